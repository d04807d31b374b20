"""The filter on both sides of the lines between its variants: two or eight outputs per
thread (by the work and the row length), one to eight views per thread of the redundancy
table, against the oracle, and the two convolutions bit for bit."""
import math

import numpy as np
import pytest
import torch

import oracle
from cases import rel_l2
from paper_2401_09283_gb300 import bp

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda", 0)
GEO = dict(pitch=0.7, sid=750.0, sdd=1200.0)


def run(raw, arc, ext):
    return bp.bp_fdk_filter(torch.as_tensor(raw, device=DEV), arc=arc, ext=ext, **GEO).cpu().numpy()


# 60 views of 160 rows are 152 * 32 * 4 - 256 pieces of work, one view more is above it;
# the full circle's weights do not depend on the number of views
@pytest.mark.parametrize("nu,ext", [(58, 0), (61, 3), (63, 0), (64, 9)])
def test_two_and_eight_outputs_per_thread_agree(nu, ext):
    raw = np.random.default_rng(nu).standard_normal((61, 160, nu)).astype(np.float32)
    few, many = run(raw[:60], 2 * math.pi, ext), run(raw, 2 * math.pi, ext)
    assert np.array_equal(few, many[:60])
    want = oracle.fdk_filter(raw[-2:], arc=2 * math.pi, ext=ext, **GEO)
    assert rel_l2(many[-2:], want) <= 1e-6


# rows at the length where few outputs go to the other variant, and odd ones
@pytest.mark.parametrize("views,nv,nu,ext", [(2, 5, 767, 0), (2, 5, 768, 7), (2, 5, 769, 0),
                                             (1, 9, 1, 2), (3, 2, 3, 0), (2, 4, 2, 5)])
def test_few_outputs_match_oracle(views, nv, nu, ext):
    raw = np.random.default_rng(nu).standard_normal((views, nv, nu)).astype(np.float32)
    want = oracle.fdk_filter(raw, arc=2 * math.pi, ext=ext, **GEO)
    assert rel_l2(run(raw, 2 * math.pi, ext), want) <= 1e-6


# views x columns per 16384: 1, 2, 3 and, clamped, 8 views per thread, with remainders
@pytest.mark.parametrize("views,nu", [(7, 500), (121, 280), (211, 247), (1023, 160)])
def test_redundancy_table_matches_oracle(views, nu):
    raw = np.random.default_rng(views).standard_normal((views, 2, nu)).astype(np.float32)
    arc = math.radians(220.0)
    want = oracle.fdk_filter(raw, arc=arc, ext=0, **GEO)
    assert rel_l2(run(raw, arc, 0), want) <= 1e-6
