"""The filter's convolution at the edges of its tiles (8 outputs and 8 taps per
step, 4 rows per group, groups per CTA, rows longer than a CTA's threads) against
the oracle's direct convolution; rows that hold an infinity or a NaN stay alone."""
import math

import numpy as np
import pytest
import torch

import oracle
from cases import rel_l2
from paper_2401_09283_gb300 import bp

pytestmark = pytest.mark.gpu

DEV = torch.device("cuda", 0)
GEO = dict(sid=750.0, sdd=1200.0, arc=2 * math.pi)


# The bound of the filter's other tests, 1e-6 in L2.
@pytest.mark.parametrize("views,nv,nu,ext", [(1, 1, 1, 0), (2, 3, 7, 0), (2, 4, 8, 0), (1, 5, 9, 3),
                                             (2, 33, 16, 1), (1, 9, 63, 5), (3, 37, 250, 25)])
def test_tiles_match_oracle(views, nv, nu, ext):
    raw = np.random.default_rng(nu + nv).standard_normal((views, nv, nu)).astype(np.float32)
    want = oracle.fdk_filter(raw, pitch=0.7, ext=ext, **GEO)
    got = bp.bp_fdk_filter(torch.as_tensor(raw, device=DEV), pitch=0.7, ext=ext, **GEO)
    assert rel_l2(got.cpu().numpy(), want) <= 1e-6


# Rows longer than a CTA's threads, one impulse per row: a product of four rounded
# factors per output and no sum, 4 * 2^-24 (the FP64 factors' rounding to FP32 and two
# products), doubled for the weight's pair of FP32 values.
@pytest.mark.parametrize("nu,ext", [(4200, 0), (8192, 0), (7999, 96)])
def test_impulses_in_long_rows_match_oracle(nu, ext):
    raw = np.zeros((1, 5, nu), np.float32)
    for b, k in enumerate((0, 1, nu // 2, nu - 9, nu - 1)):
        raw[0, b, k] = 1.0 if ext == 0 or 0 < k < nu - 1 else 0.0
    want = oracle.fdk_filter(raw, pitch=0.05, ext=ext, **GEO)
    got = bp.bp_fdk_filter(torch.as_tensor(raw, device=DEV), pitch=0.05, ext=ext, **GEO)
    assert rel_l2(got.cpu().numpy(), want) <= 8 * 2.0 ** -24


def test_non_finite_values_stay_in_their_rows():
    raw = np.random.default_rng(1).standard_normal((2, 6, 70)).astype(np.float32)
    want = bp.bp_fdk_filter(torch.as_tensor(raw, device=DEV), pitch=0.7, **GEO).cpu().numpy()
    raw[0, 2, 5], raw[1, 3, 60] = np.inf, np.nan
    got = bp.bp_fdk_filter(torch.as_tensor(raw, device=DEV), pitch=0.7, **GEO).cpu().numpy()
    assert np.isinf(got[0, 2]).all() and np.isnan(got[1, 3]).all()
    got[0, 2], got[1, 3] = want[0, 2], want[1, 3]
    assert np.array_equal(got, want)
