// FDK preprocessing of raw line integrals (the filtering of Sec. III; the
// short-scan weights that the 200-degree arcs need): per pixel the cosine
// weight SDD / sqrt(SDD^2 + x^2 + y^2) and the redundancy weight of its ray
// (Parker's, generalised to over-scan by delta = (arc - pi)/2 in place of the
// maximum fan angle; 1/2 for a full scan), then along every detector row the
// linear convolution with the Shepp-Logan ramp h[n] = -2 / (pi^2 tau^2
// (4 n^2 - 1)), tau = pitch * SID / SDD, times tau.
//
// The ramp, the redundancy weights (view, column) and the cosine weights
// (distance from the detector's centre lines) are tabulated in FP64; the
// convolution is a direct O(nu^2) sum in FP32, taken tap by tap in the same order
// for every output.  (An FP32 FFT is 2 to 3 times further from the FP64 result.)
// With ext > 0 (truncation correction, Sec. IV-D) every weighted row is extended
// by ext pixels per side falling linearly from its edge value to 0 (extension
// pixel m = 1..ext holds edge * (1 - m/ext)) and the measured nu pixels of the
// filtered, extended row are kept.
#include "bp_internal.cuh"

namespace bpk {

namespace {

constexpr double kPi = 3.14159265358979323846;

__device__ double parker_w(double beta, double gamma, double arc) {
  const double delta = 0.5 * (arc - kPi);
  double w = 1.0;
  if (beta < 2.0 * delta + 2.0 * gamma) {
    const double s = sin(0.25 * kPi * beta / (delta + gamma));
    w = s * s;
  } else if (beta > kPi + 2.0 * gamma) {
    const double s = sin(0.25 * kPi * (kPi + 2.0 * delta - beta) / (delta - gamma));
    w = s * s;
  }
  return fmin(fmax(w, 0.0), 1.0);
}

// Layout of the tables: cosine weights of a quarter of the detector, the ramp,
// redundancy weights.
struct FdkTables {
  int nuh, nvh;          // quarter detector: distance from the nearer edge
  size_t ramp, red;      // offsets in floats
  __host__ __device__ FdkTables(int nu, int nv, int ext)
      : nuh((nu + 1) / 2),
        nvh((nv + 1) / 2),
        ramp(2 * (size_t)nuh * (size_t)nvh),
        red(ramp + 2 * ((size_t)nu + 2 * (size_t)ext) - 1) {}
};

// The tables' FP64 functions: a warp's instruction takes 16 cycles of an SM's pipe, and
// one weight is a chain of some hundred.  Small tables are spread over as many SMs as
// possible (CTAs of two warps) and take one view per thread; large ones share the fan
// angle's atan between eight.  13 views of 72 x 105, whole filter: 32.9 us with eight
// views per thread in CTAs of 256, 24.7 with one, 22.7 with one in CTAs of 64.
constexpr int RED_VIEWS = 8, TABLE_THREADS = 64;

// [nvh][nuh] (high, low) FP32 parts of the cosine weight, then h[m + ne - 1] for
// |m| < ne = nu + 2 ext, then the redundancy weight of (view j, column a) at
// j nu + a.
__global__ void fdk_tables_kernel(int V, int nu, int nv, int ext, double pitch, double sid,
                                  double sdd, double arc, int rv, float* __restrict__ tab) {
  const double tau = pitch * sid / sdd;
  const bool full = arc >= 2.0 * kPi - 1e-12;
  const double dbeta = full ? arc / V : (V > 1 ? arc / (V - 1) : 0.0);
  const int ne = nu + 2 * ext;
  const FdkTables T(nu, nv, ext);
  const long long nc = (long long)T.nuh * T.nvh, nh = 2LL * ne - 1;
  const long long nr = (long long)((V + rv - 1) / rv) * nu;  // rv views per thread
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < nc + nh + nr;
       e += (long long)gridDim.x * blockDim.x) {
    if (e < nc) {
      const int b = (int)(e / T.nuh), k = (int)(e % T.nuh);
      const double x = (k - 0.5 * (nu - 1)) * pitch, y = (b - 0.5 * (nv - 1)) * pitch;
      const double c = sdd / sqrt(sdd * sdd + x * x + y * y);
      const float hi = (float)c;
      reinterpret_cast<float2*>(tab)[e] = make_float2(hi, (float)(c - (double)hi));
    } else if (e < nc + nh) {
      const double m = (double)(e - nc - (ne - 1));
      tab[T.ramp + (e - nc)] = (float)(-2.0 / (kPi * kPi * tau * tau * (4.0 * m * m - 1.0)));
    } else {
      const long long q = e - nc - nh;
      const int j0 = (int)(q / nu) * rv, a = (int)(q % nu);
      const double g = full ? 0.0 : atan((a - 0.5 * (nu - 1)) * pitch / sdd);
      for (int j = j0; j < min(V, j0 + rv); ++j)
        tab[T.red + (size_t)j * nu + a] = full ? 0.5f : (float)parker_w(j * dbeta, g, arc);
    }
  }
}

constexpr int ROWS = 4;        // detector rows of a group, interleaved as float4
constexpr int MAX_GROUPS = 8;  // groups per CTA
constexpr int MAX_THREADS = 512;

// The ramp in shared memory, element m at m + m / 8, shifted by `shift` so that
// the taps of one block of eight steps lie in one such run: the lanes' loads
// (eight elements apart) fall in different banks and their offsets are immediates.
// (With two outputs per thread a block of two steps lies in one.)
struct RampLayout {
  int c, shift, n;  // index of output 0's first tap; elements
  __host__ __device__ RampLayout(int nu, int ext) {
    const int c0 = ext + (nu + 2 * ext) - 1;
    shift = (7 - c0) & 7;
    c = c0 + shift;
    n = (nu + 7) / 8 * 8 + c;
  }
  __host__ __device__ static int at(int m) { return m + (m >> 3); }
};

typedef unsigned long long f2;
__device__ __forceinline__ f2 splat2(float a) {
  f2 r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// grid (ceil(groups / G), V), G groups of four rows per CTA.  Dynamic shared
// memory: G x ne float4 (the weighted, extended rows, interleaved), the ramp.
//
// The convolution is nu FMAs per output, bound by the FMA pipe when the operands
// are cheap: a thread owns 8 outputs of 4 rows (16 packed accumulators) and takes,
// per tap, one broadcast 16-byte load of the rows and ONE ramp value, the other
// seven being those of the step before (a window in registers, renamed by the
// unrolling).  One output of 4 rows per thread loaded 20 bytes for four FMAs.
// The cosine weight comes from a table as a pair of FP32 values, not from an FP64
// square root and division per pixel and view (2 FP64 lanes per clock and SM).
// 248 x 480 rows of 616: 3.74 -> 1.73 ms, the FMAs alone take 1.2 ms (without the
// compiler's own choice of registers, 78 and two CTAs per SM, 1.5 % more; with 8 rows
// per thread and 126 registers 13 % more).
// OUT = 2 for problems of few outputs, whose threads are a serial chain of nu taps each
// while most of the chip is idle.
template <int OUT>
__global__ void __launch_bounds__(MAX_THREADS, 2)
    fdk_conv_kernel(const float* __restrict__ raw, int nu, int nv, int ext, int G, float tau,
                    const float* __restrict__ tab, float* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int ne = nu + 2 * ext;
  const FdkTables T(nu, nv, ext);
  const RampLayout L(nu, ext);
  float4* rows = reinterpret_cast<float4*>(smem);  // [G][ne]
  float* h = reinterpret_cast<float*>(smem + sizeof(float4) * (size_t)G * ne);
  const int j = blockIdx.y, groups = (nv + ROWS - 1) / ROWS;
  const int g0 = blockIdx.x * G, ng = min(G, groups - g0);
  const float* red = tab + T.red + (size_t)j * nu;
  const float2* cosw = reinterpret_cast<const float2*>(tab);
  for (int e = threadIdx.x; e < L.n; e += blockDim.x) {
    const int m = e - L.shift;
    h[RampLayout::at(e)] = m >= 0 && m < 2 * ne - 1 ? tab[T.ramp + m] : 0.0f;
  }
  for (int e = threadIdx.x; e < ng * nu; e += blockDim.x) {
    const int g = e / nu, k = e - g * nu;
    const float p = red[k];
    float v[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const int b = (g0 + g) * ROWS + r;
      v[r] = 0.0f;
      if (b < nv) {
        const float2 c = cosw[(size_t)min(b, nv - 1 - b) * T.nuh + min(k, nu - 1 - k)];
        // the product of the FP64 cosine weight and p, rounded once
        const float hi = __fmul_rn(c.x, p);
        const float w = __fadd_rn(hi, fmaf(c.y, p, fmaf(c.x, p, -hi)));
        v[r] = w * raw[((size_t)j * nv + b) * nu + k];
      }
    }
    rows[(size_t)g * ne + ext + k] = make_float4(v[0], v[1], v[2], v[3]);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < ng * ext; e += blockDim.x) {  // linear fall-off to 0
    const int g = e / ext, m = 1 + (e - g * ext);
    float4* q = rows + (size_t)g * ne + ext;
    const float f = 1.0f - (float)m / (float)ext;
    const float4 l = q[0], r = q[nu - 1];
    q[-m] = make_float4(l.x * f, l.y * f, l.z * f, l.w * f);
    q[nu - 1 + m] = make_float4(r.x * f, r.y * f, r.z * f, r.w * f);
  }
  __syncthreads();
  const int nt = (nu + OUT - 1) / OUT;
  for (int item = threadIdx.x; item < ng * nt; item += blockDim.x) {
    const int g = item / nt, a0 = (item - g * nt) * OUT;
    const ulonglong2* p = reinterpret_cast<const ulonglong2*>(rows + (size_t)g * ne);
    const float* hb = h + RampLayout::at(a0 + L.c);  // tap kk of output a0 + i: L.c + a0 - kk + i
    f2 acc[OUT][2], w[OUT];
#pragma unroll
    for (int i = 0; i < OUT; ++i) acc[i][0] = acc[i][1] = splat2(0.0f);
#pragma unroll
    for (int i = 1; i < OUT; ++i) w[i] = splat2(h[RampLayout::at(a0 + L.c + i)]);
#pragma unroll 1
    for (int kk = 0; kk + OUT <= ne; kk += OUT) {
#pragma unroll
      for (int q = 0; q < OUT; ++q) {
        const ulonglong2 x = p[kk + q];
        w[(OUT - q) % OUT] = splat2(hb[-q]);
#pragma unroll
        for (int i = 0; i < OUT; ++i) {
          acc[i][0] = fma2(w[(i - q + OUT) % OUT], x.x, acc[i][0]);
          acc[i][1] = fma2(w[(i - q + OUT) % OUT], x.y, acc[i][1]);
        }
      }
      hb = OUT == 8 ? hb - 9 : h + RampLayout::at(a0 + L.c - kk - OUT);
    }
#pragma unroll 1
    for (int kk = ne / OUT * OUT; kk < ne; ++kk) {
      const ulonglong2 x = p[kk];
#pragma unroll
      for (int i = 0; i < OUT; ++i) {
        const f2 wi = splat2(h[RampLayout::at(a0 + L.c - kk + i)]);
        acc[i][0] = fma2(wi, x.x, acc[i][0]);
        acc[i][1] = fma2(wi, x.y, acc[i][1]);
      }
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const int b = (g0 + g) * ROWS + r;
      if (b >= nv) break;
      float* o = out + ((size_t)j * nv + b) * nu + a0;
      float s[OUT];
#pragma unroll
      for (int i = 0; i < OUT; ++i) {
        const f2 a = acc[i][r / 2];
        s[i] = tau * __uint_as_float((unsigned)(r % 2 ? a >> 32 : a));
      }
      if (OUT == 8 && nu % 4 == 0 && a0 + OUT <= nu &&
          (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
        reinterpret_cast<float4*>(o)[0] = make_float4(s[0], s[1], s[2 % OUT], s[3 % OUT]);
        reinterpret_cast<float4*>(o)[1] = make_float4(s[4 % OUT], s[5 % OUT], s[6 % OUT], s[7 % OUT]);
      } else {
#pragma unroll
        for (int i = 0; i < OUT; ++i)
          if (a0 + i < nu) o[i] = s[i];
      }
    }
  }
}

size_t conv_smem(int nu, int ext, int G) {
  const RampLayout L(nu, ext);
  return sizeof(float4) * (size_t)G * ((size_t)nu + 2 * (size_t)ext) +
         sizeof(float) * (size_t)(RampLayout::at(L.n) + 1);
}

// Threads' work (groups of four rows x eight outputs) below which a thread takes two
// outputs, four warps on each SM, and the row length up to which it does: longer rows
// take more than one turn of a CTA.  Whole filter, us, one output per thread at first /
// eight / two: 13 x 72 x 105 (views, rows, columns) 22.7 / 22.7 / 17.7, 4 x 54 x 96 18.6 /
// 21.6 / 17.7, 1 x 480 x 616 49.3 / 54.4 / 43.0; but 2 x 20 x 1200 113 / 75 / 84.
constexpr long long FEW_ITEMS = 152 * 32 * 4;
constexpr int FEW_NU = 768;

template <int OUT>
cudaError_t conv_launch(const float* raw, int V, int nv, int nu, int ext, double pitch, double sid,
                        double sdd, const float* tab, float* out, cudaStream_t s) {
  // Groups per CTA: the share of busy threads (whole warps, whole CTAs), best
  // within 56 KiB of shared memory, so that several CTAs are resident.
  const int nt = (nu + OUT - 1) / OUT, groups = (nv + ROWS - 1) / ROWS;
  int G = 1, threads = 0;
  double best = 0.0;
  for (int g = 1; g <= (OUT == 8 ? MAX_GROUPS : 1) && g <= groups; ++g) {
    if (g > 1 && conv_smem(nu, ext, g) > 56 * 1024) break;
    const int t = (g * nt + 31) / 32 * 32 < MAX_THREADS ? (g * nt + 31) / 32 * 32 : MAX_THREADS;
    const int ctas = (groups + g - 1) / g, turns = (g * nt + t - 1) / t;
    const double busy = (double)groups * nt / ((double)ctas * turns * t);
    if (busy > best + 0.01) {
      best = busy;
      G = g;
      threads = t;
    }
  }
  const size_t smem = conv_smem(nu, ext, G);
  if (smem > 48 * 1024) {  // the same limit in every call: calls in other threads agree
    const cudaError_t e = cudaFuncSetAttribute(
        fdk_conv_kernel<OUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e != cudaSuccess) return e;
  }
  dim3 grid((groups + G - 1) / G, V);
  fdk_conv_kernel<OUT><<<grid, threads, smem, s>>>(raw, nu, nv, ext, G, (float)(pitch * sid / sdd),
                                                   tab, out);
  return cudaGetLastError();
}

}  // namespace

size_t fdk_table_floats(int V, int nu, int nv, int ext) {
  return FdkTables(nu, nv, ext).red + (size_t)V * nu;
}

cudaError_t launch_fdk_filter(const float* raw, int V, int nv, int nu, int ext, double pitch,
                              double sid, double sdd, double arc, float* tab, float* out,
                              cudaStream_t s) {
  if (V == 0 || nv == 0) return cudaSuccess;
  const long long n = (long long)fdk_table_floats(V, nu, nv, ext);
  long long nb = (n + TABLE_THREADS - 1) / TABLE_THREADS, rv = (long long)V * nu / 16384;
  if (nb > 152 * 64) nb = 152 * 64;
  rv = rv < 1 ? 1 : rv > RED_VIEWS ? RED_VIEWS : rv;
  fdk_tables_kernel<<<(int)nb, TABLE_THREADS, 0, s>>>(V, nu, nv, ext, pitch, sid, sdd, arc, (int)rv,
                                                      tab);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // few outputs: two per thread, so that four warps per SM have work
  const long long items = (long long)V * ((nv + ROWS - 1) / ROWS) * ((nu + 7) / 8);
  return items < FEW_ITEMS && nu <= FEW_NU
             ? conv_launch<2>(raw, V, nv, nu, ext, pitch, sid, sdd, tab, out, s)
             : conv_launch<8>(raw, V, nv, nu, ext, pitch, sid, sdd, tab, out, s);
}

}  // namespace bpk
