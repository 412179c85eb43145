// Setup kernels of MG-CCCS (run once per grid / potential / energy).
//
//  * ECS node coordinates and the 3-point nonuniform second-difference coefficients
//    per axis and level (Sec. 2.5, Eq. (11)); coarse levels optionally on a rotated
//    contour.
//  * Diagonal D of H - E and omega/D per node, potentials injected at coincident nodes.
//  * Dense inverse of the coarsest-level operator (Gauss-Jordan, partial pivoting).
//  * Bound states of H1, H2 (Eq. (9)): of all eigenvalues (kernels_eig.cu, or here the
//    root-free implicit QR on the squared off-diagonals, Pal-Walker-Kahan form, applied
//    without conjugation to the complex-symmetric tridiagonal) the n_b with smallest real
//    part are refined by Rayleigh-quotient iteration and two shift-and-invert steps (Sec.
//    5.1.2, Sec. 5.2), normalised bilinearly, int phi^2 dz = 1 (Sec. 3.1, Remark 3).
//  * Channel potentials V^A, V^B (Sec. 4.2) and the cyclic-reduction factors of the
//    coupled-channel systems (Eqs. (28)-(29)).
#include <algorithm>

#include "common.cuh"

namespace {

__device__ __forceinline__ cplx node_z(int k, int n, double L, double R0, double ct, double st,
                                       double cg, double sg) {
  double x = (double)k * L / (double)n;
  cplx z = (x <= R0) ? cmk(x, 0.0) : cmk(R0 + (x - R0) * ct, (x - R0) * st);
  if (cg != 1.0 || sg != 0.0) z = cmul(z, cmk(cg, sg));
  return z;
}

__global__ void k_setup_axis(AxisSetup a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;   // interior index, node k = i + 1
  if (i >= a.n - 1) return;
  double ct, st, cg = 1.0, sg = 0.0;
  sincos(a.theta, &st, &ct);
  if (a.gamma != 0.0) sincos(a.gamma, &sg, &cg);
  const int k = i + 1;
  cplx zm = node_z(k - 1, a.n, a.L, a.R0, ct, st, cg, sg);
  cplx z0 = node_z(k, a.n, a.L, a.R0, ct, st, cg, sg);
  cplx zp = node_z(k + 1, a.n, a.L, a.R0, ct, st, cg, sg);
  cplx hm = csub(z0, zm), hp = csub(zp, z0);
  cplx s = cadd(hm, hp);
  cplx west = cneg(cdiv(cmk(1.0, 0.0), cmul(s, hm)));
  cplx east = cneg(cdiv(cmk(1.0, 0.0), cmul(s, hp)));
  a.west[i] = west;
  a.east[i] = east;
  a.diag[i] = cneg(cadd(west, east));
  a.w[i] = cscal(0.5, s);
}

__global__ void k_setup_diag(int mx, int my, int stride, int fine_mx, const cplx* __restrict__ dx,
                             const cplx* __restrict__ dy, const cplx* __restrict__ v1, const cplx* __restrict__ v2,
                             const cplx* __restrict__ v12, double E, double omega, cplx* __restrict__ D,
                             cplx* __restrict__ Dinv, int* status) {
  const int i = blockIdx.x * 32 + threadIdx.x;
  const int j = blockIdx.y * 8 + threadIdx.y;
  if (i >= mx || j >= my) return;
  const int fi = stride * (i + 1) - 1, fj = stride * (j + 1) - 1;   // injection at coincident nodes
  cplx d = cadd(cadd(cadd(cadd(dx[i], dy[j]), v1[fi]), v2[fj]), v12[(size_t)fj * fine_mx + fi]);
  d.x -= E;
  const size_t p = (size_t)j * mx + i;
  D[p] = d;
  if (d.x == 0.0 && d.y == 0.0) {
    atomicOr(status, MGC_ST_PIVOT);
    Dinv[p] = cmk(0.0, 0.0);
  } else {
    Dinv[p] = cdiv(cmk(omega, 0.0), d);
  }
}

// flag := 1 if a[k] != b[k] for some k (bitwise comparison of the values).
__global__ void k_compare(int n, const cplx* __restrict__ a, const cplx* __restrict__ b, int* flag) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n && (a[k].x != b[k].x || a[k].y != b[k].y)) atomicOr(flag, 1);
}

// flag := 1 if some node of the uniform box has a complex diagonal.
__global__ void k_box_real_check(int mx, int ux, int uy, const cplx* __restrict__ D, int* flag) {
  const int i = blockIdx.x * 32 + threadIdx.x;
  const int j = blockIdx.y * 8 + threadIdx.y;
  if (i >= ux || j >= uy) return;
  if (D[(size_t)j * mx + i].y != 0.0) atomicOr(flag, 1);
}

// Dense inverse of the coarsest operator by Gauss-Jordan elimination with partial
// pivoting on the augmented matrix [A | I] (nc x 2nc, row-major, in global memory),
// one pivot per pair of launches: k_gj_pivot (one block: pivot search, row swap, row
// scaling, multiplier column) and k_gj_eliminate (all SMs: rank-1 update of the
// columns right of the pivot).  A zero pivot sets MGC_ST_PIVOT and every later launch
// of the elimination returns at once.

__global__ void k_gj_assemble(StencilView s, cplx* __restrict__ aug) {
  const int nc = s.mx * s.my;
  const long long w2 = 2LL * nc;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nc * w2;
       q += (long long)gridDim.x * blockDim.x) {
    const int p = (int)(q / w2), c = (int)(q % w2);
    const int i = p % s.mx, j = p / s.mx;
    cplx v = cmk(0.0, 0.0);
    if (c == p) v = s.D[p];
    else if (i > 0 && c == p - 1) v = s.west_x[i];
    else if (i + 1 < s.mx && c == p + 1) v = s.east_x[i];
    else if (j > 0 && c == p - s.mx) v = s.west_y[j];
    else if (j + 1 < s.my && c == p + s.mx) v = s.east_y[j];
    else if (c == nc + p) v = cmk(1.0, 0.0);
    aug[q] = v;
  }
}

__global__ void __launch_bounds__(1024) k_gj_pivot(int nc, cplx* __restrict__ aug, cplx* __restrict__ fac, int k,
                                                   int* __restrict__ status) {
  __shared__ double sval[1024];
  __shared__ int sidx[1024];
  const int t = threadIdx.x;
  const long long w2 = 2LL * nc;
  if (*status & MGC_ST_PIVOT) return;
  // pivot search over rows k..nc-1 (largest modulus, lowest index on ties)
  double best = -1.0;
  int bi = k;
  for (int r = k + t; r < nc; r += blockDim.x) {
    const double v = cmod(aug[r * w2 + k]);
    if (v > best) { best = v; bi = r; }
  }
  sval[t] = best;
  sidx[t] = bi;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (t < o) {
      const double v2 = sval[t + o];
      const int i2 = sidx[t + o];
      if (v2 > sval[t] || (v2 == sval[t] && i2 < sidx[t])) { sval[t] = v2; sidx[t] = i2; }
    }
    __syncthreads();
  }
  const int piv = sidx[0];
  if (sval[0] == 0.0) {
    if (t == 0) atomicOr(status, MGC_ST_PIVOT);
    return;
  }
  if (piv != k)
    for (int c = k + t; c < w2; c += blockDim.x) {
      const cplx a = aug[k * w2 + c];
      aug[k * w2 + c] = aug[piv * w2 + c];
      aug[piv * w2 + c] = a;
    }
  __syncthreads();
  const cplx pv = aug[k * w2 + k];
  __syncthreads();
  for (int c = k + t; c < w2; c += blockDim.x) aug[k * w2 + c] = cdiv(aug[k * w2 + c], pv);
  for (int r = t; r < nc; r += blockDim.x) fac[r] = r == k ? cmk(0.0, 0.0) : aug[r * w2 + k];
}

__global__ void k_gj_eliminate(int nc, cplx* __restrict__ aug, const cplx* __restrict__ fac, int k,
                               const int* __restrict__ status) {
  if (*status & MGC_ST_PIVOT) return;
  const long long w2 = 2LL * nc;
  const long long w = w2 - k - 1;                    // columns right of the pivot
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < nc * w;
       q += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(q / w);
    if (r == k) continue;
    const long long c = k + 1 + q % w;
    aug[r * w2 + c] = cfms(fac[r], aug[k * w2 + c], aug[r * w2 + c]);
  }
}

__global__ void k_gj_extract(int nc, const cplx* __restrict__ aug, cplx* __restrict__ Ainv) {
  const long long w2 = 2LL * nc;
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < (long long)nc * nc;
       q += (long long)gridDim.x * blockDim.x) {
    const long long r = q / nc, c = q % nc;
    Ainv[q] = aug[r * w2 + nc + c];
  }
}

// ---- bound states ---------------------------------------------------------------

// 1/z = conj(z)/|z|^2 (magnitudes here stay far from under/overflow).
__device__ __forceinline__ cplx crecip(cplx z) {
  const double q = 1.0 / (z.x * z.x + z.y * z.y);
  return cmk(z.x * q, -z.y * q);
}

// Eigenvalues of the complex-symmetric tridiagonal with diagonal a[0..m) and squared
// off-diagonals b2[k] (coupling k and k+1; the squares are the products east_k west_{k+1},
// so no square root is taken) by implicit QR sweeps in the root-free form of Pal,
// Walker and Kahan (B. N. Parlett, The Symmetric Eigenvalue Problem, Sec. 8-15), applied
// without conjugation, with a Wilkinson shift from the trailing 2x2 block and deflation
// at the bottom of the unreduced block.  a is overwritten with the eigenvalues.
// Returns false on a zero pivot or when the sweep budget is exhausted.
__device__ bool qr_rootfree_eigenvalues(int m, cplx* a, cplx* b2) {
  const double eps2 = 4.93038065763132e-32;          // (2^-52)^2
  long long budget = 40LL * m + 100;
  int hi = m - 1;
  while (hi > 0) {
    int lo = hi;
    while (lo > 0 && cabs1(b2[lo - 1]) > eps2 * cabs1(a[lo - 1]) * cabs1(a[lo])) --lo;
    if (lo == hi) {
      --hi;
      continue;
    }
    if (--budget < 0) return false;
    // shift: eigenvalue of the trailing 2x2 block nearest a[hi]
    const cplx dlt = cscal(0.5, csub(a[hi - 1], a[hi]));
    const cplx rt = csqrt_p(cadd(cmul(dlt, dlt), b2[hi - 1]));
    const cplx dp = cadd(dlt, rt), dm = csub(dlt, rt);
    const cplx den = (cabs2(dp) >= cabs2(dm)) ? dp : dm;
    const cplx sigma = (den.x == 0.0 && den.y == 0.0) ? a[hi] : csub(a[hi], cmul(b2[hi - 1], crecip(den)));
    // one root-free QR sweep over lo..hi
    cplx c2 = cmk(1.0, 0.0), s2 = cmk(0.0, 0.0);
    cplx gam = csub(a[lo], sigma);
    cplx p = cmul(gam, gam);
    for (int k = lo; k < hi; ++k) {
      const cplx r = cadd(p, b2[k]);
      if (r.x == 0.0 && r.y == 0.0) return false;
      if (k > lo) b2[k - 1] = cmul(s2, r);
      const cplx c2old = c2;
      const cplx rinv = crecip(r);
      c2 = cmul(p, rinv);
      s2 = cmul(b2[k], rinv);
      const cplx gold = gam;
      const cplx alpha = csub(a[k + 1], sigma);
      gam = csub(cmul(c2, alpha), cmul(s2, gold));
      a[k] = cadd(csub(cadd(gold, alpha), gam), sigma);
      p = (c2.x == 0.0 && c2.y == 0.0) ? cmul(c2old, b2[k]) : cmul(cmul(gam, gam), crecip(c2));
    }
    b2[hi - 1] = cmul(s2, p);
    a[hi] = cadd(gam, sigma);
  }
  for (int k = 0; k < m; ++k)
    if (!isfinite(a[k].x) || !isfinite(a[k].y)) return false;
  return true;
}

// ---- refinement of the bound states: one block per state.
//
// A shift-and-invert step at an eigenvalue z known to rounding needs no elimination: with the
// quadrature weights w_k (w_k east_k = w_{k+1} west_{k+1}, diag_k = -(west_k + east_k)) and the
// flux F_k = w_k east_k (u_{k+1} - u_k), the rows of (H1 - z) u = 0 read
//   F_k = F_{k-1} + w_k (z - v_k) u_k,   u_{k+1} = u_k + F_k / (w_k east_k),
// and the solution of (H1 - z) x = gamma e_r is the solution uL started at the first row for
// k <= r and the one uR started at the last row for k >= r, matched at r.  r is taken where
// |uL uR|, proportional to the diagonal of the inverse, is largest, so neither is carried into
// a region where it decays.  Both are linear recurrences: a thread forms the 2 x 2 transfer
// matrix of its rows, a scan over the threads gives each its starting vector, and it then walks
// its rows (four warps from either end).  Values carry power-of-two exponents of their own.
constexpr int BS_THREADS = 256, BS_HALF = BS_THREADS / 2, BS_WARPS = BS_HALF / 32;
constexpr int BS_SMEM = 200 * 1024;

// Workspace of a state: 1/(w east), uL (then x), uR, and the exponents of uL and uR.
__host__ __device__ constexpr size_t states_bytes(int m) { return (sizeof(cplx) * 3 + sizeof(int) * 2) * (size_t)m; }

__device__ __forceinline__ int hi_max(int m, cplx z) {
  return max(m, max(__double2hiint(z.x) & 0x7fffffff, __double2hiint(z.y) & 0x7fffffff));
}
// 2^-e for the exponent e of the high word hm, which is added to *ex (nothing for zero and beyond 2^1000).
__device__ __forceinline__ double pow2_take(int hm, int* ex) {
  const int e = (hm >> 20) - 1023;
  if (hm < (1 << 20) || e > 1000) return 1.0;
  *ex += e;
  return __hiloint2double((1023 - e) << 20, 0);
}

// (u, F) after = [a b; c d] (u, F) before, times 2^e.
struct Transfer2 {
  cplx a, b, c, d;
  int e;
};
__device__ __forceinline__ void rescale(Transfer2& t) {
  const double f = pow2_take(hi_max(hi_max(hi_max(hi_max(0, t.a), t.b), t.c), t.d), &t.e);
  t.a = cscal(f, t.a); t.b = cscal(f, t.b); t.c = cscal(f, t.c); t.d = cscal(f, t.d);
}
__device__ __forceinline__ void rescale(cplx& u, cplx& F, int& e) {
  const double f = pow2_take(hi_max(hi_max(0, u), F), &e);
  u = cscal(f, u);
  F = cscal(f, F);
}
// t <- t o s (s acts first)
__device__ __forceinline__ Transfer2 compose(const Transfer2& t, const Transfer2& s) {
  Transfer2 r;
  r.a = cfma(t.a, s.a, cmul(t.b, s.c));
  r.b = cfma(t.a, s.b, cmul(t.b, s.d));
  r.c = cfma(t.c, s.a, cmul(t.d, s.c));
  r.d = cfma(t.c, s.b, cmul(t.d, s.d));
  r.e = t.e + s.e;
  rescale(r);
  return r;
}
__device__ __forceinline__ cplx shfl_up_c(cplx z, int o) {
  return cmk(__shfl_up_sync(0xffffffffu, z.x, o), __shfl_up_sync(0xffffffffu, z.y, o));
}
__device__ __forceinline__ Transfer2 shfl_up_t(const Transfer2& t, int o) {
  return Transfer2{shfl_up_c(t.a, o), shfl_up_c(t.b, o), shfl_up_c(t.c, o), shfl_up_c(t.d, o),
                   __shfl_up_sync(0xffffffffu, t.e, o)};
}
constexpr int HI_BIG = (1023 + 400) << 20, HI_SMALL = (1023 - 400) << 20;   // 2^400, 2^-400
__device__ __forceinline__ bool off_range(int hm) { return hm > HI_BIG || hm < HI_SMALL; }

// Sums of two complex values over the block, to every thread (fixed order).
__device__ void bs_sum2(cplx& a, cplx& b, double (*sh)[BS_THREADS / 32]) {
  double v[4] = {a.x, a.y, b.x, b.y};
#pragma unroll
  for (int c = 0; c < 4; ++c) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[c] += __shfl_down_sync(0xffffffffu, v[c], o);
    if ((threadIdx.x & 31) == 0) sh[c][threadIdx.x >> 5] = v[c];
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    v[c] = sh[c][0];
#pragma unroll
    for (int w = 1; w < BS_THREADS / 32; ++w) v[c] += sh[c][w];
  }
  __syncthreads();
  a = cmk(v[0], v[1]);
  b = cmk(v[2], v[3]);
}

// The entry of largest key (lowest index on ties) over the block, to every thread.
__device__ void bs_argmax(double& key, int& idx, double (*sh)[BS_THREADS / 32]) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double k2 = __shfl_xor_sync(0xffffffffu, key, o);
    const int i2 = __shfl_xor_sync(0xffffffffu, idx, o);
    if (k2 > key || (k2 == key && i2 < idx)) { key = k2; idx = i2; }
  }
  if ((threadIdx.x & 31) == 0) { sh[0][threadIdx.x >> 5] = key; sh[1][threadIdx.x >> 5] = (double)idx; }
  __syncthreads();
  key = sh[0][0];
  idx = (int)sh[1][0];
#pragma unroll
  for (int w = 1; w < BS_THREADS / 32; ++w) {
    const double k2 = sh[0][w];
    const int i2 = (int)sh[1][w];
    if (k2 > key || (k2 == key && i2 < idx)) { key = k2; idx = i2; }
  }
  __syncthreads();
}

// Block q: the eigenvalue with the q-th smallest real part (ties: lower index) of the m given,
// Rayleigh-quotient iteration from it (each step a shift-and-invert step and the bilinear
// quotient of its result), the paper's two shift-and-invert steps, and the bilinear
// normalisation.  The quotient x^T W H1 x = sum w v x^2 - sum w east (x_{k+1} - x_k)^2 is summed
// without the cancellation of H1 x.  Bound by the FP64 pipe of the block's one SM (a warp's FP64
// instruction occupies its quarter of an SM for 64 cycles however few lanes need it).  1023
// rows, three states: 45.8 ms with one thread per state walking pivoted tridiagonal LU factors
// in global memory, 4.3 ms with the elimination run from both ends by two threads in shared
// memory, 0.26 ms so.
__global__ void __launch_bounds__(BS_THREADS) k_bound_states(int m, const cplx* __restrict__ west,
                                                             const cplx* __restrict__ east,
                                                             const cplx* __restrict__ v, const cplx* __restrict__ w,
                                                             cplx* __restrict__ lam, cplx* __restrict__ phi,
                                                             cplx* __restrict__ scratch, int in_smem, int* status,
                                                             const cplx* __restrict__ eig) {
  extern __shared__ cplx bs_work[];
  __shared__ double sh[4][BS_THREADS / 32];
  __shared__ Transfer2 tot[2][BS_WARPS];
  __shared__ int no_eig;
  const int q = blockIdx.x, t = threadIdx.x;
  if (t == 0) no_eig = *status & MGC_ST_EIG;         // one read: another block may set it meanwhile
  __syncthreads();
  if (no_eig) return;
  cplx* base = in_smem ? bs_work : scratch + (size_t)q * ((states_bytes(m) + sizeof(cplx) - 1) / sizeof(cplx));
  cplx *ic = base, *uL = base + m, *uR = base + 2 * (size_t)m, *x = uL;
  int *eL = reinterpret_cast<int*>(base + 3 * (size_t)m), *eR = eL + m;
  const cplx zero = cmk(0.0, 0.0), one = cmk(1.0, 0.0);
  // the q-th smallest real part: q + 1 passes, each for the least (value, index) beyond the last
  double last = 0.0;
  int li = -1;
  for (int s = 0; s <= q; ++s) {
    double best = -INFINITY;
    int bi = m;
    for (int k = t; k < m; k += BS_THREADS) {
      const double r = eig[k].x;
      if (li >= 0 && !(r > last || (r == last && k > li))) continue;
      if (bi == m || -r > best) { best = -r; bi = k; }
    }
    bs_argmax(best, bi, sh);
    last = -best;
    li = bi < m ? bi : 0;
  }
  cplx lmb = eig[li];
  for (int k = t; k < m; k += BS_THREADS) ic[k] = cdiv(one, cmul(w[k], east[k]));
  const int dir = t / BS_HALF, g = t % BS_HALF, wq = g >> 5, lane = t & 31;
  const int cn = (m + BS_HALF - 1) / BS_HALF;
  const int g0 = min(g * cn, m), g1 = min(g0 + cn, m);   // this thread's steps, counted from its end
  const cplx cs = cmul(w[0], west[0]);

  // x = the solution of (H1 - z) x = gamma e_r, x_r = 1
  auto shift_invert = [&](cplx z) {
    __syncthreads();
    Transfer2 T{one, zero, zero, one, 0};
    for (int p = g0; p < g1; ++p) {
      const int k = dir ? m - 1 - p : p;
      const cplx qk = cmul(w[k], csub(z, v[k])), i = ic[k];
      if (dir == 0) {
        T.c = cfma(qk, T.a, T.c); T.d = cfma(qk, T.b, T.d);
        T.a = cfma(i, T.c, T.a);  T.b = cfma(i, T.d, T.b);
      } else {
        T.a = cfms(i, T.c, T.a);  T.b = cfms(i, T.d, T.b);
        T.c = cfms(qk, T.a, T.c); T.d = cfms(qk, T.b, T.d);
      }
      if (off_range(hi_max(hi_max(0, T.a), T.b))) rescale(T);
    }
    rescale(T);
#pragma unroll
    for (int o = 1; o < 32; o *= 2) {
      const Transfer2 s = shfl_up_t(T, o);
      if (lane >= o) T = compose(T, s);
    }
    if (lane == 31) tot[dir][wq] = T;
    Transfer2 E = shfl_up_t(T, 1);
    if (lane == 0) E = Transfer2{one, zero, zero, one, 0};
    __syncthreads();
    // (u, F) before the first row, carried to this thread's first step
    cplx u = dir ? zero : one, F = dir ? one : cs;
    int e = 0;
    auto act = [&](const Transfer2& s) {
      const cplx u2 = cfma(s.a, u, cmul(s.b, F)), F2 = cfma(s.c, u, cmul(s.d, F));
      u = u2;
      F = F2;
      e += s.e;
      rescale(u, F, e);
    };
    for (int b = 0; b < wq; ++b) act(tot[dir][b]);
    act(E);
    for (int p = g0; p < g1; ++p) {
      const int k = dir ? m - 1 - p : p;
      const cplx qk = cmul(w[k], csub(z, v[k])), i = ic[k];
      if (dir == 0) {
        uL[k] = u;
        eL[k] = e;
        F = cfma(qk, u, F);
        u = cfma(i, F, u);
      } else {
        u = cfms(i, F, u);
        uR[k] = u;
        eR[k] = e;
        F = cfms(qk, u, F);
      }
      if (off_range(hi_max(hi_max(0, u), F))) rescale(u, F, e);
    }
    __syncthreads();
    // log2 |uL uR| to within one (the high words as fixed-point numbers)
    double key = -INFINITY;
    int r = m;
    for (int k = t; k < m; k += BS_THREADS) {
      const double a = cabs1(uL[k]), b = cabs1(uR[k]);
      if (!(a > 0.0) || !(b > 0.0)) continue;
      const double l = (double)(eL[k] + eR[k]) + 0x1p-20 * (double)(__double2hiint(a) + __double2hiint(b));
      if (r == m || l > key) { key = l; r = k; }
    }
    bs_argmax(key, r, sh);
    if (r >= m) r = 0;
    const cplx sl = cdiv(one, uL[r]), sr = cdiv(one, uR[r]);
    const int el = eL[r], er = eR[r];
    __syncthreads();
    for (int k = t; k < m; k += BS_THREADS) {
      const cplx y = k <= r ? cmul(sl, uL[k]) : cmul(sr, uR[k]);
      const int sh2 = k <= r ? eL[k] - el : eR[k] - er;
      x[k] = cmk(scalbn(y.x, sh2), scalbn(y.y, sh2));
    }
    __syncthreads();
  };
  // bilinear Rayleigh quotient x^T W H1 x / x^T W x
  auto quotient = [&]() {
    cplx num = zero, den = zero;
    for (int k = t; k < m; k += BS_THREADS) {
      const cplx xk = x[k], d = csub(k + 1 < m ? x[k + 1] : zero, xk);
      const cplx wx2 = cmul(w[k], cmul(xk, xk));
      den = cadd(den, wx2);
      num = cfma(v[k], wx2, num);
      num = cfms(cmul(w[k], east[k]), cmul(d, d), num);
      if (k == 0) num = cfms(cs, cmul(xk, xk), num);
    }
    bs_sum2(num, den, sh);
    return cdiv(num, den);
  };
  for (int it = 0; it < 6; ++it) {
    shift_invert(lmb);
    const cplx ln = quotient();
    const bool conv = cabs1(csub(ln, lmb)) <= 1e-14 * fmax(1.0, cabs1(ln));
    lmb = ln;
    if (conv) break;
  }
  for (int it = 0; it < 2; ++it) {
    shift_invert(lmb);
    lmb = quotient();
  }
  // bilinear normalisation sum w x^2 = 1, then Re x > 0 at the entry of largest modulus
  cplx s = zero, unused = zero;
  for (int k = t; k < m; k += BS_THREADS) s = cfma(w[k], cmul(x[k], x[k]), s);
  bs_sum2(s, unused, sh);
  cplx inv = cdiv(one, csqrt_p(s));
  double best = -1.0;
  int kb = 0;
  for (int k = t; k < m; k += BS_THREADS) {
    const double a = cabs2(cmul(x[k], inv));
    if (a > best) { best = a; kb = k; }
  }
  bs_argmax(best, kb, sh);
  if (cmul(x[kb], inv).x < 0.0) inv = cneg(inv);
  bool fin = isfinite(lmb.x) && isfinite(lmb.y);
  for (int k = t; k < m; k += BS_THREADS) {
    const cplx y = cmul(x[k], inv);
    phi[(size_t)q * m + k] = y;
    fin = fin && isfinite(y.x) && isfinite(y.y);
  }
  if (t == 0) lam[q] = lmb;
  if (!fin) atomicOr(status, MGC_ST_EIG);
}

// Two states that refined onto the same eigenvalue mean the estimates were too poor.
__global__ void k_states_distinct(int nb, const cplx* __restrict__ lam, int* status) {
  const int a = threadIdx.x / MGC_MAX_NB, b = threadIdx.x % MGC_MAX_NB;
  if (a < b && b < nb && cabs1(csub(lam[a], lam[b])) <= 1e-10 * fmax(1.0, cabs1(lam[a])))
    atomicOr(status, MGC_ST_EIG);
}

// All eigenvalues by the FP64 root-free QR (one thread): the spectrum entry point's method 1, and
// setup's fallback when the Ehrlich-Aberth iteration does not converge.
__global__ void k_qr_spectrum(int m, const cplx* __restrict__ west, const cplx* __restrict__ east,
                              const cplx* __restrict__ diag, const cplx* __restrict__ v, cplx* __restrict__ scratch,
                              cplx* __restrict__ out, int* status) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  cplx* d = scratch;
  cplx* e2 = scratch + m;
  for (int k = 0; k < m; ++k) {
    d[k] = cadd(diag[k], v[k]);
    e2[k] = (k + 1 < m) ? cmul(east[k], west[k + 1]) : cmk(0.0, 0.0);
  }
  if (!qr_rootfree_eigenvalues(m, d, e2)) {
    atomicOr(status, MGC_ST_EIG);
    return;
  }
  for (int k = 0; k < m; ++k) out[k] = d[k];
}

__global__ void k_weight_states(int m, int nb, const cplx* __restrict__ w, const cplx* __restrict__ phi,
                                cplx* __restrict__ wphi) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= m * nb) return;
  wphi[t] = cmul(w[t % m], phi[t]);
}

// out[row][a][b] = out[row][b][a] = sum_k wst_a(k) st_b(k) v12(row, k);
// v12(row, k) = v12[row * rs + k * ks].  One block per (row, pair a <= b).
__global__ void __launch_bounds__(256) k_channel_potentials(int rows, int len, int nb, long long rs, long long ks,
                                                            const cplx* __restrict__ wst,
                                                            const cplx* __restrict__ st,
                                                            const cplx* __restrict__ v12, cplx* __restrict__ out) {
  __shared__ double sh[2][8];
  const int row = blockIdx.x;
  int pair = blockIdx.y, a = 0;
  while (pair >= nb - a) { pair -= nb - a; ++a; }
  const int b = a + pair;
  cplx acc = cmk(0.0, 0.0);
  for (int k = threadIdx.x; k < len; k += 256)
    acc = cfma(cmul(wst[(size_t)a * len + k], st[(size_t)b * len + k]), v12[row * rs + k * ks], acc);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    acc.x += __shfl_down_sync(0xffffffffu, acc.x, o);
    acc.y += __shfl_down_sync(0xffffffffu, acc.y, o);
  }
  if ((threadIdx.x & 31) == 0) { sh[0][threadIdx.x >> 5] = acc.x; sh[1][threadIdx.x >> 5] = acc.y; }
  __syncthreads();
  if (threadIdx.x == 0) {
    cplx tot = cmk(0.0, 0.0);
    for (int k = 0; k < 8; ++k) tot = cadd(tot, cmk(sh[0][k], sh[1][k]));
    out[((size_t)row * nb + a) * nb + b] = tot;
    out[((size_t)row * nb + b) * nb + a] = tot;
  }
}

// Parallel cyclic reduction factors of the two coupled-channel systems (Eqs. (28)-(29)):
// rows k = 0..m-1 of A_k x_{k-1} + B_k x_k + C_k x_{k+1} = r_k with n_b x n_b blocks
// (A_k, C_k the 1D Laplacian couplings times the identity, B_k the channel block).
// Level l (stride s = 2^l) eliminates every row's couplings to k +- s with the rows
// k +- s themselves: alpha = A_k B_{k-s}^{-1}, gamma = C_k B_{k+s}^{-1},
//   A_k <- -alpha A_{k-s},  B_k <- B_k - alpha C_{k-s} - gamma A_{k+s},  C_k <- -gamma C_{k+s};
// after ceil(log2 m) levels no coupling is left and x_k = B_k^{-1} r_k.  The first p levels
// eliminate every other remaining row: the eliminated row leaves B_k^{-1}, B_k^{-1} A_k and
// B_k^{-1} C_k of its level for the back substitution and takes no part in the later levels,
// which then couple the separators (the last row of every 2^p) only.  One launch per level
// for both systems, one warp per row with the row's blocks in shared memory; a launch ends
// with the inverses of the blocks it made, so the next one finds its neighbours'.  The state of
// a system is A, B, C and B^{-1} of every row, double-buffered: 8 m n_b^2 entries.
// Bound by the latency of the inverse's pivot chain.  Two systems of 1023 rows, n_b = 3: 6.6 ms
// as one block per system that updated every row at every level, 0.18 ms so.
constexpr int CF_WARPS = 4;

// The systems of both channels and what their first level is made from.
struct ChannelSetup {
  CRSystem S;
  const cplx *diag, *v, *lam, *Vc, *sub, *sup;
  cplx* scratch;                 // 8 m nb^2
};

// In-place inverse of the nb x nb matrix M of this warp by Gauss-Jordan elimination with
// partial pivoting on [M | I] in aug (row pitch 2 nb); false on a zero pivot.
__device__ bool warp_inverse(int nb, const cplx* M, cplx* aug, cplx* out) {
  const int lane = threadIdx.x & 31, w2 = 2 * nb;
  for (int e = lane; e < nb * w2; e += 32) {
    const int r = e / w2, c = e - r * w2;
    aug[e] = c < nb ? M[r * nb + c] : cmk(c - nb == r ? 1.0 : 0.0, 0.0);
  }
  __syncwarp();
  for (int k = 0; k < nb; ++k) {
    int piv = k;
    double best = cabs2(aug[k * w2 + k]);
    for (int r = k + 1; r < nb; ++r) {
      const double a = cabs2(aug[r * w2 + k]);
      if (a > best) { best = a; piv = r; }
    }
    if (best == 0.0) return false;                       // the same for every lane
    __syncwarp();
    if (piv != k && lane < w2) {
      const cplx t = aug[k * w2 + lane];
      aug[k * w2 + lane] = aug[piv * w2 + lane];
      aug[piv * w2 + lane] = t;
    }
    __syncwarp();
    const cplx inv = cdiv(cmk(1.0, 0.0), aug[k * w2 + k]);
    __syncwarp();
    if (lane < w2) aug[k * w2 + lane] = cmul(aug[k * w2 + lane], inv);
    // the multipliers of this lane's entries, read before column k is cleared
    cplx f[(2 * MGC_MAX_NB * MGC_MAX_NB + 31) / 32];
    __syncwarp();
#pragma unroll
    for (int q = 0; q < (2 * MGC_MAX_NB * MGC_MAX_NB + 31) / 32; ++q) {
      const int e = lane + 32 * q;
      if (e < nb * w2) f[q] = aug[e / w2 * w2 + k];
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < (2 * MGC_MAX_NB * MGC_MAX_NB + 31) / 32; ++q) {
      const int e = lane + 32 * q;
      if (e < nb * w2 && e / w2 != k) aug[e] = cfms(f[q], aug[k * w2 + e % w2], aug[e]);
    }
    __syncwarp();
  }
  for (int e = lane; e < nb * nb; e += 32) out[e] = aug[e / nb * w2 + nb + e % nb];
  return true;
}

// Entry (r, c) of X Y for nb x nb row-major blocks.
__device__ __forceinline__ cplx block_dot(int nb, const cplx* X, const cplx* Y, int r, int c) {
  cplx acc = cmk(0.0, 0.0);
  for (int k = 0; k < nb; ++k) acc = cfma(X[r * nb + k], Y[k * nb + c], acc);
  return acc;
}

// Reduction levels of the separators' system.
__host__ __device__ constexpr int sep_levels(int ns) {
  int q = 0;
  while ((1 << q) < ns) ++q;
  return q;
}

// Level l >= 0 of the reduction, or with l = -1 its start: the blocks of the unreduced rows.
__global__ void __launch_bounds__(32 * CF_WARPS) k_channel_factor(ChannelSetup ca, ChannelSetup cb, double E, int l,
                                                                  int* status) {
  extern __shared__ cplx cf_sh[];
  const ChannelSetup& P = blockIdx.y == 0 ? ca : cb;
  const CRSystem& S = P.S;
  const int nb = S.nb, nb2 = nb * nb, m = S.m;
  const int lane = threadIdx.x & 31, k = blockIdx.x * CF_WARPS + (threadIdx.x >> 5);
  // whole warps leave; no block barrier below
  const int R = 1 << S.p, rank = k / R, i = k % R, pq = S.p + sep_levels(S.ns);
  if (k >= m || l >= pq || (l > 0 && (k + 1) % (1 << min(l, S.p)) != 0)) return;
  cplx* sh = cf_sh + (size_t)(threadIdx.x >> 5) * 12 * nb2;   // ten blocks, then [B | I]
  const size_t blk = (size_t)m * nb2, row = (size_t)k * nb2;
  const int cur = (l + 2) & 1;                             // level l reads buffer cur, the start writes buffer 0
  const cplx* in = P.scratch + cur * 4 * blk;
  cplx* out = P.scratch + (l < 0 ? 0 : (cur ^ 1) * 4 * blk);
  cplx* Bn = sh + 9 * nb2;
  if (l < 0) {
    cplx base = cadd(P.diag[k], P.v[k]);
    base.x -= E;
    for (int e = lane; e < nb2; e += 32) {
      const int r = e / nb, c = e - r * nb;
      cplx val = P.Vc[row + e];
      if (r == c) val = cadd(val, cadd(base, P.lam[r]));
      Bn[e] = val;
      out[row + e] = (r == c && k > 0) ? P.sub[k] : cmk(0.0, 0.0);
      out[blk + row + e] = val;
      out[2 * blk + row + e] = (r == c && k < m - 1) ? P.sup[k] : cmk(0.0, 0.0);
    }
  } else {
    const int s = 1 << l;
    const bool lo = k - s >= 0, hi = k + s < m;
    const size_t rl = row - (lo ? (size_t)s * nb2 : 0), rh = row + (hi ? (size_t)s * nb2 : 0);
    // own A, C; the neighbours' B^{-1}, A, C (the row itself where a neighbour is missing)
    cplx *A = sh, *C = sh + nb2, *Il = sh + 2 * nb2, *Al = sh + 3 * nb2, *Cl = sh + 4 * nb2, *Ih = sh + 5 * nb2,
         *Ah = sh + 6 * nb2, *Ch = sh + 7 * nb2, *al = sh + 8 * nb2, *ga = sh + 10 * nb2;   // ga: in [B | I] until then
    for (int e = lane; e < nb2; e += 32) {
      A[e] = in[row + e];
      C[e] = in[2 * blk + row + e];
      Il[e] = in[3 * blk + rl + e];
      Al[e] = in[rl + e];
      Cl[e] = in[2 * blk + rl + e];
      Ih[e] = in[3 * blk + rh + e];
      Ah[e] = in[rh + e];
      Ch[e] = in[2 * blk + rh + e];
    }
    __syncwarp();
    cplx* pack = S.pack + rank * cr_pack_entries(R, S.p, nb);
    if (l < S.p && ((k + 1) >> l) % 2 != 0) {
      const cplx* Bi = in + 3 * blk + row;
      cplx* d = pack + ((size_t)(R - 1) * 2 + S.p + (size_t)i * 3) * nb2;
      for (int e = lane; e < nb2; e += 32) {
        const int r = e / nb, c = e - r * nb;
        d[e] = block_dot(nb, Bi, A, r, c);
        d[nb2 + e] = block_dot(nb, Bi, C, r, c);
        d[2 * nb2 + e] = Bi[e];
      }
      return;
    }
    // where alpha, gamma go, and a separator's gamma also to the next CTA
    cplx* pa = l < S.p ? pack + ((size_t)(R - (R >> l)) + (i + 1) / (2 * s) - 1) * 2 * nb2
                       : S.sfac + ((size_t)(l - S.p) * S.ns + rank) * 2 * nb2;
    cplx* pv = l < S.p && i == R - 1 && k + 1 < m
                   ? pack + cr_pack_entries(R, S.p, nb) + ((size_t)(R - 1) * 2 + l) * nb2 : nullptr;
    for (int e = lane; e < nb2; e += 32) {
      const int r = e / nb, c = e - r * nb;
      al[e] = lo ? block_dot(nb, A, Il, r, c) : cmk(0.0, 0.0);
      ga[e] = hi ? block_dot(nb, C, Ih, r, c) : cmk(0.0, 0.0);
      pa[e] = al[e];
      pa[nb2 + e] = ga[e];
      if (pv) pv[e] = ga[e];
    }
    __syncwarp();
    for (int e = lane; e < nb2; e += 32) {
      const int r = e / nb, c = e - r * nb;
      cplx b = in[blk + row + e], a2 = cmk(0.0, 0.0), c2 = a2;
      if (lo) {
        b = csub(b, block_dot(nb, al, Cl, r, c));
        a2 = cneg(block_dot(nb, al, Al, r, c));
      }
      if (hi) {
        b = csub(b, block_dot(nb, ga, Ah, r, c));
        c2 = cneg(block_dot(nb, ga, Ch, r, c));
      }
      Bn[e] = b;
      out[row + e] = a2;
      out[blk + row + e] = b;
      out[2 * blk + row + e] = c2;
    }
  }
  __syncwarp();
  // the last level's inverses (of the only level when the separators are not coupled)
  cplx* dst = l == pq - 1 && (k + 1) % R == 0 ? S.sfac + ((size_t)(pq - S.p) * S.ns * 2 + rank) * nb2
                                              : out + 3 * blk + row;
  if (!warp_inverse(nb, Bn, sh + 10 * nb2, dst)) {
    if (lane == 0) atomicOr(status, MGC_ST_PIVOT);
    for (int e = lane; e < nb2; e += 32) dst[e] = cmk(0.0, 0.0);
  }
}

// Column blockIdx.x of the inverse of the separators' system: their parallel cyclic reduction
// applied to a unit vector, one thread per (separator, component).
__global__ void __launch_bounds__(CR_CLUSTER * MGC_MAX_NB) k_separator_inverse(CRSystem SA, CRSystem SB) {
  __shared__ cplx x[2][CR_CLUSTER * MGC_MAX_NB];
  const CRSystem& S = blockIdx.y == 0 ? SA : SB;
  const int nb = S.nb, nb2 = nb * nb, n = S.ns * nb, col = blockIdx.x, e = threadIdx.x;
  if (col >= n) return;
  const int q = e / nb, c = e - q * nb;
  if (e < n) x[0][e] = cmk(e == col ? 1.0 : 0.0, 0.0);
  __syncthreads();
  int cur = 0;
  const int levels = sep_levels(S.ns);
  for (int l = 0; l < levels; ++l) {
    const int s = 1 << l;
    if (e < n) {
      const cplx* f = S.sfac + ((size_t)l * S.ns + q) * 2 * nb2 + c * nb;
      cplx v = x[cur][e];
      for (int t = 0; t < nb; ++t) {
        if (q - s >= 0) v = cfms(f[t], x[cur][(q - s) * nb + t], v);
        if (q + s < S.ns) v = cfms(f[nb2 + t], x[cur][(q + s) * nb + t], v);
      }
      x[cur ^ 1][e] = v;
    }
    __syncthreads();
    cur ^= 1;
  }
  if (e < n) {
    const cplx* f = S.sfac + ((size_t)levels * S.ns * 2 + q) * nb2 + c * nb;
    cplx v = cmk(0.0, 0.0);
    for (int t = 0; t < nb; ++t) v = cfma(f[t], x[cur][q * nb + t], v);
    S.sinv[(size_t)e * n + col] = v;
  }
}

}  // namespace

cudaError_t launch_setup_axis(const AxisSetup& a, cudaStream_t st) {
  int m = a.n - 1;
  k_setup_axis<<<(m + 127) / 128, 128, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_setup_diag(int mx, int my, int stride, int fine_mx, const cplx* dx, const cplx* dy,
                              const cplx* v1, const cplx* v2, const cplx* v12, double E, double omega,
                              cplx* D, cplx* Dinv, int* status, cudaStream_t st) {
  k_setup_diag<<<dim3((mx + 31) / 32, (my + 7) / 8), dim3(32, 8), 0, st>>>(mx, my, stride, fine_mx, dx, dy, v1, v2,
                                                                           v12, E, omega, D, Dinv, status);
  return cudaGetLastError();
}

cudaError_t launch_compare(int n, const cplx* a, const cplx* b, int* flag, cudaStream_t st) {
  k_compare<<<(n + 255) / 256, 256, 0, st>>>(n, a, b, flag);
  return cudaGetLastError();
}

cudaError_t launch_box_real_check(const StencilView& s, int* flag, cudaStream_t st) {
  if (s.cx.u <= 0 || s.cy.u <= 0) return cudaSuccess;
  k_box_real_check<<<dim3((s.cx.u + 31) / 32, (s.cy.u + 7) / 8), dim3(32, 8), 0, st>>>(s.mx, s.cx.u, s.cy.u, s.D,
                                                                                        flag);
  return cudaGetLastError();
}

size_t coarse_inverse_scratch(int nc) { return (size_t)nc * 2 * nc + nc; }

cudaError_t launch_coarse_inverse(const StencilView& s, cplx* aug, cplx* Ainv, int* status, cudaStream_t st) {
  const int nc = s.mx * s.my;
  cplx* fac = aug + (size_t)nc * 2 * nc;
  const long long total = 2LL * nc * nc;
  const int grid = (int)std::min<long long>((total + 255) / 256, 8LL * mgc_sm_count());
  k_gj_assemble<<<grid, 256, 0, st>>>(s, aug);
  cudaError_t e = cudaGetLastError();
  for (int k = 0; k < nc && e == cudaSuccess; ++k) {
    k_gj_pivot<<<1, 1024, 0, st>>>(nc, aug, fac, k, status);
    const long long work = (long long)nc * (2LL * nc - k - 1);
    const int g = (int)std::max<long long>(1, std::min<long long>((work + 255) / 256, 8LL * mgc_sm_count()));
    k_gj_eliminate<<<g, 256, 0, st>>>(nc, aug, fac, k, status);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) return e;
  k_gj_extract<<<grid, 256, 0, st>>>(nc, aug, Ainv);
  return cudaGetLastError();
}

size_t bound_states_scratch(int m, int nb) {
  // per state the workspace that does not fit in shared memory; at least the 2 m entries of the
  // QR fallback
  const size_t fac = (states_bytes(m) + sizeof(cplx) - 1) / sizeof(cplx) * sizeof(cplx) * nb;
  return std::max(fac, sizeof(cplx) * 2 * (size_t)m);
}

cudaError_t launch_bound_states(int m, const cplx* west, const cplx* east, const cplx* v, const cplx* w, int nb,
                                cplx* lam, cplx* phi, cplx* scratch, int* status,
                                cudaStream_t st, const cplx* eig) {
  const int in_smem = states_bytes(m) <= BS_SMEM;
  const size_t smem = in_smem ? states_bytes(m) : 0;
  // one constant limit, so that setups on several host threads may repeat the call
  cudaError_t e = cudaFuncSetAttribute(k_bound_states, cudaFuncAttributeMaxDynamicSharedMemorySize, BS_SMEM);
  if (e != cudaSuccess) return e;
  k_bound_states<<<nb, BS_THREADS, smem, st>>>(m, west, east, v, w, lam, phi, scratch, in_smem, status, eig);
  k_states_distinct<<<1, MGC_MAX_NB * MGC_MAX_NB, 0, st>>>(nb, lam, status);
  return cudaGetLastError();
}

cudaError_t launch_qr_spectrum(int m, const cplx* west, const cplx* east, const cplx* diag, const cplx* v,
                               cplx* scratch, cplx* out, int* status, cudaStream_t st) {
  k_qr_spectrum<<<1, 32, 0, st>>>(m, west, east, diag, v, scratch, out, status);
  return cudaGetLastError();
}

cudaError_t launch_weight_states(int m, int nb, const cplx* w, const cplx* phi, cplx* wphi, cudaStream_t st) {
  k_weight_states<<<(m * nb + 255) / 256, 256, 0, st>>>(m, nb, w, phi, wphi);
  return cudaGetLastError();
}

cudaError_t launch_channel_potentials(int mx, int my, int nb, const cplx* wphi, const cplx* phi,
                                      const cplx* wvphi, const cplx* vphi, const cplx* v12,
                                      cplx* VA, cplx* VB, cudaStream_t st) {
  const int npairs = nb * (nb + 1) / 2;
  // V^A_ab(y_j) = sum_i w_i phi_a(i) phi_b(i) V12(j, i)
  k_channel_potentials<<<dim3(my, npairs), 256, 0, st>>>(my, mx, nb, mx, 1, wphi, phi, v12, VA);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // V^B_ab(x_i) = sum_j w_j vphi_a(j) vphi_b(j) V12(j, i)
  k_channel_potentials<<<dim3(mx, npairs), 256, 0, st>>>(mx, my, nb, 1, mx, wvphi, vphi, v12, VB);
  return cudaGetLastError();
}

size_t channel_separator_entries(int ns, int nb) { return ((size_t)sep_levels(ns) * 2 + 1) * ns * nb * nb; }

int channel_factor_launches(const CRSystem& A, const CRSystem& B) {
  return 2 + std::max(A.p + sep_levels(A.ns), B.p + sep_levels(B.ns));   // the start, the levels, the separators
}

size_t channel_factor_scratch(int m, int nb) { return (size_t)8 * m * nb * nb; }

cudaError_t launch_channel_factor(const CRSystem& A, const CRSystem& B, const ChannelCoef& ca, const ChannelCoef& cb,
                                      double E, cplx* scratch, int* status, cudaStream_t st) {
  const int nb = A.nb, mm = std::max(A.m, B.m);
  const int levels = channel_factor_launches(A, B) - 2;
  cplx* scrB = scratch + channel_factor_scratch(A.m, nb);
  const ChannelSetup a{A, ca.diag, ca.v, ca.lam, ca.Vc, ca.sub, ca.sup, scratch};
  const ChannelSetup b{B, cb.diag, cb.v, cb.lam, cb.Vc, cb.sub, cb.sup, scrB};
  const dim3 grid((mm + CF_WARPS - 1) / CF_WARPS, 2);
  const size_t smem = (size_t)CF_WARPS * 12 * nb * nb * sizeof(cplx);
  for (int l = -1; l < levels; ++l) k_channel_factor<<<grid, 32 * CF_WARPS, smem, st>>>(a, b, E, l, status);
  k_separator_inverse<<<dim3(CR_CLUSTER * nb, 2), CR_CLUSTER * nb, 0, st>>>(A, B);
  return cudaGetLastError();
}
