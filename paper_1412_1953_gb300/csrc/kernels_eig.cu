// Eigenvalues of the complex-symmetric tridiagonal of a 1D bound-state problem (Eq. (9)
// on the ECS grid) by the Ehrlich-Aberth simultaneous iteration with divide-and-conquer
// starting values, after D. A. Bini, L. Gemignani and F. Tisseur, "The Ehrlich-Aberth
// method for the nonsymmetric tridiagonal eigenvalue problem", SIAM J. Matrix Anal.
// Appl. 27 (2005).
//
// Level by level the matrix is cut into blocks of bs = 2, 4, 8, ... rows; the
// eigenvalues of the two halves of a block (the previous level's converged values) are
// the starting values for the block.  G lanes own one approximation z_i and per iteration
// evaluate
//   the Newton correction N_i = p(z_i)/p'(z_i) of the block's characteristic polynomial p:
//     the value beyond the block's last row of the solution of (H1 - z) u = 0 that starts as
//     (0, 1) at its first row.  With the quadrature weights w_k (w_k east_k = w_{k+1} west_{k+1},
//     diag_k = -(west_k + east_k)) and the flux F_k = w_k east_k (u_{k+1} - u_k) a row reads
//       F_k = F_{k-1} + w_k (z - v_k) u_k,   u_{k+1} = u_k + F_k / (w_k east_k),
//     without the cancellation of the three-term recurrence in d_k - z.  Each lane forms the
//     2 x 2 transfer matrix of (u, F) over its share of the rows and the matrix's derivative in
//     z, and the lanes multiply theirs in a shuffle tree, rescaled by powers of two.  (Products
//     of transfer matrices of (p_k, p_{k-1}) lose three digits at the low end of the spectrum,
//     where successive values hardly differ: some approximations then never settled.)
//   the Aberth step z_i <- z_i - N_i / (1 - N_i sum_{j != i} 1/(z_i - z_j)), the sum as the
//     logarithmic derivative of prod (z - z_j) over each lane's share of j (one division a
//     lane instead of one a term).
// An approximation whose step falls below the tolerance is frozen.
#include "common.cuh"

namespace {

constexpr int EIG_THREADS = 64;

// Per row: the diagonal d, and the flux form's 1/(w east), w v and w west (the starting flux of
// a block that begins at the row).
struct EigRows {
  cplx *d, *ic, *wv, *cs;
  const cplx* w;
};

__global__ void k_eig_init(int m, const cplx* __restrict__ west, const cplx* __restrict__ east,
                           const cplx* __restrict__ diag, const cplx* __restrict__ v, EigRows R,
                           cplx* __restrict__ z, unsigned long long* __restrict__ scale_bits) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= m) return;
  const cplx dk = cadd(diag[k], v[k]);
  const cplx ek = (k + 1 < m) ? cmul(east[k], west[k + 1]) : cmk(0.0, 0.0);   // squared off-diagonal
  R.d[k] = dk;
  R.ic[k] = cdiv(cmk(1.0, 0.0), cmul(R.w[k], east[k]));
  R.wv[k] = cmul(R.w[k], v[k]);
  R.cs[k] = cmul(R.w[k], west[k]);
  z[k] = dk;                                     // 1 x 1 blocks: their eigenvalues
  // a bound on the spectral radius (Gershgorin with |e_k| = sqrt|e2_k|) sets the absolute
  // tolerance; nonnegative doubles order like their bit patterns
  const double bound = cabs1(dk) + 2.0 * sqrt(cabs1(ek));
  atomicMax(scale_bits, (unsigned long long)__double_as_longlong(bound));
}

// The larger of m and the high word of |x| (a nonnegative double orders like its bits).
__device__ __forceinline__ int hi_max(int m, double x) { return max(m, __double2hiint(x) & 0x7fffffff); }
__device__ __forceinline__ int hi_max(int m, cplx z) { return hi_max(hi_max(m, z.x), z.y); }

// 2^-e of the exponent in the high word hm of a finite double (1 for zero and subnormals,
// and beyond 2^1000, where the caller's values are about to overflow anyway).
__device__ __forceinline__ double pow2_inverse(int hm) {
  const int e = (hm >> 20) - 1023;
  return hm < (1 << 20) || e > 1000 ? 1.0 : __hiloint2double((1023 - e) << 20, 0);
}
constexpr int HI_BIG = (1023 + 400) << 20, HI_SMALL = (1023 - 400) << 20;   // 2^400, 2^-400

__device__ __forceinline__ cplx shfl_down_c(cplx z, int o) {
  return cmk(__shfl_down_sync(0xffffffffu, z.x, o), __shfl_down_sync(0xffffffffu, z.y, o));
}

// Transfer matrix of a run of rows, (u, F) after = T (u, F) before, and dT/dz: rows (a, b) of u
// and (fa, fb) of F; q.. the derivatives.
struct Transfer {
  cplx a, b, fa, fb, qa, qb, qfa, qfb;
};

__device__ __forceinline__ void transfer_rescale(Transfer& t) {
  int hm = hi_max(hi_max(hi_max(hi_max(0, t.a), t.b), t.fa), t.fb);
  hm = hi_max(hi_max(hi_max(hi_max(hm, t.qa), t.qb), t.qfa), t.qfb);
  const double f = pow2_inverse(hm);
  t.a = cscal(f, t.a); t.b = cscal(f, t.b); t.fa = cscal(f, t.fa); t.fb = cscal(f, t.fb);
  t.qa = cscal(f, t.qa); t.qb = cscal(f, t.qb); t.qfa = cscal(f, t.qfa); t.qfb = cscal(f, t.qfb);
}

// One iteration of a level.  The FP64 pipe bounds it: 54 operations per pair (approximation,
// row), 44 in the recurrence (two starting vectors, value and derivative, so that the lanes'
// shares are independent; one thread walking all rows needs half but leaves 32 warps on the
// whole GPU) and 10 in the deflation sum; the shuffle tree adds 96 operations a step.
// All 212 launches of a 1023-row spectrum took 81 ms with one thread per approximation and a
// complex division per deflation term, 8.8 ms so (ncu, serialised).
template <int G>
__global__ void __launch_bounds__(EIG_THREADS) k_eig_aberth(int m, int bs, EigRows R,
                                                            const cplx* __restrict__ zin, cplx* __restrict__ zout,
                                                            int* __restrict__ done, int* __restrict__ active,
                                                            const unsigned long long* __restrict__ scale_bits) {
  const int i = (blockIdx.x * EIG_THREADS + threadIdx.x) / G;
  const int g = threadIdx.x % G;
  const bool in = i < m;
  const int ic = in ? i : m - 1;
  const int s0 = (ic / bs) * bs;
  const int s1 = min(s0 + bs, m);
  const cplx zi = zin[ic];
  // a block without its second half is the previous level's block: already converged
  const bool live = in && s1 - s0 > bs / 2 && !done[ic];
  const cplx one = cmk(1.0, 0.0), zero = cmk(0.0, 0.0);
  Transfer t{one, zero, zero, one, zero, zero, zero, zero};
  cplx A = zero;
  if (live) {
    const int c = (s1 - s0 + G - 1) / G;
    const int k1 = min(s0 + (g + 1) * c, s1);
    for (int k = s0 + g * c; k < k1; ++k) {
      const cplx wk = __ldg(R.w + k), ic = __ldg(R.ic + k);
      const cplx q = csub(cmul(wk, zi), __ldg(R.wv + k));
      t.qfa = cfma(q, t.qa, cfma(wk, t.a, t.qfa));
      t.qfb = cfma(q, t.qb, cfma(wk, t.b, t.qfb));
      t.fa = cfma(q, t.a, t.fa);
      t.fb = cfma(q, t.b, t.fb);
      t.a = cfma(ic, t.fa, t.a);
      t.b = cfma(ic, t.fb, t.b);
      t.qa = cfma(ic, t.qfa, t.qa);
      t.qb = cfma(ic, t.qfb, t.qb);
      const int hm = hi_max(hi_max(hi_max(hi_max(0, t.a), t.b), t.qa), t.qb);
      if (hm > HI_BIG || hm < HI_SMALL) transfer_rescale(t);
    }
    if (G > 1) transfer_rescale(t);
    // Aberth's implicit deflation by the other approximations of the block: sum 1/(z_i - z_j)
    // is P'/P of P = prod (z - z_j)
    cplx P = one, Q = zero;
    for (int j = s0 + g; j < s1; j += G) {
      const cplx dz = csub(zi, zin[j]);
      if (j == i || !(cabs1(dz) > 0.0)) continue;
      Q = cfma(Q, dz, P);
      P = cmul(P, dz);
      const int hm = hi_max(hi_max(0, P), Q);
      if (hm > HI_BIG || hm < HI_SMALL) {
        const double f = pow2_inverse(hm);
        P = cscal(f, P);
        Q = cscal(f, Q);
      }
    }
    A = cdiv(Q, P);
  }
#pragma unroll
  for (int o = 1; o < G; o *= 2) {
    // lanes g and g + o hold neighbouring runs of rows: T <- T(g + o) T(g)
    Transfer u;
    u.a = shfl_down_c(t.a, o); u.b = shfl_down_c(t.b, o); u.fa = shfl_down_c(t.fa, o); u.fb = shfl_down_c(t.fb, o);
    u.qa = shfl_down_c(t.qa, o); u.qb = shfl_down_c(t.qb, o);
    u.qfa = shfl_down_c(t.qfa, o); u.qfb = shfl_down_c(t.qfb, o);
    const cplx As = shfl_down_c(A, o);
    if (live) {
      Transfer r;
      r.a = cfma(u.a, t.a, cmul(u.b, t.fa));
      r.b = cfma(u.a, t.b, cmul(u.b, t.fb));
      r.fa = cfma(u.fa, t.a, cmul(u.fb, t.fa));
      r.fb = cfma(u.fa, t.b, cmul(u.fb, t.fb));
      r.qa = cfma(u.qa, t.a, cfma(u.qb, t.fa, cfma(u.a, t.qa, cmul(u.b, t.qfa))));
      r.qb = cfma(u.qa, t.b, cfma(u.qb, t.fb, cfma(u.a, t.qb, cmul(u.b, t.qfb))));
      r.qfa = cfma(u.qfa, t.a, cfma(u.qfb, t.fa, cfma(u.fa, t.qa, cmul(u.fb, t.qfa))));
      r.qfb = cfma(u.qfa, t.b, cfma(u.qfb, t.fb, cfma(u.fa, t.qb, cmul(u.fb, t.qfb))));
      t = r;
      transfer_rescale(t);
      A = cadd(A, As);
    }
  }
  if (g != 0 || !in) return;
  if (!live) {
    zout[i] = zi;
    return;
  }
  const double scale = __longlong_as_double((long long)*scale_bits);
  const cplx cs = R.cs[s0];
  const cplx p = cfma(cs, t.b, t.a), dp = cfma(cs, t.qb, t.qa);
  cplx step;
  if (cabs1(dp) == 0.0) {
    step = cmk(1e-8 * scale, 1e-8 * scale);                  // critical point of p: move off it
  } else {
    const cplx N = cdiv(p, dp);                              // Newton correction p/p'
    step = cdiv(N, csub(one, cmul(N, A)));
  }
  const cplx zn = csub(zi, step);
  const bool fin = isfinite(zn.x) && isfinite(zn.y);
  zout[i] = fin ? zn : zi;
  if (fin && cabs1(step) <= 4e-15 * cabs1(zi) + 1e-14 * scale) {
    done[i] = 1;
  } else {
    atomicAdd(active, fin ? 1 : (1 << 20));                  // non-finite steps count as failure
  }
}

// Trace check: sum z_i must equal sum d_k (the trace) to rounding, else flag.
__global__ void __launch_bounds__(256) k_eig_check(int m, const cplx* __restrict__ d, const cplx* __restrict__ z,
                                                   const unsigned long long* __restrict__ scale_bits,
                                                   int* __restrict__ bad) {
  __shared__ double sh[4][256];
  double a = 0, b = 0, c = 0, e = 0;
  for (int k = threadIdx.x; k < m; k += 256) {
    a += d[k].x; b += d[k].y; c += z[k].x; e += z[k].y;
  }
  sh[0][threadIdx.x] = a; sh[1][threadIdx.x] = b; sh[2][threadIdx.x] = c; sh[3][threadIdx.x] = e;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o)
      for (int q = 0; q < 4; ++q) sh[q][threadIdx.x] += sh[q][threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double scale = __longlong_as_double((long long)*scale_bits);
    const double err = fabs(sh[0][0] - sh[2][0]) + fabs(sh[1][0] - sh[3][0]);
    *bad = !(err <= 1e-10 * scale * sqrt((double)m) + 1e-300);
  }
}

// One iteration.  A warp's FP64 instruction occupies its quarter of an SM for 64 cycles, so the
// time is the instruction count of the busiest quarter: bs/G rows of 54 and log2 G tree steps
// of 96 a lane.  G = bs/4 balances the two, up to 32 lanes and to one warp per quarter.
cudaError_t launch_iteration(int m, int bs, const EigRows& R, const cplx* zin, cplx* zout, int* done, int* active,
                             const unsigned long long* scale_bits, cudaStream_t st) {
#define MGC_EIG(G)                                                                                        \
  k_eig_aberth<G><<<(unsigned)(((long long)m * G + EIG_THREADS - 1) / EIG_THREADS), EIG_THREADS, 0, st>>>( \
      m, bs, R, zin, zout, done, active, scale_bits)
  const long long cap = 4LL * mgc_sm_count() * 32 / m;
  const long long want = bs / 4 < cap ? bs / 4 : cap;
  if (want >= 32) MGC_EIG(32);
  else if (want >= 16) MGC_EIG(16);
  else if (want >= 8) MGC_EIG(8);
  else if (want >= 4) MGC_EIG(4);
  else if (want >= 2) MGC_EIG(2);
  else MGC_EIG(1);
#undef MGC_EIG
  return cudaGetLastError();
}

}  // namespace

size_t eig_scratch_entries(int m) {
  // four row arrays, two approximation buffers, then done flags, counters and the scale (as ints)
  const size_t ints = (size_t)m + 8;
  return (size_t)6 * m + (ints * sizeof(int) + sizeof(cplx) - 1) / sizeof(cplx) + 1;
}

cudaError_t eig_aberth(int m, const cplx* west, const cplx* east, const cplx* diag, const cplx* v, const cplx* w,
                       cplx* scratch, cplx* out, bool* ok, cudaStream_t st) {
  *ok = false;
  const EigRows R{scratch, scratch + m, scratch + 2 * m, scratch + 3 * m, w};
  cplx* za = scratch + 4 * m;
  cplx* zb = scratch + 5 * m;
  int* done = reinterpret_cast<int*>(scratch + 6 * m);
  int* active = done + m;
  int* bad = done + m + 1;
  unsigned long long* scale_bits = reinterpret_cast<unsigned long long*>(
      scratch + 6 * m + ((size_t)(m + 8) * sizeof(int) + sizeof(cplx) - 1) / sizeof(cplx));
  cudaError_t e = cudaMemsetAsync(scale_bits, 0, sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  k_eig_init<<<(m + 255) / 256, 256, 0, st>>>(m, west, east, diag, v, R, za, scale_bits);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  cplx* cur = za;
  cplx* nxt = zb;
  constexpr int kChunk = 4, kMaxIter = 240;
  for (int bs = 2; bs / 2 < m; bs *= 2) {
    if ((e = cudaMemsetAsync(done, 0, sizeof(int) * (size_t)m, st)) != cudaSuccess) return e;
    bool converged = false;
    for (int it = 0; it < kMaxIter && !converged; it += kChunk) {
      for (int c = 0; c < kChunk; ++c) {
        if ((e = cudaMemsetAsync(active, 0, sizeof(int), st)) != cudaSuccess) return e;
        if ((e = launch_iteration(m, bs, R, cur, nxt, done, active, scale_bits, st)) != cudaSuccess) return e;
        cplx* x = cur; cur = nxt; nxt = x;
      }
      int act = 0;
      if ((e = cudaMemcpyAsync(&act, active, sizeof(int), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
      if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
      if (act >= (1 << 20)) return cudaSuccess;                // non-finite: *ok stays false
      converged = act == 0;
    }
    if (!converged) return cudaSuccess;
  }
  k_eig_check<<<1, 256, 0, st>>>(m, R.d, cur, scale_bits, bad);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  int b = 1;
  if ((e = cudaMemcpyAsync(&b, bad, sizeof(int), cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
  if (b) return cudaSuccess;
  if ((e = cudaMemcpyAsync(out, cur, sizeof(cplx) * (size_t)m, cudaMemcpyDeviceToDevice, st)) != cudaSuccess)
    return e;
  *ok = true;
  return cudaSuccess;
}
