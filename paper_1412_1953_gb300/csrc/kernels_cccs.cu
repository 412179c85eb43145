// Coupled Channel Correction Step kernels (Sec. 4 of Cools & Vanroose).
//
//   residual r = f - (H - E) u                                   (Sec. 4.3)
//   P^x_i(y) = sum_x w phi_i r,  P^y_j(x) = sum_y w vphi_j r      (projections, Sec. 4.1)
//   c_ij = sum_y w vphi_j P^x_i = a_ji + b_ij                     (Eq. (27))
//   a_ji = c_ij (j <= i), b_ij = c_ij (j > i)                     (Eqs. (25)-(26))
//   r^A_i = P^x_i - sum_{l>i} c_il vphi_l,  r^B_j = P^y_j - sum_{m>=j} c_mj phi_m
//   coupled-channel solves for e^A, e^B                           (Eqs. (28)-(29))
//   u += sum_m phi_m(x) e^A_m(y) + sum_l e^B_l(x) vphi_l(y)       (Eq. (30))
//
// The projections are fused into the residual pass and reduced deterministically:
// per 32 x 32 tile, sums along x and along y through a shared-memory tile give
// per-tile partials, which a second kernel sums in a fixed order; the channel solves form
// the coefficients and right-hand sides from the sums as they start.
#include <cooperative_groups.h>

#include <mutex>

#include "fixed.cuh"

namespace cg = cooperative_groups;

namespace {

constexpr int TX = 32;        // tile width (one warp per row)
constexpr int WY = 8;         // warps per block; a tile has SY rows per warp, SY = 1, 2 or 4

template <class C>
__device__ __forceinline__ C ldz(const C* __restrict__ a, int p, bool ok) {
  return ok ? __ldg(a + p) : CT<C>::make(0.0, 0.0);
}

template <int KX, int KY, int IR, int DG, class C>
__device__ __forceinline__ C residual_at(const StencilViewT<C>& s, const C* __restrict__ u, const C* __restrict__ f,
                                         int i, int j) {
  const int p = j * s.mx + i;
  return residual_vals<KX, KY, IR, DG>(s, i, j, p, __ldg(u + p), ldz(u, p - 1, i > 0), ldz(u, p + 1, i + 1 < s.mx),
                                       ldz(u, p - s.mx, j > 0), ldz(u, p + s.mx, j + 1 < s.my), __ldg(f + p));
}

// One tile of 32 x 8 SY nodes per block: each thread computes the residual at SY nodes into a
// padded shared tile; then, with the tile transposed through shared memory, one thread
// per (row, state) sums P^x over the tile's 32 columns and one thread per (column,
// state) sums P^y over its rows, without shuffle reductions.
template <int NB, int SY, class C>
__global__ void __launch_bounds__(TX * WY) k_residual_project(StencilViewT<C> s, CCViewT<C> c, const C* __restrict__ u,
                                                              const C* __restrict__ f) {
  mgc_pdl_enter();
  constexpr int TY = SY * WY;
  __shared__ C R[TY][TX + 1];
  const int lane = threadIdx.x;
  const int wy = threadIdx.y;
  const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY;
  const int i = i0 + lane;
  dispatch_kinds(s, i0, min(i0 + TX, s.mx), j0, min(j0 + TY, s.my), [&](auto kx, auto ky, auto ir, auto dg) {
    for (int q = 0; q < SY; ++q) {
      const int row = q * WY + wy;
      const int j = j0 + row;
      R[row][lane] = (i < s.mx && j < s.my)
                         ? residual_at<decltype(kx)::value, decltype(ky)::value, decltype(ir)::value,
                                       decltype(dg)::value>(s, u, f, i, j)
                         : CT<C>::make(0.0, 0.0);
    }
  });
  __syncthreads();
  const int t = wy * TX + lane;
  for (int w = t; w < (TX + TY) * NB; w += TX * WY) {
    if (w < TY * NB) {
      // P^x partial: row `row`, state m, over the tile's columns
      const int m = w / TY, row = w % TY;
      const int ncol = min(TX, s.mx - i0);
      const C* wp = c.wphi + (size_t)m * s.mx + i0;
      C acc = CT<C>::make(0.0, 0.0);
      for (int cc = 0; cc < ncol; ++cc) acc = cfma(__ldg(wp + cc), R[row][cc], acc);
      if (j0 + row < s.my) c.Px_part[((size_t)blockIdx.x * NB + m) * s.my + j0 + row] = acc;
    } else {
      // P^y partial: column `col`, state l, over the tile's rows
      const int w2 = w - TY * NB;
      const int l = w2 / TX, col = w2 % TX;
      const int nrow = min(TY, s.my - j0);
      const C* wv = c.wvphi + (size_t)l * s.my + j0;
      C acc = CT<C>::make(0.0, 0.0);
      for (int rr = 0; rr < nrow; ++rr) acc = cfma(__ldg(wv + rr), R[rr][col], acc);
      if (i0 + col < s.mx) c.Py_part[((size_t)blockIdx.y * NB + l) * s.mx + i0 + col] = acc;
    }
  }
}

// The same in complex128 with the projections on the integer pipes (fixed.cuh): the tile's
// residuals share one exponent, and so do each state's weighted values over the tile's columns
// (rows).  A residual's 2 n_b complex products then cost 24 n_b integer multiply-adds, 96 n_b
// cycles of a quarter of an SM, against 8 n_b FP64 instructions, 512 n_b cycles.  A tile with a row's
// (column's) projection whose products all lie below 2^-FX_NEAR of the tile's largest takes the FP64
// instructions: 3 to 7 % of the tiles of 32 rows in a solve at 512^2, up to 19 % at 256^2.  1023^2,
// n_b = 3, cold L2: 76.6 us with FP64 instructions, 41.8 us with integer projections (48 in a solve); 127^2: 19.2
// us in tiles of 32 rows (16 blocks), 7.4 us in tiles of 8.
template <int NB, int SY>
__global__ void __launch_bounds__(TX * WY) k_residual_project_fx(StencilView s, CCView c, const cplx* __restrict__ u,
                                                                const cplx* __restrict__ f) {
  constexpr int TY = SY * WY;
  __shared__ int4 R[TY][TX + 1];                         // limbs, or the values themselves
  __shared__ int4 wl[NB][TX], wr[NB][TY];
  __shared__ int xl[NB][TX], xr[NB][TY];                 // exponents of the weighted values
  __shared__ int ewl[NB], ewr[NB], eR, bad;
  __shared__ int pmax[NB][TX];                           // largest exponent of a column's products
  const int lane = threadIdx.x, wy = threadIdx.y, t = wy * TX + lane;
  const int i0 = blockIdx.x * TX, j0 = blockIdx.y * TY, i = i0 + lane;
  if (t == 0) eR = bad = 0;
  if (t < NB * TX) pmax[t / TX][t % TX] = 0;
  __syncthreads();
  for (int p = wy; p < 2 * NB; p += WY) {                // a warp converts one state's values of the tile
    const int m = p >> 1, n = p & 1 ? TY : TX, k = (p & 1 ? j0 : i0) + lane, len = p & 1 ? s.my : s.mx;
    const cplx w = lane < n && k < len ? __ldg((p & 1 ? c.wvphi : c.wphi) + (size_t)m * len + k) : cmk(0.0, 0.0);
    const int e = fx_exp(w), ew = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
    if (lane < n) {
      (p & 1 ? wr[m] : wl[m])[lane] = fx_limbs(w, ew, lane & 1);
      (p & 1 ? xr[m] : xl[m])[lane] = e;
    }
    if (lane == 0) {
      (p & 1 ? ewr : ewl)[m] = ew;
      if (!fx_ok(ew)) bad = 1;
    }
  }
  mgc_pdl_enter();                                       // the states were written at setup
  cplx r[SY];
  dispatch_kinds(s, i0, min(i0 + TX, s.mx), j0, min(j0 + TY, s.my), [&](auto kx, auto ky, auto ir, auto dg) {
#pragma unroll
    for (int q = 0; q < SY; ++q) {
      const int j = j0 + q * WY + wy;
      r[q] = (i < s.mx && j < s.my)
                 ? residual_at<decltype(kx)::value, decltype(ky)::value, decltype(ir)::value, decltype(dg)::value>(
                       s, u, f, i, j)
                 : cmk(0.0, 0.0);
    }
  });
  // the exponent of the residuals, and how far the largest products of any row (any column, by way of
  // pmax) stay below the largest of its state and the tile
  int e = 0, far = 0;
  __syncthreads();                                       // xl, xr, pmax
#pragma unroll
  for (int q = 0; q < SY; ++q) {
    const int eq = fx_exp(r[q]);
    e = max(e, eq);
    if (__any_sync(0xffffffffu, eq != 0)) {
#pragma unroll
      for (int m = 0; m < NB; ++m) {
        const int k = (int)__reduce_max_sync(0xffffffffu, (unsigned)(eq ? eq + xl[m][lane] : 0));
        far = max(far, ewl[m] + 4096 - k);
      }
    }
  }
#pragma unroll
  for (int m = 0; m < NB; ++m) {
    int k = 0;
#pragma unroll
    for (int q = 0; q < SY; ++q) {
      const int eq = fx_exp(r[q]);
      if (eq) k = max(k, eq + xr[m][q * WY + wy]);
    }
    atomicMax(&pmax[m][lane], k);
  }
  e = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
  if (lane == 0) atomicMax(&eR, e);
  __syncthreads();
  const int E = eR;
  if (t < NB * TX) {
    const int k = pmax[t / TX][t % TX];
    if (k) far = max(far, ewr[t / TX] + 4096 - k);
  }
  const bool ok = !__syncthreads_or(!fx_ok(E) || bad || far > 4096 - E + FX_NEAR);
#pragma unroll
  for (int q = 0; q < SY; ++q) {
    int4 v;
    if (ok) v = fx_limbs(r[q], E, (lane + q * WY + wy) & 1);
    else v = make_int4(__double2loint(r[q].x), __double2hiint(r[q].x), __double2loint(r[q].y), __double2hiint(r[q].y));
    R[q * WY + wy][lane] = v;
  }
  __syncthreads();
  for (int w = t; w < (TX + TY) * NB; w += TX * WY) {
    const bool px = w < TY * NB;                         // P^x: a row's columns; P^y: a column's rows
    const int w2 = px ? w : w - TY * NB, m = px ? w2 / TY : w2 / TX, at = px ? w2 % TY : w2 % TX;
    const int n = px ? TX : TY;
    cplx acc = cmk(0.0, 0.0);
    if (ok) {
      const int4* x = px ? &R[at][0] : &R[0][at];
      const int4* y = px ? wl[m] : wr[m];
      const int stride = px ? 1 : TX + 1;
      FxSum re{0, 0}, im{0, 0};
      for (int k0 = 0; k0 < n; k0 += FX_TERMS) {
#pragma unroll
        for (int k = 0; k < FX_TERMS; ++k) fx_cmac(re, im, y[k0 + k], x[(k0 + k) * stride]);
        fx_carry(re);
        fx_carry(im);
      }
      const int E2 = E + (px ? ewl[m] : ewr[m]);
      acc = cmk(fx_flush(re, E2, 0.0), fx_flush(im, E2, 0.0));
    } else {
      const int cnt = px ? min(TX, s.mx - i0) : min(TY, s.my - j0);
      const cplx* y = px ? c.wphi + (size_t)m * s.mx + i0 : c.wvphi + (size_t)m * s.my + j0;
      for (int k = 0; k < cnt; ++k) {
        const int4 v = px ? R[at][k] : R[k][at];
        acc = cfma(__ldg(y + k), cmk(__hiloint2double(v.y, v.x), __hiloint2double(v.w, v.z)), acc);
      }
    }
    if (px && j0 + at < s.my) c.Px_part[((size_t)blockIdx.x * NB + m) * s.my + j0 + at] = acc;
    if (!px && i0 + at < s.mx) c.Py_part[((size_t)blockIdx.y * NB + m) * s.mx + i0 + at] = acc;
  }
}

// Sum the per-tile partials (in FP64 for either partial type): eight lanes per output
// each sum a strided subset of tiles, then a fixed shuffle tree adds the eight.
template <class C>
__global__ void __launch_bounds__(256) k_reduce_partials(int nb, int mx, int my, int ntx, int nty,
                                                         const C* __restrict__ Px_part,
                                                         const C* __restrict__ Py_part,
                                                         cplx* __restrict__ Px, cplx* __restrict__ Py) {
  mgc_pdl_enter();
  const int g = blockIdx.x * 256 + threadIdx.x;
  const int t = g >> 3, sub = g & 7;
  const int nx_tot = nb * my, ny_tot = nb * mx;
  cplx acc = cmk(0.0, 0.0);
  if (t < nx_tot) {
    for (int k = sub; k < ntx; k += 8) acc = cadd(acc, to_c128(Px_part[(size_t)k * nx_tot + t]));
  } else if (t < nx_tot + ny_tot) {
    const int q = t - nx_tot;
    for (int k = sub; k < nty; k += 8) acc = cadd(acc, to_c128(Py_part[(size_t)k * ny_tot + q]));
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    acc.x += __shfl_down_sync(0xffffffffu, acc.x, o, 8);
    acc.y += __shfl_down_sync(0xffffffffu, acc.y, o, 8);
  }
  if (sub == 0) {
    if (t < nx_tot) Px[t] = acc;
    else if (t < nx_tot + ny_tot) Py[t - nx_tot] = acc;
  }
}

// Coupled-channel solves (Eqs. (28)-(29)) by cyclic reduction with setup-time factors: each
// system is solved by one thread-block cluster of CR_CLUSTER CTAs (cluster 0: channel A along y,
// cluster 1: channel B along x).  CTA `rank` owns the R = 2^p block rows [rank R, rank R + R) in
// its shared memory.  Level l < p (stride s = 2^l) eliminates every other remaining row,
// r_k -= alpha_k r_{k-s} + gamma_k r_{k+s} for the rows with k + 1 a multiple of 2s, until each
// CTA is left with its last row, the separator.  Only a separator's gamma term reaches into the
// next CTA, and nobody reads a separator meanwhile, so the next CTA sums those terms and the
// levels need block barriers only.  The separators (at most 16) are solved by the dense inverse
// of their system, every CTA gathering all their right-hand sides after one cluster barrier and
// forming the two it borders on; the eliminated rows follow in reverse order, x_k = B_k^{-1} r_k
// - alpha_k x_{k-s} - gamma_k x_{k+s}, again within the CTA.
// What bounds it is the latency of ~2 p small steps: a warp-wide FP64 instruction occupies its
// quarter of an SM for 64 cycles however few lanes need it, so LP lanes share the products of an
// item (a row's component), and the factors are copied to shared memory while the preceding
// kernel drains (large systems, and batches, read them from L2: cr_pack_in_smem).  Against
// parallel cyclic reduction over the cluster (every row updated at each of log2 m levels, a cluster barrier between them) with the
// coupling coefficients in a kernel of their own: 26.0 against 28.0 + 6.7 us for 1023 rows and
// n_b = 3, 16.2 against 18.1 + 4.1 us for 127 rows (cold L2); for 2047 rows and n_b = 6, where
// that took 11 m row updates, a step of the mixed-precision solve is 73 us shorter (50.3 to
// 44.6 ms a solve of 78 steps).
constexpr int CR_THREADS = 256;

__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void copy_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Sum over the LP lanes of an item, to all of them.
template <int LP>
__device__ __forceinline__ cplx item_sum(cplx v) {
#pragma unroll
  for (int o = 1; o < LP; o *= 2) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
  }
  return v;
}

// -(fa xl + fg xh) (+ fb r) of one component, its NB-term rows shared by LP lanes; a null x drops
// its term.
template <int NB, int LP, int NBLK>
__device__ __forceinline__ cplx item_dot(const cplx* fa, const cplx* fg, const cplx* fb, const cplx* xl,
                                         const cplx* xh, const cplx* r, int part) {
  cplx acc = cmk(0.0, 0.0);
#pragma unroll
  for (int t = 0; t < (NBLK * NB + LP - 1) / LP; ++t) {
    const int idx = t * LP + part, blk = idx / NB, q = idx - blk * NB;
    if (NBLK == 3 && blk == 2) {
      if (r) acc = cfma(fb[q], r[q], acc);
    } else if (blk < 2) {
      const cplx* f = blk == 0 ? fa : fg;
      const cplx* x = blk == 0 ? xl : xh;
      if (x) acc = cfms(f[q], x[q], acc);
    }
  }
  return item_sum<LP>(acc);
}

// What a CTA works on: rows [k0, k0 + R) of m, the rows in X, the previous separator's share in
// V, the separators' solutions xL (previous) and xO (own), null where there is none.
struct ChannelRows {
  int m, k0, R, p, rank;
  cplx *X, *V;
  const cplx *xL, *xO;
};

// Level l of the elimination.
template <int NB, int LP>
__device__ void channel_down(const ChannelRows& c, const cplx* F, int l) {
  constexpr int nb2 = NB * NB, PASS = CR_THREADS / LP;
  const int s = 1 << l, nk = c.R >> (l + 1), nit = (nk + (c.rank > 0 ? 1 : 0)) * NB, part = threadIdx.x % LP;
  const cplx* fw = F + (size_t)(c.R - (c.R >> l)) * 2 * nb2;
  const cplx* vf = F + (size_t)(c.R - 1) * 2 * nb2 + (size_t)l * nb2;
  for (int p0 = 0; p0 < nit; p0 += PASS) {
    const int it = p0 + threadIdx.x / LP, j = it / NB, comp = it - j * NB;
    const int i = j < nk ? 2 * s * (j + 1) - 1 : -1;
    const bool on = it < nit && c.k0 + i < c.m;
    const cplx* f = j < nk ? fw + (size_t)j * 2 * nb2 + comp * NB : vf - nb2 + comp * NB;
    const cplx* xl = on && j < nk ? c.X + (i - s) * NB : nullptr;
    const cplx* xh = on && i + s < c.R && c.k0 + i + s < c.m ? c.X + (i + s) * NB : nullptr;
    const cplx a = item_dot<NB, LP, 2>(f, f + nb2, nullptr, xl, xh, nullptr, part);
    if (on && part == 0) {
      cplx* t = j < nk ? c.X + i * NB + comp : c.V + comp;
      *t = cadd(*t, a);
    }
  }
}

// The rows eliminated at level l, from their neighbours' solutions.  A pass takes whole rows and
// writes after a barrier: an update in place reads all components of its row.
template <int NB, int LP>
__device__ void channel_up(const ChannelRows& c, const cplx* F, int l) {
  constexpr int nb2 = NB * NB, PASS = CR_THREADS / LP / NB * NB;
  const int s = 1 << l, nit = (c.R >> (l + 1)) * NB, part = threadIdx.x % LP, it0 = threadIdx.x / LP;
  const cplx* bk = F + ((size_t)(c.R - 1) * 2 + c.p) * nb2;
  for (int p0 = 0; p0 < nit; p0 += PASS) {
    const int it = p0 + it0, j = it / NB, comp = it - j * NB, i = s - 1 + 2 * s * j;
    const bool on = it0 < PASS && it < nit && c.k0 + i < c.m;
    const cplx* f = bk + (size_t)(on ? i : 0) * 3 * nb2 + comp * NB;
    const cplx* xl = !on ? nullptr : (j == 0 ? c.xL : c.X + (i - s) * NB);
    const cplx* xh = !on ? nullptr : (i + s == c.R - 1 ? c.xO : (c.k0 + i + s < c.m ? c.X + (i + s) * NB : nullptr));
    const cplx v = item_dot<NB, LP, 3>(f, f + nb2, f + 2 * nb2, xl, xh, on ? c.X + i * NB : nullptr, part);
    __syncthreads();
    if (on && part == 0) c.X[i * NB + comp] = v;
  }
}

template <int NB>
__global__ void __cluster_dims__(CR_CLUSTER, 1, 1) __launch_bounds__(CR_THREADS)
k_channel_solve(CRSystem SA, CRSystem SB) {
  extern __shared__ cplx cr_sh[];        // X [R][NB], then the factors when they fit
  constexpr int nb2 = NB * NB;
  __shared__ cplx cpart[nb2], csum[nb2], V[NB], xs[2][NB], rs[CR_CLUSTER * NB];
  cg::cluster_group cl = cg::this_cluster();
  const int rank = (int)cl.block_rank(), tid = threadIdx.x;
  const CRSystem S = blockIdx.x < CR_CLUSTER ? SA : SB;
  const int m = S.m, p = S.p, R = 1 << p, ns = S.ns, k0 = rank * R;
  cplx* const X = cr_sh;
  const size_t len = cr_pack_entries(R, p, NB);
  const cplx* F = S.pack + rank * len;
  const bool in_smem = cr_pack_in_smem(m, NB, S.shared_gpu);
  if (k0 < m) {
    // the factors were written at setup: fetch them ahead of the wait for the projections
    if (in_smem) {
      for (size_t e = tid; e < len; e += CR_THREADS) copy_async16(X + R * NB + e, F + e);
    } else if (tid == 0 && len > 0) {                // no factors where a CTA owns one row
      asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(F), "r"((unsigned)(len * sizeof(cplx)))
                   : "memory");
    }
  }
  mgc_pdl_enter();

  // the projections of this CTA's rows, and their share of the coupling coefficients
  // csum[a][l] = sum_k wst_l(k) P_a(k) that the conventions of Eqs. (25)-(26) use: c_al of Eq.
  // (27), l > a, in channel A, c_la, l >= a, in channel B
  for (int e = tid; e < R * NB; e += CR_THREADS) {
    const int comp = e >> p, k = k0 + (e & (R - 1));
    X[(k - k0) * NB + comp] = k < m ? S.P[comp * m + k] : cmk(0.0, 0.0);
  }
  if (tid < NB) V[tid] = cmk(0.0, 0.0);
  __syncthreads();
  {
    constexpr int CL = NB <= 3 ? 16 : NB <= 5 ? 8 : 4;   // lanes a coefficient: one warp a quarter
    const int l0 = S.chan == 0 ? 1 : 0, part = tid % CL;
    for (int q0 = 0; q0 < nb2; q0 += CR_THREADS / CL) {
      // coefficient q of the triangle, counted row by row
      int q = q0 + tid / CL, a = 0;
      while (a < NB && q >= NB - l0 - a) { q -= max(0, NB - l0 - a); ++a; }
      const int l = a + l0 + q;
      const bool on = a < NB && l < NB;
      cplx acc = cmk(0.0, 0.0);
      if (on)
        for (int k = k0 + part; k < min(k0 + R, m); k += CL)
          acc = cfma(__ldg(S.wst + l * m + k), X[(k - k0) * NB + a], acc);
      acc = item_sum<CL>(acc);
      if (on && part == 0) cpart[a * NB + l] = acc;
    }
  }
  cluster_arrive();
  cluster_wait();
  {
    const int q = tid / 4;
    cplx acc = cmk(0.0, 0.0);
    if (q < nb2 && q % NB >= q / NB + (S.chan == 0 ? 1 : 0)) {
#pragma unroll
      for (int c = 0; c < CR_CLUSTER / 4; ++c)
        acc = cadd(acc, *cl.map_shared_rank(cpart + q, (tid % 4) * (CR_CLUSTER / 4) + c));
    }
    acc = item_sum<4>(acc);
    if (q < nb2 && tid % 4 == 0) csum[q] = acc;
  }
  __syncthreads();
  for (int e = tid; e < R * NB; e += CR_THREADS) {
    const int comp = e >> p, k = k0 + (e & (R - 1));
    if (k >= m) continue;
    cplx v = X[(k - k0) * NB + comp];
    for (int l = comp + (S.chan == 0 ? 1 : 0); l < NB; ++l)
      v = cfms(csum[comp * NB + l], __ldg(S.basis + l * m + k), v);
    X[(k - k0) * NB + comp] = v;
  }
  if (in_smem) {
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    F = X + R * NB;
  }
  __syncthreads();

  const ChannelRows c{m, k0, R, p, rank, X, V, rank > 0 ? xs[0] : nullptr, rank < ns ? xs[1] : nullptr};
  for (int l = 0; l < p; ++l) {
    // four lanes an item while that still leaves one warp a quarter
    if (((R >> (l + 1)) + 1) * NB <= 32) channel_down<NB, 4>(c, F, l);
    else channel_down<NB, 2>(c, F, l);
    __syncthreads();
  }
  cluster_arrive();
  cluster_wait();
  for (int e = tid; e < ns * NB; e += CR_THREADS) {
    const int q = e / NB, comp = e - q * NB;
    cplx v = *cl.map_shared_rank(X + (R - 1) * NB + comp, q);
    if (q + 1 < CR_CLUSTER) v = cadd(v, *cl.map_shared_rank(V + comp, q + 1));
    rs[e] = v;
  }
  __syncthreads();
  cluster_arrive();                      // past this CTA's last remote read
  {
    constexpr int GL = 16;               // lanes an output
    for (int o0 = 0; o0 < 2 * NB; o0 += CR_THREADS / GL) {
      const int o = o0 + tid / GL, q = rank - 1 + o / NB, part = tid % GL;
      const bool on = o < 2 * NB && q >= 0 && q < ns;
      cplx acc = cmk(0.0, 0.0);
      if (on) {
        const cplx* g = S.sinv + (size_t)(q * NB + o % NB) * ns * NB;
        for (int e = part; e < ns * NB; e += GL) acc = cfma(__ldg(g + e), rs[e], acc);
      }
      acc = item_sum<GL>(acc);
      if (on && part == 0) xs[o / NB][o % NB] = acc;
    }
  }
  __syncthreads();
  for (int l = p - 1; l >= 0; --l) {
    if ((R >> (l + 1)) * NB <= 32) channel_up<NB, 4>(c, F, l);
    else channel_up<NB, 2>(c, F, l);
    __syncthreads();
  }
  for (int e = tid; e < R * NB; e += CR_THREADS) {
    const int comp = e >> p, i = e & (R - 1), k = k0 + i;
    if (k >= m) continue;
    const cplx v = i == R - 1 ? xs[1][comp] : X[i * NB + comp];
    S.e[comp * m + k] = v;
    if (S.e32) S.e32[comp * m + k] = make_float2((float)v.x, (float)v.y);
  }
  cluster_wait();
}

// u += sum_m phi_m(x) e^A_m(y) + sum_l e^B_l(x) vphi_l(y) (Eq. (30)), complex64.  A thread takes one
// column i and CC_ROWS consecutive rows: phi_m(i) and e^B_l(i) stay in registers
// across its rows (per node only the warp-uniform e^A_m(j), vphi_l(j) are loaded), and the
// loads of its values of u are issued together, so a warp has 8 x 256 bytes of u
// in flight (the pass is bound by how much of u is in flight).
constexpr int CC_ROWS = 8;

template <int NB, class C>
__global__ void __launch_bounds__(256) k_cccs_correct(int mx, int my, const C* __restrict__ phi,
                                                      const C* __restrict__ vphi, const C* __restrict__ eA,
                                                      const C* __restrict__ eB, C* __restrict__ u) {
  mgc_pdl_enter();
  const int i = blockIdx.x * 32 + threadIdx.x;
  const int j0 = (blockIdx.y * 8 + threadIdx.y) * CC_ROWS;
  if (i >= mx || j0 >= my) return;
  C a[NB], b[NB];
#pragma unroll
  for (int m = 0; m < NB; ++m) {
    a[m] = __ldg(phi + m * mx + i);
    b[m] = __ldg(eB + m * mx + i);
  }
  C v[CC_ROWS];
#pragma unroll
  for (int r = 0; r < CC_ROWS; ++r)
    if (j0 + r < my) v[r] = u[(j0 + r) * mx + i];
#pragma unroll
  for (int r = 0; r < CC_ROWS; ++r) {
    const int j = j0 + r;
    if (j >= my) break;
    C w = v[r];
#pragma unroll
    for (int m = 0; m < NB; ++m) w = cfma(a[m], __ldg(eA + m * my + j), w);
#pragma unroll
    for (int l = 0; l < NB; ++l) w = cfma(b[l], __ldg(vphi + l * my + j), w);
    u[j * mx + i] = w;
  }
}

// The same in complex128 on the integer pipes (fixed.cuh).  A block of 32 columns by 8 RT rows
// converts the values it needs of phi_m, e^B_l (columns) and e^A_m, vphi_l (rows), each with its
// exponent over the block, and aligns the 2 n_b products to the largest of their exponents by
// shifting e^A and vphi on conversion; a node then takes 24 n_b integer multiply-adds and four
// FP64 instructions (two conversions, two additions) against 8 n_b FP64 instructions.
// Limbs of 59 bits; a node whose products and value of u all lie below 2^-C_NEAR of the tile's largest
// product takes the FP64 multiply-adds, and so does a tile out of the integer range.
// 1023^2, n_b = 3: 45.0 us with FP64 multiply-adds, 22 us so; 127^2: 9.6 and, with RT = 1, 4.5 us
// (cold L2).
constexpr int C_NEAR = 6;

template <int NB, int RT>
__global__ void __launch_bounds__(256) k_cccs_correct_fx(int mx, int my, const cplx* __restrict__ phi,
                                                         const cplx* __restrict__ vphi, const cplx* __restrict__ eA,
                                                         const cplx* __restrict__ eB, cplx* __restrict__ u) {
  mgc_pdl_enter();
  constexpr int TYC = 8 * RT;
  __shared__ int4 col[2 * NB][32], row[2 * NB][TYC];     // [phi | e^B], [e^A | vphi]
  __shared__ int xc[2 * NB][32], xr[2 * NB][TYC];        // their exponents
  __shared__ int ec[2 * NB], er[2 * NB];
  const int lane = threadIdx.x, wy = threadIdx.y;
  const int i0 = blockIdx.x * 32, j0 = blockIdx.y * TYC, i = i0 + lane, jt = j0 + wy * RT;
  cplx v[RT];
#pragma unroll
  for (int r = 0; r < RT; ++r)
    if (i < mx && jt + r < my) v[r] = u[(size_t)(jt + r) * mx + i];
  auto value = [&](int p, int side) {                    // product p's factor at this lane's column (row)
    const int m = p < NB ? p : p - NB, k = (side ? j0 : i0) + lane, len = side ? my : mx;
    const cplx* a = p < NB ? (side ? eA : phi) : (side ? vphi : eB);
    return k < len && (!side || lane < TYC) ? __ldg(a + (size_t)m * len + k) : cmk(0.0, 0.0);
  };
  for (int p = wy; p < 4 * NB; p += 8) {
    const int ex = fx_exp(value(p >> 1, p & 1)), e = (int)__reduce_max_sync(0xffffffffu, (unsigned)ex);
    if (!(p & 1)) xc[p >> 1][lane] = ex;
    else if (lane < TYC) xr[p >> 1][lane] = ex;
    if (lane == 0) (p & 1 ? er : ec)[p >> 1] = e;
  }
  __syncthreads();
  int E2 = 0;
  bool ok = true;
#pragma unroll
  for (int p = 0; p < 2 * NB; ++p) {
    E2 = max(E2, ec[p] + er[p]);
    ok = ok && fx_ok(ec[p]) && fx_ok(er[p]);
  }
  // the rows of `which` with FP64 instructions, from the arrays
  const auto plain = [&](unsigned which) {
#pragma unroll 1
    for (; which; which &= which - 1) {
      const int j = jt + __ffs(which) - 1;
      if (j >= my) break;
      cplx w = u[(size_t)j * mx + i];
      for (int m = 0; m < NB; ++m) w = cfma(__ldg(phi + m * mx + i), __ldg(eA + m * my + j), w);
      for (int l = 0; l < NB; ++l) w = cfma(__ldg(eB + l * mx + i), __ldg(vphi + l * my + j), w);
      u[(size_t)j * mx + i] = w;
    }
  };
  if (!ok) {
    if (i < mx) plain((1u << RT) - 1);
    return;
  }
  for (int p = wy; p < 4 * NB; p += 8) {
    const int q = p >> 1;
    if (p & 1) {
      if (lane < TYC) row[q][lane] = fx_limbs<2>(value(q, 1), E2 - ec[q]);
    } else {
      col[q][lane] = fx_limbs<2>(value(q, 0), ec[q]);
    }
  }
  __syncthreads();
  if (i >= mx) return;
  int4 a[2 * NB];
#pragma unroll
  for (int p = 0; p < 2 * NB; ++p) a[p] = col[p][lane];
  unsigned low = 0;                                      // rows left to FP64 instructions
#pragma unroll
  for (int r = 0; r < RT; ++r) {
    if (jt + r >= my) break;
    int k = fx_exp(v[r]) + 1023;
    if (k < E2 - C_NEAR)
      for (int p = 0; p < 2 * NB; ++p) k = max(k, xc[p][lane] + xr[p][wy * RT + r]);
    FxSum re{0, 0}, im{0, 0};
#pragma unroll
    for (int p = 0; p < 2 * NB; ++p) {
      fx_cmac(re, im, a[p], row[p][wy * RT + r]);
      if (p + 1 == 2 * FX_TERMS_59 && p + 1 < 2 * NB) {  // the upper sum holds no more of 59 bits
        v[r].x = fx_flush<2>(re, E2, v[r].x);
        v[r].y = fx_flush<2>(im, E2, v[r].y);
      } else if ((p + 1) % FX_TERMS_59 == 0) {
        fx_carry<2>(re);
        fx_carry<2>(im);
      }
    }
    if (k < E2 - C_NEAR) low |= 1u << r;
    else u[(size_t)(jt + r) * mx + i] = cmk(fx_flush<2>(re, E2, v[r].x), fx_flush<2>(im, E2, v[r].y));
  }
  if (low) plain(low);
}

template <int NB, class C>
cudaError_t rp_launch(const StencilViewT<C>& s, const CCViewT<C>& c, const C* u, const C* f, cudaStream_t st) {
  auto go = [&](auto kern) {
    return mgc_launch(kern, dim3(cc_tiles_x(s.mx), cc_tiles_y(s.mx, s.my)), dim3(TX, WY), 0, st, s, c, u, f);
  };
  const int rows = cc_tile_rows(s.mx, s.my);
  if constexpr (sizeof(C) == sizeof(cplx))
    return rows == 1 ? go(k_residual_project_fx<NB, 1>)
                     : rows == 2 ? go(k_residual_project_fx<NB, 2>) : go(k_residual_project_fx<NB, 4>);
  else
    return rows == 1 ? go(k_residual_project<NB, 1, C>)
                     : rows == 2 ? go(k_residual_project<NB, 2, C>) : go(k_residual_project<NB, 4, C>);
}

template <int NB, class C>
cudaError_t corr_launch(const CCViewT<C>& c, C* u, cudaStream_t st) {
  if constexpr (sizeof(C) == sizeof(cplx)) {
    auto go = [&](auto kern, int rt) {
      return mgc_launch(kern, dim3((c.mx + 31) / 32, (c.my + 8 * rt - 1) / (8 * rt)), dim3(32, 8), 0, st, c.mx, c.my,
                        c.phi, c.vphi, c.eAc, c.eBc, u);
    };
    switch (cc_tile_rows(c.mx, c.my)) {
      case 1: return go(k_cccs_correct_fx<NB, 1>, 1);
      case 2: return go(k_cccs_correct_fx<NB, 2>, 2);
      default: return go(k_cccs_correct_fx<NB, 4>, 4);
    }
  } else {
    dim3 g((c.mx + 31) / 32, (c.my + 8 * CC_ROWS - 1) / (8 * CC_ROWS));
    return mgc_launch(k_cccs_correct<NB, C>, g, dim3(32, 8), 0, st, c.mx, c.my, c.phi, c.vphi, c.eAc, c.eBc, u);
  }
}

}  // namespace

int cc_tiles_x(int mx) { return (mx + TX - 1) / TX; }
// Rows per warp of a tile: four, but on grids that then have fewer than two blocks per SM (up to
// some 550 nodes an axis) two or one.
int cc_tile_rows(int mx, int my) {
  for (int sy = 4; sy > 1; sy /= 2)
    if ((long long)cc_tiles_x(mx) * ((my + WY * sy - 1) / (WY * sy)) >= 2LL * mgc_sm_count()) return sy;
  return 1;
}
int cc_tiles_y(int mx, int my) {
  const int ty = WY * cc_tile_rows(mx, my);
  return (my + ty - 1) / ty;
}

template <class C>
cudaError_t launch_residual_project(const StencilViewT<C>& s, const CCViewT<C>& c, const C* u, const C* f,
                                    cudaStream_t st) {
  switch (c.nb) {
    case 1: return rp_launch<1, C>(s, c, u, f, st);
    case 2: return rp_launch<2, C>(s, c, u, f, st);
    case 3: return rp_launch<3, C>(s, c, u, f, st);
    case 4: return rp_launch<4, C>(s, c, u, f, st);
    case 5: return rp_launch<5, C>(s, c, u, f, st);
    case 6: return rp_launch<6, C>(s, c, u, f, st);
    case 7: return rp_launch<7, C>(s, c, u, f, st);
    case 8: return rp_launch<8, C>(s, c, u, f, st);
  }
  return cudaErrorInvalidValue;
}

template <class C>
cudaError_t launch_reduce_projections(const CCViewT<C>& c, cudaStream_t st) {
  int tot = c.nb * (c.mx + c.my);
  return mgc_launch(k_reduce_partials<C>, dim3((8 * tot + 255) / 256), dim3(256), 0, st, c.nb, c.mx, c.my,
                    cc_tiles_x(c.mx), cc_tiles_y(c.mx, c.my), c.Px_part, c.Py_part, c.Px, c.Py);
}

namespace {
size_t channel_smem(int m, int nb, bool shared_gpu) {
  const int p = cr_log_rows(m);
  return sizeof(cplx) *
         (((size_t)nb << p) + (cr_pack_in_smem(m, nb, shared_gpu) ? cr_pack_entries(1 << p, p, nb) : 0));
}
}  // namespace

// Clusters of more than 8 CTAs must be allowed per kernel (once, before any launch or
// capture); called by setup.
// Raises (never lowers) the kernel's dynamic shared-memory limit to what the systems need,
// so every handle set up so far can still launch.
cudaError_t channel_solve_prepare(int nb, int mA, int mB) {
  static std::mutex mu;
  static int granted[MGC_MAX_NB + 1] = {0};
  if (nb < 1 || nb > MGC_MAX_NB) return cudaErrorInvalidValue;
  const size_t a = channel_smem(mA, nb, false), b = channel_smem(mB, nb, false);
  const int smem = (int)(a > b ? a : b);
  std::lock_guard<std::mutex> lock(mu);
  if (granted[nb] > 0 && smem <= granted[nb]) return cudaSuccess;
  const int want = smem > 48 * 1024 ? smem : 48 * 1024;
  cudaError_t e = cudaErrorInvalidValue;
  switch (nb) {
#define MGC_PREP(K)                                                                                      \
  case K:                                                                                                \
    e = cudaFuncSetAttribute(k_channel_solve<K>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);     \
    if (e == cudaSuccess)                                                                                \
      e = cudaFuncSetAttribute(k_channel_solve<K>, cudaFuncAttributeMaxDynamicSharedMemorySize, want);   \
    break;
    MGC_PREP(1) MGC_PREP(2) MGC_PREP(3) MGC_PREP(4) MGC_PREP(5) MGC_PREP(6) MGC_PREP(7) MGC_PREP(8)
#undef MGC_PREP
  }
  if (e == cudaSuccess) granted[nb] = want;
  return e;
}

cudaError_t launch_channel_solve(const CRSystem& A, const CRSystem& B, cudaStream_t st) {
  const size_t a = channel_smem(A.m, A.nb, A.shared_gpu), b = channel_smem(B.m, B.nb, B.shared_gpu);
  const size_t smem = a > b ? a : b;
  switch (A.nb) {
#define MGC_SOLVE(K) \
  case K: return mgc_launch(k_channel_solve<K>, dim3(2 * CR_CLUSTER), dim3(CR_THREADS), smem, st, A, B);
    MGC_SOLVE(1) MGC_SOLVE(2) MGC_SOLVE(3) MGC_SOLVE(4) MGC_SOLVE(5) MGC_SOLVE(6) MGC_SOLVE(7) MGC_SOLVE(8)
#undef MGC_SOLVE
    default: return cudaErrorInvalidValue;
  }
}

template <class C>
cudaError_t launch_cccs_correct(const CCViewT<C>& c, C* u, cudaStream_t st) {
  switch (c.nb) {
    case 1: return corr_launch<1, C>(c, u, st);
    case 2: return corr_launch<2, C>(c, u, st);
    case 3: return corr_launch<3, C>(c, u, st);
    case 4: return corr_launch<4, C>(c, u, st);
    case 5: return corr_launch<5, C>(c, u, st);
    case 6: return corr_launch<6, C>(c, u, st);
    case 7: return corr_launch<7, C>(c, u, st);
    case 8: return corr_launch<8, C>(c, u, st);
  }
  return cudaErrorInvalidValue;
}

#define MGC_INSTANTIATE(C)                                                                                  \
  template cudaError_t launch_residual_project<C>(const StencilViewT<C>&, const CCViewT<C>&, const C*,    \
                                                 const C*, cudaStream_t);                               \
  template cudaError_t launch_reduce_projections<C>(const CCViewT<C>&, cudaStream_t);                     \
  template cudaError_t launch_cccs_correct<C>(const CCViewT<C>&, C*, cudaStream_t);
MGC_INSTANTIATE(double2)
MGC_INSTANTIATE(float2)
#undef MGC_INSTANTIATE
