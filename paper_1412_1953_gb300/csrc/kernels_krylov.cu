// Kernels of the restarted GMRES(m) outer solver, right-preconditioned by one MG-CCCS
// iteration (Sec. 6: MG-CCCS as a Krylov preconditioner).  Arnoldi uses classical
// Gram-Schmidt (each pass: one fused multi-dot, one fused multi-axpy) with a second pass
// when a cancellation test asks for it (decided on the device);
// the Hessenberg least-squares problem is reduced by complex Givens rotations on the
// device, so the host only reads one residual estimate per step.
//
// Basis vectors are stored contiguously: V_i = V + i * ld.
#include "fixed.cuh"

namespace {

constexpr int NT = 256;

// Block sum of a complex value: warp sums in the element precision, the per-warp totals
// in FP64 by thread 0 (fixed order).  Complex64 data keeps the FP64 pipe out of the
// per-thread work.
template <int NTH, class C>
__device__ __forceinline__ cplx block_sum_c(C v, double (*sh)[NTH / 32]) {
  const int t = threadIdx.x;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v.x += __shfl_down_sync(0xffffffffu, v.x, o);
    v.y += __shfl_down_sync(0xffffffffu, v.y, o);
  }
  if ((t & 31) == 0) { sh[0][t >> 5] = (double)v.x; sh[1][t >> 5] = (double)v.y; }
  __syncthreads();
  cplx tot = cmk(0.0, 0.0);
  if (t == 0)
    for (int w = 0; w < NTH / 32; ++w) tot = cadd(tot, cmk(sh[0][w], sh[1][w]));
  return tot;
}

// partial[i][b] = sum over block b's points of conj(V_i) w   (grid: nblk x k).
// When `gate` is given and *gate == 0 the pass is skipped (partials set to zero).
// A vector V_i that is w itself gives |w|^2 (two FMAs per point; the block's branch).
// (Each thread accumulates in the element precision; the block sum is FP64.)
template <class C>
__global__ void __launch_bounds__(NT) k_multidot(long long n, const C* __restrict__ V, long long ld,
                                                 const C* __restrict__ w, cplx* __restrict__ partial,
                                                 const int* __restrict__ gate) {
  mgc_pdl_enter();
  __shared__ double sh[2][NT / 32];
  const int i = blockIdx.y;
  if (gate && *gate == 0) {
    if (threadIdx.x == 0) partial[(size_t)i * gridDim.x + blockIdx.x] = cmk(0.0, 0.0);
    return;
  }
  const C* v = V + (size_t)i * ld;
  C acc = CT<C>::make(0.0, 0.0);
  if (v == w) {
    for (long long p = blockIdx.x * (long long)NT + threadIdx.x; p < n; p += (long long)gridDim.x * NT) {
      C b = __ldg(w + p);
      acc.x = fma(b.x, b.x, fma(b.y, b.y, acc.x));
    }
  } else {
    for (long long p = blockIdx.x * (long long)NT + threadIdx.x; p < n; p += (long long)gridDim.x * NT) {
      C a = __ldg(v + p), b = __ldg(w + p);
      acc.x = fma(a.x, b.x, fma(a.y, b.y, acc.x));
      acc.y = fma(a.x, b.y, fma(-a.y, b.x, acc.y));
    }
  }
  cplx tot = block_sum_c<NT>(acc, sh);
  if (threadIdx.x == 0) partial[(size_t)i * gridDim.x + blockIdx.x] = tot;
}

// ---- complex128 Gram-Schmidt on the integer pipes (fixed.cuh).  With FP64 instructions the pair
// runs at the FP64 pipe's rate, a third of the HBM bandwidth.

// Asynchronous 16-byte copy to shared memory (_if: zeros when !ok), and the wait for all but the last
// N groups of them.  A lane reads back only what it copied, so no barrier is involved.
__device__ __forceinline__ void copy16(cplx* dst, const cplx* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy16_if(cplx* dst, const cplx* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(ok ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copy_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// The multi-dot: a block takes DG vectors, so that w is converted once for all of them, and a
// warp DU x 32 consecutive points at a time, the last 32 of them with FP64 instructions, which
// otherwise idle.  The exponents of w and of each vector are a warp's own and follow its chunks
// (within D_SLACK; a new one first rounds the sums held so far).  A chunk in which no product comes
// within 2^-FX_NEAR of the largest of both, so that its sum could be as small as what the conversions
// leave, is summed with FP64 instructions.  The sequence of chunks (w, then each
// vector, of one tile after another) is fetched DS - 1 chunks ahead.  About 90 instructions a
// product and the 16 warps that 128 registers allow bound it.  1023^2, 12 vectors (12 and 1
// of 16.7 MB read): 88.0 us with FP64 multiply-adds, 63 with 64-bit shifts of masked keys in the
// conversion, 58 before the FP64 share, 53.7 with it, 56.9 with conversions that leave no mean
// (fixed.cuh; ties alternate by lane: 4 us of a pair), 61 us with exponents that follow the chunks and
// the look for a near product, 3.3 TB/s.
constexpr int DG = 4, DU = 4, DS = 4, D_SLACK = 2;

__global__ void __launch_bounds__(NT, 2) k_multidot_fx(long long n, int k, const cplx* __restrict__ V, long long ld,
                                                       const cplx* __restrict__ w, cplx* __restrict__ partial,
                                                       const int* __restrict__ gate) {
  mgc_pdl_enter();
  extern __shared__ cplx gs_sh[];                      // [warp][DS][DU][32], then the block sums
  const int i0 = blockIdx.y * DG, nv = min(DG, k - i0), tid = threadIdx.x, lane = tid & 31;
  if (gate && *gate == 0) {
    if (tid < nv) partial[(size_t)(i0 + tid) * gridDim.x + blockIdx.x] = cmk(0.0, 0.0);
    return;
  }
  cplx* const ring = gs_sh + (size_t)(tid >> 5) * DS * DU * 32 + lane;
  const long long step = (long long)gridDim.x * NT * DU;
  long long p0 = (long long)blockIdx.x * NT * DU + (tid >> 5) * 32 * DU;   // the warp's tile
  // the next chunk to fetch: vector fi (0: w, i: vector i0 + i - 1) of the tile at fp
  const cplx* const Vg = V + (size_t)i0 * ld;
  const cplx* fv = w;
  long long fp = p0;
  int fi = 0, fs = 0;
  auto fetch = [&]() {
    if (fp < n) {
      const cplx* src = fv + fp + lane;
      if (fp + 32 * DU <= n) {
#pragma unroll
        for (int u = 0; u < DU; ++u) copy16(ring + (fs * DU + u) * 32, src + 32 * u);
      } else {
#pragma unroll
        for (int u = 0; u < DU; ++u) copy16_if(ring + (fs * DU + u) * 32, src + 32 * u, fp + lane + 32 * u < n);
      }
      fv = fi == 0 ? Vg : fv + ld;
      if (++fi > nv) {
        fi = 0;
        fv = w;
        fp += step;
      }
    }
    fs = (fs + 1) % DS;
    copy_commit();
  };
  int rs = 0;
  int ex[DU], ey[DU];                                  // exponents of the chunk taken last
  auto take = [&](cplx (&v)[DU]) {                     // the oldest chunk; returns its largest exponent
    copy_wait<DS - 2>();
    int e = 0;
#pragma unroll
    for (int u = 0; u < DU; ++u) {
      v[u] = ring[(rs * DU + u) * 32];
      ex[u] = fx_exp(v[u].x);
      ey[u] = fx_exp(v[u].y);
      e = max(max(e, ex[u]), ey[u]);
    }
    rs = (rs + 1) % DS;
    fetch();
    return (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
  };
  cplx sum[DG];
  FxSum re[DG], im[DG];
  int E[DG], Ew = 0;
#pragma unroll
  for (int i = 0; i < DG; ++i) {
    sum[i] = cmk(0.0, 0.0);
    re[i] = im[i] = FxSum{0, 0};
    E[i] = 0;
  }
  auto flush = [&](int i) {
    if (!fx_ok(Ew) || !fx_ok(E[i])) return;            // nothing was summed at these exponents
    sum[i].x = fx_flush<2>(re[i], Ew + E[i], sum[i].x);
    sum[i].y = fx_flush<2>(im[i], Ew + E[i], sum[i].y);
  };
#pragma unroll
  for (int c = 0; c < DS - 1; ++c) fetch();
  int held = 0;                                        // terms in the sums
  for (; p0 < n; p0 += step) {
    cplx v[DU];
    const int et = take(v);
    if (et > Ew || et < Ew - D_SLACK || held + DU - 1 > FX_TERMS_59) {
#pragma unroll
      for (int i = 0; i < DG; ++i) flush(i);
      held = 0;
      if (et > Ew || et < Ew - D_SLACK) Ew = et;
    }
    held += DU - 1;
    FxLimbs wx[DU - 1], wy[DU - 1];
    int ew[DU - 1];
    const cplx wl = v[DU - 1];
#pragma unroll
    for (int u = 0; u < DU - 1; ++u) {
      wx[u] = fx_limbs<2>(v[u].x, ex[u], Ew, lane & 1);
      wy[u] = fx_limbs<2>(v[u].y, ey[u], Ew, lane & 1);
      ew[u] = max(ex[u], ey[u]);
    }
#pragma unroll
    for (int i = 0; i < DG; ++i) {
      if (i >= nv) break;
      const int ei = take(v);
      if (ei > E[i] || ei < E[i] - D_SLACK) {
        flush(i);
        E[i] = ei;
      }
      int k = 0;
#pragma unroll
      for (int u = 0; u < DU - 1; ++u) k = max(k, max(ex[u], ey[u]) + ew[u]);
      if (__any_sync(0xffffffffu, k >= Ew + E[i] - FX_NEAR) && fx_ok(Ew) && fx_ok(E[i])) {
#pragma unroll
        for (int u = 0; u < DU - 1; ++u) {
          const FxLimbs ax = fx_limbs<2>(v[u].x, ex[u], E[i], lane & 1);
          const FxLimbs ay = fx_limbs<2>(v[u].y, ey[u], E[i], lane & 1);
          fx_mac(re[i], ax, wx[u]);
          fx_mac(re[i], ay, wy[u]);
          fx_mac(im[i], ax, wy[u]);
          fx_mac(im[i], fx_neg(ay), wx[u]);
        }
        const cplx a = v[DU - 1];
        sum[i].x = fma(a.x, wl.x, fma(a.y, wl.y, sum[i].x));
        sum[i].y = fma(a.x, wl.y, fma(-a.y, wl.x, sum[i].y));
      } else {
#pragma unroll
        for (int u = 0; u < DU; ++u) {
          const long long p = p0 + lane + 32 * u;
          const cplx b = p < n ? __ldg(w + p) : cmk(0.0, 0.0);
          sum[i].x = fma(v[u].x, b.x, fma(v[u].y, b.y, sum[i].x));
          sum[i].y = fma(v[u].x, b.y, fma(-v[u].y, b.x, sum[i].y));
        }
      }
    }
  }
  copy_wait<0>();
  __syncthreads();
  double (*sh)[NT] = reinterpret_cast<double (*)[NT]>(gs_sh);
#pragma unroll
  for (int i = 0; i < DG; ++i) {
    flush(i);
    sh[2 * i][tid] = sum[i].x;
    sh[2 * i + 1][tid] = sum[i].y;
  }
  __syncthreads();
  // warp q sums component q over the block's threads (fixed order)
  const int q = tid >> 5;
  static_assert(2 * DG == NT / 32, "one warp per component");
  double tot = sh[q][lane];
#pragma unroll
  for (int t = 1; t < NT / 32; ++t) tot += sh[q][lane + 32 * t];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tot += __shfl_down_sync(0xffffffffu, tot, o);
  if (lane == 0 && (q >> 1) < nv) {
    double* out = reinterpret_cast<double*>(partial + (size_t)(i0 + (q >> 1)) * gridDim.x + blockIdx.x);
    const bool self = Vg + (q >> 1) * ld == w;         // w itself: |w|^2, exactly real
    out[q & 1] = self && (q & 1) ? 0.0 : tot;
  }
}
constexpr int MULTIDOT_SMEM = NT * DS * DU * (int)sizeof(cplx);
static_assert(MULTIDOT_SMEM >= 2 * DG * NT * (int)sizeof(double), "the block sums reuse the ring");

// The update w += sgn sum_i coef[i] V_i.  The coefficients are converted once per block, each
// with its own exponent; a warp's sums over the vectors share the exponent of the largest product
// met so far (at first that of the largest coefficient and the first vector).  A warp takes
// UU x 32 points at a time and fetches the chunks (w, then each vector) ahead, as above.  Points whose
// own products and w all lie below 2^-U_NEAR of that largest product are done again with FP64
// instructions, from the arrays: 59 bits leave them fewer than a double has.
// 1023^2, 11 random vectors: 90.1 us with FP64 multiply-adds, 50 before the look for low points (UU = 4;
// 58 with UU = 2, which is the faster at 255^2: 7.6 against 11.4 us, few tiles a warp), 54 us now, 4.0 TB/s.
// In a solve, where w is near its largest term and both are small at the same points, a quarter of the
// tiles hold one, 81 against 59 us with cold L2.
constexpr int U_NEAR = 6;
constexpr int UF = 16;                                 // chunks in flight x points a lane

template <int UU>
__global__ void __launch_bounds__(NT, UU == 4 ? 2 : 3) k_multiaxpy_fx(long long n, int k, const cplx* __restrict__ V, long long ld,
                                                        const cplx* __restrict__ coef, double sgn,
                                                        cplx* __restrict__ w, double* __restrict__ norm_part,
                                                        const int* __restrict__ gate, const int* __restrict__ dk) {
  mgc_pdl_enter();
  constexpr int AS = UF / UU;
  extern __shared__ cplx gs_sh[];                      // [warp][AS][UU][32]
  __shared__ cplx sc[64];
  __shared__ int4 sl[64];                              // limbs of re and im
  __shared__ int se[64];
  __shared__ int smax;
  __shared__ double sh[NT / 32];
  if (gate && *gate == 0) return;
  if (dk) k = min(k, *dk);
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) smax = 0;
  __syncthreads();
  for (int i = tid; i < k; i += NT) {
    const cplx q = cscal(sgn, coef[i]);
    const int ex = fx_exp(q.x), ey = fx_exp(q.y), e = max(ex, ey);
    const FxLimbs x = fx_limbs<2>(q.x, ex, e), y = fx_limbs<2>(q.y, ey, e);
    sc[i] = q;
    sl[i] = make_int4(x.h, x.l, y.h, y.l);
    se[i] = e;
    atomicMax(&smax, e);
  }
  __syncthreads();
  cplx* const ring = gs_sh + (size_t)(tid >> 5) * AS * UU * 32 + lane;
  const long long step = (long long)gridDim.x * NT * UU;
  long long p0 = (long long)blockIdx.x * NT * UU + (tid >> 5) * 32 * UU;
  const cplx* fv = w;
  long long fp = p0;
  int fi = 0, fs = 0, rs = 0;
  auto fetch = [&]() {
    if (fp < n) {
      const cplx* src = fv + fp + lane;
      if (fp + 32 * UU <= n) {
#pragma unroll
        for (int u = 0; u < UU; ++u) copy16(ring + (fs * UU + u) * 32, src + 32 * u);
      } else {
#pragma unroll
        for (int u = 0; u < UU; ++u) copy16_if(ring + (fs * UU + u) * 32, src + 32 * u, fp + lane + 32 * u < n);
      }
      fv = fi == 0 ? V : fv + ld;
      if (++fi > k) {
        fi = 0;
        fv = w;
        fp += step;
      }
    }
    fs = (fs + 1) % AS;
    copy_commit();
  };
  auto take = [&](cplx (&v)[UU]) {
    copy_wait<AS - 2>();
#pragma unroll
    for (int u = 0; u < UU; ++u) v[u] = ring[(rs * UU + u) * 32];
    rs = (rs + 1) % AS;
    fetch();
  };
#pragma unroll
  for (int c = 0; c < AS - 1; ++c) fetch();
  double n2 = 0.0;
  for (; p0 < n; p0 += step) {
    cplx acc[UU];
    FxSum re[UU], im[UU];
    take(acc);
    int top[UU];                                       // exponent of a point's largest term
#pragma unroll
    for (int u = 0; u < UU; ++u) {
      re[u] = im[u] = FxSum{0, 0};
      top[u] = fx_exp(acc[u]) + 1023;
    }
    int E2 = 0, held = 0;
    auto flush = [&]() {
      if (held == 0) return;
#pragma unroll
      for (int u = 0; u < UU; ++u) {
        acc[u].x = fx_flush<2>(re[u], E2, acc[u].x);
        acc[u].y = fx_flush<2>(im[u], E2, acc[u].y);
      }
      held = 0;
    };
    for (int i = 0; i < k; ++i) {
      cplx v[UU];
      take(v);
      int ex[UU], ey[UU], e = 0;
#pragma unroll
      for (int u = 0; u < UU; ++u) {
        ex[u] = fx_exp(v[u].x);
        ey[u] = fx_exp(v[u].y);
        e = max(max(e, ex[u]), ey[u]);
      }
      const int ev = (int)__reduce_max_sync(0xffffffffu, (unsigned)e), ec = se[i];
      if (fx_ok(ev) && fx_ok(ec)) {
        if (ev + ec > E2 || held == FX_TERMS_59) {
          flush();
          // the first time: room for the largest coefficient
          E2 = max(E2, i == 0 && fx_ok(smax) ? ev + smax : ev + ec);
        }
        ++held;
        const int4 c = sl[i];
        const FxLimbs cx{c.x, c.y}, cy{c.z, c.w}, my = fx_neg(cy);
        const int E = E2 - ec;
#pragma unroll
        for (int u = 0; u < UU; ++u) {
          const FxLimbs x = fx_limbs<2>(v[u].x, ex[u], E), y = fx_limbs<2>(v[u].y, ey[u], E);
          top[u] = max(top[u], max(ex[u], ey[u]) + ec);
          fx_mac(re[u], x, cx);
          fx_mac(re[u], y, my);
          fx_mac(im[u], y, cx);
          fx_mac(im[u], x, cy);
        }
      } else {
#pragma unroll
        for (int u = 0; u < UU; ++u) acc[u] = cfma(sc[i], v[u], acc[u]);
      }
    }
    flush();
    unsigned low = 0;
#pragma unroll
    for (int u = 0; u < UU; ++u)
      if (p0 + lane + 32 * u < n && top[u] < E2 - U_NEAR) low |= 1u << u;
    if (low) {
#pragma unroll
      for (int u = 0; u < UU; ++u) {
        if (!(low >> u & 1)) continue;
        const long long p = p0 + lane + 32 * u;
        cplx a = w[p];
#pragma unroll 1
        for (int i = 0; i < k; ++i) a = cfma(sc[i], __ldg(V + i * ld + p), a);
        acc[u] = a;
      }
    }
#pragma unroll
    for (int u = 0; u < UU; ++u)
      if (p0 + lane + 32 * u < n) {
        w[p0 + lane + 32 * u] = acc[u];
        if (norm_part) n2 += cabs2(acc[u]);
      }
  }
  copy_wait<0>();
  if (norm_part) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n2 += __shfl_down_sync(0xffffffffu, n2, o);
    if (lane == 0) sh[tid >> 5] = n2;
    __syncthreads();
    if (tid == 0) {
      double tot = 0.0;
      for (int q = 0; q < NT / 32; ++q) tot += sh[q];
      norm_part[blockIdx.x] = tot;
    }
  }
}
constexpr int MULTIAXPY_SMEM = NT * UF * (int)sizeof(cplx);

// A double in units of 2^(E - 1138) for the block's largest exponent E: below 2^116, and cut below 2^-116 of
// the largest value only.
__device__ __forceinline__ __int128 fixed_128(double x, int E) {
  const int e = fx_exp(x), hi = __double2hiint(x);
  const unsigned long long m =
      (unsigned long long)(((unsigned)hi & 0xfffffu) | (e ? 0x100000u : 0u)) << 32 | (unsigned)__double2loint(x);
  const __int128 v = ((__int128)m << 63) >> min(E - e, 127);
  return hi < 0 ? -v : v;
}
__device__ __forceinline__ __int128 warp_sum_128(__int128 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long lo = __shfl_down_sync(0xffffffffu, (unsigned long long)v, o);
    const long long hi = __shfl_down_sync(0xffffffffu, (long long)(v >> 64), o);
    v += (__int128)hi << 64 | lo;
  }
  return v;
}

// out[i] = sum_b partial[i][b]; acc_into[i] += out[i] when given.  At most 2^10 partials (krylov_blocks), added exactly as
// 128-bit integers (FP64 additions out of the integer range): where a dot product of smooth vectors
// cancels, rounding their sum was most of its error, 2 to 3 times that of all the products.
__global__ void __launch_bounds__(NT) k_reduce_dots(int nblk, const cplx* __restrict__ partial,
                                                    cplx* __restrict__ out, cplx* __restrict__ acc_into) {
  mgc_pdl_enter();
  __shared__ double sh[2][NT / 32];
  __shared__ __int128 part[2][NT / 32];
  __shared__ int es;
  const int i = blockIdx.x, t = threadIdx.x;
  if (t == 0) es = 0;
  __syncthreads();
  int e = 0;
  for (int b = t; b < nblk; b += NT) e = max(e, fx_exp(partial[(size_t)i * nblk + b]));
  e = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
  if ((t & 31) == 0) atomicMax(&es, e);
  __syncthreads();
  cplx tot = cmk(0.0, 0.0);
  const int E = es;
  if (fx_ok(E)) {
    __int128 x = 0, y = 0;
    for (int b = t; b < nblk; b += NT) {
      const cplx v = partial[(size_t)i * nblk + b];
      x += fixed_128(v.x, E);
      y += fixed_128(v.y, E);
    }
    x = warp_sum_128(x);
    y = warp_sum_128(y);
    if ((t & 31) == 0) { part[0][t >> 5] = x; part[1][t >> 5] = y; }
    __syncthreads();
    if (t == 0) {
      const double sc = __hiloint2double((E - 1138 + 1023) << 20, 0);
      double r[2];
      for (int c = 0; c < 2; ++c) {
        __int128 s = part[c][0];
        for (int w = 1; w < NT / 32; ++w) s += part[c][w];
        const unsigned __int128 m = s < 0 ? -s : s;
        const double v = sc * fma((double)(unsigned long long)(m >> 64), 0x1p64, (double)(unsigned long long)m);
        r[c] = s < 0 ? -v : v;
      }
      tot = cmk(r[0], r[1]);
    }
  } else {
    cplx acc = cmk(0.0, 0.0);
    for (int b = t; b < nblk; b += NT) acc = cadd(acc, partial[(size_t)i * nblk + b]);
    tot = block_sum_c<NT>(acc, sh);
  }
  if (t == 0) {
    out[i] = tot;
    if (acc_into) acc_into[i] = cadd(acc_into[i], tot);
  }
}

// w += sgn * sum_{i<k} coef[i] V_i ; optional per-block partials of |w|^2.
template <class C>
__global__ void __launch_bounds__(NT) k_multiaxpy(long long n, int k, const C* __restrict__ V, long long ld,
                                                  const cplx* __restrict__ coef, double sgn, C* __restrict__ w,
                                                  double* __restrict__ norm_part, const int* __restrict__ gate,
                                                  const int* __restrict__ dk) {
  mgc_pdl_enter();
  __shared__ C sc[64];
  __shared__ double sh[NT / 32];
  if (gate && *gate == 0) return;
  if (dk) k = min(k, *dk);
  for (int i = threadIdx.x; i < k; i += NT) {
    const cplx q = cscal(sgn, coef[i]);
    sc[i] = CT<C>::make(q.x, q.y);
  }
  __syncthreads();
  typename CT<C>::R n2 = 0;
  for (long long p = blockIdx.x * (long long)NT + threadIdx.x; p < n; p += (long long)gridDim.x * NT) {
    C acc = w[p];
    for (int i = 0; i < k; ++i) acc = cfma(sc[i], __ldg(V + (size_t)i * ld + p), acc);
    w[p] = acc;
    n2 += cabs2(acc);
  }
  if (norm_part) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n2 += __shfl_down_sync(0xffffffffu, n2, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = (double)n2;
    __syncthreads();
    if (threadIdx.x == 0) {
      double tot = 0.0;
      for (int q = 0; q < NT / 32; ++q) tot += sh[q];
      norm_part[blockIdx.x] = tot;
    }
  }
}

// ---- complex64 update on element pairs.  With an even basis pitch every V_i + 2q and w + 2q
// is 16-byte aligned, so a thread moves two complex64 values per load; the loads of four
// basis vectors are issued before their FMAs, so each thread keeps four 16-byte loads in
// flight.  An odd last element is handled by one thread at the end.  (The same pair form
// of the multi-dot measured slower than the element form, 22.7 against 21.0 us a step,
// so the multi-dot keeps one element per thread.)

// acc += c * (a.x + i a.y) and c * (a.z + i a.w): two complex FMAs on a pair.
__device__ __forceinline__ float4 cfma2(float2 c, float4 a, float4 acc) {
  acc.x = fmaf(c.x, a.x, fmaf(-c.y, a.y, acc.x));
  acc.y = fmaf(c.x, a.y, fmaf(c.y, a.x, acc.y));
  acc.z = fmaf(c.x, a.z, fmaf(-c.y, a.w, acc.z));
  acc.w = fmaf(c.x, a.w, fmaf(c.y, a.z, acc.w));
  return acc;
}

// w += sgn * sum_{i<k} coef[i] V_i (complex64, pitch even, V and w 16-byte aligned);
// optional per-block partials of |w|^2.  Same operation as k_multiaxpy<float2>.
__global__ void __launch_bounds__(NT, 6) k_multiaxpy_c64(long long n, int k, const float2* __restrict__ V, long long ld,
                                                      const cplx* __restrict__ coef, double sgn,
                                                      float2* __restrict__ w, double* __restrict__ norm_part,
                                                      const int* __restrict__ gate, const int* __restrict__ dk) {
  mgc_pdl_enter();
  __shared__ float2 sc[64];
  __shared__ double sh[NT / 32];
  if (gate && *gate == 0) return;
  if (dk) k = min(k, *dk);
  for (int i = threadIdx.x; i < k; i += NT) {
    const cplx q = cscal(sgn, coef[i]);
    sc[i] = make_float2((float)q.x, (float)q.y);
  }
  __syncthreads();
  const float4* __restrict__ V4 = reinterpret_cast<const float4*>(V);
  float4* __restrict__ w4 = reinterpret_cast<float4*>(w);
  const long long ld4 = ld >> 1, np = n >> 1;
  float n2 = 0.f;
  for (long long q = blockIdx.x * (long long)NT + threadIdx.x; q < np; q += (long long)gridDim.x * NT) {
    float4 acc = w4[q];
    int i = 0;
    for (; i + 4 <= k; i += 4) {
      const float4 a0 = __ldg(V4 + (size_t)i * ld4 + q), a1 = __ldg(V4 + (size_t)(i + 1) * ld4 + q);
      const float4 a2 = __ldg(V4 + (size_t)(i + 2) * ld4 + q), a3 = __ldg(V4 + (size_t)(i + 3) * ld4 + q);
      acc = cfma2(sc[i], a0, acc);
      acc = cfma2(sc[i + 1], a1, acc);
      acc = cfma2(sc[i + 2], a2, acc);
      acc = cfma2(sc[i + 3], a3, acc);
    }
    for (; i < k; ++i) acc = cfma2(sc[i], __ldg(V4 + (size_t)i * ld4 + q), acc);
    w4[q] = acc;
    n2 += acc.x * acc.x + acc.y * acc.y + acc.z * acc.z + acc.w * acc.w;
  }
  if ((n & 1) && blockIdx.x == gridDim.x - 1 && threadIdx.x == NT - 1) {
    const long long p = n - 1;
    float2 acc = w[p];
    for (int i = 0; i < k; ++i) acc = cfma(sc[i], __ldg(V + (size_t)i * ld + p), acc);
    w[p] = acc;
    n2 += cabs2(acc);
  }
  if (norm_part) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) n2 += __shfl_down_sync(0xffffffffu, n2, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = (double)n2;
    __syncthreads();
    if (threadIdx.x == 0) {
      double tot = 0.0;
      for (int q = 0; q < NT / 32; ++q) tot += sh[q];
      norm_part[blockIdx.x] = tot;
    }
  }
}

// Whether the pair kernels apply: 16-byte aligned bases and an even pitch.
__host__ __forceinline__ bool pairs_ok(const void* a, const void* b, long long ld) {
  return ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b)) & 15) == 0 && (ld & 1) == 0;
}

// out = w / sqrt(*norm2) (zeros if the norm vanishes); *store = sqrt(*norm2) + 0i.
template <class C>
__global__ void __launch_bounds__(NT) k_scale_by_norm(long long n, const C* __restrict__ w, C* __restrict__ out,
                                                      const double* __restrict__ norm2, cplx* __restrict__ store) {
  mgc_pdl_enter();
  __shared__ double sb[2];
  if (threadIdx.x == 0) {
    const double b = sqrt(*norm2);
    sb[0] = b;
    sb[1] = b > 0.0 ? 1.0 / b : 0.0;
  }
  __syncthreads();
  const double beta = sb[0], s = sb[1];
  const long long p0 = blockIdx.x * (long long)NT + threadIdx.x;
  if (p0 == 0 && store) *store = cmk(beta, 0.0);
  for (long long p = p0; p < n; p += (long long)gridDim.x * NT) out[p] = cscal((typename CT<C>::R)s, w[p]);
}

// Apply rotations 0..j-1 to column j of H (h_{j+1,j} = sqrt(hn2)), build rotation j,
// update g; est = |g[j+1]|.  Called by every thread of one block.
// H is column-major with leading dimension m+1.  Rotation j maps rows (j, j+1) by
// [conj(c) conj(s); -s c] with c = a/rho, s = b/rho, rho = sqrt(|a|^2 + |b|^2).
__device__ __forceinline__ void givens_step(int j, int m, cplx* __restrict__ H, cplx* __restrict__ cs,
                                            cplx* __restrict__ sn, cplx* __restrict__ g, double* __restrict__ est,
                                            double hn2) {
  // the column and the earlier rotations are staged in shared memory by the block, so the
  // sequential chain of thread 0 waits on no global load
  __shared__ cplx col[MGC_MAX_RESTART + 1], rc[MGC_MAX_RESTART], rs[MGC_MAX_RESTART];
  cplx* colg = H + (size_t)j * (m + 1);
  for (int i = threadIdx.x; i <= j; i += blockDim.x) col[i] = colg[i];
  // h_{j+1,j} = |w| from its square (the value the normalisation of v_{j+1} uses), so the
  // rotation need not wait for that kernel
  if (threadIdx.x == 0) col[j + 1] = cmk(sqrt(hn2), 0.0);
  for (int i = threadIdx.x; i < j; i += blockDim.x) {
    rc[i] = cs[i];
    rs[i] = sn[i];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    // x carries entry i of the column through the chain in a register (rotation i - 1
    // wrote it), so each step waits on arithmetic only, not on a shared-memory round trip
    cplx x = col[0];
    for (int i = 0; i < j; ++i) {
      const cplx y = col[i + 1], c = rc[i], s = rs[i];
      col[i] = cadd(cmul(cmk(c.x, -c.y), x), cmul(cmk(s.x, -s.y), y));
      x = csub(cmul(c, y), cmul(s, x));
    }
    cplx a = x, b = col[j + 1];
    double rho = sqrt(cabs2(a) + cabs2(b));
    cplx c, s;
    if (rho == 0.0) {
      c = cmk(1.0, 0.0);
      s = cmk(0.0, 0.0);
    } else {
      c = cscal(1.0 / rho, a);
      s = cscal(1.0 / rho, b);
    }
    cs[j] = c;
    sn[j] = s;
    col[j] = cmk(rho, 0.0);
    col[j + 1] = cmk(0.0, 0.0);
    cplx gj = g[j];
    g[j + 1] = cneg(cmul(s, gj));
    g[j] = cmul(cmk(c.x, -c.y), gj);
    *est = cmod(g[j + 1]);
  }
  __syncthreads();
  for (int i = threadIdx.x; i <= j + 1; i += blockDim.x) colg[i] = col[i];
}

// The Givens update of step j on its own (after a second Gram-Schmidt pass); skipped when
// `gate` is given and *gate == 0 (the update then ran inside k_sum_dgks).
__global__ void k_givens(int j, int m, cplx* __restrict__ H, cplx* __restrict__ cs, cplx* __restrict__ sn,
                         cplx* __restrict__ g, double* __restrict__ est, const double* __restrict__ hnorm2,
                         const int* __restrict__ gate) {
  mgc_pdl_enter();
  if (gate && *gate == 0) return;
  givens_step(j, m, H, cs, sn, g, est, *hnorm2);
}

// Back substitution R y = g[0..k-1] with the rotated (upper-triangular) H.
__global__ void k_hess_solve(int k, int m, const cplx* __restrict__ H, const cplx* __restrict__ g,
                             cplx* __restrict__ y, const int* __restrict__ dk) {
  mgc_pdl_enter();
  if (threadIdx.x != 0) return;
  if (dk) k = min(k, *dk);
  for (int i = k - 1; i >= 0; --i) {
    cplx t = g[i];
    for (int q = i + 1; q < k; ++q) t = cfms(H[(size_t)q * (m + 1) + i], y[q], t);
    y[i] = cdiv(t, H[(size_t)i * (m + 1) + i]);
  }
}

// ---- device-driven GMRES: stop tests that steer the conditional nodes of a solve graph.
// One thread each; every value a test needs lives in the SolveCtl record.

// After the true residual |r|^2 of a restart: stop (converged, out of steps, non-finite,
// or a zero right-hand side) or open the next cycle with its estimate scale and target.
__global__ void k_outer_control(SolveCtl* __restrict__ c, const double* __restrict__ rn2p,
                                cudaGraphConditionalHandle h_outer, cudaGraphConditionalHandle h_cycle,
                                cudaGraphConditionalHandle h_inner, cudaGraphConditionalHandle h_switch) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  c->outer += 1;
  const double fn = sqrt(c->fn2);
  const double rn2 = *rn2p;
  bool stop = true;
  if (fn == 0.0) {
    c->rr = 0.0;
    c->status = SOLVECTL_ZERO_RHS;
  } else {
    const double rr = sqrt(rn2) / fn;
    c->rr = rr;
    if (rr < c->rr_min) c->rr_min = rr;
    if (!isfinite(rr)) {
      c->status = SOLVECTL_NONFINITE;
    } else if (rr > MGC_DIVERGENCE_FACTOR * c->rr_min) {
      c->status = SOLVECTL_DIVERGED;
    } else if (rr <= c->rtol) {
      c->status = SOLVECTL_CONVERGED;
    } else if (c->steps >= c->max_iter) {
      c->status = SOLVECTL_MAXITER;
    } else {
      const double beta = sqrt(rn2);
      if (c->mixed) {
        c->scale = beta / fn;
        c->target = fmax(c->inner_rtol, 0.5 * c->rtol * fn / beta) * beta / fn;
      } else {
        c->scale = 1.0 / fn;
        c->target = c->rtol;
      }
      c->j = 0;
      c->k = 0;
      c->cycles += 1;
      stop = false;
    }
  }
  cudaGraphSetConditional(h_outer, stop ? 0u : 1u);
  cudaGraphSetConditional(h_cycle, stop ? 0u : 1u);
  cudaGraphSetConditional(h_inner, stop ? 0u : 1u);
  cudaGraphSetConditional(h_switch, 0u);
}

// After Arnoldi step j: count it, and run step j+1 unless its residual estimate met the
// target, the step budget is spent, the cycle is full, or the estimate is not finite.
__global__ void k_step_control(SolveCtl* __restrict__ c, const double* __restrict__ est_raw,
                               cudaGraphConditionalHandle h_inner, cudaGraphConditionalHandle h_switch) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  const double est = *est_raw * c->scale;
  c->steps += 1;
  c->j += 1;
  c->k = c->j;
  const bool cont = isfinite(est) && est > c->target && c->steps < c->max_iter && c->j < c->m;
  cudaGraphSetConditional(h_switch, (unsigned)c->j);
  cudaGraphSetConditional(h_inner, cont ? 1u : 0u);
}

// Reorthogonalisation test: a second Gram-Schmidt pass runs only when the first pass
// cancelled |w| by more than a factor 1e3 (|w_after|^2 < 1e-6 |w_before|^2), so one
// pass never loses more than about 1e3 ulps of orthogonality.  (The classic threshold
// 1/sqrt(2) fires on almost every step here: with a good preconditioner A M^{-1} v_j is
// close to v_j and a first pass routinely removes half of |w|^2, harmlessly.)
// |w|^2 after the first pass comes from the block partials in the fixed summation order
// of k_sum_partials, and the decision is taken in the same kernel; in a device-driven
// solve graph it also sets the conditional node that holds the second pass (use_cond)
// and counts the passes that run.  When H is given and no second pass is needed (nearly
// every step), the Givens update of step j runs here as well, with the |w|^2 just
// summed, so it costs no launch of its own; after a second pass k_givens does it.
__global__ void __launch_bounds__(256) k_sum_dgks(const double* __restrict__ part, int n, double* __restrict__ out,
                                                  const double* __restrict__ before, int* __restrict__ gate,
                                                  cudaGraphConditionalHandle hd, int use_cond,
                                                  int* __restrict__ fired, int j, int m, cplx* __restrict__ H,
                                                  cplx* __restrict__ cs, cplx* __restrict__ sn,
                                                  cplx* __restrict__ g, double* __restrict__ est) {
  __shared__ double sh[8];
  __shared__ double s_tot;
  __shared__ int s_second;
  double v = 0.0;
  for (int k = threadIdx.x; k < n; k += 256) v += part[k];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) tot += sh[w];
    *out = tot;
    const int second = (tot < 1e-6 * *before) ? 1 : 0;
    *gate = second;
    if (use_cond) {
      cudaGraphSetConditional(hd, (unsigned)second);
      if (second) *fired += 1;
    }
    s_tot = tot;
    s_second = second;
  }
  __syncthreads();
  if (H && !s_second) givens_step(j, m, H, cs, sn, g, est, s_tot);
}

__global__ void k_zero_c(int n, cplx* __restrict__ a) {
  mgc_pdl_enter();
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) a[t] = cmk(0.0, 0.0);
}

}  // namespace

// The dynamic shared memory of the complex128 pair, allowed once per handle setup.
cudaError_t krylov_prepare() {
  cudaError_t e = cudaFuncSetAttribute(k_multidot_fx, cudaFuncAttributeMaxDynamicSharedMemorySize, MULTIDOT_SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_multiaxpy_fx<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, MULTIAXPY_SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_multiaxpy_fx<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, MULTIAXPY_SMEM);
  return e;
}

int krylov_blocks(long long n, int per_sm) {
  const long long b = (n + NT - 1) / NT, cap = (long long)per_sm * mgc_sm_count();
  return (int)(b < cap ? (b < 1 ? 1 : b) : cap);
}

// Four points a lane once they fill the resident blocks several times over, else two.
static bool axpy_wide(long long n) { return n >= 4LL * 2 * mgc_sm_count() * NT; }
int multiaxpy_blocks(long long n) {
  const long long b = (n + NT * 2 - 1) / (NT * 2), cap = (axpy_wide(n) ? 2LL : 3LL) * mgc_sm_count();
  return (int)(b < cap ? (b < 1 ? 1 : b) : cap);
}

// Blocks per vector of a k-vector multi-dot: about one full wave (8 blocks per SM) over
// all k vectors, so that each thread folds many elements before its share of the block
// reduction; never more than krylov_blocks(n), never fewer than 64.
template <class C>
int multidot_blocks(long long n, int k) {
  const int cap = krylov_blocks(n, 4);
  if constexpr (sizeof(C) == sizeof(cplx)) {
    // two resident blocks per SM over the groups of DG vectors
    const long long tiles = (n + NT * DU - 1) / (NT * DU), fill = 2LL * mgc_sm_count() / ((k + DG - 1) / DG);
    const long long b = tiles < fill ? tiles : fill;
    return (int)(b < 1 ? 1 : b < cap ? b : cap);
  }
  int b = 8 * mgc_sm_count() / (k < 1 ? 1 : k);
  if (b < 64) b = 64;
  return b < cap ? b : cap;
}

template <class C>
cudaError_t launch_multidot(long long n, int k, const C* V, long long ld, const C* w, cplx* partial,
                            int nblk, const int* gate, cudaStream_t st) {
  if constexpr (sizeof(C) == sizeof(cplx))
    return mgc_launch(k_multidot_fx, dim3(nblk, (k + DG - 1) / DG), dim3(NT), MULTIDOT_SMEM, st, n, k, V, ld, w,
                      partial, gate);
  else
    return mgc_launch(k_multidot<C>, dim3(nblk, k), dim3(NT), 0, st, n, V, ld, w, partial, gate);
}

cudaError_t launch_reduce_dots(int nblk, int k, const cplx* partial, cplx* out, cplx* acc_into, cudaStream_t st) {
  return mgc_launch(k_reduce_dots, dim3(k), dim3(NT), 0, st, nblk, partial, out, acc_into);
}

template <class C>
cudaError_t launch_multiaxpy(long long n, int k, const C* V, long long ld, const cplx* coef, double sgn,
                             C* w, double* norm_part, int nblk, const int* gate, cudaStream_t st, const int* dk) {
  if constexpr (sizeof(C) == sizeof(cplx)) {
    if (axpy_wide(n))
      return mgc_launch(k_multiaxpy_fx<4>, dim3(nblk), dim3(NT), MULTIAXPY_SMEM, st, n, k, V, ld, coef, sgn, w, norm_part,
                        gate, dk);
    return mgc_launch(k_multiaxpy_fx<2>, dim3(nblk), dim3(NT), MULTIAXPY_SMEM, st, n, k, V, ld, coef, sgn, w, norm_part,
                      gate, dk);
  } else {
    if (pairs_ok(V, w, ld)) {
      return mgc_launch(k_multiaxpy_c64, dim3(nblk), dim3(NT), 0, st, n, k, V, ld, coef, sgn, w, norm_part, gate, dk);
    }
  }
  if constexpr (sizeof(C) == sizeof(float2))
    return mgc_launch(k_multiaxpy<C>, dim3(nblk), dim3(NT), 0, st, n, k, V, ld, coef, sgn, w, norm_part, gate, dk);
}

template <class C>
cudaError_t launch_scale_by_norm(long long n, const C* w, C* out, const double* norm2, cplx* store,
                                 int nblk, cudaStream_t st) {
  return mgc_launch(k_scale_by_norm<C>, dim3(nblk), dim3(NT), 0, st, n, w, out, norm2, store);
}

#define MGC_INSTANTIATE(C)                                                                                  \
  template int multidot_blocks<C>(long long, int);                                                          \
  template cudaError_t launch_multidot<C>(long long, int, const C*, long long, const C*, cplx*, int,        \
                                         const int*, cudaStream_t);                                       \
  template cudaError_t launch_multiaxpy<C>(long long, int, const C*, long long, const cplx*, double, C*,   \
                                          double*, int, const int*, cudaStream_t, const int*);            \
  template cudaError_t launch_scale_by_norm<C>(long long, const C*, C*, const double*, cplx*, int,         \
                                              cudaStream_t);
MGC_INSTANTIATE(double2)
MGC_INSTANTIATE(float2)
#undef MGC_INSTANTIATE

cudaError_t launch_givens(int j, int m, cplx* H, cplx* cs, cplx* sn, cplx* g, double* est, const double* hnorm2,
                          cudaStream_t st, const int* gate) {
  return mgc_launch(k_givens, dim3(1), dim3(32), 0, st, j, m, H, cs, sn, g, est, hnorm2, gate);
}

cudaError_t launch_hess_solve(int k, int m, const cplx* H, const cplx* g, cplx* y, cudaStream_t st,
                              const int* dk) {
  return mgc_launch(k_hess_solve, dim3(1), dim3(32), 0, st, k, m, H, g, y, dk);
}


cudaError_t launch_outer_control(SolveCtl* c, const double* rn2, cudaGraphConditionalHandle h_outer,
                                 cudaGraphConditionalHandle h_cycle, cudaGraphConditionalHandle h_inner,
                                 cudaGraphConditionalHandle h_switch, cudaStream_t st) {
  k_outer_control<<<1, 32, 0, st>>>(c, rn2, h_outer, h_cycle, h_inner, h_switch);
  return cudaGetLastError();
}

cudaError_t launch_step_control(SolveCtl* c, const double* est, cudaGraphConditionalHandle h_inner,
                                cudaGraphConditionalHandle h_switch, cudaStream_t st) {
  k_step_control<<<1, 32, 0, st>>>(c, est, h_inner, h_switch);
  return cudaGetLastError();
}

cudaError_t launch_sum_dgks(const double* part, int n, double* out, const double* before, int* gate,
                           cudaStream_t st, cudaGraphConditionalHandle hd, int* fired, const GivensArgs* gv) {
  if (gv)
    k_sum_dgks<<<1, 256, 0, st>>>(part, n, out, before, gate, hd, fired ? 1 : 0, fired, gv->j, gv->m, gv->H, gv->cs,
                                  gv->sn, gv->g, gv->est);
  else
    k_sum_dgks<<<1, 256, 0, st>>>(part, n, out, before, gate, hd, fired ? 1 : 0, fired, 0, 0, nullptr, nullptr,
                                  nullptr, nullptr, nullptr);
  return cudaGetLastError();
}

cudaError_t launch_zero_c(int n, cplx* a, cudaStream_t st) {
  return mgc_launch(k_zero_c, dim3((n + 255) / 256), dim3(256), 0, st, n, a);
}
