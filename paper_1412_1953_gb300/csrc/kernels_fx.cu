// Complex128 level passes on the integer pipes (stencil_fx.cuh): the fused passes of a V-cycle
// level and the fine-level operator and residual.  They give what k_zero_residual_restrict,
// k_prolong_jacobi, k_apply and k_residual (kernels_mg.cu) give with FP64 instructions, to
// rounding; tiles whose exponents are out of range (all zero, subnormal, huge or not finite)
// take those instructions here as well.
#include <cmath>
#include <cstring>

#include "stencil_fx.cuh"

namespace {

constexpr int BX = 32;


// ---- level operator as limbs

// lim[0], lim[1] = largest and smallest exponent of the n values (of the larger component).
__global__ void __launch_bounds__(256) k_exponents(long long n, const cplx* __restrict__ a, int* __restrict__ lim) {
  int hi = 0, lo = 4096;
  for (long long p = blockIdx.x * 256LL + threadIdx.x; p < n; p += (long long)gridDim.x * 256) {
    const int e = fx_exp(a[p]);
    hi = max(hi, e);
    lo = min(lo, e);
  }
  hi = (int)__reduce_max_sync(0xffffffffu, (unsigned)hi);
  lo = (int)__reduce_min_sync(0xffffffffu, (unsigned)lo);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(lim, hi);
    atomicMin(lim + 1, lo);
  }
}

// most[0] = the bits of the largest sum over a node of |re| + |im| of its five coefficients, most[1] of
// that sum times |re| + |im| of the node's omega/D.
__global__ void __launch_bounds__(256) k_row_bound(StencilView s, unsigned long long* __restrict__ most) {
  const long long n = (long long)s.mx * s.my;
  double m = 0.0, g = 0.0;
  for (long long p = blockIdx.x * 256LL + threadIdx.x; p < n; p += (long long)gridDim.x * 256) {
    const int i = (int)(p % s.mx), j = (int)(p / s.mx);
    const double row =
        cabs1(s.D[p]) + cabs1(s.west_x[i]) + cabs1(s.east_x[i]) + cabs1(s.west_y[j]) + cabs1(s.east_y[j]);
    m = fmax(m, row);
    g = fmax(g, cabs1(s.Dinv[p]) * row);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    g = fmax(g, __shfl_xor_sync(0xffffffffu, g, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(most, (unsigned long long)__double_as_longlong(m));
    atomicMax(most + 1, (unsigned long long)__double_as_longlong(g));
  }
}

// the limbs of a value, or of a coefficient
__device__ __forceinline__ int4 coef_limbs(cplx z, int E) {
  const int4 v = fx_limbs(z, E);
  int4 c;
  fx_coef(((long long)v.x << 29) + v.y, &c.x, &c.y);
  fx_coef(((long long)v.z << 29) + v.w, &c.z, &c.w);
  return c;
}
template <bool COEF>
__global__ void __launch_bounds__(256) k_split(long long n, const cplx* __restrict__ a, int E, int4* __restrict__ out) {
  for (long long p = blockIdx.x * 256LL + threadIdx.x; p < n; p += (long long)gridDim.x * 256)
    out[p] = COEF ? coef_limbs(a[p], E) : fx_limbs(a[p], E);
}
// An axis' west or east coefficients.  The inner region takes its closed form here as well, as the
// FP64 passes do in a straddling block: the per-node values differ from it by the rounding of the
// grid's coordinates (4e-14 of it at 592 nodes), and the two must be the same operator.
__global__ void __launch_bounds__(256) k_split_axis(int n, AxisCoefT<cplx> ax, const cplx* __restrict__ a, int E,
                                                    int4* __restrict__ out) {
  for (int p = blockIdx.x * 256 + threadIdx.x; p < n; p += gridDim.x * 256) out[p] = coef_limbs(p < ax.u ? ax.cin : a[p], E);
}

// ---- a level's (zero-start sweep,) residual and restriction.  A block takes 16 x DBY coarse nodes:
// u on the fine nodes [2 I0 - 1, 2 I0 + 33] x [2 J0 - 1, 2 J0 + 2 DBY + 1] as integers in shared
// memory, the residuals on the tile less its rim as integers in f's and (H - E)u's common unit,
// then the weighted sums, shifts and additions only, and one conversion per coarse value.  With
// ZERO, u = (omega/D) f is formed first, with FP64 instructions (two or four, which keep each value's
// bits), and stored for the nodes the block owns.  A block of which some residual's terms all lie
// below 2^53 units takes FP64 instructions throughout: its coarse values are made of such residuals.
// Bound by the integer pipe and the latency of its barriers.  With cold L2 at 1023^2, zero start: 39.5 us
// (sweep 11.5 + residual and restriction 47.3 us with FP64 instructions).  Four blocks an SM: the
// preconditioner takes 226 us with three, 220 us with four.
constexpr int DBX = 16, DBY = 8, DT = 256, UR = 2 * DBY + 3, RR = 2 * DBY + 1, DUW = 2 * DBX + 3, DRW = 2 * DBX + 1;

template <bool ZERO>
__global__ void __launch_bounds__(DT, 4) k_zrr_fx(StencilFx x, int mcx, int mcy, const cplx* __restrict__ f,
                                               cplx* __restrict__ u, cplx* __restrict__ fc) {
  mgc_pdl_enter();
  const StencilView& s = x.s;
  __shared__ longlong2 U[UR * DUW];
  __shared__ longlong2 Rt[RR * DRW];
  __shared__ int2 eu_s, ef_s;
  const int t = threadIdx.x, I0 = blockIdx.x * DBX, J0 = blockIdx.y * DBY, i0 = 2 * I0, j0 = 2 * J0;
  if (t == 0) eu_s = ef_s = make_int2(0, 0);
  __syncthreads();
  const auto ux = [](int c) { return c == 0 ? -1 : 31 + c; };          // columns -1, 32, 33
  const auto rx = [](int) { return 32; };
  const bool box = s.rbox && i0 + DUW - 1 <= s.cx.u && j0 + UR - 1 <= s.cy.u;   // omega/D real throughout
  const auto sweep = [&](size_t p, cplx fp) {                           // (omega/D) f
    return box ? cscal(ldre(s.Dinv, (int)p), fp) : cmul(__ldg(s.Dinv + p), fp);
  };
  TileShare<DT / 32, UR, 3> tu;
  TileShare<DT / 32, RR, 1> tf;                                         // f at the residual nodes
  int2 eu_t = tu.load(ZERO ? f : u, s.mx, s.my, i0, j0 - 1, ux);
  block_exponent(tf.load(f, s.mx, s.my, i0, j0, rx), &ef_s);
  if constexpr (ZERO) {
    eu_t = make_int2(0, 0);
    tu.each(ux, [&](int r, int c, cplx& z) {
      const int i = i0 + c, j = j0 - 1 + r;
      if (i < 0 || j < 0 || i >= s.mx || j >= s.my) return;
      const size_t p = (size_t)j * s.mx + i;
      z = sweep(p, z);
      const int oi = min(i >> 1, mcx - 1), oj = min(j >> 1, mcy - 1);
      if (oi >= I0 && oi < I0 + DBX && oj >= J0 && oj < J0 + DBY) u[p] = z;
      eu_t = fx_max_exp(eu_t, z);
    });
  }
  block_exponent(eu_t, &eu_s);
  __syncthreads();
  const int eu = max(eu_s.x, eu_s.y), ef = max(ef_s.x, ef_s.y);
  bool ok = fx_tile_ok(eu_s) && fx_tile_ok(ef_s);
  // units: of u, below 2^58, and of the residuals, below 2^60, so that four of them fit
  const int qu = eu - 1080, qt = qu + x.ec - 1021, qr = max(qt, ef - 1081);
  const int i1 = min(i0 + DRW, s.mx), j1 = min(j0 + RR, s.my);
  if (ok) {
    tu.each(ux, [&](int r, int c, cplx z) { U[r * DUW + c + 1] = fx_int(z, qu); });
    __syncthreads();
    const int d = qr - qt;                               // positive only where f exceeds (H - E)u's range
    bool low = false;
    fx_kinds(s, i0, i1, j0, j1, [&](auto kx, auto ky, auto rd) {
      tf.each(rx, [&](int r, int c, cplx z) {
        const int i = i0 + c, j = j0 + r;
        if (i >= s.mx || j >= s.my) return;
        const longlong2* q = U + (r + 1) * DUW + c + 1;
        longlong2 h = fx_operator<decltype(kx)::value, decltype(ky)::value, decltype(rd)::value>(
            x, i, j, (size_t)j * s.mx + i, q, DUW);
        int lead = fx_lead5(q, DUW);
        if (d > 0) {
          const int k = min(d, 62);
          const long long b = (1LL << (k - 1)) - 1;                     // to the nearest, ties to even
          h = make_longlong2((h.x + b + (h.x >> k & 1)) >> k, (h.y + b + (h.y >> k & 1)) >> k);
          lead >>= min(d, 31);
        }
        const longlong2 fi = fx_int(z, qr);
        low = low || !fx_kept(lead | fx_lead(fi));
        Rt[r * DRW + c] = make_longlong2(fi.x - h.x, fi.y - h.y);
      });
    });
    ok = !__syncthreads_or(low);
  }
  if (!ok) {
    const auto val = [&](size_t p, bool in) {
      if (!in) return cmk(0.0, 0.0);
      const cplx z = __ldg((ZERO ? f : u) + p);
      return ZERO ? sweep(p, z) : z;
    };
    dispatch_kinds(s, i0, i1, j0, j1, [&](auto kx, auto ky, auto ir, auto dg) {
      tf.each(rx, [&](int r, int c, cplx z) {
        const int i = i0 + c, j = j0 + r;
        if (i >= s.mx || j >= s.my) return;
        const size_t p = (size_t)j * s.mx + i;
        Rt[r * DRW + c] = as_raw(
            residual_vals<decltype(kx)::value, decltype(ky)::value, decltype(ir)::value, decltype(dg)::value>(
                s, i, j, (int)p, val(p, true), val(p - 1, i > 0), val(p + 1, i + 1 < s.mx), val(p - s.mx, j > 0),
                val(p + s.mx, j + 1 < s.my), z));
      });
    });
    __syncthreads();
  }
  const int I = I0 + t % DBX, J = J0 + t / DBX;
  if (t >= DBX * DBY || I >= mcx || J >= mcy) return;
  const longlong2* c = Rt + (2 * (t / DBX) + 1) * DRW + 2 * (t % DBX) + 1;   // on fine node (2I+1, 2J+1)
  if (ok) {
    // a sixteenth of 4 centre + 2 edge + corner as a double: exact before its rounding below 2^58, else
    // first to the nearest integer, ties to even (a floor's constant bias is a smooth residual, which
    // the coarse levels amplify: measured 60 times the error)
    const double sc = fx_pow2(qr);
    auto weigh = [&](auto get) {
      const long long edge = get(-1) + get(1) + get(-DRW) + get(DRW);
      const long long corner = get(-DRW - 1) + get(-DRW + 1) + get(DRW - 1) + get(DRW + 1);
      const long long whole = (get(0) >> 2) + (edge >> 3) + (corner >> 4);
      const int rest = 4 * (int)(get(0) & 3) + 2 * (int)(edge & 7) + (int)(corner & 15);
      const bool fits = (whole ^ whole >> 63) >> 58 == 0;
      const long long sum = fits ? (whole << 4) + rest : whole + ((rest + 7 + ((int)(whole + (rest >> 4)) & 1)) >> 4);
      return (fits ? 0.0625 * sc : sc) * (double)sum;
    };
    fc[(size_t)J * mcx + I] = cmk(weigh([&](int o) { return c[o].x; }), weigh([&](int o) { return c[o].y; }));
  } else {
    auto get = [&](int o) { return as_cplx(c[o]); };
    const cplx corner = cadd(cadd(get(-DRW - 1), get(-DRW + 1)), cadd(get(DRW - 1), get(DRW + 1)));
    const cplx edge = cadd(cadd(get(-1), get(1)), cadd(get(-DRW), get(DRW)));
    const cplx m = get(0);
    fc[(size_t)J * mcx + I] =
        cscal(0.0625, cmk(fma(2.0, edge.x, fma(4.0, m.x, corner.x)), fma(2.0, edge.y, fma(4.0, m.y, corner.y))));
  }
}

// ---- a level's prolongation and first post-smoothing sweep, o = v + (omega/D)(f - (H - E) v) with
// v = u + P e.  A block forms twice the coarse values of its region interpolated along x, then v on
// its 32 x 8 nodes and a rim of one as integers in a unit that also holds (omega/D) f, the residual
// as integers, and the update as one integer per component.  A node whose terms all lie below 2^53
// units takes FP64 instructions, from the arrays (pj_node).  Bound by the integer pipe:
// 33.6 us at 1023^2 with cold L2 (prolongation 13.2 + sweep 34.9 us with FP64 instructions).  Four
// blocks an SM: 220 us for the preconditioner, against 231 us with three and 229 us with five.
constexpr int PW = BX + 2, PY = 8, PE = BX / 2 + 2, PER = PY / 2 + 2;

// One node with FP64 instructions.  Out of line: few nodes need it, and inlined its registers are
// the pass's.
__device__ __noinline__ cplx pj_node(const StencilView& s, int mcx, int mcy, const cplx* __restrict__ ec,
                                     const cplx* __restrict__ u, const cplx* __restrict__ f, int i, int j) {
  const auto v = [&](int a, int b) {
    if (a < 0 || b < 0 || a >= s.mx || b >= s.my) return cmk(0.0, 0.0);
    const auto e = [&](int q, int r) {
      return ld_or_zero(ec, (size_t)r * mcx + q, q >= 0 && r >= 0 && q < mcx && r < mcy);
    };
    // on coarse index a >> 1 where a is odd, else between that and the one before
    const int q = a >> 1, r = b >> 1;
    cplx y = e(q, r);
    double h = 1.0;
    if (!(a & 1) && !(b & 1)) {
      y = cadd(cadd(e(q - 1, r - 1), e(q, r - 1)), cadd(e(q - 1, r), y));
      h = 0.25;
    } else if (!(a & 1)) {
      y = cadd(e(q - 1, r), y);
      h = 0.5;
    } else if (!(b & 1)) {
      y = cadd(e(q, r - 1), y);
      h = 0.5;
    }
    const cplx z = __ldg(u + (size_t)b * s.mx + a);
    return cmk(fma(h, y.x, z.x), fma(h, y.y, z.y));
  };
  const int p = j * s.mx + i;
  const cplx c = v(i, j), w = v(i - 1, j), e = v(i + 1, j), so = v(i, j - 1), n = v(i, j + 1), fp = __ldg(f + p);
  if (s.cx.in_real && s.cy.in_real) return jacobi_vals<AX_GEN, AX_GEN, 1, DG_GEN>(s, i, j, p, c, w, e, so, n, fp);
  return jacobi_vals<AX_GEN, AX_GEN, 0, DG_GEN>(s, i, j, p, c, w, e, so, n, fp);
}

__global__ void __launch_bounds__(BX * PY, 4) k_pj_fx(StencilFx x, int mcx, int mcy, const cplx* __restrict__ ec,
                                                   const cplx* __restrict__ u, cplx* __restrict__ o,
                                                   const cplx* __restrict__ f) {
  mgc_pdl_enter();
  const StencilView& s = x.s;
  static_assert(PE * PER <= BX * PY && PW * PER <= BX * PY, "one coarse value per thread");
  __shared__ longlong2 T[(PY + 2) * PW];
  __shared__ longlong2 Es[PER * PE], Ex[PER * PW];
  __shared__ int2 eu_s, ef_s;
  const int t = threadIdx.y * BX + threadIdx.x, i0 = blockIdx.x * BX, j0 = blockIdx.y * PY;
  const int i = i0 + threadIdx.x, j = j0 + threadIdx.y;
  const bool mine = i < s.mx && j < s.my;
  if (t == 0) eu_s = ef_s = make_int2(0, 0);
  __syncthreads();
  const auto ux = [](int c) { return c ? BX : -1; };
  TileShare<PY, PY + 2, 2> tu;
  const int2 eu_t = tu.load(u, s.mx, s.my, i0, j0 - 1, ux);
  // coarse interior indices [i0/2 - 1, i0/2 + 16] x [j0/2 - 1, j0/2 + PY/2]
  const int er = t / PE, ei = t - er * PE, ci = i0 / 2 - 1 + ei, cj = j0 / 2 - 1 + er;
  const cplx e = t < PE * PER && ci >= 0 && cj >= 0 && ci < mcx && cj < mcy ? __ldg(ec + (size_t)cj * mcx + ci)
                                                                         : cmk(0.0, 0.0);
  const cplx fv = mine ? __ldg(f + (size_t)j * s.mx + i) : cmk(0.0, 0.0);
  block_exponent(fx_max_exp(eu_t, e), &eu_s);
  block_exponent(fx_max_exp(make_int2(0, 0), fv), &ef_s);
  __syncthreads();
  const int eu = max(eu_s.x, eu_s.y), ef = max(ef_s.x, ef_s.y);
  bool ok = fx_tile_ok(eu_s) && fx_tile_ok(ef_s);
  // units: of v (u and P e below 2^57, (omega/D) f below 2^58) and of the residual (below 2^60)
  const int qu = max(eu, ef + x.ed - 1022) - 1079, qr = qu + x.ec - 1021;
  if (ok) {
    if (t < PE * PER) Es[t] = fx_int(e, qu);
    __syncthreads();
    // column a = i0 - 1 + q odd: on coarse index a >> 1, even: between that and the one before
    if (t < PW * PER) {
      const int r = t / PW, q = t - r * PW;
      const longlong2 c = Es[r * PE + (q + 1) / 2], b = Es[r * PE + (q + 1) / 2 - (q & 1)];
      Ex[t] = fx_add(c, b);
    }
    __syncthreads();
    tu.each(ux, [&](int r, int c, cplx z) {
      const int a = i0 + c, b = j0 - 1 + r;
      longlong2 w = make_longlong2(0, 0);
      if (a >= 0 && b >= 0 && a < s.mx && b < s.my) {
        const longlong2* g = Ex + ((b >> 1) - (j0 / 2 - 1)) * PW + c + 1;
        const longlong2 y = fx_add(g[0], g[b & 1 ? 0 : -PW]);          // four times P e
        w = fx_add(fx_int(z, qu), make_longlong2(fx_quarter(y.x), fx_quarter(y.y)));
      }
      T[r * PW + c + 1] = w;
    });
    __syncthreads();
  }
  if (!mine) return;
  const size_t p = (size_t)j * s.mx + i;
  if (ok) {
    const longlong2* c = T + (threadIdx.y + 1) * PW + threadIdx.x + 1;
    const int i1 = min(i0 + BX, s.mx), j1 = min(j0 + PY, s.my);
    fx_kinds(s, i0, i1, j0, j1, [&](auto kx, auto ky, auto rd) {
      const longlong2 h = fx_operator<decltype(kx)::value, decltype(ky)::value, decltype(rd)::value>(x, i, j, p, c, PW);
      const longlong2 fi = fx_int(fv, qr);
      const longlong2 r = make_longlong2(fi.x - h.x, fi.y - h.y);
      // (omega/D) f is at least 2^(52 - kd) f in units of v
      ok = fx_kept(fx_lead5(c, PW) | fx_lead(fi) >> max(x.kd - 52, 0));
      FxSum re{0, 0}, im{0, 0};
      if constexpr (decltype(rd)::value) {
        const int2 d = __ldg(reinterpret_cast<const int2*>(x.Di + p));
        fx_rmac(re, im, d.x, d.y, r);
      } else {
        fx_cmac(re, im, __ldg(x.Di + p), r);
      }
      const double sc = fx_pow2(qu);
      if (ok) o[p] = cmk(sc * (double)(c[0].x + fx_scaled(re, x.kd)), sc * (double)(c[0].y + fx_scaled(im, x.kd)));
    });
  }
  if (!ok) o[p] = pj_node(s, mcx, mcy, ec, u, f, i, j);
}

// ---- y = (H - E) x.  Four FP64 instructions a node (two conversions, two products) and as much
// integer work bound it, beside the traffic: 22.1 us at 1023^2 with cold L2 (34.6 us with FP64
// instructions).
__global__ void __launch_bounds__(BX * PY) k_apply_fx(StencilFx x, const cplx* __restrict__ u, cplx* __restrict__ y) {
  mgc_pdl_enter();
  const StencilView& s = x.s;
  __shared__ longlong2 T[(PY + 2) * PW];
  __shared__ int2 eu_s;
  const int i0 = blockIdx.x * BX, j0 = blockIdx.y * PY, i = i0 + threadIdx.x, j = j0 + threadIdx.y;
  if (threadIdx.x + threadIdx.y == 0) eu_s = make_int2(0, 0);
  __syncthreads();
  const auto ux = [](int c) { return c ? BX : -1; };
  TileShare<PY, PY + 2, 2> tu;
  block_exponent(tu.load(u, s.mx, s.my, i0, j0 - 1, ux), &eu_s);
  __syncthreads();
  const int eu = max(eu_s.x, eu_s.y);
  bool ok = fx_tile_ok(eu_s);
  if (ok) tu.each(ux, [&](int r, int c, cplx z) { T[r * PW + c + 1] = fx_int(z, eu - 1080); });
  __syncthreads();
  if (i >= s.mx || j >= s.my) return;
  const size_t p = (size_t)j * s.mx + i;
  const longlong2* c = T + (threadIdx.y + 1) * PW + threadIdx.x + 1;
  const int i1 = min(i0 + BX, s.mx), j1 = min(j0 + PY, s.my);
  if (ok) {
    fx_kinds(s, i0, i1, j0, j1, [&](auto kx, auto ky, auto rd) {
      const longlong2 h = fx_operator<decltype(kx)::value, decltype(ky)::value, decltype(rd)::value, 3>(x, i, j, p, c, PW);
      const double sc = fx_pow2(eu + x.ec - 2104);
      ok = fx_kept(fx_lead5(c, PW));
      if (ok) y[p] = cmk(sc * (double)h.x, sc * (double)h.y);
    });
  }
  if (!ok) {
    const cplx uw = ld_or_zero(u, p - 1, i > 0), ue = ld_or_zero(u, p + 1, i + 1 < s.mx);
    const cplx us = ld_or_zero(u, p - s.mx, j > 0), un = ld_or_zero(u, p + s.mx, j + 1 < s.my);
    dispatch_kinds(s, i0, i1, j0, j1, [&](auto kx, auto ky, auto ir, auto dg) {
      y[p] = apply_vals<decltype(kx)::value, decltype(ky)::value, decltype(ir)::value, decltype(dg)::value>(
          s, i, j, (int)p, __ldg(u + p), uw, ue, us, un);
    });
  }
}

unsigned stride_blocks(long long n) {
  const long long b = (n + 255) / 256, cap = 8LL * mgc_sm_count();
  return (unsigned)(b < cap ? (b < 1 ? 1 : b) : cap);
}

}  // namespace

size_t level_fx_entries(int mx, int my) { return 2 * ((size_t)mx * my + mx + my); }

// A level's exponents and bounds into lim (FX_LIMITS device ints, 8-byte aligned: largest and smallest
// exponent of west, east, D; of omega/D; the bits of the two bounds).
cudaError_t launch_level_exponents(const StencilView& s, int* lim, cudaStream_t st) {
  static const int init[FX_LIMITS] = {0, 4096, 0, 4096, 0, 0, 0, 0};
  cudaError_t e = cudaMemcpyAsync(lim, init, sizeof(init), cudaMemcpyHostToDevice, st);
  if (e != cudaSuccess) return e;
  const long long n = (long long)s.mx * s.my;
  k_exponents<<<stride_blocks(n), 256, 0, st>>>(n, s.D, lim);
  k_exponents<<<stride_blocks(s.mx), 256, 0, st>>>(s.mx, s.west_x, lim);
  k_exponents<<<stride_blocks(s.mx), 256, 0, st>>>(s.mx, s.east_x, lim);
  k_exponents<<<stride_blocks(s.my), 256, 0, st>>>(s.my, s.west_y, lim);
  k_exponents<<<stride_blocks(s.my), 256, 0, st>>>(s.my, s.east_y, lim);
  k_exponents<<<stride_blocks(n), 256, 0, st>>>(n, s.Dinv, lim + 2);
  k_row_bound<<<stride_blocks(n), 256, 0, st>>>(s, reinterpret_cast<unsigned long long*>(lim + 4));
  return cudaGetLastError();
}

// A coefficient's limbs on the host, those of coef_limbs.
static void host_coef(double x, int E, int* h, int* l) {
  const long long m = (long long)std::floor(std::ldexp(std::fabs(x), 1079 - E) + 0.5);
  fx_coef(x < 0 ? -m : m, h, l);
}

// The level's operator as limbs in buf (level_fx_entries), if its exponents (lim, on the host)
// allow it.
cudaError_t level_fx(const StencilView& s, const int* lim, int4* buf, StencilFx* out, cudaStream_t st) {
  StencilFx x{};
  x.s = s;
  x.ec = lim[0];
  x.ed = lim[2];
  const auto ok = [](int e) { return e >= FX_MIN && e <= FX_MAX; };
  double row, gain;
  std::memcpy(&row, lim + 4, sizeof(row));
  std::memcpy(&gain, lim + 6, sizeof(gain));
  x.kd = 2100 - x.ec - x.ed;
  // the exponents within their spread; every sum (H - E)u below 2^(ec - 1020) max |u|, which keeps
  // it in 64 bits; the update's scaling within fx_scaled's range, and f's unit no coarser than
  // (omega/D) f needs (ec + ed >= 2042); and the new value of k_pj_fx in 64 bits (FX_GAIN)
  x.on = lim[0] - lim[1] <= FX_SPREAD && lim[2] - lim[3] <= FX_SPREAD && ok(x.ec) && ok(x.ed) &&
         std::isfinite(row) && row <= std::ldexp(1.0, x.ec - 1020) && x.kd >= 30 && x.kd <= 58 && gain <= FX_GAIN;
  if (x.on) {
    const long long n = (long long)s.mx * s.my;
    int4* D = buf;
    int4* Di = buf + n;
    int4* a = buf + 2 * n;
    x.D = D; x.Di = Di;
    x.wx = a; x.ex = a + s.mx; x.wy = a + 2 * s.mx; x.ey = a + 2 * s.mx + s.my;
    k_split<true><<<stride_blocks(n), 256, 0, st>>>(n, s.D, x.ec, D);
    k_split<false><<<stride_blocks(n), 256, 0, st>>>(n, s.Dinv, x.ed, Di);
    k_split_axis<<<stride_blocks(s.mx), 256, 0, st>>>(s.mx, s.cx, s.west_x, x.ec, a);
    k_split_axis<<<stride_blocks(s.mx), 256, 0, st>>>(s.mx, s.cx, s.east_x, x.ec, a + s.mx);
    k_split_axis<<<stride_blocks(s.my), 256, 0, st>>>(s.my, s.cy, s.west_y, x.ec, a + 2 * s.mx);
    k_split_axis<<<stride_blocks(s.my), 256, 0, st>>>(s.my, s.cy, s.east_y, x.ec, a + 2 * s.mx + s.my);
    host_coef(s.cx.cin.x, x.ec, &x.cx.x, &x.cx.y);
    host_coef(s.cx.cin.y, x.ec, &x.cx.z, &x.cx.w);
    host_coef(s.cy.cin.x, x.ec, &x.cy.x, &x.cy.y);
    host_coef(s.cy.cin.y, x.ec, &x.cy.z, &x.cy.w);
  }
  *out = x;
  return cudaGetLastError();
}

cudaError_t launch_zrr_fx(const StencilFx& x, const cplx* f, cplx* u, cplx* fc, bool zero, cudaStream_t st) {
  const StencilView& s = x.s;
  const int mcx = (s.mx - 1) / 2, mcy = (s.my - 1) / 2;
  if (s.mx != 2 * mcx + 1 || s.my != 2 * mcy + 1) return cudaErrorInvalidValue;
  const dim3 grid((mcx + DBX - 1) / DBX, (mcy + DBY - 1) / DBY);
  if (zero) return mgc_launch(k_zrr_fx<true>, grid, dim3(DT), 0, st, x, mcx, mcy, f, u, fc);
  return mgc_launch(k_zrr_fx<false>, grid, dim3(DT), 0, st, x, mcx, mcy, f, u, fc);
}

cudaError_t launch_pj_fx(const StencilFx& x, const cplx* ec, const cplx* u, cplx* o, const cplx* f, cudaStream_t st) {
  const StencilView& s = x.s;
  const int mcx = (s.mx - 1) / 2, mcy = (s.my - 1) / 2;
  if (s.mx != 2 * mcx + 1 || s.my != 2 * mcy + 1) return cudaErrorInvalidValue;
  return mgc_launch(k_pj_fx, dim3((s.mx + BX - 1) / BX, (s.my + PY - 1) / PY), dim3(BX, PY), 0, st, x, mcx, mcy, ec, u,
                    o, f);
}

cudaError_t launch_apply_fx(const StencilFx& x, const cplx* u, cplx* y, cudaStream_t st) {
  const dim3 g((x.s.mx + BX - 1) / BX, (x.s.my + PY - 1) / PY);
  return mgc_launch(k_apply_fx, g, dim3(BX, PY), 0, st, x, u, y);
}
