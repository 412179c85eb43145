// The 5-point operator on the integer pipes (fixed.cuh): a block turns its tile of grid values
// into integers on one exponent, the operator's coefficients are kept as limbs on one exponent
// per level, and a node's sums lose only the products of low limbs (2^-60 of the largest product).
// One exponent for a tile leaves its small values fewer bits than a double has, so a tile or a
// node takes FP64 instructions where that would show in a result (fx_tile_ok, fx_kept).
// Where the operator cancels, the coarser levels amplify what a sum leaves on smooth data by its
// condition, so every rounding here is to the nearest and without a mean.  V-cycles of 256^2 to 768 x 512
// against extended precision with the device's coefficients: l2 error 0.5 to 1.06 times that of the
// one-step FP64 kernels, on rough and on smooth data.
#pragma once
#include "fixed.cuh"

// A level's operator as limbs.  `on` when all of west, east and D lie within FX_SPREAD powers of
// two of the largest (each by the larger of its parts), and all of omega/D likewise: limbs keep 57
// bits of the largest, so within four powers of two that larger part keeps the 53 bits of its double
// (level_fx in kernels_fx.cu); otherwise the level keeps to FP64.  Square cells spread over three, cells
// of twice the height over four; at five and six a coefficient was up to 2 and 4 units of 2^-53 off.
struct StencilFx {
  StencilView s;
  int on;
  int ec, ed;                              // exponents of west, east, D, and of omega/D
  int kd;                                  // 2100 - ec - ed, between 30 and 58
  int4 cx, cy;                             // the inner regions' coefficients (fx_coef)
  const int4 *wx, *ex, *wy, *ey;           // per-node neighbour coefficients (fx_coef)
  const int4 *D, *Di;                      // [my*mx] (fx_coef; fx_limbs)
};
constexpr int FX_SPREAD = 4;
// Most a node's |omega/D| times its row's sum of coefficients (|re| + |im| of each) may be.  In the
// units of k_pj_fx v and (omega/D) f stay below 2^58, so (omega/D)(H - E) v stays below 2^58 times this
// gain and the new value below (2 + gain) 2^58, 2^62.2; beyond 30 it would wrap.  An energy close to
// the diagonal's 2/h^2 makes D small there: 2.7 at E = 0.5 on 256^2 cells of [0, 30]^2, 14 at E = 130, 47 at
// E = 135.  A level beyond it keeps to FP64.
constexpr double FX_GAIN = 16.0;
constexpr int FX_LIMITS = 8;               // ints of launch_level_exponents
// A coefficient of 57 bits as h 2^27 + l / 4, |h| <= 2^30, |l| <= 2^28: finer in the low limb than a
// value (split at 2^29), so that the products of low limbs that a sum drops are below 2^54, a quarter of
// a unit for a value's last bit times the smallest neighbour coefficient of square cells.
__host__ __device__ __forceinline__ void fx_coef(long long m, int* h, int* l) {
  *h = (int)((m + (1 << 26)) >> 27);
  *l = (int)(m - ((long long)*h << 27)) * 4;
}

// Levels of at least this many nodes run on the integer pipes: smaller ones are bound by a launch's
// latency, and the exponent's reduction and barriers lengthen that.  The preconditioner by grid size
// n, integer passes (three blocks an SM) on no level / on every level / from 60000 nodes (us): 128: 60.8 / 67.3 / 60.8,
// 256: 72.6 / 75.0 / 69.0, 512: 125 / 116 / 114, 1024: 272 / 242 / 240; from 120000: 256: 72.6,
// 1024: 242.
constexpr long long FX_NODES = 60000;

// x in units of 2^q, to the nearest integer; x must be below 2^(q + 62).  Cutting instead would
// leave a mean of half a unit towards zero on a smooth right-hand side, which the coarser levels
// amplify by the operator's condition.
__device__ __forceinline__ long long fx_int(double x, int q) {
  const int hi = __double2hiint(x), s = hi >> 31;
  const unsigned lo = (unsigned)__double2loint(x);
  const unsigned a1 = __funnelshift_l(lo, ((unsigned)hi & 0xfffffu) | 0x100000u, 11), a0 = lo << 11;
  const int t = q + 1085 - ((hi >> 20) & 0x7ff);                       // at least 0; the last place kept is a half
  const long long m = t > 63 ? 0 : (long long)((((unsigned long long)a1 << 32 | a0) >> t) + 1) >> 1;
  return (m ^ s) - s;
}
__device__ __forceinline__ longlong2 fx_int(cplx z, int q) { return make_longlong2(fx_int(z.x, q), fx_int(z.y, q)); }
__device__ __forceinline__ double fx_pow2(int q) { return __hiloint2double((q + 1023) << 20, 0); }
// v = h 2^29 + l with l in [-2^28, 2^28): the products of low limbs, which a sum drops, then have no
// mean.  With l in [0, 2^29) they leave a constant of half a unit where (H - E)u cancels, a smooth
// residual that the coarser levels amplify (25 times FP64's error on rough u, 240^2 to 767 x 511).
__device__ __forceinline__ FxLimbs fx_split(long long v) {
  const int h = (int)((v + (1LL << 28)) >> 29);
  return FxLimbs{h, (int)((unsigned)v - ((unsigned)h << 29))};
}
__device__ __forceinline__ longlong2 fx_add(longlong2 a, longlong2 b) { return make_longlong2(a.x + b.x, a.y + b.y); }
// a quarter, to the nearest, ties to even
__device__ __forceinline__ long long fx_quarter(long long a) { return (a + 1 + (a >> 2 & 1)) >> 2; }
// (re, im) += a v, a complex (limbs) or real (its first two)
__device__ __forceinline__ void fx_cmac(FxSum& re, FxSum& im, int4 a, longlong2 v) {
  const FxLimbs ax{a.x, a.y}, ay{a.z, a.w}, x = fx_split(v.x), y = fx_split(v.y);
  fx_mac(re, ax, x);
  fx_mac(re, fx_neg(ay), y);
  fx_mac(im, ax, y);
  fx_mac(im, ay, x);
}
__device__ __forceinline__ void fx_rmac(FxSum& re, FxSum& im, int ah, int al, longlong2 v) {
  const FxLimbs a{ah, al};
  fx_mac(re, a, fx_split(v.x));
  fx_mac(im, a, fx_split(v.y));
}
// The sum hh 2^58 + mid 2^29 divided by 2^k, 30 <= k <= 58, rounded; the caller knows that it fits.
__device__ __forceinline__ long long fx_scaled(const FxSum& s, int k) {
  return (s.hh << (58 - k)) + ((s.mid + (1LL << (k - 30))) >> (k - 29));
}

// How a block's nodes take the coefficients: KX, KY = AX_IN or AX_ARR as in dispatch_kinds (a
// straddling block uses the per-node arrays, which cover every node), RD = all real.
// Calls f(IntC<KX>, IntC<KY>, IntC<RD>) for interior indices [i0, i1) x [j0, j1).
template <class F>
__device__ __forceinline__ void fx_kinds(const StencilView& s, int i0, int i1, int j0, int j1, F&& f) {
  const bool xi = i1 <= s.cx.u, yi = j1 <= s.cy.u;
  if (xi && yi) {
    if (s.rbox && s.cx.in_real && s.cy.in_real) f(IntC<AX_IN>(), IntC<AX_IN>(), IntC<1>());
    else f(IntC<AX_IN>(), IntC<AX_IN>(), IntC<0>());
  } else if (xi) {
    f(IntC<AX_IN>(), IntC<AX_ARR>(), IntC<0>());
  } else if (yi) {
    f(IntC<AX_ARR>(), IntC<AX_IN>(), IntC<0>());
  } else {
    f(IntC<AX_ARR>(), IntC<AX_ARR>(), IntC<0>());
  }
}

// (H - E) u at node p = (i, j), whose value in units of 2^qu is t[0] of a tile with row pitch
// `pitch` (values below 2^58, so that a sum of two still splits into 31-bit limbs), in units of
// 2^(qu + ec - 1021 - XB), below 2^(59 + XB).  XB = 3 where a double is made of it: a coefficient of
// the spread's end times a value of 2^57 is then rounded to less than a double's last place.
template <int KX, int KY, int RD, int XB = 0>
__device__ __forceinline__ longlong2 fx_operator(const StencilFx& x, int i, int j, size_t p, const longlong2* t,
                                                 int pitch) {
  FxSum re{0, 0}, im{0, 0};
  const longlong2 w = t[-1], e = t[1], s = t[-pitch], n = t[pitch];
  if constexpr (RD) {
    fx_rmac(re, im, x.cx.x, x.cx.y, fx_add(w, e));
    fx_rmac(re, im, x.cy.x, x.cy.y, fx_add(s, n));
    const int2 d = __ldg(reinterpret_cast<const int2*>(x.D + p));
    fx_rmac(re, im, d.x, d.y, t[0]);
  } else {
    if constexpr (KX == AX_IN) {
      fx_cmac(re, im, x.cx, fx_add(w, e));
    } else {
      fx_cmac(re, im, __ldg(x.wx + i), w);
      fx_cmac(re, im, __ldg(x.ex + i), e);
    }
    if constexpr (KY == AX_IN) {
      fx_cmac(re, im, x.cy, fx_add(s, n));
    } else {
      fx_cmac(re, im, __ldg(x.wy + j), s);
      fx_cmac(re, im, __ldg(x.ey + j), n);
    }
    fx_cmac(re, im, __ldg(x.D + p), t[0]);
  }
  // the sums are hh 2^56 + mid 2^27 in products of units, hh and mid below 2^62; results in 2^58 or 2^55
  const auto total = [](const FxSum& t) {
    if constexpr (XB == 3) return (t.hh << 1) + ((t.mid + (1LL << 27)) >> 28);
    else return fx_quarter(t.hh + ((t.mid + (1LL << 28)) >> 29));
  };
  static_assert(XB == 0 || XB == 3, "units of the result");
  return make_longlong2(total(re), total(im));
}

__device__ __forceinline__ int2 fx_max_exp(int2 e, cplx z) {
  return make_int2(max(e.x, fx_exp(z.x)), max(e.y, fx_exp(z.y)));
}
// Where one exponent will do for a tile of complex values with largest exponents e.x (real parts) and
// e.y (imaginary parts): in range, and neither part more than 2^FX_NEAR below the other, unless it is zero.
__device__ __forceinline__ bool fx_tile_ok(int2 e) {
  const int hi = max(e.x, e.y), lo = min(e.x, e.y);
  return fx_ok(hi) && (lo == 0 || hi - lo <= FX_NEAR);
}
// ... and for a node of it: of the values v that its sum takes (in units that put the tile's largest
// between 2^57 and 2^58) at least one part is 2^53 or more, so that its rounding is no coarser than a
// double's.  Collect the leading bits of all of them, then ask fx_kept.
__device__ __forceinline__ int fx_lead(longlong2 v) {
  const int x = (int)(v.x >> 32), y = (int)(v.y >> 32);
  return (x ^ x >> 31) | (y ^ y >> 31);
}
__device__ __forceinline__ bool fx_kept(int lead) { return lead >= 1 << (57 - FX_NEAR - 32); }
// of a node's five values
__device__ __forceinline__ int fx_lead5(const longlong2* t, int pitch) {
  return fx_lead(t[0]) | fx_lead(t[-1]) | fx_lead(t[1]) | fx_lead(t[-pitch]) | fx_lead(t[pitch]);
}

// A thread's share of a tile of ROWS x (32 + XC) complex values around the 32 columns i0..i0+31 and
// first row jt: rows warp, warp + NW, ... at its lane's column, and one of the XC extra columns
// (column xc(c), c = 0..XC-1) of one row.  put(row, column - i0, value) is called for each.
template <int NW, int ROWS, int XC>
struct TileShare {
  static constexpr int NR = (ROWS + NW - 1) / NW;
  static_assert(XC * ROWS <= 32 * NW, "one extra value per thread");
  cplx v[NR], x;
  // loads from a (mx x my; zero outside) and returns the largest exponents of the parts
  template <class XF>
  __device__ __forceinline__ int2 load(const cplx* __restrict__ a, int mx, int my, int i0, int jt, XF xc) {
    const int lane = threadIdx.x & 31, t = threadIdx.x + threadIdx.y * blockDim.x, w = t >> 5, i = i0 + lane;
    int2 e = make_int2(0, 0);
#pragma unroll
    for (int n = 0; n < NR; ++n) {
      const int r = w + NW * n, j = jt + r;
      v[n] = r < ROWS && i < mx && j >= 0 && j < my ? __ldg(a + (size_t)j * mx + i) : cmk(0.0, 0.0);
      e = fx_max_exp(e, v[n]);
    }
    const int r = t / XC, i2 = i0 + xc(t - r * XC), j2 = jt + r;
    x = t < XC * ROWS && i2 >= 0 && i2 < mx && j2 >= 0 && j2 < my ? __ldg(a + (size_t)j2 * mx + i2) : cmk(0.0, 0.0);
    return fx_max_exp(e, x);
  }
  template <class XF, class F>
  __device__ __forceinline__ void each(XF xc, F&& put) {
    const int lane = threadIdx.x & 31, t = threadIdx.x + threadIdx.y * blockDim.x, w = t >> 5;
#pragma unroll
    for (int n = 0; n < NR; ++n) {
      const int r = w + NW * n;
      if (r < ROWS) put(r, lane, v[n]);
    }
    const int r = t / XC;
    if (t < XC * ROWS) put(r, xc(t - r * XC), x);
  }
};
__device__ __forceinline__ cplx as_cplx(longlong2 v) {
  return cmk(__longlong_as_double(v.x), __longlong_as_double(v.y));
}
__device__ __forceinline__ longlong2 as_raw(cplx v) {
  return make_longlong2(__double_as_longlong(v.x), __double_as_longlong(v.y));
}
// The largest exponents over the block, in *es (cleared before).
__device__ __forceinline__ void block_exponent(int2 e, int2* es) {
  e.x = (int)__reduce_max_sync(0xffffffffu, (unsigned)e.x);
  e.y = (int)__reduce_max_sync(0xffffffffu, (unsigned)e.y);
  if ((threadIdx.x & 31) == 0) {
    atomicMax(&es->x, e.x);
    atomicMax(&es->y, e.y);
  }
}
__device__ __forceinline__ cplx ld_or_zero(const cplx* __restrict__ a, size_t p, bool ok) {
  return ok ? __ldg(a + p) : cmk(0.0, 0.0);
}

// kernels_fx.cu
size_t level_fx_entries(int mx, int my);                                  // int4 entries of a level's limbs
cudaError_t launch_level_exponents(const StencilView& s, int* lim, cudaStream_t st);   // FX_LIMITS device ints
cudaError_t level_fx(const StencilView& s, const int* lim, int4* buf, StencilFx* out, cudaStream_t st);
cudaError_t launch_zrr_fx(const StencilFx& x, const cplx* f, cplx* u, cplx* fc, bool zero, cudaStream_t st);
cudaError_t launch_pj_fx(const StencilFx& x, const cplx* ec, const cplx* u, cplx* o, const cplx* f, cudaStream_t st);
cudaError_t launch_apply_fx(const StencilFx& x, const cplx* u, cplx* y, cudaStream_t st);

// kernels_cccs.cu (s.on 0: the residuals in FP64)
cudaError_t launch_residual_project(const StencilFx& s, const CCView& c, const cplx* u, const cplx* f, cudaStream_t st);
