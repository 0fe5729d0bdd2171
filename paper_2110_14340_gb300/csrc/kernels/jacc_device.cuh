// jacc_device.cuh - device code of the runtime-specialised stencil path.
//
// No system headers: the same text (plus jacc_params.h) is compiled by nvcc
// into the precompiled "generic" kernels, where extents and coefficients
// arrive as kernel arguments, and by NVRTC into constant-folded variants,
// where a struct with static constexpr members replaces the argument struct
// (the paper's kernel specialisation, §3.2.2: runtime-invariant parameters
// become constants).
//
// Stencils (the paper's workloads are memory-bound halo stencils, §5.2 and
// Table 1; these are the 5-, 7- and 27-point members of that family):
//   5-point Jacobi (2D)  v = (N + S + W + E) / 4
//   7-point heat   (3D)  v = u + r (sum of 6 faces - 6 u)
//   27-point box   (3D)  v = w0 c + wf (6 faces) + we (12 edges) + wc (8 corners), periodic
// Dirichlet boundary points are copied unchanged.
//
// FP64 arithmetic.  On GB300 the FP64 pipe and every conversion to or from a
// 64-bit type issue at about 2 lanes/clock/SM, against ~100-128 for INT32
// and FP32, so an FP64 stencil done in FP64 instructions is ALU-bound far
// below the HBM roof.  For convex stencils the values never leave
// [-M, M], M = max|u| of the sweep input (maximum principle), so each sweep
// runs in exact 64-bit fixed point: value = q * 2^-F with F = 57 - e(M)
// (|q| < 2^57, six bits of headroom).  Conversions FP64 <-> fixed are done
// with integer instructions; sums and power-of-two scalings are exact, so the
// only rounding is the final, correctly rounded conversion of the exact
// stencil value to FP64.  Non-dyadic coefficients use exact 128-bit products.
// Non-convex coefficients, or a non-finite or tiny input, use the native FP64
// path (chosen per launch by a uniform branch).
#pragma once

#include "jacc_params.h"

#define JD __device__ __forceinline__

// The parameter block of a table tile's kernel: the march length is the tile's
// own, known to the compiler.
template <int ZC> struct JParamsZ : JParams {
  static constexpr int zc = ZC;
};
// The parameter block with 32-bit fixed-point factors (JACC_FP_W32).
struct JParamsW32 : JParams {
  static constexpr int fpath = JACC_FP_W32;
};
// Whether extents and coefficients are constants (P is none of these blocks).
template <class P> struct Folded { static constexpr bool value = !__is_base_of(JParams, P); };

// ---------------------------------------------------------------- fixed point

// Fraction bits for the sweep from the bit pattern of max|u| (non-negative
// double).  Returns -1 when the fixed path cannot be used (Inf/NaN input, or a
// maximum below 2^-959 so that the format would leave the normal range).
JD int fx_frac_bits(u64 maxbits) {
  if (maxbits == 0ull) return 57;
  int eb = (int)(maxbits >> 52);
  if (eb >= 0x7ff || eb < 64) return -1;
  return 1079 - eb;  // M < 2^(eb-1022)  =>  |q| < 2^57
}

// x * 2^F truncated toward zero.  |x| <= M means the value is below 2^57, so
// it is the 53-bit significand in the top of a 57-bit field shifted right by
// the exponent's distance from M's; zero and subnormals are 64 or more away
// and shift to nothing.
JD i64 fx_from(double x, int F) {
  const u64 b = (u64)__double_as_longlong(x);
  const int hi = (int)(b >> 32);
  const int d = 1079 - F - ((hi >> 20) & 0x7ff);
  const u64 m = ((b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull) << 4;
  const i64 r = (i64)(m >> (d < 63 ? d : 63));
  const i64 s = (i64)(hi >> 31);
  return (r ^ s) - s;
}

// q * 2^-E rounded to nearest even, |q| < 2^62.  The magnitude is shifted to
// bit 62; adding just under half of the last place plus the last bit rounds
// half to even, and a carry out of the 53-bit significand propagates into the
// exponent field by construction.
JD double fx_to(i64 q, int E) {
  const i64 s = q >> 63;
  const u64 a = (u64)((q ^ s) - s);
  const int lz = __clzll((i64)a);
  const u64 n = a << ((lz - 1) & 63);
  const u64 mant = (n + 0x1ffull + ((n >> 10) & 1ull)) >> 10;
  const u64 bits = mant + ((u64)(u32)((63 - lz - E + 1022) << 20) << 32);
  return a ? __longlong_as_double((i64)(bits | ((u64)s & 0x8000000000000000ull))) : 0.0;
}

// Unsigned magnitude version (for residual maxima).
JD double fx_to_u(u64 a, int E) { return fx_to((i64)a, E); }

// 128-bit two's complement value.
struct s128 { u64 lo; u64 hi; };

JD s128 mul_s64_u64(i64 a, u64 b) {
  s128 r;
  r.lo = (u64)a * b;
  r.hi = __umul64hi((u64)a, b) - ((a < 0) ? b : 0ull);
  return r;
}
JD s128 add128(s128 x, s128 y) {
  s128 r;
  r.lo = x.lo + y.lo;
  r.hi = x.hi + y.hi + (u64)(r.lo < x.lo);
  return r;
}
JD s128 from_s64_shl(i64 a, int k) {  // a * 2^k, 0 <= k < 64
  s128 r;
  r.lo = (u64)a << k;
  r.hi = (k == 0) ? (u64)(a >> 63) : (u64)(a >> (64 - k));
  return r;
}
// (x.hi:x.lo) * 2^-E rounded to nearest even, by selections only: the
// magnitude's top 63 significant bits, the last one set when any bit below it
// was, then the rounding of fx_to.
JD double fx128_to(s128 x, int E) {
  const u64 s = (u64)((i64)x.hi >> 63);
  const u64 lo = (x.lo ^ s) - s;
  const u64 hi = (x.hi ^ s) + (u64)(s != 0ull && lo == 0ull);
  const bool low = hi == 0ull;
  const u64 h = low ? lo : hi, l = low ? 0ull : lo;
  const int lz = __clzll((i64)h) & 63;
  const u64 m = (h << lz) | ((l >> 1) >> (63 - lz));
  const u64 n = (m >> 1) | (m & 1ull) | (u64)((l << lz) != 0ull);
  const u64 mant = (n + 0x1ffull + ((n >> 10) & 1ull)) >> 10;
  const u64 bits = mant + ((u64)(u32)(((low ? 63 : 127) - lz - E + 1022) << 20) << 32);
  return h ? __longlong_as_double((i64)(bits | (s & 0x8000000000000000ull))) : 0.0;
}

// ---------------------------------------------------------------- load / store helpers

template <class T, int V> struct VecT;
template <> struct VecT<double, 1> { typedef double type; };
template <> struct VecT<double, 2> { typedef double2 type; };
template <> struct VecT<float, 1> { typedef float type; };
template <> struct VecT<float, 4> { typedef float4 type; };

// CG = true loads through L2 only (ld.global.cg): required where the same
// kernel launch writes the array (the persistent batched kernel), since the
// non-coherent and L1 paths may return stale lines there.
template <bool CG, class T> JD T ld1(const T* p) {
  if constexpr (CG) return __ldcg(p);
  else return __ldg(p);
}
template <class T, int V, bool CG = false> JD void ldv(const T* __restrict__ p, T (&r)[V]) {
  if constexpr (V == 1) { r[0] = ld1<CG>(p); }
  else if constexpr (V == 2) {
    double2 t = ld1<CG>(reinterpret_cast<const double2*>(p)); r[0] = t.x; r[1] = t.y;
  } else {
    float4 t = ld1<CG>(reinterpret_cast<const float4*>(p)); r[0] = t.x; r[1] = t.y; r[2] = t.z; r[3] = t.w;
  }
}
template <class T, int V> JD void stv(T* __restrict__ p, const T (&r)[V]) {
  if constexpr (V == 1) { p[0] = r[0]; }
  else if constexpr (V == 2) { double2 t; t.x = r[0]; t.y = r[1]; *reinterpret_cast<double2*>(p) = t; }
  else { float4 t; t.x = r[0]; t.y = r[1]; t.z = r[2]; t.w = r[3]; *reinterpret_cast<float4*>(p) = t; }
}

// Arithmetic modes.
#define JM_NATIVE 0
#define JM_FIXED 1

// Internal value type: T for native, int64 fixed point for JM_FIXED.
template <class T, int MODE> struct WT { typedef T type; };
template <class T> struct WT<T, JM_FIXED> { typedef i64 type; };

template <class T, int MODE> JD typename WT<T, MODE>::type cvt_in(T x, int F) {
  if constexpr (MODE == JM_FIXED) return fx_from((double)x, F);
  else return x;
}

// Per-thread residual accumulator: the magnitude of a fixed-point
// difference (converted once at the end), or a non-negative T.
template <class T, int MODE> struct RT { typedef T type; };
template <class T> struct RT<T, JM_FIXED> { typedef u64 type; };

// ---------------------------------------------------------------- block reductions

// Maximum of a 64-bit word over the (converged) warp: the maximum of the high
// halves, then the maximum of the low halves of the lanes that hold it; two
// redux.sync operations instead of five shuffle rounds.
JD u64 warp_max_u64(u64 v) {
  const u32 hi = __reduce_max_sync(0xffffffffu, (u32)(v >> 32));
  const u32 lo = __reduce_max_sync(0xffffffffu, (u32)(v >> 32) == hi ? (u32)v : 0u);
  return ((u64)hi << 32) | lo;
}
JD double warp_sum_f64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Max over the block of a non-negative double given as its bit pattern, then
// one atomicMax per block (non-negative doubles order like their bit patterns).
template <int NT> JD void block_max_to(u64 bits, double* out) {
  __shared__ u64 red[NT / 32];
  const int t = threadIdx.x + threadIdx.y * blockDim.x;
  bits = warp_max_u64(bits);
  if ((t & 31) == 0) red[t >> 5] = bits;
  __syncthreads();
  if (t < 32) {
    u64 v = (t < NT / 32) ? red[t] : 0ull;
    v = warp_max_u64(v);
    if (t == 0 && out) atomicMax(reinterpret_cast<unsigned long long*>(out), (unsigned long long)v);
  }
}

template <int NT> JD void block_sum_to(double s, double* out) {
  __shared__ double red[NT / 32];
  const int t = threadIdx.x + threadIdx.y * blockDim.x;
  s = warp_sum_f64(s);
  if ((t & 31) == 0) red[t >> 5] = s;
  __syncthreads();
  if (t < 32) {
    double v = (t < NT / 32) ? red[t] : 0.0;
    v = warp_sum_f64(v);
    if (t == 0 && out) atomicAdd(out, v);
  }
}

JD u64 dbits(double d) { return (u64)__double_as_longlong(d); }

// Programmatic dependent launch: a sweep kernel may be launched while the
// previous one still runs (its CTAs fill the SMs the previous grid frees);
// this waits until the previous grid has completed and its memory is
// visible, before the kernel touches any field.  A no-op when the launch
// did not ask for programmatic serialisation.
JD void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// Whether the word at `stop` (nullable) is set: read by one thread of the CTA,
// after griddep_wait.  Were every warp to read it, one L2 slice would serve them
// all in turn (160^3 FP32 without staging, 25600 warps: 22 us a sweep of
// jacc_sweep_until, 13 so; 128^3 FP64 17.4 and 12.4).
JD bool stopped(const int* stop) {
  return stop && __syncthreads_or(threadIdx.x == 0 && threadIdx.y == 0 && __ldcg(stop) != 0);
}

// FP32 error-free sum (Knuth TwoSum) accumulated as hi + lo.
JD void two_sum_acc(float& hi, float& lo, float x) {
  float s = hi + x;
  float bp = s - hi;
  float e = (hi - (s - bp)) + (x - bp);
  hi = s;
  lo += e;
}

// ====================================================================== 5-point Jacobi (2D)
//
// One warp owns 32*V consecutive columns starting at its lane-0 column and
// marches rows [ys, ye), keeping rows y-1, y, y+1 in registers; the x
// neighbours come from warp shuffles (lanes 0 and 31 read the edge columns
// from memory).  Row y+3 is prefetched two iterations ahead.  All 32 lanes
// must call it with the same ys, ye (full-mask shuffles).

template <class T, int V, int MODE, bool CG>
JD void jacobi_march(const T* __restrict__ u, T* __restrict__ v, i64 nx, i64 ny, i64 x0, i64 ys, i64 ye, int F,
                     typename RT<T, MODE>::type& rmax) {
  typedef typename WT<T, MODE>::type W;
  const int lane = threadIdx.x & 31;
  const bool xin = x0 < nx;
  T rup[V], rcur[V], rdn[V], rnx[V];
  W up[V], cur[V], dn[V];
#pragma unroll
  for (int e = 0; e < V; ++e) { rup[e] = rcur[e] = rdn[e] = rnx[e] = T(0); }
  if (xin) {
    if (ys >= 1) ldv<T, V, CG>(u + (ys - 1) * nx + x0, rup);
    ldv<T, V, CG>(u + ys * nx + x0, rcur);
    if (ys + 1 < ny) ldv<T, V, CG>(u + (ys + 1) * nx + x0, rdn);
    if (ys + 2 < ny) ldv<T, V, CG>(u + (ys + 2) * nx + x0, rnx);
  }
#pragma unroll
  for (int e = 0; e < V; ++e) {
    up[e] = cvt_in<T, MODE>(rup[e], F);
    cur[e] = cvt_in<T, MODE>(rcur[e], F);
    dn[e] = cvt_in<T, MODE>(rdn[e], F);
  }
  for (i64 y = ys; y < ye; ++y) {
    // x neighbours of the row
    W left = __shfl_up_sync(0xffffffffu, cur[V - 1], 1);
    W right = __shfl_down_sync(0xffffffffu, cur[0], 1);
    if (lane == 0 && xin && x0 >= 1) left = cvt_in<T, MODE>(ld1<CG>(u + y * nx + x0 - 1), F);
    if (lane == 31 && xin && x0 + V < nx) right = cvt_in<T, MODE>(ld1<CG>(u + y * nx + x0 + V), F);
    // prefetch row y+3
    T rnn[V];
#pragma unroll
    for (int e = 0; e < V; ++e) rnn[e] = T(0);
    if (xin && y + 3 < ny) ldv<T, V, CG>(u + (y + 3) * nx + x0, rnn);

    const bool yint = (y >= 1) && (y <= ny - 2);
    T out[V];
#pragma unroll
    for (int e = 0; e < V; ++e) {
      const i64 x = x0 + e;
      const W xl = (e == 0) ? left : cur[e - 1];
      const W xr = (e == V - 1) ? right : cur[e + 1];
      const bool in = yint && (x >= 1) && (x <= nx - 2);
      {
        const T s = (up[e] + dn[e]) + (xl + xr);
        const T r = T(0.25) * s;
        out[e] = in ? r : rcur[e];
        T d = r - rcur[e];
        d = d < T(0) ? -d : d;
        if (in && d > rmax) rmax = d;
      }
    }
    if (xin) stv<T, V>(v + y * nx + x0, out);
#pragma unroll
    for (int e = 0; e < V; ++e) {
      up[e] = cur[e];
      cur[e] = dn[e];
      rcur[e] = rdn[e];
      rdn[e] = rnx[e];
      dn[e] = cvt_in<T, MODE>(rnx[e], F);
      rnx[e] = rnn[e];
    }
  }
}

// ====================================================================== 3D z-marching tiles
//
// CTA = BX x BY threads covering x in [bx0, bx0 + BX*V), y in [by0, by0 + BY),
// marching z over [cz0, cz0 + ZC).  The current plane lives in shared memory
// with a one-point halo in x and y (double-buffered, so one __syncthreads per
// plane); each thread keeps its own column's z-1, z, z+1 in registers.
// Loads for plane z+1 (halo) and z+2 (own) are issued one iteration ahead.

template <class W, int BX, int BY, int V> struct alignas(16) Plane {
  // row layout: [pad V-1][left halo][TX values][right halo][pad V-1]
  static constexpr int TX = BX * V;
  static constexpr int RW = TX + 2 * V;
  static constexpr int ROWS = BY + 2;
  W a[2][ROWS][RW];
};

template <class T, int BX, int BY, int V> struct HaloFetch {
  T yrow[V];  // thread rows 0 / BY-1: the row above / below the tile
  T xl, xr;   // threads tx 0 / BX-1: the column left / right of the tile
};

template <class T, int BX, int BY, int V, class P>
JD void fetch_halo(const T* __restrict__ u, const P& p, i64 z, i64 bx0, i64 by0, bool periodic,
                   HaloFetch<T, BX, BY, V>& h) {
  const i64 nx = p.nx, ny = p.ny, nz = p.nz;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const i64 x0 = bx0 + (i64)tx * V;
  const i64 y = by0 + ty;
  if (periodic) z = (z + nz) % nz;
  const T* pl = u + z * nx * ny;
#pragma unroll
  for (int e = 0; e < V; ++e) h.yrow[e] = T(0);
  h.xl = h.xr = T(0);
  // Periodic tiles that overhang the grid load the periodic image, so the
  // slot after the last column (row) holds column (row) 0.
  const i64 xl0 = periodic ? (x0 % nx) : x0;
  if (xl0 < nx) {
    if (ty == 0) {
      i64 yy = by0 - 1;
      if (periodic) yy = (yy + ny) % ny;
      if (yy >= 0) ldv<T, V>(pl + yy * nx + xl0, h.yrow);
    }
    if (ty == BY - 1) {
      i64 yy = by0 + BY;
      if (periodic) yy = yy % ny;
      if (yy < ny) ldv<T, V>(pl + yy * nx + xl0, h.yrow);
    }
  }
  // x halo: the thread at tx == 0 fetches for its own row (and the halo rows
  // through the diagonal corners below), tx == BX-1 likewise on the right.
  if (y < ny || periodic) {
    i64 yy = periodic ? (y % ny) : y;
    if (tx == 0) {
      i64 xx = bx0 - 1;
      if (periodic) xx = (xx + nx) % nx;
      if (xx >= 0 && yy < ny) h.xl = __ldg(pl + yy * nx + xx);
    }
    if (tx == BX - 1) {
      i64 xx = bx0 + BX * V;
      if (periodic) xx = xx % nx;
      if (xx < nx && yy < ny) h.xr = __ldg(pl + yy * nx + xx);
    }
  }
}

// Write this thread's converted plane values and its halo share into buffer b.
template <class T, int BX, int BY, int V, int MODE>
JD void put_plane(Plane<typename WT<T, MODE>::type, BX, BY, V>& sm, int b, const typename WT<T, MODE>::type (&own)[V],
                  const HaloFetch<T, BX, BY, V>& h, int F) {
  const int tx = threadIdx.x, ty = threadIdx.y;
  typedef typename WT<T, MODE>::type W;
  W* row = &sm.a[b][ty + 1][V + tx * V];
#pragma unroll
  for (int e = 0; e < V; ++e) row[e] = own[e];
  if (ty == 0) {
    W* hr = &sm.a[b][0][V + tx * V];
#pragma unroll
    for (int e = 0; e < V; ++e) hr[e] = cvt_in<T, MODE>(h.yrow[e], F);
  }
  if (ty == BY - 1) {
    W* hr = &sm.a[b][BY + 1][V + tx * V];
#pragma unroll
    for (int e = 0; e < V; ++e) hr[e] = cvt_in<T, MODE>(h.yrow[e], F);
  }
  if (tx == 0) sm.a[b][ty + 1][V - 1] = cvt_in<T, MODE>(h.xl, F);
  if (tx == BX - 1) sm.a[b][ty + 1][V + BX * V] = cvt_in<T, MODE>(h.xr, F);
}


// ---------------------------------------------------------------- 7-point heat
//
// Native FP64 arithmetic, and the planes of the kernels that stage nothing.

template <class T, int BX, int BY, int V, int MODE, class P>
JD void heat3d_body(const T* __restrict__ u, T* __restrict__ v, const P& p, int zc, int F, typename RT<T, MODE>::type& rmax,
                    Plane<typename WT<T, MODE>::type, BX, BY, V>& sm, int ys_mul = 1, int ysub = 0) {
  typedef typename WT<T, MODE>::type W;
  const i64 nx = p.nx, ny = p.ny, nz = p.nz;
  const i64 sz = nx * ny;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const i64 bx0 = (i64)blockIdx.x * (BX * V);
  const i64 by0 = ((i64)blockIdx.y * ys_mul + ysub) * BY;  // a CTA may cover ys_mul tiles of BY rows
  const i64 x0 = bx0 + (i64)tx * V;
  const i64 y = by0 + ty;
  const bool act = (x0 < nx) && (y < ny);
  const i64 cz0 = (i64)blockIdx.z * zc;
  const i64 cz1 = (cz0 + zc < nz) ? cz0 + zc : nz;
  const T* urow = u + y * nx + x0;
  T* vrow = v + y * nx + x0;

  // Boundary planes are copied by the chunk that holds them.
  if (act && cz0 == 0) { T t[V]; ldv<T, V>(urow, t); stv<T, V>(vrow, t); }
  if (act && cz1 == nz) { T t[V]; ldv<T, V>(urow + (nz - 1) * sz, t); stv<T, V>(vrow + (nz - 1) * sz, t); }
  const i64 z0 = cz0 < 1 ? 1 : cz0;
  const i64 z1 = cz1 > nz - 1 ? nz - 1 : cz1;
  if (z0 >= z1) return;  // block-uniform

  const bool yint = (y >= 1) && (y <= ny - 2);
  T rcur[V], rzn[V], rzn2[V];
  W zp[V], cur[V], zn[V];
  {
    T t[V];
#pragma unroll
    for (int e = 0; e < V; ++e) t[e] = rcur[e] = rzn[e] = rzn2[e] = T(0);
    if (act) {
      ldv<T, V>(urow + (z0 - 1) * sz, t);
      ldv<T, V>(urow + z0 * sz, rcur);
      ldv<T, V>(urow + (z0 + 1) * sz, rzn);
      if (z0 + 2 < nz) ldv<T, V>(urow + (z0 + 2) * sz, rzn2);
    }
#pragma unroll
    for (int e = 0; e < V; ++e) { zp[e] = cvt_in<T, MODE>(t[e], F); cur[e] = cvt_in<T, MODE>(rcur[e], F); }
  }
  HaloFetch<T, BX, BY, V> h, hn;
  fetch_halo<T, BX, BY, V>(u, p, z0, bx0, by0, false, h);
  hn = h;
  int b = 0;
  for (i64 z = z0; z < z1; ++z) {
#pragma unroll
    for (int e = 0; e < V; ++e) zn[e] = cvt_in<T, MODE>(rzn[e], F);
    T rn3[V];
#pragma unroll
    for (int e = 0; e < V; ++e) rn3[e] = T(0);
    if (act && z + 3 < nz) ldv<T, V>(urow + (z + 3) * sz, rn3);
    if (z + 1 < z1) fetch_halo<T, BX, BY, V>(u, p, z + 1, bx0, by0, false, hn);

    put_plane<T, BX, BY, V, MODE>(sm, b, cur, h, F);
    __syncthreads();
    const W* rm = &sm.a[b][ty][V + tx * V];
    const W* r0 = &sm.a[b][ty + 1][V + tx * V];
    const W* rp = &sm.a[b][ty + 2][V + tx * V];
    T out[V];
#pragma unroll
    for (int e = 0; e < V; ++e) {
      const i64 x = x0 + e;
      const bool in = act && yint && (x >= 1) && (x <= nx - 2);
      const W xl = (e == 0) ? r0[-1] : cur[e - 1];
      const W xr = (e == V - 1) ? r0[V] : cur[e + 1];
      const W s = ((xl + xr) + (rm[e] + rp[e])) + (zp[e] + zn[e]);
      {
        const T r = (T)p.c0;
        const T o = cur[e] + r * (s - T(6) * cur[e]);
        out[e] = in ? o : rcur[e];
        T d = o - cur[e];
        d = d < T(0) ? -d : d;
        if (in && d > rmax) rmax = d;
      }
    }
    if (act) stv<T, V>(vrow + z * sz, out);
#pragma unroll
    for (int e = 0; e < V; ++e) {
      zp[e] = cur[e];
      cur[e] = zn[e];
      rcur[e] = rzn[e];
      rzn[e] = rzn2[e];
      rzn2[e] = rn3[e];
    }
    h = hn;
    b ^= 1;
  }
}

// r = fb 2^-k with 1 <= k <= 4 and fb <= 2 (r = 1/8, 1/16, ...): the
// constant-folded staged heat kernels form v 2^F directly as
// (fb S + (2^k - 6 fb) c + 2^(k-1)) >> k, which equals c + round(r L 2^F) bit
// for bit (2^k c is a multiple of 2^k); every term stays below 2^62 for
// |c| < 2^57 and |S| < 6 * 2^57.  (Every fixed-point heat kernel takes its
// residual from the increment v - c, so this changes no result.)
template <class P> JD bool heat_fold(const P& p) {
  return p.fpath == JACC_FP_SMALL && p.fk >= 1 && p.fk <= 4 && p.fb >= 1 && p.fb <= 2;
}


// Sum accumulator: FP64 for FP64 data; an FP32 error-free (hi, lo) pair for
// FP32 data, combined in FP64 once per thread.
template <class T> struct SumAcc {
  double d = 0.0;
  JD void add(T x) { d += (double)x; }
  JD double total() const { return d; }
};
template <> struct SumAcc<float> {
  float hi = 0.0f, lo = 0.0f;
  JD void add(float x) { two_sum_acc(hi, lo, x); }
  JD double total() const { return (double)hi + (double)lo; }
};

// ---------------------------------------------------------------- 27-point periodic box, native arithmetic
//
// All periodic offsets are computed once per thread (no division in the
// plane loop); plane z+2 is fetched into registers one iteration ahead and
// stored to shared memory the next.  Row reads from shared memory use 16-byte
// vectors for the thread's own V columns.

template <class W, int V> JD void lds_row(const W* p, W (&r)[V + 2]) {
  r[0] = p[-1];
  if constexpr (V * sizeof(W) == 16 && V == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    r[1] = t.x; r[2] = t.y; r[3] = t.z; r[4] = t.w;
  } else if constexpr (V * sizeof(W) == 16 && V == 2) {
    const double2 t = *reinterpret_cast<const double2*>(p);
    r[1] = t.x; r[2] = t.y;
  } else {
#pragma unroll
    for (int e = 0; e < V; ++e) r[e + 1] = p[e];
  }
  r[V + 1] = p[V];
}

// Stores a thread's V values to a shared-memory row as one 16-byte vector
// where the width allows.
template <class W, int V> JD void sts_row(W* p, const W (&r)[V]) {
  if constexpr (V * sizeof(W) == 16 && V == 4) {
    float4 t;
    t.x = r[0]; t.y = r[1]; t.z = r[2]; t.w = r[3];
    *reinterpret_cast<float4*>(p) = t;
  } else if constexpr (V * sizeof(W) == 16 && V == 2) {
    double2 t;
    t.x = r[0]; t.y = r[1];
    *reinterpret_cast<double2*>(p) = t;
  } else {
#pragma unroll
    for (int e = 0; e < V; ++e) p[e] = r[e];
  }
}

template <class T, int BX, int BY, int V>
struct Box27Fetch {
  T own[V], hrow[V], hx, cr[4];
};

template <class T, int BX, int BY, int V, class P>
JD void box27_body2(const T* __restrict__ u, T* __restrict__ v, const P& p, int zc, SumAcc<T>& acc, bool want_sum,
                    Plane<T, BX, BY, V>& sm, int ys_mul = 1, int ysub = 0) {
  const i64 nx = p.nx, ny = p.ny, nz = p.nz;
  const i64 sz = nx * ny;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const i64 bx0 = (i64)blockIdx.x * (BX * V);
  const i64 by0 = ((i64)blockIdx.y * ys_mul + ysub) * BY;  // a CTA may cover ys_mul tiles of BY rows
  const i64 x0 = bx0 + (i64)tx * V;
  const i64 y = by0 + ty;
  const bool act = (x0 < nx) && (y < ny);
  const i64 z0 = (i64)blockIdx.z * zc;
  const i64 z1 = (z0 + zc < nz) ? z0 + zc : nz;
  // periodic images, once per thread (threads overhanging the grid use them too)
  const i64 xo = x0 % nx, yo = y % ny;
  const i64 own_off = yo * nx + xo;
  const bool hy = (ty == 0) || (ty == BY - 1);
  const i64 hy_off = ((ty == 0) ? (by0 - 1 + ny) % ny : (by0 + BY) % ny) * nx + xo;
  const bool hx = (tx == 0) || (tx == BX - 1);
  const i64 hx_off = yo * nx + ((tx == 0) ? (bx0 - 1 + nx) % nx : (bx0 + BX * V) % nx);
  const bool corner = (tx == 0) && (ty == 0);
  i64 c_off[4] = {0, 0, 0, 0};
  if (corner) {
    const i64 xl = (bx0 - 1 + nx) % nx, xr = (bx0 + BX * V) % nx;
    const i64 yt = (by0 - 1 + ny) % ny, yb = (by0 + BY) % ny;
    c_off[0] = yt * nx + xl;
    c_off[1] = yt * nx + xr;
    c_off[2] = yb * nx + xl;
    c_off[3] = yb * nx + xr;
  }
  auto fetch = [&](i64 zoff, Box27Fetch<T, BX, BY, V>& f) {
    const T* pl = u + zoff;
    ldv<T, V>(pl + own_off, f.own);
    if (hy) ldv<T, V>(pl + hy_off, f.hrow);
    if (hx) f.hx = __ldg(pl + hx_off);
    if (corner) {
#pragma unroll
      for (int k = 0; k < 4; ++k) f.cr[k] = __ldg(pl + c_off[k]);
    }
  };
  auto put = [&](const Box27Fetch<T, BX, BY, V>& f, int b) {
    sts_row<T, V>(&sm.a[b][ty + 1][V + tx * V], f.own);
    if (hy) sts_row<T, V>(&sm.a[b][ty == 0 ? 0 : BY + 1][V + tx * V], f.hrow);
    if (tx == 0) sm.a[b][ty + 1][V - 1] = f.hx;
    if (tx == BX - 1) sm.a[b][ty + 1][V + BX * V] = f.hx;
    if (corner) {
      sm.a[b][0][V - 1] = f.cr[0];
      sm.a[b][0][V + BX * V] = f.cr[1];
      sm.a[b][BY + 1][V - 1] = f.cr[2];
      sm.a[b][BY + 1][V + BX * V] = f.cr[3];
    }
  };
  auto cfe = [&](int b, T (&c)[V], T (&f)[V], T (&g)[V]) {
    T m[V + 2], zz[V + 2], q[V + 2];
    lds_row<T, V>(&sm.a[b][ty][V + tx * V], m);
    lds_row<T, V>(&sm.a[b][ty + 1][V + tx * V], zz);
    lds_row<T, V>(&sm.a[b][ty + 2][V + tx * V], q);
#pragma unroll
    for (int e = 0; e < V; ++e) {
      c[e] = zz[e + 1];
      f[e] = (zz[e] + zz[e + 2]) + (m[e + 1] + q[e + 1]);
      g[e] = (m[e] + m[e + 2]) + (q[e] + q[e + 2]);
    }
  };
  auto next_plane = [&](i64 zi) { return zi + 1 == nz ? (i64)0 : zi + 1; };

  const T w0 = (T)p.c0, wf = (T)p.c1, we = (T)p.c2, wc = (T)p.c3;
  T cm[V], fm[V], gm[V], c0[V], f0[V], g0[V];
  Box27Fetch<T, BX, BY, V> fa, fb;
  i64 zi = (z0 - 1 + nz) % nz;  // plane z0 - 1
  fetch(zi * sz, fa);
  zi = next_plane(zi);           // plane z0
  fetch(zi * sz, fb);
  put(fa, 0);
  __syncthreads();
  cfe(0, cm, fm, gm);
  put(fb, 1);
  zi = next_plane(zi);           // plane z0 + 1
  fetch(zi * sz, fa);
  __syncthreads();
  cfe(1, c0, f0, g0);
  int b = 0;
  for (i64 z = z0; z < z1; ++z) {
    put(fa, b);                   // plane z + 1
    if (z + 1 < z1) {
      zi = next_plane(zi);        // plane z + 2, one iteration ahead
      fetch(zi * sz, fa);
    }
    __syncthreads();
    T cn[V], fn[V], gn[V];
    cfe(b, cn, fn, gn);
    T out[V];
#pragma unroll
    for (int e = 0; e < V; ++e)
      out[e] = (w0 * c0[e] + wf * ((f0[e] + cm[e]) + cn[e])) + (we * ((g0[e] + fm[e]) + fn[e]) + wc * (gm[e] + gn[e]));
    if (act) {
      stv<T, V>(v + z * sz + y * nx + x0, out);
      if (want_sum) {
#pragma unroll
        for (int e = 0; e < V; ++e) acc.add(out[e]);
      }
    }
#pragma unroll
    for (int e = 0; e < V; ++e) {
      cm[e] = c0[e]; fm[e] = f0[e]; gm[e] = g0[e];
      c0[e] = cn[e]; f0[e] = fn[e]; g0[e] = gn[e];
    }
    b ^= 1;
  }
}

// ---------------------------------------------------------------- bulk-copy staged planes
//
// Plane staging with the bulk-copy engine: cp.async.bulk copies rows of the
// input field from global to shared memory and counts the bytes that landed
// on an mbarrier of the stage ("full"); no register holds data in flight, so
// a CTA keeps up to S planes outstanding at no register cost.  Each stage
// also has an "empty" mbarrier on which every warp arrives once it has read
// the stage; warp 0 waits on it before it reuses the stage.  Every wait gives
// up after JParams::timeout_ns (%globaltimer), records JACC_DEV_TIMEOUT and
// lets the CTA finish; before it returns, warp 0 waits (bounded too) for the
// copies it has issued, so no copy targets the shared memory of a CTA that
// has exited.

JD u32 smem_u32(const void* ptr) { return (u32)__cvta_generic_to_shared(ptr); }
JD u64 gtimer_ns() {
  u64 t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
JD void mbar_init(u64* bar, u32 count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
JD void mbar_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
JD void mbar_expect_tx(u64* bar, u32 bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
JD void mbar_arrive(u64* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
JD bool mbar_try(u64* bar, u32 parity) {
  u32 done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done != 0;
}
// try_wait that may suspend the thread for up to `hint_ns` until the phase
// completes, so waiting warps take no issue slots.
JD bool mbar_try_suspend(u64* bar, u32 parity, u32 hint_ns) {
  u32 done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity), "r"(hint_ns)
      : "memory");
  return done != 0;
}
// Waits for the completion of the phase with the given parity; false after
// limit_ns without it.
JD bool mbar_wait(u64* bar, u32 parity, i64 limit_ns) {
  if (mbar_try(bar, parity)) return true;
  const u64 t0 = gtimer_ns();
  while (!mbar_try_suspend(bar, parity, 200000u))
    if ((i64)(gtimer_ns() - t0) > limit_ns) return false;
  return true;
}
// One bulk copy global -> shared (16-byte aligned addresses, size a multiple
// of 16), completion counted in bytes on `bar`.
JD void bulk_g2s(void* dst, const void* src, u32 bytes, u64* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// ---------------------------------------------------------------- planes staged by asynchronous copies
//
// A second way of staging planes, for the kernels whose rows need not start
// on 16-byte boundaries or whose staged values are converted in place: every
// thread copies its share of a plane (the tile with a one-point halo) with
// cp.async, CH elements per copy, into a ring of S stages in shared memory;
// one group per plane, one CTA barrier per plane.  A copy's source may be any
// element (8- or 4-byte copies for CH = 1), so odd rows, periodic images and
// clipped edges all come from a per-thread list of source offsets worked out
// once, and the thread that copied an element may convert it before the
// barrier that publishes the plane.
//
// Geometry: BX x BY threads; a thread owns V consecutive columns of RY
// consecutive rows: one column, so a warp reads and writes whole rows (no bank
// conflicts, coalesced stores at any alignment), or one 16-byte column of two
// rows.  The y neighbours inside its rows stay in registers.  A stage holds
// R x W elements in rows of W = BX V + 2 CH: column x of the tile sits at slot
// x - bx0 + CH of row y - by0 + 1.
template <class T, int BX, int BY, int CH, int V = 1> struct RingG {
  static constexpr int NT = BX * BY;
  static constexpr int RY = V > 1 ? 2 : JACC_RING_ROWS(BX, BY);
  static constexpr int TW = BX * V, TH = BY * RY;
  static constexpr int W = TW + 2 * CH, R = TH + 2;
  static constexpr int STAGE = W * R;                       // elements
  static constexpr int NCH = W / CH, NTOT = NCH * R;        // copies per row, per plane
  static constexpr int PER = (NTOT + NT - 1) / NT;          // copies per thread
  static constexpr int S0 = 46080 / (STAGE * (int)sizeof(T));
  // Stages: what 45 KB hold, but 3 at least (the march needs that many) and 6 at
  // most.  The widest tiles, FP64 of 64 x 8 and 128 x 4 threads with 16-byte
  // columns, take 57024 and 62400 bytes so.
  static constexpr int S = S0 < 3 ? 3 : (S0 > 6 ? 6 : S0);
  static_assert(S * STAGE * (int)sizeof(T) <= 62400, "static shared memory of a CTA");
};

template <int BYTES> JD void cpa_copy(void* dst, const void* src) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(dst)), "l"(src), "n"(BYTES) : "memory");
}
JD void cpa_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> JD void cpa_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// A thread's share of every staged plane: copy i moves the CH elements at
// offset off[i] of the plane to stage element (tid + i NT) CH; bit i of
// `mask` is clear where there is none (past the plane, or outside a Dirichlet
// grid, whose slots are never used).
template <class T, int BX, int BY, int CH, int V = 1> struct RingPlan {
  typedef RingG<T, BX, BY, CH, V> G;
  i64 off[G::PER];
  u32 mask;
  JD void init(i64 nx, i64 ny, i64 bx0, i64 by0, bool periodic) {
    const int tid = threadIdx.y * BX + threadIdx.x;
    mask = 0;
#pragma unroll
    for (int i = 0; i < G::PER; ++i) {
      const int c = tid + i * G::NT;
      i64 x = bx0 - CH + (c % G::NCH) * CH, y = by0 - 1 + c / G::NCH;
      bool ok = c < G::NTOT;
      if (periodic) {
        x = (x + nx) % nx;
        y = (y + ny) % ny;
      } else {
        ok = ok && x >= 0 && x < nx && y >= 0 && y < ny;
      }
      off[i] = ok ? y * nx + x : 0;
      mask |= (u32)ok << i;
    }
  }
  JD void issue(T* stage, const T* plane) const {
    const int tid = threadIdx.y * BX + threadIdx.x;
#pragma unroll
    for (int i = 0; i < G::PER; ++i)
      if ((mask >> i) & 1u) cpa_copy<CH * (int)sizeof(T)>(stage + (tid + i * G::NT) * CH, plane + off[i]);
  }
};

// Geometry of the staged 27-point FP32 kernel: BX x BY threads, each owning 4
// consecutive columns (one 16-byte vector) of 2 consecutive rows, so a CTA
// computes a TW x TH tile per plane.  A stage holds R = TH + 2 rows of
// W = TW + 8 floats: slot i of staged row r is column (bx0 - 4 + i) mod nx of
// row (by0 - 1 + r) mod ny (the periodic images, so halo columns and rows need
// no special case).  The halo is 4 columns wide on each side because bulk
// copies move whole 16-byte units; columns bx0 - 1 and bx0 + TW are used.
template <int BX, int BY> struct Box27S {
  static constexpr int RY = 2;
  static constexpr int TW = BX * 4, TH = BY * RY;
  static constexpr int W = TW + 8, R = TH + 2;
  static constexpr int STAGE_BYTES = W * R * 4;
  static constexpr int S0 = 40960 / STAGE_BYTES;
  static constexpr int S = S0 < 2 ? 2 : (S0 > 4 ? 4 : S0);  // stages, 2..4, at most ~40 KB
  static constexpr int NW = BX * BY / 32;
};

template <int BX, int BY> struct alignas(128) Box27SSmem {
  float st[Box27S<BX, BY>::S][Box27S<BX, BY>::R][Box27S<BX, BY>::W];
  u64 full[Box27S<BX, BY>::S];
  u64 empty[Box27S<BX, BY>::S];
};

// What lane r of warp 0 copies of every staged plane: staged row r, as one bulk
// copy, or as two or more where the row's slots wrap around the periodic x
// boundary.
struct Box27Row {
  i64 row;  // offset of the row in its plane
  i64 c;    // first column
};

// Whether a CTA works its rows and planes out once and carries them (every
// thread holds the registers, though only warp 0's lanes use them), or for
// every request.  Folded kernels know that a staged row wraps once at most
// (ny >= R): a comparison or two per request, and 64 registers, 8 CTAs an SM,
// instead of 72 and 7 (32 x 4 threads, us a sweep carried / not: 1024^3 1309 /
// 1294, 768^3 577 / 573, 512^3 196 / 190, 800 x 900 x 1000 1014 / 976).
// Precompiled ones would divide: 1024^3 1468 carried, 1565 not.
template <class P, int R, bool FOLDED = Folded<P>::value> struct Box27Carry { static constexpr bool value = true; };
template <class P, int R> struct Box27Carry<P, R, true> { static constexpr bool value = P::ny < R; };

// Warp 0 requests a plane into stage s: lane 0 posts the byte count, then each
// lane copies its row.
template <int BX, int BY>
JD void box27s_issue(Box27SSmem<BX, BY>& sm, int s, const float* __restrict__ plane, const Box27Row& q, i64 nx, int weff) {
  typedef Box27S<BX, BY> G;
  const int lane = threadIdx.x & 31;
  if (lane == 0) mbar_expect_tx(&sm.full[s], (u32)(G::R * weff * 4));
  __syncwarp();
  if (lane < G::R) {
    const float* row = plane + q.row;
    float* dst = &sm.st[s][lane][0];
    i64 c = q.c;
    int i = 0;
    while (i < weff) {
      i64 len = nx - c;
      if (len > weff - i) len = weff - i;
      bulk_g2s(dst + i, row + c, (u32)(len * 4), &sm.full[s]);
      i += (int)len;
      c = 0;
    }
  }
}

// One staged plane -> the per-point plane terms of the thread's 2 x 4 points:
// A = wf c + we f + wc g (the plane's contribution as an upper or lower
// neighbour plane) and B = w0 c + wf f + we g (as the centre plane), where c
// is the point, f the sum of its 4 in-plane face neighbours and g of its 4
// in-plane diagonal neighbours.  Row sums r[x-1] + r[x+1] are shared by the
// two output rows.
template <int BX, int BY>
JD void box27s_terms(const float (*st)[Box27S<BX, BY>::W], float w0, float wf, float we, float wc, float (&A)[2][4],
                     float (&B)[2][4]) {
  const int tx = threadIdx.x, ty = threadIdx.y;
  float r[4][6];
#pragma unroll
  for (int k = 0; k < 4; ++k) lds_row<float, 4>(&st[2 * ty + k][4 + 4 * tx], r[k]);
  float s[4][4];
#pragma unroll
  for (int k = 0; k < 4; ++k)
#pragma unroll
    for (int e = 0; e < 4; ++e) s[k][e] = r[k][e] + r[k][e + 2];
#pragma unroll
  for (int yy = 0; yy < 2; ++yy)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float c = r[yy + 1][e + 1];
      const float f = s[yy + 1][e] + (r[yy][e + 1] + r[yy + 2][e + 1]);
      const float g = s[yy][e] + s[yy + 2][e];
      A[yy][e] = fmaf(wc, g, fmaf(we, f, wf * c));
      B[yy][e] = fmaf(we, g, fmaf(wf, f, w0 * c));
    }
}

// The staged periodic 27-point FP32 sweep of one CTA tile: planes z0-1 ..
// z1 are staged (L = z1 - z0 + 2), output plane z = A(z-1) + B(z) + A(z+1)
// is formed as P + A(z+1) with P = A(z-1) + B(z) kept in registers.  Returns
// the thread's double-float sum of its outputs (want_sum).
template <int BX, int BY, bool BULK, class P>
JD double box27s_body(const float* __restrict__ u, float* __restrict__ v, const P& p, const JParams& rt,
                      bool want_sum) {
  typedef Box27S<BX, BY> G;
  typedef RingG<float, BX, BY, 4, 4> R;  // the same stage layout
  static_assert(R::W == G::W && R::R == G::R, "one stage layout for both ways of staging");
  __shared__ __align__(128) unsigned char raw[BULK ? sizeof(Box27SSmem<BX, BY>) : sizeof(float) * R::S * R::STAGE];
  Box27SSmem<BX, BY>& sm = *reinterpret_cast<Box27SSmem<BX, BY>*>(raw);  // BULK
  float* ring = reinterpret_cast<float*>(raw);                           // otherwise
  const i64 nx = p.nx, ny = p.ny, nz = p.nz, sz = nx * ny;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int tid = ty * BX + tx;
  const bool warp0 = tid < 32;
  const i64 bx0 = (i64)blockIdx.x * G::TW, by0 = (i64)blockIdx.y * G::TH;
  const i64 z0 = (i64)blockIdx.z * p.zc;
  const i64 z1 = (z0 + p.zc < nz) ? z0 + p.zc : nz;
  const int L = (int)(z1 - z0) + 2;
  const int weff = (int)((nx - bx0 < G::TW) ? nx - bx0 : G::TW) + 8;
  const i64 lim = rt.timeout_ns;
  const bool stall_cta = rt.stall_plane >= 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0;
  if constexpr (BULK) {
    if (tid == 0) {
#pragma unroll
      for (int s = 0; s < G::S; ++s) {
        mbar_init(&sm.full[s], 1);
        mbar_init(&sm.empty[s], G::NW);
      }
      mbar_init_fence();
    }
    __syncthreads();
  }
  static_assert(G::R <= 32, "one staged row per lane of warp 0");
  constexpr bool CARRY = Box27Carry<P, G::R>::value;
  Box27Row lrow;
  if constexpr (CARRY) lrow.row = ((by0 - 1 + (tid & 31) + ny) % ny) * nx;
  lrow.c = bx0 >= 4 ? bx0 - 4 : bx0 - 4 + nx;
  i64 zi = z0 == 0 ? nz - 1 : z0 - 1;  // the next plane to request
  auto request = [&](int j, int s) {
    if constexpr (!CARRY) {  // staged rows -1 .. ny + TH and planes -1 .. nz: one wrap at most
      const i64 y = by0 - 1 + (tid & 31);
      lrow.row = (y < 0 ? y + ny : (y >= ny ? y - ny : y)) * nx;
      zi = z0 - 1 + j;
      zi = zi < 0 ? zi + nz : (zi >= nz ? zi - nz : zi);
    }
    if (!(stall_cta && j == rt.stall_plane)) box27s_issue<BX, BY>(sm, s, u + zi * sz, lrow, nx, weff);
    if constexpr (CARRY) zi = zi + 1 == nz ? 0 : zi + 1;
  };
  int issued = 0, consumed = 0;  // warp 0: planes requested, planes waited for
  RingPlan<float, BX, BY, 4, 4> plan;
  int is = 0, cs = 0;  // asynchronous copies: stages to fill and to read, in elements
  auto copy_next = [&]() {
    if (issued < L) plan.issue(ring + is, u + zi * sz);
    cpa_commit();
    ++issued;
    zi = zi + 1 == nz ? 0 : zi + 1;
    is = is + R::STAGE == R::S * R::STAGE ? 0 : is + R::STAGE;
  };
  if constexpr (BULK) {
    if (warp0)
      for (; issued < G::S && issued < L; ++issued) request(issued, issued);
  } else {
    plan.init(nx, ny, bx0, by0, true);
#pragma unroll 1
    for (int j = 0; j < R::S - 1; ++j) copy_next();
  }

  const float w0 = (float)p.c0, wf = (float)p.c1, we = (float)p.c2, wc = (float)p.c3;
  const i64 x0 = bx0 + 4 * tx, y0 = by0 + 2 * ty;
  const bool ax = x0 < nx, ay0 = ax && y0 < ny, ay1 = ax && y0 + 1 < ny;
  float* vo = v + y0 * nx + x0 + z0 * sz;
  float hi = 0.0f, lo = 0.0f;
  // ring cursors (stage, phase parity): cn the next plane to wait for, cq
  // the plane whose stage warp 0 refills next (one step behind)
  int cn_s = 0, cq_s = 0;
  u32 cn_ph = 0, cq_ph = 0;
  auto adv = [&](int& s, u32& ph) {
    if (++s == G::S) {
      s = 0;
      ph ^= 1u;
    }
  };
  // consume plane j: wait for it, form its terms, release its stage, and let
  // warp 0 refill the stage of plane j - 1
  auto consume = [&](int j, float (&A)[2][4], float (&B)[2][4]) -> bool {
    if constexpr (!BULK) {
      cpa_wait<R::S - 2>();
      __syncthreads();
      copy_next();  // into the stage read before the barrier
      box27s_terms<BX, BY>(reinterpret_cast<const float(*)[G::W]>(ring + cs), w0, wf, we, wc, A, B);
      cs = cs + R::STAGE == R::S * R::STAGE ? 0 : cs + R::STAGE;
      return true;
    }
    if (!mbar_wait(&sm.full[cn_s], cn_ph, lim)) return false;
    ++consumed;
    box27s_terms<BX, BY>(sm.st[cn_s], w0, wf, we, wc, A, B);
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(&sm.empty[cn_s]);
    adv(cn_s, cn_ph);
    if (j >= 1) {
      if (warp0 && issued < L) {
        if (!mbar_wait(&sm.empty[cq_s], cq_ph, lim)) return false;
        request(issued, cq_s);
        ++issued;
      }
      adv(cq_s, cq_ph);
    }
    return true;
  };
  // output plane of staged plane j - 1 from P = A(j-2) + B(j-1) and the
  // terms of plane j; Anew receives A(j), Aold holds A(j-1)
  float Pz[2][4];
  auto step = [&](int j, float (&Anew)[2][4], const float (&Aold)[2][4]) -> bool {
    float B[2][4];
    if (!consume(j, Anew, B)) return false;
    float o[2][4];
#pragma unroll
    for (int yy = 0; yy < 2; ++yy)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        o[yy][e] = Pz[yy][e] + Anew[yy][e];
        Pz[yy][e] = Aold[yy][e] + B[yy][e];
      }
    if (ay0) stv<float, 4>(vo, o[0]);
    if (ay1) stv<float, 4>(vo + nx, o[1]);
    vo += sz;
    if (want_sum) {
      const float t0 = ay0 ? (o[0][0] + o[0][1]) + (o[0][2] + o[0][3]) : 0.0f;
      const float t1 = ay1 ? (o[1][0] + o[1][1]) + (o[1][2] + o[1][3]) : 0.0f;
      two_sum_acc(hi, lo, t0 + t1);
    }
    return true;
  };
  float Aa[2][4], Ab[2][4];
  bool ok;
  {
    float B[2][4];
    ok = consume(0, Aa, B) && consume(1, Ab, B);  // A of planes 0 and 1; B of plane 1
    if (ok) {
#pragma unroll
      for (int yy = 0; yy < 2; ++yy)
#pragma unroll
        for (int e = 0; e < 4; ++e) Pz[yy][e] = Aa[yy][e] + B[yy][e];
    }
  }
  if (ok) {
    // two steps per iteration: the A buffers swap roles without copies
    int j = 2;
    for (; j + 1 < L; j += 2) {
      if (!step(j, Aa, Ab) || !step(j + 1, Ab, Aa)) {
        ok = false;
        break;
      }
    }
    if (ok && j < L) ok = step(j, Aa, Ab);
  }
  if (!ok) {
    if (rt.status) atomicExch(rt.status, JACC_DEV_TIMEOUT);
    if (warp0)
      for (int j = consumed; j < issued; ++j)
        if (!(stall_cta && j == rt.stall_plane)) mbar_wait(&sm.full[j % G::S], (u32)((j / G::S) & 1), lim);
  }
  return (double)hi + (double)lo;
}

// ---------------------------------------------------------------- 27-point periodic box, temporal blocking (FP32)
//
// TT sweeps per launch.  A CTA of 32 x RY threads (4 floats each in x) loads
// an input region of 128 x RY points per plane: an output tile of 120 x
// (RY - 2 TT) points plus a halo of 4 columns (16-byte alignment) and TT rows
// on each side.  Planes stream in z; stage t (1..TT) computes sweep t for the
// plane t steps behind the input, from the three newest planes of stage t-1,
// over the region shrunk by t (values beyond it are never used).  Each stage's
// newest plane sits in shared memory, one 16-byte vector per thread and row;
// x-neighbours come from warp shuffles (a warp is one region row).  Only the
// last stage's plane is written to memory, so HBM traffic is 8/TT bytes per
// point-sweep.
constexpr int TB_BX = 32, TB_V = 4, TB_RX = TB_BX * TB_V, TB_HX = 4, TB_OX = TB_RX - 2 * TB_HX;

template <int RY> struct alignas(16) TbPlane {
  float a[RY + 2][TB_RX + 8];  // row r + 1, column c + 4 holds region point (c, r)
};

template <int RY> JD void tb_cfe(const TbPlane<RY>& sm, float (&c)[4], float (&f)[4], float (&g)[4]) {
  const int tx = threadIdx.x, ty = threadIdx.y;
  float r[3][6];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const float4 t = *reinterpret_cast<const float4*>(&sm.a[ty + k][4 + tx * 4]);
    r[k][1] = t.x; r[k][2] = t.y; r[k][3] = t.z; r[k][4] = t.w;
    r[k][0] = __shfl_up_sync(0xffffffffu, t.w, 1);
    r[k][5] = __shfl_down_sync(0xffffffffu, t.x, 1);
  }
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    c[e] = r[1][e + 1];
    f[e] = (r[1][e] + r[1][e + 2]) + (r[0][e + 1] + r[2][e + 1]);
    g[e] = (r[0][e] + r[0][e + 2]) + (r[2][e] + r[2][e + 2]);
  }
}

template <int RY> JD void tb_put(TbPlane<RY>& sm, const float (&o)[4]) {
  float4 t;
  t.x = o[0]; t.y = o[1]; t.z = o[2]; t.w = o[3];
  *reinterpret_cast<float4*>(&sm.a[threadIdx.y + 1][4 + threadIdx.x * 4]) = t;
}

template <int RY, int TT, int ZC, class P>
JD void box27_tb_body(const float* __restrict__ u, float* __restrict__ v, const P& p, SumAcc<float>& acc,
                      bool want_sum, TbPlane<RY> (&sm)[TT]) {
  const i64 nx = p.nx, ny = p.ny, nz = p.nz;
  const i64 sz = nx * ny;
  const int tx = threadIdx.x, ty = threadIdx.y;
  constexpr int OY = RY - 2 * TT;
  const i64 ox0 = (i64)blockIdx.x * TB_OX;
  const i64 oy0 = (i64)blockIdx.y * OY;
  const i64 z0 = (i64)blockIdx.z * ZC;
  const i64 z1 = (z0 + ZC < nz) ? z0 + ZC : nz;
  // this thread's 4 region columns and region row, wrapped once
  const i64 gx = ((ox0 - TB_HX + (i64)tx * 4) % nx + nx) % nx;
  const i64 gy = ((oy0 - TT + ty) % ny + ny) % ny;
  const i64 own = gy * nx + gx;
  // output: threads 1..30 hold the tile's 120 columns, rows TT..RY-TT-1
  const i64 outx = ox0 + (i64)(tx - 1) * 4;
  const i64 outy = oy0 + ty - TT;
  const bool out_ok = tx >= 1 && tx <= TB_BX - 2 && ty >= TT && ty < RY - TT && outx < nx && outy < ny;
  const float w0 = (float)p.c0, wf = (float)p.c1, we = (float)p.c2, wc = (float)p.c3;

  float cm[TT][4], fm[TT][4], gm[TT][4], c0[TT][4], f0[TT][4], g0[TT][4];
#pragma unroll
  for (int t = 0; t < TT; ++t)
#pragma unroll
    for (int e = 0; e < 4; ++e) cm[t][e] = fm[t][e] = gm[t][e] = c0[t][e] = f0[t][e] = g0[t][e] = 0.f;

  const i64 zs = z0 - TT;  // first input plane
  i64 zi = ((zs - 1) % nz + nz) % nz;
  const int nsteps = (int)(z1 - z0) + 2 * TT;
  float nxt[4];
  zi = (zi + 1 == nz) ? 0 : zi + 1;
  ldv<float, 4>(u + zi * sz + own, nxt);
  for (int j = 0; j < nsteps; ++j) {
    float cur_in[4] = {nxt[0], nxt[1], nxt[2], nxt[3]};
    if (j + 1 < nsteps) {  // prefetch the next input plane
      zi = (zi + 1 == nz) ? 0 : zi + 1;
      ldv<float, 4>(u + zi * sz + own, nxt);
    }
    tb_put<RY>(sm[0], cur_in);
    __syncthreads();
#pragma unroll
    for (int t = 0; t < TT; ++t) {
      float cn[4], fn[4], gn[4], o[4];
      tb_cfe<RY>(sm[t], cn, fn, gn);
#pragma unroll
      for (int e = 0; e < 4; ++e)
        o[e] = (w0 * c0[t][e] + wf * ((f0[t][e] + cm[t][e]) + cn[e])) +
               (we * ((g0[t][e] + fm[t][e]) + fn[e]) + wc * (gm[t][e] + gn[e]));
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        cm[t][e] = c0[t][e]; fm[t][e] = f0[t][e]; gm[t][e] = g0[t][e];
        c0[t][e] = cn[e]; f0[t][e] = fn[e]; g0[t][e] = gn[e];
      }
      if (t + 1 < TT) {
        tb_put<RY>(sm[t + 1], o);
        __syncthreads();
      } else if (j >= 2 * TT && out_ok) {
        const i64 z = zs + j - TT;  // output plane, in [z0, z1)
        stv<float, 4>(v + z * sz + outy * nx + outx, o);
        if (want_sum) {
#pragma unroll
          for (int e = 0; e < 4; ++e) acc.add(o[e]);
        }
      }
    }
  }
}

template <int RY, int TT, int ZC, class P>
JD void box27_tb_entry(const float* __restrict__ u, float* __restrict__ v, const P& p, double* resid) {
  griddep_wait();
  __shared__ TbPlane<RY> sm[TT];
  SumAcc<float> acc;
  box27_tb_body<RY, TT, ZC>(u, v, p, acc, resid != nullptr, sm);
  block_sum_to<TB_BX * RY>(acc.total(), resid);
}

// ====================================================================== resident fixed point (FP64 data)
//
// Within one sweep sequence the field stays in 64-bit fixed point in the two
// HBM buffers (the same 8 bytes per value): the first sweep reads FP64 and
// converts, intermediate sweeps read and write the int64 values directly, and
// the last sweep writes the exact stencil value correctly rounded to FP64.
// Intermediate values are rounded once per sweep to the 2^-F grid (F >= 57 -
// e(M), finer than an FP64 ulp of M).  Dirichlet boundary points keep their
// FP64 bits in both buffers throughout (the first sweep copies them; later
// sweeps write back the bits they read), so they are converted where they
// are read as neighbours.
#define JFX_IN_F64 1   // the sweep's input interior holds FP64
#define JFX_OUT_F64 2  // the sweep writes FP64 (else int64 fixed point)

JD i64 bits_i64(double d) { return (i64)__double_as_longlong(d); }
JD double i64_bits(i64 q) { return __longlong_as_double(q); }

// (x + 2^(k-1)) >> k for a 128-bit x whose result fits in int64, k in [0, 62].
JD i64 fx128_round_shift(s128 x, int k) {
  if (k == 0) return (i64)x.lo;
  s128 h;
  h.lo = (u64)1 << (k - 1);
  h.hi = 0;
  x = add128(x, h);
  return (i64)((x.lo >> k) | (x.hi << (64 - k)));
}

// Per-thread column facts of a tile: which of the thread's V columns are
// interior (bit set) and which are boundary columns (x == 0 or nx-1).
template <int V> JD void col_masks(i64 x0, i64 nx, unsigned& intm, unsigned& bndm) {
  intm = 0;
  bndm = 0;
#pragma unroll
  for (int e = 0; e < V; ++e) {
    const i64 x = x0 + e;
    if (x >= 1 && x <= nx - 2) intm |= 1u << e;
    if (x == 0 || x == nx - 1) bndm |= 1u << e;
  }
}

// ---------------------------------------------------------------- 5-point Jacobi, resident fixed point
//
// Same march as jacobi_march.  v 2^F = (S + 2) >> 2 with S the four
// neighbours (exact); the FP64 output is fx_to(S, F + 2).  Residual: max
// |S - 4u| (scale F, converted once per thread by the caller).  EDGE as for
// the 7-point kernel: intermediate sweeps (EDGE = false) convert nothing.
template <int V, bool CG, bool EDGE>
JD void jacobi_fx_march(const double* __restrict__ u, double* __restrict__ v, i64 nx, i64 ny, i64 x0, i64 ys, i64 ye,
                        int F, int flags, u64& rmax) {
  const int lane = threadIdx.x & 31;
  const bool xin = x0 < nx;
  const bool inf = EDGE && (flags & JFX_IN_F64);
  const bool outf = EDGE && (flags & JFX_OUT_F64);
  unsigned intm, bndm;
  col_masks<V>(x0, nx, intm, bndm);
  auto cvt = [&](double raw) -> i64 { return (EDGE && inf) ? fx_from(raw, F) : bits_i64(raw); };
  auto bnd_out = [&](double raw, i64 w) -> double {
    if constexpr (!EDGE) return i64_bits(w);
    if (inf && outf) return raw;
    if (outf) return fx_to(w, F);
    return i64_bits(w);
  };
  double rup[V], rcur[V], rdn[V], rnx[V];
  i64 up[V], cur[V], dn[V];
#pragma unroll
  for (int e = 0; e < V; ++e) rup[e] = rcur[e] = rdn[e] = rnx[e] = 0.0;
  if (xin) {
    if (ys >= 1) ldv<double, V, CG>(u + (ys - 1) * nx + x0, rup);
    ldv<double, V, CG>(u + ys * nx + x0, rcur);
    if (ys + 1 < ny) ldv<double, V, CG>(u + (ys + 1) * nx + x0, rdn);
    if (ys + 2 < ny) ldv<double, V, CG>(u + (ys + 2) * nx + x0, rnx);
  }
#pragma unroll
  for (int e = 0; e < V; ++e) {
    up[e] = cvt(rup[e]);
    cur[e] = cvt(rcur[e]);
    dn[e] = cvt(rdn[e]);
  }
  for (i64 y = ys; y < ye; ++y) {
    i64 left = __shfl_up_sync(0xffffffffu, cur[V - 1], 1);
    i64 right = __shfl_down_sync(0xffffffffu, cur[0], 1);
    if (lane == 0 && xin && x0 >= 1) left = cvt(ld1<CG>(u + y * nx + x0 - 1));
    if (lane == 31 && xin && x0 + V < nx) right = cvt(ld1<CG>(u + y * nx + x0 + V));
    double rnn[V];
#pragma unroll
    for (int e = 0; e < V; ++e) rnn[e] = 0.0;
    if (xin && y + 3 < ny) ldv<double, V, CG>(u + (y + 3) * nx + x0, rnn);
    const bool yint = (y >= 1) && (y <= ny - 2);
    double out[V];
#pragma unroll
    for (int e = 0; e < V; ++e) {
      const i64 xl = (e == 0) ? left : cur[e - 1];
      const i64 xr = (e == V - 1) ? right : cur[e + 1];
      const bool in = yint && ((intm >> e) & 1u);
      const i64 s = (up[e] + dn[e]) + (xl + xr);
      const double o = outf ? fx_to(s, F + 2) : i64_bits((s + 2) >> 2);
      out[e] = in ? o : bnd_out(rcur[e], cur[e]);
      const i64 d = s - cur[e] * 4;
      const u64 ad = (u64)(d ^ (d >> 63));  // |d| (one less for negative d: below the tolerance by 2^-F)
      if (in && ad > rmax) rmax = ad;
    }
    if (xin) stv<double, V>(v + y * nx + x0, out);
#pragma unroll
    for (int e = 0; e < V; ++e) {
      up[e] = cur[e];
      cur[e] = dn[e];
      rcur[e] = rdn[e];
      rdn[e] = rnx[e];
      dn[e] = cvt(rnx[e]);
      rnx[e] = rnn[e];
    }
  }
}

// The residual maximum of N increments: |d| as d ^ (d >> 63) (one less if
// negative).  Its high word is at least the running maximum's only if some
// high word of d lies outside (~t, t), so a plane usually costs two 32-bit
// compares a point instead of a 64-bit magnitude, compare and select.
template <int N> JD void fx_residual(const i64 (&d)[N], u64& rmax) {
  int hi = (int)(d[0] >> 32), lo = hi;
#pragma unroll
  for (int k = 1; k < N; ++k) {
    hi = max(hi, (int)(d[k] >> 32));
    lo = min(lo, (int)(d[k] >> 32));
  }
  const int t = (int)(rmax >> 32);
  if (hi >= t || lo <= ~t) {
#pragma unroll
    for (int k = 0; k < N; ++k) {
      const u64 a = (u64)(d[k] ^ (d[k] >> 63));
      rmax = a > rmax ? a : rmax;
    }
  }
}

// ---------------------------------------------------------------- 5-point Jacobi, strip march
//
// One warp marches rows [ys, ye) of a strip of 30 V columns, V per lane:
// lanes 0 and 31 hold the columns left and right of the strip, so every x
// neighbour comes from a shuffle, with no extra loads or selects, at the
// price of 2/30 more loads and sums (L2 serves the shared columns).  Rows
// y-1, y, y+1 stay in registers and the raw rows y+2 .. y+1+D are in flight;
// D rows per iteration rotate all of them without copies.  A warp whose
// columns are all interior runs without selects.  4096^2 FP64, 50 sweeps:
// 3.52 ms with the row march of the table's vector tiles (82 thread-
// instructions a point, an edge column loaded where it is used), 2.43 here
// (5.6 TB/s; 2.55 with 64-bit row offsets multiplied out for every row, 80
// registers instead of 66), bound by the latency of the warps an SM holds.
//
// xl: the lane's first column (may lie outside the grid).  FX: resident
// 64-bit fixed point, v 2^F = (S + 2) >> 2 with S the four neighbours, the
// FP64 output fx_to(S, F + 2), the residual |S - 4u| (EDGE: conversions, see
// JFX_*); otherwise native arithmetic on T.  All lanes of a warp share ys, ye.
template <class T, int V, bool FX, bool EDGE, int D>
JD void jacobi_strip(const T* __restrict__ u, T* __restrict__ v, i64 nx, i64 ny, i64 xl, i64 ys, i64 ye, int F,
                     int flags, typename RT<T, FX ? JM_FIXED : JM_NATIVE>::type& rmax) {
  typedef typename WT<T, FX ? JM_FIXED : JM_NATIVE>::type W;
  const int lane = threadIdx.x & 31;
  const bool inf = FX && EDGE && (flags & JFX_IN_F64);
  const bool outf = FX && EDGE && (flags & JFX_OUT_F64);
  const bool xin = xl >= 0 && xl < nx;
  const bool wr = xin && lane >= 1 && lane <= 30;  // this lane writes its columns
  bool cint[V];
  bool all = true;
#pragma unroll
  for (int e = 0; e < V; ++e) {
    cint[e] = xl + e >= 1 && xl + e <= nx - 2;
    all = all && (cint[e] || lane == 0 || lane == 31);
  }
  const bool fast = __all_sync(0xffffffffu, all);
  auto cvt = [&](T raw) -> W {
    if constexpr (FX) return inf ? fx_from(raw, F) : bits_i64(raw);
    else return raw;
  };
  const T* src = u + ys * nx + xl;  // row ys of the lane's columns
  T* dst = v + ys * nx + xl;
  // row counts relative to ys fit 32 bits; the pointers advance row by row
  const int rows = (int)(ye - ys);
  // last row needed: ye, if it is in the grid
  const int rlast = xin ? (int)((ye < ny ? ye : ny - 1) - ys) : -1;
  const int jlo = ys < 1 ? 1 : 0, jhi = (int)(ny - 2 - ys < rows ? ny - 2 - ys : rows);  // interior rows
  const T* ln = src;  // next row to load
  auto load = [&](int r, T (&q)[V]) {  // row ys + r, in order
#pragma unroll
    for (int e = 0; e < V; ++e) q[e] = T(0);
    if (r <= rlast) ldv<T, V>(ln, q);
    ln += nx;
  };
  T q[D][V];
  W w[3][V];
  {
    T t[V];
#pragma unroll
    for (int e = 0; e < V; ++e) t[e] = T(0);
    if (xin && ys >= 1) ldv<T, V>(src - nx, t);
    load(0, q[0]);
#pragma unroll
    for (int e = 0; e < V; ++e) {
      w[0][e] = cvt(t[e]);
      w[1][e] = cvt(q[0][e]);
    }
#pragma unroll
    for (int k = 0; k < D; ++k) load(1 + k, q[k]);
  }
  auto step = [&](int j, const W (&up)[V], const W (&cur)[V], W (&dn)[V], T (&qn)[V]) {
#pragma unroll
    for (int e = 0; e < V; ++e) dn[e] = cvt(qn[e]);
    load(j + 1 + D, qn);
    const W left = __shfl_up_sync(0xffffffffu, cur[V - 1], 1);
    const W right = __shfl_down_sync(0xffffffffu, cur[0], 1);
    T out[V];
    W d[V];
#pragma unroll
    for (int e = 0; e < V; ++e) {
      const W a = e == 0 ? left : cur[e == 0 ? 0 : e - 1];
      const W b = e == V - 1 ? right : cur[e == V - 1 ? e : e + 1];
      const W sm = (up[e] + dn[e]) + (a + b);
      if constexpr (FX) {
        out[e] = (EDGE && outf) ? fx_to(sm, F + 2) : i64_bits((sm + 2) >> 2);
        d[e] = sm - cur[e] * 4;
      } else {
        out[e] = T(0.25) * sm;
        d[e] = out[e] - cur[e];
      }
    }
    const bool yint = j >= jlo && j <= jhi;
    if (!(fast && yint)) {
#pragma unroll
      for (int e = 0; e < V; ++e)
        if (!(yint && cint[e])) {
          d[e] = W(0);
          if constexpr (FX) {
            if (EDGE && outf) out[e] = inf ? (wr ? src[(i64)j * nx + e] : T(0)) : fx_to(cur[e], F);
            else out[e] = i64_bits(cur[e]);
          } else {
            out[e] = cur[e];
          }
        }
    }
    if constexpr (FX) {
      fx_residual<V>(d, rmax);
    } else {
#pragma unroll
      for (int e = 0; e < V; ++e) {
        const T m = d[e] < T(0) ? -d[e] : d[e];
        rmax = m > rmax ? m : rmax;
      }
    }
    if (wr) stv<T, V>(dst, out);
    dst += nx;
  };
  int j = 0;
#pragma unroll 1
  for (; j + D <= rows; j += D) {
#pragma unroll
    for (int i = 0; i < D; ++i) step(j + i, w[i % 3], w[(i + 1) % 3], w[(i + 2) % 3], q[i]);
  }
#pragma unroll
  for (int i = 0; i < D - 1; ++i)
    if (j + i < rows) step(j + i, w[i % 3], w[(i + 1) % 3], w[(i + 2) % 3], q[i]);
  if (lane == 0 || lane == 31) rmax = 0;  // their sums lack a neighbour
}

// ---------------------------------------------------------------- 7-point heat, resident fixed point
//
// S = the six faces, L = S - 6u (exact, scale F), r = m 2^-k:
// v = u + round(m L 2^-k), the FP64 output u + r L correctly rounded, and
// |v - u| is the magnitude of the increment.  An intermediate sweep converts
// nothing: every value in both buffers, the Dirichlet boundary included, is
// in fixed point.  The first and last sweeps of a sequence (EDGE, flags
// JFX_IN_F64 / JFX_OUT_F64) convert loads and stores.
//
// The increment for any r: with fm = m 2^(62-k) < 2^60 (r <= 1/6) it is
// floor((L fm + 2^61) / 2^62).  L + 2^62 is positive (|L| < 2^61), so the
// 96-bit product of it takes four unsigned 32 x 32 -> 64-bit multiply-adds,
// and the fm that the bias adds to the quotient is exact and comes off at the
// end: 12 instructions for every r, in place of a 64 x 64 -> 128-bit product
// and a 128-bit rounding shift.
JD i64 heat_increment(i64 L, u64 fm) {
  const u64 b = (u64)L + (1ull << 62);
  const u32 bl = (u32)b, bh = (u32)(b >> 32), ml = (u32)fm, mh = (u32)(fm >> 32);
  u64 mid = (u64)bl * mh + (((u64)bl * ml) >> 32);  // < 2^61
  mid = (u64)bh * ml + mid + (1ull << 29);          // bh < 2^31
  const u64 hi = (u64)bh * mh + (mid >> 32);
  return (i64)(((hi << 2) | ((u32)mid >> 30)) - fm);
}

// For r = fb 2^-k with k <= 5 the product stays in 64 bits; fb is at most 5,
// so it takes half the multiplies (512^3 FP64, r = 1/8, precompiled tile 3:
// 413 us a sweep against 466; asynchronous copies 301^3 83 against 91).
JD i64 heat_increment_small(i64 L, i64 fb, int k) {
  const u32 f = (u32)fb;
  const i64 w = (i64)((u64)(u32)L * f + ((u64)((u32)(L >> 32) * f) << 32));
  return (w + (((i64)1 << k) >> 1)) >> k;
}

// The same increment, and in `out` the FP64 value of the exact u + r L, which
// is ce 2^62 + L fm at scale F + 62 (below 2^119): all 128 bits of the product
// are kept, so the increment and the output share it.
JD i64 heat_increment_out(i64 L, u64 fm, i64 ce, int F, double& out) {
  const u64 b = (u64)L + (1ull << 62);
  const u32 bl = (u32)b, bh = (u32)(b >> 32), ml = (u32)fm, mh = (u32)(fm >> 32);
  const u64 p0 = (u64)bl * ml;
  u64 mid = (u64)bl * mh + (p0 >> 32);
  mid = (u64)bh * ml + mid;
  s128 x;
  x.hi = (u64)bh * mh + (mid >> 32);
  x.lo = (mid << 32) | (u32)p0;
  const i64 d = (i64)((((x.hi << 3) | (x.lo >> 61)) + 1) >> 1) - (i64)fm;
  const i64 c = ce - (i64)fm;
  s128 h;
  h.lo = (u64)c << 62;
  h.hi = (u64)(c >> 2);
  x = add128(x, h);
  out = fx128_to(x, F + 62);
  return d;
}

// ---------------------------------------------------------------- 7-point heat, bulk-copy staged planes
//
// Same staging as the 27-point kernel (bulk copies on full/empty mbarriers,
// bounded waits), Dirichlet geometry: a thread owns one 16-byte column (V
// values) of 2 rows; a stage holds rows by0-1 .. by0+TH and columns
// bx0-V .. bx0+TW+V-1 of one plane, clipped to the grid (points outside are
// never needed: only interior points read neighbours).  Planes z0-1 .. z1 are
// staged; a thread keeps its own values of planes z-1 and z in registers,
// reads its own values of plane z+1 and the in-plane neighbours of plane z
// (rows y-1 and y+2, the columns left and right of its own) from the stage.
// The boundary planes z = 0 and nz-1 are written from the staged values.
//
// FX: FP64 storage in the resident 64-bit fixed point (intermediate sweeps
// only: nothing is converted); otherwise native arithmetic on T.
template <class T, int BX, int BY, int SC> struct Heat3S {
  static constexpr int V = 16 / (int)sizeof(T);
  static constexpr int RY = 2;
  static constexpr int TW = BX * V, TH = BY * RY;
  static constexpr int W = TW + 2 * V, R = TH + 2;
  static constexpr int STAGE_BYTES = W * R * (int)sizeof(T);
  static constexpr int S0 = 45056 / STAGE_BYTES;
  // stages: at most ~44 KB and SC (512^3 with 32 x 4 threads, 5.4 KB
  // stages: FP32 656 GLUP/s with 4 stages, 710 with 5, 713 with 6; FP64
  // precompiled 327.5 with 6, 295.6 with 5); larger tiles' stages fit fewer
  static constexpr int SMAX = SC;
  static constexpr int S = S0 < 2 ? 2 : (S0 > SMAX ? SMAX : S0);
  // A step needs planes z and z+1 staged.  With S >= 3 warp 0 refills the
  // stage released one step earlier (slack for lagging warps); with S = 2 it
  // refills the stage just released, and no plane is prefetched.
  static constexpr int D = S >= 3 ? 1 : 0;
  static constexpr int NW = BX * BY / 32;
};

template <class T, int BX, int BY, int SC> struct alignas(128) Heat3SSmem {
  T st[Heat3S<T, BX, BY, SC>::S][Heat3S<T, BX, BY, SC>::R][Heat3S<T, BX, BY, SC>::W];
  u64 full[Heat3S<T, BX, BY, SC>::S];
  u64 empty[Heat3S<T, BX, BY, SC>::S];
};

// 16-byte shared-memory vector reads (bit patterns kept).
JD void lds_vec(const void* p, float (&r)[4]) {
  const float4 t = *reinterpret_cast<const float4*>(p);
  r[0] = t.x; r[1] = t.y; r[2] = t.z; r[3] = t.w;
}
JD void lds_vec(const void* p, double (&r)[2]) {
  const double2 t = *reinterpret_cast<const double2*>(p);
  r[0] = t.x; r[1] = t.y;
}
JD void lds_vec(const void* p, i64 (&r)[2]) {
  const longlong2 t = *reinterpret_cast<const longlong2*>(p);
  r[0] = t.x; r[1] = t.y;
}

template <class A, class B> struct SameT { static constexpr bool value = false; };
template <class A> struct SameT<A, A> { static constexpr bool value = true; };

template <class T, bool FX> struct HeatAcc { typedef T type; };
template <> struct HeatAcc<double, true> { typedef u64 type; };

template <class T, int BX, int BY, bool FX, int SC, class P>
JD void heat3s_body(const T* __restrict__ u, T* __restrict__ v, const P& p, const JParams& rt, int F,
                    typename HeatAcc<T, FX>::type& rmax, Heat3SSmem<T, BX, BY, SC>& sm) {
  typedef Heat3S<T, BX, BY, SC> G;
  constexpr int V = G::V;
  typedef typename WT<T, FX ? JM_FIXED : JM_NATIVE>::type Wt;  // working type: i64 (fixed) or T
  const i64 nx = p.nx, ny = p.ny, nz = p.nz, sz = nx * ny;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int tid = ty * BX + tx;
  const bool warp0 = tid < 32;
  const i64 bx0 = (i64)blockIdx.x * G::TW, by0 = (i64)blockIdx.y * G::TH;
  const i64 x0 = bx0 + (i64)tx * V, y0 = by0 + 2 * ty;
  const bool ax = x0 < nx;
  const bool ay[2] = {ax && y0 < ny, ax && y0 + 1 < ny};
  // interior mask of the thread's 2 x V points: bit yy * V + e
  unsigned inm = 0;
#pragma unroll
  for (int yy = 0; yy < 2; ++yy)
#pragma unroll
    for (int e = 0; e < V; ++e)
      if (y0 + yy >= 1 && y0 + yy <= ny - 2 && x0 + e >= 1 && x0 + e <= nx - 2) inm |= 1u << (yy * V + e);
  const bool fast = __all_sync(0xffffffffu, inm == (1u << (2 * V)) - 1);  // the warp holds interior points only
  const i64 cz0 = (i64)blockIdx.z * p.zc;
  const i64 cz1 = (cz0 + p.zc < nz) ? cz0 + p.zc : nz;
  const i64 z0 = cz0 < 1 ? 1 : cz0;
  const i64 z1 = cz1 > nz - 1 ? nz - 1 : cz1;
  // raw input word -> working value, working value -> output word
  auto cvt = [&](T raw) -> Wt {
    if constexpr (FX) return bits_i64(raw);
    else return raw;
  };
  auto as_out = [&](Wt w) -> T {
    if constexpr (FX) return i64_bits(w);
    else return w;
  };
  if (z0 >= z1) {  // a chunk holding only a boundary plane (block-uniform)
    for (i64 z = cz0; z < cz1; ++z)
#pragma unroll
      for (int yy = 0; yy < 2; ++yy)
        if (ay[yy]) {
          T t[V];
          ldv<T, V>(u + z * sz + (y0 + yy) * nx + x0, t);
          stv<T, V>(v + z * sz + (y0 + yy) * nx + x0, t);
        }
    return;
  }
  const int L = (int)(z1 - z0) + 2;  // staged planes z0-1 .. z1
  const i64 lim = rt.timeout_ns;
  const bool stall_cta = rt.stall_plane >= 0 && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0;
  if (tid == 0) {
#pragma unroll
    for (int s = 0; s < G::S; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.empty[s], G::NW);
    }
    mbar_init_fence();
  }
  __syncthreads();
  // warp 0 requests a plane: one bulk copy per staged row inside the grid
  // (rows and columns clipped to it), lane r copying row r; lane 0 first posts
  // the byte count of the whole plane
  static_assert(G::R <= 32, "one staged row per lane of warp 0");
  const int lane = tid & 31;
  const i64 c0 = bx0 - V < 0 ? 0 : bx0 - V;
  const i64 c1 = bx0 + G::TW + V > nx ? nx : bx0 + G::TW + V;
  const int rlo = by0 == 0 ? 1 : 0, rhi = ny - by0 + 1 < G::R ? (int)(ny - by0 + 1) : G::R;
  const u32 row_bytes = (u32)((c1 - c0) * (i64)sizeof(T));
  const bool has_row = lane >= rlo && lane < rhi;
  const T* src = u + (z0 - 1) * sz + (by0 - 1 + lane) * nx + c0;  // the lane's row of the next plane
  const int slot = lane * G::W + (int)(c0 - (bx0 - V));
  auto request = [&](int j, int s) {
    if (!(stall_cta && j == rt.stall_plane)) {
      if (lane == 0) mbar_expect_tx(&sm.full[s], row_bytes * (u32)(rhi - rlo));
      __syncwarp();
      if (has_row) bulk_g2s(&sm.st[s][0][0] + slot, src, row_bytes, &sm.full[s]);
    }
    src += sz;
  };
  int issued = 0, consumed = 0;  // warp 0: planes requested, planes waited for
  if (warp0)
    for (; issued < G::S && issued < L; ++issued) request(issued, issued);
  // ring cursors (stage, phase parity): cn the next plane to wait for, cq the
  // plane whose stage warp 0 refills next
  int cn_s = 0, cq_s = 0;
  u32 cn_ph = 0, cq_ph = 0;
  auto adv = [&](int& s, u32& ph) {
    if (++s == G::S) {
      s = 0;
      ph ^= 1u;
    }
  };
  auto wait_next = [&]() -> bool {
    if (!mbar_wait(&sm.full[cn_s], cn_ph, lim)) return false;
    ++consumed;
    return true;
  };
  // this warp has read the plane in stage s for the last time (plane j);
  // warp 0 then refills the stage of plane j - D once every warp released it
  auto release = [&](int j, int s) -> bool {
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(&sm.empty[s]);
    if (j >= G::D) {
      if (warp0 && issued < L) {
        if (!mbar_wait(&sm.empty[cq_s], cq_ph, lim)) return false;
        request(issued, cq_s);
        ++issued;
      }
      adv(cq_s, cq_ph);
    }
    return true;
  };
  auto own = [&](int s, T (&raw)[2][V]) {
#pragma unroll
    for (int yy = 0; yy < 2; ++yy) lds_vec(&sm.st[s][2 * ty + 1 + yy][V + V * tx], raw[yy]);
  };
  auto store_bnd = [&](T* dst, const Wt (&w)[2][V]) {
#pragma unroll
    for (int yy = 0; yy < 2; ++yy)
      if (ay[yy]) {
        T t[V];
#pragma unroll
        for (int e = 0; e < V; ++e) t[e] = as_out(w[yy][e]);
        stv<T, V>(dst + yy * nx, t);
      }
  };
  Wt wa[2][V], wb[2][V], wc[2][V];  // own values of planes z-1, z, z+1 (rotating roles)
  T* vo = v + y0 * nx + x0;
  bool ok = wait_next();
  if (ok) {  // plane z0-1
    T r0[2][V];
    own(cn_s, r0);
#pragma unroll
    for (int yy = 0; yy < 2; ++yy)
#pragma unroll
      for (int e = 0; e < V; ++e) wa[yy][e] = cvt(r0[yy][e]);
    if (cz0 == 0) store_bnd(vo, wa);  // boundary plane 0
    const int s0 = cn_s;
    adv(cn_s, cn_ph);
    ok = release(0, s0) && wait_next();
  }
  int cc_s = cn_s;  // stage of the centre plane z
  if (ok) {  // plane z0
    T r0[2][V];
    own(cn_s, r0);
#pragma unroll
    for (int yy = 0; yy < 2; ++yy)
#pragma unroll
      for (int e = 0; e < V; ++e) wb[yy][e] = cvt(r0[yy][e]);
    adv(cn_s, cn_ph);
  }
  const T r = (T)p.c0;
  const i64 fb = p.fb;
  const int k = p.fk;
  const bool fold = heat_fold(p);
  constexpr bool folded = Folded<P>::value;  // extents and coefficients are constants
  vo += z0 * sz;
  // one output plane (staged plane j, 1 <= j <= L-2) from the own values of
  // planes j-1 (zp) and j (cur); fills zn with those of plane j+1
  auto step = [&](int j, const Wt (&zp)[2][V], const Wt (&cur)[2][V], Wt (&zn)[2][V]) -> bool {
    if (!wait_next()) return false;
    T rzn[2][V];
    own(cn_s, rzn);
    const Wt(*pl)[G::W] = reinterpret_cast<const Wt(*)[G::W]>(sm.st[cc_s]);
    Wt ym[V], yp[V], xl[2], xr[2];
    lds_vec(&pl[2 * ty][V + V * tx], ym);
    lds_vec(&pl[2 * ty + 3][V + V * tx], yp);
#pragma unroll
    for (int yy = 0; yy < 2; ++yy) {
      xl[yy] = pl[2 * ty + 1 + yy][V + V * tx - 1];
      xr[yy] = pl[2 * ty + 1 + yy][V + V * tx + V];
    }
#pragma unroll
    for (int yy = 0; yy < 2; ++yy)
#pragma unroll
      for (int e = 0; e < V; ++e) zn[yy][e] = cvt(rzn[yy][e]);
    T out[2][V];
    Wt dv[2 * V];  // the increments v - c
    // f(sum of the six faces, centre, increment, output) for every point
    auto each = [&](auto f) {
#pragma unroll
      for (int yy = 0; yy < 2; ++yy)
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const Wt a = (e == 0) ? xl[yy] : cur[yy][e == 0 ? 0 : e - 1];
          const Wt b = (e == V - 1) ? xr[yy] : cur[yy][e == V - 1 ? e : e + 1];
          const Wt c = yy == 0 ? ym[e] : cur[0][e];
          const Wt d = yy == 0 ? cur[1][e] : yp[e];
          f(((a + b) + (c + d)) + (zp[yy][e] + zn[yy][e]), cur[yy][e], dv[yy * V + e], out[yy][e]);
        }
    };
    if constexpr (!FX) {
      each([&](T sum, T ce, T& dk, T& o) {
        o = ce + r * (sum - T(6) * ce);
        dk = o - ce;
      });
    } else if (folded && fold) {
      each([&](i64 sum, i64 ce, i64& dk, T& o) {
        const i64 vn = (fb * sum + ((((i64)1 << k) - 6 * fb) * ce + ((i64)1 << (k - 1)))) >> k;
        dk = vn - ce;
        o = i64_bits(vn);
      });
    } else if (p.fpath == JACC_FP_SMALL) {
      each([&](i64 sum, i64 ce, i64& dk, T& o) {
        dk = heat_increment_small(sum - 6 * ce, fb, k);
        o = i64_bits(ce + dk);
      });
    } else {
      each([&](i64 sum, i64 ce, i64& dk, T& o) {
        dk = heat_increment(sum - 6 * ce, p.fm);
        o = i64_bits(ce + dk);
      });
    }
    if (!fast) {  // boundary points keep their values
#pragma unroll
      for (int yy = 0; yy < 2; ++yy)
#pragma unroll
        for (int e = 0; e < V; ++e)
          if (!((inm >> (yy * V + e)) & 1u)) {
            dv[yy * V + e] = Wt(0);
            out[yy][e] = as_out(cur[yy][e]);
          }
    }
    if constexpr (FX) {
      fx_residual<2 * V>(dv, rmax);
    } else {
#pragma unroll
      for (int q = 0; q < 2 * V; ++q) rmax = fmaxf(rmax, fabsf(dv[q]));
    }
    if (fast) {
      stv<T, V>(vo, out[0]);
      stv<T, V>(vo + nx, out[1]);
    } else {
#pragma unroll
      for (int yy = 0; yy < 2; ++yy)
        if (ay[yy]) stv<T, V>(vo + yy * nx, out[yy]);
    }
    vo += sz;
    if (j == L - 2 && cz1 == nz) store_bnd(vo, zn);  // boundary plane nz-1 = staged plane L-1
    if (!release(j, cc_s)) return false;
    cc_s = cn_s;
    adv(cn_s, cn_ph);
    return true;
  };
  if (ok) {
    // three steps per iteration: the buffers' roles rotate without copies
    int j = 1;
    for (; j + 2 <= L - 2; j += 3) {
      if (!step(j, wa, wb, wc) || !step(j + 1, wb, wc, wa) || !step(j + 2, wc, wa, wb)) {
        ok = false;
        break;
      }
    }
    if (ok && j <= L - 2) ok = step(j, wa, wb, wc);
    if (ok && j + 1 <= L - 2) ok = step(j + 1, wb, wc, wa);
  }
  if (!ok) {
    if (rt.status) atomicExch(rt.status, JACC_DEV_TIMEOUT);
    if (warp0)
      for (int j = consumed; j < issued; ++j)
        if (!(stall_cta && j == rt.stall_plane)) mbar_wait(&sm.full[j % G::S], (u32)((j / G::S) & 1), lim);
  }
}

// ---------------------------------------------------------------- planes staged by asynchronous copies: conversion
//
// Converts this thread's share of a landed FP64 plane to fixed point in place:
// 1.2 conversions a point, where the readers of a staged plane made three (one
// jacc_launch of a 256^3 7-point grid: 306 us before, 161 now, its pre-pass
// included).
template <int BX, int BY, int CH, int V>
JD void ring_to_fixed(const RingPlan<double, BX, BY, CH, V>& pl, double* stage, int F) {
  typedef RingG<double, BX, BY, CH, V> G;
  const int tid = threadIdx.y * BX + threadIdx.x;
#pragma unroll
  for (int i = 0; i < G::PER; ++i)
    if ((pl.mask >> i) & 1u) {
      double* w = stage + (tid + i * G::NT) * CH;
      if constexpr (CH == 2) {
        double2 t = *reinterpret_cast<double2*>(w);
        t.x = i64_bits(fx_from(t.x, F));
        t.y = i64_bits(fx_from(t.y, F));
        *reinterpret_cast<double2*>(w) = t;
      } else {
        *w = i64_bits(fx_from(*w, F));
      }
    }
}

// ---------------------------------------------------------------- 7-point heat, planes staged by asynchronous copies
//
// FX: FP64 storage in the resident 64-bit fixed point (EDGE: the first and
// last sweeps of a sequence and single launches, whose staged values the
// copying threads convert in place); otherwise native arithmetic on T.  A
// thread keeps its own values of planes z-1 and z in registers and reads its
// values of plane z+1 and its neighbours in plane z from the stages; two
// planes of look-ahead (stage j is free once step j is done, so plane j + S
// - 2 is requested after the barrier that opens step j - 1).  Bound by the
// integer ALU work (79 thread-instructions a point, 143 in the kernel that
// loaded halos into registers and multiplied in 128 bits): 301 x 253 x 199,
// r = 0.1, 90 us a sweep before, 57 now (4.2 TB/s); FP32 rows of odd length
// 301 x 253 x 199 27.5 us.
template <class T, int BX, int BY, int CH, int V, bool FX, bool EDGE, class P>
JD void heat3r_body(const T* __restrict__ u, T* __restrict__ v, const P& p, int F, int flags,
                    typename HeatAcc<T, FX>::type& rmax, T* sm) {
  typedef RingG<T, BX, BY, CH, V> G;
  typedef typename WT<T, FX ? JM_FIXED : JM_NATIVE>::type Wt;
  constexpr int RY = G::RY, S = G::S;
  const i64 nx = p.nx, ny = p.ny, nz = p.nz, sz = nx * ny;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const i64 bx0 = (i64)blockIdx.x * G::TW, by0 = (i64)blockIdx.y * G::TH;
  const i64 x0 = bx0 + tx * V, y0 = by0 + ty * RY;
  // rows this thread writes (a vector column lies in the grid or outside), and
  // its interior points: bit k V + e
  unsigned wrm = 0, inm = 0;
#pragma unroll
  for (int k = 0; k < RY; ++k) {
    if (x0 < nx && y0 + k < ny) wrm |= 1u << k;
#pragma unroll
    for (int e = 0; e < V; ++e)
      if (x0 + e >= 1 && x0 + e <= nx - 2 && y0 + k >= 1 && y0 + k <= ny - 2) inm |= 1u << (k * V + e);
  }
  const bool fast = __all_sync(0xffffffffu, inm == (1u << (RY * V)) - 1);  // the warp holds interior points only
  const i64 cz0 = (i64)blockIdx.z * p.zc;
  const i64 cz1 = (cz0 + p.zc < nz) ? cz0 + p.zc : nz;
  const i64 z0 = cz0 < 1 ? 1 : cz0;
  const i64 z1 = cz1 > nz - 1 ? nz - 1 : cz1;
  const bool inf = FX && EDGE && (flags & JFX_IN_F64);
  const bool outf = FX && EDGE && (flags & JFX_OUT_F64);
  const i64 own_off = y0 * nx + x0;
  T* vo = v + own_off;
  // a boundary point's output from its working value (and, where FP64 goes
  // in and out, its unchanged input at offset `at`)
  auto bnd_out = [&](Wt w, i64 at) -> T {
    if constexpr (FX && EDGE) {
      if (outf) return inf ? u[at] : fx_to(w, F);
      return i64_bits(w);
    } else if constexpr (FX) {
      return i64_bits(w);
    } else {
      return w;
    }
  };
  if (z0 >= z1) {  // a chunk holding only a boundary plane (block-uniform)
    for (i64 z = cz0; z < cz1; ++z)
#pragma unroll
      for (int k = 0; k < RY; ++k)
        if ((wrm >> k) & 1u) {
#pragma unroll
          for (int e = 0; e < V; ++e) {
            const i64 at = own_off + z * sz + k * nx + e;
            T t = u[at];
            if constexpr (FX && EDGE) {
              if (inf != outf) t = inf ? i64_bits(fx_from(t, F)) : fx_to(bits_i64(t), F);
            }
            v[at] = t;
          }
        }
    return;
  }
  const int L = (int)(z1 - z0) + 2;  // staged planes z0-1 .. z1
  RingPlan<T, BX, BY, CH, V> plan;
  plan.init(nx, ny, bx0, by0, false);
  const T* next = u + (z0 - 1) * sz;  // next plane to stage
  int is = 0, issued = 0;             // its stage, in elements
  auto issue_next = [&]() {
    if (issued < L) plan.issue(sm + is, next);
    cpa_commit();
    ++issued;
    next += sz;
    is = is + G::STAGE == S * G::STAGE ? 0 : is + G::STAGE;
  };
#pragma unroll 1
  for (int j = 0; j < S; ++j) issue_next();
  int ns = 0;  // stage of the next plane, in elements
  auto publish = [&]() {
    if constexpr (FX && EDGE) {
      if (inf) ring_to_fixed(plan, sm + ns, F);
    }
    __syncthreads();
  };
  const Wt* own0 = reinterpret_cast<const Wt*>(sm) + (ty * RY + 1) * G::W + CH + tx * V;
  auto row = [&](const Wt* q, Wt (&w)[V]) {
    if constexpr (V == 1) w[0] = q[0];
    else lds_vec(q, w);
  };
  auto own = [&](int stage, Wt (&w)[RY][V]) {
#pragma unroll
    for (int k = 0; k < RY; ++k) row(own0 + stage + k * G::W, w[k]);
  };
  auto store_bnd = [&](i64 z, const Wt (&w)[RY][V]) {
#pragma unroll
    for (int k = 0; k < RY; ++k)
      if ((wrm >> k) & 1u) {
        T t[V];
#pragma unroll
        for (int e = 0; e < V; ++e) t[e] = bnd_out(w[k][e], own_off + z * sz + k * nx + e);
        stv<T, V>(vo + z * sz + k * nx, t);
      }
  };
  Wt wa[RY][V], wb[RY][V], wc[RY][V];  // own values of planes z-1, z, z+1 (rotating roles)
  cpa_wait<S - 1>();
  publish();
  own(ns, wa);
  if (cz0 == 0) store_bnd(0, wa);  // boundary plane 0
  ns += G::STAGE;
  cpa_wait<S - 2>();
  publish();
  own(ns, wb);
  int cs = ns;  // stage of the centre plane
  ns += G::STAGE;
  const T r = (T)p.c0;
  constexpr bool folded = Folded<P>::value;
  const bool fold = folded && heat_fold(p);
  const i64 fb = p.fb;
  const int fk = p.fk;
  i64 z = z0;
  T* vz = vo + z0 * sz;
  // output plane z from the own values of planes z-1 and z; fills zn with plane z+1's
  auto step = [&](const Wt (&zp)[RY][V], const Wt (&cur)[RY][V], Wt (&zn)[RY][V]) {
    cpa_wait<S - 3>();
    publish();
    issue_next();  // into the stage of plane z-1, last read before the barrier
    own(ns, zn);
    const Wt* c0 = own0 + cs;
    Wt ym[V], yp[V];
    row(c0 - G::W, ym);
    row(c0 + RY * G::W, yp);
    T out[RY][V];
    Wt dv[RY * V];
    // f(sum of the six faces, centre, increment, output) for every point
    auto each = [&](auto f) {
#pragma unroll
      for (int k = 0; k < RY; ++k) {
        const Wt xl = c0[k * G::W - 1], xr = c0[k * G::W + V];
#pragma unroll
        for (int e = 0; e < V; ++e) {
          const Wt a = e == 0 ? xl : cur[k][e == 0 ? 0 : e - 1], b = e == V - 1 ? xr : cur[k][e == V - 1 ? e : e + 1];
          const Wt c = k == 0 ? ym[e] : cur[k == 0 ? 0 : k - 1][e], d = k == RY - 1 ? yp[e] : cur[k == RY - 1 ? k : k + 1][e];
          f(((a + b) + (c + d)) + (zp[k][e] + zn[k][e]), cur[k][e], dv[k * V + e], out[k][e]);
        }
      }
    };
    if constexpr (!FX) {
      each([&](T sum, T ce, T& dk, T& o) {
        o = ce + r * (sum - T(6) * ce);
        dk = o - ce;
      });
    } else if (EDGE && outf) {  // the exact value, rounded once
      if (p.fpath == JACC_FP_SMALL)
        each([&](i64 sum, i64 ce, i64& dk, T& o) {
          const i64 w = fb * (sum - 6 * ce);
          dk = (w + (((i64)1 << fk) >> 1)) >> fk;  // heat_increment_small
          o = fx_to(ce * ((i64)1 << fk) + w, F + fk);
        });
      else
        each([&](i64 sum, i64 ce, i64& dk, T& o) { dk = heat_increment_out(sum - 6 * ce, p.fm, ce, F, o); });
    } else if (fold) {
      each([&](i64 sum, i64 ce, i64& dk, T& o) {
        const i64 vn = (fb * sum + ((((i64)1 << fk) - 6 * fb) * ce + ((i64)1 << (fk - 1)))) >> fk;
        dk = vn - ce;
        o = i64_bits(vn);
      });
    } else if (p.fpath == JACC_FP_SMALL) {
      each([&](i64 sum, i64 ce, i64& dk, T& o) {
        dk = heat_increment_small(sum - 6 * ce, fb, fk);
        o = i64_bits(ce + dk);
      });
    } else {
      each([&](i64 sum, i64 ce, i64& dk, T& o) {
        dk = heat_increment(sum - 6 * ce, p.fm);
        o = i64_bits(ce + dk);
      });
    }
    if (!fast) {
#pragma unroll
      for (int k = 0; k < RY; ++k)
#pragma unroll
        for (int e = 0; e < V; ++e)
          if (!((inm >> (k * V + e)) & 1u)) {
            dv[k * V + e] = Wt(0);
            if ((wrm >> k) & 1u) out[k][e] = bnd_out(cur[k][e], own_off + z * sz + k * nx + e);
          }
    }
    if constexpr (FX) fx_residual<RY * V>(dv, rmax);
    else {
#pragma unroll
      for (int k = 0; k < RY * V; ++k) rmax = fmaxf(rmax, fabsf(dv[k]));
    }
    if (fast) {
#pragma unroll
      for (int k = 0; k < RY; ++k) stv<T, V>(vz + k * nx, out[k]);
    } else {
#pragma unroll
      for (int k = 0; k < RY; ++k)
        if ((wrm >> k) & 1u) stv<T, V>(vz + k * nx, out[k]);
    }
    cs = ns;
    ns = ns + G::STAGE == S * G::STAGE ? 0 : ns + G::STAGE;
    ++z;
    vz += sz;
  };
  // three steps per iteration: the buffers' roles rotate without copies
  const int n = L - 2;
  int j = 0;
#pragma unroll 1
  for (; j + 3 <= n; j += 3) {
    step(wa, wb, wc);
    step(wb, wc, wa);
    step(wc, wa, wb);
  }
  // plane nz-1 (the last staged one) is in the buffer that the last step filled
  if (n - j == 0) {
    if (cz1 == nz) store_bnd(nz - 1, wb);
  } else {
    step(wa, wb, wc);
    if (n - j == 1) {
      if (cz1 == nz) store_bnd(nz - 1, wc);
    } else {
      step(wb, wc, wa);
      if (cz1 == nz) store_bnd(nz - 1, wa);
    }
  }
  cpa_wait<0>();
}

// ---------------------------------------------------------------- 27-point box, resident fixed point
//
// v 2^F = round(sum_j fw_j class_j 2^-K) from the exact sum; the FP64 output
// is the exact sum correctly rounded.  Periodic: no boundary, every point is
// updated.  The field sum accumulates the fixed outputs exactly in 128 bits
// per thread.
//
// The weighted sum.  JACC_FP_W32 (every fw_j below 2^31 and K in [1, 31]: the
// weights of an FP32 program): with class_j = h_j 2^32 + l_j the sum is
// A 2^32 + B, A = sum fw_j h_j and B = sum fw_j l_j (below 2^64, as the fw_j
// add up to at most 2^31 (1 + 2^-20)), eight 32 x 32 -> 64-bit multiply-adds.
// Otherwise four 64 x 64 -> 128-bit products.
//
// Bound by the integer ALU work (64-bit class sums and the products), no
// longer by latency: 320 x 256 x 192, 20 sweeps, 6.21 ms with planes loaded
// and wrapped by every thread in the sweep itself (278 thread-instructions a
// point, 811 GB/s) against 1.42 ms (3.5 TB/s), weights of 32 bits; folded
// kernels, 512^3, 274 GLUP/s with 32-bit and 173 with 53-bit weights.  Four
// rows per thread share their row sums and the classes of planes z-1 and z
// stay in registers; two rows measured 2 % slower.
template <class P> JD i64 box27_weigh(const P& p, i64 c, i64 f, i64 e, i64 g, s128* exact) {
  const int K = p.fk;
  if (p.fpath == JACC_FP_W32) {
    const int w0 = (int)p.fw0, w1 = (int)p.fw1, w2 = (int)p.fw2, w3 = (int)p.fw3;
    u64 B = (u64)1 << (K - 1);  // the rounding half
    B += (u64)(u32)w0 * (u32)c;
    B += (u64)(u32)w1 * (u32)f;
    B += (u64)(u32)w2 * (u32)e;
    B += (u64)(u32)w3 * (u32)g;
    i64 A = (i64)w0 * (int)(c >> 32);
    A += (i64)w1 * (int)(f >> 32);
    A += (i64)w2 * (int)(e >> 32);
    A += (i64)w3 * (int)(g >> 32);
    if (exact) {
      B -= (u64)1 << (K - 1);
      s128 b;
      b.lo = B;
      b.hi = 0;
      *exact = add128(from_s64_shl(A, 32), b);
      return fx128_round_shift(*exact, K);
    }
    const u64 H = (u64)(A + (i64)(B >> 32));
    return (i64)((H << (32 - K)) | ((u32)B >> K));
  }
  s128 a = mul_s64_u64(c, (u64)p.fw0);
  a = add128(a, mul_s64_u64(f, (u64)p.fw1));
  a = add128(a, mul_s64_u64(e, (u64)p.fw2));
  a = add128(a, mul_s64_u64(g, (u64)p.fw3));
  if (exact) *exact = a;
  return fx128_round_shift(a, K);
}

// The running 27-point march over staged planes, for FP64 in fixed point
// (W = i64; EDGE as above) and for native FP32 (W = float: the definition's
// terms in the order of box27_body2, fused field sum in `acc32`; 501 x 487 x
// 383, rows of odd length, 447 us a sweep with planes loaded through registers
// one step ahead, 227 here).
template <class T, int BX, int BY, int CH, bool EDGE, class P>
JD void box27r_body(const T* __restrict__ u, T* __restrict__ v, const P& p, int F, int flags, bool want_sum, s128& acc,
                    SumAcc<float>& acc32, T* sm) {
  typedef RingG<T, BX, BY, CH> G;
  constexpr bool FX = sizeof(T) == 8;
  typedef typename WT<T, FX ? JM_FIXED : JM_NATIVE>::type W;
  constexpr int RY = G::RY, S = G::S;
  const i64 nx = p.nx, ny = p.ny, nz = p.nz, sz = nx * ny;
  const int zc = p.zc;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const i64 bx0 = (i64)blockIdx.x * G::TW, by0 = (i64)blockIdx.y * G::TH;
  const i64 x0 = bx0 + tx, y0 = by0 + ty * RY;
  const i64 z0 = (i64)blockIdx.z * zc;
  const i64 z1 = (z0 + zc < nz) ? z0 + zc : nz;
  const int L = (int)(z1 - z0) + 2;  // staged planes z0-1 .. z1 (periodic images)
  const int nrow = x0 < nx ? (int)(ny - y0 < RY ? (ny - y0 > 0 ? ny - y0 : 0) : RY) : 0;  // rows this thread writes
  const bool inf = EDGE && (flags & JFX_IN_F64);
  const bool outf = EDGE && (flags & JFX_OUT_F64);
  RingPlan<T, BX, BY, CH> plan;
  plan.init(nx, ny, bx0, by0, true);
  i64 zi = z0 == 0 ? nz - 1 : z0 - 1;  // next plane to stage
  int is = 0;                          // and its stage, in elements
  int issued = 0;
  auto issue_next = [&]() {
    if (issued < L) plan.issue(sm + is, u + zi * sz);
    cpa_commit();
    ++issued;
    zi = zi + 1 == nz ? 0 : zi + 1;
    is = is + G::STAGE == S * G::STAGE ? 0 : is + G::STAGE;
  };
#pragma unroll 1
  for (int j = 0; j < S - 1; ++j) issue_next();
  int cs = 0;  // the stage to read, in elements
  // own-column sums of the next staged plane: c the points, f their four
  // in-plane faces, g the four in-plane diagonals
  auto consume = [&](W (&c)[RY], W (&f)[RY], W (&g)[RY]) {
    cpa_wait<S - 2>();
    if constexpr (FX && EDGE) {
      if (inf) ring_to_fixed(plan, sm + cs, F);
    }
    __syncthreads();
    issue_next();  // into the stage read before the barrier
    const W* r = reinterpret_cast<const W*>(sm) + cs + ty * RY * G::W + CH + tx;
    W m[RY + 2], s[RY + 2];
#pragma unroll
    for (int k = 0; k < RY + 2; ++k) {
      m[k] = r[k * G::W];
      s[k] = r[k * G::W - 1] + r[k * G::W + 1];
    }
#pragma unroll
    for (int k = 0; k < RY; ++k) {
      c[k] = m[k + 1];
      f[k] = s[k + 1] + (m[k] + m[k + 2]);
      g[k] = s[k] + s[k + 2];
    }
    cs = cs + G::STAGE == S * G::STAGE ? 0 : cs + G::STAGE;
  };
  // running classes of the output plane: pf = f(z) + c(z-1), pe = g(z) + f(z-1), pc = g(z-1)
  W pf[RY], pe[RY], pc[RY];
  const float w0 = (float)p.c0, wf = (float)p.c1, we = (float)p.c2, wc = (float)p.c3;
  T* vo = v + z0 * sz + y0 * nx + x0;
  auto step = [&](const W (&c0)[RY], const W (&f0)[RY], const W (&g0)[RY], W (&cn)[RY], W (&fn)[RY], W (&gn)[RY]) {
    consume(cn, fn, gn);
    i64 rowsum = 0;  // at most four values below 2^59: exact
#pragma unroll
    for (int k = 0; k < RY; ++k) {
      const W cf = pf[k] + cn[k], ce = pe[k] + fn[k], cc = pc[k] + gn[k];
      if constexpr (FX) {
        double o;
        i64 q;
        if (EDGE && outf) {
          s128 ex;
          q = box27_weigh(p, c0[k], cf, ce, cc, &ex);
          o = fx128_to(ex, F + p.fk);
        } else {
          q = box27_weigh(p, c0[k], cf, ce, cc, nullptr);
          o = i64_bits(q);
        }
        if (k < nrow) {
          vo[k * nx] = o;
          rowsum += q;
        }
      } else {
        // the fused multiply-adds written out: one rounding pattern for every variant
        const float o = __fadd_rn(fmaf(w0, c0[k], __fmul_rn(wf, cf)), fmaf(we, ce, __fmul_rn(wc, cc)));
        if (k < nrow) {
          vo[k * nx] = o;
          if (want_sum) acc32.add(o);
        }
      }
      pf[k] = fn[k] + c0[k];
      pe[k] = gn[k] + f0[k];
      pc[k] = g0[k];
    }
    vo += sz;
    if constexpr (FX) {
      s128 t;
      t.lo = (u64)rowsum;
      t.hi = (u64)(rowsum >> 63);
      acc = add128(acc, t);
    }
  };
  W ca[RY], fa[RY], ga[RY], cb[RY], fb[RY], gb[RY];
  consume(ca, fa, ga);
  consume(cb, fb, gb);
#pragma unroll
  for (int k = 0; k < RY; ++k) {
    pf[k] = fb[k] + ca[k];
    pe[k] = gb[k] + fa[k];
    pc[k] = ga[k];
  }
  int j = 2;
#pragma unroll 1
  for (; j + 1 < L; j += 2) {
    step(cb, fb, gb, ca, fa, ga);
    step(ca, fa, ga, cb, fb, gb);
  }
  if (j < L) step(cb, fb, gb, ca, fa, ga);
  cpa_wait<0>();
}

// ---------------------------------------------------------------- 7-point heat without staging
//
// A grid that fits L2 is bound by the latency of a CTA's march, not by bytes:
// each plane of a staged march costs a wait and a barrier (64^3 FP64: 9.6 us a
// sweep at 18 planes).  Here a thread updates N planes of V consecutive
// columns of one row straight from memory: no shared memory, no barrier, every
// load independent of the others, so a sweep costs little more than one trip
// to L2.  L1 serves the neighbours that threads share.  Two planes a thread:
// 64^3 FP64 3.1 us a sweep, 5.4 with four.  These are the
// intermediate sweeps of small grids; the arithmetic is that of the staged
// kernels, term for term.
// The 7-point sweep in working type W (i64: fixed point; T: native).  Returns
// the thread's residual maximum.
template <class T, class W, int BX, int BY, int V, int N, class P, class R>
JD void heat3d_direct(const T* __restrict__ u, T* __restrict__ v, const P& p, R& rmax) {
  constexpr bool FX = SameT<W, i64>::value;
  const i64 nx = p.nx, ny = p.ny, nz = p.nz, sz = nx * ny;
  const i64 x = ((i64)blockIdx.x * BX + threadIdx.x) * V, y = (i64)blockIdx.y * BY + threadIdx.y, z0 = (i64)blockIdx.z * N;
  if (x >= nx || y >= ny) return;
  const T* col = u + y * nx + x;
  // neighbours outside the grid are replaced by points inside: only boundary points would use them
  const i64 dl = x > 0 ? -1 : 0, dr = x + V < nx ? V : 0, dm = y > 0 ? -nx : 0, dp = y < ny - 1 ? nx : 0;
  T own[N + 2][V], ym[N][V], yp[N][V], xl[N], xr[N];
#pragma unroll
  for (int k = 0; k < N + 2; ++k) {
    i64 z = z0 - 1 + k;
    z = z < 0 ? 0 : (z > nz - 1 ? nz - 1 : z);
    const T* c = col + z * sz;
    ldv<T, V>(c, own[k]);
    if (k >= 1 && k <= N) {
      ldv<T, V>(c + dm, ym[k - 1]);
      ldv<T, V>(c + dp, yp[k - 1]);
      xl[k - 1] = __ldg(c + dl);
      xr[k - 1] = __ldg(c + dr);
    }
  }
  auto w = [&](T t) -> W {
    if constexpr (FX) return bits_i64(t);
    else return t;
  };
  constexpr bool folded = Folded<P>::value;
  const bool fold = folded && heat_fold(p);
  const T r = (T)p.c0;
  T* o = v + z0 * sz + y * nx + x;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    const i64 z = z0 + k;
    if (z >= nz) break;
    const bool in = y >= 1 && y <= ny - 2 && z >= 1 && z <= nz - 2;
    T out[V];
#pragma unroll
    for (int e = 0; e < V; ++e) {
      const W ce = w(own[k + 1][e]);
      const W a = w(e == 0 ? xl[k] : own[k + 1][e == 0 ? 0 : e - 1]);
      const W b = w(e == V - 1 ? xr[k] : own[k + 1][e == V - 1 ? e : e + 1]);
      const W sum = ((a + b) + (w(ym[k][e]) + w(yp[k][e]))) + (w(own[k][e]) + w(own[k + 2][e]));
      const bool ine = in && x + e >= 1 && x + e <= nx - 2;
      if constexpr (FX) {
        i64 d;
        if (fold) d = ((p.fb * sum + ((((i64)1 << p.fk) - 6 * p.fb) * ce + ((i64)1 << (p.fk - 1)))) >> p.fk) - ce;
        else d = heat_increment(sum - 6 * ce, p.fm);
        d = ine ? d : 0;
        const u64 m = (u64)(d ^ (d >> 63));
        rmax = m > rmax ? m : rmax;
        out[e] = i64_bits(ce + d);
      } else {
        const T q = ce + r * (sum - T(6) * ce);
        T d = q - ce;
        d = d < T(0) ? -d : d;
        rmax = (ine && d > rmax) ? d : rmax;
        out[e] = ine ? q : ce;
      }
    }
    stv<T, V>(o + k * sz, out);
  }
}

// ====================================================================== kernels
//
// Every stencil kernel has the signature
//   (const T* u, T* v, JParams p, double* resid, const u64* maxword, int flags)
// and calls an entry below with P = JParams (precompiled) or P = a struct of
// constants (NVRTC); the runtime-only fields (status word, wait limits) are
// read from the JParams argument `rt` in both cases.
// resid (nullable) receives the fused reduction via one atomic per CTA (it
// must be zeroed before the launch); maxword (FP64 only, nullable) holds the
// bit pattern of max|u| written by jacc_k_maxabs, which selects the fixed
// point scale.  With maxword NULL or fpath NONE the native path runs.
// flags (JFX_*) say whether this sweep of a sequence reads and writes FP64
// or the resident fixed-point representation; native paths ignore them.
// EDGE = false instantiations run the intermediate sweeps of a fixed-point
// sequence and contain no conversion code; EDGE = true ones run the first and
// last sweeps and single launches.

// Kernel families (JACC_FAM_*, jacc_params.h): a table tile runs the kernel
// that the autotuner times for it; the library's own choice (no tile asked
// for, none remembered) may also take the strip march, the asynchronous-copy
// ring, or no staging at all.  FP64 handles that never run in fixed point
// (JACC_ARITH_NATIVE, non-convex coefficients) take kernels of their own
// (JACC_FAM_NATIVE): the fixed-point kernels also hold a native branch, for
// fields that turn out not to fit the format, but its CTAs cover several rows a
// thread one after the other, under register bounds made for integers.
// A folded grid of at most JACC_SMALL_GRID points takes the strip march also
// where a tile with 16-byte columns was asked for: its few rows in flight are
// latency-bound there (256 x 256 FP64, tile 1: 2.2 us a sweep, 3.0 by rows; at
// 4096 x 4096 52 and 50).
template <class P, bool FOLDED = Folded<P>::value> struct SmallFold { static constexpr bool value = false; };
template <class P> struct SmallFold<P, true> { static constexpr bool value = P::nx * P::ny <= JACC_SMALL_GRID; };
// A folded FP64 grid of more than JACC_LARGE_GRID points, which streams from
// HBM, has six rows in flight instead of three and marches twice the rows
// (4096^2 44.7 us a sweep against 47.6; FP32 21.7 against 20.1).
template <class P, bool FOLDED = Folded<P>::value> struct LargeFold { static constexpr bool value = false; };
template <class P> struct LargeFold<P, true> { static constexpr bool value = P::nx * P::ny > JACC_LARGE_GRID; };
template <class T, int BX, int BY, int V, int FAM, bool EDGE, class P>
JD void jacobi2d_entry(const T* __restrict__ u, T* __restrict__ v, const P& p, const JParams& rt, double* resid,
                       const u64* maxword, int flags) {
  griddep_wait();
  if (stopped(rt.stop)) return;
  u64 bits = 0;
  const i64 ys = ((i64)blockIdx.y * BY + threadIdx.y) * p.zc;
  const i64 ye = (ys + p.zc < p.ny) ? ys + p.zc : p.ny;
  // scalar columns and small folded grids march strips whatever the tile
  // (native FP64 arithmetic only the latter: its own pipe bounds it, and a strip
  // updates 2/30 of its points twice)
  constexpr bool NATIVE = FAM == JACC_FAM_NATIVE;
  constexpr bool STRIP = SmallFold<P>::value || (!NATIVE && (FAM == JACC_FAM_STRIP || V == 1));
  constexpr int DEPTH = !EDGE && V == 2 && LargeFold<P>::value ? 6 : 3;
  // STRIP: BX / 32 strips of 30 V columns across the CTA
  const i64 strip = (i64)blockIdx.x * (BX / 32) + (threadIdx.x >> 5);
  const i64 xl = STRIP ? strip * (30 * V) + ((int)(threadIdx.x & 31) - 1) * V : (i64)blockIdx.x * (BX * V) + (i64)threadIdx.x * V;
  const int F = (!NATIVE && sizeof(T) == 8 && maxword && p.fpath != JACC_FP_NONE) ? fx_frac_bits(*maxword) : -1;
  if (!NATIVE && sizeof(T) == 8 && F >= 0) {
    if constexpr (!NATIVE && sizeof(T) == 8) {
      u64 m = 0;
      if (ys < p.ny) {
        if constexpr (STRIP) jacobi_strip<double, V, true, EDGE, DEPTH>(u, v, p.nx, p.ny, xl, ys, ye, F, flags, m);
        else jacobi_fx_march<V, false, EDGE>(u, v, p.nx, p.ny, xl, ys, ye, F, flags, m);
      }
      bits = dbits(fx_to_u(m, F + 2));
    }
  } else {
    T m = T(0);
    if (ys < p.ny) {
      if constexpr (STRIP) jacobi_strip<T, V, false, false, DEPTH>(u, v, p.nx, p.ny, xl, ys, ye, -1, 0, m);
      else jacobi_march<T, V, JM_NATIVE, false>(u, v, p.nx, p.ny, xl, ys, ye, -1, m);
    }
    bits = dbits((double)m);
  }
  block_max_to<BX * BY>(bits, resid);
}

// How a 3D kernel loads.  BULK: 16-byte columns staged by bulk copies on
// mbarriers (no copy instructions, no CTA barrier).  RING: planes staged by
// asynchronous copies, which arrive sooner; also every converting FP64 sweep,
// where each staged value is converted once by the thread that copied it, and
// the FP64 table tiles of scalar columns.  DIRECT: no staging (small 7-point
// grids, and the table's scalar 32 x 8 tiles).  Otherwise (FP32 table tiles of
// scalar columns) halos loaded through registers.
template <int STENCIL, class T, int BX, int BY, int V, int FAM, bool EDGE> struct Load3D {
  static constexpr bool F64 = sizeof(T) == 8;
  static constexpr bool VEC = V * sizeof(T) == 16;
  static constexpr bool DIRECT =
      !EDGE && STENCIL == 7 && (FAM == JACC_FAM_DIRECT || (FAM == JACC_FAM_TABLE && JACC_DIRECT_TILE(BX, BY, V)));
  static constexpr bool BULK = !EDGE && VEC && (FAM == JACC_FAM_TABLE || FAM == JACC_FAM_BULK) && !(F64 && STENCIL == 27);
  static constexpr bool RING = !DIRECT && !BULK && FAM != JACC_FAM_NATIVE && (EDGE || F64 || FAM == JACC_FAM_RING);
};

template <class T, int BX, int BY, int V, int FAM, bool EDGE, class P>
JD void heat3d_entry(const T* __restrict__ u, T* __restrict__ v, const P& p, const JParams& rt, double* resid,
                     const u64* maxword, int flags) {
  griddep_wait();
  if (stopped(rt.stop)) return;
  typedef Load3D<7, T, BX, BY, V, FAM, EDGE> K;
  u64 bits = 0;
  const int F = (sizeof(T) == 8 && maxword && p.fpath != JACC_FP_NONE) ? fx_frac_bits(*maxword) : -1;
  if constexpr (FAM == JACC_FAM_NATIVE) {
    __shared__ Plane<T, BX, BY, V> sm;
    T m = T(0);
    heat3d_body<T, BX, BY, V, JM_NATIVE>(u, v, p, p.zc, -1, m, sm);
    bits = dbits((double)m);
  } else if constexpr (K::DIRECT) {
    if (sizeof(T) == 8 && F >= 0) {
      u64 m = 0;
      if constexpr (sizeof(T) == 8) heat3d_direct<T, i64, BX, BY, V, JACC_DIRECT_PLANES>(u, v, p, m);
      bits = dbits(fx_to_u(m, F));
    } else {
      T m = T(0);
      heat3d_direct<T, T, BX, BY, V, JACC_DIRECT_PLANES>(u, v, p, m);
      bits = dbits((double)m);
    }
  } else if constexpr (sizeof(T) == 8) {
    typedef RingG<double, BX, BY, V, V> G;
    // stage cap: 5 for the constant-folded intermediate sweeps (7 CTAs per SM,
    // SweepMinBlocks), else 6
    constexpr int SC = Folded<P>::value ? 5 : 6;
    // the native path covers the CTA's rows in sub-tiles of BY rows
    constexpr int SUBS = K::BULK ? 2 : G::RY;
    typedef Plane<double, BX, BY, V> NativePlane;
    constexpr size_t SM_MAIN = K::BULK ? sizeof(Heat3SSmem<double, BX, BY, SC>) : (size_t)G::S * G::STAGE * 8;
    __shared__ __align__(128) unsigned char raw[sizeof(NativePlane) > SM_MAIN ? sizeof(NativePlane) : SM_MAIN];
    if (F >= 0) {
      u64 m = 0;
      if constexpr (K::BULK)
        heat3s_body<double, BX, BY, true, SC>(u, v, p, rt, F, m, *reinterpret_cast<Heat3SSmem<double, BX, BY, SC>*>(raw));
      else
        heat3r_body<double, BX, BY, V, V, true, EDGE>(u, v, p, F, flags, m, reinterpret_cast<double*>(raw));
      bits = dbits(fx_to_u(m, F));  // max |v - c| in fixed point
    } else {
      double m = 0.0;
#pragma unroll 1
      for (int sub = 0; sub < SUBS; ++sub) {
        if (sub) __syncthreads();  // the sub-tiles share the planes
        heat3d_body<T, BX, BY, V, JM_NATIVE>(u, v, p, p.zc, -1, m, *reinterpret_cast<NativePlane*>(raw), SUBS, sub);
      }
      bits = dbits(m);
    }
  } else if constexpr (K::BULK) {
    __shared__ Heat3SSmem<float, BX, BY, 6> sm;
    float m = 0.0f;
    heat3s_body<float, BX, BY, false, 6>(u, v, p, rt, -1, m, sm);
    bits = dbits((double)m);
  } else if constexpr (K::RING) {
    typedef RingG<float, BX, BY, V, V> G;
    __shared__ __align__(16) float sm[G::S * G::STAGE];
    float m = 0.0f;
    heat3r_body<float, BX, BY, V, V, false, false>(u, v, p, -1, 0, m, sm);
    bits = dbits((double)m);
  } else {
    __shared__ Plane<T, BX, BY, V> sm;
    T m = T(0);
    heat3d_body<T, BX, BY, V, JM_NATIVE>(u, v, p, p.zc, -1, m, sm);
    bits = dbits((double)m);
  }
  block_max_to<BX * BY>(bits, resid);
}

template <class T, int BX, int BY, int V, int FAM, bool EDGE, class P>
JD void box27_entry(const T* __restrict__ u, T* __restrict__ v, const P& p, const JParams& rt, double* resid,
                    const u64* maxword, int flags) {
  griddep_wait();
  typedef Load3D<27, T, BX, BY, V, FAM, EDGE> K;
  double total = 0.0;
  const int F = (sizeof(T) == 8 && maxword && p.fpath != JACC_FP_NONE) ? fx_frac_bits(*maxword) : -1;
  if constexpr (FAM == JACC_FAM_NATIVE) {
    __shared__ Plane<T, BX, BY, V> sm;
    SumAcc<T> acc;
    box27_body2<T, BX, BY, V>(u, v, p, p.zc, acc, resid != nullptr, sm);
    total = acc.total();
  } else if constexpr (sizeof(T) == 8) {
    typedef RingG<double, BX, BY, V> G;
    constexpr size_t SM_RING = (size_t)G::S * G::STAGE * 8, SM_PLANE = sizeof(Plane<double, BX, BY, 1>);
    __shared__ __align__(16) unsigned char raw[SM_RING > SM_PLANE ? SM_RING : SM_PLANE];
    if (F >= 0) {
      s128 acc;
      acc.lo = acc.hi = 0ull;
      SumAcc<float> none;
      box27r_body<double, BX, BY, V, EDGE>(u, v, p, F, flags, false, acc, none, reinterpret_cast<double*>(raw));
      total = fx128_to(acc, F);
    } else {
      SumAcc<T> acc;
#pragma unroll 1
      for (int sub = 0; sub < G::RY; ++sub) {
        __syncthreads();  // the sub-tiles share the planes
        box27_body2<T, BX, BY, 1>(u, v, p, p.zc, acc, resid != nullptr, *reinterpret_cast<Plane<double, BX, BY, 1>*>(raw),
                                  G::RY, sub);
      }
      total = acc.total();
    }
  } else if constexpr (V == 4) {
    total = box27s_body<BX, BY, K::BULK>(u, v, p, rt, resid != nullptr);
  } else if constexpr (K::RING) {
    typedef RingG<float, BX, BY, V> G;
    __shared__ __align__(16) float sm[G::S * G::STAGE];
    SumAcc<float> acc;
    s128 none;
    box27r_body<float, BX, BY, V, false>(u, v, p, -1, 0, resid != nullptr, none, acc, sm);
    total = acc.total();
  } else {
    __shared__ Plane<T, BX, BY, V> sm;
    SumAcc<T> acc;
    box27_body2<T, BX, BY, V>(u, v, p, p.zc, acc, resid != nullptr, sm);
    total = acc.total();
  }
  block_sum_to<BX * BY>(total, resid);
}

#ifdef JACC_AUX_KERNELS
// Pre-pass: atomicMax over n doubles of the high word of |u[i]|, its last bit
// set where the low word is not zero (so only zeros give zero).  Of the
// maximum the scale takes the exponent alone: NaN and infinities select the
// native path, as does a field of subnormals.  Three 32-bit operations a value
// instead of a 64-bit mask, comparison and two selections leave the loads as
// the bound: four of 16 bytes in flight in each of a full SM's threads.
__global__ void __launch_bounds__(256, 8) jacc_k_maxabs(const double* __restrict__ u, i64 n, u64* maxword) {
  griddep_wait();
  u32 m = 0;
  const i64 n2 = n / 2;
  const uint4* u2 = reinterpret_cast<const uint4*>(u);
  auto word = [](u32 hi, u32 lo) { return (hi & 0x7fffffffu) | min(lo, 1u); };
  auto take = [&](uint4 t) { m = max(max(m, word(t.y, t.x)), word(t.w, t.z)); };
  // a block takes 1024 consecutive words of 16 bytes at a time
  const i64 full = n2 / 1024;
#pragma unroll 1
  for (i64 b = blockIdx.x; b < full; b += gridDim.x) {
    const uint4* q = u2 + b * 1024 + threadIdx.x;
    const uint4 t0 = __ldg(q), t1 = __ldg(q + 256), t2 = __ldg(q + 512), t3 = __ldg(q + 768);
    take(t0);
    take(t1);
    take(t2);
    take(t3);
  }
  if (blockIdx.x == full % gridDim.x)
    for (i64 i = full * 1024 + threadIdx.x; i < n2; i += blockDim.x) take(__ldg(u2 + i));
  if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) {
    const u64 a = dbits(u[n - 1]);
    m = max(m, word((u32)(a >> 32), (u32)a));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  __shared__ u32 red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    const u32 w = __reduce_max_sync(0xffffffffu, threadIdx.x < 8 ? red[threadIdx.x] : 0u);
    if (threadIdx.x == 0) atomicMax(reinterpret_cast<unsigned long long*>(maxword), (unsigned long long)w << 32);
  }
}

// In-place conversion of an FP64 field to the resident 64-bit fixed point,
// q = u 2^F truncated toward zero with F from the max-abs word (the same
// conversion the first sweep of a sequence applies on load), so that the
// first sweep of a long sequence of a large field can run the intermediate
// kernel.  A field routed to native FP64 (F < 0) is left unchanged.
__global__ void __launch_bounds__(256) jacc_k_to_fixed(double* __restrict__ u, i64 n, const u64* maxword) {
  griddep_wait();
  const int F = fx_frac_bits(*maxword);
  if (F < 0) return;
  const i64 stride = (i64)gridDim.x * blockDim.x;
  const i64 n2 = n / 2;
  double2* u2 = reinterpret_cast<double2*>(u);
  auto cvt = [&](double2 t) {
    double2 q;
    q.x = __longlong_as_double(fx_from(t.x, F));
    q.y = __longlong_as_double(fx_from(t.y, F));
    return q;
  };
  i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x;
  // four independent 16-byte loads in flight per thread (one resident wave)
  for (; i + 3 * stride < n2; i += 4 * stride) {
    double2 t[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) t[q] = u2[i + q * stride];
#pragma unroll
    for (int q = 0; q < 4; ++q) u2[i + q * stride] = cvt(t[q]);
  }
  for (; i < n2; i += stride) u2[i] = cvt(u2[i]);
  if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) u[n - 1] = __longlong_as_double(fx_from(u[n - 1], F));
}

// Writes NaN to resid[i] for i in [0, n) with (i + 1) % T != 0 and i != n-1:
// the sweeps a temporally blocked launch does not materialise.
__global__ void jacc_k_fill_skipped(double* resid, int n, int T) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n && ((i + 1) % T) != 0 && i != n - 1) resid[i] = __longlong_as_double(0x7ff8000000000000LL);
}

#endif  // JACC_AUX_KERNELS

// Minimum resident CTAs per SM asked of the compiler (the second launch
// bound) for a sweep kernel.  For the staged FP64 7-point kernel with 32 x 4
// threads (512^3, 200 sweeps): the constant-folded intermediate sweeps at 7
// CTAs (at most 72 registers, 5 stages of 5.4 KB) run 384.7 GLUP/s against
// 378.8 at 6; the precompiled intermediate sweeps spill at that bound (298.9)
// and, unbounded, take 124 registers (4 CTAs), so they ask for 6 (80
// registers, 6 stages); the converting sweeps at 5 CTAs (at most 102
// registers, from 157) take 2.40 ms for a 2-sweep sequence against 2.83.
// The 7-point kernels staged by asynchronous copies (scalar columns, 32 x 4
// threads): 5 CTAs (at most 102 registers); folded, 511^3 FP64 434 us a sweep
// against 445 unbounded (4 CTAs), 444 at 6 and 557 at 7 (spills).
// For the FP64 27-point kernel with 32 x 4 threads: 4 CTAs (at most 128
// registers); folded, 512^3: 490 us a sweep against 492 unbounded (3 CTAs)
// and 518 at 5 (spills).
// The precompiled staged FP32 27-point kernel: 7 CTAs (at most 72 registers;
// left alone it spills at 64).
// Table tiles of 256 or 512 threads with 16-byte columns, where a CTA fewer an
// SM costs a wave (us a sweep, unbounded / bounded): FP32 27-point of 512
// threads, 90 / 64 registers, tile 15 512^3 641 / 411, tile 21 192 x 160 x 144
// 72 / 48; FP32 7-point of 256, 80 / 64, tile 5 256^3 39 / 29 and 512^3 199 /
// 185 (64 x 60 x 62, where every CTA fits at once, 18.3 / 19.9); 5-point of 512,
// FP64 74 / 64, tile 13 4096^2 100 / 69, FP32 48 / 40, tile 21 31.8 / 29.1.
// Every other kernel: 0, no requirement (a bound of 1 is not neutral: it
// lets the compiler take registers for one CTA per SM, e.g. 111 instead of
// 80 for the staged FP32 7-point kernel).
template <int STENCIL, class T, int BX, int BY, int V, int FAM, bool EDGE, bool FOLDED> struct SweepMinBlocks {
  typedef Load3D<STENCIL, T, BX, BY, V, FAM, EDGE> K;
  static constexpr bool t32 = BX == 32 && BY == 4;
  static constexpr int heat = K::BULK ? (K::F64 ? (FOLDED ? 7 : 6) : 0) : K::RING ? (V == 1 || EDGE ? 5 : 6) : 0;
  static constexpr int box = FAM == JACC_FAM_NATIVE ? 0 : K::F64 ? (EDGE ? 0 : 4) : (V == 4 && !FOLDED ? 7 : 0);
  static constexpr bool wide = K::VEC && FAM == JACC_FAM_TABLE && !FOLDED && !EDGE;
  static constexpr int NT = BX * BY;
  static constexpr int wide5 = NT == 512 ? (K::F64 ? 2 : 3) : 0, wide7 = !K::F64 && NT == 256 ? 4 : 0,
                       wide27 = !K::F64 && NT == 512 ? 2 : 0;
  static constexpr int other = !wide ? 0 : STENCIL == 5 ? wide5 : STENCIL == 7 ? wide7 : wide27;
  static constexpr int value = !t32 ? other : STENCIL == 7 ? heat : STENCIL == 27 ? box : 0;
};

// The parameter block of a table tile's kernel.  The march length is a constant
// where the kernel marches rows or planes from registers or bulk copies: as an
// argument it costs registers, or the compiler moves the loads of the next
// plane to where they are used (us a sweep, argument / constant: FP32 27-point
// tile 0 512^3 893 / 730 and 192 x 160 x 144 35.2 / 25.9, FP64 5-point tile 7
// 4096^2 76.1 / 70.1).  Strips, rings and the kernel without staging take it as
// an argument.
template <class A, class B, bool FIRST> struct PickT { typedef A type; };
template <class A, class B> struct PickT<A, B, false> { typedef B type; };
template <int STENCIL, class T, int BX, int BY, int V, int ZC, bool NATIVE = false> struct TableP {
  typedef Load3D<STENCIL, T, BX, BY, V, JACC_FAM_TABLE, false> K;
  static constexpr bool FIXED = NATIVE || (STENCIL == 5 ? V > 1 : !(K::RING || K::DIRECT));
  typedef typename PickT<JParamsZ<STENCIL == 5 ? ZC / 4 : ZC>, JParams, FIXED>::type type;
};

// Kernel templates instantiated by the precompiled library.
template <class T, int BX, int BY, int V, int FAM, bool EDGE, class P>
__global__ void __launch_bounds__(BX * BY, (SweepMinBlocks<5, T, BX, BY, V, FAM, EDGE, false>::value))
    jacc_k_jacobi2d(const T* __restrict__ u, T* __restrict__ v, P p, double* resid, const u64* maxword, int flags) {
  jacobi2d_entry<T, BX, BY, V, FAM, EDGE>(u, v, p, p, resid, maxword, flags);
}
template <class T, int BX, int BY, int V, int FAM, bool EDGE, class P>
__global__ void __launch_bounds__(BX * BY, (SweepMinBlocks<7, T, BX, BY, V, FAM, EDGE, false>::value))
    jacc_k_heat3d(const T* __restrict__ u, T* __restrict__ v, P p, double* resid, const u64* maxword, int flags) {
  heat3d_entry<T, BX, BY, V, FAM, EDGE>(u, v, p, p, resid, maxword, flags);
}
template <class T, int BX, int BY, int V, int FAM, bool EDGE, class P>
__global__ void __launch_bounds__(BX * BY, (SweepMinBlocks<27, T, BX, BY, V, FAM, EDGE, false>::value))
    jacc_k_box27(const T* __restrict__ u, T* __restrict__ v, P p, double* resid, const u64* maxword, int flags) {
  box27_entry<T, BX, BY, V, FAM, EDGE>(u, v, p, p, resid, maxword, flags);
}
template <int RY, int TT, int ZC>
__global__ void __launch_bounds__(TB_BX * RY) jacc_k_box27_tb(const float* __restrict__ u, float* __restrict__ v,
                                                              JParams p, double* resid, const u64* maxword, int flags) {
  box27_tb_entry<RY, TT, ZC>(u, v, p, resid);
}
