// runtime.cpp - specialisation cache, launches and graph-captured sweeps.
//
// jacc_specialize follows the paper's kernel cache and specialisation
// (§3.1: code compiled once is cached and reused; §3.2.2: runtime-invariant
// parameters are substituted by constants, non-conflicting pointers are
// restrict).  Descriptors are canonicalised into a byte key; identical keys
// share one Kernel object with a reference count.  Without JACC_SPEC_JIT the
// kernel is one of the precompiled instantiations (extents and coefficients
// as arguments); with it, NVRTC compiles the same template with them folded.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>

#include "../kernels/tiles.h"
#include "jacc_internal.h"
#include "../kernels/jacobi_cluster.h"

extern "C" const void* const jacc_tab_5_64[JACC_NTILES];
extern "C" const void* const jacc_tab_5_32[JACC_NTILES];
extern "C" const void* const jacc_tab_7_64[JACC_NTILES];
extern "C" const void* const jacc_tab_7_32[JACC_NTILES];
extern "C" const void* const jacc_tab_27_64[JACC_NTILES];
extern "C" const void* const jacc_tab_27_32[JACC_NTILES];
extern "C" const void* const jacc_tab_5_64_out[JACC_NTILES];
extern "C" const void* const jacc_tab_5_32_out[JACC_NTILES];
extern "C" const void* const jacc_tab_7_64_out[JACC_NTILES];
extern "C" const void* const jacc_tab_7_32_out[JACC_NTILES];
extern "C" const void* const jacc_tab_27_64_out[JACC_NTILES];
extern "C" const void* const jacc_tab_27_32_out[JACC_NTILES];
extern "C" const void* const jacc_tab_27_64_w32[JACC_NTILES];
extern "C" const void* const jacc_tab_5_64_native[JACC_NTILES];
extern "C" const void* const jacc_tab_7_64_native[JACC_NTILES];
extern "C" const void* const jacc_tab_27_64_native[JACC_NTILES];
extern "C" const void* const jacc_tab_5_64_lib[6][2];
extern "C" const void* const jacc_tab_5_32_lib[6][2];
extern "C" const void* const jacc_tab_7_64_lib[6][2];
extern "C" const void* const jacc_tab_7_32_lib[6][2];
extern "C" const void* const jacc_tab_27_64_lib[6][2];
extern "C" const void* const jacc_tab_27_64_lib_w32[6][2];
extern "C" const void* const jacc_tab_27_32_lib[6][2];
extern "C" const void* const jacc_tab_tb[2];

namespace jacc {

static const TileCfg kTiles[JACC_NTILES] = {
#define JACC_TILE_ROW(id, BX, BY, VEC, ZC) {BX, BY, VEC, ZC},
    JACC_TILE_LIST(JACC_TILE_ROW)
#undef JACC_TILE_ROW
};

const TileCfg& tile_cfg(int id) { return kTiles[id]; }

static std::map<std::string, Kernel*>& cache() {
  static std::map<std::string, Kernel*> c;
  return c;
}

// d = m * 2^-k with m odd (d > 0 finite).  Returns false if d is not of
// that form with k in [0, 62].
static bool dyadic(double d, uint64_t* m, int* k) {
  if (!(d > 0.0) || !std::isfinite(d)) return false;
  int e = 0;
  double f = std::frexp(d, &e);  // d = f 2^e, f in [0.5, 1)
  uint64_t mm = static_cast<uint64_t>(std::ldexp(f, 53));
  int kk = 53 - e;
  while ((mm & 1u) == 0 && kk > 0) {
    mm >>= 1;
    --kk;
  }
  if ((mm & 1u) == 0 || kk > 62 || kk < 0) return false;
  *m = mm;
  *k = kk;
  return true;
}

static const void* table_entry(int stencil, int dtype, int tile, bool out) {
  const void* const* t = nullptr;
  if (stencil == 5) t = dtype == 64 ? (out ? jacc_tab_5_64_out : jacc_tab_5_64) : (out ? jacc_tab_5_32_out : jacc_tab_5_32);
  if (stencil == 7) t = dtype == 64 ? (out ? jacc_tab_7_64_out : jacc_tab_7_64) : (out ? jacc_tab_7_32_out : jacc_tab_7_32);
  if (stencil == 27)
    t = dtype == 64 ? (out ? jacc_tab_27_64_out : jacc_tab_27_64) : (out ? jacc_tab_27_32_out : jacc_tab_27_32);
  return t ? t[tile] : nullptr;
}

// Fills the fixed-point fields of p.  Returns the chosen path.
static int plan_fixed(const jacc_kernel_desc& d, JParams& p) {
  p.fpath = JACC_FP_NONE;
  if (d.dtype != JACC_F64 || d.arith != JACC_ARITH_AUTO) return p.fpath;
  if (d.stencil == JACC_STENCIL_5PT) {
    p.fpath = JACC_FP_JACOBI;
    p.fk = 2;
  } else if (d.stencil == JACC_STENCIL_7PT) {
    const double r = d.coeffs[0];
    if (r == 0.0) {
      p.fpath = JACC_FP_SMALL;
      p.fm = 0;
      p.fb = 0;
      p.fk = 0;
    } else if (r > 0.0 && r <= 1.0 / 6.0) {
      uint64_t m;
      int k;
      if (dyadic(r, &m, &k)) {
        p.fm = m << (62 - k);
        if (k <= 5) {
          p.fpath = JACC_FP_SMALL;
          p.fb = static_cast<i64>(m);
          p.fk = k;
        } else {
          p.fpath = JACC_FP_WIDE;
          p.fw0 = static_cast<i64>(m);
          p.fk = k;
        }
      }
    }
  } else if (d.stencil == JACC_STENCIL_27PT) {
    const double* w = d.coeffs;
    for (int j = 0; j < 4; ++j)
      if (!(w[j] >= 0.0) || !std::isfinite(w[j])) return p.fpath;
    const double W = w[0] + 6.0 * w[1] + 12.0 * w[2] + 8.0 * w[3];
    if (!(W <= 1.0 + std::ldexp(1.0, -20))) return p.fpath;
    uint64_t m[4] = {0, 0, 0, 0};
    int k[4] = {0, 0, 0, 0};
    int K = 0;
    for (int j = 0; j < 4; ++j) {
      if (w[j] == 0.0) continue;
      if (!dyadic(w[j], &m[j], &k[j])) return p.fpath;
      K = k[j] > K ? k[j] : K;
    }
    if (K > 62) return p.fpath;
    i64 f[4];
    for (int j = 0; j < 4; ++j) {
      if (w[j] == 0.0) {
        f[j] = 0;
        continue;
      }
      const int sh = K - k[j];
      if (sh >= 64 || (m[j] >> (63 - sh)) != 0) return p.fpath;  // factor must stay below 2^63
      f[j] = static_cast<i64>(m[j] << sh);
    }
    // weights with few bits (FP32 weights, say) take the kernel's 32-bit products
    bool narrow = K >= 1 && K <= 31;
    for (int j = 0; j < 4; ++j) narrow = narrow && f[j] < (static_cast<i64>(1) << 31);
    p.fpath = narrow ? JACC_FP_W32 : JACC_FP_WIDE;
    p.fw0 = f[0];
    p.fw1 = f[1];
    p.fw2 = f[2];
    p.fw3 = f[3];
    p.fk = K;
  }
  return p.fpath;
}

static jacc_status validate(const jacc_kernel_desc& d) {
  if (d.stencil != 5 && d.stencil != 7 && d.stencil != 27 && d.stencil != 19)
    return fail(JACC_ERR_INVALID_ARG, "unknown stencil");
  if (d.stencil == 19) {
    if (d.dtype != JACC_F32) return fail(JACC_ERR_UNSUPPORTED, "19-point variable-coefficient stencil: FP32 only");
    if (d.boundary != JACC_DIRICHLET) return fail(JACC_ERR_UNSUPPORTED, "19-point: Dirichlet only");
    if (d.nx % 4) return fail(JACC_ERR_UNSUPPORTED, "19-point: nx must be a multiple of 4 (16-byte rows)");
    if (d.flags) return fail(JACC_ERR_UNSUPPORTED, "19-point: no JIT or cluster variant");
    if (d.tblock > 1) return fail(JACC_ERR_UNSUPPORTED, "19-point: no temporal blocking");
    if (d.tile_id != -1) return fail(JACC_ERR_INVALID_ARG, "19-point: one fixed tile (tile_id must be -1)");
  }
  if (d.dtype != JACC_F32 && d.dtype != JACC_F64) return fail(JACC_ERR_INVALID_ARG, "dtype must be 32 or 64");
  if (d.tile_id < -1 || d.tile_id >= JACC_NTILES) return fail(JACC_ERR_INVALID_ARG, "tile_id out of range");
  if (d.arith != JACC_ARITH_AUTO && d.arith != JACC_ARITH_NATIVE) return fail(JACC_ERR_INVALID_ARG, "bad arith");
  if (d.flags & ~(JACC_SPEC_JIT | JACC_SPEC_CLUSTER)) return fail(JACC_ERR_INVALID_ARG, "unknown specialisation flags");
  if ((d.flags & JACC_SPEC_CLUSTER) && (d.stencil != 5 || d.dtype != JACC_F64))
    return fail(JACC_ERR_UNSUPPORTED, "JACC_SPEC_CLUSTER: 5-point FP64 only");
  if (d.nx < 3 || d.ny < 3 || d.nz < 1) return fail(JACC_ERR_INVALID_ARG, "extents must be >= 3");
  if (d.stencil == 5) {
    if (d.nz != 1) return fail(JACC_ERR_INVALID_ARG, "5-point stencil is 2D: nz must be 1");
    if (d.boundary != JACC_DIRICHLET) return fail(JACC_ERR_UNSUPPORTED, "5-point stencil supports Dirichlet only");
  } else {
    if (d.nz < 3) return fail(JACC_ERR_INVALID_ARG, "3D stencil: nz must be >= 3");
  }
  if (d.stencil == 7 && d.boundary != JACC_DIRICHLET) return fail(JACC_ERR_UNSUPPORTED, "7-point: Dirichlet only");
  if (d.stencil == 27 && d.boundary != JACC_PERIODIC) return fail(JACC_ERR_UNSUPPORTED, "27-point: periodic only");
  if (d.tblock < 0) return fail(JACC_ERR_INVALID_ARG, "tblock < 0");
  if (d.tblock > 1) {
    if (d.stencil != 27 || d.dtype != JACC_F32 || d.tblock > 3)
      return fail(JACC_ERR_UNSUPPORTED, "temporal blocking: 27-point FP32 with depth 2 or 3 only");
    if (d.nx % 4) return fail(JACC_ERR_UNSUPPORTED, "temporal blocking needs nx divisible by 4");
    if (d.flags & JACC_SPEC_JIT) return fail(JACC_ERR_UNSUPPORTED, "temporal blocking has no folded variant");
  }
  for (int j = 0; j < 4; ++j)
    if (!std::isfinite(d.coeffs[j])) return fail(JACC_ERR_INVALID_ARG, "non-finite coefficient");
  const double n = static_cast<double>(d.nx) * static_cast<double>(d.ny) * static_cast<double>(d.nz);
  if (n > 9.0e18) return fail(JACC_ERR_OVERFLOW, "element count overflows int64");
  return ok();
}

static const void* native_entry(int stencil, int tile) {
  return (stencil == 5 ? jacc_tab_5_64_native : stencil == 7 ? jacc_tab_7_64_native : jacc_tab_27_64_native)[tile];
}

// The library's own kernel (entry `row` of its table), or null.
static const void* lib_entry(const jacc_kernel_desc& d, const JParams& p, int row, bool vec) {
  const bool f64 = d.dtype == 64;
  if (d.stencil == 5) return (f64 ? jacc_tab_5_64_lib : jacc_tab_5_32_lib)[row][vec];
  if (d.stencil == 7) return (f64 ? jacc_tab_7_64_lib : jacc_tab_7_32_lib)[row][vec];
  if (!f64) return jacc_tab_27_32_lib[row][vec];
  return (p.fpath == JACC_FP_W32 ? jacc_tab_27_64_lib_w32 : jacc_tab_27_64_lib)[row][vec];
}

// The default tile: 32 x 4 threads, 16-byte columns where nx allows.  2D: they
// pay from 2^18 points on (4096^2 FP64: 50.0 us a sweep, 62.5 with scalar
// columns); below, more, narrower strips hide latency better (300^2: 2.04 us).
// 3D: the long march where it yields at least 1024 CTAs.
int default_tile(const jacc_kernel_desc& d) {
  const int V = d.dtype == 64 ? 2 : 4;
  const bool vec_ok = (d.nx % V) == 0;
  if (d.stencil == 5) return vec_ok && d.nx * d.ny >= (int64_t(1) << 18) ? 3 : 2;
  const int64_t w = 32 * (vec_ok ? V : 1);  // columns of a 32 x 4 tile
  const int64_t ctas_long = ((d.nx + w - 1) / w) * ((d.ny + 7) / 8) * ((d.nz + 63) / 64);
  if (ctas_long >= 1024) return vec_ok ? 3 : 2;
  return vec_ok ? 1 : 0;
}

// Whether the descriptor's sweeps always run native FP64 arithmetic.
static bool native_fp64(const jacc_kernel_desc& d, int fpath) {
  return d.dtype == 64 && d.stencil != 19 && fpath == JACC_FP_NONE;
}

// CTAs that a grid holds at most in y and in z.
constexpr int64_t kGridYZ = 65535;

// Whether the few planes per CTA of the kernel without staging keep its grid
// within that limit (up to 131070 planes; a loop over the rest in the kernel
// itself cost every grid 5 to 15 %).
static bool direct_fits(const jacc_kernel_desc& d) {
  return (d.nz + JACC_DIRECT_PLANES - 1) / JACC_DIRECT_PLANES <= kGridYZ;
}

// The kernel family of a table tile: its own kernel, but the ring for the
// tiles that stage nothing where those would take too many CTAs, or where the
// grid is too large for them (FP64, see default_family: 192 x 160 x 144 26.9 us a
// sweep without staging, 22.4 with the ring; 512^3 798 and 480).
static int table_family(const jacc_kernel_desc& d, int tile, int fpath) {
  const TileCfg& c = kTiles[tile];
  const bool direct = d.stencil == 7 && JACC_DIRECT_TILE(c.bx, c.by, c.vec16 ? 2 : 1), fits = direct_fits(d);
  const int64_t n = d.nx * d.ny * d.nz;
  // native FP64, us a sweep of tile 4 without staging and with its planes in
  // registers: 33^3 5.4 / 22, 101^3 31 / 43, 128^3 46 / 58, 192 x 160 x 144
  // 95 / 108
  if (native_fp64(d, fpath)) return direct && fits && n <= (int64_t(1) << 24) ? JACC_FAM_TABLE : JACC_FAM_NATIVE;
  const bool large = d.dtype == 64 && n > (int64_t(1) << 20);
  return direct && (large || !fits) ? JACC_FAM_RING : JACC_FAM_TABLE;
}

// Whether the planes per CTA are fitted to the grid: kernels of the library's
// choice, and the FP64 scalar 7-point tiles, whose ring covers four rows per
// thread: with all of the tile's planes small grids do not fill the GPU (us a
// sweep, all / fitted, but with no fewer points per CTA than one row per thread
// had: 64 x 60 x 62 tile 10 37.9 / 14.9, 192 x 160 x 144 39.7 / 20.6; large
// grids take all of them either way).
static bool fits_planes(const jacc_kernel_desc& d, int tile, int fam, bool fit) {
  return fit || (d.stencil == 7 && d.dtype == 64 && !kTiles[tile].vec16 && fam != JACC_FAM_NATIVE);
}

// The kernel family of the library's own choice.  7-point grids that live in
// L2 need no staging (us a sweep without / with the ring: FP32 64^3 1.8 / 3.3,
// 128^3 4.2 / 4.9, 160^3 9.9 / 10.4, 216^3 18.0 / 16.0; FP64 64^3 3.1 / 5.4,
// 128^3 9.9 / 10.4, 160^3 20.9 / 19.5; scalar columns FP32 81^3 3.7 / 4.1,
// 97^3 5.5 / 4.8, FP64 97^3 8.8 / 9.1, 129^3 16.9 / 12.8).  Folded kernels of
// fields that stream from HBM stage by bulk copies (bulk / ring: 7-point FP64
// 512^3 361 / 398, 320^3 98 / 95; FP32 512^3 164 / 189, 400^3 92 / 92; 27-point
// FP32 768^3 573 / 610, 512^3 190 / 179), of the precompiled ones only the FP32
// 7-point kernel (512^3 164 / 170); the rest asynchronous copies (precompiled,
// ring / bulk: 7-point FP64 512^3 396 / 480, 27-point FP32 768^3 604 / 748).
static int default_family(const jacc_kernel_desc& d, int tile, bool native) {
  if (d.tblock > 1 || d.stencil == 19) return JACC_FAM_TABLE;
  if (d.stencil == 5) return JACC_FAM_STRIP;
  const bool vec = kTiles[tile].vec16, f64 = d.dtype == 64;
  const int64_t n = d.nx * d.ny * d.nz;
  if (d.stencil == 7) {
    const int64_t direct = vec ? (f64 ? int64_t(1) << 21 : int64_t(1) << 22) : (f64 ? int64_t(1) << 20 : int64_t(5) << 17);
    if (n <= (native ? int64_t(1) << 24 : direct) && direct_fits(d)) return JACC_FAM_DIRECT;  // native: see default_tile_native
  }
  const bool bulk = d.stencil == 7 ? n * (f64 ? 8 : 4) >= (int64_t(1) << 28) : !f64 && n * 4 >= (int64_t(1) << 30);
  const bool pays = (d.flags & JACC_SPEC_JIT) || (d.stencil == 7 && !f64);
  return tile == 3 && bulk && pays ? JACC_FAM_BULK : JACC_FAM_RING;
}

// The library's own choice for native FP64 sweeps: the tile, and whether it is
// left as it is (JACC_FAM_NATIVE) or given to the family and march of the fixed-
// point sweeps of the same size (*own).  The latter bring more, shorter CTAs,
// which small grids need, but more work for the FP64 pipe, which bounds large
// ones (us a sweep, own / native: 5-point 256^2 3.2 / 5.0, 100 x 6000 14 / 26,
// 1024^2 23 / 22, 4096^2 288 / 259; 7-point without staging 64^3 9.0 / 22, 128^3
// 48 / 67, 192 x 160 x 144 96 / 107, 256^3 353 / 370;
// 27-point 64^3 23 / 27, 97 x 81 x 85 52 / 46).
static int default_tile_native(const jacc_kernel_desc& d, bool* own) {
  const int tile = default_tile(d);
  const int64_t n = d.nx * d.ny * d.nz;
  if (d.stencil == 5) {
    *own = n < (int64_t(1) << 20) || d.nx <= 384;  // 256 columns a CTA otherwise
    const int rows = d.nx % 2 ? 16 : 17;  // 128 x 2 threads, four rows each
    return !*own && tile_valid(d, rows) ? rows : tile;
  }
  *own = d.stencil == 7 ? default_family(d, tile, true) == JACC_FAM_DIRECT : n <= (int64_t(1) << 18);
  return tile;
}

// What a CTA of kernel family `fam` covers per plane (columns, rows), and how
// many planes (3D) or rows per thread row (2D) it marches.
struct CtaTile {
  int64_t cols, rows, march;
};
static CtaTile cta_tile(const jacc_kernel_desc& d, int tile, int fam, bool edge, int zc) {
  const TileCfg& c = kTiles[tile];
  const int V = c.vec16 ? (d.dtype == 64 ? 2 : 4) : 1;
  const CtaTile rows{static_cast<int64_t>(c.bx) * V, c.by, zc};
  if (d.stencil == 5) {
    const bool small = (d.flags & JACC_SPEC_JIT) && d.nx * d.ny <= JACC_SMALL_GRID;
    const bool strips = small || (fam != JACC_FAM_NATIVE && (fam == JACC_FAM_STRIP || V == 1));
    return strips ? CtaTile{static_cast<int64_t>(c.bx / 32) * 30 * V, c.by, zc} : rows;
  }
  if (fam == JACC_FAM_NATIVE) return rows;
  const bool f64 = d.dtype == 64;
  if (d.stencil == 7 && !edge && (fam == JACC_FAM_DIRECT || (fam == JACC_FAM_TABLE && JACC_DIRECT_TILE(c.bx, c.by, V))))
    return CtaTile{static_cast<int64_t>(32) * V, 8, JACC_DIRECT_PLANES};
  // one column of JACC_RING_ROWS rows per thread
  if ((d.stencil == 27 && f64) || (V == 1 && (f64 || fam == JACC_FAM_RING))) return CtaTile{c.bx, c.by * JACC_RING_ROWS(c.bx, c.by), zc};
  if (V == 1) return CtaTile{c.bx, c.by, zc};               // FP32 table tiles of scalar columns
  return CtaTile{static_cast<int64_t>(c.bx) * V, c.by * 2, zc};  // a 16-byte column of two rows
}
static dim3 cta_grid(const jacc_kernel_desc& d, const CtaTile& t) {
  auto up = [](int64_t a, int64_t b) { return static_cast<unsigned>((a + b - 1) / b); };
  if (d.stencil == 5) return dim3(up(d.nx, t.cols), up(d.ny, t.rows * t.march), 1);
  return dim3(up(d.nx, t.cols), up(d.ny, t.rows), up(d.nz, t.march));
}
// The least planes per CTA that keep a 3D grid within its limit in z: more
// than the tile's own where the library's kernels march fewer (131071 planes
// upwards).
static int least_chunk(const jacc_kernel_desc& d) {
  return d.stencil == 5 ? 1 : static_cast<int>((d.nz + kGridYZ - 1) / kGridYZ);
}

bool tile_valid(const jacc_kernel_desc& d, int t) {
  const TileCfg& c = kTiles[t];
  const int V = c.vec16 ? (d.dtype == 64 ? 2 : 4) : 1;
  if (d.nx % V) return false;
  // grid-dimension limits
  const int64_t gy = d.stencil == 5 ? (d.ny + c.by * (c.zc / 4) - 1) / (c.by * (c.zc / 4)) : (d.ny + c.by - 1) / c.by;
  const int64_t gz = d.stencil == 5 ? 1 : (d.nz + c.zc - 1) / c.zc;
  const int64_t gx = (d.nx + c.bx * V - 1) / (c.bx * V);
  return gx < (1ll << 31) && gy <= kGridYZ && gz <= kGridYZ;
}

static std::string key_of(const jacc_kernel_desc& d, int tile, bool fit, int named) {
  jacc_kernel_desc c = d;
  c.tile_id = tile;
  c.reserved = 0;
  if (c.tblock == 0) c.tblock = 1;
  return std::string(reinterpret_cast<const char*>(&c), sizeof(c)) + (fit ? "f" : "t") + std::to_string(named);
}

// Planes per CTA (3D) or rows per warp (2D) of a kernel that takes what fits
// the grid.  3D: at most the tile's own, and few enough that the grid has at
// least 2.5 times the CTAs that the device holds at once.  With fewer, the last wave leaves SMs
// idle: 301 x 253 x 199 FP64 at 64 planes (640 CTAs on 152 SMs) 65.2 us a
// sweep, at 16 planes (2080) 55.7, at 8 (4000) 57.3; 511^3, whose grid is
// large either way, within 3 % from 8 to 64.
static int fitted_chunk(const Kernel& k, int zc) {
  int dev = 0, nsm = 0, per = 6;  // a folded kernel is compiled for its chunk: 5 to 8 of them fit an SM
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      (k.func && cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k.func, static_cast<int>(k.block.x * k.block.y), 0) !=
                     cudaSuccess)) {
    cudaGetLastError();
    return zc;
  }
  const int64_t slots = static_cast<int64_t>(nsm) * (per > 0 ? per : 1);
  if (k.desc.stencil == 5) {
    // rows per warp, 2 to the tile's own: a strip's start-up (three rows of
    // loads before the first result) costs more than an unfilled wave, so 0.6
    // of the slots are enough (1000^2 FP64: 4.42 us a sweep at 8 rows, 544
    // CTAs; 4.87 at 4, 5.2 at 16)
    const int64_t rows = 10ll * k.grid.x * k.desc.ny / (6ll * slots * k.block.y);
    // twice the tile's own for the deep march of large folded FP64 grids
    // (4096^2: 45.8 us a sweep at 32 rows, 46.5 at 16, 51.3 at 64)
    if (!k.func && k.vec == 2 && k.desc.nx * k.desc.ny > JACC_LARGE_GRID && rows >= 2 * zc) return 2 * zc;
    return static_cast<int>(rows >= zc ? zc : (rows < 2 ? 2 : rows));
  }
  const int64_t columns = static_cast<int64_t>(k.grid_out.x) * k.grid_out.y;
  const int64_t want = (5 * slots / 2 + columns - 1) / columns;  // chunks
  const int64_t fit = (k.desc.nz + want - 1) / want;
  // no fewer than 4 planes, 8 for 27-point grids that are not small (their
  // halo planes cost most: FP32 64^3 3.6 us a sweep at 4, 5.0 at 8; 128^3 7.5
  // at 4, 7.0 at 8; FP64 96^3 7.3 and 8.6, 112^3 12.8 and 10.8)
  const int64_t n = k.desc.nx * k.desc.ny * k.desc.nz;
  const int least = k.desc.stencil == 7 || n <= (int64_t(1) << (k.desc.dtype == 64 ? 20 : 19)) ? 4 : 8;
  return static_cast<int>(fit >= zc ? zc : (fit < least ? least : fit));
}
// Planes per CTA of the converting 3D kernel (single launches, the first and
// last sweep of a sequence) under the same condition.  It is bound by its
// integer work, its CTAs take equally long and few waves of them run, so the
// waves are filled: the chunk with the least waves * (planes + 3 to start up),
// between 4 and 32 planes (256^3 heat, one launch: 145 us at 24 planes, 1.85
// waves; 165 at 14, 3.2 waves; 163 at 32, 1.35; 301 x 253 x 199: 153 at 24,
// 174 at 14 and at 32).
static int fitted_chunk_out(const Kernel& k, int zc) {
  int dev = 0, nsm = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k.func_out, static_cast<int>(k.block_out.x * k.block_out.y), 0) !=
          cudaSuccess ||
      per < 1) {
    cudaGetLastError();
    return zc;
  }
  const int64_t columns = static_cast<int64_t>(k.grid_out.x) * k.grid_out.y, slots = static_cast<int64_t>(nsm) * per;
  int64_t least = INT64_MAX;
  int best = zc;
  for (int z = 32; z >= 4; --z) {
    const int64_t chunks = (k.desc.nz + z - 1) / z;
    if (chunks > kGridYZ) break;
    const int64_t cost = (columns * chunks + slots - 1) / slots * (z + 3);
    if (cost < least) {
      least = cost;
      best = z;
    }
  }
  return best;
}


// Planes per CTA of a 3D kernel.  The constant-folded variants of the bulk-copy
// staged tiles with the long march take fewer planes than the table's 64: with
// the extents folded their kernels need fewer registers and more CTAs fit, and
// shallower chunks then balance better.  Measured with tile 3: heat 512^3 FP64
// best at 40 planes (396.8 against 392.1 GLUP/s at 64), 27-point 1024^3 FP32
// best at 24-32 (128.6 ms for 100 sweeps at 32 against 144.7 at 64).  The
// library's own 7-point kernels take at most 16 planes in FP32 (512^3, us a
// sweep at 12 / 16 / 24 / 32 / 64 planes: ring 170 / 170 / 174 / 178 / 181,
// bulk 162 / 164 / 164 / 166 / 184) and 24 in FP64 (ring 414 / 410 / 396 / 400 /
// 403): the CTAs that share a halo row then stay closer together.
static int plane_chunk(const jacc_kernel_desc& d, int tile, int fam) {
  const TileCfg& c = kTiles[tile];
  if (d.stencil == 5) return c.zc / 4;  // rows per warp
  const bool f64 = d.dtype == 64;
  if (fam == JACC_FAM_NATIVE) return c.zc;
  if (d.stencil == 7 && !f64 && (fam == JACC_FAM_RING || fam == JACC_FAM_BULK)) return 16;
  if (d.stencil == 7 && f64 && fam == JACC_FAM_RING) return c.zc < 24 ? c.zc : 24;
  const bool bulk = c.vec16 && !(d.stencil == 27 && f64) && (fam == JACC_FAM_TABLE || fam == JACC_FAM_BULK);
  if ((d.flags & JACC_SPEC_JIT) && bulk && c.zc == 64) return d.stencil == 27 ? 32 : 40;
  return c.zc;
}

// The NVRTC source of a folded variant: the device text plus a struct whose
// static constexpr members replace JParams, and the kernels: jacc_jit for the
// intermediate (and every FP32 or native) sweeps, and in fixed point
// jacc_jit_out, which converts FP64 on load and store, and jacc_jit_last, only on
// store.
static std::string jit_source(const Kernel& k) {
  const JParams& p = k.params;
  const TileCfg& c = kTiles[k.tile];
  const int st = k.desc.stencil;
  const std::string T = k.desc.dtype == 64 ? "double" : "float";
  char fold[1024];
  std::snprintf(fold, sizeof(fold),
                "\nstruct JFold {\n"
                "  static constexpr i64 nx = %lldll, ny = %lldll, nz = %lldll;\n"
                "  static constexpr double c0 = %a, c1 = %a, c2 = %a, c3 = %a;\n"
                "  static constexpr u64 fm = %lluull;\n"
                "  static constexpr i64 fb = %lldll;\n"
                "  static constexpr i64 fw0 = %lldll, fw1 = %lldll, fw2 = %lldll, fw3 = %lldll;\n"
                "  static constexpr int fk = %d, fpath = %d, zc = %d;\n"
                "};\n",
                (long long)p.nx, (long long)p.ny, (long long)p.nz, p.c0, p.c1, p.c2, p.c3, (unsigned long long)p.fm,
                (long long)p.fb, (long long)p.fw0, (long long)p.fw1, (long long)p.fw2, (long long)p.fw3, p.fk, p.fpath, p.zc);
  // the kernel without staging has 32 x 8 threads, the converting sweeps the tile's
  auto shape = [&](int fam, bool edge) {
    const bool direct = fam == JACC_FAM_DIRECT && !edge;
    return T + ", " + std::to_string(direct ? 32 : c.bx) + ", " + std::to_string(direct ? 8 : c.by) + ", " + std::to_string(k.vec);
  };
  auto tail = [&](int fam, bool edge) { return ", " + std::to_string(fam) + (edge ? ", true" : ", false"); };
  auto call = [&](int fam, bool edge, const char* flags) {
    return std::string(st == 5 ? "jacobi2d_entry<" : st == 7 ? "heat3d_entry<" : "box27_entry<") + shape(fam, edge) +
           tail(fam, edge) + ">(u, v, f, rt, resid, maxword, " + flags + ")";
  };
  auto kernel = [&](const char* name, int threads, const std::string& bound, const std::string& body) {
    return "extern \"C\" __global__ void __launch_bounds__(" + std::to_string(threads) + bound + ")\n" + name + "(const " + T +
           "* __restrict__ u, " + T + "* __restrict__ v, JParams rt, double* resid, const u64* maxword, int flags) {\n" +
           "  const JFold f{};\n  " + body + ";\n}\n";
  };
  auto bound = [&](int fam, bool edge) {
    if (st == 5) return std::string();
    return ", (SweepMinBlocks<" + std::to_string(st) + ", " + shape(fam, edge) + tail(fam, edge) + ", true>::value)";
  };
  std::string src = std::string(device_source()) + fold;
  src += kernel("jacc_jit", k.fam == JACC_FAM_DIRECT ? 256 : c.bx * c.by, bound(k.fam, false), call(k.fam, false, "flags"));
  if (k.desc.dtype == 64 && p.fpath != JACC_FP_NONE) {
    src += kernel("jacc_jit_out", c.bx * c.by, bound(k.fam, true), call(k.fam, true, "flags"));
    src += kernel("jacc_jit_last", c.bx * c.by, bound(k.fam, true), call(k.fam, true, "JFX_OUT_F64"));
  }
  return src;
}

static void free_kernel(Kernel* k) {
  for (auto& g : k->graphs) {
    if (g.second.exec) cudaGraphExecDestroy(g.second.exec);
    if (g.second.graph) cudaGraphDestroy(g.second.graph);
    if (g.second.scratch) cudaFree(g.second.scratch);
  }
  k->graphs.clear();
  for (auto& g : k->coeff_graphs) {
    if (g.second.exec) cudaGraphExecDestroy(g.second.exec);
    if (g.second.graph) cudaGraphDestroy(g.second.graph);
  }
  k->coeff_graphs.clear();
  free_until_graphs(*k);
  if (k->scratch) cudaFree(k->scratch);
  if (k->lib) cudaLibraryUnload(k->lib);
  delete k;
}

}  // namespace jacc

using namespace jacc;

extern "C" jacc_status jacc_tile_info(int32_t tile_id, jacc_tile* out) {
  if (tile_id < 0 || tile_id >= JACC_NTILES || !out) return fail(JACC_ERR_INVALID_ARG, "bad tile_id or NULL out");
  const TileCfg& c = kTiles[tile_id];
  out->bx = c.bx;
  out->by = c.by;
  out->vec16 = c.vec16;
  out->zc = c.zc;
  return ok();
}

static jacc_status specialize(const jacc_kernel_desc* desc, const TunedPick& pick, jacc_kernel* out);

extern "C" jacc_status jacc_specialize(const jacc_kernel_desc* desc, jacc_kernel* out) {
  if (!desc || !out) return fail(JACC_ERR_INVALID_ARG, "NULL descriptor or output");
  const jacc_status st = validate(*desc);
  return st ? st : specialize(desc, desc->tile_id < 0 && desc->stencil != 19 ? tuned_pick(*desc) : TunedPick(), out);
}

jacc_status jacc::specialize_own(const jacc_kernel_desc& desc, jacc_kernel* out) {
  const jacc_status st = validate(desc);
  return st ? st : specialize(&desc, TunedPick(), out);
}

// pick: the autotuner's, where no tile is asked for.
static jacc_status specialize(const jacc_kernel_desc* desc, const TunedPick& pick, jacc_kernel* out) {
  jacc_status st = ok();
  JParams plan{};
  plan_fixed(*desc, plan);
  const bool native = native_fp64(*desc, plan.fpath);
  int tile = desc->tile_id;
  int named = -1;    // the tile that jacc_kernel_info names, if not the kernel's
  bool fit = false;  // the library picks the kernel family and the march along with the tile
  if (desc->stencil == 19) {
    tile = 3;  // the kernel's one configuration: 32 x 4 threads, 16-byte columns, 40-plane march
  } else if (tile < 0) {
    const bool picked = pick.tile >= 0 && tile_valid(*desc, pick.tile);
    if (picked && (pick.ahead || desc->tblock > 1)) {
      tile = pick.tile;
    } else {
      bool own = true;
      tile = native ? default_tile_native(*desc, &own) : default_tile(*desc);
      fit = desc->tblock <= 1 && own;
      if (picked) named = pick.tile;
      if (picked && !tile_valid(*desc, tile)) {  // only larger tiles cover so many rows
        tile = pick.tile;
        fit = false;
      }
    }
  }
  if (!tile_valid(*desc, tile))
    return fail(JACC_ERR_INVALID_ARG, "tile " + std::to_string(tile) + " does not fit this shape (x vector width)");
  if (named < 0) named = tile;
  const std::string key = key_of(*desc, tile, fit, named);
  std::lock_guard<std::mutex> lock(global_mutex());
  auto it = cache().find(key);
  if (it != cache().end()) {
    it->second->refcount++;
    *out = reinterpret_cast<jacc_kernel>(it->second);
    return ok();
  }
  std::unique_ptr<Kernel> k(new Kernel());
  k->desc = *desc;
  k->desc.tile_id = tile;
  k->key = key;
  k->tile = tile;
  k->named = named;
  k->elem = desc->dtype / 8;
  const TileCfg& c = kTiles[tile];
  k->vec = c.vec16 ? 16 / k->elem : 1;
  JParams& p = k->params;
  p = plan;
  p.nx = desc->nx;
  p.ny = desc->ny;
  p.nz = desc->nz;
  p.c0 = desc->coeffs[0];
  p.c1 = desc->coeffs[1];
  p.c2 = desc->coeffs[2];
  p.c3 = desc->coeffs[3];
  k->fam = fit ? default_family(*desc, tile, native) : table_family(*desc, tile, p.fpath);
  const int fam = k->fam;
  // fixed-point sequences convert in their first and last sweeps, which have a kernel of their own
  const bool edge = desc->dtype == 64 && !native;
  k->block_out = dim3(c.bx, c.by, 1);
  k->block = fam == JACC_FAM_DIRECT ? dim3(32, 8, 1) : k->block_out;
  if (!(desc->flags & JACC_SPEC_JIT) && desc->stencil != 19 && desc->tblock <= 1) {
    k->func = fam == JACC_FAM_NATIVE  ? native_entry(desc->stencil, tile)
              : fam == JACC_FAM_TABLE ? table_entry(desc->stencil, desc->dtype, tile, false)
                                      : lib_entry(*desc, p, fit ? fam : 5, k->vec > 1);
    if (fam == JACC_FAM_TABLE && p.fpath == JACC_FP_W32) k->func = jacc_tab_27_64_w32[tile];
    k->func_out = !edge ? k->func
                  : fam == JACC_FAM_STRIP ? lib_entry(*desc, p, 5, k->vec > 1)
                                          : table_entry(desc->stencil, desc->dtype, tile, true);
    if (!k->func || !k->func_out) return fail(JACC_ERR_UNSUPPORTED, "no precompiled kernel for this descriptor");
  }
  p.zc = plane_chunk(*desc, tile, fam);
  k->grid = k->grid_out = cta_grid(*desc, cta_tile(*desc, tile, fam, edge, p.zc));
  if (fits_planes(*desc, tile, fam, fit)) {
    // a table tile keeps its points per CTA, and with them the tiles their order
    const int least = fit ? 1 : p.zc / JACC_RING_ROWS(c.bx, c.by);
    p.zc = std::max(fitted_chunk(*k, p.zc), least);
    if (desc->stencil == 5)
      while ((desc->ny + c.by * p.zc - 1) / (c.by * p.zc) > kGridYZ) p.zc *= 2;  // the grid's limit
  }
  if (desc->stencil != 19 && desc->tblock <= 1) p.zc = std::max(p.zc, least_chunk(*desc));
  k->zc_out = fit && edge && k->func_out && desc->stencil != 5 ? fitted_chunk_out(*k, p.zc) : p.zc;
  k->grid_out = cta_grid(*desc, cta_tile(*desc, tile, fam, edge, k->zc_out));
  k->grid = cta_grid(*desc, cta_tile(*desc, tile, fam, false, p.zc));
  if (desc->stencil == 19) {
    var19_geometry(desc->nx, desc->ny, desc->nz, &k->grid, &k->block);
    k->func = k->func_out = nullptr;  // launched by jacc_sweep_coeffs only
  } else if (desc->tblock == 2) {
    // two sweeps per launch, staged: 320 threads over a 128 x 16 output tile,
    // 64-plane chunks (box27_tb2.cu)
    k->tblock = 2;
    st = cuda_check(box27_tb2_setup(), "cudaFuncSetAttribute(two-sweep 27-point kernel)");
    if (st) return st;
    k->func = k->func_out = box27_tb2_kernel();
    k->block = box27_tb2_block();
    k->grid = box27_tb2_grid(desc->nx, desc->ny, desc->nz);
    k->smem = box27_tb2_smem();
  } else if (desc->tblock > 1) {
    // temporally blocked 27-point kernel: 32 x 16 threads over a 128 x 16 region,
    // output tile 120 x (16 - 2T), 64-plane chunks
    const int T = desc->tblock;
    k->tblock = T;
    k->func = jacc_tab_tb[T - 2];
    k->block = dim3(32, 16, 1);
    const int64_t oy = 16 - 2 * T;
    k->grid = dim3(static_cast<unsigned>((desc->nx + 119) / 120), static_cast<unsigned>((desc->ny + oy - 1) / oy),
                   static_cast<unsigned>((desc->nz + 63) / 64));
    k->func_out = k->func;
  } else if (desc->flags & JACC_SPEC_JIT) {
    static const char* const names[3] = {"jacc_jit", "jacc_jit_out", "jacc_jit_last"};
    const void* f[3] = {nullptr, nullptr, nullptr};
    st = jit_compile(jit_source(*k), names, edge ? 3 : 1, &k->lib, f, &k->compile_ms);
    if (st) return st;
    k->func = f[0];
    k->func_out = edge ? f[1] : f[0];
    k->func_last = f[2];  // fixed point only
    k->jit = true;
  }
  if (!edge) {
    k->grid_out = k->grid;
    k->block_out = k->block;
  }
  if (desc->flags & JACC_SPEC_CLUSTER) {
    int nc = 0;
    if (!jacobi_cluster_plan(desc->nx, desc->ny, &nc)) {
      if (k->lib) cudaLibraryUnload(k->lib);
      return fail(JACC_ERR_UNSUPPORTED, "JACC_SPEC_CLUSTER: the grid does not fit one cluster's shared memory");
    }
    k->cluster_nc = nc;
  }
  // scratch words: [0] max|u| bits of direct FP64 fixed-point launches, [1] the
  // device status word of bounded waits (JACC_DEV_TIMEOUT)
  st = cuda_check(cudaMalloc(reinterpret_cast<void**>(&k->scratch), 256), "cudaMalloc(scratch)");
  if (!st) st = cuda_check(cudaMemset(k->scratch, 0, 256), "cudaMemset(scratch)");
  if (st) {
    if (k->scratch) cudaFree(k->scratch);
    if (k->lib) cudaLibraryUnload(k->lib);
    return st;
  }
  p.status = reinterpret_cast<int*>(k->scratch + 1);
  p.timeout_ns = kDefaultTimeoutNs;
  p.stall_plane = -1;
  k->refcount = 1;
  Kernel* raw = k.release();
  cache()[key] = raw;
  *out = reinterpret_cast<jacc_kernel>(raw);
  return ok();
}

extern "C" jacc_status jacc_kernel_status(jacc_kernel h, int32_t* status) {
  if (!h || !status) return fail(JACC_ERR_INVALID_ARG, "NULL handle or output");
  const Kernel& k = *reinterpret_cast<Kernel*>(h);
  jacc_status st = cuda_check(cudaDeviceSynchronize(), "cudaDeviceSynchronize");
  if (st) return st;
  int v = 0;
  st = cuda_check(cudaMemcpy(&v, k.params.status, sizeof(int), cudaMemcpyDeviceToHost), "read status word");
  if (!st) st = cuda_check(cudaMemset(k.params.status, 0, sizeof(int)), "clear status word");
  if (st) return st;
  *status = v;
  return ok();
}

extern "C" jacc_status jacc_kernel_set_wait(jacc_kernel h, int32_t timeout_ms, int32_t stall_plane) {
  if (!h) return fail(JACC_ERR_INVALID_ARG, "NULL handle");
  if (timeout_ms < 0 || stall_plane < -1) return fail(JACC_ERR_INVALID_ARG, "timeout_ms < 0 or stall_plane < -1");
  std::lock_guard<std::mutex> lock(global_mutex());
  Kernel& k = *reinterpret_cast<Kernel*>(h);
  k.params.timeout_ns = timeout_ms == 0 ? kDefaultTimeoutNs : static_cast<int64_t>(timeout_ms) * 1000000;
  k.params.stall_plane = stall_plane;
  // cached graphs hold the old parameters: drop them
  for (auto& g : k.graphs) {
    if (g.second.exec) cudaGraphExecDestroy(g.second.exec);
    if (g.second.graph) cudaGraphDestroy(g.second.graph);
    if (g.second.scratch) cudaFree(g.second.scratch);
  }
  k.graphs.clear();
  free_until_graphs(k);
  return ok();
}

extern "C" jacc_status jacc_kernel_info(jacc_kernel h, jacc_kernel_info_t* out) {
  if (!h || !out) return fail(JACC_ERR_INVALID_ARG, "NULL handle or output");
  const Kernel& k = *reinterpret_cast<Kernel*>(h);
  out->tile_id = k.named;
  out->jit = k.jit ? 1 : 0;
  out->fixed_point = k.params.fpath != JACC_FP_NONE ? 1 : 0;
  out->tblock = k.tblock;
  out->block[0] = static_cast<int32_t>(k.block.x);
  out->block[1] = static_cast<int32_t>(k.block.y);
  out->block[2] = static_cast<int32_t>(k.block.z);
  out->grid[0] = static_cast<int32_t>(k.grid.x);
  out->grid[1] = static_cast<int32_t>(k.grid.y);
  out->grid[2] = static_cast<int32_t>(k.grid.z);
  out->compile_ms = k.compile_ms;
  return ok();
}

extern "C" jacc_status jacc_release(jacc_kernel h) {
  if (!h) return fail(JACC_ERR_INVALID_ARG, "NULL handle");
  std::lock_guard<std::mutex> lock(global_mutex());
  Kernel* k = reinterpret_cast<Kernel*>(h);
  auto it = cache().find(k->key);
  if (it == cache().end() || it->second != k) return fail(JACC_ERR_INVALID_ARG, "unknown or released handle");
  if (--k->refcount > 0) return ok();
  cache().erase(it);
  free_kernel(k);
  return ok();
}

extern "C" jacc_status jacc_shutdown(void) {
  std::lock_guard<std::mutex> lock(global_mutex());
  for (auto& e : cache()) free_kernel(e.second);
  cache().clear();
  static_scratch_forget();
  return ok();
}

// ---------------------------------------------------------------- launches

namespace jacc {

cudaError_t launch_sweep_kernel(const Kernel& k, const void* u, void* v, double* resid, const u64* maxword, int flags,
                                cudaStream_t s, const int* stop) {
  JParams p = k.params;
  p.stop = stop;
  const void* args[] = {&u, &v, &p, &resid, &maxword, &flags};
  // programmatic dependent launch: the kernel may start while the previous
  // sweep finishes; every sweep kernel waits (griddepcontrol.wait) for the
  // previous grid before it touches a field
  cudaLaunchConfig_t cfg = {};
  const bool edge = (flags & (kFxIn | kFxOut)) != 0;
  if (edge) p.zc = k.zc_out;
  cfg.gridDim = edge ? k.grid_out : k.grid;
  cfg.blockDim = edge ? k.block_out : k.block;
  cfg.dynamicSmemBytes = static_cast<size_t>(k.smem);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const void* f = flags == kFxOut && k.func_last ? k.func_last : (edge ? k.func_out : k.func);
  return cudaLaunchKernelExC(&cfg, f, const_cast<void**>(args));
}

jacc_status check_buffers(const Kernel& k, const void* a, const void* b) {
  if (!a || !b) return fail(JACC_ERR_INVALID_ARG, "NULL field pointer");
  if ((reinterpret_cast<uintptr_t>(a) % 16) || (reinterpret_cast<uintptr_t>(b) % 16))
    return fail(JACC_ERR_INVALID_ARG, "field pointers must be 16-byte aligned");
  const uintptr_t bytes = static_cast<uintptr_t>(k.desc.nx * k.desc.ny * k.desc.nz) * k.elem;
  const uintptr_t pa = reinterpret_cast<uintptr_t>(a), pb = reinterpret_cast<uintptr_t>(b);
  if (pa < pb + bytes && pb < pa + bytes) return fail(JACC_ERR_INVALID_ARG, "input and output fields overlap");
  return ok();
}

}  // namespace jacc

// Enqueue one sweep with its pre-pass (fixed point) and residual zeroing.
static jacc_status enqueue_one(const Kernel& k, const void* u, void* v, double* resid, u64* scratch, cudaStream_t s) {
  const u64* mw = nullptr;
  if (k.params.fpath != JACC_FP_NONE && k.desc.dtype == 64) {
    jacc_status st = cuda_check(launch_maxabs(static_cast<const double*>(u), k.desc.nx * k.desc.ny * k.desc.nz,
                                              scratch, s),
                                "max-abs pre-pass");
    if (st) return st;
    mw = scratch;
  }
  if (resid) {
    jacc_status st = cuda_check(cudaMemsetAsync(resid, 0, sizeof(double), s), "cudaMemsetAsync(resid)");
    if (st) return st;
  }
  return cuda_check(launch_sweep_kernel(k, u, v, resid, mw, kFxIn | kFxOut, s), "stencil launch");
}

extern "C" jacc_status jacc_launch(jacc_kernel h, const void* u_in, void* u_out, double* resid_dev, uintptr_t stream) {
  if (!h) return fail(JACC_ERR_INVALID_ARG, "NULL handle");
  const Kernel& k = *reinterpret_cast<Kernel*>(h);
  if (k.desc.stencil == 19) return fail(JACC_ERR_INVALID_ARG, "19-point stencil: use jacc_sweep_coeffs");
  jacc_status st = check_buffers(k, u_in, u_out);
  if (st) return st;
  return enqueue_one(k, u_in, u_out, resid_dev, k.scratch, reinterpret_cast<cudaStream_t>(stream));
}

// The full sweep sequence on stream s.  A temporally blocked kernel performs
// tblock sweeps per launch; only every tblock-th sweep is materialised and the
// residual slots of the others are set to NaN.
static jacc_status enqueue_sweeps(const Kernel& k, void* u0, void* u1, int32_t n, double* resid, u64* scratch,
                                  cudaStream_t s) {
  const u64* mw = nullptr;
  if (k.params.fpath != JACC_FP_NONE && k.desc.dtype == 64) {
    jacc_status st = cuda_check(
        launch_maxabs(static_cast<const double*>(u0), k.desc.nx * k.desc.ny * k.desc.nz, scratch, s), "max-abs pre-pass");
    if (st) return st;
    mw = scratch;
  }
  const int T = k.tblock > 1 ? k.tblock : 1;
  if (resid) {
    jacc_status st = cuda_check(cudaMemsetAsync(resid, 0, sizeof(double) * static_cast<size_t>(n), s), "memset resid");
    if (!st && T > 1) st = cuda_check(launch_fill_skipped(resid, n, T, s), "resid NaN fill");
    if (st) return st;
  }
  const int32_t launches = n / T;
  // A large FP64 fixed-point field is converted in place first, so that its
  // first sweep runs the intermediate kernel: the converting kernel holds
  // fewer CTAs per SM and converts each staged value where it is used (512^3:
  // 1.11 ms against 0.34 + 0.17 ms for the conversion).  u0 is overwritten by
  // the second sweep anyway, and the values are those the first sweep would
  // convert on load, so results do not change.  Small fields keep one launch.
  const int64_t npts = k.desc.nx * k.desc.ny * k.desc.nz;
  const bool pre = mw && launches >= 2 && npts >= (int64_t(1) << 22);
  if (pre) {
    jacc_status st = cuda_check(launch_to_fixed(static_cast<double*>(u0), npts, mw, s), "fixed-point conversion");
    if (st) return st;
  }
  for (int32_t i = 0; i < launches; ++i) {
    const void* src = (i % 2 == 0) ? u0 : u1;
    void* dst = (i % 2 == 0) ? u1 : u0;
    const int fl = (i == 0 && !pre ? kFxIn : 0) | (i == launches - 1 ? kFxOut : 0);
    double* r = resid ? resid + static_cast<int64_t>(i) * T + (T - 1) : nullptr;
    jacc_status st = cuda_check(launch_sweep_kernel(k, src, dst, r, mw, fl, s), "stencil launch");
    if (st) return st;
  }
  return ok();
}

extern "C" jacc_status jacc_sweep(jacc_kernel h, void* u0, void* u1, int32_t nsweeps, double* resid_dev, uint32_t flags,
                                  uintptr_t stream, int32_t* final_buf) {
  if (!h) return fail(JACC_ERR_INVALID_ARG, "NULL handle");
  if (nsweeps < 1) return fail(JACC_ERR_INVALID_ARG, "nsweeps must be >= 1");
  if (flags & ~JACC_SWEEP_GRAPH) return fail(JACC_ERR_INVALID_ARG, "unknown sweep flags");
  Kernel& k = *reinterpret_cast<Kernel*>(h);
  if (k.desc.stencil == 19) return fail(JACC_ERR_INVALID_ARG, "19-point stencil: use jacc_sweep_coeffs");
  jacc_status st = check_buffers(k, u0, u1);
  if (st) return st;
  if (k.tblock > 1 && nsweeps % k.tblock)
    return fail(JACC_ERR_INVALID_ARG, "nsweeps must be a multiple of the temporal-blocking depth");
  if (k.desc.stencil == 27 && k.params.fpath != JACC_FP_NONE) {
    // the fixed-point scale is taken once from u0; values may grow by W per sweep
    const double W = k.desc.coeffs[0] + 6 * k.desc.coeffs[1] + 12 * k.desc.coeffs[2] + 8 * k.desc.coeffs[3];
    if (std::pow(W, static_cast<double>(nsweeps)) > 4.0)
      return fail(JACC_ERR_UNSUPPORTED, "weight sum too far above 1 for this many fixed-point sweeps");
  }
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (final_buf) *final_buf = (nsweeps / (k.tblock > 1 ? k.tblock : 1)) % 2;
  if (k.cluster_nc > 0) {  // the whole sequence in one cluster launch (it writes every residual slot)
    JClusterArgs a = {};
    a.u = static_cast<const double*>(u0);
    a.res = static_cast<double*>((nsweeps & 1) ? u1 : u0);
    a.oth = static_cast<double*>((nsweeps & 1) ? u0 : u1);
    a.resid = resid_dev;
    a.nx = k.desc.nx;
    a.ny = k.desc.ny;
    a.nsweeps = nsweeps;
    a.native = k.params.fpath == JACC_FP_NONE ? 1 : 0;
    st = cuda_check(launch_jacobi_cluster(a, k.cluster_nc, s), "cluster sweep launch");
    if (st) return st;
    if (final_buf) *final_buf = (nsweeps & 1) ? 1 : 0;
    return ok();
  }
  if (!(flags & JACC_SWEEP_GRAPH)) return enqueue_sweeps(k, u0, u1, nsweeps, resid_dev, k.scratch, s);

  std::lock_guard<std::mutex> lock(global_mutex());
  const GraphKey gk{u0, u1, nsweeps, resid_dev};
  auto it = k.graphs.find(gk);
  if (it == k.graphs.end()) {
    SweepGraph g;
    if (k.params.fpath != JACC_FP_NONE && k.desc.dtype == 64) {
      st = cuda_check(cudaMalloc(reinterpret_cast<void**>(&g.scratch), 256), "cudaMalloc(graph scratch)");
      if (st) return st;
    }
    cudaStream_t cap = nullptr;
    st = cuda_check(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking), "cudaStreamCreate");
    if (!st) st = cuda_check(cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal), "cudaStreamBeginCapture");
    if (!st) {
      jacc_status est = enqueue_sweeps(k, u0, u1, nsweeps, resid_dev, g.scratch, cap);
      cudaGraph_t graph = nullptr;
      cudaError_t ce = cudaStreamEndCapture(cap, &graph);
      if (est) st = est;
      else st = cuda_check(ce, "cudaStreamEndCapture");
      g.graph = graph;
      if (!st) st = cuda_check(cudaGraphInstantiate(&g.exec, g.graph, 0), "cudaGraphInstantiate");
    }
    if (cap) cudaStreamDestroy(cap);
    if (st) {
      if (g.exec) cudaGraphExecDestroy(g.exec);
      if (g.graph) cudaGraphDestroy(g.graph);
      if (g.scratch) cudaFree(g.scratch);
      return st;
    }
    it = k.graphs.emplace(gk, g).first;
  }
  return cuda_check(cudaGraphLaunch(it->second.exec, s), "cudaGraphLaunch");
}
