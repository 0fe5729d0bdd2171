// jacc_params.h - the kernel parameter block, shared by the host runtime, the
// precompiled kernels and the NVRTC-compiled variants.
#pragma once

typedef unsigned long long u64;
typedef long long i64;
typedef unsigned int u32;

// Fixed-point path selector (JParams::fpath).
#define JACC_FP_NONE 0   // native arithmetic only
#define JACC_FP_SMALL 1  // 7pt, r = fb 2^-k with k <= 5: the FP64 output in 64 bits
#define JACC_FP_WIDE 2   // 7pt / 27pt: exact 128-bit products
#define JACC_FP_JACOBI 3 // 5pt: v 2^(F+2) = S
#define JACC_FP_W32 4    // 27pt: every factor below 2^31 and K in [1, 31]: 32-bit factors

// Kernel families: a table tile's kernel, and those of the library's choice.
#define JACC_FAM_TABLE 0
#define JACC_FAM_STRIP 1   // 5-point: strips of 30 lanes' columns
#define JACC_FAM_RING 2    // 3D: planes staged by asynchronous copies
#define JACC_FAM_DIRECT 3  // 7-point: no staging (32 x 8 threads)
#define JACC_FAM_BULK 4    // 3D, 16-byte columns: planes staged by bulk copies
#define JACC_FAM_NATIVE 5  // FP64 arithmetic throughout (JACC_FP_NONE): a tile's rows or planes in registers

// The 7-point table tiles that stage nothing, and the planes per thread of the
// kernel that does not.
#define JACC_DIRECT_TILE(bx, by, vec) ((bx) == 32 && (by) == 8 && (vec) == 1)
#define JACC_DIRECT_PLANES 2

// Points up to which a folded 5-point kernel marches strips whatever its tile.
#define JACC_SMALL_GRID (1 << 17)
// Points above which an FP64 one has six rows in flight.
#define JACC_LARGE_GRID (1 << 23)

// Rows per thread of the kernels that stage planes by asynchronous copies
// (bx x by threads, one column each): 4, or 2 where 4 would not leave room
// for the stages.
#define JACC_RING_ROWS(bx, by) ((bx) * (by) > 256 ? 2 : 4)

struct JParams {
  i64 nx, ny, nz;
  double c0, c1, c2, c3;   // coefficients for the native path: 7pt r; 27pt w0, wf, we, wc
  u64 fm;                  // 7pt: r 2^62
  i64 fb;                  // JACC_FP_SMALL: r = fb 2^-fk
  i64 fw0, fw1, fw2, fw3;  // JACC_FP_WIDE factors (7pt: fw0 = odd mantissa of r)
  int fk;                  // extra fraction bits of the fixed-point result
  int fpath;               // JACC_FP_*
  // Bounded waits of the bulk-copy staged kernels: each wait on an mbarrier
  // gives up after timeout_ns, writes JACC_DEV_TIMEOUT to *status (device,
  // nullable) and the CTA returns.  stall_plane >= 0 is a test hook: CTA
  // (0,0,0) never requests that staged plane, so its waits run out.
  int* status;
  i64 timeout_ns;
  int stall_plane;
  int zc;  // planes per CTA (3D) or rows per warp (2D)
  // Sweeps until a tolerance: a 5- or 7-point kernel that finds *stop set
  // (device, nullable) returns at once.
  const int* stop;
  // The twelve coefficient fields of the variable-coefficient 19-point
  // stencil (a0 a1 a2 a3 b0 b1 b2 c0 c1 c2 wrk1 bnd; FP32, device), set per
  // call; unused by the other stencils.
  const float* cf[12];
};

#define JACC_DEV_TIMEOUT (-6)  // the value of JACC_ERR_TIMEOUT
