// inst.cu - precompiled (generic) kernel instantiations.  Compiled once per
// (stencil, dtype) with -DJACC_INST_STENCIL={5,7,27} -DJACC_INST_DTYPE={32,64};
// each object exports a table of the 24 tiles' kernels and a table of the
// library's own kernels.
#include "jacc_device.cuh"
#include "tiles.h"

#if JACC_INST_DTYPE == 64
typedef double JT;
#define JVEC 2
#define JEDGE true
#else
typedef float JT;
#define JVEC 4
#define JEDGE false
#endif

#if JACC_INST_STENCIL == 5
#define JKERNP(BX, BY, V, FAM, O, ...) (const void*)jacc_k_jacobi2d<JT, BX, BY, V, FAM, O, __VA_ARGS__>
#elif JACC_INST_STENCIL == 7
#define JKERNP(BX, BY, V, FAM, O, ...) (const void*)jacc_k_heat3d<JT, BX, BY, V, FAM, O, __VA_ARGS__>
#else
#define JKERNP(BX, BY, V, FAM, O, ...) (const void*)jacc_k_box27<JT, BX, BY, V, FAM, O, __VA_ARGS__>
#endif
#define JKERN(BX, BY, V, FAM, O) JKERNP(BX, BY, V, FAM, O, JParams)
// the tile's march length, where it is a constant
#define JTABP(BX, BY, V, ZC) TableP<JACC_INST_STENCIL, JT, BX, BY, V, ZC>::type

#define JCAT3(a, b, c) a##b##_##c
#define JCAT4(a, b, c, d) a##b##_##c##d
#define JTABNAME(s, d) JCAT3(jacc_tab_, s, d)
#define JTABOUT(s, d) JCAT4(jacc_tab_, s, d, _out)
#define JTABLIB(s, d) JCAT4(jacc_tab_, s, d, _lib)
#define JENTRY(id, BX, BY, VEC, ZC) \
  JKERNP(BX, BY, ((VEC) ? JVEC : 1), JACC_FAM_TABLE, false, JTABP(BX, BY, ((VEC) ? JVEC : 1), ZC)),
#if JACC_INST_STENCIL == 5 || JACC_INST_DTYPE == 32
#define JENTRY_OUT(id, BX, BY, VEC, ZC) \
  JKERNP(BX, BY, ((VEC) ? JVEC : 1), JACC_FAM_TABLE, JEDGE, JTABP(BX, BY, ((VEC) ? JVEC : 1), ZC)),
#else  // rings, whose planes per CTA the library may choose
#define JENTRY_OUT(id, BX, BY, VEC, ZC) JKERN(BX, BY, ((VEC) ? JVEC : 1), JACC_FAM_TABLE, true),
#endif

// Table 1: the intermediate sweeps of a fixed-point sequence (and every FP32
// or native sweep).  Table 2 ("_out"): the first and last sweeps of a
// fixed-point sequence and single launches, which convert FP64 on load and/or
// store; identical to table 1 for FP32.
extern "C" const void* const JTABNAME(JACC_INST_STENCIL, JACC_INST_DTYPE)[JACC_NTILES] = {JACC_TILE_LIST(JENTRY)};
extern "C" const void* const JTABOUT(JACC_INST_STENCIL, JACC_INST_DTYPE)[JACC_NTILES] = {JACC_TILE_LIST(JENTRY_OUT)};

#if JACC_INST_DTYPE == 64
// The tiles' kernels in native FP64 arithmetic.
#define JENTRY_NATIVE(id, BX, BY, VEC, ZC)                        \
  JKERNP(BX, BY, ((VEC) ? JVEC : 1), JACC_FAM_NATIVE, false, \
         TableP<JACC_INST_STENCIL, JT, BX, BY, ((VEC) ? JVEC : 1), ZC, true>::type),
#define JTABNATIVE(s) JCAT3(jacc_tab_, s, 64_native)
extern "C" const void* const JTABNATIVE(JACC_INST_STENCIL)[JACC_NTILES] = {JACC_TILE_LIST(JENTRY_NATIVE)};
#endif

// The library's own kernels, [family][16-byte columns]; the last row holds the
// strip march of the converting sweeps (5-point FP64) and the ring of the
// table's scalar 32 x 8 tiles (7-point).
#define JPAIR(BX, BY, FAM, O) {JKERN(BX, BY, 1, FAM, O), JKERN(BX, BY, JVEC, FAM, O)}
#define JNONE {nullptr, nullptr}
extern "C" const void* const JTABLIB(JACC_INST_STENCIL, JACC_INST_DTYPE)[6][2] = {
    JNONE,
#if JACC_INST_STENCIL == 5
    JPAIR(32, 4, JACC_FAM_STRIP, false), JNONE, JNONE, JNONE, JPAIR(32, 4, JACC_FAM_STRIP, JEDGE),
#elif JACC_INST_STENCIL == 7
    JNONE, JPAIR(32, 4, JACC_FAM_RING, false), JPAIR(32, 8, JACC_FAM_DIRECT, false),
    {nullptr, JKERN(32, 4, JVEC, JACC_FAM_BULK, false)}, {JKERN(32, 8, 1, JACC_FAM_RING, false), nullptr},
#else
    JNONE, JPAIR(32, 4, JACC_FAM_RING, false), JNONE, JNONE, JNONE,
#endif
};

#if JACC_INST_STENCIL == 27 && JACC_INST_DTYPE == 64
// The same for weights with 32-bit fixed-point factors (JACC_FP_W32).
#define JW32(BX, BY, V, FAM) (const void*)jacc_k_box27<JT, BX, BY, V, FAM, false, JParamsW32>
#define JENTRY_W32(id, BX, BY, VEC, ZC) JW32(BX, BY, ((VEC) ? JVEC : 1), JACC_FAM_TABLE),
extern "C" const void* const jacc_tab_27_64_w32[JACC_NTILES] = {JACC_TILE_LIST(JENTRY_W32)};
extern "C" const void* const jacc_tab_27_64_lib_w32[6][2] = {
    JNONE, JNONE, {JW32(32, 4, 1, JACC_FAM_RING), JW32(32, 4, 2, JACC_FAM_RING)}, JNONE, JNONE, JNONE};
#endif
