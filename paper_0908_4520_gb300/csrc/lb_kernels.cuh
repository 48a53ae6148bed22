// Fused collide-stream kernels for sm_103a (templates; instantiated per
// velocity set in k_<set>.cu).
//
// One launch advances every cell by one time level of Eq. 2order:
//   pull-stream   f~_a(x) = S_a[f*_a](x)        exact shift by e_a (on-lattice) or
//                                               tensor-product Lax-Wendroff (off-lattice;
//                                               second-order upwind as an option)
//   moments       rho, rho u, 2 rho T (Sec. 2.2, D = 2)
//   equilibrium   f^eq_a = w_a rho sum_{kx+ky<=N} c_kx(u_x) c_ky(u_y) He_kx He_ky / (kx! ky!)
//                 (Sec. 2.1: the Hermite coefficients of the Maxwellian factorise per
//                 axis, c_k(u, T) = E[He_k(X)], X ~ Normal(u, T), from the recurrence
//                 c_{k+1} = u c_k + k (T - 1) c_{k-1})
//   relax         f*_a = f~_a + omega (f^eq_a - f~_a), omega = dt / (tau + dt/2)
//                 (dt / tau for the first-order scheme of Eq. slb)
//   store         f*_a (the next launch streams it)
//   diagnostics   FP64 grid sums of the observables of f~ (mass, momentum, the
//                 sin/cos Fourier amplitudes of u_y and sigma_xy, H norm)
// The stored variable is the deviation d = f - w rho0 (16-bit: d / (w S)), so
// moments and equilibrium are formed without the O(1) background and keep
// FP32 precision relative to the O(U0) signal.
//
// Work decomposition: a tile is ROWS lattice rows x 32 V columns; warp w of a
// block owns row y0 + w and each lane V consecutive cells, so every
// population-plane access of a warp is one contiguous row segment (coalesced,
// vectorised when V = 2).  The last tile of a row is shifted left to end at
// nx (its overlap with the previous tile is recomputed but neither stored nor
// counted), so every warp of a row wider than a tile is full.  The grid is
// persistent (a multiple of the SM count) and walks tiles row-major (the
// TMA-staged kernel: column-major in bands of tile rows for the exact-shift
// sets), so the halo rows a tile re-reads were fetched moments earlier by its
// neighbours and sit in L2.  Populations carry a rim of periodic images (ghost columns and
// rows), rewritten by every store, so no read ever wraps.
//
// Three step kernels share the collision code and give bitwise-identical results:
//  * lb_tma_step_kernel (the hot path): one producer warp streams, per group of
//    velocities, the tile's source box (with its halo) from HBM into a ring of
//    shared-memory stages with cp.async.bulk.tensor, completion tracked by
//    mbarriers; the consumer warps read their row from shared memory, so the
//    next tile's loads overlap this tile's collision.  Every wait is bounded:
//    on expiry the kernel flags LB_ERR_TIMEOUT in the status word and returns.
//  * lb_fused_kernel: plain coalesced loads from global memory (moments read-back,
//    the first level, FP64 storage and grids too small for the TMA tiles).
//  * lb_split_kernel: FP64 Lax-Wendroff steps of grids that leave FP64 units idle, a lane
//    for every x node of a cell.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "lb_device.h"

namespace lbk {

// ---------------------------------------------------------------- storage I/O
template <class S>
struct Is16 : std::false_type {};
template <>
struct Is16<__nv_bfloat16> : std::true_type {};
template <>
struct Is16<__half> : std::true_type {};

template <class S, class R>
__device__ __forceinline__ void st1(S* p, R v, R scinv) {
    if constexpr (std::is_same<S, __nv_bfloat16>::value) {
        *p = __float2bfloat16_rn(v * scinv);
    } else if constexpr (std::is_same<S, __half>::value) {
        *p = __float2half_rn(v * scinv);
    } else {
        (void)scinv;
        *p = v;
    }
}

template <class S, class R>
__device__ __forceinline__ R load_scale(const Tab<R>& t, int a) {
    if constexpr (Is16<S>::value) return t.sc[a];
    (void)t;
    (void)a;
    return R(1);
}

template <class S, class R>
__device__ __forceinline__ R store_scale(const Tab<R>& t, int a) {
    if constexpr (Is16<S>::value) return t.scinv[a];
    (void)t;
    (void)a;
    return R(1);
}

// ---------------------------------------------------------------- population elements
// Lax-Wendroff sets with 32- and 16-bit storage keep two velocities (a, a + 1), a even, side by side:
// plane a / 2 holds pairs, 8 or 4 bytes a cell.  The kernels collide such pairs as one packed value
// (collide_cell_pairs), so a pair is one load, one 16-bit conversion pair and one store, and a tile
// row of a TMA box has half the alignment padding.  The exact-shift sets (a shift of its own for
// every velocity) and FP64 keep one velocity a plane.
// (32 levels, one velocity a plane / pairs: D2Q36-GH FP32 4096^2 28.06 / 27.36 ms, D2Q64-GH FP32 2048^2
// 15.8 / 13.4, FP16 16.2 / 15.4; D2Q16-GH FP32 2502 x 1251, 64 levels 6.31 / 5.60.)
template <class S>
struct PairOf {
    using E = S;
};
template <>
struct PairOf<float> {
    using E = float2;
};
template <>
struct PairOf<__half> {
    using E = uint32_t;
};
template <>
struct PairOf<__nv_bfloat16> {
    using E = uint32_t;
};
template <class VS, class S>
struct Layout {
    static constexpr bool PAIRED = !VS::kOnLattice && VS::kProductWeights && VS::NA % 2 == 0 && sizeof(S) <= 4;
    static constexpr int VW = PAIRED ? 2 : 1;               // velocities of an element
    static constexpr int PLANES = VS::Q / VW;
    static constexpr int EB = VW * (int)sizeof(S);          // bytes of an element
    using E = typename std::conditional<PAIRED, typename PairOf<S>::E, S>::type;
};
// Scalar view of the populations: value of velocity a at element offset `off` of its plane is
// base[pop_index(a, plane, off)], neighbours in x lie VW apart.
template <class VS, class S>
__device__ __forceinline__ long long pop_index(int a, long long plane, long long off) {
    constexpr int VW = Layout<VS, S>::VW;
    return VW * ((a / VW) * plane + off) + a % VW;
}

// ---------------------------------------------------------------- stochastic rounding
// 16-bit stores of the step kernels round stochastically (unbiased: the stored
// value equals the FP32 value in expectation), so per-step changes smaller than
// half a 16-bit ulp are not rounded away (the decay would stagnate).  The random
// bits come from a counter-based generator: MurmurHash3's 32-bit finalizer of
// (cell, level) seeds one 32-bit linear congruential stream per cell (multiplier
// 1664525, increment 1013904223), advanced once per velocity; its high bits are
// the rounding bits.  The result does not depend on the launch geometry.
__device__ __forceinline__ uint32_t fmix32(uint32_t h) {
    h ^= h >> 16;
    h *= 0x85ebca6bu;
    h ^= h >> 13;
    h *= 0xc2b2ae35u;
    h ^= h >> 16;
    return h;
}
__device__ __forceinline__ uint32_t sr_next(uint32_t x) { return x * 1664525u + 1013904223u; }
__device__ __forceinline__ uint32_t sr_seed(long long level, long long cell) {
    return fmix32((uint32_t)cell ^ fmix32((uint32_t)level * 0x9e3779b9u + 0x7f4a7c15u));
}
// random bits below the 16-bit mantissa of an FP32 value: 13 for FP16, 16 for BF16
template <class S>
__device__ __forceinline__ uint32_t sr_bits(uint32_t r) {
    return std::is_same<S, __half>::value ? (r >> 19) : (r >> 16);
}

// Two scaled values (already multiplied by the storage scale) rounded stochastically
// into one 16-bit pair word, the first in the low half (one conversion instruction).
template <class S>
__device__ __forceinline__ uint32_t to_storage16x2(float h0, float h1, uint32_t r0, uint32_t r1) {
    const float a = __uint_as_float(__float_as_uint(h0) + sr_bits<S>(r0));
    const float b = __uint_as_float(__float_as_uint(h1) + sr_bits<S>(r1));
    uint32_t d;
    if constexpr (std::is_same<S, __half>::value) {
        asm("cvt.rz.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    } else {
        asm("cvt.rz.bf16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(b), "f"(a));
    }
    return d;
}

// compile-time loop: f(integral_constant<int, a>) for a in [A_, Q)
template <int A_, int Q, class F>
__device__ __forceinline__ void static_for(F&& f) {
    if constexpr (A_ < Q) {
        f(std::integral_constant<int, A_>{});
        static_for<A_ + 1, Q>(f);
    }
}

// ------------------------------------------------------------ packed lanes
// Two cells of a thread travel as one packed pair (f2) through the paired FP32
// instructions of sm_100-class GPUs (add/sub/mul/fma .f32x2).  Each half of a
// pair rounds exactly as the scalar instruction would, so a pair gives the
// results of two scalar evaluations bit for bit.
struct __align__(8) f2 {
    float x, y;
};

__device__ __forceinline__ unsigned long long f2_bits(f2 a) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a.x), "f"(a.y));
    return r;
}
__device__ __forceinline__ f2 f2_from(unsigned long long r) {
    f2 a;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a.x), "=f"(a.y) : "l"(r));
    return a;
}
__device__ __forceinline__ f2 vfma(f2 a, f2 b, f2 c) {
    unsigned long long d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)), "l"(f2_bits(c)));
    return f2_from(d);
}
__device__ __forceinline__ f2 vadd(f2 a, f2 b) {
    unsigned long long d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_from(d);
}
__device__ __forceinline__ f2 vsub(f2 a, f2 b) {
    unsigned long long d;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_from(d);
}
__device__ __forceinline__ f2 vmul(f2 a, f2 b) {
    unsigned long long d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(f2_bits(a)), "l"(f2_bits(b)));
    return f2_from(d);
}
__device__ __forceinline__ f2 vrcp(f2 a) { return f2{1.0f / a.x, 1.0f / a.y}; }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vrcp(float a) { return 1.0f / a; }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double vsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double vmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double vrcp(double a) { return 1.0 / a; }

template <class T>
struct LaneScalar {
    using type = T;
};
template <>
struct LaneScalar<f2> {
    using type = float;
};

template <class T>
__device__ __forceinline__ T vsplat(typename LaneScalar<T>::type c) {
    if constexpr (std::is_same<T, f2>::value) {
        return f2{c, c};
    } else {
        return c;
    }
}

// lane K of a packed value, and packing of V lane values
template <int K>
__device__ __forceinline__ float lane_get(const f2& v) {
    if constexpr (K == 0) {
        return v.x;
    } else {
        return v.y;
    }
}
template <int K>
__device__ __forceinline__ float lane_get(const float& v) {
    return v;
}
template <int K>
__device__ __forceinline__ double lane_get(const double& v) {
    return v;
}
template <class T, class R>
__device__ __forceinline__ T pack_lanes(R v0, R v1) {
    if constexpr (std::is_same<T, f2>::value) {
        return f2{v0, v1};
    } else {
        (void)v1;
        return v0;
    }
}

template <class R, int V>
struct Pack {
    using T = R;
};
template <>
struct Pack<float, 2> {
    using T = f2;
};

// Loads of the populations, from global or shared memory.  None takes the read-only path: a step launch
// may have started, and its caches filled, before the launch that writes them has ended (see
// await_previous_step).
// The cells of a lane: one value, or an aligned pair.
template <class T, class R>
__device__ __forceinline__ T ld_cells(const R* p) {
    if constexpr (std::is_same<T, f2>::value) {
        const float2 t = *reinterpret_cast<const float2*>(p);
        return f2{t.x, t.y};
    } else {
        return *p;
    }
}
// A pair of velocities of one cell, unscaled.
template <class S>
__device__ __forceinline__ f2 unpack_pair(uint32_t u) {
    float2 t;
    if constexpr (std::is_same<S, __half>::value) {
        t = __half22float2(*reinterpret_cast<const __half2*>(&u));
    } else {
        t = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u));
    }
    return f2{t.x, t.y};
}
template <class S>
__device__ __forceinline__ f2 ld_pair(const typename PairOf<S>::E* p) {
    if constexpr (std::is_same<S, float>::value) {
        const float2 t = *p;
        return f2{t.x, t.y};
    } else {
        return unpack_pair<S>(*p);
    }
}
// The stored pair (16-bit: stochastically rounded with the random bits of r0, r1).
template <class S>
__device__ __forceinline__ typename PairOf<S>::E to_storage_pair(f2 v, f2 si, uint32_t r0, uint32_t r1) {
    if constexpr (std::is_same<S, float>::value) {
        return make_float2(v.x, v.y);
    } else {
        const f2 h = vmul(v, si);
        return to_storage16x2<S>(h.x, h.y, r0, r1);
    }
}

// ------------------------------------------------------------ configuration
// Launch shapes, from sweeps at 4096^2 (FP32, N = 3) and 2048^2 (D2Q64, N = 4):
//  * Lax-Wendroff (Gauss-Hermite product) sets: one cell per lane and many warps
//    (19 consumer rows, or 15 and 11 for q = 64), stages of 6 velocities to a whole tile;
//  * exact-shift sets: two cells per lane (packed f32x2), 11 consumer rows (13 for
//    q <= 25), 18 velocities per stage.
// The plain-load kernel takes the same cells per lane as the TMA-staged one, so the
// two give the same bits.  Each value is overridable at build time (0 = the choice above).
#ifndef LB_CFG_V
#define LB_CFG_V 0
#endif
#ifndef LB_TMA_V
#define LB_TMA_V 0
#endif
#ifndef LB_CFG_ROWS
#define LB_CFG_ROWS 8
#endif
#ifndef LB_CFG_MINB
#define LB_CFG_MINB 0
#endif
#ifndef LB_TMA_ROWS
#define LB_TMA_ROWS 0
#endif
#ifndef LB_TMA_K
#define LB_TMA_K 0
#endif
#ifndef LB_TMA_EVICT_LAST
#define LB_TMA_EVICT_LAST 1  // TMA loads keep their lines in L2 for the neighbouring tiles (-3 % DRAM reads)
#endif
#ifndef LB_TMA_NS_TILES
#define LB_TMA_NS_TILES 0  // ring depth cap, in tiles of stages (0: see TmaCfg)
#endif
#ifndef LB_TMA_SMEM
#define LB_TMA_SMEM (200 * 1024)
#endif
#ifndef LB_TMA_MINB
#define LB_TMA_MINB 1
#endif
#ifndef LB_TMA_BAND
// TMA kernel tile order: -1 per set, 0 row-major, B > 0 column-major in bands of B tile rows: bands for
// the exact-shift sets, whose boxes are displaced by up to max|e| rows (row-major order cost D2Q37 a third
// of its rate at 4096^2), row-major for Lax-Wendroff (bands cost up to half)
#define LB_TMA_BAND -1
#endif
#ifndef LB_TMA_BAND_SHIFT
// band height of the exact-shift sets under LB_TMA_BAND = -1 (D2Q37 FP32 at 4096^2 and 2048^2, GLUPS:
// bands of 2 / 3 / 4 / 6 / 8 tile rows 19.63 / 19.65 / 19.40 / 18.91 / 18.44 and 19.63 / 19.77 /
// 19.43 / 19.58 / 19.36)
#define LB_TMA_BAND_SHIFT 3
#endif
#ifndef LB_TMA_WIDE_WARPS
#define LB_TMA_WIDE_WARPS 0  // consumer warps of the store-staged kernel (two per tile row); 0: 18, q = 64: 14
#endif
#ifndef LB_TMA_WIDE_SMEM
// ring + output slots of the store-staged kernel, bytes; 0: FP32 224 KB (D2Q36-GH at 4096^2, 192 / 224 KB
// and 12 velocities a stage: 788 / 751 us a level), 16-bit 192 KB (D2Q64-GH at 2048^2 525 / 563)
#define LB_TMA_WIDE_SMEM 0
#endif
#ifndef LB_DIAG_PREFETCH
// load sin/cos of the diagnostics before the collision: -1 per set and kernel, 0 never, 1 always.  Taken
// for D2Q16-GH (35.7 -> 38.5 GLUPS at 4096^2 when the stores were of single velocities) and the
// store-staged kernel (17.4 -> 17.9); D2Q37 and D2Q64-GH lost 1 to 2 % by it
#define LB_DIAG_PREFETCH -1
#endif

// cells per lane along x (FP64 storage: always 1)
template <class VS, class S, int OVERRIDE>
constexpr int cells_per_lane() {
    return sizeof(S) == 8 || Layout<VS, S>::PAIRED ? 1 : (OVERRIDE > 0 ? OVERRIDE : 2);
}

template <class VS, class S>
struct Cfg {
    static constexpr int V = cells_per_lane<VS, S, (LB_CFG_V > 0 ? LB_CFG_V : LB_TMA_V)>();
    // Lax-Wendroff, one cell per lane, FP32 arithmetic: the warp's edge lanes are halo lanes, as in
    // the TMA-staged kernel: three loads a velocity instead of six (256^2 D2Q36-GH FP32, 400 levels:
    // 9.79 -> 6.21 ms)
    static constexpr bool HALO = !VS::kOnLattice && V == 1 && Layout<VS, S>::PAIRED;
    static constexpr int TW = HALO ? 30 : 32 * V;  // cells of a warp (upwind streaming: 32 V)
    static constexpr int ROWS = LB_CFG_ROWS;
    static constexpr int THREADS = 32 * ROWS;
    // one cell per lane needs under 128 registers: two blocks (16 warps) per SM
    static constexpr int MINB = LB_CFG_MINB > 0 ? LB_CFG_MINB : (V == 1 && sizeof(S) != 8 ? 2 : 1);
};

// UPW: second-order upwind streaming of a Lax-Wendroff set (one cell per lane): lanes
// 0, 1 and 30, 31 compute the y pass of the two columns on either side of the 28 cells
// that lanes 2..29 own, and the box carries two extra rows above and below.
// WIDE: the store-staged variant of the Lax-Wendroff kernel (one cell per lane, halo lanes): two warps
// share a tile row (FP32: 30 cells each; 16-bit: 28 each, lanes 29 to 31 idle: a warp's row segment is
// whole 16-byte TMA granules), and each consumer warp writes its relaxed populations (16-bit:
// stochastically rounded) into a slot of its own in shared memory and from there to HBM with one TMA
// tensor store (cp.async.bulk.tensor, shared -> global), so no lane issues per-velocity global stores.
// A warp waits only for its own store of the tile before: one store of the whole tile by the producer
// made every warp wait for the slowest one's tile and for that store.  D2Q36-GH FP32 at 4096^2: 820 -> 774 us
// a level, with larger stages 751 (5.89 -> 6.43 TB/s).
template <class VS, class S, bool UPW = false, bool WIDE = false>
struct TmaCfg {
    static constexpr bool LW = !VS::kOnLattice;
    using E = typename Layout<VS, S>::E;
    static constexpr int VW = Layout<VS, S>::VW, EB = Layout<VS, S>::EB;
    static_assert(LW == Layout<VS, S>::PAIRED || sizeof(S) == 8, "32/16-bit Lax-Wendroff sets are paired");
    static constexpr int V = cells_per_lane<VS, S, LB_TMA_V>();
    static_assert(!UPW || (LW && V == 1), "upwind TMA staging: Lax-Wendroff sets, one cell per lane");
    static_assert(!WIDE || (LW && V == 1 && !UPW && sizeof(S) <= 4), "store staging: 32/16-bit Lax-Wendroff sets");
    // consumer warps (+ one producer warp); the register cap follows from the count
    // (exact shift at 4096^2 FP32, 11 / 13 rows, GLUPS: D2Q37 18.3 / 16.8, D2Q25 21.3 / 22.3,
    // D2Q21 25.4 / 27.7, D2Q17 41.6 / 42.1, D2Q16 44.7 / 45.1, D2Q9 68.6 / 72.6)
    static constexpr int CW = WIDE ? (LB_TMA_WIDE_WARPS > 0 ? LB_TMA_WIDE_WARPS : (VS::Q > 40 ? 14 : 18))
                                   : (LB_TMA_ROWS > 0 ? LB_TMA_ROWS
                                      : !LW           ? (VS::Q > 30 ? 11 : 13)
                                      : VS::Q > 40    ? (sizeof(S) == 2 ? 11 : 15)
                                                      : 19);
    static constexpr int WPR = WIDE ? 2 : 1;            // consumer warps per tile row
    static constexpr int ROWS = CW / WPR;               // lattice rows of a tile
    static_assert(CW % WPR == 0, "whole tile rows");
    static constexpr int TW = 32 * V;
    // Edge lanes as halo lanes: 30 cells a row (D2Q64-GH FP32 at 2048^2, us a level: 32 cells and an
    // extra column's reads 405, halo lanes 372; FP16 555 / 469).
    static constexpr bool HALO = LW && V == 1 && !UPW;
    // (No per-tile barrier of the consumer warps, which would keep the ring's stages together: with
    // populations in pairs D2Q36-GH FP32 takes 965 us a level with it and 838 without at 4094 x 4096,
    // upwind at 2048^2 271 and 224.)
    static constexpr int WCELLS = UPW || (WIDE && sizeof(S) == 2) ? 28 : (HALO ? 30 : TW);  // cells a warp produces
    static constexpr int TWO = WPR * WCELLS;            // cells a tile row produces
    static constexpr int GX = UPW ? 2 : 1;              // stencil reach (columns and rows) of the box
    static constexpr int BAND = LB_TMA_BAND >= 0 ? LB_TMA_BAND : (LW ? 0 : LB_TMA_BAND_SHIFT);  // tile order
    static constexpr int AL = 16 / EB;                  // TMA x coordinates are multiples of 16 bytes
    static_assert(!WIDE || WCELLS % AL == 0, "store-staged row segments are whole 16-byte granules");
    static constexpr int BW = WIDE ? TWO + 2 * AL : (LW ? 32 + AL : TW + AL);
    static constexpr int BH = LW ? ROWS + 2 * GX : ROWS;
    static constexpr int BOX = BW * BH;                 // elements of one plane's box
    // stride of the planes' slots in a stage: dense for one 3-D box (Lax-Wendroff),
    // 128-byte aligned for separate boxes (exact shift)
    static constexpr int SLOT = LW ? BOX : ((BOX * EB + 127) / 128 * 128) / EB;
    // Velocities per stage, in us a level: 16-bit sets take a whole tile a stage (D2Q64-GH 2048^2, 15
    // rows: 12 / 16 / 32 / 64 velocities 469 / 445 / 418 / 391, with 11 rows and no spills 382;
    // D2Q36-GH 4096^2 6 / 12 / 18 / 36 889 / 819 / 814 / 811; D2Q16-GH 4096^2 6 / 8 / 16 453 / 432 /
    // 411), FP32 D2Q16-GH 8 (4096^2 and 2502 x 1251, 6 / 8 / 16: 388 / 364 / 361 and 83.7 / 79.2 / 80.0,
    // three tiles of stages), D2Q36-GH 12 (4094 x 4096, 6 / 12 / 18: 838 / 786 / 793), D2Q64-GH 16 (2048^2,
    // 8 / 12 / 16: 391 / 372 / 369), store-staged D2Q36-GH 12, a third of a tile
    // (FP32 4096^2, 4 / 6 / 10 / 12 / 14 / 18: 820 / 774 / 758 / 751 / 784 / 804, 1024^2 6 / 12: 66 / 65; N = 1
    // alone is faster with 6, 738 / 768; FP16 1005 / 947 with 6 / 12), upwind D2Q36-GH 12 (2048^2 6 / 12: 224 /
    // 215, 4096^2 891 / 828).
    static constexpr int K = LB_TMA_K > 0          ? LB_TMA_K
                             : !LW                 ? 18
                             : WIDE || UPW         ? (VS::Q > 16 ? 12 : 6)
                             : sizeof(S) == 2      ? VS::Q
                             : VS::Q > 40          ? 16
                                                   : (VS::Q > 16 ? 12 : 8);
    static_assert(K % VW == 0, "whole elements per stage");
    static constexpr int KE = K / VW;                   // planes per stage
    static constexpr int NG = (VS::Q + K - 1) / K;      // stages per tile
    static constexpr int STAGE_BYTES = (KE * SLOT * EB + 127) / 128 * 128;
    // output slot of a warp of the store-staged kernel: [plane][WCELLS cells]
    static constexpr int OUT_SLOT = (Layout<VS, S>::PLANES * WCELLS * EB + 127) / 128 * 128;
    static constexpr int OUT_BYTES = WIDE ? CW * OUT_SLOT : 0;
    static constexpr int WIDE_SMEM = LB_TMA_WIDE_SMEM > 0 ? LB_TMA_WIDE_SMEM : (sizeof(S) == 4 ? 224 : 192) * 1024;
    static constexpr int NS_FIT = ((WIDE ? WIDE_SMEM - OUT_BYTES : LB_TMA_SMEM) - 512) / STAGE_BYTES;
    static constexpr int NS_TILES = LB_TMA_NS_TILES > 0 ? LB_TMA_NS_TILES
                                    : LW && !WIDE && !UPW && VS::Q == 16 ? (sizeof(S) == 2 ? 4 : 3) : 2;
    static constexpr int NS = NS_FIT < NS_TILES * NG ? NS_FIT : NS_TILES * NG;
    static constexpr int THREADS = 32 * (CW + 1);       // + one producer warp
    // registers a thread may hold: each SM sub-partition's 16384 registers are shared by
    // ceil(warps / 4) warps of the block (255 for 8 warps, 168 for 9..12, 128 for 13..16)
    static constexpr int WARPS_PER_SMSP = (CW + 1 + 3) / 4;
    static constexpr int MAXREG_FIT = 16384 / (32 * WARPS_PER_SMSP) / 8 * 8;
    static constexpr int MAXREG = MAXREG_FIT > 255 ? 255 : MAXREG_FIT;
    // ring, output slots, full/empty barriers of the ring
    static constexpr int SMEM = NS * STAGE_BYTES + OUT_BYTES + 2 * NS * 8 + 128;  // + alignment slack
    static constexpr int BOX_D = LW ? KE : 1;           // planes per TMA box
};

// ------------------------------------------------------------ equilibrium
// Deviation of the truncated Hermite equilibrium from w rho0, for one cell:
// deq_a = w_a (drho + rho * sum'_{kx+ky<=N} c_kx(ux) c_ky(uy) hn[ix][kx] hn[iy][ky]),
// sum' without the (0,0) term (which is rho itself).  The velocities are visited
// grouped by their x axis node, so only one row of x partial sums is live.
// emit(integral_constant<a>, deq_a) is called once per velocity.
template <class VS, int N, class R, class Emit>
__device__ __forceinline__ void equilibrium_dev(const Tab<R>& t, R drho, R rho, R ux, R uy, R th,
                                                Emit&& emit) {
    constexpr int NA = VS::NA;
    R cx[N + 1], cy[N + 1];
    cx[0] = R(1);
    cy[0] = R(1);
    cx[1] = ux;
    cy[1] = uy;
#pragma unroll
    for (int k = 1; k < N; ++k) {
        cx[k + 1] = ux * cx[k] + R(k) * th * cx[k - 1];
        cy[k + 1] = uy * cy[k] + R(k) * th * cy[k - 1];
    }
    R qy[NA][N + 1];
#pragma unroll
    for (int j = 0; j < NA; ++j) {
        qy[j][0] = R(0);
#pragma unroll
        for (int ky = 1; ky <= N; ++ky) qy[j][ky] = cy[ky] * t.hn[j][ky];
    }
    static_for<0, NA>([&](auto ic) {
        constexpr int I = decltype(ic)::value;
        // px[0] excludes kx = 0; px[ky>=1] = sum_{kx <= N-ky} cx[kx] hn[I][kx]
        R px[N + 1];
#pragma unroll
        for (int ky = 0; ky <= N; ++ky) {
            R s = (ky == 0) ? R(0) : R(1);
#pragma unroll
            for (int kx = 1; kx <= N - ky; ++kx) s = fma(cx[kx], t.hn[I][kx], s);
            px[ky] = s;
        }
        static_for<0, VS::Q>([&](auto ac) {
            constexpr int a = decltype(ac)::value;
            if constexpr (VS::ix(a) == I) {
                constexpr int iy = VS::iy(a);
                R s = px[0];
#pragma unroll
                for (int ky = 1; ky <= N; ++ky) s = fma(px[ky], qy[iy][ky], s);
                emit(ac, t.w[a] * fma(rho, s, drho));
            }
        });
    });
}

// ------------------------------------------------------------ tile geometry
struct Lane {
    int x;          // first cell of the lane
    int xl;         // column read for the lane (x, or nx for lanes past the grid)
    bool own;       // x < nx and not a recomputed overlap cell
};

// TMA-staged Lax-Wendroff with one cell per lane: the warp's edge lanes are halo lanes
// (columns x0 - 1 and x0 + 30), whose y-pass only feeds their neighbours' x-pass, so no
// lane reads an extra column; lanes 1..own own cells x0 .. x0 + own - 1.
__device__ __forceinline__ Lane halo_lane_geometry(int lane, int x0, int tile_start, int nx, int own = 30) {
    Lane g;
    g.x = x0 - 1 + lane;
    g.own = lane >= 1 && lane <= own && g.x < nx && g.x >= tile_start;
    g.xl = g.x;
    return g;
}

// The same for second-order upwind: lanes 0, 1 and 30, 31 are halo lanes (columns
// x0 - 2, x0 - 1, x0 + 28, x0 + 29); lanes 2..29 own cells x0 .. x0 + 27.
__device__ __forceinline__ Lane upwind_lane_geometry(int lane, int x0, int tile_start, int nx) {
    Lane g;
    g.x = x0 - 2 + lane;
    g.own = lane >= 2 && lane <= 29 && g.x < nx && g.x >= tile_start;
    g.xl = g.x;
    return g;
}

// Tile (ty, tx) of the TMA kernel's tile index.  Row-major (B = 0), or column-major within
// bands of B tile rows, so that the tiles in flight at one time (consecutive indices) are
// neighbours in x and in y: the exact-shift sets' boxes, displaced by up to max|e| rows
// and columns, then find the rows of the tiles above and beside them in L2.
template <int B>
__device__ __forceinline__ void tma_tile_coords(int tile, int ntiles_x, int ntiles, int& ty, int& tx) {
    if constexpr (B <= 0) {
        ty = tile / ntiles_x;
        tx = tile - ty * ntiles_x;
    } else {
        const int per_band = B * ntiles_x;
        const int band = tile / per_band;
        const int r = tile - band * per_band;
        const int ntiles_y = ntiles / ntiles_x;
        const int rows = min(B, ntiles_y - band * B);
        tx = r / rows;
        ty = band * B + (r - tx * rows);
    }
}

template <int V>
__device__ __forceinline__ Lane lane_geometry(int lane, int x0, int tile_start, int nx) {
    Lane g;
    g.x = x0 + lane * V;
    g.own = g.x < nx && g.x >= tile_start;
    g.xl = g.x < nx ? g.x : nx;  // the first column past the grid is a valid image
    return g;
}

template <class R>
__device__ __forceinline__ R warp_sum(R v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The periodic images of the V cells at (x.., y) inside the ghost rim (not (x, y) itself), one
// after another: img(xi, yi) of each.  A cell near an edge has one to three of them, on a grid
// narrower than the rim more.  The image is the outer loop and the velocities the inner, unrolled
// one, so that all q values leave from registers as independent stores: a copy of the stored
// values, velocity by velocity, was a chain of q dependent memory round trips that every warp of a
// boundary row waited for (us per level before / after: D2Q16-GH FP64 64 x 1 35.7 / 24.9, D2Q36-GH
// FP32 256^2 37.6 / 23.6, 1024^2 127 / 76, 2048^2 282 / 235, D2Q64-GH FP32 2048^2 768 / 492).
template <class R, int V, class F>
__device__ __forceinline__ void for_images(const Args<R>& A, int x, int y, F&& img) {
    int ylo = y;
    while (ylo - A.ny >= -A.gy) ylo -= A.ny;
    int xlo = x;
    while (xlo - A.nx >= -kGhostX) xlo -= A.nx;
    for (int yi = ylo; yi < A.ny + A.gy; yi += A.ny) {
        for (int xi = xlo; xi + V <= A.nx + kGhostX; xi += A.nx) {
            if (xi == x && yi == y) continue;
            img(xi, yi);
        }
    }
}

// Whether the V cells at (x.., y) have an image in the ghost rim.
template <class R, int V>
__device__ __forceinline__ bool has_images(const Args<R>& A, int x, int y) {
    return x < kGhostX || x + V > A.nx - kGhostX || y < A.gy || y >= A.ny - A.gy;
}

// Write velocity a's value at (x, y) and at every periodic image (round to nearest: used for the
// initial state).
template <class VS, class S, class R>
__device__ __forceinline__ void store_cell(const Args<R>& A, S* dst, int a, int x, int y, R v, R si) {
    S sv;
    st1<S, R>(&sv, v, si);
    auto put = [&](int xi, int yi) {
        dst[pop_index<VS, S>(a, A.plane, A.origin + (long long)yi * A.pitch + xi)] = sv;
    };
    put(x, y);
    if (has_images<R, 1>(A, x, y)) for_images<R, 1>(A, x, y, put);
}

// ------------------------------------------------------------ collision (shared)
// Result of colliding one cell (or a packed pair of cells).
template <class T>
struct CellOut {
    T drho, jx, jy;   // deviation moments: rho - rho0, rho u
    T ux, uy, th;     // velocity, T - 1
    T sig;            // sigma_xy = (1 - omega/2) sum xi_x xi_y (f~ - f^eq)   (diag)
    T h;              // sum (f~ - w rho0)^2 / w                               (diag)
};

// The state of a cell from its summed moments (deviations): velocity, temperature and sigma_xy into
// o, and (COLLIDE) the Hermite coefficients of its Maxwellian, c_{k+1} = u c_k + k (T - 1) c_{k-1},
// with the force folded into the y ones.  Returns rho.  Shared by collide_cell and the node-split
// kernel, so that both round the same.
template <int N, class R, class T, bool COLLIDE>
__device__ __forceinline__ T cell_state(R rho0, R sigma_fac, int isothermal, bool forced, T gf, R tau, R hdt, T drho,
                                        T jx, T jy, T en, T pxy, CellOut<T>& o, T (&cx)[N + 1], T (&cy)[N + 1]) {
    const T zero = vsplat<T>(R(0));
    const T rho = vadd(vsplat<T>(rho0), drho);
    const T rg = forced ? vmul(rho, gf) : zero;  // rho g
    if (forced) jy = vfma(vsplat<T>(hdt), rg, jy);
    const T inv = vrcp(rho);
    const T ux = vmul(jx, inv), uy = vmul(jy, inv);
    const T u2 = vfma(ux, ux, vmul(uy, uy));
    T th = zero;
    if (!isothermal) {
        T e2 = vsub(vsub(en, vadd(drho, drho)), vmul(rho, u2));
        if (forced) e2 = vfma(vmul(vsplat<T>(hdt + hdt), rg), uy, e2);
        th = vmul(vmul(e2, vsplat<T>(R(0.5))), inv);
    }
    o.drho = drho;
    o.jx = jx;
    o.jy = jy;
    o.ux = ux;
    o.uy = uy;
    o.th = th;
    T pneq = pxy;
    if constexpr (N >= 2) {
        pneq = vsub(pxy, vmul(rho, vmul(ux, uy)));
        if (forced) pneq = vfma(vmul(vsplat<T>(hdt), rg), ux, pneq);
    }
    o.sig = vmul(vsplat<T>(sigma_fac), pneq);
    if constexpr (COLLIDE) {
        cx[0] = cy[0] = vsplat<T>(R(1));
        cx[1] = ux;
        cy[1] = uy;
#pragma unroll
        for (int k = 1; k < N; ++k) {
            const T kth = k == 1 ? th : vmul(vsplat<T>(R(k)), th);
            cx[k + 1] = vfma(ux, cx[k], k == 1 ? kth : vmul(kth, cx[k - 1]));
            cy[k + 1] = vfma(uy, cy[k], k == 1 ? kth : vmul(kth, cy[k - 1]));
        }
        if (forced) {
            const T tg = vmul(vsplat<T>(tau), gf);
#pragma unroll
            for (int k = N; k >= 1; --k) cy[k] = vfma(vmul(vsplat<T>(R(k)), tg), cy[k - 1], cy[k]);
        }
    }
    return rho;
}

// The one definition of the per-cell arithmetic; every kernel calls it.  The
// streamed deviations are f(integral_constant<a>) (references, relaxed in place
// when COLLIDE).  T is a scalar or a packed pair of cells.
//  * moments from per-axis-node sums: C[i] = sum_{ix = i} d, Ry[j] = sum_{iy = j} d;
//    rho - rho0 = sum C, rho u_x = sum a_i C[i], rho u_y = sum a_j Ry[j],
//    sum |xi|^2 d = sum a_i^2 (C[i] + Ry[i])  (Sec. 2.2; kinetic T with D = 2)
//  * diagnostics (diag): Pi_xy = sum xi_x xi_y d and H = sum d^2 / w of the
//    streamed state; sigma_xy = (1 - omega/2) (Pi_xy - rho u_x u_y), since the
//    truncated equilibrium carries exactly the xy moment rho u_x u_y of the
//    Maxwellian when the quadrature degree is >= N + 2
//  * equilibrium (Sec. 2.1), per axis: f^eq_a - w rho0 = w_a (drho + rho S'_a),
//    S'_a = sum'_{kx+ky<=N} c_kx(u_x) c_ky(u_y) hn[ix][kx] hn[iy][ky]; for product
//    weights w_a = W_ix W_iy the weights fold into the per-axis factors, so
//    omega (f^eq_a - w_a rho0) = sum_{ky<=N} PX[ix][ky] QY[iy][ky]
//  * relaxation (Eq. 2order): f* = (1 - omega) f~ + omega f^eq, one FMA a velocity
//  * N = 1 (Sec. 3.3, Eq. lbm1): f^eq = w rho (1 + xi.u) has no xy moment, so
//    sigma_xy = (1 - omega/2) Pi_xy, and neither has its force term w rho g xi_y
//  * body force g = (0, g) (Secs. 2.1, 2.2; forced): rho u_y = sum xi_y f~ + rho g hdt,
//    2 rho T gains 2 hdt rho g u_y, sigma_xy gains hdt rho g u_x (the xy moment of
//    the force term), hdt = dt/2 (Eq. 2order; 0 for the first-order scheme of
//    Eq. slb, whose stored variable is f itself), and the force term relaxed with
//    weight omega tau (= dt for Eq. slb, where omega = dt / tau),
//    omega tau g_a = omega w_a rho g sum_{ky>=1} c_kx c_{ky-1} He_kx He_ky / (kx! (ky-1)!),
//    folds into the y factors: c_ky -> c_ky + ky tau g c_{ky-1} (ky >= 1)
template <class VS, int N, class R, class T, bool COLLIDE, class F>
__device__ __forceinline__ CellOut<T> collide_cell(const Tab<R>& t, R rho0, R omega, R sigma_fac, int isothermal,
                                                   bool diag, bool forced, T gf, R tau, R hdt, F&& f) {
    constexpr int NA = VS::NA;
    const T zero = vsplat<T>(R(0));
    T C[NA], Ry[NA];
#pragma unroll
    for (int i = 0; i < NA; ++i) C[i] = Ry[i] = zero;
    static_for<0, VS::Q>([&](auto ac) {
        constexpr int a = decltype(ac)::value;
        const T v = f(ac);
        C[VS::ix(a)] = vadd(C[VS::ix(a)], v);
        Ry[VS::iy(a)] = vadd(Ry[VS::iy(a)], v);
    });
    T drho = C[0], jx = vmul(vsplat<T>(t.a[0]), C[0]), jy = vmul(vsplat<T>(t.a[0]), Ry[0]);
    T en = vmul(vsplat<T>(t.a2[0]), vadd(C[0], Ry[0]));
#pragma unroll
    for (int i = 1; i < NA; ++i) {
        drho = vadd(drho, C[i]);
        jx = vfma(vsplat<T>(t.a[i]), C[i], jx);
        jy = vfma(vsplat<T>(t.a[i]), Ry[i], jy);
        en = vfma(vsplat<T>(t.a2[i]), vadd(C[i], Ry[i]), en);
    }
    CellOut<T> o;
    T pxy = zero, h = zero;
    if (diag) {
        T P[NA];
#pragma unroll
        for (int i = 0; i < NA; ++i) P[i] = zero;
        static_for<0, VS::Q>([&](auto ac) {
            constexpr int a = decltype(ac)::value;
            const T v = f(ac);
            P[VS::ix(a)] = vfma(vsplat<T>(t.a[VS::iy(a)]), v, P[VS::ix(a)]);
            h = vfma(vmul(v, vsplat<T>(t.winv[a])), v, h);
        });
#pragma unroll
        for (int i = 0; i < NA; ++i) pxy = vfma(vsplat<T>(t.a[i]), P[i], pxy);
    }
    o.h = h;
    T cx[N + 1], cy[N + 1];
    const T rho = cell_state<N, R, T, COLLIDE>(rho0, sigma_fac, isothermal, forced, gf, tau, hdt, drho, jx, jy, en, pxy, o,
                                               cx, cy);
    if constexpr (COLLIDE) {
        T QY[NA][N + 1];
#pragma unroll
        for (int j = 0; j < NA; ++j) {
            QY[j][0] = vsplat<T>(t.wm[j]);
#pragma unroll
            for (int ky = 1; ky <= N; ++ky)
                QY[j][ky] = vmul(vsplat<T>(VS::kProductWeights ? t.whn[j][ky] : t.hn[j][ky]), cy[ky]);
            // FP32: the first-order factor's small second term (exact momentum identity)
            if constexpr (std::is_same<R, float>::value)
                QY[j][1] = vfma(vsplat<T>(VS::kProductWeights ? t.whn1lo[j] : t.hn1lo[j]), cy[1], QY[j][1]);
        }
        const T om1 = vsplat<T>(R(1) - omega);
        static_for<0, NA>([&](auto ic) {
            constexpr int I = decltype(ic)::value;
            // px[0] = sum_{kx>=1} cx hn (the kx = ky = 0 term is rho itself); px[ky>=1] = sum_{kx<=N-ky} cx hn
            T px[N + 1];
#pragma unroll
            for (int ky = 0; ky <= N; ++ky) {
                T sacc = ky == 0 ? zero : vsplat<T>(R(1));
#pragma unroll
                for (int kx = 1; kx <= N - ky; ++kx) sacc = vfma(cx[kx], vsplat<T>(t.hn[I][kx]), sacc);
                if constexpr (std::is_same<R, float>::value) {
                    if (ky == 0) sacc = vfma(cx[1], vsplat<T>(t.hn1lo[I]), sacc);
                }
                px[ky] = sacc;
            }
            if constexpr (VS::kProductWeights) {
                const T ow = vsplat<T>(t.ow[I]);
                T PX[N + 1];
                const T s0 = vfma(rho, px[0], drho);
                PX[0] = vmul(ow, s0);
                if constexpr (std::is_same<R, float>::value) PX[0] = vfma(vsplat<T>(t.owlo[I]), s0, PX[0]);
                const T owr = vmul(ow, rho);
#pragma unroll
                for (int ky = 1; ky <= N; ++ky) PX[ky] = vmul(owr, px[ky]);
                static_for<0, VS::Q>([&](auto ac) {
                    constexpr int a = decltype(ac)::value;
                    if constexpr (VS::ix(a) == I) {
                        constexpr int iy = VS::iy(a);
                        T od = vmul(PX[0], QY[iy][0]);
#pragma unroll
                        for (int ky = 1; ky <= N; ++ky) od = vfma(PX[ky], QY[iy][ky], od);
                        T& fa = f(ac);
                        fa = vfma(fa, om1, od);
                    }
                });
            } else {
                static_for<0, VS::Q>([&](auto ac) {
                    constexpr int a = decltype(ac)::value;
                    if constexpr (VS::ix(a) == I) {
                        constexpr int iy = VS::iy(a);
                        T sacc = px[0];
#pragma unroll
                        for (int ky = 1; ky <= N; ++ky) sacc = vfma(px[ky], QY[iy][ky], sacc);
                        T od = vmul(vsplat<T>(t.oww[a]), vfma(rho, sacc, drho));
                        if constexpr (std::is_same<R, float>::value && VS::kOnLattice) {
                            if constexpr (VS::ex(a) == 0 && VS::ey(a) == 0) od = vfma(vsplat<T>(t.mass_lo), drho, od);
                        }
                        T& fa = f(ac);
                        fa = vfma(fa, om1, od);
                    }
                });
            }
        });
    }
    return o;
}

// Amplitude A_f cos(phi n dt) of the body force at time level n (0 when unforced).
template <class R>
__device__ __forceinline__ R force_at_level(const Args<R>& A, long long lvl) {
    return A.force_amp != 0.0 ? (R)(A.force_amp * cos(A.force_freq * (double)lvl * A.dt)) : R(0);
}

// Tensor-product Lax-Wendroff of a velocity pair (a, a + 1) of one lane's cell: the y pass over
// the lane's column (values of the rows y - 1, y, y + 1), then the x pass, whose neighbours'
// columns come by shuffles.  The pair has one x node and two y nodes, so both passes run as
// packed f32x2 operations: 6 instead of 12 arithmetic instructions a pair, the same rounding.
// (32 levels: D2Q36-GH FP32 4096^2 28.7 -> 28.2 ms, D2Q64-GH FP16 2048^2 17.0 -> 16.4 ms.)
template <class VS, int A_>
__device__ __forceinline__ f2 lw_y_pair(const Tab<float>& t, f2 fm, f2 f0, f2 fp) {
    constexpr int iy = VS::iy(A_);
    const f2 l0 = f2{t.lwt[0][iy], t.lwt[0][iy + 1]}, l1 = f2{t.lwt[1][iy], t.lwt[1][iy + 1]},
             l2 = f2{t.lwt[2][iy], t.lwt[2][iy + 1]};
    return vfma(l0, fm, vfma(l1, f0, vmul(l2, fp)));
}
template <class VS, int A_>
__device__ __forceinline__ f2 lw_x_pair(const Tab<float>& t, f2 gl, f2 g, f2 gr) {
    constexpr int ix = VS::ix(A_);
    return vfma(vsplat<f2>(t.lw[ix][0]), gl, vfma(vsplat<f2>(t.lw[ix][1]), g, vmul(vsplat<f2>(t.lw[ix][2]), gr)));
}
__device__ __forceinline__ f2 shfl_up2(f2 v) {
    return f2{__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1)};
}
__device__ __forceinline__ f2 shfl_down2(f2 v) {
    return f2{__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1)};
}

// The collision of collide_cell with one cell per lane and the velocities taken in pairs (a, a + 1)
// of equal x node (a = ix NA + iy, iy even), each pair one packed f32x2 value: the
// per-velocity work (moment sums, diagnostics, equilibrium, relaxation) runs at half the
// instruction count.  Product-weight Gauss-Hermite sets (NA even), FP32 arithmetic.
// Moments as in collide_cell, with the y-node sums kept as pairs and the x-node sums
// reduced when the x node changes; H = sum_ix (1/W_ix) sum_iy d^2 / W_iy.
// ow, owlo, hn1lo, whn1lo: the relaxation tables of omega (Tab), the handle's own or, in a
// batch, the instance's.
template <class VS, int N, bool COLLIDE, class F>
__device__ __forceinline__ CellOut<float> collide_cell_pairs(const Tab<float>& t, const float* ow_t, const float* owlo_t,
                                                             const float* hn1lo_t, const float* whn1lo_t,
                                                             float rho0, float omega, float sigma_fac, int isothermal,
                                                             bool diag, bool forced, float gf, float tau, float hdt,
                                                             F&& fpair) {
    using R = float;
    constexpr int NA = VS::NA, NP = VS::Q / 2, NJ = NA / 2;
    const f2 z2 = f2{0.f, 0.f};
    f2 Ryp[NJ];
    R C[NA];
#pragma unroll
    for (int j = 0; j < NJ; ++j) Ryp[j] = z2;
    // x-node sums, one pair accumulator live at a time (the pairs come in x-node order)
    static_for<0, NA>([&](auto ic) {
        constexpr int I = decltype(ic)::value;
        f2 cp = z2;
        static_for<0, NJ>([&](auto jc) {
            constexpr int J = decltype(jc)::value;
            const f2 v = fpair(std::integral_constant<int, I * NJ + J>{});
            cp = vadd(cp, v);
            Ryp[J] = vadd(Ryp[J], v);
        });
        C[I] = cp.x + cp.y;
    });
    R drho = C[0], jx = t.a[0] * C[0];
    R en = t.a2[0] * C[0];
#pragma unroll
    for (int i = 1; i < NA; ++i) {
        drho += C[i];
        jx = fmaf(t.a[i], C[i], jx);
        en = fmaf(t.a2[i], C[i], en);
    }
    f2 jyp = z2, eyp = z2;
#pragma unroll
    for (int j = 0; j < NJ; ++j) {
        jyp = vfma(f2{t.a[2 * j], t.a[2 * j + 1]}, Ryp[j], jyp);
        eyp = vfma(f2{t.a2[2 * j], t.a2[2 * j + 1]}, Ryp[j], eyp);
    }
    R jy = jyp.x + jyp.y;
    en += eyp.x + eyp.y;
    CellOut<R> o;
    R pxy = 0.f, h = 0.f;
    if (diag) {
        static_for<0, NA>([&](auto ic) {
            constexpr int I = decltype(ic)::value;
            f2 pp = z2, hp = z2;
            static_for<0, NJ>([&](auto jc) {
                constexpr int J = decltype(jc)::value;
                const f2 v = fpair(std::integral_constant<int, I * NJ + J>{});
                pp = vfma(f2{t.a[2 * J], t.a[2 * J + 1]}, v, pp);
                hp = vfma(vmul(v, f2{t.wminv[2 * J], t.wminv[2 * J + 1]}), v, hp);
            });
            pxy = fmaf(t.a[I], pp.x + pp.y, pxy);
            h = fmaf(t.wminv[I], hp.x + hp.y, h);
        });
    }
    o.h = h;
    R cx[N + 1], cy[N + 1];
    const R rho = cell_state<N, R, R, COLLIDE>(rho0, sigma_fac, isothermal, forced, gf, tau, hdt, drho, jx, jy, en, pxy, o,
                                               cx, cy);
    if constexpr (COLLIDE) {
        // y factors of the y-node pairs: QY[j][ky] = W_j He_ky(a_j)/ky! c_ky(u_y)
        f2 QYp[NJ][N + 1];
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
            QYp[j][0] = f2{t.wm[2 * j], t.wm[2 * j + 1]};
#pragma unroll
            for (int ky = 1; ky <= N; ++ky)
                QYp[j][ky] = vmul(f2{t.whnt[ky][2 * j], t.whnt[ky][2 * j + 1]}, vsplat<f2>(cy[ky]));
            // the first-order factor's small second term (exact momentum identity)
            QYp[j][1] = vfma(f2{whn1lo_t[2 * j], whn1lo_t[2 * j + 1]}, vsplat<f2>(cy[1]), QYp[j][1]);
        }
        const f2 om1 = vsplat<f2>(1.f - omega);
        static_for<0, NA>([&](auto ic) {
            constexpr int I = decltype(ic)::value;
            R PX[N + 1];
            {
                R px[N + 1];
#pragma unroll
                for (int ky = 0; ky <= N; ++ky) {
                    R sacc = ky == 0 ? 0.f : 1.f;
#pragma unroll
                    for (int kx = 1; kx <= N - ky; ++kx) sacc = fmaf(cx[kx], t.hn[I][kx], sacc);
                    if (ky == 0) sacc = fmaf(cx[1], hn1lo_t[I], sacc);
                    px[ky] = sacc;
                }
                const R ow = ow_t[I];
                const R s0 = fmaf(rho, px[0], drho);
                PX[0] = fmaf(owlo_t[I], s0, __fmul_rn(ow, s0));
                const R owr = __fmul_rn(ow, rho);
#pragma unroll
                for (int ky = 1; ky <= N; ++ky) PX[ky] = __fmul_rn(owr, px[ky]);
            }
            static_for<0, NJ>([&](auto jc) {
                constexpr int J = decltype(jc)::value;
                f2 od = vmul(vsplat<f2>(PX[0]), QYp[J][0]);
#pragma unroll
                for (int ky = 1; ky <= N; ++ky) od = vfma(vsplat<f2>(PX[ky]), QYp[J][ky], od);
                f2& fa = fpair(std::integral_constant<int, I * NJ + J>{});
                fa = vfma(fa, om1, od);
            });
        });
    }
    return o;
}

// Collision and store (or the moment outputs) of the V cells (g.x .., y) whose
// streamed populations are in ft.  Diagnostics are reduced over the warp in
// FP32 and added to acc (lane 0) in FP64.
// OSTRIDE > 0 (store-staged kernel): the relaxed populations go to the warp's output slot in shared
// memory, out[m * OSTRIDE] for plane m, instead of to HBM (the periodic images in the ghost
// rim are still written here).
template <class VS, int N, class S, class R, int V, int KIND, class T, int OSTRIDE = 0>
__device__ __forceinline__ void collide_store(const Args<R>& A, T (&ft)[VS::Q], S* dst, int y,
                                              const Lane& g, bool diag, R (&acc)[6], int lane, long long lvl,
                                              R gt, typename Layout<VS, S>::E* out = nullptr) {
    constexpr int Q = VS::Q;
    static_assert(OSTRIDE == 0 || V == 1, "output slot: one cell per lane");
    // body force g_y(x_i, t_n) = gt sin(x_i), gt = A_f cos(phi t_n) (driven standing wave, Sec. 4);
    // compiled out of the unforced step kernels
    constexpr bool STEP = (KIND == kStep || KIND == kStepForced);
    const bool forced = (KIND != kStep) && A.force_amp != 0.0;
    // sin(x_i), cos(x_i) of the diagnostics, loaded before the collision so that their
    // latency hides behind it (index clamped: lanes that own no cell add nothing)
    constexpr bool PF =
        LB_DIAG_PREFETCH > 0 || (LB_DIAG_PREFETCH < 0 && ((!VS::kOnLattice && VS::Q == 16) || OSTRIDE > 0));
    R dsin[V], dcos[V];
    if constexpr (STEP && PF) {
        if (diag) {
#pragma unroll
            for (int k = 0; k < V; ++k) {
                const int xi = min(max(g.x + k, 0), A.nx - 1);
                dsin[k] = __ldg(A.sinx + xi);
                dcos[k] = __ldg(A.cosx + xi);
            }
        }
    }
    T gf = vsplat<T>(R(0));
    if (forced) {
        R gl[V];
#pragma unroll
        for (int k = 0; k < V; ++k) gl[k] = gt * A.sinx[min(max(g.x + k, 0), A.nx - 1)];
        if constexpr (V == 2) {
            gf = pack_lanes<T, R>(gl[0], gl[1]);
        } else {
            gf = gl[0];
        }
    }
    CellOut<T> co;
    if constexpr (Layout<VS, S>::PAIRED) {
        // one cell per lane: velocity pairs as packed f32x2 values
        constexpr int NP = Q / 2;
        f2 fp[NP];
        static_for<0, NP>([&](auto mc) {
            constexpr int m = decltype(mc)::value;
            fp[m] = f2{ft[2 * m], ft[2 * m + 1]};
        });
        co = collide_cell_pairs<VS, N, STEP>(
            A.tab, A.tab.ow, A.tab.owlo, A.tab.hn1lo, A.tab.whn1lo, A.rho0, A.omega, A.sigma_fac, A.isothermal, diag || KIND == kMoments, forced, gf, A.tau,
            A.hdt, [&](auto mc) -> f2& { return fp[decltype(mc)::value]; });
        static_for<0, NP>([&](auto mc) {
            constexpr int m = decltype(mc)::value;
            ft[2 * m] = fp[m].x;
            ft[2 * m + 1] = fp[m].y;
        });
    } else {
        co = collide_cell<VS, N, R, T, STEP>(
            A.tab, A.rho0, A.omega, A.sigma_fac, A.isothermal, diag || KIND == kMoments, forced, gf, A.tau,
            A.hdt, [&](auto ac) -> T& { return ft[decltype(ac)::value]; });
    }
    if constexpr (KIND == kMoments) {
        if (g.own) {
            static_for<0, V>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                const long long c = (long long)y * A.nx + g.x + k;
                if (A.o_rho) A.o_rho[c] = (double)A.rho0 + (double)lane_get<k>(co.drho);
                if (A.o_ux) A.o_ux[c] = (double)lane_get<k>(co.ux);
                if (A.o_uy) A.o_uy[c] = (double)lane_get<k>(co.uy);
                if (A.o_T) A.o_T[c] = 1.0 + (double)lane_get<k>(co.th);
                if (A.o_sxy) A.o_sxy[c] = (double)lane_get<k>(co.sig);
                if (A.o_pop) {
                    const long long pl = (long long)A.ny * A.nx;
#pragma unroll
                    for (int a = 0; a < Q; ++a)
                        A.o_pop[a * pl + c] = (double)A.tab.w[a] * (double)A.rho0 + (double)lane_get<k>(ft[a]);
                }
            });
        }
    }
    if constexpr (STEP) {
        // The relaxed populations, straight from registers: to the cell (OSTRIDE > 0: to the
        // output slot) and, for the lanes of a boundary, to its periodic images in the ghost rim.
        // put(p) writes all planes at offset p of the first; each call draws the 16-bit rounding
        // bits anew from the cell's own stream, so every image holds the cell's bits.
        using E = typename Layout<VS, S>::E;
        auto put = [&](E* p, long long stride) {
            if constexpr (Layout<VS, S>::PAIRED) {
                uint32_t r0 = 0, r1 = 0;
                if constexpr (Is16<S>::value) r1 = sr_seed(lvl, (long long)y * A.nx + g.x);
                static_for<0, Q / 2>([&](auto mc) {
                    constexpr int a = 2 * decltype(mc)::value;
                    if constexpr (Is16<S>::value) {
                        r0 = sr_next(r1);
                        r1 = sr_next(r0);
                    }
                    *p = to_storage_pair<S>(f2{ft[a], ft[a + 1]},
                                            f2{store_scale<S, R>(A.tab, a), store_scale<S, R>(A.tab, a + 1)}, r0, r1);
                    p += stride;
                });
            } else {
                static_for<0, Q>([&](auto ac) {
                    constexpr int a = decltype(ac)::value;
                    if constexpr (V == 2) {
                        __stcs(reinterpret_cast<float2*>(p), make_float2(ft[a].x, ft[a].y));
                    } else {
                        *p = ft[a];
                    }
                    p += stride;
                });
            }
        };
        if (g.own) {
            E* const base = reinterpret_cast<E*>(dst) + A.origin;
            if constexpr (OSTRIDE > 0) {
                put(out, OSTRIDE);
                if (has_images<R, V>(A, g.x, y))
                    for_images<R, V>(A, g.x, y,
                                     [&](int xi, int yi) { put(base + (long long)yi * A.pitch + xi, A.plane); });
            } else {
                // the cell, then (lanes of a boundary) its images: one copy of the stores
                int xi = g.x, yi = y;
                bool more = has_images<R, V>(A, g.x, y), self = true;
                for (;;) {
                    put(base + (long long)yi * A.pitch + xi, A.plane);
                    if (!more) break;
                    do {
                        if (self) {  // to the first position, at the lowest row and column
                            while (yi - A.ny >= -A.gy) yi -= A.ny;
                            while (xi - A.nx >= -kGhostX) xi -= A.nx;
                            self = false;
                        } else if ((xi += A.nx) + V > A.nx + kGhostX) {
                            while (xi - A.nx >= -kGhostX) xi -= A.nx;
                            yi += A.ny;
                        }
                    } while (xi == g.x && yi == y);
                    if (yi >= A.ny + A.gy) break;
                }
            }
        }
    }
    if constexpr (STEP) {
        // per-thread partial sums over the thread's cells of every tile; reduced once per
        // launch (warp, then FP64 across warps and blocks) in finish_step
        if (diag && g.own) {
            static_for<0, V>([&](auto kc) {
                constexpr int k = decltype(kc)::value;
                acc[0] += lane_get<k>(co.drho);
                acc[1] += lane_get<k>(co.jx);
                acc[2] += lane_get<k>(co.jy);
                if constexpr (!PF) {
                    dsin[k] = A.sinx[g.x + k];
                    dcos[k] = A.cosx[g.x + k];
                }
                acc[3] = fma(lane_get<k>(co.uy), dsin[k], acc[3]);
                acc[4] = fma(lane_get<k>(co.sig), dcos[k], acc[4]);
                acc[5] += lane_get<k>(co.h);
            });
        }
    }
}

// Diagnostics of a step launch: each thread sums its own cells in R for at most kDiagFold
// tiles, then the warp folds those partials (a shuffle sum of 32 values) into its FP64 sums
// in shared memory (wsum[warp], lane 0), so the grid sums are FP64 sums of short partials at
// any grid size (a thread's cells per launch grow with the grid: ~200 at 4096^2, ~3300 at
// 16384^2).  Cost of the folds, D2Q36-GH FP32 at 4096^2 (GLUPS): every 16 tiles 17.74,
// every 64 17.87, only at the end 17.94.
#ifndef LB_DIAG_FOLD
#define LB_DIAG_FOLD 64
#endif
constexpr int kDiagFold = LB_DIAG_FOLD;

template <class R>
__device__ __forceinline__ void fold_diag(R (&acc)[6], double* wsum, int lane) {
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const R sm = warp_sum(acc[i]);
        if (lane == 0) wsum[i] += (double)sm;
        acc[i] = R(0);
    }
}

// The record of level lvl from the nb FP64 sums of a launch (kDiagSlots doubles each), added in a
// fixed order by the block that calls it: eight lanes take the quantities of one, the others
// further ones.  Sets the status word where a sum is not finite.
template <class R>
__device__ __forceinline__ void write_record(const Args<R>& A, const double* part, int nb, long long lvl) {
    __shared__ double tot[32][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)blockDim.x >> 5, q = threadIdx.x & 7;
    double s = 0.0;
    for (int b = threadIdx.x >> 3; b < nb; b += (int)blockDim.x >> 3)
        s += __ldcg(part + (long long)b * kDiagSlots + min(q, 5));
    s += __shfl_xor_sync(0xffffffffu, s, 8);
    s += __shfl_xor_sync(0xffffffffu, s, 16);
    if (nw > 1) {
        if (lane < 8) tot[warp][lane] = s;
        __syncthreads();
        if (warp > 0) return;
        s = 0.0;
        for (int w = 0; w < nw; ++w) s += tot[w][q];
    }
    // lane 0..7: mass, mom_x, mom_y, amp, shear, hnorm, t, flags
    const double v = q == 6 ? (double)lvl * A.dt : (q == 3 || q == 4 ? s * A.norm : (q == 0 ? A.mass0 + s : s));
    const bool bad = __any_sync(0xffffffffu, (q == 0 || q == 3 || q == 5) && !isfinite(v));
    double* r = reinterpret_cast<double*>(A.ring + (lvl / A.diag_every) % A.ring_cap);
    if (lane < 8) r[q == 6 ? 0 : (q == 7 ? 7 : q + 1)] = q == 7 ? (bad ? 1.0 : 0.0) : v;
    if (bad && lane == 0) atomicOr(A.status, 1);
}

// Step launches of a captured chain (plain-load and node-split kernels) leave the summing of their
// blocks' partials to the launch behind them, which has a block of its own for it (A.pending), and
// only the last launch of a chain sums its own and advances the level counter (A.advance levels):
// the fence, the ticket and the last block's pass over the partials, ~1.3 to 2.3 us at the end of a
// launch, are then not between two levels (256^2 D2Q36-GH FP32: 15.5 -> 10.0 us a level).  Blocks that
// step cells:
template <class R>
__device__ __forceinline__ int work_blocks(const Args<R>& A) {
    return (int)gridDim.x - A.pending;
}
template <class R>
__device__ __forceinline__ double* partials_of(const Args<R>& A, int parity) {
    return A.partials + (long long)parity * A.partial_stride;
}

// End of a launch once the block's partials are written (every thread of the block calls it): the
// last block to come here writes the launch's record and advances the level.
template <class R>
__device__ __forceinline__ void close_level(const Args<R>& A, long long lvl, bool diag) {
    if (A.advance == 0) return;  // the next launch writes the record
    __shared__ bool is_last;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        is_last = atomicAdd(A.ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    if (threadIdx.x == 0) {
        *A.level = lvl - A.level_add + A.advance;
        *A.ticket = 0u;
    }
    if (diag) write_record(A, partials_of(A, A.level_add & 1), A.nparts, lvl);
}

// The block beside the working ones: the record of the launch before.
template <class R>
__device__ __forceinline__ void pending_record(const Args<R>& A, long long lvl) {
    if (A.diag_every > 0 && (lvl - 1) % A.diag_every == 0) write_record(A, partials_of(A, (A.level_add - 1) & 1), A.nparts, lvl - 1);
    close_level(A, lvl, A.diag_every > 0 && lvl % A.diag_every == 0);
}

// End of a working block: the last fold, the block's FP64 partials, then close_level.  All threads
// of the block call it; wsum holds the per-warp FP64 sums (zeroed by each warp's lane 0 before its
// first fold).
template <class R, int NWARPS_DIAG>
__device__ __forceinline__ void finish_step(const Args<R>& A, R (&acc)[6], double (*wsum)[6], long long lvl,
                                            bool diag, int warp, int lane) {
    if (diag && warp < NWARPS_DIAG) fold_diag(acc, wsum[warp], lane);
    __syncthreads();
    if (diag && threadIdx.x < 6) {
        double s = 0.0;
        for (int w = 0; w < NWARPS_DIAG; ++w) s += wsum[w][threadIdx.x];
        partials_of(A, A.level_add & 1)[(long long)blockIdx.x * kDiagSlots + threadIdx.x] = s;
    }
    close_level(A, lvl, diag);
}

// Programmatic dependent launch: a step launch may start while the one before it ends (its blocks
// take the SMs that are free, set up and wait here); what that launch wrote is read only after
// this.  It then lets the launch after it do the same.  No effect on a launch without the attribute.
__device__ __forceinline__ void await_previous_step() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ------------------------------------------------------------ register kernel
// KIND = kStep:    f* (next level) into dst, diagnostics when due.
// KIND = kStepForced: the same with the body force (lb_params.force_amp != 0).
// KIND = kMoments: per-cell rho, u, T, sigma_xy (and optionally f~) of the level; no store.
// UPW: off-lattice streaming by second-order upwind instead of Lax-Wendroff.
template <class VS, int N, class S, class R, int KIND, bool UPW = false>
__global__ void __launch_bounds__(Cfg<VS, S>::THREADS, Cfg<VS, S>::MINB)
    lb_fused_kernel(const __grid_constant__ Args<R> A) {
    constexpr int Q = VS::Q;
    constexpr int V = Cfg<VS, S>::V;
    constexpr int ROWS = Cfg<VS, S>::ROWS;
    constexpr bool HALO = Cfg<VS, S>::HALO && !UPW;
    constexpr int TW = HALO ? Cfg<VS, S>::TW : 32 * V;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const S* src = static_cast<const S*>(A.src);
    S* dst = static_cast<S*>(A.dst);

    constexpr bool STEP = (KIND == kStep || KIND == kStepForced);
    long long lvl = 0;
    bool diag = false;
    if constexpr (STEP) {
        await_previous_step();
        lvl = __ldcg(A.level) + A.level_add;
        diag = (A.diag_every > 0) && (lvl % A.diag_every == 0);
        if (A.pending && (int)blockIdx.x == work_blocks(A)) {
            pending_record(A, lvl);
            return;
        }
    } else {
        // force phase of the state's level n: the device counter already points past it
        // (the launch that produced f*(n) advanced it to n + 1)
        if (A.force_amp != 0.0) lvl = __ldcg(A.level) - 1;
    }
    R gt = R(0);
    if constexpr (KIND != kStep) gt = force_at_level(A, lvl);
    R acc[6] = {0, 0, 0, 0, 0, 0};
    __shared__ double wsum[ROWS][6];
    if (lane == 0) {
#pragma unroll
        for (int i = 0; i < 6; ++i) wsum[warp][i] = 0.0;
    }
    int nfold = 0;

    const int nb = work_blocks(A);
    for (int tile = blockIdx.x; tile < A.ntiles; tile += nb) {
        const int ty = tile / A.ntiles_x;
        const int tx = tile - ty * A.ntiles_x;
        const int y = ty * ROWS + warp;
        if (y >= A.ny) continue;  // warp-uniform
        const int tile_start = tx * TW;
        const int x0 = (tx == A.ntiles_x - 1) ? A.x0_last : tile_start;
        const Lane g = HALO ? halo_lane_geometry(lane, x0, tile_start, A.nx) : lane_geometry<V>(lane, x0, tile_start, A.nx);

        using T = typename Pack<R, V>::T;
        T ft[Q];
        if constexpr (HALO) {
            // velocity pairs, as in the TMA-staged kernel (columns past nx + 1 of a grid narrower
            // than a warp lie in the row's padding and reach no cell)
            using E = typename Layout<VS, S>::E;
            const E* p = reinterpret_cast<const E*>(src) + A.origin + (long long)y * A.pitch + g.xl;
            // (the initial state is read as it is; the branch lies outside the velocity loop, whose
            // loads it would keep apart)
            auto put = [&](auto mc, f2 v) {
                constexpr int a = 2 * decltype(mc)::value;
                // the stencil is linear: 16-bit values are scaled once, after it
                if constexpr (Is16<S>::value)
                    v = vmul(v, f2{load_scale<S, R>(A.tab, a), load_scale<S, R>(A.tab, a + 1)});
                ft[a] = v.x;
                ft[a + 1] = v.y;
            };
            if (A.raw) {
                static_for<0, Q / 2>([&](auto mc) {
                    put(mc, ld_pair<S>(p));
                    p += A.plane;
                });
            } else {
                static_for<0, Q / 2>([&](auto mc) {
                    constexpr int a = 2 * decltype(mc)::value;
                    const f2 gv = lw_y_pair<VS, a>(A.tab, ld_pair<S>(p - A.pitch), ld_pair<S>(p), ld_pair<S>(p + A.pitch));
                    put(mc, lw_x_pair<VS, a>(A.tab, shfl_up2(gv), gv, shfl_down2(gv)));
                    p += A.plane;
                });
            }
        } else {
            static_for<0, Q>([&](auto ac) {
                constexpr int a = decltype(ac)::value;
                constexpr int VW = Layout<VS, S>::VW;
                const S* pl = src + pop_index<VS, S>(a, A.plane, A.origin);
                if (A.raw) {
                    const S* p = pl + VW * ((long long)y * A.pitch + g.xl);
                    ft[a] = ld_cells<T>(p);
                } else if constexpr (VS::kOnLattice) {
                    // exact shift: f~_a(x, y) = f*_a(x - ex, y - ey)
                    constexpr int ex = VS::ex(a), ey = VS::ey(a);
                    const S* p = pl + (long long)(y - ey) * A.pitch + g.xl - ex;
                    if constexpr (V == 2 && ex % 2 != 0) {
                        ft[a] = pack_lanes<T, R>(p[0], p[1]);
                    } else {
                        ft[a] = ld_cells<T>(p);
                    }
                } else if constexpr (UPW) {
                    // tensor-product second-order upwind (Beam-Warming), one cell per lane: y pass
                    // over the cell's row and the two upstream rows, x pass by shuffles from the two
                    // upstream lanes; the two lanes at the warp's downstream edge compute the two
                    // upstream columns outside the warp
                    static_assert(V == 1 && !Is16<S>::value, "upwind streaming: one cell per lane, 32/64-bit");
                    constexpr int ix = VS::ix(a), iy = VS::iy(a);
                    constexpr int sx = VS::axis_sign(ix), sy = VS::axis_sign(iy);
                    const R yf = A.tab.uw[iy][0], yn = A.tab.uw[iy][1], ys = A.tab.uw[iy][2];
                    const R xf = A.tab.uw[ix][0], xn = A.tab.uw[ix][1], xs = A.tab.uw[ix][2];
                    const S* r0 = pl + VW * (long long)y * A.pitch;
                    const S* rn = r0 - VW * (long long)sy * A.pitch;
                    const S* rf = r0 - VW * 2LL * sy * A.pitch;
                    // lanes past the grid read the images of columns 0 and 1 (nx, nx + 1)
                    const int xu = VW * min(g.x, A.nx + 1);
                    const R gv = fma(yf, rf[xu], fma(yn, rn[xu],
                                                                     ys * r0[xu]));
                    // extra column: x0 - 2 + (lane & 1) (lanes 30, 31) for sx > 0,
                    // x0 + 32 + (lane & 1) (lanes 0, 1) for sx < 0, clamped into the rim
                    const int xe = VW * (sx > 0 ? x0 - 2 + (lane & 1) : min(x0 + 32 + (lane & 1), A.nx + 1));
                    const R ge = fma(yf, rf[xe], fma(yn, rn[xe],
                                                                     ys * r0[xe]));
                    R g1, g2;
                    if constexpr (sx > 0) {
                        g1 = __shfl_up_sync(0xffffffffu, gv, 1);
                        g2 = __shfl_up_sync(0xffffffffu, gv, 2);
                        const R e2 = __shfl_sync(0xffffffffu, ge, 30);  // column x0 - 2
                        const R e1 = __shfl_sync(0xffffffffu, ge, 31);  // column x0 - 1
                        if (lane == 0) { g1 = e1; g2 = e2; }
                        if (lane == 1) g2 = e1;
                    } else {
                        g1 = __shfl_down_sync(0xffffffffu, gv, 1);
                        g2 = __shfl_down_sync(0xffffffffu, gv, 2);
                        const R e1 = __shfl_sync(0xffffffffu, ge, 0);   // column x0 + 32
                        const R e2 = __shfl_sync(0xffffffffu, ge, 1);   // column x0 + 33
                        if (lane == 31) { g1 = e1; g2 = e2; }
                        if (lane == 30) g2 = e1;
                    }
                    ft[a] = fma(xf, g2, fma(xn, g1, xs * gv));
                } else {
                    // tensor-product Lax-Wendroff (FP64): y pass in registers, x pass by shuffles; the
                    // warp's two edge lanes take their outer neighbour from one extra column
                    static_assert(V == 1 && VW == 1, "one cell per lane, one velocity a plane");
                    constexpr int ix = VS::ix(a), iy = VS::iy(a);
                    const R ly0 = A.tab.lw[iy][0], ly1 = A.tab.lw[iy][1], ly2 = A.tab.lw[iy][2];
                    const R lx0 = A.tab.lw[ix][0], lx1 = A.tab.lw[ix][1], lx2 = A.tab.lw[ix][2];
                    const S* r0 = pl + (long long)y * A.pitch;
                    const S* rm = r0 - A.pitch;
                    const S* rp = r0 + A.pitch;
                    const int xe = (lane == 31) ? min(x0 + TW, A.nx) : x0 - 1;
                    const R ge = fma(ly0, rm[xe], fma(ly1, r0[xe], ly2 * rp[xe]));
                    const R f0 = r0[g.xl];
                    const R fm = rm[g.xl];
                    const R fp = rp[g.xl];
                    const R gv = fma(ly0, fm, fma(ly1, f0, ly2 * fp));
                    R gl = __shfl_up_sync(0xffffffffu, gv, 1);
                    R gr = __shfl_down_sync(0xffffffffu, gv, 1);
                    gl = (lane == 0) ? ge : gl;
                    gr = (lane == 31) ? ge : gr;
                    ft[a] = fma(lx0, gl, fma(lx1, gv, lx2 * gr));
                }
            });
        }
        collide_store<VS, N, S, R, V, KIND>(A, ft, dst, y, g, diag, acc, lane, lvl, gt);
        if (STEP && diag && ++nfold == kDiagFold) {  // warp-uniform
            fold_diag(acc, wsum[warp], lane);
            nfold = 0;
        }
    }
    if constexpr (STEP) finish_step<R, ROWS>(A, acc, wsum, lvl, diag, warp, lane);
}

// ------------------------------------------------------------ node-split step kernel
// FP64 Lax-Wendroff steps of small grids.  The card does two FP64 operations a clock and SM, so a
// warp of 32 cells holds its SM for as long as its q x ~20 operations a cell take, while a small
// grid leaves most SMs without a warp.  Here NA lanes share a cell, lane i holding the NA
// velocities of x node i: a warp of 32 / NA cells, so that the same grid gives NA times as many
// warps of an NA-th of the work each (blocks of one or four warps, so that they spread over the SMs
// and then over an SM's four FP64 units: blocks of one warp put their warps on one unit, 128 x 64
// D2Q16-GH 74 us a level).  Sums over the
// y node and the equilibrium's own factors stay in the lane; sums over the x nodes go through
// shared memory and run in the lanes side by side, lane r summing moment r, each in the order of
// collide_cell, so the populations are those of the plain-load kernel bit for bit.
// H is summed by lane (its rounding differs from the plain-load kernel's).
template <class VS>
struct SplitCfg {
    static constexpr int NA = VS::NA;
    static constexpr int CELLS = 32 / NA;  // cells of a warp (6 nodes: lanes 30, 31 repeat the last cell's)
    // FP64 operations of a warp, about: of this kernel and of the plain-load kernel
    static constexpr int OPS = 17 * NA + 75, PLAIN_OPS = 19 * VS::Q + 100;
};

// Sums of six values over the warp in eight additions (halves, quarters and eighths of the warp
// part with the values between them); value i is returned in lane sum6_lane(i).
__device__ __forceinline__ double warp_sum6(const double (&a)[6], int lane) {
    constexpr unsigned m = 0xffffffffu;
    const bool h = lane & 16, q = lane & 8, e = lane & 4;
    double x[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) x[k] = (h ? a[k + 3] : a[k]) + __shfl_xor_sync(m, h ? a[k] : a[k + 3], 16);
    // x[0], x[1] to the first quarter of each half, x[2] to the second
    double y0 = (q ? x[2] : x[0]) + __shfl_xor_sync(m, q ? x[0] : x[2], 8);
    const double r1 = __shfl_xor_sync(m, x[1], 8);
    const double y1 = q ? 0.0 : x[1] + r1;
    double z = (e ? y1 : y0) + __shfl_xor_sync(m, e ? y0 : y1, 4);
    z += __shfl_xor_sync(m, z, 2);
    z += __shfl_xor_sync(m, z, 1);
    return z;
}
__device__ __forceinline__ int sum6_index(int lane) {  // the value a lane holds the sum of, or -1
    switch (lane) {
        case 0: return 0;
        case 4: return 1;
        case 8: return 2;
        case 16: return 3;
        case 20: return 4;
        case 24: return 5;
        default: return -1;
    }
}

template <class VS, int N, int KIND, int W>
__global__ void __launch_bounds__(32 * W) lb_split_kernel(const __grid_constant__ Args<double> A) {
    static_assert(KIND == kStep || KIND == kStepForced, "node-split kinds: step, forced step");
    constexpr int NA = VS::NA, CELLS = SplitCfg<VS>::CELLS, PAD = NA + 1;
    constexpr int ROLES = NA > 4 ? 5 : 4;  // moments summed side by side (pxy apart where the lanes do not reach)
    constexpr int EDGE = (2 * NA + CELLS - 1) / CELLS;  // edge columns' y passes of a lane
    const int lane = threadIdx.x & 31, warp = W == 1 ? 0 : threadIdx.x >> 5;
    const int c = min(lane / NA, CELLS - 1), i = lane % NA;
    const bool first = lane < CELLS * NA;  // not a repeat
    const double* src = static_cast<const double*>(A.src);
    double* dst = static_cast<double*>(A.dst);
    struct Warp {
        double sv[CELLS][NA][PAD];    // streamed values, [cell][x node][y node]
        double se[NA][2][PAD];        // y passes of the columns beside the warp, [x node][side][y node]
        double sm[CELLS][4][PAD];     // by node: C (sums over y nodes), Ry (over x nodes), C + Ry, P
        double sq[CELLS][NA][N + 1];  // y factors of the equilibrium
    };
    __shared__ Warp shared[W];
    auto& sv = shared[warp].sv;
    auto& se = shared[warp].se;
    auto& sm = shared[warp].sm;
    auto& sq = shared[warp].sq;
    // the lane's x node, and its role's coefficients of the nodes
    const Tab<double>& t = A.tab;
    const double lx0 = t.lw[i][0], lx1 = t.lw[i][1], lx2 = t.lw[i][2];
    const double ow = t.ow[i], wmi = t.wm[i], winvi = t.wminv[i];
    double hn[N + 1], whn[N + 1], role[NA];
#pragma unroll
    for (int k = 1; k <= N; ++k) {
        hn[k] = t.hn[i][k];
        whn[k] = t.whn[i][k];
    }
#pragma unroll
    for (int k = 0; k < NA; ++k) role[k] = i == 0 ? 1.0 : (i == 3 ? t.a2[k] : t.a[k]);
    const int role_sum = i == 2 ? 1 : (i == 3 ? 2 : (i == 4 ? 3 : 0));
    await_previous_step();
    const long long lvl = __ldcg(A.level) + A.level_add;
    const bool diag = (A.diag_every > 0) && (lvl % A.diag_every == 0);
    const bool forced = KIND == kStepForced;
    const int nb = work_blocks(A);
    if (A.pending && (int)blockIdx.x == nb) {
        pending_record(A, lvl);
        return;
    }
    // y node of edge pass e (of 2 NA: the left column's, then the right one's; any node past them)
    auto edge_node = [](int e) { return e < NA ? e : (e < 2 * NA ? e - NA : 0); };
    double acc[6] = {0, 0, 0, 0, 0, 0};
    const double om1 = 1.0 - A.omega;
    double gt = 0.0;
    bool have_gt = false;

    for (int tile = (int)blockIdx.x * W + warp; tile < A.ntiles; tile += nb * W) {
        const int y = tile / A.ntiles_x, x0 = (tile - y * A.ntiles_x) * CELLS;
        const int x = x0 + c;
        const bool own = first && x < A.nx;
        const double* r0 = src + (long long)(i * NA) * A.plane + A.origin + (long long)y * A.pitch;
        // the columns beside the warp (x0 - 1 and x0 + CELLS): their 2 NA y passes of x node i are
        // shared out over the lanes of that node
        double em[EDGE], e0[EDGE], ep[EDGE];
#pragma unroll
        for (int k = 0; k < EDGE; ++k) {
            const int e = k * CELLS + c;
            const double* p = r0 + edge_node(e) * A.plane + (e < NA ? x0 - 1 : min(x0 + CELLS, A.nx));
            em[k] = p[-A.pitch];
            e0[k] = *p;
            ep[k] = p[A.pitch];
        }
        double vm[NA], v0[NA], vp[NA];
#pragma unroll
        for (int j = 0; j < NA; ++j) {
            const double* p = r0 + j * A.plane + min(x, A.nx);
            vm[j] = p[-A.pitch];
            v0[j] = *p;
            vp[j] = p[A.pitch];
        }
        if (forced && !have_gt) {  // (its cosine while the loads are on their way)
            gt = force_at_level(A, lvl);
            have_gt = true;
        }
        const double sx = __ldg(A.sinx + min(x, A.nx - 1)), cxs = __ldg(A.cosx + min(x, A.nx - 1));
#pragma unroll
        for (int k = 0; k < EDGE; ++k) {
            const int e = k * CELLS + c, j = edge_node(e);
            const double ge = fma(t.lw[j][0], em[k], fma(t.lw[j][1], e0[k], t.lw[j][2] * ep[k]));
            if (first && e < 2 * NA) se[i][e < NA ? 0 : 1][j] = ge;
        }
        __syncwarp();
        double f[NA], C = 0.0, P = 0.0, h = 0.0;
#pragma unroll
        for (int j = 0; j < NA; ++j) {
            const double g = fma(t.lw[j][0], vm[j], fma(t.lw[j][1], v0[j], t.lw[j][2] * vp[j]));
            double gl = __shfl_sync(0xffffffffu, g, max(c - 1, 0) * NA + i);
            double gr = __shfl_sync(0xffffffffu, g, min(c + 1, CELLS - 1) * NA + i);
            const double el = se[i][0][j], er = se[i][1][j];
            gl = c == 0 ? el : gl;
            gr = c == CELLS - 1 ? er : gr;
            f[j] = fma(lx0, gl, fma(lx1, g, lx2 * gr));
            C = __dadd_rn(C, f[j]);
            if (diag) {
                P = fma(t.a[j], f[j], P);
                h = fma(__dmul_rn(f[j], t.wminv[j]), f[j], h);
            }
            sv[c][i][j] = f[j];
        }
        sm[c][0][i] = C;
        sm[c][3][i] = P;
        __syncwarp();
        double Ry = 0.0;
#pragma unroll
        for (int k = 0; k < NA; ++k) Ry = __dadd_rn(Ry, sv[c][k][i]);
        sm[c][1][i] = Ry;
        sm[c][2][i] = __dadd_rn(C, Ry);
        __syncwarp();
        // lane r sums moment r over the nodes: rho - rho0, rho u_x, rho u_y, sum |xi|^2 d, Pi_xy
        double s = 0.0, pxy = 0.0;
#pragma unroll
        for (int k = 0; k < NA; ++k) {
            s = fma(role[k], sm[c][role_sum][k], s);
            if (ROLES == 4) pxy = fma(t.a[k], sm[c][3][k], pxy);
        }
        const double drho = __shfl_sync(0xffffffffu, s, c * NA), jx = __shfl_sync(0xffffffffu, s, c * NA + 1),
                     jy = __shfl_sync(0xffffffffu, s, c * NA + 2), en = __shfl_sync(0xffffffffu, s, c * NA + 3);
        if (ROLES == 5) pxy = __shfl_sync(0xffffffffu, s, (c * NA + 4) & 31);
        CellOut<double> o;
        double cx[N + 1], cy[N + 1];
        const double gf = forced ? gt * sx : 0.0;
        const double rho = cell_state<N, double, double, true>(A.rho0, A.sigma_fac, A.isothermal, forced, gf, A.tau, A.hdt,
                                                               drho, jx, jy, en, pxy, o, cx, cy);
        sq[c][i][0] = wmi;
#pragma unroll
        for (int k = 1; k <= N; ++k) sq[c][i][k] = __dmul_rn(whn[k], cy[k]);
        double PX[N + 1];
        const double owr = __dmul_rn(ow, rho);
#pragma unroll
        for (int ky = 0; ky <= N; ++ky) {
            double px = ky == 0 ? 0.0 : 1.0;
#pragma unroll
            for (int kx = 1; kx <= N - ky; ++kx) px = fma(cx[kx], hn[kx], px);
            PX[ky] = ky == 0 ? __dmul_rn(ow, fma(rho, px, drho)) : __dmul_rn(owr, px);
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < NA; ++j) {
            double od = __dmul_rn(PX[0], sq[c][j][0]);
#pragma unroll
            for (int ky = 1; ky <= N; ++ky) od = fma(PX[ky], sq[c][j][ky], od);
            f[j] = fma(f[j], om1, od);
        }
        if (own) {
            double* const base = dst + (long long)(i * NA) * A.plane + A.origin;
            auto put = [&](int xi, int yi) {
                double* p = base + (long long)yi * A.pitch + xi;
#pragma unroll
                for (int j = 0; j < NA; ++j) p[j * A.plane] = f[j];
            };
            put(x, y);
            if (has_images<double, 1>(A, x, y)) for_images<double, 1>(A, x, y, put);
        }
        if (diag) {
            const bool one = own && i == 0;
            acc[0] += one ? o.drho : 0.0;
            acc[1] += one ? o.jx : 0.0;
            acc[2] += one ? o.jy : 0.0;
            acc[3] = fma(one ? o.uy : 0.0, sx, acc[3]);
            acc[4] = fma(one ? o.sig : 0.0, cxs, acc[4]);
            acc[5] = fma(winvi, own ? h : 0.0, acc[5]);
        }
        __syncwarp();  // the shared arrays are reused by the next tile
    }
    if (diag) {
        const double v = warp_sum6(acc, lane);
        const int q = sum6_index(lane);
        if (q >= 0) partials_of(A, A.level_add & 1)[((long long)blockIdx.x * W + warp) * kDiagSlots + q] = v;
    }
    close_level(A, lvl, diag);
}

// ------------------------------------------------------------ TMA-staged step kernel
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// try_wait with a suspend-time hint (ns): the waiting thread is suspended in hardware
// until the phase completes or the hint runs out, instead of spinning on issue slots
__device__ __forceinline__ bool mbar_try_wait_sleep(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        " .reg .pred p;\n"
        " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
        " selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(20000u)
        : "memory");
    return ok != 0;
}

// try_wait with the default (system-dependent) suspend window: the consumers' fast path
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n"
        " .reg .pred p;\n"
        " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n"
        "}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait for the phase of the given parity: gives up after ~2^31 cycles
// (about a second), flags LB_ERR_TIMEOUT in the status word and returns false.
static __device__ __noinline__ bool mbar_wait_slow(uint64_t* bar, uint32_t parity, int* status) {
    const long long t0 = clock64();
    for (uint32_t i = 0;; ++i) {
        if (mbar_try_wait_sleep(bar, parity)) return true;
        if ((i & 255u) == 255u && clock64() - t0 > (1LL << 31)) {
            atomicOr(status, 2);
            return false;
        }
    }
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int* status) {
    if (mbar_try_wait(bar, parity)) return true;
    return mbar_wait_slow(bar, parity, status);
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1,
                                            int c2) {
    if constexpr (LB_TMA_EVICT_LAST) {
        // the halo rows and columns of a box are read again by the neighbouring tiles:
        // ask L2 to keep the lines (evict-last) so those re-reads do not go to DRAM
        uint64_t pol;
        asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol));
        asm volatile(
            "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint "
            "[%0], [%1, {%3, %4, %5}], [%2], %6;" ::"r"(smem_u32(dst)),
            "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "l"(pol)
            : "memory");
    } else {
        asm volatile(
            "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], "
            "[%2];" ::"r"(smem_u32(dst)),
            "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2)
            : "memory");
    }
}

// Store-staged kernel: the warp's output slot to the cells (x.., y) of dst, all planes, with one TMA
// tensor store (the tensor map clips it at nx).  One lane calls it, once the warp's writes to the slot
// have been made visible to the async proxy.
__device__ __forceinline__ void store_strip(const Args<float>& A, const void* slot, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(
            reinterpret_cast<uint64_t>(&A.tmap_st)),
        "r"(smem_u32(slot)), "r"(x), "r"(y), "r"(0)
        : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// KIND = kStep: one level (store f*, diagnostics, level advance); kMoments: the per-cell
// moments (and optionally f~) of the current level, nothing stored, no level advance.
// WIDE (KIND = kStep only): the store-staged variant (see TmaCfg): consumer warp w owns half
// w % 2 of tile row w / 2, and stores it from a shared-memory slot of its own.
template <class VS, int N, class S, bool UPW = false, int KIND = kStep, bool WIDE = false>
__global__ void __maxnreg__((TmaCfg<VS, S, UPW, WIDE>::MAXREG))
    lb_tma_step_kernel(const __grid_constant__ Args<float> A) {
    static_assert(KIND == kStep || KIND == kMoments, "TMA-staged kinds: step, moments");
    static_assert(!WIDE || KIND == kStep, "the store-staged kernel is a step kernel");
    using R = float;
    using C = TmaCfg<VS, S, UPW, WIDE>;
    constexpr int Q = VS::Q, V = C::V, ROWS = C::ROWS, CW = C::CW, TW = C::TW, AL = C::AL;
    constexpr int NS = C::NS, NG = C::NG, K = C::K, BW = C::BW, BOX = C::BOX, SLOT = C::SLOT;
    using E = typename C::E;
    constexpr int STAGE_ELEMS = C::STAGE_BYTES / C::EB, KE = C::KE;
    constexpr int OSTRIDE = WIDE ? C::WCELLS : 0;  // output slot: elements per plane
    extern __shared__ __align__(128) unsigned char smem_dyn[];
    // TMA destinations must be 128-byte aligned: align the base explicitly
    unsigned char* const smem_raw =
        smem_dyn + ((128u - (smem_u32(smem_dyn) & 127u)) & 127u);
    E* const stages = reinterpret_cast<E*>(smem_raw);
    unsigned char* const slots = smem_raw + NS * C::STAGE_BYTES;  // store-staged: the warps' output slots
    uint64_t* const full = reinterpret_cast<uint64_t*>(smem_raw + NS * C::STAGE_BYTES + C::OUT_BYTES);
    uint64_t* const empty = full + NS;
    __shared__ int s_abort;

    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x == 0) {
        for (int s = 0; s < NS; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], CW);
        }
        s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();

    if constexpr (KIND == kStep) await_previous_step();
    const long long lvl = __ldcg(A.level) + A.level_add;
    const bool diag = KIND == kStep && (A.diag_every > 0) && (lvl % A.diag_every == 0);
    R acc[6] = {0, 0, 0, 0, 0, 0};
    __shared__ double wsum[CW][6];
    if (lane == 0 && warp < CW) {
#pragma unroll
        for (int i = 0; i < 6; ++i) wsum[warp][i] = 0.0;
    }
    volatile int* abort_flag = &s_abort;

    if (warp == CW) {
        // ---------------- producer: one thread streams the boxes of every tile
        if (lane == 0) {
            uint32_t it = 0;
            for (int tile = blockIdx.x; tile < A.ntiles && !*abort_flag; tile += gridDim.x) {
                int ty, tx;
                tma_tile_coords<C::BAND>(tile, A.ntiles_x, A.ntiles, ty, tx);
                // store-staged tiles are not shifted: the store clips the last one at nx
                const int x0 = (!WIDE && tx == A.ntiles_x - 1) ? A.x0_last : tx * C::TWO;
                const int y0 = ty * ROWS;
                for (int grp = 0; grp < NG; ++grp, ++it) {
                    const int s = (int)(it % NS);
                    if (it >= (uint32_t)NS && !mbar_wait(&empty[s], ((it / NS) + 1) & 1u, A.status)) {
                        *abort_flag = 1;
                        break;
                    }
                    // failure-detection test: block 0 withholds the first stage of its first tile,
                    // so its consumers' bounded waits run out (status bit 2, LB_ERR_TIMEOUT)
                    if (A.withhold_stage && blockIdx.x == 0 && tile == (int)blockIdx.x && grp == 0) continue;
                    const int a0 = grp * K;
                    const int na = (Q - a0) < K ? (Q - a0) : K;
                    E* dstage = stages + (long long)s * STAGE_ELEMS;
                    if constexpr (C::LW) {
                        mbar_arrive_expect_tx(&full[s], (uint32_t)(KE * BOX * C::EB));
                        const int xs = WIDE ? x0 - AL + kGhostX : ((x0 - C::GX + kGhostX) / AL) * AL;
                        tma_load_3d(dstage, &A.tmap, &full[s], xs, y0 - C::GX + A.gy, grp * KE);
                    } else {
                        mbar_arrive_expect_tx(&full[s], (uint32_t)(na * BOX * C::EB));
                        for (int j = 0; j < na; ++j) {
                            const int a = a0 + j;
                            const int xs = ((x0 - VS::ex(a) + kGhostX) / AL) * AL;
                            tma_load_3d(dstage + j * SLOT, &A.tmap, &full[s], xs, y0 - VS::ey(a) + A.gy, a);
                        }
                    }
                }
            }
            // drain: no box may still be in flight when the block exits
            if (*abort_flag) {
                const uint32_t first = it > (uint32_t)NS ? it - NS : 0u;
                for (uint32_t k = first; k < it; ++k) mbar_wait(&full[k % NS], (k / NS) & 1u, A.status);
            }
        }
    } else {
        // ---------------- consumers: warp w owns row y0 + w of every tile
        // stage index and parity advance with the stream of groups (NG per tile)
        int st_i = 0;
        uint32_t st_ph = 0;
        // store-staged: the warp's row of the tile and its half of the row
        const int trow = WIDE ? warp / C::WPR : warp;
        const int half = WIDE ? warp % C::WPR : 0;
        uint32_t ti = 0;  // tiles processed
        for (int tile = blockIdx.x; tile < A.ntiles; tile += gridDim.x, ++ti) {
            int ty, tx;
            tma_tile_coords<C::BAND>(tile, A.ntiles_x, A.ntiles, ty, tx);
            const int tile_start = tx * C::TWO + half * C::WCELLS;
            const int x0 = (!WIDE && tx == A.ntiles_x - 1) ? A.x0_last : tile_start;
            const int y = ty * ROWS + trow;
            const Lane g = UPW      ? upwind_lane_geometry(lane, x0, tile_start, A.nx)
                           : C::HALO ? halo_lane_geometry(lane, x0, tile_start, A.nx, C::WCELLS)
                                     : lane_geometry<V>(lane, x0, tile_start, A.nx);
            using T = typename Pack<R, V>::T;
            T ft[Q];
            bool ok = !*abort_flag;
            // Lax-Wendroff: the lane's column in the box row (column x0 - 1 for lane 0; store-staged: the
            // box starts AL columns left of the tile row)
            const int r_lw = WIDE ? AL - 1 + half * C::WCELLS : (x0 - 1 + kGhostX) & (AL - 1);
            const int c_lw = r_lw + lane;
            static_for<0, NG>([&](auto gc) {
                constexpr int grp = decltype(gc)::value;
                if (ok) {
                    ok = mbar_wait(&full[st_i], st_ph, A.status);
                    if (!ok) *abort_flag = 1;
                }
                if (ok) {
                    const E* st = stages + (long long)st_i * STAGE_ELEMS;
                    if constexpr (C::LW) {
                        static_for<0, KE>([&](auto jc) {
                            constexpr int j = decltype(jc)::value;
                            constexpr int a = grp * K + 2 * j;
                            if constexpr (a < Q) {
                                // the pair (a, a + 1); the stencil is linear: 16-bit values are scaled
                                // once, after it
                                const E* box = st + j * SLOT;
                                f2 v;
                                if constexpr (UPW) {
                                    // second-order upwind: y pass over the lane's column in the cell's
                                    // row and its two upstream rows (box row of row y: trow + 2), x pass
                                    // from the two upstream lanes (the same operation order as the
                                    // plain-load kernel, so the two give the same bits); the y nodes of a
                                    // pair may lie on either side of 0
                                    constexpr int ix = VS::ix(a), iy = VS::iy(a);
                                    constexpr int sx = VS::axis_sign(ix), sa = VS::axis_sign(iy), sb = VS::axis_sign(iy + 1);
                                    const int c = ((x0 - 2 + kGhostX) & (AL - 1)) + lane;
                                    const E* r0 = box + (trow + 2) * BW + c;
                                    auto upstream = [&](int k) {
                                        if constexpr (sa == sb) {
                                            return ld_pair<S>(r0 - k * sa * BW);
                                        } else {
                                            return f2{reinterpret_cast<const float*>(r0 - k * sa * BW)[0],
                                                      reinterpret_cast<const float*>(r0 - k * sb * BW)[1]};
                                        }
                                    };
                                    auto uw = [&](int k) { return f2{A.tab.uw[iy][k], A.tab.uw[iy + 1][k]}; };
                                    const f2 gv = vfma(uw(0), upstream(2), vfma(uw(1), upstream(1), vmul(uw(2), ld_pair<S>(r0))));
                                    const f2 g1 = sx > 0 ? shfl_up2(gv) : shfl_down2(gv);
                                    f2 g2;
                                    if constexpr (sx > 0) {
                                        g2 = f2{__shfl_up_sync(0xffffffffu, gv.x, 2), __shfl_up_sync(0xffffffffu, gv.y, 2)};
                                    } else {
                                        g2 = f2{__shfl_down_sync(0xffffffffu, gv.x, 2), __shfl_down_sync(0xffffffffu, gv.y, 2)};
                                    }
                                    v = vfma(vsplat<f2>(A.tab.uw[ix][0]), g2,
                                             vfma(vsplat<f2>(A.tab.uw[ix][1]), g1, vmul(vsplat<f2>(A.tab.uw[ix][2]), gv)));
                                } else {
                                    auto column = [&](int c) {
                                        const E* rm = box + trow * BW + c;  // row y - 1
                                        return lw_y_pair<VS, a>(A.tab, ld_pair<S>(rm), ld_pair<S>(rm + BW),
                                                                ld_pair<S>(rm + 2 * BW));
                                    };
                                    const f2 gv = column(c_lw), gl = shfl_up2(gv), gr = shfl_down2(gv);
                                    v = lw_x_pair<VS, a>(A.tab, gl, gv, gr);
                                }
                                if constexpr (Is16<S>::value)
                                    v = vmul(v, f2{load_scale<S, R>(A.tab, a), load_scale<S, R>(A.tab, a + 1)});
                                ft[a] = v.x;
                                ft[a + 1] = v.y;
                            }
                        });
                    } else {
                        static_for<0, K>([&](auto jc) {
                            constexpr int j = decltype(jc)::value;
                            constexpr int a = grp * K + j;
                            if constexpr (a < Q) {
                                constexpr int ex = VS::ex(a);
                                const int r = (x0 - ex + kGhostX) & (AL - 1);
                                const S* p = reinterpret_cast<const S*>(st + j * SLOT) + trow * BW + r + lane * V;
                                if constexpr (V == 2 && ex % 2 != 0) {
                                    ft[a] = pack_lanes<T, R>(p[0], p[1]);
                                } else {
                                    ft[a] = ld_cells<T>(p);
                                }
                            }
                        });
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&empty[st_i]);
                }
                if (++st_i == NS) {
                    st_i = 0;
                    st_ph ^= 1u;
                }
            });
            if constexpr (WIDE) {
                unsigned char* const slot = slots + warp * C::OUT_SLOT;
                const bool stores = __all_sync(0xffffffffu, ok) && y < A.ny && tile_start < A.nx;  // warp-uniform
                if (stores) {
                    // the slot is free once the warp's store before has read it
                    if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                    __syncwarp();
                    collide_store<VS, N, S, R, V, KIND, typename Pack<R, V>::T, OSTRIDE>(
                        A, ft, static_cast<S*>(A.dst), y, g, diag, acc, lane, lvl, R(0),
                        reinterpret_cast<E*>(slot) + (g.x - tile_start));
                    // the generic-proxy writes of the slot become visible to the TMA store
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                    __syncwarp();
                    if (lane == 0) store_strip(A, slot, tile_start, y);
                }
            } else {
                if (ok && y < A.ny)
                    collide_store<VS, N, S, R, V, KIND>(A, ft, static_cast<S*>(A.dst), y, g, diag, acc, lane, lvl,
                                                        R(0));
            }
            if (diag && (ti % kDiagFold) == kDiagFold - 1) fold_diag(acc, wsum[warp], lane);  // warp-uniform
            if (!ok) break;
        }
        if constexpr (WIDE) {  // the warp's stores have written HBM before the block exits
            if (lane == 0) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
            __syncwarp();
        }
    }
    __syncthreads();
    if constexpr (KIND == kStep) finish_step<R, CW>(A, acc, wsum, lvl, diag, warp, lane);
}

// ------------------------------------------------------------ init kernel
// f~(0) = f^eq(rho, u, T) per cell (raw layout, no streaming), written to dst with its images.
template <class VS, int N, class S, class R>
__global__ void __launch_bounds__(256) lb_init_kernel(const __grid_constant__ Args<R> A) {
    S* __restrict__ dst = static_cast<S*>(A.dst);
    const long long ncell = (long long)A.nx * A.ny;
    for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < ncell;
         c += (long long)gridDim.x * blockDim.x) {
        const int y = (int)(c / A.nx), x = (int)(c - (long long)y * A.nx);
        double rho = 1.0, ux = 0.0, uy, T = 1.0;
        if (A.i_uy) {
            rho = A.i_rho ? A.i_rho[c] : 1.0;
            ux = A.i_ux ? A.i_ux[c] : 0.0;
            uy = A.i_uy[c];
            T = A.i_T ? A.i_T[c] : 1.0;
        } else {
            const double sx = sinpi(2.0 * (double)x / (double)A.nx);
            const double sy = sinpi(2.0 * (double)y / (double)A.ny);
            uy = A.u0 * sx + A.u1 * sy * sx;
        }
        const R drho = (R)(rho - (double)A.rho0);
        const R th = A.isothermal ? R(0) : (R)(T - 1.0);
        equilibrium_dev<VS, N, R>(A.tab, drho, (R)rho, (R)ux, (R)uy, th, [&](auto ac, R deq) {
            constexpr int a = decltype(ac)::value;
            store_cell<VS, S, R>(A, dst, a, x, y, deq, store_scale<S, R>(A.tab, a));
        });
    }
}

// ------------------------------------------------------------ dispatch
// A step launch; `follows` makes it a programmatic dependent of the launch before it.
template <class R>
cudaError_t launch_step(void (*kernel)(const Args<R>), const Launch& L, int threads, int smem) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)L.grid);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = L.stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = L.follows ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, *static_cast<const Args<R>*>(L.args));
}

template <class VS, int N, class S, class R>
cudaError_t launch_typed(const Launch& L) {
    using C = Cfg<VS, S>;
    using T = TmaCfg<VS, S>;
    constexpr bool kTma = std::is_same<R, float>::value && T::NS >= 2;
    // second-order upwind streaming: Lax-Wendroff sets with 32/64-bit storage; TMA-staged
    // for FP32 storage
    constexpr bool kUpw = !VS::kOnLattice && !Is16<S>::value;
    constexpr bool kUpwTma = kUpw && kTma && std::is_same<S, float>::value;
    // store-staged TMA kernel: Lax-Wendroff sets, FP32 up to 36 velocities (the FP32 output
    // tile of a 64-velocity set leaves too little shared memory for the ring), 16-bit all
    constexpr bool kStore = kTma && !VS::kOnLattice && ((std::is_same<S, float>::value && VS::Q <= 40) || Is16<S>::value);
    // node-split FP64 steps of small grids
    constexpr bool kSplit = std::is_same<S, double>::value && !VS::kOnLattice;
    if (L.kind == kQueryShape) {
        Shape* sh = static_cast<Shape*>(const_cast<void*>(L.args));
        sh->vw = Layout<VS, S>::VW;
        sh->V = C::V;
        sh->tw = L.upwind ? 32 * C::V : C::TW;
        sh->rows = C::ROWS;
        sh->threads = C::THREADS;
        cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &sh->occupancy, lb_fused_kernel<VS, N, S, R, kStep>, C::THREADS, 0);
        if (e != cudaSuccess) return e;
        sh->tma = 0;
        sh->split_cells = 0;
        if constexpr (kSplit) {
            if (!L.upwind) {
                sh->split_cells = SplitCfg<VS>::CELLS;
                sh->split_ops = SplitCfg<VS>::OPS;
                sh->plain_ops = SplitCfg<VS>::PLAIN_OPS;
            }
        }
        // the TMA-staged kernel of the requested streaming, and its box
        auto tma_shape = [&](auto kernel, auto cfg) -> cudaError_t {
            using TC = decltype(cfg);
            cudaError_t r = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 TC::SMEM);  // fixed per kernel: every handle asks the same
            if (r != cudaSuccess) return r;
            r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&sh->tma_occupancy, kernel, TC::THREADS, TC::SMEM);
            if (r != cudaSuccess) return r;
            sh->tma = sh->tma_occupancy > 0 ? 1 : 0;
            sh->tma_V = TC::V;
            sh->tma_tw = TC::TWO;
            sh->tma_rows = TC::ROWS;
            sh->tma_threads = TC::THREADS;
            sh->tma_smem = TC::SMEM;
            sh->box_w = TC::BW;
            sh->box_h = TC::BH;
            sh->box_d = TC::BOX_D;
            return cudaSuccess;
        };
        if (L.upwind) {
            if constexpr (kUpwTma) {
                e = tma_shape(lb_tma_step_kernel<VS, N, S, true>, TmaCfg<VS, S, true>{});
                if (e == cudaSuccess)
                    e = cudaFuncSetAttribute(lb_tma_step_kernel<VS, N, S, true, kMoments>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, TmaCfg<VS, S, true>::SMEM);
            }
        } else {
            if constexpr (kTma) {
                e = tma_shape(lb_tma_step_kernel<VS, N, S>, T{});
                if (e == cudaSuccess)
                    e = cudaFuncSetAttribute(lb_tma_step_kernel<VS, N, S, false, kMoments>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, T::SMEM);
            }
            sh->st = 0;
            if constexpr (kStore) {
                using TS = TmaCfg<VS, S, false, true>;
                auto kernel = lb_tma_step_kernel<VS, N, S, false, kStep, true>;
                if (e == cudaSuccess)
                    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, TS::SMEM);
                if (e == cudaSuccess)
                    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&sh->st_occupancy, kernel, TS::THREADS, TS::SMEM);
                if (e == cudaSuccess) {
                    sh->st = sh->st_occupancy > 0 ? 1 : 0;
                    sh->st_tw = TS::TWO;
                    sh->st_cells = TS::WCELLS;
                    sh->st_rows = TS::ROWS;
                    sh->st_threads = TS::THREADS;
                    sh->st_smem = TS::SMEM;
                    sh->st_box_w = TS::BW;
                    sh->st_box_h = TS::BH;
                    sh->st_box_d = TS::BOX_D;
                    // D2Q16-GH and the 16-bit sets are faster with plain stores (4096^2, us a level, plain /
                    // store-staged: D2Q16-GH FP32 364 / 421, D2Q36-GH FP16 811 / 947), D2Q36-GH FP32 with
                    // staged ones (788 at 4094 x 4096 / 751)
                    sh->st_auto = (sizeof(S) == 4 && VS::Q > 16) ? 1 : 0;
                }
            }
        }
        return e;
    }
    const Args<R>& A = *static_cast<const Args<R>*>(L.args);
    if (L.upwind && (L.kind == kStepTma || L.kind == kMomentsTma)) {
        if constexpr (kUpwTma) {
            using TU = TmaCfg<VS, S, true>;
            if (L.kind == kStepTma) return launch_step<R>(lb_tma_step_kernel<VS, N, S, true>, L, TU::THREADS, TU::SMEM);
            lb_tma_step_kernel<VS, N, S, true, kMoments><<<L.grid, TU::THREADS, TU::SMEM, L.stream>>>(A);
            return cudaGetLastError();
        }
        return cudaErrorNotSupported;
    }
    if (L.upwind) {
        if constexpr (kUpw) {
            switch (L.kind) {
                case kStep:
                    return launch_step<R>(lb_fused_kernel<VS, N, S, R, kStep, true>, L, C::THREADS, 0);
                case kStepForced:
                    return launch_step<R>(lb_fused_kernel<VS, N, S, R, kStepForced, true>, L, C::THREADS, 0);
                case kMoments:
                    lb_fused_kernel<VS, N, S, R, kMoments, true><<<L.grid, C::THREADS, 0, L.stream>>>(A);
                    return cudaGetLastError();
                case kInit:
                    break;  // no streaming
                default:
                    return cudaErrorNotSupported;
            }
        } else {
            return cudaErrorNotSupported;
        }
    }
    switch (L.kind) {
        case kStep:
            return launch_step<R>(lb_fused_kernel<VS, N, S, R, kStep>, L, C::THREADS, 0);
        case kStepForced:
            return launch_step<R>(lb_fused_kernel<VS, N, S, R, kStepForced>, L, C::THREADS, 0);
        case kMoments:
            lb_fused_kernel<VS, N, S, R, kMoments><<<L.grid, C::THREADS, 0, L.stream>>>(A);
            break;
        case kInit:
            lb_init_kernel<VS, N, S, R><<<L.grid, 256, 0, L.stream>>>(A);
            break;
        case kStepTma:
            if constexpr (kTma) return launch_step<R>(lb_tma_step_kernel<VS, N, S>, L, T::THREADS, T::SMEM);
            return cudaErrorNotSupported;
        case kStepSplit:
        case kStepSplitForced:
            if constexpr (kSplit)
                return launch_step<R>(L.kind == kStepSplit ? (L.warps == 1 ? lb_split_kernel<VS, N, kStep, 1>
                                                                           : lb_split_kernel<VS, N, kStep, kSplitWarps>)
                                                           : (L.warps == 1 ? lb_split_kernel<VS, N, kStepForced, 1>
                                                                           : lb_split_kernel<VS, N, kStepForced, kSplitWarps>),
                                      L, 32 * L.warps, 0);
            return cudaErrorNotSupported;
        case kMomentsTma:
            if constexpr (kTma) {
                lb_tma_step_kernel<VS, N, S, false, kMoments><<<L.grid, T::THREADS, T::SMEM, L.stream>>>(A);
                break;
            }
            return cudaErrorNotSupported;
        case kStepTmaStore:
            if constexpr (kStore) {
                using TS = TmaCfg<VS, S, false, true>;
                return launch_step<R>(lb_tma_step_kernel<VS, N, S, false, kStep, true>, L, TS::THREADS, TS::SMEM);
            }
            return cudaErrorNotSupported;
        default:
            return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

// Entry point of one (velocity set, storage) translation unit.
template <class VS, class S, class R>
cudaError_t launch_order(const Launch& L) {
    switch (L.n_eq) {
        case 1: return launch_typed<VS, 1, S, R>(L);
        case 2: return launch_typed<VS, 2, S, R>(L);
        case 3: return launch_typed<VS, 3, S, R>(L);
        case 4: return launch_typed<VS, 4, S, R>(L);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace lbk
