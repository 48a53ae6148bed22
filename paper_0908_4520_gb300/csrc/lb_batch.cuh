// Persistent multi-instance kernel: many small, uneven lattices in one launch.
//
// A group of warps takes instances from a work queue (an atomic counter over a list ordered by
// decreasing remaining cost, i.e. longest-processing-time first) and advances one instance at a
// time by up to `chunk` time levels, with one barrier of the group between levels.  There are four
// widths of group, each with a queue of its own: a cluster of two CTAs, a CTA, four warps of it,
// and one warp.  The host gives each instance the narrowest group that still finishes within the
// launch's mean load, so a launch is not as long as its largest instance takes on one SM and a
// small instance does not hold a whole one.  Every cluster serves the wide queue first, then its
// CTAs, then their four-warp groups, then their warps go on by themselves.  Only CTAs of one
// cluster (which run at the same time) wait on one another.
//
// An instance whose two population buffers fit the group's share of the CTA's shared memory is
// copied in once per chunk and stepped entirely on chip (groups within a CTA); larger ones step
// through global memory (L2-resident at these sizes).  A warp advances strips of up to 30 cells of
// one row: each lane streams one column in y (three loads per velocity) and takes its neighbours'
// columns by shuffles for the x pass, the two edge lanes streaming the columns beside the strip, as
// the single-lattice kernels do; a row of at most 32 cells is one strip whose lanes are neighbours
// around the end.  The per-cell arithmetic is the velocity-pair stencil and collide_cell_pairs() of
// those kernels.
//
// The sums of a level (A, S, H) are taken over 64 slots: strip s belongs to slot s % 64, a slot to
// one warp, which sums its strips in order in FP32; after the level's barrier every warp finds out
// for itself whether the instance has stopped, and the last one adds the slots in a fixed order, with
// what each addition rounds off (Sum2): the history is rounded to FP32 once.  Neither a cell's
// operations nor the sums' order depend on the group or the memory path, so an instance's
// populations and history are bitwise the same whichever path runs it and whatever else shares the
// launch.  Lax-Wendroff streaming only: the batch serves the Gauss-Hermite product sets.
//
// Bound: latency of the L2 loads and of the collision's chain; 16 warps of 128 registers per SM beat
// 8 of 255, the tables are constant-bank operands (the kernel inlines its nine variants; through a
// reference they were loads), and the two wide queues take the makespan of the largest instances
// down to the mean load.  512 instances of the batching configuration, 800 levels, admission and
// histories included: 169 ms before, 72 ms, 66 ms with the populations in pairs.
#pragma once

#include "lb_batch.h"
#include "lb_kernels.cuh"

namespace lbk {

constexpr int kBatchMaxWarps = 16;  // warps per CTA (the kernel's launch bound: 512 threads of 128 registers)
constexpr int kStrip = 30;  // cells of a row per warp and pass (two lanes stream the columns beside them)
constexpr int kBatchSlots = 64;     // partial sums of a level

// the kernel's static shared memory; what belongs to a group lies at the index of its first warp
struct BatchShared {
    float red[kBatchMaxWarps][3][kBatchSlots];     // A, S, H by slot: of two levels in turn (one warp: of one)
    float relax[kBatchMaxWarps][4][kMaxNA];        // relaxation tables of the group's instance
    int next[kBatchMaxWarps];                      // queue position of the group's instance
};

// The warps that advance one instance together.
struct BatchGroup {
    int kind;        // BatchQueue: cluster, CTA, four warps, warp
    int warps;       // warps of the group, in all its CTAs
    int wid;         // this warp's number among them
    int first;       // first warp of the group in this CTA
    int threads;     // threads of the group in this CTA
    int tid;         // this thread's number among those
    int ctas;        // CTAs of the group
    int smem_cap;    // bytes of its share of the shared memory
    __device__ __forceinline__ void sync() const {
        if (kind == kBatchWarp) {
            __syncwarp();
        } else if (kind == kBatchCluster && ctas > 1) {
            __syncwarp();
            asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
        } else {
            asm volatile("bar.sync %0, %1;" ::"r"(1 + first), "r"(threads) : "memory");
        }
    }
};

// address of this CTA's shared variable in CTA r of the cluster, and a load from there
__device__ __forceinline__ uint32_t cluster_addr(const void* p, int r) {
    uint32_t d;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(d) : "r"(smem_u32(p)), "r"(r));
    return d;
}
__device__ __forceinline__ float cluster_ld(uint32_t a) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}

template <class S>
__device__ __forceinline__ float batch_load(const S* p) {
    if constexpr (std::is_same<S, __half>::value) {
        return __half2float(*p);
    } else if constexpr (std::is_same<S, __nv_bfloat16>::value) {
        return __bfloat162float(*p);
    } else {
        return *p;
    }
}

// Sums of three values over the warp in 7 shuffles: the halves of the warp, then its quarters, take
// one value each; lanes 0, 8 and 16 return the sums of a, b and c.
__device__ __forceinline__ float warp_sum3(float a, float b, float c, int lane) {
    const bool up = lane & 16;
    // lanes 0-15 keep a and b, lanes 16-31 keep c
    const float ra = __shfl_xor_sync(0xffffffffu, up ? a : c, 16);
    const float rb = __shfl_xor_sync(0xffffffffu, b, 16);
    float x = up ? c + ra : a + ra;
    float y = up ? 0.f : b + rb;
    const bool q = lane & 8;
    const float r = __shfl_xor_sync(0xffffffffu, q ? x : y, 8);
    x = q ? y + r : x + r;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// A sum of FP32 values as its FP32 rounding and what that left out: the slots' sums are exact to 2^-46
// of their terms' size.  FP64 additions, of which an SM does two a clock, cost a level of a small
// instance up to half as much again.  152 of D2Q16-GH 256 x 1, us a level: plain FP32 sums, whose
// roundings the history then has, 3.29, FP64 5.06, these in every warp 3.56, in the last warp alone, the
// others deciding by a plain sum, 2.75; 512 uneven instances 66 to 67 ms with all of them but the last, 65.
struct Sum2 {
    float hi, lo;
};
__device__ __forceinline__ Sum2 add2(Sum2 a, Sum2 b) {
    // Knuth's two-sum of the leading parts (exact); the parts left out add up
    const float s = __fadd_rn(a.hi, b.hi), t = __fsub_rn(s, a.hi);
    const float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, t)), __fsub_rn(b.hi, t));
    return {s, __fadd_rn(e, __fadd_rn(a.lo, b.lo))};
}
__device__ __forceinline__ Sum2 shfl_xor2(Sum2 v, int o) {
    return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
// the same of one more value
__device__ __forceinline__ Sum2 add1(Sum2 a, float b) {
    const float s = __fadd_rn(a.hi, b), t = __fsub_rn(s, a.hi);
    return {s, __fadd_rn(__fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, t)), __fsub_rn(b, t)), a.lo)};
}
// a b, rounded to FP32 once (a product that is not finite stays as it is)
__device__ __forceinline__ float mul2(Sum2 a, Sum2 b) {
    const float p = __fmul_rn(a.hi, b.hi);
    const float r = fmaf(a.hi, b.hi, -p) + fmaf(a.hi, b.lo, a.lo * b.hi);
    return isfinite(p) ? __fadd_rn(p, r) : p;
}
__device__ __forceinline__ Sum2 split2(double v) {
    const float hi = __double2float_rn(v);
    return {hi, __double2float_rd(v - (double)hi)};
}
// hi the FP32 rounding of the whole sum (a sum that is not finite stays as it is)
__device__ __forceinline__ Sum2 normal2(Sum2 v) {
    const float s = __fadd_rn(v.hi, v.lo);
    return isfinite(v.hi) ? Sum2{s, __fsub_rn(v.lo, __fsub_rn(s, v.hi))} : Sum2{v.hi, 0.f};
}

// Advance instance `id` by up to B.chunk levels with the group's warps (smem: the group's share of
// the CTA's shared memory).
template <class VS, int SET, int N, class S>
__device__ __forceinline__ void batch_run(const BatchArgs& B, int id, void* smem, const BatchGroup& G, BatchShared& sh) {
    constexpr int Q = VS::Q;
    BatchInst& in = B.inst[id];
    const Tab<float>& t = B.tab[SET];
    const int nx = in.nx, ny = in.ny;
    const int ncell = nx * ny;
    using E = typename PairOf<S>::E;  // the populations lie in pairs of velocities, [pair][cell]
    const long long pop = (long long)(Q / 2) * ncell;
    const float omega = in.omega, sigma_fac = in.sigma_fac;
    const int lane = threadIdx.x & 31, tid = G.tid, nthr = G.threads;
    // the instance's relaxation tables (omega W_i and the second terms of the exact FP32
    // identities) in shared memory
    float(*rt)[kMaxNA] = sh.relax[G.first];
    if (tid < VS::NA) {
        rt[0][tid] = in.ow[tid];
        rt[1][tid] = in.owlo[tid];
        rt[2][tid] = in.hn1lo[tid];
        rt[3][tid] = in.whn1lo[tid];
    }
    const float* sinx = B.trig + in.trig_off;
    const float* cosx = sinx + nx;
    float2* hist = B.hist + in.hist_off;
    // a row of at most 32 cells is one strip: its lanes are neighbours around the row's end
    const bool ring = nx <= 32;
    const int spr = ring ? 1 : (nx + kStrip - 1) / kStrip;  // strips per row
    const int nstrip = spr * ny;
    const int nslot = min(nstrip, kBatchSlots);
    const bool solo = nstrip == 1 && G.warps == 1;  // one strip, one warp: no slots to add

    const int first_level = in.level;
    int level = first_level;
    int cur = in.cur;
    const int stop = min(in.max_level, level + B.chunk - 1);
    // both buffers of an instance that fits the group's shared memory are stepped on chip
    const bool onchip = G.ctas == 1 && 2 * pop * (long long)sizeof(E) <= (long long)G.smem_cap;
    S* const arena = static_cast<S*>(B.arena);
    E* gbuf[2] = {reinterpret_cast<E*>(arena + in.off[0]), reinterpret_cast<E*>(arena + in.off[1])};
    E* buf[2] = {gbuf[0], gbuf[1]};
    if (onchip) {
        buf[0] = static_cast<E*>(smem);
        buf[1] = buf[0] + pop;
        if (level > 0)
            for (long long k = tid; k < pop; k += nthr) buf[cur][k] = gbuf[cur][k];
    }
    bool done = in.done;
    int status = 0;
    float h0 = in.h0;
    const double u0 = in.u0;
    const int isothermal = in.isothermal;
    // (what is wanted once a level is read from the descriptor there: in registers it cost the strips'
    // loop spills, D2Q64-GH FP32 N = 4 1024 x 4 44.2 for 41.7 us a level)
    // stop rule sqrt(H / H0) <= stop_ratio (none for stop_ratio = 0, also where H is 0): the largest
    // value of H that meets it, as a sum
    auto threshold = [&](float h) { return split2((double)in.stop_ratio2 * (double)h); };
    Sum2 hstop = threshold(h0);
    const Sum2 norm = split2(2.0 / (double)ncell);

    // 16-bit storage: deviation = stored * sc[a] * scale; sc (tables built with S = 1) and
    // scale are powers of two, so the load and store scales are exact inverses
    const float scale = in.scale;
    const float inv_scale = 1.0f / scale;
    G.sync();
    for (; level <= stop && !done; ++level) {
        const E* src = buf[cur];
        E* dst = buf[level == 0 ? 0 : 1 - cur];
        float(*red)[kBatchSlots] = sh.red[G.kind == kBatchWarp ? G.first : G.first + (level & 1)];
        float one = 0.f;  // A, S and H of the warp's last slot in lanes 0, 8 and 16
        for (int slot = G.wid; slot < nslot; slot += G.warps) {
            float pa = 0.f, ps = 0.f, ph = 0.f;
            // strips of up to 30 cells of one row: lanes 1..w own cells x0 .. x0 + w - 1, lanes 0
            // and w + 1 stream the columns beside the strip, so that each lane streams one column
            // in y and takes its neighbours' columns by shuffles for the x pass; lanes past w + 1
            // repeat lane w + 1's column and own nothing.  In a ring lanes 0..nx - 1 own the cells.
            for (int s = slot; s < nstrip; s += kBatchSlots) {
                const int y = s / spr, x0 = (s - y * spr) * kStrip;
                const int w = min(kStrip, nx - x0);
                int x = ring ? min(lane, nx - 1) : x0 + min(lane, w + 1) - 1;
                x = x < 0 ? x + nx : (x >= nx ? x - nx : x);
                const bool own = ring ? lane < nx : lane >= 1 && lane <= w;
                const int from_l = ring ? (lane == 0 ? nx - 1 : lane - 1) : max(lane - 1, 0);
                const int from_r = ring ? (lane >= nx - 1 ? 0 : lane + 1) : min(lane + 1, 31);
                const int c = y * nx + x;
                f2 fp[Q / 2];
                if (level == 0) {
                    // f~(0) = f^eq(rho = 1, u_y = u0 sin x, T = 1), rounded through the storage type
                    const double sx = sinpi(2.0 * (double)x / (double)nx);
                    const float uy = (float)(u0 * sx);
                    float ft[Q];
                    equilibrium_dev<VS, N, float>(t, 0.f, 1.f, 0.f, uy, 0.f, [&](auto ac, float deq) {
                        constexpr int a = decltype(ac)::value;
                        if constexpr (Is16<S>::value) {
                            S tmp;
                            st1<S, float>(&tmp, deq, t.scinv[a] * inv_scale);
                            ft[a] = batch_load<S>(&tmp) * (t.sc[a] * scale);
                        } else {
                            ft[a] = deq;
                        }
                    });
                    static_for<0, Q / 2>([&](auto mc) {
                        constexpr int m = decltype(mc)::value;
                        fp[m] = f2{ft[2 * m], ft[2 * m + 1]};
                    });
                } else {
                    const int ym = y == 0 ? ny - 1 : y - 1, yp = y + 1 == ny ? 0 : y + 1;
                    const E* p0 = src + c;
                    const E* pm = src + ym * nx + x;
                    const E* pp = src + yp * nx + x;
                    // one row: the three y taps read the same value (the branch lies outside the velocity
                    // loop, whose loads it would keep apart)
                    auto stream = [&](auto rows) {
                        static_for<0, Q / 2>([&](auto mc) {
                            constexpr int m = decltype(mc)::value, a = 2 * m;
                            auto pair = [&](const E* p) {
                                f2 v = ld_pair<S>(p);  // (plain loads: the arena or shared memory)
                                if constexpr (Is16<S>::value)
                                    v = vmul(v, f2{t.sc[a] * scale, t.sc[a + 1] * scale});
                                return v;
                            };
                            const f2 v0 = pair(p0);
                            f2 vm = v0, vp = v0;
                            if constexpr (decltype(rows)::value) {
                                vm = pair(pm);
                                vp = pair(pp);
                            }
                            p0 += ncell;
                            pm += ncell;
                            pp += ncell;
                            const f2 g = lw_y_pair<VS, a>(t, vm, v0, vp);
                            const f2 gl = f2{__shfl_sync(0xffffffffu, g.x, from_l), __shfl_sync(0xffffffffu, g.y, from_l)};
                            const f2 gr = f2{__shfl_sync(0xffffffffu, g.x, from_r), __shfl_sync(0xffffffffu, g.y, from_r)};
                            fp[m] = lw_x_pair<VS, a>(t, gl, g, gr);
                        });
                    };
                    if (ny > 1) {
                        stream(std::true_type{});
                    } else {
                        stream(std::false_type{});
                    }
                }
                const CellOut<float> co = collide_cell_pairs<VS, N, true>(
                    t, rt[0], rt[1], rt[2], rt[3], 1.f, omega, sigma_fac, isothermal, true, false, 0.f, 0.f, 0.f,
                    [&](auto mc) -> f2& { return fp[decltype(mc)::value]; });
                if (own) {
                    uint32_t r0 = 0, r1 = Is16<S>::value ? sr_seed(level, c) : 0u;
                    E* p = dst + c;
                    static_for<0, Q / 2>([&](auto mc) {
                        constexpr int m = decltype(mc)::value, a = 2 * m;
                        f2 si = f2{1.f, 1.f};
                        if constexpr (Is16<S>::value) {
                            r0 = sr_next(r1);
                            r1 = sr_next(r0);
                            si = f2{t.scinv[a] * inv_scale, t.scinv[a + 1] * inv_scale};
                        }
                        *p = to_storage_pair<S>(fp[m], si, r0, r1);
                        p += ncell;
                    });
                    pa = fma(co.uy, sinx[x], pa);
                    ps = fma(co.sig, cosx[x], ps);
                    ph += co.h;
                }
            }
            one = warp_sum3(pa, ps, ph, lane);
            if (!solo && (lane == 0 || lane == 8 || lane == 16)) red[lane >> 3][slot] = one;
        }
        G.sync();
        // Every warp finds out whether the instance has stopped, the group's last warp (none has fewer
        // strips) also writes the history.  A plain FP32 sum of H's slots, none of them negative, is
        // within 2^-21 of itself of the exact one and decides unless the threshold is nearer than twice that.
        const uint32_t at = G.ctas > 1 ? cluster_addr(&red[0][0], lane % G.ctas) : 0u;  // (slot s lies in CTA s % 2)
        auto value = [&](int k, int slot) {  // (slots past the last one are read, not used)
            const int i = k * kBatchSlots + slot;
            const float v = G.ctas > 1 ? cluster_ld(at + 4 * i) : (&red[0][0])[i];
            return slot < nslot ? v : 0.f;
        };
        const bool writes = G.wid == G.warps - 1;
        bool bad = false, near = true;
        float h = 0.f;
        if (G.warps > 1) {
            h = value(2, lane);
            bad = !isfinite(h);
            if (nslot > 32) {
                const float more = value(2, lane + 32);
                bad |= !isfinite(more);
                h += more;
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (nslot > o) h += __shfl_xor_sync(0xffffffffu, h, o);
            h = __shfl_sync(0xffffffffu, h, 0);
            bad = __any_sync(0xffffffffu, bad);
            near = !(fabsf(h - hstop.hi) > 0x1p-20f * h);
        }
        bool below = h < hstop.hi;
        if (writes || level == 0 || near) {
            // the exact sums: eight lanes each A, S and H, lane j of them slots j, j + 8, ..
            const int k = min(lane >> 3, 2), j = lane & 7;
            Sum2 tot = {solo ? one : value(k, j), 0.f};
            if (nslot > 1) {
                bool inf = k == 2 && !isfinite(tot.hi);
                auto take = [&](auto first, auto last) {
                    constexpr int I0 = decltype(first)::value, I1 = decltype(last)::value;
                    float part[I1 - I0];
#pragma unroll
                    for (int i = I0; i < I1; ++i) part[i - I0] = value(k, 8 * i + j);
#pragma unroll
                    for (int i = I0; i < I1; ++i) {
                        inf |= k == 2 && !isfinite(part[i - I0]);
                        tot = add1(tot, part[i - I0]);
                    }
                };
                if (nslot > 8) {
                    take(std::integral_constant<int, 1>{}, std::integral_constant<int, 2>{});
                    if (nslot > 16) {
                        take(std::integral_constant<int, 2>{}, std::integral_constant<int, 4>{});
                        if (nslot > 32) take(std::integral_constant<int, 4>{}, std::integral_constant<int, kBatchSlots / 8>{});
                    }
                }
                if (nslot > 4) tot = add2(tot, shfl_xor2(tot, 4));
                if (nslot > 2) tot = add2(tot, shfl_xor2(tot, 2));
                tot = normal2(add2(tot, shfl_xor2(tot, 1)));
                if (G.warps == 1) bad = __any_sync(0xffffffffu, inf);
            }
            const Sum2 H = {__shfl_sync(0xffffffffu, tot.hi, 16), __shfl_sync(0xffffffffu, tot.lo, 16)};
            if (nslot == 1) bad = !isfinite(H.hi);
            if (level == 0) {
                h0 = H.hi;
                hstop = threshold(h0);
            }
            below = H.hi < hstop.hi || (H.hi == hstop.hi && H.lo <= hstop.lo);
            if (writes && (lane == 0 || lane == 8)) reinterpret_cast<float*>(hist + level)[lane >> 3] = mul2(tot, norm);
        }
        if (bad) {
            status = 1;
            done = true;
        }
        if (G.kind == kBatchWarp) __syncwarp();  // (its next level's slots go to the same place)
        if (level > 0 && in.stop_ratio2 > 0.f && below) done = true;
        if (level == in.max_level) done = true;
        cur = (level == 0) ? 0 : 1 - cur;
    }
    if (onchip && level > first_level)
        for (long long k = tid; k < pop; k += nthr) gbuf[cur][k] = buf[cur][k];
    G.sync();  // the descriptor has been read, the shared arrays are free
    if (G.wid == 0 && lane == 0) {
        in.level = level;
        in.cur = cur;
        in.done = done;
        in.h0 = h0;
        if (status) in.status |= status;
    }
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The launch: groups from the widest to the narrowest, each taking instances from its queue until
// it is empty, then parting.
template <class S>
__global__ void __launch_bounds__(kBatchMaxWarps * 32) lb_batch_kernel(const __grid_constant__ BatchArgs B) {
    extern __shared__ __align__(16) unsigned char bsm[];
    __shared__ BatchShared sh;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    uint32_t nc, rank;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(nc));
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    // start and end of every CTA (the launch's tail: how long the last CTA runs alone)
    if (B.cta_clock && threadIdx.x == 0) B.cta_clock[2 * blockIdx.x] = global_ns();
#pragma unroll 1
    for (int kind = 0; kind < kBatchQueues; ++kind) {
        const BatchQueue& Qu = B.queue[kind];
        BatchGroup G;
        G.kind = kind;
        const int per_cta = batch_group_warps(kind, nwarp);  // warps of a group in a CTA
        if (kind == kBatchQuad && nwarp % 4 != 0) continue;  // (the host leaves that queue empty)
        G.ctas = kind == kBatchCluster ? (int)nc : 1;
        G.warps = per_cta * G.ctas;
        G.first = warp / per_cta * per_cta;
        G.wid = (warp - G.first) * G.ctas + (kind == kBatchCluster ? (int)rank : 0);
        G.threads = 32 * per_cta;
        G.tid = threadIdx.x - 32 * G.first;
        const BatchSlice slice = batch_slice(kind, G.first, B.smem_cap, nwarp);
        G.smem_cap = slice.bytes;
        void* const smem = bsm + slice.offset;
        if (!Qu.order) continue;
        const int n = *Qu.n;
        if (n == 0) continue;
        if (G.ctas > 1) G.sync();  // every CTA of the cluster runs before its shared memory is written
        for (;;) {
            if (G.wid == 0 && lane == 0) {
                const int i = atomicAdd(Qu.next, 1);
                if (G.ctas == 1) {
                    sh.next[G.first] = i;
                } else {
                    for (int r = 0; r < G.ctas; ++r)
                        asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(cluster_addr(&sh.next[G.first], r)),
                                     "r"(i)
                                     : "memory");
                }
            }
            G.sync();
            const int i = *(volatile int*)&sh.next[G.first];
            G.sync();
            if (i >= n) break;
            const int id = Qu.order[i];
            if (B.inst[id].done) continue;
            switch (B.inst[id].set * 3 + (B.inst[id].n_eq - 2)) {
                case 0: batch_run<lbvs::GH4, 0, 2, S>(B, id, smem, G, sh); break;
                case 1: batch_run<lbvs::GH4, 0, 3, S>(B, id, smem, G, sh); break;
                case 2: batch_run<lbvs::GH4, 0, 4, S>(B, id, smem, G, sh); break;
                case 3: batch_run<lbvs::GH6, 1, 2, S>(B, id, smem, G, sh); break;
                case 4: batch_run<lbvs::GH6, 1, 3, S>(B, id, smem, G, sh); break;
                case 5: batch_run<lbvs::GH6, 1, 4, S>(B, id, smem, G, sh); break;
                case 6: batch_run<lbvs::GH8, 2, 2, S>(B, id, smem, G, sh); break;
                case 7: batch_run<lbvs::GH8, 2, 3, S>(B, id, smem, G, sh); break;
                case 8: batch_run<lbvs::GH8, 2, 4, S>(B, id, smem, G, sh); break;
                default: break;
            }
        }
    }
    // a CTA of a cluster stays until the others have read its shared memory for the last time
    // (the barrier after the wide queue's last instance); the CTA's end time is that of its last warp
    __syncthreads();
    if (B.cta_clock && threadIdx.x == 0) B.cta_clock[2 * blockIdx.x + 1] = global_ns();
}

}  // namespace lbk
