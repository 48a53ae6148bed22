// Discrete velocity method (DVM) for the linearised BGK equation of the standing
// shear wave, in the reduced form of Sec. 3.3 (Eqs. LBGK, ga, gb): the unknown
// G(x, xi_k, t) at the nodes xi_k of an n-point Gauss-Hermite rule obeys
// dG/dt + xi_k dG/dx = (u - G) / tau + g with u = sum_k w_k G_k and the body force
// g(x, t) = A_f sin(x_i) cos(phi t) (0 for the free wave).  The other reduced function
// (Eq. ga) is homogeneous, starts at zero and stays zero, so the force term of Eq. gb,
// g (G_a + 1), is g itself.
//
// Space-time discretisation (independent of the lattice; the paper solves the DVM with
// Lax-Wendroff): Strang splitting of the relaxation and force, integrated exactly (u gains
// int g dt since sum w_k = 1; G - u decays by exp(-h / tau)), around one Lax-Wendroff
// advection step; dt = cfl dx / max|xi_k|.
// Observables per level: A = 2/nx sum u sin(x_i), S = 2/nx sum sigma cos(x_i),
// sigma = sum_k w_k xi_k G.
//
// A cluster of up to 8 CTAs advances one instance (one collision time) through all its levels with
// its state in shared memory (FP64); instances run in parallel.  The card does two FP64 operations
// a clock and SM, so a level of one instance is bound by FP64 issue on the SMs that share it: the
// grid columns are split over the CTAs of the cluster (one column of halo on either side, written
// by the neighbour through distributed shared memory, one cluster barrier a level), and the
// arithmetic of a level is brought down to seven operations a value:
//   the second half relaxation of a level and the first of the next are one, since u does not
//   change in a relaxation: with G' the advected state, u' = sum_k w_k G'_k, d = exp(-dt / 2 tau),
//     u_{s+1} = u' + c2 sin x,  sigma_{s+1} = d sum_k w_k xi_k G'_k  (sum_k w_k xi_k = 0),
//     P_{s+1} = u_{s+1} + c1 sin x + (G' - u') d^2   (c1, c2: the force over the half levels),
//   and P is the state that is kept and advected.
// A warp of its own sums the records and takes the force integrals (FP64 sine), 32 levels at a time.
// Measured (us a level): seven instances of 20 nodes x 128 columns 2.6, against 65 with one CTA an
// instance, ~15 operations a value, sines in every level and 2 n barriers; one of them 2.4, forty 4.3.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "lb.h"
#include "lb_host.h"

namespace {

constexpr int kDvmMaxNodes = 64;
constexpr int kDvmWarps = 8;         // warps that advance the state (+ one for records and force)
constexpr int kDvmThreads = 32 * (kDvmWarps + 1);
constexpr int kDvmNodes = 8;         // nodes a lane holds at most
constexpr int kDvmMaxCluster = 8;
#ifndef LB_DVM_FILL
// lanes of a CTA that the columns fill at least, where the nodes allow: four warps, one for each of the
// SM's FP64 units (us a level of 20 nodes x 128 columns, seven instances, 64 / 128 / 256: 2.90 / 2.58 /
// 2.59)
#define LB_DVM_FILL 128
#endif
constexpr int kDvmFill = LB_DVM_FILL;
constexpr int kDvmForceLevels = 32;  // levels of force integrals taken at a time (one a lane)

struct DvmArgs {
    int nx, nv, nsteps;
    int kg, log_kg;      // lanes that share a column (a power of two), nodes k = lane % kg + kg i
    int max_cols, stride;  // columns of a CTA at most; doubles between the nodes of a state buffer
    double dx, dt, u0;
    double force_amp, force_freq;
    const double* tau;   // n_inst collision times
    double* amp;         // n_inst x (nsteps + 1)
    double* shear;
    double* part;        // clusters of two and more: n_inst x cluster x (nsteps + 1) x 2, the records'
                         // sums over a CTA's columns
    double xi[kDvmMaxNodes], w[kDvmMaxNodes];
};

// A_f int_{t0}^{t0 + h} cos(phi t) dt
__device__ double force_integral(const DvmArgs& A, double t0, double h) {
    if (A.force_amp == 0.0) return 0.0;
    if (A.force_freq == 0.0) return A.force_amp * h;
    return A.force_amp * (sin(A.force_freq * (t0 + h)) - sin(A.force_freq * t0)) / A.force_freq;
}

// first column and number of columns of CTA r of a cluster of c
__host__ __device__ inline int dvm_first(int nx, int c, int r) { return (int)((long long)nx * r / c); }

// doubles of a CTA's shared memory: two state buffers, sin and cos, two buffers of u and sigma,
// two of force integrals
__host__ __device__ inline size_t dvm_smem_doubles(int nv, int stride, int max_cols) {
    return 2 * (size_t)nv * stride + 6 * (size_t)max_cols + 4 * kDvmForceLevels;
}

__global__ void __launch_bounds__(kDvmThreads) lb_dvm_kernel(const __grid_constant__ DvmArgs A) {
    namespace cg = cooperative_groups;
    extern __shared__ double sm[];
    cg::cluster_group cluster = cg::this_cluster();
    const int nc = (int)cluster.num_blocks(), rank = (int)cluster.block_rank(), inst = blockIdx.x / nc;
    const int x0 = dvm_first(A.nx, nc, rank), cols = dvm_first(A.nx, nc, rank + 1) - x0;
    const int nv = A.nv, stride = A.stride, mc = A.max_cols;
    // a state buffer: node k, column c at [k * stride + 1 + c], the halo columns at 0 and cols + 1
    double* const P = sm;
    double* const sn = P + 2 * (size_t)nv * stride;  // sin(x), cos(x) of the columns
    double* const cs = sn + mc;
    double* const rec = cs + mc;                     // [2][u, sigma][mc]
    double* const force = rec + 4 * mc;              // [2][c1 of the level after, c2][kDvmForceLevels]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double tau = A.tau[inst];
    const double d1 = exp(-0.5 * A.dt / tau), d2 = d1 * d1;

    for (int c = threadIdx.x; c < cols; c += blockDim.x) {
        sn[c] = sin((x0 + c) * A.dx);
        cs[c] = cos((x0 + c) * A.dx);
        // equilibrium start: psi = xi_y u_y, so G = u_y(x) at every node and sigma = 0
        rec[c] = A.u0 * sn[c];
        rec[mc + c] = 0.0;
    }
    // the force over the halves of level s: c2 of its second half, c1 of the first half of s + 1
    auto fill_force = [&](int s0) {
        const int s = s0 + lane;
        double* f = force + (s0 / kDvmForceLevels % 2) * 2 * kDvmForceLevels;
        f[lane] = force_integral(A, (s + 1) * A.dt, 0.5 * A.dt);
        f[kDvmForceLevels + lane] = force_integral(A, (s + 0.5) * A.dt, 0.5 * A.dt);
    };
    if (warp == kDvmWarps) fill_force(0);
    // P_0 = u_0 + c1 sin x at every node, the halo columns with it
    const double start = A.u0 + force_integral(A, 0.0, 0.5 * A.dt);
    for (int idx = threadIdx.x; idx < nv * (cols + 2); idx += blockDim.x) {
        const int k = idx / (cols + 2), c = idx - k * (cols + 2);
        P[k * stride + c] = start * sin(((x0 + c - 1 + A.nx) % A.nx) * A.dx);
    }
    cluster.sync();

    if (warp == kDvmWarps) {
        // records of level s (u and sigma left by the compute warps) while they advance level s + 1
        for (int s = 0;; ++s) {
            const double* u = rec + (s & 1) * 2 * mc;
            double pa = 0.0, ps = 0.0;
            for (int c = lane; c < cols; c += 32) {
                pa = fma(u[c], sn[c], pa);
                ps = fma(u[mc + c], cs[c], ps);
            }
            for (int o = 16; o > 0; o >>= 1) {
                pa += __shfl_xor_sync(0xffffffffu, pa, o);
                ps += __shfl_xor_sync(0xffffffffu, ps, o);
            }
            if (lane == 0 && nc == 1) {
                A.amp[(size_t)inst * (A.nsteps + 1) + s] = 2.0 * pa / A.nx;
                A.shear[(size_t)inst * (A.nsteps + 1) + s] = 2.0 * ps / A.nx;
            } else if (lane == 0) {
                double* out = A.part + 2 * (((size_t)inst * nc + rank) * ((size_t)A.nsteps + 1) + s);
                out[0] = pa;
                out[1] = ps;
            }
            if (s == A.nsteps) break;
            // the next 32 force integrals, half of a batch ahead of their first use
            if (s % kDvmForceLevels == kDvmForceLevels / 2) fill_force(s - s % kDvmForceLevels + kDvmForceLevels);
            __syncwarp();
            cluster.sync();
        }
    } else {
        const int kg = A.kg, sub = lane & (kg - 1), cl = lane >> A.log_kg, cpw = 32 >> A.log_kg;
        // constants of the lane's nodes: Lax-Wendroff weights, w_k, w_k xi_k (0 past the last node)
        double l0[kDvmNodes], l1[kDvmNodes], l2[kDvmNodes], wk[kDvmNodes], wx[kDvmNodes];
#pragma unroll
        for (int i = 0; i < kDvmNodes; ++i) {
            const int k = sub + kg * i;
            const bool in = k < nv;
            const double xi = in ? A.xi[in ? k : 0] : 0.0, C = xi * A.dt / A.dx;
            l0[i] = 0.5 * C * (1.0 + C);
            l1[i] = 1.0 - C * C;
            l2[i] = -0.5 * C * (1.0 - C);
            wk[i] = in ? A.w[in ? k : 0] : 0.0;
            wx[i] = wk[i] * xi;
        }
        const int npt = (nv - 1) / kg + 1;  // nodes of a lane (uniform; the last may be past the end)
        double* const left = cluster.map_shared_rank(P, (rank + nc - 1) % nc);
        double* const right = cluster.map_shared_rank(P, (rank + 1) % nc);
        const int left_cols = x0 - dvm_first(A.nx, nc, (rank + nc - 1) % nc) + (rank == 0 ? A.nx : 0);
        for (int s = 0; s < A.nsteps; ++s) {
            const double* src = P + (s & 1) * (size_t)nv * stride;
            const size_t dst = ((s & 1) ^ 1) * (size_t)nv * stride;
            double* const u = rec + ((s & 1) ^ 1) * 2 * mc;
            const double* f = force + (s / kDvmForceLevels % 2) * 2 * kDvmForceLevels;
            const double c1 = f[s % kDvmForceLevels], c2 = f[kDvmForceLevels + s % kDvmForceLevels];
            for (int cb = warp * cpw; cb < cols; cb += kDvmWarps * cpw) {  // warp-uniform
                const int c = cb + cl;
                const bool own = c < cols;
                const double* p = src + sub * stride + 1 + (own ? c : cols - 1);
                double g[kDvmNodes], su = 0.0, sx = 0.0;
#pragma unroll
                for (int i = 0; i < kDvmNodes; ++i) {
                    if (i >= npt) break;
                    // a lane past the last node reads its neighbour's column with weight 0
                    const double* q = sub + kg * i < nv ? p + kg * i * stride : p;
                    g[i] = fma(l0[i], q[-1], fma(l1[i], q[0], l2[i] * q[1]));
                    su = fma(wk[i], g[i], su);
                    sx = fma(wx[i], g[i], sx);
                }
                for (int o = 1; o < kg; o <<= 1) {
                    su += __shfl_xor_sync(0xffffffffu, su, o);
                    sx += __shfl_xor_sync(0xffffffffu, sx, o);
                }
                const double un = fma(c2, sn[own ? c : 0], su), base = fma(c1, sn[own ? c : 0], un);
                if (own && sub == 0) {
                    u[c] = un;
                    u[mc + c] = d1 * sx;
                }
#pragma unroll
                for (int i = 0; i < kDvmNodes; ++i) {
                    const int k = sub + kg * i;
                    if (i >= npt || k >= nv || !own) break;
                    const double v = fma(g[i] - su, d2, base);
                    const size_t at = dst + (size_t)k * stride + 1 + c;
                    P[at] = v;
                    if (c == 0) left[dst + (size_t)k * stride + 1 + left_cols] = v;
                    if (c == cols - 1) right[dst + (size_t)k * stride] = v;
                }
            }
            __syncwarp();
            cluster.sync();
        }
    }
    // the records of all levels: the CTAs' sums in rank order, levels split over the cluster
    cluster.sync();
    if (nc == 1) return;
    for (int s = rank * blockDim.x + threadIdx.x; s <= A.nsteps; s += nc * blockDim.x) {
        double ta = 0.0, ts = 0.0;
        for (int r = 0; r < nc; ++r) {
            const double* in = A.part + 2 * (((size_t)inst * nc + r) * ((size_t)A.nsteps + 1) + s);
            ta += in[0];
            ts += in[1];
        }
        A.amp[(size_t)inst * (A.nsteps + 1) + s] = 2.0 * ta / A.nx;
        A.shear[(size_t)inst * (A.nsteps + 1) + s] = 2.0 * ts / A.nx;
    }
}

lb_status dvm_fail(lb_status s, const std::string& m) {
    lbh::set_last_error(m);
    return s;
}

}  // namespace

extern "C" {

lb_status lb_dvm_run(int n_inst, const double* tau, int n_nodes, int nx, double cfl, double u0, int nsteps,
                     double* amp, double* shear, void* stream) {
    return lb_dvm_run_forced(n_inst, tau, n_nodes, nx, cfl, u0, 0.0, 0.0, nsteps, amp, shear, stream);
}

lb_status lb_dvm_run_forced(int n_inst, const double* tau, int n_nodes, int nx, double cfl, double u0,
                            double force_amp, double force_freq, int nsteps, double* amp, double* shear,
                            void* stream) {
    if (n_inst < 1 || !tau || !amp || !shear) return dvm_fail(LB_ERR_ARG, "n_inst >= 1 and tau, amp, shear are required");
    if (n_nodes < 1 || n_nodes > kDvmMaxNodes) return dvm_fail(LB_ERR_ARG, "n_nodes must be in [1, 64]");
    if (nx < 3 || nsteps < 0 || !(cfl > 0.0 && cfl <= 1.0) || !std::isfinite(u0))
        return dvm_fail(LB_ERR_ARG, "nx >= 3, nsteps >= 0, 0 < cfl <= 1 and a finite u0 are required");
    if (!std::isfinite(force_amp) || !std::isfinite(force_freq))
        return dvm_fail(LB_ERR_ARG, "force_amp and force_freq must be finite");
    for (int i = 0; i < n_inst; ++i)
        if (!(tau[i] > 0.0) || !std::isfinite(tau[i])) return dvm_fail(LB_ERR_ARG, "collision times must be positive");
    const size_t smem = sizeof(double) * ((size_t)n_nodes * nx + 2 * (size_t)nx);
    int dev = 0, optin = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return dvm_fail(LB_ERR_CUDA, std::string("device query: ") + cudaGetErrorString(e));
    if (smem > (size_t)optin)
        return dvm_fail(LB_ERR_UNSUPPORTED, "n_nodes x nx too large for one CTA's shared memory (" +
                                                std::to_string(smem) + " > " + std::to_string(optin) + " bytes)");
    int nsm = 0;
    e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return dvm_fail(LB_ERR_CUDA, std::string("device query: ") + cudaGetErrorString(e));
    // CTAs of an instance: as many (up to 8) as the card has SMs for, of at least four columns; more
    // where the two state buffers of a CTA would not fit otherwise (they do for 8)
    DvmArgs A{};
    int nc = 1;
    auto shape = [&]() {
        A.max_cols = (nx + nc - 1) / nc;
        // lanes a column: enough for kDvmNodes nodes a lane, then up to four warps of the CTA
        A.kg = 1;
        while (A.kg * kDvmNodes < n_nodes || (A.kg < 8 && 2 * A.kg <= n_nodes && A.max_cols * A.kg < kDvmFill)) A.kg *= 2;
        for (A.log_kg = 0; (1 << A.log_kg) < A.kg;) ++A.log_kg;
        // the 16 doubles that half a warp reads lie in different banks
        A.stride = (A.max_cols + 2 + 15) / 16 * 16 + 16 / A.kg % 16;
        return sizeof(double) * dvm_smem_doubles(n_nodes, A.stride, A.max_cols);
    };
    while (nc < kDvmMaxCluster && 2LL * nc * n_inst <= nsm && nx >= 4 * 2 * nc) nc *= 2;
    size_t bytes = shape();
    while (bytes > (size_t)optin && nc < kDvmMaxCluster) {
        nc *= 2;
        bytes = shape();
    }
    std::vector<double> x, w;
    lbh::gauss_hermite(n_nodes, x, w);
    A.nx = nx;
    A.nv = n_nodes;
    A.nsteps = nsteps;
    A.dx = 2.0 * M_PI / nx;
    double vmax = 0.0;
    for (int k = 0; k < n_nodes; ++k) {
        A.xi[k] = x[k];
        A.w[k] = w[k];
        vmax = std::max(vmax, std::fabs(x[k]));
    }
    A.dt = cfl * A.dx / (vmax > 0 ? vmax : 1.0);
    A.u0 = u0;
    A.force_amp = force_amp;
    A.force_freq = force_freq;
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    const size_t rec = (size_t)n_inst * ((size_t)nsteps + 1);
    double *d_tau = nullptr, *d_out = nullptr;
    e = cudaMalloc(&d_tau, sizeof(double) * n_inst);
    if (e == cudaSuccess) {
        // records, and the CTAs' sums of them: where those do not fit, fewer CTAs an instance
        auto out_bytes = [&]() { return sizeof(double) * 2 * (1 + (nc > 1 ? (size_t)nc : 0)) * rec; };
        while ((e = cudaMalloc(&d_out, out_bytes())) == cudaErrorMemoryAllocation && nc > 1) {
            cudaGetLastError();
            nc /= 2;
            bytes = shape();
            if (bytes > (size_t)optin) break;
        }
    }
    if (e != cudaSuccess) {
        cudaFree(d_tau);
        return dvm_fail(LB_ERR_NOMEM, "DVM device buffers");
    }
    A.tau = d_tau;
    A.amp = d_out;
    A.shear = d_out + rec;
    A.part = d_out + 2 * rec;
    e = cudaMemcpyAsync(d_tau, tau, sizeof(double) * n_inst, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(lb_dvm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
    if (e == cudaSuccess) {
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3((unsigned)n_inst * nc);
        cfg.blockDim = dim3(kDvmThreads);
        cfg.dynamicSmemBytes = bytes;
        cfg.stream = s;
        cudaLaunchAttribute at{};
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = nc;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
        cfg.attrs = &at;
        cfg.numAttrs = 1;
        e = cudaLaunchKernelEx(&cfg, lb_dvm_kernel, A);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(amp, A.amp, sizeof(double) * rec, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(shear, A.shear, sizeof(double) * rec, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(d_tau);
    cudaFree(d_out);
    if (e != cudaSuccess) return dvm_fail(LB_ERR_CUDA, std::string("DVM run: ") + cudaGetErrorString(e));
    return LB_OK;
}

}  // extern "C"
