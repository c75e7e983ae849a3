// Multi-step backward-Euler propagator of the drift operators in FP64 with one
// thread-block cluster per item: the global-state class of steps_kernel
// (pit_phi.cuh) for narrow batches, where a launch has fewer grids than the
// GPU has SMs.
//
// What bounds it: the FP64 unit of an SM (two lanes a clock).  One CTA per
// grid leaves all but 5 of the 152 SMs idle on the toggle switch (five grids
// of up to 16,129 nodes) and all but 7 on the oscillator (seven, up to 32,385),
// each of them 81 % busy.  Here up to 16 SMs share a grid: every CTA owns a run
// of consecutive nodes with the state, the BiCGStab vectors and the
// coefficient table in its shared memory (2,025 nodes x 90 bytes for the
// largest oscillator grid), so nothing of the step touches L2.
//
//   - Operands of the stencil carry halos of the stencil's reach on both sides.
//     The pass that writes p (or s) also stores the first and last nodes of its
//     run into the neighbours' halos through distributed shared memory; one
//     cluster barrier later the stencil reads its own memory only.
//   - Sums: per CTA in shared memory, one value per CTA stored to every CTA of
//     the cluster, one cluster barrier; one warp adds them (the same order in
//     every CTA, so all of them take the same branches) and works out the
//     scalars, since an FP64 division by every warp would hold the FP64 unit
//     for longer than the barrier that hands its result over.
//   - (rh, r) of the next iteration is summed with (r, r): three sums and five
//     cluster barriers an iteration.
//
// Measured, clusters of 16, one CTA of 512 threads a grid before: oscillator,
// 96 steps 117.7 -> 7.5 ms; toggle switch, 256 steps 114.7 -> 14.9 ms.
#include <cooperative_groups.h>

#include "pit_phi.cuh"

namespace cg = cooperative_groups;

namespace pit {

namespace {

constexpr int CL_THREADS = 256, CL_MAX = 16;

struct ClusterSums {
    double part[2][3][CL_MAX];  // per CTA of the cluster, double-buffered
    double warp[3][CL_THREADS / 32];
};
struct ClusterScalars {
    double beta, alpha, omega, rr, bb;
    int act;  // what every thread does next
};
enum { CL_GO = 0, CL_DONE = 1, CL_RESTART = 2 };

// Sums of K values over the cluster; on return warp 0 (all its lanes) of every
// CTA holds them in v.  One cluster barrier, which also completes earlier
// remote stores.
template <int K>
__device__ __forceinline__ void cluster_sum(cg::cluster_group &cl, ClusterSums &R, int &slot, double (&v)[K])
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, buf = slot & 1;
    ++slot;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const double s = warp_sum(v[k]);
        if (lane == 0) R.warp[k][w] = s;
    }
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            double s = lane < CL_THREADS / 32 ? R.warp[k][lane] : 0.0;
#pragma unroll
            for (int o = CL_THREADS / 64; o > 0; o >>= 1) s += __shfl_down_sync(PIT_FULL_MASK, s, o);
            s = __shfl_sync(PIT_FULL_MASK, s, 0);
            if (lane < (int)cl.num_blocks()) cl.map_shared_rank(&R, lane)->part[buf][k][cl.block_rank()] = s;
        }
    }
    cl.sync();
    if (w == 0) {
        const int C = (int)cl.num_blocks();
#pragma unroll
        for (int k = 0; k < K; ++k) {
            double s = lane < C ? R.part[buf][k][lane] : 0.0;
#pragma unroll
            for (int o = CL_MAX / 2; o > 0; o >>= 1) s += __shfl_down_sync(PIT_FULL_MASK, s, o);
            v[k] = __shfl_sync(PIT_FULL_MASK, s, 0);
        }
    }
}

template <int OP, int D>
__global__ void __launch_bounds__(CL_THREADS, 1) cluster_kernel(const __grid_constant__ StepArgs a, int reach)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ GridInfo GI;
    __shared__ ItemConst IC;
    __shared__ ClusterSums RS;
    __shared__ ClusterScalars SC;
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const int item = a.item0 + (int)blockIdx.x / C;
    const int g = a.order[item / a.n_batch];
    const int b = item % a.n_batch;
    if (a.active && !a.active[g]) return;  // uniform over the cluster
    for (int t = threadIdx.x; t < (int)(sizeof(GridInfo) / 4); t += blockDim.x)
        reinterpret_cast<int *>(&GI)[t] = reinterpret_cast<const int *>(a.grids + g)[t];
    __syncthreads();
    item_const(a, GI, IC);
    const int tid = threadIdx.x, nt = CL_THREADS, W = reach;
    const int n = GI.n, ch = (n + C - 1) / C;          // nodes of a CTA (the last may have fewer, or none)
    const int base = rank * ch, cnt = max(0, min(ch, n - base));
    const double dt = a.dt;
    constexpr int K = 2 * D + 1;
    constexpr bool CROSS = OP == PIT_OP_LSDE;
    // p and r (with halos of W nodes on both sides), x, rh, v, t, the table
    double *p = reinterpret_cast<double *>(smem) + W, *r = p + ch + 2 * W;
    double *x = r + ch + W, *rh = x + ch, *v = rh + ch, *t = v + ch, *tab = t + ch;
    uint16_t *mask = reinterpret_cast<uint16_t *>(tab + (size_t)K * ch);
    const double *in = a.in + (long long)b * a.in_stride + GI.off + base;
    const double *f0 = a.f ? a.f + (long long)b * a.f_stride + GI.off + base : nullptr;
    for (int j = tid; j < ch + 2 * W; j += nt) p[j - W] = r[j - W] = 0.0;
    for (int j = tid; j < cnt; j += nt) {
        mask[j] = a.masks[GI.off + base + j];
        x[j] = in[j];
        tab[j] = op_coef<OP>(a.op, GI, a.faces, base + j, dt, [&](int q, int, double cm, double cp) {
            tab[(1 + 2 * q) * ch + j] = cm;
            tab[(2 + 2 * q) * ch + j] = cp;
        });
        for (int k = 2 * GI.de + 1; k < K; ++k) tab[k * ch + j] = 0.0;
    }
    __syncthreads();
    // (a launch's grids may have fewer axes than D: those add nothing)
    int S[D];
#pragma unroll
    for (int i = 0; i < D; ++i) S[i] = i < GI.de ? GI.S[GI.ax[i]] : 0;
    bool mixed = false;
    if constexpr (CROSS) {
#pragma unroll
        for (int q = 0; q < D * (D - 1) / 2; ++q) mixed = mixed || (q < GI.de * (GI.de - 1) / 2 && IC.cr[q] != 0.0);
    }
    // (A u)_j, u with halos.  A coefficient towards the boundary is zero and its
    // neighbour some finite value of another line (or the zero halo's).
    auto A = [&](const double *u, int j) -> double {
        double s = tab[j] * u[j];
#pragma unroll
        for (int i = 0; i < D; ++i) {
            s = fma(tab[(1 + 2 * i) * ch + j], u[j - S[i]], s);
            s = fma(tab[(2 + 2 * i) * ch + j], u[j + S[i]], s);
        }
        if constexpr (CROSS)
            if (mixed) {
                const unsigned mk = mask[j];
                int q = 0;
#pragma unroll
                for (int i = 0; i < D; ++i)
#pragma unroll
                    for (int k = i + 1; k < D; ++k, ++q) {
                        const bool im = (mk >> (2 * i)) & 1u, ip = (mk >> (2 * i + 1)) & 1u;
                        const bool km = (mk >> (2 * k)) & 1u, kp = (mk >> (2 * k + 1)) & 1u;
                        double c = 0.0;
                        if (ip && kp) c += u[j + S[i] + S[k]];
                        if (ip && km) c -= u[j + S[i] - S[k]];
                        if (im && kp) c -= u[j - S[i] + S[k]];
                        if (im && km) c += u[j - S[i] - S[k]];
                        s = fma(IC.cr[q], c, s);
                    }
            }
        return s;
    };
    // node j of the halo'd vector u also goes to the neighbours' halos (their
    // runs of ch nodes: W <= ch, so only the two next to this one need it)
    double *pl = rank > 0 ? cl.map_shared_rank(p, rank - 1) : nullptr;
    double *pr = rank + 1 < C ? cl.map_shared_rank(p, rank + 1) : nullptr;
    double *rl = rank > 0 ? cl.map_shared_rank(r, rank - 1) : nullptr;
    double *rr_ = rank + 1 < C ? cl.map_shared_rank(r, rank + 1) : nullptr;
    auto put = [&](double *u, double *ul, double *ur, int j, double val) {
        u[j] = val;
        if (ul && j < W) ul[ch + j] = val;
        if (ur && j >= ch - W) ur[j - ch] = val;
    };
    const bool lead = tid < 32;
    int slot = 0, status = PIT_OK, iters = 0;
    const double near0 = 1e-12;
    cl.sync();  // halos cleared everywhere before the first store into them

    for (int step = 1; step <= a.nsteps; ++step) {
        const double *f = f0 ? f0 + (long long)((step - 1) / a.f_div) * a.f_step : nullptr;
        const long long sb = (long long)(step - 1);
        const double *gu = a.guess ? a.guess + (long long)b * a.guess_stride + sb * a.guess_step + GI.off + base : nullptr;
        const double *gs = a.g ? a.g + (long long)b * a.g_stride + sb * a.g_step + GI.off + base : nullptr;
        // right-hand side into rh, iterate into p (halo'd)
        double s2[2] = {0.0, 0.0};
        for (int j = tid; j < cnt; j += nt) {
            const double bj = f ? x[j] + dt * f[j] : x[j];
            rh[j] = bj;
            s2[0] += bj * bj;
            if (gu) x[j] = gs ? gu[j] - gs[j] : gu[j];
            put(p, pl, pr, j, x[j]);
        }
        cl.sync();
#pragma unroll 4
        for (int j = tid; j < cnt; j += nt) {
            const double rj = rh[j] - A(p, j);
            r[j] = rj;
            rh[j] = rj;
            v[j] = 0.0;
            s2[1] += rj * rj;
        }
        cluster_sum<2>(cl, RS, slot, s2);  // (also: every stencil has read p)
        for (int j = tid; j < cnt; j += nt) p[j] = 0.0;
        // BiCGStab as in bicgstab_core; the scalars live in warp 0
        double rho = 1.0, alpha = 1.0, omega = 1.0, rr = s2[1], rhh = s2[1], rho_n = s2[1];
        const double stop2 = a.rtol * a.rtol * s2[0];
        int k = 0, k_restart = -1, st = PIT_OK;
        for (;;) {
            if (lead) {
                int act = CL_GO;
                double beta = 0.0;
                auto breakdown = [&]() {
                    if (k != k_restart) {
                        k_restart = k;
                        rho = alpha = omega = 1.0;
                        rhh = rho_n = rr;
                        act = CL_RESTART;
                    } else {
                        st = PIT_ERR_BREAKDOWN;
                        act = CL_DONE;
                    }
                };
                if (!(rr > stop2)) {
                    if (rr != rr) st = PIT_ERR_NONFINITE;
                    act = CL_DONE;
                } else if (k >= a.maxit) {
                    st = PIT_ERR_NOCONV;
                    act = CL_DONE;
                } else if (rho_n != rho_n) {
                    st = PIT_ERR_NONFINITE;
                    act = CL_DONE;
                } else if (!(fabs(rho_n) > near0 * sqrt(rr) * sqrt(rhh))) {
                    breakdown();
                } else {
                    beta = (rho_n / rho) * (alpha / omega);
                    if (beta != beta) {
                        st = PIT_ERR_NONFINITE;
                        act = CL_DONE;
                    } else if (!(fabs(beta) < 1e30)) {
                        breakdown();
                    }
                }
                if (tid == 0) {
                    SC.act = act;
                    SC.beta = beta;
                    SC.omega = omega;
                }
            }
            __syncthreads();
            if (SC.act == CL_DONE) break;
            if (SC.act == CL_RESTART) {
                for (int j = tid; j < cnt; j += nt) {
                    rh[j] = r[j];
                    p[j] = 0.0;
                    v[j] = 0.0;
                }
                __syncthreads();  // SC read by every thread
                continue;
            }
            {
                const double beta = SC.beta, om = SC.omega;
#pragma unroll 4
                for (int j = tid; j < cnt; j += nt) put(p, pl, pr, j, fma(beta, fma(-om, v[j], p[j]), r[j]));
            }
            cl.sync();
            double s1[1] = {0.0};
#pragma unroll 4
            for (int j = tid; j < cnt; j += nt) {
                const double vj = A(p, j);
                v[j] = vj;
                s1[0] = fma(rh[j], vj, s1[0]);
            }
            cluster_sum<1>(cl, RS, slot, s1);
            if (lead) {
                int act = CL_GO;
                if (s1[0] != s1[0]) {
                    st = PIT_ERR_NONFINITE;
                    act = CL_DONE;
                } else {
                    alpha = rho_n / s1[0];
                    if (!(fabs(alpha) < 1e30)) {
                        if (k != k_restart) {
                            k_restart = k;
                            rho = alpha = omega = 1.0;
                            rhh = rho_n = rr;
                            act = CL_RESTART;
                        } else {
                            st = PIT_ERR_BREAKDOWN;
                            act = CL_DONE;
                        }
                    }
                }
                if (tid == 0) {
                    SC.act = act;
                    SC.alpha = alpha;
                }
            }
            __syncthreads();
            if (SC.act == CL_DONE) break;
            if (SC.act == CL_RESTART) {
                for (int j = tid; j < cnt; j += nt) {
                    rh[j] = r[j];
                    p[j] = 0.0;
                    v[j] = 0.0;
                }
                __syncthreads();
                continue;
            }
            {
                const double al = SC.alpha;
#pragma unroll 4
                for (int j = tid; j < cnt; j += nt) put(r, rl, rr_, j, fma(-al, v[j], r[j]));  // s
            }
            cl.sync();
            double st2[2] = {0.0, 0.0};
#pragma unroll 4
            for (int j = tid; j < cnt; j += nt) {
                const double tj = A(r, j);
                t[j] = tj;
                st2[0] = fma(tj, tj, st2[0]);
                st2[1] = fma(tj, r[j], st2[1]);
            }
            cluster_sum<2>(cl, RS, slot, st2);
            if (lead) {
                omega = st2[0] > 0.0 ? st2[1] / st2[0] : 0.0;
                const bool bad = omega != omega;
                if (bad) st = PIT_ERR_NONFINITE;
                else if (!(fabs(omega) < 1e30)) omega = 0.0;  // take the BiCG half step only
                if (tid == 0) {
                    SC.act = bad ? CL_DONE : CL_GO;
                    SC.omega = omega;
                }
            }
            __syncthreads();
            if (SC.act == CL_DONE) break;
            double sn[2] = {0.0, 0.0};
            {
                const double al = SC.alpha, om = SC.omega;
#pragma unroll 4
                for (int j = tid; j < cnt; j += nt) {
                    const double sj = r[j];
                    x[j] += fma(al, p[j], om * sj);
                    const double rj = fma(-om, t[j], sj);
                    r[j] = rj;
                    sn[0] = fma(rj, rj, sn[0]);
                    sn[1] = fma(rh[j], rj, sn[1]);
                }
            }
            cluster_sum<2>(cl, RS, slot, sn);
            ++k;
            if (lead) {
                rho = rho_n;
                rr = sn[0];
                rho_n = sn[1];
                int act = CL_GO;
                if (omega == 0.0 && rr > stop2) {
                    if (k != k_restart) {
                        k_restart = k;
                        rho = alpha = omega = 1.0;
                        rhh = rho_n = rr;
                        act = CL_RESTART;
                    } else {
                        st = PIT_ERR_BREAKDOWN;
                        act = CL_DONE;
                    }
                } else if (omega == 0.0 && rr != rr) {
                    st = PIT_ERR_NONFINITE;
                    act = CL_DONE;
                }
                if (tid == 0) SC.act = act;
            }
            __syncthreads();
            if (SC.act == CL_DONE) break;
            if (SC.act == CL_RESTART)
                for (int j = tid; j < cnt; j += nt) {
                    rh[j] = r[j];
                    p[j] = 0.0;
                    v[j] = 0.0;
                }
            __syncthreads();  // SC read before the next round writes it
        }
        // (k is the same in every thread; st is warp 0's)
        iters += k;
        if (st > status) status = st;
        __syncthreads();
        // forcing of this step and the stored outputs (own nodes only)
        if (gs)
            for (int j = tid; j < cnt; j += nt) x[j] += gs[j];
        const double *hs = a.hs ? a.hs + (long long)b * a.hs_stride + sb * a.hs_step + GI.off + base : nullptr;
        if (step < a.nsteps) {
            if (a.out_steps) {
                double *os = a.out_steps + (long long)b * a.os_stride + sb * a.os_step + GI.off + base;
                for (int j = tid; j < cnt; j += nt) os[j] = hs ? x[j] + hs[j] : x[j];
            }
        } else {
            double *ol = a.out_last + (long long)b * a.ol_stride + GI.off + base;
            const double *h = a.h ? a.h + (long long)b * a.h_stride + GI.off + base : nullptr;
            const double *cmp = a.cmp ? a.cmp + (long long)b * a.cmp_stride + GI.off + base : nullptr;
            double acc[1] = {0.0};
            for (int j = tid; j < cnt; j += nt) {
                const double xj = x[j];
                if (cmp) {
                    const double dlt = xj - cmp[j];
                    acc[0] += dlt * dlt;
                }
                ol[j] = a.out_scale * xj + (h ? a.out_hscale * h[j] : 0.0) + (hs ? hs[j] : 0.0);
            }
            if (a.cmp) {
                cluster_sum<1>(cl, RS, slot, acc);
                if (rank == 0 && tid == 0) a.norms[(long long)b * a.n_grids + g] = sqrt(acc[0]);
            }
        }
    }
    if (a.inexact && status == PIT_ERR_NOCONV) status = PIT_OK;  // fixed-iteration (inexact) solves
    if (rank == 0 && tid == 0 && a.stats) {
        atomicAdd(&a.stats->sum_iters, (unsigned long long)iters);
        atomicAdd(&a.stats->items, (unsigned long long)a.nsteps);
        atomicAdd(&a.stats->point_iters, (unsigned long long)iters * (unsigned long long)n);
        atomicAdd(&a.stats->point_passes, (unsigned long long)a.nsteps * (unsigned long long)n);
        atomicAdd(&a.stats->point_steps, (unsigned long long)a.nsteps * (unsigned long long)n);
        atomicMax(&a.stats->max_iters, iters);
        atomicMax(&a.stats->max_refine, a.nsteps);
        if (status != PIT_OK) {
            atomicAdd(&a.stats->n_failed, 1);
            atomicMax(&a.stats->worst, status);
        }
    }
    cl.sync();  // no CTA leaves while another may still store into its memory
}

// the kernel of an operator and grid dimension (listed axes), or NULL
const void *cluster_fn(int op, int de)
{
    switch (op) {
#define PIT_CL(OPV)                                                            \
    case OPV:                                                                  \
        switch (de) {                                                          \
        case 1: return (const void *)cluster_kernel<OPV, 1>;                   \
        case 2: return (const void *)cluster_kernel<OPV, 2>;                   \
        case 3: return (const void *)cluster_kernel<OPV, 3>;                   \
        default: return nullptr;                                               \
        }
        PIT_CL(PIT_OP_OU) PIT_CL(PIT_OP_LSDE) PIT_CL(PIT_OP_CME)
#undef PIT_CL
    default: return nullptr;
    }
}

}  // namespace

size_t cluster_smem_bytes(const GridInfo &G, int C, int reach)
{
    const size_t ch = (size_t)((G.n + C - 1) / C);
    return (ch * (6 + 2 * G.de + 1) + 4 * (size_t)reach) * 8 + ch * 2 + 16;
}

int cluster_reach(const GridInfo &G, int op)
{
    int far = 0, next = 0;
    for (int q = 0; q < G.de; ++q) {
        const int s = G.S[G.ax[q]];
        if (s > far) {
            next = far;
            far = s;
        } else if (s > next) {
            next = s;
        }
    }
    return op == PIT_OP_LSDE ? far + next : far;
}

bool cluster_kernel_for(int op, int de) { return cluster_fn(op, de) != nullptr; }

static cudaLaunchConfig_t cluster_config(int items, int C, size_t smem, cudaStream_t s, cudaLaunchAttribute *attr)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(items * C));
    cfg.blockDim = dim3(CL_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    attr->id = cudaLaunchAttributeClusterDimension;
    attr->val.clusterDim.x = (unsigned)C;
    attr->val.clusterDim.y = attr->val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cfg;
}

// (a kernel's limits hold for every problem of the process: they are set to the
// most that any of them asks for, and stay)
cudaError_t cluster_init(size_t max_smem)
{
    for (int op : {(int)PIT_OP_OU, (int)PIT_OP_LSDE, (int)PIT_OP_CME})
        for (int de = 1; const void *fn = cluster_fn(op, de); ++de) {
            cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_smem);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

int cluster_capacity(int op, int de, int C, size_t smem)
{
    const void *fn = cluster_fn(op, de);
    if (!fn) return 0;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = cluster_config(1, C, smem, nullptr, &attr);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, fn, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return n;
}

cudaError_t launch_cluster(const StepArgs &a, int de, int C, int reach, size_t smem, cudaStream_t s)
{
    const long long items = (long long)a.n_batch * a.n_order;
    if (items <= 0) return cudaSuccess;
    const void *fn = cluster_fn(a.op.op, de);
    if (!fn || C < 2 || C > CL_MAX || items * C > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = cluster_config((int)items, C, smem, s, &attr);
    StepArgs args = a;
    void *params[] = {&args, &reach};
    return cudaLaunchKernelExC(&cfg, fn, params);
}

}  // namespace pit
