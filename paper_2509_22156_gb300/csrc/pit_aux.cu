// Auxiliary kernels of libpit: stencil application, initial values, face
// coefficients of the variable-coefficient operator, the combination sum and
// the MGRIT residual norms.
#include "pit_internal.cuh"

namespace pit {

__device__ __forceinline__ int axis_coord(const GridInfo &G, int j, int i) { return (j / G.S[i]) % G.N[i]; }

// Variable diffusion coefficient a(x) = 1 + A prod_i f_i(x_i), f alternating
// sin(2 pi x), cos(2 pi x), ... (d = 3: 1 + A sin(2 pi x1) cos(2 pi x2) sin(2 pi x3)).
__device__ double varcoef(const OpParams &op, const double *x)
{
    double prod = 1.0;
    for (int i = 0; i < op.d; ++i) prod *= (i % 2 == 0) ? sin(2.0 * M_PI * x[i]) : cos(2.0 * M_PI * x[i]);
    return 1.0 + op.vamp * prod;
}

// (I + dt L) p at node j of grid GI, FP64 with coefficients evaluated per
// node (the reference application of the operator).
__device__ double apply_node(const GridInfo &GI, int j, const double *pg, double dt, const double *faces,
                             const OpParams &op)
{
    const int d = op.d;
    double s = 0.0, diag = 1.0;
    for (int i = 0; i < d; ++i) {
        const int c = axis_coord(GI, j, i);
        const double h = GI.h[i], ih2 = 1.0 / (h * h);
        double dd, dm, dp;
        if (op.op == PIT_OP_HEAT) {
            dd = 2.0 * ih2; dm = -ih2; dp = -ih2;
        } else if (op.op == PIT_OP_VARHEAT) {
            const double am = faces[(GI.off + j) * (2 * d) + 2 * i];
            const double ap = faces[(GI.off + j) * (2 * d) + 2 * i + 1];
            dd = (am + ap) * ih2; dm = -am * ih2; dp = -ap * ih2;
        } else if (op.op == PIT_OP_OU) {
            const double x = op.lo[i] + (double)(c + 1) * h;
            const double vp = -op.theta * (x + 0.5 * h), vm = -op.theta * (x - 0.5 * h);
            const double s2 = 0.5 * op.sigma * op.sigma * ih2;
            drift_coef(vp, vm, h, false, dd, dm, dp);
            dd += 2.0 * s2;
            dm -= s2;
            dp -= s2;
        } else if (op.op == PIT_OP_CME) {
            double xc[PIT_D];
            for (int k = 0; k < d; ++k) xc[k] = op.lo[k] + (double)(axis_coord(GI, j, k) + 1) * GI.h[k];
            cme_coef(cme_production(op, i, xc, d), op.cg[i], xc[i], h, op.central != 0, dd, dm, dp);
        } else {
            // linear SDE: face velocities (A x)_i at x -+ h/2 e_i, diagonal diffusion
            double ax = 0.0;
            for (int k = 0; k < d; ++k)
                ax += op.A[i * d + k] * (op.lo[k] + (double)(axis_coord(GI, j, k) + 1) * GI.h[k]);
            const double vp = ax + 0.5 * h * op.A[i * d + i], vm = ax - 0.5 * h * op.A[i * d + i];
            const double s2 = 0.5 * op.H[i * d + i] * ih2;
            drift_coef(vp, vm, h, op.central != 0, dd, dm, dp);
            dd += 2.0 * s2;
            dm -= s2;
            dp -= s2;
        }
        diag += dt * dd;
        if (c > 0) s += dt * dm * pg[j - GI.S[i]];
        if (c < GI.N[i] - 1) s += dt * dp * pg[j + GI.S[i]];
    }
    if (op.op == PIT_OP_LSDE) {
        // mixed derivatives: -(H_ik + H_ki)/2 (p_{++} - p_{+-} - p_{-+} + p_{--}) / (4 h_i h_k)
        for (int i = 0; i < d; ++i) {
            const int ci = axis_coord(GI, j, i);
            for (int k = i + 1; k < d; ++k) {
                const int ck = axis_coord(GI, j, k);
                const double w = -dt * 0.5 * (op.H[i * d + k] + op.H[k * d + i]) / (4.0 * GI.h[i] * GI.h[k]);
                double c4 = 0.0;
                if (ci < GI.N[i] - 1 && ck < GI.N[k] - 1) c4 += pg[j + GI.S[i] + GI.S[k]];
                if (ci < GI.N[i] - 1 && ck > 0) c4 -= pg[j + GI.S[i] - GI.S[k]];
                if (ci > 0 && ck < GI.N[k] - 1) c4 -= pg[j - GI.S[i] + GI.S[k]];
                if (ci > 0 && ck > 0) c4 += pg[j - GI.S[i] - GI.S[k]];
                s += w * c4;
            }
        }
    }
    return diag * pg[j] + s;
}

// q = (I + dt L) p, one CTA per (batch entry, grid).
__global__ void apply_kernel(const GridInfo *grids, int G, long long ntot, double dt, const double *p, double *q,
                             const double *faces, OpParams op)
{
    const int g = blockIdx.x % G, b = blockIdx.x / G;
    const GridInfo GI = grids[g];
    const double *pg = p + (long long)b * ntot + GI.off;
    double *qg = q + (long long)b * ntot + GI.off;
    for (int j = threadIdx.x; j < GI.n; j += blockDim.x) qg[j] = apply_node(GI, j, pg, dt, faces, op);
}

// Space-time residual of the backward-Euler equation at a C-point (the
// residual mode of MGRIT): rho_b = x_b + dt f_b - (I + dt L) u_b, written as
// scale * rho_b, with ||rho_b||_2 per grid in norms[b * G + g]; active grids
// only (others untouched).  One CTA of 256 threads per (batch entry, grid).
__global__ void st_resid_kernel(const GridInfo *grids, int G, long long ntot, double dt, const double *x,
                                long long xs, const double *f, long long fs, const double *u, long long us,
                                double scale, double *out, long long os, double *norms, const int *active,
                                const double *faces, OpParams op)
{
    const int g = blockIdx.x % G, b = blockIdx.x / G;
    if (active && !active[g]) return;
    const GridInfo GI = grids[g];
    const double *xg = x + b * xs + GI.off, *ug = u + b * us + GI.off;
    const double *fg = f ? f + b * fs + GI.off : nullptr;
    double *og = out + b * os + GI.off;
    double acc = 0.0;
    for (int j = threadIdx.x; j < GI.n; j += blockDim.x) {
        const double r = xg[j] + (fg ? dt * fg[j] : 0.0) - apply_node(GI, j, ug, dt, faces, op);
        og[j] = scale * r;
        acc += r * r;
    }
    __shared__ double part[8];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
        norms[(long long)b * G + g] = sqrt(t);
    }
}

cudaError_t launch_st_resid(const GridInfo *grids, int G, long long ntot, int nb, double dt, const double *x,
                            long long xs, const double *f, long long fs, const double *u, long long us, double scale,
                            double *out, long long os, double *norms, const int *active, const double *faces,
                            OpParams op, cudaStream_t s)
{
    const long long blocks = (long long)G * nb;
    if (blocks == 0) return cudaSuccess;
    st_resid_kernel<<<(unsigned)blocks, 256, 0, s>>>(grids, G, ntot, dt, x, xs, f, fs, u, us, scale, out, os, norms,
                                                      active, faces, op);
    return cudaGetLastError();
}

cudaError_t launch_apply(const GridInfo *grids, int G, long long ntot, int n_batch, double dt, const double *p,
                         double *q, const double *faces, OpParams op, cudaStream_t s)
{
    const long long blocks = (long long)G * n_batch;
    if (blocks == 0) return cudaSuccess;
    apply_kernel<<<(unsigned)blocks, 256, 0, s>>>(grids, G, ntot, dt, p, q, faces, op);
    return cudaGetLastError();
}

// Initial values at the interior nodes (kind 0: sum of product-sine modes,
// kind 1: product Gaussian); one CTA per grid.
__global__ void initial_kernel(const GridInfo *grids, OpParams op, const double *hi, int kind, const double *prm,
                               double *u)
{
    const GridInfo GI = grids[blockIdx.x];
    const int d = op.d;
    for (int j = threadIdx.x; j < GI.n; j += blockDim.x) {
        double x[PIT_D];
        for (int i = 0; i < d; ++i) x[i] = op.lo[i] + (double)(axis_coord(GI, j, i) + 1) * GI.h[i];
        double v = 0.0;
        if (kind == 0) {
            const int K = (int)prm[0];
            for (int k = 0; k < K; ++k) {
                const double *pk = prm + 1 + k * (d + 1);
                double prod = pk[0];
                for (int i = 0; i < d; ++i) prod *= sin(M_PI * pk[1 + i] * (x[i] - op.lo[i]) / (hi[i] - op.lo[i]));
                v += prod;
            }
        } else if (kind == 4) {
            // normal density with the covariance's Cholesky factor R (prm[d..]) and
            // log det R (prm[d + d*d]), prepared on the host
            double z[PIT_D], q = 0.0;
            for (int i = 0; i < d; ++i) {
                double r = x[i] - prm[i];
                for (int k = 0; k < i; ++k) r -= prm[d + i * d + k] * z[k];
                z[i] = r / prm[d + i * d + i];
                q += z[i] * z[i];
            }
            v = exp(-0.5 * q - prm[d + d * d] - 0.5 * d * log(2.0 * M_PI));
        } else if (kind == 1) {
            v = 1.0;
            for (int i = 0; i < d; ++i) {
                const double z = (x[i] - prm[i]) / prm[d + i];
                v *= exp(-0.5 * z * z) / (prm[d + i] * sqrt(2.0 * M_PI));
            }
        } else {
            // heat experiment (Sec. 4.2): u*(x,t) = rho e^{-t} S(x), rho = sqrt(|x|^2 + t^2),
            // S = prod_i sin(pi xi_i), xi_i = (x_i - a_i) / w_i; kind 3 gives
            // f = du*/dt - Laplace u* = e^{-t} [S (t/rho - rho) - S (d/rho - |x|^2/rho^3)
            //     - 2 sum_i (x_i/rho) dS/dx_i + rho pi^2 S sum_i 1/w_i^2]
            const double t = prm[0];
            double r2 = 0.0, S = 1.0, sn[PIT_D], cs[PIT_D], w[PIT_D];
            for (int i = 0; i < d; ++i) {
                w[i] = hi[i] - op.lo[i];
                sincospi((x[i] - op.lo[i]) / w[i], &sn[i], &cs[i]);
                S *= sn[i];
                r2 += x[i] * x[i];
            }
            const double rho = sqrt(r2 + t * t), et = exp(-t);
            if (kind == 2) {
                v = rho * et * S;
            } else {
                double grad = 0.0, iw2 = 0.0;
                for (int i = 0; i < d; ++i) {
                    double dS = M_PI / w[i] * cs[i];
                    for (int k = 0; k < d; ++k)
                        if (k != i) dS *= sn[k];
                    grad += x[i] / rho * dS;
                    iw2 += 1.0 / (w[i] * w[i]);
                }
                v = et * (S * (t / rho - rho) - S * (d / rho - r2 / (rho * rho * rho)) - 2.0 * grad +
                          rho * M_PI * M_PI * S * iw2);
            }
        }
        u[GI.off + j] = v;
    }
}

cudaError_t launch_initial(const GridInfo *grids, int G, OpParams op, const double *hi, int kind,
                           const double *params_dev, int n_params, double *u, cudaStream_t s)
{
    (void)n_params;
    initial_kernel<<<G, 256, 0, s>>>(grids, op, hi, kind, params_dev, u);
    return cudaGetLastError();
}

// Face values a(x -+ h_i/2 e_i) of every node (2d per node, packed like the
// state vectors), computed once per problem.
__global__ void faces_kernel(const GridInfo *grids, OpParams op, double *faces)
{
    const GridInfo GI = grids[blockIdx.x];
    const int d = op.d;
    for (int j = threadIdx.x; j < GI.n; j += blockDim.x) {
        double x[PIT_D];
        for (int i = 0; i < d; ++i) x[i] = op.lo[i] + (double)(axis_coord(GI, j, i) + 1) * GI.h[i];
        for (int i = 0; i < d; ++i) {
            const double xi = x[i];
            x[i] = xi - 0.5 * GI.h[i];
            faces[(GI.off + j) * (2 * d) + 2 * i] = varcoef(op, x);
            x[i] = xi + 0.5 * GI.h[i];
            faces[(GI.off + j) * (2 * d) + 2 * i + 1] = varcoef(op, x);
            x[i] = xi;
        }
    }
}

__global__ void masks_kernel(const GridInfo *grids, uint16_t *masks)
{
    const GridInfo GI = grids[blockIdx.x];
    for (int j = threadIdx.x; j < GI.n; j += blockDim.x) {
        unsigned mk = 0;
        for (int q = 0; q < GI.de; ++q) {
            const int i = GI.ax[q], c = axis_coord(GI, j, i);
            if (c > 0) mk |= 1u << (2 * q);
            if (c < GI.N[i] - 1) mk |= 1u << (2 * q + 1);
        }
        masks[GI.off + j] = (uint16_t)mk;
    }
}

cudaError_t launch_masks(const GridInfo *grids, int G, uint16_t *masks, cudaStream_t s)
{
    masks_kernel<<<G, 256, 0, s>>>(grids, masks);
    return cudaGetLastError();
}

cudaError_t launch_faces(const GridInfo *grids, int G, OpParams op, double *faces, cudaStream_t s)
{
    faces_kernel<<<G, 256, 0, s>>>(grids, op, faces);
    return cudaGetLastError();
}

// Combination sum (Eq. "combination_technique_solution") at arbitrary points:
// out[k] = sum_g coef_g I_g[u_g](x_k), I_g piecewise d-linear with zero
// boundary values.  One thread per point; blockIdx.y takes a contiguous chunk
// of grids in canonical order.  With one chunk the thread writes the sum;
// with several it writes its chunk's partial sum to part[chunk][k] and
// combine_sum_kernel adds the chunks in chunk order.  (One thread per point
// over all grids would keep only n_pts / 128 SMs busy, 33 of 152 for the
// 4,100 points of the d = 6 workload, on FP64 interpolation work.)
__global__ void combine_kernel(const GridInfo *grids, const double *coef, const int *levels, int G, OpParams op,
                               const double *u, int n_pts, const double *pts, int gchunk, double *dst)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_pts) return;
    const int g0 = (int)blockIdx.y * gchunk;
    const int g1 = min(G, g0 + gchunk);
    const int d = op.d;
    // position in units of the domain, once per point: the cell coordinate on
    // a grid of level l is then xr 2^l, an exact scaling (no division per grid)
    double xr[PIT_D];
    for (int i = 0; i < d; ++i) {
        // domain extent hi - lo = h 2^l of any grid (exact: h was (hi - lo) / 2^l)
        const double ext = ldexp(grids[0].h[i], levels[i]);
        xr[i] = (pts[(long long)k * d + i] - op.lo[i]) / ext;
    }
    const int dl = d / 2;  // corner weights: products over the first dl axes times the rest
    double acc = 0.0;
    for (int g = g0; g < g1; ++g) {
        const GridInfo &GI = grids[g];
        int cell[PIT_D];
        double t[PIT_D];
        for (int i = 0; i < d; ++i) {
            const int l = levels[g * d + i];
            const int M = 1 << l;
            const double s = ldexp(xr[i], l);
            int c = (int)floor(s);
            c = c < 0 ? 0 : (c > M - 1 ? M - 1 : c);
            cell[i] = c;
            t[i] = s - (double)c;
        }
        double wlo[8], whi[8];
        wlo[0] = 1.0;
        for (int i = 0; i < dl; ++i)
            for (int q = (1 << i) - 1; q >= 0; --q) {
                wlo[2 * q + 1] = wlo[q] * t[i];
                wlo[2 * q] = wlo[q] * (1.0 - t[i]);
            }
        whi[0] = 1.0;
        for (int i = dl; i < d; ++i)
            for (int q = (1 << (i - dl)) - 1; q >= 0; --q) {
                whi[2 * q + 1] = whi[q] * t[i];
                whi[2 * q] = whi[q] * (1.0 - t[i]);
            }
        double val = 0.0;
        for (int corner = 0; corner < (1 << d); ++corner) {
            long long idx = 0;
            bool inside = true;
            int lo_bits = 0, hi_bits = 0;
            for (int i = 0; i < d; ++i) {
                const int bit = (corner >> i) & 1;
                const int node = cell[i] + bit;  // 0 and 2^l are boundary nodes
                if (i < dl) lo_bits |= bit << (dl - 1 - i);
                else hi_bits |= bit << (d - 1 - i);
                if (node <= 0 || node > GI.N[i]) inside = false;
                else idx += (long long)(node - 1) * GI.S[i];
            }
            if (inside) val += (wlo[lo_bits] * whi[hi_bits]) * u[GI.off + idx];
        }
        acc += coef[g] * val;
    }
    dst[(long long)blockIdx.y * n_pts + k] = acc;
}

__global__ void combine_sum_kernel(const double *part, int n_chunks, int n_pts, double *out)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n_pts) return;
    double s = 0.0;
    for (int c = 0; c < n_chunks; ++c) s += part[(long long)c * n_pts + k];
    out[k] = s;
}

int combine_chunks(int G, int n_pts, int n_sm)
{
    const int blocks = (n_pts + 127) / 128;
    const int want = 4 * (n_sm > 0 ? n_sm : 1);  // about four 128-thread blocks per SM
    int chunks = (want + blocks - 1) / blocks;
    chunks = chunks < 1 ? 1 : (chunks > G ? G : chunks);
    const int gchunk = (G + chunks - 1) / chunks;
    return (G + gchunk - 1) / gchunk;
}

cudaError_t launch_combine(const GridInfo *grids, const double *coef, const int *levels, int G, OpParams op,
                           const double *u, int n_pts, const double *pts, double *out, int n_chunks, double *part,
                           cudaStream_t s)
{
    if (n_pts == 0 || G == 0) return cudaSuccess;
    if (n_chunks < 1 || (n_chunks > 1 && !part)) return cudaErrorInvalidValue;
    const int gchunk = (G + n_chunks - 1) / n_chunks;
    const int chunks = (G + gchunk - 1) / gchunk;
    const dim3 grid((unsigned)((n_pts + 127) / 128), (unsigned)chunks);
    combine_kernel<<<grid, 128, 0, s>>>(grids, coef, levels, G, op, u, n_pts, pts, gchunk, chunks > 1 ? part : out);
    if (chunks > 1) combine_sum_kernel<<<(n_pts + 127) / 128, 128, 0, s>>>(part, chunks, n_pts, out);
    return cudaGetLastError();
}

// The combination sum at many points.  A component grid's interpolant also lies
// in the space of any grid that is finer along one axis, so the grids that
// differ in the last axis' level only (at most d) are one function on the
// finest of them: merge_kernel adds them there, node by node, and a point then
// reads one cell of every group: 84 groups for the 195 grids of d = 4, level 7,
// and 2,002 for the 4,921 of d = 6, level 10.
//
// Interpolation weights are never negative, so a value's rounding errors keep
// to the cells that contain it, as in the sum over grids: the error at a point
// is of the size of 2^-53 sum_l |c_l| I_l[|u_l|](x), the values near that point.
// (The sum of hierarchical surpluses, with fewer terms yet, does not have this:
// its terms are of the size of the largest value anywhere, and the tails of a
// density come out as noise.)
__global__ void __launch_bounds__(256) merge_kernel(CombinePlan C, const double *u, double *M)
{
    const CombinePiece pc = C.pieces[blockIdx.x];
    const CombineGroup &G = C.groups[pc.group];
    const int j = pc.first + threadIdx.x;
    if (j >= G.n) return;
    const int d1 = G.mask >> PIT_D, de = __popc(G.mask & ((1 << PIT_D) - 1));  // last axis listed; listed axes
    const int L = d1 ? G.lev[de - 1] : 1, row = j / ((1 << L) - 1), p = j - row * ((1 << L) - 1) + 1;
    double s = 0.0;
    for (int k = G.term0; k < G.term1; ++k) {
        const CombineTerm t = C.terms[k];
        const int sh = L - t.lev, N = (1 << t.lev) - 1, c = p >> sh, rem = p & ((1 << sh) - 1);
        const double *r = u + t.off + (long long)row * N;  // r[c - 1]: node c of the member's line
        double v = 0.0;
        if (rem == 0) {
            v = r[c - 1];
        } else {
            // (boundary values are not read, nor multiplied with)
            const double f = (double)rem / (double)(1 << sh);
            if (c > 0) v = (1.0 - f) * r[c - 1];
            if (c < N) v = fma(f, r[c], v);
        }
        s = fma(t.coef, v, s);
    }
    long long at = G.at + (d1 ? p : 0);
    for (int q = de - 1 - d1, rr = row; q >= 0; --q) {
        const int N = (1 << G.lev[q]) - 1;
        at += (long long)(rr % N + 1) * G.stride[q];
        rr /= N;
    }
    M[at] = s;
}

// multilinear interpolation in the cell at p, weights t and r = 1 - t
template <int Q, int DE>
__device__ __forceinline__ double cell_value(const double *p, const int (&S)[DE + 1], const double (&t)[DE + 1],
                                             const double (&r)[DE + 1])
{
    if constexpr (Q == DE) return *p;
    else return fma(t[Q], cell_value<Q + 1, DE>(p + S[Q], S, t, r), r[Q] * cell_value<Q + 1, DE>(p, S, t, r));
}
// sum over the groups of a run that blockIdx.y takes (every gridDim.y-th); place
// and cell: this thread's columns of the tables
template <int DE>
__device__ __forceinline__ double run_value(const CombinePlan &C, const CombineRun &R, const double *M,
                                            const double *place, const int *cell)
{
    int ax[DE + 1], fine[DE + 1];
#pragma unroll
    for (int q = 0, m = R.mask; q < DE; ++q, m &= m - 1) {
        ax[q] = __ffs(m) - 1;
        fine[q] = cell[ax[q] * 128];
    }
    double v = 0.0;
    for (int g = R.first + blockIdx.y; g < R.last; g += gridDim.y) {
        const CombineGroup &G = C.groups[g];
        long long at = G.at;
        int S[DE + 1];
        double t[DE + 1], r[DE + 1];
#pragma unroll
        for (int q = 0; q < DE; ++q) {
            const int lam = G.lev[q];
            S[q] = G.stride[q];
            t[q] = place[(ax[q] * C.l_max + lam - 1) * 128];
            r[q] = 1.0 - t[q];
            at += (long long)(fine[q] >> (C.l_max - lam)) * S[q];
        }
        v += cell_value<0, DE>(M + at, S, t, r);
    }
    return v;
}
// One thread a point.  What bounds it: the loads of the cells' corners, 608 a
// point for d = 4, level 7, from L1 and L2, beside the FP64 unit (1,500
// operations a point, 0.17 ms of its time for 65,794 points).  Those points take
// 245 us with the addition of the groups (2,041 us grid by grid), 65,794 points
// on d = 3, level 9 122 us (737), 200,000 on d = 2, level 8 71 us (199).  The place in the cell is tabulated per axis and level
// on chip, once a point; the axes with one node (a grid of few listed axes has
// few corners) give one factor for a run of groups.
template <int D>
__global__ void __launch_bounds__(128) combine_eval_kernel(const __grid_constant__ CombinePlan C, const GridInfo *grids,
                                                           const int *levels, OpParams op, const double *M, int n_pts,
                                                           const double *pts, double *dst)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int k = blockIdx.x * blockDim.x + threadIdx.x, L = C.l_max;
    if (k >= n_pts) return;  // (no barrier below: every thread reads its own columns)
    double *place = reinterpret_cast<double *>(smem) + threadIdx.x;
    int *cell = reinterpret_cast<int *>(smem + (size_t)D * L * 128 * 8) + threadIdx.x;
    double one[D];
#pragma unroll
    for (int i = 0; i < D; ++i) {
        // position in units of the domain (see combine_kernel); the cell of
        // level lam is that of level L shifted down.  Outside the box the
        // boundary cell's linear piece is continued.
        const double xr = (pts[(long long)k * D + i] - op.lo[i]) / ldexp(grids[0].h[i], levels[i]);
        const double c = floor(ldexp(xr, L));
        const int top = (1 << L) - 1;
        const int fine = c < 0.0 ? 0 : c > (double)top ? top : (int)c;
        cell[i * 128] = fine;
        double f = xr;  // place in the cell of level lam, from that of the level before
        for (int lam = 1; lam <= L; ++lam) {
            const bool right = (fine >> (L - lam)) & 1;
            f = fma(2.0, f, right ? -1.0 : 0.0);
            place[(i * L + lam - 1) * 128] = f;
            if (lam == 1) one[i] = right ? 1.0 - f : f;
        }
    }
    double acc = 0.0;
    for (int q = 0; q < C.n_runs; ++q) {
        const CombineRun R = C.runs[q];
        double w = 1.0, v;
#pragma unroll
        for (int i = 0; i < D; ++i)
            if (!((R.mask >> i) & 1)) w *= one[i];
        switch (__popc(R.mask)) {
        case 0: v = run_value<0>(C, R, M, place, cell); break;
        case 1: v = run_value<1>(C, R, M, place, cell); break;
        case 2: if constexpr (D >= 2) v = run_value<2>(C, R, M, place, cell); break;
        case 3: if constexpr (D >= 3) v = run_value<3>(C, R, M, place, cell); break;
        case 4: if constexpr (D >= 4) v = run_value<4>(C, R, M, place, cell); break;
        case 5: if constexpr (D >= 5) v = run_value<5>(C, R, M, place, cell); break;
        default: if constexpr (D >= 6) v = run_value<6>(C, R, M, place, cell); break;
        }
        acc = fma(w, v, acc);
    }
    dst[(long long)blockIdx.y * n_pts + k] = acc;
}

size_t combine_eval_smem(int d, int l_max) { return (size_t)d * 128 * (8 * l_max + 4); }

cudaError_t combine_init(size_t max_smem)
{
    const void *k[] = {(const void *)combine_eval_kernel<1>, (const void *)combine_eval_kernel<2>,
                       (const void *)combine_eval_kernel<3>, (const void *)combine_eval_kernel<4>,
                       (const void *)combine_eval_kernel<5>, (const void *)combine_eval_kernel<6>};
    for (const void *f : k) {
        const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_smem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_combine_merged(const CombinePlan &C, const GridInfo *grids, const int *levels, const OpParams &op,
                                  const double *u, double *M, int n_pts, const double *pts, double *out, int n_chunks,
                                  double *part, cudaStream_t s)
{
    // (the chunks' sums, one or more, are added by a launch of their own)
    if (n_chunks < 1 || !part) return cudaErrorInvalidValue;
    merge_kernel<<<(unsigned)C.n_pieces, 256, 0, s>>>(C, u, M);
    const dim3 grid((unsigned)((n_pts + 127) / 128), (unsigned)n_chunks);
    const size_t smem = combine_eval_smem(op.d, C.l_max);
    switch (op.d) {
#define PIT_EVAL(D) \
    case D: combine_eval_kernel<D><<<grid, 128, smem, s>>>(C, grids, levels, op, M, n_pts, pts, part); break;
        PIT_EVAL(1) PIT_EVAL(2) PIT_EVAL(3) PIT_EVAL(4) PIT_EVAL(5) PIT_EVAL(6)
#undef PIT_EVAL
    default: return cudaErrorInvalidValue;
    }
    combine_sum_kernel<<<(n_pts + 127) / 128, 128, 0, s>>>(part, n_chunks, n_pts, out);
    return cudaGetLastError();
}

// resid[j*G + g] = ||a_j - b_j||_2 over grid g (one CTA per (j, g), fixed-order
// reduction).
__global__ void resid_norm_kernel(const GridInfo *grids, int G, const double *a, long long a_stride,
                                  const double *b, long long b_stride, const int *active, double *resid)
{
    const int g = blockIdx.x % G, j = blockIdx.x / G;
    if (active && !active[g]) return;
    const GridInfo GI = grids[g];
    const double *aj = a + (long long)j * a_stride + GI.off;
    const double *bj = b + (long long)j * b_stride + GI.off;
    double s = 0.0;
    for (int t = threadIdx.x; t < GI.n; t += blockDim.x) {
        const double r = aj[t] - bj[t];
        s += r * r;
    }
    __shared__ double red[32];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double tot = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
        resid[(long long)j * G + g] = sqrt(tot);
    }
}

cudaError_t launch_resid_norms(const GridInfo *grids, int G, long long ntot, int nb, const double *a,
                               long long a_stride, const double *b, long long b_stride, const int *active,
                               double *resid, cudaStream_t s)
{
    (void)ntot;
    const long long blocks = (long long)nb * G;
    if (blocks == 0) return cudaSuccess;
    resid_norm_kernel<<<(unsigned)blocks, 256, 0, s>>>(grids, G, a, a_stride, b, b_stride, active, resid);
    return cudaGetLastError();
}

// out_k = x_k + y_k on the active grids of nb consecutive states.
__global__ void add_states_kernel(const GridInfo *grids, int G, long long ntot, const double *x, const double *y,
                                  double *out, const int *active)
{
    const int g = blockIdx.x % G, k = blockIdx.x / G;
    if (active && !active[g]) return;
    const GridInfo GI = grids[g];
    const long long o = (long long)k * ntot + GI.off;
    for (int j = threadIdx.x; j < GI.n; j += blockDim.x) out[o + j] = x[o + j] + y[o + j];
}

cudaError_t launch_add_states(const GridInfo *grids, int G, long long ntot, int nb, const double *x, const double *y,
                              double *out, const int *active, cudaStream_t s)
{
    const long long blocks = (long long)nb * G;
    if (blocks == 0) return cudaSuccess;
    add_states_kernel<<<(unsigned)blocks, 256, 0, s>>>(grids, G, ntot, x, y, out, active);
    return cudaGetLastError();
}

__global__ void resid_max_kernel(int G, int nb, const double *resid, const int *active, double *rmax)
{
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= G) return;
    if (active && !active[g]) return;
    double m = 0.0;
    for (int j = 0; j < nb; ++j) {
        const double r = resid[(long long)j * G + g];
        if (r > m || r != r) m = r;
        if (m != m) break;
    }
    rmax[g] = m;
}

cudaError_t launch_resid_max(int G, int nb, const double *resid, const int *active, double *rmax, cudaStream_t s)
{
    resid_max_kernel<<<(G + 127) / 128, 128, 0, s>>>(G, nb, resid, active, rmax);
    return cudaGetLastError();
}

}  // namespace pit
