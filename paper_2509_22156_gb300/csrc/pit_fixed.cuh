// The refinement of pit_direct.cuh for launches without forcing, with the state
// held as 64-bit integers times a power of two and its residual formed by
// integer arithmetic.
//
// GB300's FP64 unit takes 16 clocks of an SM for one warp instruction, its
// integer pipes a quarter of a clock, so the FP64 check b - A x (2 de + 1
// operations a node) bounded the refinement: 45 % of the pipe busy on average,
// all of it while a block's check runs.  As integers the same residual is
//     r = (b - x) - sum_i c_i (2 x_j - x_{j-e_i} - x_{j+e_i}),  c_i = dt / h_i^2,
// with exact sums and differences and products by 60-bit fractions: per axis
// four additions and three 32 x 32 + 64-bit multiply-adds.
//
// Accuracy: ||x||_2 2^k lies in [2^52, 2^57), so a unit is at most 2^-52 of the
// norm (FP64 holds 2^-53 of every value); |x_j| <= ||x||_2, the extrapolated
// guess 2 x_s - x_{s-1} is below 3 2^57 as long as both states are below 2^57, a
// second difference below 2^60.6, and with E chosen so
// that sum c_i 2^-E < 2 the sum of products stays below 2^62.  Dropped bits and
// the final shifts leave the residual off by a few units (at most 12; times 2^E
// for large steps): 8 n^{1/2} 2^-53 max(1, sum c_i) of the norm, and the host
// takes this form only where that is below a quarter of the requested
// tolerance, the FP64 check elsewhere.  A state that has decayed by more than
// four bits is shifted up again before its next step, as far as the state before
// it, which the extrapolated guess contains, leaves room; where one step has
// shrunk the state to less than an eighth, that would leave it too few bits, and
// the step starts from x_s instead.
#pragma once

#include "pit_direct.cuh"

namespace pit {

struct FixConst {
    int hi[PIT_D + 1], lo[PIT_D + 1];  // c_i 2^{-E-1} = (hi 2^29 + lo) 2^-60 of the listed axes; [D]: sum of the others
    int E;
};
__device__ __forceinline__ void fix_const(const StepArgs &a, const GridInfo &G, FixConst &F)
{
    if (threadIdx.x < 7) {
        const double sum = a.dt * G.sum2, rest = a.dt * G.rest2;
        // (every coefficient, and the sum of any of them, is below 2^{e+1}: hi < 2^31)
        const int e = max(0, (int)((__double2hiint(sum) >> 20) & 0x7ff) - 1023);  // sum 2^-e < 2
        const int q = threadIdx.x;
        const double c = q < G.de ? a.dt * G.ih2[G.ax[q]] : q == G.de ? rest : 0.0;
        const long long C = (long long)(c * pow2d(59 - e));
        F.hi[q] = (int)(C >> 29);
        F.lo[q] = (int)(C & ((1 << 29) - 1));
        if (q == 0) F.E = e;
    }
}

// r rounded to FP32 (to within an ulp and a half)
__device__ __forceinline__ float fix_f32(long long r)
{
    const int lo = (int)r, hi = (int)((r - lo) >> 32);
    return fmaf((float)hi, 4294967296.0f, (float)lo);
}
// rv = r in FP32 and this thread's part of its squared norm, r = b - A x in units
// of 2^E; keep: r also goes to cw as an integer.  The vectors are on chip at the
// places of fixed_kernel, or (XG) x, b and cw in global memory.  A function of
// its own, like the wide transforms, for its registers.
static __shared__ FixConst fix_s;
static __shared__ GridInfo fix_g;
template <int D, bool XG>
static __device__ __noinline__ float fix_residual(const long long *xg, const long long *bg, int2 *cg, bool keep)
{
    const int n = fix_g.n, ld = (n + 3) & ~3;
    const long long *x = XG ? xg : reinterpret_cast<const long long *>(smem);
    const long long *b = XG ? bg : reinterpret_cast<const long long *>(smem) + ld;
    int2 *cw = XG ? cg : reinterpret_cast<int2 *>(smem) + 2 * ld;
    float *rv = reinterpret_cast<float *>(reinterpret_cast<long long *>(smem) + (size_t)(XG ? 0 : 3) * ld);
    const uint16_t *mask = reinterpret_cast<const uint16_t *>(rv + ld);
    int S[D], ch[D], cl[D];
#pragma unroll
    for (int i = 0; i < D; ++i) {
        S[i] = fix_g.S[fix_g.ax[i]];
        ch[i] = fix_s.hi[i];
        cl[i] = fix_s.lo[i];
    }
    const int rh = fix_s.hi[D], rl = fix_s.lo[D], E = fix_s.E;
    float acc = 0.0f;
#pragma unroll 2
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        const unsigned mk = mask[j];
        const long long xj = x[j], t0 = 2 * xj;
        long long A = 0, B = 0;
#pragma unroll
        for (int i = 0; i < D; ++i) {
            const long long xm = ((mk >> (2 * i)) & 1u) ? x[j - S[i]] : 0;
            const long long xp = ((mk >> (2 * i + 1)) & 1u) ? x[j + S[i]] : 0;
            const long long t = 4 * (t0 - xm - xp);
            const int th = (int)(t >> 32), tl = (int)((unsigned)t >> 3);
            A += (long long)th * ch[i];
            B += (long long)th * cl[i];
            B += (long long)tl * ch[i];
        }
        if (rh | rl) {
            // an axis of one node has zero neighbours: its second difference is 2 x_j
            const long long t = 4 * t0;
            const int th = (int)(t >> 32), tl = (int)((unsigned)t >> 3);
            A += (long long)th * rh;
            B += (long long)th * rl;
            B += (long long)tl * rh;
        }
        // c t 2^-E = th hi + (th lo + (tl / 8) hi) 2^-29, th and tl the halves of 4 t
        const long long r = ((b[j] - xj) >> E) - A - (B >> 29);
        const float rf = fix_f32(r);
        rv[j] = rf;
        if (keep) cw[j] = make_int2((int)r, (int)(r >> 32));
        acc += rf * rf;
    }
    return acc;
}
// e rounded to an integer, |e| < 2^59
__device__ __forceinline__ long long fix_i64(float e)
{
    const int h = __float2int_rn(e * 0x1p-28f);
    const int l = __float2int_rn(fmaf((float)h, -0x1p28f, e));
    return ((long long)h << 28) + l;
}

template <bool XG>
__global__ void __launch_bounds__(512, 1) fixed_kernel(const __grid_constant__ StepArgs a)
{
    GridInfo &GI = fix_g;
    __shared__ ItemConst IC;
    FixConst &FC = fix_s;
    __shared__ double red64[2 * 128];
    __shared__ __align__(16) float red32[2 * 128];
    for (int t = threadIdx.x; t < 256; t += blockDim.x) red32[t] = 0.0f;
    const int item = a.item0 + (int)blockIdx.x;
    const int g = a.order[item / a.n_batch];
    const int b = item % a.n_batch;
    if (a.active && !a.active[g]) return;  // uniform over the block
    for (int t = threadIdx.x; t < (int)(sizeof(GridInfo) / 4); t += blockDim.x)
        reinterpret_cast<int *>(&GI)[t] = reinterpret_cast<const int *>(a.grids + g)[t];
    __syncthreads();
    item_const(a, GI, IC);
    fix_const(a, GI, FC);
    __syncthreads();

    const int tid = threadIdx.x, nt = blockDim.x;
    const int n = GI.n, ld = (n + 3) & ~3;
    long long *s64 = reinterpret_cast<long long *>(smem);
    long long *x = XG ? reinterpret_cast<long long *>(a.xg) + (long long)b * a.n_total + GI.off : s64;
    long long *bv = XG ? reinterpret_cast<long long *>(a.bg) + (long long)b * a.n_total + GI.off : s64 + ld;
    // c_{s-1} as an integer or, in its first four bytes, the FP32 sum q (see
    // direct_kernel)
    int2 *cw = reinterpret_cast<int2 *>(
        XG ? reinterpret_cast<long long *>(a.xg) + ((long long)2 * a.n_batch + b) * a.n_total + GI.off : s64 + 2 * ld);
    float *rv = reinterpret_cast<float *>(s64 + (size_t)(XG ? 0 : 3) * ld);
    uint16_t *mask = reinterpret_cast<uint16_t *>(rv + ld);
    direct_setup(GI, IC, (int)(reinterpret_cast<float *>(mask + ld) - smem_f()));
    Reducer<double> R64{red64, 0};
    Reducer<float, true> R32{red32, 0};

    const double *in = a.in + (long long)b * a.in_stride + GI.off;
    const uint16_t *gmask = a.masks + GI.off;
    double ss[1] = {0.0};
    for (int j = tid; j < n; j += nt) {
        const double v = in[j];
        ss[0] += v * v;
        mask[j] = gmask[j];
    }
    R64.template sum<1>(ss);
    const bool bad = !(ss[0] <= 1.7976931348623157e308);  // (infinite or NaN)
    int up0 = 0;
    if (ss[0] < 0x1p-900) {
        // (squares at the double range's other end: the norm of the state times 2^500)
        up0 = 500;
        ss[0] = 0.0;
        for (int j = tid; j < n; j += nt) {
            const double v = in[j] * 0x1p500;
            ss[0] += v * v;
        }
        R64.template sum<1>(ss);
    }
    const int E = FC.E;
    int k = min(max(scale_exp(ss[0]) + 56 + up0, -900), 900);  // the state is held times 2^k
    {
        const double up = pow2d(k);
        for (int j = tid; j < n; j += nt) x[j] = bad ? 0 : __double2ll_rn(in[j] * up);
    }
    const float e2 = __uint_as_float((unsigned)(127 + E) << 23);           // a residual unit in units of x
    const float b2r = __uint_as_float((unsigned)(127 + 64 - 2 * E) << 23);  // (2^32 units of x)^2 in residual units^2
    auto residual = [&](bool keep) -> float {
        float acc[1];
        switch (GI.de) {
        case 1: acc[0] = fix_residual<1, XG>(x, bv, cw, keep); break;
        case 2: acc[0] = fix_residual<2, XG>(x, bv, cw, keep); break;
        case 3: acc[0] = fix_residual<3, XG>(x, bv, cw, keep); break;
        case 4: acc[0] = fix_residual<4, XG>(x, bv, cw, keep); break;
        case 5: acc[0] = fix_residual<5, XG>(x, bv, cw, keep); break;
        default: acc[0] = fix_residual<6, XG>(x, bv, cw, keep); break;
        }
        R32.template sum<1>(acc);
        return acc[0];
    };
    // The right-hand side's norm has fallen below 2^53 units: shifts the state
    // back up until the norm, or the larger one whose square is top, is at 2^56
    // (v: ||r||^2 and ||b||^2, updated; everything a step keeps is scaled with
    // it).  Own nodes; a barrier on both sides.
    auto rescale = [&](float (&v)[2], int cst, float top) {
        // (below 2^45 the norm's 2^32-unit parts say too little: eight bits at a
        // time, at most the width of the state)
        for (int it = 0; it < 8 && v[1] < 0x1p42f && k < 900 && (v[1] > 0.0f || v[0] > 0.0f); ++it) {
            const bool coarse = v[1] < 0x1p26f;
            const int up = min(coarse ? 8 : scale_exp(fmaxf(v[1], top)) + 24, 900 - k);
            if (up <= 0) break;
            const float sc = __uint_as_float((unsigned)(127 + up) << 23);
            float bb[1] = {0.0f};
            __syncthreads();
            for (int j = tid; j < n; j += nt) {
                x[j] <<= up;
                const long long bj = bv[j] << up;
                bv[j] = bj;
                rv[j] *= sc;
                if (cst == 2) cw[j].x = __float_as_int(__int_as_float(cw[j].x) * sc);
                const float xf = (float)(int)(bj >> 32);
                bb[0] += xf * xf;
            }
            k += up;
            R32.template sum<1>(bb);
            v[0] = (v[0] * sc) * sc;
            v[1] = bb[0];
            top = (top * sc) * sc;
        }
    };

    int status = bad ? PIT_ERR_NONFINITE : PIT_OK, iters = 0, passes = 0;
    bool have_r0 = false;
    int cst = 0, unchecked = 0;  // what cw holds: 0 nothing, 1 c, 2 q
    float b_last = 0.0f;         // ||x_{s-1}||^2 in 2^32 units
    for (int step = 1; step <= a.nsteps; ++step) {
        if (!have_r0) __syncthreads();  // state complete
        if (!bad) {
            float acc[2] = {0.0f, 0.0f};  // ||r||^2 in residual units, ||b||^2 in 2^32 units of x
            bool carried = have_r0;
            if (carried) {
                const int from = !a.predict ? 0 : cst;
                if (from == 2) {
                    for (int j0 = tid; j0 < n; j0 += 4 * nt) {
                        long long xo[4], bo[4];
                        float rs[4], qo[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int j = j0 + q * nt;
                            if (j < n) {
                                xo[q] = x[j];
                                bo[q] = bv[j];
                                rs[q] = rv[j];
                                qo[q] = __int_as_float(cw[j].x);
                            }
                        }
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int j = j0 + q * nt;
                            if (j < n) {
                                const float r0 = fmaf(2.0f, rs[q], qo[q]), xf = (float)(int)(xo[q] >> 32);
                                cw[j].x = __float_as_int(-rs[q]);
                                x[j] = 2 * xo[q] - bo[q];
                                bv[j] = xo[q];
                                rv[j] = r0;
                                acc[0] += r0 * r0;
                                acc[1] += xf * xf;
                            }
                        }
                    }
                } else {
                    for (int j = tid; j < n; j += nt) {
                        const long long xo = x[j], d = xo - bv[j];
                        const float rs = rv[j];
                        float r0;
                        if (from == 1) {
                            const int2 c = cw[j];
                            r0 = fmaf(2.0f, rs, fix_f32((d >> E) - (((long long)c.y << 32) | (unsigned)c.x)));
                            cw[j].x = __float_as_int(-rs);
                            x[j] = xo + d;
                        } else {
                            r0 = fix_f32(d >> E) + rs;
                        }
                        bv[j] = xo;
                        rv[j] = r0;
                        const float xf = (float)(int)(xo >> 32);
                        acc[0] += r0 * r0;
                        acc[1] += xf * xf;
                    }
                }
                R32.template sum<2>(acc);
                cst = from == 0 ? 0 : 2;
                if (acc[1] < 0x1p42f) {
                    if (cst == 2 && b_last > 0x1p6f * acc[1]) {  // shrunk to less than an eighth
                        for (int j = tid; j < n; j += nt) x[j] = bv[j];
                        carried = false;
                        acc[1] = 0.0f;
                    } else {
                        rescale(acc, cst, cst == 2 ? b_last : 0.0f);
                    }
                }
            }
            if (!carried) {
                for (int j = tid; j < n; j += nt) {
                    const long long xo = x[j];
                    bv[j] = xo;
                    const float xf = (float)(int)(xo >> 32);
                    acc[1] += xf * xf;
                }
                float bb[1] = {acc[1]};
                R32.template sum<1>(bb);
                acc[0] = 1.0f;
                acc[1] = bb[0];
                if (acc[1] < 0x1p42f) {
                    rescale(acc, 0, 0.0f);  // (rv is scaled too, and overwritten next)
                    __syncthreads();
                }
                acc[0] = residual(true);
                ++passes;
                cst = 1;
                unchecked = -1;
            }
            float rn = acc[0];
            const float bb = b_last = acc[1];
            have_r0 = false;
            float stop2 = a.rtol2 * bb * b2r;
            int st_step = PIT_OK;
            bool accept = !carried || unchecked < 15;
            for (int pass = 0;;) {
                if (!(rn > stop2)) {
                    if (rn != rn) st_step = PIT_ERR_NONFINITE;
                    if (st_step != PIT_OK || accept) break;
                } else {
                    if (pass >= a.ir_maxit) { st_step = PIT_ERR_NOCONV; break; }
                    direct_solve(rv, 1.0f);
                    ++iters;
                    __syncthreads();
                    for (int j0 = tid; j0 < n; j0 += 4 * nt) {
                        long long xv[4];
                        float ev[4], qo[4];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int j = j0 + q * nt;
                            if (j < n) {
                                ev[q] = rv[j];
                                xv[q] = x[j];
                                if (cst == 2) qo[q] = __int_as_float(cw[j].x);
                            }
                        }
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            const int j = j0 + q * nt;
                            if (j < n) {
                                x[j] = xv[q] + fix_i64(ev[q] * e2);
                                if (cst == 2) cw[j].x = __float_as_int(qo[q] + ev[q]);
                            }
                        }
                    }
                    ++pass;
                    __syncthreads();  // x complete
                }
                accept = true;
                unchecked = -1;
                rn = residual(false);
                ++passes;
            }
            ++unchecked;  // 0 after a check
            if (st_step > status) status = st_step;
            have_r0 = st_step == PIT_OK && step < a.nsteps;
        }
        // stored outputs (FP64, own nodes only)
        const double dn = pow2d(-k);
        auto value = [&](int j) -> double { return bad ? in[j] : (double)x[j] * dn; };
        const long long sb = (long long)(step - 1);
        const double *hs = a.hs ? a.hs + (long long)b * a.hs_stride + sb * a.hs_step + GI.off : nullptr;
        if (step < a.nsteps) {
            if (a.out_steps) {
                double *os = a.out_steps + (long long)b * a.os_stride + sb * a.os_step + GI.off;
                for (int j = tid; j < n; j += nt) os[j] = hs ? value(j) + hs[j] : value(j);
            }
        } else {
            double *ol = a.out_last + (long long)b * a.ol_stride + GI.off;
            const double *h = a.h ? a.h + (long long)b * a.h_stride + GI.off : nullptr;
            const double *cmp = a.cmp ? a.cmp + (long long)b * a.cmp_stride + GI.off : nullptr;
            double acc[1] = {0.0};
            for (int j = tid; j < n; j += nt) {
                const double xj = value(j);
                if (cmp) {
                    const double dlt = xj - cmp[j];
                    acc[0] += dlt * dlt;
                }
                ol[j] = a.out_scale * xj + (h ? a.out_hscale * h[j] : 0.0) + (hs ? hs[j] : 0.0);
            }
            if (cmp) {
                R64.template sum<1>(acc);
                if (tid == 0) a.norms[(long long)b * a.n_grids + g] = sqrt(acc[0]);
            }
        }
    }
    if (a.inexact && status == PIT_ERR_NOCONV) status = PIT_OK;  // fixed-iteration (inexact) solves
    if (tid == 0 && a.stats) {
        atomicAdd(&a.stats->sum_iters, (unsigned long long)iters);
        atomicAdd(&a.stats->items, (unsigned long long)a.nsteps);
        atomicAdd(&a.stats->point_iters, (unsigned long long)iters * (unsigned long long)n);
        atomicAdd(&a.stats->point_passes, (unsigned long long)passes * (unsigned long long)n);
        atomicAdd(&a.stats->point_steps, (unsigned long long)a.nsteps * (unsigned long long)n);
        atomicMax(&a.stats->max_iters, iters);
        atomicMax(&a.stats->max_refine, passes);
        if (status != PIT_OK) {
            atomicAdd(&a.stats->n_failed, 1);
            atomicMax(&a.stats->worst, status);
        }
    }
}

cudaError_t fixed_init(int bytes);
cudaError_t fixed_launch(const StepArgs &a, dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool xg);

}  // namespace pit
