// Multi-step backward-Euler propagator of the constant-coefficient heat
// operator with a direct FP32 solve in place of CG: the same steps, precision
// forms and stopping rules as steps_kernel (pit_phi.cuh), one CTA per item.
//
// A = I + dt L is a Kronecker sum of 1-D second differences with zero
// Dirichlet values, so the discrete sine transform (DST-I) along an axis
// diagonalises that axis' part.  A solve transforms every axis but the longest
// one, solves the remaining independent systems along the longest axis and
// transforms back: at most 2 de - 1 passes over the vector (de the axes with
// more than one node; two short axes share one), each with one barrier and no
// reduction.  On the component grids
// of the combination technique the other axes are short (at most 31 nodes up
// to level 10 in two dimensions, 15 on most grids), so a transform is a few
// multiplications a node, done line by line in registers.
//
// Why: plain CG on these grids (dt / h^2 of 0.01 to 1, condition number 1.2 to
// 5) needs four to seven iterations of about 80 instructions a node for the
// 1e-6 that a refinement asks for, and the refinement kernel spent over
// two thirds of its instructions there (640 a node and step on heat6d); the
// direct solve takes about 100.  It also needs no Krylov vectors: 30 bytes a
// node on chip instead of 50, so two CTAs share an SM where one did.
//
// What the solve returns is only trusted through the residual that the forms
// measure after it, as before (in FP64 or FP32 pairs).  The FP32 form keeps CG:
// its tolerances (1e-2 for coarse corrections) are far looser than a direct
// solve, and the corrections would differ from those of the other operators.
#pragma once

#include "pit_phi.cuh"

namespace pit {

// ----------------------------------------------------------------------------
// DST-I of N = 2^l - 1 values, X_j = sum_k v_k sin(pi j k / (N + 1)) (its own
// inverse up to the factor 2 / (N + 1)).  Folding the line about its middle
// separates odd from even outputs; the even ones are a DST-I of half the
// length: (N + 1)^2 / 4 + (N + 1)^2 / 16 + .. multiplications instead of N^2.
constexpr double cx_sin(double x)  // Taylor series, |x| <= pi / 2
{
    double t = x, s = x;
    for (int k = 1; k < 24; ++k) {
        t *= -x * x / (double)((2 * k) * (2 * k + 1));
        s += t;
    }
    return s;
}
constexpr float cx_sinpi(int num, int den)  // sin(pi num / den)
{
    int m = num % (2 * den);
    double sg = 1.0;
    if (m >= den) {
        m -= den;
        sg = -1.0;
    }
    if (2 * m > den) m = den - m;
    return (float)(sg * cx_sin(3.14159265358979323846 * m / den));
}
template <int M>
struct DstTab {
    float c[M + 1][M + 1];
    constexpr DstTab() : c()
    {
        for (int i = 0; i <= M; ++i)
            for (int k = 0; k <= M; ++k) c[i][k] = cx_sinpi((2 * i + 1) * (k + 1), 2 * M + 2);
    }
};
static __constant__ DstTab<1> dst_tab3 = DstTab<1>();
static __constant__ DstTab<3> dst_tab7 = DstTab<3>();
static __constant__ DstTab<7> dst_tab15 = DstTab<7>();
static __constant__ DstTab<15> dst_tab31 = DstTab<15>();
template <int N>
__device__ __forceinline__ const auto &dst_tab()
{
    if constexpr (N == 3) return dst_tab3;
    else if constexpr (N == 7) return dst_tab7;
    else if constexpr (N == 15) return dst_tab15;
    else return dst_tab31;
}
template <int N>
__device__ __forceinline__ void dst(float (&v)[N])
{
    if constexpr (N > 1) {
        constexpr int M = (N - 1) / 2;
        const auto &T = dst_tab<N>();
        float e[M + 1], o[M];
#pragma unroll
        for (int k = 0; k < M; ++k) {
            e[k] = v[k] + v[N - 1 - k];
            o[k] = v[k] - v[N - 1 - k];
        }
        e[M] = v[M];
#pragma unroll
        for (int i = 0; i <= M; ++i) {
            float s = e[0] * T.c[i][0];
#pragma unroll
            for (int k = 1; k <= M; ++k) s = fmaf(e[k], T.c[i][k], s);
            v[2 * i] = s;
        }
        dst<M>(o);
#pragma unroll
        for (int i = 0; i < M; ++i) v[2 * i + 1] = o[i];
    }
}

// ----------------------------------------------------------------------------
// The direct solve of one item, set up once per launch.
struct Direct {
    int n, nax;                  // nodes; transforms
    int N[PIT_D], S[PIT_D];      // transformed axis: nodes and stride
    int N2[PIT_D], S2[PIT_D];    // a second, inner one taken by the same pass (N2 = 1: none)
    int Na, Sa, nl;              // longest axis: nodes, stride, lines
    int P, L;                    // long lines (Na > 31): chunks a line, chunk length
    float norm;                  // product of 2 / (N + 1) over the transforms
    float ca;                    // dt / h^2 of the longest axis
    // tables, as offsets in floats into the dynamic shared memory
    int lam;                     // eigenvalues of the longest axis (Na <= 31)
    int base;                    // eigenvalue sum of the transformed axes, per line of the longest axis
    int sum;                     // long lines: three sums per chunk
    // words of the tables for lines of Na nodes, nl of them
    __host__ __device__ static int words(int na, int nl) { return na <= 31 ? 32 + nl : nl + 3 * (nl * (na / 8)); }
};
// One item per block; in shared memory at namespace scope, as is the vector to
// solve for, so that the solve can be a function of its own (its registers
// are not the step loop's) and still use shared-memory addresses.
static __shared__ Direct direct_s;
extern __shared__ __align__(16) unsigned char smem[];
__device__ __forceinline__ float *smem_f() { return reinterpret_cast<float *>(smem); }
// line l of an axis of N nodes and stride S starts at hi S N + lo, l = hi S + lo
// (exact for l < 2^20: l + 1/2 is at least 1 / (2 S) away from a multiple of S)
__device__ __forceinline__ int line_start(int l, int N, int S, float inv)
{
    const int hi = (int)(((float)l + 0.5f) * inv);
    return hi * S * (N - 1) + l;
}

// tab: offset of the tables
__device__ __forceinline__ void direct_setup(const GridInfo &G, const ItemConst &IC, int tab)
{
    Direct &D = direct_s;
    const int tid = threadIdx.x, nt = blockDim.x;
    int la = 0;
    for (int q = 1; q < G.de; ++q)
        if (G.N[G.ax[q]] > G.N[G.ax[la]]) la = q;
    if (tid == 0) {
        D.n = G.n;
        int nax = 0;
        float norm = 1.0f;
        for (int q = 0; q < G.de; ++q) {
            if (q == la) continue;
            const int N = G.N[G.ax[q]], S = G.S[G.ax[q]];
            norm *= 2.0f / (float)(N + 1);
            // a short axis joins an earlier pass over a short axis: 9 or 21
            // values a thread, and a barrier and a trip through shared memory
            // less each way
            int at = nax;
            for (int i = 0; i < nax; ++i)
                if (D.N2[i] == 1 && D.N[i] * N <= 21 && at == nax) at = i;
            if (at < nax) {
                D.N2[at] = N;
                D.S2[at] = S;
                continue;
            }
            D.N[nax] = N;
            D.S[nax] = S;
            D.N2[nax] = 1;
            D.S2[nax] = 0;
            ++nax;
        }
        D.nax = nax;
        D.Na = G.N[G.ax[la]];
        D.Sa = G.S[G.ax[la]];
        D.nl = G.n / D.Na;
        D.ca = IC.ch[la] + IC.cl[la];
        if (D.Na <= 31) {
            norm *= 2.0f / (float)(D.Na + 1);
            D.lam = tab;
            D.base = tab + 32;
        } else {
            D.base = tab;
            D.sum = tab + D.nl;
            int p = nt / D.nl;
            p = p < 1 ? 1 : (p > D.Na / 8 ? D.Na / 8 : p);
            D.L = (D.Na + p - 1) / p;
            D.L |= 1;  // odd: the chunks of a line start in distinct banks
            D.P = (D.Na + D.L - 1) / D.L;
        }
        D.norm = norm;
    }
    __syncthreads();
    // the axes that are not listed have one node: eigenvalue 2 dt / h^2
    const float rest = IC.rh;
    if (D.Na <= 31) {
        for (int k = tid; k < D.Na; k += nt) {
            const float s = sinpif(0.5f * (float)(k + 1) / (float)(D.Na + 1));
            smem_f()[D.lam + k] = 4.0f * D.ca * s * s;
        }
    }
    for (int l = tid; l < D.nl; l += nt) {
        const int j = line_start(l, D.Na, D.Sa, 1.0f / (float)D.Sa);
        float s = rest;
        for (int q = 0; q < G.de; ++q) {
            if (q == la) continue;
            const int ax = G.ax[q], N = G.N[ax];
            const float t = sinpif(0.5f * (float)((j / G.S[ax]) % N + 1) / (float)(N + 1));
            s += 4.0f * (IC.ch[q] + IC.cl[q]) * t * t;
        }
        smem_f()[D.base + l] = s;
    }
}

template <int N>
__device__ __forceinline__ void dst_lines(const Direct &D, float *v, int S)
{
    const int nl = D.n / N;
    const float inv = 1.0f / (float)S;
    for (int l = threadIdx.x; l < nl; l += blockDim.x) {
        float *p = v + line_start(l, N, S, inv);
        float w[N];
#pragma unroll
        for (int k = 0; k < N; ++k) w[k] = p[k * S];
        dst<N>(w);
#pragma unroll
        for (int k = 0; k < N; ++k) p[k * S] = w[k];
    }
}
// two axes at once, S2 < S1 (the inner axis' lines lie inside one step of the
// outer one)
template <int N1, int N2>
__device__ __forceinline__ void dst_slabs(const Direct &D, float *v, int S1, int S2)
{
    const int ns = D.n / (N1 * N2);
    const float inv1 = 1.0f / (float)S1, inv2 = 1.0f / (float)S2;
    for (int l = threadIdx.x; l < ns; l += blockDim.x) {
        float *p = v + line_start(line_start(l, N2, S2, inv2), N1, S1, inv1);
        float w[N1][N2];
#pragma unroll
        for (int i = 0; i < N1; ++i) {
#pragma unroll
            for (int k = 0; k < N2; ++k) w[i][k] = p[i * S1 + k * S2];
            dst<N2>(w[i]);
        }
#pragma unroll
        for (int k = 0; k < N2; ++k) {
            float c[N1];
#pragma unroll
            for (int i = 0; i < N1; ++i) c[i] = w[i][k];
            dst<N1>(c);
#pragma unroll
            for (int i = 0; i < N1; ++i) p[i * S1 + k * S2] = c[i];
        }
    }
}
// longest axis of at most 31 nodes: transform, divide by the eigenvalues, back
template <int N>
__device__ __forceinline__ void mid_lines(const Direct &D, float *v, float mul)
{
    const float *lam = smem_f() + D.lam;
    const float inv = 1.0f / (float)D.Sa;
    for (int l = threadIdx.x; l < D.nl; l += blockDim.x) {
        float *p = v + line_start(l, N, D.Sa, inv);
        const float b0 = fmaf(mul, smem_f()[D.base + l], 1.0f);
        float w[N];
#pragma unroll
        for (int k = 0; k < N; ++k) w[k] = p[k * D.Sa];
#pragma unroll 1
        for (int rep = 0; rep < 2; ++rep) {
            dst<N>(w);
            if (rep == 0) {
#pragma unroll
                for (int k = 0; k < N; ++k) w[k] *= __fdividef(D.norm, fmaf(mul, lam[k], b0));
            }
        }
#pragma unroll
        for (int k = 0; k < N; ++k) p[k * D.Sa] = w[k];
    }
}
__device__ __forceinline__ float pow_n(float r, int e)  // r^e, e >= 0
{
    float p = 1.0f;
    for (; e; e >>= 1, r *= r)
        if (e & 1) p *= r;
    return p;
}
// Longest axis of more than 31 nodes: tridiag(-c, b0 + 2c, -c) x = r on every
// line.  On the infinite line this matrix factors into (c / rho) (1 - rho S)
// (1 - rho S^-1), S the shift and rho < 1 the decay of its Green's function
// rho^|j-k| / s, s = sqrt(b0 (b0 + 4c)): a forward and a backward first-order
// recursion with one multiplication a node and no division.  The zero values
// at 0 and N + 1 are met by subtracting the two homogeneous solutions,
// alpha rho^j and beta rho^{N+1-j}, which enter as the recursions' initial
// values.  Lines are cut into chunks so that long lines keep the block busy:
// chunk sums, a short scan over the chunks by every thread, then the chunk.
__device__ __forceinline__ void long_lines(const Direct &D, float *v, float mul)
{
    const int N = D.Na, Sa = D.Sa, nl = D.nl, P = D.P, L = D.L, tasks = nl * P;
    const float inv = 1.0f / (float)Sa, invl = 1.0f / (float)nl, c = mul * D.ca;
    float *fw = smem_f() + D.sum, *bw = fw + tasks, *zs = bw + tasks;
    for (int t = threadIdx.x; t < tasks; t += blockDim.x) {
        const int q = (int)(((float)t + 0.5f) * invl), l = t - q * nl;
        const int k0 = q * L, m = min(L, N - k0);
        const float b0 = fmaf(mul, smem_f()[D.base + l], 1.0f);
        const float rho = 2.0f * c / (b0 + 2.0f * c + sqrtf(b0 * (b0 + 4.0f * c)));
        const float *p = v + line_start(l, N, Sa, inv) + k0 * Sa;
        float y = 0.0f, z = 0.0f, w = 1.0f;
        for (int k = 0; k < m; ++k) {
            const float r = p[k * Sa];
            y = fmaf(rho, y, r);  // sum of rho^{m-1-k} r_k
            z = fmaf(w, r, z);    // sum of rho^k r_k
            w *= rho;
        }
        fw[t] = y;
        bw[t] = z;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < tasks; t += blockDim.x) {
        const int q = (int)(((float)t + 0.5f) * invl), l = t - q * nl;
        const int k0 = q * L, m = min(L, N - k0);
        const float b0 = fmaf(mul, smem_f()[D.base + l], 1.0f);
        const float s = sqrtf(b0 * (b0 + 4.0f * c));
        const float rho = 2.0f * c / (b0 + 2.0f * c + s);
        const float pl = pow_n(rho, L), pz = pow_n(rho, N - (P - 1) * L), qq = pow_n(rho, N + 1);
        // w_0 s = rho sum rho^{k-1} r_k and w_{N+1} s = rho sum rho^{N-k} r_k
        float f = 0.0f, g = 0.0f, carry = 0.0f;
        for (int i = 0; i < P; ++i) {
            if (i == q) carry = f;
            f = fmaf(i == P - 1 ? pz : pl, f, fw[i * nl + l]);
            const int ib = P - 1 - i;
            g = fmaf(ib == P - 1 ? pz : pl, g, bw[ib * nl + l]);
        }
        const float den = rho / (s * (1.0f - qq * qq));
        const float alpha = (g - qq * f) * den, beta = (f - qq * g) * den;
        // y_0 that adds -alpha rho^j to the solution
        const float y0 = -alpha * c * (1.0f - rho * rho) / rho;
        float *p = v + line_start(l, N, Sa, inv) + k0 * Sa;
        float y = fmaf(pow_n(pl, q), y0, carry), z = 0.0f, w = 1.0f;
        for (int k = 0; k < m; ++k) {
            y = fmaf(rho, y, p[k * Sa]);
            p[k * Sa] = y;
            z = fmaf(w, y, z);
            w *= rho;
        }
        // (the sum of a line's first chunk is not asked for below: its place
        // takes z_{N+1}.  fw and bw are still being read by the line's other
        // threads here.)
        if (q > 0) zs[t] = z;
        // z_{N+1}: the tail rho^2 / (1 - rho^2) of y beyond the line, and -beta
        if (q == P - 1) zs[l] = (rho * y) / (1.0f - rho * rho) - beta * c / rho;
    }
    __syncthreads();
    for (int t = threadIdx.x; t < tasks; t += blockDim.x) {
        const int q = (int)(((float)t + 0.5f) * invl), l = t - q * nl;
        const int k0 = q * L, m = min(L, N - k0);
        const float b0 = fmaf(mul, smem_f()[D.base + l], 1.0f);
        const float rho = 2.0f * c / (b0 + 2.0f * c + sqrtf(b0 * (b0 + 4.0f * c)));
        const float pl = pow_n(rho, L), pz = pow_n(rho, N - (P - 1) * L), sc = rho / c * D.norm;
        float z = zs[l];
        for (int i = P - 1; i > q; --i) z = fmaf(i == P - 1 ? pz : pl, z, zs[i * nl + l]);
        float *p = v + line_start(l, N, Sa, inv) + k0 * Sa;
        for (int k = m - 1; k >= 0; --k) {
            z = fmaf(rho, z, p[k * Sa]);
            p[k * Sa] = sc * z;
        }
    }
}
// The passes that need many registers (lines of 31 values, the chunked
// recursions), v at offset voff of the shared memory.  Not inlined: together
// with the step loop's state they do not fit in 128 registers (500 bytes of
// spills inside the transforms when inlined).
static __device__ __noinline__ void wide_pass(int voff, float mul, int S)
{
    const Direct &D = direct_s;
    float *v = smem_f() + voff;
    if (S > 0) dst_lines<31>(D, v, S);
    else if (D.Na == 31) mid_lines<31>(D, v, mul);
    else long_lines(D, v, mul);
}
// v <- (I + mul dt L)^{-1} v in place (all threads; v complete on entry and, on
// return, after the caller's next barrier)
__device__ __forceinline__ void direct_solve(float *v, float mul)
{
    const Direct &D = direct_s;
#pragma unroll 1
    for (int pass = 0; pass < 2 * D.nax + 1; ++pass) {
        if (pass > 0) __syncthreads();
        if (pass == D.nax) {
            switch (D.Na) {
            case 1: if (threadIdx.x == 0) v[0] = __fdividef(v[0], 1.0f + mul * (smem_f()[D.base] + smem_f()[D.lam])); break;
            case 3: mid_lines<3>(D, v, mul); break;
            case 7: mid_lines<7>(D, v, mul); break;
            case 15: mid_lines<15>(D, v, mul); break;
            default: wide_pass((int)(v - smem_f()), mul, 0); break;
            }
        } else {
            const int i = pass < D.nax ? pass : 2 * D.nax - pass, S = D.S[i], N2 = D.N2[i];
            switch (D.N[i]) {
            case 3:
                if (N2 == 1) dst_lines<3>(D, v, S);
                else if (N2 == 3) dst_slabs<3, 3>(D, v, S, D.S2[i]);
                else dst_slabs<3, 7>(D, v, S, D.S2[i]);
                break;
            case 7:
                if (N2 == 1) dst_lines<7>(D, v, S);
                else dst_slabs<7, 3>(D, v, S, D.S2[i]);
                break;
            case 15: dst_lines<15>(D, v, S); break;
            default: wide_pass((int)(v - smem_f()), mul, S); break;
            }
        }
    }
}

// f(std::integral_constant<int, de>) for the grid's listed axes
template <class F>
__device__ __forceinline__ void by_dim(int de, F &&f)
{
    switch (de) {
    case 1: f(std::integral_constant<int, 1>{}); break;
    case 2: f(std::integral_constant<int, 2>{}); break;
    case 3: f(std::integral_constant<int, 3>{}); break;
    case 4: f(std::integral_constant<int, 4>{}); break;
    case 5: f(std::integral_constant<int, 5>{}); break;
    default: f(std::integral_constant<int, 6>{}); break;
    }
}
// stencil of I + mul dt L (mul 1 or 2, exact)
template <typename T, int D>
__device__ __forceinline__ HeatSt<T, D> heat_st(const GridInfo &G, const ItemConst &IC, const uint16_t *mask, int mul)
{
    HeatSt<T, D> H;
    H.mask = mask;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        H.S[i] = G.S[G.ax[i]];
        H.off[i] = (T)mul * (T)(sizeof(T) == 8 ? (T)IC.off[i] : (T)IC.off32[i]);
    }
    const double dg = mul == 2 ? 2.0 * IC.diag - 1.0 : IC.diag;
    H.diag = sizeof(T) == 8 ? (T)dg : mul == 2 ? (T)dg : (T)IC.diag32;
    return H;
}
template <int D>
__device__ __forceinline__ PairHeat<D> pair_st(const GridInfo &G, const ItemConst &IC, const uint16_t *mask)
{
    PairHeat<D> H;
    H.mask = mask;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        H.S[i] = G.S[G.ax[i]];
        H.ch[i] = IC.ch[i];
        H.cl[i] = IC.cl[i];
    }
    H.rh = IC.rh;
    H.rl = IC.rl;
    return H;
}

// ----------------------------------------------------------------------------
// Shared memory of one item: FP64 x, b and carried residual (MIXED) or pairs x,
// b (PAIR), unless they live in global memory (XG); FP32 vectors; neighbour
// masks; the solve's tables.
__host__ __device__ inline int direct_f64(int prec) { return prec == MIXED ? 3 : 2; }
__host__ __device__ inline int direct_f32(int prec) { return prec == MIXED ? 1 : 2; }

template <int PREC, bool XG>
__global__ void __launch_bounds__(512, 1) direct_kernel(const __grid_constant__ StepArgs a)
{
    __shared__ GridInfo GI;
    __shared__ ItemConst IC;
    __shared__ double red64[2 * 128];
    __shared__ __align__(16) float red32[2 * 128];
    for (int t = threadIdx.x; t < 256; t += blockDim.x) red32[t] = 0.0f;
    static_assert(PREC == MIXED || PREC == PAIR, "the refinement forms");
    const int item = a.item0 + (int)blockIdx.x;
    const int g = a.order[item / a.n_batch];
    const int b = item % a.n_batch;
    if (a.active && !a.active[g]) return;  // uniform over the block
    for (int t = threadIdx.x; t < (int)(sizeof(GridInfo) / 4); t += blockDim.x)
        reinterpret_cast<int *>(&GI)[t] = reinterpret_cast<const int *>(a.grids + g)[t];
    __syncthreads();
    item_const(a, GI, IC);
    __syncthreads();

    const int tid = threadIdx.x, nt = blockDim.x;
    const int n = GI.n, de = GI.de;
    const int ld = (n + 3) & ~3;
    const double dt = a.dt;
    double *s64 = reinterpret_cast<double *>(smem);
    double *x = XG ? a.xg + (long long)b * a.n_total + GI.off : s64;
    double *bvec = XG ? a.bg + (long long)b * a.n_total + GI.off : s64 + ld;
    float2 *xp = reinterpret_cast<float2 *>(x), *bp = reinterpret_cast<float2 *>(bvec);
    double *cvec = XG ? a.xg + ((long long)2 * a.n_batch + b) * a.n_total + GI.off : s64 + 2 * ld;
    // A node's 8 bytes hold c_{s-1} or, after steps from extrapolated guesses,
    // the FP32 sum q = (e_{s-1} - r_{s-2}) 2^kq_c in the first four (one access
    // type for both, so that no aliasing rule lets them pass each other).
    int2 *cw = reinterpret_cast<int2 *>(cvec);
    auto get_c = [&](int j) { const int2 v = cw[j]; return __hiloint2double(v.y, v.x); };
    auto put_c = [&](int j, double v) { cw[j] = make_int2(__double2loint(v), __double2hiint(v)); };
    auto get_q = [&](int j) { return __int_as_float(cw[j].x); };
    auto put_q = [&](int j, float v) { cw[j].x = __float_as_int(v); };
    float *f32 = reinterpret_cast<float *>(s64 + (size_t)(XG ? 0 : direct_f64(PREC)) * ld);
    uint16_t *mask = reinterpret_cast<uint16_t *>(f32 + (size_t)direct_f32(PREC) * ld);
    direct_setup(GI, IC, (int)(reinterpret_cast<float *>(mask + ld) - smem_f()));

    const double *in = a.in + (long long)b * a.in_stride + GI.off;
    const double *f0 = a.f ? a.f + (long long)b * a.f_stride + GI.off : nullptr;
    const uint16_t *gmask = a.masks + GI.off;
    Reducer<double> R64{red64, 0};
    Reducer<float, true> R32{red32, 0};
    int ks = 0;  // PAIR: the state is held times 2^ks
    if constexpr (PREC == PAIR) {
        const double *g0 = a.g ? a.g + (long long)b * a.g_stride + GI.off : nullptr;
        double acc[1] = {0.0};
        for (int j = tid; j < n; j += nt) {
            const double v = in[j];
            acc[0] += v * v;
            if (g0) acc[0] += g0[j] * g0[j];
        }
        R64.template sum<1>(acc);
        ks = scale_exp(acc[0]);
    }
    for (int j = tid; j < n; j += nt) {
        mask[j] = gmask[j];
        if constexpr (PREC == PAIR) xp[j] = split_pair(in[j], ks);
        else x[j] = in[j];
    }
    // sum over the nodes of put(j, b_j - (A x)_j), A = I + mul dt L (MIXED)
    auto residual = [&](int mul, auto &&put) -> float {
        float acc[1] = {0.0f};
        by_dim(de, [&](auto dim) {
            constexpr int D = decltype(dim)::value;
            const HeatSt<double, D> H = heat_st<double, D>(GI, IC, mask, mul);
            // (unrolled: independent nodes keep several FP64 stencil chains in
            // flight, the FP64 latency is long on GB300)
            constexpr int U = D <= 3 ? 4 : D <= 4 ? 3 : 2;
#pragma unroll U
            for (int j = tid; j < n; j += nt) {
                const float rf = put(j, H.resid(bvec[j], x, j));
                acc[0] += rf * rf;
            }
        });
        R32.template sum<1>(acc);
        return acc[0];
    };

    int status = PIT_OK, iters = 0, passes = 0;
    // (see steps_kernel for the carried residuals, the SDIRK and the
    // extrapolated steps: the algebra is the same here)
    const bool carry_ok = (f0 == nullptr) && (a.g == nullptr) && (a.guess == nullptr) && !a.sdirk && !a.ext;
    const bool carry_g = (f0 == nullptr) && (a.guess == nullptr) && !a.sdirk && !a.ext;
    const int nstage = a.sdirk ? 2 : a.ext ? 3 : 1;
    constexpr double SD_BETA = 2.4142135623730950488, SD_ALPHA = -1.4142135623730950488;
    bool have_r0 = false;
    int kr_c = 0, cst = 0, kq_c = 0, unchecked = 0;
    float rn_c = 0.0f, bb_c = 0.0f;  // PAIR
    float *rv = f32, *wv = f32 + ld;

    for (int step = 1; step <= a.nsteps; ++step) {
        const double *f = f0 ? f0 + (long long)((step - 1) / a.f_div) * a.f_step : nullptr;
        const long long sb = (long long)(step - 1);
        const double *gu = a.guess ? a.guess + (long long)b * a.guess_stride + sb * a.guess_step + GI.off : nullptr;
        const double *gs = a.g ? a.g + (long long)b * a.g_stride + sb * a.g_step + GI.off : nullptr;
        if (PREC != MIXED || !have_r0) __syncthreads();  // state complete
        if constexpr (PREC == PAIR) {
            if (gu) {
                for (int j = tid; j < n; j += nt) {
                    bp[j] = f ? pair_add(xp[j], split_pair(dt * f[j], ks)) : xp[j];
                    xp[j] = split_pair(gs ? gu[j] - gs[j] : gu[j], ks);
                }
            } else {
                for (int j = tid; j < n; j += nt) bp[j] = f ? pair_add(xp[j], split_pair(dt * f[j], ks)) : xp[j];
            }
            float rn, bb;
            if (have_r0 && bb_c >= 0x1p-20f && bb_c <= 0x1p20f) {
                // r0 = x_{s-1} - A x_{s-1}, from the last check of the previous step (in wv)
                float *t_ = rv;
                rv = wv;
                wv = t_;
                rn = rn_c;
                bb = bb_c;
                __syncthreads();  // bp complete
            } else {
                float acc[1] = {0.0f};
                for (int j = tid; j < n; j += nt) acc[0] += bp[j].x * bp[j].x;
                R32.template sum<1>(acc);  // also: bp and xp complete
                bb = acc[0];
                if (bb > 0.0f && !(bb >= 0x1p-20f && bb <= 0x1p20f)) {
                    // exact power-of-two rescale of the state
                    const int kq = scale_exp(to_f64(bb, 0));
                    const float sc = __uint_as_float((unsigned)(127 + kq) << 23);
                    for (int j = tid; j < n; j += nt) {
                        const float2 xj = xp[j], bj = bp[j];
                        xp[j] = make_float2(xj.x * sc, xj.y * sc);
                        bp[j] = make_float2(bj.x * sc, bj.y * sc);
                    }
                    bb = (bb * sc) * sc;
                    ks += kq;
                    __syncthreads();
                }
                float accf[1] = {0.0f};
                by_dim(de, [&](auto dim) {
                    constexpr int D = decltype(dim)::value;
                    const PairHeat<D> PH = pair_st<D>(GI, IC, mask);
#pragma unroll 2
                    for (int j = tid; j < n; j += nt) {
                        float xmb;
                        const float rf = PH(xp, bp, j, xmb);
                        rv[j] = rf;
                        accf[0] += rf * rf;
                    }
                });
                R32.template sum<1>(accf);
                ++passes;
                rn = accf[0];
            }
            have_r0 = false;
            const float stop2 = a.rtol2 * bb;
            int st_step = PIT_OK;
            bool carried = false;
            for (int pass = 0;; ++pass) {
                if (!(rn > stop2)) {
                    if (rn != rn) st_step = PIT_ERR_NONFINITE;
                    else if (carry_ok && pass == 0) {
                        // x unchanged: its residual is the next step's r0
                        float *t_ = rv;
                        rv = wv;
                        wv = t_;
                        rn_c = rn;
                        bb_c = bb;
                        carried = true;
                    }
                    break;
                }
                if (pass >= a.ir_maxit) { st_step = PIT_ERR_NOCONV; break; }
                // (the transforms scale linearly: a residual far below the FP32
                // range's middle is lifted first)
                const int kn = rn >= 0x1p-64f ? 0 : min(max(-scale_exp(rn), -120), 120);
                if (kn != 0) {
                    const float inv = __uint_as_float((unsigned)(127 - kn) << 23);
                    for (int j = tid; j < n; j += nt) rv[j] *= inv;
                    __syncthreads();
                }
                direct_solve(rv, 1.0f);
                ++iters;
                __syncthreads();
                const float csf = __uint_as_float((unsigned)(127 + kn) << 23);
#pragma unroll 4
                for (int j = tid; j < n; j += nt) xp[j] = pair_add(xp[j], rv[j] * csf);
                __syncthreads();  // x complete
                // check: r = b - A x; the next step's r0 = x - A x = r + (x - b)
                float accf[3] = {0.0f, 0.0f, 0.0f};
                by_dim(de, [&](auto dim) {
                    constexpr int D = decltype(dim)::value;
                    const PairHeat<D> PH = pair_st<D>(GI, IC, mask);
#pragma unroll 2
                    for (int j = tid; j < n; j += nt) {
                        float xmb;
                        const float rf = PH(xp, bp, j, xmb);
                        rv[j] = rf;
                        accf[0] += rf * rf;
                        if (carry_ok) {
                            const float cj = rf + xmb;
                            const float xf = xp[j].x;
                            wv[j] = cj;
                            accf[1] += cj * cj;
                            accf[2] += xf * xf;
                        }
                    }
                });
                R32.template sum<3>(accf);
                ++passes;
                rn = accf[0];
                if (carry_ok) {
                    rn_c = accf[1];
                    bb_c = accf[2];
                    carried = true;
                }
            }
            if (st_step > status) status = st_step;
            have_r0 = carried && st_step == PIT_OK && step < a.nsteps;
            if (gs)
                for (int j = tid; j < n; j += nt) xp[j] = pair_add(xp[j], split_pair(gs[j], ks));
        } else {
#pragma unroll 1
            for (int stage = 0; stage < nstage; ++stage) {
                const int mul = a.ext && stage == 2 ? 2 : 1;
                float rn, bb;
                int kr, kb;
                const bool carried = have_r0;
                if (carried) {
                    const int kq = kr_c;
                    const double *gp =
                        a.g ? a.g + (long long)b * a.g_stride + (long long)(step - 2) * a.g_step + GI.off : nullptr;
                    const int from =
                        !a.predict || gp ? 0 : cst == 2 && kq - kq_c <= 60 && kq_c - kq <= 60 ? 2 : cst == 1 ? 1 : 0;
                    float acc[2] = {0.0f, 0.0f};
                    if (from == 2) {
                        const float sc = scale_f(1.0f, kq - kq_c);
                        // (four nodes loaded before any is stored: in the global-state
                        // variant possibly aliasing stores would serialise the loads)
                        for (int j0 = tid; j0 < n; j0 += 4 * nt) {
                            double xo[4], bo[4];
                            float rs[4], qo[4];
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const int j = j0 + q * nt;
                                if (j < n) {
                                    xo[q] = x[j];
                                    bo[q] = bvec[j];
                                    rs[q] = rv[j];
                                    qo[q] = get_q(j);
                                }
                            }
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const int j = j0 + q * nt;
                                if (j < n) {
                                    const float r0 = fmaf(2.0f, rs[q], qo[q] * sc);
                                    const float xf = to_f32(xo[q], kq);
                                    put_q(j, -rs[q]);
                                    x[j] = fma(2.0, xo[q], -bo[q]);
                                    bvec[j] = xo[q];
                                    rv[j] = r0;
                                    acc[0] += r0 * r0;
                                    acc[1] += xf * xf;
                                }
                            }
                        }
                    } else {
#pragma unroll 2
                        for (int j = tid; j < n; j += nt) {
                            const double xo = x[j], bo = bvec[j];
                            const float rs = rv[j];
                            const double d = xo - bo;
                            const double cn = to_f64(rs, -kq) + d;
                            float r0;
                            if (from == 1) {
                                r0 = to_f32_rn(cn - get_c(j), kq) + rs;
                                x[j] = xo + d;
                                put_q(j, -rs);
                            } else {
                                r0 = to_f32_rn(cn, kq);
                                if (gp) x[j] = xo - gp[j];
                                else put_c(j, cn);
                            }
                            bvec[j] = xo;
                            rv[j] = r0;
                            const float xf = to_f32(xo, kq);
                            acc[0] += r0 * r0;
                            acc[1] += xf * xf;
                        }
                    }
                    R32.template sum<2>(acc);  // also: x, b and rv complete, cvec read
                    cst = gp ? 0 : from == 0 ? 1 : 2;
                    kq_c = kq;
                    rn = acc[0];
                    bb = acc[1];
                    kr = kb = kq;
                } else {
                    if (stage > 0 && !a.ext) {
                        for (int j = tid; j < n; j += nt) bvec[j] = SD_ALPHA * bvec[j] + SD_BETA * x[j];
                    } else if (stage == 1) {
                        for (int j = tid; j < n; j += nt) bvec[j] = x[j];
                    } else if (stage == 2) {
                        for (int j = tid; j < n; j += nt) {
                            const double un = get_c(j);
                            put_c(j, x[j]);
                            bvec[j] = un;
                        }
                    } else if (gu) {
                        for (int j = tid; j < n; j += nt) {
                            const double bj = f ? x[j] + dt * f[j] : x[j];
                            bvec[j] = bj;
                            if (a.ext) put_c(j, bj);
                            x[j] = gs ? gu[j] - gs[j] : gu[j];
                        }
                    } else {
                        for (int j = tid; j < n; j += nt) {
                            const double bj = f ? x[j] + dt * f[j] : x[j];
                            bvec[j] = bj;
                            if (a.ext) put_c(j, bj);
                        }
                    }
                    double acc[1] = {0.0};
                    for (int j = tid; j < n; j += nt) acc[0] += bvec[j] * bvec[j];
                    R64.template sum<1>(acc);  // also: bvec and x complete
                    kr = kb = scale_exp(acc[0]);
                    bb = to_f32(acc[0], 2 * kb);
                    rn = residual(mul, [&](int j, double r) {
                        const float rf = to_f32_rn(r, kr);
                        if (carry_ok) put_c(j, r);
                        rv[j] = rf;
                        return rf;
                    });
                    ++passes;
                    cst = carry_ok ? 1 : 0;
                    unchecked = -1;
                }
                have_r0 = false;
                const int kx = kb + scale_exp(bb);  // FP32 copies of this step: value 2^kx, ||b|| 2^kx in [1, 2)
                float stop2 = a.rtol2 * bb;
                int st_step = PIT_OK;
                bool accept = !carried || unchecked < 15;
                for (int pass = 0;;) {
                    if (!(rn > stop2)) {
                        if (rn != rn) st_step = PIT_ERR_NONFINITE;
                        if (st_step != PIT_OK || accept) break;
                    } else {
                        if (pass >= a.ir_maxit) { st_step = PIT_ERR_NOCONV; break; }
                        const int kn = rn >= 0x1p-64f && rn <= 0x1p64f ? 0 : min(max(-scale_exp(rn), -120), 120);
                        if (kn != 0) {
                            const float inv = __uint_as_float((unsigned)(127 - kn) << 23);
                            for (int j = tid; j < n; j += nt) rv[j] *= inv;
                            __syncthreads();
                        }
                        direct_solve(rv, (float)mul);
                        ++iters;
                        __syncthreads();
                        const double cs = pow2d(kn - kr);
                        const float cq = scale_f(1.0f, kn - kr + kq_c);
                        for (int j0 = tid; j0 < n; j0 += 4 * nt) {
                            double xv[4];
                            float ev[4], qo[4];
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const int j = j0 + q * nt;
                                if (j < n) {
                                    ev[q] = rv[j];
                                    xv[q] = x[j];
                                    if (cst == 2) qo[q] = get_q(j);
                                }
                            }
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const int j = j0 + q * nt;
                                if (j < n) {
                                    x[j] = fma(to_f64(ev[q], 0), cs, xv[q]);
                                    if (cst == 2) put_q(j, fmaf(ev[q], cq, qo[q]));
                                }
                            }
                        }
                        ++pass;
                        __syncthreads();  // x complete
                    }
                    accept = true;
                    unchecked = -1;
                    rn = residual(mul, [&](int j, double r) {
                        const float rf = to_f32_rn(r, kx);
                        rv[j] = rf;
                        return rf;
                    });
                    ++passes;
                    kr = kx;
                    stop2 = a.rtol2 * scale_f(bb, 2 * (kx - kb));
                }
                ++unchecked;  // 0 after an FP64 check
                if (st_step > status) status = st_step;
                have_r0 = carry_g && st_step == PIT_OK && step < a.nsteps;
                kr_c = kr;
            }
            // u_{n+1} = 2 U2 - U3 (the last reduction ordered every read of x)
            if (a.ext)
                for (int j = tid; j < n; j += nt) x[j] = 2.0 * get_c(j) - x[j];
            if (gs)
                for (int j = tid; j < n; j += nt) x[j] += gs[j];
        }
        // stored outputs (FP64, own nodes only)
        auto value = [&](int j) -> double {
            if constexpr (PREC == PAIR) return pair_to_f64(xp[j], ks);
            else return x[j];
        };
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

// Launchers, one translation unit per precision form.
#define PIT_DIRECT_DECL(PN)                                                                                       \
    cudaError_t direct_init_##PN(int bytes);                                                                      \
    cudaError_t direct_launch_##PN(const StepArgs &a, dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool xg);
PIT_DIRECT_DECL(mixed) PIT_DIRECT_DECL(pair)

#define PIT_DIRECT_PREC(PN, PV)                                                                                   \
    cudaError_t direct_init_##PN(int bytes)                                                                       \
    {                                                                                                             \
        const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;                                            \
        const cudaError_t e = cudaFuncSetAttribute((const void *)direct_kernel<PV, false>, attr, bytes);          \
        return e != cudaSuccess ? e : cudaFuncSetAttribute((const void *)direct_kernel<PV, true>, attr, bytes);   \
    }                                                                                                             \
    cudaError_t direct_launch_##PN(const StepArgs &a, dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool xg) \
    {                                                                                                             \
        if (xg) direct_kernel<PV, true><<<grid, block, smem, s>>>(a);                                             \
        else direct_kernel<PV, false><<<grid, block, smem, s>>>(a);                                               \
        return cudaGetLastError();                                                                                \
    }

}  // namespace pit
