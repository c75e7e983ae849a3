// Recombination of the component-grid solutions (Sec. 2.2.2): the operator
// Q = H^{-1} Qbar H of Eq. "overall_combination_operator".  H hierarchizes
// every grid's nodal values (surplus of each node over the linear
// interpolant of its two hierarchical parents along every axis), Qbar gives
// every node the sum over all grids that share the node of their
// combination coefficient times their surplus there (Eq.
// "recombination_operator"), and H^{-1} dehierarchizes.  The result on grid
// l is the nodal interpolant of the combined solution on Omega_l.
//
// The surpluses of the sparse grid are stored once, block by block: one block
// per hierarchical increment lam (a level multi-index that some grid
// contains), its 2^{|lam|_1 - d} nodes in C order.  A grid's own surpluses are
// stored in the same block order, so that the sum over grids reads whole
// blocks.  Three launches:
//   hier_kernel    one CTA per grid: values on chip, hierarchized along every
//                  axis, written block by block
//   gather_kernel  one CTA per block (or 256 nodes of it): the grids that
//                  contain the block, in slices of the list when the block has
//                  fewer nodes than the CTA has threads; slices are added in
//                  order (deterministic, no atomics)
//   dehier_kernel  one CTA per grid: the blocks' sums on chip, dehierarchized
//
// What bounds it: the FP64 unit (a surplus is one or two FP64 operations an
// axis, and the unit does two lanes a clock and SM), then memory.  Lines of up
// to 15 nodes are transformed in registers: all levels in one pass, and where a
// parent is on the boundary the operation is not there (8 operations for a
// line of 7 instead of 14).  heat6d level 10 (11.9 M nodes, 4,921 grids):
// 3,608 us before (a scan of every node for every level, and one thread that
// added all 4,921 grids of the coarsest increment), 479 us now.
#include "pit_internal.cuh"

namespace pit {

namespace {

// j / N for 0 <= j < 2^20 by a multiplication (inv = 1 / N; j + 1/2 is at least
// 1 / (2 N) away from a multiple of N, more than the product's rounding), else
// by the division.
__device__ __forceinline__ int quot(int j, int N, float inv, bool small)
{
    return small ? (int)(((float)j + 0.5f) * inv) : j / N;
}

// Levels of a line of N = 2^l - 1 nodes held in registers.  Node J (1-based)
// with t trailing zero bits has the parents J -/+ 2^t (zero on the boundary).
template <int N>
__device__ __forceinline__ void hier_line(double (&v)[N])
{
    // finest level first: parents still nodal
#pragma unroll
    for (int t = 0; (2 << t) <= N; ++t)
#pragma unroll
        for (int J = 1 << t; J <= N; J += 2 << t) {
            const int a = J - (1 << t), b = J + (1 << t);
            if (a >= 1 && b <= N) v[J - 1] = fma(-0.5, v[a - 1] + v[b - 1], v[J - 1]);
            else if (a >= 1) v[J - 1] = fma(-0.5, v[a - 1], v[J - 1]);
            else if (b <= N) v[J - 1] = fma(-0.5, v[b - 1], v[J - 1]);
        }
}
template <int N>
__device__ __forceinline__ void dehier_line(double (&v)[N])
{
    // coarsest level first: parents already nodal
#pragma unroll
    for (int st = (N + 1) / 2; st >= 1; st /= 2)
#pragma unroll
        for (int J = st; J <= N; J += 2 * st) {
            const int a = J - st, b = J + st;
            if (a >= 1 && b <= N) v[J - 1] = fma(0.5, v[a - 1] + v[b - 1], v[J - 1]);
            else if (a >= 1) v[J - 1] = fma(0.5, v[a - 1], v[J - 1]);
            else if (b <= N) v[J - 1] = fma(0.5, v[b - 1], v[J - 1]);
        }
}
template <int N, bool BACK>
__device__ __forceinline__ void lines_pass(double *v, int n, int S)
{
    const float inv = 1.0f / (float)S;
    const bool small = n < (1 << 20);
    for (int l = threadIdx.x; l < n / N; l += blockDim.x) {
        double *p = v + (quot(l, S, inv, small) * S * (N - 1) + l);
        double w[N];
#pragma unroll
        for (int k = 0; k < N; ++k) w[k] = p[k * S];
        if constexpr (BACK) dehier_line<N>(w);
        else hier_line<N>(w);
#pragma unroll
        for (int k = 0; k < N; ++k) p[k * S] = w[k];
    }
}
// longer lines: level by level with a barrier, touching the level's nodes only
template <bool BACK>
__device__ __forceinline__ void levels_pass(double *v, int n, int N, int S)
{
    const int lev = 31 - __clz(N + 1);
    const double h = BACK ? 0.5 : -0.5;
    const float inv = 1.0f / (float)S;
    const bool small = n < (1 << 20);
    for (int i = 0; i < lev; ++i) {
        const int t = BACK ? lev - 1 - i : i, sh = lev - 1 - t;  // 2^sh nodes of this level a line
        if (i) __syncthreads();
        const int cnt = (n / N) << sh;
        for (int k = threadIdx.x; k < cnt; k += blockDim.x) {
            const int l = k >> sh, J = (2 * (k & ((1 << sh) - 1)) + 1) << t, st = 1 << t;
            double *p = v + (quot(l, S, inv, small) * S * (N - 1) + l + (J - 1) * S);
            const double a = J > st ? p[-st * S] : 0.0;
            const double b = J + st <= N ? p[st * S] : 0.0;
            *p = fma(h, a + b, *p);
        }
    }
}
// every axis in turn; v complete on entry and on return
template <bool BACK>
__device__ __forceinline__ void all_axes(double *v, const GridInfo &G)
{
    for (int q = 0; q < G.de; ++q) {
        const int N = G.N[G.ax[q]], S = G.S[G.ax[q]];
        switch (N) {
        case 1: break;
        case 3: lines_pass<3, BACK>(v, G.n, S); break;
        case 7: lines_pass<7, BACK>(v, G.n, S); break;
        case 15: lines_pass<15, BACK>(v, G.n, S); break;
        default: levels_pass<BACK>(v, G.n, N, S); break;
        }
        __syncthreads();
    }
}
// Block (number in the grid's own list of increments) and position in it of
// node j.
struct Axes {  // the grid's listed axes, last (fastest) first
    int de, N[PIT_D], lev[PIT_D];
    float inv[PIT_D];
};
__device__ __forceinline__ void axes_of(const GridInfo &G, Axes &A)  // (one thread)
{
    A.de = G.de;
    for (int q = 0; q < G.de; ++q) {
        const int N = G.N[G.ax[G.de - 1 - q]];
        A.N[q] = N;
        A.lev[q] = 31 - __clz(N + 1);
        A.inv[q] = 1.0f / (float)N;
    }
}
__device__ __forceinline__ void block_of(const Axes &A, int j, bool small, int &blk, int &pos)
{
    int r = j, mul = 1, sh = 0;
    blk = 0;
    pos = 0;
    for (int q = 0; q < A.de; ++q) {
        const int N = A.N[q], hi = quot(r, N, A.inv[q], small), J = r - hi * N + 1;
        r = hi;
        const int t = __ffs(J), lam1 = A.lev[q] - t;  // lam - 1, t - 1 trailing zeros
        blk += lam1 * mul;
        mul *= A.lev[q];
        pos += (J >> t) << sh;
        sh += lam1;
    }
}

// One CTA per (grid, state).  T: natural-order scratch of a state for grids
// whose values do not fit on chip, may be u (NULL: on chip, dynamic shared
// memory).
__global__ void __launch_bounds__(256, 4) hier_kernel(RecombPlan R, const GridInfo *grids, const int *order, int n_order,
                                                   long long ntot, const double *u, double *H, double *T)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ GridInfo G;
    __shared__ Axes A;
    const int g = order[blockIdx.x % n_order];
    const long long b = blockIdx.x / n_order;
    for (int t = threadIdx.x; t < (int)(sizeof(GridInfo) / 4); t += blockDim.x)
        reinterpret_cast<int *>(&G)[t] = reinterpret_cast<const int *>(grids + g)[t];
    __syncthreads();
    if (threadIdx.x == 0) axes_of(G, A);
    const int n = G.n;
    const bool small = n < (1 << 20);
    double *v = T ? T + b * ntot + G.off : reinterpret_cast<double *>(smem);
    int *tab = reinterpret_cast<int *>(smem) + (T ? 0 : 2 * n);
    const RecombBlock *bl = R.blocks + R.grid_blocks[g];
    const int nb = (int)(R.grid_blocks[g + 1] - R.grid_blocks[g]);
    const double *src = u + b * ntot + G.off;
    for (int j = threadIdx.x; j < n; j += blockDim.x) v[j] = src[j];
    for (int k = threadIdx.x; k < nb; k += blockDim.x) tab[k] = bl[k].in_grid;
    __syncthreads();
    all_axes<false>(v, G);
    double *dst = H + b * ntot + G.off;
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        int blk, pos;
        block_of(A, j, small, blk, pos);
        dst[tab[blk] + pos] = v[j];
    }
}

// One CTA of 256 threads per piece of a block (256 nodes at most) and state.
__global__ void __launch_bounds__(256) gather_kernel(RecombPlan R, long long ntot, const double *Hb, double *Sb)
{
    __shared__ double part[256];
    const RecombPiece pc = R.pieces[blockIdx.x % R.n_pieces];
    const long long b = blockIdx.x / R.n_pieces;
    const double *H = Hb + b * ntot;
    double *S = Sb + b * R.n_sparse;
    // pc.n is a power of two up to 256: threads beyond a block's nodes take
    // further slices of its list
    const int node = threadIdx.x & (pc.n - 1), slice = threadIdx.x / pc.n, slices = 256 / pc.n;
    // (a slice is a run of the list, whose coefficients nearly cancel)
    const int len = (pc.list1 - pc.list0 + slices - 1) / slices;
    const int k0 = pc.list0 + slice * len, k1 = min(k0 + len, pc.list1);
    double acc = 0.0;
#pragma unroll 4
    for (int k = k0; k < k1; ++k) {
        const RecombTerm t = R.terms[k];
        acc = fma(t.coef, H[t.at + pc.first + node], acc);
    }
    if (slices == 1) {
        S[pc.at + node] = acc;
        return;
    }
    part[threadIdx.x] = acc;
    __syncthreads();
    // slices added in order, pairwise (fixed tree)
    for (int w = slices / 2; w >= 1; w /= 2) {
        if (slice < w) part[threadIdx.x] += part[threadIdx.x + w * pc.n];
        __syncthreads();
    }
    if (slice == 0) S[pc.at + node] = part[node];
}

__global__ void __launch_bounds__(256, 4) dehier_kernel(RecombPlan R, const GridInfo *grids, const int *order, int n_order,
                                                     long long ntot, const double *Sb, double *out, bool onchip)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ GridInfo G;
    __shared__ Axes A;
    const int g = order[blockIdx.x % n_order];
    const long long b = blockIdx.x / n_order;
    for (int t = threadIdx.x; t < (int)(sizeof(GridInfo) / 4); t += blockDim.x)
        reinterpret_cast<int *>(&G)[t] = reinterpret_cast<const int *>(grids + g)[t];
    __syncthreads();
    if (threadIdx.x == 0) axes_of(G, A);
    const int n = G.n;
    const bool small = n < (1 << 20);
    double *dst = out + b * ntot + G.off;
    double *v = onchip ? reinterpret_cast<double *>(smem) : dst;
    long long *tab = reinterpret_cast<long long *>(smem) + (onchip ? n : 0);
    const RecombBlock *bl = R.blocks + R.grid_blocks[g];
    const int nb = (int)(R.grid_blocks[g + 1] - R.grid_blocks[g]);
    const double *S = Sb + b * R.n_sparse;
    for (int k = threadIdx.x; k < nb; k += blockDim.x) tab[k] = bl[k].in_sparse;
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        int blk, pos;
        block_of(A, j, small, blk, pos);
        v[j] = S[tab[blk] + pos];
    }
    __syncthreads();
    all_axes<true>(v, G);
    if (onchip)
        for (int j = threadIdx.x; j < n; j += blockDim.x) dst[j] = v[j];
}

}  // namespace

size_t recombine_smem_bytes(int n, int n_blocks, bool onchip)
{
    return (onchip ? (size_t)n * 8 : 0) + (size_t)n_blocks * 8 + 16;
}

cudaError_t recombine_init(size_t max_smem)
{
    const cudaError_t e = cudaFuncSetAttribute((const void *)hier_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)max_smem);
    return e != cudaSuccess ? e : cudaFuncSetAttribute((const void *)dehier_kernel,
                                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)max_smem);
}

cudaError_t launch_recombine(const RecombPlan &R, const GridInfo *grids, const int *order, long long ntot, int nb,
                             const double *u, double *H, double *S, double *out, cudaStream_t s)
{
    if (nb <= 0) return cudaSuccess;
    if ((long long)R.n_pieces * nb > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    for (int c = 0; c < RECOMB_CLS; ++c)
        if ((long long)R.cls_n[c] * nb > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    for (int c = 0; c < RECOMB_CLS; ++c)
        if (R.cls_n[c] > 0)
            hier_kernel<<<(unsigned)(R.cls_n[c] * nb), 256, R.cls_smem[c], s>>>(
                R, grids, order + R.cls_first[c], R.cls_n[c], ntot, u, H, c == 0 ? out : nullptr);
    gather_kernel<<<(unsigned)(R.n_pieces * nb), 256, 0, s>>>(R, ntot, H, S);
    for (int c = 0; c < RECOMB_CLS; ++c)
        if (R.cls_n[c] > 0)
            dehier_kernel<<<(unsigned)(R.cls_n[c] * nb), 256, R.cls_smem[c], s>>>(
                R, grids, order + R.cls_first[c], R.cls_n[c], ntot, S, out, c != 0);
    return cudaGetLastError();
}

}  // namespace pit
