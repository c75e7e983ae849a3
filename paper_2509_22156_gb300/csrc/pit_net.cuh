// Learned coarse propagator (not in the paper; it replaces the coarse-level
// backward-Euler step Phi_c of Sec. 3.3.1 inside MGRIT): an axis-separable
// 1-D convolutional network, 4 layers of width-5 convolutions along every
// axis with one weight set shared by all axes, channels (u, a, s) -> 16 -> 16
// -> 16 -> 1, ReLU on the hidden layers, applied to the state normalised by
// its RMS sigma:  Phi_hat(u) = u + sigma * h4(u / sigma).  Input channels: the
// normalised state, the diffusion coefficient a at the nodes (1 for constant-
// coefficient operators) and, per axis, s_i = 1 / (1 + 4 dT / h_i^2); taps
// outside the grid read zero (Dirichlet).
//
// Weights are rounded to BF16 (round to nearest even) from FP32 master
// weights; activations and accumulation are FP32; the state and sigma FP64.
// Because the weights are shared across axes, sum_i conv_i(h; W) equals
// sum_t W_t * z_t with z_t = sum_i h(j + (t-2) e_i): each layer forms the
// axis sums once per node and mixes channels once, not d times.  In the
// inference kernel the weights travel as a kernel parameter, so every FMA
// takes its weight from the constant bank (no shared-memory traffic).
#pragma once

#include <cmath>

#include "pit_internal.cuh"

namespace pit {

__host__ __device__ constexpr int net_cin(int k) { return k == 0 ? 3 : 17; }
__host__ __device__ constexpr int net_cout(int k) { return k == 3 ? 1 : 16; }
__host__ __device__ constexpr int net_wo(int k)
{
    return k == 0 ? 0 : net_wo(k - 1) + net_cout(k - 1) * net_cin(k - 1) * 5 + net_cout(k - 1);
}
__host__ __device__ constexpr int net_bo(int k) { return net_wo(k) + net_cout(k) * net_cin(k) * 5; }
static_assert(net_bo(3) + 1 == PIT_NET_PARAMS, "parameter layout");

// Weight access from the kernel-parameter bank.
struct WParam {
    const NetWeights &w;
    __device__ __forceinline__ float operator()(int i) const { return w.w[i]; }
};

// Tap validity of node j along axis i for offset t-2 (t = 0..4): bits of the
// extended mask (4 bits per axis: -1, +1, -2, +2).
__device__ __forceinline__ bool tap_ok(uint32_t mk, int i, int t)
{
    if (t == 2) return true;
    const int bit = (t == 1) ? 0 : (t == 3) ? 1 : (t == 0) ? 2 : 3;
    return (mk >> (4 * i + bit)) & 1u;
}

template <int D>
__device__ __forceinline__ uint32_t ext_mask(const GridInfo &G, int j)
{
    uint32_t mk = 0;
#pragma unroll
    for (int i = 0; i < D; ++i) {
        const int c = (j / G.S[i]) % G.N[i];
        if (c >= 1) mk |= 1u << (4 * i);
        if (c + 1 < G.N[i]) mk |= 1u << (4 * i + 1);
        if (c >= 2) mk |= 1u << (4 * i + 2);
        if (c + 2 < G.N[i]) mk |= 1u << (4 * i + 3);
    }
    return mk;
}

// Diffusion coefficient at the nodes (the network's second input channel).
__device__ inline double node_coef(const OpParams &op, const GridInfo &G, int j, int d)
{
    if (op.op != PIT_OP_VARHEAT) return 1.0;
    double prod = 1.0;
    for (int i = 0; i < d; ++i) {
        const double x = op.lo[i] + (double)((j / G.S[i]) % G.N[i] + 1) * G.h[i];
        prod *= (i % 2 == 0) ? sin(2.0 * M_PI * x) : cos(2.0 * M_PI * x);
    }
    return 1.0 + op.vamp * prod;
}

// One convolution layer: out[o][j] = act(b_o + sum_t sum_c W[o][c][t] z_{c,t}(j)),
// z_{c,t}(j) = sum_i in[c][j + (t-2) S_i] over valid taps; the last input
// channel is the per-axis constant s_i.
template <int D, int CIN, int COUT, bool RELU, class WA>
__device__ __forceinline__ void conv_layer(const WA &W, int wo, int bo, const float *in, float *out, int n, int ld,
                                           const uint32_t *mk2, const int *S, const float *sf)
{
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
        float acc[COUT];
#pragma unroll
        for (int o = 0; o < COUT; ++o) acc[o] = W(bo + o);
        const uint32_t mk = mk2[j];
#pragma unroll
        for (int t = 0; t < 5; ++t) {
#pragma unroll
            for (int c = 0; c < CIN - 1; ++c) {
                float z = 0.0f;
#pragma unroll
                for (int i = 0; i < D; ++i)
                    if (tap_ok(mk, i, t)) z += in[c * ld + j + (t - 2) * S[i]];
#pragma unroll
                for (int o = 0; o < COUT; ++o) acc[o] = fmaf(W(wo + (o * CIN + c) * 5 + t), z, acc[o]);
            }
            float zs = 0.0f;
#pragma unroll
            for (int i = 0; i < D; ++i)
                if (tap_ok(mk, i, t)) zs += sf[i];
#pragma unroll
            for (int o = 0; o < COUT; ++o) acc[o] = fmaf(W(wo + (o * CIN + CIN - 1) * 5 + t), zs, acc[o]);
        }
#pragma unroll
        for (int o = 0; o < COUT; ++o) out[o * ld + j] = RELU ? fmaxf(acc[o], 0.0f) : acc[o];
    }
}

// Deterministic block sum in FP64 (shuffles, one barrier, same tree in every warp).
__device__ __forceinline__ double block_sum64(double v, double *red)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();  // red free
    if (lane == 0) red[w] = v;
    __syncthreads();
    double x = (lane < nw) ? red[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xffffffffu, x, o);
    return __shfl_sync(0xffffffffu, x, 0);
}

// Full forward pass of one item on normalised input already in A0 (channel 0:
// u / sigma, channel 1: a).  Result (layer-4 pre-activation) in O[0..n).
// H holds 2 x 16 channels (ping-pong).
template <int D, class WA>
__device__ void net_forward(const WA &W, const float *A0, float *H, float *O, int n, int ld, const uint32_t *mk2,
                            const int *S, const float *sf)
{
    float *H1 = H, *H2 = H + 16 * ld, *H3 = H;
    conv_layer<D, 3, 16, true>(W, net_wo(0), net_bo(0), A0, H1, n, ld, mk2, S, sf);
    __syncthreads();
    conv_layer<D, 17, 16, true>(W, net_wo(1), net_bo(1), H1, H2, n, ld, mk2, S, sf);
    __syncthreads();
    conv_layer<D, 17, 16, true>(W, net_wo(2), net_bo(2), H2, H3, n, ld, mk2, S, sf);
    __syncthreads();
    conv_layer<D, 17, 1, false>(W, net_wo(3), net_bo(3), H3, O, n, ld, mk2, S, sf);
    __syncthreads();
}

// ----------------------------------------------------------------------------
// Inference: multi-step application of the network with the StepArgs
// semantics of the backward-Euler kernels (forcing g after each step, stored
// steps, out_last = out_scale * x + h).  One CTA per item; activations in
// shared memory (act == NULL) or in a per-item global slab.
template <int D>
__global__ void __launch_bounds__(256) net_steps_kernel(StepArgs a, const __grid_constant__ NetWeights W, float *act,
                                                        long long act_stride)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ GridInfo GI;
    __shared__ double red[32];
    __shared__ int S[D];
    __shared__ float sf[D];
    const int item = a.item0 + (int)blockIdx.x;
    const int g = a.order[item / a.n_batch];
    const int b = item % a.n_batch;
    if (a.active && !a.active[g]) return;
    if (threadIdx.x == 0) GI = a.grids[g];
    __syncthreads();
    const int tid = threadIdx.x, nt = blockDim.x, n = GI.n, ld = (n + 3) & ~3;
    if (tid < D) {
        S[tid] = GI.S[tid];
        sf[tid] = (float)(1.0 / (1.0 + 4.0 * a.dt / (GI.h[tid] * GI.h[tid])));
    }
    double *x = reinterpret_cast<double *>(smem);
    uint32_t *mk2 = reinterpret_cast<uint32_t *>(x + ld);
    float *base = act ? act + (long long)blockIdx.x * act_stride : reinterpret_cast<float *>(mk2 + ld);
    float *A0 = base, *H = base + 2 * ld, *O = base + 34 * ld;
    const double *in = a.in + (long long)b * a.in_stride + GI.off;
    for (int j = tid; j < n; j += nt) {
        x[j] = in[j];
        mk2[j] = ext_mask<D>(GI, j);
        A0[ld + j] = (float)node_coef(a.op, GI, j, D);
    }
    for (int step = 1; step <= a.nsteps; ++step) {
        __syncthreads();
        double ss = 0.0;
        for (int j = tid; j < n; j += nt) ss += x[j] * x[j];
        ss = block_sum64(ss, red);
        const double sigma = sqrt(ss / (double)n);
        if (sigma > 0.0) {
            const double inv = 1.0 / sigma;
            for (int j = tid; j < n; j += nt) A0[j] = (float)(x[j] * inv);
            __syncthreads();
            net_forward<D>(WParam{W}, A0, H, O, n, ld, mk2, S, sf);
            for (int j = tid; j < n; j += nt) x[j] += sigma * (double)O[j];
        }
        const long long sb = (long long)(step - 1);
        if (a.g) {
            const double *gs = a.g + (long long)b * a.g_stride + sb * a.g_step + GI.off;
            for (int j = tid; j < n; j += nt) x[j] += gs[j];
        }
        const double *hs = a.hs ? a.hs + (long long)b * a.hs_stride + sb * a.hs_step + GI.off : nullptr;
        if (step < a.nsteps) {
            if (a.out_steps) {
                double *os = a.out_steps + (long long)b * a.os_stride + sb * a.os_step + GI.off;
                for (int j = tid; j < n; j += nt) os[j] = hs ? x[j] + hs[j] : x[j];
            }
        } else {
            double *ol = a.out_last + (long long)b * a.ol_stride + GI.off;
            const double *h = a.h ? a.h + (long long)b * a.h_stride + GI.off : nullptr;
            for (int j = tid; j < n; j += nt)
                ol[j] = a.out_scale * x[j] + (h ? a.out_hscale * h[j] : 0.0) + (hs ? hs[j] : 0.0);
        }
    }
    if (tid == 0 && a.stats) {
        atomicAdd(&a.stats->items, (unsigned long long)a.nsteps);
        atomicAdd(&a.stats->point_steps, (unsigned long long)a.nsteps * (unsigned long long)n);
    }
}

// ----------------------------------------------------------------------------
// Training: one CTA per item (a grid of one pair): forward with stored
// activations, relative squared loss ||Phi_hat(u) - y||^2 / ||y||^2, and the
// gradient with respect to every parameter, written as one row per item
// (reduced later in a fixed order, so the gradient is deterministic).
//
// What bounds it: shared-memory reads beside the FMAs of the three 85 x 16
// products a node and layer (forward, input gradient, weight gradient; FP32
// throughout, weights BF16-rounded), and the largest grid, one CTA working on
// it.  Two kernels: net_train_kernel takes an item forward and back to every
// layer's output gradient, net_wgrad_kernel one (item, layer) to its weight
// gradient, so that the layers' sums run on different SMs.  In the first,
// activations (51 channels, the gradient of a layer's input overwriting that
// input) and the layer's weights, transposed so that one 16-byte read gives
// four outputs' weights, are on chip up to 940 nodes and in the item's global
// slab beyond; neighbour indices of a node are worked out once a pass, a missing
// tap pointing at a zero element of its row; two nodes a thread share every
// weight read.  The weight gradient takes tiles of 64 nodes: axis sums of every
// (channel, tap) row and the output gradients in shared memory, then every
// thread sums eight outputs of one row over half of the tile.
// varheat3d level 8 (85 grids of up to 735 nodes), the whole call with its
// copies: 1,263 us when every FMA read its own weight from global memory and
// every row's thread formed its own axis sums, 401 us with both parts in one
// kernel, 286 us now.
constexpr int NET_THREADS = 512, NET_TILE = 64, NET_TLD = NET_TILE + 4;
constexpr int NET_CHIP = 940;  // largest grid whose activations stay on chip
__host__ __device__ constexpr int net_ld(int n) { return (n + 4) & ~3; }  // one zero element past the nodes
__host__ __device__ constexpr int net_chip_words(int n) { return 52 * net_ld(n); }
// an item's global slab: input (2 channels), H1..H3, the output gradients of
// the last layer (1) and of layers 0..2 (16 each), tap masks
__host__ __device__ constexpr int net_train_words(int n) { return 100 * net_ld(n); }
__host__ __device__ constexpr int net_h_row(int k) { return 2 + 16 * k; }               // output of layer k < 3
__host__ __device__ constexpr int net_d_row(int k) { return k == 3 ? 50 : 51 + 16 * k; }  // gradient of its pre-activations

// Indices of a node's neighbours at offsets -2, -1, +1, +2 along every axis
// (zero: the index of the zero element).
template <int D>
__device__ __forceinline__ void net_neighbours(uint32_t mk, int j, const int *S, int zero, int (&ix)[D][4])
{
#pragma unroll
    for (int i = 0; i < D; ++i) {
        ix[i][0] = (mk >> (4 * i + 2)) & 1u ? j - 2 * S[i] : zero;
        ix[i][1] = (mk >> (4 * i)) & 1u ? j - S[i] : zero;
        ix[i][2] = (mk >> (4 * i + 1)) & 1u ? j + S[i] : zero;
        ix[i][3] = (mk >> (4 * i + 3)) & 1u ? j + 2 * S[i] : zero;
    }
}
// Nodes a thread takes at a time: two share every weight read; with five or six
// axes the second node's neighbour indices no longer fit in registers.
template <int D>
constexpr bool net_two = D <= 4;
// axis sum z_t = sum_i in(j + (t - 2) e_i)
template <int D>
__device__ __forceinline__ float net_axis_sum(const float *in, int j, int t, const int (&ix)[D][4])
{
    if (t == 2) return (float)D * in[j];
    const int q = t < 2 ? t : t - 1;
    float z = 0.0f;
#pragma unroll
    for (int i = 0; i < D; ++i) z += in[ix[i][q]];
    return z;
}
// a[o] += sum over nch channels and taps of wt[(c 5 + t) 16 + o] z_{c,t} for two nodes
template <int D>
__device__ __forceinline__ void net_conv16(const float *in, int nch, int ld, const float4 *wt, int j0, int j1,
                                           const int (&x0)[D][4], const int (&x1)[D][4], float (&a0)[16], float (&a1)[16])
{
#pragma unroll 1
    for (int c = 0; c < nch; ++c) {
        const float *row = in + c * ld;
#pragma unroll
        for (int t = 0; t < 5; ++t) {
            const float z0 = net_axis_sum<D>(row, j0, t, x0);
            float z1 = 0.0f;
            if constexpr (net_two<D>) z1 = net_axis_sum<D>(row, j1, t, x1);
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 w = wt[(c * 5 + t) * 4 + q];
                a0[4 * q] = fmaf(w.x, z0, a0[4 * q]);
                if constexpr (net_two<D>) a1[4 * q] = fmaf(w.x, z1, a1[4 * q]);
                a0[4 * q + 1] = fmaf(w.y, z0, a0[4 * q + 1]);
                if constexpr (net_two<D>) a1[4 * q + 1] = fmaf(w.y, z1, a1[4 * q + 1]);
                a0[4 * q + 2] = fmaf(w.z, z0, a0[4 * q + 2]);
                if constexpr (net_two<D>) a1[4 * q + 2] = fmaf(w.z, z1, a1[4 * q + 2]);
                a0[4 * q + 3] = fmaf(w.w, z0, a0[4 * q + 3]);
                if constexpr (net_two<D>) a1[4 * q + 3] = fmaf(w.w, z1, a1[4 * q + 3]);
            }
        }
    }
}

template <int D>
struct NetItem {  // one item's geometry and buffers
    int n, ld;
    const int *S;
    const float *sf;
    const uint32_t *mk;
    float *wt, *zt, *dt;  // weights of a layer, tile of axis sums, tile of output gradients
};

// out[o][j] of one layer: ReLU of 16 channels, or the last layer's single one
// (copy: second place of the output, or NULL)
template <int D>
__device__ __forceinline__ void net_layer(const NetItem<D> &I, int k, const float *w, const float *in, float *out,
                                          float *copy)
{
    const int cin = net_cin(k), cout = net_cout(k), wo = net_wo(k), bo = net_bo(k), nt = blockDim.x;
    __syncthreads();  // in complete, wt free
    for (int q = threadIdx.x; q < cin * 5 * 16; q += nt) {
        const int r = q >> 4, o = q & 15;
        I.wt[q] = o < cout ? __ldg(w + wo + (o * cin + r / 5) * 5 + r % 5) : 0.0f;
    }
    __syncthreads();
    const float4 *wt = reinterpret_cast<const float4 *>(I.wt);
    for (int j0 = threadIdx.x; j0 < I.n; j0 += (net_two<D> ? 2 : 1) * nt) {
        const bool two = net_two<D> && j0 + nt < I.n;
        const int j1 = two ? j0 + nt : I.n;
        int x0[D][4], x1[D][4];
        const uint32_t m0 = I.mk[j0], m1 = two ? I.mk[j1] : 0u;
        net_neighbours<D>(m0, j0, I.S, I.n, x0);
        net_neighbours<D>(m1, j1, I.S, I.n, x1);
        float a0[16], a1[16];
        if (k == 3) {
            a0[0] = a1[0] = __ldg(w + bo);
#pragma unroll 1
            for (int c = 0; c < 16; ++c)
#pragma unroll
                for (int t = 0; t < 5; ++t) {
                    const float wv = I.wt[(c * 5 + t) * 16];
                    a0[0] = fmaf(wv, net_axis_sum<D>(in + c * I.ld, j0, t, x0), a0[0]);
                    if constexpr (net_two<D>) a1[0] = fmaf(wv, net_axis_sum<D>(in + c * I.ld, j1, t, x1), a1[0]);
                }
        } else {
#pragma unroll
            for (int o = 0; o < 16; ++o) a0[o] = a1[o] = __ldg(w + bo + o);
            net_conv16<D>(in, cin - 1, I.ld, wt, j0, j1, x0, x1, a0, a1);
        }
        // the s channel: s_i where the tap exists
#pragma unroll
        for (int t = 0; t < 5; ++t) {
            float z0 = 0.0f, z1 = 0.0f;
#pragma unroll
            for (int i = 0; i < D; ++i) {
                if (tap_ok(m0, i, t)) z0 += I.sf[i];
                if (tap_ok(m1, i, t)) z1 += I.sf[i];
            }
            const float *ws = I.wt + ((cin - 1) * 5 + t) * 16;
            if (k == 3) {
                a0[0] = fmaf(ws[0], z0, a0[0]);
                a1[0] = fmaf(ws[0], z1, a1[0]);
            } else {
#pragma unroll
                for (int o = 0; o < 16; ++o) {
                    a0[o] = fmaf(ws[o], z0, a0[o]);
                    a1[o] = fmaf(ws[o], z1, a1[o]);
                }
            }
        }
        if (k == 3) {
            out[j0] = a0[0];
            if (two) out[j1] = a1[0];
        } else {
#pragma unroll
            for (int o = 0; o < 16; ++o) {
                const float h0 = fmaxf(a0[o], 0.0f), h1 = fmaxf(a1[o], 0.0f);
                out[o * I.ld + j0] = h0;
                if (two) out[o * I.ld + j1] = h1;
                if (copy) {
                    copy[o * I.ld + j0] = h0;
                    if (two) copy[o * I.ld + j1] = h1;
                }
            }
        }
    }
}

// Gradient of the layer's weights and biases from its input and the gradient
// dc of its pre-activations, into grow.
template <int D>
__device__ __forceinline__ void net_weight_grad(const NetItem<D> &I, int k, const float *in, const float *dc, float *grow)
{
    const int cind = net_cin(k) - 1, cout = net_cout(k), R = (cind + 1) * 5;
    const int tid = threadIdx.x, nt = blockDim.x, warp = tid >> 5, lane = tid & 31;
    const int row = tid >> 2, grp = tid & 1, split = (tid >> 1) & 1;  // row R: the bias
    const bool active = row <= R && grp * 8 < cout;
    float acc[8];
#pragma unroll
    for (int o = 0; o < 8; ++o) acc[o] = 0.0f;
    for (int j0 = 0; j0 < I.n; j0 += NET_TILE) {
        __syncthreads();  // tile free (first: dc complete)
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const int kk = lane + 32 * half, j = j0 + kk;
            if (j < I.n) {
                int ix[D][4];
                const uint32_t m = I.mk[j];
                net_neighbours<D>(m, j, I.S, I.n, ix);
                for (int c = warp; c <= cind; c += NET_THREADS / 32) {
#pragma unroll
                    for (int t = 0; t < 5; ++t) {
                        float z = 0.0f;
                        if (c < cind) {
                            z = net_axis_sum<D>(in + c * I.ld, j, t, ix);
                        } else {
#pragma unroll
                            for (int i = 0; i < D; ++i)
                                if (tap_ok(m, i, t)) z += I.sf[i];
                        }
                        I.zt[(c * 5 + t) * NET_TLD + kk] = z;
                    }
                }
            } else {
                for (int c = warp; c <= cind; c += NET_THREADS / 32)
#pragma unroll
                    for (int t = 0; t < 5; ++t) I.zt[(c * 5 + t) * NET_TLD + kk] = 0.0f;
            }
        }
        if (tid < NET_TILE) I.zt[R * NET_TLD + tid] = 1.0f;
        for (int q = tid; q < 16 * NET_TILE; q += nt) {
            const int o = q / NET_TILE, kk = q % NET_TILE, j = j0 + kk;
            I.dt[o * NET_TLD + kk] = o < cout && j < I.n ? dc[o * I.ld + j] : 0.0f;
        }
        __syncthreads();
        if (active) {
            // (a tile's sum by itself: the rounding errors of the whole grow with
            // the tiles, not with the nodes)
            float part[8];
#pragma unroll
            for (int o = 0; o < 8; ++o) part[o] = 0.0f;
            const float4 *z4 = reinterpret_cast<const float4 *>(I.zt + row * NET_TLD + split * (NET_TILE / 2));
#pragma unroll 2
            for (int q = 0; q < NET_TILE / 8; ++q) {
                const float4 z = z4[q];
#pragma unroll
                for (int o = 0; o < 8; ++o) {
                    const float4 d = reinterpret_cast<const float4 *>(I.dt + (grp * 8 + o) * NET_TLD + split * (NET_TILE / 2))[q];
                    part[o] = fmaf(d.x, z.x, part[o]);
                    part[o] = fmaf(d.y, z.y, part[o]);
                    part[o] = fmaf(d.z, z.z, part[o]);
                    part[o] = fmaf(d.w, z.w, part[o]);
                }
            }
#pragma unroll
            for (int o = 0; o < 8; ++o) acc[o] += part[o];
        }
    }
    __syncthreads();
    if (active && split == 1) {
#pragma unroll
        for (int o = 0; o < 8; ++o) I.zt[(row * 2 + grp) * 8 + o] = acc[o];
    }
    __syncthreads();
    if (active && split == 0) {
#pragma unroll
        for (int o = 0; o < 8; ++o) {
            const int oo = grp * 8 + o;
            if (oo < cout) {
                const float v = acc[o] + I.zt[(row * 2 + grp) * 8 + o];
                grow[row == R ? net_bo(k) + oo : net_wo(k) + (oo * (cind + 1) + row / 5) * 5 + row % 5] = v;
            }
        }
    }
}

// Gradient of the layer's 16 input channels through the ReLU of the layer
// before, whose output is h, into out (may be h) and copy (or NULL):
// din[c][j] = sum_t sum_o W[o][c][t] sum_i dc[o][j - (t-2) e_i].
template <int D>
__device__ __forceinline__ void net_input_grad(const NetItem<D> &I, int k, const float *w, const float *dc, const float *h,
                                               float *out, float *copy)
{
    const int cout = net_cout(k), wo = net_wo(k), nt = blockDim.x;
    __syncthreads();  // wt and the tiles free, dc and h read
    for (int q = threadIdx.x; q < cout * 5 * 16; q += nt) {
        const int r = q >> 4, c = q & 15;  // row (o, t'), t' = 4 - t
        I.wt[q] = __ldg(w + wo + ((r / 5) * 17 + c) * 5 + (4 - r % 5));
    }
    __syncthreads();
    const float4 *wt = reinterpret_cast<const float4 *>(I.wt);
    for (int j0 = threadIdx.x; j0 < I.n; j0 += (net_two<D> ? 2 : 1) * nt) {
        const bool two = net_two<D> && j0 + nt < I.n;
        const int j1 = two ? j0 + nt : I.n;
        int x0[D][4], x1[D][4];
        net_neighbours<D>(I.mk[j0], j0, I.S, I.n, x0);
        net_neighbours<D>(two ? I.mk[j1] : 0u, j1, I.S, I.n, x1);
        float a0[16], a1[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) a0[c] = a1[c] = 0.0f;
        net_conv16<D>(dc, cout, I.ld, wt, j0, j1, x0, x1, a0, a1);
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            const float d0 = h[c * I.ld + j0] > 0.0f ? a0[c] : 0.0f;
            out[c * I.ld + j0] = d0;
            if (copy) copy[c * I.ld + j0] = d0;
            if (two) {
                const float d1 = h[c * I.ld + j1] > 0.0f ? a1[c] : 0.0f;
                out[c * I.ld + j1] = d1;
                if (copy) copy[c * I.ld + j1] = d1;
            }
        }
    }
}

// slab: the item's global slab; chip: on-chip activations, or NULL
template <int D, bool CHIP>
__device__ __forceinline__ void net_train_item(const GridInfo &GI, const int *S, const float *sf, double *red, float *tiles,
                                               float *chip, float *slab, const NetTrainItem &it, const double *u,
                                               const double *y, const float *w, double *loss, const OpParams &op)
{
    const int tid = threadIdx.x, nt = blockDim.x, n = GI.n, ld = net_ld(n);
    float *acts = CHIP ? chip : slab;
    float *A0 = acts, *H1 = acts + net_h_row(0) * ld, *H2 = acts + net_h_row(1) * ld, *H3 = acts + net_h_row(2) * ld;
    float *O = acts + net_d_row(3) * ld;
    uint32_t *mkg = reinterpret_cast<uint32_t *>(slab + 99 * ld);
    uint32_t *mk = CHIP ? reinterpret_cast<uint32_t *>(chip + 51 * ld) : mkg;
    NetItem<D> I{n, ld, S, sf, mk, tiles, nullptr, nullptr};
    const double *ui = u + it.off, *yi = y + it.off;
    double ss = 0.0, yy = 0.0;
    for (int j = tid; j < n; j += nt) {
        const uint32_t m = ext_mask<D>(GI, j);
        const float c = (float)node_coef(op, GI, j, D);
        mk[j] = m;
        A0[ld + j] = c;
        if (CHIP) {
            mkg[j] = m;
            slab[ld + j] = c;
        }
        ss += ui[j] * ui[j];
        yy += yi[j] * yi[j];
    }
    for (int c = tid; c < 99; c += nt) {  // the zero element of every row
        slab[c * ld + n] = 0.0f;
        if (CHIP && c < 51) chip[c * ld + n] = 0.0f;
    }
    ss = block_sum64(ss, red);
    yy = block_sum64(yy, red);
    const double sigma = sqrt(ss / (double)n);
    if (!(yy > 0.0)) yy = 1.0;
    if (!(sigma > 0.0)) {
        // identity map: the loss does not depend on the parameters
        double l = 0.0;
        for (int j = tid; j < n; j += nt) l += (ui[j] - yi[j]) * (ui[j] - yi[j]);
        l = block_sum64(l, red);
        for (int q = tid; q < 99 * ld; q += nt) slab[q] = 0.0f;
        if (tid == 0) *loss = l / yy;
        return;
    }
    const double inv = 1.0 / sigma;
    for (int j = tid; j < n; j += nt) {
        const float v = (float)(ui[j] * inv);
        A0[j] = v;
        if (CHIP) slab[j] = v;
    }
    auto copy = [&](int row) -> float * { return CHIP ? slab + row * ld : nullptr; };
    net_layer<D>(I, 0, w, A0, H1, copy(net_h_row(0)));
    net_layer<D>(I, 1, w, H1, H2, copy(net_h_row(1)));
    net_layer<D>(I, 2, w, H2, H3, copy(net_h_row(2)));
    net_layer<D>(I, 3, w, H3, O, nullptr);
    __syncthreads();
    // loss and dL/d(layer-4 pre-activation) = 2 e sigma / ||y||^2
    double l = 0.0;
    for (int j = tid; j < n; j += nt) {
        const double e = ui[j] + sigma * (double)O[j] - yi[j];
        l += e * e;
        const float d = (float)(2.0 * e * sigma / yy);
        O[j] = d;
        if (CHIP) slab[net_d_row(3) * ld + j] = d;
    }
    l = block_sum64(l, red);
    if (tid == 0) *loss = l / yy;
    float *D2 = CHIP ? H3 : slab + net_d_row(2) * ld, *D1 = CHIP ? H2 : slab + net_d_row(1) * ld;
    float *D0 = CHIP ? H1 : slab + net_d_row(0) * ld;
    net_input_grad<D>(I, 3, w, O, H3, D2, copy(net_d_row(2)));
    net_input_grad<D>(I, 2, w, D2, H2, D1, copy(net_d_row(1)));
    net_input_grad<D>(I, 1, w, D1, H1, D0, copy(net_d_row(0)));
}

template <int D>
__global__ void __launch_bounds__(NET_THREADS, 1)
    net_train_kernel(const GridInfo *grids, const NetTrainItem *items, const double *u, const double *y, double dT,
                     const float *w, float *act, int n_chip, double *loss_items, OpParams op)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ GridInfo GI;
    __shared__ double red[32];
    __shared__ int S[D];
    __shared__ float sf[D];
    const NetTrainItem it = items[blockIdx.x];
    if (threadIdx.x == 0) GI = grids[it.g];
    __syncthreads();
    const int tid = threadIdx.x;
    if (tid < D) {
        S[tid] = GI.S[tid];
        sf[tid] = (float)(1.0 / (1.0 + 4.0 * dT / (GI.h[tid] * GI.h[tid])));
    }
    __syncthreads();
    float *tiles = reinterpret_cast<float *>(smem), *slab = act + it.act;
    // (two calls, so that the one on chip uses shared-memory instructions)
    if (GI.n <= n_chip)
        net_train_item<D, true>(GI, S, sf, red, tiles, tiles + 85 * 16, slab, it, u, y, w, loss_items + blockIdx.x, op);
    else
        net_train_item<D, false>(GI, S, sf, red, tiles, nullptr, slab, it, u, y, w, loss_items + blockIdx.x, op);
}

// One CTA per (item, layer).
template <int D>
__global__ void __launch_bounds__(NET_THREADS, 2)
    net_wgrad_kernel(const GridInfo *grids, const NetTrainItem *items, double dT, const float *act, float *grad_rows)
{
    __shared__ __align__(16) float tiles[(86 + 16) * NET_TLD];
    __shared__ int S[D];
    __shared__ float sf[D];
    const int item = blockIdx.x >> 2, k = 3 - (int)(blockIdx.x & 3);
    const GridInfo &GI = grids[items[item].g];
    if (threadIdx.x < D) {
        S[threadIdx.x] = GI.S[threadIdx.x];
        sf[threadIdx.x] = (float)(1.0 / (1.0 + 4.0 * dT / (GI.h[threadIdx.x] * GI.h[threadIdx.x])));
    }
    const int n = GI.n, ld = net_ld(n);
    const float *slab = act + items[item].act;
    const NetItem<D> I{n, ld, S, sf, reinterpret_cast<const uint32_t *>(slab + 99 * ld), nullptr, tiles, tiles + 86 * NET_TLD};
    net_weight_grad<D>(I, k, k == 0 ? slab : slab + net_h_row(k - 1) * ld, slab + net_d_row(k) * ld,
                       grad_rows + (long long)item * PIT_NET_PARAMS);
}

// Per-dimension launchers (one translation unit per d, pit_net_d<d>.cu).
#define PIT_NET_DECL(D)                                                                                          \
    cudaError_t net_init_d##D(int bytes);                                                                        \
    void net_launch_steps_d##D(const StepArgs &a, const NetWeights &W, float *act, long long act_stride,         \
                               dim3 grid, dim3 block, size_t smem, cudaStream_t s);                              \
    void net_launch_train_d##D(const GridInfo *grids, const NetTrainItem *it, const double *u, const double *y,   \
                               double dT, const float *w, float *act, int n_chip, float *grad_rows,              \
                               double *loss_items, OpParams op, dim3 grid, size_t smem, cudaStream_t s);
PIT_NET_DECL(1) PIT_NET_DECL(2) PIT_NET_DECL(3) PIT_NET_DECL(4) PIT_NET_DECL(5) PIT_NET_DECL(6)

#define PIT_NET_DIM(D)                                                                                           \
    cudaError_t net_init_d##D(int bytes)                                                                         \
    {                                                                                                            \
        const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;                                           \
        const cudaError_t e = cudaFuncSetAttribute((const void *)net_steps_kernel<D>, attr, bytes);              \
        return e != cudaSuccess ? e : cudaFuncSetAttribute((const void *)net_train_kernel<D>, attr, bytes);      \
    }                                                                                                            \
    void net_launch_steps_d##D(const StepArgs &a, const NetWeights &W, float *act, long long act_stride,         \
                               dim3 grid, dim3 block, size_t smem, cudaStream_t s)                               \
    {                                                                                                            \
        net_steps_kernel<D><<<grid, block, smem, s>>>(a, W, act, act_stride);                                    \
    }                                                                                                            \
    void net_launch_train_d##D(const GridInfo *grids, const NetTrainItem *it, const double *u, const double *y,   \
                               double dT, const float *w, float *act, int n_chip, float *grad_rows,              \
                               double *loss_items, OpParams op, dim3 grid, size_t smem, cudaStream_t s)          \
    {                                                                                                            \
        net_train_kernel<D><<<grid, NET_THREADS, smem, s>>>(grids, it, u, y, dT, w, act, n_chip, loss_items, op); \
        net_wgrad_kernel<D><<<dim3(grid.x * 4), NET_THREADS, 0, s>>>(grids, it, dT, act, grad_rows); \
    }

}  // namespace pit
