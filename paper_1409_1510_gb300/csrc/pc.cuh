// Gauge-covariant parallel-transport network: layer, adjoint-layer and weight-gradient kernels.
//
// A layer maps A input channels to B output channels of full-lattice colour fields, for K
// samples, one output parity at a time:
//   h'_b(x) = sum_path sum_a W[path][b][a] (T_path h_a)(x),
// path 0 = identity, the 8 one-hop transports through the fat links and the 8 three-hop
// transports through the Naik links.  The transports use the packed (gathered) links of the
// Dslash, whose backward slots hold -U^dag, so the backward paths take the weight with a minus
// sign.  Channel fields are stored per parity as [Vh][3 colour][K][C] complex FP32.
#pragma once
#include "hisq_internal.cuh"
#include "link_codec.cuh"
#include "dslash_kernel.cuh"

namespace hisq {

constexpr int PC_PATHS = 17;
constexpr int PC_CH[4] = {1, 4, 4, 1};

// weight offset (complex numbers) of layer l in the packed weight vector
__host__ __device__ constexpr int pc_layer_offset(int l) {
    return l == 0 ? 0 : l == 1 ? PC_PATHS * 4 * 1 : PC_PATHS * 4 * 1 + PC_PATHS * 4 * 4;
}

// path taken by gathered link slot j (0..7 fat, 8..15 Naik) and the sign of its weight
__host__ __device__ constexpr int slot_path(int j) { return (j < 8 ? 1 : 9) + (j & 7); }
__host__ __device__ constexpr float slot_sign(int j) { return (j & 1) ? -1.0f : 1.0f; }
// adjoint path (T^{+k} <-> T^{-k})
__host__ __device__ constexpr int adjoint_path(int p) { return p == 0 ? 0 : (((p - 1) & 1) ? p - 1 : p + 1); }

struct PcLayerArgs {
    Geom g;
    LinkField fat, naik;
    const float2 *in_same;  // [Vh][3][K][A] at the output parity (identity path) or null
    const float2 *in_opp;   // [Vh][3][K][A] at the opposite parity (hop paths) or null
    float2 *out;            // [Vh][3][K][B]
    const float2 *W;        // layer weights (see pc_layer_kernel)
    int K, spb, parity;
};

// Weights in shared memory as ws[q][b][a] for q = 0 (identity) and q = 1 + slot (16 slots),
// with the backward-slot sign folded in, each complex weight as (re, re, im, im): the two packed
// operands of mix().  ADJ: the adjoint of a layer with weights W[17][A][B] (mapping B -> A
// channels): ws[q][b][a] = conj(W[adj(q)][a][b]).
template <int A, int B, bool ADJ>
__device__ __forceinline__ void stage_weights(const float2 *W, float4 *ws) {
    for (int i = threadIdx.x; i < PC_PATHS * A * B; i += blockDim.x) {
        int q = i / (A * B), rem = i - q * A * B, b = rem / A, a = rem - b * A;
        int path = q == 0 ? 0 : slot_path(q - 1);
        float sign = q == 0 ? 1.0f : slot_sign(q - 1);
        float2 w;
        if (ADJ) {
            float2 o = W[(adjoint_path(path) * A + a) * B + b];
            w = make_float2(o.x, -o.y);
        } else {
            w = W[(path * B + b) * A + a];
        }
        ws[i] = make_float4(sign * w.x, sign * w.x, sign * w.y, sign * w.y);
    }
}

// Channels of a field with C channels that are worked on together: two of four (one 16-byte load
// per colour), or the only one.  Loaded channel by channel, a warp's lanes are 32 bytes apart and every
// wavefront of the L1 carries a quarter of its bytes: that pipe was 73% (4 -> 4) and 93% (4 -> 1) busy.
// M^dag M on 16 vectors at 32^3 x 8, FP32 arithmetic bound from then on: 4.57 / 3.52 ms.
template <int C>
constexpr int PC_CHUNK = C == 4 ? 2 : 1;

// channels a0 .. a0 + PC_CHUNK<C> - 1 of sample k at site s (four-channel fields are the library's
// own, 16-byte aligned)
template <int C>
__device__ __forceinline__ void load_chunk(const float2 *f, int s, int k, int K, int a0, float2 h[PC_CHUNK<C>][3]) {
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const size_t e = (((size_t)s * 3 + c) * K + k) * C + a0;
        if constexpr (C == 4) {
            const float4 v = __ldg(reinterpret_cast<const float4 *>(f + e));
            h[0][c] = make_float2(v.x, v.y);
            h[1][c] = make_float2(v.z, v.w);
        } else {
            static_assert(C == 1, "fields have one or four channels");
            h[0][c] = __ldg(f + e);
        }
    }
}

// y = M h for N channels
template <int N>
__device__ __forceinline__ void transport(const Cplx<float> M[3][3], const float2 h[N][3], float2 y[N][3]) {
#pragma unroll
    for (int a = 0; a < N; a++)
#pragma unroll
        for (int r = 0; r < 3; r++) {
            float re = 0.f, im = 0.f;
#pragma unroll
            for (int c = 0; c < 3; c++) {
                re = fmaf(M[r][c].re, h[a][c].x, fmaf(-M[r][c].im, h[a][c].y, re));
                im = fmaf(M[r][c].re, h[a][c].y, fmaf(M[r][c].im, h[a][c].x, im));
            }
            y[a][r] = make_float2(re, im);
        }
}

// The output sum of a layer as packed pairs: with w = (wr, wi) and y = (yr, yi),
// P += (wr, wr) y and N += (wi, wi) y are two packed FMAs per complex product in place of four
// scalar ones, and the output is (P.x - N.y, P.y + N.x).
template <int B>
struct MixAcc {
    float2 P[B][3], N[B][3];
};

// channels a0 .. a0 + N - 1 of the A input channels, all B output channels
template <int A, int B, int N>
__device__ __forceinline__ void mix(const float4 *ws, int a0, const float2 y[N][3], MixAcc<B> &acc) {
#pragma unroll
    for (int a = 0; a < N; a++)
#pragma unroll
        for (int b = 0; b < B; b++) {
            const float4 w = ws[b * A + a0 + a];
            const float2 wr = make_float2(w.x, w.y), wi = make_float2(w.z, w.w);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                acc.P[b][c] = __ffma2_rn(wr, y[a][c], acc.P[b][c]);
                acc.N[b][c] = __ffma2_rn(wi, y[a][c], acc.N[b][c]);
            }
        }
}

// Calls f(q, M, nb) for every link of the site: q = 1 + slot, M the gathered link, nb the neighbour.
template <int NR, typename F>
__device__ __forceinline__ void for_each_link(const PcLayerArgs &p, int s, F &&f) {
    using FatC = LinkCodec<HISQ_FP32, 18>;
    using NaikC = LinkCodec<HISQ_FP32, NR>;
    const Geom &g = p.g;
    const SiteCoord sc = decode_site(g, s, p.parity);
#pragma unroll
    for (int grp = 0; grp < FatC::GROUPS; grp++) {
        uint32_t u[FatC::WG * 4];
        FatC::load_group(p.fat, p.parity, g.Vh, s, grp, u);
#pragma unroll
        for (int l = 0; l < FatC::G; l++) {
            const int slot = grp * FatC::G + l;
            const int nb = neighbour(g, sc, s, slot >> 1, (slot & 1) ? -1 : 1);
            Cplx<float> M[3][3];
            FatC::decode(u, l, M);
            f(1 + slot, M, nb);
        }
    }
#pragma unroll
    for (int grp = 0; grp < NaikC::GROUPS; grp++) {
        uint32_t u[NaikC::WG * 4];
        NaikC::load_group(p.naik, p.parity, g.Vh, s, grp, u);
#pragma unroll
        for (int l = 0; l < NaikC::G; l++) {
            const int slot = grp * NaikC::G + l;
            const int nb = neighbour(g, sc, s, slot >> 1, (slot & 1) ? -3 : 3);
            Cplx<float> M[3][3];
            NaikC::decode(u, l, M);
            f(9 + slot, M, nb);
        }
    }
}

// Resident blocks per SM that the register budget is set for: 24 warps for the four-to-one layer of
// 18-real links, 16 for the others (more would spill).
constexpr int pc_layer_blocks(int A, int B, int NR) { return A == 4 && B == 1 && NR == 18 ? 3 : 2; }

// one thread per (site, sample); K threads share a site's links
template <int A, int B, bool ADJ, int NR>
__global__ void __launch_bounds__(256, pc_layer_blocks(A, B, NR)) pc_layer_kernel(PcLayerArgs p) {
    constexpr int N = PC_CHUNK<A>;
    __shared__ float4 ws[PC_PATHS * A * B];
    stage_weights<A, B, ADJ>(p.W, ws);
    __syncthreads();
    const int k = threadIdx.x % p.K, sl = threadIdx.x / p.K;
    for (int tile = blockIdx.x; (long)tile * p.spb < p.g.Vh; tile += gridDim.x) {
        const int s = tile * p.spb + sl;
        if (s >= p.g.Vh || sl >= p.spb) continue;
        MixAcc<B> acc;
#pragma unroll
        for (int b = 0; b < B; b++)
#pragma unroll
            for (int c = 0; c < 3; c++) acc.P[b][c] = acc.N[b][c] = make_float2(0.f, 0.f);
        if (p.in_same) {
#pragma unroll
            for (int a0 = 0; a0 < A; a0 += N) {
                float2 h[N][3];
                load_chunk<A>(p.in_same, s, k, p.K, a0, h);
                mix<A, B, N>(ws, a0, h, acc);
            }
        }
        if (p.in_opp) {
            for_each_link<NR>(p, s, [&](int q, const Cplx<float>(&M)[3][3], int nb) {
#pragma unroll
                for (int a0 = 0; a0 < A; a0 += N) {
                    float2 h[N][3], y[N][3];
                    load_chunk<A>(p.in_opp, nb, k, p.K, a0, h);
                    transport<N>(M, h, y);
                    mix<A, B, N>(ws + q * A * B, a0, y, acc);
                }
            });
        }
#pragma unroll
        for (int c = 0; c < 3; c++) {
            float2 o[B];
#pragma unroll
            for (int b = 0; b < B; b++)
                o[b] = make_float2(acc.P[b][c].x - acc.N[b][c].y, acc.P[b][c].y + acc.N[b][c].x);
            const size_t e = (((size_t)s * 3 + c) * p.K + k) * B;
            if constexpr (B == 4) {
                float4 *d = reinterpret_cast<float4 *>(p.out + e);
                d[0] = make_float4(o[0].x, o[0].y, o[1].x, o[1].y);
                d[1] = make_float4(o[2].x, o[2].y, o[3].x, o[3].y);
            } else {
                p.out[e] = o[0];
            }
        }
    }
}

// Weight gradient of a layer A -> B channels at one output parity:
//   gW[path][b][a] += sum_x sum_colour G_b(x) conj((T_path h_a)(x))   (summed over samples)
// G: [Vh][3][K][B] at the output parity.  Result: 17*B*A complex numbers (doubles) in dot_out,
// in the weight layout [path][b][a].
//
// Each of the block's eight warps owns one direction of one link kind (its two hops are two
// paths), and the warps take turns at the identity path, so a path's 2 A B sums stay in the
// registers of one warp: over a tile of p.spb sites every lane sums its (site, sample) pairs in
// FP32, then one transposing shuffle tree (2 A B - 1 shuffles) leaves component i of the warp's sum
// in lane i, which adds it to its FP64 sum.  A lane-by-lane reduction of every component of every
// site, with lane 0 adding into FP64 sums in shared memory, was bound by those additions (75% of
// the FP64 pipe, 5 ms for a 4 -> 4 layer): at 32^3 x 8 with 16 samples the loss and gradient took
// 37.6 ms, with this kernel and the packed layers above 17.8 ms; with one body of code for both hops
// and link kinds 14.6 -> 13.9 ms (between the two the forward activations were kept instead of
// recomputed); with the blocks' sums added in groups (grad_finish) and three blocks per SM for the layers
// of four weights 13.9 -> 12.95 ms.
// Lanes add up to eight (site, sample) pairs in FP32 before the warp's tree and the FP64 sum, one before:
// the gradient's error against 64 bits on eight lattices of 6400 to 110592 sites with 2 to 16 samples is
// 3.6e-8 to 8.4e-8 either way (geometric mean of the 16 ratios 0.997).
struct PcGradArgs {
    PcLayerArgs L;       // in_same, in_opp: the layer input h; spb: sites per tile; out unused
    const float2 *G;     // gradient w.r.t. the layer output at the output parity
    RedArgs red;
};

constexpr int PC_GRAD_WARPS = 8;   // four directions of two link kinds
constexpr int PC_GRAD_GROUP = 16;  // blocks whose partials are added first

// v[0 .. N): in lane l afterwards v[0] = the warp's sum of component l % N (N a power of two <= 32)
template <int N>
__device__ __forceinline__ void transpose_sum(float v[N], int lane) {
#pragma unroll
    for (int n = N; n > 1; n /= 2) {
        const int off = n / 2;
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int i = 0; i < n / 2; i++) {
            const float keep = up ? v[i + off] : v[i], send = up ? v[i] : v[i + off];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
#pragma unroll
    for (int off = N; off < 32; off *= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
}

// acc[(b A + a) 2 ..] += sum_colour G_b conj(y_a) for channels a0 .. a0 + N - 1
template <int A, int B, int N>
__device__ __forceinline__ void outer_acc(const float2 G[B][3], const float2 y[N][3], int a0, float *acc) {
#pragma unroll
    for (int a = 0; a < N; a++)
#pragma unroll
        for (int b = 0; b < B; b++) {
            float &re = acc[(b * A + a0 + a) * 2], &im = acc[(b * A + a0 + a) * 2 + 1];
#pragma unroll
            for (int c = 0; c < 3; c++) {
                re = fmaf(G[b][c].x, y[a][c].x, fmaf(G[b][c].y, y[a][c].y, re));
                im = fmaf(G[b][c].y, y[a][c].x, fmaf(-G[b][c].x, y[a][c].y, im));
            }
        }
}

template <int C>
__device__ __forceinline__ void load_all(const float2 *f, int s, int k, int K, float2 h[C][3]) {
#pragma unroll
    for (int a0 = 0; a0 < C; a0 += PC_CHUNK<C>) load_chunk<C>(f, s, k, K, a0, h + a0);
}

// link `slot` of a record (known at run time, the same for the whole warp)
template <int NR>
__device__ __forceinline__ void load_slot(const LinkField &f, int parity, int Vh, int s, int slot, Cplx<float> M[3][3]) {
    using C = LinkCodec<HISQ_FP32, NR>;
    if constexpr (C::G == 2) {
        // two 18-float links in nine words: the second starts in the middle of word 4
        const bool odd = slot & 1;
        const uint4 *w = f.words + ((size_t)parity * f.W + (slot >> 1) * 9 + (odd ? 4 : 0)) * Vh + s;
        float u[20];
#pragma unroll
        for (int j = 0; j < 5; j++) {
            const uint4 x = __ldg(w + (size_t)j * Vh);
            u[4 * j] = __uint_as_float(x.x);
            u[4 * j + 1] = __uint_as_float(x.y);
            u[4 * j + 2] = __uint_as_float(x.z);
            u[4 * j + 3] = __uint_as_float(x.w);
        }
#pragma unroll
        for (int e = 0; e < 9; e++)
            M[e / 3][e % 3] = {odd ? u[2 * e + 2] : u[2 * e], odd ? u[2 * e + 3] : u[2 * e + 1]};
    } else {
        static_assert(C::G == 4, "records of two or four links per group");
        uint32_t u[C::WG * 4];
        C::load_group(f, parity, Vh, s, slot >> 2, u);
        switch (slot & 3) {
        case 0: C::decode(u, 0, M); break;
        case 1: C::decode(u, 1, M); break;
        case 2: C::decode(u, 2, M); break;
        default: C::decode(u, 3, M);
        }
    }
}

template <int A, int B, int NR>
__device__ __forceinline__ double grad_hop(const PcGradArgs &ga, const LinkField &f, int hop, int slot, int s0, int s1,
                                           int row, int rows, int k, int lane) {
    constexpr int N = PC_CHUNK<A>, NV = 2 * A * B;
    const PcLayerArgs &p = ga.L;
    float acc[NV];
#pragma unroll
    for (int i = 0; i < NV; i++) acc[i] = 0.f;
    if (row < rows) {
#pragma unroll 1
        for (int s = s0 + row; s < s1; s += rows) {
            Cplx<float> M[3][3];
            load_slot<NR>(f, p.parity, p.g.Vh, s, slot, M);
            const SiteCoord sc = decode_site(p.g, s, p.parity);
            const int nb = neighbour_rt(p.g, sc, s, slot >> 1, (slot & 1) ? -hop : hop);
            float2 G[B][3];
            load_all<B>(ga.G, s, k, p.K, G);
#pragma unroll
            for (int a0 = 0; a0 < A; a0 += N) {
                float2 h[N][3], y[N][3];
                load_chunk<A>(p.in_opp, nb, k, p.K, a0, h);
                transport<N>(M, h, y);
                outer_acc<A, B, N>(G, y, a0, acc);
            }
        }
    }
    transpose_sum<NV>(acc, lane);
    return (double)acc[0];
}

// s[j] = sum over rows of row[r * stride + j] (four sums in flight: an FP64 add is a 64-cycle dependent
// operation), for the thread's columns j
template <int ND, typename F>
__device__ __forceinline__ void sum_rows(const double *row, size_t stride, int rows, F &&put) {
    for (int j = threadIdx.x; j < ND; j += blockDim.x) {
        double t[4] = {0.0, 0.0, 0.0, 0.0};
        int b = 0;
        for (; b + 4 <= rows; b += 4)
#pragma unroll
            for (int u = 0; u < 4; u++) t[u] += __ldcg(row + (size_t)(b + u) * stride + j);
        for (; b < rows; b++) t[0] += __ldcg(row + (size_t)b * stride + j);
        put(j, (t[0] + t[1]) + (t[2] + t[3]));
    }
}

// The sums of the blocks' ND columns (red, shared memory) into dot_out, in a fixed order and with no block
// waiting for another: the block that finishes last of its group of 16 adds the group's partials, the
// group that finishes last adds the groups' sums.  One last block adding the partials of all 304 was a
// sixth of the time of a 4 -> 4 layer's kernel, and a fence per column more before it.
// ra.counter: one counter for the groups and then one per group, zero before and after.
template <int ND>
__device__ __forceinline__ void grad_finish(const double *red, const RedArgs &ra) {
    __shared__ int last;
    const int nb = gridDim.x, g = blockIdx.x / PC_GRAD_GROUP, groups = (nb + PC_GRAD_GROUP - 1) / PC_GRAD_GROUP;
    const int size = min(PC_GRAD_GROUP, nb - g * PC_GRAD_GROUP);
    double *mine = ra.partials + (size_t)g * PC_GRAD_GROUP * ND;
    __syncthreads();
    for (int j = threadIdx.x; j < ND; j += blockDim.x) ra.partials[(size_t)blockIdx.x * ND + j] = red[j];
    __threadfence();  // publish before the ticket is taken
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ra.counter + 1 + g, 1u) == size - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    sum_rows<ND>(mine, ND, size, [&](int j, double s) { mine[j] = s; });
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        ra.counter[1 + g] = 0u;
        last = atomicAdd(ra.counter, 1u) == groups - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    sum_rows<ND>(ra.partials, (size_t)PC_GRAD_GROUP * ND, groups, [&](int j, double s) { ra.dot_out[j] = s; });
    if (threadIdx.x == 0) ra.counter[0] = 0u;
}

// three blocks per SM where the sums of a path are eight (80 registers): the loss and gradient above 1.2 %
// faster than with two; four per SM (64 registers) spill and gain nothing more.  4 -> 4 layers need the 128.
template <int A, int B, int NR>
__global__ void __launch_bounds__(32 * PC_GRAD_WARPS, A * B < 16 ? 3 : 2) pc_grad_kernel(PcGradArgs ga) {
    constexpr int N = PC_CHUNK<A>, NV = 2 * A * B, ND = PC_PATHS * NV;  // doubles per partial
    extern __shared__ double red[];
    __shared__ double same[PC_GRAD_WARPS][NV];
    const PcLayerArgs &p = ga.L;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int rows = 32 / p.K, k = lane % p.K, row = lane / p.K;  // (site, sample) pairs of a warp
    const int mu = warp & 3;
    const bool naik_kind = warp >= 4;
    double fwd = 0.0, bwd = 0.0, idn = 0.0;
    int turn = 0;
    for (int tile = blockIdx.x; (long)tile * p.spb < p.g.Vh; tile += gridDim.x, turn++) {
        const int s0 = tile * p.spb, s1 = min(s0 + p.spb, p.g.Vh);
        if (p.in_opp) {
            // one body of code for every warp and both hops where the two encodings agree: with a body per
            // hop and kind, the warps at different places of four bodies, waiting for instructions was the
            // largest stall (3.3 warps per instruction issued in a 4 -> 4 layer; now 0.04)
#pragma unroll 1
            for (int dir = 0; dir < 2; dir++) {
                double sum;
                if constexpr (NR == 18) {
                    sum = grad_hop<A, B, 18>(ga, naik_kind ? p.naik : p.fat, naik_kind ? 3 : 1, 2 * mu + dir, s0, s1, row,
                                             rows, k, lane);
                } else {
                    if (naik_kind) sum = grad_hop<A, B, NR>(ga, p.naik, 3, 2 * mu + dir, s0, s1, row, rows, k, lane);
                    else sum = grad_hop<A, B, 18>(ga, p.fat, 1, 2 * mu + dir, s0, s1, row, rows, k, lane);
                }
                if (dir) bwd += sum;
                else fwd += sum;
            }
        }
        if (p.in_same && (turn & (PC_GRAD_WARPS - 1)) == warp) {
            float acc[NV];
#pragma unroll
            for (int i = 0; i < NV; i++) acc[i] = 0.f;
            if (row < rows) {
                for (int s = s0 + row; s < s1; s += rows) {
                    float2 G[B][3];
                    load_all<B>(ga.G, s, k, p.K, G);
#pragma unroll
                    for (int a0 = 0; a0 < A; a0 += N) {
                        float2 h[N][3];
                        load_chunk<A>(p.in_same, s, k, p.K, a0, h);
                        outer_acc<A, B, N>(G, h, a0, acc);
                    }
                }
            }
            transpose_sum<NV>(acc, lane);
            idn += (double)acc[0];
        }
    }
    if (lane < NV) {
        const int path = slot_path(2 * mu + (naik_kind ? 8 : 0));  // forward hop; the backward one follows
        red[path * NV + lane] = fwd;
        red[(path + 1) * NV + lane] = -bwd;                        // backward slots hold -U^dag
        same[warp][lane] = idn;
    }
    __syncthreads();
    if (threadIdx.x < NV) {
        double s = 0.0;
        for (int w = 0; w < PC_GRAD_WARPS; w++) s += same[w][threadIdx.x];
        red[threadIdx.x] = s;
    }
    grad_finish<ND>(red, ga.red);
}

}  // namespace hisq
