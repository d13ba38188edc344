// The 16-bit Dslash of a bundle on the tensor cores (mma.sync), one warp per output site.
//
// The stencil of one site is, for the right-hand sides of a group of 16, a sum over its 16 links of a
// 16 x 6 matrix (the neighbour's colour vectors, one right-hand side per row: three re, im pairs as
// stored) times the 6 x 6 real form of the link.  In the fragment layouts of m16n8k8 and m16n8k16
// (g = lane / 4, q = lane % 4) A has rows g and g + 8 and k = 2 q, 2 q + 1 (+ 8), B has the same k in
// column g, C rows g and g + 8 and columns 2 q, 2 q + 1.  So lane (g, q < 3) feeds colour component q of
// two right-hand sides exactly as their 16-bit words lie in memory, holds in B the link entry (row
// g / 2, column q), and receives the real and imaginary part of colour q of the same two right-hand
// sides: nothing is converted and nothing moves between lanes.
//   FP16: one m16n8k8 per link; each neighbour record has its own FP32 scale, applied in FP32 to the
//         link's product.  The lane's rows are right-hand sides g and g + 8 of the group.  Lanes q = 3
//         read the scales for their quads and feed zeros.
//   BF16: no vector scales, so two links share one m16n8k16 and accumulate in the tensor core.  The
//         lane's rows are right-hand sides 2 g and 2 g + 1, one 8-byte load.  Lanes q = 3 share
//         component 0 with lanes q = 0, each against half of its link entries (zeros in one of them
//         would turn an infinity into NaN).
// Products of 16-bit values are exact and accumulators FP32 wide, but the tensor core adds with its own
// rounding, towards zero: against 64-bit sums of the same stored values (16^3 x 8 and 28 x 20 x 12 x 10, 2 to
// 16 right-hand sides) an FP16 output's largest component is off by 7.6e-8 rms, 3.4e-8 of it common to all;
// SIMT kernels by 2.1e-7 rms and nothing in common.  A dot product over the lattice averages the rms away and
// keeps the common part: 3.4e-8 (FP16) and 5.5e-8 (BF16) of it, SIMT 1e-9.  Rounding the links and
// vectors to 16 bits puts far more on the same dots (BF16 at 28 x 20 x 36 x 10: 9.6e-6).
//
// The SIMT kernels spend two thirds of their FMA-pipe cycles on the 36 products of every link and right-hand
// side and a fifth on conversions.  Here what is left is loads, addresses and scales, and the latency of the
// loads (half of the warps' time; it is that of L1 and L2: lattices within L2 take as long per site, and
// requests into L2 ahead of use only slowed it down).
//
// A warp visits a run of consecutive sites of one x-row, U at a time: the hops in y, z and t are then
// the same index offsets for the whole run, U sites share the addresses of those neighbours, and their
// hops in x reach U + 3 sites instead of 4 U.  The warps of a block take rows adjacent in y, whose
// neighbours they find in one another's L1 lines.  Dslash at 64^3 x 16, us, SIMT / this kernel (U = 4):
// FP16 16 right-hand sides 1372 / 990, 12: 1174 / 1053, 8: 691 / 771; BF16 16: 1354 / 647, 12: 1254 / 748,
// 8: 681 / 578, 4: 373 / 820 (the tuner takes the faster).  U = 1 and 2 with 16: FP16 1238 and 1066, BF16
// 869 and 664.
//
// Links: a second copy of the 18-real records in the order the B fragments want them: 16-byte word
// ((p Vh + s) 2 + j) 9 + 3 a + b holds the entries (a, b) of links 4 j .. 4 j + 3 as 16-bit (re, im), for
// BF16 halved (exactly) for b = 0.
#pragma once
#include "dslash_kernel.cuh"

namespace hisq {

constexpr int MMA_GROUP = 16;    // right-hand sides per warp (rows of the products)
constexpr int MMA_MAX_N = 32;    // two groups at most
constexpr int MMA_THREADS = 256; // of the separate kernel

struct MmaField {
    const uint4 *frag;    // [2][Vh][2][9]
    const float *scale;   // [2][Vh]
};

struct MmaC {
    float c[4];
};

__device__ __forceinline__ MmaC mma_f16_k8(uint32_t a0, uint32_t a1, uint32_t b) {
    MmaC d;
    asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%7,%7,%7,%7};"
        : "=f"(d.c[0]), "=f"(d.c[1]), "=f"(d.c[2]), "=f"(d.c[3])
        : "r"(a0), "r"(a1), "r"(b), "f"(0.f));
    return d;
}

__device__ __forceinline__ void mma_bf16_k16(MmaC &d, uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                             uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d.c[0]), "+f"(d.c[1]), "+f"(d.c[2]), "+f"(d.c[3])
        : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The bundle sizes with a compile-time layout (strides and the distance of a lane's two right-hand sides
// as immediate offsets): N = 16 and, for BF16, N = 8; N = 0 any other.  Sites that are worked on together.
template <int P>
__host__ __device__ constexpr int mma_n(int n) {
    return n == 16 ? 16 : n == 8 && P == HISQ_BF16 ? 8 : 0;
}
__host__ __device__ constexpr int mma_u(int half) { return half % 4 == 0 ? 4 : half % 2 == 0 ? 2 : 1; }

// What a lane needs to know about its place in the fragments.
template <int P, int N>
struct MmaLane {
    int q;               // colour component of the lane (3: none)
    int r_lo, r_hi;      // its two right-hand sides
    bool has_lo, has_hi; // whether they exist
    uint32_t at;         // byte offset of its first word within a site's bundle (clamped to existing ones;
                         // FP16: lane q = 3 has the scale)
    uint32_t step;       // FP16, N = 0: bytes from the first right-hand side's words to the second's
    uint32_t bytes;      // per site of the bundle
    uint32_t link;       // word of the lane's link entry within a group of nine
    uint32_t perm, flip, keep;  // B operand from the stored entry: byte order, sign bits, mask (FP16)

    __device__ __forceinline__ MmaLane(int lane, int n, int group) {
        const int g = lane >> 2, qc = (lane & 3) < 3 ? lane & 3 : 0;
        q = lane & 3;
        if constexpr (P == HISQ_FP16) {
            r_lo = MMA_GROUP * group + g;
            r_hi = r_lo + 8;
            const uint32_t cl = min(r_lo, n - 1), ch = min(r_hi, n - 1);
            at = cl * 16 + q * 4;
            step = (ch - cl) * 16;
            bytes = n * 16;
        } else {
            r_lo = MMA_GROUP * group + 2 * g;  // n is even
            r_hi = r_lo + 1;
            at = (qc * n + min(r_lo, n - 2)) * 4;
            step = 0;
            bytes = n * 12;
        }
        has_lo = r_lo < n;
        has_hi = r_hi < n;
        link = min(g >> 1, 2) * 3 + qc;
        // column 2 a (real part): (re, -im); column 2 a + 1 (imaginary part): (im, re)
        perm = (g & 1) ? 0x1032 : 0x3210;
        flip = (g & 1) ? 0u : 0x80000000u;
        keep = q < 3 ? 0xffffffffu : 0u;
    }
    __device__ __forceinline__ uint32_t stride() const { return N ? N * (P == HISQ_FP16 ? 16 : 12) : bytes; }
    __device__ __forceinline__ uint32_t b(uint32_t entry) const {
        const uint32_t w = __byte_perm(entry, 0, perm) ^ flip;
        return P == HISQ_FP16 ? w & keep : w;
    }
};

// one neighbour's words of a lane, and (FP16, once mma_ready) the two scales
struct MmaWords {
    uint32_t lo, hi;
    float slo, shi;
};

// v: the lane's words at the site
template <int P, int N, bool COHERENT>
__device__ __forceinline__ MmaWords mma_load(const MmaLane<P, N> &L, const char *v) {
    MmaWords w;
    w.slo = w.shi = 0.f;
    if constexpr (P == HISQ_FP16) {
        w.lo = vld<COHERENT>(reinterpret_cast<const uint32_t *>(v));
        w.hi = vld<COHERENT>(reinterpret_cast<const uint32_t *>(v + (N == 16 ? 128u : L.step)));
    } else {
        const uint2 x = vld<COHERENT>(reinterpret_cast<const uint2 *>(v));
        w.lo = x.x;
        w.hi = x.y;
    }
    return w;
}

// FP16: the quad's scales from its lane q = 3, whose own words become zero
template <int P, int N>
__device__ __forceinline__ void mma_ready(const MmaLane<P, N> &L, MmaWords &w) {
    if constexpr (P == HISQ_FP16) {
        const int src = (threadIdx.x & 31) | 3;
        w.slo = __uint_as_float(__shfl_sync(0xffffffffu, w.lo, src));
        w.lo &= L.keep;
        w.shi = __uint_as_float(__shfl_sync(0xffffffffu, w.hi, src));
        w.hi &= L.keep;
    }
}

// a bundle as a lane addresses it: its words at site 0
template <int P, int N>
__device__ __forceinline__ const char *mma_ptr(const MmaLane<P, N> &L, const void *base) {
    return reinterpret_cast<const char *>(base) + L.at;
}

// A run of sites of one row: everything about the neighbours that does not change along x.
struct MmaRun {
    int row;        // even-odd index of the row's first site
    int x0, x1;     // sites [row + x0, row + x1)
    int odd;        // x = 2 xh + odd
    int off[2][6];  // index offsets of the hops +h, -h in y, z, t (h = 1, 3)
};

// Runs are numbered so that the warps of a block (consecutive numbers) take up to eight rows adjacent
// in y at the same x: run u = (8 rows of group rg) x (segment seg of the row), seg before rg.
struct MmaRuns {
    int len, nseg, rows, count;
};

__host__ __device__ __forceinline__ MmaRuns mma_runs(const Geom &g, int sites, int len) {
    MmaRuns R;
    R.len = len < g.half ? len : g.half;
    const int u = mma_u(g.half);
    R.len = (R.len + u - 1) / u * u;
    R.nseg = (g.half + R.len - 1) / R.len;
    R.rows = sites / g.half;
    R.count = (R.rows + 7) / 8 * 8 * R.nseg;
    return R;
}

// Sites per run for a grid of `warps` warps: the longest run that leaves at most 7% of the warps' time
// idle in the last round (short runs repeat the row's index arithmetic; on small lattices long ones
// leave warps without work).
inline int mma_run_length(const Geom &g, int sites, long warps) {
    int best = 1;
    double best_eff = 0.0;
    for (int len = 16; len >= 1; len /= 2) {
        const MmaRuns R = mma_runs(g, sites, len);
        const long rounds = (R.count + warps - 1) / warps;
        const double eff = (double)sites / ((double)rounds * R.len * warps);
        if (eff >= 0.93) return len;
        if (eff > best_eff + 0.01) {
            best_eff = eff;
            best = len;
        }
    }
    return best;
}

// false: no such run (the last group of rows may be short)
__device__ __forceinline__ bool mma_run(const Geom &g, const MmaRuns &R, int u, int parity, MmaRun &run) {
    const int rg = u / (8 * R.nseg), rem = u - rg * 8 * R.nseg, seg = rem >> 3, r = rg * 8 + (rem & 7);
    if (r >= R.rows) return false;
    run.row = visit_site(g, r * g.half);
    run.x0 = seg * R.len;
    run.x1 = min(run.x0 + R.len, g.half);
    const SiteCoord sc = decode_site(g, run.row, parity);
    run.odd = sc.c[0];  // x of the row's first site: 0 or 1
#pragma unroll
    for (int kind = 0; kind < 2; kind++)
#pragma unroll
        for (int mu = 1; mu < 4; mu++)
#pragma unroll
            for (int dir = 0; dir < 2; dir++) {
                const int hop = kind ? 3 : 1;
                run.off[kind][2 * (mu - 1) + dir] = neighbour(g, sc, 0, mu, dir ? -hop : hop);
            }
    return true;
}

// One field's share of a link: FP16 a product of its own, scaled by the neighbours' scales; BF16 half of a
// product of two links, accumulated in the tensor core.
template <int P, int N>
__device__ __forceinline__ void mma_link_pair(const MmaLane<P, N> &L, const MmaWords &v0, const MmaWords &v1,
                                              uint32_t e0, uint32_t e1, MmaC &acc) {
    if constexpr (P == HISQ_FP16) {
        const MmaWords *v[2] = {&v0, &v1};
        const uint32_t e[2] = {e0, e1};
#pragma unroll
        for (int i = 0; i < 2; i++) {
            const MmaC d = mma_f16_k8(v[i]->lo, v[i]->hi, L.b(e[i]));
            acc.c[0] = fmaf(v[i]->slo, d.c[0], acc.c[0]);
            acc.c[1] = fmaf(v[i]->slo, d.c[1], acc.c[1]);
            acc.c[2] = fmaf(v[i]->shi, d.c[2], acc.c[2]);
            acc.c[3] = fmaf(v[i]->shi, d.c[3], acc.c[3]);
        }
    } else {
        mma_bf16_k16(acc, v0.lo, v0.hi, v1.lo, v1.hi, L.b(e0), L.b(e1));
    }
}

// D in at the U sites row + xh .., for the lane's colour component of its two right-hand sides.  The hops
// in x of U consecutive sites reach U + 3 sites of the opposite parity's row: site u takes number u + 2
// (x + 1), u + 1 (x - 1), u + 3 (x + 3) and u (x - 3) of those that start at xh + odd - 2.
template <int P, int N, int U, bool COHERENT>
__device__ __forceinline__ void mma_sites(const Geom &g, const MmaField &fat, const MmaField &naik,
                                          const MmaLane<P, N> &L, const MmaRun &run, int parity, int xh, const char *in,
                                          MmaC w[U]) {
    const int s = run.row + xh;
    const size_t site = (size_t)parity * g.Vh + s;
    const uint32_t stride = L.stride();
    MmaWords vx[U + 3];
#pragma unroll
    for (int j = 0; j < U + 3; j++) {
        int i = xh + run.odd - 2 + j;
        i += i < 0 ? g.half : 0;
        i -= i >= g.half ? g.half : 0;
        vx[j] = mma_load<P, N, COHERENT>(L, in + (size_t)(uint32_t)(run.row + i) * stride);
    }
#pragma unroll
    for (int kind = 0; kind < 2; kind++) {
        const uint4 *frag = (kind ? naik.frag : fat.frag) + site * 18 + L.link;
        MmaC acc[U];
        uint4 e[U];
        MmaWords v[U][6];
#pragma unroll
        for (int u = 0; u < U; u++) {
            acc[u] = {{0.f, 0.f, 0.f, 0.f}};
            e[u] = __ldg(frag + 18 * u);
        }
#pragma unroll
        for (int i = 0; i < 6; i++) {
            const char *p = in + (size_t)(uint32_t)(s + run.off[kind][i]) * stride;
#pragma unroll
            for (int u = 0; u < U; u++) v[u][i] = mma_load<P, N, COHERENT>(L, p + u * stride);
        }
        if (kind == 0) {
#pragma unroll
            for (int j = 0; j < U + 3; j++) mma_ready(L, vx[j]);
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            mma_link_pair(L, vx[kind ? u + 3 : u + 2], vx[kind ? u : u + 1], e[u].x, e[u].y, acc[u]);
            mma_ready(L, v[u][0]);
            mma_ready(L, v[u][1]);
            mma_link_pair(L, v[u][0], v[u][1], e[u].z, e[u].w, acc[u]);
        }
#pragma unroll
        for (int u = 0; u < U; u++) e[u] = __ldg(frag + 18 * u + 9);
#pragma unroll
        for (int u = 0; u < U; u++) {
#pragma unroll
            for (int i = 2; i < 6; i++) mma_ready(L, v[u][i]);
            mma_link_pair(L, v[u][2], v[u][3], e[u].x, e[u].y, acc[u]);
            mma_link_pair(L, v[u][4], v[u][5], e[u].z, e[u].w, acc[u]);
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const float sf = __ldg((kind ? naik.scale : fat.scale) + site + u);
#pragma unroll
            for (int i = 0; i < 4; i++) w[u].c[i] = kind ? fmaf(sf, acc[u].c[i], w[u].c[i]) : sf * acc[u].c[i];
        }
    }
}

// stores the lane's components of the site's output vectors (FP16: with the quad's shared scales); lo, hi:
// which of the two right-hand sides
template <int P, int N>
__device__ __forceinline__ void mma_store(const MmaLane<P, N> &L, const char *out, int s, const MmaC &w, bool lo,
                                          bool hi) {
    const size_t at = (size_t)(uint32_t)s * L.stride();
    if constexpr (P == HISQ_FP16) {
        char *d = const_cast<char *>(out + at);
        float m0 = L.q < 3 ? fmaxf(fabsf(w.c[0]), fabsf(w.c[1])) : 0.f;
        float m1 = L.q < 3 ? fmaxf(fabsf(w.c[2]), fabsf(w.c[3])) : 0.f;
#pragma unroll
        for (int off = 1; off < 4; off <<= 1) {
            m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, off));
            m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, off));
        }
        const float i0 = m0 > 0.f ? 1.f / m0 : 0.f, i1 = m1 > 0.f ? 1.f / m1 : 0.f;
        const __half2 h0 = __floats2half2_rn(w.c[0] * i0, w.c[1] * i0), h1 = __floats2half2_rn(w.c[2] * i1, w.c[3] * i1);
        const uint32_t u0 = L.q < 3 ? *reinterpret_cast<const uint32_t *>(&h0) : __float_as_uint(m0);
        const uint32_t u1 = L.q < 3 ? *reinterpret_cast<const uint32_t *>(&h1) : __float_as_uint(m1);
        if (lo) *reinterpret_cast<uint32_t *>(d) = u0;
        if (hi) *reinterpret_cast<uint32_t *>(d + (N == 16 ? 128u : L.step)) = u1;
    } else {
        const __nv_bfloat162 b0 = __floats2bfloat162_rn(w.c[0], w.c[1]), b1 = __floats2bfloat162_rn(w.c[2], w.c[3]);
        const uint32_t u0 = *reinterpret_cast<const uint32_t *>(&b0), u1 = *reinterpret_cast<const uint32_t *>(&b1);
        if (L.q < 3) {
            uint32_t *d = reinterpret_cast<uint32_t *>(const_cast<char *>(out + at));
            if (lo && hi) {
                *reinterpret_cast<uint2 *>(d) = make_uint2(u0, u1);
            } else {
                if (lo) d[0] = u0;
                if (hi) d[1] = u1;
            }
        }
    }
}

// w = m^2 p - D t for the lane's components, and the lane's parts of Re <p, w> (d[0], d[1]: its two
// right-hand sides) and |w|^2 (d[2], d[3]); lanes without a component contribute nothing
template <int P, int N, bool COHERENT>
__device__ __forceinline__ void mma_aop(const MmaLane<P, N> &L, const char *pvec, int s, float m2_lo, float m2_hi,
                                        MmaC &w, float d[4]) {
    const size_t at = (size_t)(uint32_t)s * L.stride();
    MmaWords v = mma_load<P, N, COHERENT>(L, pvec + at);
    mma_ready(L, v);
    float2 p0, p1;
    if constexpr (P == HISQ_FP16) {
        p0 = __half22float2(*reinterpret_cast<const __half2 *>(&v.lo));
        p1 = __half22float2(*reinterpret_cast<const __half2 *>(&v.hi));
        p0 = f2(p0.x * v.slo, p0.y * v.slo);
        p1 = f2(p1.x * v.shi, p1.y * v.shi);
    } else {
        p0 = f2(__uint_as_float(v.lo << 16), __uint_as_float(v.lo & 0xffff0000u));
        p1 = f2(__uint_as_float(v.hi << 16), __uint_as_float(v.hi & 0xffff0000u));
    }
    w.c[0] = m2_lo * p0.x - w.c[0];
    w.c[1] = m2_lo * p0.y - w.c[1];
    w.c[2] = m2_hi * p1.x - w.c[2];
    w.c[3] = m2_hi * p1.y - w.c[3];
    const bool own = L.q < 3;
    d[0] = own ? p0.x * w.c[0] + p0.y * w.c[1] : 0.f;
    d[1] = own ? p1.x * w.c[2] + p1.y * w.c[3] : 0.f;
    d[2] = own ? w.c[0] * w.c[0] + w.c[1] * w.c[1] : 0.f;
    d[3] = own ? w.c[2] * w.c[2] + w.c[3] * w.c[3] : 0.f;
}

// the sums of d[0 .. 4) over the four lanes of a quad: lane q is left with that of d[q]
__device__ __forceinline__ float mma_quad_sums(const float d[4], int q) {
    const bool up = q & 2;
    const float a0 = (up ? d[2] : d[0]) + __shfl_xor_sync(0xffffffffu, up ? d[0] : d[2], 2);
    const float a1 = (up ? d[3] : d[1]) + __shfl_xor_sync(0xffffffffu, up ? d[1] : d[3], 2);
    const bool odd = q & 1;
    return (odd ? a1 : a0) + __shfl_xor_sync(0xffffffffu, odd ? a0 : a1, 1);
}

// The sites of a run, U at a time (rows have a multiple of U sites, runs too): f(s, w) for each
template <int P, int N, int U, bool COHERENT, class F>
__device__ __forceinline__ void mma_run_sites(const Geom &g, const MmaField &fat, const MmaField &naik,
                                              const MmaLane<P, N> &L, const MmaRun &run, int parity, const char *in,
                                              F &&f) {
    for (int xh = run.x0; xh < run.x1; xh += U) {
        MmaC w[U];
        mma_sites<P, N, U, COHERENT>(g, fat, naik, L, run, parity, xh, in, w);
#pragma unroll
        for (int u = 0; u < U; u++) f(run.row + xh + u, w[u]);
    }
}

// Resident blocks per SM that the register budget of the separate kernel is set for (measured with U = 4 at
// 64^3 x 16): FP16 2 (16 right-hand sides 990 us; 3: 1033, 4: 1205), BF16 3 with N = 16 (647; 2: 699) and
// N = 8, else 2.
constexpr int mma_blocks(int P, int N) { return P == HISQ_BF16 && N ? 3 : 2; }

// Separate kernel: EPI_PLAIN or EPI_AOP of a whole parity, n <= MMA_MAX_N right-hand sides in a.t groups
// (warps of a block alternate over the groups); a.spb = sites per run, a multiple of U.
template <int P, int EPI, int N, int U>
__global__ void __launch_bounds__(MMA_THREADS, mma_blocks(P, N)) dslash_mma_kernel(KArgs a, MmaField fat, MmaField naik) {
    extern __shared__ double red[];
    if (a.gate && *a.gate == 0) return;
    const Geom &g = a.g;
    const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0);
    const int t = N ? 1 : a.t, group = warp % t, slots = (MMA_THREADS / 32) / t;
    const MmaLane<P, N> L(lane, N ? N : a.n, group);
    const bool lo = L.has_lo && (!a.active || a.active[L.r_lo]), hi = L.has_hi && (!a.active || a.active[L.r_hi]);
    const MmaRuns R = mma_runs(g, g.Vh, a.spb);
    const char *in = mma_ptr(L, a.in), *out = mma_ptr(L, a.out), *p = mma_ptr(L, a.axpy);
    const float m2 = (float)a.mass2;
    double sum = 0.0;
    for (int u = blockIdx.x * slots + warp / t; u < R.count; u += gridDim.x * slots) {
        MmaRun run;
        if (!mma_run(g, R, u, a.parity, run)) continue;
        mma_run_sites<P, N, U, false>(g, fat, naik, L, run, a.parity, in, [&](int s, MmaC &w) {
            if constexpr (EPI == EPI_AOP) {
                float d[4];
                mma_aop<P, N, false>(L, p, s, m2, m2, w, d);
                sum += (double)mma_quad_sums(d, L.q);
            }
            mma_store(L, out, s, w, lo, hi);
        });
    }
    if constexpr (EPI == EPI_AOP) {
        const int rows = MMA_THREADS / 32;
        for (int i = threadIdx.x; i < rows * a.n; i += blockDim.x) red[i] = 0.0;
        __syncthreads();
        if (L.q == 0 && lo) red[warp * a.n + L.r_lo] = sum;
        if (L.q == 1 && hi) red[warp * a.n + L.r_hi] = sum;
        block_reduce_finish(red, rows, a.n, a.n, a.red);
    }
}

template <int P, int EPI, int N>
inline const void *mma_kernel_u(int half) {
    switch (mma_u(half)) {
    case 4: return (const void *)dslash_mma_kernel<P, EPI, N, 4>;
    case 2: return (const void *)dslash_mma_kernel<P, EPI, N, 2>;
    default: return (const void *)dslash_mma_kernel<P, EPI, N, 1>;
    }
}

template <int P, int EPI>
inline const void *mma_kernel_ptr(int n, int half) {
    if (mma_n<P>(n) == 16) return mma_kernel_u<P, EPI, 16>(half);
    if constexpr (P == HISQ_BF16)
        if (mma_n<P>(n) == 8) return mma_kernel_u<P, EPI, 8>(half);
    return mma_kernel_u<P, EPI, 0>(half);
}

template <int P, int EPI>
inline cudaError_t launch_mma_one(KArgs a, MmaField fat, MmaField naik, size_t smem, int num_sms, cudaStream_t stream,
                                  int *grid_out) {
    const void *k = mma_kernel_ptr<P, EPI>(a.n, a.g.half);
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, MMA_THREADS, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    const int slots = MMA_THREADS / 32 / a.t;
    const long tiles = (mma_runs(a.g, a.g.Vh, a.spb).count + slots - 1) / slots;
    int grid = (int)balanced_grid(tiles, std::min((long)per_sm * num_sms, tiles));
    if (EPI != EPI_PLAIN) grid = std::min(grid, a.max_grid);
    if (grid_out) *grid_out = grid;
    void *args[] = {&a, &fat, &naik};
    return cudaLaunchKernel(k, grid, MMA_THREADS, args, smem, stream);
}

}  // namespace hisq
