// Double-single ("ds") arithmetic: the FP64-accurate residual recomputation r = b - A x of the
// mixed-precision solver (the reliable update) on the FP32 pipe.
//
// A real x is held as two floats, hi = fl32(x) and lo = fl32(x - hi), so that hi + lo equals x to
// within 2^-48 |x|.  A product of two such numbers keeps the exact product of the high parts,
// split into its rounded value p = fl(a_hi b_hi) and its rounding error fma(a_hi, b_hi, -p)
// (Dekker 1971, with a fused multiply-add in place of operand splitting), plus the two cross
// terms a_hi b_lo and a_lo b_hi (a_lo b_lo is below 2^-48 of the product and dropped).  Sums of
// products add the rounded parts with Knuth's two-sum, which returns the rounding error of a
// float addition exactly, and gather every error and cross term in a second float accumulator:
// the cascaded summation of Ogita, Rump and Oishi (2005), whose result is as accurate as a sum
// computed in twice the working precision.  On this part the FP32 pipe issues 64 times as many
// operations per cycle as the FP64 pipe, so the ten float operations a real multiply-add
// costs here run about six times faster than one FP64 fused multiply-add.
//
// The error-free steps use the rounding intrinsics (__fmul_rn, __fadd_rn, __fsub_rn, __fmaf_rn),
// which the compiler neither contracts into fused operations nor reorders, or their packed forms below.
//
// Storage: a ds link record has the FP64 record's layout (16 bytes per complex number) with every
// complex number as the float4 (re_hi, im_hi, re_lo, im_lo); a ds colour vector bundle has the FP64
// bundle's layout with every complex number (re, im) stored as the float4 (re_hi, re_lo, im_hi, im_lo).
#pragma once
#include "hisq_internal.cuh"

namespace hisq {

struct dsacc {
    float hi, lo;
};

// A complex ds accumulator, real and imaginary part in the two halves of a packed pair.
struct dscplx {
    float2 hi, lo;
    __device__ __forceinline__ dsacc re() const { return {hi.x, lo.x}; }
    __device__ __forceinline__ dsacc im() const { return {hi.y, lo.y}; }
};

// Packed operations on (re, im) with one rounding each, written in PTX.  A packed product followed by a
// packed sum is fused into one multiply-add by the assembler in spite of the .rn, which two-sum does not
// survive (errors of 1e-8 in place of 1e-13); a product plus zero is not.
union ds_pair {
    float2 f;
    unsigned long long u;
    __device__ __forceinline__ ds_pair(float2 x) : f(x) {}
    __device__ __forceinline__ ds_pair() {}
};
__device__ __forceinline__ float2 ds_mul2(ds_pair a, ds_pair b) {
    ds_pair d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d.u) : "l"(a.u), "l"(b.u), "l"(0ull));
    return d.f;
}
__device__ __forceinline__ float2 ds_add2(ds_pair a, ds_pair b) {
    ds_pair d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d.u) : "l"(a.u), "l"(b.u));
    return d.f;
}
__device__ __forceinline__ float2 ds_fma2(ds_pair a, ds_pair b, ds_pair c) {
    ds_pair d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d.u) : "l"(a.u), "l"(b.u), "l"(c.u));
    return d.f;
}
__device__ __forceinline__ float2 ds_sub2(float2 a, float2 b) { return ds_fma2(b, make_float2(-1.f, -1.f), a); }

// s += a b, both halves, for ds numbers a = (a_hi, a_lo), b = (b_hi, b_lo).  With p = fl(a_hi b_hi) and
// t = fl(s.hi + p), two-sum gives z = fl(t - s.hi) and the error (s.hi - (t - z)) + (p - z); p - z is exact,
// so one fused multiply-add, a_hi b_hi - z, is that second part together with the product's own error
// a_hi b_hi - p: ten operations in place of twelve, the same error.  (nz = s.hi - t = -z exactly.)
// Packed against scalar: half the instructions and twice the independent work of each, on kernels that keep
// the FP32 pipe 40 % busy (latency, 16 and fewer warps per SM): residual of 4 right-hand sides at 32^3 x 8
// 403 -> 347 us, of one 160 -> 142, recomputations of the 64^3 x 16 solve of 16 171 -> 157 ms.
__device__ __forceinline__ void ds_mac(dscplx &s, float2 a_hi, float2 a_lo, float2 b_hi, float2 b_lo) {
    const float2 p = ds_mul2(a_hi, b_hi);
    const float2 t = ds_add2(s.hi, p);
    const float2 nz = ds_sub2(s.hi, t);
    const float2 err = ds_add2(ds_sub2(s.hi, ds_add2(t, nz)), ds_fma2(a_hi, b_hi, nz));
    float2 lo = ds_fma2(a_hi, b_lo, s.lo);
    lo = ds_fma2(a_lo, b_hi, lo);
    s.hi = t;
    s.lo = ds_add2(lo, err);
}

// the pair (hi, lo) with hi = fl(hi + lo): the accumulator in the storage form
__device__ __forceinline__ dsacc ds_normalize(dsacc s) {
    const float t = __fadd_rn(s.hi, s.lo);
    const float z = __fsub_rn(t, s.hi);
    const float err = __fadd_rn(__fsub_rn(s.hi, __fsub_rn(t, z)), __fsub_rn(s.lo, z));
    return {t, err};
}

// this lane's accumulator plus that of the lane `off` away: two-sum of the high parts, everything else low
__device__ __forceinline__ dsacc ds_add_lane(dsacc s, int off) {
    const float hi = __shfl_xor_sync(0xffffffffu, s.hi, off), lo = __shfl_xor_sync(0xffffffffu, s.lo, off);
    const float t = __fadd_rn(s.hi, hi);
    const float z = __fsub_rn(t, s.hi);
    const float err = __fadd_rn(__fsub_rn(s.hi, __fsub_rn(t, z)), __fsub_rn(hi, z));
    return {t, __fadd_rn(__fadd_rn(s.lo, lo), err)};
}
__device__ __forceinline__ dscplx ds_add_lane(const dscplx &s, int off) {
    const dsacc re = ds_add_lane(s.re(), off), im = ds_add_lane(s.im(), off);
    return {make_float2(re.hi, im.hi), make_float2(re.lo, im.lo)};
}

__device__ __forceinline__ double ds_value(dsacc s) { return (double)s.hi + (double)s.lo; }

__device__ __forceinline__ void ds_split(double x, float &hi, float &lo) {
    hi = __double2float_rn(x);
    lo = __double2float_rn(x - (double)hi);
}

// The ds colour-vector bundle: float4 per complex number at (s * 3 + c) * n + r, like the FP64 bundle's
// double2.
template <bool COHERENT>
__device__ __forceinline__ float4 ds_load(const float4 *v, long idx) {
    if constexpr (COHERENT) return __ldcg(v + idx);
    else return __ldg(v + idx);
}

__device__ __forceinline__ void ds_store3(float4 *v, int n, long s, int r, const dscplx w[3]) {
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const dsacc re = ds_normalize(w[c].re()), im = ds_normalize(w[c].im());
        v[(s * 3 + c) * n + r] = make_float4(re.hi, re.lo, im.hi, im.lo);
    }
}

// acc[a] += M_ab v_b for the three rows a of column b of one ds link: m[a] = the 16-byte word of
// entry (a, b), i.e. the floats (re_hi, im_hi, re_lo, im_lo), and one ds colour component v_b.
// (mr, mi) vr first, then (-mi, mr) vi: both parts of a complex number in one packed operation.
// The six accumulators (three rows, real and imaginary part) are independent chains.
__device__ __forceinline__ void ds_column_acc(const uint4 m[3], const float4 vb, dscplx acc[3]) {
    const float2 vr_hi = make_float2(vb.x, vb.x), vr_lo = make_float2(vb.y, vb.y);
    const float2 vi_hi = make_float2(vb.z, vb.z), vi_lo = make_float2(vb.w, vb.w);
#pragma unroll
    for (int a = 0; a < 3; a++)
        ds_mac(acc[a], make_float2(__uint_as_float(m[a].x), __uint_as_float(m[a].y)),
               make_float2(__uint_as_float(m[a].z), __uint_as_float(m[a].w)), vr_hi, vr_lo);
#pragma unroll
    for (int a = 0; a < 3; a++)
        ds_mac(acc[a], make_float2(-__uint_as_float(m[a].y), __uint_as_float(m[a].x)),
               make_float2(-__uint_as_float(m[a].w), __uint_as_float(m[a].z)), vi_hi, vi_lo);
}

// the 9 words of one link of a ds record and the neighbour vectors it multiplies
template <int R, bool COHERENT>
struct DsOperands {
    uint4 m[9];        // entry (a, b) in word 3 a + b
    float4 v[R][3];
    __device__ __forceinline__ void load(const uint4 *words, size_t plane, int nb, const float4 *in, int n,
                                         const int rr[R], const bool act[R]) {
#pragma unroll
        for (int j = 0; j < 9; j++) m[j] = __ldg(words + j * plane);
#pragma unroll
        for (int r = 0; r < R; r++)
#pragma unroll
            for (int c = 0; c < 3; c++)
                v[r][c] = act[r] ? ds_load<COHERENT>(in, ((long)nb * 3 + c) * n + rr[r]) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __device__ __forceinline__ void apply(dscplx acc[R][3]) const {
#pragma unroll
        for (int b = 0; b < 3; b++) {
            const uint4 col[3] = {m[b], m[3 + b], m[6 + b]};
#pragma unroll
            for (int r = 0; r < R; r++) ds_column_acc(col, v[r][b], acc[r]);
        }
    }
};

// The stencil of Eq. (3) at output site s of parity `parity` in ds arithmetic for the R
// right-hand sides rr[0..R) of the ds input bundle `in` (n right-hand sides): the 8 fat and 8 Naik
// links of the site's gathered ds records (slot 2 mu forward, 2 mu + 1 the backward -U^dagger, as
// in every other precision) times the neighbouring input vectors, summed into acc.  The loop runs over
// the eight (kind, direction) pairs, both hops of a direction per step, column by column (six
// independent accumulation chains); without PREFETCH a lane can take the pairs [k0, k1) only.  With
// PREFETCH the operands of each link are requested while the link before it is applied, in two sets of
// registers that take turns (one set copied into the other after every link cost 48 moves beside 360
// FP32 operations).  One link per step with its rows loaded just before their use against both hops of
// a direction per step, all of a link's words at once: recomputations of the 64^3 x 16 solve 198 / 188 ms,
// of the 32^3 x 8 single solve 1.24 / 0.98 ms.
template <int R, bool COHERENT, bool PREFETCH = false>
__device__ __forceinline__ void ds_site_stencil(const Geom &g, const LinkField &fat, const LinkField &naik, int parity,
                                                const float4 *in, int n, int s, const int rr[R], const bool act[R],
                                                dscplx acc[R][3], int k0 = 0, int k1 = 8) {
    const SiteCoord sc = decode_site(g, s, parity);
    const size_t plane = g.Vh;
#pragma unroll
    for (int r = 0; r < R; r++)
#pragma unroll
        for (int c = 0; c < 3; c++) acc[r][c] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    // first word of the forward link of pair k; the backward one is nine planes on
    auto words = [&](int k) {
        const LinkField &f = k >= 4 ? naik : fat;
        return f.words + ((size_t)parity * f.W + (size_t)(k & 3) * 18) * plane + s;
    };
    auto hop = [&](int k, int sign) { return neighbour_rt(g, sc, s, k & 3, k >= 4 ? 3 * sign : sign); };
    if constexpr (PREFETCH) {
        DsOperands<R, COHERENT> fwd, bwd;
        fwd.load(words(0), plane, hop(0, 1), in, n, rr, act);
#pragma unroll 1
        for (int k = 0; k < 8; k++) {
            bwd.load(words(k) + 9 * plane, plane, hop(k, -1), in, n, rr, act);
            fwd.apply(acc);
            if (k + 1 < 8) fwd.load(words(k + 1), plane, hop(k + 1, 1), in, n, rr, act);
            bwd.apply(acc);
        }
    } else {
#pragma unroll 1
        for (int k = k0; k < k1; k++) {
            DsOperands<R, COHERENT> op;
            op.load(words(k), plane, hop(k, 1), in, n, rr, act);
            op.apply(acc);
            op.load(words(k) + 9 * plane, plane, hop(k, -1), in, n, rr, act);
            op.apply(acc);
        }
    }
}

}  // namespace hisq
