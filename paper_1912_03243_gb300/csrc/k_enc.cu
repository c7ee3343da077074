// Two-byte adaptive amplitude code (Sec. 1 "JUQCS-A"; Sec. 3 on the cost of
// the encoding-decoding operation).
//
// Format (the paper cites but does not give its format; this is the reading
// the library implements): blocks of 256 consecutive amplitudes share one
// FP32 scale s = max over the block of max(|re|, |im|); each component is an
// int8 code q = rint(x * fl(127/s)) clamped to [-127, 127]; decoding gives
// x = sign(q) * fl(s * T[|q|]) with T[k] = fl(k / 127), so +-127 decodes to
// +-s exactly and the uniform superposition is represented exactly.
//
// A gate is one pass: every touched block is decoded into registers, the 2x2
// update runs in FP32 in a fixed fused-multiply-add order, the new block
// scale is a warp max and the block is re-encoded in place.  All arithmetic
// uses explicitly rounded intrinsics (no contraction), so codes are
// reproducible bit for bit by a CPU implementation of the same steps.
//
// Work mapping: one warp per 256-amplitude block, 8 amplitudes (16 code
// bytes, one 16-byte load, four words of two amplitudes) per lane.  Target
// bits 0-2 pair amplitudes inside a lane, bits 3-7 pair lanes, bits >= 8 pair
// two blocks that the same warp holds side by side.  A control bit >= 8
// selects whole blocks; blocks whose control bit is 0 are not touched
// (decode followed by encode with an unchanged scale returns the same codes).
//
// What bounds it: instruction issue.  A gate decodes, updates, measures and
// re-encodes 16 components per lane, so the instructions per component decide
// (about 150 per lane, block and gate; 420 for an in-block gate of a run
// before).  The FP32 work is packed: the real (imaginary) parts of a word's
// two amplitudes form one f32x2 operand, and mul / add / fma.rn.f32x2 round
// each half as the scalar instruction does, so the codes stay bit-exact at
// half the issue slots.  The decode table is addressed with one byte permute,
// the block maximum is 3-input absolute maxima and one warp reduction (REDUX
// on the bits: non-negative floats order as integers), and in-block pairs are
// formed by exchanging packed codes.  27 qubits, one gate per pass: H inside
// the blocks 138 us (172 before), H across them 128 (144), SX across 134 (159),
// T across 76 (91); 27 qubits, 160 gates in runs: 11.0 ms
// (17.5 with runs of in-block gates only).
#include "sv_internal.h"

namespace sv {
namespace {

constexpr int kWarpsPerCta = 8;
constexpr int kGateWarps = 16;  // warps that share a decode table

struct EncGateArgs {
    uint64_t nwork;     // warps of work (blocks or block pairs)
    int t, c;           // target, control (-1 none)
    int ins[2];         // ascending block-index positions where zero bits are inserted
    int nins;
    uint64_t set_mask;  // block-index bits forced to 1 (control >= 8)
    uint64_t tbit;      // block-index bit of the target (t >= 8)
    float u[8];
};

}  // namespace
}  // namespace sv

#include "enc_run.h"

namespace sv {
namespace {

__device__ __forceinline__ uint64_t insert_zero(uint64_t x, int p) {
    const uint64_t lo = x & ((uint64_t(1) << p) - 1);
    return ((x ^ lo) << 1) | lo;
}

// Zero bits inserted at the ascending positions p0, p1 (the first nins of
// them); constant indices keep the launch arguments out of local memory.
__device__ __forceinline__ uint64_t insert_zeros(uint64_t x, int nins, int p0, int p1) {
    if (nins > 0) x = insert_zero(x, p0);
    if (nins > 1) x = insert_zero(x, p1);
    return x;
}

// rint(x * fl(127/s)).  No clamp is needed: s is the exact maximum of |x| over
// the block, so |x * fl(127/s)| <= 127 (1 + 2^-24)^2 < 127.5.
__device__ __forceinline__ int enc1(float x, float inv) { return __float2int_rn(__fmul_rn(x, inv)); }

__device__ __forceinline__ void gate_pair(const float *u, float &ar, float &ai, float &br, float &bi) {
    const float r0 = __fmaf_rn(u[0], ar, __fmaf_rn(-u[1], ai, __fmaf_rn(u[2], br, -__fmul_rn(u[3], bi))));
    const float i0 = __fmaf_rn(u[0], ai, __fmaf_rn(u[1], ar, __fmaf_rn(u[2], bi, __fmul_rn(u[3], br))));
    const float r1 = __fmaf_rn(u[4], ar, __fmaf_rn(-u[5], ai, __fmaf_rn(u[6], br, -__fmul_rn(u[7], bi))));
    const float i1 = __fmaf_rn(u[4], ai, __fmaf_rn(u[5], ar, __fmaf_rn(u[6], bi, __fmul_rn(u[7], br))));
    ar = r0;
    ai = i0;
    br = r1;
    bi = i1;
}

// ---- packed FP32 pairs (each half rounded as the scalar instruction)
using F2 = unsigned long long;
__device__ __forceinline__ F2 pk(float x, float y) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ void upk(F2 r, float &x, float &y) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(r));
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
    F2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
    F2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
    return d;
}
__device__ __forceinline__ F2 dup2(float x) { return pk(x, x); }

// max(|a|, |b|, |c|) (a NaN loses, as in fmaxf)
__device__ __forceinline__ float max3abs(float a, float b, float c) {
    float d;
    asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Warp maximum of non-negative floats: their bit patterns order as integers.
__device__ __forceinline__ float warp_max(float v) {
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}

// The two amplitudes of a word, as packed real and imaginary parts.
struct Amp2 {
    F2 re, im;
};

// A code byte 0x80 (-128, which no encoder writes) reads as -127: 0x80 -> 0x81.
__device__ __forceinline__ uint32_t clamp_codes(uint32_t w) {
    const uint32_t a = (w & 0x7f7f7f7fu) + 0x7f7f7f7fu;
    return w + ((~(a | (w ^ 0x80808080u)) & 0x80808080u) >> 7);
}
__device__ __forceinline__ int4 clamp_codes(int4 v) {
    return make_int4(int(clamp_codes(uint32_t(v.x))), int(clamp_codes(uint32_t(v.y))),
                     int(clamp_codes(uint32_t(v.z))), int(clamp_codes(uint32_t(v.w))));
}

// sign(q) fl(s fl(|q| / 127)) of a word's four codes.  q: the byte with its
// sign bit flipped is q + 128, and 0x4B000000 + (q + 128) is the float
// 2^23 + q + 128, from which 2^23 + 128 is taken exactly.  fl(q / 127):
// 1/127 = hi + lo with hi = fl(1/127), and fma(q, hi, fl(q lo)) equals the
// correctly rounded quotient for every |q| <= 127 (all 255 checked).
__device__ __forceinline__ void dec_word(uint32_t w, F2 s2, Amp2 &x) {
    const uint32_t o = w ^ 0x80808080u;
    const F2 off = dup2(-8388736.0f), hi = dup2(__uint_as_float(0x3c010204u)), lo = dup2(2.9332994e-11f);
    const F2 qr = add2(pk(__uint_as_float(__byte_perm(o, 0x4B000000u, 0x7440)),
                          __uint_as_float(__byte_perm(o, 0x4B000000u, 0x7442))), off);
    const F2 qi = add2(pk(__uint_as_float(__byte_perm(o, 0x4B000000u, 0x7441)),
                          __uint_as_float(__byte_perm(o, 0x4B000000u, 0x7443))), off);
    x.re = mul2(s2, fma2(qr, hi, mul2(qr, lo)));
    x.im = mul2(s2, fma2(qi, hi, mul2(qi, lo)));
}

// The same from a table of fl(q / 127) in shared memory: row u = the code
// byte, 64 floats per row of which lane l reads the l-th (no bank conflicts,
// and one byte permute builds the byte offset 256 u + 4 l).  A code byte 0x80
// reads as -127.
constexpr int kTabBytes = 256 * 256;
struct DecTable {
    const unsigned char *tab;
    uint32_t lane4;
    __device__ __forceinline__ float at(uint32_t w, uint32_t sel) const {
        return *reinterpret_cast<const float *>(tab + __byte_perm(w, lane4, sel));
    }
    __device__ __forceinline__ void operator()(uint32_t w, F2 s2, Amp2 &x) const {
        x.re = mul2(s2, pk(at(w, 0x5504), at(w, 0x5524)));
        x.im = mul2(s2, pk(at(w, 0x5514), at(w, 0x5534)));
    }
};
__device__ __forceinline__ void fill_table(unsigned char *smem) {
    float *tab = reinterpret_cast<float *>(smem);
    for (int i = threadIdx.x; i < 256 * 32; i += blockDim.x) {
        const float q = float(int((signed char)(i >> 5)));
        tab[(i >> 5) * 64 + (i & 31)] = __fdiv_rn(fmaxf(q, -127.0f), 127.0f);
    }
}

// The codes of a word's two amplitudes.  The code byte comes without a
// float-to-integer conversion: for |v| < 2^22 the sum v + 1.5 * 2^23 lies in
// [2^23, 2^24), where the float spacing is 1, so the (round-to-nearest-even)
// addition yields exactly rint(v) + 1.5 * 2^23, whose bit pattern is
// 0x4B400000 + rint(v).  Its low byte is rint(v) mod 256, the
// two's-complement code byte.  The product is rounded on its own first, as in
// enc1: scalar multiplications, because ptxas contracts a packed
// multiplication and addition in spite of their .rn.
__device__ __forceinline__ uint32_t enc_word(const Amp2 &x, float inv) {
    const F2 magic = dup2(12582912.0f);
    float r0, r1, i0, i1;
    upk(x.re, r0, r1);
    upk(x.im, i0, i1);
    upk(add2(pk(__fmul_rn(r0, inv), __fmul_rn(r1, inv)), magic), r0, r1);
    upk(add2(pk(__fmul_rn(i0, inv), __fmul_rn(i1, inv)), magic), i0, i1);
    const uint32_t lo = __byte_perm(__float_as_uint(r0), __float_as_uint(i0), 0x0040u);
    const uint32_t hi = __byte_perm(__float_as_uint(r1), __float_as_uint(i1), 0x0040u);
    return __byte_perm(lo, hi, 0x5410u);
}

__device__ __forceinline__ float amp_max(float m, const Amp2 &x) {
    float a, b, c, d;
    upk(x.re, a, b);
    upk(x.im, c, d);
    return max3abs(max3abs(m, a, b), c, d);
}

// A lane's 8 amplitudes of a block.
struct Lane8 {
    Amp2 w[4];
};

__device__ __forceinline__ void decode_lane(const DecTable &dec, const int4 raw, float s, Lane8 &x) {
    const F2 s2 = dup2(s);
    dec(uint32_t(raw.x), s2, x.w[0]);
    dec(uint32_t(raw.y), s2, x.w[1]);
    dec(uint32_t(raw.z), s2, x.w[2]);
    dec(uint32_t(raw.w), s2, x.w[3]);
}

__device__ __forceinline__ float lane_absmax(const Lane8 &x) {
    float m = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) m = amp_max(m, x.w[k]);
    return m;
}

// Codes of a lane's 8 amplitudes, inv = fl(127 / s).
__device__ __forceinline__ int4 enc_words(const Amp2 (&w)[4], float inv) {
    return make_int4(int(enc_word(w[0], inv)), int(enc_word(w[1], inv)), int(enc_word(w[2], inv)),
                     int(enc_word(w[3], inv)));
}

// Encode a lane's 8 amplitudes with the block scale s (warp-uniform).
__device__ __forceinline__ int4 encode_lane(const Lane8 &x, float s) {
    if (s == 0.0f) return make_int4(0, 0, 0, 0);
    return enc_words(x.w, __fdiv_rn(127.0f, s));
}

// Encode a lane's share of two blocks with their scales: even lanes divide
// for the first block, odd lanes for the second.
__device__ __forceinline__ void encode_two(const Amp2 (&x)[4], float s0, const Amp2 (&y)[4], float s1, int lane,
                                           int4 &v0, int4 &v1) {
    const float inv = __fdiv_rn(127.0f, lane & 1 ? s1 : s0);
    v0 = enc_words(x, __shfl_sync(0xffffffffu, inv, 0));
    v1 = enc_words(y, __shfl_sync(0xffffffffu, inv, 1));
    if (s0 == 0.0f) v0 = make_int4(0, 0, 0, 0);
    if (s1 == 0.0f) v1 = make_int4(0, 0, 0, 0);
}

// Shape of the 2x2 matrix, chosen on the host from exact zeros: the general
// fixed-order update (gate_pair), or the same update with the terms of zero
// coefficients left out.  A left-out term contributes fmaf(0, x, y) = y up to
// the sign of a zero, and a zero (of either sign) encodes to code 0 and does
// not change a block maximum, so the codes are those of the general form (EncShape).

// The matrix as packed operands; -u for the products the update subtracts
// (a product with a negated factor is the negated product).
template <int SHAPE>
struct Mat2 {
    F2 u[8], n[8];
    __device__ __forceinline__ explicit Mat2(const float *m) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            u[k] = dup2(m[k]);
            n[k] = dup2(-m[k]);
        }
    }
};

// (a, b) <- U (a, b) on two amplitude pairs.
template <int SHAPE>
__device__ __forceinline__ void gate2(const Mat2<SHAPE> &m, Amp2 &a, Amp2 &b) {
    const F2 ar = a.re, ai = a.im, br = b.re, bi = b.im;
    if constexpr (SHAPE == ENC_REAL) {  // every imaginary part 0
        a.re = fma2(m.u[0], ar, mul2(m.u[2], br));
        a.im = fma2(m.u[0], ai, mul2(m.u[2], bi));
        b.re = fma2(m.u[4], ar, mul2(m.u[6], br));
        b.im = fma2(m.u[4], ai, mul2(m.u[6], bi));
    } else if constexpr (SHAPE == ENC_DIAG || SHAPE == ENC_DIAG1) {  // u01 = u10 = 0
        if constexpr (SHAPE == ENC_DIAG) {  // (u00 = 1: a unchanged)
            a.re = fma2(m.u[0], ar, mul2(m.n[1], ai));
            a.im = fma2(m.u[0], ai, mul2(m.u[1], ar));
        }
        b.re = fma2(m.u[6], br, mul2(m.n[7], bi));
        b.im = fma2(m.u[6], bi, mul2(m.u[7], br));
    } else {
        a.re = fma2(m.u[0], ar, fma2(m.n[1], ai, fma2(m.u[2], br, mul2(m.n[3], bi))));
        a.im = fma2(m.u[0], ai, fma2(m.u[1], ar, fma2(m.u[2], bi, mul2(m.u[3], br))));
        b.re = fma2(m.u[4], ar, fma2(m.n[5], ai, fma2(m.u[6], br, mul2(m.n[7], bi))));
        b.im = fma2(m.u[4], ai, fma2(m.u[5], ar, fma2(m.u[6], bi, mul2(m.u[7], br))));
    }
}

// old where the half's bit of the two control bits in `bits` is 0 (bit masks,
// not selects: eight loop-invariant predicates would not fit a warp's seven).
__device__ __forceinline__ F2 keep_where(F2 now, F2 old, uint32_t bits) {
    const uint32_t m0 = uint32_t(int(bits << 31) >> 31), m1 = uint32_t(int(bits << 30) >> 31);
    const F2 m = F2(m0) | F2(m1) << 32;
    return (now & m) | (old & ~m);
}

// gate2 on the pairs whose control bit is set: bits (two, for the word's two
// amplitudes) of the lane's control mask.
template <int SHAPE>
__device__ __forceinline__ void gate2_ctl(const Mat2<SHAPE> &m, Amp2 &a, Amp2 &b, uint32_t bits) {
    const Amp2 a0 = a, b0 = b;
    gate2<SHAPE>(m, a, b);
    a.re = keep_where(a.re, a0.re, bits);
    a.im = keep_where(a.im, a0.im, bits);
    b.re = keep_where(b.re, b0.re, bits);
    b.im = keep_where(b.im, b0.im, bits);
}

// Update of a block on an in-block target t.  The words are first rearranged
// so that words 0, 1 hold the lower and words 2, 3 the upper amplitudes of
// the lane's four pairs (pair p = word p / 2, half p % 2): t = 2 as stored;
// t = 1: words 1 and 2 swap; t = 0: halves; t >= 3: the lower lane of a pair
// of lanes takes the pairs of words 0, 1 and the upper lane those of words
// 2, 3 (two shuffles of packed codes instead of sixteen of amplitudes, and
// no pair computed twice).  Each rearrangement undoes itself.
__device__ __forceinline__ void arrange(uint4 &v, int t, int lane) {
    if (t == 2) return;
    if (t == 1) {
        const uint32_t s = v.y;
        v.y = v.z;
        v.z = s;
    } else if (t == 0) {
        const uint4 o = v;
        v.x = __byte_perm(o.x, o.y, 0x5410u);
        v.y = __byte_perm(o.z, o.w, 0x5410u);
        v.z = __byte_perm(o.x, o.y, 0x7632u);
        v.w = __byte_perm(o.z, o.w, 0x7632u);
    } else {
        const bool up = lane >> (t - 3) & 1;
        const uint32_t r0 = __shfl_xor_sync(0xffffffffu, up ? v.x : v.z, 1 << (t - 3));
        const uint32_t r1 = __shfl_xor_sync(0xffffffffu, up ? v.y : v.w, 1 << (t - 3));
        v.x = up ? r0 : v.x;
        v.y = up ? r1 : v.y;
        v.z = up ? v.z : r0;
        v.w = up ? v.w : r1;
    }
}
__device__ __forceinline__ void arrange_back(uint4 &v, int t, int lane) {
    if (t == 0) {
        const uint4 o = v;
        v.x = __byte_perm(o.x, o.z, 0x5410u);
        v.y = __byte_perm(o.x, o.z, 0x7632u);
        v.z = __byte_perm(o.y, o.w, 0x5410u);
        v.w = __byte_perm(o.y, o.w, 0x7632u);
    } else {
        arrange(v, t, lane);
    }
}

// Control mask of the four rearranged pairs of a lane (bit p: pair p's
// amplitudes have bit c of the in-block index set; all ones without a
// control).
__device__ __forceinline__ uint32_t pair_ctl(int t, int c, int lane) {
    if (c < 0) return 15u;
    uint32_t m = 0;
#pragma unroll
    for (int p = 0; p < 4; ++p) {
        const int k = p >> 1, h = p & 1;
        const bool up = t >= 3 && (lane >> (t - 3) & 1);
        const int j = t == 2 ? 2 * k + h : t == 1 ? 4 * k + h : t == 0 ? 4 * k + 2 * h : (up ? 4 : 0) + 2 * k + h;
        if ((lane * 8 + j) >> c & 1) m |= 1u << p;
    }
    return m;
}
// Control mask of a lane's 8 amplitudes.
__device__ __forceinline__ uint32_t amp_ctl(int c, int lane) {
    if (c < 0) return 255u;
    if (c >= 3) return lane >> (c - 3) & 1 ? 255u : 0u;
    return c == 0 ? 0xAAu : c == 1 ? 0xCCu : 0xF0u;
}

// How an in-block control is met: none; every word computed and the words'
// halves selected (runs of gates, whose few warps want instructions without
// branches in between); words left out (one gate per pass, whole words only).
enum EncCtl { CTL_NONE = 0, CTL_SELECT, CTL_SKIP };

template <int SHAPE, int CTL>
__device__ __forceinline__ void gate2_sel(const Mat2<SHAPE> &m, Amp2 &a, Amp2 &b, uint32_t bits) {
    if constexpr (CTL == CTL_SELECT) {
        gate2_ctl<SHAPE>(m, a, b, bits);
    } else if constexpr (CTL == CTL_SKIP) {
        if (bits & 1u) gate2<SHAPE>(m, a, b);
    } else {
        gate2<SHAPE>(m, a, b);
    }
}

// The rearranged words of a block, decoded and updated; returns the lane's
// absolute maximum.  cm: pair_ctl.
template <int SHAPE, int CTL>
__device__ __forceinline__ float update_in(const DecTable &dec, const Mat2<SHAPE> &m, uint32_t cm, const uint4 &v,
                                           float s, Amp2 (&x)[4]) {
    const F2 s2 = dup2(s);
    dec(v.x, s2, x[0]);
    dec(v.y, s2, x[1]);
    dec(v.z, s2, x[2]);
    dec(v.w, s2, x[3]);
    gate2_sel<SHAPE, CTL>(m, x[0], x[2], cm);
    gate2_sel<SHAPE, CTL>(m, x[1], x[3], cm >> 2);
    float mx = 0.0f;
#pragma unroll
    for (int k = 0; k < 4; ++k) mx = amp_max(mx, x[k]);
    return mx;
}
__device__ __forceinline__ uint4 as_u4(const int4 &v) {
    return make_uint4(uint32_t(v.x), uint32_t(v.y), uint32_t(v.z), uint32_t(v.w));
}
__device__ __forceinline__ int4 as_i4(const uint4 &v) { return make_int4(int(v.x), int(v.y), int(v.z), int(v.w)); }
__device__ __forceinline__ int4 arranged(const int4 &v, int t, int lane) {
    uint4 u = as_u4(v);
    arrange(u, t, lane);
    return as_i4(u);
}
__device__ __forceinline__ int4 arranged_back(const int4 &v, int t, int lane) {
    uint4 u = as_u4(v);
    arrange_back(u, t, lane);
    return as_i4(u);
}

// One in-block gate on a block: codes v, scale s.
template <int SHAPE, int CTL>
__device__ __forceinline__ void block_gate_in(const DecTable &dec, const Mat2<SHAPE> &m, int t, uint32_t cm, int lane, uint4 &v, float &s) {
    arrange(v, t, lane);
    Lane8 x;
    s = warp_max(update_in<SHAPE, CTL>(dec, m, cm, v, s, x.w));
    v = as_u4(encode_lane(x, s));
    arrange_back(v, t, lane);
}

// The same on two blocks at once (independent instructions to issue).
template <int SHAPE, int CTL>
__device__ __forceinline__ void block_gate_in2(const DecTable &dec, const Mat2<SHAPE> &m, int t, uint32_t cm, int lane, uint4 &v0, float &s0,
                                               uint4 &v1, float &s1) {
    arrange(v0, t, lane);
    arrange(v1, t, lane);
    Amp2 x[4], y[4];
    const float m0 = update_in<SHAPE, CTL>(dec, m, cm, v0, s0, x), m1 = update_in<SHAPE, CTL>(dec, m, cm, v1, s1, y);
    s0 = warp_max(m0);
    s1 = warp_max(m1);
    int4 e0, e1;
    encode_two(x, s0, y, s1, lane, e0, e1);
    v0 = as_u4(e0);
    v1 = as_u4(e1);
    arrange_back(v0, t, lane);
    arrange_back(v1, t, lane);
}

// One gate on a pair of blocks that differ in the target bit.  ENC_DIAG1
// leaves the lower block as it is: its codes are not needed.
template <int SHAPE, int CTL>
__device__ __forceinline__ void block_gate_pair(const DecTable &dec, const Mat2<SHAPE> &m, uint32_t cm, int lane, int4 &v0, float &s0,
                                                int4 &v1, float &s1) {
    Lane8 x, y;
    if constexpr (SHAPE != ENC_DIAG1) decode_lane(dec, v0, s0, x);
    decode_lane(dec, v1, s1, y);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if constexpr (SHAPE == ENC_DIAG1) x.w[k] = y.w[k];  // not used by the update
        gate2_sel<SHAPE, CTL>(m, x.w[k], y.w[k], cm >> (2 * k));
    }
    if constexpr (SHAPE != ENC_DIAG1) {
        s0 = warp_max(lane_absmax(x));
        s1 = warp_max(lane_absmax(y));
        encode_two(x.w, s0, y.w, s1, lane, v0, v1);
    } else {
        s1 = warp_max(lane_absmax(y));
        v1 = encode_lane(y, s1);
    }
}

// Target inside the block (t < 8).
template <int SHAPE>
__global__ void __launch_bounds__(32 * kGateWarps, 3) k_enc_gate_in(uint4 *__restrict__ codes, float *__restrict__ scales,
                                                                   EncGateArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    fill_table(smem);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const DecTable dec{smem, uint32_t(lane) * 4u};
    const uint64_t wid = uint64_t(blockIdx.x) * kGateWarps + (threadIdx.x >> 5);
    const uint64_t nw = uint64_t(gridDim.x) * kGateWarps;
    const Mat2<SHAPE> m(a.u);
    const bool ctl = a.c >= 0 && a.c < kEncBlockLog2;
    const uint32_t cm = pair_ctl(a.t, ctl ? a.c : -1, lane);
    for (uint64_t w = wid; w < a.nwork; w += nw) {
        const uint64_t b = insert_zeros(w, a.nins, a.ins[0], a.ins[1]) | a.set_mask;
        uint4 v = codes[b * 32 + lane];
        float s = scales[b];
        if (ctl)
            block_gate_in<SHAPE, CTL_SELECT>(dec, m, a.t, cm, lane, v, s);
        else
            block_gate_in<SHAPE, CTL_NONE>(dec, m, a.t, cm, lane, v, s);
        codes[b * 32 + lane] = v;
        if (lane == 0) scales[b] = s;
    }
}

// CTAs per SM by matrix shape: the pair of blocks of a full update takes 64
// registers per thread, the single block of ENC_DIAG1 fits 3 CTAs.
constexpr int kAcrossCtas[4] = {2, 2, 2, 3};

// Target across blocks (t >= 8): the warp holds block b0 and b0 + 2^(t-8).
// A diagonal gate with u00 = 1 (T, P, ...) keeps the blocks with the target
// bit 0, hence their scale and codes (decoding and re-encoding with an
// unchanged scale is the identity), so ENC_DIAG1 reads and rewrites only the
// blocks with the target bit 1: half the traffic, the same codes.
template <int SHAPE>
__global__ void __launch_bounds__(32 * kGateWarps, kAcrossCtas[SHAPE]) k_enc_gate_across(int4 *__restrict__ codes,
                                                                       float *__restrict__ scales, EncGateArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    fill_table(smem);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const DecTable dec{smem, uint32_t(lane) * 4u};
    const uint64_t wid = uint64_t(blockIdx.x) * kGateWarps + (threadIdx.x >> 5);
    const uint64_t nw = uint64_t(gridDim.x) * kGateWarps;
    const Mat2<SHAPE> m(a.u);
    // An in-block control selects whole words of a lane: a control on qubit 0
    // once the words are rearranged as for a target there (their upper
    // amplitudes in words 2, 3).  Words without it are left out (27 qubits, SX
    // with a control inside the blocks: 137 to 144 us; 157 with every word
    // computed and its halves selected).
    const bool ctl = a.c >= 0 && a.c < kEncBlockLog2;
    const uint32_t cm = amp_ctl(ctl ? (a.c == 0 ? 2 : a.c) : -1, lane);
    for (uint64_t w = wid; w < a.nwork; w += nw) {
        const uint64_t b0 = insert_zeros(w, a.nins, a.ins[0], a.ins[1]) | a.set_mask;
        const uint64_t b1 = b0 | a.tbit;
        int4 v0 = make_int4(0, 0, 0, 0), v1 = codes[b1 * 32 + lane];
        float s0 = 0.0f, s1 = scales[b1];
        if constexpr (SHAPE != ENC_DIAG1) {
            v0 = codes[b0 * 32 + lane];
            s0 = scales[b0];
        }
        if (ctl) {
            if (a.c == 0) {
                v0 = arranged(v0, 0, lane);
                v1 = arranged(v1, 0, lane);
            }
            block_gate_pair<SHAPE, CTL_SKIP>(dec, m, cm, lane, v0, s0, v1, s1);
            if (a.c == 0) {
                v0 = arranged_back(v0, 0, lane);
                v1 = arranged_back(v1, 0, lane);
            }
        } else {
            block_gate_pair<SHAPE, CTL_NONE>(dec, m, cm, lane, v0, s0, v1, s1);
        }
        if constexpr (SHAPE != ENC_DIAG1) {
            codes[b0 * 32 + lane] = v0;
            if (lane == 0) scales[b0] = s0;
        }
        codes[b1 * 32 + lane] = v1;
        if (lane == 0) scales[b1] = s1;
    }
}

// n < 8: one block of 2^n amplitudes, done by one thread in plain order.
__global__ void k_enc_gate_small(signed char *codes, float *scales, int n, EncGateArgs a) {
    __shared__ float re[128], im[128];
    if (threadIdx.x != 0) return;
    const int dim = 1 << n;
    const float s = scales[0];
    for (int i = 0; i < dim; ++i) {
        const int qr = codes[2 * i], qi = codes[2 * i + 1];
        const int ar = qr < 0 ? -qr : qr, ai = qi < 0 ? -qi : qi;
        const float vr = __fmul_rn(s, __fdiv_rn(float(ar), 127.0f));
        const float vi = __fmul_rn(s, __fdiv_rn(float(ai), 127.0f));
        re[i] = qr < 0 ? -vr : vr;
        im[i] = qi < 0 ? -vi : vi;
    }
    for (int i = 0; i < dim; ++i) {
        if ((i >> a.t) & 1) continue;
        if (a.c >= 0 && !((i >> a.c) & 1)) continue;
        const int j = i | (1 << a.t);
        gate_pair(a.u, re[i], im[i], re[j], im[j]);
    }
    float m = 0.0f;
    for (int i = 0; i < dim; ++i) m = fmaxf(m, fmaxf(fabsf(re[i]), fabsf(im[i])));
    scales[0] = m;
    const float inv = m == 0.0f ? 0.0f : __fdiv_rn(127.0f, m);
    for (int i = 0; i < dim; ++i) {
        codes[2 * i] = m == 0.0f ? 0 : (signed char)enc1(re[i], inv);
        codes[2 * i + 1] = m == 0.0f ? 0 : (signed char)enc1(im[i], inv);
    }
}

// c64 -> codes: one warp per block (n >= 8).  Word w of a block (amplitudes
// 2w, 2w + 1) goes to lane w % 32, so every 16-byte load and 4-byte store of
// the warp is contiguous.
__global__ void __launch_bounds__(32 * kWarpsPerCta) k_encode(const float4 *__restrict__ psi,
                                                              uint32_t *__restrict__ codes, float *__restrict__ scales,
                                                              uint64_t nblocks) {
    const int lane = threadIdx.x & 31;
    const uint64_t wid = uint64_t(blockIdx.x) * kWarpsPerCta + (threadIdx.x >> 5);
    const uint64_t nw = uint64_t(gridDim.x) * kWarpsPerCta;
    for (uint64_t b = wid; b < nblocks; b += nw) {
        Lane8 x;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float4 v = psi[b * 128 + k * 32 + lane];
            x.w[k].re = pk(v.x, v.z);
            x.w[k].im = pk(v.y, v.w);
        }
        const float s = warp_max(lane_absmax(x));
        const int4 e = encode_lane(x, s);
        codes[b * 128 + lane] = uint32_t(e.x);
        codes[b * 128 + 32 + lane] = uint32_t(e.y);
        codes[b * 128 + 64 + lane] = uint32_t(e.z);
        codes[b * 128 + 96 + lane] = uint32_t(e.w);
        if (lane == 0) scales[b] = s;
    }
}

// The same word order: contiguous 4-byte loads, contiguous 16-byte stores.
__global__ void __launch_bounds__(32 * kWarpsPerCta) k_decode(const uint32_t *__restrict__ codes,
                                                              const float *__restrict__ scales,
                                                              float4 *__restrict__ psi, uint64_t nblocks) {
    const int lane = threadIdx.x & 31;
    const uint64_t wid = uint64_t(blockIdx.x) * kWarpsPerCta + (threadIdx.x >> 5);
    const uint64_t nw = uint64_t(gridDim.x) * kWarpsPerCta;
    for (uint64_t b = wid; b < nblocks; b += nw) {
        const F2 s2 = dup2(scales[b]);
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) w[k] = codes[b * 128 + k * 32 + lane];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            Amp2 x;
            dec_word(clamp_codes(w[k]), s2, x);
            float4 v;
            upk(x.re, v.x, v.z);
            upk(x.im, v.y, v.w);
            psi[b * 128 + k * 32 + lane] = v;
        }
    }
}

__global__ void k_encode_small(const float2 *psi, signed char *codes, float *scales, int n) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int dim = 1 << n;
    float m = 0.0f;
    for (int i = 0; i < dim; ++i) m = fmaxf(m, fmaxf(fabsf(psi[i].x), fabsf(psi[i].y)));
    scales[0] = m;
    const float inv = m == 0.0f ? 0.0f : __fdiv_rn(127.0f, m);
    for (int i = 0; i < dim; ++i) {
        codes[2 * i] = m == 0.0f ? 0 : (signed char)enc1(psi[i].x, inv);
        codes[2 * i + 1] = m == 0.0f ? 0 : (signed char)enc1(psi[i].y, inv);
    }
}

__global__ void k_decode_small(const signed char *codes, const float *scales, float2 *psi, int n) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    const int dim = 1 << n;
    const float s = scales[0];
    for (int i = 0; i < dim; ++i) {
        const int qr = codes[2 * i], qi = codes[2 * i + 1];
        const float vr = __fmul_rn(s, __fdiv_rn(float(qr < 0 ? -qr : qr), 127.0f));
        const float vi = __fmul_rn(s, __fdiv_rn(float(qi < 0 ? -qi : qi), 127.0f));
        psi[i] = make_float2(qr < 0 ? -vr : vr, qi < 0 ? -vi : vi);
    }
}


// ---------------------------------------------------------------- code-level fast paths
// Exact shortcuts of the decode-gate-encode pass.  Decoding and re-encoding a
// block with an unchanged scale returns its codes (|s T[q] fl(127/s) - q| is
// far below 1/2), and a diagonal gate with entries +-1, or a permutation of
// amplitudes inside a block or of whole blocks, leaves every block maximum
// unchanged; so these gates are sign flips or moves of the codes.

struct EncFlipArgs {
    uint64_t nwork;      // int4 words (8 amplitudes) to visit
    int ins[2], nins;    // ascending block-index positions where bits are inserted
    uint64_t set_mask;   // block-index bits forced to 1
    uint32_t lo_mask;    // in-block index bits of the condition (< 8)
    uint32_t lo_val;
};

// Negate the codes of every amplitude whose in-block bits match (lo_mask, lo_val)
// in the blocks selected by the inserted / forced block bits.
__global__ void __launch_bounds__(256) k_enc_flip(uint4 *__restrict__ codes, EncFlipArgs a) {
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t w = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; w < a.nwork; w += stride) {
        uint64_t b = w >> 5;  // selected block number, 32 words per block
        b = insert_zeros(b, a.nins, a.ins[0], a.ins[1]);
        b |= a.set_mask;
        const uint32_t lane = uint32_t(w & 31);
        uint4 v = codes[b * 32 + lane];
        uint32_t *x = reinterpret_cast<uint32_t *>(&v);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            uint32_t bm = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const uint32_t idx = lane * 8 + 2 * k + h;
                if ((idx & a.lo_mask) == a.lo_val) bm |= 0xFFFFu << (16 * h);
            }
            x[k] = (x[k] & ~bm) | (__vneg4(x[k]) & bm);
        }
        codes[b * 32 + lane] = v;
    }
}

// X on in-block target t (< 8), optional control c: swap amplitude pairs
// inside each selected block; one warp per block.
__global__ void __launch_bounds__(256) k_enc_xin(uint4 *__restrict__ codes, EncGateArgs a) {
    const int lane = threadIdx.x & 31;
    const uint64_t wid = uint64_t(blockIdx.x) * 8 + (threadIdx.x >> 5);
    const uint64_t nw = uint64_t(gridDim.x) * 8;
    const uint32_t cm = amp_ctl(a.c < kEncBlockLog2 ? a.c : -1, lane);
    for (uint64_t w = wid; w < a.nwork; w += nw) {
        uint64_t b = w;
        b = insert_zeros(b, a.nins, a.ins[0], a.ins[1]);
        b |= a.set_mask;
        const uint4 v = codes[b * 32 + lane];
        uint4 p;
        if (a.t >= 3) {
            const int lb = 1 << (a.t - 3);
            p.x = __shfl_xor_sync(0xffffffffu, v.x, lb);
            p.y = __shfl_xor_sync(0xffffffffu, v.y, lb);
            p.z = __shfl_xor_sync(0xffffffffu, v.z, lb);
            p.w = __shfl_xor_sync(0xffffffffu, v.w, lb);
        } else if (a.t == 0) {
            p = make_uint4(__byte_perm(v.x, 0, 0x1032), __byte_perm(v.y, 0, 0x1032), __byte_perm(v.z, 0, 0x1032),
                           __byte_perm(v.w, 0, 0x1032));
        } else if (a.t == 1) {
            p = make_uint4(v.y, v.x, v.w, v.z);
        } else {
            p = make_uint4(v.z, v.w, v.x, v.y);
        }
        const uint32_t *xv = reinterpret_cast<const uint32_t *>(&v), *xp = reinterpret_cast<const uint32_t *>(&p);
        uint32_t out[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            uint32_t bm = 0;
#pragma unroll
            for (int h = 0; h < 2; ++h)
                if (cm >> (2 * k + h) & 1u) bm |= 0xFFFFu << (16 * h);
            out[k] = (xv[k] & ~bm) | (xp[k] & bm);
        }
        codes[b * 32 + lane] = make_uint4(out[0], out[1], out[2], out[3]);
    }
}

// X on a block-level target (>= 8) with no control or a block-level control:
// swap whole blocks (codes and scales); one warp per block pair.
__global__ void __launch_bounds__(256) k_enc_xblocks(uint4 *__restrict__ codes, float *__restrict__ scales,
                                                     EncGateArgs a) {
    const int lane = threadIdx.x & 31;
    const uint64_t wid = uint64_t(blockIdx.x) * 8 + (threadIdx.x >> 5);
    const uint64_t nw = uint64_t(gridDim.x) * 8;
    for (uint64_t w = wid; w < a.nwork; w += nw) {
        uint64_t b0 = w;
        b0 = insert_zeros(b0, a.nins, a.ins[0], a.ins[1]);
        b0 |= a.set_mask;
        const uint64_t b1 = b0 | a.tbit;
        const uint4 v0 = codes[b0 * 32 + lane], v1 = codes[b1 * 32 + lane];
        codes[b0 * 32 + lane] = v1;
        codes[b1 * 32 + lane] = v0;
        if (lane == 0) {
            const float s0 = scales[b0];
            scales[b0] = scales[b1];
            scales[b1] = s0;
        }
    }
}

// ---------------------------------------------------------------- runs of gates
// A run of consecutive gates goes through one pass: each warp holds a tile of
// 2^B blocks (the blocks that differ in B chosen block-index bits) and applies
// every gate of the run whose target is an in-block qubit or one of those
// bits, and every sign flip, in circuit order.  A gate is the same decode ->
// FP32 update -> block maximum -> encode as in its own pass (the same
// functions), so every block's codes and scale after the run are those of the
// gates applied one pass at a time: bit-exact.  A gate whose block-level
// control is 0 leaves the block as it is (decoding and re-encoding with an
// unchanged scale is the identity).
//
// The tile's codes sit in shared memory, 16 bytes per lane and block, and are
// only ever touched by their own lane (gates across blocks keep the lane,
// in-block ones exchange codes by shuffles), so no gate needs a barrier; lane
// k holds the scale of block k.  Bound: instruction issue (67% active, ALU
// pipe 50%, FMA pipe 41%, under a profiler) on about 170 instructions per block
// and gate; the HBM traffic, 1 KB per block and run, is 6% of a run of 12 gates,
// but with 16 warps on an SM little of it overlaps in a run of two (plan.cu
// weighs it).  B = 4: 8 KB per warp and the 64 KB table leave 16 warps on an SM
// at 128 registers.  (Decoding by
// arithmetic instead of the table: 11.7 against 11.0 ms on 27 qubits and 160
// gates; 24 warps at 80 registers: spills, 11.9 against 11.7.)
//
// A run inside the blocks takes one block per warp, its codes in registers
// (57 of them), so that 32 warps share an SM: 64 gates at 25 qubits 1393 us,
// 2057 in tiles of 16 blocks, 1454 with one pass each; 12 to 18 qubits 33 us
// for any of them.

constexpr int kRunWarps = 16;
constexpr int kRunCtas0 = 2;  // CTAs per SM of runs inside single blocks

struct EncRunArgs {
    uint64_t ntiles;
    int nops, nbits;
    int pos[kEncRunMaxBits];  // ascending block-index positions of the tile bits
};

// Negate the codes of the amplitudes in the 8-bit mask m (bytewise, 0 - q).
__device__ __forceinline__ uint4 flip_codes(uint4 v, uint32_t m) {
    uint32_t *x = reinterpret_cast<uint32_t *>(&v);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t bm = (m >> (2 * k) & 1u ? 0x0000FFFFu : 0u) | (m >> (2 * k + 1) & 1u ? 0xFFFF0000u : 0u);
        const uint32_t a = x[k] ^ bm, one = bm & 0x01010101u;  // ~q + 1 in the masked bytes, no carry between bytes
        x[k] = ((a & 0x7f7f7f7fu) + one) ^ (a & 0x80808080u);
    }
    return v;
}

// The gate `op` on every block (or pair of blocks) of the tile that meets its
// block-level condition.  base: block index of the tile; tile block k is
// base | spread[k].  In-block gates take two blocks at a time.
template <int SHAPE, int CTL, int NB>
__device__ __forceinline__ void run_gate(const DecTable &dec, const EncRunOp &op, uint4 *tile, float &sc, uint32_t base,
                                         const uint32_t *spread, int nblk, int lane) {
    const Mat2<SHAPE> m(op.u);
    const uint32_t hm = uint32_t(op.hi_mask), hv = uint32_t(op.hi_val);
    const int t = op.t;
    uint4 *mine = NB == 0 ? tile : tile + lane;
    if constexpr (NB == 0) {
        if ((base & hm) != hv) return;
        uint4 v = mine[0];
        block_gate_in<SHAPE, CTL>(dec, m, t, pair_ctl(t, op.c, lane), lane, v, sc);  // (every lane holds the scale)
        mine[0] = v;
    } else if (op.kind == ENC_OP_IN) {
        const uint32_t cm = pair_ctl(t, op.c, lane);
        for (int k0 = 0; k0 < nblk; k0 += 2) {
            const int k1 = k0 + 1;
            const bool on0 = ((base | spread[k0]) & hm) == hv, on1 = ((base | spread[k1]) & hm) == hv;
            if (!on0 && !on1) continue;
            uint4 v0 = mine[k0 * 32], v1 = mine[k1 * 32];
            float s0 = __shfl_sync(0xffffffffu, sc, k0), s1 = __shfl_sync(0xffffffffu, sc, k1);
            block_gate_in2<SHAPE, CTL>(dec, m, t, cm, lane, v0, s0, v1, s1);
            if (on0) {
                mine[k0 * 32] = v0;
                sc = lane == k0 ? s0 : sc;
            }
            if (on1) {
                mine[k1 * 32] = v1;
                sc = lane == k1 ? s1 : sc;
            }
        }
    } else {
        const uint32_t cm = amp_ctl(op.c, lane);
        const int hi = 1 << t;
        for (int k0 = 0; k0 < nblk; k0 = ((k0 | hi) + 1) & ~hi) {
            const int k1 = k0 | hi;
            if (((base | spread[k0]) & hm) != hv) continue;
            int4 v0 = make_int4(0, 0, 0, 0), v1 = *reinterpret_cast<const int4 *>(mine + k1 * 32);
            float s0 = 0.0f, s1 = __shfl_sync(0xffffffffu, sc, k1);
            if (SHAPE != ENC_DIAG1) {
                v0 = *reinterpret_cast<const int4 *>(mine + k0 * 32);
                s0 = __shfl_sync(0xffffffffu, sc, k0);
            }
            block_gate_pair<SHAPE, CTL>(dec, m, cm, lane, v0, s0, v1, s1);
            if (SHAPE != ENC_DIAG1) {
                mine[k0 * 32] = as_u4(v0);
                sc = lane == k0 ? s0 : sc;
            }
            mine[k1 * 32] = as_u4(v1);
            sc = lane == k1 ? s1 : sc;
        }
    }
}

template <int NB, bool FULL = false>  // tile bits, or -1: a.nbits; CTAs of kRunWarps warps
__global__ void __launch_bounds__(32 * kRunWarps, NB == 0 ? kRunCtas0 : 1) k_enc_run_in(uint4 *__restrict__ codes,
                                                                     float *__restrict__ scales,
                                                                     const EncRunOp *__restrict__ gops,
                                                                     const EncRunArgs a) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ EncRunOp ops[kEncRunMaxOps];
    __shared__ uint32_t spread[1 << kEncRunMaxBits];
    const int nblk = NB >= 0 ? 1 << NB : 1 << a.nbits;
    fill_table(smem);
    for (int i = threadIdx.x; i < a.nops; i += blockDim.x) ops[i] = gops[i];
    if (threadIdx.x < nblk) {
        uint32_t s = 0;
#pragma unroll
        for (int j = 0; j < kEncRunMaxBits; ++j)
            if (j < a.nbits && (threadIdx.x >> j & 1u)) s |= 1u << a.pos[j];
        spread[threadIdx.x] = s;
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const DecTable dec{smem, uint32_t(lane) * 4u};
    uint4 held;  // a single block's codes
    uint4 *tile = &held;
    if constexpr (NB != 0) tile = reinterpret_cast<uint4 *>(smem + kTabBytes) + (threadIdx.x >> 5) * (nblk * 32);
    const int ml = NB == 0 ? 0 : lane;  // this lane's place in a block of the tile
    const unsigned warps = FULL ? unsigned(kRunWarps) : blockDim.x >> 5;
    const uint64_t wid = uint64_t(blockIdx.x) * warps + (threadIdx.x >> 5);
    const uint64_t nw = uint64_t(gridDim.x) * warps;
    for (uint64_t w = wid; w < a.ntiles; w += nw) {
        uint64_t b64 = w;
#pragma unroll
        for (int j = 0; j < kEncRunMaxBits; ++j)
            if (NB == kEncRunMaxBits || j < a.nbits) b64 = insert_zero(b64, a.pos[j]);
        const uint32_t base = uint32_t(b64);  // at most 2^32 blocks (n <= 40)
        const uint32_t own = base | spread[lane & (nblk - 1)];
        float sc = scales[own];
#pragma unroll
        for (int k = 0; k < nblk; ++k) {
            tile[k * 32 + ml] = codes[uint64_t(base | spread[k]) * 32 + lane];
        }
        for (int i = 0; i < a.nops; ++i) {
            const EncRunOp &op = ops[i];
            if (op.kind == ENC_OP_FLIP) {
                // the consecutive flips from here on: one mask per block, applied once
                int e = i + 1;
                while (e < a.nops && ops[e].kind == ENC_OP_FLIP) ++e;
                for (int k = 0; k < nblk; ++k) {
                    const uint32_t b = base | spread[k];
                    uint32_t m = 0;
                    for (int f = i; f < e; ++f) {
                        const EncRunOp &g = ops[f];
                        const bool on = (b & uint32_t(g.hi_mask)) == uint32_t(g.hi_val) &&
                                        (uint32_t(lane * 8) & g.lo_mask & 0xF8u) == (g.lo_val & 0xF8u);
                        m ^= on ? g.amps : 0u;
                    }
                    if (__any_sync(0xffffffffu, m != 0)) tile[k * 32 + ml] = flip_codes(tile[k * 32 + ml], m);
                }
                i = e - 1;
                continue;
            }
            if (NB != 0 && op.kind == ENC_OP_SWAP) {  // X on a tile bit: the blocks change places
                const uint32_t hm = uint32_t(op.hi_mask), hv = uint32_t(op.hi_val);
                for (int k = 0; k < nblk; ++k) {
                    const int k1 = k | (1 << op.t);
                    if (k == k1 || ((base | spread[k]) & hm) != hv) continue;
                    const uint4 v = tile[k * 32 + ml];
                    tile[k * 32 + ml] = tile[k1 * 32 + ml];
                    tile[k1 * 32 + ml] = v;
                    const float s0 = __shfl_sync(0xffffffffu, sc, k), s1 = __shfl_sync(0xffffffffu, sc, k1);
                    sc = lane == k ? s1 : lane == k1 ? s0 : sc;
                }
                continue;
            }
            switch (op.shape) {
                case ENC_REAL:
                    if (op.c >= 0)
                        run_gate<ENC_REAL, CTL_SELECT, NB>(dec, op, tile, sc, base, spread, nblk, lane);
                    else
                        run_gate<ENC_REAL, CTL_NONE, NB>(dec, op, tile, sc, base, spread, nblk, lane);
                    break;
                case ENC_DIAG:
                    if (op.c >= 0)
                        run_gate<ENC_DIAG, CTL_SELECT, NB>(dec, op, tile, sc, base, spread, nblk, lane);
                    else
                        run_gate<ENC_DIAG, CTL_NONE, NB>(dec, op, tile, sc, base, spread, nblk, lane);
                    break;
                case ENC_DIAG1:
                    if (op.c >= 0)
                        run_gate<ENC_DIAG1, CTL_SELECT, NB>(dec, op, tile, sc, base, spread, nblk, lane);
                    else
                        run_gate<ENC_DIAG1, CTL_NONE, NB>(dec, op, tile, sc, base, spread, nblk, lane);
                    break;
                default:
                    if (op.c >= 0)
                        run_gate<ENC_GENERAL, CTL_SELECT, NB>(dec, op, tile, sc, base, spread, nblk, lane);
                    else
                        run_gate<ENC_GENERAL, CTL_NONE, NB>(dec, op, tile, sc, base, spread, nblk, lane);
                    break;
            }
        }
#pragma unroll
        for (int k = 0; k < nblk; ++k) codes[uint64_t(base | spread[k]) * 32 + lane] = tile[k * 32 + ml];
        if (lane < nblk) scales[own] = sc;
    }
}

// Dynamic shared memory above 48 KB: the decode table, and the tiles of a run.
cudaError_t enc_attrs(int device) {
    static std::atomic<uint64_t> configured{0};
    if (!attrs_needed(configured, device)) return cudaSuccess;
    auto set = [](auto *fn, int bytes) {
        return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    const int run = kTabBytes + kRunWarps * (512 << kEncRunMaxBits);  // 192 KB
    for (const cudaError_t e :
         {set(k_enc_gate_in<ENC_GENERAL>, kTabBytes), set(k_enc_gate_in<ENC_REAL>, kTabBytes),
          set(k_enc_gate_in<ENC_DIAG>, kTabBytes), set(k_enc_gate_in<ENC_DIAG1>, kTabBytes),
          set(k_enc_gate_across<ENC_GENERAL>, kTabBytes), set(k_enc_gate_across<ENC_REAL>, kTabBytes),
          set(k_enc_gate_across<ENC_DIAG>, kTabBytes), set(k_enc_gate_across<ENC_DIAG1>, kTabBytes),
          set(k_enc_run_in<kEncRunMaxBits, true>, run), set(k_enc_run_in<kEncRunMaxBits>, run),
          set(k_enc_run_in<-1, true>, run), set(k_enc_run_in<-1>, run),
          set(k_enc_run_in<0>, run)})
        if (e != cudaSuccess) return e;
    attrs_set(configured, device);
    return cudaSuccess;
}

int enc_grid(uint64_t nwork) {
    uint64_t b = (nwork + kWarpsPerCta - 1) / kWarpsPerCta;
    const uint64_t cap = 152ull * 16;
    return int(b < 1 ? 1 : (b < cap ? b : cap));
}

}  // namespace

cudaError_t launch_enc_gate1(sv_state *h, const Gate1 &g) {
    EncGateArgs a{};
    for (int k = 0; k < 4; ++k) {
        a.u[2 * k] = float(g.u[k].re);  // round to nearest
        a.u[2 * k + 1] = float(g.u[k].im);
    }
    a.t = g.target;
    a.c = g.control;
    const int n = h->n;
    if (n < kEncBlockLog2) {
        k_enc_gate_small<<<1, 32, 0, h->stream>>>(static_cast<signed char *>(h->data), h->scales, n, a);
        return cudaGetLastError();
    }
    const int nb_log = n - kEncBlockLog2;
    const Cplx *u = g.u;
    auto is = [](const Cplx &z, double re) { return z.re == re && z.im == 0.0; };
    // diagonal with entries +-1 (Z, CZ, ...): sign flips of codes
    if (is(u[1], 0) && is(u[2], 0) && (is(u[0], 1) || is(u[0], -1)) && (is(u[3], 1) || is(u[3], -1))) {
        if (is(u[0], 1) && is(u[3], 1)) return cudaSuccess;  // identity
        uint64_t m = g.control >= 0 ? (uint64_t(1) << g.control) : 0, v = m;
        if (!(is(u[0], -1) && is(u[3], -1))) {  // only one half flips: condition on the target bit
            m |= uint64_t(1) << g.target;
            if (is(u[3], -1)) v |= uint64_t(1) << g.target;
        }
        EncFlipArgs fa{};
        fa.lo_mask = uint32_t(m & 0xFFu);
        fa.lo_val = uint32_t(v & 0xFFu);
        int k = 0;
        for (int bit = kEncBlockLog2; bit < n; ++bit)
            if (m >> bit & 1) {
                fa.ins[k++] = bit - kEncBlockLog2;
                if (v >> bit & 1) fa.set_mask |= uint64_t(1) << (bit - kEncBlockLog2);
            }
        fa.nins = k;
        fa.nwork = (uint64_t(1) << (nb_log - k)) * 32;
        const uint64_t blocks = (fa.nwork + 255) / 256;
        k_enc_flip<<<unsigned(blocks < 152 * 32 ? blocks : 152 * 32), 256, 0, h->stream>>>(static_cast<uint4 *>(h->data),
                                                                                          fa);
        return cudaGetLastError();
    }
    const bool xgate = is(u[0], 0) && is(u[3], 0) && is(u[1], 1) && is(u[2], 1);
    int ins[2], ni = 0;
    if (a.c >= kEncBlockLog2) {
        ins[ni++] = a.c - kEncBlockLog2;
        a.set_mask = uint64_t(1) << (a.c - kEncBlockLog2);
    }
    if (a.t >= kEncBlockLog2) {
        ins[ni++] = a.t - kEncBlockLog2;
        a.tbit = uint64_t(1) << (a.t - kEncBlockLog2);
    }
    if (ni == 2 && ins[0] > ins[1]) {
        const int t = ins[0];
        ins[0] = ins[1];
        ins[1] = t;
    }
    for (int k = 0; k < ni; ++k) a.ins[k] = ins[k];
    a.nins = ni;
    a.nwork = uint64_t(1) << (nb_log - ni);
    int4 *codes = static_cast<int4 *>(h->data);
    uint4 *ucodes = static_cast<uint4 *>(h->data);
    if (xgate && a.t < kEncBlockLog2) {  // permutation inside blocks
        k_enc_xin<<<enc_grid(a.nwork), 256, 0, h->stream>>>(reinterpret_cast<uint4 *>(codes), a);
        return cudaGetLastError();
    }
    if (xgate && (a.c < 0 || a.c >= kEncBlockLog2)) {  // whole-block swaps
        k_enc_xblocks<<<enc_grid(a.nwork), 256, 0, h->stream>>>(reinterpret_cast<uint4 *>(codes), h->scales, a);
        return cudaGetLastError();
    }
    // matrix shape from exact zeros of the FP32 entries the kernel uses
    const bool real = a.u[1] == 0.0f && a.u[3] == 0.0f && a.u[5] == 0.0f && a.u[7] == 0.0f;
    const bool diag = a.u[2] == 0.0f && a.u[3] == 0.0f && a.u[4] == 0.0f && a.u[5] == 0.0f;
    const bool one = diag && a.u[0] == 1.0f && a.u[1] == 0.0f;
    const int shape = one ? ENC_DIAG1 : diag ? ENC_DIAG : real ? ENC_REAL : ENC_GENERAL;
    const cudaError_t ea = enc_attrs(h->device);
    if (ea != cudaSuccess) return ea;
    const uint64_t want = (a.nwork + kGateWarps - 1) / kGateWarps;
    // persistent CTAs (each fills a decode table): 3 per SM where the registers
    // of one block's update allow it, 2 for pairs of blocks (28 qubits: H inside
    // the blocks 255 us against 276 us with 2, H across them 240 against 290 with 3)
    const unsigned cap = 152u * unsigned(a.t < kEncBlockLog2 ? 3 : kAcrossCtas[shape]);
    const unsigned grid = unsigned(want < cap ? want : cap), block = 32 * kGateWarps;
    if (a.t < kEncBlockLog2) {
        switch (shape) {
            case ENC_REAL: k_enc_gate_in<ENC_REAL><<<grid, block, kTabBytes, h->stream>>>(ucodes, h->scales, a); break;
            case ENC_DIAG: k_enc_gate_in<ENC_DIAG><<<grid, block, kTabBytes, h->stream>>>(ucodes, h->scales, a); break;
            case ENC_DIAG1: k_enc_gate_in<ENC_DIAG1><<<grid, block, kTabBytes, h->stream>>>(ucodes, h->scales, a); break;
            default: k_enc_gate_in<ENC_GENERAL><<<grid, block, kTabBytes, h->stream>>>(ucodes, h->scales, a); break;
        }
    } else {
        switch (shape) {
            case ENC_REAL: k_enc_gate_across<ENC_REAL><<<grid, block, kTabBytes, h->stream>>>(codes, h->scales, a); break;
            case ENC_DIAG: k_enc_gate_across<ENC_DIAG><<<grid, block, kTabBytes, h->stream>>>(codes, h->scales, a); break;
            case ENC_DIAG1: k_enc_gate_across<ENC_DIAG1><<<grid, block, kTabBytes, h->stream>>>(codes, h->scales, a); break;
            default: k_enc_gate_across<ENC_GENERAL><<<grid, block, kTabBytes, h->stream>>>(codes, h->scales, a); break;
        }
    }
    return cudaGetLastError();
}

// The matrix shape of a gate from exact zeros of its FP32 entries.
static int enc_shape(const float *u) {
    const bool real = u[1] == 0.0f && u[3] == 0.0f && u[5] == 0.0f && u[7] == 0.0f;
    const bool diag = u[2] == 0.0f && u[3] == 0.0f && u[4] == 0.0f && u[5] == 0.0f;
    const bool one = diag && u[0] == 1.0f && u[1] == 0.0f;
    return one ? ENC_DIAG1 : diag ? ENC_DIAG : real ? ENC_REAL : ENC_GENERAL;
}

bool enc_run_op(int n, const Gate1 &g, EncRunOp *op) {
    if (n < kEncBlockLog2) return false;
    *op = EncRunOp{};
    const Cplx *u = g.u;
    auto is = [](const Cplx &z, double re) { return z.re == re && z.im == 0.0; };
    if (is(u[1], 0) && is(u[2], 0) && (is(u[0], 1) || is(u[0], -1)) && (is(u[3], 1) || is(u[3], -1))) {
        // +-1 diagonal: a sign flip on any qubits (identity: an empty flip)
        uint64_t m = g.control >= 0 ? (uint64_t(1) << g.control) : 0, v = m;
        if (!(is(u[0], -1) && is(u[3], -1))) {
            m |= uint64_t(1) << g.target;
            if (is(u[3], -1)) v |= uint64_t(1) << g.target;
        }
        op->kind = ENC_OP_FLIP;
        op->lo_mask = uint32_t(m & 0xFFu);
        op->lo_val = uint32_t(v & 0xFFu);
        op->hi_mask = m >> kEncBlockLog2;
        op->hi_val = v >> kEncBlockLog2;
        if (is(u[0], 1) && is(u[3], 1)) return true;  // identity: a flip of no amplitude (amps = 0)
        for (uint32_t j = 0; j < 8; ++j)
            if ((j & op->lo_mask & 7u) == (op->lo_val & 7u)) op->amps |= 1u << j;
        return true;
    }
    op->c = g.control >= 0 && g.control < kEncBlockLog2 ? g.control : -1;
    if (g.target < kEncBlockLog2) {
        op->kind = ENC_OP_IN;
        op->t = g.target;
    } else {
        const bool x = is(u[0], 0) && is(u[3], 0) && is(u[1], 1) && is(u[2], 1);
        op->kind = x && op->c < 0 ? ENC_OP_SWAP : ENC_OP_PAIR;
        op->t = g.target - kEncBlockLog2;  // a block-index bit: the caller maps it to a tile bit
    }
    if (g.control >= kEncBlockLog2) op->hi_mask = op->hi_val = uint64_t(1) << (g.control - kEncBlockLog2);
    for (int k = 0; k < 4; ++k) {
        op->u[2 * k] = float(g.u[k].re);
        op->u[2 * k + 1] = float(g.u[k].im);
    }
    op->shape = enc_shape(op->u);
    return true;
}

cudaError_t launch_enc_run(sv_state *h, const EncRunOp *d_ops, int nops, int nbits, const int *pos) {
    EncRunArgs a{};
    a.ntiles = uint64_t(1) << (h->n - kEncBlockLog2 - nbits);
    a.nops = nops;
    a.nbits = nbits;
    for (int j = 0; j < nbits; ++j) a.pos[j] = pos[j];
    uint4 *codes = static_cast<uint4 *>(h->data);
    const cudaError_t e = enc_attrs(h->device);
    if (e != cudaSuccess) return e;
    // few tiles spread over the SMs, on CTAs of at least 8 warps (22 qubits, random
    // circuit of depth 3: 485 us on 64 CTAs of 16 warps, 355 on 128 of 8; 4 warps
    // take 2 us longer to fill the decode table).  Tiles of one CTA take 16, which
    // fill it sooner (12 qubits, two SX 6.3 us, 8.2 with 8).  Full CTAs have the
    // number of warps as a constant (27 qubits, 160 gates 11.02 ms, 11.04 without).
    const uint64_t share = (a.ntiles + 151) / 152;
    const unsigned warps = unsigned(a.ntiles <= kRunWarps || share > kRunWarps ? kRunWarps : share < 8 ? 8 : share);
    const unsigned block = 32 * warps;
    const uint64_t want = (a.ntiles + warps - 1) / warps;
    const uint64_t cap = 152 * (nbits == 0 ? kRunCtas0 : 1);
    const unsigned grid = unsigned(want < cap ? want : cap);
    const int smem = kTabBytes + (nbits == 0 ? 0 : int(warps) * (512 << nbits));
    auto go = [&](auto *fn) { fn<<<grid, block, smem, h->stream>>>(codes, h->scales, d_ops, a); };
    const bool full = warps == kRunWarps;
    if (nbits == 0)
        go(k_enc_run_in<0>);
    else if (nbits == kEncRunMaxBits)
        full ? go(k_enc_run_in<kEncRunMaxBits, true>) : go(k_enc_run_in<kEncRunMaxBits>);
    else
        full ? go(k_enc_run_in<-1, true>) : go(k_enc_run_in<-1>);
    return cudaGetLastError();
}

cudaError_t launch_encode(const sv_state *src, sv_state *dst) {
    const int n = src->n;
    if (n < kEncBlockLog2) {
        k_encode_small<<<1, 32, 0, dst->stream>>>(static_cast<const float2 *>(src->data),
                                                  static_cast<signed char *>(dst->data), dst->scales, n);
    } else {
        const uint64_t nb = uint64_t(1) << (n - kEncBlockLog2);
        k_encode<<<enc_grid(nb), 32 * kWarpsPerCta, 0, dst->stream>>>(static_cast<const float4 *>(src->data),
                                                                      static_cast<uint32_t *>(dst->data), dst->scales,
                                                                      nb);
    }
    return cudaGetLastError();
}

cudaError_t launch_decode(const sv_state *src, sv_state *dst) {
    const int n = src->n;
    if (n < kEncBlockLog2) {
        k_decode_small<<<1, 32, 0, dst->stream>>>(static_cast<const signed char *>(src->data), src->scales,
                                                  static_cast<float2 *>(dst->data), n);
    } else {
        const uint64_t nb = uint64_t(1) << (n - kEncBlockLog2);
        k_decode<<<enc_grid(nb), 32 * kWarpsPerCta, 0, dst->stream>>>(static_cast<const uint32_t *>(src->data), src->scales,
                                                                      static_cast<float4 *>(dst->data), nb);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------- read-out
namespace {

__device__ __forceinline__ float dec_plain(int q, float s) {
    const float v = __fmul_rn(s, __fdiv_rn(float(q < 0 ? -q : q), 127.0f));
    return q < 0 ? -v : v;
}

__global__ void k_enc_gather(const char2 *__restrict__ codes, const float *__restrict__ scales, int n,
                             const uint64_t *__restrict__ idx, size_t m, double2 *__restrict__ out) {
    for (size_t j = size_t(blockIdx.x) * blockDim.x + threadIdx.x; j < m; j += size_t(gridDim.x) * blockDim.x) {
        const uint64_t i = idx[j];
        const float s = scales[n < kEncBlockLog2 ? 0 : (i >> kEncBlockLog2)];
        const char2 q = codes[i];
        out[j] = make_double2(dec_plain(q.x, s), dec_plain(q.y, s));
    }
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum of |decoded amplitude|^2: one warp per block, 4-amplitude FP32
// partial sums, FP64 beyond; one partial per CTA.
__global__ void __launch_bounds__(256) k_enc_norm(const int4 *__restrict__ codes, const float *__restrict__ scales,
                                                  uint64_t nblocks, double *__restrict__ partials) {
    __shared__ double sh[8];
    const int lane = threadIdx.x & 31;
    const uint64_t wid = uint64_t(blockIdx.x) * 8 + (threadIdx.x >> 5);
    const uint64_t nw = uint64_t(gridDim.x) * 8;
    double acc = 0.0;
    for (uint64_t b = wid; b < nblocks; b += nw) {
        Lane8 x;
        const int4 c = clamp_codes(codes[b * 32 + lane]);
        const F2 s2 = dup2(scales[b]);
        dec_word(uint32_t(c.x), s2, x.w[0]);
        dec_word(uint32_t(c.y), s2, x.w[1]);
        dec_word(uint32_t(c.z), s2, x.w[2]);
        dec_word(uint32_t(c.w), s2, x.w[3]);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float s = 0.0f;
#pragma unroll
            for (int k = 2 * h; k < 2 * h + 2; ++k) {
                float r0, r1, i0, i1;
                upk(x.w[k].re, r0, r1);
                upk(x.w[k].im, i0, i1);
                s = fmaf(r0, r0, fmaf(i0, i0, s));
                s = fmaf(r1, r1, fmaf(i1, i1, s));
            }
            acc += double(s);
        }
    }
    acc = warp_sum_d(acc);
    if (lane == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < 8; ++k) t += sh[k];
        partials[blockIdx.x] = t;
    }
}

__global__ void k_enc_norm_small(const signed char *codes, const float *scales, int n, double *partials, int np) {
    if (threadIdx.x != 0) return;
    double acc = 0.0;
    for (int i = 0; i < (1 << n); ++i) {
        const float a = dec_plain(codes[2 * i], scales[0]), b = dec_plain(codes[2 * i + 1], scales[0]);
        acc += double(a) * a + double(b) * b;
    }
    for (int k = 0; k < np; ++k) partials[k] = k == 0 ? acc : 0.0;
}

__global__ void k_sum_partials(const double *__restrict__ partials, int np, double *out) {
    __shared__ double sh[8];
    double acc = 0.0;
    for (int i = threadIdx.x; i < np; i += blockDim.x) acc += partials[i];
    acc = warp_sum_d(acc);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int k = 0; k < int(blockDim.x >> 5); ++k) t += sh[k];
        *out = t;
    }
}

}  // namespace

cudaError_t launch_enc_gather(sv_state *h, const uint64_t *d_idx, size_t m, double *d_out) {
    if (m == 0) return cudaSuccess;
    const int blocks = int((m + 255) / 256 < 1024 ? (m + 255) / 256 : 1024);
    k_enc_gather<<<blocks, 256, 0, h->stream>>>(static_cast<const char2 *>(h->data), h->scales, h->n, d_idx, m,
                                                reinterpret_cast<double2 *>(d_out));
    return cudaGetLastError();
}

cudaError_t launch_enc_norm(sv_state *h, double *d_out) {
    const int np = norm_partials_needed(h);
    if (h->n < kEncBlockLog2) {
        k_enc_norm_small<<<1, 32, 0, h->stream>>>(static_cast<const signed char *>(h->data), h->scales, h->n,
                                                  h->d_partials, np);
    } else {
        const uint64_t nb = uint64_t(1) << (h->n - kEncBlockLog2);
        k_enc_norm<<<np, 256, 0, h->stream>>>(static_cast<const int4 *>(h->data), h->scales, nb, h->d_partials);
    }
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_sum_partials<<<1, 256, 0, h->stream>>>(h->d_partials, np, d_out);
    return cudaGetLastError();
}

}  // namespace sv
