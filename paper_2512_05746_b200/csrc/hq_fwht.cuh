// Building blocks of the in-register fast Walsh-Hadamard transform + quantization shared by the stand-alone
// transform+quantize kernel and the fused linear kernel: two-wide fp32 arithmetic, butterfly stages, the shared-memory
// exchange between the two register phases, and rounding + packing of the codes.
#pragma once

#include "hq_common.cuh"

namespace hq {

constexpr float kMagic = 12582912.0f;            // 1.5 * 2^23: adding it rounds to an integer in the low mantissa bits
constexpr uint32_t kMagicBits = 0x4B400000u;

// ---- two-wide fp32 arithmetic (one instruction for a pair of values held in a 64-bit register) -----------------
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk2(float lo, float hi) { f32x2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi)); return r; }
__device__ __forceinline__ void upk2(f32x2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) { f32x2 r; asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) { f32x2 r; asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) { f32x2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) { f32x2 r; asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b)); return r; }

// Two pairs to 16 bytes of shared memory, as four 32-bit operands: stored as a vector of two 64-bit values, every value was moved to
// another register first (0.8 instructions per value; 32768 x 2048 bf16, two codes per byte, 43.3 -> 41.2 us).
// The kernels that transform inside the product, as vectors / so, in a graph: hq_small.cu fp32 256 x 256 -> 256 block 256 3.46 / 3.42, 70 x 512 ->
// 1024 block 512 5.31 / 5.15, 128 x 1024 -> 1024 block 128 6.21 / 6.04, 200 x 768 -> 640 block 256 4.69 / 4.67, bf16 70 x 512 -> 1024 block 512 5.11 /
// 5.02; hq_fused.cu 8192 x 512 -> 512 fp32 block 512 30.2 / 29.5, block 128 29.0 / 28.0, bf16 block 512 29.3 / 28.4.
__device__ __forceinline__ void st_shared_pairs(ulonglong2* to, f32x2 a, f32x2 b) {
    float x0, x1, x2, x3;
    upk2(a, x0, x1);
    upk2(b, x2, x3);
    *reinterpret_cast<float4*>(to) = make_float4(x0, x1, x2, x3);
}

// The largest of three values in one instruction.
__device__ __forceinline__ float max3(float a, float b, float c) { float r; asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c)); return r; }

// Butterflies over pair-index bits: element distance 2*h for h = LO .. HI (pairs stay pairs).
template <int P, int LO, int HI>
__device__ __forceinline__ void butterflies_pairs(f32x2 (&v)[P]) {
#pragma unroll
    for (int h = LO; h <= HI; h <<= 1) {
#pragma unroll
        for (int i = 0; i < P; ++i) {
            if (!(i & h)) {
                const f32x2 a = v[i], b = v[i | h];
                v[i] = add2(a, b);
                v[i | h] = sub2(a, b);
            }
        }
    }
}
// Sums with one operand in bf16 (converted exactly by the adder itself, at the rate of a plain addition): the low or the high half
// of a word.  A conversion by a shift or a mask takes a slot of the pipe that the packing needs, at half the rate.
__device__ __forceinline__ float add_bf16_lo(uint32_t w, float c) { float r; asm("{.reg .b16 l, h; mov.b32 {l, h}, %1; add.rn.f32.bf16 %0, l, %2;}" : "=f"(r) : "r"(w), "f"(c)); return r; }
__device__ __forceinline__ float add_bf16_hi(uint32_t w, float c) { float r; asm("{.reg .b16 l, h; mov.b32 {l, h}, %1; add.rn.f32.bf16 %0, h, %2;}" : "=f"(r) : "r"(w), "f"(c)); return r; }
__device__ __forceinline__ float sub_bf16_lo(uint32_t w, float c) { float r; asm("{.reg .b16 l, h; mov.b32 {l, h}, %1; sub.rn.f32.bf16 %0, l, %2;}" : "=f"(r) : "r"(w), "f"(c)); return r; }
__device__ __forceinline__ float sub_bf16_hi(uint32_t w, float c) { float r; asm("{.reg .b16 l, h; mov.b32 {l, h}, %1; sub.rn.f32.bf16 %0, h, %2;}" : "=f"(r) : "r"(w), "f"(c)); return r; }
// The stage between two neighbouring bf16 values.
__device__ __forceinline__ f32x2 butterfly_bf16(uint32_t w) {
    const float b = __uint_as_float(w & 0xFFFF0000u);
    return pk2(add_bf16_lo(w, b), sub_bf16_lo(w, b));
}

// The stage between the two values of each pair.
template <int P>
__device__ __forceinline__ void butterfly_within_pairs(f32x2 (&v)[P]) {
#pragma unroll
    for (int i = 0; i < P; ++i) {
        float a, b;
        upk2(v[i], a, b);
        v[i] = pk2(a + b, a - b);
    }
}

__host__ __device__ constexpr int ilog2_c(int v) { return v <= 1 ? 0 : 1 + ilog2_c(v >> 1); }

// Rounds E values held as pairs (ties to even, optional clamp) and packs them in register order into words: 8
// four-bit codes or 4 bytes per word.  Adding kMagic + bias leaves code + bias in the low mantissa bits.  One of two
// values is rounded F times larger (F = 256 for bytes, 16 for four-bit codes): scaling the multiplier and
// the magic number by a power of two scales the sum exactly, so the code is the same, and it lands F units up.  Taking
// the scaled magic number off again (exact) and adding the other value (exact: the sum stays below 2^22 units) leaves
// both biased codes side by side in the low bits of one float, on the floating-point pipe; byte permutes then gather
// the fields of a word, and one XOR turns the biased fields into two's complement.  Bytes: the two values come from
// neighbouring pairs, so that the additions are two-wide as well (hq_small.cu, pairs of one value each / so: bf16 200 x 768 -> 640 block 128 4.84 /
// 4.70, 256 x 256 -> 256 fp32 block 256 3.52 / 3.45; the exceptions are fp32 200 x 768 -> 640 block 256 4.49 / 4.68, 128 x 1024 -> 1024 block 128
// 5.86 / 6.07).
template <int E, bool INT8_OUT, bool CLAMP>
__device__ __forceinline__ void round_pack(const f32x2 (&v)[E / 2], float inv, int bits, uint32_t (&out)[INT8_OUT ? E / 4 : E / 8]) {
    constexpr float F = INT8_OUT ? 256.0f : 16.0f;
    const float bias = INT8_OUT ? 128.0f : 8.0f;
    const float mb = kMagic + bias;
    const float lo = mb + float(-(1 << (bits - 1))), hi = mb + float((1 << (bits - 1)) - 1);
    if (INT8_OUT) {
        const f32x2 inv0 = pk2(inv, inv), inv1 = pk2(F * inv, F * inv), mb0 = pk2(mb, mb), mb1 = pk2(F * mb, F * mb);
        const f32x2 off = pk2(-F * kMagic, -F * kMagic);
#pragma unroll
        for (int w = 0; w < E / 4; ++w) {
            f32x2 a = fma2(v[2 * w], inv0, mb0), b = fma2(v[2 * w + 1], inv1, mb1);
            if (CLAMP) {
                float a0, a1, b0, b1;
                upk2(a, a0, a1);
                upk2(b, b0, b1);
                a = pk2(fminf(fmaxf(a0, lo), hi), fminf(fmaxf(a1, lo), hi));
                b = pk2(fminf(fmaxf(b0, F * lo), F * hi), fminf(fmaxf(b1, F * lo), F * hi));
            }
            float u0, u1;                              // kMagicBits + (c0 + bias) + F (c2 + bias), and c1, c3
            upk2(add2(a, add2(b, off)), u0, u1);
            out[w] = __byte_perm(__float_as_uint(u0), __float_as_uint(u1), 0x5140) ^ 0x80808080u;
        }
    } else {
        const f32x2 inv2 = pk2(inv, F * inv), mb2 = pk2(mb, F * mb);
        uint32_t u[E / 2];                             // per pair: kMagicBits + (c0 + bias) + F (c1 + bias)
#pragma unroll
        for (int e = 0; e < E / 2; ++e) {
            float f0, f1;
            upk2(fma2(v[e], inv2, mb2), f0, f1);
            if (CLAMP) { f0 = fminf(fmaxf(f0, lo), hi); f1 = fminf(fmaxf(f1, F * lo), F * hi); }
            u[e] = __float_as_uint(f0 + (f1 - F * kMagic));
        }
#pragma unroll
        for (int w = 0; w < E / 8; ++w)
            out[w] = __byte_perm(__byte_perm(u[4 * w], u[4 * w + 1], 0x0040), __byte_perm(u[4 * w + 2], u[4 * w + 3], 0x0040),
                                 0x5410) ^ 0x88888888u;
    }
}

// Exchange-buffer geometry for a Hadamard block of 2^KLOG channels owned by N / E threads holding E values each.
template <int KLOG, int E>
struct FwhtShape {
    static constexpr int N = 1 << KLOG;
    static constexpr int LE = ilog2_c(E);
    static constexpr int P = E / 2;                    // two-wide registers per thread
    static constexpr int TB = N / E;                   // threads per Hadamard block
    static constexpr int R = KLOG - LE;                // index bits left for the second register phase
    static constexpr bool PAIR = R >= LE - 1;
    static constexpr bool SHUF = R == LE;
    static constexpr int J = PAIR ? E / 2 : E / 4;     // float4 slots a second-phase thread (pair) walks
    static constexpr int S = ilog2_c(J);
    static constexpr int GS = N / 4 + (N / 4) / J;     // padded float4 slots of the exchange buffer per Hadamard block
    static_assert(R <= LE, "block too large for this thread shape");
    static_assert(TB % J == 0 || J % TB == 0, "exchange layout needs TB and J to divide one another");
};

// All KLOG butterfly stages of one Hadamard block.  On entry thread tb of the block holds the float4s {tb + TB i} of the
// block (coalesced load order) as pairs; phase A covers index bits {0, 1} and the top log2(E) - 2 bits in registers, the
// values make one trip through the block's exchange buffer `grp` (float4 slot f at f + f / J, conflict-free both ways),
// and phase B covers the remaining bits in registers (KLOG = 12: one lane exchange more).  On exit thread u holds the E
// contiguous channels E u .. (or, PAIR, the channel pairs {4 j, 4 j + 1} + 2 (u & 1) of a 2E-channel group).
// (PAIR: the odd thread of a group holds its rows with the upper and the lower half of the pair-index range exchanged, so that
// pack_codes finds what a thread keeps and what it hands over in the same registers of both.)
// CTA_SYNC: the block's threads span more than one warp (or the caller needs a CTA-wide barrier here anyway).
// FIRST_DONE: the stage of index bit 0 has been taken as the values were read.  PAIR_STORE: without st_shared_pairs.
template <int KLOG, int E, bool CTA_SYNC, bool FIRST_DONE = false, bool PAIR_STORE = false>
__device__ __forceinline__ void fwht_stages(f32x2 (&v)[E / 2], float4* grp, int tb) {
    using Sh = FwhtShape<KLOG, E>;
    constexpr int P = Sh::P, TB = Sh::TB, J = Sh::J, S = Sh::S, R = Sh::R;
    if (!FIRST_DONE) butterfly_within_pairs<P>(v);     // index bit 0
    butterflies_pairs<P, 1, P / 2>(v);                 // index bit 1 and the top LE-2 bits
    {
        // slot f = tb + TB i sits at f + f / J; with TB and J dividing one another that is a per-thread base plus a
        // compile-time offset
        ulonglong2* wr = reinterpret_cast<ulonglong2*>(grp + tb + (tb >> S));
#pragma unroll
        for (int i = 0; i < E / 4; ++i) {
            ulonglong2* to = wr + TB * i + ((TB * i) >> S);
            if (PAIR_STORE) *to = make_ulonglong2(v[2 * i], v[2 * i + 1]);
            else st_shared_pairs(to, v[2 * i], v[2 * i + 1]);
        }
    }
    if (CTA_SYNC) __syncthreads(); else __syncwarp();
    if (!Sh::PAIR) {
        const ulonglong2* rd = reinterpret_cast<const ulonglong2*>(grp + (J + 1) * tb);
#pragma unroll
        for (int j = 0; j < E / 4; ++j) {
            const ulonglong2 q = rd[j];
            v[2 * j] = q.x; v[2 * j + 1] = q.y;
        }
        butterflies_pairs<P, 2, (2 << R) / 2>(v);      // index bits 2 .. R+1 are pair-index bits 1 .. R
    } else {
        const f32x2* rd = reinterpret_cast<const f32x2*>(grp + (J + 1) * (tb >> 1)) + (tb & 1);
        const f32x2* rd_lo = rd + (tb & 1) * P;
        const f32x2* rd_hi = rd - (tb & 1) * P;
#pragma unroll
        for (int j = 0; j < P; ++j) v[j] = (j < P / 2 ? rd_lo : rd_hi)[2 * j];
        butterflies_pairs<P, 1, P / 4>(v);             // index bits 2 .. LE are pair-index bits 0 .. LE-2
        {                                              // the last of them, whose operands the odd thread holds exchanged
            const float sg = (tb & 1) ? -1.0f : 1.0f;
            const f32x2 sg2 = pk2(sg, sg), msg2 = pk2(-sg, -sg);
#pragma unroll
            for (int i = 0; i < P / 2; ++i) {
                const f32x2 a = v[i], b = v[i + P / 2];
                v[i] = fma2(sg2, a, b);
                v[i + P / 2] = fma2(msg2, b, a);
            }
        }
        if (Sh::SHUF) {                                // index bit LE+1 lives in lane bit 1
            const float sgn = (tb & 2) ? -1.0f : 1.0f;
            const f32x2 sgn2 = pk2(sgn, sgn);
#pragma unroll
            for (int e = 0; e < P; ++e) {
                const f32x2 other = __shfl_xor_sync(0xffffffffu, v[e], 2);
                v[e] = fma2(sgn2, v[e], other);
            }
        }
    }
}

// Rounds and packs the E values a thread holds after fwht_stages into words of codes for the E contiguous channels
// E tb .. of the block (8 four-bit codes or 4 bytes per word).  In the PAIR layout the two threads of a group first
// exchange halves: w holds the codes of channel pairs {4j, 4j+1} (+2 for the odd thread); the even thread emits the first
// half of the group's bytes, the odd thread the second half (the first half of its registers), interleaved at pair granularity
// (1 byte or 2 bytes).
template <int KLOG, int E, bool INT8_OUT, bool CLAMP>
__device__ __forceinline__ void pack_codes(const f32x2 (&v)[E / 2], float inv, int bits, int tb,
                                           uint32_t (&w)[INT8_OUT ? E / 4 : E / 8]) {
    constexpr int NW = INT8_OUT ? E / 4 : E / 8;
    round_pack<E, INT8_OUT, CLAMP>(v, inv, bits, w);
    if (FwhtShape<KLOG, E>::PAIR) {
        constexpr int H = NW / 2;
        // first and second word of two: bytes (or nibbles) of the even and the odd thread in turn
        const uint32_t first = INT8_OUT ? 0x5410 : 0x5140, second = INT8_OUT ? 0x7632 : 0x7362, swap = (tb & 1) ? 0x4444 : 0;
        uint32_t o[NW];
#pragma unroll
        for (int i = 0; i < H; ++i) {
            const uint32_t recv = __shfl_xor_sync(0xffffffffu, w[i + H], 1);
            o[2 * i + 0] = __byte_perm(w[i], recv, first ^ swap);
            o[2 * i + 1] = __byte_perm(w[i], recv, second ^ swap);
        }
#pragma unroll
        for (int i = 0; i < NW; ++i) w[i] = o[i];
    }
}

// ---- the transform of Eq. 12's weight side, shared between weights and codes -----------------------------------
// The folded product sum_i q_i (H_raw W)_i needs weights of w_bits + k bits: two int8 limbs, twice the tensor work.  H_raw
// is a Kronecker product over the index bits, H_raw = prod of the factors of bits A times those of the bits not in A, and
// symmetric, so the same integers come out of z = (factors of A) q against B' = (factors of the other bits) W.  Four bits
// stay with 4-bit weights (|B'| <= 7 * 16), the other k - 4 go to the codes (|z| <= 2^(a_bits-1) * 2^(k-4)): where both fit
// a signed byte, ONE limb carries the whole product.  A is the k - 4 lowest of the order {2, 3, 4, 1, 0}: the index bits
// that a thread's 32 consecutive codes, four to a word, hold between words and then inside a word.
constexpr int kSplitWeightBits = 4;                    // index bits whose factors stay with the weights
__host__ __device__ constexpr bool split_block_ok(int klog) { return klog >= 5 && klog <= 9; }
// Blocks of 1024 .. 4096: four bits go to the codes, whatever their width, and the other k - 4 stay with the weights, whose
// integers then fit a byte (or, halved, nine bits) or not: the weight preparation looks (hq_weight.cu).
constexpr int kSplitWideCodeBits = 4;
__host__ __device__ constexpr bool split_wide(int klog) { return klog >= 10 && klog <= 12; }
__host__ __device__ constexpr int split_code_bits(int klog) { return klog <= 9 ? klog - kSplitWeightBits : kSplitWideCodeBits; }
__host__ __device__ constexpr int split_code_bit(int i) { return i < 3 ? 2 + i : 4 - i; }       // 2, 3, 4, 1, 0
// Whether z fits a signed byte for codes of a_bits bits (every row of H_raw but the first has as many -1 as +1).
__host__ __device__ constexpr bool split_fits(int klog, int a_bits) { return a_bits - 1 + split_code_bits(klog) <= 7; }

// Halved weights.  With k - 4 = 7 or 8 factors B' no longer fits a byte, but its entries have a common parity over the
// index bits that stay with the weights: that of their sum.  So with a the four code bits of a channel (bits 1 .. 4) and r the
// others, B'(a, r) = 2 B''(a, r) + w(a), w(a) = -1 or 0, and B'' is a byte again.  The product is
//   z . B' = 2 (z . B'') + sum_a w(a) sum_r z(a, r) = 2 (z . B'') + sum_p u(p) v(p),
// u(p) = sum_r q(p, r) the sums of the row's codes over r and v(p) = sum_a H(a, p) w(a).  All v(p) of a channel have one
// parity e, v = 2 v' + e, and with U = sum_p u(p) = 2 U' + Q the integer is
//   2 (z . B'' + sum_p u(p) v'(p) + e U') + e Q:
// the bracket is one product with 35 further columns on the reduction (one K block), e Q is added as the accumulator is read.
// Columns of that block, activations x weights: u(p) = 16 h + l as (h, 16 v') and (l, v'), U' = 128 c1 + c0 as (c1, 64 e) twice
// and (c0, e); the next byte of the activations' row holds Q, against a zero weight.
constexpr int kHalvedCols = 128;                       // bytes the further columns take in a row of either operand
constexpr int kHalvedH = 0, kHalvedL = 16, kHalvedC1 = 32, kHalvedC0 = 34, kHalvedQ = 35;
__host__ __device__ constexpr bool split_halved(int klog) { return klog == 11 || klog == 12; }

// u: 32 consecutive codes as bytes, biased by 128 >> A so that every sum below stays in its byte; on return z as signed
// bytes.  A byte-wise butterfly is two additions per word pair: a + b, and a - b + (the bias to come); inside a word the
// shifted copy comes from a multiplication by 2^16 +- 1 or 2^8 +- 1.  1.3 to 2 instructions per code.
template <int A>
__device__ __forceinline__ void split_butterflies(uint32_t (&u)[8]) {
    constexpr uint32_t kOnes = 0x01010101u;
#pragma unroll
    for (int i = 0; i < A; ++i) {
        const uint32_t bias = kOnes * uint32_t((128 >> A) << (i + 1));     // the bias after this stage
        if (i < 3) {
            const int h = 1 << i;
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                if (!(w & h)) {
                    const uint32_t a = u[w], b = u[w | h];
                    u[w] = a + b;
                    u[w | h] = a + bias - b;
                }
            }
        } else {
#pragma unroll
            for (int w = 0; w < 8; ++w) {
                // bytes 2, 3 of s and d: e0 + e2, e1 + e3 and e0 - e2, e1 - e3 (bit 0: bytes 1, 3: e0 + e1, e2 + e3, ...)
                const uint32_t s = u[w] * (i == 3 ? 0x00010001u : 0x00000101u);
                const uint32_t d = u[w] * (i == 3 ? 0x0000FFFFu : 0x000000FFu) + bias;
                u[w] = __byte_perm(s, d, i == 3 ? 0x7632 : 0x7351);
            }
        }
    }
#pragma unroll
    for (int w = 0; w < 8; ++w) u[w] ^= 0x80808080u;
}

// z of the 32 codes in w (8 words of bytes, or 4 words of nibbles, element 2j in the low one).
template <int KLOG, bool INT8_IN>
__device__ __forceinline__ void split_codes(const uint32_t (&w)[INT8_IN ? 8 : 4], uint32_t (&z)[8]) {
    constexpr int A = split_code_bits(KLOG);
    constexpr uint32_t kOnes = 0x01010101u, off = 128u >> A;
    if (INT8_IN) {
#pragma unroll
        for (int i = 0; i < 8; ++i) z[i] = (w[i] ^ 0x80808080u) - (128u - off) * kOnes;
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t n = w[i] ^ 0x88888888u;                         // code + 8 in every nibble
            const uint32_t ev = n & 0x0F0F0F0Fu, od = (n >> 4) & 0x0F0F0F0Fu;
            z[2 * i] = __byte_perm(ev, od, 0x5140) + off * kOnes - 8u * kOnes;
            z[2 * i + 1] = __byte_perm(ev, od, 0x7362) + off * kOnes - 8u * kOnes;
        }
    }
    split_butterflies<A>(z);
}

// The further columns of a row against halved weights.  w: the 64 consecutive codes of a thread; part: shared scratch of eight
// words per warp of the row when it has two (a row of 2^KLOG channels belongs to 2^(KLOG-6) threads, tb = 0 ..; every thread of
// the CTA calls).  Thread tb < 8 gets its 16 of the 128 bytes.
template <int KLOG, bool INT8_IN>
__device__ __forceinline__ uint4 halved_columns(const uint32_t (&w)[INT8_IN ? 16 : 8], uint32_t* part, int tb) {
    constexpr uint32_t kOnes = 0x01010101u;
    constexpr int kBias = (1 << KLOG) / 2;             // the codes are summed as code + 8, 2^KLOG / 16 to a sum
    uint32_t s[8];                                     // channel bits 2-4; the 16-bit fields are bit 1
    if (INT8_IN) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            const uint32_t t = ((w[i] ^ 0x80808080u) - 120u * kOnes) + ((w[i + 8] ^ 0x80808080u) - 120u * kOnes);
            s[i] = (t & 0x00FF00FFu) + ((t >> 8) & 0x00FF00FFu);
        }
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t n0 = w[i] ^ 0x88888888u, n1 = w[i + 4] ^ 0x88888888u;
            const uint32_t t = (n0 & 0x0F0F0F0Fu) + ((n0 >> 4) & 0x0F0F0F0Fu) + (n1 & 0x0F0F0F0Fu) + ((n1 >> 4) & 0x0F0F0F0Fu);
            s[2 * i] = __byte_perm(t, 0u, 0x4140);
            s[2 * i + 1] = __byte_perm(t, 0u, 0x4342);
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i] = __reduce_add_sync(0xffffffffu, s[i]);     // at most 32 * 60 a field
    if (KLOG == 12) {
        __syncthreads();
        if ((tb & 31) == 0) {
#pragma unroll
            for (int i = 0; i < 8; ++i) part[(tb >> 5) * 8 + i] = s[i];
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 8; ++i) s[i] += part[((tb >> 5) ^ 1) * 8 + i];
    }
    uint32_t hw[4], lw[4], tot = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t a = s[2 * i] + 0x00080008u, b = s[2 * i + 1] + 0x00080008u;
        tot += s[2 * i] + s[2 * i + 1];
        hw[i] = (__byte_perm(a >> 4, b >> 4, 0x6420) + uint32_t(128 - kBias / 16) * kOnes) ^ 0x80808080u;
        lw[i] = (__byte_perm(a & 0x000F000Fu, b & 0x000F000Fu, 0x6420) + 120u * kOnes) ^ 0x80808080u;
    }
    const int U = int(tot & 0xFFFFu) + int(tot >> 16) - 16 * kBias;
    const int half = U >> 1, c1 = (half + 64) >> 7, c0 = half - 128 * c1;
    const uint32_t c = uint32_t(c1 & 0xFF) * 0x0101u | uint32_t(c0 & 0xFF) << 16 | uint32_t(U & 1) << 24;
    if (tb == 0) return make_uint4(hw[0], hw[1], hw[2], hw[3]);
    if (tb == 1) return make_uint4(lw[0], lw[1], lw[2], lw[3]);
    return make_uint4(tb == 2 ? c : 0u, 0u, 0u, 0u);
}

}  // namespace hq
