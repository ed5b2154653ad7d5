// Offline weight side (host code): Eq. 3 per output channel, then one of
//   PLAIN   B = Q(W)
//   FOLDED  B = H_raw * Q(W)   -- the inner product of Eq. 12 / Eq. 14 kept in exact integers, computed with
//                                 integer butterflies over each block of input channels
//   DOUBLE  B = Q(H^T W)       -- Double-Hadamard weights (H orthonormal)
// and the byte layout the tensor-core kernels consume:
//   rows   128 output channels per group; with two limbs a group is 128 "hi" rows followed by 128 "lo" rows
//          (B = 256*hi + lo, lo in [-128,127]), so one 256-row operand tile carries both limbs of 128 channels;
//   K axis tap-major, each tap padded with zeros to a multiple of 128 channels; for the NIBBLE activation
//          container every 8 consecutive channels are stored in the order 0,2,4,6,1,3,5,7, which is the order
//          the in-kernel nibble unpack produces for the activation operand.
// FOLDED 4-bit weights with blocks of 32 .. 4096 channels carry a second section behind the first: the one-limb weights of
// the split fold, B' = (the factors of H_raw that stay with the weights) Q(W), whose product with the codes the fused
// layer calls' transform kernel leaves (split_codes in hq_fwht.cuh) is the same integer.  Natural channel order whatever
// the container; one row per output channel.  Up to 512 channels four factors stay and B' fits a byte whatever the weights; above,
// k - 4 stay, and the section is there where these weights' B' fit a byte or, for a linear layer of one block a row, where they
// fit when halved: rows of kHalvedCols further bytes, and behind the rows one byte per channel, the parity e (halved weights in
// hq_fwht.cuh).  Quantized Gaussian weights have B' of rms 17 at 1024 channels, 22 at 2048 (one layer of 512 rows in two has
// an entry above 127) and 30 at 4096 (four entries in 10^5 above): halved there, 8 standard deviations inside the byte.
#include <cmath>
#include <cstring>
#include <vector>

#include "hq_common.cuh"
#include "hq_fwht.cuh"

namespace hq {
namespace {

constexpr int kTileK = 128;
constexpr int kTileN = 128;

int64_t round_up(int64_t v, int64_t m) { return (v + m - 1) / m * m; }

int limbs_for(int w_bits, int had_block, hq_weight_mode mode) {
    if (mode == HQ_W_PLAIN_A2) return 2;
    if (mode != HQ_W_FOLDED || had_block <= 1) return 1;
    return (int64_t(had_block) << (w_bits - 1)) > 128 ? 2 : 1;
}

template <typename T>
void fwht_inplace(T* v, int n) {
    for (int h = 1; h < n; h <<= 1)
        for (int s = 0; s < n; s += 2 * h)
            for (int j = s; j < s + h; ++j) {
                const T a = v[j], b = v[j + h];
                v[j] = a + b;
                v[j + h] = a - b;
            }
}

bool split_section(int w_bits, int had_block, hq_weight_mode mode) {
    return mode == HQ_W_FOLDED && w_bits == 4 && had_block > 1 && is_pow2(had_block) && split_block_ok(ilog2(had_block));
}

bool wide_section(int w_bits, int had_block, hq_weight_mode mode) {
    return mode == HQ_W_FOLDED && w_bits == 4 && had_block > 1 && is_pow2(had_block) && split_wide(ilog2(had_block));
}
bool halved_layer(int RS, int64_t C, int had_block) { return RS == 1 && C == had_block && split_halved(ilog2(had_block)); }

// The factors of the index bits in `mask` of H_raw, on each block of n values.
void fwht_bits_inplace(int32_t* v, int n, int mask) {
    for (int h = 1; h < n; h <<= 1) {
        if (!(mask & h)) continue;
        for (int s = 0; s < n; s += 2 * h)
            for (int j = s; j < s + h; ++j) {
                const int32_t a = v[j], b = v[j + h];
                v[j] = a + b;
                v[j + h] = a - b;
            }
    }
}

// One channel of halved weights: B'' in `dst`, the further columns (kHalvedCols bytes) in `ext`; the parity e is returned.
int halve_channel(const int16_t* b, int n, int8_t* dst, int8_t* ext) {
    int w[16], odd = 0;
    for (int a = 0; a < 16; ++a) w[a] = -(b[2 * a] & 1);            // channel 2 a has the code bits a
    for (int c = 0; c < n; ++c) dst[c] = int8_t((b[c] - w[(c >> 1) & 15]) / 2);
    for (int a = 0; a < 16; ++a) odd ^= w[a] & 1;
    for (int p = 0; p < 16; ++p) {
        int v = 0;
        for (int a = 0; a < 16; ++a) v += __builtin_parity(unsigned(a & p)) ? -w[a] : w[a];
        v = (v - odd) / 2;                                          // -8 .. 4
        ext[kHalvedH + p] = int8_t(16 * v);
        ext[kHalvedL + p] = int8_t(v);
    }
    ext[kHalvedC1] = ext[kHalvedC1 + 1] = int8_t(64 * odd);
    ext[kHalvedC0] = int8_t(odd);
    return odd;
}

// Above 512 channels desc->bytes tells the fused calls whether and in which form the section is there.  The buffer asked for is
// a little longer than either form, so that a descriptor that was given the buffer's size instead says that there is none.
constexpr int64_t kWideSpare = 16;

void quantize_channel(const double* w, int64_t count, int w_bits, int32_t* out, float* scale) {
    const int qmax = kQmax(w_bits), qmin = kQmin(w_bits);
    double amax = 0.0;
    for (int64_t i = 0; i < count; ++i) amax = std::fmax(amax, std::fabs(w[i]));
    float s = amax > 0.0 ? float(amax / double(qmax)) : 1.0f;
    if (!(s > 0.0f)) s = 1.0f;
    *scale = s;
    for (int64_t i = 0; i < count; ++i) {
        double c = std::nearbyint(w[i] / double(s));
        c = std::fmin(std::fmax(c, double(qmin)), double(qmax));
        out[i] = int32_t(c);
    }
}

}  // namespace
}  // namespace hq

extern "C" int64_t hq_weight_blob_bytes(int64_t N, int32_t RS, int64_t C, int32_t w_bits, int32_t had_block,
                                        hq_weight_mode mode) {
    if (N <= 0 || RS <= 0 || C <= 0) return 0;
    const int limbs = hq::limbs_for(w_bits, had_block, mode);
    const int64_t Ck = mode == HQ_W_PLAIN_A2 ? 2 * C : C;          // channels per tap along K
    const int64_t limb = hq::round_up(N, hq::kTileN) * RS * hq::round_up(Ck, hq::kTileK);
    const bool wide = limbs == 2 && hq::wide_section(w_bits, had_block, mode);
    return limb * (limbs + (wide || (limbs == 2 && hq::split_section(w_bits, had_block, mode)) ? 1 : 0)) +
           (wide && hq::halved_layer(RS, C, had_block) ? hq::round_up(N, hq::kTileN) * (hq::kHalvedCols + 1) : 0) +
           (wide ? hq::kWideSpare : 0);
}

extern "C" hq_status hq_weight_prepare(const float* w, int64_t N, int32_t RS, int64_t C, int32_t w_bits,
                                       int32_t had_block, hq_weight_mode mode, hq_container container, void* blob,
                                       int64_t blob_bytes, float* s_w, hq_weight_desc* desc) {
    using namespace hq;
    if (w == nullptr || blob == nullptr || s_w == nullptr || desc == nullptr) return HQ_ERR_INVALID_ARG;
    if (w_bits != 4 && w_bits != 8) return HQ_ERR_INVALID_ARG;
    if (mode != HQ_W_PLAIN && mode != HQ_W_FOLDED && mode != HQ_W_DOUBLE && mode != HQ_W_PLAIN_A2) return HQ_ERR_INVALID_ARG;
    if (mode == HQ_W_PLAIN_A2 && container != HQ_CODES_INT8) return HQ_ERR_SHAPE;
    if (container != HQ_CODES_NIBBLE && container != HQ_CODES_INT8) return HQ_ERR_INVALID_ARG;
    if (N <= 0 || RS <= 0 || C <= 0) return HQ_ERR_SHAPE;
    const int n = had_block > 1 ? had_block : 1;
    if (n > 1 && (!is_pow2(n) || C % n != 0)) return HQ_ERR_SHAPE;
    if (container == HQ_CODES_NIBBLE && C % 8 != 0) return HQ_ERR_SHAPE;
    const int limbs = limbs_for(w_bits, had_block, mode);
    const bool a2 = mode == HQ_W_PLAIN_A2;
    const int64_t Ck = a2 ? 2 * C : C;                              // channels per tap along K
    const int64_t C_pad = round_up(Ck, kTileK), N_pad = round_up(N, kTileN);
    const int64_t Kp = int64_t(RS) * C_pad;
    const int64_t base = N_pad * limbs * Kp;
    if (blob_bytes < base) return HQ_ERR_WORKSPACE;
    // a buffer of the two-limb section's size alone is taken as well: the layer then runs on two limbs
    const bool split = limbs == 2 && split_section(w_bits, had_block, mode) && blob_bytes >= base + N_pad * Kp;
    bool wide = limbs == 2 && wide_section(w_bits, had_block, mode) && blob_bytes >= base + N_pad * Kp;
    bool halved = wide && halved_layer(RS, C, n) && blob_bytes >= base + N_pad * (Kp + kHalvedCols + 1);
    int64_t need = base + (split ? N_pad * Kp : 0);
    int weight_mask = 0;                                            // index bits whose factors stay with the one-limb weights
    if (split || wide) {
        weight_mask = n - 1;
        for (int i = 0; i < split_code_bits(ilog2(n)); ++i) weight_mask &= ~(1 << split_code_bit(i));
    }

    const int64_t KK = int64_t(RS) * C;
    std::vector<double> row(KK);
    std::vector<int32_t> B(KK);
    std::vector<int16_t> B1(wide ? size_t(N * KK) : 0);
    bool direct = wide;
    int8_t* out = static_cast<int8_t*>(blob);
    std::memset(out, 0, size_t(need));
    int32_t max_abs = 0;

    for (int64_t o = 0; o < N; ++o) {
        for (int64_t i = 0; i < KK; ++i) row[i] = double(w[o * KK + i]);
        if (mode == HQ_W_DOUBLE && n > 1) {
            const double norm = std::exp2(-0.5 * double(ilog2(n)));
            for (int64_t b = 0; b < KK / n; ++b) {
                fwht_inplace(row.data() + b * n, n);
                for (int j = 0; j < n; ++j) row[b * n + j] *= norm;
            }
        }
        quantize_channel(row.data(), KK, w_bits, B.data(), &s_w[o]);
        if (weight_mask != 0)
            for (int64_t b = 0; b < KK / n; ++b) fwht_bits_inplace(B.data() + b * n, n, weight_mask);
        if (split) {
            for (int t = 0; t < RS; ++t)
                for (int64_t c = 0; c < C; ++c) {
                    // 16 integers of -8 .. 7 (-8 only where the scale is subnormal or a weight no number) under the signs of
                    // a Hadamard row: all of one sign, at least 16 * -8 and at most 16 * 7, or eight of each, at most 8 * 8 + 8 * 7
                    out[base + o * Kp + int64_t(t) * C_pad + c] = int8_t(B[t * C + c]);
                }
        }
        if (wide) {
            for (int64_t i = 0; i < KK; ++i) {                      // at most 256 * 8
                B1[o * KK + i] = int16_t(B[i]);
                direct = direct && B[i] >= -128 && B[i] <= 127;
                halved = halved && B[i] >= -256 && B[i] <= 254;     // (B + parity) / 2 a signed byte
            }
            wide = direct || halved;
        }
        if (mode == HQ_W_FOLDED && n > 1)                           // the remaining factors
            for (int64_t b = 0; b < KK / n; ++b) fwht_bits_inplace(B.data() + b * n, n, (n - 1) & ~weight_mask);

        const int64_t grp = o / kTileN, within = o % kTileN;
        for (int t = 0; t < RS; ++t) {
            for (int64_t c = 0; c < Ck; ++c) {
                // two activation limbs: the channels of a tap are [hi(C) | lo(C)] and B = [256 Q(W) | Q(W)], whose limb
                // split below gives the "hi" rows [Q(W) | 0] and the "lo" rows [0 | Q(W)]
                const int32_t v = a2 ? (c < C ? 256 * B[t * C + c] : B[t * C + (c - C)]) : B[t * C + c];
                max_abs = std::max(max_abs, v < 0 ? -v : v);
                // position along K inside the tap
                int64_t pos = c;
                if (container == HQ_CODES_NIBBLE) {
                    // slot p of an 8-group holds channel {0,2,4,6,1,3,5,7}[p]; this is the inverse map
                    const int r = int(c & 7);
                    const int slot = (r & 1) ? 4 + (r >> 1) : (r >> 1);
                    pos = (c & ~int64_t(7)) + slot;
                }
                const int64_t k = int64_t(t) * C_pad + pos;
                if (limbs == 1) {
                    if (v < -128 || v > 127) return HQ_ERR_OVERFLOW_RISK;
                    out[(grp * kTileN + within) * Kp + k] = int8_t(v);
                } else {
                    const int32_t lo = ((v + 128) & 255) - 128;
                    const int32_t hi = (v - lo) / 256;
                    if (hi < -128 || hi > 127) return HQ_ERR_OVERFLOW_RISK;
                    out[(grp * 2 * kTileN + within) * Kp + k] = int8_t(hi);
                    out[(grp * 2 * kTileN + kTileN + within) * Kp + k] = int8_t(lo);
                }
            }
        }
    }
    if (wide) {
        const int64_t pitch = direct ? Kp : Kp + kHalvedCols;
        const int64_t section = N_pad * pitch + (direct ? 0 : N_pad);
        std::memset(out + base, 0, size_t(section));
        for (int64_t o = 0; o < N; ++o) {
            int8_t* dst = out + base + o * pitch;
            const int16_t* b1 = B1.data() + o * KK;
            if (direct) {
                for (int t = 0; t < RS; ++t)
                    for (int64_t c = 0; c < C; ++c) dst[int64_t(t) * C_pad + c] = int8_t(b1[t * C + c]);
            } else {
                out[base + N_pad * pitch + o] = int8_t(halve_channel(b1, int(C), dst, dst + Kp));
            }
        }
        need = base + section;
    }
    desc->N = N; desc->C = Ck; desc->RS = RS; desc->w_bits = w_bits; desc->had_block = had_block;
    desc->mode = int32_t(mode); desc->limbs = limbs; desc->container = int32_t(container);
    desc->C_pad = C_pad; desc->N_pad = N_pad; desc->bytes = need; desc->max_abs_b = max_abs;
    desc->reserved = split ? kBlobHasSplit : 0;
    return HQ_OK;
}

extern "C" float hq_alpha_for(const hq_weight_desc* desc) {
    if (desc == nullptr) return 1.0f;
    if (desc->mode == HQ_W_FOLDED && desc->had_block > 1)
        return float(std::exp2(-0.5 * double(hq::ilog2(desc->had_block))));
    return 1.0f;
}
