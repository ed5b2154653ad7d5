// Entry points that are not a kernel of their own: status helpers and the fused layer calls, which run
// transform+quantize (Eq. 10, Eq. 3) and then the integer product with its rescale (Eq. 12 / Eq. 14) on one stream.
#include <mutex>

#include "hq_common.cuh"
#include "hq_fwht.cuh"

// Scratch of hq_qlinear_noalloc: part of the library's device image, one copy per GPU that loads the library.
// In host code this name is only a handle for cudaGetSymbolAddress, never a device pointer.
static __device__ __align__(256) unsigned char hq_noalloc_scratch[HQ_NOALLOC_SCRATCH_BYTES];

namespace hq {
hq_status launch_hadamard_quant(const void* x, hq_dtype xdt, int64_t rows, int64_t cols, int64_t ldx, int had_block,
                                int bits, hq_scale_mode mode, const float* static_scale, void* codes,
                                hq_container cont, int64_t ld_codes, float* scales, cudaStream_t st, SplitOut* zo = nullptr);
hq_status launch_qgemm(const void* a_codes, hq_container cont, int a_bits, int64_t M, int64_t K, int64_t lda,
                       const hq_weight_desc* desc, const void* w_dev, const float* scale_a, int scale_a_is_scalar,
                       const float* scale_w, const float* bias, float alpha, int32_t* acc_out, void* y,
                       hq_dtype ydt, int64_t ldy, int32_t* dev_status, cudaStream_t st, bool after_quant,
                       const HalvedParity* halved = nullptr, ResidualAdd* res = nullptr);
bool halved_product_covers(int64_t M, const void* y, hq_dtype ydt, int64_t ldy);      // hq_gemm.cu
hq_status launch_qconv2d(const void* a_codes, hq_container cont, int a_bits, int64_t Nb, int64_t H, int64_t W,
                         int64_t C, const hq_weight_desc* desc, const void* w_dev, int R, int S, int stride, int pad,
                         const float* scale_a, int scale_a_is_scalar, const float* scale_w, const float* bias,
                         float alpha, int32_t* acc_out, void* y, hq_dtype ydt, int32_t* dev_status, cudaStream_t st,
                         bool after_quant, ResidualAdd* res = nullptr);

hq_status launch_gn_silu_quant(const void* x, hq_dtype xdt, int64_t Nb, int64_t H, int64_t W, int64_t C, int groups,
                               const float* gamma, const float* beta, float eps, int had_block, int bits,
                               hq_scale_mode mode, const float* static_scale, void* codes, hq_container cont,
                               int64_t ld_codes, float* scales, void* scratch, size_t scratch_bytes, cudaStream_t st,
                               int silu, const void* pre_bias, int64_t pre_ld, const void* x2, int64_t split, SplitOut* zo = nullptr);
hq_status launch_hadamard_quant_cat(const void* x, int64_t ldx, const void* x2, int64_t ldx2, int64_t split, hq_dtype xdt,
                                    int64_t rows, int64_t cols, int had_block, int bits, hq_scale_mode mode,
                                    const float* static_scale, void* codes, hq_container cont, int64_t ld_codes,
                                    float* scales, cudaStream_t st, SplitOut* zo = nullptr);
hq_status launch_ln_quant(const void* x, hq_dtype xdt, int64_t rows, int64_t cols, int64_t ldx, const float* weight,
                          const float* bias, int64_t rows_per_group, float eps, int had_block, int bits,
                          hq_scale_mode mode, const float* static_scale, void* codes, hq_container cont, int64_t ld_codes,
                          float* scales, cudaStream_t st, SplitOut* zo = nullptr);
hq_status launch_hadamard_quant_width(const void* x, hq_dtype xdt, int64_t Nb, int64_t H, int64_t W, int64_t C,
                                      int had_block_w, int bits, const float* static_scale, void* z, float* scale_out,
                                      cudaStream_t st);
hq_status launch_hadamard_quant_width2(const void* x, hq_dtype xdt, int64_t Nb, int64_t H, int64_t W, int64_t C,
                                       int had_block_w, int bits, const float* static_scale, void* z_limbs,
                                       float* scale_out, cudaStream_t st);

int sm_count();             // hq_gemm.cu: SM count of the current device
// hq_small.cu: a linear layer of few rows as one kernel
bool small_linear_takes(const void* x, hq_dtype xdt, int64_t M, int64_t K, int64_t ldx, const hq_weight_desc* desc, const void* w_dev,
                        const float* scale_w, int a_bits, hq_scale_mode mode, const float* static_scale, const void* y, hq_dtype ydt,
                        int64_t ldy, const void* workspace, int64_t ws_used);
hq_status launch_small_linear(const void* x, hq_dtype xdt, int64_t M, int64_t K, int64_t ldx, const hq_weight_desc* desc, const void* w_dev,
                              const float* scale_w, const float* bias, int a_bits, hq_scale_mode mode, const float* static_scale,
                              float alpha, void* y, int64_t ldy, void* codes, int64_t ld_codes, float* scales, cudaStream_t st);

namespace {
int64_t code_pitch(int64_t cols, hq_container cont) {
    const int64_t b = cont == HQ_CODES_NIBBLE ? cols / 2 : cols;
    return (b + 15) / 16 * 16;
}
int64_t scales_offset(int64_t rows, int64_t cols, hq_container cont) {
    return (rows * code_pitch(cols, cont) + 255) / 256 * 256;
}
// Codes and scales; behind them, where the caller's workspace has room for it, the split-fold codes z of the layer.
int64_t codes_bytes(int64_t rows, int64_t cols, hq_container cont) {
    return scales_offset(rows, cols, cont) + (rows > 0 ? rows : 1) * int64_t(sizeof(float));
}
int64_t split_offset(int64_t rows, int64_t cols, hq_container cont) { return (codes_bytes(rows, cols, cont) + 255) / 256 * 256; }
int64_t split_bytes(int64_t rows, int64_t cols, hq_container cont) {
    return split_offset(rows, cols, cont) + rows * code_pitch(cols, HQ_CODES_INT8);
}
int64_t halved_bytes(int64_t rows, int64_t cols, hq_container cont) {
    return split_offset(rows, cols, cont) + rows * (cols + kHalvedCols);
}

// What a fused layer call cannot do without: its codes and scales.
hq_status layer_bytes(int64_t rows, int64_t cols, hq_container cont, size_t* bytes) {
    if (cont != HQ_CODES_NIBBLE && cont != HQ_CODES_INT8) return HQ_ERR_INVALID_ARG;
    if (rows < 0 || cols <= 0) return HQ_ERR_SHAPE;
    *bytes = size_t(codes_bytes(rows, cols, cont));
    return HQ_OK;
}

// The intermediate of a fused layer call in its workspace, and the operands its product runs on: the codes and the weights
// as prepared, or (after the transform kernel has said that it wrote them) the split-fold codes and the one-limb weights
// behind the two-limb ones in the blob.  The sums are the same integers either way.
struct LayerCodes {
    unsigned char* codes;
    float* scales;
    int64_t ld;
    SplitOut z{};
    hq_weight_desc split_desc;
    const void* split_w;

    HalvedParity parity;

    // rows x cols codes.  The caller has refused a null w_dev: split_w is never null, so the product's own check no longer
    // sees one.  halved_ok: the product is one that halved weights are read by (halved_product_covers).
    LayerCodes(const hq_weight_desc* desc, const void* w_dev, int a_bits, hq_scale_mode mode, int64_t rows, int64_t cols, int stride,
               hq_container cont, void* workspace, size_t ws_bytes, bool halved_ok)
        : codes(static_cast<unsigned char*>(workspace)),
          scales(reinterpret_cast<float*>(codes + scales_offset(rows, cols, cont))), ld(code_pitch(cols, cont)) {
        const Section sec = section(desc, a_bits, cols);
        if (sec == kNone || (sec == kHalved && !halved_ok)) return;
        const int64_t room = sec == kHalved ? halved_bytes(rows, cols, cont) : split_bytes(rows, cols, cont);
        if (ws_bytes < size_t(room) || !split_taken(desc, a_bits, mode, rows, cols, stride)) return;
        z.z = codes + split_offset(rows, cols, cont);
        z.ld = sec == kHalved ? cols + kHalvedCols : code_pitch(cols, HQ_CODES_INT8);
        z.halved = sec == kHalved;
        split_desc = *desc;
        split_desc.limbs = 1;
        split_desc.container = HQ_CODES_INT8;
        split_w = static_cast<const unsigned char*>(w_dev) + desc->N_pad * 2 * desc->RS * desc->C_pad;
        if (z.halved) {
            split_desc.C += kHalvedCols;
            split_desc.C_pad += kHalvedCols;
            parity = HalvedParity{z.z + cols + kHalvedQ, z.ld, static_cast<const uint8_t*>(split_w) + desc->N_pad * split_desc.C_pad};
        }
    }
    // The one-limb section behind the two-limb weights, and whether codes of a_bits bits can be multiplied with it.
    enum Section { kNone, kBytes, kHalved };
    static Section section(const hq_weight_desc* desc, int a_bits, int64_t cols) {
        if (desc->limbs != 2 || desc->C != cols || cols >= 131072) return kNone;
        const int klog = ilog2(desc->had_block);
        if (!split_fits(klog, a_bits)) return kNone;
        if (split_block_ok(klog)) return desc->reserved == kBlobHasSplit ? kBytes : kNone;
        if (!split_wide(klog) || desc->mode != HQ_W_FOLDED) return kNone;
        const int64_t more = desc->bytes - desc->N_pad * 2 * desc->RS * desc->C_pad;      // what the preparation put there
        return more == desc->N_pad * desc->RS * desc->C_pad ? kBytes
             : more == desc->N_pad * (desc->C_pad + kHalvedCols + 1) ? kHalved : kNone;
    }
    static bool split_taken(const hq_weight_desc* desc, int a_bits, hq_scale_mode mode, int64_t rows, int64_t cols, int stride) {
        const Section sec = section(desc, a_bits, cols);
        return sec != kNone &&
               split_pays(desc, rows, cols, rows / (stride == 2 ? 4 : 1), sec == kHalved ? kHalvedCols / 128 : 0);
    }
    // One limb halves the column tiles (or the weights a CTA of the split kernel streams), and the transform kernel computes
    // and writes a second byte per code, which costs 0.7 us plus its traffic at about 5.2 TB/s.  Measured (two limbs / one):
    // 8192 x 1152 -> 4608 57.9 / 44.2 us, 64 x 32 x 32 x 512 3x3 176 / 117 us, 2 x 16 x 16 x 768 3x3 13.1 / 11.8 us; where
    // no round of tiles is saved it only costs: 256 x 256 -> 256 6.1 / 6.8 us, 8 x 64 x 64 x 256 3x3 stride 2 16.5 / 17.6.
    // Blocks above 512, the same rule: 65536 x 4096 -> 4096 1657 / 1127 us (the second byte costs the transform 84 of its 341 us),
    // 65536 x 4096 -> 1024 536 / 487, 32768 x 2048 -> 2048 195 / 161, 65536 x 1024 -> 1024 125 / 113.  The transform's threads hold 64
    // values, and the second byte travels at about 4.6 TB/s; at 4096 with one code per byte, where both bytes change lanes before
    // they are stored, at 3.4.  With one code per byte, taken: 65536 x 2048 -> 512 187.6 / 185 (bf16 input 172 / 166), 32768 x 1024 ->
    // 1024 70.0 / 66.5, 32768 x 2048 -> 768 114.6 / 109; not taken: 32768 x 2048 -> 512 95.5 / 99.0, 32768 x 1024 -> 512 50.8 / 57.8,
    // 16384 x 4096 -> 512 103.5 / 108.5, 32768 x 4096 -> 512 194 / 204.5.  At 28 shapes of 4096 to 65536 rows and 256 to 2048 channels, both
    // containers and input types, what it takes is within 3 % of the faster form.
    static bool split_pays(const hq_weight_desc* desc, int64_t rows, int64_t cols, int64_t out_rows, int more_kb) {
        const int num_kb = int(desc->RS * desc->C_pad / 128), tile_rows = out_rows < 128 ? int(out_rows > 0 ? out_rows : 1) : 128;
        // with two codes per byte the two-limb product unpacks them on one SM a tile (32768 x 2048 -> 512 52 us against 45): the whole
        // layer taken at 32768 x 1024 -> 512 53.6 / 50.0, 32768 x 2048 -> 512 96.0 / 91.3, 32768 x 4096 -> 512 199.4 / 197.4, 16384 x
        // 4096 -> 512 105.4 / 102.1; not taken at 65536 x 1024 -> 256 76.0 / 82.4, 65536 x 4096 -> 384 354 / 372
        const bool unpacks = desc->container == HQ_CODES_NIBBLE && desc->had_block > 512;
        const double two = plan_product(2, out_rows, tile_rows, desc->N_pad, num_kb).us * (unpacks ? 1.15 : 1.0);
        const double one = plan_product(1, out_rows, tile_rows, desc->N_pad, num_kb + more_kb).us;
        const bool lanes = desc->had_block == 4096 && !unpacks;              // staged_stores in hq_quant.cu
        return two - one > 0.7 + double(rows) * double(cols) / (desc->had_block <= 512 ? 5.2e6 : lanes ? 3.4e6 : 4.6e6);
    }
    const void* a() const { return z.written ? z.z : codes; }
    int64_t lda() const { return z.written ? z.ld : ld; }
    hq_container container(hq_container cont) const { return z.written ? HQ_CODES_INT8 : cont; }
    const hq_weight_desc* desc(const hq_weight_desc* d) const { return z.written ? &split_desc : d; }
    const void* w(const void* w_dev) const { return z.written ? split_w : w_dev; }
    int64_t k(int64_t K) const { return z.written && z.halved ? K + kHalvedCols : K; }
    const HalvedParity* halved() const { return z.written && z.halved ? &parity : nullptr; }
};

// A residual that a fused layer call adds to its bf16 output: checked before anything is launched, added by the product kernel
// where that takes it and by a launch of its own where not (other kernels, and halved weights).
hq_status check_residual(const void* residual, const void* y, hq_dtype ydt, int64_t N, int64_t ldy) {
    if (residual == nullptr) return HQ_OK;
    if (residual == y || ydt != HQ_BF16) return HQ_ERR_INVALID_ARG;
    if (N % 8 != 0 || ldy != N) return HQ_ERR_SHAPE;
    return aligned16(residual) && aligned16(y) ? HQ_OK : HQ_ERR_ALIGNMENT;
}
hq_status finish_residual(hq_status s, const ResidualAdd& res, void* y, int64_t count, void* stream) {
    if (s != HQ_OK || res.r == nullptr || res.done) return s;
    return hq_add(y, res.r, count, y, stream);
}
}  // namespace
}  // namespace hq

extern "C" int hq_version(void) { return 100; }

extern "C" const char* hq_status_string(hq_status s) {
    switch (s) {
        case HQ_OK: return "ok";
        case HQ_ERR_INVALID_ARG: return "invalid argument";
        case HQ_ERR_SHAPE: return "inconsistent shape";
        case HQ_ERR_UNSUPPORTED: return "unsupported configuration";
        case HQ_ERR_ALIGNMENT: return "misaligned pointer or pitch";
        case HQ_ERR_WORKSPACE: return "workspace too small";
        case HQ_ERR_OVERFLOW_RISK: return "int32 accumulator could overflow";
        case HQ_ERR_CUDA: return "CUDA call failed";
        case HQ_ERR_TIMEOUT: return "device-side wait timed out";
        case HQ_ERR_SCRATCH_LIMIT: return "layer exceeds the built-in scratch of the no-allocation entry point";
    }
    return "unknown status";
}

extern "C" hq_status hq_check_status(const int32_t* dev_status_host_copy) {
    if (dev_status_host_copy == nullptr) return HQ_ERR_INVALID_ARG;
    return *dev_status_host_copy == 0 ? HQ_OK : HQ_ERR_TIMEOUT;
}

extern "C" hq_status hq_workspace_size(int64_t rows, int64_t cols, hq_container cont, size_t* bytes) {
    if (bytes == nullptr) return HQ_ERR_INVALID_ARG;
    if (cont != HQ_CODES_NIBBLE && cont != HQ_CODES_INT8) return HQ_ERR_INVALID_ARG;
    if (rows < 0 || cols <= 0) return HQ_ERR_SHAPE;
    // Codes and scales; beyond HQ_NOALLOC_SCRATCH_BYTES also room for the split-fold codes, since the shape does not say
    // whether the layer has a use for it.  Smaller layers gain from it as well (4096 x 1152 -> 4608 30.7 / 24.5 us), but for
    // them this is the size at which the no-allocation entry point takes a layer: they ask hq_layer_workspace_size.
    *bytes = size_t(hq::codes_bytes(rows, cols, cont));
    if (*bytes > size_t(HQ_NOALLOC_SCRATCH_BYTES))
        *bytes = size_t(cols == 2048 || cols == 4096 ? hq::halved_bytes(rows, cols, cont) : hq::split_bytes(rows, cols, cont));
    return HQ_OK;
}

// Two limbs / one, whole layer: 1024 x 1152 -> 4608 12.7 / 11.3 us, 4096 x 1152 -> 4608 30.7 / 24.5, 7000 x 1024 -> 4096 41.6 / 35.3,
// 16 x 16 x 16 x 768 3x3 38.5 / 21.6, 15 x 32 x 32 x 512 3x3 51.4 / 33.2, 64 x 8 x 8 x 1024 3x3 48.7 / 30.4.
extern "C" hq_status hq_layer_workspace_size(const hq_weight_desc* desc, int a_bits, hq_scale_mode mode, int64_t rows, int stride,
                                             size_t* bytes) {
    using namespace hq;
    if (desc == nullptr || bytes == nullptr) return HQ_ERR_INVALID_ARG;
    if (mode != HQ_SCALE_PER_ROW && mode != HQ_SCALE_STATIC) return HQ_ERR_INVALID_ARG;
    if (a_bits != 3 && a_bits != 4 && a_bits != 8) return HQ_ERR_INVALID_ARG;
    if (stride != 1 && stride != 2) return HQ_ERR_UNSUPPORTED;
    const hq_container cont = hq_container(desc->container);
    const hq_status s = layer_bytes(rows, desc->C, cont, bytes);
    if (s != HQ_OK) return s;
    if (desc->had_block <= 512 && (mode == HQ_SCALE_STATIC || desc->RS == 1) &&
        LayerCodes::split_taken(desc, a_bits, mode, rows, desc->C, stride))
        *bytes = size_t(split_bytes(rows, desc->C, cont));
    return HQ_OK;
}

static hq_status qlinear_impl(const void* x, hq_dtype xdt, int64_t M, int64_t K, int64_t ldx, const hq_weight_desc* desc,
                              const void* w_dev, const float* scale_w, const float* bias, int a_bits, hq_scale_mode mode,
                              const float* static_scale, void* y, hq_dtype ydt, int64_t ldy, const void* residual, void* workspace,
                              size_t ws_bytes, int32_t* dev_status, void* stream) {
    using namespace hq;
    if (desc == nullptr || w_dev == nullptr || workspace == nullptr || y == nullptr) return HQ_ERR_INVALID_ARG;
    if (!aligned16(workspace)) return HQ_ERR_ALIGNMENT;
    const hq_container cont = hq_container(desc->container);
    size_t need = 0;
    hq_status s = layer_bytes(M, K, cont, &need);
    if (s != HQ_OK) return s;
    if (ws_bytes < need) return HQ_ERR_WORKSPACE;
    s = check_residual(residual, y, ydt, desc->N, ldy);
    if (s != HQ_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (residual == nullptr && small_linear_takes(x, xdt, M, K, ldx, desc, w_dev, scale_w, a_bits, mode, static_scale, y, ydt, ldy,
                                               workspace, int64_t(need)))
        return launch_small_linear(x, xdt, M, K, ldx, desc, w_dev, scale_w, bias, a_bits, mode, static_scale, hq_alpha_for(desc), y, ldy,
                                   workspace, code_pitch(K, cont),
                                   reinterpret_cast<float*>(static_cast<unsigned char*>(workspace) + scales_offset(M, K, cont)), st);
    ResidualAdd res{static_cast<const __nv_bfloat16*>(residual), false};
    LayerCodes lc(desc, w_dev, a_bits, mode, M, K, 1, cont, workspace, ws_bytes, halved_product_covers(M, y, ydt, ldy));
    s = launch_hadamard_quant(x, xdt, M, K, ldx, desc->had_block, a_bits, mode, static_scale, lc.codes, cont, lc.ld, lc.scales, st,
                              &lc.z);
    if (s != HQ_OK) return s;
    s = launch_qgemm(lc.a(), lc.container(cont), a_bits, M, lc.k(K), lc.lda(), lc.desc(desc), lc.w(w_dev), lc.scales, mode == HQ_SCALE_STATIC, scale_w, bias,
                     hq_alpha_for(desc), nullptr, y, ydt, ldy, dev_status, st, true, lc.halved(), residual != nullptr ? &res : nullptr);
    return finish_residual(s, res, y, M * desc->N, stream);
}

extern "C" hq_status hq_qlinear(const void* x, hq_dtype xdt, int64_t M, int64_t K, int64_t ldx,
                                const hq_weight_desc* desc, const void* w_dev, const float* scale_w,
                                const float* bias, int a_bits, hq_scale_mode mode, const float* static_scale, void* y,
                                hq_dtype ydt, int64_t ldy, void* workspace, size_t ws_bytes, int32_t* dev_status,
                                void* stream) {
    return qlinear_impl(x, xdt, M, K, ldx, desc, w_dev, scale_w, bias, a_bits, mode, static_scale, y, ydt, ldy, nullptr, workspace,
                        ws_bytes, dev_status, stream);
}

// The linear layer with a residual added to its rounded output (the output projection of an attention block).
extern "C" hq_status hq_qlinear_add(const void* x, hq_dtype xdt, int64_t M, int64_t K, int64_t ldx, const hq_weight_desc* desc,
                                    const void* w_dev, const float* scale_w, const float* bias, int a_bits, const void* residual,
                                    void* y, void* workspace, size_t ws_bytes, int32_t* dev_status, void* stream) {
    if (residual == nullptr || desc == nullptr) return HQ_ERR_INVALID_ARG;
    return qlinear_impl(x, xdt, M, K, ldx, desc, w_dev, scale_w, bias, a_bits, HQ_SCALE_PER_ROW, nullptr, y, HQ_BF16, desc->N,
                        residual, workspace, ws_bytes, dev_status, stream);
}

extern "C" hq_status hq_ln_qlinear(const void* x, hq_dtype xdt, int64_t M, int64_t K, int64_t ldx, const float* ln_weight,
                                   const float* ln_bias, int64_t rows_per_group, float eps, const hq_weight_desc* desc,
                                   const void* w_dev, const float* scale_w, const float* bias, int a_bits, void* y,
                                   hq_dtype ydt, int64_t ldy, void* workspace, size_t ws_bytes, int32_t* dev_status,
                                   void* stream) {
    using namespace hq;
    if (desc == nullptr || w_dev == nullptr || workspace == nullptr || y == nullptr) return HQ_ERR_INVALID_ARG;
    if (!aligned16(workspace)) return HQ_ERR_ALIGNMENT;
    const hq_container cont = hq_container(desc->container);
    size_t need = 0;
    hq_status s = layer_bytes(M, K, cont, &need);
    if (s != HQ_OK) return s;
    if (ws_bytes < need) return HQ_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    LayerCodes lc(desc, w_dev, a_bits, HQ_SCALE_PER_ROW, M, K, 1, cont, workspace, ws_bytes, false);
    s = launch_ln_quant(x, xdt, M, K, ldx, ln_weight, ln_bias, rows_per_group, eps, desc->had_block, a_bits, HQ_SCALE_PER_ROW,
                        nullptr, lc.codes, cont, lc.ld, lc.scales, st, &lc.z);
    if (s != HQ_OK) return s;
    return launch_qgemm(lc.a(), lc.container(cont), a_bits, M, K, lc.lda(), lc.desc(desc), lc.w(w_dev), lc.scales, 0, scale_w, bias, hq_alpha_for(desc), nullptr,
                        y, ydt, ldy, dev_status, st, true);
}

static hq_status gn_silu_qconv_impl(const void* x, const void* x2, int64_t split, hq_dtype xdt, int64_t Nb, int64_t H,
                                    int64_t W, int64_t C, int groups,
                                      const float* gamma, const float* beta, const void* pre_bias, int64_t pre_ld, float eps,
                                      const hq_weight_desc* desc,
                                      const void* w_dev, int R, int S, int stride, int pad, const float* scale_w,
                                      const float* bias, int a_bits, hq_scale_mode mode, const float* static_scale, void* y,
                                      hq_dtype ydt, const void* residual, void* workspace, size_t ws_bytes, void* scratch,
                                      size_t scratch_bytes, int32_t* dev_status, void* stream) {
    using namespace hq;
    if (desc == nullptr || w_dev == nullptr || workspace == nullptr || y == nullptr) return HQ_ERR_INVALID_ARG;
    if (!aligned16(workspace)) return HQ_ERR_ALIGNMENT;
    const hq_container cont = hq_container(desc->container);
    const int64_t rows = Nb * H * W;
    size_t need = 0;
    hq_status s = layer_bytes(rows, C, cont, &need);
    if (s != HQ_OK) return s;
    if (ws_bytes < need) return HQ_ERR_WORKSPACE;
    const int64_t ldc = code_pitch(C, cont);
    if (ldc != (cont == HQ_CODES_NIBBLE ? C / 2 : C)) return HQ_ERR_ALIGNMENT;   // conv needs densely packed pixels
    s = check_residual(residual, y, ydt, desc->N, desc->N);
    if (s != HQ_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    ResidualAdd res{static_cast<const __nv_bfloat16*>(residual), false};
    LayerCodes lc(desc, w_dev, a_bits, mode, rows, C, stride, cont, workspace, ws_bytes, false);
    s = launch_gn_silu_quant(x, xdt, Nb, H, W, C, groups, gamma, beta, eps, desc->had_block, a_bits, mode, static_scale,
                             lc.codes, cont, ldc, lc.scales, scratch, scratch_bytes, st, 1, pre_bias, pre_ld, x2, split, &lc.z);
    if (s != HQ_OK) return s;
    s = launch_qconv2d(lc.a(), lc.container(cont), a_bits, Nb, H, W, C, lc.desc(desc), lc.w(w_dev), R, S, stride, pad, lc.scales,
                       mode == HQ_SCALE_STATIC, scale_w, bias, hq_alpha_for(desc), nullptr, y, ydt, dev_status, st, true,
                       residual != nullptr ? &res : nullptr);
    if (s != HQ_OK) return s;                              // a stride of 0 is refused there
    const int64_t Ho = (H + 2 * pad - R) / stride + 1, Wo = (W + 2 * pad - S) / stride + 1;
    return finish_residual(s, res, y, Nb * Ho * Wo * desc->N, stream);
}

extern "C" hq_status hq_gn_silu_qconv(const void* x, hq_dtype xdt, int64_t Nb, int64_t H, int64_t W, int64_t C, int groups,
                                      const float* gamma, const float* beta, const void* pre_bias, float eps,
                                      const hq_weight_desc* desc, const void* w_dev, int R, int S, int stride, int pad,
                                      const float* scale_w, const float* bias, int a_bits, hq_scale_mode mode,
                                      const float* static_scale, void* y, hq_dtype ydt, void* workspace, size_t ws_bytes,
                                      void* scratch, size_t scratch_bytes, int32_t* dev_status, void* stream) {
    return gn_silu_qconv_impl(x, nullptr, 0, xdt, Nb, H, W, C, groups, gamma, beta, pre_bias, C, eps, desc, w_dev, R, S, stride,
                              pad, scale_w, bias, a_bits, mode, static_scale, y, ydt, nullptr, workspace, ws_bytes, scratch,
                              scratch_bytes, dev_status, stream);
}

// The same layer with a residual added to its rounded output (the second convolution of a residual block).
extern "C" hq_status hq_gn_silu_qconv_add(const void* x, hq_dtype xdt, int64_t Nb, int64_t H, int64_t W, int64_t C, int groups,
                                          const float* gamma, const float* beta, const void* pre_bias, int64_t ld_pre_bias, float eps,
                                          const hq_weight_desc* desc, const void* w_dev, int R, int S, int stride, int pad,
                                          const float* scale_w, const float* bias, int a_bits, hq_scale_mode mode,
                                          const float* static_scale, const void* residual, void* y, void* workspace,
                                          size_t ws_bytes, void* scratch, size_t scratch_bytes, int32_t* dev_status, void* stream) {
    if (residual == nullptr) return HQ_ERR_INVALID_ARG;
    return gn_silu_qconv_impl(x, nullptr, 0, xdt, Nb, H, W, C, groups, gamma, beta, pre_bias, ld_pre_bias, eps, desc, w_dev, R, S, stride,
                              pad, scale_w, bias, a_bits, mode, static_scale, y, HQ_BF16, residual, workspace, ws_bytes, scratch,
                              scratch_bytes, dev_status, stream);
}

// The same layer on the channel concatenation of two NHWC tensors (x: channels [0, C1), x2: channels [C1, C)), read in
// place: a skip connection joined to the up-sampling path without the concatenated tensor being written.
extern "C" hq_status hq_gn_silu_qconv_cat(const void* x, const void* x2, int64_t C1, hq_dtype xdt, int64_t Nb, int64_t H,
                                          int64_t W, int64_t C, int groups, const float* gamma, const float* beta,
                                          const void* pre_bias, float eps, const hq_weight_desc* desc, const void* w_dev,
                                          int R, int S, int stride, int pad, const float* scale_w, const float* bias,
                                          int a_bits, hq_scale_mode mode, const float* static_scale, void* y, hq_dtype ydt,
                                          void* workspace, size_t ws_bytes, void* scratch, size_t scratch_bytes,
                                          int32_t* dev_status, void* stream) {
    if (x2 == nullptr) return HQ_ERR_INVALID_ARG;
    return gn_silu_qconv_impl(x, x2, C1, xdt, Nb, H, W, C, groups, gamma, beta, pre_bias, C, eps, desc, w_dev, R, S, stride, pad,
                              scale_w, bias, a_bits, mode, static_scale, y, ydt, nullptr, workspace, ws_bytes, scratch, scratch_bytes,
                              dev_status, stream);
}

// The fused linear layer on the pixels of an NHWC tensor with GroupNorm (optionally + SiLU) in front: the QKV
// projection of an attention block, whose input is the normalised feature map.  Rows = Nb * rows_per_sample pixels.
extern "C" hq_status hq_gn_qlinear(const void* x, hq_dtype xdt, int64_t Nb, int64_t rows_per_sample, int64_t C, int groups,
                                   const float* gamma, const float* beta, float eps, int silu, const hq_weight_desc* desc,
                                   const void* w_dev, const float* scale_w, const float* bias, int a_bits, void* y,
                                   hq_dtype ydt, int64_t ldy, void* workspace, size_t ws_bytes, void* scratch,
                                   size_t scratch_bytes, int32_t* dev_status, void* stream) {
    using namespace hq;
    if (desc == nullptr || w_dev == nullptr || workspace == nullptr || y == nullptr) return HQ_ERR_INVALID_ARG;
    if (!aligned16(workspace)) return HQ_ERR_ALIGNMENT;
    if (Nb <= 0 || rows_per_sample <= 0) return HQ_ERR_SHAPE;
    const hq_container cont = hq_container(desc->container);
    const int64_t M = Nb * rows_per_sample;
    size_t need = 0;
    hq_status s = layer_bytes(M, C, cont, &need);
    if (s != HQ_OK) return s;
    if (ws_bytes < need) return HQ_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    LayerCodes lc(desc, w_dev, a_bits, HQ_SCALE_PER_ROW, M, C, 1, cont, workspace, ws_bytes, false);
    s = launch_gn_silu_quant(x, xdt, Nb, rows_per_sample, 1, C, groups, gamma, beta, eps, desc->had_block, a_bits,
                             HQ_SCALE_PER_ROW, nullptr, lc.codes, cont, lc.ld, lc.scales, scratch, scratch_bytes, st,
                             silu != 0, nullptr, 0, nullptr, 0, &lc.z);
    if (s != HQ_OK) return s;
    return launch_qgemm(lc.a(), lc.container(cont), a_bits, M, C, lc.lda(), lc.desc(desc), lc.w(w_dev), lc.scales, 0, scale_w, bias, hq_alpha_for(desc), nullptr,
                        y, ydt, ldy, dev_status, st, true);
}

static hq_status qconv_impl(const void* x, const void* x2, int64_t split, hq_dtype xdt, int64_t Nb, int64_t H, int64_t W,
                            int64_t C,
                              const hq_weight_desc* desc, const void* w_dev, int R, int S, int stride, int pad,
                              const float* scale_w, const float* bias, int a_bits, hq_scale_mode mode,
                              const float* static_scale, void* y, hq_dtype ydt, void* workspace, size_t ws_bytes,
                              int32_t* dev_status, void* stream) {
    using namespace hq;
    if (desc == nullptr || w_dev == nullptr || workspace == nullptr || y == nullptr) return HQ_ERR_INVALID_ARG;
    if (!aligned16(workspace)) return HQ_ERR_ALIGNMENT;
    const hq_container cont = hq_container(desc->container);
    const int64_t rows = Nb * H * W;
    size_t need = 0;
    hq_status s = layer_bytes(rows, C, cont, &need);
    if (s != HQ_OK) return s;
    if (ws_bytes < need) return HQ_ERR_WORKSPACE;
    const int64_t ldc = code_pitch(C, cont);
    if (ldc != (cont == HQ_CODES_NIBBLE ? C / 2 : C)) return HQ_ERR_ALIGNMENT;   // conv needs densely packed pixels
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    LayerCodes lc(desc, w_dev, a_bits, mode, rows, C, stride, cont, workspace, ws_bytes, false);
    if (x2 != nullptr)
        s = launch_hadamard_quant_cat(x, split, x2, C - split, split, xdt, rows, C, desc->had_block, a_bits, mode, static_scale,
                                      lc.codes, cont, ldc, lc.scales, st, &lc.z);
    else
        s = launch_hadamard_quant(x, xdt, rows, C, C, desc->had_block, a_bits, mode, static_scale, lc.codes, cont, lc.ld, lc.scales, st,
                              &lc.z);
    if (s != HQ_OK) return s;
    return launch_qconv2d(lc.a(), lc.container(cont), a_bits, Nb, H, W, C, lc.desc(desc), lc.w(w_dev), R, S, stride, pad, lc.scales,
                          mode == HQ_SCALE_STATIC, scale_w, bias, hq_alpha_for(desc), nullptr, y, ydt, dev_status, st, true);
}

extern "C" hq_status hq_qconv(const void* x, hq_dtype xdt, int64_t Nb, int64_t H, int64_t W, int64_t C,
                              const hq_weight_desc* desc, const void* w_dev, int R, int S, int stride, int pad,
                              const float* scale_w, const float* bias, int a_bits, hq_scale_mode mode,
                              const float* static_scale, void* y, hq_dtype ydt, void* workspace, size_t ws_bytes,
                              int32_t* dev_status, void* stream) {
    return qconv_impl(x, nullptr, 0, xdt, Nb, H, W, C, desc, w_dev, R, S, stride, pad, scale_w, bias, a_bits, mode,
                      static_scale, y, ydt, workspace, ws_bytes, dev_status, stream);
}

// The fused convolution layer on the channel concatenation of two NHWC tensors read in place (see hq_gn_silu_qconv_cat).
extern "C" hq_status hq_qconv_cat(const void* x, const void* x2, int64_t C1, hq_dtype xdt, int64_t Nb, int64_t H, int64_t W,
                                  int64_t C, const hq_weight_desc* desc, const void* w_dev, int R, int S, int stride,
                                  int pad, const float* scale_w, const float* bias, int a_bits, hq_scale_mode mode,
                                  const float* static_scale, void* y, hq_dtype ydt, void* workspace, size_t ws_bytes,
                                  int32_t* dev_status, void* stream) {
    if (x2 == nullptr) return HQ_ERR_INVALID_ARG;
    return qconv_impl(x, x2, C1, xdt, Nb, H, W, C, desc, w_dev, R, S, stride, pad, scale_w, bias, a_bits, mode, static_scale,
                      y, ydt, workspace, ws_bytes, dev_status, stream);
}

// Convolution exactly as Eq. 13-14 state it: transform along the width axis, quantization with one static scale,
// integer factor q * H_raw, integer convolution with untransformed (PLAIN, one-limb, INT8-container) weights.
// The int8 activations z and the scale S * 2^(-k/2) live in `workspace` (hq_workspace_size(Nb*H*W, C, INT8)).
extern "C" hq_status hq_qconv_width(const void* x, hq_dtype xdt, int64_t Nb, int64_t H, int64_t W, int64_t C,
                                    const hq_weight_desc* desc, const void* w_dev, int R, int S, int stride, int pad,
                                    const float* scale_w, const float* bias, int a_bits, int had_block_w,
                                    const float* static_scale, void* y, hq_dtype ydt, void* workspace, size_t ws_bytes,
                                    int32_t* dev_status, void* stream) {
    using namespace hq;
    if (desc == nullptr || workspace == nullptr || y == nullptr) return HQ_ERR_INVALID_ARG;
    if (desc->mode == HQ_W_PLAIN_A2) {
        // blocks wider than a signed byte allows: z travels as two int8 limbs per channel, [hi(C) | lo(C)] per pixel,
        // and meets weights whose "hi" rows are [Q(W) | 0] and "lo" rows [0 | Q(W)] in the two-limb product
        if (desc->limbs != 2 || desc->container != HQ_CODES_INT8 || desc->C != 2 * C) return HQ_ERR_SHAPE;
        if (!aligned16(workspace)) return HQ_ERR_ALIGNMENT;
        const int64_t rows2 = Nb * H * W;
        size_t need2 = 0;
        hq_status s2 = layer_bytes(rows2, 2 * C, HQ_CODES_INT8, &need2);
        if (s2 != HQ_OK) return s2;
        if (ws_bytes < need2) return HQ_ERR_WORKSPACE;
        if ((2 * C) % 16 != 0) return HQ_ERR_ALIGNMENT;
        cudaStream_t st2 = static_cast<cudaStream_t>(stream);
        unsigned char* z2 = static_cast<unsigned char*>(workspace);
        float* scale2 = reinterpret_cast<float*>(z2 + scales_offset(rows2, 2 * C, HQ_CODES_INT8));
        s2 = launch_hadamard_quant_width2(x, xdt, Nb, H, W, C, had_block_w, a_bits, static_scale, z2, scale2, st2);
        if (s2 != HQ_OK) return s2;
        return launch_qconv2d(z2, HQ_CODES_INT8, 8, Nb, H, W, 2 * C, desc, w_dev, R, S, stride, pad, scale2, 1, scale_w, bias,
                              1.0f, nullptr, y, ydt, dev_status, st2, true);
    }
    if (desc->mode != HQ_W_PLAIN || desc->limbs != 1 || desc->container != HQ_CODES_INT8) return HQ_ERR_SHAPE;
    if (!aligned16(workspace)) return HQ_ERR_ALIGNMENT;
    const int64_t rows = Nb * H * W;
    size_t need = 0;
    hq_status s = layer_bytes(rows, C, HQ_CODES_INT8, &need);
    if (s != HQ_OK) return s;
    if (ws_bytes < need) return HQ_ERR_WORKSPACE;
    if (C % 16 != 0) return HQ_ERR_ALIGNMENT;              // densely packed pixels for the convolution's TMA boxes
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    unsigned char* z = static_cast<unsigned char*>(workspace);
    float* scale = reinterpret_cast<float*>(z + scales_offset(rows, C, HQ_CODES_INT8));
    s = launch_hadamard_quant_width(x, xdt, Nb, H, W, C, had_block_w, a_bits, static_scale, z, scale, st);
    if (s != HQ_OK) return s;
    // |z| <= 128: the accumulator bound is that of 8-bit codes; the 2^(-k/2) is already inside `scale`
    return launch_qconv2d(z, HQ_CODES_INT8, 8, Nb, H, W, C, desc, w_dev, R, S, stride, pad, scale, 1, scale_w, bias, 1.0f,
                          nullptr, y, ydt, dev_status, st, true);
}

namespace hq {
namespace {
// Device address of hq_noalloc_scratch on the current device, looked up once per device.
hq_status noalloc_scratch_address(unsigned char** out) {
    static std::mutex mu;
    static unsigned char* addr[64] = {};
    int dev = 0;
    HQ_CUDA_OK(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return HQ_ERR_UNSUPPORTED;
    std::lock_guard<std::mutex> lock(mu);
    if (addr[dev] == nullptr) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, hq_noalloc_scratch) != cudaSuccess || p == nullptr) return HQ_ERR_CUDA;
        addr[dev] = static_cast<unsigned char*>(p);
    }
    *out = addr[dev];
    return HQ_OK;
}
}  // namespace
}  // namespace hq

// hq_qlinear for callers that cannot allocate: the codes and scales between the two kernels go to the library's
// own fixed device array (shared by all calls on a device, contents left over from the previous call, fully
// overwritten before they are read).  The first call per device resolves the array's address.
extern "C" hq_status hq_qlinear_noalloc(const void* x, hq_dtype xdt, int64_t M, int64_t K, int64_t ldx,
                                        const hq_weight_desc* desc, const void* w_dev, const float* scale_w,
                                        const float* bias, int a_bits, hq_scale_mode mode, const float* static_scale,
                                        void* y, hq_dtype ydt, int64_t ldy, int32_t* dev_status, void* stream) {
    using namespace hq;
    if (desc == nullptr || w_dev == nullptr || y == nullptr) return HQ_ERR_INVALID_ARG;
    const hq_container cont = hq_container(desc->container);
    size_t need = 0;
    hq_status s = layer_bytes(M, K, cont, &need);
    if (s != HQ_OK) return s;
    if (need > size_t(HQ_NOALLOC_SCRATCH_BYTES)) return HQ_ERR_SCRATCH_LIMIT;
    unsigned char* codes = nullptr;
    s = noalloc_scratch_address(&codes);
    if (s != HQ_OK) return s;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    LayerCodes lc(desc, w_dev, a_bits, mode, M, K, 1, cont, codes, HQ_NOALLOC_SCRATCH_BYTES, halved_product_covers(M, y, ydt, ldy));
    s = launch_hadamard_quant(x, xdt, M, K, ldx, desc->had_block, a_bits, mode, static_scale, lc.codes, cont, lc.ld, lc.scales, st,
                              &lc.z);
    if (s != HQ_OK) return s;
    return launch_qgemm(lc.a(), lc.container(cont), a_bits, M, lc.k(K), lc.lda(), lc.desc(desc), lc.w(w_dev), lc.scales, mode == HQ_SCALE_STATIC, scale_w, bias,
                        hq_alpha_for(desc), nullptr, y, ydt, ldy, dev_status, st, true, lc.halved());
}
