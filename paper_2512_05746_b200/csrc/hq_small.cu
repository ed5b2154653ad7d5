// A linear layer of few rows as ONE kernel: transform, quantization, integer product and rescale (Eq. 10, Eq. 3, Eq. 12).
//
// Latency bound: the two kernels of such a layer (256 x 256 -> 256: 5.4 us on the device one after the other, two launches of
// 2.5 us each on the host) are longer than their work.  A CTA takes 16 rows and 64 output channels; its weights land in shared
// memory (`cp.async`) while K / 32 threads a row transform and quantize as the transform kernel does (the same
// building blocks in the same order, so the same codes), every column's CTA over again -- a few hundred cycles against a trip of the
// codes through memory and a launch -- and the first column's CTA leaves codes and scales in the workspace.  The product of 16 x 64 x K
// is too small for a tensor-memory accumulator to pay its set-up: `mma.sync` m16n8k32 on fragments read from shared memory
// (rows 16 bytes apart from a multiple of 128: conflict-free), both limbs in accumulators of their own.
// Launched as a programmatic dependent, and letting the next kernel in at its start: nothing is read before the wait, weights
// included, since the kernel in front may be the one that writes them.
// Two kernels / one, in a graph: 256 x 256 -> 256 5.4 / 3.2 us (a call 6.3 / 4.2), 70 x 512 -> 1024 6.5 / 5.3, 200 x 768 -> 640 6.4 / 4.7,
// 2 x 1024 -> 1024 5.9 / 5.1, 128 x 1024 -> 1024 7.3 / 5.9, 2000 x 128 -> 64 5.1 / 3.6.  With a division per 16 bytes copied instead of
// one per thread 4.2, 6.4, 5.7, 6.2, 6.9 and 4.6; with one bulk copy a channel and limb, 55 cycles each from the warp that
// issues them, 6.3, 7.4, 7.1, 7.2, 7.8 and 6.8.
#include <type_traits>

#include "hq_common.cuh"
#include "hq_fwht.cuh"

namespace hq {
extern int g_pair_gemm;
int sm_count();

namespace {

constexpr int kSmRows = 16, kSmCols = 64;

struct SmallParams {
    const void* x; int64_t M, ldx, ldy, ld_codes;
    int K, N, m, bits;
    float norm, alpha;
    const float* static_scale;
    const float* scale_w; const float* bias;
    const unsigned char* w;          // prepared weights, rows of K bytes: 128 per group of channels, or 128 "hi" and 128 "lo"
    uint8_t* codes; float* scales;
    __nv_bfloat16* y;
};

struct SmallLayout { int a_off, b_off, xch_off, total; };
__host__ __device__ inline SmallLayout small_layout(int K, int limbs, int gs_bytes_per_row) {
    SmallLayout L;
    L.a_off = 0;                                        // codes [16][K + 16]
    L.b_off = L.a_off + kSmRows * (K + 16);             // weights [64 * limbs][K + 16]
    L.xch_off = L.b_off + kSmCols * limbs * (K + 16);
    L.total = L.xch_off + kSmRows * gs_bytes_per_row;
    return L;
}
__host__ __device__ constexpr int small_xch_bytes(int m, int gs) { return m * gs * 16; }
template <int KLOG>
__host__ __device__ constexpr int small_xch_bytes(int m) { return small_xch_bytes(m, FwhtShape<KLOG, 32>::GS); }
constexpr int kSmStatic = 8 * kSmRows + 8 * kSmCols;    // the kernel's other shared arrays
// CTAs of the kernel that an SM holds at once, by its shared memory (227 KB, 1 KB of it a CTA's own) and the registers of 128 a thread
int small_resident(int K, int limbs, int block) {
    constexpr int gs[] = {FwhtShape<5, 32>::GS, FwhtShape<6, 32>::GS, FwhtShape<7, 32>::GS, FwhtShape<8, 32>::GS, FwhtShape<9, 32>::GS};
    const int smem = small_layout(K, limbs, small_xch_bytes(K / block, gs[ilog2(block) - 5])).total + kSmStatic + 1024;
    const int by_smem = 227 * 1024 / smem, by_regs = 1024 / K, most = by_smem < by_regs ? by_smem : by_regs;
    return most < 4 ? most : 4;
}

__device__ __forceinline__ void cp_async_cg_16(void* smem, const void* gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem)), "l"(gmem) : "memory");
}
__device__ __forceinline__ void mma_s8_16x8x32(int32_t (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k32.row.col.s32.s8.s8.s32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+r"(c[0]), "+r"(c[1]), "+r"(c[2]), "+r"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int KLOG, typename InT, int LIMBS, bool STATIC>
__global__ void __launch_bounds__(512) qlinear_small_kernel(const SmallParams p) {
    constexpr int E = 32, P = E / 2, N = 1 << KLOG, TB = N / E;
    using Sh = FwhtShape<KLOG, E>;
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned int rowmax[kSmRows];
    __shared__ float sScale[kSmRows], sSw[kSmCols], sBias[kSmCols];
    const int K = p.K, pitch = K + 16;
    const SmallLayout L = small_layout(K, LIMBS, small_xch_bytes<KLOG>(p.m));
    unsigned char* sA = smem + L.a_off;
    unsigned char* sB = smem + L.b_off;
    float4* xch = reinterpret_cast<float4*>(smem + L.xch_off);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n0 = blockIdx.x * kSmCols;
    const int64_t m0 = int64_t(blockIdx.y) * kSmRows;

    griddep_launch();                                  // whoever it lets in waits for this kernel before it reads anything
    if (tid < kSmRows) rowmax[tid] = 0u;
    griddep_wait();                                    // the operands, and whoever used the workspace and the output before

    const int tpr = K / E;                             // threads per row; a Hadamard block's are neighbours in one warp
    const int r = tid / tpr, tr = tid - r * tpr;
    const int blk = tr / TB, tb = tr & (TB - 1);
    const int64_t row = m0 + r;
    const bool valid = row < p.M;                      // rows past the end are zeros (nothing is read for them: 64 CTAs all reading one
                                                       // last row again cost 2 x 1024 -> 4096 2.4 us) and store nothing
    f32x2 v[P];
    float sw = 0.f, bias = 0.f, given = 0.f;           // of column tid; the static scale
    {
        const InT* src = reinterpret_cast<const InT*>(p.x) + (valid ? row : 0) * p.ldx + blk * N;
        using Raw = typename std::conditional<sizeof(InT) == 4, float4, uint2>::type;
        Raw raw[E / 4];
#pragma unroll
        for (int i = 0; i < E / 4; ++i) raw[i] = valid ? ld_dependent_cg(reinterpret_cast<const Raw*>(src + 4 * (tb + TB * i))) : Raw{};
        // The weights, behind the rows: every thread the same 16 bytes of each eighth channel.  Channel n's rows in the blob: group n / 128
        // of 128 * LIMBS rows, "hi" in front of "lo"; rows past the last group are never read.
        const int w8 = r >> 1, c = (tid - w8 * (K / 16)) * 16;       // K / 2 threads: eight channels at a time
        const unsigned char* from = p.w + (int64_t(n0 >> 7) * (128 * LIMBS) + (n0 & 127) + w8) * K + c;
#pragma unroll
        for (int i = 0; i < 8 * LIMBS; ++i) cp_async_cg_16(sB + (w8 + 8 * i) * pitch + c, from + ((i >> 3) * 128 + 8 * (i & 7)) * K);
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (tid < kSmCols) {
            const int col = n0 + tid;
            sw = col < p.N ? ld_dependent(p.scale_w + col) : 0.f;
            bias = col < p.N && p.bias != nullptr ? ld_dependent(p.bias + col) : 0.f;
        }
        if (STATIC) given = ld_dependent(p.static_scale);
#pragma unroll
        for (int i = 0; i < E / 4; ++i) {
            float4 f;
            if constexpr (sizeof(InT) == 4) f = raw[i];
            else f = make_float4(__uint_as_float(raw[i].x << 16), __uint_as_float(raw[i].x & 0xFFFF0000u),
                                 __uint_as_float(raw[i].y << 16), __uint_as_float(raw[i].y & 0xFFFF0000u));
            v[2 * i] = pk2(f.x, f.y);
            v[2 * i + 1] = pk2(f.z, f.w);
        }
    }
    fwht_stages<KLOG, E, false>(v, xch + (tid / TB) * Sh::GS, tb);
    float inv, scale;
    if (!STATIC) {
        float amax = 0.f;
#pragma unroll
        for (int e = 0; e < P; ++e) {
            float a, b;
            upk2(v[e], a, b);
            amax = max3(amax, fabsf(a), fabsf(b));
        }
#pragma unroll
        for (int off = 1; off < TB; off <<= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
        __syncthreads();                               // rowmax is cleared
        if (tb == 0) atomicMax(&rowmax[r], __float_as_uint(amax));
        __syncthreads();
        amax = __uint_as_float(rowmax[r]);
        const float qmaxf = float((1 << (p.bits - 1)) - 1);
        if (amax > 0.f) {
            scale = amax * (p.norm / qmaxf);
            inv = qmaxf / amax;
            if (!(scale > 0.f)) { scale = 1.0f; inv = p.norm; }       // scale underflowed: same rule as an all-zero row
        } else {
            scale = 1.0f;
            inv = 0.f;
        }
    } else {
        scale = given;
        inv = p.norm / scale;
    }
    {
        uint32_t w[E / 4];
        pack_codes<KLOG, E, true, STATIC>(v, inv, p.bits, tb, w);
        const int c0 = blk * N + E * tb;               // the thread's 32 codes are channels c0 ..
        const uint4 lo = make_uint4(w[0], w[1], w[2], w[3]), hi = make_uint4(w[4], w[5], w[6], w[7]);
        *reinterpret_cast<uint4*>(sA + r * pitch + c0) = lo;
        *reinterpret_cast<uint4*>(sA + r * pitch + c0 + 16) = hi;
        if (blockIdx.x == 0 && valid) {
            uint4* dst = reinterpret_cast<uint4*>(p.codes + row * p.ld_codes + c0);
            dst[0] = lo;
            dst[1] = hi;
            if (!STATIC) { if (tr == 0) p.scales[row] = scale; }
            else if (row == 0 && tr == 0) p.scales[0] = scale;
        }
        if (tr == 0) sScale[r] = scale;
        if (tid < kSmCols) { sSw[tid] = sw; sBias[tid] = bias; }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();

    // a warp takes the 8-channel tiles warp, warp + warps, ...
    const int warps = blockDim.x >> 5, g = lane >> 2, t4 = (lane & 3) * 4;
    for (int nt = warp; nt < kSmCols / 8; nt += warps) {
        int32_t acc[LIMBS][4];
#pragma unroll
        for (int l = 0; l < LIMBS; ++l)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[l][j] = 0;
        const unsigned char* ap = sA + g * pitch + t4;
        const unsigned char* bp = sB + (nt * 8 + g) * pitch + t4;
#pragma unroll 4
        for (int k = 0; k < K; k += 32) {
            const uint32_t a[4] = {*reinterpret_cast<const uint32_t*>(ap + k), *reinterpret_cast<const uint32_t*>(ap + 8 * pitch + k),
                                   *reinterpret_cast<const uint32_t*>(ap + k + 16), *reinterpret_cast<const uint32_t*>(ap + 8 * pitch + k + 16)};
#pragma unroll
            for (int l = 0; l < LIMBS; ++l) {
                const unsigned char* b = bp + l * kSmCols * pitch + k;
                mma_s8_16x8x32(acc[l], a, *reinterpret_cast<const uint32_t*>(b), *reinterpret_cast<const uint32_t*>(b + 16));
            }
        }
        const int col = n0 + nt * 8 + 2 * (lane & 3);                 // and the next one: N is even
        if (col < p.N) {
            const float sw0 = sSw[col - n0], sw1 = sSw[col - n0 + 1], b0 = sBias[col - n0], b1 = sBias[col - n0 + 1];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int rr = g + 8 * h;
                if (m0 + rr < p.M) {
                    int32_t w0 = acc[0][2 * h], w1 = acc[0][2 * h + 1];
                    if (LIMBS == 2) { w0 = w0 * 256 + acc[LIMBS - 1][2 * h]; w1 = w1 * 256 + acc[LIMBS - 1][2 * h + 1]; }
                    const float sa = p.alpha * sScale[rr];
                    const __nv_bfloat162 o = __floats2bfloat162_rn(fmaf(float(w0) * sw0, sa, b0), fmaf(float(w1) * sw1, sa, b1));
                    *reinterpret_cast<__nv_bfloat162*>(p.y + (m0 + rr) * p.ldy + col) = o;
                }
            }
        }
        __syncwarp();
    }
}

template <int KLOG, typename InT>
cudaError_t launch_small(const SmallParams& p, int limbs, cudaStream_t st) {
    const size_t smem = size_t(small_layout(p.K, limbs, small_xch_bytes<KLOG>(p.m)).total);
    const dim3 grid(unsigned((p.N + kSmCols - 1) / kSmCols), unsigned((p.M + kSmRows - 1) / kSmRows));
    auto go = [&](auto kern) -> cudaError_t {
        if (smem > 48 * 1024) {
            const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
            if (e != cudaSuccess) return e;
        }
        return launch_dependent(kern, grid, unsigned(kSmRows * p.K / 32), smem, st, true, p);
    };
    if (p.static_scale != nullptr)
        return limbs == 2 ? go(qlinear_small_kernel<KLOG, InT, 2, true>) : go(qlinear_small_kernel<KLOG, InT, 1, true>);
    return limbs == 2 ? go(qlinear_small_kernel<KLOG, InT, 2, false>) : go(qlinear_small_kernel<KLOG, InT, 1, false>);
}

template <typename InT>
cudaError_t dispatch_small(int klog, const SmallParams& p, int limbs, cudaStream_t st) {
    switch (klog) {
        case 5: return launch_small<5, InT>(p, limbs, st);
        case 6: return launch_small<6, InT>(p, limbs, st);
        case 7: return launch_small<7, InT>(p, limbs, st);
        case 8: return launch_small<8, InT>(p, limbs, st);
        case 9: return launch_small<9, InT>(p, limbs, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace

// Whether the one-kernel form takes a layer; every argument it relies on is looked at, so that what it does not take is refused (or
// run) by the two kernels as before.  One code per byte, blocks of 32 to 512 channels, reductions of whole K blocks up to 1024 (the
// weights of 64 channels and the rows' exchange buffers fill the shared memory there), an even number of bf16 output channels in
// rows of whole pairs, and no more CTAs than the SMs hold at once
// (small_resident): within one round of CTAs it was the faster of the two at every size looked at (K = 128 to 1024, both numbers of limbs,
// M = 2 to 2000, N = 64 to 4096), beyond it the slower one almost everywhere: 512 x 512 -> 512 6.5 / 5.7 us on 256 of 296 CTAs, 48 x 512 ->
// 8192 6.4 / 8.5 on 384, 512 x 768 -> 512 7.5 / 8.6 on 256 of 148.
bool small_linear_takes(const void* x, hq_dtype xdt, int64_t M, int64_t K, int64_t ldx, const hq_weight_desc* desc, const void* w_dev,
                        const float* scale_w, int a_bits, hq_scale_mode mode, const float* static_scale, const void* y, hq_dtype ydt,
                        int64_t ldy, const void* workspace, int64_t ws_used) {
    if (g_pair_gemm != 2 || x == nullptr || y == nullptr || w_dev == nullptr || scale_w == nullptr) return false;
    if ((xdt != HQ_F32 && xdt != HQ_BF16) || ydt != HQ_BF16 || M <= 0 || K < 128 || K > 1024 || K % 128 != 0) return false;
    if (mode != HQ_SCALE_PER_ROW && (mode != HQ_SCALE_STATIC || static_scale == nullptr)) return false;
    if (a_bits != 3 && a_bits != 4 && a_bits != 8) return false;
    if (desc->container != HQ_CODES_INT8 || desc->RS != 1 || desc->C != K || desc->C_pad != K || desc->mode == HQ_W_PLAIN_A2) return false;
    if ((desc->limbs != 1 && desc->limbs != 2) || desc->N <= 0 || desc->N % 2 != 0 || desc->N_pad != (desc->N + 127) / 128 * 128) return false;
    if (desc->had_block < 32 || desc->had_block > 512 || !is_pow2(desc->had_block) || K % desc->had_block != 0) return false;
    const int elt = xdt == HQ_F32 ? 4 : 2;
    if (ldx < K || ldx % 4 != 0 || reinterpret_cast<uintptr_t>(x) % (4 * elt) != 0 || !aligned16(w_dev)) return false;
    if (ldy < desc->N || ldy % 2 != 0 || reinterpret_cast<uintptr_t>(y) % 4 != 0) return false;
    if (double(K) * double(1 << (a_bits - 1)) * double(desc->max_abs_b > 0 ? desc->max_abs_b : 1) >= 2147483648.0) return false;
    // a CTA reads its rows and the static scale while others already write: the two kernels take an output on top of either and a
    // workspace on top of the input, this one not
    const auto apart = [](const void* a, int64_t an, const void* b, int64_t bn) {
        const uintptr_t i = reinterpret_cast<uintptr_t>(a), j = reinterpret_cast<uintptr_t>(b);
        return i + uintptr_t(an) <= j || j + uintptr_t(bn) <= i;
    };
    const int64_t x_bytes = ((M - 1) * ldx + K) * elt, y_bytes = ((M - 1) * ldy + desc->N) * 2;
    if (!apart(x, x_bytes, y, y_bytes) || !apart(x, x_bytes, workspace, ws_used)) return false;
    if (mode == HQ_SCALE_STATIC && !apart(static_scale, sizeof(float), y, y_bytes)) return false;
    return ((M + kSmRows - 1) / kSmRows) * ((desc->N + kSmCols - 1) / kSmCols) <= int64_t(sm_count()) * small_resident(int(K), desc->limbs, desc->had_block);
}

hq_status launch_small_linear(const void* x, hq_dtype xdt, int64_t M, int64_t K, int64_t ldx, const hq_weight_desc* desc, const void* w_dev,
                              const float* scale_w, const float* bias, int a_bits, hq_scale_mode mode, const float* static_scale,
                              float alpha, void* y, int64_t ldy, void* codes, int64_t ld_codes, float* scales, cudaStream_t st) {
    SmallParams p{};
    const int klog = ilog2(desc->had_block);
    p.x = x; p.M = M; p.ldx = ldx; p.ldy = ldy; p.ld_codes = ld_codes;
    p.K = int(K); p.N = int(desc->N); p.m = int(K / desc->had_block); p.bits = a_bits;
    p.norm = float(exp2(-0.5 * double(klog))); p.alpha = alpha;
    p.static_scale = mode == HQ_SCALE_STATIC ? static_scale : nullptr;
    p.scale_w = scale_w; p.bias = bias;
    p.w = static_cast<const unsigned char*>(w_dev);
    p.codes = static_cast<uint8_t*>(codes); p.scales = scales;
    p.y = static_cast<__nv_bfloat16*>(y);
    const cudaError_t e = xdt == HQ_F32 ? dispatch_small<float>(klog, p, desc->limbs, st) : dispatch_small<__nv_bfloat16>(klog, p, desc->limbs, st);
    return e == cudaSuccess ? HQ_OK : HQ_ERR_CUDA;
}

}  // namespace hq
