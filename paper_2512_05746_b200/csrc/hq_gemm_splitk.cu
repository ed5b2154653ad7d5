// Integer GEMM / convolution with the rescale epilogue (Eq. 12, Eq. 14) for problems of few output tiles: the reduction of
// a tile is divided over the CTAs of a cluster.
//
// A layer of few rows leaves the persistent kernels with a handful of tiles, and a tile walks its whole reduction on one SM
// (or pair): two 8 x 8 images through a 3x3 convolution over 1024 channels are 8 tiles of 72 K blocks, 27 us on 8 of the 148
// SMs.  Here S = 2, 4 or 8 CTAs of a cluster share a tile of 128 rows x 128 output channels: each runs num_kb / S K blocks
// into its own tensor memory (A and B streamed through a TMA ring; with a programmatic dependent launch the first weight
// blocks are on their way before the transform kernel has finished), then each CTA takes 128 / S of the columns: the others
// write their integer partial sums into its shared memory (the operand ring, which is free by then), and it adds them up
// and rescales.  The sums are int32, so the result does not depend on S: bit for bit that of the other kernels.
//
// What bounds it is latency: launch, the first loads, num_kb / S K blocks at about the rate one SM takes 32-48 KB from L2,
// and the exchange of up to 56 KB per CTA through the SM-to-SM network at about 20 bytes per cycle.  The exchange has no
// cluster barrier on its path (two of them cost 1300 and 2400 cycles of the first version's 9000): the last commit of each
// CTA's MMAs arrives on a barrier of every CTA of the cluster, and the partial sums are asynchronous stores that count
// their bytes on the receiver's barrier.  Every wait is bounded; a CTA whose wait ran out waits for its own loads and
// leaves with the cluster.
#include <cuda.h>

#include "hq_cluster.cuh"
#include "hq_gemm_kernel.cuh"

namespace hq {
bool encode_4d(CUtensorMap* tm, const void* base, const uint64_t dims_in[4], const uint32_t box_in[4],
               const uint32_t estr_in[4], bool swizzle128);

namespace {
using namespace gemm;

constexpr int kSkThreads = 320;                   // producer warp, MMA warp, eight epilogue warps
constexpr int kSkCols = 128;                      // output channels per tile
constexpr int kSkMaxStages = 6;
constexpr int kSkLimbBytes = 128 * kBK;           // 128 operand-B rows of a K block

struct SplitKParams {
    int64_t M, ldy;
    int N, num_kb, tiles_n, split, tile_rows;     // tile_rows: output rows per tile (128, or the pixels of one box)
    uint32_t a_bytes;                             // bytes one activation box delivers
    const float* scale_a; int sa_scalar;
    const float* scale_w; const float* bias; float alpha;
    __nv_bfloat16* y; int y_vec_ok;
    const __nv_bfloat16* res;                     // added to the rounded output (same pitch, N a multiple of 8), or nullptr
    int pdl;
    int32_t* dev_status;
    int kb_per_tap, S, stride, pad, bw, bh, bn, tiles_w, tiles_h;       // convolution geometry
};

struct SplitKCtl {
    uint64_t full[kSkMaxStages];
    uint64_t empty[kSkMaxStages];
    uint64_t ready;                               // every CTA's MMAs have completed: accumulators done, rings free
    uint64_t recv;                                // the other CTAs' partial sums of this CTA's columns have landed
    float sw[kSkCols], bias[kSkCols];             // of the columns this CTA finishes
    uint32_t tmem_base;
    volatile int abort_flag;
};

template <int LIMBS>
struct SplitKShape {
    static constexpr int kStage = kABytes + LIMBS * kSkLimbBytes;
    static constexpr int kStages = LIMBS == 2 ? 4 : 6;                  // 192 KB of ring either way
    static constexpr int kSmem = kStages * kStage + int(sizeof(SplitKCtl)) + 1024;
    static_assert(kStages * kStage >= 128 * kSkCols * 4, "the partial sums of a column share fit the ring");
};

// Polls with a short suspend-time hint: warps parked for longer on the accumulator's barrier were resumed up to 1300 cycles
// after it had completed, a fifth of the time this kernel takes.
__device__ __forceinline__ bool try_wait_64ns(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(64u)
        : "memory");
    return ok != 0;
}
// `acquire.cluster`: what the completion publishes was written from another CTA.
__device__ __forceinline__ bool try_wait_cluster(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(64u)
        : "memory");
    return ok != 0;
}
template <bool CLUSTER = false>
__device__ __forceinline__ bool wait_splitk(uint64_t* bar, uint32_t parity, SplitKCtl* ctl, int32_t* dev_status, int32_t code) {
    auto poll = [&] { return CLUSTER ? try_wait_cluster(bar, parity) : try_wait_64ns(bar, parity); };
    if (poll()) return true;
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000000LL) {
        if (poll()) return true;
        if (ctl->abort_flag) return false;
    }
    ctl->abort_flag = 1;
    if (dev_status) atomicExch(dev_status, code);
    return false;
}

template <int LIMBS, bool CONV>
__global__ void __launch_bounds__(kSkThreads, 1)
qgemm_splitk_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const SplitKParams p) {
    griddep_launch();                                  // a small transform behind this kernel may place its CTAs (dependent_launch)
    using Sh = SplitKShape<LIMBS>;
    constexpr int STAGES = Sh::kStages;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* ring = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    SplitKCtl* ctl = reinterpret_cast<SplitKCtl*>(ring + STAGES * Sh::kStage);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int S = p.split, rank = int(cluster_rank());
    const int tile = blockIdx.x / S;
    const int m_tile = tile / p.tiles_n, n_tile = tile - m_tile * p.tiles_n;
    const int cw = kSkCols / S;                                 // columns this CTA finishes
    const int64_t row0 = int64_t(m_tile) * p.tile_rows;
    const int rows = int(p.M - row0 < p.tile_rows ? p.M - row0 : p.tile_rows);     // output rows of the tile that exist
    const int k0 = rank * p.num_kb / S, count = (rank + 1) * p.num_kb / S - k0;      // at least one: the host keeps S <= num_kb

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) { mbar_init(&ctl->full[s], 1); mbar_init(&ctl->empty[s], 1); }
        mbar_init(&ctl->ready, uint32_t(p.split));
        mbar_init(&ctl->recv, 1);
        ctl->abort_flag = 0;
        fence_barrier_init();
        mbar_expect_tx(&ctl->recv, uint32_t((S - 1) * cw * rows * 4));
        tma_prefetch_desc(&tmA);
        tma_prefetch_desc(&tmB);
    }
    if (warp == 1) { __syncwarp(); tmem_alloc(&ctl->tmem_base, kSkCols * LIMBS); tmem_relinquish(); }
    tc_fence_before();
    __syncthreads();
    cluster_arrive_release();              // this CTA's barriers exist; waited for before the first access to another CTA
    tc_fence_after();
    const uint32_t tmem_base = ctl->tmem_base;

    const int ew = warp - 2, q = warp & 3, chalf = ew >> 2;     // epilogue warps: tensor-memory lane quarter, half of the columns
    float sa_eff = 0.f;                                         // of the row this thread finishes
    bool ok = true;
    int armed = 0;                                              // K blocks requested (the producing thread's)
    if (warp != 0) cluster_wait();
    if (warp == 0) {
        // ------------------------------------------------------------------ TMA producer
        if (elect_one()) {
            int w0 = 0, h0 = 0, n0 = 0;
            if (CONV) {
                w0 = (m_tile % p.tiles_w) * p.bw;
                h0 = (m_tile / p.tiles_w % p.tiles_h) * p.bh;
                n0 = m_tile / (p.tiles_w * p.tiles_h) * p.bn;
            }
            auto load_b = [&](int i) {
                const int st = i % STAGES;
                mbar_expect_tx(&ctl->full[st], p.a_bytes + uint32_t(LIMBS * kSkLimbBytes));
#pragma unroll
                for (int l = 0; l < LIMBS; ++l)
                    tma_load_2d(ring + st * Sh::kStage + kABytes + l * kSkLimbBytes, &tmB, &ctl->full[st], (k0 + i) * kBK,
                                (n_tile * LIMBS + l) * 128);
            };
            auto load_a = [&](int i) {
                const int st = i % STAGES, kb = k0 + i;
                if (CONV) {
                    const int tap = kb / p.kb_per_tap, kc = kb - tap * p.kb_per_tap;
                    const int r = tap / p.S, s = tap - r * p.S;
                    tma_load_4d(ring + st * Sh::kStage, &tmA, &ctl->full[st], kc * kBK, w0 * p.stride + s - p.pad,
                                h0 * p.stride + r - p.pad, n0);
                } else {
                    tma_load_2d(ring + st * Sh::kStage, &tmA, &ctl->full[st], kb * kBK, m_tile * 128);
                }
            };
            const int first = count < STAGES ? count : STAGES;
            for (int i = 0; i < first; ++i) load_b(i);
            if (p.pdl) griddep_wait();                 // the codes come from the kernel before this one
            for (int i = 0; i < first; ++i) load_a(i);
            armed = first;
            for (int i = first; i < count; ++i) {
                if (!wait_splitk<false>(&ctl->empty[i % STAGES], uint32_t(i / STAGES - 1) & 1u, ctl, p.dev_status, kStatusEmptyWait)) { ok = false; break; }
                load_b(i);
                load_a(i);
                ++armed;
            }
        }
        __syncwarp();
        cluster_wait();
    } else if (warp == 1) {
        // ------------------------------------------------------------------ MMA issuer
        if (elect_one()) {
            const uint32_t idesc = make_idesc_i8(kBM, kSkCols * LIMBS);
            for (int i = 0; i < count; ++i) {
                const int st = i % STAGES;
                if (!wait_splitk<false>(&ctl->full[st], uint32_t(i / STAGES) & 1u, ctl, p.dev_status, kStatusTmaWait)) { ok = false; break; }
                tc_fence_after();
                const uint64_t a_desc = make_sw128_kmajor_desc(smem_u32(ring + st * Sh::kStage));
                const uint64_t b_desc = make_sw128_kmajor_desc(smem_u32(ring + st * Sh::kStage + kABytes));
#pragma unroll
                for (int k = 0; k < kBK / 32; ++k)
                    mma_i8(tmem_base, a_desc + uint64_t(k * 2), b_desc + uint64_t(k * 2), idesc, (i | k) != 0 ? 1u : 0u);
                mma_commit(&ctl->empty[st]);
            }
            if (ok) mma_commit_to(&ctl->ready, uint16_t((1u << S) - 1u));
        }
        __syncwarp();
    } else {
        // the column parameters, and this thread's row scale, arrive while the reduction runs
        const int e = threadIdx.x - 64, col = n_tile * kSkCols + rank * cw + e;
        if (e < cw) {
            ctl->sw[e] = col < p.N ? __ldg(p.scale_w + col) : 0.f;
            ctl->bias[e] = (p.bias != nullptr && col < p.N) ? __ldg(p.bias + col) : 0.f;
        }
        if (p.pdl) griddep_wait();                     // scale_a comes from the kernel before this one
        if ((e & 127) < rows) sa_eff = p.alpha * ld_dependent(p.scale_a + (p.sa_scalar ? 0 : row0 + (e & 127)));
        // from here on every CTA's ring is its receive buffer: [from CTA][4-column group][row] of 16-byte pieces
        uint4 resid[4];                                // the residual's share, 8 columns each (cw <= 64), requested ahead; the kernel
                                                       // in front of the transform may have written it
        if (p.res != nullptr) {
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int g = (e >> 7) + 2 * i, col0 = n_tile * kSkCols + rank * cw + g * 8;
                resid[i] = g < cw / 8 && col0 < p.N && (e & 127) < rows
                               ? ld_dependent_cs(reinterpret_cast<const uint4*>(p.res + (row0 + (e & 127)) * p.ldy + col0)) : make_uint4(0u, 0u, 0u, 0u);
            }
        }
        ok = wait_splitk<true>(&ctl->ready, 0, ctl, p.dev_status, kStatusAccumWait);
        tc_fence_after();
        const int row = q * 32 + lane;
        const uint32_t t_row = tmem_base + (uint32_t(q * 32) << 16) + uint32_t(chalf * 64);
        uint32_t hi[4][16], lo[LIMBS == 2 ? 4 : 1][16];
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            tmem_ld_32x16(t_row + uint32_t(g * 16), hi[g]);
            if (LIMBS == 2) tmem_ld_32x16(t_row + uint32_t(kSkCols + g * 16), lo[LIMBS == 2 ? g : 0]);
        }
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            tmem_ld_wait_16(hi[g]);
            if (LIMBS == 2) {
                tmem_ld_wait_16(lo[LIMBS == 2 ? g : 0]);
#pragma unroll
                for (int j = 0; j < 16; ++j) hi[g][j] = hi[g][j] * 256u + lo[LIMBS == 2 ? g : 0][j];
            }
            const int col = chalf * 64 + g * 16;       // 16 columns never straddle two owners (cw >= 16)
            const int owner = col / cw, cg = (col - owner * cw) / 4;
            const int piece = (rank * (cw / 4) + cg) * 128 + row;
            if (row >= rows || !ok) {                  // nothing to hand over
            } else if (owner == rank) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    reinterpret_cast<uint4*>(ring)[piece + j * 128] = make_uint4(hi[g][4 * j], hi[g][4 * j + 1], hi[g][4 * j + 2], hi[g][4 * j + 3]);
            } else {
                const uint32_t dst = map_to_cta(ring, uint32_t(owner)) + uint32_t(piece * 16);
                const uint32_t bar = map_to_cta(&ctl->recv, uint32_t(owner));
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    st_async_v4(dst + uint32_t(j * 128 * 16), bar, hi[g][4 * j], hi[g][4 * j + 1], hi[g][4 * j + 2], hi[g][4 * j + 3]);
            }
            __syncwarp();
        }
        tc_fence_before();
        asm volatile("bar.sync 1, 256;" ::: "memory");          // this CTA's own partial sums, written by the eight warps
        ok = ok && wait_splitk<true>(&ctl->recv, 0, ctl, p.dev_status, kStatusAccumWait);
        if (ok && (e & 127) < rows) {
            const int row = e & 127;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int g = (e >> 7) + 2 * i;
                if (g >= cw / 8) break;
                const int col0 = n_tile * kSkCols + rank * cw + g * 8;
                if (col0 >= p.N) break;
                int32_t w[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll 2
                for (int s = 0; s < S; ++s) {
                    const int4* src = reinterpret_cast<const int4*>(ring) + (s * (cw / 4) + 2 * g) * 128 + row;
                    const int4 a = src[0], b = src[128];
                    w[0] += a.x; w[1] += a.y; w[2] += a.z; w[3] += a.w;
                    w[4] += b.x; w[5] += b.y; w[6] += b.z; w[7] += b.w;
                }
                float f[8];
#pragma unroll
                for (int j = 0; j < 8; ++j) f[j] = fmaf(float(w[j]) * ctl->sw[g * 8 + j], sa_eff, ctl->bias[g * 8 + j]);
                __nv_bfloat16* dst = p.y + (row0 + row) * p.ldy + col0;
                if (p.y_vec_ok && col0 + 8 <= p.N) {
                    uint4 o = make_uint4(pack_bf16x2(f[0], f[1]), pack_bf16x2(f[2], f[3]), pack_bf16x2(f[4], f[5]), pack_bf16x2(f[6], f[7]));
                    if (p.res != nullptr)
                        o = make_uint4(add_bf16x2(o.x, resid[i].x), add_bf16x2(o.y, resid[i].y), add_bf16x2(o.z, resid[i].z),
                                       add_bf16x2(o.w, resid[i].w));
                    *reinterpret_cast<uint4*>(dst) = o;
                } else {
#pragma unroll
                    for (int j = 0; j < 8; ++j) if (col0 + j < p.N) dst[j] = __float2bfloat16_rn(f[j]);
                }
            }
        }
    }
    __syncwarp();
    cluster_arrive_relaxed();
    __syncthreads();
    if (warp == 0 && elect_one() && ctl->abort_flag)            // the copies in flight must land before the ring is given up
        for (int i = armed > STAGES ? armed - STAGES : 0; i < armed; ++i)
            mbar_wait(&ctl->full[i % STAGES], uint32_t(i / STAGES) & 1u, nullptr, 0);
    if (warp == 1) { tc_fence_after(); tmem_dealloc(tmem_base, kSkCols * LIMBS); }
    cluster_wait();                        // nobody leaves while another CTA may still write or arrive here
}

template <int LIMBS, bool CONV>
cudaError_t launch_splitk(int tiles, cudaStream_t st, const CUtensorMap& tmA, const CUtensorMap& tmB, const SplitKParams& p) {
    auto kern = qgemm_splitk_kernel<LIMBS, CONV>;
    static bool attr_set[64] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SplitKShape<LIMBS>::kSmem);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(tiles * p.split)); cfg.blockDim = dim3(kSkThreads);
    cfg.dynamicSmemBytes = SplitKShape<LIMBS>::kSmem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(p.split); attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    int na = 1;
    if (p.pdl) {
        attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[1].val.programmaticStreamSerializationAllowed = 1;
        na = 2;
    }
    cfg.attrs = attr; cfg.numAttrs = unsigned(na);
    return cudaLaunchKernelEx(&cfg, kern, tmA, tmB, p);
}

}  // namespace

// How many clusters of `ways` CTAs of this kernel the device runs at once (a cluster stays inside a GPC).
static int splitk_clusters(int ways) {
    static int cached[64][4] = {};
    int dev = 0;
    const int slot = ilog2(ways);
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    if (cached[dev][slot] == 0) {
        auto kern = qgemm_splitk_kernel<2, true>;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(unsigned(sm_count() / ways * ways)); cfg.blockDim = dim3(kSkThreads);
        cfg.dynamicSmemBytes = SplitKShape<2>::kSmem;
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = unsigned(ways); attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
        cfg.attrs = attr; cfg.numAttrs = 1;
        int n = 0;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SplitKShape<2>::kSmem) != cudaSuccess ||
            cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n <= 0) {
            (void)cudaGetLastError();
            n = sm_count() / (2 * ways);               // a safe guess
        }
        cached[dev][slot] = n;
    }
    return cached[dev][slot];
}

// Estimate of a product's time on the device and the CTAs per tile it takes (0: the persistent kernels).  A tile of the
// persistent kernels (256 rows on a pair of SMs) and a CTA here both take about 0.3 us per K block (0.27 with one limb);
// the exchange costs 1 us plus up to 2 us with the share of the sums that travels, so a wider split has to gain 0.4 us.
// Measured, persistent / split, whole layer: 2 x 8 x 8 x 2048 -> 1024 3x3 47.7 / 13.9 us (8 ways), 2 x 32 x 32 x 512 3x3
// 17.1 / 14.1 (2 ways), 2 x 1024 -> 1024 7.3 / 5.7 (8 ways), 256 x 1024 -> 1024 8.0 / 8.1 (2 or 4 ways: not taken),
// 8 x 16 x 16 x 768 3x3 22.8 / 31 (2 ways, more clusters than the device holds: not taken).
ProductPlan plan_product(int limbs, int64_t out_rows, int tile_rows, int64_t n_pad, int num_kb) {
    const int64_t pairs = sm_count() / 2;
    const int64_t old_tiles = (out_rows + 255) / 256 * (limbs == 2 ? n_pad / 128 : (n_pad + 255) / 256);
    const double kb_us = limbs == 2 ? 0.30 : 0.27;
    const double weights_us = double(n_pad) * double(num_kb) * kBK * limbs / 13.0e6;    // half of it hides behind the rest
    ProductPlan best{0, 0.30 * double((old_tiles + pairs - 1) / pairs) * num_kb + weights_us};
    const int64_t tiles = (out_rows + tile_rows - 1) / tile_rows * (n_pad / kSkCols);
    const double rows = double(out_rows < tile_rows ? out_rows : tile_rows);
    for (int ways = 2; ways <= 8 && ways <= num_kb; ways *= 2) {
        if (tiles > splitk_clusters(ways)) break;
        const double us = kb_us * double((num_kb + ways - 1) / ways) + 1.0 + 2.0 * double(ways - 1) / ways * rows / 128.0 + weights_us;
        if (us < best.us - 0.4) best = ProductPlan{ways, us};
    }
    return best;
}

// CTAs per tile for a problem planned by the one-CTA path (`g`), or 0: the persistent kernels take it.
int splitk_ways(hq_container cont, const gemm::GemmParams& g, int64_t out_rows, int tile_rows, int64_t n_pad) {
    if (cont != HQ_CODES_INT8 || g.per_tap || g.acc_out != nullptr || g.y == nullptr || !g.y_bf16 || !g.combine_fast) return 0;
    return plan_product(g.limbs, out_rows, tile_rows, n_pad, g.kb_per_tap * g.taps).ways;
}

hq_status launch_qgemm_splitk(const gemm::GemmParams& g, int ways, int tile_rows, int64_t out_rows, const CUtensorMap& tmA,
                              const hq_weight_desc* desc, const void* w_dev, cudaStream_t st) {
    SplitKParams p{};
    p.M = out_rows; p.ldy = g.ldy; p.N = g.N; p.num_kb = g.kb_per_tap * g.taps;
    p.tiles_n = (g.N + kSkCols - 1) / kSkCols; p.split = ways; p.tile_rows = tile_rows;
    p.a_bytes = g.a_box_bytes;
    p.scale_a = g.scale_a; p.sa_scalar = g.sa_scalar; p.scale_w = g.scale_w; p.bias = g.bias; p.alpha = g.alpha;
    p.y = static_cast<__nv_bfloat16*>(g.y); p.y_vec_ok = g.y_vec_ok; p.res = g.res; p.pdl = g.pdl; p.dev_status = g.dev_status;
    p.kb_per_tap = g.kb_per_tap; p.S = g.S; p.stride = g.stride; p.pad = g.pad;
    p.bw = g.bw; p.bh = g.bh; p.bn = g.bn; p.tiles_w = g.tiles_w; p.tiles_h = g.tiles_h;
    CUtensorMap tmB;
    const uint64_t Kp = uint64_t(desc->C_pad) * desc->RS;
    if (!encode_2d(&tmB, w_dev, Kp, uint64_t(desc->N_pad) * desc->limbs, Kp, kBK, 128, true)) return HQ_ERR_CUDA;
    const int tiles = int((out_rows + tile_rows - 1) / tile_rows) * p.tiles_n;
    cudaError_t e;
    if (g.conv) e = g.limbs == 2 ? launch_splitk<2, true>(tiles, st, tmA, tmB, p) : launch_splitk<1, true>(tiles, st, tmA, tmB, p);
    else e = g.limbs == 2 ? launch_splitk<2, false>(tiles, st, tmA, tmB, p) : launch_splitk<1, false>(tiles, st, tmA, tmB, p);
    return e == cudaSuccess ? HQ_OK : HQ_ERR_CUDA;
}

}  // namespace hq
