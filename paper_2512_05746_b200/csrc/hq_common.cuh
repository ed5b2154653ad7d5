// Shared device/host helpers for the sm_100a kernels of the Hadamard-quantized layer forward.
#pragma once

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include "../../include/hq.h"

namespace hq {

constexpr int kQmax(int bits) { return (1 << (bits - 1)) - 1; }
constexpr int kQmin(int bits) { return -(1 << (bits - 1)); }

inline bool is_pow2(int64_t v) { return v > 0 && (v & (v - 1)) == 0; }
inline int ilog2(int64_t v) { int k = 0; while ((int64_t(1) << k) < v) ++k; return k; }
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Device status words written when a bounded wait gives up (decoded by hq_check_status).
enum : int32_t {
    kStatusTmaWait = 0x100,      // consumer waited for a TMA stage that never landed
    kStatusEmptyWait = 0x200,    // producer waited for a stage the MMA never released
    kStatusAccumWait = 0x300,    // epilogue waited for an accumulator that never completed
    kStatusAccumFree = 0x400,    // MMA issuer waited for an accumulator the epilogue never drained
    kStatusUnpackWait = 0x500,   // unpack warps / MMA issuer waited on the staging ring
};

// Where the transform kernel may leave the codes' share of the split fold (split_codes in hq_fwht.cuh) beside the codes, with the
// further columns of halved weights behind each row (`halved`) or without; `written`: it did.
constexpr int32_t kBlobHasSplit = 1;      // hq_weight_desc::reserved: the one-limb section follows the two-limb one
struct SplitOut { uint8_t* z; int64_t ld; bool written; bool halved; };
// What a product on halved weights (hq_fwht.cuh) adds to twice its sums: 1 where the parity byte of the row (every `pitch`
// bytes) and that of the output channel are both 1.
struct HalvedParity { const uint8_t* row; int64_t pitch; const uint8_t* col; };

// A bf16 tensor of the output's shape and pitch that is added to the rounded output of a product (a residual connection);
// `done`: the product kernel has added it.
struct ResidualAdd { const __nv_bfloat16* r; bool done; };

// Whether a plain transform of `grid` CTAs is launched as a programmatic dependent of whatever precedes it in the stream: its CTAs are
// placed while that kernel drains and wait (griddep_wait) before they touch anything.  Small layers one after the other: 2 x 2048 -> 1024
// 8.2 / 6.3 us a call, 2 x 8 x 8 x 2048 -> 1024 3x3 15.1 / 13.2; with 256 CTAs (2 x 32 x 32 x 512 3x3) 14.6 / 14.9, and the thousands of
// large layers cost the kernel in front its place (four transformer linears and a convolution at 32768 rows 10 % slower).  The split
// product such layers run on lets it in (griddep_launch) as it begins; in the one-CTA product that cost 2 x 48 x 48 x 768 -> 944 1x1
// stride 2 12.5 / 12.8.
int sm_count();             // hq_gemm.cu: SM count of the current device
inline bool dependent_launch(int64_t grid) { return grid <= int64_t(sm_count()) / 2; }

// hq_gemm_splitk.cu: CTAs a tile's reduction is divided over (0: persistent kernels) and the estimated time of a product.
struct ProductPlan { int ways; double us; };
ProductPlan plan_product(int limbs, int64_t out_rows, int tile_rows, int64_t n_pad, int num_kb);

#define HQ_CUDA_OK(expr) do { cudaError_t e__ = (expr); if (e__ != cudaSuccess) return HQ_ERR_CUDA; } while (0)

#ifdef __CUDACC__

template <typename... Params, typename... Args>
cudaError_t launch_dependent(void (*kern)(Params...), dim3 grid, unsigned threads, size_t smem, cudaStream_t st, bool dependent, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid; cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = dependent ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, Params(args)...);
    if (e != cudaSuccess) (void)cudaGetLastError();    // reported here: not again by the next call's look at the last error
    return e;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// bf16(y) + r for two packed pairs of values, rounded again: what an addition of the stored output gives.
__device__ __forceinline__ uint32_t add_bf16x2(uint32_t y, uint32_t r) {
    const float lo = __uint_as_float(y << 16) + __uint_as_float(r << 16);
    const float hi = __uint_as_float(y & 0xFFFF0000u) + __uint_as_float(r & 0xFFFF0000u);
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<const uint32_t*>(&h);
}

// ---- mbarrier -------------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
// One poll of a phase.  The suspend-time hint (ns) lets the hardware park the thread until the phase completes or
// the time passes, instead of returning at once: waiting warps then leave the issue slots to the working ones.
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(1000000u)
        : "memory");
    return ok != 0;
}
// Bounded wait: gives up after about a second, records `code` and returns false.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int32_t* dev_status, int32_t code) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000000LL)
        if (mbar_try_wait(bar, parity)) return true;
    if (dev_status) atomicExch(dev_status, code);
    return false;
}

// ---- fences ---------------------------------------------------------------------------------
__device__ __forceinline__ void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// ---- TMA (tiled loads, no multicast) ------------------------------------------------------------
__device__ __forceinline__ void tma_prefetch_desc(const void* tmap) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(tmap)) : "memory");
}
__device__ __forceinline__ void tma_load_2d(void* smem_dst, const void* tmap, uint64_t* bar, int x, int y) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
        ::"r"(smem_u32(smem_dst)), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(smem_u32(bar)), "r"(x), "r"(y)
        : "memory");
}
__device__ __forceinline__ void tma_load_4d(void* smem_dst, const void* tmap, uint64_t* bar, int c0, int c1, int c2,
                                            int c3) {
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
        ::"r"(smem_u32(smem_dst)), "l"(reinterpret_cast<uint64_t>(tmap)), "r"(smem_u32(bar)), "r"(c0), "r"(c1),
        "r"(c2), "r"(c3)
        : "memory");
}

// Bulk tensor store shared -> global (no mbarrier: completion is tracked per thread in bulk groups).
__device__ __forceinline__ void tma_store_2d(const void* tmap, const void* smem_src, int x, int y) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
                 ::"l"(reinterpret_cast<uint64_t>(tmap)), "r"(smem_u32(smem_src)), "r"(x), "r"(y)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit_group() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// Waits until the bulk stores committed by this thread have finished READING shared memory (not writing global).
// Programmatic dependent launch: a kernel launched with the programmatic-serialization attribute may start while the
// kernel before it in the stream is still running; griddep_wait() then blocks until that kernel has completed and its
// writes are visible (a no-op for a normally launched kernel).  griddep_launch() in the earlier kernel lets the later
// one be scheduled once every CTA has called it or exited.
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
// Loads of what a kernel before this one wrote, for use behind griddep_wait(): through the non-coherent path (__ldg) the
// compiler may move the load in front of the wait, which gave a layer the scale that the workspace held before, and the path
// itself is for data that nothing writes while the kernel runs; the intrinsics with a caching hint (__ldcs, __ldcg) promise no
// order against the wait either.  The _cs forms carry the hint of a load that nothing reads again, the _cg forms stay out of L1.
__device__ __forceinline__ float ld_dependent(const float* p) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t ld_dependent_u8(const uint8_t* p) {
    uint32_t v;
    asm volatile("ld.global.u8 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float2 ld_dependent2(const float2* p) {
    float2 v;
    asm volatile("ld.global.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
    return v;
}
#define HQ_LD_DEPENDENT(HINT)                                                                                                          \
    __device__ __forceinline__ float4 ld_dependent_##HINT(const float4* p) {                                                           \
        float4 v;                                                                                                                      \
        asm volatile("ld.global." #HINT ".v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory"); \
        return v;                                                                                                                      \
    }                                                                                                                                  \
    __device__ __forceinline__ uint2 ld_dependent_##HINT(const uint2* p) {                                                             \
        uint2 v;                                                                                                                       \
        asm volatile("ld.global." #HINT ".v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p) : "memory");                         \
        return v;                                                                                                                      \
    }                                                                                                                                  \
    __device__ __forceinline__ uint4 ld_dependent_##HINT(const uint4* p) {                                                             \
        uint4 v;                                                                                                                       \
        asm volatile("ld.global." #HINT ".v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p) : "memory"); \
        return v;                                                                                                                      \
    }
HQ_LD_DEPENDENT(cs)
HQ_LD_DEPENDENT(cg)
#undef HQ_LD_DEPENDENT
// at most one bulk store group of this thread may still be reading shared memory
__device__ __forceinline__ void bulk_wait_read_1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// ---- tcgen05: TMEM allocation, MMA, commit, loads ----------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t* smem_result, uint32_t ncols) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_result)),
                 "r"(ncols)
                 : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// D[tmem] (+)= A[smem desc] * B[smem desc], int8 x int8 -> int32.
__device__ __forceinline__ void mma_i8(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::i8 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
// Arrive on an mbarrier once all previously issued MMAs of this thread have completed.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}
// 32 lanes x 32 consecutive 32-bit columns -> 32 registers per thread (thread i = lane i of the warp's quarter).
__device__ __forceinline__ void tmem_ld_32x32(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
// 32 lanes x 16 consecutive 32-bit columns -> 16 registers per thread.
__device__ __forceinline__ void tmem_ld_32x16(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
// 16 lanes x 32 consecutive 32-bit columns in the 16x256b fragment layout -> 16 registers per thread: for repeat n = 0..3
// (8 columns each) thread t holds r[4n], r[4n+1] = lane t/4, columns 8n + 2(t%4), +1 and r[4n+2], r[4n+3] = lane t/4 + 8,
// same columns (the layout of an m16n8 accumulator fragment).  `taddr` names the first of the 16 lanes.
__device__ __forceinline__ void tmem_ld_16x256_x4(uint32_t taddr, uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}
// tcgen05.wait::ld that also names the loaded registers, so that no use of them can be scheduled ahead of it.
__device__ __forceinline__ void tmem_ld_wait_16(uint32_t (&r)[16]) {
    asm volatile(
        "tcgen05.wait::ld.sync.aligned;"
        : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
          "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
        :
        : "memory");
}

__device__ __forceinline__ void tmem_ld_wait_32(uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.wait::ld.sync.aligned;"
        : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]),
          "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]),
          "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]),
          "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])
        :
        : "memory");
}

// Shared-memory matrix descriptor for a K-major operand tile stored as rows of 128 bytes with the
// 128-byte swizzle (what a TMA load with CU_TENSOR_MAP_SWIZZLE_128B writes): 8-row groups are 1024 bytes apart.
__device__ __forceinline__ uint64_t make_sw128_kmajor_desc(uint32_t smem_addr) {
    uint64_t d = 0;
    d |= uint64_t((smem_addr & 0x3FFFFu) >> 4);        // start address, 16-byte units
    d |= uint64_t(1) << 16;                            // leading-dimension byte offset (unused with swizzle): 1
    d |= uint64_t(1024 >> 4) << 32;                    // stride between 8-row groups
    d |= uint64_t(1) << 46;                            // descriptor version of this architecture
    d |= uint64_t(2) << 61;                            // 128-byte swizzle
    return d;
}

// Instruction descriptor for kind::i8, signed x signed -> int32, both operands K-major, tile M x N.
__host__ __device__ constexpr uint32_t make_idesc_i8(int M, int N) {
    return (2u << 4)                 // D format: S32
           | (1u << 7)               // A format: signed 8-bit
           | (1u << 10)              // B format: signed 8-bit
           | (uint32_t(N >> 3) << 17)
           | (uint32_t(M >> 4) << 24);
}

// One lane of a converged warp, the same at every call.  Unlike a comparison of the lane number it tells the compiler that what
// follows runs on one lane: the operands of tensor-core and copy instructions stay in uniform registers.  Issuing warps of the
// split and streamed paired products and of the attention core (2 x 8 x 8 x 2048 -> 1024 3x3 13.1 -> 12.0 us, 64 x 64 x 64 x 256 3x3
// 151 -> 148, 16001 x 1024 -> 1288 with 8-bit codes 39.65 -> 39.1); level or slower in the one-CTA kernel (256 x 256 -> 256 6.2 / 6.4 us,
// 32768 x 256 -> 1024 25-28 / 31-33) and in the resident paired one (32768 x 512 -> 1536 59.9 / 60.3).
__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(pred));
    return pred != 0;
}

#endif  // __CUDACC__

}  // namespace hq
