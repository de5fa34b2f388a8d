// Learned aperture surrogate on the fifth-generation tensor cores (sm_103a).
//
// The network (6 -> 128 -> 128 -> 45, ReLU) maps a proton entering the brass
// block near the opening to a transmission logit and a 4-component diagonal
// Gaussian mixture over its state on the block's exit plane.  It is not part
// of the paper.  It replaces the in-brass stepping of the aperture module
// (Sec. 2.B), which the paper reads from pre-computed brass transport data.
//
// Every layer is one 128-row tile GEMM D[128 x N] (+)= A[128 x K] B[N x K]^T:
// BF16 operands in shared memory in the canonical no-swizzle K-major layout
// (8 x 8 core matrices of 128 contiguous bytes), FP32 accumulators in tensor
// memory, issued by one thread with tcgen05.mma and completed through an
// mbarrier; the epilogues read the accumulators back with tcgen05.ld, one
// thread per row.  Training keeps the whole forward and backward of a tile in
// one CTA: the weight gradients accumulate in tensor memory over the CTA's
// tiles and the bias gradients ride along as an extra all-ones operand row.
#include <algorithm>
#include <cmath>

#include <cuda_bf16.h>

#include "device_common.cuh"
#include "vpmc_internal.cuh"

namespace vpmc {
namespace {

using namespace dev;
using namespace sur;

constexpr int kRows = 128;                // rows (tracks) per tile

// Output rows in the training kernel's order (W3P): one 16-row block per
// mixture component -- the transmission logit (component 0), its mixture
// logit, 5 means, 5 log widths, padding -- so that a component's outputs are
// 16 aligned accumulator columns.
__host__ __device__ constexpr int w3p_row(int o)
{
    if (o == 0) return 0;
    if (o < 1 + kNComp) return 16 * (o - 1) + 1;
    const int k = (o - 5) % 20, c = k / kDY, j = k % kDY;
    return 16 * c + (o < 25 ? 2 : 7) + j;
}
__host__ __device__ constexpr int w3p_output(int row)      // -1: padding
{
    const int c = row / 16, j = row % 16;
    if (j == 0) return c == 0 ? 0 : -1;
    if (j == 1) return 1 + c;
    if (j < 7) return 5 + kDY * c + (j - 2);
    return j < 12 ? 25 + kDY * c + (j - 7) : -1;
}
constexpr bool w3p_is_inverse()
{
    for (int o = 0; o < kOut; ++o)
        if (w3p_output(w3p_row(o)) != o) return false;
    return true;
}
static_assert(w3p_is_inverse(), "the training order holds every output");
constexpr int kWaitLimit = 1 << 22;       // mbarrier polls before a wait is declared failed

// What a wait returns.  A test replaces it to let one thread's wait fail
// although the work it waited for is complete.
#ifndef VPMC_WAIT_RESULT
#define VPMC_WAIT_RESULT(mbar, parity, done) (done)
#endif

// Byte offset of element (r, k) of an R x K operand in the no-swizzle
// K-major layout: core matrix (r / 8, k / 8) of 8 rows x 16 bytes.
__host__ __device__ constexpr int kmaj(int r, int k, int K)
{
    return ((((r >> 3) * (K >> 3)) + (k >> 3)) << 7) + ((r & 7) << 4) + ((k & 7) << 1);
}

// ---- tensor-core, tensor-memory and mbarrier primitives (inline PTX) ----
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: start address, leading-dimension byte
// offset (next core matrix along K), stride byte offset (next 8-row group),
// descriptor version 1, no swizzle.
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void umma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
        :: "r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void umma_commit(uint32_t mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" :: "r"(mbar)
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void mbar_init(uint32_t mbar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(mbar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// Bounded wait for the completion of the mbarrier phase with the given parity.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity)
{
    uint32_t done = 0u;
    for (int i = 0; i < kWaitLimit && !done; ++i)
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
    return VPMC_WAIT_RESULT(mbar, parity, done != 0u);
}

__device__ __forceinline__ void tmem_alloc(uint32_t slot_saddr, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(slot_saddr), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(taddr), "r"(ncols) : "memory");
}

// 16 consecutive FP32 columns of this thread's tensor-memory lane, waited for.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
        "[%16];\n\ttcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// 32 consecutive FP32 columns of this thread's tensor-memory lane, waited for.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// (a, b) + (c, d), each sum rounded as the scalar add.
__device__ __forceinline__ float2 add2(float a, float b, float c, float d)
{
    float2 r;
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 x, x, y;\n\t"
        "mov.b64 {%0, %1}, x;\n\t}"
        : "=f"(r.x), "=f"(r.y) : "f"(a), "f"(b), "f"(c), "f"(d));
    return r;
}

// relu of two BF16 values (a NaN becomes 0, as in fmaxf(x, 0)).
__device__ __forceinline__ uint32_t relu_bf16x2(uint32_t h)
{
    uint32_t r;
    asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(h), "r"(0u));
    return r;
}

// A kernel launched with programmatic serialisation starts while its
// predecessor drains; here it waits for that one's results.
__device__ __forceinline__ void wait_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_successor_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Bulk copies of bytes (a multiple of 16, both addresses 16-byte aligned):
// global to shared memory, arriving on mbar; shared to global memory.
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t mbar)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(mbar), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 :: "r"(dst), "l"(src), "r"(bytes), "r"(mbar) : "memory");
}

__device__ __forceinline__ void bulk_store(void* dst, uint32_t src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" :: "l"(dst), "r"(src), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// Until this thread's bulk stores have read their source / are complete.
__device__ __forceinline__ void bulk_store_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_store_wait() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

__device__ __forceinline__ uint32_t pack_bf16(float a, float b)
{
    __nv_bfloat162 h = __floats2bfloat162_rn(a, b);   // a in the low half (lower address)
    return *reinterpret_cast<uint32_t*>(&h);
}

__device__ __forceinline__ unsigned short bf16_bits(float a) { return __bfloat16_as_ushort(__float2bfloat16_rn(a)); }

// D[128 x N] (+)= A[128 x K] B[N x K]^T from K-major shared-memory operands.
__device__ __forceinline__ void mma_tile(uint32_t d_tmem, uint32_t a_saddr, uint32_t b_saddr, int K, int N,
                                         bool accumulate)
{
    const uint32_t idesc = idesc_bf16(kRows, N);
    const uint32_t sbo = (uint32_t)(K >> 3) << 7;
    for (int kc = 0; kc < (K >> 4); ++kc) {
        const uint64_t a = sdesc(a_saddr + (uint32_t)kc * 256u, 128u, sbo);
        const uint64_t b = sdesc(b_saddr + (uint32_t)kc * 256u, 128u, sbo);
        umma(d_tmem, a, b, idesc, (accumulate || kc > 0) ? 1u : 0u);
    }
}

// One operand of a tile GEMM in shared memory, stored as kmaj(row, column,
// columns).  K-major: rows are M or N, columns K.  MN-major (the transposed
// operand, without a transposed copy): rows are K, columns M or N; a core
// matrix then holds 8 K rows of 8 contiguous M or N values.
struct Operand {
    uint32_t saddr;
    int cols;
    bool mn_major;
};

// D[128 x N] (+)= A B^T over K, either operand K-major or MN-major.
__device__ __forceinline__ void mma_operands(uint32_t d_tmem, Operand A, Operand B, int K, int N, bool accumulate)
{
    const uint32_t idesc = idesc_bf16(kRows, N) | (A.mn_major ? 1u << 15 : 0u) | (B.mn_major ? 1u << 16 : 0u);
    const uint32_t ra = (uint32_t)(A.cols >> 3) << 7, rb = (uint32_t)(B.cols >> 3) << 7;   // 8 rows
    for (int kc = 0; kc < (K >> 4); ++kc) {
        const uint64_t a = A.mn_major ? sdesc(A.saddr + (uint32_t)kc * 2u * ra, ra, 128u)
                                      : sdesc(A.saddr + (uint32_t)kc * 256u, 128u, ra);
        const uint64_t b = B.mn_major ? sdesc(B.saddr + (uint32_t)kc * 2u * rb, rb, 128u)
                                      : sdesc(B.saddr + (uint32_t)kc * 256u, 128u, rb);
        umma(d_tmem, a, b, idesc, (accumulate || kc > 0) ? 1u : 0u);
    }
}

// Waits, as one warp, for the work committed to mbar last.  The parity moves on
// only when that work is complete: after a failed wait it still names the phase
// that is open, so that the kernel's end can wait for it once more.
__device__ __forceinline__ bool work_done(uint32_t mbar, uint32_t& parity)
{
    const bool done = __all_sync(kFull, mbar_wait(mbar, parity));
    if (done) parity ^= 1u;
    tc_fence_after();
    return done;
}

// Make this thread's generic-proxy shared-memory writes and tensor-memory
// reads visible to the next tensor-core operation, then synchronise.  Returns
// whether every thread passed ok: work is issued only when none of the waits
// before it failed, so at most one phase is ever open and nobody touches the
// operands of work in flight.
__device__ __forceinline__ bool publish(bool ok)
{
    fence_async_smem();
    tc_fence_before();
    return __syncthreads_and(ok) != 0;
}

// Barrier of one 128-thread warpgroup (named barrier 1 + g): the forward
// kernels run one tile pipeline per warpgroup, so their steps synchronise
// the group, not the CTA.
__device__ __forceinline__ void group_sync(int g)
{
    asm volatile("bar.sync %0, %1;" :: "r"(1 + g), "r"(kRows) : "memory");
}

// The same barrier, returning whether every thread of the group passed ok.
__device__ __forceinline__ bool group_sync_and(int g, bool ok)
{
    uint32_t all;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
        "bar.red.and.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(all) : "r"(ok ? 1u : 0u), "r"(1 + g), "r"(kRows) : "memory");
    return all != 0u;
}

// publish for one warpgroup's tile pipeline.
__device__ __forceinline__ bool publish_group(int g, bool ok)
{
    fence_async_smem();
    tc_fence_before();
    return group_sync_and(g, ok);
}

__device__ __forceinline__ void copy_to_smem(unsigned char* dst, const unsigned char* src, int bytes)
{
    const uint4* s = reinterpret_cast<const uint4*>(src);
    uint4* d = reinterpret_cast<uint4*>(dst);
    for (int i = threadIdx.x; i < (bytes >> 4); i += blockDim.x) d[i] = __ldg(s + i);
}

// Row r of a [128 x 16] input tile: the 6 features, then zeros.
__device__ __forceinline__ void store_input_row(unsigned char* X, int r, const float f[6])
{
    uint4 lo = make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), 0u);
    *reinterpret_cast<uint4*>(X + kmaj(r, 0, kInPad)) = lo;
    *reinterpret_cast<uint4*>(X + kmaj(r, 8, kInPad)) = make_uint4(0u, 0u, 0u, 0u);
}

// 16 consecutive FP32 columns of this thread's tensor-memory lane, issued and
// not waited for: the registers are valid after tmem_wait16 on them.
__device__ __forceinline__ void tmem_ld16_async(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
        "[%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
}

// Wait for this thread's outstanding tensor-memory loads; the registers pass
// through the wait so that no use of them moves above it.
__device__ __forceinline__ void tmem_wait16(uint32_t (&r)[16])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]),
                   "+r"(r[15])
                 :
                 : "memory");
}

// relu(D + b) of 16 columns [c0, c0 + 16) of row r, rounded to BF16 into the
// K-major [128 x 128] tile dst (bias in shared memory).  Packed adds, the
// rounding before the relu (which commutes with it): 1.5 operations and a
// quarter of a bias load per value.
__device__ __forceinline__ void relu_pack16(const uint32_t (&v)[16], const float* bias, int c0, unsigned char* dst, int r)
{
    uint32_t w[8];
#pragma unroll
    for (int j = 0; j < 16; j += 4) {
        const float4 b = *reinterpret_cast<const float4*>(bias + c0 + j);
        const float2 p = add2(__uint_as_float(v[j]), __uint_as_float(v[j + 1]), b.x, b.y);
        const float2 q = add2(__uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]), b.z, b.w);
        w[j >> 1] = relu_bf16x2(pack_bf16(p.x, p.y));
        w[(j >> 1) + 1] = relu_bf16x2(pack_bf16(q.x, q.y));
    }
    *reinterpret_cast<uint4*>(dst + kmaj(r, c0, kH)) = make_uint4(w[0], w[1], w[2], w[3]);
    *reinterpret_cast<uint4*>(dst + kmaj(r, c0 + 8, kH)) = make_uint4(w[4], w[5], w[6], w[7]);
}

// Calls f(v, c) for the ncols (a multiple of 32) FP32 columns of this
// thread's tensor-memory lane from t_row, 16 at a time: the load of the next
// 16 is in flight while f works on the current ones, so one load round trip
// is exposed per call, not one per chunk.
template <class F>
__device__ __forceinline__ void tmem_cols_pipelined(uint32_t t_row, int ncols, F&& f)
{
    uint32_t a[16], b[16];
    tmem_ld16_async(t_row, a);
    tmem_wait16(a);
#pragma unroll
    for (int c0 = 0; c0 < ncols; c0 += 32) {
        tmem_ld16_async(t_row + (uint32_t)(c0 + 16), b);
        f(a, c0);
        tmem_wait16(b);
        if (c0 + 32 < ncols) tmem_ld16_async(t_row + (uint32_t)(c0 + 32), a);
        f(b, c0 + 16);
        if (c0 + 32 < ncols) tmem_wait16(a);
    }
}

// Hidden-layer epilogue of the forward path: relu(D + b) to BF16 into the
// K-major [128 x 128] tile dst.
__device__ __forceinline__ void hidden_epilogue_fwd(uint32_t t_row, const float* bias, unsigned char* dst, int r)
{
    tmem_cols_pipelined(t_row, kH, [&](const uint32_t (&v)[16], int c0) { relu_pack16(v, bias, c0, dst, r); });
}

// z = D3 + b3 for row r (48 columns, 45 used; b3 in shared memory, padded with zeros).
__device__ __forceinline__ void output_epilogue(uint32_t t_d3, const float* b3, float (&z)[kOutPad])
{
    float v[32], u[16];
    tmem_ld32(t_d3, v);
    tmem_ld16(t_d3 + 32u, u);
#pragma unroll
    for (int j = 0; j < 32; ++j) z[j] = v[j] + b3[j];
#pragma unroll
    for (int j = 0; j < 16; ++j) z[32 + j] = u[j] + b3[32 + j];
}

// ============================================================================
// Forward: network outputs of n feature rows, and the same network drawing
// exit states for the transport's queries.
// ============================================================================
// A CTA runs kG tile pipelines, one per 128-thread warpgroup, sharing one copy
// of the weight images and biases: while one group's epilogue runs on the CUDA
// cores, another group's GEMMs run on the tensor core.  Per group: its input
// and hidden tiles, its raw inputs (and queries) and its mbarriers; in tensor
// memory, 128 columns (D1, then D2 over it once D1 is read, then D3).
//
// Forward: per 128 x 128 tile layer some 512 cycles of tensor core, 64 KB of
// tensor-memory reads and 270 issue slots of epilogue per warp, so the three
// are of one size (about 100 us each on 4.2e6 rows, whose 204 bytes a row
// take 126 us of HBM) and the time is set by how well they overlap: four
// groups, the next tile's inputs and the last one's outputs moved by bulk
// copies, and one barrier per layer: 278 us (691 TFLOP/s).  520 us with three
// groups, two barriers, scalar bias loads from global memory and copies
// through registers.
// Inference holds its queries in shared memory too: three groups fit.
template <int kG, bool kQueries>
struct FwdSmem {
    static constexpr int W = 0;                                   // W1, W2, W3 images
    static constexpr int Bias = kImgW3P;                          // b1, b2, b3 (padded), FP32
    static constexpr int G0 = (Bias + (2 * kH + kOutPad) * 4 + 127) / 128 * 128;     // the groups' regions
    // offsets within a group's region
    static constexpr int X = 0;                                   // [128 x 16]
    static constexpr int H = X + kRows * kInPad * 2;              // [128 x 128]; also the output staging
    static constexpr int XS = H + kRows * kH * 2;                 // FP32 inputs of a tile, [128 x 6]
    static constexpr int QS = XS + (kQueries ? 0 : kRows * kIn * 4);    // a tile's queries (inference)
    static constexpr int Bar = QS + (kQueries ? kRows * (int)sizeof(SurQuery) : 0);
    static constexpr int GBytes = (Bar + 16 + 127) / 128 * 128;
    static constexpr int Slot = G0 + kG * GBytes;
    static constexpr int Bytes = Slot + 8;
    static_assert(G0 % 128 == 0 && GBytes % 128 == 0, "operand tiles 128-byte aligned");
    static_assert(Bytes <= 232448, "the CTA exceeds the shared memory of one SM");
};
constexpr int kFwdGroups = 4, kInferGroups = 3;
using FwdS = FwdSmem<kFwdGroups, false>;
using InferS = FwdSmem<kInferGroups, true>;
constexpr uint32_t kFwdCols = 512;        // allocation (a power of two); group g uses columns [128 g, 128 g + 128)

// The three GEMMs of one tile whose inputs are in the group's X and published.
// On return the group's accumulator columns hold z - b3, unless ok is false in
// this warp (its wait failed) or the call returned false (the group stopped).
template <class S>
__device__ __forceinline__ bool forward_tile(unsigned char* sm, unsigned char* gs, uint32_t tcol, uint32_t t_row,
                                             uint32_t& phase, int r, int g, bool& ok)
{
    const uint32_t s0 = smem_addr(sm), gs0 = smem_addr(gs), bar = gs0 + S::Bar;
    const float* bias = reinterpret_cast<const float*>(sm + S::Bias);
    if (r == 0) {
        tc_fence_after();
        mma_tile(tcol, gs0 + S::X, s0 + S::W + kImgW1, kInPad, kH, false);
        umma_commit(bar);
    }
    ok = work_done(bar, phase);
    if (ok) hidden_epilogue_fwd(t_row, bias, gs + S::H, r);
    if (!publish_group(g, ok)) return false;
    if (r == 0) {
        tc_fence_after();
        mma_tile(tcol, gs0 + S::H, s0 + S::W + kImgW2, kH, kH, false);
        umma_commit(bar);
    }
    ok = work_done(bar, phase);
    if (ok) hidden_epilogue_fwd(t_row, bias + kH, gs + S::H, r);
    if (!publish_group(g, ok)) return false;
    if (r == 0) {
        tc_fence_after();
        mma_tile(tcol, gs0 + S::H, s0 + S::W + kImgW3, kH, kOutPad, false);
        umma_commit(bar);
    }
    ok = work_done(bar, phase);
    return true;
}

template <class S, int kG>
__device__ __forceinline__ void fwd_prologue(unsigned char* sm, const SurNet& net, uint32_t& tbase)
{
    copy_to_smem(sm + S::W, net.img, kImgW3P);
    float* bias = reinterpret_cast<float*>(sm + S::Bias);
    for (int i = threadIdx.x; i < 2 * kH + kOutPad; i += blockDim.x)
        bias[i] = i < kH ? net.params[ob1 + i]
                         : (i < 2 * kH ? net.params[ob2 + i - kH] : (i < 2 * kH + kOut ? net.params[ob3 + i - 2 * kH] : 0.0f));
    if (threadIdx.x < 2 * kG)
        mbar_init(smem_addr(sm + S::G0 + (threadIdx.x >> 1) * S::GBytes + S::Bar + 8 * (threadIdx.x & 1)));
    fence_async_smem();
    if ((threadIdx.x >> 5) == 0) tmem_alloc(smem_addr(sm + S::Slot), kFwdCols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    tbase = *reinterpret_cast<volatile uint32_t*>(sm + S::Slot);
}

template <class S>
__device__ __forceinline__ void fwd_epilogue_free(unsigned char* sm, uint32_t tbase, uint32_t bar, uint32_t phase,
                                                  bool ok, const SurNet& net)
{
    if (!ok) {
        // a wait failed in this warp: latch the error and give the tensor core
        // a last bounded chance to finish this group's work before the memory
        // is released
        atomicOr(net.status, 1);
        (void)mbar_wait(bar, phase);
    }
    tc_fence_before();
    __syncthreads();
    if ((threadIdx.x >> 5) == 0) {
        tc_fence_after();
        tmem_dealloc(tbase, kFwdCols);
    }
}

__global__ void __launch_bounds__(kFwdGroups * kRows, 1) k_sur_forward(const SurNet net, const float* __restrict__ x,
                                                                       long long n, float* __restrict__ z)
{
    using S = FwdS;
    extern __shared__ __align__(1024) unsigned char sm[];
    uint32_t tbase;
    fwd_prologue<S, kFwdGroups>(sm, net, tbase);
    const int g = threadIdx.x / kRows, r = threadIdx.x % kRows;
    unsigned char* gs = sm + S::G0 + g * S::GBytes;
    const uint32_t tcol = tbase + (uint32_t)(g * kRows);
    const uint32_t t_row = tcol + ((uint32_t)((r >> 5) * 32) << 16);
    const uint32_t bar = smem_addr(gs + S::Bar), bar_in = bar + 8u;
    uint32_t phase = 0u, phase_in = 0u;
    bool ok = true, loading = false;                // loading: a copy of inputs was started and not seen complete
    float* xs = reinterpret_cast<float*>(gs + S::XS);
    float* zs = reinterpret_cast<float*>(gs + S::H);
    const float* b3 = reinterpret_cast<const float*>(sm + S::Bias) + 2 * kH;
    const long long stride = (long long)gridDim.x * kFwdGroups;
    // a whole tile's inputs, 3 KB in a row: one bulk copy (row0 * 24 bytes is
    // a multiple of 16 when row0 is one of 128)
    auto whole = [&](long long tile) { return (tile + 1) * kRows <= n; };
    long long tile = (long long)blockIdx.x * kFwdGroups + g;
    if (whole(tile)) {
        if (r == 0) bulk_load(smem_addr(xs), x + kIn * kRows * tile, kRows * kIn * 4, bar_in);
        loading = true;
    }
    for (; tile * kRows < n; tile += stride) {
        const long long row0 = tile * kRows;
        const int rows = (int)min((long long)kRows, n - row0);
        float f[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (loading) {
            if (mbar_wait(bar_in, phase_in)) {
                phase_in ^= 1u;
                loading = false;
#pragma unroll
                for (int k = 0; k < 6; ++k) f[k] = xs[kIn * r + k];
            }
        } else if (r < rows) {
#pragma unroll
            for (int k = 0; k < 6; ++k) f[k] = __ldg(x + kIn * (row0 + r) + k);
        }
        store_input_row(gs + S::X, r, f);
        if (r == 0) bulk_store_wait_read();         // the last outputs have left the staging tile
        if (!publish_group(g, !loading)) break;
        loading = whole(tile + stride);
        if (loading && r == 0)
            bulk_load(smem_addr(xs), x + kIn * kRows * (tile + stride), kRows * kIn * 4, bar_in);
        if (!forward_tile<S>(sm, gs, tcol, t_row, phase, r, g, ok)) break;
        // outputs through shared memory (h2 is consumed): rows x 45 contiguous
        // floats (row0 * 180 bytes is a multiple of 16)
        if (ok) {
            float v[32], u[16];
            tmem_ld32(t_row, v);
            tmem_ld16(t_row + 32u, u);
#pragma unroll
            for (int j = 0; j < 32; ++j) zs[kOut * r + j] = v[j] + b3[j];
#pragma unroll
            for (int j = 32; j < kOut; ++j) zs[kOut * r + j] = u[j - 32] + b3[j];
        }
        if (!publish_group(g, ok)) break;
        if (rows == kRows) {
            if (r == 0) bulk_store(z + kOut * row0, smem_addr(zs), kRows * kOut * 4);
        } else {
            for (int i = r; i < rows * kOut; i += kRows) z[kOut * row0 + i] = zs[i];
        }
    }
    if (loading) {                                  // the group stopped: its copy ends before the memory is given back
        atomicOr(net.status, 1);
        (void)mbar_wait(bar_in, phase_in);
    }
    if (r == 0) bulk_store_wait();
    fwd_epilogue_free<S>(sm, tbase, bar, phase, ok, net);
}

// Draw of one query from the network output z (see the sampler in the oracle):
// transmitted = u0 < sigmoid(z0); component = first c with u1 < sum pi;
// y_j = mu_cj + exp(clamp(s_cj)) xi_j with xi from three Box-Muller pairs.
__device__ __forceinline__ bool sample_exit(const float (&z)[kOutPad], uint4 ua, uint4 ub, float (&y)[kDY])
{
    const float p = 1.0f / (1.0f + expf(-z[0]));
    const bool trans = u01(ua.x) < p;
    float amax = fmaxf(fmaxf(z[1], z[2]), fmaxf(z[3], z[4]));
    float e[kNComp], sum = 0.0f;
#pragma unroll
    for (int c = 0; c < kNComp; ++c) { e[c] = expf(z[1 + c] - amax); sum += e[c]; }
    const float u1 = u01(ua.y);
    int comp = kNComp - 1;
    float cum = 0.0f;
#pragma unroll
    for (int c = 0; c < kNComp; ++c) {
        cum += e[c] / sum;
        if (comp == kNComp - 1 && c < kNComp - 1 && u1 < cum) comp = c;
    }
    // the loop above takes the first c with u1 < cum_c; the last component otherwise
    const float2 x01 = box_muller(u01(ua.z), u01(ua.w));
    const float2 x23 = box_muller(u01(ub.x), u01(ub.y));
    const float2 x45 = box_muller(u01(ub.z), u01(ub.w));
    const float xi[kDY] = {x01.x, x01.y, x23.x, x23.y, x45.x};
#pragma unroll
    for (int j = 0; j < kDY; ++j) {
        float mu = 0.0f, s = 0.0f;
#pragma unroll
        for (int c = 0; c < kNComp; ++c) {
            if (c == comp) { mu = z[5 + 5 * c + j]; s = z[25 + 5 * c + j]; }
        }
        y[j] = fmaf(expf(fminf(fmaxf(s, kSMin), kSMax)), xi[j], mu);
    }
    return trans;
}

__global__ void __launch_bounds__(kInferGroups * kRows, 1) k_sur_infer(const SurNet net, const TransportParams P)
{
    using S = InferS;
    extern __shared__ __align__(1024) unsigned char sm[];
    uint32_t tbase;
    fwd_prologue<S, kInferGroups>(sm, net, tbase);
    const int g = threadIdx.x / kRows, r = threadIdx.x % kRows;
    const int lane = r & 31;
    unsigned char* gs = sm + S::G0 + g * S::GBytes;
    const uint32_t tcol = tbase + (uint32_t)(g * kRows);
    const uint32_t t_row = tcol + ((uint32_t)((r >> 5) * 32) << 16);
    const uint32_t bar = smem_addr(gs + S::Bar);
    const float* b3 = reinterpret_cast<const float*>(sm + S::Bias) + 2 * kH;
    uint32_t phase = 0u;
    bool ok = true;
    const long long nq = min((long long)*P.sq_count, P.sq_cap);
    unsigned long long acc_ap = 0ull;
    SurQuery* qs = reinterpret_cast<SurQuery*>(gs + S::QS);
    static_assert(sizeof(SurQuery) % 16 == 0, "query records are copied in 16-byte pieces");
    for (long long tile = (long long)blockIdx.x * kInferGroups + g; tile * kRows < nq;
         tile += (long long)gridDim.x * kInferGroups) {
        const long long row = tile * kRows + r;
        const int rows = (int)min((long long)kRows, nq - tile * kRows);
        // the tile's query records, contiguous: coalesced 16-byte loads
        {
            const uint4* src = reinterpret_cast<const uint4*>(P.sq + tile * kRows);
            uint4* dst = reinterpret_cast<uint4*>(qs);
            const int n16 = rows * (int)(sizeof(SurQuery) / 16);
            for (int i = r; i < n16; i += kRows) dst[i] = src[i];
        }
        group_sync(g);
        float f[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (r < rows) {
#pragma unroll
            for (int k = 0; k < 6; ++k) f[k] = qs[r].x[k];
        }
        store_input_row(gs + S::X, r, f);
        publish_group(g, true);
        if (!forward_tile<S>(sm, gs, tcol, t_row, phase, r, g, ok)) break;
        float zz[kOutPad];
        if (ok) output_epilogue(t_row, b3, zz);
        tc_fence_before();
        if (!group_sync_and(g, ok)) break;

        bool emit = false;
        PhaseRec rec;
        float pb[3] = {0.0f, 0.0f, 0.0f};       // exit point, BEV frame
        int scen0 = 0;
        const DevBeam* Bp = P.beams;
        if (row < nq) {
            const SurQuery q = qs[r];
            const DevItem& I = P.items[q.item];
            const DevBeam& B = P.beams[I.beam];
            const uint32_t hist = (uint32_t)(q.g - I.hist_off);
            const uint2 key = make_uint2(P.key0, P.key1_hi ^ (uint32_t)I.spot);
            const uint4 ua = philox(make_uint4(hist, q.step, 4u, 0u), key);
            const uint4 ub = philox(make_uint4(hist, q.step, 5u, 0u), key);
            float y[kDY];
            const bool trans = sample_exit(zz, ua, ub, y);
            if (P.track_mode) {
                if (q.g < P.total) {
                    P.trk_label[q.g] = trans ? 1 : 0;
#pragma unroll
                    for (int j = 0; j < kDY; ++j) P.trk_y[5 * q.g + j] = trans ? y[j] : 0.0f;
                }
            } else {
                const float T = B.ap_tdn - B.ap_tup;
                const float un = q.dx * q.nx + q.dy * q.ny, ut = q.dy * q.nx - q.dx * q.ny;
                const float E1 = q.E * (1.0f - 0.2f * y[0]);
                const float dn = y[1] + T * un / q.dz, dt = y[2] + T * ut / q.dz;
                float vn = fmaf(kDirScale, y[3], un), vt = fmaf(kDirScale, y[4], ut);
                const float r2 = vn * vn + vt * vt;
                if (r2 > 0.75f) {
                    const float sc = sqrtf(0.75f / r2);
                    vn *= sc;
                    vt *= sc;
                }
                if (trans && E1 > kEcut && E1 <= q.E && isfinite(dn + dt + vn + vt)) {
                    scen0 = I.scen;
                    Bp = &B;
                    pb[0] = q.px + dn * q.nx - dt * q.ny;
                    pb[1] = q.py + dn * q.ny + dt * q.nx;
                    pb[2] = B.ap_tdn;
                    const float db[3] = {vn * q.nx - vt * q.ny, vn * q.ny + vt * q.nx, sqrtf(1.0f - vn * vn - vt * vt)};
#pragma unroll
                    for (int k = 0; k < 3; ++k) rec.d[k] = db[0] * B.u[k] + db[1] * B.v[k] + db[2] * B.w[k];
                    rec.E = E1;
                    if (P.nuclear) {
                        const uint4 un6 = philox(make_uint4(hist, q.step, 6u, 0u), key);
                        rec.nlam = -logf(u01(un6.x));
                    } else {
                        rec.nlam = __int_as_float(0x7f800000);
                    }
                    rec.step = q.step + 1u;
                    rec.item = q.item;
                    rec.g = q.g;
                    emit = true;
                    acc_ap += __float2ull_rn((q.E - E1) * P.fscale) * (unsigned long long)P.n_rep;
                } else {
                    acc_ap += __float2ull_rn(q.E * P.fscale) * (unsigned long long)P.n_rep;
                    if (P.records && q.g < P.rec_cap) {
                        HistRecord hr;
                        hr.q_dep = 0;
                        hr.fate = kAbsAp;
                        hr.steps = (int)q.step;
                        hr.e_dep = 0.0f;
                        hr.e_end = 0.0f;
                        const float pe[3] = {q.px, q.py, B.ap_tup};
                        bev_to_patient(B, P.scens[I.scen], pe, hr.pos);
                        hr.pad = 0.0f;
                        P.records[q.g] = hr;
                    }
                }
            }
        }
        // hand-off into the slot the beam-line kernel reserved for this proton;
        // an absorbed proton leaves the slot empty (item -1)
        if (row < nq && !P.track_mode) {
            const long long slot = qs[r].slot;
            if (slot >= 0 && slot < P.rep_cap) {
                if (!emit) {
                    rec = PhaseRec{};
                    rec.item = -1;
                }
                // one copy per scenario sharing the beam-line transport
                const int item0 = rec.item;
                const long long g0 = rec.g;
                for (int s = 0; s < P.n_rep; ++s) {
                    if (emit) {
                        bev_to_patient(*Bp, P.scens[scen0 + s], pb, rec.p);
                        rec.item = item0 + s * P.rep_items;
                        rec.g = g0 + s * P.rep_hist;
                    }
                    P.phase[s * P.rep_cap + slot] = rec;
                }
            } else {
                atomicOr(P.status, 2);
            }
        }
        group_sync(g);                              // qs is refilled by the next tile
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) acc_ap += __shfl_xor_sync(kFull, acc_ap, o);
    if (lane == 0 && acc_ap) atomicAdd(P.stats + kStAp, acc_ap);
    fwd_epilogue_free<S>(sm, tbase, bar, phase, ok, net);
}

// ============================================================================
// Training: forward, loss, backward and weight-gradient accumulation of the
// CTA's tiles in one kernel.
// ============================================================================
// A batch of 16,384 rows is 128 tiles, one per CTA, so a launch lasts as long
// as one tile's chain of six GEMM phases, the loss between them, the operand
// load before and the gradient store after it: latency, not the tensor core
// (1 us of work).  What shortens the chain: 512 threads, four per row, each
// taking 32 columns of every epilogue and one mixture component of the loss;
// weight images by bulk copies while the inputs are read; one operand tile
// per activation, read K-major by the forward GEMMs and MN-major by the weight
// gradients and the backward ones (no transposed copies: 2-byte stores with
// 4-way bank conflicts); the b3 gradient by one butterfly per component.
// 20.7 us a launch; 40.8 us with 128 threads and transposed copies.  The Adam
// step and the next launch start while their predecessor drains (their own
// set-up runs meanwhile): 33 -> 28.6 us a training step; 29.0 with the vote on
// the waits in the barrier before each product.
constexpr int kTrainThreads = 512;
constexpr int kH1Cols = kH + 16;             // h1 and the all-ones column (b2 gradient)
struct TrainSmem {
    static constexpr int Img = 0;                                  // W1, W2, W3 images
    static constexpr int W3P = kImgW3P;                            // W3 with one 16-row block per component
    static constexpr int X = kImgBytes;                            // [128 x 16]: features, column 6 = ones (b1 gradient)
    static constexpr int H1 = X + kRows * kInPad * 2;              // [128 x 144]: h1, ones
    static constexpr int H2 = H1 + kRows * kH1Cols * 2;            // [128 x 128]: h2, then da2, then da1
    static constexpr int DZ = H2 + kRows * kH * 2;                 // [128 x 48]
    static constexpr int B1 = DZ + kRows * kOutPad * 2;            // biases (b3 in W3P's order)
    static constexpr int B2 = B1 + kH * 4;
    static constexpr int B3 = B2 + kH * 4;
    static constexpr int Alpha = B3 + kOutP * 4;                   // [128 x 4]: mixture logits of the tile
    static constexpr int Lc = Alpha + kRows * kNComp * 4;          // [128 x 4]: component log densities
    static constexpr int Db3 = Lc + kRows * kNComp * 4;            // [4 warps x 48] row sums, then [48] over the tiles
    static constexpr int Bar = Db3 + 5 * kOutPad * 4;
    static constexpr int Slot = Bar + 16;
    static constexpr int Bytes = Slot + 8;
};
static_assert(TrainSmem::Bytes <= 232448, "training tile exceeds the shared memory of one CTA");
static_assert(TrainSmem::Bar % 16 == 0 && kImgW3P % 128 == 0 && kImgBytes % 128 == 0, "alignment");
// tensor-memory columns: D1/D3/D4 at 0, D2/D5 at 128, dW2 (with db2) at 256,
// dW3^T at 400, dW1 (with db1) at 448
constexpr uint32_t kTrainCols = 512, kColW2 = 256, kColW3T = 400, kColW1 = 448;

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// relu(D + b) of this thread's 32 columns [c0, c0 + 32) of row r to BF16 into
// the tile dst of `cols` columns; returns the ReLU mask (bit j: D + b > 0).
__device__ __forceinline__ uint32_t hidden_epilogue_train(uint32_t t_row, const float* bias, unsigned char* dst, int cols,
                                                          int r, int c0)
{
    uint32_t mask = 0u;
    tmem_cols_pipelined(t_row + (uint32_t)c0, 32, [&](const uint32_t (&v)[16], int k0) {
        uint32_t w[8];
#pragma unroll
        for (int j = 0; j < 16; j += 4) {
            const float4 b = *reinterpret_cast<const float4*>(bias + c0 + k0 + j);
            const float2 p = add2(__uint_as_float(v[j]), __uint_as_float(v[j + 1]), b.x, b.y);
            const float2 q = add2(__uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]), b.z, b.w);
            mask |= (p.x > 0.0f ? 1u : 0u) << (k0 + j);
            mask |= (p.y > 0.0f ? 1u : 0u) << (k0 + j + 1);
            mask |= (q.x > 0.0f ? 1u : 0u) << (k0 + j + 2);
            mask |= (q.y > 0.0f ? 1u : 0u) << (k0 + j + 3);
            w[j >> 1] = relu_bf16x2(pack_bf16(p.x, p.y));
            w[(j >> 1) + 1] = relu_bf16x2(pack_bf16(q.x, q.y));
        }
        *reinterpret_cast<uint4*>(dst + kmaj(r, c0 + k0, cols)) = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4*>(dst + kmaj(r, c0 + k0 + 8, cols)) = make_uint4(w[4], w[5], w[6], w[7]);
    });
    return mask;
}

// D masked by the ReLU's derivative, this thread's 32 columns of row r to BF16.
__device__ __forceinline__ void masked_epilogue(uint32_t t_row, uint32_t mask, unsigned char* dst, int r, int c0)
{
    tmem_cols_pipelined(t_row + (uint32_t)c0, 32, [&](const uint32_t (&v)[16], int k0) {
        uint32_t w[8];
#pragma unroll
        for (int j = 0; j < 16; j += 2) {
            const float a0 = ((mask >> (k0 + j)) & 1u) ? __uint_as_float(v[j]) : 0.0f;
            const float a1 = ((mask >> (k0 + j + 1)) & 1u) ? __uint_as_float(v[j + 1]) : 0.0f;
            w[j >> 1] = pack_bf16(a0, a1);
        }
        *reinterpret_cast<uint4*>(dst + kmaj(r, c0 + k0, kH)) = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4*>(dst + kmaj(r, c0 + k0 + 8, kH)) = make_uint4(w[4], w[5], w[6], w[7]);
    });
}

// cols consecutive accumulator columns of this thread's row as floats at dst.
template <int kCols>
__device__ __forceinline__ void store_partial(uint32_t taddr, bool have, float* dst)
{
    uint32_t v[16];
#pragma unroll
    for (int c0 = 0; c0 < kCols; c0 += 16) {
        if (have) {
            tmem_ld16_async(taddr + (uint32_t)c0, v);
            tmem_wait16(v);
        }
#pragma unroll
        for (int j = 0; j < 16 && c0 + j < kCols; ++j) dst[c0 + j] = have ? __uint_as_float(v[j]) : 0.0f;
    }
}

__global__ void __launch_bounds__(kTrainThreads, 1) k_sur_train(const SurNet net, const float* __restrict__ x,
                                                                const float* __restrict__ yt,
                                                                const int* __restrict__ label, long long first,
                                                                long long rows, long long n, float inv_rows)
{
    using S = TrainSmem;
    extern __shared__ __align__(1024) unsigned char sm[];
    const uint32_t s0 = smem_addr(sm);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q = warp & 3, cg = warp >> 2;       // row quarter (tensor-memory lanes), column group / component
    const int r = q * 32 + lane;
    const uint32_t bar = s0 + S::Bar, bar_img = bar + 8u;
    if (threadIdx.x == 0) {
        mbar_init(bar);
        mbar_init(bar_img);
    }
    let_successor_start();
    float* b1 = reinterpret_cast<float*>(sm + S::B1);
    float* b2 = reinterpret_cast<float*>(sm + S::B2);
    float* b3 = reinterpret_cast<float*>(sm + S::B3);
    float* s_alpha = reinterpret_cast<float*>(sm + S::Alpha);
    float* s_lc = reinterpret_cast<float*>(sm + S::Lc);
    float* s_red = reinterpret_cast<float*>(sm + S::Db3);
    float* s_db3 = s_red + 4 * kOutPad;
    if (threadIdx.x < kOutPad) s_db3[threadIdx.x] = 0.0f;
    // constant operand columns: h1's ones, dz's padding
    if (cg == 0) {
        *reinterpret_cast<uint4*>(sm + S::H1 + kmaj(r, kH, kH1Cols)) = make_uint4(0x3F80u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(sm + S::H1 + kmaj(r, kH + 8, kH1Cols)) = make_uint4(0u, 0u, 0u, 0u);
    } else if (cg == 1) {
        *reinterpret_cast<uint4*>(sm + S::DZ + kmaj(r, kOutPad - 8, kOutPad)) = make_uint4(0u, 0u, 0u, 0u);
    }
    if (warp == 0) tmem_alloc(s0 + S::Slot, kTrainCols);
    // the weights of the last Adam step (and its reads of the partial
    // gradients that this launch overwrites) from here on
    wait_predecessor();
    if (threadIdx.x == 0) bulk_load(s0 + S::Img, net.img, kImgBytes, bar_img);
    if (threadIdx.x < kH) b1[threadIdx.x] = net.params[ob1 + threadIdx.x];
    else if (threadIdx.x < 2 * kH) b2[threadIdx.x - kH] = net.params[ob2 + threadIdx.x - kH];
    else if (threadIdx.x < 2 * kH + kOutP) {
        const int o = w3p_output(threadIdx.x - 2 * kH);
        b3[threadIdx.x - 2 * kH] = o >= 0 ? net.params[ob3 + o] : 0.0f;
    }
    fence_async_smem();
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = *reinterpret_cast<volatile uint32_t*>(sm + S::Slot);
    const uint32_t t_row = tbase + ((uint32_t)(q * 32) << 16);
    const int c0 = 32 * cg;
    uint32_t phase = 0u;
    const bool images = mbar_wait(bar_img, 0u);
    bool ok = true;
    int tiles_done = 0;
    double loss_acc = 0.0;
    const long long end = min(first + rows, n);
    // operands K-major (K) and MN-major (M)
    const Operand xK{s0 + S::X, kInPad, false}, h1K{s0 + S::H1, kH1Cols, false}, h2K{s0 + S::H2, kH, false},
        dzK{s0 + S::DZ, kOutPad, false};
    const Operand xM{s0 + S::X, kInPad, true}, h1M{s0 + S::H1, kH1Cols, true}, h2M{s0 + S::H2, kH, true},
        dzM{s0 + S::DZ, kOutPad, true};
    const Operand w1K{s0 + S::Img + kImgW1, kInPad, false}, w2K{s0 + S::Img + kImgW2, kH, false},
        w3pK{s0 + S::W3P, kH, false};
    const Operand w2M{s0 + S::Img + kImgW2, kH, true}, w3M{s0 + S::Img + kImgW3, kH, true};
    for (long long tile = blockIdx.x; first + tile * kRows < end; tile += gridDim.x) {
        const long long row = first + tile * kRows + r;
        const bool valid = row < end;
        // ---- inputs ----
        if (cg == 0) {
            float f[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
            if (valid) {
#pragma unroll
                for (int k = 0; k < 6; ++k) f[k] = __ldg(x + 6 * row + k);
            }
            *reinterpret_cast<uint4*>(sm + S::X + kmaj(r, 0, kInPad)) =
                make_uint4(pack_bf16(f[0], f[1]), pack_bf16(f[2], f[3]), pack_bf16(f[4], f[5]), 0x3F80u);
            *reinterpret_cast<uint4*>(sm + S::X + kmaj(r, 8, kInPad)) = make_uint4(0u, 0u, 0u, 0u);
        }
        float y[kDY] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        float t = 0.0f;
        if (valid) {
            t = __ldg(label + row) > 0 ? 1.0f : 0.0f;
#pragma unroll
            for (int j = 0; j < kDY; ++j) y[j] = __ldg(yt + 5 * row + j);
        }
        // ---- layer 1 (the CTA agrees here on the waits so far) ----
        if (!publish(ok && images)) break;
        if (threadIdx.x == 0) {
            tc_fence_after();
            mma_operands(tbase, xK, w1K, kInPad, kH, false);
            umma_commit(bar);
        }
        ok = work_done(bar, phase);
        uint32_t m1 = 0u, m2 = 0u;
        if (ok) m1 = hidden_epilogue_train(t_row, b1, sm + S::H1, kH1Cols, r, c0);
        // ---- layer 2 ----
        if (!publish(ok)) break;
        if (threadIdx.x == 0) {
            tc_fence_after();
            mma_operands(tbase + 128u, h1K, w2K, kH, kH, false);
            umma_commit(bar);
        }
        ok = work_done(bar, phase);
        if (ok) m2 = hidden_epilogue_train(t_row + 128u, b2, sm + S::H2, kH, r, c0);
        // ---- output layer: component cg's 16 columns ----
        if (!publish(ok)) break;
        if (threadIdx.x == 0) {
            tc_fence_after();
            mma_operands(tbase, h2K, w3pK, kH, kOutP, false);
            umma_commit(bar);
        }
        ok = work_done(bar, phase);
        // loss of the row and its gradient with respect to z (BCE of the
        // transmission logit plus, for transmitted tracks, the negative
        // log-likelihood of the mixture); this thread has component cg
        float zv[16] = {};
        if (ok) tmem_ld16(t_row + (uint32_t)(16 * cg), zv);
#pragma unroll
        for (int j = 0; j < 16; ++j) zv[j] += b3[16 * cg + j];
        const float alpha = zv[1];
        s_alpha[kNComp * r + cg] = alpha;
        __syncthreads();
        const float4 al = *reinterpret_cast<const float4*>(s_alpha + kNComp * r);
        const float za[kNComp] = {al.x, al.y, al.z, al.w};
        const float amax = fmaxf(fmaxf(za[0], za[1]), fmaxf(za[2], za[3]));
        float asum = 0.0f;
#pragma unroll
        for (int c = 0; c < kNComp; ++c) asum += expf(za[c] - amax);
        const float lse_a = amax + logf(asum);
        float acc = alpha - lse_a;
#pragma unroll
        for (int j = 0; j < kDY; ++j) {
            const float s = zv[7 + j];
            const float rr = (y[j] - zv[2 + j]) * expf(-s);
            acc += -0.5f * rr * rr - s - 0.91893853320467274f;
        }
        s_lc[kNComp * r + cg] = acc;
        __syncthreads();
        const float4 l4 = *reinterpret_cast<const float4*>(s_lc + kNComp * r);
        const float lc[kNComp] = {l4.x, l4.y, l4.z, l4.w};
        const float lmax = fmaxf(fmaxf(lc[0], lc[1]), fmaxf(lc[2], lc[3]));
        float lsum = 0.0f;
#pragma unroll
        for (int c = 0; c < kNComp; ++c) lsum += expf(lc[c] - lmax);
        const float L = lmax + logf(lsum);
        // gradient: 0 logit (component 0's thread), 1 mixture logit, 2.. means, 7.. log widths
        float g[12];
#pragma unroll
        for (int j = 0; j < 12; ++j) g[j] = 0.0f;
        if (valid) {
            if (cg == 0) {
                const float logit = zv[0];
                const float sig = 1.0f / (1.0f + expf(-logit));
                g[0] = sig - t;
                float loss = fmaxf(logit, 0.0f) + log1pf(expf(-fabsf(logit))) - t * logit;
                if (t > 0.0f) loss -= L;
                loss_acc += (double)loss;
            }
            if (t > 0.0f) {
                const float resp = expf(acc - L);
                const float pi = expf(alpha - lse_a);
                g[1] = pi - resp;
#pragma unroll
                for (int j = 0; j < kDY; ++j) {
                    const float s = zv[7 + j];
                    const float inv2 = expf(-2.0f * s);
                    const float diff = y[j] - zv[2 + j];
                    g[2 + j] = -resp * diff * inv2;
                    g[7 + j] = -resp * (diff * diff * inv2 - 1.0f);
                }
            }
#pragma unroll
            for (int j = 0; j < 12; ++j) g[j] *= inv_rows;
        }
        // dz [128 x 48] in the outputs' order, and b3's gradient by warp sums
        const int col[12] = {0,          1 + cg,          5 + 5 * cg,      6 + 5 * cg,      7 + 5 * cg,      8 + 5 * cg,
                             9 + 5 * cg, 25 + 5 * cg, 26 + 5 * cg, 27 + 5 * cg, 28 + 5 * cg, 29 + 5 * cg};
#pragma unroll
        for (int j = 0; j < 12; ++j) {
            if (j == 0 && cg != 0) continue;
            *reinterpret_cast<unsigned short*>(sm + S::DZ + kmaj(r, col[j], kOutPad)) = bf16_bits(g[j]);
        }
        // ---- dh2 = dz W3 and dW3^T += h2^T dz ----
        if (!publish(ok)) break;
        if (threadIdx.x == 0) {
            tc_fence_after();
            mma_operands(tbase, dzK, w3M, kOutPad, kH, false);
            mma_operands(tbase + kColW3T, h2M, dzM, kRows, kOutPad, tiles_done > 0);
            umma_commit(bar);
        }
#pragma unroll
        for (int j = 0; j < 12; ++j) {              // meanwhile: the rows' sums
            const float sum = warp_sum(g[j]);
            if (lane == 0 && (j > 0 || cg == 0)) s_red[kOutPad * q + col[j]] = sum;
        }
        ok = work_done(bar, phase);
        // ---- da2 = dh2 * relu'(a2), over h2 ----
        if (ok) masked_epilogue(t_row, m2, sm + S::H2, r, c0);
        // ---- dh1 = da2 W2 and [dW2 | db2] += da2^T [h1 | 1] ----
        if (!publish(ok)) break;
        if (threadIdx.x == 0) {
            tc_fence_after();
            mma_operands(tbase + 128u, h2K, w2M, kH, kH, false);
            mma_operands(tbase + kColW2, h2M, h1M, kRows, kH1Cols, tiles_done > 0);
            umma_commit(bar);
        }
        if (threadIdx.x < kOut) {
            double d = s_db3[threadIdx.x];          // (the order of the warps no longer shows in FP32)
#pragma unroll
            for (int k = 0; k < 4; ++k) d += s_red[kOutPad * k + threadIdx.x];
            s_db3[threadIdx.x] = (float)d;
        }
        ok = work_done(bar, phase);
        // ---- da1 = dh1 * relu'(a1), over da2 ----
        if (ok) masked_epilogue(t_row + 128u, m1, sm + S::H2, r, c0);
        // ---- [dW1 | db1] += da1^T [x | 1] ----
        if (!publish(ok)) break;
        if (threadIdx.x == 0) {
            tc_fence_after();
            mma_operands(tbase + kColW1, h2M, xM, kRows, kInPad, tiles_done > 0);
            umma_commit(bar);
        }
        ok = work_done(bar, phase);
        ++tiles_done;
    }
    // ---- loss and the accumulated weight gradients ----
    if (cg == 0) {
        const float ls = warp_sum((float)loss_acc);
        if (lane == 0 && ls != 0.0f) atomicAdd(net.loss, (double)ls);
    }
    // the CTA's partial gradient, every parameter written once (plain stores;
    // the Adam step sums the CTAs' partials: no contended atomics)
    float* part = net.gpart + (long long)blockIdx.x * kNParams;
    const bool have = __syncthreads_and(ok && images) && tiles_done > 0;
    {
        const int h = r;
        store_partial<32>(t_row + kColW2 + (uint32_t)c0, have, part + oW2 + h * kH + c0);
        if (cg == 0) store_partial<1>(t_row + kColW2 + kH, have, part + ob2 + h);
        if (cg < 3) {
            uint32_t v[16];
            if (have) {
                tmem_ld16_async(t_row + kColW3T + (uint32_t)(16 * cg), v);
                tmem_wait16(v);
            }
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (16 * cg + j < kOut) part[oW3 + (16 * cg + j) * kH + h] = have ? __uint_as_float(v[j]) : 0.0f;
        } else {
            uint32_t v[16];
            if (have) {
                tmem_ld16_async(t_row + kColW1, v);
                tmem_wait16(v);
            }
#pragma unroll
            for (int j = 0; j < kIn; ++j) part[oW1 + h * kIn + j] = have ? __uint_as_float(v[j]) : 0.0f;
            part[ob1 + h] = have ? __uint_as_float(v[kIn]) : 0.0f;
        }
        if (threadIdx.x < kOut) part[ob3 + threadIdx.x] = have ? s_db3[threadIdx.x] : 0.0f;
    }
    if (!ok || !images) {                           // a wait failed here: what it waited for ends before the CTA does
        atomicOr(net.status, 1);
        if (!ok) (void)mbar_wait(bar, phase);
        if (!images) (void)mbar_wait(bar_img, 0u);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        tmem_dealloc(tbase, kTrainCols);
    }
}

// ============================================================================
// Parameter update and BF16 operand images.
// ============================================================================
__device__ __forceinline__ void write_images(unsigned char* img, int k, float w)
{
    const unsigned short b = bf16_bits(w);
    if (k >= oW1 && k < ob1) {
        const int h = (k - oW1) / kIn, f = (k - oW1) % kIn;
        *reinterpret_cast<unsigned short*>(img + kImgW1 + kmaj(h, f, kInPad)) = b;
    } else if (k >= oW2 && k < ob2) {
        const int h = (k - oW2) / kH, i = (k - oW2) % kH;
        *reinterpret_cast<unsigned short*>(img + kImgW2 + kmaj(h, i, kH)) = b;
    } else if (k >= oW3 && k < ob3) {
        const int o = (k - oW3) / kH, h = (k - oW3) % kH;
        *reinterpret_cast<unsigned short*>(img + kImgW3 + kmaj(o, h, kH)) = b;
        *reinterpret_cast<unsigned short*>(img + kImgW3P + kmaj(w3p_row(o), h, kH)) = b;
    }
}

__global__ void k_sur_pack(const SurNet net)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < kNParams) write_images(net.img, k, net.params[k]);
}

// Sum of the parts CTAs' partial gradients of parameter k (coalesced over k),
// in the CTAs' order; 32 loads in flight.
__device__ __forceinline__ float summed_grad(const SurNet& net, int k, int parts)
{
    constexpr int kU = 32;
    float g = 0.0f;
    const float* p = net.gpart + k;
    int c = 0;
    for (; c + kU <= parts; c += kU) {
        float v[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) v[u] = p[(long long)(c + u) * kNParams];
#pragma unroll
        for (int u = 0; u < kU; ++u) g += v[u];
    }
    for (; c < parts; ++c) g += p[(long long)c * kNParams];
    return g;
}

__global__ void k_sur_reduce(const SurNet net, int parts)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k < kNParams) net.grad[k] = summed_grad(net, k, parts);
}

// Adam (Kingma & Ba 2015): moments, bias corrections c1 = 1 / (1 - beta1^t),
// c2 = 1 / (1 - beta2^t).
__global__ void k_sur_adam(const SurNet net, float lr, float c1, float c2, int parts)
{
    wait_predecessor();
    let_successor_start();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= kNParams) return;
    const float g = summed_grad(net, k, parts);
    const float m = fmaf(0.9f, net.m[k], 0.1f * g);
    const float v = fmaf(0.999f, net.v[k], 0.001f * g * g);
    net.m[k] = m;
    net.v[k] = v;
    const float w = net.params[k] - lr * (m * c1) / (sqrtf(v * c2) + 1e-8f);
    net.params[k] = w;
    write_images(net.img, k, w);
}

}  // namespace

size_t sur_forward_smem_bytes() { return std::max(FwdS::Bytes, InferS::Bytes); }
size_t sur_train_smem_bytes() { return TrainSmem::Bytes; }

cudaError_t launch_sur_pack(const SurNet& net, cudaStream_t s)
{
    k_sur_pack<<<(kNParams + 255) / 256, 256, 0, s>>>(net);
    return cudaGetLastError();
}

cudaError_t launch_sur_forward(const SurNet& net, const float* x, long long n, float* z, int grid, cudaStream_t s)
{
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_sur_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, FwdS::Bytes);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    if (n <= 0) return cudaSuccess;
    const long long tiles = (n + kRows - 1) / kRows;
    const long long ctas = (tiles + kFwdGroups - 1) / kFwdGroups;
    k_sur_forward<<<(int)std::min<long long>(ctas, grid), kFwdGroups * kRows, FwdS::Bytes, s>>>(net, x, n, z);
    return cudaGetLastError();
}

cudaError_t launch_sur_infer(const SurNet& net, const TransportParams& p, int grid, cudaStream_t s)
{
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_sur_infer, cudaFuncAttributeMaxDynamicSharedMemorySize, InferS::Bytes);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    k_sur_infer<<<grid, kInferGroups * kRows, InferS::Bytes, s>>>(net, p);
    return cudaGetLastError();
}

cudaError_t launch_sur_train(const SurNet& net, const float* x, const float* y, const int* label, long long first,
                             long long rows, long long n, float inv_rows, int grid, int* parts, cudaStream_t s)
{
    *parts = 0;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_sur_train, cudaFuncAttributeMaxDynamicSharedMemorySize, TrainSmem::Bytes);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    const long long tiles = (rows + kRows - 1) / kRows;
    if (tiles <= 0) return cudaSuccess;
    const int ctas = (int)std::min<long long>(tiles, std::min(grid, net.n_part_cap));
    *parts = ctas;
    return launch_after(k_sur_train, ctas, kTrainThreads, TrainSmem::Bytes, s, net, x, y, label, first, rows, n, inv_rows);
}

cudaError_t launch_sur_reduce(const SurNet& net, int parts, cudaStream_t s)
{
    k_sur_reduce<<<(kNParams + 255) / 256, 256, 0, s>>>(net, parts);
    return cudaGetLastError();
}

cudaError_t launch_sur_adam(const SurNet& net, int step, float lr, int parts, cudaStream_t s)
{
    const float c1 = (float)(1.0 / (1.0 - pow(0.9, step)));
    const float c2 = (float)(1.0 / (1.0 - pow(0.999, step)));
    return launch_after(k_sur_adam, (kNParams + 127) / 128, 128, 0, s, net, lr, c1, c2, parts);
}

}  // namespace vpmc
