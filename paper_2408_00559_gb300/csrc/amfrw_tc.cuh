// BF16 tensor-core GEMM on the 5th-generation tensor cores (tcgen05, sm_103a)
// for the surrogate network's dense layers.
//
//   C[M x N] = A[M x K] * B[N x K]^T        (both operands K-major, BF16;
//                                             FP32 accumulation in TMEM)
//
// One CTA of 256 threads computes a 128 x BN tile (BN <= 256, a multiple of
// 16).  K advances in chunks of 64 through a ring of up to eight shared-memory
// stages filled by TMA: one box of 64 elements of K (128 bytes, the 128-byte
// swizzle's span) by all rows per operand, in the swizzled K-major layout
// (8 rows x 128 bytes per swizzle atom, atoms 1024 bytes apart along M/N).
// (Boxes of 16 bytes a row, the unswizzled layout's, cost the TMA unit eight
// times the requests: 3 072 a chunk, which bound every product here.)  One
// elected thread issues the loads of every stage up front, then for each chunk
// waits for its stage's "full" mbarrier (the TMA transaction count), issues
// four tcgen05.mma (K = 16 each, 32 bytes further inside the atom) and commits
// them to the stage's "empty" mbarrier; the stage of the previous chunk is
// refilled with the chunk S ahead as soon as that commit completes, while the
// current chunk's MMAs run.  A final commit releases the epilogue: every warp
// reads its 32 TMEM lanes (rows; two warps share a quadrant and take its
// columns in turn, so that the GELU's arithmetic, which bounds the layers, has
// 16 warps per SM) with tcgen05.ld, applies a fused elementwise operation and
// passes 32 columns at a time through its part of the stages'
// memory, so that global accesses are whole 128-byte lines (64 bytes for the
// BF16 outputs) instead of a sector per row.  Every mbarrier wait is bounded:
// on timeout the kernel records an error, waits (bounded) once more for the
// loads and MMAs it issued, skips the rest and frees its TMEM.
// Measured (kernel alone): 65536 x 256 x 256 to FP32 60 -> 22 us (15 us at the copy rate); the training
// products 1024 x 256 x 256 36 -> 8 us, 256 x 256 x 1024 42 -> 13 us.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace amfrw {
namespace tc {

constexpr int kBM = 128;
constexpr int kBK = 64;
constexpr int kThreads = 256;
constexpr uint32_t kSpinLimit = 1u << 26;  // bounded mbarrier waits

__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

// Shared-memory matrix descriptor (tcgen05) of a K-major tile in the 128-byte
// swizzle: start address, 1024 bytes between groups of 8 rows (stride byte
// offset; the leading one is not used by this layout), descriptor version 1,
// layout type 2.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr >> 4) & 0x3FFFu);
    d |= (uint64_t)1 << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;  // version
    d |= (uint64_t)2 << 61;  // 128-byte swizzle
    return d;
}

// Instruction descriptor of tcgen05.mma.kind::f16: FP32 accumulator, BF16 A
// and B, both K-major, N >> 3 and M >> 4.
__host__ __device__ constexpr uint32_t instr_desc_bf16(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint32_t addr, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(addr), "r"(count) : "memory");
}

// Wait for the phase with the given parity; false if the bound was hit.
__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity)
{
    for (uint32_t it = 0; it < kSpinLimit; ++it) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred P1;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 P1, [%1], %2;\n\t"
            "selp.b32 %0, 1, 0, P1;\n\t}\n"
            : "=r"(done)
            : "r"(addr), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void tmem_alloc(uint32_t dst_smem, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(dst_smem),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
                 : "memory");
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc,
                                         uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(mbar)
                 : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// 32 consecutive FP32 columns of this thread's TMEM lane (one wait for all).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
        "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 8 consecutive FP32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8])
{
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                   "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// Shared memory of one CTA: S stages of A (128 rows) and B (BN rows) x 64
// elements of K, which the epilogue's buffers reuse, then, behind both, the
// mbarriers (full and empty per stage, done) and the TMEM address.  A stage's
// operand is one box of rows x 128 bytes.  (1 KB more than needed, to start on
// a 1024-byte boundary.)
constexpr int kMaxStages = 8;
constexpr int kTurnBytes = 32 * 144;  // a warp's buffer in the epilogue
constexpr int kTileA = kBM * kBK * 2;
__host__ __device__ constexpr int stage_bytes(int BN) { return kTileA + BN * kBK * 2; }
__host__ __device__ constexpr int bars_offset(int BN, int stages)
{
    const int st = stages * stage_bytes(BN), turn = kThreads / 32 * kTurnBytes;
    return st > turn ? st : turn;
}
__host__ __device__ constexpr int smem_bytes(int BN, int stages) { return 1024 + bars_offset(BN, stages) + 8 * (2 * kMaxStages + 1) + 16; }

__device__ __forceinline__ void mbar_expect_tx(uint32_t addr, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(addr), "r"(bytes) : "memory");
}

// One 2-D TMA box (x = element along K, y = row) into shared memory,
// completing on the mbarrier with its byte count.
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, int x, int y, uint32_t mbar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
            "r"(dst), "l"(reinterpret_cast<uint64_t>(tm)), "r"(x), "r"(y), "r"(mbar)
        : "memory");
}

struct Epi {
    int mode;             // 0: C = acc (FP32); 1: Z = acc + bias, H = gelu(Z) (BF16), Ht
                          // 2: D = acc * gelu'(Zprev) -> BF16 D and Dt
                          // 3: y = sum over the 256 columns of w4 * bf16(gelu(acc + bias)), + b4
    float* C;             // mode 0: [M x N] FP32, row stride ldc
    int ldc;
    const float* bias;    // mode 1: [N]
    float* Z;             // mode 1: [M x N] FP32 pre-activation (row stride N), may be null
    __nv_bfloat16* H;     // mode 1/2: [M x N] BF16 (row stride N)
    __nv_bfloat16* Ht;    // mode 1/2: [N x M] BF16 transpose (row stride ldt), may be null
    int ldt;
    const float* Zprev;   // mode 2: [M x N] FP32 pre-activation of this layer
    const float* w4;      // mode 3: [N] (N = BN = 256), then the output's bias b4
    float* y;             // mode 3: [M]
    int* error;           // set when a bounded wait gave up
};

__device__ __forceinline__ float gelu(float z)
{
    return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f));
}

__device__ __forceinline__ float gelu_grad(float z)
{
    const float cdf = 0.5f * (1.0f + erff(z * 0.70710678118654752f));
    const float pdf = 0.3989422804014327f * __expf(-0.5f * z * z);
    return cdf + z * pdf;
}

// C-tile = A[m0:m0+128, :] * B[n0:n0+BN, :]^T on one block.
__device__ __forceinline__ void gemm_tile(const CUtensorMap& tmA, const CUtensorMap& tmB, int m0, int n0, int M, int N,
                                          int K, int BN, int S, const Epi& epi)
{
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const int SB = stage_bytes(BN);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + bars_offset(BN, S));  // full[kMaxStages], empty[kMaxStages], done
    uint32_t* taddr_slot = reinterpret_cast<uint32_t*>(bars + 2 * kMaxStages + 1);
    __shared__ int s_fail;
    const int tid = threadIdx.x;
    const int warp = tid >> 5;
    const uint32_t ncols = BN <= 32 ? 32u : (BN <= 64 ? 64u : (BN <= 128 ? 128u : 256u));
    auto full = [&](int st) { return smem_u32(bars + st); };
    auto empty = [&](int st) { return smem_u32(bars + kMaxStages + st); };
    const uint32_t done = smem_u32(bars + 2 * kMaxStages);

    if (warp == 0) tmem_alloc(smem_u32(taddr_slot), ncols);
    if (tid == 0) {
        s_fail = 0;
        for (int st = 0; st < S; ++st) {
            mbar_init(full(st), 1);
            mbar_init(empty(st), 1);
        }
        mbar_init(done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *taddr_slot;
    const int nk = (K + kBK - 1) / kBK;

    if (tid == 0) {
        const uint32_t idesc = instr_desc_bf16(kBM, BN);
        const uint32_t tx = (uint32_t)SB;
        int issued = 0, waited = 0;  // chunks: loads issued, loads waited for
        auto load = [&](int i, int st) {
            const uint32_t a = smem_u32(smem + st * SB), b = a + kTileA;
            mbar_expect_tx(full(st), tx);
            tma_load_2d(a, &tmA, i * kBK, m0, full(st));
            tma_load_2d(b, &tmB, i * kBK, n0, full(st));
            issued = i + 1;
        };
        for (int i = 0; i < S && i < nk; ++i) load(i, i);
        bool ok = true;
        for (int i = 0; i < nk && ok; ++i) {
            const int st = i % S;
            const uint32_t ph = (uint32_t)((i / S) & 1);
            ok = mbar_wait(full(st), ph);
            if (!ok) break;
            waited = i + 1;
            fence_after();
            const int kc = (K - i * kBK) < kBK ? (K - i * kBK) : kBK;  // multiple of 16
            const uint32_t a = smem_u32(smem + st * SB), b = a + kTileA;
            for (int kk = 0; kk < kc / 16; ++kk) {
                mma_bf16(tmem, smem_desc(a + kk * 32), smem_desc(b + kk * 32), idesc, (i > 0 || kk > 0) ? 1u : 0u);
            }
            if (i + S < nk) mma_commit(empty(st));  // (only what a refill waits for)
            // refill the previous chunk's stage once its MMAs are done (the
            // current chunk's MMAs keep the tensor pipe busy meanwhile)
            const int prev = i - 1, next = prev + S;
            if (prev >= 0 && next < nk) {
                const int ps = prev % S;
                ok = mbar_wait(empty(ps), (uint32_t)((prev / S) & 1));
                if (ok) load(next, ps);
            }
        }
        // the last commit covers every MMA issued above
        mma_commit(done);
        if (!ok) {
            // wait (bounded) for the loads still in flight, so that none lands
            // in shared memory after the block has gone
            for (int c = waited; c < issued; ++c) mbar_wait(full(c % S), (uint32_t)((c / S) & 1));
            s_fail = 1;
        }
    }
    // every thread waits for the last commit; the block agrees on the outcome
    const bool fin = __syncthreads_and(mbar_wait(done, 0) ? 1 : 0) != 0;
    const bool ok = fin && s_fail == 0;
    fence_after();
    if (!ok) {
        if (!fin) __syncthreads_and(mbar_wait(done, 0) ? 1 : 0);  // once more before TMEM is freed
        if (tid == 0) atomicExch(epi.error, 1);
    } else {
        // epilogue: lane = row m0 + 32 warp + lane, 32 columns at a time.  The
        // stages are free now (their loads and MMAs are done; the mbarriers,
        // where an arrive may still land, lie behind them): each warp
        // turns its 32 x 32 values there, rows 144 bytes apart (FP32) or 80
        // (BF16), so that both the row-wise and the line-wise 16-byte
        // accesses are free of bank conflicts.
        const int lane = tid & 31, quad = warp & 3, half = warp >> 2, r0 = m0 + quad * 32, row = r0 + lane;
        unsigned char* tr = smem + warp * kTurnBytes;
        const uint32_t tq = tmem + ((uint32_t)(quad * 32) << 16);
        const bool vec_c = (epi.ldc & 3) == 0 && ((uintptr_t)epi.C & 15) == 0;
        auto put_f32 = [&](const float (&v)[32]) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
                *reinterpret_cast<float4*>(tr + lane * 144 + i * 16) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            __syncwarp();
        };
        // 32 (or 16) columns of FP32 from the warp's buffer to rows of `dst`
        auto store_f32 = [&](float* dst, int ld, int col0, int nc) {
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const int rr = i * 4 + (lane >> 3), c = (lane & 7) * 4;
                if (r0 + rr < M && c < nc)
                    *reinterpret_cast<float4*>(dst + (size_t)(r0 + rr) * ld + col0 + c) =
                        *reinterpret_cast<const float4*>(tr + rr * 144 + c * 4);
            }
            __syncwarp();
        };
        if (epi.mode == 3) {
            // The output layer on the spot: partial sum l of a row runs over
            // the columns l, l + 32, ..., then the 32 partial sums are added
            // pairwise (l and l + 16, then l + 8, ...).  A warp of the
            // quadrant's pair holds 16 of them; the second hands its over.
            float part[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) part[i] = 0.0f;
            for (int c32 = half * 16; c32 < BN; c32 += 32) {
                float a8[8];
#pragma unroll
                for (int g = 0; g < 2; ++g) {
                    tmem_ld8(tq + (uint32_t)(c32 + 8 * g), a8);
#pragma unroll
                    for (int i = 0; i < 8; ++i) {
                        const int col = c32 + 8 * g + i;
                        const float h = __bfloat162float(__float2bfloat16(gelu(a8[i] + epi.bias[col])));
                        part[8 * g + i] = fmaf(h, epi.w4[col], part[8 * g + i]);
                    }
                }
            }
            float* ex = reinterpret_cast<float*>(smem) + quad * 32 * 17 + lane * 17;
            if (half == 1) {
#pragma unroll
                for (int i = 0; i < 16; ++i) ex[i] = part[i];
            }
            asm volatile("bar.sync %0, 64;" ::"r"(1 + quad) : "memory");
            if (half == 0 && row < M) {
#pragma unroll
                for (int i = 0; i < 16; ++i) part[i] += ex[i];
#pragma unroll
                for (int o = 8; o > 0; o >>= 1)
#pragma unroll
                    for (int i = 0; i < 8; ++i)
                        if (i < o) part[i] += part[i + o];
                epi.y[row] = part[0] + epi.w4[BN];
            }
        } else for (int c32 = half * 32; c32 < BN; c32 += 64) {
            // (a 16-column tile's last 16 values are not read)
            float w[32];
            const uint32_t ta = tq + (uint32_t)c32;
            const int nc = BN - c32 < 32 ? 16 : 32, col0 = n0 + c32;
            if (nc == 32) {
                tmem_ld32(ta, w);
            } else {
                float a8[8], b8[8];
                tmem_ld8(ta, a8);
                tmem_ld8(ta + 8, b8);
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    w[i] = a8[i];
                    w[8 + i] = b8[i];
                    w[16 + i] = w[24 + i] = 0.f;
                }
            }
            if (epi.mode == 0) {
                put_f32(w);
                if (vec_c) {
                    store_f32(epi.C, epi.ldc, col0, nc);
                } else {
                    for (int rr = 0; rr < 32 && r0 + rr < M; ++rr)
                        if (lane < nc) epi.C[(size_t)(r0 + rr) * epi.ldc + col0 + lane] = *reinterpret_cast<const float*>(tr + rr * 144 + lane * 4);
                    __syncwarp();
                }
                continue;
            }
            __align__(16) __nv_bfloat16 h[32];
            if (epi.mode == 1) {
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                    if (i < nc) w[i] += epi.bias[col0 + i];
                    h[i] = __float2bfloat16(gelu(w[i]));
                }
                if (epi.Z) {
                    put_f32(w);
                    store_f32(epi.Z, N, col0, nc);
                }
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const int rr = i * 4 + (lane >> 3), c = (lane & 7) * 4;
                    if (r0 + rr < M && c < nc)
                        *reinterpret_cast<float4*>(tr + rr * 144 + c * 4) =
                            *reinterpret_cast<const float4*>(epi.Zprev + (size_t)(r0 + rr) * N + col0 + c);
                }
                __syncwarp();
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const float4 z = *reinterpret_cast<const float4*>(tr + lane * 144 + i * 16);
                    h[4 * i] = __float2bfloat16(w[4 * i] * gelu_grad(z.x));
                    h[4 * i + 1] = __float2bfloat16(w[4 * i + 1] * gelu_grad(z.y));
                    h[4 * i + 2] = __float2bfloat16(w[4 * i + 2] * gelu_grad(z.z));
                    h[4 * i + 3] = __float2bfloat16(w[4 * i + 3] * gelu_grad(z.w));
                }
                __syncwarp();
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                *reinterpret_cast<uint4*>(tr + lane * 80 + i * 16) = reinterpret_cast<const uint4*>(h)[i];
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int rr = i * 8 + (lane >> 2), c = (lane & 3) * 8;
                if (r0 + rr < M && c < nc)
                    *reinterpret_cast<uint4*>(epi.H + (size_t)(r0 + rr) * N + col0 + c) =
                        *reinterpret_cast<const uint4*>(tr + rr * 80 + c * 2);
            }
            __syncwarp();
            if (epi.Ht && row < M) {
#pragma unroll
                for (int i = 0; i < 32; ++i)
                    if (i < nc) epi.Ht[(size_t)(col0 + i) * epi.ldt + row] = h[i];
            }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, ncols);
}

// One product; grid (M/128, N/BN).
__global__ void __launch_bounds__(kThreads, 2)
    gemm_bf16_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, int M,
                     int N, int K, int BN, int S, const __grid_constant__ Epi epi)
{
    gemm_tile(tmA, tmB, blockIdx.x * kBM, blockIdx.y * BN, M, N, K, BN, S, epi);
}

// Up to three products of one K into FP32 results in one launch, a block per
// tile: the weight gradients of a training batch, none of which has tiles for
// more than a tenth of the SMs.
struct Jobs {
    CUtensorMap a[3], b[3];
    float* C[3];
    int ldc[3], M[3], N[3], BN[3];
    int first[4];  // the product's first block
    int K, S;
    int* error;
};
__global__ void __launch_bounds__(kThreads, 2) gemm_bf16_batch_kernel(const __grid_constant__ Jobs j)
{
    const int q = (int)blockIdx.x < j.first[1] ? 0 : ((int)blockIdx.x < j.first[2] ? 1 : 2);
    const int t = blockIdx.x - j.first[q], rt = (j.M[q] + kBM - 1) / kBM;
    Epi e{};
    e.mode = 0;
    e.C = j.C[q];
    e.ldc = j.ldc[q];
    e.error = j.error;
    gemm_tile(j.a[q], j.b[q], t % rt * kBM, t / rt * j.BN[q], j.M[q], j.N[q], j.K, j.BN[q], j.S, e);
}

}  // namespace tc
}  // namespace amfrw
