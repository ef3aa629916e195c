// BF16 tensor-core GEMM for the trailing updates of the BEM LU factorisation
// (Sec. 2.2, Eq. (matrixBEM): the dense system is the one real dense
// contraction of the method).
//
//   C[M x N] -= A[M x K] B[K x N]      C, A, B: FP32 row-major sub-blocks
//
// Operands are rounded to BF16 (round to nearest even), products accumulated in
// FP32.  K <= 128, C not too large: tc_fused_kernel, from the FP32 operands.  Else the
// operands into K-major scratch (A as is, B transposed; tc_cvt_kernel), then one
// CTA per 256 x 256 or 128 x 128 tile of C (tiles ordered in groups of 2048 rows
// for L2 reuse) runs a TMA -> shared memory -> tcgen05.mma pipeline:
//   warp 0, one lane   TMA producer: 64-wide K slices of A and B into a 3-stage
//                      ring, 128B-swizzled
//   warp 1, one lane   MMA issuer: per slice 4 K steps x 1 or 2
//                      tcgen05.mma.kind::f16 (M 128, N 128 or 256, K 16), one per
//                      128 rows, all on the stage's B; FP32 accumulation in
//                      tensor memory; tcgen05.commit frees a stage
//   warps 0-7          epilogue: tcgen05.ld of their 32 lanes and half the
//                      columns of each accumulator, through shared memory,
//                      C -= D with coalesced row accesses
// Bound: the tensor cores from K 8192 on (2.0 PFLOP/s at 32,768), C's traffic and
// latency below K 1024 (14 us per call at K 64 in 256 x 256 tiles plus 9 of
// conversion, 5.5 fused).  The updates of order 59,968 with conversions: 168 to
// 133 ms.
// Every wait on an mbarrier is bounded; a wait that runs out records
// OBEM_ERR_TIMEOUT in *err, the kernel lets its issued copies and MMAs finish
// (bounded again), frees its tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include "obem_internal.cuh"

namespace {
constexpr int TC_MM = 128;                                        // rows of one MMA and of one accumulator
constexpr int TC_BK = 64, TC_STAGES = 3, TC_THREADS = 256;
constexpr int TC_GROUP_ROWS = 2048;                              // rows of C per rasterisation group
static_assert((TC_THREADS / 32) * 32 * 33 * 4 <= 3 * 128 * TC_BK * 2, "the epilogue's staging fits the stages of A");
constexpr int TF_THREADS = 256;                                  // fused kernel
constexpr unsigned long long TC_WAIT_NS = 2000000000ull;   // 2 s per wait
// a tile of BM x BN: operand bytes of a stage, shared memory, tensor-memory columns
__host__ __device__ constexpr uint32_t tc_a_bytes(int bm) { return (uint32_t)bm * TC_BK * 2; }
__host__ __device__ constexpr uint32_t tc_stage_bytes(int bm, int bn) { return (uint32_t)(bm + bn) * TC_BK * 2; }
__host__ __device__ constexpr size_t tc_smem_bytes(int bm, int bn) { return 1024 + (size_t)TC_STAGES * tc_stage_bytes(bm, bn) + 256; }
// instruction descriptor of tcgen05.mma.kind::f16: D FP32 (bits 4-5 = 1),
// A and B BF16 (bits 7-9 = 1, 10-12 = 1), both K-major (bits 15, 16 = 0),
// N >> 3 in bits 17-22, M >> 4 in bits 24-28
__host__ __device__ constexpr uint32_t tc_idesc(int bn)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(bn >> 3) << 17) | ((uint32_t)(TC_MM >> 4) << 24);
}
}

__device__ __forceinline__ uint32_t tc_smem(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void tc_mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(tc_smem(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void tc_mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc_smem(bar)), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ unsigned long long tc_now()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// true once the phase of the given parity has completed; false when it has
// not completed within TC_WAIT_NS of the first poll
__device__ __forceinline__ bool tc_mbar_wait(uint64_t *bar, uint32_t parity)
{
    const uint32_t a = tc_smem(bar);
    const unsigned long long t0 = tc_now();
    for (unsigned i = 0;; ++i) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\t"
                     "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}"
                     : "=r"(done)
                     : "r"(a), "r"(parity)
                     : "memory");
        if (done) return true;
        if ((i & 255u) == 255u && tc_now() - t0 > TC_WAIT_NS) return false;
    }
}

__device__ __forceinline__ void tc_tma_load(const CUtensorMap *tm, uint64_t *bar, void *dst, int x, int y)
{
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                 ::"r"(tc_smem(dst)), "l"((unsigned long long)tm), "r"(tc_smem(bar)), "r"(x), "r"(y)
                 : "memory");
}

// shared-memory matrix descriptor of a K-major, 128B-swizzled operand tile
// (rows of 64 BF16 = 128 bytes, 8-row groups 1024 bytes apart): start
// address >> 4 (bits 0-13), leading offset 1 (unused with this swizzle),
// stride offset 1024 >> 4 (bits 32-45), descriptor version 1 (bit 46),
// swizzle mode 2 = 128B (bits 61-63)
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr)
{
    return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t accumulate, uint32_t idesc)
{
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "setp.ne.b32 p, %3, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %4, p;\n\t}"
                 ::"r"(d_tmem), "l"(a), "l"(b), "r"(accumulate), "r"(idesc)
                 : "memory");
}

__device__ __forceinline__ void tc_commit(uint64_t *bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc_smem(bar))
                 : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 32 consecutive FP32 columns of the warp's 32 lanes (thread t: lane t)
__device__ __forceinline__ void tc_tmem_ld32(uint32_t taddr, uint32_t (&r)[32])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                 "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                 "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                   "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
                   "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
                   "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
                   "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
                 : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Tiles of 256 x 256 (all 512 columns of tensor memory, one CTA per SM) or of
// 128 x 128 (two CTAs per SM, so that one's epilogue runs beside the other's
// main loop, and four times the tiles: updates of short K or few tiles).
template <int TC_BM, int TC_BN>
__global__ void __launch_bounds__(TC_THREADS, TC_BM == 256 ? 1 : 2)
tc_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, float *__restrict__ C,
               long long ldc, int M, int N, int K, int *err)
{
    constexpr int TC_ACC = TC_BM / TC_MM, TC_GROUP_M = TC_GROUP_ROWS / TC_BM;
    constexpr uint32_t TC_A_BYTES = tc_a_bytes(TC_BM), TC_STAGE_BYTES = tc_stage_bytes(TC_BM, TC_BN),
                       TC_B_BYTES = TC_STAGE_BYTES - TC_A_BYTES, TC_TMEM_COLS = TC_ACC * TC_BN;
    extern __shared__ uint8_t tc_smem_raw[];
    uint8_t *sm = (uint8_t *)(((uintptr_t)tc_smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sA = sm;
    uint8_t *sB = sm + TC_STAGES * TC_A_BYTES;
    uint64_t *full = (uint64_t *)(sm + TC_STAGES * TC_STAGE_BYTES);
    uint64_t *empty = full + TC_STAGES;
    uint64_t *done = empty + TC_STAGES;
    uint32_t *tmem_slot = (uint32_t *)(done + 1);
    int *s_fail = (int *)(tmem_slot + 1);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // tile of this CTA: groups of TC_GROUP_M row tiles are walked down the
    // rows first, so the CTAs resident at one time cover a compact block of C
    // and share their A and B slices in L2
    int m_tile, n_tile;
    {
        const int num_m = (M + TC_BM - 1) / TC_BM, num_n = (N + TC_BN - 1) / TC_BN;
        const int pid = blockIdx.x;
        const int per_group = TC_GROUP_M * num_n;
        const int first_m = (pid / per_group) * TC_GROUP_M;
        const int gm = min(num_m - first_m, TC_GROUP_M);
        m_tile = first_m + (pid % per_group) % gm;
        n_tile = (pid % per_group) / gm;
    }
    const int n0 = n_tile * TC_BN, m0 = m_tile * TC_BM;
    const int nk = (K + TC_BK - 1) / TC_BK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < TC_STAGES; ++s) {
            tc_mbar_init(&full[s], 1);
            tc_mbar_init(&empty[s], 1);
        }
        tc_mbar_init(done, 1);
        *s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"((unsigned long long)&tmA) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"((unsigned long long)&tmB) : "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem(tmem_slot)),
                     "r"(TC_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp >= 2) {
        // the epilogue reads and rewrites this CTA's tile of C: bring it into
        // L2 while the main loop runs (lines of 128 bytes)
        for (int e = threadIdx.x - 64; e < TC_BM * (TC_BN / 32); e += TC_THREADS - 64) {
            const int r = m0 + e / (TC_BN / 32), cc = n0 + (e % (TC_BN / 32)) * 32;
            if (r < M && cc < N)
                asm volatile("prefetch.global.L2 [%0];" ::"l"((unsigned long long)(C + (size_t)r * ldc + cc)));
        }
    }
    if (warp == 0 && lane == 0) {
        // producer
        int kb = 0;
        for (; kb < nk; ++kb) {
            const int s = kb % TC_STAGES;
            if (kb >= TC_STAGES && !tc_mbar_wait(&empty[s], ((kb / TC_STAGES) - 1) & 1)) {
                atomicExch(s_fail, 1);
                break;
            }
            tc_mbar_expect_tx(&full[s], TC_STAGE_BYTES);
            tc_tma_load(&tmA, &full[s], sA + s * TC_A_BYTES, kb * TC_BK, m0);
            tc_tma_load(&tmB, &full[s], sB + s * TC_B_BYTES, kb * TC_BK, n0);
        }
        if (*(volatile int *)s_fail) {
            // let the copies this thread issued land before the CTA exits
            for (int q = kb - 1; q >= 0 && q >= kb - TC_STAGES; --q)
                tc_mbar_wait(&full[q % TC_STAGES], (q / TC_STAGES) & 1);
        }
    } else if (warp == 1 && lane == 0) {
        // MMA issuer
        for (int kb = 0; kb < nk; ++kb) {
            const int s = kb % TC_STAGES;
            if (!tc_mbar_wait(&full[s], (kb / TC_STAGES) & 1)) {
                atomicExch(s_fail, 1);
                break;
            }
            tc_fence_after();
            const uint32_t a0 = tc_smem(sA + s * TC_A_BYTES), b0 = tc_smem(sB + s * TC_B_BYTES);
            // accumulator a: rows a*128 .. a*128+127 of the tile (their A rows
            // start a*128 rows = 16 KB into the stage, a whole number of
            // 1024-byte swizzle atoms) in tensor-memory columns a*256 ..;
            // both share the stage's B.  A half of the tile past M is skipped.
#pragma unroll
            for (int j = 0; j < TC_BK / 16; ++j)
#pragma unroll
                for (int a = 0; a < TC_ACC; ++a)
                    if (a == 0 || m0 + a * TC_MM < M)
                        tc_mma(tmem + (uint32_t)(a * TC_BN), tc_desc(a0 + (uint32_t)(a * TC_MM * 128) + 32 * j),
                               tc_desc(b0 + 32 * j), (kb | j) != 0, tc_idesc(TC_BN));
            tc_commit(&empty[s]);
        }
        // arrives once every MMA issued above has completed (also on failure)
        tc_commit(done);
    }
    __syncwarp();

    // epilogue: warp w owns accumulator lanes (rows) 32 (w % 4) .. and columns
    // (w / 4) BN / 2 .. of each accumulator, in chunks of 32 columns; the next
    // chunk's values of C (the first one's before the wait) are in flight while
    // a chunk is written back
    constexpr int CH = TC_BN / 64, NCH = TC_ACC * CH;           // chunks of a warp, accumulator by accumulator
    const int cbase = n0 + (warp >> 2) * (TC_BN / 2);
    auto chunk = [&](int q, int &rbase, int &col) {
        rbase = m0 + (q / CH) * TC_MM + (warp & 3) * 32;
        col = cbase + (q % CH) * 32 + lane;
    };
    float vn[32];
    auto load_c = [&](int q) {
        int rbase, col;
        chunk(q, rbase, col);
        const int nrow = col < N ? M - rbase : 0;
        const float *cp = C + (size_t)rbase * ldc + col;
#pragma unroll
        for (int i = 0; i < 32; ++i) vn[i] = i < nrow ? __ldcg(cp + (size_t)i * ldc) : 0.f;
    };
    load_c(0);
    const bool fine = tc_mbar_wait(done, 0);
    tc_fence_after();
    __syncthreads();
    if (fine && !*(volatile int *)s_fail) {
        float *stage = (float *)sA + warp * 32 * 33;       // pipeline smem is idle now
#pragma unroll 1
        for (int q = 0; q < NCH; ++q) {
            float v[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) v[i] = vn[i];
            if (q + 1 < NCH) load_c(q + 1);
            int rbase, col;
            chunk(q, rbase, col);
            if (rbase >= M || col - lane >= N) continue;    // warp-uniform
            uint32_t r[32];
            tc_tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) +
                             (uint32_t)((q / CH) * TC_BN + (warp >> 2) * (TC_BN / 2) + (q % CH) * 32), r);
#pragma unroll
            for (int j = 0; j < 32; ++j) stage[lane * 33 + j] = __uint_as_float(r[j]);
            __syncwarp();
            const int nrow = col < N ? M - rbase : 0;
            float *cp = C + (size_t)rbase * ldc + col;
#pragma unroll
            for (int i = 0; i < 32; ++i)
                if (i < nrow) __stcg(cp + (size_t)i * ldc, v[i] - stage[i * 33 + lane]);
            __syncwarp();
        }
    } else if (threadIdx.x == 0) {
        atomicExch(err, OBEM_ERR_TIMEOUT);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_TMEM_COLS)
                     : "memory");
}

// C[M x N] -= A[M x K] B[K x N] for K <= TF_K, from the FP32 operands: a CTA
// per 128 x BN tile converts its slices of A and B in registers, writes them to
// shared memory in the layout of the MMA's descriptors and issues the MMAs.  No
// conversion pass, no BF16 scratch, no ring: with K this short an update is its
// traffic of C (4 bytes read and written per 2 K flops) and the latency of a
// launch, and two thirds of a factorisation's updates have K <= 128.
constexpr int TF_K = 128, TF_BN = 64;
constexpr size_t tf_smem(int nk)
{
    const size_t op = (size_t)nk * tc_stage_bytes(TC_MM, TF_BN), st = (TF_THREADS / 32) * 32 * 33 * sizeof(float);
    return 1024 + (op > st ? op : st) + 64;
}
template <bool VEC>
__global__ void __launch_bounds__(TF_THREADS, 2)
tc_fused_kernel(float *__restrict__ C, long long ldc, const float *__restrict__ A, long long lda,
                const float *__restrict__ B, long long ldb, int M, int N, int K, int *err)
{
    constexpr int BN = TF_BN;
    static_assert(BN == 64, "a chunk of 32 columns per warp");
    constexpr uint32_t A_BYTES = tc_a_bytes(TC_MM), STAGE = tc_stage_bytes(TC_MM, BN);
    extern __shared__ uint8_t tc_smem_raw[];
    __shared__ uint64_t s_done;
    __shared__ uint32_t s_tmem;
    uint8_t *sm = (uint8_t *)(((uintptr_t)tc_smem_raw + 1023) & ~(uintptr_t)1023);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int num_m = (M + TC_MM - 1) / TC_MM;
    const int m0 = (blockIdx.x % num_m) * TC_MM, n0 = (blockIdx.x / num_m) * BN;
    const int nk = (K + TC_BK - 1) / TC_BK;
    if (tid == 0) {
        tc_mbar_init(&s_done, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem(&s_tmem)),
                     "r"((uint32_t)BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // the tile of C into L2 (lines of 128 bytes)
    for (int e = tid; e < TC_MM * (BN / 32); e += TF_THREADS) {
        const int r = m0 + e / (BN / 32), cc = n0 + (e % (BN / 32)) * 32;
        if (r < M && cc < N) asm volatile("prefetch.global.L2 [%0];" ::"l"((unsigned long long)(C + (size_t)r * ldc + cc)));
    }
    union Pack { __nv_bfloat162 h[4]; uint4 u; };
    auto put = [](uint8_t *tile, int row, int c, const float (&v)[8]) {        // 16-byte chunk c of a 128-byte row, swizzled
        Pack o;
#pragma unroll
        for (int q = 0; q < 4; ++q) o.h[q] = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
        *reinterpret_cast<uint4 *>(tile + row * 128 + ((c ^ (row & 7)) << 4)) = o.u;
    };
    for (int kc = 0; kc < nk; ++kc) {
        uint8_t *sA = sm + kc * STAGE, *sB = sA + A_BYTES;
        float va[4][8], vb[BN / 32][8];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = tid + TF_THREADS * q, r = m0 + (e >> 3), k = kc * TC_BK + (e & 7) * 8;
            const float *p = A + (size_t)r * lda + k;
            if (VEC && r < M && k + 8 <= K) {
                const float4 x = *reinterpret_cast<const float4 *>(p), y = *reinterpret_cast<const float4 *>(p + 4);
                va[q][0] = x.x; va[q][1] = x.y; va[q][2] = x.z; va[q][3] = x.w;
                va[q][4] = y.x; va[q][5] = y.y; va[q][6] = y.z; va[q][7] = y.w;
            } else {
#pragma unroll
                for (int i = 0; i < 8; ++i) va[q][i] = r < M && k + i < K ? p[i] : 0.f;
            }
        }
#pragma unroll
        for (int q = 0; q < BN / 32; ++q) {
            const int e = tid + TF_THREADS * q, n = n0 + e % BN, k = kc * TC_BK + (e / BN) * 8;
#pragma unroll
            for (int i = 0; i < 8; ++i) vb[q][i] = n < N && k + i < K ? B[(size_t)(k + i) * ldb + n] : 0.f;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = tid + TF_THREADS * q;
            put(sA, e >> 3, e & 7, va[q]);
        }
#pragma unroll
        for (int q = 0; q < BN / 32; ++q) {
            const int e = tid + TF_THREADS * q;
            put(sB, e % BN, e / BN, vb[q]);
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = s_tmem;
    if (tid == 0) {
        for (int kc = 0; kc < nk; ++kc) {
            const uint32_t a0 = tc_smem(sm + kc * STAGE), b0 = a0 + A_BYTES;
#pragma unroll
            for (int j = 0; j < TC_BK / 16; ++j)
                tc_mma(tmem, tc_desc(a0 + 32 * j), tc_desc(b0 + 32 * j), (kc | j) != 0, tc_idesc(BN));
        }
        tc_commit(&s_done);
    }
    __syncwarp();
    // epilogue: warp w owns accumulator lanes (rows) 32 (w % 4) .., columns
    // (w / 4) BN / 2 .. of the tile; its values of C are on the way meanwhile
    const int rbase = m0 + (warp & 3) * 32, cbase = (warp >> 2) * (BN / 2);
    const int nrow = min(32, M - rbase);
    const int col = n0 + cbase + lane;
    float *cp = C + (size_t)rbase * ldc + col;
    float v[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = (i < nrow && col < N) ? __ldcg(cp + (size_t)i * ldc) : 0.f;
    const bool fine = tc_mbar_wait(&s_done, 0);
    tc_fence_after();
    __syncthreads();
    if (fine) {
        float *stage = (float *)sm + warp * 32 * 33;            // the operands have been read
        uint32_t r[32];
        tc_tmem_ld32(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)cbase, r);
#pragma unroll
        for (int j = 0; j < 32; ++j) stage[lane * 33 + j] = __uint_as_float(r[j]);
        __syncwarp();
        if (col < N) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
                if (i < nrow) __stcg(cp + (size_t)i * ldc, v[i] - stage[i * 33 + lane]);
        }
    } else if (tid == 0) {
        atomicExch(err, OBEM_ERR_TIMEOUT);
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)BN) : "memory");
}

// Both operands of a GEMM to BF16 in one launch: blocks [0, na) round 64 x 64
// tiles of A (Ab[i][k] = bf16(A[i][k])), the others round and transpose tiles of
// B (Bb[j][k] = bf16(B[k][j])) through shared memory.  Eight values per 16-byte
// store; VEC: float4 loads (both matrices 16-byte aligned with row pitches of
// multiples of 4).  Columns K .. ldo - 1 are written as zeros.  HBM-bound for the
// large operands (6 bytes per element); most of the factorisation's 2,729
// GEMMs are small and paid the launch of a second kernel and 2- and 4-byte
// accesses: 50.3 ms of conversions at order 59,968 in two kernels.
#define CV_T 64
template <bool VEC>
__global__ void __launch_bounds__(256) tc_cvt_kernel(const float *__restrict__ A, long long lda, int M, int K,
                                                     __nv_bfloat16 *__restrict__ Ab, const float *__restrict__ B,
                                                     long long ldb, int N, __nv_bfloat16 *__restrict__ Bb, int ldo,
                                                     int na, int nk)
{
    __shared__ float t[CV_T][CV_T + 1];
    const int tid = threadIdx.x;
    union Pack { __nv_bfloat162 h[4]; uint4 u; };
    auto load8 = [](const float *p, int left, float (&v)[8]) {
        if (VEC && left >= 8) {
            const float4 x = *reinterpret_cast<const float4 *>(p), y = *reinterpret_cast<const float4 *>(p + 4);
            v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w; v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
        } else {
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = q < left ? p[q] : 0.f;
        }
    };
    auto store8 = [](__nv_bfloat16 *p, const float (&v)[8]) {
        Pack o;
#pragma unroll
        for (int q = 0; q < 4; ++q) o.h[q] = __floats2bfloat162_rn(v[2 * q], v[2 * q + 1]);
        *reinterpret_cast<uint4 *>(p) = o.u;
    };
    const bool isA = (int)blockIdx.x < na;
    const int tile = isA ? blockIdx.x : blockIdx.x - na;
    const int k0 = (tile % nk) * CV_T, i0 = (tile / nk) * CV_T;
    if (isA) {
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const int i = i0 + (tid >> 3) + 32 * q, k = k0 + (tid & 7) * 8;
            if (i >= M || k >= ldo) continue;
            float v[8];
            load8(A + (size_t)i * lda + k, K - k, v);
            store8(Ab + (size_t)i * ldo + k, v);
        }
        return;
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int r = (tid >> 3) + 32 * q, c = (tid & 7) * 8;
        float v[8];
        load8(B + (size_t)(k0 + r) * ldb + i0 + c, k0 + r < K ? N - i0 - c : 0, v);
#pragma unroll
        for (int e = 0; e < 8; ++e) t[r][c + e] = v[e];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const int c = (tid >> 3) + 32 * q, r = (tid & 7) * 8;
        if (i0 + c >= N || k0 + r >= ldo) continue;
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = t[r + e][c];
        store8(Bb + (size_t)(i0 + c) * ldo + k0 + r, v);
    }
}

// ------------------------------------------------------------------ host side
typedef CUresult (*tc_encode_fn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static tc_encode_fn tc_encoder()
{
    static tc_encode_fn fn = NULL;
    if (!fn) {
        void *p = NULL;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = (tc_encode_fn)p;
    }
    return fn;
}

// 2-D map of a K-major BF16 matrix [rows][ld] with K valid columns, boxes of
// 64 x box_rows, 128-byte swizzle, zero fill outside
static int tc_map(obem_ctx *c, CUtensorMap *m, const void *base, int rows, int K, int ld, int box_rows)
{
    tc_encode_fn enc = tc_encoder();
    if (!enc) return obem_fail(c, OBEM_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
    cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)TC_BK, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, es,
                     CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                     CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return obem_fail(c, OBEM_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
    return OBEM_OK;
}

// BF16 scratch of the context for operands up to a_elems / b_elems elements
int obem_tc_reserve(obem_ctx *c, size_t a_elems, size_t b_elems)
{
    if (a_elems * 2 > c->tc_a_bytes) {
        if (c->tc_a) cudaFree(c->tc_a);
        c->tc_a = NULL;
        c->tc_a_bytes = 0;
        OBEM_CUDA(c, cudaMalloc(&c->tc_a, a_elems * 2));
        c->tc_a_bytes = a_elems * 2;
    }
    if (b_elems * 2 > c->tc_b_bytes) {
        if (c->tc_b) cudaFree(c->tc_b);
        c->tc_b = NULL;
        c->tc_b_bytes = 0;
        OBEM_CUDA(c, cudaMalloc(&c->tc_b, b_elems * 2));
        c->tc_b_bytes = b_elems * 2;
    }
    return OBEM_OK;
}

void obem_tc_free(obem_ctx *c)
{
    if (c->tc_a) cudaFree(c->tc_a);
    if (c->tc_b) cudaFree(c->tc_b);
    c->tc_a = c->tc_b = NULL;
    c->tc_a_bytes = c->tc_b_bytes = 0;
}

// Tiles of 128 x 128 (else 256 x 256): short K, where a tile is mostly epilogue,
// and updates whose larger tiles would leave half the SMs idle.  Measured 256 /
// 128 (us, M x N x K): 30000 x 256 x 256 20.7 / 19.0, 512 x 512 x 512 22.2 / 9.0,
// 30000 x 1024 x 1024 123 / 95, 4000 x 2048 x 2048 37 / 41, 30000 x 2048 x 2048 282 /
// 255, 512 x 4096 x 4096 55 / 32, 4000 x 4096 x 4096 116 / 132.
static bool tc_small_tiles(int M, int N, int K)
{
    const long long t256 = (long long)((N + 255) / 256) * ((M + 255) / 256);
    return K <= 1024 || t256 <= 76 || (K <= 2048 && t256 > 152);
}

// From the FP32 operands in one kernel: K up to TF_K, where C is small enough for
// the latency of a second launch to count; its 64 columns a tile read A again for
// every 64 columns of C.  Measured fused / converted and 128 x 128 (us, M x N x K):
// 60000 x 128 x 64 63 / 66 and x 128 65 / 66, 2048 x 2048 x 128 53 / 55, 4096 x 4096 x 64
// 77 / 71 and x 128 88 / 82, 30000 x 512 x 128 97 / 79, 30000 x 30000 x 64 2138 / 1635 and x
// 128 2420 / 1689.
static bool tc_fused(int M, int N, int K) { return K <= TF_K && (long long)M * N <= 10000000ll; }

// C[M x N] -= A[M x K] B[K x N] with BF16 operands and FP32 accumulation;
// C, A, B are FP32 row-major blocks with leading dimensions ldc, lda, ldb.
// Uses the context's BF16 scratch (obem_tc_reserve grows it); err: device
// int receiving OBEM_ERR_TIMEOUT if a bounded wait ran out.
int obem_tc_gemm_sub(obem_ctx *c, float *C, long long ldc, const float *A, long long lda, const float *B, long long ldb,
                     int M, int N, int K, int *err, cudaStream_t s)
{
    if (M <= 0 || N <= 0 || K <= 0) return OBEM_OK;
    static unsigned long long attr = 0;   // devices done (a bit each)
    if (!(attr >> (c->device & 63) & 1ull)) {
        OBEM_CUDA(c, cudaFuncSetAttribute(tc_gemm_kernel<256, 256>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)tc_smem_bytes(256, 256)));
        OBEM_CUDA(c, cudaFuncSetAttribute(tc_gemm_kernel<128, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)tc_smem_bytes(128, 128)));
        OBEM_CUDA(c, cudaFuncSetAttribute(tc_fused_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)tf_smem(TF_K / TC_BK)));
        OBEM_CUDA(c, cudaFuncSetAttribute(tc_fused_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)tf_smem(TF_K / TC_BK)));
        attr |= 1ull << (c->device & 63);
    }
    const bool vec = (((uintptr_t)A | (uintptr_t)B) & 15) == 0 && ((lda | ldb) & 3) == 0;
    const long long t128 = (long long)((N + 127) / 128) * ((M + 127) / 128);
    if (t128 > 0x3fffffffll) return obem_fail(c, OBEM_ERR_ARG, "tensor-core GEMM: %d x %d exceeds the grid", M, N);
    if (tc_fused(M, N, K)) {
        const int nk = (K + TC_BK - 1) / TC_BK;
        const unsigned g = (unsigned)((long long)((N + TF_BN - 1) / TF_BN) * ((M + TC_MM - 1) / TC_MM));
        if (vec) tc_fused_kernel<true><<<g, TF_THREADS, tf_smem(nk), s>>>(C, ldc, A, lda, B, ldb, M, N, K, err);
        else tc_fused_kernel<false><<<g, TF_THREADS, tf_smem(nk), s>>>(C, ldc, A, lda, B, ldb, M, N, K, err);
        OBEM_LAUNCH(c);
        return OBEM_OK;
    }
    const int ldk = (K + 7) / 8 * 8;                       // 16-byte row pitch for the tensor maps
    int rc = obem_tc_reserve(c, (size_t)M * ldk, (size_t)N * ldk);
    if (rc != OBEM_OK) return rc;
    __nv_bfloat16 *Ab = (__nv_bfloat16 *)c->tc_a, *Bb = (__nv_bfloat16 *)c->tc_b;
    {
        const int nk = (ldk + CV_T - 1) / CV_T;
        const long long na = (long long)((M + CV_T - 1) / CV_T) * nk, nb = (long long)((N + CV_T - 1) / CV_T) * nk;
        if (na + nb > 0x7fffffffll) return obem_fail(c, OBEM_ERR_ARG, "tensor-core GEMM: operands exceed the grid");
        if (vec) tc_cvt_kernel<true><<<(unsigned)(na + nb), 256, 0, s>>>(A, lda, M, K, Ab, B, ldb, N, Bb, ldk, (int)na, nk);
        else tc_cvt_kernel<false><<<(unsigned)(na + nb), 256, 0, s>>>(A, lda, M, K, Ab, B, ldb, N, Bb, ldk, (int)na, nk);
        OBEM_LAUNCH(c);
    }
    const bool small = tc_small_tiles(M, N, K);
    const int bt = small ? 128 : 256;
    CUtensorMap ma, mb;
    rc = tc_map(c, &ma, Ab, M, K, ldk, bt);
    if (rc == OBEM_OK) rc = tc_map(c, &mb, Bb, N, K, ldk, bt);
    if (rc != OBEM_OK) return rc;
    if (small) {
        tc_gemm_kernel<128, 128><<<(unsigned)t128, TC_THREADS, tc_smem_bytes(128, 128), s>>>(ma, mb, C, ldc, M, N, K, err);
    } else {
        const unsigned g = (unsigned)(((N + 255) / 256) * ((M + 255) / 256));
        tc_gemm_kernel<256, 256><<<g, TC_THREADS, tc_smem_bytes(256, 256), s>>>(ma, mb, C, ldc, M, N, K, err);
    }
    OBEM_LAUNCH(c);
    return OBEM_OK;
}

// C ABI hook: the same update on caller arrays (FP32, row-major), for tests
// and measurement of the tensor-core path; synchronises the stream and
// reports a bounded-wait timeout as OBEM_ERR_TIMEOUT.
extern "C" int obem_tc_gemm(obem_ctx *c, float *C, int64_t ldc, const float *A, int64_t lda, const float *B,
                            int64_t ldb, int32_t M, int32_t N, int32_t K, obem_stream stream)
{
    if (!c || !C || !A || !B) return OBEM_ERR_ARG;
    if (M < 0 || N < 0 || K < 0 || ldc < N || lda < K || ldb < N) return obem_fail(c, OBEM_ERR_ARG, "tc_gemm: bad sizes");
    cudaStream_t s = (cudaStream_t)stream;
    int *err = NULL;
    OBEM_CUDA(c, cudaMalloc((void **)&err, sizeof(int)));
    int h = 0;
    cudaError_t e = cudaMemsetAsync(err, 0, sizeof(int), s);
    int rc = OBEM_OK;
    if (e == cudaSuccess) rc = obem_tc_gemm_sub(c, C, ldc, A, lda, B, ldb, M, N, K, err, s);
    if (e == cudaSuccess && rc == OBEM_OK) e = cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && rc == OBEM_OK) e = cudaStreamSynchronize(s);
    cudaFree(err);
    if (rc != OBEM_OK) return rc;
    if (e != cudaSuccess) return obem_fail(c, OBEM_ERR_CUDA, "tc_gemm: %s", cudaGetErrorString(e));
    if (h != 0) return obem_fail(c, OBEM_ERR_TIMEOUT, "tc_gemm: a bounded wait ran out");
    return OBEM_OK;
}
