// BEM set-up: assembly of the dense system of Eq. (matrixBEM), its LU
// factorisation, and solves with iterative refinement.  Sec. 2.2 fills the
// matrix on the GPU and keeps an inverse so that new voltages or free charges
// only need a new right-hand side; here the factors are kept instead of the
// inverse (same reuse, half the flops, better conditioned).
//
//   assemble_kernel   a thread per column, rows two at a time: Q_ij = k_C
//                     phi_j(r_i) for electrode rows, W_ij for dielectric
//                     rows; closed form for near cells (queued), FP32
//                     quadrature (7/3/1 points by distance) for far ones
//   equilibrate       scale every row by the power of two nearest below
//                     1 / max |A_ij| (exact; solution unchanged)
//   LU                partial pivoting; panels of LU_NB columns factored by
//                       panel_kernel   cooperative: one row chunk per CTA held
//                                      in shared memory, one bounded exchange
//                                      of pivot candidates per column
//                       laswp_*        the panel's row swaps on whole rows
//                                      (plan, gather to scratch, scatter)
//                     BF16 (OBEM_LU_BF16): recursive (rec_lu / rec_trsm), every
//                       trailing update and off-diagonal TRSM block a
//                       hand-written tcgen05 GEMM (lu_tc.cu: BF16 operands,
//                       FP32 accumulation into the FP32 factors)
//                     FP32 / TF32 / BF16x9: right-looking blocked, trsm_kernel
//                       for U12 = L11^-1 A12 and cuBLAS for A22 -= L21 U12
//   solve             y = L^-1 P b, x = U^-1 y (blocked, FP32 factors) inside
//                     iterative refinement with FP64 residuals r = b - A x
#include <math.h>
#include <vector>

#include "obem_internal.cuh"
#include "field_common.cuh"

template <bool B> struct AsBool { static constexpr bool value = B; };

#define LU_NB 64
#define TS_R 128               // rows of a block row of the one-launch triangular solves

#define AS_CLOSED_H2 16.0f     // d < 4 h: closed form
#define AS_7PT_H2 1024.0f      // d < 32 h: 7 points
#define AS_3PT_H2 360000.0f    // d < 600 h: 3 points, else centroid
#define AS_TH 128              // threads per block: one column (cell) each
#define AS_ROWS 64             // rows per block

// A block fills AS_ROWS rows of AS_TH columns: a thread keeps its column's cell
// in registers and takes the rows two at a time (f32x2), a far entry by the
// tier of the nearer of the two rows' centroids, evaluated without divergence
// as up to seven points c, c + a g_k, c + b g_k.  Near entries go to a
// per-warp queue of the closed form, 32 at a time: a warp-wide instruction
// costs the same with one lane as with 32, and with a thread per entry nearly
// every warp had a near one.  Electrode rows need the potential
// only, dielectric rows the field's component along their normal.
// Bound: FP32 issue of the far points (5 on average at 60k cells).  Measured at
// 59,968 cells: 174.2 to 33.0 ms, 16.5 with the near entries' closed form in pairs
// of floats.
__global__ void __launch_bounds__(AS_TH) assemble_kernel(PanelsDev P, const int *kind, const double *em,
                                                         const double *ep, float *A, int n)
{
    __shared__ u64 s_c[6][AS_ROWS / 2];              // centroids of the row pairs: x, y, z and their low parts
    __shared__ u64 s_n[3][AS_ROWS / 2];              // (eps+ - eps-) / (4 pi KC) n, 0 on electrode rows
    __shared__ int s_k[AS_ROWS / 2];                 // bit 0: an electrode row in the pair, bit 1: a dielectric one
    __shared__ uint32_t s_q[AS_TH / 32][64];         // closed-form queue: row << 8 | column of the block
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned below = (1u << lane) - 1u;
    const int i0 = blockIdx.y * AS_ROWS, rows = min(AS_ROWS, n - i0);
    const int j0 = blockIdx.x * AS_TH, j = min(j0 + tid, n - 1);
    const bool live = j0 + tid < n;
    for (int p = tid; p < AS_ROWS / 2; p += AS_TH) {
        const int a = min(i0 + 2 * p, n - 1), b = min(i0 + 2 * p + 1, n - 1);
        const float4 ca = P.c_a[a], cb = P.c_a[b], la = P.c_lo[a], lb = P.c_lo[b], na = P.nrm[a], nb = P.nrm[b];
        s_c[0][p] = pk(ca.x, cb.x); s_c[1][p] = pk(ca.y, cb.y); s_c[2][p] = pk(ca.z, cb.z);
        s_c[3][p] = pk(la.x, lb.x); s_c[4][p] = pk(la.y, lb.y); s_c[5][p] = pk(la.z, lb.z);
        const bool da = kind[a] != OBEM_CELL_ELECTRODE, db = kind[b] != OBEM_CELL_ELECTRODE;
        const float fa = da ? (float)((ep[a] - em[a]) / (4.0 * OBEM_PI * OBEM_KC)) : 0.f,
                    fb = db ? (float)((ep[b] - em[b]) / (4.0 * OBEM_PI * OBEM_KC)) : 0.f;
        s_n[0][p] = pk(fa * na.x, fb * nb.x); s_n[1][p] = pk(fa * na.y, fb * nb.y); s_n[2][p] = pk(fa * na.z, fb * nb.z);
        s_k[p] = (!da || !db ? 1 : 0) | (da || db ? 2 : 0) | (da ? 4 : 0) | (db ? 8 : 0);
    }
    __syncthreads();
    const float4 cj = P.c_a[j], lj = P.c_lo[j], g0 = P.g0_h[j], g1 = P.g1[j], g2 = P.g2[j];
    const float h2 = g0.w;
    int nq = 0;
    auto flush = [&](int m) {
        __syncwarp();
        if (lane < m) {
            const uint32_t e = s_q[warp][lane];
            const int i = i0 + (int)(e >> 8), jj = j0 + (int)(e & 255u);
            const bool pot = kind[i] == OBEM_CELL_ELECTRODE;
            const float4 ci = P.c_a[i], li = P.c_lo[i], ni = P.nrm[i];
            Dbf p, fx, fy, fz;
            float a;
            if (!pot && i == jj) {
                a = (float)(0.5 * (ep[i] + em[i]));
            } else if (tri_closed_df(P.geo2 + (size_t)OBEM_GEO2 * jj, Dbf{ci.x, li.x}, Dbf{ci.y, li.y}, Dbf{ci.z, li.z}, !pot,
                                     p, fx, fy, fz)) {
                const double w = pot ? OBEM_KC : (ep[i] - em[i]) * (1.0 / (4.0 * OBEM_PI));
                const float wh = (float)w;
                const Dbf s = pot ? p : df_sum(df_sum(df_mulf(fx, ni.x), df_mulf(fy, ni.y)), df_mulf(fz, ni.z));
                a = df_mul(Dbf{wh, (float)(w - (double)wh)}, s).h;
            } else {
                const double *vi = P.v64 + 9 * (size_t)i;
                double phi, Fx, Fy, Fz;
                tri_closed_form_g(P.v64 + 9 * (size_t)jj, P.geo + (size_t)OBEM_GEO64 * jj, (vi[0] + vi[3] + vi[6]) / 3.0,
                                  (vi[1] + vi[4] + vi[7]) / 3.0, (vi[2] + vi[5] + vi[8]) / 3.0, phi, Fx, Fy, Fz);
                a = (float)(pot ? OBEM_KC * phi : (ep[i] - em[i]) / (4.0 * OBEM_PI) * (Fx * ni.x + Fy * ni.y + Fz * ni.z));
            }
            A[(size_t)i * n + jj] = a;
        }
        __syncwarp();
    };
    for (int p = 0; 2 * p < rows; ++p) {
        const u64 DX = add2(sub2(s_c[0][p], pk(cj.x, cj.x)), sub2(s_c[3][p], pk(lj.x, lj.x))),
                  DY = add2(sub2(s_c[1][p], pk(cj.y, cj.y)), sub2(s_c[4][p], pk(lj.y, lj.y))),
                  DZ = add2(sub2(s_c[2][p], pk(cj.z, cj.z)), sub2(s_c[5][p], pk(lj.z, lj.z)));
        const int kp = s_k[p];
        float da, db;
        upk(fma2(DZ, DZ, fma2(DY, DY, mul2(DX, DX))), da, db);
        const int ia = i0 + 2 * p, ib = ia + 1;
        const bool na = da < AS_CLOSED_H2 * h2 || ia == j, nb = db < AS_CLOSED_H2 * h2 || ib == j;
        const u64 EP = pk(na ? 1e30f : 0.f, nb ? 1e30f : 0.f);
        const float dmin = fminf(na ? 3e38f : da, nb ? 3e38f : db);      // the far rows' (near entries: queue)
        const bool t1 = dmin >= AS_3PT_H2 * h2, t3 = dmin >= AS_7PT_H2 * h2;
        const float w0 = t1 ? 1.f : t3 ? 0.f : D7_W0, wa = t1 ? 0.f : t3 ? 1.0f / 3.0f : D7_W1,
                    sa = t1 ? 0.f : t3 ? 0.5f : D7_T1, wb = t3 ? 0.f : D7_W2, sb = t3 ? 0.f : D7_T2;
        u64 S = 0ull;
        auto points = [&](auto pot_c, auto fld_c) {
            constexpr bool POT = decltype(pot_c)::value, FLD = decltype(fld_c)::value;
            // mixed pair: each half has either a potential weight or a normal
            const u64 NX = s_n[0][p], NY = s_n[1][p], NZ = s_n[2][p];
            const u64 WP = pk(kp & 4 ? 0.f : 1.f, kp & 8 ? 0.f : 1.f);
            auto point = [&](float ox, float oy, float oz, float w) {
                const u64 dx = sub2(DX, pk(ox, ox)), dy = sub2(DY, pk(oy, oy)), dz = sub2(DZ, pk(oz, oz));
                float ra, rb;
                upk(fma2(dz, dz, fma2(dy, dy, fma2(dx, dx, EP))), ra, rb);
                const u64 inv = pk(rsq(ra), rsq(rb));
                const u64 wi = mul2(pk(w, w), inv);
                if (FLD) {
                    const u64 dn = fma2(dz, NZ, fma2(dy, NY, mul2(dx, NX)));
                    const u64 t = mul2(dn, mul2(inv, inv));
                    S = fma2(wi, POT ? add2(t, WP) : t, S);
                } else {
                    S = add2(S, wi);
                }
            };
            const float q = cj.w;
            if (__any_sync(0xffffffffu, w0 != 0.f)) point(0.f, 0.f, 0.f, q * w0);
            if (__any_sync(0xffffffffu, wa != 0.f)) {
                const float w = q * wa;
                point(sa * g0.x, sa * g0.y, sa * g0.z, w);
                point(sa * g1.x, sa * g1.y, sa * g1.z, w);
                point(sa * g2.x, sa * g2.y, sa * g2.z, w);
            }
            if (__any_sync(0xffffffffu, wb != 0.f)) {
                const float w = q * wb;
                point(sb * g0.x, sb * g0.y, sb * g0.z, w);
                point(sb * g1.x, sb * g1.y, sb * g1.z, w);
                point(sb * g2.x, sb * g2.y, sb * g2.z, w);
            }
        };
        if ((kp & 3) == 1) points(AsBool<true>{}, AsBool<false>{});
        else if ((kp & 3) == 2) points(AsBool<false>{}, AsBool<true>{});
        else points(AsBool<true>{}, AsBool<true>{});
        float a, b;
        upk(S, a, b);
        float *row = A + (size_t)ia * n + j;
        if (live && !na) row[0] = a;
        if (live && !nb && ib < n) row[n] = b;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
            const bool near = live && (half ? nb && ib < n : na);
            const unsigned bal = __ballot_sync(0xffffffffu, near);
            if (!bal) continue;
            if (near) s_q[warp][nq + __popc(bal & below)] = ((uint32_t)(2 * p + half) << 8) | (uint32_t)tid;
            nq += __popc(bal);
            if (nq >= 32) {
                flush(32);
                nq -= 32;
                if (lane < nq) s_q[warp][lane] = s_q[warp][32 + lane];
                __syncwarp();
            }
        }
    }
    if (nq > 0) flush(nq);
}

// Row equilibration: the rows of A scaled by 2^-floor(log2 max |a_ij|), the
// scaled matrix also written to LU (where it is factorised); the scale and the
// row's 1-norm recorded.  One block per row, read twice: the rows in flight
// (240 KB each at 60k cells) fit L2, so the second read seldom leaves it.
// HBM-bound: one read and two writes of the matrix, 43 GB at 59,968 cells in
// 8.5 ms (scaling in place 14.3 ms, the copy to LU another 4.3 ms).
#define EQ_TH 512
__global__ void __launch_bounds__(EQ_TH) equilibrate_kernel(float *A, float *LU, int n, double *rowscale,
                                                            double *rownorm)
{
    __shared__ float smax[EQ_TH / 32];
    __shared__ double ssum[EQ_TH / 32];
    float *row = A + (size_t)blockIdx.x * n, *out = LU + (size_t)blockIdx.x * n;
    const int tid = threadIdx.x;
    float m = 0.f;
    int j = tid;
    for (; j + 7 * EQ_TH < n; j += 8 * EQ_TH) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = row[j + u * EQ_TH];
#pragma unroll
        for (int u = 0; u < 8; ++u) m = fmaxf(m, fabsf(v[u]));
    }
    for (; j < n; j += EQ_TH) m = fmaxf(m, fabsf(row[j]));
    for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((tid & 31) == 0) smax[tid >> 5] = m;
    __syncthreads();
    for (int w = 0; w < EQ_TH / 32; ++w) m = fmaxf(m, smax[w]);
    // a power of two: the scaled row is exact, so the equilibrated system is
    // D A itself and the refined solution keeps FP64 accuracy for A
    const float sc = m > 0.f ? ldexpf(1.0f, -ilogbf(m)) : 1.0f;
    float s = 0.f, c = 0.f;
    for (j = tid; j + 7 * EQ_TH < n; j += 8 * EQ_TH) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = __ldcs(row + j + u * EQ_TH);
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            v[u] *= sc;
            __stcs(row + j + u * EQ_TH, v[u]);
            __stcs(out + j + u * EQ_TH, v[u]);
            two_sum_acc(s, c, fabsf(v[u]));
        }
    }
    for (; j < n; j += EQ_TH) {
        const float v = row[j] * sc;
        row[j] = v;
        out[j] = v;
        two_sum_acc(s, c, fabsf(v));
    }
    double t = (double)s + (double)c;
    for (int o = 16; o; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((tid & 31) == 0) ssum[tid >> 5] = t;
    __syncthreads();
    if (tid == 0) {
        t = 0.0;
        for (int w = 0; w < EQ_TH / 32; ++w) t += ssum[w];
        rownorm[blockIdx.x] = t;
        rowscale[blockIdx.x] = (double)sc;
    }
}

// ------------------------------------------------------------------ panel exchange
// The CTAs of the pivoting panel (a cooperative launch) meet once per column:
// each CTA publishes its pivot candidate (a 64-bit record) and the candidate's
// row, the owner of the row that receives the pivot publishes that row.  What
// is published carries the column's epoch (its number in the matrix + 1; the
// buffers are zeroed before the factorisation), so a reader polls the values
// themselves and no order among them matters.  A column is a chain of two
// trips through L2, records then the pivot row; with an arrival counter
// (release add, counter polled, then the records read) it was a chain of
// four: 3.4 to 2.5 us a column of 60,000 rows, the panels of order 59,968 203 to
// 147 ms.
// Records and rows go to two buffer sets used by alternate columns: a CTA
// rewrites a set two columns later, after it has read every CTA's record of
// the column in between, which a CTA publishes only after a block barrier
// behind its reads of the set.  A wait is bounded: after BARRIER_WAIT_NS on
// the global timer the CTA records OBEM_ERR_TIMEOUT in flag[0] and gives up.
#define BARRIER_WAIT_NS 2000000000ull
#define PAN_MAXG 1024           // largest panel grid
// record: |pivot| bits << 33 | the row in its CTA << 23 | epoch
#define PAN_ROW_SHIFT 23
#define PAN_ROW_MASK 0x3ffu
#define PAN_EPOCH_MASK 0x7fffffu
static_assert(200 * 1024 / (4 * (LU_NB + 1)) <= PAN_ROW_MASK, "a CTA's rows fit the record");
// 64-bit words: records [2][PAN_MAXG], gdiag [2][LU_NB], candidate rows [2][PAN_MAXG][LU_NB]
#define PAN_WORDS (2 * PAN_MAXG + 2 * LU_NB + 2 * PAN_MAXG * LU_NB)
#define PAN_SCRATCH_FLOATS (2 * PAN_WORDS)
#define PAN_PLAN_FLOATS 260     // the row swaps' plan (1 + 4 LU_NB ints, padded to 16 bytes)

__device__ __forceinline__ unsigned long long gb_now()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned long long pan_ld(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void pan_st(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// a bounded wait's clock (t0: 0 before its first look, at the 64th poll): true
// when it ran out (flag[0] = OBEM_ERR_TIMEOUT)
__device__ __forceinline__ bool pan_late(unsigned it, unsigned long long &t0, int *flag)
{
    if ((it & 63u) != 0u) return false;
    if (t0 == 0ull) t0 = gb_now();
    if (gb_now() - t0 <= BARRIER_WAIT_NS) return false;
    atomicExch(flag, OBEM_ERR_TIMEOUT);
    return true;
}

// Called by one warp: waits until the G records carry the epoch and returns the
// largest candidate (in every lane) as |pivot| bits << 32 | ~row (ties to the
// lower row), 1 when there is none, 0 when the wait ran out.  CTA b's rows
// start at k + b R.
__device__ unsigned long long pan_wait_records(const unsigned long long *recs, int G, unsigned epoch, int k, int R,
                                               int *flag)
{
    const int lane = threadIdx.x & 31;
    unsigned long long t0 = 0ull;
    unsigned long long best = 1ull;
    for (int g0 = 0; g0 < G; g0 += 256) {
        unsigned long long v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = 0ull;
        for (unsigned it = 1;; ++it) {
            bool ok = true;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int t = g0 + 32 * q + lane;
                if (t < G && ((unsigned)v[q] & PAN_EPOCH_MASK) != epoch) v[q] = pan_ld(recs + t);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
                ok = ok && (g0 + 32 * q + lane >= G || ((unsigned)v[q] & PAN_EPOCH_MASK) == epoch);
            if (__all_sync(0xffffffffu, ok)) break;
            int late = 0;
            if (lane == 0) late = pan_late(it, t0, flag);
            if (__shfl_sync(0xffffffffu, late, 0)) return 0ull;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const unsigned m = (unsigned)(v[q] >> 33);
            const int row = k + (g0 + 32 * q + lane) * R + (int)((unsigned)(v[q] >> PAN_ROW_SHIFT) & PAN_ROW_MASK);
            const unsigned long long key = m ? (unsigned long long)m << 32 | (unsigned)~(unsigned)row : 1ull;
            best = key > best ? key : best;
        }
    }
    const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(best >> 32));
    const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(best >> 32) == hi ? (unsigned)best : 0u);
    return (unsigned long long)hi << 32 | lo;
}

// Failure-detection self-test: the blocks wait for a record that nothing
// publishes, so every wait runs out after BARRIER_WAIT_NS and records
// OBEM_ERR_TIMEOUT in flag[0] (flag[2..3]: the record).
__global__ void barrier_timeout_kernel(int *flag)
{
    pan_wait_records((const unsigned long long *)(flag + 2), 1, 1u, 0, 1, flag);
}

extern "C" int obem_selftest_wait_timeout(obem_ctx *c, obem_stream stream)
{
    if (!c) return OBEM_ERR_ARG;
    cudaStream_t s = (cudaStream_t)stream;
    int *flag = NULL;
    OBEM_CUDA(c, cudaMalloc((void **)&flag, sizeof(int) * 8));
    int h = 0;
    cudaError_t e = cudaMemsetAsync(flag, 0, sizeof(int) * 8, s);
    if (e == cudaSuccess) {
        barrier_timeout_kernel<<<2, 32, 0, s>>>(flag);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&h, flag, sizeof(int), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    cudaFree(flag);
    if (e != cudaSuccess) return obem_fail(c, OBEM_ERR_CUDA, "wait self-test: %s", cudaGetErrorString(e));
    if (h != OBEM_ERR_TIMEOUT) return obem_fail(c, OBEM_ERR_STATE, "wait self-test: status %d, expected a timeout", h);
    return OBEM_OK;
}

struct PanelArgs {
    float *A;
    int n, k, kb, rows_per_cta;
    int *piv;
    int *flag;          // [0] status
    // published (see the panel exchange): CTA b's candidate, |pivot| 0: none;
    // epoch << 32 | value of the candidate row's panel values and of the row
    // receiving the pivot, before the swap
    unsigned long long *rec;    // [2][PAN_MAXG]
    unsigned long long *crows;  // [2][PAN_MAXG][LU_NB]
    unsigned long long *gdiag;  // [2][LU_NB]
};

// best candidate over the CTA, in every thread: v = |a| (-1: none), r = its
// row, larger |a| first, ties to the lower row.  One CTA barrier; the warps'
// results go to the buffer set `par` (calls alternate the sets, so a set is
// rewritten only after the barriers of the call in between).
__device__ __forceinline__ void pan_reduce(float &v, int &r, unsigned (*sv)[8], unsigned (*sr)[8], int par)
{
    // non-negative floats order as their bits; +1 leaves 0 for "none"
    const unsigned kv = v < 0.f ? 0u : __float_as_uint(v) + 1u;
    const unsigned m = __reduce_max_sync(0xffffffffu, kv);
    const unsigned rm = __reduce_min_sync(0xffffffffu, kv == m ? (unsigned)r : 0xffffffffu);
    if ((threadIdx.x & 31) == 0) {
        sv[par][threadIdx.x >> 5] = m;
        sr[par][threadIdx.x >> 5] = rm;
    }
    __syncthreads();
    unsigned bm = sv[par][0], br = sr[par][0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
        const unsigned m2 = sv[par][w], r2 = sr[par][w];
        if (m2 > bm || (m2 == bm && r2 < br)) { bm = m2; br = r2; }
    }
    v = bm == 0u ? -1.f : __uint_as_float(bm - 1u);
    r = bm == 0u ? 0x7fffffff : (int)br;
}

// Warp 0 publishes the CTA's candidate for column col: its record, the
// candidate row bi and, from its owner, the row that receives the pivot (both
// up to date).  With j >= 0 the two rows' columns j + 2 .. kb - 1 are first
// brought up to date with the multipliers of column j (the rest of the CTA's
// rows are updated after the publication); j = -1: no update.
__device__ __forceinline__ void pan_publish(const PanelArgs &a, int col, int j, float bv, int bi, int r0, int rows,
                                            float *sp, int ld, const float *urow)
{
    const int lane = threadIdx.x & 31, kb = a.kb, b = blockIdx.x;
    const int par = col & 1;
    const int pr = a.k + col;
    const unsigned epoch = (unsigned)(pr + 1) & PAN_EPOCH_MASK;
    unsigned long long *crow = a.crows + ((size_t)par * PAN_MAXG + b) * LU_NB;
    unsigned long long *gd = a.gdiag + par * LU_NB;
    const bool has = bi != 0x7fffffff;
    const bool own = pr >= r0 && pr < r0 + rows;
    if (lane == 0)
        pan_st(a.rec + (size_t)par * PAN_MAXG + b,
               (has ? (unsigned long long)__float_as_uint(bv) << 33 | (unsigned long long)(unsigned)(bi - r0) << PAN_ROW_SHIFT
                    : 0ull) | epoch);
    const unsigned long long tag = (unsigned long long)epoch << 32;
    for (int c = lane; c < kb; c += 32) {
        if (has) {
            float *row = sp + (size_t)(bi - r0) * ld;
            float x = row[c];
            if (j >= 0 && c >= j + 2) {
                x = fmaf(-row[j], urow[c], x);
                row[c] = x;
            }
            pan_st(crow + c, tag | __float_as_uint(x));
            if (bi == pr) pan_st(gd + c, tag | __float_as_uint(x));
        }
        if (own && bi != pr) {
            float *row = sp + (size_t)(pr - r0) * ld;
            float x = row[c];
            if (j >= 0 && c >= j + 2) {
                x = fmaf(-row[j], urow[c], x);
                row[c] = x;
            }
            pan_st(gd + c, tag | __float_as_uint(x));
        }
    }
}

// Warp 0 fetches the pivot row (row p, candidate of CTA q) to urow and swaps:
// the pivot row to row pr, row pr's old values to row p, where they are the
// CTA's.  Returns false when the wait ran out.
__device__ __forceinline__ bool pan_fetch(const PanelArgs &a, int col, int p, int q, int r0, int rows, float *sp, int ld,
                                          float *urow)
{
    static_assert(LU_NB == 64, "two columns per lane");
    const int lane = threadIdx.x & 31, kb = a.kb;
    const int par = col & 1, pr = a.k + col;
    const unsigned epoch = (unsigned)(pr + 1) & PAN_EPOCH_MASK;
    const unsigned long long *cu = a.crows + ((size_t)par * PAN_MAXG + q) * LU_NB + lane;
    const unsigned long long *cg = a.gdiag + par * LU_NB + lane;
    const bool mine = p != pr && p >= r0 && p < r0 + rows;      // warp-uniform
    const bool h0 = lane < kb, h1 = lane + 32 < kb;
    const unsigned long long none = (unsigned long long)epoch << 32;
    unsigned long long u0 = 0ull, u1 = 0ull, g0 = 0ull, g1 = 0ull;
    if (!h0) u0 = g0 = none;
    if (!h1) u1 = g1 = none;
    if (!mine) g0 = g1 = none;
    unsigned long long t0 = 0ull;
    for (unsigned it = 1;; ++it) {
        if ((unsigned)(u0 >> 32) != epoch) u0 = pan_ld(cu);
        if ((unsigned)(u1 >> 32) != epoch) u1 = pan_ld(cu + 32);
        if ((unsigned)(g0 >> 32) != epoch) g0 = pan_ld(cg);
        if ((unsigned)(g1 >> 32) != epoch) g1 = pan_ld(cg + 32);
        const bool ok = (unsigned)(u0 >> 32) == epoch && (unsigned)(u1 >> 32) == epoch &&
                        (unsigned)(g0 >> 32) == epoch && (unsigned)(g1 >> 32) == epoch;
        if (__all_sync(0xffffffffu, ok)) break;
        int late = 0;
        if (lane == 0) late = pan_late(it, t0, a.flag);
        if (__shfl_sync(0xffffffffu, late, 0)) return false;
    }
    const float x0 = __uint_as_float((unsigned)u0), x1 = __uint_as_float((unsigned)u1);
    if (h0) urow[lane] = x0;
    if (h1) urow[lane + 32] = x1;
    if (pr >= r0 && pr < r0 + rows) {
        float *row = sp + (size_t)(pr - r0) * ld;
        if (h0) row[lane] = x0;
        if (h1) row[lane + 32] = x1;
    }
    if (mine) {
        float *row = sp + (size_t)(p - r0) * ld;
        if (h0) row[lane] = __uint_as_float((unsigned)g0);
        if (h1) row[lane + 32] = __uint_as_float((unsigned)g1);
    }
    return true;
}

// Panel factorisation of A[k:n, k:k+kb] with partial pivoting.  CTA b owns
// rows k + b*R .. k + (b+1)*R - 1 of the panel in shared memory.  Per column
// j: warp 0 waits for every CTA's candidate of column j, takes the largest
// (the same pivot in every CTA), fetches the pivot row and swaps, while the
// other warps finish column j - 1's update of the own rows (never the rows of
// the swap: the CTA's candidate and the row that receives the pivot); then
// the block forms the multipliers, updates column j + 1 of the own rows and
// finds the CTA's candidate for column j + 1, which warp 0 publishes.
__global__ void __launch_bounds__(256)
panel_kernel(PanelArgs a)
{
    extern __shared__ float sp[];            // [R][kb + 1] (padded against bank conflicts)
    __shared__ unsigned sv[2][8], sr[2][8];
    __shared__ int s_stop;                   // 0, OBEM_ERR_SINGULAR or OBEM_ERR_TIMEOUT
    __shared__ float s_urow[2][LU_NB];       // pivot rows of alternate columns
    const int R = a.rows_per_cta, kb = a.kb, n = a.n, k = a.k;
    const int ld = kb + 1;
    const int b = blockIdx.x, G = gridDim.x;
    const int r0 = k + b * R;
    const int rows = max(0, min(R, n - r0));
    const int tid = threadIdx.x, warp = tid >> 5;
    // a factorisation that already failed (zero pivot, a wait that ran out)
    // stops here instead of waiting again in every later panel
    if (*(volatile const int *)a.flag != 0) return;
    {
        // 8 loads in flight per thread before the shared-memory stores
        const int tot = rows * kb;
        for (int t0 = 0; t0 < tot; t0 += 8 * 256) {
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int t = t0 + u * 256 + tid;
                v[u] = t < tot ? a.A[(size_t)(r0 + t / kb) * n + k + t % kb] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
                const int t = t0 + u * 256 + tid;
                if (t < tot) sp[(t / kb) * ld + t % kb] = v[u];
            }
        }
    }
    __syncthreads();
    {
        // candidate of column 0
        float bv = -1.f;
        int bi = 0x7fffffff;
        for (int r = tid; r < rows; r += blockDim.x) {
            const float v = fabsf(sp[r * ld]);
            if (v > bv) { bv = v; bi = r0 + r; }
        }
        pan_reduce(bv, bi, sv, sr, 0);
        if (warp == 0) pan_publish(a, 0, -1, bv, bi, r0, rows, sp, ld, s_urow[0]);
    }
    for (int j = 0; j < kb; ++j) {
        const int par = j & 1;
        const int pr = k + j;                     // row receiving the pivot
        float *urow = s_urow[par];
        if (warp == 0) {
            const unsigned long long key = pan_wait_records(a.rec + (size_t)par * PAN_MAXG, G,
                                                            (unsigned)(pr + 1) & PAN_EPOCH_MASK, k, R, a.flag);
            const float v = __uint_as_float((unsigned)(key >> 32));
            const int p = (int)(~(unsigned)(key & 0xffffffffu));
            int stop = 0;
            if (key == 0ull) stop = OBEM_ERR_TIMEOUT;
            else if (key == 1ull || !(v > 0.f)) stop = OBEM_ERR_SINGULAR;
            else if (!pan_fetch(a, j, p, (p - k) / R, r0, rows, sp, ld, urow)) stop = OBEM_ERR_TIMEOUT;
            if (tid == 0) {
                s_stop = stop;
                if (b == 0 && stop == 0) a.piv[pr] = p;
            }
        }
        __syncthreads();
        if (s_stop) {
            // singular: every CTA stops here; the panel's remaining pivots
            // are set to no swap
            if (s_stop == OBEM_ERR_SINGULAR) {
                if (tid == 0) atomicCAS(a.flag, 0, OBEM_ERR_SINGULAR);
                if (b == 0)
                    for (int jj = j + tid; jj < kb; jj += blockDim.x) a.piv[k + jj] = k + jj;
            }
            return;
        }
        const float inv = 1.0f / urow[j];
        if (j + 1 == kb) {
            for (int r = tid; r < rows; r += blockDim.x)
                if (r0 + r > pr) sp[r * ld + j] *= inv;
            break;
        }
        // multipliers of column j, column j + 1 of the own rows, candidate
        const float u1 = urow[j + 1];
        float bv = -1.f;
        int bi = 0x7fffffff;
        for (int r = tid; r < rows; r += blockDim.x) {
            const int gr = r0 + r;
            if (gr <= pr) continue;
            const float l = sp[r * ld + j] * inv;
            sp[r * ld + j] = l;
            const float x = fmaf(-l, u1, sp[r * ld + j + 1]);
            sp[r * ld + j + 1] = x;
            const float ax = fabsf(x);
            if (ax > bv) { bv = ax; bi = gr; }
        }
        pan_reduce(bv, bi, sv, sr, (j + 1) & 1);
        if (warp == 0) {
            pan_publish(a, j + 1, j, bv, bi, r0, rows, sp, ld, urow);
        } else {
            // the other rows' columns j + 2 .. kb - 1, while warp 0 waits
            // for the next column and swaps (the barrier after that comes
            // before any of them is read)
            const int nx = pr + 1;
            for (int r = tid - 32; r < rows; r += (int)blockDim.x - 32) {
                const int gr = r0 + r;
                if (gr <= pr || gr == bi || gr == nx) continue;
                float *row = sp + (size_t)r * ld;
                const float l = row[j];
#pragma unroll 8
                for (int c = j + 2; c < kb; ++c) row[c] = fmaf(-l, urow[c], row[c]);
            }
        }
    }
    __syncthreads();
    for (int t = tid; t < rows * kb; t += blockDim.x) {
        int r = t / kb, c = t % kb;
        a.A[(size_t)(r0 + r) * n + k + c] = sp[r * ld + c];
    }
}

// The panel's kb row swaps (piv[k .. k + kb)) applied to the columns outside
// the panel, unless the factorisation's status (flag[0]) records a failure,
// in three launches: laswp_plan_kernel lists the rows the swaps touch (the kb
// panel rows and the distinct pivot rows below the panel, at most 2 kb) and,
// for each, the touched row whose content it receives (the swaps undone in
// reverse order, independently per row); laswp_gather_kernel copies the
// touched rows whole into a scratch block, laswp_scatter_kernel writes each
// receiving row from it.  Whole-row copies stream at the HBM rate; a
// single-pass permutation in shared memory (every block holding a column
// slice of all touched rows) ran at a fifth of it.
#define LS_PLAN_INTS (1 + 4 * LU_NB)        // m, rows[2 LU_NB], src[2 LU_NB]
__global__ void __launch_bounds__(LU_NB) laswp_plan_kernel(int k, int kb, const int *piv, int *flag, int *plan)
{
    // a panel that stopped (zero pivot, a wait that ran out) may have left
    // pivots unwritten: no swaps then
    if (*(volatile const int *)flag != 0) {
        if (threadIdx.x == 0) plan[0] = 0;
        return;
    }
    __shared__ int s_piv[LU_NB], s_pos[LU_NB], s_row[2 * LU_NB];
    __shared__ unsigned s_first[LU_NB / 32];
    const int tid = threadIdx.x, lane = tid & 31;
    // the position of every swap's pivot row among the touched rows: panel
    // rows first, then the pivot rows below the panel by first appearance
    const int p = tid < kb ? piv[k + tid] : -1;
    s_piv[tid] = p;
    __syncthreads();
    // the first swap with the same pivot row (all 64 reads in flight)
    int f = tid;
#pragma unroll
    for (int q = LU_NB - 1; q >= 0; --q)
        if (q < tid && s_piv[q] == p) f = q;
    const bool first = tid < kb && p >= k + kb && f == tid;
    const unsigned bal = __ballot_sync(0xffffffffu, first);
    if (lane == 0) s_first[tid >> 5] = bal;
    __syncthreads();
    const unsigned long long mask = (unsigned long long)s_first[0] | ((unsigned long long)s_first[1] << 32);
    if (tid < kb) {
        s_pos[tid] = p < k + kb ? p - k : kb + __popcll(mask & ((1ull << f) - 1ull));
        s_row[tid] = k + tid;
    }
    if (first) s_row[kb + __popcll(mask & ((1ull << tid) - 1ull))] = p;
    const int m = kb + __popcll(mask);
    __syncthreads();
    // the touched row whose content ends in touched row t: the swaps
    // (position q <-> s_pos[q], q = 0 .. kb-1, in order) undone in reverse
    for (int t = tid; t < m; t += blockDim.x) {
        int j = t;
#pragma unroll
        for (int q = LU_NB - 1; q >= 0; --q) {
            const int pq = q < kb ? s_pos[q] : q;
            j = j == q ? pq : (j == pq ? q : j);
        }
        plan[1 + t] = s_row[t];
        plan[1 + 2 * LU_NB + t] = j;
    }
    if (tid == 0) plan[0] = m;
}

// S[q][:] = A[rows[q]][:] for the touched rows q < m (grid y: q)
__global__ void laswp_gather_kernel(const float *__restrict__ A, int n, const int *plan, float *__restrict__ S)
{
    const int q = blockIdx.y;
    if (q >= plan[0]) return;
    const float *a = A + (size_t)plan[1 + q] * n;
    float *d = S + (size_t)q * n;
    const int stride = gridDim.x * blockDim.x;
    if ((n & 3) == 0) {
        for (int c4 = blockIdx.x * blockDim.x + threadIdx.x; c4 < n / 4; c4 += stride)
            ((float4 *)d)[c4] = __ldcs((const float4 *)a + c4);
    } else {
        for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += stride) d[c] = __ldcs(a + c);
    }
}

// A[rows[t]][c] = S[src[t]][c] for the touched rows t < m that receive
// another row, outside the panel's own columns [k, k + kb) (the panel kernel
// already swapped those)
__global__ void laswp_scatter_kernel(float *__restrict__ A, int n, int k, int kb, const int *plan,
                                     const float *__restrict__ S)
{
    const int t = blockIdx.y;
    if (t >= plan[0]) return;
    const int sq = plan[1 + 2 * LU_NB + t];
    if (sq == t) return;
    float *d = A + (size_t)plan[1 + t] * n;
    const float *a = S + (size_t)sq * n;
    const int stride = gridDim.x * blockDim.x;
    if ((n & 3) == 0 && (k & 3) == 0 && ((k + kb) & 3) == 0) {
        for (int c4 = blockIdx.x * blockDim.x + threadIdx.x; c4 < n / 4; c4 += stride)
            if (4 * c4 < k || 4 * c4 >= k + kb) ((float4 *)d)[c4] = __ldcs((const float4 *)a + c4);
    } else {
        for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < n; c += stride)
            if (c < k || c >= k + kb) d[c] = __ldcs(a + c);
    }
}

// U12 = L11^-1 A12 with L11 unit lower triangular (kb x kb); a CTA of
// TRSM_COLS threads owns TRSM_COLS columns, held in shared memory
#define TRSM_COLS 64
__global__ void trsm_kernel(float *A, int n, int k, int kb)
{
    __shared__ float L[LU_NB][LU_NB + 1];
    __shared__ float X[LU_NB][TRSM_COLS];
    for (int t = threadIdx.x; t < kb * kb; t += blockDim.x) {
        int r = t / kb, c = t % kb;
        L[r][c] = A[(size_t)(k + r) * n + k + c];
    }
    const int c = k + kb + blockIdx.x * TRSM_COLS + threadIdx.x;
    const bool act = c < n;
    for (int r = 0; r < kb; ++r) X[r][threadIdx.x] = act ? A[(size_t)(k + r) * n + c] : 0.f;
    __syncthreads();
    for (int q = 0; q < kb; ++q) {
        const float xq = X[q][threadIdx.x];
        for (int r = q + 1; r < kb; ++r) X[r][threadIdx.x] = fmaf(-L[r][q], xq, X[r][threadIdx.x]);
    }
    if (act)
        for (int r = 0; r < kb; ++r) A[(size_t)(k + r) * n + c] = X[r][threadIdx.x];
}

// T[r][c] = M[(r0 + r) * n + c0 + c] for r, c < kb (kb <= LU_NB), loaded by
// blockDim.x (a multiple of 64) threads with 16 loads in flight per thread
// before the shared-memory stores (the loads of a few-CTA kernel are
// latency-bound otherwise)
__device__ __forceinline__ void load_block(float (*T)[LU_NB + 1], const float *M, int n, int r0, int c0, int kb,
                                           bool transpose)
{
    const int c = threadIdx.x & 63, rstep = blockDim.x >> 6;
    for (int rb = threadIdx.x >> 6; rb < kb; rb += 16 * rstep) {
        float v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int r = rb + i * rstep;
            v[i] = (r < kb && c < kb) ? M[(size_t)(r0 + r) * n + c0 + c] : 0.f;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int r = rb + i * rstep;
            if (r < kb && c < kb) {
                if (transpose) T[c][r] = v[i];
                else T[r][c] = v[i];
            }
        }
    }
}

// X = L^-1 X for the unit lower triangular block L = A[r0:r0+m, r0:r0+m]
// (m <= M) and X = A[r0:r0+m, c0:c0+nc]: one thread per column of X, the
// block's columns staged through shared memory (coalesced loads and stores)
// and each column's M values held in registers; L transposed in shared
// memory (zero outside its strict lower triangle; a column of L read as
// broadcast float4).  For q = 0 .. M-2, x[r] -= L[r][q] x[q] for every
// r > q, in FP32 (64 rows at a time in registers, each row's updates still
// in the order of q).  M = 64 or 128: the leaves of the recursive TRSM (a 128-row
// leaf replaces two 64-row leaves and the BF16 tensor-core update between
// them).
#define TRSM_LEAF 128
#define TRSM_LEAF_THREADS 128
__device__ __forceinline__ unsigned tl_smem(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
template <int M>
constexpr size_t trsm_leaf_smem() { return sizeof(float) * (size_t)M * (M + 4 + TRSM_LEAF_THREADS); }
template <int M>
__global__ void __launch_bounds__(TRSM_LEAF_THREADS)
trsm_leaf_kernel(float *A, int n, int r0, int m, int c0, int nc)
{
    constexpr int LP = M + 4;                    // pitch (the transposing stores spread over 8 banks)
    extern __shared__ float4 tl_L4[];            // [M][LP / 4]: row q = column q of L
    float *Lt = (float *)tl_L4;
    float *Xs = Lt + M * LP;                     // [M][TRSM_LEAF_THREADS]
    const int tid = threadIdx.x;
    const int col = blockIdx.x * TRSM_LEAF_THREADS + tid;
    const bool live = col < nc;
    float *x = A + (size_t)r0 * n + c0 + col;
    // every load of the block in flight at once: 4-byte asynchronous copies
    // into shared memory (a zero-size source writes a zero), lanes on
    // consecutive columns (coalesced; with lanes on consecutive rows of L, 32
    // sectors a load, the 128-row leaf took 35.7 us a call at order 59,968, now 33.8).
    for (int t = tid; t < M * M; t += blockDim.x) {
        const int r = t / M, q = t % M;
        const bool in = r < m && q < r;
        const float *src = in ? A + (size_t)(r0 + r) * n + r0 + q : A;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(tl_smem(&Lt[q * LP + r])), "l"(src),
                     "r"(in ? 4 : 0)
                     : "memory");
    }
    for (int r = 0; r < M; ++r) {
        const bool in = live && r < m;
        const float *src = in ? x + (size_t)r * n : A;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(tl_smem(&Xs[r * TRSM_LEAF_THREADS + tid])),
                     "l"(src), "r"(in ? 4 : 0)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    // 64 rows at a time in registers: the rows of the earlier blocks (already
    // solved, back in shared memory) first, then the block's own triangle
#pragma unroll
    for (int h = 0; h < M / 64; ++h) {
        float v[64];
#pragma unroll
        for (int r = 0; r < 64; ++r) v[r] = Xs[(64 * h + r) * TRSM_LEAF_THREADS + tid];
#pragma unroll 4
        for (int q = 0; q < 64 * h; ++q) {
            const float xq = Xs[q * TRSM_LEAF_THREADS + tid];
#pragma unroll
            for (int r4 = 0; r4 < 64; r4 += 4) {
                const float4 l = tl_L4[q * (LP / 4) + (64 * h + r4) / 4];
                v[r4] = fmaf(-l.x, xq, v[r4]);
                v[r4 + 1] = fmaf(-l.y, xq, v[r4 + 1]);
                v[r4 + 2] = fmaf(-l.z, xq, v[r4 + 2]);
                v[r4 + 3] = fmaf(-l.w, xq, v[r4 + 3]);
            }
        }
#pragma unroll
        for (int q = 0; q < 63; ++q) {
            const float xq = v[q];
#pragma unroll
            for (int r4 = (q + 1) & ~3; r4 < 64; r4 += 4) {
                const float4 l = tl_L4[(64 * h + q) * (LP / 4) + (64 * h + r4) / 4];
                if (r4 > q) v[r4] = fmaf(-l.x, xq, v[r4]);
                if (r4 + 1 > q) v[r4 + 1] = fmaf(-l.y, xq, v[r4 + 1]);
                if (r4 + 2 > q) v[r4 + 2] = fmaf(-l.z, xq, v[r4 + 2]);
                if (r4 + 3 > q) v[r4 + 3] = fmaf(-l.w, xq, v[r4 + 3]);
            }
        }
#pragma unroll
        for (int r = 0; r < 64; ++r) Xs[(64 * h + r) * TRSM_LEAF_THREADS + tid] = v[r];
    }
    if (!live) return;
#pragma unroll 8
    for (int r = 0; r < m; ++r) x[(size_t)r * n] = Xs[r * TRSM_LEAF_THREADS + tid];
}

// The same leaf solve for narrow X (few blocks: the latency of one block
// decides): one warp per 4 columns, lane l holding rows l, l + 32, ... of
// them in registers, L row-major in shared memory (padded: the column reads
// are conflict-free), x[q] broadcast by a shuffle at step q.  Same updates
// in the same order as trsm_leaf_kernel (the results are identical).
#define TL2_C 4
#define TL2_W 8
#define TL2_BC (TL2_C * TL2_W)
template <int M>
constexpr size_t trsm_leaf2_smem() { return sizeof(float) * ((size_t)M * (M + 1) + (size_t)M * (TL2_BC + 1)); }
template <int M>
__global__ void __launch_bounds__(TL2_W * 32)
trsm_leaf2_kernel(float *A, int n, int r0, int m, int c0, int nc)
{
    constexpr int RL = M / 32;
    extern __shared__ float tl2_s[];
    float *Ls = tl2_s;                    // [M][M + 1]: L row-major, padded (column reads conflict-free)
    float *Xs = tl2_s + M * (M + 1);      // [M][TL2_BC + 1]
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int cb = blockIdx.x * TL2_BC;
    for (int t = tid; t < M * M; t += blockDim.x) {
        const int r = t / M, q = t % M;           // coalesced over q
        const bool in = r < m && q < r;
        const float *src = in ? A + (size_t)(r0 + r) * n + r0 + q : A;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(tl_smem(&Ls[r * (M + 1) + q])), "l"(src),
                     "r"(in ? 4 : 0)
                     : "memory");
    }
    for (int e = tid; e < M * TL2_BC; e += blockDim.x) {
        const int r = e / TL2_BC, c = e % TL2_BC;
        const bool in = r < m && cb + c < nc;
        const float *src = in ? A + (size_t)(r0 + r) * n + c0 + cb + c : A;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(tl_smem(&Xs[r * (TL2_BC + 1) + c])),
                     "l"(src), "r"(in ? 4 : 0)
                     : "memory");
    }
    asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    float v[TL2_C][RL];
#pragma unroll
    for (int j = 0; j < TL2_C; ++j)
#pragma unroll
        for (int i = 0; i < RL; ++i) v[j][i] = Xs[(32 * i + lane) * (TL2_BC + 1) + warp * TL2_C + j];
    // (four steps unrolled: 127 were 50 KB of code that every block waited for, 15.0
    // us a call against 13.3)
#pragma unroll
    for (int b = 0; b < RL; ++b)
#pragma unroll 4
        for (int e = 0; e < 32; ++e) {
            const int q = 32 * b + e;
            float lq[RL];
#pragma unroll
            for (int i = b; i < RL; ++i) lq[i] = Ls[(32 * i + lane) * (M + 1) + q];
#pragma unroll
            for (int j = 0; j < TL2_C; ++j) {
                const float xq = __shfl_sync(0xffffffffu, v[j][b], e);
                // (L's upper triangle is stored as zeros; a row's own step must not touch it)
#pragma unroll
                for (int i = b; i < RL; ++i)
                    if (i > b || lane > e) v[j][i] = fmaf(-lq[i], xq, v[j][i]);
            }
        }
#pragma unroll
    for (int j = 0; j < TL2_C; ++j)
#pragma unroll
        for (int i = 0; i < RL; ++i) Xs[(32 * i + lane) * (TL2_BC + 1) + warp * TL2_C + j] = v[j][i];
    __syncthreads();
    for (int e = tid; e < M * TL2_BC; e += blockDim.x) {
        const int r = e / TL2_BC, c = e % TL2_BC;
        if (r < m && cb + c < nc) A[(size_t)(r0 + r) * n + c0 + cb + c] = Xs[r * (TL2_BC + 1) + c];
    }
}

// ------------------------------------------------------------------ solve kernels
// b_i = rowscale_i * (V_group or free density) + drhs_i  (drhs unscaled input)
__global__ void rhs_kernel(const int *kind, const int *group, const double *gv, const float *sigma_free,
                           const float *drhs, const double *rowscale, double *b, int n)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double v = 0.0;
    if (kind[i] == OBEM_CELL_ELECTRODE) v = gv[group[i]];
    else if (sigma_free) v = (double)sigma_free[i];
    if (drhs) v += (double)drhs[i];
    b[i] = v * rowscale[i];
}

// r = b - A x (FP64 accumulation over the FP32 matrix), one warp per row
// x = xh + xl in two floats (xl: the rounding remainder of xh, so that
// |x - xh - xl| <= 2^-48 |x|)
__global__ void split_kernel(const double *x, float *xh, float *xl, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float h = (float)x[i];
    xh[i] = h;
    xl[i] = (float)(x[i] - (double)h);
}

// r = b - A x in FP64 without FP64 products: a warp per row; each product
// a xh is split exactly (FMA) into its float value p and error e, p goes to
// a per-lane two-sum (s, c) and e + a xl to c; the lanes' s + c are added
// in FP64.  The result differs from the FP64 dot product by a few units of
// 2^-48 of sum |a x|.
__device__ __forceinline__ void df_acc(float &s, float &c, float a, float h, float l)
{
    const float p = __fmul_rn(a, h);
    const float e = __fmaf_rn(a, h, -p);
    const float t = __fadd_rn(s, p);
    const float z = __fsub_rn(t, s);
    const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));
    c = __fadd_rn(c, __fadd_rn(err, __fmaf_rn(a, l, e)));
    s = t;
}
__global__ void __launch_bounds__(256) residual_kernel(const float *A, const float *xh, const float *xl,
                                                       const double *b, double *r, int n)
{
    const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (row >= n) return;
    const float *a = A + (size_t)row * n;
    float s = 0.f, c = 0.f;
    int j = lane;
    for (; j + 32 * 7 < n; j += 32 * 8) {
        float av[8], hv[8], lv[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            av[u] = __ldcs(a + j + 32 * u);
            hv[u] = xh[j + 32 * u];
            lv[u] = xl[j + 32 * u];
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) df_acc(s, c, av[u], hv[u], lv[u]);
    }
    for (; j < n; j += 32) df_acc(s, c, a[j], xh[j], xl[j]);
    double v = (double)s + (double)c;
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) r[row] = b[row] - v;
}
// out[q] = max |r|, |x|, |b|: one block of 1024, the magnitudes compared as
// integers (a single SM's FP64 pipe took 155 us at 60k entries; a NaN counts as
// 0, as fmax does)
__device__ __forceinline__ unsigned long long abs_bits(double v)
{
    const unsigned long long k = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
    return k > 0x7ff0000000000000ull ? 0ull : k;
}
__global__ void __launch_bounds__(1024) norms_kernel(const double *r, const double *x, const double *b, int n,
                                                     double *out)
{
    __shared__ unsigned long long s[3][32];
    unsigned long long m[3] = {0ull, 0ull, 0ull};
#pragma unroll 4
    for (int i = threadIdx.x; i < n; i += 1024) {
        const unsigned long long a0 = abs_bits(r[i]), a1 = abs_bits(x[i]), a2 = abs_bits(b[i]);
        m[0] = a0 > m[0] ? a0 : m[0];
        m[1] = a1 > m[1] ? a1 : m[1];
        m[2] = a2 > m[2] ? a2 : m[2];
    }
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        for (int o = 16; o; o >>= 1) {
            const unsigned long long v = __shfl_xor_sync(0xffffffffu, m[q], o);
            m[q] = v > m[q] ? v : m[q];
        }
        if ((threadIdx.x & 31) == 0) s[q][threadIdx.x >> 5] = m[q];
    }
    __syncthreads();
    if (threadIdx.x < 3) {
        unsigned long long v = s[threadIdx.x][0];
        for (int w = 1; w < 32; ++w) v = s[threadIdx.x][w] > v ? s[threadIdx.x][w] : v;
        out[threadIdx.x] = __longlong_as_double((long long)v);
    }
}

// y = P r / sc in FP32 (sc = max |r|): the factorisation's row swaps as one
// gather, y[i] = r[perm[i]] / sc
__global__ void permute_kernel(const double *r, float *y, const int *perm, int n, const double *norms)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double sc = norms[0] > 0 ? norms[0] : 1.0;
    y[i] = (float)(r[perm[i]] / sc);
}



__global__ void axpy_kernel(double *x, const float *d, const double *norms, int n)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double sc = norms[0] > 0 ? norms[0] : 1.0;
    x[i] += (double)d[i] * sc;
}

__global__ void to_float_kernel(const double *x, float *a, float *b, int n)
{
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    float v = (float)x[i];
    a[i] = v;
    if (b) b[i] = v;
}

// ------------------------------------------------------------------ one-launch triangular solves
// Forward (unit lower L) or backward (upper U) substitution with the factors
// in one launch.  Block row i of TS_R rows is taken by the thread block that
// draws ticket i (in dependency order: i = 0 is the first block row of L,
// the last of U), so every block row it depends on belongs to a thread block
// that started before it, whatever the scheduling.  A thread block runs over
// the solved blocks of y in dependency order, then multiplies its right-hand
// side, less the solved part, by the inverse of its diagonal block (computed
// once after the factorisation) and publishes its y values.
//
// Bound: at 60k cells the factor's 7.2 GB (1.06 ms) and a chain of 469 steps.
// A published value carries the launch's epoch in its upper half, so a step
// waits for the data itself (one round trip to L2, no flag before it and no
// fence after it); the block's matrix entries are in flight before the wait;
// one warp polls, the more rarely the farther its block row is from its turn
// (every warp polling flags, the matrix read after them: 4.05 ms; now 1.45 ms,
// and 0.515 to 0.17 ms at 11,008 cells).
// A wait is bounded (TS_WAIT_NS): one that runs out records OBEM_ERR_TIMEOUT
// and the block waits no more, so that the launch always ends.
#define TS_WAIT_NS 2000000000ull
#define TS_TH 256
#define TS_SMEM (sizeof(float) * TS_R * TS_R)
#define TS_INV_SMEM (sizeof(float) * 2 * TS_R * (TS_R + 1))

__device__ __forceinline__ unsigned long long ts_now()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ unsigned long long ts_ld(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void ts_st(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

struct TsArgs {
    const float *LU;
    const float *dinv;  // inverses of the diagonal blocks (inv_diag_kernel)
    float *y;           // right-hand side in, solution out
    unsigned long long *z;   // [n] published values: launch epoch << 32 | y
    int n, lower;
    unsigned epoch;
    int *ticket;        // zero before the launch
    int *err;
};

// Inverses of the diagonal blocks (TS_R x TS_R) of the unit lower factor L
// (blockIdx.y = 0) and of the upper factor U (blockIdx.y = 1): thread c
// solves for column c of the inverse by substitution; rows and columns past
// the matrix are zero.
#define TS_LD (TS_R + 1)
__global__ void __launch_bounds__(TS_R) inv_diag_kernel(const float *LU, int n, float *dinv)
{
    extern __shared__ float ts_sm[];
    float *T = ts_sm, *X = ts_sm + TS_R * TS_LD;
    const int blk = blockIdx.x, upper = blockIdx.y, c = threadIdx.x;
    const int r0 = blk * TS_R, rows = min(TS_R, n - r0);
    for (int e = c; e < TS_R * TS_R; e += TS_R) {
        const int i = e / TS_R, k = e % TS_R;
        T[i * TS_LD + k] = (i < rows && k < rows) ? LU[(size_t)(r0 + i) * n + r0 + k] : 0.f;
    }
    __syncthreads();
    if (!upper) {
        for (int i = 0; i < TS_R; ++i) {
            float v = (i == c && i < rows) ? 1.f : 0.f;
            for (int k = c; k < i; ++k) v = fmaf(-T[i * TS_LD + k], X[k * TS_LD + c], v);
            X[i * TS_LD + c] = (i < rows && c < rows) ? v : 0.f;
        }
    } else {
        for (int i = TS_R - 1; i >= 0; --i) {
            float v = (i == c && i < rows) ? 1.f : 0.f;
            for (int k = i + 1; k <= c; ++k) v = fmaf(-T[i * TS_LD + k], X[k * TS_LD + c], v);
            X[i * TS_LD + c] = (i < rows && c < rows) ? v / T[i * TS_LD + i] : 0.f;
        }
    }
    __syncthreads();
    float *D = dinv + (size_t)(2 * blk + upper) * TS_R * TS_R;
    for (int e = c; e < TS_R * TS_R; e += TS_R) D[e] = X[(e / TS_R) * TS_LD + e % TS_R];
}

// Inverse of a diagonal block in shared memory, column c of row r at c ^
// ts_swz(r, c): the two halves of 16 rows are read without bank conflicts
__device__ __forceinline__ int ts_swz(int r, int c) { return c ^ ((r & 15) | ((c >> 6) << 4)); }
__device__ __forceinline__ void ts_load_inv(const TsArgs &a, int blk, int upper, float *D)
{
    const float *g = a.dinv + (size_t)(2 * blk + upper) * TS_R * TS_R;
    for (int e = threadIdx.x; e < TS_R * TS_R; e += TS_TH) {
        const int r = e / TS_R;
        D[r * TS_R + ts_swz(r, e % TS_R)] = g[e];
    }
}

// Warp 0: the values of block [c0, c0 + cols) into zs once they carry the
// launch's epoch; `behind`: block rows between this one and its turn.  `gave`:
// a wait ran out before (then nothing is waited for).
__device__ __forceinline__ void ts_wait(const TsArgs &a, int c0, int cols, int behind, float *zs, bool &gave)
{
    const int lane = threadIdx.x & 31;
    const unsigned long long t0 = ts_now();
    for (unsigned it = 0;; ++it) {
        unsigned long long v[TS_R / 32];
        bool ok = true;
#pragma unroll
        for (int q = 0; q < TS_R / 32; ++q) {
            const int c = lane + 32 * q;
            v[q] = c < cols ? ts_ld(a.z + c0 + c) : (unsigned long long)a.epoch << 32;
            ok = ok && (unsigned)(v[q] >> 32) == a.epoch;
        }
        const bool all = __all_sync(0xffffffffu, ok);
        if (!all && !gave && (it & 63u) == 63u && ts_now() - t0 > TS_WAIT_NS) {
            gave = true;
            if (lane == 0) atomicExch(a.err, OBEM_ERR_TIMEOUT);
        }
        gave = __shfl_sync(0xffffffffu, (int)gave, 0) != 0;
        if (all || gave) {
#pragma unroll
            for (int q = 0; q < TS_R / 32; ++q)
                zs[lane + 32 * q] = lane + 32 * q < cols ? __uint_as_float((unsigned)v[q]) : 0.f;
            return;
        }
        if (behind > 1) __nanosleep(behind < 32 ? 32u * behind : 1000u);
    }
}

// the block's solution: its inverse (trans: transposed) times s_b; thread
// (row, half) = (tid / 2, tid % 2).  s_b: entries 0..63, then 64..127 from 80 on
__device__ __forceinline__ void ts_publish(const TsArgs &a, const float *D, const float *s_b, bool trans, int r0,
                                           int rows)
{
    const int row = threadIdx.x >> 1, half = threadIdx.x & 1;
    const float *sb = s_b + 80 * half;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    for (int k = 0; k < 64; k += 4)
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = 64 * half + k + u;
            v[u] = fmaf(trans ? D[c * TS_R + ts_swz(c, row)] : D[row * TS_R + ts_swz(row, c)], sb[k + u], v[u]);
        }
    float t = (v[0] + v[1]) + (v[2] + v[3]);
    t += __shfl_xor_sync(0xffffffffu, t, 1);
    if (half == 0 && row < rows) {
        ts_st(a.z + r0 + row, (unsigned long long)a.epoch << 32 | __float_as_uint(t));
        a.y[r0 + row] = t;
    }
}

__global__ void __launch_bounds__(TS_TH) trsv_chain_kernel(TsArgs a)
{
    extern __shared__ float ts_sm[];         // [TS_R][TS_R] inverse of the diagonal block
    __shared__ float s_b[144], s_z[2][TS_R];
    __shared__ int s_t;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    constexpr int RW = TS_R / 8;             // rows per warp
    const int n = a.n, nbk = (n + TS_R - 1) / TS_R;
    if (tid == 0) s_t = atomicAdd(a.ticket, 1);
    __syncthreads();
    const int t = s_t;
    const int blk = a.lower ? t : nbk - 1 - t;
    const int r0 = blk * TS_R, rows = min(TS_R, n - r0);
    ts_load_inv(a, blk, a.lower ? 0 : 1, ts_sm);
    float acc[RW];
#pragma unroll
    for (int r = 0; r < RW; ++r) acc[r] = 0.f;
    // lane's row after the sum over the lanes, and its right-hand side
    const int mine = RW * w + (lane >> 1);
    const float rhs = mine < rows ? a.y[r0 + mine] : 0.f;
    bool gave = false;
    for (int st = 0; st < t; ++st) {
        const int j = a.lower ? st : nbk - 1 - st;
        const int c0 = j * TS_R, cols = min(TS_R, n - c0);
        float l[RW][4];
#pragma unroll
        for (int r = 0; r < RW; ++r) {
            const int row = RW * w + r;
            const float *arow = a.LU + (size_t)(r0 + (row < rows ? row : 0)) * n + c0;
#pragma unroll
            for (int q = 0; q < 4; ++q) l[r][q] = lane + 32 * q < cols ? arow[lane + 32 * q] : 0.f;
        }
        float *z = s_z[st & 1];
        if (w == 0) ts_wait(a, c0, cols, t - st, z, gave);
        __syncthreads();
        float zz[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) zz[q] = z[lane + 32 * q];
#pragma unroll
        for (int r = 0; r < RW; ++r)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[r] = fmaf(l[r][q], zz[q], acc[r]);
    }
    // sums over the lanes: each step halves the rows a lane holds; lanes 2 r,
    // 2 r + 1 end with row r
    int o = 16;
#pragma unroll
    for (int k = RW / 2; k > 0; k >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int r = 0; r < k; ++r) {
            const float send = up ? acc[r] : acc[r + k], keep = up ? acc[r + k] : acc[r];
            acc[r] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    const float sum = acc[0] + __shfl_xor_sync(0xffffffffu, acc[0], 1);
    if ((lane & 1) == 0) s_b[mine + (mine >= 64 ? 16 : 0)] = mine < rows ? rhs - sum : 0.f;
    __syncthreads();
    ts_publish(a, ts_sm, s_b, false, r0, rows);
}

// The transposed substitutions of the adjoint solve, A^T x = b with
// P A = L U: U^T (lower, forward; lower = 1) and L^T (unit upper, backward;
// lower = 0) in one launch each, with the same tickets and published values.
// Block row i of U^T (L^T) is block column i of U (L): thread (c, half) sums
// column c over half the rows of each solved block; the diagonal block uses
// the transposed inverse.
__global__ void __launch_bounds__(TS_TH) trsv_chain_t_kernel(TsArgs a)
{
    extern __shared__ float ts_sm[];
    __shared__ float s_b[144], s_z[2][TS_R], s_h[TS_R];
    __shared__ int s_t;
    const int tid = threadIdx.x, c = tid & (TS_R - 1), half = tid / TS_R;
    const int n = a.n, nbk = (n + TS_R - 1) / TS_R;
    if (tid == 0) s_t = atomicAdd(a.ticket, 1);
    __syncthreads();
    const int t = s_t;
    const int blk = a.lower ? t : nbk - 1 - t;
    const int i0 = blk * TS_R, ni = min(TS_R, n - i0);
    ts_load_inv(a, blk, a.lower ? 1 : 0, ts_sm);
    const float rhs = c < ni ? a.y[i0 + c] : 0.f;
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    bool gave = false;
    for (int st = 0; st < t; ++st) {
        const int j = a.lower ? st : nbk - 1 - st;
        const int j0 = j * TS_R, nj = min(TS_R, n - j0);
        const float *col = a.LU + (size_t)j0 * n + i0 + c;
        float v[TS_R / 2];
#pragma unroll
        for (int u = 0; u < TS_R / 2; ++u) {
            const int r = half * (TS_R / 2) + u;
            v[u] = c < ni && r < nj ? col[(size_t)r * n] : 0.f;
        }
        float *z = s_z[st & 1];
        if (tid < 32) ts_wait(a, j0, nj, t - st, z, gave);
        __syncthreads();
#pragma unroll
        for (int u = 0; u < TS_R / 2; ++u) acc[u & 3] = fmaf(v[u], z[half * (TS_R / 2) + u], acc[u & 3]);
    }
    const float sum = (acc[0] + acc[1]) + (acc[2] + acc[3]);
    if (half == 1) s_h[c] = sum;
    __syncthreads();
    if (half == 0) s_b[c + (c >= 64 ? 16 : 0)] = c < ni ? rhs - (sum + s_h[c]) : 0.f;
    __syncthreads();
    ts_publish(a, ts_sm, s_b, true, i0, ni);
}

// ------------------------------------------------------------------ host drivers
// A22 -= L21 U12 for the panel at column k (width kb) in cuBLAS (FP32, TF32
// or BF16x9 arithmetic).  A is row-major; cuBLAS sees it column-major, i.e.
// transposed, so the call computes A22^T -= U12^T L21^T with U12 as its first
// operand.
static int gemm_update(obem_ctx *c, int precision, float *A, int n, int k, int kb, cudaStream_t s)
{
    const int M = n - k - kb;
    if (M <= 0) return OBEM_OK;
    const float alpha = -1.0f, beta = 1.0f;
    float *A22 = A + (size_t)(k + kb) * n + (k + kb);
    float *L21 = A + (size_t)(k + kb) * n + k;
    float *U12 = A + (size_t)k * n + (k + kb);
    cublasComputeType_t ct = CUBLAS_COMPUTE_32F;
    if (precision == OBEM_LU_TF32) ct = CUBLAS_COMPUTE_32F_FAST_TF32;
    else if (precision == OBEM_LU_BF16X9) ct = CUBLAS_COMPUTE_32F_EMULATED_16BFX9;
    cublasStatus_t st = cublasGemmEx(c->cublas, CUBLAS_OP_N, CUBLAS_OP_N, M, M, kb, &alpha, U12,
                                     CUDA_R_32F, n, L21, CUDA_R_32F, n, &beta, A22, CUDA_R_32F, n, ct,
                                     CUBLAS_GEMM_DEFAULT);
    if (st != CUBLAS_STATUS_SUCCESS)
        return obem_fail(c, OBEM_ERR_CUDA, "cublasGemmEx failed (status %d)", (int)st);
    return OBEM_OK;
}

// Pivoting panel factorisation of A[k:n, k:k+kb] (cooperative panel_kernel)
// followed by its row swaps on every other column.
struct PanelScratch {
    unsigned long long *rec, *crows, *gdiag;    // of the panel exchange
    int *plan;                      // the row swaps' plan (LS_PLAN_INTS)
    float *rows;                    // [2 LU_NB][n] the touched rows during the swaps
    int nsm;
};

static int factor_panel(obem_ctx *c, const PanelScratch &P, int k, int kb, cudaStream_t s)
{
    const int n = c->nsys;
    const int rows = n - k;
    int G = (rows + 31) / 32;
    if (G > P.nsm) G = P.nsm;
    // above ~nsm x 787 rows (about 120k cells) one chunk per SM no longer
    // fits a CTA's shared memory: m = 2, 3, 4 co-resident CTAs per SM,
    // each chunk within 1/m of the SM's 224 KB (the occupancy check
    // below rejects a size that still does not fit)
    const size_t row_b = sizeof(float) * (size_t)(kb + 1);
    if ((size_t)((rows + G - 1) / G) * row_b > 200 * 1024)
        for (int m = 2; m <= 4; ++m) {
            G = m * P.nsm;
            if ((size_t)((rows + G - 1) / G) * row_b <= (size_t)224 * 1024 / m) break;
        }
    if (G > PAN_MAXG) G = PAN_MAXG;
    int R = (rows + G - 1) / G;
    G = (rows + R - 1) / R;
    size_t smem = sizeof(float) * (size_t)R * (kb + 1);
    if (smem > 200 * 1024)
        return obem_fail(c, OBEM_ERR_ARG, "LU panel of %d rows does not fit shared memory", rows);
    // host-side queries once, not per panel (they cost tens of microseconds
    // each, and the factorisation issues a panel every few hundred): the
    // attribute at the largest panel size; one CTA per SM always fits (at
    // most 200 KB of shared memory, 48 registers x 256 threads), so the
    // occupancy is checked only when there are more CTAs than SMs
    static unsigned long long attr = 0;   // devices done (a bit each)
    if (!(attr >> (c->device & 63) & 1ull)) {
        OBEM_CUDA(c, cudaFuncSetAttribute(panel_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024));
        attr |= 1ull << (c->device & 63);
    }
    if (G > P.nsm) {
        int per_sm = 0;
        OBEM_CUDA(c, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, panel_kernel, 256, smem));
        if (per_sm * P.nsm < G)
            return obem_fail(c, OBEM_ERR_CUDA, "LU panel: %d CTAs cannot be co-resident", G);
    }
    PanelArgs pa;
    pa.A = c->d_LU; pa.n = n; pa.k = k; pa.kb = kb; pa.rows_per_cta = R; pa.piv = c->d_piv;
    pa.flag = c->d_flag; pa.rec = P.rec; pa.crows = P.crows; pa.gdiag = P.gdiag;
    void *args[] = {&pa};
    OBEM_CUDA(c, cudaLaunchCooperativeKernel((void *)panel_kernel, dim3(G), dim3(256), args, smem, s));
    laswp_plan_kernel<<<1, LU_NB, 0, s>>>(k, kb, c->d_piv, c->d_flag, P.plan);
    const dim3 lg(n / 1024 + 1 < 64 ? n / 1024 + 1 : 64, 2 * LU_NB);
    laswp_gather_kernel<<<lg, 256, 0, s>>>(c->d_LU, n, P.plan, P.rows);
    laswp_scatter_kernel<<<lg, 256, 0, s>>>(c->d_LU, n, k, kb, P.plan, P.rows);
    OBEM_LAUNCH(c);
    return OBEM_OK;
}

// Split of a recursive block of w columns: a multiple of LU_NB near w / 2.
static int rec_split(int w)
{
    const int h = (w / (2 * LU_NB)) * LU_NB;
    return h > LU_NB ? h : LU_NB;
}

// X = L^-1 X with L = LU[r0:r0+m, r0:r0+m] (unit lower) and X = LU[r0:r0+m,
// c0:c0+nc], recursively: X1 = L11^-1 X1, X2 -= L21 X1 (tensor-core GEMM),
// X2 = L22^-1 X2.
static int rec_trsm(obem_ctx *c, int r0, int m, int c0, int nc, cudaStream_t s)
{
    const int n = c->nsys;
    float *A = c->d_LU;
    if (nc <= 0 || m <= 0) return OBEM_OK;
    if (m <= TRSM_LEAF) {
        const int nb = (nc + TRSM_LEAF_THREADS - 1) / TRSM_LEAF_THREADS;
        static unsigned long long attr = 0;   // devices done (a bit each)
        if (!(attr >> (c->device & 63) & 1ull)) {
            OBEM_CUDA(c, cudaFuncSetAttribute(trsm_leaf_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)trsm_leaf_smem<64>()));
            OBEM_CUDA(c, cudaFuncSetAttribute(trsm_leaf_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)trsm_leaf_smem<128>()));
            OBEM_CUDA(c, cudaFuncSetAttribute(trsm_leaf2_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)trsm_leaf2_smem<64>()));
            OBEM_CUDA(c, cudaFuncSetAttribute(trsm_leaf2_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)trsm_leaf2_smem<128>()));
            attr |= 1ull << (c->device & 63);
        }
        const int nb2 = (nc + TL2_BC - 1) / TL2_BC;
        if (nc <= 8192) {
            // narrow: the warp-per-columns form has the shorter block latency
            if (m <= 64)
                trsm_leaf2_kernel<64><<<nb2, TL2_W * 32, trsm_leaf2_smem<64>(), s>>>(A, n, r0, m, c0, nc);
            else
                trsm_leaf2_kernel<128><<<nb2, TL2_W * 32, trsm_leaf2_smem<128>(), s>>>(A, n, r0, m, c0, nc);
        } else if (m <= 64) {
            trsm_leaf_kernel<64><<<nb, TRSM_LEAF_THREADS, trsm_leaf_smem<64>(), s>>>(A, n, r0, m, c0, nc);
        } else {
            trsm_leaf_kernel<128><<<nb, TRSM_LEAF_THREADS, trsm_leaf_smem<128>(), s>>>(A, n, r0, m, c0, nc);
        }
        OBEM_LAUNCH(c);
        return OBEM_OK;
    }
    const int m1 = rec_split(m);
    int rc = rec_trsm(c, r0, m1, c0, nc, s);
    if (rc == OBEM_OK)
        rc = obem_tc_gemm_sub(c, A + (size_t)(r0 + m1) * n + c0, n, A + (size_t)(r0 + m1) * n + r0, n,
                              A + (size_t)r0 * n + c0, n, m - m1, nc, m1, c->d_flag + 4, s);
    if (rc == OBEM_OK) rc = rec_trsm(c, r0 + m1, m - m1, c0, nc, s);
    return rc;
}

// Largest BF16 operands (elements, rows x 8-padded K) of the GEMMs that
// rec_lu / rec_trsm issue, so that the scratch is reserved once.
static void rec_trsm_sizes(int m, int nc, size_t &a, size_t &b)
{
    if (nc <= 0 || m <= TRSM_LEAF) return;
    const int m1 = rec_split(m);
    const size_t k8 = ((size_t)m1 + 7) / 8 * 8;
    a = a > (size_t)(m - m1) * k8 ? a : (size_t)(m - m1) * k8;
    b = b > (size_t)nc * k8 ? b : (size_t)nc * k8;
    rec_trsm_sizes(m1, nc, a, b);
    rec_trsm_sizes(m - m1, nc, a, b);
}

static void rec_lu_sizes(int n, int k0, int w, size_t &a, size_t &b)
{
    if (w <= LU_NB) return;
    const int w1 = rec_split(w);
    const size_t k8 = ((size_t)w1 + 7) / 8 * 8;
    rec_lu_sizes(n, k0, w1, a, b);
    rec_trsm_sizes(w1, w - w1, a, b);
    a = a > (size_t)(n - k0 - w1) * k8 ? a : (size_t)(n - k0 - w1) * k8;
    b = b > (size_t)(w - w1) * k8 ? b : (size_t)(w - w1) * k8;
    rec_lu_sizes(n, k0 + w1, w - w1, a, b);
}

// Recursive LU with partial pivoting of the columns [k0, k0 + w) of rows
// [k0, n) (Toledo's recursion): factor the left half, U12 = L11^-1 A12,
// A22 -= L21 U12 on the tensor cores (BF16 operands, FP32 accumulation into
// the FP32 matrix), factor the right half.  Panels of LU_NB columns are the
// leaves; their row swaps are applied to whole rows at once.
static int rec_lu(obem_ctx *c, const PanelScratch &P, int k0, int w, cudaStream_t s)
{
    const int n = c->nsys;
    float *A = c->d_LU;
    if (w <= LU_NB) return factor_panel(c, P, k0, w, s);
    const int w1 = rec_split(w);
    int rc = rec_lu(c, P, k0, w1, s);
    if (rc == OBEM_OK) rc = rec_trsm(c, k0, w1, k0 + w1, w - w1, s);
    if (rc == OBEM_OK)
        rc = obem_tc_gemm_sub(c, A + (size_t)(k0 + w1) * n + (k0 + w1), n, A + (size_t)(k0 + w1) * n + k0, n,
                              A + (size_t)k0 * n + (k0 + w1), n, n - k0 - w1, w - w1, w1, c->d_flag + 4, s);
    if (rc == OBEM_OK) rc = rec_lu(c, P, k0 + w1, w - w1, s);
    return rc;
}

// Buffers of an n x n system (matrix, factors, pivots, scaling, refinement
// and panel scratch), reallocated when n changes.
static int alloc_system(obem_ctx *c, int n)
{
    if (c->d_A && c->nsys_alloc == n) return OBEM_OK;
    void *bufs[] = {c->d_A, c->d_LU, c->d_piv, c->d_rowscale, c->d_work64, c->d_work32, c->d_flag, c->d_panel,
                    c->d_perm, c->d_trsv, c->d_dinv};
    for (void *q : bufs)
        if (q) cudaFree(q);
    c->d_A = c->d_LU = NULL;
    c->d_piv = c->d_flag = c->d_perm = NULL;
    c->d_trsv = NULL;
    c->d_dinv = NULL;
    c->d_rowscale = c->d_work64 = NULL;
    c->d_work32 = c->d_panel = NULL;
    c->nsys_alloc = 0;
    const size_t nn = (size_t)n * n;
    OBEM_CUDA(c, cudaMalloc((void **)&c->d_A, sizeof(float) * nn));
    OBEM_CUDA(c, cudaMalloc((void **)&c->d_LU, sizeof(float) * nn));
    OBEM_CUDA(c, cudaMalloc((void **)&c->d_piv, sizeof(int) * n));
    OBEM_CUDA(c, cudaMalloc((void **)&c->d_rowscale, sizeof(double) * n));
    OBEM_CUDA(c, cudaMalloc((void **)&c->d_work64, sizeof(double) * (4 * (size_t)n + 8)));
    OBEM_CUDA(c, cudaMalloc((void **)&c->d_work32, sizeof(float) * (2 * (size_t)n + 4096)));
    OBEM_CUDA(c, cudaMalloc((void **)&c->d_flag, sizeof(int) * 8));
    OBEM_CUDA(c, cudaMalloc((void **)&c->d_panel,
                            sizeof(float) * (PAN_SCRATCH_FLOATS + PAN_PLAN_FLOATS + 2 * (size_t)LU_NB * n)));
    OBEM_CUDA(c, cudaMalloc((void **)&c->d_perm, sizeof(int) * n));
    // published values of the substitutions (no epoch yet), tickets and status
    OBEM_CUDA(c, cudaMalloc((void **)&c->d_trsv, sizeof(unsigned long long) * ((size_t)n + 4)));
    OBEM_CUDA(c, cudaMemset(c->d_trsv, 0, sizeof(unsigned long long) * ((size_t)n + 4)));
    c->trsv_epoch = 0;
    OBEM_CUDA(c, cudaMalloc((void **)&c->d_dinv, sizeof(float) * 2 * TS_R * TS_R * (size_t)((n + TS_R - 1) / TS_R)));
    c->nsys_alloc = n;
    return OBEM_OK;
}

static int factor_system(obem_ctx *c, int precision, cudaStream_t s);

int obem_assemble_and_factor(obem_ctx *c, int precision, cudaStream_t s)
{
    c->factored = 0;
    c->nsys = c->np;
    const int n = c->nsys;
    int rc0 = alloc_system(c, n);
    if (rc0 != OBEM_OK) return rc0;
    // --- assembly
    PanelsDev P;
    P.c_a = c->d_c_a; P.g0_h = c->d_g0_h; P.g1 = c->d_g1; P.g2 = c->d_g2; P.nrm = c->d_nrm;
    P.c_lo = c->d_c_lo;
    P.v64 = c->d_v64; P.geo = c->d_geo64; P.geo2 = obem_geo2_of(c->d_geo64, n); P.np = n;
    double *d_em = NULL, *d_ep = NULL;
    struct FreeOnExit { void *p; ~FreeOnExit() { if (p) cudaFree(p); } };
    OBEM_CUDA(c, cudaMalloc((void **)&d_em, sizeof(double) * n));
    FreeOnExit em_guard{d_em};
    OBEM_CUDA(c, cudaMalloc((void **)&d_ep, sizeof(double) * n));
    FreeOnExit ep_guard{d_ep};
    OBEM_CUDA(c, cudaMemcpyAsync(d_em, c->h_em, sizeof(double) * n, cudaMemcpyHostToDevice, s));
    OBEM_CUDA(c, cudaMemcpyAsync(d_ep, c->h_ep, sizeof(double) * n, cudaMemcpyHostToDevice, s));
    const dim3 ag((n + AS_TH - 1) / AS_TH, (n + AS_ROWS - 1) / AS_ROWS);
    assemble_kernel<<<ag, AS_TH, 0, s>>>(P, c->d_kind, d_em, d_ep, c->d_A, n);
    OBEM_LAUNCH(c);
    return factor_system(c, precision, s);
}

// A caller-given dense system in place of an assembled one (see obem.h).
int obem_factor_dense(obem_ctx *c, const float *A, int n, int precision, cudaStream_t s)
{
    c->factored = 0;
    c->nsys = n;
    int rc = alloc_system(c, n);
    if (rc != OBEM_OK) return rc;
    OBEM_CUDA(c, cudaMemcpyAsync(c->d_A, A, sizeof(float) * (size_t)n * n, cudaMemcpyDeviceToDevice, s));
    return factor_system(c, precision, s);
}

// Row equilibration of d_A (rows scaled by 1 / max |a_ij|, ||A||_inf kept for
// the backward error), LU factorisation into d_LU in the requested
// arithmetic, and the row permutation of the pivots.
static int factor_system(obem_ctx *c, int precision, cudaStream_t s)
{
    const int n = c->nsys;
    if (!c->cublas) {
        if (cublasCreate(&c->cublas) != CUBLAS_STATUS_SUCCESS)
            return obem_fail(c, OBEM_ERR_CUDA, "cublasCreate failed");
    }
    cublasSetStream(c->cublas, s);
    double *d_rownorm = c->d_work64;     // reused as scratch here
    equilibrate_kernel<<<n, EQ_TH, 0, s>>>(c->d_A, c->d_LU, n, c->d_rowscale, d_rownorm);
    OBEM_LAUNCH(c);
    std::vector<double> rn(n);
    OBEM_CUDA(c, cudaMemcpyAsync(rn.data(), d_rownorm, sizeof(double) * n, cudaMemcpyDeviceToHost, s));
    OBEM_CUDA(c, cudaStreamSynchronize(s));
    c->a_norm_inf = 0.0;
    for (int i = 0; i < n; ++i) c->a_norm_inf = rn[i] > c->a_norm_inf ? rn[i] : c->a_norm_inf;
    // --- factorisation
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    OBEM_CUDA(c, cudaMemsetAsync(c->d_flag, 0, sizeof(int) * 8, s));
    cudaEventRecord(e0, s);
    int nsm = 0;
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, c->device);
    PanelScratch PS;
    PS.rec = (unsigned long long *)c->d_panel;
    PS.gdiag = PS.rec + 2 * PAN_MAXG;
    PS.crows = PS.gdiag + 2 * LU_NB;
    // no epoch of an earlier factorisation
    OBEM_CUDA(c, cudaMemsetAsync(c->d_panel, 0, sizeof(float) * PAN_SCRATCH_FLOATS, s));
    PS.plan = (int *)(c->d_panel + PAN_SCRATCH_FLOATS);
    PS.rows = c->d_panel + PAN_SCRATCH_FLOATS + PAN_PLAN_FLOATS;
    PS.nsm = nsm;
    if (precision == OBEM_LU_BF16) {
        // recursive factorisation, trailing updates on the tensor cores
        size_t ea = 0, eb = 0;
        rec_lu_sizes(n, 0, n, ea, eb);
        int rc = obem_tc_reserve(c, ea, eb);
        if (rc == OBEM_OK) rc = rec_lu(c, PS, 0, n, s);
        if (rc != OBEM_OK) return rc;
    } else {
        // right-looking blocked factorisation, trailing updates in cuBLAS
        for (int k = 0; k < n; k += LU_NB) {
            const int kb = n - k < LU_NB ? n - k : LU_NB;
            int rc = factor_panel(c, PS, k, kb, s);
            if (rc != OBEM_OK) return rc;
            if (k + kb < n) {
                trsm_kernel<<<(n - k - kb + TRSM_COLS - 1) / TRSM_COLS, TRSM_COLS, 0, s>>>(c->d_LU, n, k, kb);
                OBEM_LAUNCH(c);
                rc = gemm_update(c, precision, c->d_LU, n, k, kb, s);
                if (rc != OBEM_OK) return rc;
            }
        }
    }
    cudaEventRecord(e1, s);
    int flag[8] = {0};
    OBEM_CUDA(c, cudaMemcpyAsync(flag, c->d_flag, sizeof(flag), cudaMemcpyDeviceToHost, s));
    OBEM_CUDA(c, cudaStreamSynchronize(s));
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    c->factor_ms = ms;
    if (flag[0] == OBEM_ERR_SINGULAR) return obem_fail(c, OBEM_ERR_SINGULAR, "LU: zero pivot");
    if (flag[0] == OBEM_ERR_TIMEOUT) return obem_fail(c, OBEM_ERR_TIMEOUT, "LU: a panel's wait for the pivot candidates timed out");
    if (flag[4] != 0) return obem_fail(c, OBEM_ERR_TIMEOUT, "LU: a tensor-core GEMM wait timed out");
    // the row swaps as one permutation: (P b)[i] = b[perm[i]]
    {
        std::vector<int> piv(n), perm(n);
        OBEM_CUDA(c, cudaMemcpy(piv.data(), c->d_piv, sizeof(int) * n, cudaMemcpyDeviceToHost));
        for (int i = 0; i < n; ++i) perm[i] = i;
        for (int i = 0; i < n; ++i)
            if (piv[i] != i) { const int t = perm[i]; perm[i] = perm[piv[i]]; perm[piv[i]] = t; }
        OBEM_CUDA(c, cudaMemcpy(c->d_perm, perm.data(), sizeof(int) * n, cudaMemcpyHostToDevice));
    }
    // inverses of the diagonal blocks for the one-launch substitutions
    {
        static unsigned long long attr = 0;   // devices done (a bit each)
        if (!(attr >> (c->device & 63) & 1ull)) {
            OBEM_CUDA(c, cudaFuncSetAttribute(inv_diag_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)TS_INV_SMEM));
            OBEM_CUDA(c, cudaFuncSetAttribute(trsv_chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)TS_SMEM));
            attr |= 1ull << (c->device & 63);
        }
        inv_diag_kernel<<<dim3((n + TS_R - 1) / TS_R, 2), TS_R, TS_INV_SMEM, s>>>(c->d_LU, n, c->d_dinv);
        OBEM_LAUNCH(c);
    }
    c->factored = 1;
    return OBEM_OK;
}

// y <- U^-1 L^-1 y with the stored factors: two one-launch substitutions.
// A flag wait that ran out is reported as OBEM_ERR_TIMEOUT after the launch.
static int lu_solve(obem_ctx *c, float *y, cudaStream_t s)
{
    const int n = c->nsys, nbk = (n + TS_R - 1) / TS_R;
    int *ticket = (int *)(c->d_trsv + n), *err = ticket + 2;
    OBEM_CUDA(c, cudaMemsetAsync(ticket, 0, sizeof(int) * 3, s));
    for (int lower = 1; lower >= 0; --lower) {
        TsArgs a;
        a.LU = c->d_LU;
        a.dinv = c->d_dinv;
        a.y = y;
        a.n = n;
        a.lower = lower;
        a.epoch = ++c->trsv_epoch;
        a.z = c->d_trsv;
        a.ticket = ticket + (lower ? 0 : 1);
        a.err = err;
        trsv_chain_kernel<<<nbk, TS_TH, TS_SMEM, s>>>(a);
        OBEM_LAUNCH(c);
    }
    int h = 0;
    OBEM_CUDA(c, cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    OBEM_CUDA(c, cudaStreamSynchronize(s));
    if (h != 0) return obem_fail(c, OBEM_ERR_TIMEOUT, "LU solve: a wait for a solved block timed out");
    return OBEM_OK;
}

// Failure-detection self-test of the substitutions' flag wait: one thread
// block draws ticket 1 (the counter starts at 1) and waits for block row 0,
// which no block solves; the wait runs out after TS_WAIT_NS and records
// OBEM_ERR_TIMEOUT.  Needs the factors of a system of at least 2 TS_R rows.
int obem_selftest_solve_wait(obem_ctx *c, cudaStream_t s)
{
    if (!c->factored || c->nsys < 2 * TS_R)
        return obem_fail(c, OBEM_ERR_STATE, "wait self-test: needs the factors of a system of >= %d rows", 2 * TS_R);
    const int n = c->nsys;
    int *ticket = (int *)(c->d_trsv + n), *err = ticket + 2;
    const int one = 1;
    OBEM_CUDA(c, cudaMemsetAsync(ticket, 0, sizeof(int) * 3, s));
    OBEM_CUDA(c, cudaMemcpyAsync(ticket, &one, sizeof(int), cudaMemcpyHostToDevice, s));
    TsArgs a;
    a.LU = c->d_LU;
    a.dinv = c->d_dinv;
    a.y = c->d_work32;
    a.n = n;
    a.lower = 1;
    a.epoch = ++c->trsv_epoch;
    a.z = c->d_trsv;
    a.ticket = ticket;
    a.err = err;
    trsv_chain_kernel<<<1, TS_TH, TS_SMEM, s>>>(a);
    OBEM_LAUNCH(c);
    int h = 0;
    OBEM_CUDA(c, cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    OBEM_CUDA(c, cudaStreamSynchronize(s));
    if (h != OBEM_ERR_TIMEOUT) return obem_fail(c, OBEM_ERR_STATE, "wait self-test: status %d, expected a timeout", h);
    return OBEM_OK;
}

// Iterative refinement of A x = b with the stored factors: b (device, FP64,
// rows already equilibrated) in c->d_work64[0, n), x in [n, 2n); FP64
// residuals r = b - A x from the FP32 equilibrated matrix, corrections from
// the factors.  Returns the iterations, status and backward error.
static int refine(obem_ctx *c, int &it, int &status, double &be, cudaStream_t s)
{
    const int n = c->nsys;
    double *b = c->d_work64, *x = b + n, *r = x + n, *nrm = r + n;
    float *y = c->d_work32;
    OBEM_CUDA(c, cudaMemsetAsync(x, 0, sizeof(double) * n, s));
    double be_prev = 2.0;
    be = 1.0;
    it = 0;
    status = OBEM_ERR_NOT_CONVERGED;
    const int max_it = 30;
    for (; it <= max_it; ++it) {
        if (it == 0) {
            // x = 0: the residual is b (no pass over the matrix)
            OBEM_CUDA(c, cudaMemcpyAsync(r, b, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
        } else {
            split_kernel<<<(n + 255) / 256, 256, 0, s>>>(x, y, y + n, n);
            residual_kernel<<<(n + 7) / 8, 256, 0, s>>>(c->d_A, y, y + n, b, r, n);
        }
        norms_kernel<<<1, 1024, 0, s>>>(r, x, b, n, nrm);
        OBEM_LAUNCH(c);
        double h[3];
        OBEM_CUDA(c, cudaMemcpyAsync(h, nrm, sizeof h, cudaMemcpyDeviceToHost, s));
        OBEM_CUDA(c, cudaStreamSynchronize(s));
        be = h[0] / (c->a_norm_inf * h[1] + h[2] + 1e-300);
        // converged: at the FP64 rounding level, or no longer decreasing once
        // below 1e-9 (the residual's own rounding floor for large n)
        if (be < 1e-12 || (be < 1e-9 && be > 0.5 * be_prev)) { status = OBEM_OK; break; }
        be_prev = be;
        if (it == max_it) break;
        permute_kernel<<<(n + 255) / 256, 256, 0, s>>>(r, y, c->d_perm, n, nrm);
        OBEM_LAUNCH(c);
        int rc = lu_solve(c, y, s);
        if (rc != OBEM_OK) return rc;
        axpy_kernel<<<(n + 255) / 256, 256, 0, s>>>(x, y, nrm, n);
        OBEM_LAUNCH(c);
    }
    return OBEM_OK;
}

static void fill_report(obem_ctx *c, obem_solve_report *rep, int it, int status, double be, float ms)
{
    if (!rep) return;
    rep->iterations = it;
    rep->status = status;
    rep->backward_error = be;
    rep->factor_ms = c->factor_ms;
    rep->solve_ms = ms;
}

int obem_solve_system(obem_ctx *c, const double *gv, const float *sigma_free, const float *drhs,
                      float *sigma_out, obem_solve_report *rep, cudaStream_t s)
{
    const int n = c->nsys;
    cublasSetStream(c->cublas, s);
    double *b = c->d_work64, *x = b + n;
    double *d_gv = NULL;
    int ng = c->n_groups > 0 ? c->n_groups : 1;
    OBEM_CUDA(c, cudaMalloc((void **)&d_gv, sizeof(double) * ng));
    struct FreeOnExit { void *p; ~FreeOnExit() { if (p) cudaFree(p); } } gv_guard{d_gv};
    if (c->n_groups > 0)
        OBEM_CUDA(c, cudaMemcpyAsync(d_gv, gv, sizeof(double) * c->n_groups, cudaMemcpyHostToDevice, s));
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, s);
    rhs_kernel<<<(n + 255) / 256, 256, 0, s>>>(c->d_kind, c->d_group, d_gv, sigma_free, drhs, c->d_rowscale, b, n);
    OBEM_LAUNCH(c);
    int it = 0, status = OBEM_ERR_NOT_CONVERGED;
    double be = 1.0;
    int rc = refine(c, it, status, be, s);
    if (rc != OBEM_OK) return rc;
    to_float_kernel<<<(n + 255) / 256, 256, 0, s>>>(x, sigma_out, c->d_sigma, n);
    OBEM_LAUNCH(c);
    cudaEventRecord(e1, s);
    OBEM_CUDA(c, cudaStreamSynchronize(s));
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    c->sigma_valid = 1;
    c->sigma_ver++;
    fill_report(c, rep, it, status, be, ms);
    if (status != OBEM_OK)
        return obem_fail(c, OBEM_ERR_NOT_CONVERGED, "refinement stopped at backward error %.3e after %d iterations", be, it);
    return OBEM_OK;
}

// b_i = rowscale_i * bin_i
__global__ void scale_rhs_kernel(const double *bin, const double *rowscale, double *b, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = bin[i] * rowscale[i];
}

// Solve of the dense system given to obem_dense_factor for one right-hand
// side (device FP64 b, x), with the same refinement as the BEM solve.
int obem_solve_dense_rhs(obem_ctx *c, const double *bin, double *xout, obem_solve_report *rep, cudaStream_t s)
{
    const int n = c->nsys;
    double *b = c->d_work64, *x = b + n;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, s);
    scale_rhs_kernel<<<(n + 255) / 256, 256, 0, s>>>(bin, c->d_rowscale, b, n);
    OBEM_LAUNCH(c);
    int it = 0, status = OBEM_ERR_NOT_CONVERGED;
    double be = 1.0;
    int rc = refine(c, it, status, be, s);
    if (rc != OBEM_OK) return rc;
    OBEM_CUDA(c, cudaMemcpyAsync(xout, x, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
    cudaEventRecord(e1, s);
    OBEM_CUDA(c, cudaStreamSynchronize(s));
    float ms = 0.f;
    cudaEventElapsedTime(&ms, e0, e1);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    fill_report(c, rep, it, status, be, ms);
    if (status != OBEM_OK)
        return obem_fail(c, OBEM_ERR_NOT_CONVERGED, "refinement stopped at backward error %.3e after %d iterations", be, it);
    return OBEM_OK;
}

// ====================================================================
// Adjoint of the solve: mu = A^-T g (g = dL/dsigma) is dL/db for the right-hand
// side of Eq. (matrixBEM).  With the row-equilibrated matrix At = D A and its
// factors P At = L U:  A^T mu = g  <=>  At^T nu = g,  mu = D nu,  and
// At^T = U^T L^T P, so each refinement step solves U^T z = r (forward),
// L^T w = z (backward, unit diagonal) and undoes the row swaps (nu = P^-1 w).
// The residual g - At^T nu is accumulated in FP64 from the stored FP32 At.
// ====================================================================
#define ADJ_SPLIT 16           // row ranges of the transposed residual

// part[s][j] = sum over rows i of range s of At[i][j] x[i]; one thread per column
__global__ void residual_t_part_kernel(const float *A, const float *xh, const float *xl, double *part, int n)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int s = blockIdx.y;
    const int i0 = (int)((long long)n * s / ADJ_SPLIT), i1 = (int)((long long)n * (s + 1) / ADJ_SPLIT);
    if (j >= n) return;
    float sm = 0.f, cm = 0.f;
    int i = i0;
    for (; i + 7 < i1; i += 8) {
        float av[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) av[u] = __ldcs(A + (size_t)(i + u) * n + j);
#pragma unroll
        for (int u = 0; u < 8; ++u) df_acc(sm, cm, av[u], xh[i + u], xl[i + u]);
    }
    for (; i < i1; ++i) df_acc(sm, cm, A[(size_t)i * n + j], xh[i], xl[i]);
    part[(size_t)s * n + j] = (double)sm + (double)cm;
}
__global__ void residual_t_fold_kernel(const double *part, const double *b, double *r, int n)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    double s = 0.0;
    for (int q = 0; q < ADJ_SPLIT; ++q) s += part[(size_t)q * n + j];
    r[j] = b[j] - s;
}

// column sums of |A| over a share of the rows (for the transposed system's
// infinity norm), compensated; HBM-bound (one thread per column over all rows
// in FP64 took 1.65 ms at 11,008 cells)
__global__ void colsum_kernel(const float *A, double *part, int n)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int s = blockIdx.y;
    const int i0 = (int)((long long)n * s / ADJ_SPLIT), i1 = (int)((long long)n * (s + 1) / ADJ_SPLIT);
    if (j >= n) return;
    float sm = 0.f, cm = 0.f;
    int i = i0;
    for (; i + 7 < i1; i += 8) {
        float av[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) av[u] = __ldcs(A + (size_t)(i + u) * n + j);
#pragma unroll
        for (int u = 0; u < 8; ++u) two_sum_acc(sm, cm, fabsf(av[u]));
    }
    for (; i < i1; ++i) two_sum_acc(sm, cm, fabsf(A[(size_t)i * n + j]));
    part[(size_t)s * n + j] = (double)sm + (double)cm;
}
__global__ void colsum_fold_kernel(const double *part, double *colsum, int n)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    double s = 0.0;
    for (int q = 0; q < ADJ_SPLIT; ++q) s += part[(size_t)q * n + j];
    colsum[j] = s;
}

__global__ void max_kernel(const double *v, int n, double *out)
{
    __shared__ double s[256];
    double a = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) a = fmax(a, v[i]);
    s[threadIdx.x] = a;
    __syncthreads();
    for (int o = blockDim.x / 2; o; o >>= 1) {
        if (threadIdx.x < o) s[threadIdx.x] = fmax(s[threadIdx.x], s[threadIdx.x + o]);
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = s[0];
}

__global__ void load_adjoint_kernel(const float *g, double *b, double *x, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    b[i] = (double)g[i];
    x[i] = 0.0;
}

// y = r / sc in FP32 (sc = max|r|)
__global__ void scale_to_float_kernel(const double *r, float *y, int n, const double *norms)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double sc = norms[0] > 0 ? norms[0] : 1.0;
    y[i] = (float)(r[i] / sc);
}

// x += P^T y sc: the transposed row permutation as a scatter, x[perm[i]] +=
// y[i] sc (sc = max |r|)
__global__ void axpy_unpermute_kernel(double *x, const float *y, const int *perm, const double *norms, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const double sc = norms[0] > 0 ? norms[0] : 1.0;
    x[perm[i]] += (double)y[i] * sc;
}



// y <- L^-T U^-T y with the stored factors (the adjoint's substitutions)
static int lu_solve_t(obem_ctx *c, float *y, cudaStream_t s)
{
    const int n = c->nsys, nbk = (n + TS_R - 1) / TS_R;
    int *ticket = (int *)(c->d_trsv + n), *err = ticket + 2;
    static unsigned long long attr = 0;   // devices done (a bit each)
    if (!(attr >> (c->device & 63) & 1ull)) {
        OBEM_CUDA(c, cudaFuncSetAttribute(trsv_chain_t_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)TS_SMEM));
        attr |= 1ull << (c->device & 63);
    }
    OBEM_CUDA(c, cudaMemsetAsync(ticket, 0, sizeof(int) * 3, s));
    for (int lower = 1; lower >= 0; --lower) {
        TsArgs a;
        a.LU = c->d_LU;
        a.dinv = c->d_dinv;
        a.y = y;
        a.n = n;
        a.lower = lower;
        a.epoch = ++c->trsv_epoch;
        a.z = c->d_trsv;
        a.ticket = ticket + (lower ? 0 : 1);
        a.err = err;
        trsv_chain_t_kernel<<<nbk, TS_TH, TS_SMEM, s>>>(a);
        OBEM_LAUNCH(c);
    }
    int h = 0;
    OBEM_CUDA(c, cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s));
    OBEM_CUDA(c, cudaStreamSynchronize(s));
    if (h != 0) return obem_fail(c, OBEM_ERR_TIMEOUT, "adjoint solve: a wait for a solved block timed out");
    return OBEM_OK;
}

int obem_solve_adjoint(obem_ctx *c, const float *g, double *dL_dgv, float *dL_db, obem_solve_report *rep,
                       cudaStream_t s)
{
    const int n = c->nsys;
    double *b = c->d_work64, *x = b + n, *r = x + n, *nrm = r + n;
    float *y = c->d_work32;
    double *part = NULL, *col = NULL, *mu = NULL;
    int rc = OBEM_OK, it = 0, status = OBEM_ERR_NOT_CONVERGED;
    double be = 1.0, be_prev = 2.0, a1 = 0.0;
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    cudaEventRecord(e0, s);
#define ADJ_CUDA(call)                                                                             \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess) {                                                                   \
            rc = obem_fail(c, OBEM_ERR_CUDA, "%s failed: %s", #call, cudaGetErrorString(e_));      \
            goto done;                                                                             \
        }                                                                                          \
    } while (0)
    ADJ_CUDA(cudaMalloc((void **)&part, sizeof(double) * (size_t)ADJ_SPLIT * n));
    ADJ_CUDA(cudaMalloc((void **)&col, sizeof(double) * ((size_t)n + 1)));
    colsum_kernel<<<dim3((n + 255) / 256, ADJ_SPLIT), 256, 0, s>>>(c->d_A, part, n);
    colsum_fold_kernel<<<(n + 255) / 256, 256, 0, s>>>(part, col, n);
    max_kernel<<<1, 256, 0, s>>>(col, n, col + n);
    load_adjoint_kernel<<<(n + 255) / 256, 256, 0, s>>>(g, b, x, n);
    ADJ_CUDA(cudaGetLastError());
    ADJ_CUDA(cudaMemcpyAsync(&a1, col + n, sizeof(double), cudaMemcpyDeviceToHost, s));
    for (; it <= 30; ++it) {
        if (it == 0) {
            // x = 0: the residual is b (no pass over the matrix)
            ADJ_CUDA(cudaMemcpyAsync(r, b, sizeof(double) * n, cudaMemcpyDeviceToDevice, s));
        } else {
            split_kernel<<<(n + 255) / 256, 256, 0, s>>>(x, y, y + n, n);
            residual_t_part_kernel<<<dim3((n + 255) / 256, ADJ_SPLIT), 256, 0, s>>>(c->d_A, y, y + n, part, n);
            residual_t_fold_kernel<<<(n + 255) / 256, 256, 0, s>>>(part, b, r, n);
        }
        norms_kernel<<<1, 1024, 0, s>>>(r, x, b, n, nrm);
        ADJ_CUDA(cudaGetLastError());
        double h[3];
        ADJ_CUDA(cudaMemcpyAsync(h, nrm, sizeof h, cudaMemcpyDeviceToHost, s));
        ADJ_CUDA(cudaStreamSynchronize(s));
        be = h[0] / (a1 * h[1] + h[2] + 1e-300);
        if (be < 1e-12 || (be < 1e-9 && be > 0.5 * be_prev)) { status = OBEM_OK; break; }
        be_prev = be;
        if (it == 30) break;
        scale_to_float_kernel<<<(n + 255) / 256, 256, 0, s>>>(r, y, n, nrm);
        ADJ_CUDA(cudaGetLastError());
        rc = lu_solve_t(c, y, s);
        if (rc != OBEM_OK) goto done;
        axpy_unpermute_kernel<<<(n + 255) / 256, 256, 0, s>>>(x, y, c->d_perm, nrm, n);
        ADJ_CUDA(cudaGetLastError());
    }
    // mu = D nu: the row scale of the equilibrated system
    mu = (double *)malloc(sizeof(double) * (size_t)n);
    {
        double *ds = (double *)malloc(sizeof(double) * (size_t)n);
        if (!mu || !ds) { free(ds); rc = obem_fail(c, OBEM_ERR_ARG, "adjoint: host allocation failed"); goto done; }
        ADJ_CUDA(cudaMemcpyAsync(mu, x, sizeof(double) * n, cudaMemcpyDeviceToHost, s));
        ADJ_CUDA(cudaMemcpyAsync(ds, c->d_rowscale, sizeof(double) * n, cudaMemcpyDeviceToHost, s));
        ADJ_CUDA(cudaStreamSynchronize(s));
        for (int i = 0; i < n; ++i) mu[i] *= ds[i];
        free(ds);
    }
    if (dL_dgv) {
        for (int k = 0; k < c->n_groups; ++k) dL_dgv[k] = 0.0;
        for (int i = 0; i < n; ++i)
            if (c->h_kind[i] == OBEM_CELL_ELECTRODE && c->h_group[i] >= 0 && c->h_group[i] < c->n_groups)
                dL_dgv[c->h_group[i]] += mu[i];
    }
    if (dL_db) {
        float *hf = (float *)malloc(sizeof(float) * (size_t)n);
        if (!hf) { rc = obem_fail(c, OBEM_ERR_ARG, "adjoint: host allocation failed"); goto done; }
        for (int i = 0; i < n; ++i) hf[i] = (float)mu[i];
        cudaError_t e = cudaMemcpyAsync(dL_db, hf, sizeof(float) * n, cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        free(hf);
        ADJ_CUDA(e);
    }
    cudaEventRecord(e1, s);
    ADJ_CUDA(cudaStreamSynchronize(s));
    if (rep) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        rep->iterations = it;
        rep->status = status;
        rep->backward_error = be;
        rep->factor_ms = c->factor_ms;
        rep->solve_ms = ms;
    }
    if (status != OBEM_OK)
        rc = obem_fail(c, OBEM_ERR_NOT_CONVERGED, "adjoint refinement stopped at backward error %.3e after %d iterations",
                       be, it);
done:
#undef ADJ_CUDA
    free(mu);
    if (part) cudaFree(part);
    if (col) cudaFree(col);
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    return rc;
}
