// Approximate N-body field (Sec. 3.2.4, the nearest-neighbour "NN" option of
// the paper, O(N) in the number of charges for a fixed grid): the exact
// Coulomb sum of Eq. (nbody) over the charges near a particle, charge centres
// for the farther ones.  The paper gives one sentence; the reading built here:
//   - cubic cells of edge W / G (W: the largest extent of the charges'
//     bounding box, G cells per axis); the cell of a charge is
//     floor((x - lo) * (G / W)) per axis, computed in binary32 with one
//     rounding per operation and clamped to 0..G-1;
//   - near: the exact softened pair sum over the charges of the 27 cells
//     around the particle's cell, itself excluded;
//   - far: every other cell contributes its positive and its negative charge
//     separately, each as the total charge at its charge-weighted centre.
// Pipeline: bounding box (min/max reductions on order-preserving integer
// images of the floats), cell of every charge + counts, exclusive scans
// (charges, occupied cells, groups of 8 charges), counting-sort scatter of the
// positions, per-cell aggregates of the occupied cells (FP64 sums), and the
// field.
//
// Field: a warp takes up to 8 charges of one cell (four f32x2 packs) and its
// lanes run over the sources.  The 27 cells around are 9 contiguous runs of
// the sorted charges (three cells in x each), and their centres 9 runs of the
// list of occupied cells' centres, so the far cells are the stretches between
// those runs: both sums are coalesced reads with no test per source.  Bound:
// FP32 issue (12 lane-operations and one rsqrt per charge and source); the four
// warps of a block mostly share their cell, so their sources hit in L1.
#include "obem_internal.cuh"
#include "direct_common.cuh"

#define NN_THREADS 256
#define NN_T 8                     // targets per warp
#define NN_FW 4                    // warps per block of the field kernel
#define NN_AT 128                  // threads per cell of the aggregates

// float <-> integer with the same order (for atomic min / max)
__device__ __forceinline__ int nn_ford(float f)
{
    int i = __float_as_int(f);
    return i >= 0 ? i : i ^ 0x7fffffff;
}
__device__ __forceinline__ float nn_fval(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

__global__ void nn_bbox_init_kernel(int *bb)
{
    if (threadIdx.x < 3) bb[threadIdx.x] = 0x7fffffff;              // min
    else if (threadIdx.x < 6) bb[threadIdx.x] = (int)0x80000000;    // max
    else if (threadIdx.x == 6) bb[6] = 0;                           // largest |q| (bits)
}

// bounding box of the charges and their largest |q|
__global__ void nn_bbox_kernel(const float4 *pos, const int32_t *n_dev, int n, int *bb)
{
    const int nn = n_dev ? *n_dev : n;
    float mn[3] = {INFINITY, INFINITY, INFINITY}, mx[3] = {-INFINITY, -INFINITY, -INFINITY}, mq = 0.f;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < nn; i += gridDim.x * blockDim.x) {
        const float4 p = pos[i];
        mn[0] = fminf(mn[0], p.x); mn[1] = fminf(mn[1], p.y); mn[2] = fminf(mn[2], p.z);
        mx[0] = fmaxf(mx[0], p.x); mx[1] = fmaxf(mx[1], p.y); mx[2] = fmaxf(mx[2], p.z);
        mq = fmaxf(mq, fabsf(p.w));
    }
    for (int o = 16; o; o >>= 1) mq = fmaxf(mq, __shfl_xor_sync(0xffffffffu, mq, o));
#pragma unroll
    for (int a = 0; a < 3; ++a)
        for (int o = 16; o; o >>= 1) {
            mn[a] = fminf(mn[a], __shfl_xor_sync(0xffffffffu, mn[a], o));
            mx[a] = fmaxf(mx[a], __shfl_xor_sync(0xffffffffu, mx[a], o));
        }
    // one atomic per block and bound (per warp they serialised on six words)
    __shared__ float red[7][NN_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        for (int a = 0; a < 3; ++a) { red[a][warp] = mn[a]; red[3 + a][warp] = mx[a]; }
        red[6][warp] = mq;
    }
    __syncthreads();
    if (threadIdx.x < 6) {
        float v = red[threadIdx.x][0];
        for (int w = 1; w < NN_THREADS / 32; ++w)
            v = threadIdx.x < 3 ? fminf(v, red[threadIdx.x][w]) : fmaxf(v, red[threadIdx.x][w]);
        if (threadIdx.x < 3 ? v < INFINITY : v > -INFINITY) {
            if (threadIdx.x < 3) atomicMin(&bb[threadIdx.x], nn_ford(v));
            else atomicMax(&bb[threadIdx.x], nn_ford(v));
        }
    } else if (threadIdx.x == 6) {
        float v = red[6][0];
        for (int w = 1; w < NN_THREADS / 32; ++w) v = fmaxf(v, red[6][w]);
        atomicMax(&bb[6], __float_as_int(v));
    }
}

struct NnGrid {
    float lo[3], inv;
    int G;
};

__device__ __forceinline__ NnGrid nn_grid(const int *bb, int G)
{
    NnGrid g;
    float wmax = 0.0f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        g.lo[a] = nn_fval(bb[a]);
        const float w = __fsub_rn(nn_fval(bb[3 + a]), g.lo[a]);
        wmax = w > wmax ? w : wmax;
    }
    if (!(wmax > 0.0f)) wmax = 1.0f;
    g.inv = __fdiv_rn((float)G, wmax);
    g.G = G;
    return g;
}

__device__ __forceinline__ int nn_coord(const NnGrid &g, float x, int a)
{
    const float t = __fmul_rn(__fsub_rn(x, g.lo[a]), g.inv);
    int k = (int)floorf(t);
    return k < 0 ? 0 : (k > g.G - 1 ? g.G - 1 : k);
}

// cell of every charge (packed cx | cy << 10 | cz << 20) and counts
__global__ void nn_cell_kernel(const float4 *pos, const int32_t *n_dev, int n, const int *bb, int G, int32_t *cell,
                               int32_t *count)
{
    const int nn = n_dev ? *n_dev : n;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nn) return;
    const NnGrid g = nn_grid(bb, G);
    const float4 p = pos[i];
    const int cx = nn_coord(g, p.x, 0), cy = nn_coord(g, p.y, 1), cz = nn_coord(g, p.z, 2);
    cell[i] = cx | (cy << 10) | (cz << 20);
    atomicAdd(&count[(cz * G + cy) * G + cx], 1);
}

// exclusive scans over the cells, nc + 1 entries each: start (charges; cursor
// is a copy), occ (occupied cells), grp (groups of up to NN_T charges)
__global__ void __launch_bounds__(1024) nn_scan_kernel(const int32_t *count, int nc, int32_t *start, int32_t *cursor,
                                                       int32_t *occ, int32_t *grp)
{
    __shared__ int32_t s_warp[32];
    int32_t carry[3] = {0, 0, 0};
    for (int base = 0; base < nc; base += 1024) {
        const int q = base + threadIdx.x;
        const int32_t n = q < nc ? count[q] : 0;
        const int32_t v[3] = {n, n > 0, (n + NN_T - 1) / NN_T};
        int32_t *const out[3] = {start, occ, grp};
        for (int k = 0; k < 3; ++k) {
            const int32_t inc = block_scan_1024(v[k], s_warp);
            if (q < nc) out[k][q] = carry[k] + inc - v[k];
            if (k == 0 && q < nc) cursor[q] = carry[0] + inc - v[0];
            carry[k] += s_warp[31];
        }
    }
    if (threadIdx.x == 0) {
        start[nc] = carry[0];
        occ[nc] = carry[1];
        grp[nc] = carry[2];
    }
}

__global__ void nn_scatter_kernel(const float4 *pos, const int32_t *n_dev, int n, const int32_t *cell, int G,
                                  int32_t *cursor, int32_t *sorted, float4 *spos)
{
    const int nn = n_dev ? *n_dev : n;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nn) return;
    const int32_t c = cell[i];
    const int idx = (((c >> 20) & 1023) * G + ((c >> 10) & 1023)) * G + (c & 1023);
    const int k = atomicAdd(&cursor[idx], 1);
    const float4 p = pos[i];
    sorted[k] = i;
    // a charge without a position (NaN) gives and gets no term: no charge, and out
    // of reach (its squared distance to any other is infinite, 1/r 0)
    spos[k] = isnan(p.x) || isnan(p.y) || isnan(p.z) ? make_float4(1e18f, 1e18f, 1e18f, 0.f) : p;
}

// per occupied cell: positive and negative charge centres (x, y, z, k_C Q) at
// agg[2 occ], agg[2 occ + 1] (no charge of a sign: weight 0), and the cell's
// groups (cell, first sorted charge).  One block per cell: a thread per cell
// took 11.7 ms at 3e5 charges, the densest cell's serial FP64 sum.
__global__ void __launch_bounds__(NN_AT) nn_agg_kernel(const float4 *spos, const int32_t *start, const int32_t *occ,
                                                       const int32_t *grp, float4 *agg, int2 *groups)
{
    __shared__ double red[NN_AT / 32][8];
    const int c = blockIdx.x;
    const int k0 = start[c], k1 = start[c + 1];
    if (k0 == k1) return;
    double s[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    for (int k = k0 + threadIdx.x; k < k1; k += NN_AT) {
        const float4 p = spos[k];
        const double q = (double)p.w;
        if (p.w >= 0.0f) { s[0] += q * p.x; s[1] += q * p.y; s[2] += q * p.z; s[3] += q; }
        else { s[4] += q * p.x; s[5] += q * p.y; s[6] += q * p.z; s[7] += q; }
    }
#pragma unroll
    for (int f = 0; f < 8; ++f)
        for (int o = 16; o; o >>= 1) s[f] += __shfl_xor_sync(0xffffffffu, s[f], o);
    if ((threadIdx.x & 31) == 0)
        for (int f = 0; f < 8; ++f) red[threadIdx.x >> 5][f] = s[f];
    __syncthreads();
    if (threadIdx.x < 2) {
        double t[4];
        for (int f = 0; f < 4; ++f) {
            t[f] = red[0][4 * threadIdx.x + f];
            for (int w = 1; w < NN_AT / 32; ++w) t[f] += red[w][4 * threadIdx.x + f];
        }
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        if (t[3] != 0.0) a = make_float4((float)(t[0] / t[3]), (float)(t[1] / t[3]), (float)(t[2] / t[3]),
                                         (float)(OBEM_KC * t[3]));
        agg[2 * occ[c] + threadIdx.x] = a;
    }
    const int g0 = grp[c];
    for (int g = threadIdx.x; g * NN_T < k1 - k0; g += NN_AT) groups[g0 + g] = make_int2(c, k0 + g * NN_T);
}

// Field at every charge: warp g takes group g.  E_out adds to its initial
// value when add is set, else starts from e_ext.  A pair at zero distance
// gives no term: eps2 (x 2^80) is at least what keeps k_C q / r^3 of the largest
// charge (bb[6]) finite, so that its product with the distance is 0.  That is a
// distance of 2.3e-20 m x (q / e)^(1/3), below 1.5e-4 of any at which
// k_C q / r^3 itself fits binary32: the other pairs keep their bits.  (A floor
// without regard to the charges left binary32 from 195 e on; a test of every
// pair of a cell for it took 3 % of the kernel.)
__global__ void __launch_bounds__(32 * NN_FW, 4)
nn_field_kernel(const int32_t *start, const int32_t *occ, const int32_t *grp, const int2 *groups, const int32_t *sorted,
                const float4 *spos, const float4 *agg, const int *bb, int G, float eps2, float4 *E_out, float3 e_ext, int add)
{
    constexpr int NP = NN_T / 2;
    __shared__ DfShared<NP, NN_FW> sh;
    const int nc = G * G * G;
    const int lane = threadIdx.x & 31;
    const int g = blockIdx.x * NN_FW + (threadIdx.x >> 5);
    if (g >= grp[nc]) return;                               // warp-uniform; only warp barriers below
    const int2 gr = groups[g];
    const int c = gr.x, base = gr.y;
    const int n = min(NN_T, start[c + 1] - base);
    {
        const float f = 2.15443469e-13f * cbrtf(fminf((float)OBEM_KC * __int_as_float(bb[6]) * DF_QS, 3.4e38f));   // (1e-38 k_C q)^(1/3)
        eps2 = fmaxf(eps2, fmaxf(f * f, 1e-30f));
    }
    u64 TX[NP], TY[NP], TZ[NP], A[4][NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const float4 a = spos[base + min(2 * p, n - 1)], b = spos[base + min(2 * p + 1, n - 1)];
        TX[p] = pk(a.x * DF_XS, b.x * DF_XS);
        TY[p] = pk(a.y * DF_XS, b.y * DF_XS);
        TZ[p] = pk(a.z * DF_XS, b.z * DF_XS);
#pragma unroll
        for (int k = 0; k < 4; ++k) A[k][p] = 0ull;
    }
#pragma unroll
    for (int v = 0; v < 4 * NN_T; ++v) { sh.S[v][threadIdx.x] = 0.f; sh.C[v][threadIdx.x] = 0.f; }
    const float4 none = make_float4(1e6f, 1e6f, 1e6f, 0.f);
    int since = 0;
    // the sources [b, e) of src with weights kC w
    auto run = [&](const float4 *src, int b, int e, float kC) {
        float4 nx = b + lane < e ? src[b + lane] : none;
        for (int ib = b; ib < e; ib += 32) {
            const float4 x = nx;
            nx = ib + 32 + lane < e ? src[ib + 32 + lane] : none;
            if (src == spos && ib + 32 > base && ib < base + NN_T)
                df_source<false, true>(TX, TY, TZ, x, kC, eps2, ib + lane - base, A);
            else
                df_source<false, false>(TX, TY, TZ, x, kC, eps2, 0, A);
            if (++since == DF_FOLD) {
                df_fold<false>(sh, A, 1.f);
                since = 0;
            }
        }
    };
    const int cx = c % G, cy = (c / G) % G, cz = c / (G * G);
    const int x0 = max(cx - 1, 0), x1 = min(cx + 1, G - 1);
    int fe = 0;                                             // centres before fe are done
    for (int z = max(cz - 1, 0); z <= min(cz + 1, G - 1); ++z)
        for (int y = max(cy - 1, 0); y <= min(cy + 1, G - 1); ++y) {
            const int r = (z * G + y) * G;
            run(agg, fe, 2 * occ[r + x0], DF_QS);
            fe = 2 * occ[r + x1 + 1];
            run(spos, start[r + x0], start[r + x1 + 1], (float)OBEM_KC * DF_QS);
        }
    run(agg, fe, 2 * occ[nc], DF_QS);
    df_fold<false>(sh, A, 1.f);
    float s[4 * NN_T], cc[4 * NN_T];
#pragma unroll
    for (int v = 0; v < 4 * NN_T; ++v) { s[v] = sh.S[v][threadIdx.x]; cc[v] = sh.C[v][threadIdx.x]; }
    df_reduce<4 * NN_T>(s, cc);                             // lane l: component l % 4 of target l / 4
    const int t = lane >> 2, k = lane & 3;
    if (t < n) {
        float *out = reinterpret_cast<float *>(E_out + sorted[base + t]) + k;
        float e0 = k == 0 ? e_ext.x : k == 1 ? e_ext.y : e_ext.z;
        if (add) e0 = *out;
        *out = k < 3 ? (float)((double)s[0] + (double)cc[0] + (double)e0) : 0.f;
    }
}

int obem_launch_nbody_nn(obem_ctx *c, const float4 *pos, const int32_t *n_dev, int n, int G, float eps2,
                         float4 *E_out, float3 e_ext, int add, cudaStream_t s)
{
    if (n <= 0) return OBEM_OK;
    if (G < 1 || G > OBEM_NN_GMAX) return obem_fail(c, OBEM_ERR_ARG, "nbody NN: grid %d outside 1..%d", G, OBEM_NN_GMAX);
    const int nc = G * G * G;
    const int nb = (n + NN_THREADS - 1) / NN_THREADS;
    nn_bbox_init_kernel<<<1, 32, 0, s>>>(c->nn_bbox);
    nn_bbox_kernel<<<nb < 1024 ? nb : 1024, NN_THREADS, 0, s>>>(pos, n_dev, n, c->nn_bbox);
    OBEM_CUDA(c, cudaMemsetAsync(c->nn_count, 0, sizeof(int32_t) * nc, s));
    nn_cell_kernel<<<nb, NN_THREADS, 0, s>>>(pos, n_dev, n, c->nn_bbox, G, c->nn_cell, c->nn_count);
    nn_scan_kernel<<<1, 1024, 0, s>>>(c->nn_count, nc, c->nn_start, c->nn_cursor, c->nn_occ, c->nn_grp);
    nn_scatter_kernel<<<nb, NN_THREADS, 0, s>>>(pos, n_dev, n, c->nn_cell, G, c->nn_cursor, c->nn_sorted, c->nn_spos);
    nn_agg_kernel<<<nc, NN_AT, 0, s>>>(c->nn_spos, c->nn_start, c->nn_occ, c->nn_grp, c->nn_agg, c->nn_groups);
    const int ng = n / NN_T + (n < nc ? n : nc);
    nn_field_kernel<<<(ng + NN_FW - 1) / NN_FW, 32 * NN_FW, 0, s>>>(
        c->nn_start, c->nn_occ, c->nn_grp, c->nn_groups, c->nn_sorted, c->nn_spos, c->nn_agg, c->nn_bbox, G,
        eps2 * DF_QS, E_out, e_ext, add);
    OBEM_LAUNCH(c);
    return OBEM_OK;
}
