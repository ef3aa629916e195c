// Field at few targets: one launch for the cells and one for the charges, no
// block list; the cells' targets in spatial order from OBEM_DIRECT_WIDE on.
//
// The block kernels of field.cu give a thread block 512 neighbouring targets
// and let it run over all cells (or all charges): at a few thousand targets,
// or targets spread over the chamber, that is a handful of blocks, or blocks
// with one or two live targets, each a serial pass over every cell.  Here the
// roles are swapped: a thread block holds 2 NP targets, its lanes run over the
// cells (or charges), each lane keeps the sums of its own cells for all the
// block's targets, and the lanes are added at the end.  Every SM has work from
// a few hundred targets on, and a target's own distance decides its near
// cells.  At many targets the block kernels win: they emit a cell's points
// once per 512 targets (cells) or evaluate a pair once for both charges.
//
// Bound: FP32 and rsqrt issue, 12 lane-operations and one rsqrt per point and
// target (two targets per f32x2 instruction); a lane's cell (84 bytes, from
// L2) is read once per 2 NP targets.
#include "obem_internal.cuh"
#include "direct_common.cuh"

#define DF_NBARY 140                // points of the 112- and the 28-point near rules

// this block's targets: slots [base, base + n) of the charge arrays, 0 < n <= T,
// and the range [lo, hi) of the live slots of their set (the launch's targets,
// or their chamber); false for a block without targets
template <bool BATCH, int T>
__device__ __forceinline__ bool df_targets(const FieldLaunch &L, const SymBatch &SB, int &base, int &n, int &lo,
                                           int &hi, int &cham)
{
    base = blockIdx.x * T;
    cham = 0;
    lo = 0;
    if (BATCH) {
        cham = SB.slot_cham[base / OBEM_SEG_ALIGN];
        lo = SB.seg_off[cham];
        hi = lo + SB.n[cham];
    } else {
        hi = L.nt_dev ? *L.nt_dev : L.nt;
    }
    n = min(T, hi - base);
    return n > 0;
}

// box of the block's targets (those with a position: fminf and fmaxf pass over a
// NaN) and its centre
template <int NP, int NW>
__device__ __forceinline__ float3 df_box(const DfShared<NP, NW> &sh, float (&lo)[3], float (&hi)[3])
{
#pragma unroll
    for (int c = 0; c < 3; ++c) { lo[c] = 3e38f; hi[c] = -3e38f; }
#pragma unroll
    for (int t = 0; t < 2 * NP; ++t) {
        const float4 x = sh.t[t];
        lo[0] = fminf(lo[0], x.x); lo[1] = fminf(lo[1], x.y); lo[2] = fminf(lo[2], x.z);
        hi[0] = fmaxf(hi[0], x.x); hi[1] = fmaxf(hi[1], x.y); hi[2] = fmaxf(hi[2], x.z);
    }
    return make_float3(0.5f * (lo[0] + hi[0]), 0.5f * (lo[1] + hi[1]), 0.5f * (lo[2] + hi[2]));
}

// E_out of the block's targets from the threads' slots
template <bool WANT_V, int NP, int NW>
__device__ __forceinline__ void df_finish(const FieldLaunch &L, DfShared<NP, NW> &sh, int n, int add)
{
    constexpr int V = DfShared<NP, NW>::V;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float s[V], c[V];
#pragma unroll
    for (int v = 0; v < V; ++v) { s[v] = sh.S[v][tid]; c[v] = sh.C[v][tid]; }
    df_reduce<V>(s, c);
    constexpr int per = 32 / V;
    if (lane % per == 0) { sh.red[0][warp][lane / per] = s[0]; sh.red[1][warp][lane / per] = c[0]; }
    __syncthreads();
    if (tid < 4 * n) {
        float S = 0.f, C = 0.f;
        for (int w = 0; w < NW; ++w) df_add(S, C, sh.red[0][w][tid], sh.red[1][w][tid]);
        const int k = tid & 3;
        float *out = reinterpret_cast<float *>(L.E_out + sh.ti[tid >> 2]) + k;
        float e0 = k == 0 ? L.e_ext.x : k == 1 ? L.e_ext.y : k == 2 ? L.e_ext.z : 0.f;
        if (add) e0 = *out;
        *out = (k < 3 || WANT_V) ? (float)((double)S + (double)C + (double)e0) : 0.f;
    }
}

// ---------------------------------------------------------------- cells
// A lane takes every (32 NW)-th cell.  Far cells (centroid at least 3 h from
// every target of the block) and the far targets of near cells: the rule of
// the block's nearest target, evaluated without divergence as up to seven
// points c, c + a g_k, c + b g_k (g_k: vertex - centroid) with the weights of
// the 1-, 3-, 4-, 6- or 7-point tier; a group of points that no lane of the
// warp needs is skipped.  Pairs closer than 3 h, by the target's own distance:
// the warp evaluates them together, a lane per quadrature point (28 points,
// 112 below 1.5 h), and pairs within h go to a per-warp queue of the
// closed form, 32 at a time.  All sums are formed in a fixed order.
// turn: not 0 where the kernel has the set, or NULL.
// perm: order of the targets (spatial, so that a block's targets are neighbours
// and share few near cells: 1e4 targets in a GEM of 5952 cells 1592 to 677 us),
// or NULL.
// GRP: cells in groups of 32.  A warp takes 32 groups at a time, a lane each
// tests whether the group is far from the block's targets, and these near enough
// to each other for its smallest cell; the far ones enter
// as their equivalent charges, a lane per charge of the list of all of them
// (1.5 points per lane and group, where the cells cost a point and its
// distances and weights), the others cell by cell: 60,000 targets in a GEM of
// 59,968 cells 14.8 to 11.6 ms.
template <bool WANT_V, bool BATCH, bool GRP, int NP, int NW>
__global__ void __launch_bounds__(32 * NW, NW == 8 ? 2 : 4)
direct_cells_kernel(FieldLaunch L, SymBatch SB, const int32_t *perm, CellGroups G, const int32_t *turn)
{
    if (turn && *turn == 0) return;
    constexpr int T = 2 * NP, TH = 32 * NW;
    __shared__ DfShared<NP, NW> sh;
    __shared__ float4 s_b[DF_NBARY];          // near rules: barycentric offsets of the points, weight
    __shared__ uint32_t s_q[NW][32 + T];      // closed-form queue: cell * 8 + target
    __shared__ u64 s_tp[3][NP];               // target packs
    __shared__ int s_nq[NW];
    constexpr int GW = GRP ? NW : 1, GL = GRP ? 32 : 1, GM = GRP ? OBEM_GRP_M : 1;
    __shared__ float4 s_u[GM], s_c[GW][GL];   // GRP: charges' directions; far groups' centres from the box centre, radii
    __shared__ int s_g[GW][GL];               // and numbers
    __shared__ u64 s_rp[3][NP];               // target packs from the box centre
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned below = (1u << lane) - 1u;
    int base, n, lo, hi, cham;
    if (!df_targets<BATCH, T>(L, SB, base, n, lo, hi, cham)) return;
    int poff = 0, np = L.panels.np;
    if (BATCH) {
        const int2 r = L.cham_pan[cham];
        poff = r.x;
        np = r.y;
    }
    const PanelsDev &P = L.panels;
    if (tid < T) {
        const int i = base + min(tid, n - 1);
        sh.ti[tid] = !BATCH && perm ? perm[i] : i;
        sh.t[tid] = L.targets[sh.ti[tid]];
    }
    for (int k = tid; k < DF_NBARY; k += TH) {
        float3 off;
        float wf;
        rule_point(k < 112 ? 2 : 1, k < 112 ? k : k - 112, make_float3(1.f, 0.f, 0.f), make_float3(0.f, 1.f, 0.f),
                   make_float3(0.f, 0.f, 1.f), off, wf);
        s_b[k] = make_float4(off.x, off.y, off.z, wf);
    }
#pragma unroll
    for (int v = 0; v < 4 * T; ++v) { sh.S[v][tid] = 0.f; sh.C[v][tid] = 0.f; }
    __syncthreads();
    if (tid < NP) {
        const float4 a = sh.t[2 * tid], b = sh.t[2 * tid + 1];
        s_tp[0][tid] = pk(a.x, b.x);
        s_tp[1][tid] = pk(a.y, b.y);
        s_tp[2][tid] = pk(a.z, b.z);
        if (GRP) {
            float blo[3], bhi[3];
            const float3 o = df_box(sh, blo, bhi);
            s_rp[0][tid] = pk(a.x - o.x, b.x - o.x);
            s_rp[1][tid] = pk(a.y - o.y, b.y - o.y);
            s_rp[2][tid] = pk(a.z - o.z, b.z - o.z);
        }
    }
    if (GRP)
        for (int k = tid; k < OBEM_GRP_M; k += TH) s_u[k] = G.u[k];
    __syncthreads();
    u64 A[4][NP];
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
        for (int p = 0; p < NP; ++p) A[c][p] = 0ull;
    int nq = 0;                               // queued pairs (warp-uniform, < 32)
    auto closed_pair = [&](uint32_t e) {
        const int j = (int)(e >> 3), t = (int)(e & 7u);
        const float4 x = sh.t[t];
        const float4 r = closed_terms(P.v64 + 9 * (size_t)j, P.geo ? P.geo + (size_t)OBEM_GEO64 * j : NULL,
                                      P.geo2 ? P.geo2 + (size_t)OBEM_GEO2 * j : NULL, x.x, x.y, x.z, L.sigma[j]);
        df_put(sh, 4 * t, r.x);
        df_put(sh, 4 * t + 1, r.y);
        df_put(sh, 4 * t + 2, r.z);
        if (WANT_V) df_put(sh, 4 * t + 3, r.w);
    };
    u64 D[3][NP], EP[NP];                     // target - centroid, softening of masked pairs
    auto point = [&](float ox, float oy, float oz, float w) {
        const u64 OX = pk(ox, ox), OY = pk(oy, oy), OZ = pk(oz, oz), W = pk(w, w);
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const u64 dx = sub2(D[0][p], OX), dy = sub2(D[1][p], OY), dz = sub2(D[2][p], OZ);
            const u64 r2 = fma2(dz, dz, fma2(dy, dy, fma2(dx, dx, EP[p])));
            float ra, rb;
            upk(r2, ra, rb);
            const u64 inv = pk(rsq(ra), rsq(rb));
            const u64 s = mul2(W, inv);
            const u64 s3 = mul2(s, mul2(inv, inv));
            A[0][p] = fma2(dx, s3, A[0][p]);
            A[1][p] = fma2(dy, s3, A[1][p]);
            A[2][p] = fma2(dz, s3, A[2][p]);
            if (WANT_V) A[3][p] = add2(A[3][p], s);
        }
    };
    int since = 0;
    // the warp's 32 cells (a lane each; live: the lane has one)
    auto cells32 = [&](int j, bool live) {
        const float4 ca = P.c_a[j], cl = P.c_lo[j], g0 = P.g0_h[j], g1 = P.g1[j], g2 = P.g2[j];
        const float q = live ? ca.w * L.sigma[j] : 0.f;
        const float h2 = g0.w;
        // target - centroid of every pair (exact for nearby targets)
        unsigned nm = 0u;                     // near targets of this lane's cell
        float dmin = 3e38f;
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            D[0][p] = sub2(sub2(s_tp[0][p], pk(ca.x, ca.x)), pk(cl.x, cl.x));
            D[1][p] = sub2(sub2(s_tp[1][p], pk(ca.y, ca.y)), pk(cl.y, cl.y));
            D[2][p] = sub2(sub2(s_tp[2][p], pk(ca.z, ca.z)), pk(cl.z, cl.z));
            float da, db;
            upk(fma2(D[2][p], D[2][p], fma2(D[1][p], D[1][p], mul2(D[0][p], D[0][p]))), da, db);
            dmin = fminf(dmin, fminf(da, db));
            const bool na = da < TIER_7PT_H2 * h2, nb = db < TIER_7PT_H2 * h2;
            nm |= (na ? 1u << (2 * p) : 0u) | (nb ? 2u << (2 * p) : 0u);
            // near pairs get no term here (a distance of 1e15 m)
            EP[p] = pk(na ? 1e30f : 0.f, nb ? 1e30f : 0.f);
        }
        if (!live) nm = 0u;
        nm &= (1u << n) - 1u;                 // padding repeats the last target
        const bool t1 = dmin >= TIER_1PT_H2 * h2, t3 = dmin >= TIER_3PT_H2 * h2, t4 = dmin >= TIER_4PT_H2 * h2,
                   t6 = dmin >= TIER_6PT_H2 * h2;
        const float w0 = t1 ? 1.f : t3 ? 0.f : t4 ? -27.0f / 48.0f : t6 ? 0.f : D7_W0;
        const float wa = t1 ? 0.f : t3 ? 1.0f / 3.0f : t4 ? 25.0f / 48.0f : t6 ? 0.223381589678011f : D7_W1;
        const float sa = t1 ? 0.f : t3 ? 0.5f : t4 ? 0.4f : t6 ? -0.33784547274789500f : D7_T1;
        const float wb = t4 ? 0.f : t6 ? 0.109951743655322f : D7_W2;
        const float sb = t4 ? 0.f : t6 ? 0.72527135947068800f : D7_T2;
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
        // near cells, one after the other: a lane per quadrature point
        unsigned near = __ballot_sync(0xffffffffu, nm != 0u);
        if (near) since = DF_FOLD - 1;                                  // fold their terms at once
        while (near) {
            const int src = __ffs(near) - 1, jj = __shfl_sync(0xffffffffu, j, src);      // warp-uniform
            near &= near - 1;
            const unsigned m = __shfl_sync(0xffffffffu, nm, src);
            const float4 c = P.c_a[jj], l = P.c_lo[jj], v0 = P.g0_h[jj], v1 = P.g1[jj], v2 = P.g2[jj];
            const float qq = c.w * L.sigma[jj];
            unsigned in_h = 0u, fine = 0u;
#pragma unroll
            for (int p = 0; p < NP; ++p) {
                D[0][p] = sub2(sub2(s_tp[0][p], pk(c.x, c.x)), pk(l.x, l.x));
                D[1][p] = sub2(sub2(s_tp[1][p], pk(c.y, c.y)), pk(l.y, l.y));
                D[2][p] = sub2(sub2(s_tp[2][p], pk(c.z, c.z)), pk(l.z, l.z));
                float da, db;
                upk(fma2(D[2][p], D[2][p], fma2(D[1][p], D[1][p], mul2(D[0][p], D[0][p]))), da, db);
                in_h |= (da < v0.w ? 1u << (2 * p) : 0u) | (db < v0.w ? 2u << (2 * p) : 0u);
                fine |= (da < 2.25f * v0.w ? 1u << (2 * p) : 0u) | (db < 2.25f * v0.w ? 2u << (2 * p) : 0u);
            }
            const unsigned closed = m & in_h, quad = m & ~in_h;
            if (closed) {
                if ((closed >> lane) & 1u) s_q[warp][nq + __popc(closed & below)] = ((uint32_t)jj << 3) | (uint32_t)lane;
                nq += __popc(closed);
                if (nq >= 32) {
                    __syncwarp();
                    closed_pair(s_q[warp][lane]);
                    __syncwarp();
                    nq -= 32;
                    if (lane < nq) s_q[warp][lane] = s_q[warp][32 + lane];
                    __syncwarp();
                }
            }
            if (quad) {
#pragma unroll
                for (int p = 0; p < NP; ++p)
                    EP[p] = pk((quad >> (2 * p)) & 1u ? 0.f : 1e30f, (quad >> (2 * p + 1)) & 1u ? 0.f : 1e30f);
                const bool coarse = (quad & fine) == 0u;                  // every target 1.5 h away
                for (int k = coarse ? 112 + lane : lane; k < (coarse ? 140 : 112); k += 32) {
                    const float4 b = s_b[k];
                    point(fmaf(b.z, v2.x, fmaf(b.y, v1.x, b.x * v0.x)), fmaf(b.z, v2.y, fmaf(b.y, v1.y, b.x * v0.y)),
                          fmaf(b.z, v2.z, fmaf(b.y, v1.z, b.x * v0.z)), qq * b.w);
                }
            }
        }
        if (++since == DF_FOLD) {
            df_fold<WANT_V>(sh, A, 1.f);
            since = 0;
        }
    };
    if (!GRP) {
        for (int jb = 32 * warp; jb < np; jb += TH) {
            const bool live = jb + lane < np;
            cells32(poff + (live ? jb + lane : jb), live);
        }
    } else {
        float blo[3], bhi[3];
        const float3 o = df_box(sh, blo, bhi);
        const float ex = bhi[0] - o.x, ey = bhi[1] - o.y, ez = bhi[2] - o.z;
        const float hmin2 = (FRAME_H * FRAME_H) * (ex * ex + ey * ey + ez * ez);
        // group (32 i + lane) NW + warp: neighbours, which are near together, on different warps
        for (int gb = 0; gb * NW < G.ng; gb += 32) {
            const int g = (gb + lane) * NW + warp;
            const bool have = g < G.ng;
            const float4 cr = G.cr[have ? g : 0];
            const float gx = fmaxf(fmaxf(blo[0] - cr.x, cr.x - bhi[0]), 0.f),
                        gy = fmaxf(fmaxf(blo[1] - cr.y, cr.y - bhi[1]), 0.f),
                        gz = fmaxf(fmaxf(blo[2] - cr.z, cr.z - bhi[2]), 0.f);
            const bool far = gx * gx + gy * gy + gz * gz >= OBEM_GRP_THETA2 * (cr.w * cr.w) && G.h2min[have ? g : 0] >= hmin2;
            const unsigned fm = __ballot_sync(0xffffffffu, have && far);
            unsigned nm = __ballot_sync(0xffffffffu, have && !far);
            __syncwarp();
            if (have && far) {
                const int k = __popc(fm & below);
                s_c[warp][k] = make_float4(cr.x - o.x, cr.y - o.y, cr.z - o.z, cr.w);
                s_g[warp][k] = g;
            }
            __syncwarp();
            const int nc = __popc(fm) * OBEM_GRP_M;
            for (int e0 = 0; e0 < nc; e0 += 32) {
                const int e = e0 + lane;
                const bool in = e < nc;
                const int gi = in ? e / OBEM_GRP_M : 0, k = in ? e - gi * OBEM_GRP_M : 0;
                const float4 c = s_c[warp][gi], u = s_u[k];
                const float w = in ? G.q[(size_t)s_g[warp][gi] * OBEM_GRP_M + k] : 0.f;
                const float sx = fmaf(c.w, u.x, c.x), sy = fmaf(c.w, u.y, c.y), sz = fmaf(c.w, u.z, c.z);
                const u64 SX = pk(sx, sx), SY = pk(sy, sy), SZ = pk(sz, sz), W = pk(w, w);
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    const u64 dx = sub2(s_rp[0][p], SX), dy = sub2(s_rp[1][p], SY), dz = sub2(s_rp[2][p], SZ);
                    const u64 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
                    float ra, rb;
                    upk(r2, ra, rb);
                    const u64 inv = pk(rsq(ra), rsq(rb));
                    const u64 sw = mul2(W, inv);
                    const u64 s3 = mul2(sw, mul2(inv, inv));
                    A[0][p] = fma2(dx, s3, A[0][p]);
                    A[1][p] = fma2(dy, s3, A[1][p]);
                    A[2][p] = fma2(dz, s3, A[2][p]);
                    if (WANT_V) A[3][p] = add2(A[3][p], sw);
                }
                if (++since == DF_FOLD) {
                    df_fold<WANT_V>(sh, A, 1.f);
                    since = 0;
                }
            }
            while (nm) {
                const int slot = 32 * ((gb + __ffs(nm) - 1) * NW + warp);         // warp-uniform
                nm &= nm - 1;
                const bool live = slot + lane < np;
                cells32(G.perm[live ? slot + lane : slot], live);
            }
        }
    }
    df_fold<WANT_V>(sh, A, 1.f);
    // what is left in the warps' queues, together (in warp order): a warp each
    // for its few would cost as many instructions as for 32
    if (lane == 0) s_nq[warp] = nq;
    __syncthreads();
    {
        int e = tid, w = 0;
        while (w < NW && e >= s_nq[w]) e -= s_nq[w++];
        if (w < NW) closed_pair(s_q[w][e]);
    }
    __syncthreads();
    df_finish<WANT_V>(L, sh, n, 0);
}

// ---------------------------------------------------------------- charges
// A lane takes every (32 NW)-th charge; add: on top of E_out (else e_ext).
template <bool WANT_V, int NP, int NW>
__global__ void __launch_bounds__(32 * NW, NP == 1 ? 2 : 4)
direct_pairs_kernel(FieldLaunch L, int add)
{
    constexpr int T = 2 * NP, TH = 32 * NW;
    __shared__ DfShared<NP, NW> sh;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int base = blockIdx.x * T, n = min(T, (L.nt_dev ? *L.nt_dev : L.nt) - base);
    if (n <= 0) return;
    const int ns = L.ns_dev ? *L.ns_dev : L.ns;
    if (tid < T) {
        sh.ti[tid] = base + min(tid, n - 1);
        sh.t[tid] = L.targets[sh.ti[tid]];
    }
#pragma unroll
    for (int v = 0; v < 4 * T; ++v) { sh.S[v][tid] = 0.f; sh.C[v][tid] = 0.f; }
    __syncthreads();
    u64 TX[NP], TY[NP], TZ[NP], A[4][NP];
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const float4 a = sh.t[2 * p], b = sh.t[2 * p + 1];
        TX[p] = pk(a.x * DF_XS, b.x * DF_XS);
        TY[p] = pk(a.y * DF_XS, b.y * DF_XS);
        TZ[p] = pk(a.z * DF_XS, b.z * DF_XS);
#pragma unroll
        for (int c = 0; c < 4; ++c) A[c][p] = 0ull;
    }
    const float kC = (float)OBEM_KC * DF_QS, eps2 = L.eps2 * DF_QS;
    // first charge of the block's own targets, out of reach when they are not charges
    const int own = L.self_exclude ? base + L.self_off : 0x7fffffff - T;
    int since = 0;
    const float4 none = make_float4(1e6f, 1e6f, 1e6f, 0.f);
    float4 nx = tid < ns ? L.sources[tid] : none;
    for (int ib = 32 * warp; ib < ns; ib += TH) {
        const float4 src = nx;
        const int i = ib + lane;
        nx = i + TH < ns ? L.sources[i + TH] : none;
        if (ib + 32 > own && ib < own + T) df_source<WANT_V, true>(TX, TY, TZ, src, kC, eps2, i - own, A);   // uniform
        else df_source<WANT_V, false>(TX, TY, TZ, src, kC, eps2, 0, A);
        if (++since == DF_FOLD) {
            df_fold<WANT_V>(sh, A, DF_VS);
            since = 0;
        }
    }
    df_fold<WANT_V>(sh, A, DF_VS);
    __syncthreads();
    df_finish<WANT_V>(L, sh, n, add);
}

// Targets per block: 8 (four packs, 4 warps), fewer below OBEM_DIRECT_WIDE
// targets, where blocks of 8 would leave warps idle.  Cells: 2 targets and 8 warps
// as long as those blocks fit the SMs at once (two per SM), then 2 targets and 4
// warps (four per SM: no second wave at 1000), 4 targets and 8 warps for many
// cells, whose loads a block shares.  Measured (us) at 600 and 2000 targets, 2 and
// 8 / 2 and 4 / 4 and 8: 1024 cells 55 / 68 / 72 and 148 / 125 / 144, 15,888 cells
// 147 / 202 / 204 and 448 / 437 / 479, 59,968 cells 223 / 326 / 260 and 681 / 718 /
// 619.
#define DF_ONE_WAVE 608

int obem_launch_direct_cells(obem_ctx *ctx, const FieldLaunch &L, const SymBatch *SB, int slots, const int32_t *perm,
                             const CellGroups *GR, const int32_t *turn, cudaStream_t s)
{
    SymBatch none;
    memset(&none, 0, sizeof none);
    const SymBatch &B = SB ? *SB : none;
    CellGroups G;
    memset(&G, 0, sizeof G);
    if (GR) G = *GR;
    if (SB) {
        direct_cells_kernel<false, true, false, 4, 4><<<(slots + 7) / 8, 128, 0, s>>>(L, B, NULL, G, turn);
    } else if (slots >= OBEM_DIRECT_WIDE) {
        const int g = (slots + 7) / 8;
        if (GR) {
            if (L.want_v) direct_cells_kernel<true, false, true, 4, 4><<<g, 128, 0, s>>>(L, B, perm, G, turn);
            else direct_cells_kernel<false, false, true, 4, 4><<<g, 128, 0, s>>>(L, B, perm, G, turn);
        } else if (L.want_v) {
            direct_cells_kernel<true, false, false, 4, 4><<<g, 128, 0, s>>>(L, B, perm, G, turn);
        } else {
            direct_cells_kernel<false, false, false, 4, 4><<<g, 128, 0, s>>>(L, B, perm, G, turn);
        }
    } else if (slots <= DF_ONE_WAVE) {
        const int g = (slots + 1) / 2;
        if (L.want_v) direct_cells_kernel<true, false, false, 1, 8><<<g, 256, 0, s>>>(L, B, perm, G, turn);
        else direct_cells_kernel<false, false, false, 1, 8><<<g, 256, 0, s>>>(L, B, perm, G, turn);
    } else if (L.panels.np < 32768) {
        const int g = (slots + 1) / 2;
        if (L.want_v) direct_cells_kernel<true, false, false, 1, 4><<<g, 128, 0, s>>>(L, B, perm, G, turn);
        else direct_cells_kernel<false, false, false, 1, 4><<<g, 128, 0, s>>>(L, B, perm, G, turn);
    } else {
        const int g = (slots + 3) / 4;
        if (L.want_v) direct_cells_kernel<true, false, false, 2, 8><<<g, 256, 0, s>>>(L, B, perm, G, turn);
        else direct_cells_kernel<false, false, false, 2, 8><<<g, 256, 0, s>>>(L, B, perm, G, turn);
    }
    OBEM_LAUNCH(ctx);
    return OBEM_OK;
}

int obem_launch_direct_pairs(obem_ctx *ctx, const FieldLaunch &L, int slots, int add, cudaStream_t s)
{
    if (slots >= OBEM_DIRECT_WIDE) {
        const int g = (slots + 7) / 8;
        if (L.want_v) direct_pairs_kernel<true, 4, 4><<<g, 128, 0, s>>>(L, add);
        else direct_pairs_kernel<false, 4, 4><<<g, 128, 0, s>>>(L, add);
    } else {
        const int g = (slots + 1) / 2;
        if (L.want_v) direct_pairs_kernel<true, 1, 8><<<g, 256, 0, s>>>(L, add);
        else direct_pairs_kernel<false, 1, 8><<<g, 256, 0, s>>>(L, add);
    }
    OBEM_LAUNCH(ctx);
    return OBEM_OK;
}
