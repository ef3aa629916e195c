// Device helpers of the kernels whose lanes run over the sources while a block
// (or a warp) holds a few targets: per-thread compensated sums in shared
// memory, the sum over the lanes, and the point-charge term of a source.
#pragma once
#include "field_common.cuh"

#define DF_FOLD 16                  // lane iterations summed in FP32 between compensated folds
#define DF_SELF 3.0e38f             // squared distance (x 2^80) given to a target's own charge
// Charges: positions x 2^40 and k_C q x 2^80 (exact), as in the symmetric
// kernel, so that close pairs stay finite; the potential carries 2^40
#define DF_XS 1099511627776.0f
#define DF_QS 1208925819614629174706176.0f
#define DF_VS 9.094947017729282e-13f

// (s, c) += (s2, c2), both unevaluated sums of two binary32 numbers
__device__ __forceinline__ void df_add(float &s, float &c, float s2, float c2)
{
    float e = 0.f;
    two_sum_acc(s, e, s2);
    c = __fadd_rn(c, __fadd_rn(e, c2));
}

// Sums v[0 .. V) over the warp's lanes: each step halves the values a lane
// holds and exchanges the other half, so 32 values cost 31 additions instead
// of 160; lane l ends with the total of value l >> (5 - log2 V).
template <int V>
__device__ __forceinline__ void df_reduce(float (&s)[V], float (&c)[V])
{
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int n = V; n > 1; n >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < n / 2; ++k) {
            const float ss = up ? s[k] : s[k + n / 2], sc = up ? c[k] : c[k + n / 2];
            float ks = up ? s[k + n / 2] : s[k], kc = up ? c[k + n / 2] : c[k];
            df_add(ks, kc, __shfl_xor_sync(0xffffffffu, ss, o), __shfl_xor_sync(0xffffffffu, sc, o));
            s[k] = ks;
            c[k] = kc;
        }
    }
    for (; o > 0; o >>= 1) {
        const float ss = __shfl_xor_sync(0xffffffffu, s[0], o), sc = __shfl_xor_sync(0xffffffffu, c[0], o);
        df_add(s[0], c[0], ss, sc);
    }
}

// The sums of a block: per thread, value t * 4 + component of target t, as
// compensated pairs in shared memory (own slots: no conflicts, no races)
template <int NP, int NW>
struct DfShared {
    static constexpr int T = 2 * NP, V = 4 * T, TH = 32 * NW;
    float S[V][TH], C[V][TH];
    float4 t[T];                    // the targets
    int ti[T];                      // and their indices in E_out
    float red[2][NW][V];
};
template <int NP, int NW>
__device__ __forceinline__ void df_put(DfShared<NP, NW> &sh, int v, float x)
{
    float s = sh.S[v][threadIdx.x], c = sh.C[v][threadIdx.x];
    two_sum_acc(s, c, x);
    sh.S[v][threadIdx.x] = s;
    sh.C[v][threadIdx.x] = c;
}

// accumulators of the packs, folded into the thread's slots and cleared
template <bool WANT_V, int NP, int NW>
__device__ __forceinline__ void df_fold(DfShared<NP, NW> &sh, u64 (&A)[4][NP], float vs)
{
#pragma unroll
    for (int p = 0; p < NP; ++p)
#pragma unroll
        for (int c = 0; c < (WANT_V ? 4 : 3); ++c) {
            float a, b;
            upk(A[c][p], a, b);
            if (c == 3) { a *= vs; b *= vs; }
            df_put(sh, 8 * p + c, a);
            df_put(sh, 8 * p + 4 + c, b);
            A[c][p] = 0ull;
        }
}

// one source (positions x 2^40, weight kq x 2^80) at the targets of the packs;
// OWN: rel is the source's index relative to the block's first target, whose
// own charge gives no term
template <bool WANT_V, bool OWN, int NP>
__device__ __forceinline__ void df_source(const u64 (&TX)[NP], const u64 (&TY)[NP], const u64 (&TZ)[NP], float4 src,
                                          float kC, float eps2, int rel, u64 (&A)[4][NP])
{
    const u64 SX = pk(src.x * DF_XS, src.x * DF_XS), SY = pk(src.y * DF_XS, src.y * DF_XS),
              SZ = pk(src.z * DF_XS, src.z * DF_XS);
    const float kq = kC * src.w;
#pragma unroll
    for (int p = 0; p < NP; ++p) {
        const u64 EP = OWN ? pk(rel == 2 * p ? DF_SELF : eps2, rel == 2 * p + 1 ? DF_SELF : eps2) : pk(eps2, eps2);
        const u64 Q = OWN ? pk(rel == 2 * p ? 0.f : kq, rel == 2 * p + 1 ? 0.f : kq) : pk(kq, kq);
        const u64 dx = sub2(TX[p], SX), dy = sub2(TY[p], SY), dz = sub2(TZ[p], SZ);
        const u64 r2 = fma2(dz, dz, fma2(dy, dy, fma2(dx, dx, EP)));
        float ra, rb;
        upk(r2, ra, rb);
        const u64 inv = pk(rsq(ra), rsq(rb));
        const u64 s = mul2(Q, inv);
        const u64 s3 = mul2(s, mul2(inv, inv));
        A[0][p] = fma2(dx, s3, A[0][p]);
        A[1][p] = fma2(dy, s3, A[1][p]);
        A[2][p] = fma2(dz, s3, A[2][p]);
        if (WANT_V) A[3][p] = add2(A[3][p], s);
    }
}
