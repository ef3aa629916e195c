// The tracking step (Sec. 3.2 - 3.3): recombination resolve, free flight with
// exact null-collision trials, ionisation spawn, attachment, absorption on the
// electrode planes, and a deterministic two-pass stream compaction.
//
// Built with --fmad=false: every binary32 operation of the step is one IEEE
// rounding, so that, given the same field, the collision processes, spawns,
// and the compacted order are reproducible bit for bit by any IEEE binary32
// implementation of the same operation sequence.
//
// Passes (all stream-ordered, nothing synchronises):
//   init      zero the stats and the control block
//   partners  nearest eligible cation of every electron (spatial hash, ph_*)
//   resolve   each proposing electron atomicMin's (d^2, e) into its cation
//   count     simulate every charge: its new state to scratch at its own
//             index, ionisation products to a list of records, survivors and
//             spawned pairs per chunk of charges
//   scan      one block: chunk offsets, totals, capacity check (all-or-nothing)
//   write     survivors and spawned charges from scratch to their final slots
//   moments   species counts and cloud moments of the new state, then the
//             blocks' partial sums folded and n, next_id updated
// The bt_* kernels at the end run the same passes for a batch of chambers.
#include "obem_internal.cuh"

#define ST_THREADS 256
#define ST_CT 128                  // threads of the count and write kernels (4 warps, a chunk of charges each)
// Charges per chunk: at most ST_TINY, ST_SMALL, ST_MID charges, more; by the live
// count, on the device (by the capacity, 10,000 charges of a state for 1e6 took
// 361 us to track, 345 before there were chunks, now 158).
// Few charges fill the SMs in small chunks and wait for fewer others' trials;
// larger chunks refill a warp's idle lanes from its list: 10,000 charges (us) 74
// in chunks of 32, 100,000 240 in chunks of 256 and 145 of 128, 1e6 372 and 385.
#define ST_CHUNK_T 8
#define ST_CHUNK_S 32
#define ST_CHUNK_M 128
#define ST_CHUNK_L 256
#define ST_TINY 16384
#define ST_SMALL 65536
#define ST_MID 524288
__host__ __device__ __forceinline__ int step_chunk_len(int n)
{
    return n <= ST_TINY ? ST_CHUNK_T : n <= ST_SMALL ? ST_CHUNK_S : n <= ST_MID ? ST_CHUNK_M : ST_CHUNK_L;
}
#define ST_MB 1024                 // charges per block of the moments
#define ST_MB_T 256                // in contexts of at most ST_TINY charges (bound by one SM's FP64: 1000 charges 10.5 us in one block)

typedef unsigned long long u64;

// ------------------------------------------------------------------ Philox4x32-10
// Salmon, Moraes, Dror & Shaw, SC'11: ten rounds of two 32x32->64 multiplies
// with a Weyl-sequence key schedule.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
        uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
        c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
        k0 += 0x9E3779B9u;
        k1 += 0xBB67AE85u;
    }
    return c;
}

// uniform in [0, 1) from the top 24 bits
__device__ __forceinline__ float unif01(uint32_t u)
{
    return (float)(u >> 8) * 5.9604645e-08f;
}

// -ln(U), U = ((u >> 8) + 1) 2^-24 in (0, 1]: U = 2^(e-24) f with f in [1, 2),
// ln f = 2 atanh((f-1)/(f+1)) summed to the 13th power (basic operations only)
__device__ float neg_log_unif(uint32_t u)
{
    uint32_t m = (u >> 8) + 1u;
    int e = 31 - __clz(m);
    float mf = (float)m;
    float f = mf / (float)(1u << e);
    float t = (f - 1.0f) / (f + 1.0f);
    float t2 = t * t;
    float s = 0.07692308f;
    s = s * t2 + 0.09090909f;
    s = s * t2 + 0.11111111f;
    s = s * t2 + 0.14285715f;
    s = s * t2 + 0.2f;
    s = s * t2 + 0.33333334f;
    s = s * t2 + 1.0f;
    float lnf = 2.0f * t * s;
    float a = (float)(24 - e) * 0.6931472f;
    return a - lnf;
}

// sin, cos of a in [0, pi/2) by their Taylor series in a^2 (Horner)
__device__ __forceinline__ void sincos_quadrant(float a, float &sn, float &cs)
{
    float a2 = a * a;
    float ps = -1.6059044e-10f;
    ps = ps * a2 + 2.5052108e-08f;
    ps = ps * a2 - 2.7557319e-06f;
    ps = ps * a2 + 0.0001984127f;
    ps = ps * a2 - 0.008333334f;
    ps = ps * a2 + 0.16666667f;
    ps = ps * a2 - 1.0f;
    sn = -(a * ps);
    float pc = 2.0876756e-09f;
    pc = pc * a2 - 2.755732e-07f;
    pc = pc * a2 + 2.4801588e-05f;
    pc = pc * a2 - 0.0013888889f;
    pc = pc * a2 + 0.041666668f;
    pc = pc * a2 - 0.5f;
    pc = pc * a2 + 1.0f;
    cs = pc;
}

// isotropic unit vector: cos(theta) = 1 - 2u, azimuth 2 pi u' with the
// quadrant taken from the two top bits of u''s 24-bit fraction
__device__ __forceinline__ float3 isotropic(uint32_t ua, uint32_t ub)
{
    float c = 1.0f - 2.0f * unif01(ua);
    float cc = c * c;
    float om = 1.0f - cc;
    if (om < 0.0f) om = 0.0f;
    float s = sqrtf(om);
    uint32_t b = ub >> 8;
    uint32_t q = b >> 22;
    float f = (float)(b & 0x3FFFFFu) * 5.9604645e-08f;
    float a = f * 6.2831855f;
    float sa, ca;
    sincos_quadrant(a, sa, ca);
    float cp, sp;
    if (q == 0u) { cp = ca; sp = sa; }
    else if (q == 1u) { cp = -sa; sp = ca; }
    else if (q == 2u) { cp = -ca; sp = -sa; }
    else { cp = sa; sp = -ca; }
    return make_float3(s * cp, s * sp, c);
}

// next representable float from x toward +inf (dir > 0) or -inf
__device__ __forceinline__ float next_toward(float x, float dir)
{
    if (x == 0.0f) return dir > 0.0f ? __int_as_float(1) : __int_as_float((int)0x80000001u);
    int b = __float_as_int(x);
    bool up = dir > 0.0f;
    bool pos = x > 0.0f;
    return __int_as_float(up == pos ? b + 1 : b - 1);
}

// grid segment and weight of energy eps (linear interpolation in energy): the
// segment is the last grid point <= eps, searched between the bounds that
// elut holds for eps's leading bits (the 2000-point grid: 2 steps, not 11)
__device__ __forceinline__ void egrid_locate(const GasDev &g, float eps, int &lo, float &w)
{
    lo = 0;
    if (eps < g.e_first) { lo = 0; w = 0.0f; }
    else if (eps >= g.e_last) { lo = g.n_e - 2; w = 1.0f; }
    else {
        const uint32_t b = __ldg(&g.elut[(__float_as_uint(eps) >> OBEM_ELUT_SHIFT) & (OBEM_ELUT - 1)]);
        lo = (int)(b & 0xffffu);
        int hi = (int)(b >> 16);
        while (hi - lo > 1) {
            int mid = (lo + hi) / 2;
            if (__ldg(&g.egrid[mid]) <= eps) lo = mid; else hi = mid;
        }
        float e0 = __ldg(&g.egrid[lo]), e1 = __ldg(&g.egrid[lo + 1]);
        w = (eps - e0) / (e1 - e0);
    }
}

// collision frequency of process j (zero below its threshold); the table
// holds every process of a grid point together
__device__ __forceinline__ float nu_proc(const GasDev &g, int j, float eps, float Ns, int lo, float w)
{
    if (g.mode[j] == OBEM_MODE_CONST) return g.nuc[j];
    if (eps < g.thr[j]) return Ns * 0.0f;
    const float *row = g.xs + (size_t)lo * g.n_proc + j;
    float s0 = __ldg(row);
    float s1 = __ldg(row + g.n_proc);
    float ds = s1 - s0;
    float sg = s0 + w * ds;
    return Ns * sg;
}

// ------------------------------------------------------------------ one charge
__device__ __forceinline__ ChamberP chamber_of(const GasDev &g)
{
    ChamberP c;
    c.seed_lo = g.seed_lo; c.seed_hi = g.seed_hi; c.z_lo = g.z_lo; c.z_hi = g.z_hi;
    return c;
}

struct FlightOut {
    int dead, attached, nsp, collisions, trials, overflow;
    int hit_cell;         // cell that absorbed the charge, or -1
    int rec;              // record of its last spawned pair, or -1
};

// Records of the spawned pairs (OBEM_REC_F4 float4 each, in the order of the
// race: only the links matter): electron position and the previous record of
// the same parent, electron velocity, cation position, cation velocity.  A step
// that commits spawns at most half the capacity; later records are dropped.
struct SpawnRec {
    float4 *rec;
    int *count;
    int max;
};

// One collision trial at the charge's current state: with x uniform in
// [0, scale), process j is taken when x < nu_1 + ... + nu_j (none: null).
// Returns 0 when nothing happened (null, or ionisation without the energy),
// 1 after a collision, 2 when the flight ends (attachment).
__device__ __forceinline__ int collide(const GasDev &g, const ChamberP &cp, uint32_t id, uint32_t step, uint32_t k,
                                       const uint4 &r, float x, float3 &p, float3 &v, uint8_t &sp, FlightOut &fo,
                                       const SpawnRec &R)
{
    float v2 = v.x * v.x + v.y * v.y + v.z * v.z;
    float speed = sqrtf(v2);
    if (sp == OBEM_ELECTRON) {
        float eps = g.K_e * v2;
        int lo;
        float w;
        egrid_locate(g, eps, lo, w);
        float Ns = g.N * speed;
        float cum = 0.0f;
        int proc = -1;
        for (int j = 0; j < g.n_proc; ++j) {
            cum = cum + nu_proc(g, j, eps, Ns, lo, w);
            if (x < cum) { proc = j; break; }
        }
        if (proc < 0) return 0;
        const int kind = g.kind[proc];
        if (kind == OBEM_P_ELASTIC) {
            float3 d = isotropic(r.z, r.w);
            float cosx = 0.0f;
            if (speed > 0.0f) cosx = (v.x * d.x + v.y * d.y + v.z * d.z) / speed;
            float om = 1.0f - cosx;
            float loss = g.two_m_over_M * om;
            float f = 1.0f - loss;
            float sn = speed * sqrtf(f);
            v = make_float3(sn * d.x, sn * d.y, sn * d.z);
            fo.collisions += 1;
        } else if (kind == OBEM_P_EXCITATION) {
            float e2 = eps - g.thr[proc];
            if (e2 < 0.0f) e2 = 0.0f;
            float sn = sqrtf(e2 / g.K_e);
            float3 d = isotropic(r.z, r.w);
            v = make_float3(sn * d.x, sn * d.y, sn * d.z);
            fo.collisions += 1;
        } else if (kind == OBEM_P_IONISATION) {
            float er = eps - g.thr[proc];
            er = er - g.E_therm;
            if (!(er > 0.0f)) return 0;
            float half = 0.5f * er;
            float sn = sqrtf(half / g.K_e);
            float3 d = isotropic(r.z, r.w);
            float rr = g.KCE / (2.0f * er);
            float ox = rr * d.x, oy = rr * d.y, oz = rr * d.z;
            float3 pn = make_float3(p.x + ox, p.y + oy, p.z + oz);
            float3 pp = make_float3(p.x - ox, p.y - oy, p.z - oz);
            if (pn.x == p.x && pn.y == p.y && pn.z == p.z) {
                int axi = 0;
                float a0 = fabsf(d.x), a1 = fabsf(d.y), a2 = fabsf(d.z);
                if (a1 > a0) axi = 1;
                if (a2 > (axi == 1 ? a1 : a0)) axi = 2;
                if (axi == 0) { pn.x = next_toward(p.x, d.x); pp.x = next_toward(p.x, -d.x); }
                else if (axi == 1) { pn.y = next_toward(p.y, d.y); pp.y = next_toward(p.y, -d.y); }
                else { pn.z = next_toward(p.z, d.z); pp.z = next_toward(p.z, -d.z); }
            }
            const int slot = atomicAdd(R.count, 1);
            if (slot < R.max) {
                uint4 r2 = philox4x32_10(make_uint4(id, step, k, 1u), cp.seed_lo, cp.seed_hi);
                float3 di = isotropic(r2.x, r2.y);
                float4 *o = R.rec + (size_t)OBEM_REC_F4 * slot;
                o[0] = make_float4(pn.x, pn.y, pn.z, __int_as_float(fo.rec));
                o[1] = make_float4(sn * d.x, sn * d.y, sn * d.z, 0.0f);
                o[2] = make_float4(p.x, p.y, p.z, 0.0f);
                o[3] = make_float4(g.v_th_ion * di.x, g.v_th_ion * di.y, g.v_th_ion * di.z, 0.0f);
                fo.rec = slot;
            }
            p = pp;
            v = make_float3(-sn * d.x, -sn * d.y, -sn * d.z);
            fo.nsp += 1;
            fo.collisions += 1;
        } else {
            float3 d = isotropic(r.z, r.w);
            v = make_float3(g.v_th_ion * d.x, g.v_th_ion * d.y, g.v_th_ion * d.z);
            sp = OBEM_ANION;
            fo.attached = 1;
            fo.collisions += 1;
            return 2;
        }
    } else {
        float3 d = isotropic(r.z, r.w);
        float sn = (x < g.half_nu_ion) ? speed : g.v_th_ion;
        v = make_float3(sn * d.x, sn * d.y, sn * d.z);
        fo.collisions += 1;
    }
    return 1;
}

// First cell crossed by the segment a -> b (the chord of one sub-flight), by
// the Moller-Trumbore test in binary32 with the oracle's operation order
// (this file is compiled without contraction): edges e1 = v1 - v0,
// e2 = v2 - v0, d = b - a, h = d x e2, det = e1.h (0: no hit), s = a - v0,
// u = (s.h)/det in [0, 1], q = s x e1, v = (d.q)/det >= 0 with u + v <= 1,
// t = (e2.q)/det in [0, 1]; smallest t, ties to the lower cell index.  Only
// the cells listed in the grid cells the segment's bounding box touches are
// tested (every cell is listed in all grid cells its own box touches, plus
// one on every side).  Returns the cell or -1.
__device__ int seg_hit(const GasDev &g, float3 a, float3 b)
{
    int lo[3], hi[3];
    const float mn[3] = {fminf(a.x, b.x), fminf(a.y, b.y), fminf(a.z, b.z)};
    const float mx[3] = {fmaxf(a.x, b.x), fmaxf(a.y, b.y), fmaxf(a.z, b.z)};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float t0 = (mn[k] - g.hlo[k]) * g.hinv, t1 = (mx[k] - g.hlo[k]) * g.hinv;
        if (!(t1 >= -1.0f) || !(t0 <= (float)g.hdim[k])) return -1;   // outside the grid (or NaN)
        lo[k] = max(0, min(g.hdim[k] - 1, (int)floorf(t0)));
        hi[k] = max(0, min(g.hdim[k] - 1, (int)floorf(t1)));
    }
    const float d0 = b.x - a.x, d1 = b.y - a.y, d2 = b.z - a.z;
    int best = -1;
    float bt = 0.0f;
    for (int z = lo[2]; z <= hi[2]; ++z)
        for (int y = lo[1]; y <= hi[1]; ++y)
            for (int x = lo[0]; x <= hi[0]; ++x) {
                const int q = (z * g.hdim[1] + y) * g.hdim[0] + x;
                for (int m = g.hstart[q]; m < g.hstart[q + 1]; ++m) {
                    const int k = g.htri[m];
                    const float *v = g.tri9 + 9 * (size_t)k;
                    const float e10 = v[3] - v[0], e11 = v[4] - v[1], e12 = v[5] - v[2];
                    const float e20 = v[6] - v[0], e21 = v[7] - v[1], e22 = v[8] - v[2];
                    const float h0 = d1 * e22 - d2 * e21, h1 = d2 * e20 - d0 * e22, h2 = d0 * e21 - d1 * e20;
                    const float det = e10 * h0 + e11 * h1 + e12 * h2;
                    if (det == 0.0f) continue;
                    const float inv = 1.0f / det;
                    const float s0 = a.x - v[0], s1 = a.y - v[1], s2 = a.z - v[2];
                    const float u = (s0 * h0 + s1 * h1 + s2 * h2) * inv;
                    if (!(u >= 0.0f && u <= 1.0f)) continue;
                    const float q0 = s1 * e12 - s2 * e11, q1 = s2 * e10 - s0 * e12, q2 = s0 * e11 - s1 * e10;
                    const float w = (d0 * q0 + d1 * q1 + d2 * q2) * inv;
                    if (!(w >= 0.0f && u + w <= 1.0f)) continue;
                    const float t = (e20 * q0 + e21 * q1 + e22 * q2) * inv;
                    if (!(t >= 0.0f && t <= 1.0f)) continue;
                    if (best < 0 || t < bt || (t == bt && k < best)) { best = k; bt = t; }
                }
            }
    return best;
}

// ballistic flight for time fl under acceleration a (half a in h); returns
// true when the charge crossed an absorbing plane
__device__ __forceinline__ bool flight(const GasDev &g, const ChamberP &cp, float3 &p, float3 &v, float ax, float ay, float az,
                                       float hx, float hy, float hz, float fl)
{
    {
        float w = hx * fl; float xx = v.x + w; float y = xx * fl; p.x = p.x + y; float dv = ax * fl; v.x = v.x + dv;
    }
    {
        float w = hy * fl; float xx = v.y + w; float y = xx * fl; p.y = p.y + y; float dv = ay * fl; v.y = v.y + dv;
    }
    {
        float w = hz * fl; float xx = v.z + w; float y = xx * fl; p.z = p.z + y; float dv = az * fl; v.z = v.z + dv;
    }
    return p.z <= cp.z_lo || p.z >= cp.z_hi;
}

// A charge in flight
struct Fly {
    float3 p, v;
    float ax, ay, az;
    float t;              // time since the start of the step
    uint32_t id, k;       // id, trials drawn
    uint8_t s0, sp;       // species at the start of the step, now
    FlightOut fo;
};

// One part of a charge's flight over the step under its step-start field
// (Euler in the field, exact ballistic motion between trials); returns true
// when the charge is done.  Collision sampling: null-collision trials at
// exponential waiting times -ln(U)/nu_max, process j with probability
// nu_j(eps)/nu_max (coll_mode 0; a call is one trial); or the paper's per-step
// scheme (coll_mode 1): flight over the whole step, then one interaction when
// -ln(U) < nu_tot(eps) dt, of type j with probability nu_j/nu_tot.
// Ionisation products at the distance of Eq. (distIoni).  A charge is
// absorbed where a sub-flight's chord crosses a cell (g.hit_on: charging-up)
// or where it ends beyond a plane z_lo / z_hi.
__device__ __forceinline__ bool fly_part(const GasDev &g, const ChamberP &cp, uint32_t step, Fly &f, const SpawnRec &R)
{
    const int s = f.s0;
    const float hx = 0.5f * f.ax, hy = 0.5f * f.ay, hz = 0.5f * f.az;
    if (g.coll_mode == 1) {
        const float3 p0 = f.p;
        const bool crossed = flight(g, cp, f.p, f.v, f.ax, f.ay, f.az, hx, hy, hz, g.dt);
        if (g.hit_on && (f.fo.hit_cell = seg_hit(g, p0, f.p)) >= 0) { f.fo.dead = 1; return true; }
        if (crossed) { f.fo.dead = 1; return true; }
        const uint4 r = philox4x32_10(make_uint4(f.id, step, 1u, 0u), cp.seed_lo, cp.seed_hi);
        f.fo.trials += 1;
        float nu_tot;
        if (s == OBEM_ELECTRON) {
            float v2 = f.v.x * f.v.x + f.v.y * f.v.y + f.v.z * f.v.z;
            float speed = sqrtf(v2);
            float eps = g.K_e * v2;
            int lo;
            float w;
            egrid_locate(g, eps, lo, w);
            float Ns = g.N * speed;
            nu_tot = 0.0f;
            for (int j = 0; j < g.n_proc; ++j) nu_tot = nu_tot + nu_proc(g, j, eps, Ns, lo, w);
        } else {
            nu_tot = g.nu_ion;
        }
        float pr = nu_tot * g.dt;
        if (!(neg_log_unif(r.x) < pr)) return true;
        collide(g, cp, f.id, step, 1u, r, unif01(r.y) * nu_tot, f.p, f.v, f.sp, f.fo, R);
        return true;
    }
    const float numax = (s == OBEM_ELECTRON) ? g.nu_max_e : g.nu_ion;
    float tau;
    uint4 r = make_uint4(0u, 0u, 0u, 0u);
    if (numax > 0.0f) {
        f.k += 1u;
        if ((int)f.k > g.trial_cap) { f.fo.overflow = 1; return true; }
        r = philox4x32_10(make_uint4(f.id, step, f.k, 0u), cp.seed_lo, cp.seed_hi);
        tau = neg_log_unif(r.x) / numax;
    } else {
        tau = __int_as_float(0x7f800000);
    }
    float tn = f.t + tau;
    float fl = (tn >= g.dt) ? (g.dt - f.t) : tau;
    const float3 p0 = f.p;
    const bool crossed = flight(g, cp, f.p, f.v, f.ax, f.ay, f.az, hx, hy, hz, fl);
    if (g.hit_on && (f.fo.hit_cell = seg_hit(g, p0, f.p)) >= 0) { f.fo.dead = 1; return true; }
    if (crossed) { f.fo.dead = 1; return true; }
    if (tn >= g.dt) return true;
    f.t = tn;
    f.fo.trials += 1;
    return collide(g, cp, f.id, step, f.k, r, unif01(r.y) * numax, f.p, f.v, f.sp, f.fo, R) == 2;
}

// ------------------------------------------------------------------ kernels
__device__ __forceinline__ int cur_n(const obem_state &st) { return *st.n; }

__global__ void init_kernel(obem_step_stats *stats, StepCtl *ctl, const obem_state st)
{
    if (threadIdx.x == 0) {
        memset(stats, 0, sizeof(obem_step_stats));
        memset(ctl, 0, sizeof(StepCtl));
        stats->n_before = *st.n;
    }
}

// ---------------------------------------------------------------- partner search
// Nearest eligible cation within R_c for every electron, by spatial hashing:
// cells of edge h = 2 R_c (1 + 1e-5) are hashed into PH_BUCKETS buckets, the
// eligible cations (not created in the previous step) are counting-sorted by
// bucket, and each electron scans the buckets of the 8 cells that the cube of
// half-edge R_c around it can touch (its own and, per axis, the neighbour on
// its side of the cell's middle; cells of R_c took 27), keeping the smallest
// (binary32 d^2, index) key with d^2 <= R_c^2.  Every cation within R_c lies in
// one of those cells and hash collisions only add candidates that the
// distance test rejects, so the result is the exact minimum over all cations
// (the same key as a brute-force scan, whatever the order in a bucket).  Cell
// coordinates are exact to 1e-6 of a cell, against the margin of 5e-6.
#define PH_BUCKETS (1 << 20)

__device__ __forceinline__ uint32_t ph_hash(long long cx, long long cy, long long cz)
{
    const uint32_t h = ((uint32_t)cx * 73856093u) ^ ((uint32_t)cy * 19349663u) ^ ((uint32_t)cz * 83492791u);
    return h & (PH_BUCKETS - 1);
}

// Cell of x (floor(x / h)) in c and the fraction in f.  1 / h comes as two
// floats: x / h = p + r to 2^-48 with FP32 operations (the FP64 pipe was half of
// the query), within 1e-6 of a cell below 6e7 cells; FP64 beyond.
struct PhInv {
    double d;
    float hi, lo;
};
static PhInv ph_inv(double inv_h)
{
    PhInv v;
    v.d = inv_h;
    v.hi = (float)inv_h;
    v.lo = (float)(inv_h - (double)v.hi);
    return v;
}
__device__ __forceinline__ void ph_coord(float x, const PhInv &ih, long long &c, float &f)
{
    const float p = x * ih.hi;
    if (fabsf(p) < 6e7f) {
        const float r = __fmaf_rn(x, ih.lo, __fmaf_rn(x, ih.hi, -p));
        const float k = floorf(p);
        const float t = (p - k) + r;               // p - k exact
        const float q = floorf(t);
        c = (long long)((int)k + (int)q);
        f = t - q;
    } else {
        const double t = (double)x * ih.d, k = floor(t);
        c = (long long)fmin(fmax(k, -4.0e18), 4.0e18);   // in range for the conversion
        f = (float)(t - k);
    }
}
__device__ __forceinline__ void ph_cell(float4 p, const PhInv &ih, long long &cx, long long &cy, long long &cz)
{
    float f;
    ph_coord(p.x, ih, cx, f);
    ph_coord(p.y, ih, cy, f);
    ph_coord(p.z, ih, cz, f);
}
// x's cell in c[0], the neighbour on x's side of its middle in c[1]
__device__ __forceinline__ void ph_coord2(float x, const PhInv &ih, long long (&c)[2])
{
    float f;
    ph_coord(x, ih, c[0], f);
    c[1] = c[0] + (f < 0.5f ? -1 : 1);
}

__global__ void ph_count_kernel(const obem_state st, uint32_t step, PhInv inv_h, int32_t *bucket_of,
                                int32_t *count)
{
    const int n = cur_n(st);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint32_t b = st.birth[i];
    if (st.species[i] != OBEM_CATION || (b != 0u && b == step)) { bucket_of[i] = -1; return; }
    long long cx, cy, cz;
    ph_cell(reinterpret_cast<const float4 *>(st.pos_q)[i], inv_h, cx, cy, cz);
    const uint32_t h = ph_hash(cx, cy, cz);
    bucket_of[i] = (int32_t)h;
    atomicAdd(&count[h], 1);
}

// start = exclusive scan of count (PH_BUCKETS + 1 entries), cursor = start, in
// three passes: sums of 1024-bucket blocks, scan of the block sums, scan
// within each block plus its offset.
#define PH_BLK 1024
#define PH_NBLK (PH_BUCKETS / PH_BLK)

// inclusive scan of one value per thread over a 1024-thread block
__device__ __forceinline__ int32_t ph_block_scan(int32_t v, int32_t *s_warp)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
    }
    if (lane == 31) s_warp[warp] = v;
    __syncthreads();
    if (warp == 0) {
        int32_t w = s_warp[lane];
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t u = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += u;
        }
        s_warp[lane] = w;
    }
    __syncthreads();
    return v + (warp > 0 ? s_warp[warp - 1] : 0);
}

__global__ void __launch_bounds__(PH_BLK) ph_blocksum_kernel(const int32_t *count, int32_t *bsum)
{
    __shared__ int32_t s_warp[32];
    const int32_t v = ph_block_scan(count[blockIdx.x * PH_BLK + threadIdx.x], s_warp);
    if (threadIdx.x == PH_BLK - 1) bsum[blockIdx.x] = v;
}

__global__ void __launch_bounds__(PH_BLK) ph_scan_sums_kernel(int32_t *bsum)
{
    __shared__ int32_t s_warp[32];
    const int32_t v = bsum[threadIdx.x];
    const int32_t inc = ph_block_scan(v, s_warp);
    __syncthreads();
    bsum[threadIdx.x] = inc - v;                 // exclusive offsets
    if (threadIdx.x == PH_BLK - 1) bsum[PH_NBLK] = inc;
}

__global__ void __launch_bounds__(PH_BLK) ph_scan_apply_kernel(const int32_t *count, const int32_t *bsum,
                                                                  int32_t *start, int32_t *cursor)
{
    __shared__ int32_t s_warp[32];
    const int i = blockIdx.x * PH_BLK + threadIdx.x;
    const int32_t v = count[i];
    const int32_t ex = ph_block_scan(v, s_warp) - v + bsum[blockIdx.x];
    start[i] = ex;
    cursor[i] = ex;
    if (i == PH_BUCKETS - 1) start[PH_BUCKETS] = bsum[PH_NBLK];
}

__global__ void ph_scatter_kernel(const obem_state st, const int32_t *bucket_of, int32_t *cursor, int32_t *sorted)
{
    const int n = cur_n(st);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int32_t h = bucket_of[i];
    if (h < 0) return;
    sorted[atomicAdd(&cursor[h], 1)] = i;
}

__global__ void ph_query_kernel(const obem_state st, GasDev g, PhInv inv_h, const int32_t *start,
                                const int32_t *sorted, u64 *prop)
{
    const int n = cur_n(st);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    u64 best = ~0ull;
    if (st.species[i] == OBEM_ELECTRON) {
        const float4 pe = reinterpret_cast<const float4 *>(st.pos_q)[i];
        long long cx[2], cy[2], cz[2];
        ph_coord2(pe.x, inv_h, cx);
        ph_coord2(pe.y, inv_h, cy);
        ph_coord2(pe.z, inv_h, cz);
        int k0[8], k1[8];                      // the eight buckets' loads in flight together
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const uint32_t h = ph_hash(cx[m & 1], cy[(m >> 1) & 1], cz[m >> 2]);
            k0[m] = start[h];
            k1[m] = start[h + 1];
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) {
                    for (int k = k0[m]; k < k1[m]; ++k) {
                        const int c = sorted[k];
                        const float4 pc = reinterpret_cast<const float4 *>(st.pos_q)[c];
                        const float ex = pe.x - pc.x, ey = pe.y - pc.y, ez = pe.z - pc.z;
                        const float d2 = ex * ex + ey * ey + ez * ez;
                        if (!(d2 <= g.rc2)) continue;
                        const u64 key = ((u64)__float_as_uint(d2) << 32) | (u64)(uint32_t)c;
                        if (key < best) best = key;
                    }
                }
    }
    prop[i] = best;
}

__global__ void resolve_kernel(const obem_state st, const u64 *prop, u64 *ionkey)
{
    const int n = cur_n(st);
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    u64 pr = prop[i];
    if (pr == ~0ull || st.species[i] != OBEM_ELECTRON) return;
    uint32_t ion = (uint32_t)(pr & 0xFFFFFFFFu);
    u64 key = (pr & 0xFFFFFFFF00000000ull) | (u64)(uint32_t)i;
    atomicMin(&ionkey[ion], key);
}

__device__ __forceinline__ bool recombined(int i, uint8_t s, const u64 *prop, const u64 *ionkey, int recomb_on)
{
    if (!recomb_on) return false;
    if (s == OBEM_CATION) return ionkey[i] != ~0ull;
    if (s == OBEM_ELECTRON) {
        u64 pr = prop[i];
        if (pr == ~0ull) return false;
        uint32_t ion = (uint32_t)(pr & 0xFFFFFFFFu);
        return ionkey[ion] == ((pr & 0xFFFFFFFF00000000ull) | (u64)(uint32_t)i);
    }
    return false;
}

// ---------------------------------------------------------------- simulate
// The new state of a chunk of charges, in scratch at the charges' own indices.
struct StepScratch {
    float4 *pos, *vel;
    uint32_t *id, *birth;
    uint8_t *sp;
    int32_t *keep;         // spawned pairs << 1 | survives
    int32_t *rec;          // last record of its spawned pairs, or -1
    int32_t *blk;          // (survivors, spawned pairs) per chunk; after the scan, those before it
    int32_t *hit;          // charging-up: cell << 1 | positive, or -1
    SpawnRec R;
};

struct StepCounts {
    int absorbed, attached, coll, rec, trials, ovf;
};

// Simulates the charges [i0, i0 + m), m <= WC, one warp.  The warp lists its
// charges, electrons first, and its lanes take them from the list: a lane whose
// charge is done takes the next one (once a quarter of the lanes are idle), so
// that lanes do not wait for the charge with the most trials of 32, nor ions
// (hardly a trial per step) for electrons (a dozen).  With 11.65 trials per
// electron and half the charges ions, 36 % of the lane slots are busy in array
// order and 84 % with the list (counted for Poisson trials, chunks of 256).
// Measured with the one simulation per step (it was simulated again to write):
// tracking of 1e6 charges 2124 to 725 us.
template <int WC>
__device__ __forceinline__ void step_chunk(const obem_state &st, const GasDev &g, const ChamberP &cp, const float4 *E,
                                           uint32_t step, const u64 *prop, const u64 *ionkey, int i0, int m,
                                           const StepScratch &W, uint8_t *list, int &nkeep, int &nspawn, StepCounts &n)
{
    const int lane = threadIdx.x & 31;
    const unsigned below = (1u << lane) - 1u;
    int ne = 0, ni = 0;
    for (int q = 0; q < m; q += 32) {
        const int i = i0 + q + lane;
        const bool in = q + lane < m;
        uint8_t s = 0;
        bool fly = false;
        if (in) {
            s = st.species[i];
            W.id[i] = st.id[i];
            W.birth[i] = st.birth[i];
            fly = true;
            if (recombined(i, s, prop, ionkey, g.recomb_on)) {
                fly = false;
                n.rec += s == OBEM_CATION;
                W.keep[i] = 0;
                if (g.hit_on) W.hit[i] = -1;
            }
        }
        const unsigned be = __ballot_sync(0xffffffffu, fly && s == OBEM_ELECTRON);
        const unsigned bi = __ballot_sync(0xffffffffu, fly && s != OBEM_ELECTRON);
        if ((be >> lane) & 1u) list[ne + __popc(be & below)] = (uint8_t)(q + lane);
        if ((bi >> lane) & 1u) list[WC - 1 - ni - __popc(bi & below)] = (uint8_t)(q + lane);
        ne += __popc(be);
        ni += __popc(bi);
    }
    __syncwarp();
    const int total = ne + ni;
    int head = 0, cur = -1;
    Fly f;
    nkeep = nspawn = 0;
    for (;;) {
        const unsigned idle = __ballot_sync(0xffffffffu, cur < 0);
        if (idle && head < total && (__popc(idle) >= 8 || WC <= 32)) {
            const int e = head + __popc(idle & below);
            if (cur < 0 && e < total) {
                cur = i0 + list[e < ne ? e : WC - 1 - (e - ne)];
                const float4 pq = reinterpret_cast<const float4 *>(st.pos_q)[cur];
                const float4 vv = reinterpret_cast<const float4 *>(st.vel)[cur];
                const float4 ee = E[cur];
                f.id = st.id[cur];
                f.s0 = f.sp = st.species[cur];
                f.p = make_float3(pq.x, pq.y, pq.z);
                f.v = make_float3(vv.x, vv.y, vv.z);
                const float qm = g.qm[f.s0];
                f.ax = qm * ee.x;
                f.ay = qm * ee.y;
                f.az = qm * ee.z;
                f.t = 0.0f;
                f.k = 0u;
                f.fo = {0, 0, 0, 0, 0, 0, -1, -1};
            }
            head = min(total, head + __popc(idle));
        }
        if (!__any_sync(0xffffffffu, cur >= 0)) {
            if (head >= total) break;
            continue;
        }
        if (cur >= 0 && fly_part(g, cp, step, f, W.R)) {
            const int i = cur;
            cur = -1;
            const int kp = !f.fo.dead;
            if (kp) {
                W.pos[i] = make_float4(f.p.x, f.p.y, f.p.z, st.pos_q[4 * (size_t)i + 3]);
                W.vel[i] = make_float4(f.v.x, f.v.y, f.v.z, st.vel[4 * (size_t)i + 3]);
                W.sp[i] = f.sp;
            }
            W.keep[i] = (f.fo.nsp << 1) | kp;
            if (f.fo.nsp) W.rec[i] = f.fo.rec;
            if (g.hit_on)
                W.hit[i] = f.fo.hit_cell >= 0 ? (f.fo.hit_cell << 1) | (st.pos_q[4 * (size_t)i + 3] > 0.0f ? 1 : 0) : -1;
            nkeep += kp;
            nspawn += f.fo.nsp;
            n.absorbed += f.fo.dead;
            n.attached += f.fo.attached;
            n.coll += f.fo.collisions;
            n.trials += f.fo.trials;
            n.ovf |= f.fo.overflow;
        }
    }
    nkeep = (int)__reduce_add_sync(0xffffffffu, (unsigned)nkeep);
    nspawn = (int)__reduce_add_sync(0xffffffffu, (unsigned)nspawn);
}

// the block's counts to the stats (every thread calls it)
__device__ __forceinline__ void step_counts(const StepCounts &n, obem_step_stats *stats, StepCtl *ctl)
{
    __shared__ int s_n[6];
    if (threadIdx.x < 6) s_n[threadIdx.x] = 0;
    __syncthreads();
    const int v[6] = {n.absorbed, n.attached, n.coll, n.rec, n.trials, n.ovf};
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const int t = (int)__reduce_add_sync(0xffffffffu, (unsigned)v[k]);
        if ((threadIdx.x & 31) == 0 && t) atomicAdd(&s_n[k], t);
    }
    __syncthreads();
    const int k = threadIdx.x;
    const int t = k < 6 ? s_n[k] : 0;
    if (t) {
        if (k == 0) atomicAdd(&stats->absorbed, t);
        else if (k == 1) atomicAdd(&stats->attached, t);
        else if (k == 2) atomicAdd(&stats->collisions, t);
        else if (k == 3) atomicAdd(&stats->recombined_pairs, t);
        else if (k == 4) atomicAdd((unsigned long long *)&stats->trials, (unsigned long long)t);
        else atomicOr(&ctl->trial_overflow, 1);
    }
}

template <int WC>
__device__ __forceinline__ void count_chunks(const obem_state &st, int n, const GasDev &g, const float4 *E, uint32_t step,
                                             const u64 *prop, const u64 *ionkey, const StepScratch &W, uint8_t *list,
                                             StepCounts &sc)
{
    const int ch = blockIdx.x * (ST_CT / 32) + (threadIdx.x >> 5);
    if (ch * WC >= n) return;                            // warp-uniform
    int nk, ns;
    step_chunk<WC>(st, g, chamber_of(g), E, step, prop, ionkey, ch * WC, min(WC, n - ch * WC), W, list, nk, ns, sc);
    if ((threadIdx.x & 31) == 0) { W.blk[2 * ch] = nk; W.blk[2 * ch + 1] = ns; }
}

// FIX: the chunk length of a context whose capacity leaves no other, or 0 (with the
// length a variable 1000 charges' step took 1.5 us more; a copy of the chunk's code
// for each length keeps 1e6 charges at the time of one)
template <int FIX>
__global__ void __launch_bounds__(ST_CT) count_kernel(const obem_state st, GasDev g, const float4 *E, uint32_t step,
                                                      const u64 *prop, const u64 *ionkey, StepScratch W,
                                                      obem_step_stats *stats, StepCtl *ctl)
{
    __shared__ uint8_t s_list[ST_CT / 32][FIX ? FIX : ST_CHUNK_L];
    const int n = cur_n(st), len = FIX ? FIX : step_chunk_len(n);
    if ((int)blockIdx.x * (ST_CT / 32) * len >= n) return;
    uint8_t *list = s_list[threadIdx.x >> 5];
    StepCounts sc = {0, 0, 0, 0, 0, 0};
    if (len == ST_CHUNK_T) count_chunks<ST_CHUNK_T>(st, n, g, E, step, prop, ionkey, W, list, sc);
    else if (len == ST_CHUNK_S) count_chunks<ST_CHUNK_S>(st, n, g, E, step, prop, ionkey, W, list, sc);
    else if (len == ST_CHUNK_M) count_chunks<ST_CHUNK_M>(st, n, g, E, step, prop, ionkey, W, list, sc);
    else count_chunks<ST_CHUNK_L>(st, n, g, E, step, prop, ionkey, W, list, sc);
    step_counts(sc, stats, ctl);
}

// exclusive scan of the (survivors, spawned pairs) of nb chunks, one block of
// 1024; returns the totals
__device__ __forceinline__ void step_scan(int32_t *blk, int nb, int32_t &tk, int32_t &ts)
{
    __shared__ int32_t s_warp[32];
    tk = ts = 0;
    for (int c0 = 0; c0 < nb; c0 += 1024) {
        const int b = c0 + threadIdx.x;
        const int2 v = b < nb ? reinterpret_cast<const int2 *>(blk)[b] : make_int2(0, 0);
        const int32_t ik = ph_block_scan(v.x, s_warp);
        const int32_t wk = s_warp[31];
        __syncthreads();
        const int32_t is = ph_block_scan(v.y, s_warp);
        const int32_t ws = s_warp[31];
        __syncthreads();
        if (b < nb) reinterpret_cast<int2 *>(blk)[b] = make_int2(tk + ik - v.x, ts + is - v.y);
        tk += wk;
        ts += ws;
    }
}

// single block: chunk offsets, totals, capacity and trial checks
__global__ void __launch_bounds__(1024) scan_kernel(const obem_state st, int32_t *blk, int fix,
                                                    obem_step_stats *stats, StepCtl *ctl, int cap)
{
    const int n = cur_n(st), chunk = fix ? fix : step_chunk_len(n);
    int32_t nk, nsp;
    step_scan(blk, (n + chunk - 1) / chunk, nk, nsp);
    if (threadIdx.x == 0) {
        long long total = (long long)nk + 2ll * nsp;
        ctl->n_keep = nk;
        ctl->n_spawn = nsp;
        stats->spawned_pairs = nsp;
        stats->required_capacity = total > 0x7fffffff ? 0x7fffffff : (int)total;
        if (ctl->trial_overflow) {
            ctl->abort = 1;
            stats->status = OBEM_ERR_TRIALS;
        } else if (total > cap) {
            ctl->abort = 1;
            stats->status = OBEM_ERR_CAPACITY;
        }
        stats->n_after = ctl->abort ? n : (int)total;
    }
}

// Survivors of a chunk to their slots (in order from `off`), the pairs its
// charges spawned to theirs (parents in order, a parent's pairs in trial
// order: its records are linked last to first), the charges its cells
// absorbed to the cells' counts.  Scratch is the only input: the state's
// arrays can be written in place.
__device__ __forceinline__ void write_chunk(const obem_state &st, uint32_t step, int i0, int m, int off, int n_keep,
                                            uint32_t id0, const int32_t *blk, const StepScratch &W,
                                            unsigned long long *deposit)
{
    const int lane = threadIdx.x & 31;
    int ok = blk[0], os = blk[1];
    for (int q = 0; q < m; q += 32) {
        const int i = i0 + q + lane;
        const bool in = q + lane < m;
        const int32_t v = in ? W.keep[i] : 0;
        const bool kp = v & 1;
        const int ns = v >> 1;
        const unsigned bk = __ballot_sync(0xffffffffu, kp);
        if (kp) {
            const int o = off + ok + __popc(bk & ((1u << lane) - 1u));
            reinterpret_cast<float4 *>(st.pos_q)[o] = W.pos[i];
            reinterpret_cast<float4 *>(st.vel)[o] = W.vel[i];
            st.id[o] = W.id[i];
            st.birth[o] = W.birth[i];
            st.species[o] = W.sp[i];
        }
        ok += __popc(bk);
        if (__any_sync(0xffffffffu, ns > 0)) {
            int is = ns;
            for (int o = 1; o < 32; o <<= 1) {
                const int u = __shfl_up_sync(0xffffffffu, is, o);
                if (lane >= o) is += u;
            }
            int r = ns ? W.rec[i] : -1;
            for (int k = ns - 1; k >= 0; --k) {
                const int pair = os + is - ns + k;
                const float4 *e = W.R.rec + (size_t)OBEM_REC_F4 * r;
                const float4 a = e[0], b = e[1], c = e[2], d = e[3];
                const int o = off + n_keep + 2 * pair;
                reinterpret_cast<float4 *>(st.pos_q)[o] = make_float4(a.x, a.y, a.z, -(float)OBEM_QE);
                reinterpret_cast<float4 *>(st.vel)[o] = b;
                st.id[o] = id0 + (uint32_t)(2 * pair);
                st.birth[o] = step + 1u;
                st.species[o] = OBEM_ELECTRON;
                reinterpret_cast<float4 *>(st.pos_q)[o + 1] = make_float4(c.x, c.y, c.z, (float)OBEM_QE);
                reinterpret_cast<float4 *>(st.vel)[o + 1] = d;
                st.id[o + 1] = id0 + (uint32_t)(2 * pair + 1);
                st.birth[o + 1] = step + 1u;
                st.species[o + 1] = OBEM_CATION;
                r = __float_as_int(a.w);
            }
            os += __shfl_sync(0xffffffffu, is, 31);
        }
        if (deposit && in) {
            const int32_t h = W.hit[i];
            if (h >= 0) atomicAdd(&deposit[h >> 1], (h & 1) ? 1ull : ~0ull);   // +1 or -1 (two's complement)
        }
    }
}

template <int FIX>
__global__ void __launch_bounds__(ST_CT) write_kernel(const obem_state st, uint32_t step, StepScratch W,
                                                      const StepCtl *ctl, unsigned long long *deposit)
{
    if (ctl->abort) return;
    const int n = cur_n(st), len = FIX ? FIX : step_chunk_len(n);
    const int ch = blockIdx.x * (ST_CT / 32) + (threadIdx.x >> 5);
    if (ch * len >= n) return;
    write_chunk(st, step, ch * len, min(len, n - ch * len), 0, ctl->n_keep, *st.next_id, W.blk + 2 * ch, W, deposit);
}

// free surface density of Eq. (charge-up): e * deposits / area on dielectric
// cells, 0 on electrode cells
__global__ void surface_sigma_kernel(const long long *deposit, const double *area, const int *kind, int np,
                                     float *sigma_free)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= np) return;
    sigma_free[i] = kind[i] == OBEM_CELL_DIELECTRIC ? (float)(OBEM_QE * (double)deposit[i] / area[i]) : 0.0f;
}

int obem_launch_surface_sigma(obem_ctx *c, float *sigma_free, cudaStream_t s)
{
    surface_sigma_kernel<<<(c->np + 255) / 256, 256, 0, s>>>(c->d_deposit, c->d_area, c->d_kind, c->np, sigma_free);
    OBEM_LAUNCH(c);
    return OBEM_OK;
}

// Cloud moments of the new state.  Counts go to the stats by integer atomics
// (exact in any order); the FP64 sums are formed per thread over four charges,
// reduced per block of ST_MB charges and the blocks' partial sums added by
// moments_fold in block order, so the moments are the same on every run.
// Bound: the FP64 pipe (2 FMAs per SM and clock): thirteen sums per charge
// reduced by shuffles over every 256 charges took 213 us at 1e6 charges.
#define NMOM 13    // sum_e[3], sum2_e[3], sum_i[3], sum2_i[3], sum_energy_e

// charges i0 + threadIdx.x + ST_THREADS k below end; part[f * stride]
template <int MB>
__device__ __forceinline__ void moments_block(const obem_state &st, int i0, int end, obem_step_stats *stats,
                                              double *part, int stride)
{
    __shared__ double red[ST_THREADS / 32][16];
    __shared__ int cnt[3];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < 3) cnt[threadIdx.x] = 0;
    __syncthreads();
    double v[16];
#pragma unroll
    for (int f = 0; f < 16; ++f) v[f] = 0.0;
    int ne = 0, nc = 0, na = 0;
#pragma unroll
    for (int q = 0; q < MB / ST_THREADS; ++q) {
        const int i = i0 + q * ST_THREADS + threadIdx.x;
        const uint8_t s = i < end ? st.species[i] : 255;
        const float4 p = i < end ? reinterpret_cast<const float4 *>(st.pos_q)[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        // the same FP64 operations for electrons and ions, on the sums of either
        const bool e = s == OBEM_ELECTRON;
        const float px[3] = {p.x, p.y, p.z};
        if (s != 255) {
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double x = px[c];
                const double a = (e ? v[c] : v[6 + c]) + x, b = fma(x, x, e ? v[3 + c] : v[9 + c]);
                v[c] = e ? a : v[c];
                v[6 + c] = e ? v[6 + c] : a;
                v[3 + c] = e ? b : v[3 + c];
                v[9 + c] = e ? v[9 + c] : b;
            }
        }
        if (e) {
            const float4 u = reinterpret_cast<const float4 *>(st.vel)[i];
            v[12] += (double)u.x * u.x + (double)u.y * u.y + (double)u.z * u.z;
        }
        ne += __popc(__ballot_sync(0xffffffffu, s == OBEM_ELECTRON));
        nc += __popc(__ballot_sync(0xffffffffu, s == OBEM_CATION));
        na += __popc(__ballot_sync(0xffffffffu, s != OBEM_ELECTRON && s != OBEM_CATION && s != 255));
    }
    v[12] *= 0.5 * OBEM_ME / OBEM_QE;
    if (lane == 0) {
        if (ne) atomicAdd(&cnt[0], ne);
        if (nc) atomicAdd(&cnt[1], nc);
        if (na) atomicAdd(&cnt[2], na);
    }
    // sums over the lanes, a step halves the values a lane holds: lane l ends
    // with value l >> 1
    int o = 16;
#pragma unroll
    for (int k = 8; k > 0; k >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int f = 0; f < k; ++f) {
            const double send = up ? v[f] : v[f + k], keep = up ? v[f + k] : v[f];
            v[f] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    if ((lane & 1) == 0) red[warp][lane >> 1] = v[0];
    __syncthreads();
    if (threadIdx.x < NMOM) {
        double t = red[0][threadIdx.x];
        for (int w = 1; w < ST_THREADS / 32; ++w) t += red[w][threadIdx.x];
        part[(size_t)threadIdx.x * stride] = t;
    }
    if (threadIdx.x < 3 && cnt[threadIdx.x])
        atomicAdd(threadIdx.x == 0 ? &stats->n_electron : threadIdx.x == 1 ? &stats->n_cation : &stats->n_anion,
                  cnt[threadIdx.x]);
}

// charges after the step
__device__ __forceinline__ int step_n(const obem_state &st, const StepCtl *ctl)
{
    return ctl->abort ? *st.n : ctl->n_keep + 2 * ctl->n_spawn;
}

template <int MB>
__global__ void __launch_bounds__(ST_THREADS)
moments_kernel(const obem_state st, const StepCtl *ctl, obem_step_stats *stats, double *part, int stride)
{
    const int n = step_n(st, ctl);
    const int i0 = blockIdx.x * MB;
    if (i0 >= n) return;                                 // a block with no charge adds nothing
    moments_block<MB>(st, i0, n, stats, part + blockIdx.x, stride);
}

// sums of the nb blocks' partial sums part[f * stride + b]: warp f adds moment
// f, its lanes' strides in block order and a fixed butterfly
__device__ __forceinline__ void moments_fold(const double *part, int stride, int nb, obem_step_stats *stats)
{
    const int f = threadIdx.x >> 5;
    if (f >= NMOM) return;
    double *const dst = f < 3 ? &stats->sum_e[f] : f < 6 ? &stats->sum2_e[f - 3] : f < 9 ? &stats->sum_i[f - 6]
                      : f < 12 ? &stats->sum2_i[f - 9] : &stats->sum_energy_e;
    double acc = 0.0;
    for (int b = threadIdx.x & 31; b < nb; b += 32) acc += part[(size_t)f * stride + b];
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) *dst = acc;
}

// the fold, and the new counts
__global__ void __launch_bounds__(32 * NMOM) finish_kernel(const obem_state st, const StepCtl *ctl, const double *part,
                                                           int stride, int mb, obem_step_stats *stats)
{
    const int n = step_n(st, ctl);
    moments_fold(part, stride, (n + mb - 1) / mb, stats);
    __syncthreads();                                     // every thread has read the old count
    if (threadIdx.x == 0 && !ctl->abort) {
        *st.next_id = *st.next_id + (uint32_t)(2 * ctl->n_spawn);
        *st.n = n;
    }
}

// ====================================================================
// Sharded step (the charges partitioned among shards, Sec. 2.4 / 3.2.4 run on
// several GPUs): a shard holds its own charges, sorted by id, and sees the
// charges of every shard through gathered copies (G, in shard order; its own
// at [self_off, self_off + n)).  Recombination keys are exchanged as int64 with
// INT64_MAX for "none", so that a signed MIN reduction across shards is the
// unsigned minimum of the keys (valid keys are below 2^63: a finite non-negative
// binary32 d^2 in the high word).
#define SH_NONE 0x7FFFFFFFFFFFFFFFull

// each local electron's nearest cation of the gathered set within R_c: ties to
// the lower cation id (as in the unsharded step, whose array order is id
// order); prop[i] = d^2 bits << 32 | gathered index of that cation
__global__ void sh_query_kernel(const obem_state st, const obem_state G, GasDev g, PhInv inv_h,
                                const int32_t *start, const int32_t *sorted, u64 *prop)
{
    const int n = cur_n(st);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    u64 best = ~0ull, best_idx = 0;
    if (st.species[i] == OBEM_ELECTRON) {
        const float4 pe = reinterpret_cast<const float4 *>(st.pos_q)[i];
        long long cx[2], cy[2], cz[2];
        ph_coord2(pe.x, inv_h, cx);
        ph_coord2(pe.y, inv_h, cy);
        ph_coord2(pe.z, inv_h, cz);
        int k0[8], k1[8];                      // the eight buckets' loads in flight together
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const uint32_t h = ph_hash(cx[m & 1], cy[(m >> 1) & 1], cz[m >> 2]);
            k0[m] = start[h];
            k1[m] = start[h + 1];
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) {
                    for (int k = k0[m]; k < k1[m]; ++k) {
                        const int c = sorted[k];
                        const float4 pc = reinterpret_cast<const float4 *>(G.pos_q)[c];
                        const float ex = pe.x - pc.x, ey = pe.y - pc.y, ez = pe.z - pc.z;
                        const float d2 = ex * ex + ey * ey + ez * ez;
                        if (!(d2 <= g.rc2)) continue;
                        const u64 key = ((u64)__float_as_uint(d2) << 32) | (u64)G.id[c];
                        if (key < best) { best = key; best_idx = (u64)(uint32_t)c; }
                    }
                }
    }
    prop[i] = best == ~0ull ? ~0ull : ((best & 0xFFFFFFFF00000000ull) | best_idx);
}

// the local electrons' proposals into the gathered cations' keys: (d^2, id)
__global__ void sh_propose_kernel(const obem_state st, const u64 *prop, unsigned long long *ionkey)
{
    const int n = cur_n(st);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const u64 pr = prop[i];
    if (pr == ~0ull || st.species[i] != OBEM_ELECTRON) return;
    atomicMin(&ionkey[(uint32_t)(pr & 0xFFFFFFFFu)], (pr & 0xFFFFFFFF00000000ull) | (u64)st.id[i]);
}

__global__ void sh_fill_kernel(unsigned long long *k, long long n)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        k[i] = SH_NONE;
}

// the reduced keys as the local arrays of the unsharded step: a local
// electron that won its cation gets prop = ionkey = (d^2, own index) at its
// own index; a local cation that accepted a proposal a key != ~0
__global__ void sh_localize_kernel(const obem_state st, const unsigned long long *ionkey, int self_off, u64 *prop,
                                   u64 *ionloc)
{
    const int n = cur_n(st);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint8_t sp = st.species[i];
    u64 p = ~0ull, k = ~0ull;
    if (sp == OBEM_ELECTRON) {
        const u64 pr = prop[i];
        if (pr != ~0ull &&
            ionkey[(uint32_t)(pr & 0xFFFFFFFFu)] == ((pr & 0xFFFFFFFF00000000ull) | (u64)st.id[i])) {
            p = (pr & 0xFFFFFFFF00000000ull) | (u64)(uint32_t)i;
            k = p;
        }
    } else if (sp == OBEM_CATION) {
        if (ionkey[self_off + i] != SH_NONE) k = 0ull;
    }
    prop[i] = p;
    ionloc[i] = k;
}

static GasDev step_gas(obem_ctx *c)
{
    GasDev g = c->gas;
    g.hit_on = (c->cfg.flags & OBEM_STEP_SURFACE_HITS) && c->np > 0 && c->d_tri9;
    if (g.hit_on) {
        g.tri9 = c->d_tri9;
        g.hstart = c->d_hstart;
        g.htri = c->d_htri;
        for (int k = 0; k < 3; ++k) { g.hlo[k] = c->h_hlo[k]; g.hdim[k] = c->h_hdim[k]; }
        g.hinv = c->h_hinv;
    }
    return g;
}

// the context's scratch as the count and write kernels see it
static StepScratch step_scratch(obem_ctx *c)
{
    StepScratch W;
    W.pos = c->o_pos; W.vel = c->o_vel; W.id = c->o_id; W.birth = c->o_birth; W.sp = c->o_sp;
    W.keep = c->s_keep; W.rec = c->s_nsp; W.blk = c->s_blk; W.hit = c->s_hit;
    W.R.rec = c->s_rec; W.R.count = &c->s_ctl->n_rec; W.R.max = c->cap / 2;
    return W;
}
// blocks of the count and write kernels: the most chunks that up to cap charges make
static int step_chunk_blocks(int cap)
{
    int most = 0;
    for (const int top : {ST_TINY, ST_SMALL, ST_MID, cap}) {
        const int n = top < cap ? top : cap, len = step_chunk_len(n), ch = (n + len - 1) / len;
        most = ch > most ? ch : most;
    }
    return (most + ST_CT / 32 - 1) / (ST_CT / 32);
}

static void launch_count(obem_ctx *c, const obem_state &st, const GasDev &g, const float4 *E, uint32_t step,
                         obem_step_stats *stats, cudaStream_t s)
{
    const StepScratch W = step_scratch(c);
    const int nb = step_chunk_blocks(st.capacity), fix = st.capacity <= ST_TINY ? ST_CHUNK_T : 0;
    if (fix) count_kernel<ST_CHUNK_T><<<nb, ST_CT, 0, s>>>(st, g, E, step, c->s_prop, c->s_ionkey, W, stats, c->s_ctl);
    else count_kernel<0><<<nb, ST_CT, 0, s>>>(st, g, E, step, c->s_prop, c->s_ionkey, W, stats, c->s_ctl);
    scan_kernel<<<1, 1024, 0, s>>>(st, c->s_blk, fix, stats, c->s_ctl, st.capacity < c->cap ? st.capacity : c->cap);
}

// write, moments, fold and the new counts
static void launch_write(obem_ctx *c, const obem_state &st, const GasDev &g, uint32_t step, obem_step_stats *stats,
                         cudaStream_t s)
{
    const StepScratch W = step_scratch(c);
    unsigned long long *dep = g.hit_on ? (unsigned long long *)c->d_deposit : NULL;
    const int nb = step_chunk_blocks(st.capacity);
    if (st.capacity <= ST_TINY) write_kernel<ST_CHUNK_T><<<nb, ST_CT, 0, s>>>(st, step, W, c->s_ctl, dep);
    else write_kernel<0><<<nb, ST_CT, 0, s>>>(st, step, W, c->s_ctl, dep);
    const int m = c->cap <= ST_TINY ? ST_MB_T : ST_MB, mb = (st.capacity + m - 1) / m;
    if (m == ST_MB_T) moments_kernel<ST_MB_T><<<mb, ST_THREADS, 0, s>>>(st, c->s_ctl, stats, c->s_mpart, mb);
    else moments_kernel<ST_MB><<<mb, ST_THREADS, 0, s>>>(st, c->s_ctl, stats, c->s_mpart, mb);
    finish_kernel<<<1, 32 * NMOM, 0, s>>>(st, c->s_ctl, c->s_mpart, mb, m, stats);
}

int obem_launch_shard_propose(obem_ctx *c, const obem_state *stp, const obem_state *Gp, uint32_t step,
                              unsigned long long *ionkey, cudaStream_t s)
{
    const obem_state st = *stp, G = *Gp;
    const int nblk = (st.capacity + ST_THREADS - 1) / ST_THREADS;
    const int gblk = (G.capacity + ST_THREADS - 1) / ST_THREADS;
    const GasDev g = step_gas(c);
    sh_fill_kernel<<<(G.capacity + 255) / 256 < 4096 ? (G.capacity + 255) / 256 : 4096, 256, 0, s>>>(ionkey,
                                                                                                  G.capacity);
    OBEM_LAUNCH(c);
    if (!g.recomb_on || !(g.rc2 > 0.f)) {
        OBEM_CUDA(c, cudaMemsetAsync(c->s_prop, 0xFF, sizeof(u64) * (size_t)st.capacity, s));
        return OBEM_OK;
    }
    // spatial hash of the gathered cations, queried by the local electrons
    const PhInv inv_h = ph_inv(0.5 / (sqrt((double)g.rc2) * (1.0 + 1e-5)));
    OBEM_CUDA(c, cudaMemsetAsync(c->ph_count, 0, sizeof(int32_t) * PH_BUCKETS, s));
    ph_count_kernel<<<gblk, ST_THREADS, 0, s>>>(G, step, inv_h, c->ph_bucket, c->ph_count);
    ph_blocksum_kernel<<<PH_NBLK, PH_BLK, 0, s>>>(c->ph_count, c->ph_bsum);
    ph_scan_sums_kernel<<<1, PH_BLK, 0, s>>>(c->ph_bsum);
    ph_scan_apply_kernel<<<PH_NBLK, PH_BLK, 0, s>>>(c->ph_count, c->ph_bsum, c->ph_start, c->ph_cursor);
    ph_scatter_kernel<<<gblk, ST_THREADS, 0, s>>>(G, c->ph_bucket, c->ph_cursor, c->ph_sorted);
    sh_query_kernel<<<nblk, ST_THREADS, 0, s>>>(st, G, g, inv_h, c->ph_start, c->ph_sorted, c->s_prop);
    sh_propose_kernel<<<nblk, ST_THREADS, 0, s>>>(st, c->s_prop, ionkey);
    OBEM_LAUNCH(c);
    return OBEM_OK;
}

int obem_launch_shard_count(obem_ctx *c, const obem_state *stp, const float4 *E, uint32_t step,
                            const unsigned long long *ionkey, int self_off, obem_step_stats *stats, cudaStream_t s)
{
    const obem_state st = *stp;
    const int nblk = (st.capacity + ST_THREADS - 1) / ST_THREADS;
    const GasDev g = step_gas(c);
    init_kernel<<<1, 32, 0, s>>>(stats, c->s_ctl, st);
    OBEM_LAUNCH(c);
    if (g.recomb_on) {
        sh_localize_kernel<<<nblk, ST_THREADS, 0, s>>>(st, ionkey, self_off, c->s_prop, c->s_ionkey);
        OBEM_LAUNCH(c);
    }
    launch_count(c, st, g, E, step, stats, s);
    OBEM_LAUNCH(c);
    return OBEM_OK;
}

// the shard does not commit (another shard's step failed): nothing is
// written, and a shard that had no error of its own reports OBEM_ERR_STATE
__global__ void sh_abort_kernel(StepCtl *ctl, obem_step_stats *stats)
{
    if (threadIdx.x != 0) return;
    ctl->abort = 1;
    if (stats->status == OBEM_OK) stats->status = OBEM_ERR_STATE;
    stats->n_after = stats->n_before;
}

__global__ void sh_set_id_kernel(uint32_t *next_id, uint32_t v)
{
    if (threadIdx.x == 0) *next_id = v;
}

int obem_launch_shard_commit(obem_ctx *c, const obem_state *stp, const float4 *E, uint32_t step, uint32_t id_base,
                             int commit, obem_step_stats *stats, cudaStream_t s)
{
    const obem_state st = *stp;
    const GasDev g = step_gas(c);
    (void)E;                             // the flights were simulated by obem_launch_shard_count
    if (!commit) {
        sh_abort_kernel<<<1, 32, 0, s>>>(c->s_ctl, stats);
        OBEM_LAUNCH(c);
        return OBEM_OK;
    }
    sh_set_id_kernel<<<1, 32, 0, s>>>(st.next_id, id_base);
    launch_write(c, st, g, step, stats, s);
    OBEM_LAUNCH(c);
    return OBEM_OK;
}

int obem_launch_step(obem_ctx *c, const obem_state *stp, const float4 *E, uint32_t step,
                     obem_step_stats *stats, cudaStream_t s)
{
    const obem_state st = *stp;
    const int cap = st.capacity;
    const int nblk = (cap + ST_THREADS - 1) / ST_THREADS;
    const GasDev g = step_gas(c);
    init_kernel<<<1, 32, 0, s>>>(stats, c->s_ctl, st);
    OBEM_LAUNCH(c);
    if (g.recomb_on) {
        if (g.rc2 > 0.f) {
            const PhInv inv_h = ph_inv(0.5 / (sqrt((double)g.rc2) * (1.0 + 1e-5)));
            OBEM_CUDA(c, cudaMemsetAsync(c->ph_count, 0, sizeof(int32_t) * PH_BUCKETS, s));
            ph_count_kernel<<<nblk, ST_THREADS, 0, s>>>(st, step, inv_h, c->ph_bucket, c->ph_count);
            ph_blocksum_kernel<<<PH_NBLK, PH_BLK, 0, s>>>(c->ph_count, c->ph_bsum);
            ph_scan_sums_kernel<<<1, PH_BLK, 0, s>>>(c->ph_bsum);
            ph_scan_apply_kernel<<<PH_NBLK, PH_BLK, 0, s>>>(c->ph_count, c->ph_bsum, c->ph_start, c->ph_cursor);
            ph_scatter_kernel<<<nblk, ST_THREADS, 0, s>>>(st, c->ph_bucket, c->ph_cursor, c->ph_sorted);
            ph_query_kernel<<<nblk, ST_THREADS, 0, s>>>(st, g, inv_h, c->ph_start, c->ph_sorted, c->s_prop);
            OBEM_LAUNCH(c);
        } else {
            OBEM_CUDA(c, cudaMemsetAsync(c->s_prop, 0xFF, sizeof(u64) * (size_t)cap, s));
        }
        OBEM_CUDA(c, cudaMemsetAsync(c->s_ionkey, 0xFF, sizeof(u64) * (size_t)cap, s));
        resolve_kernel<<<nblk, ST_THREADS, 0, s>>>(st, c->s_prop, c->s_ionkey);
        OBEM_LAUNCH(c);
    }
    launch_count(c, st, g, E, step, stats, s);
    OBEM_LAUNCH(c);
    launch_write(c, st, g, step, stats, s);
    OBEM_LAUNCH(c);
    if (c->prof_on) c->launches += 6 + (g.recomb_on ? 7 : 0);
    return OBEM_OK;
}

// ====================================================================
// Batch of independent chambers.  Chamber c holds slots [seg_off[c],
// seg_off[c + 1]) of one concatenated state (multiples of OBEM_SEG_ALIGN, so
// each block of ST_THREADS slots belongs to one chamber), its first n[c]
// live.  The passes of the single step, each one launch for every chamber;
// a charge meets only charges of its own chamber, and its draws are keyed by
// its chamber's seed and its own id, so every chamber evolves exactly as it
// would alone.  The step index is read from the device and advanced by the
// last pass: the launch sequence can be captured once in a CUDA graph and
// replayed step after step.  If any chamber fails (capacity, trials), no
// chamber commits.

// chamber of the block, its first slot, its live charges; slot i's index in it
struct BtSlot {
    int c, off, n, li;
};
__device__ __forceinline__ BtSlot bt_slot(const StepBatch &B)
{
    BtSlot r;
    r.c = B.blk_cham[blockIdx.x];
    r.off = B.seg_off[r.c];
    r.n = B.n[r.c];
    r.li = blockIdx.x * ST_THREADS + threadIdx.x - r.off;
    return r;
}

__global__ void bt_init_kernel(StepBatch B)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c == 0) { *B.abort = 0; *B.n_rec = 0; }
    if (c >= B.nb) return;
    memset(&B.stats[c], 0, sizeof(obem_step_stats));
    memset(&B.ctl[c], 0, sizeof(StepCtl));
    B.stats[c].n_before = B.n[c];
}

__device__ __forceinline__ uint32_t bt_hash(long long cx, long long cy, long long cz, int c)
{
    return (ph_hash(cx, cy, cz) ^ ((uint32_t)c * 0x9E3779B1u)) & (PH_BUCKETS - 1);
}

__global__ void bt_ph_count_kernel(const obem_state st, StepBatch B, PhInv inv_h, int32_t *bucket_of, int32_t *count)
{
    const BtSlot q = bt_slot(B);
    if (q.li >= q.n) return;
    const int i = q.off + q.li;
    const uint32_t step = *B.step;
    const uint32_t b = st.birth[i];
    if (st.species[i] != OBEM_CATION || (b != 0u && b == step)) { bucket_of[i] = -1; return; }
    long long cx, cy, cz;
    ph_cell(reinterpret_cast<const float4 *>(st.pos_q)[i], inv_h, cx, cy, cz);
    const uint32_t h = bt_hash(cx, cy, cz, q.c);
    bucket_of[i] = (int32_t)h;
    atomicAdd(&count[h], 1);
}

__global__ void bt_ph_scatter_kernel(const obem_state st, StepBatch B, const int32_t *bucket_of, int32_t *cursor,
                                     int32_t *sorted)
{
    const BtSlot q = bt_slot(B);
    if (q.li >= q.n) return;
    const int i = q.off + q.li;
    const int32_t h = bucket_of[i];
    if (h < 0) return;
    sorted[atomicAdd(&cursor[h], 1)] = i;
}

// nearest eligible cation of the same chamber (keys carry slots: within a
// chamber, slot order is index order, so ties resolve as in a single step)
__global__ void bt_ph_query_kernel(const obem_state st, StepBatch B, GasDev g, PhInv inv_h, const int32_t *start,
                                   const int32_t *sorted, u64 *prop)
{
    const BtSlot q = bt_slot(B);
    if (q.li >= q.n) return;
    const int i = q.off + q.li;
    u64 best = ~0ull;
    if (st.species[i] == OBEM_ELECTRON) {
        const float4 pe = reinterpret_cast<const float4 *>(st.pos_q)[i];
        long long cx[2], cy[2], cz[2];
        ph_coord2(pe.x, inv_h, cx);
        ph_coord2(pe.y, inv_h, cy);
        ph_coord2(pe.z, inv_h, cz);
        int k0[8], k1[8];                      // the eight buckets' loads in flight together
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            const uint32_t h = bt_hash(cx[m & 1], cy[(m >> 1) & 1], cz[m >> 2], q.c);
            k0[m] = start[h];
            k1[m] = start[h + 1];
        }
#pragma unroll
        for (int m = 0; m < 8; ++m) {
                    for (int k = k0[m]; k < k1[m]; ++k) {
                        const int c = sorted[k];
                        if (c < q.off || c >= q.off + q.n) continue;      // another chamber
                        const float4 pc = reinterpret_cast<const float4 *>(st.pos_q)[c];
                        const float ex = pe.x - pc.x, ey = pe.y - pc.y, ez = pe.z - pc.z;
                        const float d2 = ex * ex + ey * ey + ez * ez;
                        if (!(d2 <= g.rc2)) continue;
                        const u64 key = ((u64)__float_as_uint(d2) << 32) | (u64)(uint32_t)c;
                        if (key < best) best = key;
                    }
                }
    }
    prop[i] = best;
}

__global__ void bt_resolve_kernel(const obem_state st, StepBatch B, const u64 *prop, u64 *ionkey)
{
    const BtSlot q = bt_slot(B);
    if (q.li >= q.n) return;
    const int i = q.off + q.li;
    const u64 pr = prop[i];
    if (pr == ~0ull || st.species[i] != OBEM_ELECTRON) return;
    const uint32_t ion = (uint32_t)(pr & 0xFFFFFFFFu);
    atomicMin(&ionkey[ion], (pr & 0xFFFFFFFF00000000ull) | (u64)(uint32_t)i);
}

// chunk of a batch: WC slots of one chamber (segments are multiples of 1024);
// m: its live charges
struct BtChunk {
    int ch, c, off, i0, m;
};
template <int WC>
__device__ __forceinline__ BtChunk bt_chunk(const StepBatch &B)
{
    BtChunk r;
    r.ch = blockIdx.x * (ST_CT / 32) + (threadIdx.x >> 5);
    r.i0 = r.ch * WC;
    r.c = B.blk_cham[r.i0 / ST_THREADS];
    r.off = B.seg_off[r.c];
    r.m = min(WC, r.off + B.n[r.c] - r.i0);
    return r;
}

template <int WC>
__global__ void __launch_bounds__(ST_CT)
bt_count_kernel(const obem_state st, StepBatch B, GasDev g, const float4 *E, const u64 *prop, const u64 *ionkey,
                StepScratch W)
{
    __shared__ uint8_t s_list[ST_CT / 32][WC];
    const BtChunk q = bt_chunk<WC>(B);
    StepCounts sc = {0, 0, 0, 0, 0, 0};
    if (q.m > 0) {                                       // warp-uniform
        int nk, ns;
        step_chunk<WC>(st, g, B.cham[q.c], E, *B.step, prop, ionkey, q.i0, q.m, W, s_list[threadIdx.x >> 5], nk, ns, sc);
        if ((threadIdx.x & 31) == 0) { W.blk[2 * q.ch] = nk; W.blk[2 * q.ch + 1] = ns; }
    }
    step_counts(sc, &B.stats[q.c], &B.ctl[q.c]);         // the block's chunks are of one chamber
}

// one block per chamber: exclusive scan of its blocks' (keep, spawn) totals,
// capacity and trial checks
__global__ void __launch_bounds__(1024) bt_scan_kernel(StepBatch B, int32_t *blk, int chunk)
{
    const int c = blockIdx.x;
    const int cap = B.seg_off[c + 1] - B.seg_off[c];
    int32_t carry_k, carry_s;
    step_scan(blk + 2 * (B.seg_off[c] / chunk), (B.n[c] + chunk - 1) / chunk, carry_k, carry_s);
    if (threadIdx.x == 0) {
        StepCtl *ctl = &B.ctl[c];
        obem_step_stats *stt = &B.stats[c];
        const long long total = (long long)carry_k + 2ll * carry_s;
        ctl->n_keep = carry_k;
        ctl->n_spawn = carry_s;
        stt->spawned_pairs = carry_s;
        stt->required_capacity = total > 0x7fffffff ? 0x7fffffff : (int)total;
        if (ctl->trial_overflow) {
            stt->status = OBEM_ERR_TRIALS;
            atomicOr(B.abort, 1);
        } else if (total > cap) {
            stt->status = OBEM_ERR_CAPACITY;
            atomicOr(B.abort, 1);
        }
    }
}

template <int WC>
__global__ void __launch_bounds__(ST_CT) bt_write_kernel(const obem_state st, StepBatch B, StepScratch W)
{
    if (*B.abort) return;
    const BtChunk q = bt_chunk<WC>(B);
    if (q.m <= 0) return;
    write_chunk(st, *B.step, q.i0, q.m, q.off, B.ctl[q.c].n_keep, B.next_id[q.c], W.blk + 2 * q.ch, W, NULL);
}

// per chamber: new counts (or, when any chamber failed, the chambers that did
// not fail report OBEM_ERR_STATE: nothing was committed); the step index
// advances when the batch committed
__global__ void bt_finish_kernel(StepBatch B)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    const bool ab = *B.abort != 0;
    if (c == 0 && !ab) *B.step += 1u;
    if (c >= B.nb) return;
    obem_step_stats *stt = &B.stats[c];
    if (ab) {
        if (stt->status == OBEM_OK) stt->status = OBEM_ERR_STATE;
        stt->n_after = stt->n_before;
        return;
    }
    const StepCtl &ctl = B.ctl[c];
    B.n[c] = ctl.n_keep + 2 * ctl.n_spawn;
    B.next_id[c] = B.next_id[c] + (uint32_t)(2 * ctl.n_spawn);
    stt->n_after = B.n[c];
}

__global__ void __launch_bounds__(ST_THREADS)
bt_moments_kernel(const obem_state st, StepBatch B, double *part, int stride)
{
    const int i0 = blockIdx.x * ST_MB;
    const int c = B.blk_cham[i0 / ST_THREADS];
    const int end = B.seg_off[c] + B.n[c];
    if (i0 >= end) return;                               // a block past the chamber's charges
    moments_block<ST_MB>(st, i0, end, &B.stats[c], part + blockIdx.x, stride);
}

// one block per chamber: its blocks' partial sums in block order
__global__ void __launch_bounds__(32 * NMOM) bt_moments_fold_kernel(StepBatch B, const double *part, int stride)
{
    const int c = blockIdx.x;
    moments_fold(part + B.seg_off[c] / ST_MB, stride, (B.n[c] + ST_MB - 1) / ST_MB, &B.stats[c]);
}

// The whole batched step on stream s.  Scratch (BtScratch) is sized for the
// batch's slots; E holds the field at every live slot.
int obem_launch_step_batch(obem_ctx *c, const obem_state *stp, const StepBatch &B, const BtScratch &W,
                           const float4 *E, cudaStream_t s)
{
    const obem_state st = *stp;
    const int slots = st.capacity;
    const int nblk = slots / ST_THREADS;
    GasDev g = c->gas;
    g.hit_on = 0;
    const int cb = (B.nb + 255) / 256;
    bt_init_kernel<<<cb, 256, 0, s>>>(B);
    OBEM_LAUNCH(c);
    if (g.recomb_on) {
        if (g.rc2 > 0.f) {
            const PhInv inv_h = ph_inv(0.5 / (sqrt((double)g.rc2) * (1.0 + 1e-5)));
            OBEM_CUDA(c, cudaMemsetAsync(W.ph_count, 0, sizeof(int32_t) * PH_BUCKETS, s));
            bt_ph_count_kernel<<<nblk, ST_THREADS, 0, s>>>(st, B, inv_h, W.ph_bucket, W.ph_count);
            ph_blocksum_kernel<<<PH_NBLK, PH_BLK, 0, s>>>(W.ph_count, W.ph_bsum);
            ph_scan_sums_kernel<<<1, PH_BLK, 0, s>>>(W.ph_bsum);
            ph_scan_apply_kernel<<<PH_NBLK, PH_BLK, 0, s>>>(W.ph_count, W.ph_bsum, W.ph_start, W.ph_cursor);
            bt_ph_scatter_kernel<<<nblk, ST_THREADS, 0, s>>>(st, B, W.ph_bucket, W.ph_cursor, W.ph_sorted);
            bt_ph_query_kernel<<<nblk, ST_THREADS, 0, s>>>(st, B, g, inv_h, W.ph_start, W.ph_sorted, W.prop);
            OBEM_LAUNCH(c);
        } else {
            OBEM_CUDA(c, cudaMemsetAsync(W.prop, 0xFF, sizeof(u64) * (size_t)slots, s));
        }
        OBEM_CUDA(c, cudaMemsetAsync(W.ionkey, 0xFF, sizeof(u64) * (size_t)slots, s));
        bt_resolve_kernel<<<nblk, ST_THREADS, 0, s>>>(st, B, W.prop, W.ionkey);
        OBEM_LAUNCH(c);
    }
    StepScratch SW;
    SW.pos = W.o_pos; SW.vel = W.o_vel; SW.id = W.o_id; SW.birth = W.o_birth; SW.sp = W.o_sp;
    SW.keep = W.keep; SW.rec = W.nsp; SW.blk = W.blk; SW.hit = NULL;
    SW.R.rec = W.rec; SW.R.count = B.n_rec; SW.R.max = slots / 2;
    const int ch = slots <= ST_SMALL ? ST_CHUNK_S : ST_CHUNK_M;          // (partly filled chambers: 189 us against 300 at 256)
    const int cb2 = slots / (ch * (ST_CT / 32));
    if (ch == ST_CHUNK_S) bt_count_kernel<ST_CHUNK_S><<<cb2, ST_CT, 0, s>>>(st, B, g, E, W.prop, W.ionkey, SW);
    else bt_count_kernel<ST_CHUNK_M><<<cb2, ST_CT, 0, s>>>(st, B, g, E, W.prop, W.ionkey, SW);
    OBEM_LAUNCH(c);
    bt_scan_kernel<<<B.nb, 1024, 0, s>>>(B, W.blk, ch);
    OBEM_LAUNCH(c);
    if (ch == ST_CHUNK_S) bt_write_kernel<ST_CHUNK_S><<<cb2, ST_CT, 0, s>>>(st, B, SW);
    else bt_write_kernel<ST_CHUNK_M><<<cb2, ST_CT, 0, s>>>(st, B, SW);
    OBEM_LAUNCH(c);
    bt_finish_kernel<<<cb, 256, 0, s>>>(B);
    OBEM_LAUNCH(c);
    bt_moments_kernel<<<slots / ST_MB, ST_THREADS, 0, s>>>(st, B, W.mpart, slots / ST_MB);
    bt_moments_fold_kernel<<<B.nb, 32 * NMOM, 0, s>>>(B, W.mpart, slots / ST_MB);
    OBEM_LAUNCH(c);
    return OBEM_OK;
}
