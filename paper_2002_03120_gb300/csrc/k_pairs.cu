// k_pairs.cu -- the pair passes of one velocity-Verlet sub-step.
//
//   k_density32 (FP32), k_density or k_density_half + k_density_gather (FP64)
//                  compute_particle_dens + compute_particle_pres (Eqs. compdens,
//                  prtcpres; kernel normalisation; negative-pressure clamp)
//   k_shepard32, k_shepard  smoothe_particle_pres (Shepard-weighted pressure),
//                  density reinitialisation
//   k_drag, k_drag_law  compute_fpi_action (Eqs. fvfdef, beta, F_fpi_DG)
//   k_force_half + k_force_gather (Newton-3), k_force_draw and k_force_cached
//   (direct, FP32) or k_force_fluid (direct, FP64):
//                  compute_fluid on fluid particles + compute_fpi_reaction
//                  (Eqs. FijC, FijD, FijR, FijT, F_fpi_DG_reac) + torque
//   k_force_rigid  compute_fluid on rigid particles (Eq. F_fpi_PG) +
//                  compute_rigid (Eqs. dem_fnij .. slideref, lubri), FP64
//
// Neighbour lists hold every pair within the build radius h (1 + skin); each
// pass decides r_ij < h exactly before using a pair (float test outside a
// +-1e-5 guard band, the oracle's double expression inside it, or the double
// expression directly in FP64 mode), so the pairs evaluated are exactly the
// paper's.  No atomics on forces: a thread writes only its own particle, and
// the Newton-3 pass hands each pair result to the partner through a buffer;
// every sum has a fixed order.  The random matrix of a pair is regenerated
// from the counter (min gid, max gid, step) or, in the second evaluation of a
// step, read back from the first one's cache (same counter, same bits).
#include <algorithm>
#define BM_TABLES
#include "common.cuh"

namespace sdpd {

template <class R> struct Vec;
template <> struct Vec<float> { using T4 = float4; };
template <> struct Vec<double> { using T4 = double4_32a; };
template <class R> struct Vec2;
template <> struct Vec2<float> { using T2 = float2; };
template <> struct Vec2<double> { using T2 = double2; };

// 1 - q of q = r / h, not below 0 (q of a pair within h exceeds 1 by rounding
// at most; FP64: the sign tested on the high word)
__device__ __forceinline__ float one_minus(float q) { return q < 1.0f ? 1.0f - q : 0.0f; }
__device__ __forceinline__ double one_minus(double q)
{
    const double om = 1.0 - q;
    return __double2hiint(om) < 0 ? 0.0 : om;
}

template <class R> struct Mir;
template <> struct Mir<float> {
    using TA = int4;
    __device__ __forceinline__ static const int4 *A(const Bufs &b) { return b.A32; }
    __device__ __forceinline__ static const float4 *B(const Bufs &b) { return b.B32; }
    __device__ __forceinline__ static const float4 *C(const Bufs &b) { return b.C32; }
    __device__ __forceinline__ static float4 *D(const Bufs &b) { return b.D32; }
};
template <> struct Mir<double> {
    using TA = double4_32a;
    __device__ __forceinline__ static const double4_32a *A(const Bufs &b) { return b.A64; }
    __device__ __forceinline__ static const double4_32a *B(const Bufs &b) { return b.B64; }
    __device__ __forceinline__ static const double4_32a *C(const Bufs &b) { return b.C64; }
    __device__ __forceinline__ static double4_32a *D(const Bufs &b) { return b.D64; }
};

__device__ __forceinline__ int mir_type(const int4 &A) { return A.w; }
__device__ __forceinline__ int mir_type(const double4_32a &A) { return __double2loint(A.w); }
__device__ __forceinline__ uint32_t mir_gid(const float4 &D) { return __float_as_uint(D.w); }
__device__ __forceinline__ uint32_t mir_gid(const double4_32a &D) { return (uint32_t)__double2loint(D.w); }
// The density terms of a particle for the pair routine.  FP32 records keep
// p/d^2 in B.w and 1/d in C.w, next to the velocity and the spin, so that a
// pass reading no gid (the second evaluation, normals from the cache) needs
// two records of a partner instead of three; 1/sqrt(d_i d_j) is then formed as
// sqrt(1/d_i 1/d_j).  FP64 records: D = {p/d^2, 1/d, 1/sqrt(d), gid}.
__device__ __forceinline__ float mir_pd2(const float4 &B, const float4 &) { return B.w; }
__device__ __forceinline__ double mir_pd2(const double4_32a &, const double4_32a &D) { return D.x; }
__device__ __forceinline__ float mir_invd(const float4 &C, const float4 &) { return C.w; }
__device__ __forceinline__ double mir_invd(const double4_32a &, const double4_32a &D) { return D.y; }
template <class R> struct K;  // kernel constants in precision R
template <> struct K<float> {
    __device__ __forceinline__ static float inv_rc(const Inst &I) { return I.inv_rcf; }
    __device__ __forceinline__ static float Wc(const Inst &I) { return I.Wcf; }
    __device__ __forceinline__ static float Fc(const Inst &I) { return I.Fcf; }
    __device__ __forceinline__ static float Ca(const Inst &I) { return I.Caf; }
    __device__ __forceinline__ static float Cb(const Inst &I) { return I.Cbf; }
    __device__ __forceinline__ static float Ka(const Inst &I) { return I.Kaf; }
    __device__ __forceinline__ static float Kb(const Inst &I) { return I.Kbf; }
    __device__ __forceinline__ static float isdt(const Inst &I) { return I.isqrt_dtf; }
    __device__ __forceinline__ static float cc(const Inst &I) { return I.coeff_cf; }
    __device__ __forceinline__ static float cd(const Inst &I) { return I.coeff_df; }
    __device__ __forceinline__ static float cr(const Inst &I) { return I.coeff_rf; }
    __device__ __forceinline__ static float ct(const Inst &I) { return I.coeff_tf; }
    __device__ __forceinline__ static float lever(const Inst &I) { return I.lever_fluidf; }
};
template <> struct K<double> {
    __device__ __forceinline__ static double inv_rc(const Inst &I) { return I.inv_rc; }
    __device__ __forceinline__ static double Wc(const Inst &I) { return I.Wc; }
    __device__ __forceinline__ static double Fc(const Inst &I) { return I.Fc; }
    __device__ __forceinline__ static double Ca(const Inst &I) { return I.Ca; }
    __device__ __forceinline__ static double Cb(const Inst &I) { return I.Cb; }
    __device__ __forceinline__ static double Ka(const Inst &I) { return I.Ka; }
    __device__ __forceinline__ static double Kb(const Inst &I) { return I.Kb; }
    __device__ __forceinline__ static double isdt(const Inst &I) { return I.isqrt_dt; }
    __device__ __forceinline__ static double cc(const Inst &I) { return I.coeff_c; }
    __device__ __forceinline__ static double cd(const Inst &I) { return I.coeff_d; }
    __device__ __forceinline__ static double cr(const Inst &I) { return I.coeff_r; }
    __device__ __forceinline__ static double ct(const Inst &I) { return I.coeff_t; }
    __device__ __forceinline__ static double lever(const Inst &I) { return I.lever_fluid; }
};

// Displacement r_ij = r_i - r_j from the mirrors and the exact decision
// r_ij < h (gi: gid of i; j: slot of the partner, used only in the band).
template <class R> struct Rel;
template <> struct Rel<float> {
    __device__ __forceinline__ static bool get(const Bufs &b, const Inst &I, const Geo<float> &geo,
                                               const int4 &Ai, const int4 &Aj, int gi, int j,
                                               float &rx, float &ry, float &rz, float &r2)
    {
        geo.disp(Ai, Aj, rx, ry, rz);
        r2 = rx * rx + ry * ry + rz * rz;
        if (r2 < geo.glo) return true;
        if (r2 > geo.ghi) return false;
        return exact_within(b, I, gi, b.perm[j]);
    }
};
template <> struct Rel<double> {
    __device__ __forceinline__ static bool get(const Bufs &, const Inst &I, const Geo<double> &geo,
                                               const double4_32a &Ai, const double4_32a &Aj, int, int,
                                               double &rx, double &ry, double &rz, double &r2)
    {
        geo.disp(Ai, Aj, rx, ry, rz);
        r2 = __dadd_rn(__dadd_rn(__dmul_rn(rx, rx), __dmul_rn(ry, ry)), __dmul_rn(rz, rz));
        return lt_pos(r2, geo.rc2);
    }
};

// Compensated FP32 sums of two rows at a time (the halves of the packed
// operations).
struct Sum2 {
    F2 s, c;
    // both halves start from v0; value() takes one of them off again
    __device__ __forceinline__ explicit Sum2(float v0) : s(v0), c(0.0f) {}
    // terms v with 0 <= v <= v0, so that |s| >= |v| at every step (Dekker's
    // fast two-sum error term)
    __device__ __forceinline__ void add_small(F2 v)
    {
        const F2 t = add2(s, v);
        c = add2(c, add2(fma2(t, F2(-1.0f), s), v));
        s = t;
    }
    // any terms (Knuth's two-sum)
    __device__ __forceinline__ void add_any(F2 v)
    {
        const F2 t = add2(s, v), z = fma2(s, F2(-1.0f), t);
        const F2 es = fma2(fma2(z, F2(-1.0f), t), F2(-1.0f), s), ev = fma2(z, F2(-1.0f), v);
        c = add2(c, add2(es, ev));
        s = t;
    }
};

// Eq. prtcpres: p = p0 (rho / rho0)^alpha - beta; an integer alpha (7 in
// the paper's cases) by repeated squaring instead of the general power.
__device__ __forceinline__ double eos_pressure(const Inst &I, double rho)
{
    const double x = rho / I.rho0;
    double xa;
    if (I.alpha_int > 0) {
        double r = 1.0, b = x;
        for (int e = I.alpha_int; e; e >>= 1) {
            if (e & 1) r *= b;
            b *= b;
        }
        xa = r;
    } else {
        xa = pow(x, I.alpha);
    }
    return I.p0 * xa - I.beta_p;
}

// Per-particle quantities the force pass reads: p/d^2 and 1/d (FP32), also
// 1/sqrt(d) (FP64), in the precision of the pair arithmetic.
template <class R>
__device__ __forceinline__ void finalize_slot(const Bufs &b, long long s, double d, double p)
{
    if constexpr (sizeof(R) == 4) {
        // FP32 records: p/d^2 beside the velocity, 1/d beside the spin
        const float df = (float)d;
        b.B32[s].w = (float)p / (df * df);
        b.C32[s].w = 1.0f / df;
    } else {
        typename Vec<R>::T4 *D = Mir<R>::D(b);
        typename Vec<R>::T4 o = D[s];
        o.x = p / (d * d);
        o.y = 1.0 / d;
        o.z = 1.0 / sqrt(d);
        D[s] = o;
    }
}

// Streaming accesses (evict-first in L2): the neighbour lists and the normals
// cache are each read or written once per pass and would otherwise push the
// particle records, which every list revisits, out of L2.
__device__ __forceinline__ int ld_stream(const int *p) { return __ldcs(p); }
__device__ __forceinline__ double2 ld_stream(const double2 *p) { return __ldcs(p); }
__device__ __forceinline__ double4_32a ld_stream(const double4_32a *p)
{
    const double2 a = __ldcs((const double2 *)p), b = __ldcs((const double2 *)p + 1);
    return make_double4_32a(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st_stream(float4 *p, float4 v) { __stcs(p, v); }
__device__ __forceinline__ void st_stream(float2 *p, float2 v) { __stcs(p, v); }
__device__ __forceinline__ void st_stream(double2 *p, double2 v) { __stcs(p, v); }
__device__ __forceinline__ void st_stream(double4_32a *p, double4_32a v)
{
    __stcs((double2 *)p, make_double2(v.x, v.y));
    __stcs((double2 *)p + 1, make_double2(v.z, v.w));
}

// The pair passes give a particle LPP lanes and a warp GROUP particles at a
// time, `groups` (1 to 8) times: sub = lane % LPP takes the entries sub,
// sub + LPP, ... of its particle's list.  When a group is done its totals
// move to one lane each, so that the closing arithmetic of up to 32 particles
// (FP64 conversions, the equation of state) runs once per warp on full lanes.
// Results do not depend on `groups`; the launch takes as many as still leave
// the chip full (pass_groups).
__device__ __forceinline__ long long pass_base(int groups)
{
    return ((long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * (GROUP * groups);
}
// What a pass needs to know of a particle before its records: lane i of a warp
// holds slot base + i, loaded once for all its groups and handed to the lanes
// of a particle by shuffles.  (Loaded group by group, this chain of
// dependent loads took longer than the 33 entries a lane then walks.)
struct SlotHead {
    int gi = 0, inst = 0, type = T_OUTER, n = -1, nf = 0;   // n < 0: nothing to do (a slot past the end)
    __device__ __forceinline__ SlotHead() {}
    __device__ __forceinline__ SlotHead(const Bufs &b, long long s, bool live)
    {
        if (live && s < b.N) {
            gi = b.perm[s];
            type = b.stype[s];
            n = b.ncnt[s];
            nf = b.nfirst[s];
            inst = b.pinst[gi];
        }
    }
    __device__ __forceinline__ SlotHead of_group(int g) const
    {
        const int src = g * GROUP + (threadIdx.x & 31) / LPP;
        SlotHead h;
        h.gi = __shfl_sync(0xffffffffu, gi, src);
        h.inst = __shfl_sync(0xffffffffu, inst, src);
        h.type = __shfl_sync(0xffffffffu, type, src);
        h.n = __shfl_sync(0xffffffffu, n, src);
        h.nf = __shfl_sync(0xffffffffu, nf, src);
        return h;
    }
};
// This lane's first two entries of a list [k0, n): fetched for the next group
// while the current one is evaluated.
struct ListHead {
    int e0 = 0, e1 = 0;
    __device__ __forceinline__ ListHead() {}
    __device__ __forceinline__ ListHead(const int *nbr, long long s, int rows, int k0, int n, int sub)
    {
        const int k = k0 + sub;
        if (k < n) e0 = ld_stream(nbr + entry_at(k, s, rows));
        if (k + LPP < n) e1 = ld_stream(nbr + entry_at(k + LPP, s, rows));
    }
};

// The lists of a group asked into L2 (PTX cp.async.bulk.prefetch.L2), while
// the group before it is evaluated: its rows are one block of memory.  The
// loads one and two rows ahead then wait for L2 and not for HBM.
// (s: the group's first slot, a multiple of GROUP; n: entries of this lane's particle)
__device__ __forceinline__ void prefetch_lists(const Bufs &b, long long s, int n)
{
    const int most = __reduce_max_sync(0xffffffffu, n);
    if ((threadIdx.x & 31) == 0 && most > 0)
        asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(b.nbr + entry_at(0, s, b.rows)),
                     "r"(entry_rows(most) * (int)(ROW * sizeof(int)))
                     : "memory");
}

// lane GROUP g + p receives particle p's value (held by every lane of p) in group g
template <class T> __device__ __forceinline__ void keep_group(T v, int g, T &keep)
{
    const int lane = threadIdx.x & 31;
    const T got = __shfl_sync(0xffffffffu, v, (lane % GROUP) * LPP);
    if (lane / GROUP == g) keep = got;
}
template <class T> __device__ __forceinline__ T lanes_sum(T v)
{
#pragma unroll
    for (int o = 1; o < LPP; o <<= 1) v = v + __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ bool lanes_any(bool v)
{
    const unsigned m = __ballot_sync(0xffffffffu, v);
    return (m >> ((threadIdx.x & 31) & ~(LPP - 1))) & ((1u << LPP) - 1u);
}
// FP32 compensated sums: both halves over the lanes of a particle, error terms
// kept (Knuth's two-sum, no ordering of the operands assumed)
__device__ __forceinline__ void join(float &s, float &c, float s2, float c2)
{
    const float t = __fadd_rn(s, s2), z = __fsub_rn(t, s);
    c = __fadd_rn(__fadd_rn(c, c2), __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(s2, z)));
    s = t;
}
__device__ __forceinline__ void lanes_sum(const Sum2 &v, float &s, float &c)
{
    float s2, c2;
    v.s.get(s, s2);
    v.c.get(c, c2);
    join(s, c, s2, c2);
#pragma unroll
    for (int o = 1; o < LPP; o <<= 1) join(s, c, __shfl_xor_sync(0xffffffffu, s, o), __shfl_xor_sync(0xffffffffu, c, o));
}

// ------------------------------------------------------------------ density
// gate: nullptr = always; else only when *gate != 0 (a build just happened)
// Visits the entries k = sub, sub + LPP, ... of [k0, n) of a slot's neighbour
// list (k0 + sub first), calling f(k, entry, record of the partner, side value
// of the partner).  The list index two entries ahead and the record (and side
// value, when `side` is given) one entry ahead are fetched before f runs on
// the current one (the first two indexes by the caller: hd), so the loads of
// the next pair overlap this pair's arithmetic.  NB_FAR entries are visited too (their record is fetched
// without the flag bit).
template <class TA, class F>
__device__ __forceinline__ void for_each_entry(const int *__restrict__ nbr, long long s, int rows, int k0, int n,
                                               int sub, const ListHead &hd, const TA *__restrict__ A,
                                               const double *__restrict__ side, F &&f)
{
    int k = k0 + sub;
    if (k >= n) return;
    const int *__restrict__ nb = nbr + entry_at(k, s, rows);
    uint32_t en = (uint32_t)hd.e0, enn = (uint32_t)hd.e1;
    TA An = A[en & ~NB_FAR];
    double Sn = side ? side[en & ~NB_FAR] : 0.0;
    for (; k < n; k += LPP) {
        const uint32_t e = en;
        const TA Aj = An;
        const double Sj = Sn;
        if (k + LPP < n) {
            en = enn;
            An = A[en & ~NB_FAR];
            if (side) Sn = side[en & ~NB_FAR];
            if (k + 2 * LPP < n) enn = (uint32_t)ld_stream(nb + 2 * ROW);
        }
        nb += ROW;
        f(k, e, Aj, Sj);
    }
}

// Density, pressure and the collision mark of slot s from its kernel sum.
template <class R>
__device__ __forceinline__ void finish_density(const Bufs &b, const Inst &I, int type, long long s, double sum,
                                               bool close, int defer)
{
    // outer-wall particles are not updated (Section 2.5)
    const double d = type == T_OUTER ? I.inv_dx3 : I.Cn * sum;
    double p = eos_pressure(I, I.mf * d);
    if (I.clamp && p < 0.0) p = 0.0;
    b.aclose[s] = close ? 1 : 0;
    b.sd[s] = d;
    b.sp[s] = p;
    // (defer: bit 0 the pressure filter follows, bit 1 the reinitialisation)
    if (sizeof(R) == 4 && defer) b.side32[s] = defer & 2 ? (float)d : (float)p;
    if (!defer) {
        b.sp2[s] = p;
        finalize_slot<R>(b, s, d, p);
    }
}

// The FP64 sum of W / W(0) over the entries [k0, n) of slot s on this lane; close: a
// mobile neighbour inside the collision radius of the artificial viscosity (a
// superset: the collision pass decides exactly; CLOSE: some instance of the
// context has it)
template <bool CLOSE>
__device__ __forceinline__ double density_entries(const Bufs &b, const Inst &I, long long s, int gi, int ti, int k0,
                                                  int n, int sub, bool &close)
{
    const bool want_close = CLOSE && I.artvis && (ti == T_FLUID || ti == T_RIGID);
    const double close_r2 = (double)(I.artvis_r2f_hi * 1.0001f);
    const double4_32a *A = b.A64;
    const double4_32a Ai = A[s];
    const Geo<double> geo(I);
    const double irc = I.inv_rc;
    double acc = 0.0;
    for_each_entry(b.nbr, s, b.rows, k0, n, sub, ListHead(b.nbr, s, b.rows, k0, n, sub), A, nullptr,
                   [&](int, uint32_t e, const double4_32a &Aj, double) {
        if (e & NB_FAR) return;
        double rx, ry, rz, r2;
        if (!Rel<double>::get(b, I, geo, Ai, Aj, gi, (int)e, rx, ry, rz, r2)) return;
        if (CLOSE && want_close && r2 <= close_r2) {
            const int tj = mir_type(Aj);
            close |= (tj == T_FLUID || tj == T_RIGID);
        }
        const double q = root(r2) * irc, om = one_minus(q);
        // a separate rounding of each term (no multiply-add fused into the sum)
        acc = __dadd_rn(acc, (1.0 + 3.0 * q) * om * om * om);
    });
    return acc;
}

template <bool CLOSE>
__global__ void __launch_bounds__(256) k_density(Bufs b, int defer, const int *gate, int groups)
{
    if (gate && *gate == 0) return;
    const int lane = threadIdx.x & 31, sub = lane % LPP;
    const long long base = pass_base(groups);
    if (base == 0 && lane == 0) *b.aclose_ok = 1;   // the marks below are for these positions
    const SlotHead mine(b, base + lane, lane < groups * GROUP);
    double kown = 0.0, koth = 0.0;
    int kclose = 0;
    for (int g = 0; g < groups; ++g) {
        const long long s = base + g * GROUP + lane / LPP;
        const SlotHead h = mine.of_group(g);
        bool close = false;
        double own = 0.0, oth = 0.0;
        if (h.type != T_OUTER) {
            // the owned and the other entries apart, as the half-pair form
            // sums them (the same additions)
            const Inst &I = b.inst[h.inst];
            own = density_entries<CLOSE>(b, I, s, h.gi, h.type, 0, h.nf, sub, close);
            oth = density_entries<CLOSE>(b, I, s, h.gi, h.type, h.nf, h.n, sub, close);
        }
        keep_group(lanes_sum(own), g, kown);
        keep_group(lanes_sum(oth), g, koth);
        if constexpr (CLOSE) keep_group((int)lanes_any(close), g, kclose);
    }
    const long long s = base + lane;
    if (lane >= groups * GROUP || s >= b.N) return;
    const Inst &I = b.inst[mine.inst];
    finish_density<double>(b, I, mine.type, s, I.W0 * __dadd_rn(__dadd_rn(1.0, kown), koth), kclose, defer);
}

// FP64 density with each unordered pair evaluated once (Newton 3): phase 1
// sums W / W(0) over the owned prefix of the list and stores each for the partner
// (negated when the pair lies inside the collision radius of the artificial
// viscosity; 0 for pairs beyond h) in the partner's column of the pair
// buffer, which is free between force passes (a scattered store, which does
// not stall the thread); phase 2 reads its own column in entry order
// (coalesced).  The partner's r_ji = -r_ij bit for bit and the terms are
// added in the same order ([owned], [not owned], lane by lane) as in
// k_density, so the result is the same.
__global__ void __launch_bounds__(256) k_density_half(Bufs b, const int *gate, int groups)
{
    if (gate && *gate == 0) return;
    const int lane = threadIdx.x & 31, sub = lane % LPP;
    const long long base = pass_base(groups);
    if (base == 0 && lane == 0) *b.aclose_ok = 1;
    const double4_32a *A = Mir<double>::A(b);
    double *__restrict__ wb = (double *)b.resB;
    const int capown = b.capown;
    const SlotHead mine(b, base + lane, lane < groups * GROUP);
    double keep = 0.0;
    int kclose = 0;
    for (int g = 0; g < groups; ++g) {
        const long long s = base + g * GROUP + lane / LPP;
        const SlotHead h = mine.of_group(g);
        double acc = 0.0;
        bool close = false;
        if (s < b.N) {
            const int gi = h.gi, ti = h.type;
            const Inst &I = b.inst[h.inst];
            const double4_32a Ai = A[s];
            const Geo<double> geo(I);
            const double close_r2 = (double)(I.artvis_r2f_hi * 1.0001f);
            const bool want_close = I.artvis != 0;
            const double irc = K<double>::inv_rc(I);
            for_each_entry(b.nbr, s, b.rows, 0, h.nf, sub, ListHead(b.nbr, s, b.rows, 0, h.nf, sub), A, nullptr,
                           [&](int k, uint32_t e, const double4_32a &Aj, double) {
                double W = 0.0;
                if (!(e & NB_FAR)) {
                    double rx, ry, rz, r2;
                    if (Rel<double>::get(b, I, geo, Ai, Aj, gi, (int)e, rx, ry, rz, r2)) {
                        const double q = root(r2) * irc, om = one_minus(q);
                        W = (1.0 + 3.0 * q) * om * om * om;
                        acc = __dadd_rn(acc, W);
                        if (want_close && r2 <= close_r2) {
                            const int tj = mir_type(Aj);
                            const bool mob = (tj == T_FLUID || tj == T_RIGID);
                            if (mob && (ti == T_FLUID || ti == T_RIGID)) {
                                close = true;
                                W = flip_sign(W, 0x80000000u);   // tells the partner
                            }
                        }
                    }
                }
                // into the partner's column, at the row of its entry for this pair
                const int row = __ldg(b.rev + entry_at(k, s, b.rows));
                if (row < capown) wb[entry_at(row, e & ~NB_FAR, b.rows_own)] = W;
            });
        }
        keep_group(lanes_sum(acc), g, keep);
        keep_group((int)lanes_any(close), g, kclose);
    }
    const long long s = base + lane;
    if (lane >= groups * GROUP || s >= b.N) return;
    b.sd[s] = keep;   // partial; completed by k_density_gather
    b.aclose[s] = kclose ? 1 : 0;
}

__global__ void __launch_bounds__(256) k_density_gather(Bufs b, int defer, const int *gate, int groups)
{
    if (gate && *gate == 0) return;
    const int lane = threadIdx.x & 31, sub = lane % LPP;
    const long long base = pass_base(groups);
    const double *__restrict__ wb = (const double *)b.resB;
    const SlotHead mine(b, base + lane, lane < groups * GROUP);
    double keep = 0.0;
    int kclose = 0;
    for (int g = 0; g < groups; ++g) {
        const long long s = base + g * GROUP + lane / LPP;
        const SlotHead h = mine.of_group(g);
        double acc = 0.0;
        bool close = false;
        if (h.type != T_OUTER) {
            // the owners wrote W of this particle's non-owned entries into
            // its own column (more rows than capown only after a list error,
            // flagged; 0 for an entry beyond h)
            const int m = min(h.n - h.nf, b.capown);
            const double *__restrict__ p = wb + entry_at(sub, s, b.rows_own);
#pragma unroll 4
            for (int k = sub; k < m; k += LPP) {
                const double w = *p;
                p += ROW;
                close |= __double2hiint(w) < 0;
                acc = __dadd_rn(acc, __hiloint2double(hi_abs(w), __double2loint(w)));
            }
        }
        keep_group(lanes_sum(acc), g, keep);
        keep_group((int)lanes_any(close), g, kclose);
    }
    const long long s = base + lane;
    if (lane >= groups * GROUP || s >= b.N) return;
    const int ti = mine.type;
    const Inst &I = b.inst[mine.inst];
    const bool close = (b.aclose[s] != 0 || kclose) && (ti == T_FLUID || ti == T_RIGID);
    finish_density<double>(b, I, ti, s, I.W0 * __dadd_rn(__dadd_rn(1.0, b.sd[s]), keep), close, defer);
}

// ------------------------------------------------------ density reinitialisation
// Shepard reinitialisation of the summation density (after Colagrossi and
// Landrini; the text under Algorithm 1): d~_i = (W(0) + sum_j W_ij) /
// (W(0)/d_i + sum_j W_ij/d_j) over the density neighbours, outer walls keep
// theirs; the pressure follows from Eq. prtcpres.  The new densities go to
// sdr (the neighbours' old values are still read) and k_reinit_copy moves
// them back.
// The FP64 ratio of two kernel sums over the list of slot s (on all lanes of
// the particle): numerator and denominator of the two Shepard averages.
template <bool REINIT>
__device__ __forceinline__ void shepard_entries(const Bufs &b, const Inst &I, long long s, const SlotHead &h, int sub,
                                                double &num, double &den)
{
    const double4_32a *A = b.A64;
    const double4_32a Ai = A[s];
    const Geo<double> geo(I);
    for_each_entry(b.nbr, s, b.rows, 0, h.n, sub, ListHead(b.nbr, s, b.rows, 0, h.n, sub), A, REINIT ? b.sd : b.sp,
                   [&](int, uint32_t e, const double4_32a &Aj, double v) {
        if (e & NB_FAR) return;
        double rx, ry, rz, r2;
        if (!Rel<double>::get(b, I, geo, Ai, Aj, h.gi, (int)e, rx, ry, rz, r2)) return;
        const double q = root(r2) * I.inv_rc, om = one_minus(q);
        const double W = I.Wc * (1.0 + 3.0 * q) * om * om * om;
        // a separate rounding of each term (no multiply-add fused into the sum)
        num = __dadd_rn(num, REINIT ? W : __dmul_rn(v, W));
        den = __dadd_rn(den, REINIT ? __ddiv_rn(W, v) : W);
    });
}

// What the two averages do with their sums: reinitialised density and
// pressure, or filtered pressure.
template <class R, bool REINIT>
__device__ __forceinline__ void finish_shepard(const Bufs &b, const Inst &I, int type, long long s, double num, double den,
                                               int any_filter)
{
    const bool on = (REINIT ? I.reinit : I.filter) && type != T_OUTER;
    if constexpr (REINIT) {
        const double di = b.sd[s];
        const double d = on ? (I.W0 + num) / (I.W0 / di + den) : di;
        double p = eos_pressure(I, I.mf * d);
        if (I.clamp && p < 0.0) p = 0.0;
        b.sdr[s] = d;
        if (I.reinit) b.sp[s] = p;
        if (!any_filter) {
            b.sp2[s] = b.sp[s];
            finalize_slot<R>(b, s, d, b.sp[s]);
        }
    } else {
        const double pi = b.sp[s];
        const double pf = on ? (pi * I.W0 + num) / (I.W0 + den) : pi;
        b.sp2[s] = pf;
        finalize_slot<R>(b, s, b.sd[s], pf);
    }
}

template <bool REINIT>
__global__ void __launch_bounds__(256) k_shepard(Bufs b, int any_filter, const int *gate, int groups)
{
    if (gate && *gate == 0) return;
    const int lane = threadIdx.x & 31, sub = lane % LPP;
    const long long base = pass_base(groups);
    const SlotHead mine(b, base + lane, lane < groups * GROUP);
    double knum = 0.0, kden = 0.0;
    for (int g = 0; g < groups; ++g) {
        const SlotHead h = mine.of_group(g);
        const Inst &I = b.inst[h.inst];
        double num = 0.0, den = 0.0;
        if (h.type != T_OUTER && (REINIT ? I.reinit : I.filter))
            shepard_entries<REINIT>(b, I, base + g * GROUP + lane / LPP, h, sub, num, den);
        keep_group(lanes_sum(num), g, knum);
        keep_group(lanes_sum(den), g, kden);
    }
    const long long s = base + lane;
    if (lane >= groups * GROUP || s >= b.N) return;
    finish_shepard<double, REINIT>(b, b.inst[mine.inst], mine.type, s, knum, kden, any_filter);
}


__global__ void k_reinit_copy(Bufs b, const int *gate)
{
    if (gate && *gate == 0) return;
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= b.N) return;
    b.sd[s] = b.sdr[s];
    if (b.side32) b.side32[s] = (float)b.sp[s];   // for the pressure filter
}

// The r < h decision of a pair in the guard band, out of line: it is rare,
// and its FP64 code would cost the pair loop registers.
__device__ __noinline__ bool within_exactly(const Bufs &b, int inst, int gi, int j)
{
    return exact_within(b, b.inst[inst], gi, b.perm[j]);
}

// The loops below take ZR rows at a time, unrolled, so that a row costs no
// counters and no moves between registers.  Lists: a lane's ZR entries of the
// next rows are fetched while the present ones are evaluated (a lane without
// an entry reads record 0 and adds nothing).
constexpr int ZR = 4;
struct ListRows {
    int e[ZR];
    // (nb: this lane's entry of the first of the rows, n: entries left from it on)
    __device__ __forceinline__ void load(const int *nb, int n)
    {
#pragma unroll
        for (int i = 0; i < ZR; ++i) e[i] = i * LPP < n ? ld_stream(nb + i * ROW) : 0;
    }
};

// ---------------------------------- density and Shepard averages, FP32
// These passes are a list walk with little arithmetic a pair: bound by issue
// slots.  The 8 lanes of a particle take ZR rows at a time, unrolled, two rows
// in the halves of the packed operations: 52 instructions an entry where one
// entry at a time with branches and a library square root took 80, and 0.40
// ms where that took 0.65 (662,305 particles).  The gathers of positions then
// bound them by latency: 64 registers, with a few of them spilled, and 32 warps
// an SM beat 80 and none with 24 (0.395 -> 0.342 ms; 48 registers: 0.349), and
// the Shepard averages fetch the neighbours' values with the positions (density
// and pressure filter of 374,000 particles 0.377 -> 0.330 ms).
//
// f(W, v0, v1, ok0, ok1, r2_0, r2_1, type0, type1) sees the kernel weights of
// two entries (0 for an entry past the end, beyond h or of contact range only)
// and, with SIDE, their values in side32, fetched with the positions.
template <bool SIDE, class F>
__device__ __forceinline__ void weights32(const Bufs &b, const Inst &I, const SlotHead &h, long long s, int n, int gr,
                                          int sub, F &&f)
{
    const Geo<float> geo(I);
    const F2 u0(geo.u0), u1(geo.u1), u2(geo.u2), irc(I.inv_rcf), Wc(I.Wcf), one(1.0f), minus(-1.0f);
    const float beyond = 4.0f * geo.ghi;   // stands for r^2 of an entry left out: W = 0
    const int4 Ai = b.A32[s];
    const int *__restrict__ nb = b.nbr + entry_at(sub, s, b.rows);
    int left = n - sub;   // this lane has an entry in row i of the present ones when i LPP < left
    ListRows cur, next;
    cur.load(nb, left);
    int4 A[2] = { b.A32[cur.e[0] & ~NB_FAR], b.A32[cur.e[1] & ~NB_FAR] };   // two rows ahead
    float V[2] = { 0.f, 0.f };
    if (SIDE)
        for (int t = 0; t < 2; ++t) V[t] = b.side32[cur.e[t] & ~NB_FAR];
    for (int r0 = 0; r0 < gr; r0 += ZR) {
        nb += ZR * ROW;
        next.load(nb, left - ZR * LPP);
#pragma unroll
        for (int i = 0; i < ZR; i += 2) {
            if (i && r0 + i >= gr) break;   // uniform
            const int e0 = cur.e[i], e1 = cur.e[i + 1];
            const int4 A0 = A[0], A1 = A[1];
            const float v0 = V[0], v1 = V[1];
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const int jn = (i + 2 < ZR ? cur.e[(i + 2 + t) % ZR] : next.e[t]) & ~NB_FAR;
                A[t] = b.A32[jn];
                if (SIDE) V[t] = b.side32[jn];
            }
            const F2 rx = mul2(F2((float)fixed_diff(Ai.x, A0.x), (float)fixed_diff(Ai.x, A1.x)), u0);
            const F2 ry = mul2(F2((float)fixed_diff(Ai.y, A0.y), (float)fixed_diff(Ai.y, A1.y)), u1);
            const F2 rz = mul2(F2((float)fixed_diff(Ai.z, A0.z), (float)fixed_diff(Ai.z, A1.z)), u2);
            float a0, a1;
            fma2(rz, rz, fma2(ry, ry, mul2(rx, rx))).get(a0, a1);
            bool ok0 = i * LPP < left && e0 >= 0 && a0 < geo.ghi, ok1 = (i + 1) * LPP < left && e1 >= 0 && a1 < geo.ghi;
            if (ok0 && a0 >= geo.glo) ok0 = within_exactly(b, h.inst, h.gi, e0);
            if (ok1 && a1 >= geo.glo) ok1 = within_exactly(b, h.inst, h.gi, e1);
            // (coincident particles: r = 0 and W = W(0), not 0 times infinity)
            const float c0 = ok0 ? fmaxf(a0, 1.2e-38f) : beyond, c1 = ok1 ? fmaxf(a1, 1.2e-38f) : beyond;
            // sqrt by Newton's iteration from the hardware reciprocal root:
            // s + (x - s^2) y / 2, within an ulp's half but for rare ties
            const F2 x(c0, c1), y(rsqrt_ftz(c0), rsqrt_ftz(c1));
            const F2 t = mul2(x, y), e = fma2(mul2(t, minus), t, x);
            const F2 q = mul2(fma2(e, mul2(y, F2(0.5f)), t), irc);
            float m0, m1;
            fma2(q, minus, one).get(m0, m1);
            const F2 om(fmaxf(m0, 0.0f), fmaxf(m1, 0.0f));
            const F2 W = mul2(mul2(mul2(mul2(Wc, fma2(q, F2(3.0f), one)), om), om), om);
            f(W, v0, v1, ok0, ok1, a0, a1, A0.w, A1.w);
        }
        cur = next;
        left -= ZR * LPP;
    }
}

template <bool CLOSE>
__global__ void __launch_bounds__(256, 4) k_density32(Bufs b, int defer, const int *gate, int groups)
{
    if (gate && *gate == 0) return;
    const int lane = threadIdx.x & 31, sub = lane % LPP;
    const unsigned FULL = 0xffffffffu;
    const long long base = pass_base(groups);
    if (base == 0 && lane == 0) *b.aclose_ok = 1;   // the marks below are for these positions
    SlotHead mine(b, base + lane, lane < groups * GROUP);
    if (mine.type == T_OUTER) mine.n = 0;
    float ks = 0.f, kc = 0.f;
    int kclose = 0;
    for (int g = 0; g < groups; ++g) {
        const SlotHead h = mine.of_group(g);
        if (g + 1 < groups) prefetch_lists(b, base + (g + 1) * GROUP, mine.of_group(g + 1).n);
        const int gr = entry_rows(__reduce_max_sync(FULL, max(h.n, 0)));
        const Inst &I = b.inst[h.inst];
        const float W0 = (float)I.W0;
        Sum2 sum(W0);
        bool close = false;
        if (gr > 0) {
            const bool want_close = CLOSE && I.artvis && (h.type == T_FLUID || h.type == T_RIGID);
            const float close_r2 = want_close ? I.artvis_r2f_hi * 1.0001f : -1.0f;
            const long long s = h.n > 0 ? base + g * GROUP + lane / LPP : 0;
            weights32<false>(b, I, h, s, h.n, gr, sub,
                      [&](F2 W, float, float, bool ok0, bool ok1, float r0, float r1, int t0, int t1) {
                sum.add_small(W);
                if (CLOSE) {
                    close |= ok0 && r0 <= close_r2 && (t0 == T_FLUID || t0 == T_RIGID);
                    close |= ok1 && r1 <= close_r2 && (t1 == T_FLUID || t1 == T_RIGID);
                }
            });
        }
        float ss, cc;
        lanes_sum(sum, ss, cc);
        keep_group(ss, g, ks);
        keep_group(cc, g, kc);
        if constexpr (CLOSE) keep_group((int)lanes_any(close), g, kclose);
    }
    const long long s = base + lane;
    if (lane >= groups * GROUP || s >= b.N) return;
    const Inst &I = b.inst[mine.inst];
    // the sum held W(0) once in each half of each lane
    const double v = ((double)ks - (double)(2 * LPP - 1) * (double)(float)I.W0) + (double)kc;
    finish_density<float>(b, I, mine.type, s, v, kclose, defer);
}

template <bool REINIT>
__global__ void __launch_bounds__(256, 4) k_shepard32(Bufs b, int any_filter, const int *gate, int groups)
{
    if (gate && *gate == 0) return;
    const int lane = threadIdx.x & 31, sub = lane % LPP;
    const unsigned FULL = 0xffffffffu;
    const long long base = pass_base(groups);
    SlotHead mine(b, base + lane, lane < groups * GROUP);
    if (mine.type == T_OUTER || !(REINIT ? b.inst[mine.inst].reinit : b.inst[mine.inst].filter)) mine.n = 0;
    float kn[2] = { 0.f, 0.f }, kd[2] = { 0.f, 0.f };
    for (int g = 0; g < groups; ++g) {
        const SlotHead h = mine.of_group(g);
        if (g + 1 < groups) prefetch_lists(b, base + (g + 1) * GROUP, mine.of_group(g + 1).n);
        const int gr = entry_rows(__reduce_max_sync(FULL, max(h.n, 0)));
        Sum2 num(0.0f), den(REINIT ? 0.0f : (float)b.inst[h.inst].W0);   // (0 <= W <= W(0), see k_density32)
        if (gr > 0) {
            const Inst &I = b.inst[h.inst];
            const long long s = h.n > 0 ? base + g * GROUP + lane / LPP : 0;
            weights32<true>(b, I, h, s, h.n, gr, sub,
                      [&](F2 W, float v0, float v1, bool ok0, bool ok1, float, float, int, int) {
                if constexpr (REINIT) {
                    float w0, w1;
                    W.get(w0, w1);
                    num.add_any(W);
                    den.add_any(F2(ok0 ? w0 / v0 : 0.f, ok1 ? w1 / v1 : 0.f));
                } else {
                    num.add_any(mul2(F2(v0, v1), W));
                    den.add_small(W);
                }
            });
        }
        float ss, cc;
        lanes_sum(num, ss, cc);
        keep_group(ss, g, kn[0]);
        keep_group(cc, g, kn[1]);
        lanes_sum(den, ss, cc);
        keep_group(ss, g, kd[0]);
        keep_group(cc, g, kd[1]);
    }
    const long long s = base + lane;
    if (lane >= groups * GROUP || s >= b.N) return;
    const double den0 = REINIT ? 0.0 : (double)(2 * LPP) * (double)(float)b.inst[mine.inst].W0;   // once in each half of each lane
    finish_shepard<float, REINIT>(b, b.inst[mine.inst], mine.type, s, (double)kn[0] + (double)kn[1],
                                  ((double)kd[0] - den0) + (double)kd[1], any_filter);
}

// ---------------------------------------------------------------- drag (A5)
// r = x_i - x_j with the minimum image; returns the oracle's r^2 (no FMA).
__device__ __forceinline__ double exact_disp(const double *xi, const double *xj, const Inst &I, double r[3])
{
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double t = __dsub_rn(xi[a], xj[a]);
        if (I.periodic[a]) {
            const double hL = 0.5 * I.box[a];
            if (t > hL) t = __dsub_rn(t, I.box[a]);
            else if (t < -hL) t = __dadd_rn(t, I.box[a]);
        }
        r[a] = t;
    }
    return __dadd_rn(__dadd_rn(__dmul_rn(r[0], r[0]), __dmul_rn(r[1], r[1])), __dmul_rn(r[2], r[2]));
}

// The sphere kernels run one warp per rigid particle, RB / 32 particles per
// block: the lanes stride over its neighbour list and the partial sums are
// reduced by a fixed butterfly of shuffles, so the result does not depend on
// scheduling.
constexpr int RB = 128;
constexpr int RPB = RB / 32;   // rigid particles per block

template <int K>
__device__ __forceinline__ void warp_sum_all(double (&v)[K])
{
#pragma unroll
    for (int a = 0; a < K; ++a) v[a] = warp_sum(v[a]);
}

// Per rigid particle s (one warp each, lanes striding over its neighbour
// list, order-fixed reduction): the rigid volume within h, sum W and
// sum W v over fluid neighbours (Eq. fvfdef, Section 2.4); k_drag_law then forms
// eps_s (s included), v_f = sum W v / sum W and the drag along (v_f - v_s)
// with the Ergun (eps <= 0.8) or Wen-Yu (eps > 0.8) coefficient in the closed
// form that stays finite at eps -> 1 and |v_f - v_s| -> 0.
template <class R>
__global__ void __launch_bounds__(RB) k_drag(Bufs b)
{
    const int r = blockIdx.x * RPB + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (r >= b.nrigid) return;   // the whole warp
    const int g = b.rigid_gid[r];
    const long long s = b.slot_of[g];
    const Inst &I = b.inst[b.pinst[g]];
    double Vsum = 0.0, S = 0.0, U0 = 0.0, U1 = 0.0, U2 = 0.0;
    const int n = b.ncnt[s];
    // the kernel-weighted fluid sums in precision R on the mirrors (the
    // exact r < h decision of Rel), per lane in R; the volumes in FP64
    using T4 = typename Vec<R>::T4;
    using TA = typename Mir<R>::TA;
    const Geo<R> geo(I);
    const TA *__restrict__ A = Mir<R>::A(b);
    const T4 *__restrict__ Bm = Mir<R>::B(b);
    const TA Ai = A[s];
    const R Wc = K<R>::Wc(I), irc = K<R>::inv_rc(I);
    R Sr = 0, u0 = 0, u1 = 0, u2 = 0;
    // the loads of U entries of the lane stand before their arithmetic: a
    // list of 270 entries is two or three waits long, not nine (8,000 spheres:
    // 22 -> 15 us)
    constexpr int U = 4;
    for (int k0 = lane; k0 < n; k0 += 32 * U) {
        uint32_t e[U];
        TA Au[U];
        T4 Bu[U];
#pragma unroll
        for (int u = 0; u < U; ++u) e[u] = k0 + 32 * u < n ? (uint32_t)__ldg(b.nbr + entry_at(k0 + 32 * u, s, b.rows)) : NB_FAR;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int j = (int)(e[u] & ~NB_FAR);   // (slot 0 past the end: in range, not used)
            Au[u] = A[j];
            Bu[u] = Bm[j];
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (e[u] & NB_FAR) continue;
            const int j = (int)e[u], tj = mir_type(Au[u]);
            if (tj != T_RIGID && tj != T_FLUID) continue;
            R rx, ry, rz, r2;
            if (!Rel<R>::get(b, I, geo, Ai, Au[u], g, j, rx, ry, rz, r2)) continue;
            if (tj == T_RIGID) {
                const double Rj = b.R[b.perm[j]];
                Vsum += 4.0 / 3.0 * PI * Rj * Rj * Rj;
            } else {
                const R q = root(r2) * irc, om = R(1) - q;
                const R W = Wc * (R(1) + R(3) * q) * om * om * om;
                Sr += W;
                u0 += W * Bu[u].x;
                u1 += W * Bu[u].y;
                u2 += W * Bu[u].z;
            }
        }
    }
    S = Sr; U0 = u0; U1 = u1; U2 = u2;
    double sums[5] = { Vsum, S, U0, U1, U2 };
    warp_sum_all(sums);
    if (lane == 0)
        for (int a = 0; a < 5; ++a) b.dsum[5 * r + a] = sums[a];
}

// The drag law of each rigid particle from its sums: two lanes each, which
// share the two FP64 powers (their chain is what the kernel takes: 16.6 us with
// one lane, 13.8 us; one warp a block, so that the chains lie on many SMs).
__global__ void __launch_bounds__(32) k_drag_law(Bufs b)
{
    const int idx = (int)(blockIdx.x * 32u + threadIdx.x), r = min(idx >> 1, b.nrigid - 1), second = idx & 1;
    const int g = b.rigid_gid[r];
    const long long s = b.slot_of[g];
    const Inst &I = b.inst[b.pinst[g]];
    const double Ri = b.R[g];
    const double *sums = b.dsum + 5 * r;
    const double Vsum = sums[0] + 4.0 / 3.0 * PI * Ri * Ri * Ri;
    const double S = sums[1];
    const double U[3] = { sums[2], sums[3], sums[4] };
    double eps = fabs(I.Vf - Vsum) / I.Vf;
    eps = fmin(fmax(eps, I.eps_min), 1.0);
    double dv[3] = { 0.0, 0.0, 0.0 };
    if (S > 0.0)
        for (int a = 0; a < 3; ++a) dv[a] = U[a] / S - b.v[3 * g + a];
    const double mag = sqrt(dv[0] * dv[0] + dv[1] * dv[1] + dv[2] * dv[2]);
    const double d = 2.0 * Ri, Vs = 4.0 / 3.0 * PI * Ri * Ri * Ri;
    const double Re = I.rho0 * d * eps * mag / I.eta;
    const double power = S > 0.0 && eps > 0.8 ? pow(second ? eps : Re, second ? -2.65 : 0.687) : 0.0;
    const double eps265 = __shfl_xor_sync(0xffffffffu, power, 1);   // (the first lane's view)
    if (second || idx >> 1 >= b.nrigid) return;
    double F[3] = { 0.0, 0.0, 0.0 };
    if (S > 0.0) {
        double coef;
        if (eps <= 0.8) {
            coef = 150.0 * I.eta * (1.0 - eps) / (eps * d * d) + 1.75 * I.rho0 * mag / d;
        } else {
            const double cdre = (Re <= 1000.0) ? 24.0 * (1.0 + 0.15 * power) : 0.44 * Re;
            coef = 0.75 * cdre * I.eta * eps265 / (d * d);
        }
        for (int a = 0; a < 3; ++a) F[a] = coef * Vs * dv[a];
        b.rxn[s] = make_double4_32a(F[0] / S, F[1] / S, F[2] / S, 0.0);
        b.rxn32[s] = make_float4((float)(F[0] / S), (float)(F[1] / S), (float)(F[2] / S), 0.f);
    } else {
        b.rxn[s] = make_double4_32a(0.0, 0.0, 0.0, 0.0);
        b.rxn32[s] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    b.eps[r] = eps;
    b.fdg[3 * r] = F[0];
    b.fdg[3 * r + 1] = F[1];
    b.fdg[3 * r + 2] = F[2];
}

// External acceleration (Eq. govern, F^EXT): uniform g plus the
// reverse-Poiseuille forcing, + on the lower half of split_axis, - above.
__device__ __forceinline__ void ext_accel(const Inst &I, const double *x, double a[3])
{
    a[0] = I.g[0];
    a[1] = I.g[1];
    a[2] = I.g[2];
    if (I.body_amp != 0.0) {
        const double rel = x[I.split_axis] - I.origin[I.split_axis];
        a[I.body_axis] += (rel < 0.5 * I.box[I.split_axis]) ? I.body_amp : -I.body_amp;
    }
}

// -------------------------------------------------------- fluid force pass
// Constants of the SDPD pair force on one particle i in precision R, held in
// registers.  With om = 1 - q and g = om^2 / d_j the coefficients of Eqs. FijC,
// FijD, FijR and FijT are products of g or om and constants of i:
//   PC = cc Fc, A1 = -cd Ca Fc/d_i, A2 = cd (Ca + 2 Cb) Fc/(3 d_i),
//   A3 = -cr Ca Fc/(2 d_i) (gamma_a = Ca F/(d_i d_j), gamma_b = Cb F/(d_i d_j)),
//   T1 = ct Ka/sqrt(dt d_i), T3 = ct (Kb - Ka)/(3 sqrt(dt d_i)) (sigma = K
//   sqrt(F)/sqrt(d_i d_j)).  FP32 takes one root of the product instead, X = S/d_i
//   times 1/d_j with S = 4^m, and T1, T3 hold 2^-m in the place of 1/sqrt(d_i):
//   one hardware root a pair, the same bits seen from i and from j.  (Two, one of
//   each density, save a product: 0.7 % of a step of 1.6M particles, at 1.3 times
//   the factor's rms error.)
template <class R> struct PairK {
    R irc, Wc, PC, A1, A2, A3, T1, T3, X;
    bool noise;
    uint32_t step, key0, key1;
    template <class T4>
    __device__ __forceinline__ PairK(const Inst &I, uint32_t st, const T4 &Ci, const T4 &Di)
        : irc(K<R>::inv_rc(I)), Wc(K<R>::Wc(I)), PC(K<R>::cc(I) * K<R>::Fc(I)), noise(I.noise != 0), step(st),
          key0(I.key0), key1(I.key1)
    {
        const R fd = K<R>::Fc(I) * mir_invd(Ci, Di);
        A1 = -K<R>::cd(I) * K<R>::Ca(I) * fd;
        A2 = K<R>::cd(I) * (K<R>::Ca(I) + R(2) * K<R>::Cb(I)) * R(1.0 / 3.0) * fd;
        A3 = R(-0.5) * K<R>::cr(I) * K<R>::Ca(I) * fd;
        R t = K<R>::ct(I) * K<R>::isdt(I);
        if constexpr (sizeof(R) == 4) {
            X = mir_invd(Ci, Di) * I.d_scale;
            t *= I.d_unscale;
        } else {
            t *= Di.z;
        }
        T1 = t * K<R>::Ka(I);
        T3 = t * (K<R>::Kb(I) - K<R>::Ka(I)) * R(1.0 / 3.0);
    }
};


// om times what T1 and T3 leave of 1/sqrt(d_i d_j): FP32 x rsqrt(x) of x = X/d_j
// (the hardware reciprocal root, about 2 ulp), FP64 1/sqrt(d_j).
__device__ __forceinline__ float root_weight(const PairK<float> &P, float om, const float4 &Cj, const float4 &)
{
    const float x = P.X * Cj.w;
    return om * (x * rsqrt_ftz(x));
}
__device__ __forceinline__ double root_weight(const PairK<double> &, double om, const double4_32a &, const double4_32a &Dj)
{
    return om * Dj.z;
}

// Correctly rounded operations in precision R that the compiler may not
// contract or reorder.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float sub_rn(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ double sub_rn(double a, double b) { return __dsub_rn(a, b); }

// Kernel weight W(r) = Wc (1 + 3q)(1 - q)^3 of a pair for the drag reaction
// (Eq. F_fpi_DG_reac), every rounding explicit.
template <class R>
__device__ __forceinline__ R drag_weight(const PairK<R> &P, R q, R om)
{
    return mul_rn(mul_rn(mul_rn(mul_rn(P.Wc, fma_rn(R(3), q, R(1))), om), om), om);
}

template <class R> struct Z6 {
    R z0, z1, z2, z3, z4, z5;
};

// f = o + ce e and h = e x o of a pair in a fixed operation order, so that
// the partner of the split path, which rebuilds them from {o, ce} and its
// own (negated, bitwise equal) e, gets the owner's values exactly.
__device__ __forceinline__ void pair_fh(float ox, float oy, float oz, float ce, float ex, float ey, float ez,
                                        float &gx, float &gy, float &gz, float &hx, float &hy, float &hz)
{
    gx = __fmaf_rn(ce, ex, ox);
    gy = __fmaf_rn(ce, ey, oy);
    gz = __fmaf_rn(ce, ez, oz);
    hx = __fmaf_rn(ey, oz, -__fmul_rn(ez, oy));
    hy = __fmaf_rn(ez, ox, -__fmul_rn(ex, oz));
    hz = __fmaf_rn(ex, oy, -__fmul_rn(ey, ox));
}
__device__ __forceinline__ void pair_fh(double ox, double oy, double oz, double ce, double ex, double ey, double ez,
                                        double &gx, double &gy, double &gz, double &hx, double &hy, double &hz)
{
    gx = fma(ce, ex, ox);
    gy = fma(ce, ey, oy);
    gz = fma(ce, ez, oz);
    hx = fma(ey, oz, -__dmul_rn(ez, oy));
    hy = fma(ez, ox, -__dmul_rn(ex, oz));
    hz = fma(ex, oy, -__dmul_rn(ey, ox));
}

// SDPD force on i from j (Eqs. FijC, FijD, FijR, FijT) for a pair already
// known to lie within h, written as
//   f = o + ce * e,   o = the part not along e_ij (v_ij, rotational, random),
// so the torque (-l e) x f = -l e x o needs only o.  with_rt: rotational and
// random parts (not for pairs with a rigid particle, Section 2.4).  zmode:
// 0 draw the six normals into z, 1 use z as given.  Also returns e, q, 1 - q.
template <class R, class T4>
__device__ __forceinline__ void sdpd_pair(const PairK<R> &P, R rx, R ry, R rz, R r2, const T4 &Bi,
                                          const T4 &Ci, const T4 &Di, const T4 &Bj, const T4 &Cj,
                                          const T4 &Dj, bool with_rt, int zmode, Z6<R> &z, R &ox,
                                          R &oy, R &oz, R &ce, R &ex, R &ey, R &ez, R &q, R &om)
{
    const R is2 = R(0.70710678118654752440);
    R r, ir;
    root_and_inverse(r2, r, ir);
    q = r * P.irc;
    om = one_minus(q);
    const R om2 = om * om, g = om2 * mir_invd(Cj, Dj);
    ex = rx * ir; ey = ry * ir; ez = rz * ir;
    const R vx = Bi.x - Bj.x, vy = Bi.y - Bj.y, vz = Bi.z - Bj.z;
    const R ev = ex * vx + ey * vy + ez * vz;
    const R c1 = P.A1 * g;
    // Eq. FijC (central) + the central part of Eq. FijD
    ce = P.PC * (mir_pd2(Bi, Di) + mir_pd2(Bj, Dj)) * (om2 * r) - P.A2 * g * ev;
    ox = c1 * vx; oy = c1 * vy; oz = c1 * vz;
    if (!with_rt) return;
    // Eq. FijR
    const R wx = Ci.x + Cj.x, wy = Ci.y + Cj.y, wz = Ci.z + Cj.z;
    const R c3 = P.A3 * g;
    ox += c3 * (ry * wz - rz * wy);
    oy += c3 * (rz * wx - rx * wz);
    oz += c3 * (rx * wy - ry * wx);
    // Eq. FijT: (sa S + (sb - sa) tr(S)/3 1) . e / sqrt(dt); z holds the three
    // diagonal normals and the three others times 1/sqrt(2), the entries of S.
    // Every operation on them is spelled out (no contraction left to the
    // compiler), so normals drawn here and normals read back from the cache
    // give the same force bits.
    if (P.noise) {
        if (zmode == 0) {
            pair_normals<R>(mir_gid(Di), mir_gid(Dj), P.step, P.key0, P.key1, z.z0, z.z1, z.z2, z.z3,
                            z.z4, z.z5);
            z.z3 = mul_rn(z.z3, is2);
            z.z4 = mul_rn(z.z4, is2);
            z.z5 = mul_rn(z.z5, is2);
        }
        const R rs = root_weight(P, om, Cj, Dj);
        const R sa = P.T1 * rs;
        ce = fma_rn(P.T3 * rs, add_rn(add_rn(z.z0, z.z1), z.z2), ce);
        ox = fma_rn(sa, fma_rn(z.z4, ez, fma_rn(z.z3, ey, mul_rn(z.z0, ex))), ox);
        oy = fma_rn(sa, fma_rn(z.z5, ez, fma_rn(z.z1, ey, mul_rn(z.z3, ex))), oy);
        oz = fma_rn(sa, fma_rn(z.z2, ez, fma_rn(z.z5, ey, mul_rn(z.z4, ex))), oz);
    }
}

template <class R>
__device__ __forceinline__ void write_fluid_force(const Bufs &b, const Inst &I, int gi, R fx, R fy,
                                                  R fz, R tx, R ty, R tz, R lev)
{
    double a[3];
    const double xg[3] = { b.x[3 * gi], b.x[3 * gi + 1], b.x[3 * gi + 2] };
    ext_accel(I, xg, a);
    const double m = b.m[gi];
    b.F[3 * gi] = (double)fx + m * a[0];
    b.F[3 * gi + 1] = (double)fy + m * a[1];
    b.F[3 * gi + 2] = (double)fz + m * a[2];
    b.T[3 * gi] = -(double)(lev * tx);
    b.T[3 * gi + 1] = -(double)(lev * ty);
    b.T[3 * gi + 2] = -(double)(lev * tz);
}

// F^DG_s / S_s of rigid slot j in precision R (Eq. F_fpi_DG_reac).
__device__ __forceinline__ void rxn_of(const Bufs &b, int j, float &x, float &y, float &z)
{
    const float4 r = b.rxn32[j];
    x = r.x; y = r.y; z = r.z;
}
__device__ __forceinline__ void rxn_of(const Bufs &b, int j, double &x, double &y, double &z)
{
    const double4_32a r = b.rxn[j];
    x = r.x; y = r.y; z = r.z;
}

// Fluid particle i and a rigid neighbour j (Section 2.4): Eqs. FijC and FijD
// on i (no rotational or random part) and the drag reaction Eq.
// F_fpi_DG_reac, added to i's sums; nothing beyond h.
template <class R, class TA, class T4>
__device__ __forceinline__ void fluid_rigid_pair(const Bufs &b, const Inst &I, const Geo<R> &geo,
                                                 const PairK<R> &P, int gi, const TA &Ai, const T4 &Bi,
                                                 const T4 &Ci, const T4 &Di, int j, const TA &Aj,
                                                 const T4 &Bj, const T4 &Cj, const T4 &Dj, R &fx, R &fy,
                                                 R &fz, R &tx, R &ty, R &tz)
{
    R rx, ry, rz, r2;
    if (!Rel<R>::get(b, I, geo, Ai, Aj, gi, j, rx, ry, rz, r2)) return;
    R ox, oy, oz, ce, ex, ey, ez, q, om;
    Z6<R> z;
    sdpd_pair<R>(P, rx, ry, rz, r2, Bi, Ci, Di, Bj, Cj, Dj, false, 0, z, ox, oy, oz, ce, ex, ey, ez, q, om);
    R rcx, rcy, rcz;
    rxn_of(b, j, rcx, rcy, rcz);
    const R W = P.Wc * (R(1) + R(3) * q) * om * om * om;
    fx += ox + ce * ex - rcx * W;
    fy += oy + ce * ey - rcy * W;
    fz += oz + ce * ez - rcz * W;
    tx += ey * oz - ez * oy;
    ty += ez * ox - ex * oz;
    tz += ex * oy - ey * ox;
}

// The same, called out of line where rigid neighbours are rare and the
// caller's registers matter (the gather), loading the records itself.
template <class R>
__device__ __noinline__ void fluid_rigid_pair_call(const Bufs &b, long long s, int gi, int j, R *f)
{
    using T4 = typename Vec<R>::T4;
    using TA = typename Mir<R>::TA;
    const Inst &I = b.inst[b.pinst[gi]];
    const Geo<R> geo(I);
    const TA *__restrict__ A = Mir<R>::A(b);
    const T4 *__restrict__ Bm = Mir<R>::B(b);
    const T4 *__restrict__ Cm = Mir<R>::C(b);
    const T4 *__restrict__ Dm = Mir<R>::D(b);
    const PairK<R> P(I, (uint32_t)(*b.step), Cm[s], Dm[s]);
    fluid_rigid_pair<R>(b, I, geo, P, gi, A[s], Bm[s], Cm[s], Dm[s], j, A[j], Bm[j], Cm[j], Dm[j], f[0], f[1],
                        f[2], f[3], f[4], f[5]);
}

// The draws of a pair out of line, where they are rare and the caller's
// registers matter (an entry beyond h in the first evaluation of a step and
// within it in the second).
template <class R>
__device__ __noinline__ void draw_rare(uint32_t gi, uint32_t gj, uint32_t step, uint32_t k0, uint32_t k1, R *z)
{
    pair_normals<R>(gi, gj, step, k0, k1, z[0], z[1], z[2], z[3], z[4], z[5]);
    for (int c = 3; c < 6; ++c) z[c] = mul_rn(z[c], R(0.70710678118654752440));
}

// The force and torque totals of a warp's particles, one per lane at the end.
template <class R> struct ForceSums {
    R f[6], keep[6];
    __device__ __forceinline__ ForceSums()
    {
#pragma unroll
        for (int c = 0; c < 6; ++c) f[c] = keep[c] = R(0);
    }
    // every accumulation step rounded explicitly
    __device__ __forceinline__ void add(R gx, R gy, R gz, R hx, R hy, R hz)
    {
        f[0] = add_rn(f[0], gx);
        f[1] = add_rn(f[1], gy);
        f[2] = add_rn(f[2], gz);
        f[3] = add_rn(f[3], hx);
        f[4] = add_rn(f[4], hy);
        f[5] = add_rn(f[5], hz);
    }
    __device__ __forceinline__ void close_group(int g)
    {
#pragma unroll
        for (int c = 0; c < 6; ++c) {
            keep_group(lanes_sum(f[c]), g, keep[c]);
            f[c] = R(0);
        }
    }
};

// The second evaluation of a step reads the normals of the first for the
// instances whose lists are still the same.
struct CacheUse {
    uint32_t step;
    bool fill, maybe, all;   // maybe: some instance's normals may be cached, all: every instance's are
    __device__ __forceinline__ CacheUse(const Bufs &b, int velver)
        : step((uint32_t)(*b.step)), fill(b.use_cache && velver == 1),
          maybe(b.use_cache && velver == 2 && *b.cache_step == *b.step),
          all(maybe && b.cache_epoch[0] == b.list_epoch[0])
    {
        // only the first evaluation writes, only the second one tests them
        if (fill && blockIdx.x == 0) {
            for (int k = threadIdx.x; k <= b.n_inst; k += blockDim.x) b.cache_epoch[k] = b.list_epoch[k];
            if (threadIdx.x == 0) *b.cache_step = *b.step;
        }
    }
    __device__ __forceinline__ bool reuse(const Bufs &b, int inst) const
    {
        return all || (maybe && b.cache_epoch[1 + inst] == b.list_epoch[1 + inst]);
    }
};

// The direct (owner-computes-all) force pass in FP64 over the neighbour list of
// fluid particle s (this lane's share of it).  The index two entries ahead and the
// records of the next neighbour are fetched before the current pair is
// evaluated.  With the cache on, the first evaluation of a step (FILL) stores
// the six normals of every entry in its own column (a NaN marker for an entry
// beyond h); the second (REUSE, when the list has not been rebuilt in
// between) reads them back instead of drawing them again (same counter, so
// the same bits).
template <class R> struct NormalRow {   // a row of 32 entries of the cache
    using T4 = typename Vec<R>::T4;
    using T2 = typename Vec2<R>::T2;
    T4 a[ROW];
    T2 b[ROW];
};

template <bool REUSE>
__device__ __forceinline__ void force_fluid_entries(const Bufs &b, long long s, const SlotHead &h, const ListHead &hd,
                                                    int sub, uint32_t step, bool fill, ForceSums<double> &sums)
{
    using R = double;
    using T4 = double4_32a;
    using TA = double4_32a;
    using T2 = double2;
    const int gi = h.gi;
    const Inst &I = b.inst[h.inst];
    const Geo<R> geo(I);
    const TA *__restrict__ A = Mir<R>::A(b);
    const T4 *__restrict__ Bm = Mir<R>::B(b);
    const T4 *__restrict__ Cm = Mir<R>::C(b);
    const T4 *__restrict__ Dm = Mir<R>::D(b);
    const int n = h.n, lane = threadIdx.x & 31;   // lane: also the entry's place in its row
    int k = sub;
    if (k >= n) return;
    const int *__restrict__ nb = b.nbr + entry_at(sub, s, b.rows);
    NormalRow<R> *__restrict__ zr = (NormalRow<R> *)b.zd + (size_t)(s / GROUP) * b.rows;
    const TA Ai = A[s];
    const T4 Bi = Bm[s], Ci = Cm[s], Di = Dm[s];
    const PairK<R> P(I, step, Ci, Di);
    fill = fill && P.noise;
    int jn = hd.e0, jnn = hd.e1;
    TA An = A[jn];
    T4 Bn = Bm[jn], Cn = Cm[jn], Dn = Dm[jn];
    T4 zan;
    T2 zbn;
    if (REUSE && P.noise) { zan = ld_stream(zr->a + lane); zbn = ld_stream(zr->b + lane); }
    for (; k < n; k += LPP, nb += ROW, ++zr) {
        const int j = jn;
        const TA Aj = An;
        const T4 Bj = Bn, Cj = Cn, Dj = Dn;
        T4 za;
        T2 zb;
        if (REUSE) { za = zan; zb = zbn; }
        if (k + LPP < n) {
            jn = jnn;
            An = A[jn]; Bn = Bm[jn]; Cn = Cm[jn]; Dn = Dm[jn];
            if (REUSE && P.noise) {
                zan = ld_stream(zr[1].a + lane);
                zbn = ld_stream(zr[1].b + lane);
            }
            if (k + 2 * LPP < n) jnn = ld_stream(nb + 2 * ROW);
        }
        const bool rig = mir_type(Aj) == T_RIGID;
        R rx, ry, rz, r2;
        if (!Rel<R>::get(b, I, geo, Ai, Aj, gi, j, rx, ry, rz, r2)) {
            if (!REUSE && fill && !rig) {
                T4 nm;
                nm.x = R(NAN); nm.y = R(0); nm.z = R(0); nm.w = R(0);
                st_stream(zr->a + lane, nm);
            }
            continue;
        }
        R ox, oy, oz, ce, ex, ey, ez, q, om;
        Z6<R> z;
        int zmode = 0;
        // an entry beyond h in the first evaluation carries the NaN marker
        if (REUSE && P.noise && !rig && !is_nan(za.x)) {
            z.z0 = za.x; z.z1 = za.y; z.z2 = za.z; z.z3 = za.w; z.z4 = zb.x; z.z5 = zb.y;
            zmode = 1;
        }
        sdpd_pair<R>(P, rx, ry, rz, r2, Bi, Ci, Di, Bj, Cj, Dj, !rig, zmode, z, ox, oy, oz, ce, ex, ey, ez,
                     q, om);
        if (!REUSE && fill && !rig) {
            T4 zw;
            zw.x = z.z0; zw.y = z.z1; zw.z = z.z2; zw.w = z.z3;
            T2 zv;
            zv.x = z.z4; zv.y = z.z5;
            st_stream(zr->a + lane, zw);
            st_stream(zr->b + lane, zv);
        }
        R gx, gy, gz, hx, hy, hz;
        pair_fh(ox, oy, oz, ce, ex, ey, ez, gx, gy, gz, hx, hy, hz);
        if (rig) {
            // Eq. F_fpi_DG_reac: -F^DG_s W_sj / S_s
            R rcx, rcy, rcz;
            rxn_of(b, j, rcx, rcy, rcz);
            const R W = drag_weight(P, q, om);
            sums.f[0] = sub_rn(sums.f[0], mul_rn(rcx, W));
            sums.f[1] = sub_rn(sums.f[1], mul_rn(rcy, W));
            sums.f[2] = sub_rn(sums.f[2], mul_rn(rcz, W));
        }
        sums.add(gx, gy, gz, hx, hy, hz);
    }
}

__global__ void __launch_bounds__(256) k_force_fluid(Bufs b, int velver, int groups)
{
    using R = double;
    const CacheUse u(b, velver);
    const int lane = threadIdx.x & 31, sub = lane % LPP;
    const long long base = pass_base(groups);
    SlotHead mine(b, base + lane, lane < groups * GROUP);
    if (mine.type != T_FLUID) mine.n = -1;
    ForceSums<R> sums;
    for (int g = 0; g < groups; ++g) {
        const long long s = base + g * GROUP + lane / LPP;
        const SlotHead h = mine.of_group(g);
        const ListHead hd(b.nbr, s, b.rows, 0, h.n, sub);
        if (u.reuse(b, h.inst)) force_fluid_entries<true>(b, s, h, hd, sub, u.step, false, sums);
        else force_fluid_entries<false>(b, s, h, hd, sub, u.step, u.fill, sums);
        sums.close_group(g);
    }
    if (mine.n < 0) return;
    write_fluid_force<R>(b, b.inst[mine.inst], mine.gi, sums.keep[0], sums.keep[1], sums.keep[2], sums.keep[3],
                         sums.keep[4], sums.keep[5], K<R>::lever(b.inst[mine.inst]));
}

// ------------------------------------------------- direct force pass, FP32
// One listed pair (i, j) of the FP32 direct pass, added to i's sums where `ok`
// (within h).  Every lane runs the same straight line: an entry past the end
// or beyond h is left out of the sums at the end, and a sphere partner
// (`rig`: Eqs. FijC and FijD only) has zero rotational and random
// coefficients.  Branches for them cost the pass about a quarter of its
// instructions (divergence barriers and register moves), though some lane
// takes the long way almost always.
__device__ __forceinline__ void pair32(const Bufs &b, const PairK<float> &P, bool ok, bool rig, int j, float rx,
                                       float ry, float rz, float r2, const float4 &Bi, const float4 &Ci,
                                       const float4 &Bj, const float4 &Cj, const Z6<float> &z, float (&f)[6])
{
    float r, ir;
    root_and_inverse(r2, r, ir);
    const float q = r * P.irc, om = one_minus(q);
    const float om2 = om * om, g = om2 * Cj.w;
    const float ex = rx * ir, ey = ry * ir, ez = rz * ir;
    const float vx = Bi.x - Bj.x, vy = Bi.y - Bj.y, vz = Bi.z - Bj.z;
    const float ev = ex * vx + ey * vy + ez * vz;
    const float c1 = P.A1 * g, c3 = (rig ? 0.f : P.A3) * g;
    float ce = P.PC * (Bi.w + Bj.w) * (om2 * r) - P.A2 * g * ev;
    const float wx = Ci.x + Cj.x, wy = Ci.y + Cj.y, wz = Ci.z + Cj.z;
    float ox = c1 * vx + c3 * (ry * wz - rz * wy);
    float oy = c1 * vy + c3 * (rz * wx - rx * wz);
    float oz = c1 * vz + c3 * (rx * wy - ry * wx);
    const float rs = rig ? 0.f : root_weight(P, om, Cj, Cj);
    const float sa = P.T1 * rs, st = P.T3 * rs;
    // (explicit roundings from here on: normals drawn and normals read back
    // give the same bits)
    ce = fma_rn(st, add_rn(add_rn(z.z0, z.z1), z.z2), ce);
    ox = fma_rn(sa, fma_rn(z.z4, ez, fma_rn(z.z3, ey, mul_rn(z.z0, ex))), ox);
    oy = fma_rn(sa, fma_rn(z.z5, ez, fma_rn(z.z1, ey, mul_rn(z.z3, ex))), oy);
    oz = fma_rn(sa, fma_rn(z.z2, ez, fma_rn(z.z5, ey, mul_rn(z.z4, ex))), oz);
    float gx, gy, gz, hx, hy, hz;
    pair_fh(ox, oy, oz, ce, ex, ey, ez, gx, gy, gz, hx, hy, hz);
    if (ok && rig) {
        // Eq. F_fpi_DG_reac: -F^DG_s W_sj / S_s
        const float4 rc = b.rxn32[j];
        const float W = drag_weight(P, q, om);
        f[0] = sub_rn(f[0], mul_rn(rc.x, W));
        f[1] = sub_rn(f[1], mul_rn(rc.y, W));
        f[2] = sub_rn(f[2], mul_rn(rc.z, W));
    }
    if (ok) {
        f[0] = add_rn(f[0], gx);
        f[1] = add_rn(f[1], gy);
        f[2] = add_rn(f[2], gz);
        f[3] = add_rn(f[3], hx);
        f[4] = add_rn(f[4], hy);
        f[5] = add_rn(f[5], hz);
    }
}

// A warp's particles and their totals, in shared memory: registers are what
// these two kernels are short of.
struct WarpSlots {
    int gi[32], inst[32], n[32];   // n < 0: not a particle of this launch
    float f[32][6];
    // every lane puts its own slot's in
    __device__ __forceinline__ void set(const SlotHead &h)
    {
        const int lane = threadIdx.x & 31;
        gi[lane] = h.gi;
        inst[lane] = h.inst;
        n[lane] = h.n;
        __syncwarp();
    }
    // the totals of group g's particles: the lanes of a particle all end with them
    __device__ __forceinline__ void put(int g, float (&v)[6])
    {
#pragma unroll
        for (int c = 0; c < 6; ++c) v[c] = lanes_sum(v[c]);
        const int lane = threadIdx.x & 31;
        if (lane % LPP == 0)
#pragma unroll
            for (int c = 0; c < 6; ++c) f[g * GROUP + lane / LPP][c] = v[c];
    }
    // and written out, each by a lane of its own
    __device__ __forceinline__ void write(const Bufs &b)
    {
        __syncwarp();
        const int lane = threadIdx.x & 31;
        if (n[lane] < 0) return;
        const Inst &I = b.inst[inst[lane]];
        write_fluid_force<float>(b, I, gi[lane], f[lane][0], f[lane][1], f[lane][2], f[lane][3], f[lane][4], f[lane][5],
                                 K<float>::lever(I));
    }
};

// What a lane holds of its particle.
struct Own32 {
    Geo<float> geo;
    PairK<float> P;
    int4 A;
    float4 B, C;
    __device__ __forceinline__ Own32(const Bufs &b, int inst, uint32_t step, long long s)
        : Own32(b.inst[inst], step, b.A32[s], b.B32[s], b.C32[s])
    {}
    __device__ __forceinline__ Own32(const Inst &I, uint32_t step, const int4 &a, const float4 &bb, const float4 &c)
        : geo(I), P(I, step, c, c), A(a), B(bb), C(c)   // (FP32 keeps nothing of the pair constants in D)
    {}
};

// The displacement of a listed pair and whether it lies within h.
__device__ __forceinline__ bool near32(const Bufs &b, const Own32 &o, const WarpSlots &w, int slot, bool live, int j,
                                       const int4 &Aj, float &rx, float &ry, float &rz, float &r2)
{
    o.geo.disp(o.A, Aj, rx, ry, rz);
    r2 = rx * rx + ry * ry + rz * rz;
    bool ok = live && r2 < o.geo.ghi;
    if (ok && r2 >= o.geo.glo) ok = within_exactly(b, w.inst[slot], w.gi[slot], j);
    return ok;
}

// The drawing pass: the particles whose normals are not cached.  With the
// cache on, the first evaluation of a step (fill) stores the normals of every
// entry in its row, a NaN marker for an entry beyond h (those of a sphere
// partner are stored too and enter with a zero coefficient).  Two rows are
// drawn together for the packed Box-Muller.
__global__ void __launch_bounds__(256, 2) k_force_draw(Bufs b, int velver, int groups)
{
    __shared__ WarpSlots tables[8];
    const CacheUse u(b, velver);
    if (u.all) return;   // uniform over the launch
    WarpSlots &tab = tables[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31, sub = lane % LPP;
    const unsigned FULL = 0xffffffffu;
    const long long base = pass_base(groups);
    {
        SlotHead mine(b, base + lane, lane < groups * GROUP);
        if (mine.type != T_FLUID || u.reuse(b, mine.inst)) mine.n = -1;
        tab.set(mine);
    }
    for (int g = 0; g < groups; ++g) {
        float f[6] = { 0.f, 0.f, 0.f, 0.f, 0.f, 0.f };
        const int slot = g * GROUP + lane / LPP, n = tab.n[slot];
        if (g + 1 < groups) prefetch_lists(b, base + (g + 1) * GROUP, tab.n[slot + GROUP]);
        const int gr = entry_rows(__reduce_max_sync(FULL, max(n, 0)));
        if (gr > 0) {
            const long long s = n > 0 ? base + slot : 0;   // an idle lane reads slot 0 and adds nothing
            const Own32 o(b, tab.inst[slot], u.step, s);
            const uint32_t gid = mir_gid(b.D32[s]);
            const bool fill = u.fill && o.P.noise, draw = __any_sync(FULL, o.P.noise);
            const int *__restrict__ nb = b.nbr + entry_at(sub, s, b.rows);
            NormalRow<float> *__restrict__ zr = (NormalRow<float> *)b.zd + (size_t)(s / GROUP) * b.rows;
            int left = n - sub;   // this lane has an entry in row i of the present ones when i LPP < left
            ListRows cur, next;
            cur.load(nb, left);
            // positions and gids of the next two rows fetched ahead: the
            // draws start from them, the other records come meanwhile
            int4 A[2];
            uint32_t gj[2];
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                A[t] = b.A32[cur.e[t]];
                gj[t] = mir_gid(b.D32[cur.e[t]]);
            }
            for (int r0 = 0; r0 < gr; r0 += ZR) {
                nb += ZR * ROW;
                next.load(nb, left - ZR * LPP);
#pragma unroll
                for (int i = 0; i < ZR; i += 2) {
                    if (i && r0 + i >= gr) break;   // uniform
                    float rx[2], ry[2], rz[2], r2[2];
                    bool ok[2], live[2], rig[2];
                    float4 Bj[2], Cj[2];
                    uint32_t g2[2];
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        const int j = cur.e[i + t];
                        Bj[t] = b.B32[j];
                        Cj[t] = b.C32[j];
                        live[t] = (i + t) * LPP < left;
                        rig[t] = A[t].w == T_RIGID;
                        ok[t] = near32(b, o, tab, slot, live[t], j, A[t], rx[t], ry[t], rz[t], r2[t]);
                        g2[t] = gj[t];
                    }
#pragma unroll
                    for (int t = 0; t < 2; ++t) {
                        const int jn = i + 2 < ZR ? cur.e[(i + 2 + t) % ZR] : next.e[t];
                        A[t] = b.A32[jn];
                        gj[t] = mir_gid(b.D32[jn]);
                    }
                    float z[2][6] = { { 0.f, 0.f, 0.f, 0.f, 0.f, 0.f }, { 0.f, 0.f, 0.f, 0.f, 0.f, 0.f } };
                    if (draw) {
                        const float is2 = 0.70710678118654752440f;
                        pair_normals2(gid, g2[0], g2[1], o.P.step, o.P.key0, o.P.key1, z[0], z[1]);
#pragma unroll
                        for (int t = 0; t < 2; ++t) {
                            for (int c = 3; c < 6; ++c) z[t][c] = mul_rn(z[t][c], is2);
                            if (fill && live[t]) {
                                st_stream(zr[i + t].a + lane, make_float4(ok[t] ? z[t][0] : NAN, z[t][1], z[t][2], z[t][3]));
                                st_stream(zr[i + t].b + lane, make_float2(z[t][4], z[t][5]));
                            }
                        }
                    }
#pragma unroll
                    for (int t = 0; t < 2; ++t)
                        pair32(b, o.P, ok[t], rig[t], cur.e[i + t], rx[t], ry[t], rz[t], r2[t], o.B, o.C, Bj[t], Cj[t],
                               Z6<float>{ z[t][0], z[t][1], z[t][2], z[t][3], z[t][4], z[t][5] }, f);
                }
                cur = next;
                left -= ZR * LPP;
                zr += ZR;
            }
        }
        tab.put(g, f);
    }
    tab.write(b);
}

// The second evaluation of FP32 pairs, normals from the cache.  24 bytes of
// normals an entry are most of what the pass reads from HBM, and register
// loads one row ahead left 1.9 MB in flight on the chip where 6.8 TB/s at a
// microsecond want 7 MB: the pass ran at 2.2 TB/s and took 1.38 times what it
// takes without them.  The rows of a block are contiguous, so each warp has
// them copied into a ring in shared memory by the copy engine (PTX
// cp.async.bulk on an mbarrier), ZR rows at a time and ZS chunks ahead, across
// the groups it works through, at no registers or load instructions.
constexpr int ZS = 2, ZTHREADS = 128;
struct NormalRing {
    NormalRow<float> z[ZS][ZR];
    uint64_t bar[ZS];
    uint64_t pad[16 - ZS];   // rings start on 128 bytes
    int zrows[8];            // rows of normals of each group
    WarpSlots tab;
    int fill[24];
};
static_assert(sizeof(NormalRow<float>) == 768 && sizeof(NormalRing) % 128 == 0, "bulk copies are 16-byte aligned");
// tries of a wait: for the chunk that is next, and for what is still on its
// way when one of those gave up (a test builds the pass with no tries)
#ifndef RING_TRIES
#define RING_TRIES (1 << 22)
#endif
constexpr int RING_DRAIN_TRIES = 1 << 22;

__device__ __forceinline__ unsigned smem_addr(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

// Waits (at most `tries` times) for the phase of parity `par`; false when it gave up.
__device__ __forceinline__ bool ring_wait(uint64_t *bar, unsigned par, int tries)
{
    const unsigned a = smem_addr(bar);
    for (int it = 0; it < tries; ++it) {
        unsigned done;
        asm volatile("{\n\t.reg .pred P;\n\tmbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, P;\n\t}"
                     : "=r"(done)
                     : "r"(a), "r"(par)
                     : "memory");
        if (done) return true;
    }
    return false;
}

__global__ void __launch_bounds__(ZTHREADS, 4) k_force_cached(Bufs b, int groups)
{
    __shared__ __align__(128) NormalRing rings[ZTHREADS / 32];
    const CacheUse u(b, 2);
    if (!u.maybe) return;   // uniform over the launch
    NormalRing &ring = rings[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31, sub = lane % LPP;
    const unsigned FULL = 0xffffffffu;
    if (lane == 0) {
        for (int i = 0; i < ZS; ++i)
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(ring.bar + i)) : "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    const long long base = pass_base(groups);
    WarpSlots &tab = ring.tab;
    {
        SlotHead mine(b, base + lane, lane < groups * GROUP);
        if (mine.type != T_FLUID || !u.reuse(b, mine.inst)) mine.n = -1;
        tab.set(mine);
        // rows of each group's lists whose normals are wanted (some particle's
        // instance has noise)
        int rows = max(mine.n, 0), noisy = mine.n > 0 && b.inst[mine.inst].noise;
#pragma unroll
        for (int o = 1; o < GROUP; o <<= 1) {
            rows = max(rows, __shfl_xor_sync(FULL, rows, o));
            noisy |= __shfl_xor_sync(FULL, noisy, o);
        }
        if (lane % GROUP == 0) ring.zrows[lane / GROUP] = noisy ? entry_rows(rows) : 0;
        __syncwarp();
    }
    // the copies, chunk by chunk through the groups
    int pg = 0, pr = 0;   // next row to ask for: of group pg
    unsigned asked = 0;   // chunks asked for
    auto request = [&](int st) {
        while (pg < groups && pr >= ring.zrows[pg]) {
            ++pg;
            pr = 0;
        }
        if (pg >= groups) return;
        const int have = ring.zrows[pg];
        const unsigned bytes = (unsigned)min(ZR, have - pr) * (unsigned)sizeof(NormalRow<float>);
        if (lane == 0) {
            const void *src = (const NormalRow<float> *)b.zd + (size_t)(base / GROUP + pg) * b.rows + pr;
            const unsigned bar = smem_addr(ring.bar + st);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
            asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                             smem_addr(ring.z[st])),
                         "l"(src), "r"(bytes), "r"(bar)
                         : "memory");
        }
        pr += ZR;
        ++asked;
    };
    unsigned chunk = 0;   // chunks consumed: in stage chunk % ZS, its phase chunk / ZS
    for (int i = 0; i < ZS; ++i) request(i);
    for (int g = 0; g < groups; ++g) {
        float f[6] = { 0.f, 0.f, 0.f, 0.f, 0.f, 0.f };
        const int slot = g * GROUP + lane / LPP, n = tab.n[slot];
        if (g + 1 < groups) prefetch_lists(b, base + (g + 1) * GROUP, tab.n[slot + GROUP]);
        const int gr = entry_rows(__reduce_max_sync(FULL, max(n, 0)));
        const bool normals = ring.zrows[g] > 0;
        if (gr > 0) {
            const long long s = n > 0 ? base + slot : 0;   // an idle lane reads slot 0 and adds nothing
            const Own32 o(b, tab.inst[slot], u.step, s);
            const int *__restrict__ nb = b.nbr + entry_at(sub, s, b.rows);
            int left = n - sub;   // this lane has an entry in row i of the present ones when i LPP < left
            ListRows cur, next;
            cur.load(nb, left);
            // the records of the next row are fetched ahead
            int4 A = b.A32[cur.e[0]];
            float4 B = b.B32[cur.e[0]], C = b.C32[cur.e[0]];
            for (int r0 = 0; r0 < gr; r0 += ZR) {
                nb += ZR * ROW;
                next.load(nb, left - ZR * LPP);
                const int st = chunk % ZS;
                if (normals && !__all_sync(FULL, ring_wait(ring.bar + st, (chunk / ZS) & 1u, RING_TRIES))) {
                    // the warp leaves: no barrier is armed again within its
                    // phase, and every copy still on its way gets one more
                    // bounded wait before its buffer is left
                    if (lane == 0) atomicOr(b.err, ERR_TIMEOUT);
                    for (unsigned c = chunk; c < asked; ++c) (void)ring_wait(ring.bar + c % ZS, (c / ZS) & 1u, RING_DRAIN_TRIES);
                    return;
                }
                const NormalRow<float> *zrow = ring.z[st];
#pragma unroll
                for (int i = 0; i < ZR; ++i) {
                    if (i && r0 + i >= gr) break;   // uniform
                    const int j = cur.e[i], jn = i + 1 < ZR ? cur.e[(i + 1) % ZR] : next.e[0];
                    const int4 Aj = A;
                    const float4 Bj = B, Cj = C;
                    A = b.A32[jn];
                    B = b.B32[jn];
                    C = b.C32[jn];
                    float rx, ry, rz, r2;
                    const bool ok = near32(b, o, tab, slot, i * LPP < left, j, Aj, rx, ry, rz, r2);
                    Z6<float> z{ 0.f, 0.f, 0.f, 0.f, 0.f, 0.f };
                    if (normals) {
                        const float4 za = zrow[i].a[lane];
                        const float2 zb = zrow[i].b[lane];
                        z = Z6<float>{ za.x, za.y, za.z, za.w, zb.x, zb.y };
                        // an instance without noise has no normals, and an entry
                        // that was beyond h in the first evaluation none yet
                        if (ok && (!o.P.noise || is_nan(za.x))) {
                            float t[6] = { 0.f, 0.f, 0.f, 0.f, 0.f, 0.f };
                            if (o.P.noise)
                                draw_rare<float>(mir_gid(b.D32[s]), mir_gid(b.D32[j]), o.P.step, o.P.key0, o.P.key1, t);
                            z = Z6<float>{ t[0], t[1], t[2], t[3], t[4], t[5] };
                        }
                    }
                    pair32(b, o.P, ok, Aj.w == T_RIGID, j, rx, ry, rz, r2, o.B, o.C, Bj, Cj, z, f);
                }
                if (normals) {
                    __syncwarp();   // every lane has read the chunk
                    request(st);
                    ++chunk;
                }
                cur = next;
                left -= ZR * LPP;
            }
        }
        tab.put(g, f);
    }
    tab.write(b);
}

// Newton-3 force pass, phase 1: every fluid or wall particle evaluates the
// pairs of its owned prefix (see k_neighbors; within h, both non-rigid, at
// least one fluid) once, stores (f, e x o) in the partner's column of the
// pair buffer (at the row of the partner's entry for the pair, from k_rev)
// and keeps its own sum.  Each unordered pair is
// computed once instead of twice.  The first evaluation of a step stores the
// six normals of each pair; the second reads them back, fetched one entry
// ahead like the records, when the list has not been rebuilt in between (same
// counter, so the same bits).
// PUSH: the owner writes the finished pair result {f, e x o} into the
// partner's column (FP64, and FP32 in force mode 4); otherwise (FP32, mode 1)
// it keeps {o, ce} in its own column and the partner rebuilds f and e x o.
// Both hand the partner the same bits.
template <class R, bool REUSE, bool PUSH>
__device__ __forceinline__ void force_half_entries(const Bufs &b, long long s, const SlotHead &h, int sub,
                                                   uint32_t step, bool fill, ForceSums<R> &sums)
{
    using T4 = typename Vec<R>::T4;
    using TA = typename Mir<R>::TA;
    using T2 = typename Vec2<R>::T2;
    const int ti = h.type, gi = h.gi;
    const Inst &I = b.inst[h.inst];
    const Geo<R> geo(I);
    const TA *__restrict__ A = Mir<R>::A(b);
    const T4 *__restrict__ Bm = Mir<R>::B(b);
    const T4 *__restrict__ Cm = Mir<R>::C(b);
    const T4 *__restrict__ Dm = Mir<R>::D(b);
    T4 *__restrict__ resA = (T4 *)b.resA;
    T2 *__restrict__ resB = (T2 *)b.resB;
    const int last = h.nf;  // the owned prefix of the list
    int k = sub;
    if (k >= last) return;
    const size_t first = entry_at(sub, s, b.rows);
    size_t at = entry_at(sub, s, b.rows_own);   // own column: normals cache, split results
    T4 *__restrict__ zA = (T4 *)b.zA + at;
    T2 *__restrict__ zB = (T2 *)b.zB + at;
    const int *__restrict__ nb = b.nbr + first;
    const uint16_t *__restrict__ rv = b.rev + first;
    const TA Ai = A[s];
    const T4 Bi = Bm[s], Ci = Cm[s], Di = Dm[s];
    const PairK<R> P(I, step, Ci, Di);
    const bool fi = (ti == T_FLUID);
    const bool noise = P.noise;
    int jn = __ldg(nb);
    int jnn = k + LPP < last ? __ldg(nb + ROW) : 0;
    TA An = A[jn];
    T4 Bn = Bm[jn], Cn = Cm[jn], Dn = Dm[jn];
    T4 zan;
    T2 zbn;
    if (REUSE && noise) { zan = *zA; zbn = *zB; }
    for (; k < last; k += LPP, nb += ROW, rv += ROW, zA += ROW, zB += ROW, at += ROW) {
        const int j = jn;
        const TA Aj = An;
        const T4 Bj = Bn, Cj = Cn, Dj = Dn;
        T4 za;
        T2 zb;
        if (REUSE) { za = zan; zb = zbn; }
        if (k + LPP < last) {
            jn = jnn;
            An = A[jn]; Bn = Bm[jn]; Cn = Cm[jn]; Dn = Dm[jn];
            if (REUSE && noise) {
                zan = zA[ROW];
                zbn = zB[ROW];
            }
            if (k + 2 * LPP < last) jnn = __ldg(nb + 2 * ROW);
        }
        const int tj = mir_type(Aj);
        if (tj == T_RIGID) {
            if (fi) fluid_rigid_pair<R>(b, I, geo, P, gi, Ai, Bi, Ci, Di, j, Aj, Bj, Cj, Dj, sums.f[0], sums.f[1],
                                        sums.f[2], sums.f[3], sums.f[4], sums.f[5]);
            continue;
        }
        if (!fi && tj != T_FLUID) continue;
        // FP64 results go to the partner's column, at the row of its entry
        // for this pair (from k_rev); split results stay in the own column
        size_t pt = at;
        bool put = true;
        if constexpr (PUSH) {
            const int prow = __ldg(rv);
            put = prow < b.capown;   // false only after a list error (flagged)
            pt = entry_at(prow, j, b.rows_own);
        }
        R rx, ry, rz, r2;
        if (!Rel<R>::get(b, I, geo, Ai, Aj, gi, j, rx, ry, rz, r2)) {
            // beyond h: marked for the partner's gather and the normals cache
            T4 nm;
            nm.x = R(NAN); nm.y = R(0); nm.z = R(0); nm.w = R(0);
            if (put) resA[pt] = nm;
            if (!REUSE && fill) *zA = nm;
            continue;
        }
        Z6<R> z;
        int zmode = 0;
        // an entry beyond h in the first evaluation carries the NaN marker
        if (REUSE && noise && !is_nan(za.x)) {
            z.z0 = za.x; z.z1 = za.y; z.z2 = za.z; z.z3 = za.w; z.z4 = zb.x; z.z5 = zb.y;
            zmode = 1;
        }
        R ox, oy, oz, ce, ex, ey, ez, q, om;
        sdpd_pair<R>(P, rx, ry, rz, r2, Bi, Ci, Di, Bj, Cj, Dj, true, zmode, z, ox, oy, oz, ce, ex, ey,
                     ez, q, om);
        if (!REUSE && fill && noise) {
            T4 zw;
            zw.x = z.z0; zw.y = z.z1; zw.z = z.z2; zw.w = z.z3;
            T2 zv;
            zv.x = z.z4; zv.y = z.z5;
            *zA = zw;
            *zB = zv;
        }
        R gx, gy, gz, hx, hy, hz;
        pair_fh(ox, oy, oz, ce, ex, ey, ez, gx, gy, gz, hx, hy, hz);
        T4 ra;
        if constexpr (!PUSH) {
            // {o, ce} (16 B); the partner rebuilds f and e x o
            ra.x = ox; ra.y = oy; ra.z = oz; ra.w = ce;
        } else {
            ra.x = gx; ra.y = gy; ra.z = gz; ra.w = hx;
            T2 rb;
            rb.x = hy; rb.y = hz;
            if (put) resB[pt] = rb;
        }
        if (put) resA[pt] = ra;
        sums.add(gx, gy, gz, hx, hy, hz);
    }
}

// (FP32: at most 128 registers, so four 128-thread blocks fit on an SM)
template <class R, bool PUSH>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 2 : 1) k_force_half(Bufs b, int velver, int groups)
{
    using T4 = typename Vec<R>::T4;
    using TA = typename Mir<R>::TA;
    using T2 = typename Vec2<R>::T2;
    const CacheUse u(b, velver);
    const int lane = threadIdx.x & 31;
    const long long base = pass_base(groups);
    const SlotHead mine(b, base + lane, lane < groups * GROUP);
    ForceSums<R> sums;
    for (int g = 0; g < groups; ++g) {
        const long long s = base + g * GROUP + lane / LPP;
        const SlotHead h = mine.of_group(g);
        if (h.n >= 0 && h.type != T_RIGID) {
            if (u.reuse(b, h.inst)) force_half_entries<R, true, PUSH>(b, s, h, lane % LPP, u.step, false, sums);
            else force_half_entries<R, false, PUSH>(b, s, h, lane % LPP, u.step, u.fill, sums);
        }
        sums.close_group(g);
    }
    const long long s = base + lane;
    if (mine.n < 0 || mine.type != T_FLUID) return;
    T4 oa;
    oa.x = sums.keep[0]; oa.y = sums.keep[1]; oa.z = sums.keep[2]; oa.w = sums.keep[3];
    T2 ob;
    ob.x = sums.keep[4]; ob.y = sums.keep[5];
    ((T4 *)b.ownA)[s] = oa;
    ((T2 *)b.ownB)[s] = ob;
}

// Newton-3 force pass, phase 2 (fluid particles): own sum + the results of
// the pairs its partners own (force negated, e x o equal; pairs the owner
// found beyond h carry a NaN marker) + the pairs with rigid neighbours among
// the non-owned entries, evaluated here (Eqs. FijC, FijD and the drag
// reaction Eq. F_fpi_DG_reac) + external force.  FP64 results were written
// into this particle's column (read coalesced); split results are read from
// the owner's column through the reverse index.
template <class R, bool PUSH>
__device__ __forceinline__ void gather_entries(const Bufs &b, long long s, const SlotHead &h, int sub,
                                               ForceSums<R> &sums)
{
    using T4 = typename Vec<R>::T4;
    using TA = typename Mir<R>::TA;
    using T2 = typename Vec2<R>::T2;
    const int gi = h.gi;
    const Inst &I = b.inst[h.inst];
    const Geo<R> geo(I);
    const TA *__restrict__ A = Mir<R>::A(b);
    const T4 *__restrict__ resA = (const T4 *)b.resA;
    const T2 *__restrict__ resB = (const T2 *)b.resB;
    const TA Ai = A[s];
    const int first = h.nf;
    const bool any_rigid = b.nbflag[s] & 1;
    // more non-owned entries than capown only after a list error (flagged)
    const int m = min(h.n - first, b.capown);
    constexpr int G = PUSH ? 4 : 2;
    for (int k0 = sub; k0 < m; k0 += G * LPP) {
        size_t at[G];
        int pj[G];
        bool use[G], rig[G];
        TA Ap[G];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int k = k0 + g * LPP;
            use[g] = k < m;
            rig[g] = false;
            pj[g] = 0;
            at[g] = entry_at(k, s, b.rows_own);
            if (use[g] && (!PUSH || any_rigid)) {
                const size_t en = entry_at(first + k, s, b.rows);
                const int i = __ldg(b.nbr + en);
                pj[g] = i;
                Ap[g] = A[i];
                rig[g] = mir_type(Ap[g]) == T_RIGID;
                if constexpr (!PUSH) at[g] = entry_at(__ldg(b.rev + en), i, b.rows_own);
            }
        }
        T4 ra[G];
        T2 rb[G];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            if (use[g] && !rig[g]) {
                ra[g] = resA[at[g]];
                if constexpr (PUSH) rb[g] = resB[at[g]];
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            if (!use[g]) continue;
            if (rig[g]) {
                R f[6];   // a copy: the sums themselves stay in registers
#pragma unroll
                for (int c = 0; c < 6; ++c) f[c] = sums.f[c];
                fluid_rigid_pair_call<R>(b, s, gi, pj[g], f);
#pragma unroll
                for (int c = 0; c < 6; ++c) sums.f[c] = f[c];
                continue;
            }
            // NaN marks a pair beyond h (written by the owner)
            if (is_nan(ra[g].x)) continue;
            if constexpr (PUSH) {
                sums.add(-ra[g].x, -ra[g].y, -ra[g].z, ra[g].w, rb[g].x, rb[g].y);
            } else {
                // e of the owner = -(e seen from here), bitwise
                R rx, ry, rz;
                geo.disp(Ai, Ap[g], rx, ry, rz);
                R rr, ir;
                root_and_inverse(rx * rx + ry * ry + rz * rz, rr, ir);
                R gx, gy, gz, hx, hy, hz;
                pair_fh(ra[g].x, ra[g].y, ra[g].z, ra[g].w, -(rx * ir), -(ry * ir), -(rz * ir), gx, gy, gz,
                        hx, hy, hz);
                sums.add(-gx, -gy, -gz, hx, hy, hz);
            }
        }
    }
}

template <class R, bool PUSH>
__global__ void __launch_bounds__(256) k_force_gather(Bufs b, int groups)
{
    using T4 = typename Vec<R>::T4;
    using TA = typename Mir<R>::TA;
    using T2 = typename Vec2<R>::T2;
    const int lane = threadIdx.x & 31;
    const long long base = pass_base(groups);
    const SlotHead mine(b, base + lane, lane < groups * GROUP);
    ForceSums<R> sums;
    for (int g = 0; g < groups; ++g) {
        const long long s = base + g * GROUP + lane / LPP;
        const SlotHead h = mine.of_group(g);
        if (h.n >= 0 && h.type == T_FLUID) gather_entries<R, PUSH>(b, s, h, lane % LPP, sums);
        sums.close_group(g);
    }
    const long long s = base + lane;
    if (mine.n < 0 || mine.type != T_FLUID) return;
    const int gi = mine.gi;
    const Inst &I = b.inst[mine.inst];
    const T4 oa = ((const T4 *)b.ownA)[s];
    const T2 ob = ((const T2 *)b.ownB)[s];
    write_fluid_force<R>(b, I, gi, oa.x + sums.keep[0], oa.y + sums.keep[1], oa.z + sums.keep[2],
                         oa.w + sums.keep[3], ob.x + sums.keep[4], ob.y + sums.keep[5], K<R>::lever(I));
}

// -------------------------------------------------------- rigid force pass
__device__ __forceinline__ void cross3(const double a[3], const double c[3], double o[3])
{
    o[0] = a[1] * c[2] - a[2] * c[1];
    o[1] = a[2] * c[0] - a[0] * c[2];
    o[2] = a[0] * c[1] - a[1] * c[0];
}

__device__ __forceinline__ void dem_coeffs(const Inst &I, double Ri, double Rj, double mi, double mj,
                                           double &kn, double &kt, double &cn, double &ct)
{
    const double ms = (mj > 0.0) ? mi * mj / (mi + mj) : mi;
    if (I.dem_law == 0) {
        const double D = (1.0 - I.nu_p * I.nu_p) / (I.E_p * PI);
        const double Re = (Rj > 0.0) ? Ri * Rj / (Ri + Rj) : Ri;
        kn = 4.0 / (3.0 * PI) * (1.0 / (D + D)) * sqrt(Re);
        kt = kn * I.kt_ratio;
        cn = 2.0 * sqrt(2.0 * ms * kn);
        ct = 2.0 * sqrt(2.0 * ms * kt);
    } else {
        kn = I.kn;
        kt = kn * I.kt_ratio;
        cn = 2.0 * I.zeta * sqrt(ms * kn);
        ct = 2.0 * I.zeta * sqrt(ms * kt);
    }
}

// One DEM contact on rigid particle i (n from the partner to i, overlap < 0):
// normal spring-dashpot, tangential spring-dashpot on the stored displacement
// with the Coulomb slider, torque (-R_i n) x F; also the next tangential
// displacement |delta| t + v_t dt, capped at the slider limit (dn).
__device__ void dem_pair(const Bufs &b, const Inst &I, int r, int partner, const double n[3],
                         double overlap, const double vij[3], const double wsR[3], double Ri,
                         double kn, double kt, double cn, double ct, double F[3], double T[3],
                         double dn[3])
{
    const double vn = vij[0] * n[0] + vij[1] * n[1] + vij[2] * n[2];
    double Fn[3], wxn[3], vt[3];
    cross3(wsR, n, wxn);
    for (int a = 0; a < 3; ++a) {
        Fn[a] = -kn * overlap * n[a] - cn * vn * n[a];
        vt[a] = vij[a] - vn * n[a] - wxn[a];
    }
    double dl[3] = { 0.0, 0.0, 0.0 };
    const int K = b.K;
    const int hc = b.h_n[r];
    for (int k = 0; k < hc; ++k)
        if (b.h_part[r * K + k] == partner) {
            for (int a = 0; a < 3; ++a) dl[a] = b.h_del[((long long)r * K + k) * 3 + a];
            break;
        }
    const double vtm = sqrt(vt[0] * vt[0] + vt[1] * vt[1] + vt[2] * vt[2]);
    const double dm = sqrt(dl[0] * dl[0] + dl[1] * dl[1] + dl[2] * dl[2]);
    double t[3] = { 0.0, 0.0, 0.0 };
    if (vtm > 0.0) {
        for (int a = 0; a < 3; ++a) t[a] = vt[a] / vtm;
    } else if (dm > 0.0) {
        for (int a = 0; a < 3; ++a) t[a] = dl[a] / dm;
    }
    double Ft[3];
    for (int a = 0; a < 3; ++a) Ft[a] = -kt * dl[a] - ct * vt[a];
    const double Fnm = sqrt(Fn[0] * Fn[0] + Fn[1] * Fn[1] + Fn[2] * Fn[2]);
    const double Ftm = sqrt(Ft[0] * Ft[0] + Ft[1] * Ft[1] + Ft[2] * Ft[2]);
    if (Ftm >= I.mu_fric * Fnm)
        for (int a = 0; a < 3; ++a) Ft[a] = -I.mu_fric * Fnm * t[a];
    double Fs[3], lev[3], tq[3];
    for (int a = 0; a < 3; ++a) {
        Fs[a] = Fn[a] + Ft[a];
        lev[a] = -Ri * n[a];
    }
    cross3(lev, Fs, tq);
    for (int a = 0; a < 3; ++a) {
        F[a] += Fs[a];
        T[a] += tq[a];
    }
    for (int a = 0; a < 3; ++a) dn[a] = dm * t[a] + vt[a] * I.dt;
    const double dnm = sqrt(dn[0] * dn[0] + dn[1] * dn[1] + dn[2] * dn[2]);
    const double cap = kt > 0.0 ? I.mu_fric * Fnm / kt : 0.0;
    if (dnm > cap && dnm > 0.0) {
        const double sc = cap / dnm;
        for (int a = 0; a < 3; ++a) dn[a] *= sc;
    }
}

__device__ __forceinline__ void hist_put(const Bufs &b, int r, int slot, int partner, const double dn[3])
{
    if (slot < b.K) {
        b.hn_part[r * b.K + slot] = partner;
        for (int a = 0; a < 3; ++a) b.hn_del[((long long)r * b.K + slot) * 3 + a] = dn[a];
    } else {
        atomicOr(b.err, ERR_CONTACT_CAP);
    }
}

// Rigid particles, one warp each: pressure-gradient force from the fluid
// neighbours (Eq. F_fpi_PG), DEM + lubrication with the rigid neighbours,
// wall planes, drag, gravity.  The lanes take the neighbour list in rounds of
// 32 for the fluid pairs and collect the rigid entries, in list order, in
// shared memory.  A sphere has only a few sphere neighbours, so the block's
// RPB spheres pool theirs: the pooled pairs run one per thread, RB at a time
// (their FP64 DEM and lubrication arithmetic on every lane instead of on a
// few lanes of each warp), each result is kept in shared memory, and each
// sphere adds its own in list order.  New history entries go to slots in list
// order, so the table is deterministic.
struct RigidPairRes {
    double F[3], T[3], L[3], dn[3];   // DEM force and torque, lubrication, next tangential displacement
    int partner;                      // gid of a contact partner, -1 without contact
    int pad;
};
__host__ __device__ inline size_t rigid_list_bytes(int cap) { return ((size_t)RPB * cap * sizeof(uint32_t) + 15) / 16 * 16; }
__host__ __device__ inline size_t rigid_smem_bytes(int cap) { return rigid_list_bytes(cap) + (size_t)RB * sizeof(RigidPairRes); }

template <class R>
__global__ void __launch_bounds__(RB) k_force_rigid(Bufs b, int velver)
{
    extern __shared__ __align__(16) unsigned char rsm[];
    __shared__ double s_x[RPB][3], s_v[RPB][3], s_w[RPB][3], s_R[RPB], s_m[RPB];
    __shared__ int s_r[RPB], s_inst[RPB], s_nr[RPB], s_pre[RPB + 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r = blockIdx.x * RPB + warp;
    const bool live = r < b.nrigid;   // a warp past the end only takes part in the barriers
    uint32_t *const lists = reinterpret_cast<uint32_t *>(rsm);
    uint32_t *rl = lists + (size_t)warp * b.cap;   // this warp's rigid entries
    RigidPairRes *pres = reinterpret_cast<RigidPairRes *>(rsm + rigid_list_bytes(b.cap));
    const int g = live ? b.rigid_gid[r] : 0;
    const long long s = live ? b.slot_of[g] : 0;
    const Inst &I = b.inst[b.pinst[g]];
    double xi[3] = { 0.0, 0.0, 0.0 }, vi[3] = { 0.0, 0.0, 0.0 }, wi[3] = { 0.0, 0.0, 0.0 };
    double Ri = 0.0, mi = 0.0, di = 0.0;
    if (live) {
        for (int a = 0; a < 3; ++a) {
            xi[a] = b.x[3 * g + a];
            vi[a] = b.v[3 * g + a];
            wi[a] = b.w[3 * g + a];
        }
        Ri = b.R[g];
        mi = b.m[g];
        di = b.sd[s];
        if (lane == 0) {
            for (int a = 0; a < 3; ++a) {
                s_x[warp][a] = xi[a];
                s_v[warp][a] = vi[a];
                s_w[warp][a] = wi[a];
            }
            s_R[warp] = Ri;
            s_m[warp] = mi;
            s_r[warp] = r;
            s_inst[warp] = b.pinst[g];
        }
    }
    const bool commit = (velver == 2);
    double acc[15];
#pragma unroll
    for (int a = 0; a < 15; ++a) acc[a] = 0.0;   // pg, npg, Fdem, Tdem, Flub
    // the fluid pairs in precision R on the mirrors, as for fluid pairs (the
    // C + D part of the SDPD pair, the exact r < h decision of Rel), summed
    // per lane in R; DEM and lubrication stay FP64
    using T4 = typename Vec<R>::T4;
    using TA = typename Mir<R>::TA;
    const Geo<R> geo(I);
    const TA *__restrict__ A = Mir<R>::A(b);
    const T4 *__restrict__ Bm = Mir<R>::B(b);
    const T4 *__restrict__ Cm = Mir<R>::C(b);
    const T4 *__restrict__ Dm = Mir<R>::D(b);
    const TA Ai = A[s];
    const T4 Bi = Bm[s], Ci = Cm[s], Di = Dm[s];
    const PairK<R> P(I, 0u, Ci, Di);
    const R Rr = (R)Ri;
    R f0 = 0, f1 = 0, f2 = 0, t0 = 0, t1 = 0, t2 = 0;
    const int n = live ? b.ncnt[s] : 0;
    const unsigned below = (1u << lane) - 1u;
    int nr = 0;   // rigid entries collected
    // the entry of the next round is fetched one round ahead
    uint32_t en = lane < n ? (uint32_t)__ldg(b.nbr + entry_at(lane, s, b.rows)) : 0u;
    for (int kk = 0; kk < n; kk += 32) {
        const int k = kk + lane;
        bool rig = false;
        const uint32_t e = en;
        if (k + 32 < n) en = (uint32_t)__ldg(b.nbr + entry_at(k + 32, s, b.rows));
        if (k < n) {
            const int j = (int)(e & ~NB_FAR);
            const TA Aj = A[j];
            const int tj = mir_type(Aj);
            if (tj == T_FLUID && !(e & NB_FAR)) {
                // F^C + F^D of the pair (s, j), summed for Eq. F_fpi_PG
                R rx, ry, rz, r2;
                if (Rel<R>::get(b, I, geo, Ai, Aj, g, j, rx, ry, rz, r2)) {
                    Z6<R> z;
                    R ox, oy, oz, ce, ex, ey, ez, q, om;
                    sdpd_pair<R>(P, rx, ry, rz, r2, Bi, Ci, Di, Bm[j], Cm[j], Dm[j], false, 0, z, ox, oy, oz, ce,
                                 ex, ey, ez, q, om);
                    f0 += ox + ce * ex;
                    f1 += oy + ce * ey;
                    f2 += oz + ce * ez;
                    // lever -R e: (-R e) x (o + ce e) = -R e x o
                    t0 -= Rr * (ey * oz - ez * oy);
                    t1 -= Rr * (ez * ox - ex * oz);
                    t2 -= Rr * (ex * oy - ey * ox);
                }
            } else {
                rig = (tj == T_RIGID);
            }
        }
        const unsigned rb = __ballot_sync(0xffffffffu, rig);
        if (rig) rl[nr + __popc(rb & below)] = e;
        nr += __popc(rb);
    }
    if (lane == 0) s_nr[warp] = nr;
    __syncthreads();
    if (threadIdx.x == 0) {
        s_pre[0] = 0;
        for (int w = 0; w < RPB; ++w) s_pre[w + 1] = s_pre[w] + s_nr[w];
    }
    __syncthreads();
    // the pooled rigid pairs (sphere w's entries at [s_pre[w], s_pre[w+1])),
    // RB at a time: DEM contact, or lubrication
    const int total = s_pre[RPB];
    double mine = 0.0;   // lane c < 9 of a live warp: component c of F_dem, T_dem, F_lub
    int base = 0;        // history slots used so far (the same on every lane)
    for (int c0 = 0; c0 < total; c0 += RB) {
        const int p = c0 + threadIdx.x;
        if (p < total) {
            int ws = 0;
            while (ws + 1 < RPB && s_pre[ws + 1] <= p) ++ws;
            const uint32_t e = lists[(size_t)ws * b.cap + (p - s_pre[ws])];
            const Inst &Iw = b.inst[s_inst[ws]];
            const double xs[3] = { s_x[ws][0], s_x[ws][1], s_x[ws][2] };
            const double Rs = s_R[ws];
            RigidPairRes &o = pres[threadIdx.x];
            for (int a = 0; a < 3; ++a) {
                o.F[a] = 0.0;
                o.T[a] = 0.0;
                o.L[a] = 0.0;
                o.dn[a] = 0.0;
            }
            o.partner = -1;
            const int j = (int)(e & ~NB_FAR);
            const int gj = b.perm[j];
            const double xj[3] = { b.x[3 * gj], b.x[3 * gj + 1], b.x[3 * gj + 2] };
            double rv[3];
            const double r2 = exact_disp(xs, xj, Iw, rv);
            const double L = sqrt(r2);
            const double vij[3] = { s_v[ws][0] - b.v[3 * gj], s_v[ws][1] - b.v[3 * gj + 1],
                                    s_v[ws][2] - b.v[3 * gj + 2] };
            const double Rj = b.R[gj];
            const double dsum = Rs + Rj;
            if (L < dsum) {
                const double nn[3] = { rv[0] / L, rv[1] / L, rv[2] / L };
                double wsR[3];
                for (int a = 0; a < 3; ++a) wsR[a] = Rs * s_w[ws][a] + Rj * b.w[3 * gj + a];
                double kn, kt, cn, ct;
                dem_coeffs(Iw, Rs, Rj, s_m[ws], b.m[gj], kn, kt, cn, ct);
                dem_pair(b, Iw, s_r[ws], gj, nn, L - dsum, vij, wsR, Rs, kn, kt, cn, ct, o.F, o.T, o.dn);
                o.partner = gj;
            } else if (r2 < Iw.rc2) {
                double gap = L - dsum;
                const double gmin = Iw.lub_gap_min * dsum;
                if (gap < gmin) gap = gmin;
                const double c = 3.0 * PI * Iw.eta * dsum * dsum / (8.0 * gap);
                for (int a = 0; a < 3; ++a) o.L[a] = c * (-vij[a]);
            }
        }
        __syncthreads();
        // each sphere adds its own pairs of this chunk in list order
        if (live) {
            const int lo = max(s_pre[warp], c0) - c0, hi = min(s_pre[warp + 1], c0 + RB) - c0;
            for (int t = lo; t < hi; ++t) {
                const RigidPairRes &o = pres[t];
                if (lane < 9) mine += lane < 3 ? o.F[lane] : (lane < 6 ? o.T[lane - 3] : o.L[lane - 6]);
                if (o.partner >= 0) {
                    if (lane == 0 && commit) hist_put(b, r, base, o.partner, o.dn);
                    ++base;
                }
            }
        }
        __syncthreads();
    }
    if (!live) return;   // past the block's last barrier
    acc[0] = f0; acc[1] = f1; acc[2] = f2;
    acc[3] = t0; acc[4] = t1; acc[5] = t2;
#pragma unroll
    for (int a = 0; a < 6; ++a) acc[a] = warp_sum(acc[a]);
#pragma unroll
    for (int c = 0; c < 9; ++c) acc[6 + c] = __shfl_sync(0xffffffffu, mine, c);
    if (lane != 0) return;
    // contact with the planes bounding the domain on wall axes
    for (int a = 0; a < 3; ++a) {
        if (I.periodic[a]) continue;
        for (int side = 0; side < 2; ++side) {
            const double L = side == 0 ? xi[a] - I.origin[a] : (I.origin[a] + I.box[a]) - xi[a];
            if (!(L < Ri)) continue;
            double nn[3] = { 0, 0, 0 };
            nn[a] = side == 0 ? 1.0 : -1.0;
            double wsR[3], dn[3];
            for (int c = 0; c < 3; ++c) wsR[c] = Ri * wi[c];
            double kn, kt, cn, ct;
            dem_coeffs(I, Ri, 0.0, mi, 0.0, kn, kt, cn, ct);
            dem_pair(b, I, r, PLANE_BASE + 2 * a + side, nn, L - Ri, vi, wsR, Ri, kn, kt, cn, ct,
                     acc + 6, acc + 9, dn);
            if (commit) hist_put(b, r, base, PLANE_BASE + 2 * a + side, dn);
            ++base;
        }
    }
    if (commit) b.hn_n[r] = base < b.K ? base : b.K;
    const double Vs = 4.0 / 3.0 * PI * Ri * Ri * Ri;
    const double sc = Vs * di;
    double ax[3];
    ext_accel(I, xi, ax);
    for (int a = 0; a < 3; ++a) {
        b.F[3 * g + a] = sc * acc[a] + b.fdg[3 * r + a] + acc[6 + a] + acc[12 + a] + mi * ax[a];
        b.T[3 * g + a] = sc * acc[3 + a] + acc[9 + a];
    }
}

__global__ void k_hist_copy(Bufs b)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= b.nrigid) return;
    const int n = b.hn_n[r];
    b.h_n[r] = n;
    for (int k = 0; k < n; ++k) {
        b.h_part[r * b.K + k] = b.hn_part[r * b.K + k];
        for (int a = 0; a < 3; ++a)
            b.h_del[((long long)r * b.K + k) * 3 + a] = b.hn_del[((long long)r * b.K + k) * 3 + a];
    }
}

// ---------------------------------------------------------------- launchers
static inline unsigned nblk(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

// Groups of GROUP particles a warp of a pair pass takes one after another: as
// many (at most 8: one particle per lane at the end) as still give every SM
// 32 warps, so that small systems spread over the chip and large ones pay the
// closing arithmetic once per 32 particles.
static int pass_groups(long long N)
{
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    const long long g = N / (GROUP * 32LL * std::max(nsm, 1));
    return (int)std::min<long long>(8, std::max<long long>(1, g));
}
// Blocks of `block` threads that cover N particles at `groups` groups a warp.
static unsigned pass_blocks(long long N, int block, int groups) { return nblk(N, block / 32 * GROUP * groups); }

void launch_density(const Bufs &b, int precision, int dflags, int newton3, const int *gate, cudaStream_t st)
{
    if (!b.N) return;
    const int any_filter = dflags & 1, any_reinit = (dflags >> 1) & 1, any_artvis = (dflags >> 2) & 1;
    // the density kernels leave the mirrors to a later pass when one follows
    const int defer = any_filter | (any_reinit << 1);
    const int groups = pass_groups(b.N), bs = b.pair_block;
    const unsigned nb = pass_blocks(b.N, bs, groups);
    if (precision == SDPD_PREC_SPLIT) {
        if (any_artvis) k_density32<true><<<nb, bs, 0, st>>>(b, defer, gate, groups);
        else k_density32<false><<<nb, bs, 0, st>>>(b, defer, gate, groups);
        if (any_reinit) k_shepard32<true><<<nb, bs, 0, st>>>(b, any_filter, gate, groups);
    } else {
        if (newton3) {
            k_density_half<<<nb, bs, 0, st>>>(b, gate, groups);
            k_density_gather<<<nb, bs, 0, st>>>(b, defer, gate, groups);
        } else if (any_artvis) {
            k_density<true><<<nb, bs, 0, st>>>(b, defer, gate, groups);
        } else {
            k_density<false><<<nb, bs, 0, st>>>(b, defer, gate, groups);
        }
        if (any_reinit) k_shepard<true><<<nb, bs, 0, st>>>(b, any_filter, gate, groups);
    }
    if (any_reinit) k_reinit_copy<<<nblk(b.N, 256), 256, 0, st>>>(b, gate);
    if (any_filter) {
        if (precision == SDPD_PREC_SPLIT) k_shepard32<false><<<nb, bs, 0, st>>>(b, 0, gate, groups);
        else k_shepard<false><<<nb, bs, 0, st>>>(b, 0, gate, groups);
    }
}

void launch_drag(const Bufs &b, int precision, cudaStream_t st)
{
    if (!b.nrigid) return;
    const unsigned g = nblk(b.nrigid, RPB);
    if (precision == SDPD_PREC_SPLIT) k_drag<float><<<g, RB, 0, st>>>(b);
    else k_drag<double><<<g, RB, 0, st>>>(b);
    k_drag_law<<<nblk(b.nrigid, 16), 32, 0, st>>>(b);
}


void init_pair_kernels()
{
    // the sphere kernel's rigid lists and pooled-pair results at the largest
    // list capacity
    cudaFuncSetAttribute(k_force_rigid<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)rigid_smem_bytes(SDPD_MAX_NEIGHBORS));
    cudaFuncSetAttribute(k_force_rigid<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)rigid_smem_bytes(SDPD_MAX_NEIGHBORS));
}

void launch_forces(const Bufs &b, int precision, int velver, int newton3, cudaStream_t st, cudaStream_t rigid)
{
    if (!b.N) return;
    // the spheres' forces first: few blocks of long chains, which the fluid
    // pass then fills up around where `rigid` is a stream of its own
    if (b.nrigid) {
        const unsigned g = nblk(b.nrigid, RPB);
        const size_t smem = rigid_smem_bytes(b.cap);
        if (precision == SDPD_PREC_SPLIT) k_force_rigid<float><<<g, RB, smem, rigid>>>(b, velver);
        else k_force_rigid<double><<<g, RB, smem, rigid>>>(b, velver);
        if (velver == 2) k_hist_copy<<<nblk(b.nrigid, 64), 64, 0, rigid>>>(b);
    }
    const int bs = b.pair_block, groups = pass_groups(b.N);
    const unsigned nb = pass_blocks(b.N, bs, groups);
    if (newton3 == 1 || newton3 == 4) {
        if (precision == SDPD_PREC_SPLIT && newton3 == 4) {
            k_force_half<float, true><<<nb, bs, 0, st>>>(b, velver, groups);
            k_force_gather<float, true><<<nb, bs, 0, st>>>(b, groups);
        } else if (precision == SDPD_PREC_SPLIT) {
            k_force_half<float, false><<<nb, bs, 0, st>>>(b, velver, groups);
            k_force_gather<float, false><<<nb, bs, 0, st>>>(b, groups);
        } else {
            k_force_half<double, true><<<nb, bs, 0, st>>>(b, velver, groups);
            k_force_gather<double, true><<<nb, bs, 0, st>>>(b, groups);
        }
    } else if (precision == SDPD_PREC_SPLIT) {
        // second evaluation: the pass that reads the cached normals, then the
        // drawing pass for the instances whose lists were rebuilt since
        if (velver == 2) k_force_cached<<<pass_blocks(b.N, ZTHREADS, groups), ZTHREADS, 0, st>>>(b, groups);
        k_force_draw<<<nb, bs, 0, st>>>(b, velver, groups);
    } else {
        k_force_fluid<<<nb, bs, 0, st>>>(b, velver, groups);
    }
}

}  // namespace sdpd
