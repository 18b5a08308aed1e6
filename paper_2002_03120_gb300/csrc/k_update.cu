// k_update.cu -- update(velver) of Algorithm 1 (velocity Verlet, boundary
// treatment, collision-method artificial viscosity) and the reductions of the
// viscometer read-out and the diagnostics.
#define BM_TABLES
#include "common.cuh"

namespace sdpd {

template <class R> struct VT;
template <> struct VT<float> { using T4 = float4; };
template <> struct VT<double> { using T4 = double4_32a; };

template <class R> __device__ __forceinline__ typename VT<R>::T4 *mirB(const Bufs &b);
template <> __device__ __forceinline__ float4 *mirB<float>(const Bufs &b) { return b.B32; }
template <> __device__ __forceinline__ double4_32a *mirB<double>(const Bufs &b) { return b.B64; }
template <class R> __device__ __forceinline__ typename VT<R>::T4 *mirC(const Bufs &b);
template <> __device__ __forceinline__ float4 *mirC<float>(const Bufs &b) { return b.C32; }
template <> __device__ __forceinline__ double4_32a *mirC<double>(const Bufs &b) { return b.C64; }

template <class R>
__device__ __forceinline__ void write_vel_mirror(const Bufs &b, long long s, const double *v, const double *w)
{
    auto *B = mirB<R>(b);
    auto *C = mirC<R>(b);
    auto Bs = B[s];
    auto Cs = C[s];
    Bs.x = (R)v[0]; Bs.y = (R)v[1]; Bs.z = (R)v[2];
    Cs.x = (R)w[0]; Cs.y = (R)w[1]; Cs.z = (R)w[2];
    B[s] = Bs;
    C[s] = Cs;
}

// a / d rounded to nearest from y = RN(1/d) by Markstein's method (P.
// Markstein, IBM J. Res. Dev. 34, 1990): q0 = RN(a y), the remainder
// r = a - d q0 is exact with a fused multiply-add, and RN(q0 + r y) is the
// correctly rounded quotient (no overflow or underflow here): the result of
// the division a / d, with one multiply and two multiply-adds.
__device__ __forceinline__ double div_rn(double a, double d, double y)
{
    const double q0 = __dmul_rn(a, y);
    const double r = __fma_rn(-q0, d, a);
    return __fma_rn(r, y, q0);
}

// Comparisons on the integer pipe (the FP64 pipe of this part runs at 1/64 of
// the FP32 rate and bounds the update): key(x) orders like x for every
// non-NaN double, -0 and +0 alike; a NaN takes a branch the IEEE comparison
// would not, but stays NaN and is flagged either way.
__device__ __forceinline__ long long ord_key(double x)
{
    const long long k = __double_as_longlong(x);
    return k >= 0 ? k : (long long)(0x8000000000000000ull - (unsigned long long)k);
}
// the high word, ordered like x (never falls where x rises)
__device__ __forceinline__ int hi_key(double x)
{
    const int h = __double2hiint(x);
    return h ^ ((h >> 31) & 0x7FFFFFFF);
}
__device__ __forceinline__ bool finite_bits(double x) { return hi_abs(x) < 0x7FF00000; }

// A particle has used up half the skin: its instance's lists are rebuilt
// before the next pair pass.  In the captured step `build` opens the
// conditional node that holds the build.
__device__ __forceinline__ void request_build(const Bufs &b, int inst, cudaGraphConditionalHandle build)
{
    b.need_build[0] = 1;
    b.need_build[1 + inst] = 1;
    if (build) cudaGraphSetConditional(build, 1);
}
// The displacement since the build, from the fixed-point coordinates.  A
// single move of half the skin or more along an axis is told apart by its
// FP64 value (drift_hi), so a sum of shorter ones is requested long before
// the coordinates could wrap.
__device__ __forceinline__ bool moved_far(const int4 &now, const int4 &build, const Inst &I)
{
    const float dx = (float)fixed_diff(now.x, build.x) * I.unit[0], dy = (float)fixed_diff(now.y, build.y) * I.unit[1],
                dz = (float)fixed_diff(now.z, build.z) * I.unit[2];
    return dx * dx + dy * dy + dz * dz > I.moved2;
}

__device__ __forceinline__ void step_done(const Bufs &b)
{
    *b.step += 1;
    *b.fresh = 0;
}
__global__ void k_step_done(Bufs b) { step_done(b); }   // (a context without particles)

// Velocity Verlet (Eqs. newton1, newton2): v += dt/2 F/m, w += dt/2 N/I;
// velver 1 also drifts x += dt v, wraps periodic axes and mirrors particles
// that crossed a wall plane (normal velocity reversed); velver 2 also closes
// the step (nothing after it reads the step number).  The arithmetic is
// written without fused multiply-adds so it repeats the oracle bit for bit;
// the decisions (wrap, reflection, finiteness) are taken on the integer pipe
// from the bit patterns, with the oracle's outcomes.
//
// Bound by the FP64 pipe (36 operations a particle, 48 with the drift: three
// for each division, six conversions of the mirrors) and the latency of the
// gathers by gid, so every load stands before the first store (a store to one
// axis once held back the loads of the next).  Displacements come from the
// fixed-point coordinates instead of an FP64 sum that was read and written
// every step.  Dam break of 374,000 particles, 148,000 of them moving: 54 ->
// 26 us with the drift, 22 -> 20 us without.
template <class R>
__global__ void __launch_bounds__(256) k_integrate(Bufs b, int velver, cudaGraphConditionalHandle gate)
{
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s == 0) {
        if (velver == 1) *b.aclose_ok = 0;   // the drift moves the particles
        else step_done(b);
    }
    if (s >= b.N) return;
    const int g = b.perm[s];
    const int t = b.stype[s];
    if (t != T_FLUID && t != T_RIGID) return;
    const int inst = b.pinst[g];
    const Inst &I = b.inst[inst];
    const bool drift = velver == 1;
    double v[3], w[3], F[3], T[3], x[3] = { 0.0, 0.0, 0.0 };
    const double im = b.m[g], iI = b.Iner[g], rm = b.rm[g], rI = b.rI[g];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        F[a] = b.F[3 * g + a];
        T[a] = b.T[3 * g + a];
        v[a] = b.v[3 * g + a];
        w[a] = b.w[3 * g + a];
        if (drift) x[a] = b.x[3 * g + a];
    }
    auto *B = mirB<R>(b);
    auto *C = mirC<R>(b);
    auto Bs = B[s];
    auto Cs = C[s];
    int4 build = make_int4(0, 0, 0, 0);
    if (drift) build = b.A32_build[s];
    const double hdt = I.hdt;
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        v[a] = __dadd_rn(v[a], __dmul_rn(hdt, div_rn(F[a], im, rm)));
        w[a] = __dadd_rn(w[a], __dmul_rn(hdt, div_rn(T[a], iI, rI)));
    }
    if (drift) {
        const double dt = I.dt;
        bool far = false;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double move = __dmul_rn(dt, v[a]);
            double xa = __dadd_rn(x[a], move);
            far |= hi_abs(move) >= I.drift_hi;
            const int key = hi_key(xa);
            if (key <= I.key_lo[a] || key >= I.key_hi[a]) {   // at the faces or outside: decided on all bits
                const double lo = I.origin[a], hi = I.dom_hi[a], L = I.box[a];
                const long long kx = ord_key(xa);
                if (I.periodic[a]) {
                    if (kx < ord_key(lo)) xa = __dadd_rn(xa, L);
                    else if (kx >= ord_key(hi)) xa = __dsub_rn(xa, L);
                } else {
                    if (kx < ord_key(lo)) { xa = __dadd_rn(lo, __dsub_rn(lo, xa)); v[a] = flip_sign(v[a], 0x80000000u); }
                    else if (kx > ord_key(hi)) { xa = __dsub_rn(hi, __dsub_rn(xa, hi)); v[a] = flip_sign(v[a], 0x80000000u); }
                }
            }
            x[a] = xa;
            ok &= finite_bits(xa);
        }
        // keep the mirrors of the unchanged slot order current; the
        // displacement since the build decides whether the list still holds
        const int4 now = make_int4(fixed_coord(x[0], I, 0), fixed_coord(x[1], I, 1), fixed_coord(x[2], I, 2), t);
        if (far || moved_far(now, build, I)) request_build(b, inst, gate);
        b.A32[s] = now;
        if (b.A64) {
            double4_32a a64 = b.A64[s];
            a64.x = x[0]; a64.y = x[1]; a64.z = x[2];
            b.A64[s] = a64;
        }
#pragma unroll
        for (int a = 0; a < 3; ++a) b.x[3 * g + a] = x[a];
    }
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        b.v[3 * g + a] = v[a];
        b.w[3 * g + a] = w[a];
        ok &= finite_bits(v[a]) & finite_bits(w[a]);
    }
    if (!ok) atomicOr(b.err, ERR_NONFINITE);
    Bs.x = (R)v[0]; Bs.y = (R)v[1]; Bs.z = (R)v[2];
    Cs.x = (R)w[0]; Cs.y = (R)w[1]; Cs.z = (R)w[2];
    B[s] = Bs;
    C[s] = Cs;
}

// Absorb uploaded state (sdpd_upload_state) into a context whose lists are
// valid: each particle moves by its displacement (minimum image on periodic
// axes), the position mirrors and the displacement since the build move
// with it, and the velocity mirrors take the uploaded velocities.  A
// displacement beyond half the skin requests a rebuild (the gated build of
// the next step), exactly as after a drift; otherwise the lists still hold
// every pair within h.
template <class R>
__global__ void k_absorb(Bufs b, const double *__restrict__ xs, int has_x)
{
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= b.N) return;
    const int g = b.perm[s];
    const Inst &I = b.inst[b.pinst[g]];
    if (has_x) {
        double x[3];
        bool far = false;
        for (int a = 0; a < 3; ++a) {
            const double x0 = b.x[3 * g + a], xa = xs[3 * g + a];
            double d = xa - x0;
            if (I.periodic[a]) {
                if (d > 0.5 * I.box[a]) d -= I.box[a];
                else if (d < -0.5 * I.box[a]) d += I.box[a];
            }
            far |= hi_abs(d) >= I.drift_hi;
            x[a] = xa;
            b.x[3 * g + a] = xa;
        }
        const int4 now = make_int4(fixed_coord(x[0], I, 0), fixed_coord(x[1], I, 1), fixed_coord(x[2], I, 2), b.type[g]);
        b.A32[s] = now;
        if (b.A64) {
            double4_32a a64 = b.A64[s];
            a64.x = x[0]; a64.y = x[1]; a64.z = x[2];
            b.A64[s] = a64;
        }
        if (far || moved_far(now, b.A32_build[s], I)) request_build(b, b.pinst[g], 0);
    }
    const double v[3] = { b.v[3 * g], b.v[3 * g + 1], b.v[3 * g + 2] };
    const double w[3] = { b.w[3 * g], b.w[3 * g + 1], b.w[3 * g + 2] };
    write_vel_mirror<R>(b, s, v, w);
    if (s == 0) *b.aclose_ok = 0;   // positions changed
}

// Collision-method artificial viscosity: pairs of mobile particles closer
// than artvis_alpha dx that approach exchange momentum as an inelastic
// collision with restitution artvis_e; Jacobi form (pre-correction
// velocities), momentum-conserving.
__global__ void k_artvis(Bufs b)
{
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= b.N) return;
    const int g = b.perm[s];
    const int t = b.type[g];
    double dv[3] = { 0.0, 0.0, 0.0 };
    const Inst &I = b.inst[b.pinst[g]];
    // the density pass of these positions marked the particles that have a
    // mobile neighbour inside the collision radius; the others skip the scan
    const bool marked = !*b.aclose_ok || b.aclose[s];
    if ((t == T_FLUID || t == T_RIGID) && I.artvis && marked) {
        const double xi[3] = { b.x[3 * g], b.x[3 * g + 1], b.x[3 * g + 2] };
        const double vi[3] = { b.v[3 * g], b.v[3 * g + 1], b.v[3 * g + 2] };
        const double mi = b.m[g];
        const int n = b.ncnt[s];
        const Geo<float> geo(I);
        const int4 Ai = b.A32[s];
        const float r2hi = I.artvis_r2f_hi;
        for (int k = 0; k < n; ++k) {
            const uint32_t e = (uint32_t)b.nbr[entry_at(k, s, b.rows)];
            if (e & NB_FAR) continue;
            // float prefilter on the fixed-point mirror; exact test below
            const int4 Aj = b.A32[e];
            float fx, fy, fz;
            geo.disp(Ai, Aj, fx, fy, fz);
            if (fx * fx + fy * fy + fz * fz > r2hi) continue;
            const int gj = b.perm[e];
            const int tj = b.type[gj];
            if (tj != T_FLUID && tj != T_RIGID) continue;
            double r[3];
            for (int a = 0; a < 3; ++a) {
                double d = xi[a] - b.x[3 * gj + a];
                if (I.periodic[a]) {
                    if (d > 0.5 * I.box[a]) d -= I.box[a];
                    else if (d < -0.5 * I.box[a]) d += I.box[a];
                }
                r[a] = d;
            }
            const double rr = sqrt((r[0] * r[0] + r[1] * r[1]) + r[2] * r[2]);
            if (!(rr < I.artvis_rlim)) continue;
            const double e3[3] = { r[0] / rr, r[1] / rr, r[2] / rr };
            const double ve = (vi[0] - b.v[3 * gj]) * e3[0] + (vi[1] - b.v[3 * gj + 1]) * e3[1] +
                              (vi[2] - b.v[3 * gj + 2]) * e3[2];
            if (!(ve < 0.0)) continue;
            const double mj = b.m[gj];
            const double c = -(1.0 + I.artvis_e) * mj / (mi + mj) * ve;
            for (int a = 0; a < 3; ++a) dv[a] += c * e3[a];
        }
    }
    b.dv[3 * g] = dv[0];
    b.dv[3 * g + 1] = dv[1];
    b.dv[3 * g + 2] = dv[2];
}

template <class R>
__global__ void k_artvis_apply(Bufs b)
{
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= b.N) return;
    const int g = b.perm[s];
    const int t = b.type[g];
    if (t != T_FLUID && t != T_RIGID) return;
    double v[3], w[3];
    for (int a = 0; a < 3; ++a) {
        v[a] = b.v[3 * g + a] + b.dv[3 * g + a];
        b.v[3 * g + a] = v[a];
        w[a] = b.w[3 * g + a];
    }
    write_vel_mirror<R>(b, s, v, w);
}

// ----------------------------------------------------- viscometer read-out
// probe layout: [0, nb) velocity sums, [nb, 2nb) counts, [2nb, 2nb+4)
// signed velocity sums and counts of the two halves, [2nb+4, 3nb+4) position
// sums, [3nb+4] the error word.  The halves' sums are formed per warp (an atomic for
// every particle on two addresses was most of the time).
__global__ void k_probe(Bufs b, int inst, int nb)
{
    const Inst &I = b.inst[inst];
    const long long g = I.p_begin + (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g == I.p_begin) b.probe[3 * nb + 4] = (double)*b.err;
    const bool use = g < I.p_end && b.type[g] == T_FLUID;
    const int ax = I.split_axis, fa = I.body_axis;
    double u = 0.0;
    int half = 0;
    if (use) {
        const double rel = b.x[3 * g + ax] - I.origin[ax];
        int bin = (int)floor(rel / I.box[ax] * nb);
        bin = bin < 0 ? 0 : (bin >= nb ? nb - 1 : bin);
        u = b.v[3 * g + fa];
        atomicAdd(&b.probe[bin], u);
        atomicAdd(&b.probe[nb + bin], 1.0);
        atomicAdd(&b.probe[2 * nb + 4 + bin], rel);   // mean position of the slab's particles
        half = (rel < 0.5 * I.box[ax]) ? 0 : 1;
    }
    const double u0 = warp_sum(use && half == 0 ? u : 0.0), u1 = warp_sum(use && half == 1 ? -u : 0.0);
    const int n0 = __popc(__ballot_sync(0xffffffffu, use && half == 0)), n1 = __popc(__ballot_sync(0xffffffffu, use && half == 1));
    if ((threadIdx.x & 31) == 0) {
        if (n0) {
            atomicAdd(&b.probe[2 * nb], u0);
            atomicAdd(&b.probe[2 * nb + 2], (double)n0);
        }
        if (n1) {
            atomicAdd(&b.probe[2 * nb + 1], u1);
            atomicAdd(&b.probe[2 * nb + 3], (double)n1);
        }
    }
}

// diagnostics layout in probe: [0..2] momentum, [3] sum m v^2, [4] sum m,
// [5] count mobile, [6] max |v| (as ordered bits), [7] min d, [8] max d,
// [9] non-finite count
__global__ void k_diag(Bufs b, int inst)
{
    const Inst &I = b.inst[inst];
    const long long g = I.p_begin + (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= I.p_end) return;
    const int t = b.type[g];
    double nonf = 0.0;
    for (int a = 0; a < 3; ++a)
        nonf += (!isfinite(b.x[3 * g + a])) + (!isfinite(b.v[3 * g + a])) + (!isfinite(b.w[3 * g + a]));
    if (nonf > 0) atomicAdd(&b.probe[9], nonf);
    const long long s = b.slot_of[g];
    if (t != T_OUTER) {
        const double d = b.sd[s];
        atomicMin((unsigned long long *)&b.probe[7], (unsigned long long)__double_as_longlong(d));
        atomicMax((unsigned long long *)&b.probe[8], (unsigned long long)__double_as_longlong(d));
    }
    if (t != T_FLUID && t != T_RIGID) return;
    const double m = b.m[g];
    const double v0 = b.v[3 * g], v1 = b.v[3 * g + 1], v2 = b.v[3 * g + 2];
    atomicAdd(&b.probe[0], m * v0);
    atomicAdd(&b.probe[1], m * v1);
    atomicAdd(&b.probe[2], m * v2);
    const double v2s = v0 * v0 + v1 * v1 + v2 * v2;
    atomicAdd(&b.probe[3], m * v2s);
    atomicAdd(&b.probe[4], m);
    atomicAdd(&b.probe[5], 1.0);
    atomicMax((unsigned long long *)&b.probe[6], (unsigned long long)__double_as_longlong(sqrt(v2s)));
}

// Unordered pairs within h evaluated by the force pass (>= 1 mobile member).
__global__ void k_count_pairs(Bufs b)
{
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long c = 0;
    if (s < b.N) {
        const int ti = b.stype[s];
        if (ti == T_FLUID || ti == T_RIGID) {
            const int n = b.ncnt[s];
            const int gi = b.perm[s];
            const Inst &I = b.inst[b.pinst[gi]];
            for (int k = 0; k < n; ++k) {
                const uint32_t e = (uint32_t)b.nbr[entry_at(k, s, b.rows)];
                if (e & NB_FAR) continue;
                if (!exact_within(b, I, gi, b.perm[e])) continue;
                const int tj = b.stype[e];
                const bool mj = (tj == T_FLUID || tj == T_RIGID);
                c += mj ? ((long long)e > s ? 1u : 0u) : 1u;
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(0xffffffffu, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(b.pair_count, c);
}

// Flags of the list entries within h at the current positions (exact test).
__global__ void k_mark_pairs(Bufs b, uint8_t *flags)
{
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= b.N) return;
    const int gi = b.perm[s];
    const Inst &I = b.inst[b.pinst[gi]];
    const int n = b.ncnt[s];
    for (int k = 0; k < n; ++k) {
        const uint32_t e = (uint32_t)b.nbr[entry_at(k, s, b.rows)];
        flags[(long long)k * b.Npad + s] =
            (!(e & NB_FAR) && exact_within(b, I, gi, b.perm[e & ~NB_FAR])) ? 1 : 0;
    }
}

// ---------------------------------------------------------------- launchers
static inline unsigned nblk(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

void launch_integrate(const Bufs &b, int precision, int velver, int any_artvis, cudaStream_t st,
                      cudaGraphConditionalHandle build)
{
    if (!b.N) {
        if (velver == 2) k_step_done<<<1, 1, 0, st>>>(b);
        return;
    }
    const int bs = spread_block(b.N);
    if (precision == SDPD_PREC_SPLIT) k_integrate<float><<<nblk(b.N, bs), bs, 0, st>>>(b, velver, build);
    else k_integrate<double><<<nblk(b.N, bs), bs, 0, st>>>(b, velver, build);
    if (velver == 2 && any_artvis) {
        k_artvis<<<nblk(b.N, 128), 128, 0, st>>>(b);
        if (precision == SDPD_PREC_SPLIT) k_artvis_apply<float><<<nblk(b.N, 256), 256, 0, st>>>(b);
        else k_artvis_apply<double><<<nblk(b.N, 256), 256, 0, st>>>(b);
    }
}

void launch_probe(const Bufs &b, int inst, int nbins, cudaStream_t st, long long n)
{
    cudaMemsetAsync(b.probe, 0, sizeof(double) * (3 * nbins + 4), st);
    if (n) k_probe<<<nblk(n, spread_block(n)), spread_block(n), 0, st>>>(b, inst, nbins);
}

void launch_diag(const Bufs &b, int inst, cudaStream_t st, long long n)
{
    cudaMemsetAsync(b.probe, 0, sizeof(double) * 16, st);
    // min d starts at +inf bits
    const double big = 1e308;
    cudaMemcpyAsync(&b.probe[7], &big, sizeof(double), cudaMemcpyHostToDevice, st);
    if (n) k_diag<<<nblk(n, 256), 256, 0, st>>>(b, inst);
}

void launch_mark_pairs(const Bufs &b, uint8_t *flags, cudaStream_t st)
{
    if (b.N) k_mark_pairs<<<nblk(b.N, 128), 128, 0, st>>>(b, flags);
}

// The six normals of the random term (Eq. FijT) of given pairs, as the pair
// kernels draw them.
template <class R>
__global__ void k_noise_normals(long long n, const uint32_t *gi, const uint32_t *gj, uint32_t step, uint32_t k0,
                                uint32_t k1, double *out)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    R z[6];
    pair_normals<R>(gi[i], gj[i], step, k0, k1, z[0], z[1], z[2], z[3], z[4], z[5]);
#pragma unroll
    for (int k = 0; k < 6; ++k) out[6 * i + k] = (double)z[k];
}

// Raw Philox4x32-10 blocks for given counters and keys (the generator of
// the random term, exposed so its bits can be checked against published
// known-answer vectors).
__global__ void k_philox_raw(long long n, const uint32_t *ctr, const uint32_t *key, uint32_t *out)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint4 c = make_uint4(ctr[4 * i], ctr[4 * i + 1], ctr[4 * i + 2], ctr[4 * i + 3]);
    const uint4 r = philox4x32_10(c, key[2 * i], key[2 * i + 1]);
    out[4 * i] = r.x;
    out[4 * i + 1] = r.y;
    out[4 * i + 2] = r.z;
    out[4 * i + 3] = r.w;
}

void launch_philox_raw(long long n, const uint32_t *ctr, const uint32_t *key, uint32_t *out, cudaStream_t st)
{
    if (n) k_philox_raw<<<nblk(n, 256), 256, 0, st>>>(n, ctr, key, out);
}

void launch_noise_normals(int precision, long long n, const uint32_t *gi, const uint32_t *gj, uint32_t step,
                          uint32_t k0, uint32_t k1, double *out, cudaStream_t st)
{
    if (!n) return;
    if (precision == SDPD_PREC_FP64)
        k_noise_normals<double><<<nblk(n, 256), 256, 0, st>>>(n, gi, gj, step, k0, k1, out);
    else
        k_noise_normals<float><<<nblk(n, 256), 256, 0, st>>>(n, gi, gj, step, k0, k1, out);
}

void launch_absorb(const Bufs &b, int precision, const double *xs, int has_x, cudaStream_t st)
{
    if (!b.N) return;
    const int bs = spread_block(b.N);
    if (precision == SDPD_PREC_SPLIT) k_absorb<float><<<nblk(b.N, bs), bs, 0, st>>>(b, xs, has_x);
    else k_absorb<double><<<nblk(b.N, bs), bs, 0, st>>>(b, xs, has_x);
}

void launch_count_pairs(const Bufs &b, cudaStream_t st)
{
    cudaMemsetAsync(b.pair_count, 0, sizeof(unsigned long long), st);
    if (b.N) k_count_pairs<<<nblk(b.N, 256), 256, 0, st>>>(b);
}

}  // namespace sdpd
