// static_scratch.cu -- sdpd_density_noalloc: number density and pressure of
// one particle set without any device allocation.
//
// Some callers cannot let a library allocate device memory: applications
// whose allocator (for example a framework's caching allocator) owns the
// whole device and forbids foreign cudaMalloc calls, and control loops that
// cannot afford the implicit device-wide synchronisation cudaMalloc and
// cudaFree may cause.  This entry point serves them: its scratch (cell keys,
// slots, counts, starts and cell-ordered records) lives in one file-scope
// __device__ array of fixed size that every GPU loading the library keeps
// until process exit; the caller passes only inputs and outputs.
//
// The paper has no counterpart of this entry point; it computes the same
// quantities as sdpd_build_cells + sdpd_compute_density (Eqs. compdens and
// prtcpres with the kernel normalisation and the optional clamp) for FP64
// positions, without the pressure filter.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <string>

#include "common.cuh"

namespace sdpd {
namespace noalloc {

constexpr int NMAX = SDPD_NOALLOC_MAX_PARTICLES;
constexpr int CMAX = SDPD_NOALLOC_MAX_CELLS;
// layout of the scratch array (ints): key[NMAX] | slot[NMAX] | count[CMAX] |
// start[CMAX + 4] | records[NMAX] of four ints, in cell order
constexpr size_t OFF_KEY = 0, OFF_SLOT = NMAX, OFF_COUNT = 2 * (size_t)NMAX,
                 OFF_START = 2 * (size_t)NMAX + CMAX, OFF_REC = 2 * (size_t)NMAX + 2 * (size_t)CMAX + 4,
                 SCRATCH_INTS = OFF_REC + 4 * (size_t)NMAX;
static_assert(OFF_REC % 4 == 0, "the records are read as int4");

static __device__ __align__(256) int g_scratch[SCRATCH_INTS];

struct Grid {
    double lo[3], cs[3], inv_cs[3], box[3], inv_box[3];
    int hbox[3];                  // high word of box / 2 on periodic axes, else above every finite number's
    int fbox[3];                  // high word of 1.49 box
    int nc[3], periodic[3];
    // fixed-point coordinates of the candidate test: units of window / 2^32,
    // the window a whole fraction of a periodic box and at least 4 r_c wide.
    // The test's lengths are in r_c, so that its FP32 squares suit any r_c
    // (in the caller's units they left FP32's range beyond 1e19 and 1e-19).
    double fix[3];                // 2^32 / window
    float unit[3];                // window / (2^32 r_c)
    float r2_hi;                  // 1, widened past the error of the test
    double two_k, R, R4;          // 2^k, 2^k r_c in [1, 2) and four times it
    double self, norm;            // the weight of r = 0; d = norm x the sum of the weights
    double rc2, mf, inv_dx3, rho0, p0, alpha, beta_p;
    int clamp;
    long long n;
};

// A periodic coordinate folded into [lo, lo + box): the identity for a
// coordinate already inside (x - 0 * box = x exactly), so in-box inputs give
// the same displacements as the context path.
__device__ __forceinline__ double wrap_of(double x, const Grid &G, int a)
{
    if (!G.periodic[a]) return x;
    return x - G.box[a] * floor((x - G.lo[a]) / G.box[a]);
}

// Cell coordinate of a (wrapped) coordinate, clamped into the grid in double
// before the conversion, so that a huge or non-finite value cannot index
// outside it.  On wall axes the clamp is monotone, so two particles closer
// than r_c still fall into the same or adjacent cells.
__device__ __forceinline__ int cell_of(double x, const Grid &G, int a)
{
    const double f = floor((x - G.lo[a]) * G.inv_cs[a]);
    if (!(f >= 0.0)) return 0;   // negative or NaN
    if (f >= (double)(G.nc[a] - 1)) return G.nc[a] - 1;
    return (int)f;
}

__device__ __forceinline__ bool finite3(const double *x)
{
    return isfinite(x[0]) && isfinite(x[1]) && isfinite(x[2]);
}

__global__ void k_na_clear(int *scr, int ncell)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < ncell) scr[OFF_COUNT + c] = 0;
}

__global__ void k_na_count(int *scr, Grid G, const double *x)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= G.n) return;
    const int cx = cell_of(wrap_of(x[3 * i], G, 0), G, 0), cy = cell_of(wrap_of(x[3 * i + 1], G, 1), G, 1),
              cz = cell_of(wrap_of(x[3 * i + 2], G, 2), G, 2);
    const int key = (cz * G.nc[1] + cy) * G.nc[0] + cx;
    scr[OFF_KEY + i] = key;
    scr[OFF_SLOT + i] = atomicAdd(&scr[OFF_COUNT + key], 1);
}

// one block of 1024 threads: exclusive scan of the cell counts
__global__ void k_na_scan(int *scr, int ncell, long long n)
{
    __shared__ int part[1024];
    const int per = (ncell + 1023) / 1024;
    const int b0 = threadIdx.x * per;
    int sum = 0;
    for (int c = b0; c < b0 + per && c < ncell; ++c) sum += scr[OFF_COUNT + c];
    part[threadIdx.x] = sum;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {
        const int v = threadIdx.x >= o ? part[threadIdx.x - o] : 0;
        __syncthreads();
        part[threadIdx.x] += v;
        __syncthreads();
    }
    int run = threadIdx.x ? part[threadIdx.x - 1] : 0;
    for (int c = b0; c < b0 + per && c < ncell; ++c) {
        scr[OFF_START + c] = run;
        run += scr[OFF_COUNT + c];
    }
    if (threadIdx.x == 0) scr[OFF_START + ncell] = (int)n;
}

// Records in cell order: the coordinates in fixed point, modulo a window of at
// least 4 r_c, and the particle's index.  The difference of two such
// coordinates wraps like the minimum image, so the candidate test needs no
// branch on periodic axes, and is off by about 2^-28 r_c for positions in the
// box and by up to 2^-22 r_c for positions on periodic axes within 2^16 boxes
// of it (w below has an error of 2^-52 of its size; the cells' limit leaves an
// axis fewer than 2^11 windows), inside the margin of r2_hi.  A particle
// further out, or outside the grid on a wall axis, passes every candidate test
// (REC_FAR) and the FP64 part decides.  A non-finite position is nobody's
// neighbour: index -1.
constexpr int REC_FAR = 1 << 30;
static_assert(NMAX <= REC_FAR, "the flag bit is above every index");

__device__ __forceinline__ int fixed_of(double x, const Grid &G, int a, bool &far)
{
    const double w = (x - G.lo[a]) * G.fix[a] * 0x1p-32;   // in windows
    const double top = G.periodic[a] ? G.box[a] * 65536.0 : G.nc[a] * G.cs[a];
    far |= !(fabs(x - G.lo[a]) <= top);
    const double f = w - floor(w);                         // [0, 1], whatever the size of the box
    return (int)(unsigned)(unsigned long long)(f * 0x1p32);
}

__global__ void k_na_scatter(int *scr, Grid G, const double *x)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= G.n) return;
    const double xr[3] = { x[3 * i], x[3 * i + 1], x[3 * i + 2] };
    int4 r = make_int4(0, 0, 0, -1);
    if (finite3(xr)) {
        bool far = false;
        r.x = fixed_of(xr[0], G, 0, far);
        r.y = fixed_of(xr[1], G, 1, far);
        r.z = fixed_of(xr[2], G, 2, far);
        r.w = (int)i | (far ? REC_FAR : 0);
    }
    reinterpret_cast<int4 *>(scr + OFF_REC)[scr[OFF_START + scr[OFF_KEY + i]] + scr[OFF_SLOT + i]] = r;
}

// d of every particle, one warp each.  The kernel sum costs about 25 FP64
// instructions a neighbour, and this part issues FP64 at 1/64 of the FP32 rate:
// the FP64 pipe is the bound, so it is given nothing else to do.
//  * Candidates (27 cells, about 1,600 at r_c = 3.9 dx) are tested in fixed
//    point and FP32 from the 16-byte cell-ordered records, 32 at a time and
//    coalesced; x-adjacent cells are one run of records.
//  * The one in six that pass (a superset of the pairs within r_c) are
//    compacted through shared memory, so that all 32 lanes hold a neighbour
//    when the FP64 part runs; it re-decides r < r_c as before.
// One thread per particle over unsorted candidates, each wrapped by an FP64
// division per axis, took 13.4 ms for 46,255 particles; the call now takes
// 0.53 ms (0.82 with the image by a rounded quotient wherever a lane of a warp
// wraps; 0.56 with r / r_c by a reciprocal, whose rounding moved all densities
// one way, 0.58 by a reciprocal in two parts).  Densities are off by 1.4e-16 to
// 2.8e-16 of their value, rms against 113-bit sums at six spacings (5e-16 to
// 1.8e-15 with one thread a particle, the normalisation summed site by site).
constexpr int ND_WARPS = 4;

// `sum` plus the weight of the pair (i, j) where r < r_c.  With t = 2^k (r_c - r),
// one rounding, W is (4 R - 3 t) t^3 of R = 2^k r_c in [1, 2), but for a factor
// that the normalisation divides out: five operations from the root, the last
// of them the addition, and no quotient or reciprocal of r_c to be rounded.
__device__ __forceinline__ double na_add(const Grid &G, const double xi[3], const double *__restrict__ x, int j, double sum)
{
    double r[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        double t = __dsub_rn(xi[a], x[3 * (long long)j + a]);
        // minimum image: in-box coordinates need at most one box length, one
        // subtraction where the high words tell that it is one
        const int ht = hi_abs(t);
        if (ht >= G.hbox[a]) {
            if (ht > G.hbox[a] && ht < G.fbox[a])
                t = __dsub_rn(t, __hiloint2double(__double2hiint(G.box[a]) | (__double2hiint(t) & 0x80000000),
                                                  __double2loint(G.box[a])));
            else
                t = __dsub_rn(t, __dmul_rn(G.box[a], rint(t * G.inv_box[a])));
        }
        r[a] = t;
    }
    const double r2 = __dadd_rn(__dadd_rn(__dmul_rn(r[0], r[0]), __dmul_rn(r[1], r[1])), __dmul_rn(r[2], r[2]));
    if (!lt_pos(r2, G.rc2)) return sum;   // also a NaN
    const double t = fma(-root(r2), G.two_k, G.R);
    return fma(fma(-3.0, t, G.R4), t * t * t, sum);
}

__global__ void __launch_bounds__(ND_WARPS * 32) k_na_density(const int *scr, Grid G, const double *x, const int *type,
                                                             double *d_out)
{
    __shared__ int queue[ND_WARPS][64];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const unsigned FULL = 0xffffffffu, below = (1u << lane) - 1u;
    const int4 *__restrict__ rec = reinterpret_cast<const int4 *>(scr + OFF_REC);
    const int *__restrict__ start = scr + OFF_START;
    const long long s = (long long)blockIdx.x * ND_WARPS + wid;
    if (s >= G.n) return;   // the whole warp
    const int4 me = rec[s];
    if (me.w < 0) return;   // not finite: k_na_pressure writes its NaN
    const int i = me.w & (REC_FAR - 1);
    if (type[i] == T_OUTER) {
        if (lane == 0) d_out[i] = G.inv_dx3;
        return;
    }
    const double xi[3] = { x[3 * (long long)i], x[3 * (long long)i + 1], x[3 * (long long)i + 2] };
    const int key = scr[OFF_KEY + i], c0 = key % G.nc[0], c1 = key / G.nc[0] % G.nc[1], c2 = key / G.nc[0] / G.nc[1];
    int *q = queue[wid];
    int nq = 0;
    double sum = 0.0;
    auto run = [&](int q0, int q1) {
        for (int base = q0; base < q1; base += 32) {
            const int t = base + lane;
            bool hit = false;
            int j = -1;
            if (t < q1) {
                const int4 o = __ldg(rec + t);
                j = o.w & (REC_FAR - 1);
                const float dx = (float)(int)((unsigned)me.x - (unsigned)o.x) * G.unit[0],
                            dy = (float)(int)((unsigned)me.y - (unsigned)o.y) * G.unit[1],
                            dz = (float)(int)((unsigned)me.z - (unsigned)o.z) * G.unit[2];
                hit = o.w >= 0 && j != i && (dx * dx + dy * dy + dz * dz < G.r2_hi || ((me.w | o.w) & REC_FAR));
            }
            const unsigned m = __ballot_sync(FULL, hit);
            if (hit) q[nq + __popc(m & below)] = j;
            nq += __popc(m);
            __syncwarp();
            if (nq >= 32) {
                sum = na_add(G, xi, x, q[lane], sum);
                const int rest = lane < nq - 32 ? q[32 + lane] : 0;
                __syncwarp();
                if (lane < nq - 32) q[lane] = rest;
                nq -= 32;
                __syncwarp();
            }
        }
    };
    for (int oz = -1; oz <= 1; ++oz) {
        int cz = c2 + oz;
        if (G.periodic[2]) cz = cz < 0 ? cz + G.nc[2] : (cz >= G.nc[2] ? cz - G.nc[2] : cz);
        else if (cz < 0 || cz >= G.nc[2]) continue;
        for (int oy = -1; oy <= 1; ++oy) {
            int cy = c1 + oy;
            if (G.periodic[1]) cy = cy < 0 ? cy + G.nc[1] : (cy >= G.nc[1] ? cy - G.nc[1] : cy);
            else if (cy < 0 || cy >= G.nc[1]) continue;
            const int row = (cz * G.nc[1] + cy) * G.nc[0];
            // the x-adjacent cells are consecutive keys: one run of records,
            // and the wrapped cell's own run at the ends of a periodic axis
            const int lo = max(c0 - 1, 0), hi = min(c0 + 1, G.nc[0] - 1);
            run(start[row + lo], start[row + hi + 1]);
            if (G.periodic[0] && c0 == 0) run(start[row + G.nc[0] - 1], start[row + G.nc[0]]);
            if (G.periodic[0] && c0 == G.nc[0] - 1) run(start[row], start[row + 1]);
        }
    }
    if (lane < nq) sum = na_add(G, xi, x, q[lane], sum);
    sum = warp_sum(sum);
    if (lane == 0) d_out[i] = G.norm * (G.self + sum);
}

// The equation of state, one thread per particle (a general power: on one
// lane of the density kernel's warps it would cost as much as the sum).  A
// particle without a position has no density.
__global__ void k_na_pressure(Grid G, const double *x, double *d_out, double *p_out)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= G.n) return;
    const double xr[3] = { x[3 * i], x[3 * i + 1], x[3 * i + 2] };
    if (!finite3(xr)) {
        d_out[i] = NAN;
        p_out[i] = NAN;
        return;
    }
    double p = G.p0 * pow(G.mf * d_out[i] / G.rho0, G.alpha) - G.beta_p;
    if (G.clamp && p < 0.0) p = 0.0;
    p_out[i] = p;
}

// Device address of the scratch array, resolved once per device (with that
// device current) on the first call made on it and kept for the process.  A
// device reset (cudaDeviceReset, or another library resetting the primary
// context) reloads the module and may move the array, so the library must
// not be used across one.
std::mutex g_mu;
int *g_addr[64] = { nullptr };

}  // namespace noalloc
}  // namespace sdpd

namespace {
struct NaErr {
    void operator=(const std::string &m) { sdpd::set_last_error(m.c_str()); }
} g_na_err;

}  // namespace

extern "C" sdpd_status sdpd_density_noalloc(const sdpd_params *p, long long n, const double *x,
                                            const int *type, double *d_out, double *p_out,
                                            void *stream)
{
    using namespace sdpd::noalloc;
    if (!p || n < 0 || (n && (!x || !type || !d_out || !p_out))) {
        g_na_err = "sdpd_density_noalloc: NULL argument or negative count";
        return SDPD_E_INVALID;
    }
    if (n > NMAX) {
        g_na_err = "sdpd_density_noalloc: " + std::to_string(n) + " particles exceed the static scratch limit of " +
                   std::to_string(NMAX);
        return SDPD_E_INVALID;
    }
    if (!(p->dx > 0) || !(p->r_c > 0) || !(p->rho0 > 0)) {
        g_na_err = "sdpd_density_noalloc: dx, r_c, rho0 must be > 0";
        return SDPD_E_INVALID;
    }
    // the kernel normalisation sums W over a lattice of (2 ceil(r_c/dx) + 3)^3
    // sites on the host
    if (!(p->r_c / p->dx <= 32.0)) {
        g_na_err = "sdpd_density_noalloc: r_c / dx must be finite and at most 32";
        return SDPD_E_INVALID;
    }
    Grid G{};
    // every axis: a finite origin, a finite box > 0 and a finite number of
    // cells in [1, CMAX] decided in double before any integer conversion,
    // so that no product of cell counts can overflow or turn negative
    for (int a = 0; a < 3; ++a) {
        if (!std::isfinite(p->origin[a]) || !std::isfinite(p->box[a]) || !(p->box[a] > 0.0) ||
            !std::isfinite(p->r_c) || !std::isfinite(p->dx)) {
            g_na_err = "sdpd_density_noalloc: origin, box, dx and r_c must be finite, box > 0 on every axis";
            return SDPD_E_INVALID;
        }
        G.box[a] = p->box[a];
        G.periodic[a] = p->periodic[a] ? 1 : 0;
        const double ncd = G.periodic[a] ? std::floor(p->box[a] / p->r_c)
                                         : std::ceil((p->box[a] + 4.0 * p->r_c) / p->r_c);
        if (!std::isfinite(ncd) || ncd < (G.periodic[a] ? 3.0 : 1.0)) {
            g_na_err = G.periodic[a] ? "sdpd_density_noalloc: periodic axis narrower than 3 r_c"
                                     : "sdpd_density_noalloc: box / r_c is not a finite positive cell count";
            return SDPD_E_INVALID;
        }
        if (ncd > (double)CMAX) {
            g_na_err = "sdpd_density_noalloc: " + std::to_string((long long)ncd) + " cells along axis " +
                       std::to_string(a) + " exceed the static scratch limit of " + std::to_string(CMAX);
            return SDPD_E_INVALID;
        }
        G.nc[a] = (int)ncd;
        if (G.periodic[a]) {
            G.cs[a] = p->box[a] / G.nc[a];
            G.lo[a] = p->origin[a];
        } else {
            // the fluid region plus two kernel radii of dummy-particle layers;
            // particles beyond are clamped into the boundary cells (still exact)
            G.cs[a] = p->r_c;
            G.lo[a] = p->origin[a] - 2.0 * p->r_c;
        }
        G.inv_cs[a] = 1.0 / G.cs[a];
    }
    const long long ncell = (long long)G.nc[0] * G.nc[1] * G.nc[2];   // each factor <= CMAX
    if (ncell > CMAX) {
        g_na_err = "sdpd_density_noalloc: " + std::to_string(ncell) + " cells exceed the static scratch limit of " +
                   std::to_string(CMAX);
        return SDPD_E_INVALID;
    }
    const double h = p->r_c;
    G.rc2 = h * h;
    int ex = 0;
    G.R = 2.0 * std::frexp(h, &ex);
    G.two_k = std::ldexp(1.0, 1 - ex);
    G.R4 = 4.0 * G.R;
    for (int a = 0; a < 3; ++a) {
        // a periodic box is a whole number of windows (the fixed-point
        // coordinates wrap with it); a box below 8 r_c is one window
        const double k = std::max(1.0, std::floor(G.box[a] / (4.0 * h)));
        const double window = G.periodic[a] ? G.box[a] / k : 4.0 * h;
        G.fix[a] = 4294967296.0 / window;
        G.unit[a] = (float)(window / h / 4294967296.0);
        G.inv_box[a] = 1.0 / G.box[a];
        const double hb = 0.5 * G.box[a];
        unsigned long long bits;
        std::memcpy(&bits, &hb, sizeof hb);
        G.hbox[a] = G.periodic[a] ? (int)(bits >> 32) : 0x7FFFFFFF;
        const double fb = 1.49 * G.box[a];
        std::memcpy(&bits, &fb, sizeof fb);
        G.fbox[a] = (int)(bits >> 32);
    }
    // FP32 products of fixed-point differences: relative error of r^2 below 1e-6
    G.r2_hi = 1.0f + 1e-5f;
    // the normalisation: the weights of a perfect lattice, self included, sum to
    // 1 / (norm dx^3).  Sums of rows of planes: rounded a dozen times on the way,
    // not once a site.
    auto weight = [&](double r) {
        if (r >= h) return 0.0;
        const double t = std::fma(-r, G.two_k, G.R);
        return std::fma(-3.0, t, G.R4) * (t * t * t);
    };
    const int m = (int)std::ceil(h / p->dx) + 1;
    double lat = 0.0;
    for (int k = -m; k <= m; ++k) {
        double plane = 0.0;
        for (int j = -m; j <= m; ++j) {
            double row = 0.0;
            for (int i = -m; i <= m; ++i) row += weight(std::sqrt((double)(i * i + j * j + k * k)) * p->dx);
            plane += row;
        }
        lat += plane;
    }
    G.norm = 1.0 / (p->dx * p->dx * p->dx * lat);
    G.self = weight(0.0);
    G.mf = p->rho0 * p->dx * p->dx * p->dx;
    G.inv_dx3 = 1.0 / (p->dx * p->dx * p->dx);
    G.rho0 = p->rho0;
    G.p0 = p->p0;
    G.alpha = p->alpha;
    G.beta_p = p->beta_p;
    G.clamp = p->clamp_negative_p ? 1 : 0;
    G.n = n;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
        g_na_err = "sdpd_density_noalloc: no current CUDA device";
        return SDPD_E_CUDA;
    }
    int *scr = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_mu);
        if (!g_addr[dev]) {
            void *ptr = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&ptr, g_scratch);
            if (e != cudaSuccess) {
                g_na_err = std::string("sdpd_density_noalloc: cudaGetSymbolAddress: ") + cudaGetErrorString(e);
                return SDPD_E_CUDA;
            }
            g_addr[dev] = (int *)ptr;
        }
        scr = g_addr[dev];
    }
    if (n == 0) return SDPD_OK;
    cudaStream_t st = (cudaStream_t)stream;
    (void)cudaGetLastError();
    const int nc_i = (int)ncell;
    k_na_clear<<<(nc_i + 255) / 256, 256, 0, st>>>(scr, nc_i);
    k_na_count<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(scr, G, x);
    k_na_scan<<<1, 1024, 0, st>>>(scr, nc_i, n);
    k_na_scatter<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(scr, G, x);
    k_na_density<<<(unsigned)((n + ND_WARPS - 1) / ND_WARPS), ND_WARPS * 32, 0, st>>>(scr, G, x, type, d_out);
    k_na_pressure<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(G, x, d_out, p_out);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        g_na_err = std::string("sdpd_density_noalloc: launch: ") + cudaGetErrorString(e);
        return SDPD_E_CUDA;
    }
    return SDPD_OK;
}
