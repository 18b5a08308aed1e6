// k_cells.cu -- compute_neighbor_list (Algorithm 1, Section 3.2) on the GPU.
//
// The paper's background grid with linked lists is replaced by a counting
// sort of the particles into Morton-ranked cells:
//   K1 cell key per particle + atomic per-cell count      (HBM bound, 1 pass)
//   K2 exclusive scan of the counts -> cell starts
//   K3 scatter into cell ranges, K4 rank by gid inside each cell (deterministic
//      order, so every later sum is reproducible bit for bit)
//   K5 gather of the cell-sorted mirrors (float4 / double4 records)
//   K6 per particle, the list of neighbours j != i within the build
//      radius rb = h (1 + skin) from the surrounding cells
//   K7 reverse index of the Newton-3 force pass
// The list is a superset of the pairs within h; every consumer re-decides
// r_ij < h exactly, so the evaluated pair set equals the paper's.  The list
// stays valid while no particle has moved more than skin h / 2 since the
// build; the drift raises `need_build` when one has and opens the conditional
// node of the captured step that holds these kernels (a build enqueued after
// an upload has the flag as its gate instead).  Only the instances whose
// own flag is up are rebuilt: an instance's slots are the range of its gids,
// so the others keep their cells, slots and lists.
#include <algorithm>

#include "common.cuh"

namespace sdpd {

#define GATE                                                                                    \
    if (gate && *gate == 0) return;

__device__ __forceinline__ int cell_coord(double x, double lo, double inv_cs, int nc, bool &out, bool &nonfinite)
{
    const double f = floor((x - lo) * inv_cs);
    nonfinite = !(fabs(f) < 1e9);   // NaN or a runaway coordinate
    const int k = nonfinite ? 0 : (int)f;
    out = (k < 0) || (k >= nc);
    return k < 0 ? 0 : (k >= nc ? nc - 1 : k);
}

__global__ void k_cell_clear(Bufs b, const int *gate)
{
    GATE;
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    if (c < b.ncell_total && rebuilds(b, gate, b.cell_inst[c])) b.ccount[c] = 0;
}

__global__ void k_cell_keys(Bufs b, const int *gate)
{
    GATE;
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= b.N || !rebuilds(b, gate, b.pinst[g])) return;
    const Inst &I = b.inst[b.pinst[g]];
    int c[3];
    bool bad = false, nf = false;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        bool o, f;
        c[a] = cell_coord(b.x[3 * g + a], I.lo[a], I.inv_cs[a], I.nc[a], o, f);
        bad |= o;
        nf |= f;
    }
    if (nf) atomicOr(b.err, ERR_NONFINITE);
    else if (bad) atomicOr(b.err, ERR_DOMAIN);
    const int lin = (c[2] * I.nc[1] + c[1]) * I.nc[0] + c[0];
    const int key = I.cell_base + b.cell_rank[I.cell_base + lin];
    b.key[g] = key;
    b.slot_in_cell[g] = atomicAdd(&b.ccount[key], 1);
}

// --- exclusive scan of the cell counts (three phases, 1024 cells per block)
__device__ __forceinline__ int warp_incl_scan(int v)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) >= o) v += t;
    }
    return v;
}

__device__ int block_excl_scan(int v, int *total)
{
    __shared__ int ws[32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int inc = warp_incl_scan(v);
    if (lane == 31) ws[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        int s = (lane < (int)(blockDim.x >> 5)) ? ws[lane] : 0;
        s = warp_incl_scan(s);
        ws[lane] = s;
    }
    __syncthreads();
    const int off = wid ? ws[wid - 1] : 0;
    *total = ws[(blockDim.x >> 5) - 1];
    __syncthreads();
    return off + inc - v;
}

__global__ void k_scan_local(Bufs b, const int *gate)
{
    GATE;
    const int n = b.ncell_total;
    const int i = blockIdx.x * 1024 + threadIdx.x;
    const int v = i < n ? b.ccount[i] : 0;
    int tot;
    const int e = block_excl_scan(v, &tot);
    if (i < n) b.cstart[i] = e;
    if (threadIdx.x == 0) b.scan_partials[blockIdx.x] = tot;
}

__global__ void k_scan_partials(Bufs b, int nblk, const int *gate)
{
    GATE;
    // one block of 1024 threads, sequential over chunks
    int carry = 0;
    for (int base = 0; base < nblk; base += 1024) {
        const int i = base + threadIdx.x;
        const int v = i < nblk ? b.scan_partials[i] : 0;
        int tot;
        const int e = block_excl_scan(v, &tot);
        if (i < nblk) b.scan_partials[i] = carry + e;
        carry += tot;
        __syncthreads();
    }
}

__global__ void k_scan_add(Bufs b, const int *gate)
{
    GATE;
    const int n = b.ncell_total;
    const int i = blockIdx.x * 1024 + threadIdx.x;
    if (i < n) b.cstart[i] += b.scan_partials[blockIdx.x];
    if (i == 0) b.cstart[n] = (int)b.N;
}

__global__ void k_scatter(Bufs b, const int *gate)
{
    GATE;
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= b.N || !rebuilds(b, gate, b.pinst[g])) return;
    b.tmp_perm[b.cstart[b.key[g]] + b.slot_in_cell[g]] = (int)g;
}

// Rank of each particle among its cell's members by gid (stable, unique).
__global__ void k_rank(Bufs b, const int *gate)
{
    GATE;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= b.N) return;
    const int g = b.tmp_perm[t];   // (of the last build where this one leaves the instance as it is)
    if (!rebuilds(b, gate, b.pinst[g])) return;
    const int c = b.key[g];
    const int s0 = b.cstart[c], s1 = b.cstart[c + 1];
    int r = 0;
    for (int u = s0; u < s1; ++u) r += (b.tmp_perm[u] < g);
    b.perm[s0 + r] = g;
    b.slot_of[g] = s0 + r;
}

// Cell-sorted mirrors for the pair kernels; displacements count from here.
__global__ void k_gather(Bufs b, int precision, const int *gate)
{
    GATE;
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= b.N) return;
    const int g = b.perm[s];
    const int ii = b.pinst[g];
    if (!rebuilds(b, gate, ii)) return;
    const Inst &I = b.inst[ii];
    const int t = b.type[g];
    b.stype[s] = t;
    const double x0 = b.x[3 * g], x1 = b.x[3 * g + 1], x2 = b.x[3 * g + 2];
    const uint32_t lg = (uint32_t)(g - I.p_begin);
    // (both precisions: the neighbour search and the split-precision pair
    // kernels work on the fixed-point coordinates)
    b.A32[s] = b.A32_build[s] = make_int4(fixed_coord(x0, I, 0), fixed_coord(x1, I, 1), fixed_coord(x2, I, 2), t);
    if (precision == SDPD_PREC_SPLIT) {
        b.B32[s] = make_float4((float)b.v[3 * g], (float)b.v[3 * g + 1], (float)b.v[3 * g + 2],
                               (float)b.R[g]);
        b.C32[s] = make_float4((float)b.w[3 * g], (float)b.w[3 * g + 1], (float)b.w[3 * g + 2],
                               (float)b.m[g]);
        b.D32[s].w = __uint_as_float(lg);
    } else {
        b.A64[s] = make_double4_32a(x0, x1, x2, __longlong_as_double(t));
        b.B64[s] = make_double4_32a(b.v[3 * g], b.v[3 * g + 1], b.v[3 * g + 2], b.R[g]);
        b.C64[s] = make_double4_32a(b.w[3 * g], b.w[3 * g + 1], b.w[3 * g + 2], b.m[g]);
        b.D64[s].w = __longlong_as_double((long long)lg);
    }
}

// Neighbour list of particle (slot) s: candidates from the cells around s's
// cell (cells are at least max(rb, largest sphere diameter + skin) / sub
// wide and the stencil reaches sub cells each way, sub = 1 or 2; periodic
// axes at least 2 sub + 1 cells).  A pair is listed when r < rb (float test:
// the list only has to be a superset of the pairs within h), or when both are
// rigid and r < R_i + R_j + skin h (contact range; flagged NB_FAR).
//
// In FP32 contexts with a direct force pass (b.split == 0) the list is
// ascending in slot.  Otherwise it is split by Newton-3 ownership, balanced so that every particle owns about half of its
// pairs whatever its position in the cell: the pair of instance-local slots
// a < b belongs to a when bit 15 of the hash (a * 0x9E3779B1) ^
// (b * 0x85EBCA77) is set, else to b.  The list is written as [owned][not
// owned], the owned part ascending in slot (cells visited in ascending key),
// the other descending, so the owned pairs are the prefix [0, nfirst) and a
// partner's position is found by binary search in it.
__device__ __forceinline__ bool pair_owned(long long s, int j, int base)
{
    // instance-local slots: an instance owns the same pairs alone or batched
    const uint32_t lo = (uint32_t)(min((long long)j, s) - base), hi = (uint32_t)(max((long long)j, s) - base);
    const uint32_t h = (lo * 0x9E3779B1u) ^ (hi * 0x85EBCA77u);
    const bool low_owns = (h >> 15) & 1u;
    return low_owns == (s < j);
}


// The candidate test of a pair (i, j) with j's record Aj: within rb (float),
// or both rigid and within contact range (flagged NB_FAR).
__device__ __forceinline__ bool nb_test(const Bufs &b, const Inst &I, const Geo<float> &geo, const int4 &Ai, int ti,
                                        float Ri, int j, const int4 &Aj, uint32_t &entry, int &tj)
{
    tj = Aj.w;
    float dx, dy, dz;
    geo.disp(Ai, Aj, dx, dy, dz);
    const float r2f = dx * dx + dy * dy + dz * dz;
    entry = (uint32_t)j;
    if (r2f < I.rb2f) return true;
    if (ti == T_RIGID && tj == T_RIGID) {
        const float lim = (Ri + (float)b.R[b.perm[j]] + (float)(2.0 * I.half_skin)) * 1.0001f;
        entry |= NB_FAR;
        return r2f < lim * lim;
    }
    return false;
}

// The fallback for cells with a crowded neighbour (below): one lane per
// particle, 32 at a time, every lane testing the same candidates, which are
// staged 32 at a time in shared memory and visited in ascending order.
// The lists of cell c's particles [s0, s1), one lane per particle; stage:
// 32 int4 of this warp's shared memory.
__device__ void nb_scan_cell(const Bufs &b, int c, int s0, int s1, int4 *stage, int lane)
{
    const int *adj = b.cell_adj + (long long)c * ADJ;
    const Inst &I = b.inst[b.pinst[b.perm[s0]]];   // a cell belongs to one instance
    const int base = b.cstart[I.cell_base];           // first slot of the instance
    const int rows = b.rows;
    const int cap = b.cap;
    const bool split = b.split != 0;
    const Geo<float> geo(I);
    for (int chunk = s0; chunk < s1; chunk += 32) {
        const int s = chunk + lane;
        const bool act = s < s1;
        int ti = T_FLUID;
        float Ri = 0.f;
        int4 Ai = make_int4(0, 0, 0, 0);
        if (act) {
            ti = b.stype[s];
            Ri = (ti == T_RIGID) ? (float)b.R[b.perm[s]] : 0.f;
            Ai = b.A32[s];
        }
        auto col = [&](int k) -> int & { return b.nbr[entry_at(k, s, rows)]; };   // this particle's column
        // one scan in ascending slot order: owned pairs from the front, the
        // others from the back of the column (so in descending positions)
        int nf = 0, m = 0;
        bool rig = false;
        for (int q = 0; q < ADJ; ++q) {
            const int key = adj[q];
            if (key < 0) break;
            const int j0 = b.cstart[key], j1 = b.cstart[key + 1];
            for (int jb = j0; jb < j1; jb += 32) {
                const int jj = jb + lane;
                __syncwarp();
                stage[lane] = jj < j1 ? b.A32[jj] : make_int4(0, 0, 0, 0);
                __syncwarp();
                if (!act) continue;
                const int cnt = min(32, j1 - jb);
                for (int t = 0; t < cnt; ++t) {
                    const int j = jb + t;
                    uint32_t entry;
                    int tj;
                    if (j == s || !nb_test(b, I, geo, Ai, ti, Ri, j, stage[t], entry, tj)) continue;
                    rig |= (tj == T_RIGID);
                    if (!split || pair_owned(s, j, base)) {
                        if (nf + m < cap) col(nf) = (int)entry;
                        ++nf;
                    } else {
                        if (nf + m < cap) col(cap - 1 - m) = (int)entry;
                        ++m;
                    }
                }
            }
        }
        if (!act) continue;
        const int n = nf + m;
        // the pair buffer holds capown rows of owned and of non-owned entries
        if (split && (nf > b.capown || m > b.capown)) atomicOr(b.err, ERR_PAIR_CAP);
        if (n > cap) {
            atomicOr(b.err, ERR_NBR_CAP);
        } else {
            // the back region [cap - m, cap) holds the non-owned entries in
            // descending slot order: move it down to [nf, n) as it is
            // (destination below the source, so an ascending copy never
            // overwrites an entry still to be read); only the owned prefix
            // needs ascending order (the reverse index searches it)
            if (nf < cap - m)
                for (int k = 0; k < m; ++k) col(nf + k) = col(cap - m + k);
        }
        b.nfirst[s] = min(nf, split ? min(cap, b.capown) : cap);
        b.ncnt[s] = min(n, cap);
        b.nbflag[s] = rig ? 1 : 0;
    }
}

// The lists: lanes are candidates.  `parts` warps share a cell, each taking
// every parts-th group of NG_G of its particles.  A warp is a block of its own:
// latency bounds the scan, shared memory (9 KB a warp) the warps on an SM, and
// in a block of four the memory of those that are done, or had no group, stayed
// taken until the last one was (374,000 particles: 811 us a build in blocks of
// four, 647 in blocks of one with the records of a batch fetched a batch ahead;
// 662,000: 1.58 -> 1.43 ms).  A warp flattens the
// candidates of the cell's neighbour cells (ascending key, then slot; cells
// whose slots follow one another are one run).  For each group:
// * Every batch of 32 candidates is tested against the group's bounding box,
//   widened to the list radius: about 40 % of the 27-cell stencil of full
//   cells survives, about half of the 125-cell stencil of half cells.
// * The survivors are compacted in order into a staging area.
// * Each full stage of 32 runs one round per particle of the group: every
//   lane tests its candidate against that particle. Ballots place the hits in
//   scan order.
// * The group's lists are collected in shared memory as 16-bit entries (the
//   run, the offset in it, the contact-only flag): in FP32 direct contexts in
//   order, else owned entries from the front and the others from the back.
// * The lists are then written out LPP entries of a particle at a time, four
//   particles side by side, instead of one scattered entry per lane.
// A cell with a crowded neighbour cell (beyond the offsets of the entries) is
// scanned by the lane-per-particle routine above instead, which writes the
// same lists: the same entries in the same order, the same counts and flags.
// Full cells were once scanned by that routine alone, one warp for a cell of
// some 70 particles: 2.9 ms for 8,192 particles (128 warps on the chip), 0.1
// ms by this one.
constexpr int NG_G = 8;        // particles per group
constexpr int NG_TAB = 128;    // runs (>= ADJ)
constexpr int NG_STAGE = 64;   // staged candidates (one batch on top of a partial stage)

// 16-bit entries: offset bits, and the largest neighbour cell; a run never
// exceeds twice that (it is cut where the flattened index passes a multiple).
// Full cells: up to 27 runs of 1,024; half cells: up to 125 runs of 256.
template <int SUB> struct NgEntry {
    static constexpr int BITS = SUB == 1 ? 10 : 8;
    static constexpr int CELL = 1 << (BITS - 1);
};

struct NgShared {
    int4 sa[NG_STAGE];         // staged candidates: record,
    int sj[NG_STAGE];          //   slot,
    float sr[NG_STAGE];        //   radius where it can be a contact partner, else 0
    int sq[NG_STAGE];          //   16-bit entry
    int pre[NG_TAB + 1];       // candidates before each run (flattened index)
    int js[NG_TAB];            // first slot of each run
    int4 ai[NG_G];             // the group's records,
    float ri[NG_G];            //   rigid radii
};

// list-buffer row stride (16-bit entries): stride % 64 == 8 puts the rows
// of consecutive particles 16 bytes (4 banks) apart
__host__ __device__ constexpr int ng_stride(int cap) { return cap + ((72 - cap % 64) % 64); }
__host__ __device__ constexpr size_t ng_head() { return (sizeof(NgShared) + 15) / 16 * 16; }
__host__ __device__ constexpr size_t ng_warp_bytes(int cap)
{
    return ng_head() + (size_t)NG_G * ng_stride(cap) * sizeof(uint16_t);
}

template <int SUB, bool SPLIT>
__global__ void __launch_bounds__(32, 24) k_neighbors(Bufs b, int parts, const int *gate)
{
    GATE;
    constexpr int BITS = NgEntry<SUB>::BITS, CELL = NgEntry<SUB>::CELL;
    constexpr int NADJ = (2 * SUB + 1) * (2 * SUB + 1) * (2 * SUB + 1);
    extern __shared__ __align__(16) unsigned char ng_smem[];
    const int lane = threadIdx.x;
    const int c = blockIdx.x / parts, part = blockIdx.x % parts;
    if (!rebuilds(b, gate, b.cell_inst[c])) return;
    const int s0 = b.cstart[c], s1 = b.cstart[c + 1];
    if (s0 + part * NG_G >= s1) return;
    const int cap = b.cap, stride = ng_stride(cap);
    NgShared &S = *reinterpret_cast<NgShared *>(ng_smem);
    uint16_t *buf = reinterpret_cast<uint16_t *>(ng_smem + ng_head());
    const unsigned FULL = 0xffffffffu, lt = (1u << lane) - 1u;

    // the runs of the neighbour cells (valid keys are a prefix of the row)
    const int *adj = b.cell_adj + (long long)c * ADJ;
    int total = 0, nq = 0, last_end = -1, last_bucket = 0;
    bool fat = false;
    // (all the loads of the chain key -> start first: one latency, not one
    // for each 32 cells)
    constexpr int NQ = (NADJ + 31) / 32;
    int qkey[NQ], qjs[NQ], qend[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) qkey[q] = q * 32 + lane < NADJ ? adj[q * 32 + lane] : -1;
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        qjs[q] = qkey[q] >= 0 ? b.cstart[qkey[q]] : 0;
        qend[q] = qkey[q] >= 0 ? b.cstart[qkey[q] + 1] : 0;
    }
#pragma unroll
    for (int q0 = 0; q0 < NQ; ++q0) {
        const int key = qkey[q0], js = qjs[q0], cnt = qend[q0] - js;
        fat = fat || __any_sync(FULL, cnt > CELL);
        int v = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(FULL, v, o);
            if (lane >= o) v += t;
        }
        const int first = total + v - cnt, bucket = first / CELL;
        // the filled cell before this one: where it ended
        const unsigned filled = __ballot_sync(FULL, cnt > 0), before = filled & lt;
        const int src = before ? 31 - __clz(before) : 0;
        int pe = __shfl_sync(FULL, js + cnt, src), pb = __shfl_sync(FULL, bucket, src);
        if (!before) {
            pe = last_end;
            pb = last_bucket;
        }
        const unsigned starts = __ballot_sync(FULL, cnt > 0 && (js != pe || bucket != pb));
        if ((starts >> lane) & 1u) {
            const int r = nq + __popc(starts & lt);
            S.pre[r] = first;
            S.js[r] = js;
        }
        nq += __popc(starts);
        total += __shfl_sync(FULL, v, 31);
        if (filled) {
            const int l = 31 - __clz(filled);
            last_end = __shfl_sync(FULL, js + cnt, l);
            last_bucket = __shfl_sync(FULL, bucket, l);
        }
        if (__ballot_sync(FULL, key >= 0) != FULL) break;
    }
    if (fat) {
        // the staging records, idle here, serve as the routine's stage (the list
        // buffer is smaller than 32 records for capacities up to 8)
        static_assert(NG_STAGE >= 32, "the routine stages 32 records");
        if (part == 0) nb_scan_cell(b, c, s0, s1, S.sa, lane);
        return;
    }
    if (lane == 0) S.pre[nq] = total;
    __syncwarp();

    const Inst &I = b.inst[b.cell_inst[c]];   // a cell belongs to one instance
    const int base = b.cstart[I.cell_base];   // first slot of the instance
    const int rows = b.rows;
    const float rb2 = I.rb2f, rb2_box = rb2 * 1.001f;   // conservative: the pair test decides
    const float two_hs = (float)(2.0 * I.half_skin);
    const Geo<float> geo(I);
    const float BIG = 3.0e38f;

    for (int g0 = s0 + part * NG_G; g0 < s1; g0 += parts * NG_G) {
        const int P = min(NG_G, s1 - g0);
        int4 a = make_int4(0, 0, 0, 0);
        int t = T_FLUID;
        float r = 0.f;
        if (lane < P) {
            a = b.A32[g0 + lane];
            t = a.w;
            r = (t == T_RIGID) ? (float)b.R[b.perm[g0 + lane]] : 0.f;
            S.ai[lane] = a;
            S.ri[lane] = r;
        }
        // the group's bounding box, relative to its first particle (all in one cell)
        const int4 ref = make_int4(__shfl_sync(FULL, a.x, 0), __shfl_sync(FULL, a.y, 0), __shfl_sync(FULL, a.z, 0), 0);
        float ax, ay, az;
        geo.disp(a, ref, ax, ay, az);
        float lx = lane < P ? ax : BIG, ly = lane < P ? ay : BIG, lz = lane < P ? az : BIG;
        float hx = lane < P ? ax : -BIG, hy = lane < P ? ay : -BIG, hz = lane < P ? az : -BIG;
        float rg = r;
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {   // lanes >= NG_G hold the neutral values
            lx = fminf(lx, __shfl_xor_sync(FULL, lx, o));
            ly = fminf(ly, __shfl_xor_sync(FULL, ly, o));
            lz = fminf(lz, __shfl_xor_sync(FULL, lz, o));
            hx = fmaxf(hx, __shfl_xor_sync(FULL, hx, o));
            hy = fmaxf(hy, __shfl_xor_sync(FULL, hy, o));
            hz = fmaxf(hz, __shfl_xor_sync(FULL, hz, o));
            rg = fmaxf(rg, __shfl_xor_sync(FULL, rg, o));
        }
        lx = __shfl_sync(FULL, lx, 0); ly = __shfl_sync(FULL, ly, 0); lz = __shfl_sync(FULL, lz, 0);
        hx = __shfl_sync(FULL, hx, 0); hy = __shfl_sync(FULL, hy, 0); hz = __shfl_sync(FULL, hz, 0);
        rg = __shfl_sync(FULL, rg, 0);
        // its centre and half widths: the wrapping difference to the centre is
        // the image of a candidate nearest to the box, also where a periodic
        // axis holds only three cells
        const float bx = 0.5f * (hx - lx), by = 0.5f * (hy - ly), bz = 0.5f * (hz - lz);
        const int4 mid = make_int4((int)((unsigned)ref.x + (unsigned)__float2int_rn(0.5f * (lx + hx) / geo.u0)),
                                   (int)((unsigned)ref.y + (unsigned)__float2int_rn(0.5f * (ly + hy) / geo.u1)),
                                   (int)((unsigned)ref.z + (unsigned)__float2int_rn(0.5f * (lz + hz) / geo.u2)), 0);
        const bool grp_rigid = __any_sync(FULL, lane < P && t == T_RIGID);
        __syncwarp();

        // nf: entries (SPLIT: owned ones), m: not owned ones, rig: any sphere
        int nf[NG_G], m[NG_G];
        unsigned rig = 0;
#pragma unroll
        for (int p = 0; p < NG_G; ++p) { nf[p] = 0; m[p] = 0; }

        // one round per particle over the first nv staged candidates
        auto rounds = [&](int nv) {
            int4 Aj = make_int4(0, 0, 0, T_FLUID);
            int j = -1;
            uint32_t e16 = 0;
            float rj = 0.f;
            if (lane < nv) {
                Aj = S.sa[lane];
                j = S.sj[lane];
                rj = S.sr[lane];
                e16 = (uint32_t)S.sq[lane];
            }
            const unsigned valid = nv >= 32 ? FULL : (1u << nv) - 1u;
            const bool rigid_j = Aj.w == T_RIGID;
            const unsigned mrig = __ballot_sync(FULL, rigid_j);
#pragma unroll
            for (int p = 0; p < NG_G; ++p) {
                if (p < P) {
                    const int4 Ai = S.ai[p];
                    const int s = g0 + p;
                    uint32_t entry = e16;
                    float dx, dy, dz;
                    geo.disp(Ai, Aj, dx, dy, dz);
                    const float r2f = dx * dx + dy * dy + dz * dz;
                    bool hit = r2f < rb2 && j != s;
                    if (grp_rigid && Ai.w == T_RIGID && rigid_j && !hit && j != s) {
                        const float lim = (S.ri[p] + rj + two_hs) * 1.0001f;
                        entry |= 0x8000u;   // contact range only
                        hit = r2f < lim * lim;
                    }
                    const unsigned mh = __ballot_sync(FULL, hit) & valid;
                    if (!SPLIT) {
                        const int pos = nf[p] + __popc(mh & lt);
                        if (((mh >> lane) & 1u) && pos < cap) buf[p * stride + pos] = (uint16_t)entry;
                        nf[p] += __popc(mh);
                    } else {
                        const unsigned mo = __ballot_sync(FULL, pair_owned(s, j, base)) & mh;
                        // rank in scan order decides whether the entry fits, as
                        // the per-particle scan writes while nf + m < cap
                        if (((mh >> lane) & 1u) && nf[p] + m[p] + __popc(mh & lt) < cap) {
                            const int pos = ((mo >> lane) & 1u) ? nf[p] + __popc(mo & lt)
                                                               : cap - 1 - (m[p] + __popc(mh & ~mo & lt));
                            buf[p * stride + pos] = (uint16_t)entry;
                        }
                        nf[p] += __popc(mo);
                        m[p] += __popc(mh & ~mo);
                    }
                    if (mh & mrig) rig |= 1u << p;
                }
            }
            __syncwarp();
        };

        int nst = 0, qc = 0;   // staged candidates; the run of the batch's first candidate
        // the records of a batch are fetched while the one before it is tested
        int4 An = make_int4(0, 0, 0, 0);
        int jn = 0, en = 0;
        auto fetch = [&](int f0) {
            const int f = f0 + lane;
            // the runs that begin inside this batch, as bits at their first
            // candidate (runs are not empty: at most one begins at a place)
            int nx = qc + 1 + lane < nq ? S.pre[qc + 1 + lane] - f0 : 32;
            const unsigned begin = __reduce_or_sync(FULL, nx < 32 ? 1u << nx : 0u);
            const int q = qc + __popc(begin & (lt | (1u << lane)));
            if (f < total) {
                const int off = f - S.pre[q];
                jn = S.js[q] + off;
                en = (q << BITS) | off;
                An = b.A32[jn];
            }
            qc += __popc(begin);
        };
        if (total > 0) fetch(0);
        for (int f0 = 0; f0 < total; f0 += 32) {
            const int4 Aj = An;
            const int j = jn, eq = en;
            if (f0 + 32 < total) fetch(f0 + 32);
            bool keep = false;
            float rj = 0.f;
            if (f0 + lane < total) {
                float px, py, pz;
                geo.disp(Aj, mid, px, py, pz);
                const float ex = fmaxf(fabsf(px) - bx, 0.f), ey = fmaxf(fabsf(py) - by, 0.f),
                            ez = fmaxf(fabsf(pz) - bz, 0.f);
                const float d2 = ex * ex + ey * ey + ez * ez;
                float lim2 = rb2_box;
                if (grp_rigid && Aj.w == T_RIGID) {
                    rj = (float)b.R[b.perm[j]];
                    const float L = (rg + rj + two_hs) * (1.0001f * 1.0005f);
                    lim2 = fmaxf(lim2, L * L);
                }
                keep = d2 < lim2;
            }
            const unsigned km = __ballot_sync(FULL, keep);
            if (keep) {
                const int pos = nst + __popc(km & lt);
                S.sa[pos] = Aj;
                S.sj[pos] = j;
                S.sq[pos] = eq;
                S.sr[pos] = rj;
            }
            nst += __popc(km);
            __syncwarp();
            if (nst >= 32) {
                rounds(32);
                // move the remainder to the front of the stage
                const bool mv = lane < nst - 32;
                int4 ma;
                int mj = 0, mq = 0;
                float mr = 0.f;
                if (mv) {
                    ma = S.sa[32 + lane];
                    mj = S.sj[32 + lane];
                    mq = S.sq[32 + lane];
                    mr = S.sr[32 + lane];
                }
                __syncwarp();
                if (mv) {
                    S.sa[lane] = ma;
                    S.sj[lane] = mj;
                    S.sq[lane] = mq;
                    S.sr[lane] = mr;
                }
                nst -= 32;
                __syncwarp();
            }
        }
        if (nst > 0) rounds(nst);

        // counts and flags of the group's particles
        int mynf = 0, mym = 0;
#pragma unroll
        for (int p = 0; p < NG_G; ++p)
            if (lane == p) { mynf = nf[p]; mym = m[p]; }
        int myn = 0;
        if (lane < P) {
            const int s = g0 + lane;
            myn = mynf + mym;
            if (SPLIT && (mynf > b.capown || mym > b.capown)) atomicOr(b.err, ERR_PAIR_CAP);
            if (myn > cap) atomicOr(b.err, ERR_NBR_CAP);
            b.nfirst[s] = min(mynf, SPLIT ? min(cap, b.capown) : cap);
            b.ncnt[s] = min(myn, cap);
            b.nbflag[s] = (rig >> lane) & 1u;
        }
        const int maxn = __reduce_max_sync(FULL, lane < P ? min(myn, cap) : 0);
        // write-out: LPP lanes a particle, GROUP particles side by side; without
        // overflow the back region [cap - m, cap) moves down to [nf, n) as it is
        for (int p0 = 0; p0 < P; p0 += GROUP) {
            const int p = p0 + lane / LPP;   // < NG_G: the shuffles below stay in range
            const int pnf = __shfl_sync(FULL, mynf, p), pm = __shfl_sync(FULL, mym, p);
            const int pn = pnf + pm, pcnt = p < P ? min(pn, cap) : 0;
            int *out = b.nbr + entry_at(lane % LPP, g0 + p, rows);
            for (int k = lane % LPP; k < maxn; k += LPP, out += ROW) {
                if (k < pcnt) {
                    const int src = (!SPLIT || pn > cap || k < pnf) ? k : cap - pm + (k - pnf);
                    const uint32_t e = buf[p * stride + src];
                    const int slot = S.js[(e & 0x7FFFu) >> BITS] + (int)(e & ((1u << BITS) - 1u));
                    *out = (int)((uint32_t)slot | ((e & 0x8000u) ? NB_FAR : 0u));
                }
            }
        }
        __syncwarp();
    }
}

// For every non-owned entry k of s (positions [nfirst, n)), the position r
// of s in the partner j's owned prefix (ascending), by binary search; LPP
// lanes share a list and four searches of a lane run interleaved so their
// loads overlap.  Both directions are kept, in disjoint entries of rev:
// rev[k of s] = r (where s reads j's result in j's column) and rev[r of j] =
// k - nfirst(s) (where j writes its result in s's column); each owned entry
// of j gets exactly one.
__device__ __forceinline__ int nb_at(const Bufs &b, int i, int k)
{
    return (int)((uint32_t)__ldg(b.nbr + entry_at(k, i, b.rows)) & ~NB_FAR);
}

__global__ void k_rev(Bufs b, const int *gate)
{
    GATE;
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long s = t / LPP;
    if (s >= b.N || !rebuilds(b, gate, b.pinst[b.perm[s]])) return;
    const int rows = b.rows;
    const int first = b.nfirst[s], n = b.ncnt[s];
    constexpr int G = 4;  // (owned prefixes are <= capown, checked at the build)
    for (int k0 = first + (int)(t % LPP); k0 < n; k0 += G * LPP) {
        int part[G], lo[G], hi[G];
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int k = k0 + g * LPP;
            part[g] = k < n ? nb_at(b, (int)s, k) : -1;
            lo[g] = 0;
            hi[g] = part[g] >= 0 ? b.nfirst[part[g]] : 0;
        }
        int end[G];
#pragma unroll
        for (int g = 0; g < G; ++g) end[g] = hi[g];
        bool active = true;
        while (active) {
            active = false;
#pragma unroll
            for (int g = 0; g < G; ++g) {
                if (lo[g] < hi[g]) {
                    const int mid = (lo[g] + hi[g]) >> 1;
                    if (nb_at(b, part[g], mid) < (int)s) lo[g] = mid + 1;
                    else hi[g] = mid;
                    active = true;
                }
            }
        }
#pragma unroll
        for (int g = 0; g < G; ++g) {
            const int k = k0 + g * LPP;
            if (k >= n) break;
            const bool ok = lo[g] < end[g] && nb_at(b, part[g], lo[g]) == (int)s;
            if (!ok || k - first >= b.capown) atomicOr(b.err, ERR_REV);
            b.rev[entry_at(k, s, rows)] = (uint16_t)(ok ? lo[g] : 0);
            if (ok && k - first < b.capown) b.rev[entry_at(lo[g], part[g], rows)] = (uint16_t)(k - first);
        }
    }
}

// Closes the build: a new list epoch of each instance built, its gate shut
// until the skin is used up (one block).
__global__ void k_build_done(Bufs b, const int *gate)
{
    GATE;
    for (int k = threadIdx.x; k < b.n_inst; k += blockDim.x)
        if (rebuilds(b, gate, k)) {
            b.list_epoch[1 + k] += 1u;
            b.need_build[1 + k] = 0;
        }
    __syncthreads();   // the gate itself is read above
    if (threadIdx.x == 0) {
        b.list_epoch[0] += 1u;
        b.need_build[0] = 0;
        *b.fresh = 1;
        *b.aclose_ok = 0;   // slots were reassigned
    }
}

// ---------------------------------------------------------------- launchers
static inline unsigned nblk(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

// dynamic shared memory of the lane-per-candidate list kernel: at least one
// warp's buffers at the largest list capacity
constexpr size_t NG_SMEM_MAX = 200 * 1024;
static_assert(ng_warp_bytes(SDPD_MAX_NEIGHBORS) <= NG_SMEM_MAX, "list buffers of one warp exceed the limit");

void init_cell_kernels()
{
    cudaFuncSetAttribute(k_neighbors<1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)NG_SMEM_MAX);
    cudaFuncSetAttribute(k_neighbors<1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)NG_SMEM_MAX);
    cudaFuncSetAttribute(k_neighbors<2, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)NG_SMEM_MAX);
    cudaFuncSetAttribute(k_neighbors<2, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)NG_SMEM_MAX);
}

template <int SUB>
static void launch_lists(const Bufs &b, const int *gate, cudaStream_t st)
{
    // Warps per cell: a full cell holds 8 to 24 groups (cells per axis are
    // whole numbers), a half cell one or two.  More than one warp for half
    // cells only where the cells alone leave SMs idle (16,000 particles: 166 us
    // a build with one, 115 with four; 662,000: 1.53 ms with one, 1.66 with four);
    // a warp without a group leaves at once.  8,192 particles in full cells: 381
    // us with 8, 198 with 24; fewer where most cells are empty, so that
    // a large domain is not a launch of idle blocks.
    const int parts = SUB == 1 ? (int)std::min<long long>(24, std::max<long long>(1, 4 * b.N / b.ncell_total))
                               : std::min(4, std::max(1, 16384 / b.ncell_total));
    const size_t wb = ng_warp_bytes(b.cap);
    const unsigned nb = (unsigned)b.ncell_total * parts;
    if (b.split) k_neighbors<SUB, true><<<nb, 32, wb, st>>>(b, parts, gate);
    else k_neighbors<SUB, false><<<nb, 32, wb, st>>>(b, parts, gate);
}

void launch_build(const Bufs &b, int precision, int need_rev, const int *gate, cudaStream_t st)
{
    const int nc = b.ncell_total;
    const int nbk = (nc + 1023) / 1024, bs = spread_block(b.N);
    k_cell_clear<<<nblk(nc, 256), 256, 0, st>>>(b, gate);
    if (b.N) k_cell_keys<<<nblk(b.N, bs), bs, 0, st>>>(b, gate);
    k_scan_local<<<nbk, 1024, 0, st>>>(b, gate);
    k_scan_partials<<<1, 1024, 0, st>>>(b, nbk, gate);
    k_scan_add<<<nbk, 1024, 0, st>>>(b, gate);
    if (b.N) {
        k_scatter<<<nblk(b.N, bs), bs, 0, st>>>(b, gate);
        k_rank<<<nblk(b.N, bs), bs, 0, st>>>(b, gate);
        k_gather<<<nblk(b.N, bs), bs, 0, st>>>(b, precision, gate);
        if (b.cell_sub == 2) launch_lists<2>(b, gate, st);
        else launch_lists<1>(b, gate, st);
        if (need_rev) k_rev<<<nblk(b.N * LPP, 128), 128, 0, st>>>(b, gate);
    }
    k_build_done<<<1, 64, 0, st>>>(b, gate);
}

}  // namespace sdpd
