// Symmetric near-field pair kernel: every unordered pair is met once and its
// force (or Jacobian product) is added to both particles.
//
// F(x_j - x_i) = -F(x_i - x_j), and the adjoint's J (g_j - g_i) changes sign
// with the exchange of i and j, so one evaluation serves both particles: 14
// FP32 lane operations and one rsqrt per unordered pair in the forward
// direction (separation 3, r^2 3, r^-3 2, sums 3 + 3) where two directed ones
// cost 22 and two; 25 against 44 in the adjoint.
//
// Work decomposition.  As in nf_force.cu a pencil centred at cell (i, j, k)
// has the sinks (i+c, j, k), |c| <= R, and the sources lie in the plane x = i;
// here only half of that plane is taken, (i, j+b, k+d) with b > 0 or b = 0 and
// d > 0, plus the centre cell.  Exchanging the roles maps the offset
// (-c, b, d) to (c, -b, -d), so the half planes of all pencils hold every pair
// of cells once.  The centre cell meets the sinks with c < 0 (both get the
// force) and itself (c = 0: ordered pairs, one-sided).  A particle collects
// 2R+1 partial sums as a sink and 1 + ((2R+1)^2 - 1)/2 as a source, each in a
// slot of its own; k_combine adds them without rounding error.  No result
// depends on the order in which warps run.
//
// One warp runs one unit: the pencil's sinks (in chunks of 64 G, two per lane
// in the halves of G packed registers) against a run of source tiles of 32.
// A tile's sources are written to shared memory twice over, each value
// duplicated for the packed arithmetic; in step t lane l meets source
// (l + t) mod 32, whose reaction sum travels with it from lane l + 1 by six
// shuffles (a packed pair per component), so after 32 steps every source is
// back in its own lane with the sum over the chunk's 64 G sinks.  A step of G
// groups costs 14 G packed FMA-pipe instructions, 2 G rsqrt, 6 shuffles and 2
// shared loads for 4 G ordered pairs per lane.  Later chunks of the same pencil add to the tile's
// slots with red.add from the same thread that stored them, in chunk order.
//
// Balance (count_units).  A dear pencil's tiles are split into `groups` runs (a
// rule on N, with slots of their own for the sinks); where even a run is dearer
// than one warp's share of the box, the sinks' half and the sources' half of
// the work become one-sided units per chunk (22 operations a pair instead of
// 14, any number of warps).  A box with much of its work in such pencils, or whose
// pencils fill the lanes badly, is left to the directed kernel (box_is_sym, on the
// device: the counts are not known on the host).
//
// Softening and the density follow nf_force.cu: tiles that can hold a pair
// closer than a cell track the smallest r^2 and are run again on the exact
// path if some pair was closer than eps_s; the centre cell's tiles take the
// exact path from the start.
#include <cuda_runtime.h>

#include "nf_pair.cuh"

namespace nf {

namespace {

// Groups of two residents per lane (64 * groups particles a chunk) and resident
// blocks of 8 warps per SM, measured on GB300 (pair kernel, clustered 200^3):
// forward 3 groups at 16 warps 33.5 ms (4: 33.3, 5: 33.0; on a uniform 256^3 box,
// whose pencils hold 320 sinks, 45.8, 48.2 and 46.6; 8 warps are slower), adjoint
// 5 groups at 8 warps 55.0 ms (4: 59.2; 6: 57.3; 3 at 16 warps: 58).  The
// directed kernel takes 38.7 and 72.9 ms (uniform 256^3: 51.6 and 97.4).
// What bounds the loop is not the FMA pipe's issue rate but its operands: run alone in a
// loop, a packed FMA with three different 64-bit sources (the six sums of a group) took
// 3.1 cycles a scheduler where one with two took 2.0, and a shuffle held up the FMAs for
// 2.65.  The bare tile loop reached 13 ordered pairs per clock and SM of the 18.3 that 14
// operations allow (directed: 10.3 of 11.6).  Unrolling, scalar sums, sums rotated through
// shared memory and prefetched sources all measured slower.  The registers are full:
// forward 128, with 24 bytes of spills written and 52 read, adjoint 255, with 68 and 128.
constexpr int kGroupsFwd = 3, kBlocksFwd = 2;
constexpr int kGroupsAdj = 5, kBlocksAdj = 1;
constexpr int kWarps = 8;
// Chains in which a resident's tile sums are added, tile t in chain t mod kChains (a power
// of two).  One chain over all tiles of a pencil (26 at 64 particles per cell, hundreds in a
// dense pencil) lost up to 8 % against the directed kernel in the median error; four
// have a sixteenth of its variance and stay below the directed kernel.  Median error of
// symmetric over directed with one, two and four chains: forward 2 10^6 uniform 1.06, 0.86,
// 0.81, 36 10^6 clustered 1.07, 0.86, 0.79; adjoint 1.4 10^6 uniform 1.07, 0.98, 0.95,
// 17 10^6 clustered 1.07, 0.97, 0.92, R = 3 1.08, 0.95, 0.88.  Call times with four over
// one: forward 1.003, adjoint 256^3 1.008, 64^3 1.03.  Folding every eight tiles into a
// second sum has the same errors and takes as long or longer.
constexpr int kChains = 4;

// (the density build cuts its chunks as the plain one does: its accelerations are the same bits)
constexpr int sym_groups_max(bool adj) { return adj ? kGroupsAdj : kGroupsFwd; }
// Warps that run at once on 152 SMs: a box's work is balanced over these.
constexpr int sym_warps(bool adj) { return 152 * kWarps * (adj ? kBlocksAdj : kBlocksFwd); }

// The share of a box's cost in pencils that need one-sided units above which the
// directed kernel is the better one.  Measured on boxes from the clustered recipe
// to half of all particles in a few cells (directed time over symmetric): forward
// 1.19 at a share of 0.26, 1.07 at 0.35, 1.05 at 0.51, 0.92 at 0.57, 0.78 at 0.66;
// adjoint 1.36 at 0.01, 0.92 at 0.085 (3e5 particles), 1.04 at 0.09 (9e5), 0.74 at
// 0.15 (3e5), 0.96 at 0.24.
__host__ __device__ constexpr double dear_share(bool adj) { return adj ? 0.08 : 0.5; }

// Units of one pencil, by its cost against a warp's share of the box: one unit
// for a light pencil (at most half a share), `groups` units for a dearer one,
// and the one-sided units of both halves where even such a unit is dearer than
// a share: per sink chunk and tile group, and per source chunk (the centre
// cell's sources in chunks of their own).  Splitting every pencil cost 2 to 6 %
// (set-up and a reload of the sinks per unit); splitting none left the last
// warps running alone (64^3 clustered forward: 1.18 ms against 0.89).
struct UnitCount {
    bool heavy;  // one-sided units
    bool light;  // one unit for all groups
    int nch;     // sink chunks
    int n0, n1;  // heavy: source chunks of the centre cell and of the rest
    int units;
    int bucket;
};
__device__ __forceinline__ UnitCount count_units(int n_sink, int n_src, int n_c0, int groups, int GM,
                                                 double share)
{
    UnitCount u;
    const unsigned long long cost = sym_cost(n_sink, n_src, GM);
    u.heavy = (double)cost > share * groups;
    u.light = (double)cost <= 0.5 * share;
    const int ng = (n_sink + 63) >> 6, CH = 64 * GM;
    u.nch = (ng + GM - 1) / GM;
    u.n0 = (n_c0 + CH - 1) / CH;
    u.n1 = (n_src - n_c0 + CH - 1) / CH;
    if (n_sink == 0 && n_src == 0) {
        u.heavy = false;
        u.units = 0;
        u.bucket = kBuckets - 1;
    } else if (u.heavy) {
        u.units = u.nch * groups + u.n0 + u.n1;
        const unsigned long long a = cost / (unsigned long long)(groups * u.nch);
        const unsigned long long b = sym_cost(min(n_src, CH), n_sink, GM);
        u.bucket = cost_bucket(a > b ? a : b);
    } else {
        u.units = u.light ? 1 : groups;
        u.bucket = cost_bucket(cost / (unsigned long long)u.units);
    }
    return u;
}

// Which pencils need one-sided units: their cost, per box, in total[nboxes + b].
__global__ void k_sym_dear(const BoxDev* __restrict__ boxes, int nboxes, int Ctot, const int* __restrict__ off,
                           const int2* __restrict__ dims, unsigned long long* __restrict__ total, int GM, int warps)
{
    for (int gb = blockIdx.x * blockDim.x; gb < Ctot; gb += gridDim.x * blockDim.x) {
        const int c = gb + (int)threadIdx.x;
        if (c >= Ctot) continue;
        const int b = find_box_by_cell(boxes, nboxes, c);
        if (!boxes[b].sym) continue;
        const int2 d = dims[c];
        const UnitCount u =
            count_units(d.x, d.y, off[c + 1] - off[c], boxes[b].groups, GM, (double)total[b] / warps);
        if (u.heavy) atomicAdd(&total[nboxes + b], sym_cost(d.x, d.y, GM));  // few pencils
    }
}

// Boxes in which dear pencils hold much of the work run directed, and those whose
// pencils fill the symmetric kernel's lanes badly: few sinks to a pencil (padded to
// 64; the directed kernel pads to 32) or few sources to a half plane.  fill is the
// directed kernel's lane pairs over twice the symmetric kernel's, the latter with
// what a step costs beside its groups (28 and 10 cycles, sym_cost); the fewer
// particles, the more its longer work list and combine weigh.  Measured over N =
// 2.65e5 .. 6e6, 40 .. 90 particles per cell, R = 1 .. 3, uniform and clustered, the
// directed call's time over the symmetric one's: forward N = 6e6 0.98 at a fill of
// 0.728, 1.14 at 0.795; 2.5e6 1.00 at 0.743, 1.08 at 0.785; 1.2e6 0.94 at 0.728, 1.03
// at 0.801, 1.11 at 0.814; 4e5 0.98 at 0.768, 1.04 at 0.797, 1.10 at 0.815 (and with
// the density, which takes the forward's kernel, 0.98 at 0.801, 1.04 at 0.814; 0.95 at
// 0.797, 1.01 at 0.815); adjoint 7e5 0.99 at 0.747, 1.05 at 0.763; 4e5 0.97 at 0.777,
// 1.14 at 0.795.  R = 1 boxes of 20 to 60 particles per cell stay directed by this.
__device__ __forceinline__ double fill_needed(int N, bool adj)
{
    if (adj) return N < 450000 ? 0.78 : 0.75;
    return N < 450000 ? 0.82 : N < 1500000 ? 0.805 : 0.775;
}
__device__ __forceinline__ bool box_is_sym(const BoxDev* boxes, int nboxes, const unsigned long long* total, int b,
                                           bool adjoint)
{
    if (!boxes[b].sym) return false;
    const double cost = (double)total[b];
    const double fill = (double)total[2 * nboxes + b] * 28.0 / (128.0 * cost);
    return (double)total[nboxes + b] <= dear_share(adjoint) * cost && fill >= fill_needed(boxes[b].N, adjoint);
}

// Counts the units of the lot's boxes and, in lot 0, the chunks of all that turn out directed.
__global__ void k_sym_count(const BoxDev* __restrict__ boxes, int nboxes, int lot, int c0, int c1,
                            const int* __restrict__ off,
                            const int2* __restrict__ dims, const unsigned long long* __restrict__ total, int GM,
                            int warps, bool adjoint, const int* __restrict__ chunks,
                            const unsigned char* __restrict__ bucket_of, unsigned* __restrict__ sym_count,
                            unsigned* __restrict__ dir_count)
{
    __shared__ bool one_sym;
    if (threadIdx.x == 0) one_sym = nboxes == 1 && box_is_sym(boxes, nboxes, total, 0, adjoint);
    __syncthreads();
    for (int gb = c0 + blockIdx.x * blockDim.x; gb < c1; gb += gridDim.x * blockDim.x) {
        const int c = gb + (int)threadIdx.x;
        int n = 0, bk = -1;  // bucket, + kBuckets on the directed list
        if (c < c1) {
            const int b = find_box_by_cell(boxes, nboxes, c);
            if (nboxes == 1 ? one_sym : box_is_sym(boxes, nboxes, total, b, adjoint)) {
                if (boxes[b].lot == lot) {
                    const int2 d = dims[c];
                    const UnitCount u =
                        count_units(d.x, d.y, off[c + 1] - off[c], boxes[b].groups, GM, (double)total[b] / warps);
                    n = u.units;
                    if (n) bk = u.bucket;
                }
            } else if (lot == 0 && boxes[b].sym) {  // a candidate: its chunks are not counted yet
                n = chunks[c];
                if (n) bk = kBuckets + (int)bucket_of[c];
            }
        }
        const unsigned peers = __match_any_sync(kFull, bk);
        const unsigned tot = __reduce_add_sync(peers, (unsigned)n);
        if (bk >= 0 && (int)(threadIdx.x & 31) == __ffs(peers) - 1)
            atomicAdd(bk < kBuckets ? &sym_count[bk] : &dir_count[bk - kBuckets], tot);
    }
}

// Exclusive scans of both lists' buckets (lot 0; later the units' alone, in kBuckets
// threads); the boxes' kernels for good.
__global__ void k_sym_scan(BoxDev* boxes, int nboxes, const unsigned long long* __restrict__ total, bool adjoint,
                           SymCtl* ctl, unsigned* dir_count, WsHeader* hdr)
{
    __shared__ unsigned v[2][kBuckets];
    const int t = threadIdx.x & (kBuckets - 1), list = threadIdx.x / kBuckets;
    unsigned* count = list ? dir_count : ctl->bucket;
    v[list][t] = count[t];
    __syncthreads();
    if (t == 0) {
        unsigned run = 0;
        for (int b = 0; b < kBuckets; ++b) {
            const unsigned c = v[list][b];
            v[list][b] = run;
            run += c;
        }
        if (list) hdr->n_items = (int)run;
        else hdr->sym_units += ctl->n_units = (int)run;
    }
    __syncthreads();
    count[t] = v[list][t];
    for (int b = threadIdx.x; b < nboxes; b += blockDim.x)
        boxes[b].sym = box_is_sym(boxes, nboxes, total, b, adjoint);
}

// Unit types (item .w)
constexpr int kUnitSym = 0, kUnitSinks = 1, kUnitSources = 2;

// Writes both lists bucket by bucket (as k_items): the lot's symmetric units and, in
// lot 0, the directed items of the other boxes.
__global__ void k_sym_units(const BoxDev* __restrict__ boxes, int nboxes, int lot, int c0, int c1,
                            const int* __restrict__ off,
                            const int2* __restrict__ dims, const unsigned long long* __restrict__ total, int GM,
                            int warps, const int* __restrict__ chunks, const unsigned char* __restrict__ bucket_of,
                            unsigned* __restrict__ sym_cursor, unsigned* __restrict__ dir_cursor,
                            int4* __restrict__ units, int4* __restrict__ items)
{
    const int lane = threadIdx.x & 31;
    for (int gb = c0 + blockIdx.x * blockDim.x; gb < c1; gb += gridDim.x * blockDim.x) {
        const int c = gb + (int)threadIdx.x;
        int bk = -1, b = 0, groups = 1, n = 0;
        UnitCount u = {};
        if (c < c1) {
            b = find_box_by_cell(boxes, nboxes, c);
            if (boxes[b].sym) {
                if (boxes[b].lot == lot) {
                    const int2 d = dims[c];
                    groups = boxes[b].groups;
                    u = count_units(d.x, d.y, off[c + 1] - off[c], groups, GM, (double)total[b] / warps);
                    n = u.units;
                    if (n) bk = u.bucket;
                }
            } else if (lot == 0) {
                n = chunks[c];
                if (n) bk = kBuckets + (int)bucket_of[c];
            }
        }
        const unsigned peers = __match_any_sync(kFull, bk);
        const int leader = __ffs(peers) - 1;
        unsigned pre = 0, tot = 0;
        for (int src = 0; src < 32; ++src) {
            const unsigned v = __shfl_sync(kFull, (unsigned)n, src);
            if ((peers >> src) & 1u) {
                tot += v;
                if (src < lane) pre += v;
            }
        }
        unsigned base = 0;
        if (bk >= 0 && lane == leader)
            base = atomicAdd(bk < kBuckets ? &sym_cursor[bk] : &dir_cursor[bk - kBuckets], tot);
        base = __shfl_sync(kFull, base, leader) + pre;
        if (bk < 0) continue;  // no warp-wide operation follows in this iteration
        if (bk >= kBuckets) {
            for (int q = 0; q < n; ++q) items[base + q] = make_int4(c, q, b, 0);
        } else if (!u.heavy) {
            for (int q = 0; q < n; ++q) units[base + q] = make_int4(c, u.light ? -1 : q, b, kUnitSym);
        } else {
            unsigned at = base;
            for (int q = 0; q < u.nch * groups; ++q) units[at++] = make_int4(c, q, b, kUnitSinks);
            for (int q = 0; q < u.n0 + u.n1; ++q) units[at++] = make_int4(c, q, b, kUnitSources);
        }
    }
}

// ---------------------------------------------------------------------------
// Pair kernel
// ---------------------------------------------------------------------------

// Resident particles of a lane: two per group, one in each half.
template <int G, bool ADJ>
struct Residents {
    f2 nx[G], ny[G], nz[G];                                      // -position
    f2 ngx[ADJ ? G : 1], ngy[ADJ ? G : 1], ngz[ADJ ? G : 1];     // -g
    f2 sx[G], sy[G], sz[G];                                      // sums of the current tile
};

// Reaction sums of the source a lane holds in this step (they travel with it):
// the halves belong to the two residents of a group.
struct Reaction {
    f2 x, y, z, w;
};

// A warp's tile in shared memory, every value in both halves of a pair, the 32
// sources twice over so that lane l reads source (l + t) mod 32 at l + t.
struct Tile {
    const ulonglong2* xy;
    const f2* z;
    const ulonglong2* gxy;
    const f2* gz;
};

__device__ __forceinline__ f2 shfl2(f2 v, int src)
{
    return pk(__shfl_sync(kFull, lo(v), src), __shfl_sync(kFull, hi(v), src));
}

// One tile, f = r^-3 for every pair.  FORCE off: the density alone.  The density's
// sums live only in the loops that take it (few tiles) and join the running ones in
// shared memory at once: totw[s * stride], stride TS.
template <int G, bool REACT, bool TRK, bool DENS, bool FORCE, int TS>
__device__ __forceinline__ void tile_fwd(const Tile& v, Residents<G, false>& k, Reaction& a, float& trk, f2 b2,
                                         f2* totw)
{
    f2 sw[DENS ? G : 1];
    if constexpr (DENS)
#pragma unroll
        for (int s = 0; s < G; ++s) sw[s] = 0ull;
    const f2 tiny = pk(kTiny, kTiny);
    const int next = (threadIdx.x + 1) & 31;
#pragma unroll 1
    for (int t = 0; t < 32; ++t) {
        const ulonglong2 xy = v.xy[t];
        const f2 pz = v.z[t];
#pragma unroll
        for (int s = 0; s < G; ++s) {
            const f2 dx = add2(xy.x, k.nx[s]), dy = add2(xy.y, k.ny[s]), dz = add2(pz, k.nz[s]);
            f2 r2 = fma2(dx, dx, tiny);
            r2 = fma2(dy, dy, r2);
            r2 = fma2(dz, dz, r2);
            if constexpr (TRK) trk = track_min(trk, r2);
            if constexpr (DENS) {
                const f2 w = tophat2(r2, b2);
                sw[s] = add2(sw[s], w);
                if constexpr (REACT) a.w = add2(a.w, w);
            }
            if constexpr (FORCE) {
                const f2 ri = rsqrt2(r2);
                const f2 f = mul2(mul2(ri, ri), ri);
                k.sx[s] = fma2(dx, f, k.sx[s]);
                k.sy[s] = fma2(dy, f, k.sy[s]);
                k.sz[s] = fma2(dz, f, k.sz[s]);
                if constexpr (REACT) {
                    a.x = fma2(dx, f, a.x);
                    a.y = fma2(dy, f, a.y);
                    a.z = fma2(dz, f, a.z);
                }
            }
        }
        if constexpr (REACT) {
            if constexpr (FORCE) {
                a.x = shfl2(a.x, next);
                a.y = shfl2(a.y, next);
                a.z = shfl2(a.z, next);
            }
            if constexpr (DENS) a.w = shfl2(a.w, next);
        }
    }
    if constexpr (DENS)
#pragma unroll
        for (int s = 0; s < G; ++s) totw[s * TS] = add2(totw[s * TS], sw[s]);
}

// Keeps the halves of v whose bits are set.
__device__ __forceinline__ f2 keep2(f2 v, unsigned bits)
{
    return pk((bits & 1u) ? lo(v) : 0.0f, (bits & 2u) ? hi(v) : 0.0f);
}

// One tile, f = min(poly(r), r^-3) (Eq. (spline) with the min hand-off).  Bit
// 2s + h of ms0 / mr0: the resident s, h receives the force / acts on the source,
// for the tile's first n_self sources.
template <int G, bool REACT, bool DENS, int TS>
__device__ __forceinline__ void tile_fwd_exact(const Tile& v, Residents<G, false>& k, Reaction& a, const Coef& cf,
                                               f2 b2, unsigned ms0, unsigned mr0, int n_self, f2* totw)
{
    f2 sw[DENS ? G : 1];
    if constexpr (DENS)
#pragma unroll
        for (int s = 0; s < G; ++s) sw[s] = 0ull;
    const f2 tiny = pk(kTiny, kTiny);
    const f2 c0 = pk(cf.c0, cf.c0), c1 = pk(cf.c1, cf.c1), c2 = pk(cf.c2, cf.c2);
    const int next = (threadIdx.x + 1) & 31;
#pragma unroll 1
    for (int t = 0; t < 32; ++t) {
        // the masks apply to the sources of the residents' own cell
        const bool self = (int)((threadIdx.x + t) & 31) < n_self;
        const unsigned ms = self ? ms0 : ~0u, mr = self ? mr0 : ~0u;
        const ulonglong2 xy = v.xy[t];
        const f2 pz = v.z[t];
#pragma unroll
        for (int s = 0; s < G; ++s) {
            const f2 dx = add2(xy.x, k.nx[s]), dy = add2(xy.y, k.ny[s]), dz = add2(pz, k.nz[s]);
            f2 r2 = fma2(dx, dx, tiny);
            r2 = fma2(dy, dy, r2);
            r2 = fma2(dz, dz, r2);
            if constexpr (DENS) {
                const f2 w = tophat2(r2, b2);
                sw[s] = add2(sw[s], keep2(w, ms >> (2 * s)));
                if constexpr (REACT) a.w = add2(a.w, keep2(w, mr >> (2 * s)));
            }
            const f2 ri = rsqrt2(r2);
            const f2 p = fma2(r2, fma2(c1, ri, c2), c0);
            const f2 r3 = mul2(mul2(ri, ri), ri);
            const f2 f = pk(fminf(lo(p), lo(r3)), fminf(hi(p), hi(r3)));
            const f2 fs = keep2(f, ms >> (2 * s));
            k.sx[s] = fma2(dx, fs, k.sx[s]);
            k.sy[s] = fma2(dy, fs, k.sy[s]);
            k.sz[s] = fma2(dz, fs, k.sz[s]);
            if constexpr (REACT) {
                const f2 fr = keep2(f, mr >> (2 * s));
                a.x = fma2(dx, fr, a.x);
                a.y = fma2(dy, fr, a.y);
                a.z = fma2(dz, fr, a.z);
            }
        }
        if constexpr (REACT) {
            a.x = shfl2(a.x, next);
            a.y = shfl2(a.y, next);
            a.z = shfl2(a.z, next);
            if constexpr (DENS) a.w = shfl2(a.w, next);
        }
    }
    if constexpr (DENS)
#pragma unroll
        for (int s = 0; s < G; ++s) totw[s * TS] = add2(totw[s * TS], sw[s]);
}

// Adjoint, one tile: J v = r^-3 (v - 3 r^-2 (d.v) d), v = g_j - g_i.
template <int G, bool REACT, bool TRK>
__device__ __forceinline__ void tile_adj(const Tile& v, Residents<G, true>& k, Reaction& a, float& trk)
{
    const f2 tiny = pk(kTiny, kTiny), m3 = pk(-3.0f, -3.0f);
    const int next = (threadIdx.x + 1) & 31;
#pragma unroll 1
    for (int t = 0; t < 32; ++t) {
        const ulonglong2 xy = v.xy[t], gxy = v.gxy[t];
        const f2 pz = v.z[t], qz = v.gz[t];
#pragma unroll
        for (int s = 0; s < G; ++s) {
            const f2 dx = add2(xy.x, k.nx[s]), dy = add2(xy.y, k.ny[s]), dz = add2(pz, k.nz[s]);
            f2 r2 = fma2(dx, dx, tiny);
            r2 = fma2(dy, dy, r2);
            r2 = fma2(dz, dz, r2);
            if constexpr (TRK) trk = track_min(trk, r2);
            const f2 ri = rsqrt2(r2);
            const f2 ri2 = mul2(ri, ri);
            const f2 ri3 = mul2(ri2, ri);
            const f2 vx = add2(gxy.x, k.ngx[s]), vy = add2(gxy.y, k.ngy[s]), vz = add2(qz, k.ngz[s]);
            f2 dv = mul2(dx, vx);
            dv = fma2(dy, vy, dv);
            dv = fma2(dz, vz, dv);
            const f2 c = mul2(dv, mul2(ri2, m3));
            const f2 ux = fma2(c, dx, vx), uy = fma2(c, dy, vy), uz = fma2(c, dz, vz);
            k.sx[s] = fma2(ri3, ux, k.sx[s]);
            k.sy[s] = fma2(ri3, uy, k.sy[s]);
            k.sz[s] = fma2(ri3, uz, k.sz[s]);
            if constexpr (REACT) {
                a.x = fma2(ri3, ux, a.x);
                a.y = fma2(ri3, uy, a.y);
                a.z = fma2(ri3, uz, a.z);
            }
        }
        if constexpr (REACT) {
            a.x = shfl2(a.x, next);
            a.y = shfl2(a.y, next);
            a.z = shfl2(a.z, next);
        }
    }
}

// Adjoint, one tile, exact: the softened branch selected per pair (as nf_force.cu's stage_adj_exact).
template <int G, bool REACT>
__device__ __forceinline__ void tile_adj_exact(const Tile& v, Residents<G, true>& k, Reaction& a,
                                               const Coef& cf, unsigned ms0, unsigned mr0, int n_self)
{
    const f2 tiny = pk(kTiny, kTiny), m3 = pk(-3.0f, -3.0f);
    const f2 c0 = pk(cf.c0, cf.c0), c1 = pk(cf.c1, cf.c1), c2 = pk(cf.c2, cf.c2);
    const f2 e0 = pk(cf.e0, cf.e0), e1 = pk(cf.e1, cf.e1);
    const int next = (threadIdx.x + 1) & 31;
#pragma unroll 1
    for (int t = 0; t < 32; ++t) {
        // the masks apply to the sources of the residents' own cell
        const bool self = (int)((threadIdx.x + t) & 31) < n_self;
        const unsigned ms = self ? ms0 : ~0u, mr = self ? mr0 : ~0u;
        const ulonglong2 xy = v.xy[t], gxy = v.gxy[t];
        const f2 pz = v.z[t], qz = v.gz[t];
#pragma unroll
        for (int s = 0; s < G; ++s) {
            const f2 dx = add2(xy.x, k.nx[s]), dy = add2(xy.y, k.ny[s]), dz = add2(pz, k.nz[s]);
            f2 r2 = fma2(dx, dx, tiny);
            r2 = fma2(dy, dy, r2);
            r2 = fma2(dz, dz, r2);
            const f2 ri = rsqrt2(r2);
            const f2 ri2 = rcp2(r2);
            const f2 Fs = fma2(r2, fma2(c1, ri, c2), c0);
            const f2 Gs = mul2(fma2(e0, ri, e1), rcp2(Fs));
            const f2 Fr = mul2(ri2, ri);
            const f2 Gr = mul2(ri2, m3);
            const bool sl = lo(r2) < cf.eps2, sh = hi(r2) < cf.eps2;
            const f2 F = pk(sl ? lo(Fs) : lo(Fr), sh ? hi(Fs) : hi(Fr));
            const f2 Gm = pk(sl ? lo(Gs) : lo(Gr), sh ? hi(Gs) : hi(Gr));
            const f2 vx = add2(gxy.x, k.ngx[s]), vy = add2(gxy.y, k.ngy[s]), vz = add2(qz, k.ngz[s]);
            f2 dv = mul2(dx, vx);
            dv = fma2(dy, vy, dv);
            dv = fma2(dz, vz, dv);
            const f2 c = mul2(dv, Gm);
            const f2 ux = fma2(c, dx, vx), uy = fma2(c, dy, vy), uz = fma2(c, dz, vz);
            const f2 Fi = keep2(F, ms >> (2 * s));
            k.sx[s] = fma2(Fi, ux, k.sx[s]);
            k.sy[s] = fma2(Fi, uy, k.sy[s]);
            k.sz[s] = fma2(Fi, uz, k.sz[s]);
            if constexpr (REACT) {
                const f2 Fj = keep2(F, mr >> (2 * s));
                a.x = fma2(Fj, ux, a.x);
                a.y = fma2(Fj, uy, a.y);
                a.z = fma2(Fj, uz, a.z);
            }
        }
        if constexpr (REACT) {
            a.x = shfl2(a.x, next);
            a.y = shfl2(a.y, next);
            a.z = shfl2(a.z, next);
        }
    }
}

// Per-warp shared memory: the tile (and its g), the cp.async targets, the
// residents' running sums (kChains of them, and the density's) and the segment tables of
// both lists.
template <int GM, bool ADJ, bool DENS>
struct SymSmem {
    static constexpr size_t xy = 0;
    static constexpr size_t z = xy + 64 * 16;
    static constexpr size_t gxy = z + 64 * 8;
    static constexpr size_t gz = gxy + (ADJ ? 64 * 16 : 0);
    static constexpr size_t raw = gz + (ADJ ? 64 * 8 : 0);
    static constexpr size_t graw = raw + 32 * 16;
    static constexpr size_t tot = graw + (ADJ ? 32 * 16 : 0);
    static constexpr int chain = GM * 3 * 32;  // sums of one chain
    static constexpr size_t totw = tot + (size_t)kChains * chain * 8;
    static constexpr size_t tab = totw + (DENS ? (size_t)GM * 32 * 8 : 0);
    static constexpr int NA = 2 * NF_MAX_R + 1;
    static constexpr size_t ints = (NA + 1) + NA + (kHalfMax + 1) + 2 * kHalfMax;
    static constexpr size_t bytes = (tab + 4 * ints + 15) & ~size_t(15);
};

// One of a unit's two particle lists (the pencil's sinks, or the half plane's
// sources): segment q holds the flat positions [pre[q], pre[q+1]), sorted slot
// base[q] + position.
struct List {
    const int* pre;
    const int* base;
    const int* shift;  // packed (dy, dz), or null: dx = q - R
    int slot0, slot_step, slot_add;  // partial slot of segment q: slot0 + q * slot_step + slot_add
};

__device__ __forceinline__ void list_shift(const List& l, int q, int R, float4& r)
{
    if (l.shift) {
        const int c = l.shift[q];
        r.y += (float)((c & 15) - 8);
        r.z += (float)((c >> 4) - 8);
    } else {
        r.x += (float)(q - R);
    }
}

struct Pass {
    List res, til;
    int r0, r1;        // resident positions [r0, r1)
    int t0, t1;        // tiles
    int n;             // length of the tile list
    int n_self;        // its positions below this are the residents' own cell: exact, masked
    bool exact;        // every tile on the exact path
    int far_from;      // tiles starting here or later are untracked
    int n_act, n_get;  // self sources: residents below n_act act on them, below n_get receive
    bool first;        // the tile sums are stored (else added)
    int zero;          // slots after the residents' own that are cleared (groups run in one unit)
};

__device__ __forceinline__ void red_add(float* p, float v)
{
    asm volatile("red.relaxed.gpu.global.add.f32 [%0], %1;" ::"l"(p), "f"(v) : "memory");
}

template <int G, int GM, bool ADJ, bool DENS, bool REACT>
__device__ __forceinline__ void run_pass(const Pass& ps, int R, const Coef& cf, f2 b2, const float4* __restrict__ rel,
                                         const float4* __restrict__ gs, unsigned char* sm, float* __restrict__ planes,
                                         int N, int part_base, int nslot, WsHeader* hdr)
{
    using L = SymSmem<GM, ADJ, DENS>;
    const int lane = threadIdx.x & 31;
    ulonglong2* xy = reinterpret_cast<ulonglong2*>(sm + L::xy);
    f2* zz = reinterpret_cast<f2*>(sm + L::z);
    ulonglong2* gxy = reinterpret_cast<ulonglong2*>(sm + L::gxy);
    f2* gz = reinterpret_cast<f2*>(sm + L::gz);
    float4* raw = reinterpret_cast<float4*>(sm + L::raw);
    float4* graw = reinterpret_cast<float4*>(sm + L::graw);
    f2* tot = reinterpret_cast<f2*>(sm + L::tot) + lane;
    const size_t dens0 = 3 * (size_t)nslot;  // first density plane

    int cur = 0;
    int at = -1;
    // issues the copy of this lane's source of tile t; its sorted slot goes to `at`
    auto issue = [&](int t) {
        const int p = 32 * t + lane;
        at = -1;
        if (p < ps.n) {
            while (p >= ps.til.pre[cur + 1]) ++cur;
            at = ps.til.base[cur] + p;
            cp_async16(&raw[lane], &rel[at]);
            if constexpr (ADJ) cp_async16(&graw[lane], &gs[at]);
        }
        cp_async_commit();
    };
    if (ps.t0 < ps.t1) issue(ps.t0);

    Residents<G, ADJ> k;
    unsigned ms = 0, mr = 0;
    {
        int q = 0;
#pragma unroll
        for (int s = 0; s < G; ++s) {
            float4 r[2], g[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int p = ps.r0 + (2 * s + h) * 32 + lane;
                r[h] = make_float4(kFarSink, kFarSink, kFarSink, 0.0f);
                g[h] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (p < ps.r1) {
                    while (p >= ps.res.pre[q + 1]) ++q;
                    r[h] = rel[ps.res.base[q] + p];
                    list_shift(ps.res, q, R, r[h]);
                    if constexpr (ADJ) g[h] = gs[ps.res.base[q] + p];
                }
                if (p < ps.n_get) ms |= 1u << (2 * s + h);
                if (p < ps.n_act) mr |= 1u << (2 * s + h);
            }
            k.nx[s] = pk(-r[0].x, -r[1].x);
            k.ny[s] = pk(-r[0].y, -r[1].y);
            k.nz[s] = pk(-r[0].z, -r[1].z);
            if constexpr (ADJ) {
                k.ngx[s] = pk(-g[0].x, -g[1].x);
                k.ngy[s] = pk(-g[0].y, -g[1].y);
                k.ngz[s] = pk(-g[0].z, -g[1].z);
            }
        }
    }
    const bool dens_near_only = lo(b2) <= 1.0f;   // b <= one cell width
    const bool soft_near_only = cf.eps2 <= 1.0f;  // eps_s <= one cell width
    const bool dens_defer = DENS && cf.dens_defer != 0 && dens_near_only;
    const Tile tv = {xy + lane, zz + lane, gxy + lane, gz + lane};
    constexpr int TS = 32;
    f2* totw = reinterpret_cast<f2*>(sm + L::totw) + lane;
    if constexpr (DENS)
#pragma unroll
        for (int s = 0; s < G; ++s) totw[s * TS] = 0ull;

    for (int t = ps.t0; t < ps.t1; ++t) {
        const int my_at = at, my_seg = cur;
        cp_async_wait<0>();
        {
            float4 v = make_float4(kFarSrc, kFarSrc, kFarSrc, 0.0f);
            if (my_at >= 0) {
                v = raw[lane];
                list_shift(ps.til, my_seg, R, v);
            }
            const ulonglong2 w = make_ulonglong2(pk(v.x, v.x), pk(v.y, v.y));
            xy[lane] = w;
            xy[lane + 32] = w;
            zz[lane] = pk(v.z, v.z);
            zz[lane + 32] = pk(v.z, v.z);
            if constexpr (ADJ) {
                float4 g = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (my_at >= 0) g = graw[lane];
                const ulonglong2 gw = make_ulonglong2(pk(g.x, g.x), pk(g.y, g.y));
                gxy[lane] = gw;
                gxy[lane + 32] = gw;
                gz[lane] = pk(g.z, g.z);
                gz[lane + 32] = pk(g.z, g.z);
            }
        }
        __syncwarp();
        if (t + 1 < ps.t1) issue(t + 1);
        const int n_self = ps.n_self - 32 * t;  // sources of the tile below this are self
        const bool far = 32 * t >= ps.far_from;
        bool exact = ps.exact || n_self > 0;
        const bool dens = DENS && (!dens_near_only || !far);
        bool fused = false;  // the density is taken in the fast loop
        const bool plain = !exact && far && soft_near_only;  // no pair of this tile can need the exact path
        Reaction a;
        auto clear = [&]() {
#pragma unroll
            for (int s = 0; s < G; ++s) {
                k.sx[s] = k.sy[s] = k.sz[s] = 0ull;
            }
            a.x = a.y = a.z = 0ull;
        };
        a.w = 0ull;
        clear();
        if (!exact) {
            float trk = kBig;
            if (plain) {
                if constexpr (ADJ) tile_adj<G, REACT, false>(tv, k, a, trk);
                else {
                    if constexpr (DENS) {
                        if (dens) tile_fwd<G, REACT, false, true, true, TS>(tv, k, a, trk, b2, totw);
                    }
                    if (!dens) tile_fwd<G, REACT, false, false, true, TS>(tv, k, a, trk, b2, totw);
                }
            } else {
                if constexpr (ADJ) tile_adj<G, REACT, true>(tv, k, a, trk);
                else {
                    fused = dens && !dens_defer;
                    if constexpr (DENS) {
                        if (fused) tile_fwd<G, REACT, true, true, true, TS>(tv, k, a, trk, b2, totw);
                    }
                    if (!fused) tile_fwd<G, REACT, true, false, true, TS>(tv, k, a, trk, b2, totw);
                }
                exact = __any_sync(kFull, trk < cf.eps2);
                if (exact && lane == 0) atomicAdd(&hdr->stages_rerun, 1ull);  // rare
                if constexpr (DENS && !ADJ) {
                    // a pair closer than b gives a positive term; elsewhere every term is +0
                    if (dens && dens_defer && !exact && __any_sync(kFull, trk < lo(b2)))
                        tile_fwd<G, REACT, false, true, false, TS>(tv, k, a, trk, b2, totw);
                }
                if (exact) clear();
            }
        }
        if (exact) {
            if constexpr (ADJ) tile_adj_exact<G, REACT>(tv, k, a, cf, ms, mr, n_self);
            else {
                if constexpr (DENS) {
                    if (dens && !fused) tile_fwd_exact<G, REACT, true, TS>(tv, k, a, cf, b2, ms, mr, n_self, totw);
                }
                // (a re-run keeps the density that the fused loop has taken: the term is the same)
                if (!dens || fused) tile_fwd_exact<G, REACT, false, TS>(tv, k, a, cf, b2, ms, mr, n_self, totw);
            }
        }
        // the tile's sums (chains of at most 32 sources) join one of the running ones
        f2* const chain = tot + (t & (kChains - 1)) * L::chain;
#pragma unroll
        for (int s = 0; s < G; ++s) {
            f2* p = chain + s * 96;
            if (t < ps.t0 + kChains) {
                p[0] = k.sx[s];
                p[32] = k.sy[s];
                p[64] = k.sz[s];
            } else {
                p[0] = add2(p[0], k.sx[s]);
                p[32] = add2(p[32], k.sy[s]);
                p[64] = add2(p[64], k.sz[s]);
            }
        }
        if constexpr (REACT) {
            if (my_at >= 0) {
                const int slot = ps.til.slot0 + my_seg * ps.til.slot_step + ps.til.slot_add;
                float* d = planes + 3 * (size_t)slot * (size_t)N + (size_t)(my_at - part_base);
                const float rx = -(lo(a.x) + hi(a.x)), ry = -(lo(a.y) + hi(a.y)), rz = -(lo(a.z) + hi(a.z));
                if (ps.first) {
                    d[0] = rx;
                    d[N] = ry;
                    d[2 * (size_t)N] = rz;
                } else {
                    red_add(d, rx);
                    red_add(d + N, ry);
                    red_add(d + 2 * (size_t)N, rz);
                }
                if constexpr (DENS) {
                    float* w = planes + (dens0 + (size_t)slot) * (size_t)N + (size_t)(my_at - part_base);
                    const float rw = lo(a.w) + hi(a.w);
                    if (ps.first) *w = rw;
                    else red_add(w, rw);
                }
            }
        }
        __syncwarp();
    }
    // the residents' partial sums: the chains join the first tile's
    f2* const sums = tot + (ps.t0 & (kChains - 1)) * L::chain;
#pragma unroll 1
    for (int t = ps.t0 + 1; t < min(ps.t0 + kChains, ps.t1); ++t) {
        const f2* other = tot + (t & (kChains - 1)) * L::chain;
#pragma unroll
        for (int q = 0; q < 3 * G; ++q) sums[q * 32] = add2(sums[q * 32], other[q * 32]);
    }
    {
        int q = 0;
#pragma unroll
        for (int s = 0; s < G; ++s) {
            const f2* p = sums + s * 96;
            const bool any = ps.t0 < ps.t1;
            const f2 x = any ? p[0] : 0ull, y = any ? p[32] : 0ull, z = any ? p[64] : 0ull;
            const f2 w = DENS ? totw[s * TS] : 0ull;
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int pos = ps.r0 + (2 * s + h) * 32 + lane;
                if (pos < ps.r1) {
                    while (pos >= ps.res.pre[q + 1]) ++q;
                    const size_t e = (size_t)(ps.res.base[q] + pos - part_base);
                    const int slot = ps.res.slot0 + q * ps.res.slot_step + ps.res.slot_add;
                    float* d = planes + 3 * (size_t)slot * (size_t)N + e;
                    d[0] = h ? hi(x) : lo(x);
                    d[N] = h ? hi(y) : lo(y);
                    d[2 * (size_t)N] = h ? hi(z) : lo(z);
                    if constexpr (DENS) planes[(dens0 + (size_t)slot) * (size_t)N + e] = h ? hi(w) : lo(w);
                    for (int u = 1; u <= ps.zero; ++u) {
                        float* o = d + 3 * (size_t)u * (size_t)N;
                        o[0] = o[N] = o[2 * (size_t)N] = 0.0f;
                        if constexpr (DENS) planes[(dens0 + (size_t)(slot + u)) * (size_t)N + e] = 0.0f;
                    }
                }
            }
        }
    }
    __syncwarp();
}

template <int GM, bool ADJ, bool DENS, int MINB>
__global__ void __launch_bounds__(kWarps * 32, MINB)
k_sym(const BoxDev* __restrict__ boxes, const int* __restrict__ off, const float4* __restrict__ rel,
      const float4* __restrict__ gs, const int4* __restrict__ units, SymCtl* ctl, WsHeader* hdr,
      float* __restrict__ planes0)
{
    extern __shared__ __align__(16) unsigned char smem[];
    using L = SymSmem<GM, ADJ, DENS>;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned char* sm = smem + (size_t)wid * L::bytes;
    int* preA = reinterpret_cast<int*>(sm + L::tab);
    int* baseA = preA + L::NA + 1;
    int* preB = baseA + L::NA;
    int* baseB = preB + kHalfMax + 1;
    int* shB = baseB + kHalfMax;
    const int n_units = *((volatile int*)&ctl->n_units);

    for (;;) {
        int un = 0;
        if (lane == 0) un = atomicAdd(&ctl->queue, 1);
        un = __shfl_sync(kFull, un, 0);
        if (un >= n_units) break;
        const int4 unit = units[un];
        const BoxDev& Bx = boxes[unit.z];
        const int K = Bx.K, R = Bx.R, cb = Bx.cell_base, N = Bx.N, part_base = Bx.part_base, groups = Bx.groups;
        Coef cf;
        cf.c0 = Bx.c0;
        cf.c1 = Bx.c1;
        cf.c2 = Bx.c2;
        cf.e0 = Bx.e0;
        cf.e1 = Bx.e1;
        cf.eps2 = Bx.eps2;
        cf.dens_defer = Bx.dens_defer;
        const f2 b2 = pk(Bx.dens_b2, Bx.dens_b2);
        float* planes = planes0 + Bx.plane_base;
        const int ns = 2 * R + 1, nb = 1 + (ns * ns - 1) / 2, nslot = ns * groups + nb;
        const int l = unit.x - cb;
        const int ci = l / (K * K), cj = (l / K) % K, ck = l % K;
        // sink segments: cells i-R .. i+R of the pencil
        {
            int cnt = 0, st = 0;
            if (lane < ns) cnt = cell_count(off, cb + (wrap(ci + lane - R, K) * K + cj) * K + ck, &st);
            int inc = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(kFull, inc, o);
                if (lane >= o) inc += y;
            }
            if (lane < ns) {
                preA[lane] = inc - cnt;
                baseA[lane] = st - (inc - cnt);
                if (lane == ns - 1) preA[ns] = inc;
            }
        }
        // source segments: the half plane in rings
        int carry = 0;
        for (int s0 = 0; s0 < nb; s0 += 32) {
            const int q = s0 + lane;
            int cnt = 0, st = 0, b = 0, d = 0;
            if (q < nb) {
                b = c_half[q][0];
                d = c_half[q][1];
                cnt = cell_count(off, cb + (ci * K + wrap(cj + b, K)) * K + wrap(ck + d, K), &st);
            }
            int inc = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(kFull, inc, o);
                if (lane >= o) inc += y;
            }
            if (q < nb) {
                preB[q] = carry + inc - cnt;
                baseB[q] = st - (carry + inc - cnt);
                shB[q] = (b + 8) | ((d + 8) << 4);
            }
            carry += __shfl_sync(kFull, inc, 31);
        }
        if (lane == 0) preB[nb] = carry;
        __syncwarp();
        const int n_sink = preA[ns], n_src = carry, n_c0 = preB[1];
        const int n_near = preB[min(nb, 5)];            // the centre cell and its half first ring
        const int n_before = preA[R], n_le0 = preA[R + 1];  // sinks with c < 0, c <= 0
        const int n_lo = preA[R - 1], n_hi = preA[R + 2];   // sinks with |c| <= 1
        const List LA = {preA, baseA, nullptr, 0, groups, 0};
        const List LB = {preB, baseB, shB, ns * groups, 1, 0};
        const int ng = (n_sink + 63) >> 6, nch = (ng + GM - 1) / GM;

#define NF_SYM_RUN(REACT)                                                                                            \
    do {                                                                                                             \
        const int g_ = (ps.r1 - ps.r0 + 63) >> 6;                                                                    \
        if (GM >= 5 && g_ == 5)                                                                                 \
            run_pass<(GM >= 5 ? 5 : 1), GM, ADJ, DENS, REACT>(ps, R, cf, b2, rel, gs, sm, planes, N, part_base, nslot, hdr); \
        else if (GM >= 4 && g_ == 4)                                                                                 \
            run_pass<(GM >= 4 ? 4 : 1), GM, ADJ, DENS, REACT>(ps, R, cf, b2, rel, gs, sm, planes, N, part_base, nslot, hdr); \
        else if (GM >= 3 && g_ == 3)                                                                                 \
            run_pass<(GM >= 3 ? 3 : 1), GM, ADJ, DENS, REACT>(ps, R, cf, b2, rel, gs, sm, planes, N, part_base, nslot, hdr); \
        else if (GM >= 2 && g_ == 2)                                                                                 \
            run_pass<(GM >= 2 ? 2 : 1), GM, ADJ, DENS, REACT>(ps, R, cf, b2, rel, gs, sm, planes, N, part_base, nslot, hdr); \
        else                                                                                                         \
            run_pass<1, GM, ADJ, DENS, REACT>(ps, R, cf, b2, rel, gs, sm, planes, N, part_base, nslot, hdr);         \
    } while (0)

        Pass ps;
        if (unit.w != kUnitSources) {
            // sinks resident, half plane in tiles
            const int nt = (n_src + 31) >> 5;
            const bool all = unit.w == kUnitSym && unit.y < 0;  // one unit for all tile groups
            const int gi = all ? 0 : unit.w == kUnitSym ? unit.y : unit.y % groups;
            const int t0 = all ? 0 : (int)((long long)nt * gi / groups);
            const int t1 = all ? nt : (int)((long long)nt * (gi + 1) / groups);
            ps.res = LA;
            ps.res.slot_add = gi;
            ps.til = LB;
            ps.n = n_src;
            ps.n_self = n_c0;
            ps.exact = false;
            ps.zero = all ? groups - 1 : 0;
            ps.n_act = n_before;
            ps.n_get = n_le0;
            const int q0 = unit.w == kUnitSym ? 0 : unit.y / groups;
            // a pencil without sinks still clears the slots of its sources
            const int q1 = unit.w == kUnitSym ? max(nch, 1) : q0 + 1;
            for (int q = q0; q < q1; ++q) {
                ps.r0 = nch ? 64 * (int)((long long)ng * q / nch) : 0;
                ps.r1 = nch ? min(64 * (int)((long long)ng * (q + 1) / nch), n_sink) : 0;
                // the centre cell's tiles: nothing to do for a chunk of sinks beyond it
                // (the first chunk stores the tiles' slots, so it runs them all)
                ps.t0 = q > 0 && ps.r0 >= n_le0 ? max(t0, min(n_c0 >> 5, t1)) : t0;
                ps.t1 = t1;
                ps.far_from = ps.r0 < n_hi && ps.r1 > n_lo ? n_near : 0;
                ps.first = q == 0;
                if (unit.w == kUnitSym) NF_SYM_RUN(true);
                else NF_SYM_RUN(false);
            }
        } else {
            // sources resident, the pencil's sinks in tiles
            const int CH = 64 * GM, n0ch = (n_c0 + CH - 1) / CH;
            const bool self = unit.y < n0ch;
            ps.res = LB;
            ps.til = LA;
            ps.r0 = self ? unit.y * CH : n_c0 + (unit.y - n0ch) * CH;
            ps.r1 = min(ps.r0 + CH, self ? n_c0 : n_src);
            ps.n = self ? n_before : n_sink;
            ps.t0 = 0;
            ps.t1 = (ps.n + 31) >> 5;
            ps.n_self = 0;
            ps.exact = self;
            ps.far_from = ps.r0 >= n_near ? 0 : 0x7fffffff;
            ps.n_act = ps.n_get = 0;
            ps.first = false;
            ps.zero = 0;
            NF_SYM_RUN(false);
        }
#undef NF_SYM_RUN
    }
}

int grid_for(size_t n, int threads)
{
    size_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 65535ull * 16) b = 65535ull * 16;
    return (int)b;
}

typedef void (*SymKernel)(const BoxDev*, const int*, const float4*, const float4*, const int4*, SymCtl*, WsHeader*,
                          float*);

template <bool ADJ, bool DENS>
cudaError_t launch_kernel(const BoxDev* boxes, const int* off, const float4* rel, const float4* gs, const int4* units,
                          SymCtl* ctl, WsHeader* hdr, float* planes, cudaStream_t s)
{
    constexpr int GM = sym_groups_max(ADJ);
    SymKernel fn = k_sym<GM, ADJ, DENS, ADJ ? kBlocksAdj : kBlocksFwd>;
    const size_t smem = kWarps * SymSmem<GM, ADJ, DENS>::bytes;
    cudaError_t e = ensure_smem((const void*)fn, (int)smem, true);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, nb = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, (const void*)fn, kWarps * 32, smem);
    if (e != cudaSuccess) return e;
    if (nb < 1) return cudaErrorInvalidConfiguration;
    fn<<<sms * nb, kWarps * 32, smem, s>>>(boxes, off, rel, gs, units, ctl, hdr, planes);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace

int sym_gmax(bool adjoint) { return sym_groups_max(adjoint); }

int sym_slots(int R, int groups) { return (2 * R + 1) * groups + 1 + ((2 * R + 1) * (2 * R + 1) - 1) / 2; }

long long sym_max_units(long long N, long long C, int R, int groups)
{
    // symmetric units: `groups` per cell.  One-sided units: the chunks hold at least 64 particles
    // each but the last of a list (balanced chunks of 64 .. 64 G), over the 2R+1 pencils that a
    // particle is a sink of and the half planes that it is a source of.
    const long long ns = 2 * R + 1, nb = 1 + (ns * ns - 1) / 2;
    return C * (2 * (long long)groups + 2) + (ns * groups + nb) * (N / 64 + 1);
}

cudaError_t launch_sym_units(bool adjoint, BoxDev* boxes, int nboxes, int lot, int c0, int c1, const int* cell_off,
                             const int2* dims, SymCtl* ctl, unsigned long long* total, int4* units,
                             const int* chunks, const unsigned char* bucket_of, unsigned* bucket_count, int4* items,
                             WsHeader* hdr, cudaStream_t s)
{
    const int grid = grid_for(c1 - c0, 256), warps = sym_warps(adjoint), GM = sym_groups_max(adjoint);
    if (lot == 0) {
        k_sym_dear<<<grid, 256, 0, s>>>(boxes, nboxes, c1, cell_off, dims, total, GM, warps);
        count_launches(1);
    } else {
        const cudaError_t e = cudaMemsetAsync(ctl, 0, sizeof(SymCtl), s);
        if (e != cudaSuccess) return e;
    }
    k_sym_count<<<grid, 256, 0, s>>>(boxes, nboxes, lot, c0, c1, cell_off, dims, total, GM, warps, adjoint, chunks,
                                     bucket_of, ctl->bucket, bucket_count);
    k_sym_scan<<<1, (lot == 0 ? 2 : 1) * kBuckets, 0, s>>>(boxes, nboxes, total, adjoint, ctl, bucket_count, hdr);
    k_sym_units<<<grid, 256, 0, s>>>(boxes, nboxes, lot, c0, c1, cell_off, dims, total, GM, warps, chunks,
                                     bucket_of, ctl->bucket, bucket_count, units, items);
    count_launches(3);
    return cudaGetLastError();
}

cudaError_t launch_sym_force(bool adjoint, bool density, const BoxDev* boxes, const int* cell_off, const float4* rel,
                             const float4* gs, const int4* units, SymCtl* ctl, WsHeader* hdr, float* planes,
                             cudaStream_t s)
{
    if (adjoint) return launch_kernel<true, false>(boxes, cell_off, rel, gs, units, ctl, hdr, planes, s);
    if (density) return launch_kernel<false, true>(boxes, cell_off, rel, gs, units, ctl, hdr, planes, s);
    return launch_kernel<false, false>(boxes, cell_off, rel, gs, units, ctl, hdr, planes, s);
}

}  // namespace nf
