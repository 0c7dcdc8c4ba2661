// Collision detection (Alg. 1, first line) on the device.
//
// Broad phase: uniform grid hash.  Every body's inflated AABB is computed in IEEE single
// precision with a fixed operation order.  The cell size is the widest grid box of the step
// (times 1.01), so two overlapping grid boxes always sit in the same or in adjacent cells.
// A scene caps it at creation (grid_cell_cap: the widest box at rest, or below it when a few
// much wider boxes make that cheaper): a body whose inflated box is wider than the cap this
// step -- one flagged larger than the scene's `large_he`, or one moving fast -- goes off the
// grid and is tested against all bodies instead of widening every cell.  Scenes with such
// bodies by design use a multilevel grid instead (below), where a fast body moves up a level
// rather than off the grid.  Bodies are counting-sorted into hash buckets; each body scans
// the 27 cells around its own, each bucket once (cells that share one never duplicate a pair),
// and keeps the neighbours j > i whose boxes overlap, that share its group and are not joined to
// it by a user bond.  Each body's partner list is sorted, so the final
// list is the sorted set of overlapping pairs -- independent of bucket order.
//
// Narrow phase: box-box contact manifold (reference face by separating axis over the six
// face normals, incident face clipped against the reference face's side planes) and
// corner-vs-ground-plane contacts, all in single precision with the same fixed operation
// order as the specification in the tests' oracle; contacts are written in pair order
// (then ground, in body order) through prefix sums, so the contact list is deterministic.
#include <algorithm>

#include "contacts.cuh"
#include "csr.cuh"
#include "sort_slices.cuh"
#include "predict.cuh"

namespace pabd {

constexpr int CT = 256;  // threads per block for per-body / per-pair kernels
__global__ void k_aabb(Dev d) {
    pdl_enter();
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= d.N) return;
    aabb_body(d, b);
}

__device__ __forceinline__ int cell_coord(float x, float inv_cs) {
    float t = floorf(x * inv_cs);
    t = fminf(fmaxf(t, -1048576.f), 1048576.f);
    return (int)t;
}

__device__ __forceinline__ int cell_hash(unsigned x, unsigned y, unsigned z, int bits) {
    unsigned h = x * 73856093u ^ y * 19349663u ^ z * 83492791u;
    h ^= h >> 16;
    h *= 0x7feb352du;
    h ^= h >> 15;
    return (int)(h & ((1u << bits) - 1u));
}

// Cell size of grid level lv: the widest box of that level or any finer one (times 1.01), so
// that a box of one level and a box of a coarser level that overlap sit in the same or in
// adjacent cells of the coarser level.
__device__ __forceinline__ float level_cell(const Dev& d, int lv) {
    float cs = __int_as_float(d.ctr[C_CELLBITS]);
    if (lv >= 1) cs = fmaxf(cs, __int_as_float(d.ctr[C_CELLBITS1]));
    if (lv >= 2) cs = fmaxf(cs, __int_as_float(d.ctr[C_CELLBITS2]));
    return cs;
}

// bucket of cell (x, y, z) of level lv for the bodies of a group (levels apart: coordinates stay
// within +-2^20; groups apart, so that scenes in the same place do not fill each other's buckets:
// 24 piles of 8000 boxes counted their pairs in 27 us, now 11)
__device__ __forceinline__ int level_hash(int x, int y, int z, int lv, int group, int bits) {
    return cell_hash((unsigned)x + ((unsigned)lv << 22) + (unsigned)group * 0x2545f491u, (unsigned)y, (unsigned)z, bits);
}

__global__ void k_cells(Dev d) {
    pdl_enter();
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= d.N) return;
    if (d.cell[b].w < 0) return;  // off the grid (k_aabb)
    const int lv = d.blevel ? d.blevel[b] : 0;
    const float cs = level_cell(d, lv);
    float inv = 1.0f / cs;
    float4 a = d.qn[3 * b];
    int x = cell_coord(a.x, inv), y = cell_coord(a.y, inv), z = cell_coord(a.z, inv);
    int hb = level_hash(x, y, z, lv, d.group[b], d.table_bits);
    d.cell[b] = make_int4(x, y, z, hb);
    atomicAdd(&d.bucket_cnt[hb], 1);
}

// Bodies into their buckets, with a copy of what the pair test reads -- the box, the group, the id,
// level and pinned flag -- in one 32-byte record (Dev::brec): the candidates lie anywhere, and
// waiting for them is most of what the pair search costs (262 144 boxes: 9 of 20 cycles per issued
// instruction at 42 warps per SM, L1 68 % busy).  (The cell, too, made it three sectors; that no
// partner is met twice is the scan's business, which takes each bucket once.  262 144 boxes: pairs
// counted in 164 us, now 132; a quadruped on 50 000 grains 77, now 62.)
constexpr int REC_ID_BITS = 28;  // (a body takes kilobytes of device memory: more do not fit)
__device__ __forceinline__ int rec_id(float w) { return __float_as_int(w) & ((1 << REC_ID_BITS) - 1); }
__device__ __forceinline__ int rec_level(float w) { return (__float_as_int(w) >> REC_ID_BITS) & 7; }
__device__ __forceinline__ bool rec_pinned(float w) { return __float_as_int(w) < 0; }
__global__ void k_bucket_fill(Dev d) {
    pdl_enter();
    int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= d.N) return;
    const int4 c = d.cell[b];
    if (c.w < 0) return;
    const int pos = d.bucket_off[c.w] + atomicAdd(&d.bucket_cur[c.w], 1);
    const float4 lo = d.lo[b], hi = d.hi[b];
    const unsigned id = (unsigned)b | (unsigned)(d.blevel ? d.blevel[b] : 0) << REC_ID_BITS | (d.bflags[b] & BF_PINNED ? 1u << 31 : 0u);
    d.brec[2 * pos] = make_float4(lo.x, lo.y, lo.z, __uint_as_float(id));
    d.brec[2 * pos + 1] = make_float4(hi.x, hi.y, hi.z, __int_as_float(d.group[b]));
}

// Calls test(record lo, record hi) for every body in the buckets of the 27 cells around (x, y, z)
// of level l (the cell of a warp's lane c: dx, dy, dz = c % 3 - 1, c / 3 % 3 - 1, c / 9 - 1), each
// bucket once: of the lanes whose cells share one, the first scans it.  Whatever else a bucket
// holds is for the test to turn down; a box that overlaps one centred in (x, y, z) is in the 27.
// All lanes of the warp call it together.
template <class F>
__device__ __forceinline__ void scan_cells(const Dev& d, int x, int y, int z, int l, int group, int lane, F&& test) {
    if (lane >= 27) return;
    const int hb = level_hash(x + lane % 3 - 1, y + (lane / 3) % 3 - 1, z + lane / 9 - 1, l, group, d.table_bits);
    const int s = d.bucket_off[hb];
    int e = d.bucket_off[hb + 1];
    if (__match_any_sync(0x07ffffffu, hb) & ((1u << lane) - 1u)) e = s;
    for (int k = s; k < e; k += 2) {  // (two records in flight)
        const int k1 = min(k + 1, e - 1);
        const float4 l0 = d.brec[2 * k], h0 = d.brec[2 * k + 1], l1 = d.brec[2 * k1], h1 = d.brec[2 * k1 + 1];
        test(l0, h0);
        if (k + 1 < e) test(l1, h1);
    }
}

// Pair finding, one warp per body i.  A grid body: lane c < 27 scans neighbour cell c
// (dx, dy, dz = c % 3 - 1, c / 3 % 3 - 1, c / 9 - 1), then the lanes stride over the large
// bodies; the partners are written at per-lane offsets and the body's slice is sorted.  A
// large body: the warp sweeps j = i+1 .. N-1 in chunks of 32 and compacts with a ballot,
// which keeps j ascending.  Accepted partners: j > i, same group, not both pinned, inflated
// boxes overlap, not joined by a user bond.
template <class F>
__device__ __forceinline__ int lane_partners(const Dev& d, int i, int lane, F&& f) {
    const int gi = d.group[i], fi = d.bflags[i];
    const float4 li = d.lo[i], hi_ = d.hi[i];
    const int4 ci = d.cell[i];
    int n = 0;
    scan_cells(d, ci.x, ci.y, ci.z, 0, gi, lane, [&](const float4& lj, const float4& hj) {
        const int j = rec_id(lj.w);
        if (j <= i || __float_as_int(hj.w) != gi || ((fi & BF_PINNED) && rec_pinned(lj.w))) return;
        if (!overlap(li, hi_, lj, hj) || adj_has(d, i, j)) return;
        f(j, n);
        ++n;
    });
    const int nl = d.large_ids ? d.ctr[C_NLARGE] : 0;
    for (int k = lane; k < nl; k += 32) {
        const int j = d.large_ids[k];
        if (j > i && pair_ok(d, i, j, gi, fi, li, hi_)) { f(j, n); ++n; }
    }
    return n;
}

__device__ __forceinline__ int warp_sum(int v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ int warp_excl(int v, int lane) {
    int inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    return inc - v;
}

// Counts body i's partners (a warp per body) and, when there are at most PAIR_LIST of them and no
// lane found more than four, leaves them in order in its list, so that writing the pairs is a
// copy; a body with partners and no list is noted for the writing pass (Dev::pair_rest).
__global__ void __launch_bounds__(CT) k_pair_count(Dev d) {
    pdl_enter();
    __shared__ int found[CT / 32][PAIR_LIST];
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (i >= d.N) return;
    int n = 0;
    bool listed = false;
    const int gi = d.group[i], fi = d.bflags[i];
    if (d.cell[i].w < 0) {
        const float4 li = d.lo[i], hi_ = d.hi[i];
        for (int j0 = i + 1; j0 < d.N; j0 += 32) {
            const int j = j0 + lane;
            n += (j < d.N && pair_ok(d, i, j, gi, fi, li, hi_)) ? 1 : 0;
        }
        n = warp_sum(n);
    } else {
        int id[4];
        const int mine = lane_partners(d, i, lane, [&](int j, int k) {
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (k == c) id[c] = j;
        });
        n = warp_sum(mine);
        listed = n > 0 && n <= PAIR_LIST && !__any_sync(0xffffffffu, mine > 4);
        if (listed) {
            const int at = warp_excl(mine, lane);
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (c < mine) found[w][at + c] = id[c];
            __syncwarp();
            const int v = lane < n ? found[w][lane] : 0x7fffffff;
            const int r = warp_rank32(v, n, lane);
            if (r >= 0) d.pair_list[(size_t)i * PAIR_LIST + r] = v;
        }
    }
    if (lane == 0) {
        d.pair_cnt[i] = n;
        if (n > 0 && !listed) {  // found again when written
            d.pair_list[(size_t)i * PAIR_LIST] = -1;
            d.pair_rest[atomicAdd(&d.ctr[C_NREST], 1)] = i;
        }
    }
}

// The pairs of a body that was not listed while counting, by a warp: an off-grid body's (the
// whole rest in order), or those of a body with many partners (found again, in any order, then
// sorted; a slice that the capacity cuts keeps any of them).  cur: a word of shared memory.
__device__ __forceinline__ void write_unlisted_pairs(const Dev& d, int i, int lane, int* cur) {
    const int s = d.pair_off[i], cap = d.cap_pairs;
    const int gi = d.group[i], fi = d.bflags[i];
    if (d.cell[i].w < 0) {
        int pos = s;
        const float4 li = d.lo[i], hi_ = d.hi[i];
        for (int j0 = i + 1; j0 < d.N; j0 += 32) {
            const int j = j0 + lane;
            const bool ok = j < d.N && pair_ok(d, i, j, gi, fi, li, hi_);
            const unsigned bal = __ballot_sync(0xffffffffu, ok);
            const int at = pos + __popc(bal & ((1u << lane) - 1u));
            if (ok && at < cap) d.pairs[at] = make_int2(i, j);
            pos += __popc(bal);
        }
        return;
    }
    if (lane == 0) *cur = s;
    __syncwarp();
    lane_partners(d, i, lane, [&](int j, int) {
        const int at = atomicAdd(cur, 1);
        if (at < cap) d.pairs[at] = make_int2(i, j);
    });
    __syncwarp();
    const int e = min(d.pair_off[i + 1], cap), n = e - s;
    if (n <= 32) {  // the slice sorted by j: each partner's rank among the slice
        const int j = lane < n ? d.pairs[s + lane].y : 0x7fffffff;
        const int r = warp_rank32(j, n, lane);
        __syncwarp();
        if (r >= 0) d.pairs[s + r] = make_int2(i, j);
    } else if (n <= 64) {  // by the bitonic network in registers
        int v0 = (2 * lane < n) ? d.pairs[s + 2 * lane].y : 0x7fffffff;
        int v1 = (2 * lane + 1 < n) ? d.pairs[s + 2 * lane + 1].y : 0x7fffffff;
        warp_sort64(v0, v1, lane);
        __syncwarp();
        if (2 * lane < n) d.pairs[s + 2 * lane] = make_int2(i, v0);
        if (2 * lane + 1 < n) d.pairs[s + 2 * lane + 1] = make_int2(i, v1);
    } else if (lane == 0) {
        for (int a = s + 1; a < e; ++a) {  // insertion sort of the slice by j
            int2 v = d.pairs[a];
            int b = a - 1;
            while (b >= s && d.pairs[b].y > v.y) { d.pairs[b + 1] = d.pairs[b]; --b; }
            d.pairs[b + 1] = v;
        }
    }
}

// Copies the listed partners, WRITE_LANES lanes per body; then the warps share out the bodies that
// were not listed, each its first by its index and the next ones from a counter (an off-grid body's
// sweep takes the longer the smaller its id).  (A warp per body that replayed every lane's finds
// took 120 us for 262 144 boxes, and without room for them, in the allocation-free call, it scanned
// the cells twice more: 50 us for 16 384 boxes.  Now 13 and 13.  Left to the warps that copy around
// them, eight to a warp, the unlisted ones were the launch's length: detection of 60 000 cubes of
// which 568 are off the grid 3077 us, now 1850, of 1000 crowded ones, 42 partners each, 1294, now
// 350.)
constexpr int WRITE_LANES = 4;
__global__ void __launch_bounds__(CT) k_pair_write(Dev d) {
    pdl_enter();
    __shared__ int cur[CT / 32];
    const int t = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const int i = t / WRITE_LANES, sub = t % WRITE_LANES, cap = d.cap_pairs;
    if (i < d.N) {
        const int s = d.pair_off[i], n = d.pair_off[i + 1] - s;
        const int* list = d.pair_list + (size_t)i * PAIR_LIST;
        if (n > 0 && list[0] >= 0)
            for (int k = sub; k < n; k += WRITE_LANES)
                if (s + k < cap) d.pairs[s + k] = make_int2(i, list[k]);
    }
    const int rest = d.ctr[C_NREST], warps = gridDim.x * (CT / 32);
    for (int r = t >> 5; r < rest;) {
        write_unlisted_pairs(d, d.pair_rest[r], lane, &cur[threadIdx.x >> 5]);
        if (rest <= warps) break;
        if (lane == 0) r = warps + atomicAdd(&d.ctr[C_REST_NEXT], 1);
        r = __shfl_sync(0xffffffffu, r, 0);
    }
    if (t == 0) {
        const int tot = d.pair_off[d.N];
        if (tot > cap) latch_status(d, ST_CAPACITY);
        d.ctr[C_NPAIRS] = min(tot, cap);
    }
}

// ---- multilevel grid (Dev::multilevel: scenes with bodies of very different widths) ----
//
// A grid body sits at the first level l whose cap, cell cap x 4^l, holds its box (NLEV
// levels); a wider one, or one flagged large, goes off the grid.  Level l's cell is the widest
// box of that level or a finer one, so a body meets every overlapping body of its own or a
// coarser level in the 27 cells around its centre at that level.  Each body therefore scans
// its own level (keeping partners j > i, as the single-level grid does) and every non-empty
// coarser level (keeping all partners): a partner j > i joins i's slice, a partner j < i is
// delivered to j's slice (counted, then placed, with atomics).  The off-grid bodies take all
// j > i by a block-parallel sweep (k_offgrid_pairs) and the grid bodies test the off-grid
// list for j > i.  Every slice is then sorted (launch_pair_sort), so the list is again the
// sorted set of overlapping pairs whatever the order of the atomics.

template <class Own, class Deliver>
__device__ __forceinline__ int lane_partners_ml(const Dev& d, int i, int lane, Own&& own, Deliver&& deliver) {
    const int gi = d.group[i], fi = d.bflags[i];
    const int lvi = d.blevel[i];
    const float4 li = d.lo[i], hi_ = d.hi[i];
    const int4 ci = d.cell[i];
    const float4 pos = d.qn[3 * i];
    int n = 0;
    // its own level, then each coarser one that holds any body
    for (int l = lvi; l < NLEV; ++l) {
        int bx = ci.x, by = ci.y, bz = ci.z;
        if (l != lvi) {
            if (d.ctr[C_CELLBITS1 + l - 1] == 0) continue;
            const float inv = 1.0f / level_cell(d, l);
            bx = cell_coord(pos.x, inv); by = cell_coord(pos.y, inv); bz = cell_coord(pos.z, inv);
        }
        scan_cells(d, bx, by, bz, l, gi, lane, [&](const float4& lj, const float4& hj) {
            const int j = rec_id(lj.w);
            if (rec_level(lj.w) != l || j == i) return;
            if (l == lvi && j < i) return;  // same level: found by the smaller id
            if (__float_as_int(hj.w) != gi || ((fi & BF_PINNED) && rec_pinned(lj.w))) return;
            if (!overlap(li, hi_, lj, hj) || adj_has(d, i, j)) return;
            if (j > i) { own(j, n); ++n; }
            else deliver(j);
        });
        __syncwarp();
    }
    const int nl = d.ctr[C_NLARGE];
    for (int k = lane; k < nl; k += 32) {
        const int j = d.large_ids[k];
        if (j > i && pair_ok(d, i, j, gi, fi, li, hi_)) { own(j, n); ++n; }
    }
    return n;
}

// counts: pair_cnt (zeroed before) gains each body's own partners and the deliveries to it
__global__ void k_ml_pair_count(Dev d) {
    pdl_enter();
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= d.N || !d.p.body_contacts || d.cell[i].w < 0) return;
    int* st = d.pair_stash + (size_t)(32 * i + lane) * PAIR_STASH;
    int tot = 0;  // entries: own partners and deliveries, in the order found
    int n = lane_partners_ml(d, i, lane,
        [&](int j, int) { if (tot < PAIR_STASH) st[tot] = j; ++tot; },
        [&](int j) {
            atomicAdd(&d.pair_cnt[j], 1);
            if (tot < PAIR_STASH) st[tot] = j | STASH_DELIVER;
            ++tot;
        });
    d.lane_cnt[32 * i + lane] = n;
    d.lane_tot[32 * i + lane] = tot;
    n = warp_sum(n);
    if (lane == 0) {
        d.pair_own[i] = n;
        atomicAdd(&d.pair_cnt[i], n);
    }
}

// partner ids into pair_j: own partners at per-lane offsets, deliveries after the receiver's
// own ones through its cursor (pair_cur, zeroed before)
__global__ void k_ml_pair_write(Dev d) {
    pdl_enter();
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= d.N) return;
    const int cap = d.cap_pairs;
    if (d.p.body_contacts && d.cell[i].w >= 0) {
        const int base = d.pair_off[i] + warp_excl(d.lane_cnt[32 * i + lane], lane);
        auto own = [&](int j, int k) { if (base + k < cap) d.pair_j[base + k] = j; };
        auto deliver = [&](int j) {
            const int at = d.pair_off[j] + d.pair_own[j] + atomicAdd(&d.pair_cur[j], 1);
            if (at < cap) d.pair_j[at] = i;
        };
        const int tot = d.lane_tot[32 * i + lane];
        // the entries found while counting, unless a lane of the warp found too many (the scan is the
        // whole warp's)
        if (!__any_sync(0xffffffffu, tot > PAIR_STASH)) {
            const int* st = d.pair_stash + (size_t)(32 * i + lane) * PAIR_STASH;
            int k = 0;
            for (int t = 0; t < tot; ++t) {
                const int v = st[t];
                if (v & STASH_DELIVER) deliver(v & ~STASH_DELIVER);
                else own(v, k++);
            }
        } else {
            lane_partners_ml(d, i, lane, own, deliver);
        }
    }
    if (i == d.N - 1 && lane == 0) {
        const int tot = d.pair_off[d.N];
        if (tot > cap) latch_status(d, ST_CAPACITY);
        d.ctr[C_NPAIRS] = min(tot, cap);
    }
}

// Pairs of the off-grid bodies: body i of the off-grid list against every j > i, by 32 warps, warp
// w taking the w-th of 32 contiguous runs of (i, N), so the warps' hits concatenated in warp order
// keep the slice sorted by j.  The warps of all off-grid bodies are spread over the grid and each
// keeps four chunks of 32 bodies in flight (32 warps of one block read 2 MB per body through one
// SM: 13 off-grid bodies among 50 077 took 140 us for both passes, now 29; spread but with the
// pair filter's loads one after the other 103).
// WRITE = false counts (into pair_cnt[i], and each warp's count in lane_cnt[32 i + w]); true
// stores the partners into pair_j.
constexpr int OFF_T = 128;

template <bool WRITE>
__global__ void __launch_bounds__(OFF_T) k_offgrid_pairs(Dev d) {
    pdl_enter();
    if (!d.p.body_contacts) return;
    const int nl = d.ctr[C_NLARGE];
    const int lane = threadIdx.x & 31, cap = d.cap_pairs;
    // (neighbouring tasks of one body on different SMs)
    const int warp0 = (threadIdx.x >> 5) * gridDim.x + blockIdx.x, warps = gridDim.x * (OFF_T / 32);
    for (int task = warp0; task < 32 * nl; task += warps) {
        const int i = d.large_ids[task >> 5], w = task & 31;
        const int gi = d.group[i], fi = d.bflags[i];
        const float4 li = d.lo[i], hi_ = d.hi[i];
        const int len = (((d.N - i - 1) + 31) / 32 + 31) & ~31;  // per warp, a multiple of 32
        const int j_beg = i + 1 + w * len, j_end = min(d.N, j_beg + len);
        int pos = 0;
        if (WRITE) {
            int before = lane < w ? d.lane_cnt[32 * i + lane] : 0;
            pos = d.pair_off[i] + warp_sum(before);
        }
        for (int j0 = j_beg; j0 < j_end; j0 += 4 * 32) {
            bool ok[4];
            float4 lj[4], hj[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {  // (the boxes of all four chunks before any test)
                const int j = min(j0 + 32 * k + lane, d.N - 1);
                lj[k] = d.lo[j];
                hj[k] = d.hi[j];
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int j = j0 + 32 * k + lane;
                ok[k] = j < j_end && overlap(li, hi_, lj[k], hj[k]) && d.group[j] == gi &&
                        !((fi & BF_PINNED) && (d.bflags[j] & BF_PINNED)) && !adj_has(d, i, j);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const unsigned bal = __ballot_sync(0xffffffffu, ok[k]);
                if (WRITE) {
                    const int at = pos + __popc(bal & ((1u << lane) - 1u));
                    if (ok[k] && at < cap) d.pair_j[at] = j0 + 32 * k + lane;
                }
                pos += __popc(bal);
            }
        }
        if (!WRITE && lane == 0) {
            d.lane_cnt[32 * i + w] = pos;
            if (pos > 0) atomicAdd(&d.pair_cnt[i], pos);
        }
    }
}

// ---- narrow phase ----

// contacts of a tile of k_narrow's items, counted again by a warp (out of line: hardly ever wanted)
__device__ __noinline__ int tile_contacts(const Dev& d, int tile, int np) {
    int n = 0;
    for (int t = threadIdx.x & 31; t < NARROW_T; t += 32) {
        const int item = tile * NARROW_T + t;
        if (item < np + d.N) n += narrow_item_contacts(d, item, np);
    }
    return __reduce_add_sync(0xffffffffu, n);
}

// The whole narrow phase in one pass.  Items [0, np) are this step's pairs, items np + b the ground
// corners of body b; a tile of NARROW_T items is a block's, a thread each.  The block keeps its
// items' contacts in shared memory while it learns how many contacts precede its tile -- the
// tiles' counts are published as they are known, and a tile adds up its predecessors' from the
// nearest one whose whole prefix is known (decoupled look-back, Merrill and Garland 2016) -- and
// then writes them, a thread per contact.  Contacts come out in item order whatever the order of
// the blocks.  Tiles are taken from a counter, so a tile's predecessors are running or done; the
// wait for them is bounded all the same, and where it runs out the waiting warp counts the missing
// tile's contacts itself (tile_contacts): a late tile costs time, and every contact keeps its one
// slot.  The bodies' bond ends are counted on the way, on top of their static ones.
//
// It replaced a counting pass, two prefix sums, a pass that derived every manifold again to write
// it, and the count of bond ends.  Bound by latency at 16 warps per SM (its 46 KB a block): the
// block's barriers, where a tile waits for its longest item and for the look-back (5.0 of 13 cycles
// per issued instruction on a pile), then the boxes' loads (3.7), the clipping's dependent steps
// and divergence (half the lanes idle on a settled bed).  532 325 pairs of a settled bed 115 us
// (counting 156 and writing 187 us; in one pass with the polygons in local memory 274), 258 048
// pairs of a pile, all touching, 78 us (57 and 90).
__global__ void __launch_bounds__(NARROW_T) k_narrow(const __grid_constant__ Dev d) {
    constexpr int T = NARROW_T, MAXC = 8;
    __shared__ float corners[2 * MAXC * 5 * T];  // the items' polygons, then their contacts (SharedPoly)
    __shared__ float nrm[3][T], wgt[T], dht[T], face_x[T];
    __shared__ int bi[T], bj[T];                 // bj < 0: ground contacts
    __shared__ unsigned char face[T], buf[T];    // incident face's axis; the buffer that holds the contacts
    __shared__ unsigned short map[MAXC * T];  // contact of the tile -> item + T * its number there
    __shared__ int wsum[T / 32], s_tile, s_before;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    pdl_enter();
    const int np = d.ctr[C_NPAIRS], items = np + d.N, ntile = (items + T - 1) / T;
    const unsigned limit = *d.wait_limit;
    volatile unsigned long long* const state = d.tile_state;
    constexpr unsigned long long PART = 1ull << 32, WHOLE = 2ull << 32;  // count of the tile, of all up to it
    for (;;) {
        if (t == 0) s_tile = atomicAdd(&d.ctr[C_NARROW_NEXT], 1);
        __syncthreads();
        const int tile = s_tile;
        if (tile >= ntile) return;
        const int item = tile * T + t;
        int n = 0;
        SharedPoly<T> poly{corners + t};
        if (item < np) {
            const int2 pr = d.pairs[item];
            FBox fa, fb;
            load_box(d, pr.x, fa);
            load_box(d, pr.y, fb);
            Manifold mf;
            int out = 0;
            n = box_box(fa, fb, pr.x, pr.y, poly, mf, out, [&](const Corner& c, int k) { st_corner(poly, out, k, c); });
            if (n > 0) {
                bi[t] = mf.ii;
                bj[t] = mf.ir;
                buf[t] = (unsigned char)out;
                face[t] = (unsigned char)mf.ki;
                face_x[t] = mf.xk;
#pragma unroll
                for (int k = 0; k < 3; ++k) nrm[k][t] = mf.N[k];
            }
        } else if (item < items && d.p.has_ground && !(d.bflags[item - np] & BF_PINNED)) {
            // (a ground contact's corner by number: its coordinates are the half extents, signed)
            FBox fa;
            load_box(d, item - np, fa);
            n = ground_corners(d, fa, item - np, [&](int, int corner, const float*, const float* anc, int k) {
                st_corner(poly, 0, k, Corner{{anc[0], anc[1], anc[2]}, __int_as_float(corner), 0.f});
            });
            if (n > 0) {
                bi[t] = item - np;
                bj[t] = -1;
                buf[t] = 0;
#pragma unroll
                for (int k = 0; k < 3; ++k) nrm[k][t] = fa.he[k];
            }
        }
        int inc = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        int start = inc - n, total = 0;
#pragma unroll
        for (int k = 0; k < T / 32; ++k) {
            if (k < warp) start += wsum[k];
            total += wsum[k];
        }
        if (warp == 0) {  // publish, and look back
            int before = 0;
            if (tile > 0) {
                if (lane == 0) state[tile] = PART | (unsigned)total;
                for (int first = tile - 1;; first -= 32) {  // tiles first, first - 1, ...: one per lane
                    const int k = first - lane;
                    unsigned long long v = WHOLE;  // (before tile 0: nothing)
                    unsigned whole, late;  // lanes with a whole prefix; unpublished ones before the nearest
                    int last;              // the nearest lane with a whole prefix
                    for (unsigned polls = 0;; ++polls) {
                        if (k >= 0) v = state[k];
                        whole = __ballot_sync(0xffffffffu, (v >> 32) == 2);
                        last = whole ? __ffs(whole) - 1 : 31;
                        late = __ballot_sync(0xffffffffu, v == 0 && lane <= last);
                        if (late == 0 || polls >= limit) break;
                    }
                    for (; late; late &= late - 1) {
                        const int l = __ffs(late) - 1, n = tile_contacts(d, first - l, np);
                        if (lane == l) v = PART | (unsigned)n;
                    }
                    int c = lane <= last ? (int)(unsigned)v : 0;
                    c = __reduce_add_sync(0xffffffffu, c);
                    before += c;
                    if (whole) break;
                }
            }
            if (lane == 0) {
                state[tile] = WHOLE | (unsigned)(before + total);
                s_before = before;
            }
        }
        for (int k = 0; k < n; ++k) map[start + k] = (unsigned short)(t + T * k);
        if (n > 0) {
            const int i = bi[t], j = bj[t];
            wgt[t] = contact_weight(d, i, j);
            dht[t] = pair_dhat(d, i, j);
        }
        __syncthreads();
        const int before = s_before;
        for (int c = t; c < total; c += T) {
            const int o = map[c] % T, k = map[c] / T;
            SharedPoly<T> his{corners + o};
            const Corner p = ld_corner(his, buf[o], k);
            const bool ground = bj[o] < 0;
            float x[3];
            if (ground) {
                const int corner = __float_as_int(p.xa);
#pragma unroll
                for (int a = 0; a < 3; ++a) x[a] = (corner >> a) & 1 ? nrm[a][o] : -nrm[a][o];
            } else {
                corner_point(face[o], face_x[o], p.xa, p.xb, x);
            }
            Contact q;
            q.m = make_int4(bi[o], bj[o], ground ? K_GROUND : K_CONTACT, 0);
            q.xi = make_float4(x[0], x[1], x[2], wgt[o]);
            q.xj = make_float4(p.u[0], p.u[1], p.u[2], dht[o]);
            q.bn = ground ? make_float4(d.p.gn[0], d.p.gn[1], d.p.gn[2], d.p.mu)
                          : make_float4(nrm[0][o], nrm[1][o], nrm[2][o], d.p.mu);
            store_contact(d, before + c, q);
        }
        if (n > 0) {  // (those with room)
            const int m = min(n, d.cap_contacts - (before + start));
            if (m > 0) {
                if (end_live(d, bi[t])) atomicAdd(&d.end_cnt[bi[t]], m);
                if (end_live(d, bj[t])) atomicAdd(&d.end_cnt[bj[t]], m);
            }
        }
        if (tile == ntile - 1 && t == 0) {
            int nk = before + total;
            if (nk > d.cap_contacts) { latch_status(d, ST_CAPACITY); nk = d.cap_contacts; }
            d.ctr[C_NCONTACTS] = nk;
            d.ctr[C_NBONDS] = d.Nc + nk;
        }
        __syncthreads();  // the tile's shared memory is reused
    }
}

static inline int nblk(int n) { return (n + CT - 1) / CT > 0 ? (n + CT - 1) / CT : 1; }

// ---- the front of a step in scenes whose only contacts are with the ground ----
//
// Three launches in place of the AABB, ground-count, scan, contact-write, CSR and predictor
// kernels (the same arithmetic, fewer launch boundaries): k_ground_prelude per body, the scan of
// its blocks' totals, k_ground_bonds_csr per static end and per body.

// per body: AABB and inflation, ground contacts counted, predictor; per block of CT bodies, the
// exclusive prefix of the counts inside the block (Dev::gnd_loc) and their total (Dev::gnd_blk)
__global__ void __launch_bounds__(CT) k_ground_prelude(Dev d) {
    pdl_enter();
    __shared__ int wsum[CT / 32];
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    int n = 0;
    if (b < d.N) {
        aabb_body(d, b);
        if (d.p.has_ground && !(d.bflags[b] & BF_PINNED)) {
            FBox fa;
            load_box(d, b, fa);
            n = ground_corners(d, fa, b, [](int, int, const float*, const float*, int) {});
        }
        predict_body(d, b);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += t;
    }
    if (lane == 31) wsum[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int w = lane < CT / 32 ? wsum[lane] : 0;
#pragma unroll
        for (int o = 1; o < CT / 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += t;
        }
        if (lane < CT / 32) wsum[lane] = w;
    }
    __syncthreads();
    if (b < d.N) d.gnd_loc[b] = (warp ? wsum[warp - 1] : 0) + inc - n;
    if (threadIdx.x == 0) d.gnd_blk[blockIdx.x] = wsum[CT / 32 - 1];
}

// ground contacts of the bodies before b (b <= N), from the prelude's block prefixes and the
// scan of its block totals (Dev::gnd_bof, whose last entry is the total)
__device__ __forceinline__ int gnd_prefix(const Dev& d, int b) {
    return b < d.N ? d.gnd_bof[b / CT] + d.gnd_loc[b] : d.gnd_bof[(d.N + CT - 1) / CT];
}

// After the scan: items [0, Ns) are the static ends in Dev::sta_id order -- end e of body b
// takes slot e + g0(b), g0(b) = the ground contacts of the bodies before b (at most the
// contact capacity); items Ns + b, b <= N, the bodies -- slice start sta_off[b] + g0(b), the
// body's ground contacts written as bonds Nc + g0(b) + k and given slots after its static ends,
// and the heavy list.  The same CSR, in the same order, as counting, filling and sorting it.
template <int WANT>
__global__ void k_ground_bonds_csr(Dev d) {
    pdl_enter();
    const int nb = d.N, Ns = d.sta_off[nb], cap = d.cap_contacts;
    const int items = Ns + nb + 1;
    for (int tt = blockIdx.x * blockDim.x + threadIdx.x; tt < items; tt += gridDim.x * blockDim.x) {
        if (tt < Ns) {
            const int b = d.sta_body[tt];
            const int slot = tt + min(gnd_prefix(d, b), cap);
            place_end<WANT>(d, d.sta_id[tt], slot);
            continue;
        }
        const int b = tt - Ns;
        const int gb = gnd_prefix(d, b), g0 = min(gb, cap);
        d.end_off[b] = d.sta_off[b] + g0;
        if (b == nb) continue;
        const int gn = min(gnd_prefix(d, b + 1), cap) - g0;
        if (gn > 0) {
            FBox fa;
            load_box(d, b, fa);
            const int p0 = d.sta_off[b + 1] + g0;
            ground_corners(d, fa, b, [&](int i, int, const float* xi, const float* xj, int k) {
                if (k >= gn) return;  // past the contact capacity (latched below)
                const Contact c = write_contact(d, g0 + k, K_GROUND, i, -1, xi, xj, d.p.gn);
                place_end<WANT>(d, 2 * (d.Nc + g0 + k), p0 + k, c.m, c.xi, c.xj, c.bn);
            });
        }
        if (d.sta_off[b + 1] - d.sta_off[b] + gn > HEAVY_ENDS) d.heavy[atomicAdd(&d.ctr[C_NHEAVY], 1)] = b;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        int nk = gnd_prefix(d, nb);
        if (nk > cap) { latch_status(d, ST_CAPACITY); nk = cap; }
        d.ctr[C_NCONTACTS] = nk;
        d.ctr[C_NBONDS] = d.Nc + nk;
    }
}

void launch_ground_front(const Dev& d, cudaStream_t st, long long* launches) {
    launch_pdl(k_ground_prelude, dim3(nblk(d.N)), dim3(CT), 0, st, d);
    scan_exclusive(d.gnd_blk, d.gnd_bof, nblk(d.N), d.scan_scratch, st, launches);
    with_want(d.csr_want, [&](auto w) {
        launch_pdl(k_ground_bonds_csr<decltype(w)::value>, dim3(stride_grid((long long)d.cap_ends + d.N + 1, CT)), dim3(CT), 0, st, d);
    });
    *launches += 2;
}

// k_pair_write's grid: WRITE_LANES threads per body, and at least a warp per body while all are
// resident at once
static inline int pair_write_blocks(int n) { return std::max(nblk(n * WRITE_LANES), stride_grid(32ll * n, CT)); }

// The broad phase alone (bucket / counter resets, AABBs, grid, sorted pair list), on whatever
// buffers `d` points at; used by the allocation-free entry point.
void launch_broadphase(const Dev& d, cudaStream_t st, long long* launches) {
    const int T = 1 << d.table_bits;
    cudaMemsetAsync(d.bucket_cnt, 0, sizeof(int) * T, st);
    cudaMemsetAsync(d.bucket_cur, 0, sizeof(int) * T, st);
    cudaMemsetAsync(d.ctr, 0, sizeof(int) * C_COUNT, st);
    launch_pdl(k_aabb, dim3(nblk(d.N)), dim3(CT), 0, st, d);
    launch_pdl(k_cells, dim3(nblk(d.N)), dim3(CT), 0, st, d);
    scan_exclusive(d.bucket_cnt, d.bucket_off, T, d.scan_scratch, st, launches);
    launch_pdl(k_bucket_fill, dim3(nblk(d.N)), dim3(CT), 0, st, d);
    const int wblk = (d.N * 32 + CT - 1) / CT > 0 ? (d.N * 32 + CT - 1) / CT : 1;
    launch_pdl(k_pair_count, dim3(wblk), dim3(CT), 0, st, d);
    scan_exclusive(d.pair_cnt, d.pair_off, d.N, d.scan_scratch, st, launches);
    launch_pdl(k_pair_write, dim3(pair_write_blocks(d.N)), dim3(CT), 0, st, d);
    *launches += 5;
}

// (the counters and buckets it accumulates into are zeroed by launch_step_reset)
void launch_collision(const Dev& d, cudaStream_t st, long long* launches) {
    if (!d.p.body_contacts) {  // ground contacts only: no broad phase
        launch_ground_front(d, st, launches);
        return;
    }
    launch_pdl(k_aabb, dim3(nblk(d.N)), dim3(CT), 0, st, d);
    *launches += 1;
    if (d.p.broadphase == 1) {
        launch_lbvh_pairs(d, st, launches);
    } else {
        const int T = 1 << d.table_bits;
        launch_pdl(k_cells, dim3(nblk(d.N)), dim3(CT), 0, st, d);
        scan_exclusive(d.bucket_cnt, d.bucket_off, T, d.scan_scratch, st, launches);
        launch_pdl(k_bucket_fill, dim3(nblk(d.N)), dim3(CT), 0, st, d);
        const int wblk = (d.N * 32 + CT - 1) / CT > 0 ? (d.N * 32 + CT - 1) / CT : 1;  // one warp per body
        if (d.multilevel) {
            launch_pdl(k_ml_pair_count, dim3(wblk), dim3(CT), 0, st, d);
            launch_pdl(k_offgrid_pairs<false>, dim3(resident_slots(4)), dim3(OFF_T), 0, st, d);
            scan_exclusive(d.pair_cnt, d.pair_off, d.N, d.scan_scratch, st, launches);
            launch_pdl(k_ml_pair_write, dim3(wblk), dim3(CT), 0, st, d);
            launch_pdl(k_offgrid_pairs<true>, dim3(resident_slots(4)), dim3(OFF_T), 0, st, d);
            *launches += 6;
            launch_pair_sort(d, st, launches);
        } else {
            launch_pdl(k_pair_count, dim3(wblk), dim3(CT), 0, st, d);
            scan_exclusive(d.pair_cnt, d.pair_off, d.N, d.scan_scratch, st, launches);
            launch_pdl(k_pair_write, dim3(pair_write_blocks(d.N)), dim3(CT), 0, st, d);
            *launches += 4;
        }
    }
    // resident blocks, or a block per tile where the capacities leave fewer
    const long long tiles = ((long long)d.cap_pairs + d.N + NARROW_T - 1) / NARROW_T;
    launch_pdl(k_narrow, dim3((unsigned)std::min<long long>(tiles, resident_slots(4))), dim3(NARROW_T), 0, st, d);
    *launches += 1;
}

}  // namespace pabd
