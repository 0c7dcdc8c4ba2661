// The front of a small scene's step in one launch of one block: counters, drive anchors, AABBs,
// pairs, contact manifolds, CSR of bond ends, predictor and augmented Lagrangian warm start.
//
// A scene of up to FRONT_N bodies spends these stages waiting: some twenty launches of two
// microseconds each, most of it launch and first loads.  Here a stage ends at a block barrier and
// what it hands to the next -- boxes, counts, offsets, pairs, end ids -- stays in shared memory
// (lists that outgrow it use the larger scenes' arrays).  The items of every stage are those of
// the kernels for larger scenes (contacts.cuh, csr.cuh, predict.cuh), except that the pairs come
// from testing every body against the later bodies of its group (a warp per body, partners found
// in order): the same sorted list of overlapping pairs as the grid's, without a grid.
//
// Bound by latency: first loads, block barriers and instruction fetch (every line of it runs
// once).  Front of the step against the kernels it replaces, both with 6 us of stage events: 8
// chained bodies 18.5 us (42.4), 40 of them 23.9 (42.3), a pile of 30 boxes 33.6 (52.5), of 128
// 44.8 (54.7), a slab under 121 boxes 45.1 (73.1); without body contacts, 19 bodies 18.3 (22.5)
// but 121 bodies 20.2 (18.5).  Spread over a cluster, with global memory between the stages, it
// took longer than the kernels from 250 bodies on.  (Not for a state with many contacts, see
// choose_front in pabd_capi.cu.)
#include "contacts.cuh"
#include "csr.cuh"
#include "predict.cuh"

namespace pabd {

constexpr int FT = 512;            // threads
constexpr int FRONT_N = 128;       // most bodies
constexpr int FRONT_N_GROUND = 32; // without body contacts, whose own front is three launches
constexpr int FRONT_PAIRS = 1024;  // pairs kept in shared memory
constexpr int FRONT_ENDS = 2048;   // bond ends kept in shared memory

// out[0..n] = exclusive prefix sums of in[0..n); every thread of the block calls it, and the
// results are visible to all once it returns
__device__ __forceinline__ void block_scan(const int* in, int* out, int n, int* smem) {
    constexpr int ITEMS = 4;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int carry = 0;
    for (int c0 = 0; c0 < n; c0 += FT * ITEMS) {
        const int base = c0 + t * ITEMS;
        int v[ITEMS], s = 0;
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            v[k] = base + k < n ? in[base + k] : 0;
            s += v[k];
        }
        int inc = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) smem[warp] = inc;
        __syncthreads();
        int before = 0, all = 0;
#pragma unroll
        for (int k = 0; k < FT / 32; ++k) {
            const int w = smem[k];
            if (k < warp) before += w;
            all += w;
        }
        int run = carry + before + inc - s;
#pragma unroll
        for (int k = 0; k < ITEMS; ++k) {
            if (base + k < n) out[base + k] = run;
            run += v[k];
        }
        carry += all;
        __syncthreads();  // smem is rewritten by the next pass
    }
    if (t == 0) out[n] = carry;
    __syncthreads();
}

template <int WANT>
__global__ void __launch_bounds__(FT, 1) k_front(Dev d0) {
    __shared__ float4 lo[FRONT_N], hi[FRONT_N];
    __shared__ int cnt[FRONT_N], off[FRONT_N + 1], gcnt[FRONT_N], goff[FRONT_N + 1], ends[FRONT_N], cur[FRONT_N];
    __shared__ int scan[FT / 32];
    // the lists, and once they are done with, the heavy bodies' ranking
    constexpr int LISTS = 4 * FRONT_PAIRS + 4 + FRONT_ENDS;
    __shared__ int2 list[(LISTS > 2 * LONG_SMEM ? LISTS : 2 * LONG_SMEM) / 2];
    int2* const pairs = list;
    int* const npc = reinterpret_cast<int*>(pairs + FRONT_PAIRS);
    int* const npc_off = npc + FRONT_PAIRS;
    int* const ids = npc_off + FRONT_PAIRS + 4;
    int* const key = reinterpret_cast<int*>(list);
    const int t = threadIdx.x, w = t >> 5, lane = t & 31, W = FT / 32;
    const int N = d0.N, cap = d0.cap_pairs;
    // the stages' view of the scene: what they hand on in shared memory
    Dev d = d0;
    d.gnd_cnt = gcnt;
    d.gnd_off = goff;
    d.end_cnt = ends;
    d.end_cur = cur;
    pdl_enter();

    if (t == 0) reset_counters(d);
    if (t < FRONT_N) {
        ends[t] = t < N ? d.sta_cnt[t] : 0;
        cur[t] = 0;
    }
    for (int k = t; k < 2 * END_BINS; k += FT) {
        d.bin_cnt[k] = 0;
        d.bin_cur[k] = 0;
    }
    for (int k = t; k < d.Ndrive; k += FT) drive_update(d, k);
    if (d.Nal)
        for (int k = t; k < d.Nc; k += FT) al_warm(d, k);
    __syncthreads();

    // (aabb_body's reductions expect the lanes of a warp below N)
    if (t < N) {
        aabb_body(d, t);
        lo[t] = d.lo[t];
        hi[t] = d.hi[t];
    } else if (t >= FRONT_N && t - FRONT_N < N) {
        predict_body(d, t - FRONT_N);
    }
    __syncthreads();

    int np = 0;
    if (d.p.body_contacts) {
        // pairs: body i against the later bodies of its group, counted and then written in order
        auto partners = [&](int i, auto&& chunk) {
            const int gi = d.group[i], fi = d.bflags[i], end = d.group_off[gi + 1];
            const float4 li = lo[i], hi_ = hi[i];
            for (int j0 = i + 1; j0 < end; j0 += 32) {
                const int j = j0 + lane;
                chunk(j, j < end && overlap(li, hi_, lo[j], hi[j]) && !((fi & BF_PINNED) && (d.bflags[j] & BF_PINNED)) &&
                             !adj_has(d, i, j));
            }
        };
        for (int i = w; i < N; i += W) {
            int n = 0;
            partners(i, [&](int, bool ok) { n += __popc(__ballot_sync(0xffffffffu, ok)); });
            if (lane == 0) cnt[i] = n;
        }
        __syncthreads();
        block_scan(cnt, off, N, scan);
        const int tot = off[N];
        np = min(tot, cap);
        if (np > 0) {
            for (int i = w; i < N; i += W) {
                int pos = off[i];
                if (off[i + 1] == pos) continue;
                partners(i, [&](int j, bool ok) {
                    const unsigned bal = __ballot_sync(0xffffffffu, ok);
                    const int at = pos + __popc(bal & ((1u << lane) - 1u));
                    if (ok && at < cap) {
                        d.pairs[at] = make_int2(i, j);
                        if (at < FRONT_PAIRS) pairs[at] = make_int2(i, j);
                    }
                    pos += __popc(bal);
                });
            }
            __syncthreads();
        }
        if (t == 0) {
            if (tot > cap) latch_status(d, ST_CAPACITY);
            d.ctr[C_NPAIRS] = np;
        }
        if (np <= FRONT_PAIRS) {
            d.pairs = pairs;
            d.npc = npc;
            d.npc_off = npc_off;
        }
    }

    // contacts (without body contacts the pair contacts' prefix is the zero of creation)
    for (int k = t; k < np + N; k += FT) narrow_count_item(d, k, np);
    __syncthreads();
    if (np > 0) block_scan(d.npc, d.npc_off, np, scan);
    block_scan(gcnt, goff, N, scan);
    const int n_pc = np > 0 ? d.npc_off[np] : 0;
    for (int k = t; k < np + N; k += FT)
        narrow_write_item(d, k, np, n_pc, [&](int i, int j) {
            if (end_live(d, i)) atomicAdd(&ends[i], 1);
            if (end_live(d, j)) atomicAdd(&ends[j], 1);
        });
    if (t == 0) set_contact_counts(d, n_pc);
    __syncthreads();

    // CSR (the slices' offsets also in shared memory; the ends' ids there too while they fit and
    // no slice needs the block's sort)
    int* const end_off = d.end_off;
    d.end_off = off;
    block_scan(ends, off, N, scan);
    for (int b = t; b <= N; b += FT) end_off[b] = off[b];
    bool many = t < N && ends[t] > HEAVY_ENDS;
    many = __syncthreads_or(many);
    if (!many && off[N] <= FRONT_ENDS) d.end_id = ids;
    const int nb = d.Nc + min(n_pc + goff[N], d.cap_contacts);
    for (int b = t; b < nb; b += FT) csr_fill_bond(d, b);
    __syncthreads();
    for (int b = t / CSR_LANES; b < N; b += FT / CSR_LANES) csr_place_body<WANT>(d, b, t % CSR_LANES);
    if (!many) return;
    __syncthreads();
    const int nheavy = d.ctr[C_NHEAVY];
    for (int h = 0; h < nheavy; ++h) csr_sort_heavy<FT, WANT>(d, d.heavy[h], key);
}

bool front_fits(int n_bodies, bool contacts) { return n_bodies > 0 && n_bodies <= (contacts ? FRONT_N : FRONT_N_GROUND); }

void launch_front(const Dev& d, cudaStream_t st, long long* launches) {
    with_want(d.csr_want, [&](auto w) { launch_pdl(k_front<decltype(w)::value>, dim3(1), dim3(FT), 0, st, d); });
    *launches += 1;
}

}  // namespace pabd
