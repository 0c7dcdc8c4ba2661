// Linear BVH broad phase (the paper's choice for collision detection, Sec. 5), beside the
// grid hash: it needs no cell size, so boxes of any mix of sizes and speeds cost the same.
//
//   1. scene box of the bodies' box centres (min / max over order-preserving int bits: exact
//      and order-independent);
//   2. 30-bit Morton code of every centre (10 bits per axis over the scene box);
//   3. stable LSD radix sort of (code, body) -- 8-bit digits, tiles of 1024 keys, a block of
//      1024 threads each: per-(digit, tile) counts (taken by the pass before), their prefix sums,
//      and a stable scatter that ranks equal digits by warp match masks and the warps' counts, so
//      the order is deterministic;
//   4. the binary radix tree over the sorted codes by Karras' construction ("Maximizing
//      parallelism in the construction of BVHs, octrees, and k-d trees", HPG 2012): each
//      internal node finds its range and split from the longest common prefixes (equal codes
//      broken by leaf index);
//   5. bottom-up refit (the second child to arrive merges): an internal node is one 64-byte
//      record of both children's boxes, their ids and the largest body id below each;
//   6. every body i walks the tree for the leaves j > i its box overlaps that the pair filter
//      accepts, the bodies in leaf order so that a warp's walks stay together: a counting walk
//      that keeps the first partners it finds, prefix sums, a write that replays them (or walks
//      again where a body has more), then each body's partner slice sorted (warp or block).
//      The list is the sorted set of overlapping pairs: the same pairs, bit for bit, as the grid
//      hash's.
//
// Bound by the latency of its dependent steps: 20 011 boxes leave four warps per SM.  One node
// record per visit (one dependent load instead of three), leaf order, subtrees without a larger
// id skipped, the replayed write and 1024-thread tiles (a tile of 1024 keys was one warp's, 32
// steps in series) took its collision stage from 387 to 156 us.
#include "pair_filter.cuh"
#include "sort_slices.cuh"

namespace pabd {

constexpr int BT = 256;        // threads per block for per-body / per-node kernels
constexpr int RX_TILE = 1024;  // keys per radix tile (a block, one thread each)

static inline int bblk(long long n) { return (int)((n + BT - 1) / BT > 0 ? (n + BT - 1) / BT : 1); }

__device__ __forceinline__ float o2f(int i) { return __int_as_float(i >= 0 ? i : i ^ 0x7fffffff); }

// spread the low 10 bits of v to every third bit
__device__ __forceinline__ unsigned spread3(unsigned v) {
    v &= 0x3ffu;
    v = (v | (v << 16)) & 0x030000ffu;
    v = (v | (v << 8)) & 0x0300f00fu;
    v = (v | (v << 4)) & 0x030c30c3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

// per tile of 1024 bodies: their codes, the counts of the first digit, and the scratch of the
// passes that follow zeroed (the second digit's counts, the refit's arrivals)
__global__ void __launch_bounds__(RX_TILE) k_bvh_morton(Dev d, int ntile) {
    pdl_enter();
    __shared__ int c[256];
    const int tile = blockIdx.x, t = threadIdx.x;
    if (t < 256) c[t] = 0;
    __syncthreads();
    const int b = tile * RX_TILE + t;
    if (b == 0) d.bvh_parent[0] = -1;
    if (b < d.N - 1) d.bvh_visit[b] = 0;
    if (b < d.N) {
        const float4 lo = d.lo[b], hi = d.hi[b];
        const float x[3] = {0.5f * (lo.x + hi.x), 0.5f * (lo.y + hi.y), 0.5f * (lo.z + hi.z)};
        unsigned q[3];
        bool finite = true;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const float b0 = o2f(d.bvh_bounds[k]), b1 = o2f(d.bvh_bounds[3 + k]);
            const float ext = b1 - b0;
            float u = ext > 0.f ? (x[k] - b0) / ext : 0.f;
            finite = finite && isfinite(u);
            u = fminf(fmaxf(u, 0.f), 1.f);
            q[k] = min((unsigned)(u * 1024.f), 1023u);
        }
        const unsigned key = finite ? (spread3(q[0]) << 2) | (spread3(q[1]) << 1) | spread3(q[2]) : 0xffffffffu;
        d.bvh_key[b] = key;
        d.bvh_id[b] = b;
        atomicAdd(&c[key & 255u], 1);
    }
    __syncthreads();
    if (t < 256) {
        d.rx_cnt[t * ntile + tile] = c[t];
        d.rx_cnt2[t * ntile + tile] = 0;
    }
}

// ---- stable radix sort of (key, id), 8 bits per pass ----

// One pass over a tile: each key's rank among the tile's equal digits is its rank in its warp
// plus the equal digits of the warps before; the tile's first place for a digit comes from the
// scanned counts.  The next pass's digit is counted at the key's destination (cnt_next), and
// this pass's counts, already scanned, are zeroed for the pass after.
__global__ void __launch_bounds__(RX_TILE) k_rx_scatter(const unsigned* key_in, const int* id_in, unsigned* key_out,
                                                        int* id_out, int n, int shift, int ntile, const int* off,
                                                        int* cnt, int* cnt_next) {
    pdl_enter();
    constexpr int NW = RX_TILE / 32;
    __shared__ unsigned short wc[NW][256];
    const int tile = blockIdx.x, t = threadIdx.x, w = t >> 5, lane = t & 31;
    for (int k = t; k < NW * 256 / 2; k += RX_TILE) reinterpret_cast<unsigned*>(wc)[k] = 0;
    __syncthreads();
    const int idx = tile * RX_TILE + t;
    const bool valid = idx < n;
    const unsigned k = valid ? key_in[idx] : 0u;
    const int id = valid ? id_in[idx] : 0;
    const int digit = valid ? (int)((k >> shift) & 255u) : 256 + lane;  // unmatched if invalid
    const unsigned peers = __match_any_sync(0xffffffffu, digit);
    const int rank = __popc(peers & ((1u << lane) - 1u));
    if (valid && rank == 0) wc[w][digit] = (unsigned short)__popc(peers);
    __syncthreads();
    if (t < 256) {
        int run = 0;
#pragma unroll 8
        for (int v = 0; v < NW; ++v) {
            const int c = wc[v][t];
            wc[v][t] = (unsigned short)run;
            run += c;
        }
        cnt[t * ntile + tile] = 0;
    }
    __syncthreads();
    if (valid) {
        const int dst = off[digit * ntile + tile] + wc[w][digit] + rank;
        key_out[dst] = k;
        id_out[dst] = id;
        if (cnt_next) atomicAdd(&cnt_next[((k >> (shift + 8)) & 255u) * ntile + dst / RX_TILE], 1);
    }
}

// ---- Karras radix tree ----

__device__ __forceinline__ int prefix(const unsigned* __restrict__ key, int n, int i, int j) {
    if (j < 0 || j >= n) return -1;
    const unsigned a = key[i], b = key[j];
    return a == b ? 32 + __clz(i ^ j) : __clz(a ^ b);
}

__global__ void k_bvh_build(Dev d) {
    pdl_enter();
    const int n = d.N;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n - 1) return;
    const unsigned* key = d.bvh_key;
    const int dir = prefix(key, n, i, i + 1) - prefix(key, n, i, i - 1) > 0 ? 1 : -1;
    const int dmin = prefix(key, n, i, i - dir);
    int lmax = 2;
    while (prefix(key, n, i, i + lmax * dir) > dmin) lmax <<= 1;
    int l = 0;
    for (int t = lmax >> 1; t >= 1; t >>= 1)
        if (prefix(key, n, i, i + (l + t) * dir) > dmin) l += t;
    const int j = i + l * dir;
    const int dnode = prefix(key, n, i, j);
    int s = 0;
    for (int div = 2;; div <<= 1) {
        const int t = (l + div - 1) / div;
        if (prefix(key, n, i, i + (s + t) * dir) > dnode) s += t;
        if (t <= 1) break;
    }
    const int gamma = i + s * dir + min(dir, 0);
    const int left = min(i, j) == gamma ? (n - 1) + gamma : gamma;
    const int right = max(i, j) == gamma + 1 ? (n - 1) + gamma + 1 : gamma + 1;
    d.bvh_kids[i] = make_int2(left, right);
    d.bvh_parent[left] = i;
    d.bvh_parent[right] = i;
}

// An internal node's record (Dev::bvh_node, four float4): (lo, id) and (hi, largest body id) of
// the left child, then of the right.  A leaf's id is n - 1 + its place; its largest body id is
// its body.

// the box of node c and the largest body id below it
__device__ __forceinline__ void node_box(const Dev& d, int c, float4& lo, float4& hi) {
    const int n = d.N;
    if (c >= n - 1) {
        const int b = d.bvh_id[c - (n - 1)];
        lo = d.lo[b];
        hi = d.hi[b];
        hi.w = __int_as_float(b);
    } else {
        const float4* r = d.bvh_node + 4 * (size_t)c;
        const float4 al = __ldcg(r), ah = __ldcg(r + 1), bl = __ldcg(r + 2), bh = __ldcg(r + 3);
        lo = make_float4(fminf(al.x, bl.x), fminf(al.y, bl.y), fminf(al.z, bl.z), 0.f);
        hi = make_float4(fmaxf(ah.x, bh.x), fmaxf(ah.y, bh.y), fmaxf(ah.z, bh.z),
                         __int_as_float(max(__float_as_int(ah.w), __float_as_int(bh.w))));
    }
}

__global__ void k_bvh_refit(Dev d) {
    pdl_enter();
    const int n = d.N;
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= n || n < 2) return;
    int node = d.bvh_parent[(n - 1) + k];
    while (node >= 0) {
        __threadfence();
        if (atomicAdd(&d.bvh_visit[node], 1) == 0) return;  // the sibling's walk is not here yet
        __threadfence();
        const int2 ch = d.bvh_kids[node];
        float4 al, ah, bl, bh;
        node_box(d, ch.x, al, ah);
        node_box(d, ch.y, bl, bh);
        al.w = __int_as_float(ch.x);
        bl.w = __int_as_float(ch.y);
        float4* r = d.bvh_node + 4 * (size_t)node;
        __stcg(r, al);
        __stcg(r + 1, ah);
        __stcg(r + 2, bl);
        __stcg(r + 3, bh);
        node = d.bvh_parent[node];
    }
}

// every accepted partner j > i of body i, in tree order
template <class F>
__device__ __forceinline__ int bvh_partners(const Dev& d, int i, F&& f) {
    const int n = d.N;
    if (n < 2 || !d.p.body_contacts) return 0;
    const float4 li = d.lo[i], hi = d.hi[i];
    const int gi = d.group[i], fi = d.bflags[i];
    int stack[64];
    int sp = 0, cnt = 0;
    int node = 0;
    for (;;) {
        const float4* r = d.bvh_node + 4 * (size_t)node;
        const float4 box[4] = {r[0], r[1], r[2], r[3]};
        int next = -1;
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const int kid = __float_as_int(box[2 * c].w), top = __float_as_int(box[2 * c + 1].w);
            if (top <= i || !overlap(li, hi, box[2 * c], box[2 * c + 1])) continue;
            if (kid >= n - 1) {  // the leaf of body `top`, whose box is the one just tested
                if (d.group[top] != gi || ((fi & BF_PINNED) && (d.bflags[top] & BF_PINNED)) || adj_has(d, i, top)) continue;
                f(top, cnt);
                ++cnt;
            } else if (next < 0) {
                next = kid;
            } else if (sp < 64) {
                stack[sp++] = kid;
            } else {
                latch_status(d, ST_CAPACITY);  // deeper than any tree of 30-bit codes
            }
        }
        if (next < 0) {
            if (sp == 0) return cnt;
            next = stack[--sp];
        }
        node = next;
    }
}

// counts the partners of the bodies in leaf order, keeping the first BVH_STASH of each (slot k of
// body i at k N + i)
__global__ void k_bvh_pair_count(Dev d) {
    pdl_enter();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.N) return;
    const int i = d.bvh_id[k];
    d.pair_cnt[i] = bvh_partners(d, i, [&](int j, int c) {
        if (c < BVH_STASH) d.bvh_stash[(size_t)c * d.N + i] = j;
    });
}

__global__ void k_bvh_pair_write(Dev d) {
    pdl_enter();
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= d.N) return;
    const int i = d.bvh_id[k];
    const int s = d.pair_off[i], n = d.pair_off[i + 1] - s, cap = d.cap_pairs;
    if (n <= BVH_STASH) {
        for (int c = 0; c < n; ++c)
            if (s + c < cap) d.pair_j[s + c] = d.bvh_stash[(size_t)c * d.N + i];
    } else {
        bvh_partners(d, i, [&](int j, int c) {
            if (s + c < cap) d.pair_j[s + c] = j;
        });
    }
    if (k == d.N - 1) {
        const int tot = d.pair_off[d.N];
        if (tot > cap) latch_status(d, ST_CAPACITY);
        d.ctr[C_NPAIRS] = min(tot, cap);
    }
}

// each body's partners ascending (a warp each; longer than 64: the block sort below); shared
// by the LBVH and the multilevel grid
__global__ void k_pair_sort(Dev d) {
    pdl_enter();
    const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (i >= d.N) return;
    const int cap = d.cap_pairs;
    const int s = min(d.pair_off[i], cap), e = min(d.pair_off[i + 1], cap), n = e - s;
    if (n > 64) {
        if (lane == 0) d.pair_heavy[atomicAdd(&d.ctr[C_NPHEAVY], 1)] = i;
        return;
    }
    warp_sort_slice64(d.pair_j + s, n, lane);
    __syncwarp();
    for (int p = s + lane; p < e; p += 32) d.pairs[p] = make_int2(i, d.pair_j[p]);
}

// (an off-grid body's partners come in order: nothing to sort; the others are ranked by a bitmap
// over the bodies, or sorted)
__global__ void __launch_bounds__(LONG_T) k_pair_sort_long(Dev d) {
    pdl_enter();
    extern __shared__ int key[];
    const int nh = d.ctr[C_NPHEAVY], cap = d.cap_pairs;
    for (int h = blockIdx.x; h < nh; h += gridDim.x) {
        const int i = d.pair_heavy[h];
        const int s = min(d.pair_off[i], cap), e = min(d.pair_off[i + 1], cap);
        bool unsorted = false;
        for (int p = s + threadIdx.x; p + 1 < e; p += LONG_T) unsorted |= d.pair_j[p] > d.pair_j[p + 1];
        if (__syncthreads_or(unsorted)) {
            if (rank_pays(e - s, d.N)) {
                block_rank_ids<LONG_T>(d.pair_j + s, e - s, d.N, reinterpret_cast<unsigned*>(key), key + LONG_SMEM,
                                       [&](int j, int r) { d.pairs[s + r] = make_int2(i, j); });
                continue;
            }
            block_sort_slice<LONG_T>(d.pair_j + s, e - s, d.pair_tmp + s, key);
        }
        for (int p = s + threadIdx.x; p < e; p += LONG_T) d.pairs[p] = make_int2(i, d.pair_j[p]);
        __syncthreads();
    }
}

void launch_pair_sort(const Dev& d, cudaStream_t st, long long* launches) {
    launch_pdl(k_pair_sort, dim3(bblk((long long)d.N * 32)), dim3(BT), 0, st, d);
    launch_pdl(k_pair_sort_long, dim3(152), dim3(LONG_T), 2 * LONG_SMEM * sizeof(int), st, d);
    *launches += 2;
}

// (the bounds of the centres are zeroed by launch_step_reset and taken by k_aabb)
void launch_lbvh_pairs(const Dev& d, cudaStream_t st, long long* launches) {
    const int n = d.N;
    const int ntile = (n + RX_TILE - 1) / RX_TILE > 0 ? (n + RX_TILE - 1) / RX_TILE : 1;
    launch_pdl(k_bvh_morton, dim3(ntile), dim3(RX_TILE), 0, st, d, ntile);
    unsigned* ka = d.bvh_key;
    unsigned* kb = d.bvh_key2;
    int* ia = d.bvh_id;
    int* ib = d.bvh_id2;
    int* ca_ = d.rx_cnt;
    int* cb = d.rx_cnt2;
    for (int shift = 0; shift < 32; shift += 8) {
        scan_exclusive(ca_, d.rx_off, 256 * ntile, d.scan_scratch, st, launches);
        launch_pdl(k_rx_scatter, dim3(ntile), dim3(RX_TILE), 0, st, ka, ia, kb, ib, n, shift, ntile, d.rx_off, ca_,
                   shift < 24 ? cb : (int*)nullptr);
        unsigned* tk = ka; ka = kb; kb = tk;
        int* ti = ia; ia = ib; ib = ti;
        int* tc = ca_; ca_ = cb; cb = tc;
    }
    // four passes: the sorted keys and ids are back in bvh_key / bvh_id
    launch_pdl(k_bvh_build, dim3(bblk(n - 1)), dim3(BT), 0, st, d);
    launch_pdl(k_bvh_refit, dim3(bblk(n)), dim3(BT), 0, st, d);
    launch_pdl(k_bvh_pair_count, dim3((n + 63) / 64 > 0 ? (n + 63) / 64 : 1), dim3(64), 0, st, d);
    scan_exclusive(d.pair_cnt, d.pair_off, n, d.scan_scratch, st, launches);
    launch_pdl(k_bvh_pair_write, dim3(bblk(n)), dim3(BT), 0, st, d);
    *launches += 9;
    launch_pair_sort(d, st, launches);
}

}  // namespace pabd
