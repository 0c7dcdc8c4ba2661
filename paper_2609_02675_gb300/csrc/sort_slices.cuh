// Sorting of short integer slices in place (ascending, keys unique within a slice): a warp's
// ranking for up to 32 keys, its bitonic network in registers for up to 64, and a block's for
// longer slices -- runs of up
// to LONG_SMEM keys in shared memory, then merge passes through a scratch slice.  Used for
// the CSR of bond ends (k_step.cu) and for the pair lists of both broad phases (k_collision.cu,
// k_lbvh.cu).
#pragma once
#include "pabd_internal.h"

namespace pabd {

constexpr int LONG_T = 1024;
constexpr int LONG_SMEM = 4096;  // keys of a sorted run, words of a bitmap (launches that may rank take two arrays of them, 32 KB)

// 64 keys held two per lane (key k in lane k / 2, slot k % 2) sorted ascending by the 32
// lanes of a warp: a bitonic network of shuffles
__device__ __forceinline__ void warp_sort64(int& v0, int& v1, int lane) {
    for (int size = 2; size <= 64; size <<= 1) {
        const bool up = ((2 * lane) & size) == 0;       // ascending block (same for both slots)
        for (int stride = size >> 1; stride > 1; stride >>= 1) {
            const bool lower = ((2 * lane) & stride) == 0; // partner k ^ stride is in lane ^ stride/2
            const int o0 = __shfl_xor_sync(0xffffffffu, v0, stride >> 1);
            const int o1 = __shfl_xor_sync(0xffffffffu, v1, stride >> 1);
            v0 = (lower == up) ? min(v0, o0) : max(v0, o0);
            v1 = (lower == up) ? min(v1, o1) : max(v1, o1);
        }
        const int mn = min(v0, v1), mx = max(v0, v1);  // stride 1: the lane's own pair
        v0 = up ? mn : mx;
        v1 = up ? mx : mn;
    }
}

// up to 32 unique keys, one per lane (lanes >= n hold nothing): each key's rank among the n,
// counted through n broadcasts -- independent shuffles, no dependent network
__device__ __forceinline__ int warp_rank32(int v, int n, int lane) {
    int r = 0;
    for (int k = 0; k < n; ++k) {
        const int o = __shfl_sync(0xffffffffu, v, k);
        r += (o < v) ? 1 : 0;
    }
    return lane < n ? r : -1;
}

// slice v[0..n), n <= 64, by the 32 lanes of a warp: by rank up to 32 keys, else the bitonic
// network (padding INT_MAX)
__device__ __forceinline__ void warp_sort_slice64(int* v, int n, int lane) {
    if (n <= 32) {
        const int x = lane < n ? v[lane] : 0x7fffffff;
        const int r = warp_rank32(x, n, lane);
        __syncwarp();
        if (r >= 0) v[r] = x;
        return;
    }
    int v0 = (2 * lane < n) ? v[2 * lane] : 0x7fffffff;
    int v1 = (2 * lane + 1 < n) ? v[2 * lane + 1] : 0x7fffffff;
    warp_sort64(v0, v1, lane);
    if (2 * lane < n) v[2 * lane] = v0;
    if (2 * lane + 1 < n) v[2 * lane + 1] = v1;
}

// slice v[0..n) by a whole block of T threads with `key` LONG_SMEM ints of shared memory
// and tmp[0..n) scratch: runs of up to LONG_SMEM keys by a bitonic network in shared memory,
// then runs merged pairwise (run length doubling), each key placed at its index in its run
// plus its rank in the partner run (a binary search), ping-ponging between v and tmp.  Every
// thread of the block calls it with the same slice.
template <int T>
__device__ __forceinline__ void block_sort_slice(int* v, int n, int* tmp, int* key) {
    for (int r0 = 0; r0 < n; r0 += LONG_SMEM) {
        const int rn = min(LONG_SMEM, n - r0);
        int m = 2;
        while (m < rn) m <<= 1;
        for (int k = threadIdx.x; k < m; k += T) key[k] = k < rn ? v[r0 + k] : 0x7fffffff;
        __syncthreads();
        for (int size = 2; size <= m; size <<= 1) {
            for (int stride = size >> 1; stride > 0; stride >>= 1) {
                for (int k = threadIdx.x; k < m; k += T) {
                    const int l = k ^ stride;
                    if (l > k) {
                        const bool up = (k & size) == 0;
                        const int a = key[k], b = key[l];
                        if ((a > b) == up) { key[k] = b; key[l] = a; }
                    }
                }
                __syncthreads();
            }
        }
        for (int k = threadIdx.x; k < rn; k += T) v[r0 + k] = key[k];
        __syncthreads();
    }
    int* src = v;
    int* dst = tmp;
    for (int R = LONG_SMEM; R < n; R <<= 1) {
        for (int k = threadIdx.x; k < n; k += T) {
            const int run = k / R, start = run * R, pstart = (run ^ 1) * R;
            const int plen = max(0, min(R, n - pstart));
            const int x = src[k];
            int lo = 0, hi = plen;  // keys of the partner run below x
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (src[pstart + mid] < x) lo = mid + 1; else hi = mid;
            }
            dst[min(start, pstart) + (k - start) + lo] = x;
        }
        __syncthreads();
        int* t = src; src = dst; dst = t;
    }
    if (src != v) {
        for (int k = threadIdx.x; k < n; k += T) v[k] = src[k];
        __syncthreads();
    }
}

// Ranks of unique ids in [0, universe) by a whole block of T threads: place(id, r) for every
// id of v[0..n), r its place among them.  A bitmap of the ids in shared memory (LONG_SMEM words,
// a window of the universe at a time) and the running count of its words: O(n + universe / 32)
// instead of a sort's O(n log^2 n).  v is not changed.
template <int T, class Place>
__device__ __forceinline__ void block_rank_ids(const int* v, int n, int universe, unsigned* bits, int* before,
                                               Place&& place) {
    constexpr int PER = LONG_SMEM / T;
    static_assert(PER * T == LONG_SMEM, "whole words per thread");
    __shared__ int wsum[T / 32];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int base = 0;  // ids below the window
    for (long long w0 = 0; w0 < universe; w0 += 32ll * LONG_SMEM) {
        for (int k = t; k < LONG_SMEM; k += T) bits[k] = 0u;
        __syncthreads();
        for (int k = t; k < n; k += T) {
            const long long i = v[k] - w0;
            if (i >= 0 && i < 32ll * LONG_SMEM) atomicOr(&bits[i >> 5], 1u << (i & 31));
        }
        __syncthreads();
        int c[PER], s = 0;
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            c[k] = __popc(bits[t * PER + k]);
            s += c[k];
        }
        int inc = s;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int u = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += u;
        }
        if (lane == 31) wsum[warp] = inc;
        __syncthreads();
        int run = base + inc - s, all = 0;
        for (int k = 0; k < T / 32; ++k) {
            if (k < warp) run += wsum[k];
            all += wsum[k];
        }
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            before[t * PER + k] = run;
            run += c[k];
        }
        __syncthreads();
        for (int k = t; k < n; k += T) {
            const int id = v[k];
            const long long i = id - w0;
            if (i >= 0 && i < 32ll * LONG_SMEM)
                place(id, before[i >> 5] + __popc(bits[i >> 5] & ((1u << (i & 31)) - 1u)));
        }
        base += all;
        __syncthreads();  // the bitmap is cleared for the next window
    }
}

// ranking pays against sorting in place unless a short slice's ids spread over many windows
__device__ __forceinline__ bool rank_pays(int n, long long universe) {
    return universe <= 4ll * 32 * LONG_SMEM || n > LONG_SMEM;
}

}  // namespace pabd
