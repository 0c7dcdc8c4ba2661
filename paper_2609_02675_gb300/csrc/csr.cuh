// The CSR of bond ends: ends of dynamic bodies, sorted by (body, 2 * bond + side).  Shared by the
// CSR kernels (k_step.cu), the ground-only front (k_collision.cu) and the one-launch front of
// small scenes (k_front.cu).
#pragma once
#include <type_traits>

#include "end_record.cuh"
#include "sort_slices.cuh"

namespace pabd {

__device__ __forceinline__ bool end_live(const Dev& d, int body) {
    return body >= 0 && !(d.bflags[body] & BF_PINNED);
}

// end `id` (2 bond + side) takes slot p: what the step's sweeps read of it -- its slot and
// material point for the bond and solve launches (WANT_SLOTS), its record for the others
// (WANT_RECORDS)
template <int WANT>
__device__ __forceinline__ void place_end(const Dev& d, int id, int p, int4 m, float4 xi, float4 xj, float4 bn) {
    const bool side_j = id & 1;
    if (WANT & WANT_SLOTS) {
        d.end_pos[id] = p;
        d.end_x[p] = side_j ? make_float4(xj.x, xj.y, xj.z, 0.f) : make_float4(xi.x, xi.y, xi.z, 0.f);
    }
    if (WANT & WANT_RECORDS) pack_end(d.rec + 3 * (size_t)p, id >> 1, m, xi, xj, bn, side_j);
}
template <int WANT>
__device__ __forceinline__ void place_end(const Dev& d, int id, int p) {
    const int bond = id >> 1;
    if (WANT == WANT_SLOTS) {  // (one material point to load)
        const float4 x = (id & 1) ? d.bxj[bond] : d.bxi[bond];
        d.end_pos[id] = p;
        d.end_x[p] = make_float4(x.x, x.y, x.z, 0.f);
    } else {
        place_end<WANT>(d, id, p, d.bmeta[bond], d.bxi[bond], d.bxj[bond], d.bn[bond]);
    }
}

__device__ __forceinline__ void csr_fill_bond(const Dev& d, int b) {
    const int4 m = d.bmeta[b];
    auto put = [&](int body, int id) {
        if (end_live(d, body)) d.end_id[d.end_off[body] + atomicAdd(&d.end_cur[body], 1)] = id;
        else d.end_pos[id] = -1;
    };
    put(m.x, 2 * b);
    put(m.y, 2 * b + 1);
}

// Place a body's ends in ascending end id, by CSR_LANES lanes: an end's slot is the slice's start
// plus the number of smaller ids in it.  A body with more than HEAVY_ENDS (64) ends goes on the
// heavy list, whose slices csr_sort_heavy sorts.  Eight lanes: a body of a pile has about as
// many ends (a warp per body left 24 lanes idle: 64 us for 262 144 bodies, now 19; a settled
// bed's grains, with 29 ends, took 79 us of CSR stage on a warp each against 65).
constexpr int CSR_LANES = 8;
template <int WANT>
__device__ __forceinline__ void csr_place_body(const Dev& d, int body, int lane) {
    const int s = d.end_off[body], n = d.end_off[body + 1] - s;
    if (n > HEAVY_ENDS) {
        if (lane == 0) d.heavy[atomicAdd(&d.ctr[C_NHEAVY], 1)] = body;
        return;
    }
    const int* ids = d.end_id + s;
    for (int k = lane; k < n; k += CSR_LANES) {
        const int id = ids[k];
        int r = 0;
#pragma unroll 4
        for (int m = 0; m < n; ++m) r += ids[m] < id ? 1 : 0;
        place_end<WANT>(d, id, s + r);
    }
}

// A heavy body's ends, by a block of T threads: ranked by a bitmap over the step's ends, or sorted
// first with the bond launch's end-record buffer (unused at this stage) as scratch (the slab
// under 48 x 48 boxes: CSR stage 73 us with the sort, 29 with the ranking).  key: 2 LONG_SMEM
// ints.
template <int T, int WANT>
__device__ __forceinline__ void csr_sort_heavy(const Dev& d, int body, int* key) {
    const int s = d.end_off[body], e = d.end_off[body + 1], n = e - s;
    const long long universe = 2ll * d.ctr[C_NBONDS];
    if (rank_pays(n, universe)) {
        block_rank_ids<T>(d.end_id + s, n, (int)universe, reinterpret_cast<unsigned*>(key), key + LONG_SMEM,
                          [&](int id, int r) { place_end<WANT>(d, id, s + r); });
        return;
    }
    block_sort_slice<T>(d.end_id + s, n, reinterpret_cast<int*>(d.ends) + s, key);
    for (int p = s + threadIdx.x; p < e; p += T) place_end<WANT>(d, d.end_id[p], p);
    __syncthreads();
}

// calls f(want) with Dev::csr_want as a compile-time constant
template <class F>
void with_want(int want, F&& f) {
    if (want == WANT_SLOTS) f(std::integral_constant<int, WANT_SLOTS>{});
    else if (want == WANT_RECORDS) f(std::integral_constant<int, WANT_RECORDS>{});
    else f(std::integral_constant<int, WANT_SLOTS | WANT_RECORDS>{});
}

}  // namespace pabd
