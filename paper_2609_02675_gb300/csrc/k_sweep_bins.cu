// All n_iter sweeps of a step in one launch, for scenes whose groups are small (sweep mode 2).
//
// Bodies interact only inside their group (a scene whose user bonds join groups is swept by
// launches), so whole groups are dealt to bins of consecutive
// bodies and each bin is swept by one thread-block cluster on its own: nothing is exchanged
// between clusters.  The bin's iterates live in shared memory, twice (Jacobi), a copy in every
// block of the cluster: a body's new iterate is stored into all the copies through distributed
// shared memory and the next sweep reads only its own block's.  Sweeps are separated by the
// cluster's hardware barrier (a block barrier in a cluster of one) instead of a launch; a
// body's other data (predictor, mass, end records) stay in the L1 caches from the second sweep
// on.  The blocks of a cluster take equal runs of the bin's bodies, ordered by (extended path,
// end count) as the light order does for the whole scene.  Same arithmetic per body as
// k_sweep_one, so the results are the same bit for bit.
//
// What bounds it: instruction issue of one warp per scheduler along the dependent chain of a
// body's sum, factorisation and rotation (8 chained bodies: 2160 instructions a sweep, 2.7 cycles
// each, of which 0.65 wait for the previous result and 0.57 for instruction fetch; a 121-body net
// 4.7, with the cluster's barrier and its stores 1.1).  Per sweep,
// against one launch per sweep: 8 chained bodies 3.0 us (5.4), 121-body spring net 3.7 (4.9),
// 250-box pile 3.8 (4.5).
#include "sweep_shape.h"

namespace pabd {

constexpr int BIN_KEYS = 2 * END_BINS;  // bins of the order; one more for the heavy bodies
constexpr int BINS_T = 256;             // most threads per block (leaves a thread 255 registers: no spills)

__device__ __forceinline__ unsigned cluster_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cluster_size() {
    unsigned n;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(n));
    return n;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// three float4 into block `rank`'s copy of the shared array at local address p
__device__ __forceinline__ void store_remote(float4* p, unsigned rank, const float* c, const float* A) {
    unsigned a = (unsigned)__cvta_generic_to_shared(p), ra;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(ra), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(A[0]) : "memory");
    asm volatile("st.shared::cluster.v4.f32 [%0+16], {%1, %2, %3, %4};" ::"r"(ra), "f"(A[1]), "f"(A[2]), "f"(A[3]), "f"(A[4]) : "memory");
    asm volatile("st.shared::cluster.v4.f32 [%0+32], {%1, %2, %3, %4};" ::"r"(ra), "f"(A[5]), "f"(A[6]), "f"(A[7]), "f"(A[8]) : "memory");
}

// iterates of the bin's bodies (from body b0 on) in shared memory, for gather_ends
struct BinQ {
    const float4* q;
    int b0;
    __device__ __forceinline__ void operator()(const EndBond& e, float* c, float* A) const {
        ld_other(q, e.other < 0 ? -1 : e.other - b0, e.xo, c, A);
    }
};

// a light body of the block's run, in its order, with what its solve reads besides iterates and
// bonds: kept in shared memory for all the sweeps
struct alignas(16) BinSlot {
    int b, e0, e1, fl;
    BodyData body;
};

// shared memory of a block: the two iterates, its run of bodies in order, the heavy teams'
static size_t bins_smem(int cap, int cluster, int threads) {
    const size_t run = (size_t)(cap + cluster - 1) / cluster;
    return 2 * 3 * sizeof(float4) * (size_t)cap + sizeof(BinSlot) * run + sizeof(HeavyShared) * (threads / HEAVY_T);
}

template <int L, class X>
__global__ void __launch_bounds__(BINS_T, 1) k_sweep_bins(Dev d, int cap) {
    extern __shared__ float4 sm[];
    __shared__ int hist[BIN_KEYS + 1], start[BIN_KEYS + 2];
    const int tid = threadIdx.x, T = blockDim.x;
    const int C = (int)cluster_size(), rank = (int)cluster_rank();
    const int2 range = d.bin_range[blockIdx.x / C];
    const int b0 = range.x, nb = range.y - range.x;
    float4* const q[2] = {sm, sm + 3 * cap};
    BinSlot* const slots = reinterpret_cast<BinSlot*>(sm + 6 * cap);
    HeavyShared* const heavy_sh = reinterpret_cast<HeavyShared*>(slots + (cap + C - 1) / C);
    for (int k = tid; k <= BIN_KEYS; k += T) hist[k] = 0;
    pdl_enter();
    // both buffers start from the predictor's iterate: pinned and held bodies keep it
    for (int k = tid; k < 3 * nb; k += T) {
        const float4 v = d.qa[3 * (size_t)b0 + k];
        q[0][k] = v;
        q[1][k] = v;
    }
    // this block's run of the bin's bodies, by (class, end count): a counting sort
    const int run = (nb + C - 1) / C, r0 = min(nb, rank * run), r1 = min(nb, r0 + run);
    auto key_of = [&](int b) {
        const int fl = d.bflags[b];
        if ((fl & BF_PINNED) || held(d, b)) return -1;
        const int n = d.end_off[b + 1] - d.end_off[b];
        if (n > HEAVY_ENDS) return BIN_KEYS;
        const bool ext = d.p.precision_policy == 3 || (d.p.precision_policy && (fl & BF_FP64));
        return (ext ? 0 : END_BINS) + (HEAVY_ENDS - n);
    };
    __syncthreads();
    for (int i = r0 + tid; i < r1; i += T) {
        const int k = key_of(b0 + i);
        if (k >= 0) atomicAdd(&hist[k], 1);
        if (d.bflags[b0 + i] & BF_PINNED) d.resid_body[b0 + i] = 0.0;
    }
    __syncthreads();
    if (tid < 32) {  // exclusive prefix of the bins by one warp
        int carry = 0;
        for (int k0 = 0; k0 <= BIN_KEYS; k0 += 32) {
            const int k = k0 + tid, v = k <= BIN_KEYS ? hist[k] : 0;
            int inc = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int t = __shfl_up_sync(0xffffffffu, inc, o);
                if (tid >= o) inc += t;
            }
            if (k <= BIN_KEYS) { start[k] = carry + inc - v; hist[k] = carry + inc - v; }
            carry += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (tid == 0) start[BIN_KEYS + 1] = carry;
    }
    __syncthreads();
    for (int i = r0 + tid; i < r1; i += T) {
        const int b = b0 + i, k = key_of(b);
        if (k < 0) continue;
        BinSlot& s = slots[atomicAdd(&hist[k], 1)];
        s.b = b;
        s.e0 = d.end_off[b];
        s.e1 = d.end_off[b + 1];
        s.fl = d.bflags[b];
        s.body = ld_body(d, b, s.fl);
    }
    const int nl = start[BIN_KEYS], nall = start[BIN_KEYS + 1];
    if (C > 1) cluster_sync();
    else __syncthreads();

    constexpr int P = L;  // one thread per lane: the bodies are few
    const int plane = tid & (P - 1), warp = tid >> 5, lane = tid & 31;
    float4* const q_out = (d.p.n_iter & 1) ? d.qb : d.qa;
#pragma unroll 1
    for (int it = 0; it < d.p.n_iter; ++it) {
        const float4* qi = q[it & 1];
        float4* qo = q[(it + 1) & 1];
        const int last = it == d.p.n_iter - 1;
        const BinQ other{qi, b0};
        const auto gather = end_gather(d, other, it);
        auto self = [&](int b, float* c, float* A) { ld_q(qi, b - b0, c, A); };
        // (by the first `threads` threads of the body, pl this one's index among them)
        auto store = [&](int b, int pl, int threads, const float* c, const float* A) {
            if (last) {
                if (pl == 0) store_iterate(q_out, b, c, A);
            } else if (C == 1) {
                if (pl == 0) store_iterate(qo, b - b0, c, A);
            } else {
                for (int k = pl; k < C; k += threads) store_remote(qo + 3 * (b - b0), k, c, A);
            }
        };
        // the bodies with many ends first: a warp each, or a team of HEAVY_T threads
        for (int h = nl + warp; h < nall; h += T / 32) {
            const BinSlot& s = slots[h];
            if (s.e1 - s.e0 > WIDE_ENDS) continue;
            solve_free_body<32, 32, X>(d, s.b, lane, 0xffffffffu, s.fl, s.e0, s.e1, last, [&] { return s.body; }, self,
                [&](int o, const float* c, const float* A, int n) { store(o, lane, n, c, A); }, gather);
        }
        const HeavyTeam heavy{tid % HEAVY_T, 1 + tid / HEAVY_T};
        for (int h = nl + tid / HEAVY_T; h < nall; h += T / HEAVY_T) {
            const BinSlot& s = slots[h];
            if (s.e1 - s.e0 <= WIDE_ENDS) continue;
            solve_heavy<X>(d, s.b, heavy, heavy_sh[tid / HEAVY_T], last, self,
                [&](int o, const float* c, const float* A) { store(o, 0, 1, c, A); }, gather);
        }
        for (int k0 = warp * (32 / P); k0 < nl; k0 += T / P) {
            const int k = k0 + lane / P;
            const unsigned team = __ballot_sync(0xffffffffu, k < nl);
            if (k < nl) {
                const BinSlot& s = slots[k];
                solve_free_body<L, P, X>(d, s.b, plane, team, s.fl, s.e0, s.e1, last, [&] { return s.body; }, self,
                    [&](int o, const float* c, const float* A, int n) { store(o, plane, n, c, A); }, gather);
            }
            __syncwarp();
        }
        if (last) break;
        if (C > 1) cluster_sync();
        else __syncthreads();
    }
}

static cudaLaunchConfig_t bins_config(const BinsShape& b, cudaLaunchAttribute* attr) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(b.n * b.cluster);
    cfg.blockDim = dim3(b.block);
    cfg.dynamicSmemBytes = bins_smem(b.cap, b.cluster, b.block);
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = b.cluster;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cfg;
}

cudaError_t setup_sweep_bins(const BinsShape& b, int lanes, bool f64, int* fit) {
    cudaError_t e = cudaSuccess;
    with_lanes(lanes, f64, [&](auto l, auto x) {
        auto kernel = k_sweep_bins<decltype(l)::value, typename decltype(x)::type>;
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = bins_config(b, attr);
        // (the attribute is the kernel's, not the scene's: all that a block may have, whatever
        // other scenes need; bins that need more fit nowhere)
        cudaFuncAttributes fa;
        e = cudaFuncGetAttributes(&fa, kernel);
        if (e != cudaSuccess) return;
        const int most = 227 * 1024 - (int)fa.sharedSizeBytes;
        *fit = 0;
        if ((long long)cfg.dynamicSmemBytes > most) return;
        e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
        if (e == cudaSuccess && b.cluster > 8) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        cfg.numAttrs = 1;
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(fit, kernel, &cfg);
    });
    return e;
}

void launch_sweep_bins(const Dev& d, const BinsShape& b, int lanes, cudaStream_t st, long long* launches) {
    with_lanes(lanes, d.p.precision_policy == 2, [&](auto l, auto x) {
        cudaLaunchAttribute attr[2];
        cudaLaunchConfig_t cfg = bins_config(b, attr);
        cfg.stream = st;
        cudaLaunchKernelEx(&cfg, k_sweep_bins<decltype(l)::value, typename decltype(x)::type>, d, b.cap);
    });
    *launches += 1;
}

}  // namespace pabd
