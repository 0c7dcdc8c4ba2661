// Exclusive prefix sums of int arrays.
// Chunks of 4096 values (1024 threads x 4) are scanned per block; block totals go to a
// scratch array that one block scans; a third pass adds the block offsets.  Arrays of one
// chunk take one block, arrays of up to 131 072 values one cluster of blocks.
#include "pabd_internal.h"

namespace pabd {

constexpr int SCAN_THREADS = 1024;
constexpr int SCAN_ITEMS = 4;
constexpr int SCAN_CHUNK = SCAN_THREADS * SCAN_ITEMS;

__device__ __forceinline__ int warp_incl_scan(int v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int t = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// inclusive block scan of one value per thread; returns the inclusive prefix, block total in *total
__device__ __forceinline__ int block_incl_scan(int v, int* smem, int* total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int inc = warp_incl_scan(v);
    if (lane == 31) smem[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        int w = (lane < (blockDim.x >> 5)) ? smem[lane] : 0;
        int wi = warp_incl_scan(w);
        smem[lane] = wi;  // inclusive over warps
    }
    __syncthreads();
    int base = warp ? smem[warp - 1] : 0;
    *total = smem[(blockDim.x >> 5) - 1];
    return base + inc;
}

__global__ void __launch_bounds__(SCAN_THREADS) k_scan_chunks(const int* __restrict__ in, int* __restrict__ out,
                                                              int n, int* block_sums, int single) {
    pdl_enter();
    __shared__ int smem[32];
    const int base = blockIdx.x * SCAN_CHUNK + threadIdx.x * SCAN_ITEMS;
    int v[SCAN_ITEMS];
    int s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        v[k] = (base + k < n) ? in[base + k] : 0;
        s += v[k];
    }
    int total;
    int incl = block_incl_scan(s, smem, &total);
    int run = incl - s;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        if (base + k < n) out[base + k] = run;
        run += v[k];
    }
    if (threadIdx.x == 0) {
        if (single) out[n] = total;
        else block_sums[blockIdx.x] = total;
    }
}

__global__ void __launch_bounds__(SCAN_THREADS) k_scan_totals(int* block_sums, int nb, int* out, int n) {
    pdl_enter();
    __shared__ int smem[32];
    const int base = threadIdx.x * SCAN_ITEMS;
    int v[SCAN_ITEMS];
    int s = 0;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        v[k] = (base + k < nb) ? block_sums[base + k] : 0;
        s += v[k];
    }
    int total;
    int incl = block_incl_scan(s, smem, &total);
    int run = incl - s;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k) {
        if (base + k < nb) block_sums[base + k] = run;
        run += v[k];
    }
    if (threadIdx.x == 0) out[n] = total;
}

__global__ void __launch_bounds__(SCAN_THREADS) k_scan_add(int* out, int n, const int* block_sums) {
    pdl_enter();
    if (blockIdx.x == 0) return;
    const int add = block_sums[blockIdx.x];
    const int base = blockIdx.x * SCAN_CHUNK + threadIdx.x * SCAN_ITEMS;
#pragma unroll
    for (int k = 0; k < SCAN_ITEMS; ++k)
        if (base + k < n) out[base + k] += add;
}

// Arrays of up to SCAN_CLUSTER_MAX values: one cluster of SCAN_BLOCKS blocks (the portable
// maximum), each scanning a run of CL_CHUNK values per pass; the runs' totals are exchanged
// through distributed shared memory (a copy in every block) and a cluster barrier, and the
// running total is carried to the next pass.  Bound by latency: a load, two block barriers and a
// cluster barrier per 65 536 values, in one launch.  One block looping over chunks took that
// long per 4096 values: with it the 50 077-body quadruped step took 1434 us, now 1388, and the
// 16 384-box broad phase 111 us, now 102.
constexpr int SCAN_BLOCKS = 8;
constexpr int CL_ITEMS = 8;
constexpr int CL_CHUNK = SCAN_THREADS * CL_ITEMS;
// Two passes cost what the three launches do (262 144 values take four: 2 us more).
constexpr int SCAN_CLUSTER_MAX = 2 * SCAN_BLOCKS * CL_CHUNK;

__global__ void __launch_bounds__(SCAN_THREADS) k_scan_cluster(const int* __restrict__ in, int* __restrict__ out, int n) {
    __shared__ int smem[32];
    __shared__ int totals[2][SCAN_BLOCKS];
    unsigned rank;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
    // (every block of the cluster has started before another writes to its shared memory)
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    pdl_enter();
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
    int carry = 0;
    // (every block takes every pass, whether its run holds values or not: the barriers match)
    for (int c0 = 0, pass = 0; c0 < n; c0 += SCAN_BLOCKS * CL_CHUNK, ++pass) {
        const int base = c0 + (int)rank * CL_CHUNK + threadIdx.x * CL_ITEMS;
        int v[CL_ITEMS];
        if (base + CL_ITEMS <= n) {  // (arrays start on 16-byte boundaries, base is a multiple of 8)
#pragma unroll
            for (int k = 0; k < CL_ITEMS; k += 4) {
                const int4 q = *reinterpret_cast<const int4*>(in + base + k);
                v[k] = q.x; v[k + 1] = q.y; v[k + 2] = q.z; v[k + 3] = q.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < CL_ITEMS; ++k) v[k] = (base + k < n) ? in[base + k] : 0;
        }
        int s = 0;
#pragma unroll
        for (int k = 0; k < CL_ITEMS; ++k) s += v[k];
        int total;
        const int incl = block_incl_scan(s, smem, &total);
        // two sets of totals in turn: a block past this pass's barrier writes the other set
        int* const tot = totals[pass & 1];
        if (threadIdx.x < SCAN_BLOCKS) {
            const unsigned a = (unsigned)__cvta_generic_to_shared(&tot[rank]);
            unsigned ra;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"((unsigned)threadIdx.x));
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(ra), "r"(total) : "memory");
        }
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
        int before = carry, all = 0;
#pragma unroll
        for (int k = 0; k < SCAN_BLOCKS; ++k) {
            const int t = tot[k];
            all += t;
            if (k < (int)rank) before += t;
        }
        carry += all;
        int run = before + incl - s;
        if (base + CL_ITEMS <= n) {
#pragma unroll
            for (int k = 0; k < CL_ITEMS; k += 4) {
                int4 q;
                q.x = run; run += v[k];
                q.y = run; run += v[k + 1];
                q.z = run; run += v[k + 2];
                q.w = run; run += v[k + 3];
                *reinterpret_cast<int4*>(out + base + k) = q;
            }
        } else {
#pragma unroll
            for (int k = 0; k < CL_ITEMS; ++k) {
                if (base + k < n) out[base + k] = run;
                run += v[k];
            }
        }
    }
    if (rank == 0 && threadIdx.x == 0) out[n] = carry;
}

static void launch_scan_cluster(const int* in, int* out, int n, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(SCAN_BLOCKS);
    cfg.blockDim = dim3(SCAN_THREADS);
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = SCAN_BLOCKS;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    cudaLaunchKernelEx(&cfg, k_scan_cluster, in, out, n);
}

int scan_scratch_ints(int n) { return (n + SCAN_CHUNK - 1) / SCAN_CHUNK + 1; }

void scan_exclusive(const int* in, int* out, int n, int* scratch, cudaStream_t st, long long* launches) {
    const int nb = n > 0 ? (n + SCAN_CHUNK - 1) / SCAN_CHUNK : 1;
    if (nb == 1) {
        launch_pdl(k_scan_chunks, dim3(1), dim3(SCAN_THREADS), 0, st, in, out, n, scratch, 1);
        *launches += 1;
        return;
    }
    if (n <= SCAN_CLUSTER_MAX) {
        launch_scan_cluster(in, out, n, st);
        *launches += 1;
        return;
    }
    // the level-2 scan handles up to SCAN_CHUNK block totals (n <= 16.7 M)
    launch_pdl(k_scan_chunks, dim3(nb), dim3(SCAN_THREADS), 0, st, in, out, n, scratch, 0);
    launch_pdl(k_scan_totals, dim3(1), dim3(SCAN_THREADS), 0, st, scratch, nb, out, n);
    launch_pdl(k_scan_add, dim3(nb), dim3(SCAN_THREADS), 0, st, out, n, scratch);
    *launches += 3;
}

}  // namespace pabd
