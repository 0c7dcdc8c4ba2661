// One launch per sweep (sweep mode 2): every body gathers its bond ends from the CSR-ordered
// end records, evaluates each bond's split force from q^k (Eq. 15-17) and solves its 4x4
// system and local rotation (Eq. 19-24, Sec. 4.3); the launch boundary orders the sweeps.
#include "sweep_shape.h"

namespace pabd {

// One sweep per launch: the same per-body work as the fused kernel, with the launch boundary
// (a graph edge) in place of the grid barrier.  Capped at 128 registers (4 blocks per SM),
// without spills (the fused kernel, which loops over the sweeps, spills a few bytes).  The
// first HEAVY_BLOCKS blocks take the heavy bodies (more than HEAVY_ENDS ends) and are
// dispatched first; the blocks after them stay resident and take the light bodies (L lanes
// each, in the step's light order), a warp's worth at a time (for_light_slots).
template <int L, int P, class X>
__global__ void __launch_bounds__(128, 4) k_sweep_one(Dev d, const float4* __restrict__ qi, float4* __restrict__ qo,
                                                   int it) {
    // Programmatic dependent launch: wait until the previous sweep has completed and its writes
    // are visible (a no-op when launched without the attribute); no early signal to the next
    // sweep, whose waiting blocks would take SM slots (measured slower)
    pdl_enter();
    int last = it == d.p.n_iter - 1;
    if (it < 0) {
        // under a residual threshold: the sweep index and buffers from the device, the
        // per-body residual every sweep; nothing once the loop has ended (eager launches)
        if (!d.sweep_ctl[2]) return;
        it = d.sweep_ctl[0];
        qi = (it & 1) ? d.qb : d.qa;
        qo = (it & 1) ? d.qa : d.qb;
        last = 1;
    }
    // this sweep's counter of light chunks, and the next sweep's zeroed (the previous sweep,
    // which used it, has finished)
    int* next = &d.ctr[C_SWEEP_NEXT + (it & 1)];
    if (blockIdx.x == 0 && threadIdx.x == 0) d.ctr[C_SWEEP_NEXT + ((it + 1) & 1)] = 0;
    if ((int)blockIdx.x < HEAVY_BLOCKS) {
        heavy_role<X>(d, blockIdx.x, qi, qo, last, end_gather(d, GlobalQ{qi}, it));
        return;
    }
    // the light bodies in this step's (class, end count) order, or in body order (a body on
    // the heavy list then returns at once); either way the same arithmetic per body
    const int plane = threadIdx.x & (P - 1);
    for_light_slots<P>(next, d.light_sorted ? d.ctr[C_NLIGHT] : d.N, HEAVY_BLOCKS, [&](int slot, unsigned team) {
        const int b = d.light_sorted ? d.order[slot] : slot;
        solve_body<L, P, X>(d, b, plane, team, qi, qo, last, end_gather(d, GlobalQ{qi}, it));
    });
}

// `pdl`: launched as a programmatic dependent of the previous kernel on the stream (the
// previous sweep), so that its launch overlaps that sweep's tail.  The extended type of
// ill-conditioned bodies: FP64 under policy 2, double-float otherwise.
void launch_sweep_one(const Dev& d, const float4* qi, float4* qo, int it, int lanes, int threads, cudaStream_t st,
                      long long* launches, bool pdl) {
    static_assert(HEAVY_T == 128, "the sweep launch's blocks are the heavy bodies' blocks");
    const long long n = (long long)(d.N > 0 ? d.N : 1) * threads;
    const long long need = (n + 127) / 128;
    const int slots = resident_slots(4);
    const int grid = HEAVY_BLOCKS + (int)(need < slots ? need : slots);
    with_sweep_shape(lanes, threads, d.p.precision_policy == 2, [&](auto l, auto p, auto x) {
        auto kernel = k_sweep_one<decltype(l)::value, decltype(p)::value, typename decltype(x)::type>;
        if (pdl) launch_pdl(kernel, dim3(grid), dim3(128), 0, st, d, qi, qo, it);
        else kernel<<<grid, 128, 0, st>>>(d, qi, qo, it);
    });
    *launches += 1;
}

}  // namespace pabd
