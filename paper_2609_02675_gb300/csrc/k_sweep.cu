// The semi-implicit successive-substitution sweep (Sec. 4.2-4.3), one launch pair per
// global/local iteration:
//
//   k_bond   one thread per bond: from q^k, the bond's split force (Eq. 15-17) as the two
//            ends' records (w, f'), w = h^2 phi+(d)/d and f' = f - w y_self, the right-hand
//            side term of Eq. 19 minus H's own-body term (the "delta" form) -- equal and
//            opposite f' on the two ends; each record is stored at the end's CSR slot.
//   k_solve  L lanes per body, a thread each or a thread per two (the warp-cooperative
//            gather): each lane adds its share of
//            the body's CSR slice and a fixed shuffle tree combines them; it forms, by the Kronecker
//            structure of H (Eq. 20, 23-24: H = P (G (x) I3) P^T with G the 4x4
//            diag(m, Pi) + sum w [1;x][1;x]^T), the 4x3 system G dX = M(s - q^k) + sum
//            [1;x] f'^T; factors G by Cholesky (the 12x12 Cholesky factor is L (x) I3),
//            solves the three right-hand sides, then takes the rotation of A^{k+1/2}
//            (the polar decomposition of sweep_math.cuh: Higham's scaled Newton
//            iteration, with an eigen-decomposition of A^T A as the fallback).
//            FP32, except bodies whose 4x4 factorisation is ill-conditioned (statically
//            flagged, or a Cholesky pivot below 1e-3 of its diagonal): those sum the same
//            single-precision records and factor in an extended type -- double-float on
//            the FP32 pipes (precision policy 1), or FP64 (policy 2).
#include "predict.cuh"
#include "sweep_shape.h"

namespace pabd {

constexpr int BOND_T = 256;
constexpr int SOLVE_T = 128;

// What a bond's records need that no sweep writes: its metadata and material points, the CSR
// slots of its ends and the ends' body flags (set at creation or by this step's front).
struct BondStatic {
    int4 m;
    float4 xi, xj;
    int p0, p1, fi, fj;
};

__device__ __forceinline__ BondStatic bond_static(const Dev& d, int b) {
    BondStatic s;
    s.m = d.bmeta[b];
    s.xi = d.bxi[b];
    s.xj = d.bxj[b];
    s.p0 = d.end_pos[2 * b];
    s.p1 = s.m.y >= 0 ? d.end_pos[2 * b + 1] : -1;
    s.fi = d.bflags[s.m.x];
    s.fj = s.m.y >= 0 ? d.bflags[s.m.y] : BF_PINNED;
    return s;
}

// one bond's end records from q^k
__device__ __forceinline__ void bond_one(const Dev& d, const float4* __restrict__ q, int it, int b,
                                         const BondStatic& s) {
    float c[3], A[9];
    ld_q(q, s.m.x, c, A);
    float co[3], Ao[9];
    ld_other(q, s.m.y, s.xj, co, Ao);
    EndBond e;
    e.xs = s.xi; e.xo = s.xj;
    e.nm = (s.m.z == K_CONTACT || s.m.z == K_GROUND) ? d.bn[b] : make_float4(0.f, 0.f, 0.f, 0.f);
    e.type = s.m.z; e.other = s.m.y; e.side_j = false; e.bond = b;
    // a bond between two fixed ends is advanced by the final update alone (as in the sweep kernels)
    const bool writer = !(s.fi & BF_PINNED) || !(s.fj & BF_PINNED);
    float f[3];
    const float w = end_force(d, e, co, Ao, c, A, it, writer, f);
    if (s.p0 >= 0) d.ends[s.p0] = make_float4(w, f[0], f[1], f[2]);
    if (s.p1 >= 0) d.ends[s.p1] = make_float4(w, -f[0], -f[1], -f[2]);
}

// (strides over this step's bonds with a grid capped at GS_BLOCKS blocks: the bond capacity
// holds room for every possible contact, far more than a step has).  Each thread loads its
// first bond's static part before it waits for the previous sweep (pdl_enter), so that the
// loads overlap that sweep's last blocks; q^k and the augmented Lagrangian state are read after.
// The first sweep follows the step's front itself, in a small scene the launch that writes the
// bonds and their slots: there nothing is read before the wait.
__global__ void __launch_bounds__(BOND_T, 5) k_bond(Dev d, const float4* __restrict__ q, int it) {
    if (it == 0) pdl_enter();
    const int nb = d.ctr[C_NBONDS];  // (set by the step's front, before the sweeps)
    const int b0 = blockIdx.x * blockDim.x + threadIdx.x;
    BondStatic s0;
    if (b0 < nb) s0 = bond_static(d, b0);
    if (it > 0) pdl_enter();
    // the solve launch that follows hands out its light bodies from this counter (the previous
    // solve launch has finished: pdl_enter waited for it)
    if (blockIdx.x == 0 && threadIdx.x == 0) d.ctr[C_SOLVE_NEXT] = 0;
    if (b0 < nb) bond_one(d, q, it, b0, s0);
    for (int b = b0 + gridDim.x * blockDim.x; b < nb; b += gridDim.x * blockDim.x) bond_one(d, q, it, b, bond_static(d, b));
}

// Sums a body's ends from the bond kernel's records, each loaded one round ahead of its sum (the
// loads of the next end overlap the arithmetic of this one).
struct RecordGather {
    const Dev& d;

    template <class T>
    __device__ __forceinline__ void one(Sys<T>& s, const float*, const float*, const float* xs, int p, int e1, int L) const {
        if (p >= e1) return;
        float4 e = d.ends[p], x = d.end_x[p];
        for (; p < e1; p += L) {
            const float4 ec = e, xc = x;
            if (p + L < e1) {
                e = d.ends[p + L];
                x = d.end_x[p + L];
            }
            sys_add(s, ec, xc, xs);
        }
    }
    // a heavy body's: few warps share its many ends, so a thread keeps several of them in flight
    // (a slab under 48 x 48 boxes: one end ahead 12.7 us a sweep, four at a time 10.6, eight,
    // which spills, 11.4)
    template <class T>
    __device__ __forceinline__ void many(Sys<T>& s, const float* c, const float* A, const float* xs, int p, int e1,
                                         int L) const {
        constexpr int U = sizeof(T) == 4 ? 4 : 2;
        for (; p + (U - 1) * L < e1; p += U * L) {
            float4 e[U], x[U];
#pragma unroll
            for (int k = 0; k < U; ++k) {
                e[k] = d.ends[p + k * L];
                x[k] = d.end_x[p + k * L];
            }
#pragma unroll
            for (int k = 0; k < U; ++k) sys_add(s, e[k], x[k], xs);
        }
        one(s, c, A, xs, p, e1, L);
    }
    template <class T>
    __device__ __forceinline__ void two(Sys<T>& s, Sys<T>& t, const float* c, const float* A, const float* xs, int p,
                                        int e1, int L) const {
        if (sizeof(T) != 4) {  // (a lane after the other: the second sum starts once the first is complete)
            one(s, c, A, xs, p, e1, L);
            one(t, c, A, xs, p + 1, e1, L);
            return;
        }
        for (; p + 1 < e1; p += L) {
            const float4 e0 = d.ends[p], x0 = d.end_x[p], e1_ = d.ends[p + 1], x1 = d.end_x[p + 1];
            sys_add(s, e0, x0, xs);
            sys_add(t, e1_, x1, xs);
        }
        if (p < e1) sys_add(s, d.ends[p], d.end_x[p], xs);
    }
};

// One body per P threads, which sum its L logical lanes (sys_sum_lanes); lane l adds the bond
// kernel's records of the body's ends l, l + L, ... -- in FP32, or in the extended type for a
// body on the extended path (the same records and order as the one-launch sweep, so the two
// modes agree bit for bit).  The first HEAVY_BLOCKS blocks take the heavy bodies (more than
// HEAVY_ENDS ends), and are dispatched first; the blocks after them stay resident and take the
// light bodies.
template <int L, int P, class X>
__global__ void __launch_bounds__(SOLVE_T, 4) k_solve(Dev d, const float4* __restrict__ qi, float4* __restrict__ qo,
                                                   int it) {
    pdl_enter();
    const int last = it == d.p.n_iter - 1;
    if ((int)blockIdx.x < HEAVY_BLOCKS) {
        heavy_role<X>(d, blockIdx.x, qi, qo, last, RecordGather{d});
        return;
    }
    // the light bodies in this step's (class, end count) order, or in body order (a body on
    // the heavy list then returns at once); either way the same arithmetic per body
    const int plane = threadIdx.x & (P - 1);
    for_light_slots<P>(&d.ctr[C_SOLVE_NEXT], d.light_sorted ? d.ctr[C_NLIGHT] : d.N, HEAVY_BLOCKS, [&](int slot, unsigned team) {
        const int b = d.light_sorted ? d.order[slot] : slot;
        solve_body<L, P, X>(d, b, plane, team, qi, qo, last, RecordGather{d});
    });
}

void launch_bond(const Dev& d, const float4* q, int it, cudaStream_t st, long long* launches) {
    launch_pdl(k_bond, dim3(stride_grid(d.cap_bonds > 0 ? d.cap_bonds : 1, BOND_T)), dim3(BOND_T), 0, st, d, q, it);
    *launches += 1;
}

void launch_solve(const Dev& d, const float4* q_in, float4* q_out, int it, int lanes, int threads, cudaStream_t st,
                  long long* launches) {
    static_assert(SOLVE_T == HEAVY_T, "the solve launch's blocks are the heavy bodies' blocks");
    // resident light blocks: as many as fit beside each other (4 per SM by the launch bounds),
    // fewer when the bodies do not need them
    const int slots = resident_slots(4);
    const long long n = (long long)(d.N > 0 ? d.N : 1) * threads;
    const long long need = (n + SOLVE_T - 1) / SOLVE_T;
    const int light = (int)(need < slots ? need : slots);
    with_sweep_shape(lanes, threads, d.p.precision_policy == 2, [&](auto l, auto p, auto x) {
        launch_pdl(k_solve<decltype(l)::value, decltype(p)::value, typename decltype(x)::type>,
                   dim3(HEAVY_BLOCKS + light), dim3(SOLVE_T), 0, st, d, q_in, q_out, it);
    });
    *launches += 1;
}

__global__ void k_al_warm(Dev d) {
    pdl_enter();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < d.Nc) al_warm(d, b);
}

// the dual update from the step's final iterate (after the last sweep), into parity n_iter
__global__ void k_al_final(Dev d, const float4* __restrict__ q) {
    pdl_enter();
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= d.Nc) return;
    const int4 m = d.bmeta[b];
    if (m.z != K_AL) return;
    const float4 xi = d.bxi[b], xj = d.bxj[b];
    float ci[3], Ai[9], cj[3], Aj[9], r[3];
    ld_q(q, m.x, ci, Ai);
    ld_other(q, m.y, xj, cj, Aj);
    bond_vec_dot2(ci, Ai, xi, cj, Aj, xj, false, r);
    const float cc = sqrtf(r[0] * r[0] + r[1] * r[1] + r[2] * r[2]) - xj.w;
    const int it = d.p.n_iter;
    const float beta = d.al_par[b].y;
    float2* out = (it & 1) ? d.al_st1 : d.al_st0;
    const bool fixed_i = d.bflags[m.x] & BF_PINNED, fixed_j = m.y < 0 || (d.bflags[m.y] & BF_PINNED);
    if (fixed_i && fixed_j) {
        // no sweep evaluates a bond between two fixed ends; its constraint is the same at every
        // iterate, so all n_iter updates are taken here from the warm start
        float2 kl = d.al_st0[b];
        for (int k = 0; k < it; ++k) kl = make_float2(kl.x + beta * fabsf(cc), kl.x * cc + kl.y);
        out[b] = kl;
        return;
    }
    const float2 kl = ((it - 1) & 1) ? d.al_st1[b] : d.al_st0[b];
    out[b] = make_float2(kl.x + beta * fabsf(cc), kl.x * cc + kl.y);
}

void launch_al_warm(const Dev& d, cudaStream_t st, long long* launches) {
    if (d.Nal == 0) return;
    launch_pdl(k_al_warm, dim3((d.Nc + 255) / 256), dim3(256), 0, st, d);
    *launches += 1;
}

void launch_al_final(const Dev& d, const float4* q, cudaStream_t st, long long* launches) {
    if (d.Nal == 0) return;
    launch_pdl(k_al_final, dim3((d.Nc + 255) / 256), dim3(256), 0, st, d, q);
    *launches += 1;
}

}  // namespace pabd
