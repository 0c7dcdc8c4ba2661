// Boxes, contact manifolds and the narrow phase's items, shared by the collision kernels
// (k_collision.cu) and the one-launch front of small scenes (k_front.cu).
//
// All arithmetic here that decides an integer (overlap, inside, face) uses __fmul_rn /
// __fadd_rn / __fsub_rn so that no multiply-add is contracted into an FMA.
#pragma once
#include "pair_filter.cuh"

namespace pabd {

#define FM(a, b) __fmul_rn((a), (b))
#define FA(a, b) __fadd_rn((a), (b))
#define FS(a, b) __fsub_rn((a), (b))

constexpr int NLEV = 3;           // levels of the multilevel grid
constexpr float LEV_RATIO = 4.f;  // cap ratio of consecutive levels

struct FBox {
    float c[3], A[9], he[3], infl;
};

__device__ __forceinline__ void load_q(const float4* q, int b, float* c, float* A) {
    float4 a = q[3 * b], bb = q[3 * b + 1], cc = q[3 * b + 2];
    c[0] = a.x; c[1] = a.y; c[2] = a.z;
    A[0] = a.w; A[1] = bb.x; A[2] = bb.y; A[3] = bb.z; A[4] = bb.w;
    A[5] = cc.x; A[6] = cc.y; A[7] = cc.z; A[8] = cc.w;
}

__device__ __forceinline__ void load_box(const Dev& d, int b, FBox& f) {
    load_q(d.qn, b, f.c, f.A);
    float4 h = d.he[b];
    f.he[0] = h.x; f.he[1] = h.y; f.he[2] = h.z;
    f.infl = d.lo[b].w;
}

// inflation of one body: (dhat + h*|v|) + margin, dhat = d_hat_rel * (2 * min he)
__device__ __forceinline__ float body_infl(const Dev& d, int b) {
    float4 h = d.he[b];
    float4 v = d.vel[b];
    float dh = FM(d.p.d_hat_rel, FM(2.0f, fminf(fminf(h.x, h.y), h.z)));
    float sp = __fsqrt_rn(FA(FA(FM(v.x, v.x), FM(v.y, v.y)), FM(v.z, v.z)));
    return FA(FA(dh, FM(d.p.h, sp)), d.p.margin);
}

// One body's AABB, inflation and grid level (one thread per body, b = the thread's global
// index, the threads at and above N already returned: the per-warp maximum below relies on it).
__device__ __forceinline__ void aabb_body(const Dev& d, int b) {
    float c[3], A[9];
    load_q(d.qn, b, c, A);
    float4 h = d.he[b];
    float infl = body_infl(d, b);
    float lo[3], hi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float e = FA(FA(FA(FM(fabsf(A[3 * k]), h.x), FM(fabsf(A[3 * k + 1]), h.y)), FM(fabsf(A[3 * k + 2]), h.z)), infl);
        lo[k] = FS(c[k], e);
        hi[k] = FA(c[k], e);
    }
    d.lo[b] = make_float4(lo[0], lo[1], lo[2], infl);
    d.hi[b] = make_float4(hi[0], hi[1], hi[2], 0.f);
    // off the grid: flagged large, or (with a fixed cell size) a box wider than a cell -- a fast
    // body whose inflation grew its box -- or a box that is not finite
    // The cell is the widest grid box of this step (times 1.01); with a scene cap p.cell, a box
    // wider than the cap leaves the grid instead of widening every cell.
    const float w = fmaxf(fmaxf(FS(hi[0], lo[0]), FS(hi[1], lo[1])), FS(hi[2], lo[2]));
    bool large = d.bflags[b] & BF_LARGE;
    int lv = 0;
    if (d.p.cell > 0.f) {
        if (d.multilevel) {  // the first level whose cap (cell cap x 4^level) holds the box
            float cap = d.p.cell;
            while (lv < NLEV - 1 && !(w <= cap)) { cap *= LEV_RATIO; ++lv; }
            large = large || !(w <= cap);
        } else {
            large = large || !(w <= d.p.cell);
        }
    }
    // the widest box of each level (positive floats order as ints): a warp's maximum first, then
    // one atomic per warp and level -- one per body on a single word serialises in L2
    const float wc = w * 1.01f + 1e-6f;
    const int bits = (!large && wc < 1e30f) ? __float_as_int(wc) : 0;
    const int wbase = b - (int)(threadIdx.x & 31);  // the warp's lanes below N (those above returned)
    const unsigned act = d.N - wbase >= 32 ? 0xffffffffu : ((1u << (d.N - wbase)) - 1u);
    const bool leader = (threadIdx.x & 31) == 0;
    for (int l = 0; l < (d.multilevel ? NLEV : 1); ++l) {
        const int m = __reduce_max_sync(act, lv == l ? bits : 0);
        if (leader && m > 0) atomicMax(&d.ctr[l == 0 ? C_CELLBITS : C_CELLBITS1 + l - 1], m);
    }
    if (d.bvh_bounds) {  // LBVH: the box of the finite centres, as order-preserving ints
        const float x[3] = {0.5f * (lo[0] + hi[0]), 0.5f * (lo[1] + hi[1]), 0.5f * (lo[2] + hi[2])};
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int i = __float_as_int(x[k]), o = i >= 0 ? i : i ^ 0x7fffffff;
            const bool fin = isfinite(x[k]);
            const int mn = __reduce_min_sync(act, fin ? o : 0x7fffffff), mx = __reduce_max_sync(act, fin ? o : (int)0x80000000);
            if (leader) {
                atomicMin(&d.bvh_bounds[k], mn);
                atomicMax(&d.bvh_bounds[3 + k], mx);
            }
        }
    }
    d.cell[b] = make_int4(0, 0, 0, large ? -1 : 0);
    if (d.blevel) d.blevel[b] = large ? -1 : lv;
    if (large && d.large_ids) d.large_ids[atomicAdd(&d.ctr[C_NLARGE], 1)] = b;
}

struct CPt {
    float u[3], x[3];
};

__device__ __forceinline__ float dot_col(const float* A, int l, const float* r) {
    return FA(FA(FM(A[l], r[0]), FM(A[3 + l], r[1])), FM(A[6 + l], r[2]));
}

// Manifold of the pair (a, b); calls emit(i, j, x_i, x_j, N) for each contact, returns count.
template <class Emit>
__device__ int box_box(const FBox& fa, const FBox& fb, int a, int b, Emit&& emit) {
    const float delta = FA(fa.infl, fb.infl);
    float dv[3], dab[3], dba[3], R[9];
#pragma unroll
    for (int k = 0; k < 3; ++k) dv[k] = FS(fa.c[k], fb.c[k]);
#pragma unroll
    for (int l = 0; l < 3; ++l) dab[l] = dot_col(fb.A, l, dv);
    float dn[3] = {-dv[0], -dv[1], -dv[2]};
#pragma unroll
    for (int k = 0; k < 3; ++k) dba[k] = dot_col(fa.A, k, dn);
#pragma unroll
    for (int l = 0; l < 3; ++l)
#pragma unroll
        for (int k = 0; k < 3; ++k)
            R[3 * l + k] = FA(FA(FM(fb.A[l], fa.A[k]), FM(fb.A[3 + l], fa.A[3 + k])), FM(fb.A[6 + l], fa.A[6 + k]));
    float best = 0.f;
    int ref_b = 1, l = 0;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        float ext = FA(FA(FM(fabsf(R[3 * ax]), fa.he[0]), FM(fabsf(R[3 * ax + 1]), fa.he[1])), FM(fabsf(R[3 * ax + 2]), fa.he[2]));
        float sep = FS(fabsf(dab[ax]), FA(fb.he[ax], ext));
        if (ax == 0 || sep > best) { best = sep; ref_b = 1; l = ax; }
    }
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
        float ext = FA(FA(FM(fabsf(R[ax]), fb.he[0]), FM(fabsf(R[3 + ax]), fb.he[1])), FM(fabsf(R[6 + ax]), fb.he[2]));
        float sep = FS(fabsf(dba[ax]), FA(fa.he[ax], ext));
        if (sep > best) { best = sep; ref_b = 0; l = ax; }
    }
    if (!(best <= delta)) return 0;
    const FBox& fr = ref_b ? fb : fa;
    const FBox& fi = ref_b ? fa : fb;
    const int ir = ref_b ? b : a, ii = ref_b ? a : b;
    const float sg = ref_b ? (dab[l] >= 0.f ? 1.f : -1.f) : (dba[l] >= 0.f ? 1.f : -1.f);
    float N[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) N[k] = FM(sg, fr.A[3 * k + l]);
    int ki = 0;
    float bestd = 0.f, dsel = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float dk = dot_col(fi.A, k, N);
        if (k == 0 || fabsf(dk) > bestd) { bestd = fabsf(dk); ki = k; dsel = dk; }
    }
    const float si = dsel > 0.f ? -1.f : 1.f;
    const int k1 = (ki + 1) % 3, k2 = (ki + 2) % 3;
    const float sgn1[4] = {1.f, -1.f, -1.f, 1.f}, sgn2[4] = {1.f, 1.f, -1.f, -1.f};
    CPt poly[8], tmp[8];
    int np = 4;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        float x[3], y[3], r[3];
        x[ki] = FM(si, fi.he[ki]);
        x[k1] = FM(sgn1[v], fi.he[k1]);
        x[k2] = FM(sgn2[v], fi.he[k2]);
#pragma unroll
        for (int dd = 0; dd < 3; ++dd) {
            y[dd] = FA(FA(FA(fi.c[dd], FM(fi.A[3 * dd], x[0])), FM(fi.A[3 * dd + 1], x[1])), FM(fi.A[3 * dd + 2], x[2]));
            r[dd] = FS(y[dd], fr.c[dd]);
        }
#pragma unroll
        for (int m = 0; m < 3; ++m) { poly[v].u[m] = dot_col(fr.A, m, r); poly[v].x[m] = x[m]; }
    }
    const int m1 = (l + 1) % 3, m2 = (l + 2) % 3;
    for (int pl = 0; pl < 4 && np > 0; ++pl) {
        const int m = pl < 2 ? m1 : m2;
        const float ps = (pl & 1) ? -1.f : 1.f, lim = fr.he[m];
        int nt = 0;
        for (int v = 0; v < np; ++v) {
            const CPt& P = poly[v];
            const CPt& Q = poly[(v + 1) % np];
            float dp = FS(FM(ps, P.u[m]), lim), dq = FS(FM(ps, Q.u[m]), lim);
            bool pin = dp <= 0.f, qin = dq <= 0.f;
            if (pin) tmp[nt++] = P;
            if (pin != qin) {
                float t = __fdiv_rn(dp, FS(dp, dq));
                CPt X;
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    X.u[c] = FA(P.u[c], FM(t, FS(Q.u[c], P.u[c])));
                    X.x[c] = FA(P.x[c], FM(t, FS(Q.x[c], P.x[c])));
                }
                tmp[nt++] = X;
            }
        }
        np = nt;
        for (int v = 0; v < nt; ++v) poly[v] = tmp[v];
    }
    int cnt = 0;
    for (int v = 0; v < np; ++v) {
        float hgt = FS(FM(sg, poly[v].u[l]), fr.he[l]);
        if (!(hgt < delta)) continue;
        float xj[3] = {poly[v].u[0], poly[v].u[1], poly[v].u[2]};
        xj[l] = FM(sg, fr.he[l]);
        emit(ii, ir, poly[v].x, xj, N, cnt);
        ++cnt;
    }
    return cnt;
}

template <class Emit>
__device__ int ground_corners(const Dev& d, const FBox& fa, int a, Emit&& emit) {
    int cnt = 0;
#pragma unroll 1
    for (int k = 0; k < 8; ++k) {
        float x[3] = {(k & 1) ? fa.he[0] : -fa.he[0], (k & 2) ? fa.he[1] : -fa.he[1], (k & 4) ? fa.he[2] : -fa.he[2]};
        float y[3];
#pragma unroll
        for (int dd = 0; dd < 3; ++dd)
            y[dd] = FA(FA(FA(fa.c[dd], FM(fa.A[3 * dd], x[0])), FM(fa.A[3 * dd + 1], x[1])), FM(fa.A[3 * dd + 2], x[2]));
        float g = FS(FA(FA(FM(d.p.gn[0], y[0]), FM(d.p.gn[1], y[1])), FM(d.p.gn[2], y[2])), d.p.gd);
        if (!(g < fa.infl)) continue;
        float anc[3] = {FS(y[0], FM(g, d.p.gn[0])), FS(y[1], FM(g, d.p.gn[1])), FS(y[2], FM(g, d.p.gn[2]))};
        emit(a, -1, x, anc, d.p.gn, cnt);
        ++cnt;
    }
    return cnt;
}

__device__ __forceinline__ float pair_dhat(const Dev& d, int i, int j) {
    float di = d.he[i].w;
    return j < 0 ? di : fminf(di, d.he[j].w);
}

// a contact as a bond's four arrays hold it
struct Contact {
    int4 m;
    float4 xi, xj, bn;
};

// contact number `slot` of the step, written as bond Nc + slot while there is room
__device__ __forceinline__ Contact write_contact(const Dev& d, int slot, int type, int i, int j, const float* xi,
                                                 const float* xj, const float* N) {
    Contact c;
    if (slot >= d.cap_contacts) return c;
    const int b = d.Nc + slot;
    float mi = d.mass[i].x;
    float mm;
    if (j < 0) mm = mi;
    else {
        float mj = d.mass[j].x;
        bool pi = d.bflags[i] & BF_PINNED, pj = d.bflags[j] & BF_PINNED;
        mm = pj ? mi : (pi ? mj : fminf(mi, mj));
    }
    c.m = make_int4(i, j, type, 0);
    c.xi = make_float4(xi[0], xi[1], xi[2], d.p.c_kappa * mm);
    c.xj = make_float4(xj[0], xj[1], xj[2], pair_dhat(d, i, j));
    c.bn = make_float4(N[0], N[1], N[2], d.p.mu);
    d.bmeta[b] = c.m;
    d.bxi[b] = c.xi;
    d.bxj[b] = c.xj;
    d.bn[b] = c.bn;
    return c;
}

// One item of the narrow phase's two passes.  Items [0, np) are this step's pairs, items np + b
// the ground corners of body b (apart, so that no item runs both manifolds in series).
__device__ __forceinline__ void narrow_count_item(const Dev& d, int tt, int np) {
    if (tt < np) {
        int2 pr = d.pairs[tt];
        FBox fa, fb;
        load_box(d, pr.x, fa);
        load_box(d, pr.y, fb);
        d.npc[tt] = box_box(fa, fb, pr.x, pr.y, [](int, int, const float*, const float*, const float*, int) {});
    } else {
        const int t = tt - np;
        int n = 0;
        if (d.p.has_ground && !(d.bflags[t] & BF_PINNED)) {
            FBox fa;
            load_box(d, t, fa);
            n = ground_corners(d, fa, t, [](int, int, const float*, const float*, const float*, int) {});
        }
        d.gnd_cnt[t] = n;
    }
}

// writes the item's contacts from npc_off and, after the npc pair contacts, gnd_off on;
// written(i, j) follows each one that has room
template <class Written>
__device__ __forceinline__ void narrow_write_item(const Dev& d, int tt, int np, int npc, Written&& written) {
    if (tt < np) {
        int2 pr = d.pairs[tt];
        FBox fa, fb;
        load_box(d, pr.x, fa);
        load_box(d, pr.y, fb);
        const int base = d.npc_off[tt];
        box_box(fa, fb, pr.x, pr.y, [&](int i, int j, const float* xi, const float* xj, const float* N, int k) {
            write_contact(d, base + k, K_CONTACT, i, j, xi, xj, N);
            if (base + k < d.cap_contacts) written(i, j);
        });
    } else {
        const int t = tt - np;
        if (d.gnd_cnt[t] > 0) {
            FBox fa;
            load_box(d, t, fa);
            const int base = npc + d.gnd_off[t];
            ground_corners(d, fa, t, [&](int i, int j, const float* xi, const float* xj, const float* N, int k) {
                write_contact(d, base + k, K_GROUND, i, j, xi, xj, N);
                if (base + k < d.cap_contacts) written(i, j);
            });
        }
    }
}

// the step's contact and bond counts, once both prefix sums are known (one thread)
__device__ __forceinline__ void set_contact_counts(const Dev& d, int npc) {
    int nk = npc + d.gnd_off[d.N];
    if (nk > d.cap_contacts) { latch_status(d, ST_CAPACITY); nk = d.cap_contacts; }
    d.ctr[C_NPC] = min(npc, d.cap_contacts);
    d.ctr[C_NGC] = nk - min(npc, d.cap_contacts);
    d.ctr[C_NBONDS] = d.Nc + nk;
}

}  // namespace pabd
