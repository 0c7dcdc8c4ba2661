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

// A corner of the clipped incident face: u, its place in the reference box's frame, and (xa, xb),
// its two coordinates along the incident face in the incident box's frame (the third is the
// face's).  A polygon under clipping is read from one buffer of eight corners and written to
// another; Poly::at(buffer, corner, component) says where they are.
struct Corner {
    float u[3], xa, xb;
};
struct LocalPoly {
    float c[2][8][5];
    __device__ __forceinline__ float& at(int b, int v, int k) { return c[b][v][k]; }
};
// in shared memory, element e of thread t at e T + t: no bank conflicts whatever the corner.
// (Indexed by run-time corners, the buffers cannot be registers; in local memory the 384 bytes
// of 800 threads per SM did not fit the L1 cache beside the shared memory.)
template <int T>
struct SharedPoly {
    float* base;  // the thread's element 0
    __device__ __forceinline__ float& at(int b, int v, int k) const { return base[((b * 8 + v) * 5 + k) * T]; }
};
template <class Poly>
__device__ __forceinline__ Corner ld_corner(Poly& poly, int b, int v) {
    return Corner{{poly.at(b, v, 0), poly.at(b, v, 1), poly.at(b, v, 2)}, poly.at(b, v, 3), poly.at(b, v, 4)};
}
template <class Poly>
__device__ __forceinline__ void st_corner(Poly& poly, int b, int v, const Corner& c) {
#pragma unroll
    for (int k = 0; k < 3; ++k) poly.at(b, v, k) = c.u[k];
    poly.at(b, v, 3) = c.xa;
    poly.at(b, v, 4) = c.xb;
}
__device__ __forceinline__ float pick3(const float* v, int k) { return k == 0 ? v[0] : (k == 1 ? v[1] : v[2]); }

__device__ __forceinline__ float dot_col(const float* A, int l, const float* r) {
    return FA(FA(FM(A[l], r[0]), FM(A[3 + l], r[1])), FM(A[6 + l], r[2]));
}

// What a pair's contacts share: the incident and the reference body, the normal, and the incident
// face (its axis ki and the coordinate xk along it).
struct Manifold {
    int ii, ir, ki;
    float xk, N[3];
};
// the contact point in the incident body's frame
__device__ __forceinline__ void corner_point(int ki, float xk, float xa, float xb, float* x) {
    x[0] = ki == 0 ? xk : (ki == 2 ? xa : xb);
    x[1] = ki == 1 ? xk : (ki == 0 ? xa : xb);
    x[2] = ki == 2 ? xk : (ki == 1 ? xa : xb);
}

// Manifold of the pair (a, b); calls emit(corner, k) for contact k, whose corner's u is the point
// in the reference body's frame, returns the count.  emit may write to buffer `out` of the
// polygon up to corner k.
template <class Poly, class Emit>
__device__ __forceinline__ int box_box(const FBox& fa, const FBox& fb, int a, int b, Poly& poly, Manifold& mf, int& out,
                                       Emit&& emit) {
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
    // the reference and the incident box (selected value by value: an index into the two boxes
    // would put them in memory)
    FBox fr, fi;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        fr.c[k] = ref_b ? fb.c[k] : fa.c[k];
        fi.c[k] = ref_b ? fa.c[k] : fb.c[k];
        fr.he[k] = ref_b ? fb.he[k] : fa.he[k];
        fi.he[k] = ref_b ? fa.he[k] : fb.he[k];
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        fr.A[k] = ref_b ? fb.A[k] : fa.A[k];
        fi.A[k] = ref_b ? fa.A[k] : fb.A[k];
    }
    mf.ir = ref_b ? b : a;
    mf.ii = ref_b ? a : b;
    const float dl = ref_b ? pick3(dab, l) : pick3(dba, l);
    const float sg = dl >= 0.f ? 1.f : -1.f, hl = pick3(fr.he, l);
    float N[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) mf.N[k] = N[k] = FM(sg, pick3(fr.A + 3 * k, l));
    int ki = 0;
    float bestd = 0.f, dsel = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        float dk = dot_col(fi.A, k, N);
        if (k == 0 || fabsf(dk) > bestd) { bestd = fabsf(dk); ki = k; dsel = dk; }
    }
    const float si = dsel > 0.f ? -1.f : 1.f;
    const int k1 = ki == 2 ? 0 : ki + 1, k2 = ki == 0 ? 2 : ki - 1;
    mf.ki = ki;
    mf.xk = FM(si, pick3(fi.he, ki));
    const float h1 = pick3(fi.he, k1), h2 = pick3(fi.he, k2);
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const float sgn1 = v == 0 || v == 3 ? 1.f : -1.f, sgn2 = v < 2 ? 1.f : -1.f;
        Corner c;
        c.xa = FM(sgn1, h1);
        c.xb = FM(sgn2, h2);
        float x[3], r[3];
        corner_point(ki, mf.xk, c.xa, c.xb, x);
#pragma unroll
        for (int dd = 0; dd < 3; ++dd) {
            const float y = FA(FA(FA(fi.c[dd], FM(fi.A[3 * dd], x[0])), FM(fi.A[3 * dd + 1], x[1])), FM(fi.A[3 * dd + 2], x[2]));
            r[dd] = FS(y, fr.c[dd]);
        }
#pragma unroll
        for (int m = 0; m < 3; ++m) c.u[m] = dot_col(fr.A, m, r);
        st_corner(poly, 0, v, c);
    }
    const int m1 = l == 2 ? 0 : l + 1, m2 = l == 0 ? 2 : l - 1;
    int np = 4, src = 0;
    for (int pl = 0; pl < 4 && np > 0; ++pl) {
        const int m = pl < 2 ? m1 : m2;
        const float ps = (pl & 1) ? -1.f : 1.f, lim = pick3(fr.he, m);
        const Corner first = ld_corner(poly, src, 0);
        const float dfirst = FS(FM(ps, pick3(first.u, m)), lim);
        Corner P = first;
        float dp = dfirst;
        int nt = 0;
        for (int v = 0; v < np; ++v) {
            Corner Q = first;
            float dq = dfirst;
            if (v + 1 < np) {
                Q = ld_corner(poly, src, v + 1);
                dq = FS(FM(ps, pick3(Q.u, m)), lim);
            }
            const bool pin = dp <= 0.f, qin = dq <= 0.f;
            if (pin && nt < 8) st_corner(poly, src ^ 1, nt++, P);
            if (pin != qin && nt < 8) {
                const float t = __fdiv_rn(dp, FS(dp, dq));
                Corner X;
#pragma unroll
                for (int c = 0; c < 3; ++c) X.u[c] = FA(P.u[c], FM(t, FS(Q.u[c], P.u[c])));
                X.xa = FA(P.xa, FM(t, FS(Q.xa, P.xa)));
                X.xb = FA(P.xb, FM(t, FS(Q.xb, P.xb)));
                st_corner(poly, src ^ 1, nt++, X);
            }
            P = Q;
            dp = dq;
        }
        np = nt;
        src ^= 1;
    }
    out = src ^ 1;
    int cnt = 0;
    const float top = FM(sg, hl);
    for (int v = 0; v < np; ++v) {
        Corner c = ld_corner(poly, src, v);
        const float hgt = FS(FM(sg, pick3(c.u, l)), hl);
        if (!(hgt < delta)) continue;
#pragma unroll
        for (int k = 0; k < 3; ++k)
            if (k == l) c.u[k] = top;
        emit(c, cnt);
        ++cnt;
    }
    return cnt;
}

// contacts of body a's corners with the ground; emit(a, corner, x, anchor, k) for contact k
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
        emit(a, k, x, anc, cnt);
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

// h^2 kappa_c of the contacts of bodies i and j (the ground: j < 0)
__device__ __forceinline__ float contact_weight(const Dev& d, int i, int j) {
    float mi = d.mass[i].x;
    float mm;
    if (j < 0) mm = mi;
    else {
        float mj = d.mass[j].x;
        bool pi = d.bflags[i] & BF_PINNED, pj = d.bflags[j] & BF_PINNED;
        mm = pj ? mi : (pi ? mj : fminf(mi, mj));
    }
    return d.p.c_kappa * mm;
}

// contact number `slot` of the step, written as bond Nc + slot while there is room
__device__ __forceinline__ void store_contact(const Dev& d, int slot, const Contact& c) {
    if (slot >= d.cap_contacts) return;
    const int b = d.Nc + slot;
    d.bmeta[b] = c.m;
    d.bxi[b] = c.xi;
    d.bxj[b] = c.xj;
    d.bn[b] = c.bn;
}

__device__ __forceinline__ Contact write_contact(const Dev& d, int slot, int type, int i, int j, const float* xi,
                                                 const float* xj, const float* N) {
    Contact c;
    if (slot >= d.cap_contacts) return c;
    c.m = make_int4(i, j, type, 0);
    c.xi = make_float4(xi[0], xi[1], xi[2], contact_weight(d, i, j));
    c.xj = make_float4(xj[0], xj[1], xj[2], pair_dhat(d, i, j));
    c.bn = make_float4(N[0], N[1], N[2], d.p.mu);
    store_contact(d, slot, c);
    return c;
}

// Contacts of one narrow-phase item, counted alone.  Items [0, np) are this step's pairs, items
// np + b the ground corners of body b (apart, so that no item runs both manifolds in series).
__device__ __forceinline__ int narrow_item_contacts(const Dev& d, int tt, int np) {
    if (tt < np) {
        int2 pr = d.pairs[tt];
        FBox fa, fb;
        load_box(d, pr.x, fa);
        load_box(d, pr.y, fb);
        LocalPoly poly;
        Manifold mf;
        int out;
        return box_box(fa, fb, pr.x, pr.y, poly, mf, out, [](const Corner&, int) {});
    }
    const int t = tt - np;
    if (!d.p.has_ground || (d.bflags[t] & BF_PINNED)) return 0;
    FBox fa;
    load_box(d, t, fa);
    return ground_corners(d, fa, t, [](int, int, const float*, const float*, int) {});
}

// an item of the first of the small front's two narrow passes
__device__ __forceinline__ void narrow_count_item(const Dev& d, int tt, int np) {
    const int n = narrow_item_contacts(d, tt, np);
    if (tt < np) d.npc[tt] = n;
    else d.gnd_cnt[tt - np] = n;
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
        LocalPoly poly;
        Manifold mf;
        int out;
        box_box(fa, fb, pr.x, pr.y, poly, mf, out, [&](const Corner& c, int k) {
            float x[3];
            corner_point(mf.ki, mf.xk, c.xa, c.xb, x);
            write_contact(d, base + k, K_CONTACT, mf.ii, mf.ir, x, c.u, mf.N);
            if (base + k < d.cap_contacts) written(mf.ii, mf.ir);
        });
    } else {
        const int t = tt - np;
        if (d.gnd_cnt[t] > 0) {
            FBox fa;
            load_box(d, t, fa);
            const int base = npc + d.gnd_off[t];
            ground_corners(d, fa, t, [&](int i, int, const float* xi, const float* xj, int k) {
                write_contact(d, base + k, K_GROUND, i, -1, xi, xj, d.p.gn);
                if (base + k < d.cap_contacts) written(i, -1);
            });
        }
    }
}

// the step's contact and bond counts, once both prefix sums are known (one thread)
__device__ __forceinline__ void set_contact_counts(const Dev& d, int npc) {
    int nk = npc + d.gnd_off[d.N];
    if (nk > d.cap_contacts) { latch_status(d, ST_CAPACITY); nk = d.cap_contacts; }
    d.ctr[C_NCONTACTS] = nk;
    d.ctr[C_NBONDS] = d.Nc + nk;
}

}  // namespace pabd
