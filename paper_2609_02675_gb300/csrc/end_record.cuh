// The bond-end records that the sweeps read (written where the CSR is built, read by unpack_end).
#pragma once
#include "pabd_internal.h"

namespace pabd {

// ---- bond-end records in CSR order (Dev::rec, three float4 per end) ----
// (x of the end, w0), (x of the other end, p1) and (N, code): everything one evaluation of the
// bond reads but the two iterates, in 48 contiguous bytes.  code packs the other body + 1 (24
// bits; 0: the world), the side (bit 24) and the type (from bit 25); a bond without a normal
// keeps its id in N's place.  mu is the scene's.  Four separate records (metadata, x_i, x_j, and
// the normal by bond id) took 64 bytes and a fourth cache line per end.
__device__ __forceinline__ void pack_end(float4* __restrict__ rec, int bond, int4 m, float4 xi, float4 xj, float4 bn,
                                         bool side_j) {
    const int other = side_j ? m.x : m.y;
    const int code = (other + 1) | (side_j ? 1 << 24 : 0) | (m.z << 25);
    const bool contact = m.z == K_CONTACT || m.z == K_GROUND;
    rec[0] = side_j ? make_float4(xj.x, xj.y, xj.z, xi.w) : xi;
    rec[1] = side_j ? make_float4(xi.x, xi.y, xi.z, xj.w) : xj;
    rec[2] = contact ? make_float4(bn.x, bn.y, bn.z, __int_as_float(code))
                     : make_float4(__int_as_float(bond), 0.f, 0.f, __int_as_float(code));
}

}  // namespace pabd
