// Device helpers shared by the structured-mesh kernels: the field kernel
// (lbfsi_fields.cu) and the step kernel (lbfsi_step.cu).
#pragma once

#include "lbfsi_device.cuh"
#include "lbfsi_internal.h"

namespace lbfsi {

template <typename R>
struct Vec2;
template <>
struct Vec2<float> {
    using T = float2;
};
template <>
struct Vec2<double> {
    using T = double2;
};

// Four consecutive table entries (16-byte aligned) in one or two loads.
__device__ __forceinline__ void ld4(const float* p, float& a, float& b, float& c, float& d) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    a = v.x; b = v.y; c = v.z; d = v.w;
}
__device__ __forceinline__ void ld4(const double* p, double& a, double& b, double& c, double& d) {
    const double2 u = *reinterpret_cast<const double2*>(p);
    const double2 v = *reinterpret_cast<const double2*>(p + 2);
    a = u.x; b = u.y; c = v.x; d = v.y;
}

// Bounds-checked build (LBFSI_BOUNDS_CHECK): the shared-memory windows the
// step reads and the global slots it writes are checked; an index outside
// its buffer sets ST_BOUNDS and the access is skipped.  The substitute for a
// memory checker where none can run; without the macro every check is true.
#ifdef LBFSI_BOUNDS_CHECK
__device__ __forceinline__ bool in_bounds(bool ok, unsigned* st) {
    if (!ok) atomicOr(st, ST_BOUNDS);
    return ok;
}
#else
__device__ __forceinline__ bool in_bounds(bool, unsigned*) { return true; }
#endif

// Derivative along an index direction of the 1-D quadratic Lagrange interpolant
// through a node and its neighbours, evaluated at the node (Eq. ddx+fem):
// central inside, one-sided (-3 c0 + 4 c1 - c2)/2 on the first row,
// (3 cN - 4 cN-1 + cN-2)/2 on the last.  p points at the node.
template <typename R>
__device__ __forceinline__ R d_row(const R* p, int stride, int i, int nr) {
    if (i == 0) return R(0.5) * fm(R(-3), p[0], fm(R(4), p[stride], -p[2 * stride]));
    if (i == nr - 1) return R(0.5) * fm(R(3), p[0], fm(R(-4), p[-stride], p[-2 * stride]));
    return R(0.5) * (p[stride] - p[-stride]);
}
template <typename R>
__device__ __forceinline__ R d_col(const R* p) {
    return R(0.5) * (p[1] - p[-1]);
}
// The same stencils on a general mesh that may be a C-grid (cg): central
// along i at row-0 nodes whose row below is the mirrored row across the cut
// (across), one-sided along j at the outlet columns and, at the two copies of
// the rear point, along the cut.  With cg == 0 and across == false they are
// d_row and d_col.
template <typename R>
__device__ __forceinline__ R d_row_c(const R* p, int stride, int i, int nr, bool across, bool wrap_rows = false) {
    if (!wrap_rows) {   // a periodic box has no first or last row
        if (i == 0 && !across) return R(0.5) * fm(R(-3), p[0], fm(R(4), p[stride], -p[2 * stride]));
        if (i == nr - 1) return R(0.5) * fm(R(3), p[0], fm(R(-4), p[-stride], p[-2 * stride]));
    }
    return R(0.5) * (p[stride] - p[-stride]);
}
// jdir: at a row-0 junction of a C-grid, +1 (the cut is the next column) or
// -1 (the previous one); 0 elsewhere.
template <typename R>
__device__ __forceinline__ R d_col_c(const R* p, int j, int nt, int cg, int jdir) {
    if (cg) {
        if (j == 0 || jdir > 0) return R(0.5) * fm(R(-3), p[0], fm(R(4), p[1], -p[2]));
        if (j == nt - 1 || jdir < 0) return R(0.5) * fm(R(3), p[0], fm(R(-4), p[-1], p[-2]));
    }
    return R(0.5) * (p[1] - p[-1]);
}

template <typename R>
__device__ __forceinline__ void lagrange3(R t, R* L) {
    L[0] = t * fm(R(0.5), t, R(-0.5));
    L[1] = fm(-t, t, R(1));
    L[2] = t * fm(R(0.5), t, R(0.5));
}

// Map from index derivatives (C_xi, C_eta) at a node to the physical gradient:
// grad_X C = J^{-1} (C_xi, C_eta) (Eq. ddx+fem) with the separable O-grid
// metric, then grad_x = g^{-1} grad_X = F^{-T} grad_X (Eq. dx_ref).
template <typename R>
__device__ __forceinline__ void grad_map_j(R j00, R j01, R j10, R j11, R F00, R F01, R F10, R F11,
                                           R* G) {
    const R idet = rcp_(fm(F00, F11, -(F01 * F10)));
    const R i00 = F11 * idet, i01 = -F01 * idet, i10 = -F10 * idet, i11 = F00 * idet;
    G[0] = fm(i00, j00, i10 * j10);
    G[1] = fm(i00, j01, i10 * j11);
    G[2] = fm(i01, j00, i11 * j10);
    G[3] = fm(i01, j01, i11 * j11);
}

// J^{-1} of the separable O-grid from its row and column tables.
template <typename R>
__device__ __forceinline__ void grad_map(const R* row, const R* col, R F00, R F01, R F10, R F11,
                                         R* G) {
    R c0, c1, c2, c3;
    ld4(col + CT_G, c0, c1, c2, c3);
    grad_map_j(row[RT_IDRC] * c0, -row[RT_IR] * c1, -row[RT_IDRC] * c2, row[RT_IR] * c3, F00, F01, F10,
               F11, G);
}

// Asynchronous 4- or 8-byte copy global -> shared (cp.async): no register
// round trip, so every copy of the tile is in flight at once.
__device__ __forceinline__ void cp_async4(void* dst, const void* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}

// Angular index modulo nt (the tile's halo may wrap more than once on very
// coarse rings).
__device__ __forceinline__ int wrap_nt(int j, int nt) {
    if ((unsigned)j >= (unsigned)nt) {
        j %= nt;
        if (j < 0) j += nt;
    }
    return j;
}

template <typename R>
__device__ __forceinline__ R pick(double d, float f);
template <>
__device__ __forceinline__ float pick<float>(double, float f) {
    return f;
}
template <>
__device__ __forceinline__ double pick<double>(double d, float) {
    return d;
}

}  // namespace lbfsi
