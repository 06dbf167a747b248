// Departure points (Eq. depPnt) on separable O-grids (closed form) and on
// meshes given by node coordinates (Newton), and the boundary targets built
// with them (Sec. III A), shared by the float step kernel (lbfsi_step.cu) and
// the float64 stream kernel (lbfsi_stream64.cu).
#pragma once

#include "lbfsi_stencil.cuh"

namespace lbfsi {

// Per-cell element coefficients of a general mesh (entries per cell).
constexpr int CELLC = 8;

// Departure point of node (i, j) displaced by d, in the reference coordinates
// of its element (Eq. depPnt).  On the subparametric O-grid the bilinear map
// of every element factorises, X(xi, eta) = R(xi) E(eta) with R linear in xi
// (radius) and E linear in eta (a point on the chord between two direction
// vectors), so the inverse is closed-form and relative to the node:
//   eta - eta_node = s = -(e_j x d) / (r_i (dE x e_j) + dE x d)
//   R - r_i = (d . E - r_i s dE . E) / |E|^2,   E = e_j + s dE
// with dE = dE/deta of the element.  The adjacent cell is picked by the signs
// of e_j x d (which side of the ray through the node) and of R - r_i (which
// side of the ring through the node); lines of constant eta are rays and of
// constant xi are rings, so this choice is exact.
//
// NodeGeo holds the table entries of one node; a solve picks the cells (da, db)
// in {-1, 0}^2 as flags, window() gives their element's first node.
template <typename R>
struct NodeGeo {
    R ex, ey, ri;
    R eta0, dEx0, dEy0, cq0, eta1, dEx1, dEy1, cq1;   // angular cells j-1 (0) and j (1)
    R xin0, idR0, xin1, idR1;                       // radial cells i-1 (0) and i (1)
    int wa0, wa1, wb0, wb1;                         // their elements' first row and column
};

template <typename R>
__device__ __forceinline__ void node_geo(int i, int j, int nr, const R* row, const R* col, NodeGeo<R>& G) {
    R u0, u1;
    ld4(col + CT_E, G.ex, G.ey, u0, u1);
    G.ri = row[RT_R];
    ld4(col + CT_C0, G.eta0, G.dEx0, G.dEy0, G.cq0);
    ld4(col + CT_C1, G.eta1, G.dEx1, G.dEy1, G.cq1);
    ld4(row + RT_XIN0, G.xin0, G.idR0, G.xin1, G.idR1);
    G.wa0 = min((max(i - 1, 0) >> 1) * 2, nr - 3);   // the wall row has no cell i-1
    G.wa1 = min((i >> 1) * 2, nr - 3);
    G.wb0 = ((j - 1) >> 1) * 2;
    G.wb1 = (j >> 1) * 2;
}

template <typename R>
__device__ __forceinline__ bool depart(const NodeGeo<R>& G, int i, R dx, R dy, int& wa, int& wb, R& xi,
                                       R& eta) {
    const R cr = fm(G.ex, dy, -(G.ey * dx));
    const bool db = !(cr < R(0));
    const R dEx = db ? G.dEx1 : G.dEx0, dEy = db ? G.dEy1 : G.dEy0;
    const R s = -cr * rcp_(fm(G.ri, db ? G.cq1 : G.cq0, fm(dEx, dy, -(dEy * dx))));
    const R Ex = fm(s, dEx, G.ex), Ey = fm(s, dEy, G.ey);
    const R dR = fm(-(G.ri * s), fm(dEx, Ex, dEy * Ey), fm(dx, Ex, dy * Ey)) * rcp_(fm(Ex, Ex, Ey * Ey));
    const bool da = !(dR < R(0)) || i == 0;   // on the wall: round-off of a tangential departure
    const R dxi = dR * (da ? G.idR1 : G.idR0);
    xi = (da ? G.xin1 : G.xin0) + dxi;
    eta = (db ? G.eta1 : G.eta0) + s;
    wa = da ? G.wa1 : G.wa0;
    wb = db ? G.wb1 : G.wb0;
    const R lim = R(1) + R(1e-4);
    return abs_(s) <= lim && abs_(dxi) <= lim;
}

// The same solve for a node the blend does not move (g = I, V_G = 0), where
// the displacement is the constant d = -dt c for the lattice velocity
// c = (CX, CY): the products with d reduce to sums of table entries.
template <int CX, int CY, typename R>
__device__ __forceinline__ bool depart_static(const NodeGeo<R>& G, R dt, int& wa, int& wb, R& xi, R& eta) {
    // e x c and dE x c for the two angular cells; d = -dt c
    const R exc = (CY ? G.ex * R(CY) : R(0)) - (CX ? G.ey * R(CX) : R(0));
    const R cr = -dt * exc;
    const bool db = !(cr < R(0));
    const R dEx = db ? G.dEx1 : G.dEx0, dEy = db ? G.dEy1 : G.dEy0;
    const R dexc = (CY ? dEx * R(CY) : R(0)) - (CX ? dEy * R(CX) : R(0));
    const R s = -cr * rcp_(fm(G.ri, db ? G.cq1 : G.cq0, -(dt * dexc)));
    const R Ex = fm(s, dEx, G.ex), Ey = fm(s, dEy, G.ey);
    const R cE = (CX ? R(CX) * Ex : R(0)) + (CY ? R(CY) * Ey : R(0));
    const R dR = fm(-dt, cE, -(G.ri * s) * fm(dEx, Ex, dEy * Ey)) * rcp_(fm(Ex, Ex, Ey * Ey));
    const bool da = !(dR < R(0));
    const R dxi = dR * (da ? G.idR1 : G.idR0);
    xi = (da ? G.xin1 : G.xin0) + dxi;
    eta = (db ? G.eta1 : G.eta0) + s;
    wa = da ? G.wa1 : G.wa0;
    wb = db ? G.wb1 : G.wb0;
    const R lim = R(1) + R(1e-4);
    return abs_(s) <= lim && abs_(dxi) <= lim;
}

// One Newton step of (b + d eta0) u + (c + d xi0) v + d u v = (dx, dy), with
// B = b + d eta0, C = c + d xi0 (written with fixed rounding: see fma_rn);
// ONCE false: and a second one with the same Jacobian.  Returns the size of the
// first step.
template <bool ONCE, typename R>
__device__ __forceinline__ R newton_step(const R* c, R Bx, R By, R Cx, R Cy, R dx, R dy, R& u, R& v) {
    const R a11 = fma_rn(c[4], v, Bx), a12 = fma_rn(c[4], u, Cx);
    const R a21 = fma_rn(c[5], v, By), a22 = fma_rn(c[5], u, Cy);
    const R idet = rcp_(fma_rn(a11, a22, -mul_rn(a12, a21)));
    R size = R(0);
#pragma unroll
    for (int it = 0; it < (ONCE ? 1 : 2); ++it) {
        const R uv = mul_rn(u, v);
        const R rx = fma_rn(c[4], uv, fma_rn(Cx, v, fma_rn(Bx, u, -dx)));
        const R ry = fma_rn(c[5], uv, fma_rn(Cy, v, fma_rn(By, u, -dy)));
        const R du = mul_rn(fma_rn(a22, rx, -mul_rn(a12, ry)), idet), dv = mul_rn(fma_rn(a11, ry, -mul_rn(a21, rx)), idet);
        u = add_rn(u, -du);
        v = add_rn(v, -dv);
        if (it == 0) size = max(abs_(du), abs_(dv));
    }
    return size;
}

// Departure point on a general mesh (Eq. depPnt): the node's Q2 element for
// the adjacent cell (a, b) the displacement d points into (its index-space
// direction J^{-1} d at the node), then Newton's method on the element's
// bilinear map X0 + b xi + c eta + d xi eta relative to the node's own local
// coordinates (xi0, eta0): (b + d eta0) u + (c + d xi0) v + d u v = d, which
// involves no absolute coordinates.  If the point falls outside that element
// the other adjacent cell is tried in the direction it left by; a point in no
// adjacent cell is a CFL violation.  jn: the node's (j00, j01, j10, j11) with
// d/dX = j00 d/di + j01 d/dj, d/dY = j10 d/di + j11 d/dj.
// gc: element coefficients of the mesh (global memory; a node that solves its
// departures reads four cells, which its neighbours share in L1).
template <typename R>
__device__ __forceinline__ bool depart_gen(const R* __restrict__ gc, const R* jn, int i, int j, int nr, int nt, bool cg,
                                           R dx, R dy, int& wo, int& wp, R& xi, R& eta, bool below = false, bool wrap_rows = false,
                                           unsigned* st = nullptr, int cbmax = -1) {
    // below: the node has cells below row 0 (the mirrored cells across a
    // C-grid's cut, or the wrapped rows of a periodic box); otherwise a row-0
    // node only has the cells of row 0.  wrap_rows: no last window to clamp to.
    // cbmax >= 0: only the cell columns 0..cbmax exist (a C-grid's outlet
    // columns, whose points on the column line may round to either side)
    // (written with fixed rounding: see fma_rn)
    const R di = fma_rn(jn[0], dx, mul_rn(jn[2], dy)), dj = fma_rn(jn[1], dx, mul_rn(jn[3], dy));
    const bool down = i > 0 || below;
    auto cb_ok = [&](int d) { return cbmax < 0 || (unsigned)(j + d) <= (unsigned)cbmax; };
    // no cells beyond the last row
    const bool up = wrap_rows || i < nr - 1;
    int da = ((!(di < R(0)) || !down) && up) ? 0 : -1;
    int db = !(dj < R(0)) ? 0 : -1;
    if (!cb_ok(db)) db = -1 - db;
    // an element is taken when the point lies in it up to round-off (tin);
    // failing that, the first candidate within the CFL margin (lim), as for
    // a wall departure that grazes the body
    const R tin = R(1) + (sizeof(R) == 4 ? R(1e-5) : R(1e-12));
    const R lim = R(1) + R(1e-4);
    bool have = false;
    int b_wa = 0, b_wb = 0;
    R b_xi = R(0), b_eta = R(0), b_du = R(2);
#pragma unroll 1
    for (int attempt = 0; attempt < 3; ++attempt) {
        const int ca = i + da, cb = j + db;
        const int wa = wrap_rows ? (ca >> 1) * 2 : min((ca >> 1) * 2, nr - 3), wb = (cb >> 1) * 2;
        const int cr = wrap_rows ? wrap_nt(ca, nr) : ca, cc = cg ? cb : wrap_nt(cb, nt);
        if (!in_bounds(cr >= (cg ? -1 : 0) && cr <= (wrap_rows ? nr - 1 : nr - 2) && cc >= 0 && cc < nt, st)) break;
        R c[8];
        {
            const R* g = gc + ((ptrdiff_t)cr * nt + cc) * CELLC;
            ld4(g, c[0], c[1], c[2], c[3]);
            ld4(g + 4, c[4], c[5], c[6], c[7]);
        }
        const R xi0 = R(i - wa - 1), et0 = R(j - wb - 1);
        const R Bx = fma_rn(c[4], et0, c[0]), By = fma_rn(c[5], et0, c[1]);
        const R Cx = fma_rn(c[4], xi0, c[2]), Cy = fma_rn(c[5], xi0, c[3]);
        R u = R(0), v = R(0);
        if constexpr (sizeof(R) == 4) {
#pragma unroll 1
            for (int it = 0; it < 3; ++it) newton_step<true>(c, Bx, By, Cx, Cy, dx, dy, u, v);
        } else {
            // float iterations for the start (their arithmetic is free beside
            // float64's) until one moves by less than 1e-5 of a cell: the error
            // is then float round-off, below 1e-5, goes to 1e-10 in one float64
            // step and below round-off in a second with the first's Jacobian.
            // Where they do not get there (cells skewed so far that float
            // round-off is more, values beyond float's range) float64 from zero
            const float cf[6] = {0.f, 0.f, 0.f, 0.f, (float)c[4], (float)c[5]};
            const float bx = (float)Bx, by = (float)By, ex = (float)Cx, ey = (float)Cy, fx = (float)dx, fy = (float)dy;
            float uf = 0.f, vf = 0.f;
            bool near = false;
#pragma unroll 1
            for (int it = 0; it < 12 && !near; ++it) near = newton_step<true>(cf, bx, by, ex, ey, fx, fy, uf, vf) < 1e-5f;
            if (near) {
                u = (R)uf;
                v = (R)vf;
            }
#pragma unroll 1
            for (int it = near ? 15 : 0; it < 16; ++it) newton_step<false>(c, Bx, By, Cx, Cy, dx, dy, u, v);
        }
        const R x = add_rn(xi0, u), e = add_rn(et0, v);
        const R du = max(abs_(u), abs_(v));   // displacement in cells (CFL)
        if (abs_(x) <= tin && abs_(e) <= tin) {
            wo = wa;
            wp = wb;
            xi = x;
            eta = e;
            return du <= lim;
        }
        if (!have && abs_(x) <= lim && abs_(e) <= lim) {
            have = true;
            b_wa = wa;
            b_wb = wb;
            b_xi = x;
            b_eta = e;
            b_du = du;
        }
        bool next = false;
        if (x > tin && da == -1 && up) { da = 0; next = true; }
        else if (x < -tin && da == 0 && down) { da = -1; next = true; }
        if (e > tin && db == -1 && cb_ok(0)) { db = 0; next = true; }
        else if (e < -tin && db == 0 && cb_ok(-1)) { db = -1; next = true; }
        if (!next) break;
    }
    wo = b_wa;
    wp = b_wb;
    xi = b_xi;
    eta = b_eta;
    return have && b_du <= lim;
}

// Far-field targets (Sec. III A 2), built like the wall's: a quantity the
// boundary does not prescribe takes a zero normal gradient through the point
// B = A - dt n_out one step inside along the outward unit direction, by Q2
// interpolation of M^k (the previous step's field).  An inlet (where the free
// stream enters) prescribes the free stream's u and T, its density is the
// value at B; an outlet prescribes nothing.  Interpolated as the node's own
// value plus the weighted differences from it: B lies a fraction of a cell
// from the node, and the weights' round-off (their sum is 1 to an ulp, the
// same at every step) then acts on the small differences, not on the values.
// mat(c, r, cc): moment c of node (r, cc).  Returns component c.
template <typename R, typename Mat>
__device__ __forceinline__ R far_target(Mat mat, int c, int i, int j, bool found, int wa, int wb, R xi, R eta) {
    const R own = mat(c, i, j);
    if (!found) return own;
    R Lx[3], Ly[3];
    lagrange3(xi, Lx);
    lagrange3(eta, Ly);
    R d = R(0);
#pragma unroll
    for (int aa = 0; aa < 3; ++aa)
#pragma unroll
        for (int bb = 0; bb < 3; ++bb) d = fm(Lx[aa] * Ly[bb], mat(c, wa + aa, wb + bb) - own, d);
    return own + d;
}

// Targets of a wall node (Sec. III A): rho, T at B = A + dt n0 by Q2
// interpolation of M^k (found, wa, wb, xi, eta: B's window), u = the wall's
// velocity, gradients of M^k at the node mapped by G.  mirror: the window lies
// below row 0 of a C-grid, whose row 0 is the other side's (column nt-1-c).
template <typename R, typename Mat>
__device__ __forceinline__ void wall_rho_T(Mat mat, int j, int nt, bool found, int wa, int wb, R xi, R eta, bool mirror, R& rho,
                                           R& T) {
    const R rhoA = mat(0, 0, j), TA = mat(3, 0, j);
    rho = rhoA;
    T = TA;
    if (!found) return;
    R Lx[3], Ly[3];
    lagrange3(xi, Lx);
    lagrange3(eta, Ly);
    R dr = R(0), dT = R(0);
#pragma unroll
    for (int aa = 0; aa < 3; ++aa)
#pragma unroll
        for (int bb = 0; bb < 3; ++bb) {
            const R w = Lx[aa] * Ly[bb];
            const int cc = (aa == 2 && mirror) ? nt - 1 - wb - bb : wb + bb;
            dr = fm(w, mat(0, wa + aa, cc) - rhoA, dr);
            dT = fm(w, mat(3, wa + aa, cc) - TA, dT);
        }
    rho += dr;
    T += dT;
}

// Gradient of moment c at wall node j.  rear: a C-grid's junction (its
// derivative along i is central across the cut, along j one-sided in
// direction jd).
template <typename R, typename Mat>
__device__ __forceinline__ void wall_gradient(Mat mat, int c, int j, bool rear, int jd, const R* G, R& gx, R& gy) {
    const R v0 = mat(c, 0, j), v1 = mat(c, 1, j);
    const R cxi = rear ? R(0.5) * (v1 - mat(c, -1, j)) : R(0.5) * fm(R(-3), v0, fm(R(4), v1, -mat(c, 2, j)));
    const R cet = jd > 0   ? R(0.5) * fm(R(-3), v0, fm(R(4), mat(c, 0, j + 1), -mat(c, 0, j + 2)))
                  : jd < 0 ? R(0.5) * fm(R(3), v0, fm(R(-4), mat(c, 0, j - 1), mat(c, 0, j - 2)))
                           : R(0.5) * (mat(c, 0, j + 1) - mat(c, 0, j - 1));
    gx = fm(G[0], cxi, G[1] * cet);
    gy = fm(G[2], cxi, G[3] * cet);
}

}  // namespace lbfsi
