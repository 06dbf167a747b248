// Field launch of the structured-mesh step, run between two step launches
// (lbfsi_step.cu): its blocks do two independent jobs on the current state k
// (moments M^k and post-propagation populations).
//
//   loads    one warp per 32 wall columns: the wall stress of the streamed
//            populations in float64 (Sec. III), the columns' Simpson shares of
//            force and moment; the last block of a solve sums them in a fixed
//            order, advances its bodies by RK4 (Sec. III B) and writes the
//            blended maps of the next stream (Sec. II D)
//   fields   one block per tile: Y_a = d_a[(mu/p) d_a dQ_a] (Sec. II C; FE
//            gradients, Eq. ddx+fem, mapped by g^{-1} of the blended map of
//            step k), once per node; in float64 the node's collision (Eq.
//            f_boltz) follows at once, into the post-collision buffer
//
// Why a launch of its own: Y is a second derivative, so a step that forms it
// inside its streaming tiles does so on the tile's +-2 halo from D on +-3 and
// dQ on +-4 (1.4 to 1.9 evaluations per node), and holds M^k, dQ, D and the
// gradient maps of that halo in shared memory, which left two blocks per SM.
// Here dQ and D reach one or two nodes beyond the tile, and the step stages
// two floats per node instead.  The loads' float64 chain (2 lanes per SM on
// this part) and the RK4 tail run beside the fields instead of at the end of
// the step launch.  Measured: float fields 22 us at 512 x 256 x 16 (50 MB read
// and written: 7.4 us at 6.8 TB/s; bound by issue and the latency of a strip's
// loads), 24 us on an ellipse 512 x 256 x 8 by coordinates; the loads' chain alone
// 8 to 12 us, which is what bounds the launch on small meshes; float64 with the
// collision 13 us at 128 x 64.
#include <algorithm>

#include "lbfsi_record.cuh"
#include "lbfsi_stencil.cuh"

namespace lbfsi {

// (double)x of a normal float in integer instructions: a conversion runs at
// the float64 rate, and a wall node has 18.
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) {
    const unsigned u = __float_as_uint(x), e = (u >> 23) & 255u;
    if (e == 0u || e == 255u) return (double)x;
    return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}

constexpr int LOAD_WARPS = 4;   // wall tiles (32 columns) per loads block
// float64 rate: 2 lanes per SM and cycle, and a chain of dependent operations
// waits for each: sums as trees, no division (one Newton reciprocal each for
// the velocity and omega), the RK4 step as its linear map
template <typename R, bool GEN>
__device__ __forceinline__ void wall_loads(const FieldArgs& a, const SolveDev& S, const MeshDev& G, int sb, int blk,
                                           unsigned kk, unsigned* ctr) {
    using R2 = typename Vec2<R>::T;
    __shared__ StepMaps s_rec;
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, NW = (int)blockDim.x >> 5;
    const int cur = (int)(kk & 1u), nt = G.nt, ntj = G.ntj, nb = GEN ? S.nbody : 1;
    const int nblk = (ntj + LOAD_WARPS - 1) / LOAD_WARPS;
    const size_t N = (size_t)G.N;
    const StepMaps* prev = S.maps[cur ^ 1] + (size_t)sb * nb;   // the streamed step's record
    double* part = S.part + (size_t)sb * nb * ntj * 3;
    for (int q0 = w; q0 < LOAD_WARPS; q0 += NW) {
        const int tj = blk * LOAD_WARPS + q0, j = tj * TILE_J + l;
        double fc[3] = {0.0, 0.0, 0.0};
        int bid = 0;
        bool wall = j < nt;
        if constexpr (GEN) {
            if (G.box) wall = false;
            if (wall && G.cgrid) {
                const int ct = __ldg(G.coltype + j);
                wall = (ct & CT_WALL) && !(ct & CT_DUP);
                bid = (ct >> CT_BODY_SHIFT) & (MAX_BODIES - 1);
            }
        }
        if (wall) {
            // wall stress sigma = -p I - (1 - omega/2) P^(1), P^(1) = sum f c c -
            // rho (u u + T I) (Sec. III), this node's Simpson share of its edges:
            // float64 from the populations on
            const R2* p = reinterpret_cast<const R2*>(S.p[cur]) + (size_t)sb * 9 * N + j;
            double f[9], g[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const R2 v = p[(size_t)q * N];
                f[q] = widen(v.x);
                g[q] = widen(v.y);
            }
            const double E2 = ((g[0] + g[1]) + (g[2] + g[3])) + ((g[4] + g[5]) + (g[6] + g[7])) + g[8];   // 2 rho E
            const double sx = f[1] + f[3], sy = f[2] + f[4], da = f[5] + f[7], db = f[6] + f[8], sd = da + db;
            const double rho = (f[0] + sx) + (sy + sd), ir = rcp_(rho);
            const double dx = f[5] - f[7], dy = f[6] - f[8];
            const double ux = ((f[1] - f[3]) + (dx - dy)) * ir, uy = ((f[2] - f[4]) + (dx + dy)) * ir;
            const double T = fm(-0.5, fm(ux, ux, uy * uy), 0.5 * E2 * ir) * S.iCv;
            const double p0 = rho * T;
            // 1 - omega/2 with omega = 1 / (1/2 + mu / (p dt))
            const double am = S.mu * rcp_(fm(0.5 * S.dt, p0, S.mu));
            const double pxx = fm(-rho, fm(ux, ux, T), sx + sd), pyy = fm(-rho, fm(uy, uy, T), sy + sd);
            const double pxy = fm(-rho, ux * uy, da - db);
            const double sxx = fm(-am, pxx, -p0), sxy = -am * pxy, syy = fm(-am, pyy, -p0);
            // the wall node moves with its own body: rotation and moment
            // reference of that body
            const BodyMap<double>& mw = prev[bid].Sd;
            const double R00 = 1.0 + mw.a00, R01 = mw.a01, R10 = mw.a10, R11 = 1.0 + mw.a11;
            const double Xd = G.xw[2 * j] - mw.xp, Yd = G.xw[2 * j + 1] - mw.yp;
            const double rx = fm(R00, Xd, R01 * Yd), ry = fm(R10, Xd, R11 * Yd);
            const double ex = G.wall_share[2 * j], ey = G.wall_share[2 * j + 1];
            const double nx = fm(R00, ex, R01 * ey), ny = fm(R10, ex, R11 * ey);
            fc[0] = fm(sxx, nx, sxy * ny);
            fc[1] = fm(sxy, nx, syy * ny);
            fc[2] = fm(rx, fc[1], -(ry * fc[0]));
        }
        for (int b = 0; b < nb; ++b)
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const double v = warp_sum(bid == b ? fc[c] : 0.0);
                if (l == 0 && tj < ntj) __stcg(part + ((size_t)b * ntj + tj) * 3 + c, v);
            }
    }
    __syncthreads();
    if (w != 0) return;
    // the bodies' steps, four lanes per body: lane r of a group state entry
    // r.  What they need besides the loads is read before the count below, so
    // that the solve's last block does not wait for it in turn
    const int bo = min(l >> 2, nb - 1);
    const size_t sbo = (size_t)sb * nb + bo;
    const BodyLane bl = body_lane(S.body[sbo], S.prop[sbo], prev[bo], S.dt, kk, l);
    // the acquire-release count publishes this block's partials and makes
    // every other block's visible to the solve's last
    if (nblk > 1) {
        unsigned done = 0u;
        if (l == 0) asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(done) : "l"(ctr + 2) : "memory");
        if (__shfl_sync(FULL, done, 0) != (unsigned)nblk - 1u) return;
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
    }
    double F[3] = {0.0, 0.0, 0.0};   // the load of this lane's body
    for (int b = 0; b < nb; ++b) {
        // lane t holds the partials of tiles t, t + 32, ...; then the warp's tree
        double v[3] = {0.0, 0.0, 0.0};
        for (int t = l; t < ntj; t += 32)
#pragma unroll
            for (int c = 0; c < 3; ++c) v[c] += __ldcg(part + ((size_t)b * ntj + t) * 3 + c);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const double t = warp_sum(v[c]);
            if (b == bo) F[c] = t;
        }
    }
    body_records(bl, F, S.idt, nb, l, s_rec, S.maps[cur] + (size_t)sb * nb, a.rec ? a.rec + (size_t)sb * nb * 7 : nullptr);
    if (l == 0) {
        ctr[1] = kk;
        ctr[2] = 0u;
    }
}

// The blended maps of step k into shared memory: the record's collision maps,
// or, behind the step that streamed it (whose record of step k the loads
// blocks of this launch are still writing), the stream maps of the record
// before, built from the same states.
template <typename R>
__device__ __forceinline__ void stage_maps(const FieldArgs& a, const SolveDev& S, int sb, int nb, int cur,
                                           BodyMap<R>* smap) {
    constexpr int W = (int)(sizeof(BodyMap<R>) / 4);
    const StepMaps* rec = S.maps[a.loads ? cur ^ 1 : cur] + (size_t)sb * nb;
    for (int t = threadIdx.x; t < nb * W; t += blockDim.x) {
        const int b = t / W, q = t - b * W;
        const void* src;
        if constexpr (sizeof(R) == 4) src = a.loads ? &rec[b].Sf : &rec[b].Kf;
        else src = a.loads ? &rec[b].Sd : &rec[b].Kd;
        reinterpret_cast<unsigned*>(&smap[b])[q] = __ldcg(reinterpret_cast<const unsigned*>(src) + q);
    }
}

// ---- float fields: a warp covers a strip of 32 columns x ROWS + 4 rows, lane
// l column j0 - H + l, all rows in registers: every load of the strip is in
// flight at once (marching row by row with one row loaded ahead waited for
// memory at each: 34 us on 2 M nodes against 22), and the neighbours along j
// come by shuffles, so there is no barrier behind the loads.  dQ and D of a
// node are formed 1.14 times over along j and 1.7 and 1.3 times along i.  The
// gradient maps go through shared memory: strips in a blended region map
// theirs by F^{-T} in a loop of its own (unrolled into every row it filled the
// instruction cache), the others skip it.
constexpr int MARCH_WARPS = 4;
template <bool GEN>
struct March {
    static constexpr int ROWS = GEN ? 4 : 6, K = ROWS + 4;   // rows a strip writes and reads
    static constexpr int H = GEN ? 3 : 2;   // (a C-grid's one-sided stencils reach two nodes)
    static constexpr int W = 32 - 2 * H;    // columns a strip writes
};

// sG: this warp's gradient maps [K][32]; sX: general meshes, its node
// coordinates [K][32]; sR: separable meshes, its rows' tables [K].
template <bool GEN>
__device__ __forceinline__ void fields_march(const SolveDev& S, const MeshDev& G, int sb, int unit, int cur,
                                             const BodyMap<float>* smap, const float* rout2, float4* sG, float2* sX,
                                             float4* sR, unsigned* status) {
    using T = March<GEN>;
    constexpr int H = T::H, W = T::W, K = T::K;
    const int l = threadIdx.x & 31, nr = G.nr, nt = G.nt, N = G.N;
    const int nsx = (nt + W - 1) / W, sy = unit / nsx, sx = unit - sy * nsx;
    const int i0 = sy * T::ROWS, i1 = min(i0 + T::ROWS, nr);   // (past the mesh: nothing is written)
    const int cg = GEN ? G.cgrid : 0, pb = GEN ? G.box : 0, nb = GEN ? S.nbody : 1;
    const int j = sx * W - H + l;
    const int jc = cg ? min(max(j, 0), nt - 1) : wrap_nt(j, nt);
    const bool mine = l >= H && l < 32 - H && j < nt && !(cg && (j == 0 || j == nt - 1));   // writes this column
    const float* __restrict__ M = reinterpret_cast<const float*>(S.M[cur]) + (size_t)sb * 4 * N;
    const int rlo = cg ? -CGRID_GHOST_ROWS : 0;
    // node of row i0 - 2 + k in this column (outside the mesh: the nearest, unused)
    auto node = [&](int k) -> int {
        const int i = min(i0, nr - 1) - 2 + k;
        return (pb ? wrap_nt(i, nr) : min(max(i, rlo), nr - 1)) * nt + jc;
    };
    if constexpr (GEN) {
#pragma unroll
        for (int k = 1; k < K - 1; ++k) {
            const int n = node(k);
            cp_async16(sG + 32 * k + l, reinterpret_cast<const float4*>(G.jinv) + n);
            cp_async8(sX + 32 * k + l, reinterpret_cast<const float2*>(G.nodex) + n);
        }
    } else {
        // the rows' tables, one row per lane (read after the barrier below)
        const int i = min(max(min(i0, nr - 1) - 2 + l, 0), nr - 1);
        if (l < K) cp_async16(sR + l, reinterpret_cast<const float*>(G.rowtab) + (size_t)i * ROWTAB + RT_R);
    }
    float m[K][4];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const int n = node(k);
#pragma unroll
        for (int c = 0; c < 4; ++c) m[k][c] = M[c * N + n];
    }
    // class of this column on row 0 of a C-grid
    const int ct = cg && j >= 0 && j < nt ? __ldg(G.coltype + jc) : 0;
    const bool across = (ct & (CT_CUT | CT_JUNC)) != 0;
    const int jdir0 = (ct & CT_JUNC) ? ((ct & CT_JFWD) ? 1 : -1) : 0;
    const bool low = !pb && i0 == 0;   // the strip starts on row 0
    const bool onesided = low && !(GEN && across);
    // column tables of the separable mesh
    float c0 = 0.f, c1 = 0.f, c2 = 0.f, c3 = 0.f, ex = 0.f, ey = 0.f;
    if constexpr (!GEN) {
        const float* col = reinterpret_cast<const float*>(G.coltab) + jc * COLTAB;
        float u0, u1;
        ld4(col + CT_G, c0, c1, c2, c3);
        ld4(col + CT_E, ex, ey, u0, u1);
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();   // (the maps, staged by the block ahead of these loads)

    // gradient maps: inverse metric, mapped by F^{-T} where the blend moves the
    // node.  Whether a node may lie in a blended region by a bound with a margin
    // above its rounding (kinematics() decides)
    auto place = [&](int k) -> float2 {
        if constexpr (GEN) return sX[32 * k + l];
        const float r = sR[k].x;
        return make_float2(fm(r, ex, G.xm_f), fm(r, ey, G.ym_f));
    };
    bool any = false;
    for (int b = 0; b < nb; ++b) {
        const float xc = smap[b].xc, yc = smap[b].yc, r2 = rout2[b];
#pragma unroll
        for (int k = 1; k < K - 1; ++k) {
            const float2 x = place(k);
            const float dx = x.x - xc, dy = x.y - yc;
            any = any || fm(dx, dx, dy * dy) <= r2;
        }
    }
    any = __any_sync(FULL, any);
    if (any) {
#pragma unroll 1
        for (int k = 1; k < K - 1; ++k) {
            float4 g;
            if constexpr (GEN) {
                g = sG[32 * k + l];
            } else {
                const float4 r = sR[k];   // r, 1/r', 1/r
                g = make_float4(r.y * c0, -r.z * c1, -r.y * c2, r.z * c3);
            }
            const float2 x = place(k);
            float F00, F01, F10, F11, vx, vy, t[4];
            if (kinematics_sum(smap, nb, x.x, x.y, F00, F01, F10, F11, vx, vy)) {
                grad_map_j(g.x, g.y, g.z, g.w, F00, F01, F10, F11, t);
                g = make_float4(t[0], t[1], t[2], t[3]);
            }
            sG[32 * k + l] = g;
        }
    }
    auto gmap = [&](int k) -> float4 {
        if (GEN || any) return sG[32 * k + l];
        const float4 r = sR[k];
        return make_float4(r.y * c0, -r.z * c1, -r.y * c2, r.z * c3);
    };
    // derivative along j (one-sided on a C-grid's outlet columns, which a strip
    // may hold in its halo alone, and at a row-0 junction)
    const bool edge = cg && (sx == 0 || sx * W - H + 31 >= nt - 1);
    auto dj = [&](float v, bool row0) -> float {
        const float up = __shfl_down_sync(FULL, v, 1), dn = __shfl_up_sync(FULL, v, 1);
        float d = 0.5f * (up - dn);
        if (GEN && (edge || (cg && row0))) {
            const float up2 = __shfl_down_sync(FULL, v, 2), dn2 = __shfl_up_sync(FULL, v, 2);
            const int jd = j == 0 ? 1 : j == nt - 1 ? -1 : row0 ? jdir0 : 0;
            if (jd > 0) d = 0.5f * fm(-3.0f, v, fm(4.0f, up, -up2));
            if (jd < 0) d = 0.5f * fm(3.0f, v, fm(-4.0f, dn, dn2));
        }
        return d;
    };
    // one-sided row stencils (first and last row) as central ones with the row
    // beyond extrapolated quadratically: 3 v0 - 3 v1 + v2
    auto beyond = [](float2 v0, float2 v1, float2 v2) {
        return make_float2(fm(3.0f, v0.x - v1.x, v2.x), fm(3.0f, v0.y - v1.y, v2.y));
    };
    float2 q[K];
    float mup[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const float rho = m[k][0], ux = m[k][1], uy = m[k][2], Tn = m[k][3];
        const float t = fm(-3.0f, Tn, 1.0f);
        q[k] = make_float2(rho * ux * fm(-ux, ux, t), rho * uy * fm(-uy, uy, t));
        mup[k] = S.mu_f * rcp_(rho * Tn);
    }
    const float2 ghq = beyond(q[2], q[3], q[4]);   // (low: row -1)
    if (!pb && i0 - 2 + K > nr) {                  // the row beyond the last
#pragma unroll
        for (int k = 3; k < K; ++k)
            if (i0 - 2 + k == nr) q[k] = beyond(q[k - 1], q[k - 2], q[k - 3]);
    }
    float* Y = reinterpret_cast<float*>(S.Y) + (size_t)sb * 2 * N;
    float2 d[K];
    float4 g[K];
    auto make_y = [&](int k, float2 db) {   // Y of row i0 - 2 + k
        const int i = i0 - 2 + k;
        const bool row0 = !pb && i == 0;
        const float xe = dj(d[k].x, row0), ye = dj(d[k].y, row0);
        const float Yx = fm(g[k].x, 0.5f * (d[k + 1].x - db.x), g[k].y * xe);
        const float Yy = fm(g[k].z, 0.5f * (d[k + 1].y - db.y), g[k].w * ye);
        const int n = i * nt + j;
        if (i < i1 && (pb || i < nr - 1) && mine && !(row0 && (ct & CT_DUP)) && in_bounds(n >= 0 && n < nr * nt, status)) {
            Y[n] = Yx;
            Y[N + n] = Yy;
            if (row0 && across) {   // a C-grid's second copies take the first copies' values
                Y[nt - 1 - j] = Yx;
                Y[N + nt - 1 - j] = Yy;
            }
        }
    };
#pragma unroll
    for (int k = 1; k < K - 1; ++k) {
        g[k] = gmap(k);
        const bool row0 = !pb && i0 - 2 + k == 0;
        const float2 qb = (k == 2 && onesided) ? ghq : q[k - 1];
        const float xe = dj(q[k].x, row0), ye = dj(q[k].y, row0);
        d[k] = make_float2(mup[k] * fm(g[k].x, 0.5f * (q[k + 1].x - qb.x), g[k].y * xe),
                           mup[k] * fm(g[k].z, 0.5f * (q[k + 1].y - qb.y), g[k].w * ye));
        // (Y of row 0 needs D of rows 0, 1, 2)
        if (k == 4) make_y(2, onesided ? beyond(d[2], d[3], d[4]) : d[1]);
        if (k > 4) make_y(k - 2, d[k - 3]);
    }
    make_y(K - 3, d[K - 4]);
}

// ---- float64 fields and collision: one block per tile of TI x 32 nodes, dQ
// and D of its halo in shared memory; then two warps per tile row, one for
// the row's f and one for its g (each forms the moments both relax by).  A
// float64 warp instruction holds the SM's unit for some 16 cycles, so what
// counts is the operations and the longest warp's chain of them.
// Two rows: a 128 x 64 mesh is 128 blocks, about one per SM.
constexpr int FIELD_ROWS_FP64 = 2;
template <bool GEN, int TI>
__device__ __forceinline__ void fields_tile(const FieldArgs& a, const SolveDev& S, const MeshDev& G, int sb, int blk,
                                            int cur, const BodyMap<double>* smap) {
    using R = double;
    using R2 = double2;
    constexpr int NT = 64 * TI, TJ = TILE_J;
    // halo of D and dQ along j: a C-grid's one-sided stencils reach two nodes
    constexpr int HD = GEN ? 2 : 1, HQ = HD + 1;
    constexpr int DH = TI + 2, DW = TJ + 2 * HD, DS = DH * DW;
    constexpr int QH = TI + 4, QW = TJ + 2 * HQ, QS = QH * QW;
    __shared__ R sQ[2][QS], sP[QS], sD[2][DS], sG[4][DS];

    const int tid = threadIdx.x, nr = G.nr, nt = G.nt;
    const int i0 = (blk / G.ntj) * TI, j0 = (blk - (blk / G.ntj) * G.ntj) * TJ;
    const int cg = GEN ? G.cgrid : 0, pb = GEN ? G.box : 0;
    const int* ctab = G.coltype;
    auto ctype = [&](int j) -> int { return cg ? __ldg(ctab + j) : 0; };
    auto jdir_of = [&](int c) -> int { return (c & CT_JUNC) ? ((c & CT_JFWD) ? 1 : -1) : 0; };
    const int rlo = cg ? -CGRID_GHOST_ROWS : 0;
    auto rowok = [&](int i) { return pb || (i >= rlo && i < nr); };
    auto rw = [&](int i) { return pb ? wrap_nt(i, nr) : i; };
    const ptrdiff_t N = G.N;
    const R* __restrict__ M = reinterpret_cast<const R*>(S.M[cur]) + (size_t)sb * 4 * N;
    const int nb = GEN ? S.nbody : 1;
    const R mu = pick<R>(S.mu, S.mu_f), dt = pick<R>(S.dt, S.dt_f), Cv = pick<R>(S.Cv, S.Cv_f);
    for (int t = tid; t < QS; t += NT) {
        const int li = t / QW, lj = t - li * QW;
        const int i = i0 - 2 + li, j = j0 - HQ + lj;
        if (!rowok(i) || (cg && (unsigned)j >= (unsigned)nt)) continue;
        const ptrdiff_t n = (ptrdiff_t)rw(i) * nt + (cg ? j : wrap_nt(j, nt));
        if (!in_bounds(n >= (ptrdiff_t)rlo * nt && n < (ptrdiff_t)nr * nt, a.status)) continue;
        const R rho = M[n], ux = M[N + n], uy = M[2 * N + n], T = M[3 * N + n];
        const R s = fm(R(-3), T, R(1));
        sQ[0][t] = rho * ux * fm(-ux, ux, s);
        sQ[1][t] = rho * uy * fm(-uy, uy, s);
        sP[t] = mu * rcp_(rho * T);
    }
    __syncthreads();
    const R* __restrict__ rowtab = reinterpret_cast<const R*>(G.rowtab);
    const R* __restrict__ coltab = reinterpret_cast<const R*>(G.coltab);
    const R* __restrict__ gx = reinterpret_cast<const R*>(G.nodex);
    const R* __restrict__ gj = reinterpret_cast<const R*>(G.jinv);
    const R xm = pick<R>(G.xm, G.xm_f), ym = pick<R>(G.ym, G.ym_f);
    for (int t = tid; t < DS; t += NT) {
        const int li = t / DW, lj = t - li * DW;
        const int i = i0 - 1 + li, j = j0 - HD + lj;
        if (!rowok(i) || (cg && (unsigned)j >= (unsigned)nt)) continue;
        R F00, F01, F10, F11, vx, vy, m[4], q[4];
        bool moved;
        const int s = (li + 1) * QW + lj + 1;
        if constexpr (GEN) {
            const ptrdiff_t n = (ptrdiff_t)rw(i) * nt + (cg ? j : wrap_nt(j, nt));
            const R2 x = __ldg(reinterpret_cast<const R2*>(gx) + n);
            ld4(gj + 4 * n, m[0], m[1], m[2], m[3]);
            moved = kinematics_sum(smap, nb, x.x, x.y, F00, F01, F10, F11, vx, vy);
            const int ct = (cg && i == 0) ? ctype(j) : 0;
            const bool across = (ct & (CT_CUT | CT_JUNC)) != 0;
            q[0] = d_row_c(sQ[0] + s, QW, i, nr, across, pb);
            q[1] = d_col_c(sQ[0] + s, j, nt, cg, jdir_of(ct));
            q[2] = d_row_c(sQ[1] + s, QW, i, nr, across, pb);
            q[3] = d_col_c(sQ[1] + s, j, nt, cg, jdir_of(ct));
        } else {
            const R* row = rowtab + (size_t)i * ROWTAB;
            const R* col = coltab + (size_t)wrap_nt(j, nt) * COLTAB;
            R c[4], r[4], ex, ey, u0, u1;
            ld4(col + CT_G, c[0], c[1], c[2], c[3]);
            ld4(row + RT_R, r[0], r[1], r[2], r[3]);   // r, 1/r', 1/r
            m[0] = r[1] * c[0]; m[1] = -r[2] * c[1]; m[2] = -r[1] * c[2]; m[3] = r[2] * c[3];
            moved = smap[0].active;
            if (moved) {
                ld4(col + CT_E, ex, ey, u0, u1);
                moved = kinematics(smap[0], xm + r[0] * ex, ym + r[0] * ey, F00, F01, F10, F11, vx, vy);
            }
            q[0] = d_row(sQ[0] + s, QW, i, nr);
            q[1] = d_col(sQ[0] + s);
            q[2] = d_row(sQ[1] + s, QW, i, nr);
            q[3] = d_col(sQ[1] + s);
        }
        if (moved) {
            R g[4];
            grad_map_j(m[0], m[1], m[2], m[3], F00, F01, F10, F11, g);
#pragma unroll
            for (int c = 0; c < 4; ++c) m[c] = g[c];
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) sG[c][t] = m[c];
        sD[0][t] = sP[s] * fm(m[0], q[0], m[1] * q[1]);
        sD[1][t] = sP[s] * fm(m[2], q[2], m[3] * q[3]);
    }
    __syncthreads();
    {
        const bool gh = tid >= 32 * TI;   // the g half
        const int t = gh ? tid - 32 * TI : tid;
        const int li = t / TJ, lj = t - li * TJ;
        const int i = i0 + li, j = j0 + lj;
        if (i >= nr || j >= nt) return;
        const ptrdiff_t n = (ptrdiff_t)i * nt + j;
        // a C-grid's second copies take the first copies' values
        const int ct = (cg && i == 0) ? ctype(j) : 0;
        if (ct & CT_DUP) return;
        const bool two = (ct & (CT_CUT | CT_JUNC)) != 0;
        const ptrdiff_t n2 = nt - 1 - j;
        const bool far = (!pb && i == nr - 1) || (cg && (j == 0 || j == nt - 1));
        R Yx = R(0), Yy = R(0);
        if (!far && !gh) {
            const int s = (li + 1) * DW + lj + HD;
            R d[4];
            if constexpr (GEN) {
                const bool across = two;
                d[0] = d_row_c(sD[0] + s, DW, i, nr, across, pb);
                d[1] = d_col_c(sD[0] + s, j, nt, cg, jdir_of(ct));
                d[2] = d_row_c(sD[1] + s, DW, i, nr, across, pb);
                d[3] = d_col_c(sD[1] + s, j, nt, cg, jdir_of(ct));
            } else {
                d[0] = d_row(sD[0] + s, DW, i, nr);
                d[1] = d_col(sD[0] + s);
                d[2] = d_row(sD[1] + s, DW, i, nr);
                d[3] = d_col(sD[1] + s);
            }
            Yx = fm(sG[0][s], d[0], sG[1][s] * d[1]);
            Yy = fm(sG[2][s], d[2], sG[3][s] * d[3]);
        }
        R* po = reinterpret_cast<R*>(S.ppost) + (size_t)sb * 18 * N + (gh ? 1 : 0);   // this half's slots
        R v[9];
        if (far) {
            // the far field's post-collision state: the equilibria of its targets
            if (gh) g_equilibrium(M[n], M[N + n], M[2 * N + n], M[3 * N + n], Cv, v);
            else f_equilibrium(M[n], M[N + n], M[2 * N + n], M[3 * N + n], v);
        } else {
            const R2* p = reinterpret_cast<const R2*>(S.p[cur]) + (size_t)sb * 9 * N;
            R2 pq[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) pq[q] = p[q * N + n];
            Collision<R> c;
            c.moments(pq, mu, S.muP, dt, S.iCv);
            if (gh) {
                c.g_target(v);
#pragma unroll
                for (int q = 0; q < 9; ++q) v[q] = fm(c.w1, v[q] - pq[q].y, pq[q].y);
            } else {
                c.f_target(v);
#pragma unroll
                for (int q = 0; q < 9; ++q) v[q] = fm(c.w, v[q] - pq[q].x, pq[q].x);
                // dt phi on the axis velocities
                const R hyx = 0.5 * dt * Yx, hyy = 0.5 * dt * Yy;
                v[1] -= hyx;
                v[3] += hyx;
                v[2] -= hyy;
                v[4] += hyy;
            }
        }
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            po[2 * (q * N + n)] = v[q];
            if (two) po[2 * (q * N + n2)] = v[q];
        }
    }
}

// ---- float64, step 0: the initial state, which is streamed as it is, into the
// post-collision buffer (the same tiles; a thread's five or four directions).
template <int TI>
__device__ __forceinline__ void copy_state(const FieldArgs& a, const SolveDev& S, const MeshDev& G, int sb, int blk) {
    const int half = (int)threadIdx.x / (32 * TI), t = (int)threadIdx.x - half * 32 * TI;
    const int i = (blk / G.ntj) * TI + t / TILE_J, j = (blk % G.ntj) * TILE_J + t % TILE_J;
    if (i >= G.nr || j >= G.nt) return;
    const ptrdiff_t N = G.N, n = (ptrdiff_t)i * G.nt + j;
    const double2* p = reinterpret_cast<const double2*>(S.p[0]) + (size_t)sb * 9 * N;
    double2* po = reinterpret_cast<double2*>(S.ppost) + (size_t)sb * 9 * N;
    for (int q = half ? 5 : 0; q < (half ? 9 : 5); ++q) po[q * N + n] = p[q * N + n];
}

// Uniform launches (a mesh handle: the records are launch arguments) and table
// launches (the batch runtime).  R float: TI unused (marching strips).  R double: tiles of TI rows.
template <typename R, bool GEN, int TI, bool UNIFORM>
__global__ void __launch_bounds__(sizeof(R) == 4 ? 32 * MARCH_WARPS : 64 * TI, sizeof(R) == 4 ? 5 : 4)
    k_fields(const __grid_constant__ FieldArgs a) {
    wait_previous();
    __shared__ BodyMap<R> smap[GEN ? MAX_BODIES : 1];
    int sb = 0, blk = (int)blockIdx.x;
    bool loads;
    FieldTile t{};
    if constexpr (UNIFORM) {
        const int nl = (a.umesh.ntj + LOAD_WARPS - 1) / LOAD_WARPS, n = a.loads ? a.nbatch * nl : 0;
        loads = blk < n;
        if (!loads) blk -= n;
        const int per = loads ? nl : a.nfield;
        sb = blk / per;
        blk -= sb * per;
    } else {
        t = a.tiles[blockIdx.x];
        loads = !t.fields;
        blk = t.block;
    }
    const SolveDev& S = [&]() -> const SolveDev& {
        if constexpr (UNIFORM) return a.usol;
        else return a.solves[t.solve];
    }();
    const MeshDev& G = [&]() -> const MeshDev& {
        if constexpr (UNIFORM) return a.umesh;
        else return a.meshes[t.mesh];
    }();
    unsigned* ctr = S.counter + 4 * sb;
    const unsigned kk = (UNIFORM && a.ustep >= 0) ? (unsigned)a.ustep : __ldcg(ctr + 1);
    if (loads) {
        wall_loads<R, GEN>(a, S, G, sb, blk, kk, ctr);
        return;
    }
    if (kk == 0u) {   // the first launch streams the initial state, nothing collides
        if constexpr (sizeof(R) == 8) copy_state<TI>(a, S, G, sb, blk);
        return;
    }
    const int cur = (int)(kk & 1u);
    stage_maps(a, S, sb, GEN ? S.nbody : 1, cur, smap);
    if constexpr (sizeof(R) == 4) {
        constexpr int K = March<GEN>::K;
        __shared__ float4 sG[MARCH_WARPS][K][32], sR[MARCH_WARPS][K];
        __shared__ float2 sX[GEN ? MARCH_WARPS : 1][K][32];
        __shared__ float rout2[GEN ? MAX_BODIES : 1];
        // the blended regions' radii (with a margin), negative for a body at rest
        const StepMaps* rec = S.maps[a.loads ? cur ^ 1 : cur] + (size_t)sb * (GEN ? S.nbody : 1);
        if ((int)threadIdx.x < (GEN ? S.nbody : 1)) {
            const BodyMap<float>& bm = rec[threadIdx.x].Sf;
            const float r = (bm.r_in + rcp_(bm.inv_w)) * 1.0001f;
            rout2[threadIdx.x] = bm.active ? r * r : -1.0f;
        }
        const int w = (int)threadIdx.x >> 5;
        fields_march<GEN>(S, G, sb, blk * MARCH_WARPS + w, cur, smap, rout2, &sG[w][0][0], &sX[GEN ? w : 0][0][0], &sR[w][0],
                          a.status);
    } else {
        fields_tile<GEN, TI>(a, S, G, sb, blk, cur, smap);
    }
}

// Post-collision populations of the current state from Y (float path; the
// accessor's read of them, no part of a step).
__global__ void k_post(const SolveDev S, const MeshDev G, int cur, int nbatch) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const ptrdiff_t N = G.N;
    const int nodes = G.nr * G.nt;
    if (t >= (size_t)nodes * nbatch) return;
    const size_t sb = t / nodes;
    const int n = (int)(t - sb * nodes), i = n / G.nt, j = n - i * G.nt;
    const float2* p = reinterpret_cast<const float2*>(S.p[cur]) + sb * 9 * N;
    const float* M = reinterpret_cast<const float*>(S.M[cur]) + sb * 4 * N;
    const float* Y = reinterpret_cast<const float*>(S.Y) + sb * 2 * N;
    float2* po = reinterpret_cast<float2*>(S.ppost) + sb * 9 * N;
    float2 pq[9];
    if ((!G.box && i == G.nr - 1) || (G.cgrid && (j == 0 || j == G.nt - 1))) {
        float f[9], g[9];
        f_equilibrium(M[n], M[N + n], M[2 * N + n], M[3 * N + n], f);
        g_equilibrium(M[n], M[N + n], M[2 * N + n], M[3 * N + n], S.Cv_f, g);
        for (int q = 0; q < 9; ++q) pq[q] = pair(f[q], g[q]);
    } else {
        for (int q = 0; q < 9; ++q) pq[q] = p[q * N + n];
        collide_pairs(pq, Y[n], Y[N + n], S.mu_f, S.muP_f, S.dt_f, S.iCv_f);
    }
    for (int q = 0; q < 9; ++q) po[q * N + n] = pq[q];
}

template <typename R, bool GEN, bool UNIFORM>
static cudaError_t launch_t(const FieldArgs& a, unsigned blocks, cudaStream_t s) {
    constexpr int TI = sizeof(R) == 4 ? 0 : FIELD_ROWS_FP64;
    return launch_behind(k_fields<R, GEN, TI, UNIFORM>, blocks, sizeof(R) == 4 ? 32 * MARCH_WARPS : 64 * FIELD_ROWS_FP64, 0,
                         s, sizeof(R) == 4 || blocks <= OVERLAP_BLOCKS_FP64, a);
}

template <bool UNIFORM>
static cudaError_t launch_any(const FieldArgs& a, int precision, bool general, unsigned blocks, cudaStream_t s) {
    if (precision == 0) return general ? launch_t<double, true, UNIFORM>(a, blocks, s) : launch_t<double, false, UNIFORM>(a, blocks, s);
    return general ? launch_t<float, true, UNIFORM>(a, blocks, s) : launch_t<float, false, UNIFORM>(a, blocks, s);
}

int field_blocks(int precision, bool general, int nr, int nt) {
    if (precision == 0) return ((nr + FIELD_ROWS_FP64 - 1) / FIELD_ROWS_FP64) * tiles_j(nt);
    const int w = general ? March<true>::W : March<false>::W, rows_ = general ? March<true>::ROWS : March<false>::ROWS;
    const int units = ((nr + rows_ - 1) / rows_) * ((nt + w - 1) / w);
    return (units + MARCH_WARPS - 1) / MARCH_WARPS;
}

int load_blocks(int ntj) { return (ntj + LOAD_WARPS - 1) / LOAD_WARPS; }

cudaError_t launch_fields(FieldArgs a, int precision, bool general, cudaStream_t s) {
    unsigned blocks = (unsigned)a.ntiles;
    if (a.uniform) {
        a.nfield = field_blocks(precision, general, a.umesh.nr, a.umesh.nt);
        blocks = (unsigned)a.nbatch * (unsigned)((a.loads ? load_blocks(a.umesh.ntj) : 0) + (a.fields ? a.nfield : 0));
    }
    if (!blocks) return cudaSuccess;
    return a.uniform ? launch_any<true>(a, precision, general, blocks, s) : launch_any<false>(a, precision, general, blocks, s);
}

cudaError_t launch_post(const SolveDev& S, const MeshDev& G, int cur, int nbatch, cudaStream_t s) {
    const size_t total = (size_t)G.nr * G.nt * nbatch;
    k_post<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(S, G, cur, nbatch);
    return cudaGetLastError();
}

}  // namespace lbfsi
