// Stream launch of the float64 path on structured meshes: streaming of step
// k+1 from the post-collision populations of step k, which the field launch
// (lbfsi_fields.cu) has formed (k = 0: a copy of the initial state).  The two
// population buffers are the state's and the post-collision one, not a ping-pong
// pair: the field launch reads the first and writes the second, this one back.
//
// Float64 arithmetic is what bounds it: a warp instruction holds the SM's unit
// for some 16 cycles, so every operation counts, and so does the chain of one
// thread: a node's nine departure points and interpolations (about 70
// operations each) one after another are latency on small meshes, twice that
// at a wall.  Four warps therefore share each row of 32 nodes: warp w streams
// the directions {0, 1, 2}, {3, 4}, {5, 6} or {7, 8} of all 32 and adds its
// sums to the moments in shared memory.  Measured at 128 x 64 nodes: one
// kernel that staged, corrected, collided and streamed with a thread per node
// 118 us a step, this launch 25 us and the field launch 13 us.
// The windows are gathered from global memory (they hit L1 and L2): staging
// them would cost a barrier and the halo, and no float64 work is saved by it.
#include <algorithm>

#include "lbfsi_departure.cuh"

namespace lbfsi {

// a direction component as a double by selection (a conversion runs at the
// float64 rate)
__device__ __forceinline__ double sgn(int c) { return c > 0 ? 1.0 : c < 0 ? -1.0 : 0.0; }

constexpr int S64_WARPS = 4, S64_THREADS = 32 * S64_WARPS;

template <bool GEN, bool UNIFORM>
__global__ void __launch_bounds__(S64_THREADS, 4) k_stream64(const __grid_constant__ StepArgs a, int nbatch, int rows) {
    constexpr int TJ = TILE_J;
    wait_previous();
    __shared__ BodyMap<double> mapS[GEN ? MAX_BODIES : 1];
    __shared__ double s_sum[4][S64_WARPS][TJ];   // rho, rho u_x, rho u_y, 2 rho E of each warp's directions
    __shared__ double s_far[4][TJ];
    __shared__ double s_tgt[8][TJ];              // wall nodes: rho, T and the gradients of the targets
    __shared__ double s_grad[2][9][TJ];          // and their populations by Grad's approximation
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    int sb, ti0, j0;
    TileDev t{};
    if constexpr (UNIFORM) {
        // the solve varies fastest, then the column tile (neighbouring blocks
        // share the mesh's tables)
        const int b = (int)blockIdx.x, r = b / nbatch, ntj = a.umesh.ntj;
        sb = b - r * nbatch;
        j0 = (r % ntj) * TJ;
        ti0 = (r / ntj) * rows;
    } else {
        t = a.tiles[blockIdx.x];
        sb = 0;
        j0 = t.j0;
        ti0 = t.i0;
    }
    const SolveDev& S = [&]() -> const SolveDev& {
        if constexpr (UNIFORM) return a.usol;
        else return a.solves[t.solve];
    }();
    const MeshDev& G = [&]() -> const MeshDev& {
        if constexpr (UNIFORM) return a.umesh;
        else return a.meshes[t.mesh];
    }();
    const int nr = G.nr, nt = G.nt, j = j0 + l, nb = GEN ? S.nbody : 1;
    const int cg = GEN ? G.cgrid : 0, pb = GEN ? G.box : 0;
    const ptrdiff_t N = G.N;
    unsigned* ctr = S.counter + 4 * sb;
    const unsigned kstep = (UNIFORM && a.ustep >= 0) ? (unsigned)a.ustep : __ldcg(ctr + 1);
    const int cur = (int)(kstep & 1u);
    const bool record = a.record;
    {
        const StepMaps* rec = S.maps[cur] + (size_t)sb * nb;
        constexpr int W = (int)(sizeof(BodyMap<double>) / 4);
        for (int t = threadIdx.x; t < nb * W; t += S64_THREADS) {
            const int b = t / W, q = t - b * W;
            reinterpret_cast<unsigned*>(&mapS[b])[q] = __ldcg(reinterpret_cast<const unsigned*>(&rec[b].Sd) + q);
        }
    }
    __syncthreads();
    const double2* __restrict__ pin = reinterpret_cast<const double2*>(S.ppost) + (size_t)sb * 9 * N;
    const double* __restrict__ M = reinterpret_cast<const double*>(S.M[cur]) + (size_t)sb * 4 * N;
    double2* __restrict__ pout = reinterpret_cast<double2*>(S.p[cur ^ 1]) + (size_t)sb * 9 * N;
    double* __restrict__ Mout = reinterpret_cast<double*>(S.M[cur ^ 1]) + (size_t)sb * 4 * N;
    const double* __restrict__ gcell = reinterpret_cast<const double*>(G.cellc);
    const double dt = S.dt;
    const int rlo = cg ? -CGRID_GHOST_ROWS : 0;
    auto rw = [&](int i) { return pb ? wrap_nt(i, nr) : i; };
    auto cw = [&](int c) { return cg ? c : wrap_nt(c, nt); };
    // moment c at node (r, cc) of M^k (a C-grid stores mirrored rows below row 0)
    auto Mat = [&](int c, int r, int cc) -> double { return M[(ptrdiff_t)c * N + (ptrdiff_t)rw(r) * nt + cw(cc)]; };

    for (int i = ti0; i < ti0 + rows && i < nr; ++i) {
        const bool live = j < nt;
        // C-grid: the second copies of the row-0 cut nodes (and of the rear
        // point) are written by their first copies; rows 1-4 also write
        // their moments into their mirrored slots below row 0
        const int ct = (cg && i == 0 && live) ? __ldg(G.coltype + j) : 0;
        const bool mine = live && !(ct & CT_DUP);
        const int n = i * nt + j, n2 = i == 0 ? nt - 1 - j : -i * nt + (nt - 1 - j);
        const bool dup2_ = (ct & (CT_CUT | CT_JUNC)) != 0, mir_ = cg && i >= 1 && i <= CGRID_GHOST_ROWS;
        const bool n2ok = !(dup2_ || mir_) || !live || in_bounds(n2 >= rlo * nt && n2 < nr * nt, a.status);
        const bool dup2 = dup2_ && n2ok, mir = mir_ && n2ok;
        const bool farj = cg && i < nr - 1 && (j == 0 || j == nt - 1);
        const bool far = mine && ((!pb && i == nr - 1) || farj);
        double jn[4] = {0.0, 0.0, 0.0, 0.0};
        NodeGeo<double> geo;
        double F00 = 1.0, F01 = 0.0, F10 = 0.0, F11 = 1.0, vx = 0.0, vy = 0.0;
        bool moved = false;
        if (mine) {
            if constexpr (GEN) {
                ld4(reinterpret_cast<const double*>(G.jinv) + 4 * (ptrdiff_t)n, jn[0], jn[1], jn[2], jn[3]);
                if (!far) {
                    const double2 x = __ldg(reinterpret_cast<const double2*>(G.nodex) + n);
                    moved = kinematics_sum(mapS, nb, x.x, x.y, F00, F01, F10, F11, vx, vy);
                }
            } else {
                const double* row = reinterpret_cast<const double*>(G.rowtab) + (size_t)i * ROWTAB;
                const double* col = reinterpret_cast<const double*>(G.coltab) + (size_t)j * COLTAB;
                node_geo(i, j, nr, row, col, geo);
                if (!far && mapS[0].active)
                    moved = kinematics(mapS[0], G.xm + geo.ri * geo.ex, G.ym + geo.ri * geo.ey, F00, F01, F10, F11, vx, vy);
            }
        }
        double i00 = 1.0, i01 = 0.0, i10 = 0.0, i11 = 1.0;
        if (moved) {
            const double idF = rcp_(fm(F00, F11, -(F01 * F10)));
            i00 = F11 * idF;
            i01 = -F01 * idF;
            i10 = -F10 * idF;
            i11 = F00 * idF;
        }
        auto departure = [&](int inode, double dx, double dy, int& wa, int& wb, double& xi, double& eta, int cbmax) -> bool {
            bool ok;
            if constexpr (GEN)
                ok = depart_gen<double>(gcell, jn, inode, j, nr, nt, cg, dx, dy, wa, wb, xi, eta, dup2 || pb, pb, a.status, cbmax);
            else
                ok = depart(geo, inode, dx, dy, wa, wb, xi, eta);
            return ok && in_bounds(pb || (wa >= (cg ? -2 : 0) && wa + 2 < nr && (!cg || (wb >= 0 && wb + 2 < nt))), a.status);
        };
        if (record) {
            // departure cache of the static nodes: one warp
            // per row solves and writes all nine
            if (w == 0 && mine && !far) {
                if (!moved && i > 0) {
                    double2* gxe = reinterpret_cast<double2*>(a.usol.dep_xe);
                    unsigned long long code = 0ull;
                    bool ok = true;
#pragma unroll 1
                    for (int q = 0; q < 9; ++q) {
                        int wa = i, wb = j;
                        double2 xe;
                        unsigned nib = 16u;   // a lost departure
                        if (departure(i, -dt * sgn(cxq(q)), -dt * sgn(cyq(q)), wa, wb, xe.x, xe.y, -1)) {
                            const int dr = wa - i, dc = wb - j;
                            if (dr < -3 || dr > 0 || dc < -3 || dc > 0) ok = false;
                            nib = (unsigned)(((dr + 3) << 2) | (dc + 3));
                        }
                        code |= (unsigned long long)nib << (5 * q);
                        gxe[(size_t)q * N + n] = xe;
                    }
                    a.usol.dep_code[n] = ok ? code : ~0ull;
                }
            }
            continue;
        }
        const int q0 = w == 0 ? 0 : 2 * w + 1, q1 = 2 * w + 3;   // this warp's directions
        const bool wall = mine && !far && !pb && i == 0 && (!cg || (ct & CT_WALL));
        if (i == 0 && !pb) {
            // wall nodes (Sec. III A), in parts (the four warps share the SM's
            // float64 lanes: nothing is computed twice): targets and gradients,
            // one warp each; then Grad's f by the first and g by the second
            if (wall) {
                const int jd = (ct & CT_JUNC) ? ((ct & CT_JFWD) ? 1 : -1) : 0;
                if (w == 0) {
                    int wa = 0, wb = 0;
                    double xi = 0.0, eta = 0.0;
                    const bool ok = departure(0, dt * G.n0[2 * j], dt * G.n0[2 * j + 1], wa, wb, xi, eta, -1);
                    if (!ok) atomicOr(a.status, ST_BPOINT);
                    wall_rho_T<double>(Mat, j, nt, ok, wa, wb, xi, eta, GEN && cg && wa == -2, s_tgt[0][l], s_tgt[1][l]);
                } else {
                    double Gm[4], gx, gy;
                    if constexpr (GEN) grad_map_j(jn[0], jn[1], jn[2], jn[3], F00, F01, F10, F11, Gm);
                    else grad_map(reinterpret_cast<const double*>(G.rowtab), reinterpret_cast<const double*>(G.coltab) + (size_t)j * COLTAB,
                                  F00, F01, F10, F11, Gm);
                    wall_gradient<double>(Mat, w, j, (ct & CT_JUNC) != 0, jd, Gm, gx, gy);
                    s_tgt[2 * w][l] = gx;
                    s_tgt[2 * w + 1][l] = gy;
                }
            }
            __syncthreads();
            if (wall && w < 2) {
                WallTarget<double> t;
                t.rho = s_tgt[0][l];
                t.T = s_tgt[1][l];
                t.ux = vx;
                t.uy = vy;
#pragma unroll
                for (int c = 0; c < 6; ++c) t.gr[c] = s_tgt[2 + c][l];
                double v[9];
                if (w == 0) grad_f(t, S.mu, dt, S.iCv, v);
                else grad_g(t, S.mu, dt, S.Cv, S.iCv, S.iPr, v);
#pragma unroll
                for (int q = 0; q < 9; ++q) s_grad[w][q][l] = v[q];
            }
            __syncthreads();
        }
        if (far) {
            // far field: component w of the targets
            const double* fd = farj ? G.fardirj + 4 * i + (j == 0 ? 0 : 2) : G.fardir + 2 * j;
            const bool inlet = S.uinf_x * fd[0] + S.uinf_y * fd[1] < 0.0;
            int wa = 0, wb = 0;
            double xi = 0.0, eta = 0.0;
            const bool ok = departure(i, -dt * fd[0], -dt * fd[1], wa, wb, xi, eta, cg ? nt - 2 : -1);
            if (!ok) atomicOr(a.status, ST_BPOINT);
            double v;
            if (inlet && w > 0) v = w == 1 ? S.uinf_x : w == 2 ? S.uinf_y : S.T_inf;
            else v = far_target<double>(Mat, w, i, j, ok, wa, wb, xi, eta);
            s_far[w][l] = v;
            Mout[(ptrdiff_t)w * N + n] = v;
            if (dup2 || mir) Mout[(ptrdiff_t)w * N + n2] = v;
        } else if (mine) {
            double f[3] = {0.0, 0.0, 0.0}, g[3] = {0.0, 0.0, 0.0};
            unsigned missing = 0u;
            if (wall) {
                // missing populations: departure point inside the body (Sec. III A)
                const double n0x = G.n0[2 * j], n0y = G.n0[2 * j + 1];
                for (int q = q0; q < q1; ++q) {
                    const double cx = sgn(cxq(q)), cy = sgn(cyq(q));
                    const double hx = fm(i00, cx, fm(i01, cy, -vx)), hy = fm(i10, cx, fm(i11, cy, -vy));
                    if (fm(hx, n0x, hy * n0y) > 1e-12) missing |= 1u << q;
                }
            }
            unsigned long long dcode = ~0ull;
            if (UNIFORM && a.usol.dep_code != nullptr && !moved && i > 0) dcode = __ldg(a.usol.dep_code + n);
            bool lost = false;
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                const int q = q0 + t;
                if (q >= q1) continue;
                if (missing & (1u << q)) {
                    f[t] = s_grad[0][q][l];
                    g[t] = s_grad[1][q][l];
                    continue;
                }
                int wa, wb;
                double xi, eta;
                bool ok;
                if (dcode != ~0ull) {
                    // a node the blend does not move takes its cached departures
                    const unsigned nib = (unsigned)(dcode >> (5 * q)) & 31u;
                    const double2 xe = __ldg(reinterpret_cast<const double2*>(a.usol.dep_xe) + (size_t)q * N + n);
                    ok = !(nib & 16u);
                    wa = i + (int)(nib >> 2) - 3;
                    wb = j + (int)(nib & 3u) - 3;
                    xi = xe.x;
                    eta = xe.y;
                } else {
                    const double cx = sgn(cxq(q)), cy = sgn(cyq(q));
                    const double hx = fm(i00, cx, fm(i01, cy, -vx)), hy = fm(i10, cx, fm(i11, cy, -vy));
                    ok = departure(i, -dt * hx, -dt * hy, wa, wb, xi, eta, -1);
                }
                const double2* __restrict__ p = pin + (ptrdiff_t)q * N;
                if (!ok) {
                    lost = true;
                    f[t] = p[n].x;
                    g[t] = p[n].y;
                    continue;
                }
                // Q2 interpolation over the window; below row 0 of a C-grid
                // its mirror on the other side of the cut, its row 0 included
                double Lx[3], Ly[3];
                lagrange3(xi, Lx);
                lagrange3(eta, Ly);
                int c[3];
#pragma unroll
                for (int b = 0; b < 3; ++b) c[b] = cw(wb + b);
                double ax = 0.0, ay = 0.0;
#pragma unroll
                for (int aa = 0; aa < 3; ++aa) {
                    const int r = wa + aa;
                    const bool m = GEN && cg && wa < 0;
                    const double2* pr = p + (m ? (ptrdiff_t)-r * nt + nt - 1 : (ptrdiff_t)rw(r) * nt);
                    const double2 v0 = m ? pr[-c[0]] : pr[c[0]], v1 = m ? pr[-c[1]] : pr[c[1]], v2 = m ? pr[-c[2]] : pr[c[2]];
                    ax = fm(Lx[aa], fm(Ly[2], v2.x, fm(Ly[1], v1.x, Ly[0] * v0.x)), ax);
                    ay = fm(Lx[aa], fm(Ly[2], v2.y, fm(Ly[1], v1.y, Ly[0] * v0.y)), ay);
                }
                f[t] = ax;
                g[t] = ay;
            }
            if (lost) atomicOr(a.status, ST_DEPARTURE);
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                if (q0 + t >= q1) continue;
                const double2 v = make_double2(f[t], g[t]);
                pout[(ptrdiff_t)(q0 + t) * N + n] = v;
                if (dup2) pout[(ptrdiff_t)(q0 + t) * N + n2] = v;
            }
            // this warp's share of the moments (f[2] is zero but in the first)
            double jx, jy;
            if (w == 0) {          // directions 0, (1, 0), (0, 1)
                jx = f[1];
                jy = f[2];
            } else if (w == 1) {   // (-1, 0), (0, -1)
                jx = -f[0];
                jy = -f[1];
            } else if (w == 2) {   // (1, 1), (-1, 1)
                jx = f[0] - f[1];
                jy = f[0] + f[1];
            } else {               // (-1, -1), (1, -1)
                jx = f[1] - f[0];
                jy = -(f[0] + f[1]);
            }
            s_sum[0][w][l] = f[0] + f[1] + f[2];
            s_sum[1][w][l] = jx;
            s_sum[2][w][l] = jy;
            s_sum[3][w][l] = g[0] + g[1] + g[2];
        }
        __syncthreads();
        if (far) {
            // equilibria at the targets: f by the first warp, g by the others
            double v[9];
            if (w == 0) f_equilibrium(s_far[0][l], s_far[1][l], s_far[2][l], s_far[3][l], v);
            else g_equilibrium(s_far[0][l], s_far[1][l], s_far[2][l], s_far[3][l], S.Cv, v);
            double* po = reinterpret_cast<double*>(pout) + (w ? 1 : 0);
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                if (w > 0 && q / 3 != w - 1) continue;
                po[2 * ((ptrdiff_t)q * N + n)] = v[q];
                if (dup2) po[2 * ((ptrdiff_t)q * N + n2)] = v[q];
            }
        } else if (mine && w == 0) {
            double s[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) s[c] = (s_sum[c][0][l] + s_sum[c][1][l]) + (s_sum[c][2][l] + s_sum[c][3][l]);
            const double ir = rcp_(s[0]), ux = s[1] * ir, uy = s[2] * ir;
            const double T = fm(-0.5, fm(ux, ux, uy * uy), 0.5 * s[3] * ir) * S.iCv;
            if (!(s[0] > 0.0) || !(T > 0.0) || !isfinite(ux) || !isfinite(uy)) atomicOr(a.status, ST_NONPHYS);
            const double m[4] = {s[0], ux, uy, T};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                Mout[(ptrdiff_t)c * N + n] = m[c];
                if (dup2 || mir) Mout[(ptrdiff_t)c * N + n2] = m[c];
            }
        }
        if (i + 1 < ti0 + rows) __syncthreads();   // (the sums are the next row's)
    }
    // a launch that took its step number from the device counter advances it
    // when the last block of the solve has read it (the barrier above: every
    // thread of this one has)
    if (!record && !(UNIFORM && a.ustep >= 0) && threadIdx.x == 0) {
        if (atomicAdd(ctr, 1u) == (unsigned)S.ntiles - 1u) {
            ctr[0] = 0u;
            ctr[1] = kstep + 1u;
        }
    }
}

cudaError_t launch_stream64(const StepArgs& a, bool uniform, bool general, int rows, int nbatch, cudaStream_t s) {
    const int nti = (a.umesh.nr + rows - 1) / rows;
    const unsigned grid = uniform ? (unsigned)nbatch * a.umesh.ntj * nti : (unsigned)a.ntiles;
    auto go = [&](auto kernel) { return launch_behind(kernel, grid, S64_THREADS, 0, s, grid <= OVERLAP_BLOCKS_FP64, a, nbatch, rows); };
    if (uniform) return general ? go(k_stream64<true, true>) : go(k_stream64<false, true>);
    return general ? go(k_stream64<true, false>) : go(k_stream64<false, false>);
}

}  // namespace lbfsi
