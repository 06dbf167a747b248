// The step of a solve's bodies behind its loads and the next step's record,
// one warp per solve: the structured meshes' loads (lbfsi_fields.cu) and the
// element lists' (lbfsi_elements.cu).  Bound by the chain of float64
// operations of a single warp, so a body's step is the linear map it is
// (BodyProp) on four lanes, not a serial Runge-Kutta on one.
#pragma once

#include <cstddef>

#include "lbfsi_device.cuh"
#include "lbfsi_internal.h"

namespace lbfsi {
namespace {

constexpr unsigned FULL = 0xffffffffu;

// Sum over the warp's lanes (the same tree for every caller).
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(FULL, v, o);
    return v;
}

// Lane r of a body's group of four: state entry r (h, alpha, hdot, adot) before
// the step (zero where the new one is prescribed), the part of its increment that
// does not depend on the loads, and the weights of F_y and M.
struct BodyLane {
    BodyStateDev Sn;
    BodyMap<double> ms;
    double p4, p5, y, base;
};

// The step to step kk from the record prev of the step before; whole warp.
__device__ __forceinline__ BodyLane body_lane(const BodyDev& bd, const BodyProp& prop, const StepMaps& prev, double dt,
                                              unsigned kk, int l) {
    const int r = l & 3;
    const BodyStateDev Sn = prev.S_next;
    const double t1 = (double)kk * dt;
    const bool forced = bd.dof == 2 && t1 <= bd.t_forced;
    double pr[6], sv[4] = {Sn.h, Sn.alpha, Sn.hdot, Sn.adot};
    {
        const double* p = forced ? prop.forced[r >> 1] : prop.free[r];
#pragma unroll
        for (int c = 0; c < 6; ++c) pr[c] = p[c];
    }
    double y = 0.0, base = r == 0 ? Sn.h : r == 1 ? Sn.alpha : r == 2 ? Sn.hdot : Sn.adot;
    if (forced) {
        // forced pitching (Sec. IV D): alpha = amp sin(w t) prescribed, its
        // acceleration at the step's start, middle and end
        const double ww = bd.w_a, amp = bd.pitch_amp;
        const double ang = ww * (r == 0 ? t1 - dt : r == 1 ? ((double)kk - 0.5) * dt : t1);
        const double sn = amp * (r == 3 ? cos(ang) : sin(ang));
        const int g4 = l & ~3;
        const unsigned grp = 0xfu << g4;   // (the body's lanes take this branch together)
        const double a0 = __shfl_sync(grp, sn, g4), ah = __shfl_sync(grp, sn, g4 + 1), a1 = __shfl_sync(grp, sn, g4 + 2);
        const double c1 = __shfl_sync(grp, sn, g4 + 3);
        if (r == 1) y = a1;
        else if (r == 3) y = ww * c1;
        else y = fm(-ww * ww, fm(pr[3], a0, fm(pr[4], ah, pr[5] * a1)), fm(pr[0], sv[0], pr[1] * sv[2]));
        if (r & 1) base = 0.0;
        pr[4] = (r & 1) ? 0.0 : pr[2];
        pr[5] = 0.0;
    } else {
        y = fm(pr[0], sv[0], pr[1] * sv[1]) + fm(pr[2], sv[2], pr[3] * sv[3]);
    }
    return BodyLane{Sn, prev.Sd, pr[4], pr[5], y, base};
}

// The new states from the loads F (x, y, moment of the lane's body) and the
// records maps[0 .. nb) of the new step; rec: seven values per body, or null.
__device__ __forceinline__ void body_records(const BodyLane& bl, const double* F, double idt, int nb, int l,
                                             StepMaps& s_rec, StepMaps* maps, double* rec) {
    const int g4 = min(l >> 2, nb - 1) * 4, r = l & 3;
    const double y = bl.base + fm(bl.p4, F[1], fm(bl.p5, F[2], bl.y));
    const BodyStateDev& Sn = bl.Sn;
    const BodyMap<double>& ms = bl.ms;
    const double h = __shfl_sync(FULL, y, g4), al = __shfl_sync(FULL, y, g4 + 1);
    const double hd = __shfl_sync(FULL, y, g4 + 2), ad = __shfl_sync(FULL, y, g4 + 3);
    // sin(alpha) and cos(alpha) - 1 = -2 sin^2(alpha / 2) (body_rot)
    double sn = (r & 1) ? al : 0.5 * al;
    if (al != 0.0) sn = sin(sn);
    const double hs = __shfl_sync(FULL, sn, g4), sa = __shfl_sync(FULL, sn, g4 + 1), cm = -2.0 * hs * hs;
    for (int b = 0; b < nb; ++b) {
        // the record (build_maps): the collision map is the streamed map at
        // rest, the stream map the new state's with the rates from the last
        if (l == 4 * b) {
            s_rec.S_cur = s_rec.S_vgprev = Sn;
            s_rec.S_next = BodyStateDev{h, al, hd, ad};
            for (int c = 0; c < 3; ++c) s_rec.loads[c] = F[c];
            BodyMap<double> m = ms;
            m.va00 = m.va01 = m.va10 = m.va11 = m.vtx = m.vty = 0.0;
            s_rec.Kd = m;
            m.va00 = m.va11 = (cm - ms.a00) * idt;
            m.va10 = (sa - ms.a10) * idt;
            m.va01 = -m.va10;
            m.vty = (h - Sn.h) * idt;
            m.a00 = m.a11 = cm;
            m.a01 = -sa;
            m.a10 = sa;
            m.ty = h;
            s_rec.Sd = m;
        }
        __syncwarp();
        // their float copies, an entry per lane
        constexpr int ND = (int)((sizeof(BodyMap<double>) - offsetof(BodyMap<double>, xc)) / 8);
        for (int t = l; t < 2 * ND; t += 32) {
            const BodyMap<double>& d = t < ND ? s_rec.Sd : s_rec.Kd;
            BodyMap<float>& f = t < ND ? s_rec.Sf : s_rec.Kf;
            const int c = t < ND ? t : t - ND;
            (&f.xc)[c] = (float)(&d.xc)[c];
            if (c == 0) f.active = d.active;
        }
        __syncwarp();
        unsigned* out = reinterpret_cast<unsigned*>(maps + b);
        for (int t = l; t < (int)(sizeof(StepMaps) / 4); t += 32) out[t] = reinterpret_cast<const unsigned*>(&s_rec)[t];
        if (rec && l < 7) rec[b * 7 + l] = l < 3 ? s_rec.loads[l] : (&s_rec.S_next.h)[l - 3];
        __syncwarp();
    }
}

}  // namespace
}  // namespace lbfsi
