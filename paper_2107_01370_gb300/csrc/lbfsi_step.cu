// Step kernel of the two-population compressible semi-Lagrangian LBM on a
// blended structured mesh (Sec. II-III of the paper), for sm_103a.
//
// One launch L_k advances the solver by one step in the order
//     collide(step k)  ->  stream(step k+1)
// which is the paper's stream-then-collide cycle shifted by half a step: the
// state kept in HBM between launches is the post-propagation (pre-collision)
// population set of step k, plus its moment field M^k.  Collision first lets
// the correction term phi (a second derivative of moments of the *current*
// step, Sec. II C) use the moment field written by the previous launch.  That
// derivative and the loads are the field launch's (lbfsi_fields.cu), which
// runs between two step launches.  This is the float path; the float64 path
// collides in the field launch and streams in lbfsi_stream64.cu.
//
//   prologue   the solve's step number; the blended maps of the stream
//              (Sec. II D)
//   phase 1    stage the populations of the tile +-2 nodes and Y of
//              the same nodes in shared memory as asynchronous copies
//   phase 2    collision of the +-2 region in place (Eq. f_boltz)
//   phase 3    stream every tile node: c_hat = g^{-T} c - V_G, departure point,
//              bilinear inverse (Eq. depPnt) and Q2 interpolation (Eq.
//              SemiLagrProp) from the collided tile; wall nodes rebuild their
//              missing populations by Grad's approximation (Sec. III A); far
//              field nodes take equilibria at their targets; write the
//              populations and M^{k+1}
//
// Populations are kept in HBM as (f_q, g_q) pairs, [q][node] (both share the
// departure point and the interpolation weights), so staging moves 16-byte
// chunks and the stream writes one 64-bit pair per direction.  The redundant
// work is the collision of the 2-node halo; the HBM traffic per node is the
// 18 populations read and written once plus the 4-value moment field and Y.
//
// Bound by instruction issue: 41.7 warp instructions per node on the VIV ring
// (59.9 when this kernel also formed dQ, D and Y in its halo and reduced the
// loads).  Measured at 512 x 256 x 16 solves, half the nodes moving: that one
// kernel 155 us a step; this launch 113 us and the field launch 22.  At 256 x 128
// x 1: 29.6 us against 11.3 and 9.5 (the loads' chain no longer ends the step).
#include <algorithm>
#include <cstdio>
#include <type_traits>

#include "lbfsi_departure.cuh"

namespace lbfsi {

template <int TI, int TJ>
struct Tile {
    static constexpr int HP = 2;
    static constexpr int PH = TI + 2 * HP, PW = TJ + 2 * HP, PS = PH * PW;
    // staged populations: rows of PWS nodes from j0 - 4 (16-byte aligned
    // chunks), so the +-2 region starts at column 2 of a row
    static constexpr int PWS = TJ + 8, PSS = PH * PWS;
};


// Shared-memory strides of the geometry tables: a row is read by whole warps
// (broadcast); consecutive columns are 20 words apart, so the 16-byte loads of
// eight threads (one shared-memory wavefront) cover distinct banks.
constexpr int RS = ROWTAB;
constexpr int CS = COLTAB + 4;

// Dynamic shared memory of a block: the staged populations and Y, then the
// geometry tables of the tile's nodes (separable meshes) or the mirrored row 0
// of a C-grid.
template <int TI, int TJ, bool GEN>
constexpr size_t step_smem_bytes() {
    using T = Tile<TI, TJ>;
    return sizeof(float) * (size_t)(20 * T::PSS + (GEN ? 20 * T::PWS : TI * RS + TJ * CS));
}

__device__ __forceinline__ void cp_async_wait_all() {
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}
// A record of 4-byte words copied by the 32 lanes of one warp.
__device__ __forceinline__ void cp_async_words(void* dst, const void* src, int words, int lane) {
    for (int q = lane; q < words; q += 32)
        cp_async4(static_cast<unsigned*>(dst) + q, static_cast<const unsigned*>(src) + q);
}

// Tensor copies (TMA): one thread moves a whole 4-D box global -> shared, the
// bytes arriving on a shared-memory transaction barrier (mbarrier) that every
// reader waits on.  Each barrier of a CTA is used for one phase (parity 0).
__device__ __forceinline__ void mbar_init(unsigned long long* bar) {
    const unsigned b = (unsigned)__cvta_generic_to_shared(bar);
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(b) : "memory");
}
// make the initialised barriers visible to the tensor-copy (async) proxy
__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;\nfence.proxy.async.shared::cta;\n" ::: "memory");
}
// the one arrival of the phase, announcing the bytes the copies will deliver
__device__ __forceinline__ void mbar_expect_tx(unsigned long long* bar, unsigned bytes) {
    const unsigned b = (unsigned)__cvta_generic_to_shared(bar);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(b), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait0(unsigned long long* bar) {
    const unsigned b = (unsigned)__cvta_generic_to_shared(bar);
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(b)
        : "memory");
    return done != 0u;
}
// Wait for phase 0 of a barrier with an iteration limit; a wait that runs out
// flags the launch (the host then reports the step as failed) and returns.
constexpr int TMA_WAIT_LIMIT = 1 << 22;
__device__ __forceinline__ void mbar_wait0(unsigned long long* bar, unsigned* status) {
    for (int it = 0; it < TMA_WAIT_LIMIT; ++it)
        if (mbar_try_wait0(bar)) return;
    atomicOr(status, ST_TMA);
}
// Box of a 4-D tensor map at element coordinates (x innermost) into shared
// memory; x times the element size must be a multiple of 16 bytes.
__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, unsigned long long* bar, int x,
                                            int y, int z, int w) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    const unsigned b = (unsigned)__cvta_generic_to_shared(bar);
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
        "%5}], [%6];\n" ::"r"(d),
        "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(z), "r"(w), "r"(b)
        : "memory");
}

// Q2 interpolation of one (f, g) pair over a 3x3 window (rows rowstride
// apart, columns adjacent): separable sums t_a = sum_b L_b(eta) v(a, b), then
// sum_a L_a(xi) t_a (Eq. SemiLagrProp), with packed two-wide FMAs (f and g
// share the weights).
// Reads the first two pairs of a window row with one 16-byte
// load: window origins are even columns of a staged row that starts on a
// 16-byte boundary.
__device__ __forceinline__ float2 gather9(const float2* p, int rowstride, const float* Lx,
                                                  const float* Ly) {
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int aa = 0; aa < 3; ++aa) {
        const float2* pr = p + aa * rowstride;
        const float4 p01 = *reinterpret_cast<const float4*>(pr);
        float2 t = __fmul2_rn(make_float2(Ly[0], Ly[0]), make_float2(p01.x, p01.y));
        t = __ffma2_rn(make_float2(Ly[1], Ly[1]), make_float2(p01.z, p01.w), t);
        t = __ffma2_rn(make_float2(Ly[2], Ly[2]), pr[2], t);
        acc = __ffma2_rn(make_float2(Lx[aa], Lx[aa]), t, acc);
    }
    return acc;
}
// The same over a window whose last row is elsewhere (p2): a window below row
// 0 of a C-grid is the mirror of one on the other side of the cut, its row 0
// included, which next to a junction differs from the tile's row 0.
__device__ __forceinline__ float2 gather9_rows(const float2* p, int rowstride, const float2* p2, const float* Lx,
                                               const float* Ly) {
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int aa = 0; aa < 3; ++aa) {
        const float2* pr = aa == 2 ? p2 : p + aa * rowstride;
        float2 t = pmul(pair(Ly[0], Ly[0]), pr[0]);
        t = pfma(pair(Ly[1], Ly[1]), pr[1], t);
        t = pfma(pair(Ly[2], Ly[2]), pr[2], t);
        acc = pfma(pair(Lx[aa], Lx[aa]), t, acc);
    }
    return acc;
}

template <int TI, int TJ, int NT, int MINB, bool UNIFORM, bool GEN>
__global__ void __launch_bounds__(NT, MINB) k_step(const __grid_constant__ StepArgs a) {
    using T = Tile<TI, TJ>;
    using R = float;
    using R2 = float2;
    // tile nodes streamed per thread
    constexpr int NPT = (TI * TJ + NT - 1) / NT;
    constexpr bool RAGGED = NPT * NT != TI * TJ;
    wait_previous();
    extern __shared__ __align__(128) unsigned char smraw[];
    R2* sp = reinterpret_cast<R2*>(smraw);                        // [9][PH][PWS] (f_q, g_q) pairs
    R* sY = reinterpret_cast<R*>(sp + 9 * T::PSS);                // [2][PH][PWS] Y_x, Y_y
    R* srow = sY + 2 * T::PSS;                                    // separable: [TI][ROWTAB] (stride RS)
    R* scol = srow + TI * RS;                                     // separable: [TJ][COLTAB] (stride CS)
    R2* sx = reinterpret_cast<R2*>(srow);                         // C-grid: [9][PWS] the mirrored row 0
    R* sYx = reinterpret_cast<R*>(sx + 9 * T::PWS);               // C-grid: [2][PWS] its Y

    // blended maps of the solve's bodies (several only on general meshes)
    constexpr int MB = GEN ? MAX_BODIES : 1;
    __shared__ BodyMap<R> mapS[MB];
    __shared__ BodyMap<double> mapSd[MB];
    __shared__ SolveDev s_sol;
    __shared__ MeshDev s_mesh;
    __shared__ __align__(8) unsigned long long s_bar;   // tensor copies
    // wall nodes of the tile: which populations are missing; theirs go to the
    // staged columns that no window reaches (0, 1, 38, 39 of the first rows)
    __shared__ unsigned s_miss[TJ];
    static_assert(TJ == 32 && T::PH >= 8 && T::PWS == 40, "slots of the wall populations");
    auto s_wall = [&](int q, int tj) -> R2& { return sp[q * T::PSS + (tj >> 2) * T::PWS + (tj & 3) + ((tj & 2) ? 36 : 0)]; };
    __shared__ int s_next;   // the next chunk of the collision (tiles on the wall)

    const int tid = threadIdx.x;
    // ---- prologue: this CTA's tile and solve; the solve's step number k
    // (current buffer k & 1; k == 0 streams the initial state without
    // colliding).  Every thread reads what it needs to address its copies
    // itself, so the whole staging below is one batch of asynchronous copies
    // and one barrier.
    int sb, i0, j0, nr, nt, N;
    int ttma = 0, tsol = 0;   // table launch: the tile's tensor-copy flag and solve
    const SolveDev* sg = nullptr;   // table launch: the solve and mesh records
    const MeshDev* mg = nullptr;
    unsigned* ctr;
    StepMaps* const* mptr;
    if constexpr (UNIFORM) {
        sb = a.uorder ? (int)blockIdx.x : (int)blockIdx.z;
        j0 = (a.uorder ? (int)blockIdx.y : (int)blockIdx.x) * TJ;
        i0 = (a.uorder ? (int)blockIdx.z : (int)blockIdx.y) * TI;
        nr = a.umesh.nr; nt = a.umesh.nt; N = a.umesh.N;
        ctr = a.usol.counter + 4 * sb;
        mptr = a.usol.maps;
    } else {
        const TileDev* tg = a.tiles + blockIdx.x;
        sb = 0;
        j0 = tg->j0; i0 = tg->i0;
        ttma = tg->tma; tsol = tg->solve;
        sg = a.solves + tg->solve;
        mg = a.meshes + tg->mesh;
        nr = mg->nr; nt = mg->nt; N = mg->N;
        ctr = tg->counter;
        mptr = tg->maps;
    }
    // bodies of the solve (maps and body records per body)
    int nb = 1;
    if constexpr (GEN) nb = UNIFORM ? a.usol.nbody : __ldg(&sg->nbody);
    // C-grid (general meshes): the angular index does not wrap; rows below
    // row 0 are the mirrored rows across the cut, node (-k, j) = node (k, nt-1-j)
    int cg = 0, pb = 0;
    const int* ctab = nullptr;
    if constexpr (GEN) {
        cg = UNIFORM ? a.umesh.cgrid : mg->cgrid;
        ctab = UNIFORM ? a.umesh.coltype : mg->coltype;
        pb = UNIFORM ? a.umesh.box : mg->box;
    }
    // class of a C-grid's row-0 column (CT_*); the one-sided direction of a
    // row-0 junction's derivative along j
    auto ctype = [&](int j) -> int { return cg ? __ldg(ctab + j) : 0; };
    auto jdir_of = [&](int c) -> int { return (c & CT_JUNC) ? ((c & CT_JFWD) ? 1 : -1) : 0; };
    const int rlo = cg ? -CGRID_GHOST_ROWS : 0;
    auto rw = [&](int i) { return pb ? wrap_nt(i, nr) : i; };
    auto cw = [&](int j) { return cg ? j : wrap_nt(j, nt); };
    // a uniform launch from the host knows the step number; otherwise it is
    // the solve's device counter
    const unsigned kstep = (UNIFORM && a.ustep >= 0) ? (unsigned)a.ustep : __ldcg(ctr + 1);
    const int cur = (int)(kstep & 1u);
    const bool collide = kstep != 0u;
    {
        const int w = tid >> 5, l = tid & 31;
        constexpr int NW = NT / 32;
        const StepMaps* mi = (cur ? mptr[1] : mptr[0]) + (size_t)sb * nb;
        if (!UNIFORM && w == 0) cp_async_words(&s_sol, sg, (int)(sizeof(SolveDev) / 4), l);
        if (!UNIFORM && w == 1 % NW) cp_async_words(&s_mesh, mg, (int)(sizeof(MeshDev) / 4), l);
        for (int b = 0; b < nb; ++b) {
            if (w == 2 % NW) cp_async_words(&mapS[b], &mi[b].Sf, (int)(sizeof(BodyMap<R>) / 4), l);
            if (i0 == 0 && w == 3 % NW) cp_async_words(&mapSd[b], &mi[b].Sd, (int)(sizeof(BodyMap<double>) / 4), l);
        }
    }
    // solve / mesh fields: kernel parameters for a uniform launch, the copied
    // records for a table launch (valid after the staging barrier)
#define SD(x) (UNIFORM ? a.usol.x : s_sol.x)
#define MD(x) (UNIFORM ? a.umesh.x : s_mesh.x)
    const size_t o9 = (size_t)sb * 9 * N, o4 = (size_t)sb * 4 * N;
    const void* psrc = UNIFORM ? (cur ? a.usol.p[1] : a.usol.p[0]) : sg->p[cur];
    const void* Msrc = UNIFORM ? (cur ? a.usol.M[1] : a.usol.M[0]) : sg->M[cur];
    const R2* __restrict__ p_in = reinterpret_cast<const R2*>(psrc) + o9;
    const R* __restrict__ M_in = reinterpret_cast<const R*>(Msrc) + o4;
    const R* __restrict__ Y_in = reinterpret_cast<const R*>(UNIFORM ? a.usol.Y : sg->Y) + (size_t)sb * 2 * N;
    const R* __restrict__ rowtab = reinterpret_cast<const R*>(UNIFORM ? a.umesh.rowtab : mg->rowtab);
    const R* __restrict__ coltab = reinterpret_cast<const R*>(UNIFORM ? a.umesh.coltab : mg->coltab);
    const R* __restrict__ gcell = reinterpret_cast<const R*>(UNIFORM ? a.umesh.cellc : mg->cellc);
    const int pi0 = i0 - T::HP, sj0 = j0 - 4;       // global index of sp row 0, column 0
    const bool record = GEN && a.record;
    // float launches: the population and Y boxes of a tile whose columns do
    // not wrap come by two tensor copies that one thread issues (rows outside
    // the mesh arrive as zeros and are never read); uniform launches through
    // the handle's maps, the batch's separable table launches through each
    // solve's own.  C-grids (odd row lengths: no 16-byte strides) and the
    // general kernel's table launches stage by per-thread copies
    bool use_tma = false;
    if constexpr (UNIFORM || !GEN) {
        // (the boxes' shared-memory destinations are 128-byte aligned by the
        // layout; checked, so that another layout falls back instead of faulting)
        const unsigned sa = (unsigned)__cvta_generic_to_shared(sp), ya = (unsigned)__cvta_generic_to_shared(sY);
        const bool fits = sj0 >= 0 && sj0 + T::PWS <= nt && ((sa | ya) & 127u) == 0u;
        const CUtensorMap *tmP, *tmY;
        if constexpr (UNIFORM) {
            use_tma = a.tma != 0 && fits && !pb && !record;
            tmP = &a.tm_p[cur];
            tmY = &a.tm_Y;
        } else {
            use_tma = ttma != 0 && a.tmaps != nullptr && fits;
            tmP = a.tmaps + 4 * tsol + cur;
            tmY = a.tmaps + 4 * tsol + 2;
        }
        if (use_tma && tid == 0) {
            mbar_init(&s_bar);
            mbar_fence_init();
            mbar_expect_tx(&s_bar, 9u * T::PSS * (unsigned)sizeof(R2) + (collide ? 2u * T::PSS * (unsigned)sizeof(R) : 0u));
            tma_load_4d(sp, tmP, &s_bar, 2 * sj0, pi0, 0, UNIFORM ? sb : 0);
            if (collide) tma_load_4d(sY, tmY, &s_bar, sj0, pi0, 0, UNIFORM ? sb : 0);
        }
    }

    // ---- phase 1: stage the geometry tables, the populations and Y ---------
    if constexpr (!GEN) {
        constexpr int CE = 16 / (int)sizeof(R);   // table entries per 16-byte chunk
        for (int t = tid; t < TI * (ROWTAB / CE); t += NT) {
            const int li = t / (ROWTAB / CE), c = (t - li * (ROWTAB / CE)) * CE;
            cp_async16(srow + li * RS + c, rowtab + min(i0 + li, nr - 1) * ROWTAB + c);
        }
        for (int t = tid; t < TJ * (COLTAB / CE); t += NT) {
            const int lj = t / (COLTAB / CE), c = (t - lj * (COLTAB / CE)) * CE;
            cp_async16(scol + lj * CS + c, coltab + wrap_nt(j0 + lj, nt) * COLTAB + c);
        }
    }
    if (GEN && cg && !record) {
        // odd rows: one thread per node of the +-2 region, the nine
        // directions N apart; behind the tile's rows, in its first row of
        // tiles, the mirrored row 0 (node (0, nt-1-j))
        const int rows = T::PH + (i0 == 0 ? 1 : 0);
        for (int idx = tid; idx < rows * T::PW; idx += NT) {
            const int li = idx / T::PW, lj = idx - li * T::PW;
            const int i = pi0 + li, jj = j0 - T::HP + lj;
            const bool extra = li == T::PH;
            if ((unsigned)jj >= (unsigned)nt || (!extra && i >= nr)) continue;
            const ptrdiff_t n = extra ? nt - 1 - jj : i < 0 ? (ptrdiff_t)-i * nt + (nt - 1 - jj) : (ptrdiff_t)i * nt + jj;
            if (!in_bounds(n >= 0 && n < (ptrdiff_t)nr * nt, a.status)) continue;
            R2* dst = extra ? sx + lj + 2 : sp + li * T::PWS + lj + 2;
            const int ds = extra ? T::PWS : T::PSS;
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                cp_async8(dst + q * ds, p_in + (ptrdiff_t)q * N + n);
            }
            if (collide) {
                R* dy = extra ? sYx + lj + 2 : sY + li * T::PWS + lj + 2;
                cp_async4(dy, Y_in + n);
                cp_async4(dy + ds, Y_in + N + n);
            }
        }
    } else if (!use_tma && !record) {
        // rows of PWS (f, g) pairs per direction in 16-byte chunks (two float
        // pairs or one double pair); one thread per (row, chunk), the nine
        // directions N apart.  Row lengths are even.
        constexpr int CP = 16 / (int)sizeof(R2), NCH = T::PWS / CP;
        auto rowin = [&](int i) { return pb || (i >= 0 && i < nr); };
        for (int idx = tid; idx < T::PH * NCH; idx += NT) {
            const int ch = idx % NCH, li = idx / NCH;
            const int i = pi0 + li;
            if (!rowin(i)) continue;
            R2* dst = sp + li * T::PWS + ch * CP;
            const R2* src = p_in + (ptrdiff_t)rw(i) * nt + wrap_nt(sj0 + ch * CP, nt);
#pragma unroll
            for (int q = 0; q < 9; ++q) cp_async16(dst + q * T::PSS, src + (size_t)q * N);
        }
        if (collide) {
            for (int idx = tid; idx < T::PH * T::PW; idx += NT) {
                const int li = idx / T::PW, lj = idx - li * T::PW;
                const int i = pi0 + li;
                if (!rowin(i)) continue;
                const R* src = Y_in + (ptrdiff_t)rw(i) * nt + wrap_nt(j0 - T::HP + lj, nt);
                R* dst = sY + li * T::PWS + lj + 2;
                cp_async4(dst, src);
                cp_async4(dst + T::PSS, src + N);
            }
        }
    }
    // general meshes: the cached static departures are read per node in the
    // stream phase (the solves of a handle share them, so they are mostly
    // L2 hits); here a prefetch of the tile's entries into L2
    const bool dcache = GEN && UNIFORM && !record && a.usol.dep_code != nullptr;
    if (dcache) {
        const int len = min(TJ, nt - j0);
        for (int t = tid; t < 2 * 10 * TI; t += NT) {
            const int c = t / (2 * TI), r = (t >> 1) % TI, end = t & 1;
            const int i = i0 + r;
            if (i >= nr || len <= 0) continue;
            const size_t off = (size_t)i * nt + j0 + (end ? len - 1 : 0);
            const void* ad = c < 9 ? (const void*)(reinterpret_cast<const R2*>(a.usol.dep_xe) + (size_t)c * N + off)
                                   : (const void*)(a.usol.dep_code + off);
            asm volatile("prefetch.global.L2 [%0];" ::"l"(ad));
        }
    }
    const bool wtile = i0 == 0 && !pb && !record;   // the tile has wall nodes
    if (wtile && tid == 0) s_next = 0;
    cp_async_wait_all();
    __syncthreads();
    R2* __restrict__ p_out = reinterpret_cast<R2*>(SD(p[cur ^ 1])) + o9;
    R* __restrict__ M_out = reinterpret_cast<R*>(SD(M[cur ^ 1])) + o4;
    const R dt = SD(dt_f), mu = SD(mu_f), Cv = SD(Cv_f), iCv = SD(iCv_f), muP = SD(muP_f);
    const R xm = MD(xm_f), ym = MD(ym_f);
    // shared memory holds the post-collision pairs as deviations from the
    // free-stream pair of their direction, so that the Q2 weights (which sum
    // to 1 only up to round-off, the same way at every step of a node that
    // does not move) act on the deviation; an interpolated pair gets the
    // reference back
    auto ref_of = [&](int q) -> R2 { return pair(SD(fgref)[2 * q], SD(fgref)[2 * q + 1]); };
    auto add_ref = [&](int q, R2 v) -> R2 { return padd(v, ref_of(q)); };
    // static tile: no node of the tile lies in the blended region of the body
    // (F = I, V_G = 0 there), from a lower bound of the distance to the blend
    // centre on the separable O-grid (r of the tile's first row x min |e_j| -
    // |mesh centre - blend centre|) with a margin; such tiles skip the
    // kinematics.  Tiles near the boundary take the general path, which
    // gives the same result.
    bool tile_static = false;
    if constexpr (!GEN) {
        if (!mapS[0].active) {
            tile_static = true;
        } else {
            // in the element type of the path (no float64 on the float path),
            // with a margin well above its rounding
            const R rmin = srow[RT_R] * MD(emin_f);
            const R ox = xm - mapS[0].xc, oy = ym - mapS[0].yc;
            const R r_out = mapS[0].r_in + rcp_(mapS[0].inv_w);
            tile_static = rmin - sqrt_(ox * ox + oy * oy) > r_out * (R(1) + R(1e-4)) + R(1e-5);
        }
    }

    // moment c at node (r, cc) of M^k
    auto Mat = [&](int c, int r, int cc) -> R { return M_in[(ptrdiff_t)c * N + (ptrdiff_t)rw(r) * nt + cw(cc)]; };
    // inverse metric and coordinates of node n (general meshes)
    auto metric = [&](int n, R* jn) {
        if constexpr (GEN) ld4(reinterpret_cast<const R*>(MD(jinv)) + 4 * (ptrdiff_t)n, jn[0], jn[1], jn[2], jn[3]);
    };
    // blended map of the stream at node (i, j): F and V_G; false where the
    // blend does not move it
    auto motion = [&](int n, int ti, int tj, R& F00, R& F01, R& F10, R& F11, R& vx, R& vy) -> bool {
        if constexpr (GEN) {
            const R2 x = __ldg(reinterpret_cast<const R2*>(MD(nodex)) + n);
            return kinematics_sum(mapS, nb, x.x, x.y, F00, F01, F10, F11, vx, vy);
        } else {
            if (tile_static) {
                F00 = R(1); F01 = R(0); F10 = R(0); F11 = R(1); vx = R(0); vy = R(0);
                return false;
            }
            const R r = srow[ti * RS + RT_R], ex = scol[tj * CS + CT_E], ey = scol[tj * CS + CT_E + 1];
            return kinematics(mapS[0], xm + r * ex, ym + r * ey, F00, F01, F10, F11, vx, vy);
        }
    };

    // ---- wall nodes (Sec. III A), by the first warp while the others start
    // the collision: which populations are missing, and theirs by Grad's
    // approximation, from M^k alone (this row's chain of loads and arithmetic
    // is twice a whole row of the stream; behind it, it made the wall tiles
    // last 21.5 thousand cycles against 10.4 of the others on a 256 x 128
    // O-grid)
    if (wtile && tid < TJ) {
        const int j = j0 + tid;
        const int ct = (cg && j < nt) ? ctype(j) : 0;
        unsigned missing = 0u;
        R fw[9], gw[9];
        if (j < nt && (!cg || ((ct & CT_WALL) && !(ct & CT_DUP)))) {
            R F00, F01, F10, F11, vx, vy, jn[4];
            metric(j, jn);
            motion(j, 0, tid, F00, F01, F10, F11, vx, vy);
            const R idF = rcp_(fm(F00, F11, -(F01 * F10)));
            const R i00 = F11 * idF, i01 = -F01 * idF, i10 = -F10 * idF, i11 = F00 * idF;
            // missing populations: departure point inside the body,
            // c_hat . n0 > 0, decided in float64.  A wall moves rigidly with
            // its own body (it lies in that body's rigid zone and outside
            // every other's blended region).  A float value beyond its
            // rounding error has the float64 value's sign; the others, the
            // directions along the wall, are decided below.  The error: some
            // ten roundings (2^-24) each of the inverse map's entries, the
            // velocity and the coordinates that it is formed from; sixteen
            // times the sum of all of them
            const BodyMap<double>& mw = mapSd[GEN ? (ct >> CT_BODY_SHIFT) & (MAX_BODIES - 1) : 0];
            const BodyMap<R>& mf = mapS[GEN ? (ct >> CT_BODY_SHIFT) & (MAX_BODIES - 1) : 0];
            const double n0x = MD(n0)[2 * j], n0y = MD(n0)[2 * j + 1];
            const R fx = (R)n0x, fy = (R)n0y;
            R reach = abs_(i00) + abs_(i01) + abs_(i10) + abs_(i11);
            if (mw.active) {
                R X, Y;
                if constexpr (GEN) {
                    const R2 x = __ldg(reinterpret_cast<const R2*>(MD(nodex)) + j);
                    X = x.x;
                    Y = x.y;
                } else {
                    const R r = srow[RT_R];
                    X = abs_(xm) + abs_(r * scol[tid * CS + CT_E]);
                    Y = abs_(ym) + abs_(r * scol[tid * CS + CT_E + 1]);
                }
                reach += abs_(vx) + abs_(vy) + abs_(mf.vtx) + abs_(mf.vty) +
                         (abs_(mf.va00) + abs_(mf.va01) + abs_(mf.va10) + abs_(mf.va11)) *
                             (abs_(X) + abs_(Y) + abs_(mf.xp) + abs_(mf.yp));
            }
            const R round = R(16.0 / (1 << 24)) * reach;
            unsigned near = 0u;
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const R v = (i00 * R(cxq(q)) + i01 * R(cyq(q)) - vx) * fx + (i10 * R(cxq(q)) + i11 * R(cyq(q)) - vy) * fy;
                if (v > round) missing |= 1u << q;
                else if (!(v < -round)) near |= 1u << q;
            }
            if (!mw.active) near &= ~1u;   // (a wall at rest: the rest population's is zero)
            if (near) {
                double D00 = 1.0, D01 = 0.0, D10 = 0.0, D11 = 1.0, dvx = 0.0, dvy = 0.0;
                if (mw.active) {
                    const double px = MD(xw)[2 * j] - mw.xp, py = MD(xw)[2 * j + 1] - mw.yp;
                    D00 = 1.0 + mw.a00; D01 = mw.a01; D10 = mw.a10; D11 = 1.0 + mw.a11;
                    dvx = mw.va00 * px + mw.va01 * py + mw.vtx;
                    dvy = mw.va10 * px + mw.va11 * py + mw.vty;
                    const double idd = rcp_(D00 * D11 - D01 * D10);
                    D00 *= idd; D01 *= idd; D10 *= idd; D11 *= idd;
                }
#pragma unroll
                for (int q = 0; q < 9; ++q) {
                    if (!(near & (1u << q))) continue;
                    const double cx = cxq(q), cy = cyq(q);
                    const double hx = (D11 * cx - D01 * cy) - dvx, hy = (-D10 * cx + D00 * cy) - dvy;
                    if (hx * n0x + hy * n0y > 1e-12) missing |= 1u << q;
                }
            }
            if (missing) {
                const bool rear = (ct & CT_JUNC) != 0, below = (ct & (CT_CUT | CT_JUNC)) != 0;
                int wa, wb;
                R xi, eta, G[4];
                bool found;
                if constexpr (GEN) {
                    found = depart_gen<R>(gcell, jn, 0, j, nr, nt, cg, dt * fx, dt * fy, wa, wb, xi, eta, below, false, a.status);
                    grad_map_j(jn[0], jn[1], jn[2], jn[3], F00, F01, F10, F11, G);
                } else {
                    NodeGeo<R> geo;
                    node_geo(0, j, nr, srow, scol + tid * CS, geo);
                    found = depart(geo, 0, dt * fx, dt * fy, wa, wb, xi, eta);
                    grad_map(srow, scol + tid * CS, F00, F01, F10, F11, G);
                }
                if (found) found = in_bounds(wa >= (cg ? -2 : 0) && wa + 2 < nr && (!cg || (wb >= 0 && wb + 2 < nt)), a.status);
                if (!found) atomicOr(a.status, ST_BPOINT);
                WallTarget<R> t;
                t.ux = vx;
                t.uy = vy;
                wall_rho_T<R>(Mat, j, nt, found, wa, wb, xi, eta, GEN && cg && wa == -2, t.rho, t.T);
#pragma unroll
                for (int c = 0; c < 3; ++c) wall_gradient<R>(Mat, c + 1, j, rear, jdir_of(ct), G, t.gr[2 * c], t.gr[2 * c + 1]);
                grad_f(t, mu, dt, iCv, fw);
                grad_g(t, mu, dt, Cv, iCv, SD(iPr_f), gw);
            }
        }
        s_miss[tid] = missing;
        if (use_tma) mbar_wait0(&s_bar, a.status);
        if (missing) {
#pragma unroll
            for (int q = 0; q < 9; ++q) s_wall(q, tid) = pair(fw[q], gw[q]);
        }
    } else if (use_tma) {
        mbar_wait0(&s_bar, a.status);   // (the barrier above ordered the init)
    }

    // ---- phase 2: collision of step k on the +-2 region ---------------------
    if (collide) {
        const bool xrow = GEN && cg && i0 == 0;
        const int total = T::PS + (xrow ? T::PW : 0);
        auto collide_node = [&](int idx) {
            const int li = idx / T::PW, lj = idx - li * T::PW;
            const int i = pi0 + li, jj = j0 - T::HP + lj;
            const bool extra = GEN && li == T::PH;
            if (!pb && !extra && (i >= nr || (i < 0 && !(GEN && cg)))) return;
            if (cg && (unsigned)jj >= (unsigned)nt) return;
            R2* s = sp + li * T::PWS + lj + 2;
            const R* y = sY + li * T::PWS + lj + 2;
            int ds = T::PSS;
            if (extra) {
                s = sx + lj + 2;
                y = sYx + lj + 2;
                ds = T::PWS;
            }
            R2 pq[9];
            if ((!pb && !extra && i == nr - 1) || (cg && (jj == 0 || jj == nt - 1))) {
                // far field: the equilibria of its targets
                const ptrdiff_t n = extra ? nt - 1 - jj : i < 0 ? (ptrdiff_t)-i * nt + (nt - 1 - jj) : (ptrdiff_t)i * nt + cw(jj);
                const R rho = M_in[n], ux = M_in[N + n], uy = M_in[(ptrdiff_t)2 * N + n], Tn = M_in[(ptrdiff_t)3 * N + n];
                R f[9], g[9];
                f_equilibrium(rho, ux, uy, Tn, f);
                g_equilibrium(rho, ux, uy, Tn, Cv, g);
#pragma unroll
                for (int q = 0; q < 9; ++q) pq[q] = pair(f[q], g[q]);
            } else {
#pragma unroll
                for (int q = 0; q < 9; ++q) pq[q] = s[q * ds];
                collide_pairs(pq, y[0], y[ds], mu, muP, dt, iCv);
            }
#pragma unroll
            for (int q = 0; q < 9; ++q) s[q * ds] = psub(pq[q], ref_of(q));
        };
        // fixed shares, or in a tile with wall nodes chunks as the warps come
        // (the first one after its wall nodes); one copy of the code, so that a
        // node's collision rounds alike in both
        const int lane = tid & 31;
        auto grab = [&]() {
            int c = 0;
            if (lane == 0) c = atomicAdd(&s_next, 32);
            return __shfl_sync(0xffffffffu, c, 0);
        };
        for (int c = wtile ? grab() : tid - lane; c < total; c = wtile ? grab() : c + NT)
            if (c + lane < total) collide_node(c + lane);
        __syncthreads();
    } else if (!record) {
        // the initial state is streamed as it is: the staged pairs are full
        // values (nothing collided them), made deviations like collided ones
        for (int idx = tid; idx < 9 * T::PSS; idx += NT) {
            const int col = idx % T::PWS;
            if (col >= 2 && col < T::PWS - 2) sp[idx] = psub(sp[idx], ref_of(idx / T::PSS));
        }
        if (GEN && cg && i0 == 0)
            for (int idx = tid; idx < 9 * T::PWS; idx += NT) sx[idx] = psub(sx[idx], ref_of(idx / T::PWS));
        __syncthreads();
    }

    // ---- phase 3: stream step k+1 ----------------------------------------
#pragma unroll 1
    for (int k = 0; k < NPT; ++k) {
        const int t = tid + k * NT;
        const int ti = t / TJ, tj = t - (t / TJ) * TJ;
        const int i = i0 + ti, j = j0 + tj;
        if ((RAGGED && ti >= TI) || i >= nr || j >= nt) continue;
        // C-grid: the second copies of the row-0 cut nodes (and of the rear
        // point) are written by their first copies; rows 1-4 also write
        // their moments into their mirrored slots below row 0
        const int ct = (cg && i == 0) ? ctype(j) : 0;
        if (ct & CT_DUP) continue;
        const int n2 = i == 0 ? nt - 1 - j : -i * nt + (nt - 1 - j);
        const bool dup2_ = (ct & (CT_CUT | CT_JUNC)) != 0, mir_ = cg && i >= 1 && i <= CGRID_GHOST_ROWS;
        const bool n2ok = !(dup2_ || mir_) || in_bounds(n2 >= rlo * nt && n2 < nr * nt, a.status);
        const bool dup2 = dup2_ && n2ok;
        const bool mir = mir_ && n2ok;
        const int n = i * nt + j;
        const R* row = srow + ti * RS;
        const R* col = scol + tj * CS;
        const bool farj = cg && i < nr - 1 && (j == 0 || j == nt - 1);
        if ((!pb && i == nr - 1) || farj) {
            if (record) continue;
            // far field, on a C-grid also the outlet columns (direction along j)
            const double* fd = farj ? MD(fardirj) + 4 * i + (j == 0 ? 0 : 2) : MD(fardir) + 2 * j;
            const double un = SD(uinf_x) * fd[0] + SD(uinf_y) * fd[1];
            const R bx = -dt * (R)fd[0], by = -dt * (R)fd[1];
            int wa = 0, wb = 0;
            R xi, eta;
            bool ok;
            if constexpr (GEN) {
                R jn[4];
                metric(n, jn);
                ok = depart_gen<R>(gcell, jn, i, j, nr, nt, cg, bx, by, wa, wb, xi, eta, dup2 || pb, pb, a.status, cg ? nt - 2 : -1);
            } else {
                NodeGeo<R> fg;
                node_geo(i, j, nr, row, col, fg);
                ok = depart(fg, i, bx, by, wa, wb, xi, eta);
            }
            if (!ok) atomicOr(a.status, ST_BPOINT);
            ok = ok && in_bounds(wa >= (cg ? -2 : 0) && wa + 2 < nr && (!cg || (wb >= 0 && wb + 2 < nt)), a.status);
            const R rho = far_target<R>(Mat, 0, i, j, ok, wa, wb, xi, eta);
            const bool inlet = un < 0.0;
            const R ux = inlet ? SD(uinf_x_f) : far_target<R>(Mat, 1, i, j, ok, wa, wb, xi, eta);
            const R uy = inlet ? SD(uinf_y_f) : far_target<R>(Mat, 2, i, j, ok, wa, wb, xi, eta);
            const R Tt = inlet ? SD(T_inf_f) : far_target<R>(Mat, 3, i, j, ok, wa, wb, xi, eta);
            R f[9], g[9];
            f_equilibrium(rho, ux, uy, Tt, f);
            g_equilibrium(rho, ux, uy, Tt, Cv, g);
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const R2 v = pair(f[q], g[q]);
                p_out[(size_t)q * N + n] = v;
                if (dup2) p_out[(ptrdiff_t)q * N + n2] = v;
            }
            M_out[n] = rho; M_out[(size_t)N + n] = ux; M_out[(size_t)2 * N + n] = uy;
            M_out[(size_t)3 * N + n] = Tt;
            if (dup2 || mir) {
                M_out[n2] = rho; M_out[(ptrdiff_t)N + n2] = ux; M_out[(ptrdiff_t)2 * N + n2] = uy;
                M_out[(ptrdiff_t)3 * N + n2] = Tt;
            }
            continue;
        }
        const bool wall = !pb && i == 0 && (!cg || (ct & CT_WALL));
        NodeGeo<R> geo;
        if constexpr (!GEN) {
            // window origins as offsets in the staged tile
            node_geo(i, j, nr, row, col, geo);
            geo.wa0 = (geo.wa0 - pi0) * T::PWS;
            geo.wa1 = (geo.wa1 - pi0) * T::PWS;
            geo.wb0 -= sj0;
            geo.wb1 -= sj0;
        }
        R F00, F01, F10, F11, vx, vy;
        const bool moved = motion(n, ti, tj, F00, F01, F10, F11, vx, vy);
        const R idF = rcp_(fm(F00, F11, -(F01 * F10)));
        const R i00 = F11 * idF, i01 = -F01 * idF, i10 = -F10 * idF, i11 = F00 * idF;
        const unsigned missing = wall && !record ? s_miss[tj] : 0u;
        bool lost = false;
        const int own = (ti + T::HP) * T::PWS + tj + T::HP + 2;   // this node in the staged tile
        // population q of the node: written as it is found, its share added to
        // the moments (in the order of q on every path)
        R rho = R(0), jx = R(0), jy = R(0), s2 = R(0);
        // v: the population, d: its deviation from the free stream's.  The moments
        // are summed over the deviations (nine small numbers), which keeps their
        // rounding to that of the last addition
        auto put = [&](int q, R2 v, R2 d) {
            p_out[(size_t)q * N + n] = v;
            if (dup2) p_out[(ptrdiff_t)q * N + n2] = v;
            rho += d.x;
            s2 += d.y;
            const int cx = cxq(q), cy = cyq(q);
            if (cx) jx += cx > 0 ? d.x : -d.x;
            if (cy) jy += cy > 0 ? d.x : -d.x;
        };
        R jn[4] = {R(0), R(0), R(0), R(0)};
        // departure solve of this node for a displacement (dx, dy): the window's
        // offset in the staged tile
        auto departure = [&](int inode, R dx, R dy, int& base, R& xi, R& eta) -> bool {
            int wa, wb;
            bool ok;
            if constexpr (GEN) {
                ok = depart_gen<R>(gcell, jn, inode, j, nr, nt, cg, dx, dy, wa, wb, xi, eta, dup2 || pb, pb, a.status);
                base = (wa - pi0) * T::PWS + (wb - sj0);
            } else {
                ok = depart(geo, inode, dx, dy, wa, wb, xi, eta);
                base = wa + wb;
            }
            return ok && in_bounds(base >= 0 && base + 2 * T::PWS + 2 < T::PSS, a.status);
        };
        // general meshes: a node the blend does not move takes its cached
        // departures (the same solves, made once for the handle's dt)
        unsigned long long dcode = ~0ull;
        if constexpr (GEN) {
            if (dcache && !moved && i > 0) dcode = __ldg(a.usol.dep_code + n);
            if (dcode == ~0ull) metric(n, jn);
            if (record) {
                if (!moved && i > 0) {
                    R2* gxe = reinterpret_cast<R2*>(a.usol.dep_xe);
                    unsigned long long code = 0ull;
                    bool ok = true;
#pragma unroll 1
                    for (int q = 0; q < 9; ++q) {
                        const R cx = (R)cxq(q), cy = (R)cyq(q);
                        const R hx = fm(i00, cx, fm(i01, cy, -vx)), hy = fm(i10, cx, fm(i11, cy, -vy));
                        int base;
                        R2 xe;
                        unsigned nib = 16u;   // a lost departure
                        if (departure(i, -dt * hx, -dt * hy, base, xe.x, xe.y)) {
                            const int dr = base / T::PWS - (i - pi0), dc = base % T::PWS - (j - sj0);
                            if (dr < -3 || dr > 0 || dc < -3 || dc > 0) ok = false;
                            nib = (unsigned)(((dr + 3) << 2) | (dc + 3));
                        }
                        code |= (unsigned long long)nib << (5 * q);
                        gxe[(size_t)q * N + n] = xe;
                    }
                    a.usol.dep_code[n] = ok ? code : ~0ull;
                }
                continue;
            }
        }
        if (GEN && dcode != ~0ull) {
            R2 xe[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) xe[q] = __ldg(reinterpret_cast<const R2*>(a.usol.dep_xe) + (size_t)q * N + n);
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const unsigned nib = (unsigned)(dcode >> (5 * q)) & 31u;
                R2 v;
                if (nib & 16u) {
                    lost = true;
                    v = sp[q * T::PSS + own];
                } else {
                    const int base = own + ((int)(nib >> 2) - 3) * T::PWS + ((int)(nib & 3u) - 3);
                    R Lx[3], Ly[3];
                    lagrange3(xe[q].x, Lx);
                    lagrange3(xe[q].y, Ly);
                    v = gather9(sp + q * T::PSS + base, T::PWS, Lx, Ly);
                }
                put(q, add_ref(q, v), v);
            }
        } else if (!GEN && !moved && i > 0) {
            // a node the blend does not move: c_hat = c, and the rest
            // population's departure point is the node itself
            put(0, add_ref(0, sp[own]), sp[own]);
            auto pull = [&](auto cxc, auto cyc, int q) {
                int wa, wb;
                R xi, eta;
                R2 v;
                const bool ok = depart_static<decltype(cxc)::value, decltype(cyc)::value>(geo, dt, wa, wb, xi, eta);
                const int base = wa + wb;
                if (ok && in_bounds(base >= 0 && base + 2 * T::PWS + 2 < T::PSS, a.status)) {
                    R Lx[3], Ly[3];
                    lagrange3(xi, Lx);
                    lagrange3(eta, Ly);
                    v = gather9(sp + q * T::PSS + base, T::PWS, Lx, Ly);
                } else {
                    lost = true;
                    v = sp[q * T::PSS + own];
                }
                put(q, add_ref(q, v), v);
            };
            using P1 = std::integral_constant<int, 1>;
            using Z0 = std::integral_constant<int, 0>;
            using M1 = std::integral_constant<int, -1>;
            pull(P1{}, Z0{}, 1);
            pull(Z0{}, P1{}, 2);
            pull(M1{}, Z0{}, 3);
            pull(Z0{}, M1{}, 4);
            pull(P1{}, P1{}, 5);
            pull(M1{}, P1{}, 6);
            pull(M1{}, M1{}, 7);
            pull(P1{}, M1{}, 8);
        } else {
            // moving nodes and walls: one copy of the solve, not nine (the
            // kernel's instructions have to fit the instruction cache)
#pragma unroll 1
            for (int q = 0; q < 9; ++q) {
                if (missing & (1u << q)) {
                    put(q, s_wall(q, tj), psub(s_wall(q, tj), ref_of(q)));   // Grad's approximation
                    continue;
                }
                const R cx = (R)cxq(q), cy = (R)cyq(q);
                const R hx = fm(i00, cx, fm(i01, cy, -vx)), hy = fm(i10, cx, fm(i11, cy, -vy));
                int base;
                R xi, eta;
                R2 v;
                if (departure(i, -dt * hx, -dt * hy, base, xi, eta)) {
                    R Lx[3], Ly[3];
                    lagrange3(xi, Lx);
                    lagrange3(eta, Ly);
                    const R2* p = sp + q * T::PSS + base;
                    // (the mirrored windows of a C-grid's cut nodes start at row
                    // -2, the tile's first staged row)
                    if (GEN && dup2 && base < T::PWS) v = gather9_rows(p, T::PWS, sx + q * T::PWS + base, Lx, Ly);
                    else v = gather9(p, T::PWS, Lx, Ly);
                } else {
                    lost = true;
                    v = sp[q * T::PSS + own];
                }
                put(q, add_ref(q, v), v);
            }
        }
        if (lost) atomicOr(a.status, ST_DEPARTURE);
        rho += SD(mref)[0];
        jx += SD(mref)[1];
        jy += SD(mref)[2];
        s2 += SD(mref)[3];
        const R ir = rcp_(rho), ux = jx * ir, uy = jy * ir;
        const R Tn = fm(R(-0.5), fm(ux, ux, uy * uy), R(0.5) * s2 * ir) * iCv;
        if (!(rho > R(0)) || !(Tn > R(0)) || !isfinite(ux) || !isfinite(uy)) atomicOr(a.status, ST_NONPHYS);
        M_out[n] = rho; M_out[(size_t)N + n] = ux; M_out[(size_t)2 * N + n] = uy;
        M_out[(size_t)3 * N + n] = Tn;
        if (dup2 || mir) {
            M_out[n2] = rho; M_out[(ptrdiff_t)N + n2] = ux; M_out[(ptrdiff_t)2 * N + n2] = uy;
            M_out[(ptrdiff_t)3 * N + n2] = Tn;
        }
    }
    // a launch that took its step number from the device counter advances it
    // when the last CTA of the solve has read it (a host launch's number is
    // written by the loads that follow)
    if (!record && !(UNIFORM && a.ustep >= 0) && tid == 0) {
        const unsigned ntiles = UNIFORM ? (unsigned)a.usol.ntiles : (unsigned)s_sol.ntiles;
        if (atomicAdd(ctr, 1u) == ntiles - 1u) {
            ctr[0] = 0u;
            ctr[1] = kstep + 1u;
        }
    }
}

#undef SD
#undef MD

// ---------------------------------------------------------------------------
template <typename R>
__global__ void k_init(const double* __restrict__ M, typename Vec2<R>::T* __restrict__ P,
                       R* __restrict__ Mout, int N, int nbatch, double Cv) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (size_t)N * nbatch) return;
    const size_t b = t / N, n = t - b * N;
    const double* Mb = M + b * 4 * N;
    const R rho = (R)Mb[n], ux = (R)Mb[N + n], uy = (R)Mb[2 * (size_t)N + n], T = (R)Mb[3 * (size_t)N + n];
    R fe[9], ge[9];
    f_equilibrium(rho, ux, uy, T, fe);
    g_equilibrium(rho, ux, uy, T, (R)Cv, ge);
    for (int q = 0; q < 9; ++q) {
        typename Vec2<R>::T v;
        v.x = fe[q];
        v.y = ge[q];
        P[(b * 9 + q) * N + n] = v;
    }
    for (int c = 0; c < 4; ++c) Mout[(b * 4 + c) * N + n] = (R)Mb[c * (size_t)N + n];
}

// Rows of node values to float64 for a caller's array, in its node order (node i
// of the row is order[i]; null: as it lies).  Bound by the 8 bytes per value it
// writes and their copy (150 GB/s to pageable memory); copying the path's type
// and widening it on the host took nine times as long (2 M values: 0.11 against
// 0.9 ms; an element list's reordering came on top).
template <typename R>
__global__ void k_read(const R* __restrict__ src, size_t stride, const int* __restrict__ order, double* __restrict__ dst,
                       int N, size_t total) {
    const size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= total) return;
    const size_t row = t / N;
    const int i = (int)(t - row * N);
    dst[t] = (double)src[row * stride + (order ? order[i] : i)];
}

__global__ void k_prepare(const BodyDev* __restrict__ bodies, const BodyStateDev* S_cur,
                          const BodyStateDev* S_next, const BodyStateDev* S_vgprev,
                          const double* loads, double dt, int nbatch, StepMaps* maps) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nbatch) return;
    StepMaps m = maps[b];
    const BodyStateDev sc = S_cur ? S_cur[b] : m.S_cur;
    const BodyStateDev sn = S_next ? S_next[b] : m.S_next;
    const BodyStateDev sp = S_vgprev ? S_vgprev[b] : m.S_vgprev;
    build_maps(bodies[b], sc, sn, sp, dt, m);
    if (loads)
        for (int c = 0; c < 3; ++c) m.loads[c] = loads[b * 3 + c];
    maps[b] = m;
}

__global__ void k_advance(const BodyDev* __restrict__ bodies, const double* __restrict__ loads,
                          double dt, long long n, int nbatch, StepMaps* maps) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nbatch) return;
    StepMaps m = maps[b];
    const BodyStateDev s = m.S_next;
    const BodyStateDev ns = rk4_body(bodies[b], s, loads[b * 3 + 1], loads[b * 3 + 2], dt, n);
    build_maps(bodies[b], m.S_cur, ns, s, dt, m);
    maps[b] = m;
}

// Tile shapes of the step kernel (angular tile width one warp).
constexpr int TJ = TILE_J;

template <int TI, int NT, int MINB, bool UNIFORM, bool GEN = false>
struct StepKernel {
    static cudaError_t configure() {
        static const cudaError_t e = cudaFuncSetAttribute(k_step<TI, TJ, NT, MINB, UNIFORM, GEN>,
                                                          cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                          (int)step_smem_bytes<TI, TJ, GEN>());
        return e;
    }

    static cudaError_t launch(const StepArgs& a, int nbatch, cudaStream_t s) {
        const cudaError_t e = configure();
        if (e != cudaSuccess) return e;
        const int nti = (a.umesh.nr + TI - 1) / TI;
        const dim3 grid = !UNIFORM   ? dim3(a.ntiles)
                          : a.uorder ? dim3(nbatch, a.umesh.ntj, nti)
                                     : dim3(a.umesh.ntj, nti, nbatch);
        return launch_behind(k_step<TI, TJ, NT, MINB, UNIFORM, GEN>, grid, NT, step_smem_bytes<TI, TJ, GEN>(), s, true, a);
    }
};

// The float kernel of a tile shape: separable shapes by variant, on general
// meshes those of default_shape_general.
template <bool UNIFORM, typename Fn>
static cudaError_t with_kernel(bool general, int variant, Fn fn) {
    if (general) switch (variant) {
        case 0: return fn(StepKernel<8, 256, 3, UNIFORM, true>());
        case 1: return fn(StepKernel<16, 256, 3, UNIFORM, true>());
        default: return fn(StepKernel<16, 512, 2, UNIFORM, true>());
    }
    switch (variant) {
        case 1: return fn(StepKernel<16, 256, 3, UNIFORM>());
        case 2: return fn(StepKernel<12, 192, 4, UNIFORM>());
        case 3: return fn(StepKernel<12, 384, 2, UNIFORM>());
        case 4: return fn(StepKernel<16, 512, 2, UNIFORM>());
        default: return fn(StepKernel<8, 256, 3, UNIFORM>());
    }
}

int step_variants(int precision) { return precision == 0 ? 3 : 5; }

// Tile shape where no schedule was asked for, by the tiles of 16 rows (float64:
// one row per block).  Below a tile per SM more and smaller tiles spread the
// work; up to four per SM a tile's own time counts, which 512 threads shorten;
// beyond, the three blocks of 256 threads that an SM holds overlap better.
// Measured per step with 8 x 32 tiles, 16 x 32 / 512 threads, 16 x 32 / 256
// threads: 256 x 128 (64 tiles) 20.2, 21.3, 23.3 us; 256 x 128 x 4 (256) 25.3, 24.7,
// 25.6; 201 x 150 x 5 (325) 28.3, 27.3, 29.5; 512 x 256 x 2 (512) 32.7, 31.8, 32.8;
// x 3 (768) 43.0, 40.3, 39.8; x 16 (4096) 150, 140.7, 139.9; 8192 x 512 (8192) 259,
// 242.3, 240.6.
int default_shape(int precision, long long tiles16) {
    if (precision == 0) return 0;
    return tiles16 < 152 ? 0 : tiles16 < 608 ? 4 : 1;
}

// The same on general meshes (0: 8 x 32 tiles, 1: 16 x 32 / 256 threads, 2: 16 x 32 /
// 512 threads; 456 blocks of the first two are resident at once, 304 of the
// third).  8-row tiles as long as they are one wave; then a tile's own time
// counts, which its nodes that solve their departures and its per-thread copies
// make long and 512 threads halve; tiles staged by tensor copies keep 256 where no
// body moves and they are one wave, and from four per SM on.  Measured per step
// (us) with 0, 1, 2, body at rest and moving.  Ellipse, tensor copies: 40 x 64 (6
// tiles) 26.4 30.5 28.4, 28.0 38.2 31.7; 200 x 128 x 4 (208) 28.5 28.9 29.1, 31.6
// 38.5 32.7; 300 x 160 x 4 (380) 34.4 33.1 34.9, 39.7 44.8 38.1; 512 x 256 x 2 (512)
// 40.6 41.6 38.1, 44.6 44.5 45.0; x 4 (1024, order 0) 61.2 57.9 60.6, 72.3 74.8 69.8;
// x 15 (3840) - 159.8 170.1, - 202.3 204.5.  C-grid: 60 x 129 x 4 (80) 34.2 38.9 34.9,
// 34.0 51.5 41.0; 192 x 257 x 4 (432) 40.7 44.0 37.9, 43.9 58.0 44.6; 192 x 385 x 16
// (2496) 140.0 141.1 131.8, 167.7 173.2 159.8.
int default_shape_general(bool tma, bool moving, long long tiles16) {
    if (tiles16 <= 228) return 0;
    if (!tma) return 2;
    return tiles16 >= 608 || (!moving && tiles16 <= 456) ? 1 : 2;
}

// CTA order of a handle where none was asked for (0: solve by solve, 1: the solves
// of a tile together).  Order 1 shares the mesh's tables between neighbouring
// blocks; from half the L2's size on (184 bytes of state a node against 129 MB)
// order 0 finds more of a solve's populations there, as long as a launch is not
// many waves.  Measured per step (us) with 0 and 1: separable 512 x 256 x 2 32.0
// 32.2; x 4 43.5 47.5, moving 46.7 50.4; x 8 71.0 75.8, 78.3 79.7; x 16 127.0 128.3,
// 140.3 139.1; ellipse 256 x 256 x 5 (60 MB) 44.6 43.3, 54.9 52.2; 512 x 256 x 3 (72
// MB) 52.3 55.1, 57.7 67.1; x 4 57.9 73.8, 74.8 81.2; x 15 159.8 167.5, 202.3 206.5.
// Without tensor copies (C-grids) the two agree within 2%.
int default_order(bool tma, bool general, long long nodes, long long tiles16) {
    return tma && nodes * 184 > 66000000ll && (general || tiles16 < 3040) ? 0 : 1;
}

int tile_rows(int precision, int variant) {
    if (precision == 0) return 1 << variant;
    switch (variant) {
        case 1: return 16;
        case 2: return 12;
        case 3: return 12;
        case 4: return 16;
        default: return 8;
    }
}

cudaError_t prepare_step(int precision, int variant, bool uniform, bool general) {
    if (precision == 0) return cudaSuccess;
    auto conf = [](auto k) { return k.configure(); };
    return uniform ? with_kernel<true>(general, variant, conf) : with_kernel<false>(general, variant, conf);
}

cudaError_t launch_step(const StepArgs& a, int precision, bool general, int variant, cudaStream_t s) {
    if (precision == 0) return launch_stream64(a, false, general, tile_rows(0, variant), 0, s);
    return with_kernel<false>(general, variant, [&](auto k) { return k.launch(a, 0, s); });
}

cudaError_t launch_step_uniform(const StepArgs& a, int precision, int variant, int nbatch, cudaStream_t s) {
    const bool general = a.umesh.general != 0;
    if (precision == 0) return launch_stream64(a, true, general, tile_rows(0, variant), nbatch, s);
    return with_kernel<true>(general, variant, [&](auto k) { return k.launch(a, nbatch, s); });
}

cudaError_t launch_init(int precision, const double* M, void* P, void* Mout, int N, int nbatch,
                        double Cv, cudaStream_t s) {
    const size_t total = (size_t)N * nbatch;
    const int bs = 256;
    const unsigned nb = (unsigned)((total + bs - 1) / bs);
    if (precision == 0)
        k_init<double><<<nb, bs, 0, s>>>(M, (double2*)P, (double*)Mout, N, nbatch, Cv);
    else
        k_init<float><<<nb, bs, 0, s>>>(M, (float2*)P, (float*)Mout, N, nbatch, Cv);
    return cudaGetLastError();
}

cudaError_t launch_read(int precision, const void* src, size_t stride, const int* order, double* dst, int N, size_t rows,
                        cudaStream_t s) {
    const size_t total = rows * (size_t)N;
    const unsigned nb = (unsigned)((total + 255) / 256);
    if (precision == 0) k_read<double><<<nb, 256, 0, s>>>((const double*)src, stride, order, dst, N, total);
    else k_read<float><<<nb, 256, 0, s>>>((const float*)src, stride, order, dst, N, total);
    return cudaGetLastError();
}

cudaError_t launch_prepare(const BodyDev* bodies, const BodyStateDev* S_cur,
                           const BodyStateDev* S_next, const BodyStateDev* S_vgprev,
                           const double* loads, double dt, int nbatch, StepMaps* maps,
                           cudaStream_t s) {
    k_prepare<<<(nbatch + 127) / 128, 128, 0, s>>>(bodies, S_cur, S_next, S_vgprev, loads, dt, nbatch, maps);
    return cudaGetLastError();
}

cudaError_t launch_advance(const BodyDev* bodies, const double* loads, double dt, long long n,
                           int nbatch, StepMaps* maps, cudaStream_t s) {
    k_advance<<<(nbatch + 127) / 128, 128, 0, s>>>(bodies, loads, dt, n, nbatch, maps);
    return cudaGetLastError();
}

}  // namespace lbfsi
