// Internal declarations shared by the kernels and the C-ABI layer.
#pragma once

#include <utility>
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>

namespace lbfsi {

// Status bits written by the kernels (OR-ed into a device word).
enum : unsigned {
    ST_DEPARTURE = 1u,   // departure point outside the adjacent cells
    ST_NONPHYS = 2u,     // rho <= 0, T <= 0 or NaN
    ST_BPOINT = 4u,      // wall or outlet target point B outside the cells next to its node
    ST_BOUNDS = 8u,      // bounds-checked build: an index outside its buffer (access skipped)
    ST_TMA = 16u,        // a tensor-copy wait of the step ran out of iterations
};

// Body model with dimensional ODE coefficients (Sec. III, Sec. IV).
struct BodyDev {
    int dof;                 // 0 fixed, 1 transverse, 2 pitch-plunge
    double xc, yc, xp, yp;   // blend centre, reference point
    double r_in, r_out, inv_w;   // blend radii, 1 / (r_out - r_in)
    double m, k, c;          // transverse: m h'' + c h' + k h = F_y
    double s_a, i_a, k_h, k_a;  // pitch-plunge: [m S; S I] y'' + diag(k_h, k_a) y = [F_y; M]
    double pitch_amp, w_a, t_forced;  // forced pitch amp sin(w_a t) while (n + 1) dt <= t_forced
};

struct BodyStateDev {
    double h, alpha, hdot, adot;
};

// The increment of one RK4 step of a body over the flow's dt under a held load
// (Sec. III B) as the linear map it is: row r of free gives that of state entry r
// from (h, alpha, hdot, adot, F_y, M); forced gives those of (h, hdot) of a step
// in the forcing interval from (h, hdot, F_y, alpha'' at the step's start, middle
// and end).  The increment, not the state: it is some hundredths of the state, so
// the state's own rounding is the addition's alone (as a whole map its products
// rounded it again, and 1 / dt carries that into the mesh velocity).
struct BodyProp {
    double free[4][6], forced[2][6];
};

// Per-row and per-column geometry of the O-grid X = centre + r_i e_j (see
// the table builder in lbfsi_api.cu for the meaning of each entry).
// Entries are grouped in fours so that a kernel reads each group with one
// 16-byte load.
constexpr int ROWTAB = 8;
constexpr int COLTAB = 16;
// row i: [0..3] xi of the node and 1 / (dR/dxi) in the cells i-1 and i
// (element coordinates), [4] r_i, [5] 1 / (dr/dxi) at the node (centred),
// [6] 1 / r_i, [7] unused
enum : int { RT_XIN0 = 0, RT_IDR0 = 1, RT_XIN1 = 2, RT_IDR1 = 3, RT_R = 4, RT_IDRC = 5, RT_IR = 6 };
// column j: [0..3] (de_y, e_y, de_x, e_x) / (e x de) with de the centred
// difference of the direction vectors (inverse metric), [4..5] e_j, [6..7]
// unused, [8..11] and [12..15] for the cells j-1 and j: eta of the node,
// dE/deta (x, y) and dE x e_j
enum : int { CT_G = 0, CT_E = 4, CT_C0 = 8, CT_C1 = 12 };

// Blended rigid map of one body for one body state (defined in
// lbfsi_device.cuh); declared here so the per-step record can hold it.
template <typename R>
struct BodyMap {
    int active;
    R xc, yc, xp, yp, r_in, inv_w;
    R a00, a01, a10, a11, tx, ty;
    R va00, va01, va10, va11, vtx, vty;
};

// Per-solve record handed from one launch to the next: the body state of the
// last streamed step (used by the next collision), the state and previous
// state for the next stream (V_G), the loads of the last streamed step and
// the blended maps built from those states.
struct StepMaps {
    BodyStateDev S_cur, S_next, S_vgprev;
    double loads[3];
    BodyMap<double> Kd, Sd;
    BodyMap<float> Kf, Sf;
};

// Mirrored rows kept below row 0 of a C-grid (the moments' halo).
constexpr int CGRID_GHOST_ROWS = 4;
// Classes of a C-grid's row-0 columns: on the cut, on a wall chain, a
// junction (a chain's end next to the cut, one point with its mirror), a
// second copy of the mirrored column's node (past the middle of row 0), and
// for a junction whether its cut neighbour is the next column (else the
// previous one).
enum : int { CT_CUT = 1, CT_WALL = 2, CT_JUNC = 4, CT_DUP = 8, CT_JFWD = 16 };
// A wall column's body (C-grids with independent bodies): bits from
// CT_BODY_SHIFT of its class.  At most MAX_BODIES bodies per solve.
constexpr int MAX_BODIES = 4;
enum : int { CT_BODY_SHIFT = 5 };

// Geometry of one O-grid mesh shape, shared by every solve on it (device).
struct MeshDev {
    int nr, nt, N, ntj;            // N: node slots per field component (nr nt, plus the
                                   // mirrored rows of a C-grid)
    double xm, ym;                 // mesh centre
    const double* r;               // [nr]
    const double* e;               // [nt][2]
    const double* n0;              // [nt][2] wall normals (undeformed)
    const double* wall_share;      // [nt][2] a wall node's Simpson share of its edges: sum of weight
                                   // times length times unit normal (undeformed)
    const void* rowtab;            // [nr][ROWTAB] per-row geometry (element type of the path)
    const void* coltab;            // [nt][COLTAB] per-column geometry
    float xm_f, ym_f;
    double emin;                   // separable O-grid: min over j of |e_j| (static-tile test)
    float emin_f;
    const double* xw;              // [nt][2] wall node coordinates
    const double* fardir;          // [nt][2] outward unit direction at the far-field row
    // general meshes (node coordinates given): element type of the path
    int general;
    const void* nodex;             // [N][2] node coordinates
    const void* jinv;              // [N][4] inverse metric (index derivatives -> d/dX, d/dY)
    const void* cellc;             // [(nr-1) nt][8] element coefficients per cell
    // C-grid (general meshes only): the node, metric and cell arrays and every
    // field component hold mirrored rows -4..-1 below row 0 (their pointers
    // point at row 0); coltype classes the row-0 columns (CT_*); columns 0
    // and nt-1 are outlets
    int cgrid;
    const int* coltype;            // [nt]
    const double* fardirj;         // [nr][2][2] outward unit directions of columns 0 and nt-1
    // doubly periodic box (general meshes only): rows wrap like columns,
    // every node is interior (no wall, no far field)
    int box;
};

// One solve (one set of fields on one mesh and its bodies: nbody > 1 only on
// general meshes, where the maps, body and load-partial arrays hold nbody
// consecutive records).  Buffers are
// ping-pong pairs; which one holds the current state follows from the solve's
// step number k (counter[1]): after k step launches the state is in buffer
// k & 1, and the launch with k == 0 streams from the initial (post-collision)
// state without colliding.  counter[0] counts the CTAs of the solve that have
// finished a step launch that reads k from the device (the last one resets it
// and writes k + 1), counter[2] its finished loads blocks (the last one
// advances the bodies).
struct SolveDev {
    int mesh;
    int ntiles;                    // CTAs of this solve in every step launch
    int nbody = 1;                 // bodies (maps / body records per solve)
    // flow (float64 and float copies, so that no thread of the float path
    // converts or divides in float64)
    double dt, mu, Cv, Pr, rho_inf, uinf_x, uinf_y, T_inf;
    float dt_f, mu_f, Cv_f, Pr_f, iPr_f, rho_inf_f, uinf_x_f, uinf_y_f, T_inf_f, pad_f;
    // float path: the free-stream equilibrium pairs (f_q, g_q), q = 0..8.  The
    // step interpolates deviations from them, so that the round-off of the
    // float Q2 weights (their sum is 1 only to within an ulp, the same way
    // every step at a node that does not move) scales with the deviation, not
    // with the population
    float fgref[18];
    float mref[4];   // its moments: rho, rho u_x, rho u_y, 2 rho E
    void* p[2];                    // populations, (f_q, g_q) pairs [9][N] (float64: both the one
                                   // buffer of the state, ppost the other)
    void* M[2];                    // moments [4][N]
    StepMaps* maps[2];             // [nbody] each
    void* ppost;                   // post-collision pairs [9][N] (float64 path: written by the field
                                   // launch, read by the stream; float: only for the accessor)
    void* Y;                       // float path: correction field [2][N] of the current state
    double* part;                  // [nbody][ntj][3] load partials of the streamed step
    unsigned* counter;             // [4]: CTA count of the step launch, step number k, loads
                                   // blocks done, unused
    const BodyDev* body;           // [nbody]
    const BodyProp* prop;          // [nbody]
    double iCv, idt, iPr, muP;     // 1 / Cv, 1 / dt, 1 / Pr, mu / Pr
    float iCv_f, muP_f;
    // general meshes and float64, uniform launches: departure points of the nodes the
    // blend does not move (g = I, V_G = 0, so the displacement of direction q
    // is -dt c_q for every step): (xi, eta) pairs [9][N] in the element type
    // of the path and per node a code [N] (5 bits per direction: the window
    // origin relative to the node, row and column offsets in -3..0, or a lost
    // departure; all ones: not cached), shared by the solves of the handle
    // (one mesh, one dt), or null
    void* dep_xe = nullptr;
    unsigned long long* dep_code = nullptr;
};

// One CTA of a step launch: a tile of one solve.  The entry repeats the
// solve's counter and maps pointers so that a CTA can read its step number
// and fetch its maps without first loading the solve record.  tma: stage the
// tile's populations and Y by tensor copies (StepArgs::tmaps).
struct TileDev {
    int solve, mesh, i0, j0, tma;
    unsigned* counter;
    StepMaps* maps[2];
};

struct StepArgs {
    MeshDev umesh;                 // uniform launch: the mesh
    SolveDev usol;                 // uniform launch: solve 0 (others by stride)
    const MeshDev* meshes;
    const SolveDev* solves;
    const TileDev* tiles;
    int ntiles;
    int ustep;                     // uniform launch: the solves' step number (they advance
                                   // together), or -1 to read it from the device counters
    int uorder;                    // uniform launch: CTA order, 0 = (tile column, tile row,
                                   // solve), 1 = (solve, tile column, tile row)
    int record;                    // general meshes, uniform: fill usol.dep_* (departures of
                                   // the static nodes of solve 0) and write nothing else
    unsigned* status;
    // uniform launch of the float kernel: stage the populations and Y of a
    // tile whose columns do not wrap by two tensor copies (TMA) into shared
    // memory instead of per-thread copies.  tm_p[c] describes population
    // buffer c (c = k & 1) of all solves as a 4-D float array (2 nt, nr, 9,
    // nbatch) with boxes (2 (TJ + 8), TI + 4, 9, 1), tm_Y the correction field
    // as (nt, nr, 2, nbatch) with boxes (TJ + 8, TI + 4, 2, 1) (lbfsi_api.cu).
    int tma;
    // table launch of the float separable kernel: per solve the tensor maps of
    // its populations (buffers 0, 1) and of Y, in device memory, [solve][4]
    // (the last unused), each an array of one solve with the boxes above;
    // used by the tiles whose TileDev::tma is set
    const CUtensorMap* tmaps;
    alignas(64) CUtensorMap tm_p[2];
    alignas(64) CUtensorMap tm_Y;
};

// One block of a table launch of the field kernel: block number 'block' of a
// solve's fields, or (fields == 0) of its loads.
struct FieldTile {
    int solve, mesh, fields, block;
};

// Field launch (lbfsi_fields.cu): the loads of the step that produced the
// current state (loads) and the current state's correction field, in float64
// its collision (fields).
struct FieldArgs {
    MeshDev umesh;                 // uniform launch: the mesh and solve 0
    SolveDev usol;
    const MeshDev* meshes;         // table launch
    const SolveDev* solves;
    const FieldTile* tiles;
    int ntiles;
    int uniform, nbatch;
    int nfield;                    // uniform: field blocks per solve (set by the launcher)
    int loads, fields;
    int ustep;                     // uniform: the current state's step number, or -1 (device counters)
    double* rec;                   // uniform: this step's records [nbatch][nbody][7] (Fx, Fy, M, h,
                                   // alpha, hdot, adot), or null
    unsigned* status;
};
// Blocks of a solve: of its fields and of its loads.
int field_blocks(int precision, bool general, int nr, int nt);
int load_blocks(int ntj);
cudaError_t launch_fields(FieldArgs a, int precision, bool general, cudaStream_t s);
// Post-collision populations of the current state of a float handle into
// ppost, from its Y.
cudaError_t launch_post(const SolveDev& S, const MeshDev& G, int cur, int nbatch, cudaStream_t s);

// The step launch's tile shape is chosen by variant (see tile_rows).

// Tensor map of a float array of dims (dx, dy, dz, dw), x fastest and dense,
// read in boxes of (bx, by, bz, 1), elements outside the array as zeros;
// false if the map cannot be made (defined in lbfsi_api.cu).
bool encode_box4(CUtensorMap* map, void* base, size_t dx, size_t dy, size_t dz, size_t dw, unsigned bx,
                 unsigned by, unsigned bz);

// Record msg as the calling thread's last error and return code (defined in
// lbfsi_api.cu).
int set_error(int code, const std::string& msg);

// Launchers (defined in lbfsi_step.cu).  variant selects the tile shape of
// the step kernel (see tile_rows): five float shapes on separable meshes, one
// on general meshes, float64 blocks of 1, 2 or 4 rows.  Table launch (the batch
// runtime) of the separable or the general-geometry kernel:
cudaError_t launch_step(const StepArgs& a, int precision, bool general, int variant, cudaStream_t s);
// Uniform launch over nbatch solves of one mesh (see StepArgs).
cudaError_t launch_step_uniform(const StepArgs& a, int precision, int variant, int nbatch,
                                cudaStream_t s);
int default_shape(int precision, long long tiles16);
int default_shape_general(bool tma, bool moving, long long tiles16);
int default_order(bool tma, bool general, long long nodes, long long tiles16);
int tile_rows(int precision, int variant);
// Stream launch of the float64 path (lbfsi_stream64.cu): blocks of 'rows' rows
// x 32 columns, each row by four warps that share the directions.
cudaError_t launch_stream64(const StepArgs& a, bool uniform, bool general, int rows, int nbatch, cudaStream_t s);
// Tile rows of the general-geometry kernel (float: default_shape_general).
inline int general_tile_rows(int precision, int variant) {
    return precision == 0 ? tile_rows(0, variant) : variant == 0 ? 8 : 16;
}
// Number of tile shapes of the step kernel of a precision (variants 0 .. n-1).
int step_variants(int precision);
// One-time configuration of a step kernel (shared-memory limit, occupancy);
// done by the first launch, and by this call before a stream capture.
cudaError_t prepare_step(int precision, int variant, bool uniform, bool general = false);
constexpr int TILE_J = 32;
inline int tiles_j(int nt) { return (nt + TILE_J - 1) / TILE_J; }
cudaError_t launch_init(int precision, const double* M, void* P, void* Mout, int N, int nbatch,
                        double Cv, cudaStream_t s);
// The kernels of a step are launched while the one before still runs
// (programmatic stream serialization) and wait for its end and its writes
// themselves, first thing (wait_previous): a launch's start -- some 2 to 3 us
// behind the end of the last, a tenth to a quarter of a small mesh's step --
// then overlaps the previous kernel's last wave.  Float: every launch (measured
// per step: 256 x 128 one solve 25.1 -> 22.1 us, 201 x 150 x 5 32.4 -> 29.2,
// ellipse 512 x 256 x 8 132 -> 127).  Float64: launches of few blocks only, which
// find SMs of their own (24 x 32: 91.5 -> 87.9 us); more of them are packed
// beside the running kernel's on some SMs, whose float64 rate then bounds the
// step while others idle (128 x 64: 47.4 -> 59.4 us, a 97 x 161 C-grid 106 -> 120).
// The line is on the safe side: with the overlap and without, by blocks of the
// stream launch, 76: 43.0 and 47.2 us; 160: 44.9 and 47.8; 200: 46.3 and 47.2; by
// coordinates 128: 50.4 and 53.3, 192: 54.4 and 54.6; 256 (128 x 64) the other way.
constexpr unsigned OVERLAP_BLOCKS_FP64 = 76;   // half the SMs
template <typename... P, typename... A>
cudaError_t launch_behind(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, bool overlap,
                          A&&... args) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = overlap ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);
    if (e != cudaSuccess) cudaGetLastError();
    return e;
}

// rows x N values of the path's type, rows stride apart, as float64 [rows][N] in
// the order given (null: as they lie)
cudaError_t launch_read(int precision, const void* src, size_t stride, const int* order, double* dst, int N, size_t rows,
                        cudaStream_t s);
// Build the maps record from explicit states: S_cur (collision), S_next and
// S_vgprev (stream); loads copied from 'loads' if non-null.
cudaError_t launch_prepare(const BodyDev* bodies, const BodyStateDev* S_cur,
                           const BodyStateDev* S_next, const BodyStateDev* S_vgprev,
                           const double* loads, double dt, int nbatch, StepMaps* maps,
                           cudaStream_t s);
// RK4 of every body over dt with the given loads from maps->S_next; the
// result becomes S_next and the old S_next S_vgprev and S_cur.
cudaError_t launch_advance(const BodyDev* bodies, const double* loads, double dt, long long n,
                           int nbatch, StepMaps* maps, cudaStream_t s);

}  // namespace lbfsi
