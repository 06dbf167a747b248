// C-ABI of the library (declared in include/lbfsi.h): the mesh handle (one
// O-grid, nbatch independent solves advanced together), its device memory and
// the launch sequence of the coupled step.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <string>
#include <vector>

#include "lbfsi.h"
#include "lbfsi_host.h"
#include "lbfsi_internal.h"

using lbfsi::BodyDev;
using lbfsi::BodyStateDev;
using lbfsi::SolveDev;
using lbfsi::StepMaps;
using lbfsi::TileDev;

namespace lbfsi {

// cuTensorMapEncodeTiled through the runtime's driver entry point (no link
// against the driver library)
using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled() {
    static const EncodeTiledFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q{};
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            return static_cast<EncodeTiledFn>(nullptr);
        }
        return reinterpret_cast<EncodeTiledFn>(p);
    }();
    return fn;
}

// A float array of dims (dx, dy, dz, dw), x fastest and dense, read in boxes
// of (bx, by, bz, 1); elements outside the array arrive as zeros.
bool encode_box4(CUtensorMap* map, void* base, size_t dx, size_t dy, size_t dz, size_t dw, unsigned bx,
                 unsigned by, unsigned bz) {
    const EncodeTiledFn fn = encode_tiled();
    if (!fn) return false;
    const cuuint64_t dims[4] = {dx, dy, dz, dw};
    const cuuint64_t strides[3] = {dx * 4, dx * dy * 4, dx * dy * dz * 4};   // bytes, dims 1..3
    const cuuint32_t box[4] = {bx, by, bz, 1};
    const cuuint32_t estr[4] = {1, 1, 1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
              CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace lbfsi

namespace {

thread_local std::string g_last_error;

int fail(int code, const std::string& msg) {
    g_last_error = msg;
    return code;
}

int cuda_fail(cudaError_t e, const char* where) {
    return fail(LBFSI_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

}  // namespace

int lbfsi::set_error(int code, const std::string& msg) { return fail(code, msg); }

struct lbfsi_mesh_s {
    lbfsi::HostMesh host;
    lbfsi::DeviceMesh dmesh;
    lbfsi::CudaMallocMemory mem;
    int nbatch = 0, precision = 0, variant = 4, order = 1, tile_rows = 16, tiles_per_solve = 0;
    bool own_shape = true, own_order = true;   // no schedule asked for: the shape and the order follow the size
    int shape = 4, launch_order = 1;     // what is launched (set_shape)
    // the step whose correction field (float64: and post-collision populations)
    // the last call left behind its last step, or -1; and the step at which the
    // last call ended, or -1 once anything changed the state since
    long long fields_of = -1, ended_at = -1;
    bool handed_out = false;   // a field's device address: what is written there between calls counts
    int nbody = 1;                       // bodies per solve (independent bodies of a C-grid)
    size_t slots() const { return (size_t)nbatch * (size_t)nbody; }   // body records
    size_t esize = 8;
    cudaStream_t stream = nullptr;
    std::vector<lbfsi_body_desc> bodies;
    void* d_p[2] = {nullptr, nullptr};   // populations, (f_q, g_q) pairs [nbatch][9][N]: float a
                                         // ping-pong pair; float64 the post-collision ones and the state
    void* d_M[2] = {nullptr, nullptr};
    void* d_ppost = nullptr;             // float: post-collision populations, same layout (made when
                                         // the accessor asks)
    void* d_Y = nullptr;                 // float: correction field [nbatch][2][N] (where the device has
                                         // no room for it, in d_stage, which is idle but for transfers)
    void* d_dep = nullptr;               // general meshes, float64: cached static departures ((xi, eta)
                                         // [9][Nx], then codes [Nx]; see SolveDev::dep_xe)
    double* d_stage = nullptr;  // [nbatch][4][N] float64 staging
    // pinned copies of the records and the status word for the small reads
    // between steps (null: could not be had, the reads go to pageable memory)
    StepMaps* h_maps = nullptr;
    unsigned* h_status = nullptr;
    std::mutex reading;         // held by a read from its first copy until it has taken its values out
    StepMaps* d_maps[2] = {nullptr, nullptr};  // [nbatch][nbody] each
    BodyStateDev* d_state_a = nullptr;          // host-given states staging
    BodyStateDev* d_state_b = nullptr;
    double* d_loads_tmp = nullptr;
    double* d_part = nullptr;        // [nbatch][nbody][ntj][3] load partials
    unsigned* d_counter = nullptr;   // [nbatch][4] (SolveDev::counter)
    BodyDev* d_bodies = nullptr;     // [nbatch][nbody]
    lbfsi::BodyProp* d_prop = nullptr;   // [nbatch][nbody]
    lbfsi::MeshDev* d_meshdev = nullptr;
    SolveDev* d_solves = nullptr;    // [nbatch]
    unsigned* d_status = nullptr;
    std::vector<SolveDev> solves;
    unsigned host_k = 0;             // step number of every solve (mirror of counter[1])
    bool initialized = false;
    double dt = 0;
    int64_t launches = 0;
    // CUDA graph of graph_steps step launches (step number from the device
    // counters), captured on a private stream and replayed on 'stream'
    int graph_steps = 0;
    cudaGraphExec_t graph = nullptr;
    int64_t graph_launches = 0;
    cudaStream_t cap_stream = nullptr;
    // pinned staging of lbfsi_step_record
    void* h_rec = nullptr;
    size_t h_rec_bytes = 0;
    double* d_rec = nullptr;         // device history of lbfsi_step_record: [steps][records][7]
    size_t d_rec_count = 0;
    // tensor maps of the float step (StepArgs::tm_p, tm_Y) for tiles of
    // tma_rows rows: -1 not built yet, 0 not used (float64, C-grids, periodic
    // boxes, Ntheta not a multiple of 4, LBFSI_TMA=0, or no encoder)
    int tma_rows = -1;
    CUtensorMap tm_p[2], tm_Y;

    int cur() const { return (int)(host_k & 1u); }
    bool first() const { return host_k == 0u; }
    void* pops() const { return d_p[precision == LBFSI_FP64 ? 1 : cur()]; }   // the state's populations
    void changed() { fields_of = ended_at = -1; }   // the state, other than by steps
};

namespace {

template <typename T>
cudaError_t dalloc(T** p, size_t count) {
    return cudaMalloc(reinterpret_cast<void**>(p), count * sizeof(T));
}

int status_code(unsigned st) {
    if (st & lbfsi::ST_BOUNDS)
        return lbfsi::set_error(LBFSI_EBOUNDS, "an index of the step outside its buffer (bounds-checked build)");
    if (st & lbfsi::ST_TMA)
        return lbfsi::set_error(LBFSI_ECUDA, "a tensor copy of the step did not complete within its wait limit");
    if (st & lbfsi::ST_DEPARTURE)
        return fail(LBFSI_EDEPARTURE, "departure point outside the cells adjacent to its node (CFL)");
    if (st & lbfsi::ST_BPOINT)
        return fail(LBFSI_EDEPARTURE, "wall or outlet target point B outside the cells next to its node");
    if (st & lbfsi::ST_NONPHYS) return fail(LBFSI_ENONPHYS, "non-physical state (rho<=0, T<=0 or NaN)");
    return LBFSI_OK;
}

// The status word behind the stream's work (and the records, whose copy was
// enqueued before): one copy into pinned memory, one wait.  The caller holds
// 'reading'.
int read_status(lbfsi_mesh m) {
    unsigned own = 0, *st = m->h_status ? m->h_status : &own;
    cudaError_t e = cudaMemcpyAsync(st, m->d_status, sizeof(unsigned), cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "status read");
    return status_code(*st);
}

int check_status(lbfsi_mesh m) {
    std::lock_guard<std::mutex> hold(m->reading);
    return read_status(m);
}

void to_double(const void* src, double* dst, size_t n, int precision) {
    if (precision == LBFSI_FP64) {
        std::memcpy(dst, src, n * sizeof(double));
    } else {
        const float* s = static_cast<const float*>(src);
        for (size_t k = 0; k < n; ++k) dst[k] = (double)s[k];
    }
}

int download(lbfsi_mesh m, const void* dsrc, double* host, size_t n) {
    std::vector<unsigned char> tmp(n * m->esize);
    cudaError_t e = cudaMemcpyAsync(tmp.data(), dsrc, n * m->esize, cudaMemcpyDeviceToHost, m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "download");
    e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "download sync");
    to_double(tmp.data(), host, n, m->precision);
    return LBFSI_OK;
}

int upload(lbfsi_mesh m, const double* host, void* ddst, size_t n) {
    std::vector<unsigned char> tmp(n * m->esize);
    if (m->precision == LBFSI_FP64) {
        std::memcpy(tmp.data(), host, n * sizeof(double));
    } else {
        float* t = reinterpret_cast<float*>(tmp.data());
        for (size_t k = 0; k < n; ++k) t[k] = (float)host[k];
    }
    cudaError_t e = cudaMemcpyAsync(ddst, tmp.data(), n * m->esize, cudaMemcpyHostToDevice, m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "upload");
    e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "upload sync");
    return LBFSI_OK;
}

// Field blocks of w values per node: the caller's [blocks][N] layout to the
// device's [blocks][Nx] (a C-grid's mirrored rows below row 0 filled from
// their nodes, node (-k, j) = node (k, nt-1-j)), and back.
std::vector<double> expand_rows(const lbfsi::HostMesh& h, const double* user, size_t blocks, int w) {
    const size_t N = (size_t)h.N, Nx = (size_t)h.Nx, nt = (size_t)h.nt, g0 = (size_t)h.G * nt;
    std::vector<double> dev(blocks * Nx * w);
    for (size_t b = 0; b < blocks; ++b) {
        const double* u = user + b * N * w;
        double* d = dev.data() + b * Nx * w;
        std::memcpy(d + g0 * w, u, N * w * sizeof(double));
        for (int k = 1; k <= h.G; ++k)
            for (size_t j = 0; j < nt; ++j)
                for (int c = 0; c < w; ++c)
                    d[(g0 - k * nt + j) * w + c] = u[(k * nt + (nt - 1 - j)) * w + c];
    }
    return dev;
}

void compact_rows(const lbfsi::HostMesh& h, const double* dev, double* user, size_t blocks, int w) {
    const size_t N = (size_t)h.N, Nx = (size_t)h.Nx, g0 = (size_t)h.G * h.nt;
    for (size_t b = 0; b < blocks; ++b)
        std::memcpy(user + b * N * w, dev + (b * Nx + g0) * w, N * w * sizeof(double));
}

// A C-grid's second copies of the row-0 cut nodes (and of the rear point)
// take the first copies' values in caller-given fields of w values per node.
void unify_cut_copies(const lbfsi::HostMesh& h, double* user, size_t blocks, int w) {
    if (!h.cgrid) return;
    for (size_t b = 0; b < blocks; ++b)
        for (int j = 0; j < h.nt; ++j)
            if (h.coltype[j] & lbfsi::CT_DUP)
                for (int c = 0; c < w; ++c)
                    user[(b * h.N + (size_t)j) * w + c] = user[(b * h.N + (size_t)(h.nt - 1 - j)) * w + c];
}

lbfsi::StepArgs make_args(lbfsi_mesh m);

// Float meshes whose tiles are staged by tensor copies (LBFSI_TMA aside).
bool tma_mesh(const lbfsi::HostMesh& h) { return !h.box && !h.cgrid && h.nt % 4 == 0; }

// Tile shape, rows and tiles and the CTA order of the handle's schedule or, as
// long as none was asked for, by its size.
void set_shape(lbfsi_mesh m) {
    const lbfsi::HostMesh& h = m->host;
    const long long tiles16 = (long long)m->nbatch * h.ntj * ((h.nr + 15) / 16);
    const bool tma = tma_mesh(h);
    bool moving = false;
    for (const lbfsi_body_desc& b : m->bodies) moving = moving || b.dof != LBFSI_BODY_FIXED;
    m->shape = !m->own_shape ? m->variant
               : m->precision == LBFSI_FP32 && h.general ? lbfsi::default_shape_general(tma, moving, tiles16)
                                                         : lbfsi::default_shape(m->precision, tiles16);
    // (the third dimension of a grid, here the solves, has 16 bits)
    m->launch_order = m->own_order && m->nbatch <= 65535 ? lbfsi::default_order(tma, h.general, (long long)m->nbatch * h.N, tiles16)
                                                         : m->order;
    m->tile_rows = m->host.general ? lbfsi::general_tile_rows(m->precision, m->shape)
                                   : lbfsi::tile_rows(m->precision, m->shape);
    m->tiles_per_solve = ((m->host.nr + m->tile_rows - 1) / m->tile_rows) * m->host.ntj;
}

// Field launch (lbfsi_fields.cu) on the current state of every solve.
cudaError_t launch_fields(lbfsi_mesh m, const lbfsi::StepArgs& a, int loads, int fields, int ustep, double* rec,
                          cudaStream_t s) {
    lbfsi::FieldArgs f{};
    f.umesh = a.umesh;
    f.usol = a.usol;
    f.uniform = 1;
    f.nbatch = m->nbatch;
    f.loads = loads;
    f.fields = fields;
    f.ustep = ustep;
    f.rec = rec;
    f.status = m->d_status;
    return lbfsi::launch_fields(f, m->precision, m->host.general, s);
}

// n coupled steps of every solve on stream s, two launches per step: the
// fields of the current state; then per step the step launch and the field
// launch behind it (the step's loads and bodies, and the next step's fields).
// A call that follows another with the state unchanged also leaves the fields of
// its last state to the next, which takes them over, one launch less, if it too
// follows unchanged: a run of one call, and calls with the state or the bodies
// set in between, form no field that nobody takes (8192 x 512: a fresh run of
// two steps 502 -> 465 us, blend_mesh and one step 289 -> 252).  With a field's
// address handed out every call forms them anew; so does one that a caller's
// stream captures, which may be replayed behind anything.
// rec: device history of the steps' records, or null.
// host_step < 0: the step numbers come from the device counters.
cudaError_t launch_steps(lbfsi_mesh m, int n, long long host_step, double* rec, cudaStream_t s, int64_t* launches) {
    if (n <= 0) return cudaSuccess;
    lbfsi::StepArgs a = make_args(m);
    const bool host = host_step >= 0;
    cudaError_t e = cudaSuccess;
    // (an error, on the legacy stream beside another's capture, comes back from the launches)
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (host && cudaStreamIsCapturing(s, &st) != cudaSuccess) cudaGetLastError();
    const bool keep = host && st == cudaStreamCaptureStatusNone;
    const bool carry = keep && !m->handed_out && m->ended_at == host_step, have = carry && m->fields_of == host_step;
    m->changed();
    // (the initial state is streamed without colliding; float64 copies it)
    if (!have && (!host || host_step > 0 || m->precision == LBFSI_FP64)) {
        e = launch_fields(m, a, 0, 1, host ? (int)host_step : -1, nullptr, s);
        ++*launches;
    }
    for (int k = 0; k < n && e == cudaSuccess; ++k) {
        a.ustep = host ? (int)(host_step + k) : -1;
        e = lbfsi::launch_step_uniform(a, m->precision, m->shape, m->nbatch, s);
        if (e == cudaSuccess)
            e = launch_fields(m, a, 1, carry || k + 1 < n, host ? (int)(host_step + k + 1) : -1,
                              rec ? rec + (size_t)k * m->slots() * 7 : nullptr, s);
        *launches += 2;
    }
    if (keep && e == cudaSuccess) {
        m->ended_at = host_step + n;
        if (carry) m->fields_of = m->ended_at;
    }
    return e;
}

void free_all(lbfsi_mesh m) {
    void* ptrs[] = {m->d_p[0], m->d_p[1], m->d_M[0], m->d_M[1], m->d_ppost, m->d_Y == m->d_stage ? nullptr : m->d_Y, m->d_dep, m->d_stage, m->d_maps[0], m->d_maps[1], m->d_state_a, m->d_state_b,
                    m->d_loads_tmp, m->d_part, m->d_counter, m->d_bodies, m->d_prop, m->d_meshdev, m->d_solves,
                    m->d_status};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    if (m->graph) cudaGraphExecDestroy(m->graph);
    if (m->cap_stream) cudaStreamDestroy(m->cap_stream);
    if (m->h_rec) cudaFreeHost(m->h_rec);
    if (m->h_maps) cudaFreeHost(m->h_maps);
    if (m->d_rec) cudaFree(m->d_rec);
    lbfsi::release_mesh(m->dmesh, m->mem);
}

// Per-solve descriptors of the handle: solve b's buffers are slices of the
// batch-contiguous arrays.
int upload_solves(lbfsi_mesh m) {
    // field pointers at row 0 of solve b (a C-grid's mirrored rows before it)
    const size_t N = (size_t)m->host.Nx, es = m->esize, g0 = (size_t)m->host.G * m->host.nt;
    for (int b = 0; b < m->nbatch; ++b) {
        SolveDev& s = m->solves[b];
        s.mesh = 0;
        s.ntiles = m->tiles_per_solve;
        s.nbody = m->nbody;
        const size_t bb = (size_t)b * m->nbody;
        for (int p = 0; p < 2; ++p) {
            s.p[p] = (char*)m->d_p[m->precision == LBFSI_FP64 ? 1 : p] + ((size_t)b * 18 * N + 2 * g0) * es;
            s.M[p] = (char*)m->d_M[p] + ((size_t)b * 4 * N + g0) * es;
            s.maps[p] = m->d_maps[p] + bb;
        }
        char* post = (char*)(m->precision == LBFSI_FP64 ? m->d_p[0] : m->d_ppost);
        s.ppost = post ? post + ((size_t)b * 18 * N + 2 * g0) * es : nullptr;
        s.Y = m->d_Y ? (char*)m->d_Y + ((size_t)b * 2 * N + g0) * es : nullptr;
        s.part = m->d_part + bb * m->host.ntj * 3;
        s.counter = m->d_counter + 4 * b;
        s.body = m->d_bodies + bb;
        s.prop = m->d_prop + bb;
        s.dep_xe = m->d_dep ? (char*)m->d_dep + g0 * 2 * es : nullptr;
        s.dep_code = m->d_dep ? reinterpret_cast<unsigned long long*>((char*)m->d_dep + 9 * N * 2 * es) + g0
                              : nullptr;
    }
    cudaError_t e = cudaMemcpyAsync(m->d_solves, m->solves.data(), m->solves.size() * sizeof(SolveDev),
                                    cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "solve descriptors upload");
    return LBFSI_OK;
}

// Tensor maps of the handle's two population buffers and its correction
// field for its current tile shape (built again after a schedule change);
// false where the step stages by per-thread copies.  Populations: (f, g) float
// pairs as (2 Ntheta, nr, 9, nbatch) floats, box (2 (32 + 8), rows + 4, 9, 1);
// Y: (Ntheta, nr, 2, nbatch), box (32 + 8, rows + 4, 2, 1) -- the staged tiles
// of the step kernel (+-2 rows and -4 .. +4 columns around the tile).
bool tma_maps(lbfsi_mesh m) {
    if (m->tma_rows == m->tile_rows) return true;
    if (m->tma_rows == 0) return false;
    const char* env = std::getenv("LBFSI_TMA");
    bool ok = m->precision == LBFSI_FP32 && tma_mesh(m->host) && !(env && std::atoi(env) == 0);
    const size_t nt = (size_t)m->host.nt, nr = (size_t)m->host.nr, nb = (size_t)m->nbatch;
    const unsigned rows = (unsigned)m->tile_rows, w = (unsigned)(lbfsi::TILE_J + 8);
    for (int c = 0; c < 2 && ok; ++c) ok = lbfsi::encode_box4(&m->tm_p[c], m->d_p[c], 2 * nt, nr, 9, nb, 2 * w, rows + 4, 9);
    ok = ok && lbfsi::encode_box4(&m->tm_Y, m->d_Y, nt, nr, 2, nb, w, rows + 4, 2);
    m->tma_rows = ok ? m->tile_rows : 0;
    return ok;
}

lbfsi::StepArgs make_args(lbfsi_mesh m) {
    lbfsi::StepArgs a{};
    if (tma_maps(m)) {
        a.tma = 1;
        for (int c = 0; c < 2; ++c) a.tm_p[c] = m->tm_p[c];
        a.tm_Y = m->tm_Y;
    }
    a.umesh = m->dmesh.dev;
    a.usol = m->solves[0];
    a.meshes = m->d_meshdev;
    a.solves = m->d_solves;
    a.tiles = nullptr;
    a.ntiles = m->nbatch * m->tiles_per_solve;
    a.ustep = (int)m->host_k;
    a.uorder = m->launch_order;
    a.status = m->d_status;
    return a;
}

// Capture graph_steps step launches that take the step number from the
// device counters (so the same graph serves every replay).
int capture_graph(lbfsi_mesh m) {
    lbfsi::TraceRange trace_("lbfsi graph capture");
    cudaError_t e = lbfsi::prepare_step(m->precision, m->shape, true, m->host.general);
    if (e == cudaSuccess && !m->cap_stream) e = cudaStreamCreateWithFlags(&m->cap_stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) return cuda_fail(e, "graph capture setup");
    e = cudaStreamBeginCapture(m->cap_stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return cuda_fail(e, "begin capture");
    m->graph_launches = 0;
    const cudaError_t le = launch_steps(m, m->graph_steps, -1, nullptr, m->cap_stream, &m->graph_launches);
    cudaGraph_t graph = nullptr;
    e = cudaStreamEndCapture(m->cap_stream, &graph);
    if (le != cudaSuccess || e != cudaSuccess) {
        if (graph) cudaGraphDestroy(graph);
        return cuda_fail(le != cudaSuccess ? le : e, "step capture");
    }
    e = cudaGraphInstantiate(&m->graph, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
        m->graph = nullptr;
        return cuda_fail(e, "graph instantiate");
    }
    return LBFSI_OK;
}

void drop_graph(lbfsi_mesh m) {
    if (m->graph) {
        cudaStreamSynchronize(m->stream);
        cudaGraphExecDestroy(m->graph);
        m->graph = nullptr;
    }
}

}  // namespace

extern "C" {

const char* lbfsi_last_error(void) { return g_last_error.c_str(); }

namespace {

int check_common(int nr, int nt, int precision, int nbatch, const lbfsi_body_desc* bodies, lbfsi_mesh* out) {
    if (!out) return fail(LBFSI_EINVAL, "null argument");
    *out = nullptr;
    if (precision != LBFSI_FP64 && precision != LBFSI_FP32)
        return fail(LBFSI_EINVAL, "precision must be LBFSI_FP64 or LBFSI_FP32");
    if (nbatch < 1) return fail(LBFSI_EINVAL, "nbatch must be >= 1");
    if (!bodies) return fail(LBFSI_EINVAL, "null body pointer");
    const long long Nll = (long long)nr * nt;
    if (nr > 0 && nt > 0 && Nll * 9 * nbatch > (1ll << 31))
        return fail(LBFSI_EINVAL, "mesh too large for 32-bit node indexing");
    return LBFSI_OK;
}

int create_common(lbfsi_mesh m, int precision, int nbatch, const lbfsi_body_desc* bodies, void* cuda_stream,
                  lbfsi_mesh* out);

}  // namespace

int lbfsi_create_mesh(const lbfsi_mesh_desc* d, void* cuda_stream, lbfsi_mesh* out) {
    g_last_error.clear();
    if (!d) return fail(LBFSI_EINVAL, "null argument");
    int rc = check_common(d->nr, d->ntheta, d->precision, d->nbatch, d->bodies, out);
    if (rc) return rc;
    auto m = new lbfsi_mesh_s();
    rc = lbfsi::build_host_mesh(d->nr, d->ntheta, d->r, d->e, d->xc, d->yc, m->host);
    if (rc) {
        delete m;
        return rc;
    }
    return create_common(m, d->precision, d->nbatch, d->bodies, cuda_stream, out);
}

int lbfsi_create_mesh_xy(const lbfsi_mesh_xy_desc* d, void* cuda_stream, lbfsi_mesh* out) {
    g_last_error.clear();
    if (!d) return fail(LBFSI_EINVAL, "null argument");
    int rc = check_common(d->nr, d->ntheta, d->precision, d->nbatch, d->bodies, out);
    if (rc) return rc;
    auto m = new lbfsi_mesh_s();
    rc = lbfsi::build_host_mesh_xy(d->nr, d->ntheta, d->X, d->xc, d->yc, m->host);
    if (rc) {
        delete m;
        return rc;
    }
    return create_common(m, d->precision, d->nbatch, d->bodies, cuda_stream, out);
}

int lbfsi_create_mesh_box(const lbfsi_mesh_box_desc* d, void* cuda_stream, lbfsi_mesh* out) {
    g_last_error.clear();
    if (!d) return fail(LBFSI_EINVAL, "null argument");
    int rc = check_common(d->ni, d->nj, d->precision, d->nbatch, d->bodies, out);
    if (rc) return rc;
    auto m = new lbfsi_mesh_s();
    rc = lbfsi::build_host_mesh_box(d->ni, d->nj, d->X, d->shift_i, d->shift_j, m->host);
    if (rc) {
        delete m;
        return rc;
    }
    return create_common(m, d->precision, d->nbatch, d->bodies, cuda_stream, out);
}

int lbfsi_create_mesh_cgrid(const lbfsi_mesh_cgrid_desc* d, void* cuda_stream, lbfsi_mesh* out) {
    g_last_error.clear();
    if (!d) return fail(LBFSI_EINVAL, "null argument");
    int rc = check_common(d->nr + lbfsi::CGRID_GHOST_ROWS, d->ntheta, d->precision, d->nbatch, d->bodies, out);
    if (rc) return rc;
    auto m = new lbfsi_mesh_s();
    const int walls[2] = {d->n_cut, d->ntheta - 1 - d->n_cut};
    rc = lbfsi::build_host_mesh_c(d->nr, d->ntheta, 1, walls, d->X, d->xc, d->yc, m->host);
    if (rc) {
        delete m;
        return rc;
    }
    return create_common(m, d->precision, d->nbatch, d->bodies, cuda_stream, out);
}

int lbfsi_create_mesh_cgrid_walls(const lbfsi_mesh_cgrid_walls_desc* d, void* cuda_stream, lbfsi_mesh* out) {
    g_last_error.clear();
    if (!d) return fail(LBFSI_EINVAL, "null argument");
    int rc = check_common(d->nr + lbfsi::CGRID_GHOST_ROWS, d->ntheta, d->precision, d->nbatch, d->bodies, out);
    if (rc) return rc;
    auto m = new lbfsi_mesh_s();
    const int nbody = d->nbody < 1 ? 1 : d->nbody;
    rc = lbfsi::build_host_mesh_c(d->nr, d->ntheta, d->nwalls, d->walls, d->X, d->xc, d->yc, m->host, nbody,
                                  d->wall_body);
    if (rc) {
        delete m;
        return rc;
    }
    m->nbody = nbody;
    return create_common(m, d->precision, d->nbatch, d->bodies, cuda_stream, out);
}

namespace {

int create_common(lbfsi_mesh m, int precision, int nbatch, const lbfsi_body_desc* bodies, void* cuda_stream,
                  lbfsi_mesh* out) {
    int rc = lbfsi::validate_bodies(m->host, bodies, nbatch);
    if (rc) {
        delete m;
        return rc;
    }
    m->nbatch = nbatch;
    m->precision = precision;
    m->esize = precision == LBFSI_FP64 ? sizeof(double) : sizeof(float);
    m->stream = static_cast<cudaStream_t>(cuda_stream);
    // tile shape of the float kernel (a tuning knob, every variant computes the
    // same result; see lbfsi_step_variants): default 4 with the solve-minor
    // CTA order (the autotuner's choice on a GB300 for batched meshes), or
    // LBFSI_STEP_VARIANT
    m->variant = 4;
    m->order = 1;
    if (const char* v = std::getenv("LBFSI_STEP_VARIANT")) {
        const int k = std::atoi(v);
        m->variant = (k >= 0 && k < lbfsi::step_variants(LBFSI_FP32)) ? k : 4;
        m->own_shape = m->precision == LBFSI_FP64 || m->host.general;
    }
    if (m->precision == LBFSI_FP64 || m->host.general) m->variant = 0;   // (general: the one shape)
    m->bodies.assign(bodies, bodies + m->slots());
    set_shape(m);
    m->solves.assign(m->nbatch, SolveDev{});
    rc = lbfsi::upload_mesh(m->host, m->precision, m->mem, m->stream, m->dmesh);
    if (rc) {
        delete m;
        return rc;
    }
    const size_t N = (size_t)m->host.Nx, nb = (size_t)m->nbatch, ns = m->slots();
    const int ntj = m->host.ntj;
    cudaError_t e = cudaSuccess;
#define LB_ALLOC(ptr, cnt) \
    if (e == cudaSuccess) e = dalloc(&(ptr), (cnt));
    LB_ALLOC(m->d_stage, nb * 4 * N);
    if (cudaMallocHost((void**)&m->h_maps, ns * sizeof(StepMaps) + sizeof(unsigned)) == cudaSuccess) {
        m->h_status = reinterpret_cast<unsigned*>(m->h_maps + ns);
    } else {
        m->h_maps = nullptr;
        cudaGetLastError();
    }
    LB_ALLOC(m->d_maps[0], ns);
    LB_ALLOC(m->d_maps[1], ns);
    LB_ALLOC(m->d_state_a, ns);
    LB_ALLOC(m->d_state_b, ns);
    LB_ALLOC(m->d_loads_tmp, ns * 3);
    LB_ALLOC(m->d_part, ns * ntj * 3);
    LB_ALLOC(m->d_counter, 4 * nb);
    LB_ALLOC(m->d_bodies, ns);
    LB_ALLOC(m->d_prop, ns);
    LB_ALLOC(m->d_meshdev, 1);
    LB_ALLOC(m->d_solves, nb);
    LB_ALLOC(m->d_status, 1);
#undef LB_ALLOC
    for (int k = 0; k < 2 && e == cudaSuccess; ++k) {
        e = cudaMalloc(&m->d_p[k], nb * 18 * N * m->esize);
        if (e == cudaSuccess) e = cudaMalloc(&m->d_M[k], nb * 4 * N * m->esize);
    }
    // (what a step can do without is left out where the device has no room)
    auto spare = [&](void** p, size_t bytes) {
        if (e != cudaSuccess || cudaMalloc(p, bytes) == cudaSuccess) return;
        *p = nullptr;
        cudaGetLastError();
    };
    if (m->precision == LBFSI_FP32) {
        spare(&m->d_Y, nb * 2 * N * m->esize);
        if (!m->d_Y) m->d_Y = m->d_stage;
    }
    // general meshes and float64: departures of the static nodes, solved once
    // per time step size (a float step solves the separable mesh's closed form
    // faster than it reads them; LBFSI_NO_DEPARTURE_CACHE=1, or a device without
    // room for them, solves them every step instead; the results are the same)
    const char* nc = std::getenv("LBFSI_NO_DEPARTURE_CACHE");
    if ((m->host.general || m->precision == LBFSI_FP64) && !(nc && std::atoi(nc) != 0))
        spare(&m->d_dep, 9 * N * 2 * m->esize + N * sizeof(unsigned long long));
    if (e != cudaSuccess) {
        free_all(m);
        delete m;
        cudaGetLastError();
        return fail(LBFSI_ENOMEM, std::string("device allocation failed: ") + cudaGetErrorString(e));
    }
    e = cudaMemcpy(m->d_meshdev, &m->dmesh.dev, sizeof(lbfsi::MeshDev), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemset(m->d_status, 0, sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMemset(m->d_counter, 0, 4 * nb * sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMemset(m->d_part, 0, ns * ntj * 3 * sizeof(double));
    if (e != cudaSuccess) {
        free_all(m);
        delete m;
        return cuda_fail(e, "create_mesh copy");
    }
    *out = m;
    return LBFSI_OK;
}

}  // namespace

int lbfsi_destroy_mesh(lbfsi_mesh m) {
    if (!m) return fail(LBFSI_EINVAL, "null mesh");
    cudaStreamSynchronize(m->stream);
    free_all(m);
    delete m;
    return LBFSI_OK;
}

int lbfsi_init_fields(lbfsi_mesh m, const lbfsi_flow_params* p, const double* rho_u_T) {
    lbfsi::TraceRange trace_("lbfsi_init_fields");
    if (!m || !p) return fail(LBFSI_EINVAL, "null argument");
    SolveDev proto{};
    int rc = lbfsi::fill_flow(*p, proto);
    if (rc) return rc;
    const size_t N = (size_t)m->host.N, nb = (size_t)m->nbatch;
    for (auto& s : m->solves) s = proto;
    m->dt = p->dt;
    const size_t ns = m->slots();
    std::vector<BodyDev> bd(ns);
    for (size_t b = 0; b < ns; ++b) bd[b] = lbfsi::body_dev(m->bodies[b], proto.rho_inf, proto.uinf_x);
    std::vector<lbfsi::BodyProp> prop(ns);
    for (size_t b = 0; b < ns; ++b) prop[b] = lbfsi::body_prop(bd[b], p->dt);
    // the caller's field goes to the device as it is unless the C-grid's
    // rows need rearranging (cut copies unified, mirrored rows added)
    const bool direct = rho_u_T && !m->host.cgrid && !m->host.G;
    std::vector<double> M(direct ? 0 : nb * 4 * N);
    if (direct) {
    } else if (rho_u_T) {
        std::memcpy(M.data(), rho_u_T, M.size() * sizeof(double));
    } else {
        for (size_t b = 0; b < nb; ++b)
            for (size_t n = 0; n < N; ++n) {
                M[(b * 4 + 0) * N + n] = proto.rho_inf;
                M[(b * 4 + 1) * N + n] = proto.uinf_x;
                M[(b * 4 + 2) * N + n] = 0.0;
                M[(b * 4 + 3) * N + n] = proto.T_inf;
            }
    }
    std::vector<BodyStateDev> zero(ns, BodyStateDev{0.0, 0.0, 0.0, 0.0});
    std::vector<double> zl(ns * 3, 0.0);
    if (!direct) unify_cut_copies(m->host, M.data(), nb * 4, 1);
    if (m->host.G) M = expand_rows(m->host, M.data(), nb * 4, 1);
    cudaError_t e = cudaMemcpyAsync(m->d_bodies, bd.data(), ns * sizeof(BodyDev), cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->d_prop, prop.data(), ns * sizeof(lbfsi::BodyProp), cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess)
        e = direct ? cudaMemcpyAsync(m->d_stage, rho_u_T, nb * 4 * N * sizeof(double), cudaMemcpyHostToDevice, m->stream)
                   : cudaMemcpyAsync(m->d_stage, M.data(), M.size() * sizeof(double), cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->d_state_a, zero.data(), ns * sizeof(BodyStateDev), cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->d_loads_tmp, zl.data(), zl.size() * sizeof(double), cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->d_status, 0, sizeof(unsigned), m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->d_counter, 0, 4 * nb * sizeof(unsigned), m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "init_fields upload");
    m->host_k = 0;
    m->changed();
    rc = upload_solves(m);
    if (rc) return rc;
    e = lbfsi::launch_init(m->precision, m->d_stage, m->pops(), m->d_M[0], m->host.Nx, m->nbatch,
                           proto.Cv, m->stream);
    m->launches++;
    if (e != cudaSuccess) return cuda_fail(e, "init kernel");
    e = lbfsi::launch_prepare(m->d_bodies, m->d_state_a, m->d_state_a, m->d_state_a, m->d_loads_tmp, m->dt,
                              (int)ns, m->d_maps[0], m->stream);
    m->launches++;
    if (e != cudaSuccess) return cuda_fail(e, "prepare kernel");
    if (m->d_dep) {
        // the static nodes' departures for this dt (one pass of the step
        // kernel over solve 0 that writes nothing else)
        const size_t Nx = (size_t)m->host.Nx;
        e = cudaMemsetAsync((char*)m->d_dep + 9 * Nx * 2 * m->esize, 0xff, Nx * sizeof(unsigned long long),
                            m->stream);
        lbfsi::StepArgs a = make_args(m);
        a.ustep = 0;
        a.record = 1;
        if (e == cudaSuccess) e = lbfsi::launch_step_uniform(a, m->precision, m->shape, 1, m->stream);
        m->launches++;
        if (e != cudaSuccess) return cuda_fail(e, "departure cache");
    }
    e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "init sync");
    m->initialized = true;
    return LBFSI_OK;
}

int lbfsi_blend_mesh(lbfsi_mesh m, const lbfsi_body_state* state, const lbfsi_body_state* prev) {
    if (!m || !state) return fail(LBFSI_EINVAL, "null argument");
    if (!m->initialized) return fail(LBFSI_ESTATE, "init_fields first");
    const size_t nb = m->slots();
    static_assert(sizeof(lbfsi_body_state) == sizeof(BodyStateDev), "layout");
    const lbfsi_body_state* pv = prev ? prev : state;
    m->changed();
    cudaError_t e = cudaMemcpyAsync(m->d_state_a, state, nb * sizeof(BodyStateDev), cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->d_state_b, pv, nb * sizeof(BodyStateDev), cudaMemcpyHostToDevice, m->stream);
    // before the first step the collision map is unused; later it stays the
    // state of the last streamed step
    if (e == cudaSuccess)
        e = lbfsi::launch_prepare(m->d_bodies, m->first() ? m->d_state_a : nullptr, m->d_state_a, m->d_state_b,
                                  nullptr, m->dt, (int)nb, m->d_maps[m->cur()], m->stream);
    m->launches++;
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "blend_mesh");
    return LBFSI_OK;
}

int lbfsi_step(lbfsi_mesh m, int nsteps) {
    lbfsi::TraceRange trace_("lbfsi_step");
    if (!m) return fail(LBFSI_EINVAL, "null mesh");
    if (!m->initialized) return fail(LBFSI_ESTATE, "init_fields first");
    if (nsteps < 0) return fail(LBFSI_EINVAL, "nsteps must be >= 0");
    int s = 0;
    if (m->graph_steps > 0 && nsteps >= m->graph_steps) {
        if (!m->graph) {
            const int rc = capture_graph(m);
            if (rc) return rc;
        }
        m->changed();
        for (; nsteps - s >= m->graph_steps; s += m->graph_steps) {
            const cudaError_t e = cudaGraphLaunch(m->graph, m->stream);
            if (e != cudaSuccess) return cuda_fail(e, "graph launch");
            m->launches += m->graph_launches;
            m->host_k += (unsigned)m->graph_steps;
        }
    }
    const cudaError_t e = launch_steps(m, nsteps - s, (long long)m->host_k, nullptr, m->stream, &m->launches);
    if (e != cudaSuccess) return cuda_fail(e, "step kernel launch");
    m->host_k += (unsigned)(nsteps - s);
    return LBFSI_OK;
}

int lbfsi_field_ptr(lbfsi_mesh m, int which, void** ptr, int64_t* slots, int64_t* row0) {
    if (!m || !ptr) return fail(LBFSI_EINVAL, "null argument");
    if (which != LBFSI_FIELD_MOMENTS && which != LBFSI_FIELD_POPULATIONS)
        return fail(LBFSI_EINVAL, "which must be LBFSI_FIELD_MOMENTS or LBFSI_FIELD_POPULATIONS");
    if (!m->initialized) return fail(LBFSI_ESTATE, "init_fields first");
    m->handed_out = true;
    *ptr = which == LBFSI_FIELD_MOMENTS ? m->d_M[m->cur()] : m->pops();
    if (slots) *slots = (int64_t)m->host.Nx;
    if (row0) *row0 = (int64_t)m->host.G * m->host.nt;
    return LBFSI_OK;
}

int lbfsi_synchronize(lbfsi_mesh m) {
    if (!m) return fail(LBFSI_EINVAL, "null mesh");
    return check_status(m);
}

static int download_maps(lbfsi_mesh m, std::vector<StepMaps>& out) {
    out.resize(m->slots());
    std::lock_guard<std::mutex> hold(m->reading);
    StepMaps* to = m->h_maps ? m->h_maps : out.data();
    cudaError_t e = cudaMemcpyAsync(to, m->d_maps[m->cur()], out.size() * sizeof(StepMaps),
                                    cudaMemcpyDeviceToHost, m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "maps copy");
    const int rc = read_status(m);
    if (!rc && m->h_maps) std::memcpy(out.data(), m->h_maps, out.size() * sizeof(StepMaps));
    return rc;
}

int lbfsi_step_record(lbfsi_mesh m, int nsteps, double* loads_out, lbfsi_body_state* states_out) {
    lbfsi::TraceRange trace_("lbfsi_step_record");
    if (!m || !loads_out) return fail(LBFSI_EINVAL, "null argument");
    if (!m->initialized) return fail(LBFSI_ESTATE, "init_fields first");
    if (nsteps < 0) return fail(LBFSI_EINVAL, "nsteps must be >= 0");
    const size_t nb = m->slots();   // one record per (solve, body)
    // the loads blocks of each step write its records into a device history,
    // which comes back in one copy at the end
    const size_t cnt = (size_t)nsteps * nb * 7;
    if (cnt > m->d_rec_count || cnt * sizeof(double) > m->h_rec_bytes) {
        cudaError_t e = cudaStreamSynchronize(m->stream);
        if (e == cudaSuccess && cnt > m->d_rec_count) {
            if (m->d_rec) cudaFree(m->d_rec);
            m->d_rec = nullptr;
            m->d_rec_count = 0;
            e = cudaMalloc(&m->d_rec, cnt * sizeof(double));
            if (e == cudaSuccess) m->d_rec_count = cnt;
        }
        if (e == cudaSuccess && cnt * sizeof(double) > m->h_rec_bytes) {
            if (m->h_rec) cudaFreeHost(m->h_rec);
            m->h_rec = nullptr;
            m->h_rec_bytes = 0;
            e = cudaHostAlloc(&m->h_rec, cnt * sizeof(double), cudaHostAllocDefault);
            if (e == cudaSuccess) m->h_rec_bytes = cnt * sizeof(double);
        }
        if (e != cudaSuccess) {
            cudaGetLastError();
            return fail(LBFSI_ENOMEM, "staging for the step records");
        }
    }
    cudaError_t e = launch_steps(m, nsteps, (long long)m->host_k, m->d_rec, m->stream, &m->launches);
    if (e != cudaSuccess) return cuda_fail(e, "step kernel launch");
    m->host_k += (unsigned)nsteps;
    if (cnt) e = cudaMemcpyAsync(m->h_rec, m->d_rec, cnt * sizeof(double), cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "step record copy");
    static_assert(sizeof(lbfsi_body_state) == sizeof(BodyStateDev), "layout");
    const double* h = static_cast<const double*>(m->h_rec);
    for (size_t r = 0; r < (size_t)nsteps * nb; ++r) {
        std::memcpy(loads_out + 3 * r, h + 7 * r, 3 * sizeof(double));
        if (states_out) std::memcpy(states_out + r, h + 7 * r + 3, sizeof(BodyStateDev));
    }
    return check_status(m);
}

int lbfsi_body_forces(lbfsi_mesh m, double* out) {
    lbfsi::TraceRange trace_("lbfsi_body_forces");
    if (!m || !out) return fail(LBFSI_EINVAL, "null argument");
    if (!m->initialized) return fail(LBFSI_ESTATE, "init_fields first");
    std::vector<StepMaps> mp;
    const int rc = download_maps(m, mp);
    if (rc) return rc;
    for (size_t b = 0; b < m->slots(); ++b)
        for (int c = 0; c < 3; ++c) out[b * 3 + c] = mp[b].loads[c];
    return LBFSI_OK;
}

int lbfsi_advance_bodies(lbfsi_mesh m, const double* loads, double dt) {
    if (!m) return fail(LBFSI_EINVAL, "null mesh");
    if (!m->initialized) return fail(LBFSI_ESTATE, "init_fields first");
    const size_t nb = m->slots();
    std::vector<double> ld(nb * 3);
    if (loads) {
        std::memcpy(ld.data(), loads, ld.size() * sizeof(double));
    } else {
        std::vector<StepMaps> mp;
        const int rc = download_maps(m, mp);
        if (rc) return rc;
        for (size_t b = 0; b < nb; ++b)
            for (int c = 0; c < 3; ++c) ld[b * 3 + c] = mp[b].loads[c];
    }
    m->changed();
    cudaError_t e = cudaMemcpyAsync(m->d_loads_tmp, ld.data(), ld.size() * sizeof(double), cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess)
        e = lbfsi::launch_advance(m->d_bodies, m->d_loads_tmp, dt, (long long)m->host_k, (int)nb,
                                  m->d_maps[m->cur()], m->stream);
    m->launches++;
    if (e != cudaSuccess) return cuda_fail(e, "advance_bodies");
    return check_status(m);
}

int lbfsi_get_body_state(lbfsi_mesh m, lbfsi_body_state* out) {
    if (!m || !out) return fail(LBFSI_EINVAL, "null argument");
    if (!m->initialized) return fail(LBFSI_ESTATE, "init_fields first");
    std::vector<StepMaps> mp;
    const int rc = download_maps(m, mp);
    if (rc) return rc;
    for (size_t b = 0; b < m->slots(); ++b) {
        out[b].h = mp[b].S_next.h;
        out[b].alpha = mp[b].S_next.alpha;
        out[b].hdot = mp[b].S_next.hdot;
        out[b].adot = mp[b].S_next.adot;
    }
    return LBFSI_OK;
}

int lbfsi_get_fields(lbfsi_mesh m, double* rho_u_T) {
    if (!m || !rho_u_T) return fail(LBFSI_EINVAL, "null argument");
    if (!m->initialized) return fail(LBFSI_ESTATE, "init_fields first");
    // rows 0 .. nr-1 of each component (Nx slots apart) straight into the
    // caller's array, float values widened on the device first
    const size_t N = (size_t)m->host.N, Nx = (size_t)m->host.Nx, rows = (size_t)m->nbatch * 4, w = sizeof(double);
    const char* src = (const char*)m->d_M[m->cur()] + (size_t)m->host.G * m->host.nt * m->esize;
    cudaError_t e;
    if (m->precision == LBFSI_FP64) {
        e = cudaMemcpy2DAsync(rho_u_T, N * w, src, Nx * w, N * w, rows, cudaMemcpyDeviceToHost, m->stream);
    } else {
        e = lbfsi::launch_read(m->precision, src, Nx, nullptr, m->d_stage, (int)N, rows, m->stream);
        m->launches++;
        if (m->d_Y == m->d_stage) m->fields_of = -1;
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(rho_u_T, m->d_stage, rows * N * w, cudaMemcpyDeviceToHost, m->stream);
    }
    if (e != cudaSuccess) return cuda_fail(e, "fields download");
    return check_status(m);
}

int lbfsi_get_populations(lbfsi_mesh m, int which, double* f, double* g) {
    if (!m || !f || !g) return fail(LBFSI_EINVAL, "null argument");
    if (which != 0 && which != 1) return fail(LBFSI_EINVAL, "which must be 0 or 1");
    if (!m->initialized) return fail(LBFSI_ESTATE, "init_fields first");
    const size_t cnt = (size_t)m->nbatch * 9 * m->host.N, cntx = (size_t)m->nbatch * 9 * m->host.Nx;
    const void* ps = m->pops();
    if (which == 1 && !m->first()) {
        cudaError_t e = cudaSuccess;
        if (m->precision == LBFSI_FP32 && !m->d_ppost) {
            e = cudaMalloc(&m->d_ppost, 2 * cntx * m->esize);
            if (e != cudaSuccess) return fail(LBFSI_ENOMEM, "post-collision staging allocation failed");
            const int rc = upload_solves(m);
            if (rc) return rc;
        }
        // the field launch on the current state (float64: it collides)
        e = launch_fields(m, make_args(m), 0, 1, (int)m->host_k, nullptr, m->stream);
        m->launches++;
        if (e == cudaSuccess && m->precision == LBFSI_FP32) {
            e = lbfsi::launch_post(m->solves[0], m->dmesh.dev, m->cur(), m->nbatch, m->stream);
            m->launches++;
        }
        if (e != cudaSuccess) return cuda_fail(e, "collide kernel launch");
        ps = m->precision == LBFSI_FP64 ? m->d_p[0] : m->d_ppost;
    }
    std::vector<double> pairs(2 * cnt);
    int rc;
    if (m->host.G) {
        std::vector<double> all(2 * cntx);
        rc = download(m, ps, all.data(), all.size());
        if (!rc) compact_rows(m->host, all.data(), pairs.data(), (size_t)m->nbatch * 9, 2);
    } else {
        rc = download(m, ps, pairs.data(), 2 * cnt);
    }
    if (rc) return rc;
    for (size_t k = 0; k < cnt; ++k) {
        f[k] = pairs[2 * k];
        g[k] = pairs[2 * k + 1];
    }
    return check_status(m);
}

int lbfsi_set_populations(lbfsi_mesh m, const double* f, const double* g, const double* rho_u_T) {
    if (!m || !f || !g || !rho_u_T) return fail(LBFSI_EINVAL, "null argument");
    if (!m->initialized) return fail(LBFSI_ESTATE, "init_fields first");
    const size_t cnt = (size_t)m->nbatch * 9 * m->host.N;
    const int c = m->cur();
    m->changed();
    std::vector<double> pairs(2 * cnt);
    for (size_t k = 0; k < cnt; ++k) {
        pairs[2 * k] = f[k];
        pairs[2 * k + 1] = g[k];
    }
    int rc;
    if (m->host.G) {
        std::vector<double> mu(rho_u_T, rho_u_T + (size_t)m->nbatch * 4 * m->host.N);
        unify_cut_copies(m->host, pairs.data(), (size_t)m->nbatch * 9, 2);
        unify_cut_copies(m->host, mu.data(), (size_t)m->nbatch * 4, 1);
        const std::vector<double> px = expand_rows(m->host, pairs.data(), (size_t)m->nbatch * 9, 2);
        const std::vector<double> mx = expand_rows(m->host, mu.data(), (size_t)m->nbatch * 4, 1);
        rc = upload(m, px.data(), m->pops(), px.size());
        if (!rc) rc = upload(m, mx.data(), m->d_M[c], mx.size());
    } else {
        rc = upload(m, pairs.data(), m->pops(), 2 * cnt);
        if (!rc) rc = upload(m, rho_u_T, m->d_M[c], (size_t)m->nbatch * 4 * m->host.N);
    }
    if (rc) return rc;
    // the restored state is post-propagation: make the next launch collide it
    // (step number >= 2 with the same parity)
    m->host_k = 2u + (unsigned)c;
    std::vector<unsigned> ctr(4 * (size_t)m->nbatch, 0u);
    for (int b = 0; b < m->nbatch; ++b) ctr[4 * b + 1] = m->host_k;
    cudaError_t e = cudaMemcpyAsync(m->d_counter, ctr.data(), ctr.size() * sizeof(unsigned),
                                    cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "step number upload");
    return LBFSI_OK;
}

int64_t lbfsi_launch_count(lbfsi_mesh m) { return m ? m->launches : -1; }

namespace {
struct CheckpointHeader {
    char magic[8];
    int32_t version, precision, nbatch, nr, nt, esize;
    uint32_t step;
    uint32_t nbody;   // 0 in checkpoints of one-body handles
};
constexpr char kMagic[8] = {'L', 'B', 'F', 'S', 'I', 'C', 'K', '1'};

size_t checkpoint_bytes(lbfsi_mesh m) {
    const size_t N = (size_t)m->host.Nx, nb = (size_t)m->nbatch;
    return sizeof(CheckpointHeader) + nb * 18 * N * m->esize + nb * 4 * N * m->esize + m->slots() * sizeof(StepMaps);
}
}  // namespace

size_t lbfsi_checkpoint_bytes(lbfsi_mesh m) { return m ? checkpoint_bytes(m) : 0; }

int lbfsi_checkpoint(lbfsi_mesh m, void* buf, size_t bytes) {
    lbfsi::TraceRange trace_("lbfsi_checkpoint");
    if (!m || !buf) return fail(LBFSI_EINVAL, "null argument");
    if (!m->initialized) return fail(LBFSI_ESTATE, "init_fields first");
    if (bytes < checkpoint_bytes(m)) return fail(LBFSI_EINVAL, "checkpoint buffer too small");
    const int rc = check_status(m);   // a failed state is not saved
    if (rc) return rc;
    CheckpointHeader h{};
    std::memcpy(h.magic, kMagic, sizeof(kMagic));
    h.version = 1;
    h.precision = m->precision;
    h.nbatch = m->nbatch;
    h.nr = m->host.nr;
    h.nt = m->host.nt;
    h.esize = (int32_t)m->esize;
    h.step = m->host_k;
    h.nbody = m->nbody > 1 ? (uint32_t)m->nbody : 0u;
    const size_t N = (size_t)m->host.Nx, nb = (size_t)m->nbatch;
    char* p = static_cast<char*>(buf);
    std::memcpy(p, &h, sizeof(h));
    p += sizeof(h);
    const int c = m->cur();
    cudaError_t e = cudaMemcpyAsync(p, m->pops(), nb * 18 * N * m->esize, cudaMemcpyDeviceToHost, m->stream);
    p += nb * 18 * N * m->esize;
    if (e == cudaSuccess) e = cudaMemcpyAsync(p, m->d_M[c], nb * 4 * N * m->esize, cudaMemcpyDeviceToHost, m->stream);
    p += nb * 4 * N * m->esize;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(p, m->d_maps[c], m->slots() * sizeof(StepMaps), cudaMemcpyDeviceToHost, m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "checkpoint copy");
    return LBFSI_OK;
}

int lbfsi_restore(lbfsi_mesh m, const void* buf, size_t bytes) {
    lbfsi::TraceRange trace_("lbfsi_restore");
    if (!m || !buf) return fail(LBFSI_EINVAL, "null argument");
    if (!m->initialized) return fail(LBFSI_ESTATE, "init_fields first (the flow of the checkpointed run)");
    if (bytes < checkpoint_bytes(m)) return fail(LBFSI_EINVAL, "checkpoint buffer too small for this handle");
    CheckpointHeader h;
    std::memcpy(&h, buf, sizeof(h));
    if (std::memcmp(h.magic, kMagic, sizeof(kMagic)) != 0 || h.version != 1)
        return fail(LBFSI_EINVAL, "not a checkpoint of this library");
    if (h.precision != m->precision || h.nbatch != m->nbatch || h.nr != m->host.nr || h.nt != m->host.nt ||
        h.esize != (int32_t)m->esize || (h.nbody > 1 ? (int)h.nbody : 1) != m->nbody)
        return fail(LBFSI_EINVAL, "checkpoint of a different mesh, batch or precision");
    drop_graph(m);
    m->changed();
    m->host_k = h.step;
    const size_t N = (size_t)m->host.Nx, nb = (size_t)m->nbatch;
    const char* p = static_cast<const char*>(buf) + sizeof(h);
    const int c = m->cur();
    cudaError_t e = cudaMemcpyAsync(m->pops(), p, nb * 18 * N * m->esize, cudaMemcpyHostToDevice, m->stream);
    p += nb * 18 * N * m->esize;
    if (e == cudaSuccess) e = cudaMemcpyAsync(m->d_M[c], p, nb * 4 * N * m->esize, cudaMemcpyHostToDevice, m->stream);
    p += nb * 4 * N * m->esize;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->d_maps[c], p, m->slots() * sizeof(StepMaps), cudaMemcpyHostToDevice, m->stream);
    std::vector<unsigned> ctr(4 * nb, 0u);
    for (size_t b = 0; b < nb; ++b) ctr[4 * b + 1] = m->host_k;
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(m->d_counter, ctr.data(), ctr.size() * sizeof(unsigned), cudaMemcpyHostToDevice, m->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(m->d_status, 0, sizeof(unsigned), m->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
    if (e != cudaSuccess) return cuda_fail(e, "restore copy");
    return LBFSI_OK;
}

int lbfsi_step_variants(int precision) {
    if (precision != LBFSI_FP32 && precision != LBFSI_FP64) return fail(LBFSI_EINVAL, "unknown precision");
    return lbfsi::step_variants(precision);
}

int lbfsi_set_schedule(lbfsi_mesh m, int variant, int order) {
    if (!m) return fail(LBFSI_EINVAL, "null mesh");
    if (variant < 0 || variant >= (m->host.general ? 1 : lbfsi::step_variants(m->precision)) ||
        (order != 0 && order != 1))
        return fail(LBFSI_EINVAL, "variant or order out of range");
    if (!m->own_order && variant == m->variant && order == m->order) return LBFSI_OK;
    drop_graph(m);
    m->own_order = false;
    m->own_shape = m->host.general;   // (general meshes have the one variant)
    m->variant = variant;
    m->order = order;
    set_shape(m);
    return m->initialized ? upload_solves(m) : LBFSI_OK;
}

int lbfsi_get_schedule(lbfsi_mesh m, int* variant, int* order) {
    if (!m) return fail(LBFSI_EINVAL, "null mesh");
    if (variant) *variant = m->variant;
    if (order) *order = m->order;
    return LBFSI_OK;
}

int lbfsi_set_graph_steps(lbfsi_mesh m, int graph_steps) {
    if (!m) return fail(LBFSI_EINVAL, "null mesh");
    if (graph_steps < 0) return fail(LBFSI_EINVAL, "graph_steps must be >= 0");
    if (graph_steps != m->graph_steps) drop_graph(m);
    m->graph_steps = graph_steps;
    return LBFSI_OK;
}

int lbfsi_autotune(lbfsi_mesh m, int steps_per_trial, int* best_variant, int* best_order, float* ms_per_step) {
    lbfsi::TraceRange trace_("lbfsi_autotune");
    if (!m) return fail(LBFSI_EINVAL, "null mesh");
    if (!m->initialized) return fail(LBFSI_ESTATE, "init_fields first");
    if (steps_per_trial < 1) return fail(LBFSI_EINVAL, "steps_per_trial must be >= 1");
    const int nv = m->host.general ? 1 : lbfsi::step_variants(m->precision);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    if (e != cudaSuccess) return cuda_fail(e, "tuner events");
    int bv = m->variant, bo = m->order, rc = LBFSI_OK;
    float best = -1.0f;
    const int graph_steps = m->graph_steps;   // trials use plain launches
    lbfsi_set_graph_steps(m, 0);
    for (int v = 0; v < nv && !rc; ++v)
        for (int o = 0; o < 2 && !rc; ++o) {
            rc = lbfsi_set_schedule(m, v, o);
            if (rc) break;
            lbfsi_step(m, 1);   // first launch of a shape configures it
            cudaEventRecord(e0, m->stream);
            rc = lbfsi_step(m, steps_per_trial);
            cudaEventRecord(e1, m->stream);
            e = cudaEventSynchronize(e1);
            if (e != cudaSuccess) {
                rc = cuda_fail(e, "tuner trial");
                break;
            }
            float ms = 0.0f;
            cudaEventElapsedTime(&ms, e0, e1);
            ms /= (float)steps_per_trial;
            if (ms_per_step) ms_per_step[2 * v + o] = ms;
            if (best < 0.0f || ms < best) {
                best = ms;
                bv = v;
                bo = o;
            }
        }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    lbfsi_set_graph_steps(m, graph_steps);
    if (rc) return rc;
    rc = lbfsi_set_schedule(m, bv, bo);
    if (rc) return rc;
    if (best_variant) *best_variant = bv;
    if (best_order) *best_order = bo;
    return check_status(m);
}

}  // extern "C"
