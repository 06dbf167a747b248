// Batch runtime (declared in include/lbfsi.h): solves on O-grids of different
// sizes admitted into a device memory pool and retired while others run, all
// active solves advanced together by table launches, per step a step launch and
// a field launch for each mesh kind that is there (separable, by coordinates).
// Native pieces: a first-fit pool allocator over one cudaMalloc, a cache of
// device mesh geometry shared by solves on identical O-grids, slot bookkeeping
// and the tile tables (the node-to-CTA schedule) of the launches.
#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "lbfsi.h"
#include "lbfsi_host.h"
#include "lbfsi_internal.h"

using lbfsi::BodyDev;
using lbfsi::BodyStateDev;
using lbfsi::MeshDev;
using lbfsi::SolveDev;
using lbfsi::StepMaps;
using lbfsi::TileDev;

namespace {

// First-fit allocator over one device block; 256-byte granularity; free
// neighbours coalesce.
class Pool : public lbfsi::DevMemory {
public:
    int init(size_t bytes) {
        size_ = (bytes + 255) & ~size_t(255);
        if (cudaMalloc(&base_, size_) != cudaSuccess) {
            cudaGetLastError();
            base_ = nullptr;
            return lbfsi::set_error(LBFSI_ENOMEM, "device pool allocation failed");
        }
        free_[0] = size_;
        return LBFSI_OK;
    }
    ~Pool() override {
        if (base_) cudaFree(base_);
    }
    void* alloc(size_t bytes) override {
        const size_t need = (bytes + 255) & ~size_t(255);
        for (auto it = free_.begin(); it != free_.end(); ++it) {
            if (it->second < need) continue;
            const size_t off = it->first, len = it->second;
            free_.erase(it);
            if (len > need) free_[off + need] = len - need;
            used_[off] = need;
            return base_ + off;
        }
        return nullptr;
    }
    void release(void* p) override {
        if (!p) return;
        const size_t off = (size_t)((char*)p - base_);
        auto u = used_.find(off);
        if (u == used_.end()) return;
        size_t start = off, len = u->second;
        used_.erase(u);
        auto next = free_.lower_bound(start);
        if (next != free_.end() && next->first == start + len) {
            len += next->second;
            free_.erase(next);
        }
        auto prev = free_.lower_bound(start);
        if (prev != free_.begin()) {
            --prev;
            if (prev->first + prev->second == start) {
                start = prev->first;
                len += prev->second;
                free_.erase(prev);
            }
        }
        free_[start] = len;
    }
    size_t free_bytes() const {
        size_t s = 0;
        for (auto& kv : free_) s += kv.second;
        return s;
    }
    size_t largest() const {
        size_t s = 0;
        for (auto& kv : free_) s = std::max(s, kv.second);
        return s;
    }

private:
    char* base_ = nullptr;
    size_t size_ = 0;
    std::map<size_t, size_t> free_, used_;
};

// The body's step map at the head of a solve's workspace.
constexpr size_t WORK_HEAD = 512;
static_assert(sizeof(lbfsi::BodyProp) <= WORK_HEAD, "workspace head");

struct MeshEntry {
    lbfsi::HostMesh host;
    lbfsi::DeviceMesh dev;
    int refs = 0;
    bool used = false;
};

struct Slot {
    bool used = false, finished = false;
    bool general = false;   // on a mesh given by node coordinates (the general kernel)
    int mesh = -1;
    int steps_target = 0, steps_done = 0;
    int ntiles = 0;
    SolveDev dev{};
    std::vector<void*> blocks;
    void* work = nullptr;   // its step workspace (SolveDev::prop, Y), null: among the blocks
    // the tile rows its tensor maps were made for (-1: none yet, 0: not used)
    int tma_rows = -1;
};

}  // namespace

struct lbfsi_batch_s {
    Pool pool;
    // step workspaces of the admitted solves (the bodies' step maps and the float
    // path's correction field), beside the pool so that it admits the solves it
    // always did; made with the batch, for as many as the pool can hold (or
    // empty: the workspaces then come from the pool)
    Pool work;
    int precision = LBFSI_FP32, variant = 4, order = 0, tile_rows = 16;
    // reading a solve back: pinned copies of its record and the status word
    // (null: could not be had)
    struct Small {
        StepMaps maps;
        unsigned status;
    }* h_get = nullptr;
    std::mutex reading;      // held by a read from its first copy until it has taken its values out
    bool own_shape = true;   // no schedule asked for: the shape follows the active solves' sizes
    int shape = 4, gshape = 1;   // tile shapes launched, separable and general meshes (rebuild_tiles)
    size_t esize = 4;
    cudaStream_t stream = nullptr;
    std::vector<MeshEntry> meshes;
    std::vector<Slot> slots;
    MeshDev* d_meshes = nullptr;
    SolveDev* d_solves = nullptr;
    TileDev* d_tiles = nullptr;
    size_t tiles_cap = 0;
    lbfsi::FieldTile* d_ftiles = nullptr;
    size_t ftiles_cap = 0;
    int max_meshes = 256, max_slots = 4096;
    unsigned* d_status = nullptr;
    // float separable solves: tensor maps of each slot's populations and Y,
    // [max_slots][4] (StepArgs::tmaps)
    CUtensorMap* d_tmaps = nullptr;
    BodyStateDev* d_zero_state = nullptr;
    double* d_zero_loads = nullptr;
    // per part of the tables (0 separable, 1 general meshes): step tiles, and
    // in the field table loads blocks followed by field tiles
    int ntiles[2] = {0, 0}, nload[2] = {0, 0}, nfield[2] = {0, 0};
    bool dirty = true;
    // CUDA graph of graph_steps launches over the current tile table,
    // captured on a private stream, dropped whenever the table changes
    int graph_steps = 0;
    cudaGraphExec_t graph = nullptr;
    cudaStream_t cap_stream = nullptr;
};

namespace {

int cuda_err(cudaError_t e, const char* where) {
    return lbfsi::set_error(LBFSI_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

bool same_mesh(const lbfsi::HostMesh& h, const lbfsi_solve_desc& d) {
    return !h.general && h.nr == d.nr && h.nt == d.ntheta && h.xm == d.xc && h.ym == d.yc &&
           std::memcmp(h.r.data(), d.r, sizeof(double) * d.nr) == 0 &&
           std::memcmp(h.e.data(), d.e, sizeof(double) * 2 * d.ntheta) == 0;
}

bool same_mesh_xy(const lbfsi::HostMesh& h, const lbfsi_solve_xy_desc& d) {
    return h.general && !h.cgrid && h.nr == d.nr && h.nt == d.ntheta && h.xm == d.xc && h.ym == d.yc &&
           std::memcmp(h.X.data(), d.X, sizeof(double) * 2 * (size_t)d.nr * d.ntheta) == 0;
}

bool same_mesh_c(const lbfsi::HostMesh& h, const lbfsi_solve_cgrid_desc& d) {
    // the stored coordinates carry the mirrored rows before row 0
    return h.cgrid && h.nr == d.nr && h.nt == d.ntheta && h.walls.size() == 2 && h.walls[0] == d.n_cut &&
           h.xm == d.xc && h.ym == d.yc &&
           std::memcmp(h.X.data() + 2 * (size_t)h.G * h.nt, d.X, sizeof(double) * 2 * (size_t)d.nr * d.ntheta) == 0;
}

// Find or create the device geometry of a mesh (match: an existing entry's
// host mesh equals the request; build: the host mesh of a new one); returns
// the mesh index.
template <typename Match, typename Build>
int acquire_mesh(lbfsi_batch b, Match match, Build build_host, int* out) {
    for (size_t k = 0; k < b->meshes.size(); ++k)
        if (b->meshes[k].used && match(b->meshes[k].host)) {
            b->meshes[k].refs++;
            *out = (int)k;
            return LBFSI_OK;
        }
    int k = -1;
    for (size_t q = 0; q < b->meshes.size(); ++q)
        if (!b->meshes[q].used) {
            k = (int)q;
            break;
        }
    if (k < 0) {
        if ((int)b->meshes.size() >= b->max_meshes) return lbfsi::set_error(LBFSI_ENOMEM, "too many distinct meshes");
        b->meshes.emplace_back();
        k = (int)b->meshes.size() - 1;
    }
    MeshEntry& me = b->meshes[k];
    me = MeshEntry{};
    int rc = build_host(me.host);
    if (rc) return rc;
    rc = lbfsi::upload_mesh(me.host, b->precision, b->pool, b->stream, me.dev);
    if (rc) return rc;
    cudaError_t e = cudaMemcpyAsync(b->d_meshes + k, &me.dev.dev, sizeof(MeshDev), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) {
        lbfsi::release_mesh(me.dev, b->pool);
        return cuda_err(e, "mesh descriptor upload");
    }
    me.used = true;
    me.refs = 1;
    *out = k;
    return LBFSI_OK;
}

void drop_mesh(lbfsi_batch b, int k) {
    MeshEntry& me = b->meshes[k];
    if (--me.refs > 0) return;
    cudaStreamSynchronize(b->stream);
    lbfsi::release_mesh(me.dev, b->pool);
    me.used = false;
}

void release_slot_memory(lbfsi_batch b, Slot& s) {
    for (void* p : s.blocks) b->pool.release(p);
    s.blocks.clear();
    if (s.work) b->work.release(s.work);
    s.work = nullptr;
}

void drop_graph(lbfsi_batch b) {
    if (b->graph) {
        cudaStreamSynchronize(b->stream);
        cudaGraphExecDestroy(b->graph);
        b->graph = nullptr;
    }
}

int step_rows(lbfsi_batch b, bool general) {
    return general ? lbfsi::general_tile_rows(b->precision, b->gshape) : b->tile_rows;
}

// CTAs of a slot's step launches in the current tile shape (SolveDev::ntiles,
// the completion count), uploaded where it changed.
cudaError_t update_counts(lbfsi_batch b) {
    cudaError_t e = cudaSuccess;
    for (size_t k = 0; k < b->slots.size() && e == cudaSuccess; ++k) {
        Slot& s = b->slots[k];
        if (!s.used) continue;
        const lbfsi::HostMesh& h = b->meshes[s.mesh].host;
        const int rows = step_rows(b, s.general), n = ((h.nr + rows - 1) / rows) * h.ntj;
        if (n == s.ntiles) continue;
        s.dev.ntiles = s.ntiles = n;
        e = cudaMemcpyAsync(b->d_solves + k, &s.dev, sizeof(SolveDev), cudaMemcpyHostToDevice, b->stream);
    }
    return e;
}

// Upload of a host table into a device array that grows as needed.
template <typename T>
cudaError_t put_table(lbfsi_batch b, const std::vector<T>& v, T*& dev, size_t& cap) {
    cudaError_t e = cudaSuccess;
    if (v.size() > cap) {
        e = cudaStreamSynchronize(b->stream);
        if (dev) cudaFree(dev);
        dev = nullptr;
        cap = std::max(v.size(), 2 * cap);
        if (e == cudaSuccess) e = cudaMalloc(&dev, cap * sizeof(T));
        if (e != cudaSuccess) {
            cap = 0;
            return e;
        }
    }
    // stream-ordered: launches already queued read the previous table
    if (!v.empty()) e = cudaMemcpyAsync(dev, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, b->stream);
    return e;
}

// Tables of the next launches: every tile of every active solve, in the
// batch's order: 0, the tiles of each solve together; 1, tile rows outermost
// across all solves, so that the wall and blending-region rows (the most
// expensive tiles) start first and the far-field rows fill the tail.
int rebuild_tiles(lbfsi_batch b) {
    lbfsi::TraceRange trace_("lbfsi tile table");
    drop_graph(b);
    cudaError_t e = cudaSuccess;
    auto active = [&](const Slot& s, int part) { return s.used && !s.finished && (s.general ? 1 : 0) == part; };
    b->shape = b->gshape = b->variant;
    if (b->precision == LBFSI_FP32) {
        // as the mesh handle (step_shape)
        long long n[2] = {0, 0};
        for (int part = 0; part < 2; ++part)
            for (const Slot& s : b->slots)
                if (active(s, part)) n[part] += (long long)b->meshes[s.mesh].host.ntj * ((b->meshes[s.mesh].host.nr + 15) / 16);
        if (b->own_shape) b->shape = lbfsi::default_shape(b->precision, n[0]);
        b->gshape = lbfsi::default_shape_general(false, true, n[1]);   // (staged by per-thread copies)
    }
    b->tile_rows = lbfsi::tile_rows(b->precision, b->shape);
    e = update_counts(b);
    if (e != cudaSuccess) return cuda_err(e, "solve record upload");
    // float separable solves: tensor maps for the current tile shape (made
    // once per slot and shape, uploaded behind the launches already queued)
    const char* tenv = std::getenv("LBFSI_TMA");
    const bool tma_on = b->precision == LBFSI_FP32 && b->d_tmaps && !(tenv && std::atoi(tenv) == 0);
    for (size_t k = 0; k < b->slots.size() && tma_on; ++k) {
        Slot& s = b->slots[k];
        if (!s.used || s.finished || s.general || s.tma_rows == b->tile_rows) continue;
        const lbfsi::HostMesh& h = b->meshes[s.mesh].host;
        bool ok = h.nt % 4 == 0;
        CUtensorMap maps[4]{};
        const size_t nt = (size_t)h.nt, nr = (size_t)h.nr;
        const unsigned rows = (unsigned)b->tile_rows, w = (unsigned)(lbfsi::TILE_J + 8);
        for (int c = 0; c < 2 && ok; ++c) ok = lbfsi::encode_box4(&maps[c], s.dev.p[c], 2 * nt, nr, 9, 1, 2 * w, rows + 4, 9);
        ok = ok && lbfsi::encode_box4(&maps[2], s.dev.Y, nt, nr, 2, 1, w, rows + 4, 2);
        if (ok) {
            e = cudaMemcpyAsync(b->d_tmaps + 4 * k, maps, sizeof(maps), cudaMemcpyHostToDevice, b->stream);
            if (e != cudaSuccess) return cuda_err(e, "tensor map upload");
        }
        s.tma_rows = ok ? b->tile_rows : 0;
    }
    std::vector<TileDev> tiles;
    std::vector<lbfsi::FieldTile> ftiles;
    for (int part = 0; part < 2; ++part) {
        const int rows = step_rows(b, part == 1);
        const size_t t0 = tiles.size(), f0 = ftiles.size();
        auto push = [&](size_t k, int ti, int tj) {
            const Slot& s = b->slots[k];
            TileDev t{};
            t.solve = (int)k;
            t.mesh = s.mesh;
            t.i0 = ti * rows;
            t.j0 = tj * lbfsi::TILE_J;
            // a separable tile whose columns do not wrap, of a solve with maps
            const int ntm = b->meshes[s.mesh].host.nt;
            t.tma = part == 0 && tma_on && s.tma_rows == rows && t.j0 >= 4 && t.j0 + lbfsi::TILE_J + 4 <= ntm;
            t.counter = s.dev.counter;
            t.maps[0] = s.dev.maps[0];
            t.maps[1] = s.dev.maps[1];
            tiles.push_back(t);
        };
        auto nti_of = [&](size_t k) { return (b->meshes[b->slots[k].mesh].host.nr + rows - 1) / rows; };
        if (b->order == 0) {
            for (size_t k = 0; k < b->slots.size(); ++k) {
                if (!active(b->slots[k], part)) continue;
                const int nti = nti_of(k), ntj = b->meshes[b->slots[k].mesh].host.ntj;
                for (int ti = 0; ti < nti; ++ti)
                    for (int tj = 0; tj < ntj; ++tj) push(k, ti, tj);
            }
        } else {
            int max_nti = 0;
            for (size_t k = 0; k < b->slots.size(); ++k)
                if (active(b->slots[k], part)) max_nti = std::max(max_nti, nti_of(k));
            for (int ti = 0; ti < max_nti; ++ti)
                for (size_t k = 0; k < b->slots.size(); ++k) {
                    if (!active(b->slots[k], part) || ti >= nti_of(k)) continue;
                    const int ntj = b->meshes[b->slots[k].mesh].host.ntj;
                    for (int tj = 0; tj < ntj; ++tj) push(k, ti, tj);
                }
        }
        b->ntiles[part] = (int)(tiles.size() - t0);
        b->nload[part] = b->nfield[part] = 0;
        for (int fields = 0; fields < 2; ++fields)
            for (size_t k = 0; k < b->slots.size(); ++k) {
                if (!active(b->slots[k], part)) continue;
                const lbfsi::HostMesh& h = b->meshes[b->slots[k].mesh].host;
                const int n = fields ? lbfsi::field_blocks(b->precision, part == 1, h.nr, h.nt) : lbfsi::load_blocks(h.ntj);
                for (int t = 0; t < n; ++t) ftiles.push_back({(int)k, b->slots[k].mesh, fields, t});
                (fields ? b->nfield : b->nload)[part] += n;
            }
    }
    e = put_table(b, tiles, b->d_tiles, b->tiles_cap);
    if (e == cudaSuccess) e = put_table(b, ftiles, b->d_ftiles, b->ftiles_cap);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return cuda_err(e, "tile table upload");
    b->dirty = false;
    return LBFSI_OK;
}

// (one copy behind the stream's work, one wait; the caller holds 'reading')
int read_status(lbfsi_batch b) {
    unsigned own = 0, *hs = b->h_get ? &b->h_get->status : &own;
    cudaError_t e = cudaMemcpyAsync(hs, b->d_status, sizeof(unsigned), cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return cuda_err(e, "status read");
    const unsigned st = *hs;
    if (st & lbfsi::ST_BOUNDS)
        return lbfsi::set_error(LBFSI_EBOUNDS, "an index of the step outside its buffer (bounds-checked build)");
    if (st & (lbfsi::ST_DEPARTURE | lbfsi::ST_BPOINT))
        return lbfsi::set_error(LBFSI_EDEPARTURE, "departure point outside the cells adjacent to its node (CFL)");
    if (st & lbfsi::ST_TMA)
        return lbfsi::set_error(LBFSI_ECUDA, "a tensor copy of the step did not complete within its wait limit");
    if (st & lbfsi::ST_NONPHYS) return lbfsi::set_error(LBFSI_ENONPHYS, "non-physical state (rho<=0, T<=0 or NaN)");
    return LBFSI_OK;
}

int check_status(lbfsi_batch b) {
    std::lock_guard<std::mutex> hold(b->reading);
    return read_status(b);
}

// Step launch of one part of the tile table (0 separable, 1 general meshes).
cudaError_t launch_step_part(lbfsi_batch b, int part, cudaStream_t s) {
    if (b->ntiles[part] == 0) return cudaSuccess;
    lbfsi::StepArgs a{};
    a.meshes = b->d_meshes;
    a.solves = b->d_solves;
    a.tiles = b->d_tiles + (part ? b->ntiles[0] : 0);
    a.ntiles = b->ntiles[part];
    a.ustep = -1;
    a.status = b->d_status;
    a.tmaps = part == 0 && b->precision == LBFSI_FP32 ? b->d_tmaps : nullptr;
    return lbfsi::launch_step(a, b->precision, part == 1, part == 1 ? b->gshape : b->shape, s);
}

// Field launch of one part: the loads of the last step, the fields of the
// current state, or both.
cudaError_t launch_field_part(lbfsi_batch b, int part, int loads, int fields, cudaStream_t s) {
    lbfsi::FieldArgs f{};
    f.meshes = b->d_meshes;
    f.solves = b->d_solves;
    f.tiles = b->d_ftiles + (part ? b->nload[0] + b->nfield[0] : 0) + (loads ? 0 : b->nload[part]);
    f.ntiles = (loads ? b->nload[part] : 0) + (fields ? b->nfield[part] : 0);
    f.loads = loads;
    f.fields = fields;
    f.ustep = -1;
    f.status = b->d_status;
    return lbfsi::launch_fields(f, b->precision, part == 1, s);
}

// n steps of every active solve (as launch_steps of the mesh handle): the
// current state's fields, then per step the step launches of both parts
// (independent solves, so their order is free) and the field launches.
cudaError_t launch_run(lbfsi_batch b, int n, cudaStream_t s) {
    cudaError_t e = cudaSuccess;
    auto both = [&](auto fn) {
        for (int part = 0; part < 2 && e == cudaSuccess; ++part) e = fn(part);
    };
    if (n > 0) both([&](int p) { return launch_field_part(b, p, 0, 1, s); });
    for (int k = 0; k < n && e == cudaSuccess; ++k) {
        both([&](int p) { return launch_step_part(b, p, s); });
        both([&](int p) { return launch_field_part(b, p, 1, k + 1 < n, s); });
    }
    return e;
}

// Capture graph_steps launches over the current tile table (every launch
// reads the step numbers from the device counters, so the graph is valid for
// every replay until the table changes).
int capture_graph(lbfsi_batch b) {
    lbfsi::TraceRange trace_("lbfsi batch graph capture");
    cudaError_t e = lbfsi::prepare_step(b->precision, b->shape, false);
    if (e == cudaSuccess && b->ntiles[1] > 0) e = lbfsi::prepare_step(b->precision, b->gshape, false, true);
    if (e == cudaSuccess && !b->cap_stream) e = cudaStreamCreateWithFlags(&b->cap_stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) return cuda_err(e, "graph capture setup");
    e = cudaStreamBeginCapture(b->cap_stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return cuda_err(e, "begin capture");
    const cudaError_t le = launch_run(b, b->graph_steps, b->cap_stream);
    cudaGraph_t graph = nullptr;
    e = cudaStreamEndCapture(b->cap_stream, &graph);
    if (le != cudaSuccess || e != cudaSuccess) {
        if (graph) cudaGraphDestroy(graph);
        return cuda_err(le != cudaSuccess ? le : e, "batch step capture");
    }
    e = cudaGraphInstantiate(&b->graph, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) {
        b->graph = nullptr;
        return cuda_err(e, "graph instantiate");
    }
    return LBFSI_OK;
}

}  // namespace

extern "C" {

int lbfsi_batch_create(size_t pool_bytes, int precision, void* cuda_stream, lbfsi_batch* out) {
    if (!out) return lbfsi::set_error(LBFSI_EINVAL, "null argument");
    *out = nullptr;
    if (precision != LBFSI_FP64 && precision != LBFSI_FP32)
        return lbfsi::set_error(LBFSI_EINVAL, "precision must be LBFSI_FP64 or LBFSI_FP32");
    if (pool_bytes < (1u << 20)) return lbfsi::set_error(LBFSI_EINVAL, "pool must be at least 1 MiB");
    auto b = new lbfsi_batch_s();
    b->precision = precision;
    b->esize = precision == LBFSI_FP64 ? sizeof(double) : sizeof(float);
    b->stream = static_cast<cudaStream_t>(cuda_stream);
    if (precision == LBFSI_FP64) b->variant = 0;
    b->shape = b->gshape = b->variant;
    b->tile_rows = lbfsi::tile_rows(precision, b->shape);
    int rc = b->pool.init(pool_bytes);
    if (rc) {
        delete b;
        return rc;
    }
    // a node takes 176 bytes of the pool and in float 8 of the workspaces
    b->work.init((size_t)b->max_slots * (WORK_HEAD + 256) + (precision == LBFSI_FP32 ? pool_bytes / 22 : 0));
    cudaError_t e = cudaMalloc(&b->d_meshes, b->max_meshes * sizeof(MeshDev));
    if (e == cudaSuccess) e = cudaMalloc(&b->d_solves, b->max_slots * sizeof(SolveDev));
    if (e == cudaSuccess) e = cudaMalloc(&b->d_status, sizeof(unsigned));
    if (e == cudaSuccess && precision == LBFSI_FP32)
        e = cudaMalloc(&b->d_tmaps, (size_t)b->max_slots * 4 * sizeof(CUtensorMap));
    if (e == cudaSuccess) e = cudaMalloc(&b->d_zero_state, sizeof(BodyStateDev));
    if (e == cudaSuccess) e = cudaMalloc(&b->d_zero_loads, 3 * sizeof(double));
    if (e == cudaSuccess) e = cudaMemset(b->d_status, 0, sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMemset(b->d_zero_state, 0, sizeof(BodyStateDev));
    if (e == cudaSuccess) e = cudaMemset(b->d_zero_loads, 0, 3 * sizeof(double));
    if (e != cudaSuccess) {
        lbfsi_batch_destroy(b);
        return lbfsi::set_error(LBFSI_ENOMEM, std::string("batch allocation: ") + cudaGetErrorString(e));
    }
    if (cudaMallocHost((void**)&b->h_get, sizeof(*b->h_get)) != cudaSuccess) {
        b->h_get = nullptr;
        cudaGetLastError();
    }
    *out = b;
    return LBFSI_OK;
}

int lbfsi_batch_destroy(lbfsi_batch b) {
    if (!b) return lbfsi::set_error(LBFSI_EINVAL, "null batch");
    cudaStreamSynchronize(b->stream);
    if (b->h_get) cudaFreeHost(b->h_get);
    void* ptrs[] = {b->d_meshes, b->d_solves, b->d_tiles, b->d_ftiles, b->d_status, b->d_zero_state,
                    b->d_zero_loads, b->d_tmaps};
    for (void* p : ptrs)
        if (p) cudaFree(p);
    if (b->graph) cudaGraphExecDestroy(b->graph);
    if (b->cap_stream) cudaStreamDestroy(b->cap_stream);
    delete b;   // the pool frees its block
    return LBFSI_OK;
}

}  // extern "C"

namespace {

// Admission of one solve whose mesh is given by 'acquire' (which finds or
// creates its device geometry): pool memory, initial state, slot.
template <typename Acquire>
int add_solve(lbfsi_batch b, const lbfsi_body_desc& body_desc, const lbfsi_flow_params& flow,
              const double* rho_u_T, int steps, int nr, int nt, Acquire acquire, int* slot) {
    if (!slot) return lbfsi::set_error(LBFSI_EINVAL, "null argument");
    *slot = -1;
    if (steps <= 0) return lbfsi::set_error(LBFSI_EINVAL, "steps must be > 0");
    const long long Nll = (long long)nr * nt;
    if (nr < 5 || nt < 4 || Nll * 9 > (1ll << 31)) return lbfsi::set_error(LBFSI_EINVAL, "invalid mesh size");
    SolveDev sd{};
    int rc = lbfsi::fill_flow(flow, sd);
    if (rc) return rc;
    // a free slot
    int k = -1;
    for (size_t q = 0; q < b->slots.size(); ++q)
        if (!b->slots[q].used) {
            k = (int)q;
            break;
        }
    if (k < 0) {
        if ((int)b->slots.size() >= b->max_slots) return lbfsi::set_error(LBFSI_ENOMEM, "no free slot");
        b->slots.emplace_back();
        k = (int)b->slots.size() - 1;
    }
    int mk = -1;
    rc = acquire(&mk);
    if (rc) return rc;
    const lbfsi::HostMesh& h = b->meshes[mk].host;
    rc = lbfsi::validate_bodies(h, &body_desc, 1);
    if (rc) {
        drop_mesh(b, mk);
        return rc;
    }
    Slot s;
    // slots per component: nr nt, plus a C-grid's mirrored rows before row 0
    const size_t N = (size_t)h.N, Nx = (size_t)h.Nx, es = b->esize, g0 = (size_t)h.G * h.nt;
    auto take = [&](size_t bytes) -> void* {
        void* p = b->pool.alloc(bytes);
        if (p) s.blocks.push_back(p);
        return p;
    };
    bool ok = true;
    void* p0 = nullptr;   // population block of the initial state (float64: the state's, the second)
    void* m0 = nullptr;
    for (int p = 0; p < 2 && ok; ++p) {
        void* pb = take(18 * Nx * es);
        void* mb = take(4 * Nx * es);
        ok = ok && pb && mb;
        if (p == (b->precision == LBFSI_FP64 ? 1 : 0)) p0 = pb;
        if (p == 0) m0 = mb;
        if (ok) {
            sd.p[p] = (char*)pb + 2 * g0 * es;   // row 0
            sd.M[p] = (char*)mb + g0 * es;
        }
        ok = ok && (sd.maps[p] = (StepMaps*)take(sizeof(StepMaps))) != nullptr;
    }
    ok = ok && (sd.part = (double*)take((size_t)h.ntj * 3 * sizeof(double))) != nullptr;
    ok = ok && (sd.counter = (unsigned*)take(4 * sizeof(unsigned))) != nullptr;
    BodyDev* body = nullptr;
    ok = ok && (body = (BodyDev*)take(sizeof(BodyDev))) != nullptr;
    double* stage = nullptr;
    ok = ok && (stage = (double*)take(4 * Nx * sizeof(double))) != nullptr;
    if (ok) {
        // the body's step map, then float the correction field
        const bool f64 = b->precision == LBFSI_FP64;
        const size_t bytes = WORK_HEAD + (f64 ? 0 : 2 * Nx * es);
        void* work = s.work = b->work.alloc(bytes);
        if (!work) work = take(bytes);
        ok = work != nullptr;
        if (ok) {
            sd.prop = (const lbfsi::BodyProp*)work;
            if (!f64) sd.Y = (char*)work + WORK_HEAD + g0 * es;
        }
        if (f64) {   // (SolveDev::p, ppost)
            sd.ppost = sd.p[0];
            sd.p[0] = sd.p[1];
        }
    }
    if (!ok) {
        release_slot_memory(b, s);
        drop_mesh(b, mk);
        return lbfsi::set_error(LBFSI_ENOMEM, "the pool has no room for this solve now");
    }
    sd.body = body;
    sd.mesh = mk;
    const int rows = step_rows(b, h.general);
    sd.ntiles = ((h.nr + rows - 1) / rows) * h.ntj;
    // initial state: equilibria of the initial field, bodies at rest
    std::vector<double> M(4 * N);
    if (rho_u_T) {
        std::memcpy(M.data(), rho_u_T, M.size() * sizeof(double));
    } else {
        for (size_t n = 0; n < N; ++n) {
            M[n] = sd.rho_inf;
            M[N + n] = sd.uinf_x;
            M[2 * N + n] = 0.0;
            M[3 * N + n] = sd.T_inf;
        }
    }
    if (h.cgrid) {
        // the two copies of a cut node start from the first copy's values;
        // the mirrored rows below row 0 from their nodes
        for (int c = 0; c < 4; ++c)
            for (int j = 0; j < h.nt; ++j)
                if (h.coltype[j] & lbfsi::CT_DUP) M[c * N + (size_t)j] = M[c * N + (size_t)(h.nt - 1 - j)];
        std::vector<double> Mx(4 * Nx);
        for (int c = 0; c < 4; ++c) {
            std::memcpy(&Mx[c * Nx + g0], &M[c * N], N * sizeof(double));
            for (int k2 = 1; k2 <= h.G; ++k2)
                for (int j = 0; j < h.nt; ++j)
                    Mx[c * Nx + g0 - (size_t)k2 * h.nt + j] = M[c * N + (size_t)k2 * h.nt + (h.nt - 1 - j)];
        }
        M.swap(Mx);
    }
    const BodyDev bd = lbfsi::body_dev(body_desc, sd.rho_inf, sd.uinf_x);
    const lbfsi::BodyProp prop = lbfsi::body_prop(bd, sd.dt);
    cudaError_t e = cudaMemcpyAsync(stage, M.data(), M.size() * sizeof(double), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(body, &bd, sizeof(BodyDev), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync((void*)sd.prop, &prop, sizeof(prop), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(sd.counter, 0, 4 * sizeof(unsigned), b->stream);
    if (e == cudaSuccess) e = lbfsi::launch_init(b->precision, stage, p0, m0, (int)Nx, 1, sd.Cv, b->stream);
    if (e == cudaSuccess)
        e = lbfsi::launch_prepare(body, b->d_zero_state, b->d_zero_state, b->d_zero_state, b->d_zero_loads, sd.dt,
                                  1, sd.maps[0], b->stream);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(b->d_solves + k, &sd, sizeof(SolveDev), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    // the staging block is no longer needed
    b->pool.release(stage);
    s.blocks.erase(std::remove(s.blocks.begin(), s.blocks.end(), (void*)stage), s.blocks.end());
    if (e != cudaSuccess) {
        release_slot_memory(b, s);
        drop_mesh(b, mk);
        return cuda_err(e, "solve initialisation");
    }
    s.used = true;
    s.finished = false;
    s.general = h.general;
    s.mesh = mk;
    s.steps_target = steps;
    s.steps_done = 0;
    s.ntiles = sd.ntiles;
    s.dev = sd;
    b->slots[k] = std::move(s);
    b->dirty = true;
    *slot = k;
    return LBFSI_OK;
}

}  // namespace

extern "C" {

int lbfsi_batch_add(lbfsi_batch b, const lbfsi_solve_desc* d, int* slot) {
    lbfsi::TraceRange trace_("lbfsi_batch_add");
    if (!b || !d || !slot) return lbfsi::set_error(LBFSI_EINVAL, "null argument");
    auto acquire = [&](int* mk) {
        return acquire_mesh(
            b, [&](const lbfsi::HostMesh& h) { return same_mesh(h, *d); },
            [&](lbfsi::HostMesh& h) { return lbfsi::build_host_mesh(d->nr, d->ntheta, d->r, d->e, d->xc, d->yc, h); },
            mk);
    };
    return add_solve(b, d->body, d->flow, d->rho_u_T, d->steps, d->nr, d->ntheta, acquire, slot);
}

int lbfsi_batch_add_xy(lbfsi_batch b, const lbfsi_solve_xy_desc* d, int* slot) {
    lbfsi::TraceRange trace_("lbfsi_batch_add_xy");
    if (!b || !d || !slot) return lbfsi::set_error(LBFSI_EINVAL, "null argument");
    auto acquire = [&](int* mk) {
        return acquire_mesh(
            b, [&](const lbfsi::HostMesh& h) { return same_mesh_xy(h, *d); },
            [&](lbfsi::HostMesh& h) { return lbfsi::build_host_mesh_xy(d->nr, d->ntheta, d->X, d->xc, d->yc, h); },
            mk);
    };
    return add_solve(b, d->body, d->flow, d->rho_u_T, d->steps, d->nr, d->ntheta, acquire, slot);
}

int lbfsi_batch_add_cgrid(lbfsi_batch b, const lbfsi_solve_cgrid_desc* d, int* slot) {
    lbfsi::TraceRange trace_("lbfsi_batch_add_cgrid");
    if (!b || !d || !slot) return lbfsi::set_error(LBFSI_EINVAL, "null argument");
    auto acquire = [&](int* mk) {
        return acquire_mesh(
            b, [&](const lbfsi::HostMesh& h) { return same_mesh_c(h, *d); },
            [&](lbfsi::HostMesh& h) {
                const int walls[2] = {d->n_cut, d->ntheta - 1 - d->n_cut};
                return lbfsi::build_host_mesh_c(d->nr, d->ntheta, 1, walls, d->X, d->xc, d->yc, h);
            },
            mk);
    };
    return add_solve(b, d->body, d->flow, d->rho_u_T, d->steps, d->nr, d->ntheta, acquire, slot);
}

int lbfsi_batch_step(lbfsi_batch b, int nsteps, int* active_after) {
    lbfsi::TraceRange trace_("lbfsi_batch_step");
    if (!b) return lbfsi::set_error(LBFSI_EINVAL, "null batch");
    if (nsteps < 0) return lbfsi::set_error(LBFSI_EINVAL, "nsteps must be >= 0");
    int st = 0;
    while (st < nsteps) {
        if (b->dirty) {
            const int rc = rebuild_tiles(b);
            if (rc) return rc;
        }
        if (b->ntiles[0] + b->ntiles[1] == 0) break;
        // steps until the next solve finishes: the tile table is fixed over them
        int run = nsteps - st;
        for (auto& s : b->slots)
            if (s.used && !s.finished) run = std::min(run, s.steps_target - s.steps_done);
        int done = 0;
        if (b->graph_steps > 0 && run >= b->graph_steps) {
            if (!b->graph) {
                const int rc = capture_graph(b);
                if (rc) return rc;
            }
            for (; run - done >= b->graph_steps; done += b->graph_steps) {
                const cudaError_t e = cudaGraphLaunch(b->graph, b->stream);
                if (e != cudaSuccess) return cuda_err(e, "batch graph launch");
            }
        }
        const cudaError_t e = launch_run(b, run - done, b->stream);
        if (e != cudaSuccess) return cuda_err(e, "batch step launch");
        st += run;
        for (auto& s : b->slots) {
            if (!s.used || s.finished) continue;
            s.steps_done += run;
            if (s.steps_done >= s.steps_target) {
                s.finished = true;
                b->dirty = true;
            }
        }
    }
    if (active_after) {
        int n = 0;
        for (auto& s : b->slots) n += (s.used && !s.finished) ? 1 : 0;
        *active_after = n;
    }
    return LBFSI_OK;
}

int lbfsi_batch_set_schedule(lbfsi_batch b, int variant, int order) {
    if (!b) return lbfsi::set_error(LBFSI_EINVAL, "null batch");
    if (variant < 0 || variant >= lbfsi::step_variants(b->precision) || (order != 0 && order != 1))
        return lbfsi::set_error(LBFSI_EINVAL, "variant or order out of range");
    if (!b->own_shape && variant == b->variant && order == b->order) return LBFSI_OK;
    drop_graph(b);
    b->own_shape = false;
    b->variant = variant;
    b->order = order;
    b->dirty = true;   // (rebuild_tiles: the tile shape, the per-solve CTA counts, the tables)
    return LBFSI_OK;
}

int lbfsi_batch_get_schedule(lbfsi_batch b, int* variant, int* order) {
    if (!b) return lbfsi::set_error(LBFSI_EINVAL, "null batch");
    if (variant) *variant = b->variant;
    if (order) *order = b->order;
    return LBFSI_OK;
}

int lbfsi_batch_set_graph_steps(lbfsi_batch b, int graph_steps) {
    if (!b) return lbfsi::set_error(LBFSI_EINVAL, "null batch");
    if (graph_steps < 0) return lbfsi::set_error(LBFSI_EINVAL, "graph_steps must be >= 0");
    if (graph_steps != b->graph_steps) drop_graph(b);
    b->graph_steps = graph_steps;
    return LBFSI_OK;
}

int lbfsi_batch_autotune(lbfsi_batch b, int steps_per_trial, int* best_variant, int* best_order,
                         float* ns_per_node) {
    lbfsi::TraceRange trace_("lbfsi_batch_autotune");
    if (!b) return lbfsi::set_error(LBFSI_EINVAL, "null batch");
    if (steps_per_trial < 1) return lbfsi::set_error(LBFSI_EINVAL, "steps_per_trial must be >= 1");
    const int nv = lbfsi::step_variants(b->precision);
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    if (e != cudaSuccess) return cuda_err(e, "tuner events");
    const int graph_steps = b->graph_steps;   // trials use plain launches
    lbfsi_batch_set_graph_steps(b, 0);
    int bv = b->variant, bo = b->order, rc = LBFSI_OK;
    float best = -1.0f;
    for (int v = 0; v < nv && !rc; ++v)
        for (int o = 0; o < 2 && !rc; ++o) {
            rc = lbfsi_batch_set_schedule(b, v, o);
            if (rc) break;
            rc = lbfsi_batch_step(b, 1, nullptr);   // configures the shape, rebuilds the table
            if (rc) break;
            // node updates of the trial, from the steps each solve takes
            std::vector<int> before(b->slots.size());
            for (size_t k = 0; k < b->slots.size(); ++k) before[k] = b->slots[k].steps_done;
            cudaEventRecord(e0, b->stream);
            rc = lbfsi_batch_step(b, steps_per_trial, nullptr);
            cudaEventRecord(e1, b->stream);
            e = cudaEventSynchronize(e1);
            if (!rc && e != cudaSuccess) rc = cuda_err(e, "tuner trial");
            if (rc) break;
            double nodes = 0.0;
            for (size_t k = 0; k < b->slots.size(); ++k)
                if (b->slots[k].used)
                    nodes += (double)(b->slots[k].steps_done - before[k]) * b->meshes[b->slots[k].mesh].host.N;
            float ms = 0.0f;
            cudaEventElapsedTime(&ms, e0, e1);
            const float ns = nodes > 0.0 ? (float)(ms * 1e6 / nodes) : -1.0f;
            if (ns_per_node) ns_per_node[2 * v + o] = ns;
            if (ns > 0.0f && (best < 0.0f || ns < best)) {
                best = ns;
                bv = v;
                bo = o;
            }
        }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    lbfsi_batch_set_graph_steps(b, graph_steps);
    if (rc) return rc;
    rc = lbfsi_batch_set_schedule(b, bv, bo);
    if (rc) return rc;
    if (best_variant) *best_variant = bv;
    if (best_order) *best_order = bo;
    return check_status(b);
}

int lbfsi_batch_poll(lbfsi_batch b, int slot, int* steps_done, int* finished) {
    if (!b || slot < 0 || slot >= (int)b->slots.size() || !b->slots[slot].used)
        return lbfsi::set_error(LBFSI_EINVAL, "invalid slot");
    if (steps_done) *steps_done = b->slots[slot].steps_done;
    if (finished) *finished = b->slots[slot].finished ? 1 : 0;
    return LBFSI_OK;
}

int lbfsi_batch_get(lbfsi_batch b, int slot, double* rho_u_T, double* loads, lbfsi_body_state* state) {
    if (!b || slot < 0 || slot >= (int)b->slots.size() || !b->slots[slot].used)
        return lbfsi::set_error(LBFSI_EINVAL, "invalid slot");
    const Slot& s = b->slots[slot];
    const int cur = s.steps_done & 1;
    const size_t N = (size_t)b->meshes[s.mesh].host.N, Nx = (size_t)b->meshes[s.mesh].host.Nx;
    cudaError_t e = cudaSuccess;
    // rows 0 .. nr-1 of the four components (Nx slots apart) straight into the
    // caller's array, float values widened on the device first: in the population
    // buffer that the next step writes (72 bytes a node; 32 are needed)
    if (rho_u_T && b->precision == LBFSI_FP32) {
        double* wide = (double*)s.dev.p[cur ^ 1];
        e = lbfsi::launch_read(b->precision, s.dev.M[cur], Nx, nullptr, wide, (int)N, 4, b->stream);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(rho_u_T, wide, 4 * N * sizeof(double), cudaMemcpyDeviceToHost, b->stream);
    } else if (rho_u_T) {
        e = cudaMemcpy2DAsync(rho_u_T, N * sizeof(double), s.dev.M[cur], Nx * sizeof(double), N * sizeof(double), 4,
                              cudaMemcpyDeviceToHost, b->stream);
    }
    std::lock_guard<std::mutex> hold(b->reading);
    StepMaps own{}, *rec = b->h_get ? &b->h_get->maps : &own;
    if (e == cudaSuccess && (loads || state))
        e = cudaMemcpyAsync(rec, s.dev.maps[cur], sizeof(StepMaps), cudaMemcpyDeviceToHost, b->stream);
    if (e != cudaSuccess) return cuda_err(e, "batch results copy");
    const int rc = read_status(b);
    const StepMaps& mp = *rec;
    if (loads)
        for (int c = 0; c < 3; ++c) loads[c] = mp.loads[c];
    if (state) {
        state->h = mp.S_next.h;
        state->alpha = mp.S_next.alpha;
        state->hdot = mp.S_next.hdot;
        state->adot = mp.S_next.adot;
    }
    return rc;
}

int lbfsi_batch_remove(lbfsi_batch b, int slot) {
    if (!b || slot < 0 || slot >= (int)b->slots.size() || !b->slots[slot].used)
        return lbfsi::set_error(LBFSI_EINVAL, "invalid slot");
    const cudaError_t e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return cuda_err(e, "batch remove");
    Slot& s = b->slots[slot];
    release_slot_memory(b, s);
    drop_mesh(b, s.mesh);
    if (!s.finished) b->dirty = true;
    s = Slot{};
    return LBFSI_OK;
}

int lbfsi_batch_memory(lbfsi_batch b, size_t* free_bytes, size_t* largest_free) {
    if (!b) return lbfsi::set_error(LBFSI_EINVAL, "null batch");
    if (free_bytes) *free_bytes = b->pool.free_bytes();
    if (largest_free) *largest_free = b->pool.largest();
    return LBFSI_OK;
}

}  // extern "C"
