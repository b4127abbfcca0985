// dugks_batch.cu -- many independent grids per launch (declared in include/dugks.h).
//
// Host side of the batch: per-grid device memory and descriptors (BatchGrid), the
// work list of strip segments, the launches of a group of steps and their CUDA-graph
// replay. The arithmetic is the row march's, unchanged.
//
// Nothing on the path of a running batch waits for the device: grid memory comes
// from a stream-ordered pool of the batch's own and goes back to it in stream
// order, descriptors and initial fields are uploaded from pinned staging buffers,
// results are read out into pinned buffers, and every host buffer or graph that
// the stream may still use is released only once a fence (an event recorded on
// the stream, numbered in order) shows the stream has passed it. So a server can
// add, retire and collect grids while steps are in flight.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <map>
#include <string>
#include <tuple>
#include <vector>

#include "../../include/dugks.h"
#include "dugks_host.h"
#include "dugks_internal.h"

using namespace dugks;
using namespace dugks::host;

namespace {

struct Slot {
    bool used = false;
    bool retiring = false;   // read-out enqueued (dugks_batch_retire), result not yet collected
    int nx = 0, ny = 0, pitch = 0;
    size_t plane = 0;
    void *X[2] = {nullptr, nullptr};
    void *phi[3] = {nullptr, nullptr, nullptr};
    int64_t step = 0, target = -1;
    bool mass_known = false;        // h_mass of this slot is the mass of its state
    int vel_kind = DUGKS_VEL_UNIFORM;
    double vel[3] = {0, 0, 0};
    uint64_t ticket = 0;            // fence after the read-out
    void *pinned = nullptr;         // host buffer the read-out lands in
    size_t pinned_bytes = 0;
};

// what follows the status word (dugks_batch_mass)
constexpr size_t MASS_COUNT = 16, MASS_PART = MASS_COUNT + MASS_LIST * sizeof(unsigned);
constexpr size_t STATUS_BYTES = MASS_PART + (size_t)MASS_LIST * MASS_TILES * sizeof(double);

// pinned host buffers kept for reuse beyond this are given back
constexpr size_t PINNED_KEEP = (size_t)1 << 30;

}  // namespace

struct dugks_batch {
    dugks_params p{};
    int dev = 0, sms = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    size_t tsize = 4, ssize = 4;
    int nphi = 2;
    int variant = 4;    // segment length: by the rule of march_plan
    MarchPlan plan{};
    MarchWork work;             // segments of the grids that advance, and their sizes there by slot (0: none)
    std::vector<int2> counted;
    int rows = 0;       // the longest segment of the work list
    int ctas = 0;
    int resident = 0, resident_cols = 0, resident_rows = 0;   // CTAs that the GPU holds, for segments of that shape
    int ctas_req = 0;   // 0: resident CTAs (grid-stride); < 0: one CTA per segment; > 0: at most that many
    std::vector<Slot> slots;
    cudaMemPool_t pool = nullptr;   // grid memory, descriptors and the work list
    // device side
    void *d_grids = nullptr;
    int grids_cap = 0;
    int4 *d_items = nullptr;
    int items_cap = 0, nitems = 0;
    int *d_status = nullptr;     // status word, then the counters and the tiles' sums of dugks_batch_mass
    double *h_mass = nullptr;    // pinned: its results, by slot
    size_t h_mass_bytes = 0;
    bool mass_asked = false;     // a mass of the present state has been asked for
    void *d_tmp = nullptr;       // phi read-out of the waiting call
    size_t tmp_bytes = 0;
    bool dirty = true;
    cudaGraphExec_t graph = nullptr;
    std::vector<unsigned char> coefs, uniform;
    // fences: events recorded on the stream with increasing tickets
    std::deque<std::pair<uint64_t, cudaEvent_t>> fences;
    std::vector<cudaEvent_t> spare_events;
    uint64_t next_ticket = 1, reached = 0;
    // pinned host buffers free for reuse (by size), and those waiting for a fence
    std::multimap<size_t, void *> pinned_free;
    size_t pinned_free_bytes = 0;
    std::vector<std::tuple<uint64_t, void *, size_t>> pinned_later;
    std::vector<std::pair<uint64_t, cudaGraphExec_t>> graphs_later;
    int sticky = DUGKS_OK;
    std::string err;
};

namespace {

int bfail(dugks_batch *b, int code, const std::string &msg) {
    if (b) {
        if (b->sticky == DUGKS_OK) b->sticky = code;
        b->err = msg;
    }
    return code;
}
int bcuda(dugks_batch *b, cudaError_t e, const char *where) {
    return bfail(b, DUGKS_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

bool fp64(const dugks_batch *b) { return b->p.precision == DUGKS_FP64; }

// ---- stream-ordered device memory ------------------------------------------
cudaError_t pool_alloc(dugks_batch *b, void **p, size_t bytes) {
    cudaError_t e = dev_malloc_pool(p, bytes, b->pool, b->stream);
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
    }
    return e;
}
template <typename P>
cudaError_t pool_alloc(dugks_batch *b, P **p, size_t bytes) {
    return pool_alloc(b, reinterpret_cast<void **>(p), bytes);
}
// freed once the work queued on the stream before it has run
void pool_free(dugks_batch *b, void *p) {
    if (p) cudaFreeAsync(p, b->stream);
}

// ---- fences -----------------------------------------------------------------
void consume_not_ready() {
    if (cudaPeekAtLastError() == cudaErrorNotReady) cudaGetLastError();
}

int fence(dugks_batch *b, uint64_t *ticket) {
    cudaEvent_t ev = nullptr;
    if (!b->spare_events.empty()) {
        ev = b->spare_events.back();
        b->spare_events.pop_back();
    } else {
        cudaError_t e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
        if (e != cudaSuccess) return bcuda(b, e, "fence event");
    }
    cudaError_t e = cudaEventRecord(ev, b->stream);
    if (e != cudaSuccess) {
        b->spare_events.push_back(ev);
        return bcuda(b, e, "fence record");
    }
    *ticket = b->next_ticket++;
    b->fences.emplace_back(*ticket, ev);
    return DUGKS_OK;
}

void pinned_put(dugks_batch *b, void *p, size_t bytes) {
    if (!p) return;
    b->pinned_free.emplace(bytes, p);
    b->pinned_free_bytes += bytes;
    while (b->pinned_free_bytes > PINNED_KEEP && !b->pinned_free.empty()) {
        auto it = std::prev(b->pinned_free.end());   // the largest goes first
        b->pinned_free_bytes -= it->first;
        cudaFreeHost(it->second);
        b->pinned_free.erase(it);
    }
}

// a pinned buffer of at least `bytes` (reused when one of at most twice the size is free)
int pinned_get(dugks_batch *b, size_t bytes, void **p, size_t *got) {
    bytes = std::max<size_t>(bytes, 256);
    auto it = b->pinned_free.lower_bound(bytes);
    if (it != b->pinned_free.end() && it->first <= 2 * bytes) {
        *p = it->second;
        *got = it->first;
        b->pinned_free_bytes -= it->first;
        b->pinned_free.erase(it);
        return DUGKS_OK;
    }
    if (cudaMallocHost(p, bytes) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return DUGKS_ENOMEM;
    }
    *got = bytes;
    return DUGKS_OK;
}

// gives `p` back once the stream has passed fence `ticket`
void pinned_later(dugks_batch *b, void *p, size_t bytes, uint64_t ticket) {
    if (p) b->pinned_later.emplace_back(ticket, p, bytes);
}

// moves b->reached over every fence the stream has passed and releases what
// waited for them
int advance(dugks_batch *b) {
    int r = DUGKS_OK;
    while (!b->fences.empty()) {
        cudaError_t e = cudaEventQuery(b->fences.front().second);
        if (e == cudaErrorNotReady) {
            consume_not_ready();
            break;
        }
        if (e != cudaSuccess) {
            r = bcuda(b, e, "batch fence");
            break;
        }
        b->reached = b->fences.front().first;
        b->spare_events.push_back(b->fences.front().second);
        b->fences.pop_front();
    }
    auto &pl = b->pinned_later;
    for (size_t i = 0; i < pl.size();) {
        if (std::get<0>(pl[i]) <= b->reached) {
            pinned_put(b, std::get<1>(pl[i]), std::get<2>(pl[i]));
            pl[i] = pl.back();
            pl.pop_back();
        } else {
            i++;
        }
    }
    auto &gl = b->graphs_later;
    for (size_t i = 0; i < gl.size();) {
        if (gl[i].first <= b->reached) {
            cudaGraphExecDestroy(gl[i].second);
            gl[i] = gl.back();
            gl.pop_back();
        } else {
            i++;
        }
    }
    return r;
}

// blocks until the stream has passed fence `ticket`
int wait_ticket(dugks_batch *b, uint64_t ticket) {
    for (auto &f : b->fences)
        if (f.first >= ticket) {
            cudaError_t e = cudaEventSynchronize(f.second);
            if (e != cudaSuccess) return bcuda(b, e, "batch fence wait");
            break;
        }
    return advance(b);
}


size_t plane_of(int nx, int ny, int *pitch_out) {
    const int pitch = (nx + 2 * GHOST + 31) / 32 * 32;
    if (pitch_out) *pitch_out = pitch;
    return (size_t)(ny + 2 * GHOST) * pitch;
}

int resident_ctas(dugks_batch *b) {
    if (b->resident > 0 && b->resident_cols == b->plan.cols && b->resident_rows == b->rows) return b->resident;
    int per = 1;
    switch (b->p.precision) {
    case DUGKS_FP64: per = Launch<double, double>::batch_ctas_per_sm(b->p.flux, b->plan.cols, b->rows); break;
    case DUGKS_FP32: per = Launch<float, float>::batch_ctas_per_sm(b->p.flux, b->plan.cols, b->rows); break;
    default: per = Launch<float, __half>::batch_ctas_per_sm(b->p.flux, b->plan.cols, b->rows); break;
    }
    b->resident = std::max(1, b->sms) * std::max(1, per);
    b->resident_cols = b->plan.cols;
    b->resident_rows = b->rows;
    return b->resident;
}

// By default resident CTAs striding over a list that is little longer (32 grids of 64^2 to
// 512^2: 79.5 us a step against 82.8), else one CTA a segment, which the hardware hands out as
// others finish (512 such grids: 897 us against 1353). In FP64 a warp that joins a busy scheduler
// halves its rate, so the resident set is kept (32 grids: 1966 us against 2389).
void choose_ctas(dugks_batch *b) {
    b->ctas = b->ctas_req < 0 ? INT_MAX : b->ctas_req;
    if (b->ctas_req != 0) return;
    b->ctas = resident_ctas(b);
    if (!fp64(b) && 2 * (int64_t)b->nitems > 3 * (int64_t)b->ctas) b->ctas = INT_MAX;
}

template <typename T>
void fill_uniform(dugks_batch *b) {
    BatchUniform<T> u;
    std::memset(&u, 0, sizeof u);
    const double dt = b->p.cfl, tau = 3.0 * b->p.M, h = 0.5 * dt;
    const double bb = (dt + h) / (2.0 * tau + dt);   // bar f^+ = X + b (g - X)
    u.b = (T)bb;
    u.c2 = (T)(h / (2.0 * tau + h));
    u.c3 = (T)(tau * h / (2.0 * tau + h));
    u.be1 = (T)(4.0 / 3.0 * bb);
    u.ga1 = (T)dt;
    u.tau = (T)tau;
    u.theta_c = (T)(-4.0 / (b->p.W * (b->p.phiA - b->p.phiB)));
    u.phiA = (T)b->p.phiA;
    u.phiB = (T)b->p.phiB;
    u.inv_dt = (T)(1.0 / dt);
    u.qscale = (T)256.0;
    u.qinv = (T)(1.0 / 256.0);
    u.dt = dt;
    u.dtphiu = b->p.dtphiu;
    u.status = b->d_status;
    b->uniform.assign(reinterpret_cast<unsigned char *>(&u), reinterpret_cast<unsigned char *>(&u) + sizeof u);
    const MarchCoefs<T> cf = make_march_coefs<T>(b->p.order, h);
    b->coefs.assign(reinterpret_cast<const unsigned char *>(&cf),
                    reinterpret_cast<const unsigned char *>(&cf) + sizeof cf);
}

// the current graph is destroyed once the stream has passed its launches
void drop_graph(dugks_batch *b) {
    if (!b->graph) return;
    uint64_t t = 0;
    if (fence(b, &t) == DUGKS_OK) {
        b->graphs_later.emplace_back(t, b->graph);
    } else {
        cudaStreamSynchronize(b->stream);
        cudaGraphExecDestroy(b->graph);
    }
    b->graph = nullptr;
}

// Descriptors and work list of all grids, uploaded in stream order from pinned
// staging (the steps already queued keep the old ones). Grids that reached their
// target, or are retiring, keep a frozen descriptor and contribute no tiles.
template <typename T>
int rebuild_t(dugks_batch *b) {
    drop_graph(b);
    const int n = (int)b->slots.size();
    if (n > b->grids_cap) {
        const int cap = std::max(16, n * 2);
        void *grids = nullptr;
        if (pool_alloc(b, &grids, (size_t)cap * sizeof(BatchGrid<T>)) != cudaSuccess)
            return bfail(b, DUGKS_ENOMEM, "batch descriptors");
        pool_free(b, b->d_grids);
        b->d_grids = grids;
        b->grids_cap = cap;
    }
    const MarchShape &shape = march_shape(2, b->p.flux);
    auto live = [](const Slot &s) { return s.used && !s.retiring && (s.target < 0 || s.step < s.target); };
    std::vector<int2> sizes;
    b->counted.resize(n, make_int2(0, 0));
    for (int i = 0; i < n; i++) {
        const Slot &s = b->slots[i];
        const int2 now = live(s) ? make_int2(s.nx, s.ny) : make_int2(0, 0);
        int2 &was = b->counted[i];
        if (now.x) sizes.push_back(now);
        if (now.x == was.x && now.y == was.y) continue;
        if (was.x) b->work.count(shape, was, -1);
        if (now.x) b->work.count(shape, now, 1);
        was = now;
    }
    b->plan = march_plan(shape, b->variant, b->work, sizes.data(), (int)sizes.size(), b->p.precision, b->sms);
    int nitems = 0;
    b->rows = 1;
    for (const int2 &q : sizes) {
        nitems += march_strips(b->plan.cols, q.x) * march_segments(b->plan.rows, q.y);
        b->rows = std::max(b->rows, march_segment_rows(b->plan.rows, q.y));
    }
    b->nitems = nitems;
    choose_ctas(b);
    if (nitems > b->items_cap) {
        pool_free(b, b->d_items);
        b->d_items = nullptr;
        b->items_cap = 0;
        const int cap = nitems * 2;
        if (pool_alloc(b, &b->d_items, (size_t)cap * sizeof(int4)) != cudaSuccess)
            return bfail(b, DUGKS_ENOMEM, "batch work list");
        b->items_cap = cap;
    }
    const size_t gbytes = (size_t)std::max(n, 1) * sizeof(BatchGrid<T>);
    const size_t ibytes = (size_t)std::max(nitems, 1) * sizeof(int4);
    void *hg = nullptr, *hi = nullptr;
    size_t hgs = 0, his = 0;
    if (pinned_get(b, gbytes, &hg, &hgs) != DUGKS_OK) return bfail(b, DUGKS_ENOMEM, "descriptor staging");
    if (pinned_get(b, ibytes, &hi, &his) != DUGKS_OK) {
        pinned_put(b, hg, hgs);
        return bfail(b, DUGKS_ENOMEM, "work-list staging");
    }
    BatchGrid<T> *G = static_cast<BatchGrid<T> *>(hg);
    int4 *I = static_cast<int4 *>(hi);
    int k = 0;
    for (int i = 0; i < n; i++) {
        const Slot &s = b->slots[i];
        BatchGrid<T> &d = G[i];
        std::memset(&d, 0, sizeof d);   // step 0, target 0: frozen
        if (!s.used || s.retiring) continue;
        for (int q = 0; q < 2; q++) d.X[q] = s.X[q];
        for (int q = 0; q < b->nphi; q++) d.phi[q] = static_cast<T *>(s.phi[q]);
        d.plane = s.plane;
        d.nx = s.nx;
        d.ny = s.ny;
        d.pitch = s.pitch;
        d.tile_w = march_width(b->plan.cols, s.nx);
        d.vel_kind = s.vel_kind;
        for (int q = 0; q < 3; q++) d.vp[q] = s.vel[q];
        d.step = s.step;
        d.target = s.target < 0 ? (long long)1 << 62 : s.target;
        if (!live(s)) continue;
        const int strips = march_strips(b->plan.cols, s.nx), rows = march_segment_rows(b->plan.rows, s.ny);
        for (int y = 0; y < s.ny; y += rows)
            for (int x = 0; x < strips; x++) I[k++] = make_int4(i, x, y, std::min(rows, s.ny - y));
    }
    cudaError_t e = cudaSuccess;
    if (n > 0) e = cudaMemcpyAsync(b->d_grids, hg, (size_t)n * sizeof(BatchGrid<T>), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess && nitems > 0)
        e = cudaMemcpyAsync(b->d_items, hi, (size_t)nitems * sizeof(int4), cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess)
        e = launch_batch_advance<T>(static_cast<BatchGrid<T> *>(b->d_grids), n, 0, b->p.cfl, b->stream);
    uint64_t t = 0;
    const int fr = e == cudaSuccess ? fence(b, &t) : DUGKS_ECUDA;
    if (fr == DUGKS_OK) {
        pinned_later(b, hg, hgs, t);
        pinned_later(b, hi, his, t);
    } else {
        cudaStreamSynchronize(b->stream);
        pinned_put(b, hg, hgs);
        pinned_put(b, hi, his);
    }
    if (e != cudaSuccess) return bcuda(b, e, "batch descriptors upload");
    if (fr != DUGKS_OK) return fr;
    b->dirty = false;
    return DUGKS_OK;
}

int rebuild(dugks_batch *b) { return fp64(b) ? rebuild_t<double>(b) : rebuild_t<float>(b); }

// `n` steps (at most GRAPH_STEPS) and the step counters
template <typename T, typename ST>
cudaError_t launch_steps(dugks_batch *b, int n) {
    const BatchUniform<T> &u = *reinterpret_cast<const BatchUniform<T> *>(b->uniform.data());
    const MarchCoefs<T> &cf = *reinterpret_cast<const MarchCoefs<T> *>(b->coefs.data());
    BatchGrid<T> *G = static_cast<BatchGrid<T> *>(b->d_grids);
    for (int i = 0; i < n; i++)
        if (cudaError_t e = Launch<T, ST>::batch_step(u, cf, G, b->d_items, b->nitems, b->rows, i, b->p.flux,
                                                      b->plan.cols, b->ctas, b->stream);
            e != cudaSuccess)
            return e;
    return launch_batch_advance<T>(G, (int)b->slots.size(), n, u.dt, b->stream);
}

cudaError_t steps(dugks_batch *b, int n) {
    switch (b->p.precision) {
    case DUGKS_FP64: return launch_steps<double, double>(b, n);
    case DUGKS_FP32: return launch_steps<float, float>(b, n);
    default: return launch_steps<float, __half>(b, n);
    }
}

template <typename T, typename ST>
StepParams<T> slot_view(const dugks_batch *b, const Slot &s) {
    StepParams<T> q;
    std::memset(&q, 0, sizeof q);
    q.nx = s.nx;
    q.ny = s.ny;
    q.pitch = s.pitch;
    q.plane = s.plane;
    q.status = b->d_status;
    q.theta_c = (T)(-4.0 / (b->p.W * (b->p.phiA - b->p.phiB)));
    q.phiA = (T)b->p.phiA;
    q.phiB = (T)b->p.phiB;
    q.vel_kind = s.vel_kind;
    q.vp0 = (T)s.vel[0];
    q.vp1 = (T)s.vel[1];
    q.vp2 = (T)s.vel[2];
    q.qscale = (T)256.0;
    q.qinv = (T)(1.0 / 256.0);
    q.X = s.X[s.step & 1];
    if (Store<T, ST>::phi_plane) q.phi_cur = static_cast<const T *>(s.phi[(3 - (int)(s.step % 3)) % 3]);
    return q;
}

// The masses of the given slots, queued into h_mass. Tiles go by the grid's size alone, so that the sum's order
// (and its last bit) is the same in every batch: 8 rows (one a warp) of at most 1024 cells while that
// gives up to 512 tiles, about three CTAs an SM; more rows from there up. At most 64 columns of tiles, so
// never more than 576.
template <typename T, typename ST>
cudaError_t queue_masses(dugks_batch *b, const std::vector<int> &ids) {
    char *base = reinterpret_cast<char *>(b->d_status);
    for (size_t first = 0; first < ids.size(); first += MASS_LIST) {
        MassList<T> list;
        int tiles = 0;
        const int n = (int)std::min<size_t>(MASS_LIST, ids.size() - first);
        for (int i = 0; i < n; i++) {
            const Slot &s = b->slots[ids[first + i]];
            const StepParams<T> q = slot_view<T, ST>(b, s);
            const int w = std::max(std::min(s.nx, 1024), (s.nx + 63) / 64);
            const int64_t across = (s.nx + w - 1) / w;
            const int h = (int)std::max<int64_t>(8, (s.ny * across + 511) / 512);
            list.g[i] = MassGrid<T>{q.X, q.phi_cur, s.plane, s.nx, s.ny, s.pitch, w, h, ids[first + i]};
            tiles = std::max(tiles, (int)across * ((s.ny + h - 1) / h));
        }
        cudaError_t e = Launch<T, ST>::mass(list, n, tiles, reinterpret_cast<double *>(base + MASS_PART),
                                            reinterpret_cast<unsigned *>(base + MASS_COUNT), b->h_mass, b->d_status,
                                            b->stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// The initial equilibrium of a new grid, queued on the stream: the ghost-bordered
// field goes through pinned staging into a pool buffer that is freed in stream
// order after the init kernel.
template <typename T, typename ST>
int init_slot(dugks_batch *b, Slot &s, const double *phi0) {
    const size_t bytes = s.plane * sizeof(T);
    void *d_phi0 = nullptr;
    if (pool_alloc(b, &d_phi0, bytes) != cudaSuccess) return DUGKS_ENOMEM;
    void *h = nullptr;
    size_t hs = 0;
    if (pinned_get(b, bytes, &h, &hs) != DUGKS_OK) {
        pool_free(b, d_phi0);
        return DUGKS_ENOMEM;
    }
    fill_ghosted_plane(static_cast<T *>(h), phi0, s.nx, s.ny, s.pitch);
    cudaError_t e = cudaMemcpyAsync(d_phi0, h, bytes, cudaMemcpyHostToDevice, b->stream);
    if (e == cudaSuccess) {
        StepParams<T> q = slot_view<T, ST>(b, s);
        q.t = (T)0;
        q.out1 = s.X[0];
        q.phi_out = static_cast<T *>(s.phi[0]);
        e = Launch<T, ST>::init(q, static_cast<const T *>(d_phi0), (T)(0.5 * b->p.cfl), b->p.order, b->stream);
    }
    pool_free(b, d_phi0);
    uint64_t t = 0;
    if (e == cudaSuccess && fence(b, &t) == DUGKS_OK) {
        pinned_later(b, h, hs, t);
    } else {
        cudaStreamSynchronize(b->stream);
        cudaGetLastError();
        pinned_put(b, h, hs);
    }
    return e == cudaSuccess ? DUGKS_OK : bcuda(b, e, "batch init");
}

// device memory back to the pool in stream order; a pending read-out's host
// buffer waits for its fence
void free_slot(dugks_batch *b, Slot &s) {
    for (void *q : {s.X[0], s.X[1], s.phi[0], s.phi[1], s.phi[2]}) pool_free(b, q);
    if (s.pinned) pinned_later(b, s.pinned, s.pinned_bytes, s.ticket);
    s = Slot();
}

int check_common(const dugks_params *p) {
    if (!p) return DUGKS_EINVAL;
    if (!(p->W > 0) || !(p->M > 0) || !(p->cfl > 0) || p->cfl > 1.0) return DUGKS_EINVAL;
    if ((p->order != 2 && p->order != 3) || (p->flux != 0 && p->flux != 1) || p->stages != 2) return DUGKS_EINVAL;
    if (p->precision < DUGKS_FP64 || p->precision > DUGKS_FP16F) return DUGKS_EINVAL;
    if (!(p->phiA != p->phiB)) return DUGKS_EINVAL;
    return DUGKS_OK;
}

}  // namespace

extern "C" {

int dugks_batch_create(const dugks_params *common, void *cuda_stream, dugks_batch **out) {
    if (!out) return DUGKS_EINVAL;
    *out = nullptr;
    int r = check_common(common);
    if (r != DUGKS_OK) return r;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev == 0) {
        cudaGetLastError();
        return DUGKS_ECUDA;
    }
    dugks_batch *b = new dugks_batch();
    b->p = *common;
    cudaGetDevice(&b->dev);
    if (cuda_stream) {
        b->stream = static_cast<cudaStream_t>(cuda_stream);
    } else if (cudaStreamCreateWithFlags(&b->stream, cudaStreamNonBlocking) == cudaSuccess) {
        b->own_stream = true;
    } else {
        delete b;
        return DUGKS_ECUDA;
    }
    b->tsize = fp64(b) ? 8 : 4;
    b->ssize = common->precision == DUGKS_FP64 ? 8 : common->precision == DUGKS_FP32 ? 4 : 2;
    b->nphi = common->precision == DUGKS_FP64 ? 2 : 3;   // FP32 and FP16F: phi is a plane of its own
    cudaDeviceGetAttribute(&b->sms, cudaDevAttrMultiProcessorCount, b->dev);
    if (const char *ev = std::getenv("DUGKS_FAST_VARIANT")) {
        const int v = std::atoi(ev);
        if (v >= 0 && v < FAST_VARIANTS) b->variant = v;
    }
    int pools = 0;
    cudaDeviceGetAttribute(&pools, cudaDevAttrMemoryPoolsSupported, b->dev);
    cudaMemPoolProps props;
    std::memset(&props, 0, sizeof props);
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = b->dev;
    if (!pools || cudaMemPoolCreate(&b->pool, &props) != cudaSuccess) {
        cudaGetLastError();
        b->pool = nullptr;
        dugks_batch_destroy(b);
        return DUGKS_ECUDA;
    }
    if (dev_malloc(&b->d_status, STATUS_BYTES) != cudaSuccess) {
        cudaGetLastError();
        dugks_batch_destroy(b);
        return DUGKS_ENOMEM;
    }
    cudaMemset(b->d_status, 0, MASS_PART);
    if (fp64(b)) fill_uniform<double>(b);
    else fill_uniform<float>(b);
    *out = b;
    return DUGKS_OK;
}

size_t dugks_batch_grid_bytes(const dugks_params *common, int32_t nx, int32_t ny) {
    if (!common || nx < 8 || ny < 8) return 0;
    const size_t plane = plane_of(nx, ny, nullptr);
    const size_t ts = common->precision == DUGKS_FP64 ? 8 : 4;
    const size_t ss = common->precision == DUGKS_FP64 ? 8 : common->precision == DUGKS_FP32 ? 4 : 2;
    const int nphi = common->precision == DUGKS_FP64 ? 2 : 3;
    return 2 * 9 * plane * ss + (size_t)nphi * plane * ts;
}

int dugks_batch_add(dugks_batch *b, int32_t nx, int32_t ny, const double *phi0_host, int vel_kind,
                    const double *vel_params, int64_t target_steps, int32_t *grid_id) {
    if (!b || !phi0_host || !grid_id || nx < 8 || ny < 8) return DUGKS_EINVAL;
    if (b->sticky != DUGKS_OK) return b->sticky;
    if (vel_kind != DUGKS_VEL_UNIFORM && vel_kind != DUGKS_VEL_ROTATION && vel_kind != DUGKS_VEL_VORTEX)
        return bfail(b, DUGKS_EINVAL, "batch grids take uniform, rotation or vortex velocity");
    if (!vel_params) return bfail(b, DUGKS_EINVAL, "velocity parameters missing");
    if (vel_kind == DUGKS_VEL_VORTEX && (!(vel_params[0] > 0) || !(vel_params[2] > 0)))
        return bfail(b, DUGKS_EINVAL, "vortex needs (L > 0, U, T > 0)");
    for (size_t i = 0; i < (size_t)nx * ny; i++)
        if (!std::isfinite(phi0_host[i])) return DUGKS_ENONFINITE;
    cudaSetDevice(b->dev);
    int r = advance(b);
    if (r != DUGKS_OK) return r;
    Slot s;
    s.used = true;
    s.nx = nx;
    s.ny = ny;
    s.plane = plane_of(nx, ny, &s.pitch);
    s.vel_kind = vel_kind;
    const int nv = vel_kind == DUGKS_VEL_UNIFORM ? 2 : 3;
    for (int k = 0; k < nv; k++) s.vel[k] = vel_params[k];
    s.target = target_steps;
    bool ok = true;
    for (int k = 0; k < 2 && ok; k++) ok = pool_alloc(b, &s.X[k], 9 * s.plane * b->ssize) == cudaSuccess;
    for (int k = 0; k < b->nphi && ok; k++) ok = pool_alloc(b, &s.phi[k], s.plane * b->tsize) == cudaSuccess;
    if (!ok) {
        free_slot(b, s);
        return DUGKS_ENOMEM;   // not sticky: the caller may retry later
    }
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < 2 && e == cudaSuccess; k++) e = cudaMemsetAsync(s.X[k], 0, 9 * s.plane * b->ssize, b->stream);
    for (int k = 0; k < b->nphi && e == cudaSuccess; k++)
        e = cudaMemsetAsync(s.phi[k], 0, s.plane * b->tsize, b->stream);
    if (e != cudaSuccess) {
        free_slot(b, s);
        return bcuda(b, e, "batch grid clear");
    }
    switch (b->p.precision) {
    case DUGKS_FP64: r = init_slot<double, double>(b, s, phi0_host); break;
    case DUGKS_FP32: r = init_slot<float, float>(b, s, phi0_host); break;
    default: r = init_slot<float, __half>(b, s, phi0_host); break;
    }
    if (r != DUGKS_OK) {
        free_slot(b, s);
        return r;
    }
    int id = -1;
    for (size_t i = 0; i < b->slots.size(); i++)
        if (!b->slots[i].used) {
            id = (int)i;
            break;
        }
    if (id < 0) {
        id = (int)b->slots.size();
        b->slots.push_back(Slot());
    }
    b->slots[id] = s;
    b->dirty = true;
    *grid_id = id;
    return DUGKS_OK;
}

int dugks_batch_remove(dugks_batch *b, int32_t grid_id) {
    if (!b || grid_id < 0 || grid_id >= (int)b->slots.size() || !b->slots[grid_id].used) return DUGKS_EINVAL;
    cudaSetDevice(b->dev);
    free_slot(b, b->slots[grid_id]);
    b->dirty = true;
    return advance(b);
}

int dugks_batch_retire(dugks_batch *b, int32_t grid_id, uint64_t *ticket) {
    if (!b || !ticket || grid_id < 0 || grid_id >= (int)b->slots.size() || !b->slots[grid_id].used ||
        b->slots[grid_id].retiring)
        return DUGKS_EINVAL;
    if (b->sticky != DUGKS_OK) return b->sticky;
    cudaSetDevice(b->dev);
    Slot &s = b->slots[grid_id];
    const size_t bytes = (size_t)s.nx * s.ny * sizeof(double);
    void *h = nullptr;
    size_t hs = 0;
    if (pinned_get(b, bytes, &h, &hs) != DUGKS_OK) return DUGKS_ENOMEM;   // not sticky
    // phi widened to FP64 into the state set the last step read (no longer needed:
    // 9 planes of at least 2 bytes hold ny * nx doubles), then one copy to the host
    double *d = static_cast<double *>(s.X[1 - (int)(s.step & 1)]);
    cudaError_t e;
    switch (b->p.precision) {
    case DUGKS_FP64: e = Launch<double, double>::phi64(slot_view<double, double>(b, s), d, b->stream); break;
    case DUGKS_FP32: e = Launch<float, float>::phi64(slot_view<float, float>(b, s), d, b->stream); break;
    default: e = Launch<float, __half>::phi64(slot_view<float, __half>(b, s), d, b->stream); break;
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, d, bytes, cudaMemcpyDeviceToHost, b->stream);
    if (e != cudaSuccess) {
        cudaStreamSynchronize(b->stream);
        cudaGetLastError();
        pinned_put(b, h, hs);
        return bcuda(b, e, "retire read-out");
    }
    uint64_t t = 0;
    int r = fence(b, &t);
    if (r != DUGKS_OK) {
        cudaStreamSynchronize(b->stream);
        pinned_put(b, h, hs);
        return r;
    }
    s.retiring = true;
    s.target = s.step;   // frozen where it stands
    s.ticket = t;
    s.pinned = h;
    s.pinned_bytes = hs;
    b->dirty = true;
    *ticket = t;
    return DUGKS_OK;
}

int dugks_batch_collect(dugks_batch *b, int32_t grid_id, double *out_host, int wait) {
    if (!b || !out_host || grid_id < 0 || grid_id >= (int)b->slots.size() || !b->slots[grid_id].used ||
        !b->slots[grid_id].retiring)
        return DUGKS_EINVAL;
    cudaSetDevice(b->dev);
    Slot &s = b->slots[grid_id];
    int r = advance(b);
    if (r != DUGKS_OK) return r;
    if (b->reached < s.ticket) {
        if (!wait) return DUGKS_EAGAIN;
        r = wait_ticket(b, s.ticket);
        if (r != DUGKS_OK) return r;
    }
    if (b->sticky != DUGKS_OK) return b->sticky;
    std::memcpy(out_host, s.pinned, (size_t)s.nx * s.ny * sizeof(double));
    pinned_put(b, s.pinned, s.pinned_bytes);
    s.pinned = nullptr;
    free_slot(b, s);
    b->dirty = true;
    return DUGKS_OK;
}

int dugks_batch_fence(dugks_batch *b, uint64_t *ticket) {
    if (!b || !ticket) return DUGKS_EINVAL;
    if (b->sticky != DUGKS_OK) return b->sticky;
    cudaSetDevice(b->dev);
    return fence(b, ticket);
}

int dugks_batch_reached(dugks_batch *b, uint64_t ticket, int32_t *done) {
    if (!b || !done || ticket >= b->next_ticket) return DUGKS_EINVAL;
    cudaSetDevice(b->dev);
    const int r = advance(b);
    *done = b->reached >= ticket ? 1 : 0;
    return r;
}

int dugks_batch_set_ctas(dugks_batch *b, int32_t ctas) {
    if (!b) return DUGKS_EINVAL;
    cudaSetDevice(b->dev);
    b->ctas_req = ctas;
    if (!b->dirty) choose_ctas(b);   // (else with the work list)
    drop_graph(b);   // the next replay is captured with the new grid size
    return DUGKS_OK;
}

int dugks_batch_step(dugks_batch *b, int64_t nsteps) {
    if (!b || nsteps < 0) return DUGKS_EINVAL;
    if (b->sticky != DUGKS_OK) return b->sticky;
    cudaSetDevice(b->dev);
    int ar = advance(b);
    if (ar != DUGKS_OK) return ar;
    if (b->dirty) {
        int r = rebuild(b);
        if (r != DUGKS_OK) return r;
    }
    if (nsteps > 0) {
        for (auto &s : b->slots) s.mass_known = false;
        b->mass_asked = false;
    }
    int64_t left = nsteps;
    cudaError_t e = cudaSuccess;
    while (left > 0 && e == cudaSuccess) {
        const int m = (int)std::min<int64_t>(left, GRAPH_STEPS);
        if (m == GRAPH_STEPS) {
            if (!b->graph) {   // capture a group once; replayed while the work list is unchanged
                cudaGraph_t g = nullptr;
                e = cudaStreamBeginCapture(b->stream, cudaStreamCaptureModeThreadLocal);
                if (e == cudaSuccess) e = steps(b, m);
                cudaError_t e2 = cudaStreamEndCapture(b->stream, &g);
                if (e == cudaSuccess) e = e2;
                if (e == cudaSuccess) e = cudaGraphInstantiate(&b->graph, g, 0);
                if (g) cudaGraphDestroy(g);
                if (e != cudaSuccess) break;
            }
            e = cudaGraphLaunch(b->graph, b->stream);
        } else {
            e = steps(b, m);
        }
        left -= m;
        for (auto &s : b->slots)
            if (s.used) s.step = s.target < 0 ? s.step + m : std::min(s.target, s.step + m);
    }
    if (e != cudaSuccess) return bcuda(b, e, "batch step");
    return DUGKS_OK;
}

int64_t dugks_batch_step_index(const dugks_batch *b, int32_t grid_id) {
    if (!b || grid_id < 0 || grid_id >= (int)b->slots.size() || !b->slots[grid_id].used) return -1;
    return b->slots[grid_id].step;
}

int64_t dugks_batch_active_cells(const dugks_batch *b) {
    if (!b) return 0;
    int64_t n = 0;
    for (auto &s : b->slots)
        if (s.used && (s.target < 0 || s.step < s.target)) n += (int64_t)s.nx * s.ny;
    return n;
}

int dugks_batch_read_phi(dugks_batch *b, int32_t grid_id, double *out_host) {
    if (!b || !out_host || grid_id < 0 || grid_id >= (int)b->slots.size() || !b->slots[grid_id].used)
        return DUGKS_EINVAL;
    if (b->sticky != DUGKS_OK) return b->sticky;
    cudaSetDevice(b->dev);
    const Slot &s = b->slots[grid_id];
    const size_t n = (size_t)s.nx * s.ny, bytes = n * sizeof(double);
    if (bytes > b->tmp_bytes) {
        cudaStreamSynchronize(b->stream);
        if (b->d_tmp) cudaFree(b->d_tmp);
        b->d_tmp = nullptr;
        b->tmp_bytes = 0;
        if (dev_malloc(&b->d_tmp, bytes) != cudaSuccess) {
            cudaGetLastError();
            return bfail(b, DUGKS_ENOMEM, "read-out buffer");
        }
        b->tmp_bytes = bytes;
    }
    // phi widened to double on the device, then one copy into the caller's buffer
    cudaError_t e;
    double *d = static_cast<double *>(b->d_tmp);
    switch (b->p.precision) {
    case DUGKS_FP64: e = Launch<double, double>::phi64(slot_view<double, double>(b, s), d, b->stream); break;
    case DUGKS_FP32: e = Launch<float, float>::phi64(slot_view<float, float>(b, s), d, b->stream); break;
    default: e = Launch<float, __half>::phi64(slot_view<float, __half>(b, s), d, b->stream); break;
    }
    if (e != cudaSuccess) return bcuda(b, e, "phi kernel");
    e = cudaMemcpyAsync(out_host, d, bytes, cudaMemcpyDeviceToHost, b->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(b->stream);
    return e == cudaSuccess ? b->sticky : bcuda(b, e, "read phi");
}

int dugks_batch_mass(dugks_batch *b, int32_t grid_id, double *out) {
    if (!b || !out || grid_id < 0 || grid_id >= (int)b->slots.size() || !b->slots[grid_id].used) return DUGKS_EINVAL;
    if (b->sticky != DUGKS_OK) return b->sticky;
    cudaSetDevice(b->dev);
    // One grid when a state is first asked; who asks for a second one is likely to ask for all (64 grids of 64^2:
    // 960 us one at a time, 200 together; 730 where every step summed every mass and the call copied it)
    if (!b->slots[grid_id].mass_known) {
        const size_t need = b->slots.size() * sizeof(double);
        if (b->h_mass_bytes < need) {   // (nothing is in flight into the old buffer)
            pinned_put(b, b->h_mass, b->h_mass_bytes);
            b->h_mass = nullptr;
            b->h_mass_bytes = 0;
            for (auto &s : b->slots) s.mass_known = false;
            void *h = nullptr;
            size_t hs = 0;
            if (pinned_get(b, 2 * need, &h, &hs) != DUGKS_OK) return bfail(b, DUGKS_ENOMEM, "mass buffer");
            b->h_mass = static_cast<double *>(h);
            b->h_mass_bytes = hs;
        }
        std::vector<int> ids{grid_id};
        if (b->mass_asked)
            for (int i = 0; i < (int)b->slots.size(); i++)
                if (i != grid_id && b->slots[i].used && !b->slots[i].mass_known) ids.push_back(i);
        cudaError_t e;
        switch (b->p.precision) {
        case DUGKS_FP64: e = queue_masses<double, double>(b, ids); break;
        case DUGKS_FP32: e = queue_masses<float, float>(b, ids); break;
        default: e = queue_masses<float, __half>(b, ids); break;
        }
        if (e != cudaSuccess) return bcuda(b, e, "batch mass");
        for (int i : ids) b->slots[i].mass_known = true;
        b->mass_asked = true;
    }
    cudaError_t e = cudaStreamSynchronize(b->stream);   // (the call waits, also where the mass is there)
    if (e != cudaSuccess) return bcuda(b, e, "batch mass");
    *out = b->h_mass[grid_id];
    if (!std::isfinite(*out)) return bfail(b, DUGKS_ENONFINITE, "the field holds NaN or Inf");
    return DUGKS_OK;
}

int dugks_batch_set_variant(dugks_batch *b, int variant) {
    if (!b || variant < 0 || variant >= FAST_VARIANTS) return DUGKS_EINVAL;
    cudaSetDevice(b->dev);
    cudaError_t e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return bcuda(b, e, "batch synchronize");
    b->variant = variant;
    b->dirty = true;
    return DUGKS_OK;
}

int dugks_batch_status(dugks_batch *b) {
    if (!b) return DUGKS_EINVAL;
    cudaSetDevice(b->dev);
    cudaError_t e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return bcuda(b, e, "batch synchronize");
    int flags = 0;
    e = cudaMemcpy(&flags, b->d_status, sizeof(int), cudaMemcpyDeviceToHost);
    if (e != cudaSuccess) return bcuda(b, e, "read status");
    if (flags & 2) return bfail(b, DUGKS_ETIMEOUT, "a device wait ran out");
    if (flags & 1) return bfail(b, DUGKS_ENONFINITE, "a grid holds NaN or Inf");
    return b->sticky;
}

const char *dugks_batch_last_error(const dugks_batch *b) { return b ? b->err.c_str() : "null batch"; }

void dugks_batch_destroy(dugks_batch *b) {
    if (!b) return;
    cudaSetDevice(b->dev);
    if (b->stream) cudaStreamSynchronize(b->stream);
    if (b->graph) cudaGraphExecDestroy(b->graph);
    b->graph = nullptr;
    for (auto &g : b->graphs_later) cudaGraphExecDestroy(g.second);
    if (b->pool) {
        for (auto &s : b->slots) free_slot(b, s);
        for (void *q : {b->d_grids, (void *)b->d_items}) pool_free(b, q);
        cudaStreamSynchronize(b->stream);
    }
    for (void *q : {(void *)b->d_status, b->d_tmp})
        if (q) cudaFree(q);
    for (auto &f : b->fences) cudaEventDestroy(f.second);
    for (cudaEvent_t ev : b->spare_events) cudaEventDestroy(ev);
    if (b->h_mass) cudaFreeHost(b->h_mass);
    for (auto &q : b->pinned_later) cudaFreeHost(std::get<1>(q));
    for (auto &q : b->pinned_free) cudaFreeHost(q.second);
    if (b->pool) cudaMemPoolDestroy(b->pool);
    if (b->own_stream && b->stream) cudaStreamDestroy(b->stream);
    delete b;
}

}  // extern "C"
