// ensemble.cu -- pools of independent runs advanced together by the batched
// cluster kernel (batch.cu): slot table, arena allocator, admission, the
// advance launches and result access.  The pool holds no device memory of
// its own: everything lives in the caller's arena.
//
// Arena layout: [descriptor table | order table | ticket + error word] then
// the runs, each a 256-byte-aligned block from a first-fit free list:
//   x[N], v[N] (float32), [x'[N], v'[N]: the sort's destination, when the run
//   sorts], E32[NG], E64[NG], phi[NG], rho[NG], rho_q_last[NG], history[H],
//   step counter.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <vector>

#include "pic_internal.cuh"
#include "staging.h"

using namespace pic;

namespace {

constexpr size_t kAlign = 256;
// least idle arena space for a read-back's device conversion: below it the
// pieces' launches and copies cost more than the host's own conversion
constexpr size_t kMinScratch = 256 * 1024;
size_t align_up(size_t v) { return (v + kAlign - 1) / kAlign * kAlign; }

struct RunLayout {
    size_t x, v, xa, va, E32, E64, phi, rho, rq, hist, step, total;
};

RunLayout run_layout(const pic_params *p, int history) {
    RunLayout L;
    const size_t n = (size_t)p->npart, ng = (size_t)p->ncell;
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off = align_up(off + b); return o; };
    L.x = take(4 * n);
    L.v = take(4 * n);
    L.xa = p->sort_interval > 0 ? take(4 * n) : 0;
    L.va = p->sort_interval > 0 ? take(4 * n) : 0;
    L.E32 = take(4 * ng);
    L.E64 = take(8 * ng);
    L.phi = take(8 * ng);
    L.rho = take(8 * ng);
    L.rq = take(8 * ng);
    L.hist = take((size_t)history * sizeof(pic_diag_row));
    L.step = take(8);
    L.total = off;
    return L;
}

struct TableLayout {
    size_t runs, order, scalars, total;
};

TableLayout table_layout(int max_slots) {
    TableLayout T;
    size_t off = 0;
    auto take = [&](size_t b) { size_t o = off; off = align_up(off + b); return o; };
    T.runs = take((size_t)max_slots * sizeof(BatchRun));
    T.order = take((size_t)max_slots * sizeof(int));
    T.scalars = take(2 * sizeof(unsigned));
    T.total = off;
    return T;
}

int check_cfg(const pic_pool_config *c) {
    if (!c || c->max_slots < 1 || c->ncell_max < 1 || c->ncell_max > PIC_NCELL_MAX ||
        c->history < 1)
        return PIC_EINVAL;
    return PIC_OK;
}

// The shape of a pool whose caller leaves it open: per-particle adds in the
// 64-register build, clusters of 8 blocks, and kPoolBlock threads a block, or
// twice that while every active run has a cluster of the larger blocks.
// Measured on 512 runs of 1e4-1e6 particles (ms per step of all, steps 0-20,
// 40-100 and 200-400): 0.61, 0.43, 0.40; MATCH in the 128-register build
// 3.0; QUAD 0.61, 0.44, 0.42; PAIR 0.47, 0.43, 0.43 (in lattice order, at the
// start, lanes share nodes and its runs combine; they mix within 50 steps).
// On 40 runs: 0.14, 0.11, 0.09 with 256 threads, 0.10, 0.07, 0.06 with 512.
constexpr int kPoolVariant = PIC_DEPOSIT_ATOMIC + 16;
constexpr int kPoolBlock = 256;

// variant + 16 (two blocks per SM, 64 registers) is accepted too.
int check_shape(int code, int cluster, int block, int ncell_max) {
    const int variant = code & 15;
    if (code >> 4 > 1) return PIC_EINVAL;
    if (variant != PIC_DEPOSIT_ATOMIC && variant != PIC_DEPOSIT_MATCH && variant != PIC_DEPOSIT_QUAD &&
        variant != PIC_DEPOSIT_PAIR)
        return PIC_EINVAL;
    if (cluster != 1 && cluster != 2 && cluster != 4 && cluster != 8) return PIC_EINVAL;
    if (block < 128 || block > 512 || block % 32) return PIC_EINVAL;
    const int P = (ncell_max + cluster - 1) / cluster;
    if (P > block) return PIC_EINVAL;   // one slice node per thread
    return PIC_OK;
}

int cuda_fail(cudaError_t e) {
    if (e == cudaSuccess) return PIC_OK;
    std::fprintf(stderr, "libpic: CUDA error %d: %s\n", (int)e, cudaGetErrorString(e));
    return PIC_ECUDA;
}

#define PIC_CUDA(call)                               \
    do {                                             \
        cudaError_t e_ = (call);                     \
        if (e_ != cudaSuccess) return cuda_fail(e_); \
    } while (0)

}  // namespace

struct pic_pool {
    pic_pool_config cfg{};
    cudaStream_t stream = nullptr;
    unsigned char *arena = nullptr;
    size_t arena_bytes = 0;
    TableLayout tab{};
    std::map<size_t, size_t> free_list;   // offset -> size
    size_t used = 0;
    struct Slot {
        bool used = false, needs_init = false;
        bool lost = false;            // in a launch whose wait ran out
        pic_params p{};
        size_t off = 0, size = 0;
        RunLayout lay{};
        BatchRun desc{};
        int64_t target = 0, done = 0;
        float *buf_x[2] = {nullptr, nullptr}, *buf_v[2] = {nullptr, nullptr};

        // The buffers holding the state after `done` steps: a sort precedes
        // every step n > 0 with n % S == 0, so floor((done - 1) / S) sorts
        // have run; each swaps the pair.
        void point_at_state() {
            const int S = p.sort_interval;
            const int cur = (S > 0 && done >= 1) ? (int)(((done - 1) / S) & 1) : 0;
            desc.x = buf_x[cur];
            desc.v = buf_v[cur];
            desc.xa = buf_x[1 - cur];
            desc.va = buf_v[1 - cur];
        }
    };
    std::vector<Slot> slots;
    std::vector<BatchRun> h_runs;
    std::vector<int> h_order;
    int variant = kPoolVariant, cluster = 8, block = kPoolBlock, nclusters = 1;
    int wide_clusters = 0;        // > 0: up to so many runs take blocks twice as large
    int sms = 0;
    int resident_sms = 0;         // SMs of the many-step launch (0: not available)
    bool many_step = true;        // few runs may take it (pic_pool_many_step)
    unsigned wait_limit = 0, wait_missing = 0;   // pic_pool_set_wait_limit
    pic::Staging stage;
    // what is handed out of the arena, or used of its idle space
    std::mutex arena_mutex;

    BatchRun *d_runs() const { return reinterpret_cast<BatchRun *>(arena + tab.runs); }
    int *d_order() const { return reinterpret_cast<int *>(arena + tab.order); }
    unsigned *d_next() const { return reinterpret_cast<unsigned *>(arena + tab.scalars); }
    unsigned *d_err() const { return d_next() + 1; }

    bool alloc(size_t bytes, size_t *off) {
        for (auto it = free_list.begin(); it != free_list.end(); ++it) {
            if (it->second >= bytes) {
                *off = it->first;
                const size_t rest = it->second - bytes;
                const size_t roff = it->first + bytes;
                free_list.erase(it);
                if (rest) free_list[roff] = rest;
                used += bytes;
                return true;
            }
        }
        return false;
    }

    // The largest free piece of the arena (for a call's own use).
    bool idle_space(size_t *off, size_t *bytes) const {
        *bytes = 0;
        for (const auto &kv : free_list)
            if (kv.second > *bytes) {
                *off = kv.first;
                *bytes = kv.second;
            }
        return *bytes > 0;
    }

    void release(size_t off, size_t bytes) {
        used -= bytes;
        auto it = free_list.emplace(off, bytes).first;
        auto nx = std::next(it);
        if (nx != free_list.end() && it->first + it->second == nx->first) {
            it->second += nx->second;
            free_list.erase(nx);
        }
        if (it != free_list.begin()) {
            auto pv = std::prev(it);
            if (pv->first + pv->second == it->first) {
                pv->second += it->second;
                free_list.erase(it);
            }
        }
    }
};

namespace {

int set_shape(pic_pool *pool, int variant, int cluster, int block) {
    int rc = check_shape(variant, cluster, block, pool->cfg.ncell_max);
    if (rc) return rc;
    const int nc = batch_max_clusters(variant, cluster, block, pool->cfg.ncell_max);
    if (nc < 1) return PIC_EINVAL;
    pool->variant = variant;
    pool->cluster = cluster;
    pool->block = block;
    pool->nclusters = nc;
    pool->wide_clusters = 0;      // a chosen shape is kept
    return PIC_OK;
}

// Upload the descriptors of `order` and launch one batched pass.
int launch(pic_pool *pool, const std::vector<int> &order, bool push) {
    if (order.empty()) return PIC_OK;
    for (size_t i = 0; i < order.size(); i++) pool->h_order[i] = order[i];
    for (int s : order) pool->h_runs[s] = pool->slots[s].desc;
    // the table is small; copy the whole of it
    PIC_CUDA(cudaMemcpyAsync(pool->d_runs(), pool->h_runs.data(),
                             pool->h_runs.size() * sizeof(BatchRun), cudaMemcpyHostToDevice,
                             pool->stream));
    PIC_CUDA(cudaMemcpyAsync(pool->d_order(), pool->h_order.data(), order.size() * sizeof(int),
                             cudaMemcpyHostToDevice, pool->stream));
    PIC_CUDA(cudaMemsetAsync(pool->d_next(), 0, sizeof(unsigned), pool->stream));
    BatchArgs a;
    a.runs = pool->d_runs();
    a.order = pool->d_order();
    a.nrun = (int)order.size();
    a.next = pool->d_next();
    a.err = pool->d_err();
    a.push = push ? 1 : 0;
    a.ng_max = pool->cfg.ncell_max;
    const bool wide = (int)order.size() <= pool->wide_clusters;
    int nc = wide ? pool->wide_clusters : pool->nclusters;
    if (nc > (int)order.size()) nc = (int)order.size();
    PIC_CUDA(launch_batch(a, pool->variant, pool->cluster, wide ? 2 * pool->block : pool->block, nc,
                          pool->stream));
    // the copies above read pageable host memory: wait so the next launch
    // may rewrite the host tables
    PIC_CUDA(cudaStreamSynchronize(pool->stream));
    return PIC_OK;
}

// ---- few active runs: the many-step launch (steps.cu) ---------------------------
//
// A cluster of 8 SMs per run leaves most of the GPU idle when few runs are
// active, and the largest run decides when the launch ends.  The many-step
// launch gives every run as many SMs as evens out the runs' times.

// Blocks of the runs in `order` on `sms` SMs: one for the diagnostics and at
// least one worker each, the rest one by one to the run that would take
// longest.  A step takes about 6 us and 1.5 us per 1024 cells, and a worker
// 0.4 ns a particle.  *time: of the launch (us); false when there are too many
// runs.
bool allot(const pic_pool *pool, const std::vector<int> &order, int sms, std::vector<int> *workers,
           double *time) {
    const int spare = sms - 2 * (int)order.size();
    if (spare < 0) return false;
    workers->assign(order.size(), 1);
    auto run_time = [&](size_t i) {
        const pic_pool::Slot &sl = pool->slots[order[i]];
        return sl.desc.steps * (6.0 + 1.5 * sl.p.ncell / 1024.0 +
                                0.4e-3 * (double)sl.p.npart / (*workers)[i]);
    };
    std::vector<std::pair<double, size_t>> heap;
    for (size_t i = 0; i < order.size(); i++) heap.emplace_back(run_time(i), i);
    std::make_heap(heap.begin(), heap.end());
    *time = 0.0;                      // of the runs that can use no more workers
    for (int k = 0; k < spare && !heap.empty();) {
        std::pop_heap(heap.begin(), heap.end());
        const double t = heap.back().first;
        const size_t i = heap.back().second;
        heap.pop_back();
        // a worker takes a group of 4 particles per thread at least
        const int64_t most = (pool->slots[order[i]].p.npart + 4 * kStepsPoolBlock - 1) / (4 * kStepsPoolBlock);
        if ((*workers)[i] < most && (*workers)[i] < kStepsMaxGrid - 2) {
            (*workers)[i]++;
            heap.emplace_back(run_time(i), i);
            std::push_heap(heap.begin(), heap.end());
            k++;
        } else {
            *time = std::max(*time, t);
        }
    }
    for (const auto &h : heap) *time = std::max(*time, h.first);
    return true;
}

// Time of the cluster launch (us): its longest run, on 8 SMs that other clusters
// share when there are more than fit side by side, or the whole work at the
// rate of a full GPU.
double cluster_time(const pic_pool *pool, const std::vector<int> &order) {
    const double each = 8 * (int)order.size() > pool->sms ? 0.1e-3 : 0.07e-3;
    double longest = 0.0, work = 0.0;
    for (int s : order) {
        const pic_pool::Slot &sl = pool->slots[s];
        longest = std::max(longest, sl.desc.steps * (14.0 + each * (double)sl.p.npart));
        work += (double)sl.desc.steps * (double)sl.p.npart;
    }
    return std::max(longest, work / 2.3e5);
}

// Whether the runs of `order` take the many-step launch, and its workers.
// Measured (us per step of all, cluster launch and this one):
//   runs of 1e4-1e6: 1 run 13-20, 5.8; 10 runs 51-78, 12; 24 runs 72-81, 23-26;
//     38 runs 123-135, 36-39; 60 runs 136, 89-96; 76 runs 150, 345
//   equal runs: 20 of 2e6 210, 133; 40 of 1e6 179, 190; 10 of 4e6 287, 120; 65 of
//     2e5 55, 78; 60 of 5e4 24, 24; 76 of 1e4 25, 9; 8 of 1.2e7 825, 276
bool resident(const pic_pool *pool, const std::vector<int> &order, std::vector<int> *workers) {
    if (!pool->resident_sms || !pool->many_step) return false;
    for (int s : order) {
        const pic_pool::Slot &sl = pool->slots[s];
        const int64_t S = sl.p.sort_interval;
        if (S > 0) {                  // a sort falls before a step n > 0 with n % S == 0
            const int64_t next = sl.done == 0 ? S : (sl.done + S - 1) / S * S;
            if (next < sl.done + sl.desc.steps) return false;
        }
        if (sl.p.ncell > kStepsMaxCells || sl.p.npart > (((int64_t)1 << 38) / sl.p.ncell)) return false;
    }
    double time = 0.0;
    if (!allot(pool, order, pool->resident_sms, workers, &time)) return false;
    for (size_t i = 0; i < order.size(); i++)       // a worker's counts share words with carries
        if (pool->slots[order[i]].p.npart / (*workers)[i] >= kPackedCount - 64) return false;
    return time < cluster_time(pool, order);
}

int read_error_word(pic_pool *pool, unsigned *err);

// Advance the runs of `order` by their steps; *done false (and nothing done) when
// the arena has no room for the launch's accumulators.  PIC_ETIMEOUT: a wait ran out;
// the runs of the launch are lost, the others are as before.
int launch_resident(pic_pool *pool, const std::vector<int> &order, const std::vector<int> &workers,
                    bool *done) {
    *done = false;
    size_t off = align_up(order.size() * sizeof(StepsArgs)), clear = off;
    struct Part { size_t acc, sync, partials; };
    std::vector<Part> parts(order.size());
    for (size_t i = 0; i < order.size(); i++) {     // what starts at zero, first
        parts[i].acc = off;
        off = align_up(off + (size_t)kStepsSlots * pool->slots[order[i]].p.ncell * 8);
        parts[i].sync = off;
        off = align_up(off + 4 * sizeof(unsigned));
    }
    const size_t cleared = off;
    for (size_t i = 0; i < order.size(); i++) {
        parts[i].partials = off;
        off = align_up(off + (size_t)kStepsSlots * kStepsMaxGrid * 16);
    }
    size_t soff = 0, sbytes = 0;
    std::lock_guard<std::mutex> lock(pool->arena_mutex);          // till the launch is done
    if (!pool->idle_space(&soff, &sbytes) || sbytes < off) return PIC_OK;
    unsigned char *mem = pool->arena + soff;
    std::vector<StepsArgs> args(order.size());
    int first = 0, ng_max = 1;
    for (size_t i = 0; i < order.size(); i++) {
        const pic_pool::Slot &sl = pool->slots[order[i]];
        const BatchRun &d = sl.desc;
        StepsArgs &a = args[i];
        a.x = d.x;
        a.v = d.v;
        a.n = d.n;
        a.E32 = d.E32;
        a.E64 = d.E64;
        a.phi = d.phi;
        a.rho = d.rho;
        a.rho_q_last = d.rho_q_last;
        a.acc = reinterpret_cast<unsigned long long *>(mem + parts[i].acc);
        a.partials = reinterpret_cast<double *>(mem + parts[i].partials);
        a.err = pool->d_err();
        a.sync = reinterpret_cast<unsigned *>(mem + parts[i].sync);
        a.base[0] = pool->wait_missing;
        a.base[1] = a.base[2] = 0;
        a.wait_limit = pool->wait_limit ? pool->wait_limit : kStepsWaitLimit;
        a.diag_blocks = 1;
        a.first_block = first;
        a.blocks = workers[i] + 1;
        a.log_copies = steps_pool_copies();
        a.hist = d.hist;
        a.hist_len = d.hist_len;
        a.step0 = sl.done;
        a.dstep = d.step;
        a.steps = d.steps;
        a.c = d.pc;
        a.weight_total = d.weight_total;
        a.k_rho = d.k_rho;
        a.k_e = d.k_e;
        a.k_phi = d.k_phi;
        a.k_mode = d.k_mode;
        a.dx = d.dx;
        a.mass = d.mass;
        first += a.blocks;
        ng_max = std::max(ng_max, sl.p.ncell);
    }
    PIC_CUDA(cudaMemcpyAsync(mem, args.data(), args.size() * sizeof(StepsArgs), cudaMemcpyHostToDevice,
                             pool->stream));
    PIC_CUDA(cudaMemsetAsync(mem + clear, 0, cleared - clear, pool->stream));
    PIC_CUDA(launch_steps_pool(reinterpret_cast<const StepsArgs *>(mem), (int)args.size(), first, ng_max,
                               pool->stream));
    // the scratch is free again, and the host's arguments read, when this is done
    unsigned err = 0;
    const int rc = read_error_word(pool, &err);
    if (rc) return rc;
    *done = true;
    if (!(err & kErrWait)) return PIC_OK;
    // the word is the pool's: what the other runs have set stays
    for (int s : order) pool->slots[s].lost = true;
    err &= ~kErrWait;
    PIC_CUDA(cudaMemcpyAsync(pool->d_err(), &err, sizeof(err), cudaMemcpyHostToDevice, pool->stream));
    PIC_CUDA(cudaStreamSynchronize(pool->stream));
    return PIC_ETIMEOUT;
}

bool slot_ok(const pic_pool *pool, int32_t slot) {
    return pool && slot >= 0 && slot < (int)pool->slots.size() && pool->slots[slot].used;
}

// Whether a run has results to read.
int readable(const pic_pool::Slot &sl) {
    return sl.lost ? PIC_ETIMEOUT : sl.needs_init ? PIC_ESTATE : PIC_OK;
}

// Wait for the stream and what was queued into the staging memory; the error
// word comes with it.  The caller holds the staging's mutex.
int finish_read(pic_pool *pool, unsigned *err) {
    *err = 0;
    cudaError_t e = pool->stage.add(err, pool->d_err(), sizeof(*err), pool->stream);
    const cudaError_t f = pool->stage.finish(pool->stream);
    if (e == cudaSuccess) e = f;
    return e == cudaSuccess ? PIC_OK : cuda_fail(e);
}

int finish_read(pic_pool *pool) {
    unsigned err;
    const int rc = finish_read(pool, &err);
    return rc ? rc : err ? PIC_EDEVICE : PIC_OK;
}

int read_error_word(pic_pool *pool, unsigned *err) {
    std::lock_guard<std::mutex> lock(pool->stage.mutex);
    return finish_read(pool, err);
}

int read_error(pic_pool *pool) {
    std::lock_guard<std::mutex> lock(pool->stage.mutex);
    return finish_read(pool);
}

}  // namespace

extern "C" {

int pic_pool_run_bytes(const pic_params *p, int32_t history, size_t *bytes) {
    if (!p || !bytes || history < 1) return PIC_EINVAL;
    int rc = validate_params(p);
    if (rc) return rc;
    if (p->precision != PIC_FP32_FIXED) return PIC_EINVAL;
    if (p->field_solver != PIC_SOLVER_EXACT || p->shape != PIC_SHAPE_CIC) return PIC_EINVAL;
    *bytes = run_layout(p, history).total;
    return PIC_OK;
}

int pic_pool_table_bytes(const pic_pool_config *cfg, size_t *bytes) {
    int rc = check_cfg(cfg);
    if (rc) return rc;
    if (!bytes) return PIC_EINVAL;
    *bytes = table_layout(cfg->max_slots).total;
    return PIC_OK;
}

int pic_pool_create(const pic_pool_config *cfg, void *arena, size_t arena_bytes, void *stream,
                    pic_pool **out) {
    if (!out) return PIC_EINVAL;
    *out = nullptr;
    int rc = check_cfg(cfg);
    if (rc) return rc;
    if (!arena || ((uintptr_t)arena % kAlign)) return PIC_EINVAL;
    const TableLayout T = table_layout(cfg->max_slots);
    if (arena_bytes < T.total) return PIC_ENOMEM;
    pic_pool *pool = new (std::nothrow) pic_pool();
    if (!pool) return PIC_ENOMEM;
    pool->cfg = *cfg;
    pool->arena = (unsigned char *)arena;
    pool->arena_bytes = arena_bytes;
    pool->stream = (cudaStream_t)stream;
    pool->tab = T;
    if (arena_bytes > T.total) pool->free_list[T.total] = arena_bytes - T.total;
    pool->slots.resize(cfg->max_slots);
    pool->h_runs.resize(cfg->max_slots);
    pool->h_order.resize(cfg->max_slots);
    std::memset(pool->h_runs.data(), 0, pool->h_runs.size() * sizeof(BatchRun));
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&pool->sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = batch_prepare_attributes();
    int coop = 0, per_sm = 0;
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e == cudaSuccess && coop) e = steps_pool_prepare(&per_sm);
    if (e != cudaSuccess) { delete pool; return cuda_fail(e); }
    if (per_sm > 0) pool->resident_sms = pool->sms;
    rc = set_shape(pool, cfg->variant ? cfg->variant : kPoolVariant,
                   cfg->cluster ? cfg->cluster : 8, cfg->block ? cfg->block : kPoolBlock);
    if (rc) { delete pool; return rc; }
    pool->many_step = !cfg->variant && !cfg->cluster && !cfg->block;
    if (!cfg->block)
        pool->wide_clusters = batch_max_clusters(pool->variant, pool->cluster, 2 * kPoolBlock,
                                                 pool->cfg.ncell_max);
    e = cudaMemsetAsync(pool->arena + T.scalars, 0, 2 * sizeof(unsigned), pool->stream);
    if (e != cudaSuccess) { delete pool; return cuda_fail(e); }
    *out = pool;
    return PIC_OK;
}

void pic_pool_destroy(pic_pool *pool) { delete pool; }

int pic_pool_configure(pic_pool *pool, int32_t variant, int32_t cluster, int32_t block) {
    if (!pool) return PIC_EINVAL;
    const int rc = set_shape(pool, variant, cluster, block);
    if (!rc) pool->many_step = false;
    return rc;
}

int pic_pool_many_step(pic_pool *pool, int32_t on) {
    if (!pool) return PIC_EINVAL;
    pool->many_step = on != 0;
    return PIC_OK;
}

}  // extern "C"

namespace {

// Take a slot and arena space for a run; fill its descriptor; zero its
// counters.  The particles are written by the caller.
int admit_common(pic_pool *pool, const pic_params *p, int64_t steps, int32_t *slot) {
    int s = -1;
    for (int i = 0; i < (int)pool->slots.size(); i++)
        if (!pool->slots[i].used) { s = i; break; }
    if (s < 0) return PIC_ENOMEM;
    const RunLayout L = run_layout(p, pool->cfg.history);
    size_t off;
    {
        std::lock_guard<std::mutex> lock(pool->arena_mutex);
        if (!pool->alloc(L.total, &off)) return PIC_ENOMEM;
    }
    pic_pool::Slot &sl = pool->slots[s];
    sl.used = true;
    sl.needs_init = true;
    sl.p = *p;
    sl.off = off;
    sl.size = L.total;
    sl.lay = L;
    sl.target = steps;
    sl.done = 0;
    unsigned char *base = pool->arena + off;
    BatchRun &d = sl.desc;
    sl.buf_x[0] = (float *)(base + L.x);
    sl.buf_v[0] = (float *)(base + L.v);
    sl.buf_x[1] = p->sort_interval > 0 ? (float *)(base + L.xa) : nullptr;
    sl.buf_v[1] = p->sort_interval > 0 ? (float *)(base + L.va) : nullptr;
    sl.point_at_state();
    d.sort_interval = p->sort_interval;
    d.n = p->npart;
    d.pc.ng = p->ncell;
    d.pc.ngf = (float)p->ncell;
    d.pc.kdrift = (float)(p->dt * (double)p->ncell / p->length);
    d.pc.qmdt = (float)(p->qm * p->dt);
    d.E32 = (float *)(base + L.E32);
    d.E64 = (double *)(base + L.E64);
    d.phi = (double *)(base + L.phi);
    d.rho = (double *)(base + L.rho);
    d.rho_q_last = (unsigned long long *)(base + L.rq);
    d.hist = (pic_diag_row *)(base + L.hist);
    d.hist_len = pool->cfg.history;
    d.steps = 0;
    d.step = (long long *)(base + L.step);
    d.weight_total = (long long)p->npart << kFixBits;
    d.dx = p->length / (double)p->ncell;
    const double q0 = (p->rho_ion * p->length / (double)p->npart) * (p->qm / std::fabs(p->qm));
    d.mass = q0 / p->qm;
    d.k_rho = p->rho_ion / std::ldexp((double)p->npart, kFixBits);
    d.k_e = 0.5 * d.dx * d.k_rho / (double)p->ncell;
    d.k_phi = -d.dx * d.dx * d.k_rho / (double)p->ncell;
    d.k_mode = 2.0 / (double)p->ncell;
    cudaError_t e = cudaMemsetAsync(d.step, 0, 8, pool->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(d.E32, 0, 4 * (size_t)p->ncell, pool->stream);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(d.hist, 0xFF, (size_t)pool->cfg.history * sizeof(pic_diag_row), pool->stream);
    if (e != cudaSuccess) {
        sl = pic_pool::Slot();
        std::lock_guard<std::mutex> lock(pool->arena_mutex);
        pool->release(off, L.total);
        return cuda_fail(e);
    }
    *slot = s;
    return PIC_OK;
}

int check_admit(const pic_pool *pool, const pic_params *p) {
    int rc = validate_params(p);
    if (rc) return rc;
    if (p->precision != PIC_FP32_FIXED || p->ncell > pool->cfg.ncell_max) return PIC_EINVAL;
    if (p->field_solver != PIC_SOLVER_EXACT || p->shape != PIC_SHAPE_CIC) return PIC_EINVAL;
    return PIC_OK;
}

void drop_slot(pic_pool *pool, int s) {
    pic_pool::Slot &sl = pool->slots[s];
    std::lock_guard<std::mutex> lock(pool->arena_mutex);
    pool->release(sl.off, sl.size);
    sl = pic_pool::Slot();
}

}  // namespace

extern "C" {

int pic_pool_admit(pic_pool *pool, const pic_params *p, const void *x0, const void *v0,
                   int64_t steps, int32_t *slot) {
    pic::TraceRange trace_("pic_pool_admit");
    if (!pool || !p || !x0 || !v0 || !slot || steps < 0) return PIC_EINVAL;
    *slot = -1;
    int rc = check_admit(pool, p);
    if (rc) return rc;
    const float Lf = (float)p->length;
    const float *xf = (const float *)x0;
    for (int64_t i = 0; i < p->npart; i++)
        if (!(xf[i] >= 0.0f && xf[i] < Lf)) return PIC_EINVAL;
    int32_t s;
    rc = admit_common(pool, p, steps, &s);
    if (rc) return rc;
    const BatchRun &d = pool->slots[s].desc;
    const size_t pb = (size_t)p->npart * 4;
    cudaError_t e = cudaMemcpyAsync(d.x, x0, pb, cudaMemcpyHostToDevice, pool->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(d.v, v0, pb, cudaMemcpyHostToDevice, pool->stream);
    if (e == cudaSuccess)
        e = launch_to_cells(d.x, p->npart, (double)p->ncell / p->length, (float)p->ncell, Lf,
                            pool->d_err(), pool->sms, pool->stream);
    if (e != cudaSuccess) { drop_slot(pool, s); return cuda_fail(e); }
    *slot = s;
    return PIC_OK;
}

int pic_pool_admit_loaded(pic_pool *pool, const pic_params *p, const pic_loading *ld,
                          int64_t steps, int32_t *slot) {
    pic::TraceRange trace_("pic_pool_admit_loaded");
    if (!pool || !p || !ld || !slot || steps < 0) return PIC_EINVAL;
    *slot = -1;
    int rc = check_admit(pool, p);
    if (rc) return rc;
    LoadArgs a;
    rc = make_load_args(ld, p->npart, p->length, (float *)pool->arena, (float *)pool->arena, &a);
    if (rc) return rc;
    int32_t s;
    rc = admit_common(pool, p, steps, &s);
    if (rc) return rc;
    a.x = pool->slots[s].desc.x;
    a.v = pool->slots[s].desc.v;
    cudaError_t e = launch_load(a, pool->sms, pool->stream);
    if (e == cudaSuccess)
        e = launch_to_cells(a.x, p->npart, (double)p->ncell / p->length, (float)p->ncell,
                            (float)p->length, pool->d_err(), pool->sms, pool->stream);
    if (e != cudaSuccess) { drop_slot(pool, s); return cuda_fail(e); }
    *slot = s;
    return PIC_OK;
}

int pic_pool_advance(pic_pool *pool, int64_t k, int32_t *active) {
    pic::TraceRange trace_("pic_pool_advance");
    if (!pool || k < 0) return PIC_EINVAL;
    if (active) *active = 0;
    std::vector<int> order;
    for (int i = 0; i < (int)pool->slots.size(); i++)
        if (pool->slots[i].used && pool->slots[i].needs_init) order.push_back(i);
    if (!order.empty()) {
        std::sort(order.begin(), order.end(), [&](int a, int b) {
            return pool->slots[a].p.npart > pool->slots[b].p.npart;
        });
        int rc = launch(pool, order, false);
        if (rc) return rc;
        for (int i : order) pool->slots[i].needs_init = false;
    }
    if (k == 0) return PIC_OK;
    order.clear();
    for (int i = 0; i < (int)pool->slots.size(); i++) {
        pic_pool::Slot &sl = pool->slots[i];
        if (!sl.used || sl.lost) continue;
        const int64_t left = sl.target - sl.done;
        const int64_t take = left < k ? left : k;
        // one launch advances at most INT_MAX steps (the descriptor's int)
        sl.desc.steps = (int)(take > INT_MAX ? INT_MAX : take);
        if (sl.desc.steps > 0) order.push_back(i);
    }
    // longest work first (particles x steps)
    std::sort(order.begin(), order.end(), [&](int a, int b) {
        const double wa = (double)pool->slots[a].p.npart * pool->slots[a].desc.steps;
        const double wb = (double)pool->slots[b].p.npart * pool->slots[b].desc.steps;
        return wa > wb;
    });
    std::vector<int> workers;
    bool done = order.empty();
    int rc = PIC_OK;
    if (!done && resident(pool, order, &workers)) rc = launch_resident(pool, order, workers, &done);
    if (!rc && !done) rc = launch(pool, order, true);
    if (rc) return rc;
    for (int i : order) {
        pool->slots[i].done += pool->slots[i].desc.steps;
        pool->slots[i].point_at_state();
    }
    if (active) *active = (int32_t)order.size();
    return PIC_OK;
}

int pic_pool_set_wait_limit(pic_pool *pool, int32_t polls, int32_t missing) {
    if (!pool || (polls != 0 && polls < PIC_WAIT_LIMIT_MIN) || missing < 0 || missing > 1) return PIC_EINVAL;
    pool->wait_limit = (unsigned)polls;
    pool->wait_missing = (unsigned)missing;
    return PIC_OK;
}

int pic_pool_finished(const pic_pool *pool, int32_t *slots, int32_t max, int32_t *n) {
    if (!pool || !n || max < 0) return PIC_EINVAL;
    int c = 0;
    for (int i = 0; i < (int)pool->slots.size(); i++) {
        const pic_pool::Slot &sl = pool->slots[i];
        if (sl.used && !sl.needs_init && !sl.lost && sl.done >= sl.target) {
            if (slots && c < max) slots[c] = i;
            c++;
        }
    }
    *n = c;
    return PIC_OK;
}

int pic_pool_step_count(const pic_pool *pool, int32_t slot, int64_t *step) {
    if (!slot_ok(pool, slot) || !step) return PIC_EINVAL;
    *step = pool->slots[slot].done;
    return PIC_OK;
}

int pic_pool_get_cells(pic_pool *pool, int32_t slot, float *u, float *v) {
    pic::TraceRange trace_("pic_pool_get_cells");
    if (!slot_ok(pool, slot)) return PIC_EINVAL;
    const pic_pool::Slot &sl = pool->slots[slot];
    if (const int rc = readable(sl)) return rc;
    const size_t pb = (size_t)sl.p.npart * 4;
    if (u) PIC_CUDA(cudaMemcpyAsync(u, sl.desc.x, pb, cudaMemcpyDeviceToHost, pool->stream));
    if (v) PIC_CUDA(cudaMemcpyAsync(v, sl.desc.v, pb, cudaMemcpyDeviceToHost, pool->stream));
    return read_error(pool);
}

int pic_pool_get_state(pic_pool *pool, int32_t slot, void *x, void *v) {
    pic::TraceRange trace_("pic_pool_get_state");
    if (!slot_ok(pool, slot)) return PIC_EINVAL;
    const pic_pool::Slot &sl = pool->slots[slot];
    if (const int rc = readable(sl)) return rc;
    const size_t pb = (size_t)sl.p.npart * 4;
    const double to_phys = sl.p.length / (double)sl.p.ncell;
    const float Lf = (float)sl.p.length;
    size_t soff = 0, sbytes = 0;
    std::unique_lock<std::mutex> lock(pool->arena_mutex);         // till the copies are queued
    const bool scratch = x && pool->idle_space(&soff, &sbytes) && sbytes >= std::min(pb, kMinScratch);
    if (!scratch) {
        lock.unlock();
        // the arena is full: cell coordinates down, converted here with the
        // same two float64-rounded steps as the device conversion
        const int rc = pic_pool_get_cells(pool, slot, (float *)x, (float *)v);
        if (rc || !x) return rc;
        const float top = below(Lf);
        float *xf = (float *)x;
        for (int64_t i = 0; i < sl.p.npart; i++) {
            const float xi = (float)((double)xf[i] * to_phys);
            xf[i] = xi > top ? top : xi;
        }
        return PIC_OK;
    }
    // physical positions into idle arena space, piece by piece, then down; the
    // stream orders each piece's copy before the next piece's conversion and
    // before anything admitted into that space later
    float *tmp = (float *)(pool->arena + soff);
    const int64_t piece = (int64_t)(std::min(pb, sbytes) / 4);
    for (int64_t i = 0; i < sl.p.npart; i += piece) {
        const int64_t m = std::min(piece, sl.p.npart - i);
        PIC_CUDA(launch_to_physical(sl.desc.x + i, tmp, m, to_phys, Lf, pool->sms, pool->stream));
        PIC_CUDA(cudaMemcpyAsync((float *)x + i, tmp, (size_t)m * 4, cudaMemcpyDeviceToHost,
                                 pool->stream));
    }
    lock.unlock();
    if (v) PIC_CUDA(cudaMemcpyAsync(v, sl.desc.v, pb, cudaMemcpyDeviceToHost, pool->stream));
    return read_error(pool);
}

int pic_pool_get_field(pic_pool *pool, int32_t slot, double *rho, double *phi, double *E,
                       int64_t *rho_q) {
    pic::TraceRange trace_("pic_pool_get_field");
    if (!slot_ok(pool, slot)) return PIC_EINVAL;
    const pic_pool::Slot &sl = pool->slots[slot];
    if (const int rc = readable(sl)) return rc;
    const size_t nb = (size_t)sl.p.ncell * 8;
    struct { void *dst; const void *src; } const want[] = {
        {rho, sl.desc.rho}, {phi, sl.desc.phi}, {E, sl.desc.E64}, {rho_q, sl.desc.rho_q_last}};
    std::lock_guard<std::mutex> lock(pool->stage.mutex);
    for (const auto &w : want) {
        if (!w.dst) continue;
        const cudaError_t e = pool->stage.add(w.dst, w.src, nb, pool->stream);
        if (e != cudaSuccess) { pool->stage.abandon(pool->stream); return cuda_fail(e); }
    }
    return finish_read(pool);
}

int pic_pool_diagnostics(pic_pool *pool, int32_t slot, int64_t first, int32_t count,
                         pic_diag_row *rows) {
    pic::TraceRange trace_("pic_pool_diagnostics");
    if (!slot_ok(pool, slot) || !rows || count < 0 || first < 0) return PIC_EINVAL;
    const pic_pool::Slot &sl = pool->slots[slot];
    if (sl.lost) return PIC_ETIMEOUT;
    const int64_t H = pool->cfg.history;
    if (count == 0) return PIC_OK;
    if (first + count - 1 > sl.done || first < sl.done - H + 1) return PIC_EINVAL;
    std::lock_guard<std::mutex> lock(pool->stage.mutex);
    int64_t got = 0;
    while (got < count) {
        const int64_t pos = (first + got) % H;
        int64_t len = count - got;
        if (pos + len > H) len = H - pos;
        const cudaError_t e = pool->stage.add(rows + got, sl.desc.hist + pos,
                                              (size_t)len * sizeof(pic_diag_row), pool->stream);
        if (e != cudaSuccess) { pool->stage.abandon(pool->stream); return cuda_fail(e); }
        got += len;
    }
    return finish_read(pool);
}

int pic_pool_release(pic_pool *pool, int32_t slot) {
    if (!slot_ok(pool, slot)) return PIC_EINVAL;
    pic_pool::Slot &sl = pool->slots[slot];
    // the arena space may be reused by the next admission: its uploads are
    // stream-ordered after every launch already enqueued
    std::lock_guard<std::mutex> lock(pool->arena_mutex);
    pool->release(sl.off, sl.size);
    sl = pic_pool::Slot();
    return PIC_OK;
}

int pic_pool_sync(pic_pool *pool) {
    if (!pool) return PIC_EINVAL;
    return read_error(pool);
}

int pic_pool_usage(const pic_pool *pool, size_t *used, size_t *largest_free) {
    if (!pool) return PIC_EINVAL;
    if (used) *used = pool->used;
    if (largest_free) {
        size_t m = 0;
        for (auto &kv : pool->free_list) m = kv.second > m ? kv.second : m;
        *largest_free = m;
    }
    return PIC_OK;
}

}  // extern "C"
