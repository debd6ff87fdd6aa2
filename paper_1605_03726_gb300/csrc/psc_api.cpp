// psc_api.cpp -- host runtime of the hop engine: the C ABI of include/psc.h.
//
// The host owns the model (species, reactions), derives the per-species
// constants of the paper (hop interval, Sec. 2.3; acceptance p_AB,
// Sec. 2.4.2; first-order firing, Sec. 2.4.1), runs the event scheduler
// (Sec. 2.2) and queues the kernels of each event on the lattice's stream.
// No step of an event runs on the host: the kernels read the molecule counts
// from device memory, so the host never waits for the device between events.
#include "psc.h"
#include "psc_internal.h"
#include "psc_readout.h"
#include "psc_runtime.h"

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <thread>
#include <vector>

#include <sys/mman.h>
#include <unistd.h>

using namespace psc;

namespace {

psc_alloc_fn g_alloc = nullptr;
psc_free_fn g_free = nullptr;
void* g_alloc_ctx = nullptr;
std::mutex g_alloc_mu;

// floor(min(p, 1) * 2^32): a 32-bit uniform u passes with probability p iff u < T
uint64_t prob_threshold(double p)
{
    if (!(p > 0.0)) return 0;
    if (p >= 1.0) return 1ull << 32;
    return (uint64_t)std::floor(p * 4294967296.0);
}

// Sec. 2.3, Eq. 3: mean time to hop one voxel diameter, tau_d = 2 r_v^2 / (3 D)
double hop_interval(double rv, double D) { return (2.0 * rv * rv) / (3.0 * D); }

// Sec. 2.4.2, Eq. 6: discrete Collins-Kimball acceptance of a collision
double acceptance(double k, double DA, double DB, double rv)
{
    return k / (6.0 * std::sqrt(2.0) * (DA + DB) * rv);
}

}  // namespace

namespace psc_rt {

int cuda_fail(psc_lattice* L, cudaError_t e)
{
    if (e == cudaSuccess) return PSC_OK;
    if (L) L->sticky = (e == cudaErrorMemoryAllocation) ? PSC_E_NOMEM : PSC_E_CUDA;
    return e == cudaErrorMemoryAllocation ? PSC_E_NOMEM : PSC_E_CUDA;
}

void* dev_alloc(psc_lattice* L, size_t bytes)
{
    if (bytes == 0) bytes = 256;
    bytes = (bytes + 255) & ~(size_t)255;
    void* p = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_alloc_mu);
        if (g_alloc) p = g_alloc(bytes, L->device, L->stream, g_alloc_ctx);
        else if (cudaMalloc(&p, bytes) != cudaSuccess) p = nullptr;
    }
    if (!p) cudaGetLastError();                      // reported by the caller; not the next launch's error
    if (p) L->allocs.push_back(p);
    return p;
}

namespace {

// Buffers carved from one allocation: a lattice of 64^3 voxels spent more on some
// thirty allocations and their release than on its placement.
struct Carve {
    std::vector<std::pair<void*, size_t>> parts;     // address of the pointer, offset
    size_t bytes = 0;
    template <typename T>
    void add(T** p, size_t n)
    {
        parts.emplace_back((void*)p, bytes);
        bytes += (std::max<size_t>(n, 1) + 255) & ~(size_t)255;
    }
    char* commit(psc_lattice* L)
    {
        char* base = (char*)dev_alloc(L, bytes);
        for (const auto& x : parts) {
            char* q = base ? base + x.second : nullptr;
            std::memcpy(x.first, &q, sizeof(q));
        }
        return base;
    }
};

// Pages of a host buffer that a read-out is about to fill, made present by
// several threads: a copy into fresh pages faults them in one after the other
// (64 MB 2.49 ms; made present by one thread, and copied, 2.33, two 1.53, four
// 1.22, eight 2.05).  Contents stay as they are; a buffer whose pages are there
// already (its ends and middle say so), or a small one, is left alone.
void make_present(void* buf, size_t bytes)
{
    const size_t kPart = (size_t)2 << 20;
    if (bytes < 2 * kPart) return;
    const uintptr_t page = (uintptr_t)sysconf(_SC_PAGESIZE);
    const uintptr_t lo = ((uintptr_t)buf + page - 1) & ~(page - 1), hi = ((uintptr_t)buf + bytes) & ~(page - 1);
    unsigned char there = 1;
    const uintptr_t look[3] = {lo, (lo + (hi - lo) / 2) & ~(page - 1), hi - page};
    for (int x = 0; x < 3 && (there & 1); ++x)
        if (mincore((void*)look[x], page, &there) != 0) return;
    if (there & 1) return;
    const size_t want = std::min<size_t>({bytes / kPart, (size_t)4, (size_t)std::max(1u, std::thread::hardware_concurrency())});
    const int parts = (int)std::max<size_t>(want, 1);
    auto part = [=](int x) {
        const uintptr_t step = ((hi - lo) / (uintptr_t)parts) & ~(page - 1);
        const uintptr_t a = lo + step * (uintptr_t)x, b = x == parts - 1 ? hi : a + step;
        (void)madvise((void*)a, b - a, MADV_POPULATE_WRITE);       // a kernel without it: the copy faults them in
    };
    std::vector<std::thread> helpers;
    int mine = 1;
    try {
        helpers.reserve((size_t)parts);
        for (; mine < parts; ++mine) helpers.emplace_back(part, mine);
    } catch (...) {                                    // no more threads: the rest here
    }
    part(0);
    for (; mine < parts; ++mine) part(mine);
    for (auto& h : helpers) h.join();
}

}  // namespace

void dev_free_all(psc_lattice* L)
{
    std::lock_guard<std::mutex> lk(g_alloc_mu);
    for (void* p : L->allocs) {
        if (g_free) g_free(p, L->device, L->stream, g_alloc_ctx);
        else cudaFree(p);
    }
    L->allocs.clear();
}

void dev_free_one(psc_lattice* L, void* p)
{
    auto it = std::find(L->allocs.begin(), L->allocs.end(), p);
    if (it == L->allocs.end()) return;
    L->allocs.erase(it);
    std::lock_guard<std::mutex> lk(g_alloc_mu);
    if (g_free) g_free(p, L->device, L->stream, g_alloc_ctx);
    else cudaFree(p);
}

int event_blocks(const psc_lattice* L, int64_t work)
{
    const int64_t want = (work + L->opt.block_threads - 1) / L->opt.block_threads;
    const int64_t cap = (int64_t)L->sm_count * L->opt.blocks_per_sm;
    return (int)std::max<int64_t>(1, std::min(want, cap));
}

// Grid of a per-event launch over list x: the list's grid class (4, 32 or
// 256 blocks, or the full grid for its capacity).
int list_blocks(const psc_lattice* L, int x)
{
    return std::min(event_blocks(L, L->cap[x]), L->grid_class[x]);
}

// The grid class for a list estimated at n entries, given its class so far:
// a class holds at least one block per 128 entries; it grows as soon as the
// list outgrows it and shrinks only once the list needs a sixteenth of it, so
// that captured graphs (keyed by the grids) stay valid while a count hovers.
static int grid_class_for(const psc_lattice* L, int x, int64_t n, int cur)
{
    static const int kClasses[3] = {4, 32, 256};
    const int full = event_blocks(L, L->cap[x]);
    const int64_t need = (2 * n + L->opt.block_threads - 1) / L->opt.block_threads + 1;
    int fit = INT32_MAX;
    for (int c : kClasses)
        if (need <= c && c < full) { fit = c; break; }
    if (cur <= 0 || fit > cur) return fit;                      // first class, or grown out of it
    const int64_t cur_blocks = std::min(cur, full);
    return need * 16 <= cur_blocks ? fit : cur;
}

// How many leading entries of list x a Morton re-sort takes: a list in a
// small grid class sorts twice what its class holds, at most its capacity
// (entries beyond keep their places; list order never changes results).  The
// sort's tiles and scans follow this bound, not the capacity, which for
// reaction products is the whole lattice.
int32_t sort_limit(const psc_lattice* L, int x)
{
    int64_t n = std::min<int64_t>(L->cap[x], 256 * (int64_t)L->grid_class[x]);
    // a full-grid list: an eighth over its estimate
    if (L->counts_h && L->est[x] > 0) n = std::min<int64_t>(n, L->est[x] + L->est[x] / 8 + 65536);
    return (int32_t)n;
}

// Does Morton order pay for list x?  Only if the list holds at least 1/256 of
// the voxels (by its estimate): sparser lists share too few cache lines
// between neighbours in any order, and their re-sorts cost more than they
// save.  (Long lists on large lattices always: their claim launches read a
// mirror that does not fit in L2; 2.1M walkers on 1024^3 118 us per event, 140
// unsorted.)  A skipped re-sort changes no result.
bool sorted_order_pays(const psc_lattice* L, int x)
{
    return !L->counts_h || L->est[x] * 256 >= L->V ||
           (L->open_claims && L->est[x] >= kOpenList);
}

// Lists come from the placement in no order: the first sort of list s is due
// at its first event, not a period later (1.23M walkers at 30 %: 33 us per
// event before it, 21 after).  It takes as long as a few events gain: calls of fewer
// put it off.
constexpr int64_t kSortFirst = 8;
static bool first_sort_due(const psc_lattice* L, int s)
{
    return L->placed_order[s] && (L->ahead >= kSortFirst || L->since_resort[s] >= (uint64_t)kSortFirst);
}

int sort_first(psc_lattice* L, int s)
{
    if (L->opt.resort_period > 0 && first_sort_due(L, s)) {
        L->placed_order[s] = false;
        if (sorted_order_pays(L, s)) return resort(L, s);
    }
    return PSC_OK;
}

// Take the last background copy of the list lengths if it has landed, and
// start the next one every 64 events.  The host queues events far faster than
// the device runs them; once a copy is 256 events old the host waits for it,
// so the estimates stay recent (the device still has that many queued).
constexpr size_t kCountsBytes = offsetof(Scalars, next_id) + sizeof(uint32_t);   // counts to next_id
constexpr size_t kStateBytes = offsetof(Scalars, err) + sizeof(int32_t);         // counts to err
constexpr size_t kStateAt = 2048;           // of check_device's copy, in the same page
static_assert(kCountsBytes <= kStateAt && kStateAt + kStateBytes <= 4096, "both fit a page");

static void counts_free(psc_lattice* L)
{
    if (!L->counts_h) return;
    cudaHostUnregister(L->counts_h);
    std::free(L->counts_h);
    L->counts_h = nullptr;
}

void refresh_estimates(psc_lattice* L)
{
    if (!L->counts_h) return;
    if (L->counts_pending) {
        if (cudaEventQuery(L->counts_ev) != cudaSuccess) {
            if (L->g - L->counts_g < 256u) return;
            if (cudaEventSynchronize(L->counts_ev) != cudaSuccess) {
                L->counts_pending = false;
                return;
            }
        }
        if (L->counts_g >= L->next_id_g) {           // (a batch may have brought newer ones)
            for (int s = 0; s < L->nsp; ++s) {
                L->est[s] = L->counts_h[s];
                L->grid_class[s] = grid_class_for(L, s, L->est[s], L->grid_class[s]);
            }
            L->next_id_known = (uint32_t)L->counts_h[offsetof(Scalars, next_id) / 4];
            L->next_id_g = L->counts_g;
        }
        L->counts_pending = false;
    }
    if (L->g - L->counts_g < 64u) return;
    if (cudaMemcpyAsync(L->counts_h, L->sc, kCountsBytes, cudaMemcpyDeviceToHost, L->stream) != cudaSuccess ||
        cudaEventRecord(L->counts_ev, L->stream) != cudaSuccess)
        return;
    L->d2h += kCountsBytes;
    L->counts_pending = true;
    L->counts_g = L->g;
}

// set-up of one event of species s, everything passed by value
EventArgs event_args(const psc_lattice* L, int s)
{
    EventArgs a{};
    a.geo = L->geo;
    a.geo.slot_map = (uint32_t)(L->opt.slot_map - 1);
    a.occ = L->occ;
    a.bits = L->bits + (size_t)L->sp[s].comp * L->mirror_n;
    a.ct.direct = L->claim;
    if (L->tables[0]) {
        const int cur = (int)(L->g & 1u), other = cur ^ 1;
        a.ct.hash = L->tables[cur];
        a.ct.hash_bits = L->hash_bits[s];
        a.ct.clear = L->tables[other];
        a.ct.clear_n = L->table_used[other];
    }
    a.live = L->live[s] ? 1 : 0;
    a.list = L->model_h.lists[s];
    a.count = &L->sc->counts[s];
    a.model = L->model_d;
    a.sc = L->sc;
    a.births = L->births;
    a.births_cap = L->births_cap;
    a.key0 = (uint32_t)L->seed;
    a.key1 = (uint32_t)(L->seed >> 32);
    a.g = L->g;
    a.g_base = nullptr;
    if (L->capture_g0 >= 0) {                         // captured for replay: index relative to the run's first
        a.g = L->g - (uint32_t)L->capture_g0;
        a.g_base = &L->sc->g_base;
    }
    a.dirty[0] = L->dirty[0];
    a.dirty[1] = L->dirty[1];
    a.dirty_words = L->dirty_words;
    // the claim outcomes live in the scratch list's third array between claim
    // and commit, the due species' leavers in its first (its capacity is the
    // largest list's; the list passes that use it come after)
    a.dec = reinterpret_cast<uint8_t*>(L->tmp.img);
    a.leave = L->tmp.vox;
    a.holes = reinterpret_cast<int32_t*>(L->tmp.ids);
    a.surv = reinterpret_cast<int32_t*>(L->tmp.img);
    a.g_bump = nullptr;
    a.s = s;
    a.collect_stats = L->opt.collect_stats > 0 ? 1 : 0;
    return a;
}

enum SpanKind { kSpanClaim = 0, kSpanCommit, kSpanReconcile, kSpanResort, kSpanRun, kSpanTile, kSpanTileLean };

cudaEvent_t take_event(psc_lattice* L)
{
    if (!L->event_pool.empty()) {
        cudaEvent_t e = L->event_pool.back();
        L->event_pool.pop_back();
        return e;
    }
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
    return e;
}

// open a span: returns its start event (recorded now) or null when timing is off
cudaEvent_t span_open(psc_lattice* L)
{
    if (L->opt.time_kernels <= 0) return nullptr;
    cudaEvent_t a = take_event(L);
    if (a) cudaEventRecord(a, L->stream);
    return a;
}

void span_close(psc_lattice* L, cudaEvent_t a, int kind, int64_t events = 1)
{
    if (!a) return;
    cudaEvent_t b = take_event(L);
    if (!b) { L->event_pool.push_back(a); return; }
    cudaEventRecord(b, L->stream);
    L->spans.push_back({a, b, kind, events});
}

int resort(psc_lattice* L, int s)
{
    L->placed_order[s] = false;
    if (int rc = grid_current(L, true)) return rc;
    const int blocks = list_blocks(L, s);
    const SpeciesList& list = L->model_h.lists[s];
    const int32_t* count = &L->sc->counts[s];
    const int32_t limit = sort_limit(L, s);
    if (limit > kCellSortMax) {
        launch_morton_keys(list, count, limit, L->geo, L->rs_keys, L->rs_vals, blocks, L->stream);
        if (radix_sort_pairs(L->rs_keys, L->rs_vals, count, limit, limit, (int)morton_sort_bits(L->geo),
                             L->rs_scratch, L->stream, &L->launches) != 0)
            return cuda_fail(L, cudaErrorUnknown);
        launch_permute(list, L->tmp, L->rs_vals, count, limit, blocks, L->stream);
        launch_copy_list(L->tmp, list, count, limit, blocks, L->stream);
        L->launches += 3;
        return PSC_OK;
    }
    // as many cells as the scratch counts: 8 to 16 entries in each, at most 2^20
    uint32_t bits = 8;
    while (bits < 20 && bits < L->geo.mort_bits && (2ll << bits) <= std::min<int64_t>(limit / 8, L->rs_scratch.hist_len))
        ++bits;
    bits = std::min(bits, L->geo.mort_bits);
    uint32_t* cells = L->rs_scratch.hist;
    if (int rc = cuda_fail(L, cudaMemsetAsync(cells, 0, sizeof(uint32_t) << bits, L->stream))) return rc;
    launch_cell_count(list, count, limit, L->geo, bits, cells, blocks, L->stream);
    exclusive_scan(cells, (int64_t)1 << bits, L->rs_scratch.block_sums, L->stream, &L->launches);
    launch_cell_scatter(list, L->tmp, count, limit, L->geo, bits, cells, blocks, L->stream);
    launch_copy_list(L->tmp, list, count, limit, blocks, L->stream);
    L->launches += 3;
    return PSC_OK;
}

ReconcileArgs reconcile_args(const psc_lattice* L, int x)
{
    ReconcileArgs r{};
    r.geo = L->geo;
    r.occ = L->occ;
    r.bits = L->bits + (size_t)L->sp[x].comp * L->mirror_n;
    r.x = x;
    r.list = L->model_h.lists[x];
    r.tmp = L->tmp;
    r.model = L->model_d;
    r.sc = L->sc;
    r.dirty[0] = L->dirty[0];
    r.dirty[1] = L->dirty[1];
    r.g = L->g;
    r.g_base = nullptr;
    r.g_bump = nullptr;
    if (L->capture_g0 >= 0) {
        r.g = L->g - (uint32_t)L->capture_g0;
        r.g_base = &L->sc->g_base;
    }
    return r;
}

// Do claim and commit launches of species s look for hops that need no claim
// (psc_open.cuh)?  Long lists of species without reactions, on lattices whose
// claim words do not fit in the L2 cache and that are not crowded.
static bool open_pays(const psc_lattice* L, int s)
{
    if (L->general[s] || L->est[s] < kOpenList || L->V <= kWalkVoxels) return false;
    int64_t molecules = 0;
    for (int x = 0; x < L->nsp; ++x) molecules += L->est[x];
    return (double)molecules <= kOpenOccupied * (double)L->V;
}

int enqueue_event(psc_lattice* L, int s)
{
    const EventArgs a = event_args(L, s);
    const int threads = L->opt.block_threads;
    const int blocks = list_blocks(L, s);
    // captured as a single-event graph: the event's last launch advances the
    // device's event index to the next event
    uint32_t* bump = L->capture_single ? &L->sc->g_base : nullptr;
    const std::vector<int>& Q = L->reconcile[s];
    // a list of at most a few hundred molecules: claim, commit and its own
    // fill in one block, one launch
    const bool one = L->general[s] && L->grid_class[s] <= 4;
    cudaEvent_t sp = span_open(L);
    if (one) {
        EventArgs a1 = a;
        if (!L->fo2[s] && Q.size() == 1) a1.g_bump = bump;
        launch_event_one(a1, L->stream);
        span_close(L, sp, kSpanClaim);
        L->launches += 1;
    } else if (open_pays(L, s)) {
        launch_open_claim(a, L->est[s], L->sm_count, L->stream);
        span_close(L, sp, kSpanClaim);
        sp = span_open(L);
        launch_open_commit(a, L->est[s], L->sm_count, L->stream);
        span_close(L, sp, kSpanCommit);
        L->launches += 2;
    } else {
        launch_claim(a, L->general[s], blocks, threads, L->stream);
        span_close(L, sp, kSpanClaim);
        sp = span_open(L);
        launch_commit(a, L->general[s], blocks, threads, L->stream);
        span_close(L, sp, kSpanCommit);
        L->launches += 2;
    }
    if (L->tables[0]) {
        const int cur = (int)(L->g & 1u);
        L->table_used[cur] = 1u << L->hash_bits[s];
        L->table_used[cur ^ 1] = 0;
    }
    sp = (!L->reconcile[s].empty() || L->fo2[s]) ? span_open(L) : nullptr;
    // the due species' own list changes only through its own molecules, whose
    // commit noted the leavers; partner lists are checked against the grid,
    // one after the other; then one launch fills every list (but the own one
    // of a one-block event), a block each (list order: the due species, then
    // the partners; each list's scratch range follows those of the lists
    // before it)
    uint32_t before = 0;
    for (int x : Q) {
        if (x != s) {
            launch_reconcile(reconcile_args(L, x), before, list_blocks(L, x), threads, L->stream);
            L->launches += 1;
        }
        before |= 1u << x;
    }
    if (Q.size() > (one ? 1u : 0u)) {
        ListFill f{};
        f.r = reconcile_args(L, s);
        before = 0;
        for (size_t q = 0; q < Q.size(); ++q) {
            if (one && Q[q] == s) {
                before |= 1u << s;
                continue;
            }
            f.x[f.n] = Q[q];
            f.list[f.n] = L->model_h.lists[Q[q]];
            f.before[f.n] = before;
            before |= 1u << Q[q];
            if (++f.n == kListFillMax || q + 1 == Q.size()) {
                if (!L->fo2[s] && q + 1 == Q.size()) f.r.g_bump = bump;
                launch_fill(f, L->stream);
                L->launches += 1;
                f.n = 0;
            }
        }
    }
    if (L->fo2[s]) {
        EventArgs ab = a;
        ab.g_bump = bump;
        launch_births(ab, L->stream);
        L->launches += 1;
    }
    span_close(L, sp, kSpanReconcile);
    L->events++;
    if (L->opt.resort_period > 0 && ++L->since_resort[s] >= (uint64_t)L->opt.resort_period) {
        L->since_resort[s] = 0;
        if (sorted_order_pays(L, s)) {
            sp = span_open(L);
            int rc = resort(L, s);
            span_close(L, sp, kSpanResort);
            if (rc) return rc;
        }
    }
    return cuda_fail(L, cudaPeekAtLastError());
}

// Can a stretch of events of species s run in one persistent launch?
int run_width(const psc_lattice* L, int s, int* threads, int* blocks)
{
    if (L->opt.persistent <= 0 || L->general[s]) return 0;
    if (L->tables[0] && L->hash_bits[s] > 27) return 0;
    return run_capacity(L->cap[s], threads, blocks, L->sm_count, L->opt.run_per_thread);
}

int enqueue_run(psc_lattice* L, int s, int n_events, int per_thread, int threads, int blocks)
{
    cudaStream_t st = L->stream;
    // both claim tables must start empty
    for (int t = 0; t < 2; ++t) {
        if (L->tables[t] && L->table_used[t]) {
            launch_fill_u64(L->tables[t], kEmptySlot, L->table_used[t], L->sm_count * 4, st);
            L->table_used[t] = 0;
            L->launches += 1;
        }
    }
    RunArgs r{};
    r.ev = event_args(L, s);
    r.tables[0] = L->tables[0];
    r.tables[1] = L->tables[1];
    r.n_events = n_events;
    r.barrier = L->barrier;
    r.barrier_timeout_ns = (uint64_t)L->opt.barrier_timeout_us * 1000ull;
    r.barrier_phantom = (uint32_t)L->opt.barrier_phantom;
    int rc = cuda_fail(L, cudaMemsetAsync(L->barrier, 0, sizeof(BarrierState), st));
    if (rc) return rc;
    cudaEvent_t sp = span_open(L);
    rc = cuda_fail(L, launch_run(r, blocks, threads, per_thread, st));
    span_close(L, sp, kSpanRun, n_events);
    if (rc) return rc;
    L->launches += 1;
    L->events += (uint64_t)n_events;
    return PSC_OK;
}

// ---------------------------------------------------------------------------
// tile kernel (owner-computes stretches)
// ---------------------------------------------------------------------------
// Does the plan spread the species' molecules evenly enough over the boxes?
// Every event waits for the fullest box, so the tile kernel's time grows with
// max / mean of the box loads, while the molecule-list kernel is balanced by
// construction and takes about 1.4 times the tile kernel's time on evenly
// spread molecules (measured at 512^3).  Decided once per species, from the
// loads at its first stretch (one count kernel and one small read-back);
// molecules confined to part of the lattice (a compartment, a cluster) pick
// the molecule-list kernel.
static bool tile_balanced(psc_lattice* L, int s, const TilePlan& P)
{
    const int64_t n = L->sp[s].n0;
    if (n <= 0 || P.regions <= 0) return false;
    int32_t* counts = (int32_t*)dev_alloc(L, (size_t)P.regions * 4);
    if (!counts) return false;
    TileArgs A{};
    A.ev = event_args(L, s);
    A.plan = P;
    std::vector<int32_t> h((size_t)P.regions, 0);
    bool ok = cudaMemsetAsync(counts, 0, (size_t)P.regions * 4, L->stream) == cudaSuccess;
    if (ok) {
        launch_tile_count(A, counts, std::max(1, std::min(2 * L->sm_count, (int)((n + 4095) / 4096))), L->stream);
        L->launches += 1;
        ok = cudaMemcpyAsync(h.data(), counts, (size_t)P.regions * 4, cudaMemcpyDeviceToHost, L->stream) ==
                 cudaSuccess &&
             cudaStreamSynchronize(L->stream) == cudaSuccess;
        L->d2h += (uint64_t)P.regions * 4;
    }
    dev_free_one(L, counts);
    if (!ok) return false;
    const int32_t mx = *std::max_element(h.begin(), h.end());
    return (double)mx * P.regions <= kTileMaxImbalance * (double)n;
}

bool tile_plan(psc_lattice* L, int s, TilePlan* P)
{
    if (L->opt.tiles < 0 || L->general[s] || L->live[s] || !(L->sp[s].D > 0.0)) return false;
    // automatic choice: the tile kernel wins from about 2^18 molecules on
    // lattices whose claims go to hash tables; on lattices of up to 2^22
    // voxels the molecule-list kernel's per-voxel claim words stay in L2 and
    // it wins at every density (measured on 128^3, 256^3 and 512^3)
    if (L->opt.tiles == 0 && (L->sp[s].n0 < ((int64_t)1 << 18) || L->V <= ((int64_t)1 << 22))) return false;
    if (L->sp[s].n0 <= 0) return false;
    // periodic axes must wrap whole bricks
    if ((L->bflags & PSC_PERIODIC_I) && (L->ni & 3)) return false;
    if ((L->bflags & PSC_PERIODIC_J) && (L->nj & 3)) return false;
    if ((L->bflags & PSC_PERIODIC_K) && (L->nk & 1)) return false;
    if (L->tile_smem < 0) L->tile_smem = tile_smem_limit(L->device);
    const int nbi = (L->ni + 3) / 4, nbj = (L->nj + 3) / 4, nbk = (L->nk + 1) / 2;
    int S = kTileBlocksPerSM * L->sm_count;
    if (L->opt.tile_regions > 0) S = std::min(S, L->opt.tile_regions);
    // the cut that minimises the largest box (work of the slowest block), then
    // the halo
    int64_t best_work = -1, best_box = 0;
    TilePlan best{};
    // owner tables, neighbourhood masks, outbox
    const int fcc = (L->bflags & PSC_FCC) ? 1 : 0;
    const int64_t owners = ((nbi + nbj + nbk + 15) & ~15) + (fcc ? 96 : 32) * 8 * 4 + kTileOutbox * 12 +
                           kTileQueue * 4;
    for (int pi = 1; pi <= std::min(std::min(nbi, S), 255); ++pi) {
        for (int pj = 1; pj <= std::min(std::min(nbj, S / pi), 255); ++pj) {
            for (int pk = 1; pk <= std::min(std::min(nbk, S / (pi * pj)), 255); ++pk) {
                const int ei = (nbi + pi - 1) / pi, ej = (nbj + pj - 1) / pj, ek = (nbk + pk - 1) / pk;
                const int64_t box = (int64_t)(ei + 2) * (ej + 2) * (ek + 2);
                if (((box + 3) & ~3) * 4 + owners > L->tile_smem) continue;
                if (ei > 512 || ej > 512 || ek > 512) continue;   // packed region coordinates
                const int64_t work = (int64_t)ei * ej * ek;
                if (best_work < 0 || work < best_work || (work == best_work && box < best_box)) {
                    best_work = work;
                    best_box = box;
                    best = TilePlan{pi, pj, pk, nbi, nbj, nbk, ei, ej, ek, pi * pj * pk, (int32_t)box, 0, fcc};
                }
            }
        }
    }
    if (best_work < 0) return false;
    const double share = (double)best_work / ((double)nbi * nbj * nbk);
    const int64_t cap = std::min<int64_t>(best_work * 32, (int64_t)(2.0 * share * (double)L->sp[s].n0) + 8192);
    if (cap > INT32_MAX / 2) return false;
    best.cap = (int32_t)cap;
    // the lean variant: HCP, whole bricks on every axis (so reflective walls
    // fall on brick faces), boxes at least two bricks thick (neighbour waits),
    // two or more boxes along every periodic axis (no box wraps onto itself)
    {
        const bool whole = (L->ni % 4) == 0 && (L->nj % 4) == 0 && (L->nk % 2) == 0;
        const bool thick = nbi / best.pi >= 2 && nbj / best.pj >= 2 && nbk / best.pk >= 2;
        const bool wraps = (!(L->bflags & PSC_PERIODIC_I) || best.pi >= 2) &&
                           (!(L->bflags & PSC_PERIODIC_J) || best.pj >= 2) &&
                           (!(L->bflags & PSC_PERIODIC_K) || best.pk >= 2);
        best.lean = (!fcc && whole && thick && wraps && L->opt.tile_lean >= 0 &&
                     lean_smem_bytes(best) <= L->tile_smem) ? 1 : 0;
    }
    if (L->opt.tiles == 0) {
        if (L->open_claims && (!best.lean || L->sp[s].n0 >= kOpenOverLean)) return false;
        if (L->tile_auto[s] == 0) L->tile_auto[s] = tile_balanced(L, s, best) ? 1 : -1;
        if (L->tile_auto[s] < 0) return false;
    }
    *P = best;
    return true;
}

static int tile_buffers(psc_lattice* L, const TilePlan& P, int64_t ids)
{
    auto& T = L->tile;
    const int64_t slots = (int64_t)P.regions * P.cap;
    if (slots > T.slots || P.regions > T.regions) {
        for (void* p : {(void*)T.b_vox[0], (void*)T.b_vox[1], (void*)T.b_ids[0], (void*)T.b_ids[1],
                        (void*)T.b_state, (void*)T.b_cnt, (void*)T.in_vox, (void*)T.in_ids, (void*)T.in_cnt,
                        (void*)T.claimed, (void*)T.done})
            if (p) dev_free_one(L, p);
        const int64_t ns = std::max(slots, T.slots);
        const int32_t nr = std::max(P.regions, T.regions);
        for (int x = 0; x < 2; ++x) {
            T.b_vox[x] = (int32_t*)dev_alloc(L, (size_t)ns * 4);
            T.b_ids[x] = (uint32_t*)dev_alloc(L, (size_t)ns * 4);
        }
        T.b_state = (uint32_t*)dev_alloc(L, (size_t)ns * 4);
        T.in_vox = (int32_t*)dev_alloc(L, (size_t)ns * 4);
        T.in_ids = (uint32_t*)dev_alloc(L, (size_t)ns * 4);
        T.b_cnt = (int32_t*)dev_alloc(L, (size_t)nr * 4);
        T.in_cnt = (int32_t*)dev_alloc(L, (size_t)nr * 4);
        T.claimed = (uint32_t*)dev_alloc(L, (size_t)nr * 4);
        T.done = (uint32_t*)dev_alloc(L, (size_t)nr * 4);
        T.slots = ns;
        T.regions = nr;
        if (!T.b_vox[0] || !T.b_vox[1] || !T.b_ids[0] || !T.b_ids[1] || !T.b_state || !T.in_vox || !T.in_ids ||
            !T.b_cnt || !T.in_cnt || !T.claimed || !T.done) {
            T.slots = 0;
            return PSC_E_NOMEM;
        }
    }
    if (!L->claim && !T.claim) {
        // contested targets are claimed in per-voxel words, free (all ones) between events
        T.claim = (uint32_t*)dev_alloc(L, (size_t)L->V * 4);
        if (!T.claim) return PSC_E_NOMEM;
        launch_fill_u32(T.claim, kNoClaim, (size_t)L->V, L->sm_count * 8, L->stream);
    }
    if (P.lean && (int64_t)P.regions * lean_halo_cap(P) > T.halo_entries) {
        if (T.halo_tab) dev_free_one(L, T.halo_tab);
        const int64_t ne = (int64_t)P.regions * lean_halo_cap(P);
        T.halo_tab = (uint2*)dev_alloc(L, (size_t)ne * sizeof(uint2));
        T.halo_entries = T.halo_tab ? ne : 0;
        if (!T.halo_tab) return PSC_E_NOMEM;
    }
    if (ids > T.ids) {
        if (T.img_id) dev_free_one(L, T.img_id);
        T.img_id = (uint64_t*)dev_alloc(L, (size_t)ids * 8);
        T.ids = T.img_id ? ids : 0;
        if (!T.img_id) return PSC_E_NOMEM;
    }
    return PSC_OK;
}

// Do events of species s take claim and commit launches (psc_open.cuh)
// although stretches are on?  Long lists of large lattices without reactions,
// unless the tile kernel takes them.  Decided once (options reset it).
static bool open_route(psc_lattice* L, int s)
{
    if (!L->open_claims || L->opt.persistent <= 0 || L->opt.run_per_thread > 0 || L->sp[s].n0 < kOpenList) return false;
    if (L->open_auto[s] == 0) {
        TilePlan P{};
        L->open_auto[s] = tile_plan(L, s, &P) ? -1 : 1;
    }
    return L->open_auto[s] > 0;
}

int enqueue_tiles(psc_lattice* L, int s, int64_t n_events, const TilePlan& P)
{
    cudaStream_t st = L->stream;
    int64_t id_lo = 0;
    for (int q = 0; q < s; ++q) id_lo += L->sp[q].n0;
    int rc = tile_buffers(L, P, L->sp[s].n0);
    if (rc) return rc;
    TileArgs A{};
    A.ev = event_args(L, s);
    A.ev.ct.hash = nullptr;
    A.ev.ct.clear = nullptr;
    A.ev.ct.clear_n = 0;
    A.claim = L->claim ? L->claim : L->tile.claim;
    A.claimed = L->tile.claimed;
    A.done = L->tile.done;
    // Neighbour waits instead of grid barriers need boxes at least two bricks
    // thick: then everything a phase reads from outside its box (halo bits,
    // arrivals, the claim words of targets next to it) is written only by
    // boxes adjacent to it, and all boxes touching one claim word are
    // adjacent to each other.
    A.nbr_sync = (P.nbi / P.pi >= 2 && P.nbj / P.pj >= 2 && P.nbk / P.pk >= 2) ? 1 : 0;
    A.plan = P;
    for (int x = 0; x < 2; ++x) {
        A.b_vox[x] = L->tile.b_vox[x];
        A.b_ids[x] = L->tile.b_ids[x];
    }
    A.b_state = L->tile.b_state;
    A.b_cnt = L->tile.b_cnt;
    A.in_vox = L->tile.in_vox;
    A.in_ids = L->tile.in_ids;
    A.in_cnt = L->tile.in_cnt;
    A.img_id = L->tile.img_id;
    A.halo_tab = L->tile.halo_tab;
    A.halo_cap = P.lean ? (int32_t)lean_halo_cap(P) : 0;
    A.id_lo = (uint32_t)id_lo;
    A.n_events = (int32_t)n_events;
    A.barrier = L->barrier;
    A.barrier_timeout_ns = (uint64_t)L->opt.barrier_timeout_us * 1000ull;
    A.barrier_phantom = (uint32_t)L->opt.barrier_phantom;
    if ((rc = cuda_fail(L, cudaMemsetAsync(L->tile.b_cnt, 0, (size_t)P.regions * 4, st)))) return rc;
    if ((rc = cuda_fail(L, cudaMemsetAsync(L->tile.in_cnt, 0, (size_t)P.regions * 4, st)))) return rc;
    if ((rc = cuda_fail(L, cudaMemsetAsync(L->tile.done, 0, (size_t)P.regions * 4, st)))) return rc;
    if ((rc = cuda_fail(L, cudaMemsetAsync(L->tile.claimed, 0, (size_t)P.regions * 4, st)))) return rc;
    if ((rc = cuda_fail(L, cudaMemsetAsync(L->barrier, 0, sizeof(BarrierState), st)))) return rc;
    cudaEvent_t sp = span_open(L);
    const int64_t n = L->sp[s].n0;
    const int sblocks = (int)std::max<int64_t>(1, std::min<int64_t>((n + 8191) / 8192, 2 * L->sm_count));
    launch_tile_scatter(A, sblocks, st);
    rc = cuda_fail(L, launch_tile_run(A, st));
    if (!rc) launch_tile_gather(A, st);
    span_close(L, sp, P.lean ? kSpanTileLean : kSpanTile, n_events);
    if (rc) return rc;
    L->launches += 3;
    L->events += (uint64_t)n_events;
    return cuda_fail(L, cudaPeekAtLastError());
}

// the sub-volume rule: one cooperative launch over a stretch of events
int enqueue_subvol(psc_lattice* L, int s, int64_t n_events)
{
    cudaStream_t st = L->stream;
    SubvolArgs A{};
    A.ev = event_args(L, s);
    A.word = L->subvol.word;
    A.head = L->subvol.head;
    A.next = L->subvol.next;
    A.state = L->subvol.state;
    A.colour0 = L->subvol.colour0;
    A.lead = L->subvol.lead;
    A.lead_vox = L->subvol.lead_vox;
    A.counters = L->subvol.counters;
    A.n_events = (int32_t)n_events;
    A.barrier = L->barrier;
    A.barrier_timeout_ns = (uint64_t)L->opt.barrier_timeout_us * 1000ull;
    A.barrier_phantom = (uint32_t)L->opt.barrier_phantom;
    int rc = cuda_fail(L, cudaMemsetAsync(L->barrier, 0, sizeof(BarrierState), st));
    if (rc) return rc;
    if ((rc = cuda_fail(L, cudaMemsetAsync(L->subvol.counters, 0, 32 * sizeof(uint32_t), st)))) return rc;
    cudaEvent_t sp = span_open(L);
    rc = cuda_fail(L, launch_subvol(A, L->subvol.blocks, 256, st));
    span_close(L, sp, kSpanRun, n_events);
    if (rc) return rc;
    L->launches += 1;
    L->events += (uint64_t)n_events;
    return PSC_OK;
}

// What stretches of k_small_run and k_walk_run may take on the lattice's
// device: asked of the device once (it does not change).
static void device_shapes(psc_lattice* L)
{
    struct Shapes {
        bool known = false;
        int cluster = 0, grid = 0, walk_cluster = 0, walk_smem = 0;
    };
    static std::mutex mu;
    static Shapes all[64];
    std::lock_guard<std::mutex> lk(mu);
    Shapes one;
    Shapes& S = L->device < 64 ? all[L->device] : one;
    if (!S.known) {
        small_limits(L->sm_count, &S.cluster, &S.grid);
        walk_limits(&S.walk_cluster, &S.walk_smem);
        S.known = true;
    }
    L->small.cluster = S.cluster;
    L->small.grid = S.grid;
    L->walk_cluster = S.walk_cluster;
    L->walk_smem = S.walk_smem;
    L->shapes_known = true;
}

// Set-up of the first stretch: which species react, have partners, make what;
// the argument templates.
static int small_setup(psc_lattice* L)
{
    auto& B = L->small;
    for (int s = 0; s < L->nsp; ++s) {
        if (L->general[s]) B.general |= 1u << s;
        if (L->fo2[s]) B.fo2 |= 1u << s;
        for (int x : L->reconcile[s]) B.closes[s] |= 1u << x;
        auto products = [&](const Reaction& R) {
            for (int q = 0; q < R.np; ++q) B.products[s] |= 1u << R.p[q];
        };
        for (int x = 0; x < L->nsp; ++x) {
            if (L->pair[s][x] < 0) continue;
            products(L->rx[L->pair[s][x]]);
        }
        for (int u = 0; u < L->sp[s].n_fo; ++u) products(L->rx[L->sp[s].fo[u]]);
    }
    std::vector<EventArgs> ev((size_t)L->nsp);
    for (int s = 0; s < L->nsp; ++s) ev[(size_t)s] = event_args(L, s);
    if (!B.ev) B.ev = (EventArgs*)dev_alloc(L, sizeof(EventArgs) * ev.size());
    if (!B.ev) return PSC_E_NOMEM;
    // (from pageable memory: the copy has left it when the call returns)
    const int rc = cuda_fail(L, cudaMemcpyAsync(B.ev, ev.data(), sizeof(EventArgs) * ev.size(), cudaMemcpyHostToDevice,
                                                L->stream));
    if (rc) return rc;
    L->h2d += sizeof(EventArgs) * ev.size();
    B.ev_set = true;
    return PSC_OK;
}

// No id is at or above this: an event makes at most births_cap of them.
int64_t ids_bound(const psc_lattice* L)
{
    return L->next_id_known + (L->births_cap > 1 ? (int64_t)(L->g - L->next_id_g) * L->births_cap : 0);
}

// Do the events of walkers s among species with reactions, whose diffusion
// coefficients add up to `others`, come in runs too long for k_small_run?
static bool small_run_long(const psc_lattice* L, int s, double others)
{
    const double n = (double)L->est[s];
    int threads, blocks;
    if (n < (double)kSmallRunList) return false;
    const double run = L->V > kWalkVoxels ? kSmallRunLarge / n
                                          : run_width(L, s, &threads, &blocks) > 0 ? kSmallRun / n : kSmallRunDense;
    return L->sp[s].D > std::max(run, kSmallRunLeast) * others;
}

// Do the lattice's events run in stretches of k_small_run?  Every mobile
// species' list holds at most kSmallList molecules, in lattices without
// reactions kSmallWalk, and no long list of walkers among species with reactions
// has its events in long runs (by the estimates: a list that has grown past it in the
// meantime only takes longer).  All of them or none: the other kernels want
// mirrors and codes, which these stretches bring up to date by a pass over the
// lattice.
static bool small_fits(psc_lattice* L)
{
    if (!L->claim || L->opt.persistent <= 0 || L->V > kCellVoxels ||
        ids_bound(L) > kCellIds || L->small.no_room)
        return false;
    for (int s = 0; s < L->nsp; ++s)
        if (L->model_h.lists[s].cap > kCellVoxels) return false;
    if (!L->shapes_known) device_shapes(L);
    if (L->small.cluster <= 0 || L->small.grid <= 0) return false;
    const int64_t most = L->nrx > 0 ? kSmallList : kSmallWalk;
    double rate = 0.0;                               // of all species' events
    for (int s = 0; s < L->nsp; ++s) rate += L->sp[s].D;
    for (int s = 0; s < L->nsp; ++s) {
        if (!(L->sp[s].D > 0.0)) continue;
        if (L->est[s] > most) return false;
        if (!L->general[s] && small_run_long(L, s, rate - L->sp[s].D)) return false;
        // kernel timing keeps the phases of a reaction event apart; without the background
        // copies of the list lengths nothing is known of them
        if (L->general[s] && (L->opt.time_kernels > 0 || !L->counts_h)) return false;
        if (L->general[s]) continue;
        if (L->opt.run_per_thread > 0) return false; // the caller picks the molecule-list kernel's shape
        TilePlan P{};
        if (L->opt.tiles > 0 && tile_plan(L, s, &P)) return false;
    }
    return true;
}

// Bytes of the buffers a lattice's stretches of k_small_run still lack, and
// their allocation; scratch: lists are closed up in a grid or a group of blocks.
static int32_t small_scratch(const psc_lattice* L)
{
    // two tombstones per molecule of the due species and event, and as many
    // again from the events before; lists may have grown by half
    int64_t cap = 0, est = 0;
    for (int x = 0; x < L->nsp; ++x) {
        cap = std::max<int64_t>(cap, L->model_h.lists[x].cap);
        if (L->sp[x].D > 0.0) est = std::max<int64_t>(est, L->est[x]);
    }
    return (int32_t)std::min<int64_t>(std::max<int64_t>(6 * est, 1200000), 4 * cap + 4096);
}

int64_t small_lacks(const psc_lattice* L, bool scratch)
{
    const auto& B = L->small;
    bool general = false;
    for (int s = 0; s < L->nsp; ++s) general = general || L->general[s];
    int64_t b = B.ev ? 0 : (int64_t)L->nsp * (int64_t)sizeof(EventArgs);
    if (!B.cell) b += (int64_t)L->mirror_n * 128;
    if (scratch && general && !B.scratch) b += (int64_t)small_scratch(L) * 8;
    return b;
}

int small_buffers(psc_lattice* L, bool scratch)
{
    auto& B = L->small;
    if (!B.ev_set) {
        const int rc = small_setup(L);
        if (rc) return rc;
    }
    if (!B.cell) {
        B.cell = (uint32_t*)dev_alloc(L, (size_t)L->mirror_n * 128);
        if (!B.cell) return PSC_E_NOMEM;
    }
    // (a list that has doubled since wants more)
    if (scratch && B.general && (!B.scratch || (int64_t)small_scratch(L) > 2 * (int64_t)B.scratch_n)) {
        B.version++;
        if (B.scratch) dev_free_one(L, B.scratch);
        B.scratch_n = small_scratch(L);
        B.scratch = (int32_t*)dev_alloc(L, (size_t)B.scratch_n * 8);
        if (!B.scratch) {
            B.scratch_n = 0;
            return PSC_E_NOMEM;
        }
    }
    return PSC_OK;
}

// The arguments of a stretch but its events; the cells are built if need be.
int small_args(psc_lattice* L, SmallArgs* A)
{
    auto& B = L->small;
    if (!B.cells_hold) {
        L->waited = 0;
        launch_cells_build(B.cell, L->bits, L->mirror_n, L->labels.empty() ? 1 : L->ncomp, L->model_d, L->sc->counts,
                           L->nsp, L->geo, L->sm_count * 8, L->stream);
        L->launches += 2;
        if (int rc = cuda_fail(L, cudaPeekAtLastError())) return rc;
        B.cells_hold = true;
    }
    B.grid_stale = true;
    A->ev = B.ev;
    A->model = L->model_d;
    A->sc = L->sc;
    A->cell = B.cell;
    A->holes = B.scratch;
    A->surv = B.scratch + B.scratch_n;
    A->scratch_n = B.scratch_n;
    A->barrier = L->barrier;
    A->barrier_timeout_ns = (uint64_t)L->opt.barrier_timeout_us * 1000ull;
    A->barrier_phantom = (uint32_t)L->opt.barrier_phantom;
    A->nsp = L->nsp;
    A->collect_stats = L->opt.collect_stats > 0 ? 1 : 0;
    A->general = B.general;
    A->fo2 = B.fo2;
    std::memcpy(A->products, B.products, sizeof(A->products));
    return PSC_OK;
}

int grid_current(psc_lattice* L, bool leave)
{
    auto& B = L->small;
    if (B.grid_stale) {
        launch_cells_grid(B.cell, L->bits, L->mirror_n, L->labels.empty() ? 1 : L->ncomp, L->occ, L->geo,
                          L->sm_count * 8, L->stream);
        L->launches += 1;
        B.grid_stale = false;
        if (int rc = cuda_fail(L, cudaPeekAtLastError())) return rc;
    }
    if (leave) B.cells_hold = false;
    return PSC_OK;
}

// A stretch of consecutive events, starting with species s at time t: one
// launch.  *n = events queued.
// Without room for its buffers *n is 0, and the events take the kernels that need
// none, until options are set the next time.
static int small_stretch(psc_lattice* L, int s, double t, double t_end, int64_t max_events, int64_t* n)
{
    auto& B = L->small;
    bool grid = false;                               // the stretch takes a grid
    for (int x = 0; x < L->nsp; ++x) grid = grid || (L->sp[x].D > 0.0 && L->est[x] > kSmallCluster);
    *n = 0;
    const int sticky = L->sticky;
    int rc = small_buffers(L, grid);
    if (rc == PSC_E_NOMEM) {
        L->sticky = sticky;
        B.no_room = true;
        return PSC_OK;
    }
    if (rc) return rc;
    SmallArgs A{};
    const int64_t limit = std::min<int64_t>(std::min<int64_t>(max_events, kSmallEvents),
                                            (int64_t)UINT32_MAX - L->g);
    A.g = L->g;
    int64_t longest = 0, closed = 0;                 // lists of due species; lists that may be closed up
    double spare = 0.0;                              // events that a cluster makes faster, less for longer lists
    do {
        A.seq[A.n_events++] = (uint8_t)s;
        longest = std::max(longest, L->est[s]);
        spare += std::max(0.0, 1.0 - (double)L->est[s] / (double)kSmallCluster);
        for (int x : L->reconcile[s]) closed = std::max(closed, L->est[x]);
        L->sp[s].done++;
        L->g++;
        L->clock = t;
    } while (A.n_events < limit && next_event(L, &s, &t) && t <= t_end);
    // the shape: a cluster of 16 blocks up to kSmallCluster entries (with fewer
    // blocks, or 128 threads in each, short lists got slower: 2621 walkers 3.9 us
    // per event, 4.4 on 8 blocks, 5.5 with 128 threads), but for few events where
    // closing up the lists would take longer than the cluster spares; then a block
    // per SM, of half the threads while they suffice
    // (a cluster's hardware barrier knows no phantoms)
    bool cluster = longest <= kSmallCluster && L->opt.barrier_phantom <= 0;
    if (cluster && (double)closed > kSmallClosed + kSmallClosedEvent * spare) {
        rc = small_buffers(L, true);
        if (rc == PSC_E_NOMEM) L->sticky = sticky;   // (no scratch: in a cluster all the same)
        else if (rc) return rc;
        else cluster = false;
    }
    if ((rc = small_args(L, &A))) return rc;
    const int threads = !cluster && longest <= 65536 && closed <= 1 << 20 ? kSmallThreads / 2 : kSmallThreads;
    const int blocks = cluster ? B.cluster : B.grid;
    if (!cluster && !B.barrier_set) {
        // (it goes on from whatever complete barriers left there; after one that ran out
        // the lattice runs no more)
        if ((rc = cuda_fail(L, cudaMemsetAsync(L->barrier, 0, sizeof(BarrierState), L->stream)))) return rc;
        B.barrier_set = true;
    }
    cudaEvent_t sp = span_open(L);
    rc = cuda_fail(L, launch_small(A, blocks, threads, cluster, L->stream));
    span_close(L, sp, kSpanRun, A.n_events);
    if (rc) return rc;
    L->launches += 1;
    L->events += (uint64_t)A.n_events;
    *n = A.n_events;
    return PSC_OK;
}

int claims_free(psc_lattice* L)
{
    if (!L->claim_vacancy) return PSC_OK;
    L->claim_vacancy = false;
    launch_fill_u32(L->claim, kNoClaim, (size_t)L->claim_n, L->sm_count * 8, L->stream);
    L->launches += 1;
    return cuda_fail(L, cudaPeekAtLastError());
}

// Molecules of all mobile species a thread of k_walk_run holds in a grid of
// one block per SM.
static int64_t walk_slots(const psc_lattice* L, int64_t threads)
{
    int64_t slots = 0;
    for (int s = 0; s < L->nsp; ++s)
        if (L->sp[s].D > 0.0) slots += (L->sp[s].n0 + threads - 1) / threads;
    return slots;
}

// A lattice of a size that k_walk_run takes with its molecules
static bool walk_size(const psc_lattice* L)
{
    if (L->V <= kWalkVoxels) return true;
    if (L->V > kWalkVoxelsFew) return false;
    for (int s = 0; s < L->nsp; ++s)
        if (L->sp[s].D > 0.0 && L->sp[s].n0 >= kOpenList) return false;
    return true;
}

// Can the lattice's events run in stretches of k_walk_run?  No reactions, no
// compartments, a claim word per voxel, molecules that fit in shared memory.
static bool walk_fits(psc_lattice* L, int s)
{
    // (kernel timing keeps to the kernels it tells apart)
    if (!L->walk_only || !L->claim || L->opt.persistent <= 0 || L->opt.run_per_thread > 0 || L->opt.time_kernels > 0)
        return false;
    if (!walk_size(L)) return false;
    if (!L->shapes_known) device_shapes(L);
    if (walk_slots(L, (int64_t)kWalkThreads * L->sm_count) * kWalkThreads * 12 > L->walk_smem) return false;
    TilePlan P{};
    return !(L->opt.tiles > 0 && tile_plan(L, s, &P));
}

// Does Morton order pay for list x there?
static bool walk_sorts(const psc_lattice* L, int x)
{
    return L->opt.resort_period > 0 && L->sp[x].D > 0.0 && L->sp[x].n0 >= kWalkSorted && sorted_order_pays(L, x);
}

static int walk_stretch(psc_lattice* L, int s, double t, double t_end, int64_t max_events, int64_t* n)
{
    WalkArgs A{};
    A.geo = L->geo;
    A.div_nbi = make_fastdiv(L->geo.nbi);
    A.div_nbij = make_fastdiv(L->geo.nbi * L->geo.nbj);
    A.word = L->claim;
    A.bits = L->bits;
    A.sc = L->sc;
    A.barrier = L->barrier;
    A.barrier_timeout_ns = (uint64_t)L->opt.barrier_timeout_us * 1000ull;
    A.barrier_phantom = (uint32_t)L->opt.barrier_phantom;
    A.key0 = (uint32_t)L->seed;
    A.key1 = (uint32_t)(L->seed >> 32);
    A.g = L->g;
    A.collect_stats = L->opt.collect_stats > 0 ? 1 : 0;
    // claims stay below all ones: epochs 1 .. 2^(32 - id bits) - 2
    int64_t largest = 0;
    for (int x = 0; x < L->nsp; ++x) largest = std::max<int64_t>(largest, L->sp[x].D > 0.0 ? L->sp[x].n0 : 0);
    while ((1ll << A.id_bits) < largest) ++A.id_bits;
    const int64_t epochs = ((int64_t)1 << (32 - A.id_bits)) - 2;
    const bool words = !L->claim_vacancy || (int64_t)L->walk_epoch >= epochs;      // they are made (anew)
    const int64_t limit = std::min<int64_t>({max_events, kWalkEvents, (int64_t)UINT32_MAX - L->g,
                                             epochs - (words ? 0 : (int64_t)L->walk_epoch)});
    const uint64_t period = L->opt.resort_period > 0 ? (uint64_t)L->opt.resort_period : UINT64_MAX;
    bool due = false;                                // a list's re-sort ends the stretch
    bool used[kMaxSpecies] = {};                     // species with events in it: the others' molecules stay put
    do {
        A.seq[A.n_events++] = (uint8_t)s;
        used[s] = true;
        if (++L->since_resort[s] >= period && walk_sorts(L, s)) due = true;
        L->sp[s].done++;
        L->g++;
        L->clock = t;
    } while (!due && A.n_events < limit && next_event(L, &s, &t) && t <= t_end);
    auto slots = [&](int64_t threads) {
        int64_t m = 0;
        for (int x = 0; x < L->nsp; ++x) m += used[x] ? (L->sp[x].n0 + threads - 1) / threads : 0;
        return m;
    };
    int64_t most = 0;
    for (int x = 0; x < L->nsp; ++x) most = std::max<int64_t>(most, used[x] ? L->sp[x].n0 : 0);
    const bool cluster = most <= kWalkCluster && L->walk_cluster > 0 && A.barrier_phantom == 0 &&
                         slots((int64_t)kWalkClusterThreads * L->walk_cluster) * kWalkClusterThreads * 12 <=
                             kWalkClusterSmem - 1024;
    const int blocks = cluster ? L->walk_cluster : L->sm_count;
    const int64_t T = (int64_t)blocks * (cluster ? kWalkClusterThreads : kWalkThreads);
    int place[kMaxSpecies] = {};
    uint32_t id_lo = 0;                              // ids are the ones placement gave, species by species
    for (int x = 0; x < L->nsp; id_lo += (uint32_t)L->sp[x].n0, ++x) {
        if (!used[x]) continue;
        A.id_lo[A.n_species] = id_lo;
        place[x] = A.n_species;
        A.n[A.n_species] = (int32_t)L->sp[x].n0;
        A.slot0[A.n_species] = A.slots;
        A.species[A.n_species] = (uint8_t)x;
        A.list[A.n_species] = L->model_h.lists[x];
        A.slots += (int32_t)((L->sp[x].n0 + T - 1) / T);
        A.n_species++;
    }
    for (int e = 0; e < A.n_events; ++e) A.seq[e] = (uint8_t)place[A.seq[e]];
    int rc = PSC_OK;
    for (int x = 0; x < L->nsp; ++x) {
        if (!used[x] || !first_sort_due(L, x) || !walk_sorts(L, x)) continue;
        if ((rc = resort(L, x))) return rc;
    }
    if (words) {
        L->waited = 0;
        launch_walk_words(L->claim, L->claim_vacancy ? nullptr : L->bits, L->mirror_n, L->sm_count * 8, L->stream);
        L->launches += 1;
        L->claim_vacancy = true;
        L->walk_epoch = 0;
    }
    A.epoch = L->walk_epoch + 1;
    L->walk_epoch += (uint32_t)A.n_events;
    if (!cluster && (rc = cuda_fail(L, cudaMemsetAsync(L->barrier, 0, sizeof(BarrierState), L->stream)))) return rc;
    if ((rc = cuda_fail(L, launch_walk(A, blocks, cluster, L->stream)))) return rc;
    L->launches += 1;
    L->events += (uint64_t)A.n_events;
    *n = A.n_events;
    for (int x = 0; due && x < L->nsp; ++x) {
        if (L->since_resort[x] < period || !walk_sorts(L, x)) continue;
        L->since_resort[x] = 0;
        if ((rc = resort(L, x))) return rc;
    }
    return PSC_OK;
}

// Sec. 2.2: the next event belongs to the mobile species whose next diffusion
// time (events done + 1) * tau is earliest; ties go to the lower index.
bool next_event(const psc_lattice* L, int* s_out, double* t_out)
{
    int best = -1;
    double tb = 0.0;
    for (int s = 0; s < L->nsp; ++s) {
        if (!(L->sp[s].D > 0.0)) continue;
        const double t = (double)(L->sp[s].done + 1) * L->sp[s].tau;
        if (best < 0 || t < tb) { best = s; tb = t; }
    }
    *s_out = best;
    *t_out = tb;
    return best >= 0;
}

int note_errors(psc_lattice* L, int32_t err)
{
    if (err & kErrBarrierTimeout) L->sticky = PSC_E_TIMEOUT;
    else if (err) L->sticky = PSC_E_CAPACITY;
    return L->sticky;
}

int check_device(psc_lattice* L)
{
    if (!L->populated) {
        const cudaError_t e = cudaStreamSynchronize(L->stream);
        return e != cudaSuccess ? cuda_fail(L, e) : L->sticky;
    }
    // list lengths and error bits come with the wait itself
    int32_t* state = L->counts_h ? L->counts_h + kStateAt / 4 : L->state;
    cudaError_t e = cudaMemcpyAsync(state, L->sc, kStateBytes, cudaMemcpyDeviceToHost, L->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(L->stream);
    if (e != cudaSuccess) return cuda_fail(L, e);
    if (state != L->state) std::memcpy(L->state, state, kStateBytes);
    L->d2h += kStateBytes;
    return note_errors(L, L->state[offsetof(Scalars, err) / 4]);
}



}  // namespace psc_rt

using namespace psc_rt;

extern "C" {

const char* psc_status_string(int s)
{
    switch (s) {
    case PSC_OK: return "PSC_OK";
    case PSC_E_ARG: return "PSC_E_ARG";
    case PSC_E_DIMS: return "PSC_E_DIMS";
    case PSC_E_ORDER: return "PSC_E_ORDER";
    case PSC_E_FULL: return "PSC_E_FULL";
    case PSC_E_UNSUPPORTED: return "PSC_E_UNSUPPORTED";
    case PSC_E_NOMEM: return "PSC_E_NOMEM";
    case PSC_E_CUDA: return "PSC_E_CUDA";
    case PSC_E_TIMEOUT: return "PSC_E_TIMEOUT";
    case PSC_E_LIMIT: return "PSC_E_LIMIT";
    case PSC_E_CAPACITY: return "PSC_E_CAPACITY";
    case PSC_W_PCLAMP: return "PSC_W_PCLAMP";
    default: return "PSC_UNKNOWN";
    }
}

int psc_set_allocator(psc_alloc_fn alloc, psc_free_fn release, void* ctx)
{
    if ((alloc == nullptr) != (release == nullptr)) return PSC_E_ARG;
    std::lock_guard<std::mutex> lk(g_alloc_mu);
    g_alloc = alloc;
    g_free = release;
    g_alloc_ctx = ctx;
    return PSC_OK;
}

int psc_lattice_create(psc_lattice** out, int32_t ni, int32_t nj, int32_t nk, double rv,
                       uint32_t bflags, int device, void* cuda_stream)
{
    if (!out) return PSC_E_ARG;
    *out = nullptr;
    if (!(rv > 0.0) || !std::isfinite(rv) || bflags > 15u || device < 0) return PSC_E_ARG;
    if (ni < 1 || nj < 1 || nk < 1) return PSC_E_DIMS;
    const int64_t V = (int64_t)ni * nj * nk;
    if (V >= (1ll << 31)) return PSC_E_DIMS;
    if ((bflags & PSC_PERIODIC_I) && ni < 3) return PSC_E_DIMS;
    if ((bflags & PSC_PERIODIC_J) && (nj < 4 || (nj & 1))) return PSC_E_DIMS;
    if (!(bflags & PSC_FCC) && (bflags & PSC_PERIODIC_K) && (nk < 4 || (nk & 1))) return PSC_E_DIMS;
    if ((bflags & PSC_FCC) && (bflags & PSC_PERIODIC_K) && (nk < 3 || nk % 3)) return PSC_E_DIMS;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device >= ndev) return PSC_E_CUDA;
    psc_lattice* L = new (std::nothrow) psc_lattice();
    if (!L) return PSC_E_NOMEM;
    L->ni = ni; L->nj = nj; L->nk = nk; L->V = V; L->rv = rv; L->bflags = bflags; L->device = device;
    std::memset(L->pair, -1, sizeof(L->pair));
    DevGuard dg(device);
    cudaDeviceProp prop;
    if (cudaGetDeviceProperties(&prop, device) != cudaSuccess) { delete L; return PSC_E_CUDA; }
    L->sm_count = prop.multiProcessorCount;
    if (cuda_stream) {
        L->stream = static_cast<cudaStream_t>(cuda_stream);
    } else {
        if (cudaStreamCreateWithFlags(&L->stream, cudaStreamNonBlocking) != cudaSuccess) { delete L; return PSC_E_CUDA; }
        L->own_stream = true;
    }
    L->geo.ni = ni; L->geo.nj = nj; L->geo.nk = nk; L->geo.bflags = bflags;
    L->geo.ninj = (uint32_t)ni * (uint32_t)nj;
    L->geo.div_ni = make_fastdiv((uint32_t)ni);
    L->geo.div_ninj = make_fastdiv(L->geo.ninj);
    L->geo.nbi = (uint32_t)((ni + 3) / 4);
    L->geo.nbj = (uint32_t)((nj + 3) / 4);
    *out = L;
    return PSC_OK;
}

int psc_add_species(psc_lattice* L, double D, int64_t n0, int32_t* species_out)
{
    if (!L) return PSC_E_ARG;
    if (L->populated) return PSC_E_ORDER;
    if (!(D >= 0.0) || !std::isfinite(D) || n0 < 0) return PSC_E_ARG;
    if (L->nsp >= kMaxSpecies) return PSC_E_UNSUPPORTED;
    Species& S = L->sp[L->nsp];
    S = Species();
    S.D = D;
    S.n0 = n0;
    S.tau = D > 0.0 ? hop_interval(L->rv, D) : 0.0;
    if (species_out) *species_out = L->nsp;
    L->nsp++;
    return PSC_OK;
}

int psc_add_reaction(psc_lattice* L, const int32_t* re, int32_t nr, const int32_t* pr, int32_t np,
                     double k, int32_t* rx_out)
{
    if (!L) return PSC_E_ARG;
    if (L->populated) return PSC_E_ORDER;
    if (nr < 1 || nr > 2 || np < 0 || !re || (np > 0 && !pr)) return PSC_E_ARG;
    if (!(k >= 0.0) || !std::isfinite(k)) return PSC_E_ARG;
    if (np > 2) return PSC_E_UNSUPPORTED;
    for (int a = 0; a < nr; ++a) if (re[a] < 0 || re[a] >= L->nsp) return PSC_E_ARG;
    for (int a = 0; a < np; ++a) if (pr[a] < 0 || pr[a] >= L->nsp) return PSC_E_ARG;
    if (L->nrx >= kMaxReactions) return PSC_E_UNSUPPORTED;
    if (nr == 2) {
        if (re[0] == re[1]) return PSC_E_UNSUPPORTED;
        if (!(L->sp[re[0]].D + L->sp[re[1]].D > 0.0)) return PSC_E_UNSUPPORTED;
        if (L->pair[re[0]][re[1]] >= 0) return PSC_E_UNSUPPORTED;
    } else {
        if (!(L->sp[re[0]].D > 0.0)) return PSC_E_UNSUPPORTED;
        if (L->sp[re[0]].n_fo >= kMaxFirstOrder) return PSC_E_UNSUPPORTED;
    }
    Reaction& R = L->rx[L->nrx];
    R = Reaction();
    R.nr = nr; R.np = np; R.k = k;
    for (int a = 0; a < nr; ++a) R.r[a] = re[a];
    for (int a = 0; a < np; ++a) R.p[a] = pr[a];
    if (nr == 2) {
        L->pair[re[0]][re[1]] = (int8_t)L->nrx;
        L->pair[re[1]][re[0]] = (int8_t)L->nrx;
    } else {
        Species& S = L->sp[re[0]];
        S.fo[S.n_fo++] = L->nrx;
    }
    if (rx_out) *rx_out = L->nrx;
    L->nrx++;
    return PSC_OK;
}

int psc_set_compartments(psc_lattice* L, const uint8_t* labels, int32_t n)
{
    if (!L || !labels) return PSC_E_ARG;
    if (L->populated) return PSC_E_ORDER;
    if (n < 1 || n > kMaxCompartments) return PSC_E_ARG;
    for (int64_t v = 0; v < L->V; ++v)
        if (labels[v] >= n) return PSC_E_ARG;
    for (int s = 0; s < L->nsp; ++s)
        if (L->sp[s].comp >= n) return PSC_E_ARG;
    L->labels.assign(labels, labels + L->V);
    L->ncomp = n;
    return PSC_OK;
}

int psc_species_compartment(psc_lattice* L, int32_t s, int32_t c)
{
    if (!L || s < 0 || s >= L->nsp) return PSC_E_ARG;
    if (L->populated) return PSC_E_ORDER;
    if (c < 0 || c >= L->ncomp) return PSC_E_ARG;
    L->sp[s].comp = c;
    return PSC_OK;
}

double psc_tau(const psc_lattice* L, int32_t s)
{
    if (!L || s < 0 || s >= L->nsp || !(L->sp[s].D > 0.0)) return 0.0;
    return L->sp[s].tau;
}

double psc_p_ab(const psc_lattice* L, int32_t r)
{
    if (!L || r < 0 || r >= L->nrx || L->rx[r].nr != 2) return 0.0;
    const Reaction& R = L->rx[r];
    return acceptance(R.k, L->sp[R.r[0]].D, L->sp[R.r[1]].D, L->rv);
}

// spare: claim words and list room that only stretches and the open kernels want
// may be taken (claim words then instead of hash tables).
static int populate(psc_lattice* L, uint64_t seed, bool spare)
{
    int64_t N = 0;
    for (int s = 0; s < L->nsp; ++s) N += L->sp[s].n0;
    if (N > L->V) return PSC_E_FULL;
    // compartments: room in each for its species, and products that can land
    // in theirs
    const bool comps = !L->labels.empty();
    int64_t start[kMaxSpecies] = {};                 // first sorted voxel of each species (placement)
    {
        int64_t room[kMaxCompartments] = {}, used[kMaxCompartments] = {};
        if (comps) {
            for (int64_t v = 0; v < L->V; ++v) room[L->labels[v]]++;
        } else {
            room[0] = L->V;
        }
        for (int s = 0; s < L->nsp; ++s) {
            const int c = L->sp[s].comp;
            used[c] += L->sp[s].n0;
            if (used[c] > room[c]) return PSC_E_FULL;
        }
        for (int r = 0; r < L->nrx; ++r) {
            const Reaction& R = L->rx[r];
            const int ca = L->sp[R.r[0]].comp;
            if (R.nr == 1) {
                if (R.np >= 1 && L->sp[R.p[0]].comp != ca) return PSC_E_UNSUPPORTED;
                continue;
            }
            const int cb = L->sp[R.r[1]].comp;
            if (R.np == 1 && L->sp[R.p[0]].comp != ca && L->sp[R.p[0]].comp != cb) return PSC_E_UNSUPPORTED;
            if (R.np == 2) {
                const int c0 = L->sp[R.p[0]].comp, c1 = L->sp[R.p[1]].comp;
                if (!((c0 == ca && c1 == cb) || (c0 == cb && c1 == ca))) return PSC_E_UNSUPPORTED;
            }
        }
    }
    DevGuard dg(L->device);
    L->seed = seed;

    // ---- frozen constants (Sec. 2.3, 2.4.1, 2.4.2) ----
    ModelDev& M = L->model_h;
    std::memset(&M, 0, sizeof(M));
    std::memcpy(M.pair, L->pair, sizeof(M.pair));
    bool growth = false;
    bool is_product[kMaxSpecies] = {};
    for (int r = 0; r < L->nrx; ++r) {
        Reaction& R = L->rx[r];
        ReactionDev& D = M.rx[r];
        D.np = R.np;
        D.p0 = R.np > 0 ? R.p[0] : 0;
        D.p1 = R.np > 1 ? R.p[1] : 0;
        for (int a = 0; a < R.np; ++a) is_product[R.p[a]] = true;
        if (R.nr == 2) {
            R.prob = acceptance(R.k, L->sp[R.r[0]].D, L->sp[R.r[1]].D, L->rv);
            if (R.prob > 1.0) L->clamped = true;
            D.T = prob_threshold(R.prob);
        } else if (R.np == 2) {
            growth = true;
        }
    }
    for (int s = 0; s < L->nsp; ++s) {
        const Species& S = L->sp[s];
        M.n_fo[s] = S.n_fo;
        if (S.n_fo == 0) continue;
        // per molecule and per own diffusion event: fire with 1 - exp(-a0 tau)
        double ktot = 0.0;
        for (int u = 0; u < S.n_fo; ++u) ktot += L->rx[S.fo[u]].k;
        M.T_fire[s] = prob_threshold(-std::expm1(-ktot * S.tau));
        // Eq. 5: reaction u is the first whose cumulative share reaches a0 R
        double cum = 0.0;
        for (int u = 0; u < S.n_fo; ++u) {
            cum += L->rx[S.fo[u]].k;
            M.fo_rx[s][u] = S.fo[u];
            M.fo_cum[s][u] = (u == S.n_fo - 1) ? (1ull << 32)
                                               : prob_threshold(ktot > 0.0 ? cum / ktot : 1.0);
        }
    }
    // ---- which lists an event can touch ----
    for (int s = 0; s < L->nsp; ++s) L->live[s] = false;
    for (int r = 0; r < L->nrx; ++r) {
        for (int a = 0; a < L->rx[r].nr; ++a) L->live[L->rx[r].r[a]] = true;
        for (int a = 0; a < L->rx[r].np; ++a) L->live[L->rx[r].p[a]] = true;
    }
    for (int s = 0; s < L->nsp; ++s) {
        bool so = false;
        L->reconcile[s].clear();
        for (int r = 0; r < L->nsp; ++r) if (L->pair[s][r] >= 0) so = true;
        L->general[s] = so || L->sp[s].n_fo > 0;
        L->fo2[s] = false;
        for (int u = 0; u < L->sp[s].n_fo; ++u)
            if (L->rx[L->sp[s].fo[u]].np == 2) L->fo2[s] = true;
        if (L->general[s]) {
            L->reconcile[s].push_back(s);
            for (int r = 0; r < L->nsp; ++r) if (L->pair[s][r] >= 0) L->reconcile[s].push_back(r);
        }
    }
    // ---- the sub-volume rule takes species without reactions on colour-consistent periods ----
    if (L->opt.subvolume > 0) {
        for (int s = 0; s < L->nsp; ++s)
            if (L->sp[s].D > 0.0 && L->general[s]) return PSC_E_UNSUPPORTED;
        if (((L->bflags & PSC_PERIODIC_I) && L->ni % 4) || ((L->bflags & PSC_PERIODIC_J) && L->nj % 4) ||
            ((L->bflags & PSC_PERIODIC_K) && L->nk % 4))
            return PSC_E_DIMS;
    }
    // ---- capacities: a list only grows if its species is a product ----
    const int64_t total_bound = growth ? L->V : N;
    int64_t max_cap = 1, max_mobile = 1;
    for (int s = 0; s < L->nsp; ++s) {
        int64_t c = is_product[s] ? std::min<int64_t>(L->V, std::max<int64_t>(total_bound, L->sp[s].n0))
                                  : L->sp[s].n0;
        c = std::max<int64_t>(c, 1);
        L->cap[s] = (int32_t)c;
        max_cap = std::max(max_cap, c);
        if (L->sp[s].D > 0.0) max_mobile = std::max(max_mobile, c);
    }
    // lists of products that are not sized for the lattice keep room for the
    // tombstones of k_small_run
    L->list_slack = growth || !L->stretches || !spare ? 0 : std::min<int64_t>(2 * N, 262144);
    bool any_fo2 = false;
    for (int s = 0; s < L->nsp; ++s) any_fo2 = any_fo2 || L->fo2[s];

    // ---- device memory ----
    const size_t V = (size_t)L->V;
    const size_t nwords = (size_t)mirror_words(L->ni, L->nj, L->nk);
    const int nmirror = comps ? L->ncomp : 1;
    L->mirror_n = nwords;
    L->dirty_words = (uint32_t)((nwords + 31) / 32);
    uint32_t* mort = nullptr;
    Carve carve;
    carve.add(&L->occ, V * sizeof(uint16_t));
    carve.add(&L->bits, nwords * nmirror * sizeof(uint32_t));
    for (int x = 0; x < 2; ++x) carve.add(&L->dirty[x], (size_t)L->dirty_words * 4);
    carve.add(&L->sc, sizeof(Scalars));
    carve.add(&L->model_d, sizeof(ModelDev));
    carve.add(&L->barrier, sizeof(BarrierState));
    carve.add(&mort, (size_t)(L->ni + L->nj + L->nk) * sizeof(uint32_t));
    // claims: a word per voxel on small lattices, else two hash tables with at
    // least two slots per molecule of the largest mobile species
    uint32_t hb_max = 0;
    for (int s = 0; s < L->nsp; ++s) {
        uint32_t hb = 10;
        while (hb < 31 && (1ll << hb) < (int64_t)L->opt.claim_slots * L->cap[s]) ++hb;
        L->hash_bits[s] = hb;
        if (L->sp[s].D > 0.0 && hb > hb_max) hb_max = hb;
    }
    // (tables at least as large as a word per voxel buy nothing, and the
    // per-event kernels empty the previous table in full every event: species
    // that are reaction products get lists sized for the lattice)
    bool direct = L->V <= (1ll << 22) || hb_max == 0 ||
                  2.0 * 8.0 * (double)(1ll << hb_max) >= 4.0 * (double)L->V;
    if (L->opt.claim_table == 1) direct = true;
    if (L->opt.claim_table == 2 && hb_max > 0) direct = spare = false;
    L->batchable = direct;                           // batches take the lattices that have claim words by these rules
    // lattices without reactions take k_walk_run while their molecules fit in
    // shared memory
    L->walk_only = L->nrx == 0 && !comps && L->opt.subvolume <= 0;
    const bool walk = L->walk_only && walk_size(L) &&
                      walk_slots(L, (int64_t)kWalkThreads * L->sm_count) * kWalkThreads * 12 <= kWalkSmem;
    // larger ones with long lists and no reactions skip most claims: words need
    // no table to be emptied (and the tile kernel wants them too)
    bool open = false;
    for (int s = 0; s < L->nsp; ++s)
        open = open || (L->nrx == 0 && L->V > kWalkVoxels && L->sp[s].D > 0.0 && L->sp[s].n0 >= kOpenList &&
                        L->opt.subvolume <= 0);
    // the rest, as far as their events run in stretches of k_small_run (tables and
    // a launch per phase before: A + B <-> C of 2000 + 1000 molecules on 200^3 9.9 ->
    // 3.9 us per event, 200,000 + 100,000 on 256^3 27.5 -> 15.1, 100,000 + 50,000 on
    // 400^3 24.6 -> 12.2; 60,000 walkers on 400^3 15.9 -> 4.7)
    bool stretch = L->stretches && L->V <= kCellVoxels && L->opt.subvolume <= 0;
    for (int s = 0; s < L->nsp; ++s)
        stretch = stretch && (!(L->sp[s].D > 0.0) || L->sp[s].n0 <= (L->nrx > 0 ? kSmallList : kSmallWalk));
    // with stretches off their words pay only where they fit in the L2 cache or the lists
    // are short (400^3, A + B -> C of 1.0M each 121 us per event in tables, 139 in words; of
    // 100,000 26 and 23)
    int64_t longest = 0;
    for (int s = 0; s < L->nsp; ++s) longest = std::max<int64_t>(longest, L->sp[s].D > 0.0 ? L->sp[s].n0 : 0);
    const bool others = L->opt.persistent > 0 || L->V <= kWalkVoxels || longest <= kSmallWalk;
    // (k_walk_run orders them as the mirror's bits, whole bricks)
    const int64_t claim_n = std::max<int64_t>(L->V, L->walk_only ? (int64_t)nwords * 32 : 0);
    L->spare_claims = !direct && spare &&
                      (open || (others && (stretch || (walk && (L->stretches || L->V <= kWalkVoxels)))));
    if (L->spare_claims) {
        L->claim_n = claim_n;
        L->claim = (uint32_t*)dev_alloc(L, (size_t)claim_n * sizeof(uint32_t));
        direct = L->claim != nullptr;                // no room: tables
    }
    L->open_claims = open && direct;
    if (direct && !L->claim) {
        L->claim_n = claim_n;
        carve.add(&L->claim, (size_t)L->claim_n * sizeof(uint32_t));
    } else if (!direct) {
        L->table_slots = (int64_t)1 << hb_max;
        for (int t = 0; t < 2; ++t) carve.add(&L->tables[t], ((size_t)1 << hb_max) * sizeof(uint64_t));
    }
    for (int s = 0; s < L->nsp; ++s) {
        SpeciesList& l = M.lists[s];
        l.cap = L->cap[s] + (is_product[s] ? (int32_t)L->list_slack : 0);
        carve.add(&l.vox, (size_t)l.cap * 4);
        carve.add(&l.ids, (size_t)l.cap * 4);
        carve.add(&l.img, (size_t)l.cap * 8);
    }
    // from here to the end: scratch of events and re-sorts, and first of the placement
    const size_t scratch_at = carve.bytes;
    // the list passes of an event note up to two leavers per reaction, at most
    // one reaction per molecule of the due species
    L->tmp.cap = (int32_t)max_cap;
    carve.add(&L->tmp.vox, (size_t)max_cap * 8);
    carve.add(&L->tmp.ids, (size_t)max_cap * 8);
    carve.add(&L->tmp.img, (size_t)max_cap * 8);
    L->births_cap = any_fo2 ? 8192 : 1;
    carve.add(&L->births, (size_t)L->births_cap * sizeof(Birth));
    L->rs_max = max_mobile;
    void* rs = nullptr;
    carve.add(&L->rs_keys, (size_t)max_mobile * 4);
    carve.add(&L->rs_vals, (size_t)max_mobile * 4);
    carve.add(&rs, sort_scratch_bytes(max_mobile));
    char* const carved = carve.commit(L);
    if (!carved) return PSC_E_NOMEM;
    char* const place_scratch = L->scratch = carved + scratch_at;
    const size_t place_room = L->scratch_bytes = carve.bytes - scratch_at;
    sort_scratch_bind(L->rs_scratch, rs, max_mobile);
    for (int s = 0; s < L->nsp; ++s) {
        M.comp[s] = (uint8_t)(comps ? L->sp[s].comp : 0);
        M.mirror[s] = L->bits + (size_t)M.comp[s] * nwords;
    }
    {
        std::vector<uint32_t> mt((size_t)(L->ni + L->nj + L->nk));
        uint32_t mbits = 0;
        build_morton_tables(L->ni, L->nj, L->nk, mt.data(), &mbits);
        int rc0 = cuda_fail(L, cudaMemcpy(mort, mt.data(), mt.size() * 4, cudaMemcpyHostToDevice));
        if (rc0) return rc0;
        L->h2d += mt.size() * 4;
        L->geo.mort = mort;
        L->geo.mort_bits = mbits;
    }

    if (L->opt.subvolume > 0) {
        auto& SV = L->subvol;
        const size_t nsub = (size_t)((L->ni + 1) / 2) * (size_t)((L->nj + 1) / 2) * (size_t)((L->nk + 1) / 2);
        SV.word = (uint32_t*)dev_alloc(L, nsub * 4);
        SV.head = (uint32_t*)dev_alloc(L, nsub * 4);
        SV.next = (uint32_t*)dev_alloc(L, (size_t)max_mobile * 4);
        SV.state = (uint32_t*)dev_alloc(L, (size_t)max_mobile * 4);
        SV.colour0 = (uint8_t*)dev_alloc(L, (size_t)max_mobile);
        SV.lead = (uint32_t*)dev_alloc(L, (size_t)max_mobile * 4);
        SV.lead_vox = (uint32_t*)dev_alloc(L, (size_t)max_mobile * 4);
        SV.counters = (uint32_t*)dev_alloc(L, 32 * 4);
        if (!SV.word || !SV.head || !SV.next || !SV.state || !SV.colour0 || !SV.lead || !SV.lead_vox ||
            !SV.counters)
            return PSC_E_NOMEM;
        SV.subvols = (int64_t)nsub;
        SV.slots = max_mobile;
        SV.blocks = subvol_max_blocks(L->sm_count);
        if (SV.blocks <= 0) return PSC_E_CUDA;
        launch_fill_u32(SV.word, kNoClaim, nsub, L->sm_count * 4, L->stream);
        launch_fill_u32(SV.head, kNoClaim, nsub, L->sm_count * 4, L->stream);
    }

    cudaStream_t st = L->stream;
    upload_stencil(st);
    int rc = cuda_fail(L, cudaMemcpyAsync(L->model_d, &M, sizeof(M), cudaMemcpyHostToDevice, st));
    if (rc) return rc;
    L->h2d += sizeof(M) + 5 * sizeof(uint32_t) + sizeof(Scalars);
    Scalars sh;
    std::memset(&sh, 0, sizeof(sh));
    for (int s = 0; s < L->nsp; ++s) sh.counts[s] = (int32_t)L->sp[s].n0;
    sh.next_id = (uint32_t)N;
    if ((rc = cuda_fail(L, cudaMemcpyAsync(L->sc, &sh, sizeof(sh), cudaMemcpyHostToDevice, st)))) return rc;
    if ((rc = cuda_fail(L, cudaMemsetAsync(L->occ, 0, V * sizeof(uint16_t), st)))) return rc;
    for (int x = 0; x < 2; ++x)
        if ((rc = cuda_fail(L, cudaMemsetAsync(L->dirty[x], 0, (size_t)L->dirty_words * 4, st)))) return rc;
    const int fill_blocks = L->sm_count * 8;
    uint8_t* labels_d = nullptr;
    if (comps) {
        // the labels are needed on the device only while placing
        labels_d = (uint8_t*)dev_alloc(L, V);
        if (!labels_d) return PSC_E_NOMEM;
        if ((rc = cuda_fail(L, cudaMemcpyAsync(labels_d, L->labels.data(), V, cudaMemcpyHostToDevice, st))))
            return rc;
        L->h2d += V;
        launch_mirror_walls(L->bits, nwords, nmirror, labels_d, L->geo, fill_blocks, st);
        L->launches += 1;
    } else if ((rc = cuda_fail(L, cudaMemsetAsync(L->bits, 0, nwords * sizeof(uint32_t), st)))) {
        return rc;
    }
    if (L->claim) launch_fill_u32(L->claim, kNoClaim, (size_t)L->claim_n, fill_blocks, st);
    for (int t = 0; t < 2; ++t)
        if (L->tables[t]) launch_fill_u64(L->tables[t], kEmptySlot, (size_t)1 << hb_max, fill_blocks, st);

    // ---- placement (Sec. 3.4): voxels in (Philox key, voxel) order, per
    // compartment, dealt to the species.  Only the first voxels of each
    // compartment matter: a histogram of the keys' top bits finds the bin
    // that covers them, and only the voxels up to it are sorted (by key, equal
    // keys by voxel, then stably by compartment). ----
    if (N > 0) {
        const int nc = comps ? L->ncomp : 1;
        const int bins = 1 << kPlaceBits;
        int64_t need[kMaxCompartments] = {};
        for (int s = 0; s < L->nsp; ++s) need[comps ? L->sp[s].comp : 0] += L->sp[s].n0;
        // histogram and count, then the candidates and their sort: in the scratch of
        // the lattice's events, which nothing uses yet, or in blocks of their own
        const size_t head = (size_t)nc * bins * 4 + 256;
        char* const own_head = head <= place_room ? nullptr : (char*)dev_alloc(L, head);
        if (head > place_room && !own_head) return PSC_E_NOMEM;
        uint32_t* hist = (uint32_t*)(own_head ? own_head : place_scratch);
        int32_t* pick_n = (int32_t*)(hist + (size_t)nc * bins);
        if ((rc = cuda_fail(L, cudaMemsetAsync(hist, 0, head, st)))) return rc;
        launch_place_hist((uint32_t)V, (uint32_t)seed, (uint32_t)(seed >> 32), labels_d, nc, hist, fill_blocks, st);
        std::vector<uint32_t> h((size_t)nc * bins);
        if ((rc = cuda_fail(L, cudaMemcpyAsync(h.data(), hist, h.size() * 4, cudaMemcpyDeviceToHost, st)))) return rc;
        if ((rc = cuda_fail(L, cudaStreamSynchronize(st)))) return rc;
        L->d2h += h.size() * 4;
        PlaceLimits lim;
        int64_t cand[kMaxCompartments] = {}, cbase[kMaxCompartments + 1] = {};
        for (int c = 0; c < kMaxCompartments; ++c) lim.bin[c] = -1;
        for (int c = 0; c < nc; ++c) {
            int64_t cum = 0;
            for (int b = 0; b < bins && need[c] > 0; ++b) {
                cum += h[(size_t)c * bins + b];
                if (cum >= need[c]) { lim.bin[c] = b; break; }
            }
            if (need[c] > 0 && lim.bin[c] < 0) return PSC_E_FULL;      // cannot happen: room was checked
            cand[c] = need[c] > 0 ? cum : 0;
            cbase[c + 1] = cbase[c] + cand[c];
        }
        const int64_t M = cbase[nc];
        {
            int64_t used[kMaxCompartments] = {};
            for (int s = 0; s < L->nsp; ++s) {
                const int c = comps ? L->sp[s].comp : 0;
                start[s] = cbase[c] + used[c];
                used[c] += L->sp[s].n0;
            }
        }
        const size_t part = ((size_t)M * 4 + 255) & ~(size_t)255, body = 2 * part + sort_scratch_bytes(M);
        const size_t head_at = own_head ? 0 : (head + 255) & ~(size_t)255;
        char* const own_body = head_at + body <= place_room ? nullptr : (char*)dev_alloc(L, body);
        if (head_at + body > place_room && !own_body) return PSC_E_NOMEM;
        char* const at = own_body ? own_body : place_scratch + head_at;
        uint32_t* cvox = (uint32_t*)at;
        uint32_t* ckey = (uint32_t*)(at + part);
        void* scratch = at + 2 * part;
        SortScratch ss;
        sort_scratch_bind(ss, scratch, M);
        launch_place_pick((uint32_t)V, (uint32_t)seed, (uint32_t)(seed >> 32), labels_d, lim, cvox, ckey, pick_n,
                          (int32_t)M, &L->sc->err, fill_blocks, st);
        int kbits = 32 - kPlaceBits;                   // of the candidates' keys
        for (int c = 0; c < nc; ++c)
            while (kbits < 32 && (lim.bin[c] >> (kbits - (32 - kPlaceBits))) > 0) ++kbits;
        if (radix_sort_pairs(ckey, cvox, nullptr, M, M, kbits, ss, st, &L->launches) != 0)
            return cuda_fail(L, cudaErrorUnknown);
        launch_sort_ties(ckey, cvox, M, fill_blocks, st);
        L->launches += 1;
        if (comps) {
            launch_label_keys(cvox, labels_d, ckey, M, fill_blocks, st);
            if (radix_sort_pairs(ckey, cvox, nullptr, M, M, 8, ss, st, &L->launches) != 0)
                return cuda_fail(L, cudaErrorUnknown);
            L->launches += 1;
        }
        int64_t off[kMaxSpecies + 1];
        off[0] = 0;
        for (int s = 0; s < L->nsp; ++s) off[s + 1] = off[s] + L->sp[s].n0;
        launch_populate_scatter(cvox, N, off, start, L->nsp, L->occ, L->geo, L->model_d, fill_blocks, st);
        L->launches += 3;
        int32_t picked = 0;
        if ((rc = cuda_fail(L, cudaMemcpyAsync(&picked, pick_n, 4, cudaMemcpyDeviceToHost, st)))) return rc;
        if ((rc = cuda_fail(L, cudaStreamSynchronize(st)))) return rc;
        if (picked != M) return PSC_E_CUDA;                             // the two passes disagree
        if (own_body) dev_free_one(L, own_body);
        if (own_head) dev_free_one(L, own_head);
    }
    if (labels_d) {
        if ((rc = cuda_fail(L, cudaStreamSynchronize(st)))) return rc;
        dev_free_one(L, labels_d);
    }
    if (N == 0 && (rc = cuda_fail(L, cudaStreamSynchronize(st)))) return rc;     // (else the placement waited)
    // reactions on lattices of up to 2^22 voxels run in stretches: their templates and
    // cells come with the lattice (16 MB at most), so that events allocate nothing
    bool reacts = false;
    for (int s = 0; s < L->nsp; ++s) reacts = reacts || L->general[s];
    if (reacts && stretch && direct && L->opt.persistent > 0 && L->V <= (1ll << 22)) {
        L->small.ev = (EventArgs*)dev_alloc(L, sizeof(EventArgs) * (size_t)L->nsp);
        L->small.cell = (uint32_t*)dev_alloc(L, nwords * 128);
        if (!L->small.ev || !L->small.cell) return PSC_E_NOMEM;
    }
    L->g = 0;
    L->clock = 0.0;
    L->populated = true;
    // the list-length estimates start from the placed counts (without the
    // pinned copy the grids follow the capacities)
    for (int s = 0; s < L->nsp; ++s) {
        L->est[s] = L->sp[s].n0;
        L->grid_class[s] = INT32_MAX;
        L->placed_order[s] = true;
    }
    L->counts_g = 0;
    L->next_id_known = N;
    L->next_id_g = 0;
    if (!L->counts_h) {
        // a page of the heap, registered: 37 us with its release, 270 from cudaMallocHost
        const size_t page = (size_t)sysconf(_SC_PAGESIZE);
        L->counts_h = (int32_t*)std::aligned_alloc(page, page);
        if (L->counts_h && cudaHostRegister(L->counts_h, page, cudaHostRegisterDefault) != cudaSuccess) {
            std::free(L->counts_h);
            L->counts_h = nullptr;
        }
        if (!L->counts_h) cudaGetLastError();
    }
    if (L->counts_h && !L->counts_ev &&
        cudaEventCreateWithFlags(&L->counts_ev, cudaEventDisableTiming) != cudaSuccess) {
        counts_free(L);
        L->counts_ev = nullptr;
        cudaGetLastError();
    }
    // lists that start empty take the full grid until their first estimate
    if (L->counts_h)
        for (int s = 0; s < L->nsp; ++s)
            if (L->est[s] > 0) L->grid_class[s] = grid_class_for(L, s, L->est[s], 0);
    return L->clamped ? PSC_W_PCLAMP : PSC_OK;
}

int psc_populate(psc_lattice* L, uint64_t seed)
{
    if (!L) return PSC_E_ARG;
    if (L->populated) return PSC_E_ORDER;
    const int sticky = L->sticky;
    int rc = populate(L, seed, true);
    // what was allocated goes back; where claim words were taken that the lattice can do
    // without, it may fit with tables
    for (bool again = true; rc < 0; again = false) {
        const bool retry = again && rc == PSC_E_NOMEM && L->spare_claims;
        DevGuard dg(L->device);
        cudaStreamSynchronize(L->stream);
        dev_free_all(L);
        L->claim = nullptr;
        L->claim_n = 0;
        L->tables[0] = L->tables[1] = nullptr;
        L->table_slots = 0;
        L->small.ev = nullptr;
        L->small.cell = nullptr;
        L->subvol = {};
        if (!retry) break;
        L->sticky = sticky;
        rc = populate(L, seed, false);
    }
    return rc;
}

}  // extern "C"

namespace psc_rt {

// The per-event grids a captured event takes (they follow the list estimates;
// so do the re-sort bounds, through the grid classes).
static void append_grids(const psc_lattice* L, std::vector<uint8_t>& key)
{
    for (int x = 0; x < L->nsp; ++x) {
        const int b = list_blocks(L, x);
        key.push_back((uint8_t)(b & 0xFF));
        key.push_back((uint8_t)(b >> 8));
    }
}

void graph_cache_clear(psc_lattice* L)
{
    for (auto& G : L->graphs)
        if (G.exec) cudaGraphExecDestroy(G.exec);
    L->graphs.clear();
    L->graph_seen.clear();
    for (auto& G : L->graphs1)
        if (G.exec) cudaGraphExecDestroy(G.exec);
    L->graphs1.clear();
    L->graph_seen1.clear();
}

// One event of species s (time t) replayed from a CUDA graph: its launches are
// fixed by the species, the event's parity, the claim tables' fill and whether
// the species' list is re-sorted after it; the event index comes from device
// memory.  Met for the first time, the event runs as usual; met again, it is
// captured once and replayed from then on.  For workloads whose runs of many
// events never recur (species with unrelated hop intervals), where launching
// dominates.  A failed capture turns graphs off for the lattice.
static int single_event(psc_lattice* L, int s, double t)
{
    auto finish = [&]() {
        L->sp[s].done++;
        L->g++;
        L->clock = t;
    };
    if (L->opt.graph_events < 2 || L->opt.time_kernels > 0 || L->g == UINT32_MAX - 1) {
        int rc = enqueue_event(L, s);
        finish();
        return rc;
    }
    // the re-sort counter runs out after this event (1: the list is re-sorted,
    // 2: its order does not pay, no re-sort)
    const uint8_t resort_now =
        (L->opt.resort_period > 0 && L->since_resort[s] + 1 >= (uint64_t)L->opt.resort_period)
            ? (sorted_order_pays(L, s) ? 1 : 2)
            : 0;
    std::vector<uint8_t> key;
    key.push_back((uint8_t)s);
    key.push_back((uint8_t)(L->g & 1u));
    key.push_back(resort_now);
    const uint8_t* tu = reinterpret_cast<const uint8_t*>(L->table_used);
    key.insert(key.end(), tu, tu + sizeof(L->table_used));
    append_grids(L, key);
    // the event index: events of species with reactions advance it on the
    // device, so a run of their replays sets it once
    auto set_index = [&]() {
        if (L->g_dev != (int64_t)L->g) {
            launch_fill_u32(&L->sc->g_base, L->g, 1, 1, L->stream);
            L->launches += 1;
        }
        L->g_dev = L->general[s] ? (int64_t)L->g + 1 : (int64_t)L->g;
    };
    for (const auto& G : L->graphs1) {
        if (G.key != key) continue;
        set_index();
        int rc = cuda_fail(L, cudaGraphLaunch(G.exec, L->stream));
        if (rc) return rc;
        L->table_used[0] = G.table_used[0];
        L->table_used[1] = G.table_used[1];
        L->since_resort[s] = resort_now ? 0 : L->since_resort[s] + 1;
        L->launches += G.launches;
        L->events += 1;
        finish();
        return PSC_OK;
    }
    if (std::find(L->graph_seen1.begin(), L->graph_seen1.end(), key) == L->graph_seen1.end()) {
        if (L->graph_seen1.size() >= 256) L->graph_seen1.erase(L->graph_seen1.begin());
        L->graph_seen1.push_back(key);
        int rc = enqueue_event(L, s);
        finish();
        return rc;
    }
    // seen before: capture once, then launch the graph
    const uint64_t since0 = L->since_resort[s];
    const uint32_t used0[2] = {L->table_used[0], L->table_used[1]};
    const int64_t launches0 = L->launches;
    const uint64_t events0 = L->events;
    const int sticky0 = L->sticky;
    auto restore = [&]() {
        L->since_resort[s] = since0;
        L->table_used[0] = used0[0];
        L->table_used[1] = used0[1];
        L->launches = launches0;
        L->events = events0;
        L->sticky = sticky0;
        L->opt.graph_events = 0;
        cudaGetLastError();
    };
    cudaGraphExec_t exec = nullptr;
    if (cudaStreamBeginCapture(L->stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
        L->capture_g0 = L->g;
        L->capture_single = true;
        int rc = enqueue_event(L, s);
        L->capture_g0 = -1;
        L->capture_single = false;
        cudaGraph_t graph = nullptr;
        cudaError_t ce = cudaStreamEndCapture(L->stream, &graph);
        if (rc == PSC_OK && ce == cudaSuccess && graph) ce = cudaGraphInstantiate(&exec, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        if (rc != PSC_OK || ce != cudaSuccess) {
            if (exec) cudaGraphExecDestroy(exec);
            exec = nullptr;
        }
    }
    if (!exec) {                                   // no graphs for this lattice: the ordinary way
        restore();
        int rc = enqueue_event(L, s);
        finish();
        return rc;
    }
    psc_lattice::GraphRun G;
    G.key = key;
    G.exec = exec;
    G.table_used[0] = L->table_used[0];
    G.table_used[1] = L->table_used[1];
    G.launches = L->launches - launches0;
    if (L->graphs1.size() >= 128) {
        cudaGraphExecDestroy(L->graphs1.front().exec);
        L->graphs1.erase(L->graphs1.begin());
    }
    L->graphs1.push_back(std::move(G));
    set_index();
    int rc = cuda_fail(L, cudaGraphLaunch(exec, L->stream));
    if (rc) return rc;
    finish();
    return PSC_OK;
}

// Runs of per-event launches replayed from CUDA graphs (psc_options.
// graph_events = K; small lattices, where launching dominates).  The next K
// events are planned with the scheduler; all must take per-event launches.
// Their pattern -- species in order, the claim tables' parity and fill, the
// re-sort counters -- fixes every launch but the event index, which the
// kernels then read from device memory.  A pattern met for the first time
// runs as usual; met again it is captured once and replayed from then on,
// the host bookkeeping advanced from what the capture recorded.  Any failure
// to capture turns graphs off for the lattice and leaves the events to the
// ordinary path.  *done = events queued (0: none, take one the ordinary way).
static int graph_run(psc_lattice* L, double t_end, int64_t room, int64_t* done)
{
    *done = 0;
    const int K = L->opt.graph_events;
    if (K < 2 || room < K || L->opt.time_kernels > 0 || (int64_t)L->g + K >= (int64_t)UINT32_MAX) return PSC_OK;
    uint64_t next[kMaxSpecies];
    for (int s = 0; s < L->nsp; ++s) next[s] = L->sp[s].done;
    std::vector<int> seq((size_t)K);
    std::vector<double> at((size_t)K);
    for (int e = 0; e < K; ++e) {
        int best = -1;
        double tb = 0.0;
        for (int s = 0; s < L->nsp; ++s) {
            if (!(L->sp[s].D > 0.0)) continue;
            const double t = (double)(next[s] + 1) * L->sp[s].tau;
            if (best < 0 || t < tb) { best = s; tb = t; }
        }
        if (best < 0 || tb > t_end) return PSC_OK;
        if (!L->general[best] && L->opt.persistent > 0 && !open_route(L, best)) return PSC_OK;   // a stretch comes first
        seq[(size_t)e] = best;
        at[(size_t)e] = tb;
        next[best]++;
    }
    std::vector<uint8_t> key;
    auto put = [&key](const void* p, size_t n) {
        const uint8_t* b = static_cast<const uint8_t*>(p);
        key.insert(key.end(), b, b + n);
    };
    bool in_run[kMaxSpecies] = {};
    for (int s2 : seq) {
        key.push_back((uint8_t)s2);
        in_run[s2] = true;
    }
    const uint32_t parity = L->g & 1u;
    put(&parity, 4);
    put(L->table_used, sizeof(L->table_used));
    for (int s = 0; s < L->nsp; ++s)                 // only the run's species can re-sort in it
        if (in_run[s]) put(&L->since_resort[s], sizeof(uint64_t));
    append_grids(L, key);
    auto advance = [&](int e) {
        L->sp[seq[(size_t)e]].done++;
        L->g++;
        L->clock = at[(size_t)e];
    };
    for (const auto& G : L->graphs) {
        if (G.key != key) continue;
        launch_fill_u32(&L->sc->g_base, L->g, 1, 1, L->stream);
        L->g_dev = (int64_t)L->g;
        int rc = cuda_fail(L, cudaGraphLaunch(G.exec, L->stream));
        if (rc) return rc;
        for (int e = 0; e < K; ++e) advance(e);
        L->table_used[0] = G.table_used[0];
        L->table_used[1] = G.table_used[1];
        for (int s = 0; s < L->nsp; ++s)
            if (in_run[s]) L->since_resort[s] = G.since[(size_t)s];
        L->launches += G.launches + 1;
        L->events += (uint64_t)K;
        *done = K;
        return PSC_OK;
    }
    if (std::find(L->graph_seen.begin(), L->graph_seen.end(), key) == L->graph_seen.end()) {
        if (L->graph_seen.size() >= 32) L->graph_seen.erase(L->graph_seen.begin());
        L->graph_seen.push_back(key);
        for (int e = 0; e < K; ++e) {                // event by event, each from its own graph
            int rc = single_event(L, seq[(size_t)e], at[(size_t)e]);
            if (rc) return rc;
        }
        *done = K;
        return PSC_OK;
    }
    // seen before: capture once
    uint64_t done0[kMaxSpecies], since0[kMaxSpecies];
    for (int s = 0; s < L->nsp; ++s) { done0[s] = L->sp[s].done; since0[s] = L->since_resort[s]; }
    const uint32_t g0 = L->g, used0[2] = {L->table_used[0], L->table_used[1]};
    const double clock0 = L->clock;
    const int64_t launches0 = L->launches;
    const uint64_t events0 = L->events;
    const int sticky0 = L->sticky;
    auto restore = [&]() {
        for (int s = 0; s < L->nsp; ++s) { L->sp[s].done = done0[s]; L->since_resort[s] = since0[s]; }
        L->g = g0;
        L->table_used[0] = used0[0];
        L->table_used[1] = used0[1];
        L->clock = clock0;
        L->launches = launches0;
        L->events = events0;
        L->sticky = sticky0;
        L->opt.graph_events = 0;
        cudaGetLastError();
    };
    if (cudaStreamBeginCapture(L->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        restore();
        return PSC_OK;
    }
    L->capture_g0 = g0;
    int rc = PSC_OK;
    for (int e = 0; e < K && rc == PSC_OK; ++e) {
        rc = enqueue_event(L, seq[(size_t)e]);
        advance(e);
    }
    L->capture_g0 = -1;
    cudaGraph_t graph = nullptr;
    cudaError_t ce = cudaStreamEndCapture(L->stream, &graph);
    cudaGraphExec_t exec = nullptr;
    if (rc == PSC_OK && ce == cudaSuccess && graph) ce = cudaGraphInstantiate(&exec, graph, 0);
    if (graph) cudaGraphDestroy(graph);
    if (rc != PSC_OK || ce != cudaSuccess || !exec) {
        if (exec) cudaGraphExecDestroy(exec);
        restore();
        return PSC_OK;
    }
    psc_lattice::GraphRun G;
    G.key = key;
    G.exec = exec;
    G.table_used[0] = L->table_used[0];
    G.table_used[1] = L->table_used[1];
    G.since.assign(L->since_resort, L->since_resort + L->nsp);
    G.launches = L->launches - launches0;
    if (L->graphs.size() >= 8) {
        cudaGraphExecDestroy(L->graphs.front().exec);
        L->graphs.erase(L->graphs.begin());
    }
    L->graphs.push_back(std::move(G));
    launch_fill_u32(&L->sc->g_base, g0, 1, 1, L->stream);
    L->g_dev = (int64_t)g0;
    if ((rc = cuda_fail(L, cudaGraphLaunch(exec, L->stream)))) return rc;
    L->launches += 1;
    *done = K;
    return PSC_OK;
}

// Events of a call up to t_end, at most max_events (an estimate).
static int64_t events_ahead(const psc_lattice* L, double t_end, int64_t max_events)
{
    double n = 0.0;
    for (int s = 0; s < L->nsp && t_end < INFINITY; ++s)
        if (L->sp[s].D > 0.0) n += std::max(0.0, std::floor(t_end / L->sp[s].tau) - (double)L->sp[s].done);
    return t_end < INFINITY && n < (double)max_events ? (int64_t)n : max_events;
}

// Stretches of large lattices start with a pass over the voxels, their first ones with
// an allocation too: 100 us at 400^3 for k_walk_run, 280 for k_small_run, as long as 15
// and 30 events of short lists in the other kernels (events of lists of a million gain
// twice as much).  Calls with fewer events than these stay there, until as many have run so.
// us of a first call of 1 / 5 events on 400^3, with the pass / put off: 100,000 walkers
// 143 / 170, 34 / 82; A + B -> C of 1000 molecules each 320 / 330, 38 / 119.
static bool pass_pays(const psc_lattice* L, int64_t events)
{
    int64_t longest = 0;
    for (int s = 0; s < L->nsp; ++s)
        if (L->sp[s].D > 0.0) longest = std::max<int64_t>(longest, L->est[s]);
    return L->ahead >= events * (1 << 20) / ((1 << 20) + longest) - L->waited;
}

// Queue events in scheduler order until max_events are queued or the next
// event lies after t_end.  Consecutive events of one species without
// reactions are grouped into persistent stretches (cut at re-sort points).
int drive(psc_lattice* L, double t_end, int64_t max_events)
{
    int64_t queued = 0;
    L->ahead = events_ahead(L, t_end, max_events);
    const bool walks = L->claim_vacancy || L->V <= kWalkVoxels || pass_pays(L, L->V >> 22);
    const bool smalls = L->small.cells_hold || L->V <= (1ll << 22) || pass_pays(L, L->V >> 21);
    while (queued < max_events) {
        int s;
        double t;
        if (!next_event(L, &s, &t) || t > t_end) break;
        refresh_estimates(L);
        if (L->g == UINT32_MAX) return PSC_E_LIMIT;
        if (L->opt.subvolume > 0) {
            // the sub-volume rule: stretches of the species' events, one launch each
            const uint32_t g0 = L->g;
            const int64_t limit = std::max<int64_t>(
                1, std::min<int64_t>(std::min<int64_t>(max_events - queued, (int64_t)1 << 16),
                                     (int64_t)UINT32_MAX - L->g));
            int64_t e = 0;
            for (;;) {
                L->sp[s].done++;
                L->g++;
                L->clock = t;
                ++e;
                if (e >= limit) break;
                int s2;
                double t2;
                if (!next_event(L, &s2, &t2) || s2 != s || t2 > t_end) break;
                t = t2;
            }
            L->g = g0;
            int rc = enqueue_subvol(L, s, e);
            L->g = g0 + (uint32_t)e;
            if (rc) return rc;
            queued += e;
            continue;
        }
        const bool walk = walk_fits(L, s);
        if (walk && walks) {
            int64_t e = 0;
            if (int rc = grid_current(L, true)) return rc;
            int rc = walk_stretch(L, s, t, t_end, max_events - queued, &e);
            if (rc) return rc;
            queued += e;
            continue;
        }
        if (int rc = claims_free(L)) return rc;
        const bool small = small_fits(L);
        if (small && smalls) {
            int64_t e = 0;
            int rc = small_stretch(L, s, t, t_end, max_events - queued, &e);
            if (rc) return rc;
            queued += e;
            if (e > 0) continue;
        }
        const bool waits = (walk && !walks) || (small && !smalls);
        if (waits) L->waited++;
        if (int rc = grid_current(L, true)) return rc;
        int threads = 0, blocks = 0;
        const bool open = open_route(L, s);
        const int per = open ? 0 : run_width(L, s, &threads, &blocks);
        TilePlan plan{};
        // the tile kernel needs no molecule slots per thread: it also takes
        // species above the molecule-list kernel's capacity
        const bool tiles = !open && L->opt.persistent > 0 && !L->general[s] && tile_plan(L, s, &plan);
        if (!tiles)
            if (int rc = sort_first(L, s)) return rc;
        if (per > 0 || tiles) {
            // how long does species s stay next?  (Tile stretches keep their
            // own spatial order: no re-sort points.)
            const uint32_t g0 = L->g;
            int64_t limit = max_events - queued;
            if (L->opt.resort_period > 0 && !tiles)
                limit = std::min<int64_t>(limit, (int64_t)L->opt.resort_period - (int64_t)L->since_resort[s]);
            if (tiles) limit = std::min<int64_t>(limit, (int64_t)1 << 16);   // bounded launch length
            limit = std::max<int64_t>(1, std::min<int64_t>(limit, (int64_t)UINT32_MAX - L->g));
            int64_t e = 0;
            for (;;) {
                L->sp[s].done++;
                L->g++;
                L->clock = t;
                ++e;
                if (e >= limit) break;
                int s2;
                double t2;
                if (!next_event(L, &s2, &t2) || s2 != s || t2 > t_end) break;
                t = t2;
            }
            L->g = g0;                                   // event_args reads the first index
            int rc = tiles ? enqueue_tiles(L, s, e, plan) : enqueue_run(L, s, (int)e, per, threads, blocks);
            L->g = g0 + (uint32_t)e;
            if (rc) return rc;
            queued += e;
            if (waits) L->waited += e - 1;
            if (tiles) continue;
            L->since_resort[s] += (uint64_t)e;
            if (L->opt.resort_period > 0 && L->since_resort[s] >= (uint64_t)L->opt.resort_period) {
                L->since_resort[s] = 0;
                if (sorted_order_pays(L, s)) {
                    cudaEvent_t sp = span_open(L);
                    rc = resort(L, s);
                    span_close(L, sp, kSpanResort);
                    if (rc) return rc;
                }
            }
            continue;
        }
        if (waits) {                                 // (nor are graphs captured for these few)
            int rc = enqueue_event(L, s);
            L->sp[s].done++;
            L->g++;
            L->clock = t;
            if (rc) return rc;
            ++queued;
            continue;
        }
        if (L->opt.graph_events > 1) {
            int64_t done = 0;
            int rc = graph_run(L, t_end, max_events - queued, &done);
            if (rc) return rc;
            if (done > 0) {
                queued += done;
                continue;
            }
        }
        int rc = single_event(L, s, t);
        if (rc) return rc;
        ++queued;
    }
    return PSC_OK;
}

}  // namespace psc_rt

extern "C" {

int psc_run(psc_lattice* L, double t_end)
{
    if (!L || !std::isfinite(t_end)) return PSC_E_ARG;
    if (!L->populated) return PSC_E_ORDER;
    if (L->sticky) return L->sticky;
    DevGuard dg(L->device);
    int rc = drive(L, t_end, INT64_MAX);
    if (rc) return rc;
    if (t_end > L->clock) L->clock = t_end;
    return PSC_OK;
}

int psc_run_events(psc_lattice* L, int64_t n_events)
{
    if (!L || n_events < 0) return PSC_E_ARG;
    if (!L->populated) return PSC_E_ORDER;
    if (L->sticky) return L->sticky;
    DevGuard dg(L->device);
    return drive(L, INFINITY, n_events);
}

int psc_synchronize(psc_lattice* L)
{
    if (!L) return PSC_E_ARG;
    DevGuard dg(L->device);
    return check_device(L);
}

int psc_counts(psc_lattice* L, int64_t* counts, int32_t n)
{
    if (!L || !counts || n < L->nsp) return PSC_E_ARG;
    for (int s = 0; s < n; ++s) counts[s] = s < L->nsp ? L->sp[s].n0 : 0;
    if (!L->populated) return PSC_OK;
    DevGuard dg(L->device);
    int rc = check_device(L);
    if (rc) return rc;
    for (int s = 0; s < L->nsp; ++s) counts[s] = L->state[s];
    return PSC_OK;
}

static int read_list(psc_lattice* L, int32_t s, std::vector<int32_t>& vox, std::vector<uint32_t>& ids,
                     std::vector<uint64_t>* img)
{
    int rc = check_device(L);
    if (rc) return rc;
    const int32_t n = L->state[s];
    L->d2h += (uint64_t)n * (img ? 16 : 8);
    const SpeciesList& l = L->model_h.lists[s];
    vox.resize(n);
    ids.resize(n);
    if (n > 0) {
        if ((rc = cuda_fail(L, cudaMemcpy(vox.data(), l.vox, (size_t)n * 4, cudaMemcpyDeviceToHost)))) return rc;
        if ((rc = cuda_fail(L, cudaMemcpy(ids.data(), l.ids, (size_t)n * 4, cudaMemcpyDeviceToHost)))) return rc;
        if (img) {
            img->resize(n);
            if ((rc = cuda_fail(L, cudaMemcpy(img->data(), l.img, (size_t)n * 8, cudaMemcpyDeviceToHost)))) return rc;
        }
    }
    return PSC_OK;
}

// The number of molecules of species s, for a call that only sizes its buffers
static int list_size(psc_lattice* L, int32_t s, int64_t* n_out)
{
    int rc = check_device(L);
    if (rc) return rc;
    const int32_t n = L->state[s];
    *n_out = n;
    return n > 0 ? PSC_E_ARG : PSC_OK;
}

// Read-out order by molecule id.  Ids are never reused, so when the ids of a
// list span exactly as many values as it has entries (every species without
// reactions keeps the ids placement gave it) each entry goes straight to
// its place; otherwise they are sorted.
static void order_by_id(const std::vector<uint32_t>& ids, std::vector<int64_t>& order)
{
    const int64_t n = (int64_t)ids.size();
    order.assign((size_t)n, -1);
    if (n == 0) return;
    const auto mm = std::minmax_element(ids.begin(), ids.end());
    const uint32_t lo = *mm.first;
    bool placed = (int64_t)*mm.second - (int64_t)lo + 1 == n;
    for (int64_t a = 0; placed && a < n; ++a) {
        int64_t& slot = order[ids[a] - lo];
        if (slot >= 0) placed = false;                   // a repeated id: sort instead
        slot = a;
    }
    if (placed) return;
    for (int64_t a = 0; a < n; ++a) order[a] = a;
    std::sort(order.begin(), order.end(), [&](int64_t x, int64_t y) { return ids[x] < ids[y]; });
}

// The n molecules of list s in id order, built on the device and copied to the
// caller's host buffers in one piece each: entries of a species without
// reactions go straight to their places, its ids being the ones placement gave
// it; else the ids are sorted with their slots, where the list fits the
// re-sort scratch.  Returns PSC_OK, an error, or 1 when the caller should build
// the answer on the host.
static int device_positions(psc_lattice* L, int32_t s, int64_t n, bool unwrapped, int32_t* out,
                            uint32_t* ids_out)
{
    const bool by_id = !L->live[s] && n == L->sp[s].n0;
    if (n <= 0 || (n > L->rs_max && !by_id)) return 1;
    // the list passes' scratch, 24 bytes per entry of the longest list (16 are used)
    int32_t* pos = L->tmp.vox;
    uint32_t* ids = reinterpret_cast<uint32_t*>(pos + 3 * n);
    const int blocks = event_blocks(L, n);
    if (by_id) {
        uint32_t id_lo = 0;
        for (int x = 0; x < s; ++x) id_lo += (uint32_t)L->sp[x].n0;
        if (readout_by_id(L->model_h.lists[s], (int32_t)n, id_lo, L->ni, L->nj, L->nk, unwrapped,
                          (L->bflags & PSC_FCC) != 0, pos, ids, &L->sc->err, blocks, L->stream, &L->launches) != 0)
            return cuda_fail(L, cudaErrorUnknown);
    } else if (readout_positions(L->model_h.lists[s], (int32_t)n, L->ni, L->nj, L->nk, unwrapped,
                          (L->bflags & PSC_FCC) != 0, L->rs_keys, L->rs_vals, L->rs_scratch, pos, ids, blocks,
                          L->stream, &L->launches) != 0)
        return cuda_fail(L, cudaErrorUnknown);
    make_present(out, (size_t)n * 12);
    if (ids_out) make_present(ids_out, (size_t)n * 4);
    int rc = cuda_fail(L, cudaMemcpyAsync(out, pos, (size_t)n * 12, cudaMemcpyDeviceToHost, L->stream));
    if (!rc && ids_out)
        rc = cuda_fail(L, cudaMemcpyAsync(ids_out, ids, (size_t)n * 4, cudaMemcpyDeviceToHost, L->stream));
    if (!rc) rc = cuda_fail(L, cudaStreamSynchronize(L->stream));
    if (rc) return rc;
    L->d2h += (uint64_t)n * (ids_out ? 16 : 12);
    return PSC_OK;
}

int psc_coords(psc_lattice* L, int32_t s, int32_t* ijk, uint32_t* ids_out, int64_t cap, int64_t* n_out)
{
    if (!L || !n_out || s < 0 || s >= L->nsp) return PSC_E_ARG;
    if (!L->populated) return PSC_E_ORDER;
    DevGuard dg(L->device);
    if (!ijk || cap <= 0) return list_size(L, s, n_out);
    int rc = list_size(L, s, n_out);               // E_ARG here only says the list is not empty
    if (rc != PSC_OK && rc != PSC_E_ARG) return rc;
    if (*n_out > cap) return PSC_E_ARG;
    if ((rc = device_positions(L, s, *n_out, false, ijk, ids_out)) <= 0) return rc;
    std::vector<int32_t> vox;
    std::vector<uint32_t> ids;
    rc = read_list(L, s, vox, ids, nullptr);
    if (rc) return rc;
    const int64_t n = (int64_t)vox.size();
    *n_out = n;
    if (n > cap) return PSC_E_ARG;
    std::vector<int64_t> order;
    order_by_id(ids, order);
    const uint32_t ni = (uint32_t)L->ni, nj = (uint32_t)L->nj;
    for (int64_t a = 0; a < n; ++a) {
        const uint32_t v = (uint32_t)vox[order[a]], q = v / ni;
        ijk[3 * a + 0] = (int32_t)(v - q * ni);
        ijk[3 * a + 1] = (int32_t)(q % nj);
        ijk[3 * a + 2] = (int32_t)(q / nj);
        if (ids_out) ids_out[a] = ids[order[a]];
    }
    return PSC_OK;
}

int psc_unwrapped(psc_lattice* L, int32_t s, int32_t* xyz, uint32_t* ids_out, int64_t cap, int64_t* n_out)
{
    if (!L || !n_out || s < 0 || s >= L->nsp) return PSC_E_ARG;
    if (!L->populated) return PSC_E_ORDER;
    DevGuard dg(L->device);
    if (!xyz || cap <= 0) return list_size(L, s, n_out);
    int rc = list_size(L, s, n_out);               // E_ARG here only says the list is not empty
    if (rc != PSC_OK && rc != PSC_E_ARG) return rc;
    if (*n_out > cap) return PSC_E_ARG;
    if ((rc = device_positions(L, s, *n_out, true, xyz, ids_out)) <= 0) return rc;
    std::vector<int32_t> vox;
    std::vector<uint32_t> ids;
    std::vector<uint64_t> img;
    rc = read_list(L, s, vox, ids, &img);
    if (rc) return rc;
    const int64_t n = (int64_t)vox.size();
    *n_out = n;
    if (n > cap) return PSC_E_ARG;
    std::vector<int64_t> order;
    order_by_id(ids, order);
    const uint32_t ni = (uint32_t)L->ni, nj = (uint32_t)L->nj;
    for (int64_t a = 0; a < n; ++a) {
        const uint32_t v = (uint32_t)vox[order[a]], q = v / ni;
        const uint64_t w = img[order[a]];
        const int32_t i = (int32_t)(v - q * ni), j = (int32_t)(q % nj), k = (int32_t)(q / nj);
        const int32_t I = i + (int32_t)(int16_t)(w & 0xFFFF) * L->ni;
        const int32_t J = j + (int32_t)(int16_t)((w >> 16) & 0xFFFF) * L->nj;
        const int32_t K = k + (int32_t)(int16_t)((w >> 32) & 0xFFFF) * L->nk;
        if (L->bflags & PSC_FCC) {
            const int32_t c3 = ((K % 3) + 3) % 3;
            xyz[3 * a + 0] = 2 * I + ((J + (c3 == 1 ? 1 : 0)) & 1);
            xyz[3 * a + 1] = 3 * J + c3;
        } else {
            xyz[3 * a + 0] = 2 * I + ((J + K) & 1);
            xyz[3 * a + 1] = 3 * J + (K & 1);
        }
        xyz[3 * a + 2] = K;
        if (ids_out) ids_out[a] = ids[order[a]];
    }
    return PSC_OK;
}

int psc_grid(psc_lattice* L, uint16_t* occ)
{
    if (!L || !occ) return PSC_E_ARG;
    if (!L->populated) return PSC_E_ORDER;
    DevGuard dg(L->device);
    int rc = check_device(L);
    if (rc) return rc;
    if ((rc = grid_current(L, false))) return rc;
    if (L->small.cells_hold) {                       // grid_current wrote the code of every voxel
        make_present(occ, (size_t)L->V * 2);
        rc = cuda_fail(L, cudaMemcpyAsync(occ, L->occ, (size_t)L->V * 2, cudaMemcpyDeviceToHost, L->stream));
        if (!rc) rc = cuda_fail(L, cudaStreamSynchronize(L->stream));
        L->d2h += (uint64_t)L->V * 2;
        return rc;
    }
    // exact codes: mirror-masked codes of species with reactions, then the
    // species without reactions from their lists
    const bool own = (size_t)L->V * 2 > L->scratch_bytes;
    uint16_t* tmp = own ? (uint16_t*)dev_alloc(L, (size_t)L->V * 2) : (uint16_t*)L->scratch;
    if (!tmp) return PSC_E_NOMEM;
    const int blocks = L->sm_count * 8;
    launch_materialize(tmp, L->occ, L->bits, L->mirror_n, L->labels.empty() ? 1 : L->ncomp, L->geo, L->V, blocks,
                       L->stream);
    for (int s = 0; s < L->nsp; ++s)
        if (!L->live[s])
            launch_scatter_codes(tmp, L->model_h.lists[s], &L->sc->counts[s], (uint16_t)(s + 1), blocks,
                                 L->stream);
    L->launches += 1;
    make_present(occ, (size_t)L->V * 2);
    rc = cuda_fail(L, cudaStreamSynchronize(L->stream));
    if (!rc) rc = cuda_fail(L, cudaMemcpy(occ, tmp, (size_t)L->V * 2, cudaMemcpyDeviceToHost));
    L->d2h += (uint64_t)L->V * 2;
    if (own) dev_free_one(L, tmp);
    return rc;
}

int psc_time(const psc_lattice* L, double* t)
{
    if (!L || !t) return PSC_E_ARG;
    *t = L->clock;
    return PSC_OK;
}

int psc_event_index(const psc_lattice* L, uint32_t* g)
{
    if (!L || !g) return PSC_E_ARG;
    *g = L->g;
    return PSC_OK;
}

int psc_stats_get(psc_lattice* L, psc_stats* out)
{
    if (!L || !out) return PSC_E_ARG;
    std::memset(out, 0, sizeof(*out));
    out->events = L->events;
    out->launches = (uint64_t)L->launches;
    out->h2d_bytes = L->h2d;
    out->d2h_bytes = L->d2h;
    if (!L->populated) return PSC_OK;
    DevGuard dg(L->device);
    int rc = check_device(L);
    if (rc) return rc;
    unsigned long long st[kNumStats];
    if ((rc = cuda_fail(L, cudaMemcpy(st, L->sc->stats, sizeof(st), cudaMemcpyDeviceToHost)))) return rc;
    L->d2h += sizeof(st);
    out->attempts = st[kStatAttempts];
    out->hops = st[kStatHops];
    out->collisions = st[kStatCollisions];
    out->accepted = st[kStatAccepted];
    out->reactions2 = st[kStatReactions2];
    out->fires = st[kStatFires];
    out->reactions1 = st[kStatReactions1];
    out->births = st[kStatBirths];
    return PSC_OK;
}

int psc_set_options(psc_lattice* L, const psc_options* o)
{
    if (!L || !o) return PSC_E_ARG;
    if (o->block_threads && (o->block_threads < 32 || o->block_threads > 256 || (o->block_threads & 31)))
        return PSC_E_ARG;
    if (o->blocks_per_sm < 0) return PSC_E_ARG;
    graph_cache_clear(L);                            // captured launches follow the options
    std::memset(L->open_auto, 0, sizeof(L->open_auto));
    L->small.no_room = false;
    L->small.version++;
    if (o->resort_period) L->opt.resort_period = o->resort_period;
    if (o->block_threads) L->opt.block_threads = o->block_threads;
    if (o->blocks_per_sm) L->opt.blocks_per_sm = o->blocks_per_sm;
    if (o->collect_stats) L->opt.collect_stats = o->collect_stats;
    if (o->graph_events) L->opt.graph_events = o->graph_events < 0 ? 0 : o->graph_events;
    if (o->time_kernels) L->opt.time_kernels = o->time_kernels;
    if (o->claim_table) {
        if (o->claim_table < -1 || o->claim_table > 2) return PSC_E_ARG;
        if (L->populated) return PSC_E_ORDER;
        L->opt.claim_table = o->claim_table;
    }
    if (o->persistent) L->opt.persistent = o->persistent;
    if (o->run_per_thread) L->opt.run_per_thread = o->run_per_thread < 0 ? 0 : o->run_per_thread;
    if (o->barrier_timeout_us) {
        if (o->barrier_timeout_us < 0) return PSC_E_ARG;
        L->opt.barrier_timeout_us = o->barrier_timeout_us;
    }
    if (o->barrier_phantom) L->opt.barrier_phantom = o->barrier_phantom < 0 ? 0 : o->barrier_phantom;
    if (o->tiles) L->opt.tiles = o->tiles > 0 ? 1 : -1;
    if (o->subvolume) {
        if (L->populated) return PSC_E_ORDER;
        L->opt.subvolume = o->subvolume > 0 ? 1 : -1;
    }
    if (o->tile_regions) L->opt.tile_regions = o->tile_regions < 0 ? 0 : o->tile_regions;
    if (o->tile_lean) L->opt.tile_lean = o->tile_lean > 0 ? 1 : -1;
    if (o->slot_map) {
        if (o->slot_map < 1 || o->slot_map > 3) return PSC_E_ARG;
        L->opt.slot_map = o->slot_map;
    }
    if (o->claim_slots) {
        if (o->claim_slots < 2 || o->claim_slots > 64) return PSC_E_ARG;
        if (L->populated) return PSC_E_ORDER;
        L->opt.claim_slots = o->claim_slots;
    }
    return PSC_OK;
}

int psc_kernel_times_get(psc_lattice* L, psc_kernel_times* out)
{
    if (!L || !out) return PSC_E_ARG;
    std::memset(out, 0, sizeof(*out));
    DevGuard dg(L->device);
    cudaError_t e = cudaStreamSynchronize(L->stream);
    if (e != cudaSuccess) return cuda_fail(L, e);
    for (const auto& sp : L->spans) {
        float ms = 0.0f;
        if (cudaEventElapsedTime(&ms, sp.a, sp.b) != cudaSuccess) ms = 0.0f;
        switch (sp.kind) {
        case kSpanClaim: out->claim_ms += ms; out->claim_launches++; break;
        case kSpanCommit: out->commit_ms += ms; out->commit_launches++; break;
        case kSpanReconcile: out->reconcile_ms += ms; out->reconcile_events++; break;
        case kSpanRun: out->run_ms += ms; out->run_launches++; out->run_events += sp.events; break;
        case kSpanTile:
        case kSpanTileLean:
            out->run_ms += ms; out->run_launches++; out->run_events += sp.events;
            out->tile_launches++; out->tile_events += sp.events;
            if (sp.kind == kSpanTileLean) out->tile_lean_events += sp.events;
            break;
        default: out->resort_ms += ms; out->resorts++; break;
        }
        L->event_pool.push_back(sp.a);
        L->event_pool.push_back(sp.b);
    }
    L->spans.clear();
    return PSC_OK;
}

int psc_device_bytes(const psc_lattice* L, int64_t* bytes)
{
    if (!L || !bytes) return PSC_E_ARG;
    const int64_t mirrors = L->labels.empty() ? 1 : L->ncomp;
    const int64_t mwords = (int64_t)mirror_words(L->ni, L->nj, L->nk);
    int64_t b = L->V * 2 + mwords * 4 * mirrors + 2 * ((mwords + 31) / 32) * 4 + (int64_t)sizeof(Scalars) +
                (int64_t)sizeof(ModelDev);
    if (L->small.ev) b += (int64_t)L->nsp * (int64_t)sizeof(EventArgs);
    if (L->small.cell) b += mwords * 128;
    b += (int64_t)L->small.scratch_n * 8;
    if (L->claim) b += L->claim_n * 4;
    b += 2 * L->table_slots * 8;
    int64_t N = 0;
    for (int s = 0; s < L->nsp; ++s) N += L->sp[s].n0;
    if (L->populated) {
        int64_t mx = 1, mm = 1;
        for (int s = 0; s < L->nsp; ++s) {
            b += (int64_t)L->model_h.lists[s].cap * 16;
            mx = std::max<int64_t>(mx, L->cap[s]);
            if (L->sp[s].D > 0.0) mm = std::max<int64_t>(mm, L->cap[s]);
        }
        b += mx * 24 + (int64_t)L->births_cap * (int64_t)sizeof(Birth) + mm * 8 +
             (int64_t)sort_scratch_bytes(mm);
    } else {
        b += 2 * N * 16 + 2 * N * 8;
    }
    // sub-volume rule buffers
    b += L->subvol.subvols * 8 + L->subvol.slots * 17 + (L->subvol.counters ? 128 : 0);
    // tile kernel buffers, once a stretch has used them
    const auto& T = L->tile;
    b += T.slots * 4 * 5 + (int64_t)T.regions * 4 * 4 + T.ids * 8 + T.halo_entries * (int64_t)sizeof(uint2);
    if (T.claim) b += L->V * 4;
    *bytes = b;
    return PSC_OK;
}

void psc_lattice_destroy(psc_lattice* L)
{
    if (!L) return;
    {
        DevGuard dg(L->device);
        if (L->stream) cudaStreamSynchronize(L->stream);
        for (const auto& sp : L->spans) { cudaEventDestroy(sp.a); cudaEventDestroy(sp.b); }
        for (cudaEvent_t ev : L->event_pool) cudaEventDestroy(ev);
        if (L->counts_ev) cudaEventDestroy(L->counts_ev);
        counts_free(L);
        graph_cache_clear(L);
        dev_free_all(L);
        if (L->own_stream && L->stream) cudaStreamDestroy(L->stream);
    }
    delete L;
}

}  // extern "C"
