// psc_batch.cpp -- batches of lattices advanced by shared launches, and the
// serving loop built on them (continuous batching with admission by device
// memory).  Each member of a batch keeps its own scheduler (Sec. 2.2); one
// batched launch per event phase covers every member's next event.
#include "psc.h"
#include "psc_internal.h"
#include "psc_runtime.h"

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstring>
#include <deque>
#include <map>
#include <new>
#include <vector>

using namespace psc;
using namespace psc_rt;

namespace {

constexpr int kItemBlocksMaxDefault = 64;   // blocks per member per launch (grid-stride inside)
constexpr int kItemThreadsDefault = 256;   // threads per block of the batched launches

struct Member {
    psc_lattice* L = nullptr;
    double t_stop = INFINITY;             // run events up to this time
    uint32_t args = 0;                    // SmallBuffers::version of what args_d holds of it (0: nothing)
    bool stretch = false;                 // runs in stretches (else in batched launches per event phase)
};

}  // namespace

constexpr int kNarrow = 2;
constexpr int kNarrowMost = 8;             // times stretch_blocks, at most
constexpr int kNarrowThreads[kNarrow] = {kSmallThreads / 2, kSmallThreads / 4};

struct psc_batch {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    Member slot[kBatchMax];
    int32_t size = 0;
    EventArgs* tmpl_ev = nullptr;         // [kBatchMax][kMaxSpecies] on the device
    ReconcileArgs* tmpl_rc = nullptr;
    int64_t launches = 0;
    int threads = kItemThreadsDefault;
    int item_blocks_max = kItemBlocksMaxDefault;
    int32_t resort_period = -1;           // events of a member's species between Morton re-sorts (-1 never)
    // stretches of the members' events, one launch for many members
    int stretch_blocks = -1;              // most blocks of a launch (-1: not asked, 0: no stretches)
    int narrow_blocks[kNarrow][2] = {{-1, -1}, {-1, -1}};       // of fewer threads; without and with births
    int sm_count = 0;
    bool use_stretches = true;
    SmallArgs* args_d = nullptr;          // [kBatchMax], device: a member's, but for its events
    char* upload_d = nullptr;             // stretches, blocks' groups and events of a call
    int32_t* counts_d = nullptr;          // [kBatchMax][kSmallCounts] list lengths after a stretch
    int32_t* counts_h = nullptr;          // pinned copy, for the next stretch's groups
    cudaEvent_t counts_ev = nullptr;
    bool counts_pending = false;
    int64_t counts_age = INT64_MAX / 2;   // events of a call since the last copy was queued
    std::vector<std::pair<psc_lattice*, uint32_t>> counts_of;  // whose lengths counts_h holds (null: no member
                                                               // any more), after which event
};

namespace {

int item_blocks(const psc_batch* B, int64_t work)
{
    const int64_t b = (work + B->threads - 1) / B->threads;
    return (int)std::max<int64_t>(1, std::min<int64_t>(b, B->item_blocks_max));
}

// Queue the next event of every member whose next event time is <= its
// t_stop (and <= t_cap); returns how many members had one.
// (all: members that could run in stretches too.)
int batch_event(psc_batch* B, double t_cap, bool all, int* rc_out)
{
    *rc_out = PSC_OK;
    struct Act {
        int slot, s;
        double t;
    };
    Act acts[kBatchMax];
    int na = 0;
    static thread_local BatchLaunch bl;
    bl.n = 0;
    int total = 0;
    for (int i = 0; i < kBatchMax; ++i) {
        psc_lattice* L = B->slot[i].L;
        if (!L || L->sticky || (!all && B->slot[i].stretch)) continue;
        int s;
        double t;
        if (!next_event(L, &s, &t) || t > B->slot[i].t_stop || t > t_cap || L->g == UINT32_MAX) continue;
        acts[na++] = {i, s, t};
        if ((*rc_out = claims_free(L)) || (*rc_out = grid_current(L, true))) return 1;
        BatchItem& it = bl.item[bl.n++];
        it.rep = i;
        it.sel = s;
        it.g = L->g;
        it.block0 = total;
        it.mask = 0;
        total += item_blocks(B, L->cap[s]);
    }
    if (na == 0) return 0;
    bl.total_blocks = total;
    launch_claim_batch(B->tmpl_ev, bl, B->threads, B->stream);
    launch_commit_batch(B->tmpl_ev, bl, B->threads, B->stream);
    B->launches += 2;
    // list passes: the k-th partner list of each member's event checked
    // against the member's grid (list 0 is the member's own species, whose
    // commit noted its leavers), then every list of every member's event
    // filled, a block each; a list's scratch range follows those of the lists
    // before it in the member's order
    for (int k = 1;; ++k) {
        bl.n = 0;
        total = 0;
        for (int a = 0; a < na; ++a) {
            psc_lattice* L = B->slot[acts[a].slot].L;
            const std::vector<int>& rec = L->reconcile[acts[a].s];
            if (k >= (int)rec.size()) continue;
            BatchItem& it = bl.item[bl.n++];
            it.rep = acts[a].slot;
            it.sel = rec[k];
            it.g = L->g;                  // the event's parity picks the commit's dirty map
            it.block0 = total;
            it.mask = 0;
            for (int q = 0; q < k; ++q) it.mask |= 1u << rec[q];
            total += item_blocks(B, L->cap[rec[k]]);
        }
        if (bl.n == 0) break;
        bl.total_blocks = total;
        launch_reconcile_batch(B->tmpl_rc, bl, B->threads, B->stream);
        B->launches += 1;
    }
    bl.n = 0;
    for (int a = 0; a < na; ++a) {
        psc_lattice* L = B->slot[acts[a].slot].L;
        const std::vector<int>& rec = L->reconcile[acts[a].s];
        uint32_t before = 0;
        for (int x : rec) {
            BatchItem& it = bl.item[bl.n++];
            it.rep = acts[a].slot;
            it.sel = x;
            it.g = L->g;
            it.block0 = bl.n - 1;
            it.mask = before;
            before |= 1u << x;
            if (bl.n == kBatchMax) {
                bl.total_blocks = bl.n;
                launch_fill_batch(B->tmpl_rc, bl, B->stream);
                B->launches += 1;
                bl.n = 0;
            }
        }
    }
    if (bl.n > 0) {
        bl.total_blocks = bl.n;
        launch_fill_batch(B->tmpl_rc, bl, B->stream);
        B->launches += 1;
    }
    bl.n = 0;
    for (int a = 0; a < na; ++a) {
        psc_lattice* L = B->slot[acts[a].slot].L;
        if (!L->fo2[acts[a].s]) continue;
        BatchItem& it = bl.item[bl.n];
        it.rep = acts[a].slot;
        it.sel = acts[a].s;
        it.g = L->g;
        it.block0 = bl.n;
        it.mask = 0;
        bl.n++;
    }
    if (bl.n > 0) {
        bl.total_blocks = bl.n;
        launch_births_batch(B->tmpl_ev, bl, B->stream);
        B->launches += 1;
    }
    const cudaError_t e = cudaPeekAtLastError();
    if (e != cudaSuccess) {
        *rc_out = PSC_E_CUDA;
        return na;
    }
    for (int a = 0; a < na; ++a) {
        psc_lattice* L = B->slot[acts[a].slot].L;
        L->sp[acts[a].s].done++;
        L->g++;
        L->clock = acts[a].t;
        L->events++;
        L->launches += 2;
        // the member's list in Morton order again every resort_period of its events (the order of a
        // list never changes results)
        if (B->resort_period > 0 && ++L->since_resort[acts[a].s] >= (uint64_t)B->resort_period) {
            L->since_resort[acts[a].s] = 0;
            const int rc = psc_rt::resort(L, acts[a].s);
            if (rc) {
                *rc_out = rc;
                return na;
            }
        }
    }
    return na;
}

// ---------------------------------------------------------------------------
// stretches: every member's events in a group of blocks of its own, at its own
// pace, one launch for as many members as there are blocks on the device
// ---------------------------------------------------------------------------
// of a call that advances kBatchMax members by kSmallEvents events, in launches of at
// most `blocks` blocks, at least one for each member
constexpr int kUploadLaunches = 16;
size_t upload_bytes(int blocks)
{
    return kBatchMax * (sizeof(SmallStretch) + kSmallEvents + sizeof(int32_t)) +
           (kUploadLaunches + 1) * (size_t)blocks * sizeof(int32_t);
}

// Launches of a call over `total` members with so many bytes of cells and molecules
// an event: as few as there are blocks for.  Where the cells do not fit in the L2
// cache together, members take turns instead, each launch with the cells that fit, as
// long as it has kSplitMolecules molecules per block and its groups fill the blocks
// to 0.85.  us for an event of every member, launches per event phase / all members
// at once / in turns, calls of 64 events: 64 walkers' lattices of 160^3 at 2 % 455 / 517 /
// 250, of 96^3 at 30 % 834 / 973 / 641, 32 of 128^3 at 20 % 761 / 884 / 544, 64 of A + B -> C on
// 160^3 at 2 % 401 / 236 / 173; calls of one event: 470 / 560 / 470, 828 / 1029 / 708,
// 759 / 941 / 613, 420 / 283 / 300.
constexpr double kSplitMolecules = 4096.0, kSplitBytes = 4.0 * (double)kWalkVoxels;
int stretch_launches(int total, int blocks, double bytes, double molecules)
{
    const int least = (total + blocks - 1) / blocks;
    const int most = (int)std::min<double>({molecules / (kSplitMolecules * blocks), (double)total, (double)kUploadLaunches});
    for (int l = std::min((int)std::min(std::ceil(bytes / kSplitBytes), (double)kUploadLaunches), most); l <= most; ++l) {
        const int members = (total + std::max(l, 1) - 1) / std::max(l, 1);
        if (l > least && blocks / members * members >= 0.85 * blocks) return l;
    }
    return least;
}

int stretch_buffers(psc_batch* B, psc_lattice* L)
{
    if (B->stretch_blocks < 0) B->stretch_blocks = small_batch_blocks(L->sm_count, kSmallThreads, true);
    B->sm_count = L->sm_count;
    if (B->stretch_blocks == 0 || B->args_d) return PSC_OK;
    if (cudaMalloc(&B->args_d, sizeof(SmallArgs) * kBatchMax) != cudaSuccess ||
        cudaMalloc(&B->upload_d, upload_bytes(kNarrowMost * B->stretch_blocks)) != cudaSuccess ||
        cudaMalloc(&B->counts_d, sizeof(int32_t) * kBatchMax * kSmallCounts) != cudaSuccess ||
        cudaMallocHost(&B->counts_h, sizeof(int32_t) * kBatchMax * kSmallCounts) != cudaSuccess ||
        cudaEventCreateWithFlags(&B->counts_ev, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        B->stretch_blocks = 0;            // what was allocated goes with the batch
    }
    return PSC_OK;
}

// May L run in stretches (*yes)?  extra: bytes of its buffers for that, at most
// `room`.  Without room on the device it runs in batched launches.
int member_stretches(psc_batch* B, psc_lattice* L, int64_t room, int64_t* extra, bool* yes)
{
    *extra = 0;
    *yes = false;
    if (L->opt.persistent <= 0 || L->opt.time_kernels > 0 || L->opt.subvolume > 0) return PSC_OK;
    stretch_buffers(B, L);
    if (B->stretch_blocks <= 0) return PSC_OK;
    if (L->V > kCellVoxels) return PSC_OK;
    for (int s = 0; s < L->nsp; ++s)
        if (L->model_h.lists[s].cap > kCellVoxels) return PSC_OK;
    const int64_t lacks = small_lacks(L, true);
    if (lacks > room) return PSC_OK;
    const int sticky = L->sticky;         // an error it brings along stays
    const int rc = small_buffers(L, true);
    if (rc == PSC_E_NOMEM) {
        cudaGetLastError();
        L->sticky = sticky;
        return PSC_OK;
    }
    if (rc) return rc;
    // a group's barrier goes on from whatever complete barriers left there
    if (cudaMemsetAsync(L->barrier, 0, sizeof(BarrierState), B->stream) != cudaSuccess) return PSC_E_CUDA;
    *extra = lacks;
    *yes = true;
    return PSC_OK;
}

// A copy of the members' list lengths every so many events; the host waits for it
// when the call would take its age to that number (the groups of a long call follow
// the lengths after the one before: served replicas whose lists fall from step to step
// took 4 % longer with older ones).  Waited for by every call, with two copies up
// and a memset in every launch, run_events(1) took 52 us of 64 A + B -> C members on 48^3
// and 133 of 300 on 32^3; now 27 and 40; in launches per event phase 38 and 55.
constexpr int64_t kCountsEvery = 64;

// Up to n_events next events of every member that runs in stretches, up to
// its t_stop and t_cap; the number of members that had any.
int batch_stretch(psc_batch* B, double t_cap, int64_t n_events, int* rc_out)
{
    *rc_out = PSC_OK;
    if (!B->use_stretches || B->stretch_blocks <= 0) return 0;
    // list lengths after an earlier stretch: groups follow them
    if (B->counts_pending && (B->counts_age + n_events >= kCountsEvery || cudaEventQuery(B->counts_ev) == cudaSuccess)) {
        if (cudaEventSynchronize(B->counts_ev) != cudaSuccess) {
            *rc_out = PSC_E_CUDA;
            return 1;
        }
        B->counts_pending = false;
        for (size_t r = 0; r < B->counts_of.size(); ++r) {
            psc_lattice* L = B->counts_of[r].first;
            // (null: it left the batch; it may also have run on by itself and know better)
            if (!L || B->counts_of[r].second < L->next_id_g) continue;
            const int32_t* h = B->counts_h + r * kSmallCounts;
            if (note_errors(L, h[kMaxSpecies + 1])) continue;      // (a wait that ran out: no further events of it)
            for (int s = 0; s < L->nsp; ++s)
                if (h[s] >= 0) L->est[s] = h[s];
            if (h[kMaxSpecies] > 0) {
                L->next_id_known = h[kMaxSpecies];
                L->next_id_g = B->counts_of[r].second;
            }
        }
    }
    std::vector<SmallStretch> stretch;
    std::vector<uint8_t> seq;
    std::vector<double> work;             // molecules per event, entries looked through at the end among them
    std::vector<std::pair<psc_lattice*, uint32_t>> of;
    bool births = false;
    SmallArgs A{};
    for (int i = 0; i < kBatchMax; ++i) {
        psc_lattice* L = B->slot[i].L;
        if (!L || L->sticky || !B->slot[i].stretch) continue;
        if (ids_bound(L) > kCellIds) {    // no more ids for the cells' claims
            B->slot[i].stretch = false;
            continue;
        }
        int s;
        double t;
        if (!next_event(L, &s, &t) || t > B->slot[i].t_stop || t > t_cap || L->g == UINT32_MAX) continue;
        if ((*rc_out = claims_free(L))) return 1;
        if (!L->small.cells_hold || B->slot[i].args != L->small.version) {
            if ((*rc_out = small_args(L, &A))) return 1;
            if (cudaMemcpyAsync(B->args_d + i, &A, offsetof(SmallArgs, seq), cudaMemcpyHostToDevice, B->stream) !=
                cudaSuccess) {
                *rc_out = PSC_E_CUDA;
                return 1;
            }
            B->slot[i].args = L->small.version;
        }
        L->small.grid_stale = true;
        SmallStretch x{};
        x.slot = i;
        x.g = L->g;
        x.seq = (uint32_t)seq.size();
        const int64_t limit = std::min<int64_t>(std::min<int64_t>(n_events, kSmallEvents), (int64_t)UINT32_MAX - L->g);
        double molecules = 0.0, closed = 0.0;                    // closed: lists that may be closed up at the end
        uint32_t may_close = 0;
        do {
            seq.push_back((uint8_t)s);
            x.n_events++;
            molecules += (double)L->est[s];
            may_close |= L->small.closes[s];
            L->sp[s].done++;
            L->g++;
            L->clock = t;
        } while (x.n_events < limit && next_event(L, &s, &t) && t <= B->slot[i].t_stop && t <= t_cap);
        births = births || L->small.fo2 != 0u;
        L->events += (uint64_t)x.n_events;
        L->launches += 1;
        for (; may_close != 0; may_close &= may_close - 1) closed += (double)L->est[__builtin_ctz(may_close)];
        work.push_back((molecules + 0.25 * closed) / x.n_events);
        stretch.push_back(x);
        of.emplace_back(L, L->g);
    }
    if (stretch.empty()) return 0;
    B->counts_age += n_events;
    const int total = (int)stretch.size();
    double bytes = 0.0, molecules = 0.0;
    for (int r = 0; r < total; ++r) {
        bytes += 128.0 * (double)of[(size_t)r].first->mirror_n;
        molecules += work[(size_t)r];
    }
    int blocks_most = B->stretch_blocks, threads = kSmallThreads;
    int launches = stretch_launches(total, blocks_most, bytes, molecules);
    // more members than blocks: narrower blocks, several on an SM, as long as their
    // threads hold the molecules of an event (500 members of 400 molecules on 24^3, calls of
    // 1 / 64 events: 64 / 19.7 us per event in launches one after the other, 27 / 9.6 so)
    for (int w = 0; w < kNarrow && total > B->stretch_blocks; ++w) {
        int& narrow = B->narrow_blocks[w][births ? 1 : 0];
        if (narrow < 0)
            narrow = std::min(small_batch_blocks(B->sm_count, kNarrowThreads[w], births), kNarrowMost * B->stretch_blocks);
        if (narrow <= blocks_most || molecules > 2.0 * kNarrowThreads[w] * total ||
            (total + narrow - 1) / narrow >= launches)
            continue;
        blocks_most = narrow;
        threads = kNarrowThreads[w];
        launches = (total + narrow - 1) / narrow;
    }
    std::vector<int32_t> group;           // of all launches' blocks
    std::vector<int> first;               // block of each launch
    for (int l = 0; l < launches; ++l) {
        const int lo = (int)((int64_t)total * l / launches), hi = (int)((int64_t)total * (l + 1) / launches);
        // blocks by work; an event takes about as long with no molecules as
        // with 600 per block
        double sum = 0.0;
        for (int r = lo; r < hi; ++r) sum += work[(size_t)r] + 600.0;
        const int spare = blocks_most - (hi - lo);
        first.push_back((int)group.size());
        for (int r = lo; r < hi; ++r) {
            const int more = (int)(spare * (work[(size_t)r] + 600.0) / sum);
            const int most = (int)(work[(size_t)r] / threads);           // with it, a molecule per thread
            stretch[(size_t)r].blocks = 1 + std::min(more, most);
            stretch[(size_t)r].block0 = (int)group.size() - first.back();
            group.insert(group.end(), (size_t)stretch[(size_t)r].blocks, r);
        }
    }
    first.push_back((int)group.size());
    // one copy up: stretches, groups, events
    const size_t at_group = sizeof(SmallStretch) * (size_t)total, at_seq = at_group + sizeof(int32_t) * group.size();
    std::vector<char> up(at_seq + seq.size());
    std::memcpy(up.data(), stretch.data(), at_group);
    std::memcpy(up.data() + at_group, group.data(), at_seq - at_group);
    std::memcpy(up.data() + at_seq, seq.data(), seq.size());
    if (cudaMemcpyAsync(B->upload_d, up.data(), up.size(), cudaMemcpyHostToDevice, B->stream) != cudaSuccess) {
        *rc_out = PSC_E_CUDA;
        return total;
    }
    for (int l = 0; l < launches; ++l) {
        if (launch_small_batch(B->args_d, (const SmallStretch*)B->upload_d,
                               (const int32_t*)(B->upload_d + at_group) + first[(size_t)l],
                               (const uint8_t*)B->upload_d + at_seq, B->counts_d,
                               first[(size_t)l + 1] - first[(size_t)l], threads, births, B->stream) != cudaSuccess) {
            *rc_out = PSC_E_CUDA;
            return total;
        }
        B->launches += 1;
    }
    if (B->counts_pending || B->counts_age < kCountsEvery) return total;
    B->counts_of.swap(of);
    if (cudaMemcpyAsync(B->counts_h, B->counts_d, sizeof(int32_t) * kSmallCounts * (size_t)total,
                        cudaMemcpyDeviceToHost, B->stream) != cudaSuccess ||
        cudaEventRecord(B->counts_ev, B->stream) != cudaSuccess) {
        *rc_out = PSC_E_CUDA;
    } else {
        B->counts_pending = true;
        B->counts_age = 0;
    }
    return total;
}

// Up to n_events next events of every member, up to t_cap; false when none had
// any left.
bool batch_advance(psc_batch* B, double t_cap, int64_t n_events, int* rc_out)
{
    const int64_t e = std::min<int64_t>(n_events, kSmallEvents);
    bool any = batch_stretch(B, t_cap, e, rc_out) > 0;
    if (*rc_out) return true;
    for (int64_t x = 0; x < e; ++x) {
        if (batch_event(B, t_cap, !B->use_stretches, rc_out) == 0) break;
        any = true;
        if (*rc_out) return true;
    }
    return any;
}

int upload_templates(psc_batch* B, int slot, psc_lattice* L)
{
    std::vector<EventArgs> ev(kMaxSpecies);
    std::vector<ReconcileArgs> rc(kMaxSpecies);
    for (int s = 0; s < L->nsp; ++s) {
        ev[s] = event_args(L, s);
        rc[s] = reconcile_args(L, s);
    }
    if (cudaMemcpy(B->tmpl_ev + (size_t)slot * kMaxSpecies, ev.data(), sizeof(EventArgs) * kMaxSpecies,
                   cudaMemcpyHostToDevice) != cudaSuccess)
        return PSC_E_CUDA;
    if (cudaMemcpy(B->tmpl_rc + (size_t)slot * kMaxSpecies, rc.data(), sizeof(ReconcileArgs) * kMaxSpecies,
                   cudaMemcpyHostToDevice) != cudaSuccess)
        return PSC_E_CUDA;
    L->h2d += sizeof(EventArgs) * kMaxSpecies + sizeof(ReconcileArgs) * kMaxSpecies;
    return PSC_OK;
}

int batch_add_until(psc_batch* B, psc_lattice* L, double t_stop, int64_t room, int64_t* extra)
{
    if (!B || !L) return PSC_E_ARG;
    if (!L->populated) return PSC_E_ORDER;
    if (L->device != B->device || L->stream != B->stream || !L->claim || !L->batchable) return PSC_E_UNSUPPORTED;
    int free_slot = -1;
    for (int i = 0; i < kBatchMax; ++i) {
        if (B->slot[i].L == L) return PSC_E_ARG;
        if (!B->slot[i].L && free_slot < 0) free_slot = i;
    }
    if (free_slot < 0) return PSC_E_CAPACITY;
    DevGuard dg(B->device);
    int rc = upload_templates(B, free_slot, L);
    if (rc) return rc;
    bool stretch = false;
    if ((rc = member_stretches(B, L, room, extra, &stretch))) return rc;
    B->slot[free_slot].L = L;
    B->slot[free_slot].t_stop = t_stop;
    B->slot[free_slot].stretch = stretch;
    B->slot[free_slot].args = 0;
    B->size++;
    return PSC_OK;
}

}  // namespace

extern "C" {

int psc_batch_create(psc_batch** out, int device, void* cuda_stream)
{
    if (!out || device < 0) return PSC_E_ARG;
    *out = nullptr;
    int ndev = 0;
    if (cudaGetDeviceCount(&ndev) != cudaSuccess || device >= ndev) return PSC_E_CUDA;
    psc_batch* B = new (std::nothrow) psc_batch();
    if (!B) return PSC_E_NOMEM;
    B->device = device;
    DevGuard dg(device);
    if (cuda_stream) {
        B->stream = static_cast<cudaStream_t>(cuda_stream);
    } else {
        if (cudaStreamCreateWithFlags(&B->stream, cudaStreamNonBlocking) != cudaSuccess) { delete B; return PSC_E_CUDA; }
        B->own_stream = true;
    }
    if (cudaMalloc(&B->tmpl_ev, sizeof(EventArgs) * kBatchMax * kMaxSpecies) != cudaSuccess ||
        cudaMalloc(&B->tmpl_rc, sizeof(ReconcileArgs) * kBatchMax * kMaxSpecies) != cudaSuccess) {
        cudaFree(B->tmpl_ev);
        if (B->own_stream) cudaStreamDestroy(B->stream);
        delete B;
        return PSC_E_NOMEM;
    }
    *out = B;
    return PSC_OK;
}

int psc_batch_add(psc_batch* B, psc_lattice* L)
{
    int64_t extra = 0;
    return batch_add_until(B, L, INFINITY, INT64_MAX, &extra);
}

int psc_batch_remove(psc_batch* B, psc_lattice* L)
{
    if (!B || !L) return PSC_E_ARG;
    for (int i = 0; i < kBatchMax; ++i) {
        if (B->slot[i].L == L) {
            B->slot[i].L = nullptr;
            B->size--;
            // list lengths on their way are of the lattice as it was: it may be destroyed,
            // and its address the next member's, before they are looked at
            for (auto& c : B->counts_of)
                if (c.first == L) c.first = nullptr;
            return PSC_OK;
        }
    }
    return PSC_E_ARG;
}

int psc_batch_size(const psc_batch* B, int32_t* n)
{
    if (!B || !n) return PSC_E_ARG;
    *n = B->size;
    return PSC_OK;
}

int64_t psc_batch_launches(const psc_batch* B) { return B ? B->launches : 0; }

int psc_batch_run_events(psc_batch* B, int64_t n_events)
{
    if (!B || n_events < 0) return PSC_E_ARG;
    DevGuard dg(B->device);
    // every member with events left takes part
    for (int64_t e = 0; e < n_events; e += kSmallEvents) {
        int rc;
        if (!batch_advance(B, INFINITY, n_events - e, &rc)) break;
        if (rc) return rc;
    }
    return PSC_OK;
}

int psc_batch_run(psc_batch* B, double t_end)
{
    if (!B || !std::isfinite(t_end)) return PSC_E_ARG;
    DevGuard dg(B->device);
    for (;;) {
        int rc;
        if (!batch_advance(B, t_end, kSmallEvents, &rc)) break;
        if (rc) return rc;
    }
    for (int i = 0; i < kBatchMax; ++i) {
        psc_lattice* L = B->slot[i].L;
        if (L && t_end > L->clock) L->clock = t_end;
    }
    return PSC_OK;
}

// Block shape of the batched launches, tuned by timing batched events.  Like
// the lattice tuner it changes only how work is laid out on the GPU, so the
// trial rounds are real events of every member.
int psc_batch_autotune(psc_batch* B, int64_t max_rounds, psc_batch_tune_result* out)
{
    if (!B || !out || max_rounds < 0) return PSC_E_ARG;
    std::memset(out, 0, sizeof(*out));
    DevGuard dg(B->device);
    cudaEvent_t a = nullptr, b = nullptr;
    if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) {
        if (a) cudaEventDestroy(a);
        return PSC_E_CUDA;
    }
    const int64_t W = std::max<int64_t>(2, std::min<int64_t>(64, max_rounds / 14));
    int64_t budget = max_rounds;
    int rc = PSC_OK;
    // run up to n batched events; *us = microseconds per batched event (timed)
    auto rounds = [&](int64_t n, bool time_it, double* us) -> int {
        n = std::min(n, budget);
        int64_t done = 0;
        if (time_it && cudaEventRecord(a, B->stream) != cudaSuccess) return PSC_E_CUDA;
        for (; done < n; ++done) {
            int r;
            if (batch_event(B, INFINITY, true, &r) == 0) break;
            if (r) return r;
        }
        budget -= done;
        out->rounds += done;
        if (!time_it) return PSC_OK;
        if (cudaEventRecord(b, B->stream) != cudaSuccess || cudaEventSynchronize(b) != cudaSuccess)
            return PSC_E_CUDA;
        float ms = 0.f;
        if (cudaEventElapsedTime(&ms, a, b) != cudaSuccess) return PSC_E_CUDA;
        out->trials++;
        *us = done > 0 ? 1e3 * (double)ms / (double)done : INFINITY;
        return PSC_OK;
    };
    int best_t = B->threads, best_m = B->item_blocks_max;
    double best_us = INFINITY;
    rc = rounds(1, false, nullptr);
    if (!rc) rc = rounds(W, true, &best_us);
    out->us_per_round_before = best_us;
    const int threads[] = {128, 256};
    const int per_member[] = {8, 16, 32, 64, 128, 256};
    for (int th : threads) {
        for (int m : per_member) {
            if (rc || budget <= 0) break;
            if (th == best_t && m == best_m) continue;
            B->threads = th;
            B->item_blocks_max = m;
            double us;
            if (!(rc = rounds(W, true, &us)) && us < best_us) { best_us = us; best_t = th; best_m = m; }
        }
    }
    B->threads = best_t;
    B->item_blocks_max = best_m;
    // the members' re-sort period: none, or every 64 or 256 of a member's
    // events; each trial spans at least one period of the fastest member
    int best_r = B->resort_period;
    for (const int period : {-1, 64, 256}) {
        if (rc || budget <= 0) break;
        if (period == best_r) continue;
        B->resort_period = period;
        double us;
        const int64_t span = period > 0 ? std::max<int64_t>(W, period) : W;
        if (!(rc = rounds(span, true, &us)) && us < best_us) { best_us = us; best_r = period; }
    }
    B->resort_period = best_r;
    // the members' stretches against the best of these launches
    B->use_stretches = true;
    if (!rc && budget >= W) {
        auto stretch = [&](bool time_it, double* us) -> int {
            if (time_it && cudaEventRecord(a, B->stream) != cudaSuccess) return PSC_E_CUDA;
            int r;
            const bool any = batch_advance(B, INFINITY, W, &r);
            if (r || !any) return r;
            budget -= W;
            out->rounds += W;
            if (!time_it) return PSC_OK;
            if (cudaEventRecord(b, B->stream) != cudaSuccess || cudaEventSynchronize(b) != cudaSuccess)
                return PSC_E_CUDA;
            float ms = 0.f;
            if (cudaEventElapsedTime(&ms, a, b) != cudaSuccess) return PSC_E_CUDA;
            out->trials++;
            *us = 1e3 * (double)ms / (double)W;
            return PSC_OK;
        };
        double us = INFINITY;
        if (budget >= 2 * W) rc = stretch(false, nullptr);
        if (!rc) rc = stretch(true, &us);
        if (!rc && us < best_us) best_us = us;
        else B->use_stretches = false;
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    out->threads = best_t;
    out->blocks_per_member = best_m;
    out->resort_period = best_r;
    out->us_per_round = best_us;
    return rc;
}

void psc_batch_destroy(psc_batch* B)
{
    if (!B) return;
    {
        DevGuard dg(B->device);
        cudaStreamSynchronize(B->stream);
        cudaFree(B->tmpl_ev);
        cudaFree(B->tmpl_rc);
        cudaFree(B->args_d);
        cudaFree(B->upload_d);
        cudaFree(B->counts_d);
        if (B->counts_h) cudaFreeHost(B->counts_h);
        if (B->counts_ev) cudaEventDestroy(B->counts_ev);
        if (B->own_stream) cudaStreamDestroy(B->stream);
    }
    delete B;
}

}  // extern "C"

// ---------------------------------------------------------------------------
// serving loop
// ---------------------------------------------------------------------------
namespace {

using Clock = std::chrono::steady_clock;

struct Request {
    int64_t ticket = 0;
    psc_request r{};
    std::vector<double> D, k;
    std::vector<int64_t> n0;
    std::vector<int32_t> nre, re, npr, pr;
    Clock::time_point submitted;
};

struct Running {
    psc_lattice* L = nullptr;
    int64_t ticket = 0;
    int64_t bytes = 0;
    double t_end = 0.0;
    int32_t n_species = 0;
    Clock::time_point submitted;
};

struct Outcome {
    int status = PSC_OK;
    std::vector<int64_t> counts;
    double seconds = 0.0;
};

// create and populate a lattice for a request; *bytes = its device footprint
int build_lattice(const Request& q, int device, cudaStream_t stream, psc_lattice** out)
{
    const psc_request& r = q.r;
    psc_lattice* L = nullptr;
    int rc = psc_lattice_create(&L, r.ni, r.nj, r.nk, r.voxel_radius_m, r.boundary_flags, device, stream);
    if (rc) return rc;
    psc_options o{};
    o.claim_table = 1;
    o.resort_period = -1;
    psc_set_options(L, &o);
    L->stretches = false;                            // the batch runs its events
    for (int s = 0; s < r.n_species && !rc; ++s) rc = psc_add_species(L, q.D[s], q.n0[s], nullptr);
    for (int x = 0; x < r.n_reactions && !rc; ++x)
        rc = psc_add_reaction(L, &q.re[2 * x], q.nre[x], &q.pr[2 * x], q.npr[x], q.k[x], nullptr);
    if (rc) {
        psc_lattice_destroy(L);
        return rc;
    }
    *out = L;
    return PSC_OK;
}

}  // namespace

struct psc_server {
    int device = 0;
    cudaStream_t stream = nullptr;
    bool own_stream = false;
    int64_t max_bytes = 0;
    int64_t used = 0;
    int64_t peak = 0;
    int32_t max_active = 0;
    psc_batch* batch = nullptr;
    int64_t next_ticket = 1;
    std::deque<Request> queue;
    std::vector<Running> running;
    std::map<int64_t, Outcome> done;
};

extern "C" {

int psc_server_create(psc_server** out, int device, void* cuda_stream, int64_t max_device_bytes, int32_t max_active)
{
    if (!out || max_device_bytes <= 0 || max_active < 1) return PSC_E_ARG;
    *out = nullptr;
    psc_server* S = new (std::nothrow) psc_server();
    if (!S) return PSC_E_NOMEM;
    S->device = device;
    S->max_bytes = max_device_bytes;
    S->max_active = std::min<int32_t>(max_active, kBatchMax);
    {
        DevGuard dg(device);
        if (cuda_stream) {
            S->stream = static_cast<cudaStream_t>(cuda_stream);
        } else {
            if (cudaStreamCreateWithFlags(&S->stream, cudaStreamNonBlocking) != cudaSuccess) {
                delete S;
                return PSC_E_CUDA;
            }
            S->own_stream = true;
        }
    }
    int rc = psc_batch_create(&S->batch, device, S->stream);
    if (rc) {
        if (S->own_stream) cudaStreamDestroy(S->stream);
        delete S;
        return rc;
    }
    *out = S;
    return PSC_OK;
}

int psc_server_submit(psc_server* S, const psc_request* r, int64_t* ticket)
{
    if (!S || !r || !ticket) return PSC_E_ARG;
    if (r->n_species < 1 || r->n_species > kMaxSpecies || r->n_reactions < 0 || r->n_reactions > kMaxReactions ||
        !r->D || !r->initial_count || !std::isfinite(r->t_end))
        return PSC_E_ARG;
    if (r->n_reactions > 0 && (!r->n_reactants || !r->reactants || !r->n_products || !r->k)) return PSC_E_ARG;
    Request q;
    q.r = *r;
    q.D.assign(r->D, r->D + r->n_species);
    q.n0.assign(r->initial_count, r->initial_count + r->n_species);
    q.nre.assign(r->n_reactions, 0);
    q.npr.assign(r->n_reactions, 0);
    q.re.assign(2 * (size_t)r->n_reactions, 0);
    q.pr.assign(2 * (size_t)r->n_reactions, 0);
    q.k.assign(r->n_reactions, 0.0);
    for (int x = 0; x < r->n_reactions; ++x) {
        q.nre[x] = r->n_reactants[x];
        q.npr[x] = r->n_products[x];
        if (q.nre[x] < 1 || q.nre[x] > 2 || q.npr[x] < 0 || q.npr[x] > 2) return PSC_E_ARG;
        for (int a = 0; a < q.nre[x]; ++a) q.re[2 * x + a] = r->reactants[2 * x + a];
        for (int a = 0; a < q.npr[x]; ++a) q.pr[2 * x + a] = r->products[2 * x + a];
        q.k[x] = r->k[x];
    }
    q.ticket = S->next_ticket++;
    q.submitted = Clock::now();
    *ticket = q.ticket;
    S->queue.push_back(std::move(q));
    return PSC_OK;
}

int psc_server_step(psc_server* S, int32_t n_events, int32_t* n_active, int32_t* n_waiting)
{
    if (!S || n_events < 0) return PSC_E_ARG;
    DevGuard dg(S->device);
    // admit in arrival order while memory and slots allow
    while (!S->queue.empty() && (int32_t)S->running.size() < S->max_active) {
        Request& q = S->queue.front();
        psc_lattice* L = nullptr;
        int rc = build_lattice(q, S->device, S->stream, &L);
        if (rc) {
            Outcome& o = S->done[q.ticket];
            o.status = rc;
            S->queue.pop_front();
            continue;
        }
        int64_t bytes = 0;
        psc_device_bytes(L, &bytes);
        if (S->used + bytes > S->max_bytes) {
            psc_lattice_destroy(L);
            if (S->running.empty()) {          // can never fit
                Outcome& o = S->done[q.ticket];
                o.status = PSC_E_NOMEM;
                S->queue.pop_front();
                continue;
            }
            break;
        }
        rc = psc_populate(L, q.r.seed);
        if (rc < 0) {
            psc_lattice_destroy(L);
            Outcome& o = S->done[q.ticket];
            o.status = rc;
            S->queue.pop_front();
            continue;
        }
        psc_device_bytes(L, &bytes);
        int64_t extra = 0;
        rc = batch_add_until(S->batch, L, q.r.t_end, S->max_bytes - S->used - bytes, &extra);
        bytes += extra;
        if (rc) {
            psc_lattice_destroy(L);
            Outcome& o = S->done[q.ticket];
            o.status = rc;
            S->queue.pop_front();
            continue;
        }
        Running run;
        run.L = L;
        run.ticket = q.ticket;
        run.bytes = bytes;
        run.t_end = q.r.t_end;
        run.n_species = q.r.n_species;
        run.submitted = q.submitted;
        S->running.push_back(run);
        S->used += bytes;
        S->peak = std::max(S->peak, S->used);
        S->queue.pop_front();
    }
    // advance every running simulation by up to n_events of its events
    for (int64_t e = 0; e < n_events; e += kSmallEvents) {
        int rc;
        if (!batch_advance(S->batch, INFINITY, n_events - e, &rc)) break;
        if (rc) return rc;
    }
    // retire the finished ones
    for (size_t x = 0; x < S->running.size();) {
        Running& run = S->running[x];
        int s;
        double t;
        const bool more = next_event(run.L, &s, &t) && t <= run.t_end && run.L->g != UINT32_MAX;
        if (more && !run.L->sticky) {
            ++x;
            continue;
        }
        Outcome& o = S->done[run.ticket];
        o.counts.assign(run.n_species, 0);
        o.status = run.L->sticky ? run.L->sticky : psc_counts(run.L, o.counts.data(), run.n_species);
        o.seconds = std::chrono::duration<double>(Clock::now() - run.submitted).count();
        psc_batch_remove(S->batch, run.L);
        psc_lattice_destroy(run.L);
        S->used -= run.bytes;
        run = S->running.back();
        S->running.pop_back();
    }
    if (n_active) *n_active = (int32_t)S->running.size();
    if (n_waiting) *n_waiting = (int32_t)S->queue.size();
    return PSC_OK;
}

int psc_server_result(psc_server* S, int64_t ticket, int64_t* counts, int32_t n, double* seconds)
{
    if (!S) return PSC_E_ARG;
    auto it = S->done.find(ticket);
    if (it == S->done.end()) return PSC_E_ORDER;
    const Outcome& o = it->second;
    if (o.status < 0) return o.status;
    if (counts) {
        if (n < (int32_t)o.counts.size()) return PSC_E_ARG;
        for (size_t s = 0; s < o.counts.size(); ++s) counts[s] = o.counts[s];
    }
    if (seconds) *seconds = o.seconds;
    return PSC_OK;
}

int psc_server_memory(const psc_server* S, int64_t* in_use, int64_t* peak)
{
    if (!S) return PSC_E_ARG;
    if (in_use) *in_use = S->used;
    if (peak) *peak = S->peak;
    return PSC_OK;
}

void psc_server_destroy(psc_server* S)
{
    if (!S) return;
    {
        DevGuard dg(S->device);
        cudaStreamSynchronize(S->stream);
        for (Running& run : S->running) psc_lattice_destroy(run.L);
        psc_batch_destroy(S->batch);
        if (S->own_stream) cudaStreamDestroy(S->stream);
    }
    delete S;
}

}  // extern "C"
