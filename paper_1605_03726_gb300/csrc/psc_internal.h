// psc_internal.h -- device-side data layout and launch interfaces of the hop
// engine.  Shared by the CUDA translation units and the host runtime; not part
// of the public ABI (include/psc.h).
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace psc {

constexpr int kMaxSpecies = 32;
constexpr int kMaxReactions = 128;
constexpr int kMaxFirstOrder = 8;          // first-order reactions per species
constexpr int kMaxCompartments = 16;
constexpr uint32_t kNoClaim = 0xFFFFFFFFu;  // claim word of an unclaimed voxel
constexpr uint16_t kBlocked = 0xFFFFu;      // occupancy code reserved for walls
constexpr uint32_t kTagEvent = 0u;          // Philox counter word 2 domain tags
constexpr uint32_t kTagPopulate = 1u;

// Error bits raised on the device, read back by psc_synchronize.
constexpr int32_t kErrListOverflow = 1;
constexpr int32_t kErrBirthOverflow = 2;
constexpr int32_t kErrClaimTableFull = 4;
constexpr int32_t kErrBarrierTimeout = 8;
constexpr int32_t kErrBadInput = 16;       // caller-supplied molecules: voxel out of range,
                                            // two on one voxel, or the reserved id

// grid-wide barrier state of the persistent hop kernel: one arrival word whose
// top bit flips each time every block has arrived
struct BarrierState {
    unsigned int arrive;
    unsigned int pad;
};

// n / d for n, d < 2^31 by one high multiply (round-up reciprocal).
struct FastDiv {
    uint32_t d;
    uint32_t m;
    int32_t s;  // -1 marks d == 1
};
FastDiv make_fastdiv(uint32_t d);

struct Geometry {
    int32_t ni, nj, nk;
    uint32_t bflags;      // bit a set: axis a periodic
    uint32_t ninj;
    FastDiv div_ni;
    FastDiv div_ninj;
    uint32_t nbi, nbj;    // vacancy-mirror bricks (4 x 4 x 2 voxels per word) along i, j
    // compact Morton code of a voxel = mort[i] | mort[ni + j] | mort[ni + nj + k]
    // (bits of the three axes interleaved, axes with fewer bits dropping out
    // at the top), mort_bits wide
    const uint32_t* mort;
    uint32_t mort_bits;
    uint32_t slot_map;    // claim-table home slot: 0 hashed voxel index, 1 Morton,
                          // 2 Morton with the low 10 bits permuted
};
// host: spread tables of the compact Morton code (ni + nj + nk words)
void build_morton_tables(int32_t ni, int32_t nj, int32_t nk, uint32_t* out, uint32_t* bits);
// words of the vacancy mirror for an ni x nj x nk lattice
inline uint64_t mirror_words(int32_t ni, int32_t nj, int32_t nk)
{
    return (uint64_t)((ni + 3) / 4) * (uint64_t)((nj + 3) / 4) * (uint64_t)((nk + 1) / 2);
}

// Structure-of-arrays list of the molecules of one species.  img packs three
// 16-bit periodic wrap counters (i at bits 0-15, j at 16-31, k at 32-47).
struct SpeciesList {
    int32_t* vox;
    uint32_t* ids;
    uint64_t* img;
    int32_t cap;
};

struct ReactionDev {
    uint64_t T;           // acceptance threshold (second order), floor(p 2^32)
    int32_t np;           // products
    int32_t p0, p1;       // product species
};

// Model tables, uploaded once at populate and read through a pointer.
struct ModelDev {
    int8_t pair[kMaxSpecies][kMaxSpecies];   // second-order reaction or -1
    ReactionDev rx[kMaxReactions];
    uint64_t T_fire[kMaxSpecies];            // first-order firing threshold
    int32_t n_fo[kMaxSpecies];
    int32_t fo_rx[kMaxSpecies][kMaxFirstOrder];
    uint64_t fo_cum[kMaxSpecies][kMaxFirstOrder];
    SpeciesList lists[kMaxSpecies];
    // Compartments (Sec. 2): one vacancy mirror per compartment, in which the
    // voxels of every other compartment are set for good, so a species tests
    // vacancy-and-own-compartment with one bit of its own mirror
    uint32_t* mirror[kMaxSpecies];           // the mirror of the species' compartment
    uint8_t comp[kMaxSpecies];               // the species' compartment
};

enum StatIndex {
    kStatAttempts = 0, kStatHops, kStatCollisions, kStatAccepted, kStatReactions2,
    kStatFires, kStatReactions1, kStatBirths, kNumStats
};

// Small device-resident scalars of one lattice.
struct Scalars {
    int32_t counts[kMaxSpecies];     // molecules per species list
    int32_t tmp_count[kMaxSpecies];  // entries of each list that left in the current event
    uint32_t next_id;                // next fresh molecule id
    int32_t births;                  // births queued in the current event
    int32_t err;                     // kErr* bits
    uint32_t g_base;                 // index of the first event of a replayed graph
    uint32_t touched[2];             // by event parity, in k_small_run: the event had births
    int32_t hole_n[kMaxSpecies], surv_n[kMaxSpecies];   // while k_small_run closes its lists up
    unsigned long long stats[kNumStats];
};

struct Birth {
    uint32_t parent;
    int32_t t;
    int32_t species;
    int32_t pad;
    uint64_t img;
};

// Where the claims of one event go.  Direct: one 32-bit word per voxel (small
// lattices), reset by the winner.  Hash: open addressing over 64-bit slots
// holding (voxel << 32 | lowest id); two tables alternate between events and
// the commit kernel of one event empties the table of the previous one.
struct ClaimTable {
    uint32_t* direct;
    uint64_t* hash;
    uint32_t hash_bits;        // log2 of the slots in use this event
    uint64_t* clear;           // table of the previous event (hash mode)
    uint32_t clear_n;          // its slots to reset
};
constexpr uint64_t kEmptySlot = ~0ull;

// Everything one event kernel needs, passed by value.
struct EventArgs {
    Geometry geo;
    uint16_t* occ;             // species codes (exact for species with reactions)
    uint32_t* bits;            // vacancy mirror: bit v set = voxel v occupied
    ClaimTable ct;
    SpeciesList list;          // list of the due species
    const int32_t* count;      // its length (device)
    const ModelDev* model;
    Scalars* sc;
    Birth* births;
    int32_t births_cap;
    uint32_t key0, key1;       // Philox key = seed
    uint32_t g;                // global event index (with g_base: its offset from *g_base)
    const uint32_t* g_base;    // null, or the device word holding the index a replayed graph starts at
    uint32_t* dirty[2];        // by event parity: a bit per mirror word whose voxels changed species
    uint32_t dirty_words;      // words of one dirty map
    uint8_t* dec;              // null, or per list entry the claim's outcome for the commit (kDec*)
    int32_t* leave;            // species with reactions: the commit notes here the slots of the due
                               // species' entries that react away (count in Scalars::tmp_count[s])
    uint32_t* g_bump;          // null, or the word the event's last launch sets to its index + 1
    int32_t* holes;            // scratch of the own-list fill of a one-block event (the scratch
    int32_t* surv;             // list's ids and img; img's decision bytes are read by then)
    int32_t s;                 // due species
    int32_t live;              // 1: the species writes its code into occ
    int32_t collect_stats;
};

// Outcome of a molecule's claim phase, kept for its commit phase: the
// direction 0-11 of the voxel it claimed, no claim, or a first-order firing
// (the commit redraws those)
constexpr uint8_t kDecNone = 12;
constexpr uint8_t kDecFire = 13;

// A stretch of consecutive events of one species without reactions, run by
// one persistent cooperative launch.
struct RunArgs {
    EventArgs ev;              // g = index of the first event
    uint64_t* tables[2];       // claim tables, alternating by event parity
    int32_t n_events;
    BarrierState* barrier;
    uint64_t barrier_timeout_ns;  // a block gives up waiting at a barrier after this long
    uint32_t barrier_phantom;     // arrivals awaited from blocks that do not exist (0; tests only)
};

// Owner-computes decomposition of a stretch (tile kernel): the mirror's brick
// grid (nbi x nbj x nbk words) is cut into pi x pj x pk boxes of whole bricks,
// one per block; region a along an axis of nb bricks spans bricks
// [a nb / p, (a + 1) nb / p).
struct TilePlan {
    int32_t pi, pj, pk;
    int32_t nbi, nbj, nbk;
    int32_t ei, ej, ek;        // largest region extent in bricks
    int32_t regions;
    int32_t box_words;         // (ei + 2)(ej + 2)(ek + 2): region plus one brick of halo
    int32_t cap;               // molecule slots per region (bucket, inbox)
    int32_t fcc;               // FCC lattice: stencil and neighbourhood masks by k mod 3
    int32_t lean;              // 1: the stretch runs k_tile_lean (HCP, whole bricks, boxes of
                               // at least two bricks, two or more boxes along periodic axes)
};

// A stretch of a species without reactions under the tile kernel.  Each
// region's molecules live in its bucket; a molecule that hops into another
// region is appended to that region's inbox and joins its bucket at the next
// event.  Wrap counters are kept by id (the species' ids are id_lo .. id_lo +
// n - 1: it never reacts, so they are the ones populate gave it).
struct TileArgs {
    EventArgs ev;              // g = index of the first event
    TilePlan plan;
    uint32_t* claim;           // per-voxel claim words (kNoClaim when free), for contested targets
    uint32_t* claimed;         // [regions] events whose claim phase the region has finished
    uint32_t* done;            // [regions] events whose commit phase the region has finished
    int32_t nbr_sync;          // 1: phases wait for the neighbouring boxes only; 0: grid barriers
    int32_t* b_vox[2];         // [regions][cap] voxel of each molecule; event e
    uint32_t* b_ids[2];        // reads buffer e & 1 and keeps its survivors in the other
    uint32_t* b_state;         // claim-phase decision of each bucket slot
    int32_t* b_cnt;            // [regions]
    int32_t* in_vox;           // [regions][cap] arrivals of the last event
    uint32_t* in_ids;
    int32_t* in_cnt;           // [regions]
    uint64_t* img_id;          // wrap counters by id - id_lo
    uint2* halo_tab;           // lean kernel: [regions][halo_cap] (box word, global word or ~0 behind a wall)
    int32_t halo_cap;
    uint32_t id_lo;
    int32_t n_events;
    BarrierState* barrier;
    uint64_t barrier_timeout_ns;
    uint32_t barrier_phantom;
};

// A stretch of events of one species under the sub-volume rule (the paper's
// sub-volume scheme on the lattice; species without reactions).
struct SubvolArgs {
    EventArgs ev;              // g = index of the first event
    uint32_t* word;            // per 2x2x2 sub-volume: lowest waiting id of the colour's turn (kNoClaim: free)
    uint32_t* head;            // per sub-volume: first list slot of its chain of waiting molecules (kNoClaim: none)
    uint32_t* next;            // per list slot: the next slot of its sub-volume's chain
    uint32_t* state;           // per list slot: its sub-volume at the event's start, bit 31 it leads it, bit 30 alone
    uint8_t* colour0;          // per list slot: colour of its sub-volume when the event began
    uint32_t* lead;            // per list slot: the leaders' slots, colour by colour (top bit: alone)
    uint32_t* lead_vox;        // per list slot: the voxel of an alone leader, in the same order
    uint32_t* counters;        // [2][16] by event parity: molecules and leaders per colour
    int32_t n_events;
    BarrierState* barrier;
    uint64_t barrier_timeout_ns;
    uint32_t barrier_phantom;
};

struct ReconcileArgs {
    Geometry geo;
    uint16_t* occ;
    const uint32_t* bits;
    int32_t x;                 // species whose list is reconciled
    SpeciesList list;
    SpeciesList tmp;           // scratch: the slots that leave, then the holes and the tail's survivors
                               // (vox and ids hold twice the capacity: one reaction can remove two entries)
    const ModelDev* model;
    Scalars* sc;
    const uint32_t* dirty[2];  // the commit's dirty maps, by event parity
    uint32_t g;                // event index (with g_base: its offset from *g_base)
    const uint32_t* g_base;
    uint32_t* g_bump;          // null, or the word the event's last launch sets to its index + 1
};

// A stretch of events, of any species in scheduler order, of a lattice with
// per-voxel claim words (k_small_run).
constexpr int kSmallEvents = 512;          // events of one launch
constexpr int kSmallThreads = 512;         // threads of a block
constexpr int kSmallCounts = kMaxSpecies + 2;      // list lengths, next id and error bits, per lattice of a batch
// limits of a cell's fields
constexpr int64_t kCellVoxels = 1ll << 26; // (list slots)
constexpr int64_t kCellIds = (1ll << 27) - (1ll << 23);    // next id when a stretch starts; a stretch makes at
                                                           // most 512 x 8192 (births_cap) of them
// The longest list of a mobile species of a lattice that runs in stretches:
// with reactions as far as was measured (3.2M molecules 126 us per event, 180 in
// per-event launches), else where the molecule-list and tile kernels take over
// (128^3: 63,000 walkers 6.0 us per event against 10.8, 210,000 14.4 against 13.0).
constexpr int64_t kSmallList = 1 << 22;
constexpr int64_t kSmallWalk = 131072;
// Walkers among species with reactions: the tile and molecule-list kernels take
// fewer accesses for a walker, but start anew after every event of another species.
// So long lists of walkers leave these stretches to them, with all events of the
// lattice, where a run (walkers' events for one of all other species) is longer
// than kSmallRun / molecules; than kSmallRunLarge / molecules where the cells do not
// fit in the L2 cache; than kSmallRunDense where they do and the list is too long
// for the molecule-list kernel; and in no case for runs of kSmallRunLeast.  us per
// event, those kernels / stretches, with a pair of 2000 molecules each that react, at
// runs of 0.5, 4 and 50 events: 270,000 walkers on 256^3 35.0 / 9.4, 19.8 / 13.8,
// 14.1 / 15.6; 1.0M on 256^3 45.0 / 19.0, 37.9 / 36.6, 34.9 / 43.4; 2.5M on 256^3
// 81.7 / 36.8, 87.9 / 78.8, 90.4 / 94.9; 500,000 on 128^3 19.9 / 12.1, 19.8 / 20.4,
// 19.8 / 23.6; 1.0M on 400^3 48.3 / 30.1, 34.7 / 62.7, 29.6 / 75.4; 2.5M on 400^3
// 81.0 / 70.8, 77.5 / 160, 76.9 / 195.
// 131,072 walkers are faster in stretches at any run (400^3 at 50 events 12.4 / 9.8).
constexpr int64_t kSmallRunList = 1 << 18;
constexpr double kSmallRun = 1.5e6, kSmallRunLarge = 1e6, kSmallRunDense = 3.0, kSmallRunLeast = 0.6;
// The longest list that runs in one cluster of 16 blocks: A + B -> C of 2000
// molecules each takes 4.2 us per event there and 6.3 in a grid, of 12,000 6.4 and
// 6.7, of 24,000 10.3 and 6.8.
constexpr int64_t kSmallCluster = 16384;
// There one block closes up a list, 1.2 us for 1000 entries; a grid does it together.
// An event of few molecules is 2 us faster in a cluster: a stretch of few events
// with lists to close up longer than kSmallClosed, and kSmallClosedEvent for each event
// (less for longer due lists, which gain less), runs in a grid.  us per call of one event, in a
// cluster / in a grid (launches per event phase): 2000 A meeting 2000 B on 64^3 25 / -
// (33), 15,000 and 15,000 49 / 29 (34), 2000 and 200,000 immobile ones on 128^3 294 / 29
// (33), 2000 and 4 million on 256^3 8470 / 37 (46).
constexpr double kSmallClosed = 2048.0, kSmallClosedEvent = 2500.0;
struct SmallArgs {
    const EventArgs* ev;       // [nsp] templates on the device (event_args with g unset)
    const ModelDev* model;
    Scalars* sc;
    uint32_t* cell;            // a word per voxel (psc_small.cuh)
    int32_t* holes;            // [scratch_n] slots of tombstones and of the entries that take them
    int32_t* surv;
    int32_t scratch_n;
    BarrierState* barrier;
    uint64_t barrier_timeout_ns;
    uint32_t barrier_phantom;
    uint32_t g;                // index of the first event
    int32_t n_events;
    int32_t nsp;
    int32_t collect_stats;
    uint32_t general;          // bit s: species s has reactions
    uint32_t fo2;              // bit s: a first-order reaction of s has two products
    uint32_t products[kMaxSpecies];        // bit y: an event of s may append to list y
    uint8_t seq[kSmallEvents]; // species of each event (batched launches: see SmallStretch)
};

// A lattice's stretch in a batched launch: what changes from one to the next (the
// rest of its SmallArgs stays on the device)
struct SmallStretch {
    int32_t slot;              // of its SmallArgs
    int32_t block0, blocks;    // its group of the launch's blocks
    uint32_t g;
    int32_t n_events;
    uint32_t seq;              // where its events' species begin
};

// A stretch of events of a lattice without reactions (k_walk_run): every
// mobile species' molecules in shared memory, claim words that tell vacancy.
constexpr int kWalkEvents = 512;           // events of one launch
constexpr int kWalkThreads = 1024;         // threads of a block: one per SM, a cooperative grid
constexpr int kWalkClusterThreads = 512;   // or one cluster
constexpr int64_t kWalkCluster = 16384;    // molecules a cluster takes
// Shorter lists run as fast in any order: 168,000 walkers on 256^3 8.4 us per
// event either way, 629,000 on 128^3 13.7 sorted every 64 events, 15.1 unsorted.
constexpr int64_t kWalkSorted = 200000;
constexpr int kWalkClusterSmem = 36 * 1024;        // shared memory of its blocks, at most
// Largest lattice that runs in them, its claim words in the L2 cache (112 MB);
// and with lists shorter than kOpenList, where the claims are too few for that
// to matter: 100,000 walkers on 320^3 9.3 -> 7.0 us per event (k_small_run),
// 200,000 on 400^3 17.2 -> 10.2 (tables, a launch per phase), 125,000 on 500^3
// 15.2 -> 10.9; but 640,000 on 400^3 22.1 -> 32, 400,000 on 500^3 19.3 -> 24.9
// (the lean tile kernel).
constexpr int64_t kWalkVoxels = 28000000;
constexpr int64_t kWalkVoxelsFew = 1 << 27;
constexpr int64_t kWalkSmem = 225 * 1024;  // shared memory of its blocks
struct WalkArgs {
    Geometry geo;
    FastDiv div_nbi, div_nbij; // by the mirror's words along i, and along i and j
    uint32_t* word;            // per voxel, in the mirror's order (word << 5 | bit): all ones vacant, else the
                               // last claim that won it (0: occupied since the words were made)
    uint32_t epoch;            // of the first event; claims are epoch << id_bits | id - id_lo
    int32_t id_bits;
    uint32_t id_lo[kMaxSpecies];
    uint32_t* bits;            // vacancy mirror
    Scalars* sc;
    BarrierState* barrier;
    uint64_t barrier_timeout_ns;
    uint32_t barrier_phantom;
    uint32_t key0, key1;
    uint32_t g;                // index of the first event
    int32_t n_events;
    int32_t collect_stats;
    int32_t n_species;         // species with events in the stretch
    int32_t slots;             // molecules a thread holds at most, over all species
    int32_t n[kMaxSpecies];    // per species: molecules, first slot, index, list
    int32_t slot0[kMaxSpecies];
    uint8_t species[kMaxSpecies];
    SpeciesList list[kMaxSpecies];
    uint8_t seq[kWalkEvents];  // species of each event (place in the arrays above)
};

// ---- launchers (psc_kernels.cu) ----
void upload_stencil(cudaStream_t st);
void launch_claim(const EventArgs& a, bool general, int blocks, int threads, cudaStream_t st);
void launch_commit(const EventArgs& a, bool general, int blocks, int threads, cudaStream_t st);
// claim and commit of a species without reactions (n molecules) that skip the
// claim where no other molecule is next to the target
void launch_open_claim(const EventArgs& a, int64_t n, int sm_count, cudaStream_t st);
void launch_open_commit(const EventArgs& a, int64_t n, int sm_count, cudaStream_t st);
constexpr int64_t kOpenList = 1 << 18;      // shortest list they take
// They take lattices of more than kWalkVoxels voxels up to this share of occupied ones.
// us per event, plain claims / these, both in claim words: 320^3 at 5 / 10 / 20 / 30 / 50 %
// 69.8 / 54.1, 130 / 110, 221 / 207, 286 / 284, 346 / 416; 512^3 at 5 / 30 / 50 % 338 / 219,
// 1213 / 1117, 1457 / 1691.  Where the words fit in the L2 cache a claim costs less than
// the test: 256^3 at 2 / 5 / 10 / 30 % 16.4 / 18.7, 29.2 / 32.6, 50.6 / 57.5, 134 / 151,
// 160^3 at 10 / 30 % 17.4 / 22.3, 37.3 / 47.2.
constexpr double kOpenOccupied = 0.3;
// Where the lean tile kernel can run, it does up to here: 2.5M walkers on 512^3
// 70.7 us per event against 73.0, 2.7M 79.9 against 76.8, 3.4M 118 against 101.
// (The general tile kernel never: 1.4M on a ragged lattice 102 against 45.)
constexpr int64_t kOpenOverLean = 2600000;
// claim, commit and the own-list fill of one event of a species with
// reactions in a single block (lists of a few hundred molecules)
constexpr int kEventOneThreads = 512;
void launch_event_one(const EventArgs& a, cudaStream_t st);
void launch_walk_words(uint32_t* word, const uint32_t* bits, uint64_t words, int blocks, cudaStream_t st);
// blocks of the largest cluster, shared memory of a block on the current
// device (0: none); sets the kernels' attributes there
void walk_limits(int* cluster, int* smem);
cudaError_t launch_walk(const WalkArgs& A, int blocks, bool cluster, cudaStream_t st);
void launch_fill_u64(uint64_t* p, uint64_t value, size_t n, int blocks, cudaStream_t st);
// Molecules per thread the persistent kernel holds in registers (0 = the
// stretch does not fit); threads = its launch width.
int run_capacity(int64_t n, int* threads_per_block, int* blocks, int sm_count, int min_per_thread);
cudaError_t launch_run(const RunArgs& r, int blocks, int threads, int per_thread, cudaStream_t st);
cudaError_t launch_subvol(const SubvolArgs& A, int blocks, int threads, cudaStream_t st);
int subvol_max_blocks(int sm_count);        // co-resident 256-thread blocks of the sub-volume kernel
// tile kernel: dynamic shared memory a block may use, its need for a plan,
// the three launches of a stretch (list -> buckets, the persistent events,
// buckets -> list)
int tile_smem_limit(int device);
constexpr int kTileOutbox = 1024;           // departures a block stages per event
constexpr int kTileQueue = 1024;            // molecules a block defers per commit phase (contested, leaving)
// largest max / mean box load at which the automatic choice keeps the tile kernel
constexpr double kTileMaxImbalance = 1.4;
inline int tile_smem_bytes(const TilePlan& P)
{
    return ((P.box_words + 3) & ~3) * 4 + (P.fcc ? 96 : 32) * 8 * 4 + kTileOutbox * 12 + kTileQueue * 4 +
           ((P.nbi + P.nbj + P.nbk + 15) & ~15);
}
// the lean tile kernel: shared-memory tables per (place in the brick word,
// direction), per-axis halo tables, plus the areas of the general kernel
constexpr int kLeanEntries = 32 * 12;
constexpr int kLeanClaimBits = 10;          // block-local claim table: 2^10 slots of 8 bytes
constexpr int kLeanOutbox = 512;            // departures staged per event (more go straight to the inboxes)
// halo words of the largest box of a plan (the lean kernel's per-box halo table)
inline int64_t lean_halo_cap(const TilePlan& P)
{
    const int64_t BI = P.ei + 2, BJ = P.ej + 2, BK = P.ek + 2;
    return 2 * BI * BJ + 2 * (BK - 2) * BI + 2 * (BK - 2) * (BJ - 2);
}
inline int lean_smem_bytes(const TilePlan& P)
{
    const int halo_tables = ((P.ei + 2) + (P.ej + 2) + (P.ek + 2) + 3) & ~3;
    return ((P.box_words + 3) & ~3) * 4 + (8 << kLeanClaimBits) + kLeanEntries * 8 * 4 + kLeanEntries * 2 * 4 +
           kLeanOutbox * 12 + halo_tables * 4 + ((P.box_words + 31) >> 5) * 4 +
           ((P.nbi + P.nbj + P.nbk + 15) & ~15);
}
constexpr int kTileThreads = 512;
constexpr int kTileBlocksPerSM = 2;
void launch_tile_count(const TileArgs& A, int32_t* counts, int blocks, cudaStream_t st);
void launch_tile_scatter(const TileArgs& A, int blocks, cudaStream_t st);
cudaError_t launch_tile_run(const TileArgs& A, cudaStream_t st);
void launch_tile_gather(const TileArgs& A, cudaStream_t st);
// mirror c of n: bit v set where labels[v] != c (walls), the rest clear
void launch_mirror_walls(uint32_t* bits0, uint64_t words, int n, const uint8_t* labels, const Geometry& geo,
                         int blocks, cudaStream_t st);
// placement by selection (psc_populate): per compartment, a histogram of the
// top kPlaceBits bits of the voxels' placement keys, then the voxels whose
// key bin is at most that compartment's limit (-1: none), in no order
constexpr int kPlaceBits = 10;
struct PlaceLimits {
    int32_t bin[kMaxCompartments];
};
void launch_place_hist(uint32_t V, uint32_t key0, uint32_t key1, const uint8_t* labels, int nc, uint32_t* hist,
                       int blocks, cudaStream_t st);
void launch_place_pick(uint32_t V, uint32_t key0, uint32_t key1, const uint8_t* labels, const PlaceLimits& lim,
                       uint32_t* out_vox, uint32_t* out_key, int32_t* count, int32_t cap, int32_t* err, int blocks,
                       cudaStream_t st);
// keys[r] = labels[vals[r]]: the compartment of each sorted voxel
void launch_label_keys(const uint32_t* vals, const uint8_t* labels, uint32_t* keys, int64_t n, int blocks,
                       cudaStream_t st);
// codes where a voxel is occupied (its bit set in all n_mirrors mirrors of
// `words` words each, starting at bits0), zero elsewhere
void launch_materialize(uint16_t* out, const uint16_t* occ, const uint32_t* bits0, uint64_t words,
                        int n_mirrors, const Geometry& geo, int64_t V, int blocks, cudaStream_t st);
void launch_scatter_codes(uint16_t* out, const SpeciesList& list, const int32_t* count, uint16_t code,
                          int blocks, cudaStream_t st);
// Partner list r.x checked against the grid; its leavers' slots go after
// those of the lists in `before` (a bit per species).
void launch_reconcile(const ReconcileArgs& r, uint32_t before, int blocks, int threads, cudaStream_t st);
// The event's lists filled from their tails, one block each, side by side.
constexpr int kListFillMax = 8;
struct ListFill {
    ReconcileArgs r;                       // the event's arguments; x and list per block
    int32_t n;
    int32_t x[kListFillMax];
    SpeciesList list[kListFillMax];
    uint32_t before[kListFillMax];         // lists whose scratch ranges come first
};
void launch_fill(const ListFill& f, cudaStream_t st);
void launch_births(const EventArgs& a, cudaStream_t st);
// Most blocks of a stretch on the current device: as one cluster, as a
// cooperative grid (0: not at all).  Sets the kernels' attributes there.
void small_limits(int sm_count, int* cluster, int* grid);
// cells from mirrors and lists; mirrors and codes from cells
void launch_cells_build(uint32_t* cell, const uint32_t* bits0, uint64_t words, int n_mirrors, const ModelDev* model,
                        const int32_t* counts, int nsp, const Geometry& geo, int blocks, cudaStream_t st);
void launch_cells_grid(const uint32_t* cell, uint32_t* bits0, uint64_t words, int n_mirrors, uint16_t* occ,
                       const Geometry& geo, int blocks, cudaStream_t st);
// stretches of many lattices in one launch of `blocks` blocks: per block the
// stretch it belongs to, species of all their events; stretch r leaves list
// lengths in counts + r * kSmallCounts (all on the device)
int small_batch_blocks(int sm_count, int threads, bool births);    // most blocks on the current device (0: not at all)
cudaError_t launch_small_batch(const SmallArgs* args, const SmallStretch* stretch, const int32_t* group,
                               const uint8_t* seq, int32_t* counts, int blocks, int threads, bool births,
                               cudaStream_t st);
cudaError_t launch_small(const SmallArgs& A, int blocks, int threads, bool cluster, cudaStream_t st);
void launch_fill_u32(uint32_t* p, uint32_t value, size_t n, int blocks, cudaStream_t st);
// molecule r (ids in species order, species s owning [offsets[s],
// offsets[s+1])) takes sorted_vox[starts[s] + r - offsets[s]]; its bit goes
// to the mirror of its species' compartment
void launch_populate_scatter(const uint32_t* sorted_vox, int64_t n_total, const int64_t* offsets,
                             const int64_t* starts, int n_species, uint16_t* occ, const Geometry& geo,
                             const ModelDev* model, int blocks, cudaStream_t st);
// The Morton re-sort of a list's first min(*count, limit) entries (the rest,
// if any, keep their places: list order never changes results): by the whole
// code (keys and values for the radix sort, then a permutation), or by cells, the
// top `cell_bits` bits of the Morton code: the entries per cell are counted
// (cells zeroed before), and after an exclusive scan of the counts every entry
// takes the next place of its cell in dst.
constexpr int32_t kCellSortMax = 1 << 22;  // longer lists sort by the whole code: with cells, 10.7M walkers on 1024^3
                                           // took 920 us per event against 843
void launch_morton_keys(const SpeciesList& list, const int32_t* count, int32_t limit, const Geometry& geo,
                        uint32_t* keys, uint32_t* vals, int blocks, cudaStream_t st);
uint32_t morton_sort_bits(const Geometry& geo);
void launch_permute(const SpeciesList& src, const SpeciesList& dst, const uint32_t* perm,
                    const int32_t* count, int32_t limit, int blocks, cudaStream_t st);
void launch_cell_count(const SpeciesList& list, const int32_t* count, int32_t limit, const Geometry& geo,
                       uint32_t cell_bits, uint32_t* cells, int blocks, cudaStream_t st);
void launch_cell_scatter(const SpeciesList& src, const SpeciesList& dst, const int32_t* count, int32_t limit,
                         const Geometry& geo, uint32_t cell_bits, uint32_t* cells, int blocks, cudaStream_t st);
void launch_copy_list(const SpeciesList& src, const SpeciesList& dst, const int32_t* count, int32_t limit,
                      int blocks, cudaStream_t st);
// set the vacancy-mirror bit of every molecule of a list (mirror cleared before)
void launch_mirror_from_list(uint32_t* bits, const Geometry& geo, const SpeciesList& list, const int32_t* count,
                             int blocks, cudaStream_t st);
// the same for a list the library did not build: entries whose voxel is
// outside [0, V), that land on a voxel already set, or whose id is kNoClaim
// are skipped and raise kErrBadInput in *err
void launch_mirror_from_list_checked(uint32_t* bits, const Geometry& geo, const SpeciesList& list,
                                     const int32_t* count, int64_t V, int32_t* err, int blocks, cudaStream_t st);

// ---- slabs along k with ghost layers (psc_slab.cuh, psc_slab.cpp) ----
struct SlabEntry {                 // a molecule handed to a neighbouring slab
    int32_t i, j, k;               // global coordinates of the voxel it entered
    uint32_t id;
    uint64_t img;                  // packed wrap counters
};

struct SlabArgs {
    int32_t ni, nj, nk, m, k0;     // global extents, owned layers, first owned layer
    uint32_t bflags;
    uint32_t lw;                   // words per layer of the bit array (layers start on words)
    uint32_t* bits;                // (m + 2) * lw words: bit i + ni j of layer L, set = occupied or wall
    uint32_t* claim;               // (m + 2) * ni * nj words, kNoClaim when free
    int32_t* vox[2];               // molecule lists by buffer: local voxel i + ni (j + nj L)
    uint32_t* ids[2];
    uint64_t* img[2];
    int32_t* count;                // [2] molecules per buffer
    int32_t cap;
    int32_t cur;                   // buffer holding the molecules at the start of the event
    uint8_t* dec;                  // claim-phase decision per molecule
    uint8_t* send_commit[2];       // [0] to the lower neighbour, [1] to the upper one
    const uint8_t* recv_commit[2];
    const uint32_t* recv_claim[2];
    int32_t tcap;                  // entries a commit message holds
    int32_t has[2];                // a neighbour on that side (else a wall)
    int32_t* err;
    uint32_t key0, key1, g, s;     // Philox key, event index, species
};

void launch_slab_claim(const SlabArgs& A, int blocks, cudaStream_t st);
void launch_slab_commit(const SlabArgs& A, int blocks, cudaStream_t st);
void launch_slab_apply(const SlabArgs& A, int blocks, cudaStream_t st);

// ---- batched launches: many lattices (replicas) per launch ----
// Item x covers blocks [block0, next block0) of the launch and runs the event
// (or list) `sel` of replica `rep` with event index g.  Argument templates of
// every (replica, species) live on the device: tmpl[rep * kMaxSpecies + sel].
constexpr int kBatchMax = 512;
struct BatchItem {
    int32_t rep;
    int32_t sel;
    uint32_t g;
    int32_t block0;
    uint32_t mask;             // list passes: lists whose scratch ranges come before list sel's
};
struct BatchLaunch {
    int32_t n;
    int32_t total_blocks;
    BatchItem item[kBatchMax];
};
void launch_claim_batch(const EventArgs* tmpl, const BatchLaunch& bl, int threads, cudaStream_t st);
void launch_commit_batch(const EventArgs* tmpl, const BatchLaunch& bl, int threads, cudaStream_t st);
void launch_reconcile_batch(const ReconcileArgs* tmpl, const BatchLaunch& bl, int threads, cudaStream_t st);
void launch_fill_batch(const ReconcileArgs* tmpl, const BatchLaunch& bl, cudaStream_t st);
void launch_births_batch(const EventArgs* tmpl, const BatchLaunch& bl, cudaStream_t st);

// ---- radix sort (psc_sort.cu) ----
// Stable LSD radix sort of (key, value) pairs by the low `bits` bits of key.
// n is n_host, or the count in device memory (n_dev) capped at n_host;
// max_n (at least n_host) sizes the tiles and the scratch.
struct SortScratch {
    uint32_t* keys_alt = nullptr;
    uint32_t* vals_alt = nullptr;
    uint32_t* hist = nullptr;       // 256 * blocks
    uint32_t* block_sums = nullptr; // scan partials
    int64_t max_n = 0;
    int64_t hist_len = 0;
    int64_t sums_len = 0;
};
size_t sort_scratch_bytes(int64_t max_n);
void sort_scratch_bind(SortScratch& s, void* base, int64_t max_n);
// exclusive scan of data[len] in place; sums: a word per 4096 of them
void exclusive_scan(uint32_t* data, int64_t len, uint32_t* sums, cudaStream_t st, int64_t* launches);
// values of equal keys, side by side after a sort, into ascending order
void launch_sort_ties(const uint32_t* keys, uint32_t* vals, int64_t n, int blocks, cudaStream_t st);
// After the call the sorted data is in (keys, vals) again.
int radix_sort_pairs(uint32_t* keys, uint32_t* vals, const int32_t* n_dev, int64_t n_host,
                     int64_t max_n, int bits, SortScratch& scratch, cudaStream_t st,
                     int64_t* launches);

}  // namespace psc
