// psc_small.cuh -- a stretch of events of a lattice, whatever their species,
// in one launch.  Part of psc_kernels.cu's translation unit.
//
// What bounds it: an event of a short list is a chain of dependent L2
// accesses, not work.  A load that another SM wrote takes about 700 cycles, a
// fence with claims or moves in flight 1300, a cluster's hardware barrier 270
// and a grid barrier 1100 more than that fence; a launch per phase (claim,
// commit, list passes) or a grid barrier over every SM costs several times the
// chain.  So the blocks of one launch run the events of a stretch one after
// the other: claim phase, barrier, commit phase, barrier.  What keeps an event
// at two phases:
//   - a thread carries its molecules from the claim to the commit phase in
//     registers, and the counts, the list entries and what may be left to do
//     from the last event are loaded together;
//   - one word per voxel, its cell, tells vacancy and compartment, takes the
//     claims of a vacant voxel, and holds species and list slot of the molecule
//     on an occupied one.  A hop reads its target's cell, claims in it, reads it
//     back, and writes it and the one it leaves (with mirror, codes, claim words
//     and slots apart there were about ten accesses).  A reacting molecule finds
//     its partner's list entry there, so the commit itself takes both entries off
//     their lists and appends the products: no list is checked against the grid.
//     Mirror and codes are brought up to date when another kernel or a read-out
//     wants them;
//   - an entry that leaves stays behind as a tombstone (voxel -1); the lists
//     are closed up at the end of the stretch, or when one could run out of
//     room.
// Births need a pass of their own (ids in parent order) in events that have
// any: a rank for each among the parents, by all blocks (small_births).
//
// One block of 512 threads per SM: the events need about 110 registers (two
// blocks per SM spilled: crowded 256^3 30.1 us per event against 25.3), and two
// molecules in flight per thread (three 27.2, four 32.1).
//
// Measured (us per event; before: claim, commit, list check and fill launches
// replayed from CUDA graphs, or the molecule-list kernel for walkers): A + B -> C
// of 2000 + 2000 molecules on 64^3 12.5 -> 4.1, a cascade of 22 species of up to
// 16,000 molecules on 200^3 10.5 -> 3.1, 30,000 ligands and 5000 receptors in a
// cell on 128^3 19.8 -> 6.2, reversible A + B <-> C under 30 % crowding with 839,000
// A on 256^3 40.0 -> 24.6, with 1.6M on 320^3 92 -> 48, with 3.2M on 400^3
// 180 -> 126.  Tried: the next event's entries read, and their draws made, before
// the barrier that ends an event (the first 4.2 -> 4.5, the second 3.1 -> 3.7: every
// thread's extra instructions cost more than the load they hide); molecules kept in
// shared memory between the phases (crowded 256^3 26.1).  The order of a list makes
// little difference: two species of 400,000 on 256^3 22.6 us per event as placed, 22.2
// sorted, of 1.0M on 400^3, whose cells do not fit in the L2 cache, 81.0 and 82.6, 64 members
// of 160^3 at 2 % 182 and 182; only the longest gain (3.2M on 400^3 243 and 204).  So these
// stretches have no re-sorts.

// Event arguments and model of the lattice, copied to shared memory once per
// launch: after a barrier a load of them from global memory would go to L2.
struct SmallShared {
    EventArgs ev[kMaxSpecies];
    ModelDev model;
    int32_t n[kMaxSpecies], k[kMaxSpecies];     // lengths and tombstones while the lists are closed up
    uint8_t seq[kSmallEvents];
};

__device__ __forceinline__ void small_copy(void* dst, const void* src, size_t bytes)
{
    uint32_t* d = static_cast<uint32_t*>(dst);
    const uint32_t* s = static_cast<const uint32_t*>(src);
    for (uint32_t x = threadIdx.x; x < bytes / 4; x += blockDim.x) d[x] = s[x];
}

// Barrier of a cluster's blocks.  One fence per block, made cumulative over
// the block by the block barrier: a release by every warp took 500 cycles longer.
__device__ __forceinline__ void cluster_barrier()
{
    __syncthreads();
    if (threadIdx.x == 0) __threadfence();
    __syncwarp();
    asm volatile("barrier.cluster.arrive.relaxed.aligned;\n"
                 "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// The blocks of a stretch: all of the launch, as one cluster or a cooperative
// grid, or a group of the blocks of a batched launch.
enum SmallMode { kSmallInCluster, kSmallInGrid, kSmallInGroup };
struct SmallBlocks {
    int blk, nblk;
};

template <SmallMode MODE>
__device__ __forceinline__ bool small_barrier(const SmallArgs& A, const SmallBlocks& B)
{
    if (MODE == kSmallInCluster) {
        cluster_barrier();
        return true;
    }
    if (MODE == kSmallInGroup && B.nblk == 1 && A.barrier_phantom == 0u) {
        __syncthreads();                                        // what a block wrote, the block sees
        return true;
    }
    return block_barrier(A.barrier, &A.sc->err, A.barrier_timeout_ns, A.barrier_phantom, B.blk, B.nblk);
}

// Cells, in the mirror's order (place = mirror word << 5 | bit).  Top bit set:
// vacant, compartment in bits 27 to 30, in the low 27 the id of the lowest
// claimant (all ones: none).  Clear: occupied, species in bits 26 to 30, list
// slot below.
constexpr uint32_t kCellVacant = 0x80000000u;
constexpr uint32_t kCellNone = 0x07FFFFFFu;                    // no claimant
__device__ __forceinline__ uint32_t cell_claim(uint32_t comp, uint32_t id) { return kCellVacant | (comp << 27) | id; }
__device__ __forceinline__ uint32_t cell_free(uint32_t comp) { return cell_claim(comp, kCellNone); }
__device__ __forceinline__ uint32_t cell_of_entry(int s, uint32_t slot) { return ((uint32_t)s << 26) | slot; }

// vacant in compartment comp at the start of the event (claimed or not)
__device__ __forceinline__ bool cell_open(uint32_t w, uint32_t comp)
{
    return (w & kCellVacant) && ((w >> 27) & 15u) == comp;
}

__device__ __forceinline__ uint32_t small_place(const Geometry& G, int32_t i, int32_t j, int32_t k)
{
    const uint32_t word = (((uint32_t)k >> 1) * G.nbj + ((uint32_t)j >> 2)) * G.nbi + ((uint32_t)i >> 2);
    return (word << 5) | ((uint32_t)i & 3u) | (((uint32_t)j & 3u) << 2) | (((uint32_t)k & 1u) << 4);
}
__device__ __forceinline__ BitPos small_bit(uint32_t place) { return BitPos{place >> 5, 1u << (place & 31u)}; }

// Cells of all voxels from the mirrors (occupied ones 0: their lists' entries
// follow, k_cells_lists), a thread per voxel of a mirror word
__global__ void k_cells_vacant(uint32_t* cell, const uint32_t* bits0, uint64_t words, int n_mirrors)
{
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < words * 32;
         x += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t w = 0u;
        for (int c = 0; c < n_mirrors; ++c)
            if (!((bits0[(uint64_t)c * words + (x >> 5)] >> (x & 31u)) & 1u)) w = cell_free((uint32_t)c);
        cell[x] = w;
    }
}

__global__ void k_cells_lists(uint32_t* cell, const ModelDev* model, const int32_t* counts, int nsp, Geometry G)
{
    for (int s = 0; s < nsp; ++s) {
        const SpeciesList& list = model->lists[s];
        const int n = counts[s];
        for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += gridDim.x * blockDim.x) {
            int32_t i, j, k;
            decode(G, (uint32_t)list.vox[idx], i, j, k);
            cell[small_place(G, i, j, k)] = cell_of_entry(s, (uint32_t)idx);
        }
    }
}

// Mirrors and codes from the cells: a warp per mirror word.  A voxel's bit is
// set in every mirror if it is occupied, else in all but its compartment's.
__global__ void k_cells_grid(const uint32_t* cell, uint32_t* bits0, uint64_t words, int n_mirrors, uint16_t* occ,
                             Geometry G)
{
    const uint32_t lane = threadIdx.x & 31;
    for (uint64_t x = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5; x < words;
         x += ((uint64_t)gridDim.x * blockDim.x) >> 5) {
        const uint32_t w = cell[x * 32 + lane];
        const int32_t i = (int32_t)((uint32_t)(x % G.nbi) * 4u + (lane & 3u));
        const int32_t j = (int32_t)((uint32_t)((x / G.nbi) % G.nbj) * 4u + ((lane >> 2) & 3u));
        const int32_t k = (int32_t)((uint32_t)(x / ((uint64_t)G.nbi * G.nbj)) * 2u + (lane >> 4));
        const bool inside = i < G.ni && j < G.nj && k < G.nk;   // else its bit stays clear
        for (int c = 0; c < n_mirrors; ++c) {
            const unsigned m = __ballot_sync(0xFFFFFFFFu, inside && !cell_open(w, (uint32_t)c));
            if (lane == 0) bits0[(uint64_t)c * words + x] = m;
        }
        if (inside)
            occ[(uint64_t)i + (uint64_t)G.ni * ((uint64_t)j + (uint64_t)G.nj * (uint64_t)k)] =
                (w & kCellVacant) ? (uint16_t)0 : (uint16_t)((w >> 26) + 1u);
    }
}

void launch_cells_build(uint32_t* cell, const uint32_t* bits0, uint64_t words, int n_mirrors, const ModelDev* model,
                        const int32_t* counts, int nsp, const Geometry& geo, int blocks, cudaStream_t st)
{
    k_cells_vacant<<<blocks, 256, 0, st>>>(cell, bits0, words, n_mirrors);
    k_cells_lists<<<blocks, 256, 0, st>>>(cell, model, counts, nsp, geo);
}

void launch_cells_grid(const uint32_t* cell, uint32_t* bits0, uint64_t words, int n_mirrors, uint16_t* occ,
                       const Geometry& geo, int blocks, cudaStream_t st)
{
    k_cells_grid<<<blocks, 256, 0, st>>>(cell, bits0, words, n_mirrors, occ, geo);
}

// molecule (id, img) on voxel v, place p, joins list y
__device__ __forceinline__ void small_append(const SmallArgs& A, const ModelDev& M, int y, uint32_t v, uint32_t p,
                                             uint32_t id, uint64_t img)
{
    const SpeciesList dst = M.lists[y];
    const int slot = atomicAdd(&A.sc->counts[y], 1);
    if (slot >= dst.cap) {
        atomicOr(&A.sc->err, kErrListOverflow);
        return;
    }
    dst.vox[slot] = (int32_t)v;
    dst.ids[slot] = id;
    dst.img[slot] = img;
    A.cell[p] = cell_of_entry(y, (uint32_t)slot);
}

// the entry at `slot` of list x leaves it
__device__ __forceinline__ void small_leave(const SmallArgs& A, const ModelDev& M, int x, uint32_t slot)
{
    M.lists[x].vox[slot] = -1;
    atomicAdd(&A.sc->tmp_count[x], 1);
}

// A molecule between its claim and its commit phase: its voxel, id, the
// claim's outcome (kDec*; with a direction, kSmallWrap where the hop crosses a
// periodic boundary and kSmallReact where it is an accepted collision), the
// target voxel, the places of both, and the target's cell as it was.
struct SmallMol {
    int32_t v;
    uint32_t id, dec, t, pv, pt, w;
};
constexpr uint32_t kSmallWrap = 0x80u, kSmallReact = 0x40u;

// the target of direction d; false behind a reflective wall
__device__ __forceinline__ bool small_target(const Geometry& G, SmallMol& m, int32_t i, int32_t j, int32_t k, int d,
                                             uint64_t* wrap)
{
    Nb nb;
    if (!neighbor(G, i, j, k, d, nb)) return false;
    m.t = (uint32_t)nb.t;
    m.pv = small_place(G, i, j, k);
    m.pt = small_place(G, nb.i, nb.j, nb.k);
    *wrap = nb.wrap;
    return true;
}

// Claim phase of molecule (m.v, m.id) up to its target: m.dec is kDecFire (its
// claim, if it has one, is made), kDecNone or the direction; returns u1.
template <bool GENERAL>
__device__ __forceinline__ uint32_t small_aim(const SmallArgs& A, const EventArgs& a, const ModelDev& M, uint32_t g,
                                              SmallMol& m, unsigned& n_fire)
{
    int32_t i, j, k;
    decode(a.geo, (uint32_t)m.v, i, j, k);
    uint32_t u[4];
    philox(m.id, g, ((uint32_t)a.s << 4) | kTagEvent, 0u, a.key0, a.key1, u);
    m.dec = kDecNone;
    if (GENERAL && M.n_fo[a.s] > 0 && (uint64_t)u[2] < M.T_fire[a.s]) {
        ++n_fire;
        m.dec = kDecFire;
        const int r = pick_first_order(&M, a.s, u[3]);
        if (M.rx[r].np != 2) return 0u;
        // second product: uniform pick among the neighbours vacant now in its compartment
        const uint32_t comp = M.comp[M.rx[r].p1];
        uint32_t open = 0u;
        for (int d = 0; d < 12; ++d) {
            Nb nb;
            if (neighbor(a.geo, i, j, k, d, nb) &&
                cell_open(__ldcg(&A.cell[small_place(a.geo, nb.i, nb.j, nb.k)]), comp))
                open |= 1u << d;
        }
        if (!open) return 0u;
        for (int want = (int)__umulhi(u[0], (uint32_t)__popc(open)); want > 0; --want) open &= open - 1u;
        Nb nb;
        neighbor(a.geo, i, j, k, __ffs(open) - 1, nb);
        red_min(&A.cell[small_place(a.geo, nb.i, nb.j, nb.k)], cell_claim(comp, m.id));
        return 0u;
    }
    const int d = (int)__umulhi(u[0], 12u);
    uint64_t wrap;
    if (small_target(a.geo, m, i, j, k, d, &wrap)) m.dec = (uint32_t)d | (wrap ? kSmallWrap : 0u);
    return u[1];
}

// The rest of it, the target's cell being m.w: a claim or kDecNone.
template <bool GENERAL>
__device__ __forceinline__ void small_decide(const SmallArgs& A, const EventArgs& a, const ModelDev& M, SmallMol& m,
                                             uint32_t u1, unsigned& n_col, unsigned& n_acc)
{
    const uint32_t comp = M.comp[a.s];
    if (cell_open(m.w, comp)) {
        red_min(&A.cell[m.pt], cell_claim(comp, m.id));
        return;
    }
    bool go = false;
    if (GENERAL && !(m.w & kCellVacant)) {
        const int r = M.pair[a.s][m.w >> 26];
        if (r >= 0) {
            ++n_col;
            go = (uint64_t)u1 < M.rx[r].T;
            if (go) {
                ++n_acc;
                red_min(&a.ct.direct[m.t], m.id);               // its partner's voxel: a claim word
                m.dec |= kSmallReact;
            }
        }
    }
    if (!go) m.dec = kDecNone;
}

// the word the commit phase reads back: the claim word of a collision, else
// the target's cell
__device__ __forceinline__ uint32_t small_readback(const SmallArgs& A, const EventArgs& a, const SmallMol& m)
{
    return __ldcg((m.dec & kSmallReact) ? &a.ct.direct[m.t] : &A.cell[m.pt]);
}

// Commit phase of the molecule at list slot idx whose claim phase did not end
// with kDecNone; `back` is the word read back (not used for kDecFire).  A hop
// sets m.v.
template <bool GENERAL>
__device__ __forceinline__ void small_commit(const SmallArgs& A, const EventArgs& a, const ModelDev& M, uint32_t g,
                                             int idx, SmallMol& m, uint32_t back, unsigned& n_hop, unsigned& n_r2,
                                             unsigned& n_r1)
{
    const int s = a.s;
    const uint32_t v = (uint32_t)m.v, id = m.id;
    if (GENERAL && m.dec == kDecFire) {
        int32_t i, j, k;
        decode(a.geo, v, i, j, k);
        const uint32_t pv = small_place(a.geo, i, j, k);
        uint32_t u[4];
        philox(id, g, ((uint32_t)s << 4) | kTagEvent, 0u, a.key0, a.key1, u);
        const ReactionDev R = M.rx[pick_first_order(&M, s, u[3])];
        if (R.np == 2) {
            // the neighbour this molecule claimed, if it won it
            const uint32_t mine = cell_claim(M.comp[R.p1], id);
            for (int d = 0; d < 12; ++d) {
                Nb nb;
                if (!neighbor(a.geo, i, j, k, d, nb)) continue;
                if (__ldcg(&A.cell[small_place(a.geo, nb.i, nb.j, nb.k)]) != mine) continue;
                const uint64_t img = a.list.img[idx];
                if (R.p0 != s) {
                    small_leave(A, M, s, (uint32_t)idx);
                    small_append(A, M, R.p0, v, pv, id, img);
                }
                // (its cell follows with its list entry, in the births' pass)
                const int slot = atomicAdd(&A.sc->births, 1);
                A.sc->touched[g & 1u] = 1u;
                if (slot < a.births_cap) {
                    Birth b;
                    b.parent = id; b.t = nb.t; b.species = R.p1; b.pad = 0;
                    b.img = img_add(img, nb.wrap);
                    a.births[slot] = b;
                } else {
                    atomicOr(&A.sc->err, kErrBirthOverflow);
                }
                ++n_r1;
                break;
            }
            return;
        }
        ++n_r1;
        if (R.np && R.p0 == s) return;
        const uint64_t img = a.list.img[idx];
        small_leave(A, M, s, (uint32_t)idx);
        if (R.np) small_append(A, M, R.p0, v, pv, id, img);
        else A.cell[pv] = cell_free(M.comp[s]);
        return;
    }
    if (!GENERAL || !(m.dec & kSmallReact)) {
        if (back != cell_claim(M.comp[s], id)) return;
        A.cell[m.pt] = cell_of_entry(s, (uint32_t)idx);         // move (Sec. 2.3)
        A.cell[m.pv] = cell_free(M.comp[s]);
        a.list.vox[idx] = (int32_t)m.t;
        if (m.dec & kSmallWrap) {
            int32_t i, j, k;
            decode(a.geo, v, i, j, k);
            Nb nb;
            neighbor(a.geo, i, j, k, (int)(m.dec & 15u), nb);
            a.list.img[idx] = img_add(a.list.img[idx], nb.wrap);
        }
        m.v = (int32_t)m.t;
        ++n_hop;
        return;
    }
    // accepted collision with partner y (Sec. 2.4.2), if it won it: first
    // product on the partner's voxel, second on the mover's, unless that puts a
    // product outside its compartment (then they trade places)
    if (back != id) return;
    a.ct.direct[m.t] = kNoClaim;
    const int y = (int)(m.w >> 26);
    const uint32_t slot = m.w & 0x03FFFFFFu;
    const ReactionDev R = M.rx[M.pair[s][y]];
    const bool straight = R.np == 0 ||
                          (M.comp[R.p0] == M.comp[y] && (R.np < 2 || M.comp[R.p1] == M.comp[s]));
    int at_t = 0, at_v = 0;                                     // species + 1 afterwards
    if (R.np == 1) {
        if (straight) at_t = R.p0 + 1;
        else at_v = R.p0 + 1;
    } else if (R.np == 2) {
        at_t = (straight ? R.p0 : R.p1) + 1;
        at_v = (straight ? R.p1 : R.p0) + 1;
    }
    if (at_v != s + 1) {
        const uint64_t img = a.list.img[idx];
        small_leave(A, M, s, (uint32_t)idx);
        if (at_v) small_append(A, M, at_v - 1, v, m.pv, id, img);
        else A.cell[m.pv] = cell_free(M.comp[s]);
    }
    if (at_t != y + 1) {
        const uint32_t pid = __ldcg(&M.lists[y].ids[slot]);
        const uint64_t pimg = __ldcg(&M.lists[y].img[slot]);
        small_leave(A, M, y, slot);
        if (at_t) small_append(A, M, at_t - 1, m.t, m.pt, pid, pimg);
        else A.cell[m.pt] = cell_free(M.comp[y]);
    }
    ++n_r2;
}

// the entry of list x on voxel v is at slot h now
__device__ __forceinline__ void small_entry(const SmallArgs& A, const SmallShared& S, int x, int32_t v, uint32_t h)
{
    const Geometry& G = S.ev[0].geo;
    int32_t i, j, k;
    decode(G, (uint32_t)v, i, j, k);
    A.cell[small_place(G, i, j, k)] = cell_of_entry(x, h);
}

// The lists closed up.  In a cluster one block packs a list chunk by chunk
// (lists of a few thousand entries: a few microseconds).  In a grid every
// thread looks through its share of the lists with tombstones and notes the
// tombstones below the new length and the entries at or above it (as many);
// after a barrier these move into those.  Where the scratch does not hold them
// all (lists that grew far past their estimates) the blocks pack there too.
// The caller has a barrier before, if counts were read, and one after, if the
// stretch goes on.
template <SmallMode MODE>
__device__ bool small_close(const SmallArgs& A, SmallShared& S, const SmallBlocks& B, int t0, int stride)
{
    __shared__ int32_t s_warp[32];
    const ModelDev& M = S.model;
    if ((int)threadIdx.x < A.nsp) {
        S.n[threadIdx.x] = min(__ldcg(&A.sc->counts[threadIdx.x]), M.lists[threadIdx.x].cap);
        S.k[threadIdx.x] = __ldcg(&A.sc->tmp_count[threadIdx.x]);
    }
    __syncthreads();
    int64_t total = 0;
    for (int x = 0; x < A.nsp; ++x) total += S.k[x];
    if (total == 0) return true;
    const bool fits = MODE != kSmallInCluster && total <= A.scratch_n;
    int32_t base = 0;
    for (int x = 0; fits && x < A.nsp; ++x) {
        if (S.k[x] <= 0) continue;
        const int32_t n = S.n[x], n2 = n - S.k[x];
        const int32_t* vox = M.lists[x].vox;
        constexpr int U = 4;                                    // entries in flight
        for (int idx0 = t0; idx0 - (t0 & 31) < n; idx0 += U * stride) {      // whole warps
            int32_t v[U];
#pragma unroll
            for (int u = 0; u < U; ++u) v[u] = idx0 + u * stride < n ? __ldcg(vox + idx0 + u * stride) : -1;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int idx = idx0 + u * stride;
                const int h = warp_alloc(&A.sc->hole_n[x], idx < n2 && v[u] < 0);
                if (h >= 0) A.holes[base + h] = idx;
                const int q = warp_alloc(&A.sc->surv_n[x], idx >= n2 && v[u] >= 0);
                if (q >= 0) A.surv[base + q] = idx;
            }
        }
        base += S.k[x];
    }
    if (MODE != kSmallInCluster && !small_barrier<MODE>(A, B)) return false;
    base = 0;
    for (int x = 0; fits && x < A.nsp; ++x) {
        if (S.k[x] <= 0) continue;
        const SpeciesList list = M.lists[x];
        const int32_t moves = __ldcg(&A.sc->hole_n[x]);
        for (int q = t0; q < moves; q += stride) {
            const int32_t h = __ldcg(A.holes + base + q), p = __ldcg(A.surv + base + q);
            const int32_t v = __ldcg(list.vox + p);
            list.vox[h] = v;
            list.ids[h] = __ldcg(list.ids + p);
            list.img[h] = __ldcg(list.img + p);
            small_entry(A, S, x, v, (uint32_t)h);
        }
        if (t0 == 0) {
            A.sc->counts[x] = S.n[x] - S.k[x];
            A.sc->tmp_count[x] = 0;
        }
        base += S.k[x];
    }
    for (int x = B.blk; !fits && x < A.nsp; x += B.nblk) {
        if (S.k[x] <= 0) continue;
        const SpeciesList list = M.lists[x];
        const int32_t n = S.n[x];
        int32_t out = 0;                                        // entries kept so far
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
        for (int32_t at0 = 0; at0 < n; at0 += blockDim.x) {
            const int32_t p = at0 + threadIdx.x;
            const int32_t v = p < n ? __ldcg(list.vox + p) : -1;
            const uint32_t id = v >= 0 ? __ldcg(list.ids + p) : 0u;
            const uint64_t img = v >= 0 ? __ldcg(list.img + p) : 0ull;
            const unsigned live = __ballot_sync(0xFFFFFFFFu, v >= 0);
            if (lane == 0) s_warp[warp] = __popc(live);
            __syncthreads();                                    // the chunk is in registers
            int32_t at = out + __popc(live & ((1u << lane) - 1u));
            for (int w = 0; w < warps; ++w) {
                if (w < warp) at += s_warp[w];
                out += s_warp[w];
            }
            if (v >= 0 && at != p) {
                list.vox[at] = v;
                list.ids[at] = id;
                list.img[at] = img;
                small_entry(A, S, x, v, (uint32_t)at);
            }
            __syncthreads();
        }
        if (threadIdx.x == 0) {
            A.sc->counts[x] = out;
            A.sc->tmp_count[x] = 0;
        }
    }
    return true;
}

// Births of the event of a by many blocks: a warp counts the parents below one
// birth's, its rank among the ids handed out, and appends it.  Up to 8192 of them
// sorted and appended by one block as in launches per event phase, which have twice the
// threads there, took longer than the rest of an event (500,000 molecules that split
// 0.7 % an event and another 500,000 on 256^3 99 us per event so, 60 in ranks, 90 in
// launches).  Returns their number; the caller has a barrier, then moves the next id.
constexpr int kSmallBirthBlocks = 8;        // fewer blocks sort
__device__ __forceinline__ int small_births(const SmallArgs& A, const ModelDev& M, const EventArgs& a, const SmallBlocks& B)
{
    extern __shared__ unsigned long long keys[];
    uint32_t* parent = reinterpret_cast<uint32_t*>(keys);
    const int nb = min(min(__ldcg(&A.sc->births), a.births_cap), kBirthSortMax);
    for (int x = threadIdx.x; x < nb; x += blockDim.x) parent[x] = __ldcg(&a.births[x].parent);
    const uint32_t base_id = __ldcg(&A.sc->next_id);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int x = ((int)threadIdx.x >> 5) * B.nblk + B.blk; x < nb; x += B.nblk * ((int)blockDim.x >> 5)) {
        const uint32_t p = parent[x];
        unsigned below = 0;
        for (int y = lane; y < nb; y += 32) below += parent[y] < p ? 1u : 0u;
        below = __reduce_add_sync(0xFFFFFFFFu, below);
        if (lane != 0) continue;
        const uint32_t v = (uint32_t)__ldcg(&a.births[x].t);
        int32_t i, j, k;
        decode(a.geo, v, i, j, k);
        small_append(A, M, __ldcg(&a.births[x].species), v, small_place(a.geo, i, j, k), base_id + below,
                     __ldcg(&a.births[x].img));
    }
    return nb;
}

constexpr int kSmallCarry = 2;              // molecules a thread carries in registers

// One event of species s.  m: the entries (voxel, id) of the thread's first
// molecules (idx = t0 + c * stride), loaded by the caller; n: the list's
// length.  `next`: null, or the arguments of the next event, whose entries of
// this thread nobody else changes: they are loaded before the barrier.
template <bool GENERAL, SmallMode MODE>
__device__ __forceinline__ bool small_event(const SmallArgs& A, const SmallBlocks& B, const EventArgs& a,
                                            const ModelDev& M, uint32_t g, int t0, int stride, int n, SmallMol (&m)[kSmallCarry],
                                            const EventArgs* next)
{
    unsigned n_att = 0, n_col = 0, n_acc = 0, n_fire = 0, n_hop = 0, n_r2 = 0, n_r1 = 0;
    // kSmallCarry molecules of the thread at a time, from slot t0 + c0 * stride:
    // the cells' loads go out together
    auto claims = [&](int c0, SmallMol (&q)[kSmallCarry]) {
        uint32_t u1[kSmallCarry];
#pragma unroll
        for (int c = 0; c < kSmallCarry; ++c) {
            if (t0 + (c0 + c) * stride < n && q[c].v >= 0) {
                ++n_att;
                u1[c] = small_aim<GENERAL>(A, a, M, g, q[c], n_fire);
            } else {
                q[c].dec = kDecNone;
            }
        }
#pragma unroll
        for (int c = 0; c < kSmallCarry; ++c)
            if (q[c].dec != kDecNone && q[c].dec != kDecFire) q[c].w = __ldcg(&A.cell[q[c].pt]);
#pragma unroll
        for (int c = 0; c < kSmallCarry; ++c)
            if (q[c].dec != kDecNone && q[c].dec != kDecFire)
                small_decide<GENERAL>(A, a, M, q[c], u1[c], n_col, n_acc);
    };
    auto commits = [&](int c0, SmallMol (&q)[kSmallCarry]) {
        uint32_t back[kSmallCarry];
#pragma unroll
        for (int c = 0; c < kSmallCarry; ++c)
            if (q[c].dec != kDecNone && q[c].dec != kDecFire) back[c] = small_readback(A, a, q[c]);
#pragma unroll
        for (int c = 0; c < kSmallCarry; ++c)
            if (q[c].dec != kDecNone)
                small_commit<GENERAL>(A, a, M, g, t0 + (c0 + c) * stride, q[c], back[c], n_hop, n_r2, n_r1);
    };
    claims(0, m);
    for (int c0 = kSmallCarry; t0 + c0 * stride < n; c0 += kSmallCarry) {
        SmallMol q[kSmallCarry];
#pragma unroll
        for (int c = 0; c < kSmallCarry; ++c) {
            const int idx = t0 + (c0 + c) * stride;
            q[c].v = idx < n ? __ldcg(&a.list.vox[idx]) : -1;
            q[c].id = idx < n ? __ldcg(&a.list.ids[idx]) : 0u;
        }
        claims(c0, q);
#pragma unroll
        for (int c = 0; c < kSmallCarry; ++c) {
            const int idx = t0 + (c0 + c) * stride;
            if (idx < n) a.dec[idx] = (uint8_t)q[c].dec;        // read back by this thread
        }
    }
    if (!small_barrier<MODE>(A, B)) return false;
    commits(0, m);
    for (int c0 = kSmallCarry; t0 + c0 * stride < n; c0 += kSmallCarry) {
        SmallMol q[kSmallCarry];
#pragma unroll
        for (int c = 0; c < kSmallCarry; ++c) {
            const int idx = t0 + (c0 + c) * stride;
            q[c].dec = idx < n ? a.dec[idx] : (uint32_t)kDecNone;
            q[c].v = idx < n ? __ldcg(&a.list.vox[idx]) : -1;
            q[c].id = idx < n ? __ldcg(&a.list.ids[idx]) : 0u;
        }
#pragma unroll
        for (int c = 0; c < kSmallCarry; ++c) {
            if (q[c].dec == kDecNone || q[c].dec == kDecFire) continue;
            int32_t i, j, k;
            decode(a.geo, (uint32_t)q[c].v, i, j, k);
            uint64_t wrap;
            small_target(a.geo, q[c], i, j, k, (int)(q[c].dec & 15u), &wrap);
            if (q[c].dec & kSmallReact) q[c].w = __ldcg(&A.cell[q[c].pt]);
        }
        commits(c0, q);
    }
    if (next != nullptr && next != &a) {
#pragma unroll
        for (int c = 0; c < kSmallCarry; ++c) {
            const int idx = t0 + c * stride;
            if (idx >= next->list.cap) continue;
            m[c].v = __ldcg(&next->list.vox[idx]);
            m[c].id = __ldcg(&next->list.ids[idx]);
        }
    }
    if (A.collect_stats) {
        flush_stat(&A.sc->stats[kStatAttempts], n_att);
        flush_stat(&A.sc->stats[kStatHops], n_hop);
        if (GENERAL) {
            flush_stat(&A.sc->stats[kStatCollisions], n_col);
            flush_stat(&A.sc->stats[kStatAccepted], n_acc);
            flush_stat(&A.sc->stats[kStatFires], n_fire);
            flush_stat(&A.sc->stats[kStatReactions2], n_r2);
            flush_stat(&A.sc->stats[kStatReactions1], n_r1);
        }
    }
    return small_barrier<MODE>(A, B);
}

// false: a wait ran out
template <SmallMode MODE>
__device__ __forceinline__ bool small_run(const SmallArgs& A, SmallShared& S, const SmallBlocks& B)
{
    // a list is dealt out warp by warp over the blocks, so that a short one
    // keeps every SM of the launch busy
    const int blk = B.blk, nblk = B.nblk;
    const int lane = (int)threadIdx.x & 31;
    const int t0 = (((int)threadIdx.x >> 5) * nblk + blk) * 32 + lane;
    const int stride = nblk * (int)blockDim.x;
    small_copy(S.ev, A.ev, sizeof(EventArgs) * A.nsp);
    small_copy(&S.model, A.model, sizeof(ModelDev));
    for (int e = threadIdx.x; e < A.n_events; e += blockDim.x) S.seq[e] = A.seq[e];
    if (t0 < kMaxSpecies) {
        A.sc->tmp_count[t0] = 0;                                // tombstones per list
        A.sc->hole_n[t0] = 0;
        A.sc->surv_n[t0] = 0;
    }
    if (t0 < 2) A.sc->touched[t0] = 0u;
    __syncthreads();
    if ((int)threadIdx.x < A.nsp) {
        S.ev[threadIdx.x].collect_stats = A.collect_stats;
        S.n[threadIdx.x] = A.sc->counts[threadIdx.x];
    }
    __syncthreads();
    if (!small_barrier<MODE>(A, B)) return false;
    const ModelDev& M = S.model;
    bool prev_fo2 = false, loaded = false;
    SmallMol m[kSmallCarry];
    for (int e = 0; e <= A.n_events; ++e) {
        const bool last = e == A.n_events;
        const uint32_t g = A.g + (uint32_t)e;
        const int s = last ? 0 : S.seq[e];
        const EventArgs& a = S.ev[s];
        int n = 0;
        for (;;) {
            // one round of loads: the list's length and first entries, the
            // lengths of the lists the event may append to, and whether the
            // last event left births
            uint32_t born = 0u;
            int32_t room = INT32_MAX, holes = 0;
            if (prev_fo2) born = __ldcg(&A.sc->touched[(g & 1u) ^ 1u]);
            if (!last) {
                // without reactions the lengths stay
                n = A.general ? __ldcg(&A.sc->counts[s]) : S.n[s];
                if ((A.products[s] >> lane) & 1u) room = M.lists[lane].cap - __ldcg(&A.sc->counts[lane]);
                if (A.products[s] && lane < A.nsp) holes = __ldcg(&A.sc->tmp_count[lane]);
                if (!loaded) {
#pragma unroll
                    for (int c = 0; c < kSmallCarry; ++c) {
                        const int idx = t0 + c * stride;
                        if (idx >= a.list.cap) continue;
                        m[c].v = __ldcg(&a.list.vox[idx]);
                        m[c].id = __ldcg(&a.list.ids[idx]);
                    }
                }
            }
            // the same decision in every warp: nothing read here changes
            // between the last event's end and this event's commit phase
            if (born) {
                int nb = -1;
                if (nblk >= kSmallBirthBlocks) nb = small_births(A, M, S.ev[S.seq[e - 1]], B);
                else if (blk == 0) births_body(S.ev[S.seq[e - 1]], A.cell);
                prev_fo2 = false;
                if (!small_barrier<MODE>(A, B)) return false;
                if (nb >= 0 && t0 == 0) {                       // everybody has read them
                    A.sc->next_id += (uint32_t)nb;
                    A.sc->births = 0;
                    if (A.collect_stats) A.sc->stats[kStatBirths] += (unsigned long long)nb;
                }
                continue;
            }
            if (last) break;
            // (a list without tombstones has room for what the event can add)
            const bool tight = __any_sync(0xFFFFFFFFu, holes > 0 && room < 2 * (int64_t)n) ||
                               (A.scratch_n > 0 && __any_sync(0xFFFFFFFFu, holes > 0) &&
                                (int64_t)__reduce_add_sync(0xFFFFFFFFu, holes) + 2 * (int64_t)n >
                                    (int64_t)A.scratch_n);
            if (!tight) break;
            if (!small_barrier<MODE>(A, B)) return false;             // the counts are read
            if (!small_close<MODE>(A, S, B, t0, stride)) return false;
            if (!small_barrier<MODE>(A, B)) return false;
            if (t0 < kMaxSpecies) A.sc->hole_n[t0] = A.sc->surv_n[t0] = 0;
        }
        if (last) {
            return A.general ? small_close<MODE>(A, S, B, t0, stride) : true;
        }
        n = min(n, a.list.cap);
        if ((A.general >> s) & 1u) {
            // word g & 1 was last read an event ago
            if (t0 == 0) A.sc->touched[g & 1u] = 0u;
            if (!small_event<true, MODE>(A, B, a, M, g, t0, stride, n, m, nullptr)) return false;
        } else {
            const EventArgs* next = (A.general || e + 1 == A.n_events) ? nullptr : &S.ev[S.seq[e + 1]];
            if (!small_event<false, MODE>(A, B, a, M, g, t0, stride, n, m, next)) return false;
            loaded = next != nullptr;
        }
        prev_fo2 = (A.fo2 >> s) & 1u;
    }
    return true;
}

template <bool CLUSTER>
__global__ void __launch_bounds__(kSmallThreads, 1) k_small_run(const SmallArgs A)
{
    __shared__ SmallShared S;
    small_run<CLUSTER ? kSmallInCluster : kSmallInGrid>(A, S, SmallBlocks{(int)blockIdx.x, (int)gridDim.x});
}

// Stretches of many lattices in one cooperative launch, each with a group of
// consecutive blocks and at its own pace: no lattice waits for another.
// Measured (us for an event of every member, the first 64 events / after 450;
// before: a launch per phase for all of them): 64 members of 96^3 with 5 % A and B
// 171 / 31 -> 106 / 15; 64 of 160^3 with 2 % 446 / 155 -> 261 / 74, bound by
// scattered DRAM accesses, as the members' cells are 1 GB.
// counts: list lengths (-1 where they are not known), next id and error bits
// afterwards, [lattice][kSmallCounts], for the next launch's groups.
__global__ void __launch_bounds__(kSmallThreads, 1) k_small_batch(const SmallArgs* args, const SmallStretch* stretch,
                                                                  const int32_t* group, const uint8_t* seq,
                                                                  int32_t* counts)
{
    __shared__ SmallShared S;
    __shared__ SmallArgs A;
    static_assert(offsetof(SmallArgs, seq) % 4 == 0, "copied by words");
    const int32_t r = group[blockIdx.x];
    const SmallStretch mine = stretch[r];
    small_copy(&A, args + mine.slot, offsetof(SmallArgs, seq));
    for (int e = threadIdx.x; e < mine.n_events; e += blockDim.x) A.seq[e] = seq[mine.seq + e];
    __syncthreads();
    if (threadIdx.x == 0) {
        A.g = mine.g;
        A.n_events = mine.n_events;
    }
    __syncthreads();
    const SmallBlocks B{(int)blockIdx.x - mine.block0, mine.blocks};
    const bool done = small_run<kSmallInGroup>(A, S, B);
    int32_t* out = counts + r * kSmallCounts;
    if (B.blk == 0 && (int)threadIdx.x < A.nsp)
        out[threadIdx.x] = done && A.general ? S.n[threadIdx.x] - S.k[threadIdx.x] : -1;
    if (B.blk == 0 && threadIdx.x == 0) {
        out[kMaxSpecies] = (int32_t)min(A.sc->next_id, 0x7FFFFFFFu);
        out[kMaxSpecies + 1] = __ldcg(&A.sc->err);
    }
}

int small_batch_blocks(int sm_count, int threads, bool births)
{
    const void* f = (const void*)k_small_batch;
    const int smem = kBirthSortMax * (int)sizeof(unsigned long long);
    int per_sm = 0;
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, threads, births ? smem : 0) != cudaSuccess)
        per_sm = 0;
    cudaGetLastError();
    return per_sm * sm_count;
}

cudaError_t launch_small_batch(const SmallArgs* args, const SmallStretch* stretch, const int32_t* group,
                               const uint8_t* seq, int32_t* counts, int blocks, int threads, bool births,
                               cudaStream_t st)
{
    void* p[] = {&args, &stretch, &group, &seq, &counts};
    return cudaLaunchCooperativeKernel((const void*)k_small_batch, dim3(blocks), dim3(threads), p,
                                       births ? (size_t)kBirthSortMax * sizeof(unsigned long long) : 0, st);
}

static void small_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute& at, int blocks, int threads, bool cluster, bool births)
{
    if (cluster) {
        at.id = cudaLaunchAttributeClusterDimension;
        at.val.clusterDim.x = (unsigned)blocks;
        at.val.clusterDim.y = at.val.clusterDim.z = 1;
    } else {
        at.id = cudaLaunchAttributeCooperative;
        at.val.cooperative = 1;
    }
    cfg.gridDim = dim3(blocks);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = births ? (size_t)kBirthSortMax * sizeof(unsigned long long) : 0;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
}

void small_limits(int sm_count, int* cluster, int* grid)
{
    const void* fc = (const void*)k_small_run<true>;
    const void* fg = (const void*)k_small_run<false>;
    const int smem = kBirthSortMax * (int)sizeof(unsigned long long);
    *cluster = 0;
    *grid = 0;
    if (cudaFuncSetAttribute(fc, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess &&
        cudaFuncSetAttribute(fc, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        for (int m = 16; m >= 8 && *cluster == 0; m /= 2) {
            cudaLaunchConfig_t cfg{};
            cudaLaunchAttribute at{};
            small_config(cfg, at, m, kSmallThreads, true, true);
            int clusters = 0;
            if (cudaOccupancyMaxActiveClusters(&clusters, fc, &cfg) == cudaSuccess && clusters > 0) *cluster = m;
        }
    }
    int per_sm = 0;
    if (cudaFuncSetAttribute(fg, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess &&
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fg, kSmallThreads, smem) == cudaSuccess)
        *grid = per_sm * sm_count;
    cudaGetLastError();
}

cudaError_t launch_small(const SmallArgs& A, int blocks, int threads, bool cluster, cudaStream_t st)
{
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    small_config(cfg, at, blocks, threads, cluster, A.fo2 != 0u);
    cfg.stream = st;
    return cluster ? cudaLaunchKernelEx(&cfg, k_small_run<true>, A) : cudaLaunchKernelEx(&cfg, k_small_run<false>, A);
}
