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
//   - a map from voxel to list slot (of the species that can be a partner)
//     tells a reacting molecule where its partner's entry is, so the commit
//     itself takes both entries off their lists and appends the products: no
//     list is checked against the grid;
//   - an entry that leaves stays behind as a tombstone (voxel -1); the lists
//     are closed up at the end of the stretch, or when one could run out of
//     room.
// Births need a pass of their own (ids in parent order) in events that have
// any.
//
// Measured (us per event; before: CUDA graphs of per-event launches, or the
// molecule-list kernel for walkers): A + B -> C of 2000 + 2000 molecules on
// 64^3 12.5 -> 4.9, a cascade of 22 species of up to 16,000 molecules on 200^3
// 10.5 -> 3.6, 30,000 ligands and 5000 receptors in a cell on 128^3 19.8 -> 8.0,
// 2621 walkers on 64^3 8.2 -> 3.9.

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
    if (MODE == kSmallInGroup && B.nblk == 1) {
        __syncthreads();                                        // what a block wrote, the block sees
        return true;
    }
    return block_barrier(A.barrier, &A.sc->err, A.barrier_timeout_ns, 0u, B.blk, B.nblk);
}

// molecule (id, img) on voxel v joins list y
__device__ __forceinline__ void small_append(const SmallArgs& A, const ModelDev& M, int y, uint32_t v, uint32_t id,
                                             uint64_t img)
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
    if ((A.mapped >> y) & 1u) A.slot[v] = (uint32_t)slot;
}

// the entry at `slot` of list x leaves it
__device__ __forceinline__ void small_leave(const SmallArgs& A, const ModelDev& M, int x, uint32_t slot)
{
    M.lists[x].vox[slot] = -1;
    atomicAdd(&A.sc->tmp_count[x], 1);
}

// A molecule between its claim and its commit phase: its voxel, id, the
// claim's outcome (kDec*, with kSmallWrap where the hop crosses a periodic
// boundary), the target voxel, and the places of both in the vacancy mirror
// (word << 5 | bit).
struct SmallMol {
    int32_t v;
    uint32_t id, dec, t, wv, wt;
};
constexpr uint32_t kSmallWrap = 0x80u;

__device__ __forceinline__ uint32_t small_place(const Geometry& G, int32_t i, int32_t j, int32_t k)
{
    const uint32_t word = (((uint32_t)k >> 1) * G.nbj + ((uint32_t)j >> 2)) * G.nbi + ((uint32_t)i >> 2);
    return (word << 5) | ((uint32_t)i & 3u) | (((uint32_t)j & 3u) << 2) | (((uint32_t)k & 1u) << 4);
}
__device__ __forceinline__ BitPos small_bit(uint32_t place) { return BitPos{place >> 5, 1u << (place & 31u)}; }

// the target of direction d; false behind a reflective wall
__device__ __forceinline__ bool small_target(const Geometry& G, SmallMol& m, int32_t i, int32_t j, int32_t k, int d,
                                             uint64_t* wrap)
{
    Nb nb;
    if (!neighbor(G, i, j, k, d, nb)) return false;
    m.t = (uint32_t)nb.t;
    m.wv = small_place(G, i, j, k);
    m.wt = small_place(G, nb.i, nb.j, nb.k);
    *wrap = nb.wrap;
    return true;
}

// Claim phase of molecule (m.v, m.id): the rest of m.
template <bool GENERAL>
__device__ __forceinline__ void small_claim(const EventArgs& a, const ModelDev& M, uint32_t g, SmallMol& m,
                                            unsigned& n_col, unsigned& n_acc, unsigned& n_fire)
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
        if (M.rx[r].np != 2) return;
        // second product: uniform pick among the neighbours vacant now in its compartment
        const uint32_t* pb = M.mirror[M.rx[r].p1];
        uint32_t open = 0u;
        for (int d = 0; d < 12; ++d) {
            Nb nb;
            if (neighbor(a.geo, i, j, k, d, nb) && !occupied(pb, bitpos(a.geo, nb.i, nb.j, nb.k))) open |= 1u << d;
        }
        if (!open) return;
        for (int want = (int)__umulhi(u[0], (uint32_t)__popc(open)); want > 0; --want) open &= open - 1u;
        Nb nb;
        neighbor(a.geo, i, j, k, __ffs(open) - 1, nb);
        claim<false>(a, nb, m.id);
        return;
    }
    const int d = (int)__umulhi(u[0], 12u);
    uint64_t wrap;
    if (!small_target(a.geo, m, i, j, k, d, &wrap)) return;
    bool go = !occupied(a.bits, small_bit(m.wt));
    if (GENERAL && !go) {
        const uint16_t o = __ldcg(&a.occ[m.t]);
        if (o != 0 && o != kBlocked) {
            const int r = M.pair[a.s][o - 1];
            if (r >= 0) {
                ++n_col;
                go = (uint64_t)u[1] < M.rx[r].T;
                if (go) ++n_acc;
            }
        }
    }
    if (!go) return;
    atomicMin(&a.ct.direct[m.t], m.id);
    m.dec = (uint32_t)d | (wrap ? kSmallWrap : 0u);
}

// did molecule id win voxel t?  (the winner resets the word)
__device__ __forceinline__ bool small_won(const EventArgs& a, uint32_t t, uint32_t id)
{
    if (__ldcg(&a.ct.direct[t]) != id) return false;
    a.ct.direct[t] = kNoClaim;
    return true;
}

// Commit phase of the molecule at list slot idx whose claim phase did not end
// with kDecNone; a hop sets m.v.
template <bool GENERAL>
__device__ __forceinline__ void small_commit(const SmallArgs& A, const EventArgs& a, const ModelDev& M, uint32_t g,
                                             int idx, SmallMol& m, unsigned& n_hop, unsigned& n_r2, unsigned& n_r1)
{
    const int s = a.s;
    const uint32_t v = (uint32_t)m.v, id = m.id;
    if (GENERAL && m.dec == kDecFire) {
        int32_t i, j, k;
        decode(a.geo, v, i, j, k);
        const BitPos bv = bitpos(a.geo, i, j, k);
        uint32_t u[4];
        philox(id, g, ((uint32_t)s << 4) | kTagEvent, 0u, a.key0, a.key1, u);
        const ReactionDev R = M.rx[pick_first_order(&M, s, u[3])];
        if (R.np == 2) {
            // the neighbour this molecule claimed, if it won it; only its
            // winner changes the bit of a claimed voxel
            uint32_t* pb = M.mirror[R.p1];
            for (int d = 0; d < 12; ++d) {
                Nb nb;
                if (!neighbor(a.geo, i, j, k, d, nb)) continue;
                const BitPos bt = bitpos(a.geo, nb.i, nb.j, nb.k);
                if (occupied(pb, bt) || !small_won(a, (uint32_t)nb.t, id)) continue;
                a.occ[v] = (uint16_t)(R.p0 + 1);
                a.occ[nb.t] = (uint16_t)(R.p1 + 1);
                bit_set(pb, bt);
                const uint64_t img = a.list.img[idx];
                if (R.p0 != s) {
                    small_leave(A, M, s, (uint32_t)idx);
                    small_append(A, M, R.p0, v, id, img);
                }
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
        if (R.np == 0) {
            a.occ[v] = 0;
            bit_clear(a.bits, bv);
        } else {
            a.occ[v] = (uint16_t)(R.p0 + 1);
            if (R.p0 == s) return;
        }
        const uint64_t img = a.list.img[idx];
        small_leave(A, M, s, (uint32_t)idx);
        if (R.np) small_append(A, M, R.p0, v, id, img);
        return;
    }
    // the bit of a claimed voxel only changes through its winner, so it still
    // tells a vacant target (hop) from a partner (reaction)
    const BitPos bv = small_bit(m.wv), bt = small_bit(m.wt);
    const uint32_t word = GENERAL ? __ldcg(&a.bits[bt.word]) : 0u;
    if (!small_won(a, m.t, id)) return;
    if (!GENERAL || !(word & bt.mask)) {
        bit_move(a.bits, bv, bt);                               // move (Sec. 2.3)
        if (a.live) {
            a.occ[m.t] = (uint16_t)(s + 1);
            a.occ[v] = 0;
        }
        a.list.vox[idx] = (int32_t)m.t;
        if (GENERAL && ((A.mapped >> s) & 1u)) A.slot[m.t] = (uint32_t)idx;
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
    // accepted collision with partner y (Sec. 2.4.2): first product on the
    // partner's voxel, second on the mover's, unless that puts a product
    // outside its compartment (then they trade places)
    const int y = (int)__ldcg(&a.occ[m.t]) - 1;
    const ReactionDev R = M.rx[M.pair[s][y]];
    const bool straight = R.np == 0 ||
                          (M.comp[R.p0] == M.comp[y] && (R.np < 2 || M.comp[R.p1] == M.comp[s]));
    int at_t = 0, at_v = 0;                                     // codes afterwards
    if (R.np == 1) {
        if (straight) at_t = R.p0 + 1;
        else at_v = R.p0 + 1;
    } else if (R.np == 2) {
        at_t = (straight ? R.p0 : R.p1) + 1;
        at_v = (straight ? R.p1 : R.p0) + 1;
    }
    a.occ[m.t] = (uint16_t)at_t;
    a.occ[v] = (uint16_t)at_v;
    if (at_t == 0) bit_clear(M.mirror[y], bt);
    if (at_v == 0) bit_clear(a.bits, bv);
    if (at_v != s + 1) {
        const uint64_t img = a.list.img[idx];
        small_leave(A, M, s, (uint32_t)idx);
        if (at_v) small_append(A, M, at_v - 1, v, id, img);
    }
    if (at_t != y + 1) {
        const uint32_t slot = __ldcg(&A.slot[m.t]);            // the partner's entry
        const uint32_t pid = __ldcg(&M.lists[y].ids[slot]);
        const uint64_t pimg = __ldcg(&M.lists[y].img[slot]);
        small_leave(A, M, y, slot);
        if (at_t) small_append(A, M, at_t - 1, m.t, pid, pimg);
    }
    ++n_r2;
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
        for (int idx = t0; idx - (t0 & 31) < n; idx += stride) {      // whole warps
            const bool live = idx < n && __ldcg(vox + idx) >= 0;
            const int h = warp_alloc(&A.sc->hole_n[x], idx < n2 && !live);
            if (h >= 0) A.holes[base + h] = idx;
            const int q = warp_alloc(&A.sc->surv_n[x], idx >= n2 && live);
            if (q >= 0) A.surv[base + q] = idx;
        }
        base += S.k[x];
    }
    if (MODE != kSmallInCluster && !small_barrier<MODE>(A, B)) return false;
    base = 0;
    for (int x = 0; fits && x < A.nsp; ++x) {
        if (S.k[x] <= 0) continue;
        const SpeciesList list = M.lists[x];
        const int32_t moves = __ldcg(&A.sc->hole_n[x]);
        const bool mapped = (A.mapped >> x) & 1u;
        for (int q = t0; q < moves; q += stride) {
            const int32_t h = __ldcg(A.holes + base + q), p = __ldcg(A.surv + base + q);
            const int32_t v = __ldcg(list.vox + p);
            list.vox[h] = v;
            list.ids[h] = __ldcg(list.ids + p);
            list.img[h] = __ldcg(list.img + p);
            if (mapped) A.slot[v] = (uint32_t)h;
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
                if ((A.mapped >> x) & 1u) A.slot[v] = (uint32_t)at;
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
#pragma unroll
    for (int c = 0; c < kSmallCarry; ++c) {
        if (t0 + c * stride < n && m[c].v >= 0) {
            ++n_att;
            small_claim<GENERAL>(a, M, g, m[c], n_col, n_acc, n_fire);
        } else {
            m[c].dec = kDecNone;
        }
    }
    for (int idx = t0 + kSmallCarry * stride; idx < n; idx += stride) {
        SmallMol w;
        w.v = __ldcg(&a.list.vox[idx]);
        w.id = __ldcg(&a.list.ids[idx]);
        w.dec = kDecNone;
        if (w.v >= 0) {
            ++n_att;
            small_claim<GENERAL>(a, M, g, w, n_col, n_acc, n_fire);
        }
        a.dec[idx] = (uint8_t)w.dec;                            // read back by this thread
    }
    if (!small_barrier<MODE>(A, B)) return false;
#pragma unroll
    for (int c = 0; c < kSmallCarry; ++c)
        if (m[c].dec != kDecNone) small_commit<GENERAL>(A, a, M, g, t0 + c * stride, m[c], n_hop, n_r2, n_r1);
    for (int idx = t0 + kSmallCarry * stride; idx < n; idx += stride) {
        SmallMol w;
        w.dec = a.dec[idx];
        if (w.dec == kDecNone) continue;
        w.v = __ldcg(&a.list.vox[idx]);
        w.id = __ldcg(&a.list.ids[idx]);
        if (w.dec != kDecFire) {
            int32_t i, j, k;
            decode(a.geo, (uint32_t)w.v, i, j, k);
            uint64_t wrap;
            small_target(a.geo, w, i, j, k, (int)(w.dec & 15u), &wrap);
        }
        small_commit<GENERAL>(A, a, M, g, idx, w, n_hop, n_r2, n_r1);
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

template <SmallMode MODE>
__device__ __forceinline__ void small_run(const SmallArgs& A, SmallShared& S, const SmallBlocks& B)
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
    // the voxel -> slot map, where it does not hold from the last stretch
    if (A.build_map) {
        for (uint32_t m = A.mapped; m; m &= m - 1u) {
            const int x = __ffs(m) - 1;
            const SpeciesList& list = A.model->lists[x];
            const int n = A.sc->counts[x];
            for (int idx = t0; idx < n; idx += stride) A.slot[list.vox[idx]] = (uint32_t)idx;
        }
    }
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
    if (!small_barrier<MODE>(A, B)) return;
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
                if (blk == 0) births_body(S.ev[S.seq[e - 1]], A.slot, A.mapped);
                prev_fo2 = false;
                if (!small_barrier<MODE>(A, B)) return;
                continue;
            }
            if (last) break;
            // (a list without tombstones has room for what the event can add)
            const bool tight = __any_sync(0xFFFFFFFFu, holes > 0 && room < 2 * (int64_t)n) ||
                               (A.scratch_n > 0 && __any_sync(0xFFFFFFFFu, holes > 0) &&
                                (int64_t)__reduce_add_sync(0xFFFFFFFFu, holes) + 2 * (int64_t)n >
                                    (int64_t)A.scratch_n);
            if (!tight) break;
            if (!small_barrier<MODE>(A, B)) return;             // the counts are read
            if (!small_close<MODE>(A, S, B, t0, stride)) return;
            if (!small_barrier<MODE>(A, B)) return;
            if (t0 < kMaxSpecies) A.sc->hole_n[t0] = A.sc->surv_n[t0] = 0;
        }
        if (last) {
            if (A.general) small_close<MODE>(A, S, B, t0, stride);
            return;
        }
        n = min(n, a.list.cap);
        if ((A.general >> s) & 1u) {
            // word g & 1 was last read an event ago
            if (t0 == 0) A.sc->touched[g & 1u] = 0u;
            if (!small_event<true, MODE>(A, B, a, M, g, t0, stride, n, m, nullptr)) return;
        } else {
            const EventArgs* next = (A.general || e + 1 == A.n_events) ? nullptr : &S.ev[S.seq[e + 1]];
            if (!small_event<false, MODE>(A, B, a, M, g, t0, stride, n, m, next)) return;
            loaded = next != nullptr;
        }
        prev_fo2 = (A.fo2 >> s) & 1u;
    }
}

template <bool CLUSTER>
__global__ void __launch_bounds__(kSmallThreads, CLUSTER ? 1 : 2) k_small_run(const SmallArgs A)
{
    __shared__ SmallShared S;
    small_run<CLUSTER ? kSmallInCluster : kSmallInGrid>(A, S, SmallBlocks{(int)blockIdx.x, (int)gridDim.x});
}

// Stretches of many lattices in one cooperative launch, each with a group of
// consecutive blocks and at its own pace: no lattice waits for another.
// counts: list lengths afterwards, [lattice][kMaxSpecies], for the next
// launch's groups.
__global__ void __launch_bounds__(kSmallThreads, 2) k_small_batch(const SmallArgs* args, const int2* group,
                                                                  int32_t* counts)
{
    __shared__ SmallShared S;
    __shared__ SmallArgs A;
    const int2 mine = group[blockIdx.x];                        // lattice, first block of its group
    small_copy(&A, args + mine.x, sizeof(SmallArgs));
    __syncthreads();
    const SmallBlocks B{(int)blockIdx.x - mine.y, A.blocks};
    small_run<kSmallInGroup>(A, S, B);
    if (A.general && B.blk == 0 && (int)threadIdx.x < A.nsp)
        counts[mine.x * kMaxSpecies + threadIdx.x] = S.n[threadIdx.x] - S.k[threadIdx.x];
}

int small_batch_blocks(int sm_count)
{
    const void* f = (const void*)k_small_batch;
    const int smem = kBirthSortMax * (int)sizeof(unsigned long long);
    int per_sm = 0;
    if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, f, kSmallThreads, smem) != cudaSuccess)
        per_sm = 0;
    cudaGetLastError();
    return per_sm * sm_count;
}

cudaError_t launch_small_batch(const SmallArgs* args, const int2* group, int32_t* counts, int blocks, bool births,
                               cudaStream_t st)
{
    void* p[] = {&args, &group, &counts};
    return cudaLaunchCooperativeKernel((const void*)k_small_batch, dim3(blocks), dim3(kSmallThreads), p,
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
