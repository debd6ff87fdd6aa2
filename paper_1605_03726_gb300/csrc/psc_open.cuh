// psc_open.cuh -- claim and commit launches of one event of a species without
// reactions on a large, sparse lattice (kOpenList, kWalkVoxels, kOpenOccupied).  Part
// of psc_kernels.cu's translation unit.
//
// What bounds them: scattered accesses, to DRAM where the claim words (or
// tables) of the lattice do not fit in the L2 cache.  A molecule whose target is
// vacant and has no other molecule among its twelve neighbours needs no claim,
// since only molecules next to a voxel can hop into it (the rule is the tile
// kernels').  At 1 % occupancy that is nine hops of ten.  The test reads the up
// to eight mirror words around the target; in a list in Morton order a block's
// molecules share them in the L1 cache (the mirror does not change during the
// claim launch), so each block takes a stretch of consecutive entries.
// Entries load a row or two ahead: a thread's loads would otherwise be one chain
// per molecule (1024^3 339 us per event without, 512^3 338, the closed one 172).
// Measured, us per event (before: plain claims of every hop in hash tables, or
// the tile kernel where its boxes fit in shared memory): 10.7M walkers on
// 1024^3 843 -> 331, 9.4M on 512^3 547 -> 325, 4.8M on a closed
// 401 x 399 x 301 lattice 348 -> 167.
constexpr uint8_t kDecOpen = 16;            // flag: hop without a claim, direction in the low bits

// Occupied voxels among the target (ti, tj, tk) and its neighbours: 1 is the
// mover itself alone.  2 where the mirror's bricks do not line up across a
// periodic boundary next to the target (the claim decides then).
__device__ __forceinline__ int open_count(const Geometry& G, const uint32_t* bits, const uint32_t* nbmask, int ti,
                                          int tj, int tk)
{
    const int nbi = (int)G.nbi, nbj = (int)G.nbj, nbk = (G.nk + 1) >> 1;
    if (((G.bflags & 1u) && (G.ni & 3) && (ti == 0 || ti == G.ni - 1)) ||
        ((G.bflags & 2u) && (G.nj & 3) && (tj == 0 || tj == G.nj - 1)) ||
        ((G.bflags & 4u) && (G.nk & 1) && (tk == 0 || tk == G.nk - 1)))
        return 2;
    const int c3 = (G.bflags & 8u) ? tk % 3 : 0;
    const int c = ((ti & 3) | ((tj & 3) << 2) | ((tk & 1) << 4)) + 32 * c3;
    int x[2] = {(ti - 1) >> 2, ((ti - 1) >> 2) + 1}, y[2] = {(tj - 1) >> 2, ((tj - 1) >> 2) + 1},
        z[2] = {(tk - 1) >> 1, ((tk - 1) >> 1) + 1};
    // across a periodic boundary; behind a wall (or the end of the last
    // brick) there is nobody
    if (x[0] < 0) x[0] = (G.bflags & 1u) ? nbi - 1 : -1;
    if (x[1] >= nbi) x[1] = (G.bflags & 1u) ? 0 : -1;
    if (y[0] < 0) y[0] = (G.bflags & 2u) ? nbj - 1 : -1;
    if (y[1] >= nbj) y[1] = (G.bflags & 2u) ? 0 : -1;
    if (z[0] < 0) z[0] = (G.bflags & 4u) ? nbk - 1 : -1;
    if (z[1] >= nbk) z[1] = (G.bflags & 4u) ? 0 : -1;
    const uint4 m0 = *reinterpret_cast<const uint4*>(nbmask + c * 8);
    const uint4 m1 = *reinterpret_cast<const uint4*>(nbmask + c * 8 + 4);
    const uint32_t m[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
    int n = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int bx = x[q & 1], by = y[(q >> 1) & 1], bz = z[q >> 2];
        if (m[q] != 0u && (bx | by | bz) >= 0) n += __popc(__ldg(&bits[(bz * nbj + by) * nbi + bx]) & m[q]);
    }
    return n;
}

// tile_build_nbmask with a thread per (place, direction): the blocks here are
// short-lived
__device__ __forceinline__ void open_build_masks(uint32_t* mask, int fcc)
{
    const int entries = fcc ? 96 : 32;
    for (int e = threadIdx.x; e < entries * 8; e += blockDim.x) mask[e] = 0u;
    __syncthreads();
    for (int e = threadIdx.x; e < entries * 13; e += blockDim.x) {
        const int c = e / 13, d = e - 13 * c - 1;
        const int x = 4 + (c & 3), y = 4 + ((c >> 2) & 3), z = 2 + ((c >> 4) & 1);
        int dx = 0, dy = 0, dz = 0;
        if (d >= 0) tile_step(d, y, z, fcc ? (c >> 5) : -1, dx, dy, dz);
        const int nx = x + dx, ny = y + dy, nz = z + dz;
        const int q = ((nx >> 2) - ((x - 1) >> 2)) | (((ny >> 2) - ((y - 1) >> 2)) << 1) |
                      (((nz >> 1) - ((z - 1) >> 1)) << 2);
        atomicOr(&mask[c * 8 + q], 1u << ((nx & 3) | ((ny & 3) << 2) | ((nz & 1) << 4)));
    }
    __syncthreads();
}

// target of direction d from (i, j, k); false behind a reflective wall
__device__ __forceinline__ bool open_target(const Geometry& G, const uint8_t* step, int32_t i, int32_t j, int32_t k,
                                            uint32_t d, Nb& nb)
{
    const uint32_t o = step[walk_class(G, j, k) * 12 + (int)d];
    nb.i = i + (int32_t)(o & 3u) - 1;
    nb.j = j + (int32_t)((o >> 2) & 3u) - 1;
    nb.k = k + (int32_t)(o >> 4) - 1;
    nb.wrap = 0ull;
    if ((uint32_t)nb.i < (uint32_t)G.ni && (uint32_t)nb.j < (uint32_t)G.nj && (uint32_t)nb.k < (uint32_t)G.nk) {
        nb.t = nb.i + G.ni * (nb.j + G.nj * nb.k);
        return true;
    }
    return neighbor(G, i, j, k, (int)d, nb);
}

// the block's stretch of the n list entries, a multiple of its threads long
__device__ __forceinline__ void open_range(int n, int& lo, int& hi)
{
    const int rows = (n + (int)blockDim.x - 1) / (int)blockDim.x;
    lo = (int)((int64_t)rows * blockIdx.x / gridDim.x) * (int)blockDim.x;
    hi = min(n, (int)((int64_t)rows * (blockIdx.x + 1) / gridDim.x) * (int)blockDim.x);
}

template <bool HASH>
__global__ void __launch_bounds__(256, 6) k_open_claim(const EventArgs a)
{
    __shared__ __align__(16) uint32_t s_mask[96 * 8];
    __shared__ uint8_t s_step[kWalkSteps];
    const Geometry& G = a.geo;
    walk_steps(G, s_step);
    open_build_masks(s_mask, (G.bflags & 8u) ? 1 : 0);
    if (blockIdx.x == 0 && threadIdx.x < kMaxSpecies) a.sc->tmp_count[threadIdx.x] = 0;
    const uint32_t g = event_index(a), c2 = ((uint32_t)a.s << 4) | kTagEvent;
    const int n = *a.count;
    int lo, hi;
    open_range(n, lo, hi);
    unsigned n_att = 0;
    uint32_t v1 = 0u, id1 = 0u;                                 // the next row's entry, on its way
    if (lo + (int)threadIdx.x < hi) {
        v1 = (uint32_t)a.list.vox[lo + threadIdx.x];
        id1 = a.list.ids[lo + threadIdx.x];
    }
    for (int idx = lo + threadIdx.x; idx < hi; idx += blockDim.x) {
        const uint32_t v = v1, id = id1;
        if (idx + (int)blockDim.x < hi) {
            v1 = (uint32_t)a.list.vox[idx + blockDim.x];
            id1 = a.list.ids[idx + blockDim.x];
        }
        const uint32_t d = walk_draw(a.key0, a.key1, id, g, c2);
        int32_t i, j, k;
        decode(G, v, i, j, k);
        Nb nb;
        uint8_t out = kDecNone;
        if (open_target(G, s_step, i, j, k, d, nb)) {
            if (open_count(G, a.bits, s_mask, nb.i, nb.j, nb.k) == 1) {
                out = (uint8_t)(kDecOpen | d);
            } else {
                const BitPos b = bitpos(G, nb.i, nb.j, nb.k);
                if (!(__ldg(&a.bits[b.word]) & b.mask)) {
                    claim<HASH>(a, nb, id);
                    out = (uint8_t)d;
                }
            }
        }
        a.dec[idx] = out;
        ++n_att;
    }
    if (a.collect_stats) flush_stat(&a.sc->stats[kStatAttempts], n_att);
}

template <bool HASH>
__global__ void __launch_bounds__(256, 6) k_open_commit(const EventArgs a)
{
    __shared__ uint8_t s_step[kWalkSteps];
    const Geometry& G = a.geo;
    walk_steps(G, s_step);
    __syncthreads();
    const int n = *a.count;
    int lo, hi;
    open_range(n, lo, hi);
    if (HASH) {
        // empty the table of the previous event for the next one
        for (uint32_t x = blockIdx.x * blockDim.x + threadIdx.x; x < a.ct.clear_n; x += gridDim.x * blockDim.x)
            a.ct.clear[x] = kEmptySlot;
    }
    unsigned n_hop = 0;
    constexpr int A = 2;                                        // rows on their way
    uint32_t dn[A], vn[A];
#pragma unroll
    for (int u = 0; u < A; ++u) {
        const int x = lo + u * (int)blockDim.x + (int)threadIdx.x;
        dn[u] = x < hi ? a.dec[x] : (uint32_t)kDecNone;
        vn[u] = x < hi ? (uint32_t)a.list.vox[x] : 0u;
    }
    for (int idx = lo + threadIdx.x; idx < hi; idx += blockDim.x) {
        const uint32_t dec = dn[0], v = vn[0];
#pragma unroll
        for (int u = 0; u + 1 < A; ++u) {
            dn[u] = dn[u + 1];
            vn[u] = vn[u + 1];
        }
        const int x = idx + A * (int)blockDim.x;
        dn[A - 1] = x < hi ? a.dec[x] : (uint32_t)kDecNone;
        vn[A - 1] = x < hi ? (uint32_t)a.list.vox[x] : 0u;
        if (dec == kDecNone) continue;
        int32_t i, j, k;
        decode(G, v, i, j, k);
        Nb nb;
        open_target(G, s_step, i, j, k, dec & 15u, nb);
        if (!(dec & kDecOpen) && !won<HASH>(a, nb, a.list.ids[idx])) continue;
        bit_move(a.bits, bitpos(G, i, j, k), bitpos(G, nb.i, nb.j, nb.k));
        if (a.live) {
            a.occ[nb.t] = (uint16_t)(a.s + 1);
            a.occ[v] = 0;
        }
        a.list.vox[idx] = nb.t;
        if (nb.wrap) a.list.img[idx] = img_add(a.list.img[idx], nb.wrap);
        ++n_hop;
    }
    if (a.collect_stats) flush_stat(&a.sc->stats[kStatHops], n_hop);
}

// Blocks for n entries: one to eight rows of 256 each, so that the longest
// lists fill several waves and the shortest every SM (a wave is six blocks per
// SM; 1.34M walkers on 512^3 44 us per event with four rows, 48 with two; 10.7M on
// 1024^3 331 with eight, 348 with sixteen).
static int open_blocks(int64_t n, int sm_count)
{
    const int64_t rows = (n + 255) / 256;
    const int64_t per = std::max<int64_t>(1, std::min<int64_t>(8, rows / (8 * (int64_t)sm_count)));
    return (int)std::max<int64_t>(1, (rows + per - 1) / per);
}

void launch_open_claim(const EventArgs& a, int64_t n, int sm_count, cudaStream_t st)
{
    const int blocks = open_blocks(n, sm_count);
    if (a.ct.hash) k_open_claim<true><<<blocks, 256, 0, st>>>(a);
    else k_open_claim<false><<<blocks, 256, 0, st>>>(a);
}

void launch_open_commit(const EventArgs& a, int64_t n, int sm_count, cudaStream_t st)
{
    const int blocks = open_blocks(n, sm_count);
    if (a.ct.hash) k_open_commit<true><<<blocks, 256, 0, st>>>(a);
    else k_open_commit<false><<<blocks, 256, 0, st>>>(a);
}
