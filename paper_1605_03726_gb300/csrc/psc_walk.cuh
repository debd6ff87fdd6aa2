// psc_walk.cuh -- stretches of events of lattices without reactions whose
// claim words fit in the L2 cache.  Part of psc_kernels.cu's translation unit.
//
// What bounds it: scattered L2 accesses, about 0.55 per cycle and SM (then the
// instructions of the draw and the neighbour, and for short lists the chain
// of two barriers).  What keeps the accesses at three per molecule and event:
//   - the claim words tell vacancy too.  While these stretches run, the word
//     of a vacant voxel is all ones and that of an occupied one less than any
//     claim to come: a claim is a minimum with (epoch << id bits | id within
//     the species), the epoch one higher in every event.  It leaves an occupied
//     voxel's word alone, so the claim phase reads nothing; in the commit phase
//     a word holds a molecule's claim exactly if the voxel was vacant and the
//     molecule its lowest claimant; and the winner's claim marks the voxel
//     occupied from then on.  So: the claim, one read-back, and on success the
//     word of the voxel left.  (With the vacancy mirror there were seven: a
//     bit read and a claim, the read-back, the word's reset, the mirror's
//     update of one or two words.)
//   - words lie as the mirror's bits do, a brick of 4 x 4 x 2 voxels on one
//     cache line, so that neighbours in a sorted list share lines.
//   - the molecules of every species stay in shared memory, each with one
//     thread, for the whole stretch; lists and mirror are brought up to date
//     at its end.
//   - the next event's directions, which depend on no position, are drawn
//     while the read-backs are on their way.
// Several species may take turns in a stretch; immobile ones are voxels whose
// word is 0.
// Measured (us per event; before: the molecule-list kernel, the tile kernels one
// species at a time): 2621 walkers on 64^3 8.2 -> 3.2, 1.23M (30 %) on 160^3
// 39.2 -> 19.5, 708,000 on FCC 192^3 37.7 -> 15.4, 797,000 on 301 x 251 x 211
// 39.6 -> 17.8, two species of 503,000 and 336,000 among crowders on 256^3
// 69.7 -> 13.2.
// Tried: the words in the shared memory of a cluster, for lattices they fit in
// (2621 walkers on 64^3 the same, 16,000 on 92^3 6.5 against 5.1: minima on another
// SM's memory are slower than L2's).  Claims that return the old value, with losses noted through a map
// from id to list entry instead of the read-back (two accesses): a returning
// atomic takes as long as a claim and a read-back (160^3 at 30 % 22.3 us per
// event against 22.0, 256^3 at 5 % 18.5 against 19.9, 2621 walkers on 64^3 3.4
// against 2.8).

// word[32 w + b] = 0 where bit b of mirror word w is set, all ones elsewhere;
// without a mirror (bits null): 0 where the word is not all ones
__global__ void k_walk_words(uint32_t* word, const uint32_t* bits, uint64_t words)
{
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < words * 32;
         x += (uint64_t)gridDim.x * blockDim.x)
        word[x] = (bits ? (bits[x >> 5] >> (x & 31u)) & 1u : word[x] != kNoClaim) ? 0u : kNoClaim;
}

void launch_walk_words(uint32_t* word, const uint32_t* bits, uint64_t words, int blocks, cudaStream_t st)
{
    k_walk_words<<<blocks, 256, 0, st>>>(word, bits, words);
}

template <bool CLUSTER>
__device__ __forceinline__ bool walk_barrier(const WalkArgs& A)
{
    if (CLUSTER) {
        cluster_barrier();
        return true;
    }
    return grid_barrier(A.barrier, &A.sc->err, A.barrier_timeout_ns, A.barrier_phantom);
}

// coordinates of place p = mirror word << 5 | bit
__device__ __forceinline__ void walk_decode(const WalkArgs& A, uint32_t p, int32_t& i, int32_t& j, int32_t& k)
{
    const uint32_t w = p >> 5;
    const uint32_t bk = fdiv(w, A.div_nbij);
    const uint32_t r = w - bk * A.div_nbij.d;
    const uint32_t bj = fdiv(r, A.div_nbi);
    i = (int32_t)((r - bj * A.div_nbi.d) * 4u + (p & 3u));
    j = (int32_t)(bj * 4u + ((p >> 2) & 3u));
    k = (int32_t)(bk * 2u + ((p >> 4) & 1u));
}

// Steps by class and direction, packed (di + 1) | (dj + 1) << 2 | (dk + 1) << 4.
// Class: HCP (j + k) & 1 | (k & 1) << 1; FCC row parity | (k mod 3) << 1.
constexpr int kWalkSteps = 6 * 12;
__device__ __forceinline__ int walk_class(const Geometry& G, int32_t j, int32_t k)
{
    if (G.bflags & 8u) {
        const int c = k % 3;
        return ((j + (c == 1 ? 1 : 0)) & 1) | (c << 1);
    }
    return ((j + k) & 1) | ((k & 1) << 1);
}
__device__ __forceinline__ void walk_steps(const Geometry& G, uint8_t* step)
{
    for (int x = threadIdx.x; x < kWalkSteps; x += blockDim.x) {
        const int c = x / 12, d = x % 12, p = c & 1, l = c >> 1;        // l: k & 1, or k mod 3
        const uint32_t wi = c_stencil[p];
        const uint32_t wj = c_stencil[(G.bflags & 8u) ? 5 + l : 2 + (l & 1)];
        const uint32_t wk = c_stencil[4];
        step[x] = (uint8_t)(((wi >> (2 * d)) & 3u) | (((wj >> (2 * d)) & 3u) << 2) | (((wk >> (2 * d)) & 3u) << 4));
    }
}

constexpr uint32_t kWalkNone = 0xFFFFFFFFu;     // no target: the hop goes through a reflective wall
constexpr uint32_t kWalkWrap = 0x80000000u;     // the hop crosses a periodic boundary

// place of the target of direction d from place p
__device__ __forceinline__ uint32_t walk_target(const WalkArgs& A, const uint8_t* step, uint32_t p, uint32_t d)
{
    const Geometry& G = A.geo;
    int32_t i, j, k;
    walk_decode(A, p, i, j, k);
    const uint32_t o = step[walk_class(G, j, k) * 12 + (int)d];
    const int32_t ti = i + (int32_t)(o & 3u) - 1, tj = j + (int32_t)((o >> 2) & 3u) - 1,
                  tk = k + (int32_t)(o >> 4) - 1;
    if ((uint32_t)ti < (uint32_t)G.ni && (uint32_t)tj < (uint32_t)G.nj && (uint32_t)tk < (uint32_t)G.nk)
        return small_place(G, ti, tj, tk);
    Nb nb;
    if (!neighbor(G, i, j, k, (int)d, nb)) return kWalkNone;
    return small_place(G, nb.i, nb.j, nb.k) | kWalkWrap;
}

__device__ __forceinline__ uint32_t walk_draw(uint32_t key0, uint32_t key1, uint32_t id, uint32_t g, uint32_t c2)
{
    uint32_t u[4];
    philox(id, g, c2, 0u, key0, key1, u);
    return __umulhi(u[0], 12u);
}

// change of a wrap counter between coordinates a and b of one hop that differ
// by more than one voxel
__device__ __forceinline__ uint64_t walk_wrap(int32_t a, int32_t b, int shift)
{
    return b - a > 1 ? 0xFFFFull << shift : (a - b > 1 ? 1ull << shift : 0ull);
}

template <bool CLUSTER>
__global__ void __launch_bounds__(CLUSTER ? kWalkClusterThreads : kWalkThreads, 1) k_walk_run(const WalkArgs A)
{
    constexpr int NT = CLUSTER ? kWalkClusterThreads : kWalkThreads;
    constexpr int U = 8;                                        // read-backs in flight per thread
    extern __shared__ uint32_t sm[];                            // [place, id, target][slot][thread]
    __shared__ uint8_t s_step[kWalkSteps];
    uint32_t* s_v = sm + threadIdx.x;
    uint32_t* s_id = s_v + A.slots * NT;
    uint32_t* s_t = s_id + A.slots * NT;
    // molecules are dealt out warp by warp over the blocks, so that a short
    // list keeps every SM of the launch busy; the lanes of a warp hold
    // neighbours in list order (space, after a re-sort)
    const int t0 = (((int)threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x) * 32 + ((int)threadIdx.x & 31);
    const int T = (int)gridDim.x * NT;
    for (int q = 0; q < A.n_species; ++q) {
        int m = A.slot0[q];
        for (int idx = t0; idx < A.n[q]; idx += T, ++m) {
            int32_t i, j, k;
            decode(A.geo, (uint32_t)A.list[q].vox[idx], i, j, k);
            s_v[m * NT] = small_place(A.geo, i, j, k);
            s_id[m * NT] = A.list[q].ids[idx];
        }
    }
    walk_steps(A.geo, s_step);
    __syncthreads();
    const Geometry& G = A.geo;
    uint32_t n_hop = 0;
    unsigned long long n_att = 0;
    auto count = [&](int q) { return t0 < A.n[q] ? (A.n[q] - t0 + T - 1) / T : 0; };
    // directions of event e, into the places of the targets
    auto draw = [&](int e) {
        const int q = A.seq[e], mine = count(q);
        for (int m = A.slot0[q]; m < A.slot0[q] + mine; ++m)
            s_t[m * NT] = walk_draw(A.key0, A.key1, s_id[m * NT], A.g + (uint32_t)e, ((uint32_t)A.species[q] << 4) | kTagEvent);
    };
    draw(0);
    for (int e = 0; e < A.n_events; ++e) {
        const int q = A.seq[e], mine = count(q);
        // claims, less the id
        const uint32_t claim0 = ((A.epoch + (uint32_t)e) << A.id_bits) - A.id_lo[q];
        uint32_t* v0 = s_v + A.slot0[q] * NT;
        uint32_t* id0 = s_id + A.slot0[q] * NT;
        uint32_t* tt0 = s_t + A.slot0[q] * NT;
#pragma unroll 2
        for (int m = 0; m < mine; ++m) {
            const uint32_t t = walk_target(A, s_step, v0[m * NT], tt0[m * NT]);
            if (t != kWalkNone) red_min(&A.word[t & ~kWalkWrap], claim0 + id0[m * NT]);
            tt0[m * NT] = t;
        }
        n_att += (unsigned long long)mine;
        if (!walk_barrier<CLUSTER>(A)) return;
        const bool again = e + 1 < A.n_events && A.seq[e + 1] == q;
        for (int m = 0; m < mine; m += U) {
            uint32_t t[U], w[U], id[U], d[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                t[u] = m + u < mine ? tt0[(m + u) * NT] : kWalkNone;
                id[u] = m + u < mine ? id0[(m + u) * NT] : 0u;
                w[u] = 0u;
                if (t[u] != kWalkNone) w[u] = __ldcg(&A.word[t[u] & ~kWalkWrap]);
            }
            if (again) {
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (m + u < mine) d[u] = walk_draw(A.key0, A.key1, id[u], A.g + (uint32_t)e + 1u, ((uint32_t)A.species[q] << 4) | kTagEvent);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (m + u >= mine) continue;
                if (again) tt0[(m + u) * NT] = d[u];
                if (t[u] == kWalkNone || w[u] != claim0 + id[u]) continue;
                const uint32_t v = v0[(m + u) * NT], to = t[u] & ~kWalkWrap;
                A.word[v] = kNoClaim;
                v0[(m + u) * NT] = to;
                ++n_hop;
                if (t[u] & kWalkWrap) {
                    int32_t i, j, k, ti, tj, tk;
                    walk_decode(A, v, i, j, k);
                    walk_decode(A, to, ti, tj, tk);
                    uint64_t* img = &A.list[q].img[t0 + (m + u) * T];
                    *img = img_add(*img, walk_wrap(i, ti, 0) | walk_wrap(j, tj, 16) | walk_wrap(k, tk, 32));
                }
            }
        }
        if (e + 1 < A.n_events) {
            if (!again) draw(e + 1);
            if (!walk_barrier<CLUSTER>(A)) return;
        }
    }
    // the lists, and the mirror: every molecule that moved flips the bits of
    // the voxels it stood on before and after the stretch
    for (int q = 0; q < A.n_species; ++q) {
        int m = A.slot0[q];
        for (int idx = t0; idx < A.n[q]; idx += T, ++m) {
            const uint32_t from = (uint32_t)A.list[q].vox[idx], to = s_v[m * NT];
            int32_t i, j, k;
            walk_decode(A, to, i, j, k);
            const uint32_t v = (uint32_t)(i + G.ni * (j + G.nj * k));
            if (from == v) continue;
            A.list[q].vox[idx] = (int32_t)v;
            decode(G, from, i, j, k);
            const BitPos bf = bitpos(G, i, j, k), bt = small_bit(to);
            if (bf.word == bt.word) {
                atomicXor(&A.bits[bf.word], bf.mask ^ bt.mask);
            } else {
                atomicXor(&A.bits[bf.word], bf.mask);
                atomicXor(&A.bits[bt.word], bt.mask);
            }
        }
    }
    if (A.collect_stats) {
        flush_stat(&A.sc->stats[kStatHops], n_hop);
        flush_stat(&A.sc->stats[kStatAttempts], n_att);
    }
}

void walk_limits(int* cluster, int* smem)
{
    const void* fc = (const void*)k_walk_run<true>;
    const void* fg = (const void*)k_walk_run<false>;
    *cluster = 0;
    *smem = 0;
    int dev = 0, optin = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess)
        return;
    const int room = optin - 1024;
    if (cudaFuncSetAttribute(fg, cudaFuncAttributeMaxDynamicSharedMemorySize, room) == cudaSuccess) *smem = room;
    if (cudaFuncSetAttribute(fc, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        for (int m = 16; m >= 8 && *cluster == 0; m /= 2) {
            cudaLaunchConfig_t cfg{};
            cudaLaunchAttribute at{};
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = (unsigned)m;
            at.val.clusterDim.y = at.val.clusterDim.z = 1;
            cfg.gridDim = dim3(m);
            cfg.blockDim = dim3(kWalkClusterThreads);
            cfg.dynamicSmemBytes = kWalkClusterSmem;
            cfg.attrs = &at;
            cfg.numAttrs = 1;
            int clusters = 0;
            if (cudaOccupancyMaxActiveClusters(&clusters, fc, &cfg) == cudaSuccess && clusters > 0) *cluster = m;
        }
    }
    cudaGetLastError();
}

cudaError_t launch_walk(const WalkArgs& A, int blocks, bool cluster, cudaStream_t st)
{
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at{};
    const int threads = cluster ? kWalkClusterThreads : kWalkThreads;
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
    cfg.dynamicSmemBytes = (size_t)A.slots * threads * 12;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cluster ? cudaLaunchKernelEx(&cfg, k_walk_run<true>, A) : cudaLaunchKernelEx(&cfg, k_walk_run<false>, A);
}
