// kernels_rebuild.cu -- binning, scan, deterministic reorder and neighbour
// list construction (Secs. 3.2-3.3 of Tang & Karniadakis).
//
// The chain runs inside captured CUDA graphs every step; each kernel first
// reads the device rebuild flag set by the integrator's displacement check
// and returns at once when no rebuild is due, so the graph never changes.
//
//   k_bin      cell of each particle (cells ranked along a Morton curve, the
//              first level of the paper's two-level Morton order) + an
//              arrival slot from a per-cell counter, and a 6-bit Morton key
//              of the particle's sub-cell (the second level)
//   k_scan_*   exclusive scan of the cell counts -> cell_start; its first
//              kernel also flips the live buffer set (nothing between the
//              binning and the scan's end reads which set is live)
//   k_scatter  the in-cell sort keys (sub-cell key, caller index), cell by cell
//   k_place    final position = cell_start + rank of the key inside the cell:
//              independent of the atomics' order, so the particle order and
//              the lists are deterministic; the particle arrays go there, into
//              the other buffer set
//   k_sort_small  all of the above in one launch, for small boxes
//   k_nbuild_brick / k_nbuild
//              packed neighbour lists of groups of 4 to 32 particles, hits
//              compacted by warp ballots as in the paper's builder (Sec. 3.3);
//              the list order depends only on the positions
#include "dpd_internal.cuh"

#include <type_traits>
#include "dpd_math.cuh"
#include "brick.cuh"

namespace dpd {

namespace {

constexpr int kThreads = 256;
constexpr int kScanThreads = 512;
constexpr int kScanPerThread = 4;
constexpr int kScanTile = kScanThreads * kScanPerThread;  // 2048 cells per block
constexpr uint32_t kCellMask = (1u << 26) - 1u;

int grid_for(int n)
{
    int g = (n + kThreads - 1) / kThreads;
    return g < 1 ? 1 : (g > 152 * 8 ? 152 * 8 : g);  // grid-stride beyond 8 blocks per SM (measured faster)
}

__device__ __forceinline__ int cell_axis(float x, float cpl, int nc, float *frac)
{
    float f = x * cpl;
    int c = (int)f;  // x >= 0; NaN converts to 0
    c = c < 0 ? 0 : (c >= nc ? nc - 1 : c);
    *frac = f - (float)c;
    return c;
}

__device__ __forceinline__ uint32_t sub_axis(float frac)
{
    int s = (int)(frac * 4.0f);
    return (uint32_t)(s < 0 ? 0 : (s > 3 ? 3 : s));
}

// Morton interleave of three 2-bit coordinates (x in the lowest bit).
__device__ __forceinline__ uint32_t morton2bit(uint32_t x, uint32_t y, uint32_t z)
{
    return (x & 1u) | ((y & 1u) << 1) | ((z & 1u) << 2) | ((x & 2u) << 2) | ((y & 2u) << 3) | ((z & 2u) << 4);
}

__device__ __forceinline__ uint32_t cell_rank_of(const SimParams &P, const uint32_t *rank_of_cell, float4 p,
                                                 uint32_t *sub)
{
    float fx, fy, fz;
    int cx = cell_axis(p.x, P.cells_per_len[0], P.nc[0], &fx);
    int cy = cell_axis(p.y, P.cells_per_len[1], P.nc[1], &fy);
    int cz = cell_axis(p.z, P.cells_per_len[2], P.nc[2], &fz);
    if (sub) *sub = morton2bit(sub_axis(fx), sub_axis(fy), sub_axis(fz));
    return rank_of_cell[(cz * P.nc[1] + cy) * P.nc[0] + cx];
}

// Rank of cell (x, y, z) along the Morton curve through an nx x ny x nz grid (x
// in the lowest bit): the cells before it, counted from the top down as the
// sizes of the child blocks before its own, clipped to the grid.
__device__ uint32_t morton_rank(const int (&n)[3], int x, int y, int z)
{
    uint32_t r = 0;
    for (int b = 9; b >= 0; --b) {  // at most 1024 cells along an axis
        const int size = 1 << b, k = ((x >> b) & 1) | (((y >> b) & 1) << 1) | (((z >> b) & 1) << 2);
        const int ox = (x >> (b + 1)) << (b + 1), oy = (y >> (b + 1)) << (b + 1), oz = (z >> (b + 1)) << (b + 1);
        for (int c = 0; c < k; ++c) {
            const int ex = min(size, n[0] - ox - (c & 1) * size), ey = min(size, n[1] - oy - ((c >> 1) & 1) * size),
                      ez = min(size, n[2] - oz - (c >> 2) * size);
            if (ex > 0 && ey > 0 && ez > 0) r += (uint32_t)ex * (uint32_t)ey * (uint32_t)ez;
        }
    }
    return r;
}

// The cell tables of a handle, built once: ranks, bricks (an aligned block of
// cells is one interval of ranks, and the bricks follow each other as the cells
// of their own grid do), or, without bricks, each cell's neighbour ranks in
// ascending order, no cell twice where an axis has fewer than three.
__global__ void k_geometry(SimParams P, uint32_t *rank_of_cell, uint32_t *stencil, uint32_t *brick_lo, uint32_t *brick_hi,
                           uint32_t *brick_ord)
{
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < P.ncell; c += gridDim.x * blockDim.x) {
        const int x = c % P.nc[0], y = c / P.nc[0] % P.nc[1], z = c / (P.nc[0] * P.nc[1]);
        const uint32_t r = morton_rank(P.nc, x, y, z);
        rank_of_cell[c] = r;
        if (!P.use_bricks) {
            uint32_t *st = stencil + (size_t)r * kStencil;
            int m = 0;
            for (int o = 0; o < kStencil; ++o) {
                // offsets {-1, 0, 1}, {0, 1} or {0} along each axis
                const int d[3] = {o % 3 - 1, o / 3 % 3 - 1, o / 9 - 1};
                bool use = true;
                for (int a = 0; a < 3; ++a)
                    use = use && (P.nc[a] >= 3 || d[a] == 0 || (P.nc[a] == 2 && d[a] == 1));
                if (!use) continue;
                const uint32_t q = morton_rank(P.nc, (x + d[0] + P.nc[0]) % P.nc[0], (y + d[1] + P.nc[1]) % P.nc[1],
                                               (z + d[2] + P.nc[2]) % P.nc[2]);
                int k = m++;
                for (; k > 0 && st[k - 1] > q; --k) st[k] = st[k - 1];
                st[k] = q;
            }
            for (; m < kStencil; ++m) st[m] = kNone;
        }
    }
    for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < P.nbricks; b += gridDim.x * blockDim.x) {
        const int x = b % P.nb[0], y = b / P.nb[0] % P.nb[1], z = b / (P.nb[0] * P.nb[1]);
        const int ex = min(kBrick, P.nc[0] - x * kBrick), ey = min(kBrick, P.nc[1] - y * kBrick),
                  ez = min(kBrick, P.nc[2] - z * kBrick);
        const uint32_t lo = morton_rank(P.nc, x * kBrick, y * kBrick, z * kBrick);
        brick_lo[b] = lo;
        brick_hi[b] = lo + (uint32_t)(ex * ey * ez) - 1u;
        brick_ord[b] = morton_rank(P.nb, x, y, z);
    }
}

__global__ void k_bin(SimParams P, Ptrs D)
{
    dependency_wait();
    if (!D.ctl->rebuild) return;
    const uint32_t par = D.ctl->parity;
    const float4 *pos = D.pos[par];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += gridDim.x * blockDim.x) {
        uint32_t sub;
        uint32_t c = cell_rank_of(P, D.rank_of_cell, pos[i], &sub);
        D.key[i] = (sub << 26) | c;
        D.slot[i] = atomicAdd(&D.cell_count[c], 1u);
    }
}

// Block-level exclusive scan of up to kScanTile values; returns the total.
__device__ uint32_t block_exclusive_scan(uint32_t (&v)[kScanPerThread], uint32_t *warp_sums)
{
    uint32_t t = 0;
#pragma unroll
    for (int k = 0; k < kScanPerThread; ++k) {
        uint32_t x = v[k];
        v[k] = t;
        t += x;
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t incl = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) warp_sums[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        uint32_t w = lane < (kScanThreads / 32) ? warp_sums[lane] : 0u;
        uint32_t wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xFFFFFFFFu, wi, o);
            if (lane >= o) wi += y;
        }
        if (lane < (kScanThreads / 32)) warp_sums[lane] = wi - w;  // exclusive warp offsets
        if (lane == 31) warp_sums[32] = wi;                        // block total
    }
    __syncthreads();
    uint32_t off = warp_sums[warp] + incl - t;
#pragma unroll
    for (int k = 0; k < kScanPerThread; ++k) v[k] += off;
    uint32_t total = warp_sums[32];
    __syncthreads();
    return total;
}

// The rebuilt order becomes the live one: the kernels that follow read the
// old set as parity ^ 1.  Called by one thread, in a kernel that reads none
// of these words itself.
__device__ __forceinline__ void commit_order(DevCtl *c)
{
    c->parity ^= 1u;
    c->oparity ^= 1u;
    c->since_rebuild = 0u;
    c->nrebuild += 1ull;
    c->max_nnb = 0u;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_blocks(SimParams P, Ptrs D)
{
    dependency_wait();
    if (!D.ctl->rebuild) return;
    __shared__ uint32_t ws[33];
    const int base = blockIdx.x * kScanTile + threadIdx.x * kScanPerThread;
    uint32_t v[kScanPerThread];
#pragma unroll
    for (int k = 0; k < kScanPerThread; ++k) v[k] = (base + k < P.ncell) ? D.cell_count[base + k] : 0u;
    uint32_t total = block_exclusive_scan(v, ws);
#pragma unroll
    for (int k = 0; k < kScanPerThread; ++k)
        if (base + k < P.ncell) D.cell_start[base + k] = v[k];
    if (threadIdx.x == 0) {
        D.scan_part[blockIdx.x] = total;
        if (blockIdx.x == 0) {
            D.cell_start[P.ncell] = (uint32_t)P.n;
            commit_order(D.ctl);
        }
    }
}

// Scans the block totals (one block, loops over tiles of kScanTile).
__global__ void __launch_bounds__(kScanThreads) k_scan_top(int nblocks, Ptrs D)
{
    dependency_wait();
    if (!D.ctl->rebuild) return;
    __shared__ uint32_t ws[33];
    uint32_t carry = 0;
    for (int tile = 0; tile < nblocks; tile += kScanTile) {
        const int base = tile + threadIdx.x * kScanPerThread;
        uint32_t v[kScanPerThread];
#pragma unroll
        for (int k = 0; k < kScanPerThread; ++k) v[k] = (base + k < nblocks) ? D.scan_part[base + k] : 0u;
        uint32_t total = block_exclusive_scan(v, ws);
#pragma unroll
        for (int k = 0; k < kScanPerThread; ++k)
            if (base + k < nblocks) D.scan_part[base + k] = v[k] + carry;
        carry += total;
    }
}

// Adds to each tile the sum of the tiles before it: from the scanned totals
// (SCANNED), or summed here by every block, which up to kScanSelf tiles costs
// less than the launch of k_scan_top.
constexpr int kScanSelf = 1024;
template <bool SCANNED>
__global__ void __launch_bounds__(kScanThreads) k_scan_add(SimParams P, Ptrs D)
{
    dependency_wait();
    if (!D.ctl->rebuild) return;
    const int tile = blockIdx.x + 1;  // the first tile needs no offset
    uint32_t off;
    if (SCANNED) {
        off = D.scan_part[tile];
    } else {
        __shared__ uint32_t ws[kScanThreads / 32];
        uint32_t t = 0;
        for (int k = threadIdx.x; k < tile; k += kScanThreads) t += D.scan_part[k];
        t = __reduce_add_sync(0xFFFFFFFFu, t);
        if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = t;
        __syncthreads();
        off = 0;
        for (int w = 0; w < kScanThreads / 32; ++w) off += ws[w];
    }
    const int base = tile * kScanTile;
#pragma unroll
    for (int k = 0; k < kScanPerThread; ++k) {
        const int c = base + k * kScanThreads + (int)threadIdx.x;
        if (c < P.ncell) D.cell_start[c] += off;
    }
}

__global__ void k_scatter(SimParams P, Ptrs D)
{
    dependency_wait();
    if (!D.ctl->rebuild) return;
    const uint32_t *pid = D.pid[D.ctl->oparity ^ 1u];
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += gridDim.x * blockDim.x) {
        const uint32_t k = D.key[i];
        D.skey[D.cell_start[k & kCellMask] + D.slot[i]] = ((unsigned long long)(k >> 26) << 32) | pid[i];
    }
}

// Particle i of the old set goes to place dst of the new one.  IDENT (reorder
// ablation): it keeps its place, and the order goes to perm.
template <bool LHALF, bool IDENT>
__device__ __forceinline__ void place_particle(const SimParams &P, const Ptrs &D, int i, uint32_t dst, uint32_t id,
                                               uint32_t s, uint32_t t, uint32_t os, uint32_t ot)
{
    if (kChecked && dst >= (uint32_t)P.n) {
        atomicOr(&D.ctl->err, kErrBadIndex);
        return;
    }
    if (IDENT) D.perm[dst] = (uint32_t)i;
    const uint32_t p = IDENT ? (uint32_t)i : dst;
    // the inputs first: the stores may alias them as far as the compiler knows
    const float4 x = D.pos[s][i], v = D.vel[s][i];
    const uint32_t tg = D.tag[os][i];
    float4 u = v;
    if (!LHALF) u = D.vkick[s][i];
    D.pos[t][p] = x;
    D.xref[p] = x;
    D.vel[t][p] = v;
    if (!LHALF) D.vkick[t][p] = u;
    // force[] is not carried: every reader finds it rewritten first
    // (a force evaluation, or the last step of a run)
    D.tag[ot][p] = tg;
    D.pid[ot][p] = id;
    if (P.has_bonds) D.idx_of_pid[id] = p;  // bond partners are found by caller index
}

template <bool LHALF, bool IDENT>
__global__ void k_place(SimParams P, Ptrs D)
{
    dependency_wait();
    if (!D.ctl->rebuild) return;
    const uint32_t t = D.ctl->parity, s = t ^ 1u;
    const uint32_t ot = D.ctl->oparity, os = ot ^ 1u;
    const int lim = P.n > P.ncell ? P.n : P.ncell;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < lim; i += gridDim.x * blockDim.x) {
        if (i < P.n) {
            const uint32_t k = D.key[i], id = D.pid[os][i];
            const uint32_t b = D.cell_start[k & kCellMask], e = D.cell_start[(k & kCellMask) + 1u];
            const unsigned long long my = ((unsigned long long)(k >> 26) << 32) | id;
            uint32_t r = 0;
            for (uint32_t q = b; q < e; ++q) r += (D.skey[q] < my) ? 1u : 0u;
            place_particle<LHALF, IDENT>(P, D, i, b + r, id, s, t, os, ot);
        }
        if (i < P.ncell) D.cell_count[i] = 0u;
    }
}

// Binning, scan and reorder of a small box in one launch in place of five whose
// work is a microsecond each: every block bins all particles into its own shared
// memory (counts, starts and sort keys), then places its share of them, so that
// no block waits for another; the last one to finish flips the live set.  3,000
// particles: 17.7 us per step with the five launches, 15.8 with one block for
// everything (11.7 us a rebuild), 15.2 with the stores spread over 12
// (8.3).  The bounds are what one block holds: eight particles and cells per
// thread.
constexpr int kSortThreads = 1024;
constexpr int kSortPer = 8;
constexpr int kSortMax = kSortThreads * kSortPer;  // particles, and cells, it takes
constexpr int kSortShare = 256;                    // particles a block places

template <bool LHALF, bool IDENT>
__global__ void __launch_bounds__(kSortThreads) k_sort_small(SimParams P, Ptrs D)
{
    dependency_wait();
    DevCtl *ctl = D.ctl;
    if (!ctl->rebuild) return;
    extern __shared__ unsigned long long s_key[];                   // [n]
    uint32_t *s_start = reinterpret_cast<uint32_t *>(s_key + P.n);  // [ncell + 1]: counts, then starts
    __shared__ uint32_t ws[32];
    const uint32_t s = ctl->parity, t = s ^ 1u;
    const uint32_t os = ctl->oparity, ot = os ^ 1u;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int c = tid; c < P.ncell; c += kSortThreads) s_start[c] = 0u;
    __syncthreads();
    uint32_t key[kSortPer], slot[kSortPer], id[kSortPer];
#pragma unroll
    for (int k = 0; k < kSortPer; ++k) {
        const int i = k * kSortThreads + tid;
        if (i < P.n) {
            uint32_t sub;
            const uint32_t c = cell_rank_of(P, D.rank_of_cell, D.pos[s][i], &sub);
            key[k] = (sub << 26) | c;
            id[k] = D.pid[os][i];
            slot[k] = atomicAdd(&s_start[c], 1u);
        }
    }
    __syncthreads();
    // exclusive scan: thread tid owns cells [tid per, tid per + per)
    const int per = (P.ncell + kSortThreads - 1) / kSortThreads;
    uint32_t v[kSortPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kSortPer; ++k) {
        const int c = tid * per + k;
        v[k] = k < per && c < P.ncell ? s_start[c] : 0u;
        sum += v[k];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    const uint32_t w = ws[lane];
    uint32_t run = incl - sum + __reduce_add_sync(0xFFFFFFFFu, lane < warp ? w : 0u);
#pragma unroll
    for (int k = 0; k < kSortPer; ++k) {
        const int c = tid * per + k;
        if (k < per && c < P.ncell) {
            s_start[c] = run;
            if (blockIdx.x == 0) D.cell_start[c] = run;
            run += v[k];
        }
    }
    if (tid == 0) {
        s_start[P.ncell] = (uint32_t)P.n;
        if (blockIdx.x == 0) D.cell_start[P.ncell] = (uint32_t)P.n;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSortPer; ++k)
        if (k * kSortThreads + tid < P.n)
            s_key[s_start[key[k] & kCellMask] + slot[k]] = ((unsigned long long)(key[k] >> 26) << 32) | id[k];
    __syncthreads();
    // this block's share: kSortShare consecutive particles, whose keys are in the
    // registers of kSortShare consecutive threads
    const int lo = blockIdx.x * kSortShare;
#pragma unroll
    for (int k = 0; k < kSortPer; ++k) {
        const int i = k * kSortThreads + tid;
        if (i >= lo && i < lo + kSortShare && i < P.n) {
            const uint32_t c = key[k] & kCellMask;
            const uint32_t b = s_start[c], e = s_start[c + 1];
            const unsigned long long my = ((unsigned long long)(key[k] >> 26) << 32) | id[k];
            uint32_t r = 0;
            for (uint32_t q = b; q < e; ++q) r += (s_key[q] < my) ? 1u : 0u;
            place_particle<LHALF, IDENT>(P, D, i, b + r, id[k], s, t, os, ot);
        }
    }
    // every thread of every block has read the control words by now
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        if (atomicAdd(&ctl->done, 1u) + 1u == gridDim.x) {
            ctl->done = 0u;
            commit_order(ctl);
        }
    }
}

// idx_of_pid of the live order (when bonds are first set)
__global__ void k_index(SimParams P, Ptrs D)
{
    const uint32_t *pid = D.pid[D.ctl->oparity];
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < P.n; p += gridDim.x * blockDim.x) D.idx_of_pid[pid[p]] = (uint32_t)p;
}

// ---------------------------------------------------------------------------
// Neighbour build into packed group lists.  A warp builds one group: lane l
// owns particle first + l and walks its own candidate sequence (the
// particles of its surrounding cells, cell by cell, each cell in index
// order); all lanes take one candidate per iteration in lockstep, and the
// hits of an iteration are compacted with a ballot and appended to the
// group's list in lane order.  The list content and order depend only on the
// positions: deterministic, with no atomics.  In Newton-3 mode a particle
// keeps only partners j > i, and a cell's walk starts past i.

// Append the hits of one lockstep iteration to a group list; returns the
// group's new running total (entries past gcap are counted, not written).
__device__ __forceinline__ uint32_t append_hits(bool hit, uint32_t lane, uint32_t j, uint32_t total,
                                                uint32_t *list, uint32_t gcap)
{
    const uint32_t m = __ballot_sync(0xFFFFFFFFu, hit);
    if (hit) {
        const uint32_t k = total + (uint32_t)__popc(m & ((1u << lane) - 1u));
        if (k < gcap) list[k] = (lane << kOwnerShift) | j;
    }
    return total + (uint32_t)__popc(m);
}

// Group descriptor and overflow flag, written by lane 0.
__device__ __forceinline__ void write_group(const Ptrs &D, const SimParams &P, uint32_t g, uint32_t first,
                                            uint32_t owners, uint32_t total)
{
    const uint32_t ne = total < (uint32_t)P.gcap ? total : (uint32_t)P.gcap;
    D.gdesc[g] = make_uint2(first, owners | (ne << 6));
    if (total > (uint32_t)P.gcap) atomicOr(&D.ctl->err, kErrNbrOverflow);
}

// Builder for grids with fewer than three cells along some axis (no
// bricks): groups are the 32-aligned tiles, candidates come from the
// deduplicated cell stencil in global memory.  NOREORDER (reorder ablation):
// the particles stay in load order, so a cell's members are found through
// the sort permutation and the half-list rule is tested per candidate.
template <bool NOREORDER>
__global__ void k_nbuild(SimParams P, Ptrs D)
{
    dependency_wait();
    if (!D.ctl->rebuild) return;
    const uint32_t par = D.ctl->parity;
    const float4 *__restrict__ pos = D.pos[par];
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t nwarps = gridDim.x * blockDim.x / 32u;
    uint32_t local_max = 0;
    for (uint32_t g = (blockIdx.x * blockDim.x + threadIdx.x) / 32u; g < (uint32_t)P.ngroups; g += nwarps) {
        const uint32_t i = g * kGroup + lane;
        const bool valid = i < (uint32_t)P.n;
        const float4 pi = valid ? pos[i] : make_float4(0.f, 0.f, 0.f, 0.f);
        const uint32_t *st = D.stencil + (size_t)(valid ? cell_rank_of(P, D.rank_of_cell, pi, nullptr) : 0u) * kStencil;
        uint32_t s = valid ? 0u : (uint32_t)kStencil, b = 0, n = 0, e = 0;
        auto next_cell = [&]() {
            while (e >= n && s < (uint32_t)kStencil) {
                const uint32_t cc = st[s++];
                if (cc == kNone) {
                    s = kStencil;
                    break;
                }
                b = D.cell_start[cc];
                n = D.cell_start[cc + 1] - b;
                e = (!NOREORDER && P.newton3 && i >= b) ? i + 1u - b : 0u;
            }
        };
        next_cell();
        uint32_t *list = D.nbr + (size_t)g * P.gcap;
        uint32_t total = 0;
        for (;;) {
            const bool act = e < n;
            if (!__any_sync(0xFFFFFFFFu, act)) break;
            bool hit = false;
            uint32_t j = 0;
            if (act) {
                j = NOREORDER ? D.perm[b + e] : b + e;
                const float4 pj = pos[j];
                const float dx = min_image_rn(pj.x, pi.x, P.L[0], P.halfL[0]);
                const float dy = min_image_rn(pj.y, pi.y, P.L[1], P.halfL[1]);
                const float dz = min_image_rn(pj.z, pi.z, P.L[2], P.halfL[2]);
                hit = (dist2_rn(dx, dy, dz) < P.rlist2) & (P.newton3 ? (!NOREORDER || j > i) : j != i);
                ++e;
                if (e >= n) next_cell();
            }
            total = append_hits(hit, lane, j, total, list, (uint32_t)P.gcap);
        }
        if (lane == 0) {
            const uint32_t owners = (uint32_t)P.n - g * kGroup < 32u ? (uint32_t)P.n - g * kGroup : 32u;
            write_group(D, P, g, g * kGroup, owners, total);
        }
        local_max = total > local_max ? total : local_max;
    }
    if (lane == 0 && local_max) atomicMax(&D.ctl->max_nnb, local_max);
}

// Brick builder: P.brick_split CTAs per brick (see brick.cuh).  Each stages the
// positions of the brick's halo in shared memory with bulk (TMA) copies;
// their warps take the brick's particles in groups of P.group and build each
// group cell by cell.  For a cell C the warp lays out one candidate
// sequence: C's own particles (index order), then the particles of the
// stencil cells it needs -- in Newton-3 mode those of higher rank than C,
// otherwise all 26 -- and copies it, in chunks, to a per-warp buffer
// (position, index).  The candidates j > i of an owner i at place p of C are
// then exactly the suffix from p + 1 on, because cells are index ranges in
// rank order; full lists take the whole sequence minus i.  For each owner of
// the group in C, all 32 lanes test 32 consecutive candidates per
// iteration, the owner's position broadcast from shared memory, and append
// the hits with a ballot.  No lane diverges and the list order is fixed by
// the positions.  The groups of brick b get the ids lo / P.group + ord(b) onwards,
// where ord is the brick's position in rank order: unique ids with no count
// pass; the ids a brick leaves unused (at most one or two) get empty
// descriptors.  A brick whose halo exceeds the staging buffer reads
// positions from global memory.
constexpr int kBuildThreads = 32 * kBuildWarps;
constexpr int kSlots = 3;               // candidates per lane and chunk, held in registers
constexpr int kChunk = 32 * kSlots;     // chunk of the candidate sequence
// Three candidates per lane and four resident blocks per SM (64 registers,
// no spill): 0.809 against 0.848 ms per rebuild on the 3M fluid with four
// candidates and three blocks (80 registers).  A cell whose sequence needs a
// second chunk interleaves its owners' entries chunk by chunk, which costs the
// pair kernel 1 % (0.311 against 0.308 ms); two candidates per lane cost it
// 2.5 % for a smaller builder gain.
constexpr int kBuildMinBlocks = 4;

template <bool WRAP>
__device__ __forceinline__ bool within_list(const SimParams &P, float4 pj, float4 pi)
{
    float dx, dy, dz;
    if (WRAP) {
        dx = min_image_rn(pj.x, pi.x, P.L[0], P.halfL[0]);
        dy = min_image_rn(pj.y, pi.y, P.L[1], P.halfL[1]);
        dz = min_image_rn(pj.z, pi.z, P.L[2], P.halfL[2]);
    } else {
        dx = __fsub_rn(pj.x, pi.x);
        dy = __fsub_rn(pj.y, pi.y);
        dz = __fsub_rn(pj.z, pi.z);
    }
    return dist2_rn(dx, dy, dz) < P.rlist2;
}

template <bool WRAP>
__device__ __forceinline__ float pair_d2(const SimParams &P, float4 pj, float4 pi)
{
    float dx, dy, dz;
    if (WRAP) {
        dx = min_image_rn(pj.x, pi.x, P.L[0], P.halfL[0]);
        dy = min_image_rn(pj.y, pi.y, P.L[1], P.halfL[1]);
        dz = min_image_rn(pj.z, pi.z, P.L[2], P.halfL[2]);
    } else {
        dx = __fsub_rn(pj.x, pi.x);
        dy = __fsub_rn(pj.y, pi.y);
        dz = __fsub_rn(pj.z, pi.z);
    }
    return dist2_rn(dx, dy, dz);
}

// fn(std::integral_constant<int, m>) with m = ns clamped to [1, M]: the pass
// instantiated for the chunk's number of live slots (never more than the
// candidate registers hold).
template <int M, typename F>
__device__ __forceinline__ void with_slots(uint32_t ns, F &&fn)
{
    if constexpr (M > 1) {
        if (ns < (uint32_t)M) {
            with_slots<M - 1>(ns, fn);
            return;
        }
    }
    fn(std::integral_constant<int, M>{});
}

// Per-warp table of one slot of the candidate sequence: head[l] is the
// sequence entry (cell) whose first candidate falls on lane l.
struct CellSeq {
    uint8_t head[32];
    uint32_t count;    // atomic-append variant: the group's running total
    uint32_t rows[32]; // row layout: each owner's counts, core | skin << 16
};

// Row layout (list_layout 1, the paper's Sec. 3.3): owner io has the row
// nbr[io * cap, io * cap + cap).  A warp works on one owner at a time; the
// pairs inside r_c at build time (core) are appended at the front of the row
// in sequence order, the other pairs inside r_list (skin) at its back in
// reverse order -- the double insertion, one table and two counters -- and
// k_rows_join later moves the skin part behind the core part.  Full lists:
// every pair is listed by both of its particles.
template <bool WRAP, bool STAGED, int NS>
__device__ __forceinline__ void owner_pass_rows(const SimParams &P, const float4 *__restrict__ pos,
                                                const float4 *s_pos, const uint32_t *s_off,
                                                const float4 (&cand)[kSlots], int t, uint32_t g_own, uint32_t p_lo,
                                                uint32_t p_hi, uint32_t c0, uint32_t c1, uint32_t first, uint32_t lane,
                                                uint32_t *nbr, uint32_t cap, uint32_t *rows)
{
    const uint32_t lt = (1u << lane) - 1u;
    for (uint32_t p = p_lo; p < p_hi; ++p) {
        const uint32_t io = g_own + p;
        const float4 pio = STAGED ? s_pos[s_off[t] + p] : pos[io];
        const uint32_t o = io - first;
        uint32_t core = rows[o] & 0xFFFFu, skin = rows[o] >> 16;
        uint32_t *row = nbr + (size_t)io * cap;
#pragma unroll
        for (int sl = 0; sl < NS; ++sl) {
            const uint32_t k = c0 + 32u * sl + lane;
            const uint32_t j = __float_as_uint(cand[sl].w);
            const float d2 = pair_d2<WRAP>(P, cand[sl], pio);
            const bool cand_ok = (k < c1) & (j != io);
            const uint32_t m_core = __ballot_sync(0xFFFFFFFFu, cand_ok & (d2 < P.rc2));
            const uint32_t m_skin = __ballot_sync(0xFFFFFFFFu, cand_ok & (d2 < P.rlist2) & !(d2 < P.rc2));
            if ((m_core >> lane) & 1u) {
                const uint32_t q = core + (uint32_t)__popc(m_core & lt);
                if (q < cap) row[q] = j;
            }
            if ((m_skin >> lane) & 1u) {
                const uint32_t q = skin + (uint32_t)__popc(m_skin & lt);
                if (q < cap) row[cap - 1u - q] = j;
            }
            core += (uint32_t)__popc(m_core);
            skin += (uint32_t)__popc(m_skin);
        }
        __syncwarp();
        if (lane == 0) rows[o] = min(core, 0xFFFFu) | (min(skin, 0xFFFFu) << 16);
        __syncwarp();
    }
}

// One chunk against the owners [p_lo, p_hi) of cell slot t, one at a time over
// the NS live slots, so that an owner's entries stay contiguous in the list.
//
// ATOMIC (an ablation of the paper's Table 2, ballot against atomic
// insertion): every hit takes its slot with an atomic add on the group's
// shared counter instead of a ballot prefix; the list order then varies run
// to run.
template <bool WRAP, bool STAGED, bool HALF, int NS, bool ATOMIC>
__device__ __forceinline__ uint32_t owner_pass(const SimParams &P, const float4 *__restrict__ pos,
                                               const float4 *s_pos, const uint32_t *s_off, const float4 (&cand)[kSlots],
                                               int t, uint32_t g_own, uint32_t p_lo, uint32_t p_hi, uint32_t c0,
                                               uint32_t c1, uint32_t first, uint32_t lane, uint32_t *list,
                                               uint32_t gcap, uint32_t total, uint32_t *count)
{
    const uint32_t lt = (1u << lane) - 1u;
    if constexpr (ATOMIC) {
        for (uint32_t p = p_lo; p < p_hi; ++p) {
            const uint32_t io = g_own + p;
            const float4 pio = STAGED ? s_pos[s_off[t] + p] : pos[io];
            const uint32_t k0 = HALF ? max(p + 1u, c0) : c0;
            const uint32_t entry_owner = (io - first) << kOwnerShift;
#pragma unroll
            for (int sl = 0; sl < NS; ++sl) {
                const uint32_t k = c0 + 32u * sl + lane;
                const uint32_t j = __float_as_uint(cand[sl].w);
                if ((k < c1) & (k >= k0) & within_list<WRAP>(P, cand[sl], pio) & (HALF || j != io)) {
                    const uint32_t q = atomicAdd(count, 1u);
                    if (q < gcap) list[q] = entry_owner | j;
                }
            }
        }
        return total;
    } else {
        const float4 *own = s_pos + s_off[t];
        for (uint32_t p = p_lo; p < p_hi; ++p) {
            const uint32_t io = g_own + p;
            const float4 pio = STAGED ? own[p] : pos[io];
            // every ballot of the pass first (no branches between them, so the
            // tests overlap); the hits stay in predicates for the stores.  The
            // empty places of the last slot lie outside every cutoff.
            bool hit[NS];
            uint32_t m[NS], at = total;
#pragma unroll
            for (int sl = 0; sl < NS; ++sl) {
                hit[sl] = within_list<WRAP>(P, cand[sl], pio) &
                          (HALF ? c0 + 32u * sl + lane > p : __float_as_uint(cand[sl].w) != io);
                m[sl] = __ballot_sync(0xFFFFFFFFu, hit[sl]);
                total += (uint32_t)__popc(m[sl]);
            }
            const uint32_t entry_owner = (io - first) << kOwnerShift;
            if (total <= gcap) {
#pragma unroll
                for (int sl = 0; sl < NS; ++sl) {
                    if (hit[sl]) list[at + (uint32_t)__popc(m[sl] & lt)] = entry_owner | __float_as_uint(cand[sl].w);
                    at += (uint32_t)__popc(m[sl]);
                }
            } else {  // counted, not written past the capacity
#pragma unroll
                for (int sl = 0; sl < NS; ++sl) {
                    const uint32_t q = at + (uint32_t)__popc(m[sl] & lt);
                    if (hit[sl] && q < gcap) list[q] = entry_owner | __float_as_uint(cand[sl].w);
                    at += (uint32_t)__popc(m[sl]);
                }
            }
        }
        return total;
    }
}

// The owners [p_lo, p_hi) (places in cell slot t) of a group whose first
// particle is `first`: their pairs with the candidate sequence, appended to
// the group list; returns the new running total.  A chunk of kChunk
// candidates is held in registers, lane l holding entries c0 + 32 s + l;
// every owner of the cell tests against the same registers (owner_pass).
template <bool WRAP, bool STAGED, bool HALF, bool ATOMIC, bool ROWS = false>
__device__ __forceinline__ uint32_t build_cell(const SimParams &P, const float4 *__restrict__ pos,
                                               const float4 *s_pos, const uint32_t *s_off, const uint32_t *s_gstart,
                                               const uint32_t *s_cnt, CellSeq &w, int t, uint32_t p_lo, uint32_t p_hi,
                                               uint32_t first, uint32_t lane, uint32_t *list, uint32_t gcap,
                                               uint32_t total)
{
    const uint32_t g_own = s_gstart[t], n_own = s_cnt[t];
    // lanes 0..26: stencil cell (dz, dy, dx) = (l / 9, l / 3 % 3, l % 3) - 1;
    // lane 13 is the cell itself
    uint32_t n_use = 0;
    int ts = t;
    if (lane < (uint32_t)kStencil) {
        ts = t + ((int)(lane / 9u) - 1) * (kHalo * kHalo) + ((int)(lane / 3u % 3u) - 1) * kHalo + ((int)(lane % 3u) - 1);
        const uint32_t n = s_cnt[ts];
        const bool use = lane != 13u && (!HALF || s_gstart[ts] > g_own);
        n_use = use ? n : 0u;
    }
    uint32_t incl = n_use;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if ((int)lane >= o) incl += y;
    }
    const uint32_t total_seq = n_own + __shfl_sync(0xFFFFFFFFu, incl, 31);
    // this lane's sequence entry (lanes 0..26): own cell first (lane 13),
    // then the used stencil cells in lane order
    const uint32_t my_start = lane == 13u ? 0u : n_own + incl - n_use;
    const uint32_t my_n = lane == 13u ? n_own : n_use;
    const uint32_t my_g = lane < (uint32_t)kStencil ? s_gstart[ts] : 0u;
    const uint32_t my_o = lane < (uint32_t)kStencil ? s_off[ts] : 0u;
    for (uint32_t c0 = 0; c0 < total_seq; c0 += (uint32_t)kChunk) {
        const uint32_t c1 = min(total_seq, c0 + (uint32_t)kChunk);
        float4 cand[kSlots];
#pragma unroll
        for (int sl = 0; sl < kSlots; ++sl) {
            const uint32_t kb = c0 + 32u * sl;
            cand[sl] = make_float4(1.0e30f, 1.0e30f, 1.0e30f, 0.f);  // outside every cutoff
            if (kb < c1) {
                // the cell of candidate kb + lane: the last cell starting at or
                // below it in this slot, else the cell covering kb
                const bool covers = my_n > 0u && my_start <= kb && kb < my_start + my_n;
                const bool starts = my_n > 0u && my_start > kb && my_start < kb + 32u;
                if (covers) w.head[0] = (uint8_t)lane;
                if (starts) w.head[my_start - kb] = (uint8_t)lane;
                const uint32_t hmask = __reduce_or_sync(0xFFFFFFFFu, starts ? 1u << (my_start - kb) : 0u) | 1u;
                __syncwarp();
                const int h = 31 - __clz(hmask & (0xFFFFFFFFu >> (31u - lane)));
                const int c = w.head[h];
                __syncwarp();
                const uint32_t cs = __shfl_sync(0xFFFFFFFFu, my_start, c);
                const uint32_t cg = __shfl_sync(0xFFFFFFFFu, my_g, c);
                const uint32_t co = __shfl_sync(0xFFFFFFFFu, my_o, c);
                const uint32_t k = kb + lane;
                if (k < c1) {
                    const uint32_t e = k - cs;
                    const uint32_t j = cg + e;
                    float4 pj = STAGED ? s_pos[co + e] : pos[j];
                    pj.w = __uint_as_float(j);
                    cand[sl] = pj;
                }
            }
        }
        const uint32_t ns = (c1 - c0 + 31u) / 32u;  // live slots of this chunk
        if (ROWS) {
            // list = the whole table, gcap = the row capacity
            with_slots<kSlots>(ns, [&](auto m) {
                owner_pass_rows<WRAP, STAGED, decltype(m)::value>(P, pos, s_pos, s_off, cand, t, g_own, p_lo, p_hi, c0,
                                                                  c1, first, lane, list, gcap, w.rows);
            });
            continue;
        }
        with_slots<kSlots>(ns, [&](auto m) {
            total = owner_pass<WRAP, STAGED, HALF, decltype(m)::value, ATOMIC>(P, pos, s_pos, s_off, cand, t, g_own,
                                                                           p_lo, p_hi, c0, c1, first, lane, list, gcap,
                                                                           total, &w.count);
        });
    }
    return total;
}

template <bool ATOMIC, bool ROWS>
__global__ void __launch_bounds__(kBuildThreads, kBuildMinBlocks) k_nbuild_brick(SimParams P, Ptrs D)
{
    // (not releasing the pair kernel early: two handles of 250,000 particles side by
    // side 125 us a step each when it did, 116 now, four of 81,000 95 and 88; one
    // alone 71.2 and 71.2, 36.1 and 36.1)
    dependency_wait_long();
    if (!D.ctl->rebuild) return;
    extern __shared__ float4 s_pos[];  // [P.brick_cap] staged halo positions
    __shared__ uint32_t s_off[kHaloCells + 1];
    __shared__ uint32_t s_gstart[kHaloCells];
    __shared__ uint32_t s_cnt[kHaloCells];
    __shared__ uint32_t s_wsum[kBuildWarps];
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ CellSeq s_seq[kBuildWarps];
    const uint32_t par = D.ctl->parity;
    const float4 *pos = D.pos[par];
    const int b = blockIdx.x / P.brick_split, part = blockIdx.x % P.brick_split;
    const BrickRange br = brick_halo(P, D, b, s_off, s_gstart, s_cnt, s_wsum);
    const uint32_t ord = D.brick_ord[b];
    const uint32_t G = (uint32_t)P.group;
    const uint32_t gbase = br.lo / G + ord, gnext = br.hi / G + ord + 1u;
    const uint32_t nloc = br.hi - br.lo, ngrp = (nloc + G - 1) / G;
    const bool local = s_off[kHaloCells] <= (uint32_t)P.brick_cap;  // halo fits the staging buffer
    bool staged = true;
    if (local) staged = brick_stage_bulk(D, &s_bar, s_pos, pos, nullptr, nullptr, s_off, s_gstart, s_cnt);
    if (!staged) {  // the error word is set; leave no lists behind for the force kernel
        for (uint32_t g = gbase + threadIdx.x; g < gnext; g += blockDim.x) D.gdesc[g] = make_uint2(0u, 0u);
        return;
    }
    const int bx = b % P.nb[0], by = (b / P.nb[0]) % P.nb[1], bz = b / (P.nb[0] * P.nb[1]);
    const uint32_t gcap = (uint32_t)P.gcap;
    const bool grid5 = P.nc[0] >= 5 && P.nc[1] >= 5 && P.nc[2] >= 5;
    const uint32_t lane = threadIdx.x & 31u;
    CellSeq &w = s_seq[threadIdx.x / 32u];
    uint32_t local_max = 0;
    for (uint32_t q = part * kBuildWarps + threadIdx.x / 32u; q < ngrp; q += kBuildWarps * P.brick_split) {
        const uint32_t first = br.lo + q * G;
        const uint32_t owners = min(nloc - q * G, G);
        // halo slot of each lane's cell (the own cells of the brick are at 1..kBrick per axis)
        int t_lane = -1, inner_lane = 1;
        if (lane < owners) {
            const float4 pi = pos[first + lane];
            float f;
            const int cx = cell_axis(pi.x, P.cells_per_len[0], P.nc[0], &f);
            const int cy = cell_axis(pi.y, P.cells_per_len[1], P.nc[1], &f);
            const int cz = cell_axis(pi.z, P.cells_per_len[2], P.nc[2], &f);
            t_lane = brick_halo_slot(cx - bx * kBrick + 1, cy - by * kBrick + 1, cz - bz * kBrick + 1);
            // a cell one layer or more inside a grid of >= 5 cells per axis
            // never sees a periodic image in its stencil
            inner_lane = grid5 && cx >= 1 && cx <= P.nc[0] - 2 && cy >= 1 && cy <= P.nc[1] - 2 && cz >= 1 &&
                         cz <= P.nc[2] - 2;
        }
        uint32_t *list = ROWS ? D.nbr : D.nbr + (size_t)(gbase + q) * gcap;
        uint32_t total = 0;
        if (ATOMIC) {
            if (lane == 0) w.count = 0u;
            __syncwarp();
        }
        if (ROWS) {
            w.rows[lane] = 0u;
            __syncwarp();
        }
        // the group's particles are sorted by cell: take the cells in turn
        for (uint32_t l0 = 0; l0 < owners;) {
            const int t = __shfl_sync(0xFFFFFFFFu, t_lane, (int)l0);
            const uint32_t same = __ballot_sync(0xFFFFFFFFu, t_lane == t);
            const uint32_t run = (uint32_t)__popc(same);  // lanes of this cell (consecutive)
            const bool inner = __shfl_sync(0xFFFFFFFFu, inner_lane, (int)l0) != 0;
            const uint32_t p_lo = first + l0 - s_gstart[t];
            const uint32_t p_hi = p_lo + run;
            if (ROWS) {
                const uint32_t rcap = (uint32_t)P.cap;
                if (!local)
                    build_cell<true, false, false, false, true>(P, pos, s_pos, s_off, s_gstart, s_cnt, w, t, p_lo, p_hi, first, lane, list, rcap, 0u);
                else if (inner)
                    build_cell<false, true, false, false, true>(P, pos, s_pos, s_off, s_gstart, s_cnt, w, t, p_lo, p_hi, first, lane, list, rcap, 0u);
                else
                    build_cell<true, true, false, false, true>(P, pos, s_pos, s_off, s_gstart, s_cnt, w, t, p_lo, p_hi, first, lane, list, rcap, 0u);
            } else if (P.newton3) {
                if (!local)
                    total = build_cell<true, false, true, ATOMIC>(P, pos, s_pos, s_off, s_gstart, s_cnt, w, t, p_lo, p_hi, first, lane, list, gcap, total);
                else if (inner)
                    total = build_cell<false, true, true, ATOMIC>(P, pos, s_pos, s_off, s_gstart, s_cnt, w, t, p_lo, p_hi, first, lane, list, gcap, total);
                else
                    total = build_cell<true, true, true, ATOMIC>(P, pos, s_pos, s_off, s_gstart, s_cnt, w, t, p_lo, p_hi, first, lane, list, gcap, total);
            } else {
                if (!local)
                    total = build_cell<true, false, false, ATOMIC>(P, pos, s_pos, s_off, s_gstart, s_cnt, w, t, p_lo, p_hi, first, lane, list, gcap, total);
                else if (inner)
                    total = build_cell<false, true, false, ATOMIC>(P, pos, s_pos, s_off, s_gstart, s_cnt, w, t, p_lo, p_hi, first, lane, list, gcap, total);
                else
                    total = build_cell<true, true, false, ATOMIC>(P, pos, s_pos, s_off, s_gstart, s_cnt, w, t, p_lo, p_hi, first, lane, list, gcap, total);
            }
            l0 += run;
        }
        if (ATOMIC) {
            __syncwarp();
            total = w.count;
        }
        if (ROWS) {
            // each owner's counts; a row whose two parts do not fit its
            // capacity reports an overflow (the list is rebuilt larger)
            __syncwarp();
            const uint32_t rc = w.rows[lane];
            const uint32_t len = (rc & 0xFFFFu) + (rc >> 16);
            if (lane < owners) {
                D.rowcnt[first + lane] = rc;
                if (len > (uint32_t)P.cap) atomicOr(&D.ctl->err, kErrNbrOverflow);
            }
            total = __reduce_max_sync(0xFFFFFFFFu, lane < owners ? len : 0u);
            __syncwarp();
        } else if (lane == 0) {
            write_group(D, P, gbase + q, first, owners, total);
        }
        local_max = total > local_max ? total : local_max;
    }
    // ids of this brick's range that no group took
    if (part == 0) for (uint32_t g = gbase + ngrp + threadIdx.x; g < gnext; g += blockDim.x) D.gdesc[g] = make_uint2(0u, 0u);
    if (lane == 0 && local_max) atomicMax(&D.ctl->max_nnb, local_max);
}

// Row layout: join the two parts of every row (the paper's NeighborListJoin):
// the skin entries, stored from the row's end backwards, are moved behind the
// core entries in their insertion order, so a row reads core pairs first and
// skin pairs after them.  One thread per row: reverse the skin block in
// place, then copy it down to the end of the core block (copying towards
// lower addresses in increasing order never overwrites an unread entry).
__global__ void k_rows_join(SimParams P, Ptrs D)
{
    dependency_wait();
    if (!D.ctl->rebuild) return;
    const uint32_t cap = (uint32_t)P.cap;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += gridDim.x * blockDim.x) {
        const uint32_t rc = D.rowcnt[i];
        uint32_t core = rc & 0xFFFFu, skin = rc >> 16;
        if (core > cap) core = cap;
        if (skin > cap - core) skin = cap - core;  // overflowed: reported by the builder
        uint32_t *row = D.nbr + (size_t)i * cap;
        for (uint32_t a = cap - skin, b = cap - 1u; a < b; ++a, --b) {
            const uint32_t x = row[a];
            row[a] = row[b];
            row[b] = x;
        }
        for (uint32_t k = 0; k < skin; ++k) row[core + k] = row[cap - skin + k];
        D.rowcnt[i] = core + skin;
    }
}

// Row layout: transpose every 32 x 32 tile of the table in place (the paper's
// local transposition, NeighborListTranspose): rows 32 g .. 32 g + 31 and
// entries 32 c .. 32 c + 31 swap their roles, so that entry k of particle
// 32 g + l ends up at row 32 g + (k mod 32), entry 32 (k div 32) + l, and a
// warp whose lane l walks particle 32 g + l reads each entry index with one
// coalesced load.  One warp per group of 32 rows, over the tiles its
// longest row reaches.
__global__ void k_rows_transpose(SimParams P, Ptrs D)
{
    dependency_wait();
    if (!D.ctl->rebuild) return;
    __shared__ uint32_t tile[kBuildWarps][32][33];
    const uint32_t cap = (uint32_t)P.cap, lane = threadIdx.x & 31u, wl = threadIdx.x / 32u;
    const uint32_t ngroups = ((uint32_t)P.n + 31u) / 32u;
    const uint32_t nwarps = gridDim.x * blockDim.x / 32u;
    for (uint32_t g = (blockIdx.x * blockDim.x + threadIdx.x) / 32u; g < ngroups; g += nwarps) {
        const uint32_t i = g * 32u + lane;
        const uint32_t len = i < (uint32_t)P.n ? D.rowcnt[i] : 0u;
        const uint32_t ntiles = (__reduce_max_sync(0xFFFFFFFFu, len) + 31u) / 32u;
        uint32_t *base = D.nbr + (size_t)g * 32u * cap;
        for (uint32_t c = 0; c < ntiles; ++c) {
#pragma unroll 8
            for (uint32_t r = 0; r < 32u; ++r) tile[wl][r][lane] = base[(size_t)r * cap + 32u * c + lane];
            __syncwarp();
#pragma unroll 8
            for (uint32_t r = 0; r < 32u; ++r) base[(size_t)r * cap + 32u * c + lane] = tile[wl][lane][r];
            __syncwarp();
        }
    }
}

// Failure-detection probe: the bounded mbarrier wait of the brick staging,
// on a transaction that nothing delivers (expect_tx with no copy issued).
// The wait gives up after `polls` polls and the timeout bit is set; no
// asynchronous copy is in flight, so the block exits cleanly.
__global__ void k_wait_probe(Ptrs D, uint32_t polls)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_arrive_expect_tx(&bar, 16u);
    }
    __syncthreads();
    const bool ok = mbar_wait(&bar, 0u, polls);
    if (!__syncthreads_and(ok) && threadIdx.x == 0) atomicOr(&D.ctl->err, kErrTimeout);
}

}  // namespace

cudaError_t launch_wait_probe(const Ptrs &D, uint32_t polls, cudaStream_t s)
{
    k_wait_probe<<<1, 32, 0, s>>>(D, polls);
    return cudaGetLastError();
}

cudaError_t launch_geometry(const SimParams &P, const Ptrs &D, cudaStream_t s)
{
    k_geometry<<<grid_for(P.ncell), kThreads, 0, s>>>(P, (uint32_t *)D.rank_of_cell, (uint32_t *)D.stencil,
                                                      (uint32_t *)D.brick_rank_lo, (uint32_t *)D.brick_rank_hi,
                                                      (uint32_t *)D.brick_ord);
    return cudaGetLastError();
}

int scan_blocks_for(int ncell) { return (ncell + kScanTile - 1) / kScanTile; }

// fn(lambda is 1/2, identity order) as integral constants
template <typename F>
static void with_place(const SimParams &P, F &&fn)
{
    if (P.lambda_half) {
        if (P.no_reorder) fn(std::true_type{}, std::true_type{});
        else fn(std::true_type{}, std::false_type{});
    } else {
        if (P.no_reorder) fn(std::false_type{}, std::true_type{});
        else fn(std::false_type{}, std::false_type{});
    }
}

static size_t sort_smem(int n, int ncell) { return 8 * (size_t)n + 4 * ((size_t)ncell + 1); }

bool sort_fits_block(int64_t n, int ncell) { return n <= kSortMax && ncell <= kSortMax; }

int rebuild_kernels(const SimParams &P, int n_scan_blocks)
{
    const int sort = P.sort_small ? 1 : (n_scan_blocks > kScanSelf ? 6 : (n_scan_blocks > 1 ? 5 : 4));
    return sort + (P.list_layout == 1 ? 3 : 1);
}

cudaError_t init_build_attributes(int max_dyn_smem)
{
    cudaError_t e = cudaFuncSetAttribute(k_nbuild_brick<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dyn_smem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_nbuild_brick<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dyn_smem);
    const int sort_max = (int)sort_smem(kSortMax, kSortMax);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sort_small<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sort_max);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sort_small<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sort_max);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sort_small<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sort_max);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sort_small<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sort_max);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_nbuild_brick<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_dyn_smem);
    return e;
}

cudaError_t launch_index(const SimParams &P, const Ptrs &D, cudaStream_t s)
{
    k_index<<<grid_for(P.n), kThreads, 0, s>>>(P, D);
    return cudaGetLastError();
}

cudaError_t launch_rebuild(const SimParams &P, const Ptrs &D, cudaStream_t s, int n_scan_blocks, bool overlap)
{
    cudaError_t e = cudaSuccess;
    auto go = [&](auto k, int grid, int block, size_t smem, auto... args) {
        if (e == cudaSuccess) e = launch_kernel(k, grid, block, smem, s, overlap, args...);
    };
    const int g = grid_for(P.n);
    if (P.sort_small) {
        with_place(P, [&](auto lh, auto id) {
            go(k_sort_small<decltype(lh)::value, decltype(id)::value>, (P.n + kSortShare - 1) / kSortShare, kSortThreads, sort_smem(P.n, P.ncell), P, D);
        });
    } else {
        go(k_bin, g, kThreads, 0, P, D);
        go(k_scan_blocks, n_scan_blocks, kScanThreads, 0, P, D);
        if (n_scan_blocks > kScanSelf) {
            go(k_scan_top, 1, kScanThreads, 0, n_scan_blocks, D);
            go(k_scan_add<true>, n_scan_blocks - 1, kScanThreads, 0, P, D);
        } else if (n_scan_blocks > 1) {
            go(k_scan_add<false>, n_scan_blocks - 1, kScanThreads, 0, P, D);
        }
        go(k_scatter, g, kThreads, 0, P, D);
        const int gg = grid_for(P.n > P.ncell ? P.n : P.ncell);
        with_place(P, [&](auto lh, auto id) {
            go(k_place<decltype(lh)::value, decltype(id)::value>, gg, kThreads, 0, P, D);
        });
    }
    if (P.use_bricks) {
        const size_t smem = sizeof(float4) * (size_t)P.brick_cap;
        const int gb = P.nbricks * P.brick_split;
        if (P.list_layout == 1) {
            go(k_nbuild_brick<false, true>, gb, kBuildThreads, smem, P, D);
            go(k_rows_join, g, kThreads, 0, P, D);
            go(k_rows_transpose, grid_for((P.n + 31) / 32 * 32), kBuildThreads, 0, P, D);
        } else if (P.list_builder == 1) {
            go(k_nbuild_brick<true, false>, gb, kBuildThreads, smem, P, D);
        } else {
            go(k_nbuild_brick<false, false>, gb, kBuildThreads, smem, P, D);
        }
    } else if (P.no_reorder) {
        go(k_nbuild<true>, g, kThreads, 0, P, D);
    } else {
        go(k_nbuild<false>, g, kThreads, 0, P, D);
    }
    return e;
}

}  // namespace dpd
