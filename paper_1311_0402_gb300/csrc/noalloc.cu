// noalloc.cu -- dpd_forces_static: the pair force of a small system computed
// without any device allocation, for callers that cannot allocate device
// memory themselves (a host application that hands the library memory it
// manages in its own pool, code running inside another framework's memory
// budget, or a caller in a context where cudaMalloc is not allowed).
//
// Every call uses one file-scope scratch array in device global memory
// (kScratchBytes, fixed at compile time; every GPU that loads the library
// holds it until the process exits).  Its device address is looked up once
// per device with cudaGetSymbolAddress, on the first call made on that
// device (so that first call must come before any stream capture), and is
// passed to the kernels.  Calls share the array: two calls whose kernels
// overlap on the GPU (different streams, or different host threads on the
// same device without ordering) race on it and give wrong results.
#include "dpd.h"
#include "dpd_internal.cuh"
#include "dpd_math.cuh"

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <string>

namespace {

using namespace dpd;

constexpr int kNAMaxParticles = 131072;
constexpr int kNAMaxCells = 65536;
constexpr int kNAThreads = 256;
constexpr int kNAForceThreads = 128;

// scratch layout (byte offsets, 256-aligned)
constexpr size_t kOffPos = 0;                                           // float4 [max particles]
constexpr size_t kOffVel = kOffPos + 16 * (size_t)kNAMaxParticles;      // float4 [max particles]
constexpr size_t kOffIdx = kOffVel + 16 * (size_t)kNAMaxParticles;      // u32 [max particles]
constexpr size_t kOffKey = kOffIdx + 4 * (size_t)kNAMaxParticles;       // u32 [max particles]
constexpr size_t kOffSlot = kOffKey + 4 * (size_t)kNAMaxParticles;      // u32 [max particles]
constexpr size_t kOffFill = kOffSlot + 4 * (size_t)kNAMaxParticles;     // u32 [max particles]
constexpr size_t kOffCount = kOffFill + 4 * (size_t)kNAMaxParticles;    // u32 [max cells]
constexpr size_t kOffStart = kOffCount + 4 * (size_t)kNAMaxCells;       // u32 [max cells + 1]
constexpr size_t kOffTile = kOffStart + 4 * ((size_t)kNAMaxCells + 64);   // u32 [max cells]
constexpr size_t kOffTotal = kOffTile + 4 * (size_t)kNAMaxCells;        // u32 [scan tiles]
constexpr size_t kScratchBytes = kOffTotal + 256;

static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

struct NAParams {
    int n;
    int nc[3];
    int ncell;
    float L[3], halfL[3], cells_per_len[3];
    float rc2, inv_rc, gamma, sigma_isdt, s;
    int s_mode;
    int n_species;
    float a[kMaxSpecies * kMaxSpecies];
    int body_mode;
    float body[3];
    uint32_t key[4];
    uint32_t step;
};

struct NAScratch {
    float4 *pos, *vel;  // the particles cell by cell, each cell in index order (vel.w: signature)
    uint32_t *idx;      // their caller indices
    uint32_t *key;      // cell of each particle
    uint32_t *slot;     // its arrival slot in the cell
    uint32_t *fill;     // cell members in arrival order
    uint32_t *count;    // particles of each cell
    uint32_t *start;    // [ncell + 1] first particle of each cell
    uint32_t *tile;     // the same counted from the cell's scan tile
    uint32_t *total;    // sums of the scan tiles
};

__device__ __forceinline__ int na_cell_axis(float x, float cpl, int nc)
{
    int c = (int)(x * cpl);
    return c < 0 ? 0 : (c >= nc ? nc - 1 : c);
}

__device__ __forceinline__ uint32_t na_cell(const NAParams &P, float4 p)
{
    const int cx = na_cell_axis(p.x, P.cells_per_len[0], P.nc[0]);
    const int cy = na_cell_axis(p.y, P.cells_per_len[1], P.nc[1]);
    const int cz = na_cell_axis(p.z, P.cells_per_len[2], P.nc[2]);
    return (uint32_t)((cz * P.nc[1] + cy) * P.nc[0] + cx);
}

__global__ void k_na_clear(NAParams P, NAScratch S)
{
    dependency_wait();
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < P.ncell; c += gridDim.x * blockDim.x) S.count[c] = 0u;
}

__global__ void k_na_bin(NAParams P, NAScratch S, const float4 *pos)
{
    dependency_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.n) return;
    const uint32_t c = na_cell(P, pos[i]);
    S.key[i] = c;
    S.slot[i] = atomicAdd(&S.count[c], 1u);
}

// Exclusive scan of the counts inside tiles of 2048 cells (at most 32 of
// them), and the tiles' sums; na_start() adds the sums before a tile.
constexpr int kNATile = 2048;
constexpr int kNAScanThreads = 512;

__global__ void __launch_bounds__(kNAScanThreads) k_na_scan(NAParams P, NAScratch S)
{
    __shared__ uint32_t ws[kNAScanThreads / 32];
    dependency_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int base = blockIdx.x * kNATile + threadIdx.x * 4;
    uint32_t v[4], t = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const uint32_t x = base + k < P.ncell ? S.count[base + k] : 0u;
        v[k] = t;
        t += x;
    }
    uint32_t incl = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    const uint32_t w = lane < kNAScanThreads / 32 ? ws[lane] : 0u;
    const uint32_t off = __reduce_add_sync(0xFFFFFFFFu, lane < warp ? w : 0u) + incl - t;
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if (base + k < P.ncell) S.tile[base + k] = off + v[k];
    if (threadIdx.x == kNAScanThreads - 1) S.total[blockIdx.x] = off + t;
}

// Offsets of the scan tiles, into shared memory (called by whole blocks).
__device__ __forceinline__ void na_tiles(const NAParams &P, const NAScratch &S, uint32_t *s_tile)
{
    if (threadIdx.x < 32) {
        const uint32_t t = (int)threadIdx.x * kNATile < P.ncell ? S.total[threadIdx.x] : 0u;
        uint32_t incl = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
            if ((int)threadIdx.x >= o) incl += y;
        }
        s_tile[threadIdx.x] = incl - t;
    }
    __syncthreads();
}

__device__ __forceinline__ uint32_t na_start(const NAParams &P, const NAScratch &S, const uint32_t *s_tile, uint32_t c)
{
    return c < (uint32_t)P.ncell ? S.tile[c] + s_tile[c / kNATile] : (uint32_t)P.n;
}

__global__ void __launch_bounds__(kNAThreads) k_na_fill(NAParams P, NAScratch S)
{
    __shared__ uint32_t s_tile[32];
    dependency_wait();
    na_tiles(P, S, s_tile);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < P.n) S.fill[na_start(P, S, s_tile, S.key[i]) + S.slot[i]] = (uint32_t)i;
}

// Each particle's place in its cell is the number of members with a smaller
// index, so every cell is in index order whatever order the atomics filled it
// in, and the force sums run in a fixed order.  One thread per particle reads
// its own cell once: no thread does more than the cell's occupancy in work.
__global__ void __launch_bounds__(kNAThreads) k_na_place(NAParams P, NAScratch S, const float4 *pos, const float4 *vel,
                                                         const uint32_t *tag)
{
    __shared__ uint32_t s_tile[32];
    dependency_wait();
    na_tiles(P, S, s_tile);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i <= P.ncell) S.start[i] = na_start(P, S, s_tile, (uint32_t)i);
    if (i >= P.n) return;
    const float4 x = pos[i], v = vel[i];
    const uint32_t tg = tag ? tag[i] : (uint32_t)i;
    const uint32_t c = S.key[i];
    const uint32_t b = na_start(P, S, s_tile, c), e = na_start(P, S, s_tile, c + 1);
    uint32_t r = b;
    for (uint32_t q = b; q < e; ++q) r += S.fill[q] < (uint32_t)i ? 1u : 0u;
    S.pos[r] = x;
    S.vel[r] = make_float4(v.x, v.y, v.z, __uint_as_float(signature(tg, P.step, P.key)));
    S.idx[r] = (uint32_t)i;
}

// All of the above for a small system in one launch: every block bins all
// particles into its own shared memory (counts, starts, members), then places
// its share of them, so that no block waits for another and the signatures and
// stores are spread over the blocks.
constexpr int kNASortThreads = 1024;
constexpr int kNASortPer = 4;
constexpr int kNASortMax = kNASortThreads * kNASortPer;  // particles, and cells, it takes
constexpr int kNASortShare = 256;                        // particles a block places

__global__ void __launch_bounds__(kNASortThreads) k_na_sort_small(NAParams P, NAScratch S, const float4 *pos,
                                                                  const float4 *vel, const uint32_t *tag)
{
    __shared__ uint32_t s_start[kNASortMax + 1];
    __shared__ uint16_t s_fill[kNASortMax];
    __shared__ uint32_t ws[32];
    static_assert(kNASortMax <= 65536, "members are 16-bit");
    dependency_wait();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // the particle this thread places
    const int mine = blockIdx.x * kNASortShare + tid;
    const bool places = tid < kNASortShare && mine < P.n;
    float4 x, u;
    uint32_t tg = (uint32_t)mine;
    if (places) {
        x = pos[mine];
        u = vel[mine];
        if (tag) tg = tag[mine];
    }
    for (int c = tid; c < P.ncell; c += kNASortThreads) s_start[c] = 0u;
    __syncthreads();
    uint32_t cell[kNASortPer], slot[kNASortPer];
#pragma unroll
    for (int k = 0; k < kNASortPer; ++k) {
        const int i = k * kNASortThreads + tid;
        cell[k] = i < P.n ? na_cell(P, pos[i]) : 0u;
    }
#pragma unroll
    for (int k = 0; k < kNASortPer; ++k)
        if (k * kNASortThreads + tid < P.n) slot[k] = atomicAdd(&s_start[cell[k]], 1u);
    __syncthreads();
    const int per = (P.ncell + kNASortThreads - 1) / kNASortThreads;  // thread tid owns cells [tid per, tid per + per)
    uint32_t v[kNASortPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kNASortPer; ++k) {
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
    for (int k = 0; k < kNASortPer; ++k) {
        const int c = tid * per + k;
        if (k < per && c < P.ncell) {
            s_start[c] = run;
            if (blockIdx.x == 0) S.start[c] = run;
            run += v[k];
        }
    }
    if (tid == 0) {
        s_start[P.ncell] = (uint32_t)P.n;
        if (blockIdx.x == 0) S.start[P.ncell] = (uint32_t)P.n;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kNASortPer; ++k)
        if (k * kNASortThreads + tid < P.n) s_fill[s_start[cell[k]] + slot[k]] = (uint16_t)(k * kNASortThreads + tid);
    __syncthreads();
    if (!places) return;
    const uint32_t c = na_cell(P, x);
    const uint32_t b = s_start[c], e = s_start[c + 1];
    uint32_t r = b;
    for (uint32_t q = b; q < e; ++q) r += s_fill[q] < mine ? 1u : 0u;
    S.pos[r] = x;
    S.vel[r] = make_float4(u.x, u.y, u.z, __uint_as_float(signature(tg, P.step, P.key)));
    S.idx[r] = (uint32_t)mine;
}

// Pair force of Eqs. 2-9 for each particle over the particles of its 27
// surrounding cells (cells of side >= r_c), FP32 predicate d^2 < r_c^2.  T
// lanes share a particle: its nine rows of cells along x are dealt to them in
// turn, and their sums are added in a fixed order.  The cells of a row are
// consecutive, so a lane walks a few index ranges of the sorted particles.
// Testing a candidate takes some 15 instructions, evaluating a pair 150, and
// one in six candidates is a pair: a lane therefore only notes its pairs in
// shared memory while it walks, and the warp evaluates them together, each lane
// its own in the order found, when a lane's notes run out.  131,000 particles:
// 181 us when every lane evaluated a pair as it met it, 46 now (idle lanes:
// pairs per lane vary between the lanes of a warp, and loads of starts and
// partners); 3,000 particles, where T = 8 spreads the work: 94 to 11 us (ncu,
// cold caches).
constexpr int kNANotes = 24;  // pairs a lane notes
constexpr int kNABurst = 4;   // candidates between looks at the notes

template <int T>
struct NAWarp {
    uint2 range[2 * ((9 + T - 1) / T)][32];
    uint32_t note[kNANotes][32];
};

template <int SMODE, int T, bool WRAP>
__device__ __forceinline__ void na_walk(const NAParams &P, const NAScratch &S, uint32_t p, bool valid,
                                        int sub, NAWarp<T> &w, float &fx, float &fy, float &fz, bool &bad)
{
    const int lane = threadIdx.x & 31;
    const float4 pi = S.pos[valid ? p : 0u], vi = S.vel[valid ? p : 0u];
    const uint32_t si = __float_as_uint(vi.w);
    const int ti = __float_as_int(pi.w);
    // a species outside 0..n_species-1 (in this particle or a partner within
    // r_c) makes the force NaN; the parameter table is never read with it
    bad = (unsigned)ti >= (unsigned)P.n_species;
    const int cx = na_cell_axis(pi.x, P.cells_per_len[0], P.nc[0]);
    const int cy = na_cell_axis(pi.y, P.cells_per_len[1], P.nc[1]);
    const int cz = na_cell_axis(pi.z, P.cells_per_len[2], P.nc[2]);
    // distinct neighbour cells per axis: {-1, 0, 1}, {0, 1} or {0}; a row is cut
    // in two where it crosses the boundary
    const int ny = min(P.nc[1], 3), nz = min(P.nc[2], 3), rows = ny * nz;
    int x0 = P.nc[0] >= 3 ? cx - 1 : (P.nc[0] == 2 ? cx : 0);
    const int nx = min(P.nc[0], 3);
    if (x0 < 0) x0 += P.nc[0];
    const int n1 = min(nx, P.nc[0] - x0);  // cells up to the boundary; nx - n1 from cell 0 on
    // this lane's index ranges: rows sub, sub + T, ... in order
    int nr = 0;
    if (valid) {
#pragma unroll
        for (int k = 0; k < (9 + T - 1) / T; ++k) {
            const int row = sub + k * T;
            if (row < rows) {
                int y = cy + row % ny - (P.nc[1] >= 3 ? 1 : 0), z = cz + row / ny - (P.nc[2] >= 3 ? 1 : 0);
                y = y < 0 ? y + P.nc[1] : (y >= P.nc[1] ? y - P.nc[1] : y);
                z = z < 0 ? z + P.nc[2] : (z >= P.nc[2] ? z - P.nc[2] : z);
                const uint32_t base = (uint32_t)((z * P.nc[1] + y) * P.nc[0]);
                const uint32_t b0 = S.start[base + (uint32_t)x0], e0 = S.start[base + (uint32_t)(x0 + n1)];
                if (e0 > b0) w.range[nr++][lane] = make_uint2(b0, e0);
                if (n1 < nx) {
                    const uint32_t b1 = S.start[base], e1 = S.start[base + (uint32_t)(nx - n1)];
                    if (e1 > b1) w.range[nr++][lane] = make_uint2(b1, e1);
                }
            }
        }
    }
    auto delta = [&](float4 pj) {
        if (WRAP)
            return make_float3(min_image_rn(pj.x, pi.x, P.L[0], P.halfL[0]), min_image_rn(pj.y, pi.y, P.L[1], P.halfL[1]),
                               min_image_rn(pj.z, pi.z, P.L[2], P.halfL[2]));
        return make_float3(__fsub_rn(pj.x, pi.x), __fsub_rn(pj.y, pi.y), __fsub_rn(pj.z, pi.z));
    };
    int noted = 0, r = 0;
    uint2 range = make_uint2(0u, 0u);
    if (r < nr) range = w.range[r++][lane];
    for (;;) {
        const bool more = __any_sync(0xFFFFFFFFu, range.x < range.y);
        if (more) {
            // kNABurst candidates of the range, their loads in flight together
            float4 pj[kNABurst];
#pragma unroll
            for (int u = 0; u < kNABurst; ++u) pj[u] = S.pos[min(range.x + (uint32_t)u, (uint32_t)P.n - 1u)];
#pragma unroll
            for (int u = 0; u < kNABurst; ++u) {
                const float3 d = delta(pj[u]);
                const float d2 = dist2_rn(d.x, d.y, d.z);
                const uint32_t q = range.x + (uint32_t)u;
                if ((q < range.y) & (d2 < P.rc2) & (d2 > 0.0f) & (q != p)) w.note[noted++][lane] = q;
            }
            range.x += kNABurst;
            if (range.x >= range.y && r < nr) range = w.range[r++][lane];
            if (!__any_sync(0xFFFFFFFFu, noted > kNANotes - kNABurst)) continue;
        }
        const int most = __reduce_max_sync(0xFFFFFFFFu, noted);
        uint32_t j = noted > 0 ? w.note[0][lane] : 0u;
        float4 xj = S.pos[j], vj = S.vel[j];
        for (int k = 0; k < most; ++k) {
            const float4 xk = xj, vk = vj;
            if (k + 1 < noted) {
                j = w.note[k + 1][lane];
                xj = S.pos[j];
                vj = S.vel[j];
            }
            if (k < noted) {
                const float3 d = delta(xk);
                const float d2 = dist2_rn(d.x, d.y, d.z);
                const float inv_r = rsqrtf(d2);
                const float rr = d2 * inv_r;
                const float wg = fmaxf(fmaf(-rr, P.inv_rc, 1.0f), 0.0f);
                const float wR = weight_R<SMODE>(wg, P.s);
                const float ev = -((d.x * (vi.x - vk.x) + d.y * (vi.y - vk.y)) + d.z * (vi.z - vk.z)) * inv_r;
                uint32_t A, B;
                pair_hash(si, __float_as_uint(vk.w), P.key, A, B);
                const float xi = gauss_from_hash(A, B);
                const int tj = __float_as_int(xk.w);
                bad |= (unsigned)tj >= (unsigned)P.n_species;
                const float a = bad ? 0.0f : P.a[ti * P.n_species + tj];
                const float F = fmaf(a, wg, fmaf(-P.gamma * wR * wR, ev, P.sigma_isdt * wR * xi));
                const float sc = -F * inv_r;
                fx = fmaf(sc, d.x, fx);
                fy = fmaf(sc, d.y, fy);
                fz = fmaf(sc, d.z, fz);
            }
        }
        if (!more) return;
        noted = 0;
    }
}

template <int SMODE, int T>
__global__ void __launch_bounds__(kNAForceThreads) k_na_force(NAParams P, NAScratch S, float4 *fout)
{
    __shared__ NAWarp<T> s_warp[kNAForceThreads / 32];
    // (no launch_dependents: what the caller launches next starts afterwards)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const uint32_t p = (uint32_t)(t / T);
    const int sub = t % T;
    const bool valid = p < (uint32_t)P.n;
    const float4 pi = S.pos[valid ? p : 0u];
    // a warp whose cells all lie inside a grid of >= 5 cells per axis meets no
    // periodic image, and d = x_j - x_i is the minimum image already
    const int cx = na_cell_axis(pi.x, P.cells_per_len[0], P.nc[0]);
    const int cy = na_cell_axis(pi.y, P.cells_per_len[1], P.nc[1]);
    const int cz = na_cell_axis(pi.z, P.cells_per_len[2], P.nc[2]);
    const bool inner = P.nc[0] >= 5 && P.nc[1] >= 5 && P.nc[2] >= 5 && cx >= 1 && cx <= P.nc[0] - 2 && cy >= 1 &&
                       cy <= P.nc[1] - 2 && cz >= 1 && cz <= P.nc[2] - 2;
    float fx = 0.f, fy = 0.f, fz = 0.f;
    bool bad = false;
    NAWarp<T> &w = s_warp[threadIdx.x >> 5];
    if (__all_sync(0xFFFFFFFFu, inner || !valid))
        na_walk<SMODE, T, false>(P, S, p, valid, sub, w, fx, fy, fz, bad);
    else
        na_walk<SMODE, T, true>(P, S, p, valid, sub, w, fx, fy, fz, bad);
#pragma unroll
    for (int o = 1; o < T; o <<= 1) {
        fx += __shfl_xor_sync(0xFFFFFFFFu, fx, o);
        fy += __shfl_xor_sync(0xFFFFFFFFu, fy, o);
        fz += __shfl_xor_sync(0xFFFFFFFFu, fz, o);
        bad |= __shfl_xor_sync(0xFFFFFFFFu, (int)bad, o) != 0;
    }
    if (!valid || sub != 0) return;
    if (P.body_mode == 1) {
        fx += P.body[0]; fy += P.body[1]; fz += P.body[2];
    } else if (P.body_mode == 2) {
        const float sg = pi.y < P.halfL[1] ? 1.0f : -1.0f;
        fx = fmaf(sg, P.body[0], fx); fy = fmaf(sg, P.body[1], fy); fz = fmaf(sg, P.body[2], fz);
    }
    if (bad) fx = fy = fz = __int_as_float(0x7FC00000);  // quiet NaN
    fout[S.idx[p]] = make_float4(fx, fy, fz, 0.0f);
}

// Lanes per particle: 8 up to kNALanes8 particles, 4 up to kNALanes4, else 2.
// us per call with 8 / 4 / 2 / 1 lanes: 240 particles 14.5 / 16.5 / 20.5 /
// 30.8; 17,496 32.4 / 36.1 / 44.7 / 60.4; 36,501 42.6 / 37.2 / 45.6 / 61.5;
// 65,856 59.0 / 48.0 / 46.3 / 62.7; 129,150 94.2 / 73.3 / 62.9 / 64.7.
constexpr int kNALanes8 = 20000, kNALanes4 = 50000;

template <int T>
cudaError_t na_force(const NAParams &P, const NAScratch &S, float4 *f, cudaStream_t s)
{
    const int g = (P.n * T + kNAForceThreads - 1) / kNAForceThreads;
    switch (P.s_mode) {
    case 1: return launch_kernel(k_na_force<1, T>, g, kNAForceThreads, 0, s, true, P, S, f);
    case 2: return launch_kernel(k_na_force<2, T>, g, kNAForceThreads, 0, s, true, P, S, f);
    case 3: return launch_kernel(k_na_force<3, T>, g, kNAForceThreads, 0, s, true, P, S, f);
    default: return launch_kernel(k_na_force<0, T>, g, kNAForceThreads, 0, s, true, P, S, f);
    }
}

constexpr int kMaxDevices = 64;
std::mutex g_na_mutex;
void *g_na_addr[kMaxDevices] = {};
thread_local std::string g_na_err;

dpd_status na_fail(dpd_status st, const std::string &m)
{
    g_na_err = m;
    return st;
}

}  // namespace

extern "C" {

const char *dpd_forces_static_last_error(void) { return g_na_err.c_str(); }

int64_t dpd_forces_static_max_particles(void) { return kNAMaxParticles; }

dpd_status dpd_forces_static(const dpd_static_params *prm, int64_t n, const float *pos, const float *vel,
                             const uint32_t *tag, uint64_t step, float *force_out, void *stream)
{
    if (!prm || !pos || !vel || !force_out) return na_fail(DPD_ERR_ARG, "params, pos, vel and force_out are required");
    if (n < 1 || n > kNAMaxParticles)
        return na_fail(DPD_ERR_ARG, "n = " + std::to_string(n) + " is outside 1.." + std::to_string(kNAMaxParticles) +
                                        " (the size of the static scratch of dpd_forces_static)");
    if (prm->n_species < 1 || prm->n_species > kMaxSpecies) return na_fail(DPD_ERR_ARG, "n_species must be in 1..8");
    if (!(prm->rc > 0) || !(prm->dt > 0) || !(prm->gamma >= 0) || !(prm->kT >= 0) || !(prm->s > 0))
        return na_fail(DPD_ERR_ARG, "need rc > 0, dt > 0, gamma >= 0, kT >= 0, s > 0");
    if (prm->body_force_mode < 0 || prm->body_force_mode > 2) return na_fail(DPD_ERR_ARG, "body_force_mode in 0..2");
    NAParams P;
    std::memset(&P, 0, sizeof(P));
    P.n = (int)n;
    int64_t ncell = 1;
    for (int a = 0; a < 3; ++a) {
        double L = prm->box[a];
        if (!(L > 2.0 * prm->rc) || !std::isfinite(L)) return na_fail(DPD_ERR_ARG, "each box length must exceed 2 rc");
        int nc = (int)std::floor(L / (prm->rc * (1.0 + 1e-4)));
        P.nc[a] = nc < 1 ? 1 : nc;
        ncell *= P.nc[a];
        P.L[a] = (float)L;
        P.halfL[a] = 0.5f * P.L[a];
        P.cells_per_len[a] = (float)(P.nc[a] / L);
        P.body[a] = (float)prm->body_force[a];
    }
    if (ncell > kNAMaxCells)
        return na_fail(DPD_ERR_ARG, "the box needs " + std::to_string(ncell) + " cells, more than the " +
                                        std::to_string(kNAMaxCells) + " of the static scratch");
    for (int i = 0; i < prm->n_species; ++i)
        for (int j = 0; j < prm->n_species; ++j) {
            double x = prm->a_ij[i * prm->n_species + j];
            if (!std::isfinite(x) || x != prm->a_ij[j * prm->n_species + i])
                return na_fail(DPD_ERR_ARG, "a_ij must be finite and symmetric");
            P.a[i * prm->n_species + j] = (float)x;
        }
    P.ncell = (int)ncell;
    const float rcf = (float)prm->rc;
    P.rc2 = rcf * rcf;
    P.inv_rc = (float)(1.0 / prm->rc);
    P.gamma = (float)prm->gamma;
    P.sigma_isdt = (float)(std::sqrt(2.0 * prm->gamma * prm->kT) / std::sqrt(prm->dt));
    P.s = (float)prm->s;
    P.s_mode = prm->s == 1.0 ? 1 : (prm->s == 0.5 ? 2 : (prm->s == 2.0 ? 3 : 0));
    P.n_species = prm->n_species;
    P.body_mode = prm->body_force_mode;
    P.key[0] = (uint32_t)(prm->seed & 0xFFFFFFFFull);
    P.key[1] = (uint32_t)(prm->seed >> 32);
    P.key[2] = 0x243F6A88u;
    P.key[3] = 0x85A308D3u;
    P.step = (uint32_t)step;

    // device address of the scratch array, looked up once per device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return na_fail(DPD_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= kMaxDevices) return na_fail(DPD_ERR_ARG, "device ordinal beyond 64");
    void *base = nullptr;
    {
        std::lock_guard<std::mutex> lk(g_na_mutex);
        if (!g_na_addr[dev]) {
            void *p = nullptr;
            e = cudaGetSymbolAddress(&p, g_scratch);
            if (e != cudaSuccess || !p)
                return na_fail(DPD_ERR_CUDA, std::string("cudaGetSymbolAddress(scratch): ") + cudaGetErrorString(e));
            g_na_addr[dev] = p;
        }
        base = g_na_addr[dev];
    }
    unsigned char *b = (unsigned char *)base;
    NAScratch S;
    S.pos = (float4 *)(b + kOffPos);
    S.vel = (float4 *)(b + kOffVel);
    S.idx = (uint32_t *)(b + kOffIdx);
    S.key = (uint32_t *)(b + kOffKey);
    S.slot = (uint32_t *)(b + kOffSlot);
    S.fill = (uint32_t *)(b + kOffFill);
    S.count = (uint32_t *)(b + kOffCount);
    S.start = (uint32_t *)(b + kOffStart);
    S.tile = (uint32_t *)(b + kOffTile);
    S.total = (uint32_t *)(b + kOffTotal);

    cudaStream_t s = (cudaStream_t)stream;
    const float4 *p4 = (const float4 *)pos;
    const float4 *v4 = (const float4 *)vel;
    float4 *f4 = (float4 *)force_out;
    const int gn = (P.n + kNAThreads - 1) / kNAThreads;
    // the first kernel starts when the caller's work before it has finished
    if (P.n <= kNASortMax && P.ncell <= kNASortMax) {
        e = launch_kernel(k_na_sort_small, (P.n + kNASortShare - 1) / kNASortShare, kNASortThreads, 0, s, false, P, S, p4, v4, tag);
    } else {
        e = launch_kernel(k_na_clear, (P.ncell + kNAThreads - 1) / kNAThreads, kNAThreads, 0, s, false, P, S);
        if (e == cudaSuccess) e = launch_kernel(k_na_bin, gn, kNAThreads, 0, s, true, P, S, p4);
        if (e == cudaSuccess)
            e = launch_kernel(k_na_scan, (P.ncell + kNATile - 1) / kNATile, kNAScanThreads, 0, s, true, P, S);
        if (e == cudaSuccess) e = launch_kernel(k_na_fill, gn, kNAThreads, 0, s, true, P, S);
        const int gp = (std::max(P.n, P.ncell + 1) + kNAThreads - 1) / kNAThreads;
        if (e == cudaSuccess) e = launch_kernel(k_na_place, gp, kNAThreads, 0, s, true, P, S, p4, v4, tag);
    }
    if (e == cudaSuccess) {
        e = P.n <= kNALanes8 ? na_force<8>(P, S, f4, s) : (P.n <= kNALanes4 ? na_force<4>(P, S, f4, s) : na_force<2>(P, S, f4, s));
    }
    if (e != cudaSuccess) return na_fail(DPD_ERR_CUDA, std::string("launch: ") + cudaGetErrorString(e));
    return DPD_OK;
}

}  // extern "C"
