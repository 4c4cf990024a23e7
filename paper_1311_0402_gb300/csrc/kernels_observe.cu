// kernels_observe.cu -- observables of the live state: kinetic sums and
// the virial (Eq. 3 pressure), binned velocity profiles (Sec. 4.2), and the
// pair random numbers exported for checking (Sec. 3.5).  None of these runs
// inside the stepping graphs.
#include "dpd_internal.cuh"
#include "dpd_math.cuh"

#include <algorithm>

namespace dpd {

namespace {

constexpr int kThreads = 256;

// Compensated FP32 accumulation (FP64 arithmetic is scarce on this part):
// Knuth's TwoSum for each addition, a square as its exact two-term split hi + lo,
// hi = v v rounded, lo = fma(v, v, -hi).  Of the m terms one thread adds, s + c is
// off by at most m^2 2^-48 of the sum of their magnitudes (the bound of Ogita,
// Rump and Oishi).
struct Sum2 {
    float s = 0.0f, c = 0.0f;
    // every operation rounded on its own: a contracted multiply-add would
    // break the error-free transformations
    __device__ __forceinline__ void add(float x)
    {
        const float t = __fadd_rn(s, x);
        const float bp = __fsub_rn(t, s);
        c = __fadd_rn(c, __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(x, bp)));
        s = t;
    }
    __device__ __forceinline__ void add_square(float v)
    {
        const float hi = __fmul_rn(v, v);
        add(hi);
        c = __fadd_rn(c, fmaf(v, v, -hi));
    }
    // by whole warps; a thread that added one term holds it in s alone
    __device__ __forceinline__ double value() const
    {
        const double x = (double)s;
        return __any_sync(0xFFFFFFFFu, c != 0.0f) ? x + (double)c : x;
    }
};

// FP64 sums of four values over the warp, in a fixed order: lane 8 k returns the
// sum of v[k].  Half the lanes hand two of their values over and keep the
// other two, then a quarter one, so a lane makes 6 additions where four separate
// trees make 20: FP64 additions are what limits this (one warp's take 16 cycles
// of an SM).
__device__ __forceinline__ double warp_sum4(const double (&v)[4], int lane)
{
    const bool hi2 = (lane & 16) != 0, hi1 = (lane & 8) != 0;
    const double a = (hi2 ? v[2] : v[0]) + __shfl_xor_sync(0xFFFFFFFFu, hi2 ? v[0] : v[2], 16);
    const double b = (hi2 ? v[3] : v[1]) + __shfl_xor_sync(0xFFFFFFFFu, hi2 ? v[1] : v[3], 16);
    double x = (hi1 ? b : a) + __shfl_xor_sync(0xFFFFFFFFu, hi1 ? a : b, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
    return x;
}

// Observables: sum v^2, sum v (3) over the particles, and the virial sum over
// pairs inside r_c of r_ij . F^C_ij plus the bonds' share (Eq. 3 and Sec. 4.5).
// The virial comes from the force evaluation that closed the last call (a force
// evaluation, or the last step of a run): its positions are the current ones,
// and the pair kernel left one partial per block in vir_part, summed here in a
// fixed order.  Each thread adds its particles as Sum2 (one particle up to
// 155,648 of them); everything above a thread is FP64.  Each block leaves its
// partials in red; the last one to finish adds all of
// them in block order (whichever it is, the order is the same) and stores the
// finished dpd_obs, nine 8-byte words: step, n, kinetic, temperature, virial,
// pressure, momentum[3], with the divisors 3N - 3 and 3V passed in.  One launch
// where there were three: 81,000 particles, a step and its record each time: 91
// to 78 us a step.
constexpr int kSums = 5;  // v^2, v (3), virial
__global__ void __launch_bounds__(kThreads) k_observe(SimParams P, Ptrs D, double dof, double three_v)
{
    __shared__ double sh[kSums][kThreads / 32];
    __shared__ int s_last;
    dependency_wait();
    DevCtl *ctl = D.ctl;
    const float4 *__restrict__ vel = D.vel[ctl->parity];
    Sum2 sums[4];
    double vir = 0.0;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x, first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    for (int64_t i = first; i < P.n; i += stride) {
        const float4 v = vel[i];
        sums[0].add_square(v.x);
        sums[0].add_square(v.y);
        sums[0].add_square(v.z);
        sums[1].add(v.x);
        sums[2].add(v.y);
        sums[3].add(v.z);
    }
    const int64_t nvir = (P.ngroups + kForceWarps - 1) / kForceWarps;
    for (int64_t k = first; k < nvir; k += stride) vir += D.vir_part[k];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto warp_sum = [&](double x) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xFFFFFFFFu, x, o);
        return x;
    };
    // the block's sum of sh[k] over the warps, on thread k
    auto block_sums = [&]() {
        __syncthreads();
        double x = 0.0;
        if (threadIdx.x < kSums)
            for (int w = 0; w < kThreads / 32; ++w) x += sh[threadIdx.x][w];
        __syncthreads();
        return x;
    };
    const double v4[4] = {sums[0].value(), sums[1].value(), sums[2].value(), sums[3].value()};
    const double w4 = warp_sum4(v4, lane);
    if ((lane & 7) == 0) sh[lane >> 3][warp] = w4;
    // most warps hold no virial partial
    if (__any_sync(0xFFFFFFFFu, first < nvir)) vir = warp_sum(vir);
    if (lane == 0) sh[4][warp] = vir;
    const double mine = block_sums();
    if (threadIdx.x < kSums) {
        D.red[(size_t)blockIdx.x * 8 + threadIdx.x] = mine;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&ctl->obs_done, 1u) + 1u == gridDim.x;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (threadIdx.x == 0) ctl->obs_done = 0u;
    double acc[kSums] = {0, 0, 0, 0, 0};
    for (int b = threadIdx.x; b < (int)gridDim.x; b += kThreads)
#pragma unroll
        for (int k = 0; k < kSums; ++k) acc[k] += __ldcg(D.red + (size_t)b * 8 + k);
    const double a4[4] = {acc[0], acc[1], acc[2], acc[3]};
    const double t4 = warp_sum4(a4, lane), t5 = warp_sum(acc[4]);
    if ((lane & 7) == 0) sh[lane >> 3][warp] = t4;
    if (lane == 0) sh[4][warp] = t5;
    const double total = block_sums();
    if (threadIdx.x < kSums) sh[threadIdx.x][0] = total;
    __syncthreads();
    if (threadIdx.x == 0) {
        const double s0 = sh[0][0], virial = sh[4][0];
        auto bits = [](double x) { return (unsigned long long)__double_as_longlong(x); };
        D.obs[0] = ctl->step;
        D.obs[1] = (unsigned long long)P.n;
        D.obs[2] = bits(0.5 * s0);
        D.obs[3] = bits(dof > 0.0 ? s0 / dof : 0.0);
        D.obs[4] = bits(virial);
        D.obs[5] = bits((s0 + virial) / three_v);
        for (int k = 0; k < 3; ++k) D.obs[6 + k] = bits(sh[1 + k][0]);
    }
}

__device__ __forceinline__ float axis_of(float4 x, int axis) { return axis == 0 ? x.x : (axis == 1 ? x.y : x.z); }

__device__ __forceinline__ int profile_bin(float4 x, int axis, float scale, int nbins)
{
    const int b = (int)(axis_of(x, axis) * scale);
    return b < 0 ? 0 : (b >= nbins ? nbins - 1 : b);
}

// Binned profile.  Block b handles the particles [b chunk, (b + 1) chunk), its
// warps in runs of 32: a warp reduces its lanes' velocities bin by bin (the
// cell order puts a run into a few bins) and lane 0 adds them to the warp's own
// table in shared memory, so every partial is summed in a fixed order without
// atomics, each particle read once.  Partials (sum, count): red[b][2 nbins].
// 262,144 particles, 60 bins: 195 us when each thread owned a bin and read the
// whole chunk, 15 us now (ncu, cold caches; the loads' latency), with the blocks' partials
// summed on the device instead of the host: 201 to 46 us per call.
__global__ void k_profile(SimParams P, Ptrs D, int bin_axis, int vel_axis, int nbins, int chunk)
{
    extern __shared__ double s_sum[];  // [warps][nbins], then the counts
    const int W = blockDim.x / 32, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t *s_cnt = reinterpret_cast<uint32_t *>(s_sum + (size_t)W * nbins);
    for (int k = threadIdx.x; k < W * nbins; k += blockDim.x) {
        s_sum[k] = 0.0;
        s_cnt[k] = 0u;
    }
    __syncthreads();
    const uint32_t par = D.ctl->parity;
    const float4 *__restrict__ pos = D.pos[par];
    const float4 *__restrict__ vel = D.vel[par];
    const int b1 = min((int64_t)P.n, ((int64_t)blockIdx.x + 1) * chunk);
    const float scale = (float)nbins / P.L[bin_axis];
    double *sum = s_sum + (size_t)warp * nbins;
    uint32_t *cnt = s_cnt + (size_t)warp * nbins;
    for (int64_t p0 = (int64_t)blockIdx.x * chunk + 32 * warp; p0 < b1; p0 += 32 * W) {
        const int64_t p = p0 + lane;
        const bool valid = p < b1;
        int bin = -1;
        float v = 0.0f;
        if (valid) {
            const float4 x = pos[p], u = vel[p];
            bin = profile_bin(x, bin_axis, scale, nbins);
            v = axis_of(u, vel_axis);
        }
        uint32_t left = __ballot_sync(0xFFFFFFFFu, valid);
        while (left) {
            const int b = __shfl_sync(0xFFFFFFFFu, bin, __ffs(left) - 1);
            const uint32_t same = __ballot_sync(0xFFFFFFFFu, bin == b);
            double x = bin == b ? (double)v : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xFFFFFFFFu, x, o);
            if (lane == 0) {
                sum[b] += x;
                cnt[b] += (uint32_t)__popc(same);
            }
            left &= ~same;
        }
    }
    __syncthreads();
    double *out = D.red + (size_t)blockIdx.x * 2 * nbins;
    for (int bin = threadIdx.x; bin < nbins; bin += blockDim.x) {
        double s = 0.0, c = 0.0;
        for (int w = 0; w < W; ++w) {
            s += s_sum[(size_t)w * nbins + bin];
            c += (double)s_cnt[(size_t)w * nbins + bin];
        }
        out[2 * bin] = s;
        out[2 * bin + 1] = c;
    }
}

// The same for more bins than a warp's table holds: thread t owns bins t,
// t + blockDim, ... and scans the chunk in order.
__global__ void __launch_bounds__(kThreads) k_profile_wide(SimParams P, Ptrs D, int bin_axis, int vel_axis, int nbins,
                                                           int chunk)
{
    const uint32_t par = D.ctl->parity;
    const float4 *pos = D.pos[par];
    const float4 *vel = D.vel[par];
    const int64_t b0 = (int64_t)blockIdx.x * chunk;
    const int64_t b1 = min((int64_t)P.n, b0 + chunk);
    const float scale = (float)nbins / P.L[bin_axis];
    double *out = D.red + (size_t)blockIdx.x * 2 * nbins;
    for (int bin = threadIdx.x; bin < nbins; bin += blockDim.x) {
        double s = 0.0, c = 0.0;
        for (int64_t p = b0; p < b1; ++p) {
            if (profile_bin(pos[p], bin_axis, scale, nbins) == bin) {
                s += axis_of(vel[p], vel_axis);
                c += 1.0;
            }
        }
        out[2 * bin] = s;
        out[2 * bin + 1] = c;
    }
}

// Sum of the blocks' partials, one warp per entry, in a fixed order.
__global__ void __launch_bounds__(kThreads) k_profile_sum(const double *part, int nblocks, int n2, double *out)
{
    const int lane = threadIdx.x & 31, e = (blockIdx.x * kThreads + threadIdx.x) / 32;
    if (e >= n2) return;
    double x = 0.0;
    for (int b = lane; b < nblocks; b += 32) x += part[(size_t)b * n2 + e];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_down_sync(0xFFFFFFFFu, x, o);
    if (lane == 0) out[e] = x;
}

__global__ void k_pair_rng(uint64_t seed, uint32_t step, int64_t m, const uint32_t *ti, const uint32_t *tj,
                           uint32_t *out_hash, float *out_xi)
{
    const uint32_t key[4] = {(uint32_t)(seed & 0xFFFFFFFFull), (uint32_t)(seed >> 32), 0x243F6A88u, 0x85A308D3u};
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < m; k += (int64_t)gridDim.x * blockDim.x) {
        uint32_t si = signature(ti[k], step, key);
        uint32_t sj = signature(tj[k], step, key);
        uint32_t A, B;
        pair_hash(si, sj, key, A, B);
        out_hash[2 * k] = A;
        out_hash[2 * k + 1] = B;
        if (out_xi) out_xi[k] = gauss_from_hash(A, B);
    }
}

}  // namespace

int observe_blocks_for(int n)
{
    const int g = (n + kThreads - 1) / kThreads;
    return g < 1 ? 1 : (g > 152 * 4 ? 152 * 4 : g);  // grid-stride beyond 4 blocks per SM
}

cudaError_t launch_observe(const SimParams &P, const Ptrs &D, double dof, double three_v, cudaStream_t s)
{
    return launch_kernel(k_observe, observe_blocks_for(P.n), kThreads, 0, s, true, P, D, dof, three_v);
}

// Up to this many bins a block of one warp or more has its tables in the 48 KB
// of shared memory every launch may ask for.
constexpr int kProfileBins = 4096;

static int profile_warps(int nbins) { return std::max(1, std::min(8, kProfileBins / nbins)); }

int profile_blocks_for(int64_t n, int nbins)
{
    if (nbins > kProfileBins) return (int)std::min<int64_t>(std::max<int64_t>(1, n / 1024), 1024);
    const int64_t run = 32 * profile_warps(nbins);
    return (int)std::min<int64_t>((n + run - 1) / run, 152 * 2);
}

cudaError_t launch_profile(const SimParams &P, const Ptrs &D, int bin_axis, int vel_axis, int nbins, int nblocks,
                           cudaStream_t s)
{
    const int chunk = (P.n + nblocks - 1) / nblocks;
    if (nbins > kProfileBins) {
        k_profile_wide<<<nblocks, kThreads, 0, s>>>(P, D, bin_axis, vel_axis, nbins, chunk);
    } else {
        const int W = profile_warps(nbins), run = 32 * W;
        k_profile<<<nblocks, 32 * W, (size_t)W * nbins * 12, s>>>(P, D, bin_axis, vel_axis, nbins, (chunk + run - 1) / run * run);
    }
    k_profile_sum<<<(2 * nbins * 32 + kThreads - 1) / kThreads, kThreads, 0, s>>>(D.red, nblocks, 2 * nbins,
                                                                                  D.red + (size_t)nblocks * 2 * nbins);
    return cudaGetLastError();
}

cudaError_t launch_pair_rng(uint64_t seed, uint64_t step, int64_t m, const uint32_t *ti, const uint32_t *tj,
                            uint32_t *out_hash, float *out_xi, cudaStream_t s)
{
    int64_t g = (m + kThreads - 1) / kThreads;
    if (g > 152 * 16) g = 152 * 16;
    if (g < 1) g = 1;
    k_pair_rng<<<(int)g, kThreads, 0, s>>>(seed, (uint32_t)step, m, ti, tj, out_hash, out_xi);
    return cudaGetLastError();
}

}  // namespace dpd
