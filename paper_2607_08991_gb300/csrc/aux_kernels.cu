// aux_kernels.cu -- weight repacking, token routing (Sec. 3.2, Eq. 13) and the
// percentile threshold selection (Sec. 2, Eq. 3) for sm_103a.
#include <cmath>

#include "common.cuh"
#include "internal.h"

namespace sats {
namespace {

// ------------------------------------------------------------------ repacking
// Wg [H][N] -> wg_t [N][H];  Wu [H][N] -> w_ud[:, 0:H] (transposed);
// Wd [N][H] -> w_ud[:, H:2H] (row copy).  32x32 tiles through shared memory.
constexpr int kTile = 32;

__global__ void transpose_kernel(const uint16_t *__restrict__ src, int rows, int cols,
                                 uint16_t *__restrict__ dst, int dst_stride)
{
    // src [rows][cols] -> dst[c * dst_stride + r]
    __shared__ uint16_t tile[kTile][kTile + 2];
    const int c0 = blockIdx.x * kTile, r0 = blockIdx.y * kTile;
    for (int dy = threadIdx.y; dy < kTile; dy += blockDim.y) {
        const int r = r0 + dy, c = c0 + threadIdx.x;
        if (r < rows && c < cols) tile[dy][threadIdx.x] = src[(size_t)r * cols + c];
    }
    __syncthreads();
    for (int dy = threadIdx.y; dy < kTile; dy += blockDim.y) {
        const int c = c0 + dy, r = r0 + threadIdx.x;
        if (r < rows && c < cols) dst[(size_t)c * dst_stride + r] = tile[threadIdx.x][dy];
    }
}

__global__ void copy_rows_kernel(const uint16_t *__restrict__ src, int rows, int cols,
                                 uint16_t *__restrict__ dst, int dst_stride)
{
    const size_t total = (size_t)rows * cols;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
        const size_t r = i / cols, c = i - r * cols;
        dst[r * dst_stride + c] = src[i];
    }
}

// ------------------------------------------------------------------ routing
// One CTA of 1024 threads.  Pass 1 counts base-path tokens; pass 2 walks the
// batch in tiles of 1024 with a block-wide exclusive scan, placing each token
// at its rank within its group: a stable partition, identical on every run.
constexpr int kRouteThreads = 1024;

__device__ __forceinline__ int route_flag(const int32_t *ids, int b, const uint8_t *lut, int V, int32_t *status)
{
    const int id = ids[b];
    if (id < 0 || id >= V) {
        if (status) atomicOr(status, kStatusBadToken);
        return 1;   // unknown ids take the base path
    }
    return lut[id] ? 1 : 0;
}

__device__ int block_excl_scan(int v, int *warp_tot, int *total)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int w = lane < (int)(blockDim.x >> 5) ? warp_tot[lane] : 0;
        int wi = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int t = __shfl_up_sync(0xffffffffu, wi, o);
            if (lane >= o) wi += t;
        }
        warp_tot[lane] = wi - w;   // exclusive prefix of warp totals
        if (lane == 31) *total = wi;
    }
    __syncthreads();
    const int r = warp_tot[warp] + incl - v;
    __syncthreads();
    return r;
}

__global__ void __launch_bounds__(kRouteThreads) route_kernel(const int32_t *ids, int B, const uint8_t *lut, int V,
                                                              int32_t *perm, int32_t *n_dense, uint8_t *flags,
                                                              int32_t *status)
{
    __shared__ int warp_tot[32];
    __shared__ int total;
    int cnt = 0;
    for (int b = threadIdx.x; b < B; b += kRouteThreads) cnt += route_flag(ids, b, lut, V, nullptr);
    (void)block_excl_scan(cnt, warp_tot, &total);
    const int nd = total;
    __syncthreads();
    int dense_before = 0;
    for (int base = 0; base < B; base += kRouteThreads) {
        const int b = base + threadIdx.x;
        const int f = b < B ? route_flag(ids, b, lut, V, status) : 0;
        const int excl = block_excl_scan(f, warp_tot, &total);
        if (b < B) {
            const int d = dense_before + excl;                 // base-path tokens before b
            perm[f ? d : nd + (b - d)] = b;
            if (flags) flags[b] = (uint8_t)f;
        }
        dense_before += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) *n_dense = nd;
}

// ------------------------------------------------------------------ selection
// The m-th smallest |a_i| for up to kSelRanks ranks m at once, by a radix select on
// the IEEE bit pattern of |a_i| (non-negative floats order as their unsigned bit
// patterns), 11 + 10 + 10 bits.  Level 0 counts the top 11 bits of every value;
// levels 1 and 2 count the next 10 bits of the values that share their leading bits
// with one of the ranks (a slot each; ranks in one bin share its slot).  At each level
// a CTA counts its values in shared memory and adds the non-zero counts to the level's
// histogram; once all CTAs have, every one of them finds every rank's bin by itself (after
// the last level the first CTA alone).  The three levels are one cooperative launch; a CTA whose
// bounded wait for the others runs out records it in *status, and the results are then NaN.
//
// What bounds it: passes over values that sit in L2, and the meetings.  Post-gate
// magnitudes fall into a few dozen of the top bins, so counting them with atomics in
// global memory ran at the rate of one address (263 us per pass over 3.7 M values,
// and 36 us to search 65536 bins with one CTA); level 0 therefore keeps kSelCopies
// histograms per CTA in shared memory, and 2048-bin levels leave the search a few
// microseconds.  All percentiles of a calibration grid share the three passes.
// As three launches, the last CTA of each searching, a whole call took 37 / 45 / 46 / 59 us for
// 39 k / 0.9 M / 3.7 M / 7.3 M values; as one it takes 33 / 35 / 43 / 47 (the kernel 20 us at 3.7 M, of which
// the second and third pass are 2 each and a meeting with the additions before it about 4).
constexpr int kSelBins0 = 2048, kSelBins = 1024, kSelCopies = 4;
constexpr int kSelThreads = 1024, kSelWarps = kSelThreads / 32;

// Workspace of a selection of R ranks; cleared as a whole before it.
struct SelWs {
    int *done;              // [3] CTAs finished per level; the words behind them are the caller's (kSelStatusWord)
    unsigned *hist0;        // [kSelBins0]
    unsigned *hist;         // [2][R][kSelBins] levels 1 and 2
};

__host__ __device__ inline size_t sel_layout(char *base, int R, SelWs *w)
{
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char *p = base + off;
        off += (bytes + 255) & ~(size_t)255;
        return p;
    };
    w->done = reinterpret_cast<int *>(take((kSelResultWord + kSelRanks) * sizeof(int)));
    w->hist0 = reinterpret_cast<unsigned *>(take(kSelBins0 * sizeof(unsigned)));
    w->hist = reinterpret_cast<unsigned *>(take((size_t)2 * R * kSelBins * sizeof(unsigned)));
    return off;
}

// Calls f(bits of |a_i|) for this thread's share of the n values.
template <typename F>
__device__ __forceinline__ void for_each_bits(const float *__restrict__ a, int64_t n, F f)
{
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, T = (int64_t)gridDim.x * blockDim.x;
    int64_t done = 0;
    if ((reinterpret_cast<uintptr_t>(a) & 15u) == 0) {   // 16-byte loads, two in flight
        const uint4 *v = reinterpret_cast<const uint4 *>(a);
        const int64_t nv = n >> 2;
        done = nv << 2;
        for (int64_t i = t; i < nv; i += 2 * T) {
            const uint4 p = v[i];
            const bool two = i + T < nv;
            const uint4 q = two ? v[i + T] : p;
            f(p.x & 0x7fffffffu);
            f(p.y & 0x7fffffffu);
            f(p.z & 0x7fffffffu);
            f(p.w & 0x7fffffffu);
            if (two) {
                f(q.x & 0x7fffffffu);
                f(q.y & 0x7fffffffu);
                f(q.z & 0x7fffffffu);
                f(q.w & 0x7fffffffu);
            }
        }
    }
    for (int64_t i = done + t; i < n; i += T) f(__float_as_uint(a[i]) & 0x7fffffffu);
}

// Sum over the lanes up to this one.
__device__ __forceinline__ long long warp_incl_scan(long long v)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const long long t = __shfl_up_sync(0xffffffffu, v, o);
        if ((int)(threadIdx.x & 31) >= o) v += t;
    }
    return v;
}

// The bin of NBINS counts (in shared memory) that holds the 1-based rank r, and r within it, by one warp: each lane
// sums NBINS / 32 counts, then the lanes share the counts of the lane that the rank falls in.
template <int NBINS>
__device__ __forceinline__ int find_bin(const unsigned *hist, long long r, long long *within)
{
    constexpr int kPer = NBINS / 32;
    const int lane = threadIdx.x & 31;
    long long sum = 0;
#pragma unroll 8
    for (int k = 0; k < kPer; ++k) sum += hist[lane * kPer + ((k + lane) & (kPer - 1))];   // (no two lanes in a bank)
    const long long incl = warp_incl_scan(sum);
    const unsigned at = __ballot_sync(0xffffffffu, incl >= r);
    const int src = at ? __ffs(at) - 1 : 31;   // (1 <= r <= the sum of the counts)
    long long run = __shfl_sync(0xffffffffu, incl - sum, src);
#pragma unroll
    for (int k = 0; k < kPer / 32; ++k) {
        const long long v = hist[src * kPer + 32 * k + lane], in = run + warp_incl_scan(v);
        const unsigned hit = __ballot_sync(0xffffffffu, in >= r);
        if (hit) {
            const int l = __ffs(hit) - 1;
            *within = r - __shfl_sync(0xffffffffu, in - v, l);
            return src * kPer + 32 * k + l;
        }
        run = __shfl_sync(0xffffffffu, in, 31);
    }
    *within = 1;   // not reached
    return NBINS - 1;
}

// Counts that a CTA keeps in shared memory: level 0's copies, or a slot per rank.
__host__ __device__ constexpr int sel_counts(int R)
{
    return kSelCopies * kSelBins0 > R * kSelBins ? kSelCopies * kSelBins0 : R * kSelBins;
}

struct SelRankList {
    long long m[kSelRanks];
};

// This CTA has added its counts of a level.
__device__ __forceinline__ void sel_arrive(int *done)
{
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) atomicAdd(done, 1);
}

// `ctas` CTAs of the (cooperative) grid have; false, and a timeout in *status, if they do not within kWaitLimitNs.
__device__ __forceinline__ bool sel_meet(const int *done, int ctas, int *status, bool *met)
{
    if (threadIdx.x == 0) {
        const unsigned long long t0 = global_ns();
        bool ok = true;
        while (ld_acquire_gpu(done) < ctas)
            if (global_ns() - t0 > kWaitLimitNs) { ok = false; break; }
        if (!ok) atomicOr(status, kStatusTimeout);
        *met = ok;
    }
    __syncthreads();
    return *met;
}

__global__ void __launch_bounds__(kSelThreads) select_kernel(const float *__restrict__ a, int64_t n, int R,
                                                             const SelRankList ranks, char *ws, int ctas, int *status,
                                                             float *__restrict__ t_out)
{
    extern __shared__ __align__(16) unsigned sel_smem[];   // (stored to in 16-byte vectors)
    __shared__ int bins[kSelRanks], slot[kSelRanks], nslots;
    __shared__ long long rest[kSelRanks];        // rank within the bins chosen so far (1-based)
    __shared__ uint32_t prefix[kSelRanks];       // bits chosen so far
    __shared__ bool met;
    SelWs w;
    sel_layout(ws, R, &w);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    unsigned *h = sel_smem;
    uint8_t *map0 = reinterpret_cast<uint8_t *>(h + sel_counts(R));   // [kSelBins0] slot + 1 of level 1, or 0
    uint8_t *map1 = map0 + kSelBins0;                                 // [R][kSelBins] slot + 1 of level 2, or 0
    for (int i = tid; i < (kSelBins0 + R * kSelBins) / 4; i += kSelThreads) reinterpret_cast<uint32_t *>(map0)[i] = 0u;
    if (tid < R) {
        rest[tid] = ranks.m[tid];
        prefix[tid] = 0u;
        slot[tid] = 0;
    }
#pragma unroll
    for (int level = 0; level < 3; ++level) {
        const int nh = level == 0 ? kSelCopies * kSelBins0 : nslots * kSelBins;
        for (int i = tid; i < nh; i += kSelThreads) h[i] = 0u;
        __syncthreads();
        if (level == 0) {
            unsigned *mine = h + (warp % kSelCopies) * kSelBins0;
            for_each_bits(a, n, [&](uint32_t b) { atomicAdd(mine + (b >> 20), 1u); });
        } else {
            for_each_bits(a, n, [&](uint32_t b) {
                const int s0 = map0[b >> 20];
                if (s0 == 0) return;
                if (level == 1) {
                    atomicAdd(h + (s0 - 1) * kSelBins + ((b >> 10) & 1023u), 1u);
                } else {
                    const int s1 = map1[(s0 - 1) * kSelBins + ((b >> 10) & 1023u)];
                    if (s1) atomicAdd(h + (s1 - 1) * kSelBins + (b & 1023u), 1u);
                }
            });
        }
        __syncthreads();
        unsigned *gh = level == 0 ? w.hist0 : w.hist + (size_t)(level - 1) * R * kSelBins;
        if (level == 0) {
            for (int i = tid; i < kSelBins0; i += kSelThreads) {
                unsigned c = 0;
                for (int k = 0; k < kSelCopies; ++k) c += h[k * kSelBins0 + i];
                if (c) atomicAdd(gh + i, c);
            }
        } else {
            for (int i = tid; i < nh; i += kSelThreads)
                if (h[i]) atomicAdd(gh + i, h[i]);
        }
        sel_arrive(w.done + level);
        if (level == 2 && blockIdx.x != 0) return;
        if (!sel_meet(w.done + level, ctas, status, &met)) {
            // (where another CTA gives up, the first one does at the last level)
            if (blockIdx.x == 0 && tid < R) t_out[tid] = __int_as_float(0x7fffffff);
            return;
        }
        // all CTAs' counts (past L1: the other CTAs wrote them)
        for (int i = tid; i < (level == 0 ? kSelBins0 : nh) / 4; i += kSelThreads)
            reinterpret_cast<uint4 *>(h)[i] = __ldcg(reinterpret_cast<const uint4 *>(gh) + i);
        __syncthreads();
        for (int i = warp; i < R; i += kSelWarps) {   // a warp per rank finds its bin
            long long within;
            const int bin = level == 0 ? find_bin<kSelBins0>(h, rest[i], &within)
                                       : find_bin<kSelBins>(h + slot[i] * kSelBins, rest[i], &within);
            if (lane == 0) {
                bins[i] = bin;
                rest[i] = within;
                prefix[i] |= (uint32_t)bin << (20 - 10 * level);
                if (level == 2) t_out[i] = __uint_as_float(prefix[i]);
            }
        }
        if (level == 2) return;
        __syncthreads();
        if (tid == 0) {   // ranks that share a bin share a slot of the next level
            int ns = 0;
            for (int i = 0; i < R; ++i) {
                uint8_t *m = level == 0 ? map0 + bins[i] : map1 + slot[i] * kSelBins + bins[i];
                if (*m == 0) *m = (uint8_t)++ns;
                slot[i] = *m - 1;
            }
            nslots = ns;
        }
        __syncthreads();
    }
}

size_t sel_smem_bytes(int R) { return (size_t)sel_counts(R) * sizeof(unsigned) + kSelBins0 + (size_t)R * kSelBins; }

}  // namespace

cudaError_t launch_pack(const uint16_t *Wg, const uint16_t *Wu, const uint16_t *Wd, int H, int N,
                        uint16_t *wg_t, uint16_t *w_ud, cudaStream_t stream)
{
    const dim3 block(kTile, 8);
    const dim3 grid((N + kTile - 1) / kTile, (H + kTile - 1) / kTile);
    transpose_kernel<<<grid, block, 0, stream>>>(Wg, H, N, wg_t, H);
    transpose_kernel<<<grid, block, 0, stream>>>(Wu, H, N, w_ud, 2 * H);
    copy_rows_kernel<<<1024, 256, 0, stream>>>(Wd, N, H, w_ud + H, 2 * H);
    return cudaGetLastError();
}

// LoRA adapter layout of the fused kernel (one element per thread, grid-stride):
//   blk [ceil(N/8)][8][3r]: neuron j = 8c + i holds B_gate[:, j], B_up[:, j], A_down[j, :]
//   (neurons past N are zero); agu [H][2r]: A_gate[h, :], A_up[h, :]; bd = B_down [r][H].
__global__ void pack_lora_kernel(const uint16_t *__restrict__ Ag, const uint16_t *__restrict__ Bg,
                                 const uint16_t *__restrict__ Au, const uint16_t *__restrict__ Bu,
                                 const uint16_t *__restrict__ Ad, const uint16_t *__restrict__ Bd, int H, int N, int r,
                                 uint16_t *__restrict__ blk, uint16_t *__restrict__ agu, uint16_t *__restrict__ bd)
{
    const size_t nblk = (size_t)((N + 7) / 8) * 8 * 3 * r, nagu = (size_t)H * 2 * r, nbd = (size_t)r * H;
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < nblk + nagu + nbd;
         i += (size_t)gridDim.x * blockDim.x) {
        if (i < nblk) {
            const int j = (int)(i / (3 * r)), e = (int)(i % (3 * r));
            const int part = e / r, q = e % r;
            uint16_t v = 0;
            if (j < N) v = part == 0 ? Bg[(size_t)q * N + j] : (part == 1 ? Bu[(size_t)q * N + j] : Ad[(size_t)j * r + q]);
            blk[i] = v;
        } else if (i < nblk + nagu) {
            const size_t k = i - nblk;
            const int h = (int)(k / (2 * r)), e = (int)(k % (2 * r));
            agu[k] = e < r ? Ag[(size_t)h * r + e] : Au[(size_t)h * r + (e - r)];
        } else {
            const size_t k = i - nblk - nagu;
            bd[k] = Bd[k];
        }
    }
}

cudaError_t launch_pack_lora(const uint16_t *Ag, const uint16_t *Bg, const uint16_t *Au, const uint16_t *Bu,
                             const uint16_t *Ad, const uint16_t *Bd, int H, int N, int r, sats_lora *l,
                             cudaStream_t stream)
{
    pack_lora_kernel<<<1024, 256, 0, stream>>>(Ag, Bg, Au, Bu, Ad, Bd, H, N, r, l->blk, l->agu, l->bd);
    return cudaGetLastError();
}

cudaError_t launch_route(const int32_t *ids, int B, const uint8_t *lut, int V, int32_t *perm, int32_t *n_dense,
                         uint8_t *flags, int32_t *status, cudaStream_t stream)
{
    route_kernel<<<1, kRouteThreads, 0, stream>>>(ids, B, lut, V, perm, n_dense, flags, status);
    return cudaGetLastError();
}

// The library's bounded waits, made to run out: an mbarrier phase that no thread
// completes (the wait every ring of the MLP kernels uses) and a counter in the
// workspace that no CTA raises (the form of the fused kernel's prologue wait).
// Each gives up after kWaitLimitNs and records a timeout in the status word.
__global__ void wait_timeout_kernel(int *ctl)
{
    __shared__ uint64_t bar;
    __shared__ int never;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        never = 0;
        mbar_init_fence();
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    if (!mbar_wait(&bar, 0u, &never)) atomicOr(ctl + kCtlStatus, kStatusTimeout);
    const unsigned long long t0 = global_ns();
    while (ld_acquire_gpu(ctl + kCtlSelftest) == 0) {
        if (global_ns() - t0 > kWaitLimitNs) {
            atomicOr(ctl + kCtlStatus, kStatusTimeout);
            break;
        }
        __nanosleep(256);
    }
}

cudaError_t launch_wait_timeout(int *ctl, cudaStream_t stream)
{
    wait_timeout_kernel<<<1, 32, 0, stream>>>(ctl);
    return cudaGetLastError();
}

// The workspace of one percentile: what sats_select_workspace_bytes has always asked for.
size_t select_ws_bytes() { return (size_t)65536 * sizeof(unsigned) + 256; }

size_t select_multi_ws_bytes(int R)
{
    SelWs w;
    return sel_layout(nullptr, R, &w);
}

// t_dev[i] = the m[i]-th smallest of |a_0 .. a_{n-1}| for R <= kSelRanks ranks in [1, n];
// ws: select_multi_ws_bytes(R) bytes, 16-byte aligned.  A wait that gives up sets kStatusTimeout in *status (device; a
// word of its own, or ws's word kSelStatusWord, which is cleared here).  absent: CTAs that are waited for and do not exist (the
// self-test's; 0).
cudaError_t launch_select(const float *a, int64_t n, const int64_t *m, int R, void *ws, float *t_dev, int *status,
                          cudaStream_t stream, int absent)
{
    if (R < 1 || R > kSelRanks) return cudaErrorInvalidValue;
    SelRankList ranks;
    for (int i = 0; i < kSelRanks; ++i) ranks.m[i] = i < R ? m[i] : 1;
    char *base = static_cast<char *>(ws);
    cudaError_t e = cudaMemsetAsync(base, 0, select_multi_ws_bytes(R), stream);
    if (e != cudaSuccess) return e;
    // one CTA per SM, fewer where a CTA would have less than 4 values a thread
    const int64_t want = (n + 4 * kSelThreads - 1) / (4 * kSelThreads);
    const int sms = fused_grid(kMaxGrid);
    const int grid = (int)(want < sms ? want : sms);
    const size_t smem = sel_smem_bytes(R);
    // (the limit is set to the most that any call needs, so calls never lower it under one another)
    if (smem > 48 * 1024) {
        e = cudaFuncSetAttribute(select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sel_smem_bytes(kSelRanks));
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kSelThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // the CTAs wait for one another
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, select_kernel, a, n, R, ranks, base, grid + absent, status, t_dev);
}

}  // namespace sats
