// tc_common.cuh -- helpers shared by the tensor-core kernels (gemm_tc.cu,
// union_mlp.cu): tcgen05 descriptors and instructions, TMEM access, TMA tile
// loads, and the host side of tensor maps, shared-memory limits and launches
// with programmatic dependent launch.  Included once per translation unit;
// everything is in an unnamed namespace.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <atomic>
#include <cmath>
#include <mutex>
#include <utility>

#include "common.cuh"
#include "internal.h"

namespace sats {
namespace tc {
namespace {

constexpr int BM = 128;              // MMA M: rows of the A operand
constexpr int BK = 64;               // K per TMA box: one 128-byte swizzle row of bf16
constexpr int kThreads = 192;
// Epilogue groups of four warps in the prefill kernels: the last tile's epilogue of the
// persistent gate/up kernel, and every tile's of the down projection, follow their MMAs.
constexpr int kWideGuGroups = 4;     // at most: 128-neuron tiles, two 16-neuron blocks each
constexpr int kWideDownGroups = 4;   // 256 columns: four 16-column blocks each
constexpr int kWideMaxThreads = 64 + 128 * 4;
// Epilogue groups of four warps of the batched-decode gate/up kernel, at most: seven (64 registers a
// thread) take 97-112 and 193-224 tokens in one turn less than six (Llama-shaped layer, 112 bf16 / fp32
// tokens 65.5 / 74.5 -> 63.9 / 73.0 us, 224 tokens 95.0 / 125.2 -> 91.9 / 122.5); elsewhere the seventh only
// costs (hidden 1024 / intermediate 4096, 250 tokens 30.8 -> 31.3).
constexpr int kSkinnyMaxGroups = 7;
constexpr int kSkinnyMaxThreads = 64 + 128 * kSkinnyMaxGroups;  // of the batched-decode gate/up kernel
constexpr int kSmemBudget = 196608;  // stage ring (one CTA per SM)
constexpr int kSmemWide = 225280;    // stage ring of the persistent prefill kernels, at most
constexpr int kMaxStages = 8;
constexpr int kMaxSkinny = 256;      // largest batch on the skinny orientation (MMA N <= 256)
// with fp32 activations (bf16 high and low parts), larger batches run faster on the prefill
// kernels: at hidden 4096 / intermediate 14336, 256 tokens took 135 us skinny and 129 us wide
// (224 tokens: 125 and 126 us); with bf16 activations the skinny kernels stay ahead up to 256
constexpr int kMaxSkinnySplit = 224;
constexpr int kMaxUnion = 8;         // largest batch on the union path (sparse-path tokens only)
constexpr int kTileBytes = BK * 2;   // bytes of one tile row
// The prefill kernels bring their weight stages into L2 this many stages ahead of
// the loads: every weight stage is read by the CTAs of all token tiles at about
// the same time, and a ring of four or five stages does not cover a miss to HBM.
constexpr int kWidePrefetch = 16;

// ---------------------------------------------------------------------- device helpers
// Shared-memory matrix descriptor of a K-major bf16 tile written by TMA with
// 128-byte swizzle: rows of 128 bytes, 8-row atoms 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr)
{
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);     // start address
    d |= (uint64_t)(16u >> 4) << 16;               // leading byte offset (unused for swizzled K-major)
    d |= (uint64_t)(1024u >> 4) << 32;             // stride byte offset: one 8-row atom
    d |= (uint64_t)1 << 46;                        // descriptor version of this architecture
    d |= (uint64_t)2 << 61;                        // 128-byte swizzle
    return d;
}

// Instruction descriptor of kind::f16: bf16 A and B (K-major), fp32 D, M x N.
__host__ __device__ constexpr uint32_t instr_desc(int M, int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// The load and MMA roles are run by whole warps, whose loops and operands are then uniform, and issued by one
// elected lane.  With a role's loop in one lane's branch every address and descriptor had to be moved into uniform
// registers before each instruction: about 100 cycles per MMA, commit or copy, more than the MMAs of a batched-
// decode K block or the eight copies of a prefill stage leave (the same box, us; before -> MMA role -> both roles):
// Llama-shaped layer 8 bf16 tokens 57.5 -> 54.3 -> 53.5 and 2048 (a few calls; in a loop at the power limit about 600
// either way) 610 -> 601 -> 560, hidden 8192 / intermediate 7168
// 8 tokens 75 -> 61 -> 54, hidden 2048 / intermediate 8192 25.4 -> 22.5 -> 20.1.
__device__ __forceinline__ uint32_t elect_one()
{
    uint32_t lead;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(lead));
    return lead;
}

// warp = threadIdx.x / 32, known to be the same in all its lanes.
__device__ __forceinline__ int uniform_warp() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }

// mbar_wait by all lanes of a warp (of one barrier or of one each), with one answer.
__device__ __forceinline__ bool warp_wait(uint64_t *bar, uint32_t parity, volatile int *abort)
{
    const bool ok = __all_sync(0xffffffffu, mbar_wait(bar, parity, abort));
    __syncwarp();
    return ok;
}

__device__ __forceinline__ void mma_bf16_if(uint32_t lead, uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                            uint32_t acc)
{
    asm volatile(
        "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
        "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(lead)
        : "memory");
}

// The mbarrier receives one arrival when all MMAs that the elected lane issued before are done.
__device__ __forceinline__ void mma_commit_if(uint32_t lead, uint64_t *bar)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
                 "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}"
                 ::"r"(smem_addr(bar)), "r"(lead) : "memory");
}

__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols)
{
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(slot)), "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols)
{
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

// 16 consecutive fp32 columns of this warp's 32 TMEM lanes (one row per thread).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16])
{
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// As tmem_ld16, 8 columns.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8])
{
    uint32_t r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Error path only (a role gave up waiting): before the CTA releases its TMEM
// and exits, wait -- again bounded -- for the tile loads still in flight
// (stages issued but never consumed) and for the MMAs already issued.
__device__ void drain_after_abort(uint64_t *full, int stages, int issued, int consumed, uint64_t *acc_full)
{
    int never = 0;
    for (int k = consumed; k < issued; ++k)
        mbar_wait(&full[k % stages], (uint32_t)((k / stages) & 1), &never);
    mbar_wait(acc_full, 0u, &never);
}

// The load role's instructions (lead: whether this lane issues them).
__device__ __forceinline__ void mbar_expect_if(uint32_t lead, uint64_t *bar, uint32_t bytes)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t"
                 "@q mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;\n\t}"
                 ::"r"(smem_addr(bar)), "r"(bytes), "r"(lead) : "memory");
}

__device__ __forceinline__ void bulk_load_if(uint32_t lead, void *dst, const void *src, uint32_t bytes, uint64_t *bar,
                                             uint64_t policy)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
                 "@q cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
                 " [%0], [%1], %2, [%3], %4;\n\t}"
                 ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar)), "l"(policy), "r"(lead)
                 : "memory");
}

__device__ __forceinline__ void bulk_load_shared_if(uint32_t lead, void *dst, const void *src, uint32_t bytes,
                                                    uint64_t *bar)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %4, 0;\n\t"
                 "@q cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n\t}"
                 ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar)), "r"(lead)
                 : "memory");
}

__device__ __forceinline__ void bulk_prefetch_l2_if(uint32_t lead, const void *src, uint32_t bytes)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t"
                 "@q cp.async.bulk.prefetch.L2.global [%0], %1;\n\t}" ::"l"(src), "r"(bytes), "r"(lead) : "memory");
}

// One 2D TMA tile load: inner coordinate c0 (elements, a multiple of 64), row c1.
__device__ __forceinline__ void tma_load_if(uint32_t lead, void *dst, const CUtensorMap *map, int c0, int c1,
                                            uint64_t *bar)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
                 "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%2, %3}], [%4];\n\t}"
                 ::"r"(smem_addr(dst)), "l"(map), "r"(c0), "r"(c1), "r"(smem_addr(bar)), "r"(lead)
                 : "memory");
}

// Starts bringing one TMA box (inner coordinate c0, row c1) of the tensor into L2;
// no completion to wait for.
__device__ __forceinline__ void tma_prefetch_l2_if(uint32_t lead, const CUtensorMap *map, int c0, int c1)
{
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %3, 0;\n\t"
                 "@q cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];\n\t}"
                 ::"l"(map), "r"(c0), "r"(c1), "r"(lead)
                 : "memory");
}

__device__ __forceinline__ uint16_t bf16_bits(float v)
{
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    return *reinterpret_cast<const uint16_t *>(&h);
}

__device__ __forceinline__ uint8_t *align1024(uint8_t *p)
{
    return reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(p) + 1023) & ~(uintptr_t)1023);
}


__device__ __forceinline__ void set_timeout(int *ctl, volatile int *abort_flag)
{
    *abort_flag = 1;
    atomicOr(ctl + kCtlStatus, kStatusTimeout);
}

// ---------------------------------------------------------------------- kept lists
// The ascending kept lists of a batch, from the keep bytes of the gate/up epilogue (0 or 1 per row
// and neuron): row m's list is written as the list of token perm[m] (token m without a permutation).
// The down projections' epilogue warps write them while their first MMAs run.
struct KeepLists {
    const uint8_t *keep;
    int stride;             // a multiple of 16
    int N;
    int32_t *idx;           // [tokens][N], or nullptr: no lists
    int32_t *cnt;           // [tokens] or nullptr
    const int32_t *perm;
};

// Row m, by `threads` (a multiple of 32) threads that share hardware barrier `bar`; t is the thread's
// number among them, warp_sums holds an int per warp.  Thread t takes the 16-byte vectors [t per,
// (t + 1) per) of the row: it counts their kept bytes, a scan gives its first position, and it writes
// its entries in order (two passes over the row, the second from L1/L2).
__device__ __forceinline__ void write_keep_list(const KeepLists &L, int m, int t, int threads, int *warp_sums, int bar)
{
    const int tok = L.perm ? L.perm[m] : m;
    const uint4 *k = reinterpret_cast<const uint4 *>(L.keep + (size_t)m * L.stride);
    const int lane = t & 31, w = t >> 5;
    const int nv = (L.N + 15) >> 4;
    const int per = (nv + threads - 1) / threads;
    const int v0 = min(nv, t * per), v1 = min(nv, v0 + per);
    // the kept bytes of vector v as a 16-bit mask; bytes at or past N are not counted
    auto mask16 = [&](int v) {
        const uint4 q = k[v];
        const uint32_t wq[4] = {q.x, q.y, q.z, q.w};
        uint32_t bits = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            bits |= ((wq[i] & 1u) | ((wq[i] >> 7) & 2u) | ((wq[i] >> 14) & 4u) | ((wq[i] >> 21) & 8u)) << (4 * i);
        const int rest = L.N - 16 * v;
        return rest >= 16 ? bits : bits & ((1u << rest) - 1u);
    };
    int c = 0;
    for (int v = v0; v < v1; ++v) c += __popc(mask16(v));
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
    }
    if (lane == 31) warp_sums[w] = incl;
    named_barrier(bar, threads);
    int pos = incl - c, total = 0;
    for (int i = 0; i < threads >> 5; ++i) {
        if (i < w) pos += warp_sums[i];
        total += warp_sums[i];
    }
    int32_t *out = L.idx + (size_t)tok * L.N;
    for (int v = v0; v < v1; ++v)
        for (uint32_t bits = mask16(v); bits; bits &= bits - 1u) out[pos++] = 16 * v + __ffs(bits) - 1;
    if (t == 0 && L.cnt) L.cnt[tok] = total;
    named_barrier(bar, threads);   // warp_sums may be written again
}

// ---------------------------------------------------------------------- host
PFN_cuTensorMapEncodeTiled_v12000 encode_fn()
{
    static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
    static std::once_flag once;
    std::call_once(once, [] {
        void *ptr = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
                cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
    });
    return fn;
}

// bf16 matrix [rows][cols] with the given row stride (a multiple of 16 bytes),
// read in boxes of box_rows x 64 with 128-byte swizzle.
bool make_map(CUtensorMap *map, const void *base, uint64_t rows, uint64_t cols, uint64_t row_stride_bytes,
              uint32_t box_rows)
{
    auto fn = encode_fn();
    if (!fn) return false;
    const cuuint64_t dims[2] = {cols, rows};
    const cuuint64_t strides[1] = {row_stride_bytes};
    const cuuint32_t box[2] = {(cuuint32_t)BK, box_rows};
    const cuuint32_t es[2] = {1, 1};
    return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, es,
              CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The device's opt-in limit of shared memory per CTA.
int smem_optin()
{
    static int by_dev[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    int &n = by_dev[dev & 63];
    if (n == 0) cudaDeviceGetAttribute(&n, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return n;
}

// Raises the kernel's dynamic shared-memory limit on the current device to at
// least `bytes`; `configured` is the caller's per-device record for this kernel.
template <typename K>
cudaError_t set_smem(K kernel, size_t bytes, std::atomic<int> (&configured)[64])
{
    int dev = 0;
    cudaGetDevice(&dev);
    std::atomic<int> &have = configured[dev & 63];
    if ((int)bytes <= have.load()) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e == cudaSuccess) have.store((int)bytes);
    return e;
}

// Launch with programmatic dependent launch: the kernel may start while the
// preceding kernel in the stream finishes; it calls griddepcontrol.wait before
// touching anything that kernel produces.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, size_t smem, cudaStream_t stream, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// As launch_pdl, for the small kernels (no dynamic shared memory, `threads` per CTA).
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl_threads(void (*kernel)(KArgs...), dim3 grid, int threads, cudaStream_t stream, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// As launch_pdl, with `threads` per CTA and `smem` bytes of dynamic shared memory; overlap: whether to start
// before the preceding kernel has ended.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl_if(bool overlap, void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem,
                          cudaStream_t stream, Args &&...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl_cfg(void (*kernel)(KArgs...), dim3 grid, int threads, size_t smem, cudaStream_t stream,
                           Args &&...args)
{
    return launch_pdl_if(true, kernel, grid, threads, smem, stream, std::forward<Args>(args)...);
}

// Dynamic shared memory of a launch: the stage ring, 1 KB of alignment slack and the barriers.
size_t smem_for(int stages, int stage_bytes) { return (size_t)stages * stage_bytes + 1024 + 256; }

// Ring budget of the prefill kernels: kSmemWide, or less if the device allows
// less (the opt-in limit covers the kernel's static shared memory as well).
int wide_budget()
{
    const int lim = smem_optin() - 1024 - 256 - 64;
    return lim < kSmemWide ? lim : kSmemWide;
}

int stages_for(int stage_bytes, int budget = kSmemBudget)
{
    const int s = budget / stage_bytes;
    return s > kMaxStages ? kMaxStages : s;
}

uint32_t tmem_cols_for(int cols)
{
    uint32_t c = 32;
    while ((int)c < cols) c <<= 1;
    return c;
}

int sm_count()
{
    static int by_dev[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    int &n = by_dev[dev & 63];
    if (n == 0) cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

// Neurons per tile: the multiple of 16 (<= 128) that minimises waves x rows,
// so that the neuron tiles cover the SMs in about one wave.
int choose_rows(int N, int sms)
{
    int best = 16;
    long long best_cost = -1;
    for (int R = 16; R <= BM; R += 16) {
        const long long tiles = (N + R - 1) / R;
        const long long cost = ((tiles + sms - 1) / sms) * R;
        if (best_cost < 0 || cost <= best_cost) {
            best_cost = cost;
            best = R;
        }
    }
    return best;
}

// Neurons per tile of the prefill gate/up kernel: the multiple of 16 (<= 128,
// spanning at most two of the packed R-neuron tiles) that minimises waves x
// shared-memory bytes per K step.  Each operand byte is
// written to shared memory once by the copy engine and read once by the MMA; that
// traffic (the x tile, twice for split activations, plus 2 Rw weight rows) paces
// the MMA loop, while the tile's work grows with Rw.
int wide_rows(int N, int R, int mtiles, int sms, bool split)
{
    int best = 16;
    long long best_cost = -1;
    for (int Rw = 16; Rw <= BM; Rw += 16) {
        int g = Rw, r = R;   // gcd(Rw, R): a wide tile then spans at most two tiles of R neurons
        while (r) {
            const int t = g % r;
            g = r;
            r = t;
        }
        if (Rw - g > R) continue;
        const long long tiles = (long long)mtiles * ((N + Rw - 1) / Rw);
        const long long cost = ((tiles + sms - 1) / sms) * (BM * (split ? 2 : 1) + 2 * Rw);
        if (best_cost < 0 || cost <= best_cost) {
            best_cost = cost;
            best = Rw;
        }
    }
    return best;
}

// Splits of the neuron range in the prefill down projection: the count (<= 8,
// none empty) that minimises waves x (K blocks per unit + 4), the 4 standing for
// a unit's fixed cost (its accumulator's reductions into the output).
int wide_down_splits(int tiles, int KBn, int sms)
{
    int best = 1;
    long long best_cost = -1;
    for (int s = 1; s <= 8 && s <= KBn; ++s) {
        const int kps = (KBn + s - 1) / s;
        if ((KBn + kps - 1) / kps != s) continue;
        const long long units = (long long)tiles * s;
        const long long cost = ((units + sms - 1) / sms) * (kps + 4);
        if (best_cost < 0 || cost < best_cost) {
            best_cost = cost;
            best = s;
        }
    }
    return best;
}

}  // namespace
}  // namespace tc
}  // namespace sats
