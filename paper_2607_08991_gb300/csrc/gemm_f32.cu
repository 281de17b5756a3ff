// gemm_f32.cu -- products on the tensor cores of sm_103a whose results are as
// accurate as fp32 FMAs, for the paths that promise fp32 arithmetic: the post-gate
// activations of the calibrations (Sec. 2, Eqs. 1-3; Sec. 3.1).
//
// Two things keep tcgen05.mma (bf16 operands, fp32 accumulator) from that accuracy:
//  - its operands.  The weights are bf16 as they are; an fp32 activation is cut into
//    three bf16 parts by truncation (8 + 8 + 8 significant bits: the cut is exact), all
//    multiplied by the same weights.  Converter warps cut the tiles on their way into
//    shared memory, so the activations need no staging in memory.
//  - its accumulator, which is truncated after every K = 16 step: over 4096 products the
//    sum came out 1.2e-5 short (256 steps of half a unit of the 24th bit).  Here an
//    accumulator takes K = 32 only (the small parts first); every K block of 64 fills
//    two of them, and the epilogue warps read both from TMEM while the next block's MMAs
//    run, add the two and add the sum to totals that they keep in registers (rounded to
//    nearest).  Measured against fp64 on the Llama-shaped layer: 1.1e-7 relative, as the
//    fp32 FMA chains that this replaced.
//
// What bounds it: at up to 128 tokens the weight stream, beyond that the MMAs (about 70
// cycles each up to N = 128) and the TMEM reads (two accumulators per K block), which
// take about as long as each other; three MMAs per step with fp32 activations.
#include "tc_common.cuh"

namespace sats {
namespace tc {
namespace {

constexpr int kPreciseTok = 128;     // tokens per CTA tile: four accumulators of this width fill TMEM
constexpr int kConvThreads = 192;    // converter warps (fp32 activations)
// copy and MMA warps, converters, epilogue groups (fp32: two of 64 totals a thread within the
// 128 registers that 16 warps leave; bf16: four of 32)
template <bool F32> constexpr int kPreciseThreads = F32 ? 64 + kConvThreads + 256 : 64 + 512;
constexpr int kPartStages = 2;       // cut tiles in shared memory
constexpr int kParts = 3;
constexpr int kSubBlocks = 8;        // K blocks summed before they join the totals

struct PreciseGateParams {
    const uint16_t *w;     // gu_blk
    const float *x;        // fp32 activations [B][H] (the converter warps read them; bf16 ones come by TMA)
    int B, H, N, R, KBh;
    int NT;                // tokens per tile, a multiple of 16
    float *a;              // [B][N]
    int stages, stage_bytes, w_bytes, ring_bytes;
    uint32_t tmem_cols;    // four accumulators of NT columns
};

// x = the sum of three bf16 values, cut off the top 8 significant bits at a time.  (x - top is
// exact; the comparison keeps an infinity from becoming inf - inf.)
__device__ __forceinline__ float cut_bf16(float &x)
{
    const float top = __uint_as_float(__float_as_uint(x) & 0xffff0000u);
    x = top == x ? 0.f : x - top;
    return top;
}

__device__ __forceinline__ uint32_t pack_tops(float lo, float hi)
{
    return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}

// Eight fp32 values -> one 16-byte chunk of each part.
__device__ __forceinline__ void cut8(const float4 &p, const float4 &q, uint4 (&part)[kParts])
{
    float v[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < kParts; ++i) {
        float t[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) t[e] = cut_bf16(v[e]);
        part[i] = make_uint4(pack_tops(t[0], t[1]), pack_tops(t[2], t[3]), pack_tops(t[4], t[5]), pack_tops(t[6], t[7]));
    }
}

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// The converter warps (threads 64 .. 64 + kConvThreads - 1): fp32 tiles of NT rows x 64 columns, one
// per step, cut into kPartStages stages of swizzled bf16 parts [kParts][NT][64].  Unit u of a tile is
// 8 consecutive values (chunk u mod 8 of row u / 8), load(row, chunk, step, lo, hi) fetches one (zero
// unless set); the next step's units are loaded while this one's are cut.
template <int TOK, typename Load>
__device__ __forceinline__ bool cut_tiles(uint8_t *parts, int NT, int steps, uint64_t *pfull, uint64_t *pempty,
                                          volatile int *abort, Load load)
{
    constexpr int kUnits = (TOK * 8 + kConvThreads - 1) / kConvThreads;
    const int ct = threadIdx.x - 64, nu = NT * 8;
    float4 lo[kUnits], hi[kUnits];
    auto fetch = [&](int i, int step) {
        const int u = ct + kConvThreads * i;
        lo[i] = hi[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (u < nu) load(u >> 3, u & 7, step, lo[i], hi[i]);
    };
#pragma unroll
    for (int i = 0; i < kUnits; ++i)
        if (steps > 0) fetch(i, 0);
    for (int step = 0; step < steps; ++step) {
        const int ps = step % kPartStages;
        if (!mbar_wait(&pempty[ps], (uint32_t)((step / kPartStages) & 1) ^ 1u, abort)) return false;
        uint8_t *dst = parts + (size_t)ps * kParts * NT * kTileBytes;
#pragma unroll
        for (int i = 0; i < kUnits; ++i) {
            const int u = ct + kConvThreads * i, r = u >> 3, c = u & 7;
            uint4 part[kParts];
            cut8(lo[i], hi[i], part);
            if (step + 1 < steps) fetch(i, step + 1);
            if (u < nu) {
#pragma unroll
                for (int q = 0; q < kParts; ++q)
                    *reinterpret_cast<uint4 *>(dst + (size_t)(q * NT + r) * kTileBytes + ((c ^ (r & 7)) << 4)) = part[q];
            }
        }
        fence_async_smem();   // the MMAs read the tile through the async proxy
        mbar_arrive(&pfull[ps]);
    }
    return true;
}

// a = SiLU(x W_gate) for one tile of NT tokens and R neurons per CTA (neurons are the MMA's
// M, tokens its N).  Grid: token tiles x neuron tiles, the token tiles of one neuron tile
// next to each other, so that its weights come from L2 for all but the first of them.
template <bool F32>
__global__ void __launch_bounds__(kPreciseThreads<F32>, 1)
    gate_precise_kernel(const __grid_constant__ CUtensorMap tmX, const PreciseGateParams p)
{
    constexpr int kEpi0 = 2 + (F32 ? kConvThreads / 32 : 0);        // first epilogue warp
    constexpr int G = (kPreciseThreads<F32> / 32 - kEpi0) / 4;           // epilogue groups of four warps
    constexpr int kBlocks = (kPreciseTok / 16 + G - 1) / G;         // 16-token blocks per thread
    constexpr int kXParts = F32 ? kParts : 1;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *ring = align1024(smem_raw);
    uint8_t *parts = ring + p.ring_bytes;   // F32: [kPartStages][kParts][NT][64] bf16
    uint64_t *full = reinterpret_cast<uint64_t *>(parts + (F32 ? kPartStages * kParts * p.NT * kTileBytes : 0));
    uint64_t *empty = full + kMaxStages;
    uint64_t *pfull = empty + kMaxStages;     // [kPartStages]
    uint64_t *pempty = pfull + kPartStages;   // [kPartStages]
    uint64_t *acc_full = pempty + kPartStages;   // [2]
    uint64_t *acc_empty = acc_full + 2;          // [2]
    uint64_t *mma_done = acc_empty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mma_done + 1);
    __shared__ int abort_flag, issued_s, consumed_s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int R = p.R, NT = p.NT, S = p.stages, KBh = p.KBh;
    const int m0 = (int)blockIdx.x * NT, t = blockIdx.y;
    const int n_quads = (R + 31) / 32;   // TMEM lane quarters that hold neurons

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < kPartStages; ++s) {
            mbar_init(&pfull[s], kConvThreads);
            mbar_init(&pempty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 128 * G);
        }
        mbar_init(mma_done, 1);
        abort_flag = 0;
        issued_s = 0;
        consumed_s = 0;
        mbar_init_fence();
    }
    if (warp == 1) tmem_alloc(tmem_slot, p.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    grid_launch_dependents();

    if (warp == 0 && lane == 0) {
        const uint32_t load_bytes = (uint32_t)p.w_bytes + (F32 ? 0u : (uint32_t)(NT * kTileBytes));
        // (each weight tile is read once with one token tile, else by its neighbours through L2)
        const uint64_t once = l2_policy_evict_first();
        auto load_w = [&](int s, int kb) {
            const uint16_t *src = p.w + (size_t)((size_t)t * KBh + kb) * 2 * R * BK;
            if (gridDim.x == 1) bulk_load(ring + (size_t)s * p.stage_bytes, src, (uint32_t)p.w_bytes, &full[s], once);
            else bulk_load_shared(ring + (size_t)s * p.stage_bytes, src, (uint32_t)p.w_bytes, &full[s]);
        };
        const int npre = KBh < S ? KBh : S;
        for (int i = 0; i < npre; ++i) {   // the weights do not depend on the preceding kernel
            mbar_arrive_expect_tx(&full[i], load_bytes);
            load_w(i, i);
        }
        if (!F32) grid_dependency_wait();
        int kb = 0;
        for (int s = 0, ph = 0; kb < KBh; ++kb) {
            if (kb >= npre) {
                if (!mbar_wait(&empty[s], (uint32_t)ph ^ 1u, &abort_flag)) { abort_flag = 1; break; }
                mbar_arrive_expect_tx(&full[s], load_bytes);
                load_w(s, kb);
            }
            if (!F32) tma_load(ring + (size_t)s * p.stage_bytes + p.w_bytes, &tmX, kb * BK, m0, &full[s]);
            if (++s == S) { s = 0; ph ^= 1; }
        }
        issued_s = kb;
    } else if (warp == 1 && lane == 0) {
        const uint32_t idesc = instr_desc(BM, NT);
        int kb = 0;
        for (int s = 0, ph = 0; kb < KBh; ++kb) {
            const int buf = kb & 1, ps = kb % kPartStages;
            const uint32_t bph = (uint32_t)((kb >> 1) & 1);
            if (!mbar_wait(&acc_empty[buf], bph ^ 1u, &abort_flag) || !mbar_wait(&full[s], (uint32_t)ph, &abort_flag) ||
                (F32 && !mbar_wait(&pfull[ps], (uint32_t)((kb / kPartStages) & 1), &abort_flag))) {
                abort_flag = 1;
                break;
            }
            tc_fence_after();
            const uint32_t st = smem_addr(ring + (size_t)s * p.stage_bytes);
            const uint32_t xs = F32 ? smem_addr(parts + (size_t)ps * kParts * NT * kTileBytes) : st + p.w_bytes;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                const uint32_t d = tmem + (uint32_t)((buf * 2 + half) * NT);
#pragma unroll
                for (int q = kXParts - 1; q >= 0; --q)   // the smallest part first
#pragma unroll
                    for (int kk = 2 * half; kk < 2 * half + 2; ++kk)
                        mma_bf16(d, smem_desc(st + kk * 32), smem_desc(xs + q * NT * kTileBytes + kk * 32), idesc,
                                 (q < kXParts - 1 || (kk & 1)) ? 1u : 0u);
            }
            mma_commit(&empty[s]);
            if (F32) mma_commit(&pempty[ps]);
            mma_commit(&acc_full[buf]);
            if (++s == S) { s = 0; ph ^= 1; }
        }
        consumed_s = kb;
        mma_commit(mma_done);
    } else if (F32 && warp >= 2 && warp < kEpi0) {
        grid_dependency_wait();
        auto load = [&](int r, int c, int kb, float4 &lo, float4 &hi) {
            const int m = m0 + r, k = kb * BK + c * 8;
            if (m < p.B && k < p.H) {   // H is a multiple of 8
                const float4 *src = reinterpret_cast<const float4 *>(p.x + (size_t)m * p.H + k);
                lo = src[0];
                hi = src[1];
            }
        };
        if (!cut_tiles<kPreciseTok>(parts, NT, KBh, pfull, pempty, &abort_flag, load)) abort_flag = 1;
    } else if (warp >= kEpi0) {
        const int quad = warp & 3, grp = (warp - kEpi0) >> 2;
        const uint32_t lane0 = tmem + ((uint32_t)(32 * quad) << 16);
        const int n = t * R + 32 * quad + lane;
        // acc: totals; sub: the sums of up to kSubBlocks K blocks, added to the totals together, so that
        // a total takes few roundings at its full size (bf16: 64 more registers than fp32's have)
        float acc[kBlocks][16], sub[F32 ? 1 : kBlocks][16];
#pragma unroll
        for (int k = 0; k < kBlocks; ++k)
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                acc[k][e] = 0.f;
                if (!F32) sub[F32 ? 0 : k][e] = 0.f;
            }
        bool ok = true;
        for (int kb = 0; kb < KBh; ++kb) {
            const int buf = kb & 1;
            if (!mbar_wait(&acc_full[buf], (uint32_t)((kb >> 1) & 1), &abort_flag)) { ok = false; break; }
            tc_fence_after();
            if (quad < n_quads) {
#pragma unroll
                for (int k = 0; k < kBlocks; ++k) {
                    const int c0 = 16 * (grp + G * k);
                    if (c0 >= NT) break;
#pragma unroll
                    for (int o = 0; o < 16; o += 8) {
                        float v0[8], v1[8];
                        tmem_ld8(lane0 + (uint32_t)(2 * buf * NT + c0 + o), v0);
                        tmem_ld8(lane0 + (uint32_t)((2 * buf + 1) * NT + c0 + o), v1);
                        tmem_ld_wait();
#pragma unroll
                        for (int e = 0; e < 8; ++e) {
                            if (F32) acc[k][o + e] += v0[e] + v1[e];
                            else sub[F32 ? 0 : k][o + e] += v0[e] + v1[e];
                        }
                    }
                }
            }
            tc_fence_before();
            mbar_arrive(&acc_empty[buf]);
            if (!F32 && (kb % kSubBlocks == kSubBlocks - 1 || kb + 1 == KBh)) {
#pragma unroll
                for (int k = 0; k < kBlocks; ++k)
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        acc[k][e] += sub[F32 ? 0 : k][e];
                        sub[F32 ? 0 : k][e] = 0.f;
                    }
            }
        }
        grid_dependency_wait();   // a may still be in use by the preceding kernel
        if (32 * quad + lane < R && n < p.N) {
#pragma unroll
            for (int k = 0; k < kBlocks; ++k)
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const int j = 16 * (grp + G * k) + e;
                    if (j < NT && m0 + j < p.B) {
                        // (a wait that gave up leaves NaN: this call has no status word)
                        const float g = ok ? acc[k][e] : __int_as_float(0x7fffffff);
                        p.a[(size_t)(m0 + j) * p.N + n] = g / (1.0f + expf(-g));   // SiLU, Eq. 2
                    }
                }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        // the copies in flight and the arrival on mma_done must land before the CTA's shared memory is released
        int never = 0;
        if (abort_flag)
            for (int k = consumed_s; k < issued_s; ++k) mbar_wait(&full[k % S], (uint32_t)((k / S) & 1), &never);
        mbar_wait(mma_done, 0u, &never);
    }
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        tmem_dealloc(tmem, p.tmem_cols);
    }
}

template <bool F32>
cudaError_t launch_gate_precise(const sats_layer *layer, const void *x, int B, float *a, cudaStream_t stream)
{
    PreciseGateParams p{};
    p.w = layer->gu_blk;
    p.x = F32 ? static_cast<const float *>(x) : nullptr;
    p.B = B;
    p.H = layer->H;
    p.N = layer->N;
    p.R = layer->tc_R;
    p.KBh = layer->tc_kbh;
    const int mt = (B + kPreciseTok - 1) / kPreciseTok;
    p.NT = ((B + mt - 1) / mt + 15) & ~15;   // the tokens evenly over the fewest tiles
    p.a = a;
    p.tmem_cols = tmem_cols_for(4 * p.NT);
    p.w_bytes = p.R * kTileBytes;
    p.stage_bytes = p.w_bytes + (F32 ? 0 : p.NT * kTileBytes);
    const int parts = F32 ? kPartStages * kParts * p.NT * kTileBytes : 0;
    // the MMAs read 128 rows from a stage's start (rows R..127 of D are not used)
    const int over = BM * kTileBytes - p.stage_bytes;
    const int slack = over > 0 ? ((over + 1023) & ~1023) : 0;
    p.stages = stages_for(p.stage_bytes, wide_budget() - parts - slack);
    p.ring_bytes = p.stages * p.stage_bytes + slack;
    CUtensorMap mX{};
    if (!F32 && !make_map(&mX, x, (uint64_t)B, (uint64_t)p.H, (uint64_t)p.H * 2, (uint32_t)p.NT))
        return cudaErrorInvalidValue;
    static std::atomic<int> cfg[64];
    const size_t smem = smem_for(1, p.ring_bytes + parts);
    const cudaError_t e = set_smem(gate_precise_kernel<F32>, smem, cfg);
    if (e != cudaSuccess) return e;
    return launch_pdl_cfg(gate_precise_kernel<F32>, dim3(mt, layer->tc_T), kPreciseThreads<F32>, smem, stream, mX, p);
}

}  // namespace
}  // namespace tc

cudaError_t launch_gate_act(const sats_layer *layer, const uint16_t *x, int B, float *a, cudaStream_t stream)
{
    return tc::launch_gate_precise<false>(layer, x, B, a, stream);
}

cudaError_t launch_gate_act_f32(const sats_layer *layer, const float *x, int B, float *a, cudaStream_t stream)
{
    return tc::launch_gate_precise<true>(layer, x, B, a, stream);
}

}  // namespace sats
