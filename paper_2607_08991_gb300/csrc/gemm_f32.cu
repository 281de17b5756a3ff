// gemm_f32.cu -- products on the tensor cores of sm_103a whose results are as
// accurate as fp32 FMAs, for the paths that promise fp32 arithmetic: the post-gate
// activations of the calibrations (Sec. 2, Eqs. 1-3; Sec. 3.1), and a u of Eq. 6.
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
//    run, add the two, and add the sums (rounded to nearest) in two levels or, up to hidden
//    2048 with bf16 activations, to totals whose roundings are summed beside them.
//
// The error of a = SiLU(x W_gate) against fp64 (2-norm, units of 1e-8), before the tensor cores (fp32 FMA
// chains) / with sums in two levels of 8 blocks, fp32 tiles of more than 64 tokens in one, and a plain SiLU / now:
//   hidden                 256              512               1024              2048               4096               8192
//   bf16              7.1 /      6.7   7.7 /  9.0 / 6.8   8.5 /  9.5 /  6.8   9.5 / 10.1 /  6.7  10.9 / 11.0 / 10.5  13.5 / 12.2 / 11.8
//   fp32,  64 tokens  9.3 /      8.9  10.7 / 10.4 / 9.5  13.1 / 10.9 / 10.2  16.9 / 11.4 / 11.1  22.5 / 12.1 / 11.7  30.7 / 13.3 / 12.9
//   fp32, 256 tokens  9.3 /      8.9  10.7 / 10.4 / 9.5  13.1 / 12.2 / 10.2  16.9 / 14.9 / 11.1  22.5 / 18.8 / 11.7  30.7 / 24.3 / 12.8
// The worst of the elements, in units of the result's rms, 1e-6: 4096 bf16 1.4 / 1.8 / 1.6, fp32 2.2 / 3.7 / 1.7;
// 8192 bf16 1.3 / 1.7 / 1.7, fp32 2.8 / 4.0 / 1.8.  An Eq. 3 threshold of the Llama-shaped layer, 256 bf16
// tokens: 1.1e-7 / 9.5e-8 / 9.3e-8 of its value on average over 27 quantiles, 5.7e-7 / 5.0e-7 / 4.3e-7 at worst.
//
// What bounds it: neither the weight stream (17 us on that layer) nor the MMAs, but what the
// roles issue per K block: waits and commits of about 100 cycles each, the TMEM reads and
// additions of two accumulators (two at a time, f32x2; fp32: the next columns' read in
// flight), and with fp32 activations the converters (no test for infinities but one vote at
// the end of a step).  Llama-shaped layer, us: bf16 16 / 128 / 256 tokens 24.6 / 34.1 / 67.1, fp32 40.1 / 84.0 / 170.
// Without the accuracy that the last column above has over the middle one: 24.6 / 32.7 / 63.9 and 39.2 / 75.5 / 153.
#include "tc_common.cuh"

namespace sats {
namespace tc {
namespace {

constexpr int kPreciseTok = 128;     // tokens per CTA tile: four accumulators of this width fill TMEM
constexpr int kConvThreads = 192;    // converter warps (fp32 activations)
// copy and MMA warps, converters, epilogue groups (fp32: two of 64 totals a thread within the
// 128 registers that 16 warps leave; bf16: four of 32)
template <bool F32> constexpr int kPreciseThreads = F32 ? 64 + kConvThreads + 256 : 64 + 512;
// Largest hidden size at which bf16 totals keep their roundings: above it sums in two levels are as near to 64 bits as
// FMA chains were (the table above), and keeping them everywhere costs 36 % (Llama-shaped layer, 256 tokens 67.1 -> 87.3 us;
// here hidden 1024 / intermediate 4096 24.8 -> 32.1).
constexpr int kKeepH = 2048;
constexpr int kPartStages = 2;       // cut tiles in shared memory
constexpr int kParts = 3;
constexpr int kBarrierBytes = 256;   // the barriers and the TMEM slot, after the operand tiles

struct PreciseGateParams {
    const uint16_t *w;     // gu_blk
    const float *x;        // fp32 activations [B][H] (the converter warps read them; bf16 ones come by TMA)
    int B, H, N, R, KBh;
    int NT;                // tokens per tile, a multiple of 16
    float *a;              // [B][N]: written, or read for h (UP)
    uint16_t *hhi, *hlo;   // UP: [B][ldh] bf16
    int ldh;
    int *status;           // takes kStatusTimeout if a wait gives up, or nullptr
    int sub;               // K blocks summed before they join the totals
    int stages, stage_bytes, w_bytes, ring_bytes;
    uint32_t tmem_cols;    // four accumulators of NT columns
};

__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b)
{
    f32x2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
    return d;
}

// SiLU(g) = g / (1 + e^-g), Eq. 2, with the quotient's remainder and what 1 + e^-g was rounded by brought back in.
__device__ __forceinline__ float silu_rounded(float g)
{
    const float e = expf(-g), d = 1.0f + e, b = __fadd_rn(d, -1.0f);
    const float rest = __fadd_rn(1.0f, -__fadd_rn(d, -b)) + __fadd_rn(e, -b);   // d + rest = 1 + e
    const float q = g / d;
    const float c = __fdividef(fmaf(-q, rest, fmaf(-q, d, g)), d);
    return fabsf(c) < INFINITY ? q + c : q;   // (not a number where e or g is infinite)
}

__device__ __forceinline__ float bf16_top(float x) { return __uint_as_float(__float_as_uint(x) & 0xffff0000u); }

__device__ __forceinline__ uint32_t pack_tops(float lo, float hi)
{
    return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}

// Eight fp32 values -> one 16-byte chunk of each part: the top 8 significant bits, the next 8, the
// last 8 (each difference x - top is exact, so the parts' sum is x).  With SPECIAL an infinity leaves
// nothing after its top; without, inf - inf, and `odd` becomes NaN if any value was not finite.
template <bool SPECIAL>
__device__ __forceinline__ void cut8(const float4 &p, const float4 &q, uint4 (&part)[kParts], f32x2 &odd)
{
    const float v[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
    const f32x2 minus1 = pack2(-1.f, -1.f);
    uint32_t out[kParts][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float a = v[2 * e], b = v[2 * e + 1];
        out[0][e] = pack_tops(a, b);
        float2 d = unpack2(ffma2(pack2(bf16_top(a), bf16_top(b)), minus1, pack2(a, b)));
        if (SPECIAL) {   // a value that is its own top leaves nothing
            d.x = __float_as_uint(a) & 0xffffu ? d.x : 0.f;
            d.y = __float_as_uint(b) & 0xffffu ? d.y : 0.f;
        }
        out[1][e] = pack_tops(d.x, d.y);
        const f32x2 r = ffma2(pack2(bf16_top(d.x), bf16_top(d.y)), minus1, pack2(d.x, d.y));
        const float2 f = unpack2(r);
        out[2][e] = pack_tops(f.x, f.y);
        if (!SPECIAL) odd = ffma2(r, pack2(0.f, 0.f), odd);
    }
#pragma unroll
    for (int i = 0; i < kParts; ++i) part[i] = make_uint4(out[i][0], out[i][1], out[i][2], out[i][3]);
}

// One arrival per warp once all its lanes have read their TMEM columns: hundreds of threads
// arriving one by one on a barrier cost more than a K block's MMAs.
__device__ __forceinline__ void warp_arrive_tmem(uint64_t *bar, int lane)
{
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
}

__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// The converter warps (threads 64 .. 64 + kConvThreads - 1): fp32 tiles of NT rows x 64 columns, one
// per step, cut into kPartStages stages of swizzled bf16 parts [kParts][NT][64].  Unit u of a tile is
// 8 consecutive values (chunk u mod 8 of row u / 8), load(row, chunk, step, lo, hi) fetches one (zero
// unless set); the next step's units are loaded while this one's are cut.  (Loads up to four steps ahead
// cost more in code than they hid: LoRA layer, 8 tokens, 84.4 us with four, 81.0 with two, 79.7 with one.)
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
        if (u < nu && step < steps) load(u >> 3, u & 7, step, lo[i], hi[i]);
    };
#pragma unroll
    for (int i = 0; i < kUnits; ++i) fetch(i, 0);
    for (int step = 0; step < steps; ++step) {
        const int ps = step % kPartStages;
        if (!mbar_wait(&pempty[ps], (uint32_t)((step / kPartStages) & 1) ^ 1u, abort)) return false;
        uint8_t *dst = parts + (size_t)ps * kParts * NT * kTileBytes;
        auto put = [&](int u, const uint4 (&part)[kParts]) {
            const int r = u >> 3, c = u & 7;
            if (u >= nu) return;
#pragma unroll
            for (int q = 0; q < kParts; ++q)
                *reinterpret_cast<uint4 *>(dst + (size_t)(q * NT + r) * kTileBytes + ((c ^ (r & 7)) << 4)) = part[q];
        };
        f32x2 odd = pack2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < kUnits; ++i) {
            uint4 part[kParts];
            cut8<false>(lo[i], hi[i], part, odd);
            fetch(i, step + 1);
            put(ct + kConvThreads * i, part);
        }
        const float2 o = unpack2(odd);
        if (!(o.x == 0.f && o.y == 0.f)) {   // not all finite: once more
#pragma unroll 1
            for (int u = ct; u < nu; u += kConvThreads) {
                float4 p = make_float4(0.f, 0.f, 0.f, 0.f), q = p;
                uint4 part[kParts];
                load(u >> 3, u & 7, step, p, q);
                cut8<true>(p, q, part, odd);
                put(u, part);
            }
        }
        fence_async_smem();   // the MMAs read the tile through the async proxy
        __syncwarp();
        if ((threadIdx.x & 31) == 0) mbar_arrive(&pfull[ps]);
    }
    return true;
}

// a = SiLU(x W_gate) for one tile of NT tokens and R neurons per CTA (neurons are the MMA's
// M, tokens its N).  Grid: token tiles x neuron tiles, the token tiles of one neuron tile
// next to each other, so that its weights come from L2 for all but the first of them.
// TOK: the most tokens of a tile (64 leaves registers for a second level of sums with fp32 activations).
// UP: u = x W_up instead, and from it and the a of an earlier launch h = a u in two bf16 parts.
// KEEP: what a total is rounded by is summed beside it and added at the end (bf16 activations).
template <bool F32, int TOK, bool UP, bool KEEP>
__global__ void __launch_bounds__(kPreciseThreads<F32>, 1)
    gate_precise_kernel(const __grid_constant__ CUtensorMap tmX, const PreciseGateParams p)
{
    constexpr int kEpi0 = 2 + (F32 ? kConvThreads / 32 : 0);        // first epilogue warp
    constexpr int G = (kPreciseThreads<F32> / 32 - kEpi0) / 4;           // epilogue groups of four warps
    constexpr int kBlocks = (TOK / 16 + G - 1) / G;         // 16-token blocks per thread
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
    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    const int R = p.R, NT = p.NT, S = p.stages, KBh = p.KBh;
    const int m0 = (int)blockIdx.x * NT, t = blockIdx.y;
    const int n_quads = (R + 31) / 32;   // TMEM lane quarters that hold neurons
    auto give_up = [&]() {
        abort_flag = 1;
        if (p.status) atomicOr(p.status, kStatusTimeout);
    };

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < kPartStages; ++s) {
            mbar_init(&pfull[s], kConvThreads / 32);
            mbar_init(&pempty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], 4 * G);
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

    // (bf16: one lane runs the load role, 256 tokens 69 us so and 75 with a whole warp; fp32: the warp, 64
    // tokens 48.0 us and 51.6 with one lane)
    if (warp == 0 && (F32 || lane == 0)) {
        const uint32_t lead = F32 ? elect_one() : 1u;
        const uint32_t load_bytes = (uint32_t)p.w_bytes + (F32 ? 0u : (uint32_t)(NT * kTileBytes));
        // (each weight tile is read once with one token tile, else by its neighbours through L2)
        const uint64_t once = l2_policy_evict_first();
        auto load_w = [&](int s, int kb) {
            const uint16_t *src = p.w + ((size_t)((size_t)t * KBh + kb) * 2 + (UP ? 1 : 0)) * R * BK;
            if (gridDim.x == 1) bulk_load_if(lead, ring + (size_t)s * p.stage_bytes, src, (uint32_t)p.w_bytes, &full[s], once);
            else bulk_load_shared_if(lead, ring + (size_t)s * p.stage_bytes, src, (uint32_t)p.w_bytes, &full[s]);
        };
        const int npre = KBh < S ? KBh : S;
        for (int i = 0; i < npre; ++i) {   // the weights do not depend on the preceding kernel
            mbar_expect_if(lead, &full[i], load_bytes);
            load_w(i, i);
        }
        if (!F32) grid_dependency_wait();
        int kb = 0;
        for (int s = 0, ph = 0; kb < KBh; ++kb) {
            if (kb >= npre) {
                if (!(F32 ? warp_wait(&empty[s], (uint32_t)ph ^ 1u, &abort_flag)
                          : mbar_wait(&empty[s], (uint32_t)ph ^ 1u, &abort_flag))) {
                    give_up();
                    break;
                }
                mbar_expect_if(lead, &full[s], load_bytes);
                load_w(s, kb);
            }
            if (!F32) tma_load_if(lead, ring + (size_t)s * p.stage_bytes + p.w_bytes, &tmX, kb * BK, m0, &full[s]);
            if (++s == S) { s = 0; ph ^= 1; }
        }
        issued_s = kb;
    } else if (warp == 1) {
        const uint32_t lead = elect_one();
        const uint32_t idesc = instr_desc(BM, NT);
        int kb = 0;
        for (int s = 0, ph = 0; kb < KBh; ++kb) {
            const int buf = kb & 1, ps = kb % kPartStages;
            const uint32_t bph = (uint32_t)((kb >> 1) & 1);
            // fp32: the three barriers by a lane each (a wait costs about 100 cycles even when its phase is over)
            uint64_t *const bar = lane == 1 ? &acc_empty[buf] : F32 && lane == 2 ? &pfull[ps] : &full[s];
            if (F32 ? !warp_wait(bar, lane == 1 ? bph ^ 1u : lane == 2 ? bph : (uint32_t)ph, &abort_flag)
                    : !warp_wait(&acc_empty[buf], bph ^ 1u, &abort_flag) || !warp_wait(&full[s], (uint32_t)ph, &abort_flag)) {
                give_up();
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
                        mma_bf16_if(lead, d, smem_desc(st + kk * 32), smem_desc(xs + q * NT * kTileBytes + kk * 32), idesc,
                                 (q < kXParts - 1 || (kk & 1)) ? 1u : 0u);
            }
            mma_commit_if(lead, &empty[s]);
            if (F32) mma_commit_if(lead, &pempty[ps]);
            mma_commit_if(lead, &acc_full[buf]);
            if (++s == S) { s = 0; ph ^= 1; }
        }
        consumed_s = kb;
        mma_commit_if(lead, mma_done);
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
        if (!cut_tiles<TOK>(parts, NT, KBh, pfull, pempty, &abort_flag, load)) give_up();
    } else if (warp >= kEpi0) {
        const int quad = warp & 3, grp = (warp - kEpi0) >> 2;
        const uint32_t lane0 = tmem + ((uint32_t)(32 * quad) << 16);
        const int n = t * R + 32 * quad + lane;
        // sum: the sums of up to p.sub K blocks, which join the totals together, so that a total takes few roundings at
        // its full size; with KEEP every K block joins, and sum holds what the totals were rounded by.  64 totals a
        // thread (fp32 activations, tiles of more than 64 tokens) are kept in shared memory.
        constexpr bool kShared = kBlocks > 2;
        constexpr int kPairs = 8 * kBlocks;
        static_assert(!KEEP || !(kShared || UP), "kept roundings need the totals in registers");
        f32x2 sum[kPairs], tot[kShared ? 1 : kPairs];
        f32x2 *const shared_tot = reinterpret_cast<f32x2 *>(reinterpret_cast<uint8_t *>(full) + kBarrierBytes) +
                                  (threadIdx.x - 32 * kEpi0);   // [kPairs] of this thread, 128 G apart
        const bool busy = quad < n_quads;   // (uniform in the warp, as is the next)
        auto in_tile = [&](int pair) { return 16 * (grp + G * (pair >> 3)) < NT; };
#pragma unroll
        for (int k = 0; k < kPairs; ++k) {
            sum[k] = pack2(0.f, 0.f);
            if (!kShared) tot[kShared ? 0 : k] = sum[k];
            else if (in_tile(k)) shared_tot[k * 128 * G] = sum[k];
        }
        int since = 0;
        bool ok = true;
        for (int kb = 0; kb < KBh; ++kb) {
            const int buf = kb & 1;
            if (!mbar_wait(&acc_full[buf], (uint32_t)((kb >> 1) & 1), &abort_flag)) {
                give_up();
                ok = false;
                break;
            }
            tc_fence_after();
            if (busy) {
                const uint32_t a0 = lane0 + (uint32_t)(2 * buf * NT);
                constexpr int kV = F32 ? 2 : 1;
                float v[kV][2][8];
                auto fetch = [&](int o) {   // 8 columns of both accumulators
                    const uint32_t c = (uint32_t)(16 * (grp + G * (o >> 1)) + 8 * (o & 1));
                    tmem_ld8(a0 + c, v[o % kV][0]);
                    tmem_ld8(a0 + (uint32_t)NT + c, v[o % kV][1]);
                };
                if (F32 && 16 * grp < NT) fetch(0);
#pragma unroll
                for (int o = 0; o < 2 * kBlocks; ++o) {
                    if (16 * (grp + G * (o >> 1)) >= NT) break;
                    if (!F32) fetch(o);
                    tmem_ld_wait();
                    if (F32 && o + 1 < 2 * kBlocks && 16 * (grp + G * ((o + 1) >> 1)) < NT) fetch(o + 1);
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const f32x2 w = add2(pack2(v[o % kV][0][2 * e], v[o % kV][0][2 * e + 1]),
                                             pack2(v[o % kV][1][2 * e], v[o % kV][1][2 * e + 1]));
                        f32x2 &s = sum[4 * o + e], &t0 = tot[kShared ? 0 : 4 * o + e];
                        if (KEEP) {
                            const f32x2 minus1 = pack2(-1.f, -1.f), t1 = add2(t0, w);
                            s = add2(s, ffma2(ffma2(t0, minus1, t1), minus1, w));   // += w - (t1 - t0)
                            t0 = t1;
                        } else {
                            s = add2(s, w);
                        }
                    }
                }
            }
            warp_arrive_tmem(&acc_empty[buf], lane);
            if (!KEEP && (++since == p.sub || kb + 1 == KBh)) {
                since = 0;
#pragma unroll
                for (int k = 0; k < kPairs; ++k) {
                    if (!busy || !in_tile(k)) break;
                    f32x2 &to = kShared ? shared_tot[k * 128 * G] : tot[kShared ? 0 : k];
                    to = add2(to, sum[k]);
                    sum[k] = pack2(0.f, 0.f);
                }
            }
        }
        grid_dependency_wait();   // a (h) may still be in use by the preceding kernel
        if (32 * quad + lane < R && n < p.N) {
#pragma unroll
            for (int k = 0; k < kBlocks; ++k) {
                float av[UP ? 16 : 1];
                if (UP)
#pragma unroll
                    for (int e = 0; e < 16; ++e) {
                        const int j = 16 * (grp + G * k) + e;
                        av[UP ? e : 0] = j < NT && m0 + j < p.B ? p.a[(size_t)(m0 + j) * p.N + n] : 0.f;
                    }
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    const int j = 16 * (grp + G * k) + e;
                    if (j < NT && m0 + j < p.B) {
                        const int pair = 8 * k + e / 2;
                        const float2 two = unpack2(kShared ? shared_tot[pair * 128 * G] : tot[kShared ? 0 : pair]);
                        float g = e & 1 ? two.y : two.x;
                        if (KEEP && fabsf(g) < INFINITY) {   // (what an infinite total was rounded by is no number)
                            const float2 r = unpack2(sum[pair]);
                            g += e & 1 ? r.y : r.x;
                        }
                        if (!ok) g = __int_as_float(0x7fffffff);   // (some callers have no status word)
                        if (!UP) {
                            p.a[(size_t)(m0 + j) * p.N + n] = silu_rounded(g);
                        } else {
                            const float h = av[UP ? e : 0] * g;
                            const uint16_t hb = bf16_bits(h);
                            p.hhi[(size_t)(m0 + j) * p.ldh + n] = hb;
                            p.hlo[(size_t)(m0 + j) * p.ldh + n] = bf16_bits(h - __uint_as_float((uint32_t)hb << 16));
                        }
                    }
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

// K blocks summed before they join the totals.
int sub_blocks(int KBh) { return KBh <= 32 ? 4 : 8; }

template <bool F32, int TOK, bool UP = false, bool KEEP = false>
cudaError_t launch_gate_precise(const sats_layer *layer, const void *x, int B, float *a, int *status,
                                cudaStream_t stream, uint16_t *hhi = nullptr, uint16_t *hlo = nullptr)
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
    p.hhi = hhi;
    p.hlo = hlo;
    p.ldh = layer->ldn;
    p.status = status;
    p.tmem_cols = tmem_cols_for(4 * p.NT);
    p.w_bytes = p.R * kTileBytes;
    p.stage_bytes = p.w_bytes + (F32 ? 0 : p.NT * kTileBytes);
    p.sub = sub_blocks(p.KBh);
    const int parts = F32 ? kPartStages * kParts * p.NT * kTileBytes : 0;
    const int totals = F32 && TOK > 64 ? TOK * BM * 4 : 0;
    // the MMAs read 128 rows from a stage's start (rows R..127 of D are not used)
    const int over = BM * kTileBytes - p.stage_bytes;
    const int slack = over > 0 ? ((over + 1023) & ~1023) : 0;
    p.stages = stages_for(p.stage_bytes, wide_budget() - parts - slack - totals);
    p.ring_bytes = p.stages * p.stage_bytes + slack;
    CUtensorMap mX{};
    if (!F32 && !make_map(&mX, x, (uint64_t)B, (uint64_t)p.H, (uint64_t)p.H * 2, (uint32_t)p.NT))
        return cudaErrorInvalidValue;
    static std::atomic<int> cfg[64];
    const size_t smem = smem_for(1, p.ring_bytes + parts + totals);
    const cudaError_t e = set_smem(gate_precise_kernel<F32, TOK, UP, KEEP>, smem, cfg);
    if (e != cudaSuccess) return e;
    return launch_pdl_cfg(gate_precise_kernel<F32, TOK, UP, KEEP>, dim3(mt, layer->tc_T), kPreciseThreads<F32>, smem, stream, mX, p);
}

// ---------------------------------------------------------------------- LoRA batches
// The sparse path of a fine-tuned model (Sec. 4) for batches of three tokens and more, in the
// accuracy of the fused kernel, which runs the smaller ones:
//   lora_z_kernel        z = x A_gate | x A_up, per slice of hidden rows
//   lora_gate_up_kernel  g = x W_gate + s z B_gate[:, n], u likewise, h = keep ? SiLU(g) u : 0, w += h A_down
//   lora_down_kernel     y += h W_down + s w B_down
// W is streamed once for up to kLoraTok tokens, where the fused kernel streamed it once per pass of one or two
// (129 us for four tokens on the Llama-shaped layer at 70 % sparsity, 267 us for eight; 77 here; with A_down as one
// more tile of outputs and w B_down in a kernel of its own 79 and 80).  What bounds it: that stream and the roles'
// serial issue; with at most 32 tokens the parts of an operand are the rows of one tile, so a K step is one MMA per
// weight tile however many parts there are, and their products are added in the epilogue.
constexpr int kLoraTok = 32;
constexpr int kLoraWRow = kMaxLoraRank;        // row pitch of w
constexpr int kLoraZRow = 2 * kMaxLoraRank;    // row pitch of z
constexpr int kLoraEpiThreads = 256;           // two groups of four warps, one per 16 tokens
template <bool F32> constexpr int kLoraGuThreads = 64 + (F32 ? kConvThreads : 0) + kLoraEpiThreads;
constexpr int kLoraDownThreads = 64 + kConvThreads + kLoraEpiThreads;

// z[b][s][0 .. 2r) over the hidden rows of slice s, and w[b] cleared.  Grid: (slices, B).
template <typename X>
__global__ void __launch_bounds__(256) lora_z_kernel(const X *__restrict__ x, int H, const uint16_t *__restrict__ agu,
                                                     int r, float *__restrict__ z, float *__restrict__ wsum)
{
    __shared__ float red[256][9];
    const int s = blockIdx.x, slices = gridDim.x, b = blockIdx.y, t = threadIdx.x;
    const int C = r / 4, rows = 256 / C;   // 16-byte chunks of a row of agu (2r values), rows per pass
    const int c = t % C, row = t / C;
    const int h0 = (int)((long long)H * s / slices), h1 = (int)((long long)H * (s + 1) / slices);
    grid_dependency_wait();
    grid_launch_dependents();
    if (s == 0 && t < kLoraWRow) wsum[(size_t)b * kLoraWRow + t] = 0.f;   // the gate/up kernel adds into it
    float acc[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.f;
    if (row < rows) {
#pragma unroll 4
        for (int h = h0 + row; h < h1; h += rows) {
            float xv;
            if constexpr (sizeof(X) == 2) xv = __uint_as_float((uint32_t)x[(size_t)b * H + h] << 16);
            else xv = x[(size_t)b * H + h];
            float w[8];
            unpack8(*reinterpret_cast<const uint4 *>(agu + (size_t)h * 2 * r + 8 * c), w);
#pragma unroll
            for (int e = 0; e < 8; ++e) acc[e] = fmaf(xv, w[e], acc[e]);
        }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) red[t][e] = acc[e];
    __syncthreads();
    if (t < 2 * r) {
        float sum = 0.f;
        for (int k = 0; k < rows; ++k) sum += red[k * C + t / 8][t % 8];
        z[((size_t)b * slices + s) * kLoraZRow + t] = sum;
    }
}

struct LoraGuParams {
    const uint16_t *w;      // gu_blk
    const float *x;         // fp32 activations [B][H] (bf16 ones come by TMA)
    int B, H, N, R, KBh;
    int NT;                 // tokens per tile (16 or 32)
    int halves;             // accumulators per K block and weight matrix: K = 32 each (2) or 64 (1)
    int sub;                // K blocks summed before they join the totals
    float t_l, scale;
    const uint16_t *blk;    // adapter columns per neuron: B_gate, B_up, A_down
    int r;
    const float *z;         // [B][slices][kLoraZRow]
    int slices;
    float *h;               // [B][ldh] fp32
    int ldh;
    uint8_t *keep;          // [B][keep_stride] or nullptr
    int keep_stride;
    float *y;               // [B][H], cleared here for the down kernel's additions
    float *wsum;            // [B][kLoraWRow]: w = h A_down, added to
    int *ctl;
    int stages, stage_bytes, w_bytes, ring_bytes;
    uint32_t tmem_cols;
};

// One tile of NT tokens and R neurons per CTA, as gate_precise_kernel; grid: token tiles x neuron tiles.
template <bool F32>
__global__ void __launch_bounds__(kLoraGuThreads<F32>, 1)
    lora_gate_up_kernel(const __grid_constant__ CUtensorMap tmX, const LoraGuParams p)
{
    constexpr int kEpi0 = 2 + (F32 ? kConvThreads / 32 : 0);
    constexpr int kXParts = F32 ? kParts : 1;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *ring = align1024(smem_raw);
    uint8_t *parts = ring + p.ring_bytes;
    uint64_t *full = reinterpret_cast<uint64_t *>(parts + (F32 ? kPartStages * kParts * p.NT * kTileBytes : 0));
    uint64_t *empty = full + kMaxStages;
    uint64_t *pfull = empty + kMaxStages;
    uint64_t *pempty = pfull + kPartStages;
    uint64_t *acc_full = pempty + kPartStages;   // [2]
    uint64_t *acc_empty = acc_full + 2;          // [2]
    uint64_t *mma_done = acc_empty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mma_done + 1);
    __shared__ int abort_flag, issued_s, consumed_s;
    __shared__ float zs[kLoraTok][kLoraZRow];
    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    const int R = p.R, NT = p.NT, S = p.stages, KBh = p.KBh, halves = p.halves;
    const int NX = kXParts * NT;   // accumulator columns: the parts side by side
    const int m0 = (int)blockIdx.x * NT, t = blockIdx.y;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < kPartStages; ++s) {
            mbar_init(&pfull[s], kConvThreads / 32);
            mbar_init(&pempty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], kLoraEpiThreads / 32);
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

    if (warp == 0) {
        const uint32_t lead = elect_one();
        const uint32_t load_bytes = (uint32_t)p.w_bytes + (F32 ? 0u : (uint32_t)(NT * kTileBytes));
        const uint64_t once = l2_policy_evict_first();
        auto load_w = [&](int s, int kb) {
            const uint16_t *src = p.w + ((size_t)t * KBh + kb) * 2 * R * BK;
            if (gridDim.x == 1) bulk_load_if(lead, ring + (size_t)s * p.stage_bytes, src, (uint32_t)p.w_bytes, &full[s], once);
            else bulk_load_shared_if(lead, ring + (size_t)s * p.stage_bytes, src, (uint32_t)p.w_bytes, &full[s]);
        };
        const int npre = KBh < S ? KBh : S;
        for (int i = 0; i < npre; ++i) {
            mbar_expect_if(lead, &full[i], load_bytes);
            load_w(i, i);
        }
        if (!F32) grid_dependency_wait();
        int kb = 0;
        for (int s = 0, ph = 0; kb < KBh; ++kb) {
            if (kb >= npre) {
                if (!warp_wait(&empty[s], (uint32_t)ph ^ 1u, &abort_flag)) { set_timeout(p.ctl, &abort_flag); break; }
                mbar_expect_if(lead, &full[s], load_bytes);
                load_w(s, kb);
            }
            if (!F32) tma_load_if(lead, ring + (size_t)s * p.stage_bytes + p.w_bytes, &tmX, kb * BK, m0, &full[s]);
            if (++s == S) { s = 0; ph ^= 1; }
        }
        issued_s = kb;
    } else if (warp == 1) {
        const uint32_t lead = elect_one();
        const uint32_t idesc = instr_desc(BM, NX);
        const int per = 4 / halves;   // K = 16 steps per accumulator
        int kb = 0;
        for (int s = 0, ph = 0; kb < KBh; ++kb) {
            const int buf = kb & 1, ps = kb % kPartStages;
            if (!warp_wait(&acc_empty[buf], (uint32_t)((kb >> 1) & 1) ^ 1u, &abort_flag) ||
                !warp_wait(&full[s], (uint32_t)ph, &abort_flag) ||
                (F32 && !warp_wait(&pfull[ps], (uint32_t)((kb / kPartStages) & 1), &abort_flag))) {
                set_timeout(p.ctl, &abort_flag);
                break;
            }
            tc_fence_after();
            const uint32_t st = smem_addr(ring + (size_t)s * p.stage_bytes);
            const uint32_t xs = F32 ? smem_addr(parts + (size_t)ps * kParts * NT * kTileBytes) : st + p.w_bytes;
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk) {
                const uint32_t d = tmem + (uint32_t)((buf * halves + kk / per) * 2 * NX), acc = kk % per ? 1u : 0u;
                const uint64_t b = smem_desc(xs + kk * 32);
                mma_bf16_if(lead, d, smem_desc(st + kk * 32), b, idesc, acc);
                mma_bf16_if(lead, d + NX, smem_desc(st + R * kTileBytes + kk * 32), b, idesc, acc);
            }
            mma_commit_if(lead, &empty[s]);
            if (F32) mma_commit_if(lead, &pempty[ps]);
            mma_commit_if(lead, &acc_full[buf]);
            if (++s == S) { s = 0; ph ^= 1; }
        }
        consumed_s = kb;
        mma_commit_if(lead, mma_done);
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
        if (!cut_tiles<kLoraTok>(parts, NT, KBh, pfull, pempty, &abort_flag, load)) set_timeout(p.ctl, &abort_flag);
    } else if (warp >= kEpi0) {
        const int et = threadIdx.x - 32 * kEpi0;
        const int quad = warp & 3, grp = (warp - kEpi0) >> 2;
        const int c0 = 16 * grp;
        const int n = t * R + 32 * quad + lane;
        const bool busy = c0 < NT && 32 * quad < R;   // (uniform in the warp)
        const uint32_t lane0 = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)c0;
        // acc: the sums of up to p.sub K blocks; they join the totals together, so that a total takes few roundings
        // at its full size.  The totals are kept in shared memory with fp32 activations (whose parts take the registers).
        float acc[2][16], tot[2][F32 ? 1 : 16];
        float *const shared_tot = reinterpret_cast<float *>(reinterpret_cast<uint8_t *>(full) + kBarrierBytes) +
                                  et;   // [2][16] of this thread, kLoraEpiThreads apart
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                acc[q][e] = 0.f;
                if (F32) shared_tot[(16 * q + e) * kLoraEpiThreads] = 0.f;
                else tot[q][F32 ? 0 : e] = 0.f;
            }
        bool ok = true;
        int kb = 0;
        auto blocks = [&](int end) {
            for (; kb < end; ++kb) {
                const int buf = kb & 1;
                if (!mbar_wait(&acc_full[buf], (uint32_t)((kb >> 1) & 1), &abort_flag)) {
                    set_timeout(p.ctl, &abort_flag);
                    return false;
                }
                tc_fence_after();
                if (busy) {
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        float sum[16];
#pragma unroll
                        for (int e = 0; e < 16; ++e) sum[e] = 0.f;
                        for (int f = 0; f < halves; ++f) {
                            float v[kXParts][16];
#pragma unroll
                            for (int k = 0; k < kXParts; ++k)
                                tmem_ld16(lane0 + (uint32_t)(((buf * halves + f) * 2 + q) * NX + k * NT), v[k]);
                            tmem_ld_wait();
#pragma unroll
                            for (int e = 0; e < 16; ++e) {
                                float w = v[kXParts - 1][e];   // the small parts first
#pragma unroll
                                for (int k = kXParts - 2; k >= 0; --k) w += v[k][e];
                                sum[e] += w;
                            }
                        }
#pragma unroll
                        for (int e = 0; e < 16; ++e) acc[q][e] += sum[e];
                    }
                }
                warp_arrive_tmem(&acc_empty[buf], lane);
            }
            return true;
        };
        while (ok && kb < KBh) {
            ok = blocks(min(KBh, kb + p.sub));
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    float &to = F32 ? shared_tot[(16 * q + e) * kLoraEpiThreads] : tot[q][F32 ? 0 : e];
                    to += acc[q][e];
                    acc[q][e] = 0.f;
                }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
            for (int e = 0; e < 16; ++e) acc[q][e] = F32 ? shared_tot[(16 * q + e) * kLoraEpiThreads] : tot[q][F32 ? 0 : e];
        grid_dependency_wait();   // z, and y, w, h and the keep bytes may still be in use by the preceding kernels
        const int ctas = (int)(gridDim.x * gridDim.y), cta = (int)(blockIdx.y * gridDim.x + blockIdx.x);
        for (long long i = (long long)cta * kLoraEpiThreads + et; i < (long long)p.B * (p.H >> 2);
             i += (long long)ctas * kLoraEpiThreads)
            reinterpret_cast<float4 *>(p.y)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        const int r = p.r, r2 = 2 * r;
        for (int i = et; i < NT * r2; i += kLoraEpiThreads) {
            const int j = i / r2, c = i % r2;
            float v = 0.f;
            if (m0 + j < p.B)
                for (int k = 0; k < p.slices; ++k) v += p.z[((size_t)(m0 + j) * p.slices + k) * kLoraZRow + c];
            zs[j][c] = v;
        }
        named_barrier(1, kLoraEpiThreads);
        const bool mine = ok && busy && 32 * quad + lane < R && n < p.N;
        const uint16_t *col = p.blk + (size_t)n * 3 * r;
        float hv[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) hv[e] = 0.f;
        if (mine) {
            float lg[16], lu[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) lg[e] = lu[e] = 0.f;
            for (int q0 = 0; q0 < r; q0 += 8) {
                float bg[8], bu[8];
                unpack8(*reinterpret_cast<const uint4 *>(col + q0), bg);
                unpack8(*reinterpret_cast<const uint4 *>(col + r + q0), bu);
#pragma unroll
                for (int e = 0; e < 16; ++e)
#pragma unroll
                    for (int q = 0; q < 8; ++q) {
                        lg[e] = fmaf(zs[c0 + e][q0 + q], bg[q], lg[e]);
                        lu[e] = fmaf(zs[c0 + e][r + q0 + q], bu[q], lu[e]);
                    }
            }
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                const int j = m0 + c0 + e;
                if (j < p.B && c0 + e < NT) {
                    const float g = fmaf(p.scale, lg[e], acc[0][e]);
                    const float u = fmaf(p.scale, lu[e], acc[1][e]);
                    const float a = g / (1.0f + expf(-g));   // SiLU, Eq. 2
                    const bool keep = fabsf(a) >= p.t_l;     // Eqs. 4-5
                    hv[e] = keep ? a * u : 0.f;
                    p.h[(size_t)j * p.ldh + n] = hv[e];
                    if (p.keep) p.keep[(size_t)j * p.keep_stride + n] = keep ? 1 : 0;
                }
            }
        }
        // w += h A_down: 4 tokens x 8 rank columns at a time, summed over the warp's neurons so that lane k is left
        // with token k mod 4, column k / 4
        for (int q0 = 0; busy && q0 < r; q0 += 8) {
            float ad[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) ad[q] = 0.f;
            if (mine) unpack8(*reinterpret_cast<const uint4 *>(col + 2 * r + q0), ad);
#pragma unroll
            for (int t0 = 0; t0 < 16; t0 += 4) {
                if (m0 + c0 + t0 >= p.B) break;
                float x[32];
#pragma unroll
                for (int k = 0; k < 32; ++k) x[k] = hv[t0 + (k & 3)] * ad[k >> 2];
#pragma unroll
                for (int o = 16; o >= 1; o >>= 1)
#pragma unroll
                    for (int k = 0; k < o; ++k) {
                        const bool up = lane & o;
                        const float give = up ? x[k] : x[k + o], have = up ? x[k + o] : x[k];
                        x[k] = have + __shfl_xor_sync(0xffffffffu, give, o);
                    }
                const int j = m0 + c0 + t0 + (lane & 3);
                if (j < p.B && c0 + t0 + (lane & 3) < NT) atomicAdd(p.wsum + (size_t)j * kLoraWRow + q0 + (lane >> 2), x[0]);
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
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

struct LoraDownParams {
    const uint16_t *w;      // wd_blk
    const float *h;         // [B][ldh] fp32
    int ldh, B, H, N;
    int NT, halves;
    int KBn, units;         // units = hidden tiles x KBn: (hidden tile, neuron block) pairs
    const uint16_t *bd;     // B_down [r][H]
    int r;
    float scale;
    float *y;               // [B][H], added to
    const float *wsum;      // [B][kLoraWRow]
    int *ctl;
    int stages, ring_bytes;
    uint32_t tmem_cols;
    KeepLists lists;        // the kept lists to write, if any
};

// CTA c takes units [c U / G, (c + 1) U / G) in order for the tokens of tile blockIdx.y; consecutive
// units of one output tile are summed in registers and added into y, with s w B_down by the CTA of the tile's
// first unit.
__global__ void __launch_bounds__(kLoraDownThreads, 1) lora_down_kernel(const LoraDownParams p)
{
    constexpr int kEpi0 = 2 + kConvThreads / 32;
    constexpr int kA = BM * kTileBytes;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *ring = align1024(smem_raw);
    uint8_t *parts = ring + p.ring_bytes;
    uint64_t *full = reinterpret_cast<uint64_t *>(parts + kPartStages * kParts * p.NT * kTileBytes);
    uint64_t *empty = full + kMaxStages;
    uint64_t *pfull = empty + kMaxStages;
    uint64_t *pempty = pfull + kPartStages;
    uint64_t *acc_full = pempty + kPartStages;   // [2]
    uint64_t *acc_empty = acc_full + 2;          // [2]
    uint64_t *mma_done = acc_empty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(mma_done + 1);
    __shared__ int abort_flag, issued_s, consumed_s;
    __shared__ float tr[kLoraEpiThreads / 32][16][33];
    __shared__ __align__(16) float ws[kLoraTok][kLoraWRow];   // s w
    const int warp = uniform_warp(), lane = threadIdx.x & 31;
    const int NT = p.NT, S = p.stages, KBn = p.KBn, halves = p.halves, NX = kParts * NT;
    const int m0 = (int)blockIdx.y * NT;
    const int u0 = (int)((long long)blockIdx.x * p.units / gridDim.x);
    const int u1 = (int)((long long)(blockIdx.x + 1) * p.units / gridDim.x);
    const int nu = u1 - u0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int s = 0; s < kPartStages; ++s) {
            mbar_init(&pfull[s], kConvThreads / 32);
            mbar_init(&pempty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&acc_full[b], 1);
            mbar_init(&acc_empty[b], kLoraEpiThreads / 32);
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

    if (warp == 0) {
        const uint32_t lead = elect_one();
        // nothing but weights is copied, so the whole stream runs ahead of the preceding kernel's end
        const uint64_t once = l2_policy_evict_first();
        int i = 0;
        for (int s = 0, ph = 0; i < nu; ++i) {
            if (!warp_wait(&empty[s], (uint32_t)ph ^ 1u, &abort_flag)) { set_timeout(p.ctl, &abort_flag); break; }
            const uint16_t *src = p.w + (size_t)(u0 + i) * BM * BK;
            mbar_expect_if(lead, &full[s], (uint32_t)kA);
            if (gridDim.y == 1) bulk_load_if(lead, ring + (size_t)s * kA, src, (uint32_t)kA, &full[s], once);
            else bulk_load_shared_if(lead, ring + (size_t)s * kA, src, (uint32_t)kA, &full[s]);
            if (++s == S) { s = 0; ph ^= 1; }
        }
        issued_s = i;
    } else if (warp == 1) {
        const uint32_t lead = elect_one();
        const uint32_t idesc = instr_desc(BM, NX);
        const int per = 4 / halves;
        int i = 0;
        for (int s = 0, ph = 0; i < nu; ++i) {
            const int buf = i & 1, ps = i % kPartStages;
            if (!warp_wait(&acc_empty[buf], (uint32_t)((i >> 1) & 1) ^ 1u, &abort_flag) ||
                !warp_wait(&full[s], (uint32_t)ph, &abort_flag) ||
                !warp_wait(&pfull[ps], (uint32_t)((i / kPartStages) & 1), &abort_flag)) {
                set_timeout(p.ctl, &abort_flag);
                break;
            }
            tc_fence_after();
            const uint32_t st = smem_addr(ring + (size_t)s * kA);
            const uint32_t hs = smem_addr(parts + (size_t)ps * kParts * NT * kTileBytes);
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
                mma_bf16_if(lead, tmem + (uint32_t)((buf * halves + kk / per) * NX), smem_desc(st + kk * 32),
                         smem_desc(hs + kk * 32), idesc, kk % per ? 1u : 0u);
            mma_commit_if(lead, &empty[s]);
            mma_commit_if(lead, &pempty[ps]);
            mma_commit_if(lead, &acc_full[buf]);
            if (++s == S) { s = 0; ph ^= 1; }
        }
        consumed_s = i;
        mma_commit_if(lead, mma_done);
    } else if (warp >= 2 && warp < kEpi0) {
        grid_dependency_wait();   // h is written by the preceding gate/up kernel
        auto load = [&](int r, int c, int step, float4 &lo, float4 &hi) {
            const int m = m0 + r, k = ((u0 + step) % KBn) * BK + c * 8;
            if (m >= p.B || k >= p.N) return;
            const float *src = p.h + (size_t)m * p.ldh + k;   // (ldh is a multiple of 8)
            if (k + 8 <= p.N) {
                lo = reinterpret_cast<const float4 *>(src)[0];
                hi = reinterpret_cast<const float4 *>(src)[1];
            } else {   // columns past N hold anything
                const int left = p.N - k;
                lo.x = src[0];
                if (left > 1) lo.y = src[1];
                if (left > 2) lo.z = src[2];
                if (left > 3) lo.w = src[3];
                if (left > 4) hi.x = src[4];
                if (left > 5) hi.y = src[5];
                if (left > 6) hi.z = src[6];
            }
        };
        if (!cut_tiles<kLoraTok>(parts, NT, nu, pfull, pempty, &abort_flag, load)) set_timeout(p.ctl, &abort_flag);
    } else if (warp >= kEpi0) {
        grid_dependency_wait();   // y is cleared, w and the keep bytes written by the preceding kernel
        const int et = threadIdx.x - 32 * kEpi0;
        for (int i = et; i < NT * kLoraWRow; i += kLoraEpiThreads) {
            const int j = i / kLoraWRow, q = i % kLoraWRow;
            ws[j][q] = m0 + j < p.B && q < p.r ? p.scale * p.wsum[(size_t)(m0 + j) * kLoraWRow + q] : 0.f;
        }
        named_barrier(1, kLoraEpiThreads);
        __shared__ int warp_sums[kLoraEpiThreads / 32];
        if (blockIdx.y == 0)
            for (int m = blockIdx.x; p.lists.idx && m < p.B; m += gridDim.x)
                write_keep_list(p.lists, m, et, kLoraEpiThreads, warp_sums, 1);
        const int quad = warp & 3, grp = (warp - kEpi0) >> 2;
        const int c0 = 16 * grp;
        const bool busy = c0 < NT;
        const uint32_t lane0 = tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)c0;
        float(*T)[33] = tr[warp - kEpi0];
        const int te = lane >> 1, r0 = (lane & 1) * 16;   // this lane's token in the block, first row
        float acc[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) acc[e] = 0.f;
        for (int i = 0; i < nu; ++i) {
            const int buf = i & 1, u = u0 + i, d = u / KBn;
            if (!mbar_wait(&acc_full[buf], (uint32_t)((i >> 1) & 1), &abort_flag)) {
                set_timeout(p.ctl, &abort_flag);
                break;
            }
            tc_fence_after();
            if (busy) {
                float sum[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) sum[e] = 0.f;
                for (int f = 0; f < halves; ++f) {
                    float v[kParts][16];
#pragma unroll
                    for (int k = 0; k < kParts; ++k)
                        tmem_ld16(lane0 + (uint32_t)((buf * halves + f) * NX + k * NT), v[k]);
                    tmem_ld_wait();
#pragma unroll
                    for (int e = 0; e < 16; ++e) sum[e] += (v[2][e] + v[1][e]) + v[0][e];
                }
#pragma unroll
                for (int e = 0; e < 16; ++e) acc[e] += sum[e];
            }
            warp_arrive_tmem(&acc_empty[buf], lane);
            if (i + 1 < nu && (u + 1) / KBn == d) continue;
            // the last unit of this output tile: 32 rows x 16 tokens through shared memory, so that each
            // lane adds four vectors of four hidden units of one token
            if (busy) {
                const int row = d * BM + 32 * quad + lane;
                if (d * KBn >= u0 && row < p.H) {   // this CTA has the tile's first unit
                    float l[16];
#pragma unroll
                    for (int e = 0; e < 16; ++e) l[e] = 0.f;
                    for (int q = 0; q < p.r; q += 4) {   // (ranks are multiples of 8)
                        float b[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) b[k] = __uint_as_float((uint32_t)p.bd[(size_t)(q + k) * p.H + row] << 16);
#pragma unroll
                        for (int e = 0; e < 16; ++e) {
                            const float4 w = *reinterpret_cast<const float4 *>(&ws[c0 + e][q]);
                            l[e] = fmaf(w.w, b[3], fmaf(w.z, b[2], fmaf(w.y, b[1], fmaf(w.x, b[0], l[e]))));
                        }
                    }
#pragma unroll
                    for (int e = 0; e < 16; ++e) acc[e] += l[e];
                }
#pragma unroll
                for (int e = 0; e < 16; ++e) T[e][lane] = acc[e];
                __syncwarp();
                const int j = m0 + c0 + te, h0 = d * BM + 32 * quad + r0;
                if (j < p.B && c0 + te < NT) {
                    float *dst = p.y + (size_t)j * p.H + h0;
#pragma unroll
                    for (int k = 0; k < 4; ++k)   // H is a multiple of 8: a vector is in range or not at all
                        if (h0 + 4 * k < p.H)
                            red_add_v4(dst + 4 * k, T[te][r0 + 4 * k], T[te][r0 + 4 * k + 1], T[te][r0 + 4 * k + 2],
                                       T[te][r0 + 4 * k + 3]);
                }
                __syncwarp();
            }
#pragma unroll
            for (int e = 0; e < 16; ++e) acc[e] = 0.f;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
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
cudaError_t launch_lora_gate_up(LoraGuParams &p, const sats_layer *layer, const void *x, int mt, cudaStream_t stream)
{
    p.w_bytes = 2 * p.R * kTileBytes;
    p.stage_bytes = p.w_bytes + (F32 ? 0 : p.NT * kTileBytes);
    const int parts = F32 ? kPartStages * kParts * p.NT * kTileBytes : 0;
    // the up tile's MMA reads 128 rows from row R (rows R..127 of D are not used)
    const int over = (p.R + BM) * kTileBytes - p.stage_bytes;
    const int slack = over > 0 ? ((over + 1023) & ~1023) : 0;
    const int totals = F32 ? 32 * kLoraEpiThreads * 4 : 0;
    // (half of the totals fit beside the ring's budget, zs and the barriers)
    p.stages = stages_for(p.stage_bytes, kSmemBudget - parts - slack - totals / 2);
    p.ring_bytes = p.stages * p.stage_bytes + slack;
    p.halves = F32 && p.NT > 16 ? 1 : 2;
    // One sum over 64 blocks is as near to 64 bits as the fused kernel's (hidden 4096, fp32: 3.0e-7 both); longer ones go
    // in parts (8192 / intermediate 3584, bf16: 3.4e-7 as one sum, 2.2e-7 so, 2.7e-7 on the fused kernel; 1 % of the call).
    p.sub = p.KBh <= 64 ? p.KBh : 32;
    p.tmem_cols = tmem_cols_for(2 * p.halves * 2 * (F32 ? kParts : 1) * p.NT);
    CUtensorMap mX{};
    if (!F32 && !make_map(&mX, x, (uint64_t)p.B, (uint64_t)p.H, (uint64_t)p.H * 2, (uint32_t)p.NT))
        return cudaErrorInvalidValue;
    static std::atomic<int> cfg[64];
    const size_t smem = smem_for(1, p.ring_bytes + parts + totals);
    const cudaError_t e = set_smem(lora_gate_up_kernel<F32>, smem, cfg);
    if (e != cudaSuccess) return e;
    return launch_pdl_cfg(lora_gate_up_kernel<F32>, dim3(mt, layer->tc_T), kLoraGuThreads<F32>, smem, stream, mX, p);
}

}  // namespace
}  // namespace tc

cudaError_t launch_gate_act(const sats_layer *layer, const uint16_t *x, int B, float *a, cudaStream_t stream)
{
    return layer->H <= tc::kKeepH ? tc::launch_gate_precise<false, tc::kPreciseTok, false, true>(layer, x, B, a, nullptr, stream)
                                  : tc::launch_gate_precise<false, tc::kPreciseTok>(layer, x, B, a, nullptr, stream);
}

cudaError_t launch_gate_act_f32(const sats_layer *layer, const float *x, int B, float *a, int *status,
                                cudaStream_t stream)
{
    return B <= 64 ? tc::launch_gate_precise<true, 64>(layer, x, B, a, status, stream)
                   : tc::launch_gate_precise<true, tc::kPreciseTok>(layer, x, B, a, status, stream);
}

cudaError_t launch_up_f32(const sats_layer *layer, const float *x, int B, const float *a, uint16_t *hhi, uint16_t *hlo,
                          int *status, cudaStream_t stream)
{
    float *const in = const_cast<float *>(a);   // (read only)
    return B <= 64 ? tc::launch_gate_precise<true, 64, true>(layer, x, B, in, status, stream, hhi, hlo)
                   : tc::launch_gate_precise<true, tc::kPreciseTok, true>(layer, x, B, in, status, stream, hhi, hlo);
}

// Scratch of a LoRA batch inside the tensor-core region of a workspace: z and w where the other
// paths keep bf16 copies of x (4 H bytes per token), h in fp32 where they keep its two parts.
static int lora_slices(int H) { return H / 128 < 1 ? 1 : (H / 128 > 8 ? 8 : H / 128); }

bool lora_tc_ok(int H, int B)
{
    const int need = lora_slices(H) * tc::kLoraZRow * 4 + tc::kLoraWRow * 4;
    // Two tokens of hidden sizes above 4096 stay two passes: at 85 % sparsity those read less than all weights
    // once (hidden 4448 / intermediate 6883: 73 us in passes, 81 here).  (B is a grid dimension.)
    return use_tc_path(H, B) && B >= 3 && B <= 65535 && need <= 4 * H;
}

cudaError_t run_lora_tc(const sats_layer *layer, const sats_lora *lora, bool x_f32, const void *x, int B, float t_l,
                        float *y, int32_t *active_idx, int32_t *active_cnt, void *tc_ws, int *ctl, cudaStream_t stream)
{
    using namespace tc;
    const int H = layer->H, N = layer->N;
    const TcRegions W = tc_regions(H, N, B);
    char *base = static_cast<char *>(tc_ws);
    const int slices = lora_slices(H);
    float *z = reinterpret_cast<float *>(base + W.x);
    float *wsum = z + (size_t)B * slices * kLoraZRow;
    float *h = reinterpret_cast<float *>(base + W.h);
    uint8_t *keep = reinterpret_cast<uint8_t *>(base + W.keep);
    auto failed = [](cudaError_t e, const char *where) {
        cuda_fail(e, where);
        return e;
    };
    cudaError_t e =
        x_f32 ? launch_pdl_threads(lora_z_kernel<float>, dim3(slices, B), 256, stream, static_cast<const float *>(x), H,
                                   static_cast<const uint16_t *>(lora->agu), lora->r, z, wsum)
              : launch_pdl_threads(lora_z_kernel<uint16_t>, dim3(slices, B), 256, stream,
                                   static_cast<const uint16_t *>(x), H, static_cast<const uint16_t *>(lora->agu),
                                   lora->r, z, wsum);
    if (e != cudaSuccess) return failed(e, "adapter input kernel launch");

    const int mt = (B + kLoraTok - 1) / kLoraTok;
    LoraGuParams gp{};
    gp.w = layer->gu_blk;
    gp.x = x_f32 ? static_cast<const float *>(x) : nullptr;
    gp.B = B;
    gp.H = H;
    gp.N = N;
    gp.R = layer->tc_R;
    gp.KBh = layer->tc_kbh;
    gp.NT = ((B + mt - 1) / mt + 15) & ~15;
    gp.t_l = t_l;
    gp.scale = lora->scale;
    gp.blk = lora->blk;
    gp.r = lora->r;
    gp.z = z;
    gp.slices = slices;
    gp.h = h;
    gp.ldh = layer->ldn;
    gp.keep = active_idx ? keep : nullptr;
    gp.keep_stride = (N + 15) & ~15;
    gp.y = y;
    gp.wsum = wsum;
    gp.ctl = ctl;
    e = x_f32 ? launch_lora_gate_up<true>(gp, layer, x, mt, stream) : launch_lora_gate_up<false>(gp, layer, x, mt, stream);
    if (e != cudaSuccess) return failed(e, "adapted gate/up kernel launch");

    LoraDownParams dp{};
    dp.w = layer->wd_blk;
    dp.h = h;
    dp.ldh = layer->ldn;
    dp.B = B;
    dp.H = H;
    dp.N = N;
    dp.NT = gp.NT;
    dp.halves = 2;
    dp.KBn = layer->tc_kbn;
    dp.units = layer->tc_dt * dp.KBn;
    dp.bd = lora->bd;
    dp.r = lora->r;
    dp.scale = lora->scale;
    dp.y = y;
    dp.wsum = wsum;
    dp.lists = {keep, gp.keep_stride, N, active_idx, active_cnt, nullptr};
    dp.ctl = ctl;
    const int parts = kPartStages * kParts * dp.NT * kTileBytes;
    dp.stages = stages_for(BM * kTileBytes, kSmemBudget - parts);
    dp.ring_bytes = dp.stages * BM * kTileBytes;
    dp.tmem_cols = tmem_cols_for(2 * dp.halves * kParts * dp.NT);
    static std::atomic<int> cfg[64];
    const size_t smem = smem_for(1, dp.ring_bytes + parts);
    if ((e = set_smem(lora_down_kernel, smem, cfg)) != cudaSuccess) return failed(e, "shared-memory attribute");
    const int sms = sm_count();
    e = launch_pdl_cfg(lora_down_kernel, dim3(dp.units < sms ? dp.units : sms, mt), kLoraDownThreads, smem, stream, dp);
    return e == cudaSuccess ? e : failed(e, "adapted down kernel launch");
}

}  // namespace sats
