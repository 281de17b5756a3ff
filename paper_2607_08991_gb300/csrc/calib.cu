// calib.cu -- SATS threshold calibration (Sec. 3.1, Eqs. 6-10; Sec. 4 guardrail)
// on the GPU, with the same kernels that run the thresholded MLP.
//
// Eq. 6, Err_l(t) = E_x[ ||y(x) - y~_t(x)|| / (||y(x)|| + eps) ], is evaluated for
// many candidate thresholds at once per block: on the tensor cores from one pass
// over the gate and up projections and one GEMM over the dropped neurons of all
// candidates, for one or two inputs from the fused kernel's outputs (the dense one,
// then one per candidate); small reduction kernels add the per-token relative
// distortion and realised sparsity into device accumulators.  Eqs. 7-10 (budget selection) run on the
// host; the coarse-to-fine driver chains everything for a whole stack.
#include <algorithm>
#include <cmath>
#include <cstddef>
#include <cstring>
#include <vector>

#include "common.cuh"
#include "internal.h"

namespace sats {
namespace {

constexpr int kErrGroup = 32;     // candidate thresholds per group of Eq. 6
// Bytes of a group's rows (candidates x inputs: h's two parts and the output) at most
constexpr size_t kErrRowBytes = (size_t)512 << 20;
constexpr size_t kErrKeep = (size_t)1 << 30;   // of a calibration's kept inputs, at most

size_t al256(size_t v) { return (v + 255) & ~(size_t)255; }

// A launch that may start while the preceding kernel ends; the kernel waits for that before it reads or writes.
template <typename... KArgs, typename... Args>
cudaError_t launch_after(void (*kernel)(KArgs...), dim3 grid, int threads, cudaStream_t st, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// out[b] = x[b] / sqrt(mean_i x[b][i]^2 + eps) * w  (one CTA per row).
__global__ void __launch_bounds__(256) rmsnorm_kernel(const float *__restrict__ x, int H, const float *__restrict__ w,
                                                      float eps, float *__restrict__ out)
{
    grid_dependency_wait();
    grid_launch_dependents();
    const float *xr = x + (size_t)blockIdx.x * H;
    float *o = out + (size_t)blockIdx.x * H;
    __shared__ float red[8];
    float s = 0.f;
    for (int i = threadIdx.x; i < H; i += 256) s = fmaf(xr[i], xr[i], s);
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    float tot = 0.f;
    for (int i = 0; i < 8; ++i) tot += red[i];
    const float inv = 1.0f / sqrtf(tot / (float)H + eps);
    for (int i = threadIdx.x; i < H; i += 256) o[i] = xr[i] * inv * w[i];
}

// Token c: acc[0] += ||yd_c - yk_c|| / (||yd_c|| + eps), acc[1] += (N - kept_c) / N.
__global__ void __launch_bounds__(256) err_accum_kernel(const float *__restrict__ yd, const float *__restrict__ yk,
                                                        int H, const int32_t *__restrict__ cnt, int N, float eps,
                                                        double *__restrict__ acc)
{
    const int c = blockIdx.x;
    const float *a = yd + (size_t)c * H, *b = yk + (size_t)c * H;
    double dd = 0.0, yy = 0.0;
    for (int i = threadIdx.x; i < H; i += 256) {
        const double d = (double)a[i] - (double)b[i];
        dd += d * d;
        yy += (double)a[i] * (double)a[i];
    }
    __shared__ double r0[8], r1[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        dd += __shfl_xor_sync(0xffffffffu, dd, o);
        yy += __shfl_xor_sync(0xffffffffu, yy, o);
    }
    if ((threadIdx.x & 31) == 0) {
        r0[threadIdx.x >> 5] = dd;
        r1[threadIdx.x >> 5] = yy;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double d = 0.0, y = 0.0;
        for (int i = 0; i < 8; ++i) {
            d += r0[i];
            y += r1[i];
        }
        atomicAdd(acc, sqrt(d) / (sqrt(y) + (double)eps));
        atomicAdd(acc + 1, (double)(N - cnt[c]) / (double)N);
    }
}

// Candidates of one group: the threshold of each; with dev, candidate k's is dev[at[k]].
struct Candidates {
    float t[kErrGroup];
    int at[kErrGroup];
    const float *dev;
};

// The rows of a group of K candidates, in bf16 parts: row (0, c) is h of every neuron (for the dense output), row
// (k + 1, c) is h where |a| < t_k, 0 elsewhere; counts[k] += the neurons dropped.  h (hi, lo) is [C][ld], a [C][N],
// the rows [K + 1][C][ld]; ld is a multiple of 8, and columns N .. ld - 1 are never read as neurons.  Grid: (C,
// column blocks of 8 x 256).  Bound by its writes (4 K C N bytes, mostly into L2).
__global__ void __launch_bounds__(256) drop_rows_kernel(const float *__restrict__ a, const uint16_t *__restrict__ hhi,
                                                        const uint16_t *__restrict__ hlo, int C, int N, int ld,
                                                        const Candidates cand, int K, uint16_t *__restrict__ rhi,
                                                        uint16_t *__restrict__ rlo, unsigned long long *counts,
                                                        float4 *__restrict__ out, size_t n4)
{
    __shared__ unsigned dropped[kErrGroup];
    if (threadIdx.x < kErrGroup) dropped[threadIdx.x] = 0u;
    grid_dependency_wait();   // h and a are the gate/up kernel's
    grid_launch_dependents();
    // the rows' projection adds into out
    for (size_t i = ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 256 + threadIdx.x; i < n4;
         i += (size_t)gridDim.x * gridDim.y * 256)
        out[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    __syncthreads();
    const int c = blockIdx.x, n0 = (blockIdx.y * 256 + threadIdx.x) * 8;
    const bool in = n0 < N;
    float av[8];
    uint4 hh = make_uint4(0u, 0u, 0u, 0u), hl = hh;
    if (in) {
        const size_t at = (size_t)c * ld + n0;
        const float *ar = a + (size_t)c * N + n0;
        if ((N & 7) == 0) {
            const float4 p = reinterpret_cast<const float4 *>(ar)[0], q = reinterpret_cast<const float4 *>(ar)[1];
            av[0] = p.x; av[1] = p.y; av[2] = p.z; av[3] = p.w;
            av[4] = q.x; av[5] = q.y; av[6] = q.z; av[7] = q.w;
        } else {
#pragma unroll
            for (int e = 0; e < 8; ++e) av[e] = n0 + e < N ? ar[e] : 0.f;
        }
        hh = *reinterpret_cast<const uint4 *>(hhi + at);
        hl = *reinterpret_cast<const uint4 *>(hlo + at);
        *reinterpret_cast<uint4 *>(rhi + at) = hh;
        *reinterpret_cast<uint4 *>(rlo + at) = hl;
    }
    for (int k = 0; k < K; ++k) {
        const float t = cand.dev ? cand.dev[cand.at[k]] : cand.t[k];
        unsigned m[4] = {0u, 0u, 0u, 0u}, cnt = 0u;
        if (in) {
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                // not kept (Eqs. 4-5: a neuron is kept if |a| >= t)
                const bool drop = n0 + e < N && !(fabsf(av[e]) >= t);
                cnt += drop ? 1u : 0u;
                m[e / 2] |= drop ? (e & 1 ? 0xffff0000u : 0xffffu) : 0u;
            }
            const size_t at = ((size_t)(k + 1) * C + c) * ld + n0;
            *reinterpret_cast<uint4 *>(rhi + at) = make_uint4(hh.x & m[0], hh.y & m[1], hh.z & m[2], hh.w & m[3]);
            *reinterpret_cast<uint4 *>(rlo + at) = make_uint4(hl.x & m[0], hl.y & m[1], hl.z & m[2], hl.w & m[3]);
        }
        cnt = __reduce_add_sync(0xffffffffu, cnt);
        if ((threadIdx.x & 31) == 0 && cnt) atomicAdd(dropped + k, cnt);
    }
    __syncthreads();
    if (threadIdx.x < K && dropped[threadIdx.x]) atomicAdd(counts + threadIdx.x, (unsigned long long)dropped[threadIdx.x]);
}

// A sum of squares as an unevaluated sum of three floats (the product's error by FMA, the sums' by Knuth's TwoSum),
// more than the 53 bits of a double: this GPU's 64-bit rate is 1/64 of its 32-bit one (1344 rows of 4096: 33 us in
// doubles, 10 so).
struct SquareSum {
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
    static __device__ float two_sum(float &s, float v)   // s += v; returns what the sum was rounded by
    {
        const float t = __fadd_rn(s, v), b = __fadd_rn(t, -s);
        const float e = __fadd_rn(__fadd_rn(s, -__fadd_rn(t, -b)), __fadd_rn(v, -b));
        s = t;
        return e;
    }
    __device__ void join(float v0, float v1, float v2)
    {
        const float e0 = two_sum(s1, two_sum(s0, v0)), e1 = two_sum(s1, v1);
        s2 += (e0 + e1) + v2;
    }
    __device__ void add(float v)
    {
        const float p = __fmul_rn(v, v);
        join(p, __fmaf_rn(v, v, -p), 0.f);
    }
    __device__ double value() const { return ((double)s2 + (double)s1) + (double)s0; }
};

// sq[r] = ||row r||^2 of the group's outputs [rows][H].  Grid: rows.
__global__ void __launch_bounds__(256) row_squares_kernel(const float *__restrict__ out, int H, double *__restrict__ sq)
{
    grid_dependency_wait();
    grid_launch_dependents();
    const float *row = out + (size_t)blockIdx.x * H;
    SquareSum s;
    for (int i = threadIdx.x; i < (H >> 2); i += 256) {   // H is a multiple of 8
        const float4 p = reinterpret_cast<const float4 *>(row)[i];
        s.add(p.x); s.add(p.y); s.add(p.z); s.add(p.w);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        s.join(__shfl_xor_sync(0xffffffffu, s.s0, o), __shfl_xor_sync(0xffffffffu, s.s1, o),
               __shfl_xor_sync(0xffffffffu, s.s2, o));
    __shared__ float part[8][3];
    __shared__ double wide[8];
    __shared__ bool again;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        part[warp][0] = s.s0;
        part[warp][1] = s.s1;
        part[warp][2] = s.s2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) s.join(part[w][0], part[w][1], part[w][2]);
        const double v = s.value();
        again = !(v > 1e-24 && v < 1e36);   // 32-bit squares may have over- or underflown
        sq[blockIdx.x] = v;
    }
    __syncthreads();
    if (!again) return;
    double d = 0.0;
    for (int i = threadIdx.x; i < H; i += 256) d += (double)row[i] * (double)row[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    if (lane == 0) wide[warp] = d;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) d += wide[w];
        sq[blockIdx.x] = d;
    }
}

// err[k] += sum_c ||d_kc|| / (||y_c|| + eps), with d = y - y~_t (the dropped neurons' output) and y the dense one:
// sq is [K + 1][C], the dense rows first.  A dense output that is not finite has no distortion (infinity less infinity,
// were the outputs subtracted).  Grid: K.
__global__ void __launch_bounds__(256) err_ratio_kernel(const double *__restrict__ sq, int C, float eps,
                                                        double *__restrict__ err)
{
    grid_dependency_wait();
    grid_launch_dependents();
    const double *d = sq + (size_t)(blockIdx.x + 1) * C;
    double s = 0.0;
    for (int c = threadIdx.x; c < C; c += 256)
        s += isfinite(sq[c]) ? sqrt(d[c]) / (sqrt(sq[c]) + (double)eps) : (double)NAN;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    __shared__ double part[8];
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int w = 1; w < 8; ++w) s += part[w];
        err[blockIdx.x] += s;   // (the groups and their kernels follow one another)
    }
}

// What the candidates of one block are formed from.
struct ErrInputs {
    float *a;                // [C][N]: SiLU(x W_gate)
    uint16_t *hhi, *hlo;     // [C][ldn]: a u of every neuron
    static size_t a_bytes(int N, int C) { return al256((size_t)C * N * 4); }
    static size_t h_bytes(int N, int C) { return al256((size_t)C * ((N + 7) & ~7) * 4); }
    ErrInputs(void *a, void *h, int N, int C)
        : a(static_cast<float *>(a)), hhi(static_cast<uint16_t *>(h)), hlo(hhi + (size_t)C * ((N + 7) & ~7)) {}
};

// Workspace of Eq. 6.  Batches on the fused kernel (at most two tokens) compare whole outputs
// (yd, yk, idx, cnt); batches on the tensor cores project the dropped neurons of a group of
// candidates (a: the gate activations of a call that has no other place for them; rows, y: the group's outputs, sq: their
// squared norms).  mlp is an ordinary workspace; h takes the place of its h.
struct ErrLayout {
    size_t mlp, yd, yk, idx, cnt, a, h, rhi, rlo, y, sq, acc, total;
};

// Candidates of a group and inputs of a chunk: as many candidates as a launch takes, and inputs within kErrRowBytes (but
// one, whose rows are 140 MB at the largest layer), the dense rows among them.
struct ErrGroup {
    int candidates, inputs;
    size_t rows() const { return (size_t)(candidates + 1) * inputs; }
};

ErrGroup err_group(int H, int N, int C, int K)
{
    const int g = std::max(1, std::min(K, kErrGroup));
    const size_t row = ((size_t)((N + 7) & ~7) + H) * 4, fit = std::max<size_t>(1, kErrRowBytes / (row * (g + 1)));
    const int chunks = (int)((C + fit - 1) / fit);
    return {g, (C + chunks - 1) / chunks};
}

ErrLayout err_layout(int H, int N, int C, int K, bool own_a)
{
    ErrLayout L{};
    size_t off = 0;
    auto take = [&](size_t bytes) {
        const size_t at = off;
        off += al256(bytes);
        return at;
    };
    L.mlp = take(ws_layout(H, N, C).total);
    if (use_tc_path(H, C)) {
        const size_t ldn = ((size_t)N + 7) & ~(size_t)7, rows = err_group(H, N, C, K).rows();
        if (own_a) L.a = take(ErrInputs::a_bytes(N, C));
        L.h = L.mlp + ws_layout(H, N, C).tc + tc_regions(H, N, C).h;
        L.rhi = take(rows * ldn * 2);
        L.rlo = take(rows * ldn * 2);
        L.y = take(rows * H * sizeof(float));
        L.sq = take(rows * sizeof(double));
        L.acc = take((size_t)std::max(K, 1) * (sizeof(double) + sizeof(unsigned long long)));   // ErrSums
    } else {
        L.yd = take((size_t)C * H * sizeof(float));
        L.yk = take((size_t)C * H * sizeof(float));
        L.idx = take((size_t)C * N * sizeof(int32_t));
        L.cnt = take((size_t)C * sizeof(int32_t));
        L.acc = take((size_t)2 * (K > 0 ? K : 1) * sizeof(double));
    }
    L.total = off;
    return L;
}

// Eq. 6 on the tensor cores: a and h = a u of every neuron once, in fp32 accuracy, then y - y~_t = (h where |a| < t)
// W_down directly, for all candidates of a group as the rows of one GEMM, and y itself as C more of its rows.
// That is one pass over W_gate and W_up and one over W_down per group instead of both per candidate (20 passes of
// 72 us for 19 candidates of 64 inputs on the Llama-shaped layer).  What its accuracy rests on: an accumulator that is
// truncated after every K = 16 step comes out short, the shorter the longer its chain.  g and u short by 1e-5 change a
// and h of small and of large |a| by different shares, so they are taken in fp32 accuracy; y and y - y~_t take the same
// chains and keep little of it in their ratio.  Against 64 bits (2-norm over the candidates), with both / with h from
// the batched gate/up kernel and y from a GEMM of its own: that layer 2.6e-7 / 1.6e-6, hidden 2048 / intermediate
// 5633, 48 inputs 2.8e-7 / 2.4e-6.  What bounds it: the down projection's MMAs (two per product: h's high and low
// parts).
struct ErrSums {
    double *err;                     // [K]
    unsigned long long *dropped;     // [K]
    static size_t bytes(int K) { return (size_t)K * (sizeof(double) + sizeof(unsigned long long)); }
    ErrSums(void *p, int K) : err(static_cast<double *>(p)), dropped(reinterpret_cast<unsigned long long *>(err + K)) {}
};

// The dense rows and those of kg candidates (cand), and their product with W_down, into out [kg + 1][C][H].
sats_status enqueue_rows(const sats_layer *layer, const float *a, const uint16_t *hhi, const uint16_t *hlo, int C,
                         const Candidates &cand, int kg, unsigned long long *dropped, float *out, char *base,
                         const ErrLayout &W, int *ctl, cudaStream_t st)
{
    const int H = layer->H, N = layer->N, ld = layer->ldn;
    uint16_t *rhi = reinterpret_cast<uint16_t *>(base + W.rhi), *rlo = reinterpret_cast<uint16_t *>(base + W.rlo);
    const cudaError_t e = launch_after(drop_rows_kernel, dim3(C, (ld / 8 + 255) / 256), 256, st, a, hhi, hlo, C, N, ld, cand,
                                       kg, rhi, rlo, dropped, reinterpret_cast<float4 *>(out), (size_t)(kg + 1) * C * H / 4);
    if (e != cudaSuccess) return cuda_fail(e, "dropped rows kernel launch");
    return run_tc_down(layer, rhi, rlo, (kg + 1) * C, out, ctl, st) == cudaSuccess ? SATS_OK : SATS_ECUDA;
}

__global__ void __launch_bounds__(256) add_rows_kernel(float4 *__restrict__ x, const float4 *__restrict__ y, size_t n4)
{
    grid_dependency_wait();
    grid_launch_dependents();
    const size_t i = blockIdx.x * (size_t)256 + threadIdx.x;
    if (i >= n4) return;
    const float4 a = x[i], b = y[i];
    x[i] = make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

// x += the dense output, projected on its own: up to 256 inputs take the batched-decode kernel, whose shorter
// accumulator chains are the more accurate ones.  In chunks of what the groups' output holds (rows).
sats_status enqueue_residual(const sats_layer *layer, float *x, int C, const ErrInputs &in, size_t rows, char *base,
                             const ErrLayout &W, int *ctl, cudaStream_t st)
{
    const int H = layer->H;
    float *y = reinterpret_cast<float *>(base + W.y);
    for (size_t c0 = 0; c0 < (size_t)C; c0 += rows) {
        const int m = (int)std::min(rows, C - c0);
        const size_t n = (size_t)m * H, at = c0 * layer->ldn;
        cudaError_t e = cudaMemsetAsync(y, 0, n * sizeof(float), st);
        if (e != cudaSuccess) return cuda_fail(e, "dense output clear");
        if (run_tc_down(layer, in.hhi + at, in.hlo + at, m, y, ctl, st) != cudaSuccess) return SATS_ECUDA;
        e = launch_after(add_rows_kernel, dim3((unsigned)((n / 4 + 255) / 256)), 256, st,
                         reinterpret_cast<float4 *>(x + c0 * H), reinterpret_cast<const float4 *>(y), n / 4);
        if (e != cudaSuccess) return cuda_fail(e, "residual kernel launch");
    }
    return SATS_OK;
}

// Enqueues the sums for K candidates: thresholds t (host), or q[at(k)] on the device where q is given; group: that of the
// call's workspace.  sums: cleared device memory of ErrSums::bytes(K).
template <typename At>
sats_status enqueue_err(const sats_layer *layer, const ErrInputs &in, int C, const float *t, const float *q, At at, int K,
                        float eps, const ErrSums &sums, const ErrGroup &group, char *base, const ErrLayout &W, int *ctl,
                        cudaStream_t st)
{
    float *out = reinterpret_cast<float *>(base + W.y);
    double *sq = reinterpret_cast<double *>(base + W.sq);
    for (int c0 = 0; c0 < C; c0 += group.inputs) {
        const int cc = std::min(group.inputs, C - c0);
        const size_t h0 = (size_t)c0 * layer->ldn;
        for (int k0 = 0; k0 < K; k0 += group.candidates) {
            const int kg = std::min(group.candidates, K - k0);
            Candidates cand{};
            cand.dev = q;
            for (int k = 0; k < kg; ++k) {
                cand.t[k] = q ? 0.f : t[k0 + k];
                cand.at[k] = at(k0 + k);
            }
            const sats_status s = enqueue_rows(layer, in.a + (size_t)c0 * layer->N, in.hhi + h0, in.hlo + h0, cc, cand, kg,
                                               sums.dropped + k0, out, base, W, ctl, st);
            if (s != SATS_OK) return s;
            cudaError_t e = launch_after(row_squares_kernel, dim3((kg + 1) * cc), 256, st, (const float *)out, layer->H, sq);
            if (e == cudaSuccess)
                e = launch_after(err_ratio_kernel, dim3(kg), 256, st, (const double *)sq, cc, eps, sums.err + k0);
            if (e != cudaSuccess) return cuda_fail(e, "error reduction kernel launch");
        }
    }
    return SATS_OK;
}

// The means of a candidate table's rows from their sums (host copies).
void err_means(const void *host_sums, int K, int C, int N, double *err, double *sp)
{
    const char *p = static_cast<const char *>(host_sums);
    for (int k = 0; k < K; ++k) {
        double e;
        unsigned long long d;
        std::memcpy(&e, p + sizeof(double) * k, sizeof e);
        std::memcpy(&d, p + sizeof(double) * K + sizeof d * k, sizeof d);
        err[k] = e / C;
        sp[k] = (double)d / ((double)C * N);
    }
}

sats_status layer_err_tc(const sats_layer *layer, const float *x, int C, const float *t, int K, float eps, double *err,
                         double *sp, char *base, const ErrLayout &W, cudaStream_t st)
{
    char *mlp = base + W.mlp;
    const size_t sum_bytes = ErrSums::bytes(K);
    cudaError_t e = clear_fused_state(mlp, layer->H, layer->N, C, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(base + W.acc, 0, sum_bytes, st);
    if (e != cudaSuccess) return cuda_fail(e, "layer error workspace clear");
    const ErrInputs in(base + W.a, base + W.h, layer->N, C);
    int *ctl = reinterpret_cast<int *>(mlp + ws_layout(layer->H, layer->N, C).ctl);
    e = launch_gate_act_f32(layer, x, C, in.a, ctl + kCtlStatus, st);
    if (e == cudaSuccess) e = launch_up_f32(layer, x, C, in.a, in.hhi, in.hlo, ctl + kCtlStatus, st);
    if (e != cudaSuccess) return cuda_fail(e, "gate and up kernels launch");
    sats_status s = enqueue_err(layer, in, C, t, nullptr, [](int k) { return k; }, K, eps, ErrSums(base + W.acc, K),
                                err_group(layer->H, layer->N, C, K), base, W, ctl, st);
    if (s != SATS_OK) return s;
    std::vector<char> h(sum_bytes);
    e = cudaMemcpyAsync(h.data(), base + W.acc, sum_bytes, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "layer error read-back");
    s = sats_get_error(mlp, ws_layout(layer->H, layer->N, C).total, st);
    if (s != SATS_OK) return s;
    err_means(h.data(), K, C, layer->N, err, sp);
    return SATS_OK;
}

struct SatsLayout {
    size_t x, n, sel, q, sums, a, in_each, err, total;   // in_each: 0 if the blocks share one
};

SatsLayout sats_layout(int H, int N, int C, int L, int K0, int K)
{
    SatsLayout S{};
    size_t off = 0;
    S.x = off;
    off += al256((size_t)C * H * sizeof(float));
    S.n = off;
    off += al256((size_t)L * C * H * sizeof(float));
    S.sel = off;
    off += al256(select_multi_ws_bytes(kSelRanks));
    S.q = off;   // every block's percentiles: the coarse candidates, the largest |a|, the guardrail's
    off += al256((size_t)L * (K0 + 1) * sizeof(float));
    S.sums = off;   // every block's ErrSums
    off += al256((size_t)L * ErrSums::bytes(K));
    // every block's a and h, kept from the coarse candidates for the fine ones, up to kErrKeep bytes; else one a (and the
    // h of Eq. 6's workspace)
    const size_t each = use_tc_path(H, C) ? ErrInputs::a_bytes(N, C) + ErrInputs::h_bytes(N, C) : 0;
    S.in_each = each * L <= kErrKeep ? each : 0;
    S.a = off;
    off += S.in_each ? S.in_each * L : ErrInputs::a_bytes(N, C);
    S.err = off;
    off += err_layout(H, N, C, K, false).total;
    S.total = off;
    return S;
}

bool bad_t(double t) { return std::isnan(t) || t < 0.0; }

}  // namespace
}  // namespace sats

using namespace sats;

extern "C" {

sats_status sats_rmsnorm(const float *x, int B, int H, const float *w, float eps, float *out, void *stream)
{
    if (B < 0 || H < 1 || std::isnan(eps) || eps < 0.0f) return SATS_EINVAL;
    if (B == 0) return SATS_OK;
    if (!x || !w || !out) return SATS_EINVAL;
    const cudaError_t e = launch_after(rmsnorm_kernel, dim3(B), 256, static_cast<cudaStream_t>(stream), x, H, w, eps, out);
    return e == cudaSuccess ? SATS_OK : cuda_fail(e, "rmsnorm kernel launch");
}

sats_status sats_gate_act_f32(const sats_layer *layer, const float *x, int B, float *a, void *stream)
{
    if (!layer || B < 0) return SATS_EINVAL;
    if (B == 0) return SATS_OK;
    if (!x || !a || (reinterpret_cast<uintptr_t>(x) & 15u)) return SATS_EINVAL;
    const cudaError_t e = launch_gate_act_f32(layer, x, B, a, nullptr, static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? SATS_OK : cuda_fail(e, "gate activation kernel launch");
}

size_t sats_layer_err_workspace_bytes(int H, int N, int C, int K)
{
    if (H < 8 || H > kMaxH || (H % 8) != 0 || N < 1 || N > kMaxN || C < 1 || K < 0) return 0;
    return err_layout(H, N, C, K, true).total;
}

sats_status sats_layer_err(const sats_layer *layer, const float *x, int C, const float *t, int K, float eps,
                           double *err, double *sp, void *ws, size_t ws_bytes, void *stream)
{
    if (!layer || !x || C < 1 || K < 0 || !ws || (reinterpret_cast<uintptr_t>(x) & 15u) ||
        (reinterpret_cast<uintptr_t>(ws) & 255u))
        return SATS_EINVAL;
    if (K > 0 && (!t || !err || !sp)) return SATS_EINVAL;
    if (std::isnan(eps) || eps < 0.0f) return SATS_EINVAL;
    for (int k = 0; k < K; ++k)
        if (bad_t(t[k])) return SATS_EINVAL;
    const int H = layer->H, N = layer->N;
    const ErrLayout W = err_layout(H, N, C, K, true);
    if (ws_bytes < W.total) return SATS_ENOSPACE;
    if (K == 0) return SATS_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char *base = static_cast<char *>(ws);
    if (use_tc_path(H, C)) return layer_err_tc(layer, x, C, t, K, eps, err, sp, base, W, st);
    void *mlp = base + W.mlp;
    float *yd = reinterpret_cast<float *>(base + W.yd), *yk = reinterpret_cast<float *>(base + W.yk);
    int32_t *idx = reinterpret_cast<int32_t *>(base + W.idx), *cnt = reinterpret_cast<int32_t *>(base + W.cnt);
    double *acc = reinterpret_cast<double *>(base + W.acc);
    cudaError_t e = clear_fused_state(mlp, H, N, C, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(acc, 0, (size_t)2 * K * sizeof(double), st);
    if (e != cudaSuccess) return cuda_fail(e, "layer error workspace clear");
    const float zero = 0.0f;
    sats_status s = run_layer(layer, kXF32, x, C, &zero, nullptr, 0.f, nullptr, kOutY, yd, nullptr, nullptr,
                              nullptr, mlp, st);
    for (int k = 0; k < K && s == SATS_OK; ++k) {
        s = run_layer(layer, kXF32, x, C, &t[k], nullptr, 0.f, nullptr, kOutY, yk, idx, cnt, nullptr, mlp, st);
        if (s != SATS_OK) break;
        err_accum_kernel<<<C, 256, 0, st>>>(yd, yk, H, cnt, N, eps, acc + 2 * k);
        if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "error reduction kernel launch");
    }
    if (s != SATS_OK) return s;
    std::vector<double> h((size_t)2 * K);
    e = cudaMemcpyAsync(h.data(), acc, h.size() * sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "layer error read-back");
    s = sats_get_error(mlp, ws_layout(H, N, C).total, stream);
    if (s != SATS_OK) return s;
    for (int k = 0; k < K; ++k) {
        err[k] = h[2 * (size_t)k] / C;
        sp[k] = h[2 * (size_t)k + 1] / C;
    }
    return SATS_OK;
}

sats_status sats_sats_select(const double *t, const double *err, const double *sp, int L, int K, double s_tar,
                             int guard, double guard_t, double guard_sp, double *b_out, double *t_out,
                             double *S_out)
{
    if (L < 1 || K < 0 || !t_out || !b_out || !S_out || std::isnan(s_tar)) return SATS_EINVAL;
    if (K > 0 && (!t || !err || !sp)) return SATS_EINVAL;
    if (guard >= L || (guard >= 0 && (std::isnan(guard_t) || std::isnan(guard_sp)))) return SATS_EINVAL;
    // per block, candidate indices by decreasing threshold (stable: the first listed wins a tie)
    std::vector<std::vector<int>> order((size_t)L);
    std::vector<double> budgets(1, 0.0);
    for (int l = 0; l < L; ++l) {
        std::vector<int> &o = order[(size_t)l];
        for (int k = 0; k < K; ++k) {
            const size_t i = (size_t)l * K + k;
            if (std::isnan(t[i]) || std::isnan(err[i]) || std::isnan(sp[i])) return SATS_EINVAL;
            o.push_back(k);
            budgets.push_back(err[i]);
        }
        std::stable_sort(o.begin(), o.end(), [&](int p, int q) { return t[(size_t)l * K + p] > t[(size_t)l * K + q]; });
    }
    std::sort(budgets.begin(), budgets.end());
    budgets.erase(std::unique(budgets.begin(), budgets.end()), budgets.end());
    // Eq. 7 for one block at budget b: the largest admissible threshold (index, or -1 for t = 0)
    auto pick = [&](int l, double b) {
        for (int k : order[(size_t)l]) {
            const size_t i = (size_t)l * K + k;
            if (t[i] <= 0.0) break;
            if (err[i] <= b) return k;
        }
        return -1;
    };
    double best_gap = INFINITY, best_b = 0.0, best_S = 0.0;
    for (double b : budgets) {   // Eqs. 8-10; increasing b, so a tie keeps the smaller budget
        double S = 0.0;
        for (int l = 0; l < L; ++l) {
            if (l == guard) {
                S += guard_sp;
                continue;
            }
            const int k = pick(l, b);
            S += k < 0 ? 0.0 : sp[(size_t)l * K + k];
        }
        S /= L;
        const double gap = std::fabs(S - s_tar);
        if (gap < best_gap) {
            best_gap = gap;
            best_b = b;
            best_S = S;
        }
    }
    for (int l = 0; l < L; ++l) {
        if (l == guard) {
            t_out[l] = guard_t;
            continue;
        }
        const int k = pick(l, best_b);
        t_out[l] = k < 0 ? 0.0 : t[(size_t)l * K + k];
    }
    *b_out = best_b;
    *S_out = best_S;
    return SATS_OK;
}

size_t sats_sats_workspace_bytes(int H, int N, int C, int L, int K0, int K1)
{
    if (H < 8 || H > kMaxH || (H % 8) != 0 || N < 1 || N > kMaxN || C < 1 || L < 1 || K0 < 2 || K1 < 0) return 0;
    const int K = std::max(K0, K1);   // (the coarse candidates and the guardrail threshold)
    return sats_layout(H, N, C, L, K0, K).total;
}

sats_status sats_sats_calibrate(const sats_layer *const *layers, const float *const *norm_w, int L, float eps,
                                const float *x_cal, int C, double s_tar, int K0, int K1, int guardrail, float err_eps,
                                float *t_out, double *b_out, double *S_out, double *table_t, double *table_err,
                                double *table_sp, void *ws, size_t ws_bytes, void *stream)
{
    if (!layers || !norm_w || L < 1 || !x_cal || C < 1 || K0 < 2 || K1 < 0 || !t_out || !ws) return SATS_EINVAL;
    if (std::isnan(eps) || eps < 0.0f || std::isnan(err_eps) || err_eps < 0.0f || !(s_tar >= 0.0 && s_tar <= 1.0))
        return SATS_EINVAL;
    if ((reinterpret_cast<uintptr_t>(x_cal) & 15u) || (reinterpret_cast<uintptr_t>(ws) & 255u)) return SATS_EINVAL;
    const int H = layers[0] ? layers[0]->H : 0, N = layers[0] ? layers[0]->N : 0;
    for (int l = 0; l < L; ++l)
        if (!layers[l] || layers[l]->H != H || layers[l]->N != N || !norm_w[l]) return SATS_EINVAL;
    const int Kc = K0 - 1, Kmax = std::max(Kc + 1, K1), Kt = Kc + K1;
    const SatsLayout W = sats_layout(H, N, C, L, K0, Kmax);
    if (ws_bytes < W.total) return SATS_ENOSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char *base = static_cast<char *>(ws);
    float *x = reinterpret_cast<float *>(base + W.x);
    float *nall = reinterpret_cast<float *>(base + W.n);
    void *sel = base + W.sel;
    float *q = reinterpret_cast<float *>(base + W.q);
    char *ews = base + W.err;
    const ErrLayout E = err_layout(H, N, C, Kmax, false);
    const ErrGroup group = err_group(H, N, C, Kmax);
    char *sums = base + W.sums;
    const size_t sum_bytes = ErrSums::bytes(Kmax);
    const bool batched = use_tc_path(H, C);
    // (the masks take the gate activations that the thresholds are percentiles of)
    auto inputs_of = [&](int l) {
        char *a = base + W.a + l * W.in_each;
        return ErrInputs(a, W.in_each ? a + ErrInputs::a_bytes(N, C) : ews + E.h, N, C);
    };
    char *mlp = ews + E.mlp;
    // every bounded wait of the call reports here
    int *ctl = reinterpret_cast<int *>(mlp + ws_layout(H, N, C).ctl), *status = ctl + kCtlStatus;
    auto n_of = [&](int l) { return nall + (size_t)l * C * H; };
    auto up_of = [&](int l) {
        const ErrInputs in = inputs_of(l);
        return launch_up_f32(layers[l], n_of(l), C, in.a, in.hhi, in.hlo, status, st);
    };
    auto gate_of = [&](int l) { return batched ? inputs_of(l).a : reinterpret_cast<float *>(base + W.a); };
    const size_t ews_bytes = W.total - W.err;
    const int guard = guardrail ? L - 1 : -1;

    // 1-2: the dense stack gives each block's MLP inputs; coarse candidates from |SiLU(n W_gate)|
    cudaError_t e = cudaMemcpyAsync(x, x_cal, (size_t)C * H * sizeof(float), cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess) e = clear_fused_state(mlp, H, N, C, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(q, 0, W.a - W.q, st);   // (the sums follow the percentiles)
    if (e != cudaSuccess) return cuda_fail(e, "calibration set-up");
    std::vector<double> tc((size_t)L * Kc), amax((size_t)L), errc((size_t)L * Kc), spc((size_t)L * Kc);
    double g_t = 0.0, g_sp = 0.0;
    const float zero = 0.0f;
    sats_status s;
    const int64_t n = (int64_t)C * N;
    std::vector<int64_t> rank((size_t)K0 + 1);
    for (int l = 0; l < L; ++l) {
        if ((s = sats_rmsnorm(x, C, H, norm_w[l], eps, n_of(l), stream)) != SATS_OK) return s;
        float *a = gate_of(l);
        if ((e = launch_gate_act_f32(layers[l], n_of(l), C, a, status, st)) != cudaSuccess)
            return cuda_fail(e, "gate activation kernel launch");
        // Eq. 3 at k / K0, the largest |a|, and the guardrail block's percentile at the target, all
        // from shared passes over |a|; read back once after the last block
        float *ql = q + (size_t)l * (K0 + 1);
        const int nq = l == guard && s_tar > 0.0 ? Kc + 2 : Kc + 1;
        for (int k = 0; k < nq; ++k)
            rank[(size_t)k] = percentile_rank(n, k < Kc ? (double)(k + 1) / K0 : k == Kc ? 1.0 : s_tar);
        for (int k = 0; k < nq; k += kSelRanks)
            if ((e = launch_select(a, n, rank.data() + k, std::min(kSelRanks, nq - k), sel, ql + k, status, st)) !=
                cudaSuccess)
                return cuda_fail(e, "percentile kernels launch");
        if (batched) {
            // 3: Eq. 6 for every coarse candidate (and, with them, the guardrail's CATS threshold), the
            // thresholds read on the device; then x <- x + MLP_l(n_l)
            const int K = l == guard ? Kc + 1 : Kc;
            if ((e = up_of(l)) != cudaSuccess) return cuda_fail(e, "up kernel launch");
            if ((s = enqueue_err(layers[l], inputs_of(l), C, nullptr, ql, [&](int k) { return k < Kc ? k : Kc + 1; }, K,
                                 err_eps, ErrSums(sums + l * sum_bytes, K), group, ews, E, ctl, st)) != SATS_OK)
                return s;
            if ((s = enqueue_residual(layers[l], x, C, inputs_of(l), group.rows(), ews, E, ctl, st)) != SATS_OK)
                return s;
            continue;
        }
        // x <- x + MLP_l(n_l) with every neuron kept
        if ((s = run_layer(layers[l], kXF32, n_of(l), C, &zero, nullptr, 0.f, nullptr, kOutResid, x, nullptr,
                           nullptr, nullptr, mlp, st)) != SATS_OK)
            return s;
    }
    std::vector<float> qh((size_t)L * (K0 + 1), 0.f);
    std::vector<char> hs((size_t)L * sum_bytes);
    e = cudaMemcpyAsync(qh.data(), q, qh.size() * sizeof(float), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess && batched) e = cudaMemcpyAsync(hs.data(), sums, hs.size(), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "percentile read-back");
    for (int l = 0; l < L; ++l) {
        const float *ql = qh.data() + (size_t)l * (K0 + 1);
        std::copy(ql, ql + Kc, tc.begin() + (size_t)l * Kc);
        amax[(size_t)l] = ql[Kc];
        if (l == guard) g_t = s_tar > 0.0 ? ql[Kc + 1] : 0.f;
    }
    if ((s = sats_get_error(mlp, ws_layout(H, N, C).total, stream)) != SATS_OK) return s;
    // 3 (without a batch): Eq. 6 block by block
    std::vector<float> tf((size_t)Kmax);
    std::vector<double> eb((size_t)Kmax), sb((size_t)Kmax);
    for (int l = 0; l < L; ++l) {
        const int K = l == guard ? Kc + 1 : Kc;
        if (batched) {
            err_means(hs.data() + l * sum_bytes, K, C, N, eb.data(), sb.data());
        } else {
            for (int k = 0; k < Kc; ++k) tf[(size_t)k] = (float)tc[(size_t)l * Kc + k];
            if (l == guard) tf[(size_t)Kc] = (float)g_t;
            if ((s = sats_layer_err(layers[l], n_of(l), C, tf.data(), K, err_eps, eb.data(), sb.data(), ews, ews_bytes,
                                    stream)) != SATS_OK)
                return s;
        }
        for (int k = 0; k < Kc; ++k) {
            errc[(size_t)l * Kc + k] = eb[(size_t)k];
            spc[(size_t)l * Kc + k] = sb[(size_t)k];
        }
        if (l == guard) g_sp = sb[(size_t)Kc];
    }
    // 4: Eqs. 7-10 over the coarse candidates
    double b0 = 0.0, S0 = 0.0;
    std::vector<double> t0((size_t)L);
    if ((s = sats_sats_select(tc.data(), errc.data(), spc.data(), L, Kc, s_tar, guard, g_t, g_sp, &b0, t0.data(),
                              &S0)) != SATS_OK)
        return s;
    // 5-6: K1 candidates strictly between the coarse neighbours of each block's choice, then
    // Eqs. 6-10 over coarse and fine candidates together
    std::vector<double> ta((size_t)L * Kt), ea((size_t)L * Kt), sa((size_t)L * Kt);
    tf.assign((size_t)L * std::max(K1, 1), 0.f);
    if (batched && K1 > 0 && (e = cudaMemsetAsync(sums, 0, (size_t)L * sum_bytes, st)) != cudaSuccess)
        return cuda_fail(e, "layer error workspace clear");
    for (int l = 0; l < L; ++l) {
        double lo = 0.0, hi = amax[(size_t)l];
        bool above = false;
        for (int k = 0; k < Kc; ++k) {
            const double v = tc[(size_t)l * Kc + k];
            if (v < t0[(size_t)l]) lo = std::max(lo, v);
            if (v > t0[(size_t)l]) {
                hi = above ? std::min(hi, v) : v;
                above = true;
            }
        }
        for (int k = 0; k < Kc; ++k) {
            ta[(size_t)l * Kt + k] = tc[(size_t)l * Kc + k];
            ea[(size_t)l * Kt + k] = errc[(size_t)l * Kc + k];
            sa[(size_t)l * Kt + k] = spc[(size_t)l * Kc + k];
        }
        for (int k = 0; k < K1; ++k) {
            const float t = (float)(lo + (hi - lo) * (k + 1) / (K1 + 1));
            tf[(size_t)l * K1 + k] = t;
            ta[(size_t)l * Kt + Kc + k] = t;
        }
        if (K1 == 0) continue;
        if (batched && W.in_each == 0) {
            if ((e = launch_gate_act_f32(layers[l], n_of(l), C, gate_of(l), status, st)) != cudaSuccess)
                return cuda_fail(e, "gate activation kernel launch");
            if ((e = up_of(l)) != cudaSuccess) return cuda_fail(e, "up kernel launch");
        }
        s = batched ? enqueue_err(layers[l], inputs_of(l), C, tf.data() + (size_t)l * K1, nullptr, [](int k) { return k; },
                                  K1, err_eps, ErrSums(sums + l * sum_bytes, K1), group, ews, E, ctl, st)
                    : sats_layer_err(layers[l], n_of(l), C, tf.data() + (size_t)l * K1, K1, err_eps,
                                     ea.data() + (size_t)l * Kt + Kc, sa.data() + (size_t)l * Kt + Kc, ews, ews_bytes,
                                     stream);
        if (s != SATS_OK) return s;
    }
    if (batched && K1 > 0) {
        e = cudaMemcpyAsync(hs.data(), sums, hs.size(), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return cuda_fail(e, "layer error read-back");
        if ((s = sats_get_error(mlp, ws_layout(H, N, C).total, stream)) != SATS_OK) return s;
        for (int l = 0; l < L; ++l)
            err_means(hs.data() + l * sum_bytes, K1, C, N, ea.data() + (size_t)l * Kt + Kc, sa.data() + (size_t)l * Kt + Kc);
    }
    double b = 0.0, S = 0.0;
    std::vector<double> tt((size_t)L);
    if ((s = sats_sats_select(ta.data(), ea.data(), sa.data(), L, Kt, s_tar, guard, g_t, g_sp, &b, tt.data(), &S)) !=
        SATS_OK)
        return s;
    for (int l = 0; l < L; ++l) t_out[l] = (float)tt[(size_t)l];
    if (b_out) *b_out = b;
    if (S_out) *S_out = S;
    if (table_t && table_err && table_sp) {
        std::copy(ta.begin(), ta.end(), table_t);
        std::copy(ea.begin(), ea.end(), table_err);
        std::copy(sa.begin(), sa.end(), table_sp);
    }
    return SATS_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------- routing calibration (Sec. 3.2)
namespace sats {
namespace {

// Where token v's total and count are kept: neighbouring ids go to different cache lines.  Ids are often
// given out by frequency, and additions to one line queue up behind one another (a million occurrences,
// Zipf ids in order of rank: 57 us, most of it on the first few lines).
constexpr int kSpread = 64;

__host__ __device__ inline int spread_rows(int V) { return V / kSpread + (V % kSpread != 0); }

__device__ __forceinline__ size_t spread(int v, int rows)
{
    return (size_t)(v & (kSpread - 1)) * rows + v / kSpread;   // (up to V + 62, beyond int for the largest V)
}

int blocks_of(int V, int per) { return (int)(((int64_t)V + per - 1) / per); }

// A warp's table of the token ids it has met: sums of the occurrences it has seen, added to the
// device totals once at the end.  Token frequencies are far from even (a corpus' most common token
// is several per cent of it), and atomics on one address go one after the other: 290 us for a
// million occurrences added straight to global memory.  Tables of one warp need no atomics:
// lanes with the same id take turns.  An id whose slot another id holds is added to the totals
// directly.
constexpr int kTallySlots = 512, kTallyWarps = 16;
constexpr int kNoToken = -1;

template <bool SUMS>
struct Tally {
    int id[kTallySlots];
    unsigned count[kTallySlots];
    double sum[SUMS ? kTallySlots : 1];
};

// Adds one occurrence per lane (id kNoToken: none) with excess loss v.
template <bool SUMS>
__device__ __forceinline__ void tally_add(Tally<SUMS> &T, int id, float v, double *__restrict__ total,
                                          unsigned *__restrict__ count, int rows)
{
    const unsigned lane = threadIdx.x & 31u;
    const unsigned same = __match_any_sync(0xffffffffu, id);
    const int slot = (int)(((unsigned)id * 2654435761u) >> (32 - 9));
    static_assert(kTallySlots == 1 << 9, "slot hash width");
    const unsigned turn = __popc(same & ((1u << lane) - 1u));   // of the lanes with this id
    bool mine = false;
    if (id != kNoToken && turn == 0 && T.id[slot] == kNoToken) T.id[slot] = id;   // one id wins an empty slot
    __syncwarp();
    if (id != kNoToken) mine = T.id[slot] == id;
    if (id != kNoToken && !mine) {
        if (SUMS) atomicAdd(total + spread(id, rows), (double)v);
        atomicAdd(count + spread(id, rows), 1u);
    }
    if (mine && turn == 0) T.count[slot] += (unsigned)__popc(same);
    if (!SUMS) {
        __syncwarp();
        return;
    }
    const unsigned turns = __reduce_max_sync(0xffffffffu, mine ? turn + 1u : 0u);
    for (unsigned k = 0; k < turns; ++k) {
        if (mine && turn == k) T.sum[slot] += (double)v;
        __syncwarp();
    }
}

// Eqs. 11-12, the sums (SUMS): for every occurrence, d = max(0, l_sparse - l_base) into the token's
// total, and the occurrences per token; without SUMS the occurrences only.
template <bool SUMS>
__global__ void __launch_bounds__(32 * kTallyWarps) tally_kernel(const int32_t *__restrict__ ids,
                                                                 const float *__restrict__ lb,
                                                                 const float *__restrict__ ls, int64_t n, int V,
                                                                 double *__restrict__ total,
                                                                 unsigned *__restrict__ count,
                                                                 int32_t *__restrict__ status)
{
    extern __shared__ __align__(16) char tally_smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    Tally<SUMS> &T = reinterpret_cast<Tally<SUMS> *>(tally_smem)[warp];
    for (int i = lane; i < kTallySlots; i += 32) {
        T.id[i] = kNoToken;
        T.count[i] = 0u;
        if (SUMS) T.sum[i] = 0.0;
    }
    __syncwarp();
    const int rows = spread_rows(V);
    constexpr int kAhead = 4;   // loads in flight per lane
    const int64_t step = (int64_t)gridDim.x * kTallyWarps * 32;
    for (int64_t base = ((int64_t)blockIdx.x * kTallyWarps + warp) * 32; base < n; base += kAhead * step) {
        int id[kAhead];
        float v[kAhead];
#pragma unroll
        for (int k = 0; k < kAhead; ++k) {
            const int64_t i = base + k * step + lane;
            id[k] = kNoToken;
            v[k] = 0.f;
            if (i < n) {
                id[k] = ids[i];
                if (SUMS) v[k] = fmaxf(0.0f, ls[i] - lb[i]);
                if (id[k] < 0 || id[k] >= V) {
                    atomicOr(status, kStatusBadToken);
                    id[k] = kNoToken;
                }
            }
        }
#pragma unroll
        for (int k = 0; k < kAhead; ++k) tally_add<SUMS>(T, id[k], v[k], total, count, rows);
    }
    __syncthreads();
    // the CTA's tables together, a thread per slot: common tokens have the slot in every table
    const Tally<SUMS> *all = reinterpret_cast<const Tally<SUMS> *>(tally_smem);
    for (int i = threadIdx.x; i < kTallySlots; i += 32 * kTallyWarps) {
        int first = kNoToken;
        unsigned c = 0u;
        double v = 0.0;
        for (int w = 0; w < kTallyWarps; ++w) {
            const int id = all[w].id[i];
            if (id == kNoToken) continue;
            if (first == kNoToken) first = id;
            if (id == first) {
                c += all[w].count[i];
                if (SUMS) v += all[w].sum[i];
            } else {
                if (SUMS) atomicAdd(total + spread(id, rows), all[w].sum[i]);
                atomicAdd(count + spread(id, rows), all[w].count[i]);
            }
        }
        if (first != kNoToken) {
            if (SUMS) atomicAdd(total + spread(first, rows), v);
            atomicAdd(count + spread(first, rows), c);
        }
    }
}

// Eq. 12, the means; +inf for a token that never occurs (it keeps the base path).
__global__ void score_final_kernel(const double *__restrict__ total, const unsigned *__restrict__ count, int V,
                                   float *__restrict__ score)
{
    grid_dependency_wait();
    grid_launch_dependents();
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= V) return;
    const size_t at = spread(v, spread_rows(V));
    const unsigned c = count[at];
    if (c == 0u) {
        score[v] = INFINITY;
        return;
    }
    // total / c rounded to fp32, with one 64-bit multiply-add instead of a 64-bit division (this GPU has
    // few 64-bit units): a quotient q in fp32 and its remainder's share
    const double t = total[at];
    const float cf = (float)c, q = (float)t / cf;
    if (q > 1e-30f && q < 1e38f) score[v] = q + (float)__fma_rn(-(double)q, (double)c, t) / cf;
    else score[v] = (float)(t / (double)c);   // 0, and the ends of fp32's range
}

// Eq. 14 on the device.  With the held-out occurrences' scores in increasing order, the candidates
// around the target are the occurrence at rank K + 1 (K: the most occurrences that may lie below tau
// for R(tau) <= r_tar) and the next larger score.  A radix search over the V scores, weighted by the
// occurrences (11 + 11 + 10 bits of the ordered bit pattern; each level one kernel whose last CTA
// picks the bin), finds the first; one more pass sums the occurrences below it and at it, and takes
// the smallest score above it.  Sorting the scores on the host took 2 ms of the call.
struct TauSearch {
    unsigned done[3];
    uint32_t prefix;                 // bits of the rank's score chosen so far
    unsigned long long rest;         // rank within the chosen bins (1-based)
    unsigned long long below, at;    // occurrences with a smaller score, with the same score
    unsigned long long negative;     // occurrences with a score below 0
    unsigned long long finite;       // occurrences with a score below +inf
    uint32_t not_above;              // complement of the ordered bits of the smallest larger score (0: none)
    uint32_t pad;
    unsigned long long hist[3][2048];
};

// Floats in increasing order as unsigned numbers (-0 as +0).
__device__ __forceinline__ uint32_t ordered_bits(float f)
{
    const uint32_t b = __float_as_uint(f + 0.0f);
    return (b & 0x80000000u) ? ~b : b | 0x80000000u;
}

constexpr int kTauThreads = 512;

template <int LEVEL>
__global__ void __launch_bounds__(kTauThreads) tau_level_kernel(const float *__restrict__ score,
                                                                const unsigned *__restrict__ freq, int V,
                                                                unsigned long long rank, TauSearch *S)
{
    constexpr int kShift = LEVEL == 0 ? 21 : LEVEL == 1 ? 10 : 0;
    constexpr int kBins = LEVEL == 2 ? 1024 : 2048;
    __shared__ unsigned long long h[kBins];
    __shared__ unsigned long long warp_sum_s[kTauThreads / 32];
    __shared__ bool last;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int i = tid; i < kBins; i += kTauThreads) h[i] = 0ull;
    grid_dependency_wait();
    grid_launch_dependents();
    const uint32_t prefix = LEVEL == 0 ? 0u : S->prefix;
    const int rows = spread_rows(V);
    __syncthreads();
    for (unsigned v = blockIdx.x * kTauThreads + tid; v < (unsigned)V; v += gridDim.x * kTauThreads) {   // (int would overflow)
        const unsigned f = freq[spread((int)v, rows)];
        const uint32_t b = ordered_bits(score[v]);
        const bool in = LEVEL == 0 || (LEVEL == 1 ? (b >> 21) == (prefix >> 21) : (b >> 10) == (prefix >> 10));
        if (f && in) atomicAdd(h + ((b >> kShift) & (kBins - 1)), (unsigned long long)f);
    }
    __syncthreads();
    for (int i = tid; i < kBins; i += kTauThreads)
        if (h[i]) atomicAdd(&S->hist[LEVEL][i], h[i]);
    __threadfence();
    __syncthreads();
    if (tid == 0) last = atomicAdd(&S->done[LEVEL], 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    constexpr int kPer = kBins / kTauThreads;
    unsigned long long c[kPer], s = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
        c[k] = __ldcg(&S->hist[LEVEL][tid * kPer + k]);
        s += c[k];
    }
    unsigned long long incl = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_sum_s[warp] = incl;
    const unsigned long long r = LEVEL == 0 ? rank : S->rest;
    __syncthreads();
    for (int w = 0; w < warp; ++w) incl += warp_sum_s[w];
    unsigned long long run = incl - s;
    if (run < r && incl >= r) {   // one thread's bins hold the rank (1 <= rank <= the occurrences)
        for (int k = 0; k < kPer; ++k) {
            if (run + c[k] >= r) {
                S->prefix = prefix | ((uint32_t)(tid * kPer + k) << kShift);
                S->rest = r - run;
                break;
            }
            run += c[k];
        }
    }
}

// The occurrences around the score at the rank (S->prefix), and those below 0 and below +inf.
__global__ void __launch_bounds__(kTauThreads) tau_sums_kernel(const float *__restrict__ score,
                                                               const unsigned *__restrict__ freq, int V, TauSearch *S)
{
    __shared__ unsigned long long sums[4];
    __shared__ uint32_t not_above;
    if (threadIdx.x < 4) sums[threadIdx.x] = 0ull;
    if (threadIdx.x == 4) not_above = 0u;
    grid_dependency_wait();
    __syncthreads();
    const int rows = spread_rows(V);
    const uint32_t at = S->prefix, zero = 0x80000000u, inf = 0xff800000u;
    unsigned long long s[4] = {0ull, 0ull, 0ull, 0ull};
    uint32_t na = 0u;
    for (unsigned v = blockIdx.x * kTauThreads + threadIdx.x; v < (unsigned)V; v += gridDim.x * kTauThreads) {
        const unsigned f = freq[spread((int)v, rows)];
        if (!f) continue;
        const uint32_t b = ordered_bits(score[v]);
        s[0] += b < at ? f : 0u;
        s[1] += b == at ? f : 0u;
        s[2] += b < zero ? f : 0u;
        s[3] += b < inf ? f : 0u;
        if (b > at) na = max(na, ~b);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], o);
        if ((threadIdx.x & 31) == 0 && s[k]) atomicAdd(sums + k, s[k]);
    }
    na = __reduce_max_sync(0xffffffffu, na);
    if ((threadIdx.x & 31) == 0 && na) atomicMax(&not_above, na);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (sums[0]) atomicAdd(&S->below, sums[0]);
        if (sums[1]) atomicAdd(&S->at, sums[1]);
        if (sums[2]) atomicAdd(&S->negative, sums[2]);
        if (sums[3]) atomicAdd(&S->finite, sums[3]);
        if (not_above) atomicMax(&S->not_above, not_above);
    }
}

// Eq. 13 as a table: 1 (base path) where score >= tau, 0 (sparse path) where score < tau.
__global__ void lut_kernel(const float *__restrict__ score, int V, float tau, uint8_t *__restrict__ lut)
{
    const int v = blockIdx.x * blockDim.x + threadIdx.x;
    if (v < V) lut[v] = score[v] < tau ? 0 : 1;
}

struct ScoreLayout {
    size_t status, search, total, count, total_bytes;
};

ScoreLayout score_layout(int V)
{
    ScoreLayout S{};
    size_t off = 0;
    S.status = off;
    off += 256;
    S.search = off;   // sats_route_calibrate
    off += al256(sizeof(TauSearch));
    S.total = off;
    off += al256((size_t)kSpread * spread_rows(V) * sizeof(double));
    S.count = off;
    off += al256((size_t)kSpread * spread_rows(V) * sizeof(unsigned));
    S.total_bytes = off;
    return S;
}

sats_status read_status_word(int32_t *word, cudaStream_t st)
{
    int32_t v = 0;
    cudaError_t e = cudaMemcpyAsync(&v, word, sizeof v, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "status read");
    return (v & kStatusBadToken) ? SATS_EDEVICE : SATS_OK;
}

template <bool SUMS>
cudaError_t launch_tally(const int32_t *ids, const float *lb, const float *ls, int64_t n, int V, double *total,
                         unsigned *count, int32_t *status, cudaStream_t st)
{
    const size_t smem = sizeof(Tally<SUMS>) * kTallyWarps;
    const cudaError_t e = cudaFuncSetAttribute(tally_kernel<SUMS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const int64_t want = (n + 32 * kTallyWarps - 1) / (32 * kTallyWarps);
    const int sms = fused_grid(kMaxGrid);
    tally_kernel<SUMS><<<(int)(want < sms ? want : sms), 32 * kTallyWarps, smem, st>>>(ids, lb, ls, n, V, total, count,
                                                                                     status);
    return cudaGetLastError();
}

template <typename... KArgs, typename... Args>
cudaError_t launch_search(void (*kernel)(KArgs...), int V, cudaStream_t st, Args... args)
{
    const int want = blocks_of(V, 2 * kTauThreads), sms = fused_grid(kMaxGrid);
    return launch_after(kernel, dim3(want < sms ? want : sms), kTauThreads, st, args...);
}

float score_of(uint32_t ordered)
{
    const uint32_t b = (ordered & 0x80000000u) ? ordered & 0x7fffffffu : ~ordered;
    float f;
    std::memcpy(&f, &b, sizeof f);
    return f;
}

}  // namespace
}  // namespace sats

extern "C" {

size_t sats_route_calib_workspace_bytes(int V)
{
    if (V < 1) return 0;
    return score_layout(V).total_bytes;
}

sats_status sats_token_scores(const int32_t *ids, const float *l_base, const float *l_sparse, int64_t n, int V,
                              float *score, void *ws, size_t ws_bytes, void *stream)
{
    if (V < 1 || n < 0 || !score || !ws || (n > 0 && (!ids || !l_base || !l_sparse))) return SATS_EINVAL;
    const ScoreLayout S = score_layout(V);
    if (ws_bytes < S.total_bytes || (reinterpret_cast<uintptr_t>(ws) & 255u)) return ws_bytes < S.total_bytes ? SATS_ENOSPACE : SATS_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char *base = static_cast<char *>(ws);
    int32_t *status = reinterpret_cast<int32_t *>(base + S.status);
    double *total = reinterpret_cast<double *>(base + S.total);
    unsigned *count = reinterpret_cast<unsigned *>(base + S.count);
    cudaError_t e = cudaMemsetAsync(ws, 0, S.total_bytes, st);
    if (e != cudaSuccess) return cuda_fail(e, "score workspace clear");
    if (n > 0 && (e = launch_tally<true>(ids, l_base, l_sparse, n, V, total, count, status, st)) != cudaSuccess)
        return cuda_fail(e, "score kernel launch");
    e = launch_after(score_final_kernel, dim3(blocks_of(V, 256)), 256, st, (const double *)total, (const unsigned *)count, V,
                     score);
    if (e != cudaSuccess) return cuda_fail(e, "score kernel launch");
    return read_status_word(status, st);
}

sats_status sats_route_calibrate(const float *score, int V, const int32_t *heldout_ids, int64_t m, double r_tar,
                                 float *tau_out, double *R_out, uint8_t *lut, void *ws, size_t ws_bytes, void *stream)
{
    if (V < 1 || m < 0 || !score || !tau_out || !ws || std::isnan(r_tar) || (m > 0 && !heldout_ids)) return SATS_EINVAL;
    const ScoreLayout S = score_layout(V);
    if (ws_bytes < S.total_bytes || (reinterpret_cast<uintptr_t>(ws) & 255u)) return ws_bytes < S.total_bytes ? SATS_ENOSPACE : SATS_EINVAL;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char *base = static_cast<char *>(ws);
    int32_t *status = reinterpret_cast<int32_t *>(base + S.status);
    unsigned *freq = reinterpret_cast<unsigned *>(base + S.count);
    TauSearch *search = reinterpret_cast<TauSearch *>(base + S.search);
    cudaError_t e = cudaMemsetAsync(status, 0, 256 + sizeof(TauSearch), st);   // (the search follows the status word)
    if (e == cudaSuccess) e = cudaMemsetAsync(freq, 0, (size_t)kSpread * spread_rows(V) * sizeof(unsigned), st);
    if (e != cudaSuccess) return cuda_fail(e, "held-out count clear");
    if (m > 0 && (e = launch_tally<false>(heldout_ids, nullptr, nullptr, m, V, nullptr, freq, status, st)) != cudaSuccess)
        return cuda_fail(e, "held-out count kernel launch");
    // K: the most occurrences c <= m with c / m <= r_tar (-1: none); R(tau) = (occurrences below tau) / m
    const double M = m > 0 ? (double)m : 1.0;
    int64_t K = m;
    if (!(r_tar >= 1.0)) {
        K = r_tar < 0.0 ? -1 : (int64_t)(r_tar * M);
        while (K >= 0 && (double)K / M > r_tar) --K;
        while (K < m && (double)(K + 1) / M <= r_tar) ++K;
    }
    struct {
        int32_t status;
        char pad[252];
        unsigned done[3];
        uint32_t prefix;
        unsigned long long rest, below, at, negative, finite;
        uint32_t not_above, pad2;
    } got;
    static_assert(offsetof(TauSearch, hist) == sizeof(got) - 256, "layout of the search's results");
    const unsigned long long rank = (unsigned long long)(K < 0 ? 1 : K >= m ? m : K + 1);   // 1-based
    if (m > 0) {
        e = launch_search(tau_level_kernel<0>, V, st, score, (const unsigned *)freq, V, rank, search);
        if (e == cudaSuccess) e = launch_search(tau_level_kernel<1>, V, st, score, (const unsigned *)freq, V, rank, search);
        if (e == cudaSuccess) e = launch_search(tau_level_kernel<2>, V, st, score, (const unsigned *)freq, V, rank, search);
        if (e == cudaSuccess) e = launch_search(tau_sums_kernel, V, st, score, (const unsigned *)freq, V, search);
        if (e != cudaSuccess) return cuda_fail(e, "threshold search kernels launch");
    }
    e = cudaMemcpyAsync(&got, status, sizeof got, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "threshold search read-back");
    if (got.status & kStatusBadToken) return SATS_EDEVICE;
    // The candidates are 0, each distinct finite positive held-out score, and +inf; R never falls from
    // one to the next, so the nearest to the target is one of the two around it (a tie: the smaller).
    double best_gap = INFINITY, best_R = 0.0;
    float best_tau = 0.0f;
    auto consider = [&](float tau, uint64_t below) {   // in increasing order of tau
        const double R = (double)below / M;
        const double gap = std::fabs(R - r_tar);
        if (gap < best_gap) {
            best_gap = gap;
            best_tau = tau;
            best_R = R;
        }
    };
    consider(0.0f, got.negative);
    if (m > 0) {
        const float at = score_of(got.prefix);
        if (at > 0.0f && std::isfinite(at)) consider(at, got.below);
        const float above = got.not_above ? score_of(~got.not_above) : INFINITY;
        if (std::isfinite(above) && above > 0.0f) consider(above, got.below + got.at);
    }
    consider(INFINITY, m > 0 ? got.finite : 0);
    *tau_out = best_tau;
    if (R_out) *R_out = best_R;
    if (lut) {
        lut_kernel<<<blocks_of(V, 256), 256, 0, st>>>(score, V, best_tau, lut);
        if ((e = cudaGetLastError()) != cudaSuccess) return cuda_fail(e, "table kernel launch");
    }
    return SATS_OK;
}

}  // extern "C"
