// Learned move proposal (growth path, not in the paper): a small network
// 12 -> 64 -> 64 -> 1 (ReLU) predicts each variable's best-shift score from
// per-variable features; the exact best-shift evaluation then runs on the
// top-k predicted variables only, and a full exact pass every E iterations is
// both the fallback move and the judge of the proposal's top-1 misses.  The
// scores that decide moves are always exact.
//
// Kernels: features, refresh of the pass-time features, network forward
// (BF16 parameters and features, FP32 accumulation with explicit FMAs), loss
// gradient over a minibatch (tiles of 64 rows, activations in shared memory),
// Adam, the proposal's scores (features, forward pass and first histogram),
// deterministic top-k by three-level radix select + stable compaction in one
// cluster, exact flip scores of the selected binary columns, and the glue that
// hands the chosen move to the apply kernel of the exact path.
#include "chap_handle.h"

#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <mutex>
#include <string>

namespace chap {
namespace {

namespace cg = cooperative_groups;

#define FULLMASK 0xffffffffu

constexpr int kF = 12, kH = 64;
constexpr int kOffW1 = 0, kOffB1 = kF * kH, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH;
constexpr int kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kH, kNParams = kOffB3 + 1;  // 5057
constexpr int kTileRows = 64;        // rows of one network tile
constexpr int kTileThreads = 256;    // threads of its CTA: 4 rows x 4 columns of a layer each
constexpr int kTPad = kTileRows + 4; // rows of a transposed activation, padded (16-byte aligned, 17 x 16 bytes)
constexpr int kPropThreads = 128;    // proposal scores: 4 warps of 32 variables
constexpr int kTkThreads = 1024;     // top-k: threads of a CTA of the cluster
constexpr int kTkCtas = 16;          // its largest cluster
constexpr int kTkKeys = 1024;        // keys of a warp kept in shared memory
constexpr int kTkSmem = (kTkThreads / 32) * kTkKeys * (int)sizeof(unsigned);
constexpr int kVarBits = 22;

// Device state of the learned driver of one handle.
struct __align__(16) LearnCtl {
    unsigned long long key;     // best proposal move: score << 22 | (2^22 - 1 - var), 0 = none
    long long smax;             // max |score| at the last exact pass
    long long passes, misses;   // exact passes and top-1 misses
    long long pass_iter;        // iteration of the last exact pass
    unsigned ticket;            // CTAs of the subset kernel that are done
};

struct Learn {
    double *xh;                   // value of the best shift of each proposed non-binary column [n]
    float *colviol, *colwv;       // pass-time column features [n]
    long long *s_last;            // exact scores of the last pass [n]
    __nv_bfloat16 *feat;          // [n x 12]
    float *y;                     // predictions [n]
    uint2 *fixed;                 // features 8..11 of each variable [n]: they never change
    unsigned *hist;               // 3 x 2048 bins, zero between selections
    int *bcnt;                    // per-CTA counts of the selection [2 x kTkCtas]
    int *list;                    // selected variables [k]
    LearnCtl *lc;
};

__device__ __forceinline__ unsigned long long lglobal_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool done_gate(const Dev &d) { return *(volatile int *)&d.ctl->done != 0; }

__device__ __forceinline__ long long i4_r(const int4 &v)
{
    return (long long)(((unsigned long long)(unsigned)v.y << 32) | (unsigned)v.x);
}

__device__ __forceinline__ bool dbl_neg_bits(long long b) { return b < 0; }

// ---------------------------------------------------------------- features

// Column features recorded at an exact pass: share of violated halves and the
// weighted (w |a|) share, one thread per variable, and the largest |score|
// (one atomic per CTA: one per variable on the same word was most of the
// kernel, 132 us for 200k variables 13 without it).
__global__ void k_refresh(Dev d, Learn L)
{
    unsigned long long top = 0;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < d.n; j += gridDim.x * blockDim.x) {
        const int q = d.vpos[j];
        int halves = 0, viol = 0;
        float wall = 0.0f, wviol = 0.0f;
        for (int e = d.ci_ptr[q]; e < d.ci_ptr[q + 1]; ++e) {
            const RowState s = d.rs[d.ci_row[e]];
            const float a = fabsf((float)d.ci_val[e]);
            halves += 1; wall += s.w1 * a;
            if (s.r > 0) { viol += 1; wviol += s.w1 * a; }
            if (s.w2 >= 0) {
                halves += 1; wall += s.w2 * a;
                if (s.r < 0) { viol += 1; wviol += s.w2 * a; }
            }
        }
        for (int e = d.cf_ptr[q]; e < d.cf_ptr[q + 1]; ++e) {
            const RowState s = d.rs[d.cf_row[e]];
            const float a = fabsf((float)d.cf_val[e]);
            halves += 1; wall += s.w1 * a;
            if (dbl_neg_bits(__double_as_longlong(s.m1))) { viol += 1; wviol += s.w1 * a; }
            if (s.w2 >= 0) {
                halves += 1; wall += s.w2 * a;
                if (dbl_neg_bits(__double_as_longlong(s.m2))) { viol += 1; wviol += s.w2 * a; }
            }
        }
        L.colviol[j] = halves ? (float)viol / (float)halves : 0.0f;
        L.colwv[j] = wall > 0.0f ? wviol / wall : 0.0f;
        const long long sa = L.s_last[j] < 0 ? -L.s_last[j] : L.s_last[j];
        top = max(top, (unsigned long long)sa);
    }
    __shared__ unsigned long long s_top[8];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(FULLMASK, top, o));
    if ((threadIdx.x & 31) == 0) s_top[threadIdx.x >> 5] = top;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < (int)blockDim.x / 32; ++i) top = max(top, s_top[i]);
        if (top) atomicMax(reinterpret_cast<unsigned long long *>(&L.lc->smax), top);
    }
}

__global__ void k_refresh_begin(Dev d, Learn L, int gate)
{
    if (gate && done_gate(d)) return;
    L.lc->smax = 0;
    L.lc->pass_iter = d.ctl->iter;
}

// The 12 features of variable j, rounded to BF16: x/(u-l), (x-l)/(u-l),
// (u-x)/(u-l), min(tabu age, 64)/64, violated share, violated weighted share,
// last exact score / (1 + max |score|), iterations since the exact pass / 50,
// log2(1 + column length)/16, is_binary, is_integer, c_j / max |c|.
//
// The last four do not change: they are laid out once with the driver's state
// (column length through two gathers per variable, 19 us of each proposal over
// 200k variables, with the others, when each formed them).
__global__ void k_fixed_features(Dev d, Learn L, float cmax)
{
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < d.n; j += gridDim.x * blockDim.x) {
        const int q = d.vpos[j];
        const int len = (d.ci_ptr[q + 1] - d.ci_ptr[q]) + (d.cf_ptr[q + 1] - d.cf_ptr[q]);
        const int vt = d.vtype[j];
        const float f8 = log2f(1.0f + (float)len) / 16.0f;
        const float f9 = vt == kVarBin ? 1.0f : 0.0f, f10 = vt == kVarInt ? 1.0f : 0.0f;
        const float f11 = cmax > 0.0f ? (float)d.obj[j] / cmax : 0.0f;
        const __nv_bfloat162 a = __floats2bfloat162_rn(f8, f9), b = __floats2bfloat162_rn(f10, f11);
        L.fixed[j] = make_uint2(*reinterpret_cast<const unsigned *>(&a), *reinterpret_cast<const unsigned *>(&b));
    }
}

struct VarRaw {
    double x, l, u;
    long long s;
    int ti, td;
    float cv, cw;
    uint2 fx;
};

__device__ __forceinline__ VarRaw var_load(const Dev &d, const Learn &L, int j)
{
    VarRaw v;
    v.x = d.x[j]; v.l = d.lb[j]; v.u = d.ub[j];
    v.s = L.s_last[j];
    v.ti = d.tabu_inc[j]; v.td = d.tabu_dec[j];
    v.cv = L.colviol[j]; v.cw = L.colwv[j];
    v.fx = L.fixed[j];
    return v;
}

__device__ __forceinline__ void var_features(const VarRaw &v, int tenure, long long iter, float smax, float since,
                                             __nv_bfloat162 (&out)[kF / 2])
{
    const bool fin = isfinite(v.u - v.l) && v.u > v.l;
    const float w = fin ? (float)(v.u - v.l) : 1.0f;
    float f[8];
    f[0] = fin ? (float)v.x / w : 0.0f;
    f[1] = fin ? (float)(v.x - v.l) / w : 0.0f;
    f[2] = fin ? (float)(v.u - v.x) / w : 0.0f;
    const int st = v.ti > v.td ? v.ti : v.td;
    long long age = st > 0 ? iter - (long long)(st - 1 - tenure) : 64;
    if (age > 64) age = 64;
    f[3] = (float)age / 64.0f;
    f[4] = v.cv;
    f[5] = v.cw;
    f[6] = (float)v.s / (1.0f + smax);
    f[7] = since / 50.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i) out[i] = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);
    out[4] = *reinterpret_cast<const __nv_bfloat162 *>(&v.fx.x);
    out[5] = *reinterpret_cast<const __nv_bfloat162 *>(&v.fx.y);
}

__global__ void k_features(Dev d, Learn L)
{
    const long long iter = d.ctl->iter;
    const float smax = (float)L.lc->smax;
    const float since = (float)(iter - L.lc->pass_iter);
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < d.n; j += gridDim.x * blockDim.x) {
        __nv_bfloat162 f[kF / 2];
        var_features(var_load(d, L, j), d.tenure, iter, smax, since, f);
        // a row is 24 bytes, 8-byte aligned
        uint2 *out = reinterpret_cast<uint2 *>(L.feat + (long long)j * kF);
        const uint2 *in = reinterpret_cast<const uint2 *>(f);
#pragma unroll
        for (int k = 0; k < kF / 4; ++k) out[k] = in[k];
    }
}

// Targets: the last exact scores scaled by 1 / (1 + max |score|).  Formed here:
// the scores went to the host and back before (a logged pass of 90k variables
// 399 -> 300 us with the copies and the wait gone).
__global__ void k_targets(int n, Learn L, float *target)
{
    const double sc = __ddiv_rn(1.0, __dadd_rn(1.0, (double)L.lc->smax));
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
        target[j] = (float)__dmul_rn((double)L.s_last[j], sc);
}

// ----------------------------------------------------------------- network

// A tile of kTileRows rows in shared memory.  Activations are stored by
// column (hT[j][row]), so that a thread's 4 rows are one 16-byte load.
struct MlpTile {
    float w1[kF * kH], b1[kH];
    float w2[kH * kH], b2[kH];
    float w3[kH], b3[4];
    float xT[kF * kTPad];
    float h1T[kH * kTPad];
    float h2T[kH * kTPad];
    float out[kTileRows];
};

__device__ __forceinline__ void mlp_load_weights(MlpTile &s, const __nv_bfloat16 *w)
{
    for (int i = threadIdx.x; i < kF * kH; i += kTileThreads) s.w1[i] = __bfloat162float(w[kOffW1 + i]);
    for (int i = threadIdx.x; i < kH * kH; i += kTileThreads) s.w2[i] = __bfloat162float(w[kOffW2 + i]);
    if (threadIdx.x < kH) {
        s.b1[threadIdx.x] = __bfloat162float(w[kOffB1 + threadIdx.x]);
        s.b2[threadIdx.x] = __bfloat162float(w[kOffB2 + threadIdx.x]);
        s.w3[threadIdx.x] = __bfloat162float(w[kOffW3 + threadIdx.x]);
    }
    if (threadIdx.x == 0) s.b3[0] = __bfloat162float(w[kOffB3]);
}

// One layer of the tile: act[j][r] = relu(b[j] + sum_k in[k][r] W[k][j]), terms
// added in increasing k with FMAs; rows past `rows` become 0.  A thread owns
// rows 4 (t / 16) .. + 3 and columns 4 (t % 16) .. + 3: per k two 16-byte loads
// for 16 FMAs.
__device__ __forceinline__ void mlp_layer(const float *inT, const float *W, const float *b, int K, int rows, float *actT)
{
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    float acc[4][4];
    const float4 bb = *reinterpret_cast<const float4 *>(b + 4 * tx);
#pragma unroll
    for (int r = 0; r < 4; ++r) { acc[r][0] = bb.x; acc[r][1] = bb.y; acc[r][2] = bb.z; acc[r][3] = bb.w; }
#pragma unroll 4
    for (int k = 0; k < K; ++k) {
        const float4 x = *reinterpret_cast<const float4 *>(inT + k * kTPad + 4 * ty);
        const float4 w = *reinterpret_cast<const float4 *>(W + k * kH + 4 * tx);
        const float xr[4] = {x.x, x.y, x.z, x.w}, wc[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) acc[r][c] = __fmaf_rn(xr[r], wc[c], acc[r][c]);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
        float4 v;
        v.x = 4 * ty < rows ? fmaxf(acc[0][c], 0.0f) : 0.0f;
        v.y = 4 * ty + 1 < rows ? fmaxf(acc[1][c], 0.0f) : 0.0f;
        v.z = 4 * ty + 2 < rows ? fmaxf(acc[2][c], 0.0f) : 0.0f;
        v.w = 4 * ty + 3 < rows ? fmaxf(acc[3][c], 0.0f) : 0.0f;
        *reinterpret_cast<float4 *>(actT + (4 * tx + c) * kTPad + 4 * ty) = v;
    }
}

// Forward pass of the tile's rows [r0, r0 + rows): s.out; ends with a barrier.
__device__ __forceinline__ void mlp_tile_forward(MlpTile &s, const __nv_bfloat16 *x, long long r0, int rows)
{
    __syncthreads();   // the previous tile is done with the buffers
    for (int i = threadIdx.x; i < kTileRows * kF; i += kTileThreads) {
        const int r = i / kF, f = i % kF;
        s.xT[f * kTPad + r] = r < rows ? __bfloat162float(x[r0 * kF + i]) : 0.0f;
    }
    __syncthreads();
    mlp_layer(s.xT, s.w1, s.b1, kF, rows, s.h1T);
    __syncthreads();
    mlp_layer(s.h1T, s.w2, s.b2, kH, rows, s.h2T);
    __syncthreads();
    if (threadIdx.x < kTileRows) {
        float o = s.b3[0];
#pragma unroll 8
        for (int j = 0; j < kH; ++j) o = __fmaf_rn(s.h2T[j * kTPad + threadIdx.x], s.w3[j], o);
        s.out[threadIdx.x] = o;
    }
    __syncthreads();
}

// Forward pass (FP32 activations; every sum in increasing index with FMAs): a
// persistent grid over the tiles.  Bound by the FP32 FMAs and their operand
// loads from shared memory: a 4 x 4 block per thread reads 2 words an FMA less
// than one row per thread did.
__global__ void __launch_bounds__(kTileThreads) k_mlp_forward(const __nv_bfloat16 *w, const __nv_bfloat16 *x, long long n,
                                                              float *y)
{
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    MlpTile &s = *reinterpret_cast<MlpTile *>(mlp_smem);
    mlp_load_weights(s, w);
    const long long tiles = (n + kTileRows - 1) / kTileRows;
    for (long long t = blockIdx.x; t < tiles; t += gridDim.x) {
        const long long r0 = t * kTileRows;
        const int rows = (int)(n - r0 < kTileRows ? n - r0 : kTileRows);
        mlp_tile_forward(s, x, r0, rows);
        if ((int)threadIdx.x < rows) y[r0 + threadIdx.x] = s.out[threadIdx.x];
    }
}

// Order-preserving bits of a float.
__device__ __forceinline__ unsigned fkey(float v)
{
    const unsigned b = __float_as_uint(v);
    return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// The digit of the `need`-th largest key, from a histogram of it over the keys
// that match the digits before (a block-wide suffix scan, two bins a thread);
// need becomes its rank among the keys of that digit.
__device__ __forceinline__ int topk_pick(const unsigned *hist, int &need)
{
    __shared__ int wsum[kTkThreads / 32];
    __shared__ int s_dig, s_need;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // thread t owns bins 2047 - 2t and 2046 - 2t: higher bins first
    const uint2 v = __ldcg(reinterpret_cast<const uint2 *>(hist) + 1023 - threadIdx.x);
    const int c0 = (int)v.y, tot = c0 + (int)v.x;
    int incl = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(FULLMASK, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    const int ws = wsum[lane];
    const int before = incl - tot + __reduce_add_sync(FULLMASK, lane < wid ? ws : 0);
    if (before < need && before + tot >= need) {
        const bool first = before + c0 >= need;
        s_dig = 2047 - 2 * (int)threadIdx.x - (first ? 0 : 1);
        s_need = need - before - (first ? 0 : c0);
    }
    __syncthreads();
    need = s_need;
    return s_dig;
}

// True in the CTA that is the last of the grid to get here (all threads call
// it; what the others wrote before is visible to it).
__device__ bool last_cta(const Learn &L)
{
    __shared__ int s_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        s_last = atomicAdd(&L.lc->ticket, 1u) == gridDim.x - 1;
        if (s_last) L.lc->ticket = 0u;
    }
    __syncthreads();
    if (s_last) __threadfence();
    return s_last != 0;
}

// Features and predictions of every variable, with the first histogram of the
// top-k: the forward pass with the second layer on the tensor cores.  A warp
// takes 32 variables: each lane forms one variable's features (BF16, kept in
// shared memory), then for the two 16-row tiles together every lane computes, in
// FP32 on the CUDA cores, exactly the first-layer activations its A fragments of
// mma.m16n8k16 need (rows g and g + 8 of a tile, 16 hidden units per 16-wide K
// chunk; the 12 weights of a unit are three 16-byte loads for 4 rows), rounds
// them to BF16, and the warp multiplies the tiles by W2 (64 x 64, BF16 from
// shared memory, one fragment load for both) into FP32 accumulators; the output
// layer is reduced across the four lanes that share a row.  Activations of the
// first layer are BF16 here (FP32 in k_mlp_forward and in training).  Bound by
// the operand loads from shared memory and the first layer's FMAs; the next
// group's inputs are loaded under this one's arithmetic.  200k variables: 27 us,
// against 49 as three kernels (features 19, forward 25 one tile at a time,
// histogram 5).
__global__ void __launch_bounds__(kPropThreads, 3) k_propose_scores(Dev d, Learn L, const __nv_bfloat16 *w, int gate)
{
    constexpr int kPadF = kF + 4;                               // padded feature rows
    __shared__ __align__(16) float s1[kH * kF + kH];            // W1 by hidden unit ([c][f]), b1
    __shared__ float s2[kH + kH + 1];                           // b2, w3, b3
    __shared__ __align__(16) unsigned short sW2t[kH * (kH + 8)];  // W2 transposed, [n][k], padded rows
    __shared__ __align__(16) float sx[kPropThreads / 32][32 * kPadF];  // features of each warp's 32 variables
    __shared__ unsigned h[2048];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const int n = d.n, groups = (n + 31) / 32, step = gridDim.x * (kPropThreads / 32);
    int gr = blockIdx.x * (kPropThreads / 32) + warp;
    chain_next();
    // the weights do not depend on the kernel before
    for (int i = threadIdx.x; i < kF * kH; i += blockDim.x) s1[(i % kH) * kF + i / kH] = __bfloat162float(w[kOffW1 + i]);
    for (int i = threadIdx.x; i < kH; i += blockDim.x) s1[kF * kH + i] = __bfloat162float(w[kOffB1 + i]);
    for (int i = threadIdx.x; i < 2 * kH + 1; i += blockDim.x) s2[i] = __bfloat162float(w[kOffB2 + i]);
    for (int i = threadIdx.x; i < 2048; i += blockDim.x) h[i] = 0u;
    const unsigned short *wraw = reinterpret_cast<const unsigned short *>(w);
#pragma unroll 8
    for (int i = threadIdx.x; i < kH * kH; i += kPropThreads) {
        const int kk = i / kH, nn = i % kH;                     // W2[kk][nn]
        sW2t[nn * (kH + 8) + kk] = wraw[kOffW2 + i];
    }
    chain_wait();
    if (gate && done_gate(d)) return;
    __syncthreads();
    VarRaw raw = var_load(d, L, min(gr * 32 + lane, n - 1));
    const long long iter = d.ctl->iter;
    const float smax = (float)L.lc->smax;
    const float since = (float)(iter - L.lc->pass_iter);
    float *xw = sx[warp];
    for (; gr < groups; gr += step) {
        {
            __nv_bfloat162 f[kF / 2];
            var_features(raw, d.tenure, iter, smax, since, f);
            __syncwarp();
#pragma unroll
            for (int i = 0; i < kF / 2; i += 2) {
                const float2 a = __bfloat1622float2(f[i]), b = __bfloat1622float2(f[i + 1]);
                *reinterpret_cast<float4 *>(xw + lane * kPadF + 2 * i) = make_float4(a.x, a.y, b.x, b.y);
            }
            __syncwarp();
        }
        // the next group's loads run under this one's arithmetic
        raw = var_load(d, L, min((int)min((long long)gr + step, (long long)groups - 1) * 32 + lane, n - 1));
        // rows g, g + 8 (first tile), g + 16, g + 24 (second)
        float x[4][kF];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int i = 0; i < kF; i += 4) {
                const float4 a = *reinterpret_cast<const float4 *>(xw + (8 * r + g) * kPadF + i);
                x[r][i] = a.x; x[r][i + 1] = a.y; x[r][i + 2] = a.z; x[r][i + 3] = a.w;
            }
        float acc[2][8][4];
#pragma unroll
        for (int nt = 0; nt < 8; ++nt)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[0][nt][e] = acc[1][nt][e] = 0.0f;
#pragma unroll 1
        for (int kc = 0; kc < 4; ++kc) {
            // A fragments: hidden units 16 kc + {2t, 2t+1} and {2t+8, 2t+9}
            unsigned a[2][4];
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                float v[4][2];
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int c = 16 * kc + 2 * t + 8 * half + e;
                    const float b = s1[kF * kH + c];
#pragma unroll
                    for (int r = 0; r < 4; ++r) v[r][e] = b;
#pragma unroll
                    for (int i = 0; i < kF; i += 4) {
                        const float4 wv = *reinterpret_cast<const float4 *>(s1 + c * kF + i);
#pragma unroll
                        for (int r = 0; r < 4; ++r) {
                            v[r][e] = __fmaf_rn(x[r][i], wv.x, v[r][e]);
                            v[r][e] = __fmaf_rn(x[r][i + 1], wv.y, v[r][e]);
                            v[r][e] = __fmaf_rn(x[r][i + 2], wv.z, v[r][e]);
                            v[r][e] = __fmaf_rn(x[r][i + 3], wv.w, v[r][e]);
                        }
                    }
                }
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const __nv_bfloat162 pr = __floats2bfloat162_rn(fmaxf(v[r][0], 0.0f), fmaxf(v[r][1], 0.0f));
                    a[r >> 1][(r & 1) + 2 * half] = *reinterpret_cast<const unsigned *>(&pr);
                }
            }
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                // B fragment: k = 16 kc + {2t, 2t+1} and {2t+8, 2t+9}, n = 8 nt + g
                const unsigned short *bp = sW2t + (8 * nt + g) * (kH + 8) + 16 * kc + 2 * t;
                const unsigned b0 = *reinterpret_cast<const unsigned *>(bp);
                const unsigned b1 = *reinterpret_cast<const unsigned *>(bp + 8);
#pragma unroll
                for (int m = 0; m < 2; ++m)
                    asm volatile(
                        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
                        "{%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                        : "+f"(acc[m][nt][0]), "+f"(acc[m][nt][1]), "+f"(acc[m][nt][2]), "+f"(acc[m][nt][3])
                        : "r"(a[m][0]), "r"(a[m][1]), "r"(a[m][2]), "r"(a[m][3]), "r"(b0), "r"(b1));
            }
        }
        // output layer: rows g (acc[.][.][0..1]) and g + 8 (acc[.][.][2..3]) of a tile, columns 8 nt + 2t (+1)
#pragma unroll
        for (int m = 0; m < 2; ++m) {
            float o0 = 0.0f, o1 = 0.0f;
#pragma unroll
            for (int nt = 0; nt < 8; ++nt) {
                const int c = 8 * nt + 2 * t;
                o0 = __fmaf_rn(fmaxf(acc[m][nt][0] + s2[c], 0.0f), s2[kH + c], o0);
                o0 = __fmaf_rn(fmaxf(acc[m][nt][1] + s2[c + 1], 0.0f), s2[kH + c + 1], o0);
                o1 = __fmaf_rn(fmaxf(acc[m][nt][2] + s2[c], 0.0f), s2[kH + c], o1);
                o1 = __fmaf_rn(fmaxf(acc[m][nt][3] + s2[c + 1], 0.0f), s2[kH + c + 1], o1);
            }
            o0 += __shfl_xor_sync(FULLMASK, o0, 1);
            o0 += __shfl_xor_sync(FULLMASK, o0, 2);
            o1 += __shfl_xor_sync(FULLMASK, o1, 1);
            o1 += __shfl_xor_sync(FULLMASK, o1, 2);
            const int r0 = gr * 32 + 16 * m + g, r1 = r0 + 8;
            if (t == 0) {
                if (r0 < n) {
                    const float y = o0 + s2[2 * kH];
                    L.y[r0] = y;
                    atomicAdd(&h[fkey(y) >> 21], 1u);
                }
                if (r1 < n) {
                    const float y = o1 + s2[2 * kH];
                    L.y[r1] = y;
                    atomicAdd(&h[fkey(y) >> 21], 1u);
                }
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2048; i += blockDim.x)
        if (h[i]) atomicAdd(&L.hist[i], h[i]);
}

// Gradient of the mean squared error over n rows (scale 2/n), accumulated into
// grad[kNParams] and the sum of squared errors into loss[0] (FP32 atomics, one
// per parameter and CTA).  A CTA takes tiles of kTileRows rows in turn, keeps
// its share of the gradient in registers (16 weights of the second layer, 3 of
// the first per thread) and adds it once at the end.  Bound by the FP32 FMAs
// (0.9M a tile) and their shared-memory operands.  8 training steps of
// 8,192 rows and a forward pass of 100,003 take 370 us; with one row per thread
// and one parameter per thread and pass they took 697.
struct MlpGradTile {
    MlpTile f;
    float w2T[kH * kH];          // second layer transposed, [j][i]
    float gy[kTileRows];
};

__global__ void __launch_bounds__(kTileThreads) k_mlp_grad(const __nv_bfloat16 *w, const __nv_bfloat16 *x, const float *t,
                                                           long long n, float scale, float *grad, float *loss)
{
    extern __shared__ __align__(16) unsigned char mlp_smem[];
    MlpGradTile &g = *reinterpret_cast<MlpGradTile *>(mlp_smem);
    MlpTile &s = g.f;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    mlp_load_weights(s, w);
    for (int i = tid; i < kH * kH; i += kTileThreads) g.w2T[(i % kH) * kH + i / kH] = __bfloat162float(w[kOffW2 + i]);
    float gw2[4][4], gw1[3], gb = 0.0f, gw3 = 0.0f, gb3 = 0.0f, lsum = 0.0f;
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) gw2[i][j] = 0.0f;
    gw1[0] = gw1[1] = gw1[2] = 0.0f;
    float gb1 = 0.0f;
    const long long tiles = (n + kTileRows - 1) / kTileRows;
    for (long long tl = blockIdx.x; tl < tiles; tl += gridDim.x) {
        const long long r0 = tl * kTileRows;
        const int rows = (int)(n - r0 < kTileRows ? n - r0 : kTileRows);
        mlp_tile_forward(s, x, r0, rows);
        if (tid < kTileRows) {
            const float err = tid < rows ? s.out[tid] - t[r0 + tid] : 0.0f;
            g.gy[tid] = scale * err;
            lsum = __fmaf_rn(err, err, lsum);
        }
        __syncthreads();
        // output layer (threads 0..63: w3, 64: b3); then ga2 = gy w3 [h2 > 0] in place of h2
        if (tid < kH) {
            for (int r = 0; r < kTileRows; ++r) gw3 = __fmaf_rn(s.h2T[tid * kTPad + r], g.gy[r], gw3);
        } else if (tid == kH) {
            for (int r = 0; r < kTileRows; ++r) gb3 += g.gy[r];
        }
        __syncthreads();
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float4 *p = reinterpret_cast<float4 *>(s.h2T + (4 * tx + c) * kTPad + 4 * ty);
            const float4 y = *reinterpret_cast<const float4 *>(g.gy + 4 * ty);
            const float w3 = s.w3[4 * tx + c];
            float4 v = *p;
            v.x = v.x > 0.0f ? y.x * w3 : 0.0f;
            v.y = v.y > 0.0f ? y.y * w3 : 0.0f;
            v.z = v.z > 0.0f ? y.z * w3 : 0.0f;
            v.w = v.w > 0.0f ? y.w * w3 : 0.0f;
            *p = v;
        }
        __syncthreads();
        // gW2[i][j] = sum_r h1[r][i] ga2[r][j] for i = ty + 16 a, j = tx + 16 b
        // (strided, so that the 16-byte loads of 4 rows meet different banks)
#pragma unroll 2
        for (int r = 0; r < kTileRows; r += 4) {
            float4 h[4], q[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                h[a] = *reinterpret_cast<const float4 *>(s.h1T + (ty + 16 * a) * kTPad + r);
                q[a] = *reinterpret_cast<const float4 *>(s.h2T + (tx + 16 * a) * kTPad + r);
            }
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    gw2[a][b] = __fmaf_rn(h[a].x, q[b].x, gw2[a][b]);
                    gw2[a][b] = __fmaf_rn(h[a].y, q[b].y, gw2[a][b]);
                    gw2[a][b] = __fmaf_rn(h[a].z, q[b].z, gw2[a][b]);
                    gw2[a][b] = __fmaf_rn(h[a].w, q[b].w, gw2[a][b]);
                }
        }
        if (tid < kH)
            for (int r = 0; r < kTileRows; ++r) gb += s.h2T[tid * kTPad + r];
        // ga1 = (ga2 W2^T) [h1 > 0]
        float a1[4][4];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) a1[r][c] = 0.0f;
#pragma unroll 4
        for (int j = 0; j < kH; ++j) {
            const float4 q = *reinterpret_cast<const float4 *>(s.h2T + j * kTPad + 4 * ty);
            const float4 v = *reinterpret_cast<const float4 *>(g.w2T + j * kH + 4 * tx);
            const float qr[4] = {q.x, q.y, q.z, q.w}, vc[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
                for (int c = 0; c < 4; ++c) a1[r][c] = __fmaf_rn(qr[r], vc[c], a1[r][c]);
        }
        __syncthreads();   // h1 has been read by every thread
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            float4 *p = reinterpret_cast<float4 *>(s.h1T + (4 * tx + c) * kTPad + 4 * ty);
            float4 v = *p;
            v.x = v.x > 0.0f ? a1[0][c] : 0.0f;
            v.y = v.y > 0.0f ? a1[1][c] : 0.0f;
            v.z = v.z > 0.0f ? a1[2][c] : 0.0f;
            v.w = v.w > 0.0f ? a1[3][c] : 0.0f;
            *p = v;
        }
        __syncthreads();
        // gW1[f][i] for i = tid % 64, f = tid / 64 + 4 m
        {
            const int i = tid & (kH - 1), f0 = tid / kH;
            for (int r = 0; r < kTileRows; r += 4) {
                const float4 a = *reinterpret_cast<const float4 *>(s.h1T + i * kTPad + r);
#pragma unroll
                for (int m = 0; m < 3; ++m) {
                    const float4 v = *reinterpret_cast<const float4 *>(s.xT + (f0 + 4 * m) * kTPad + r);
                    gw1[m] = __fmaf_rn(v.x, a.x, gw1[m]);
                    gw1[m] = __fmaf_rn(v.y, a.y, gw1[m]);
                    gw1[m] = __fmaf_rn(v.z, a.z, gw1[m]);
                    gw1[m] = __fmaf_rn(v.w, a.w, gw1[m]);
                }
                if (f0 == 0) gb1 += (a.x + a.y) + (a.z + a.w);
            }
        }
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) atomicAdd(grad + kOffW2 + (ty + 16 * a) * kH + tx + 16 * b, gw2[a][b]);
#pragma unroll
    for (int m = 0; m < 3; ++m) atomicAdd(grad + kOffW1 + (tid / kH + 4 * m) * kH + (tid & (kH - 1)), gw1[m]);
    if (tid < kH) {
        atomicAdd(grad + kOffB1 + tid, gb1);
        atomicAdd(grad + kOffB2 + tid, gb);
        atomicAdd(grad + kOffW3 + tid, gw3);
    }
    if (tid == kH) atomicAdd(grad + kOffB3, gb3);
    if (tid < kTileRows) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(FULLMASK, lsum, o);
        if ((tid & 31) == 0) atomicAdd(loss, lsum);
    }
}

// Adam on FP32 master parameters; writes the BF16 copy and clears the gradient.
__global__ void k_adam(float *w32, __nv_bfloat16 *wbf, float *m, float *v, float *g, int n, float lr, float b1,
                       float b2, float eps, float c1, float c2)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.0f - b1) * gi;
    const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float wi = w32[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w32[i] = wi;
    wbf[i] = __float2bfloat16_rn(wi);
    g[i] = 0.0f;
}

// ------------------------------------------------------------------- top-k

// The variables with the k largest predictions, ties by the lower index, in
// index order (above the k-th value first, then those equal to it): a radix
// select over the order-preserving keys in one cluster.  The first digit (bits
// 31..21) is counted where the predictions are made; a warp owns a run of
// consecutive keys, keeps the first kTkKeys of it in shared memory and counts
// the second (bits 20..10) and third digit (bits 9..0) of those that match, then
// the keys above and equal, then writes.  Bound by its three cluster-wide
// barriers and the L2 round trip of the counts around each; 18 us for
// 200k variables (cold cache) against 44 with a launch over the whole GPU for
// each step.
__global__ void __launch_bounds__(kTkThreads) k_topk(Dev d, Learn L, int n, int k, int gate)
{
    chain_next();
    chain_wait();
    if (gate && done_gate(d)) return;
    extern __shared__ unsigned tk_keys[];
    __shared__ unsigned h[2048];
    __shared__ int sg[kTkThreads / 32], se[kTkThreads / 32];
    cg::cluster_group cl = cg::this_cluster();
    const int C = (int)gridDim.x, rank = (int)blockIdx.x;   // the grid is one cluster
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nw = C * (kTkThreads / 32);
    const int chunk = ((n + nw - 1) / nw + 31) & ~31;
    const long long lo = (long long)(rank * (kTkThreads / 32) + wid) * chunk;
    const int j0 = (int)(lo < n ? lo : n), cnt = min(chunk, n - j0);
    unsigned *kw = tk_keys + wid * kTkKeys;
    auto key_at = [&](int i) { return i < kTkKeys ? kw[i] : fkey(__ldcg(L.y + j0 + i)); };
    for (int i = threadIdx.x; i < 2048; i += kTkThreads) h[i] = 0u;
#pragma unroll 8
    for (int i = lane; i < min(cnt, kTkKeys); i += 32) kw[i] = fkey(__ldcg(L.y + j0 + i));
    int need = k;
    unsigned prefix = (unsigned)topk_pick(L.hist, need);
    for (int i = lane; i < cnt; i += 32) {
        const unsigned key = key_at(i);
        if (key >> 21 == prefix) atomicAdd(&h[(key >> 10) & 0x7ffu], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 2048; i += kTkThreads) {
        if (h[i]) atomicAdd(&L.hist[2048 + i], h[i]);
        h[i] = 0u;
    }
    cl.sync();
    // every CTA has read the first histogram: clear it for the next selection
    if (rank == 0)
        for (int i = threadIdx.x; i < 2048; i += kTkThreads) L.hist[i] = 0u;
    prefix = (prefix << 11) | (unsigned)topk_pick(L.hist + 2048, need);
    for (int i = lane; i < cnt; i += 32) {
        const unsigned key = key_at(i);
        if (key >> 10 == prefix) atomicAdd(&h[key & 0x3ffu], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 1024; i += kTkThreads)
        if (h[i]) atomicAdd(&L.hist[4096 + i], h[i]);
    cl.sync();
    if (rank == 0)
        for (int i = threadIdx.x; i < 2048; i += kTkThreads) L.hist[2048 + i] = 0u;
    const unsigned thr = (prefix << 10) | (unsigned)topk_pick(L.hist + 4096, need);
    int gt = 0, eq = 0;
    for (int i = lane; i < chunk; i += 32) {
        const unsigned key = i < cnt ? key_at(i) : 0u;
        gt += __popc(__ballot_sync(FULLMASK, i < cnt && key > thr));
        eq += __popc(__ballot_sync(FULLMASK, i < cnt && key == thr));
    }
    if (lane == 0) { sg[wid] = gt; se[wid] = eq; }
    __syncthreads();
    const int tg = __reduce_add_sync(FULLMASK, sg[lane]), te = __reduce_add_sync(FULLMASK, se[lane]);
    int pg = __reduce_add_sync(FULLMASK, lane < wid ? sg[lane] : 0);
    int pe = __reduce_add_sync(FULLMASK, lane < wid ? se[lane] : 0);
    if (threadIdx.x == 0) {
        L.bcnt[2 * rank] = tg;
        L.bcnt[2 * rank + 1] = te;
    }
    cl.sync();
    if (rank == 0)
        for (int i = threadIdx.x; i < 1024; i += kTkThreads) L.hist[4096 + i] = 0u;
    const int cgt = lane < C ? __ldcg(L.bcnt + 2 * lane) : 0, ceq = lane < C ? __ldcg(L.bcnt + 2 * lane + 1) : 0;
    const int total_gt = __reduce_add_sync(FULLMASK, cgt);
    pg += __reduce_add_sync(FULLMASK, lane < rank ? cgt : 0);
    pe += __reduce_add_sync(FULLMASK, lane < rank ? ceq : 0);
    for (int i = lane; i < chunk; i += 32) {
        const unsigned key = i < cnt ? key_at(i) : 0u;
        const unsigned mg = __ballot_sync(FULLMASK, i < cnt && key > thr);
        const unsigned me = __ballot_sync(FULLMASK, i < cnt && key == thr);
        const unsigned below = (1u << lane) - 1u;
        if (mg >> lane & 1u) L.list[pg + __popc(mg & below)] = j0 + i;
        const int r = pe + __popc(me & below);
        if ((me >> lane & 1u) && r < need) L.list[total_gt + r] = j0 + i;
        pg += __popc(mg);
        pe += __popc(me);
    }
}

// ------------------------------------------------ exact scores of the subset

__device__ __forceinline__ int lflip_f(bool v0, bool v1, bool dec)
{
    return 2 * ((int)v0 - (int)v1) + ((v0 && v1) ? (dec ? 1 : -1) : 0);
}

__device__ __forceinline__ unsigned long long dkey_bits(long long b)
{
    const unsigned long long u = (unsigned long long)b;
    return (u & 0x8000000000000000ull) ? ~u : (u | 0x8000000000000000ull);
}

__device__ __forceinline__ long long flip_sign(long long b)
{
    long long r;
    asm("xor.b64 %0, %1, 0x8000000000000000;" : "=l"(r) : "l"(b));
    return r;
}

// Hand the proposal's move to the apply kernel of the exact path.
__device__ __forceinline__ void learn_select(const Dev &d, const Learn &L)
{
    Ctl *c = d.ctl;
    const unsigned long long key = __ldcg(&L.lc->key);
    L.lc->key = 0ull;
    if (key != 0ull) {
        const int j = (1 << kVarBits) - 1 - (int)(key & ((1ull << kVarBits) - 1));
        const double x = d.x[j];
        c->mv_var = j;
        c->mv_s = (long long)(key >> kVarBits);
        c->mv_dc = 0;
        c->mv_old = x;
        c->mv_new = d.vtype[j] == kVarBin ? (__double_as_longlong(x) == 0 ? 1.0 : 0.0) : L.xh[j];
    } else {
        c->mv_var = -1;
        c->mv_s = 0;
        c->mv_dc = 0;
        c->mv_new = 0.0;
        c->mv_old = 0.0;
    }
}

// Flip score of every listed binary variable (8 lanes per variable, as the
// exact binary kernel); the best admissible positive flip is folded into
// lc->key with one 64-bit atomicMax (larger score, then lower variable).  Row
// states are read through L2: the apply kernel before may still be writing them
// when this one starts.
// select: the last CTA hands the move to the apply kernel.
__global__ void __launch_bounds__(256) k_subset_eval(Dev d, Learn L, int k, int select, int gate)
{
    chain_next();
    chain_wait();
    if (gate && done_gate(d)) return;
    const int lane = threadIdx.x & 31, g = lane >> 3, sub = lane & 7;
    const long long iter = d.ctl->iter, nviol = d.ctl->nviol, bestnv = d.ctl->best_nviol;
    const int nwarps = gridDim.x * (blockDim.x >> 5);
    for (int base = (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 4; base < k; base += nwarps * 4) {
        const int idx = base + g;
        const int jl = idx < k ? L.list[idx] : 0;
        const bool live = idx < k && d.vtype[jl] == kVarBin;   // other columns: k_subset_eval_nb
        const int j = live ? jl : 0;
        const int q = d.vpos[j];
        const bool up = __double_as_longlong(d.x[j]) == 0;
        long long s = 0;
        int dc = 0;
        // integral rows
        {
            const int e0 = d.ci_ptr[q], e1 = live ? d.ci_ptr[q + 1] : e0;
            int len = e1 - e0, lmax = len;
#pragma unroll
            for (int o = 16; o >= 8; o >>= 1) lmax = max(lmax, __shfl_xor_sync(FULLMASK, lmax, o));
            for (int v0 = 0; v0 < lmax; v0 += 8) {
                const int v = v0 + sub;
                if (v < len) {
                    const int e = e0 + v;
                    const int4 st = __ldcg(reinterpret_cast<const int4 *>(d.rs + d.ci_row[e]));
                    const long long r = i4_r(st);
                    const int ad = up ? d.ci_val[e] : -d.ci_val[e];
                    const long long r1 = r + ad;
                    s += (long long)lflip_f(r > 0, r1 > 0, ad < 0) * st.z;
                    dc += (int)(r1 > 0) - (int)(r > 0);
                    if (st.w >= 0) {
                        s += (long long)lflip_f(r < 0, r1 < 0, ad > 0) * st.w;
                        dc += (int)(r1 < 0) - (int)(r < 0);
                    }
                }
            }
        }
        // other rows: violated <=> m < 0; violated after the move <=> change > m
        {
            const int e0 = d.cf_ptr[q], e1 = live ? d.cf_ptr[q + 1] : e0;
            int len = e1 - e0, lmax = len;
#pragma unroll
            for (int o = 16; o >= 8; o >>= 1) lmax = max(lmax, __shfl_xor_sync(FULLMASK, lmax, o));
            for (int v0 = 0; v0 < lmax; v0 += 8) {
                const int v = v0 + sub;
                if (v < len) {
                    const int e = e0 + v;
                    const int4 *st = reinterpret_cast<const int4 *>(d.rs + d.cf_row[e]);
                    const int4 s0 = __ldcg(st), s1 = __ldcg(st + 1);
                    const long long ab = __double_as_longlong(d.cf_val[e]);
                    const long long ad = up ? ab : flip_sign(ab);
                    const long long m1 = i4_r(s1);
                    const long long m2 = (long long)(((unsigned long long)(unsigned)s1.w << 32) | (unsigned)s1.z);
                    const bool neg = ad < 0;
                    const bool v0b = m1 < 0, v1b = dkey_bits(ad) > dkey_bits(m1);
                    s += (long long)lflip_f(v0b, v1b, neg) * s0.z;
                    dc += (int)v1b - (int)v0b;
                    if (s0.w >= 0) {
                        const bool u0 = m2 < 0, u1 = dkey_bits(flip_sign(ad)) > dkey_bits(m2);
                        s += (long long)lflip_f(u0, u1, !neg) * s0.w;
                        dc += (int)u1 - (int)u0;
                    }
                }
            }
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
            s += __shfl_xor_sync(FULLMASK, s, o);
            dc += __shfl_xor_sync(FULLMASK, dc, o);
        }
        if (sub == 0 && live && s > 0) {
            const int stamp = up ? d.tabu_inc[j] : d.tabu_dec[j];
            if (iter >= (long long)stamp || nviol + (long long)dc < bestnv) {
                const unsigned long long key =
                    ((unsigned long long)s << kVarBits) | (unsigned long long)((1 << kVarBits) - 1 - j);
                atomicMax(&L.lc->key, key);
            }
        }
    }
    if (select && last_cta(L) && threadIdx.x == 0) learn_select(d, L);
}

__global__ void k_learn_select(Dev d, Learn L, int gate)
{
    if (gate && done_gate(d)) return;
    learn_select(d, L);
}

// At an exact pass: the proposal misses when the exact best score exceeds the
// best score found in the proposed subset.
__global__ void k_learn_miss(Dev d, Learn L, int gate)
{
    if (gate && done_gate(d)) return;
    const unsigned long long key = L.lc->key;
    L.lc->key = 0ull;
    const long long ls = key ? (long long)(key >> kVarBits) : 0;
    const Ctl *c = d.ctl;
    L.lc->passes += 1;
    if (c->mv_var >= 0 && c->mv_s > ls) L.lc->misses += 1;
}

}  // namespace
}  // namespace chap

// ------------------------------------------------------------------ host

namespace chap {

struct LearnHost {
    Learn L{};
    int tk_ctas = 8;             // CTAs of the top-k cluster
    std::vector<void *> allocs;
    cudaGraphExec_t gexec = nullptr;
    int g_key[4] = {0, 0, 0, 0};   // topk, exact_every, propose_every, graph weights pointer (low bits)
    const void *g_w = nullptr;
    LearnCtl *h_lc = nullptr;      // pinned
    float cmax = 0.0f;
};

void learn_free(chap_bs *h)
{
    if (!h || !h->learn) return;
    LearnHost *lh = static_cast<LearnHost *>(h->learn);
    if (lh->gexec) cudaGraphExecDestroy(lh->gexec);
    for (void *p : lh->allocs) cudaFree(p);
    if (lh->h_lc) cudaFreeHost(lh->h_lc);
    delete lh;
    h->learn = nullptr;
}

namespace {

template <class T>
T *lalloc(LearnHost *lh, size_t count)
{
    void *p = nullptr;
    if (cudaMalloc(&p, sizeof(T) * std::max<size_t>(count, 1)) != cudaSuccess) {
        cudaGetLastError();
        return nullptr;
    }
    lh->allocs.push_back(p);
    return static_cast<T *>(p);
}

chap_status lfail(chap_bs *h, chap_status s, const std::string &msg)
{
    h->err = msg;
    return s;
}

#define LCK(h, expr, what)                                                                   \
    do {                                                                                     \
        cudaError_t e_ = (expr);                                                             \
        if (e_ != cudaSuccess) {                                                             \
            cudaGetLastError();                                                              \
            return lfail(h, CHAP_E_CUDA, std::string(what) + ": " + cudaGetErrorString(e_)); \
        }                                                                                    \
    } while (0)

int grid_n(long long n, int threads, int cap = 152 * 8)
{
    long long g = (n + threads - 1) / threads;
    return (int)std::max<long long>(1, std::min<long long>(g, cap));
}

// Adds the attribute of a chained launch to cfg (whose attrs, if any, are at) for
// the iterations of a captured run (51 -> 48 us an iteration of 5 kernels over 200k
// variables); a kernel launched by itself follows work of the
// caller's, which may still be writing the weights, and takes none.
void chain_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *at, int gate)
{
    if (!gate) return;
    at[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[cfg.numAttrs].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs += 1;
}

void topk_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute *at, int ctas, cudaStream_t st)
{
    cfg.gridDim = dim3((unsigned)ctas);
    cfg.blockDim = dim3(kTkThreads);
    cfg.dynamicSmemBytes = kTkSmem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)ctas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
}

// Cluster of the top-k kernel: 16 CTAs where the GPU can hold such a cluster, else 8.
cudaError_t topk_shape(LearnHost *lh)
{
    cudaError_t e = cudaFuncSetAttribute(k_topk, cudaFuncAttributeMaxDynamicSharedMemorySize, kTkSmem);
    if (e != cudaSuccess) return e;
    lh->tk_ctas = 8;
    if (cudaFuncSetAttribute(k_topk, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at[1];
        topk_config(cfg, at, kTkCtas, nullptr);
        int fits = 0;
        if (cudaOccupancyMaxActiveClusters(&fits, k_topk, &cfg) == cudaSuccess && fits > 0) lh->tk_ctas = kTkCtas;
    }
    cudaGetLastError();
    return cudaSuccess;
}

// Learned-driver state of the handle, created on first use.
chap_status ensure_learn(chap_bs *h, LearnHost **out)
{
    if (h->learn) {
        *out = static_cast<LearnHost *>(h->learn);
        return CHAP_OK;
    }
    LearnHost *lh = new (std::nothrow) LearnHost();
    if (!lh) return CHAP_E_OOM;
    const int n = h->n;
    Learn &L = lh->L;
    L.colviol = lalloc<float>(lh, n);
    L.colwv = lalloc<float>(lh, n);
    L.s_last = lalloc<long long>(lh, n);
    L.feat = lalloc<__nv_bfloat16>(lh, (size_t)n * kF);
    L.y = lalloc<float>(lh, n);
    L.fixed = lalloc<uint2>(lh, n);
    L.hist = lalloc<unsigned>(lh, 3 * 2048);
    L.bcnt = lalloc<int>(lh, 2 * kTkCtas);
    L.list = lalloc<int>(lh, n);
    L.xh = lalloc<double>(lh, n);
    L.lc = lalloc<LearnCtl>(lh, 1);
    bool ok = L.colviol && L.colwv && L.s_last && L.feat && L.y && L.fixed && L.hist && L.bcnt && L.list && L.xh && L.lc &&
              cudaMallocHost(&lh->h_lc, sizeof(LearnCtl)) == cudaSuccess;
    for (int j = 0; j < n; ++j) lh->cmax = std::max(lh->cmax, (float)std::fabs(h->obj[j]));
    cudaError_t e = cudaSuccess;
    if (ok) {
        e = topk_shape(lh);
        if (e == cudaSuccess) e = cudaMemsetAsync(L.colviol, 0, sizeof(float) * std::max(1, n), h->st);
        if (e == cudaSuccess) e = cudaMemsetAsync(L.colwv, 0, sizeof(float) * std::max(1, n), h->st);
        if (e == cudaSuccess) e = cudaMemsetAsync(L.s_last, 0, sizeof(long long) * std::max(1, n), h->st);
        if (e == cudaSuccess) e = cudaMemsetAsync(L.hist, 0, sizeof(unsigned) * 3 * 2048, h->st);
        if (e == cudaSuccess) e = cudaMemsetAsync(L.lc, 0, sizeof(LearnCtl), h->st);
        if (e == cudaSuccess) {
            k_fixed_features<<<grid_n(n, 256), 256, 0, h->st>>>(h->dev, L, lh->cmax);
            e = cudaGetLastError();
        }
        if (e == cudaSuccess) e = cudaStreamSynchronize(h->st);
    }
    if (!ok || e != cudaSuccess) {
        cudaGetLastError();
        h->learn = lh;
        learn_free(h);
        return ok ? CHAP_E_CUDA : CHAP_E_OOM;
    }
    h->learn = lh;
    *out = lh;
    return CHAP_OK;
}

// exact scores into s_last and the pass-time column features
cudaError_t launch_refresh(chap_bs *h, LearnHost *lh, int gate, cudaStream_t st)
{
    const Dev &d = h->dev;
    VarOut o{nullptr, lh->L.s_last, nullptr};
    cudaError_t e = launch_eval_gated(d, h->plan, o, gate, st);
    if (e == cudaSuccess) e = launch_select_gated(d, h->plan, gate, st);
    if (e != cudaSuccess) return e;
    k_refresh_begin<<<1, 1, 0, st>>>(d, lh->L, gate);
    // the refresh reads the state before the move; gated like the rest
    k_refresh<<<grid_n(d.n, 256), 256, 0, st>>>(d, lh->L);
    return cudaGetLastError();
}

cudaError_t launch_propose(chap_bs *h, LearnHost *lh, const __nv_bfloat16 *w, int k, int gate, cudaStream_t st)
{
    const Dev &d = h->dev;
    const Learn &L = lh->L;
    const int n = d.n;
    if (n < 1) return cudaSuccess;
    cudaLaunchConfig_t cfg{};
    cudaLaunchAttribute at[2];
    cfg.gridDim = dim3((unsigned)grid_n((n + 31) / 32 * 32LL, kPropThreads, 152 * 3));
    cfg.blockDim = dim3(kPropThreads);
    cfg.stream = st;
    chain_config(cfg, at, gate);
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_propose_scores, d, L, w, gate);
    if (e != cudaSuccess) return e;
    topk_config(cfg, at, lh->tk_ctas, st);
    chain_config(cfg, at, gate);
    return cudaLaunchKernelEx(&cfg, k_topk, d, L, n, k, gate);
}

// Exact scores of the listed variables; select: their best move goes to the
// apply kernel.
cudaError_t launch_subset(chap_bs *h, LearnHost *lh, int k, int select, int gate, cudaStream_t st)
{
    const bool nb = h->info.n_bin < h->n - h->info.n_fixed;
    const bool fuse = select && !nb && h->info.n_bin > 0;   // the flips' last CTA selects
    cudaError_t e = cudaSuccess;
    if (h->info.n_bin > 0) {
        cudaLaunchConfig_t cfg{};
        cudaLaunchAttribute at[1];
        cfg.gridDim = dim3((unsigned)grid_n((long long)k * 8, 256, 152 * 4));
        cfg.blockDim = dim3(256);
        cfg.stream = st;
        chain_config(cfg, at, gate);
        e = cudaLaunchKernelEx(&cfg, k_subset_eval, h->dev, lh->L, k, fuse ? 1 : 0, gate);
    }
    if (e == cudaSuccess && nb) e = launch_subset_nb(h->dev, h->plan, lh->L.list, k, lh->L.xh, &lh->L.lc->key, gate, st);
    if (e == cudaSuccess && select && !fuse) {
        k_learn_select<<<1, 1, 0, st>>>(h->dev, lh->L, gate);
        e = cudaGetLastError();
    }
    return e;
}

// Shared-memory limit of a network kernel, once per device (slot: kernel).
cudaError_t mlp_smem_limit(const void *fn, int slot, int bytes)
{
    constexpr int kMaxDevices = 64;
    static std::mutex s_mu;
    static bool s_set[kMaxDevices][2] = {};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(s_mu);
    if (s_set[dev][slot]) return cudaSuccess;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess) s_set[dev][slot] = true;
    return e;
}

}  // namespace
}  // namespace chap

using namespace chap;

extern "C" {

chap_status chap_bs_refresh_features(chap_bs *h)
{
    if (!h) return CHAP_E_INVALID;
    if (h->broken) return lfail(h, CHAP_E_STATE, "handle unusable after a CUDA fault");
    if (own_scratch_ok(h) != CHAP_OK || whole_instance_ok(h) != CHAP_OK) return CHAP_E_STATE;
    LearnHost *lh = nullptr;
    chap_status s = ensure_learn(h, &lh);
    if (s != CHAP_OK) return lfail(h, s, "learned-driver state");
    LCK(h, launch_refresh(h, lh, 0, h->st), "refresh");
    LCK(h, cudaStreamSynchronize(h->st), "synchronise");
    return CHAP_OK;
}

chap_status chap_bs_features(chap_bs *h, uint16_t *feat, float *target)
{
    if (!h) return CHAP_E_INVALID;
    if (h->broken) return lfail(h, CHAP_E_STATE, "handle unusable after a CUDA fault");
    LearnHost *lh = nullptr;
    chap_status s = ensure_learn(h, &lh);
    if (s != CHAP_OK) return lfail(h, s, "learned-driver state");
    k_features<<<grid_n(h->n, 256), 256, 0, h->st>>>(h->dev, lh->L);
    LCK(h, cudaGetLastError(), "features");
    if (feat && h->n)
        LCK(h, cudaMemcpyAsync(feat, lh->L.feat, sizeof(uint16_t) * kF * (size_t)h->n, cudaMemcpyDeviceToDevice, h->st),
            "copy features");
    if (target && h->n) {
        k_targets<<<grid_n(h->n, 256), 256, 0, h->st>>>(h->n, lh->L, target);
        LCK(h, cudaGetLastError(), "targets");
    }
    LCK(h, cudaStreamSynchronize(h->st), "synchronise");
    return CHAP_OK;
}

chap_status chap_bs_propose(chap_bs *h, const uint16_t *weights, int32_t k, int32_t *list, float *pred)
{
    if (!h || !weights || k < 1) return h ? lfail(h, CHAP_E_INVALID, "bad proposal arguments") : CHAP_E_INVALID;
    if (h->broken) return lfail(h, CHAP_E_STATE, "handle unusable after a CUDA fault");
    LearnHost *lh = nullptr;
    chap_status s = ensure_learn(h, &lh);
    if (s != CHAP_OK) return lfail(h, s, "learned-driver state");
    k = std::min(k, h->n);
    LCK(h, launch_propose(h, lh, reinterpret_cast<const __nv_bfloat16 *>(weights), k, 0, h->st), "proposal");
    if (list) LCK(h, cudaMemcpyAsync(list, lh->L.list, sizeof(int) * k, cudaMemcpyDeviceToDevice, h->st), "copy list");
    if (pred) LCK(h, cudaMemcpyAsync(pred, lh->L.y, sizeof(float) * h->n, cudaMemcpyDeviceToDevice, h->st), "copy predictions");
    LCK(h, cudaStreamSynchronize(h->st), "synchronise");
    return CHAP_OK;
}

chap_status chap_learned_run(chap_bs *h, const uint16_t *weights, const chap_learned_options *lo,
                             chap_learned_result *res)
{
    if (!h || !weights || !lo || !res) return h ? lfail(h, CHAP_E_INVALID, "NULL argument") : CHAP_E_INVALID;
    if (h->broken) return lfail(h, CHAP_E_STATE, "handle unusable after a CUDA fault");
    if (lo->topk < 1 || lo->exact_every < 1 || lo->propose_every < 1 || lo->max_iters < 0)
        return lfail(h, CHAP_E_INVALID, "bad learned-run options");
    if (own_scratch_ok(h) != CHAP_OK || whole_instance_ok(h) != CHAP_OK) return CHAP_E_STATE;
    if (h->n >= (1 << kVarBits))
        return lfail(h, CHAP_E_UNSUPPORTED, "the learned driver handles instances below 2^22 variables");
    LearnHost *lh = nullptr;
    chap_status s = ensure_learn(h, &lh);
    if (s != CHAP_OK) return lfail(h, s, "learned-driver state");
    const int k = std::min<int>(lo->topk, h->n);
    const auto t0 = std::chrono::steady_clock::now();
    LCK(h, cudaMemcpyAsync(h->h_ctl, h->dev.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, h->st), "read control");
    LCK(h, cudaStreamSynchronize(h->st), "synchronise");
    const long long iter0 = h->h_ctl->iter, moves0 = h->h_ctl->moves;
    if (iter0 + lo->max_iters + h->opt.tenure + 1 >= (long long)INT_MAX)
        return lfail(h, CHAP_E_UNSUPPORTED, "iteration counter would exceed the 32-bit tabu stamps");
    LCK(h, cudaMemsetAsync(&lh->L.lc->passes, 0, 2 * sizeof(long long), h->st), "reset counters");
    LCK(h, launch_begin_run(h->dev, lo->max_iters, lo->stop_at_feasible, h->st), "begin run");
    const __nv_bfloat16 *w = reinterpret_cast<const __nv_bfloat16 *>(weights);
    const int key[4] = {k, lo->exact_every, lo->propose_every, 0};
    if (!lh->gexec || lh->g_w != weights || !std::equal(key, key + 3, lh->g_key)) {
        if (lh->gexec) { cudaGraphExecDestroy(lh->gexec); lh->gexec = nullptr; }
        cudaGraph_t g = nullptr;
        cudaStream_t cs = h->cap_st;
        LCK(h, cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal), "begin capture");
        cudaError_t e = cudaSuccess;
        // one block: the exact iteration, then exact_every - 1 proposal iterations
        e = launch_propose(h, lh, w, k, 1, cs);
        if (e == cudaSuccess) e = launch_subset(h, lh, k, 0, 1, cs);
        if (e == cudaSuccess) e = launch_refresh(h, lh, 1, cs);
        if (e == cudaSuccess) { k_learn_miss<<<1, 1, 0, cs>>>(h->dev, lh->L, 1); e = cudaGetLastError(); }
        if (e == cudaSuccess) e = launch_apply_gated(h->dev, h->plan, 1, cs, true);
        for (int i = 1; i < lo->exact_every && e == cudaSuccess; ++i) {
            if (i % lo->propose_every == 0) e = launch_propose(h, lh, w, k, 1, cs);
            if (e == cudaSuccess) e = launch_subset(h, lh, k, 1, 1, cs);
            if (e == cudaSuccess) e = launch_apply_gated(h->dev, h->plan, 1, cs, true);
        }
        cudaError_t e2 = cudaStreamEndCapture(cs, &g);
        if (e != cudaSuccess) { if (g) cudaGraphDestroy(g); LCK(h, e, "capture"); }
        LCK(h, e2, "end capture");
        cudaError_t e3 = cudaGraphInstantiate(&lh->gexec, g, 0);
        cudaGraphDestroy(g);
        if (e3 != cudaSuccess) { lh->gexec = nullptr; LCK(h, e3, "instantiate graph"); }
        std::copy(key, key + 3, lh->g_key);
        lh->g_w = weights;
    }
    const long long max_replays = lo->max_iters / lo->exact_every + 2;
    for (long long r = 0; r < max_replays; ++r) {
        LCK(h, cudaGraphLaunch(lh->gexec, h->st), "graph launch");
        LCK(h, cudaMemcpyAsync(h->h_ctl, h->dev.ctl, sizeof(Ctl), cudaMemcpyDeviceToHost, h->st), "read control");
        LCK(h, cudaStreamSynchronize(h->st), "synchronise");
        if (h->h_ctl->done) break;
    }
    const auto t1 = std::chrono::steady_clock::now();
    LCK(h, cudaMemcpyAsync(lh->h_lc, lh->L.lc, sizeof(LearnCtl), cudaMemcpyDeviceToHost, h->st), "read state");
    LCK(h, cudaStreamSynchronize(h->st), "synchronise");
    const Ctl c = *h->h_ctl;
    res->iters = c.iter - iter0;
    res->moves = c.moves - moves0;
    res->feasible_iter = c.feasible_iter;
    res->final_nviol = c.nviol;
    res->best_nviol = c.best_nviol;
    res->seconds = std::chrono::duration<double>(t1 - t0).count();
    res->time_to_feasible_s = c.feasible_iter >= 0 ? (double)(c.t_feas_ns - c.t_start_ns) * 1e-9 : -1.0;
    res->exact_passes = lh->h_lc->passes;
    res->misses = lh->h_lc->misses;
    return CHAP_OK;
}

chap_status chap_mlp_forward(const uint16_t *weights, const uint16_t *x, int64_t n, float *y, void *stream)
{
    if (!weights || !x || !y || n < 0) return CHAP_E_INVALID;
    if (n == 0) return CHAP_OK;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (mlp_smem_limit((const void *)k_mlp_forward, 0, (int)sizeof(MlpTile)) != cudaSuccess) {
        cudaGetLastError();
        return CHAP_E_CUDA;
    }
    const long long tiles = (n + kTileRows - 1) / kTileRows;
    k_mlp_forward<<<(unsigned)std::min<long long>(tiles, 152 * 4), kTileThreads, sizeof(MlpTile), st>>>(
        reinterpret_cast<const __nv_bfloat16 *>(weights), reinterpret_cast<const __nv_bfloat16 *>(x), n, y);
    return cudaGetLastError() == cudaSuccess ? CHAP_OK : CHAP_E_CUDA;
}

chap_status chap_mlp_loss_grad(const uint16_t *weights, const uint16_t *x, const float *target, int64_t n, float *grad,
                               float *loss, void *stream)
{
    if (!weights || !x || !target || !grad || !loss || n < 1) return CHAP_E_INVALID;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (mlp_smem_limit((const void *)k_mlp_grad, 1, (int)sizeof(MlpGradTile)) != cudaSuccess) {
        cudaGetLastError();
        return CHAP_E_CUDA;
    }
    const long long tiles = (n + kTileRows - 1) / kTileRows;
    k_mlp_grad<<<(unsigned)std::min<long long>(tiles, 152 * 2), kTileThreads, sizeof(MlpGradTile), st>>>(
        reinterpret_cast<const __nv_bfloat16 *>(weights), reinterpret_cast<const __nv_bfloat16 *>(x), target, n,
        2.0f / (float)n, grad, loss);
    return cudaGetLastError() == cudaSuccess ? CHAP_OK : CHAP_E_CUDA;
}

chap_status chap_mlp_adam(float *w32, uint16_t *wbf, float *m, float *v, float *grad, int32_t step, float lr,
                          void *stream)
{
    if (!w32 || !wbf || !m || !v || !grad || step < 1 || !(lr > 0.0f)) return CHAP_E_INVALID;
    const float b1 = 0.9f, b2 = 0.999f;
    const float c1 = 1.0f - std::pow(b1, (float)step), c2 = 1.0f - std::pow(b2, (float)step);
    k_adam<<<(kNParams + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(
        w32, reinterpret_cast<__nv_bfloat16 *>(wbf), m, v, grad, kNParams, lr, b1, b2, 1e-8f, c1, c2);
    return cudaGetLastError() == cudaSuccess ? CHAP_OK : CHAP_E_CUDA;
}

}  // extern "C"
