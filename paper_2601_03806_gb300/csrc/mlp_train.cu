// mlp_train.cu -- training of the learned-collision network on the GPU: the
// loss gradient and Adam (the training pairs are made in aux.cu).
//
// Gradient of L = mean over samples and outputs of (y - t)^2, FP32 on the
// CUDA cores.  A CTA takes tiles of T samples (8, 16 or 32) whose features,
// targets and activations live in shared memory beside the weights (rows
// padded to conflict-free strides).  A thread computes one output of a layer
// for 4 or 8 samples, so a weight fetched once (four inputs per 128-bit load)
// serves all of them: the shared-memory pipe bounds these phases, and 128
// threads of 4 samples read 40 % less of it than 256 of 2.
//
// One gradient (k_mlp_grad): the weight gradients are register blocks (4 x 4
// of W2, 2 x 4 of W1, 4 x 2 of W3) summed over the tile's samples and added
// to the CTA's totals per tile; sums over CTAs are FP64 in CTA order.
//
// Training (k_mlp_train): an epoch's mini-batches in one cooperative launch.
// A mini-batch of 1024 samples is bound by latency, not by work, so it is
// spread over as many SMs as it has tiles -- T is the smallest with one tile
// per SM -- and an iteration is two phases with a grid barrier after each:
//   A  forward and backward of the CTA's tile; activations and dL/dz go to
//      L2, feature by feature (312 rows of the batch's samples);
//   B  a CTA owns about 64 parameters (an 8 x 8 block of W2, 8 x 7 of W1, 7 x
//      8 of W3, and the biases of its rows): it reads the 16 rows they need,
//      sums each parameter over 128 samples in order (a warp per 128
//      samples), adds those sums in FP64 and applies Adam.
// Parameters are summed where they are updated, so no partial gradients
// cross the chip.  On batches of 1024 (262,144 samples, 7771 parameters) an
// iteration takes 11 us; one CTA per 128 samples doing all of it, with two
// more kernels for the sums and Adam, took 130 us (8 of 152 SMs busy).
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <numeric>
#include <random>
#include <string>
#include <type_traits>
#include <vector>

#include "../../include/flbm.h"
#include "internal.h"
#include "lattice.cuh"
#include "step_kernel.cuh"

namespace flbm {

namespace {

constexpr int kNin = 28, kNh = 64, kNout = 27, kNp = 7771;
constexpr int kOffW1 = 0, kOffB1 = 1792, kOffW2 = 1856, kOffB2 = 5952, kOffW3 = 6016, kOffB3 = 7744;
constexpr int kNpPad = 7776;       // row length of the per-CTA partial gradients
constexpr int kGradThreads = 256;
constexpr int kSw = 68;            // padded row stride of W2 and W3 in shared memory
// The network as the kernels hold it, in shared memory and (training) in
// global memory: W1 [64][28], W2 [64][68], W3 [28][68] (row 27 zero), b1, b2,
// b3 [32]; the pads keep 128-bit row reads free of bank conflicts.
constexpr int kImgW2 = kNh * kNin, kImgW3 = kImgW2 + kNh * kSw, kImgB1 = kImgW3 + 28 * kSw, kImgB2 = kImgB1 + kNh,
              kImgB3 = kImgB2 + kNh, kImg = kImgB3 + 32;
__host__ __device__ constexpr int image_index(int p)
{
    return p < kOffB1   ? p
           : p < kOffW2 ? kImgB1 + p - kOffB1
           : p < kOffB2 ? kImgW2 + (p - kOffW2) / kNh * kSw + (p - kOffW2) % kNh
           : p < kOffW3 ? kImgB2 + p - kOffB2
           : p < kOffB3 ? kImgW3 + (p - kOffW3) / kNh * kSw + (p - kOffW3) % kNh
                        : kImgB3 + p - kOffB3;
}
constexpr int kFlushTiles = 64;    // tiles summed in FP32 before they enter the FP64 partials

// Threads that compute the layers of a tile of T samples (all of the CTA's
// 256 at T = 32), and the samples a thread then takes: kN4 where a thread
// owns one of 64 outputs, kN8 where a lane owns one of 28 or two of 64.
template <int T>
struct TileShape {
    static constexpr int kThreads = T == 32 ? 256 : 128;
    static constexpr int kN4 = T * 64 / kThreads, kN8 = T * 32 / kThreads;
};

// Shared memory of a CTA with tiles of T samples (every array a multiple of
// 16 bytes, so rows take 128-bit loads).
template <int T>
struct GradSmem {
    float img[kImg];               // the network, image_index order
    float x[2][T * kNin];          // this tile's and the next one's features
    float t[2][T * 28];            // and targets (27 used)
    float h1[T * kNh], h2[T * kNh];
    float s1[T * kNh];             // silu'(z1), then dL/dz1
    float s2[T * kNh];             // silu'(z2), then dL/dz2
    float dy[T * 28];              // column 27 zero
    uint64_t idx[2][T];            // sample rows of the next tiles
};

// Training, phase B: 16 rows of kChunk samples and the sums per 128 samples.
constexpr int kRun = 128;                  // samples a parameter's FP32 sum spans
constexpr int kChunk = 8 * kRun;           // a run per warp
constexpr int kRowPad = kChunk + 4;        // 8 rows' 128-bit loads in distinct banks
constexpr int kMaxRuns = 152;              // batches of up to 19,456 samples
constexpr int kActRows = kNin + 4 * kNh + 28;   // X, H1, Z1, H2, Z2, DY (312)
constexpr int kRowH1 = kNin, kRowZ1 = kRowH1 + kNh, kRowH2 = kRowZ1 + kNh, kRowZ2 = kRowH2 + kNh,
              kRowDY = kRowZ2 + kNh;
constexpr int kBlocks = 128;               // parameter blocks: 64 of W2, 32 of W1, 32 of W3
template <int T>
struct TrainSmem {
    GradSmem<T> g;
    float d[8][kRowPad], in[8][kRowPad];
    float sum[kMaxRuns][72];               // 8 x 8 parameters, then 8 biases
};

__device__ __forceinline__ float sigm(float z) { return 1.0f / (1.0f + expf(-z)); }

// Sample s of the epoch order: (mult s + off) mod n, a bijection of [0, n)
// for mult coprime to n (mult = 1, off = 0: the identity).  s < n < 2^32 and
// mult < n keep the product below 2^64.
__device__ __forceinline__ uint64_t sample_index(uint64_t s, uint64_t mult, uint64_t off, uint64_t n)
{
    return (mult * s + off) % n;
}

// The samples of the batches a kernel goes through: batch b of the epoch
// order holds samples b batch .. , `count` of them (the last one fewer).
struct Samples {
    const float *X, *T;
    uint64_t n, batch, mult, off;
    __device__ __forceinline__ uint64_t count(uint64_t b) const
    {
        const uint64_t rest = n - b * batch;
        return rest < batch ? rest : batch;
    }
};

// A CTA's tiles: tile blockIdx.x, blockIdx.x + gridDim.x, ... of batch b0,
// then those of batch b0 + 1, up to batch b1.
template <int T>
struct TileWalk {
    uint64_t b, b1, tile;
    __device__ __forceinline__ TileWalk(const Samples &s, uint64_t first, uint64_t last)
        : b(first), b1(last), tile(blockIdx.x)
    {
        settle(s);
    }
    __device__ __forceinline__ bool done() const { return b >= b1; }
    __device__ __forceinline__ void settle(const Samples &s)
    {
        while (b < b1 && tile * T >= s.count(b)) {
            ++b;
            tile = blockIdx.x;
        }
    }
    __device__ __forceinline__ void next(const Samples &s)
    {
        tile += gridDim.x;
        settle(s);
    }
    __device__ __forceinline__ uint64_t live(const Samples &s) const
    {
        const uint64_t left = s.count(b) - tile * T;
        return left < T ? left : T;
    }
};

// Threads kGradThreads - T ..: the sample rows of the tile at w into idx.
template <int T>
__device__ __forceinline__ void tile_rows(uint64_t (&idx)[T], const Samples &s, const TileWalk<T> &w)
{
    const int j = int(threadIdx.x) - (kGradThreads - T);
    if (j >= 0 && !w.done() && uint64_t(j) < w.live(s))
        idx[j] = sample_index(w.b * s.batch + w.tile * T + uint64_t(j), s.mult, s.off, s.n);
}

// Start the copies of a tile's features and targets (4 bytes each: rows of
// 112 and 108 bytes in arrays the caller aligns to 4); rows past the batch
// get zero features.
template <int T>
__device__ __forceinline__ void fetch_tile(float (&x)[T * kNin], float (&t)[T * 28], const uint64_t (&idx)[T],
                                           const Samples &s, const TileWalk<T> &w)
{
    if (!w.done()) {
        const uint32_t live = uint32_t(w.live(s));
        for (uint32_t e = threadIdx.x; e < uint32_t(T * kNin); e += kGradThreads) {
            const uint32_t j = e / kNin, k = e % kNin;
            if (j < live) {
                cp_async4(&x[e], s.X + idx[j] * kNin + k);
                if (k < uint32_t(kNout)) cp_async4(&t[e], s.T + idx[j] * kNout + k);
            } else {
                x[e] = 0.0f;
            }
        }
    }
    cp_async_commit();
}

// Start the copy of the network image into shared memory (from L2: in
// k_mlp_train other SMs have just written it).
template <int T>
__device__ __forceinline__ void fetch_image(GradSmem<T> &sm, const float *img)
{
    static_assert(kImg % 4 == 0, "16-byte copies");
    for (int i = threadIdx.x; i < kImg / 4; i += kGradThreads)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(sm.img + 4 * i)), "l"(img + 4 * i)
                     : "memory");
    cp_async_commit();
}

// z_i = b + W row . input row of sample i, K inputs (a multiple of 4), one
// FMA per input in order.
template <int K, int NS>
__device__ __forceinline__ void dense(const float *w, float b, const float *in, int stride, float (&z)[NS])
{
#pragma unroll
    for (int i = 0; i < NS; ++i) z[i] = b;
#pragma unroll
    for (int k = 0; k < K; k += 4) {
        const float4 wv = *reinterpret_cast<const float4 *>(w + k);
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            const float4 v = *reinterpret_cast<const float4 *>(in + i * stride + k);
            z[i] = fmaf(wv.x, v.x, z[i]);
            z[i] = fmaf(wv.y, v.y, z[i]);
            z[i] = fmaf(wv.z, v.z, z[i]);
            z[i] = fmaf(wv.w, v.w, z[i]);
        }
    }
}

// g_i = (columns k, k + 1 of W)^T . d row of sample i, O outputs in order.
template <int O, int NS>
__device__ __forceinline__ void dense_t(const float *w, const float *d, int stride, float2 (&g)[NS])
{
#pragma unroll
    for (int i = 0; i < NS; ++i) g[i] = make_float2(0.0f, 0.0f);
#pragma unroll
    for (int o = 0; o < O; o += 4) {
        float2 wv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) wv[q] = *reinterpret_cast<const float2 *>(w + (o + q) * kSw);
#pragma unroll
        for (int i = 0; i < NS; ++i) {
            const float4 v = *reinterpret_cast<const float4 *>(d + i * stride + o);
            const float dv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                g[i].x = fmaf(dv[q], wv[q].x, g[i].x);
                g[i].y = fmaf(dv[q], wv[q].y, g[i].y);
            }
        }
    }
}

// A thread's share of the gradient: W2 rows 4 (t / 16) .. + 3, columns 4 (t %
// 16) .. + 3; warps 0-6: W1 rows 2 lane, 2 lane + 1, columns 4 warp .. + 3,
// and W3 rows 4 warp .. + 3, columns 2 lane, 2 lane + 1; warp 7: in w1, the
// biases b1[lane], b1[lane + 32], b2[lane], b2[lane + 32], b3[lane].
struct GradAcc {
    float w2[4][4], w1[2][4], w3[4][2];
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
#pragma unroll
            for (int c = 0; c < 4; ++c) w2[a][c] = 0.0f;
#pragma unroll
            for (int c = 0; c < 2; ++c) w1[c][a] = w3[a][c] = 0.0f;
        }
    }
    __device__ __forceinline__ void add(const GradAcc &o)
    {
#pragma unroll
        for (int a = 0; a < 4; ++a) {
#pragma unroll
            for (int c = 0; c < 4; ++c) w2[a][c] += o.w2[a][c];
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                w1[c][a] += o.w1[c][a];
                w3[a][c] += o.w3[a][c];
            }
        }
    }
    // f(parameter index, value) for every parameter of this thread
    template <typename F>
    __device__ __forceinline__ void each(F &&f) const
    {
        const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c) f(kOffW2 + (4 * (t >> 4) + a) * kNh + 4 * (t & 15) + c, w2[a][c]);
        if (warp < 7) {
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int c = 0; c < 4; ++c) f(kOffW1 + (2 * lane + a) * kNin + 4 * warp + c, w1[a][c]);
#pragma unroll
            for (int a = 0; a < 4; ++a)
                if (4 * warp + a < kNout)
#pragma unroll
                    for (int c = 0; c < 2; ++c) f(kOffW3 + (4 * warp + a) * kNh + 2 * lane + c, w3[a][c]);
        } else {
            f(kOffB1 + lane, w1[0][0]);
            f(kOffB1 + 32 + lane, w1[0][1]);
            f(kOffB2 + lane, w1[0][2]);
            f(kOffB2 + 32 + lane, w1[0][3]);
            if (lane < kNout) f(kOffB3 + lane, w1[1][0]);
        }
    }
};

// Forward, loss and backward of the tile in x, t (live samples; the others
// get zero activations and derivatives).  The caller's barrier makes the
// results visible.
template <int T>
__device__ __forceinline__ void forward_backward(GradSmem<T> &sm, const float *x, const float *t, int live,
                                                 float inv_norm, double &loss)
{
    using Shape = TileShape<T>;
    constexpr int N4 = Shape::kN4, N8 = Shape::kN8;
    const int tid = threadIdx.x, lane = tid & 31;
    const int o = tid & 63, s4 = (tid >> 6) * N4, s8 = (tid >> 5) * N8;
    const bool on = tid < Shape::kThreads;
    // hidden layer: silu(z) and silu'(z) of output o
    auto hidden = [&](auto K, const float *w, float b, const float *in, int stride, float *h, float *s) {
        float z[N4];
        dense<decltype(K)::value, N4>(w, b, in + s4 * stride, stride, z);
#pragma unroll
        for (int i = 0; i < N4; ++i) {
            const bool ok = s4 + i < live;
            const float g = sigm(z[i]);
            h[(s4 + i) * kNh + o] = ok ? z[i] * g : 0.0f;
            s[(s4 + i) * kNh + o] = ok ? g * (1.0f + z[i] * (1.0f - g)) : 0.0f;
        }
    };
    if (on) hidden(std::integral_constant<int, kNin>{}, sm.img + o * kNin, sm.img[kImgB1 + o], x, kNin, sm.h1, sm.s1);
    __syncthreads();
    if (on)
        hidden(std::integral_constant<int, kNh>{}, sm.img + kImgW2 + o * kSw, sm.img[kImgB2 + o], sm.h1, kNh, sm.h2,
               sm.s2);
    __syncthreads();
    if (!on) return;
    if (lane < 28) {
        float y[N8];
        dense<kNh, N8>(sm.img + kImgW3 + lane * kSw, sm.img[kImgB3 + lane], sm.h2 + s8 * kNh, kNh, y);
#pragma unroll
        for (int i = 0; i < N8; ++i) {
            const float d = (s8 + i < live && lane < kNout) ? y[i] - t[(s8 + i) * 28 + lane] : 0.0f;
            loss += double(d) * double(d);
            sm.dy[(s8 + i) * 28 + lane] = 2.0f * d * inv_norm;
        }
    }
    __syncwarp();   // backwards a warp keeps its samples
    float2 v[N8];
    auto scale = [&](float *s) {
#pragma unroll
        for (int i = 0; i < N8; ++i) {
            float2 *p = reinterpret_cast<float2 *>(s + (s8 + i) * kNh + 2 * lane);
            *p = make_float2(p->x * v[i].x, p->y * v[i].y);
        }
    };
    dense_t<28, N8>(sm.img + kImgW3 + 2 * lane, sm.dy + s8 * 28, 28, v);
    scale(sm.s2);
    __syncwarp();
    dense_t<kNh, N8>(sm.img + kImgW2 + 2 * lane, sm.s2 + s8 * kNh, kNh, v);
    scale(sm.s1);
}

// The gradient sums of the tile in sm (features in x).
template <int T>
__device__ __forceinline__ void weight_grads(const GradSmem<T> &sm, const float *x, GradAcc &g)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    g.zero();
    const int o4 = 4 * (tid >> 4), k4 = 4 * (tid & 15);
#pragma unroll 4
    for (int s = 0; s < T; ++s) {
        const float4 dv = *reinterpret_cast<const float4 *>(sm.s2 + s * kNh + o4);
        const float4 hv = *reinterpret_cast<const float4 *>(sm.h1 + s * kNh + k4);
        const float d[4] = {dv.x, dv.y, dv.z, dv.w}, h[4] = {hv.x, hv.y, hv.z, hv.w};
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int c = 0; c < 4; ++c) g.w2[a][c] = fmaf(d[a], h[c], g.w2[a][c]);
    }
    if (warp < 7) {
#pragma unroll 4
        for (int s = 0; s < T; ++s) {
            const float2 dv = *reinterpret_cast<const float2 *>(sm.s1 + s * kNh + 2 * lane);
            const float4 xv = *reinterpret_cast<const float4 *>(x + s * kNin + 4 * warp);
            const float4 ev = *reinterpret_cast<const float4 *>(sm.dy + s * 28 + 4 * warp);
            const float2 hv = *reinterpret_cast<const float2 *>(sm.h2 + s * kNh + 2 * lane);
            const float xs[4] = {xv.x, xv.y, xv.z, xv.w}, es[4] = {ev.x, ev.y, ev.z, ev.w};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                g.w1[0][c] = fmaf(dv.x, xs[c], g.w1[0][c]);
                g.w1[1][c] = fmaf(dv.y, xs[c], g.w1[1][c]);
                g.w3[c][0] = fmaf(es[c], hv.x, g.w3[c][0]);
                g.w3[c][1] = fmaf(es[c], hv.y, g.w3[c][1]);
            }
        }
    } else {
#pragma unroll 4
        for (int s = 0; s < T; ++s) {
            g.w1[0][0] += sm.s1[s * kNh + lane];
            g.w1[0][1] += sm.s1[s * kNh + 32 + lane];
            g.w1[0][2] += sm.s2[s * kNh + lane];
            g.w1[0][3] += sm.s2[s * kNh + 32 + lane];
            if (lane < kNout) g.w1[1][0] += sm.dy[s * 28 + lane];
        }
    }
}

// Gradient and loss sums of batch b into partials[cta][kNpPad] (FP64) and
// lpart[cta][8] (per warp).  Tiles add up in FP32 kFlushTiles at a time.
template <int T>
__global__ void __launch_bounds__(kGradThreads, 2) k_mlp_grad(const float *__restrict__ img, const Samples s,
                                                              uint64_t b, float inv_norm,
                                                              double *__restrict__ partials,
                                                              double *__restrict__ lpart)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    GradSmem<T> &sm = *reinterpret_cast<GradSmem<T> *>(smraw);
    TileWalk<T> cur(s, b, b + 1), nxt(cur);
    nxt.next(s);
    tile_rows<T>(sm.idx[0], s, cur);
    tile_rows<T>(sm.idx[1], s, nxt);
    fetch_image(sm, img);
    __syncthreads();
    fetch_tile<T>(sm.x[0], sm.t[0], sm.idx[0], s, cur);
    double *out = partials + size_t(blockIdx.x) * kNpPad;
    GradAcc acc, g;
    acc.zero();
    double loss = 0.0;
    uint32_t q = 0;
    bool first = true;
    for (; !cur.done(); ++q) {
        cp_async_wait_all();
        __syncthreads();
        fetch_tile<T>(sm.x[(q + 1) & 1], sm.t[(q + 1) & 1], sm.idx[(q + 1) & 1], s, nxt);
        TileWalk<T> after(nxt);
        if (!after.done()) after.next(s);
        forward_backward<T>(sm, sm.x[q & 1], sm.t[q & 1], int(cur.live(s)), inv_norm, loss);
        __syncthreads();
        tile_rows<T>(sm.idx[q & 1], s, after);
        weight_grads<T>(sm, sm.x[q & 1], g);
        acc.add(g);
        if (nxt.done() || q % kFlushTiles == kFlushTiles - 1) {
            acc.each([&](int p, float v) { out[p] = first ? double(v) : out[p] + double(v); });
            first = false;
            acc.zero();
        }
        cur = nxt;
        nxt = after;
    }
    loss = warp_sum(loss);
    if ((threadIdx.x & 31) == 0) lpart[blockIdx.x * 8 + (threadIdx.x >> 5)] = loss;
}

// A grid barrier in two halves.  The counter only grows: the k-th barrier of
// a launch waits for k gridDim.x arrivals beyond `base`.  The wait is bounded
// (about 2^22 polls, seconds) and reports failure to the whole CTA.
__device__ __forceinline__ void grid_arrive(unsigned int *bar)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(bar, 1u);
    }
}
__device__ __forceinline__ bool grid_wait(unsigned int *bar, unsigned int target, unsigned int *flag)
{
    int late = 0;
    if (threadIdx.x == 0) {
        late = 1;
        for (uint32_t it = 0; it < (1u << 22); ++it) {
            unsigned int v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(bar) : "memory");
            if (int(v - target) >= 0) {
                late = 0;
                break;
            }
            if (it > 64) __nanosleep(64);
        }
        if (late) atomicOr(flag, 2u);
        __threadfence();
    }
    return __syncthreads_or(late) == 0;
}

struct TrainArgs {
    Samples s;
    uint64_t b0, b1;               // the batches of this launch
    float inv_full, inv_last;      // 1 / (samples x outputs) of a full batch and of the epoch's last
    float beta1, beta2, eps;
    float *img, *m1, *m2;          // network image; moments in parameter order
    const float *lr;               // step size of batch b at lr[b - b0]
    float *act;                    // [kActRows + 1][stride]: phase A's results
    uint32_t stride;               // samples of a full batch, rounded up to 128
    double *lpart;                 // [gridDim.x][8]: loss sums of the warps
    double *loss;                  // loss sum of batch b at loss[b]
    unsigned int *bar;             // 0 at launch
    unsigned int *flag;            // bit 1: a bounded wait ran out
};

// The tile's activations and derivatives into rows of act from sample s0 (a
// multiple of T): four samples of a row per 16-byte store.
template <int T>
__device__ __forceinline__ void store_rows(const GradSmem<T> &sm, const float *x, float *act, uint32_t stride,
                                           uint32_t s0)
{
    for (int e = threadIdx.x; e < kActRows * (T / 4); e += kGradThreads) {
        const int row = e % kActRows, q = 4 * (e / kActRows);
        const float *src;
        int st = kNh;
        if (row < kRowH1) { src = x + row; st = kNin; }
        else if (row < kRowZ1) src = sm.h1 + row - kRowH1;
        else if (row < kRowH2) src = sm.s1 + row - kRowZ1;
        else if (row < kRowZ2) src = sm.h2 + row - kRowH2;
        else if (row < kRowDY) src = sm.s2 + row - kRowZ2;
        else { src = sm.dy + row - kRowDY; st = 28; }
        __stcg(reinterpret_cast<float4 *>(act + size_t(row) * stride + s0 + q),
               make_float4(src[q * st], src[(q + 1) * st], src[(q + 2) * st], src[(q + 3) * st]));
    }
}

// Parameter block blk: rows d0 .. d0 + 7 (dL/dz) and in0 .. in0 + 7 (inputs)
// of act, and the parameter index of (row a, column c), c = 8 for a's bias
// (-1: none).
struct Block {
    int d0, in0, blk;
    __device__ __forceinline__ explicit Block(int b) : blk(b)
    {
        if (b < 64) {
            d0 = kRowZ2 + 8 * (b >> 3);
            in0 = kRowH1 + 8 * (b & 7);
        } else if (b < 96) {
            d0 = kRowZ1 + 8 * ((b - 64) >> 2);
            in0 = 7 * (b & 3);
        } else {
            d0 = kRowDY + 7 * ((b - 96) >> 3);
            in0 = kRowH2 + 8 * (b & 7);
        }
    }
    __device__ __forceinline__ int param(int a, int c) const
    {
        if (blk < 64) {
            const int o = d0 - kRowZ2 + a;
            return c < 8 ? kOffW2 + o * kNh + in0 - kRowH1 + c : ((blk & 7) ? -1 : kOffB2 + o);
        }
        if (blk < 96) {
            const int o = d0 - kRowZ1 + a;
            return c < 7 ? kOffW1 + o * kNin + in0 + c : (c == 7 || (blk & 3)) ? -1 : kOffB1 + o;
        }
        const int o = d0 - kRowDY + a;
        if (a == 7 || o >= kNout) return -1;
        return c < 8 ? kOffW3 + o * kNh + in0 - kRowH2 + c : ((blk & 7) ? -1 : kOffB3 + o);
    }
};

// Adam (Kingma & Ba 2015) over the batches b0 .. b1 - 1: one cooperative
// launch, one CTA per SM at most; a batch has at most kMaxRuns runs.
template <int T>
__global__ void __launch_bounds__(kGradThreads, 1) k_mlp_train(const __grid_constant__ TrainArgs a)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    TrainSmem<T> &ts = *reinterpret_cast<TrainSmem<T> *>(smraw);
    GradSmem<T> &sm = ts.g;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    TileWalk<T> cur(a.s, a.b0, a.b1), nxt(cur);
    if (!nxt.done()) nxt.next(a.s);
    tile_rows<T>(sm.idx[0], a.s, cur);
    tile_rows<T>(sm.idx[1], a.s, nxt);
    __syncthreads();
    fetch_tile<T>(sm.x[0], sm.t[0], sm.idx[0], a.s, cur);
    uint32_t q = 0;
    unsigned int target = 0;
    for (uint64_t b = a.b0; b < a.b1; ++b) {
        // ---- phase A
        const uint32_t count = uint32_t(a.s.count(b)), ntiles = (count + T - 1) / T;
        const uint32_t active = min(ntiles, gridDim.x);   // CTAs with a tile
        const float inv_norm = count == a.s.batch ? a.inv_full : a.inv_last;
        if (blockIdx.x < active) fetch_image(sm, a.img);
        double loss = 0.0;
        for (; !cur.done() && cur.b == b; ++q) {
            cp_async_wait_all();
            __syncthreads();
            fetch_tile<T>(sm.x[(q + 1) & 1], sm.t[(q + 1) & 1], sm.idx[(q + 1) & 1], a.s, nxt);
            TileWalk<T> after(nxt);
            if (!after.done()) after.next(a.s);
            forward_backward<T>(sm, sm.x[q & 1], sm.t[q & 1], int(cur.live(a.s)), inv_norm, loss);
            __syncthreads();
            store_rows<T>(sm, sm.x[q & 1], a.act, a.stride, uint32_t(cur.tile) * T);
            tile_rows<T>(sm.idx[q & 1], a.s, after);
            cur = nxt;
            nxt = after;
        }
        if (blockIdx.x < active) {
            loss = warp_sum(loss);
            if (lane == 0) __stcg(a.lpart + blockIdx.x * 8 + warp, loss);
        }
        target += gridDim.x;
        grid_arrive(a.bar);
        if (!grid_wait(a.bar, target, a.flag)) break;
        // ---- phase B
        const uint32_t runs = (count + kRun - 1) / kRun;
        const float lr = a.lr[b - a.b0];
        if (blockIdx.x == gridDim.x - 1 && warp == 7) {   // a CTA without a block, where there are 129
            double sum = 0.0;
            for (uint32_t c = uint32_t(lane); c < 8 * active; c += 32) sum += __ldcg(a.lpart + c);
            sum = warp_sum(sum);
            if (lane == 0) a.loss[b] = sum;
        }
        for (int blk = int(blockIdx.x); blk < kBlocks; blk += int(gridDim.x)) {
            const Block B(blk);
            // thread t < 72 updates parameter (t / 8, t % 8), or bias t - 64
            const int p = tid < 64 ? B.param(tid >> 3, tid & 7) : (tid < 72 ? B.param(tid - 64, 8) : -1);
            float m = 0.0f, v = 0.0f, th = 0.0f;
            if (p >= 0) {
                m = __ldcg(a.m1 + p);
                v = __ldcg(a.m2 + p);
                th = __ldcg(a.img + image_index(p));
            }
            for (uint32_t r0 = 0; r0 < runs; r0 += kChunk / kRun) {
                const uint32_t s0 = r0 * kRun;
                // samples of the chunk: whole groups of four (phase A wrote
                // zeros up to the end of the last tile)
                const uint32_t len = min(uint32_t(kChunk), (count - s0 + 3) / 4 * 4);
                if (r0) __syncthreads();   // the previous chunk's rows are done with
                for (uint32_t e = tid; e < 16 * (kChunk / 4); e += kGradThreads) {
                    const uint32_t row = e / (kChunk / 4), k = 4 * (e % (kChunk / 4));
                    if (k < len)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(
                                         smem_u32(row < 8 ? &ts.d[row][k] : &ts.in[row - 8][k])),
                                     "l"(a.act + size_t(row < 8 ? B.d0 + row : B.in0 + row - 8) * a.stride + s0 + k)
                                     : "memory");
                }
                cp_async_commit();
                cp_async_wait_all();
                __syncthreads();
                const uint32_t run = r0 + uint32_t(warp), k0 = uint32_t(warp) * kRun;
                if (run < runs) {
                    // lane: row a = lane / 4, columns c, c + 1 with c = 2 (lane % 4)
                    const float *dr = ts.d[lane >> 2], *i0 = ts.in[2 * (lane & 3)], *i1 = ts.in[2 * (lane & 3) + 1];
                    const uint32_t k1 = min(k0 + kRun, len);
                    float g0 = 0.0f, g1 = 0.0f, gb = 0.0f;
#pragma unroll 4
                    for (uint32_t k = k0; k < k1; k += 4) {
                        const float4 d = *reinterpret_cast<const float4 *>(dr + k);
                        const float4 u = *reinterpret_cast<const float4 *>(i0 + k);
                        const float4 w = *reinterpret_cast<const float4 *>(i1 + k);
                        g0 = fmaf(d.w, u.w, fmaf(d.z, u.z, fmaf(d.y, u.y, fmaf(d.x, u.x, g0))));
                        g1 = fmaf(d.w, w.w, fmaf(d.z, w.z, fmaf(d.y, w.y, fmaf(d.x, w.x, g1))));
                        gb = (((gb + d.x) + d.y) + d.z) + d.w;
                    }
                    *reinterpret_cast<float2 *>(&ts.sum[run][2 * lane]) = make_float2(g0, g1);
                    if ((lane & 3) == 0) ts.sum[run][64 + (lane >> 2)] = gb;
                }
            }
            __syncthreads();
            if (p >= 0) {
                double sum = 0.0;
#pragma unroll 8
                for (uint32_t r = 0; r < runs; ++r) sum += double(ts.sum[r][tid]);
                const float gr = float(sum);
                m = a.beta1 * m + (1.0f - a.beta1) * gr;
                v = a.beta2 * v + (1.0f - a.beta2) * gr * gr;
                __stcg(a.m1 + p, m);
                __stcg(a.m2 + p, v);
                __stcg(a.img + image_index(p), th - lr * m / (sqrtf(v) + a.eps));
            }
        }
        target += gridDim.x;
        grid_arrive(a.bar);
        if (!grid_wait(a.bar, target, a.flag)) break;
    }
    cp_async_wait_all();   // no copy may land after the CTA has left
}

// grad[p] = sum over CTAs of partials[cta][p]; grad[kNp]: the loss sum
__global__ void k_mlp_reduce(const double *__restrict__ partials, const double *__restrict__ lpart, int nblocks,
                             double *__restrict__ grad)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p > kNp) return;
    double s = 0.0;
    if (p < kNp)
        for (int b = 0; b < nblocks; ++b) s += partials[size_t(b) * kNpPad + p];
    else
        for (int b = 0; b < 8 * nblocks; ++b) s += lpart[b];
    grad[p] = s;
}

// Adam (Kingma & Ba 2015) with bias-corrected step size lr_t.
__global__ void k_mlp_adam(float *__restrict__ img, float *__restrict__ m1, float *__restrict__ m2,
                           const double *__restrict__ grad, float lr_t, float beta1, float beta2, float eps)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= kNp) return;
    const float g = float(grad[p]);
    const float a = beta1 * m1[p] + (1.0f - beta1) * g;
    const float b = beta2 * m2[p] + (1.0f - beta2) * g * g;
    m1[p] = a;
    m2[p] = b;
    img[image_index(p)] -= lr_t * a / (sqrtf(b) + eps);
}

// Samples per tile for batches of `count`: the smallest tile with at most
// one per SM (a tile of 8 takes less than half the time of one of 32, so
// spreading a small batch over more SMs wins), else 32 (twice the reuse of
// each weight fetched from shared memory of T = 8).
int tile_for(uint64_t count, int nsm)
{
    if (count <= uint64_t(8) * nsm) return 8;
    if (count <= uint64_t(16) * nsm) return 16;
    return 32;
}

// f(std::integral_constant<int, T>) for the tile size T.
template <typename F>
auto with_tile(int T, F &&f)
{
    if (T == 8) return f(std::integral_constant<int, 8>{});
    if (T == 16) return f(std::integral_constant<int, 16>{});
    return f(std::integral_constant<int, 32>{});
}

constexpr uint64_t kTrainChunk = 1024;   // mini-batches of one training launch at most

// A call's device workspace: one allocation, cut up by take(), and the partial
// gradients of a training call whose cooperative launch was refused.
struct Scratch {
    unsigned char *base = nullptr;
    double *partials = nullptr;
    size_t used = 0;
    cudaStream_t s = nullptr;
    template <typename P>
    void take(P *&p, size_t count)
    {
        p = reinterpret_cast<P *>(base + used);
        used += (count * sizeof(P) + 255) / 256 * 256;
    }
    ~Scratch()
    {
        if (s) cudaStreamSynchronize(s);
        cudaFree(base);
        cudaFree(partials);
        if (s) cudaStreamDestroy(s);
    }
};

int fail(const std::string &m, int code)
{
    set_thread_error(m.c_str());
    return code;
}

// Whether p is device (or managed) memory; a host pointer handed to a
// kernel would fault instead of failing.
bool is_device_memory(const void *p)
{
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// The workspace of a gradient or training call on batches of B samples,
// nb of them in an epoch.
struct Work {
    std::vector<float> host;       // the network image on its way in and out
    int nsm = 0;
    int T = 32, grid = 1;          // tile size and CTAs
    uint32_t stride = 0;           // samples of a row of act
    bool epochs_in_one = false;    // training: k_mlp_train serves the batch
    float *img = nullptr, *m1 = nullptr, *m2 = nullptr, *lr = nullptr, *act = nullptr;
    double *partials = nullptr, *grad = nullptr, *lpart = nullptr, *loss = nullptr;
    unsigned int *bar = nullptr;   // [0] barrier arrivals, [1] flag
};

int prepare(Scratch &sc, Work &w, const float *params, uint64_t B, uint64_t nb, bool train)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&w.nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&sc.s, cudaStreamNonBlocking);
    w.T = tile_for(B, w.nsm);
    const uint64_t tiles = (B + w.T - 1) / w.T;
    // larger batches (thousands of tiles) gain nothing from one launch
    w.epochs_in_one = train && B <= uint64_t(kRun) * std::min(w.nsm, kMaxRuns);
    // the training kernel: one CTA on every SM (tiles of phase A, blocks of
    // phase B and, on the last, the loss sums); the gradient kernel: two
    w.grid = w.epochs_in_one ? w.nsm : int(std::min<uint64_t>(tiles, uint64_t(2) * w.nsm));
    w.stride = uint32_t((B + kRun - 1) / kRun * kRun);
    if (e == cudaSuccess)
        e = with_tile(w.T, [&](auto tag) {
            constexpr int T = decltype(tag)::value;
            const cudaError_t r = cudaFuncSetAttribute(k_mlp_grad<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       int(sizeof(GradSmem<T>)));
            return r != cudaSuccess ? r
                                    : cudaFuncSetAttribute(k_mlp_train<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                           int(sizeof(TrainSmem<T>)));
        });
    if (e != cudaSuccess) return fail(std::string("mlp: device set-up: ") + cudaGetErrorString(e), FLBM_E_CUDA);
    const auto lay_out = [&] {
        sc.used = 0;
        sc.take(w.img, kImg);
        sc.take(w.lpart, size_t(w.grid) * 8);
        sc.take(w.grad, kNp + 1);
        if (train) {
            sc.take(w.m1, kNpPad);
            sc.take(w.m2, kNpPad);
            sc.take(w.loss, nb);
        }
        if (w.epochs_in_one) {
            sc.take(w.lr, kTrainChunk);
            sc.take(w.bar, 2);
            sc.take(w.act, size_t(kActRows + 1) * w.stride);
        } else {
            sc.take(w.partials, size_t(w.grid) * kNpPad);
        }
    };
    lay_out();
    e = cudaMalloc(&sc.base, sc.used);
    if (e != cudaSuccess) return fail(std::string("mlp: cudaMalloc: ") + cudaGetErrorString(e), FLBM_E_NOMEM);
    lay_out();
    w.host.assign(kImg, 0.0f);
    for (int p = 0; p < kNp; ++p) w.host[size_t(image_index(p))] = params[p];
    e = cudaMemcpyAsync(w.img, w.host.data(), kImg * sizeof(float), cudaMemcpyHostToDevice, sc.s);
    if (e == cudaSuccess && train) e = cudaMemsetAsync(w.m1, 0, kNpPad * sizeof(float), sc.s);
    if (e == cudaSuccess && train) e = cudaMemsetAsync(w.m2, 0, kNpPad * sizeof(float), sc.s);
    if (e == cudaSuccess && w.epochs_in_one) e = cudaMemsetAsync(w.bar, 0, 2 * sizeof(unsigned int), sc.s);
    if (e != cudaSuccess) return fail(std::string("mlp: upload: ") + cudaGetErrorString(e), FLBM_E_CUDA);
    return FLBM_OK;
}

// Training continues without k_mlp_train: a gradient, its sums and Adam per
// mini-batch, as for larger batches (three launches, slower, the same
// accuracy: a partial sum spans a tile or two of samples).
int without_cooperation(Scratch &sc, Work &w, uint64_t B)
{
    cudaGetLastError();   // clear the refusal
    w.epochs_in_one = false;
    w.grid = int(std::min<uint64_t>((B + w.T - 1) / w.T, uint64_t(2) * w.nsm));
    const size_t bytes = (size_t(w.grid) * kNpPad + size_t(w.grid) * 8) * sizeof(double);
    const cudaError_t e = cudaMalloc(&sc.partials, bytes);
    if (e != cudaSuccess) return fail(std::string("mlp: cudaMalloc: ") + cudaGetErrorString(e), FLBM_E_NOMEM);
    w.partials = sc.partials;
    w.lpart = sc.partials + size_t(w.grid) * kNpPad;
    return FLBM_OK;
}

float norm_of(uint64_t count) { return float(1.0 / (double(count) * kNout)); }

// gradient (and loss sum) of batch b of the epoch order into w.grad
cudaError_t launch_grad(Scratch &sc, Work &w, const Samples &s, uint64_t b)
{
    const uint64_t count = std::min<uint64_t>(s.batch, s.n - b * s.batch), tiles = (count + w.T - 1) / w.T;
    const int grid = int(std::min<uint64_t>(tiles, uint64_t(w.grid)));
    with_tile(w.T, [&](auto tag) {
        constexpr int T = decltype(tag)::value;
        k_mlp_grad<T><<<grid, kGradThreads, sizeof(GradSmem<T>), sc.s>>>(w.img, s, b, norm_of(count), w.partials,
                                                                           w.lpart);
    });
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_mlp_reduce<<<(kNp + 1 + 255) / 256, 256, 0, sc.s>>>(w.partials, w.lpart, grid, w.grad);
    return cudaGetLastError();
}

// Whether a cooperative launch was refused for want of the SMs or of the
// feature: a process may hold only part of the device's SMs (MPS, green
// contexts), and the grid takes every one that the device has.
bool refused(cudaError_t e) { return e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported; }

// FLBM_INJECT_REFUSE=1 (environment, failure-injection tests only): the
// cooperative launch is refused.
cudaError_t launch_train(Scratch &sc, const Work &w, TrainArgs &a)
{
    const char *inject = std::getenv("FLBM_INJECT_REFUSE");
    if (inject && std::atoi(inject) == 1) return cudaErrorCooperativeLaunchTooLarge;
    void *args[] = {&a};
    return with_tile(w.T, [&](auto tag) {
        constexpr int T = decltype(tag)::value;
        return cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(k_mlp_train<T>), dim3(unsigned(w.grid)),
                                           dim3(kGradThreads), args, sizeof(TrainSmem<T>), sc.s);
    });
}

}  // namespace

}  // namespace flbm

using namespace flbm;

extern "C" int flbm_mlp_grad(const float *params, const float *dev_x, const float *dev_t, int64_t n, float *grad,
                             double *loss)
{
    if (!params || !dev_x || !dev_t || !grad || n < 1 || n >= (int64_t(1) << 32))
        return fail("flbm_mlp_grad: NULL argument or n outside [1, 2^32)", FLBM_E_INVALID);
    if (!is_device_memory(dev_x) || !is_device_memory(dev_t))
        return fail("flbm_mlp_grad: dev_x and dev_t must be device (or managed) memory", FLBM_E_INVALID);
    Work w;
    Scratch sc;
    int rc = prepare(sc, w, params, uint64_t(n), 1, false);
    if (rc) return rc;
    cudaError_t e = launch_grad(sc, w, Samples{dev_x, dev_t, uint64_t(n), uint64_t(n), 1, 0}, 0);
    std::vector<double> h(kNp + 1);
    if (e == cudaSuccess) e = cudaMemcpyAsync(h.data(), w.grad, (kNp + 1) * sizeof(double), cudaMemcpyDeviceToHost, sc.s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(sc.s);
    if (e != cudaSuccess) return fail(std::string("flbm_mlp_grad: ") + cudaGetErrorString(e), FLBM_E_CUDA);
    for (int p = 0; p < kNp; ++p) grad[p] = float(h[p]);
    if (loss) *loss = h[kNp] / (double(n) * kNout);
    return FLBM_OK;
}

extern "C" int flbm_mlp_train(float *params, const float *dev_x, const float *dev_t, int64_t n, int epochs,
                              int batch, double lr, uint64_t seed, double *epoch_loss)
{
    if (!params || !dev_x || !dev_t || n < 1 || n >= (int64_t(1) << 32) || epochs < 1 || batch < 1 ||
        !(lr > 0.0) || !std::isfinite(lr))
        return fail("flbm_mlp_train: bad argument", FLBM_E_INVALID);
    if (!is_device_memory(dev_x) || !is_device_memory(dev_t))
        return fail("flbm_mlp_train: dev_x and dev_t must be device (or managed) memory", FLBM_E_INVALID);
    const uint64_t N = uint64_t(n);
    const uint64_t B = std::min<uint64_t>(uint64_t(batch), N);
    const uint64_t nb = (N + B - 1) / B;
    const uint64_t total = uint64_t(epochs) * nb;
    // host buffers of copies in flight: they outlive the workspace's stream
    std::vector<double> losses(size_t(epochs), 0.0), h(nb);
    std::vector<float> lrs;
    Work w;
    Scratch sc;
    int rc = prepare(sc, w, params, B, nb, true);
    if (rc) return rc;
    if (w.epochs_in_one) lrs.resize(nb);
    std::mt19937_64 rng(seed);
    const float beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
    double p1 = 1.0, p2 = 1.0;
    uint64_t it = 0;
    // bias-corrected step size of the next mini-batch: cosine decay to 5 %
    // over the run
    const auto next_lr = [&] {
        const double frac = double(it++) / double(std::max<uint64_t>(total - 1, 1));
        const double lr_it = lr * (0.05 + 0.95 * 0.5 * (1.0 + std::cos(3.141592653589793 * frac)));
        p1 *= beta1;
        p2 *= beta2;
        return float(lr_it * std::sqrt(1.0 - p2) / (1.0 - p1));
    };
    cudaError_t e = cudaSuccess;
    unsigned int book[2] = {0, 0};
    for (int ep = 0; ep < epochs && e == cudaSuccess; ++ep) {
        // epoch order: an affine bijection of [0, n) with a random multiplier coprime to n
        uint64_t mult = 1, off = 0;
        if (N > 1) {
            do mult = 1 + rng() % (N - 1);
            while (std::gcd(mult, N) != 1);
            off = rng() % N;
        }
        const Samples s{dev_x, dev_t, N, B, mult, off};
        uint64_t b = 0, planned = 0;   // the next batch; step sizes drawn so far
        if (w.epochs_in_one) {
            for (; b < nb && e == cudaSuccess; b = planned) {
                const uint64_t b1 = std::min(b + kTrainChunk, nb);
                for (uint64_t k = b; k < b1; ++k) lrs[k] = next_lr();
                planned = b1;
                TrainArgs a{s,     b,     b1,   norm_of(B), norm_of(N - (nb - 1) * B), beta1,  beta2, eps, w.img, w.m1,
                            w.m2,  w.lr,  w.act, w.stride, w.lpart, w.loss, w.bar, w.bar + 1};
                e = cudaMemcpyAsync(w.lr, lrs.data() + b, (b1 - b) * sizeof(float), cudaMemcpyHostToDevice, sc.s);
                if (e == cudaSuccess) e = cudaMemsetAsync(w.bar, 0, sizeof(unsigned int), sc.s);
                if (e == cudaSuccess) e = launch_train(sc, w, a);
                if (refused(e)) {
                    if ((rc = without_cooperation(sc, w, B)) != FLBM_OK) return rc;
                    e = cudaSuccess;
                    break;
                }
            }
        }
        for (; b < nb && e == cudaSuccess; ++b) {
            e = launch_grad(sc, w, s, b);
            if (e != cudaSuccess) break;
            e = cudaMemcpyAsync(w.loss + b, w.grad + kNp, sizeof(double), cudaMemcpyDeviceToDevice, sc.s);
            const float lr_b = b < planned ? lrs[b] : next_lr();
            k_mlp_adam<<<(kNp + 255) / 256, 256, 0, sc.s>>>(w.img, w.m1, w.m2, w.grad, lr_b, beta1, beta2, eps);
            if (e == cudaSuccess) e = cudaGetLastError();
        }
        if (e != cudaSuccess) break;
        e = cudaMemcpyAsync(h.data(), w.loss, sizeof(double) * nb, cudaMemcpyDeviceToHost, sc.s);
        if (e == cudaSuccess && w.bar)
            e = cudaMemcpyAsync(book, w.bar, sizeof(book), cudaMemcpyDeviceToHost, sc.s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(sc.s);
        if (e == cudaSuccess && (book[1] & 2u))
            return fail("flbm_mlp_train: a bounded device wait ran out", FLBM_E_TIMEOUT);
        double sum = 0.0;
        for (double v : h) sum += v;
        losses[size_t(ep)] = sum / (double(N) * kNout);
    }
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(w.host.data(), w.img, kImg * sizeof(float), cudaMemcpyDeviceToHost, sc.s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(sc.s);
    if (e == cudaSuccess)
        for (int p = 0; p < kNp; ++p) params[p] = w.host[size_t(image_index(p))];
    if (e != cudaSuccess) return fail(std::string("flbm_mlp_train: ") + cudaGetErrorString(e), FLBM_E_CUDA);
    if (epoch_loss)
        for (int ep = 0; ep < epochs; ++ep) epoch_loss[ep] = losses[size_t(ep)];
    return FLBM_OK;
}
