// Network tail (Sec. 2.2), fp32: sum of the dense-1 partial-sum rows in row
// order, times the dense-1 scale s1 (1, or the inverse of the operand scales
// of the e4m3 path), + bias + ReLU, dense 128->32 + ReLU, the 3-way softmax
// head (track, em, none) and the Michel sigmoid head.  The rows of a hit come
// from the stream-K CTAs that shared its tile.
// Two kernels, chosen by launch_head:
//   head_rows_kernel  small launches, whose tiles are spread over many CTAs: a
//                     warp per hit sums its many rows, 16 deep (from 32 rows
//                     on, four warps per hit each sum a quarter of the rows
//                     and the quarters are added in order);
//   head_hits_kernel  the others: a CTA per 32 hits, the share of one epilogue
//                     warp of the network kernels.
// Both add the rows in order (but for the four quarters) and the inputs of
// every dense-2 and head sum in order, so they give the same bits.
#include "emtk_internal.h"

namespace emtk {
namespace {

__device__ __forceinline__ unsigned long long global_timer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The dense-2 weights [128][32] into shared memory (16-byte aligned): every
// load issued before the first store, so that staging costs one round trip.
template <int kThreads>
__device__ __forceinline__ void stage_w2(float *w2, const float *__restrict__ fc2_w) {
    constexpr int kN4 = kN1 * kN2 / 4;
    static_assert(kN4 % kThreads == 0, "whole float4s per thread");
    float4 v[kN4 / kThreads];
#pragma unroll
    for (int k = 0; k < kN4 / kThreads; ++k)
        v[k] = __ldg(reinterpret_cast<const float4 *>(fc2_w) + threadIdx.x + k * kThreads);
#pragma unroll
    for (int k = 0; k < kN4 / kThreads; ++k) reinterpret_cast<float4 *>(w2)[threadIdx.x + k * kThreads] = v[k];
}
constexpr int kManyRows = 4;    // up to this many partial rows per hit, head_hits_kernel at any size
constexpr int kSplitRows = 32;  // from this many, head_rows_kernel with four warps per hit

// The tail when a hit has many partial rows (a small launch, whose tiles are
// split over many CTAs): one warp per hit sums the rows, lane l taking dense-1
// outputs 4l .. 4l+3 of every row (512 contiguous bytes per row), and writes
// bias + ReLU to shared memory; every thread then computes dense-2 outputs (one
// per hit and output), and one thread per hit the heads.
constexpr int kThreadsRows = 256;
constexpr int kSmallLaunch = 2048;
constexpr int kH1Stride = kN1 + 1;  // shared h1 rows padded: thread t reads row t conflict-free

// kSplit warps share a hit: warp k of the hit sums its rows [k R / kSplit,
// (k+1) R / kSplit) in order, and the kSplit partial sums are then added in
// k order (kSplit = 1: all rows in order).  More warps
// per hit put more of the GPU on a small launch's many rows.
template <int kHitsRows, int kSplit = 1>
__global__ void __launch_bounds__(kThreadsRows) head_rows_kernel(const float *__restrict__ partials, int G,
                                                                int upt, int n_pad, int32_t n, float s1,
                                                                const float *__restrict__ fc1_b,
                                                                const float *__restrict__ fc2_w,
                                                                const float *__restrict__ fc2_b,
                                                                const float *__restrict__ cls_w,
                                                                const float *__restrict__ cls_b,
                                                                const float *__restrict__ mic_w,
                                                                const float *__restrict__ mic_b, OutRows out_rows,
                                                                int debug_logits) {
    static_assert(kHitsRows * kSplit <= kThreadsRows / 32 || kSplit == 1, "a warp per (hit, row share)");
    __shared__ float h1s[kHitsRows * kH1Stride];
    __shared__ __align__(16) float4 part[kSplit > 1 ? kHitsRows * kSplit * 32 : 1];
    __shared__ float h2s[kHitsRows * (kN2 + 1)];
    __shared__ __align__(16) float w2[kN1][kN2];
    __shared__ __align__(16) float wc[kN2][kNC + 1];
    __shared__ float b2[kN2];
    pdl_trigger();  // the next call's first kernel may be scheduled; it waits for this one
    stage_w2<kThreadsRows>(&w2[0][0], fc2_w);
    for (int i = threadIdx.x; i < kN2 * kNC; i += blockDim.x) wc[i / kNC][i % kNC] = cls_w[i];
    for (int i = threadIdx.x; i < kN2; i += blockDim.x) {
        wc[i][kNC] = mic_w[i];
        b2[i] = fc2_b[i];
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    pdl_wait();  // the partial sums and output rows come from the kernels before
    const int64_t h0 = (int64_t)blockIdx.x * kHitsRows;
    const int64_t row_stride = (int64_t)n_pad * kN1 / 4;  // float4s between partial rows
    const float4 bb = reinterpret_cast<const float4 *>(fc1_b)[lane];
    for (int jw = warp; jw < kHitsRows * kSplit; jw += kThreadsRows / 32) {
        const int j = jw / kSplit, share = jw % kSplit;
        const int64_t h = h0 + j;
        if (h >= n) {
            if (kSplit > 1) continue;
            break;
        }
        const int rows = tile_partial_rows(h >> 7, (int64_t)((n + 127) / 128) * upt, G, upt);
        const int r_end = (int)((int64_t)rows * (share + 1) / kSplit);
        const float4 *p = reinterpret_cast<const float4 *>(partials + h * kN1) + lane;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        // this warp's rows in order, loaded kDepth at a time (the last batch
        // predicated), so that a hit's rows cost one round trip per kDepth rows
        constexpr int kDepth = 16;
        for (int r = (int)((int64_t)rows * share / kSplit); r < r_end; r += kDepth) {
            float4 v[kDepth];
#pragma unroll
            for (int k = 0; k < kDepth; ++k)
                if (r + k < r_end) v[k] = p[(r + k) * row_stride];
#pragma unroll
            for (int k = 0; k < kDepth; ++k) {
                if (r + k < r_end) {
                    a.x += v[k].x;
                    a.y += v[k].y;
                    a.z += v[k].z;
                    a.w += v[k].w;
                }
            }
        }
        if (kSplit > 1) {
            part[jw * 32 + lane] = a;
            continue;
        }
        float *o = h1s + j * kH1Stride + 4 * lane;
        o[0] = fmaxf(fmaf(a.x, s1, bb.x), 0.f);
        o[1] = fmaxf(fmaf(a.y, s1, bb.y), 0.f);
        o[2] = fmaxf(fmaf(a.z, s1, bb.z), 0.f);
        o[3] = fmaxf(fmaf(a.w, s1, bb.w), 0.f);
    }
    if (kSplit > 1) {  // the shares of each hit, added in share order
        __syncthreads();
        for (int jw = warp; jw < kHitsRows; jw += kThreadsRows / 32) {
            float4 a = part[(jw * kSplit) * 32 + lane];
#pragma unroll
            for (int k = 1; k < kSplit; ++k) {
                const float4 v = part[(jw * kSplit + k) * 32 + lane];
                a.x += v.x;
                a.y += v.y;
                a.z += v.z;
                a.w += v.w;
            }
            float *o = h1s + jw * kH1Stride + 4 * lane;
            o[0] = fmaxf(fmaf(a.x, s1, bb.x), 0.f);
            o[1] = fmaxf(fmaf(a.y, s1, bb.y), 0.f);
            o[2] = fmaxf(fmaf(a.z, s1, bb.z), 0.f);
            o[3] = fmaxf(fmaf(a.w, s1, bb.w), 0.f);
        }
    }
    __syncthreads();
    // dense-2 with every thread: output j of hit i is thread (32 i + j) mod 256's,
    // an fmaf chain over k in order
    for (int o = threadIdx.x; o < kHitsRows * kN2; o += kThreadsRows) {
        const int i = o / kN2, j = o % kN2;
        const float *h1 = h1s + i * kH1Stride;
        float acc = b2[j];
#pragma unroll 8
        for (int k = 0; k < kN1; ++k) acc = fmaf(h1[k], w2[k][j], acc);
        h2s[i * (kN2 + 1) + j] = acc;
    }
    __syncthreads();
    if (threadIdx.x >= kHitsRows) return;
    const int64_t h = h0 + threadIdx.x;
    if (h >= n) return;
    const float *h2 = h2s + threadIdx.x * (kN2 + 1);
    float z[kNC + 1] = {cls_b[0], cls_b[1], cls_b[2], mic_b[0]};
#pragma unroll
    for (int j = 0; j < kN2; ++j) {
        const float v = fmaxf(h2[j], 0.f);
        const float4 wv = *reinterpret_cast<const float4 *>(&wc[j][0]);
        z[0] = fmaf(v, wv.x, z[0]);
        z[1] = fmaf(v, wv.y, z[1]);
        z[2] = fmaf(v, wv.z, z[2]);
        z[3] = fmaf(v, wv.w, z[3]);
    }
    const float m = fmaxf(fmaxf(z[0], z[1]), z[2]);
    const float e0 = expf(z[0] - m), e1 = expf(z[1] - m), e2 = expf(z[2] - m);
    const float sum = e0 + e1 + e2;
    float *out = out_rows.rows ? out_rows.rows + h * (int64_t)out_rows.stride : out_rows.dest[h];
    out[0] = e0 / sum;
    out[1] = e1 / sum;
    out[2] = e2 / sum;
    out[3] = 1.0f / (1.0f + expf(-z[kNC]));
    if (debug_logits) {
        out[4] = z[0];
        out[5] = z[1];
        out[6] = z[2];
        out[7] = z[3];
    }
}

// The tail of the other launches: one CTA of 128 threads per 32 hits, the hits
// whose partial rows one epilogue warp of each contributing network CTA stores.
//   1. warp w sums the rows of hits 8w .. 8w + 7, lane l taking dense-1 outputs
//      4l .. 4l + 3 (512 contiguous bytes per row), four hits x four rows in
//      flight, and writes bias + ReLU to h1[hit][k];
//   2. dense-2: a thread keeps 4 hits x 2 outputs, four inputs per step;
//   3. four threads per hit: the head logits, then softmax and sigmoid.
// What bounds it: the latency of this chain after the last network CTA of a
// tile, and in a large launch the rows' L2 reads.  With a CTA per 128-hit tile
// (256 threads) a launch of 7,692 hits, 61 tiles, ended 24 us after its network
// kernel; this one ends about 8 us after it.
constexpr int kHeadHits = 32;
constexpr int kThreadsHits = 128;
constexpr int kH1Pitch = kN1 + 4;  // h1 rows: 16-byte aligned, hits 8 apart in different banks

__global__ void __launch_bounds__(kThreadsHits) head_hits_kernel(const float *__restrict__ partials, int G,
                                                                int upt, int n_pad, int32_t n, float s1,
                                                                const float *__restrict__ fc1_b,
                                                                const float *__restrict__ fc2_w,
                                                                const float *__restrict__ fc2_b,
                                                                const float *__restrict__ cls_w,
                                                                const float *__restrict__ cls_b,
                                                                const float *__restrict__ mic_w,
                                                                const float *__restrict__ mic_b, OutRows out_rows,
                                                                int debug_logits, int *tile_done, int *status,
                                                                long long timeout_ns) {
    __shared__ __align__(16) float h1[kHeadHits][kH1Pitch];
    __shared__ __align__(16) float w2[kN1][kN2];
    __shared__ float h2s[kHeadHits][kN2 + 1];
    __shared__ float wc[kN2][kNC + 1];
    __shared__ int go;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    pdl_trigger();  // the next call's first kernel may be scheduled; it waits for this one
    stage_w2<kThreadsHits>(&w2[0][0], fc2_w);
    for (int i = tid; i < kN2 * kNC; i += kThreadsHits) wc[i / kNC][i % kNC] = cls_w[i];
    for (int i = tid; i < kN2; i += kThreadsHits) wc[i][kNC] = mic_w[i];
    const int64_t h0 = (int64_t)blockIdx.x * kHeadHits;
    const int rows = tile_partial_rows(h0 >> 7, (int64_t)((n + 127) / 128) * upt, G, upt);
    if (tile_done != nullptr) {
        // the hits' partial rows are complete once one epilogue warp of each of the tile's
        // `rows` CTAs counted its own; the output rows were written before those CTAs read
        // their windows.  Every network CTA is running (this kernel is scheduled after all of
        // them started), so the wait ends unless the network kernel gave up (bit 0 of *status)
        if (tid == 0) {
            int ok = 1;
            const long long t0 = (long long)global_timer();
            for (;;) {
                int v;
                asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(tile_done + blockIdx.x) : "memory");
                if (v >= rows) break;
                if (*reinterpret_cast<volatile int *>(status) & 1) {
                    ok = 0;
                    break;
                }
                if ((long long)global_timer() - t0 > timeout_ns) {
                    atomicOr(status, 2);
                    ok = 0;
                    break;
                }
                __nanosleep(200);
            }
            tile_done[blockIdx.x] = 0;  // every row is counted (or the launch gave up): zero for the next launch
            // one block lasts as long as the network kernel, so that the completion of this
            // kernel implies that one's
            if (blockIdx.x == gridDim.x - 1) pdl_wait();
            go = ok;
        }
        __syncthreads();
        if (!go) return;
    } else {
        pdl_wait();  // the partial sums and output rows come from the kernels before
    }
    const int64_t row_stride = (int64_t)n_pad * kN1 / 4;  // float4s between partial rows
    const float4 bb = reinterpret_cast<const float4 *>(fc1_b)[lane];
    constexpr int kB = 4;  // hits, and rows, in flight.  Rows past n are read (the tile's padding), never used
#pragma unroll
    for (int j0 = 0; j0 < kHeadHits / 4; j0 += kB) {
        const float4 *p = reinterpret_cast<const float4 *>(partials + (h0 + warp * (kHeadHits / 4) + j0) * kN1) + lane;
        float4 a[kB];
#pragma unroll
        for (int u = 0; u < kB; ++u) a[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int r = 0; r < rows; r += kB) {
            float4 v[kB][kB];
#pragma unroll
            for (int k = 0; k < kB; ++k)
                if (r + k < rows) {
#pragma unroll
                    for (int u = 0; u < kB; ++u) v[k][u] = __ldcg(p + (r + k) * row_stride + u * (kN1 / 4));
                }
#pragma unroll
            for (int k = 0; k < kB; ++k)
                if (r + k < rows) {
#pragma unroll
                    for (int u = 0; u < kB; ++u) {
                        a[u].x += v[k][u].x;
                        a[u].y += v[k][u].y;
                        a[u].z += v[k][u].z;
                        a[u].w += v[k][u].w;
                    }
                }
        }
#pragma unroll
        for (int u = 0; u < kB; ++u)  // s1 is a power of two: a * s1 + b rounds once, as a + b does for s1 = 1
            *reinterpret_cast<float4 *>(&h1[warp * (kHeadHits / 4) + j0 + u][4 * lane]) =
                make_float4(fmaxf(fmaf(a[u].x, s1, bb.x), 0.f), fmaxf(fmaf(a[u].y, s1, bb.y), 0.f),
                            fmaxf(fmaf(a[u].z, s1, bb.z), 0.f), fmaxf(fmaf(a[u].w, s1, bb.w), 0.f));
    }
    __syncthreads();
    {
        const int hg = lane & 7, og = 4 * warp + (lane >> 3);  // hits hg + 8 i, outputs 2 og, 2 og + 1
        float acc[4][2];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int q = 0; q < 2; ++q) acc[i][q] = __ldg(fc2_b + 2 * og + q);
#pragma unroll 2
        for (int k = 0; k < kN1; k += 4) {
            float x[4][4];
            float2 w[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const float4 v = *reinterpret_cast<const float4 *>(&h1[hg + 8 * i][k]);
                x[i][0] = v.x, x[i][1] = v.y, x[i][2] = v.z, x[i][3] = v.w;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) w[e] = *reinterpret_cast<const float2 *>(&w2[k + e][2 * og]);
#pragma unroll
            for (int e = 0; e < 4; ++e)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    acc[i][0] = fmaf(x[i][e], w[e].x, acc[i][0]);
                    acc[i][1] = fmaf(x[i][e], w[e].y, acc[i][1]);
                }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int q = 0; q < 2; ++q) h2s[hg + 8 * i][2 * og + q] = acc[i][q];
    }
    __syncthreads();
    const int i = tid >> 2, c = tid & 3;  // hit i, logit c: track, em, none, michel
    float z = c < kNC ? __ldg(cls_b + c) : __ldg(mic_b);
#pragma unroll
    for (int j = 0; j < kN2; ++j) z = fmaf(fmaxf(h2s[i][j], 0.f), wc[j][c], z);
    const float z0 = __shfl_sync(0xffffffffu, z, 0, 4), z1 = __shfl_sync(0xffffffffu, z, 1, 4),
                z2 = __shfl_sync(0xffffffffu, z, 2, 4);
    const float m = fmaxf(fmaxf(z0, z1), z2);
    const float e = expf(c < kNC ? z - m : -z);
    const float sum = __shfl_sync(0xffffffffu, e, 0, 4) + __shfl_sync(0xffffffffu, e, 1, 4) +
                      __shfl_sync(0xffffffffu, e, 2, 4);
    const int64_t h = h0 + i;
    if (h >= n) return;
    // through L2: the rows were written by a kernel that is not ordered before this one by its launch
    float *out = out_rows.rows ? out_rows.rows + h * (int64_t)out_rows.stride
                               : reinterpret_cast<float *>(
                                     __ldcg(reinterpret_cast<const unsigned long long *>(out_rows.dest + h)));
    out[c] = c < kNC ? e / sum : 1.0f / (1.0f + e);
    if (debug_logits) out[4 + c] = z;
}

}  // namespace

bool head_counts_tiles(int32_t n, int rows) {
    return n > kSmallLaunch && rows <= kManyRows;
}

cudaError_t launch_head(const DeviceWeights &w, const float *partials, int G, int upt, int rows, int n_pad, int32_t n,
                        OutRows out_rows, int debug_logits, int *tile_done, int *status, int64_t timeout_ns,
                        cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    // launched as dependents of the network kernel: the weights are staged while it finishes
    const float s1 = w.fc1_scale;
    const float *b1 = w.fc1_b, *w2 = w.fc2_w, *b2 = w.fc2_b, *wc = w.cls_w, *bc = w.cls_b, *wm = w.mic_w,
                *bm = w.mic_b;
    if (rows > kManyRows) {
        if (rows >= kSplitRows && n <= kSmallLaunch)  // a hit's rows over 4 warps, 2 hits per block
            return launch_pdl(head_rows_kernel<2, 4>, dim3((n + 1) / 2), dim3(kThreadsRows), 0, s, partials, G,
                              upt, n_pad, n, s1, b1, w2, b2, wc, bc, wm, bm, out_rows, debug_logits);
        if (n <= kSmallLaunch)  // 8 hits per block: more blocks, so more rows summed at once
            return launch_pdl(head_rows_kernel<8>, dim3((n + 7) / 8), dim3(kThreadsRows), 0, s, partials, G, upt,
                              n_pad, n, s1, b1, w2, b2, wc, bc, wm, bm, out_rows, debug_logits);
    }
    return launch_pdl(head_hits_kernel, dim3((n + kHeadHits - 1) / kHeadHits), dim3(kThreadsHits), 0, s, partials, G,
                      upt, n_pad, n, s1, b1, w2, b2, wc, bc, wm, bm, out_rows, debug_logits, tile_done, status,
                      (long long)timeout_ns);
}

}  // namespace emtk
