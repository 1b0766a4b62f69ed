// Network tail (Sec. 2.2), fp32: sum of the dense-1 partial-sum rows in row
// order, times the dense-1 scale s1 (1, or the inverse of the operand scales
// of the e4m3 path), + bias + ReLU, dense 128->32 + ReLU, the 3-way softmax
// head (track, em, none) and the Michel sigmoid head.  The rows of a hit come
// from the stream-K CTAs that shared its tile.
// Two kernels, chosen by launch_head, each with its sums in a fixed order:
//   head_rows_kernel  small launches, whose tiles are spread over many CTAs: a
//                     CTA per one, two or four hits, its warps share the hit's many rows;
//   head_hits_kernel  the others: a CTA per 32 hits, the share of one epilogue
//                     warp of the network kernels.
#include "emtk_internal.h"

namespace emtk {
namespace {

__device__ __forceinline__ unsigned long long global_timer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The dense-2 weights [128][32]: a thread's share, then into shared memory
// (16-byte aligned).
template <int kThreads>
struct W2Share {
    static constexpr int kN4 = kN1 * kN2 / 4 / kThreads;
    static_assert(kN1 * kN2 / 4 % kThreads == 0, "whole float4s per thread");
    float4 v[kN4];
    __device__ __forceinline__ void load(const float *__restrict__ fc2_w) {
#pragma unroll
        for (int k = 0; k < kN4; ++k) v[k] = __ldg(reinterpret_cast<const float4 *>(fc2_w) + threadIdx.x + k * kThreads);
    }
    __device__ __forceinline__ void store(float *w2) const {
#pragma unroll
        for (int k = 0; k < kN4; ++k) reinterpret_cast<float4 *>(w2)[threadIdx.x + k * kThreads] = v[k];
    }
};
constexpr int kManyRows = 4;  // up to this many partial rows per hit, head_hits_kernel at any size

// The tail when a hit has many partial rows (a small launch, whose tiles are
// split over many CTAs), HITS hits per CTA of 8 warps.  What bounds it is its
// chain of latencies after the network kernel's last row, so nothing but the rows
// is loaded on it and every step is spread over the warps:
//   before the wait  thread (warp w, lane j) takes the dense-2 weights of inputs
//                    16 w .. 16 w + 15 to output j into registers;
//   1. kSplit = 8 / HITS warps per hit: warp k sums rows [k R / kSplit,
//      (k + 1) R / kSplit) in order, lane l dense-1 outputs 4 l .. 4 l + 3, up to
//      kDepth rows in one round trip;
//   2. a thread per (hit, dense-1 output) adds the shares in order, bias + ReLU;
//   3. dense-2: every warp its 16 inputs, for all hits;
//   4. a warp per hit adds the 8 parts in order, bias + ReLU, and the head logits
//      by warp sums.
// Against a kernel with the dense-2 weights staged in shared memory, one thread per
// dense-2 output and one per hit for the heads: 256 hits of one plane (76 rows per
// hit) 26.6 -> 23.8 us per call, 128 patches 21.3 -> 18.3, 1,693 54.9 -> 53.9.
constexpr int kThreadsRows = 256;
constexpr int kSmallLaunch = 2048;  // above it, head_hits_kernel
// Up to kOneHit hits one per CTA, up to kTwoHits two, else four: each the fewest that
// keep the launch in one wave of 2 or 3 CTAs per SM (256 hits: 23.8 us per call with
// one, 24.9 with two; 1,000: 38.4 with two, 35.4 with four).
constexpr int kOneHit = 256, kTwoHits = 912;
constexpr int kDepth = 10;          // rows per round trip: all of a share from 129 hits on (77 rows)

template <int HITS>
__global__ void __launch_bounds__(kThreadsRows, HITS == 1 ? 2 : 3) head_rows_kernel(const float *__restrict__ partials, int G,
                                                                int upt, int n_pad, int32_t n, float s1,
                                                                const float *__restrict__ fc1_b,
                                                                const float *__restrict__ fc2_w,
                                                                const float *__restrict__ fc2_b,
                                                                const float *__restrict__ cls_w,
                                                                const float *__restrict__ cls_b,
                                                                const float *__restrict__ mic_w,
                                                                const float *__restrict__ mic_b, OutRows out_rows,
                                                                int debug_logits) {
    constexpr int kWarps = kThreadsRows / 32, kSplit = kWarps / HITS, kShare = kN1 / kWarps;
    static_assert(kThreadsRows % kN1 == 0 && kWarps % HITS == 0, "whole dense-1 rows per pass, whole warps per hit");
    __shared__ __align__(16) float part[kWarps][kN1];        // row sums of each warp's share
    __shared__ __align__(16) float h1[HITS][kN1];
    __shared__ float part2[HITS][kWarps][kN2];
    pdl_trigger();  // the next call's first kernel may be scheduled; it waits for this one
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    float w2[kShare];
#pragma unroll
    for (int i = 0; i < kShare; ++i) w2[i] = __ldg(fc2_w + (kShare * warp + i) * kN2 + lane);
    const float b1 = __ldg(fc1_b + (tid & (kN1 - 1))), b2 = __ldg(fc2_b + lane);
    const float wc[kNC + 1] = {__ldg(cls_w + lane * kNC), __ldg(cls_w + lane * kNC + 1), __ldg(cls_w + lane * kNC + 2),
                               __ldg(mic_w + lane)};
    const float bc[kNC + 1] = {__ldg(cls_b), __ldg(cls_b + 1), __ldg(cls_b + 2), __ldg(mic_b)};
    const int64_t h0 = (int64_t)blockIdx.x * HITS;
    const int64_t units = (int64_t)((n + 127) / 128) * upt;
    const int j = warp / kSplit, share = warp % kSplit;  // this warp's hit and share of its rows
    const int rows = tile_partial_rows((h0 + j) >> 7, units, G, upt);
    int r = rows * share / kSplit;
    const int r_end = rows * (share + 1) / kSplit;
    const int64_t row_stride = (int64_t)n_pad * kN1 / 4;  // float4s between partial rows
    const float4 *p = reinterpret_cast<const float4 *>(partials + (h0 + j) * kN1) + lane;
    pdl_wait();  // the partial sums and output rows come from the kernels before
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (; r < r_end; r += kDepth) {  // a row past n lies in the tile's padding: read, never used
        float4 v[kDepth];
#pragma unroll
        for (int k = 0; k < kDepth; ++k)
            if (r + k < r_end) v[k] = p[(r + k) * row_stride];
#pragma unroll
        for (int k = 0; k < kDepth; ++k)
            if (r + k < r_end) {
                a.x += v[k].x;
                a.y += v[k].y;
                a.z += v[k].z;
                a.w += v[k].w;
            }
    }
    *reinterpret_cast<float4 *>(&part[warp][4 * lane]) = a;
    __syncthreads();
#pragma unroll
    for (int e = tid; e < HITS * kN1; e += kThreadsRows) {
        const int i = e / kN1, k = tid % kN1;
        float s = part[i * kSplit][k];
#pragma unroll
        for (int q = 1; q < kSplit; ++q) s += part[i * kSplit + q][k];
        h1[i][k] = fmaxf(fmaf(s, s1, b1), 0.f);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < HITS; ++i) {
        float acc = 0.f;
#pragma unroll
        for (int k = 0; k < kShare; k += 4) {
            const float4 x = *reinterpret_cast<const float4 *>(&h1[i][kShare * warp + k]);
            acc = fmaf(x.x, w2[k], acc);
            acc = fmaf(x.y, w2[k + 1], acc);
            acc = fmaf(x.z, w2[k + 2], acc);
            acc = fmaf(x.w, w2[k + 3], acc);
        }
        part2[i][warp][lane] = acc;
    }
    __syncthreads();
    const int64_t h = h0 + warp;
    if (warp >= HITS || h >= n) return;
    float v = b2;
#pragma unroll
    for (int q = 0; q < kWarps; ++q) v += part2[warp][q][lane];
    v = fmaxf(v, 0.f);
    float z[kNC + 1];
#pragma unroll
    for (int c = 0; c <= kNC; ++c) {
        z[c] = v * wc[c];
#pragma unroll
        for (int o = 16; o; o >>= 1) z[c] += __shfl_xor_sync(0xffffffffu, z[c], o);
        z[c] += bc[c];
    }
    const float m = fmaxf(fmaxf(z[0], z[1]), z[2]);
    const float e0 = expf(z[0] - m), e1 = expf(z[1] - m), e2 = expf(z[2] - m);
    const float sum = e0 + e1 + e2;
    float *out = out_rows.rows ? out_rows.rows + h * (int64_t)out_rows.stride : out_rows.dest[h];
    if (lane < 4) out[lane] = lane < kNC ? (lane == 0 ? e0 : lane == 1 ? e1 : e2) / sum : 1.0f / (1.0f + expf(-z[kNC]));
    if (debug_logits && lane < 4) out[4 + lane] = lane == 0 ? z[0] : lane == 1 ? z[1] : lane == 2 ? z[2] : z[3];
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
// kernel; this one ends about 6 us after it.
// LATE: the dense-2 weights, loaded first, go to shared memory only after the rows,
// one round trip off the chain of a launch of a single wave of CTAs (5,000 patches
// 127.3 -> 125.1 us, one APA in three calls 469.7 -> 464.3); in a launch of several
// waves the registers that hold them cost more (full event 1,210 -> 1,217).
constexpr int kHeadHits = 32;
constexpr int kThreadsHits = 128;
constexpr int kH1Pitch = kN1 + 4;  // h1 rows: 16-byte aligned, hits 8 apart in different banks
constexpr int kLateHits = 3 * 152 * kHeadHits;  // hits of one wave: three CTAs per SM

template <bool LATE>
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
    W2Share<kThreadsHits> w2v;
    w2v.load(fc2_w);
    if (!LATE) w2v.store(&w2[0][0]);
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
    if (LATE) w2v.store(&w2[0][0]);
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
    if (rows > kManyRows && n <= kSmallLaunch) {
        if (n <= kOneHit)
            return launch_pdl(head_rows_kernel<1>, dim3(n), dim3(kThreadsRows), 0, s, partials, G, upt, n_pad, n, s1,
                              b1, w2, b2, wc, bc, wm, bm, out_rows, debug_logits);
        if (n <= kTwoHits)
            return launch_pdl(head_rows_kernel<2>, dim3((n + 1) / 2), dim3(kThreadsRows), 0, s, partials, G, upt, n_pad,
                              n, s1, b1, w2, b2, wc, bc, wm, bm, out_rows, debug_logits);
        return launch_pdl(head_rows_kernel<4>, dim3((n + 3) / 4), dim3(kThreadsRows), 0, s, partials, G, upt, n_pad, n,
                          s1, b1, w2, b2, wc, bc, wm, bm, out_rows, debug_logits);
    }
    return launch_pdl(n <= kLateHits ? head_hits_kernel<true> : head_hits_kernel<false>,
                      dim3((n + kHeadHits - 1) / kHeadHits), dim3(kThreadsHits), 0, s, partials, G, upt, n_pad, n, s1, b1,
                      w2, b2, wc, bc, wm, bm, out_rows, debug_logits, tile_done, status, (long long)timeout_ns);
}

}  // namespace emtk
