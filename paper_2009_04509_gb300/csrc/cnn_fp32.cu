// fp32 network path on CUDA cores (EMTK_FP32): conv 5x5x48 + ReLU fused
// with dense-1 (Sec. 2.2).
//
// Work units are (tile of 128 hits, pair of conv positions (x, x + 1), x even):
// 968 per tile.  One persistent CTA per SM takes a contiguous range of units
// (stream-K), across tile boundaries, so every SM gets the same work (+-1 pair)
// whatever the hit count; a grid of whole K splits left the last of 2 to 5
// waves mostly empty (628 CTAs on 152 SMs for 20,000 hits).  256 threads, a conv
// warp and a dense-1 warp on each SM sub-partition, joined by a ring of two
// shared-memory slots (one pair each: its 96 x 128 dense-1 weights and its
// 96 x 128 activations):
//   conv warps     bring the pair's dense-1 weights in (cp.async) and compute
//                  its activations: the 5 x 8 window of a quad of positions is
//                  staged in shared memory, a thread takes two hits and 24
//                  filters, one window row per loop iteration;
//   dense-1 warps  16 hits x 8 outputs per thread in 64 packed pairs of hits,
//                  the next input's 6 shared-memory loads in flight under the
//                  current one's 64 FMAs.
// Both use the packed FMA (two IEEE fp32 FMAs per instruction): the FMA pipe
// runs 128 FMAs per cycle and SM either way, but the packed form leaves half
// the issue slots to loads, to the copies that put a scalar into both halves of
// a pair, and to the other warp.  Both loops are short on purpose: straight-line
// code that does not fit the instruction cache ran at a quarter of its rate (a
// fully unrolled conv took 6,000 cycles per position for 1,200 FMAs).
//
// What bounds it: the FMA pipe.  A position is 7,344 pipe cycles; it takes about
// 9,400 (one APA, 20,000 hits: 9.3 ms, 61 TFLOP/s, 0.75 of the derived peak; the
// kernel before this one 13.6 ms).  Operands that are all 64-bit pairs straight from
// shared memory (each activation stored twice, no copies) ran at 42 TFLOP/s, an
// 8 x 8 register tile on twice the warps at 59, scalar FMAs at 53.
//
// The dense-1 sums restart every kSeg positions of a tile and are added to
// the CTA's partial row of the tile with one fp32 add per segment, in order
// (deterministic; shorter chains of sums round less: scores of 2,080 patches
// are off by 9.8e-7 against 64 bits with 16 positions, 1.4e-6 with 44, 8.0e-7
// with 8, and 1.7e-6 in the kernel before this one; with 44 the kernel is 1.2 %
// faster, with 8 3 % slower).  The head kernel adds
// the partial rows of the CTAs that shared a tile, in CTA order.
#include "emtk_internal.h"

namespace emtk {
namespace {

constexpr int kHT = 128;          // hits per tile
constexpr int kRole = 128;        // threads of each role
constexpr int kThreads = 2 * kRole;
constexpr int kPairs = kPos / 2;   // units per tile: pairs of conv positions (x, x + 1), x even
constexpr int kSlots = 4;          // ring slots (positions)
constexpr int kSeg = 16;           // positions per dense-1 segment
constexpr int kW1Pos = kF * kN1;   // 6144 weights of one position (24 KB)
constexpr int kActPos = kF * kHT;  // 6144 activations of one position
constexpr int kWinHalf = kK * kHT * 4;      // 5 rows x 128 hits x 4 columns of a quad's window
constexpr int kConvF = kK * kK * kF + kF;   // conv weights [25][48], then the bias [48]
constexpr int kSmemBytes = (kSlots * (kW1Pos + kActPos) + 2 * kWinHalf + kConvF) * 4;
static_assert(kSmemBytes <= 232448, "shared memory budget");
static_assert((kSlots & (kSlots - 1)) == 0, "slot index by mask");
static_assert(kW1Pos % (4 * kRole) == 0 && kQ % 4 == 0, "whole vectors per thread; quads do not straddle rows");

__device__ __forceinline__ void cp_async16(float *smem_dst, const float *gmem_src) {
    const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(smem_dst));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Named barriers of the ring: pair b (two slots) is full at kBarFull + b (conv
// warps arrive, dense-1 warps wait) and free at kBarFree + b (the other way
// round); kBarConv joins the conv warps.
constexpr int kBarFull = 1, kBarFree = 3, kBarConv = 5;
__device__ __forceinline__ void bar_wait(int id) { asm volatile("bar.sync %0, %1;" ::"r"(id), "n"(kThreads) : "memory"); }
__device__ __forceinline__ void bar_arrive(int id) {
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "n"(kThreads) : "memory");
}
__device__ __forceinline__ void bar_conv() { asm volatile("bar.sync %0, %1;" ::"n"(kBarConv), "n"(kRole) : "memory"); }

// The 48 x 128 dense-1 weights of position p into dst: thread t's share, copied
// asynchronously.
__device__ __forceinline__ void load_w1(float *dst, const float *__restrict__ fc1_w, int p, int t) {
    const float *src = fc1_w + (int64_t)p * kW1Pos;
#pragma unroll
    for (int k = 0; k < kW1Pos / 4 / kRole; ++k) cp_async16(dst + (t + k * kRole) * 4, src + (t + k * kRole) * 4);
}

// Conv + ReLU of positions x, x + 1 (window columns C0 .. C0 + 5 of the staged
// quad) for two hits, 32 apart, and 24 filters, into the pair's activations.  One
// window row's 5 taps per iteration (a loop that stays in the instruction
// cache): per tap, 12 packed filter pairs x 2 positions x 2 hits on 6 weight
// loads, which every lane reads at once.
template <int C0>
__device__ __forceinline__ void conv_pair(const float *win, const float *cw, float *act) {
    float2 s[2][2][12];  // [hit][position][filter pair]
    const float2 *bias = reinterpret_cast<const float2 *>(cw + kK * kK * kF);
#pragma unroll
    for (int f = 0; f < 12; ++f) s[0][0][f] = s[0][1][f] = s[1][0][f] = s[1][1][f] = bias[f];
#pragma unroll 1
    for (int r = 0; r < kK; ++r, cw += kK * kF, win += kHT * 4) {
        float px[2][8];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const float4 lo = *reinterpret_cast<const float4 *>(win + h * 32 * 4);
            const float4 hi = *reinterpret_cast<const float4 *>(win + h * 32 * 4 + kWinHalf);
            px[h][0] = lo.x, px[h][1] = lo.y, px[h][2] = lo.z, px[h][3] = lo.w;
            px[h][4] = hi.x, px[h][5] = hi.y, px[h][6] = hi.z, px[h][7] = hi.w;
        }
#pragma unroll
        for (int j = 0; j < kK; ++j)
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const float4 w = *reinterpret_cast<const float4 *>(cw + j * kF + 4 * q);
                const float2 wl = make_float2(w.x, w.y), wh = make_float2(w.z, w.w);
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        const float2 v = make_float2(px[h][C0 + j + x], px[h][C0 + j + x]);
                        s[h][x][2 * q] = __ffma2_rn(v, wl, s[h][x][2 * q]);
                        s[h][x][2 * q + 1] = __ffma2_rn(v, wh, s[h][x][2 * q + 1]);
                    }
            }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
            for (int f = 0; f < 12; ++f) {
                float *d = act + x * kActPos + 2 * f * kHT + 32 * h;
                d[0] = fmaxf(s[h][x][f].x, 0.0f);
                d[kHT] = fmaxf(s[h][x][f].y, 0.0f);
            }
}

// One input's operands of a dense-1 thread: 16 hits (4 x 4, 32 apart) and 8
// outputs (2 x 4, 64 apart).
struct Frag {
    float4 a[4], b[2];
    __device__ __forceinline__ void load(const float *act, const float *w1, int c) {
#pragma unroll
        for (int j = 0; j < 4; ++j) a[j] = *reinterpret_cast<const float4 *>(act + c * kHT + 32 * j);
#pragma unroll
        for (int j = 0; j < 2; ++j) b[j] = *reinterpret_cast<const float4 *>(w1 + c * kN1 + 64 * j);
    }
};

// acc[q][o] (pair of hits q, output o) += the pair's activations x the weight of o.
__device__ __forceinline__ void fma_frag(const Frag &f, float2 (&acc)[8][8]) {
    const float b[8] = {f.b[0].x, f.b[0].y, f.b[0].z, f.b[0].w, f.b[1].x, f.b[1].y, f.b[1].z, f.b[1].w};
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const float4 v = f.a[q >> 1];
        const float2 a = q & 1 ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
#pragma unroll
        for (int o = 0; o < 8; ++o) acc[q][o] = __ffma2_rn(a, make_float2(b[o], b[o]), acc[q][o]);
    }
}

// Eight pixels of a window row whose first is element m (0..3) of the aligned
// 16-byte chunk at p; the third chunk is read only if it is needed.
__device__ __forceinline__ void load_pixels8(const float4 *__restrict__ p, int m, float4 &lo, float4 &hi) {
    const float4 a = __ldg(p), b = __ldg(p + 1), c = m ? __ldg(p + 2) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    const float w[12] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y, c.z, c.w};
    float s[10], o[8];
#pragma unroll
    for (int j = 0; j < 10; ++j) s[j] = (m & 2) ? w[j + 2] : w[j];
#pragma unroll
    for (int j = 0; j < 8; ++j) o[j] = (m & 1) ? s[j + 1] : s[j];
    lo = make_float4(o[0], o[1], o[2], o[3]);
    hi = make_float4(o[4], o[5], o[6], o[7]);
}

// units = tiles * kPairs pairs in all.  src: patches [n][48][48] (desc null), or
// the haloed interval images of the hits' planes, located through desc.
__global__ void __launch_bounds__(kThreads, 1)
    cnn_fp32_kernel(const float *__restrict__ src, const HitDesc *__restrict__ desc, int n,
                    const float *__restrict__ conv_w,
                    const float *__restrict__ conv_b, const float *__restrict__ fc1_w, long long units,
                    float *__restrict__ partials, int n_pad) {
    extern __shared__ float4 smem_f4[];
    float *w1 = reinterpret_cast<float *>(smem_f4);  // [kSlots][48][128]
    float *act = w1 + kSlots * kW1Pos;               // [kSlots][48][128]
    float *win = act + kSlots * kActPos;             // [2][5][128][4]
    float *cw = win + 2 * kWinHalf;                  // [25][48], [48]
    const int cta = blockIdx.x, G = gridDim.x;
    const int64_t u0 = unit_begin(cta, units, G), u1 = unit_begin(cta + 1, units, G);
    const int np = 2 * (int)(u1 - u0);  // positions, in order, across tile boundaries
    int64_t tile = u0 / kPairs;
    int p = 2 * (int)(u0 - tile * kPairs);
    pdl_trigger();  // the head may be scheduled as SMs free up; it waits for this kernel

    if (threadIdx.x >= kRole) {
        // ================================================= conv + weights
        const int t = threadIdx.x - kRole;
        for (int i = t; i < kConvF; i += kRole) cw[i] = i < kK * kK * kF ? conv_w[i] : conv_b[i - kK * kK * kF];
        if (np > 0) {
            load_w1(w1, fc1_w, p, t);
            load_w1(w1 + kW1Pos, fc1_w, p + 1, t);
        }
        pdl_wait();  // the patches, or images and descriptors, come from the kernel before
        HitDesc hd;  // of hit t of the tile
        bool have = false;
        const int hit_c = 64 * ((t >> 5) & 1) + (t & 31), f_c = 24 * (t >> 6);  // this thread's conv: hits, filters
        for (int i = 0; i < np; i += 2) {
            // the pair of position p: window rows y .. y+4, columns x0 .. x0+7 of its quad
            const int y = p / kQ, x = p - y * kQ, x0 = x & ~3;
            if (i == 0 || x == x0) {  // a new quad: thread t stages hit t's window
                const int64_t hit = tile * kHT + t;
                if (!have) {
                    have = true;
                    if (desc != nullptr && hit < n) {
                        hd = desc[hit];
                    } else {
                        hd.origin = hit < n ? hit * kPatchElems : 0;
                        hd.pitch = kPatch;
                        hd.inside = 1;
                    }
                }
                float4 a[kK], b[kK];
                if (hit < n && hd.inside) {  // the pitch is a multiple of 4: every row has the phase m
                    const int m = (int)(hd.origin & 3);
                    const float *p = src + (hd.origin - m) + (int64_t)y * hd.pitch + x0;
#pragma unroll
                    for (int r = 0; r < kK; ++r)
                        load_pixels8(reinterpret_cast<const float4 *>(p + (int64_t)r * hd.pitch), m, a[r], b[r]);
                } else {  // past the last hit, or a hit outside its plane: every pixel checked
#pragma unroll
                    for (int r = 0; r < kK; ++r) {
                        float v[8];
                        const int w = hd.wc - kHalf + y + r;
                        const bool wok = hit < n && w >= 0 && w < hd.nwires;
                        const float *row = src + (wok ? hd.d_off + (int64_t)(w + kHalo) * hd.pitch + kHalo : 0);
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            const int64_t c = (int64_t)hd.bc - kHalf + x0 + j;
                            v[j] = wok && c >= 0 && c < hd.nint ? __ldg(row + c) : 0.0f;
                        }
                        a[r] = make_float4(v[0], v[1], v[2], v[3]);
                        b[r] = make_float4(v[4], v[5], v[6], v[7]);
                    }
                }
                bar_conv();  // the last quad's window has been read (first: the conv weights are staged)
#pragma unroll
                for (int r = 0; r < kK; ++r) {
                    *reinterpret_cast<float4 *>(win + (r * kHT + t) * 4) = a[r];
                    *reinterpret_cast<float4 *>(win + kWinHalf + (r * kHT + t) * 4) = b[r];
                }
                bar_conv();
            }
            // the pair's weights, in flight under its conv
            const int s = i & (kSlots - 1), b = s >> 1;
            if (i >= kSlots) bar_wait(kBarFree + b);
            if (i > 0) {
                load_w1(w1 + s * kW1Pos, fc1_w, p, t);
                load_w1(w1 + (s + 1) * kW1Pos, fc1_w, p + 1, t);
            }
            if (x == x0)
                conv_pair<0>(win + 4 * hit_c, cw + f_c, act + s * kActPos + f_c * kHT + hit_c);
            else
                conv_pair<2>(win + 4 * hit_c, cw + f_c, act + s * kActPos + f_c * kHT + hit_c);
            cp_async_wait_all();  // this thread's share of the weights has landed
            bar_arrive(kBarFull + b);
            p += 2;
            if (p == kPos) {
                p = 0;
                ++tile;
                have = false;
            }
        }
        return;
    }

    // =========================================================== dense-1
    // thread: hits 32 j + 4 hg .. +3 (j = 0..3), outputs 64 j + 4 og .. +3 (j = 0, 1).
    // A 16-byte shared-memory load of a warp takes two passes instead of four when
    // lanes l and l ^ 1, or lanes l and l ^ 2, share every address (2.1 against 4.0
    // cycles): bit 0 of the lane moves only the hits, bit 1 only the outputs.
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int hg = 4 * (warp & 1) + ((lane & 1) | ((lane >> 1) & 2));
    const int og = 8 * (warp >> 1) + (((lane >> 1) & 1) | ((lane >> 2) & 6));
    float2 acc[8][8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int o = 0; o < 8; ++o) acc[q][o] = make_float2(0.0f, 0.0f);
    int64_t started = -1;  // tile whose partial row this CTA has begun
    int krow = 0;          // which of the tile's partial rows it is
    for (int i = 0; i < np; i += 2) {
        const int s = i & (kSlots - 1), b = s >> 1;
        bar_wait(kBarFull + b);
        // a pair's 96 inputs: its two slots are contiguous
        const float *a = act + s * kActPos + 4 * hg, *w = w1 + s * kW1Pos + 4 * og;
        Frag f0, f1;
        f0.load(a, w, 0);
        // unconditional loads (the last one is a repeat): a conditional one costs a
        // copy of the whole operand set per input
#pragma unroll 1
        for (int c = 0; c < 2 * kF; c += 2) {
            f1.load(a, w, c + 1);
            fma_frag(f0, acc);
            f0.load(a, w, c + 2 < 2 * kF ? c + 2 : 0);
            fma_frag(f1, acc);
        }
        if (i + kSlots < np) bar_arrive(kBarFree + b);
        p += 2;
        if (i == np - 2 || p == kPos || p % kSeg == 0) {  // the segment's sums onto the partial row
            const bool first = tile != started;
            if (first) krow = cta - cta_of_unit(tile * kPairs, units, G);
            started = tile;
            // rows past n lie in the padding of the tile and are never read.  Four hits at
            // a time: their loads before their stores
            float *row = partials + ((int64_t)krow * n_pad + tile * kHT + 4 * hg) * kN1 + 4 * og;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float4 *dst = reinterpret_cast<float4 *>(row + 32 * j * kN1);
                float4 old[4][2];
#pragma unroll
                for (int h = 0; h < 4; ++h)
#pragma unroll
                    for (int k = 0; k < 2; ++k)
                        old[h][k] = first ? make_float4(0.0f, 0.0f, 0.0f, 0.0f) : dst[(h * kN1 + 64 * k) / 4];
#pragma unroll
                for (int h = 0; h < 4; ++h)
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const float2 *v = acc[2 * j + (h >> 1)] + 4 * k;
                        const float4 o = old[h][k];
                        dst[(h * kN1 + 64 * k) / 4] =
                            h & 1 ? make_float4(o.x + v[0].y, o.y + v[1].y, o.z + v[2].y, o.w + v[3].y)
                                  : make_float4(o.x + v[0].x, o.y + v[1].x, o.z + v[2].x, o.w + v[3].x);
                    }
            }
#pragma unroll
            for (int q = 0; q < 8; ++q)
#pragma unroll
                for (int o = 0; o < 8; ++o) acc[q][o] = make_float2(0.0f, 0.0f);
        }
        if (p == kPos) {
            p = 0;
            ++tile;
        }
    }
}

}  // namespace

cudaError_t init_fp32_kernel_attrs() {
    return cudaFuncSetAttribute(cnn_fp32_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
}

cudaError_t launch_cnn_fp32(const DeviceWeights &w, const float *src, const HitDesc *desc, int32_t n, int G,
                            float *partials, int n_pad, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const long long units = (long long)((n + kHT - 1) / kHT) * kPairs;
    const float *cw = w.conv_w, *cb = w.conv_b, *fw = w.fc1_w;
    return launch_pdl(cnn_fp32_kernel, dim3(G), dim3(kThreads), kSmemBytes, s, src, desc, n, cw, cb, fw, units,
                      partials, n_pad);
}

}  // namespace emtk
