// Patch extraction (Sec. 2.1): every hit gets a 48x48 patch, rows = wires,
// columns = time intervals of 6 ticks, centred on the hit (row 24 / column
// 24); pixels outside the plane are zero.
//
// Two HBM-friendly passes instead of one gather per hit:
//   1. interval image: each plane's ticks are reduced once to its interval
//      values (fp32 sum of the 6 ticks left to right, one fp32 divide by 6),
//      stored in the patch format.  Reads every plane byte exactly once
//      (16-byte vector loads, streaming), writes 1/6 of it (stays in L2).
//   2. gather: each patch is copied out of the L2-resident interval image.
// Hits of windows that overlap read the same interval values, so the plane
// is never re-read per hit.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "emtk_internal.h"

namespace emtk {
namespace {

__device__ __forceinline__ float interval_sum(float a0, float a1, float a2, float a3, float a4, float a5) {
    // fixed order: ((((a0 + a1) + a2) + a3) + a4) + a5, no contraction possible
    float s = __fadd_rn(a0, a1);
    s = __fadd_rn(s, a2);
    s = __fadd_rn(s, a3);
    s = __fadd_rn(s, a4);
    s = __fadd_rn(s, a5);
    return __fdiv_rn(s, 6.0f);
}

// One pixel of the EMTK_TF32 image: the fp16 head of v * s_p in the low half,
// the fp16 tail (v * s_p - head, rounded) in the high half.  s_p is a power
// of two, so the product is exact.
__device__ __forceinline__ uint32_t split_word(float v) {
    const float x = __fmul_rn(v, kSplitPatchScale);
    const __half h = __float2half_rn(x);
    const __half t = __float2half_rn(__fsub_rn(x, __half2float(h)));
    return (uint32_t)__half_as_ushort(h) | ((uint32_t)__half_as_ushort(t) << 16);
}

template <int FMT>
__device__ __forceinline__ void store2(void *base, int64_t idx, float v0, float v1, bool two) {
    if (FMT == kPatchSplit16) {
        uint32_t *p = static_cast<uint32_t *>(base) + idx;
        if (two) {
            *reinterpret_cast<uint2 *>(p) = make_uint2(split_word(v0), split_word(v1));
        } else {
            p[0] = split_word(v0);
        }
    } else if (FMT == EMTK_PATCH_F32) {
        float *p = static_cast<float *>(base) + idx;
        if (two) {
            *reinterpret_cast<float2 *>(p) = make_float2(v0, v1);
        } else {
            p[0] = v0;
        }
    } else if (FMT == EMTK_PATCH_BF16) {
        __nv_bfloat16 *p = static_cast<__nv_bfloat16 *>(base) + idx;
        if (two) {
            __nv_bfloat162 h;
            h.x = __float2bfloat16_rn(v0);
            h.y = __float2bfloat16_rn(v1);
            *reinterpret_cast<__nv_bfloat162 *>(p) = h;
        } else {
            p[0] = __float2bfloat16_rn(v0);
        }
    } else {
        __half *p = static_cast<__half *>(base) + idx;
        if (two) {
            *reinterpret_cast<__half2 *>(p) = __halves2half2(__float2half_rn(v0), __float2half_rn(v1));
        } else {
            p[0] = __float2half_rn(v0);
        }
    }
}

// One column pair = two consecutive image columns of one image row; inside the
// plane that is two intervals of one wire (12 ticks = 48 bytes, 16-byte
// aligned because ld % 4 == 0, the plane is 16-byte aligned and the halo is
// even), outside it (the zero halo, the pitch padding) zeros.  The image of
// request r, grid-stride over its column pairs along x, kPairsPerStep per thread and
// step with all their loads before the first sum: a plane of 800 wires is then one
// wave of blocks.  The pitch and the image offset are even, so the pair store is
// aligned too.  I: 32-bit pair indices, unless the image has 2^31 pairs or more (a
// 64-bit division per pair showed: with it and one pair per step one APA in three
// calls took 464.8 us, now 461.0; the cut of one plane 19.7, now 19.0).
constexpr int kPairsPerStep = 2;

template <int FMT, class I>
__device__ __forceinline__ void interval_request(const ReqDesc &r, void *img) {
    if (r.nwires == 0) return;
    constexpr int kU = kPairsPerStep;
    const I npairs = (I)(r.pitch >> 1);
    const I work = (I)((int64_t)r.nwires + 2 * r.halo) * npairs;
    const I step = (I)gridDim.x * blockDim.x;
    for (I i0 = (I)blockIdx.x * blockDim.x + threadIdx.x; i0 < work; i0 += kU * step) {
        float4 xa[kU], xd[kU];
        float2 xb[kU], xc[kU];
        bool in0[kU], in1[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const I i = i0 + u * step, wr = i / npairs;
            const int64_t w = (int64_t)wr - r.halo;
            const int b = 2 * (int)(i - wr * npairs) - r.halo;
            in0[u] = i < work && w >= 0 && w < r.nwires && b >= 0 && b < r.nint;
            in1[u] = in0[u] && b + 1 < r.nint;
            const float *src = r.adc + w * r.ld + 6 * b;
            if (in0[u]) {
                xa[u] = __ldcs(reinterpret_cast<const float4 *>(src));
                xb[u] = __ldcs(reinterpret_cast<const float2 *>(src + 4));
            }
            if (in1[u]) {
                xc[u] = __ldcs(reinterpret_cast<const float2 *>(src + 6));
                xd[u] = __ldcs(reinterpret_cast<const float4 *>(src + 8));
            }
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const I i = i0 + u * step;
            if (i >= work) break;
            const float v0 = in0[u] ? interval_sum(xa[u].x, xa[u].y, xa[u].z, xa[u].w, xb[u].x, xb[u].y) : 0.0f;
            const float v1 = in1[u] ? interval_sum(xc[u].x, xc[u].y, xd[u].x, xd[u].y, xd[u].z, xd[u].w) : 0.0f;
            store2<FMT>(img, r.d_off + 2 * (int64_t)i, v0, v1, true);  // rows are npairs pairs apart
        }
    }
}

// grid.y = request.
template <int FMT, class I>
__global__ void __launch_bounds__(256) interval_image_kernel(const __grid_constant__ ReqTable t, void *img) {
    pdl_begin();  // the next kernel may set up while this one runs; it waits for it
    interval_request<FMT, I>(t.r[blockIdx.y], img);
}

constexpr int kGatherThreads = 96;

template <int FMT>
struct Elem;
template <>
struct Elem<EMTK_PATCH_F32> {
    using T = float;
};
template <>
struct Elem<EMTK_PATCH_BF16> {
    using T = unsigned short;
};
template <>
struct Elem<EMTK_PATCH_F16> {
    using T = unsigned short;
};

__device__ __forceinline__ int find_request(const ReqTable &t, int64_t g) {
    int lo = 0, hi = t.n - 1;
    while (lo < hi) {  // last request with hit_begin <= g
        const int mid = (lo + hi + 1) >> 1;
        if (t.r[mid].hit_begin <= g)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int64_t floor_div6(int64_t a) {
    int64_t q = a / 6;
    if ((a % 6) != 0 && a < 0) q -= 1;
    return q;
}

// One block per hit: thread t copies 16-byte chunk t % CH of patch rows t / CH,
// t / CH + RG, ...  A window that lies in the image (halo included) is read with
// aligned 16-byte loads: a chunk of the patch spans two of them, moved down by
// the window's phase (the same for every row: the pitch is a multiple of 8
// elements) with selects and, for an odd 16-bit phase, a funnel shift.  All of a
// thread's loads are issued before its first store, so a block is one round trip
// for the hit and one for the window.  Bound by the L1 (76 % of its rate: two
// loads and a store per chunk); the cut of 7,692 hits of an 800 x 6000 plane in
// fp32 (71 MB written) took 36.9 us with scalar checked reads by 288 threads per
// hit and takes 22.6 us.  Other windows (hits outside the plane; hits near its
// edge when the image has no halo) read every pixel checked.
template <int FMT>
struct Gather {
    using T = typename Elem<FMT>::T;
    static constexpr int V = 16 / sizeof(T);  // elements per chunk
    static constexpr int CH = kPatch / V;     // chunks per patch row: 12 or 6
    static constexpr int RG = kGatherThreads / CH;
    static constexpr int RN = kPatch / RG;    // rows per thread: 6 or 3
    static_assert(kGatherThreads % CH == 0 && kPatch % RG == 0, "whole rows per thread");
};

// Words s .. s + 3 of two consecutive chunks and, if odd, half a word further.
__device__ __forceinline__ uint4 shift_chunk(const uint4 &lo, const uint4 &hi, int s, bool odd) {
    const uint32_t w[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    uint32_t a[6], b[5];
#pragma unroll
    for (int j = 0; j < 6; ++j) a[j] = (s & 2) ? w[j + 2] : w[j];
#pragma unroll
    for (int j = 0; j < 5; ++j) b[j] = (s & 1) ? a[j + 1] : a[j];
    if (!odd) return make_uint4(b[0], b[1], b[2], b[3]);
    return make_uint4(__funnelshift_r(b[0], b[1], 16), __funnelshift_r(b[1], b[2], 16),
                      __funnelshift_r(b[2], b[3], 16), __funnelshift_r(b[3], b[4], 16));
}

template <int FMT>
__global__ void __launch_bounds__(kGatherThreads) gather_kernel(const __grid_constant__ ReqTable t, const void *img,
                                                                void *patches) {
    using G = Gather<FMT>;
    using T = typename G::T;
    pdl_trigger();  // the next kernel may set up while this one runs; it waits for it
    const int64_t g = blockIdx.x;
    const ReqDesc &r = t.r[find_request(t, g)];
    if (r.nwires == 0) pdl_wait();  // no image kernel may stand between this one and what wrote the hits
    const emtk_hit hit = r.hits[g - r.hit_begin];
    const int64_t wc = hit.wire;
    const int64_t bc = floor_div6(hit.tick);
    T *out = static_cast<T *>(patches) + g * kPatchElems;
    const int c = threadIdx.x % G::CH, row0 = threadIdx.x / G::CH;
    pdl_wait();  // the images come from the kernel before
    const T *src = static_cast<const T *>(img) + r.d_off;
    const int64_t w0 = wc - kHalf + r.halo, b0 = bc - kHalf + r.halo;  // the window's first image row, column
    if (r.nwires > 0 && w0 >= 0 && w0 + kPatch <= r.nwires + 2 * (int64_t)r.halo && b0 >= 0 &&
        b0 + kPatch <= r.pitch) {
        const int m = (int)(b0 % G::V);
        const uint4 *p = reinterpret_cast<const uint4 *>(src + (w0 + row0) * r.pitch + (b0 - m)) + c;
        const int64_t step = (int64_t)G::RG * r.pitch / G::V;
        uint4 lo[G::RN], hi[G::RN];
#pragma unroll
        for (int k = 0; k < G::RN; ++k) lo[k] = __ldg(p + k * step);
        if (m != 0) {  // the second chunk holds at least one of the window's elements: it is in the image
#pragma unroll
            for (int k = 0; k < G::RN; ++k) hi[k] = __ldg(p + k * step + 1);
            const int s = m * (int)sizeof(T) / 4;
            const bool odd = sizeof(T) == 2 && (m & 1);
#pragma unroll
            for (int k = 0; k < G::RN; ++k) lo[k] = shift_chunk(lo[k], hi[k], s, odd);
        }
        uint4 *q = reinterpret_cast<uint4 *>(out + row0 * kPatch) + c;
#pragma unroll
        for (int k = 0; k < G::RN; ++k) q[k * G::RG * G::CH] = lo[k];
        return;
    }
    for (int row = row0; row < kPatch; row += G::RG) {
        const int64_t w = wc - kHalf + row;
        union {
            T e[G::V];
            uint4 u;
        } v;
        const bool wire_ok = (w >= 0 && w < r.nwires);
#pragma unroll
        for (int e = 0; e < G::V; ++e) {
            const int64_t b = bc - kHalf + c * G::V + e;
            v.e[e] = (wire_ok && b >= 0 && b < r.nint) ? src[(w + r.halo) * r.pitch + b + r.halo] : T(0);
        }
        *reinterpret_cast<uint4 *>(out + row * kPatch + c * G::V) = v.u;
    }
}

// Pre-cut fp32 patches -> the split-fp16 head / tail words of the EMTK_TF32
// network (emtk_infer_patches; the 16-bit kernels read fp32 patches
// themselves): eight values per thread and step (two 16-byte streaming loads,
// so the dense-1 weights keep their place in L2), four steps in flight; the
// same word per value as the interval images.  n8 = values / 8 (a patch is
// 2,304 values).
__global__ void convert_split_kernel(const float *__restrict__ src, uint4 *__restrict__ dst, int64_t n8) {
    pdl_begin();  // the network kernel may set up while this one runs; it waits for it
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
    const float4 *s4 = reinterpret_cast<const float4 *>(src);
    constexpr int kU = 4;
    for (int64_t base = tid; base < n8; base += nthreads * kU) {
        float4 a[kU], b[kU];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int64_t i = base + u * nthreads;
            if (i < n8) {
                a[u] = __ldcs(s4 + 2 * i);
                b[u] = __ldcs(s4 + 2 * i + 1);
            }
        }
#pragma unroll
        for (int u = 0; u < kU; ++u) {
            const int64_t i = base + u * nthreads;
            if (i >= n8) continue;
            dst[2 * i] = make_uint4(split_word(a[u].x), split_word(a[u].y), split_word(a[u].z), split_word(a[u].w));
            dst[2 * i + 1] =
                make_uint4(split_word(b[u].x), split_word(b[u].y), split_word(b[u].z), split_word(b[u].w));
        }
    }
}

// The window descriptor of hit g0 + local of the table (and its output row).
__device__ __forceinline__ void hit_desc_one(const ReqTable &t, int64_t g0, int64_t local, HitDesc *desc,
                                             float **dest, int out_stride) {
    const int64_t g = g0 + local;
    const ReqDesc &r = t.r[find_request(t, g)];
    const int64_t hloc = g - r.hit_begin;
    const emtk_hit hit = r.hits[hloc];
    const int64_t bc = floor_div6(hit.tick);
    HitDesc d;
    d.wc = hit.wire;
    d.bc = (int32_t)bc;  // |tick| < 2^31, so the interval fits
    d.nwires = r.nwires;
    d.nint = r.nint;
    d.pitch = r.pitch;
    d.d_off = r.d_off;
    // the window [wc-24, wc+24) x [bc-24, bc+24) lies in the haloed image iff
    // the hit itself lies in the plane (the halo is 24 wide)
    d.inside = (hit.wire >= 0 && hit.wire < r.nwires && bc >= 0 && bc < r.nint) ? 1 : 0;
    d.origin = d.inside ? r.d_off + (int64_t)(hit.wire - kHalf + r.halo) * r.pitch + (bc - kHalf + r.halo) : 0;
    desc[local] = d;
    if (dest != nullptr) dest[local] = r.scores + hloc * out_stride;
}

__global__ void hit_desc_kernel(const __grid_constant__ ReqTable t, int64_t g0, int32_t count, HitDesc *desc,
                                float **dest, int out_stride) {
    pdl_begin();
    const int64_t local = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (local < count) hit_desc_one(t, g0, local, desc, dest, out_stride);
}

// The images (grid rows 0 .. t.n - 1) and, in one more grid row, the window
// descriptors of hits g0 .. g0 + count - 1: the descriptors' few bytes ride
// along with the images' stream instead of taking a launch of their own.
template <int FMT, class I>
__global__ void __launch_bounds__(256) interval_desc_kernel(const __grid_constant__ ReqTable t, void *img, int64_t g0,
                                                            int32_t count, HitDesc *desc, float **dest,
                                                            int out_stride) {
    pdl_begin();
    if ((int)blockIdx.y < t.n) {
        interval_request<FMT, I>(t.r[blockIdx.y], img);
        return;
    }
    for (int64_t local = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; local < count;
         local += (int64_t)gridDim.x * blockDim.x)
        hit_desc_one(t, g0, local, desc, dest, out_stride);
}

// The tiles of request r's image that the window of `hit` touches: image rows
// [wire, wire + 47] x image columns [bc, bc + 47] (halo 24), clipped to the
// image; a hit outside its plane marks the part of its window inside the
// image (its in-plane pixels are all there).  The window spans at most 7
// bands and 48 / kTileInts + 1 tile columns, in at most 2 mask words;
// `valid` false marks nothing.
struct WindowTiles {
    int64_t band0;    // first band
    int nbands;       // 0 .. 7
    int w0, nwords;   // first mask word of a band row, 1 or 2
    uint32_t bits[2]; // tile bits in words w0, w0 + 1
};
__device__ __forceinline__ WindowTiles window_tiles(const ReqDesc &r, const emtk_hit &hit, bool valid) {
    WindowTiles wt{0, 0, 0, 0, {0u, 0u}};
    if (!valid) return wt;
    const int64_t rows = (int64_t)r.nwires + 2 * r.halo;
    const int64_t bc = floor_div6(hit.tick);
    const int64_t r0 = hit.wire > 0 ? hit.wire : 0;
    const int64_t r1 = (int64_t)hit.wire + 2 * kHalf - 1 < rows - 1 ? (int64_t)hit.wire + 2 * kHalf - 1 : rows - 1;
    const int64_t c0 = bc > 0 ? bc : 0;
    const int64_t c1 = bc + 2 * kHalf - 1 < r.pitch - 1 ? bc + 2 * kHalf - 1 : (int64_t)r.pitch - 1;
    if (r0 > r1 || c0 > c1) return wt;
    const int t0 = (int)(c0 / kTileInts), t1 = (int)(c1 / kTileInts);
    wt.band0 = r0 / kTileRows;
    wt.nbands = (int)(r1 / kTileRows - wt.band0 + 1);
    wt.w0 = t0 >> 5;
    wt.nwords = (t1 >> 5) - wt.w0 + 1;
    for (int k = 0; k < wt.nwords; ++k) {
        const int wd = wt.w0 + k;
        const int lo = t0 > 32 * wd ? t0 - 32 * wd : 0;
        const int hi = t1 < 32 * wd + 31 ? t1 - 32 * wd : 31;
        wt.bits[k] = (hi == 31 ? 0xffffffffu : ((1u << (hi + 1)) - 1u)) & ~((1u << lo) - 1u);
    }
    return wt;
}

// Every hit of request blockIdx.y marks its window's tiles (one thread per
// hit).  The hits of a block (consecutive in the list: a track or a shower
// of one plane) mostly mark the same few words, and atomics to one word
// serialize in L2, so a block first ORs its marks into a shared-memory copy
// of the plane's mask and then sends each non-zero word once.  A plane whose
// mask is larger than kMarkSmemWords words marks global memory directly.
constexpr int kMarkSmemWords = 8192;  // 32 KB
__global__ void __launch_bounds__(256) mark_tiles_kernel(const __grid_constant__ ReqTable t, uint32_t *mask,
                                                         int smem_words) {
    extern __shared__ uint32_t plane_mask[];
    pdl_begin();  // the tile kernel may be scheduled; it waits for this one
    const ReqDesc &r = t.r[blockIdx.y];
    const int64_t rows = r.nwires > 0 ? (int64_t)r.nwires + 2 * r.halo : 0;
    const int64_t words = (rows + kTileRows - 1) / kTileRows * r.m_wpb;
    const bool local = words <= smem_words;
    if (local) {
        for (int64_t i = threadIdx.x; i < words; i += blockDim.x) plane_mask[i] = 0u;
        __syncthreads();
    }
    uint32_t *dst = local ? plane_mask : mask + r.m_off;
    for (int64_t h = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; h < r.nhits;
         h += (int64_t)gridDim.x * blockDim.x) {
        const WindowTiles wt = window_tiles(r, r.hits[h], r.nwires > 0);
        uint32_t *row0 = dst + wt.band0 * r.m_wpb + wt.w0;
        for (int b = 0; b < wt.nbands; ++b)
            for (int k = 0; k < wt.nwords; ++k) atomicOr(row0 + b * r.m_wpb + k, wt.bits[k]);
    }
    if (local) {
        __syncthreads();
        for (int64_t i = threadIdx.x; i < words; i += blockDim.x)
            if (plane_mask[i]) atomicOr(mask + r.m_off + i, plane_mask[i]);
    }
}

// One warp per tile (kTileRows rows x kTileInts intervals = 8 x 8 column
// pairs) of request blockIdx.y: a tile no window touches is left as it is;
// the others are computed as in interval_request (same sums, same rounding),
// two column pairs per lane with every load issued before the first sum.
// Grid row blockIdx.y == t.n builds the window descriptors and output rows
// of hits [g0, g0 + count).  All threads together clear mask_next for the
// next launch.
constexpr int kTileWarps = 8;
template <int FMT>
__global__ void __launch_bounds__(kTileWarps * 32) interval_tiles_kernel(const __grid_constant__ ReqTable t, void *img,
                                                                         const uint32_t *mask_cur, uint32_t *mask_next,
                                                                         int64_t mask_cap, int64_t g0, int32_t count,
                                                                         HitDesc *desc, float **dest, int out_stride) {
    pdl_trigger();  // the network kernel may set up while this one runs; it waits for it
    const int64_t nthr = (int64_t)gridDim.x * gridDim.y * blockDim.x;
    for (int64_t i = ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x; i < mask_cap;
         i += nthr)
        mask_next[i] = 0u;
    if ((int)blockIdx.y == t.n) {  // the descriptors need nothing from the marking kernel
        for (int64_t local = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; local < count;
             local += (int64_t)gridDim.x * blockDim.x)
            hit_desc_one(t, g0, local, desc, dest, out_stride);
        return;
    }
    pdl_wait();     // the marks come from the kernel before
    const ReqDesc &r = t.r[blockIdx.y];
    if (r.nwires == 0) return;
    const int lane = threadIdx.x & 31;
    const int rows = r.nwires + 2 * r.halo;
    const int npairs = r.pitch >> 1;
    const int nbands = (rows + kTileRows - 1) / kTileRows;
    const int nchunks = (r.pitch + kTileInts - 1) / kTileInts;
    const int64_t tile = (int64_t)blockIdx.x * kTileWarps + (threadIdx.x >> 5);
    if (tile >= (int64_t)nbands * nchunks) return;
    const int band = (int)(tile / nchunks), chunk = (int)(tile - (int64_t)band * nchunks);
    if (((mask_cur[r.m_off + (int64_t)band * r.m_wpb + (chunk >> 5)] >> (chunk & 31)) & 1u) == 0) return;
    constexpr int kPairs = kTileInts / 2;          // column pairs per tile row
    constexpr int kU = kTileRows * kPairs / 32;    // pairs per lane
    float4 xa[kU], xd[kU];
    float2 xb[kU], xc[kU];
    bool in0[kU], in1[kU];
    int64_t dst[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
        const int j = lane + 32 * u;
        const int wr = band * kTileRows + j / kPairs;
        const int cp = chunk * kPairs + j % kPairs;
        const int cb = 2 * cp;
        const int w = wr - r.halo, b = cb - r.halo;
        in0[u] = wr < rows && cp < npairs && w >= 0 && w < r.nwires && b >= 0 && b < r.nint;
        in1[u] = in0[u] && b + 1 < r.nint;
        dst[u] = (wr < rows && cp < npairs) ? r.d_off + (int64_t)wr * r.pitch + cb : -1;
        const float *src = r.adc + (int64_t)w * r.ld + 6 * b;
        if (in0[u]) {
            xa[u] = __ldcs(reinterpret_cast<const float4 *>(src));
            xb[u] = __ldcs(reinterpret_cast<const float2 *>(src + 4));
        }
        if (in1[u]) {
            xc[u] = __ldcs(reinterpret_cast<const float2 *>(src + 6));
            xd[u] = __ldcs(reinterpret_cast<const float4 *>(src + 8));
        }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
        if (dst[u] < 0) continue;
        const float v0 = in0[u] ? interval_sum(xa[u].x, xa[u].y, xa[u].z, xa[u].w, xb[u].x, xb[u].y) : 0.0f;
        const float v1 = in1[u] ? interval_sum(xc[u].x, xc[u].y, xd[u].x, xd[u].y, xd[u].z, xd[u].w) : 0.0f;
        store2<FMT>(img, dst[u], v0, v1, true);
    }
}

template <class I>
auto *image_kernel_for(emtk_patch_format fmt) {
    return fmt == kPatchSplit16     ? interval_image_kernel<kPatchSplit16, I>
           : fmt == EMTK_PATCH_F32  ? interval_image_kernel<EMTK_PATCH_F32, I>
           : fmt == EMTK_PATCH_BF16 ? interval_image_kernel<EMTK_PATCH_BF16, I>
                                    : interval_image_kernel<EMTK_PATCH_F16, I>;
}
template <class I>
auto *desc_kernel_for(emtk_patch_format fmt) {
    return fmt == kPatchSplit16     ? interval_desc_kernel<kPatchSplit16, I>
           : fmt == EMTK_PATCH_F32  ? interval_desc_kernel<EMTK_PATCH_F32, I>
           : fmt == EMTK_PATCH_BF16 ? interval_desc_kernel<EMTK_PATCH_BF16, I>
                                    : interval_desc_kernel<EMTK_PATCH_F16, I>;
}

}  // namespace

cudaError_t launch_interval_images(const ReqTable &t, void *dimg, emtk_patch_format fmt, cudaStream_t s,
                                   const DescJob *job) {
    int64_t most = 0;
    for (int i = 0; i < t.n; ++i) {
        const int64_t w = t.r[i].nwires ? (int64_t)(t.r[i].nwires + 2 * t.r[i].halo) * (t.r[i].pitch / 2) : 0;
        most = w > most ? w : most;
    }
    const bool small = most < (int64_t)1 << 31;
    if (job != nullptr && job->count > 0) {
        if (most == 0 || t.n == 0)  // no image to cut: the descriptors alone
            return launch_hit_desc(t, job->g0, job->count, job->desc, job->dest, job->out_stride, s);
        const int64_t steps = (most + kPairsPerStep - 1) / kPairsPerStep;
        const int64_t want = steps > job->count ? steps : job->count;
        int64_t bx = (want + 255) / 256;
        if (bx > 4096) bx = 4096;
        const dim3 grid((unsigned)bx, (unsigned)t.n + 1);
        auto *kernel = small ? desc_kernel_for<uint32_t>(fmt) : desc_kernel_for<int64_t>(fmt);
        return launch_pdl(kernel, grid, dim3(256), 0, s, t, dimg, job->g0, job->count, job->desc, job->dest,
                          job->out_stride);
    }
    if (most == 0 || t.n == 0) return cudaSuccess;
    int64_t bx = (most + 256 * kPairsPerStep - 1) / (256 * kPairsPerStep);
    if (bx > 4096) bx = 4096;
    auto *kernel = small ? image_kernel_for<uint32_t>(fmt) : image_kernel_for<int64_t>(fmt);
    return launch_pdl(kernel, dim3((unsigned)bx, (unsigned)t.n), dim3(256), 0, s, t, dimg);
}

cudaError_t launch_cut_tiles(const ReqTable &t, int64_t total_hits, void *dimg, emtk_patch_format fmt,
                             const DescJob &job, uint32_t *mask_cur, uint32_t *mask_next, int64_t mask_cap,
                             cudaStream_t s) {
    if (total_hits <= 0 || t.n == 0) return cudaSuccess;
    int64_t most_hits = 0, most_words = 0;
    for (int i = 0; i < t.n; ++i) {
        const ReqDesc &r = t.r[i];
        most_hits = r.nhits > most_hits ? r.nhits : most_hits;
        const int64_t rows = r.nwires > 0 ? (int64_t)r.nwires + 2 * r.halo : 0;
        const int64_t words = (rows + kTileRows - 1) / kTileRows * r.m_wpb;
        most_words = words > most_words ? words : most_words;
    }
    int64_t mb = (most_hits + 255) / 256;
    if (mb > 4096) mb = 4096;
    const int smem_words = (int)(most_words < kMarkSmemWords ? most_words : kMarkSmemWords);
    // not a dependent launch: with one, the tile kernel after it takes 62 us instead of 46 us on the
    // full event (measured, cause unknown), and the launch it would hide is 0.1 % of such a call
    mark_tiles_kernel<<<dim3((unsigned)(mb > 0 ? mb : 1), (unsigned)t.n), 256, (size_t)smem_words * 4, s>>>(
        t, mask_cur, smem_words);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    int64_t most = 0;  // tiles of the largest image
    for (int i = 0; i < t.n; ++i) {
        const ReqDesc &r = t.r[i];
        if (r.nwires == 0) continue;
        const int64_t tiles = (((int64_t)r.nwires + 2 * r.halo + kTileRows - 1) / kTileRows) *
                              ((r.pitch + kTileInts - 1) / kTileInts);
        most = tiles > most ? tiles : most;
    }
    int64_t bx = (most + kTileWarps - 1) / kTileWarps;
    const int64_t desc_blocks = (job.count + kTileWarps * 32 - 1) / (kTileWarps * 32);
    bx = bx > desc_blocks ? bx : desc_blocks;
    bx = bx > 0 ? bx : 1;
    const dim3 grid((unsigned)bx, (unsigned)t.n + 1);  // the last row builds the descriptors
    const uint32_t *mc = mask_cur;
    if (fmt == kPatchSplit16)
        return launch_pdl(interval_tiles_kernel<kPatchSplit16>, grid, dim3(kTileWarps * 32), 0, s, t, dimg, mc,
                          mask_next, mask_cap, job.g0, job.count, job.desc, job.dest, job.out_stride);
    if (fmt == EMTK_PATCH_F16)
        return launch_pdl(interval_tiles_kernel<EMTK_PATCH_F16>, grid, dim3(kTileWarps * 32), 0, s, t, dimg, mc,
                          mask_next, mask_cap, job.g0, job.count, job.desc, job.dest, job.out_stride);
    return launch_pdl(interval_tiles_kernel<EMTK_PATCH_BF16>, grid, dim3(kTileWarps * 32), 0, s, t, dimg, mc,
                      mask_next, mask_cap, job.g0, job.count, job.desc, job.dest, job.out_stride);
}

cudaError_t launch_gather(const ReqTable &t, const void *dimg, emtk_patch_format fmt, int32_t count, void *patches,
                          cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    auto *kernel = fmt == EMTK_PATCH_F32    ? gather_kernel<EMTK_PATCH_F32>
                   : fmt == EMTK_PATCH_BF16 ? gather_kernel<EMTK_PATCH_BF16>
                                            : gather_kernel<EMTK_PATCH_F16>;
    return launch_pdl(kernel, dim3((unsigned)count), dim3(kGatherThreads), 0, s, t, dimg, patches);
}

cudaError_t launch_convert_split(const float *src, void *dst, int64_t n, int sms, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int64_t n8 = n / 8;
    int64_t blocks = (n8 + 256 * 4 - 1) / (256 * 4);
    if (blocks > (int64_t)sms * 8) blocks = (int64_t)sms * 8;
    if (blocks < 1) blocks = 1;
    return launch_pdl(convert_split_kernel, dim3((unsigned)blocks), dim3(256), 0, s, src, static_cast<uint4 *>(dst), n8);
}

cudaError_t launch_hit_desc(const ReqTable &t, int64_t g0, int32_t count, HitDesc *desc, float **dest,
                            int out_stride, cudaStream_t s) {
    if (count <= 0) return cudaSuccess;
    return launch_pdl(hit_desc_kernel, dim3((count + 255) / 256), dim3(256), 0, s, t, g0, count, desc, dest, out_stride);
}

}  // namespace emtk
