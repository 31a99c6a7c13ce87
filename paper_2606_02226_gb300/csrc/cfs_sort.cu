// cfs_sort.cu -- spatial reordering of a stored point cloud.
//
// Streaming a stored cloud through a smooth deformation keeps neighbours
// together (Section 3's staged alternative; the deformation use of Section
// 4): if the cloud is stored in Morton (Z-curve) order of its positions,
// consecutive points splat into neighbouring pixels and the depth layer's
// sectors are reused in L1/L2 instead of being fetched at random.  This file
// sorts a cloud by a Morton key of 10 bits per coordinate with a stable LSD
// radix sort, 10 bits per pass (three passes in 3D, two in 2D).  Stable
// sorting makes the permutation unique: ties keep their original order.
//
// What bounds it and how it is laid out (16.8 M points, 3D, GB300; the whole
// call went from 2.08 to 0.85 ms):
//  - The final gather reads every point at a random place.  From the SoA
//    arrays that is four sectors in four lines per point, 4.3 GB of DRAM
//    traffic, 780 us.  The key pass, which reads the cloud anyway, therefore
//    also writes it as 16-byte records, so that the gather touches one line
//    per point.
//  - A pass ranks a tile of 8192 keys with warp ballots (ten per key, against
//    the match instruction's unit, which was the limit at 8 bits a pass) and
//    per-warp counters; the tile's keys go through shared memory in sorted
//    order, so that writes leave in runs.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "cfs_device.cuh"
#include "cfs_internal.h"

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kItems = 16;                    // keys per thread per tile
constexpr int kTile = kThreads * kItems;      // 8192 keys per tile
constexpr int kBits = 10;
constexpr int kRadix = 1 << kBits;

// float <-> order-preserving unsigned
__device__ __forceinline__ u32 f2o(float f)
{
    const u32 u = __float_as_uint(f);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float o2f(u32 o)
{
    return __uint_as_float((o & 0x80000000u) ? (o & 0x7FFFFFFFu) : ~o);
}

// box[0..2]: smallest coordinate (ordered bits), box[3..5]: complement of the
// largest; both start at all ones.  NaNs are skipped.
__global__ void __launch_bounds__(kThreads) bbox_kernel(const float* __restrict__ xyz, u32 n,
                                                        int dim, u32* box)
{
    __shared__ u32 s_lo[kWarps], s_hi[kWarps];
    const size_t i0 = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    for (int d = 0; d < dim; ++d) {
        const float* row = xyz + (size_t)d * n;
        u32 lo = 0xFFFFFFFFu, hi = 0xFFFFFFFFu;
        auto take = [&](float v) {
            if (v == v) {
                lo = min(lo, f2o(v));
                hi = min(hi, ~f2o(v));
            }
        };
        auto take4 = [&](float4 v) { take(v.x); take(v.y); take(v.z); take(v.w); };
        // scalars up to the row's first 16-byte boundary and after its last
        // whole vector; two vectors in flight per thread (scalar loads, four
        // in flight, ran at 1.6 TB/s)
        const size_t head = min((size_t)n, (size_t)((4u - (u32)((uintptr_t)row >> 2 & 3u)) & 3u));
        const size_t vecs = (n - head) / 4;
        const float4* v4 = reinterpret_cast<const float4*>(row + head);
        size_t i = i0;
        for (; i + 3 * stride < vecs; i += 4 * stride) {
            const float4 a = v4[i], b = v4[i + stride], c = v4[i + 2 * stride],
                         e = v4[i + 3 * stride];
            take4(a); take4(b); take4(c); take4(e);
        }
        for (; i < vecs; i += stride) take4(v4[i]);
        if (i0 < head) take(row[i0]);
        if (i0 < n - head - 4 * vecs) take(row[head + 4 * vecs + i0]);
        lo = __reduce_min_sync(0xffffffffu, lo);
        hi = __reduce_min_sync(0xffffffffu, hi);
        __syncthreads();                // the previous row's sums have been read
        if ((threadIdx.x & 31) == 0) {
            s_lo[threadIdx.x >> 5] = lo;
            s_hi[threadIdx.x >> 5] = hi;
        }
        __syncthreads();
        if (threadIdx.x < 32) {
            lo = threadIdx.x < kWarps ? s_lo[threadIdx.x] : 0xFFFFFFFFu;
            hi = threadIdx.x < kWarps ? s_hi[threadIdx.x] : 0xFFFFFFFFu;
            lo = __reduce_min_sync(0xffffffffu, lo);
            hi = __reduce_min_sync(0xffffffffu, hi);
            if (threadIdx.x == 0) {
                atomicMin(box + d, lo);
                atomicMin(box + 3 + d, hi);
            }
        }
    }
}

__device__ __forceinline__ u32 spread10(u32 v)
{
    v &= 0x3FFu;
    v = (v | (v << 16)) & 0x030000FFu;
    v = (v | (v << 8)) & 0x0300F00Fu;
    v = (v | (v << 4)) & 0x030C30C3u;
    v = (v | (v << 2)) & 0x09249249u;
    return v;
}

__device__ __forceinline__ u32 spread10_2(u32 v)
{
    v &= 0x3FFu;
    v = (v | (v << 8)) & 0x00FF00FFu;
    v = (v | (v << 4)) & 0x0F0F0F0Fu;
    v = (v | (v << 2)) & 0x33333333u;
    v = (v | (v << 1)) & 0x55555555u;
    return v;
}

// a tile's digit counts to its row of hist [n_tiles][kRadix] (cnt complete
// after the caller's barrier)
__device__ __forceinline__ void store_counts(const u32* cnt, u32* hist)
{
    for (int d = threadIdx.x; d < kRadix; d += kThreads)
        hist[(size_t)blockIdx.x * kRadix + d] = cnt[d];
}

// Morton key: each coordinate quantized to 10 bits over the box,
// q = min(1023, (int)((v - lo) * (1024 / (hi - lo)))) in FP32 (no
// contraction), bits interleaved x lowest.  Non-finite coordinates map to 0.
// Also the first pass's digit counts and, with `pack`, the points as records
// (x, y, z or 0, map index).
template <int DIM>
__global__ void __launch_bounds__(kThreads) key_kernel(const float* __restrict__ xyz,
                                                       const unsigned char* __restrict__ fn, u32 n,
                                                       const u32* box, u32* keys, uint4* pack,
                                                       u32* hist)
{
    __shared__ u32 cnt[kRadix];
    __shared__ float s_lo[3], s_scale[3];
    for (int d = threadIdx.x; d < kRadix; d += kThreads) cnt[d] = 0;
    if (threadIdx.x < DIM) {
        const float lo = o2f(box[threadIdx.x]), hi = o2f(~box[3 + threadIdx.x]);
        const float ext = hi - lo;
        s_lo[threadIdx.x] = lo;
        s_scale[threadIdx.x] = ext > 0.0f ? 1024.0f / ext : 0.0f;
    }
    __syncthreads();
    const size_t base = (size_t)blockIdx.x * kTile;
    const u32 here = (u32)min((size_t)kTile, (size_t)n - base);
#pragma unroll 4
    for (int q = 0; q < kItems; ++q) {
        const u32 t = (u32)q * kThreads + threadIdx.x;
        if (t >= here) break;
        const size_t i = base + t;
        u32 key = 0;
        float v[3] = {0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int d = 0; d < DIM; ++d) {
            v[d] = xyz[(size_t)d * n + i];
            const float u = __fmul_rn(__fsub_rn(v[d], s_lo[d]), s_scale[d]);
            const u32 c = (u >= 0.0f) ? (u32)min((int)u, 1023) : 0u;   // NaN fails the test
            key |= (DIM == 3 ? spread10(c) : spread10_2(c)) << d;
        }
        keys[i] = key;
        if (pack)
            pack[i] = make_uint4(__float_as_uint(v[0]), __float_as_uint(v[1]),
                                 __float_as_uint(v[2]), (u32)fn[i]);
        atomicAdd(&cnt[key & (kRadix - 1)], 1u);
    }
    __syncthreads();
    store_counts(cnt, hist);
}

// digit counts per tile of a later pass
__global__ void __launch_bounds__(kThreads) hist_kernel(const u32* __restrict__ keys, u32 n,
                                                        int shift, u32* hist)
{
    __shared__ u32 cnt[kRadix];
    for (int d = threadIdx.x; d < kRadix; d += kThreads) cnt[d] = 0;
    __syncthreads();
    const size_t base = (size_t)blockIdx.x * kTile;
    const u32 here = (u32)min((size_t)kTile, (size_t)n - base);
    u32 k[kItems];
#pragma unroll
    for (int q = 0; q < kItems; ++q) {
        const u32 t = (u32)q * kThreads + threadIdx.x;
        k[q] = t < here ? keys[base + t] : 0u;
    }
#pragma unroll
    for (int q = 0; q < kItems; ++q)
        if ((u32)q * kThreads + threadIdx.x < here)
            atomicAdd(&cnt[(k[q] >> shift) & (kRadix - 1)], 1u);
    __syncthreads();
    store_counts(cnt, hist);
}

// Per digit: exclusive sums of the counts over the tiles, in place, and the
// digit's total.  A block takes 8 digits (32-byte rows, so that 128 blocks
// share the work); a warp's lanes are four tiles by eight digits, its warps
// take consecutive runs of tiles, which they read twice.
constexpr int kScanThreads = 1024;
constexpr int kScanDigits = 8;
__global__ void __launch_bounds__(kScanThreads) tile_scan_kernel(u32* hist, u32 n_tiles, u32* total)
{
    constexpr u32 W = kScanThreads / kScanDigits;        // runs of tiles
    __shared__ u32 sums[W][kScanDigits];
    const u32 d = threadIdx.x % kScanDigits, run = threadIdx.x / kScanDigits;
    const u32 per = (n_tiles + W - 1) / W;
    const u32 t0 = min((size_t)n_tiles, (size_t)run * per), t1 = min(n_tiles, t0 + per);
    u32* col = hist + blockIdx.x * kScanDigits + d;
    u32 s = 0;
#pragma unroll 8
    for (u32 t = t0; t < t1; ++t) s += col[(size_t)t * kRadix];
    sums[run][d] = s;
    __syncthreads();
    u32 before = 0, all = 0;
#pragma unroll 8
    for (u32 w = 0; w < W; ++w) {
        const u32 v = sums[w][d];
        before += w < run ? v : 0u;
        all += v;
    }
    if (run == 0) total[blockIdx.x * kScanDigits + d] = all;
#pragma unroll 8
    for (u32 t = t0; t < t1; ++t) {
        const u32 v = col[(size_t)t * kRadix];
        col[(size_t)t * kRadix] = before;
        before += v;
    }
}

// exclusive sums of kRadix values v[d] in shared memory, in place (two per
// thread; all threads, barriers inside)
__device__ __forceinline__ void scan_digits(u32* v, u32* s_warp)
{
    static_assert(kRadix == 2 * kThreads, "two digits per thread");
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const u32 a = v[2 * threadIdx.x], b = v[2 * threadIdx.x + 1];
    u32 s = a + b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u32 t = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += t;
    }
    if (lane == 31) s_warp[warp] = s;
    __syncthreads();
    u32 before = 0;
    for (int w = 0; w < warp; ++w) before += s_warp[w];
    v[2 * threadIdx.x] = before + s - a - b;
    v[2 * threadIdx.x + 1] = before + s - b;
    __syncthreads();
}

// shared memory of a sorting pass
struct PassSmem {
    u32 key[kTile], val[kTile];                     // the tile in sorted order
    unsigned short cnt[kWarps][kRadix];             // per warp and digit
    u32 start[kRadix];                              // first place of a digit in the tile
    u32 dest[kRadix];                               // its global place less `start`
    u32 warp[kWarps];
};

// One stable pass over a tile; vin == null: the value is the index i itself;
// kout == null (the last pass): only the values are wanted.  (Moving 16-byte
// records with the keys instead of indices, to save the random gather: their
// scattered half-sector stores made a pass 370 instead of 122 us.)
__global__ void __launch_bounds__(kThreads, 2) pass_kernel(const u32* __restrict__ kin,
                                                           const u32* __restrict__ vin, u32 n,
                                                           int shift, const u32* __restrict__ offs,
                                                           const u32* __restrict__ total,
                                                           u32* kout, u32* vout)
{
    extern __shared__ __align__(16) unsigned char raw[];
    PassSmem& sm = *reinterpret_cast<PassSmem*>(raw);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const size_t base = (size_t)blockIdx.x * kTile;
    const u32 here = (u32)min((size_t)kTile, (size_t)n - base);
    // a warp's keys are consecutive, 32 at a time
    const u32 first = (u32)warp * (32 * kItems) + lane;
    u32 k[kItems];
#pragma unroll
    for (int q = 0; q < kItems; ++q) {
        const u32 t = first + 32 * q;
        k[q] = t < here ? kin[base + t] : 0xFFFFFFFFu;     // past the end: the last digit
    }
    // the digits' global starts while the keys arrive
    for (int d = threadIdx.x; d < kRadix; d += kThreads) sm.dest[d] = total[d];
    u32* c32 = reinterpret_cast<u32*>(&sm.cnt[0][0]);
    for (int e = threadIdx.x; e < kWarps * kRadix / 2; e += kThreads) c32[e] = 0u;
    __syncthreads();
    scan_digits(sm.dest, sm.warp);
    // rank among the warp's equal digits, in the high half of a word whose
    // low half keeps the digit
    u32 at[kItems];
    const u32 lt = (1u << lane) - 1u;
#pragma unroll
    for (int q = 0; q < kItems; ++q) {
        const u32 d = (k[q] >> shift) & (kRadix - 1);
        u32 peers = 0xFFFFFFFFu;
#pragma unroll
        for (int b = 0; b < kBits; ++b) {
            const bool bit = (d >> b) & 1u;
            const u32 with = __ballot_sync(0xffffffffu, bit);
            peers &= bit ? with : ~with;
        }
        const u32 old = sm.cnt[warp][d];
        const u32 below = __popc(peers & lt);
        at[q] = (old + below) << 16 | d;
        __syncwarp();
        if (below == 0) sm.cnt[warp][d] = (unsigned short)(old + __popc(peers));
        __syncwarp();
    }
    __syncthreads();
    // per digit: exclusive sums over the warps, and the tile's total
    for (int d = threadIdx.x; d < kRadix; d += kThreads) {
        u32 acc = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) {
            const u32 v = sm.cnt[w][d];
            sm.cnt[w][d] = (unsigned short)acc;
            acc += v;
        }
        sm.start[d] = acc;
    }
    __syncthreads();
    scan_digits(sm.start, sm.warp);
    for (int d = threadIdx.x; d < kRadix; d += kThreads)
        sm.dest[d] += offs[(size_t)blockIdx.x * kRadix + d] - sm.start[d];
#pragma unroll
    for (int q = 0; q < kItems; ++q) {
        const u32 d = at[q] & 0xFFFFu;
        at[q] = sm.start[d] + sm.cnt[warp][d] + (at[q] >> 16);
        sm.key[at[q]] = k[q];
    }
    if (vin) {
#pragma unroll
        for (int q = 0; q < kItems; ++q) {
            const u32 t = first + 32 * q;
            sm.val[at[q]] = t < here ? vin[base + t] : 0u;
        }
    } else {
#pragma unroll
        for (int q = 0; q < kItems; ++q) sm.val[at[q]] = (u32)base + first + 32 * q;
    }
    __syncthreads();
    // (the keys past the end came last: places here .. kTile - 1)
#pragma unroll 4
    for (int q = 0; q < kItems; ++q) {
        const u32 p = (u32)q * kThreads + threadIdx.x;
        if (p >= here) break;
        const u32 key = sm.key[p];
        const u32 dst = sm.dest[(key >> shift) & (kRadix - 1)] + p;
        if (kout) kout[dst] = key;
        vout[dst] = sm.val[p];
    }
}

// The points in sorted order, from packed records or from the SoA arrays.
// (One plain 16-byte load per point; streaming hints made it 25% slower, and
// gathering in the last sorting pass, at its occupancy, 633 against 390 us
// for both.)
template <int DIM>
__global__ void __launch_bounds__(256) gather_kernel(const uint4* __restrict__ pack,
                                                     const float* __restrict__ xyz,
                                                     const unsigned char* __restrict__ fn,
                                                     const u32* __restrict__ perm, u32 n,
                                                     float* xyz_out, unsigned char* fn_out)
{
    const size_t j = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const u32 i = perm[j];
    if (pack) {
        const uint4 r = pack[i];
        const u32 v[3] = {r.x, r.y, r.z};
#pragma unroll
        for (int d = 0; d < DIM; ++d) xyz_out[(size_t)d * n + j] = __uint_as_float(v[d]);
        fn_out[j] = (unsigned char)r.w;
    } else {
#pragma unroll
        for (int d = 0; d < DIM; ++d) xyz_out[(size_t)d * n + j] = xyz[(size_t)d * n + i];
        fn_out[j] = fn[i];
    }
}

// scratch, 16-byte aligned parts: box and totals | counts | records | keys
// and indices of one pass [2][n] | the permutation, unless the caller takes it
struct Layout {
    size_t hist, pack, kv, perm, bytes;
};

Layout layout(u32 n, bool packed, bool own_perm)
{
    const size_t n_tiles = ((size_t)n + kTile - 1) / kTile;
    Layout l;
    l.hist = 256 + 4 * (size_t)kRadix;
    l.pack = l.hist + 4 * (size_t)kRadix * n_tiles;
    l.kv = l.pack + (packed ? 16 * (size_t)n : 0);
    l.perm = l.kv + 8 * (size_t)n;
    l.bytes = l.perm + (own_perm ? 4 * (size_t)n : 0);
    return l;
}

template <int DIM>
cudaError_t reorder(const float* xyz, const unsigned char* fn, u32 n, float* xyz_out,
                    unsigned char* fn_out, u32* perm_out, unsigned char* ws, bool packed,
                    cudaStream_t s)
{
    const u32 n_tiles = (u32)(((size_t)n + kTile - 1) / kTile);
    const Layout l = layout(n, packed, perm_out == nullptr);
    u32* box = reinterpret_cast<u32*>(ws);
    u32* total = box + 64;
    u32* hist = reinterpret_cast<u32*>(ws + l.hist);
    u32* kv = reinterpret_cast<u32*>(ws + l.kv);
    u32* perm = perm_out ? perm_out : reinterpret_cast<u32*>(ws + l.perm);
    uint4* pack = packed ? reinterpret_cast<uint4*>(ws + l.pack) : nullptr;
    // xyz_out, written last, holds the keys and indices of one pass until
    // then: in 3D kv -> xyz_out -> kv -> permutation, in 2D xyz_out -> kv ->
    // permutation
    u32* xo = reinterpret_cast<u32*>(xyz_out);
    u32* k0 = DIM == 3 ? kv : xo;
    cudaError_t e = cudaMemsetAsync(box, 0xFF, 24, s);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(pass_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(PassSmem));
    if (e != cudaSuccess) return e;
    const u32 sms = (u32)std::max(1, cfs::device_sm_count());
    bbox_kernel<<<std::min((n - 1) / kThreads + 1, sms * 4u), kThreads, 0, s>>>(xyz, n, DIM, box);
    key_kernel<DIM><<<n_tiles, kThreads, 0, s>>>(xyz, fn, n, box, k0, pack, hist);
    const u32 *kin = k0, *vin = nullptr;
    constexpr int passes = DIM == 3 ? 3 : 2;                // 30 or 20 key bits
    for (int p = 0; p < passes; ++p) {
        const int shift = kBits * p;
        const bool last = p == passes - 1;
        if (p > 0) hist_kernel<<<n_tiles, kThreads, 0, s>>>(kin, n, shift, hist);
        tile_scan_kernel<<<kRadix / kScanDigits, kScanThreads, 0, s>>>(hist, n_tiles, total);
        u32* to = (DIM == 3 && p == 0) ? xo : kv;
        u32* ko = last ? nullptr : to;
        u32* vo = last ? perm : to + n;
        pass_kernel<<<n_tiles, kThreads, sizeof(PassSmem), s>>>(kin, vin, n, shift, hist, total, ko,
                                                                vo);
        kin = ko;
        vin = vo;
    }
    gather_kernel<DIM><<<(n - 1) / 256 + 1, 256, 0, s>>>(pack, xyz, fn, perm, n, xyz_out, fn_out);
    return cudaGetLastError();
}

}  // namespace

extern "C" cfs_status cfs_pointcloud_reorder(const float* xyz, const uint8_t* fn, uint32_t n,
                                             int dim, float* xyz_out, uint8_t* fn_out,
                                             uint32_t* perm_out, void* stream_)
{
    using cfs::check_cuda;
    using cfs::fail;
    cfs::clear_error();
    if (n == 0) return CFS_OK;
    if (dim != 2 && dim != 3) return fail(CFS_ERR_INVALID_ARG, "dim must be 2 or 3");
    if (!xyz || !fn || !xyz_out || !fn_out)
        return fail(CFS_ERR_INVALID_ARG, "NULL cloud pointer");
    if (xyz_out == xyz || fn_out == fn)
        return fail(CFS_ERR_INVALID_ARG, "the reorder cannot run in place");
    cudaStream_t s = (cudaStream_t)stream_;
    // with the points as records, or, where that much memory is not to be
    // had, gathering from the SoA arrays
    unsigned char* ws = nullptr;
    bool packed = true;
    cudaError_t e = cudaMallocAsync((void**)&ws, layout(n, true, perm_out == nullptr).bytes, s);
    if (e == cudaErrorMemoryAllocation) {
        (void)cudaGetLastError();
        packed = false;
        e = cudaMallocAsync((void**)&ws, layout(n, false, perm_out == nullptr).bytes, s);
    }
    if (e != cudaSuccess) return check_cuda(e, "cudaMallocAsync");
    e = dim == 3 ? reorder<3>(xyz, fn, n, xyz_out, fn_out, perm_out, ws, packed, s)
                 : reorder<2>(xyz, fn, n, xyz_out, fn_out, perm_out, ws, packed, s);
    const cudaError_t e2 = cudaFreeAsync(ws, s);
    if (e != cudaSuccess) return check_cuda(e, "cloud reorder");
    return check_cuda(e2, "cudaFreeAsync");
}
