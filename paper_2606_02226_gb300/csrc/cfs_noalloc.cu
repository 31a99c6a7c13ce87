// cfs_noalloc.cu -- batched histogram rendering that allocates nothing.
//
// Some callers cannot allocate device memory while they render: a
// real-time or embedded host whose memory budget is fixed after start-up
// (an allocation can fail or stall a frame), or a process whose GPU memory
// is handed out by another allocator that owns the device's free memory.
// cfs_render_batch needs a per-batch workspace (frame descriptors, a work
// counter, discard counters) and gets it with cudaMalloc; this variant keeps
// that workspace in one file-scope device array instead, sized for at most
// CFS_NOALLOC_MAX_FRAMES frames.  The caller still passes every input and
// output (systems, targets).
//
// The array lives as long as the library is loaded, on every GPU that
// loads it, and all calls share it: calls whose GPU work overlaps (two
// streams, or two host threads) race on it.  Everything that must start
// at zero (work counter, discard counters) is cleared on the stream at the
// start of every call.
//
// A call is four kinds of launches: the frame descriptors travel as kernel
// arguments (kUpload frames each), one kernel clears every histogram, one
// places the frames' privatized windows (one CTA per frame), and the
// persistent renderer draws work items.  The renderer is the windowed batch
// renderer of the generated programs (cfs_window.cuh) with the channel count
// read at run time: before it, every splat was a global reduction and 24
// frames of 2^12..2^17 points x 150 steps took 1.93 ms of kernel time at 14%
// of the issue slots, held up by reductions to the same few pixels.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstring>
#include <mutex>

#include "cfs_device.cuh"
#include "cfs_internal.h"

namespace {

constexpr int kMaxFrames = CFS_NOALLOC_MAX_FRAMES;
constexpr int kBlock = CFS_WIN_THREADS;
// shared counters of the windows (208 KB): with the tables that leaves one
// CTA per SM
constexpr uint32_t kCounters = 53248;

struct NaTarget {
    unsigned long long data;
    int W, H, C, pad;
    float x0, x1, y0, y1, sx, sy;
};

struct NaFrame {
    u32 T[16];
    int n_cmp;
    u32 n_points, point_begin, system_id;
    u32 item_begin, pad0, pad1, pad2;
    float prm[6][16];               // a b c d e f of every map, SoA
    NaTarget tg;
};

struct NaScratch {
    NaFrame frames[kMaxFrames];
    int4 box[kMaxFrames][16];       // the windows' pixel boxes, per channel
    unsigned int counter;
    unsigned int pad[63];
    unsigned long long discards[kMaxFrames];
};

// the workspace: one per GPU that loads the library, shared by every call
static __device__ __align__(256) unsigned char g_noalloc_scratch[sizeof(NaScratch)];

// frames whose descriptors one launch carries in its argument block (at most
// 32764 bytes)
constexpr int kUpload = 48;
struct NaUpload {
    NaScratch* ws;
    u32 first, count, reset, pad;   // reset: also zero the counters
    NaFrame f[kUpload];
};
static_assert(sizeof(NaUpload) <= 32764, "kernel argument block");

__global__ void __launch_bounds__(256) noalloc_upload_kernel(const __grid_constant__ NaUpload u)
{
    constexpr u32 kWords = sizeof(NaFrame) / 4;
    const u32* src = reinterpret_cast<const u32*>(u.f);
    u32* dst = reinterpret_cast<u32*>(u.ws->frames + u.first);
    for (u32 e = blockIdx.x * blockDim.x + threadIdx.x; e < u.count * kWords;
         e += gridDim.x * blockDim.x)
        dst[e] = src[e];
    if (u.reset && blockIdx.x == 0) {
        if (threadIdx.x == 0) u.ws->counter = 0u;
        for (int f = threadIdx.x; f < kMaxFrames; f += blockDim.x) u.ws->discards[f] = 0ull;
    }
}

// zeroes every frame's histogram: block (x, f) a slice of frame f's words
__global__ void __launch_bounds__(256) noalloc_clear_kernel(const NaScratch* ws)
{
    const NaTarget& t = ws->frames[blockIdx.y].tg;
    const size_t n = (size_t)t.W * (size_t)t.H * (size_t)t.C;
    u32* p = reinterpret_cast<u32*>(t.data);
    // words up to the first 16-byte boundary, whole vectors, the rest
    const size_t head = min(n, (size_t)((4u - (u32)((t.data >> 2) & 3u)) & 3u));
    const size_t vecs = (n - head) / 4;
    const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t stride = (size_t)gridDim.x * blockDim.x;
    uint4* v = reinterpret_cast<uint4*>(p + head);
    for (size_t e = i; e < vecs; e += stride) v[e] = make_uint4(0u, 0u, 0u, 0u);
    if (i < head) p[i] = 0u;
    const size_t tail = head + 4 * vecs;
    if (i < n - tail) p[tail + i] = 0u;
}

struct NaArgs {
    unsigned int rk[10][2];
    u32 iters, burn_in, n_frames, n_items, chunk, pad;
    NaScratch* ws;
};

// the frame's tables in shared memory
struct NaTables {
    float4 abcd[16];
    float2 ef[16];
    u32 T[16];
    int n_cmp;
    u32 n_points, point_begin, system_id, item_begin;
};

__device__ __forceinline__ void load_tables(const NaFrame& f, NaTables& t, cfs_dev_target& tg)
{
    const int k = threadIdx.x;
    if (k < 16) {
        t.abcd[k] = make_float4(f.prm[0][k], f.prm[1][k], f.prm[2][k], f.prm[3][k]);
        t.ef[k] = make_float2(f.prm[4][k], f.prm[5][k]);
        t.T[k] = f.T[k];
    }
    if (k == 16) {
        t.n_cmp = f.n_cmp;
        t.n_points = f.n_points;
        t.point_begin = f.point_begin;
        t.system_id = f.system_id;
        t.item_begin = f.item_begin;
        tg.data = f.tg.data;
        tg.W = f.tg.W; tg.H = f.tg.H; tg.C = f.tg.C;
        tg.x0 = f.tg.x0; tg.x1 = f.tg.x1; tg.y0 = f.tg.y0; tg.y1 = f.tg.y1;
        tg.sx = f.tg.sx; tg.sy = f.tg.sy;
    }
}

__device__ __forceinline__ void apply_map(const NaTables& t, int k, float& x, float& y)
{
    const float4 m = t.abcd[k];
    const float2 e = t.ef[k];
    cfs_affine2(m.x, m.y, m.z, m.w, e.x, e.y, x, y);
}

__device__ __forceinline__ void start_point(const NaArgs& a, u32 i, u32 sid, float& x, float& y)
{
    const uint4 r = cfs_philox_rk(a.rk, i, 0u, sid, 1u);
    x = (float)(r.x >> 8) * CFS_INV_2_24;
    y = (float)(r.y >> 8) * CFS_INV_2_24;
}

__global__ void __launch_bounds__(kBlock) noalloc_place_kernel(const __grid_constant__ NaArgs a)
{
    extern __shared__ u32 s_samples[];
    __shared__ NaTables tab;
    __shared__ cfs_dev_target tg;
    __shared__ CfsPlace place;
    __shared__ CfsKtab kt;
    load_tables(a.ws->frames[blockIdx.x], tab, tg);
    __syncthreads();
    cfs_build_ktab(tab.T, tab.n_cmp, kt);
    __syncthreads();
    const CfsChooseKtab<true> choose{kt, kt.more};
    const int C = tg.C;
    cfs_place_windows(tg, C, kCounters, place, s_samples,
                      reinterpret_cast<unsigned char*>(s_samples + CFS_WIN_SAMPLES * blockDim.x),
                      a.ws->box[blockIdx.x], [&](auto emit) {
        const u32 j = threadIdx.x;
        if (j >= tab.n_points) return;
        const u32 i = tab.point_begin + j, sid = tab.system_id;
        float x, y;
        start_point(a, i, sid, x, y);
        const CfsStream ps = cfs_stream(a.rk, i, sid);
        // (burn_in <= iters < 2^32 - 32 or the sum is cut at iters)
        const u32 n1 = a.iters - a.burn_in > (u32)CFS_WIN_SAMPLES ? a.burn_in + CFS_WIN_SAMPLES
                                                                  : a.iters;
#pragma unroll 1
        for (u32 nb = 0; 4u * nb < n1; ++nb) {
            uint4 r = cfs_stream_block(a.rk, ps, nb, sid);
#pragma unroll 1
            for (u32 n = 4u * nb; n < min(n1, 4u * nb + 4u); ++n) {
                const int k = choose(r.x);
                r = make_uint4(r.y, r.z, r.w, 0u);
                apply_map(tab, k, x, y);
                if (n < a.burn_in) continue;
                const int ix = cfs_bin(x, tg.x0, tg.x1, tg.sx, tg.W);
                const int iy = cfs_bin(y, tg.y0, tg.y1, tg.sy, tg.H);
                if (ix >= 0 && iy >= 0) emit(ix, iy, k % C);
            }
        }
    });
}

__global__ void __launch_bounds__(kBlock, 1) noalloc_batch_kernel(const __grid_constant__ NaArgs a)
{
    extern __shared__ u32 s_cnt[];
    __shared__ NaTables tab;
    __shared__ cfs_dev_target tg;
    __shared__ CfsKtab kt;
    __shared__ int4 win[16];                // per channel (cfs_pack_windows)
    __shared__ int4 mapwin[16];             // per map (CfsTile)
    __shared__ u32 maprow[16];
    __shared__ u32 s_item, s_frame;
    const CfsTile tile{mapwin, maprow, &tg};
    for (u32 e = threadIdx.x; e < kCounters; e += blockDim.x) s_cnt[e] = 0u;
    NaScratch* ws = a.ws;
    int cur = -1;
    u32 disc = 0;
    CfsBinTarget bt = {};
    auto leave_frame = [&]() {
        const u32 s = __reduce_add_sync(0xffffffffu, disc);
        if ((threadIdx.x & 31) == 0 && s) atomicAdd(&ws->discards[cur], (u64)s);
        disc = 0;
        cfs_flush_tile(tg, s_cnt, win, tg.C);
    };
    for (;;) {
        if (threadIdx.x == 0) {
            const u32 item = atomicAdd(&ws->counter, 1u);
            u32 lo = 0;
            if (item < a.n_items) {
                u32 hi = a.n_frames;
                while (hi - lo > 1) {
                    const u32 mid = (lo + hi) >> 1;
                    if (ws->frames[mid].item_begin <= item) lo = mid; else hi = mid;
                }
            }
            s_item = item;
            s_frame = lo;
        }
        __syncthreads();
        const u32 item = s_item;
        if (item >= a.n_items) break;
        const int f = (int)s_frame;
        if (f != cur) {
            if (cur >= 0) leave_frame();
            __syncthreads();
            load_tables(ws->frames[f], tab, tg);
            if (threadIdx.x == 32)
                cfs_pack_windows(ws->box[f], ws->frames[f].tg.C, kCounters, false, win);
            __syncthreads();
            cfs_build_ktab(tab.T, tab.n_cmp, kt);
            if (threadIdx.x < 16) {
                const int c = (int)threadIdx.x % tg.C;
                mapwin[threadIdx.x] = cfs_win_record(win[c], s_cnt);
                maprow[threadIdx.x] = (u32)(c * tg.H) - CFS_BIN_MAGIC;
            }
            bt = cfs_bin_target(tg);
            __syncthreads();
            cur = f;
        }
        const u32 j0 = (item - tab.item_begin) * a.chunk;
        const u32 n_here = min(a.chunk, tab.n_points - j0);
        const u32 pbeg = tab.point_begin, sid = tab.system_id;
        const int C = tg.C;
        auto run_item = [&](const auto& choose) {
            for (u32 t = threadIdx.x; t < n_here; t += blockDim.x) {
                const u32 i = pbeg + j0 + t;
                float x, y;
                start_point(a, i, sid, x, y);
                const CfsStream ps = cfs_stream(a.rk, i, sid);
                auto step = [&](u32 w) {
                    const int k = choose(w);
                    apply_map(tab, k, x, y);
                    cfs_splat_hist_tile(bt, tile, x, y, true, k, C, disc);
                };
                // blocks whole before the burn-in, whole past it, and the
                // (at most two) others with a test per step
                const u32 plain = min(a.burn_in, a.iters) >> 2, whole = a.iters >> 2;
                u32 nb = 0;
#pragma unroll 1
                for (; nb < plain; ++nb) {
                    const uint4 r = cfs_stream_block(a.rk, ps, nb, sid);
                    apply_map(tab, choose(r.x), x, y);
                    apply_map(tab, choose(r.y), x, y);
                    apply_map(tab, choose(r.z), x, y);
                    apply_map(tab, choose(r.w), x, y);
                }
#pragma unroll 1
                while (4u * nb < a.iters) {
                    if (4u * nb >= a.burn_in && nb < whole) {
#pragma unroll 1
                        for (; nb < whole; ++nb) {
                            const uint4 r = cfs_stream_block(a.rk, ps, nb, sid);
                            step(r.x);
                            step(r.y);
                            step(r.z);
                            step(r.w);
                        }
                        continue;
                    }
                    uint4 r = cfs_stream_block(a.rk, ps, nb, sid);
#pragma unroll 1
                    for (u32 n = 4u * nb; n < min(a.iters, 4u * nb + 4u); ++n) {
                        if (n < a.burn_in) apply_map(tab, choose(r.x), x, y);
                        else step(r.x);
                        r = make_uint4(r.y, r.z, r.w, 0u);
                    }
                    ++nb;
                }
            }
        };
        // (a copy of the step code for each choice; the generated batch kernel's
        // third, one lookup, took 242 us here as without it: the table's part for
        // it is built and not read)
        if (kt.more <= 1) run_item(CfsChooseKtab<false>{kt, 1});
        else run_item(CfsChooseKtab<true>{kt, kt.more});
        __syncthreads();
    }
    if (cur >= 0) leave_frame();
}

// per-device set-up: the device address of the array, the grid size and the
// kernels' shared-memory limits
struct DeviceSetup {
    bool ready = false;
    NaScratch* ws = nullptr;
    int sms = 0;
};
constexpr int kMaxDevices = 64;
DeviceSetup g_setup[kMaxDevices];
std::mutex g_setup_mu;

cfs_status setup_device(int dev, DeviceSetup** out)
{
    using cfs::check_cuda;
    if (dev < 0 || dev >= kMaxDevices) return cfs::fail(CFS_ERR_UNSUPPORTED, "device index");
    std::lock_guard<std::mutex> lock(g_setup_mu);
    DeviceSetup& s = g_setup[dev];
    if (!s.ready) {
        // host code must not use g_noalloc_scratch directly: it is a host
        // stand-in; the device address comes from the runtime
        void* p = nullptr;
        cfs_status st = check_cuda(cudaGetSymbolAddress(&p, g_noalloc_scratch),
                                   "cudaGetSymbolAddress(no-alloc scratch)");
        if (st != CFS_OK) return st;
        int sms = 0;
        st = check_cuda(cudaFuncSetAttribute(noalloc_batch_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)(kCounters * sizeof(u32))),
                        "cudaFuncSetAttribute");
        if (st == CFS_OK)
            st = check_cuda(cudaFuncSetAttribute(noalloc_place_kernel,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 CFS_WIN_SMEM),
                            "cudaFuncSetAttribute");
        if (st != CFS_OK) return st;
        st = check_cuda(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev),
                        "cudaDeviceGetAttribute");
        if (st != CFS_OK) return st;
        s.ws = static_cast<NaScratch*>(p);
        s.sms = sms > 0 ? sms : 1;
        s.ready = true;
    }
    *out = &s;
    return CFS_OK;
}

}  // namespace

extern "C" cfs_status cfs_render_batch_noalloc(const cfs_frame* frames, int n_frames,
                                               uint32_t iters, uint32_t burn_in, uint64_t seed,
                                               int clear, unsigned long long* discards,
                                               void* stream_)
{
    using cfs::check_cuda;
    using cfs::fail;
    cfs::clear_error();
    if (!frames || n_frames <= 0) return fail(CFS_ERR_INVALID_ARG, "need at least one frame");
    if (n_frames > kMaxFrames)
        return fail(CFS_ERR_INVALID_ARG,
                    "cfs_render_batch_noalloc takes at most CFS_NOALLOC_MAX_FRAMES (256) frames");
    for (int f = 0; f < n_frames; ++f) {
        const cfs_frame& fr = frames[f];
        const cfs_system* s = fr.system;
        const cfs_target& t = fr.targets[0];
        if (!s || s->dim != 2) return fail(CFS_ERR_INVALID_ARG, "every frame needs a 2D system");
        for (int k = 0; k < s->n_maps; ++k)
            if (s->maps[k].kind != CFS_MAP_AFFINE)
                return fail(CFS_ERR_UNSUPPORTED, "the no-allocation batch renders affine maps");
        if (t.kind != CFS_TARGET_HIST_U32 || !t.data || t.width <= 0 || t.height <= 0 ||
            t.channels < 1 || t.channels > CFS_MAX_MAPS || !(t.x1 > t.x0) || !(t.y1 > t.y0) ||
            t.width > 65536 || t.height > 65536)
            return fail(CFS_ERR_INVALID_ARG, "every frame needs one u32 histogram target");
        if ((uint64_t)fr.point_begin + fr.n_points > (1ull << 32))
            return fail(CFS_ERR_INVALID_ARG, "point indices exceed 2^32");
        if ((uint64_t)fr.n_points > (1ull << 32) - 1024)
            return fail(CFS_ERR_INVALID_ARG, "a frame may hold at most 2^32 - 1024 points");
        if (fr.start)
            return fail(CFS_ERR_UNSUPPORTED,
                        "the no-allocation batch starts every point from Philox");
    }
    int dev = 0;
    cfs_status st = check_cuda(cudaGetDevice(&dev), "cudaGetDevice");
    if (st != CFS_OK) return st;
    DeviceSetup* ds = nullptr;
    st = setup_device(dev, &ds);
    if (st != CFS_OK) return st;
    cudaStream_t s = (cudaStream_t)stream_;
    if (burn_in > iters) burn_in = iters;

    // work items: the same rule as a planned batch's; their numbers come from
    // a 32-bit counter that runs up to n_items + grid (256 frames of less
    // than 2^32 points in items of at least 256 stay below 2^32)
    uint64_t points = 0;
    for (int f = 0; f < n_frames; ++f) points += frames[f].n_points;
    const uint32_t chunk = cfs::default_item_points(points, (uint32_t)ds->sms);
    uint64_t n_items = 0;
    for (int f = 0; f < n_frames; ++f) n_items += ((uint64_t)frames[f].n_points + chunk - 1) / chunk;
    if (n_items + (uint64_t)ds->sms >= (1ull << 32))
        return fail(CFS_ERR_INVALID_ARG, "too many points in one call");

    // frame descriptors go up as kernel arguments, copied at the launch
    uint32_t item = 0;
    size_t most = 0;                    // words of the largest histogram
    for (int first = 0; first < n_frames; first += kUpload) {
        NaUpload u;
        u.ws = ds->ws;
        u.first = (u32)first;
        u.count = (u32)std::min(kUpload, n_frames - first);
        u.reset = first == 0 ? 1u : 0u;
        u.pad = 0;
        std::memset(u.f, 0, sizeof(NaFrame) * u.count);
        for (u32 q = 0; q < u.count; ++q) {
            const cfs_frame& fr = frames[first + (int)q];
            const cfs_system& sy = *fr.system;
            const cfs_target& t = fr.targets[0];
            NaFrame& d = u.f[q];
            for (int j = 0; j < sy.n_cmp; ++j) d.T[j] = sy.T[j];
            d.n_cmp = sy.n_cmp;
            d.n_points = fr.n_points;
            d.point_begin = fr.point_begin;
            d.system_id = fr.system_id;
            d.item_begin = item;
            for (int k = 0; k < sy.n_maps; ++k)
                for (int j = 0; j < 6; ++j) d.prm[j][k] = sy.maps[k].params[j];
            d.tg.data = (unsigned long long)(uintptr_t)t.data;
            d.tg.W = t.width;
            d.tg.H = t.height;
            d.tg.C = t.channels;
            d.tg.x0 = t.x0; d.tg.x1 = t.x1; d.tg.y0 = t.y0; d.tg.y1 = t.y1;
            d.tg.sx = (float)t.width / (t.x1 - t.x0);
            d.tg.sy = (float)t.height / (t.y1 - t.y0);
            item += (uint32_t)(((uint64_t)fr.n_points + chunk - 1) / chunk);
            most = std::max(most, (size_t)t.width * (size_t)t.height * (size_t)t.channels);
        }
        noalloc_upload_kernel<<<8, 256, 0, s>>>(u);
        st = check_cuda(cudaGetLastError(), "noalloc_upload_kernel launch");
        if (st != CFS_OK) return st;
    }
    if (clear) {
        // 16 KB per block of a typical frame, at most 8 blocks per SM a frame
        const size_t want = std::min<size_t>((most + 4095) / 4096, (size_t)ds->sms * 8);
        noalloc_clear_kernel<<<dim3((unsigned)std::max<size_t>(1, want), (unsigned)n_frames), 256, 0,
                               s>>>(ds->ws);
        st = check_cuda(cudaGetLastError(), "noalloc_clear_kernel launch");
        if (st != CFS_OK) return st;
    }
    if (item > 0) {
        NaArgs a;
        std::memset(&a, 0, sizeof(a));
        cfs::philox_round_keys(seed, a.rk);
        a.iters = iters;
        a.burn_in = burn_in;
        a.n_frames = (u32)n_frames;
        a.n_items = item;
        a.chunk = chunk;
        a.ws = ds->ws;
        const unsigned grid = std::min<unsigned>((unsigned)ds->sms, item);
        noalloc_place_kernel<<<(unsigned)n_frames, kBlock, CFS_WIN_SMEM, s>>>(a);
        st = check_cuda(cudaGetLastError(), "noalloc_place_kernel launch");
        if (st != CFS_OK) return st;
        noalloc_batch_kernel<<<grid, kBlock, kCounters * sizeof(u32), s>>>(a);
        st = check_cuda(cudaGetLastError(), "noalloc_batch_kernel launch");
        if (st != CFS_OK) return st;
    }
    if (discards)
        st = check_cuda(cudaMemcpyAsync(discards, ds->ws->discards,
                                        sizeof(unsigned long long) * (size_t)n_frames,
                                        cudaMemcpyDeviceToDevice, s),
                        "cudaMemcpyAsync(discards)");
    return st;
}
