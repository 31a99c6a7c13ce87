// cfs_sampler.cu -- the learned warm-start sampler.
//
// The paper leaves the initial distribution of the primitive to future work
// (Section 4: generate it automatically from the function systems).  The
// sampler is that idea made concrete: an MLP maps Gaussian noise, the affine
// parameters of a system (up to 8 maps) and the frame time t to a point near
// the system's attractor, so a render can start its points there and skip
// most of the burn-in.  It is trained on chaos-game points the library
// itself generates, with a sliced-Wasserstein loss.
//
// Network: u (64) -> 128 -> 128 -> 128 -> 2, SiLU after the first three
// layers; BF16 weights and activations, FP32 accumulation on the tensor
// cores, FP32 master weights and Adam state.  Training and inference run their
// products on the fifth-generation tensor cores (tcgen05.mma, accumulators in
// tensor memory).
//
// Parameter vector (FP32, this order): W1 [128][64], b1 [128], W2 [128][128],
// b2, W3 [128][128], b3, W4 [2][128], b4 [2] -- 41602 floats.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "cfs_device.cuh"
#include "cfs_internal.h"

namespace {

typedef unsigned short bf16r;

constexpr int D_IN = 64, HID = 128, D_OUT = 2;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + HID * D_IN;
constexpr int OFF_W2 = OFF_B1 + HID, OFF_B2 = OFF_W2 + HID * HID;
constexpr int OFF_W3 = OFF_B2 + HID, OFF_B3 = OFF_W3 + HID * HID;
constexpr int OFF_W4 = OFF_B3 + HID, OFF_B4 = OFF_W4 + D_OUT * HID;
constexpr int N_PARAMS = OFF_B4 + D_OUT;   // 41602
constexpr int MAX_SYS_MAPS = 8;
constexpr int COND = 6 * MAX_SYS_MAPS;     // 48 conditioning parameters

__device__ __forceinline__ bf16r to_bf16(float v)
{
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    return *reinterpret_cast<const bf16r*>(&h);
}

__device__ __forceinline__ float from_bf16(bf16r v)
{
    return __uint_as_float(((u32)v) << 16);
}

// SiLU and its derivative in training: sigma(z) = 1 / (1 + e^-z) with the
// hardware exponential and reciprocal (relative error a few ulps, far below
// the BF16 rounding of the activations and gradients they feed)
__device__ __forceinline__ float sigmoid_f(float z)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(1.0f + __expf(-z)));
    return r;
}

__device__ __forceinline__ float silu_f(float z) { return z * sigmoid_f(z); }

__device__ __forceinline__ float silu_grad_f(float z)
{
    const float s = sigmoid_f(z);
    return s * (1.0f + z * (1.0f - s));
}

// ---------------------------------------------------------------------------
// GEMM on the fifth-generation tensor cores:
//   D[M][N] = A[M][K] B[N][K]^T,  A and B BF16 and K-major in global memory,
//   D accumulated in FP32 in tensor memory (TMEM).
// CTA tile: 128 rows x the whole width N (64 or 128).  K runs in chunks of
// 64, staged by the CTA's 128 threads into shared memory in the no-swizzle
// K-major layout of 8-row x 16-byte core matrices (K-adjacent cores 128 B
// apart, 8-row groups 1024 B apart).  Thread 0 issues the four tcgen05.mma of
// a chunk (M = 128, N, K = 16 each) and commits them to an mbarrier; the chunk's
// place is refilled only after that barrier completes.  It serves batches of
// fewer than 128 rows: K is at most 128, two chunks.  The epilogue reads the accumulator with tcgen05.ld: warp w
// owns TMEM lanes 32w..32w+31, so every thread holds one output row.
// Every wait is bounded: on a time-out the CTA records it in g_tc_error,
// skips its epilogue, frees its TMEM and returns.
// ---------------------------------------------------------------------------
enum Epi { EPI_SILU = 1, EPI_SILU_GRAD = 2, EPI_ATOMIC = 3 };

constexpr int TC_M = 128, TC_K = 64, TC_THREADS = 256;
constexpr int TC_NV = 128 * 8 / TC_THREADS;   // 16-byte vectors per thread per operand tile
constexpr int TC_TILE_BYTES = 128 * TC_K * 2;             // 16 KB: 128 rows x 64 K
// dynamic shared memory: a chunk of A and B, barrier and alignment, padded so that
// at most four CTAs share an SM (four times 128 TMEM columns fill its 512)
constexpr int TC_SMEM = 50 * 1024;
constexpr u32 TC_WAIT_LIMIT = 1u << 24;
constexpr int TC_COPIES = 16;   // copies of the bias-gradient sums (spread the atomics)

__device__ unsigned int g_tc_error = 0;

struct TcArgs {
    int M, N, K;                 // N in {64, 128}
    const bf16r* A; int lda;     // [M][lda], K contiguous
    const bf16r* B; int ldb;     // [N][ldb], K contiguous
    int mode;
    const float* bias;           // SILU: [N]
    float* C; int ldc;           // SILU: pre-activation Z out; ATOMIC: C += D
    bf16r* H; int ldh;           // SILU: activation out; SILU_GRAD: dZ out
    bf16r* HT; int ldt;          // SILU, SILU_GRAD: transposed copy [N][ldt] (or null)
    const float* Zin; int ldz;   // SILU_GRAD: pre-activation of the layer
    float* colsum;               // SILU_GRAD: bias gradient partials, [TC_COPIES][N]; CTA b
                                 // adds its column sums into copy b % TC_COPIES
};

// Waits for the grid before this one in the stream where this one was launched
// to start early (launch_after), and lets the next one do so.  In this order:
// what ran before the previous grid is then complete for the next one's part
// before its own wait, which loads weights and touches nothing else.  The
// previous grid's output is written while this one lives, so it is read with
// ordinary loads: __ldg and const __restrict__ would promise otherwise and
// could be moved above the wait (loss and gradients of 65536 rows: 184.0 us with
// them, 183.1 without)
__device__ __forceinline__ void after_previous()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ u32 smem_addr(const void* p)
{
    return (u32)__cvta_generic_to_shared(p);
}

// shared-memory matrix descriptor: start address, leading (K) byte offset
// 128, stride (8-row group) byte offset 1024, descriptor version 1 (bit 46),
// base offset 0, no swizzle
__device__ __forceinline__ u64 tc_desc(u32 saddr)
{
    return (u64)((saddr >> 4) & 0x3FFFu) | ((u64)(128u >> 4) << 16) |
           ((u64)(1024u >> 4) << 32) | ((u64)1 << 46);
}

// instruction descriptor of kind::f16: D F32 (bit 4), A and B BF16 (bits 7,
// 10), both K-major, N >> 3 at bit 17, M >> 4 at bit 24
__device__ __forceinline__ u32 tc_idesc(int N)
{
    return (1u << 4) | (1u << 7) | (1u << 10) | ((u32)(N >> 3) << 17) |
           ((u32)(TC_M >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(u32 d_tmem, u64 adesc, u64 bdesc, u32 idesc, u32 acc)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n"
        :
        : "r"(d_tmem), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void tc_commit(u32 bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                 :
                 : "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void mbar_init(u32 bar, u32 count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" : : "r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_wait(u32 bar, u32 parity)
{
    for (u32 it = 0; it < TC_WAIT_LIMIT; ++it) {
        u32 done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done)
            : "r"(bar), "r"(parity)
            : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// 16 consecutive FP32 columns of this thread's TMEM lane, without the wait
// (the caller issues tcgen05.wait::ld before using them)
__device__ __forceinline__ void tc_ld16_nowait(u32 taddr, u32 (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

// the loads of this thread so far have arrived; r (one of them) may be used
// from here on
__device__ __forceinline__ void tc_wait_ld(u32 (&r)[16])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]),
                   "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]),
                   "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
                 :
                 : "memory");
}

// f(c0, the 16 FP32 columns c0 .. c0 + 15 of this thread's TMEM lane) for the
// 128 columns from taddr: the next 16 are on their way while f works
template <class F>
__device__ __forceinline__ void tc_for_columns(u32 taddr, F f)
{
    u32 a[16], b[16];
    tc_ld16_nowait(taddr, a);
#pragma unroll 1
    for (int c0 = 0; c0 < 128; c0 += 32) {
        tc_wait_ld(a);
        tc_ld16_nowait(taddr + (u32)(c0 + 16), b);
        f(c0, a);
        tc_wait_ld(b);
        if (c0 + 32 < 128) tc_ld16_nowait(taddr + (u32)(c0 + 32), a);
        f(c0 + 16, b);
    }
}

// 16 consecutive FP32 columns of this thread's TMEM lane
__device__ __forceinline__ void tc_ld16(u32 taddr, float (&v)[16])
{
    u32 r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// Staging of rows row0 .. row0 + n_rows - 1 (those < rows_valid), K columns
// k0 .. k0 + 63 (those < k_end) of a K-major BF16 matrix into the core-matrix
// layout, zeros elsewhere.  Vector v -> row (v / 64) * 8 + v % 8, K group
// (v / 8) % 8, so each 8-lane phase of a warp writes one contiguous 128-byte
// core matrix.  Two phases -- every load of the tile first, then the shared
// stores -- keep TC_NV loads per thread in flight.
__device__ __forceinline__ void tc_stage_load(uint4 (&val)[TC_NV], const bf16r* src, int ld,
                                              int rows_valid, int row0, int n_rows, int k0,
                                              int k_end)
{
#pragma unroll
    for (int i = 0; i < TC_NV; ++i) {
        const int v = (int)threadIdx.x + i * TC_THREADS;
        const int r = ((v >> 6) << 3) | (v & 7), k8 = (v >> 3) & 7;
        const int gr = row0 + r, gk = k0 + 8 * k8;
        val[i] = make_uint4(0u, 0u, 0u, 0u);
        if (v < n_rows * 8 && gr < rows_valid && gk < k_end) {
            const bf16r* p = src + (size_t)gr * ld + gk;
            if (gk + 8 <= k_end) {
                val[i] = __ldg(reinterpret_cast<const uint4*>(p));
            } else {
                u32 w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (gk + e < k_end) w[e >> 1] |= (u32)p[e] << (16 * (e & 1));
                val[i] = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
    }
}

__device__ __forceinline__ void tc_stage_store(u32 dst, const uint4 (&val)[TC_NV], int n_rows)
{
#pragma unroll
    for (int i = 0; i < TC_NV; ++i) {
        const int v = (int)threadIdx.x + i * TC_THREADS;
        if (v < n_rows * 8) {
            const int r = ((v >> 6) << 3) | (v & 7), k8 = (v >> 3) & 7;
            const u32 a = dst + (u32)((r >> 3) * 1024 + k8 * 128 + (r & 7) * 16);
            asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};"
                         :
                         : "r"(a), "r"(val[i].x), "r"(val[i].y), "r"(val[i].z), "r"(val[i].w)
                         : "memory");
        }
    }
}

__device__ __forceinline__ u32 pack_bf16x2(float a, float b)
{
    return (u32)to_bf16(a) | ((u32)to_bf16(b) << 16);
}

// pre-activations of columns c0 .. c0 + 15 of this thread's row (SILU_GRAD)
__device__ __forceinline__ void tc_load_z(const TcArgs& g, int row, int c0, float (&z)[16])
{
    if (g.mode != EPI_SILU_GRAD || row >= g.M) return;
    const float4* zp = reinterpret_cast<const float4*>(g.Zin + (size_t)row * g.ldz + c0);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const float4 t = __ldg(zp + q);
        z[4 * q] = t.x; z[4 * q + 1] = t.y; z[4 * q + 2] = t.z; z[4 * q + 3] = t.w;
    }
}

// sums of 16 values over the warp's 32 lanes by halving exchanges (16
// shuffles instead of 80): on return lanes 2c and 2c + 1 hold the sum of
// value c
__device__ __forceinline__ float warp_colsum16(float (&h)[16])
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int w = 8; w >= 1; w >>= 1) {
        // this lane keeps values [0, w) or [w, 2w) of the current 2w and
        // adds the partner's copy of the same ones; the bit that decides is
        // lane bit log2(w) + 1 (16, 8, 4, 2 for w = 8, 4, 2, 1)
        const bool upper = (lane & (2 * w)) != 0;
#pragma unroll
        for (int k = 0; k < w; ++k) {
            const float send = upper ? h[k] : h[k + w];
            const float keep = upper ? h[k + w] : h[k];
            h[k] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * w);
        }
    }
    return h[0] + __shfl_xor_sync(0xffffffffu, h[0], 1);
}

__device__ __forceinline__ void tc_epilogue(const TcArgs& g, int row, int c0, const float (&v)[16],
                                            const float (&zi)[16], float* s_col,
                                            const float* bias)
{
    const bool in = row < g.M;
    if (g.mode == EPI_ATOMIC) {
        if (in) {
            float* c = g.C + (size_t)row * g.ldc + c0;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                cfs_red_add_v4f32(c + 4 * q, make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2],
                                                         v[4 * q + 3]));
        }
        return;
    }
    float h[16];
    if (g.mode == EPI_SILU) {
        float z[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
            z[j] = v[j] + bias[c0 + j];
            h[j] = silu_f(z[j]);
        }
        if (in && g.C) {
            float4* zc = reinterpret_cast<float4*>(g.C + (size_t)row * g.ldc + c0);
#pragma unroll
            for (int q = 0; q < 4; ++q) zc[q] = make_float4(z[4 * q], z[4 * q + 1], z[4 * q + 2], z[4 * q + 3]);
        }
    } else {   // EPI_SILU_GRAD
#pragma unroll
        for (int j = 0; j < 16; ++j) h[j] = in ? v[j] * silu_grad_f(zi[j]) : 0.0f;
        // bias gradient: column sums over the warp's 32 rows, one atomic per column
        float hs[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) hs[j] = h[j];
        const float s = warp_colsum16(hs);
        const int lane = threadIdx.x & 31;
        if (!(lane & 1) && s != 0.0f) atomicAdd(s_col + c0 + (lane >> 1), s);
    }
    if (in && g.H) {
        uint4* hp = reinterpret_cast<uint4*>(g.H + (size_t)row * g.ldh + c0);
        hp[0] = make_uint4(pack_bf16x2(h[0], h[1]), pack_bf16x2(h[2], h[3]),
                           pack_bf16x2(h[4], h[5]), pack_bf16x2(h[6], h[7]));
        hp[1] = make_uint4(pack_bf16x2(h[8], h[9]), pack_bf16x2(h[10], h[11]),
                           pack_bf16x2(h[12], h[13]), pack_bf16x2(h[14], h[15]));
    }
    if (in && g.HT) {
        // consecutive lanes hold consecutive rows: each column's stores coalesce
#pragma unroll
        for (int j = 0; j < 16; ++j) g.HT[(size_t)(c0 + j) * g.ldt + row] = to_bf16(h[j]);
    }
}

__global__ void __launch_bounds__(TC_THREADS) tc_gemm_kernel(const __grid_constant__ TcArgs g)
{
    extern __shared__ unsigned char tc_smem_raw[];
    unsigned char* sm = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~(uintptr_t)1023);
    // A at sm, B right after it
    const u32 sA = smem_addr(sm), sB = sA + TC_TILE_BYTES;
    const u32 bar = smem_addr(sm + 2 * TC_TILE_BYTES);
    u32* s_tmem = reinterpret_cast<u32*>(sm + 2 * TC_TILE_BYTES + 64);
    float* s_col = reinterpret_cast<float*>(sm + 2 * TC_TILE_BYTES + 128);   // [128]
    const int tid = threadIdx.x, warp = tid >> 5;
    const int m0 = blockIdx.x * TC_M;
    const int n_chunks = (g.K + TC_K - 1) / TC_K;
    const u32 ncols = g.N <= 64 ? 64u : 128u;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :
                     : "r"(smem_addr(s_tmem)), "r"(ncols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid < 128) s_col[tid] = 0.0f;
    if (tid == 0) {
        mbar_init(bar, 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const u32 tmem = *s_tmem;
    const u32 idesc = tc_idesc(g.N);

    bool ok = true;
    for (int c = 0; c < n_chunks; ++c) {
        // (the barrier completes once per chunk: the previous one must have left
        // the tensor core)
        if (c > 0) ok = mbar_wait(bar, (u32)(c - 1) & 1u);
        if (!__syncthreads_and(ok)) { ok = false; break; }
        const int k0 = c * TC_K;
        {
            uint4 va[TC_NV], vb[TC_NV];
            tc_stage_load(va, g.A, g.lda, g.M, m0, TC_M, k0, g.K);
            tc_stage_load(vb, g.B, g.ldb, g.N, 0, g.N, k0, g.K);
            tc_stage_store(sA, va, TC_M);
            tc_stage_store(sB, vb, g.N);
        }
        // generic-proxy stores -> visible to the tensor core (async proxy)
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (tid == 0) {
            tc_fence_after();
#pragma unroll
            for (int kk = 0; kk < TC_K / 16; ++kk)
                tc_mma(tmem, tc_desc(sA + kk * 256), tc_desc(sB + kk * 256), idesc,
                       (c > 0 || kk > 0) ? 1u : 0u);
            tc_commit(bar);
        }
    }
    // epilogue split: warp w reads TMEM lanes 32 (w % 4) .. + 31 (its rows)
    // and the columns of half w / 4
    const int quad = warp & 3, half = warp >> 2;
    const int row = m0 + quad * 32 + (tid & 31);
    const int c_begin = half * (g.N / 2), c_end = c_begin + g.N / 2;
    float z_next[16];
    tc_load_z(g, row, c_begin, z_next);   // independent of the MMAs: overlaps them
    if (ok && n_chunks > 0) ok = mbar_wait(bar, (u32)(n_chunks - 1) & 1u);
    ok = __syncthreads_and(ok) != 0;
    tc_fence_after();
    if (ok && n_chunks > 0) {
        const u32 lane_base = tmem + ((u32)(quad * 32) << 16);
        for (int c0 = c_begin; c0 < c_end; c0 += 16) {
            float z[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) z[j] = z_next[j];
            if (c0 + 16 < c_end) tc_load_z(g, row, c0 + 16, z_next);
            float v[16];
            tc_ld16(lane_base + (u32)c0, v);
            tc_epilogue(g, row, c0, v, z, s_col, g.bias);
        }
    } else if (!ok && tid == 0) {
        atomicOr(&g_tc_error, (unsigned)CFS_DEVICE_ERR_TC_TIMEOUT);
        // give in-flight MMAs a bounded chance to drain before TMEM is freed
        if (n_chunks > 0) mbar_wait(bar, (u32)(n_chunks - 1) & 1u);
    }
    tc_fence_before();
    __syncthreads();
    // the CTA's bias-gradient column sums: one atomic per column into copy
    // blockIdx.x % TC_COPIES
    if (g.mode == EPI_SILU_GRAD && ok && tid < g.N && s_col[tid] != 0.0f)
        atomicAdd(g.colsum + (blockIdx.x % TC_COPIES) * g.N + tid, s_col[tid]);
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;"
                     :
                     : "r"(tmem), "r"(ncols)
                     : "memory");
    }
}

// ---------------------------------------------------------------------------
// shared-memory descriptors of TMA boxes, TMA and mbarriers
// ---------------------------------------------------------------------------
// K-major operand in the 128-byte swizzle: 8 rows of 64 K elements are one
// 1024-byte atom (stride offset between 8-row groups); within it a step of 16
// K elements is 32 bytes of the start address
__device__ __forceinline__ u64 tc_desc_ksw(u32 saddr)
{
    return (u64)((saddr >> 4) & 0x3FFFu) | ((u64)1 << 16) | ((u64)(1024u >> 4) << 32) |
           ((u64)1 << 46) | ((u64)2 << 61);
}

// MN-major operand with the 128-byte swizzle: 64 features of 8 rows are one
// 1024-byte atom; 8-row groups 1024 B apart (stride offset), 64-feature
// blocks `block` bytes apart (leading offset); swizzle mode 2 at bit 61
__device__ __forceinline__ u64 tc_desc_mn(u32 saddr, u32 block)
{
    return (u64)((saddr >> 4) & 0x3FFFu) | ((u64)(block >> 4) << 16) |
           ((u64)(1024u >> 4) << 32) | ((u64)1 << 46) | ((u64)2 << 61);
}

__device__ __forceinline__ u64 tc_desc_kn(u32 saddr, u32 lbo, u32 sbo)
{
    return (u64)((saddr >> 4) & 0x3FFFu) | ((u64)((lbo >> 4) & 0x3FFFu) << 16) |
           ((u64)((sbo >> 4) & 0x3FFFu) << 32) | ((u64)1 << 46);
}

__device__ __forceinline__ void mbar_expect_tx(u32 bar, u32 bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

// one box of a 2D tensor map at element coordinates (x = K, y = row)
__device__ __forceinline__ void tma_load_2d(u32 dst, const CUtensorMap* map, int x, int y, u32 bar)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, "
        "{%2, %3}], [%4];" ::"r"(dst),
        "l"(reinterpret_cast<u64>(map)), "r"(x), "r"(y), "r"(bar)
        : "memory");
}

// sums of the gradient copies in bias_part (the output layer's and the bias
// gradients) added to grads, by one block
constexpr int OB_PART = 3 * HID + 4;
constexpr int PART_FLOATS = TC_COPIES * (2 * HID + OB_PART);
__device__ __forceinline__ void part_reduce(const float* part, float* grads)
{
    for (int e = threadIdx.x; e < 2 * HID + 3 * HID + 2; e += blockDim.x) {
        float s = 0.0f;
        if (e < 2 * HID) {
            const int l = e / HID, c = e % HID;
            for (int k = 0; k < TC_COPIES; ++k) s += part[((size_t)l * TC_COPIES + k) * HID + c];
            grads[(l == 0 ? OFF_B2 : OFF_B1) + c] += s;
        } else {
            const int q = e - 2 * HID;
            const float* ob = part + (size_t)2 * TC_COPIES * HID;
            for (int k = 0; k < TC_COPIES; ++k) s += ob[(size_t)k * OB_PART + q];
            grads[q < 2 * HID ? OFF_W4 + q : (q < 3 * HID ? OFF_B3 + q - 2 * HID
                                                          : OFF_B4 + q - 3 * HID)] += s;
        }
    }
}

// ---------------------------------------------------------------------------
// The three weight gradients dW_l[128][N] += dZ_l^T A (A: the layer's input, N
// = 128, 128 or 64) in one launch, split over the rows: the CTAs are dealt to
// the gradients in proportion to what they read, and each takes a run of
// 64-row chunks.  Both operands are the row-major activations themselves:
// their rows are the contraction, so they are MN-major operands (transpose
// bits of the instruction descriptor) and nothing has to be stored
// transposed.  A chunk is one or two TMA boxes of 64 rows x 64 features an
// operand (128-byte swizzle).  Warp 0 loads the chunks into a ring of
// DW_STAGES slots, one thread of warp 1 accumulates them into one TMEM
// accumulator, and warps 2..5 add it to dW with vector reductions at the end.
// One more CTA sums the bias-gradient copies.  Every wait is bounded: a time-out
// sets g_tc_error and the role stops.
// What it measured (65536 rows): 54 us for three launches on K-major operands,
// whose 16-byte box rows the TMA unit took one by one, besides the transposed
// copies that every producer wrote.
// ---------------------------------------------------------------------------
constexpr int DW_STAGES = 4;
constexpr int DW_THREADS = 32 * 6;
constexpr int DW_ROWS = 64;
constexpr int DW_BOX = DW_ROWS * 128;         // 64 rows x 64 BF16 features
constexpr int DW_SLOT = 4 * DW_BOX;           // A and B chunk of up to 128 features each
constexpr int DW_SMEM = 1024 + DW_STAGES * DW_SLOT + 256;


struct DwArgs {
    int chunks;                  // of DW_ROWS rows
    int cta0[4];                 // first CTA of each gradient, and the end
    int N[3];
    float* C[3];                 // [128][N]
    const float* part;           // the bias-gradient copies and
    float* grads;                // where their sums go
};

struct DwMaps {
    CUtensorMap a[3], b[3];
};

__global__ void __launch_bounds__(DW_THREADS, 1) tc_dw_kernel(const __grid_constant__ DwMaps maps,
                                                              const __grid_constant__ DwArgs g)
{
    extern __shared__ unsigned char dw_smem_raw[];
    if ((int)blockIdx.x >= g.cta0[3]) {
        after_previous();
        part_reduce(g.part, g.grads);
        return;
    }
    unsigned char* sm = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(dw_smem_raw) + 1023) & ~(uintptr_t)1023);
    const u32 s0 = smem_addr(sm);
    u64* bars = reinterpret_cast<u64*>(sm + DW_STAGES * DW_SLOT);
    auto full = [&](int s) { return smem_addr(&bars[s]); };
    auto empty = [&](int s) { return smem_addr(&bars[DW_STAGES + s]); };
    const u32 tdone = smem_addr(&bars[2 * DW_STAGES]);
    u32* s_tmem = reinterpret_cast<u32*>(bars + 16);
    __shared__ int s_err;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int p = (int)blockIdx.x < g.cta0[1] ? 0 : ((int)blockIdx.x < g.cta0[2] ? 1 : 2);
    const int ctas = g.cta0[p + 1] - g.cta0[p], N = g.N[p];
    const int per = (g.chunks + ctas - 1) / ctas;
    const int c_first = min(g.chunks, ((int)blockIdx.x - g.cta0[p]) * per);
    const int c_last = min(g.chunks, c_first + per);

    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :
                     : "r"(smem_addr(s_tmem)), "r"(128u)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (threadIdx.x == 0) {
        s_err = 0;
        for (int s = 0; s < DW_STAGES; ++s) {
            mbar_init(full(s), 1u);
            mbar_init(empty(s), 1u);
        }
        mbar_init(tdone, 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const u32 tmem = *s_tmem;
    after_previous();
    // slot s: A at s0 + s DW_SLOT (two boxes), B after it (N / 64 boxes)
    if (warp == 0) {
        if (lane == 0) {
            const CUtensorMap* ma = &maps.a[p];
            const CUtensorMap* mb = &maps.b[p];
            int i = 0, issued = 0;
            for (int c = c_first; c < c_last; ++c, ++i) {
                const int s = i % DW_STAGES;
                if (i >= DW_STAGES && !mbar_wait(empty(s), (u32)(i / DW_STAGES - 1) & 1u)) {
                    atomicExch(&s_err, 1);
                    break;
                }
                mbar_expect_tx(full(s), (u32)((2 + N / 64) * DW_BOX));
                const u32 a = s0 + (u32)(s * DW_SLOT);
                tma_load_2d(a, ma, 0, c * DW_ROWS, full(s));
                tma_load_2d(a + DW_BOX, ma, 64, c * DW_ROWS, full(s));
                tma_load_2d(a + 2 * DW_BOX, mb, 0, c * DW_ROWS, full(s));
                if (N == 128) tma_load_2d(a + 3 * DW_BOX, mb, 64, c * DW_ROWS, full(s));
                issued = i + 1;
            }
            for (int j = (issued > DW_STAGES ? issued - DW_STAGES : 0); j < issued; ++j)
                mbar_wait(full(j % DW_STAGES), (u32)(j / DW_STAGES) & 1u);
        }
    } else if (warp == 1) {
        if (lane == 0) {
            // both operands MN-major: transpose bits 15 and 16
            const u32 idesc = tc_idesc(N) | (1u << 15) | (1u << 16);
            bool ok = true;
            int i = 0;
            for (int c = c_first; c < c_last; ++c, ++i) {
                const int s = i % DW_STAGES;
                if (!mbar_wait(full(s), (u32)(i / DW_STAGES) & 1u)) { ok = false; break; }
                tc_fence_after();
                const u32 a = s0 + (u32)(s * DW_SLOT);
#pragma unroll
                for (int kk = 0; kk < DW_ROWS / 16; ++kk)      // 16 rows: two 1024-byte groups
                    tc_mma(tmem, tc_desc_mn(a + kk * 2048, DW_BOX),
                           tc_desc_mn(a + 2 * DW_BOX + kk * 2048, DW_BOX), idesc,
                           (i > 0 || kk > 0) ? 1u : 0u);
                tc_commit(empty(s));
            }
            if (!ok) atomicExch(&s_err, 1);
            tc_commit(tdone);   // every MMA issued above (none: arrives at once)
        }
    } else {
        const int quad = warp & 3;
        const bool any = c_last > c_first;
        if (!mbar_wait(tdone, 0u)) {
            atomicExch(&s_err, 1);
        } else if (any && !s_err) {
            tc_fence_after();
            const int row = quad * 32 + lane;
            const u32 base = tmem + ((u32)(quad * 32) << 16);
            for (int c0 = 0; c0 < N; c0 += 16) {
                float v[16];
                tc_ld16(base + (u32)c0, v);
                float* c = g.C[p] + (size_t)row * N + c0;
#pragma unroll
                for (int q = 0; q < 4; ++q)
                    cfs_red_add_v4f32(c + 4 * q, make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2],
                                                             v[4 * q + 3]));
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (threadIdx.x == 0 && s_err) atomicOr(&g_tc_error, (unsigned)CFS_DEVICE_ERR_TC_TIMEOUT);
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                     "r"(128u)
                     : "memory");
    }
}

// output layer forward Y = H3 W4^T + b4 (N = 2: a dot product per output,
// not a tensor-core shape): one thread per row
__global__ void __launch_bounds__(256) out_forward_kernel(const bf16r* __restrict__ H3,
                                                          const bf16r* __restrict__ wb,
                                                          const float* __restrict__ w, int B,
                                                          float* Y)
{
    __shared__ float w4[D_OUT][HID];
    for (int e = threadIdx.x; e < D_OUT * HID; e += blockDim.x)
        w4[e / HID][e % HID] = from_bf16(wb[OFF_W4 + e]);
    __syncthreads();
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= B) return;
    const uint4* h = reinterpret_cast<const uint4*>(H3 + (size_t)r * HID);
    float y0 = 0.0f, y1 = 0.0f;
#pragma unroll 4
    for (int q = 0; q < HID / 8; ++q) {
        const uint4 p = h[q];
        const u32 pw[4] = {p.x, p.y, p.z, p.w};
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float x = from_bf16((bf16r)(pw[e >> 1] >> (16 * (e & 1))));
            y0 = fmaf(x, w4[0][8 * q + e], y0);
            y1 = fmaf(x, w4[1][8 * q + e], y1);
        }
    }
    Y[2 * r] = y0 + w[OFF_B4];
    Y[2 * r + 1] = y1 + w[OFF_B4 + 1];
}

// bias_part: gradient partial sums in TC_COPIES copies to spread the atomics:
// [2][TC_COPIES][HID] bias gradients b2 and b1 (GEMM epilogues), then
// [TC_COPIES][OB_PART] of the output layer's backward: W4 rows 0 and 1
// (2 x HID), b3 (HID), b4 (2), padding
__global__ void __launch_bounds__(512) part_reduce_kernel(const float* part, float* grads)
{
    part_reduce(part, grads);
}

// U [rows][D_IN] -> UT [D_IN][ldt] (the K-major operand of dW1; batches of
// fewer than 64 rows)
__global__ void __launch_bounds__(256) transpose_in_kernel(const bf16r* __restrict__ U, int rows,
                                                           bf16r* UT, int ldt)
{
    __shared__ bf16r tile[32][D_IN + 2];
    const int r0 = blockIdx.x * 32;
    for (int e = threadIdx.x; e < 32 * D_IN; e += blockDim.x) {
        const int r = e / D_IN, c = e % D_IN;
        tile[r][c] = r0 + r < rows ? U[(size_t)(r0 + r) * D_IN + c] : (bf16r)0;
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 32 * D_IN; e += blockDim.x) {
        const int c = e / 32, r = e % 32;
        if (r0 + r < rows) UT[(size_t)c * ldt + r0 + r] = tile[r][c];
    }
}

// output layer backward: dH3 = dY W4 (N = 2, not a tensor-core shape), dZ3 =
// dH3 * silu'(Z3); dW4 = dY^T H3, db3 = sum dZ3, db4 = sum dY.  Lane l of a
// warp takes the units 4l .. 4l+3 of a row (16-byte loads of Z3, from which H3
// is formed again); blocks stride over runs of OB_ROWS rows, and their sums
// combine across warps in shared memory before one atomic per value into copy
// blockIdx.x % TC_COPIES of `part`.  SMALL (batches of fewer than 128 rows, a
// run per block) also writes the transpose dZ3^T.
constexpr int OB_ROWS = 64;
constexpr int OB_THREADS = 256;

template <bool SMALL>
__global__ void __launch_bounds__(OB_THREADS) out_backward_kernel(const float* dY,
                                                                  const bf16r* __restrict__ wb,
                                                                  const float* Z3, int B,
                                                                  bf16r* dZ3, bf16r* dZ3T, int ldt,
                                                                  float* part)
{
    // the block's dZ3 tile, transposed
    __shared__ bf16r tT[SMALL ? HID : 1][SMALL ? OB_ROWS + 1 : 1];
    __shared__ float s_sum[3 * HID + 2];     // W4 rows 0 and 1, b3, b4
    constexpr int WARPS = OB_THREADS / 32, RUN = OB_ROWS / WARPS;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int c = 4 * lane;
    float w0[4], w1[4], a0[4], a1[4], ab[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        w0[j] = from_bf16(wb[OFF_W4 + c + j]);
        w1[j] = from_bf16(wb[OFF_W4 + HID + c + j]);
        a0[j] = a1[j] = ab[j] = 0.0f;
    }
    float b40 = 0.0f, b41 = 0.0f;
    // rows of dY on eight-byte boundaries are read as one word
    const bool wide = ((uintptr_t)dY & 7u) == 0;
    after_previous();       // (the weights are older)
    for (int e = threadIdx.x; e < 3 * HID + 2; e += OB_THREADS) s_sum[e] = 0.0f;
    // a warp's RUN consecutive rows, four of them in flight
    for (int r0 = blockIdx.x * OB_ROWS; r0 < B; r0 += gridDim.x * OB_ROWS) {
#pragma unroll 1
        for (int k = 0; k < RUN; k += 4) {
            const int r = r0 + warp * RUN + k;
            float4 z[4];
            float2 y[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const bool in = r + q < B;
                const float* p = dY + 2 * (size_t)(r + q);
                y[q] = !in ? make_float2(0.0f, 0.0f)
                           : (wide ? *reinterpret_cast<const float2*>(p)
                                   : make_float2(p[0], p[1]));
                z[q] = in ? __ldcs(reinterpret_cast<const float4*>(Z3 + (size_t)(r + q) * HID + c))
                          : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                if (r + q >= B) break;
                const float zz[4] = {z[q].x, z[q].y, z[q].z, z[q].w};
                bf16r db[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float dh = fmaf(y[q].x, w0[j], y[q].y * w1[j]);
                    const float d = dh * silu_grad_f(zz[j]);
                    // H3 again, the forward's bits (the two share their sigmoid)
                    const float h = from_bf16(to_bf16(silu_f(zz[j])));
                    db[j] = to_bf16(d);
                    if constexpr (SMALL) tT[c + j][warp * RUN + k + q] = db[j];
                    ab[j] += d;
                    a0[j] = fmaf(y[q].x, h, a0[j]);
                    a1[j] = fmaf(y[q].y, h, a1[j]);
                }
                *reinterpret_cast<uint2*>(dZ3 + (size_t)(r + q) * HID + c) =
                    make_uint2((u32)db[0] | ((u32)db[1] << 16), (u32)db[2] | ((u32)db[3] << 16));
                b40 += y[q].x;
                b41 += y[q].y;
            }
        }
    }
    __syncthreads();   // tT complete, s_sum zeroed
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        atomicAdd(&s_sum[c + j], a0[j]);
        atomicAdd(&s_sum[HID + c + j], a1[j]);
        atomicAdd(&s_sum[2 * HID + c + j], ab[j]);
    }
    if (lane == 0) {
        atomicAdd(&s_sum[3 * HID], b40);
        atomicAdd(&s_sum[3 * HID + 1], b41);
    }
    if constexpr (SMALL) {
        // dZ3^T rows (one run of rows per block): a warp writes 64 consecutive
        // rows of one unit as 32 words
        const int r0 = blockIdx.x * OB_ROWS;
        for (int e = threadIdx.x; e < HID * (OB_ROWS / 2); e += OB_THREADS) {
            const int u = e / (OB_ROWS / 2), jp = 2 * (e % (OB_ROWS / 2));
            const int r = r0 + jp;
            if (r + 1 < B) {
                *reinterpret_cast<u32*>(dZ3T + (size_t)u * ldt + r) =
                    (u32)tT[u][jp] | ((u32)tT[u][jp + 1] << 16);
            } else if (r < B) {
                dZ3T[(size_t)u * ldt + r] = tT[u][jp];
            }
        }
    }
    __syncthreads();   // s_sum complete
    float* cp = part + (size_t)(blockIdx.x % TC_COPIES) * OB_PART;
    for (int e = threadIdx.x; e < 3 * HID + 2; e += OB_THREADS)
        if (s_sum[e] != 0.0f) atomicAdd(cp + e, s_sum[e]);
}

// ---------------------------------------------------------------------------
// sliced-Wasserstein loss and gradient.  A pair of warps takes the sorts of
// 1024 / N projections at once: a group of G = N / 32 lanes of the first warp
// sorts the projected predicted points of one, the same lanes of the second
// warp its projected target points, each lane holding 32 keys.
//
// Sorting network: every lane sorts its 32 keys in registers (Batcher's
// odd-even merge sort); bitonic merges do the rest.  Merge k (blocks of 2^k
// positions) runs compare-exchange stages on position bits k-1, ..., 0.  A
// position's bits are split into a window of 5 register bits [a, a + 5) -- the
// key's slot in its lane -- and the others, which number the lane; a stage on a
// bit of the window is a min/max of two slots of one lane.  The stages on
// bits k-1 .. 5 run in the topmost window and those on bits 4 .. 0 in the lowest,
// so a merge moves the keys twice through shared memory, 32 stores and 32 loads
// of a warp without bank conflicts and no barrier but the warp's own.  Blocks
// that a merge sorts descending hold their keys negated, so every stage puts
// the smaller key at the lower position and a merge boundary only flips signs.
//
// A point's rank is then found by binary search of its own key (recomputed bit
// for bit) among the sorted predicted keys, so the network carries no indices.
// The gradients of a CTA's projections are summed per point, and added to dX
// with one atomic per coordinate, system and round of sorts.  Keys must be
// finite.
//
// What it measured (64 systems x 1024 points x 64 projections): 50.6 us.  8 keys of
// either kind a thread and 128 threads a sort took 67 us, four fifths of the
// shared memory's cycles for 19 moves; half the moves leave the ALU pipe (min and
// max, 29 us), the moves (30 us) and the issue slots (27 us) about even.  One
// warp for both kinds had half the parallelism: 63 us there, and 20 us
// instead of 12 for 32 sorts.
// ---------------------------------------------------------------------------
constexpr int SW_LG = 5;           // register bits of a window
constexpr int SW_E = 1 << SW_LG;   // keys per lane
constexpr int SW_PAIRS = 4;        // of warps per CTA at most
// per multiprocessor: 64 registers a thread; 27 of the 4096 sorts of 64 x 64 fall to
// one, two rounds of its 16 pairs (with 3 CTAs three rounds: 53 us)
constexpr int SW_CTAS = 4;

__host__ __device__ constexpr int sw_log2(int n)
{
    return n > 1 ? 1 + sw_log2(n / 2) : 0;
}

__device__ __forceinline__ float sw_key(float u0, float u1, float c, float sn)
{
    return fmaf(u0, c, u1 * sn);
}

// word of position p in a group's array: one word of padding per 32 positions.
// Positions with disjoint bits add up, so a lane's keys lie at constant
// distances from its first one; and bit b moves a word by an odd multiple of
// 2^(b mod 5) banks, so the lanes of both windows hit all banks (the groups of
// a warp lie at odd multiples of G words)
__host__ __device__ constexpr int sw_word(int p)
{
    return p + (p >> 5);
}

// words of one group's array
template <int N>
constexpr int SW_WORDS = N + N / SW_E;

// all keys of a kind in a CTA
constexpr int SW_ALL = SW_PAIRS * 32 * (SW_E + 1);

// word of lane t's first key in window A
template <int A>
__device__ __forceinline__ int sw_first(int t)
{
    return sw_word((t & ((1 << A) - 1)) | ((t >> A) << (A + SW_LG)));
}

__device__ __forceinline__ void sw_exchange(float& a, float& b)
{
    const float lo = fminf(a, b), hi = fmaxf(a, b);
    a = lo;
    b = hi;
}

// Batcher's odd-even merge sort of a lane's keys, from the exchanges over a
// distance of D in the merge of runs of P
template <int P, int D>
__device__ __forceinline__ void sw_lane_sort(float (&x)[SW_E])
{
#pragma unroll
    for (int e = 0; e + D < SW_E; ++e)
        if (e >= D % P && (e - D % P) % (2 * D) < D && e / (2 * P) == (e + D) / (2 * P))
            sw_exchange(x[e], x[e + D]);
    if constexpr (D > 1)
        sw_lane_sort<P, D / 2>(x);
    else if constexpr (2 * P < SW_E)
        sw_lane_sort<2 * P, 2 * P>(x);
}

// compare-exchange of the slot pairs that differ in register bit M
template <int M>
__device__ __forceinline__ void sw_reg_stage(float (&x)[SW_E])
{
#pragma unroll
    for (int e = 0; e < SW_E; ++e)
        if (!(e & (1 << M))) sw_exchange(x[e], x[e | (1 << M)]);
}

// the stages on register bits M .. 0
template <int M>
__device__ __forceinline__ void sw_reg_stages(float (&x)[SW_E])
{
    sw_reg_stage<M>(x);
    if constexpr (M > 0) sw_reg_stages<M - 1>(x);
}

// merge k's stages on position bits 5 and up, from register bit M of window A down
template <int M, int A>
__device__ __forceinline__ void sw_high_stages(float (&x)[SW_E], int k)
{
    if (A + M < k) sw_reg_stage<M>(x);
    if constexpr (A + M > SW_LG) sw_high_stages<M - 1, A>(x, k);
}

// moves the group's keys from window A to window NA
template <int A, int NA>
__device__ __forceinline__ void sw_move(float (&x)[SW_E], int t, float* buf)
{
    float* w = buf + sw_first<A>(t);
    __syncwarp();               // the last move has read the buffer
#pragma unroll
    for (int e = 0; e < SW_E; ++e) w[sw_word(e << A)] = x[e];
    __syncwarp();
    const float* r = buf + sw_first<NA>(t);
#pragma unroll
    for (int e = 0; e < SW_E; ++e) x[e] = r[sw_word(e << NA)];
}

// sorts the group's keys: ranks 32 t .. 32 t + 31 in lane t on return.  The
// keys of odd lanes come negated where N > 32
template <int N>
__device__ __forceinline__ void sw_sort(float (&x)[SW_E], int t, float* buf)
{
    constexpr int L = sw_log2(N), A = L - SW_LG;
    sw_lane_sort<1, 1>(x);
    if constexpr (A > 0) {
        // one body for all the merges: unrolled, with the moves and stages of
        // each, the kernel spent its time fetching instructions
        bool down = t & 1;
#pragma unroll 1
        for (int k = SW_LG + 1; k <= L; ++k) {
            // lane t of window 0 holds positions (t << 5) | e: its keys are
            // negated where position bit k is set (not in the last merge)
            const bool next = k < L && ((t >> (k - SW_LG)) & 1);
            const float sg = next != down ? -1.0f : 1.0f;
            down = next;
#pragma unroll
            for (int e = 0; e < SW_E; ++e) x[e] *= sg;
            sw_move<0, A>(x, t, buf);
            sw_high_stages<SW_LG - 1, A>(x, k);
            sw_move<A, 0>(x, t, buf);
            sw_reg_stages<SW_LG - 1>(x);
        }
    }
}

// barrier of a pair's 64 threads
__device__ __forceinline__ void sw_pair_sync(int pair)
{
    asm volatile("bar.sync %0, 64;" ::"r"(pair + 1) : "memory");
}

template <int N>
__global__ void __launch_bounds__(64 * SW_PAIRS, SW_CTAS) sw_kernel(
    const float* X, const float* T, const float* phi, int P, u64 n_sorts, float scale, float* loss,
    float* dX)
{
    constexpr int G = N / SW_E, HALF = SW_E / 2;
    __shared__ float s_key[2 * SW_ALL];      // [predicted, target][groups][SW_WORDS]
    __shared__ float2 s_dir[32 * SW_PAIRS / G];
    __shared__ float s_loss[2 * SW_PAIRS];
    after_previous();
    const int pair = threadIdx.x >> 6, role = (threadIdx.x >> 5) & 1, lane = threadIdx.x & 31;
    const u32 g = pair * (32 / G) + lane / G;
    const int t = lane % G;
    const u32 groups = (blockDim.x >> 6) * (32 / G);
    float* key = s_key + g * SW_WORDS<N>;
    float* buf = key + role * SW_ALL;
    // points of eight-byte alignment are read as one word
    const bool wide = (((uintptr_t)X | (uintptr_t)T) & 7u) == 0;
    auto point = [&](const float* p) -> float2 {
        return wide ? *reinterpret_cast<const float2*>(p) : make_float2(p[0], p[1]);
    };
    // the sorts (system s, projection j) are numbered s P + j; this CTA takes an
    // equal run of them, one for every group at a time
    const u64 q1 = n_sorts / gridDim.x * (blockIdx.x + 1) +
                   min((u64)blockIdx.x + 1, n_sorts % gridDim.x);
    u64 q0 = n_sorts / gridDim.x * blockIdx.x + min((u64)blockIdx.x, n_sorts % gridDim.x);
    u32 s0 = (u32)(q0 / (u32)P), j0 = (u32)(q0 - (u64)s0 * (u32)P);
    float lacc = 0.0f;
    while (q0 < q1) {
        const u32 n = (u32)min((u64)groups, q1 - q0);
        if ((u32)(pair * (32 / G)) < n) {
            // (a group without a sort repeats the first one and counts for nothing)
            const u32 j = j0 + (g < n ? g : 0u), s = s0 + j / (u32)P;
            float sn, c;
            sincosf(phi[j % (u32)P], &sn, &c);
            if (role == 0 && t == 0) s_dir[g] = make_float2(c, sn);
            // slot e of lane t starts with point e G + t
            const size_t at = ((size_t)s * N + t) * 2;
            {
                const float* p = (role ? T : X) + at;
                const float sg = N > SW_E && (t & 1) ? -1.0f : 1.0f;
                float x[SW_E];
                if (wide) {
#pragma unroll
                    for (int e = 0; e < SW_E; ++e) {
                        const float2 u = reinterpret_cast<const float2*>(p)[e * G];
                        x[e] = sw_key(u.x, u.y, sg * c, sg * sn);
                    }
                } else {
#pragma unroll
                    for (int e = 0; e < SW_E; ++e)
                        x[e] = sw_key(p[2 * e * G], p[2 * e * G + 1], sg * c, sg * sn);
                }
                sw_sort<N>(x, t, buf);
                __syncwarp();       // the last move has read the buffer
#pragma unroll
                for (int e = 0; e < SW_E; ++e) buf[sw_first<0>(t) + e] = x[e];
            }
            sw_pair_sync(pair);
            // squared differences, and each rank's gradient in place of its
            // target, half of them by each warp
            {
                float* k = key + sw_first<0>(t) + role * HALF;
#pragma unroll
                for (int e = 0; e < HALF; ++e) {
                    const float d = k[e] - k[SW_ALL + e];
                    if (g < n) lacc = fmaf(d, d, lacc);
                    k[SW_ALL + e] = 2.0f * d / (float)N;
                }
            }
            sw_pair_sync(pair);
            // half of the points' ranks by bisection.  The first six pivots of
            // a search lie in different banks for different halves, so only the
            // last levels, 64 pivots and more, have conflicts
            float grad[HALF];
            const float* p = X + at + 2 * G * HALF * role;
#pragma unroll
            for (int e = 0; e < HALF; ++e) {
                const float2 u = point(p + 2 * G * e);
                const float kx = sw_key(u.x, u.y, c, sn);
                const float* r = key;
#pragma unroll
                for (int h = N / 2; h >= 1; h >>= 1) r += r[sw_word(h - 1)] < kx ? sw_word(h) : 0;
                grad[e] = r[SW_ALL];
            }
            sw_pair_sync(pair);     // the searches have read the keys
#pragma unroll
            for (int e = 0; e < HALF; ++e) key[(e + HALF * role) * G + t] = grad[e];
        }
        __syncthreads();
        for (u32 a = 0; a < n;) {
            const u32 b = min(n, a + ((u32)P - j0));    // the round's sorts of system s0
            for (int i = threadIdx.x; i < N; i += blockDim.x) {
                float ax = 0.0f, ay = 0.0f;
                for (u32 h = a; h < b; ++h) {
                    const float v = s_key[h * SW_WORDS<N> + i];
                    ax = fmaf(v, s_dir[h].x, ax);
                    ay = fmaf(v, s_dir[h].y, ay);
                }
                atomicAdd(dX + ((size_t)s0 * N + i) * 2, ax * scale);
                atomicAdd(dX + ((size_t)s0 * N + i) * 2 + 1, ay * scale);
            }
            j0 += b - a;
            if (j0 == (u32)P) {
                j0 = 0;
                ++s0;
            }
            a = b;
        }
        q0 += n;
        __syncthreads();        // the arrays serve the next round
    }
    for (int o = 16; o > 0; o >>= 1) lacc += __shfl_xor_sync(0xffffffffu, lacc, o);
    if (lane == 0) s_loss[threadIdx.x >> 5] = lacc;
    __syncthreads();
    if (threadIdx.x == 0) {
        float tot = 0.0f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += s_loss[w];
        atomicAdd(loss, tot * scale / (float)N);
    }
}

// Launches `kernel`, which calls after_previous(); where the stream's previous
// operation is a kernel of this file that does so too (`after`), it may start
// while that one's last CTAs run: their tail hides its launch, its TMEM and its
// weights (loss and gradients of 65536 rows 191 -> 184 us; replayed in a graph,
// where the launches are cheaper, 1 us a step).
template <class... Params, class... Args>
void launch_after(bool after, void (*kernel)(Params...), unsigned grid, unsigned threads,
                  size_t smem, cudaStream_t st, const Args&... args)
{
    cudaLaunchConfig_t c = {};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &attr;
    c.numAttrs = after ? 1 : 0;
    cudaLaunchKernelEx(&c, kernel, Params(args)...);
}

// launches the SW kernel for N points per system (a power of two, 32..1024)
void sw_launch(bool after, const float* X, const float* T, const float* phi, int P, int N, int n_sys,
               float scale, float* loss, float* dX, cudaStream_t st)
{
    const u64 sms = (u64)std::max(1, cfs::device_sm_count());
    const u64 n_sorts = (u64)(u32)n_sys * (u64)P;
    // as many pairs of warps as there are sorts for, first one on every
    // multiprocessor; then as many CTAs as fit, each an equal share of the sorts
    const u64 pairs = (n_sorts - 1) / (u64)(32 * SW_E / N) + 1;
    const unsigned w = (unsigned)std::min<u64>(SW_PAIRS, (pairs - 1) / sms + 1);
    const unsigned grid = (unsigned)std::min<u64>(sms * SW_CTAS, (pairs - 1) / w + 1);
    auto sw = [&](auto* kernel) {
        launch_after(after, kernel, grid, 64 * w, 0, st, X, T, phi, P, n_sorts, scale, loss, dX);
    };
    switch (N) {
    case 32: sw(&sw_kernel<32>); break;
    case 64: sw(&sw_kernel<64>); break;
    case 128: sw(&sw_kernel<128>); break;
    case 256: sw(&sw_kernel<256>); break;
    case 512: sw(&sw_kernel<512>); break;
    default: sw(&sw_kernel<1024>); break;
    }
}

// ---------------------------------------------------------------------------
// Adam (Kingma & Ba) with bias correction on the FP32 master weights; writes
// the BF16 copies the GEMMs read.  t (1-based) is *step + 1.
// ---------------------------------------------------------------------------
// BF16 copy of parameter i; W2 and W3 also go transposed into wbT
// ([2][in][out]): the K-major operands of the backward GEMMs
__device__ __forceinline__ void store_bf16_weight(bf16r* wb, bf16r* wbT, int i, float wi)
{
    const bf16r b = to_bf16(wi);
    wb[i] = b;
    if (i >= OFF_W2 && i < OFF_W2 + HID * HID) {
        const int e = i - OFF_W2;
        wbT[(e % HID) * HID + e / HID] = b;
    } else if (i >= OFF_W3 && i < OFF_W3 + HID * HID) {
        const int e = i - OFF_W3;
        wbT[HID * HID + (e % HID) * HID + e / HID] = b;
    }
}

// Step size of a training run of `total` steps that started at step `first`:
// cosine decay from lr to lr_final (Loshchilov & Hutter's schedule without
// restarts); lr_final == lr keeps it constant.
__device__ __forceinline__ float lr_at(u32 step, u32 first, u32 total, float lr, float lr_final)
{
    if (lr_final == lr || total < 2) return lr;
    const float x = fminf(1.0f, (float)(step - first) / (float)(total - 1));
    return lr_final + 0.5f * (lr - lr_final) * (1.0f + cosf(3.14159265358979f * x));
}

__global__ void __launch_bounds__(256) adam_kernel(float* w, float* m, float* v,
                                                   const float* g, bf16r* wb, bf16r* wbT, int n,
                                                   u32* step, u32 t_explicit, float lr0,
                                                   float lr_final, u32 first, u32 total,
                                                   float b1, float b2, float eps,
                                                   const float* loss, float* hist)
{
    after_previous();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) {
        const u32 t = step ? (*step + 1u) : t_explicit;
        const float lr = step ? lr_at(*step, first, total, lr0, lr_final) : lr0;
        const float c1 = 1.0f - powf(b1, (float)t), c2 = 1.0f - powf(b2, (float)t);
        const float gi = g[i];
        const float mi = fmaf(b1, m[i], (1.0f - b1) * gi);
        const float vi = fmaf(b2, v[i], (1.0f - b2) * gi * gi);
        m[i] = mi;
        v[i] = vi;
        const float wi = w[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
        w[i] = wi;
        store_bf16_weight(wb, wbT, i, wi);
    }
    if (!step) return;
    // training: the block that finishes last (every block has read *step by
    // then) puts the step's loss into the run's history and counts the step;
    // step[1] holds the blocks done and is back at 0 after the last
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicInc(step + 1, gridDim.x - 1) == gridDim.x - 1) {
            const u32 at = *step - first;
            if (at < total) hist[at] = *loss;
            *step += 1u;
        }
    }
}

__global__ void to_bf16_kernel(const float* w, bf16r* wb, bf16r* wbT, int n)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) store_bf16_weight(wb, wbT, i, w[i]);
}

// ---------------------------------------------------------------------------
// training data, inputs, per-step randomness
// ---------------------------------------------------------------------------
// one system of the training family: threshold table + maps (chaos game)
// and the conditioning vector of the network
struct SysRec {
    u32 T[16];
    int n_cmp, n_maps, pad0, pad1;
    float prm[MAX_SYS_MAPS][6];
    float cond[COND];
    float t;
    float pad[3];
};

__device__ __forceinline__ uint4 philox_key(u64 seed, u32 c0, u32 c1, u32 c2, u32 c3)
{
    unsigned int rk[10][2];
    u32 k0 = (u32)seed, k1 = (u32)(seed >> 32);
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        rk[r][0] = k0; rk[r][1] = k1;
        k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
    }
    return cfs_philox_rk(rk, c0, c1, c2, c3);
}

constexpr u32 TAG_NOISE = 3, TAG_PROJ = 4, TAG_DATA = 8, TAG_DATA_INIT = 9, TAG_PICK = 10;

// network inputs of row r: Gaussian noise (Box-Muller on a Philox block),
// the conditioning vector of its system and t, written as eight 16-byte
// vectors
__device__ __forceinline__ void write_inputs_row(const SysRec& q, int r, u32 st,
                                                 const unsigned int (&rk)[10][2], bf16r* U)
{
    const uint4 w = cfs_philox_rk(rk, (u32)r, st, 0u, TAG_NOISE);
    const float u1 = ((float)(w.x >> 8) + 0.5f) * CFS_INV_2_24;
    const float u2 = (float)(w.y >> 8) * CFS_INV_2_24;
    const float rad = sqrtf(-2.0f * logf(u1));
    float sn, c;
    sincosf(6.28318530717958647692f * u2, &sn, &c);
    u32 w32[D_IN / 2];
    w32[0] = (u32)to_bf16(rad * c) | ((u32)to_bf16(rad * sn) << 16);
#pragma unroll
    for (int j = 0; j < COND / 2; ++j)
        w32[1 + j] = (u32)to_bf16(q.cond[2 * j]) | ((u32)to_bf16(q.cond[2 * j + 1]) << 16);
    w32[1 + COND / 2] = (u32)to_bf16(q.t);
#pragma unroll
    for (int j = 2 + COND / 2; j < D_IN / 2; ++j) w32[j] = 0u;
    uint4* row = reinterpret_cast<uint4*>(U + (size_t)r * D_IN);
#pragma unroll
    for (int v = 0; v < D_IN / 8; ++v)
        row[v] = make_uint4(w32[4 * v], w32[4 * v + 1], w32[4 * v + 2], w32[4 * v + 3]);
}

struct DataArgs {
    unsigned int rk[10][2];      // Philox round keys of the run's seed
    const SysRec* sys;           // [n_sys]: the family
    int n_sys;
    const u32* step;
    int N, rows, steps, P;       // rows a system, all rows, chaos-game steps, projections
    float* T;                    // [rows][2]: the targets
    bf16r* U;                    // [rows][D_IN]: the network's inputs
    float* phi;                  // [P]: the projection angles
    float *zero_a, *zero_b, *dY; // cleared for the step: gradients and loss, the
    int n_a, n_b;                // gradient copies, and dL/dY [rows][2]
};

// One training step's inputs.  Row r = s * N + j gets the chaos-game point of
// its system after `steps` steps from a uniform start (the target) and its
// network inputs; the systems are picked per step, the angles rotated.  What
// the step accumulates into is cleared here too: a launch of its own each for
// that, the picks and the angles were a sixth of the step's launches.  The
// comparisons of the map choice are unrolled over registers (looping over
// the record's thresholds in shared memory was 18 us of a 65536-row step).
__global__ void __launch_bounds__(256) data_kernel(const __grid_constant__ DataArgs a)
{
    __shared__ SysRec s_sys[256 / 32];   // rows of a block: at most 8 systems (N >= 32)
    __shared__ u32 s_sel[256 / 32];
    after_previous();
    const u32 st = *a.step;
    const int r0 = blockIdx.x * blockDim.x;
    const int first = r0 / a.N, last = min(r0 + (int)blockDim.x - 1, a.rows - 1) / a.N;
    const int tid = threadIdx.x, all = gridDim.x * blockDim.x, me = r0 + tid;
    if (tid <= last - first)
        s_sel[tid] = cfs_philox_rk(a.rk, (u32)(first + tid), st, 0u, TAG_PICK).x % (u32)a.n_sys;
    for (int e = me; e < a.n_a; e += all) a.zero_a[e] = 0.0f;
    for (int e = me; e < a.n_b; e += all) a.zero_b[e] = 0.0f;
    if (me < a.P) {
        const float u = (float)(cfs_philox_rk(a.rk, 0u, st, 0u, TAG_PROJ).x >> 8) * CFS_INV_2_24;
        a.phi[me] = ((float)me + u) * (6.28318530717958647692f / (float)a.P);
    }
    for (int j = me + all; j < a.P; j += all) {       // fewer rows than projections
        const float u = (float)(cfs_philox_rk(a.rk, 0u, st, 0u, TAG_PROJ).x >> 8) * CFS_INV_2_24;
        a.phi[j] = ((float)j + u) * (6.28318530717958647692f / (float)a.P);
    }
    __syncthreads();
    constexpr int W = (int)(sizeof(SysRec) / 4);
    for (int e = tid; e < (last - first + 1) * W; e += blockDim.x) {
        const int q = e / W, w = e % W;
        reinterpret_cast<u32*>(&s_sys[q])[w] = reinterpret_cast<const u32*>(&a.sys[s_sel[q]])[w];
    }
    __syncthreads();
    const int r = me;
    if (r >= a.rows) return;
    const SysRec& q = s_sys[r / a.N - first];
    reinterpret_cast<float2*>(a.dY)[r] = make_float2(0.0f, 0.0f);
    write_inputs_row(q, r, st, a.rk, a.U);
    // last word of each map but the last (T - 1); thresholds of 0 are below
    // every word, those past n_cmp above
    u32 lastw[MAX_SYS_MAPS - 1];
    int k0 = 0;
#pragma unroll
    for (int j = 0; j < MAX_SYS_MAPS - 1; ++j) {
        const u32 t = q.T[j];
        const bool zero = j < q.n_cmp && t == 0u;
        k0 += zero ? 1 : 0;
        lastw[j] = j < q.n_cmp && !zero ? t - 1u : 0xFFFFFFFFu;
    }
    const uint4 s0 = cfs_philox_rk(a.rk, (u32)r, st, 0u, TAG_DATA_INIT);
    float x = (float)(s0.x >> 8) * CFS_INV_2_24, y = (float)(s0.y >> 8) * CFS_INV_2_24;
    for (int n = 0; n < a.steps; n += 4) {
        const uint4 w = cfs_philox_rk(a.rk, (u32)r, st, (u32)(n >> 2), TAG_DATA);
        const u32 ws[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int h = 0; h < 4; ++h) {
            if (n + h >= a.steps) break;
            int k = k0;
#pragma unroll
            for (int j = 0; j < MAX_SYS_MAPS - 1; ++j) k += ws[h] > lastw[j] ? 1 : 0;
            const float* m = q.prm[k];
            const float nx = fmaf(m[0], x, fmaf(m[1], y, m[4]));
            const float ny = fmaf(m[2], x, fmaf(m[3], y, m[5]));
            x = nx;
            y = ny;
        }
    }
    reinterpret_cast<float2*>(a.T)[r] = make_float2(x, y);
}


// ---------------------------------------------------------------------------
// fused inference on the tensor cores: start points of many frames straight
// from noise, 128 rows (points) per tile.
// Layer 1 is a rank-2 update: only the noise varies from row to row, so
// z1 = c1 + W1[:, 0] n0 + W1[:, 1] n1 with c1 = W1[:, 2:51] u_cond + b1 (one
// vector per frame, cond_kernel); each thread computes its row's 128
// activations and writes them, BF16, as the A operand of layer 2 in shared
// memory (no-swizzle K-major core matrices: 8-column K groups 2048 B apart,
// 8-row groups 128 B apart).  Layers 2 and 3 (128 x 128) and the output
// layer (padded to N = 16) are one tcgen05.mma chain each (M = 128, K = 16
// per instruction) into the group's 128 TMEM columns; the epilogue reads
// each thread's row back (tcgen05.ld, TMEM lane = row), adds the bias,
// applies SiLU and writes the next layer's A tile in place.
// A CTA holds the weights once and runs IT_GROUPS independent warpgroups,
// each on its own tiles with its own A tile, TMEM columns and mbarrier, so
// one group's MMAs overlap the other groups' SiLU epilogues.  Every wait is
// bounded (a time-out sets the device error flag and the group stops).
// ---------------------------------------------------------------------------
// SiLU for inference: z sigma(z) = z (1 + tanh(z / 2)) / 2 with the hardware
// tanh (one special-function operation instead of an exponential and a
// reciprocal; relative error about 2^-11, below the BF16 rounding of the
// activation that follows)
__device__ __forceinline__ float silu_fast(float z)
{
    float t;
    asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(0.5f * z));
    const float h = 0.5f * z;
    return fmaf(h, t, h);
}

// c1 = W1[:, 2:51] u_cond + b1 with the BF16-rounded operands (one block
// per frame)
__global__ void cond_kernel(const bf16r* __restrict__ wb, const float* __restrict__ w,
                            const SysRec* __restrict__ recs, float* c1_all)
{
    const int j = threadIdx.x;
    if (j >= HID) return;
    const SysRec* rec = recs + blockIdx.x;
    float* c1 = c1_all + (size_t)blockIdx.x * HID;
    float acc = w[OFF_B1 + j];
    for (int q = 0; q < COND; ++q)
        acc = fmaf(from_bf16(wb[OFF_W1 + j * D_IN + 2 + q]), from_bf16(to_bf16(rec->cond[q])), acc);
    acc = fmaf(from_bf16(wb[OFF_W1 + j * D_IN + 2 + COND]), from_bf16(to_bf16(rec->t)), acc);
    c1[j] = acc;
}

constexpr int IT_GROUPS = 4;
constexpr int IT_THREADS = 128 * IT_GROUPS;
constexpr int IT_W = HID * HID * 2;            // W2 or W3 in shared memory (bytes)
constexpr int IT_N4 = 16;                      // output layer rows, padded
constexpr int IT_W4 = IT_N4 * HID * 2;
constexpr int IT_A = 128 * HID * 2;            // one group's activation tile
constexpr int IT_SMEM = 1024 + 2 * IT_W + IT_W4 + IT_GROUPS * IT_A + 256;

// byte offset of element (row r, column k) of a K-major tile whose 8-row
// groups are 128 B apart and whose 8-column K groups are `kstride` apart
__device__ __forceinline__ u32 it_off(int r, int k, u32 kstride)
{
    return (u32)(k >> 3) * kstride + (u32)r * 16u + (u32)(k & 7) * 2u;
}

// two floats to packed BF16 (round to nearest even), lo in the low half
__device__ __forceinline__ u32 it_bf16x2(float lo, float hi)
{
    u32 r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

__device__ __forceinline__ void it_st16(u32 addr, u32 a, u32 b, u32 c, u32 d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c),
                 "r"(d)
                 : "memory");
}

// a [128][K] BF16 weight matrix (16-byte aligned) into a K-major tile (K
// groups 2048 B apart), 16 bytes = 8 columns of one row at a time.  A warp's
// lanes take 8 rows x 4 K groups: 64-byte runs in global memory and no bank
// conflicts in shared memory (a row per lane was 32 lines an instruction, and
// element by element the loop took 15 us of every launch)
template <int K, int THREADS>
__device__ __forceinline__ void it_stage_weights(u32 dst, const bf16r* __restrict__ w)
{
    constexpr int KG4 = K / 32;                 // runs of 4 K groups
#pragma unroll
    for (int e = threadIdx.x; e < 128 * (K / 8); e += THREADS) {
        const int l = e & 31, run = e >> 5;
        const int n = (run / KG4) * 8 + (l & 7), kg = (run % KG4) * 4 + (l >> 3);
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(w + (size_t)n * K + 8 * kg));
        it_st16(dst + (u32)kg * 2048u + (u32)n * 16u, v.x, v.y, v.z, v.w);
    }
}

__device__ __forceinline__ void it_fence_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

template <int THREADS = 128>
__device__ __forceinline__ void it_group_sync(int g)
{
    asm volatile("bar.sync %0, %1;" ::"r"(g + 1), "n"(THREADS) : "memory");
}

// group barrier that also ANDs a flag over the group's 128 threads: every
// thread leaves with the same answer, so a time-out seen by one thread
// stops the whole group together
template <int THREADS = 128>
__device__ __forceinline__ bool it_group_all(int g, bool v)
{
    u32 r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.and.pred q, %2, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}\n"
        : "=r"(r)
        : "r"((u32)v), "r"(g + 1), "n"(THREADS)
        : "memory");
    return r != 0;
}

// frames of one inference launch: tile_begin[f] = first 128-row tile of
// frame f (tile_begin[n_sys] = all tiles), its c1 vector, row count, seed
// and output (SoA [2][count])
struct InferFrames {
    const float* c1;          // [n_sys][HID]
    const u32* tile_begin;    // [n_sys + 1]
    const u32* count;         // [n_sys]
    const u64* seed;          // [n_sys]
    float* const* out;        // [n_sys]
    int n_sys;
};

__global__ void __launch_bounds__(IT_THREADS, 1) infer_tc_kernel(const bf16r* __restrict__ wb,
                                                                 const float* __restrict__ w,
                                                                 const InferFrames fs)
{
    extern __shared__ unsigned char it_raw[];
    unsigned char* sm = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(it_raw) + 1023) & ~(uintptr_t)1023);
    const u32 sW2 = smem_addr(sm), sW3 = sW2 + IT_W, sW4 = sW3 + IT_W;
    const u32 sA0 = sW4 + IT_W4;
    u64* bars = reinterpret_cast<u64*>(sm + 2 * IT_W + IT_W4 + IT_GROUPS * IT_A);
    u32* s_tmem = reinterpret_cast<u32*>(bars + IT_GROUPS);
    __shared__ __align__(16) float s_w10[HID], s_w11[HID], s_b2[HID], s_b3[HID], s_b4[4];
    __shared__ int s_err;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    // weights into the B-operand layout (rows = output features n, K = inputs)
    it_stage_weights<HID, IT_THREADS>(sW2, wb + OFF_W2);
    it_stage_weights<HID, IT_THREADS>(sW3, wb + OFF_W3);
    for (int e = tid; e < IT_N4 * HID; e += IT_THREADS) {
        const int n = e / HID, k = e % HID;
        *reinterpret_cast<bf16r*>(sm + 2 * IT_W + it_off(n, k, (u32)IT_N4 * 16u)) =
            n < D_OUT ? wb[OFF_W4 + e] : (bf16r)0;
    }
    for (int j = tid; j < HID; j += IT_THREADS) {
        s_w10[j] = from_bf16(wb[OFF_W1 + j * D_IN]);
        s_w11[j] = from_bf16(wb[OFF_W1 + j * D_IN + 1]);
        s_b2[j] = w[OFF_B2 + j];
        s_b3[j] = w[OFF_B3 + j];
    }
    if (tid < 2) s_b4[tid] = w[OFF_B4 + tid];
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :
                     : "r"(smem_addr(s_tmem)), "r"(128u * IT_GROUPS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        s_err = 0;
        for (int g = 0; g < IT_GROUPS; ++g) mbar_init(smem_addr(&bars[g]), 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    it_fence_async_smem();          // the weights, written by st.shared, feed the MMAs
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    const int g = warp >> 2, wq = warp & 3, r = wq * 32 + lane;   // r: row in the tile
    const u32 sA = sA0 + (u32)(g * IT_A);
    const u32 bar = smem_addr(&bars[g]);
    const u32 tcol = *s_tmem + (u32)(g * 128);                    // the group's columns
    const u32 tlane = tcol + ((u32)(wq * 32) << 16);              // this warp's lanes
    const bool issuer = wq == 0 && lane == 0;
    const u32 idesc128 = tc_idesc(128), idesc16 = tc_idesc(IT_N4);
    u32 phase = 0;
    int pending = 0;               // commits issued and not yet waited for (issuer)
    bool ok = true;

    // layer k's MMAs on the A tile into the group's columns, committed to bar
    auto mma_layer = [&](u32 sW, u32 lbo_w, u32 idesc) {
        it_fence_async_smem();
        tc_fence_before();
        it_group_sync(g);
        if (issuer) {
            tc_fence_after();
            for (int kk = 0; kk < HID / 16; ++kk)
                tc_mma(tcol, tc_desc_kn(sA + (u32)kk * 4096u, 2048u, 128u),
                       tc_desc_kn(sW + (u32)kk * 2u * lbo_w, lbo_w, 128u), idesc,
                       kk > 0 ? 1u : 0u);
            tc_commit(bar);
            pending = 1;
        }
    };
    auto wait_layer = [&]() -> bool {
        const bool done = it_group_all(g, mbar_wait(bar, phase));
        if (done) {
            phase ^= 1u;
            if (issuer) pending = 0;
        }
        tc_fence_after();
        return done;
    };
    // epilogue of a hidden layer: bias, SiLU, BF16, written as the next A tile
    auto hidden_epilogue = [&](const float* bias) {
        const float4* b4 = reinterpret_cast<const float4*>(bias);
        tc_for_columns(tlane, [&](int c0, const u32 (&v)[16]) {
            u32 q[8];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 bb = b4[c0 / 4 + j];
                q[2 * j] = it_bf16x2(silu_fast(__uint_as_float(v[4 * j]) + bb.x),
                                     silu_fast(__uint_as_float(v[4 * j + 1]) + bb.y));
                q[2 * j + 1] = it_bf16x2(silu_fast(__uint_as_float(v[4 * j + 2]) + bb.z),
                                         silu_fast(__uint_as_float(v[4 * j + 3]) + bb.w));
            }
            it_st16(sA + it_off(r, c0, 2048u), q[0], q[1], q[2], q[3]);
            it_st16(sA + it_off(r, c0 + 8, 2048u), q[4], q[5], q[6], q[7]);
        });
    };

    const u32 tiles = fs.tile_begin[fs.n_sys];
    // a tile's frame, row and noise; those of the group's next tile are
    // computed while this tile's first MMAs run
    struct Tile {
        int f;
        u32 row;
        float n0, n1;
    };
    auto tile_of = [&](u32 tile) {
        // the frame of this tile: last f with tile_begin[f] <= tile
        int lo = 0, hi = fs.n_sys;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (fs.tile_begin[mid] <= tile) lo = mid; else hi = mid;
        }
        Tile t;
        t.f = lo;
        t.row = (tile - fs.tile_begin[lo]) * 128u + (u32)r;
        // Box-Muller on Philox (row, 0, 0, 3)
        const uint4 q = philox_key(fs.seed[lo], t.row, 0u, 0u, TAG_NOISE);
        const float u1 = ((float)(q.x >> 8) + 0.5f) * CFS_INV_2_24;
        const float u2 = (float)(q.y >> 8) * CFS_INV_2_24;
        const float rad = sqrtf(-2.0f * logf(u1));
        float sn, cs;
        sincosf(6.28318530717958647692f * u2, &sn, &cs);
        t.n0 = from_bf16(to_bf16(rad * cs));
        t.n1 = from_bf16(to_bf16(rad * sn));
        return t;
    };
    u32 tile = blockIdx.x * IT_GROUPS + (u32)g;
    Tile next = {};
    if (tile < tiles) next = tile_of(tile);
    for (; tile < tiles; tile += gridDim.x * IT_GROUPS) {
        const int f = next.f;
        const u32 row = next.row;
        const float n0 = next.n0, n1 = next.n1;
        const u32 n = fs.count[f];
        const float* c1 = fs.c1 + (size_t)f * HID;
        // layer 1 (rank-2 update) into the A tile (16-byte loads of c1 and
        // of the two noise columns of W1, shared by the whole group)
        const float4* c14 = reinterpret_cast<const float4*>(c1);
        const float4* w04 = reinterpret_cast<const float4*>(s_w10);
        const float4* w14 = reinterpret_cast<const float4*>(s_w11);
        // (unrolled: the loads of one group of columns hide behind the others'
        // tanh; one group at a time took a fifth of the kernel, 206 us for 256 x
        // 4096 samples against 167)
#pragma unroll 8
        for (int c0 = 0; c0 < HID; c0 += 8) {
            u32 q[4];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const float4 cc = __ldg(c14 + c0 / 4 + h);
                const float4 a0 = w04[c0 / 4 + h], a1 = w14[c0 / 4 + h];
                q[2 * h] = it_bf16x2(silu_fast(fmaf(a1.x, n1, fmaf(a0.x, n0, cc.x))),
                                     silu_fast(fmaf(a1.y, n1, fmaf(a0.y, n0, cc.y))));
                q[2 * h + 1] = it_bf16x2(silu_fast(fmaf(a1.z, n1, fmaf(a0.z, n0, cc.z))),
                                         silu_fast(fmaf(a1.w, n1, fmaf(a0.w, n0, cc.w))));
            }
            it_st16(sA + it_off(r, c0, 2048u), q[0], q[1], q[2], q[3]);
        }
        mma_layer(sW2, 2048u, idesc128);
        if (tile + gridDim.x * IT_GROUPS < tiles) next = tile_of(tile + gridDim.x * IT_GROUPS);
        if (!(ok = wait_layer())) break;
        hidden_epilogue(s_b2);
        mma_layer(sW3, 2048u, idesc128);
        if (!(ok = wait_layer())) break;
        hidden_epilogue(s_b3);
        mma_layer(sW4, (u32)IT_N4 * 16u, idesc16);
        if (!(ok = wait_layer())) break;
        float y[16];
        tc_ld16(tlane, y);
        tc_fence_before();          // TMEM read: the next tile's MMAs may overwrite it
        if (row < n) {
            float* out = fs.out[f];
            out[row] = y[0] + s_b4[0];
            out[(size_t)n + row] = y[1] + s_b4[1];
        }
    }
    if (!ok) {
        atomicExch(&s_err, 1);
        // the MMAs of an unfinished commit complete before TMEM is freed
        if (issuer && pending) mbar_wait(bar, phase);
    }
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && s_err) atomicOr(&g_tc_error, (unsigned)CFS_DEVICE_ERR_TC_TIMEOUT);
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*s_tmem),
                     "r"(128u * IT_GROUPS)
                     : "memory");
    }
}

// ---------------------------------------------------------------------------
// The training forward pass fused per 128-row tile (the same structure as
// infer_tc_kernel): layer 1 (K = 64), layer 2 and layer 3 run as tcgen05.mma
// chains into the group's TMEM columns, each epilogue adding the bias,
// applying SiLU and writing the next A tile in place; the output layer itself
// (N = 2) runs on the CUDA cores in the layer-3 epilogue.  What the backward
// pass reads is written on the way, row-major: H1, H2 and Z3.
// All tiles are in the 128-byte-swizzled K-major layout (128 rows of 128
// bytes a block), which the MMAs read and TMA moves: the weights and a tile of
// inputs arrive, and H1 and H2 leave straight from the A tile while the next
// layer's MMAs read it, with no thread's loads or stores.  The epilogues' two
// special-function operations an element (13 us at 65536 rows) are the bound
// left: 27.5 us there.  The same arithmetic took 53 us with a row per lane for
// every load and store, and 40 through shared memory in whole lines.
// ---------------------------------------------------------------------------
constexpr int TF_GROUPS = 4;
constexpr int TF_THREADS = 128 * TF_GROUPS;
constexpr int TF_W1 = HID * D_IN * 2;          // 16 KB
constexpr int TF_BLOCK = 128 * 128;            // 128 rows of 128 bytes
constexpr int TF_SMEM = 1024 + TF_W1 + 2 * IT_W + TF_GROUPS * IT_A + 256;

struct TrainFwdMaps {
    CUtensorMap U, W1, W2, W3;     // boxes of 128 rows x 64 BF16
    CUtensorMap H1, H2, Z3;        // Z3 as [B][2 * HID] 16-bit words: 32 floats a box
};

struct TrainFwdArgs {
    int B;
    float* Y;                      // [B][2]
};

// a box of shared memory to the tensor map's matrix at (x, y); rows and
// columns outside it are not written
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, u32 src, int x, int y)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];" ::"l"(
                     reinterpret_cast<u64>(map)),
                 "r"(x), "r"(y), "r"(src)
                 : "memory");
}

__device__ __forceinline__ void tma_store_commit()
{
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// all but the newest N of this thread's store groups have read their source
template <int N>
__device__ __forceinline__ void tma_store_read_wait()
{
    asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}

__global__ void __launch_bounds__(TF_THREADS, 1) train_fwd_kernel(
    const __grid_constant__ TrainFwdMaps m, const bf16r* __restrict__ wb,
    const float* __restrict__ w, const TrainFwdArgs g)
{
    extern __shared__ unsigned char tf_raw[];
    unsigned char* sm = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(tf_raw) + 1023) & ~(uintptr_t)1023);
    const u32 sW1 = smem_addr(sm), sW2 = sW1 + TF_W1, sW3 = sW2 + IT_W;
    const u32 sA0 = sW3 + IT_W;
    // barriers: weights, then per group the inputs and the MMAs
    u64* bars = reinterpret_cast<u64*>(sm + TF_W1 + 2 * IT_W + TF_GROUPS * IT_A);
    u32* s_tmem = reinterpret_cast<u32*>(bars + 1 + 2 * TF_GROUPS);
    __shared__ __align__(16) float s_b1[HID], s_b2[HID], s_b3[HID], s_w4[D_OUT][HID];
    __shared__ float s_b4[2];
    __shared__ int s_err;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const u32 wfull = smem_addr(&bars[0]);

    for (int j = tid; j < HID; j += TF_THREADS) {
        s_b1[j] = w[OFF_B1 + j];
        s_b2[j] = w[OFF_B2 + j];
        s_b3[j] = w[OFF_B3 + j];
        s_w4[0][j] = from_bf16(wb[OFF_W4 + j]);
        s_w4[1][j] = from_bf16(wb[OFF_W4 + HID + j]);
    }
    if (tid < 2) s_b4[tid] = w[OFF_B4 + tid];
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :
                     : "r"(smem_addr(s_tmem)), "r"(128u * TF_GROUPS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        s_err = 0;
        for (int q = 0; q < 1 + 2 * TF_GROUPS; ++q) mbar_init(smem_addr(&bars[q]), 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_expect_tx(wfull, (u32)(TF_W1 + 2 * IT_W));
        tma_load_2d(sW1, &m.W1, 0, 0, wfull);
        for (int c = 0; c < 2; ++c) {
            tma_load_2d(sW2 + c * TF_BLOCK, &m.W2, 64 * c, 0, wfull);
            tma_load_2d(sW3 + c * TF_BLOCK, &m.W3, 64 * c, 0, wfull);
        }
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    after_previous();       // (the weights are older)

    const int gi = warp >> 2, wq = warp & 3, r = wq * 32 + lane;
    const u32 sA = sA0 + (u32)(gi * IT_A);
    const u32 ubar = smem_addr(&bars[1 + gi]), bar = smem_addr(&bars[1 + TF_GROUPS + gi]);
    const u32 tcol = *s_tmem + (u32)(gi * 128);
    const u32 tlane = tcol + ((u32)(wq * 32) << 16);
    const bool issuer = wq == 0 && lane == 0;
    const u32 idesc = tc_idesc(128);
    u32 phase = 0, uphase = 0;
    int pending = 0;
    bool ok = true;

    // 16 bytes of this thread's row: chunk c of the block at `block`
    auto chunk = [&](u32 block, int c) { return block + (u32)r * 128u + (u32)((c ^ (r & 7)) * 16); };
    // the issuer's part of a layer: the MMAs of the A tile with sW
    auto issue = [&](u32 sW, int K) {
        tc_fence_after();
        for (int kk = 0; kk < K / 16; ++kk) {
            const u32 at = (u32)((kk >> 2) * TF_BLOCK + (kk & 3) * 32);
            tc_mma(tcol, tc_desc_ksw(sA + at), tc_desc_ksw(sW + at), idesc, kk > 0 ? 1u : 0u);
        }
        tc_commit(bar);
        pending = 1;
    };
    // layers 2 and 3: the A tile just written, to the MMAs and to H
    auto mma_layer = [&](u32 sW, const CUtensorMap* H, int row0) {
        it_fence_async_smem();
        tc_fence_before();
        it_group_sync(gi);
        if (issuer) {
            issue(sW, HID);
            tma_store_2d(H, sA, 0, row0);
            tma_store_2d(H, sA + TF_BLOCK, 64, row0);
            tma_store_commit();
        }
    };
    // the layer's accumulator is complete, and the A tile has been read
    auto wait_layer = [&](bool in_ok) -> bool {
        const bool mine = in_ok && mbar_wait(bar, phase);
        if (issuer) tma_store_read_wait<0>();
        const bool done = it_group_all(gi, mine);
        if (done) {
            phase ^= 1u;
            if (issuer) pending = 0;
        }
        tc_fence_after();
        return done;
    };
    // epilogue of layers 1 and 2: H = SiLU(acc + b) as BF16 into the next A
    // tile
    auto hidden_epilogue = [&](const float* bias) {
        const float4* b4 = reinterpret_cast<const float4*>(bias);
        tc_for_columns(tlane, [&](int c0, const u32 (&acc)[16]) {
            u32 q[8];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float4 bb = b4[c0 / 4 + j];
                q[2 * j] = pack_bf16x2(silu_f(__uint_as_float(acc[4 * j]) + bb.x),
                                       silu_f(__uint_as_float(acc[4 * j + 1]) + bb.y));
                q[2 * j + 1] = pack_bf16x2(silu_f(__uint_as_float(acc[4 * j + 2]) + bb.z),
                                           silu_f(__uint_as_float(acc[4 * j + 3]) + bb.w));
            }
            const u32 block = sA + (u32)((c0 >> 6) * TF_BLOCK);
            const int c = (c0 & 63) / 8;
            it_st16(chunk(block, c), q[0], q[1], q[2], q[3]);
            it_st16(chunk(block, c + 1), q[4], q[5], q[6], q[7]);
        });
    };

    const int n_tiles = (g.B + 127) / 128;
    for (int tile = blockIdx.x * TF_GROUPS + gi; tile < n_tiles; tile += gridDim.x * TF_GROUPS) {
        const int row0 = tile * 128, row = row0 + r;
        const bool in = row < g.B;
        bool go = true;
        if (issuer) {
            // (the A tile is free: the last tile's stores have read it, below)
            mbar_expect_tx(ubar, (u32)TF_BLOCK);
            tma_load_2d(sA, &m.U, 0, row0, ubar);
            go = mbar_wait(ubar, uphase) && mbar_wait(wfull, 0u);
            if (go) issue(sW1, D_IN);
        }
        uphase ^= 1u;
        if (!(ok = wait_layer(go))) break;
        hidden_epilogue(s_b1);
        mma_layer(sW2, &m.H1, row0);
        if (!(ok = wait_layer(true))) break;
        hidden_epilogue(s_b2);
        mma_layer(sW3, &m.H2, row0);
        if (!(ok = wait_layer(true))) break;
        // layer 3: Z3 (FP32) out, and the output layer on the BF16 activations
        // (which the backward pass forms again from Z3), columns in order.  Z3
        // leaves in quarters of 32 columns through the A tile's two blocks
        float y0 = 0.0f, y1 = 0.0f;
        u32 a[16], b[16];
        tc_ld16_nowait(tlane, a);
#pragma unroll 1
        for (int q = 0; q < 4; ++q) {
            const u32 block = sA + (u32)((q & 1) * TF_BLOCK);
            auto work = [&](int c0, const u32 (&v)[16]) {
                const float4* b4 = reinterpret_cast<const float4*>(s_b3 + c0);
                const float4* p0 = reinterpret_cast<const float4*>(&s_w4[0][c0]);
                const float4* p1 = reinterpret_cast<const float4*>(&s_w4[1][c0]);
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const float4 bb = b4[j], w0 = p0[j], w1 = p1[j];
                    const float z[4] = {
                        __uint_as_float(v[4 * j]) + bb.x, __uint_as_float(v[4 * j + 1]) + bb.y,
                        __uint_as_float(v[4 * j + 2]) + bb.z, __uint_as_float(v[4 * j + 3]) + bb.w};
                    const u32 q0 = pack_bf16x2(silu_f(z[0]), silu_f(z[1]));
                    const u32 q1 = pack_bf16x2(silu_f(z[2]), silu_f(z[3]));
                    const float h[4] = {__uint_as_float(q0 << 16), __uint_as_float(q0 & 0xFFFF0000u),
                                        __uint_as_float(q1 << 16), __uint_as_float(q1 & 0xFFFF0000u)};
                    y0 = fmaf(h[0], w0.x, y0); y1 = fmaf(h[0], w1.x, y1);
                    y0 = fmaf(h[1], w0.y, y0); y1 = fmaf(h[1], w1.y, y1);
                    y0 = fmaf(h[2], w0.z, y0); y1 = fmaf(h[2], w1.z, y1);
                    y0 = fmaf(h[3], w0.w, y0); y1 = fmaf(h[3], w1.w, y1);
                    it_st16(chunk(block, (c0 & 31) / 4 + j), __float_as_uint(z[0]),
                            __float_as_uint(z[1]), __float_as_uint(z[2]), __float_as_uint(z[3]));
                }
            };
            if (q >= 2) {       // the block's last quarter has left
                if (issuer) tma_store_read_wait<1>();
                it_group_sync(gi);
            }
            tc_wait_ld(a);
            tc_ld16_nowait(tlane + (u32)(32 * q + 16), b);
            work(32 * q, a);
            tc_wait_ld(b);
            if (q < 3) tc_ld16_nowait(tlane + (u32)(32 * q + 32), a);
            work(32 * q + 16, b);
            it_fence_async_smem();
            if (q == 3) tc_fence_before();   // TMEM read: the next tile's MMAs may overwrite it
            it_group_sync(gi);
            if (issuer) {
                tma_store_2d(&m.Z3, block, 64 * q, row0);
                tma_store_commit();
                if (q == 3) tma_store_read_wait<0>();
            }
        }
        if (in) {
            g.Y[2 * (size_t)row] = y0 + s_b4[0];
            g.Y[2 * (size_t)row + 1] = y1 + s_b4[1];
        }
    }
    if (!ok) {
        atomicExch(&s_err, 1);
        if (issuer) {
            if (pending) mbar_wait(bar, phase);
            mbar_wait(ubar, uphase ^ 1u);      // the last tile's inputs
        }
    }
    // the copies into and out of this CTA's shared memory are over before it
    // may leave: the weights (all of them, also where no tile waited for them)
    // and every group's stores
    if (tid == 0) mbar_wait(wfull, 0u);
    if (issuer) asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    if (tid == 0 && s_err) atomicOr(&g_tc_error, (unsigned)CFS_DEVICE_ERR_TC_TIMEOUT);
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*s_tmem),
                     "r"(128u * TF_GROUPS)
                     : "memory");
    }
}

// ---------------------------------------------------------------------------
// The input gradients of training in one launch, per tile of 128 rows:
//   dZ2 = (dZ3 W3) * silu'(H1 W2^T + b2),  dZ1 = (dZ2 W2) * silu'(U W1^T + b1),
// and the column sums of both (the bias gradients).  A group of 8 warps takes a
// tile, two groups a CTA.  A layer's two products are two accumulators of one
// MMA chain: the gradient, whose weights are an MN-major operand (their rows
// are the contraction), and the pre-activation again, the same MMAs the
// forward ran on the same bits, so no Z has to be stored.  The epilogue writes
// dZ2 over dZ3, the next layer's A tile, from where TMA takes it out while
// the MMAs read it; U and the next tile's H1 arrive under the epilogues.
// All tiles are TMA boxes of 128 rows x 64 columns (128-byte swizzle).  Each
// wait is bounded; a time-out sets g_tc_error and the group stops.
// What it measured (65536 rows): 32.4 us, where a launch a layer took 22.4 us each
// and read dZ2 back.
// ---------------------------------------------------------------------------
constexpr int BR_GROUPS = 2;
constexpr int BR_GT = 256;                     // threads of a group
constexpr int BR_THREADS = BR_GT * BR_GROUPS;
constexpr int BR_WEIGHTS = 2 * IT_W + TF_W1;
constexpr int BR_SLOT = 2 * IT_A;              // a group's dZ, and H1 or U
constexpr int BR_SMEM = 1024 + BR_WEIGHTS + BR_GROUPS * BR_SLOT + 256;

struct BackRowsMaps {
    CUtensorMap W1, W2, W3, dZ3, H1, U, dZ2, dZ1;
};

struct BackRowsArgs {
    int B;
    const float* b2;
    const float* b1;
    float* col2;                   // bias gradient partials, [TC_COPIES][HID]: CTA b adds
    float* col1;                   // its column sums into copy b % TC_COPIES
};

__global__ void __launch_bounds__(BR_THREADS, 1) back_rows_kernel(
    const __grid_constant__ BackRowsMaps m, const __grid_constant__ BackRowsArgs g)
{
    extern __shared__ unsigned char br_raw[];
    unsigned char* sm = reinterpret_cast<unsigned char*>(
        (reinterpret_cast<uintptr_t>(br_raw) + 1023) & ~(uintptr_t)1023);
    const u32 sW3 = smem_addr(sm), sW2 = sW3 + IT_W, sW1 = sW2 + IT_W;
    // barriers: weights, then per group dZ3, H1, U and the MMAs
    u64* bars = reinterpret_cast<u64*>(sm + BR_WEIGHTS + BR_GROUPS * BR_SLOT);
    u32* s_tmem = reinterpret_cast<u32*>(bars + 1 + 4 * BR_GROUPS);
    __shared__ __align__(16) float s_b[2][HID];
    __shared__ float s_col[2][HID];
    __shared__ int s_err;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const u32 wfull = smem_addr(&bars[0]);

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :
                     : "r"(smem_addr(s_tmem)), "r"(256u * BR_GROUPS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid < HID) {
        s_b[0][tid] = g.b2[tid];
        s_b[1][tid] = g.b1[tid];
        s_col[0][tid] = s_col[1][tid] = 0.0f;
    }
    if (tid == 0) {
        s_err = 0;
        for (int q = 0; q < 1 + 4 * BR_GROUPS; ++q) mbar_init(smem_addr(&bars[q]), 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        mbar_expect_tx(wfull, (u32)BR_WEIGHTS);
        for (int c = 0; c < 2; ++c) {
            tma_load_2d(sW3 + c * TF_BLOCK, &m.W3, 64 * c, 0, wfull);
            tma_load_2d(sW2 + c * TF_BLOCK, &m.W2, 64 * c, 0, wfull);
        }
        tma_load_2d(sW1, &m.W1, 0, 0, wfull);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();

    after_previous();       // (the weights are older)

    const int gi = tid / BR_GT, quad = warp & 3, half = (warp >> 2) & 1;
    const int r = quad * 32 + lane;
    const u32 sD = sW1 + TF_W1 + (u32)(gi * BR_SLOT), sH = sD + IT_A;
    const u32 dbar = smem_addr(&bars[1 + 4 * gi]), hbar = dbar + 8, ubar = dbar + 16,
              bar = dbar + 24;
    const u32 tcol = *s_tmem + (u32)(256 * gi);
    // this thread's row and half of the columns
    const u32 tlane = tcol + ((u32)(quad * 32) << 16) + (u32)(64 * half);
    const bool issuer = tid % BR_GT == 0;
    // the weights of the gradient are MN-major B operands: transpose bit 16
    const u32 idesc = tc_idesc(HID), idesc_mn = idesc | (1u << 16);
    const int n_tiles = (g.B + 127) / 128, step = (int)gridDim.x * BR_GROUPS;
    const int first = (int)blockIdx.x * BR_GROUPS + gi;
    u32 phase = 0;
    int pending = 0, n_d = 0, n_h = 0, n_u = 0;    // MMAs and loads (issuer)
    bool ok = true;

    auto load_d = [&](int row0) {
        mbar_expect_tx(dbar, (u32)IT_A);
        tma_load_2d(sD, &m.dZ3, 0, row0, dbar);
        tma_load_2d(sD + TF_BLOCK, &m.dZ3, 64, row0, dbar);
        ++n_d;
    };
    auto load_h = [&](int row0) {
        mbar_expect_tx(hbar, (u32)IT_A);
        tma_load_2d(sH, &m.H1, 0, row0, hbar);
        tma_load_2d(sH + TF_BLOCK, &m.H1, 64, row0, hbar);
        ++n_h;
    };
    auto loaded = [&](u32 b, int n) { return n == 0 || mbar_wait(b, (u32)(n - 1) & 1u); };
    // the gradient of the tile in sD through W into columns 0 .. 127, the
    // pre-activation of the K columns in sH by WZ into the next 128
    auto issue = [&](u32 W, u32 WZ, int K) {
        tc_fence_after();
        for (int kk = 0; kk < HID / 16; ++kk)
            tc_mma(tcol, tc_desc_ksw(sD + (u32)((kk >> 2) * TF_BLOCK + (kk & 3) * 32)),
                   tc_desc_mn(W + (u32)(kk * 2048), TF_BLOCK), idesc_mn, kk > 0 ? 1u : 0u);
        for (int kk = 0; kk < K / 16; ++kk) {
            const u32 at = (u32)((kk >> 2) * TF_BLOCK + (kk & 3) * 32);
            tc_mma(tcol + 128u, tc_desc_ksw(sH + at), tc_desc_ksw(WZ + at), idesc,
                   kk > 0 ? 1u : 0u);
        }
        tc_commit(bar);
        pending = 1;
    };
    // the MMAs are complete, and the copy out of sD has read it
    auto wait_layer = [&](bool in_ok) -> bool {
        const bool mine = in_ok && mbar_wait(bar, phase);
        if (issuer) tma_store_read_wait<0>();
        const bool done = it_group_all<BR_GT>(gi, mine);
        if (done) {
            phase ^= 1u;
            if (issuer) pending = 0;
        }
        tc_fence_after();
        return done;
    };
    // dZ of 16 columns from c0 (of this thread's half) into sD, their sums over
    // the warp's rows added to col (lanes 2c and 2c + 1: column c)
    auto columns = [&](int c0, const u32 (&acc)[16], const u32 (&z)[16], const float* bias, bool in,
                       float& col) {
        float h[16];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const float4 bb = *reinterpret_cast<const float4*>(bias + 64 * half + c0 + 4 * j);
            const float b[4] = {bb.x, bb.y, bb.z, bb.w};
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int e = 4 * j + q;
                const float d = silu_grad_f(__uint_as_float(z[e]) + b[q]);
                h[e] = in ? __uint_as_float(acc[e]) * d : 0.0f;
            }
        }
        u32 p[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) p[j] = pack_bf16x2(h[2 * j], h[2 * j + 1]);
        const u32 line = sD + (u32)(half * TF_BLOCK + r * 128);
        const int c = c0 / 8;
        it_st16(line + (u32)((c ^ (r & 7)) * 16), p[0], p[1], p[2], p[3]);
        it_st16(line + (u32)(((c + 1) ^ (r & 7)) * 16), p[4], p[5], p[6], p[7]);
        col += warp_colsum16(h);
    };
    float col[2][4] = {};
    auto epilogue = [&](const float* bias, bool in, float (&cs)[4]) {
        u32 a0[16], z0[16], a1[16], z1[16];
        tc_ld16_nowait(tlane, a0);
        tc_ld16_nowait(tlane + 128u, z0);
#pragma unroll
        for (int q = 0; q < 4; q += 2) {
            tc_wait_ld(a0);
            tc_wait_ld(z0);
            tc_ld16_nowait(tlane + (u32)(16 * q + 16), a1);
            tc_ld16_nowait(tlane + (u32)(16 * q + 144), z1);
            columns(16 * q, a0, z0, bias, in, cs[q]);
            tc_wait_ld(a1);
            tc_wait_ld(z1);
            if (q == 0) {
                tc_ld16_nowait(tlane + 32u, a0);
                tc_ld16_nowait(tlane + 160u, z0);
            }
            columns(16 * q + 16, a1, z1, bias, in, cs[q + 1]);
        }
        it_fence_async_smem();
        tc_fence_before();
        it_group_sync<BR_GT>(gi);
    };
    auto store = [&](const CUtensorMap* map, int row0) {
        tma_store_2d(map, sD, 0, row0);
        tma_store_2d(map, sD + TF_BLOCK, 64, row0);
        tma_store_commit();
    };

    if (issuer && first < n_tiles) {
        load_d(first * 128);
        load_h(first * 128);
    }
    for (int tile = first; tile < n_tiles; tile += step) {
        const int row0 = tile * 128, next0 = row0 + step * 128;
        const bool in = row0 + r < g.B, more = tile + step < n_tiles;
        bool go = true;
        if (issuer) {
            go = loaded(dbar, n_d) && loaded(hbar, n_h) && mbar_wait(wfull, 0u);
            if (go) issue(sW3, sW2, HID);
        }
        if (!(ok = wait_layer(go))) break;
        if (issuer) {                   // H1 has been read
            mbar_expect_tx(ubar, (u32)TF_BLOCK);
            tma_load_2d(sH, &m.U, 0, row0, ubar);
            ++n_u;
        }
        epilogue(s_b[0], in, col[0]);
        if (issuer) {
            go = loaded(ubar, n_u);
            if (go) issue(sW2, sW1, D_IN);
            store(&m.dZ2, row0);
        }
        if (!(ok = wait_layer(go))) break;
        if (issuer && more) load_h(next0);
        epilogue(s_b[1], in, col[1]);
        if (issuer) {
            store(&m.dZ1, row0);
            tma_store_read_wait<0>();
            if (more) load_d(next0);
        }
    }
    if (!ok) {
        atomicExch(&s_err, 1);
        if (issuer && pending) mbar_wait(bar, phase);
    }
    // the copies into and out of this CTA's shared memory are over before it
    // may leave
    if (tid == 0) mbar_wait(wfull, 0u);
    if (issuer) {
        loaded(dbar, n_d);
        loaded(hbar, n_h);
        loaded(ubar, n_u);
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    if (!(lane & 1)) {
#pragma unroll
        for (int l = 0; l < 2; ++l)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                atomicAdd(&s_col[l][64 * half + 16 * q + (lane >> 1)], col[l][q]);
    }
    tc_fence_before();
    __syncthreads();
    if (!s_err && tid < 2 * HID) {
        const float v = s_col[tid / HID][tid % HID];
        if (v != 0.0f)
            atomicAdd((tid < HID ? g.col2 : g.col1) + (blockIdx.x % TC_COPIES) * HID + tid % HID, v);
    }
    if (tid == 0 && s_err) atomicOr(&g_tc_error, (unsigned)CFS_DEVICE_ERR_TC_TIMEOUT);
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(*s_tmem),
                     "r"(256u * BR_GROUPS)
                     : "memory");
    }
}

}  // namespace

// ---------------------------------------------------------------------------
// host object
// ---------------------------------------------------------------------------
struct cfs_sampler {
    int device = 0;
    float* w = nullptr;      // master params [N_PARAMS]
    float* m = nullptr;
    float* v = nullptr;
    bf16r* wb = nullptr;     // bf16 copies
    bf16r* wbT = nullptr;    // bf16 W2^T, W3^T ([2][in][out]) for the backward GEMMs
    float* bias_part = nullptr;   // PART_FLOATS gradient partial sums (part_reduce_kernel)
    u32* d_step = nullptr;   // Adam step counter (device)
    u32 step = 0;            // host mirror (checkpoints)
    // inference workspace for n frames (grown on demand): records, c1,
    // tile offsets, counts, seeds, output pointers
    int cap_frames = 0;
    unsigned char* inf = nullptr;
    unsigned char* inf_host = nullptr;   // pinned staging of the same layout
    cudaEvent_t uploaded = nullptr;      // the staging buffer's last upload
    bool upload_pending = false;
    // activations for B rows (grown on demand)
    int cap_rows = 0;
    int ldt = 0;             // row stride of the transposed copies (TC_M)
    unsigned char* act = nullptr;
    float *Z1, *Z2, *Z3, *Y;
    bf16r *H1, *H2, *H3, *dZ1, *dZ2, *dZ3;
    // transposed copies [features][ldt]: the K-major operands of dW = dZ^T A
    // of batches of fewer than DW_ROWS rows (written up to TC_M)
    bf16r *UT, *H1T, *H2T, *dZ1T, *dZ2T, *dZ3T;
};

namespace {
using namespace cfs;

cfs_status ensure_rows(cfs_sampler* s, int B)
{
    if (B <= s->cap_rows) return CFS_OK;
    if (s->act) cudaFree(s->act);
    s->act = nullptr;
    s->cap_rows = 0;
    const size_t fz = (size_t)B * HID * 4, fh = (size_t)B * HID * 2;
    const int ldt = TC_M;    // the transposed copies serve batches of fewer rows only
    const size_t ft = (size_t)ldt * HID * 2, fu = (size_t)ldt * D_IN * 2;
    const size_t bytes = 3 * fz + (size_t)B * 2 * 4 + 6 * fh + 5 * ft + fu + 13 * 256;
    cfs_status st = check_cuda(cudaMalloc(&s->act, bytes), "cudaMalloc(sampler activations)");
    if (st != CFS_OK) return st;
    unsigned char* p = s->act;
    auto take = [&](size_t n) {
        unsigned char* r = p;
        p += (n + 255) & ~(size_t)255;
        return r;
    };
    s->Z1 = (float*)take(fz); s->Z2 = (float*)take(fz); s->Z3 = (float*)take(fz);
    s->Y = (float*)take((size_t)B * 2 * 4);
    s->H1 = (bf16r*)take(fh); s->H2 = (bf16r*)take(fh); s->H3 = (bf16r*)take(fh);
    s->dZ1 = (bf16r*)take(fh); s->dZ2 = (bf16r*)take(fh); s->dZ3 = (bf16r*)take(fh);
    s->UT = (bf16r*)take(fu);
    s->H1T = (bf16r*)take(ft); s->H2T = (bf16r*)take(ft);
    s->dZ1T = (bf16r*)take(ft); s->dZ2T = (bf16r*)take(ft); s->dZ3T = (bf16r*)take(ft);
    s->ldt = ldt;
    s->cap_rows = B;
    return CFS_OK;
}

// D = A B^T on the tensor cores (both operands K-major; ATOMIC adds it to C)
cfs_status tc_gemm(cudaStream_t st, int M, int N, int K, const bf16r* A, int lda, const bf16r* B,
             int ldb, int mode, const float* bias, float* C, int ldc, bf16r* H, int ldh,
             bf16r* HT, int ldt, const float* Zin, int ldz, float* colsum)
{
    // the staging reads 16-byte vectors, the epilogue writes them: every
    // operand and output of this library is laid out for that; anything
    // else is a bug here, so stop before a misaligned launch
    const bool aligned =
        ((uintptr_t)A % 16 == 0) && ((uintptr_t)B % 16 == 0) && lda % 8 == 0 && ldb % 8 == 0 &&
        (!C || ((uintptr_t)C % 16 == 0 && ldc % 4 == 0)) &&
        (!H || ((uintptr_t)H % 16 == 0 && ldh % 8 == 0)) &&
        (!Zin || ((uintptr_t)Zin % 16 == 0 && ldz % 4 == 0)) && (N == 64 || N == 128);
    if (!aligned)
        return fail(CFS_ERR_INVALID_ARG, "tensor-core GEMM operands not 16-byte aligned");
    TcArgs g;
    g.M = M; g.N = N; g.K = K;
    g.A = A; g.lda = lda;
    g.B = B; g.ldb = ldb;
    g.mode = mode; g.bias = bias; g.C = C; g.ldc = ldc; g.H = H; g.ldh = ldh;
    g.HT = HT; g.ldt = ldt; g.Zin = Zin; g.ldz = ldz; g.colsum = colsum;
    tc_gemm_kernel<<<(M + TC_M - 1) / TC_M, TC_THREADS, TC_SMEM, st>>>(g);
    return CFS_OK;
}

// whether a batch of M rows runs on the fused forward, back_rows_kernel and
// tc_dw_kernel; smaller ones use the register-staged tc_gemm_kernel (no tensor
// map with an extent below its box)
bool rows_on_tma(int M) { return M >= TC_M; }

// a tensor map of [rows][cols] BF16 in boxes of 128 rows x 64 columns
cfs_status box_map(CUtensorMap* t, const void* p, int rows, int cols)
{
    return make_tmap_2d_bf16(t, p, (uint64_t)cols, (uint64_t)rows, (uint64_t)cols, 64u, 128u, true);
}

// forward of B rows of U: H1..H3 (bf16), Z3 (fp32), Y (fp32 [B][2]); with fewer
// rows than one tile also Z1, Z2, H1^T, H2^T
// (after: as for launch_after)
cfs_status forward(cfs_sampler* s, const bf16r* U, int B, cudaStream_t st, bool after = false)
{
    const bf16r* wb = s->wb;
    if ((uintptr_t)U % 16)
        return fail(CFS_ERR_INVALID_ARG, "sampler inputs must be 16-byte aligned");
    if (rows_on_tma(B)) {
        // the fused pass (one launch): what the backward reads, and Y
        static int smem_dev = -1;
        if (smem_dev != s->device) {
            cfs_status r = check_cuda(cudaFuncSetAttribute(train_fwd_kernel,
                                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                           TF_SMEM),
                                      "cudaFuncSetAttribute(train_fwd_kernel)");
            if (r != CFS_OK) return r;
            smem_dev = s->device;
        }
        TrainFwdMaps m;
        cfs_status r = box_map(&m.U, U, B, D_IN);
        if (r == CFS_OK) r = box_map(&m.W1, wb + OFF_W1, HID, D_IN);
        if (r == CFS_OK) r = box_map(&m.W2, wb + OFF_W2, HID, HID);
        if (r == CFS_OK) r = box_map(&m.W3, wb + OFF_W3, HID, HID);
        if (r == CFS_OK) r = box_map(&m.H1, s->H1, B, HID);
        if (r == CFS_OK) r = box_map(&m.H2, s->H2, B, HID);
        if (r == CFS_OK) r = box_map(&m.Z3, s->Z3, B, 2 * HID);
        if (r != CFS_OK) return r;
        const int tiles = (B + 127) / 128;
        const int grid = std::max(1, std::min(device_sm_count(), (tiles + TF_GROUPS - 1) / TF_GROUPS));
        launch_after(after, train_fwd_kernel, grid, TF_THREADS, TF_SMEM, st, m, wb, s->w,
                     TrainFwdArgs{B, s->Y});
        return check_cuda(cudaGetLastError(), "train_fwd_kernel launch");
    }
    // with Z1, Z2 and the transposed copies, which the backward of so few rows
    // reads
    auto layer = [&](int K, const bf16r* A, int off_w, int off_b, float* Z, bf16r* H, bf16r* HT) {
        return tc_gemm(st, B, HID, K, A, K, wb + off_w, K, EPI_SILU, s->w + off_b, Z, HID, H, HID,
                       HT, s->ldt, nullptr, 0, nullptr);
    };
    cfs_status r = layer(D_IN, U, OFF_W1, OFF_B1, s->Z1, s->H1, s->H1T);
    if (r == CFS_OK) r = layer(HID, s->H1, OFF_W2, OFF_B2, s->Z2, s->H2, s->H2T);
    if (r == CFS_OK) r = layer(HID, s->H2, OFF_W3, OFF_B3, s->Z3, s->H3, nullptr);
    if (r != CFS_OK) return r;
    out_forward_kernel<<<(B + 255) / 256, 256, 0, st>>>(s->H3, wb, s->w, B, s->Y);
    return CFS_OK;
}

// dZ2, dZ1 and their column sums from dZ3 (B >= 128 rows)
cfs_status back_rows(cfs_sampler* s, const bf16r* U, int B, float* col2, float* col1,
                     cudaStream_t st)
{
    const bf16r* wb = s->wb;
    BackRowsMaps m;
    cfs_status r = box_map(&m.W1, wb + OFF_W1, HID, D_IN);
    if (r == CFS_OK) r = box_map(&m.W2, wb + OFF_W2, HID, HID);
    if (r == CFS_OK) r = box_map(&m.W3, wb + OFF_W3, HID, HID);
    if (r == CFS_OK) r = box_map(&m.dZ3, s->dZ3, B, HID);
    if (r == CFS_OK) r = box_map(&m.H1, s->H1, B, HID);
    if (r == CFS_OK) r = box_map(&m.U, U, B, D_IN);
    if (r == CFS_OK) r = box_map(&m.dZ2, s->dZ2, B, HID);
    if (r == CFS_OK) r = box_map(&m.dZ1, s->dZ1, B, HID);
    if (r != CFS_OK) return r;
    const int tiles = (B + 127) / 128;
    const int grid = std::max(1, std::min(device_sm_count(), (tiles + BR_GROUPS - 1) / BR_GROUPS));
    launch_after(true, back_rows_kernel, grid, BR_THREADS, BR_SMEM, st, m,
                 BackRowsArgs{B, s->w + OFF_B2, s->w + OFF_B1, col2, col1});
    return check_cuda(cudaGetLastError(), "back_rows_kernel launch");
}

// the weight gradients of W1..W3 and the sums of the bias-gradient copies
// (B >= DW_ROWS rows)
cfs_status tc_dw(cfs_sampler* s, const bf16r* U, int B, float* grads, cudaStream_t st)
{
    const bf16r* dz[3] = {s->dZ3, s->dZ2, s->dZ1};
    const bf16r* in[3] = {s->H2, s->H1, U};
    DwMaps m;
    DwArgs g;
    std::memset(&g, 0, sizeof(g));
    g.chunks = (B + DW_ROWS - 1) / DW_ROWS;
    g.part = s->bias_part;
    g.grads = grads;
    const int off[3] = {OFF_W3, OFF_W2, OFF_W1};
    // CTAs in proportion to the bytes read (256, 256 and 192 B a row)
    const int sms = std::max(3, device_sm_count());
    const int n01 = std::max(1, std::min(g.chunks, sms * 256 / 704));
    const int n2 = std::max(1, std::min(g.chunks, sms - 2 * n01));
    g.cta0[1] = n01;
    g.cta0[2] = 2 * n01;
    g.cta0[3] = 2 * n01 + n2;
    for (int l = 0; l < 3; ++l) {
        g.N[l] = l == 2 ? D_IN : HID;
        g.C[l] = grads + off[l];
        cfs_status r = make_tmap_2d_bf16(&m.a[l], dz[l], HID, (uint64_t)B, HID, 64u, DW_ROWS, true);
        if (r == CFS_OK)
            r = make_tmap_2d_bf16(&m.b[l], in[l], (uint64_t)g.N[l], (uint64_t)B, (uint64_t)g.N[l],
                                  64u, DW_ROWS, true);
        if (r != CFS_OK) return r;
    }
    if ((uintptr_t)grads % 16)
        return fail(CFS_ERR_INVALID_ARG, "weight-gradient GEMM operands not aligned");
    launch_after(true, tc_dw_kernel, g.cta0[3] + 1, DW_THREADS, DW_SMEM, st, m, g);
    return check_cuda(cudaGetLastError(), "tc_dw_kernel launch");
}

// backward of sum(dY * Y), after a kernel of this file; forward() has run and
// bias_part is zero: adds into grads [N_PARAMS]
cfs_status backward(cfs_sampler* s, const bf16r* U, int B, const float* dY, float* grads,
                    cudaStream_t st)
{
    const bf16r* wb = s->wb;
    // fewer rows than one tile: the register-staged GEMMs, whose weight
    // gradients read transposed copies (of fewer than DW_ROWS rows)
    const bool small = !rows_on_tma(B);
    // gradient sums of the output layer and of the biases gather in copies
    // (bias_part) first: fewer atomics on the same address
    float* ob = s->bias_part + 2 * TC_COPIES * HID;
    const int runs = (B + OB_ROWS - 1) / OB_ROWS;
    if (small)
        launch_after(true, &out_backward_kernel<true>, runs, OB_THREADS, 0, st, dY, wb, s->Z3, B,
                     s->dZ3, s->dZ3T, s->ldt, ob);
    else
        launch_after(true, &out_backward_kernel<false>,
                     std::min(runs, 4 * std::max(1, device_sm_count())), OB_THREADS, 0, st, dY, wb,
                     s->Z3, B, s->dZ3, nullptr, 0, ob);
    // dZ2 = (dZ3 W3) * silu'(Z2), then dZ1
    float *col2 = s->bias_part, *col1 = s->bias_part + TC_COPIES * HID;
    cfs_status r;
    if (!small) {
        r = back_rows(s, U, B, col2, col1, st);
        return r == CFS_OK ? tc_dw(s, U, B, grads, st) : r;
    }
    auto rows = [&](const bf16r* A, const bf16r* W, bf16r* dZ, bf16r* dZT, const float* Z,
                    float* col) {
        return tc_gemm(st, B, HID, HID, A, HID, W, HID, EPI_SILU_GRAD, nullptr, nullptr, 0, dZ, HID,
                       dZT, s->ldt, Z, HID, col);
    };
    // (the K-major B operand is W3^T, then W2^T)
    r = rows(s->dZ3, s->wbT + HID * HID, s->dZ2, s->dZ2T, s->Z2, col2);
    // (from one chunk of tc_dw_kernel's rows on its one launch reads the row-major
    // copies: the whole backward of 127 rows 126 -> 89 us, 64 rows 81 where 63 on
    // the GEMMs below take 113)
    const bool dw_rows = B >= DW_ROWS;
    if (r == CFS_OK)
        r = rows(s->dZ2, s->wbT, dw_rows ? s->dZ1 : nullptr, s->dZ1T, s->Z1, col1);
    if (r != CFS_OK || dw_rows) return r == CFS_OK ? tc_dw(s, U, B, grads, st) : r;
    part_reduce_kernel<<<1, 512, 0, st>>>(s->bias_part, grads);
    transpose_in_kernel<<<(B + 31) / 32, 256, 0, st>>>(U, B, s->UT, s->ldt);
    // weight gradients dW = dZ^T A from the transposed copies: K = the rows
    auto dw = [&](int N, const bf16r* dZT, const bf16r* AT, float* C) {
        return tc_gemm(st, HID, N, B, dZT, s->ldt, AT, s->ldt, EPI_ATOMIC, nullptr, C, N, nullptr,
                       0, nullptr, 0, nullptr, 0, nullptr);
    };
    r = dw(HID, s->dZ3T, s->H2T, grads + OFF_W3);
    if (r == CFS_OK) r = dw(HID, s->dZ2T, s->H1T, grads + OFF_W2);
    if (r == CFS_OK) r = dw(D_IN, s->dZ1T, s->UT, grads + OFF_W1);
    return r;
}

void init_params_host(uint64_t seed, std::vector<float>& p)
{
    // uniform +-1/sqrt(fan_in) from Philox (host), zero biases
    p.assign(N_PARAMS, 0.0f);
    const int offs[4] = {OFF_W1, OFF_W2, OFF_W3, OFF_W4};
    const int outs[4] = {HID, HID, HID, D_OUT}, ins[4] = {D_IN, HID, HID, HID};
    for (int l = 0; l < 4; ++l) {
        const float bound = 1.0f / std::sqrt((float)ins[l]);
        for (int e = 0; e < outs[l] * ins[l]; ++e) {
            uint32_t c[4] = {(uint32_t)e, (uint32_t)l, 0u, 6u};
            // Philox on the host for the initial weights (Salmon et al.)
            uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
            uint32_t c0 = c[0], c1 = c[1], c2 = c[2], c3 = c[3];
            for (int r = 0; r < 10; ++r) {
                const uint64_t p0 = (uint64_t)0xD2511F53u * c0, p1 = (uint64_t)0xCD9E8D57u * c2;
                const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ k0, n2 = (uint32_t)(p0 >> 32) ^ c3 ^ k1;
                c1 = (uint32_t)p1; c3 = (uint32_t)p0; c0 = n0; c2 = n2;
                k0 += 0x9E3779B9u; k1 += 0xBB67AE85u;
            }
            const float u = (float)(c0 >> 8) * (1.0f / 16777216.0f);
            p[offs[l] + e] = (2.0f * u - 1.0f) * bound;
        }
    }
}

cfs_status upload_params(cfs_sampler* s, const float* host)
{
    cfs_status st = check_cuda(cudaMemcpy(s->w, host, sizeof(float) * N_PARAMS,
                                          cudaMemcpyHostToDevice), "cudaMemcpy(params)");
    if (st != CFS_OK) return st;
    to_bf16_kernel<<<(N_PARAMS + 255) / 256, 256>>>(s->w, s->wb, s->wbT, N_PARAMS);
    return check_cuda(cudaDeviceSynchronize(), "sampler params");
}

// The system's record: thresholds and maps in their own order (the chaos
// game that makes training targets), and the conditioning vector with the
// maps in canonical order -- decreasing |det A| = |a d - b c| (in double
// from the FP32 parameters), ties by index -- because the attractor does
// not depend on the order in which the maps are listed.
void pack_system(const cfs_system* sys, float t, SysRec* r)
{
    std::memset(r, 0, sizeof(*r));
    for (int j = 0; j < sys->n_cmp; ++j) r->T[j] = sys->T[j];
    r->n_cmp = sys->n_cmp;
    r->n_maps = sys->n_maps;
    const int n = std::min(sys->n_maps, MAX_SYS_MAPS);
    int order[MAX_SYS_MAPS];
    double adet[MAX_SYS_MAPS];
    for (int k = 0; k < n; ++k) {
        const float* v = sys->maps[k].params;
        order[k] = k;
        adet[k] = std::fabs((double)v[0] * (double)v[3] - (double)v[1] * (double)v[2]);
        for (int j = 0; j < 6; ++j) r->prm[k][j] = v[j];
    }
    std::stable_sort(order, order + n, [&](int a, int b) { return adet[a] > adet[b]; });
    for (int q = 0; q < n; ++q)
        for (int j = 0; j < 6; ++j) r->cond[6 * q + j] = sys->maps[order[q]].params[j];
    r->t = t;
}

}  // namespace

namespace cfs {
cfs_status take_device_flags(unsigned int* flags)
{
    unsigned int v = 0;
    cfs_status st = check_cuda(cudaMemcpyFromSymbol(&v, g_tc_error, sizeof(v)), "error flags");
    if (st == CFS_OK && v) {
        const unsigned int zero = 0;
        st = check_cuda(cudaMemcpyToSymbol(g_tc_error, &zero, sizeof(zero)), "error flags");
    }
    *flags = v;
    return st;
}

cfs_status raise_device_flags(unsigned int flags)
{
    unsigned int v = 0;
    cfs_status st = check_cuda(cudaMemcpyFromSymbol(&v, g_tc_error, sizeof(v)), "error flags");
    v |= flags;
    if (st == CFS_OK)
        st = check_cuda(cudaMemcpyToSymbol(g_tc_error, &v, sizeof(v)), "error flags");
    return st;
}
}  // namespace cfs

namespace {
cfs_status check_sampler_system(const cfs_system* sys)
{
    if (!sys) return fail(CFS_ERR_INVALID_ARG, "NULL system");
    if (sys->dim != 2 || sys->n_maps > MAX_SYS_MAPS)
        return fail(CFS_ERR_UNSUPPORTED, "the sampler conditions on 2D systems of up to 8 maps");
    for (int k = 0; k < sys->n_maps; ++k)
        if (sys->maps[k].kind != CFS_MAP_AFFINE)
            return fail(CFS_ERR_UNSUPPORTED, "the sampler conditions on affine maps");
    return CFS_OK;
}
}  // namespace

extern "C" {

cfs_status cfs_sampler_create(const float* params, uint64_t seed, cfs_sampler** out)
{
    clear_error();
    if (!out) return fail(CFS_ERR_INVALID_ARG, "out is NULL");
    *out = nullptr;
    cfs_sampler* s = new (std::nothrow) cfs_sampler();
    if (!s) return fail(CFS_ERR_OOM, "host allocation failed");
    cudaGetDevice(&s->device);
    // w | m | v (FP32), then the BF16 copies on 256-byte boundaries: the
    // tensor-core GEMMs read the weights with 16-byte loads
    const size_t off_wb = (sizeof(float) * N_PARAMS * 3 + 255) & ~(size_t)255;
    const size_t off_wbT = off_wb + ((sizeof(bf16r) * N_PARAMS + 255) & ~(size_t)255);
    const size_t off_part = off_wbT + sizeof(bf16r) * 2 * HID * HID;
    cfs_status st = check_cuda(cudaMalloc(&s->w, off_part + sizeof(float) * PART_FLOATS),
                               "cudaMalloc(sampler params)");
    if (st != CFS_OK) { delete s; return st; }
    s->m = s->w + N_PARAMS;
    s->v = s->m + N_PARAMS;
    s->wb = reinterpret_cast<bf16r*>(reinterpret_cast<unsigned char*>(s->w) + off_wb);
    s->wbT = reinterpret_cast<bf16r*>(reinterpret_cast<unsigned char*>(s->w) + off_wbT);
    s->bias_part = reinterpret_cast<float*>(reinterpret_cast<unsigned char*>(s->w) + off_part);
    // the tensor-core GEMM stages its chunk pairs in dynamic shared memory
    if (st == CFS_OK)
        st = check_cuda(cudaFuncSetAttribute(tc_gemm_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM),
                        "cudaFuncSetAttribute(tc_gemm_kernel)");
    if (st == CFS_OK)
        st = check_cuda(cudaFuncSetAttribute(back_rows_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, BR_SMEM),
                        "cudaFuncSetAttribute(back_rows_kernel)");
    if (st == CFS_OK)
        st = check_cuda(cudaFuncSetAttribute(tc_dw_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, DW_SMEM),
                        "cudaFuncSetAttribute(tc_dw_kernel)");
    if (st == CFS_OK) st = check_cuda(cudaMalloc(&s->d_step, 256), "cudaMalloc(step)");
    if (st == CFS_OK) st = check_cuda(cudaMemset(s->m, 0, sizeof(float) * N_PARAMS * 2), "memset");
    if (st == CFS_OK) st = check_cuda(cudaMemset(s->d_step, 0, 256), "memset");
    std::vector<float> init;
    if (!params) { init_params_host(seed, init); params = init.data(); }
    if (st == CFS_OK) st = upload_params(s, params);
    if (st != CFS_OK) { cfs_sampler_destroy(s); return st; }
    *out = s;
    return CFS_OK;
}

cfs_status cfs_sampler_destroy(cfs_sampler* s)
{
    if (!s) return CFS_OK;
    cudaDeviceSynchronize();
    if (s->act) cudaFree(s->act);
    if (s->inf) cudaFree(s->inf);
    if (s->inf_host) cudaFreeHost(s->inf_host);
    if (s->uploaded) cudaEventDestroy(s->uploaded);
    if (s->w) cudaFree(s->w);
    if (s->d_step) cudaFree(s->d_step);
    delete s;
    return CFS_OK;
}

uint32_t cfs_sampler_param_count(void) { return N_PARAMS; }

cfs_status cfs_sampler_get_params(const cfs_sampler* s, float* params, float* adam_m,
                                  float* adam_v, uint32_t* step)
{
    clear_error();
    if (!s) return fail(CFS_ERR_INVALID_ARG, "NULL sampler");
    cfs_status st = check_cuda(cudaDeviceSynchronize(), "sampler sync");
    const float* src[3] = {s->w, s->m, s->v};
    float* dst[3] = {params, adam_m, adam_v};
    for (int j = 0; j < 3 && st == CFS_OK; ++j)
        if (dst[j])
            st = check_cuda(cudaMemcpy(dst[j], src[j], sizeof(float) * N_PARAMS,
                                       cudaMemcpyDeviceToHost), "cudaMemcpy(params)");
    if (st == CFS_OK && step)
        st = check_cuda(cudaMemcpy(step, s->d_step, 4, cudaMemcpyDeviceToHost), "step");
    // a tensor-core GEMM whose barrier wait ran out of time skipped its
    // output: report it once
    unsigned int flags = 0;
    if (st == CFS_OK) st = take_device_flags(&flags);
    if (st == CFS_OK && (flags & CFS_DEVICE_ERR_TC_TIMEOUT))
        return fail(CFS_ERR_TIMEOUT, "a tensor-core GEMM timed out waiting for its mbarrier");
    return st;
}

cfs_status cfs_sampler_set_params(cfs_sampler* s, const float* params, const float* adam_m,
                                  const float* adam_v, uint32_t step)
{
    clear_error();
    if (!s || !params) return fail(CFS_ERR_INVALID_ARG, "NULL sampler or params");
    cfs_status st = check_cuda(cudaDeviceSynchronize(), "sampler sync");
    if (st == CFS_OK) st = upload_params(s, params);
    if (st == CFS_OK && adam_m)
        st = check_cuda(cudaMemcpy(s->m, adam_m, sizeof(float) * N_PARAMS, cudaMemcpyHostToDevice), "m");
    if (st == CFS_OK && adam_v)
        st = check_cuda(cudaMemcpy(s->v, adam_v, sizeof(float) * N_PARAMS, cudaMemcpyHostToDevice), "v");
    if (st == CFS_OK)
        st = check_cuda(cudaMemcpy(s->d_step, &step, 4, cudaMemcpyHostToDevice), "step");
    return st;
}

cfs_status cfs_sampler_forward(cfs_sampler* s, const void* U, uint32_t B, float* Y, void* stream)
{
    clear_error();
    if (!s || !U || !Y) return fail(CFS_ERR_INVALID_ARG, "NULL argument");
    if (B == 0) return CFS_OK;
    if (B > (1u << 24)) return fail(CFS_ERR_INVALID_ARG, "B too large");
    cfs_status st = ensure_rows(s, (int)B);
    if (st != CFS_OK) return st;
    cudaStream_t sm = (cudaStream_t)stream;
    st = forward(s, (const bf16r*)U, (int)B, sm);
    if (st != CFS_OK) return st;
    st = check_cuda(cudaMemcpyAsync(Y, s->Y, sizeof(float) * 2 * B, cudaMemcpyDeviceToDevice, sm),
                    "copy Y");
    if (st != CFS_OK) return st;
    return check_cuda(cudaGetLastError(), "sampler forward");
}

cfs_status cfs_sampler_backward(cfs_sampler* s, const void* U, uint32_t B, const float* dY,
                                float* grads, void* stream)
{
    clear_error();
    if (!s || !U || !dY || !grads) return fail(CFS_ERR_INVALID_ARG, "NULL argument");
    if (B == 0) return CFS_OK;
    if (B > (1u << 24)) return fail(CFS_ERR_INVALID_ARG, "B too large");
    cfs_status st = ensure_rows(s, (int)B);
    if (st != CFS_OK) return st;
    cudaStream_t sm = (cudaStream_t)stream;
    cudaMemsetAsync(s->bias_part, 0, sizeof(float) * PART_FLOATS, sm);
    st = forward(s, (const bf16r*)U, (int)B, sm);
    if (st == CFS_OK) st = backward(s, (const bf16r*)U, (int)B, dY, grads, sm);
    if (st != CFS_OK) return st;
    return check_cuda(cudaGetLastError(), "sampler backward");
}

cfs_status cfs_sw_loss(const float* X, const float* T, uint32_t n_sys, uint32_t n_per,
                       const float* phi, uint32_t n_proj, float* loss, float* dX, void* stream)
{
    clear_error();
    if (!X || !T || !phi || !loss || !dX) return fail(CFS_ERR_INVALID_ARG, "NULL argument");
    if (n_per < 32 || n_per > 1024 || (n_per & (n_per - 1)))
        return fail(CFS_ERR_INVALID_ARG, "points per system must be a power of two in 32..1024");
    if (n_sys == 0 || n_proj == 0) return CFS_OK;
    const float scale = 1.0f / ((float)n_sys * (float)n_proj);
    sw_launch(false, X, T, phi, (int)n_proj, (int)n_per, (int)n_sys, scale, loss, dX,
              (cudaStream_t)stream);
    return check_cuda(cudaGetLastError(), "sw_kernel launch");
}

cfs_status cfs_sampler_adam(cfs_sampler* s, const float* grads, uint32_t t, float lr,
                            void* stream)
{
    clear_error();
    if (!s || !grads || t == 0) return fail(CFS_ERR_INVALID_ARG, "bad arguments");
    adam_kernel<<<(N_PARAMS + 255) / 256, 256, 0, (cudaStream_t)stream>>>(
        s->w, s->m, s->v, grads, s->wb, s->wbT, N_PARAMS, nullptr, t, lr, lr, 0u, 0u, 0.9f,
        0.999f, 1e-8f, nullptr, nullptr);
    return check_cuda(cudaGetLastError(), "adam launch");
}

cfs_status cfs_sampler_train(cfs_sampler* s, const cfs_system* const* systems,
                             const float* t_values, int n_systems, uint32_t steps,
                             uint32_t systems_per_step, uint32_t points_per_system,
                             uint32_t n_proj, float lr, uint64_t seed, float* loss_history,
                             void* stream)
{
    cfs_train_options o;
    o.steps = steps;
    o.systems_per_step = systems_per_step;
    o.points_per_system = points_per_system;
    o.n_proj = n_proj;
    o.lr = lr;
    o.lr_final = lr;
    o.seed = seed;
    return cfs_sampler_train_ex(s, systems, t_values, n_systems, &o, loss_history, stream);
}

cfs_status cfs_sampler_train_ex(cfs_sampler* s, const cfs_system* const* systems,
                                const float* t_values, int n_systems,
                                const cfs_train_options* opt, float* loss_history, void* stream)
{
    clear_error();
    if (!s || !systems || !t_values || n_systems <= 0 || !opt)
        return fail(CFS_ERR_INVALID_ARG, "NULL sampler, systems or options");
    const uint32_t steps = opt->steps, systems_per_step = opt->systems_per_step;
    const uint32_t points_per_system = opt->points_per_system, n_proj = opt->n_proj;
    const float lr = opt->lr, lr_final = opt->lr_final;
    const uint64_t seed = opt->seed;
    if (!(lr > 0.0f) || !(lr_final > 0.0f) || !std::isfinite(lr) || !std::isfinite(lr_final))
        return fail(CFS_ERR_INVALID_ARG, "learning rates must be positive and finite");
    if (points_per_system < 32 || points_per_system > 1024 ||
        (points_per_system & (points_per_system - 1)))
        return fail(CFS_ERR_INVALID_ARG, "points per system must be a power of two in 32..1024");
    if (systems_per_step == 0 || systems_per_step > 1024 || n_proj == 0 || n_proj > 1024)
        return fail(CFS_ERR_INVALID_ARG, "systems per step and projections must be in 1..1024");
    for (int i = 0; i < n_systems; ++i) {
        cfs_status st = check_sampler_system(systems[i]);
        if (st != CFS_OK) return st;
    }
    cudaStream_t sm = (cudaStream_t)stream;
    const int S = (int)systems_per_step, N = (int)points_per_system, B = S * N;
    cfs_status st = ensure_rows(s, B);
    if (st != CFS_OK) return st;
    // device workspace of the run
    std::vector<SysRec> recs(n_systems);
    for (int i = 0; i < n_systems; ++i) pack_system(systems[i], t_values[i], &recs[i]);
    const size_t bytes = sizeof(SysRec) * n_systems + 4 * 1024 +
                         sizeof(float) * (size_t)B * 2 * 2 + sizeof(bf16r) * (size_t)B * D_IN +
                         sizeof(float) * (N_PARAMS + 1) + sizeof(float) * (steps + 1) + 8 * 256;
    unsigned char* ws = nullptr;
    st = check_cuda(cudaMalloc(&ws, bytes), "cudaMalloc(training workspace)");
    if (st != CFS_OK) return st;
    unsigned char* p = ws;
    auto take = [&](size_t n) {
        unsigned char* r = p;
        p += (n + 255) & ~(size_t)255;
        return r;
    };
    SysRec* d_sys = (SysRec*)take(sizeof(SysRec) * n_systems);
    float* d_phi = (float*)take(4 * 1024);
    float* d_T = (float*)take(sizeof(float) * (size_t)B * 2);
    float* d_dY = (float*)take(sizeof(float) * (size_t)B * 2);
    bf16r* d_U = (bf16r*)take(sizeof(bf16r) * (size_t)B * D_IN);
    float* d_g = (float*)take(sizeof(float) * (N_PARAMS + 1));
    float* d_loss = d_g + N_PARAMS;
    float* d_hist = (float*)take(sizeof(float) * (steps + 1));
    u32 step0 = 0;
    cudaStream_t cap = nullptr;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    st = check_cuda(cudaMemcpy(d_sys, recs.data(), sizeof(SysRec) * n_systems,
                               cudaMemcpyHostToDevice), "upload systems");
    if (st == CFS_OK) st = check_cuda(cudaMemcpy(&step0, s->d_step, 4, cudaMemcpyDeviceToHost), "step");
    if (st == CFS_OK) st = check_cuda(cudaMemset(d_hist, 0, sizeof(float) * (steps + 1)), "memset");
    if (st == CFS_OK) st = check_cuda(cudaStreamCreateWithFlags(&cap, cudaStreamNonBlocking), "stream");
    // one training step, captured once and replayed
    if (st == CFS_OK) st = check_cuda(cudaStreamBeginCapture(cap, cudaStreamCaptureModeThreadLocal), "capture");
    if (st == CFS_OK) {
        DataArgs da;
        std::memset(&da, 0, sizeof(da));
        philox_round_keys(seed, da.rk);
        da.sys = d_sys; da.n_sys = n_systems; da.step = s->d_step;
        da.N = N; da.rows = B; da.steps = 40; da.P = (int)n_proj;
        da.T = d_T; da.U = d_U; da.phi = d_phi;
        da.zero_a = d_g; da.n_a = N_PARAMS + 1;          // and the loss behind them
        da.zero_b = s->bias_part; da.n_b = PART_FLOATS;
        da.dY = d_dY;
        data_kernel<<<(B + 255) / 256, 256, 0, cap>>>(da);
        cfs_status fst = forward(s, d_U, B, cap, true);
        sw_launch(true, s->Y, d_T, d_phi, (int)n_proj, N, S, 1.0f / ((float)S * (float)n_proj),
                  d_loss, d_dY, cap);
        if (fst == CFS_OK) fst = backward(s, d_U, B, d_dY, d_g, cap);
        launch_after(true, adam_kernel, (N_PARAMS + 255) / 256, 256, 0, cap, s->w, s->m, s->v, d_g,
                     s->wb, s->wbT, N_PARAMS, s->d_step, 0u, lr, lr_final, step0, steps, 0.9f,
                     0.999f, 1e-8f, d_loss, d_hist);
        cudaError_t e = cudaGetLastError();
        cudaError_t e2 = cudaStreamEndCapture(cap, &graph);
        st = check_cuda(e != cudaSuccess ? e : e2, "training step capture");
        if (st == CFS_OK && fst != CFS_OK) st = fst;
    }
    if (st == CFS_OK) st = check_cuda(cudaGraphInstantiate(&exec, graph, 0), "instantiate");
    for (uint32_t i = 0; i < steps && st == CFS_OK; ++i)
        st = check_cuda(cudaGraphLaunch(exec, sm), "cudaGraphLaunch");
    if (st == CFS_OK) st = check_cuda(cudaStreamSynchronize(sm), "training");
    if (st == CFS_OK && loss_history && steps > 0)
        st = check_cuda(cudaMemcpy(loss_history, d_hist, sizeof(float) * steps,
                                   cudaMemcpyDeviceToHost), "loss history");
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
    if (cap) cudaStreamDestroy(cap);
    cudaFree(ws);
    return st;
}

namespace {
struct InferLayout {
    size_t rec, c1, tiles, count, seed, out, total;
};

InferLayout infer_layout(int n)
{
    auto up = [](size_t v) { return (v + 255) & ~(size_t)255; };
    InferLayout l;
    l.rec = 0;
    l.c1 = up(l.rec + sizeof(SysRec) * (size_t)n);
    l.tiles = up(l.c1 + sizeof(float) * HID * (size_t)n);
    l.count = up(l.tiles + sizeof(u32) * ((size_t)n + 1));
    l.seed = up(l.count + sizeof(u32) * (size_t)n);
    l.out = up(l.seed + sizeof(u64) * (size_t)n);
    l.total = up(l.out + sizeof(float*) * (size_t)n);
    return l;
}
}  // namespace

cfs_status cfs_sampler_start_points_batch(cfs_sampler* s, int n_frames,
                                          const cfs_system* const* systems, const float* t,
                                          const uint32_t* counts, const uint64_t* seeds,
                                          float* const* starts, void* stream)
{
    clear_error();
    if (!s || !systems || !t || !counts || !seeds || !starts || n_frames <= 0)
        return fail(CFS_ERR_INVALID_ARG, "NULL argument or no frames");
    uint64_t tiles = 0;
    for (int f = 0; f < n_frames; ++f) {
        cfs_status st = check_sampler_system(systems[f]);
        if (st != CFS_OK) return st;
        if (counts[f] > (1u << 30)) return fail(CFS_ERR_INVALID_ARG, "count too large");
        if (counts[f] && !starts[f]) return fail(CFS_ERR_INVALID_ARG, "NULL output");
        tiles += (counts[f] + 127) / 128;
    }
    if (tiles >= (1ull << 31)) return fail(CFS_ERR_INVALID_ARG, "too many rows");
    cudaStream_t sm = (cudaStream_t)stream;
    const InferLayout L = infer_layout(n_frames);
    if (n_frames > s->cap_frames) {
        // the previous staging buffer may still feed an upload
        cfs_status st = check_cuda(cudaDeviceSynchronize(), "sampler sync");
        if (st != CFS_OK) return st;
        if (s->inf) cudaFree(s->inf);
        if (s->inf_host) cudaFreeHost(s->inf_host);
        s->inf = nullptr;
        s->inf_host = nullptr;
        s->cap_frames = 0;
        st = check_cuda(cudaMalloc(&s->inf, L.total), "cudaMalloc(inference workspace)");
        if (st == CFS_OK)
            st = check_cuda(cudaMallocHost(&s->inf_host, L.total), "cudaMallocHost(inference)");
        if (st != CFS_OK) return st;
        s->cap_frames = n_frames;
    } else if (s->upload_pending) {
        // the staging buffer is rewritten: wait for its last upload only
        cfs_status st = check_cuda(cudaEventSynchronize(s->uploaded), "sampler upload sync");
        if (st != CFS_OK) return st;
    }
    if (!s->uploaded) {
        cfs_status st = check_cuda(cudaEventCreateWithFlags(&s->uploaded, cudaEventDisableTiming),
                                   "cudaEventCreate");
        if (st != CFS_OK) return st;
    }
    unsigned char* h = s->inf_host;
    u32* h_tiles = reinterpret_cast<u32*>(h + L.tiles);
    u32 acc = 0;
    for (int f = 0; f < n_frames; ++f) {
        pack_system(systems[f], t[f], reinterpret_cast<SysRec*>(h + L.rec) + f);
        h_tiles[f] = acc;
        acc += (counts[f] + 127) / 128;
        reinterpret_cast<u32*>(h + L.count)[f] = counts[f];
        reinterpret_cast<u64*>(h + L.seed)[f] = seeds[f];
        reinterpret_cast<float**>(h + L.out)[f] = starts[f];
    }
    h_tiles[n_frames] = acc;
    cfs_status st = check_cuda(cudaMemcpyAsync(s->inf, h, L.total, cudaMemcpyHostToDevice, sm),
                               "cudaMemcpyAsync(inference frames)");
    if (st == CFS_OK) st = check_cuda(cudaEventRecord(s->uploaded, sm), "cudaEventRecord");
    if (st != CFS_OK) return st;
    s->upload_pending = true;
    unsigned char* d = s->inf;
    cond_kernel<<<n_frames, HID, 0, sm>>>(s->wb, s->w, reinterpret_cast<const SysRec*>(d + L.rec),
                                         reinterpret_cast<float*>(d + L.c1));
    if (acc == 0) return check_cuda(cudaGetLastError(), "sampler conditioning");
    static int smem_set = -1;
    if (smem_set != s->device) {
        st = check_cuda(cudaFuncSetAttribute(infer_tc_kernel,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             IT_SMEM),
                        "cudaFuncSetAttribute");
        if (st != CFS_OK) return st;
        smem_set = s->device;
    }
    // persistent: one CTA per SM (its shared memory and 512 TMEM columns),
    // IT_GROUPS tiles in flight per CTA
    const int sms = std::max(1, device_sm_count());
    const int grid = (int)std::min<uint64_t>((uint64_t)sms, (acc + IT_GROUPS - 1) / IT_GROUPS);
    InferFrames fs;
    fs.c1 = reinterpret_cast<const float*>(d + L.c1);
    fs.tile_begin = reinterpret_cast<const u32*>(d + L.tiles);
    fs.count = reinterpret_cast<const u32*>(d + L.count);
    fs.seed = reinterpret_cast<const u64*>(d + L.seed);
    fs.out = reinterpret_cast<float* const*>(d + L.out);
    fs.n_sys = n_frames;
    infer_tc_kernel<<<grid, IT_THREADS, IT_SMEM, sm>>>(s->wb, s->w, fs);
    return check_cuda(cudaGetLastError(), "sampler start points");
}

cfs_status cfs_sampler_start_points(cfs_sampler* s, const cfs_system* sys, float t, uint32_t n,
                                    uint64_t seed, float* start, void* stream)
{
    if (n == 0) {
        clear_error();
        if (!s || !start) return fail(CFS_ERR_INVALID_ARG, "NULL sampler or output");
        return check_sampler_system(sys);
    }
    return cfs_sampler_start_points_batch(s, 1, &sys, &t, &n, &seed, &start, stream);
}

}  // extern "C"
