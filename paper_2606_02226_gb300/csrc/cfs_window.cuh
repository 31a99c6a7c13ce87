/*
 * cfs_window.cuh -- what the batched histogram renderers share: a frame's map
 * choice table, the privatized shared-memory windows of its histogram, their
 * splats, and the pre-pass that places them.  Included by cfs_device.cuh (the
 * generated programs and the no-allocation batch).
 */
#ifndef CFS_WINDOW_CUH
#define CFS_WINDOW_CUH

/* ---- map choice of a frame ------------------------------------------------
 * k = #{ j < n_cmp : w >= T_j } through a bucket table.  Where no bucket of the
 * word's top 5 bits holds more than one threshold (`more5`, most systems), one
 * lookup does: bucket b's entry has the other 27 bits of the threshold's
 * predecessor, the last word of the bucket that stays, above the count k at
 * the bucket's start (32 words, one a bank: no conflicts).  That is one
 * shared-memory cycle a warp instead of two, of 14.7 a step in a kernel that
 * they bound: 142.0 -> 136.8 ms for the 256 animation frames.
 * In other frames the top 7 bits of the word pick one of 128 buckets (128
 * bytes: every bank holds one word of them, so a warp's lookups never
 * conflict), whose entry is 16 times the count at the bucket's start; the word
 * is then compared with the thresholds the bucket may hold.  `more` is the
 * largest number of thresholds in one of these; the loop for more than one,
 * compiled into a copy of its own, cost 5% of the animation's time when every
 * step tested for it.  A finer table with a fallback (12 bits, one lookup) took
 * 3.4 shared-memory cycles per warp instead of 2 and a divergent branch. */
#define CFS_KTAB_BITS 7
struct CfsKtab {
    unsigned char k16[1 << CFS_KTAB_BITS];
    u32 last[CFS_A_MAX_MAPS][4];    /* [k][0]: T_k - 1, the last word that stays at k */
    u32 one[32];                    /* [bucket]: (T_k - 1) << 5 | k */
    int more, more5;
};

struct CfsChooseOne {
    const CfsKtab& t;               /* shared memory */
    __device__ __forceinline__ int operator()(u32 w) const
    {
        const u32 e = t.one[w >> 27];
        return (int)((e & 31u) + (w << 5 > e ? 1u : 0u));
    }
};

template <bool MORE>
struct CfsChooseKtab {
    const CfsKtab& t;               /* shared memory */
    int more;
    __device__ __forceinline__ int operator()(u32 w) const
    {
        u32 o = t.k16[w >> (32 - CFS_KTAB_BITS)];
        const char* last = reinterpret_cast<const char*>(&t.last[0][0]);
        o += w > *reinterpret_cast<const u32*>(last + o) ? 16u : 0u;
        for (int r = 1; MORE && r < more; ++r)
            o += w > *reinterpret_cast<const u32*>(last + o) ? 16u : 0u;
        __builtin_assume((o & 15u) == 0u);
        return (int)(o >> 4);
    }
};

/* the frame's table from its n_cmp ascending thresholds (all threads; the
 * caller synchronizes before and after) */
__device__ __forceinline__ void cfs_build_ktab(const u32* T, int n_cmp, CfsKtab& t)
{
    /* (a threshold of 0 is below every word and so never the next one) */
    for (u32 k = threadIdx.x; k < CFS_A_MAX_MAPS; k += blockDim.x)
        t.last[k][0] = (int)k < n_cmp ? T[k] - 1u : 0xFFFFFFFFu;
    if (threadIdx.x < 32) {
        int more = 1;
        for (u32 b = threadIdx.x; b < (1u << CFS_KTAB_BITS); b += 32) {
            const u32 w0 = b << (32 - CFS_KTAB_BITS);
            const u32 w1 = w0 | ((1u << (32 - CFS_KTAB_BITS)) - 1u);
            int k0 = 0, k1 = 0;
            for (int j = 0; j < n_cmp; ++j) {
                k0 += w0 >= T[j] ? 1 : 0;
                k1 += w1 >= T[j] ? 1 : 0;
            }
            t.k16[b] = (unsigned char)(16 * k0);
            more = max(more, k1 - k0);
        }
        more = __reduce_max_sync(0xffffffffu, more);
        const u32 w0 = threadIdx.x << 27, w1 = w0 | 0x07FFFFFFu;
        int k0 = 0, k1 = 0;
        for (int j = 0; j < n_cmp; ++j) {
            k0 += w0 >= T[j] ? 1 : 0;
            k1 += w1 >= T[j] ? 1 : 0;
        }
        /* (no threshold: no word passes 27 ones) */
        t.one[threadIdx.x] = (k1 > k0 ? (T[k0] - 1u) << 5 : 0xFFFFFFE0u) | (u32)k0;
        const int more5 = __reduce_max_sync(0xffffffffu, k1 - k0);
        if (threadIdx.x == 0) {
            t.more = more;
            t.more5 = more5;
        }
    }
}

/* ---- privatized windows of a batch frame's u32 histogram ------------------
 * One pixel box per channel (a channel's splats come from its own maps, whose
 * images are smaller copies of the attractor, so each channel's box sits over
 * that channel's densest region), the channels' counters packed one after the
 * other in shared memory.
 *
 * A splat's bin is floor((x - x0) sx): with 2^23 added in round-down mode the
 * sum's bits are 0x4B000000 + that floor for 0 <= . < 2^23, and every other
 * value (negative, infinite, NaN) gives bits that are no such number, so one
 * unsigned comparison after subtracting a box's origin tests the box and all
 * of them.  This stands for the view test too where a box holds only "safe"
 * columns and rows: those to which no coordinate outside the view has its
 * product rounded (cfs_safe_bins). */
#define CFS_BIN_MAGIC 0x4B000000u

/* The columns (rows) of an axis that only coordinates inside the view reach,
 * and those without the last bin's clamp: first in .x, their number in .y.
 * (u - lo) * scale never decreases with u, so the two view bounds and their
 * outer neighbours tell; for u > hi it is within two roundings of n or above,
 * so with n <= 65536 it passes n - 1 in any case. */
__device__ __forceinline__ int2 cfs_safe_bins(float lo, float hi, float scale, int n)
{
    const float inf = __int_as_float(0x7f800000);
    const float below = (nextafterf(lo, -inf) - lo) * scale;
    const float above = (nextafterf(hi, inf) - lo) * scale;
    const int first = below < 0.0f ? 0 : 1;
    const int last = above >= (float)n && (hi - lo) * scale < (float)n ? n - 1 : n - 2;
    return make_int2(first, max(0, last - first + 1));
}

/* What a windowed splat reads of its target: the frame's values, copied to
 * the kernel's locals once per frame so that they stay in registers instead
 * of being read from shared memory on every splat. */
struct CfsBinTarget {
    float x0, sx, y0, sy;
    u32 bx, nx, by, ny;         /* safe bins: first (+ CFS_BIN_MAGIC), number */
    u32 W4;                     /* bytes of a row */
    unsigned long long base;    /* data - 4 CFS_BIN_MAGIC */
};

template <class F>
__device__ __forceinline__ CfsBinTarget cfs_bin_target(const F& t)
{
    const int2 sx = cfs_safe_bins(t.x0, t.x1, t.sx, t.W), sy = cfs_safe_bins(t.y0, t.y1, t.sy, t.H);
    return CfsBinTarget{t.x0, t.sx, t.y0, t.sy, (u32)sx.x + CFS_BIN_MAGIC, (u32)sx.y,
                        (u32)sy.x + CFS_BIN_MAGIC, (u32)sy.y, 4u * (u32)t.W,
                        t.data - 4ull * CFS_BIN_MAGIC};
}

struct CfsTile {
    /* shared, per generator map k (the window of its channel):
     * (x0 + magic, y0 + magic, w | h << 16, byte address of the first
     * counter); w = 0: no window */
    const int4* win;
    /* shared, per map: its channel's first row of the histogram, channel H,
     * less CFS_BIN_MAGIC */
    const u32* row;
    const cfs_dev_target* tg;   /* shared: the target, for the general path */
};

/* the record of one channel's box for CfsTile::win */
__device__ __forceinline__ int4 cfs_win_record(int4 box, u32* cnt)
{
    return make_int4((int)((u32)box.x + CFS_BIN_MAGIC), (int)((u32)box.y + CFS_BIN_MAGIC), box.z,
                     (int)((u32)__cvta_generic_to_shared(cnt) + 4u * (u32)box.w));
}

/* u32 histogram splat of map index kc: adds to the shared window of its
 * channel when the bin lies in it (one shared atomic per group of lanes
 * hitting the same counter with CFS_WARP_AGG) and to global memory otherwise.
 * Two in five warps have a lane that misses its window, so the miss path is
 * kept short too: safe bins need no view test and no clamp.  (Both
 * reductions under predicates, without the branch, ran 17% more instructions
 * and the animation in 193 instead of 167 ms.) */
__device__ __forceinline__ void cfs_splat_hist_tile(const CfsBinTarget& t, const CfsTile& tl,
                                                    float x, float y, bool alive, int kc,
                                                    int channels, u32& disc)
{
    const u32 bu = __float_as_uint(__fadd_rd((x - t.x0) * t.sx, 8388608.0f));
    const u32 bv = __float_as_uint(__fadd_rd((y - t.y0) * t.sy, 8388608.0f));
    const int4 g = tl.win[kc];
    const u32 lx = bu - (u32)g.x, ly = bv - (u32)g.y;
    const u32 w = (u32)g.z & 0xFFFFu, h = (u32)g.z >> 16;
    if (alive && lx < w && ly < h) {
        const u32 at = (u32)g.w + 4u * (ly * w + lx);
#if defined(CFS_WARP_AGG) && CFS_WARP_AGG
        const u32 act = __activemask();
        const u32 peers = __match_any_sync(act, at);
        if ((int)(threadIdx.x & 31) == __ffs(peers) - 1)
            asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(at), "r"(__popc(peers)));
#else
        asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(at), "r"(1u));
#endif
    } else if (alive && bu - t.bx < t.nx && bv - t.by < t.ny) {
        const u32 row = bv + tl.row[kc];
        cfs_red_add_u32(reinterpret_cast<u32*>(t.base + (u64)row * t.W4 + (u64)bu * 4ull), 1u);
    } else {
        cfs_splat_hist(*tl.tg, x, y, alive, kc % channels, disc);
    }
}

/* (the pre-pass records the chain's points and never splats) */
__device__ __forceinline__ void cfs_splat_hist_tile(const cfs_dev_target& t, const CfsTile&,
                                                    float x, float y, bool alive, int kc,
                                                    int channels, u32& disc)
{
    cfs_splat_hist(t, x, y, alive, kc % channels, disc);
}

/* Adds the windows' nonzero counters to the global histogram and zeroes
 * them; every thread of the CTA takes part.  win: per channel (x0, y0,
 * w | h << 16, first counter). */
template <class F>
__device__ __forceinline__ void cfs_flush_tile(const F& t, u32* cnt, const int4* win, int C)
{
    u32* base = reinterpret_cast<u32*>(t.data);
    for (int ch = 0; ch < C; ++ch) {
        const int4 g = win[ch];
        const u32 w = (u32)g.z & 0xFFFFu, h = (u32)g.z >> 16;
        u32* cc = cnt + (u32)g.w;
        for (u32 e = threadIdx.x; e < w * h; e += blockDim.x) {
            const u32 v = cc[e];
            cc[e] = 0u;
            if (v) {
                const u32 ly = e / w, lx = e - ly * w;
                const size_t off = ((size_t)ch * (size_t)t.H + (size_t)(g.y + (int)ly)) *
                                       (size_t)t.W + (size_t)(g.x + (int)lx);
                cfs_red_add_u32(base + off, v);
            }
        }
    }
}

/* ---- placing the windows ---------------------------------------------------
 * One CTA per frame samples the frame's first blockDim trajectories, up to
 * CFS_WIN_SAMPLES steps each past the burn-in, and gives each channel the
 * pixel box its window covers (empty when no sample of the channel landed).
 * The channels share the counters in proportion to their sampled splats (a
 * channel's capacity, in pixels, is its share, rounded down, so the windows
 * together never pass them).
 * When the channel's sampled box fits its window, the window is that box.
 * Otherwise the channel's samples are binned into a coarse grid over the
 * box, and of the windows of the channel's capacity (five aspect ratios,
 * positions on the grid's cell boundaries) the one holding the most
 * samples wins: attractors are far from uniform, and the densest region is
 * where privatizing the counters saves the most L2 reductions.  Splats
 * outside the windows still go to global memory, so the choice changes the
 * speed only, never the histogram.
 * The samples stay in shared memory (5 bytes each), so the trajectories run
 * once: running them again for every channel's box and grid took 570 us of
 * the 256-frame animation and most of a batch of a few small frames. */
#define CFS_WG 64                        /* coarse density grid: CFS_WG x CFS_WG cells */
#define CFS_WIN_SHAPES 5                 /* window aspect ratios 1/4, 1/2, 1, 2, 4 */

#define CFS_WGP (CFS_WG + 1)             /* row pitch of the grid: a column's cells in 32 banks */
struct CfsPlace {
    u32 grid[CFS_WG * CFS_WGP];
    u32 mass[CFS_A_MAX_MAPS];
    int box[CFS_A_MAX_MAPS][4];
    int2 shape[CFS_WIN_SHAPES];
    unsigned long long best;
};

/* inclusive scan of 64 values of stride `step`, two per lane, by one warp */
__device__ __forceinline__ void cfs_scan64(u32* v, int step)
{
    const int lane = (int)(threadIdx.x & 31u);
    const u32 a = v[2 * lane * step], b = v[(2 * lane + 1) * step];
    u32 s = a + b;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const u32 t = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += t;
    }
    v[2 * lane * step] = s - b;
    v[(2 * lane + 1) * step] = s;
}

/* Window shape q (width / height = 2^(q - 2), q = 0..4): at most cap pixels,
 * inside a bw x bh box, widened to the cap once the height is clamped. */
__device__ __forceinline__ int2 cfs_window_shape(int q, int cap, int bw, int bh)
{
    int ww = (int)sqrtf((float)cap * ldexpf(1.0f, q - 2));
    ww = max(1, min(ww, bw));
    const int wh = max(1, min(bh, cap / ww));
    ww = max(1, min(bw, cap / wh));
    return make_int2(ww, wh);
}

/* run(emit): this thread's trajectory, calling emit(ix, iy, channel) for at
 * most CFS_WIN_SAMPLES samples that land (ix, iy < 65536).  pos and chan:
 * CFS_WIN_SAMPLES blockDim entries each.  Writes box c of C to out[c]. */
template <class F, class Run>
__device__ __forceinline__ void cfs_place_windows(const F& t0, int C, u32 counters, CfsPlace& p,
                                                  u32* pos, unsigned char* chan, int4* out, Run run)
{
    const u32 nt = blockDim.x, tid = threadIdx.x;
    if (tid < CFS_A_MAX_MAPS) {
        p.mass[tid] = 0u;
        p.box[tid][0] = 0x7fffffff; p.box[tid][1] = 0x7fffffff;
        p.box[tid][2] = -1; p.box[tid][3] = -1;
    }
    u32 mine = 0;                       /* samples of this thread */
    run([&](int ix, int iy, int ch) {
        pos[mine * nt + tid] = (u32)ix | ((u32)iy << 16);
        chan[mine * nt + tid] = (unsigned char)ch;
        ++mine;
    });
    const int2 safe_x = cfs_safe_bins(t0.x0, t0.x1, t0.sx, t0.W);
    const int2 safe_y = cfs_safe_bins(t0.y0, t0.y1, t0.sy, t0.H);
    __syncthreads();
    /* every channel's samples and box */
    for (int c = 0; c < C; ++c) {
        int bx0 = 0x7fffffff, by0 = 0x7fffffff, bx1 = -1, by1 = -1;
        u32 n = 0;
        for (u32 q = 0; q < mine; ++q) {
            if (chan[q * nt + tid] != c) continue;
            const u32 v = pos[q * nt + tid];
            const int ix = (int)(v & 0xFFFFu), iy = (int)(v >> 16);
            bx0 = min(bx0, ix); by0 = min(by0, iy);
            bx1 = max(bx1, ix); by1 = max(by1, iy);
            ++n;
        }
        n = __reduce_add_sync(0xffffffffu, n);
        if (n == 0u) continue;
        bx0 = __reduce_min_sync(0xffffffffu, bx0);
        by0 = __reduce_min_sync(0xffffffffu, by0);
        bx1 = __reduce_max_sync(0xffffffffu, bx1);
        by1 = __reduce_max_sync(0xffffffffu, by1);
        if ((tid & 31) == 0) {
            atomicAdd(&p.mass[c], n);
            atomicMin(&p.box[c][0], bx0); atomicMin(&p.box[c][1], by0);
            atomicMax(&p.box[c][2], bx1); atomicMax(&p.box[c][3], by1);
        }
    }
    __syncthreads();
    u32 total = 0;
    for (int c = 0; c < C; ++c) total += p.mass[c];
    for (int c = 0; c < C; ++c) {
        /* window pixels of this channel */
        const int cap = total ? (int)(((unsigned long long)counters * p.mass[c]) / total) : 0;
        int4 box = make_int4(p.box[c][0], p.box[c][1], p.box[c][2], p.box[c][3]);
        const int bw = box.z - box.x + 1, bh = box.w - box.y + 1;
        if (box.z >= box.x && box.w >= box.y && cap >= 1 && (long long)bw * bh > cap) {
            /* the grid: cells of cw x ch pixels over the box, gx x gy of them */
            const int cw = (bw + CFS_WG - 1) / CFS_WG, ch = (bh + CFS_WG - 1) / CFS_WG;
            const int gx = (bw + cw - 1) / cw, gy = (bh + ch - 1) / ch;
            if (tid < CFS_WIN_SHAPES) p.shape[tid] = cfs_window_shape((int)tid, cap, bw, bh);
            if (tid == 0) p.best = 0ull;
            for (u32 e = tid; e < CFS_WG * CFS_WGP; e += nt) p.grid[e] = 0u;
            __syncthreads();
            /* a sample's cell: (v + 1/2) / cw is at least 1 / 2048 from an
             * integer and below 64, so its rounding never moves the floor */
            const float rw = 1.0f / (float)cw, rh = 1.0f / (float)ch;
            for (u32 q = 0; q < mine; ++q) {
                if (chan[q * nt + tid] != c) continue;
                const u32 v = pos[q * nt + tid];
                const int i0 = (int)(((float)((int)(v & 0xFFFFu) - box.x) + 0.5f) * rw);
                const int j0 = (int)(((float)((int)(v >> 16) - box.y) + 0.5f) * rh);
                atomicAdd(&p.grid[j0 * CFS_WGP + i0], 1u);
            }
            __syncthreads();
            /* summed-area table: rows, then columns */
            for (u32 r = tid >> 5; r < CFS_WG; r += nt >> 5) cfs_scan64(p.grid + r * CFS_WGP, 1);
            __syncthreads();
            for (u32 r = tid >> 5; r < CFS_WG; r += nt >> 5) cfs_scan64(p.grid + r, CFS_WGP);
            __syncthreads();
            /* candidates: shape q, cell position (i0, j0); the window's whole
             * cells nw x nh are counted */
            unsigned long long best = 0ull;
            for (int q = 0; q < CFS_WIN_SHAPES; ++q) {
                const int2 s = p.shape[q];
                const int nw = max(1, s.x / cw), nh = max(1, s.y / ch);
                for (u32 at = tid; at < CFS_WG * CFS_WG; at += nt) {
                    const int j0 = (int)(at / CFS_WG), i0 = (int)(at % CFS_WG);
                    if (i0 + nw > gx || j0 + nh > gy) continue;
                    auto sum = [&](int r, int col) -> u32 {
                        return (r < 0 || col < 0) ? 0u : p.grid[r * CFS_WGP + col];
                    };
                    const int r1 = j0 + nh - 1, c1 = i0 + nw - 1;
                    const u32 mass = sum(r1, c1) - sum(j0 - 1, c1) - sum(r1, i0 - 1) +
                                     sum(j0 - 1, i0 - 1);
                    /* most samples; ties to the lowest candidate number */
                    const u32 cand = (u32)q * (CFS_WG * CFS_WG) + at;
                    const unsigned long long key =
                        ((unsigned long long)mass << 32) | (unsigned long long)(0xffffffffu - cand);
                    best = key > best ? key : best;
                }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long v = __shfl_xor_sync(0xffffffffu, best, o);
                best = v > best ? v : best;
            }
            if ((tid & 31) == 0) atomicMax(&p.best, best);
            __syncthreads();
            int2 s;
            int x0, y0;
            if (p.best != 0ull) {
                const u32 cand = 0xffffffffu - (u32)(p.best & 0xffffffffull);
                const int q = (int)(cand / (CFS_WG * CFS_WG)), at = (int)(cand % (CFS_WG * CFS_WG));
                const int j0 = at / CFS_WG, i0 = at % CFS_WG;
                s = p.shape[q];
                const int nw = max(1, s.x / cw), nh = max(1, s.y / ch);
                /* centre the window on the counted cells */
                x0 = box.x + i0 * cw + (nw * cw - s.x) / 2;
                y0 = box.y + j0 * ch + (nh * ch - s.y) / 2;
            } else {                   /* (no candidate) the square shape, centred */
                s = p.shape[2];
                x0 = box.x + (bw - s.x) / 2;
                y0 = box.y + (bh - s.y) / 2;
            }
            /* inside the box */
            x0 = max(box.x, min(x0, box.z - s.x + 1));
            y0 = max(box.y, min(y0, box.w - s.y + 1));
            box = make_int4(x0, y0, x0 + s.x - 1, y0 + s.y - 1);
        } else if (cap < 1) {
            box = make_int4(0, 0, -1, -1);
        }
        /* only bins that need no view test */
        box = make_int4(max(box.x, safe_x.x), max(box.y, safe_y.x),
                        min(box.z, safe_x.x + safe_x.y - 1), min(box.w, safe_y.x + safe_y.y - 1));
        if (box.z < box.x || box.w < box.y) box = make_int4(0, 0, -1, -1);
        if (tid == 0) out[c] = box;
        __syncthreads();                /* grid, shape and best are reused */
    }
}

/* The windows of a frame from its boxes (thread 0; `off`: none): their
 * counters packed one channel after the other; none for an empty box and, as
 * a guard, for one that would pass the counters' end.  win[c]: (x0, y0,
 * w | h << 16, first counter). */
__device__ __forceinline__ void cfs_pack_windows(const int4* box, int C, u32 counters, bool off,
                                                 int4* win)
{
    u32 used = 0;
    for (int c = 0; c < C; ++c) {
        const int4 b = box[c];
        const long long w = (long long)b.z - b.x + 1, h = (long long)b.w - b.y + 1;
        if (off || w < 1 || h < 1 || w > 0xFFFF || h > 0x7FFF ||
            (long long)used + w * h > (long long)counters) {
            win[c] = make_int4(0, 0, 0, 0);
            continue;
        }
        win[c] = make_int4(b.x, b.y, (int)((u32)w | ((u32)h << 16)), (int)used);
        used += (u32)(w * h);
    }
}

#endif /* CFS_WINDOW_CUH */
