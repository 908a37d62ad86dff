// Spreading by column strips: the exponential-of-semicircle spreading of
// spread.cuh (same grid, same kernel values) for plans that sort their
// records by origin cell instead of by the tiles their supports touch.
//
// Sort.  A record is kept once, under the key of its first support cell
// (s1, s2): live 32 x 32 tile of the grid, 8-column strip of the tile, row.
// The keys of one strip are consecutive rows, so the sorted records of a
// strip come row by row.  Key starts need no order between strips: blocks of
// 1024 keys reserve their records' places with one atomic add each
// (k_strip_starts), instead of a scan through one block.  The node kernel's
// counting atomic returns each record's rank within its key, so the scatter
// needs no atomics of its own.
//
// Spread.  A warp takes a fixed range of sorted records, whatever strips
// they fall in (dense clusters and empty regions balance by themselves), and
// sweeps each strip downwards: the strip's 8 origin columns plus the support
// are at most 7 + w columns wide, and only w rows are open at a time, kept as
// accumulators indexed by the row modulo their number.  Moving on by d rows
// adds the d finished rows to the grid with vector reductions; a record's
// kernel values along y are read from the slot (row - s2), which changes only
// when the sweep moves.  The grid must be zero on entry: the row pass of the
// FFT zeroes the nonzero cells that it reads.
//
// Rounding.  An addition to the grid rounds the whole sum of a cell, so where
// much of a problem's sum lies in a few cells (a starshade on a coarse pupil
// grid) the additions per cell decide the error.  Plans with such a problem
// (see build_plan) run with MERGE: a block takes the tile kernel's chunk of
// records (512 in FP32, 256 in FP64, more in large plans), its warps
// neighbouring ranges of it, and the rows that the warps hold at the end are
// summed in shared memory before they are added: a cell gets one addition per
// block, strip and row sweep, about as many as the tile kernel made, whatever
// the density.  FP32 adds in two levels besides, a batch's sums and the
// range's: runs of 128 additions to one cell would round 10 to 25 % more than
// the tile kernel's interleaved warps.
//
// FP32 (k_spread_strips_f32): accumulators in registers, a lane owning 4
// columns of one row (w <= 8: 16 x 8 cells on 32 lanes; wider kernels own
// more rows), so a record costs a 16-byte and an 8-byte shared load and 8
// multiply-adds per lane.  Half of the 16 columns are padding, which costs
// less than the tile kernel's read-modify-writes and duplicated records (1.5
// per node at w = 8).  Bound by the shared-memory return path (6 words per
// lane and record; L1 89 % busy at 4.3M records) and, where runs are short,
// by issue.  Cold L2, start (tiles) and now: star at F = 100, 524,288 records,
// 65.5 -> 28.7 us; Koch snowflake, 4.27M, 379 -> 141 us; starshade sweep, 978k on 64
// x 28 keys, 71.7 -> 32.8 us (MERGE; 34.8 without).
// FP64 (k_spread_strips_f64): the FP64 pipe (1/58 of the FP32 rate) bounds
// it, so no multiply-add goes to padding: lanes walk the w x w support
// (ceil(w^2 / 32) steps) on a private 16-row window in shared memory.  Star,
// w = 13: 1649 -> 609 us; w = 10: 1016 -> 392 us.
#pragma once
#include <algorithm>

#include "spread.cuh"

namespace fres {

// Most warps of a block; MERGE: by registers (FP32: a lane holds one row up to
// w = 8, then two, then four) and shared memory (FP64: 19 KB per warp at w = 16).
template <typename T, int W, bool MERGE>
constexpr int strip_warps() {
    return !MERGE ? 4 : (sizeof(T) == 8 ? 12 : (W <= 8 ? 32 : (W == 9 ? 16 : 8)));
}

// The rows that the block's warps hold open at the end, added to the grid:
// open = (strip, first row) of the calling warp (strip -1: none), whose cell
// (y, x) is win(the warp's Smem, y, x), for open.y <= y < open.y + W.
// Warps that hold the same strip of one tile row (neighbours: records are
// sorted) are summed first, each adding its share of the rows.  V: the sum of
// STEP neighbouring cells; add takes the first one's place in the (periodic,
// stacked) grids and the sum.
template <typename V, int W, int COLS, int STEP, class Smem, class Win, class Add>
__device__ __forceinline__ void add_open_rows(Smem* sm, int2 open, int nf1, int nf2, Win win, Add add) {
    __shared__ int2 s_open[32];
    constexpr int QC = COLS / STEP;
    const int warps = blockDim.x >> 5, lane = threadIdx.x & 31, me = threadIdx.x >> 5;
    if (lane == 0) s_open[me] = open;
    __syncthreads();
    // this warp's neighbours v .. e - 1 of the same strip, first rows ascending
    const int2 o = lane < warps ? s_open[lane] : make_int2(-1, 0);
    const int pa = __shfl_up_sync(0xffffffffu, o.x, 1), pb = __shfl_up_sync(0xffffffffu, o.y, 1);
    const unsigned first = __ballot_sync(
        0xffffffffu, lane == 0 || lane >= warps || o.x != pa || (o.y >> 5) != (pb >> 5) || o.y < pb);
    const int v = 31 - __clz(first & (0xffffffffu >> (31 - me)));
    const unsigned next = me < 31 ? first >> (me + 1) : 0u;
    const int e = next ? me + __ffs(next) : warps;
    if (open.x >= 0) {
        const int y0 = s_open[v].y, yend = (y0 / nf2 + 1) * nf2;
        for (int t = (me - v) * 32 + lane; t < (s_open[e - 1].y - y0 + W) * QC; t += (e - v) * 32) {
            const int y = y0 + t / QC, x = t % QC * STEP;
            V s{};
            for (int u = v; u < e; ++u) {
                const int d = y - s_open[u].y;
                if (d >= 0 && d < W) {
                    const V c = win(sm[u], y, x);
                    s.x += c.x;
                    s.y += c.y;
                    if constexpr (STEP == 2) {
                        s.z += c.z;
                        s.w += c.w;
                    }
                }
            }
            int gx = open.x * 8 + x;
            if (gx >= nf1) gx -= nf1;
            add(gx, y >= yend ? y - nf2 : y, s);
        }
    }
}

// ------------------------------------------------------------------ FP32
template <int W>
struct StripMap {
    static constexpr int COLG = W <= 9 ? 4 : 8;          // 4-column groups
    static constexpr int COLS = 4 * COLG;                // >= 7 + W
    static constexpr int ROWS = W <= 8 ? 8 : 16;         // open rows (power of two >= W)
    static constexpr int RSTEP = 32 / COLG;
    static constexpr int RPL = ROWS / RSTEP;             // rows per lane
    static constexpr int NQ = (W + 3 + 3) / 4;           // quads of a kernel row shifted by 0..3
};

// 16-byte rows whose strides (20 or 36 words) keep the staging stores and
// the row reads free of bank conflicts.  At the end a warp's open rows take
// the place of kx: row y in slot y mod ROWS
template <int W>
struct StripSmemF {
    using M = StripMap<W>;
    float kx[32][M::COLS + 4];
    float2 ck[32][M::ROWS + 2];
};

template <int W, bool MERGE>
__global__ void __launch_bounds__(strip_warps<float, W, MERGE>() * 32)
k_spread_strips_f32(const NodeRec<float>* __restrict__ sorted, long long n, int range,
                    float2* __restrict__ grid, int nf1, int nf2, float beta, const HornerTab hz) {
    using M = StripMap<W>;
    static_assert(M::ROWS * M::COLS * sizeof(float2) <= sizeof(StripSmemF<W>::kx), "open rows");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    StripSmemF<W>* sm = reinterpret_cast<StripSmemF<W>*>(smem_raw);
    kernel_begin();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const long long beg = ((long long)blockIdx.x * (blockDim.x >> 5) + warp) * range;
    const long long end = beg + range < n ? beg + range : n;   // <= beg: no records
    float(*kx)[M::COLS + 4] = sm[warp].kx;
    float2(*ck)[M::ROWS + 2] = sm[warp].ck;
#pragma unroll
    for (int b = W; b < M::ROWS; ++b) ck[lane][b] = make_float2(0.0f, 0.0f);
    const int cg = lane % M::COLG, rg = lane / M::COLG;
    float2 acc[M::RPL][4];           // this batch's sums
    float2 sum[M::RPL][4];           // the earlier batches'
    int slot[M::RPL];                // this lane's rows relative to the open row
    const float2* ckp[M::RPL];       // their staged values (of record 0)
    const float4* kxp = reinterpret_cast<const float4*>(&kx[0][4 * cg]);
    constexpr int KXS = (M::COLS + 4) / 4, CKS = M::ROWS + 2;   // strides of a record
    int cur_a = -1, cur_b = 0;       // open strip (s1 / 8) and row
    int yend = 0;                    // end of the problem's rows (stacked grids)
    float2* colp = grid;             // this lane's first column
#pragma unroll
    for (int k = 0; k < M::RPL; ++k) {
        slot[k] = 0;
        ckp[k] = &ck[0][0];
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[k][i] = sum[k][i] = make_float2(0.0f, 0.0f);
    }
    auto fold = [&](int k) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            sum[k][i].x += acc[k][i].x;
            sum[k][i].y += acc[k][i].y;
            acc[k][i] = make_float2(0.0f, 0.0f);
        }
    };
    // adds the rows less than d below the open one to the grid (a row's zero
    // cells too: they stay inside the grid, and testing costs more)
    auto flush = [&](int d) {
#pragma unroll
        for (int k = 0; k < M::RPL; ++k)
            if (slot[k] < d) {
                int y = cur_b + slot[k];
                if (y >= yend) y -= nf2;
                float2* dst = colp + (long long)y * nf1;
                fold(k);
                asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst),
                             "f"(sum[k][0].x), "f"(sum[k][0].y), "f"(sum[k][1].x),
                             "f"(sum[k][1].y)
                             : "memory");
                asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst + 2),
                             "f"(sum[k][2].x), "f"(sum[k][2].y), "f"(sum[k][3].x),
                             "f"(sum[k][3].y)
                             : "memory");
#pragma unroll
                for (int i = 0; i < 4; ++i) sum[k][i] = make_float2(0.0f, 0.0f);
            }
    };
    NodeRec<float> r{};
    if (beg + lane < end) r = sorted[beg + lane];
    for (long long base = beg; base < end; base += 32) {
        const int cnt = (int)(end - base < 32 ? end - base : 32);
        const int a = r.s1 >> 3, b = r.s2;
        {
            // lanes beyond the last record stage zeros (strength 0)
            float kxv[W], kyv[W];
            kernel_values<float, W>(r.f1, beta, hz, kxv);
            kernel_values<float, W>(r.f2, beta, hz, kyv);
            const float cre = lane < cnt ? r.cre : 0.0f, cim = lane < cnt ? r.cim : 0.0f;
            // the x values shifted right by s1 mod 8: by 0..3 in registers, by
            // 0 or 4 through the address; the other slots are zero
            const int dx = r.s1 & 7;
            float t1[W + 1], t2[4 * M::NQ];
#pragma unroll
            for (int i = 0; i <= W; ++i) {
                const float v0 = i < W ? kxv[i < W ? i : 0] : 0.0f;
                const float v1 = i >= 1 ? kxv[i >= 1 ? i - 1 : 0] : 0.0f;
                t1[i] = (dx & 1) ? v1 : v0;
            }
#pragma unroll
            for (int i = 0; i < 4 * M::NQ; ++i) {
                const float v0 = i <= W ? t1[i <= W ? i : 0] : 0.0f;
                const float v2 = i >= 2 && i - 2 <= W ? t1[i >= 2 && i - 2 <= W ? i - 2 : 0] : 0.0f;
                t2[i] = (dx & 2) ? v2 : v0;
            }
            float4* kq = reinterpret_cast<float4*>(kx[lane]);
            const int q0 = dx >> 2;
#pragma unroll
            for (int q = 0; q < M::COLG; ++q) {
                float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (q < M::NQ) {
                    v.x = t2[q < M::NQ ? 4 * q : 0];
                    v.y = t2[q < M::NQ ? 4 * q + 1 : 0];
                    v.z = t2[q < M::NQ ? 4 * q + 2 : 0];
                    v.w = t2[q < M::NQ ? 4 * q + 3 : 0];
                }
                kq[(q0 + q) & (M::COLG - 1)] = v;
            }
#pragma unroll
            for (int i = 0; i + 1 < W; i += 2)
                *reinterpret_cast<float4*>(&ck[lane][i]) =
                    make_float4(cre * kyv[i], cim * kyv[i], cre * kyv[i + 1], cim * kyv[i + 1]);
            if (W % 2) ck[lane][W - 1] = make_float2(cre * kyv[W - 1], cim * kyv[W - 1]);
        }
        // the next batch's records, in flight during this one
        if (base + 32 + lane < end) r = sorted[base + 32 + lane];
        int pa = __shfl_up_sync(0xffffffffu, a, 1), pb = __shfl_up_sync(0xffffffffu, b, 1);
        if (lane == 0) {
            pa = cur_a;
            pb = cur_b;
        }
        // records where the sweep moves to another row or strip
        unsigned moves = __ballot_sync(0xffffffffu, lane < cnt && (a != pa || b != pb));
        __syncwarp();
#pragma unroll 1
        for (int j0 = 0; j0 < cnt; j0 += 4, moves >>= 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int j = j0 + u;
                if (moves & (1u << u)) {
                    const int na = __shfl_sync(0xffffffffu, a, j);
                    const int nb = __shfl_sync(0xffffffffu, b, j);
                    const bool same = na == cur_a && (nb >> 5) == (cur_b >> 5) && nb > cur_b;
                    if (cur_a >= 0) flush(same ? nb - cur_b : M::ROWS);
                    if (!same) {
                        int x = na * 8 + 4 * cg;
                        if (x >= nf1) x -= nf1;
                        colp = grid + x;
                        yend = (nb / nf2 + 1) * nf2;
                        cur_a = na;
                    }
                    cur_b = nb;
#pragma unroll
                    for (int k = 0; k < M::RPL; ++k) {
                        slot[k] = (rg + k * M::RSTEP - nb) & (M::ROWS - 1);
                        ckp[k] = &ck[0][slot[k]];
                    }
                }
                const float4 kv = kxp[j * KXS];
#pragma unroll
                for (int k = 0; k < M::RPL; ++k) {
                    const float2 c = ckp[k][j * CKS];
                    acc[k][0].x = fmaf(c.x, kv.x, acc[k][0].x);
                    acc[k][0].y = fmaf(c.y, kv.x, acc[k][0].y);
                    acc[k][1].x = fmaf(c.x, kv.y, acc[k][1].x);
                    acc[k][1].y = fmaf(c.y, kv.y, acc[k][1].y);
                    acc[k][2].x = fmaf(c.x, kv.z, acc[k][2].x);
                    acc[k][2].y = fmaf(c.y, kv.z, acc[k][2].y);
                    acc[k][3].x = fmaf(c.x, kv.w, acc[k][3].x);
                    acc[k][3].y = fmaf(c.y, kv.w, acc[k][3].y);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < M::RPL; ++k) fold(k);
        __syncwarp();   // the next batch overwrites the staged values
    }
    if constexpr (!MERGE) {
        if (cur_a >= 0) flush(M::ROWS);
        return;
    }
    // what is still open, summed over the block's warps
    float2* win = reinterpret_cast<float2*>(kx);
#pragma unroll
    for (int k = 0; k < M::RPL; ++k) {
        fold(k);
#pragma unroll
        for (int i = 0; i < 4; i += 2)
            *reinterpret_cast<float4*>(win + (rg + k * M::RSTEP) * M::COLS + 4 * cg + i) =
                make_float4(sum[k][i].x, sum[k][i].y, sum[k][i + 1].x, sum[k][i + 1].y);
    }
    add_open_rows<float4, W, M::COLS, 2>(
        sm, make_int2(cur_a, cur_b), nf1, nf2,
        [](const StripSmemF<W>& w, int y, int x) {
            return *reinterpret_cast<const float4*>(reinterpret_cast<const float2*>(w.kx) +
                                                    (y & (M::ROWS - 1)) * M::COLS + x);
        },
        [&](int x, int y, float4 v) {
            if (v.x == 0.0f && v.y == 0.0f && v.z == 0.0f && v.w == 0.0f) return;
            asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(
                             grid + (long long)y * nf1 + x),
                         "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
                         : "memory");
        });
}

// ------------------------------------------------------------------ FP64
template <int W>
struct StripSmemD {
    static constexpr int COLS = W + 7;
    double2 win[16 * COLS];
    double2 ck[32][W | 1];
    double kx[32][W | 1];
};

template <int W, bool MERGE>
__global__ void __launch_bounds__(strip_warps<double, W, MERGE>() * 32)
k_spread_strips_f64(const NodeRec<double>* __restrict__ sorted, long long n, int range,
                    double2* __restrict__ grid, int nf1, int nf2, double beta,
                    const HornerTabD hz) {
    constexpr int COLS = StripSmemD<W>::COLS;
    constexpr int NP = (W * W + 31) / 32;      // support cells per lane
    extern __shared__ __align__(16) unsigned char smem_raw[];
    kernel_begin();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    StripSmemD<W>* all = reinterpret_cast<StripSmemD<W>*>(smem_raw);
    StripSmemD<W>& sm = all[warp];
    const long long beg = ((long long)blockIdx.x * (blockDim.x >> 5) + warp) * range;
    const long long end = beg + range < n ? beg + range : n;   // <= beg: no records
    double2* win = sm.win;
    for (int e = lane; e < 16 * COLS; e += 32) win[e] = make_double2(0.0, 0.0);
    int ca[NP], cb[NP], off[NP];               // cell (a, b) of step k, its window offset
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int e = lane + 32 * k;
        ca[k] = e % W;
        cb[k] = e / W;                         // >= W: no cell
        off[k] = 0;
    }
    int cur_a = -1, cur_b = 0, yend = 0;
    auto flush = [&](int d) {
        __syncwarp();
        d = d < W ? d : W;
        int x = cur_a * 8 + lane;
        if (x >= nf1) x -= nf1;
        for (int o = 0; o < d; o += 2) {
            double2 v[2];
#pragma unroll
            for (int i = 0; i < 2; ++i)
                v[i] = o + i < d && lane < COLS ? win[((cur_b + o + i) & 15) * COLS + lane]
                                                : make_double2(0.0, 0.0);
#pragma unroll
            for (int i = 0; i < 2; ++i)
                if (nonzero(v[i])) {
                    const int y = cur_b + o + i;
                    win[(y & 15) * COLS + lane] = make_double2(0.0, 0.0);
                    double2* g = grid + (long long)(y >= yend ? y - nf2 : y) * nf1 + x;
                    atomicAdd(&g->x, v[i].x);
                    atomicAdd(&g->y, v[i].y);
                }
        }
        __syncwarp();
    };
    NodeRec<double> r{};
    if (beg + lane < end) r = sorted[beg + lane];
    for (long long base = beg; base < end; base += 32) {
        const int cnt = (int)(end - base < 32 ? end - base : 32);
        const int a = r.s1 >> 3, b = r.s2, dx = r.s1 & 7;
        if (lane < cnt) {
            double kv[W];
            kernel_values<double, W>(r.f1, beta, hz, kv);
#pragma unroll
            for (int i = 0; i < W; ++i) sm.kx[lane][i] = kv[i];
            kernel_values<double, W>(r.f2, beta, hz, kv);
#pragma unroll
            for (int i = 0; i < W; ++i)
                sm.ck[lane][i] = make_double2(r.cre * kv[i], r.cim * kv[i]);
        }
        if (base + 32 + lane < end) r = sorted[base + 32 + lane];
        int pa = __shfl_up_sync(0xffffffffu, a, 1), pb = __shfl_up_sync(0xffffffffu, b, 1);
        if (lane == 0) {
            pa = cur_a;
            pb = cur_b;
        }
        const unsigned moves = __ballot_sync(0xffffffffu, lane < cnt && (a != pa || b != pb));
        __syncwarp();
        for (int j = 0; j < cnt; ++j) {
            if ((moves >> j) & 1u) {
                const int na = __shfl_sync(0xffffffffu, a, j), nb = __shfl_sync(0xffffffffu, b, j);
                const bool same = na == cur_a && (nb >> 5) == (cur_b >> 5) && nb > cur_b;
                if (cur_a >= 0) flush(same ? nb - cur_b : W);
                if (!same) {
                    yend = (nb / nf2 + 1) * nf2;
                    cur_a = na;
                }
                cur_b = nb;
#pragma unroll
                for (int k = 0; k < NP; ++k) off[k] = ((nb + cb[k]) & 15) * COLS + ca[k];
            }
            const int x0 = __shfl_sync(0xffffffffu, dx, j);
#pragma unroll
            for (int k = 0; k < NP; ++k)
                if (cb[k] < W) {
                    const double kv = sm.kx[j][ca[k]];
                    const double2 c = sm.ck[j][cb[k]];
                    double2* cell = win + off[k] + x0;
                    double2 o = *cell;
                    o.x += c.x * kv;
                    o.y += c.y * kv;
                    *cell = o;
                }
            __syncwarp();
        }
    }
    if constexpr (!MERGE) {
        if (cur_a >= 0) flush(W);
        return;
    }
    add_open_rows<double2, W, COLS, 1>(
        all, make_int2(cur_a, cur_b), nf1, nf2,
        [](const StripSmemD<W>& w, int y, int x) { return w.win[(y & 15) * COLS + x]; },
        [&](int x, int y, double2 v) {
            if (!nonzero(v)) return;
            double2* g = grid + (long long)y * nf1 + x;
            atomicAdd(&g->x, v.x);
            atomicAdd(&g->y, v.y);
        });
}

// Records per warp and warps per block.  FP32: enough warps for every SM's
// resident set (152 x 32), at least one batch and at most four.  FP64 records
// cost far more than a flush, so the split that balances the SMs wins: two
// batches per warp, one below 16 warps per SM.  MERGE: a block takes `cap`
// records, the plan's chunk of the tile kernel, or up to twice as many where
// that loads the fullest SM less (117,000 records: 800 instead of 2 x 512); in
// large FP32 plans (cap above its base) eight warps, so that the last blocks
// are short.
inline void strip_shape(long long n, int cap, bool dbl, bool merge, int most, int* range, int* warps) {
    const int base = dbl ? 256 : 512;
    const int few = dbl ? 64 : 128;
    long long r = dbl ? (n < 152LL * 16 * 64 ? 32 : 64) : (n / (152 * 32) + 31) / 32 * 32;
    r = r < 32 ? 32 : (r > few ? few : r);
    *warps = most;
    *range = (int)r;
    if (!merge) return;
    while (base % r || base / r > most) r += 32;   // 32, 64 or 128
    int w = !dbl && cap > base ? 8 : (int)(base / r);
    long long load = -1;
    for (int k = w; cap == base && k <= std::min(most, (int)(2 * base / r)); ++k) {
        const long long per = k * r, l = ((n + per - 1) / per + 151) / 152 * per;
        if (load < 0 || l < load) {
            load = l;
            w = k;
        }
    }
    *warps = w;
    *range = std::max((int)r, (cap / w + 31) / 32 * 32);
}

template <typename T, int W, bool MERGE>
void launch_strips_w(const NodeRec<T>* sorted, long long n, int cap, cx_t<T>* grid, int nf1, int nf2,
                     const KernelShape& ks, cudaStream_t st) {
    int range, warps;
    strip_shape(n, cap, sizeof(T) == 8, MERGE, strip_warps<T, W, MERGE>(), &range, &warps);
    const long long per = (long long)range * warps;
    auto launch = [&](auto kernel, size_t smem, auto beta, const auto& horner) {
        if (smem > 48 * 1024)
            cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        kernel<<<(unsigned)((n + per - 1) / per), warps * 32, smem, st>>>(sorted, n, range, grid, nf1,
                                                                          nf2, beta, horner);
    };
    if constexpr (sizeof(T) == 4)
        launch(k_spread_strips_f32<W, MERGE>, warps * sizeof(StripSmemF<W>), ks.betaf, ks.horner);
    else
        launch(k_spread_strips_f64<W, MERGE>, warps * sizeof(StripSmemD<W>), ks.beta, ks.hornerd);
}

template <typename T>
void launch_strips_impl(const NodeRec<T>* sorted, long long n, int cap, bool merge, cx_t<T>* grid,
                        int nf1, int nf2, const KernelShape& ks, cudaStream_t st) {
    if (n <= 0) return;
#define FRES_STRIP_CASE(WW)                                                                  \
    case WW:                                                                                 \
        if (merge) launch_strips_w<T, WW, true>(sorted, n, cap, grid, nf1, nf2, ks, st);     \
        else launch_strips_w<T, WW, false>(sorted, n, cap, grid, nf1, nf2, ks, st);          \
        break;
    switch (ks.w) {
        FRES_STRIP_CASE(2) FRES_STRIP_CASE(3) FRES_STRIP_CASE(4) FRES_STRIP_CASE(5)
        FRES_STRIP_CASE(6) FRES_STRIP_CASE(7) FRES_STRIP_CASE(8) FRES_STRIP_CASE(9)
        FRES_STRIP_CASE(10) FRES_STRIP_CASE(11) FRES_STRIP_CASE(12) FRES_STRIP_CASE(13)
        FRES_STRIP_CASE(14) FRES_STRIP_CASE(15) FRES_STRIP_CASE(16)
        default: break;
    }
#undef FRES_STRIP_CASE
}

}  // namespace fres
