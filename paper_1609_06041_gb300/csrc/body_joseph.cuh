// body_joseph.cuh -- bodies of the mirrored Joseph projector and of the rotation-orbit backprojector, shared by their kernels
// (k_joseph.cu) and the persistent batched kernel (persist.cu).  Each body
// takes its block index and shared memory explicitly and runs on the
// threads of a context (a whole block or a group of a persistent block).
#pragma once

#include "ctpd_internal.cuh"

namespace ctpd {

__device__ __forceinline__ float joseph_h(int n) { return 0.5f * (float)(n - 1); }
__device__ __forceinline__ float joseph_dp(int d, int B) { return __fsub_rn((float)d, 0.5f * (float)(B - 1)); }

constexpr int PG = 16;         // views per block
constexpr int MR = 16;         // steps per band (two bands per block)

// Conservative integer range [lo, hi] within [s_lo, s_hi] of the steps s
// for which u'(s) = q + (s - h) m can lie in [ulo, uhi] (empty if lo > hi).
__device__ __forceinline__ void step_range(float q, float m, float inv_m, float h, float ulo, float uhi,
                                           int s_lo, int s_hi, int &lo, int &hi)
{
    if (m == 0.0f) {
        lo = s_lo;
        hi = (q >= ulo && q <= uhi) ? s_hi : s_lo - 1;
        return;
    }
    // explicit roundings: every kernel that walks a ray finds the same range
    float sa = __fmaf_rn(__fsub_rn(ulo, q), inv_m, h), sb = __fmaf_rn(__fsub_rn(uhi, q), inv_m, h);
    float smin = fminf(sa, sb), smax = fmaxf(sa, sb);
    // clamp before converting: far-off rays give huge (or infinite) s
    smin = fminf(fmaxf(smin, (float)s_lo - 2.0f), (float)s_hi + 2.0f);
    smax = fminf(fmaxf(smax, (float)s_lo - 2.0f), (float)s_hi + 2.0f);
    lo = max(s_lo, (int)floorf(smin) - 1);
    hi = min(s_hi, (int)ceilf(smax) + 1);
}

// Shared memory of the mirrored projector's staged band pair at image side
// N: float4 entries (one per step and pair), or raw (float2 pixel pairs).
__host__ __device__ __forceinline__ size_t quad_smem(int N, bool raw = false)
{
    return raw ? sizeof(float2) * (size_t)MR * ((N + 4) | 1) : sizeof(float4) * (size_t)MR * ((N + 3) | 1);
}
// Band pairs of N image lines: pair bp holds the lines s0 .. s0 + 15, s0 = 16
// bp, of the first half (the middle line of an odd N included) and their
// mirrors N-1-s.
__host__ __device__ __forceinline__ int quad_bands(int N) { return (N + 2 * MR - 1) / (2 * MR); }

// ---------------------------------------------------------------------
// Forward projection with the detector mirror and, at the default angles t_v
// = v pi / V, the view mirror.  Ray B-1-d meets step N-1-s at the mirrored
// coordinate N-1-u of ray d at step s, so a block that stages band A (steps
// s0 .. s0+15) and band B (steps N-1-s0-15 .. N-1-s0) turned by 180 degrees
// (step and pair order reversed) reads, for one evaluation of (u', g) at (d,
// s), the sample of ray d in band A and of ray B-1-d in band B at the same
// shared offset.  View V-v is view v reflected in the image's vertical axis:
// its a and m are those of view v with the signs a row view (a -> -a, m ->
// -m) or a column view (m -> -m) gets from t -> pi - t.  For a row view that
// puts ray d of view V-v at coordinate N-1-u on the same row; for a column
// view ray d of view V-v meets column N-1-c where ray d of view v meets
// column c, i.e. the other band's line.  Either way the reflected sample
// sits at pair N-2-i0 of a staged line with weight -g: one evaluation yields
// four samples, two of view v and two of view V-v:
//     rows:    A[i0] (v, d)  B[i0] (v, B-1-d)  A[N-2-i0] (V-v, d)    B[N-2-i0] (V-v, B-1-d)
//     columns: A[i0] (v, d)  B[i0] (v, B-1-d)  A[N-2-i0] (V-v, B-1-d) B[N-2-i0] (V-v, d)
// Work items are view pairs (v, V-v) and the views without a partner (v = 0,
// v = V/2 for even V; at custom angles every view), pg items per block, tpi
// threads per item.
// ---------------------------------------------------------------------
// Walks one ray through the staged steps lo..hi (ROWS steps per pass, one
// coordinate evaluation per step) and returns its four sums: band A and
// band B at the pair i0, and (PAIR) at the reflected pair N-2-i0.  Q holds
// per step and pair (A mid, B mid, A delta, B delta), so one 16-byte load
// serves both bands and the two bands' samples are one packed two-wide
// FMA, mid + g delta, into a pair accumulator (the reflected pair with -g).
// The coordinates of two steps are evaluated as one packed pair as well.
// RAW: the staged entries are the bands' pixels (A_i, B_i) instead, and a
// sample reads the entries i and i + 1: with mid = (a + b) / 2 and delta =
// b - a formed on the fly, mid + g delta is rounded exactly as from float4
// entries, at half the shared memory and two more packed operations.
// A pass of ROWS = 4 is two passes of ROWS = 2 whose loads are issued
// together: the same coordinates (u' = (s - h) m + q for even steps,
// (s - 1 - h) m + (q + m) for odd ones), the same two accumulators (even
// and odd steps) updated in the same order and the same tail, so both
// give the same sums to the bit.
template <bool PAIR, int ROWS, bool RAW>
__device__ __forceinline__ float4 quad_walk(const void *Qv, int SP, float q, float m, int lo, int hi,
                                            int s0, float h, unsigned top)
{
    static_assert(ROWS == 2 || ROWS == 4, "steps are evaluated in pairs, one or two pairs per pass");
    // one sample's entry: (mid A, mid B, delta A, delta B), or raw pixels (A_i, B_i, A_i+1, B_i+1)
    auto entry = [&](int k) {
        if constexpr (RAW) {
            const float2 *R = static_cast<const float2 *>(Qv);
            const float2 x0 = R[k], x1 = R[k + 1];
            return make_float4(x0.x, x0.y, x1.x, x1.y);
        } else {
            return static_cast<const float4 *>(Qv)[k];
        }
    };
    // acc + mid + g delta: acc + mid rounds, then the FMA
    auto sample = [&](float2 acc, const float4 &p, float g) {
        if constexpr (RAW) {
            const float2 x0 = pk(p.x, p.y), x1 = pk(p.z, p.w);
            return pfma(pk(g, g), psub(x1, x0), pfma(pk(0.5f, 0.5f), padd(x0, x1), acc));
        } else {
            return pfma(pk(g, g), pk(p.z, p.w), padd(acc, pk(p.x, p.y)));
        }
    };
    const float2 qk = pk(q, __fmaf_rn(1.0f, m, q));   // q + k m for the steps k = 0, 1 of a pair
    const float2 mm = pk(m, m), bias = pk(JOSEPH_BIAS, JOSEPH_BIAS);
    float spk = (float)lo - h;
    int ridx = (lo - s0) * SP;
    float2 ab[2], ce[2];   // (band A, band B) sums of the even and odd steps, at i0 and at the reflected pair
    ab[0] = ab[1] = ce[0] = ce[1] = pk(0.0f, 0.0f);
    // the samples of the steps s and s + 1, at (s - h) = sp
    auto pair_samples = [&](float sp, int rr, float4 &p0, float4 &p1, float4 &r0, float4 &r1, float2 &g) {
        const float2 up = pfma(pk(sp, sp), mm, qk);
        const float2 t = padd(up, bias);
        const float2 tb = psub(t, bias);
        g = psub(up, tb);
        const unsigned i0 = min((unsigned)(__float_as_int(t.x) - (JOSEPH_BIAS_BITS - 2)), top);
        const unsigned i1 = min((unsigned)(__float_as_int(t.y) - (JOSEPH_BIAS_BITS - 2)), top);
        p0 = entry(rr + (int)i0);
        p1 = entry(rr + SP + (int)i1);
        if (PAIR) {
            r0 = entry(rr + (int)(top - i0));
            r1 = entry(rr + SP + (int)(top - i1));
        }
    };
    auto pair_add = [&](const float4 &p0, const float4 &p1, const float4 &r0, const float4 &r1, float2 g) {
        ab[0] = sample(ab[0], p0, g.x);
        ab[1] = sample(ab[1], p1, g.y);
        if (PAIR) {
            ce[0] = sample(ce[0], r0, -g.x);
            ce[1] = sample(ce[1], r1, -g.y);
        }
    };
    int s = lo;
    for (; s + ROWS - 1 <= hi; s += ROWS) {
        float4 p[ROWS], r[ROWS];
        float2 g[ROWS / 2];
#pragma unroll
        for (int k = 0; k < ROWS / 2; ++k)
            pair_samples(k == 0 ? spk : __fadd_rn(spk, (float)(2 * k)), ridx + 2 * k * SP, p[2 * k], p[2 * k + 1],
                         r[2 * k], r[2 * k + 1], g[k]);
#pragma unroll
        for (int k = 0; k < ROWS / 2; ++k) pair_add(p[2 * k], p[2 * k + 1], r[2 * k], r[2 * k + 1], g[k]);
        spk = __fadd_rn(spk, (float)ROWS);
        ridx += ROWS * SP;
    }
    if (ROWS == 4 && s + 1 <= hi) {   // the pair ROWS = 2 would still take
        float4 p0, p1, r0, r1;
        float2 g;
        pair_samples(spk, ridx, p0, p1, r0, r1, g);
        pair_add(p0, p1, r0, r1, g);
        spk = __fadd_rn(spk, 2.0f);
        ridx += 2 * SP;
        s += 2;
    }
    if (s <= hi) {   // one step left
        const float up = joseph_u(spk, m, qk.x);
        const float t = __fadd_rn(up, JOSEPH_BIAS);
        const unsigned i = min((unsigned)(__float_as_int(t) - (JOSEPH_BIAS_BITS - 2)), top);
        const float g = __fsub_rn(up, __fsub_rn(t, JOSEPH_BIAS));
        ab[0] = sample(ab[0], entry(ridx + (int)i), g);
        if (PAIR) ce[0] = sample(ce[0], entry(ridx + (int)(top - i)), -g);
    }
    ab[0] = padd(ab[0], ab[1]);
    ce[0] = padd(ce[0], ce[1]);
    return make_float4(ab[0].x, ab[0].y, ce[0].x, ce[0].y);
}

// Stages band pair s0 of image img: entry i of step t (stored at i + 2,
// -2 <= i <= N) holds (A mid, B mid, A delta, B delta), band A the image line
// s0 + t and band B the line N-1-s0-t read backwards (image value at N-1-i);
// the lines are image rows (rows) or columns.  RAW: the pixels (A_i, B_i),
// i <= N + 1.  Steps past the first half hold zeros, as does band B on the
// middle line of an odd N (band A has it).  Every pixel is loaded once and
// its neighbour comes by shuffle; a thread issues the loads of four entries
// before it stores any, and the index arithmetic has no division (staging a
// 512-line segment took 170 instructions per 32 entries with both, about 30
// now).  Runs on the threads of c and ends without a barrier.
template <bool RAW, class Ctx>
__device__ __forceinline__ void quad_stage(const Ctx &c, void *Qv, const float *img, int N, int s0, bool rows)
{
    static_assert(MR == 16, "a warp's lanes take the 16 steps of two entries (columns)");
    constexpr unsigned FULL = 0xffffffffu;
    constexpr int SU = 4;
    const int CW = RAW ? N + 4 : N + 3, SP = CW | 1;
    const int lane = c.tid() & 31, nw = c.nth() >> 5;
    const int na = min(MR, (N + 1) / 2 - s0), nb = min(MR, N / 2 - s0);   // lines of bands A and B
    const int last = N * N - 1;                                            // N N < 2^31
    auto store = [&](int at, float a0, float a1, float b0, float b1) {
        if constexpr (RAW) static_cast<float2 *>(Qv)[at] = make_float2(a0, b0);
        else
            static_cast<float4 *>(Qv)[at] = make_float4(0.5f * (a0 + a1), 0.5f * (b0 + b1), a1 - a0, b1 - b0);
    };
    if (rows) {
        // a warp takes a chunk of 31 entries (RAW: 32) of one step; lane 31 loads the last entry's neighbour
        constexpr int CH = RAW ? 32 : 31;
        const int nc = MR * ((CW + CH - 1) / CH);
        for (int k0 = c.tid() >> 5; k0 < nc; k0 += SU * nw) {
            float av[SU], bv[SU];
#pragma unroll
            for (int u = 0; u < SU; ++u) {
                const int k = k0 + u * nw, t = k & (MR - 1), i = (k >> 4) * CH + lane - 2, o = (s0 + t) * N + i;
                const bool in = k < nc && (unsigned)i < (unsigned)N;
                av[u] = in && t < na ? img[o] : 0.0f;
                bv[u] = in && t < nb ? img[last - o] : 0.0f;
            }
#pragma unroll
            for (int u = 0; u < SU; ++u) {
                const int k = k0 + u * nw, t = k & (MR - 1), ii = (k >> 4) * CH + lane;
                float a1 = 0.0f, b1 = 0.0f;
                if (!RAW) {
                    a1 = __shfl_down_sync(FULL, av[u], 1);
                    b1 = __shfl_down_sync(FULL, bv[u], 1);
                }
                if (k < nc && lane < CH && ii < CW) store(t * SP + ii, av[u], a1, bv[u], b1);
            }
        }
    } else {
        // a warp takes 2 SU neighbouring entries: the lane's step t, entries e0 + 2 u + (lane >> 4) (64-byte row
        // segments in, conflict-free stores: odd SP)
        const int t = lane & 15, hf = lane >> 4;
        const bool ina = t < na, inb = t < nb;
        for (int e0 = 2 * SU * (c.tid() >> 5); e0 < CW; e0 += 2 * SU * nw) {
            constexpr int SL = RAW ? SU : SU + 1;   // one more for the last entry's neighbour
            float av[SL], bv[SL];
#pragma unroll
            for (int u = 0; u < SL; ++u) {
                const int i = e0 + 2 * u + hf - 2, o = i * N + s0 + t;
                const bool in = (unsigned)i < (unsigned)N && (u < SU || hf == 0);
                av[u] = in && ina ? img[o] : 0.0f;
                bv[u] = in && inb ? img[last - o] : 0.0f;
            }
#pragma unroll
            for (int u = 0; u < SU; ++u) {
                const int ii = e0 + 2 * u + hf;
                float a1 = 0.0f, b1 = 0.0f;
                if constexpr (!RAW) {   // the other half-warp's entry after this one
                    a1 = __shfl_xor_sync(FULL, hf ? av[u] : av[u + 1], 16);
                    b1 = __shfl_xor_sync(FULL, hf ? bv[u] : bv[u + 1], 16);
                }
                if (ii < CW) store(t * SP + ii, av[u], a1, bv[u], b1);
            }
        }
    }
}

// Ray position idx of an item: rays d and its detector mirror B-1-d.
// Positions map to rays in whole blocks of 8 stride positions, where the
// eight lanes of a quarter warp take rays `stride` apart, spreading their
// 16-byte loads over the bank groups; the last partial block maps to itself.
__device__ __forceinline__ int quad_ray(int idx, int cs, int npair)
{
    const int blk = 8 * cs, b = idx / blk, r = idx - b * blk;
    return (b + 1) * blk <= npair ? b * blk + (r & 7) * cs + (r >> 3) : idx;
}

// Walks rays d and dm = B-1-d of item `it` through the staged band pair
// (steps s0 .. s1): the band sums of view v in (x, y) and, for vp >= 0, of
// view vp in (z, w), ray d first (in x and z alone when dm == d).
template <int ROWS, bool RAW>
__device__ __forceinline__ float4 quad_sums(const void *Q, int SP, const QuadItem &it, bool rows, int d, int N, int B,
                                            int s0, int s1, float h, float hq, unsigned top)
{
    const float a = it.a, m = it.m, inv_m = it.inv_m;
    const int dm = B - 1 - d;
    float ov[2] = {0.0f, 0.0f}, op[2] = {0.0f, 0.0f};   // view v / vp: [0] ray d, [1] ray dm
#pragma unroll
    for (int which = 0; which < 2; ++which) {
        if (which == 1 && dm == d) break;
        const int dd = which == 0 ? d : dm;
        const float q = joseph_q(joseph_dp(dd, B), a, hq);
        int lo, hi;
        step_range(q, m, inv_m, h, -2.5f, (float)N + 0.5f, s0, s1, lo, hi);
        const float4 r = it.vp >= 0 ? quad_walk<true, ROWS, RAW>(Q, SP, q, m, lo, hi, s0, h, top)
                                    : quad_walk<false, ROWS, RAW>(Q, SP, q, m, lo, hi, s0, h, top);
        ov[which] += r.x;
        ov[1 - which] += r.y;
        if (rows) {
            op[which] += r.z;
            op[1 - which] += r.w;
        } else {
            op[1 - which] += r.z;
            op[which] += r.w;
        }
    }
    if (dm == d) {
        ov[0] = ov[0] + ov[1];
        op[0] = op[0] + op[1];
    }
    return make_float4(ov[0], ov[1], op[0], op[1]);
}

// quad_sums of position idx, stored into the partial slot out (V x B).
template <int ROWS, bool RAW>
__device__ __forceinline__ void quad_position(const void *Q, int SP, const QuadItem &it, bool rows, int idx, int npair,
                                              int N, int B, int s0, int s1, float h, float hq, unsigned top,
                                              float *out)
{
    const int d = quad_ray(idx, it.stride, npair), dm = B - 1 - d;
    const float4 r = quad_sums<ROWS, RAW>(Q, SP, it, rows, d, N, B, s0, s1, h, hq, top);
    float *o = out + (size_t)it.v * B;
    o[d] = r.x;
    if (dm != d) o[dm] = r.y;
    if (it.vp >= 0) {
        float *o2 = out + (size_t)it.vp * B;
        o2[d] = r.z;
        if (dm != d) o2[dm] = r.w;
    }
}

// Body of block (bx, by, bz) of a grid of nbp band pairs: smraw holds
// quad_smem(N) bytes, the block's c.nth() = tpi pg threads.  The block
// stages its band pair once and then walks gpb groups of pg view-pair
// items of one class (rows or columns) one after the other, so that the
// staging is spread over gpb groups.
template <int ROWS, class Ctx>
__device__ __forceinline__ void quad_body(const Ctx &c, int bx, int by, int bz, int nbp, unsigned char *smraw,
                                          const float *x, const QuadItem *row_items, int n_row,
                                          const QuadItem *col_items, int n_col, int N, int V, int B, int pg, int gpb, int tpi,
                                          float *partial)
{
    const int SP = (N + 3) | 1;
    void *Q = smraw;   // [step][pair]: band A pair, band B pair

    const int bp = bx;
    const int row_groups = (n_row + pg - 1) / pg, col_groups = (n_col + pg - 1) / pg;
    const int row_blocks = (row_groups + gpb - 1) / gpb;
    const bool rows = by < row_blocks;
    const int grp0 = (rows ? by : by - row_blocks) * gpb;
    const int ngrp = min(gpb, (rows ? row_groups : col_groups) - grp0);
    const QuadItem *list = rows ? row_items : col_items;
    const int nl = rows ? n_row : n_col;
    float *out = partial + ((size_t)bz * nbp + bp) * V * B;
    const int s0 = bp * MR, s1 = min(s0 + MR, (N + 1) / 2) - 1;
    const float h = joseph_h(N), hq = joseph_hq(N);
    const int tid = c.tid();

    // the first item's constants arrive while the band pair is staged
    const int vi = tid / tpi;
    QuadItem it = list[min(grp0 * pg + vi, nl - 1)];
    quad_stage<false>(c, Q, x + (size_t)bz * N * N, N, s0, rows);
    c.sync();
    const int npair = (B + 1) / 2;
    const unsigned top = (unsigned)(N + 2);
    for (int gi = 0; gi < ngrp; ++gi) {
        const int grp = grp0 + gi;
        if (vi >= min(pg, nl - grp * pg)) break;
        if (gi > 0) it = list[grp * pg + vi];
        for (int idx = tid - vi * tpi; idx < npair; idx += tpi)
            quad_position<ROWS, false>(Q, SP, it, rows, idx, npair, N, B, s0, s1, h, hq, top,
                                       out);
    }
}

// Work-balanced form of the same projection.  The work of a batch is cut
// into units (slice, class, band pair, item, chunk of 32 or 64 ray
// positions), ordered so that the units of one staged band pair (a segment)
// are consecutive; each block takes the range [u0, u1) of units, stages
// each segment the range touches once, and its warps take the segment's
// units one at a time from a shared counter.  Blocks thus carry equal work
// whatever the number of items, and a block holds as many warps as its
// registers allow.  The sums are those of quad_body, unit for unit.
struct QuadUnits {
    int upl;        // ray positions of a unit per lane (1 or 2)
    int nch;        // chunks of 32 upl positions per item
    int u_rows;     // units of one row-class segment: n_row items x nch
    int u_cols;     // units of one column-class segment
    long long u_z;  // units per slice: band pairs x (u_rows + u_cols)
};
__host__ __device__ __forceinline__ QuadUnits quad_units(int N, int B, int n_row, int n_col, int upl)
{
    QuadUnits U;
    U.upl = upl;
    U.nch = ((B + 1) / 2 + 32 * upl - 1) / (32 * upl);
    U.u_rows = n_row * U.nch;
    U.u_cols = n_col * U.nch;
    U.u_z = (long long)quad_bands(N) * (U.u_rows + U.u_cols);
    return U;
}

template <int ROWS, bool RAW, class Ctx>
__device__ __forceinline__ void quad_balanced_body(const Ctx &c, long long u0, long long u1, const QuadUnits &U,
                                                   unsigned char *smraw, int *next, const float *x,
                                                   const QuadItem *row_items, const QuadItem *col_items, int N,
                                                   int V, int B, float *partial)
{
    const int SP = RAW ? (N + 4) | 1 : (N + 3) | 1, nbp = quad_bands(N);
    const float h = joseph_h(N), hq = joseph_hq(N);
    const int npair = (B + 1) / 2;
    const unsigned top = (unsigned)(N + 2);
    const int tid = c.tid(), lane = tid & 31;
    const long long rows_all = (long long)nbp * U.u_rows;
    long long u = u0;
    while (u < u1) {
        // the segment of unit u: slice z, class, band pair bp
        const long long z = u < U.u_z ? 0 : u / U.u_z, r = u - z * U.u_z;
        const bool rows = r < rows_all;
        const long long r2 = rows ? r : r - rows_all;
        const int per = rows ? U.u_rows : U.u_cols;
        const int bp = r2 < 0x7fffffffLL ? (int)((unsigned)r2 / (unsigned)per) : (int)(r2 / per);
        const long long seg0 = u - (r2 - (long long)bp * per);
        const long long e = min(u1, seg0 + per);
        const int s0 = bp * MR, s1 = min(s0 + MR, (N + 1) / 2) - 1;
        const QuadItem *list = rows ? row_items : col_items;
        float *out = partial + ((size_t)z * nbp + bp) * V * B;
        const int n_units = (int)(e - seg0);
        quad_stage<RAW>(c, smraw, x + (size_t)z * N * N, N, s0, rows);
        if (tid == 0) *next = (int)(u - seg0);
        c.sync();
        for (;;) {
            int w = 0;
            if (lane == 0) w = atomicAdd(next, 1);
            w = __shfl_sync(0xffffffffu, w, 0);
            if (w >= n_units) break;
            const int item = (int)((unsigned)w / (unsigned)U.nch), chunk = w - item * U.nch;
            const QuadItem it = list[item];
#pragma unroll 1
            for (int k = 0; k < U.upl; ++k) {
                const int idx = (chunk * U.upl + k) * 32 + lane;
                if (idx < npair)
                    quad_position<ROWS, RAW>(smraw, SP, it, rows, idx, npair, N, B, s0, s1, h,
                                             hq, top, out);
            }
        }
        c.sync();
        u = e;
    }
}

// =====================================================================
// Backprojection by rotation orbits (default angles, V and N even).
// View v + V/2 is view v turned by 90 degrees and the detector mirror
// d -> B-1-d is the turn by 180 degrees, so for a pixel P the detector
// coordinate e of (P, view v) is also that of (R90 P, view v + V/2), and the
// mirrored coordinate B-1-e is that of (R180 P, v) and (R270 P, v + V/2).
// One weight evaluation (floor, fraction, two hat weights) therefore
// serves four pixel-views; a block takes a 16 x 16 tile of one image
// quadrant and evaluates, per base view v < V/2, the weights of P and of
// R90 P, which cover all eight (pixel, view) pairs of the orbit
// {P, R90 P, R180 P, R270 P} x {v, v + V/2}.  Each of the block's
// 16 ORB_TY threads takes the orbits of ORB_PX pixels of one tile column
// (rows r, r + ORB_TY, ..), so the per-view constants, window bases and
// loop control are shared by 8 ORB_PX pixel-views.  Base views are split into
// nsl slices (grid.z; by rule or tuned, at most ORB_SL_MAX), added in slice
// order: in a thread-block cluster of the slices' blocks
// (k_backproject_orbit_cl), or from slice images (the persistent batched
// kernel's reduction phase).  The weights are the
// pixel-side Joseph weights of k_backproject_tiles, so both kernels compute
// the same A^T.
// =====================================================================
constexpr int ORB_T = 16;        // quadrant tile side
constexpr int ORB_TY = 8;        // thread rows of a block: tile rows r, r + ORB_TY, ... each
constexpr int ORB_TH = ORB_T * ORB_TY;
constexpr int ORB_PX = ORB_T / ORB_TY;   // pixel orbits per thread
constexpr int ORB_SL = 4;        // base-view slices where no rule applies
constexpr int ORB_SL_MAX = 8;
constexpr int ORB_VC = 8;        // base views staged per chunk
constexpr int ORB_RW = 36;       // values per window: pairs (k, k+1), k <= ORB_RW - 2
constexpr int ORB_MAXS = 1024;   // base views per slice (V <= 8192)

__device__ __forceinline__ void cp_async16(float *dst, const float *src, bool valid)
{
    const unsigned sdst = (unsigned)__cvta_generic_to_shared(dst);
    const int n = valid ? 16 : 0;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(sdst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async4(float *dst, const float *src, bool valid)
{
    const unsigned sdst = (unsigned)__cvta_generic_to_shared(dst);
    const int n = valid ? 4 : 0;
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(sdst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int K>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(K) : "memory"); }

// Body of block (bx, by, bz) (c.nth() = ORB_TH threads, as ORB_T x ORB_TY);
// osm holds orbit_smem() bytes.  FORM ORB_PAIR: y holds per image V/2 pairs
// of rows, views v and v + V/2 interleaved, ld values each, ld a multiple of
// 4, zeros past the B-th, 16-byte aligned: so every window, whose start is a
// multiple of 4, is copied in aligned 16-byte pieces, each wholly on or
// wholly off the padded row, and one 8-byte load serves both views (their
// windows, places and weights are the same).  A load per view took 5 us more
// a launch at 512^2 / 720 views / 736 bins (a 30-iteration solve's 42: 6669
// -> 6453 us).  ORB_PAIR4: also B % 4 == 0, which makes the mirrored windows'
// place a constant (one addition a view less, 2 %).  ORB_PLAIN: y holds rows
// of B values, ld = B apart, copied value by value (25 us more there: for
// small sinograms).  ORB_PLAIN4: such rows with B % 4 == 0, copied in 16-byte
// pieces, two 4-byte loads for a pair's two views (for all but large
// sinograms: no pass before it).  ct_backproject, which interleaves a large
// input first, takes 65.6 us a call at 512^2 / 720 (62.5 in a replayed graph,
// the pass included) and 225 at 1024^2, 67.7 and 238 from the plain rows.
// CL: instead of storing its sums, the block leaves them in osm, entry (k ORB_PX + j) ORB_TH + tid for rotation
// k of the thread's pixel orbit j, for a cluster reduction over slices.
// SEQ (nsl a power of two): bz counts the csz blocks of a tile, a divisor of
// nsl, instead of the slices; each takes nsl / csz slices one after the other.
// CL: the sums of those before its last are kept one by one in
// orbit_kept(osm), the last one's are left as above.  Otherwise csz is 1: the
// block adds its slices' sums up there and writes the result.
enum { ORB_PLAIN = 0, ORB_PLAIN4, ORB_PAIR, ORB_PAIR4 };
constexpr int ORB_E = 4 * ORB_PX * ORB_TH;   // sums of a tile
__device__ __forceinline__ float *orbit_kept(unsigned char *osm)
{
    return reinterpret_cast<float *>(osm) + 2 * ORB_VC * 8 * ORB_RW + 4 * 4 * ORB_VC;
}
// Sets of sums a block keeps: one of csz that share nsl slices.
__host__ __device__ __forceinline__ int orbit_kept_sets(int nsl, int csz) { return csz == 1 ? 1 : nsl / csz - 1; }
template <int FORM, class Ctx, bool CL = false, bool SEQ = false>
__device__ __forceinline__ void orbit_body(const Ctx &cb, int bx, int by, int bz, unsigned char *osm, const float *y,
                                           int ld, float *partial, const float4 *trig, int N, int V, int B, int nsl,
                                           int fin, float *out, const float *xin, const double *scal, int csz = 1)
{
    // raw[buffer][view][window (e, mirror e, e90, mirror e90)][value][row (v, v+V/2)]; ORB_PLAIN4: [row][window][value]
    float *raw = reinterpret_cast<float *>(osm);                               // 2 x ORB_VC x 8 x ORB_RW
    float4 *tt = reinterpret_cast<float4 *>(raw + 2 * ORB_VC * 8 * ORB_RW);    // 2 x ORB_VC x 2
    float *kept = orbit_kept(osm);                                             // SEQ: orbit_kept_sets x ORB_E
    int *wbs = reinterpret_cast<int *>(kept + (SEQ ? orbit_kept_sets(nsl, csz) * ORB_E : 0));   // base views x 2
    const int tid = cb.tid();   // tid / ORB_T < ORB_TY
    const int tx = tid % ORB_T, ty = tid / ORB_T;
    const int half = N / 2, V2 = V / 2;
    const int share = SEQ ? nsl / csz : 1, slice = SEQ ? bz % csz * share : bz % nsl, img = bz / (SEQ ? csz : nsl);
    const int slice1 = slice + share;   // the block's slices: slice .. slice1 - 1
    auto first_view = [&](int s) { return SEQ ? V2 * s >> (31 - __clz(nsl)) : (int)((long long)V2 * s / nsl); };
    const int r0 = by * ORB_T, c0 = half + bx * ORB_T;   // quadrant r < N/2, c >= N/2
    const int r = r0 + ty, c = c0 + tx;                  // pixels (r + j ORB_TY, c)
    const bool inside = r < half && c < N;
    const float h = 0.5f * (float)(N - 1), hb = 0.5f * (float)(B - 1), hb_lo = hb - 0.5f;
    const float xq = (float)c - h, yq = (float)r - h;               // P = (x, y); R90 P = (-y, x)
    const float *ys = y + (size_t)img * V * ld;
    const int ms = FORM == ORB_PAIR4 || FORM == ORB_PLAIN4 ? 3 : (B - ORB_RW + 3) & 3;   // see the mirrored windows below
    const int vb0 = first_view(slice), vb1 = first_view(slice1);
    const int nvs = vb1 - vb0;
    static_assert(ORB_PX == 2, "a thread's two orbits are packed");
    const float2 xq2 = pk(xq, xq), yq2 = pk(yq, yq + (float)ORB_TY), nyq2 = pk(-yq, -(yq + (float)ORB_TY));
    const float2 hb2 = pk(hb_lo, hb_lo), bias2 = pk(JOSEPH_BIAS, JOSEPH_BIAS);
    float acc[ORB_PX][4];   // per pixel orbit: P, R90 P, R180 P, R270 P
#pragma unroll
    for (int j = 0; j < ORB_PX; ++j) acc[j][0] = acc[j][1] = acc[j][2] = acc[j][3] = 0.0f;

    // window bases (multiples of 4) of the tile for every base view of this
    // slice: floor(e) - wb lies in [1, 29] for every pixel of the tile, as
    // e spans at most 15 (|cos| + |sin|) < 21.3 over it
    for (int vi = tid; vi < nvs; vi += ORB_TH) {
        const float4 T = trig[vb0 + vi];
        float emin = 3.0e38f, e9min = 3.0e38f;
#pragma unroll
        for (int cr = 0; cr < 4; ++cr) {
            const float xx = (float)(c0 + (cr & 1) * (ORB_T - 1)) - h;
            const float yy = (float)(r0 + (cr >> 1) * (ORB_T - 1)) - h;
            emin = fminf(emin, xx * T.x + yy * T.y);
            e9min = fminf(e9min, -yy * T.x + xx * T.y);
        }
        emin = fminf(fmaxf(emin + hb, -1.0e6f), 1.0e6f);
        e9min = fminf(fmaxf(e9min + hb, -1.0e6f), 1.0e6f);
        wbs[2 * vi] = ((int)floorf(emin) - 2) & ~3;
        wbs[2 * vi + 1] = ((int)floorf(e9min) - 2) & ~3;
    }
    cb.sync();

    // raw window values y[start + w], w < ORB_RW, start = wb (windows e, e90) or, for their mirrors, the multiple of
    // 4 at or below B - ORB_RW + 3 - wb, so that pair B-2-f sits at ORB_RW-5 + ms - (f - wb), ms = 0 .. 3;
    // per view (cos, sin, |a|^2, |a| (1 - |a|/2)), each twice: the hat weights times |a|
    auto issue = [&](int v0, int nv, int buf) {
        float *dst0 = raw + (size_t)buf * ORB_VC * 8 * ORB_RW;
        if (tid < nv) {
            const float4 T = trig[v0 + tid];
            tt[2 * (buf * ORB_VC + tid)] = make_float4(T.x, T.x, T.y, T.y);
            tt[2 * (buf * ORB_VC + tid) + 1] = make_float4(T.z * T.z, T.z * T.z, T.z * T.w, T.z * T.w);
        }
        if (FORM == ORB_PLAIN4) {
            constexpr int CH = ORB_RW / 4;   // copies per window
            for (int k = tid; k < nv * 8 * CH; k += ORB_TH) {
                const int q = k / CH, j = k - q * CH;
                const int win = q & 3, row = (q >> 2) & 1, vi = q >> 3;
                const int base = wbs[2 * (v0 - vb0 + vi) + (win >> 1)];
                const int d = ((win & 1) ? B - ORB_RW - base : base) + 4 * j;
                const bool ok = d >= 0 && d < B;
                cp_async16(dst0 + (size_t)q * ORB_RW + 4 * j, ys + (size_t)(v0 + vi + row * V2) * ld + (ok ? d : 0), ok);
            }
        } else if (FORM != ORB_PLAIN) {
            constexpr int CH = ORB_RW / 2;   // copies per window
            for (int k = tid; k < nv * 4 * CH; k += ORB_TH) {
                const int q = k / CH, j = k - q * CH;
                const int win = q & 3, vi = q >> 2;
                const int base = wbs[2 * (v0 - vb0 + vi) + (win >> 1)];
                const int d = ((win & 1) ? B - ORB_RW + 3 - ms - base : base) + 2 * j;
                const bool ok = d >= 0 && d < B;
                cp_async16(dst0 + 2 * (size_t)q * ORB_RW + 4 * j, ys + 2 * ((size_t)(v0 + vi) * ld + (ok ? d : 0)), ok);
            }
        } else {
            for (int k = tid; k < nv * 8 * ORB_RW; k += ORB_TH) {
                const int q = k / ORB_RW, j = k - q * ORB_RW;
                const int win = q & 3, row = (q >> 2) & 1, vi = q >> 3;
                const int base = wbs[2 * (v0 - vb0 + vi) + (win >> 1)];
                const int d = ((win & 1) ? B - ORB_RW + 3 - ms - base : base) + j;
                const bool ok = d >= 0 && d < B;
                cp_async4(dst0 + 2 * ((size_t)(vi * 4 + win) * ORB_RW + j) + row,
                          ys + (size_t)(v0 + vi + row * V2) * ld + (ok ? d : 0), ok);
            }
        }
        cp_async_commit();
    };
    // SEQ: the sums of a slice that ends before view v are kept, and the next slice's start at zero
    int cur = slice, bnd = 0x7fffffff;
    auto bound = [&]() { bnd = cur + 1 < slice1 ? first_view(cur + 1) : 0x7fffffff; };
    auto keep = [&](int v) {
        while (v >= bnd) {
            float *dst = kept + (CL ? (cur - slice) * ORB_E : 0) + tid;
#pragma unroll
            for (int j = 0; j < ORB_PX; ++j)
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    float *q = dst + (k * ORB_PX + j) * ORB_TH;
                    *q = !CL && cur > 0 ? *q + acc[j][k] : acc[j][k];
                    acc[j][k] = 0.0f;
                }
            ++cur;
            bound();
        }
    };
    if constexpr (SEQ) bound();
    const int nch = (nvs + ORB_VC - 1) / ORB_VC;
    if (nch > 0) issue(vb0, min(ORB_VC, nvs), 0);
    for (int ch = 0; ch < nch; ++ch) {
        const int v0 = vb0 + ch * ORB_VC, nv = min(ORB_VC, vb1 - v0);
        if (ch + 1 < nch) {
            issue(v0 + ORB_VC, min(ORB_VC, vb1 - v0 - ORB_VC), (ch + 1) & 1);
            cp_async_wait<1>();
        } else {
            cp_async_wait<0>();
        }
        cb.sync();
        const float *tb = raw + (size_t)(ch & 1) * ORB_VC * 8 * ORB_RW;
        const float4 *tv = tt + 2 * (ch & 1) * ORB_VC;
        auto view = [&](int vi) {
            const float4 Ta = tv[2 * vi], Tb = tv[2 * vi + 1];
            const float2 Tx = pk(Ta.x, Ta.y), Ty = pk(Ta.z, Ta.w), Tz = pk(Tb.x, Tb.y), Tw = pk(Tb.z, Tb.w);
            const int2 wb = *reinterpret_cast<const int2 *>(wbs + 2 * (v0 - vb0 + vi));
            // value i of window w: (view v, view v + V/2)
            const float *win = tb + (size_t)vi * 8 * ORB_RW;
            auto at = [&](int w, unsigned i) {
                if constexpr (FORM == ORB_PLAIN4) return pk(win[w * ORB_RW + i], win[(4 + w) * ORB_RW + i]);
                else return reinterpret_cast<const float2 *>(win)[w * ORB_RW + i];
            };
            // e - 1/2 of P and of R90 P for the thread's two orbits, (x, y) = (xq, yq) and (xq, yq + ORB_TY),
            // their windows' places and weights: packed (14 issue slots a view for 28; ct_backproject 63.8 -> 62.7 us
            // in a replayed graph at 512^2 / 720 views, each value rounded as before)
            const float2 e = pfma(xq2, Tx, pfma(yq2, Ty, hb2)), e9 = pfma(xq2, Ty, pfma(nyq2, Tx, hb2));
            const float2 t = padd(e, bias2), t9 = padd(e9, bias2);
            const float2 u = psub(t, bias2), u9 = psub(t9, bias2);
            const float2 g = psub(e, u), g9 = psub(e9, u9), ng = psub(u, e), ng9 = psub(u9, e9);
            const float2 a0 = pfma(ng, Tz, Tw), a1 = pfma(g, Tz, Tw), a09 = pfma(ng9, Tz, Tw), a19 = pfma(g9, Tz, Tw);
            auto orbit = [&](int j, float &cP, float &c90, float &c180, float &c270) {
                const unsigned k = min((unsigned)(__float_as_int((j ? t.y : t.x)) - (JOSEPH_BIAS_BITS + wb.x)),
                                       (unsigned)(ORB_RW - 5));
                const unsigned k9 = min((unsigned)(__float_as_int((j ? t9.y : t9.x)) - (JOSEPH_BIAS_BITS + wb.y)),
                                        (unsigned)(ORB_RW - 5));
                const float w0 = fmaxf(0.0f, (j ? a0.y : a0.x)), w1 = fmaxf(0.0f, (j ? a1.y : a1.x));
                const float w09 = fmaxf(0.0f, (j ? a09.y : a09.x)), w19 = fmaxf(0.0f, (j ? a19.y : a19.x));
                const unsigned km = ORB_RW - 5 + ms - k, km9 = ORB_RW - 5 + ms - k9;
                const float2 e0 = at(0, k), e1 = at(0, k + 1), m0 = at(1, km), m1 = at(1, km + 1);
                const float2 f0 = at(2, k9), f1 = at(2, k9 + 1), n0 = at(3, km9), n1 = at(3, km9 + 1);
                cP = fmaf(w0, e0.x, fmaf(w1, e1.x, cP));           // P at v
                c180 = fmaf(w1, m0.x, fmaf(w0, m1.x, c180));       // R180 P at v
                c90 = fmaf(w0, e0.y, fmaf(w1, e1.y, c90));         // R90 P at v + V/2
                c270 = fmaf(w1, m0.y, fmaf(w0, m1.y, c270));       // R270 P at v + V/2
                c90 = fmaf(w09, f0.x, fmaf(w19, f1.x, c90));       // R90 P at v
                c270 = fmaf(w19, n0.x, fmaf(w09, n1.x, c270));     // R270 P at v
                c180 = fmaf(w09, f0.y, fmaf(w19, f1.y, c180));     // R180 P at v + V/2
                cP = fmaf(w19, n0.y, fmaf(w09, n1.y, cP));         // P at v + V/2
            };
#pragma unroll
            for (int j = 0; j < ORB_PX; ++j)
                orbit(j, acc[j][0], acc[j][1], acc[j][2], acc[j][3]);   // (a row past the quadrant is not stored)
        };
        if (inside) {
            if constexpr (SEQ) {
                for (int vi = 0; vi < nv;) {
                    keep(v0 + vi);
                    for (const int ve = min(nv, bnd - v0); vi < ve; ++vi) view(vi);
                }
            } else {
                for (int vi = 0; vi < nv; ++vi) view(vi);
            }
        }
        cb.sync();   // the buffer is refilled two chunks later
    }
    if constexpr (SEQ) {
        keep(vb1);
        if constexpr (!CL) {   // the only block of the tile: the sums are complete
            if (cur > 0)
#pragma unroll
                for (int j = 0; j < ORB_PX; ++j)
#pragma unroll
                    for (int k = 0; k < 4; ++k) acc[j][k] = kept[(k * ORB_PX + j) * ORB_TH + tid] + acc[j][k];
        }
    }
    if constexpr (CL) {
        float *red = reinterpret_cast<float *>(osm);   // the staging buffers are free again
#pragma unroll
        for (int j = 0; j < ORB_PX; ++j)
#pragma unroll
            for (int k = 0; k < 4; ++k) red[(k * ORB_PX + j) * ORB_TH + tid] = acc[j][k];
        return;
    }
    // fin 0: the slice's partial image; with a single slice the sums are
    // complete and the block writes the result itself: fin 1 out = sum,
    // fin 2 out = xin - tau sum
    float *pp = (fin ? out : partial) + ((size_t)img * (fin ? 1 : nsl) + (fin ? 0 : slice)) * N * N;
    const float *xq0 = fin == 2 ? xin + (size_t)img * N * N : nullptr;
    const float tau = fin == 2 ? fscal(scal, F_TAU) : 0.0f;
#pragma unroll
    for (int j = 0; j < ORB_PX; ++j) {
        const int rj = r + j * ORB_TY;
        if (rj < half && c < N) {
            const size_t o[4] = {(size_t)rj * N + c,                    // P
                                 (size_t)c * N + (N - 1 - rj),          // R90 (r, c) = (c, N-1-r)
                                 (size_t)(N - 1 - rj) * N + (N - 1 - c), // R180 (r, c) = (N-1-r, N-1-c)
                                 (size_t)(N - 1 - c) * N + rj};         // R270 (r, c) = (N-1-c, r)
#pragma unroll
            for (int k = 0; k < 4; ++k) pp[o[k]] = fin == 2 ? __fmaf_rn(-tau, acc[j][k], xq0[o[k]]) : acc[j][k];
        }
    }
}

}  // namespace ctpd
