// body_tv.cuh -- body of the temporally blocked, register-resident TV prox
// (Eq. 17) shared by its kernel (k_tv.cu) and the persistent batched kernel
// (persist.cu).
#pragma once

#include "ctpd_internal.cuh"

namespace ctpd {

constexpr int TV_WARPS = 16;
constexpr int TV_THREADS = TV_WARPS * 32;
constexpr int TV_J = 5;                     // most region rows per warp
constexpr int TV_ROWS = TV_WARPS * TV_J;    // 80
constexpr int TV_MAX_STEPS = 16;            // H = 17: 30 interior columns
constexpr int TV_MIN_TR = 16;               // fewest interior rows per tile

// Shared memory of one tile: what a warp's rows publish for the rows above
// and below them, in two buffers used in turn (so one barrier a step).
struct TvPub {
    float4 first[2][TV_WARPS + 1][32];   // (r_x, r_y) of warp w's first row; the last entry: zeros
    float2 last[2][TV_WARPS + 1][32];    // r_y of warp w - 1's last row; entry 0: zeros
};

// Halo: steps + 1; the trajectory variant rounds it up to even, so that tile
// origins (and every lane's column pair) fall on even columns: with N even
// each pair of its many stores is one aligned 8-byte store.
__host__ __device__ __forceinline__ int tv_halo(int steps, bool even) { return even ? (steps + 2) & ~1 : steps + 1; }

// bz selects the image of a batch (z, x: N x N each; p: 2 N x N).
// traj, when not NULL, receives p after each of the first steps - 1 steps:
// step l + 1 (l = 0 .. steps - 2) at traj + (l * gz + image) * 2 N N.
//
// FGP: the fast gradient projection (Beck and Teboulle): each step is the
// projected-gradient step taken at r = p + theta (p - p_prev) instead of p,
// with theta_k = (t_k - 1) / t_{k+1}, t_1 = 1, t_{k+1} = (1 + sqrt(1 + 4 t_k^2)) / 2
// (momentum restarted at every call).  Each cell keeps p_prev as well, and
// the field published for the divergence is r_y (p_y after the last step).
// Body of tile (bx, by) of image bz of a batch of gz images, on the
// TV_THREADS threads of context cb.  Warp w holds the J consecutive region
// rows w J .. w J + J - 1, so that a row's vertical neighbours are in the
// same thread's registers except at the J-row runs' ends.  There a step
// needs r_y of the row above and x of the row below; the latter is computed
// again from that row's published r and its z, so a step has one barrier and
// four shared-memory accesses.  A column pair's arithmetic is packed
// (f32x2).  Bound: one 16-warp block an SM, its chain of steps (issue 47 %,
// FP pipe and barrier waits); 512^2, 10 steps: 13.6 us with rows dealt out
// in turn (two barriers, 4 J accesses a step, 5.9 M instructions), 11.1 to
// 12.1 us now (4.2 M), cold cache.
template <bool FGP, bool TRAJ, int J, class Ctx>
__device__ __forceinline__ void tv_body(const Ctx &cb, int bx, int by, int bz, int gz, TvPub &pub,
                                        const float *z, const float *p_in, float *p_out, float *x, int N,
                                        int steps, int final_, int tc, int tr, const double *scal, float *traj)
{
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = cb.tid() & 31, w = cb.tid() >> 5;
    const int H = tv_halo(steps, TRAJ), Sr = tr + 2 * H;
    const bool vec2 = TRAJ && (N & 1) == 0;   // column pairs 8-byte aligned
    const int R0 = by * tr - H, C0 = bx * tc - H;
    const int c0 = C0 + 2 * lane;   // image columns c0, c0 + 1 of this lane
    const int l0 = w * J;           // region row of j = 0
    const size_t NN = (size_t)N * N, img = bz;
    z += img * NN;
    p_in += img * 2 * NN;
    p_out += img * 2 * NN;
    if (final_) x += img * NN;
    const float lam = fscal(scal, F_LAMBDA);
    const float inv8 = fscal(scal, F_INV8LAM);
    const float2 lam2 = pk(lam, lam);
    // forward differences: along x on columns 0..N-2, along y on columns 0..N-1
    const bool cx0 = (unsigned)c0 < (unsigned)(N - 1), cx1 = (unsigned)(c0 + 1) < (unsigned)(N - 1);
    const bool cy0 = (unsigned)c0 < (unsigned)N, cy1 = (unsigned)(c0 + 1) < (unsigned)N;
    // the dual step's factors: 0 on p_x of columns -1 and N-1 and on p_y of
    // rows -1 and N-1, which cuts the image off from the cells around it
    // (those evolve from zeros and are never read by an image cell)
    const float2 mx = pk(c0 == -1 || c0 == N - 1 ? 0.0f : inv8, c0 + 1 == -1 || c0 + 1 == N - 1 ? 0.0f : inv8);
    float my[J];

    // per column pair: z (the run's rows and the row below it), p_x, p_y
    float2 zr[J + 1], pxr[J], pyr[J];
    float2 pxo[FGP ? J : 1], pyo[FGP ? J : 1];   // FGP: p of the previous step
#pragma unroll
    for (int j = 0; j <= J; ++j) {
        const int li = l0 + j, rr = R0 + li;
        const bool rin = li < Sr && (unsigned)rr < (unsigned)N;
        const size_t gi = (size_t)rr * N + c0;   // c0 may be -1..: only valid columns are read
        zr[j] = pk(rin && cy0 ? z[gi] : 0.0f, rin && cy1 ? z[gi + 1] : 0.0f);
        if (j < J) {
            const bool ryd = li < Sr && (unsigned)rr < (unsigned)(N - 1);
            pxr[j] = pk(rin && cx0 ? p_in[gi] : 0.0f, rin && cx1 ? p_in[gi + 1] : 0.0f);
            pyr[j] = pk(ryd && cy0 ? p_in[NN + gi] : 0.0f, ryd && cy1 ? p_in[NN + gi + 1] : 0.0f);
            my[j] = rr == -1 || rr == N - 1 ? 0.0f : inv8;
            if constexpr (FGP) {
                pxo[j] = pxr[j];
                pyo[j] = pyr[j];
            }
        }
    }
    if (w < 2) {   // the entries beyond the region
        pub.first[w][TV_WARPS][lane] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        pub.last[w][0][lane] = make_float2(0.0f, 0.0f);
    }
    pub.first[0][w][lane] = make_float4(pxr[0].x, pxr[0].y, pyr[0].x, pyr[0].y);
    pub.last[0][w + 1][lane] = pyr[J - 1];
    cb.sync();
    const bool busy = l0 < Sr;   // otherwise the warp holds no region row (its p stays zero)
    int ph = 0;

    if (lam > 0.0f) {
        float t = 1.0f, th = 0.0f;   // FGP: t_k and theta_{k-1} (theta_0 = 0)
        for (int it = 0; it < steps; ++it) {
            // FGP: theta_k for the next extrapolation
            const float t1 = FGP ? 0.5f * (1.0f + sqrtf(fmaf(4.0f * t, t, 1.0f))) : 1.0f;
            const float thn = FGP ? (t - 1.0f) / t1 : 0.0f;
            const bool last = it + 1 == steps;
            if (busy) {
                const float2 up = pub.last[ph][w][lane];
                const float4 dn = pub.first[ph][w + 1][lane];
                // r = p (GP) or p + theta (p - p_prev) (FGP)
                auto ext = [](float f, float2 p, float2 o) { return pfma(pk(f, f), psub(p, o), p); };
                auto rx = [&](int j) { return FGP ? ext(th, pxr[j], pxo[FGP ? j : 0]) : pxr[j]; };
                auto ry = [&](int j) { return FGP ? ext(th, pyr[j], pyo[FGP ? j : 0]) : pyr[j]; };
                // x = max(0, z + lam div r), the run and the row below it
                float2 xr[J + 1];
#pragma unroll
                for (int j = 0; j <= J; ++j) {
                    const float2 rxj = j < J ? rx(j < J ? j : 0) : pk(dn.x, dn.y);
                    const float2 ryj = j < J ? ry(j < J ? j : 0) : pk(dn.z, dn.w);
                    const float2 ryu = j > 0 ? ry(j > 0 ? j - 1 : 0) : up;
                    float pl = __shfl_up_sync(FULL, rxj.y, 1);
                    if (lane == 0) pl = 0.0f;
                    const float2 v = pfma(lam2, padd(pk(rxj.x - pl, rxj.y - rxj.x), psub(ryj, ryu)), zr[j]);
                    xr[j] = pk(fmaxf(0.0f, v.x), fmaxf(0.0f, v.y));
                }
                // p = Pi(p + grad x / (8 lam)), Pi(q) = q / max(1, |q|)
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    const float xrt = __shfl_down_sync(FULL, xr[j].x, 1);
                    const float2 qx = pfma(pk(xr[j].y - xr[j].x, xrt - xr[j].y), mx, rx(j));
                    const float2 qy = pfma(psub(xr[j + 1], xr[j]), pk(my[j], my[j]), ry(j));
                    const float2 n2 = pfma(qx, qx, pmul(qy, qy));
                    const float2 sc = pk(fminf(1.0f, rsqrt_ftz(n2.x)), fminf(1.0f, rsqrt_ftz(n2.y)));
                    if constexpr (FGP) {
                        pxo[j] = pxr[j];
                        pyo[j] = pyr[j];
                    }
                    pxr[j] = pmul(qx, sc);
                    pyr[j] = pmul(qy, sc);
                }
                // r of the next step (p after the last one)
                auto nx = [&](float2 p, float2 o) { return FGP && !last ? ext(thn, p, o) : p; };
                const float2 fx = nx(pxr[0], pxo[0]), fy = nx(pyr[0], pyo[0]);
                pub.first[ph ^ 1][w][lane] = make_float4(fx.x, fx.y, fy.x, fy.y);
                pub.last[ph ^ 1][w + 1][lane] = nx(pyr[J - 1], pyo[FGP ? J - 1 : 0]);
            } else if (it < 2) {   // its neighbour reads zeros
                pub.first[ph ^ 1][w][lane] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            }
            if (TRAJ && !last) {   // the tile interior's p after this step
                float *tp = traj + ((size_t)it * gz + img) * 2 * NN;
#pragma unroll
                for (int j = 0; j < J; ++j) {
                    const int li = l0 + j, rr = R0 + li, lj = 2 * lane;
                    if (li >= H && li < H + tr && rr < N) {
                        const size_t gi = (size_t)rr * N + c0;
                        const bool in0 = lj >= H && lj < H + tc && c0 < N;
                        const bool in1 = lj + 1 >= H && lj + 1 < H + tc && c0 + 1 < N;
                        if (vec2) {   // H, tc even: both columns of the pair are interior, or neither
                            if (in0) {
                                *reinterpret_cast<float2 *>(tp + gi) = pxr[j];
                                *reinterpret_cast<float2 *>(tp + NN + gi) = pyr[j];
                            }
                        } else {
                            if (in0) {
                                tp[gi] = pxr[j].x;
                                tp[NN + gi] = pyr[j].x;
                            }
                            if (in1) {
                                tp[gi + 1] = pxr[j].y;
                                tp[NN + gi + 1] = pyr[j].y;
                            }
                        }
                    }
                }
            }
            cb.sync();
            ph ^= 1;
            t = t1;
            th = thn;
        }
    }

    // the tile interior: p, and x = max(0, z + lam div p) on the last chunk
    const float2 up = pub.last[ph][w][lane];
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int li = l0 + j, rr = R0 + li;
        if (li >= H && li < H + tr && rr < N) {
            const float2 ryu = j > 0 ? pyr[j > 0 ? j - 1 : 0] : up;
            float pl = __shfl_up_sync(FULL, pxr[j].y, 1);
            if (lane == 0) pl = 0.0f;
            const float2 v = pfma(lam2, padd(pk(pxr[j].x - pl, pxr[j].y - pxr[j].x), psub(pyr[j], ryu)), zr[j]);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int lj = 2 * lane + e, cc = C0 + lj;
                if (lj >= H && lj < H + tc && cc < N) {
                    const size_t gi = (size_t)rr * N + cc;
                    if (lam > 0.0f) {
                        p_out[gi] = e == 0 ? pxr[j].x : pxr[j].y;
                        p_out[NN + gi] = e == 0 ? pyr[j].x : pyr[j].y;
                    }
                    if (final_) x[gi] = fmaxf(0.0f, e == 0 ? v.x : v.y);
                }
            }
        }
    }
}

}  // namespace ctpd
