// body_fft.cuh -- register-resident FFT of the frequency-domain
// preconditioner D (k_fft.cu) and the body of the fused dual step, shared by
// its kernel and the persistent batched kernel (persist.cu).
//
// D applies, along the detector of every view, the linear (zero-padded)
// convolution with the taps t[k], |k| < half.  With the view zero-padded to
// the period P >= 2B, the circular convolution with the taps placed at k
// mod P equals that linear convolution on bins 0..B-1, so D =
// IFFT_P(Hhat . FFT_P(.)) with Hhat the P-point DFT of the circularly placed
// taps.  Two real views travel as one complex sequence.
//
// Layout.  P / 8 threads run one transform; thread t holds the 8 elements
// t + r P/8 in registers, before and after every transform.  A transform is
// a Stockham autosort of radix-8 stages (the last one of radix 8, 4 or 2),
// with one exchange through shared memory between stages.  The ownership at
// both ends is what the layout is chosen for: the multiply by Hhat, the
// inverse's first stage, the dual update and the next filter's first stage
// all run on the registers the previous stage left.  B <= P/2, so the inputs
// r >= 4 are zero and the outputs r >= 4 are not used.
//
// Code size is part of the design: every thread runs through the code once,
// so straight-line copies of the transform are fetched, not reused (with the
// four transforms of a dual step written out, 113 KB of instructions, its
// warps waited for instructions two thirds of the time, 39 us at 512^2 / 720
// views).  One copy of the transform therefore serves both directions (a
// sign, folded into additions as exact FMAs by +-1) and both filters of a
// step, in loops that are not unrolled.
#pragma once

#include "ctpd_internal.cuh"

namespace ctpd {

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// The DFTs take the direction as s: +1 forward (e^{-i..}), -1 inverse.
__device__ __forceinline__ void dft2(float2 &a, float2 &b)
{
    const float2 t = a;
    a = cadd(t, b);
    b = csub(t, b);
}

__device__ __forceinline__ void dft4(float2 &a0, float2 &a1, float2 &a2, float2 &a3, float s)
{
    const float2 t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), d = csub(a1, a3);
    a0 = cadd(t0, t2);
    a2 = csub(t0, t2);
    // t1 +- (-+i) d
    a1 = make_float2(__fmaf_rn(s, d.y, t1.x), __fmaf_rn(-s, d.x, t1.y));
    a3 = make_float2(__fmaf_rn(-s, d.y, t1.x), __fmaf_rn(s, d.x, t1.y));
}

// FUSE: the multiplication by 1/sqrt 2 of w8^3 and the addition after it
// round once (the filters and the dual step); otherwise each rounds (Hhat and
// the adjoint of the dual step).
template <bool FUSE>
__device__ __forceinline__ float mul_add(float a, float b, float c)
{
    return FUSE ? __fmaf_rn(a, b, c) : __fadd_rn(__fmul_rn(a, b), c);
}

template <bool FUSE>
__device__ __forceinline__ void dft8(float2 *v, float s)
{
    // even / odd 4-point DFTs, then the radix-2 combination with w8^k
    float2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    float2 o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4(e0, e1, e2, e3, s);
    dft4(o0, o1, o2, o3, s);
    const float c = 0.70710678118654752440f;
    // w8^1 = c(1 -+ i), w8^2 = -+i, w8^3 = c(-1 -+ i)
    const float2 u1 = make_float2(__fmaf_rn(s, o1.y, o1.x), __fmaf_rn(-s, o1.x, o1.y));
    const float2 u3 = make_float2(__fmaf_rn(s, o3.y, -o3.x), __fmaf_rn(s, o3.x, o3.y));
    v[0] = cadd(e0, o0);
    v[4] = csub(e0, o0);
    v[1] = make_float2(__fmaf_rn(c, u1.x, e1.x), __fmaf_rn(c, u1.y, e1.y));
    v[5] = make_float2(__fmaf_rn(-c, u1.x, e1.x), __fmaf_rn(-c, u1.y, e1.y));
    v[2] = make_float2(__fmaf_rn(s, o2.y, e2.x), __fmaf_rn(-s, o2.x, e2.y));
    v[6] = make_float2(__fmaf_rn(-s, o2.y, e2.x), __fmaf_rn(s, o2.x, e2.y));
    v[3] = make_float2(mul_add<FUSE>(c, u3.x, e3.x), mul_add<FUSE>(-c, u3.y, e3.y));
    v[7] = make_float2(mul_add<FUSE>(-c, u3.x, e3.x), mul_add<FUSE>(c, u3.y, e3.y));
}

// Shared-memory exchange buffers hold element i at fp(i) = i + i/16: the
// first stage's stride-16 stores and every contiguous access are free of
// bank conflicts.
__host__ __device__ __forceinline__ constexpr int fp(int i) { return i + (i >> 4); }
__host__ __device__ __forceinline__ constexpr int fft_elems(int P) { return P + (P >> 4); }
// threads of one transform
__host__ __device__ __forceinline__ constexpr int fft_threads(int P) { return P / 8; }
// radix of the last stage: 8, or what is left of P
__host__ __device__ __forceinline__ constexpr int fft_last_radix(int P) { return P > 8 ? fft_last_radix(P / 8) : P; }
// Twiddle table of a P-point transform (float2, from double precision): for
// every stage after the first, of radix R after stages of total length Ns,
// the entries e^{-2 pi i r k / (Ns R)}, r < R, k < Ns, at fft_tw_off(Ns) + r Ns + k
// (contiguous in k); then the same conjugated for the inverse.
__host__ __device__ __forceinline__ constexpr int fft_tw_off(int Ns) { return Ns <= 8 ? 0 : fft_tw_off(Ns / 8) + Ns; }
__host__ __device__ __forceinline__ constexpr int fft_tw_half(int P)
{
    return fft_tw_off(P / fft_last_radix(P)) + P;
}
__host__ __device__ __forceinline__ constexpr int fft_tw_elems(int P) { return 2 * fft_tw_half(P); }

template <int N>
struct IntC {
    static constexpr int value = N;
};

// Unnormalised P-point DFT of the values v[r] = element t + r P/8, in place
// (inv: e^{+..}, s = -1; else s = +1).  buf holds one exchange buffer of
// fft_elems(P) values (DBL: two, used in turn from number ph, which saves
// the barrier between an exchange's reads and the next one's writes).  A
// stage's twiddles are loaded before the barrier it waits at.  Every thread
// of context c must call it.
template <int P, bool FUSE, bool DBL, class Ctx>
__device__ __forceinline__ void fft_regs(const Ctx &c, int t, float2 (&v)[8], float2 *buf, int &ph,
                                         const float2 *__restrict__ tw, float s)
{
    constexpr int T = P / 8, RL = fft_last_radix(P), NL = P / RL, Q = 8 / RL;
    static_assert(P >= 64 && P <= 8192 && (P & (P - 1)) == 0, "two stages or more, at most 1024 threads");
    auto next = [&]() {
        float2 *b = buf;
        if (DBL) {
            b += ph * fft_elems(P);
            ph ^= 1;
        } else {
            c.sync();   // the previous exchange has been read
        }
        return b;
    };
    dft8<FUSE>(v, s);
    float2 *src = next();
#pragma unroll
    for (int r = 0; r < 8; ++r) src[fp(8 * t + r)] = v[r];
    float2 w[8];
    auto middle = [&](auto ns) {
        constexpr int Ns = decltype(ns)::value;
        if constexpr (8 * Ns <= NL) {
            const int k = t & (Ns - 1);
#pragma unroll
            for (int r = 1; r < 8; ++r) w[r] = __ldg(tw + fft_tw_off(Ns) + r * Ns + k);
            c.sync();
#pragma unroll
            for (int r = 0; r < 8; ++r) v[r] = src[fp(t + r * T)];
#pragma unroll
            for (int r = 1; r < 8; ++r) v[r] = cmul(v[r], w[r]);
            dft8<FUSE>(v, s);
            src = next();
#pragma unroll
            for (int r = 0; r < 8; ++r) src[fp((t - k) * 8 + k + r * Ns)] = v[r];
        }
    };
    middle(IntC<8>{});
    middle(IntC<64>{});
    middle(IntC<512>{});
    // last stage: butterflies t + q T, elements and results at t + (q + r Q) T
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int r = 1; r < RL; ++r) w[q + r * Q] = __ldg(tw + fft_tw_off(NL) + r * NL + t + q * T);
    c.sync();
#pragma unroll
    for (int r = 0; r < 8; ++r) v[r] = src[fp(t + r * T)];
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int r = 1; r < RL; ++r) v[q + r * Q] = cmul(v[q + r * Q], w[q + r * Q]);
    if constexpr (RL == 8) dft8<FUSE>(v, s);
    else if constexpr (RL == 4) {
        dft4(v[0], v[2], v[4], v[6], s);
        dft4(v[1], v[3], v[5], v[7], s);
    } else {
        dft2(v[0], v[4]);
        dft2(v[1], v[5]);
        dft2(v[2], v[6]);
        dft2(v[3], v[7]);
    }
}

// v <- D v (up to the factor P), v's elements r >= 4 zero on entry: forward
// transform, times Hhat (CONJ: its conjugate, D^T), inverse.  On return
// v[r], r < 4, hold the outputs t + r P/8 < P/2.
template <int P, bool CONJ, bool DBL, class Ctx>
__device__ __forceinline__ void fft_apply(const Ctx &c, int t, float2 (&v)[8], float2 *buf, int &ph,
                                          const float2 *hhat, const float2 *__restrict__ tw)
{
    float s = 1.0f;
#pragma unroll 1
    for (int inv = 0; inv < 2; ++inv) {
        fft_regs<P, !CONJ, DBL>(c, t, v, buf, ph, tw + inv * fft_tw_half(P), s);
        s = -1.0f;
        if (inv == 0) {
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                float2 h = hhat[t + r * (P / 8)];
                if (CONJ) h.y = -h.y;
                v[r] = cmul(v[r], h);
            }
        }
    }
}

// Band partial sums of A x for the rays o0 + i and o1 + i (band k at p + k
// VB), added in band order; the loads of 16 bands are issued together.
__device__ __forceinline__ void band_sum2(const float *__restrict__ p0, const float *__restrict__ p1, size_t VB,
                                          int nb, float &s0, float &s1)
{
    s0 = 0.0f;
    s1 = 0.0f;
    asm volatile("" : "+l"(VB));   // keeps the 16 offsets out of the registers a caller's loop would hold them in
    for (int kb = 0; kb < nb; kb += 16) {
        float a[16], c[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const bool ok = kb + k < nb;
            a[k] = ok ? p0[(size_t)(kb + k) * VB] : 0.0f;
            c[k] = ok ? p1[(size_t)(kb + k) * VB] : 0.0f;
        }
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            if (kb + k < nb) {
                s0 += a[k];
                s1 += c[k];
            }
        }
    }
}

// Stages f(i, s0, s1), i < B, at stage[fp(i)], s0 and s1 the band sums of
// the rays p0 + i and p1 + i; thread t of n takes the elements t, t + n, ...
// With at most four bands, four elements' loads are issued together instead
// of one's.
template <class F>
__device__ __forceinline__ void stage_bands(int t, int n, int B, const float *__restrict__ p0,
                                            const float *__restrict__ p1, size_t VB, int nb, float2 *stage, F f)
{
    if (nb <= 4) {
#pragma unroll 1
        for (int i0 = t; i0 < B; i0 += 4 * n) {
            float a[4][4], c[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + u * n;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const bool ok = k < nb && i < B;
                    a[u][k] = ok ? p0[(size_t)k * VB + i] : 0.0f;
                    c[u][k] = ok ? p1[(size_t)k * VB + i] : 0.0f;
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int i = i0 + u * n;
                float s0 = 0.0f, s1 = 0.0f;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    if (k < nb) {
                        s0 += a[u][k];
                        s1 += c[u][k];
                    }
                if (i < B) stage[fp(i)] = f(i, s0, s1);
            }
        }
        return;
    }
#pragma unroll 1
    for (int i = t; i < B; i += n) {
        float s0, s1;
        band_sum2(p0 + i, p1 + i, VB, nb, s0, s1);
        stage[fp(i)] = f(i, s0, s1);
    }
}

// Fused Step 3 and next Step 1 for the pair of views (v, v+1):
//   r     = scale_v sum_b partial[b] - b [- winv mu]     (A x^{k+1} - b [- W^-1 mu^k])
//   mu'   = mu + sigma D r                               (Step 3)
//   mubar = 2 mu' - mu [- sigma D (winv .* (mu' - mu))]  (Step 1, Alg. 1 / Alg. 2)
// Thread t of the fft_threads(P) of view pair `pair` of slice `by` of a
// batch; buf: one exchange buffer (DBL: two).  A pair past the last view
// only takes part in the barriers.  dual_stage leaves the residual in shared
// memory (LATER: in the second buffer, which the exchanges write after a
// barrier; in a loop, for the code's size) and may run on more threads than
// the transform has; the caller has them meet when it does.  KEEP: mu stays in registers between the two filters and mu', mu_bar
// are written once; otherwise (the persistent kernel's 64 registers a
// thread) mu is read again and 2 mu' - mu waits in mu_bar, each element
// touched by one thread only.  Both round alike.
struct DualArgs {
    const float2 *hhat, *tw;
    const float *partial;
    int nb;
    const float *b, *mu_in;   // mu_in may equal mu (each thread reads its elements before writing them)
    float *mu, *mu_bar;
    const float *winv;
    int lowdose;
    const ViewP *views;
    const double *scal;
    int V, B;
    Rows rows;   // of mu_bar; zeros are written past B
};

template <int P, bool DBL>
__device__ __forceinline__ void dual_stage(int t, int n, int pair, int by, float2 *buf, const DualArgs &g)
{
    const int v0 = 2 * pair, v1 = v0 + 1, V = g.V, B = g.B;
    const bool has0 = v0 < V, has1 = v1 < V;
    const size_t VB = (size_t)V * B, so = (size_t)by * VB;
    const size_t o0 = so + (size_t)(has0 ? v0 : 0) * B, o1 = so + (size_t)(has1 ? v1 : 0) * B;
    const float *partial = g.partial + (size_t)by * (g.nb - 1) * VB;   // band k of slice by at (by nb + k) VB
    const float sc0 = has0 ? g.views[v0].scale : 0.0f, sc1 = has1 ? g.views[v1].scale : 0.0f;
    const float *b = g.b, *winv = g.winv, *mu_in = g.mu_in;
    const int lowdose = g.lowdose;
    stage_bands(t, n, B, partial + o0, partial + (has1 ? o1 : o0), VB, g.nb, buf + (DBL ? fft_elems(P) : 0),
                [&](int i, float s0, float s1) {
                    float r0 = 0.0f, r1 = 0.0f;
                    if (has0) {
                        r0 = __fmaf_rn(s0, sc0, -b[o0 + i]);
                        if (lowdose) r0 = __fmaf_rn(-winv[o0 + i], mu_in[o0 + i], r0);
                    }
                    if (has1) {
                        r1 = __fmaf_rn(s1, sc1, -b[o1 + i]);
                        if (lowdose) r1 = __fmaf_rn(-winv[o1 + i], mu_in[o1 + i], r1);
                    }
                    return make_float2(r0, r1);
                });
}

template <int P, bool DBL, bool KEEP, class Ctx>
__device__ __forceinline__ void dual_update(const Ctx &c, int t, int pair, int by, float2 *buf, const DualArgs &g)
{
    constexpr int T = P / 8;
    const int v0 = 2 * pair, v1 = v0 + 1, V = g.V, B = g.B, lowdose = g.lowdose;
    const bool has0 = v0 < V, has1 = v1 < V;
    const size_t so = (size_t)by * V * B;
    const size_t o0 = so + (size_t)(has0 ? v0 : 0) * B, o1 = so + (size_t)(has1 ? v1 : 0) * B;
    const float *winv = g.winv, *mu_in = g.mu_in;
    float *mu = g.mu;
    float *mb0 = g.mu_bar + g.rows.row(by, has0 ? v0 : 0, V);
    // the second view's row from the first's
    const int m1 = has1 ? (int)((ptrdiff_t)g.rows.row(0, v1, V) - (ptrdiff_t)g.rows.row(0, v0, V)) : 0;
    const int rs = g.rows.step();
    const float sp = fscal(g.scal, F_SIGMA) * (1.0f / (float)P);
    const float2 *stage = buf + (DBL ? fft_elems(P) : 0);
    int ph = 0;
    float2 v[8];
    float2 mo[KEEP ? 4 : 1], mn[KEEP ? 4 : 1];   // mu, then 2 mu' - mu, and mu' of elements r < 4
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int i = t + r * T;
        v[r] = r < 4 && i < B ? stage[fp(i)] : make_float2(0.0f, 0.0f);
        if constexpr (KEEP)
            if (r < 4) mo[r] = make_float2(has0 && i < B ? mu_in[o0 + i] : 0.0f, has1 && i < B ? mu_in[o1 + i] : 0.0f);
    }
#pragma unroll 1
    for (int pass = 0;; ++pass) {
        fft_apply<P, false, DBL>(c, t, v, buf, ph, g.hhat, g.tw);
        if (pass) break;
        // the dual update, which leaves the second filter's input in v
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int i = t + r * T;
            float2 d = make_float2(0.0f, 0.0f);
            if (i < B && has0) {
                float2 m = KEEP ? mo[KEEP ? r : 0] : make_float2(mu_in[o0 + i], has1 ? mu_in[o1 + i] : 0.0f);
                const float2 n = make_float2(__fmaf_rn(sp, v[r].x, m.x), __fmaf_rn(sp, v[r].y, m.y));
                const float2 e = make_float2(__fmaf_rn(2.0f, n.x, -m.x), __fmaf_rn(2.0f, n.y, -m.y));
                if (lowdose) {
                    d.x = __fmul_rn(winv[o0 + i], __fsub_rn(n.x, m.x));
                    if (has1) d.y = __fmul_rn(winv[o1 + i], __fsub_rn(n.y, m.y));
                }
                if constexpr (KEEP) {
                    mo[r] = e;
                    mn[r] = n;
                }
                if (!KEEP || !lowdose) {   // Alg. 2: mu_bar = 2 mu' - mu, no second filter
                    mu[o0 + i] = n.x;
                    mb0[i * rs] = e.x;
                    if (has1) {
                        mu[o1 + i] = n.y;
                        mb0[i * rs + m1] = e.y;
                    }
                }
            } else if (i < g.rows.ld && has0) {
                mb0[i * rs] = mb0[i * rs + m1] = 0.0f;
            }
            v[r] = d;
        }
        if (!lowdose) return;
#pragma unroll
        for (int r = 4; r < 8; ++r) v[r] = make_float2(0.0f, 0.0f);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = t + r * T;
        if (i < B && has0) {
            if constexpr (KEEP) mu[o0 + i] = mn[r].x;
            mb0[i * rs] = __fmaf_rn(-sp, v[r].x, KEEP ? mo[KEEP ? r : 0].x : mb0[i * rs]);
            if (has1) {
                if constexpr (KEEP) mu[o1 + i] = mn[r].y;
                mb0[i * rs + m1] = __fmaf_rn(-sp, v[r].y, KEEP ? mo[KEEP ? r : 0].y : mb0[i * rs + m1]);
            }
        }
    }
}

}  // namespace ctpd
