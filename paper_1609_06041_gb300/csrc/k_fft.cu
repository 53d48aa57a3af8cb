// k_fft.cu -- the preconditioner D as a frequency-domain filter.
//
// D applies, along the detector of every view, the linear (zero-padded)
// convolution with the taps t[k], |k| < half (Eq. 24 / Eq. 32 give the
// taps from H).  With the view zero-padded to the period P >= 2B, the
// circular convolution with the taps placed at k mod P equals that linear
// convolution on bins 0..B-1, so D = IFFT_P(Hhat . FFT_P(.)) with Hhat the
// P-point DFT of the circularly placed taps.  The taps are real, so two
// views travel as the real and imaginary parts of one complex sequence.
//
// P / 8 threads run one transform with its elements in registers
// (body_fft.cuh); the kernels are instantiated per length, so that all
// index arithmetic is constant, and a block holds one transform (more for
// P < 256, to fill a warp).
#include <math.h>

#include <algorithm>

#include "body_fft.cuh"

namespace ctpd {

// Convolution length: the period n_fft of the taps, at least the shortest
// transform.
int fft_length(int n_bins)
{
    int p = 64;
    while (p < 2 * n_bins) p <<= 1;
    return p;
}

size_t fft_table_elems(int p) { return fft_tw_elems(p); }

// tw: fft_table_elems(p) twiddles of a p-point transform (see fft_tw_elems)
void fft_table(int p, float2 *tw)
{
    const int half = fft_tw_half(p), last = fft_last_radix(p);
    for (int ns = 8; ns < p; ns *= 8) {
        const int R = p / ns >= 8 ? 8 : last;
        for (int r = 0; r < R; ++r)
            for (int k = 0; k < ns; ++k) {
                const double ang = -2.0 * M_PI * (double)((long)r * k * (p / (ns * R))) / (double)p;
                const float2 w = make_float2((float)cos(ang), (float)sin(ang));
                tw[fft_tw_off(ns) + r * ns + k] = w;
                tw[half + fft_tw_off(ns) + r * ns + k] = make_float2(w.x, -w.y);
            }
    }
}

namespace {

constexpr int block_threads(int P) { return fft_threads(P) < 32 ? 32 : fft_threads(P); }
constexpr int block_transforms(int P) { return block_threads(P) / fft_threads(P); }
constexpr size_t buf_bytes(int P) { return sizeof(float2) * fft_elems(P); }
// dynamic shared memory: two exchange buffers per transform
constexpr size_t block_smem(int P) { return 2 * buf_bytes(P) * block_transforms(P); }
// three blocks of 256 threads an SM (85 registers): 360 view pairs on 152 SMs are one wave
constexpr int min_blocks(int P) { return block_threads(P) >= 768 ? 1 : 768 / block_threads(P); }

// Threads of a block that reads band sums.  A grid with a block or more for
// every SM takes the transforms' threads only.  A smaller one (few views,
// small images) is bound by the latency of its 16 loads an element, so there
// 512 threads stage the residual and the transforms' threads go on alone (the
// dual step without and with the extra threads, cold: 512^2 / 32 views 12.8
// and 10.6 us, 64^2 / 90 8.7 and 6.8; a solve's iteration 29.5 and 28.3, 18.8
// and 17.3 us).
constexpr int wide_threads(int P) { return block_threads(P) < 512 ? 512 : block_threads(P); }
bool wide_grid(const Geometry *g, int batch)
{
    const int per = std::max(1, 32 / fft_threads(g->p_fft));   // transforms a block
    return wide_threads(g->p_fft) > block_threads(g->p_fft) &&
           (long long)((g->n_views + 1) / 2) * batch < (long long)g->n_sm * per;
}

// Calls f(IntC<P>) for the transform length p.
template <class F>
void with_length(int p, F f)
{
    switch (p) {
    case 64: f(IntC<64>{}); break;
    case 128: f(IntC<128>{}); break;
    case 256: f(IntC<256>{}); break;
    case 512: f(IntC<512>{}); break;
    case 1024: f(IntC<1024>{}); break;
    case 2048: f(IntC<2048>{}); break;
    case 4096: f(IntC<4096>{}); break;
    case 8192: f(IntC<8192>{}); break;
    default: break;
    }
}

// This thread's place: element offset t, transform number, exchange buffers.
template <int P>
struct Place {
    int t, which;
    float2 *buf;
    __device__ __forceinline__ Place(float2 *sm)
    {
        constexpr int T = fft_threads(P);
        t = threadIdx.x % T;
        const int sub = threadIdx.x / T;
        which = blockIdx.x * block_transforms(P) + sub;
        buf = sm + (size_t)sub * 2 * fft_elems(P);
    }
};

}  // namespace

// Hhat = DFT_P of the taps placed circularly (t[k] at k mod P).
template <int P>
__global__ void __launch_bounds__(block_threads(P), min_blocks(P))
k_hhat(const float *__restrict__ taps, int half, const float2 *__restrict__ tw, float2 *__restrict__ hhat)
{
    extern __shared__ float2 fsm[];
    pdl_wait();
    pdl_launch();   // a filter launched after this one stages its input meanwhile
    const Place<P> pl(fsm);
    float2 v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        // index i holds t[k] with k = i (i < half) or k = i - P (i > P - half)
        const int i = pl.t + r * fft_threads(P);
        float x = 0.0f;
        if (i < half) x = taps[half - 1 + i];
        else if (i > P - half) x = taps[half - 1 + (i - P)];
        v[r] = make_float2(x, 0.0f);
    }
    int ph = 0;
    fft_regs<P, false, true>(whole_block(), pl.t, v, pl.buf, ph, tw, 1.0f);
    if (pl.which != 0) return;
#pragma unroll
    for (int r = 0; r < 8; ++r) hhat[pl.t + r * fft_threads(P)] = v[r];
}

void launch_hhat(const Geometry *g, const float *taps, int half, float2 *hhat, cudaStream_t st)
{
    counted();
    with_length(g->p_fft, [&](auto L) {
        constexpr int P = decltype(L)::value;
        launch_kernel(k_hhat<P>, dim3(1), dim3(block_threads(P)), block_smem(P), st, taps, half, g->d_tw, hhat);
    });
}

// out = post .* D(pre .* in) * sc, sc = 1 (mode 0) or -sigma (mode 1);
// one transform per pair of views (v, v+1) of image `blockIdx.y`.  BANDS: the
// input is A x given as band partial sums (in = partial, nb bands), added
// in band order and scaled by the views' path lengths.  early: the kernel's
// predecessor wrote hhat only, so the input is staged before the wait for it.
// The plain form keeps no state, so it runs at 64 registers, four 256-thread
// blocks an SM: 4 x 720 views x 736 bins 39.0 -> 22.3 us (issue 58 %; 23.8 us
// at three blocks), the transform of the taps before it 12 -> 5.3 us.
template <int P, bool BANDS, bool WIDE>
__global__ void __launch_bounds__(WIDE ? wide_threads(P) : block_threads(P),
                                  WIDE ? 1 : BANDS ? min_blocks(P) : 4 * min_blocks(P) / 3)
k_filter_fft(const float2 *__restrict__ hhat, const float *__restrict__ in, float *__restrict__ out, Rows ldo,
             const float *__restrict__ pre, const float *__restrict__ post, int mode,
             const double *__restrict__ scal, int V, int B, const float2 *__restrict__ tw, int nb,
             const ViewP *__restrict__ views, int early)
{
    extern __shared__ float2 fsm[];
    if (!early) pdl_wait();
    constexpr int T = fft_threads(P);
    const Place<P> pl(fsm);
    const int v0 = 2 * pl.which, v1 = v0 + 1;
    const bool has0 = v0 < V, has1 = v1 < V;
    const size_t VB = (size_t)V * B, base = (size_t)blockIdx.y * VB;
    const size_t o0 = base + (size_t)(has0 ? v0 : 0) * B, o1 = base + (size_t)(has1 ? v1 : 0) * B;
    if constexpr (BANDS) {
        // every thread stages elements of the block's transforms, in the second buffer (the exchanges write it
        // after a barrier)
        for (int q = 0; q < block_transforms(P); ++q) {
            const int w0 = 2 * (blockIdx.x * block_transforms(P) + q), w1 = w0 + 1 < V ? w0 + 1 : w0;
            if (w0 >= V) break;
            const float *p = in + (size_t)blockIdx.y * nb * VB;
            const float c0 = views[w0].scale, c1 = w1 > w0 ? views[w1].scale : 0.0f;
            stage_bands(threadIdx.x, blockDim.x, B, p + (size_t)w0 * B, p + (size_t)w1 * B, VB, nb,
                        fsm + (2 * q + 1) * fft_elems(P),
                        [&](int, float s0, float s1) { return make_float2(s0 * c0, s1 * c1); });
        }
        __syncthreads();
        if (WIDE && threadIdx.x >= block_threads(P)) return;
    } else {
#pragma unroll 1
        for (int i = pl.t; i < B; i += T) {
            float x0 = has0 ? in[o0 + i] : 0.0f, x1 = has1 ? in[o1 + i] : 0.0f;
            if (pre) {
                if (has0) x0 *= pre[o0 + i];
                if (has1) x1 *= pre[o1 + i];
            }
            pl.buf[fft_elems(P) + fp(i)] = make_float2(x0, x1);
        }
    }
    if (early) pdl_wait();
    const float2 *stage = pl.buf + fft_elems(P);
    float2 v[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) {
        const int i = pl.t + r * T;
        v[r] = r < 4 && i < B && has0 ? stage[fp(i)] : make_float2(0.0f, 0.0f);
    }
    int ph = 0;
    const GroupCtx ctx{(int)threadIdx.x, block_threads(P), 1};
    fft_apply<P, false, true>(ctx, pl.t, v, pl.buf, ph, hhat, tw);
    const float sc = ((mode == 1) ? -fscal(scal, F_SIGMA) : 1.0f) / (float)P;
    float *q0 = out + ldo.row(blockIdx.y, has0 ? v0 : 0, V), *q1 = has1 ? out + ldo.row(blockIdx.y, v1, V) : q0;
    const int rs = ldo.step();
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = pl.t + r * T;
        if (i < B && has0) {
            float y0 = v[r].x * sc, y1 = v[r].y * sc;
            if (post) {
                y0 *= post[o0 + i];
                if (has1) y1 *= post[o1 + i];
            }
            q0[i * rs] = y0;
            if (has1) q1[i * rs] = y1;
        } else if (i < ldo.ld && has0) {
            q0[i * rs] = q1[i * rs] = 0.0f;
        }
    }
}

// grid of one transform per view pair (views: per view) and image
template <int P>
static dim3 fft_grid(int transforms, int batch)
{
    return dim3((transforms + block_transforms(P) - 1) / block_transforms(P), batch);
}

// out = D (A x) from the projector's band partial sums
void launch_filter_fft_bands(const Geometry *g, const float2 *hhat, const float *partial, float *out, int batch,
                             cudaStream_t st, Rows ldo)
{
    counted();
    with_length(g->p_fft, [&](auto L) {
        constexpr int P = decltype(L)::value;
        const bool wide = wide_grid(g, batch);
        launch_kernel(wide ? k_filter_fft<P, true, true> : k_filter_fft<P, true, false>,
                      fft_grid<P>((g->n_views + 1) / 2, batch), dim3(wide ? wide_threads(P) : block_threads(P)),
                      block_smem(P), st, hhat, partial, out, ldo, nullptr, nullptr, 0, nullptr, g->n_views, g->n_bins,
                      g->d_tw, proj_bands(g->n), g->d_views, 0);
    });
}

void launch_filter_fft(const Geometry *g, const float2 *hhat, const float *in, float *out,
                       const float *pre, const float *post, int mode, const double *scal, int batch,
                       cudaStream_t st, Rows ldo, bool early)
{
    counted();
    PdlScope pdl(early || t_pdl);
    with_length(g->p_fft, [&](auto L) {
        constexpr int P = decltype(L)::value;
        launch_kernel(k_filter_fft<P, false, false>, fft_grid<P>((g->n_views + 1) / 2, batch), dim3(block_threads(P)),
                      block_smem(P), st, hhat, in, out, ldo, pre, post, mode, scal, g->n_views, g->n_bins, g->d_tw, 0,
                      nullptr, early ? 1 : 0);
    });
}

// The fused dual step.  Bound: the latency of the 16 band loads an element
// and of the exchanges between stages (issue 46 %, 29 % of the warp slots).
// 512^2 / 720 views / 736 bins (360 view pairs, one wave of three 256-thread
// blocks an SM): 35.3 -> 22.7 us; 32 views (16 pairs, the wide form): 16.6 ->
// 10.6 us; 64^2 / 90 / 95: 14.6 -> 6.8 us (cold cache).
template <int P, bool WIDE>
__global__ void __launch_bounds__(WIDE ? wide_threads(P) : block_threads(P), WIDE ? 1 : min_blocks(P))
k_dual_fft(const DualArgs a)
{
    extern __shared__ float2 fsm[];
    pdl_wait();
    const Place<P> pl(fsm);
    if (WIDE) {
        for (int q = 0; q < block_transforms(P); ++q)
            dual_stage<P, true>(threadIdx.x, blockDim.x, blockIdx.x * block_transforms(P) + q, blockIdx.y,
                                fsm + 2 * q * fft_elems(P), a);
        __syncthreads();
        if (threadIdx.x >= block_threads(P)) return;
    } else {
        dual_stage<P, true>(pl.t, fft_threads(P), pl.which, blockIdx.y, pl.buf, a);
    }
    const GroupCtx ctx{(int)threadIdx.x, block_threads(P), 1};
    dual_update<P, true, true>(ctx, pl.t, pl.which, blockIdx.y, pl.buf, a);
}

// =====================================================================
// The shift-variant preconditioner D = T_lo + S T_hi S (S = diag(s),
// s_i = sqrt(kappa w_i)): T_lo and T_hi are the convolutions with the taps
// of the low and high bands H_lo + H_hi = H of Eq. 24, so that D tends to
// the pure ramp of Eq. 32 at low frequency and to W at high frequency, the
// two limits of D = (tau A A^T + W^-1)^-1 (Eq. 23).  One view y per block:
// the real sequences y and S y travel as one complex sequence,
//     Z = FFT(y + i S y),  F y = (Z + conj Z(-k)) / 2,  F(S y) = (Z - conj Z(-k)) / 2i,
// and one inverse transform of
//     Y = H_lo F y + i H_hi F(S y) = hs Z + hd conj Z(-k),   hs, hd = (H_lo +- H_hi) / 2,
// returns u + i v with u = P T_lo y and v = P T_hi S y (both real, as
// H_lo and H_hi are Hermitian), so D y = (u + s v) / P.
// =====================================================================
__global__ void k_sv_combine(float2 *__restrict__ hs, float2 *__restrict__ hd, int P)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= P) return;
    const float2 lo = hs[k], hi = hd[k];
    hs[k] = make_float2(0.5f * (lo.x + hi.x), 0.5f * (lo.y + hi.y));
    hd[k] = make_float2(0.5f * (lo.x - hi.x), 0.5f * (lo.y - hi.y));
}

void launch_sv_hhat(const Geometry *g, const float *taps_lo, const float *taps_hi, int half, float2 *hs, float2 *hd,
                    cudaStream_t st)
{
    launch_hhat(g, taps_lo, half, hs, st);
    launch_hhat(g, taps_hi, half, hd, st);
    counted();
    k_sv_combine<<<(g->p_fft + 255) / 256, 256, 0, st>>>(hs, hd, g->p_fft);
}

// v <- the shift-variant D's (u, v) pair (up to the factor P) of the
// sequence (y, S y) in v: forward transform, Y(k) = hs(k) Z(k) + hd(k) conj
// Z(P-k) with the mirrored elements taken through an exchange buffer, inverse.
template <int P>
__device__ __forceinline__ void sv_apply(int t, float2 (&v)[8], float2 *buf, int &ph, const float2 *__restrict__ hs,
                                         const float2 *__restrict__ hd, const float2 *__restrict__ tw)
{
    constexpr int T = fft_threads(P);
    float s = 1.0f;
#pragma unroll 1
    for (int inv = 0; inv < 2; ++inv) {
        fft_regs<P, true, true>(whole_block(), t, v, buf, ph, tw + inv * fft_tw_half(P), s);
        s = -1.0f;
        if (inv == 0) {
            float2 *m = buf + ph * fft_elems(P);
            ph ^= 1;
#pragma unroll
            for (int r = 0; r < 8; ++r) m[fp(t + r * T)] = v[r];
            __syncthreads();
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                const int k = t + r * T;
                const float2 z = m[fp((P - k) & (P - 1))];
                v[r] = cadd(cmul(hs[k], v[r]), cmul(hd[k], make_float2(z.x, -z.y)));
            }
        }
    }
}

// sum of the nb band partial sums of one ray, in band order
__device__ __forceinline__ float band_sum(const float *__restrict__ p, size_t VB, int nb)
{
    float acc = 0.0f;
    for (int q = 0; q < nb; ++q) acc += p[q * VB];
    return acc;
}

// out = post .* D(pre .* in) * sc, sc = 1 (mode 0) or -sigma (mode 1), D the
// shift-variant form; one transform per view of image blockIdx.y.
// BANDS: the input is A x as the projector's nb band partial sums.
template <int P, bool BANDS>
__global__ void __launch_bounds__(block_threads(P), min_blocks(P))
k_filter_sv(const float2 *__restrict__ hs, const float2 *__restrict__ hd, const float *__restrict__ sv,
            const float *__restrict__ in, float *__restrict__ out, Rows ldo, const float *__restrict__ pre,
            const float *__restrict__ post, int mode, const double *__restrict__ scal, int V, int B,
            const float2 *__restrict__ tw, int nb, const ViewP *__restrict__ views)
{
    extern __shared__ float2 fsm[];
    pdl_wait();
    constexpr int T = fft_threads(P);
    const Place<P> pl(fsm);
    const bool has = pl.which < V;
    const int vw = has ? pl.which : 0;
    const size_t VB = (size_t)V * B;
    const size_t o = (size_t)blockIdx.y * VB + (size_t)vw * B;
    const float *s = sv + (size_t)vw * B;   // the weights, so S, are one slice's
    float2 v[8];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = pl.t + r * T;
        float y = 0.0f, sy = 0.0f;
        if (i < B && has) {
            if (BANDS) {
                y = band_sum(in + (size_t)blockIdx.y * nb * VB + (size_t)vw * B + i, VB, nb) * views[vw].scale;
            } else {
                y = in[o + i];
                if (pre) y *= pre[o + i];
            }
            sy = s[i] * y;
        }
        v[r] = make_float2(y, sy);
        v[r + 4] = make_float2(0.0f, 0.0f);
    }
    int ph = 0;
    sv_apply<P>(pl.t, v, pl.buf, ph, hs, hd, tw);
    float *q = out + ldo.row(blockIdx.y, vw, V);
    const int rs = ldo.step();
    const float sc = ((mode == 1) ? -fscal(scal, F_SIGMA) : 1.0f) / (float)P;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = pl.t + r * T;
        if (i < B && has) {
            float y = fmaf(s[i], v[r].y, v[r].x) * sc;
            if (post) y *= post[o + i];
            q[i * rs] = y;
        } else if (i < ldo.ld && has) {
            q[i * rs] = 0.0f;
        }
    }
}

void launch_filter_sv(const Geometry *g, const float2 *hs, const float2 *hd, const float *sv, const float *in,
                      float *out, const float *pre, const float *post, int mode, const double *scal, int batch,
                      cudaStream_t st, Rows ldo)
{
    counted();
    with_length(g->p_fft, [&](auto L) {
        constexpr int P = decltype(L)::value;
        launch_kernel(k_filter_sv<P, false>, fft_grid<P>(g->n_views, batch), dim3(block_threads(P)), block_smem(P), st,
                      hs, hd, sv, in, out, ldo, pre, post, mode, scal, g->n_views, g->n_bins, g->d_tw, 0, nullptr);
    });
}

void launch_filter_sv_bands(const Geometry *g, const float2 *hs, const float2 *hd, const float *sv,
                            const float *partial, float *out, int batch, cudaStream_t st, Rows ldo)
{
    counted();
    with_length(g->p_fft, [&](auto L) {
        constexpr int P = decltype(L)::value;
        launch_kernel(k_filter_sv<P, true>, fft_grid<P>(g->n_views, batch), dim3(block_threads(P)), block_smem(P), st,
                      hs, hd, sv, partial, out, ldo, nullptr, nullptr, 0, nullptr, g->n_views, g->n_bins, g->d_tw,
                      proj_bands(g->n), g->d_views);
    });
}

// Fused Step 3 and next Step 1 of Algorithm 1 with the shift-variant D, one
// view per transform (the form of k_dual_fft):
//   r = scale_v sum_b partial[b] - b - winv mu;  mu' = mu + sigma D r;
//   mubar = 2 mu' - mu - sigma D (winv .* (mu' - mu)).
template <int P>
__global__ void __launch_bounds__(block_threads(P), min_blocks(P))
k_dual_sv(const float2 *__restrict__ hs, const float2 *__restrict__ hd, const float *__restrict__ sv,
          const float *__restrict__ partial, int nb, const float *__restrict__ b, float *mu,
          float *__restrict__ mu_bar, Rows rows, const float *__restrict__ winv, const ViewP *__restrict__ views,
          const double *__restrict__ scal, int V, int B, const float2 *__restrict__ tw)
{
    extern __shared__ float2 fsm[];
    pdl_wait();
    constexpr int T = fft_threads(P);
    const Place<P> pl(fsm);
    const bool has = pl.which < V;
    const int vw = has ? pl.which : 0;
    const size_t VB = (size_t)V * B, o = (size_t)vw * B;
    const float *s = sv + o;
    const float sc = views[vw].scale;
    const float sp = fscal(scal, F_SIGMA) * (1.0f / (float)P);
    float2 v[8];
    float mo[4], mn[4];   // mu, then 2 mu' - mu, and mu'
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = pl.t + r * T;
        float res = 0.0f, sr = 0.0f;
        mo[r] = 0.0f;
        if (i < B && has) {
            mo[r] = mu[o + i];
            res = band_sum(partial + o + i, VB, nb) * sc - b[o + i] - winv[o + i] * mo[r];
            sr = s[i] * res;
        }
        v[r] = make_float2(res, sr);
        v[r + 4] = make_float2(0.0f, 0.0f);
    }
    int ph = 0;
#pragma unroll 1
    for (int pass = 0;; ++pass) {
        sv_apply<P>(pl.t, v, pl.buf, ph, hs, hd, tw);
        if (pass) break;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int i = pl.t + r * T;
            float d = 0.0f, sd = 0.0f;
            if (i < B && has) {
                mn[r] = fmaf(sp, fmaf(s[i], v[r].y, v[r].x), mo[r]);
                d = winv[o + i] * (mn[r] - mo[r]);
                sd = s[i] * d;
                mo[r] = fmaf(2.0f, mn[r], -mo[r]);
            }
            v[r] = make_float2(d, sd);
            v[r + 4] = make_float2(0.0f, 0.0f);
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = pl.t + r * T;
        if (i < B && has) {
            mu[o + i] = mn[r];
            mu_bar[rows.row(0, vw, V) + i * rows.step()] = fmaf(-sp, fmaf(s[i], v[r].y, v[r].x), mo[r]);
        } else if (i < rows.ld && has) {
            mu_bar[rows.row(0, vw, V) + i * rows.step()] = 0.0f;
        }
    }
}

void launch_dual_sv(const Geometry *g, const float2 *hs, const float2 *hd, const float *sv, const float *partial,
                    const float *b, float *mu, float *mu_bar, const float *winv, const double *scal,
                    cudaStream_t st)
{
    counted();
    with_length(g->p_fft, [&](auto L) {
        constexpr int P = decltype(L)::value;
        launch_kernel(k_dual_sv<P>, fft_grid<P>(g->n_views, 1), dim3(block_threads(P)), block_smem(P), st, hs, hd, sv,
                      partial, proj_bands(g->n), b, mu, mu_bar, at_rows(g), winv, g->d_views, scal, g->n_views, g->n_bins,
                      g->d_tw);
    });
}

// one exchange buffer, per thread group of a transform (the persistent kernel)
size_t dual_fft_smem(const Geometry *g) { return buf_bytes(g->p_fft); }

void launch_dual_fft(const Geometry *g, const float2 *hhat, const float *partial, const float *b, float *mu,
                     float *mu_bar, const float *winv, int lowdose, const double *scal, cudaStream_t st)
{
    launch_dual_fft_batched(g, hhat, partial, b, mu, mu, mu_bar, winv, lowdose, scal, 1, st);
}

void launch_dual_fft_batched(const Geometry *g, const float2 *hhat, const float *partial, const float *b,
                             const float *mu_in, float *mu_out, float *mu_bar, const float *winv, int lowdose,
                             const double *scal, int batch, cudaStream_t st)
{
    counted();
    with_length(g->p_fft, [&](auto L) {
        constexpr int P = decltype(L)::value;
        const bool wide = wide_grid(g, batch);
        const DualArgs a{hhat, g->d_tw, partial, proj_bands(g->n), b, mu_in, mu_out, mu_bar, winv, lowdose,
                         g->d_views, scal, g->n_views, g->n_bins, at_rows(g)};
        launch_kernel(wide ? k_dual_fft<P, true> : k_dual_fft<P, false>, fft_grid<P>((g->n_views + 1) / 2, batch),
                      dim3(wide ? wide_threads(P) : block_threads(P)), block_smem(P), st, a);
    });
}

// Adjoint of one dual step (Step 3 and the next Step 1) for the pair of
// views (v, v+1) of slice blockIdx.y.  Forward (W = diag(winv), low-dose):
//   r      = A x' - b - W mu
//   mu'    = mu + sigma D r
//   mubar' = 2 mu' - mu - sigma D W (mu' - mu)
// Given gm = dL/dmu' and gmb = dL/dmubar', with D^T applied through the
// conjugate response:
//   h   = D^T gmb
//   gm1 = gm + 2 gmb - sigma W h          (total dL/dmu')
//   gr  = sigma D^T gm1                   (dL/dr)
//   gmu = gm1 - W gr - gmb + sigma W h    (dL/dmu)
// and writes r and v = W (mu' - mu) for the tap correlations
// dL/dt += sigma (gm1 * r) - sigma (gmb * v).  Few-view drops every W term.
template <int P>
__global__ void __launch_bounds__(block_threads(P), min_blocks(P))
k_dual_bwd_fft(const float2 *__restrict__ hhat, const float *__restrict__ partial, int nb,
               const float *__restrict__ b, const float *__restrict__ winv, const float *__restrict__ mu,
               const float *__restrict__ mu1, const float *__restrict__ gm, const float *__restrict__ gmb,
               float *__restrict__ gmu_out, float *__restrict__ gr_out, float *gm1_out,
               float *__restrict__ r_out, float *__restrict__ v_out, int lowdose,
               const ViewP *__restrict__ views, const double *__restrict__ scal, int V, int B, Rows rows,
               const float2 *__restrict__ tw)
{
    extern __shared__ float2 fsm[];
    pdl_wait();
    constexpr int T = fft_threads(P);
    const Place<P> pl(fsm);
    const int v0 = 2 * pl.which, v1 = v0 + 1;
    const bool has0 = v0 < V, has1 = v1 < V;
    const size_t VB = (size_t)V * B, so = (size_t)blockIdx.y * VB;
    const size_t o0 = so + (size_t)(has0 ? v0 : 0) * B, o1 = so + (size_t)(has1 ? v1 : 0) * B;
    partial += (size_t)blockIdx.y * (nb - 1) * VB;
    const float sigma = fscal(scal, F_SIGMA);
    const float invP = 1.0f / (float)P;
    const float sc0 = has0 ? views[v0].scale : 0.0f, sc1 = has1 ? views[v1].scale : 0.0f;

    // pass 0: h = D^T gmb, which forms gm1 = gm + 2 gmb - sigma W h; pass 1: gr = sigma D^T gm1
    float2 v[8], hr[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = pl.t + r * T;
        v[r] = make_float2(i < B && has0 ? gmb[o0 + i] : 0.0f, i < B && has1 ? gmb[o1 + i] : 0.0f);
        v[r + 4] = make_float2(0.0f, 0.0f);
    }
    int ph = 0;
#pragma unroll 1
    for (int pass = 0;; ++pass) {
        fft_apply<P, true, true>(whole_block(), pl.t, v, pl.buf, ph, hhat, tw);
        if (pass) break;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            const int i = pl.t + r * T;
            float g0 = 0.0f, g1 = 0.0f;
            hr[r] = make_float2(v[r].x * invP, v[r].y * invP);
            if (i < B && has0) {
                g0 = gm[o0 + i] + 2.0f * gmb[o0 + i];
                if (lowdose) g0 -= sigma * winv[o0 + i] * hr[r].x;
                gm1_out[o0 + i] = g0;
            }
            if (i < B && has1) {
                g1 = gm[o1 + i] + 2.0f * gmb[o1 + i];
                if (lowdose) g1 -= sigma * winv[o1 + i] * hr[r].y;
                gm1_out[o1 + i] = g1;
            }
            v[r] = make_float2(g0, g1);
            v[r + 4] = make_float2(0.0f, 0.0f);
        }
    }
    // the rest element by element, in a loop (for the code's size): the
    // thread's own D^T gm1 and h wait in the free exchange buffer
    float2 *st = pl.buf + ph * fft_elems(P);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = pl.t + r * T;
        st[fp(i)] = v[r];
        st[fp(P / 2 + i)] = hr[r];
    }
    if (!has0) return;
    // dL/dr, the adjoint's input of A^T: zeros past B
    float *gp0 = gr_out + rows.row(blockIdx.y, v0, V), *gp1 = gr_out + rows.row(blockIdx.y, has1 ? v1 : v0, V);
    const int rs = rows.step();
    for (int i = B + pl.t; i < rows.ld; i += T) gp0[i * rs] = gp1[i * rs] = 0.0f;
#pragma unroll 1
    for (int i = pl.t; i < B; i += T) {
        float s[2];
        band_sum2(partial + o0 + i, partial + (has1 ? o1 : o0) + i, VB, nb, s[0], s[1]);
        const float2 res = st[fp(i)], h = st[fp(P / 2 + i)];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (k == 1 && !has1) break;
            const size_t o = (k == 0 ? o0 : o1) + i;
            const float gr = sigma * ((k == 0 ? res.x : res.y) * invP);
            const float g1v = gm1_out[o], hv = k == 0 ? h.x : h.y;
            float gmu = g1v - gmb[o];
            float r = s[k] * (k == 0 ? sc0 : sc1) - b[o];
            float vv = 0.0f;
            if (lowdose) {
                gmu += -winv[o] * gr + sigma * winv[o] * hv;
                r -= winv[o] * mu[o];
                vv = winv[o] * (mu1[o] - mu[o]);
            }
            gmu_out[o] = gmu;
            (k == 0 ? gp0 : gp1)[i * rs] = gr;
            r_out[o] = r;
            v_out[o] = vv;
        }
    }
}

void launch_dual_bwd_fft(const Geometry *g, const float2 *hhat, const float *partial, const float *b,
                         const float *winv, const float *mu, const float *mu1, const float *gm, const float *gmb,
                         float *gmu, float *gr, float *gm1, float *r, float *v, int lowdose, const double *scal,
                         int batch, cudaStream_t st)
{
    counted();
    with_length(g->p_fft, [&](auto L) {
        constexpr int P = decltype(L)::value;
        launch_kernel(k_dual_bwd_fft<P>, fft_grid<P>((g->n_views + 1) / 2, batch), dim3(block_threads(P)),
                      block_smem(P), st, hhat, partial, proj_bands(g->n), b, winv, mu, mu1, gm, gmb, gmu, gr, gm1, r,
                      v, lowdose, g->d_views, scal, g->n_views, g->n_bins, at_rows(g), g->d_tw);
    });
}

bool fft_supported(const Geometry *g) { return g->n_fft <= FFT_MAX_P; }

void kernel_attrs_fft(const Geometry *g)
{
    if (!fft_supported(g)) return;
    with_length(g->p_fft, [&](auto L) {
        constexpr int P = decltype(L)::value;
        const int sm = (int)block_smem(P);
        cudaFuncSetAttribute(k_hhat<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        cudaFuncSetAttribute(k_filter_fft<P, false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        cudaFuncSetAttribute(k_filter_fft<P, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        cudaFuncSetAttribute(k_filter_fft<P, true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        cudaFuncSetAttribute(k_dual_fft<P, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        cudaFuncSetAttribute(k_dual_fft<P, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        cudaFuncSetAttribute(k_dual_bwd_fft<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        cudaFuncSetAttribute(k_filter_sv<P, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        cudaFuncSetAttribute(k_filter_sv<P, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
        cudaFuncSetAttribute(k_dual_sv<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, sm);
    });
}

}  // namespace ctpd
