// k_misc.cu -- element-wise helpers, deterministic reductions and the
// scalar program of the step-size setup (Alg. 1 / Alg. 2 boxes).
#include <math.h>

#include <algorithm>

#include <cooperative_groups.h>

#include "ctpd_internal.cuh"

namespace ctpd {

static int grid_for(size_t n, int threads)
{
    size_t b = (n + threads - 1) / threads;
    return (int)(b < 152 * 16 ? (b == 0 ? 1 : b) : 152 * 16);
}

__global__ void k_fill(float *p, float v, size_t n)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        p[i] = v;
}

void launch_fill(float *p, float v, size_t n, cudaStream_t st)
{
    counted();
    k_fill<<<grid_for(n, 256), 256, 0, st>>>(p, v, n);
}

__global__ void k_recip(const float *w, float *winv, size_t n)
{
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        winv[i] = 1.0f / w[i];
}

void launch_recip(const float *w, float *winv, size_t n, cudaStream_t st)
{
    counted();
    k_recip<<<grid_for(n, 256), 256, 0, st>>>(w, winv, n);
}

// s = sqrt(kappa w): the diagonal of the shift-variant preconditioner
__global__ void k_sv_scale(const float *w, const double *scal, float *s, size_t n)
{
    const float kappa = (float)scal[S_KAPPA];
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        s[i] = sqrtf(kappa * w[i]);
}

void launch_sv_scale(const float *w, const double *scal, float *s, size_t n, cudaStream_t st)
{
    counted();
    k_sv_scale<<<grid_for(n, 256), 256, 0, st>>>(w, scal, s, n);
}

// +-1 from a 32-bit integer hash of i (the lowbias32 mixing of C. Wellons):
// a start vector with components in every symmetry class
__device__ __forceinline__ float hash_sign(size_t i)
{
    unsigned x = (unsigned)i * 2654435761u + 12345u;
    x ^= x >> 16;
    x *= 0x7feb352du;
    x ^= x >> 15;
    x *= 0x846ca68bu;
    x ^= x >> 16;
    return (x & 1u) ? 1.0f : -1.0f;
}

// Deterministic reductions: a fixed grid of DOT_BLOCKS blocks; each thread
// sums its grid-stride elements in float, warps add their lanes by a fixed
// shuffle tree, the warp sums of a block are added in order, and the block
// partials the same way.  Everything is float (FP64 arithmetic is slow on
// this GPU); the relative error stays near 1e-6, well inside what the
// step-size setup needs.
constexpr int DOT_BLOCKS = 1216;   // 8 blocks per SM of 152: one element group per thread
constexpr int DOT_THREADS = 256;
size_t dot_partials_doubles() { return DOT_BLOCKS + 64; }   // + room for the ticket counter

__device__ __forceinline__ float warp_sum(float v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// block total (valid in thread 0) of the float per-thread sums: warp trees,
// then the warp sums in order
__device__ __forceinline__ float block_sum(float v)
{
    __shared__ float wsum[DOT_THREADS / 32];
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = v;
    __syncthreads();
    float t = 0.0f;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < DOT_THREADS / 32; ++k) t += wsum[k];
    }
    return t;
}

// sum of the np block partials (strided runs per thread, then block_sum),
// valid in thread 0; every thread of the block calls it.  The partials are
// read from L2 (written by other blocks before their fence).
__device__ __forceinline__ float partials_sum(const double *partials, int np)
{
    float t = 0.0f;
    for (int i = threadIdx.x; i < np; i += blockDim.x) t += (float)__ldcg(partials + i);
    return block_sum(t);
}

// The float copies of the scalars the per-iteration kernels read
__device__ __forceinline__ void float_copies(double *s)
{
    float *f = reinterpret_cast<float *>(s + S_F32);
    f[F_TAU] = (float)s[S_TAU];
    f[F_SIGMA] = (float)s[S_SIGMA];
    f[F_LAMBDA] = (float)s[S_LAMBDA];
    f[F_INV8LAM] = (float)s[S_INV8LAM];
}

// The solve's setup around its Lanczos runs, in three launches.  Each part is
// an element-wise pass or a few scalars, far shorter than a launch; as a
// chain of some fifteen kernels and memsets they cost a 64^2 / 90-view solve
// (20 iterations) 21 of its 607 us.
//
// First: the input checks (w > 0 and finite, b finite; bits in the flag
// word), W^-1 and, where the Lanczos runs follow, W^-1/2 and both start
// vectors; partial sums of 1 / w by the deterministic reduction above.
__global__ void __launch_bounds__(DOT_THREADS)
k_setup_data(const float *b, const float *w, size_t n, float *winv, float *sw, float *t_sino, float *t_img,
             size_t n_img, double *partials, unsigned *flags, unsigned *ticket, unsigned *ticket2)
{
    const size_t tid = blockIdx.x * (size_t)blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
    if (tid == 0) {   // the reductions' counters
        *ticket = 0u;
        *ticket2 = 0u;
    }
    unsigned f = 0;
    float acc = 0.0f;
    for (size_t i = tid; i < n; i += stride) {
        if (!isfinite(b[i])) f |= CHK_NONFINITE_INPUT;
        if (w) {
            const float wi = w[i], v = 1.0f / wi;
            if (!isfinite(wi)) f |= CHK_NONFINITE_INPUT;
            else if (!(wi > 0.0f)) f |= CHK_WEIGHT_NOT_POSITIVE;
            winv[i] = v;
            if (sw) sw[i] = sqrtf(v);
            acc += v;
        }
        if (t_sino) t_sino[i] = hash_sign(i);
    }
    if (t_img)
        for (size_t i = tid; i < n_img; i += stride) t_img[i] = hash_sign(i);
    f = __reduce_or_sync(0xffffffffu, f);
    if ((threadIdx.x & 31) == 0 && f) atomicOr(flags, f);
    if (!w) return;
    const float t = block_sum(acc);
    if (threadIdx.x == 0) partials[blockIdx.x] = (double)t;
}

// blocks of the first launch: at most DOT_BLOCKS, fewer where each thread then
// has one element at most (the blocks left out would add zeros)
static int setup_blocks(size_t n, size_t n_img)
{
    return (int)std::min<size_t>((std::max(n, n_img) + DOT_THREADS - 1) / DOT_THREADS, DOT_BLOCKS);
}

void launch_setup_data(const float *b, const float *w, size_t n, float *winv, float *sw, float *t_sino, float *t_img,
                       size_t n_img, double *partials, unsigned *flags, unsigned *ticket, unsigned *ticket2,
                       cudaStream_t st)
{
    counted();
    launch_kernel(k_setup_data, dim3(setup_blocks(n, n_img)), dim3(DOT_THREADS), 0, st, b, w, n, winv, sw, t_sino, t_img, n_img,
                  partials, flags, ticket, ticket2);
}

// Second: kappa = mean(1/w) (Eq. 24; low-dose) or the given one, tau, and the
// norms of the Lanczos start vectors.
__global__ void __launch_bounds__(DOT_THREADS)
k_setup_scalars(double *s, const double *partials, int np, int mode, double n, double tau, double n_views, double kappa,
                double norm_img, double norm_sino)
{
    pdl_wait();
    const float t = mode == CT_LOWDOSE ? partials_sum(partials, np) : 0.0f;
    if (threadIdx.x != 0) return;
    if (mode == CT_LOWDOSE) {
        s[S_RED0] = (double)t;
        s[S_KAPPA] = s[S_RED0] / n;
    }
    if (tau > 0.0) s[S_TAU] = tau;
    else s[S_TAU] = mode == CT_LOWDOSE ? 3.14159265358979323846 * s[S_KAPPA] / (2.0 * n_views) : 0.01;
    if (kappa > 0.0) s[S_KAPPA] = kappa;
    s[S_LN0] = norm_img;
    s[S_LN0B] = norm_sino;
    float_copies(s);
}

void launch_setup_scalars(double *scal, const double *partials, int mode, size_t n, size_t n_img, double tau,
                          int n_views, double kappa, double norm_img, double norm_sino, cudaStream_t st)
{
    counted();
    launch_kernel(k_setup_scalars, dim3(1), dim3(DOT_THREADS), 0, st, scal, partials, setup_blocks(n, n_img), mode,
                  (double)n, tau, (double)n_views, kappa, norm_img, norm_sino);
}

// Third, after the norms: sigma and lambda (thread 0), and x = p = mu = 0.
// The arrays start on 16-byte boundaries.
__global__ void __launch_bounds__(256)
k_setup_finish(double *s, double sigma, double rho, int mode, double beta, float *x, float *p0, float *p1, size_t J,
               float *mu, size_t I)
{
    const size_t tid = blockIdx.x * (size_t)blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
    if (tid == 0) {
        if (sigma > 0.0) {
            s[S_SIGMA] = sigma;
        } else {
            double bound = 1.0 / (s[S_TAU] * s[S_NADA]);
            if (mode == CT_LOWDOSE && s[S_NWDW] > 0.0) bound = fmin(bound, 2.0 / s[S_NWDW]);
            s[S_SIGMA] = rho * bound;
        }
        const double lam = mode == CT_LOWDOSE ? s[S_TAU] * beta : s[S_TAU];
        s[S_LAMBDA] = lam;
        s[S_INV8LAM] = lam > 0.0 ? 1.0 / (8.0 * lam) : 0.0;
        float_copies(s);
    }
    auto zero = [&](float *a, size_t n) {
        for (size_t i = tid; i < n / 4; i += stride)
            reinterpret_cast<float4 *>(a)[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (tid < n % 4) a[n / 4 * 4 + tid] = 0.0f;
    };
    zero(x, J);
    zero(p0, 2 * J);
    zero(p1, 2 * J);
    zero(mu, I);
}

void launch_setup_finish(double *scal, double sigma, double rho, int mode, double beta, float *x, float *p0,
                         float *p1, size_t J, float *mu, size_t I, cudaStream_t st)
{
    counted();
    k_setup_finish<<<grid_for(std::max(2 * J, I) / 4 + 1, 256), 256, 0, st>>>(scal, sigma, rho, mode, beta, x, p0, p1,
                                                                              J, mu, I);
}

// The scalars of the unrolled form: tau, sigma, lambda and -tau (the factor
// of mu_bar's adjoint) with both accumulators at zero, and in s2 the factor
// of a backprojection that adds.  (As eight launches, twice per forward and
// backward: 36 us more in 6000 at 16 x 256^2.)
__global__ void k_unrolled_scalars(double *s, double *s2, double tau, double sigma, double lam, int acc_a, int acc_b)
{
    s[S_TAU] = tau;
    s[S_SIGMA] = sigma;
    s[S_LAMBDA] = lam;
    s[S_INV8LAM] = lam > 0.0 ? 1.0 / (8.0 * lam) : 0.0;
    s[S_RED0] = -tau;
    s[acc_a] = 0.0;
    s[acc_b] = 0.0;
    float_copies(s);
    s2[S_TAU] = -1.0;
    float_copies(s2);
}

void launch_unrolled_scalars(double *scal, double *scal2, double tau, double sigma, double lam, int acc_a, int acc_b,
                             cudaStream_t st)
{
    counted();
    k_unrolled_scalars<<<1, 1, 0, st>>>(scal, scal2, tau, sigma, lam, acc_a, acc_b);
}

// One-thread scalar program: s[i0] = a0, or s[i0] += a0 s[(int)a1].
__global__ void k_scalars(double *s, int op, double a0, double a1, int i0)
{
    if (op == SC_SET) s[i0] = a0;
    else s[i0] += a0 * s[(int)a1];
    float_copies(s);
}

// Largest eigenvalue of the Lanczos tridiagonal T_k (diagonal s[base + 2j],
// off-diagonal s[base + 2j + 1]) into s[out]: multisection on the Sturm
// count of T - x I (the number of negative pivots of its LDL^T is the
// number of eigenvalues below x), 32 points per round.  The count runs in
// float on T scaled by its Gershgorin bound (backward stable: the count is
// exact for a matrix within a few float ulps of T); the result is the upper
// end of the final bracket, so it errs high.
__global__ void k_lanczos_max(double *s, int base, int k, int out)
{
    __shared__ float ta[LANCZOS_MAX], tb[LANCZOS_MAX];
    __shared__ double y[LANCZOS_MAX], inv_d[LANCZOS_MAX], da[LANCZOS_MAX], od[LANCZOS_MAX];
    pdl_wait();
    const int lane = threadIdx.x;
    for (int j = lane; j < k; j += 32) {
        da[j] = s[base + 2 * j];
        od[j] = s[base + 2 * j + 1];   // T's off-diagonal; theta I - T holds -od
        ta[j] = (float)da[j];
        tb[j] = (float)od[j];
    }
    __syncwarp();
    float glo = 0.0f, ghi = 0.0f;
    for (int j = 0; j < k; ++j) {   // Gershgorin interval
        const float rad = (j > 0 ? fabsf(tb[j - 1]) : 0.0f) + (j + 1 < k ? fabsf(tb[j]) : 0.0f);
        glo = j == 0 ? ta[j] - rad : fminf(glo, ta[j] - rad);
        ghi = j == 0 ? ta[j] + rad : fmaxf(ghi, ta[j] + rad);
    }
    const float big = fmaxf(fabsf(glo), fabsf(ghi));
    if (!(big > 0.0f)) {
        if (lane == 0) s[out] = 0.0;
        return;
    }
    const float inv = 1.0f / big;
    float lo = glo * inv, hi = ghi * inv;
    for (int round = 0; round < 8 && hi - lo > 4e-7f * fmaxf(fabsf(hi), 1e-30f); ++round) {
        const float x = lo + (hi - lo) * (float)(lane + 1) * (1.0f / 33.0f);
        int below = 0;
        float d = 1.0f;
        for (int j = 0; j < k; ++j) {
            const float b = j > 0 ? tb[j - 1] * inv : 0.0f;
            d = (ta[j] * inv - x) - (j > 0 ? b * b / d : 0.0f);
            if (d == 0.0f) d = -1e-30f;
            if (d < 0.0f) ++below;
        }
        // lowest point with all k eigenvalues below it bounds lambda_max from above
        const unsigned all = __ballot_sync(0xffffffffu, below == k);
        const int first = all ? __ffs(all) - 1 : 32;     // lanes >= first have below == k
        const float nlo = first == 0 ? lo : lo + (hi - lo) * (float)first * (1.0f / 33.0f);
        const float nhi = first == 32 ? hi : lo + (hi - lo) * (float)(first + 1) * (1.0f / 33.0f);
        lo = nlo;
        hi = fmaxf(nhi, nlo);
    }
    if (lane != 0) return;
    // theta = the upper end of the bracket; the estimate is theta + beta_k |y_k|,
    // the Ritz value plus its residual norm (y the unit eigenvector of T for
    // theta, beta_k the norm left after the last step), so that it lies above
    // lambda_max once the Ritz vector has found the top of the spectrum.
    // y by two steps of inverse iteration with theta I - T (positive definite,
    // as theta is above every eigenvalue of T): tridiagonal elimination in
    // double on this one thread.
    // One elimination serves both steps: the pivots' reciprocals are the only
    // divisions (with a division per element and step the kernel took 35 us).
    const double theta = (double)(hi * big) * (1.0 + 1e-6);
    for (int j = 0; j < k; ++j) {
        double d = theta - da[j];
        if (j > 0) d -= od[j - 1] * od[j - 1] * inv_d[j - 1];
        if (!(d > 0.0)) d = 1e-300;
        inv_d[j] = 1.0 / d;
        y[j] = 1.0;
    }
    for (int itr = 0; itr < 2; ++itr) {
        for (int j = 1; j < k; ++j) y[j] = fma(od[j - 1] * inv_d[j - 1], y[j - 1], y[j]);
        y[k - 1] *= inv_d[k - 1];
        for (int j = k - 2; j >= 0; --j) y[j] = fma(od[j], y[j + 1], y[j]) * inv_d[j];
    }
    double nrm = 0.0;
    for (int j = 0; j < k; ++j) nrm += y[j] * y[j];
    const double res = fabs(od[k - 1] * y[k - 1]) / sqrt(nrm);
    s[out] = isfinite(res) ? theta + res : theta;
}

void launch_lanczos_max(double *scal, int base, int k, int out, cudaStream_t st)
{
    counted();
    launch_kernel(k_lanczos_max, dim3(1), dim3(32), 0, st, scal, base, k, out);
}

// One half of a Lanczos step on unnormalised vectors (t_j = n_j q_j with
// n_0 = s[n0slot] and n_j = beta_{j-1} = s[base + 2j - 1]):
//   phase 0:  w = w / n_j - (n_j / n_{j-1}) t_{j-1}   (w held op(t_j));
//             alpha_j = <w, t_j> / n_j                 -> s[base + 2j]
//   phase 1:  w -= (alpha_j / n_j) t_j;  beta_j = |w|  -> s[base + 2j + 1]
// The dot is the deterministic reduction above; the last block to finish
// (ticket counter) adds the partials in block order and resets the counter.
__global__ void __launch_bounds__(DOT_THREADS)
k_lanczos_step(float *__restrict__ w, const float *__restrict__ tp, const float *__restrict__ tc, size_t n,
               double *s, int base, int n0slot, int j, int phase, double *partials, unsigned *ticket)
{
    __shared__ bool last;
    __shared__ float coef[3];
    pdl_wait();
    const float *x2 = phase == 0 ? tp : tc;
    const size_t tid = blockIdx.x * (size_t)blockDim.x + threadIdx.x, stride = (size_t)gridDim.x * blockDim.x;
    const bool vec = ((reinterpret_cast<uintptr_t>(w) | reinterpret_cast<uintptr_t>(tc) |
                       reinterpret_cast<uintptr_t>(x2)) & 15) == 0;
    const size_t n4 = vec ? n / 4 : 0;   // four elements per load
    float4 *w4 = reinterpret_cast<float4 *>(w);
    const float4 *x4 = reinterpret_cast<const float4 *>(x2), *t4 = reinterpret_cast<const float4 *>(tc);
    // the first group's loads go out before the coefficients are known
    const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    float4 a0 = zero, xa = zero, ta = zero;
    if (tid < n4) {
        a0 = w4[tid];
        xa = x4[tid];
        if (phase == 0) ta = t4[tid];
    }
    // coefficients from the double slots, once per block (FP64 is slow here)
    if (threadIdx.x == 0) {
        const float nj = (float)(j == 0 ? s[n0slot] : s[base + 2 * j - 1]);
        float c1 = 1.0f, c2 = 0.0f;
        if (phase == 0) {
            const float njm1 = (float)(j <= 1 ? s[n0slot] : s[base + 2 * j - 3]);
            c1 = nj > 0.0f ? 1.0f / nj : 0.0f;
            c2 = (j > 0 && njm1 > 0.0f) ? nj / njm1 : 0.0f;
        } else {
            c2 = nj > 0.0f ? (float)s[base + 2 * j] / nj : 0.0f;
        }
        coef[0] = c1;
        coef[1] = c2;
        coef[2] = nj;
    }
    __syncthreads();
    const float c1 = coef[0], c2 = coef[1];
    float acc = 0.0f;
    auto group = [&](float4 a, float4 x, float4 t, size_t i) {
        if (c2 == 0.0f) x = zero;   // t_{-1} is never read (it may hold anything)
        a.x = fmaf(-c2, x.x, a.x * c1);
        a.y = fmaf(-c2, x.y, a.y * c1);
        a.z = fmaf(-c2, x.z, a.z * c1);
        a.w = fmaf(-c2, x.w, a.w * c1);
        w4[i] = a;
        const float4 d = phase == 0 ? t : a;
        acc = fmaf(a.x, d.x, acc);
        acc = fmaf(a.y, d.y, acc);
        acc = fmaf(a.z, d.z, acc);
        acc = fmaf(a.w, d.w, acc);
    };
    if (tid < n4) group(a0, xa, ta, tid);
    for (size_t i = tid + stride; i < n4; i += stride) group(w4[i], x4[i], phase == 0 ? t4[i] : zero, i);
    const size_t done = n4 * 4;
    for (size_t i = done + tid; i < n; i += stride) {
        float wi = w[i] * c1;
        if (c2 != 0.0f) wi = fmaf(-c2, x2[i], wi);
        w[i] = wi;
        acc = fmaf(wi, phase == 0 ? tc[i] : wi, acc);
    }
    const float t = block_sum(acc);
    if (threadIdx.x == 0) {
        partials[blockIdx.x] = (double)t;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    const float tf = partials_sum(partials, gridDim.x);
    if (threadIdx.x == 0) {
        const float nj = coef[2];
        if (phase == 0) s[base + 2 * j] = nj > 0.0f ? (double)(tf / nj) : 0.0;
        else s[base + 2 * j + 1] = (double)sqrtf(fmaxf(tf, 0.0f));
        *ticket = 0u;
    }
}

void launch_lanczos_step(float *w, const float *tp, const float *tc, size_t n, double *scal, int base, int n0slot,
                         int j, int phase, double *partials, unsigned *ticket, cudaStream_t st)
{
    // one four-element group per thread: no block without elements, so the
    // ticket sees only as many arrivals as the vector needs (256 blocks for
    // a 512^2 image instead of the full reduction grid)
    const size_t groups = (n + 4 * (size_t)DOT_THREADS - 1) / (4 * (size_t)DOT_THREADS);
    const int blocks = (int)std::min<size_t>(std::max<size_t>(groups, 1), DOT_BLOCKS);
    counted();
    launch_kernel(k_lanczos_step, dim3(blocks), dim3(DOT_THREADS), 0, st, w, tp, tc, n, scal, base, n0slot, j, phase,
                  partials, ticket);
}

// Both halves of a Lanczos step in one launch of a thread-block cluster, for
// vectors of at most LANCZOS_FUSED elements: the halves of k_lanczos_step are
// two launches whose work (a 64^2 or 256^2 image) is far shorter than their
// launch and their ticket.  Groups of 256 threads stand in for that kernel's
// blocks, each forming the same partial (four elements a thread, the same
// trees), and every block adds all partials in that kernel's order, so the
// coefficients are the same to the bit.  Eight blocks take 32768 elements in
// one pass, the limit; on a 512^2 image they need eight and lose to the two
// launches by about 14 us a step (64^2 / 90 views, with k_lanczos_max and the
// backprojector's slice rule: 685 -> 603 us a solve).  Partials of both halves sit in the
// first block's shared memory (distributed shared memory).
constexpr int LF_THREADS = 1024;
constexpr int LF_PARTS = (int)(LANCZOS_FUSED / (4 * DOT_THREADS));   // stand-in blocks
static_assert(LANCZOS_FUSED % (4 * DOT_THREADS) == 0 && LF_PARTS <= DOT_THREADS, "one partial per thread of a group");

__global__ void __launch_bounds__(LF_THREADS)
k_lanczos_fused(float *w, const float *tp, const float *tc, size_t n, double *s, int base, int n0slot, int j)
{
    namespace cg = cooperative_groups;
    __shared__ float part[2][LF_PARTS];
    __shared__ float wsum[LF_THREADS / 32];
    __shared__ float total, coef[3];
    cg::cluster_group cl = cg::this_cluster();
    // a block may store into the first block's shared memory once that block runs: every block arrives here and
    // waits just before its first remote store, behind the loads in between
    cl.barrier_arrive();
    pdl_wait();
    const int grp = threadIdx.x >> 8, t = threadIdx.x & 255, ng = LF_THREADS / DOT_THREADS;
    const size_t n4 = n / 4, done = n4 * 4;
    const int nparts = (int)((n + 4 * (size_t)DOT_THREADS - 1) / (4 * (size_t)DOT_THREADS));
    float4 *w4 = reinterpret_cast<float4 *>(w);
    const float4 *tc4 = reinterpret_cast<const float4 *>(tc), *tp4 = reinterpret_cast<const float4 *>(tp);
    if (threadIdx.x == 0) {   // from the double slots once per block (FP64 is slow here)
        const float n0 = (float)(j == 0 ? s[n0slot] : s[base + 2 * j - 1]);
        const float nm = (float)(j <= 1 ? s[n0slot] : s[base + 2 * j - 3]);
        coef[0] = n0 > 0.0f ? 1.0f / n0 : 0.0f;
        coef[1] = (j > 0 && nm > 0.0f) ? n0 / nm : 0.0f;
        coef[2] = n0;
    }
    __syncthreads();
    float c1 = coef[0], c2 = coef[1];
    const float nj = coef[2];
    const float4 zero = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    cl.barrier_wait();
#pragma unroll 1
    for (int phase = 0; phase < 2; ++phase) {
        const float4 *x4 = phase == 0 ? tp4 : tc4;
        const float *x2 = phase == 0 ? tp : tc;
        for (int b0 = blockIdx.x * ng; b0 < nparts; b0 += gridDim.x * ng) {   // uniform over the block
            const int b = b0 + grp;
            const size_t i = (size_t)b * DOT_THREADS + t;
            float acc = 0.0f;
            if (b < nparts && i < n4) {
                float4 a = w4[i], x = x4[i];
                const float4 tt = phase == 0 ? tc4[i] : zero;
                if (c2 == 0.0f) x = zero;   // t_{-1} is never read (it may hold anything)
                a.x = fmaf(-c2, x.x, a.x * c1);
                a.y = fmaf(-c2, x.y, a.y * c1);
                a.z = fmaf(-c2, x.z, a.z * c1);
                a.w = fmaf(-c2, x.w, a.w * c1);
                w4[i] = a;
                const float4 d = phase == 0 ? tt : a;
                acc = fmaf(a.x, d.x, acc);
                acc = fmaf(a.y, d.y, acc);
                acc = fmaf(a.z, d.z, acc);
                acc = fmaf(a.w, d.w, acc);
            }
            if (b < nparts && done + i < n) {   // the last one to three elements
                float wi = w[done + i] * c1;
                if (c2 != 0.0f) wi = fmaf(-c2, x2[done + i], wi);
                w[done + i] = wi;
                acc = fmaf(wi, phase == 0 ? tc[done + i] : wi, acc);
            }
            const float v = warp_sum(acc);
            if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = v;
            __syncthreads();
            if (t == 0 && b < nparts) {
                float q = 0.0f;
#pragma unroll
                for (int k = 0; k < DOT_THREADS / 32; ++k) q += wsum[grp * (DOT_THREADS / 32) + k];
                *cl.map_shared_rank(&part[phase][b], 0) = q;
            }
            __syncthreads();
        }
        cl.sync();
        // every block adds the partials, as k_lanczos_step's last block does
        if (grp == 0) {
            float v = 0.0f;
            if (t < nparts) v += *cl.map_shared_rank(&part[phase][t], 0);
            v = warp_sum(v);
            if ((t & 31) == 0) wsum[t >> 5] = v;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            float q = 0.0f;
#pragma unroll
            for (int k = 0; k < DOT_THREADS / 32; ++k) q += wsum[k];
            total = q;
        }
        __syncthreads();
        const float tf = total;
        if (phase == 0) {
            const float alpha = nj > 0.0f ? tf / nj : 0.0f;
            c2 = nj > 0.0f ? alpha / nj : 0.0f;
            c1 = 1.0f;
            if (blockIdx.x == 0 && threadIdx.x == 0) s[base + 2 * j] = (double)alpha;
        } else if (blockIdx.x == 0 && threadIdx.x == 0) {
            s[base + 2 * j + 1] = (double)sqrtf(fmaxf(tf, 0.0f));
        }
    }
    cl.sync();   // the first block's partials outlive every read of them
}

void launch_lanczos_fused(float *w, const float *tp, const float *tc, size_t n, double *scal, int base, int n0slot,
                          int j, cudaStream_t st)
{
    const int ng = LF_THREADS / DOT_THREADS;
    const int nparts = (int)((n + 4 * (size_t)DOT_THREADS - 1) / (4 * (size_t)DOT_THREADS));
    int blocks = 1;
    while (blocks < 8 && blocks * ng < nparts) blocks *= 2;
    counted();
    launch_kernel_cluster(k_lanczos_fused, dim3(blocks), dim3(LF_THREADS), 0, st, dim3(blocks), w, tp, tc, n, scal,
                          base, n0slot, j);
}

void launch_scalars(double *scal, int op, double a0, double a1, int i0, cudaStream_t st)
{
    counted();
    k_scalars<<<1, 1, 0, st>>>(scal, op, a0, a1, i0);
}

}  // namespace ctpd
