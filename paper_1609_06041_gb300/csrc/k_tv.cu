// k_tv.cu -- prox of tau*g (Eq. 17): argmin_{x>=0} lam TV(x) + 1/2 ||x - z||^2
// by projected-gradient steps on the TV dual field p = (px, py), |p_j| <= 1:
//     x_l = max(0, z + lam div p),   p <- Pi(p + grad x_l / (8 lam)),
// then x = max(0, z + lam div p).  grad is the forward difference (zero
// across the last row/column), div = -grad^T.  lam = 0 gives max(0, z).
//
// Temporal blocking: one block owns a tile of tc x tr pixels and holds it
// with a halo of H >= steps + 1 pixels on every side.  Each step spoils one
// more ring of the halo (its outermost cells see zeros instead of their
// neighbours), so after `steps` steps the tile holds exactly what a
// whole-image iteration would give, with no grid-wide synchronisation and
// one pass over global memory per call.  p is double-buffered (p_in ->
// p_out) because neighbouring blocks read the old p in their halos.
//
// The held region is 64 columns (lane l owns columns 2l, 2l+1) by up to
// TV_ROWS rows (warp w owns the J rows from w J), so tc = 64 - 2H.  Every
// cell's z, p and x stay in registers for the whole call; left/right
// neighbours come from the adjacent lane by shuffle, vertical ones from the
// thread's own rows and, at the ends of a warp's run of rows, through shared
// memory (tv_body).  Where a forward difference does not exist (p_x on the
// last column, p_y on the last row) and just before the first column and
// row, p is zero and stays zero: the dual step's factor is 0 there, so the
// divergence needs no boundary tests, and the cells outside the image never
// reach it.
#include <algorithm>

#include "body_tv.cuh"

namespace ctpd {

int tv_max_steps() { return TV_MAX_STEPS; }

struct TvTiles {
    int tc, tr, ncb, nrb;
};

// Column tiles are as wide as the region allows; rows are split so that the
// tiles of one image about fill the GPU once (one block per SM), but no
// narrower than TV_MIN_TR rows and no taller than the region.
static TvTiles tv_tiles(int N, int steps, int n_sm, int min_tr, bool even = false, int rows = TV_ROWS)
{
    const int H = tv_halo(steps, even);
    TvTiles t;
    t.tc = 64 - 2 * H;
    t.ncb = (N + t.tc - 1) / t.tc;
    const int tr_max = rows - 2 * H;
    int nrb = std::max(1, n_sm / t.ncb);
    nrb = std::min(nrb, (N + min_tr - 1) / min_tr);
    nrb = std::max(nrb, (N + tr_max - 1) / tr_max);
    t.tr = (N + nrb - 1) / nrb;
    t.nrb = (N + t.tr - 1) / t.tr;
    return t;
}

template <bool FGP, bool TRAJ, int J>
__global__ void __launch_bounds__(TV_THREADS, 1)
k_tv(const float *__restrict__ z, const float *__restrict__ p_in, float *__restrict__ p_out,
     float *__restrict__ x, int N, int steps, int final_, int tc, int tr, const double *__restrict__ scal,
     float *__restrict__ traj)
{
    __shared__ TvPub pub;
    pdl_wait();
    tv_body<FGP, TRAJ, J>(whole_block(), blockIdx.x, blockIdx.y, blockIdx.z, gridDim.z, pub, z, p_in, p_out, x, N,
                          steps, final_, tc, tr, scal, traj);
}

void tv_tile_shape(int n, int steps, int n_sm, int min_rows, int *tc, int *tr, int *ncb, int *nrb, int rows)
{
    const TvTiles t = tv_tiles(n, steps, std::max(1, n_sm), min_rows > 0 ? min_rows : TV_MIN_TR, false,
                               rows > 0 ? rows : TV_ROWS);
    *tc = t.tc;
    *tr = t.tr;
    *ncb = t.ncb;
    *nrb = t.nrb;
}

void launch_tv(const float *z, const float *p_in, float *p_out, float *x,
               int n, int n_sm, int min_rows, int steps, int final_, const double *scal, cudaStream_t st, bool fgp,
               int batch, float *traj)
{
    // a batch fills the GPU with its images: the tiles of one image only
    // need to cover n_sm / batch SMs
    const TvTiles t = tv_tiles(n, steps, std::max(1, n_sm / std::max(1, batch)), min_rows > 0 ? min_rows : TV_MIN_TR,
                               traj != nullptr);
    const dim3 grid(t.ncb, t.nrb, std::max(1, batch));
    counted();
    // rows per warp: as few as hold the region, so that all 16 warps carry a share of it
    const int rows = t.tr + 2 * tv_halo(steps, traj != nullptr);
    auto pick = [&](auto k1, auto k2, auto k3, auto k4, auto k5) {
        return rows <= TV_WARPS ? k1 : rows <= 2 * TV_WARPS ? k2 : rows <= 3 * TV_WARPS ? k3 : rows <= 4 * TV_WARPS ? k4 : k5;
    };
    auto kern = traj  ? pick(k_tv<false, true, 1>, k_tv<false, true, 2>, k_tv<false, true, 3>, k_tv<false, true, 4>,
                             k_tv<false, true, 5>)
                : fgp ? pick(k_tv<true, false, 1>, k_tv<true, false, 2>, k_tv<true, false, 3>, k_tv<true, false, 4>,
                             k_tv<true, false, 5>)
                      : pick(k_tv<false, false, 1>, k_tv<false, false, 2>, k_tv<false, false, 3>, k_tv<false, false, 4>,
                             k_tv<false, false, 5>);
    launch_kernel(kern, grid, dim3(TV_THREADS), 0, st, z, p_in, p_out, x, n, steps, final_, t.tc, t.tr, scal, traj);
}



// =====================================================================
// Whole-image single steps of the same projected-gradient iteration, and
// their adjoints, for the differentiable unrolled solve.  One thread per
// pixel, blockIdx.z = image of a batch; p = (px, py) stored as two N x N
// planes.  The adjoints use div = -grad^T, the mask of max(0, .), and the
// Jacobian of the unit-ball projection Pi(q) = q / max(1, |q|), which is I
// inside the ball and (I - qhat qhat^T) / |q| outside it.
// =====================================================================
namespace {

__device__ __forceinline__ float tv_div(const float *px, const float *py, int r, int c, int N)
{
    const size_t j = (size_t)r * N + c;
    return ((c < N - 1 ? px[j] : 0.0f) - (c > 0 ? px[j - 1] : 0.0f)) +
           ((r < N - 1 ? py[j] : 0.0f) - (r > 0 ? py[j - N] : 0.0f));
}

// s = z + lam div p (before the max(0, .))
__device__ __forceinline__ float tv_s(const float *z, const float *px, const float *py, int r, int c, int N, float lam)
{
    return z[(size_t)r * N + c] + lam * tv_div(px, py, r, c, N);
}

// q = p + inv8 grad max(0, s) at (r, c)
__device__ __forceinline__ float2 tv_q(const float *z, const float *px, const float *py, int r, int c, int N,
                                       float lam, float inv8)
{
    const size_t j = (size_t)r * N + c;
    const float x0 = fmaxf(0.0f, tv_s(z, px, py, r, c, N, lam));
    const float gx = c < N - 1 ? fmaxf(0.0f, tv_s(z, px, py, r, c + 1, N, lam)) - x0 : 0.0f;
    const float gy = r < N - 1 ? fmaxf(0.0f, tv_s(z, px, py, r + 1, c, N, lam)) - x0 : 0.0f;
    return make_float2(px[j] + gx * inv8, py[j] + gy * inv8);
}

// J_Pi(q)^T g
__device__ __forceinline__ float2 proj_adj(float2 q, float2 g)
{
    const float n2 = fmaf(q.x, q.x, q.y * q.y);
    const float inv = rsqrtf(n2);
    const float hx = q.x * inv, hy = q.y * inv;
    const float d = hx * g.x + hy * g.y;
    return n2 <= 1.0f ? g : make_float2((g.x - hx * d) * inv, (g.y - hy * d) * inv);
}

// Block sums of the per-thread float terms va, vb: a fixed shuffle tree per
// warp, then the block's warp sums in order (compensated FP32, FSum) into
// part[2 block], part[2 block + 1].  launch_pair_sums adds the partials of
// many launches at the end.  Blocks of 256 threads.
__device__ __forceinline__ void block_pair_to(float va, float vb, float *part)
{
    __shared__ float wa[8], wb[8];
    const int t = threadIdx.y * blockDim.x + threadIdx.x;
    const size_t blk = ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        va += __shfl_down_sync(0xffffffffu, va, o);
        vb += __shfl_down_sync(0xffffffffu, vb, o);
    }
    if ((t & 31) == 0) {
        wa[t >> 5] = va;
        wb[t >> 5] = vb;
    }
    __syncthreads();
    if (t == 0) {
        FSum sa{0.0f, 0.0f}, sb{0.0f, 0.0f};
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            fsum_add(sa, wa[k]);
            fsum_add(sb, wb[k]);
        }
        part[2 * blk] = sa.s + sa.c;
        part[2 * blk + 1] = sb.s + sb.c;
    }
}

}  // namespace

// p_out = Pi(p_in + inv8 grad max(0, z + lam div p_in))
__global__ void __launch_bounds__(256)
k_tv_step(const float *__restrict__ z, const float *__restrict__ p_in, float *__restrict__ p_out, int N,
          const double *__restrict__ scal)
{
    const int c = blockIdx.x * 32 + threadIdx.x, r = blockIdx.y * 8 + threadIdx.y;
    if (r >= N || c >= N) return;
    const size_t NN = (size_t)N * N, j = (size_t)r * N + c;
    const float *zz = z + blockIdx.z * NN;
    const float *px = p_in + blockIdx.z * 2 * NN, *py = px + NN;
    float *ox = p_out + blockIdx.z * 2 * NN, *oy = ox + NN;
    const float lam = fscal(scal, F_LAMBDA), inv8 = fscal(scal, F_INV8LAM);
    const float2 q = tv_q(zz, px, py, r, c, N, lam, inv8);
    const float sc = fminf(1.0f, rsqrtf(fmaf(q.x, q.x, q.y * q.y)));
    ox[j] = q.x * sc;
    oy[j] = q.y * sc;
}

// x = max(0, z + lam div p)
__global__ void __launch_bounds__(256)
k_tv_final(const float *__restrict__ z, const float *__restrict__ p, float *__restrict__ x, int N,
           const double *__restrict__ scal)
{
    const int c = blockIdx.x * 32 + threadIdx.x, r = blockIdx.y * 8 + threadIdx.y;
    if (r >= N || c >= N) return;
    const size_t NN = (size_t)N * N;
    const float *px = p + blockIdx.z * 2 * NN, *py = px + NN;
    x[blockIdx.z * NN + (size_t)r * N + c] =
        fmaxf(0.0f, tv_s(z + blockIdx.z * NN, px, py, r, c, N, fscal(scal, F_LAMBDA)));
}

// Adjoint of x = max(0, s), s = z + lam div p, with the adjoint gp_next of p
// flowing in from later: gs = gx [s > 0]; gz = gs; gp = gp_next - lam grad gs;
// partial sums of <gs, div p> (the lam derivative).
__global__ void __launch_bounds__(256)
k_tv_final_bwd(const float *__restrict__ z, const float *__restrict__ p, const float *__restrict__ gx,
               const float *__restrict__ gp_next, float *__restrict__ gz, float *__restrict__ gp, int N,
               const double *__restrict__ scal, float *__restrict__ part)
{
    const int c = blockIdx.x * 32 + threadIdx.x, r = blockIdx.y * 8 + threadIdx.y;
    float contrib = 0.0f;
    if (r < N && c < N) {
        const size_t NN = (size_t)N * N, j = (size_t)r * N + c;
        const float *zz = z + blockIdx.z * NN, *g = gx + blockIdx.z * NN;
        const float *px = p + blockIdx.z * 2 * NN, *py = px + NN;
        const float lam = fscal(scal, F_LAMBDA);
        auto gs_at = [&](int rr, int cc) {
            return tv_s(zz, px, py, rr, cc, N, lam) > 0.0f ? g[(size_t)rr * N + cc] : 0.0f;
        };
        const float gs0 = gs_at(r, c);
        const float gsr = c < N - 1 ? gs_at(r, c + 1) : 0.0f;
        const float gsd = r < N - 1 ? gs_at(r + 1, c) : 0.0f;
        gz[blockIdx.z * NN + j] = gs0;
        const float *gnx = gp_next + blockIdx.z * 2 * NN, *gny = gnx + NN;
        float *ox = gp + blockIdx.z * 2 * NN, *oy = ox + NN;
        ox[j] = gnx[j] - lam * (c < N - 1 ? gsr - gs0 : 0.0f);
        oy[j] = gny[j] - lam * (r < N - 1 ? gsd - gs0 : 0.0f);
        contrib = gs0 * tv_div(px, py, r, c, N);
    }
    block_pair_to(0.0f, contrib, part);
}

// Adjoint of one step p' = Pi(q), q = p + inv8 grad x, x = max(0, s),
// s = z + lam div p, with the adjoint gp_next of p' flowing in from later:
//   gq = J_Pi(q)^T gp_next;   gx = -inv8 div gq;   gs = gx [s > 0];
//   gz += gs;   gp = gq - lam grad gs;
// and the derivative terms <gq, grad x> (for inv8) and <gs, div p> (for
// lam).
//
// Several steps run per launch, temporally blocked as the prox itself
// (body_tv.cuh): a block holds a region of 64 columns by 16 J rows, lane l
// the columns 2l and 2l + 1, warp w the J rows from w J, with z, gz and gp in
// registers; its interior is the region minus a halo of steps + 1 (rounded up
// to even) on every side.  A step reads its p from shared memory, copied there
// by cp.async while the step before it computes; it publishes gq_y of a
// warp's last row (for gs below) and gs of its first row (for gp above), with
// a barrier after each.  One step per launch staged every field with halos
// and read and wrote the adjoints each time: 17.7 us a step on 16 x 256^2; five
// steps take 48 us, bound by their instructions (64 % of the issue slots, 16
// warps an SM).  Both forms of a warp's cells (border tests or none), no masks
// on cells whose values go nowhere, and a branch-free projection adjoint took
// the five steps there from 60 us.
constexpr int TVB_J = 4;       // most region rows per warp: 5 spill
constexpr int TVB_STEPS = 5;   // most steps per launch: halo 6, 52 interior columns
__host__ __device__ __forceinline__ int tvb_halo(int steps) { return (steps + 2) & ~1; }
struct TvbPub {
    float2 gqy[TV_WARPS + 1][32];   // gq_y of warp w - 1's last row; entry 0: zeros
    float2 gs[TV_WARPS + 1][32];    // gs of warp w's first row; the last entry: zeros
};
template <int J>
constexpr size_t tvb_smem() { return sizeof(TvbPub) + sizeof(float) * 2 * 2 * TV_WARPS * J * 64; }

// p0: p before the prox's first step (l = 0); traj: p before step l at traj +
// (l - 1) tstride.  Runs the adjoints of steps l_hi, l_hi - 1, .., l_hi - steps + 1.
template <int J>
__global__ void __launch_bounds__(TV_THREADS, 1)
k_tv_bwd(const float *__restrict__ z, const float *__restrict__ p0, const float *__restrict__ traj, size_t tstride,
         int l_hi, int steps, const float *__restrict__ gp_next, float *__restrict__ gz, float *__restrict__ gp, int N,
         int tc, int tr, const double *__restrict__ scal, float *__restrict__ part)
{
    extern __shared__ __align__(16) unsigned char tvsm[];
    TvbPub &pub = *reinterpret_cast<TvbPub *>(tvsm);
    float *P = reinterpret_cast<float *>(tvsm + sizeof(TvbPub));   // [buffer][x, y][row][column]
    constexpr int ROWS = TV_WARPS * J;
    constexpr unsigned FULL = 0xffffffffu;
    pdl_wait();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int H = tvb_halo(steps), Sr = tr + 2 * H;
    const int R0 = blockIdx.y * tr - H, C0 = blockIdx.x * tc - H, c0 = C0 + 2 * lane, l0 = w * J;
    const size_t NN = (size_t)N * N;
    z += blockIdx.z * NN;
    gz += blockIdx.z * NN;
    gp_next += blockIdx.z * 2 * NN;
    gp += blockIdx.z * 2 * NN;
    const float lam = fscal(scal, F_LAMBDA), inv8 = fscal(scal, F_INV8LAM);
    bool in[2], lt[2], gt[2], own[2];   // columns: inside, before the last, after the first, interior of the tile
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int c = c0 + e, lj = 2 * lane + e;
        in[e] = (unsigned)c < (unsigned)N;
        lt[e] = c < N - 1;
        gt[e] = c > 0;
        own[e] = in[e] && lj >= H && lj < H + tc;
    }
    auto row_in = [&](int li) { return li < Sr && (unsigned)(R0 + li) < (unsigned)N; };

    // the region's p before step l into buffer b (zeros outside the image)
    auto fetch = [&](int l, int b) {
        const float *src = (l == 0 ? p0 : traj + (size_t)(l - 1) * tstride) + blockIdx.z * 2 * NN;
#pragma unroll
        for (int j = 0; j < J; ++j) {
            const int li = l0 + j;
            const size_t gi = (size_t)(R0 + li) * N + c0;
            const bool ok = row_in(li);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                float *dst = P + ((b * 2 + k) * ROWS + li) * 64 + 2 * lane;
                const float *sp = src + k * NN;
                const unsigned sd = (unsigned)__cvta_generic_to_shared(dst);
                if ((N & 1) == 0) {   // C0 is even: an aligned pair, inside or outside as a whole
                    const int n = ok && in[0] ? 8 : 0;
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(sd), "l"(n ? sp + gi : src), "r"(n)
                                 : "memory");
                } else {
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int n = ok && in[e] ? 4 : 0;
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(sd + 4 * e),
                                     "l"(n ? sp + gi + e : src), "r"(n)
                                     : "memory");
                    }
                }
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    fetch(l_hi, 0);
    for (int i = threadIdx.x; i < (int)(sizeof(TvbPub) / sizeof(float2)); i += TV_THREADS)
        reinterpret_cast<float2 *>(tvsm)[i] = make_float2(0.0f, 0.0f);

    float zr[J + 1][2], gzr[J][2], gx[J][2], gy[J][2];   // gx, gy: the adjoint field gp
#pragma unroll
    for (int j = 0; j <= J; ++j) {
        const int li = l0 + j;
        const bool rin = row_in(li), rown = li >= H && li < H + tr;
        const size_t gi = (size_t)(R0 + li) * N + c0;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            zr[j][e] = rin && in[e] ? z[gi + e] : 0.0f;
            if (j < J) {
                gx[j < J ? j : 0][e] = rin && in[e] ? gp_next[gi + e] : 0.0f;
                gy[j < J ? j : 0][e] = rin && in[e] ? gp_next[NN + gi + e] : 0.0f;
                gzr[j < J ? j : 0][e] = rin && rown && own[e] ? gz[gi + e] : 0.0f;
            }
        }
    }
    FSum si[2], sl[2];   // <gq, grad x>, <gs, div p> of a column
    si[0] = si[1] = sl[0] = sl[1] = FSum{0.0f, 0.0f};
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();
    const bool busy = l0 < Sr;
    // No value of a cell outside the image, or beyond the region's good part,
    // reaches an interior cell: its differences across the border are dropped
    // and the halo takes the rest, so only the sums and the stores ask whether
    // a cell is the tile's own.  Warps whose cells all have four neighbours in
    // the image take the form without the border's tests.
    const bool inner = C0 >= 1 && C0 + 64 < N && R0 + l0 >= 1 && R0 + l0 + J < N - 1;
    for (int st = 0; st < steps; ++st) {
        const int b = st & 1;
        if (st + 1 < steps) fetch(l_hi - st - 1, b ^ 1);
        const float *PX = P + (b * 2) * ROWS * 64 + 2 * lane, *PY = PX + ROWS * 64;
        float s[J + 1][2], dv[J][2], qx[J][2], qy[J][2], gs[J][2];
        float ti[2] = {0.0f, 0.0f}, tl[2] = {0.0f, 0.0f};
        auto first = [&](auto form) {   // s and gq
            constexpr bool INT = decltype(form)::value;
            const bool lt0 = INT || lt[0], lt1 = INT || lt[1], gt0 = INT || gt[0];
            float2 pu = l0 > 0 ? *reinterpret_cast<const float2 *>(PY + (l0 - 1) * 64) : make_float2(0.0f, 0.0f);
            float px[J][2], py[J][2];
#pragma unroll
            for (int j = 0; j <= J; ++j) {   // s = z + lam div p, the run and the row below it
                const int li = l0 + j, a = R0 + li;
                const bool rlt = INT || a < N - 1, rgt = INT || a > 0;
                float2 vx = make_float2(0.0f, 0.0f), vy = vx;
                if (j < J || li < ROWS) {
                    vx = *reinterpret_cast<const float2 *>(PX + li * 64);
                    vy = *reinterpret_cast<const float2 *>(PY + li * 64);
                }
                const float left = __shfl_up_sync(FULL, vx.y, 1);
                const float d0 = ((lt0 ? vx.x : 0.0f) - (gt0 ? left : 0.0f)) + ((rlt ? vy.x : 0.0f) - (rgt ? pu.x : 0.0f));
                const float d1 = ((lt1 ? vx.y : 0.0f) - vx.x) + ((rlt ? vy.y : 0.0f) - (rgt ? pu.y : 0.0f));
                s[j][0] = fmaf(lam, d0, zr[j][0]);
                s[j][1] = fmaf(lam, d1, zr[j][1]);
                if (j < J) {
                    const int jj = j < J ? j : 0;
                    px[jj][0] = vx.x;
                    px[jj][1] = vx.y;
                    py[jj][0] = vy.x;
                    py[jj][1] = vy.y;
                    dv[jj][0] = d0;
                    dv[jj][1] = d1;
                }
                pu = vy;
            }
#pragma unroll
            for (int j = 0; j < J; ++j) {   // gq = J_Pi(q)^T gp_next
                const int li = l0 + j;
                const bool rlt = INT || R0 + li < N - 1;
                const float right = __shfl_down_sync(FULL, s[j][0], 1);
                const bool rown = li >= H && li < H + tr;
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float x0 = fmaxf(0.0f, s[j][e]), sr = e == 0 ? s[j][1] : right;
                    const float gxv = (e == 0 ? lt0 : lt1) ? fmaxf(0.0f, sr) - x0 : 0.0f;
                    const float gyv = rlt ? fmaxf(0.0f, s[j + 1][e]) - x0 : 0.0f;
                    const float2 q = make_float2(px[j][e] + gxv * inv8, py[j][e] + gyv * inv8);
                    const float2 g = proj_adj(q, make_float2(gx[j][e], gy[j][e]));
                    qx[j][e] = g.x;
                    qy[j][e] = g.y;
                    if (rown) ti[e] = fmaf(g.x, gxv, fmaf(g.y, gyv, ti[e]));
                }
            }
            pub.gqy[w + 1][lane] = make_float2(qy[J - 1][0], qy[J - 1][1]);
        };
        auto second = [&](auto form) {   // gs
            constexpr bool INT = decltype(form)::value;
            const bool lt0 = INT || lt[0], lt1 = INT || lt[1], gt0 = INT || gt[0];
            float2 qu = pub.gqy[w][lane];
#pragma unroll
            for (int j = 0; j < J; ++j) {   // gs = [s > 0] (-inv8 div gq)
                const int li = l0 + j, a = R0 + li;
                const bool rlt = INT || a < N - 1, rgt = INT || a > 0, rown = li >= H && li < H + tr;
                const float left = __shfl_up_sync(FULL, qx[j][1], 1);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float ql = e == 0 ? left : qx[j][0], qup = e == 0 ? qu.x : qu.y;
                    const float d = (((e == 0 ? lt0 : lt1) ? qx[j][e] : 0.0f) - ((e == 1 || gt0) ? ql : 0.0f)) +
                                    ((rlt ? qy[j][e] : 0.0f) - (rgt ? qup : 0.0f));
                    const float v = s[j][e] > 0.0f ? -inv8 * d : 0.0f;
                    gs[j][e] = v;
                    gzr[j][e] = gzr[j][e] + v;
                    if (rown) tl[e] = fmaf(v, dv[j][e], tl[e]);
                }
                qu = make_float2(qy[j][0], qy[j][1]);
            }
            pub.gs[w][lane] = make_float2(gs[0][0], gs[0][1]);
        };
        auto third = [&](auto form) {   // gp
            constexpr bool INT = decltype(form)::value;
            const bool lt0 = INT || lt[0], lt1 = INT || lt[1];
            const float2 dn = pub.gs[w + 1][lane];
#pragma unroll
            for (int j = 0; j < J; ++j) {   // gp = gq - lam grad gs
                const bool rlt = INT || R0 + l0 + j < N - 1;
                const float right = __shfl_down_sync(FULL, gs[j][0], 1);
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float g0 = gs[j][e], gr = e == 0 ? gs[j][1] : right;
                    const float gd = j + 1 < J ? gs[j + 1 < J ? j + 1 : 0][e] : (e == 0 ? dn.x : dn.y);
                    gx[j][e] = qx[j][e] - lam * ((e == 0 ? lt0 : lt1) ? gr - g0 : 0.0f);
                    gy[j][e] = qy[j][e] - lam * (rlt ? gd - g0 : 0.0f);
                }
            }
        };
        constexpr std::true_type yes{};
        constexpr std::false_type no{};
        if (busy) inner ? first(yes) : first(no);
        __syncthreads();
        if (busy) inner ? second(yes) : second(no);
        asm volatile("cp.async.wait_group 0;" ::: "memory");   // the next step's p
        __syncthreads();
        if (busy) inner ? third(yes) : third(no);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            fsum_add(si[e], ti[e]);
            fsum_add(sl[e], tl[e]);
        }
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
        const int li = l0 + j;
        if (li >= H && li < H + tr && row_in(li)) {
            const size_t gi = (size_t)(R0 + li) * N + c0;
#pragma unroll
            for (int e = 0; e < 2; ++e)
                if (own[e]) {
                    gz[gi + e] = gzr[j][e];
                    gp[gi + e] = gx[j][e];
                    gp[NN + gi + e] = gy[j][e];
                }
        }
    }
    // block sums of the derivative terms: a fixed shuffle tree per warp, then the warps in order
    float va = 0.0f, vb = 0.0f;
#pragma unroll
    for (int e = 0; e < 2; ++e)
        if (own[e]) {
            va += si[e].s + si[e].c;
            vb += sl[e].s + sl[e].c;
        }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        va += __shfl_down_sync(FULL, va, o);
        vb += __shfl_down_sync(FULL, vb, o);
    }
    float2 *red = &pub.gqy[0][0];   // read by every warp before the last barrier
    if (lane == 0) red[w] = make_float2(va, vb);
    __syncthreads();
    if (threadIdx.x == 0) {
        FSum ta{0.0f, 0.0f}, tb{0.0f, 0.0f};
        for (int k = 0; k < TV_WARPS; ++k) {
            fsum_add(ta, red[k].x);
            fsum_add(tb, red[k].y);
        }
        const size_t blk = ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
        part[2 * blk] = ta.s + ta.c;
        part[2 * blk + 1] = tb.s + tb.c;
    }
}

namespace {
dim3 tv_px_grid(int n, int batch) { return dim3((n + 31) / 32, (n + 7) / 8, batch); }
}

// partials (two floats per block) of the adjoint kernels: the final step's grid, the larger one (its blocks hold 32 x
// 8 pixels, k_tv_bwd's at least 34 x 8)
size_t tv_px_blocks(int n, int batch)
{
    return 2 * (size_t)((n + 31) / 32) * ((n + 7) / 8) * batch;
}

void launch_tv_step(const float *z, const float *p_in, float *p_out, int n, int batch, const double *scal,
                    cudaStream_t st)
{
    counted();
    k_tv_step<<<tv_px_grid(n, batch), dim3(32, 8), 0, st>>>(z, p_in, p_out, n, scal);
}

void launch_tv_final(const float *z, const float *p, float *x, int n, int batch, const double *scal, cudaStream_t st)
{
    counted();
    k_tv_final<<<tv_px_grid(n, batch), dim3(32, 8), 0, st>>>(z, p, x, n, scal);
}

void launch_tv_final_bwd(const float *z, const float *p, const float *gx, const float *gp_next, float *gz,
                         float *gp, int n, int batch, const double *scal, float *part, cudaStream_t st)
{
    counted();
    k_tv_final_bwd<<<tv_px_grid(n, batch), dim3(32, 8), 0, st>>>(z, p, gx, gp_next, gz, gp, n, scal, part);
}

int tv_bwd_max_steps() { return TVB_STEPS; }

void launch_tv_bwd(const float *z, const float *p0, const float *traj, size_t tstride, int l_hi, int steps,
                   const float *gp_next, float *gz, float *gp, int n, int n_sm, int batch, const double *scal,
                   float *part, cudaStream_t st)
{
    // row tiles by the least rows per warp times waves of blocks (one block an SM);
    // the row below the run is computed too, hence j + 1
    const int H = tvb_halo(steps), tc = 64 - 2 * H, ncb = (n + tc - 1) / tc;
    int best_j = 0, best_tr = 0;
    long best = -1;
    for (int j = 2; j <= TVB_J; ++j) {
        const int most = TV_WARPS * j - 2 * H;
        if (most < 8) continue;
        const int nrb = (n + most - 1) / most, tr = (n + nrb - 1) / nrb;
        const long blocks = (long)ncb * nrb * batch, cost = (blocks + n_sm - 1) / n_sm * (j + 1);
        if (best < 0 || cost < best) {
            best = cost;
            best_j = j;
            best_tr = std::max(tr, 8);
        }
    }
    const dim3 grid(ncb, (n + best_tr - 1) / best_tr, batch);
    counted();
    auto go = [&](auto kern, size_t smem) {
        launch_kernel(kern, grid, dim3(TV_THREADS), smem, st, z, p0, traj, tstride, l_hi, steps, gp_next, gz, gp, n, tc,
                      best_tr, scal, part);
    };
    if (best_j == 2) go(k_tv_bwd<2>, tvb_smem<2>());
    else if (best_j == 3) go(k_tv_bwd<3>, tvb_smem<3>());
    else go(k_tv_bwd<4>, tvb_smem<4>());
}

// scal[slot_a] += sum of part[2 i], scal[slot_b] += sum of part[2 i + 1],
// i < npairs, in a fixed order and compensated FP32: PS_BLOCKS blocks add
// contiguous runs, one warp adds their results; the one thread then adds
// the two totals to the double slots.
constexpr int PS_BLOCKS = 152;

__global__ void __launch_bounds__(256) k_pair_sums(const float *__restrict__ part, size_t npairs, float *out)
{
    const size_t per = (npairs + gridDim.x - 1) / gridDim.x, lo = blockIdx.x * per;
    const size_t hi = lo + per < npairs ? lo + per : npairs;
    FSum a{0.0f, 0.0f}, b{0.0f, 0.0f};
    for (size_t i = lo + threadIdx.x; i < hi; i += 256) {
        const float2 v = reinterpret_cast<const float2 *>(part)[i];
        fsum_add(a, v.x);
        fsum_add(b, v.y);
    }
    __shared__ FSum ra[256], rb[256];
    ra[threadIdx.x] = a;
    rb[threadIdx.x] = b;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            fsum_merge(ra[threadIdx.x], ra[threadIdx.x + o]);
            fsum_merge(rb[threadIdx.x], rb[threadIdx.x + o]);
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[4 * blockIdx.x] = ra[0].s;
        out[4 * blockIdx.x + 1] = ra[0].c;
        out[4 * blockIdx.x + 2] = rb[0].s;
        out[4 * blockIdx.x + 3] = rb[0].c;
    }
}

// one warp: strided lanes, then a fixed shuffle tree
__global__ void k_pair_final(const float *__restrict__ r, int nb, double *scal, int slot_a, int slot_b)
{
    FSum a{0.0f, 0.0f}, b{0.0f, 0.0f};
    for (int i = threadIdx.x; i < nb; i += 32) {
        fsum_merge(a, FSum{r[4 * i], r[4 * i + 1]});
        fsum_merge(b, FSum{r[4 * i + 2], r[4 * i + 3]});
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        fsum_merge(a, FSum{__shfl_down_sync(0xffffffffu, a.s, o), __shfl_down_sync(0xffffffffu, a.c, o)});
        fsum_merge(b, FSum{__shfl_down_sync(0xffffffffu, b.s, o), __shfl_down_sync(0xffffffffu, b.c, o)});
    }
    if (threadIdx.x == 0) {
        scal[slot_a] += (double)a.s + (double)a.c;
        scal[slot_b] += (double)b.s + (double)b.c;
    }
}

size_t pair_sums_scratch_floats() { return 4 * PS_BLOCKS; }

void launch_pair_sums(const float *part, size_t npairs, float *scratch, double *scal, int slot_a, int slot_b,
                      cudaStream_t st)
{
    counted(2);
    k_pair_sums<<<PS_BLOCKS, 256, 0, st>>>(part, npairs, scratch);
    k_pair_final<<<1, 32, 0, st>>>(scratch, PS_BLOCKS, scal, slot_a, slot_b);
}

void kernel_attrs_tv()
{
    cudaFuncSetAttribute(k_tv_bwd<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tvb_smem<2>());
    cudaFuncSetAttribute(k_tv_bwd<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tvb_smem<3>());
    cudaFuncSetAttribute(k_tv_bwd<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tvb_smem<4>());
}

}  // namespace ctpd
