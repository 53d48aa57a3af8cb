// k_joseph.cu -- Joseph forward projector A (ray-driven) and its transpose
// A^T (pixel-driven gather), the A and A^T of Eqs. 18-20 / 29-31.  Both are
// deterministic (fixed summation orders, no atomics).
#include <algorithm>
#include <cmath>
#include <mutex>
#include <new>
#include <type_traits>
#include <vector>

#include <cooperative_groups.h>

#include "body_joseph.cuh"

namespace ctpd {


// =====================================================================
// Forward projection without mirrors: images of over about 1800 pixels a
// side (a mirrored band pair does not fit in shared memory) and the unrolled
// form on sides that are not a multiple of 32.
// A block owns a band of PROJ_R consecutive steps (rows for row-stepping
// views, columns for column-stepping views) and a group of PG views of one
// class.  It stages the band in shared memory as interpolation pairs
//     P[i] = ((x[i] + x[i+1]) / 2, x[i+1] - x[i]),  i = -2 .. N (zero padded),
// so one sample is fma(g, P.y, P.x) = (1/2 - g) x[i0] + (1/2 + g) x[i0+1].
// Each thread walks whole rays across the band and writes the band's
// partial ray sum; launch_band_reduce adds the bands in a fixed order.
// Images wider than one staged row (PROJ_CW pairs) are staged in several
// column passes; a sample is taken in the pass that holds its pair and the
// pass sums are added to the partial in pass order.
// =====================================================================
constexpr int PT = 1024;       // threads per block
constexpr int PROJ_CW = 640;   // pairs per staged band row

static int proj_cw(int n) { return (n + 3) < PROJ_CW ? (n + 3) : PROJ_CW; }
static int proj_stride(int n) { return proj_cw(n) | 1; }   // odd: spreads smem banks
constexpr int QUAD_SMEM_MAX = 227 * 1024;   // shared memory a block may have
static size_t proj_smem(int n) { return sizeof(float2) * (size_t)PROJ_R * proj_stride(n) + sizeof(ViewP) * PG + 64; }

__device__ __forceinline__ int d_proj_cw(int n) { return (n + 3) < PROJ_CW ? (n + 3) : PROJ_CW; }

template <bool MULTI>
__global__ void __launch_bounds__(PT)
k_project_bands(const float *__restrict__ x, const ViewP *__restrict__ views,
                const int *__restrict__ row_list, int n_row, const int *__restrict__ col_list, int n_col,
                int N, int V, int B, float *__restrict__ partial)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    const int CW = d_proj_cw(N), SP = CW | 1;
    float2 *P = reinterpret_cast<float2 *>(smraw);
    ViewP *sv = reinterpret_cast<ViewP *>(P + (size_t)PROJ_R * SP);
    int *svi = reinterpret_cast<int *>(sv + PG);

    const int band = blockIdx.x, nb = gridDim.x;
    const int row_groups = (n_row + PG - 1) / PG;
    const bool rows = (int)blockIdx.y < row_groups;
    const int grp = rows ? blockIdx.y : blockIdx.y - row_groups;
    const int *list = rows ? row_list : col_list;
    const int nl = rows ? n_row : n_col;
    const int nv = min(PG, nl - grp * PG);
    const float *img = x + (size_t)blockIdx.z * N * N;
    float *out = partial + ((size_t)blockIdx.z * nb + band) * V * B;
    const int s0 = band * PROJ_R, ns = min(PROJ_R, N - s0);
    const float h = joseph_h(N), hq = joseph_hq(N);
    const int tid = threadIdx.x;

    if (tid < nv) {
        svi[tid] = list[grp * PG + tid];
        sv[tid] = views[svi[tid]];
    }
    for (int I0 = -2; I0 <= N; I0 += CW) {
        const int I1 = min(I0 + CW, N + 1);   // this pass holds pairs I0 .. I1-1
        const int w = I1 - I0;
        __syncthreads();
        if (rows) {
            for (int k = tid; k < ns * w; k += PT) {
                const int si = k / w, i = I0 + (k - si * w);
                const float *rowp = img + (size_t)(s0 + si) * N;
                const float a = (i >= 0 && i < N) ? rowp[i] : 0.0f;
                const float b = (i + 1 >= 0 && i + 1 < N) ? rowp[i + 1] : 0.0f;
                P[si * SP + (i - I0)] = make_float2(0.5f * (a + b), b - a);
            }
        } else {
            // column band: pair i of step (column) c = s0 + si is (x[i][c], x[i+1][c]);
            // neighbouring threads take neighbouring columns (coalesced rows)
            for (int k = tid; k < ns * w; k += PT) {
                const int ii = k / ns, si = k - ii * ns, i = I0 + ii, c = s0 + si;
                const float a = (i >= 0 && i < N) ? img[(size_t)i * N + c] : 0.0f;
                const float b = (i + 1 >= 0 && i + 1 < N) ? img[(size_t)(i + 1) * N + c] : 0.0f;
                P[si * SP + ii] = make_float2(0.5f * (a + b), b - a);
            }
        }
        __syncthreads();
        // samples with non-zero weight have u' in (-1.5, N - 0.5); this pass
        // takes those with round(u') in [I0, I1)
        const float ulo = (float)max(I0, -1) - 1.5f, uhi = (float)min(I1, N) + 0.5f;
        for (int slot = tid; slot < nv * B; slot += PT) {
            const int vi = slot / B, d = slot - vi * B;
            const float a = sv[vi].a, m = sv[vi].m, inv_m = sv[vi].inv_m;
            const float q = joseph_q(joseph_dp(d, B), a, hq);
            int lo, hi;
            step_range(q, m, inv_m, h, ulo, uhi, s0, s0 + ns - 1, lo, hi);
            const float sp = (float)lo - h;
            int ridx = (lo - s0) * SP;                 // pair array offset of step lo
            float acc0 = 0.0f, acc1 = 0.0f, acc2 = 0.0f, acc3 = 0.0f;
            if (!MULTI) {
                // steps lo, lo+1, ... as u'(s) = sp_k m + q with sp_k = (s - h) exact;
                // the pair index i0 + 2 is clamped to [0, N + 2] (both ends are zero pairs)
                const unsigned top = (unsigned)(N + 2);
                // q_u = q + u m: u'(s + u) = (s - h) m + q_u
                const float qu1 = __fadd_rn(q, m), qu2 = __fmaf_rn(2.0f, m, q), qu3 = __fmaf_rn(3.0f, m, q);
                float spk = sp;
                int s = lo;
                for (; s + 3 <= hi; s += 4) {
                    float2 pr[4];
                    float gg[4];
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float qq = u == 0 ? q : (u == 1 ? qu1 : (u == 2 ? qu2 : qu3));
                        const float up = joseph_u(spk, m, qq);
                        const float t = __fadd_rn(up, JOSEPH_BIAS);
                        const unsigned ip = min((unsigned)(__float_as_int(t) - (JOSEPH_BIAS_BITS - 2)), top);
                        gg[u] = __fsub_rn(up, __fsub_rn(t, JOSEPH_BIAS));
                        pr[u] = P[ridx + u * SP + (int)ip];
                    }
                    acc0 += __fmaf_rn(gg[0], pr[0].y, pr[0].x);
                    acc1 += __fmaf_rn(gg[1], pr[1].y, pr[1].x);
                    acc2 += __fmaf_rn(gg[2], pr[2].y, pr[2].x);
                    acc3 += __fmaf_rn(gg[3], pr[3].y, pr[3].x);
                    spk = __fadd_rn(spk, 4.0f);
                    ridx += 4 * SP;
                }
                for (; s <= hi; ++s) {
                    const float up = joseph_u(spk, m, q);
                    const float t = __fadd_rn(up, JOSEPH_BIAS);
                    const unsigned ip = min((unsigned)(__float_as_int(t) - (JOSEPH_BIAS_BITS - 2)), top);
                    const float g = __fsub_rn(up, __fsub_rn(t, JOSEPH_BIAS));
                    const float2 p = P[ridx + (int)ip];
                    acc0 += __fmaf_rn(g, p.y, p.x);
                    spk = __fadd_rn(spk, 1.0f);
                    ridx += SP;
                }
            } else {
                float spk = sp;
                for (int s = lo; s <= hi; ++s) {
                    int i0;
                    float g;
                    joseph_round(joseph_u(spk, m, q), i0, g);
                    i0 = min(max(i0, -2), N);
                    if (i0 >= I0 && i0 < I1) {
                        const float2 p = P[ridx + (i0 - I0)];
                        acc0 += __fmaf_rn(g, p.y, p.x);
                    }
                    spk = __fadd_rn(spk, 1.0f);
                    ridx += SP;
                }
            }
            const float sum = (acc0 + acc1) + (acc2 + acc3);
            float *o = out + (size_t)svi[vi] * B + d;
            if (!MULTI || I0 == -2) *o = sum;
            else *o += sum;                       // this thread wrote it in the previous pass
        }
    }
}

// ROWS = 2: up to 1024 threads (64 registers); ROWS = 4: more loads in flight
// per thread, up to 768 threads (85 registers).
template <int ROWS>
__global__ void __launch_bounds__(ROWS == 2 ? 1024 : 768)
k_project_quad(const float *__restrict__ x, const QuadItem *__restrict__ row_items, int n_row,
               const QuadItem *__restrict__ col_items, int n_col, int N, int V, int B, int pg, int gpb, int tpi,
               float *__restrict__ partial)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    pdl_wait();
    quad_body<ROWS>(whole_block(), blockIdx.x, blockIdx.y, blockIdx.z, gridDim.x, smraw, x, row_items, n_row,
                    col_items, n_col, N, V, B, pg, gpb, tpi, partial);
}

// A x of small images in one launch, without partial sums.  A block takes one
// item: it stages all band pairs of the item's line class (at most
// DIRECT_BANDS, 76 KB at N = 96), a thread walks one of a position's two rays
// through one band pair, and the sums meet in shared memory, where each ray's
// are added in quad_position's and k_band_reduce's order and scaled (the same
// bits).  Such a projection is a call's latency: one kernel and no scratch,
// instead of two kernels and an allocation (64^2 / 90 views: 21 us a call),
// and walks as short as can be (8 items a block with both rays and all bands
// on one thread took 10.5 us, six SMs busy).
constexpr int DIRECT_BANDS = 3;
constexpr int DIRECT_THREADS = 1024;

__global__ void __launch_bounds__(DIRECT_THREADS)
k_project_direct(const float *__restrict__ x, const QuadItem *__restrict__ row_items, int n_row,
                 const QuadItem *__restrict__ col_items, int N, int V, int B, int tpi,
                 const ViewP *__restrict__ views, float *__restrict__ out)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    const bool rows = (int)blockIdx.x < n_row;
    const QuadItem it = rows ? row_items[blockIdx.x] : col_items[blockIdx.x - n_row];
    const int nb = quad_bands(N), SP = (N + 3) | 1, npair = (B + 1) / 2;
    const float *img = x + (size_t)blockIdx.y * N * N;
    for (int b = 0; b < nb; ++b)
        quad_stage<false>(whole_block(), smraw + b * quad_smem(N), img, N, b * MR, rows);
    float4 *red = reinterpret_cast<float4 *>(smraw + nb * quad_smem(N));   // [2 band + ray][position]
    __syncthreads();
    const int part = threadIdx.x / tpi, idx = threadIdx.x - part * tpi, b = part >> 1;
    const int d = idx < npair ? quad_ray(idx, it.stride, npair) : 0, dm = B - 1 - d;
    float4 r = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    if (idx < npair && !((part & 1) && dm == d)) {
        const float q = joseph_q(joseph_dp((part & 1) ? dm : d, B), it.a, joseph_hq(N));
        const int s0 = b * MR, s1 = min(s0 + MR, (N + 1) / 2) - 1;
        const float h = joseph_h(N);
        const unsigned top = (unsigned)(N + 2);
        const void *Q = smraw + b * quad_smem(N);
        int lo, hi;
        step_range(q, it.m, it.inv_m, h, -2.5f, (float)N + 0.5f, s0, s1, lo, hi);
        r = it.vp >= 0 ? quad_walk<true, 2, false>(Q, SP, q, it.m, lo, hi, s0, h, top)
                       : quad_walk<false, 2, false>(Q, SP, q, it.m, lo, hi, s0, h, top);
    }
    red[part * tpi + idx] = r;
    __syncthreads();
    if (part != 0 || idx >= npair) return;
    float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);   // view v: rays d, dm; view vp: rays d, dm
    for (int k = 0; k < nb; ++k) {
        const float4 u = red[2 * k * tpi + idx], v = red[(2 * k + 1) * tpi + idx];   // the walks of rays d and dm
        float o0 = u.x + v.y, o1 = u.y + v.x;
        float p0 = rows ? u.z + v.w : u.w + v.z, p1 = rows ? u.w + v.z : u.z + v.w;
        if (dm == d) {   // one walk: both its sums are ray d's
            o0 = u.x + u.y;
            p0 = rows ? u.z + u.w : u.w + u.z;
        }
        acc.x += o0;
        acc.y += o1;
        acc.z += p0;
        acc.w += p1;
    }
    float *o = out + (size_t)blockIdx.y * V * B + (size_t)it.v * B;
    const float sc = views[it.v].scale;
    o[d] = acc.x * sc;
    if (dm != d) o[dm] = acc.y * sc;
    if (it.vp >= 0) {
        float *o2 = out + (size_t)blockIdx.y * V * B + (size_t)it.vp * B;
        const float sp = views[it.vp].scale;
        o2[d] = acc.z * sp;
        if (dm != d) o2[dm] = acc.w * sp;
    }
}

// Served by k_project_direct: the whole image's bands staged at once, the
// threads of one item in a block, and few enough blocks that staging an
// image per item does not show (16 x 64^2 / 90 views, 720 blocks: as fast as
// the band-pair form and its reduction).
bool project_direct_ok(const Geometry *g, int batch)
{
    const int nb = quad_bands(g->n), tpi = ((g->n_bins + 1) / 2 + 31) / 32 * 32;
    return nb <= DIRECT_BANDS && 2 * nb * tpi <= DIRECT_THREADS &&
           (long long)(g->n_row_items + g->n_col_items) * batch <= 8LL * g->n_sm;
}

static size_t direct_smem(int n, int tpi) { return quad_bands(n) * (quad_smem(n) + 2 * sizeof(float4) * tpi); }

void launch_project_direct(const Geometry *g, const float *x, float *out, int batch, cudaStream_t st)
{
    const int tpi = ((g->n_bins + 1) / 2 + 31) / 32 * 32;
    counted();
    k_project_direct<<<dim3(g->n_row_items + g->n_col_items, batch), 2 * quad_bands(g->n) * tpi,
                       direct_smem(g->n, tpi), st>>>(x, g->d_row_items, g->n_row_items, g->d_col_items, g->n,
                                                     g->n_views, g->n_bins, tpi, g->d_views, out);
}

// The work-balanced form: block b takes units [total b / nb, total (b+1) / nb)
// (see quad_balanced_body); its unit counter sits after the staged pairs.
__device__ __forceinline__ unsigned long long global_time()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// bounds (optional): block b takes units [bounds[b], bounds[b+1]), a table
// of the geometry's written before any launch that reads it (so it is read
// before the wait for the previous kernel); else equal unit counts.
// times (optional): block b writes its start and end times (ns) to
// times[2b], times[2b+1].
template <int ROWS, bool RAW>
__global__ void __launch_bounds__(ROWS == 2 ? 1024 : 768)
k_project_qbal(const float *__restrict__ x, const QuadItem *__restrict__ row_items,
               const QuadItem *__restrict__ col_items, int N, int V, int B, QuadUnits U, long long total,
               long long share, const long long *__restrict__ bounds, unsigned long long *__restrict__ times,
               float *__restrict__ partial)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    const long long nb = gridDim.x;
    long long u0, u1;
    if (bounds) {   // clamped: a table is never read outside [0, total)
        u0 = min(max(bounds[blockIdx.x], 0LL), total);
        u1 = min(max(bounds[blockIdx.x + 1], u0), total);
    } else {
        // equal counts, the first blocks one more
        u0 = (long long)blockIdx.x * share + min((long long)blockIdx.x, total - share * nb);
        u1 = u0 + share + (blockIdx.x < total - share * nb ? 1 : 0);
    }
    pdl_wait();
    const unsigned long long t0 = times ? global_time() : 0ull;
    quad_balanced_body<ROWS, RAW>(whole_block(), u0, u1, U, smraw, reinterpret_cast<int *>(smraw + quad_smem(N, RAW)),
                                  x, row_items, col_items, N, V, B, partial);
    if (times) {
        __syncthreads();
        if (threadIdx.x == 0) {
            times[2 * blockIdx.x] = t0;
            times[2 * blockIdx.x + 1] = global_time();
        }
    }
}

// Launch shapes of the mirrored projector.
//
// k_project_quad: a block stages one band pair and walks gpb groups of pg
// items, tpi threads an item.  k_project_qbal: about one block an SM, each
// with an equal range of units.  The built-in rule takes the shape with the
// least modelled time, in SM cycles:
//   staging a band pair: 45 instructions per 32 entries, and a round trip of
//     700 cycles per four entries of a thread;
//   walking a ray position (both of its rays): 800 instructions per warp
//     (450 for an item of one view), a chain of 1100 cycles;
//   an SM issues 2.4 instructions a cycle for its resident blocks.
// The constants are fitted to a sweep of (pg, tpi) over 16 geometries, 32^2
// to 512^2, 12 to 720 views.  What it is for: with 64 threads an item, few-view
// grids left most warp slots empty and each thread six positions of serial
// walk (512^2 / 32 views: 80 blocks of 8 warps 13.6 us, 144 blocks of 24 warps
// 8.4 us; 256^2 / 90: 8.9 and 6.8 us).  Launches in a graph, warm cache, with
// the staging of quad_stage: 512^2 / 32 views 18.1 -> 8.3 us, 64^2 / 90 5.4 ->
// 4.3, 256^2 / 180 11.9 -> 9.5, 512^2 / 720 69.9 -> 65.3.  Sides that are not a
// multiple of 32, over 637, or custom angles took unmirrored or unpaired
// kernels before: 1024^2 / 720 718 -> 313 us, 900^2 / 300 258 -> 82, 2 x 333^2
// / 101 27.2 -> 16.8, 512^2 / 720 golden angles 97.8 -> 77.7.
struct QuadShape {
    int pg, gpb, tpi;
    double cost;
};
static double stage_cycles(int N, int warps, double share)
{
    const double entries = MR * ((N + 33) / 32);
    return entries * 45.0 * share / 2.4 + ceil(entries / (4.0 * warps)) * 700.0;
}
static double walk_instr(const Geometry *g) { return g->vpair ? 800.0 : 450.0; }

// the projector's settings in force: all by the rule when the tuner found the rule's shape best
struct ProjSettings {
    int pg, tpi, rows, form;
};
static ProjSettings settings(const Geometry *g)
{
    if (g->tune_tpi < 0) return ProjSettings{0, 0, 0, 0};
    return ProjSettings{g->tune_pg, g->tune_tpi, g->tune_qrows, g->tune_qbal};
}

static QuadShape quad_shape(const Geometry *g, int batch, int rows4)
{
    const ProjSettings t = settings(g);
    const int N = g->n, npair = (g->n_bins + 1) / 2, bands = quad_bands(N);
    const int max_threads = rows4 ? 768 : 1024;
    const int by_smem = std::max(1, QUAD_SMEM_MAX / (int)(quad_smem(N) + 1024));
    static const int tpis[] = {32, 64, 96, 128, 192, 256, 384, 512};
    QuadShape best{0, 1, 64, -1.0};
    const int pg_fix = t.pg;
    for (int pg = pg_fix > 0 ? pg_fix : 1; pg <= (pg_fix > 0 ? pg_fix : PG); ++pg) {
        const long rg = (g->n_row_items + pg - 1) / pg, cg = (g->n_col_items + pg - 1) / pg;
        for (int tpi : tpis) {
            if (t.tpi > 0 ? tpi != t.tpi : pg_fix > 0 && tpi != 64) continue;
            const int threads = pg * tpi;
            if (threads > max_threads || threads < 64 || (tpi > 64 && tpi >= npair + 64)) continue;
            const int occ = std::max(1, std::min(by_smem, max_threads / threads));
            for (int gpb = 1; gpb <= 8; ++gpb) {
                const long blocks = bands * ((rg + gpb - 1) / gpb + (cg + gpb - 1) / gpb) * (long)batch;
                const double share = (double)std::min<long>(occ, (blocks + g->n_sm - 1) / g->n_sm);
                const double waves = ceil((double)blocks / ((double)g->n_sm * occ));
                const double walk = gpb * pg * (double)((npair + 31) / 32) * walk_instr(g) * share / 2.4 +
                                    gpb * (double)((npair + tpi - 1) / tpi) * 1100.0;
                const double cost = waves * (stage_cycles(N, threads / 32, share) + walk);
                if (best.cost < 0.0 || cost < best.cost) best = QuadShape{pg, gpb, tpi, cost};
                if (rg <= gpb && cg <= gpb) break;
            }
        }
    }
    return best;
}

// Launch shape of the work-balanced form: as many blocks as fit on the
// device at once (fewer when the work would leave a warp under two units).
// Four steps a pass and 12 items' threads unless set (512^2 / 720 views: 64.6
// us, against 66.5 with two steps and 16 items' threads).
struct QbalShape {
    QuadUnits U;
    long long total;
    int rows4, raw, pgb, threads, blocks, key;
    size_t smem;
    double cost;
};
using QbalKernel = decltype(&k_project_qbal<2, false>);
static QbalKernel qbal_kernel(const QbalShape &q)
{
    return q.rows4 ? (q.raw ? k_project_qbal<4, true> : k_project_qbal<4, false>)
                   : (q.raw ? k_project_qbal<2, true> : k_project_qbal<2, false>);
}
static bool quad_raw(const Geometry *g) { return quad_smem(g->n) + 16 > (size_t)QUAD_SMEM_MAX; }
static QbalShape qbal_shape(const Geometry *g, int batch)
{
    QbalShape q;
    const ProjSettings t = settings(g);
    const int N = g->n;
    q.rows4 = t.rows == 4 || (t.rows == 0 && t.pg <= 12);
    q.raw = quad_raw(g);
    const int max_pg = q.rows4 ? 12 : PG;
    q.pgb = t.pg > 0 ? std::min(t.pg, max_pg) : max_pg;
    q.threads = q.pgb * 64;
    q.smem = quad_smem(N, q.raw) + 16;
    // blocks per SM, queried once per (steps per pass, items) for the geometry
    int &occ_slot = const_cast<Geometry *>(g)->qbal_occ[q.rows4][q.pgb];
    int occ = occ_slot;
    if (occ < 1) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, qbal_kernel(q), q.threads, q.smem) != cudaSuccess ||
            occ < 1)
            occ = 1;
        occ_slot = occ;
    }
    // units of 64 positions, or of 32 when a warp would take fewer than eight of the former
    q.U = quad_units(N, g->n_bins, g->n_row_items, g->n_col_items, 2);
    if (q.U.u_z * batch < (long long)g->n_sm * occ * q.pgb * 2 * 8)
        q.U = quad_units(N, g->n_bins, g->n_row_items, g->n_col_items, 1);
    q.total = q.U.u_z * batch;
    q.key = (q.U.upl * 2 + q.rows4) * 64 + q.pgb;
    const long long by_work = (q.total + 4 * q.pgb - 1) / (4 * q.pgb);   // two units per warp
    q.blocks = (int)std::max(1LL, std::min((long long)g->n_sm * occ, by_work));
    const double share = std::min<double>(occ, ceil((double)q.blocks / g->n_sm));
    const double segs = 1.0 + (double)(2 * quad_bands(N)) * batch / q.blocks;   // segments a block's range touches
    q.cost = segs * stage_cycles(N, q.pgb * 2, share) +
             (double)q.total / q.blocks * q.U.upl * walk_instr(g) * share / 2.4 + 2.0 * q.U.upl * 1100.0;
    return q;
}

// The mirrored projector's launch for one batch size, kept in the geometry
// (the shape model is too slow for every call) until its tuning changes.
struct ProjPlan {
    int batch = 0, balanced, rows4;
    QuadShape quad;
    QbalShape qbal;
};
struct ProjPlans {
    std::mutex mu;
    ProjPlan p[4];
    int next = 0;
};
static ProjPlan make_plan(const Geometry *g, int batch)
{
    ProjPlan p;
    p.batch = batch;
    const ProjSettings t = settings(g);
    p.rows4 = t.rows == 4;
    p.qbal = qbal_shape(g, batch);
    p.balanced = quad_raw(g) || t.form == 2;
    // The factor is fitted: without it the rule took the balanced form for 4 x
    // 384^2 / 90 views (27.4 us against 25.3), 512^2 / 90 (17.2, 15.0) and 4 x
    // 512^2 / 32 (21.5, 18.3); with it, it still takes it for 512^2 / 720 (65.3
    // us against 66.5) and 512^2 / 360.
    if (!p.balanced) {
        p.quad = quad_shape(g, batch, p.rows4);
        p.balanced = p.quad.cost < 0.0 || (t.form == 0 && 1.16 * p.qbal.cost < p.quad.cost);
    }
    return p;
}
static ProjPlan proj_plan(const Geometry *g, int batch)
{
    ProjPlans &c = *static_cast<ProjPlans *>(g->proj_plans);
    std::lock_guard<std::mutex> lock(c.mu);
    for (const ProjPlan &p : c.p)
        if (p.batch == batch) return p;
    ProjPlan &p = c.p[c.next];
    c.next = (c.next + 1) % 4;
    p = make_plan(g, batch);
    return p;
}
void *proj_plans_create() { return new (std::nothrow) ProjPlans; }
void proj_plans_free(void *p) { delete static_cast<ProjPlans *>(p); }
void proj_plans_clear(Geometry *g)
{
    ProjPlans &c = *static_cast<ProjPlans *>(g->proj_plans);
    std::lock_guard<std::mutex> lock(c.mu);
    for (ProjPlan &p : c.p) p.batch = 0;
}

void launch_project_bands(const Geometry *g, const float *x, float *partial, int batch, cudaStream_t st, bool plain)
{
    const int N = g->n;
    counted();
    if (quad_ok(g) && !plain) {
        // mirrored 16-step bands: ceil(N/32) partial slots
        const ProjPlan p = proj_plan(g, batch);
        if (p.balanced) {
            const QbalShape &q = p.qbal;
            // the tuner's measured-balance ranges, for the launch they were made for
            const long long *bounds =
                batch == 1 && g->d_qbounds && g->qbounds_nb > 0 && g->qbounds_nb == q.blocks && g->qbounds_key == q.key
                    ? g->d_qbounds
                    : nullptr;
            launch_kernel(qbal_kernel(q), dim3(q.blocks), dim3(q.threads), q.smem, st, x, g->d_row_items,
                          g->d_col_items, N, g->n_views, g->n_bins, q.U, q.total, q.total / q.blocks, bounds,
                          g->d_qtimes, partial);
            return;
        }
        const QuadShape &q = p.quad;
        const int rg = (g->n_row_items + q.pg - 1) / q.pg, cg = (g->n_col_items + q.pg - 1) / q.pg;
        const dim3 grd(quad_bands(N), (rg + q.gpb - 1) / q.gpb + (cg + q.gpb - 1) / q.gpb, batch);
        launch_kernel(p.rows4 ? k_project_quad<4> : k_project_quad<2>, grd, dim3(q.pg * q.tpi), quad_smem(N), st, x,
                      g->d_row_items, g->n_row_items, g->d_col_items, g->n_col_items, N, g->n_views, g->n_bins, q.pg,
                      q.gpb, q.tpi, partial);
        return;
    }
    dim3 grd(proj_bands(N), (g->n_row + PG - 1) / PG + (g->n_col + PG - 1) / PG, batch);
    const size_t smem = proj_smem(N);
    if (N + 3 <= PROJ_CW)
        k_project_bands<false><<<grd, PT, smem, st>>>(x, g->d_views, g->d_row_list, g->n_row, g->d_col_list,
                                                      g->n_col, N, g->n_views, g->n_bins, partial);
    else
        k_project_bands<true><<<grd, PT, smem, st>>>(x, g->d_views, g->d_row_list, g->n_row, g->d_col_list,
                                                     g->n_col, N, g->n_views, g->n_bins, partial);
}

// out[v][d] = scale_v * sum_b partial[b][v][d]; SCALED: times fac[0]
template <bool SCALED>
__global__ void k_band_reduce(const float *__restrict__ partial, float *__restrict__ out,
                              const ViewP *__restrict__ views, int nb, int V, int B, const double *__restrict__ fac)
{
    pdl_wait();
    const int d = blockIdx.x * blockDim.x + threadIdx.x, v = blockIdx.y;
    if (d >= B) return;
    const size_t VB = (size_t)V * B;
    const float *p = partial + (size_t)blockIdx.z * nb * VB + (size_t)v * B + d;
    float acc = 0.0f;
    for (int k = 0; k < nb; ++k) acc += p[k * VB];
    float val = acc * views[v].scale;
    if (SCALED) val *= (float)*fac;
    out[(size_t)blockIdx.z * VB + (size_t)v * B + d] = val;
}

// The plain sum for B % 4 == 0, four bins a thread and four bands'
// loads together: with the projector before it, 512^2 / 720 views 70.3 -> 68.7
// us, 1024^2 / 720 341.6 -> 329.9 (eight and sixteen bands together are slower,
// 71.0 and 71.4 us: more rows of the partial sums open at once).
constexpr int BR_BANDS = 4;
__global__ void __launch_bounds__(256)
k_band_reduce4(const float4 *__restrict__ partial, float4 *__restrict__ out, const ViewP *__restrict__ views, int nb,
               unsigned vb4, unsigned b4)
{
    pdl_wait();
    const unsigned i = blockIdx.x * 256 + threadIdx.x;
    if (i >= vb4) return;
    const float4 *p = partial + (size_t)blockIdx.y * nb * vb4 + i;
    float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    for (int k0 = 0; k0 < nb; k0 += BR_BANDS) {
        float4 t[BR_BANDS];
#pragma unroll
        for (int k = 0; k < BR_BANDS; ++k)
            t[k] = k0 + k < nb ? p[(size_t)(k0 + k) * vb4] : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
        for (int k = 0; k < BR_BANDS; ++k)
            if (k0 + k < nb) {
                acc.x += t[k].x;
                acc.y += t[k].y;
                acc.z += t[k].z;
                acc.w += t[k].w;
            }
    }
    const float s = views[i / b4].scale;
    out[(size_t)blockIdx.y * vb4 + i] = make_float4(acc.x * s, acc.y * s, acc.z * s, acc.w * s);
}

void launch_band_reduce(const Geometry *g, const float *partial, float *out, int batch, cudaStream_t st)
{
    dim3 grd((g->n_bins + 255) / 256, g->n_views, batch);
    const int nb = proj_bands(g->n);
    counted();
    const unsigned b4 = g->n_bins / 4, vb4 = b4 * g->n_views;
    // below 20000 rays the grid of four-bin threads is too small (256^2 / 32 views: 7.6 against 7.3 us)
    if (g->n_bins % 4 == 0 && 4 * vb4 >= 20000 &&
        (reinterpret_cast<uintptr_t>(partial) | reinterpret_cast<uintptr_t>(out)) % 16 == 0) {
        launch_kernel(k_band_reduce4, dim3((vb4 + 255) / 256, batch), dim3(256), 0, st, (const float4 *)partial,
                      (float4 *)out, g->d_views, nb, vb4, b4);
        return;
    }
    launch_kernel(k_band_reduce<false>, grd, dim3(256), 0, st, partial, out, g->d_views, nb, g->n_views, g->n_bins,
                  nullptr);
}

// out = fac * A x from the band partials (fac: one device double)
void launch_band_reduce_scaled(const Geometry *g, const float *partial, float *out, const double *fac, int batch,
                               cudaStream_t st)
{
    dim3 grd((g->n_bins + 255) / 256, g->n_views, batch);
    counted();
    k_band_reduce<true><<<grd, 256, 0, st>>>(partial, out, g->d_views, proj_bands(g->n), g->n_views, g->n_bins, fac);
}

// =====================================================================
// Backprojection: a pixel-driven gather.  Pixel (r, c) sits at detector
// coordinate e = (c - h) cos t + (r - h) sin t + hb of view t, and ray d
// reaches it with Joseph's weight 1 - |u(d) - j| = 1 - |d - e| |a| (u the
// coordinate along the stepping direction, j the pixel's index along it,
// |a| = 1/max(|cos t|, |sin t|)), non-zero only for d = floor(e) and
// floor(e) + 1.  In exact arithmetic this is the weight the projector
// uses, so A^T is the transpose of A up to the float rounding of the
// weight (a few ulp); every pixel sums its rays in a fixed order, so the
// result is deterministic and needs no atomics.
//
// One block per BT x BT tile.  Views are staged in chunks: per view
// (cos, sin, |a|, 1 - |a|/2) and a window of ray pairs
// (y[d], y[d+1]) * |a| covering the rays that reach the tile.  The block's
// 256 threads form BSL view slices of 64 threads; a thread owns four
// pixels of one row and sums the views of its slice; the slices are added
// in a fixed order at the end.
// =====================================================================
constexpr int BT = 16;          // tile side
constexpr int BSL = 4;          // view slices per block
constexpr int BTH = 64 * BSL;   // threads per block
constexpr int BVC = 64;         // views staged per chunk
constexpr int BWW = 32;         // staged ray pairs per view (>= 15 (|cos|+|sin|) + 3)

template <int MODE>
__global__ void __launch_bounds__(BTH)
k_backproject_tiles(const float *__restrict__ y, float *__restrict__ out,
                    const float4 *__restrict__ trig, int N, int V, int B,
                    const float *__restrict__ xin, const double *__restrict__ scal)
{
    __shared__ float2 tab[BVC][BWW];
    __shared__ float4 sv[BVC];
    __shared__ int wbase[BVC];
    __shared__ float red[BSL][BT * BT];

    const int tid = threadIdx.x;
    const int slice = tid >> 6, l = tid & 63;
    const int R0 = blockIdx.y * BT, C0 = blockIdx.x * BT;
    const int r = R0 + (l >> 2), c0 = C0 + (l & 3) * 4;
    const float *ys = y + (size_t)blockIdx.z * V * B;
    const float h = 0.5f * (float)(N - 1);
    const float hb_lo = 0.5f * (float)(B - 1) - 0.5f;   // e - 1/2 is rounded to find floor(e)
    const float yr = (float)r - h;
    float xc[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) xc[k] = (float)(c0 + k) - h;
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};

    for (int v0 = 0; v0 < V; v0 += BVC) {
        const int nv = min(BVC, V - v0);
        __syncthreads();
        if (tid < nv) {
            const float4 T = trig[v0 + tid];   // cos, sin, |a|, 1 - |a|/2
            sv[tid] = T;
            // lowest detector coordinate over the tile corners
            float emin = 3.0e38f;
#pragma unroll
            for (int cr = 0; cr < 4; ++cr) {
                const float xx = (float)(C0 + (cr & 1) * (BT - 1)) - h;
                const float yy = (float)(R0 + (cr >> 1) * (BT - 1)) - h;
                emin = fminf(emin, xx * T.x + yy * T.y);
            }
            emin = fminf(fmaxf(emin + 0.5f * (float)(B - 1), -1.0e6f), 1.0e6f);
            wbase[tid] = (int)floorf(emin) - 2;
        }
        __syncthreads();
        for (int k = tid; k < nv * BWW; k += BTH) {
            const int vi = k / BWW, w = k - vi * BWW;
            const int d = wbase[vi] + w;
            const float *yv = ys + (size_t)(v0 + vi) * B;
            const float sc = sv[vi].z;
            const float y0 = (d >= 0 && d < B) ? yv[d] : 0.0f;
            const float y1 = (d + 1 >= 0 && d + 1 < B) ? yv[d + 1] : 0.0f;
            tab[vi][w] = make_float2(y0 * sc, y1 * sc);
        }
        __syncthreads();
        if (r < N) {
            for (int vi = slice; vi < nv; vi += BSL) {
                const float4 T = sv[vi];
                const int fb = JOSEPH_BIAS_BITS + wbase[vi];
                const float eb = fmaf(yr, T.y, hb_lo);
                const float2 *tv = tab[vi];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const float e = fmaf(xc[k], T.x, eb);               // e - 1/2
                    const float t = __fadd_rn(e, JOSEPH_BIAS);
                    // floor(e) - wbase, kept inside the staged window
                    const unsigned f = min((unsigned)(__float_as_int(t) - fb), (unsigned)(BWW - 1));
                    const float g = __fsub_rn(e, __fsub_rn(t, JOSEPH_BIAS));   // frac(e) - 1/2
                    const float w0 = fmaxf(0.0f, fmaf(-g, T.z, T.w));   // 1 - frac |a|
                    const float w1 = fmaxf(0.0f, fmaf(g, T.z, T.w));    // 1 - (1 - frac) |a|
                    const float2 yy = tv[f];
                    acc[k] = fmaf(w0, yy.x, fmaf(w1, yy.y, acc[k]));
                }
            }
        }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) red[slice][(l >> 2) * BT + (l & 3) * 4 + k] = acc[k];
    __syncthreads();
    if (tid < BT * BT) {
        const int rr = R0 + tid / BT, cc = C0 + tid % BT;
        if (rr < N && cc < N) {
            float tot = red[0][tid];
#pragma unroll
            for (int k = 1; k < BSL; ++k) tot += red[k][tid];
            const size_t o = (size_t)blockIdx.z * N * N + (size_t)rr * N + cc;
            if (MODE == 0) out[o] = tot;
            else out[o] = xin[o] - fscal(scal, F_TAU) * tot;
        }
    }
}

template <int FORM>
__global__ void __launch_bounds__(ORB_TH, 8)
k_backproject_orbit(const float *__restrict__ y, int ld, float *__restrict__ partial, const float4 *__restrict__ trig,
                    int N, int V, int B, int nsl, int fin, float *out, const float *xin,
                    const double *__restrict__ scal)
{
    extern __shared__ __align__(16) unsigned char osm[];
    pdl_wait();
    orbit_body<FORM>(Block2D{}, blockIdx.x, blockIdx.y, blockIdx.z, osm, y, ld, partial, trig, N, V, B, nsl, fin, out, xin,
                   scal);
}

// The orbit backprojector with its base-view slices added in a thread-block
// cluster: the nsl blocks of one tile (grid.z = images x slices, cluster
// (1, 1, nsl)) each leave their partial sums in shared memory; block s then
// adds, for its share of the tile's 4 ORB_PX ORB_TH sums, the nsl partials
// in slice order through distributed shared memory and writes the sum
// (mode 0) or xin - tau sum (mode 1).  No slice images are written, and no
// reduction pass runs.
template <int FORM>
__global__ void __launch_bounds__(ORB_TH, 8)
k_backproject_orbit_cl(const float *__restrict__ y, int ld, const float4 *__restrict__ trig, int N, int V, int B, int nsl,
                       int mode, float *out, const float *xin, const double *__restrict__ scal)
{
    extern __shared__ __align__(16) unsigned char osm[];
    pdl_wait();
    orbit_body<FORM, Block2D, true>(Block2D{}, blockIdx.x, blockIdx.y, blockIdx.z, osm, y, ld, nullptr, trig, N, V, B, nsl, 0,
                                  nullptr, nullptr, scal);
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    cl.sync();   // every slice's partial sums are in its shared memory
    const int slice = blockIdx.z % nsl, img = blockIdx.z / nsl;   // the block's rank in its cluster
    float *red = reinterpret_cast<float *>(osm);
    constexpr int E = 4 * ORB_PX * ORB_TH;
    const int e0 = E * slice / nsl, e1 = E * (slice + 1) / nsl;
    const int half = N / 2;
    const float tau = mode ? fscal(scal, F_TAU) : 0.0f;
    float *o_img = out + (size_t)img * N * N;
    const float *x_img = mode ? xin + (size_t)img * N * N : nullptr;
    for (int e = e0 + (int)(threadIdx.y * blockDim.x + threadIdx.x); e < e1; e += ORB_TH) {
        float t = *cl.map_shared_rank(red + e, 0);
        for (int s = 1; s < nsl; ++s) t += *cl.map_shared_rank(red + e, s);
        const int k = e / (ORB_PX * ORB_TH), rem = e - k * (ORB_PX * ORB_TH);
        const int j = rem / ORB_TH, th = rem - j * ORB_TH;
        const int rj = blockIdx.y * ORB_T + th / ORB_T + j * ORB_TY, c = half + blockIdx.x * ORB_T + th % ORB_T;
        if (rj < half && c < N) {
            const size_t o = k == 0   ? (size_t)rj * N + c
                             : k == 1 ? (size_t)c * N + (N - 1 - rj)
                             : k == 2 ? (size_t)(N - 1 - rj) * N + (N - 1 - c)
                                      : (size_t)(N - 1 - c) * N + rj;
            o_img[o] = mode ? __fmaf_rn(-tau, t, x_img[o]) : t;
        }
    }
    cl.sync();   // no block leaves while its partial sums may still be read
}

// The same sums with fewer blocks than slices: the csz blocks of a tile share
// the nsl slices (orbit_body, SEQ), whose sums are added in slice order still,
// so the result has k_backproject_orbit_cl's bits whatever csz is.  CL: csz >
// 1 blocks in a cluster; else one block, which writes its sums itself.
template <int FORM, bool CL>
__global__ void __launch_bounds__(ORB_TH, 8)
k_backproject_orbit_seq(const float *__restrict__ y, int ld, const float4 *__restrict__ trig, int N, int V, int B,
                        int nsl, int csz, float *__restrict__ out)
{
    extern __shared__ __align__(16) unsigned char osm[];
    pdl_wait();
    orbit_body<FORM, Block2D, CL, true>(Block2D{}, blockIdx.x, blockIdx.y, blockIdx.z, osm, y, ld, nullptr, trig, N, V,
                                        B, nsl, 1, out, nullptr, nullptr, csz);
    if constexpr (CL) {
        namespace cg = cooperative_groups;
        cg::cluster_group cl = cg::this_cluster();
        cl.sync();   // every slice's sums are in its block's shared memory
        const int rank = blockIdx.z % csz, img = blockIdx.z / csz;
        const int sets = orbit_kept_sets(nsl, csz), lg = 31 - __clz(sets + 1);   // a block's slices: sets + 1 = 2^lg
        float *red = reinterpret_cast<float *>(osm), *kept = orbit_kept(osm);
        const int half = N / 2;
        float *o_img = out + (size_t)img * N * N;
        for (int e = ORB_E / csz * rank + (int)(threadIdx.y * blockDim.x + threadIdx.x); e < ORB_E / csz * (rank + 1);
             e += ORB_TH) {
            // the loads of all slices are issued together
            float p[ORB_SL_MAX];
#pragma unroll
            for (int s = 0; s < ORB_SL_MAX; ++s) {
                const int l = s & sets;
                if (s < nsl) p[s] = *cl.map_shared_rank(l < sets ? kept + l * ORB_E + e : red + e, s >> lg);
            }
            float t = p[0];
#pragma unroll
            for (int s = 1; s < ORB_SL_MAX; ++s)
                if (s < nsl) t += p[s];
            const int k = e / (ORB_PX * ORB_TH), rem = e - k * (ORB_PX * ORB_TH);
            const int j = rem / ORB_TH, th = rem - j * ORB_TH;
            const int rj = blockIdx.y * ORB_T + th / ORB_T + j * ORB_TY, c = half + blockIdx.x * ORB_T + th % ORB_T;
            if (rj < half && c < N)
                o_img[k == 0   ? (size_t)rj * N + c
                      : k == 1 ? (size_t)c * N + (N - 1 - rj)
                      : k == 2 ? (size_t)(N - 1 - rj) * N + (N - 1 - c)
                               : (size_t)(N - 1 - c) * N + rj] = t;
        }
        cl.sync();   // no block leaves while its sums may still be read
    }
}

// shared memory of a block that holds the window bases of `views` base views, and `kept` sets of sums
static size_t orbit_smem(int views = ORB_MAXS, int kept = 0)
{
    return sizeof(float) * 2 * ORB_VC * 8 * ORB_RW + sizeof(float4) * 4 * ORB_VC + sizeof(float) * ORB_E * kept +
           sizeof(int) * 2 * views;
}

// out = sum of the slice images (mode 0), or xin - tau * sum (mode 1)
template <int MODE>
__global__ void k_orbit_reduce(const float *__restrict__ partial, float *__restrict__ out, const float *xin,
                               const double *__restrict__ scal, size_t NN, int nsl)
{
    pdl_wait();
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i >= NN) return;
    const float *pp = partial + (size_t)blockIdx.y * nsl * NN + i;
    float t = pp[0];
    for (int s = 1; s < nsl; ++s) t += pp[s * NN];
    const size_t o = (size_t)blockIdx.y * NN + i;
    if (MODE == 0) out[o] = t;
    else out[o] = __fmaf_rn(-fscal(scal, F_TAU), t, xin[o]);   // one rounding, as every form of z
}

bool orbit_ok(const Geometry *g) { return g->orbit; }
size_t orbit_partial_floats(const Geometry *g, int batch) { return (size_t)ORB_SL_MAX * g->n * g->n * batch; }

// base-view slices of the orbit kernel: a slice holds at most ORB_MAXS base views
bool orbit_slices_ok(const Geometry *g, int nsl)
{
    return nsl >= 1 && nsl <= ORB_SL_MAX && (g->n_views / 2 + nsl - 1) / nsl <= ORB_MAXS;
}
int orbit_slices(const Geometry *g, bool cluster)
{
    const int t = cluster ? g->tune_orb : g->tune_orb_si;
    return t > 0 ? t : g->orb_rule;
}

// Modelled time, in us, of A^T of `images` images by `blocks` blocks a tile,
// each taking `share` slices of `views` base views.  A block costs about 0.3,
// 0.07 per slice after its first and, per base view, 0.19 alone on its SM,
// 0.135 with another, 0.118 as one of three and 0.105 of four and more, the
// most blocks of any SM counting; adding the blocks' sums in a cluster costs 1
// and 0.6 per slice after a block's first.
static double orbit_cost(const Geometry *g, int images, int blocks, int share, double views)
{
    static const double per[] = {0.19, 0.135, 0.118, 0.105};
    const int q = (g->n / 2 + ORB_T - 1) / ORB_T;
    const long long k = ((long long)q * q * images * blocks + g->n_sm - 1) / g->n_sm;
    return (double)k * (share * views * per[std::min(k, 4LL) - 1] + 0.3 + 0.07 * (share - 1)) +
           (blocks > 1 ? 1.0 + 0.6 * (share - 1) : 0.0);
}

// The built-in count of base-view slices, which fixes the order of the sums:
// the least modelled time of one image over 1 .. 8 slices, or over 1, 2, 4
// and 8 (pow2; ct_backproject, whose batches share them out, orbit_blocks).
// (Warm launches: 512^2 / 32 views 7.1 us with one slice, 8.2 with four;
// 64^2 / 90 6.1 with four, 4.7 with eight; 256^2 / 180 9.9 and 9.0; 512^2 /
// 720 and 384^2 / 90 keep four.)
int orbit_slices_rule(const Geometry *g, bool pow2)
{
    if (!g->orbit) return ORB_SL;
    int best = ORB_SL;
    double cost = -1.0;
    for (int nsl = 1; nsl <= ORB_SL_MAX; ++nsl) {
        if (!orbit_slices_ok(g, nsl) || (pow2 && (nsl & (nsl - 1)))) continue;
        const double c = orbit_cost(g, 1, nsl, 1, (double)(g->n_views / 2) / nsl);
        if (cost < 0.0 || c < cost) {
            cost = c;
            best = nsl;
        }
    }
    return best;
}

// Blocks that share a tile's nsl slices (a power of two) in a launch of
// several images, by the same model: a batch that fills the device wants
// fewer than a lone image.  The count of slices stays, so an image has the
// same bits in any batch.  (Launches in a graph, aligned rows, a block per
// slice of a lone image's eight -> the rule's blocks; with four slices always:
// 64 x 64^2 / 90 15.0 -> 13.9, 13.2; 256 x 64^2 / 90 48.7 -> 36.0, 41.4; 128 x
// 48^2 / 60 22.8 -> 16.6, 16.8; 64 x 128^2 / 60 42.0 -> 26.3, 32.0; 4 x 256^2 /
// 90 15.3 -> 14.0, 13.7; 8 x 256^2 / 90 26.8 -> 22.4, 23.0; 4 x 256^2 / 180
// 22.0 -> 21.3, 20.7; 16 x 256^2 / 180 73.7 -> 63.7, 68.5 us.)
int orbit_blocks(const Geometry *g, int nsl, int images)
{
    int best = nsl;
    double cost = -1.0;
    for (int c = nsl; c >= 1; c /= 2) {
        const double t = orbit_cost(g, images, c, nsl / c, (double)(g->n_views / 2) / nsl);
        if (cost < 0.0 || t < cost) {
            cost = t;
            best = c;
        }
    }
    return best;
}
size_t orbit_smem_bytes() { return orbit_smem(); }
bool quad_ok(const Geometry *g) { return quad_smem(g->n, true) + 16 <= (size_t)QUAD_SMEM_MAX; }

// Measured balance of the work-balanced projector for one image.  Equal
// unit counts per block leave the blocks' times about 20 % apart at
// 512^2 / 720 views (views whose rays cross fewer staged steps, bank
// conflicts that differ by view, the two line classes), and the launch
// lasts as long as its slowest block.  The tuner keeps a cost per unit,
// uniform at first.  Each round times every block of a few launches
// (%globaltimer at its start and end), scales the costs of each block's
// units by (measured / modelled time)^0.7, and cuts the units again at
// equal shares of the modelled cost; as the ranges move between rounds the
// model resolves finer than one block.  The ranges of the round whose
// launch time (CUDA events) is least are kept, if they beat equal counts.
// A range only decides which block forms which units' sums, so results do
// not change.  The geometry's table (QB_CAP entries) is allocated once and
// kept until the geometry is destroyed, so that a graph captured before a
// later tuning never reads freed memory (and the kernel clamps what it
// reads); the rounds run on a scratch table.
constexpr int QB_CAP = 4096;
ct_status qbal_balance(Geometry *g, const float *x, float *band, cudaStream_t st)
{
    g->qbounds_nb = 0;   // no table until a better one is written
    if (!quad_ok(g) || !proj_plan(g, 1).balanced) return CT_OK;
    const QbalShape q = qbal_shape(g, 1);
    const int nb = q.blocks;
    if (nb < 2 || nb + 1 > QB_CAP) return CT_OK;
    const long long uz = q.U.u_z;
    unsigned long long *times = nullptr;
    long long *bounds = nullptr, *keep = g->d_qbounds;
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    cudaError_t e = cudaSuccess;
    if (!keep) {
        e = cudaMalloc(&keep, sizeof(long long) * QB_CAP);
        if (e == cudaSuccess) g->d_qbounds = keep;
    }
    if (e == cudaSuccess) e = cudaMalloc(&times, sizeof(unsigned long long) * 2 * nb);
    if (e == cudaSuccess) e = cudaMalloc(&bounds, sizeof(long long) * (nb + 1));
    if (e == cudaSuccess) e = cudaEventCreate(&e0);
    if (e == cudaSuccess) e = cudaEventCreate(&e1);
    std::vector<long long> b(nb + 1), best;
    for (int i = 0; i <= nb; ++i) b[i] = uz * i / nb;
    std::vector<unsigned long long> h(2 * nb);
    std::vector<double> dur(nb), cost((size_t)uz, 1.0), cum((size_t)uz + 1);
    float best_ms = -1.0f;
    // the mean time of 8 launches with the current table (none: equal counts)
    auto time_it = [&](float &ms) {
        launch_project_bands(g, x, band, 1, st);
        cudaEventRecord(e0, st);
        for (int r = 0; r < 8; ++r) launch_project_bands(g, x, band, 1, st);
        cudaEventRecord(e1, st);
        e = cudaEventSynchronize(e1);
        if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
        ms /= 8.0f;
    };
    if (e == cudaSuccess) time_it(best_ms);
    g->qbounds_key = q.key;
    for (int round = 0; round < 12 && e == cudaSuccess; ++round) {
        // block times of four launches with the current ranges
        e = cudaMemcpy(bounds, b.data(), sizeof(long long) * (nb + 1), cudaMemcpyHostToDevice);
        g->d_qbounds = bounds;   // the scratch table for the rounds' launches
        g->qbounds_nb = nb;
        g->d_qtimes = times;
        std::fill(dur.begin(), dur.end(), 0.0);
        for (int r = 0; r < 4 && e == cudaSuccess; ++r) {
            launch_project_bands(g, x, band, 1, st);
            e = cudaStreamSynchronize(st);
            if (e == cudaSuccess) e = cudaMemcpy(h.data(), times, sizeof(unsigned long long) * 2 * nb,
                                                 cudaMemcpyDeviceToHost);
            for (int i = 0; i < nb && e == cudaSuccess; ++i) dur[i] += (double)(h[2 * i + 1] - h[2 * i]);
        }
        g->d_qtimes = nullptr;
        if (e != cudaSuccess) break;
        // scale each block's unit costs towards its measured time, then cut
        // the units at equal shares of the modelled cost
        for (int i = 0; i < nb; ++i) {
            double model = 0.0;
            for (long long u = b[i]; u < b[i + 1]; ++u) model += cost[(size_t)u];
            if (model <= 0.0 || b[i + 1] == b[i]) continue;
            const double f = std::pow(std::max(dur[i], 1.0) / model, 0.7);
            for (long long u = b[i]; u < b[i + 1]; ++u) cost[(size_t)u] *= f;
        }
        cum[0] = 0.0;
        for (long long u = 0; u < uz; ++u) cum[(size_t)u + 1] = cum[(size_t)u] + cost[(size_t)u];
        b[0] = 0;
        b[nb] = uz;
        for (int k = 1; k < nb; ++k) {
            const double t = cum[(size_t)uz] * k / nb;
            const long long u = (long long)(std::lower_bound(cum.begin(), cum.end(), t) - cum.begin());
            b[k] = std::min(uz, std::max(b[k - 1], u));
        }
        e = cudaMemcpy(bounds, b.data(), sizeof(long long) * (nb + 1), cudaMemcpyHostToDevice);
        float ms = -1.0f;
        if (e == cudaSuccess) time_it(ms);
        if (e == cudaSuccess && ms > 0.0f && ms < best_ms) {
            best_ms = ms;
            best = b;
        }
    }
    g->d_qtimes = nullptr;
    g->d_qbounds = keep;
    g->qbounds_nb = 0;
    if (e == cudaSuccess && !best.empty() && keep) {
        e = cudaMemcpy(keep, best.data(), sizeof(long long) * (nb + 1), cudaMemcpyHostToDevice);
        if (e == cudaSuccess) g->qbounds_nb = nb;
    }
    if (bounds) cudaFree(bounds);
    if (times) cudaFree(times);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
    if (e != cudaSuccess) {
        cudaGetLastError();
        set_error("ct_geometry_autotune: %s", cudaGetErrorString(e));
        return e == cudaErrorMemoryAllocation ? CT_ERR_OOM : CT_ERR_CUDA;
    }
    return CT_OK;
}

// the rows of at_rows (half > 0): views v and v + V/2 interleaved, zeros past B
__global__ void k_pair_rows(const float *__restrict__ in, float2 *__restrict__ out, size_t n, int B, int ld, int half)
{
    const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    const size_t pair = i / (unsigned)ld, row = pair + pair / (unsigned)half * (unsigned)half;   // of its first view
    const int d = (int)(i - pair * ld);
    out[i] = d < B ? make_float2(in[row * B + d], in[(row + half) * B + d]) : make_float2(0.0f, 0.0f);
}

void launch_pair_rows(const Geometry *g, const float *in, float *out, int batch, cudaStream_t st)
{
    const int half = g->n_views / 2;
    const size_t n = (size_t)batch * half * g->ld;
    counted();
    k_pair_rows<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(in, reinterpret_cast<float2 *>(out), n, g->n_bins, g->ld,
                                                             half);
}

// Whether a caller's sinogram is better read in its own rows than interleaved
// first, which takes a pass, a launch and scratch (about 1.2 us in a graph, 2
// to 4 as a call).  Rows of whole 16-byte pieces are copied so, and interleaving
// gains 4 to 6 % of a large launch only (graph, own rows / interleaved: 64^2 /
// 90 views 4.5 / 5.8 us, 256^2 / 90 6.4 / 7.6, 512^2 / 90 13.1 / 13.7, 512^2 /
// 360 34.6 / 34.2, 512^2 / 720 65.0 / 62.5, 1024^2 / 720 235 / 222).  Others
// are copied value by value: for little work and few views (64^2 / 90 4.9 /
// 5.8 us, 128^2 / 90 5.7 / 6.4, 256^2 / 32 5.3 / 6.4; but 128^2 / 180 7.6 /
// 7.6, 64^2 / 720 15.7 / 12.1, 512^2 / 32 7.8 / 7.0).
bool orbit_plain_rows(const Geometry *g, int batch)
{
    const double pixel_views = (double)g->n * g->n * g->n_views * batch;
    return g->ld == g->n_bins ? pixel_views <= 1.2e8 : g->n_views <= 128 && pixel_views <= 2.5e6;
}

void launch_backproject_orbit(const Geometry *g, const float *y, float *out, int mode, const float *xin,
                              const double *scal, int batch, float *partial, cudaStream_t st, bool cluster, int slices,
                              bool plain, int blocks)
{
    const int q = g->n / 2;
    const bool cl = cluster || !partial;
    const int nsl = slices > 0 ? slices : orbit_slices(g, cl);
    const int csz = blocks > 0 ? blocks : nsl;
    const bool al = g->ld == g->n_bins;
    const int ld = plain ? g->n_bins : g->ld;
    const size_t NN = (size_t)g->n * g->n;
    const float4 *trig = g->d_trig;
    const dim3 th(ORB_T, ORB_TY);
    auto launch = [&](auto form, const float *yi, float *o, const float *xi, dim3 grd) {
        constexpr int FORM = decltype(form)::value;
        if (csz < nsl) {
            // fewer blocks than slices
            const size_t smem = orbit_smem(g->n_views / 2 / csz + 1, orbit_kept_sets(nsl, csz));
            counted();
            if (csz > 1)
                launch_kernel_cluster(k_backproject_orbit_seq<FORM, true>, grd, th, smem, st, dim3(1, 1, csz), yi, ld,
                                      trig, g->n, g->n_views, g->n_bins, nsl, csz, o);
            else
                launch_kernel(k_backproject_orbit_seq<FORM, false>, grd, th, smem, st, yi, ld, trig, g->n, g->n_views,
                              g->n_bins, nsl, csz, o);
            return;
        }
        if (nsl > 1 && cl) {
            // several slices: their sums are added in a cluster of the slices' blocks
            counted();
            launch_kernel_cluster(k_backproject_orbit_cl<FORM>, grd, th, orbit_smem(), st, dim3(1, 1, nsl), yi, ld, trig,
                                  g->n, g->n_views, g->n_bins, nsl, mode != 0 ? 1 : 0, o, xi, scal);
            return;
        }
        // one slice: the block's sums are complete and it writes the result;
        // several slices without a cluster: slice images, then k_orbit_reduce
        const int fin = nsl == 1 ? 1 + (mode != 0) : 0;
        counted(fin ? 1 : 2);
        launch_kernel(k_backproject_orbit<FORM>, grd, th, orbit_smem(), st, yi, ld, partial, trig, g->n, g->n_views,
                      g->n_bins, nsl, fin, o, xi, scal);
        if (fin) return;
        launch_kernel(mode == 0 ? k_orbit_reduce<0> : k_orbit_reduce<1>,
                      dim3((unsigned)((NN + 255) / 256), grd.z / nsl), dim3(256), 0, st, (const float *)partial, o, xi,
                      scal, NN, nsl);
    };
    // grid.z holds 65535: larger batches go in several launches
    const int most = 65535 / csz;
    for (int i0 = 0; i0 < batch; i0 += most) {
        const dim3 grd((q + ORB_T - 1) / ORB_T, (q + ORB_T - 1) / ORB_T, csz * std::min(most, batch - i0));
        const float *yi = y + (size_t)i0 * g->n_views * ld, *xi = xin ? xin + i0 * NN : nullptr;
        float *o = out + i0 * NN;
        if (plain && al) launch(std::integral_constant<int, ORB_PLAIN4>{}, yi, o, xi, grd);
        else if (plain) launch(std::integral_constant<int, ORB_PLAIN>{}, yi, o, xi, grd);
        else if (al) launch(std::integral_constant<int, ORB_PAIR4>{}, yi, o, xi, grd);
        else launch(std::integral_constant<int, ORB_PAIR>{}, yi, o, xi, grd);
    }
}

void launch_backproject(const Geometry *g, const float *y, float *out, int mode,
                        const float *xin, const double *scal, int batch, cudaStream_t st)
{
    dim3 grd((g->n + BT - 1) / BT, (g->n + BT - 1) / BT, batch);
    counted();
    if (mode == 0)
        k_backproject_tiles<0><<<grd, BTH, 0, st>>>(y, out, g->d_trig, g->n, g->n_views, g->n_bins, xin, scal);
    else
        k_backproject_tiles<1><<<grd, BTH, 0, st>>>(y, out, g->d_trig, g->n, g->n_views, g->n_bins, xin, scal);
}

void kernel_attrs_joseph(const Geometry *g)
{
    cudaFuncSetAttribute(k_project_direct, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (int)(DIRECT_BANDS * quad_smem(2 * MR * DIRECT_BANDS) + sizeof(float4) * DIRECT_THREADS));
    auto orbit_attrs = [](auto form) {
        constexpr int FORM = decltype(form)::value;
        cudaFuncSetAttribute(k_backproject_orbit<FORM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)orbit_smem());
        cudaFuncSetAttribute(k_backproject_orbit_cl<FORM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)orbit_smem());
        // at most all base views with one set of kept sums, or half of them with three
        const int shared = (int)orbit_smem(4 * ORB_MAXS + 1, 3);
        cudaFuncSetAttribute(k_backproject_orbit_seq<FORM, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, shared);
        cudaFuncSetAttribute(k_backproject_orbit_seq<FORM, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, shared);
    };
    if (g->orbit && g->ld == g->n_bins) {
        orbit_attrs(std::integral_constant<int, ORB_PLAIN4>{});
        orbit_attrs(std::integral_constant<int, ORB_PAIR4>{});
    } else if (g->orbit) {
        orbit_attrs(std::integral_constant<int, ORB_PLAIN>{});
        orbit_attrs(std::integral_constant<int, ORB_PAIR>{});
    }
    for (auto k : {k_project_quad<2>, k_project_quad<4>})
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, QUAD_SMEM_MAX);
    for (auto k : {k_project_qbal<2, false>, k_project_qbal<2, true>, k_project_qbal<4, false>, k_project_qbal<4, true>})
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, QUAD_SMEM_MAX);
    cudaFuncSetAttribute(k_project_bands<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)proj_smem(8192));
    cudaFuncSetAttribute(k_project_bands<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)proj_smem(8192));
}

}  // namespace ctpd
