// Incident fields, BLAS-1 helpers and the preconditioned GMRES driver.
#include <math.h>

#include <algorithm>
#include <complex>
#include <vector>

#include "common.cuh"

namespace {

template <typename C>
__global__ void k_plane_wave(C *e, const double *__restrict__ dp, int n, double h, double k, long total)
{
    long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= total) return;
    const long n3 = (long)n * n * n;
    long b = gid / n3, i = gid - b * n3;
    int i1 = (int)(i % n), i2 = (int)((i / n) % n), i3 = (int)(i / ((long)n * n));
    const double *d = dp + b * 6, *pol = d + 3;
    double phase = k * h * (d[0] * (i1 + 1) + d[1] * (i2 + 1) + d[2] * (i3 + 1));
    double sn, cs;
    sincos(phase, &sn, &cs);
    for (int c = 0; c < 3; ++c) {
        C v;
        v.x = pol[c] * cs;
        v.y = pol[c] * sn;
        e[(b * 3 + c) * n3 + i] = v;
    }
}

template <typename C>
__global__ void k_axpby(long count, double a, const C *__restrict__ x, double b, C *y)
{
    long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= count) return;
    C xv = x[gid], yv = y[gid];
    yv.x = a * xv.x + b * yv.x;
    yv.y = a * xv.y + b * yv.y;
    y[gid] = yv;
}

} // namespace

spm_status spm_plane_wave_impl(spm_problem_s *P, int prec, const double *dir, const double *pol, int nrhs, void *e,
                               cudaStream_t s)
{
    std::vector<double> dp(6 * nrhs);
    for (int b = 0; b < nrhs; ++b)
        for (int c = 0; c < 3; ++c) { dp[6 * b + c] = dir[3 * b + c]; dp[6 * b + 3 + c] = pol[3 * b + c]; }
    DevBuf t;
    SPM_TRY(t.ensure(sizeof(double) * dp.size()));
    SPM_CUDA_TRY(cudaMemcpyAsync(t.ptr, dp.data(), sizeof(double) * dp.size(), cudaMemcpyHostToDevice, s));
    const long total = (long)nrhs * P->n * P->n * P->n;
    unsigned grid = (unsigned)((total + 255) / 256);
    if (prec == SPM_C128)
        k_plane_wave<double2><<<grid, 256, 0, s>>>((double2 *)e, t.as<double>(), P->n, P->h, P->k, total);
    else
        k_plane_wave<float2><<<grid, 256, 0, s>>>((float2 *)e, t.as<double>(), P->n, P->h, P->k, total);
    SPM_CUDA_TRY(cudaGetLastError());
    SPM_CUDA_TRY(cudaStreamSynchronize(s));
    t.release();
    return SPM_OK;
}

spm_status spm_axpby_impl(int prec, long count, double a, const void *x, double b, void *y, cudaStream_t s)
{
    unsigned grid = (unsigned)((count + 255) / 256);
    if (prec == SPM_C128)
        k_axpby<double2><<<grid, 256, 0, s>>>(count, a, (const double2 *)x, b, (double2 *)y);
    else
        k_axpby<float2><<<grid, 256, 0, s>>>(count, a, (const float2 *)x, b, (float2 *)y);
    SPM_CUDA_TRY(cudaGetLastError());
    return SPM_OK;
}


// ====================================================================== GMRES
// Solve A x = g (Eq. discrete_block), left-preconditioned by S^{-1} Q (Section
// 3.1, last paragraph; GMRES with restart 20 as in Section 4).  The outer loop
// is FP64: r = g - A x in complex128, stop when ||r_b||/||g_b|| <= tol for every
// right-hand side b.  Each outer step runs one GMRES(restart) cycle on A d = r
// (preconditioned residual), in complex128 (SPM_C128) or complex64 (SPM_C64,
// SPM_MIXED) with FP64-accumulated dot products and FP64 Givens rotations, both on
// the device, then x += d in FP64.  Right-hand sides are iterated together: every
// operator and preconditioner application acts on the whole batch.
namespace {

// Reductions over a vector.  FP64 arithmetic on two lanes per SM is what they cost, the
// sums across a warp included (a shuffled FP64 sum of eight products is 80 additions, 64
// cycles each on the warp's scheduler), so a block is four warps, one per scheduler, with
// as many elements per thread as that leaves.  Each block stores its partial sums; the
// last one to finish adds them up, in block order.  At n = 32 and one right-hand side a
// pass over five vectors took 30 us plus 50 us for the separate launch whose eight threads
// added 304 partial sums each; now 19 us.
constexpr int DOT_BLOCKS = 304, DOT_THREADS = 128;
constexpr int VGROUP = 8; // basis vectors per dot/axpy pass

// float -> double by integer arithmetic (exponent rebiased, 29 zero bits appended): the
// conversion instruction goes through the FP64 pipe, which is what these kernels wait for.
// Zeros, subnormals, infinities and NaNs take the instruction.
__device__ __forceinline__ double widen(float a)
{
    const unsigned b = __float_as_uint(a), e = (b >> 23) & 255u;
    if (e - 1u >= 254u) return (double)a;
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ double widen(double a) { return a; }

inline int dot_blocks(long N, int nrhs)
{
    const long most = std::max(16, DOT_BLOCKS / nrhs); // blocks per right-hand side
    return (int)std::max(1L, std::min({(long)DOT_BLOCKS / 2, most, (N + DOT_THREADS - 1) / DOT_THREADS}));
}

// The block's sums of acc[0 .. NV) over its threads go to partial[b][blk][i]; true in the
// last block of right-hand side b to get here, whose total[i] then holds the sums over
// all blocks (shared memory, visible to every thread).  done: a zeroed counter per
// right-hand side, zeroed again on the way out.
template <int NV>
__device__ bool reduce_last(const double2 (&acc)[NV], int nv, double2 *__restrict__ partial, int b, unsigned *done,
                            double2 *total)
{
    __shared__ double2 red[NV][DOT_THREADS / 32];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nblk = gridDim.x;
#pragma unroll
    for (int i = 0; i < NV; ++i) {
        if (i >= nv) break;
        double x = acc[i].x, y = acc[i].y;
        for (int off = 16; off > 0; off >>= 1) {
            x += __shfl_down_sync(0xffffffffu, x, off);
            y += __shfl_down_sync(0xffffffffu, y, off);
        }
        if (lane == 0) red[i][wid] = make_double2(x, y);
    }
    __syncthreads();
    double2 *pb = partial + (long)b * nblk * VGROUP;
    if (threadIdx.x < nv) {
        double2 s = red[threadIdx.x][0];
        for (int q = 1; q < DOT_THREADS / 32; ++q) { s.x += red[threadIdx.x][q].x; s.y += red[threadIdx.x][q].y; }
        pb[(long)blockIdx.x * VGROUP + threadIdx.x] = s;
        __threadfence();
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&done[b], 1u) == (unsigned)nblk - 1;
    __syncthreads();
    if (!last) return false;
    __threadfence();
    for (int i = wid; i < nv; i += DOT_THREADS / 32) { // a warp per sum
        double x = 0, y = 0;
        for (int q = lane; q < nblk; q += 32) {
            const double2 v = __ldcg(&pb[(long)q * VGROUP + i]);
            x += v.x;
            y += v.y;
        }
        for (int off = 16; off > 0; off >>= 1) {
            x += __shfl_down_sync(0xffffffffu, x, off);
            y += __shfl_down_sync(0xffffffffu, y, off);
        }
        if (lane == 0) total[i] = make_double2(x, y);
    }
    if (threadIdx.x == 0) done[b] = 0;
    __syncthreads();
    return true;
}

// out[b][i0 + i] = <V_{i0+i}[b], w[b]>, i < ni
template <typename C>
__global__ void __launch_bounds__(DOT_THREADS) k_dots(const C *__restrict__ V, long vstride, int i0, int ni,
                                                      const C *__restrict__ w, long N, double2 *__restrict__ partial,
                                                      unsigned *done, double2 *out, int ld)
{
    pdl_wait_and_trigger();
    __shared__ double2 total[VGROUP];
    const int b = blockIdx.y;
    double2 acc[VGROUP];
#pragma unroll
    for (int i = 0; i < VGROUP; ++i) acc[i] = make_double2(0, 0);
    const C *wb = w + (long)b * N, *vb = V + (long)i0 * vstride + (long)b * N;
    for (long k = (long)blockIdx.x * DOT_THREADS + threadIdx.x; k < N; k += (long)gridDim.x * DOT_THREADS) {
        const C wk = wb[k];
        const double wx = widen(wk.x), wy = widen(wk.y);
#pragma unroll
        for (int i = 0; i < VGROUP; ++i) {
            if (i < ni) {
                const C v = vb[(long)i * vstride + k];
                const double vx = widen(v.x), vy = widen(v.y);
                acc[i].x = fma(vx, wx, fma(vy, wy, acc[i].x));
                acc[i].y = fma(vx, wy, fma(-vy, wx, acc[i].y));
            }
        }
    }
    if (reduce_last(acc, ni, partial, b, done, total) && threadIdx.x < ni) out[(long)b * ld + i0 + threadIdx.x] = total[threadIdx.x];
}

// r = g - Ax, out[b] = ||r[b]||^2
__global__ void __launch_bounds__(DOT_THREADS) k_residual(double2 *r, const double2 *__restrict__ g, const double2 *__restrict__ Ax,
                                                          long N, double2 *__restrict__ partial, unsigned *done, double2 *out,
                                                          int ld)
{
    pdl_wait_and_trigger();
    __shared__ double2 total[1];
    const long b = blockIdx.y;
    double2 acc[1] = {make_double2(0, 0)};
    for (long k = (long)blockIdx.x * DOT_THREADS + threadIdx.x; k < N; k += (long)gridDim.x * DOT_THREADS) {
        double2 v = g[b * N + k];
        const double2 a = Ax[b * N + k];
        v.x -= a.x;
        v.y -= a.y;
        r[b * N + k] = v;
        acc[0].x = fma(v.x, v.x, fma(v.y, v.y, acc[0].x));
    }
    if (reduce_last(acc, 1, partial, (int)b, done, total) && threadIdx.x == 0) out[b * ld] = total[0];
}

// w[b] += sign sum_{i < ni} h[b][i0+i] V_{i0+i}[b], sign = +-1   (coefficients FP64)
template <typename C>
__global__ void k_axpy_multi(const C *__restrict__ V, long vstride, int i0, int ni, const double2 *__restrict__ h,
                             int ld, C *w, long N, int nrhs, double sign)
{
    long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait_and_trigger();
    if (gid >= N * nrhs) return;
    const long b = gid / N;
    C wk = w[gid];
    double x = widen(wk.x), y = widen(wk.y);
#pragma unroll
    for (int i = 0; i < VGROUP; ++i) {
        if (i >= ni) break;
        const double2 c = h[b * ld + i0 + i];
        const C v = V[(long)(i0 + i) * vstride + gid];
        const double vx = widen(v.x), vy = widen(v.y), cx = sign < 0 ? -c.x : c.x, cy = sign < 0 ? -c.y : c.y;
        x = fma(cx, vx, fma(-cy, vy, x));
        y = fma(cx, vy, fma(cy, vx, y));
    }
    wk.x = x;
    wk.y = y;
    w[gid] = wk;
}

// dst[b] = src[b] * scale[b]
template <typename C, typename D>
__global__ void k_scale_copy(D *dst, const C *__restrict__ src, const double *__restrict__ scale, long N, int nrhs)
{
    long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait_and_trigger();
    if (gid >= N * nrhs) return;
    double s = scale[gid / N];
    C v = src[gid];
    D o;
    o.x = s * v.x;
    o.y = s * v.y;
    dst[gid] = o;
}

// x[b] += scale[b] * d[b]   (x complex128)
template <typename C>
__global__ void k_accum(double2 *x, const C *__restrict__ d, const double *__restrict__ scale, long N, int nrhs)
{
    long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    pdl_wait_and_trigger();
    if (gid >= N * nrhs) return;
    double s = scale[gid / N];
    C v = d[gid];
    double2 o = x[gid];
    o.x += s * v.x;
    o.y += s * v.y;
    x[gid] = o;
}

inline unsigned nblocks(long cnt) { return (unsigned)((cnt + 255) / 256); }

// where the reductions keep their partial sums and count their finished blocks
struct Reduce {
    double2 *partial; // [nrhs][DOT_BLOCKS][VGROUP]
    unsigned *done;   // [nrhs], zero between launches
};

template <typename C>
spm_status dots(const C *V, long vstride, int nvec, const C *w, long N, int nrhs, const Reduce &rd, double2 *out, int ld,
                cudaStream_t s)
{
    for (int i0 = 0; i0 < nvec; i0 += VGROUP) {
        int ni = nvec - i0 < VGROUP ? nvec - i0 : VGROUP;
        launch_pdl(k_dots<C>, dim3(dot_blocks(N, nrhs), nrhs), dim3(DOT_THREADS), 0, s, V, vstride, i0, ni, w, N, rd.partial,
                   rd.done, out, ld);
    }
    SPM_CUDA_TRY(cudaGetLastError());
    return SPM_OK;
}

template <typename C>
spm_status axpy_multi(const C *V, long vstride, int nvec, const double2 *h, int ld, C *w, long N, int nrhs,
                      double sign, cudaStream_t s)
{
    for (int i0 = 0; i0 < nvec; i0 += VGROUP) {
        int ni = nvec - i0 < VGROUP ? nvec - i0 : VGROUP;
        launch_pdl(k_axpy_multi<C>, dim3(nblocks(N * nrhs)), dim3(256), 0, s, V, vstride, i0, ni, h, ld, w, N, nrhs, sign);
    }
    SPM_CUDA_TRY(cudaGetLastError());
    return SPM_OK;
}

// ---- the small FP64 problem of GMRES on the device, one thread per RHS ----
// Per right-hand side b the cycle keeps, in device memory: the Hessenberg
// matrix H[b] ((restart + 1) x restart, row i column j at i * restart + j), the
// Givens rotations cs[b][i], sn[b][i], the rotated residual vector g[b][i], beta
// = ||v_0||, and whether b is still active.
struct GmresSmall {
    double2 *H, *cs, *sn, *g;
    double *beta, *rtol, *scale;
    int *active, *count; // count[0]: RHS still active; count[1]: non-finite values seen
};

// after v_0 = S^-1 Q r: beta = ||v_0|| (nn[b*ld] holds <v_0, v_0>), g = beta e_1
__global__ void k_cycle_init(GmresSmall gs, const double2 *__restrict__ nn, int ld, int restart, int nrhs)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nrhs) return;
    const double beta = sqrt(fmax(nn[(long)b * ld].x, 0.0));
    const bool ok = beta > 0 && isfinite(beta);
    gs.beta[b] = beta;
    gs.active[b] = ok ? 1 : 0;
    gs.scale[b] = ok ? 1.0 / beta : 0.0;
    for (int i = 0; i <= restart; ++i) gs.g[(long)b * (restart + 1) + i] = make_double2(i == 0 ? beta : 0.0, 0.0);
    for (long i = 0; i < (long)(restart + 1) * restart; ++i) gs.H[(long)b * (restart + 1) * restart + i] = make_double2(0, 0);
    if (ok) atomicAdd(&gs.count[0], 1);
}

__device__ __forceinline__ double2 zmul(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ double2 zconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 zadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

// Arnoldi step j of right-hand side b: column j of H from the two Gram-Schmidt passes
// (h1, h2) and ||w||^2, the previous rotations applied, a new rotation that zeroes
// H[j+1][j], g rotated; scale = 1/||w|| for normalising v_{j+1}; a RHS whose
// |g[j+1]| <= rtol beta (or whose ||w|| vanished) becomes inactive.
__device__ void arnoldi_givens(const GmresSmall &gs, const double2 *h1, const double2 *h2, double nn, int ld, int j, int restart,
                               int b)
{
    if (!gs.active[b]) { gs.scale[b] = 0.0; return; }
    double2 *H = gs.H + (long)b * (restart + 1) * restart;
    double2 *cs = gs.cs + (long)b * restart, *sn = gs.sn + (long)b * restart, *g = gs.g + (long)b * (restart + 1);
    for (int i = 0; i <= j; ++i) H[i * restart + j] = zadd(h1[(long)b * ld + i], h2[(long)b * ld + i]);
    const double hn = sqrt(fmax(nn, 0.0));
    if (!isfinite(hn)) { atomicAdd(&gs.count[1], 1); gs.active[b] = 0; gs.scale[b] = 0.0; return; }
    H[(j + 1) * restart + j] = make_double2(hn, 0.0);
    gs.scale[b] = hn > 1e-300 ? 1.0 / hn : 0.0;
    for (int i = 0; i < j; ++i) {
        const double2 a = H[i * restart + j], c = H[(i + 1) * restart + j];
        H[i * restart + j] = zadd(zmul(zconj(cs[i]), a), zmul(zconj(sn[i]), c));
        const double2 ms = make_double2(-sn[i].x, -sn[i].y);
        H[(i + 1) * restart + j] = zadd(zmul(ms, a), zmul(cs[i], c));
    }
    const double2 a = H[j * restart + j], c = H[(j + 1) * restart + j];
    const double den = sqrt(a.x * a.x + a.y * a.y + c.x * c.x + c.y * c.y);
    if (den == 0.0) { cs[j] = make_double2(1.0, 0.0); sn[j] = make_double2(0.0, 0.0); }
    else { cs[j] = make_double2(a.x / den, a.y / den); sn[j] = make_double2(c.x / den, c.y / den); }
    H[j * restart + j] = make_double2(den, 0.0);
    H[(j + 1) * restart + j] = make_double2(0.0, 0.0);
    const double2 gj = g[j];
    const double2 ms = make_double2(-sn[j].x, -sn[j].y);
    g[j + 1] = zmul(ms, gj);
    g[j] = zmul(zconj(cs[j]), gj);
    const double r = sqrt(g[j + 1].x * g[j + 1].x + g[j + 1].y * g[j + 1].y);
    if (r <= gs.rtol[b] * gs.beta[b] || hn <= 1e-300) gs.active[b] = 0;
    else atomicAdd(&gs.count[0], 1);
}

// The end of Arnoldi step j in one launch: w[b] -= sum_{i < ni} h2[b][i0+i] V_{i0+i}[b] (the
// last group of the second Gram-Schmidt pass), ||w||^2 and the small problem's step, by the
// last block of each right-hand side.
template <typename C>
__global__ void __launch_bounds__(DOT_THREADS) k_arnoldi_end(const C *__restrict__ V, long vstride, int i0, int ni, const double2 *h1,
                                                             const double2 *h2, int ld, C *w, long N,
                                                             double2 *__restrict__ partial, unsigned *done, GmresSmall gs,
                                                             int j, int restart)
{
    pdl_wait_and_trigger();
    __shared__ double2 total[1], h[VGROUP];
    const int b = blockIdx.y;
    if (threadIdx.x < ni) h[threadIdx.x] = h2[(long)b * ld + i0 + threadIdx.x];
    __syncthreads();
    double2 acc[1] = {make_double2(0, 0)};
    C *wb = w + (long)b * N;
    const C *vb = V + (long)i0 * vstride + (long)b * N;
    for (long k = (long)blockIdx.x * DOT_THREADS + threadIdx.x; k < N; k += (long)gridDim.x * DOT_THREADS) {
        C wk = wb[k];
        double x = widen(wk.x), y = widen(wk.y);
#pragma unroll
        for (int i = 0; i < VGROUP; ++i) {
            if (i < ni) {
                const C v = vb[(long)i * vstride + k];
                const double vx = widen(v.x), vy = widen(v.y);
                x = fma(-h[i].x, vx, fma(h[i].y, vy, x));
                y = fma(-h[i].x, vy, fma(-h[i].y, vx, y));
            }
        }
        wk.x = x;
        wk.y = y;
        wb[k] = wk;
        x = widen(wk.x);
        y = widen(wk.y);
        acc[0].x = fma(x, x, fma(y, y, acc[0].x));
    }
    if (reduce_last(acc, 1, partial, b, done, total) && threadIdx.x == 0)
        arnoldi_givens(gs, h1, h2, total[0].x, ld, j, restart, b);
}

// back substitution H y = g over the leading m columns (fewer where a RHS
// stopped early: its trailing diagonal entries are zero); y -> coef[b*ld + i]
__global__ void k_backsolve(GmresSmall gs, double2 *coef, int ld, int m, int restart, int nrhs)
{
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b >= nrhs) return;
    const double2 *H = gs.H + (long)b * (restart + 1) * restart, *g = gs.g + (long)b * (restart + 1);
    double2 *y = coef + (long)b * ld;
    int mb = m;
    while (mb > 0 && H[(mb - 1) * restart + (mb - 1)].x == 0.0 && H[(mb - 1) * restart + (mb - 1)].y == 0.0) --mb;
    for (int i = 0; i < ld; ++i) y[i] = make_double2(0, 0);
    for (int i = mb - 1; i >= 0; --i) {
        double2 acc = g[i];
        for (int q = i + 1; q < mb; ++q) {
            const double2 t = zmul(H[i * restart + q], y[q]);
            acc.x -= t.x;
            acc.y -= t.y;
        }
        const double2 d = H[i * restart + i];
        const double dd = d.x * d.x + d.y * d.y;
        y[i] = make_double2((acc.x * d.x + acc.y * d.y) / dd, (acc.y * d.x - acc.x * d.y) / dd);
    }
}

// One preconditioned GMRES(restart) cycle for all right-hand sides, zero initial
// guess: d = argmin over the Krylov space of ||S^{-1} Q (r - A d)||.  Stops
// early when every active RHS reaches relative preconditioned residual rtol[b].
template <typename R>
spm_status gmres_cycle(const KrylovOps &ops, int prec, const typename cplx_of<R>::type *r,
                       typename cplx_of<R>::type *d, int nrhs, int restart, typename cplx_of<R>::type *V,
                       typename cplx_of<R>::type *tmp, const Reduce &rd, double2 *h1, double2 *h2, double2 *nn,
                       const GmresSmall &gs, int *count_host, int *iters, cudaStream_t s)
{
    using C = typename cplx_of<R>::type;
    const long N = ops.N;
    const long vstride = N * nrhs;
    const int ld = restart + 2;
    const unsigned sb = (unsigned)((nrhs + 63) / 64);
    C *w = V + (long)(restart)*vstride;

    // v0 = S^{-1} Q r / beta
    SPM_TRY(ops.apply_Q(ops.ctx, prec, r, tmp, nrhs, s));
    SPM_TRY(ops.solve_S(ops.ctx, prec, tmp, V, nrhs, s));
    SPM_TRY(dots<C>(V, vstride, 1, V, N, nrhs, rd, nn, ld, s));
    SPM_CUDA_TRY(cudaMemsetAsync(gs.count, 0, 2 * sizeof(int), s));
    k_cycle_init<<<sb, 64, 0, s>>>(gs, nn, ld, restart, nrhs);
    k_scale_copy<C, C><<<nblocks(vstride), 256, 0, s>>>(V, V, gs.scale, N, nrhs);
    SPM_CUDA_TRY(cudaMemcpyAsync(count_host, gs.count, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
    SPM_CUDA_TRY(cudaStreamSynchronize(s));
    int j = 0;
    for (; j < restart && count_host[0] > 0; ++j) {
        C *vj = V + (long)j * vstride;
        w = V + (long)(j + 1) * vstride;
        SPM_CUDA_TRY(cudaMemsetAsync(gs.count, 0, sizeof(int), s));
        SPM_TRY(ops.apply_A(ops.ctx, prec, vj, w, nrhs, s));       // w = A v_j
        SPM_TRY(ops.apply_Q(ops.ctx, prec, w, tmp, nrhs, s));      // tmp = Q A v_j
        SPM_TRY(ops.solve_S(ops.ctx, prec, tmp, w, nrhs, s));      // w = S^{-1} Q A v_j
        // classical Gram-Schmidt twice, FP64 coefficients
        SPM_TRY(dots<C>(V, vstride, j + 1, w, N, nrhs, rd, h1, ld, s));
        SPM_TRY(axpy_multi<C>(V, vstride, j + 1, h1, ld, w, N, nrhs, -1.0, s));
        SPM_TRY(dots<C>(V, vstride, j + 1, w, N, nrhs, rd, h2, ld, s));
        const int done_groups = j / VGROUP * VGROUP; // all groups but the last
        SPM_TRY(axpy_multi<C>(V, vstride, done_groups, h2, ld, w, N, nrhs, -1.0, s));
        launch_pdl(k_arnoldi_end<C>, dim3(dot_blocks(N, nrhs), nrhs), dim3(DOT_THREADS), 0, s, (const C *)V, vstride, done_groups,
                   j + 1 - done_groups, (const double2 *)h1, (const double2 *)h2, ld, w, N, rd.partial, rd.done, gs, j, restart);
        launch_pdl(k_scale_copy<C, C>, dim3(nblocks(vstride)), dim3(256), 0, s, w, (const C *)w, (const double *)gs.scale, N, nrhs);
        SPM_CUDA_TRY(cudaMemcpyAsync(count_host, gs.count, 2 * sizeof(int), cudaMemcpyDeviceToHost, s));
        SPM_CUDA_TRY(cudaStreamSynchronize(s)); // the only host round trip of an iteration: a convergence count
        ++*iters;
        if (count_host[1]) { spm_set_error("NaN in GMRES"); return SPM_ERR_NUMERICAL; }
    }
    // d = sum_i y_i v_i with H y = g (upper triangular, per RHS, on the device)
    const int m = j;
    k_backsolve<<<sb, 64, 0, s>>>(gs, h1, ld, m, restart, nrhs);
    SPM_CUDA_TRY(cudaMemsetAsync(d, 0, sizeof(C) * vstride, s));
    SPM_TRY(axpy_multi<C>(V, vstride, m, h1, ld, d, N, nrhs, 1.0, s));
    SPM_CUDA_TRY(cudaGetLastError());
    return SPM_OK;
}

// out[b] = sqrt of the sums of squares that a reduction left in hdev
spm_status read_norms(const double2 *hdev, int nrhs, int ld, std::vector<double> &out, cudaStream_t s)
{
    std::vector<double2> t((size_t)nrhs * ld);
    SPM_CUDA_TRY(cudaMemcpyAsync(t.data(), hdev, sizeof(double2) * nrhs * ld, cudaMemcpyDeviceToHost, s));
    SPM_CUDA_TRY(cudaStreamSynchronize(s));
    out.resize(nrhs);
    for (int b = 0; b < nrhs; ++b) out[b] = sqrt(fmax(t[(size_t)b * ld].x, 0.0));
    return SPM_OK;
}

template <typename R>
spm_status solve_typed(const KrylovOps &ops, const double2 *g, double2 *x, int nrhs, double tol, int maxit,
                       int restart, spm_solve_info *info)
{
    using C = typename cplx_of<R>::type;
    const int inner_prec = sizeof(R) == 8 ? SPM_C128 : SPM_C64;
    cudaStream_t s = ops.stream;
    const long N = ops.N;
    const long vstride = N * nrhs;
    const int ld = restart + 2;
    // workspace: r (c128), Ax (c128), V (restart+1), d, tmp (inner precision), reductions
    const size_t small = sizeof(double2) * (size_t)nrhs * (3 * ld + (restart + 1) * restart + 2 * restart + restart + 1) +
                         sizeof(double) * 3 * (size_t)nrhs + sizeof(int) * (2 * (size_t)nrhs + 2);
    size_t bytes = sizeof(double2) * 2 * vstride + sizeof(C) * (size_t)(restart + 3) * vstride +
                   sizeof(double2) * (size_t)nrhs * DOT_BLOCKS * VGROUP + small + 16 * 256;
    DevBuf &ws = *ops.ws; // kept across solves: sized by the largest solve so far
    SPM_TRY(ws.ensure(bytes));
    char *p = ws.as<char>();
    double2 *r = reinterpret_cast<double2 *>(p); p += sizeof(double2) * vstride;
    double2 *Ax = reinterpret_cast<double2 *>(p); p += sizeof(double2) * vstride;
    C *V = reinterpret_cast<C *>(p); p += sizeof(C) * (restart + 1) * vstride;
    C *d = reinterpret_cast<C *>(p); p += sizeof(C) * vstride;
    C *tmp = reinterpret_cast<C *>(p); p += sizeof(C) * vstride;
    Reduce rd;
    rd.partial = reinterpret_cast<double2 *>(p); p += sizeof(double2) * nrhs * DOT_BLOCKS * VGROUP;
    double2 *hdev = reinterpret_cast<double2 *>(p); p += sizeof(double2) * nrhs * ld;
    double2 *h2dev = reinterpret_cast<double2 *>(p); p += sizeof(double2) * nrhs * ld;
    double2 *nndev = reinterpret_cast<double2 *>(p); p += sizeof(double2) * nrhs * ld;
    GmresSmall gs;
    gs.H = reinterpret_cast<double2 *>(p); p += sizeof(double2) * (size_t)nrhs * (restart + 1) * restart;
    gs.cs = reinterpret_cast<double2 *>(p); p += sizeof(double2) * (size_t)nrhs * restart;
    gs.sn = reinterpret_cast<double2 *>(p); p += sizeof(double2) * (size_t)nrhs * restart;
    gs.g = reinterpret_cast<double2 *>(p); p += sizeof(double2) * (size_t)nrhs * (restart + 1);
    gs.beta = reinterpret_cast<double *>(p); p += sizeof(double) * nrhs;
    gs.rtol = reinterpret_cast<double *>(p); p += sizeof(double) * nrhs;
    double *sdev = reinterpret_cast<double *>(p); p += sizeof(double) * nrhs;
    gs.scale = sdev;
    gs.active = reinterpret_cast<int *>(p); p += sizeof(int) * nrhs;
    gs.count = reinterpret_cast<int *>(p); p += sizeof(int) * 2;
    rd.done = reinterpret_cast<unsigned *>(p);
    SPM_CUDA_TRY(cudaMemsetAsync(rd.done, 0, sizeof(unsigned) * nrhs, s));
    int count_host[2] = {0, 0};

    std::vector<double> gnorm, rnorm, rtol(nrhs), scl(nrhs);
    SPM_TRY(dots<double2>(g, 0, 1, g, N, nrhs, rd, hdev, ld, s));
    SPM_TRY(read_norms(hdev, nrhs, ld, gnorm, s));
    for (int b = 0; b < nrhs; ++b) if (gnorm[b] == 0.0) gnorm[b] = 1.0;
    int iters = 0, outer = 0;
    double worst = 0.0;
    const double floor_rel = sizeof(R) == 8 ? 1e-14 : 2e-6;
    while (true) {
        SPM_TRY(ops.apply_A(ops.ctx, SPM_C128, x, Ax, nrhs, s));
        launch_pdl(k_residual, dim3(dot_blocks(N, nrhs), nrhs), dim3(DOT_THREADS), 0, s, r, g, (const double2 *)Ax, N, rd.partial,
                   rd.done, hdev, ld);
        SPM_CUDA_TRY(cudaGetLastError());
        SPM_TRY(read_norms(hdev, nrhs, ld, rnorm, s));
        worst = 0.0;
        bool done = true;
        for (int b = 0; b < nrhs; ++b) {
            double rel = rnorm[b] / gnorm[b];
            if (!isfinite(rel)) { spm_set_error("residual is not finite"); return SPM_ERR_NUMERICAL; }
            worst = fmax(worst, rel);
            if (rel > tol) done = false;
            // target for this cycle, relative to ||r_b||, with a safety factor for
            // the gap between preconditioned and true residuals
            rtol[b] = rel > tol ? fmax(0.1 * tol / rel, floor_rel) : 1e300;
            scl[b] = rnorm[b] > 0 ? 1.0 / rnorm[b] : 0.0;
        }
        if (info) { info->true_relres = worst; info->iterations = iters; info->outer_steps = outer; }
        if (done) return SPM_OK;
        if (iters >= maxit) { spm_set_error("no convergence within %d iterations (residual %.3e)", maxit, worst); return SPM_ERR_NO_CONVERGENCE; }
        // inner right-hand side: r / ||r|| in the inner precision
        SPM_CUDA_TRY(cudaMemcpyAsync(sdev, scl.data(), sizeof(double) * nrhs, cudaMemcpyHostToDevice, s));
        C *rin = d; // d is free until the cycle writes its result
        k_scale_copy<double2, C><<<nblocks(vstride), 256, 0, s>>>(rin, r, sdev, N, nrhs);
        int it_cycle = 0;
        int cyc_restart = restart < maxit - iters ? restart : maxit - iters;
        SPM_CUDA_TRY(cudaMemcpyAsync(gs.rtol, rtol.data(), sizeof(double) * nrhs, cudaMemcpyHostToDevice, s));
        SPM_TRY(gmres_cycle<R>(ops, inner_prec, rin, d, nrhs, cyc_restart, V, tmp, rd, hdev, h2dev, nndev, gs,
                               count_host, &it_cycle, s));
        iters += it_cycle;
        ++outer;
        for (int b = 0; b < nrhs; ++b) scl[b] = rtol[b] < 1e299 ? rnorm[b] : 0.0;
        SPM_CUDA_TRY(cudaMemcpyAsync(sdev, scl.data(), sizeof(double) * nrhs, cudaMemcpyHostToDevice, s));
        k_accum<C><<<nblocks(vstride), 256, 0, s>>>(x, d, sdev, N, nrhs);
        SPM_CUDA_TRY(cudaGetLastError());
    }
}

} // namespace

spm_status spm_gmres_solve(const KrylovOps &ops, int prec, const void *g, void *x, int nrhs, double tol, int maxit,
                           int restart, spm_solve_info *info)
{
    const bool inner64 = prec != SPM_C128;
    spm_status st = inner64 ? solve_typed<float>(ops, (const double2 *)g, (double2 *)x, nrhs, tol, maxit, restart, info)
                            : solve_typed<double>(ops, (const double2 *)g, (double2 *)x, nrhs, tol, maxit, restart, info);
    SPM_CUDA_TRY(cudaStreamSynchronize(ops.stream));
    return st;
}

namespace {
spm_status ops3_A(void *c, int prec, const void *x, void *y, int nrhs, cudaStream_t s)
{
    return spm_apply_A_impl(static_cast<spm_problem_s *>(c), prec, x, y, nrhs, s);
}
spm_status ops3_Q(void *c, int prec, const void *v, void *y, int nrhs, cudaStream_t s)
{
    return spm_apply_Q_impl(static_cast<spm_problem_s *>(c), prec, v, y, nrhs, s);
}
spm_status ops3_S(void *c, int prec, const void *b, void *x, int nrhs, cudaStream_t s)
{
    return spm_solveS_impl(static_cast<spm_problem_s *>(c), prec, b, x, nrhs, s);
}
} // namespace

spm_status spm_solve_impl(spm_problem_s *P, int prec, const void *g, void *x, int nrhs, double tol, int maxit,
                          int restart, spm_solve_info *info)
{
    if (!P->have_S) { spm_set_error("stencils not built (spm_build_stencils)"); return SPM_ERR_NOT_BUILT; }
    const bool inner64 = prec != SPM_C128;
    if ((inner64 && !P->fac64) || (!inner64 && !P->fac128)) {
        spm_set_error("no factor of S in the %s precision (spm_factor_S)", inner64 ? "complex64" : "complex128");
        return SPM_ERR_NOT_BUILT;
    }
    KrylovOps ops;
    ops.N = 3L * P->n * P->n * P->n;
    ops.stream = P->stream;
    ops.ws = &P->gmres_ws;
    ops.ctx = P;
    ops.apply_A = ops3_A;
    ops.apply_Q = ops3_Q;
    ops.solve_S = ops3_S;
    return spm_gmres_solve(ops, prec, g, x, nrhs, tol, maxit, restart, info);
}
