// Nested-dissection multifrontal LU of the sparse system S (Section 3.1: the
// sparse system "can be solved efficiently by the nested dissection
// algorithm"; complexity in Section 3.3).
//
// Geometric dissection: a box of grid points is cut by one plane normal to its
// longest axis (a line on a 2-D grid); one plane separates because S couples
// only points with ||j - i||_inf <= 1.  The grid, the unknowns per point and the
// block layout of S come from a SparseSys (3-D: n^3 points, 3 unknowns, 27
// neighbours; 2-D variant: n^2 points, 2 unknowns, 9 neighbours).  Node = box B.  Its own unknowns are the separator plane
// (or every point of B for a leaf); its boundary unknowns are the points
// outside B within distance 1 of B, which all lie on ancestor separators.  The
// front is [own; boundary] x [own; boundary]:
//   original rows and columns of the own unknowns are assembled from S,
//   children's Schur complements are extend-added,
//   F11 = P L U (partial pivoting inside the own block),
//   X = F11^{-1} F12,   update = F22 - F21 X  -> parent.
// Each node keeps G = [F11^{-1}; F21 F11^{-1}] (front x own) and X = F11^{-1} F12,
// in the factor's precision or (SPM_C64H) as binary16 pairs scaled per column by
// the column's largest component, which halves the bytes every solve reads.
// Solve, one launch per tree level and direction (k_nd_level): nodes of one level
// have disjoint own unknowns, and their boundaries lie on shallower separators.  Dense front
// work (dense.cu): F11^{-1} by Gauss-Jordan with partial pivoting, then
// X = F11^{-1} F12, F21 F11^{-1} and the update F22 - F21 X as complex GEMMs;
// assembly, extend-add and the solve's levels are kernels here.
#include <cuda_fp16.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>
#include <vector>

#include "common.cuh"

namespace {

struct Node {
    int lo[3], hi[3];     // box [lo, hi) of grid points
    int axis = -1, cut = -1; // separator plane (axis, coordinate); -1 for a leaf
    int left = -1, right = -1;
    int nown = 0, nbnd = 0;  // points
    long own_off = 0, bnd_off = 0; // offsets into the point lists
    long map_off = 0;        // offset of the local map over the expanded box
    int elo[3], ehi[3];      // expanded box (B grown by 1, clipped)
    long rel_off = 0;        // offset of the child-bnd -> parent-front map (unknowns)
    long fac_off = 0;        // persistent factor storage (elements)
    long piv_off = 0;        // pivots
    long scale_off = 0;      // per-column scales of G then X (half storage)
    int depth = 0;
};

// ---------------------------------------------------------------- kernels

// Assemble the own rows and own columns of S into a zeroed front (column-major,
// ld = f); unknown (point a, component c) of the front is D a + c.
struct GridDesc {
    int n1, n2, n3, D, nsten;
};

template <typename C>
__global__ void k_front_assemble(C *F, int f, const C *__restrict__ S, const int *__restrict__ own_pts, int nown,
                                 const int *__restrict__ lmap, int e0, int e1, int e2, int ew0, int ew1, GridDesc g)
{
    int gid = blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= nown * g.nsten) return;
    const int D = g.D, DD = g.D * g.D;
    int a = gid / g.nsten, s = gid % g.nsten;
    int o1 = s % 3 - 1, o2 = (s / 3) % 3 - 1, o3 = g.nsten == 27 ? s / 9 - 1 : 0;
    int i = own_pts[a];
    int i1 = i % g.n1, i2 = (i / g.n1) % g.n2, i3 = i / (g.n1 * g.n2);
    int j1 = i1 + o1, j2 = i2 + o2, j3 = i3 + o3;
    if (j1 < 0 || j2 < 0 || j3 < 0 || j1 >= g.n1 || j2 >= g.n2 || j3 >= g.n3) return;
    int lj = lmap[((j3 - e2) * ew1 + (j2 - e1)) * ew0 + (j1 - e0)];
    if (lj < 0) return; // neighbour eliminated in a child subtree
    long j = ((long)j3 * g.n2 + j2) * g.n1 + j1;
    const C *blk = S + ((long)i * g.nsten + s) * DD; // rows (i,c), columns (j,f)
    for (int c = 0; c < D; ++c)
        for (int q = 0; q < D; ++q) F[(long)(D * lj + q) * f + D * a + c] = blk[c * D + q];
    if (lj >= nown) { // row of a boundary unknown j, column of own unknown i
        int sr = g.nsten - 1 - s; // offset -o
        const C *bj = S + (j * g.nsten + sr) * DD;
        for (int c = 0; c < D; ++c)
            for (int q = 0; q < D; ++q) F[(long)(D * a + q) * f + D * lj + c] = bj[c * D + q];
    }
}

// ---- batched fronts: a level's fronts advance together, panel by panel
// A front of f unknowns (o3 own first) is assembled from S and the children's updates,
// then swept by Gauss-Jordan over its o3 own pivots with partial pivoting among the own
// rows (row swaps) and the static pivot floor: after the sweep the front holds
// [(P F11)^-1, F11^-1 F12; -F21 (P F11)^-1, F22 - F21 F11^-1 F12], from which
// G = [F11^-1; F21 F11^-1] (columns put back in place), X = F11^-1 F12 and the update
// F22 - F21 X are stored: the same quantities as the per-front path (dense inverse and
// GEMMs).  Every front of a level lies in global scratch and takes one panel of BP_NB
// pivots at a time, K its rows and columns:
//   k_bp_panel   (a block per front) the steps on the unpivoted own rows of the panel's
//                columns, in shared memory
//   k_bp_cross   the same steps on the other rows of the panel's columns, and on the
//                pivot rows of the other columns (where it also swaps the rows)
//   k_bp_update  the same steps on everything else: A[i][j] -= M[i][:] S[:][j]
// Step jj divides the pivot row by the pivot and subtracts the row's multiple M[i][jj]
// (the entry of the pivot's column before the step) from every other row i.  The first
// two kernels keep the multipliers M (moved along by later row swaps) and the scaled pivot
// rows S as each step leaves them, so every entry of the front sees the same operations in
// the same order as in an unblocked sweep.  (Forming P^-1 of the pivot block and adding the product
// of M P^-1 and the pivot rows is the same work in fewer steps, but its factors' probe
// residuals were 1.3 to 2 times as large.)
// Bound: the FP64 pipe for complex128 (4 o3 f^2 FMAs; two lanes per SM) and the chain of
// pivots.  With one block per front, the few fronts near the root had one SM each: of
// the 204 ms of a 2-D factor at n = 119 the last five levels took 192.  Spread over the
// chip the factor takes 14 ms (n = 239: 361 -> 137; 3-D complex64 n = 16: 86 -> 12,
// n = 32: 406 -> 231, n = 64: 5.5 -> 4.8 s; 3-D complex128 n = 16: 338 -> 79 ms).  At
// n = 119 the updates take 6 ms of it (their FP64 work alone 3.2), the panels' chains 3.2
// (4 us a pivot), k_bp_cross 1.2.
struct BatchFront {
    int own_off, nown, map_off, e0, e1, e2, ew0, ew1, f, o3, nch;
    int ch_bc[2], ch_rel[2];
    long fac_off;
    void *upd;
    const void *ch_upd[2];
};

constexpr int BP_NB = 8, BP_THREADS = 256;
constexpr int BATCH_LINES[] = {1536, 1024, 512}; // unknowns of the largest fronts batched
template <typename C> struct BatchPanel {
    C prow[BP_NB][BP_NB];               // scaled pivot row of each step ([jj][jj]: 1 / pivot)
    int nmove;                          // rows the panel's swaps gave new contents
    int dst[2 * BP_NB], src[2 * BP_NB]; // the first are the pivot rows
};

// The sweep's arithmetic, rounding fixed: a - m b with the product first (six FP64
// instructions where chained FMAs would be four, but the factors' residuals are smaller,
// 0.85 of the others' in 3-D complex64), m b, and |d|^2.  A box of the dissection that is
// nearly singular magnifies the last bit of any of these to 1e-8 in S^-1, so the kernels
// must not leave the contraction to each one's context.
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
template <typename C> __device__ __forceinline__ C csub_mul(C a, C m, C b)
{
    a.x -= fma(m.x, b.x, -mul_rn(m.y, b.y));
    a.y -= fma(m.y, b.x, mul_rn(m.x, b.y));
    return a;
}
template <typename C> __device__ __forceinline__ C cmul_rn(C a, C b)
{
    C r;
    r.x = fma(a.x, b.x, -mul_rn(a.y, b.y));
    r.y = fma(a.x, b.y, mul_rn(a.y, b.x));
    return r;
}
template <typename C> __device__ __forceinline__ C neg_mul(C m, C b)
{
    C r = cmul_rn(m, b);
    r.x = -r.x;
    r.y = -r.y;
    return r;
}
template <typename C> __device__ __forceinline__ auto norm2_rn(C a) { return fma(a.x, a.x, mul_rn(a.y, a.y)); }

// F (zeroed) <- the front's entries of S
template <typename C>
__global__ void __launch_bounds__(BP_THREADS) k_bp_assemble(const BatchFront *__restrict__ fronts, const C *__restrict__ S,
                                                            const int *__restrict__ pts, const int *__restrict__ maps,
                                                            GridDesc g, C *scratch, long stride, int *perm, int permld)
{
    pdl_wait_and_trigger();
    const BatchFront fr = fronts[blockIdx.x];
    C *F = scratch + (long)blockIdx.x * stride;
    const int f = fr.f, D = g.D, DD = g.D * g.D, first = blockIdx.y * blockDim.x + threadIdx.x, step = gridDim.y * blockDim.x;
    const int *own_pts = pts + fr.own_off, *lmap = maps + fr.map_off;
    for (int i = first; i < fr.o3; i += step) perm[(long)blockIdx.x * permld + i] = i;
    for (int gid = first; gid < fr.nown * g.nsten; gid += step) {
        const int a = gid / g.nsten, s = gid % g.nsten;
        const int o1 = s % 3 - 1, o2 = (s / 3) % 3 - 1, oz = g.nsten == 27 ? s / 9 - 1 : 0;
        const int i = own_pts[a];
        const int j1 = i % g.n1 + o1, j2 = (i / g.n1) % g.n2 + o2, j3 = i / (g.n1 * g.n2) + oz;
        if (j1 < 0 || j2 < 0 || j3 < 0 || j1 >= g.n1 || j2 >= g.n2 || j3 >= g.n3) continue;
        const int lj = lmap[((j3 - fr.e2) * fr.ew1 + (j2 - fr.e1)) * fr.ew0 + (j1 - fr.e0)];
        if (lj < 0) continue; // eliminated in a child
        const long j = ((long)j3 * g.n2 + j2) * g.n1 + j1;
        const C *blk = S + ((long)i * g.nsten + s) * DD;
        for (int c = 0; c < D; ++c)
            for (int q = 0; q < D; ++q) F[(long)(D * lj + q) * f + D * a + c] = blk[c * D + q];
        if (lj >= fr.nown) {
            const C *bj = S + (j * g.nsten + (g.nsten - 1 - s)) * DD;
            for (int c = 0; c < D; ++c)
                for (int q = 0; q < D; ++q) F[(long)(D * a + q) * f + D * lj + c] = bj[c * D + q];
        }
    }
}

// F += the update of child ch (the children one after the other: their maps overlap)
template <typename C>
__global__ void __launch_bounds__(BP_THREADS) k_bp_extend(const BatchFront *__restrict__ fronts, int ch,
                                                          const int *__restrict__ rels, C *scratch, long stride)
{
    pdl_wait_and_trigger();
    const BatchFront &fr = fronts[blockIdx.x];
    if (ch >= fr.nch) return;
    C *F = scratch + (long)blockIdx.x * stride;
    const C *U = reinterpret_cast<const C *>(fr.ch_upd[ch]);
    const int bc = fr.ch_bc[ch], f = fr.f;
    const int *rel = rels + fr.ch_rel[ch];
    for (int c = blockIdx.y; c < bc; c += gridDim.y) {
        C *col = F + (long)rel[c] * f;
        for (int r = threadIdx.x; r < bc; r += BP_THREADS) {
            const C u = U[(long)c * bc + r];
            C d = col[rel[r]];
            d.x += u.x;
            d.y += u.y;
            col[rel[r]] = d;
        }
    }
}

// amax2[front] = the largest |entry|^2 of F11, as the bits of a double (zeroed before)
template <typename C>
__global__ void __launch_bounds__(BP_THREADS) k_bp_absmax(const BatchFront *__restrict__ fronts, const C *scratch, long stride,
                                                          unsigned long long *amax2)
{
    pdl_wait_and_trigger();
    const int f = fronts[blockIdx.x].f, o3 = fronts[blockIdx.x].o3;
    const C *F = scratch + (long)blockIdx.x * stride;
    unsigned long long mx = 0;
    for (int c = blockIdx.y; c < o3; c += gridDim.y)
        for (int r = threadIdx.x; r < o3; r += BP_THREADS) {
            const C a = F[(long)c * f + r];
            mx = max(mx, (unsigned long long)__double_as_longlong((double)norm2_rn(a)));
        }
    for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if ((threadIdx.x & 31) == 0 && mx) atomicMax(&amax2[blockIdx.x], mx);
}

// A step's rows x BP_NB entries are spread over the block: thread t takes row t % rows and
// the columns of group t / rows.  M: [front][BP_NB][fm].
template <typename C>
__global__ void __launch_bounds__(BP_THREADS) k_bp_panel(const BatchFront *__restrict__ fronts, C *scratch, long stride, int k0,
                                                         double tau, const unsigned long long *__restrict__ amax2, int *perm,
                                                         int permld, C *M, int fm, BatchPanel<C> *panels, int *raised)
{
    using R = decltype(C{}.x);
    pdl_wait_and_trigger();
    const int f = fronts[blockIdx.x].f, o3 = fronts[blockIdx.x].o3;
    if (k0 >= o3) return;
    const int kb = min(BP_NB, o3 - k0), m = o3 - k0;
    extern __shared__ unsigned char smem_raw[];
    C *P = reinterpret_cast<C *>(smem_raw); // [BP_NB][m]
    C *pc = P + BP_NB * m;                  // [m] the step's column before elimination
    __shared__ C prow[BP_NB];
    __shared__ unsigned long long cand[BP_THREADS / 32];
    __shared__ int candi[BP_THREADS / 32], pivs[BP_NB];
    C *F = scratch + (long)blockIdx.x * stride + k0;
    C *Mf = M + (long)blockIdx.x * BP_NB * fm + k0;
    BatchPanel<C> &bp = panels[blockIdx.x];
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, wid = tid >> 5;
    for (int e = tid; e < kb * m; e += nt) P[e] = F[(long)(k0 + e / m) * f + e % m];
    const R fl = (R)(tau * sqrt(__longlong_as_double((long long)amax2[blockIdx.x])));
    // column groups: 1, 2, 4 or 8, as many as give every thread work
    int gr = 1;
    while (gr < BP_NB && m * gr * 2 <= nt) gr *= 2;
    const int cw = BP_NB / gr, rows = gr == 1 ? nt : m, r0 = tid % rows, cg = tid / rows * cw;
    __syncthreads();
    for (int jj = 0; jj < kb; ++jj) {
        // the largest |P[jj][i]| over the unpivoted own rows, the lowest row on ties;
        // magnitudes compared as the bits of non-negative doubles
        unsigned long long best = 0;
        int bi = m;
        for (int i = tid; i < m; i += nt) {
            const C a = P[jj * m + i];
            pc[i] = a;
            if (i < jj) continue;
            const unsigned long long v = (unsigned long long)__double_as_longlong((double)norm2_rn(a));
            if (v > best || bi == m) { best = v; bi = i; }
        }
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long ov = __shfl_xor_sync(0xffffffffu, best, o);
            const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
            if (oi < m && (bi == m || ov > best || (ov == best && oi < bi))) { best = ov; bi = oi; }
        }
        if (lane == 0) { cand[wid] = best; candi[wid] = bi; }
        __syncthreads();
        if (wid == 0) {
            best = cand[0];
            bi = candi[0];
            for (int w = 1; w < nt / 32; ++w)
                if (candi[w] < m && (bi == m || cand[w] > best || (cand[w] == best && candi[w] < bi))) { best = cand[w]; bi = candi[w]; }
            const int p = bi;
            // the pivot row, divided by the (floored) pivot; rows p and jj change places
            C v = czero<C>();
            if (lane < kb) {
                v = P[lane * m + p];
                P[lane * m + p] = P[lane * m + jj];
            }
            C d;
            d.x = __shfl_sync(0xffffffffu, v.x, jj);
            d.y = __shfl_sync(0xffffffffu, v.y, jj);
            R d2 = norm2_rn(d);
            if (d2 < fl * fl) { // the static pivot floor
                const R ad = sqrt(d2);
                const R sx = ad > 0 ? d.x / ad : (R)1, sy = ad > 0 ? d.y / ad : (R)0;
                d.x = fl * sx;
                d.y = fl * sy;
                d2 = norm2_rn(d);
                if (lane == 0) atomicAdd(raised, 1);
            }
            // conj(d) / |d|^2: the two divisions in two lanes at once
            const R quo = (lane & 1 ? -d.y : d.x) / d2;
            C inv_d;
            inv_d.x = __shfl_sync(0xffffffffu, quo, 0);
            inv_d.y = __shfl_sync(0xffffffffu, quo, 1);
            if (lane < kb) {
                const C w = lane == jj ? inv_d : cmul_rn(v, inv_d);
                prow[lane] = w;
                bp.prow[jj][lane] = w;
            }
            if (lane == 0) {
                pivs[jj] = p;
                pc[p] = pc[jj];
            }
        }
        __syncthreads();
        if (r0 < m && cg < kb) {
            for (int i = r0; i < m; i += rows) {
                const C a = pc[i];
                if (cg == 0) Mf[jj * fm + i] = a;
#pragma unroll 1
                for (int c = cg; c < min(cg + cw, kb); ++c)
                    P[c * m + i] = i == jj ? prow[c] : (c == jj ? neg_mul(a, prow[jj]) : csub_mul(P[c * m + i], a, prow[c]));
            }
        }
        if (wid == nt / 32 - 1 && lane < jj && pivs[jj] != jj) { // the swapped rows' earlier multipliers
            C *u = Mf + lane * fm + jj, *w = Mf + lane * fm + pivs[jj];
            const C t = *u;
            *u = *w;
            *w = t;
        }
        __syncthreads();
    }
    for (int e = tid; e < kb * m; e += nt) F[(long)(k0 + e / m) * f + e % m] = P[e];
    if (tid == 0) { // the rows whose contents the swaps moved
        int nmove = kb;
        for (int jj = 0; jj < kb; ++jj) bp.dst[jj] = bp.src[jj] = k0 + jj;
        int *pm = perm + (long)blockIdx.x * permld;
        for (int jj = 0; jj < kb; ++jj) {
            const int p = k0 + pivs[jj];
            if (p == k0 + jj) continue;
            const int t = pm[p];
            pm[p] = pm[k0 + jj];
            pm[k0 + jj] = t;
            int q = 0;
            while (q < nmove && bp.dst[q] != p) ++q;
            if (q == nmove) {
                bp.dst[q] = bp.src[q] = p;
                ++nmove;
            }
            const int u = bp.src[q];
            bp.src[q] = bp.src[jj];
            bp.src[jj] = u;
        }
        bp.nmove = nmove;
    }
}

// blockIdx.y < row_blocks: the panel's columns on the other rows (pivoted before, and
// boundary), eight rows and four column groups per warp, the step's multiplier passed
// between the groups.  The other blocks: the pivot rows of the other columns, a thread per
// (pivot row, column): the panel's row swaps first, then the steps, S kept.
constexpr int BX_THREADS = 128, BX_ROWS = BX_THREADS / 4, BX_COLS = BX_THREADS / BP_NB;
template <typename C>
__global__ void __launch_bounds__(BX_THREADS) k_bp_cross(const BatchFront *__restrict__ fronts, C *scratch, long stride, int k0,
                                                         int row_blocks, C *M, C *S, int fm,
                                                         const BatchPanel<C> *__restrict__ panels)
{
    constexpr int CW = BP_NB / 4;
    pdl_wait_and_trigger();
    const int f = fronts[blockIdx.x].f, o3 = fronts[blockIdx.x].o3;
    if (k0 >= o3) return;
    const int kb = min(BP_NB, o3 - k0);
    const BatchPanel<C> &bp = panels[blockIdx.x];
    C *F = scratch + (long)blockIdx.x * stride;
    C *Mf = M + (long)blockIdx.x * BP_NB * fm;
    if ((int)blockIdx.y < row_blocks) {
        if (blockIdx.y * BX_ROWS >= f - (o3 - k0)) return;
        const int lane = threadIdx.x & 31, g = lane >> 3;
        const int e = blockIdx.y * BX_ROWS + (threadIdx.x >> 5) * 8 + (lane & 7), i = e < k0 ? e : e + o3 - k0;
        F += (long)k0 * f;
        C a[CW];
#pragma unroll
        for (int c = 0; c < CW; ++c) a[c] = g * CW + c < kb && i < f ? F[(long)(g * CW + c) * f + i] : czero<C>();
#pragma unroll
        for (int jj = 0; jj < BP_NB; ++jj) {
            if (jj >= kb) break;
            C w;
            w.x = __shfl_sync(0xffffffffu, a[jj % CW].x, (jj / CW) * 8 + (lane & 7));
            w.y = __shfl_sync(0xffffffffu, a[jj % CW].y, (jj / CW) * 8 + (lane & 7));
            if (g == 0 && i < f) Mf[jj * fm + i] = w;
#pragma unroll
            for (int c = 0; c < CW; ++c)
                if (g * CW + c < kb) a[c] = g * CW + c == jj ? neg_mul(w, bp.prow[jj][jj]) : csub_mul(a[c], w, bp.prow[jj][g * CW + c]);
        }
        if (i >= f) return;
#pragma unroll
        for (int c = 0; c < CW; ++c)
            if (g * CW + c < kb) F[(long)(g * CW + c) * f + i] = a[c];
        return;
    }
    const int c0 = (blockIdx.y - row_blocks) * BX_COLS;
    if (c0 >= f - kb) return;
    __shared__ C sr[BP_NB][BX_COLS];
    const int k = threadIdx.x / BX_COLS, c = threadIdx.x % BX_COLS;
    const bool act = k < kb && c0 + c < f - kb;
    const int j = c0 + c < k0 ? c0 + c : c0 + c + kb; // the column
    C *col = F + (long)j * f;
    const int q = kb + k; // a displaced row, if there are as many (at most kb)
    const bool dis = c0 + c < f - kb && q < bp.nmove;
    C r = act ? col[bp.src[k]] : czero<C>(), away = dis ? col[bp.src[q]] : czero<C>(), mk[BP_NB];
#pragma unroll
    for (int jj = 0; jj < BP_NB; ++jj) mk[jj] = act && jj < kb ? Mf[jj * fm + k0 + k] : czero<C>();
    const C inv = act ? bp.prow[k][k] : czero<C>();
    __syncthreads(); // every source row has been read
    if (dis) col[bp.dst[q]] = away;
#pragma unroll
    for (int jj = 0; jj < BP_NB; ++jj) {
        if (jj >= kb) break;
        if (act && k == jj) {
            r = cmul_rn(r, inv);
            sr[jj][c] = r;
            S[((long)blockIdx.x * fm + j) * BP_NB + jj] = r;
        }
        __syncthreads();
        if (act && k != jj) r = csub_mul(r, mk[jj], sr[jj][c]);
    }
    if (act) col[k0 + k] = r;
}

template <typename C, int CT>
__global__ void __launch_bounds__(BP_THREADS, 2) k_bp_update(const BatchFront *__restrict__ fronts, C *scratch, long stride,
                                                          int k0, const C *__restrict__ M, const C *__restrict__ S, int fm)
{
    pdl_wait_and_trigger();
    const int f = fronts[blockIdx.x].f, o3 = fronts[blockIdx.x].o3;
    if (k0 >= o3) return;
    const int kb = min(BP_NB, o3 - k0), c0 = blockIdx.y * CT, nc = min(CT, f - kb - c0);
    if (nc <= 0) return;
    __shared__ C sr[CT][BP_NB];
    C *F = scratch + (long)blockIdx.x * stride;
    const C *Mf = M + (long)blockIdx.x * BP_NB * fm;
    auto col = [&](int c) { return c0 + c < k0 ? c0 + c : c0 + c + kb; };
    for (int e = threadIdx.x; e < CT * BP_NB; e += blockDim.x) {
        const int c = e / BP_NB, q = e % BP_NB;
        sr[c][q] = c < nc && q < kb ? S[((long)blockIdx.x * fm + col(c)) * BP_NB + q] : czero<C>();
    }
    __syncthreads();
    for (int i = threadIdx.x; i < f; i += blockDim.x) {
        if (i >= k0 && i < k0 + kb) continue;
        C t[BP_NB];
#pragma unroll
        for (int q = 0; q < BP_NB; ++q) t[q] = q < kb ? Mf[q * fm + i] : czero<C>();
#pragma unroll 2
        for (int c = 0; c < nc; ++c) {
            C *at = F + (long)col(c) * f + i;
            C a = *at;
#pragma unroll
            for (int q = 0; q < BP_NB; ++q)
                if (q < kb) a = csub_mul(a, t[q], sr[c][q]);
            *at = a;
        }
    }
}

// the swept fronts -> G = [F11^-1; F21 F11^-1] (columns put back in place), X, update
template <typename C>
__global__ void __launch_bounds__(BP_THREADS) k_bp_store(const BatchFront *__restrict__ fronts, const C *scratch, long stride,
                                                         const int *__restrict__ perm, int permld, C *fac)
{
    pdl_wait_and_trigger();
    const BatchFront &fr = fronts[blockIdx.x];
    const C *F = scratch + (long)blockIdx.x * stride;
    const int f = fr.f, o3 = fr.o3, b3 = f - o3;
    C *G = fac + fr.fac_off, *X = G + (long)f * o3, *U = reinterpret_cast<C *>(fr.upd);
    for (int j = blockIdx.y; j < f; j += gridDim.y) {
        const C *col = F + (long)j * f;
        C *g = j < o3 ? G + (long)perm[(long)blockIdx.x * permld + j] * f : nullptr;
        for (int r = threadIdx.x; r < f; r += BP_THREADS) {
            C v = col[r];
            if (j < o3) {
                if (r >= o3) { v.x = -v.x; v.y = -v.y; }
                g[r] = v;
            } else if (r < o3) {
                X[(long)(j - o3) * o3 + r] = v;
            } else {
                U[(long)(j - o3) * b3 + r - o3] = v;
            }
        }
    }
}

template <typename C>
__global__ void k_extend_add(C *F, int f, const C *__restrict__ U, int bc, const int *__restrict__ rel)
{
    long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (long)bc * bc) return;
    int r = (int)(gid % bc), c = (int)(gid / bc);
    long dst = (long)rel[c] * f + rel[r];
    C u = U[gid], v = F[dst];
    v.x += u.x;
    v.y += u.y;
    F[dst] = v;
}

// copy an (m x n) block between column-major matrices
template <typename C>
__global__ void k_copy_block(C *dst, int ldd, const C *__restrict__ src, int lds, int m, int ncol)
{
    long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (long)m * ncol) return;
    int r = (int)(gid % m), c = (int)(gid / m);
    dst[(long)c * ldd + r] = src[(long)c * lds + r];
}

template <typename C> __global__ void k_zero(C *a, long cnt)
{
    long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid < cnt) { a[gid].x = 0; a[gid].y = 0; }
}

inline unsigned blocks(long cnt, int t = 256) { return (unsigned)((cnt + t - 1) / t); }

// ---------------------------------------------------------------- solve kernels
// Vectors of a solve live in elimination order, [unknown u][rhs], u = D x (rank of
// the point among all nodes' own points, in postorder) + component: a node's own
// unknowns are contiguous and its boundary is a list of u, so a level needs no
// packing pass.  W holds the right-hand side as it is updated, Y the solution.
//   forward, deepest level first:  [y; t] = G w_own,  Y_own = y,  W_bnd -= t
//   backward, root first:          Y_own -= X Y_bnd
// One launch per level and direction.  Every node's matrix (column-major, ld rows)
// is cut into tiles (of at most st_elems entries where they are copied to shared memory, 256
// columns where they stream through registers, below); a block of 256 threads owns one tile:
// thread t takes row t % nrow and the columns t / nrow + groups k,
// groups = 256 / nrow, so that a tile of 49 rows keeps 245 threads busy.
// Bound: complex64 by reading the factor; complex128 by the FP64 pipe (4 FMAs per
// 16 bytes at 1.25 TFLOP/s: 2.5 TB/s); small grids by the 2 x levels dependent
// launches (3.3 us each at n = 16).  S^-1, against the packing, GEMV and scatter launches
// this replaced (four per level and direction): 2-D complex128 n = 119 139 us (1063
// before), n = 239 294 (1970; 137 by the FP64 pipe); 3-D complex64 n = 16 40 (378), n = 32
// 314 (1067; 219 by the factor's bytes), n = 64 4090 (4655); 16 right-hand sides n = 16 222
// (1439), n = 32 1072 (2887; 300 by the FP32 pipe), n = 64 13200 (22170).
struct SolveTile {
    long mat, scale;  // first entry of the tile; scale of its first column (half storage)
    int ld, nrow, ncol;
    int in;           // forward: unknown of the first column; backward: its place in the boundary list
    int out, nown;    // unknown of the first row; rows that are own unknowns
    int bout;         // place of row nown in the boundary list
    int full;         // the tile spans every column: no other block adds to its own rows
};
constexpr int ST_THREADS = 256, ST_GROUPS = 16;
// Tiles go through shared memory whole (cp.async) in complex128, where the registers are
// better spent on more warps for the FP64 pipe (n = 239: 339 us against 500), and in
// complex64 for factors that stay in the L2 (3-D n = 16: 43 us against 63); larger ones
// stream through registers, eight entries ahead (n = 64: 4.49 ms against 5.43).
constexpr size_t ST_STAGED_BYTES = 256u << 20;
template <typename C> constexpr int st_rows() { return 1024 / (int)sizeof(C); } // 1 KB of each column
template <typename C> constexpr int st_elems() { return sizeof(C) == 8 ? 6144 : 2048; } // of a staged tile: 48, 32 KB

__device__ __forceinline__ float2 value_of(float2 v) { return v; }
__device__ __forceinline__ double2 value_of(double2 v) { return v; }
__device__ __forceinline__ float2 value_of(__half2 v) { return __half22float2(v); }

__device__ __forceinline__ void add_to(float2 *p, float2 v) { atomicAdd(p, v); }
__device__ __forceinline__ void add_to(double2 *p, double2 v)
{
    atomicAdd(&p->x, v.x);
    atomicAdd(&p->y, v.y);
}

// acc of g x over a tile's columns, NB right-hand sides.  complex64 keeps the sums
// of g.x x and g.y x apart (two packed FP32x2 FMAs each) and joins them at the end.
template <typename C, int NB> struct TileAcc {
    C s[NB];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int b = 0; b < NB; ++b) s[b] = czero<C>();
    }
    __device__ __forceinline__ void mac(C g, const C *x)
    {
#pragma unroll
        for (int b = 0; b < NB; ++b) s[b] = cfma(g, x[b], s[b]);
    }
    __device__ __forceinline__ C get(int b) const { return s[b]; }
};
template <int NB> struct TileAcc<float2, NB> {
    float2 p[NB], q[NB];
    __device__ __forceinline__ void clear()
    {
#pragma unroll
        for (int b = 0; b < NB; ++b) p[b] = q[b] = make_float2(0.f, 0.f);
    }
    __device__ __forceinline__ void mac(float2 g, const float2 *x)
    {
        const float2 gx = make_float2(g.x, g.x), gy = make_float2(g.y, g.y);
#pragma unroll
        for (int b = 0; b < NB; ++b) {
            p[b] = __ffma2_rn(gx, x[b], p[b]);
            q[b] = __ffma2_rn(gy, x[b], q[b]);
        }
    }
    __device__ __forceinline__ float2 get(int b) const { return make_float2(p[b].x - q[b].y, p[b].y + q[b].x); }
};

// Blocks per SM that the registers are held to.  complex64, one right-hand side: loads in
// flight against blocks to overlap their starts and ends (3-D n = 32: four 392 us, five
// 346, six 314, eight 562; n = 64: 4.60, 3.94, 4.09, 6.46 ms).  At six the streamed kernels
// spill a few registers (one right-hand side 48 bytes a thread, two 104), at eight many.  Several wait on
// shared memory between their packed FMAs and gain from warps (8 of them at n = 32: one
// block 1050 us, two 686, three 606, four 586; 16, whose sums alone are 64 registers: one
// 1599, two 1072, three 1585).  complex128 (2-D n = 239): one right-hand side four 342 us,
// five 312, six 294, eight 343; four 843, 840, 870, 884; eight 1802 with two, 1680 with four.
// Half storage streamed, one or two right-hand sides: eight, and no batches held in
// registers: sixteen loads issued together straight into their FMAs (one right-hand side at
// n = 64 2.49 ms; batches of eight at six blocks 3.34, of sixteen at four 3.54; two 2.59
// against 3.71; n = 32 274 us against 283).
template <typename C, typename S, int NB, bool STAGED> constexpr bool st_direct() { return !STAGED && sizeof(S) == 4 && NB <= 2; }
template <typename C, typename S, int NB, bool STAGED> constexpr int st_blocks()
{
    if (st_direct<C, S, NB, STAGED>()) return 8;
    if (sizeof(C) == 16) return NB <= 2 ? 6 : (NB == 4 ? 5 : 4);
    return NB <= 2 ? 6 : (NB <= 8 ? 4 : 2);
}

template <typename C, typename S, int NB, bool FWD, bool STAGED, bool DIRECT = st_direct<C, S, NB, STAGED>()>
__global__ void __launch_bounds__(ST_THREADS, st_blocks<C, S, NB, STAGED>()) k_nd_level(const S *__restrict__ M, const float *__restrict__ scales,
                                                         const SolveTile *__restrict__ tiles,
                                                         const int *__restrict__ bnd, C *W, C *Y, int nrhs, int tile_elems)
{
    constexpr bool SCALED = !std::is_same<S, C>::value;
    constexpr int UNR = STAGED || DIRECT ? 1 : (NB == 8 ? 4 : 8); // matrix entries a thread has in flight in registers
    extern __shared__ __align__(16) unsigned char smem_raw[];
    S *ts = reinterpret_cast<S *>(smem_raw); // the tile, [ncol][nrow]
    C *xs = reinterpret_cast<C *>(smem_raw + (STAGED ? sizeof(S) * (size_t)tile_elems : 0)); // columns, then sums
    const SolveTile tl = tiles[blockIdx.x];
    const int groups = min(ST_THREADS / tl.nrow, ST_GROUPS);
    const int row = threadIdx.x % tl.nrow, g = threadIdx.x / tl.nrow;
    const bool act = g < groups;
    const S *src = M + tl.mat + row;
    const int steps = (tl.ncol + groups - 1) / groups; // columns per thread
    S cur[UNR];
    auto fetch = [&](int k0) {
#pragma unroll
        for (int k = 0; k < UNR; ++k) {
            const int c = g + (k0 + k) * groups;
            if (act && c < tl.ncol) cur[k] = __ldcs(src + (long)c * tl.ld);
        }
    };
    // the factor does not change: the tile is on its way before the previous level's
    // results are waited for.  A thread copies the entries that it multiplies.
    if constexpr (STAGED) {
        if (act)
            for (int c = g; c < tl.ncol; c += groups) cp_async<sizeof(S)>(&ts[c * tl.nrow + row], src + (long)c * tl.ld);
        cp_async_commit();
    } else if constexpr (!DIRECT) {
        fetch(0);
    }
    pdl_wait_and_trigger();
    for (int b0 = 0; b0 < nrhs; b0 += NB) {
        const int nb = min(NB, nrhs - b0);
        if (b0 > 0) {
            __syncthreads(); // the sums of the previous group have been read
            if constexpr (!STAGED && !DIRECT) fetch(0);
        }
        for (int i = threadIdx.x; i < tl.ncol * NB; i += ST_THREADS) {
            const int c = i / NB, b = i % NB;
            C v = czero<C>();
            if (b < nb) {
                v = FWD ? __ldcg(W + (long)(tl.in + c) * nrhs + b0 + b) : __ldcg(Y + (long)bnd[tl.in + c] * nrhs + b0 + b);
                if constexpr (SCALED) v = cscale(v, scales[tl.scale + c]);
            }
            xs[i] = v;
        }
        if constexpr (STAGED) cp_async_wait<0>();
        __syncthreads();
        TileAcc<C, NB> acc;
        acc.clear();
        if constexpr (STAGED) {
            if (act) {
#pragma unroll 4
                for (int c = g; c < tl.ncol; c += groups) acc.mac(value_of(ts[c * tl.nrow + row]), xs + c * NB);
            }
        } else if constexpr (DIRECT) {
            if (act) {
                const S *q = src + (long)g * tl.ld;
                const long step = (long)groups * tl.ld;
#pragma unroll 16
                for (int c = g; c < tl.ncol; c += groups, q += step) acc.mac(value_of(__ldcs(q)), xs + c * NB);
            }
        } else {
            for (int k0 = 0; k0 < steps; k0 += UNR) {
                S now[UNR];
#pragma unroll
                for (int k = 0; k < UNR; ++k) now[k] = cur[k];
                if (k0 + UNR < steps) fetch(k0 + UNR);
#pragma unroll
                for (int k = 0; k < UNR; ++k) {
                    const int c = g + (k0 + k) * groups;
                    if (act && c < tl.ncol) acc.mac(value_of(now[k]), xs + c * NB);
                }
            }
        }
        __syncthreads();
        if (act) {
#pragma unroll
            for (int b = 0; b < NB; ++b) xs[threadIdx.x * NB + b] = acc.get(b);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < tl.nrow * NB; i += ST_THREADS) {
            const int r = i / NB, b = i % NB;
            if (b >= nb) continue;
            C v = xs[i];
            for (int q = 1; q < groups; ++q) v = v + xs[i + q * tl.nrow * NB];
            C neg;
            neg.x = -v.x;
            neg.y = -v.y;
            if (r < tl.nown) {
                C *dst = Y + (long)(tl.out + r) * nrhs + b0 + b;
                if (FWD) {
                    if (tl.full) *dst = v;
                    else add_to(dst, v);
                } else {
                    if (tl.full) *dst = __ldcg(dst) - v;
                    else add_to(dst, neg);
                }
            } else {
                add_to(W + (long)bnd[tl.bout + r - tl.nown] * nrhs + b0 + b, neg);
            }
        }
    }
}

// W[u][b] = b[b][c][point], Y = 0; and x[b][c][point] = Y[u][b]
template <typename C>
__global__ void k_nd_enter(C *W, C *Y, const C *__restrict__ in, const int *__restrict__ ptof, int D, long npts, int nrhs)
{
    const long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const long u = gid / nrhs, b = gid - u * nrhs;
    pdl_wait_and_trigger();
    if (u >= D * npts) return;
    const int rank = (int)(u / D), c = (int)(u - (long)rank * D);
    W[gid] = in[(b * D + c) * npts + ptof[rank]];
    Y[gid] = czero<C>();
}
template <typename C>
__global__ void k_nd_leave(C *out, const C *Y, const int *__restrict__ rankof, int D, long npts, int nrhs)
{
    const long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    const long bc = gid / npts, pt = gid - bc * npts, b = bc / D, c = bc - b * D;
    pdl_wait_and_trigger();
    if (b >= nrhs) return;
    out[gid] = __ldcg(Y + ((long)rankof[pt] * D + c) * nrhs + b);
}

// scale[c] = largest |component| of column c of an (m x ncol, ld m) block (1 if zero)
__global__ void k_col_scales(const float2 *__restrict__ a, int m, int ncol, float *scale)
{
    const int c = blockIdx.x;
    float mx = 0.f;
    for (int r = threadIdx.x; r < m; r += blockDim.x) {
        float2 v = a[(long)c * m + r];
        mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y)));
    }
    for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_down_sync(0xffffffffu, mx, off));
    __shared__ float red[32];
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = mx;
    __syncthreads();
    if (threadIdx.x == 0) {
        float t = 0.f;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = fmaxf(t, red[w]);
        scale[c] = t > 0.f ? t : 1.f;
    }
}

// dst = src / scale[column] as binary16 pairs
__global__ void k_to_half(__half2 *dst, const float2 *__restrict__ src, int m, int ncol,
                          const float *__restrict__ scale)
{
    long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= (long)m * ncol) return;
    const float inv = 1.f / scale[gid / m];
    const float2 v = src[gid];
    dst[gid] = __floats2half2_rn(v.x * inv, v.y * inv);
}

} // namespace

// ---------------------------------------------------------------- factor object

struct NDFactor {
    int prec = 0;
    int variant = 0;         // nested-dissection tree variant (cut offsets)
    int batch_line = 0;      // unknowns up to which fronts were batched
    int raised_pivots = 0;   // pivots raised by the static perturbation
    size_t stored_bytes = 0; // bytes of the stored blocks (G and X, plus half-storage scales)
    bool half_store = false; // blocks as scaled binary16 pairs (complex64 factor only)
    DevBuf scales;           // per-column scales (half storage)
    int D = 3;               // unknowns per point
    long npts = 0;           // grid points
    std::vector<Node> nodes; // post-order
    DevBuf pts, maps, rels;  // int lists
    DevBuf fac;              // persistent: per node [F11;F21] (f x nown3) then X (nown3 x nbnd3)
    DevBuf piv;
    DevBuf front, stack, work, info; // factor scratch (released after factoring)
    DevBuf solve_ws;
    size_t max_front_unknowns = 0, max_own3 = 0, max_bnd3 = 0;
    // tiles of the solve's levels; levels[0] is the deepest
    struct Level {
        long tiles_f, tiles_b; // offsets into the tile table: forward (G), backward (X)
        int ntiles_f, ntiles_b;
    };
    std::vector<Level> levels;
    int tile_elems = 0, tile_cols = 0; // of the largest tiles (entries rounded up to four)
    bool staged = false;               // tiles copied to shared memory whole
    DevBuf st_tiles, st_bnd, st_rank, st_point; // tiles, boundary unknowns, rank of each point and back
    DenseWork *dense = nullptr; // Gauss-Jordan workspace
    ~NDFactor()
    {
        spm_dense_work_free(dense);
        pts.release(); maps.release(); rels.release(); fac.release(); piv.release();
        front.release(); stack.release(); work.release(); info.release(); solve_ws.release();
        st_tiles.release(); st_bnd.release(); st_rank.release(); st_point.release(); scales.release();
    }
};

void spm_factor_free(NDFactor *f) { delete f; }


namespace {

constexpr int LEAF_SIDE = 5;

// Separator offset of tree variant v at a given depth.  Variant 0 cuts every box
// through its middle plane; the others move the cuts by one plane (all down,
// all up, alternating by depth), so that every box of the tree changes.  A box
// whose restriction of S is nearly singular makes its separator's Schur block
// nearly singular too (det S_box = det S_children * det F11), and the pivots of
// the multifrontal LU stay inside each front, so such a box spoils the factor;
// a different tree has different boxes.
constexpr int TREE_VARIANTS = 4;

// relative floor of the pivots of a front (about the square root of the
// precision's unit roundoff: near-singular boxes only, since S itself is well
// conditioned)
template <typename R> constexpr double pivot_floor() { return sizeof(R) == 8 ? 1e-8 : 1e-4; }
inline int cut_offset(int variant, int depth)
{
    switch (variant) {
    case 1: return -1;
    case 2: return 1;
    case 3: return (depth & 1) ? 1 : -1;
    default: return 0;
    }
}

int build_tree(std::vector<Node> &nodes, const int lo[3], const int hi[3], int variant, int depth = 0)
{
    Node nd;
    nd.depth = depth;
    for (int d = 0; d < 3; ++d) { nd.lo[d] = lo[d]; nd.hi[d] = hi[d]; }
    int axis = 0;
    for (int d = 1; d < 3; ++d) if (hi[d] - lo[d] > hi[axis] - lo[axis]) axis = d;
    int len = hi[axis] - lo[axis];
    if (len > LEAF_SIDE) {
        nd.axis = axis;
        int cut = lo[axis] + len / 2 + cut_offset(variant, depth);
        cut = std::max(lo[axis] + 1, std::min(hi[axis] - 2, cut)); // both halves non-empty
        nd.cut = cut;
        int lhi[3] = {hi[0], hi[1], hi[2]}, rlo[3] = {lo[0], lo[1], lo[2]};
        lhi[axis] = nd.cut;
        rlo[axis] = nd.cut + 1;
        nd.left = build_tree(nodes, lo, lhi, variant, depth + 1);
        nd.right = build_tree(nodes, rlo, hi, variant, depth + 1);
    }
    nodes.push_back(nd);
    return (int)nodes.size() - 1;
}

} // namespace

// Elimination ranks, boundary lists and tiles of every level.  A level's tiles hold
// at most st_rows rows (a node's rows are cut evenly) and as many columns as leave
// about five tiles for every SM (four or eight are 1 to 4 % slower), 8 to 256 of them and
// at most st_elems entries if staged: levels of few nodes spread over the chip, levels of
// many add each row's sum less often.
template <typename R> static spm_status build_solve_tiles(NDFactor *F, const std::vector<int> &pts)
{
    using C = typename cplx_of<R>::type;
    const std::vector<Node> &nodes = F->nodes;
    const int NN = (int)nodes.size(), D = F->D;
    F->staged = sizeof(R) == 8 || F->stored_bytes <= ST_STAGED_BYTES;
    std::vector<int> rank(F->npts), point(F->npts), bnd;
    std::vector<int> base(NN), boff(NN);
    int next = 0;
    for (int id = 0; id < NN; ++id) {
        base[id] = D * next;
        for (int a = 0; a < nodes[id].nown; ++a, ++next) {
            const int p = pts[nodes[id].own_off + a];
            rank[p] = next;
            point[next] = p;
        }
    }
    int maxd = 0;
    for (int id = 0; id < NN; ++id) {
        const Node &nd = nodes[id];
        boff[id] = (int)bnd.size();
        for (int b = 0; b < nd.nbnd; ++b)
            for (int c = 0; c < D; ++c) bnd.push_back(D * rank[pts[nd.bnd_off + b]] + c);
        maxd = std::max(maxd, nd.depth);
    }
    std::vector<std::vector<int>> at(maxd + 1);
    for (int id = 0; id < NN; ++id) at[nodes[id].depth].push_back(id);
    std::vector<SolveTile> tt;
    auto cut = [&](const std::vector<int> &ids, bool fwd, long &first, int &count) {
        first = (long)tt.size();
        double level = 0;
        for (int id : ids) {
            const double o = D * (double)nodes[id].nown, b = D * (double)nodes[id].nbnd;
            level += fwd ? (o + b) * o : o * b;
        }
        const double per_tile = level / (5 * 152);
        for (int id : ids) {
            const Node &nd = nodes[id];
            const int o = D * nd.nown, b = D * nd.nbnd;
            const int rows = fwd ? o + b : o, cols = fwd ? o : b;
            if (cols == 0) continue;
            const int nr = (rows + st_rows<C>() - 1) / st_rows<C>(), rt = (rows + nr - 1) / nr;
            int ct = std::min({ST_THREADS, std::max(1, F->staged ? st_elems<C>() / rt : ST_THREADS), (int)std::min(1e6, std::max(8.0, per_tile / rt))});
            const int nc = (cols + ct - 1) / ct;
            ct = (cols + nc - 1) / nc;
            for (int r0 = 0; r0 < rows; r0 += rt)
                for (int c0 = 0; c0 < cols; c0 += ct) {
                    SolveTile t;
                    t.ld = rows;
                    t.nrow = std::min(rt, rows - r0);
                    t.ncol = std::min(ct, cols - c0);
                    t.mat = nd.fac_off + (fwd ? 0 : (long)(o + b) * o) + (long)c0 * rows + r0;
                    t.scale = nd.scale_off + (fwd ? 0 : o) + c0;
                    t.in = fwd ? base[id] + c0 : boff[id] + c0;
                    t.out = base[id] + r0;
                    t.nown = std::max(0, std::min(t.nrow, o - r0));
                    t.bout = boff[id] + std::max(0, r0 - o);
                    t.full = t.ncol == cols;
                    F->tile_elems = std::max(F->tile_elems, t.nrow * t.ncol);
                    F->tile_cols = std::max(F->tile_cols, t.ncol);
                    tt.push_back(t);
                }
        }
        count = (int)((long)tt.size() - first);
    };
    F->levels.clear();
    for (int d = maxd; d >= 0; --d) {
        NDFactor::Level lv;
        cut(at[d], true, lv.tiles_f, lv.ntiles_f);
        cut(at[d], false, lv.tiles_b, lv.ntiles_b);
        F->levels.push_back(lv);
    }
    // the vectors lie behind a staged tile: whole 16-byte units, also of 4-byte entries
    F->tile_elems = (F->tile_elems + 3) / 4 * 4;
    auto put = [](DevBuf &buf, const void *src, size_t bytes) -> spm_status {
        SPM_TRY(buf.ensure(std::max<size_t>(bytes, 1)));
        if (bytes) SPM_CUDA_TRY(cudaMemcpy(buf.ptr, src, bytes, cudaMemcpyHostToDevice));
        return SPM_OK;
    };
    SPM_TRY(put(F->st_tiles, tt.data(), sizeof(SolveTile) * tt.size()));
    SPM_TRY(put(F->st_bnd, bnd.data(), sizeof(int) * bnd.size()));
    SPM_TRY(put(F->st_rank, rank.data(), sizeof(int) * rank.size()));
    return put(F->st_point, point.data(), sizeof(int) * point.size());
}

// One level's batched fronts (fm, om: the largest front and own block), all at once.
// ws: panel_ws_bytes(count, fm, om), scratch: count fm^2 entries.
template <typename C> static size_t panel_ws_bytes(size_t count, int fm, int om)
{
    return count * (sizeof(C) * 2 * BP_NB * (size_t)fm + sizeof(BatchPanel<C>) + sizeof(unsigned long long) + sizeof(int) * (size_t)om);
}
template <typename C>
static spm_status factor_panels(const BatchFront *fronts, int count, int fm, int om, const C *S, const int *pts,
                                const int *maps, const int *rels, GridDesc g, C *scratch, char *ws, C *fac, double tau,
                                int *raised, cudaStream_t s)
{
    const long stride = (long)fm * fm;
    const size_t b_amax = sizeof(unsigned long long) * (size_t)count;
    C *M = reinterpret_cast<C *>(ws); // most aligned first
    C *srow = M + (size_t)count * BP_NB * fm;
    BatchPanel<C> *panels = reinterpret_cast<BatchPanel<C> *>(srow + (size_t)count * BP_NB * fm);
    unsigned long long *amax2 = reinterpret_cast<unsigned long long *>(panels + count);
    int *perm = reinterpret_cast<int *>(amax2 + count);
    SPM_CUDA_TRY(cudaMemsetAsync(amax2, 0, b_amax, s));
    SPM_CUDA_TRY(cudaMemsetAsync(scratch, 0, sizeof(C) * stride * count, s));
    const unsigned rows = (unsigned)std::max(1, std::min(fm, (8 * 152 + count - 1) / count)); // blocks per front
    const size_t smem = sizeof(C) * (BP_NB + 1) * (size_t)om;
    const int threads = std::min(BP_THREADS, std::max(64, (fm + 31) / 32 * 32)); // a thread per row, up to 256
    // om <= 1536: at most 216 KB, with the static shared memory below the 227 KB of a block
    SPM_CUDA_TRY(cudaFuncSetAttribute(k_bp_panel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, 216 * 1024));
    launch_pdl(k_bp_assemble<C>, dim3(count, rows), dim3(BP_THREADS), 0, s, fronts, S, pts, maps, g, scratch, stride, perm, om);
    for (int ch = 0; ch < 2; ++ch)
        launch_pdl(k_bp_extend<C>, dim3(count, rows), dim3(BP_THREADS), 0, s, fronts, ch, rels, scratch, stride);
    launch_pdl(k_bp_absmax<C>, dim3(count, rows), dim3(BP_THREADS), 0, s, fronts, (const C *)scratch, stride, amax2);
    // columns per update block: as many as leave two blocks for every SM
    auto blocks_of = [&](int ct) { return (unsigned)((fm + ct - 1) / ct); };
    const int ct = blocks_of(8) * count >= 304 ? 8 : (blocks_of(4) * count >= 304 ? 4 : 2);
    for (int k0 = 0; k0 < om; k0 += BP_NB) {
        launch_pdl(k_bp_panel<C>, dim3(count), dim3(om - k0 > 64 ? BP_THREADS : 128), smem, s, fronts, scratch, stride, k0, tau,
                   (const unsigned long long *)amax2, perm, om, M, fm, panels, raised);
        const int row_blocks = (fm + BX_ROWS - 1) / BX_ROWS;
        launch_pdl(k_bp_cross<C>, dim3(count, row_blocks + (fm + BX_COLS - 1) / BX_COLS), dim3(BX_THREADS), 0, s, fronts, scratch,
                   stride, k0, row_blocks, M, srow, fm, (const BatchPanel<C> *)panels);
        const dim3 grid(count, blocks_of(ct));
        auto update = [&](auto kernel) {
            launch_pdl(kernel, grid, dim3(threads), 0, s, fronts, scratch, stride, k0, (const C *)M, (const C *)srow, fm);
        };
        if (ct == 8) update(k_bp_update<C, 8>);
        else if (ct == 4) update(k_bp_update<C, 4>);
        else update(k_bp_update<C, 2>);
    }
    launch_pdl(k_bp_store<C>, dim3(count, rows), dim3(BP_THREADS), 0, s, fronts, (const C *)scratch, stride, (const int *)perm,
               om, fac);
    SPM_CUDA_TRY(cudaGetLastError());
    return SPM_OK;
}

template <typename R>
static spm_status factor_typed(const SparseSys &SY, NDFactor *F, bool half_store, int variant, int most)
{
    using C = typename cplx_of<R>::type;
    const int n1 = SY.dims[0], n2 = SY.dims[1], n3d = SY.dims[2], D = SY.D;
    const GridDesc gd{n1, n2, n3d, D, SY.nsten};
    cudaStream_t s = SY.stream;
    F->D = D;
    F->npts = SY.points();
    F->nodes.clear();
    int lo[3] = {0, 0, 0}, hi[3] = {n1, n2, n3d};
    build_tree(F->nodes, lo, hi, variant);
    F->variant = variant;
    std::vector<Node> &nodes = F->nodes;
    const int NN = (int)nodes.size();

    // point lists and local maps (host)
    std::vector<int> pts, maps;
    for (Node &nd : nodes) {
        nd.own_off = pts.size();
        int olo[3], ohi[3];
        for (int d = 0; d < 3; ++d) { olo[d] = nd.lo[d]; ohi[d] = nd.hi[d]; }
        if (nd.axis >= 0) { olo[nd.axis] = nd.cut; ohi[nd.axis] = nd.cut + 1; }
        for (int z = olo[2]; z < ohi[2]; ++z)
            for (int y = olo[1]; y < ohi[1]; ++y)
                for (int x = olo[0]; x < ohi[0]; ++x) pts.push_back((z * n2 + y) * n1 + x);
        nd.nown = (int)(pts.size() - nd.own_off);
        nd.bnd_off = pts.size();
        for (int d = 0; d < 3; ++d) { nd.elo[d] = std::max(nd.lo[d] - 1, 0); nd.ehi[d] = std::min(nd.hi[d] + 1, hi[d]); }
        for (int z = nd.elo[2]; z < nd.ehi[2]; ++z)
            for (int y = nd.elo[1]; y < nd.ehi[1]; ++y)
                for (int x = nd.elo[0]; x < nd.ehi[0]; ++x) {
                    bool inside = x >= nd.lo[0] && x < nd.hi[0] && y >= nd.lo[1] && y < nd.hi[1] && z >= nd.lo[2] &&
                                  z < nd.hi[2];
                    if (!inside) pts.push_back((z * n2 + y) * n1 + x);
                }
        nd.nbnd = (int)(pts.size() - nd.bnd_off);
        // local map over the expanded box: own -> [0,nown), bnd -> nown + rank, else -1
        nd.map_off = maps.size();
        int ew[3] = {nd.ehi[0] - nd.elo[0], nd.ehi[1] - nd.elo[1], nd.ehi[2] - nd.elo[2]};
        size_t base = maps.size();
        maps.resize(base + (size_t)ew[0] * ew[1] * ew[2], -1);
        auto mi = [&](int p) {
            int x = p % n1, y = (p / n1) % n2, z = p / (n1 * n2);
            return base + ((size_t)(z - nd.elo[2]) * ew[1] + (y - nd.elo[1])) * ew[0] + (x - nd.elo[0]);
        };
        for (int a = 0; a < nd.nown; ++a) maps[mi(pts[nd.own_off + a])] = a;
        for (int b = 0; b < nd.nbnd; ++b) maps[mi(pts[nd.bnd_off + b])] = nd.nown + b;
    }
    // child boundary unknowns -> parent front unknowns
    std::vector<int> rels;
    for (Node &nd : nodes) {
        for (int ch : {nd.left, nd.right}) {
            if (ch < 0) continue;
            Node &c = nodes[ch];
            c.rel_off = rels.size();
            int ew[3] = {nd.ehi[0] - nd.elo[0], nd.ehi[1] - nd.elo[1], nd.ehi[2] - nd.elo[2]};
            for (int b = 0; b < c.nbnd; ++b) {
                int p = pts[c.bnd_off + b];
                int x = p % n1, y = (p / n1) % n2, z = p / (n1 * n2);
                int l = maps[nd.map_off + ((size_t)(z - nd.elo[2]) * ew[1] + (y - nd.elo[1])) * ew[0] + (x - nd.elo[0])];
                if (l < 0) { spm_set_error("nested dissection: child boundary point outside the parent front"); return SPM_ERR_NUMERICAL; }
                for (int q = 0; q < D; ++q) rels.push_back(D * l + q);
            }
        }
    }
    // storage
    F->half_store = half_store;
    long fac_total = 0, piv_total = 0, scale_total = 0;
    std::vector<size_t> upd_size(NN, 0);
    for (int id = 0; id < NN; ++id) {
        Node &nd = nodes[id];
        long o3 = (long)D * nd.nown, b3 = (long)D * nd.nbnd, f = o3 + b3;
        nd.fac_off = fac_total;
        fac_total += f * o3 + o3 * b3;
        nd.piv_off = piv_total;
        piv_total += o3;
        nd.scale_off = scale_total;
        scale_total += f;
        F->max_own3 = std::max(F->max_own3, (size_t)o3);
        F->max_bnd3 = std::max(F->max_bnd3, (size_t)b3);
        upd_size[id] = (size_t)(b3 * b3);
    }
    // Concurrency across fronts.  A subtree whose fronts all have a fully summed
    // block of at most GJ_ONE_BLOCK unknowns (inverted by one block, no grid
    // barrier) is a unit of work; the maximal such subtrees are dealt round-robin
    // to a pool of streams, each stream factoring its subtrees in postorder with
    // its own front, update stack and dense workspace.  A subtree root's update
    // goes to a buffer of its own, where its parent (above the subtrees, factored
    // afterwards on the problem's stream) finds it.
    // Fronts of at most fmax unknowns whose subtrees are batched too are factored
    // first, level by level, all of a level at once (factor_panels); their updates go to
    // buffers of their own.  The stream pool below handles the rest.  In 3-D 1536 is the
    // fastest line where the updates fit (n = 32 complex64: 512 327 ms, 1024 275, 1536
    // 231, 2048 255); where they would take more than 12 GB the next smaller one serves
    // (n = 64: 15 GB at 1536, 10 at 1024, at the same speed).  In 2-D the line stays at
    // 512: larger fronts would be faster batched too (n = 239: 137 -> 66 ms), but the
    // per-front path rounds differently, and 2-D factors have near-singular boxes often
    // enough (one medium in twelve at n = 239) that S^-1 moves by 5e-9.
    std::vector<char> batched(NN, 0);
    for (const int fmax : BATCH_LINES) {
        if (fmax > (n3d == 1 ? 512 : most)) continue;
        F->batch_line = fmax;
        double bytes = 0;
        for (int id = 0; id < NN; ++id) { // postorder: children before parents
            const Node &nd = nodes[id];
            bool ok = !half_store && D * (nd.nown + nd.nbnd) <= fmax;
            for (int ch : {nd.left, nd.right})
                if (ch >= 0 && !batched[ch]) ok = false;
            batched[id] = ok ? 1 : 0;
            if (ok) bytes += sizeof(C) * (double)upd_size[id];
        }
        if (bytes <= 12e9) break;
    }
    const size_t one_block = sizeof(R) == 4 ? 768 : 384;
    std::vector<size_t> smax(NN, 0);
    std::vector<int> parent(NN, -1);
    for (int id = 0; id < NN; ++id) { // postorder: children before parents
        const Node &nd = nodes[id];
        smax[id] = batched[id] ? 0 : D * (size_t)nd.nown;
        for (int ch : {nd.left, nd.right})
            if (ch >= 0) { smax[id] = std::max(smax[id], smax[ch]); parent[ch] = id; }
    }
    std::vector<int> group(NN, -1);     // stream slot of the node, -1: above the subtrees
    std::vector<char> sub_root(NN, 0);
    const int NSTREAM = 16;
    int nsub = 0;
    for (int id = 0; id < NN; ++id)
        if (!batched[id] && smax[id] <= one_block && (parent[id] < 0 || smax[parent[id]] > one_block)) {
            sub_root[id] = 1;
            ++nsub;
        }
    {   // deal the subtrees (each a contiguous postorder range ending at its root)
        int k = 0;
        for (int id = 0; id < NN; ++id) {
            if (!sub_root[id]) continue;
            int first = id;
            while (true) { // leftmost descendant = first node of the subtree's range
                const Node &nd = nodes[first];
                if (nd.left >= 0) first = nd.left;
                else if (nd.right >= 0) first = nd.right;
                else break;
            }
            for (int j = first; j <= id; ++j)
                if (!batched[j]) group[j] = k % NSTREAM;
            ++k;
        }
    }
    const int ngroups = std::min(NSTREAM, std::max(nsub, 0)) + 1; // + the problem's stream (slot ngroups - 1)
    auto slot = [&](int id) { return group[id] < 0 ? ngroups - 1 : group[id]; };
    // per-slot workspace sizes: front, update stack (postorder within the slot; a
    // subtree root's update lives in its own buffer), half-storage staging
    std::vector<size_t> g_front(ngroups, 1), g_stack(ngroups, 1), g_now(ngroups, 0), g_gx(ngroups, 1);
    std::vector<size_t> root_upd_off(NN, 0);
    size_t root_upd_total = 0;
    std::vector<size_t> batch_upd_off(NN, 0);
    size_t batch_upd_total = 0;
    for (int id = 0; id < NN; ++id) {
        const Node &nd = nodes[id];
        if (batched[id]) {
            batch_upd_off[id] = batch_upd_total;
            batch_upd_total += upd_size[id];
            continue;
        }
        const size_t o3 = D * (size_t)nd.nown, b3 = D * (size_t)nd.nbnd, f = o3 + b3;
        const int g = slot(id);
        g_front[g] = std::max(g_front[g], f * f);
        g_gx[g] = std::max(g_gx[g], f * o3 + o3 * b3);
        for (int ch : {nd.left, nd.right})
            if (ch >= 0 && !sub_root[ch] && !batched[ch]) g_now[g] -= upd_size[ch];
        if (sub_root[id]) {
            root_upd_off[id] = root_upd_total;
            root_upd_total += upd_size[id];
        } else {
            g_now[g] += upd_size[id];
            g_stack[g] = std::max(g_stack[g], g_now[g]);
        }
    }
    F->max_front_unknowns = 0;
    for (const Node &nd : nodes) F->max_front_unknowns = std::max(F->max_front_unknowns, (size_t)(D * (nd.nown + nd.nbnd)));
    SPM_TRY(F->pts.ensure(sizeof(int) * pts.size()));
    SPM_TRY(F->maps.ensure(sizeof(int) * maps.size()));
    SPM_TRY(F->rels.ensure(sizeof(int) * std::max<size_t>(rels.size(), 1)));
    SPM_CUDA_TRY(cudaMemcpy(F->pts.ptr, pts.data(), sizeof(int) * pts.size(), cudaMemcpyHostToDevice));
    SPM_CUDA_TRY(cudaMemcpy(F->maps.ptr, maps.data(), sizeof(int) * maps.size(), cudaMemcpyHostToDevice));
    if (!rels.empty())
        SPM_CUDA_TRY(cudaMemcpy(F->rels.ptr, rels.data(), sizeof(int) * rels.size(), cudaMemcpyHostToDevice));
    SPM_TRY(F->fac.ensure((half_store ? sizeof(__half2) : sizeof(C)) * fac_total));
    F->stored_bytes = (half_store ? sizeof(__half2) : sizeof(C)) * (size_t)fac_total +
                      (half_store ? sizeof(float) * (size_t)scale_total : 0);
    if (half_store) SPM_TRY(F->scales.ensure(sizeof(float) * scale_total));
    SPM_TRY(F->info.ensure(sizeof(int) * 3)); // expired grid barrier, unused, raised pivots
    SPM_CUDA_TRY(cudaMemsetAsync(F->info.ptr, 0, sizeof(int) * 3, s));
    const C *Sdev = reinterpret_cast<const C *>(sizeof(R) == 8 ? SY.S128 : SY.S64);
    const int *dpts = F->pts.as<int>(), *dmaps = F->maps.as<int>(), *drels = F->rels.as<int>();
    C *fac = F->fac.as<C>();
    int *dinfo = F->info.as<int>();
    std::vector<const C *> upd_ptr(NN, nullptr); // where each node's update sits
    // the batched levels, deepest first, on the problem's stream
    DevBuf batch_upd, batch_desc;
    {
        SPM_TRY(batch_upd.ensure(sizeof(C) * std::max<size_t>(batch_upd_total, 1)));
        C *bu = batch_upd.as<C>();
        int maxd = 0;
        for (const Node &nd : nodes) maxd = std::max(maxd, nd.depth);
        std::vector<std::vector<BatchFront>> lv(maxd + 1);
        size_t nbf = 0;
        for (int id = 0; id < NN; ++id) {
            if (!batched[id]) continue;
            const Node &nd = nodes[id];
            upd_ptr[id] = bu + batch_upd_off[id];
            BatchFront b;
            b.own_off = (int)nd.own_off;
            b.nown = nd.nown;
            b.map_off = (int)nd.map_off;
            b.e0 = nd.elo[0]; b.e1 = nd.elo[1]; b.e2 = nd.elo[2];
            b.ew0 = nd.ehi[0] - nd.elo[0];
            b.ew1 = nd.ehi[1] - nd.elo[1];
            b.o3 = D * nd.nown;
            b.f = b.o3 + D * nd.nbnd;
            b.fac_off = nd.fac_off;
            b.upd = bu + batch_upd_off[id];
            b.nch = 0;
            for (int ch : {nd.left, nd.right}) {
                if (ch < 0 || nodes[ch].nbnd == 0) continue;
                b.ch_bc[b.nch] = D * nodes[ch].nbnd;
                b.ch_rel[b.nch] = (int)nodes[ch].rel_off;
                b.ch_upd[b.nch] = upd_ptr[ch];
                ++b.nch;
            }
            lv[nd.depth].push_back(b);
            ++nbf;
        }
        if (nbf > 0) {
            SPM_TRY(batch_desc.ensure(sizeof(BatchFront) * nbf));
            std::vector<BatchFront> all;
            struct Launch { size_t first, count; int fm, om; };
            std::vector<Launch> launches;
            size_t scratch_max = 0, ws_max = 0;
            for (int d = maxd; d >= 0; --d) {
                if (lv[d].empty()) continue;
                Launch ln{all.size(), lv[d].size(), 1, 1};
                for (const BatchFront &b : lv[d]) {
                    all.push_back(b);
                    ln.fm = std::max(ln.fm, b.f);
                    ln.om = std::max(ln.om, b.o3);
                }
                const size_t per = (size_t)ln.fm * ln.fm; // chunks of at most 2 GB of scratch
                const size_t chunk = std::max<size_t>(1, ((size_t)2 << 30) / (sizeof(C) * per));
                for (size_t c0 = 0; c0 < ln.count; c0 += chunk) {
                    Launch part = ln;
                    part.first = ln.first + c0;
                    part.count = std::min(chunk, ln.count - c0);
                    scratch_max = std::max(scratch_max, part.count * per);
                    ws_max = std::max(ws_max, panel_ws_bytes<C>(part.count, ln.fm, ln.om));
                    launches.push_back(part);
                }
            }
            SPM_CUDA_TRY(cudaMemcpy(batch_desc.ptr, all.data(), sizeof(BatchFront) * nbf, cudaMemcpyHostToDevice));
            DevBuf gscratch, panel_ws;
            SPM_TRY(gscratch.ensure(sizeof(C) * scratch_max));
            SPM_TRY(panel_ws.ensure(ws_max));
            const GridDesc gd2{n1, n2, n3d, D, SY.nsten};
            for (const Launch &ln : launches)
                SPM_TRY(factor_panels<C>(batch_desc.as<BatchFront>() + ln.first, (int)ln.count, ln.fm, ln.om, Sdev, dpts, dmaps,
                                         drels, gd2, gscratch.as<C>(), panel_ws.as<char>(), fac, pivot_floor<R>(), dinfo + 2, s));
            SPM_CUDA_TRY(cudaStreamSynchronize(s)); // before the scratch is freed
        }
    }
    // per-slot buffers and streams (slot ngroups - 1 is the problem's stream)
    struct Slot {
        DevBuf front, stack, gx;
        DenseWork *dense = nullptr;
        cudaStream_t st = nullptr;
        cudaEvent_t done = nullptr;
        ~Slot()
        {
            spm_dense_work_free(dense);
            if (st) cudaStreamDestroy(st);
            if (done) cudaEventDestroy(done);
        }
    };
    std::vector<Slot> slots(ngroups);
    DevBuf root_upd;
    SPM_TRY(root_upd.ensure(sizeof(C) * std::max<size_t>(root_upd_total, 1)));
    cudaEvent_t start_ev = nullptr;
    SPM_CUDA_TRY(cudaEventCreateWithFlags(&start_ev, cudaEventDisableTiming));
    SPM_CUDA_TRY(cudaEventRecord(start_ev, s)); // the streams start after the work queued so far
    for (int g = 0; g < ngroups; ++g) {
        Slot &sl = slots[g];
        SPM_TRY(sl.front.ensure(sizeof(C) * g_front[g]));
        SPM_TRY(sl.stack.ensure(sizeof(C) * g_stack[g]));
        if (half_store) SPM_TRY(sl.gx.ensure(sizeof(C) * g_gx[g]));
        sl.dense = spm_dense_work_new();
        if (g == ngroups - 1) {
            sl.st = nullptr; // use s
        } else {
            SPM_CUDA_TRY(cudaStreamCreateWithFlags(&sl.st, cudaStreamNonBlocking));
            SPM_CUDA_TRY(cudaEventCreateWithFlags(&sl.done, cudaEventDisableTiming));
            SPM_CUDA_TRY(cudaStreamWaitEvent(sl.st, start_ev, 0));
        }
    }
    cudaEventDestroy(start_ev);

    std::vector<size_t> top(ngroups, 0);
    auto factor_node = [&](int id) -> spm_status {
        Node &nd = nodes[id];
        const int g = slot(id);
        Slot &sl = slots[g];
        cudaStream_t ss = sl.st ? sl.st : s;
        C *front = sl.front.as<C>(), *stack = sl.stack.as<C>();
        const int o3 = D * nd.nown, b3 = D * nd.nbnd, f = o3 + b3;
        k_zero<C><<<blocks((long)f * f), 256, 0, ss>>>(front, (long)f * f);
        int ew0 = nd.ehi[0] - nd.elo[0], ew1 = nd.ehi[1] - nd.elo[1];
        k_front_assemble<C><<<blocks((long)nd.nown * gd.nsten), 256, 0, ss>>>(front, f, Sdev, dpts + nd.own_off,
                                                                               nd.nown, dmaps + nd.map_off, nd.elo[0],
                                                                               nd.elo[1], nd.elo[2], ew0, ew1, gd);
        // extend-add the children's updates
        for (int ch : {nd.left, nd.right}) {
            if (ch < 0) continue;
            Node &c = nodes[ch];
            int bc = D * c.nbnd;
            if (bc == 0) continue;
            k_extend_add<C><<<blocks((long)bc * bc), 256, 0, ss>>>(front, f, upd_ptr[ch], bc, drels + c.rel_off);
        }
        for (int ch : {nd.left, nd.right})
            if (ch >= 0 && !sub_root[ch] && !batched[ch]) top[g] -= upd_size[ch];
        SPM_CUDA_TRY(cudaGetLastError());
        // F11^{-1} by Gauss-Jordan (partial pivoting inside the own block, static
        // pivot floor), then with G = [F11^{-1}; F21 F11^{-1}] (f x o3, ld f) and
        // X = F11^{-1} F12 (o3 x b3, ld o3) stored after it:
        //   X = F11^{-1} F12,  G_bottom = F21 F11^{-1},  update = F22 - F21 X.
        C *G = half_store ? sl.gx.as<C>() : fac + nd.fac_off;
        SPM_TRY(spm_dense_inverse<C>(o3, front, f, G, f, pivot_floor<R>(), dinfo + 2, dinfo, sl.dense, ss));
        if (b3 > 0) {
            C *X = G + (long)f * o3;
            SPM_TRY(spm_dense_gemm<C>(o3, b3, o3, 1.0, G, f, front + (long)o3 * f, f, 0.0, X, o3, ss));
            SPM_TRY(spm_dense_gemm<C>(b3, o3, o3, 1.0, front + o3, f, G, f, 0.0, G + o3, f, ss));
            SPM_TRY(spm_dense_gemm<C>(b3, b3, o3, -1.0, front + o3, f, X, o3, 1.0, front + (long)o3 * f + o3, f, ss));
            // keep the update: on the slot's stack, or in the subtree root's own buffer
            C *dst = sub_root[id] ? root_upd.as<C>() + root_upd_off[id] : stack + top[g];
            if (!sub_root[id]) top[g] += upd_size[id];
            k_copy_block<C><<<blocks((long)b3 * b3), 256, 0, ss>>>(dst, b3, front + (long)o3 * f + o3, f, b3, b3);
            upd_ptr[id] = dst;
        }
        if constexpr (sizeof(R) == 4) {
            if (half_store) {
                float *sc = F->scales.as<float>() + nd.scale_off;
                __half2 *h = F->fac.as<__half2>() + nd.fac_off;
                const float2 *g2 = reinterpret_cast<const float2 *>(G);
                k_col_scales<<<o3, 256, 0, ss>>>(g2, f, o3, sc);
                k_to_half<<<blocks((long)f * o3), 256, 0, ss>>>(h, g2, f, o3, sc);
                if (b3 > 0) {
                    k_col_scales<<<b3, 256, 0, ss>>>(g2 + (long)f * o3, o3, b3, sc + o3);
                    k_to_half<<<blocks((long)o3 * b3), 256, 0, ss>>>(h + (long)f * o3, g2 + (long)f * o3, o3, b3, sc + o3);
                }
            }
        }
        SPM_CUDA_TRY(cudaGetLastError());
        return SPM_OK;
    };
    // the subtrees on the stream pool, then the nodes above them on the problem's stream
    for (int id = 0; id < NN; ++id)
        if (group[id] >= 0) SPM_TRY(factor_node(id));
    for (int g = 0; g < ngroups - 1; ++g) {
        SPM_CUDA_TRY(cudaEventRecord(slots[g].done, slots[g].st));
        SPM_CUDA_TRY(cudaStreamWaitEvent(s, slots[g].done, 0));
    }
    for (int id = 0; id < NN; ++id)
        if (group[id] < 0 && !batched[id]) SPM_TRY(factor_node(id));
    int hinfo[3] = {0, 0, 0};
    SPM_CUDA_TRY(cudaMemcpyAsync(hinfo, dinfo, sizeof(int) * 3, cudaMemcpyDeviceToHost, s));
    SPM_CUDA_TRY(cudaStreamSynchronize(s));
    slots.clear();
    root_upd.release();
    F->raised_pivots = hinfo[2];
    if (hinfo[0] != 0) {
        spm_set_error("a grid barrier of the Gauss-Jordan panel expired (code %d)", hinfo[0]);
        return SPM_ERR_TIMEOUT;
    }
    return build_solve_tiles<R>(F, pts);
}

// forward, deepest level first; backward, root first: launch(kernel of the direction, tiles, count)
template <typename KF, typename KB, typename L>
static void each_level(NDFactor *F, KF fwd, KB bwd, L launch)
{
    const SolveTile *tiles = F->st_tiles.as<const SolveTile>();
    const int NL = (int)F->levels.size();
    for (int l = 0; l < NL; ++l)
        if (F->levels[l].ntiles_f > 0) launch(fwd, tiles + F->levels[l].tiles_f, F->levels[l].ntiles_f);
    for (int l = NL - 1; l >= 0; --l)
        if (F->levels[l].ntiles_b > 0) launch(bwd, tiles + F->levels[l].tiles_b, F->levels[l].ntiles_b);
}

// Opt in to the shared memory, and, where tiles stream through registers, ask for the L1:
// lines in flight live there, and without a request the SM keeps the division that the
// kernel before it wanted (S^-1 at n = 32: 314 us among its like, 440 after Q).
template <typename K> static bool opt_in(K kernel, bool staged, int percent)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024) == cudaSuccess &&
           (staged || cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, percent) == cudaSuccess);
}

template <typename C, typename S, int NB, bool STAGED>
static void launch_levels(NDFactor *F, const S *M, C *W, C *Y, int nrhs, cudaStream_t s)
{
    // percent of 228 KB for the blocks that fit: NB x 256 sums and a reserved kilobyte each
    constexpr int percent = st_blocks<C, S, NB, STAGED>() * ((int)sizeof(C) * NB * ST_THREADS + 1024) / 2334 + 1;
    static PerDevice<bool> opted;
    opted.get([]() -> std::optional<bool> { // a failure is the last error, which the solve checks after its launches
        if (opt_in(k_nd_level<C, S, NB, true, STAGED>, STAGED, percent) && opt_in(k_nd_level<C, S, NB, false, STAGED>, STAGED, percent))
            return true;
        return std::nullopt;
    });
    // at most a 48 KB tile and 32 KB of sums
    const size_t smem = (STAGED ? sizeof(S) * (size_t)F->tile_elems : 0) + sizeof(C) * NB * std::max(ST_THREADS, F->tile_cols);
    each_level(F, k_nd_level<C, S, NB, true, STAGED>, k_nd_level<C, S, NB, false, STAGED>, [&](auto kernel, const SolveTile *t, int n) {
        launch_pdl(kernel, dim3(n), dim3(ST_THREADS), smem, s, M, (const float *)F->scales.as<float>(), t,
                   F->st_bnd.as<const int>(), W, Y, nrhs, F->tile_elems);
    });
}

// right-hand sides per pass over a tile: a tile is read once per group of NB
template <typename C, typename S>
static void launch_solve(NDFactor *F, const S *M, C *W, C *Y, int nrhs, cudaStream_t s)
{
    constexpr bool DBL = sizeof(C) == 16;
    if (nrhs > 8 && !DBL) launch_levels<C, S, DBL ? 8 : 16, DBL>(F, M, W, Y, nrhs, s);
    else if (nrhs > 4) launch_levels<C, S, 8, DBL>(F, M, W, Y, nrhs, s);
    else if (F->staged) {
        if (nrhs == 1) launch_levels<C, S, 1, true>(F, M, W, Y, nrhs, s);
        else if (nrhs == 2) launch_levels<C, S, 2, true>(F, M, W, Y, nrhs, s);
        else launch_levels<C, S, 4, true>(F, M, W, Y, nrhs, s);
    } else {
        if (nrhs == 1) launch_levels<C, S, 1, DBL>(F, M, W, Y, nrhs, s);
        else if (nrhs == 2) launch_levels<C, S, 2, DBL>(F, M, W, Y, nrhs, s);
        else launch_levels<C, S, 4, DBL>(F, M, W, Y, nrhs, s);
    }
}

template <typename R>
static spm_status solve_typed(NDFactor *F, const void *bv, void *xv, int nrhs, cudaStream_t s)
{
    using C = typename cplx_of<R>::type;
    const long N = F->D * F->npts;
    SPM_TRY(F->solve_ws.ensure(sizeof(C) * 2 * N * nrhs));
    C *W = F->solve_ws.as<C>(), *Y = W + N * nrhs;
    const unsigned grid = blocks(N * nrhs);
    launch_pdl(k_nd_enter<C>, dim3(grid), dim3(256), 0, s, W, Y, reinterpret_cast<const C *>(bv),
               F->st_point.as<const int>(), F->D, F->npts, nrhs);
    bool half = false;
    if constexpr (sizeof(R) == 4) {
        half = F->half_store;
        if (half) launch_solve<C, __half2>(F, F->fac.as<__half2>(), W, Y, nrhs, s);
    }
    if (!half) launch_solve<C, C>(F, F->fac.as<C>(), W, Y, nrhs, s);
    launch_pdl(k_nd_leave<C>, dim3(grid), dim3(256), 0, s, reinterpret_cast<C *>(xv), (const C *)Y,
               F->st_rank.as<const int>(), F->D, F->npts, nrhs);
    SPM_CUDA_TRY(cudaGetLastError());
    return SPM_OK;
}

namespace {

// probe right-hand side: components uniform in [-1, 1] from a splitmix64 hash of the index
__global__ void k_probe_rhs(double2 *b128, float2 *b64, long N)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N) return;
    uint64_t z = (uint64_t)i * 0x9E3779B97F4A7C15ull + 0x2545F4914F6CDD1Dull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    double2 v;
    v.x = (double)(z >> 40) * (2.0 / 16777216.0) - 1.0;
    v.y = (double)((z >> 16) & 0xFFFFFF) * (2.0 / 16777216.0) - 1.0;
    b128[i] = v;
    if (b64) b64[i] = make_float2((float)v.x, (float)v.y);
}

__global__ void k_widen(const float2 *a, double2 *b, long N)
{
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < N) b[i] = make_double2(a[i].x, a[i].y);
}

// acc[0] += sum |y - b|^2, acc[1] += sum |b|^2
__global__ void k_resid_norms(const double2 *y, const double2 *b, long N, double *acc)
{
    __shared__ double s0[256], s1[256];
    double r = 0, q = 0;
    for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < N; i += (long)gridDim.x * blockDim.x) {
        const double dx = y[i].x - b[i].x, dy = y[i].y - b[i].y;
        r += dx * dx + dy * dy;
        q += b[i].x * b[i].x + b[i].y * b[i].y;
    }
    s0[threadIdx.x] = r;
    s1[threadIdx.x] = q;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
        if (threadIdx.x < w) { s0[threadIdx.x] += s0[threadIdx.x + w]; s1[threadIdx.x] += s1[threadIdx.x + w]; }
        __syncthreads();
    }
    if (threadIdx.x == 0) { atomicAdd(acc, s0[0]); atomicAdd(acc + 1, s1[0]); }
}

// ||S x - b|| / ||b|| for x = S^{-1} b through the factor of precision `prec`,
// with b a fixed pseudo-random vector and S x formed in complex128.
spm_status probe_factor(const SparseSys &SY, int prec, double *relres)
{
    const long N = (long)SY.D * SY.points();
    cudaStream_t s = SY.stream;
    DevBuf buf;
    SPM_TRY(buf.ensure(sizeof(double2) * 3 * N + sizeof(float2) * 2 * N + 2 * sizeof(double)));
    double2 *b = buf.as<double2>(), *x = b + N, *y = x + N;
    float2 *b64 = reinterpret_cast<float2 *>(y + N), *x64 = b64 + N;
    double *acc = reinterpret_cast<double *>(x64 + N);
    const bool single = prec != SPM_C128;
    const unsigned g = (unsigned)((N + 255) / 256);
    k_probe_rhs<<<g, 256, 0, s>>>(b, single ? b64 : nullptr, N);
    if (single) {
        SPM_TRY(spm_nd_solve(*SY.slot64, SPM_C64, b64, x64, 1, s));
        k_widen<<<g, 256, 0, s>>>(x64, x, N);
    } else {
        SPM_TRY(spm_nd_solve(*SY.slot128, SPM_C128, b, x, 1, s));
    }
    SPM_TRY(SY.apply_S128(SY.ctx, x, y, s));
    SPM_CUDA_TRY(cudaMemsetAsync(acc, 0, 2 * sizeof(double), s));
    k_resid_norms<<<1024, 256, 0, s>>>(y, b, N, acc);
    double h[2];
    SPM_CUDA_TRY(cudaMemcpyAsync(h, acc, sizeof(h), cudaMemcpyDeviceToHost, s));
    SPM_CUDA_TRY(cudaStreamSynchronize(s));
    *relres = h[1] > 0 ? sqrt(h[0] / h[1]) : 0.0;
    if (!(*relres == *relres)) *relres = HUGE_VAL; // NaN: an unusable factor
    return SPM_OK;
}

// probe residual below which a factor is accepted without trying another tree
// (measured on the n = 48 / 64 media: complex64 factors up to 3e-2 and
// half-storage factors up to 0.3 keep GMRES within a few iterations of the
// best tree; factors above 1 stall it)
double probe_accept(int prec)
{
    return prec == SPM_C128 ? 1e-6 : (prec == SPM_C64H ? 3e-1 : 3e-2);
}

spm_status factor_once(const SparseSys &SY, int prec, int variant, NDFactor *&slot)
{
    spm_factor_free(slot);
    slot = nullptr;
    // A higher line takes more memory (3-D complex128 n = 32: 9.8 GB at the most with 1536,
    // 7.9 with 512): where it ends, the next lower line is tried.
    NDFactor *F = nullptr;
    spm_status st = SPM_ERR_OOM;
    int most = BATCH_LINES[0];
    while (st == SPM_ERR_OOM && most > 0) {
        if (F) cudaGetLastError(); // of the allocation that failed
        delete F;
        F = new NDFactor();
        F->prec = prec == SPM_C128 ? SPM_C128 : SPM_C64;
        st = prec == SPM_C128 ? factor_typed<double>(SY, F, false, variant, most)
                              : factor_typed<float>(SY, F, prec == SPM_C64H, variant, most);
        most = 0;
        for (const int line : BATCH_LINES)
            if (line < F->batch_line && !F->half_store) most = std::max(most, line);
    }
    if (st != SPM_OK) {
        delete F;
        return st;
    }
    slot = F;
    return SPM_OK;
}

} // namespace

// Factor, probe the factor's accuracy, and if the probe residual is above the
// acceptance level try the other tree variants, keeping the most accurate.
spm_status spm_nd_factor(const SparseSys &SY, int prec)
{
    const int fi = prec == SPM_C128 ? 0 : 1;
    NDFactor *&slot = fi == 0 ? *SY.slot128 : *SY.slot64;
    int best_v = -1, attempts = 0;
    double best = HUGE_VAL, last = HUGE_VAL;
    for (int v = 0; v < TREE_VARIANTS; ++v) {
        SPM_TRY(factor_once(SY, prec, v, slot));
        ++attempts;
        SPM_TRY(probe_factor(SY, prec, &last));
        if (last < best) { best = last; best_v = v; }
        if (last <= probe_accept(prec)) break;
    }
    if (best_v != slot->variant) { // a later variant was worse: rebuild the best one
        SPM_TRY(factor_once(SY, prec, best_v, slot));
        ++attempts;
    }
    SY.info[fi].variant = best_v;
    SY.info[fi].attempts = attempts;
    SY.info[fi].raised_pivots = slot->raised_pivots;
    SY.info[fi].stored_bytes = slot->stored_bytes;
    SY.info[fi].probe_relres = best;
    SY.info[fi].half_store = prec == SPM_C64H;
    return SPM_OK;
}

// Factor on one given tree variant (no retry); the probe is still recorded.
spm_status spm_nd_factor_tree(const SparseSys &SY, int prec, int variant)
{
    if (variant < 0 || variant >= TREE_VARIANTS) {
        spm_set_error("tree variant must be in [0, %d)", TREE_VARIANTS);
        return SPM_ERR_INVALID_ARG;
    }
    const int fi = prec == SPM_C128 ? 0 : 1;
    NDFactor *&slot = fi == 0 ? *SY.slot128 : *SY.slot64;
    SPM_TRY(factor_once(SY, prec, variant, slot));
    double r = 0;
    SPM_TRY(probe_factor(SY, prec, &r));
    SY.info[fi].variant = variant;
    SY.info[fi].attempts = 1;
    SY.info[fi].raised_pivots = slot->raised_pivots;
    SY.info[fi].stored_bytes = slot->stored_bytes;
    SY.info[fi].probe_relres = r;
    SY.info[fi].half_store = prec == SPM_C64H;
    return SPM_OK;
}

spm_status spm_nd_solve(NDFactor *F, int prec, const void *b, void *x, int nrhs, cudaStream_t s)
{
    if (!F) { spm_set_error("no factor of S in this precision"); return SPM_ERR_NOT_BUILT; }
    return prec == SPM_C128 ? solve_typed<double>(F, b, x, nrhs, s) : solve_typed<float>(F, b, x, nrhs, s);
}

// ---------------------------------------------------------------- 3-D problem
namespace {
spm_status apply_S128_3d(void *ctx, const void *x, void *y, cudaStream_t s)
{
    return spm_apply_S_impl(static_cast<spm_problem_s *>(ctx), SPM_C128, x, y, 1, s);
}

SparseSys sys_of(spm_problem_s *P)
{
    SparseSys S;
    S.dims[0] = S.dims[1] = S.dims[2] = P->n;
    S.D = 3;
    S.nsten = 27;
    S.S128 = P->S128.ptr;
    S.S64 = P->S64.ptr;
    S.stream = P->stream;
    S.slot128 = &P->fac128;
    S.slot64 = &P->fac64;
    S.info = P->fac_info;
    S.apply_S128 = apply_S128_3d;
    S.ctx = P;
    return S;
}
} // namespace

spm_status spm_factor_impl(spm_problem_s *P, int prec) { return spm_nd_factor(sys_of(P), prec); }

spm_status spm_factor_tree_impl(spm_problem_s *P, int prec, int variant)
{
    return spm_nd_factor_tree(sys_of(P), prec, variant);
}

spm_status spm_solveS_impl(spm_problem_s *P, int prec, const void *b, void *x, int nrhs, cudaStream_t s)
{
    return spm_nd_solve(prec == SPM_C128 ? P->fac128 : P->fac64, prec, b, x, nrhs, s);
}
