// Matrix-free apply of the Nystrom operator A = I + [k^2 G, G^d][m; p]
// (Eq. discrete_block) by zero-padded FFT convolution, plus the sparsifying
// row combination Q (Eq. nbr_i_block_alpha).
//
// Five passes per chunk of right-hand sides, each a batch of 1-D FFTs along
// one axis, register-resident with shared-memory exchanges between stages
// (fft_reg.cuh; fft.cuh serves only the one-time FP64 kernel spectra):
//   xfwd : w = [m E^1, m E^2, m E^3, p.E] formed on the fly, FFT along x
//          (n inputs zero-padded to L = 2n)          -> W1[b][4][z<n][y<n][xi<L]
//   yfwd : FFT along y (n -> L)                      -> W2[b][4][z<n][eta<L][xi<L]
//   zprod: FFT along z (n -> L), Fourier-side product
//          yhat_d = K0 what_d + K_d what_4  (K0 = k^2 Ghat/L^3, K_d = Ghat^d/L^3),
//          inverse FFT along z, keep z < n           -> W2 fields 0..2 (in place)
//   yinv : inverse FFT along eta, keep y < n         -> V1[b][3][z][y][xi] (in W1)
//   xinv : inverse FFT along xi, keep x < n, y = x + result
// The kernel spectra are stored as one octant [4][n+1]^3: Ghat is even in each
// frequency, Ghat^d is odd in frequency d and even in the others.
#include <cuda.h> // CUtensorMap (the encoder is reached through the runtime, no libcuda link)

#include <atomic>
#include <cstdio>
#include <cstring>
#include <string>
#include <mutex>
#include <type_traits>
#include <vector>

#include "fft.cuh"
#include "fft16.cuh"
#include "fft_reg.cuh"

namespace {

constexpr int NT = 256; // threads per block for every FFT pass

// -------------------------------------------------------------- strided lines
// Lines along a strided axis.  Element (b, f, z, pos, i) of the input sits at
//   in[b*ib + f*if_ + z*iz + pos*inner + i], 0 <= pos < nin, 0 <= i < inner,
// and is written to out[b*ob + f*of + z*oz + pos*inner + i], 0 <= pos < nout.
// grid = (inner/TX, nz, nb*F); each block transforms TX adjacent lines.
template <typename R, int DIR>
__global__ void __launch_bounds__(NT) k_cols(const typename cplx_of<R>::type *in,
                                             typename cplx_of<R>::type *out, int L, int logL,
                                             int nin, int nout, long inner, int F, long ib,
                                             long if_, long iz, long ob, long of, long oz, int TX,
                                             const typename cplx_of<R>::type *__restrict__ tw)
{
    using C = typename cplx_of<R>::type;
    extern __shared__ unsigned char smem_raw[];
    const int ls = L + 1;
    C *buf0 = reinterpret_cast<C *>(smem_raw);
    C *buf1 = buf0 + TX * ls;
    const long i0 = (long)blockIdx.x * TX;
    const int z = blockIdx.y;
    const int b = blockIdx.z / F, f = blockIdx.z - (blockIdx.z / F) * F;
    const C *src = in + b * ib + f * if_ + z * iz + i0;
    C *dst = out + b * ob + f * of + z * oz + i0;
    for (int idx = threadIdx.x; idx < TX * L; idx += blockDim.x) {
        int pos = idx / TX, t = idx - pos * TX;
        buf0[t * ls + pos] = pos < nin ? src[pos * inner + t] : czero<C>();
    }
    __syncthreads();
    C *res = smem_fft<DIR>(buf0, buf1, L, logL, TX, ls, tw);
    for (int idx = threadIdx.x; idx < TX * nout; idx += blockDim.x) {
        int pos = idx / TX, t = idx - pos * TX;
        dst[pos * inner + t] = res[t * ls + pos];
    }
}

// ================================================================ v2 passes
// Register-resident line FFTs (fft_reg.cuh): thread t of a line holds elements
// t + T m, m = 0..7, T = L/8.  Strided passes use TX adjacent columns per block
// with thread (c, t) at tid = c + TX t, so each load/store instruction of a warp
// touches whole 128-byte rows.

// columns per strided-pass block: 128-byte rows, fewer at L = 512 so the block
// (TX * L/8 threads) keeps at least 128 registers per thread
template <typename R, int L> struct tx_of {
    static constexpr int w = (sizeof(R) == 4 ? 16 : 8) / (L >= 512 ? 2 : 1);
    static constexpr int v = w < L ? w : L; // never wider than a row of L elements
};

// Blocks per SM asked of the compiler for a strided pass whose threads get at
// most `regs` registers; 0 leaves its own choice.  Asked for at L = 128 in
// complex64 only, where that choice is a bad one: k2_cols2 took 74 registers
// (three blocks; 14.0 us against 12.1 with four), k2_zprod4 100 (still two
// blocks, its loads in shorter batches; 30.7 us against 26.7 with 128).  One
// application at n = 64: 70.9 us, 74.1 without.  From L = 256 on it already
// compiles to these numbers, and a bound of one block there makes k2_cols2 keep
// fewer blocks resident (L = 512: 946 us against 633); below L = 64 it
// takes up to 70, not measured with a bound.
template <typename R, int L> constexpr int pass_blocks(int regs)
{
    return sizeof(R) == 4 && L == 128 ? 65536 / (regs * tx_of<R, L>::v * L / 8) : 0;
}

constexpr int ZPROD_FOUR = 0, ZPROD_ONE = 1, ZPROD_TMA = 2, ZPROD_E16 = 3, ZPROD_STAGED = 4, ZPROD_SPLIT = 5; // z-pass kernels
constexpr int ZPLAN_FUSED_XY = 8; // plan bit: x and y passes fused per z-plane (L = 64, 128)

template <int L> __device__ __forceinline__ int xpad(int pos) { return pos + (pos >> 3); }

// xfwd: w_f of one grid row per line, FFT along x (pruned), 4 fields in turn, or (APART)
// one field per block, blockIdx.y.
template <typename R, int L, bool APART>
__global__ void __launch_bounds__(256) k2_xfwd(const typename cplx_of<R>::type *__restrict__ x,
                                               const typename cplx_of<R>::type *__restrict__ m,
                                               const typename cplx_of<R>::type *__restrict__ p,
                                               typename cplx_of<R>::type *__restrict__ W1, int nrows,
                                               const typename cplx_of<R>::type *__restrict__ tw)
{
    pdl_wait_and_trigger();
    using C = typename cplx_of<R>::type;
    constexpr int E = line_elems(L), H = E / 2;
    constexpr int T = L / E, n = L / 2, LS = L + L / 8;
    extern __shared__ unsigned char smem_raw[];
    C *sm = reinterpret_cast<C *>(smem_raw);
    const int line = threadIdx.x / T, t = threadIdx.x % T;
    const int g = blockIdx.x * (blockDim.x / T) + line;
    const bool ok = g < nrows;
    const long n2 = (long)n * n, n3 = n2 * n;
    const long b = ok ? g / n2 : 0, zy = ok ? g - b * n2 : 0;
    const C *xb = x + b * 3 * n3;
    C *lb = sm + line * LS;
    auto buf = [&](int pos) -> C & { return lb[xpad<L>(pos)]; };
    auto sync = [&]() { if (T <= 32) __syncwarp(); else __syncthreads(); };
    // E = 8: the 7 inputs of the row stay in registers for the 4 fields;
    // E = 12: reloaded per field (cached in L1) to keep register pressure down
    constexpr bool CACHE = (E == 8);
    constexpr int HC = CACHE ? H : 1;
    C e[3][HC], mm[HC], pp[3][HC];
    if constexpr (CACHE) {
#pragma unroll
        for (int q = 0; q < H; ++q) {
            const long off = zy * n + t + T * q;
            if (ok) {
                e[0][q] = xb[off]; e[1][q] = xb[n3 + off]; e[2][q] = xb[2 * n3 + off];
                mm[q] = m[off];
                pp[0][q] = p[off]; pp[1][q] = p[n3 + off]; pp[2][q] = p[2 * n3 + off];
            } else {
                e[0][q] = e[1][q] = e[2][q] = mm[q] = pp[0][q] = pp[1][q] = pp[2][q] = czero<C>();
            }
        }
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        if (APART && f != (int)blockIdx.y) continue;
        C v[E];
#pragma unroll
        for (int q = 0; q < H; ++q) {
            C w = czero<C>();
            if constexpr (CACHE) {
                if (f < 3) w = cmul(mm[q], e[f][q]);
                else w = cfma(pp[0][q], e[0][q], cfma(pp[1][q], e[1][q], cmul(pp[2][q], e[2][q])));
            } else if (ok) {
                const long off = zy * n + t + T * q;
                if (f < 3) w = cmul(m[off], xb[f * n3 + off]);
                else w = cfma(p[off], xb[off], cfma(p[n3 + off], xb[n3 + off], cmul(p[2 * n3 + off], xb[2 * n3 + off])));
            }
            v[q] = w;
            v[q + H] = czero<C>();
        }
        line_fft<-1, L, true>(v, t, buf, sync, tw);
        if (ok) {
            C *dst = W1 + ((b * 4 + f) * n2 + zy) * L;
#pragma unroll
            for (int q = 0; q < E; ++q) dst[t + T * q] = v[q];
        }
        sync();
    }
}

// Strided lines: element (b, f, z, pos, i) at in[b*ib + f*if_ + z*iz + pos*inner + i];
// grid (inner/TX, nz, nb*F).  nin, nout in {L/2, L}.
template <typename R, int L, int DIR, bool PRUNE>
__global__ void __launch_bounds__(tx_of<R, L>::v * L / line_elems(L)) k2_cols(const typename cplx_of<R>::type *in, typename cplx_of<R>::type *out,
                                                int nout, long inner, int F, long ib, long if_, long iz, long ob,
                                                long of, long oz, const typename cplx_of<R>::type *__restrict__ tw)
{
    pdl_wait_and_trigger();
    using C = typename cplx_of<R>::type;
    constexpr int E = line_elems(L), H = E / 2;
    constexpr int T = L / E, TX = tx_of<R, L>::v;
    extern __shared__ unsigned char smem_raw[];
    C *sm = reinterpret_cast<C *>(smem_raw);
    const int c = threadIdx.x % TX, t = threadIdx.x / TX;
    const long i0 = (long)blockIdx.x * TX;
    const int z = blockIdx.y;
    const int b = blockIdx.z / F, f = blockIdx.z % F;
    const C *src = in + b * ib + f * if_ + z * iz + i0 + c;
    C *dst = out + b * ob + f * of + z * oz + i0 + c;
    C v[E];
#pragma unroll
    for (int q = 0; q < E; ++q) v[q] = (!PRUNE || q < H) ? src[(long)(t + T * q) * inner] : czero<C>();
    auto buf = [&](int pos) -> C & { return sm[pos * TX + c]; };
    auto sync = [&]() { __syncthreads(); };
    line_fft<DIR, L, PRUNE>(v, t, buf, sync, tw);
#pragma unroll
    for (int q = 0; q < E; ++q)
        if (t + T * q < nout) dst[(long)(t + T * q) * inner] = v[q];
}

// Same strided lines, two z planes per block (E = 8 lengths): both planes'
// columns are loaded before either is transformed, and the two transforms share
// every barrier (fft_lines), so each thread keeps twice the loads in flight.
template <typename R, int L, int DIR, bool PRUNE>
__global__ void __launch_bounds__(tx_of<R, L>::v * L / 8, pass_blocks<R, L>(64)) k2_cols2(const typename cplx_of<R>::type *in, typename cplx_of<R>::type *out,
                                                                 int nout, long inner, int F, long ib, long if_, long iz, long ob,
                                                                 long of, long oz, const typename cplx_of<R>::type *__restrict__ tw)
{
    pdl_wait_and_trigger();
    using C = typename cplx_of<R>::type;
    constexpr int T = L / 8, TX = tx_of<R, L>::v;
    extern __shared__ unsigned char smem_raw[];
    C *sm = reinterpret_cast<C *>(smem_raw); // [2][L][TX]
    const int c = threadIdx.x % TX, t = threadIdx.x / TX;
    const long i0 = (long)blockIdx.x * TX;
    const int z0 = 2 * blockIdx.y;
    const int b = blockIdx.z / F, f = blockIdx.z % F;
    C v[2][8];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const C *src = in + b * ib + f * if_ + (z0 + k) * iz + i0 + c;
#pragma unroll
        for (int q = 0; q < 8; ++q) v[k][q] = (!PRUNE || q < 4) ? src[(long)(t + T * q) * inner] : czero<C>();
    }
    auto buf = [&](int k, int pos) -> C & { return sm[(k * L + pos) * TX + c]; };
    auto sync = [&]() { __syncthreads(); };
    fftr::fft_lines<DIR, L, PRUNE, 2>(v, t, buf, sync, tw);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        C *dst = out + b * ob + f * of + (z0 + k) * oz + i0 + c;
#pragma unroll
        for (int q = 0; q < 8; ++q)
            if (t + T * q < nout) dst[(long)(t + T * q) * inner] = v[k][q];
    }
}

// zprod: lines along z of W2[b][4][z<n][eta][xi] (TX adjacent columns), product
// with the octant spectra, inverse along z, keep z < n (in place, fields 0..2).
// The four fields' columns are prefetched into shared memory with cp.async at
// the start (one commit group per field, in the order they are consumed); each
// thread reads back only the elements it copied, so no block barrier is needed
// for the prefetch.
template <typename R, int L>
__global__ void __launch_bounds__(tx_of<R, L>::v * L / line_elems(L)) k2_zprod1(typename cplx_of<R>::type *W2,
                                                 const typename cplx_of<R>::type *__restrict__ spec,
                                                 const typename cplx_of<R>::type *__restrict__ tw)
{
    pdl_wait_and_trigger();
    using C = typename cplx_of<R>::type;
    constexpr int E = line_elems(L), H = E / 2;
    constexpr int T = L / E, TX = tx_of<R, L>::v, n = L / 2, n1 = n + 1;
    constexpr long L2 = (long)L * L, oct = (long)n1 * n1 * n1, fs = (long)n * L * L;
    extern __shared__ unsigned char smem_raw[];
    C *sm = reinterpret_cast<C *>(smem_raw);
    C *pre = sm + L * TX; // [4 fields in consumption order][n][TX]
    const int c = threadIdx.x % TX, t = threadIdx.x / TX;
    const long col = (long)blockIdx.x * TX + c;
    const int b = blockIdx.y;
    C *base = W2 + (long)b * 4 * fs + col;
    const int eta = (int)(col / L), xi = (int)(col % L);
    const int a1 = xi <= n ? xi : L - xi, a2 = eta <= n ? eta : L - eta;
    auto buf = [&](int pos) -> C & { return sm[pos * TX + c]; };
    auto sync = [&]() { __syncthreads(); };
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const int f = g == 0 ? 3 : g - 1;
#pragma unroll
        for (int q = 0; q < H; ++q) {
            const int z = t + T * q;
            cp_async<sizeof(C)>(&pre[(g * n + z) * TX + c], base + f * fs + (long)z * L2);
        }
        cp_async_commit();
    }
    C w4[E];
    cp_async_wait<3>();
#pragma unroll
    for (int q = 0; q < H; ++q) w4[q] = pre[(0 * n + t + T * q) * TX + c];
#pragma unroll
    for (int q = H; q < E; ++q) w4[q] = czero<C>();
    line_fft<-1, L, true>(w4, t, buf, sync, tw);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        C v[E];
        if (d == 0) cp_async_wait<2>();
        else if (d == 1) cp_async_wait<1>();
        else cp_async_wait<0>();
#pragma unroll
        for (int q = 0; q < H; ++q) v[q] = pre[((d + 1) * n + t + T * q) * TX + c];
#pragma unroll
        for (int q = H; q < E; ++q) v[q] = czero<C>();
        line_fft<-1, L, true>(v, t, buf, sync, tw);
        const int fr_fixed = d == 0 ? xi : eta;
#pragma unroll
        for (int q = 0; q < E; ++q) {
            const int zeta = t + T * q;
            const int a3 = zeta <= n ? zeta : L - zeta;
            const long o = ((long)a3 * n1 + a2) * n1 + a1;
            C K0 = spec[o], Kd = spec[(1 + d) * oct + o];
            const int fr = d == 2 ? zeta : fr_fixed;
            if (fr > n) { Kd.x = -Kd.x; Kd.y = -Kd.y; }
            v[q] = cfma(K0, v[q], cmul(Kd, w4[q]));
        }
        line_fft<1, L, false>(v, t, buf, sync, tw);
#pragma unroll
        for (int q = 0; q < H; ++q) base[d * fs + (long)(t + T * q) * L2] = v[q];
    }
}

// zprod, staged: as k2_zprod1 (the four fields' columns prefetched with
// cp.async, one field transformed at a time), and also the tile's kernel
// spectra and the twiddle table staged in shared memory, so that no global load
// remains between the transforms.  The tile's spectra: for each kernel K and
// folded z-frequency a3 in [0, n], the TX values at the tile's folded (a2, a1)
// (ks[K][a3][c]); K(zeta) and K(L - zeta) share the entry (with the sign of K_3
// flipped), so n + 1 rows cover all L frequencies.
template <typename R, int L> struct zst {
    using C = typename cplx_of<R>::type;
    static constexpr int TX = tx_of<R, L>::v, n = L / 2, THREADS = TX * L / line_elems(L);
    static constexpr size_t elems = (size_t)L * TX + 4 * n * TX + 4 * (n + 1) * TX + L;
    static constexpr size_t smem = sizeof(C) * elems;
};

template <typename R, int L>
__global__ void __launch_bounds__(zst<R, L>::THREADS) k2_zstaged(typename cplx_of<R>::type *W2,
                                                                const typename cplx_of<R>::type *__restrict__ spec,
                                                                const typename cplx_of<R>::type *__restrict__ tw)
{
    pdl_wait_and_trigger();
    using C = typename cplx_of<R>::type;
    constexpr int E = line_elems(L), H = E / 2;
    constexpr int T = L / E, TX = tx_of<R, L>::v, n = L / 2, n1 = n + 1, THR = zst<R, L>::THREADS;
    constexpr long L2 = (long)L * L, oct = (long)n1 * n1 * n1, fs = (long)n * L * L;
    extern __shared__ unsigned char smem_raw[];
    C *sm = reinterpret_cast<C *>(smem_raw); // exchange [L][TX]
    C *pre = sm + L * TX;                    // [4 fields in consumption order][n][TX]
    C *ks = pre + 4 * n * TX;                // [4 kernels][n + 1][TX]
    C *stw = ks + 4 * n1 * TX;               // [L] twiddles
    const int c = threadIdx.x % TX, t = threadIdx.x / TX;
    const long col0 = (long)blockIdx.x * TX, col = col0 + c;
    const int b = blockIdx.y;
    C *base = W2 + (long)b * 4 * fs + col;
    const int eta = (int)(col / L), xi = (int)(col % L);
    const int a1 = xi <= n ? xi : L - xi, a2 = eta <= n ? eta : L - eta;
    // group 0: p.E (consumed first)
#pragma unroll
    for (int q = 0; q < H; ++q) {
        const int z = t + T * q;
        cp_async<sizeof(C)>(&pre[z * TX + c], base + 3 * fs + (long)z * L2);
    }
    cp_async_commit();
    // group 1: the tile's spectra (every thread copies a share; read after a barrier)
    {
        const int xi0 = (int)(col0 % L);
        for (int i = threadIdx.x; i < 4 * n1 * TX; i += THR) {
            const int k = i / (n1 * TX), a3 = (i / TX) % n1, cc = i % TX;
            const int x = xi0 + cc, b1 = x <= n ? x : L - x;
            cp_async<sizeof(C)>(&ks[i], spec + k * oct + ((long)a3 * n1 + a2) * n1 + b1);
        }
    }
    cp_async_commit();
    // groups 2..4: E^1, E^2, E^3
#pragma unroll
    for (int g = 1; g < 4; ++g) {
#pragma unroll
        for (int q = 0; q < H; ++q) {
            const int z = t + T * q;
            cp_async<sizeof(C)>(&pre[(g * n + z) * TX + c], base + (g - 1) * fs + (long)z * L2);
        }
        cp_async_commit();
    }
    for (int i = threadIdx.x; i < L; i += THR) stw[i] = tw[i];
    auto buf = [&](int pos) -> C & { return sm[pos * TX + c]; };
    auto sync = [&]() { __syncthreads(); };
    C w4[E];
    cp_async_wait<4>();
#pragma unroll
    for (int q = 0; q < H; ++q) w4[q] = pre[(t + T * q) * TX + c];
#pragma unroll
    for (int q = H; q < E; ++q) w4[q] = czero<C>();
    __syncthreads(); // the twiddle table
    line_fft<-1, L, true>(w4, t, buf, sync, stw);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        C v[E];
        // this thread's copies of E^(d+1) and of the spectra have landed; the
        // barriers inside the forward transform below make every thread's
        // spectrum copies visible before the product reads them
        if (d == 0) cp_async_wait<2>();
        else if (d == 1) cp_async_wait<1>();
        else cp_async_wait<0>();
#pragma unroll
        for (int q = 0; q < H; ++q) v[q] = pre[((d + 1) * n + t + T * q) * TX + c];
#pragma unroll
        for (int q = H; q < E; ++q) v[q] = czero<C>();
        line_fft<-1, L, true>(v, t, buf, sync, stw);
        const int fr_fixed = d == 0 ? xi : eta;
#pragma unroll
        for (int q = 0; q < E; ++q) {
            const int zeta = t + T * q;
            const int a3 = zeta <= n ? zeta : L - zeta;
            const C K0 = ks[a3 * TX + c];
            C Kd = ks[((1 + d) * n1 + a3) * TX + c];
            const int fr = d == 2 ? zeta : fr_fixed;
            if (fr > n) { Kd.x = -Kd.x; Kd.y = -Kd.y; }
            v[q] = cfma(K0, v[q], cmul(Kd, w4[q]));
        }
        line_fft<1, L, false>(v, t, buf, sync, stw);
#pragma unroll
        for (int q = 0; q < H; ++q) base[d * fs + (long)(t + T * q) * L2] = v[q];
    }
}

// zprod, split into even and odd frequencies (L = 64, 128, 256): with
// H = L/2 = n and x[z] = 0 for z >= H,
//   X[2k]     = DFT_H(x)[k],   X[2k + 1] = DFT_H(x . w_L^z)[k],
// and the inverse restricted to z < H is
//   y[z] = IDFT_H(Y_even)[z] + conj(w_L^z) IDFT_H(Y_odd)[z],
// so every length-L transform of the z-pass becomes two length-H transforms
// that share their exchanges (fftr::fft_lines with K = 2), and the radix-2
// stage of L = 128 disappears.  256 threads: TX = 256 / (H/8) columns.
template <typename R, int L> struct zsp {
    using C = typename cplx_of<R>::type;
    static constexpr int H = L / 2, T = H / 8, TX = 256 / T;
    // exchange [2][H][TX], transformed p.E [16][256] (each thread its own), tables H + L
    static constexpr size_t smem = sizeof(C) * ((size_t)2 * H * TX + 16 * 256 + H + L);
    static_assert(L == 64 || L == 128 || L == 256, "split z-pass lengths");
};

template <typename R, int L>
__global__ void __launch_bounds__(256, 2) k2_zsplit(typename cplx_of<R>::type *W2,
                                                 const typename cplx_of<R>::type *__restrict__ spec,
                                                 const typename cplx_of<R>::type *__restrict__ tw)
{
    pdl_wait_and_trigger();
    using C = typename cplx_of<R>::type;
    constexpr int H = zsp<R, L>::H, T = zsp<R, L>::T, TX = zsp<R, L>::TX, n = H, n1 = n + 1;
    constexpr long L2 = (long)L * L, oct = (long)n1 * n1 * n1, fs = (long)n * L * L;
    extern __shared__ unsigned char smem_raw[];
    C *xch = reinterpret_cast<C *>(smem_raw); // [2 lines][H][TX]
    C *w4s = xch + 2 * H * TX;               // transformed p.E: [16][256], thread-private columns
    C *stw = w4s + 16 * 256;                 // length-H twiddles: w_H^j = w_L^(2j)
    C *stl = stw + H;                        // length-L twiddles w_L^j
    const int c = threadIdx.x % TX, t = threadIdx.x / TX;
    const long col = (long)blockIdx.x * TX + c;
    const int b = blockIdx.y;
    C *base = W2 + (long)b * 4 * fs + col;
    const int eta = (int)(col / L), xi = (int)(col % L);
    const int a1 = xi <= n ? xi : L - xi, a2 = eta <= n ? eta : L - eta;
    for (int i = threadIdx.x; i < L; i += blockDim.x) {
        const C w = tw[i];
        stl[i] = w;
        if ((i & 1) == 0) stw[i >> 1] = w;
    }
    __syncthreads();
    auto buf = [&](int k, int pos) -> C & { return xch[(k * H + pos) * TX + c]; };
    auto sync = [&]() { __syncthreads(); };
    // forward: field f -> (even, odd) halves of its spectrum at k = t + T m
    auto forward = [&](int f, C (&v)[2][8]) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const C xz = base[f * fs + (long)(t + T * q) * L2];
            v[0][q] = xz;
            v[1][q] = cmul(xz, stl[t + T * q]);
        }
        fftr::fft_lines<-1, H, false, 2>(v, t, buf, sync, stw);
    };
    {
        C w4[2][8];
        forward(3, w4);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < 8; ++q) w4s[(h * 8 + q) * 256 + threadIdx.x] = w4[h][q];
    }
#pragma unroll 1
    for (int d = 0; d < 3; ++d) {
        C v[2][8];
        forward(d, v);
        const int fr_fixed = d == 0 ? xi : eta;
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const int zeta = 2 * (t + T * q) + h;
                const int a3 = zeta <= n ? zeta : L - zeta;
                const long o = ((long)a3 * n1 + a2) * n1 + a1;
                C K0 = spec[o], Kd = spec[(1 + d) * oct + o];
                const int fr = d == 2 ? zeta : fr_fixed;
                if (fr > n) { Kd.x = -Kd.x; Kd.y = -Kd.y; }
                v[h][q] = cfma(K0, v[h][q], cmul(Kd, w4s[(h * 8 + q) * 256 + threadIdx.x]));
            }
        fftr::fft_lines<1, H, false, 2>(v, t, buf, sync, stw);
#pragma unroll
        for (int q = 0; q < 8; ++q) base[d * fs + (long)(t + T * q) * L2] = v[0][q] + cmulc(v[1][q], stl[t + T * q]);
    }
}

// zprod, E = 8: the four forward z-transforms run together (shared barriers),
// then the three products and the three inverse transforms together.
template <typename R, int L>
__global__ void __launch_bounds__(tx_of<R, L>::v * L / 8, pass_blocks<R, L>(128)) k2_zprod4(typename cplx_of<R>::type *W2,
                                                                  const typename cplx_of<R>::type *__restrict__ spec,
                                                                  const typename cplx_of<R>::type *__restrict__ tw)
{
    pdl_wait_and_trigger();
    using C = typename cplx_of<R>::type;
    constexpr int T = L / 8, TX = tx_of<R, L>::v, n = L / 2, n1 = n + 1;
    constexpr long L2 = (long)L * L, oct = (long)n1 * n1 * n1, fs = (long)n * L * L;
    extern __shared__ unsigned char smem_raw[];
    C *sm = reinterpret_cast<C *>(smem_raw); // 4 exchange buffers [4][L][TX]
    const int c = threadIdx.x % TX, t = threadIdx.x / TX;
    const long col = (long)blockIdx.x * TX + c;
    const int b = blockIdx.y;
    C *base = W2 + (long)b * 4 * fs + col;
    const int eta = (int)(col / L), xi = (int)(col % L);
    const int a1 = xi <= n ? xi : L - xi, a2 = eta <= n ? eta : L - eta;
    auto buf = [&](int k, int pos) -> C & { return sm[(k * L + pos) * TX + c]; };
    auto sync = [&]() { __syncthreads(); };
    C w[4][8]; // fields 0, 1, 2 and p.E (index 3)
#pragma unroll
    for (int f = 0; f < 4; ++f) {
#pragma unroll
        for (int q = 0; q < 4; ++q) w[f][q] = base[f * fs + (long)(t + T * q) * L2];
#pragma unroll
        for (int q = 4; q < 8; ++q) w[f][q] = czero<C>();
    }
    fftr::fft_lines<-1, L, true, 4>(w, t, buf, sync, tw);
    C v[3][8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int zeta = t + T * q;
        const int a3 = zeta <= n ? zeta : L - zeta;
        const long o = ((long)a3 * n1 + a2) * n1 + a1;
        const C K0 = spec[o];
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            C Kd = spec[(1 + d) * oct + o];
            const int fr = d == 0 ? xi : (d == 1 ? eta : zeta);
            if (fr > n) { Kd.x = -Kd.x; Kd.y = -Kd.y; }
            v[d][q] = cfma(K0, w[d][q], cmul(Kd, w[3][q]));
        }
    }
    fftr::fft_lines<1, L, false, 3>(v, t, buf, sync, tw);
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int q = 0; q < 4; ++q) base[d * fs + (long)(t + T * q) * L2] = v[d][q];
}

// The same on small grids, a line per thread group: a quarter of the block's threads per
// field, TX adjacent columns.  The groups transform their fields side by side, a warp each;
// p.E's transform goes to the other three through shared memory; they form the product and
// transform back.  Four times the warps, each with two transforms instead of seven one after
// another: in complex128 a warp's FP64 instruction takes 64 cycles, and at n = 16 the
// four-line kernel is 128 warps on 608 schedulers (33.9 us; this one 14.3; n = 8 28.7 and
// 12.3).  It serves complex128 up to L = 32 and complex64 up to 16; at L = 32 in complex64
// the four-line kernel, which shares its twiddles and spectra between the fields, is little
// slower for one right-hand side (6.8 us against 5.8) and faster for blocks of them (A with
// 8 16.9 us against 18.0, with 64 39.7 against 49.8), as it is from L = 64 on in both
// (complex64 n = 64: 30.7 against 45.1 us, complex128 567 against 590).  By L alone, so that
// a block of right-hand sides gives the bits of single ones.
template <typename R, int L> constexpr bool zfield_serves() { return L <= (sizeof(R) == 8 ? 32 : 16); }
template <typename R, int L> struct zfl {
    using C = typename cplx_of<R>::type;
    static constexpr int T = L / 8;
    static constexpr int TX = 32 / T; // a warp per field
    static_assert(L <= 32, "small grids");
    static constexpr int GROUP = TX * T, THREADS = 4 * GROUP;
    static constexpr size_t smem = sizeof(C) * 4 * L * TX;
};
template <typename R, int L>
__global__ void __launch_bounds__(zfl<R, L>::THREADS) k2_zfield(typename cplx_of<R>::type *W2,
                                                                  const typename cplx_of<R>::type *__restrict__ spec,
                                                             const typename cplx_of<R>::type *__restrict__ tw)
{
    pdl_wait_and_trigger();
    using C = typename cplx_of<R>::type;
    constexpr int T = zfl<R, L>::T, TX = zfl<R, L>::TX, GROUP = zfl<R, L>::GROUP, n = L / 2, n1 = n + 1;
    constexpr long L2 = (long)L * L, oct = (long)n1 * n1 * n1, fs = (long)n * L * L;
    extern __shared__ unsigned char smem_raw[];
    C *sm = reinterpret_cast<C *>(smem_raw); // 4 exchange buffers [4][L][TX]
    const int f = threadIdx.x / GROUP, tid = threadIdx.x % GROUP, c = tid % TX, t = tid / TX;
    const long col = (long)blockIdx.x * TX + c;
    C *base = W2 + (long)blockIdx.y * 4 * fs + f * fs + col;
    C *own = sm + f * L * TX;
    auto buf = [&](int pos) -> C & { return own[pos * TX + c]; };
    auto sync = [&]() { __syncwarp(); }; // a group is a warp
    static_assert(GROUP == 32, "one warp per field");
    C v[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = base[(long)(t + T * q) * L2];
#pragma unroll
    for (int q = 4; q < 8; ++q) v[q] = czero<C>();
    fftr::fft_line<-1, L, true>(v, t, buf, sync, tw);
    C *w4 = sm + 3 * L * TX; // group 3's buffer; its last exchange has been read
    if (f == 3) {
#pragma unroll
        for (int q = 0; q < 8; ++q) w4[(t + T * q) * TX + c] = v[q];
    }
    __syncthreads();
    if (f == 3) return;
    const int eta = (int)(col / L), xi = (int)(col % L);
    const int a1 = xi <= n ? xi : L - xi, a2 = eta <= n ? eta : L - eta;
    const C *Kf = spec + (long)a2 * n1 + a1;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int zeta = t + T * q;
        const int o = (zeta <= n ? zeta : L - zeta) * n1 * n1;
        const C K0 = Kf[o];
        C Kd = Kf[(1 + f) * oct + o];
        const int fr = f == 0 ? xi : (f == 1 ? eta : zeta);
        if (fr > n) { Kd.x = -Kd.x; Kd.y = -Kd.y; }
        v[q] = cfma(K0, v[q], cmul(Kd, w4[zeta * TX + c]));
    }
    fftr::fft_line<1, L, false>(v, t, buf, sync, tw);
#pragma unroll
    for (int q = 0; q < 4; ++q) base[(long)(t + T * q) * L2] = v[q];
}

// Exchange buffer of a 16-per-thread line shared by TX columns: position pos of
// column c at (pos + pos/16) TX + c.  The pad of one row per 16 positions keeps
// the stage-0 writes (positions 16 t + q) of the T threads of a half-warp on
// distinct banks when TX < 16.
template <int L> __host__ __device__ constexpr int xch16_rows() { return L + L / 16; }
__device__ __forceinline__ int xch16(int pos, int TX, int c) { return (pos + (pos >> 4)) * TX + c; }

template <typename R, int L> struct zp16 {
    // 128 threads (complex64) or 64 (complex128) per block: TX columns x L/16
    static constexpr int TX = (sizeof(R) == 4 ? 16 : 8) * 128 / L;
    static constexpr int THREADS = TX * (L / 16);
    // blocks per SM the register budget is sized for: about 168 registers a thread
    // in complex64, 255 in complex128
    static constexpr int MINB = 65536 / (THREADS * (sizeof(R) == 4 ? 168 : 255));
    static constexpr size_t smem()
    {
        using C = typename cplx_of<R>::type;
        return sizeof(C) * ((size_t)(xch16_rows<L>() + L) * TX + 4 * (L / 2) * TX + (L == 512 ? L : 0));
    }
};

// z-pass with 16 values per thread (fft16.cuh; L = 128, 256, 512): TX adjacent
// columns per block, the four fields' columns (pruned half) prefetched into
// shared memory with cp.async in consumption order (p.E first), the middle
// stage's twiddles computed once per thread and kept in registers, p.E
// transformed once and kept in registers, then per d: forward transform,
// Fourier-side product, inverse transform, z < n stored in place.
template <typename R, int L>
__global__ void __launch_bounds__(zp16<R, L>::THREADS, zp16<R, L>::MINB) k3_zpass(typename cplx_of<R>::type *W2,
                                                              const typename cplx_of<R>::type *__restrict__ spec,
                                                              const typename cplx_of<R>::type *__restrict__ tw)
{
    pdl_wait_and_trigger();
    using C = typename cplx_of<R>::type;
    constexpr int T = L / 16, TX = zp16<R, L>::TX, n = L / 2, n1 = n + 1;
    constexpr long L2 = (long)L * L, oct = (long)n1 * n1 * n1, fs = (long)n * L * L;
    extern __shared__ unsigned char smem_raw[];
    C *xch = reinterpret_cast<C *>(smem_raw); // exchange buffer [L + L/16][TX]
    C *w4s = xch + xch16_rows<L>() * TX;      // transformed p.E [L][TX]
    C *pre = w4s + L * TX;                    // [4 fields in consumption order][n][TX]
    C *stw = pre + 4 * n * TX;                // [L] forward twiddles (L = 512)
    const int c = threadIdx.x % TX, t = threadIdx.x / TX;
    const long col = (long)blockIdx.x * TX + c;
    const int b = blockIdx.y;
    C *base = W2 + (long)b * 4 * fs + col;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
        const int f = g == 0 ? 3 : g - 1;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            const int z = t + T * q;
            cp_async<sizeof(C)>(&pre[(g * n + z) * TX + c], base + f * fs + (long)z * L2);
        }
        cp_async_commit();
    }
    if constexpr (L == 512) {
        for (int i = threadIdx.x; i < L; i += blockDim.x) stw[i] = tw[i];
        __syncthreads();
    }
    fft16::Tw16<C, L> twr;
    twr.init(t, tw);
    const int eta = (int)(col / L), xi = (int)(col % L);
    const int a1 = xi <= n ? xi : L - xi, a2 = eta <= n ? eta : L - eta;
    auto buf = [&](int pos) -> C & { return xch[xch16(pos, TX, c)]; };
    auto sync = [&]() { __syncthreads(); };
    {
        C w4[16];
        cp_async_wait<3>();
#pragma unroll
        for (int q = 0; q < 8; ++q) w4[q] = pre[(t + T * q) * TX + c];
#pragma unroll
        for (int q = 8; q < 16; ++q) w4[q] = czero<C>();
        fft16::line<-1, L, true>(w4, t, buf, sync, twr, stw);
        // kept in shared memory; each thread reads back only its own positions
#pragma unroll
        for (int q = 0; q < 16; ++q) w4s[(t + T * q) * TX + c] = w4[q];
    }
    cp_async_wait<0>(); // the other three fields (copies of this thread's own elements)
#pragma unroll 1
    for (int d = 0; d < 3; ++d) {
        C v[16];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = pre[((d + 1) * n + t + T * q) * TX + c];
#pragma unroll
        for (int q = 8; q < 16; ++q) v[q] = czero<C>();
        fft16::line<-1, L, true>(v, t, buf, sync, twr, stw);
        const int fr_fixed = d == 0 ? xi : eta;
#pragma unroll
        for (int q = 0; q < 16; ++q) {
            const int zeta = t + T * q;
            const int a3 = zeta <= n ? zeta : L - zeta;
            const long o = ((long)a3 * n1 + a2) * n1 + a1;
            C K0 = spec[o], Kd = spec[(1 + d) * oct + o];
            const int fr = d == 2 ? zeta : fr_fixed;
            if (fr > n) { Kd.x = -Kd.x; Kd.y = -Kd.y; }
            v[q] = cfma(K0, v[q], cmul(Kd, w4s[(t + T * q) * TX + c]));
        }
        fft16::line<1, L, false>(v, t, buf, sync, twr, stw);
#pragma unroll
        for (int q = 0; q < 8; ++q) base[d * fs + (long)(t + T * q) * L2] = v[q];
    }
}

// Fused x and y passes of one z-plane (lengths with 8 values per thread,
// L <= 128): the plane's n x L intermediate stays in shared memory instead of
// going through W1.
//   k2_xyfwd, block (z, f, b): the x-transforms of the plane's n rows of w_f
//     (formed on the fly), kept in S[y][xi]; then the y-transforms of its L
//     columns (n nonzero inputs), written to W2[b][f][z][eta][xi].
//   k2_yxinv, block (z, d, b): the inverse y-transforms of the L columns of
//     W2[b][d][z], rows eta < n kept in S; then the inverse x-transforms of the n
//     rows, x < n kept, plus the identity term: y[b][d][z][y][x].
// 256 threads: LPR = 256 / (L/8) lines per round.  S rows are padded like the
// row passes (xpad), columns go through a separate [L][LPR] exchange buffer.
template <typename R, int L> struct xyf {
    using C = typename cplx_of<R>::type;
    static constexpr int n = L / 2, T = L / 8, LPR = 256 / T, LS = L + L / 8;
    static constexpr size_t smem = sizeof(C) * ((size_t)n * LS + (size_t)L * LPR);
    static_assert(L == 64 || L == 128, "fused plane passes: L = 64 or 128");
    static_assert(n % LPR == 0 && L % LPR == 0, "whole rounds of lines");
};

template <typename R, int L>
__global__ void __launch_bounds__(256) k2_xyfwd(const typename cplx_of<R>::type *__restrict__ x,
                                                const typename cplx_of<R>::type *__restrict__ m,
                                                const typename cplx_of<R>::type *__restrict__ p,
                                                typename cplx_of<R>::type *__restrict__ W2,
                                                const typename cplx_of<R>::type *__restrict__ tw)
{
    pdl_wait_and_trigger();
    using C = typename cplx_of<R>::type;
    constexpr int n = xyf<R, L>::n, T = xyf<R, L>::T, LPR = xyf<R, L>::LPR, LS = xyf<R, L>::LS;
    constexpr long n2 = (long)n * n, n3 = n2 * n, L2 = (long)L * L;
    extern __shared__ unsigned char smem_raw[];
    C *S = reinterpret_cast<C *>(smem_raw); // [n][LS]
    C *X = S + n * LS;                      // [L][LPR]
    const int z = blockIdx.x, f = blockIdx.y, b = blockIdx.z;
    const C *xb = x + (long)b * 3 * n3;
    auto sync = [&]() { __syncthreads(); };
    {   // x-transforms of the rows
        const int line = threadIdx.x / T, t = threadIdx.x % T;
        for (int y0 = 0; y0 < n; y0 += LPR) {
            const int y = y0 + line;
            C v[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const long off = ((long)z * n + y) * n + t + T * q;
                v[q] = f < 3 ? cmul(m[off], xb[f * n3 + off])
                             : cfma(p[off], xb[off], cfma(p[n3 + off], xb[n3 + off], cmul(p[2 * n3 + off], xb[2 * n3 + off])));
                v[q + 4] = czero<C>();
            }
            C *row = S + y * LS; // the row's slot is also its exchange buffer
            auto buf = [&](int pos) -> C & { return row[xpad<L>(pos)]; };
            fftr::fft_line<-1, L, true>(v, t, buf, sync, tw);
#pragma unroll
            for (int q = 0; q < 8; ++q) row[xpad<L>(t + T * q)] = v[q];
        }
        __syncthreads();
    }
    {   // y-transforms of the columns
        const int c = threadIdx.x % LPR, t = threadIdx.x / LPR;
        auto buf = [&](int pos) -> C & { return X[pos * LPR + c]; };
        C *dst = W2 + (((long)b * 4 + f) * n + z) * L2;
        for (int xi0 = 0; xi0 < L; xi0 += LPR) {
            const int xi = xi0 + c;
            C v[8];
#pragma unroll
            for (int q = 0; q < 4; ++q) v[q] = S[(t + T * q) * LS + xpad<L>(xi)];
#pragma unroll
            for (int q = 4; q < 8; ++q) v[q] = czero<C>();
            fftr::fft_line<-1, L, true>(v, t, buf, sync, tw);
#pragma unroll
            for (int q = 0; q < 8; ++q) dst[(long)(t + T * q) * L + xi] = v[q];
        }
    }
}

template <typename R, int L>
__global__ void __launch_bounds__(256) k2_yxinv(const typename cplx_of<R>::type *__restrict__ W2,
                                                const typename cplx_of<R>::type *__restrict__ xin,
                                                typename cplx_of<R>::type *__restrict__ y,
                                                const typename cplx_of<R>::type *__restrict__ tw)
{
    pdl_wait_and_trigger();
    using C = typename cplx_of<R>::type;
    constexpr int n = xyf<R, L>::n, T = xyf<R, L>::T, LPR = xyf<R, L>::LPR, LS = xyf<R, L>::LS;
    constexpr long n2 = (long)n * n, n3 = n2 * n, L2 = (long)L * L;
    extern __shared__ unsigned char smem_raw[];
    C *S = reinterpret_cast<C *>(smem_raw); // [n][LS]
    C *X = S + n * LS;                      // [L][LPR]
    const int z = blockIdx.x, d = blockIdx.y, b = blockIdx.z;
    auto sync = [&]() { __syncthreads(); };
    {   // inverse y-transforms of the columns, eta < n kept
        const int c = threadIdx.x % LPR, t = threadIdx.x / LPR;
        auto buf = [&](int pos) -> C & { return X[pos * LPR + c]; };
        const C *src = W2 + (((long)b * 4 + d) * n + z) * L2;
        for (int xi0 = 0; xi0 < L; xi0 += LPR) {
            const int xi = xi0 + c;
            C v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = src[(long)(t + T * q) * L + xi];
            fftr::fft_line<1, L, false>(v, t, buf, sync, tw);
#pragma unroll
            for (int q = 0; q < 4; ++q) S[(t + T * q) * LS + xpad<L>(xi)] = v[q];
        }
    }
    __syncthreads();
    {   // inverse x-transforms of the rows, x < n kept, + x
        const int line = threadIdx.x / T, t = threadIdx.x % T;
        const C *xb = xin + ((long)b * 3 + d) * n3;
        C *yb = y + ((long)b * 3 + d) * n3;
        for (int y0 = 0; y0 < n; y0 += LPR) {
            const int yy = y0 + line;
            C *row = S + yy * LS;
            C v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = row[xpad<L>(t + T * q)];
            C xi[4];
            const long off = ((long)z * n + yy) * n;
#pragma unroll
            for (int q = 0; q < 4; ++q) xi[q] = xb[off + t + T * q];
            __syncthreads(); // the rows are in registers before they serve as exchange buffers
            auto buf = [&](int pos) -> C & { return row[xpad<L>(pos)]; };
            fftr::fft_line<1, L, false>(v, t, buf, sync, tw);
#pragma unroll
            for (int q = 0; q < 4; ++q) yb[off + t + T * q] = xi[q] + v[q];
        }
    }
}

// xinv: rows of V1 (length L) -> y = x + IFFT(row)[x < n]
template <typename R, int L>
__global__ void __launch_bounds__(256) k2_xinv(const typename cplx_of<R>::type *__restrict__ V1,
                                               const typename cplx_of<R>::type *__restrict__ xin,
                                               typename cplx_of<R>::type *__restrict__ y, long nrows,
                                               const typename cplx_of<R>::type *__restrict__ tw)
{
    pdl_wait_and_trigger();
    using C = typename cplx_of<R>::type;
    constexpr int E = line_elems(L), H = E / 2;
    constexpr int T = L / E, n = L / 2, LS = L + L / 8;
    extern __shared__ unsigned char smem_raw[];
    C *sm = reinterpret_cast<C *>(smem_raw);
    const int line = threadIdx.x / T, t = threadIdx.x % T;
    const long g = (long)blockIdx.x * (blockDim.x / T) + line;
    const bool ok = g < nrows;
    C v[E];
#pragma unroll
    for (int q = 0; q < E; ++q) v[q] = ok ? V1[g * L + t + T * q] : czero<C>();
    C *lb = sm + line * LS;
    auto buf = [&](int pos) -> C & { return lb[xpad<L>(pos)]; };
    auto sync = [&]() { if (T <= 32) __syncwarp(); else __syncthreads(); };
    C xi[H]; // the identity term, loaded before the transform so its latency overlaps it
#pragma unroll
    for (int q = 0; q < H; ++q) xi[q] = ok ? xin[g * n + t + T * q] : czero<C>();
    line_fft<1, L, false>(v, t, buf, sync, tw);
    if (ok) {
#pragma unroll
        for (int q = 0; q < H; ++q) y[g * n + t + T * q] = xi[q] + v[q];
    }
}


// Half of the L1 for shared memory unless a pass needs more: without a request a pass runs
// with what the one before it wanted (A complex64, asked for 50 / 75 / 100 %: n = 32 13.2,
// 13.1, 12.6 us against 14.9; n = 128 438, 460, 514 against 463; n = 256 4077, 4278, 4953
// against 4114; n = 64 54.2, 56.1, 57.8 against 54.2).  In complex128 the request costs
// (n = 96 3643 us against 3472, n = 16 50 against 47), so there is none.
template <typename R, typename K> void allow_smem(K kernel, size_t bytes)
{
    if (sizeof(R) == 4) cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 50);
    if (bytes > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// ---------------------------------------------------------------- TMA z-pass
// mbarrier and bulk-tensor copy primitives (PTX ISA, sm_90 and later)
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_fence_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
// bounded wait for phase `parity`: about 2^22 polls (each may suspend briefly)
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, unsigned parity)
{
    const unsigned a = smem_u32(bar);
    for (int it = 0; it < (1 << 22); ++it) {
        unsigned done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done)
                     : "r"(a), "r"(parity)
                     : "memory");
        if (done) return true;
    }
    return false;
}
__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, int x, int y, int z, uint64_t *bar)
{
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];\n" ::"r"(
                     smem_u32(dst)),
                 "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
                 : "memory");
}

// Self-test of the bounded wait: an mbarrier expecting 16 bytes that no copy
// delivers; every thread waits with the same bound as the TMA z-pass, and the
// expired wait is recorded in *err (code 2) exactly as the z-pass records one.
__global__ void k_wait_selftest(int *err)
{
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        mbar_fence_init();
        mbar_expect_tx(&bar, 16);
    }
    __syncthreads();
    const bool ok = mbar_wait(&bar, 0);
    if (__syncthreads_or(!ok) && threadIdx.x == 0) atomicExch(err, 2);
}

// zpass fed by TMA: a persistent grid walks the tiles (TX adjacent columns of
// one right-hand side); while a tile is transformed, the next tile's four
// fields (n z-values x TX columns each, the pruned half) stream into the other
// of two shared-memory stages through cp.async.bulk.tensor, completion counted
// on that stage's mbarrier.  Per tile: forward z-transform of p.E, then per d
// forward transform, Fourier-side product, inverse transform, z < n stored in
// place (fields 0..2), as in the other z-pass kernels.  Tensor map: W2 viewed as
// [nb 4 n][L][L x (complex size / 8)] 8-byte words, box {TX words, 1, n}.
template <typename R, int L>
__global__ void __launch_bounds__(tx_of<R, L>::v * L / line_elems(L)) k2_ztma(const __grid_constant__ CUtensorMap tmap,
                                                                            typename cplx_of<R>::type *W2,
                                                                            const typename cplx_of<R>::type *__restrict__ spec,
                                                                            const typename cplx_of<R>::type *__restrict__ tw,
                                                                            int ntiles, int tiles_per_rhs, int *err)
{
    using C = typename cplx_of<R>::type;
    constexpr int E = line_elems(L), H = E / 2;
    constexpr int T = L / E, TX = tx_of<R, L>::v, n = L / 2, n1 = n + 1;
    constexpr long L2 = (long)L * L, oct = (long)n1 * n1 * n1, fs = (long)n * L * L;
    constexpr int STAGE = 4 * n * TX;
    constexpr unsigned STAGE_BYTES = STAGE * sizeof(C);
    constexpr int WPC = sizeof(C) / 8; // 8-byte words per complex
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    C *stages = reinterpret_cast<C *>(smem_raw);
    C *xch = stages + 2 * STAGE; // exchange buffer [L][TX]
    uint64_t *bar = reinterpret_cast<uint64_t *>(xch + L * TX);
    const int c = threadIdx.x % TX, t = threadIdx.x / TX;
    auto issue = [&](int tile, int st) { // thread 0
        const int b = tile / tiles_per_rhs;
        const long col0 = (long)(tile % tiles_per_rhs) * TX;
        const int eta = (int)(col0 / L), xi0 = (int)(col0 % L);
        mbar_expect_tx(&bar[st], STAGE_BYTES);
#pragma unroll
        for (int g = 0; g < 4; ++g) {
            const int f = g == 0 ? 3 : g - 1; // consumption order: p.E first
            tma_load_3d(stages + st * STAGE + g * n * TX, &tmap, xi0 * WPC, eta, (b * 4 + f) * n, &bar[st]);
        }
    };
    if (threadIdx.x == 0) {
        mbar_init(&bar[0], 1);
        mbar_init(&bar[1], 1);
        mbar_fence_init();
    }
    __syncthreads();
    pdl_wait_and_trigger();
    if (threadIdx.x == 0) {
        if ((int)blockIdx.x < ntiles) issue(blockIdx.x, 0);
        if ((int)(blockIdx.x + gridDim.x) < ntiles) issue(blockIdx.x + gridDim.x, 1);
    }
    auto buf = [&](int pos) -> C & { return xch[pos * TX + c]; };
    auto sync = [&]() { __syncthreads(); };
    int it = 0;
    bool failed = false;
    for (int tile = blockIdx.x; tile < ntiles; tile += gridDim.x, ++it) {
        const int st = it & 1;
        const bool ok = mbar_wait(&bar[st], (it >> 1) & 1);
        if (__syncthreads_or(!ok)) { failed = true; break; } // every thread leaves together
        const C *pre = stages + st * STAGE; // [g][z][TX]
        const int b = tile / tiles_per_rhs;
        const long col = (long)(tile % tiles_per_rhs) * TX + c;
        C *base = W2 + (long)b * 4 * fs + col;
        const int eta = (int)(col / L), xi = (int)(col % L);
        const int a1 = xi <= n ? xi : L - xi, a2 = eta <= n ? eta : L - eta;
        C w4[E];
#pragma unroll
        for (int q = 0; q < H; ++q) w4[q] = pre[(t + T * q) * TX + c];
#pragma unroll
        for (int q = H; q < E; ++q) w4[q] = czero<C>();
        line_fft<-1, L, true>(w4, t, buf, sync, tw);
#pragma unroll 1
        for (int d = 0; d < 3; ++d) {
            C v[E];
#pragma unroll
            for (int q = 0; q < H; ++q) v[q] = pre[((d + 1) * n + t + T * q) * TX + c];
#pragma unroll
            for (int q = H; q < E; ++q) v[q] = czero<C>();
            line_fft<-1, L, true>(v, t, buf, sync, tw);
            const int fr_fixed = d == 0 ? xi : eta;
#pragma unroll
            for (int q = 0; q < E; ++q) {
                const int zeta = t + T * q;
                const int a3 = zeta <= n ? zeta : L - zeta;
                const long o = ((long)a3 * n1 + a2) * n1 + a1;
                C K0 = spec[o], Kd = spec[(1 + d) * oct + o];
                const int fr = d == 2 ? zeta : fr_fixed;
                if (fr > n) { Kd.x = -Kd.x; Kd.y = -Kd.y; }
                v[q] = cfma(K0, v[q], cmul(Kd, w4[q]));
            }
            line_fft<1, L, false>(v, t, buf, sync, tw);
#pragma unroll
            for (int q = 0; q < H; ++q) base[d * fs + (long)(t + T * q) * L2] = v[q];
        }
        __syncthreads(); // stage st and the exchange buffer are free again
        if (threadIdx.x == 0 && tile + 2 * (int)gridDim.x < ntiles) issue(tile + 2 * gridDim.x, st);
    }
    if (failed && threadIdx.x == 0) {
        // Both stages may still have copies in flight: the one whose wait expired
        // and the next one.  Wait for each (bounded) before the block leaves, so
        // that no bulk copy writes into shared memory after the exit.  Code 1: the
        // wait expired and both copies then landed; code 3: a copy was still
        // outstanding after the second bounded wait (the exit is then best effort).
        bool drained = mbar_wait(&bar[it & 1], (it >> 1) & 1);
        const int nxt = it + 1;
        if ((int)(blockIdx.x + (unsigned)nxt * gridDim.x) < ntiles) drained = mbar_wait(&bar[nxt & 1], (nxt >> 1) & 1) && drained;
        atomicExch(err, drained ? 1 : 3);
    }
}


// tensor-map encoder from the driver, fetched once through the runtime
typedef CUresult (*encode_tiled_fn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                    const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
encode_tiled_fn tensor_map_encoder()
{
    static encode_tiled_fn fn = nullptr;
    static std::once_flag once;
    std::call_once(once, []() {
        void *p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
            q == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<encode_tiled_fn>(p);
    });
    return fn;
}

template <typename R, int L> constexpr size_t ztma_smem()
{
    using C = typename cplx_of<R>::type;
    constexpr int TX = tx_of<R, L>::v, n = L / 2;
    return sizeof(C) * (2 * 4 * n * TX + L * TX) + 2 * sizeof(uint64_t);
}

template <typename R, int L>
spm_status launch_ztma(typename cplx_of<R>::type *W2, const typename cplx_of<R>::type *spec,
                       const typename cplx_of<R>::type *tw, int nb, int *err, cudaStream_t s)
{
    using C = typename cplx_of<R>::type;
    constexpr int TX = tx_of<R, L>::v, n = L / 2, THR = TX * L / line_elems(L);
    constexpr int WPC = sizeof(C) / 8;
    encode_tiled_fn enc = tensor_map_encoder();
    if (!enc) { spm_set_error("cuTensorMapEncodeTiled is not available"); return SPM_ERR_CUDA; }
    CUtensorMap map;
    const cuuint64_t dims[3] = {(cuuint64_t)L * WPC, (cuuint64_t)L, (cuuint64_t)nb * 4 * n};
    const cuuint64_t strides[2] = {(cuuint64_t)L * sizeof(C), (cuuint64_t)L * L * sizeof(C)};
    const cuuint32_t box[3] = {(cuuint32_t)(TX * WPC), 1u, (cuuint32_t)n};
    const cuuint32_t estr[3] = {1u, 1u, 1u};
    if (enc(&map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 3, W2, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS) {
        spm_set_error("tensor map for the z-pass rejected (L = %d)", L);
        return SPM_ERR_CUDA;
    }
    constexpr size_t smem = ztma_smem<R, L>();
    static int grid_per_sm = 0;
    static int sms = 0;
    if (!grid_per_sm) {
        allow_smem<R>(k2_ztma<R, L>, smem);
        int dev = 0;
        SPM_CUDA_TRY(cudaGetDevice(&dev));
        SPM_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        int per = 0;
        SPM_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k2_ztma<R, L>, THR, smem));
        grid_per_sm = per > 0 ? per : 1;
    }
    const int tiles_per_rhs = L * L / TX, ntiles = tiles_per_rhs * nb;
    const int grid = std::min(ntiles, grid_per_sm * sms);
    launch_pdl(k2_ztma<R, L>, dim3(grid), dim3(THR), smem, s, map, W2, spec, tw, ntiles, tiles_per_rhs, err);
    return SPM_OK;
}


// ev (may be NULL): events recorded after each pass on s, so that the caller can
// time every pass of one apply (spm_profile_apply); *nev counts them.
template <typename R, int L>
spm_status apply_chunk_v2(const typename cplx_of<R>::type *xb, typename cplx_of<R>::type *yb,
                    const typename cplx_of<R>::type *m, const typename cplx_of<R>::type *p,
                    const typename cplx_of<R>::type *spec, const typename cplx_of<R>::type *tw,
                    typename cplx_of<R>::type *W1, typename cplx_of<R>::type *W2, int nb, int zvar, int *err,
                    cudaStream_t s, cudaEvent_t *ev = nullptr, int *nev = nullptr)
{
    auto mark = [&]() {
        if (ev) cudaEventRecord(ev[(*nev)++], s);
    };
    using C = typename cplx_of<R>::type;
    constexpr int n = L / 2, T = L / line_elems(L), TX = tx_of<R, L>::v;
    constexpr int LPB = 256 / T > 0 ? 256 / T : 1;
    constexpr size_t sm_rows = sizeof(C) * LPB * (L + L / 8), sm_cols = sizeof(C) * L * TX;
    constexpr bool APART = (long)n * n * T < 32 * 4 * 152; // one field's rows may be that few
    // rows per block: 256 threads, fewer (down to a warp) while that leaves under two
    // blocks for each of 152 SMs: x-forward at n = 16 in complex128 was 4 blocks and
    // 40 us, with 32 it takes 21
    auto launch_rows = [&](auto kernel, long rows, int fields, auto... args) {
        int lines = LPB;
        while (lines % 2 == 0 && lines * T >= 64 && (rows + lines - 1) / lines < 2 * 152) lines /= 2;
        launch_pdl(kernel, dim3((unsigned)((rows + lines - 1) / lines), fields), dim3(lines * T), sizeof(C) * lines * (L + L / 8), s,
                   args...);
    };
    const bool fused = (zvar & ZPLAN_FUSED_XY) != 0; // x and y passes fused per z-plane
    zvar &= ZPLAN_FUSED_XY - 1;
    constexpr size_t sm_zprod = sm_cols + sizeof(C) * 4 * n * TX;
    constexpr size_t sm_zprod4 = 4 * sm_cols;
    static bool attrs = false;
    if (!attrs) {
        if constexpr (APART) allow_smem<R>(k2_xfwd<R, L, true>, sm_rows);
        allow_smem<R>(k2_xfwd<R, L, false>, sm_rows);
        allow_smem<R>(k2_xinv<R, L>, sm_rows);
        allow_smem<R>(k2_cols<R, L, -1, true>, sm_cols);
        allow_smem<R>(k2_cols<R, L, 1, false>, sm_cols);
        if constexpr (line_elems(L) == 8) {
            allow_smem<R>(k2_cols2<R, L, -1, true>, 2 * sm_cols);
            allow_smem<R>(k2_cols2<R, L, 1, false>, 2 * sm_cols);
        }
        if constexpr (line_elems(L) == 8 && !zfield_serves<R, L>()) allow_smem<R>(k2_zprod4<R, L>, sm_zprod4);
        allow_smem<R>(k2_zprod1<R, L>, sm_zprod);
        attrs = true;
    }
    const long n2 = (long)n * n, L2 = (long)L * L;
    const int THR = TX * T; // threads of a strided-pass block
    bool fused_done = false;
    if constexpr (L == 64 || L == 128) {
        if (fused) {
            static bool axy = false;
            if (!axy) {
                allow_smem<R>(k2_xyfwd<R, L>, xyf<R, L>::smem);
                allow_smem<R>(k2_yxinv<R, L>, xyf<R, L>::smem);
                axy = true;
            }
            launch_pdl(k2_xyfwd<R, L>, dim3(n, 4, nb), dim3(256), xyf<R, L>::smem, s, xb, m, p, W2, tw);
            mark();
            fused_done = true;
        }
    }
    if (!fused_done) {
        long rows = (long)nb * n2;
        // too few rows for a warp on every scheduler (4 x 152): the fields apart (n = 16 in
        // complex128: 20 us one after another)
        bool apart = false;
        if constexpr (APART) {
            apart = rows * T < 32 * 4 * 152;
            if (apart) launch_rows(k2_xfwd<R, L, true>, rows, 4, xb, m, p, W1, (int)rows, tw);
        }
        if (!apart) launch_rows(k2_xfwd<R, L, false>, rows, 1, xb, m, p, W1, (int)rows, tw);
        mark();
        if constexpr (line_elems(L) == 8 && n % 2 == 0)
            launch_pdl(k2_cols2<R, L, -1, true>, dim3(L / TX, n / 2, nb * 4), dim3(THR), 2 * sm_cols, s, (const C *)W1,
                       W2, L, (long)L, 4, 4 * n2 * L, n2 * L, n * (long)L, 4 * (long)n * L2, (long)n * L2, L2, tw);
        else
            launch_pdl(k2_cols<R, L, -1, true>, dim3(L / TX, n, nb * 4), dim3(THR), sm_cols, s, (const C *)W1, W2, L,
                       (long)L, 4, 4 * n2 * L, n2 * L, n * (long)L, 4 * (long)n * L2, (long)n * L2, L2, tw);
        mark();
    }
    bool done = false;
    if constexpr (L >= 32) {
        if (zvar == ZPROD_TMA) {
            SPM_TRY((launch_ztma<R, L>(W2, spec, tw, nb, err, s)));
            done = true;
        }
    }
    if constexpr (L == 128 || L == 256 || L == 512) {
        if (zvar == ZPROD_E16) {
            constexpr size_t sm16 = zp16<R, L>::smem();
            static bool a16 = false;
            if (!a16) {
                allow_smem<R>(k3_zpass<R, L>, sm16);
                a16 = true;
            }
            launch_pdl(k3_zpass<R, L>, dim3((unsigned)(L2 / zp16<R, L>::TX), nb), dim3(zp16<R, L>::THREADS), sm16, s,
                       W2, spec, tw);
            done = true;
        }
    }
    if constexpr (L >= 32) {
        if (!done && zvar == ZPROD_STAGED) {
            constexpr size_t smz = zst<R, L>::smem;
            static bool ast = false;
            if (!ast) {
                allow_smem<R>(k2_zstaged<R, L>, smz);
                ast = true;
            }
            launch_pdl(k2_zstaged<R, L>, dim3((unsigned)(L2 / TX), nb), dim3(zst<R, L>::THREADS), smz, s, W2, spec, tw);
            done = true;
        }
    }
    if constexpr (L == 64 || L == 128 || L == 256) {
        if (!done && zvar == ZPROD_SPLIT) {
            static bool asp = false;
            if (!asp) {
                allow_smem<R>(k2_zsplit<R, L>, zsp<R, L>::smem);
                asp = true;
            }
            launch_pdl(k2_zsplit<R, L>, dim3((unsigned)(L2 / zsp<R, L>::TX), nb), dim3(256), zsp<R, L>::smem, s, W2,
                       spec, tw);
            done = true;
        }
    }
    if constexpr (line_elems(L) == 8) {
        if (!done && zvar == ZPROD_FOUR) {
            if constexpr (zfield_serves<R, L>())
                launch_pdl(k2_zfield<R, L>, dim3((unsigned)(L2 / zfl<R, L>::TX), nb), dim3(zfl<R, L>::THREADS), zfl<R, L>::smem,
                           s, W2, spec, tw);
            else
                launch_pdl(k2_zprod4<R, L>, dim3((unsigned)(L2 / TX), nb), dim3(THR), sm_zprod4, s, W2, spec, tw);
            done = true;
        }
    }
    if (!done) launch_pdl(k2_zprod1<R, L>, dim3((unsigned)(L2 / TX), nb), dim3(THR), sm_zprod, s, W2, spec, tw);
    mark();
    if (fused_done) {
        if constexpr (L == 64 || L == 128)
            launch_pdl(k2_yxinv<R, L>, dim3(n, 3, nb), dim3(256), xyf<R, L>::smem, s, (const C *)W2, xb, yb, tw);
        mark();
        return SPM_OK;
    }
    if constexpr (line_elems(L) == 8 && n % 2 == 0)
        launch_pdl(k2_cols2<R, L, 1, false>, dim3(L / TX, n / 2, nb * 3), dim3(THR), 2 * sm_cols, s, (const C *)W2, W1,
                   n, (long)L, 3, 4 * (long)n * L2, (long)n * L2, L2, 3 * n2 * L, n2 * L, n * (long)L, tw);
    else
        launch_pdl(k2_cols<R, L, 1, false>, dim3(L / TX, n, nb * 3), dim3(THR), sm_cols, s, (const C *)W2, W1, n,
                   (long)L, 3, 4 * (long)n * L2, (long)n * L2, L2, 3 * n2 * L, n2 * L, n * (long)L, tw);
    mark();
    {
        long rows = (long)nb * 3 * n2;
        launch_rows(k2_xinv<R, L>, rows, 1, (const C *)W1, xb, yb, rows, tw);
    }
    mark();
    return SPM_OK;
}

template <typename R>
spm_status run_chunk(int L, const typename cplx_of<R>::type *xb, typename cplx_of<R>::type *yb,
                     const typename cplx_of<R>::type *m, const typename cplx_of<R>::type *p,
                     const typename cplx_of<R>::type *spec, const typename cplx_of<R>::type *tw,
                     typename cplx_of<R>::type *W1, typename cplx_of<R>::type *W2, int nb, int zvar, int *err,
                     cudaStream_t s, cudaEvent_t *ev = nullptr, int *nev = nullptr)
{
    switch (L) {
    case 8: return apply_chunk_v2<R, 8>(xb, yb, m, p, spec, tw, W1, W2, nb, zvar, err, s, ev, nev);
    case 16: return apply_chunk_v2<R, 16>(xb, yb, m, p, spec, tw, W1, W2, nb, zvar, err, s, ev, nev);
    case 32: return apply_chunk_v2<R, 32>(xb, yb, m, p, spec, tw, W1, W2, nb, zvar, err, s, ev, nev);
    case 64: return apply_chunk_v2<R, 64>(xb, yb, m, p, spec, tw, W1, W2, nb, zvar, err, s, ev, nev);
    case 128: return apply_chunk_v2<R, 128>(xb, yb, m, p, spec, tw, W1, W2, nb, zvar, err, s, ev, nev);
    case 256: return apply_chunk_v2<R, 256>(xb, yb, m, p, spec, tw, W1, W2, nb, zvar, err, s, ev, nev);
    case 512: return apply_chunk_v2<R, 512>(xb, yb, m, p, spec, tw, W1, W2, nb, zvar, err, s, ev, nev);
    case 96: return apply_chunk_v2<R, 96>(xb, yb, m, p, spec, tw, W1, W2, nb, zvar, err, s, ev, nev);
    case 192: return apply_chunk_v2<R, 192>(xb, yb, m, p, spec, tw, W1, W2, nb, zvar, err, s, ev, nev);
    default: spm_set_error("unsupported FFT length %d", L); return SPM_ERR_INVALID_ARG;
    }
}

// Apply plan.  The z-pass kernel is the choice with more than one candidate:
// the four-line kernel (all fields in registers, shared barriers; lengths with
// 8 elements per thread), the one-field-at-a-time kernel (all four fields
// prefetched into shared memory by cp.async, then transformed one after
// another), and the persistent TMA-fed kernel (double-buffered stages, L >= 32).  The first apply of each (length, precision) in the process
// times both candidates on the caller's own data and keeps the faster for every
// later apply; during stream capture the default kernel is used untimed.
std::atomic<int> g_zplan[2][10];
std::atomic<int> g_zplan_init(0);
// per-apply ms of each candidate when the plan timed them (0: not timed)
float g_ztime[2][10][6];
float g_ztime_fused[2][10]; // the chosen z-pass with fused x and y passes (0: not timed)
std::mutex g_ztime_mu;

int len_index(int L)
{
    switch (L) {
    case 8: return 0; case 16: return 1; case 32: return 2; case 64: return 3; case 128: return 4;
    case 256: return 5; case 512: return 6; case 96: return 7; case 192: return 8; default: return 9;
    }
}

int zplan_get(int prec_idx, int L)
{
    int expected = 0;
    if (g_zplan_init.compare_exchange_strong(expected, 1)) {
        for (auto &row : g_zplan)
            for (auto &e : row) e.store(-1);
        g_zplan_init.store(2);
    }
    while (g_zplan_init.load() != 2) {}
    return g_zplan[prec_idx][len_index(L)].load();
}

template <typename R>
spm_status choose_zplan(int L, const typename cplx_of<R>::type *xb, typename cplx_of<R>::type *yb,
                        const typename cplx_of<R>::type *m, const typename cplx_of<R>::type *p,
                        const typename cplx_of<R>::type *spec, const typename cplx_of<R>::type *tw,
                        typename cplx_of<R>::type *W1, typename cplx_of<R>::type *W2, int nb, int *err, cudaStream_t s,
                        int *zvar)
{
    const int pi = sizeof(R) == 8 ? 0 : 1;
    int z = zplan_get(pi, L);
    if (z >= 0) { *zvar = z; return SPM_OK; }
    const int fallback = line_elems(L) == 8 ? ZPROD_FOUR : ZPROD_ONE;
    int cands[6], nc = 0;
    if (line_elems(L) == 8) cands[nc++] = ZPROD_FOUR;
    if (line_elems(L) != 8 || L >= 32) cands[nc++] = ZPROD_ONE;
    if (L >= 32) cands[nc++] = ZPROD_TMA;
    if (L == 128 || L == 256 || L == 512) cands[nc++] = ZPROD_E16;
    if (L >= 32) cands[nc++] = ZPROD_STAGED;
    if (L == 64 || L == 128 || L == 256) cands[nc++] = ZPROD_SPLIT;
    if (nc == 1) { g_zplan[pi][len_index(L)].store(cands[0]); *zvar = cands[0]; return SPM_OK; }
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    SPM_CUDA_TRY(cudaStreamIsCapturing(s, &cap));
    if (cap != cudaStreamCaptureStatusNone) { *zvar = fallback; return SPM_OK; }
    cudaEvent_t e0, e1;
    SPM_CUDA_TRY(cudaEventCreate(&e0));
    SPM_CUDA_TRY(cudaEventCreate(&e1));
    float best = 0;
    int best_z = fallback;
    spm_status st = SPM_OK;
    const int reps = L >= 512 ? 3 : (L >= 256 ? 5 : 10);
    float times[6] = {0, 0, 0, 0, 0, 0};
    for (int ci = 0; ci < nc; ++ci) {
        const int cand = cands[ci];
        st = run_chunk<R>(L, xb, yb, m, p, spec, tw, W1, W2, nb, cand, err, s); // warm-up
        if (st != SPM_OK) break;
        cudaEventRecord(e0, s);
        for (int r = 0; r < reps && st == SPM_OK; ++r) st = run_chunk<R>(L, xb, yb, m, p, spec, tw, W1, W2, nb, cand, err, s);
        cudaEventRecord(e1, s);
        if (st != SPM_OK || cudaEventSynchronize(e1) != cudaSuccess) { st = st != SPM_OK ? st : SPM_ERR_CUDA; break; }
        float ms = 0;
        cudaEventElapsedTime(&ms, e0, e1);
        times[cand] = ms / reps;
        if (ci == 0 || ms < best) { best = ms; best_z = cand; }
    }
    float fused_ms = 0;
    if (st == SPM_OK && (L == 64 || L == 128)) {
        // the best z-pass again with the x and y passes fused per plane
        const int cand = best_z | ZPLAN_FUSED_XY;
        st = run_chunk<R>(L, xb, yb, m, p, spec, tw, W1, W2, nb, cand, err, s);
        if (st == SPM_OK) {
            cudaEventRecord(e0, s);
            for (int r = 0; r < reps && st == SPM_OK; ++r) st = run_chunk<R>(L, xb, yb, m, p, spec, tw, W1, W2, nb, cand, err, s);
            cudaEventRecord(e1, s);
            if (st == SPM_OK && cudaEventSynchronize(e1) == cudaSuccess) {
                float ms = 0;
                cudaEventElapsedTime(&ms, e0, e1);
                fused_ms = ms / reps;
                if (ms < best) { best = ms; best_z = cand; }
            } else if (st == SPM_OK) {
                st = SPM_ERR_CUDA;
            }
        }
    }
    if (st == SPM_OK) {
        std::lock_guard<std::mutex> lock(g_ztime_mu);
        for (int v = 0; v < 6; ++v) g_ztime[pi][len_index(L)][v] = times[v];
        g_ztime_fused[pi][len_index(L)] = fused_ms;
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (st != SPM_OK) {
        if (st == SPM_ERR_CUDA) spm_set_error("timing the z-pass candidates failed: %s", cudaGetErrorString(cudaGetLastError()));
        return st;
    }
    g_zplan[pi][len_index(L)].store(best_z);
    *zvar = best_z;
    return SPM_OK;
}

template <typename R>
spm_status apply_A_typed(spm_problem_s *P, const void *xv, void *yv, int nrhs, cudaStream_t s)
{
    using C = typename cplx_of<R>::type;
    const int n = P->n, L = P->L;
    const long n2 = (long)n * n, n3 = n2 * n, L2 = (long)L * L;
    const C *x = reinterpret_cast<const C *>(xv);
    C *y = reinterpret_cast<C *>(yv);
    const bool dbl = sizeof(R) == 8;
    const C *m = dbl ? P->m128.as<C>() : P->m64.as<C>();
    const C *p = dbl ? P->p128.as<C>() : P->p64.as<C>();
    const C *spec = dbl ? P->spec128.as<C>() : P->spec64.as<C>();
    const C *tw = dbl ? P->tw128.as<C>() : P->tw64.as<C>();
    const int chunk = dbl ? P->chunk128 : P->chunk64;
    const long w1 = 4 * n2 * L, w2 = 4 * (long)n * L2; // per RHS, complex elements
    SPM_TRY(P->work.ensure(sizeof(C) * (size_t)chunk * (w1 + w2)));
    C *W1 = P->work.as<C>();
    C *W2 = W1 + (long)chunk * w1;
    int zvar = ZPROD_FOUR;
    SPM_TRY(choose_zplan<R>(L, x, y, m, p, spec, tw, W1, W2, nrhs < chunk ? nrhs : chunk, P->dev_err.as<int>(), s, &zvar));
    for (int b0 = 0; b0 < nrhs; b0 += chunk) {
        const int nb = nrhs - b0 < chunk ? nrhs - b0 : chunk;
        SPM_TRY(run_chunk<R>(L, x + (long)b0 * 3 * n3, y + (long)b0 * 3 * n3, m, p, spec, tw, W1, W2, nb, zvar, P->dev_err.as<int>(), s));
    }
    SPM_CUDA_TRY(cudaGetLastError());
    return SPM_OK;
}

// Q gather in complex64, one launch of 128-thread blocks of three kinds (block-uniform
// branch), boundary blocks first so that their latency overlaps the interior:
// * face blocks: the points with exactly one coordinate on the boundary belong
//   to one of six face classes; a block owns a 32 x 4 tile of one face, stages
//   the face layer and the next layer inward (three components, one-point halo)
//   and its class's 18-neighbour coefficients (remapped to face-local order) in
//   shared memory, and each thread forms its point's three outputs;
// * edge blocks: the 12 (n-2) + 8 points on edges and corners, one warp per
//   point; lane l takes the terms (d, o) with d * 27 + o in {l, l + 32, l + 64}
//   (of 81) from the expanded table [cls][d][o][c] (zero outside the class
//   neighbourhood, which is also where a neighbour would leave the grid) and
//   the warp sums its partials;
// * interior blocks (1 <= i_d <= n-2, one class): a 32 x 4 x QZ tile whose three
//   components plus a one-point halo are staged in shared memory; each thread
//   owns QZ = 4 points stacked along z, so every staged value it loads feeds the
//   three z-offsets of up to three of its points (6 loads per (d, o1, o2) serve
//   36 complex MACs per output component instead of one load per MAC); the
//   class's 243 coefficients arrive as a by-value kernel parameter, so they sit
//   in the constant bank, and each feeds QZ points once in registers.
constexpr int Q_THREADS = 128;
constexpr int QX = 32, QY = 4, QZ = 4;
constexpr int QHX = QX + 2, QHY = QY + 2, QHZ = QZ + 2, QH = QHX * QHY * QHZ;
constexpr int QF_U = 32, QF_W = 4;
constexpr int QF_HU = QF_U + 2, QF_HW = QF_W + 2, QF_HALO = 3 * 2 * QF_HW * QF_HU;
constexpr int Q_SMEM = (3 * QH > QF_HALO + 162) ? 3 * QH : QF_HALO + 162; // complex elements
static_assert(QX * QY == Q_THREADS && QF_U * QF_W == Q_THREADS, "Q block shapes");

// interior coefficients [d][o][c], o = (o3+1)*9 + (o2+1)*3 + (o1+1): each coefficient a
// as the packed pairs (a.x, a.x, -a.y, a.y), so a complex MAC acc += a v is two packed
// FP32x2 FMAs, (a.x, a.x) (v.x, v.y) and (-a.y, a.y) (v.y, v.x)
struct QInterior {
    float4 a[243];
};
static_assert(sizeof(QInterior) + 64 <= 4096, "kernel parameter space");

// edge point number e (0 <= e < 12 (n-2) + 8) -> (i1, i2, i3): corners, then the
// edges along x, y, z (four each)
__device__ __forceinline__ void edge_point(int e, int n, int &i1, int &i2, int &i3)
{
    if (e < 8) {
        i1 = (e & 1) ? n - 1 : 0;
        i2 = (e & 2) ? n - 1 : 0;
        i3 = (e & 4) ? n - 1 : 0;
        return;
    }
    const int r = e - 8, k = r / (n - 2), t = 1 + r % (n - 2);
    const int a = k >> 2, b0 = (k & 1) ? n - 1 : 0, b1 = (k & 2) ? n - 1 : 0;
    if (a == 0) { i1 = t; i2 = b0; i3 = b1; }
    else if (a == 1) { i1 = b0; i2 = t; i3 = b1; }
    else { i1 = b0; i2 = b1; i3 = t; }
}

__device__ __forceinline__ void q_interior_block(int blk, const float2 *__restrict__ vb, const QInterior &qa,
                                                 float2 *__restrict__ yb, int n, float2 *sv)
{
    const long n3 = (long)n * n * n;
    const int m = n - 2; // interior extent
    const int tiles_x = (m + QX - 1) / QX, tiles_y = (m + QY - 1) / QY;
    const int txy = blk % (tiles_x * tiles_y), tz = blk / (tiles_x * tiles_y);
    const int tx0 = 1 + (txy % tiles_x) * QX, ty0 = 1 + (txy / tiles_x) * QY, tz0 = 1 + tz * QZ;
    // halo [d][hz][hy][hx], x fastest: each warp's loads below read 32 consecutive x.
    // All copies are issued before any is waited for (cp.async, zero fill outside
    // the grid), so their latencies overlap.
    for (int i = threadIdx.x; i < 3 * QH; i += Q_THREADS) {
        int d = i / QH, h = i % QH;
        int hx = h % QHX, hy = (h / QHX) % QHY, hz = h / (QHX * QHY);
        int gx = tx0 + hx - 1, gy = ty0 + hy - 1, gz = tz0 + hz - 1;
        const bool in = gx < n && gy < n && gz < n;
        cp_async_zfill<sizeof(float2)>(&sv[i], in ? vb + d * n3 + ((long)gz * n + gy) * n + gx : vb, in);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    const int lx = threadIdx.x % QX, ly = threadIdx.x / QX;
    const int i1 = tx0 + lx, i2 = ty0 + ly;
    if (i1 > n - 2 || i2 > n - 2) return;
    float2 acc[QZ][3];
#pragma unroll
    for (int q = 0; q < QZ; ++q) acc[q][0] = acc[q][1] = acc[q][2] = czero<float2>();
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int o2 = -1; o2 <= 1; ++o2)
#pragma unroll
            for (int o1 = -1; o1 <= 1; ++o1) {
                // the z-column (d, i2 + o2, i1 + o1) over the tile's QZ + 2 halo planes
                float2 col[QZ + 2];
#pragma unroll
                for (int j = 0; j < QZ + 2; ++j) col[j] = sv[d * QH + (j * QHY + ly + 1 + o2) * QHX + lx + 1 + o1];
                float2 cs[QZ + 2]; // (im, re) of each value, for the second packed FMA
#pragma unroll
                for (int j = 0; j < QZ + 2; ++j) cs[j] = make_float2(col[j].y, col[j].x);
#pragma unroll
                for (int o3 = -1; o3 <= 1; ++o3) {
                    const int o = (o3 + 1) * 9 + (o2 + 1) * 3 + (o1 + 1);
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        const float4 a = qa.a[(d * 27 + o) * 3 + c];
                        const float2 ar = make_float2(a.x, a.y), ai = make_float2(a.z, a.w);
#pragma unroll
                        for (int q = 0; q < QZ; ++q)
                            acc[q][c] = __ffma2_rn(ai, cs[q + o3 + 1], __ffma2_rn(ar, col[q + o3 + 1], acc[q][c]));
                    }
                }
            }
#pragma unroll
    for (int q = 0; q < QZ; ++q) {
        const int i3 = tz0 + q;
        if (i3 > n - 2) break;
        const long i = ((long)i3 * n + i2) * n + i1;
        yb[i] = acc[q][0];
        yb[n3 + i] = acc[q][1];
        yb[2 * n3 + i] = acc[q][2];
    }
}

__device__ __forceinline__ void q_face_block(int blk, const float2 *__restrict__ vb, const float2 *__restrict__ qtab,
                                             float2 *__restrict__ yb, int n, float2 *sv)
{
    float2 *sa = sv + QF_HALO; // 162 coefficients [d][la][ou][ow][c]
    const long n3 = (long)n * n * n, n2 = (long)n * n;
    const int m = n - 2;
    const int tiles_u = (m + QF_U - 1) / QF_U, tiles_w = (m + QF_W - 1) / QF_W;
    const int per_face = tiles_u * tiles_w;
    const int face = blk / per_face, tile = blk % per_face;
    const int a = face >> 1, side = face & 1;          // face i_a = 0 (side 0) or n-1 (side 1)
    const int ua = a == 0 ? 1 : 0, wa = a == 2 ? 1 : 2; // the face's in-plane axes, ascending
    const int inward = side ? -1 : 1;
    const int u0 = (tile % tiles_u) * QF_U, w0 = (tile / tiles_u) * QF_W; // halo origin (grid coords)
    const long sa_ = a == 0 ? 1 : (a == 1 ? n : n2); // strides of the face normal and in-plane axes
    const long su = ua == 0 ? 1 : n, sw = wa == 1 ? n : n2;
    const int ia0 = side ? n - 1 : 0;
    const int cf = side ? 2 : 0;
    const int cls = (a == 0 ? cf : 1) + 3 * (a == 1 ? cf : 1) + 9 * (a == 2 ? cf : 1);
    const float2 *al = qtab + (long)cls * 243;
    for (int i = threadIdx.x; i < 162; i += Q_THREADS) {
        const int c = i % 3, l = (i / 3) % 18, d = i / 54;
        const int la = l / 9, ou = (l / 3) % 3 - 1, ow = l % 3 - 1;
        const int on = la ? inward : 0;
        const int o1 = a == 0 ? on : ou;
        const int o2 = a == 1 ? on : (a == 0 ? ou : ow);
        const int o3 = a == 2 ? on : ow;
        const int o = (o3 + 1) * 9 + (o2 + 1) * 3 + (o1 + 1);
        sa[i] = al[(d * 27 + o) * 3 + c];
    }
    for (int i = threadIdx.x; i < QF_HALO; i += Q_THREADS) {
        const int hu = i % QF_HU, hw = (i / QF_HU) % QF_HW, la = (i / (QF_HU * QF_HW)) % 2, d = i / (2 * QF_HU * QF_HW);
        const int gu = u0 + hu, gw = w0 + hw; // halo starts one point before the first face point (u = 1)
        const bool in = gu < n && gw < n;
        cp_async_zfill<sizeof(float2)>(&sv[i], in ? vb + d * n3 + (ia0 + (la ? inward : 0)) * sa_ + gu * su + gw * sw : vb, in);
    }
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    const int lu = threadIdx.x % QF_U, lw = threadIdx.x / QF_U;
    const int pu = 1 + u0 + lu, pw = 1 + w0 + lw;
    if (pu > m || pw > m) return;
    float2 acc0 = czero<float2>(), acc1 = czero<float2>(), acc2 = czero<float2>();
#pragma unroll
    for (int d = 0; d < 3; ++d)
#pragma unroll
        for (int la = 0; la < 2; ++la)
#pragma unroll
            for (int ou = -1; ou <= 1; ++ou)
#pragma unroll
                for (int ow = -1; ow <= 1; ++ow) {
                    const float2 val = sv[((d * 2 + la) * QF_HW + (lw + 1 + ow)) * QF_HU + (lu + 1 + ou)];
                    const float2 *ar = sa + ((d * 18 + la * 9 + (ou + 1) * 3 + (ow + 1)) * 3);
                    acc0 = cfma(ar[0], val, acc0);
                    acc1 = cfma(ar[1], val, acc1);
                    acc2 = cfma(ar[2], val, acc2);
                }
    const long i = ia0 * sa_ + pu * su + pw * sw;
    yb[i] = acc0;
    yb[n3 + i] = acc1;
    yb[2 * n3 + i] = acc2;
}

__device__ __forceinline__ void q_edge_block(int blk, const float2 *__restrict__ vb, const float2 *__restrict__ qtab,
                                             float2 *__restrict__ yb, int n, int nedge)
{
    const long n3 = (long)n * n * n;
    const int e = blk * (Q_THREADS / 32) + (int)(threadIdx.x >> 5);
    const int lane = threadIdx.x & 31;
    if (e >= nedge) return; // whole warps leave together
    int i1, i2, i3;
    edge_point(e, n, i1, i2, i3);
    const int c1 = i1 == 0 ? 0 : (i1 == n - 1 ? 2 : 1);
    const int c2 = i2 == 0 ? 0 : (i2 == n - 1 ? 2 : 1);
    const int c3 = i3 == 0 ? 0 : (i3 == n - 1 ? 2 : 1);
    const float2 *al = qtab + (long)(c1 + 3 * c2 + 9 * c3) * 243;
    float2 acc0 = czero<float2>(), acc1 = czero<float2>(), acc2 = czero<float2>();
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int term = lane + 32 * k;
        if (term >= 81) break;
        const int d = term / 27, o = term % 27;
        const int j1 = i1 + o % 3 - 1, j2 = i2 + (o / 3) % 3 - 1, j3 = i3 + o / 9 - 1;
        if (j1 < 0 || j2 < 0 || j3 < 0 || j1 >= n || j2 >= n || j3 >= n) continue;
        const float2 val = vb[d * n3 + ((long)j3 * n + j2) * n + j1];
        const float2 *ar = al + (d * 27 + o) * 3;
        acc0 = cfma(ar[0], val, acc0);
        acc1 = cfma(ar[1], val, acc1);
        acc2 = cfma(ar[2], val, acc2);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        acc0.x += __shfl_down_sync(0xffffffffu, acc0.x, off);
        acc0.y += __shfl_down_sync(0xffffffffu, acc0.y, off);
        acc1.x += __shfl_down_sync(0xffffffffu, acc1.x, off);
        acc1.y += __shfl_down_sync(0xffffffffu, acc1.y, off);
        acc2.x += __shfl_down_sync(0xffffffffu, acc2.x, off);
        acc2.y += __shfl_down_sync(0xffffffffu, acc2.y, off);
    }
    if (lane == 0) {
        const long i = ((long)i3 * n + i2) * n + i1;
        yb[i] = acc0;
        yb[n3 + i] = acc1;
        yb[2 * n3 + i] = acc2;
    }
}

__global__ void __launch_bounds__(Q_THREADS) k_q(const float2 *__restrict__ v,
                                                 const QInterior qa,
                                                 const float2 *__restrict__ qtab,
                                                 float2 *__restrict__ y, int n, int face_blocks,
                                                 int edge_blocks, int nedge)
{
    pdl_wait_and_trigger();
    extern __shared__ unsigned char smem_raw[];
    float2 *sv = reinterpret_cast<float2 *>(smem_raw); // Q_SMEM complex elements
    const long n3 = (long)n * n * n;
    const long b = blockIdx.y;
    const float2 *vb = v + b * 3 * n3;
    float2 *yb = y + b * 3 * n3;
    const int blk = blockIdx.x;
    if (blk < face_blocks) q_face_block(blk, vb, qtab, yb, n, sv);
    else if (blk < face_blocks + edge_blocks) q_edge_block(blk - face_blocks, vb, qtab, yb, n, nedge);
    else q_interior_block(blk - face_blocks - edge_blocks, vb, qa, yb, n, sv);
}

// Q in complex128: one thread per (point, output component), values and coefficients
// straight from the caches.  Bound: the FP64 pipe (two lanes per SM: a warp's FMA takes 16
// cycles of the SM's pipe, 64 of its scheduler's share): 972 n^3 FMAs, 6.3 us at n = 16 and
// 1.37 ms at n = 96.  Loads are nearly free beside that, and what counts is that every SM
// gets the same share of full warps: the 32 x 4 x 4 tiles of the complex64 kernel left one
// tile's work on each of 16 SMs at n = 16 (157 us; this kernel 17 us) and half-empty tiles
// elsewhere (n = 64: 600 against 416 us, n = 96: 1780 against 1395 us).  In complex64 the
// tiles win from n = 16 on (n = 64: 21 against 33 us) and the two are equal below.
// SPLIT = 3, for grids of fewer warps than schedulers: the three components d of a point
// in three warps of a block, their sums joined through shared memory.
template <typename C, int SPLIT>
__global__ void __launch_bounds__(SPLIT == 1 ? Q_THREADS : 96) k_q_direct(const C *__restrict__ v, const C *__restrict__ qtab,
                                                                         C *__restrict__ y, int n)
{
    pdl_wait_and_trigger();
    constexpr int PTS = SPLIT == 1 ? Q_THREADS : 32; // points per block
    const int n2 = n * n, n3 = n2 * n;
    const int i = blockIdx.x * PTS + threadIdx.x % PTS, c = blockIdx.y, d0 = threadIdx.x / PTS;
    const bool ok = i < n3;
    if (SPLIT == 1 && !ok) return;
    const int i1 = i % n, i2 = (i / n) % n, i3 = i / n2;
    const bool lo[3] = {i1 > 0, i2 > 0, i3 > 0}, hi[3] = {i1 < n - 1, i2 < n - 1, i3 < n - 1};
    const int cls = (lo[0] ? (hi[0] ? 1 : 2) : 0) + 3 * (lo[1] ? (hi[1] ? 1 : 2) : 0) + 9 * (lo[2] ? (hi[2] ? 1 : 2) : 0);
    const C *al = qtab + cls * 243 + c + d0 * 81;
    const C *vb = v + ((long)blockIdx.z * 3 + d0) * n3 + i;
    C acc = czero<C>();
#pragma unroll 1
    for (int d = 0; d < 3 / SPLIT; ++d, vb += n3, al += 81) {
        C a[27], u[27]; // all loads of a component before its FMAs
#pragma unroll
        for (int o = 0; o < 27; ++o) {
            const int o1 = o % 3 - 1, o2 = (o / 3) % 3 - 1, o3 = o / 9 - 1;
            const bool in = ok && (o1 == 0 || (o1 < 0 ? lo[0] : hi[0])) && (o2 == 0 || (o2 < 0 ? lo[1] : hi[1])) &&
                            (o3 == 0 || (o3 < 0 ? lo[2] : hi[2]));
            a[o] = al[3 * o];
            u[o] = czero<C>();
            if (in) u[o] = vb[o3 * n2 + o2 * n + o1];
        }
#pragma unroll
        for (int o = 0; o < 27; ++o) acc = cfma(a[o], u[o], acc);
    }
    if constexpr (SPLIT == 3) {
        __shared__ C part[2][32];
        if (d0 > 0) part[d0 - 1][threadIdx.x % 32] = acc;
        __syncthreads();
        if (d0 > 0 || !ok) return;
        acc = acc + part[0][threadIdx.x] + part[1][threadIdx.x];
    }
    y[((long)blockIdx.z * 3 + c) * n3 + i] = acc;
}

template <typename R>
spm_status apply_Q_typed(spm_problem_s *P, const void *vv, void *yv, int nrhs, cudaStream_t s)
{
    using C = typename cplx_of<R>::type;
    const int n = P->n;
    const C *qtab = sizeof(R) == 8 ? P->qtab128.as<C>() : P->qtab64.as<C>();
    if constexpr (sizeof(R) == 8) {
        // by n alone, so that a block of right-hand sides gives the bits of single ones
        if (3 * n * n * n <= 32 * 4 * 152) {
            launch_pdl(k_q_direct<C, 3>, dim3((unsigned)((n * n * n + 31) / 32), 3, (unsigned)nrhs), dim3(96), 0, s, (const C *)vv,
                       qtab, (C *)yv, n);
        } else {
            const dim3 grid((unsigned)((n * n * n + Q_THREADS - 1) / Q_THREADS), 3, (unsigned)nrhs);
            static PerDevice<EvenPlacement> even;
            launch_pdl(k_q_direct<C, 1>, grid, dim3(Q_THREADS), even_smem(even, k_q_direct<C, 1>, Q_THREADS, grid), s, (const C *)vv,
                       qtab, (C *)yv, n);
        }
        SPM_CUDA_TRY(cudaGetLastError());
        return SPM_OK;
    } else {
    // interior coefficients (class 13) by value, from the host copy of the table
    QInterior qa;
    for (int i = 0; i < 243; ++i) {
        const float ax = (float)P->qtab_h[2 * (13 * 243 + i)], ay = (float)P->qtab_h[2 * (13 * 243 + i) + 1];
        qa.a[i] = make_float4(ax, ax, -ay, ay);
    }
    const C *v = reinterpret_cast<const C *>(vv);
    C *y = reinterpret_cast<C *>(yv);
    const int m = n - 2;
    const int interior_blocks = ((m + QX - 1) / QX) * ((m + QY - 1) / QY) * ((m + QZ - 1) / QZ);
    const int face_blocks = 6 * ((m + QF_U - 1) / QF_U) * ((m + QF_W - 1) / QF_W);
    const int nedge = 12 * m + 8;
    const int edge_blocks = (nedge + Q_THREADS / 32 - 1) / (Q_THREADS / 32);
    constexpr size_t smem = sizeof(C) * Q_SMEM;
    static_assert(smem <= 48 * 1024, "no opt-in");
    const dim3 grid((unsigned)(face_blocks + edge_blocks + interior_blocks), (unsigned)nrhs);
    // Half of the L1 for shared memory, as the passes before it, while the blocks are few:
    // three on an SM, and no change of the division in between (Q A n = 32 19.1 us against
    // 21.8, n = 48 51 against 61, n = 64 70.5 against 78).  From about 2400 blocks on more
    // of them on an SM count (Q n = 96 45.6 us against 46.8, 16 fields at n = 64 212
    // against 225, 64 at n = 16 48.9 against 52.1).
    const int shared = (long)grid.x * grid.y <= 16 * 152 ? 50 : -1;
    launch_pdl_l1(shared, k_q, grid, dim3(Q_THREADS), smem, s, v, qa, qtab, y, n, face_blocks, edge_blocks, nedge);
    SPM_CUDA_TRY(cudaGetLastError());
    return SPM_OK;
    }
}

} // namespace

// alpha of every class spread over all 27 offsets [cls][d][o][c], o = (o3+1)*9 + (o2+1)*3 + (o1+1)
spm_status spm_build_qtable(spm_problem_s *P)
{
    std::vector<double> t(2 * 27 * 243, 0.0);
    for (int cls = 0; cls < 27; ++cls) {
        const int c[3] = {cls % 3, (cls / 3) % 3, cls / 9};
        int lo[3], hi[3], w[3];
        for (int d = 0; d < 3; ++d) {
            lo[d] = c[d] == 0 ? 0 : -1;
            hi[d] = c[d] == 2 ? 0 : 1;
            w[d] = hi[d] - lo[d] + 1;
        }
        const int T = w[0] * w[1] * w[2];
        for (int o3 = lo[2]; o3 <= hi[2]; ++o3)
            for (int o2 = lo[1]; o2 <= hi[1]; ++o2)
                for (int o1 = lo[0]; o1 <= hi[0]; ++o1) {
                    const int oi = ((o3 - lo[2]) * w[1] + (o2 - lo[1])) * w[0] + (o1 - lo[0]);
                    const int of = (o3 + 1) * 9 + (o2 + 1) * 3 + (o1 + 1);
                    for (int d = 0; d < 3; ++d)
                        for (int cc = 0; cc < 3; ++cc)
                            for (int ri = 0; ri < 2; ++ri)
                                t[2 * ((long)cls * 243 + (d * 27 + of) * 3 + cc) + ri] =
                                    P->alpha_h[2 * (((long)cls * 81 + d * T + oi) * 3 + cc) + ri];
                }
    }
    std::vector<float> t32(t.size());
    for (size_t i = 0; i < t.size(); ++i) t32[i] = (float)t[i];
    P->qtab_h = t;
    SPM_TRY(P->qtab128.ensure(sizeof(double) * t.size()));
    SPM_TRY(P->qtab64.ensure(sizeof(float) * t32.size()));
    SPM_CUDA_TRY(cudaMemcpy(P->qtab128.ptr, t.data(), sizeof(double) * t.size(), cudaMemcpyHostToDevice));
    SPM_CUDA_TRY(cudaMemcpy(P->qtab64.ptr, t32.data(), sizeof(float) * t32.size(), cudaMemcpyHostToDevice));
    return SPM_OK;
}

// supported z-pass kernels of a length: bit v set if variant v can run
static int zplan_supported(int L)
{
    const bool e8 = !(L == 96 || L == 192);
    return (e8 ? 1 << ZPROD_FOUR : 0) | ((!e8 || L >= 32) ? 1 << ZPROD_ONE : 0) | (L >= 32 ? 1 << ZPROD_TMA : 0) |
           ((L == 128 || L == 256 || L == 512) ? 1 << ZPROD_E16 : 0) | (L >= 32 ? 1 << ZPROD_STAGED : 0) |
           ((L == 64 || L == 128 || L == 256) ? 1 << ZPROD_SPLIT : 0);
}

spm_status spm_wait_selftest_impl(spm_problem_s *P)
{
    k_wait_selftest<<<1, 32, 0, P->stream>>>(P->dev_err.as<int>());
    SPM_CUDA_TRY(cudaGetLastError());
    return SPM_OK;
}

spm_status spm_apply_plan_impl(int prec, int L, int *get, const int *set)
{
    if (len_index(L) > 8) { spm_set_error("no apply plan for FFT length %d", L); return SPM_ERR_INVALID_ARG; }
    const int pi = prec == SPM_C128 ? 0 : 1;
    if (set) {
        const int zpart = *set & (ZPLAN_FUSED_XY - 1);
        const bool fz = *set >= 0 && (*set & ZPLAN_FUSED_XY) != 0;
        if (*set != -1 && (*set < 0 || *set > (ZPLAN_FUSED_XY | 5) || !(zplan_supported(L) & (1 << zpart)) ||
                           (fz && L != 64 && L != 128))) {
            spm_set_error("z-pass variant %d is not available for FFT length %d", *set, L);
            return SPM_ERR_INVALID_ARG;
        }
        zplan_get(pi, L); // initialise the table
        g_zplan[pi][len_index(L)].store(*set);
    }
    if (get) *get = zplan_get(pi, L);
    return SPM_OK;
}

// ---- persistence of the apply plans (JSON) ----
static const int k_plan_lengths[9] = {8, 16, 32, 64, 128, 256, 512, 96, 192};

static std::string device_name()
{
    int dev = 0;
    cudaDeviceProp prop;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaGetDeviceProperties(&prop, dev) != cudaSuccess) return "unknown";
    return prop.name;
}

spm_status spm_save_plans_impl(const char *path)
{
    std::string out = "{\n  \"device\": \"" + device_name() + "\",\n  \"plans\": [";
    bool first = true;
    for (int pi = 0; pi < 2; ++pi)
        for (int li = 0; li < 9; ++li) {
            const int L = k_plan_lengths[li];
            const int z = zplan_get(pi, L);
            if (z < 0) continue;
            char buf[256];
            float t[6];
            {
                std::lock_guard<std::mutex> lock(g_ztime_mu);
                for (int v = 0; v < 6; ++v) t[v] = g_ztime[pi][li][v];
            }
            float tf;
            {
                std::lock_guard<std::mutex> lock(g_ztime_mu);
                tf = g_ztime_fused[pi][li];
            }
            snprintf(buf, sizeof buf,
                     "%s\n    {\"prec\": \"%s\", \"L\": %d, \"variant\": %d, \"ms\": [%.6g, %.6g, %.6g, %.6g, %.6g, %.6g], "
                     "\"fused_xy_ms\": %.6g}",
                     first ? "" : ",", pi == 0 ? "c128" : "c64", L, z, t[0], t[1], t[2], t[3], t[4], t[5], tf);
            out += buf;
            first = false;
        }
    out += "\n  ]\n}\n";
    FILE *f = fopen(path, "w");
    if (!f) { spm_set_error("cannot open %s for writing", path); return SPM_ERR_INVALID_ARG; }
    const size_t w = fwrite(out.data(), 1, out.size(), f);
    fclose(f);
    if (w != out.size()) { spm_set_error("short write to %s", path); return SPM_ERR_INVALID_ARG; }
    return SPM_OK;
}

// Reads the file written above: the device name must match the current
// device's; each {"prec", "L", "variant"} entry with a variant the length
// supports is installed.  *loaded = number of entries installed.
spm_status spm_load_plans_impl(const char *path, int *loaded)
{
    FILE *f = fopen(path, "r");
    if (!f) { spm_set_error("cannot open %s", path); return SPM_ERR_INVALID_ARG; }
    std::string txt;
    char buf[4096];
    size_t r;
    while ((r = fread(buf, 1, sizeof buf, f)) > 0) txt.append(buf, r);
    fclose(f);
    auto str_after = [&](size_t pos, const char *key, std::string &val) -> bool {
        size_t k = txt.find(key, pos);
        if (k == std::string::npos) return false;
        size_t q0 = txt.find('"', txt.find(':', k) + 1);
        size_t q1 = q0 == std::string::npos ? q0 : txt.find('"', q0 + 1);
        if (q1 == std::string::npos) return false;
        val = txt.substr(q0 + 1, q1 - q0 - 1);
        return true;
    };
    std::string dev;
    if (!str_after(0, "\"device\"", dev)) { spm_set_error("%s: no device name", path); return SPM_ERR_INVALID_ARG; }
    if (dev != device_name()) {
        spm_set_error("%s was tuned on \"%s\", this device is \"%s\"", path, dev.c_str(), device_name().c_str());
        return SPM_ERR_INVALID_ARG;
    }
    int count = 0;
    size_t pos = txt.find("\"plans\"");
    while (pos != std::string::npos) {
        size_t ob = txt.find('{', pos);
        if (ob == std::string::npos) break;
        size_t cb = txt.find('}', ob);
        if (cb == std::string::npos) break;
        const std::string obj = txt.substr(ob, cb - ob + 1);
        pos = cb + 1;
        int L = 0, z = -1;
        char pr[8] = "";
        const size_t kp = obj.find("\"prec\""), kl = obj.find("\"L\""), kv = obj.find("\"variant\"");
        if (kp == std::string::npos || kl == std::string::npos || kv == std::string::npos) continue;
        if (sscanf(obj.c_str() + obj.find(':', kp) + 1, " \"%7[^\"]\"", pr) != 1) continue;
        if (sscanf(obj.c_str() + obj.find(':', kl) + 1, " %d", &L) != 1) continue;
        if (sscanf(obj.c_str() + obj.find(':', kv) + 1, " %d", &z) != 1) continue;
        const int prec = strcmp(pr, "c128") == 0 ? SPM_C128 : (strcmp(pr, "c64") == 0 ? SPM_C64 : -1);
        if (prec < 0 || len_index(L) > 8) continue;
        if (spm_apply_plan_impl(prec, L, nullptr, &z) == SPM_OK) ++count;
    }
    if (loaded) *loaded = count;
    return SPM_OK;
}

// Per-pass device times of one apply (A, or Q A), averaged over reps applies:
// an event after every pass, so the passes run serialised (no overlap of one
// pass's tail with the next one's start) and their sum exceeds the pipelined
// apply time.
namespace {
template <typename R>
spm_status profile_typed(spm_problem_s *P, const void *xv, void *yv, int with_q, int reps, float *pass_ms, int *npasses,
                         cudaStream_t s)
{
    using C = typename cplx_of<R>::type;
    const int n = P->n, L = P->L;
    const long n2 = (long)n * n, L2 = (long)L * L;
    const bool dbl = sizeof(R) == 8;
    const C *m = dbl ? P->m128.as<C>() : P->m64.as<C>();
    const C *p = dbl ? P->p128.as<C>() : P->p64.as<C>();
    const C *spec = dbl ? P->spec128.as<C>() : P->spec64.as<C>();
    const C *tw = dbl ? P->tw128.as<C>() : P->tw64.as<C>();
    const int chunk = dbl ? P->chunk128 : P->chunk64;
    const long w1 = 4 * n2 * L, w2 = 4 * (long)n * L2;
    SPM_TRY(P->work.ensure(sizeof(C) * (size_t)chunk * (w1 + w2)));
    C *W1 = P->work.as<C>();
    C *W2 = W1 + (long)chunk * w1;
    const C *x = reinterpret_cast<const C *>(xv);
    C *y = reinterpret_cast<C *>(yv);
    C *ax = y;
    if (with_q) {
        SPM_TRY(P->kry.ensure(std::max(P->kry.bytes, sizeof(C) * 3 * (size_t)n2 * n)));
        ax = P->kry.as<C>();
    }
    int zvar = ZPROD_FOUR;
    SPM_TRY(choose_zplan<R>(L, x, ax, m, p, spec, tw, W1, W2, 1, P->dev_err.as<int>(), s, &zvar));
    cudaEvent_t ev[8];
    for (int k = 0; k < 8; ++k) SPM_CUDA_TRY(cudaEventCreate(&ev[k]));
    float acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    int nev = 0;
    spm_status st = SPM_OK;
    for (int r = 0; r < reps && st == SPM_OK; ++r) {
        nev = 0;
        cudaEventRecord(ev[nev++], s);
        st = run_chunk<R>(L, x, ax, m, p, spec, tw, W1, W2, 1, zvar, P->dev_err.as<int>(), s, ev, &nev);
        if (st == SPM_OK && with_q) {
            st = spm_apply_Q_impl(P, dbl ? SPM_C128 : SPM_C64, ax, y, 1, s);
            cudaEventRecord(ev[nev++], s);
        }
        if (st == SPM_OK && cudaEventSynchronize(ev[nev - 1]) != cudaSuccess) st = SPM_ERR_CUDA;
        for (int k = 1; k < nev && st == SPM_OK; ++k) {
            float ms = 0;
            cudaEventElapsedTime(&ms, ev[k - 1], ev[k]);
            acc[k - 1] += ms;
        }
    }
    for (int k = 0; k < 8; ++k) cudaEventDestroy(ev[k]);
    if (st != SPM_OK) {
        if (st == SPM_ERR_CUDA) spm_set_error("profiled apply failed: %s", cudaGetErrorString(cudaGetLastError()));
        return st;
    }
    *npasses = nev - 1;
    for (int k = 0; k < nev - 1; ++k) pass_ms[k] = acc[k] / reps;
    return SPM_OK;
}
} // namespace

spm_status spm_profile_apply_impl(spm_problem_s *P, int prec, const void *x, void *y, int with_q, int reps,
                                  float *pass_ms, int *npasses, cudaStream_t s)
{
    return prec == SPM_C128 ? profile_typed<double>(P, x, y, with_q, reps, pass_ms, npasses, s)
                            : profile_typed<float>(P, x, y, with_q, reps, pass_ms, npasses, s);
}

spm_status spm_apply_A_impl(spm_problem_s *P, int prec, const void *x, void *y, int nrhs, cudaStream_t s)
{
    return prec == SPM_C128 ? apply_A_typed<double>(P, x, y, nrhs, s) : apply_A_typed<float>(P, x, y, nrhs, s);
}

spm_status spm_apply_Q_impl(spm_problem_s *P, int prec, const void *v, void *y, int nrhs, cudaStream_t s)
{
    return prec == SPM_C128 ? apply_Q_typed<double>(P, v, y, nrhs, s) : apply_Q_typed<float>(P, v, y, nrhs, s);
}

// ------------------------------------------------------------------ spectra
namespace {

// Circulant embedding of one kernel on the L^3 grid: slot v in [0,L) holds the
// entry for offset t = v (v < n) or v - L (v > n); slot n is zero.
// Entries (Section 2): G_t = h^3 G(t h), G^d_t = h^3 dG/dx_d(t h) off the
// diagonal; ORDER4 corrections at t = 0 (G) and t = +-e_d (G^d).
__device__ void kernel_entry_dev(int t1, int t2, int t3, double h, double k, int quad, double Z, double2 out[4])
{
    const double inv4pi = 0.079577471545947667884; // 1/(4 pi)
    if (t1 == 0 && t2 == 0 && t3 == 0) {
        double zc = quad == 0 ? Z : 0.0;
        out[0] = make_double2(-h * h * zc * inv4pi, h * h * h * k * inv4pi);
        out[1] = out[2] = out[3] = make_double2(0.0, 0.0);
        return;
    }
    double x1 = t1 * h, x2 = t2 * h, x3 = t3 * h;
    double r = sqrt(x1 * x1 + x2 * x2 + x3 * x3);
    double sn, cs;
    sincos(k * r, &sn, &cs);
    double h3 = h * h * h;
    double g = h3 * inv4pi / r;
    out[0] = make_double2(g * cs, g * sn);
    // (i k r - 1) e^{ikr} = (-cs - k r sn) + i (k r cs - sn)
    double re = -cs - k * r * sn, im = k * r * cs - sn;
    double f = h3 * inv4pi / (r * r * r);
    double xs[3] = {x1, x2, x3};
    int ts[3] = {t1, t2, t3};
    for (int d = 0; d < 3; ++d) {
        out[1 + d] = make_double2(f * xs[d] * re, f * xs[d] * im);
        if (quad == 0) {
            bool axis = (ts[(d + 1) % 3] == 0) && (ts[(d + 2) % 3] == 0) && (ts[d] == 1 || ts[d] == -1);
            if (axis) out[1 + d].x += ts[d] * h * Z / (24.0 * 3.14159265358979323846);
        }
    }
}

__global__ void k_fill_circulant(double2 *out, int q, int n, int L, double h, double k, int quad, double Z)
{
    long L3 = (long)L * L * L;
    long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= L3) return;
    int v1 = (int)(gid % L), v2 = (int)((gid / L) % L), v3 = (int)(gid / ((long)L * L));
    if (v1 == n || v2 == n || v3 == n) { out[gid] = make_double2(0, 0); return; }
    int t1 = v1 < n ? v1 : v1 - L, t2 = v2 < n ? v2 : v2 - L, t3 = v3 < n ? v3 : v3 - L;
    double2 e[4];
    kernel_entry_dev(t1, t2, t3, h, k, quad, Z, e);
    out[gid] = e[q];
}

__global__ void k_entries_table(double2 *out, int n, double h, double k, int quad, double Z)
{
    int W = 2 * n - 1;
    long W3 = (long)W * W * W;
    long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= W3) return;
    int a1 = (int)(gid % W), a2 = (int)((gid / W) % W), a3 = (int)(gid / ((long)W * W));
    double2 e[4];
    kernel_entry_dev(a1 - (n - 1), a2 - (n - 1), a3 - (n - 1), h, k, quad, Z, e);
    for (int q = 0; q < 4; ++q) out[q * W3 + gid] = e[q];
}

__global__ void k_octant(const double2 *__restrict__ full, double2 *spec128, float2 *spec64, int n, int L,
                         double scale)
{
    int n1 = n + 1;
    long tot = (long)n1 * n1 * n1;
    long gid = (long)blockIdx.x * blockDim.x + threadIdx.x;
    if (gid >= tot) return;
    int a1 = (int)(gid % n1), a2 = (int)((gid / n1) % n1), a3 = (int)(gid / ((long)n1 * n1));
    double2 v = full[((long)a3 * L + a2) * L + a1];
    v.x *= scale;
    v.y *= scale;
    spec128[gid] = v;
    spec64[gid] = to_c64(v);
}

// plain rows: FFT of contiguous rows of length L, in place
__global__ void __launch_bounds__(NT) k_rows_plain(double2 *a, int L, int logL, long nrows, int nl,
                                                   const double2 *__restrict__ tw)
{
    extern __shared__ unsigned char smem_raw[];
    double2 *buf0 = reinterpret_cast<double2 *>(smem_raw);
    double2 *buf1 = buf0 + nl * L;
    long row0 = (long)blockIdx.x * nl;
    for (int idx = threadIdx.x; idx < nl * L; idx += blockDim.x) {
        long g = row0 + idx / L;
        buf0[idx] = g < nrows ? a[row0 * L + idx] : make_double2(0, 0);
    }
    __syncthreads();
    double2 *res = smem_fft<-1>(buf0, buf1, L, logL, nl, L, tw);
    for (int idx = threadIdx.x; idx < nl * L; idx += blockDim.x) {
        long g = row0 + idx / L;
        if (g < nrows) a[row0 * L + idx] = res[idx];
    }
}

} // namespace

spm_status spm_build_spectra(spm_problem_s *P)
{
    const int n = P->n, L = P->L, logL = P->logL;
    const long L3 = (long)L * L * L, L2 = (long)L * L;
    const int n1 = n + 1;
    const long oct = (long)n1 * n1 * n1;
    DevBuf full;
    SPM_TRY(full.ensure(sizeof(double2) * L3));
    SPM_TRY(P->spec128.ensure(sizeof(double2) * 4 * oct));
    SPM_TRY(P->spec64.ensure(sizeof(float2) * 4 * oct));
    cudaStream_t s = P->stream;
    double2 *F = full.as<double2>();
    const double2 *tw = P->tw128.as<double2>();
    int TX = 8;
    while (TX > 2 && 2 * TX * (L + 1) * 16 > 100 * 1024) TX >>= 1;
    if (TX > L) TX = L;
    const int nlx = L >= 256 ? 1 : 256 / L;
    for (int q = 0; q < 4; ++q) {
        k_fill_circulant<<<(unsigned)((L3 + 255) / 256), 256, 0, s>>>(F, q, n, L, P->h, P->k, P->quad, P->zconst);
        k_rows_plain<<<(unsigned)((L2 + nlx - 1) / nlx), NT, 2 * 16 * nlx * L, s>>>(F, L, logL, L2, nlx, tw);
        // y: lines along y of [z][y][x]; in place is safe (each block owns its columns)
        k_cols<double, -1><<<dim3(L / TX, L, 1), NT, 2 * 16 * TX * (L + 1), s>>>(
            F, F, L, logL, L, L, L, 1, 0, 0, L2, 0, 0, L2, TX, tw);
        // z: lines along z, inner = L^2
        k_cols<double, -1><<<dim3((unsigned)(L2 / TX), 1, 1), NT, 2 * 16 * TX * (L + 1), s>>>(
            F, F, L, logL, L, L, L2, 1, 0, 0, 0, 0, 0, 0, TX, tw);
        double scale = (q == 0 ? P->k * P->k : 1.0) / (double)L3;
        k_octant<<<(unsigned)((oct + 255) / 256), 256, 0, s>>>(F, P->spec128.as<double2>() + q * oct,
                                                               P->spec64.as<float2>() + q * oct, n, L, scale);
    }
    SPM_CUDA_TRY(cudaGetLastError());
    SPM_CUDA_TRY(cudaStreamSynchronize(s));
    full.release();
    return SPM_OK;
}

spm_status spm_entries_device(spm_problem_s *P, DevBuf &t)
{
    const int n = P->n, W = 2 * n - 1;
    const long W3 = (long)W * W * W;
    SPM_TRY(t.ensure(sizeof(double2) * 4 * W3));
    k_entries_table<<<(unsigned)((W3 + 255) / 256), 256, 0, P->stream>>>(t.as<double2>(), n, P->h, P->k, P->quad,
                                                                        P->zconst);
    SPM_CUDA_TRY(cudaGetLastError());
    return SPM_OK;
}

spm_status spm_entries_impl(spm_problem_s *P, double *out_host)
{
    const int n = P->n, W = 2 * n - 1;
    const long W3 = (long)W * W * W;
    DevBuf t;
    SPM_TRY(spm_entries_device(P, t));
    SPM_CUDA_TRY(cudaMemcpyAsync(out_host, t.ptr, sizeof(double2) * 4 * W3, cudaMemcpyDeviceToHost, P->stream));
    SPM_CUDA_TRY(cudaStreamSynchronize(P->stream));
    t.release();
    return SPM_OK;
}

// The largest smem request of the FFT passes exceeds the 48 KB default; opt in once.
spm_status spm_apply_init_attributes()
{
    const int big = 200 * 1024;
    SPM_CUDA_TRY(cudaFuncSetAttribute(k_cols<float, -1>, cudaFuncAttributeMaxDynamicSharedMemorySize, big));
    SPM_CUDA_TRY(cudaFuncSetAttribute(k_cols<float, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, big));
    SPM_CUDA_TRY(cudaFuncSetAttribute(k_cols<double, -1>, cudaFuncAttributeMaxDynamicSharedMemorySize, big));
    SPM_CUDA_TRY(cudaFuncSetAttribute(k_cols<double, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, big));
    SPM_CUDA_TRY(cudaFuncSetAttribute(k_rows_plain, cudaFuncAttributeMaxDynamicSharedMemorySize, big));
    return SPM_OK;
}

// ================================================================ no-allocation apply
// Some callers cannot allocate device memory when they apply the operator: a
// process whose device memory is owned by another allocator or budget (a pool
// reserved up front, where a raw cudaMalloc could fail or fragment it), or a
// latency-bound loop that cannot afford cudaMalloc/cudaFree, which may block
// or synchronise the device.  spm_apply_A_noalloc serves them: it runs the same
// passes as spm_apply_A but keeps the pass intermediates (24 n^3 complex values
// per right-hand side, right-hand sides taken one at a time) in this file-scope
// device array instead of library-allocated workspace.  Every GPU that loads
// the library holds the array until the process exits.
#define SPM_NOALLOC_SCRATCH_BYTES (64ull << 20)
static __device__ __align__(256) unsigned char g_spm_noalloc_scratch[SPM_NOALLOC_SCRATCH_BYTES];

namespace {
// Host code cannot use the array's name as a device address: look the address
// up on the current device.  The lookup is cheap and allocates nothing, so it is
// repeated on every call (a cached address would go stale after a device reset).
spm_status noalloc_scratch(void **out)
{
    void *p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_spm_noalloc_scratch);
    if (e != cudaSuccess || !p) {
        spm_set_error("cudaGetSymbolAddress of the no-allocation scratch failed: %s", cudaGetErrorString(e));
        return SPM_ERR_CUDA;
    }
    *out = p;
    return SPM_OK;
}

template <typename R>
spm_status apply_A_noalloc_typed(spm_problem_s *P, const void *xv, void *yv, int nrhs, cudaStream_t s)
{
    using C = typename cplx_of<R>::type;
    const int n = P->n, L = P->L;
    const long n2 = (long)n * n, n3 = n2 * n, L2 = (long)L * L;
    const long w1 = 4 * n2 * L, w2 = 4 * (long)n * L2;
    const unsigned long long need = sizeof(C) * (unsigned long long)(w1 + w2);
    if (need > SPM_NOALLOC_SCRATCH_BYTES) {
        spm_set_error("spm_apply_A_noalloc: n = %d in %s needs %llu bytes of scratch, above the fixed %llu", n,
                      sizeof(R) == 8 ? "complex128" : "complex64", need, SPM_NOALLOC_SCRATCH_BYTES);
        return SPM_ERR_INVALID_ARG;
    }
    void *scratch = nullptr;
    SPM_TRY(noalloc_scratch(&scratch));
    C *W1 = reinterpret_cast<C *>(scratch);
    C *W2 = W1 + w1;
    const bool dbl = sizeof(R) == 8;
    const C *m = dbl ? P->m128.as<C>() : P->m64.as<C>();
    const C *p = dbl ? P->p128.as<C>() : P->p64.as<C>();
    const C *spec = dbl ? P->spec128.as<C>() : P->spec64.as<C>();
    const C *tw = dbl ? P->tw128.as<C>() : P->tw64.as<C>();
    const C *x = reinterpret_cast<const C *>(xv);
    C *y = reinterpret_cast<C *>(yv);
    // Every pass writes its whole output before the next pass reads it, so no
    // part of the shared scratch has to be cleared between calls.  The z-pass
    // kernel is the one the timed applies chose, if any (no timing here).
    const int zcached = zplan_get(dbl ? 0 : 1, L);
    const int zvar = zcached >= 0 ? zcached : (L == 96 || L == 192 ? ZPROD_ONE : ZPROD_FOUR);
    for (int b = 0; b < nrhs; ++b) {
        const C *xb = x + (long)b * 3 * n3;
        C *yb = y + (long)b * 3 * n3;
        SPM_TRY(run_chunk<R>(L, xb, yb, m, p, spec, tw, W1, W2, 1, zvar, P->dev_err.as<int>(), s));
    }
    SPM_CUDA_TRY(cudaGetLastError());
    return SPM_OK;
}
} // namespace

extern "C" spm_status spm_apply_A_noalloc(spm_problem P, spm_prec prec, const void *x, void *y, int nrhs,
                                          void *stream)
{
    if (!P) { spm_set_error("NULL problem"); return SPM_ERR_INVALID_ARG; }
    if (prec != SPM_C128 && prec != SPM_C64) { spm_set_error("precision must be SPM_C128 or SPM_C64"); return SPM_ERR_INVALID_ARG; }
    if (nrhs < 0) { spm_set_error("nrhs < 0"); return SPM_ERR_INVALID_ARG; }
    if (nrhs > 0 && (!x || !y)) { spm_set_error("NULL buffer"); return SPM_ERR_INVALID_ARG; }
    if (nrhs > 0 && x == y) { spm_set_error("input and output alias"); return SPM_ERR_INVALID_ARG; }
    if (nrhs == 0) return SPM_OK;
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    return prec == SPM_C128 ? apply_A_noalloc_typed<double>(P, x, y, nrhs, s)
                            : apply_A_noalloc_typed<float>(P, x, y, nrhs, s);
}
