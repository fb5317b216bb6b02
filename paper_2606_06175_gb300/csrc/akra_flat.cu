// akra_flat.cu -- the flat-sky variant of the operator (Sec. II B: each SHT replaced by a 2D
// FFT, the four-step structure of A and the CG solver unchanged).
//
// On an n x n periodic patch the unknown is x = F z, the unitary 2D Fourier transform of the
// complex field z = κ_E + i κ_B (rows k2, columns k1, FFT frequency order), and
//   A x   = F^-1 (D x)            γ1 + i γ2 at the pixels,  D(k) = (k1² - k2² + 2i k1 k2)/|k|²
//   A^T u = conj(D) F (u1 + i u2) (the exact adjoint: F is unitary and |D| <= 1)
//   H x   = conj(D) F (W F^-1 (D x)) + λ_eff x,   W = M N^-1 on the pixels,
// the flat-sky Kaiser-Squires kernel (D(0) = 0) in place of D_l and the spin-2 SHTs.
//
// A 2D transform is two passes of row FFTs; a pass writes its result transposed, so that the next one
// reads rows again, and for H the second and third passes (inverse along y, ×W, forward along y) are one
// kernel per row of the transposed field, as the ring FFT fuses W between its two DFTs.
//
// Row FFTs are radix-16 Stockham passes (plus one pass of radix 2, 4 or 8 where log2 n is no multiple of 4; radix 4
// for FP64 rows up to 256),
// 16 elements of a row in each thread's registers: a row of 2048 crosses shared memory twice instead of the
// six times of radix-4 passes, consecutive threads load consecutive twiddles, and the first pass reads and the
// last writes global memory directly.  n is a template argument, which leaves one address and immediate
// offsets per pass: with n at run time the index arithmetic was 35% of the issue slots and H took 129 us.
// H at n = 2048, FP32: 95 us in three launches (0.2 GB through the L2), 247 us as five launches of radix-4
// passes and transposes (0.34 GB); 512: 24 against 36; 8192: 1545 against 4429; 2048 FP64: 1.46 ms against 1.75.
// FP32 is bound by issue and the L2 latency of the loads, which two blocks per SM cover in part; FP64 by the
// FP64 pipe.
#include "akra_internal.cuh"

namespace akra {
namespace flat {

constexpr int kMaxN = 8192;        // largest grid side

// a row's slots in shared memory: one of padding in 17, and 4 so that the rows of a transposed store are
// read from different banks
__host__ __device__ constexpr int slots(int n) { return n + (n >> 4) + 4; }
__device__ __forceinline__ int pd(int i) { return i + (i >> 4); }   // bank-conflict padding

// complex helpers on float2 / double2 (C)
template <typename C> __device__ __forceinline__ C cmul(C a, C b)
{
    return C{fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x)};
}
template <typename C> __device__ __forceinline__ C cadd(C a, C b) { return C{a.x + b.x, a.y + b.y}; }
template <typename C> __device__ __forceinline__ C csub(C a, C b) { return C{a.x - b.x, a.y - b.y}; }
template <int S, typename C> __device__ __forceinline__ C mul_si(C a)   // S i a
{
    return S > 0 ? C{-a.y, a.x} : C{a.y, -a.x};
}

// DFTs of sign S in registers, natural order in and out: v[r] <- Σ_q v[q] e^{S 2πi qr/N}
template <int S, typename C> __device__ __forceinline__ void dft4(C &a, C &b, C &c, C &d)
{
    const C s0 = cadd(a, c), d0 = csub(a, c), s1 = cadd(b, d), d1 = mul_si<S>(csub(b, d));
    a = cadd(s0, s1);
    b = cadd(d0, d1);
    c = csub(s0, s1);
    d = csub(d0, d1);
}

// e^{S 2πi m/16}: cosines of 0, π/8, .. π/2 and symmetry (m a compile-time constant after unrolling)
template <int S, typename T> __device__ __forceinline__ cx_t<T> root16(int m)
{
    const T c[5] = {T(1), T(0.92387953251128675613), T(0.70710678118654752440), T(0.38268343236508977173), T(0)};
    auto cs = [&](int k) { k &= 15; return k <= 4 ? c[k] : k <= 8 ? -c[8 - k] : k <= 12 ? -c[k - 8] : c[16 - k]; };
    return cx_t<T>{cs(m), S > 0 ? cs(m + 12) : -cs(m + 12)};
}

// R-point DFT of v[0..R) for R = 2, 4, 8, 16 as 4-point DFTs over the high digit, roots, and DFTs over the low one
template <int S, typename T, int R> __device__ __forceinline__ void dft(cx_t<T> *v)
{
    using C = cx_t<T>;
    if constexpr (R == 2) {
        const C a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    } else if constexpr (R == 4) {
        dft4<S>(v[0], v[1], v[2], v[3]);
    } else {
        constexpr int B = R / 4;   // q = B a + b, r = c + 4 d
#pragma unroll
        for (int b = 0; b < B; b++) {
            dft4<S>(v[b], v[b + B], v[b + 2 * B], v[b + 3 * B]);   // over a: slot b + B c
#pragma unroll
            for (int c = 1; c < 4; c++)
                if (b > 0) v[b + B * c] = cmul(v[b + B * c], root16<S, T>(b * c * (16 / R)));
        }
        C o[R];
#pragma unroll
        for (int c = 0; c < 4; c++) {
            C w[B];
#pragma unroll
            for (int b = 0; b < B; b++) w[b] = v[B * c + b];
            dft<S, T, B>(w);
#pragma unroll
            for (int d = 0; d < B; d++) o[c + 4 * d] = w[d];
        }
#pragma unroll
        for (int r = 0; r < R; r++) v[r] = o[r];
    }
}

// log2 of the elements E of a row in a thread: 16 elements and radix-16 passes, but 4 for the FP64 rows up to 256,
// whose few warps are bound by each warp's own FP64 instructions (H at n = 64: 70 us with 16, 27 with 4;
// 39 with radix-4 passes through shared memory).
template <typename T> __host__ __device__ constexpr int log_elems(int logn) { return sizeof(T) == 8 && logn <= 8 ? 2 : 4; }

// A row of N = 2^LOGN in N/E threads: radix-E passes and one of R0 = 2^(LOGN mod log2 E) where that is not 1.
// Everything but the thread's index is a compile-time constant, so that the accesses of a pass are one
// address and immediate offsets.
template <typename T, int LOGN>
struct Row {
    using C = cx_t<T>;
    static constexpr int LE = log_elems<T>(LOGN), E = 1 << LE;
    static constexpr int N = 1 << LOGN, TN = N / E, R0 = 1 << (LOGN % LE);
    static constexpr int R1 = R0 > 1 ? R0 : E;   // first pass of the backward transform, last of the forward one

    // offset from t of the place of v[i] as the first pass of radix R reads it and the last one leaves it
    template <int R> static __host__ __device__ constexpr int place(int i) { return (i / R) * TN + (i % R) * (E / R) * TN; }

    // slot of element i + off
    static __device__ __forceinline__ int at(int i, int off)
    {
        return off % 16 == 0 ? pd(i) + off + off / 16 : pd(i + off);
    }

    // Stockham pass of radix R after passes of product Ns: butterflies j = t + u TN (u < E/R), inputs
    // x[j + q N/R] in v[u R + q], twiddled by e^{S 2πi qk/(Ns R)}, k = j mod Ns (table w[(q - 1) Ns + k],
    // sign -), outputs x[(j - k) R + k + r Ns]
    template <int S, int R, int Ns> static __device__ __forceinline__ void pass(C (&v)[E], int t, const C *__restrict__ w)
    {
#pragma unroll
        for (int u = 0; u < E / R; u++) {
            if (Ns > 1) {
                const C *wk = w + ((t + u * TN) & (Ns - 1));
#pragma unroll
                for (int q = 1; q < R; q++) {
                    C c = wk[(q - 1) * Ns];
                    if (S > 0) c.y = -c.y;
                    v[u * R + q] = cmul(v[u * R + q], c);
                }
            }
            dft<S, T, R>(v + u * R);
        }
    }
    // its outputs to the row's buffer; (k + r Ns) / 16 = r Ns / 16 for every pass
    template <int R, int Ns> static __device__ __forceinline__ void put(C *buf, const C (&v)[E], int t)
    {
#pragma unroll
        for (int u = 0; u < E / R; u++) {
            const int k = (t + u * TN) & (Ns - 1);
            const int o = Ns == 1 ? at(t * R, u * TN * R) : pd((t + u * TN - k) * R + k);
#pragma unroll
            for (int r = 0; r < R; r++) buf[o + r * Ns + (r * Ns >> 4)] = v[u * R + r];
        }
    }
    // inputs of a pass of radix R
    template <int R> static __device__ __forceinline__ void get(const C *buf, C (&v)[E], int t)
    {
#pragma unroll
        for (int i = 0; i < E; i++) v[i] = buf[at(t, place<R>(i))];
    }

    // radix-E passes from Ns to the product M; then the buffer holds the inputs of a pass of radix R0, or v the row
    template <int S, int Ns, int M> static __device__ __forceinline__ void passes(C (&v)[E], C *buf, int t, const C *__restrict__ w)
    {
        if constexpr (Ns < M) {
            pass<S, E, Ns>(v, t, w);
            if constexpr (Ns * E < N) {
                __syncthreads();   // the buffer's last readers
                put<E, Ns>(buf, v, t);
                __syncthreads();
                if constexpr (Ns * E < M) get<E>(buf, v, t);
            }
            passes<S, Ns * E, M>(v, buf, t, w + (Ns > 1 ? (E - 1) * Ns : 0));
        } else if constexpr (M < N) {
            get<R0>(buf, v, t);
            pass<S, R0, M>(v, t, w);
        }
    }
    // Backward: R0, E, E, ..; forward: E, E, .., R0.  The backward transform ends and the forward one starts
    // with the same radix-E places, so ×W between them needs no exchange.
    static __device__ __forceinline__ void backward(C (&v)[E], C *buf, int t, const C *__restrict__ w)
    {
        if constexpr (R0 > 1) {
            pass<+1, R0, 1>(v, t, w);
            put<R0, 1>(buf, v, t);
            __syncthreads();
            get<E>(buf, v, t);
        }
        passes<+1, R0, N>(v, buf, t, w);
    }
    static __device__ __forceinline__ void forward(C (&v)[E], C *buf, int t, const C *__restrict__ w)
    {
        passes<-1, 1, N / R0>(v, buf, t, w);
    }
};

// flat-sky Kaiser-Squires kernel at frequencies (a, b)
template <typename T>
__device__ __forceinline__ cx_t<T> ks(T a, T b)
{
    const T q = a * a + b * b;
    if (q == T(0)) return cx_t<T>{0, 0};
    const T inv = T(1) / q;
    return cx_t<T>{(a * a - b * b) * inv, T(2) * a * b * inv};
}

template <typename T>
struct Args {
    bool tr;                 // the result goes to out[r][column][row]
    const cx_t<T> *wb, *wf;  // twiddles of the backward and of the forward passes
    const cx_t<T> *in;       // [R][n][n]
    cx_t<T> *out;            // [R][n][n]
    const T *Wt;             // middle pass: [n][n] weights, transposed, scaled by 1/n^2
    const cx_t<T> *xreg;     // mode 2: x for the λ_eff term (nullptr: none)
    T lam, scale;
    const int *skip;         // device flag: return at once if set
};

// Up to 4096 a pass stores its rows transposed; rows of 8192, of which a block would hold too few for a
// sector, are stored as they are and go through k_transpose.
__host__ __device__ constexpr bool fused_transpose(int n) { return n <= 4096; }

// Rows of a block.  A transposed store joins 32 bytes, a sector, from 4 FP32 rows: at n = 2048 H takes 95 us against
// 100 with two, at 4096 (1024 threads) 361 against 425.  FP64 blocks are of 256 threads where that holds a row: at
// 4096 one row takes 6.03 ms against 6.43 with two, the FP64 pipe being the bound.  Short rows fill a warp: the few
// blocks of a small grid would otherwise leave most SMs idle.
template <typename T> __host__ __device__ constexpr int rows_per_block(int logn)
{
    const int n = 1 << logn, per_row = n >> log_elems<T>(logn);
    const int sector = 32 / (int)sizeof(cx_t<T>), threads = sizeof(T) == 8 ? 256 : fused_transpose(n) ? 1024 : 512;
    const int most = threads < per_row ? 1 : threads / per_row;
    const int least = per_row >= 32 ? 1 : 32 / per_row < n ? 32 / per_row : n;
    const int rows = sector < most ? sector : most;
    return least > rows ? least : rows;
}

template <typename T> __host__ __device__ constexpr int row_threads(int logn)
{
    return rows_per_block<T>(logn) * ((1 << logn) >> log_elems<T>(logn));
}

// Registers: 64 a thread in FP32 (1024 threads per SM; 768 take 101 us for H at 2048, where 1024 take 95), 128 in FP64.
template <typename T> constexpr int row_blocks(int logn)
{
    return (sizeof(T) == 4 ? 1024 : 512) / (row_threads<T>(logn) < 128 ? 128 : row_threads<T>(logn));
}

// rows_per_block rows of one RHS per block, n/E threads a row.  MODE
//   0: ×D(k1 = column, k2 = row), inverse FFT along the row
//   1: inverse FFT, ×Wt[row][y], forward FFT (the transposed middle of H)
//   2: forward FFT, then ×conj(D(k1 = column, k2 = row)) × scale + λ x
//   3: inverse FFT, × scale
//   4: forward FFT
template <typename T, int MODE, int LOGN>
__global__ void __launch_bounds__(row_threads<T>(LOGN), row_blocks<T>(LOGN)) k_rows(Args<T> a)
{
    using C = cx_t<T>;
    using F = Row<T, LOGN>;
    constexpr int n = F::N, tn = F::TN, E = F::E, rpb = rows_per_block<T>(LOGN);
    if (a.skip && *a.skip) return;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int lt = threadIdx.x / tn, t = threadIdx.x % tn;
    const int row = blockIdx.x * rpb + lt;
    C *buf = reinterpret_cast<C *>(smem_raw) + lt * slots(n);
    const size_t base = ((size_t)blockIdx.y * n + row) * n + t;
    constexpr bool fwd_only = MODE == 2 || MODE == 4;
    constexpr int RI = fwd_only ? E : F::R1;                          // first pass
    constexpr int RO = MODE == 0 || MODE == 3 ? E : F::R1;            // last pass
    const T ft = (T)t, fr = (T)(row < n / 2 ? row : row - n);          // frequencies; n/2 is a multiple of tn
    auto fcol = [&](int off) { return ft + (T)(off < n / 2 ? off : off - n); };
    C v[E];
    const C *in = a.in + base;
#pragma unroll
    for (int i = 0; i < E; i++) {
        const int off = F::template place<RI>(i);
        v[i] = in[off];
        if (MODE == 0) v[i] = cmul(ks<T>(fcol(off), fr), v[i]);
    }
    if (!fwd_only) F::backward(v, buf, t, a.wb);
    if (MODE == 1) {
        const T *wt = a.Wt + (size_t)row * n + t;
#pragma unroll
        for (int i = 0; i < E; i++) {
            const T wy = wt[F::template place<E>(i)];
            v[i].x *= wy;
            v[i].y *= wy;
        }
    }
    if (fwd_only || MODE == 1) F::forward(v, buf, t, a.wf);
    if (MODE == 3) {
#pragma unroll
        for (int i = 0; i < E; i++) {
            v[i].x *= a.scale;
            v[i].y *= a.scale;
        }
    }
    if (MODE == 2) {
#pragma unroll
        for (int i = 0; i < E; i++) {
            const int off = F::template place<RO>(i);
            const C d = ks<T>(fcol(off), fr);
            v[i] = cmul(C{d.x, -d.y}, v[i]);
            v[i].x *= a.scale;
            v[i].y *= a.scale;
            if (a.xreg) {
                const C xr = a.xreg[base + off];
                v[i].x = fma(a.lam, xr.x, v[i].x);
                v[i].y = fma(a.lam, xr.y, v[i].y);
            }
        }
    }
    if (MODE == 2 || !a.tr) {
        C *out = a.out + base;
#pragma unroll
        for (int i = 0; i < E; i++) out[F::template place<RO>(i)] = v[i];
    } else if constexpr (rpb * sizeof(C) >= 16) {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < E; i++) buf[F::at(t, F::template place<RO>(i))] = v[i];
        __syncthreads();
        constexpr int RC = 16 / sizeof(C);   // rows in a 16-byte store
        struct alignas(16) Chunk { C c[RC]; };
        constexpr int nc = rpb / RC;         // stores side by side in a column
        const int k = threadIdx.x / nc, r = (threadIdx.x % nc) * RC;
        const C *src = reinterpret_cast<const C *>(smem_raw) + r * slots(n);
        C *dst = a.out + ((size_t)blockIdx.y * n + k) * n + blockIdx.x * rpb + r;
#pragma unroll
        for (int i = 0; i < E / RC; i++) {
            Chunk o;
#pragma unroll
            for (int q = 0; q < RC; q++) o.c[q] = src[q * slots(n) + F::at(k, i * tn * RC)];
            *reinterpret_cast<Chunk *>(dst + (size_t)i * (tn * RC) * n) = o;
        }
    }
}

// out[r][j][i] = in[r][i][j] in 32 x 32 tiles
template <typename T>
__global__ void k_transpose(int n, const cx_t<T> *__restrict__ in, cx_t<T> *__restrict__ out, const int *skip)
{
    if (skip && *skip) return;
    __shared__ cx_t<T> tile[32][33];
    const size_t off = (size_t)blockIdx.z * n * n;
    const int x0 = blockIdx.x * 32, y0 = blockIdx.y * 32;
    for (int j = threadIdx.y; j < 32; j += blockDim.y) {
        const int y = y0 + j, x = x0 + threadIdx.x;
        if (y < n && x < n) tile[j][threadIdx.x] = in[off + (size_t)y * n + x];
    }
    __syncthreads();
    for (int j = threadIdx.y; j < 32; j += blockDim.y) {
        const int y = x0 + j, x = y0 + threadIdx.x;
        if (y < n && x < n) out[off + (size_t)y * n + x] = tile[threadIdx.x][j];
    }
}

// complex [R][n²] <-> maps [R][2][n²] (γ1 = real part, γ2 = imaginary part), optional ×W
template <typename T>
__global__ void k_split(long long npix, int R, const cx_t<T> *__restrict__ z, const T *__restrict__ W, T *__restrict__ map)
{
    const long long tot = (long long)R * npix;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < tot; i += (long long)gridDim.x * blockDim.x) {
        const long long r = i / npix, pix = i - r * npix;
        const cx_t<T> v = z[i];
        const T wv = W ? W[pix] : T(1);
        map[(2 * r) * npix + pix] = wv * v.x;
        map[(2 * r + 1) * npix + pix] = wv * v.y;
    }
}

template <typename T>
__global__ void k_join(long long npix, int R, const T *__restrict__ map, const T *__restrict__ W, cx_t<T> *__restrict__ z)
{
    const long long tot = (long long)R * npix;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < tot; i += (long long)gridDim.x * blockDim.x) {
        const long long r = i / npix, pix = i - r * npix;
        const T wv = W ? W[pix] : T(1);
        z[i] = cx_t<T>{wv * map[(2 * r) * npix + pix], wv * map[(2 * r + 1) * npix + pix]};
    }
}

// per-device statistics of N^-1 and the weight tables
__global__ void k_weights(int n, const double *ninv, double *W64, float *W32, double *Wt64, float *Wt32,
                          double *stats)
{
    const long long npix = (long long)n * n;
    double s = 0, c = 0, bad = 0;
    const double scale = 1.0 / (double)npix;
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < npix; i += (long long)gridDim.x * blockDim.x) {
        const double v = ninv[i];
        const bool ok = isfinite(v) && v >= 0;
        const double w = (ok && v > 0) ? v : 0.0;
        W64[i] = w;
        W32[i] = (float)w;
        const long long y = i / n, x = i - y * n;
        Wt64[x * n + y] = w * scale;
        Wt32[x * n + y] = (float)(w * scale);
        if (!ok) bad += 1;
        if (ok && v > 0) {
            s += v;
            c += 1;
        }
    }
    __shared__ double sh[3][256];
    sh[0][threadIdx.x] = s;
    sh[1][threadIdx.x] = c;
    sh[2][threadIdx.x] = bad;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o)
            for (int q = 0; q < 3; q++) sh[q][threadIdx.x] += sh[q][threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0)
        for (int q = 0; q < 3; q++) atomicAdd(&stats[q], sh[q][0]);
}

// twiddles of one pass: w[(q - 1) Ns + k] = e^{-2πi qk/(Ns R)}, 1 <= q < R, k < Ns
template <typename T>
__global__ void k_twiddles(int Ns, int R, cx_t<T> *w)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < (R - 1) * Ns) {
        const int q = 1 + i / Ns, k = i % Ns;
        double s, c;
        sincospi(-2.0 * (double)(q * k) / (double)(Ns * R), &s, &c);
        w[i] = cx_t<T>{(T)c, (T)s};
    }
}

// the passes' twiddles in order: of the backward transform (R0, E, E, ..) from 0, of the forward one (E, .., R0) from n
template <typename T>
static void build_twiddles(int logn, cx_t<T> *w)
{
    const int n = 1 << logn, le = log_elems<T>(logn), E = 1 << le, r0 = 1 << (logn % le);
    for (int dir = 0; dir < 2; dir++) {
        cx_t<T> *at = w + dir * n;
        auto pass = [&](int Ns, int R) {
            if (Ns == 1 || R == 1) return;   // no twiddles
            k_twiddles<T><<<((R - 1) * Ns + 255) / 256, 256>>>(Ns, R, at);
            at += (R - 1) * Ns;
        };
        for (int Ns = dir == 0 ? r0 : 1; Ns < (dir == 0 ? n : n / r0); Ns *= E) pass(Ns, E);
        if (dir == 1) pass(n / r0, r0);
    }
}

template <typename T> const cx_t<T> *twiddles(akra_plan p);
template <> const double2 *twiddles<double>(akra_plan p) { return p->d_ftw64; }
template <> const float2 *twiddles<float>(akra_plan p) { return p->d_ftw32; }
template <typename T> const T *wt(akra_plan p);
template <> const double *wt<double>(akra_plan p) { return p->d_fWt64; }
template <> const float *wt<float>(akra_plan p) { return p->d_fWt32; }
template <typename T> const T *wmap(akra_plan p);
template <> const double *wmap<double>(akra_plan p) { return p->d_W64; }
template <> const float *wmap<float>(akra_plan p) { return p->d_W32; }

template <typename T, int MODE, int LOGN>
static void launch_rows(const Args<T> &a, int R, cudaStream_t st)
{
    constexpr int n = 1 << LOGN, rpb = rows_per_block<T>(LOGN);
    k_rows<T, MODE, LOGN><<<dim3(n / rpb, R), row_threads<T>(LOGN), rpb * slots(n) * sizeof(cx_t<T>), st>>>(a);
}

template <typename T, int MODE>
static akra_status rows(akra_plan p, const void *in, void *out, bool tr, int R, const void *xreg, double lam,
                        double scale, cudaStream_t st)
{
    Args<T> a{};
    a.tr = tr;
    a.wb = twiddles<T>(p);
    a.wf = a.wb + p->nside;
    a.in = (const cx_t<T> *)in;
    a.out = (cx_t<T> *)out;
    a.Wt = wt<T>(p);
    a.xreg = (const cx_t<T> *)xreg;
    a.lam = (T)lam;
    a.scale = (T)scale;
    a.skip = p->cur_skip;
    switch (p->flat_logn) {
    case 4: launch_rows<T, MODE, 4>(a, R, st); break;
    case 5: launch_rows<T, MODE, 5>(a, R, st); break;
    case 6: launch_rows<T, MODE, 6>(a, R, st); break;
    case 7: launch_rows<T, MODE, 7>(a, R, st); break;
    case 8: launch_rows<T, MODE, 8>(a, R, st); break;
    case 9: launch_rows<T, MODE, 9>(a, R, st); break;
    case 10: launch_rows<T, MODE, 10>(a, R, st); break;
    case 11: launch_rows<T, MODE, 11>(a, R, st); break;
    case 12: launch_rows<T, MODE, 12>(a, R, st); break;
    default: launch_rows<T, MODE, 13>(a, R, st); break;
    }
    AKRA_CUDA_TRY(cudaGetLastError());
    p->launches++;
    return AKRA_OK;
}

template <typename T>
static akra_status transpose(akra_plan p, const void *in, void *out, int R, cudaStream_t st)
{
    const int n = p->nside, g = (n + 31) / 32;
    k_transpose<T><<<dim3(g, g, R), dim3(32, 8), 0, st>>>(n, (const cx_t<T> *)in, (cx_t<T> *)out, p->cur_skip);
    AKRA_CUDA_TRY(cudaGetLastError());
    p->launches++;
    return AKRA_OK;
}

// a pass whose result is wanted transposed; tmp (as large) is used where the store does not transpose
template <typename T, int MODE>
static akra_status rows_t(akra_plan p, const void *in, void *out, void *tmp, int R, double scale, cudaStream_t st)
{
    if (fused_transpose(p->nside)) return rows<T, MODE>(p, in, out, true, R, nullptr, 0.0, scale, st);
    AKRA_TRY((rows<T, MODE>(p, in, tmp, false, R, nullptr, 0.0, scale, st)));
    return transpose<T>(p, tmp, out, R, st);
}

template <typename T>
static akra_status buffers(akra_plan p, int R, cx_t<T> **b1, cx_t<T> **b2)
{
    const size_t v = (size_t)R * p->npix;
    AKRA_TRY(ws_reserve(p, p->phi, 2 * v * sizeof(cx_t<T>)));
    *b1 = (cx_t<T> *)p->phi.ptr;
    *b2 = *b1 + v;
    return AKRA_OK;
}

// the shared-memory opt-in of the row kernels that take more than 48 KB (at plan creation, never inside a capture)
template <typename T, int MODE, int LOGN>
static cudaError_t prepare_one()
{
    constexpr int n = 1 << LOGN, bytes = rows_per_block<T>(LOGN) * slots(n) * (int)sizeof(cx_t<T>);
    if (bytes <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(k_rows<T, MODE, LOGN>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}
template <typename T, int MODE> static cudaError_t prepare_mode()
{
    cudaError_t e = prepare_one<T, MODE, 11>();
    if (e == cudaSuccess) e = prepare_one<T, MODE, 12>();
    if (e == cudaSuccess) e = prepare_one<T, MODE, 13>();
    return e;
}
template <typename T> static cudaError_t prepare_type()
{
    cudaError_t e = prepare_mode<T, 0>();
    if (e == cudaSuccess) e = prepare_mode<T, 1>();
    if (e == cudaSuccess) e = prepare_mode<T, 2>();
    if (e == cudaSuccess) e = prepare_mode<T, 3>();
    if (e == cudaSuccess) e = prepare_mode<T, 4>();
    return e;
}
static cudaError_t rows_prepare()
{
    const cudaError_t e = prepare_type<float>();
    return e == cudaSuccess ? prepare_type<double>() : e;
}

}  // namespace flat

template <typename T>
akra_status flat_op_A(akra_plan p, const void *x, void *map, bool weighted, int R, cudaStream_t st)
{
    cx_t<T> *b1, *b2;
    AKRA_TRY(flat::buffers<T>(p, R, &b1, &b2));
    const double s = 1.0 / (double)p->nside;
    AKRA_TRY((flat::rows_t<T, 0>(p, x, b2, b1, R, 1.0, st)));   // ×D, inverse along k1; [x][k2]
    // inverse along k2, × 1/n; [y][x].  In place where the store transposes separately
    AKRA_TRY((flat::rows_t<T, 3>(p, b2, b1, b2, R, s, st)));
    flat::k_split<T><<<1216, 256, 0, st>>>(p->npix, R, b1, weighted ? flat::wmap<T>(p) : nullptr, (T *)map);
    AKRA_CUDA_TRY(cudaGetLastError());
    p->launches++;
    return AKRA_OK;
}

template <typename T>
akra_status flat_op_At(akra_plan p, const void *map, void *x, bool weighted, int R, cudaStream_t st)
{
    cx_t<T> *b1, *b2;
    AKRA_TRY(flat::buffers<T>(p, R, &b1, &b2));
    flat::k_join<T><<<1216, 256, 0, st>>>(p->npix, R, (const T *)map, weighted ? flat::wmap<T>(p) : nullptr, b1);
    AKRA_CUDA_TRY(cudaGetLastError());
    p->launches++;
    AKRA_TRY(flat::transpose<T>(p, b1, b2, R, st));                            // [x][y]
    AKRA_TRY((flat::rows_t<T, 4>(p, b2, b1, b2, R, 1.0, st)));                 // forward along y; [k2][x]
    return flat::rows<T, 2>(p, b1, x, false, R, nullptr, 0.0, 1.0 / (double)p->nside, st);   // along x, ×conj D / n
}

template <typename T>
akra_status flat_op_H(akra_plan p, const void *x, void *y, int R, cudaStream_t st)
{
    cx_t<T> *b1, *b2;
    AKRA_TRY(flat::buffers<T>(p, R, &b1, &b2));
    AKRA_TRY((flat::rows_t<T, 0>(p, x, b2, b1, R, 1.0, st)));        // ×D, inverse along k1; [x][k2]
    AKRA_TRY((flat::rows_t<T, 1>(p, b2, b1, b2, R, 1.0, st)));       // along k2: F^-1, ×W/n², F; [k2][x]
    return flat::rows<T, 2>(p, b1, y, false, R, x, p->lambda_eff, 1.0, st);   // along x, ×conj D, + λ x
}

template akra_status flat_op_A<float>(akra_plan, const void *, void *, bool, int, cudaStream_t);
template akra_status flat_op_A<double>(akra_plan, const void *, void *, bool, int, cudaStream_t);
template akra_status flat_op_At<float>(akra_plan, const void *, void *, bool, int, cudaStream_t);
template akra_status flat_op_At<double>(akra_plan, const void *, void *, bool, int, cudaStream_t);
template akra_status flat_op_H<float>(akra_plan, const void *, void *, int, cudaStream_t);
template akra_status flat_op_H<double>(akra_plan, const void *, void *, int, cudaStream_t);

akra_status flat_set_weights(akra_plan p, const double *d_ninv, double lambda, cudaStream_t st)
{
    double *d_stats = nullptr;
    if (cudaMalloc(&d_stats, 3 * sizeof(double)) != cudaSuccess) {
        cudaGetLastError();
        set_error("akra_plan_set_weights: allocation failed");
        return AKRA_ENOMEM;
    }
    double h[3] = {0, 0, 0};
    p->has_weights = false;   // until the new ones are complete
    p->ws_gen++;   // captured CG iterations hold the previous λ_eff
    cudaError_t e = cudaMemsetAsync(d_stats, 0, 3 * sizeof(double), st);
    if (e == cudaSuccess) {
        flat::k_weights<<<1216, 256, 0, st>>>(p->nside, d_ninv, p->d_W64, p->d_W32, p->d_fWt64, p->d_fWt32, d_stats);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(h, d_stats, sizeof(h), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    cudaFree(d_stats);
    AKRA_CUDA_TRY(e);
    if (h[2] > 0) {
        set_error("akra_plan_set_weights: %.0f negative or non-finite N^-1 entries", h[2]);
        return AKRA_EINVAL;
    }
    p->lambda = lambda;
    p->omega = 1.0;
    p->lambda_eff = h[1] > 0 ? lambda * h[0] / h[1] : 0.0;
    p->precond = 1.0 / (h[0] / (double)p->npix + p->lambda_eff);
    if (!std::isfinite(p->precond)) p->precond = 1.0;
    p->has_weights = true;
    return AKRA_OK;
}

}  // namespace akra

using namespace akra;

extern "C" akra_status akra_flat_plan_create(int n, akra_plan *out)
{
    if (!out) {
        set_error("akra_flat_plan_create: out is NULL");
        return AKRA_EINVAL;
    }
    *out = nullptr;
    if (n < 16 || n > flat::kMaxN || (n & (n - 1))) {
        set_error("akra_flat_plan_create: n = %d must be a power of two in [16, %d]", n, flat::kMaxN);
        return AKRA_EINVAL;
    }
    akra_plan p = new (std::nothrow) akra_plan_s();
    if (!p) {
        set_error("akra_flat_plan_create: host allocation failed");
        return AKRA_ENOMEM;
    }
    p->kind = 1;
    p->nside = n;
    p->lmax = -1;
    p->npix = (long long)n * n;
    p->ntri = p->npix / 2;
    int lg = 0;
    while ((1 << lg) < n) lg++;
    p->flat_logn = lg;
    cudaGetDevice(&p->device);
    const size_t np = (size_t)p->npix;
    auto fail = [&](const char *what) {
        cudaGetLastError();
        set_error("akra_flat_plan_create: %s", what);
        akra_plan_destroy(p);
        return AKRA_ENOMEM;
    };
    if (cudaMalloc(&p->d_ftw64, sizeof(double2) * 2 * n) != cudaSuccess ||
        cudaMalloc(&p->d_ftw32, sizeof(float2) * 2 * n) != cudaSuccess ||
        cudaMalloc(&p->d_W64, sizeof(double) * np) != cudaSuccess ||
        cudaMalloc(&p->d_W32, sizeof(float) * np) != cudaSuccess ||
        cudaMalloc(&p->d_fWt64, sizeof(double) * np) != cudaSuccess ||
        cudaMalloc(&p->d_fWt32, sizeof(float) * np) != cudaSuccess)
        return fail("table allocation failed");
    p->bytes_tables = (sizeof(double2) + sizeof(float2)) * 2 * n + 2 * (sizeof(double) + sizeof(float)) * np;
    flat::build_twiddles<double>(lg, p->d_ftw64);
    flat::build_twiddles<float>(lg, p->d_ftw32);
    cudaError_t e = cudaGetLastError();
    // row kernels: shared memory of the largest block, set once for every plan
    if (e == cudaSuccess) e = flat::rows_prepare();
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&p->stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p->ev_a, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&p->ev_b, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        set_error("akra_flat_plan_create: %s", cudaGetErrorString(e));
        akra_plan_destroy(p);
        return AKRA_ECUDA;
    }
    *out = p;
    return AKRA_OK;
}
