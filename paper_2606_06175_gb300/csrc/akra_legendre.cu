// akra_legendre.cu -- spin-2 Legendre stages of the synthesis (Eq. 1) and of its exact
// transpose, fused with the KS factor (Eq. 3) and the E/B <-> spin ±2 recombination (Eq. 2).
//
// Work unit: one m and one ring pair (north ring θ, south ring π-θ; the equator ring alone).
// Two recurrences run in ℓ, one per spin s = ±2 (x = cos θ, A_l, B_l the normalised
// Wigner-d coefficients):
//     sλ_{l+1} = (A_l x + s A_l m/(l(l+1))) sλ_l - A_l B_l sλ_{l-1},
// carried in monic form μ_l = sλ_l / σ_l (σ from the plan's table, between 0.17 and 1), so a
// step is μ_{l+1} = (A'_l x ± c'_l) μ_l - μ_{l-1}: 2 FMA per spin; σ_l is folded into the staged
// alm (synthesis) and into the per-l partial sums (adjoint).
// (kept separate: near the poles one spin is O(1) and the other tiny, and any mixed
// combination would leak the large one's rounding into the small one).  The mirror ring
// follows from  sλ_lm(π-θ) = (-1)^{l+m} (-s)λ_lm(θ), so one pair of recurrences feeds both
// rings through even/odd (l+m) accumulators.  Seeds at l0 = max(m,2) are formed in FP64 in
// log2 form; the recurrence carries a per-unit exponent index e (value = v 2^(Q e)) and
// contributes only once e == 0.
#include <type_traits>

#include "akra_legendre_impl.cuh"

namespace akra {

// ---------------------------------------------------------------------------
// epilogue: sum chunk partials, apply f_l/2 and the spin ±2 -> E/B recombination
//   E = (f/2) E-part,  B = (-i f/2) B-part,  optional + λ x
// ---------------------------------------------------------------------------
template <typename T>
__global__ void k_adj_epilogue(int L, long long ntri, int nchunks, int R,
                               const T *__restrict__ partial, const T *__restrict__ fl,
                               const cx_t<T> *__restrict__ xreg, T lam, cx_t<T> *__restrict__ out,
                               const int *__restrict__ skip, int fields)
{
    if (skip && *skip) return;
    using C2 = cx_t<T>;
    const int m = blockIdx.x, r = blockIdx.y;
    const long long mbase = (long long)m * (2 * L + 1 - m) / 2;
    const long long qbound = (long long)nchunks * R * ntri * 4;   // extent of the partial sums
    const long long abound = (long long)R * 2 * ntri;             // extent of x and out
    (void)qbound;
    (void)abound;
    for (int l = m + threadIdx.x; l <= L; l += blockDim.x) {
        const long long idx = mbase + l;
        T a0 = 0, a1 = 0, a2 = 0, a3 = 0;
        if (l >= 2) {
            for (int c = 0; c < nchunks; c++) {
                const long long pq = (((size_t)c * R + r) * ntri + idx) * 4;
                a0 += partial[AKRA_IX(pq + 0, qbound, kDbgPartialRead)];
                a1 += partial[AKRA_IX(pq + 1, qbound, kDbgPartialRead)];
                a2 += partial[AKRA_IX(pq + 2, qbound, kDbgPartialRead)];
                a3 += partial[AKRA_IX(pq + 3, qbound, kDbgPartialRead)];
            }
        }
        const T h = (fl ? fl[AKRA_IX(l, L + 1, kDbgKsFactor)] : T(-1)) * T(0.5);
        C2 E{h * a0, h * a1};
        C2 B{h * a3, -h * a2};
        if (xreg) {
            C2 xe = xreg[AKRA_IX(((size_t)r * 2 + 0) * ntri + idx, abound, kDbgAlm)];
            C2 xb = xreg[AKRA_IX(((size_t)r * 2 + 1) * ntri + idx, abound, kDbgAlm)];
            E.x += lam * xe.x;
            E.y += lam * xe.y;
            B.x += lam * xb.x;
            B.y += lam * xb.y;
        }
        if (m == 0) E.y = B.y = 0;
        // a field outside the solve's field set is held at zero (its block row is dropped)
        if (!(fields & 1)) E = C2{0, 0};
        if (!(fields & 2)) B = C2{0, 0};
        out[AKRA_IX(((size_t)r * 2 + 0) * ntri + idx, abound, kDbgAlmOut)] = E;
        out[AKRA_IX(((size_t)r * 2 + 1) * ntri + idx, abound, kDbgAlmOut)] = B;
    }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <typename T> const v4_t<T> *coef_ptr(akra_plan p);
template <> const float4 *coef_ptr<float>(akra_plan p) { return p->d_coef32; }
template <> const double4_32a *coef_ptr<double>(akra_plan p) { return p->d_coef64; }
template <typename T> const v4_t<T> *seed_ptr(akra_plan p);
template <> const float4 *seed_ptr<float>(akra_plan p) { return p->d_seed32; }
template <> const double4_32a *seed_ptr<double>(akra_plan p) { return p->d_seed64; }
template <typename T> static const int2 *start_ptr(akra_plan p);
template <> const int2 *start_ptr<float>(akra_plan p) { return p->d_start32; }
template <> const int2 *start_ptr<double>(akra_plan p) { return p->d_start64; }
template <typename T> const T *D_ptr(akra_plan p);
template <> const float *D_ptr<float>(akra_plan p) { return p->d_D32; }
template <> const double *D_ptr<double>(akra_plan p) { return p->d_D64; }

template <typename T>
LegArgs<T> leg_args(akra_plan p, const LegShape &s, LegMode mode, const int *units, int nunits, int R)
{
    LegArgs<T> a{};
    a.L = p->lmax;
    a.nring = p->nring;
    a.nchunks = (nunits + s.NT * s.P - 1) / (s.NT * s.P);
    a.nunits = nunits;
    a.nunit_all = p->nunit;
    a.R = R;
    a.ntri = p->ntri;
    a.units = units;
    a.uinfo = p->d_units;
    a.coef = coef_ptr<T>(p);
    a.seeds = seed_ptr<T>(p);
    a.dseeds = p->d_dseed32;
    a.start = start_ptr<T>(p);
    a.fl = mode == LegMode::KS ? D_ptr<T>(p) : nullptr;
    a.ring_active = units == p->d_all_units ? nullptr : p->d_ring_active;
    a.skip = p->cur_skip;
    a.err = p->d_tc_err;
    a.bpre = (const float *)p->bpre.ptr;
    a.tc_tilebase = p->d_tc_tilebase;
    a.tc_groups = s.TC > 0 ? (R + s.TC - 1) / s.TC : 0;
    a.tc_tiles = p->tc_tiles;
    const BlkTables &bt = blk_tables(p, units);
    a.blk_rows = bt.rows;
    a.blk_info = bt.info;
    a.blk_vtab = bt.vtab;
    a.blk_nrows = bt.nrows;
    a.blk_chunks = bt.nchunks;
    return a;
}

template <typename T, int P, int RG, int NT>
static void launch_synth(akra_plan p, LegMode mode, const void *alm, void *phi, int R,
                         const int *units, int nunits, cudaStream_t st)
{
    LegArgs<T> a = leg_args<T>(p, LegShape{P, NT, RG}, mode, units, nunits, R);
    a.alm = (const cx_t<T> *)alm;
    a.phi = (cx_t<T> *)phi;
    dim3 grid((unsigned)(p->lmax + 1) * a.nchunks, (R + RG - 1) / RG);
    k_leg_synth<T, P, RG, NT><<<grid, NT, 0, st>>>(a);
}

template <typename T, int P, int RG, int NT, int ONE = 0>
static int launch_adjoint(akra_plan p, const void *phi, void *partial, int R, const int *units,
                          int nunits, cudaStream_t st)
{
    LegArgs<T> a = leg_args<T>(p, LegShape{P, NT, RG}, LegMode::Synth, units, nunits, R);
    a.phi_in = (const cx_t<T> *)phi;
    a.partial = (T *)partial;
    dim3 grid((unsigned)(p->lmax + 1) * a.nchunks, (R + RG - 1) / RG);
    k_leg_adjoint<T, P, RG, NT, ONE><<<grid, NT, 0, st>>>(a);
    return a.nchunks;
}

// Whether the block-jump kernels take a list's ring pairs (FP32, unless the plan's shape rules them out).
// They treat every ring by itself, the direct kernels share a pair's recurrence between its two rings, so
// the line lies where most of the work is on pairs that need one ring.  One RHS, direct -> block-jump:
// footprints of one hemisphere at (Nside, lmax) = (64, 128) synthesis 13.6 -> 10.9 us, adjoint 23.2 -> 14.3;
// (512, 1024) 181 -> 125, 311 -> 223; (2048, 4096) 8.19 -> 4.16 ms, 10.31 -> 8.84 ms.  Full sky, whole
// transforms: (1024, 2048) 2.08 -> 2.35 ms, 3.83 -> 4.66; (2048, 4096) 13.7 -> 12.1 ms, 19.7 -> 24.9: only
// the synthesis, and only from lmax 4096 on.
bool blk_pays(akra_plan p, const int *units, bool adjoint)
{
    if (p->lmax < kBlkMinLmax) return false;
    if (units != p->d_all_units && p->mostly_one_ring) return true;
    return !adjoint && p->lmax >= 4096;
}

// Synthesis of R right-hand sides on a list of blk_pays.  A block-jump block takes one right-hand side, a direct
// block of shape (1, 4) four that share the recurrence, so from four on the direct kernel is the faster one where its
// slots are full and lmax is low.  Time of (1, 4) over block jumps at full slots (R = 4, 8) on DES-like footprints: 256 / 512
// 0.66, 300 / 600 0.78, 512 / 1024 1.01, 1024 / 1024 1.04, 1024 / 2048 1.25; caps 0.63, 0.63, 0.84, 0.85, 1.00; about 0.62 + 0.3 lmax / 1000
// between them, more by the empty slots (R = 5 at 400 / 800: 1.18 to 1.32).  One to three right-hand sides: 1.18 to 1.97 with
// one, 0.9 to 1.35 with two or three (below 1 at a few sizes of lmax 250 to 800 only, and the block jumps are the
// more accurate ones).  All rings, 2048 / 4096: R = 1 1.14, 2 1.08, 3 1.16, 4 0.94, 6 1.09.
static bool jump_synth(akra_plan p, const LegShape &s, const int *units, int R)
{
    if (!s.BS || !blk_pays(p, units, false)) return false;
    if (s.BS == 2 || R < 4) return true;
    const double pad = (R + 3) / 4 * 4 / (double)R;
    return units == p->d_all_units ? pad >= 1.06 : pad * (0.62 + 0.3e-3 * p->lmax) >= 0.95;
}

// The adjoint's shape on a list of blk_pays: whether the block jumps take it (BA 2 or 0), for all of R, and the direct
// shape where they do not.  The block jumps have the smaller errors (A^T by 1.1 to 1.6 times, growing with lmax), so they
// stay wherever they are about as fast as the direct kernel they replaced at five pairs a thread.  They repeat for
// every right-hand side what a direct block does once, compute the rings that pad a chunk, and pay a set-up, a slow first phase and
// a padded last tile per block.  Whole A^T in us, that direct kernel, block jumps, this rule:
//   lmax below Nside, many chunks: 1500 / 1024 cap 929, 1047, 910; 2048 / 1024 cap 1177, 1307, 1122, DES-like 1336, 1417, 1256
//   several right-hand sides at low lmax (errors differ by a quarter at most there): 64 / 128 strip, R = 5 26, 36, 25; 128 / 256
//          strip, R = 3 39, 45, 37; 200 / 250 DES-like, R = 5 154, 142, 112
//   badly filled chunks: 400 / 800 strip R = 3 246, 325, 230, R = 8 632, 829, 536, R = 1 98, 119, 110 (a list that needs one
//          side alone, for which the direct kernel does half the work); DES-like, 555 pairs in three chunks, R = 5 841, 884, 793
//   the rest: DES-like, R = 5: 600 / 700 1291, 1225; 600 / 1200 2699, 2356; R = 1: 400 / 800 205, 191; 1024 / 1024 577, 579
// (the strip: -0.45 < cos(theta) < 0).  The direct shape is the one with the fewest pairs of padding: a single chunk up to 640 pairs,
// chunks of 384 or 512 beyond (adjoint alone, R = 5: 400 / 800, 555 pairs (5, 1) 648, (3, 1) 612, (4, 1) 728; 200 / 400, 278 pairs (3, 1) 113,
// (2, 1) 139, (5, 1) 181).
LegShape adjoint_shape(akra_plan p, const LegShape &s, const int *units, int nunits, int R)
{
    LegShape t = s;
    if (s.BA != 1 || nunits <= 0 || !blk_pays(p, units, true)) return t;
    const BlkTables &bt = blk_tables(p, units);
    const bool badly_filled = bt.nrows < 0.8 * 256 * bt.nchunks && bt.nchunks >= (p->one_side ? 2 : R >= 3 ? 3 : kNeverLive);
    bool direct = bt.nchunks >= 3 && p->lmax < p->nside;
    if (R >= 3 || (R == 2 && bt.nchunks >= 2)) direct |= p->lmax < 350 || badly_filled;
    if (R == 1) direct |= badly_filled && p->nside * (double)p->lmax >= 2.2e5;
    t.BA = direct ? 0 : 2;
    if (!direct) return t;
    const int c = (nunits + 127) / 128;
    t.PA = c <= 5 ? c : (c + 3) / 4 * 4 <= (c + 2) / 3 * 3 ? 4 : 3;
    t.RGA = 1;
    return t;
}

// The tensor-core group that a synthesis of shape s runs with (0: none).  Groups of 4 and 8 RHS leave the tensor-core
// GEMM's columns thin: on one-ring lists what the default runs there is faster.  Synthesis of 8 RHS in us, groups of
// 4, of 8, the default: (128, 256) 65, 55, 34; (300, 600) 465, 357, 228 (direct); (1024, 2048) 12700, 9160, 5400 (block
// jumps).  Larger groups stay: 16 RHS of 16 10.3 ms against 10.8 at (1024, 2048).
int synth_tc_group(akra_plan p, const LegShape &s, const int *units)
{
    return s.BS && s.TC <= 8 && blk_pays(p, units, true) ? 0 : s.TC;
}

// shape dispatch: (P, RG) combinations compiled for each precision, NT = 128
template <typename T>
akra_status legendre_synth(akra_plan p, const LegShape &s, LegMode mode, const void *alm,
                           void *phi, int R, const int *units, int nunits, cudaStream_t st)
{
    if (nunits <= 0) return AKRA_OK;
    if constexpr (std::is_same<T, float>::value) {
        const int tcg = synth_tc_group(p, s, units);
        if (tcg > 0) return legendre_synth_tc(p, tcg, mode, alm, phi, R, units, nunits, st);
        if (jump_synth(p, s, units, R)) {
            // the polar ring pairs (the first of the list) keep the difference-form kernels
            const int npolar = blk_tables(p, units).npolar;
            LegShape sp = s;
            sp.BS = sp.TC = 0;
            AKRA_TRY(legendre_synth<T>(p, sp, mode, alm, phi, R, units, npolar, st));
            return legendre_synth_blk(p, mode, alm, phi, R, units, st);
        }
    }
#define AKRA_S(PP, RR)                                                                      \
    if (s.P == PP && s.RG == RR) {                                                          \
        launch_synth<T, PP, RR, 128>(p, mode, alm, phi, R, units, nunits, st);              \
        AKRA_CUDA_TRY(cudaGetLastError());                                                  \
        p->launches++;                                                                      \
        return AKRA_OK;                                                                     \
    }
    AKRA_S(1, 1) AKRA_S(2, 1) AKRA_S(4, 1) AKRA_S(1, 2) AKRA_S(2, 2) AKRA_S(1, 4)
    if constexpr (std::is_same<T, float>::value) { AKRA_S(3, 1) AKRA_S(5, 1) AKRA_S(6, 1) AKRA_S(8, 1) }
#undef AKRA_S
    set_error("no synthesis kernel for P=%d RG=%d", s.P, s.RG);
    return AKRA_EINVAL;
}

template <typename T>
akra_status legendre_adjoint(akra_plan p, const LegShape &s, const void *phi, void *partial,
                             int R, const int *units, int nunits, int *nchunks_out,
                             cudaStream_t st)
{
    *nchunks_out = 0;
    if (nunits <= 0) return AKRA_OK;
    const int pa = s.adjP();
    if constexpr (std::is_same<T, float>::value) {
        if (s.BA && blk_pays(p, units, true)) {
            // chunks of the block-jump kernel first, then those of the polar ring pairs (the first of the list)
            const BlkTables &t = blk_tables(p, units);
            LegShape sp = s;
            sp.BA = 0;
            int np = 0;
            AKRA_TRY(legendre_adjoint<T>(p, sp, phi, (T *)partial + (size_t)t.nchunks * R * p->ntri * 4, R, units,
                                         t.npolar, &np, st));
            *nchunks_out = t.nchunks + np;
            return legendre_adjoint_blk(p, phi, partial, R, units, *nchunks_out, st);
        }
    }
    {
        // the active ring pairs of a one-hemisphere footprint all need the same single ring: the
        // kernel compiled for that form alone (fewer registers); FP32 at 3-8 ring pairs per
        // thread, FP64 at 1, 2 and 4, one RHS per block
        const int one = (units != p->d_all_units && s.adjRG() == 1) ? p->one_side : 0;
#define AKRA_A1(PP)                                                                          \
        if (one && pa == PP) {                                                               \
            *nchunks_out = one == 1 ? launch_adjoint<T, PP, 1, 128, 1>(p, phi, partial, R, units, nunits, st) \
                                    : launch_adjoint<T, PP, 1, 128, 2>(p, phi, partial, R, units, nunits, st); \
            AKRA_CUDA_TRY(cudaGetLastError());                                               \
            p->launches++;                                                                   \
            return AKRA_OK;                                                                  \
        }
        if constexpr (std::is_same<T, float>::value) { AKRA_A1(3) AKRA_A1(4) AKRA_A1(5) AKRA_A1(6) AKRA_A1(8) }
        else { AKRA_A1(1) AKRA_A1(2) AKRA_A1(4) }
#undef AKRA_A1
    }
#define AKRA_A(PP, RR)                                                                      \
    if (pa == PP && s.adjRG() == RR) {                                                      \
        *nchunks_out = launch_adjoint<T, PP, RR, 128>(p, phi, partial, R, units, nunits, st); \
        AKRA_CUDA_TRY(cudaGetLastError());                                                  \
        p->launches++;                                                                      \
        return AKRA_OK;                                                                     \
    }
    AKRA_A(1, 1) AKRA_A(2, 1) AKRA_A(4, 1) AKRA_A(1, 2) AKRA_A(2, 2) AKRA_A(1, 4)
    if constexpr (std::is_same<T, float>::value) { AKRA_A(3, 1) AKRA_A(5, 1) AKRA_A(6, 1) AKRA_A(8, 1) }
#undef AKRA_A
    set_error("no adjoint kernel for P=%d RG=%d", pa, s.adjRG());
    return AKRA_EINVAL;
}

template <typename T>
akra_status adjoint_epilogue(akra_plan p, LegMode mode, const void *partial, int nchunks,
                             const void *x_reg, double lam, void *alm_out, int R, cudaStream_t st,
                             int fields)
{
    dim3 grid(p->lmax + 1, R);
    k_adj_epilogue<T><<<grid, 128, 0, st>>>(p->lmax, p->ntri, nchunks, R, (const T *)partial,
                                            mode == LegMode::KS ? D_ptr<T>(p) : nullptr,
                                            (const cx_t<T> *)x_reg, (T)lam, (cx_t<T> *)alm_out,
                                            p->cur_skip, fields);
    AKRA_CUDA_TRY(cudaGetLastError());
    p->launches++;
    return AKRA_OK;
}

// chunks of the adjoint (its partial sums are laid out per chunk)
int legendre_chunks(akra_plan p, const int *units, int nunits, const LegShape &s)
{
    const int per = s.NT * s.adjP();
    if (s.BA && nunits > 0 && blk_pays(p, units, true)) {
        const BlkTables &t = blk_tables(p, units);
        return t.nchunks + (t.npolar + per - 1) / per;
    }
    return (nunits + per - 1) / per;
}

// Right-hand sides whose partial sums are formed at a time.  Chunks of 256 rings have about twice the partial
// sums of the direct kernel's 640 pairs: 12 chunks against 5 on the DES-like footprint at Nside 2048 / lmax 4096, 1.6 GB
// per right-hand side against 0.67, 103 GB against 43 at 64.  They take no more than the direct kernel's, or 4 GB (where
// launches of a millisecond and more are split, which costs nothing that can be measured), so that a call that
// fits with the direct kernel fits with these.
int adjoint_rhs(akra_plan p, const int *units, int nunits, const LegShape &s, int R, size_t real_bytes)
{
    if (!s.BA || nunits <= 0 || !blk_pays(p, units, true)) return R;
    const size_t vec = (size_t)p->ntri * 4 * real_bytes;
    const size_t most = std::max((size_t)((nunits + 639) / 640) * R * vec, (size_t)4 << 30);
    const size_t fit = std::max<size_t>(most / (vec * legendre_chunks(p, units, nunits, s)), 1);
    if (fit >= (size_t)R) return R;
    const int groups = (int)((R + fit - 1) / fit);
    return (R + groups - 1) / groups;   // of even size
}

size_t partial_bytes(akra_plan p, const int *units, int nunits, const LegShape &shape, int R, size_t real_bytes)
{
    const LegShape s = adjoint_shape(p, shape, units, nunits, R);
    return (size_t)legendre_chunks(p, units, nunits, s) * adjoint_rhs(p, units, nunits, s, R, real_bytes) * p->ntri * 4 * real_bytes;
}

template LegArgs<float> leg_args<float>(akra_plan, const LegShape &, LegMode, const int *, int, int);
template LegArgs<double> leg_args<double>(akra_plan, const LegShape &, LegMode, const int *, int, int);
template akra_status legendre_synth<float>(akra_plan, const LegShape &, LegMode, const void *, void *,
                                           int, const int *, int, cudaStream_t);
template akra_status legendre_synth<double>(akra_plan, const LegShape &, LegMode, const void *,
                                            void *, int, const int *, int, cudaStream_t);
template akra_status legendre_adjoint<float>(akra_plan, const LegShape &, const void *, void *, int,
                                             const int *, int, int *, cudaStream_t);
template akra_status legendre_adjoint<double>(akra_plan, const LegShape &, const void *, void *, int,
                                              const int *, int, int *, cudaStream_t);
template akra_status adjoint_epilogue<float>(akra_plan, LegMode, const void *, int, const void *,
                                             double, void *, int, cudaStream_t, int);
template akra_status adjoint_epilogue<double>(akra_plan, LegMode, const void *, int, const void *,
                                              double, void *, int, cudaStream_t, int);

AKRA_DEBUG_COLLECTOR(legendre)

}  // namespace akra
