// akra_legendre_blk.cuh -- FP32 Legendre stages by blocks of 16 l-steps with the blocks' transfer
// polynomials interpolated on the tensor core.
//
// Over 16 steps from l the recurrence is linear in its state: ξ_{l+k}(x) = p_k(x) ξ_l + q_k(x) ξ_{l-1},
// p_k and q_k polynomials in x = cos θ of degree k and k - 1 that do not depend on the ring.  A polynomial
// of degree <= 15 is given exactly by its values at 16 nodes, so for a chunk of 256 rings (close in
// latitude) the recurrence runs once per node instead of once per ring:
//   * nodes: the FP32 recurrence of p, q at 16 Chebyshev nodes of the chunk's x-interval, for 8 blocks
//     (128 l-steps, a tile) at once -- the blocks do not depend on each other;
//   * rings: p and q at every ring are V · (node values), V[ring][node] the Lagrange basis at the ring's x
//     (one table per chunk), M = 128, K = 16 products on the tensor core;
//   * the ring's state then takes one 16-step jump with four products per spin.
// Synthesis: the sums Σ_k c_{l+k} ξ_{l+k} = (Σ c p_k) ξ_l + (Σ c q_k) ξ_{l-1} are interpolated the same
// way (the node threads accumulate Σ c p_k and Σ c q_k).  Adjoint: the rings' products ξ_l X, ξ_{l-1} X
// are contracted with V over the rings (a second tensor-core product, K = 256 rings), which gives 16 node
// moments per block, and the node recurrence started from the moments gives the 16 sums over the rings.
//
// Per (l, ring) step that needs one ring this leaves 16 tensor-core multiply-adds and about 2 FP32 ones where
// the direct recurrence has 8 FP32 ones.  Measured on the DES-like footprint, one RHS, direct -> this:
// Nside 2048 / lmax 4096 synthesis 8.19 -> 4.16 ms, adjoint 10.3 (9.7 in its best shape) -> 8.8 ms; 512 / 1024 0.181 ->
// 0.125 ms, 0.311 -> 0.223 ms.  Where they are not faster: akra_legendre.cu (jump_synth, adjoint_shape).  What
// bounds it: no unit is busy half of the time (FMA pipe 43 % in the synthesis, 29 % in the adjoint, tensor pipe 15 and 9 %);
// with TMEM for two blocks per SM a tile's way node threads -> product -> ring threads -> freed columns (the
// product's round trip alone is 600 cycles) is not fully hidden, and phase A is more than a quarter of the time
// (cycles a block at 2048 / 4096: synthesis 14.6k beside 13 tiles of 2.6k, adjoint 27.8k beside 13 of 4.8k).
//
// Precision: node values and V are split into two FP16 parts (22 bits), products head·head + head·rest +
// rest·head with FP32 accumulation; nodes are FP32 numbers and V is computed in FP64 from the rings' FP64 x,
// so the ring's x enters without FP32 rounding -- the direct recurrence's largest error, which grows with l.
// Relative error of H against FP64 at 512 / 1024: 9.3e-6 -> 7.4e-6; 2048 / 4096: 2.8e-5 -> 1.8e-5.
//
// Where a ring of the chunk is still before its turning point (l sin θ < m) p_k grows like e^{k κ} with κ
// varying over the chunk, and interpolation would lose bits; until the chunk's most polar ring is past it
// the rings run the direct recurrence (phase A; a tenth to a fifth of the steps).  Rings within 0.1 rad of a
// pole are left to the difference-form kernels (akra_legendre_impl.cuh).
#pragma once
#include <cuda_fp16.h>

#include "akra_legendre_impl.cuh"
#include "akra_tc.cuh"

namespace akra {

constexpr int BLK_RINGS = 256;   // rings per chunk: two MMA row tiles of 128
constexpr int BLK_NT = 128;      // ring threads, two rings each
constexpr int BLK_NN = 128;      // node threads
constexpr int BLK_K = 16;        // l-steps per block = nodes = MMA K
constexpr int BLK_NB = 8;        // blocks per tile
constexpr int BLK_TILE = BLK_K * BLK_NB;
constexpr int BLK_VBYTES = 16384;   // V of a chunk: 256 rows x 16 nodes, FP16 head and rest
constexpr int kBlkWaitLimit = 1 << 20;

// byte offset of V(row, node) of part h in a chunk's table: K-major A operand of the interpolation
// (lbo 128, sbo 512) and, read as MN-major, B operand of the moments (rows = part x node, sbo 128, lbo 512)
__host__ __device__ __forceinline__ int blk_voff(int row, int node, int h)
{
    return (row >> 3) * 512 + h * 256 + (node >> 3) * 128 + (row & 7) * 16 + (node & 7) * 2;
}

// ring (position in the chunk) of MMA row r = 128 k + thread: a warp owns 64 consecutive rings, its lanes
// ring 32 k + lane of them in row tile k
__host__ __device__ __forceinline__ int blk_ring_of_row(int r)
{
    return ((r & 127) >> 5) * 64 + (r >> 7) * 32 + (r & 31);
}

// node values of a tile, K-major B operand: column n, node k.  Strides padded so that the 32-bit stores of
// a warp (8 node pairs x 2 spins x 2 blocks) fall into 32 different banks.
constexpr int BLK_BLBO = 160, BLK_BSBO = 288;
__device__ __forceinline__ int blk_boff(int n, int kpair)
{
    return (n >> 3) * BLK_BSBO + (kpair >> 2) * BLK_BLBO + (n & 7) * 16 + (kpair & 3) * 4;
}

// staged values of step i of block b: {rA', rc'} (float2) and {c.re, c.im, ±d.re, ±d.im} (float4); a block's
// row is padded so that the blocks a warp reads fall into different banks
constexpr int BLK_CROW = BLK_K + 2;
__device__ __forceinline__ int blk_coff(int b, int i) { return b * BLK_CROW + i; }

// one row = one ring of the chunk
struct BlkRow {
    int ring, uid, gs, e;
    bool south;
    float x;
    float2 V, VO;   // (ξ+, ξ-) at the current l and at l - 1
    float4 seed;    // start state, loaded ahead
};

__device__ __forceinline__ void blk_row_init(const LegArgs<float> &a, int m, int chunk, int k, BlkRow &w)
{
    const int iu = chunk * BLK_RINGS + blk_ring_of_row(128 * k + threadIdx.x);
    w.ring = w.uid = -1;
    w.gs = kNeverLive;
    w.e = 0;
    w.south = false;
    w.x = 0.f;
    w.V = w.VO = make_float2(0.f, 0.f);
    if (iu < a.blk_nrows) {
        w.ring = a.blk_rows[AKRA_IX(iu, a.blk_nrows, kDbgUnits)];
        w.south = w.ring >= a.nunit_all;   // rows 0 .. 2N-1 are the north rings and the equator
        w.uid = w.south ? a.nring - 1 - w.ring : w.ring;
        const float x = (float)a.uinfo[AKRA_IX(w.uid, a.nunit_all, kDbgUnitInfo)].x;
        w.x = w.south ? -x : x;
        const long long tbound = (long long)(a.L + 1) * a.nunit_all;
        (void)tbound;
        const int2 st = a.start[AKRA_IX((size_t)m * a.nunit_all + w.uid, tbound, kDbgStart)];
        w.gs = st.x;
        w.e = st.y;
        w.seed = a.seeds[AKRA_IX((size_t)m * a.nunit_all + w.uid, tbound, kDbgSeeds)];
    }
}

// the state of a ring whose recurrence starts at the grid point lt (until then it is zero).  A south ring's λ
// follow from its pair's: sλ(π-θ) = (-1)^{l+m} (-s)λ(θ).  Exponent index -1 (state x 2^64) becomes 0 at
// once: 2^-96 and the smaller spin's 2^-17 of it are normal FP32 numbers.  Only states below 2^-96 keep it.
__device__ __forceinline__ void blk_settle(BlkRow &w)
{
    if (w.e == -1) {
        const float2 s = make_float2(Scale<float>::inv(), Scale<float>::inv());
        w.V = __fmul2_rn(w.V, s);
        w.VO = __fmul2_rn(w.VO, s);
        w.e = 0;
    }
}

__device__ __forceinline__ void blk_row_start(int m, int lt, BlkRow &w)
{
    if (w.gs != lt) return;
    const float4 s = w.seed;
    if (w.south) {
        const float sg = ((lt + m) & 1) ? -1.f : 1.f;
        w.V = make_float2(sg * s.y, sg * s.x);
        w.VO = make_float2(sg * s.w, sg * s.z);
    } else {
        w.V = make_float2(s.x, s.y);
        w.VO = make_float2(-s.z, -s.w);   // ξ_{g-1} = -μ_{g-1}
    }
    blk_settle(w);
}

// after 8 steps of phase A: a state that has grown past 2^32 at its exponent index moves to the next one
__device__ __forceinline__ void blk_rescale(BlkRow &w)
{
    if (w.e < 0 && (fabsf(w.V.x) > Scale<float>::hi() || fabsf(w.V.y) > Scale<float>::hi())) {
        const float2 s = make_float2(Scale<float>::inv(), Scale<float>::inv());
        w.V = __fmul2_rn(w.V, s);
        w.VO = __fmul2_rn(w.VO, s);
        w.e++;
        blk_settle(w);
    }
}

// the true state, whatever its exponent index (entering the block phase; past its turning point a ring's λ is
// of order 1, so the index is 0 there)
__device__ __forceinline__ void blk_unscale(BlkRow &w)
{
    for (; w.e < 0; w.e++) {
        const float2 s = make_float2(Scale<float>::inv(), Scale<float>::inv());
        w.V = __fmul2_rn(w.V, s);
        w.VO = __fmul2_rn(w.VO, s);
    }
}

// first l of the block phase: past every ring's turning point of either spin (sqrt(m^2 + 4 + 4 m |x|) / sin θ)
// and start, a whole number of 16-step blocks after l_first
__device__ __forceinline__ int blk_switch(int m, float zmax, int l_first, int last_start)
{
    const float lt = sqrtf(((float)m * m + 4.f + 4.f * m * zmax) / fmaxf(1.f - zmax * zmax, 1e-6f)) + 4.f;
    const int l = max((int)fminf(lt, 1e6f), last_start + 1);
    return l_first + (max(l - l_first, 0) + BLK_K - 1) / BLK_K * BLK_K;
}

// the inputs of one l-step as loaded (kept raw until they are staged, so that nothing waits for the loads)
struct BlkRaw {
    float4 c;        // recurrence coefficients {A', c', σ, A' - 2}
    float2 E, B;
    float f;         // KS factor, or -1
    __device__ __forceinline__ void load(const LegArgs<float> &a, int m, long long mbase, int l, int r, bool in)
    {
        const long long ntri = a.ntri, abound = (long long)a.R * 2 * ntri;
        (void)abound;
        c = make_float4(0.f, 0.f, 0.f, 0.f);
        E = B = make_float2(0.f, 0.f);
        f = -1.f;
        if (in) {
            c = a.coef[AKRA_IX(mbase + l, ntri, kDbgCoef)];
            E = a.alm[AKRA_IX(((size_t)r * 2 + 0) * ntri + mbase + l, abound, kDbgAlm)];
            B = a.alm[AKRA_IX(((size_t)r * 2 + 1) * ntri + mbase + l, abound, kDbgAlm)];
            if (a.fl) f = a.fl[AKRA_IX(l, a.L + 1, kDbgKsFactor)];
        }
    }
    // {c.re, d.re, c.im, d.im} with c = f (E + iB), d = f (E - iB), f including the monic scale and the state
    // sign s_l of step i
    __device__ __forceinline__ float4 cd(int m, int i) const
    {
        const float g = f * (c.z * f2_sign(i)), ei = m == 0 ? 0.f : E.y, bi = m == 0 ? 0.f : B.y;
        return make_float4(g * (E.x - bi), g * (E.x + bi), g * (ei + B.x), g * (ei - B.x));
    }
};

// inverse of the power of two at or below a magnitude (bits of a non-negative float)
__device__ __forceinline__ float blk_down(unsigned bits)
{
    const int e = (int)(bits >> 23);
    // infinities and NaN give NaN; 2^-127 is a subnormal number
    return e == 255 ? __int_as_float(0x7fc00000) : e == 254 ? __int_as_float(0x00400000)
                                                 : __uint_as_float((unsigned)(254 - max(e, 1)) << 23);
}

__device__ __forceinline__ float blk_up(unsigned bits)   // its inverse
{
    const int e = (int)(bits >> 23);
    return e == 255 ? __int_as_float(0x7fc00000) : __uint_as_float((unsigned)max(e, 1) << 23);
}

// split v into two FP16 parts and store the node pair's values of one column.  No scaling: past the turning
// point |p_k|, |q_k| <= ~20, and the sums are of c, d scaled to at most 2.
__device__ __forceinline__ void blk_put(unsigned char *bh, unsigned char *bl, int off, float2 v)
{
    const __half2 h = __float22half2_rn(v);
    const float2 hf = __half22float2(h);
    const __half2 g = __float22half2_rn(make_float2(v.x - hf.x, v.y - hf.y));
    *reinterpret_cast<__half2 *>(bh + off) = h;
    *reinterpret_cast<__half2 *>(bl + off) = g;
}

__device__ __forceinline__ float blk_absmax(float2 v) { return fmaxf(fabsf(v.x), fabsf(v.y)); }

// barrier of the ring threads
__device__ __forceinline__ void blk_bar_rings() { asm volatile("bar.sync 1, %0;" :: "n"(BLK_NT) : "memory"); }

// first start, last start and |X| maximum over the block's rings (x: magnitude bits, ring threads only)
struct BlkRange { int first, last; unsigned xmax; };
__device__ __forceinline__ BlkRange blk_range(const BlkRow (&w)[2], bool ringt, unsigned x)
{
    __shared__ BlkRange s_rg;
    if (threadIdx.x == 0) s_rg = BlkRange{kNeverLive, 0, 0u};
    __syncthreads();
    if (ringt) {
        const int lo = __reduce_min_sync(0xffffffffu, min(w[0].gs, w[1].gs));
        const int hi = __reduce_max_sync(0xffffffffu, max(w[0].ring < 0 ? 0 : w[0].gs, w[1].ring < 0 ? 0 : w[1].gs));
        const unsigned xm = __reduce_max_sync(0xffffffffu, x);
        if ((threadIdx.x & 31) == 0) {
            atomicMin(&s_rg.first, lo);
            atomicMax(&s_rg.last, hi);
            atomicMax(&s_rg.xmax, xm);
        }
    }
    __syncthreads();
    return s_rg;
}

// node recurrences of one block and spin at a pair of nodes, in the variable x for spin + and -x for spin -:
// t_-(x) = A'x - c' = -t_+(-x), so η_k = (-1)^k ξ_k of spin - obeys spin +'s recurrence at -x and both
// spins read the same coefficients.  After 15 steps p, q hold p_14, q_14 and po, qo hold ±p_15, ±q_15.
struct BlkNode {
    float2 p, po, q, qo;
    __device__ __forceinline__ void init(float sg)   // sg: +1 for spin +, -1 for spin -
    {
        p = make_float2(1.f, 1.f);
        qo = make_float2(sg, sg);
        po = q = make_float2(0.f, 0.f);
    }
    __device__ __forceinline__ void step(int k, const float2 c, const float2 xn)
    {
        const float2 tt = f2fma(make_float2(c.x, c.x), xn, make_float2(c.y, c.y));
        if (k & 1) {
            p = f2fma(tt, po, p);
            q = f2fma(tt, qo, q);
        } else {
            po = f2fma(tt, p, po);
            qo = f2fma(tt, q, qo);
        }
    }
    // signs of the odd step's values
    __device__ __forceinline__ void fix(float sg)
    {
        po = __fmul2_rn(po, make_float2(sg, sg));
        qo = __fmul2_rn(qo, make_float2(sg, sg));
    }
};

// jump of a ring's state over a block: g = (p_14, q_14, p_15, q_15) at the ring, spin-paired; A, C the last
// step's coefficients
__device__ __forceinline__ void blk_jump(BlkRow &w, const float *g, float A, float C)
{
    const float2 tt = f2fma(make_float2(A, A), make_float2(w.x, w.x), make_float2(C, -C));
    const float2 x14 = f2fma(make_float2(g[2], g[3]), w.VO, __fmul2_rn(make_float2(g[0], g[1]), w.V));
    const float2 x15 = f2fma(make_float2(g[6], g[7]), w.VO, __fmul2_rn(make_float2(g[4], g[5]), w.V));
    w.V = f2fma(tt, x15, x14);
    w.VO = x15;
}

// A block of the grid: 128 threads own two rings each (phase A, jumps: what a shared-memory load costs is its
// words per lane, a broadcast included, so every coefficient loaded serves two rings), four warps run the node recurrences,
// each its own two blocks of a tile, and two threads issue the tensor-core products, one per row tile of 128
// rings.  They hand tiles over through mbarriers, so that the node warps work ahead (also while the ring
// threads are in phase A) and nobody but the issuing threads spends time on the issue (about 40 cycles a
// product, 600 for its round trip).  A wait names the use of its barrier (parity): each barrier's next use
// depends on the waiter, so that it is never more than one use ahead of a wait.
struct BlkBars {
    uint64_t ready[2];      // node values of a tile stored (4 node warps), by buffer
    uint64_t bfree[2];      // ... read by the products of both row tiles, by buffer
    uint64_t full[2][2];    // interpolated values in TMEM (completion, issuing thread), by row tile and half tile
    uint64_t empty[2][2];   // ... read by the row tile's 4 ring warps
    uint64_t yready[2];     // adjoint: products of a row tile stored (4 ring warps)
    uint64_t yfree[2];      // adjoint: ... read by the moments' product
    uint64_t full2[2];      // adjoint: moments of both row tiles in TMEM, by buffer
    uint64_t empty2[2];     // adjoint: ... read by the 4 node warps
};
constexpr int BLK_THREADS = BLK_NT + BLK_NN + 64;
constexpr int BLK_SLOTS = 4;     // ring of per-tile hand-over values (last-step coefficients, scales)

__device__ __forceinline__ bool blk_wait(const LegArgs<float> &a, uint64_t *bar, uint32_t use)
{
    return tc::mbar_wait(bar, use & 1, kBlkWaitLimit, a.err);
}
// The item's last arrivals at bfree (and, in the adjoint, at yfree) come from the tensor core's completions and
// have no other waiter: waited for here by the thread that issued them, so that none is in flight when the block
// gives its shared memory back (to a block that initialises barriers at the same addresses).
template <bool ADJ>
__device__ __forceinline__ bool blk_drain(const LegArgs<float> &a, BlkBars *bars, int T, int h)
{
    bool ok = true;
    if (T > 0) ok &= blk_wait(a, &bars->bfree[(T - 1) & 1], (T - 1) >> 1);
    if (T > 1) ok &= blk_wait(a, &bars->bfree[T & 1], (T - 2) >> 1);
    if (ADJ && T > 0) ok &= blk_wait(a, &bars->yfree[h], T - 1);
    return ok;
}

__device__ __forceinline__ void blk_warp_arrive(uint64_t *bar)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0) tc::mbar_arrive(bar);
}
__device__ __forceinline__ void blk_warp_arrive2(uint64_t *bar, uint64_t *bar2)
{
    __syncwarp();
    if ((threadIdx.x & 31) == 0) {
        tc::mbar_arrive(bar);
        tc::mbar_arrive(bar2);
    }
}

// ---------------------------------------------------------------------------
// synthesis item: Φ(ring, ±m) of one chunk of rings and one RHS
// ---------------------------------------------------------------------------
struct BlkSynthSmem {
    static constexpr int BBUF = 16 * BLK_BSBO;   // one part of a tile's node values (128 columns)
    static constexpr int OFF_B = BLK_VBYTES;     // [2 buffers][2 parts]
    static constexpr int ROWS = BLK_NB * BLK_CROW;
    static constexpr int OFF_CF = OFF_B + 4 * BBUF;                     // coefficients
    static constexpr int OFF_AL = OFF_CF + ROWS * 8;                    // alm
    static constexpr int OFF_CT = OFF_AL + ROWS * 16;               // [slots][8] {rA', rc'} of a block's last step, scale of its sums
    static constexpr int OFF_PA = OFF_CT + BLK_SLOTS * BLK_NB * 16;     // phase A: coefficients and alm of 64 steps
    static constexpr int USED = OFF_PA + 2 * 64 * 16;
    static constexpr int BYTES = USED > 76 * 1024 ? USED : 76 * 1024;   // at most 2 blocks per SM (TMEM: 256 columns each)
};

// returns the number of tiles (uses of the barriers)
__device__ __forceinline__ int blk_synth_item(const LegArgs<float> &a, const int m, const int chunk, const int r,
                                              unsigned char *smem, BlkBars *bars, const uint32_t tmem)
{
    using S = BlkSynthSmem;
    const int L = a.L;
    const bool ringt = threadIdx.x < BLK_NT, nodet = !ringt && threadIdx.x < BLK_NT + BLK_NN;
    const int tid = ringt ? threadIdx.x : threadIdx.x - BLK_NT;
    const long long mbase = (long long)m * (2 * L + 1 - m) / 2, ntri = a.ntri;
    (void)ntri;
    float4 *s_ct = reinterpret_cast<float4 *>(smem + S::OFF_CT);
    const BlkChunk &ci = a.blk_info[AKRA_IX(chunk, a.blk_chunks, kDbgUnits)];

    BlkRow w[2];
    if (ringt) {
        blk_row_init(a, m, chunk, 0, w[0]);
        blk_row_init(a, m, chunk, 1, w[1]);
    }
    const BlkRange rg = blk_range(w, ringt, 0u);
    // first l of the block phase; a ring that never starts keeps the chunk in phase A
    const int lB = rg.last == kNeverLive ? L + 1 : blk_switch(m, ci.zmax, min(rg.first, L + 1), rg.last);
    const int T = lB <= L ? (L - lB) / BLK_TILE + 1 : 0;

    bool ok = true;
    if (nodet) {
        if (T > 0) {
            for (int i = tid; i < BLK_VBYTES / 16; i += BLK_NN)
                reinterpret_cast<uint4 *>(smem)[i] =
                    a.blk_vtab[AKRA_IX((size_t)chunk * (BLK_VBYTES / 16) + i, (long long)a.blk_chunks * (BLK_VBYTES / 16), kDbgUnits)];
            const int kp = tid & 7, sp = (tid >> 3) & 1, pb = tid >> 4;   // node pair, spin, block
            const float sg = sp ? -1.f : 1.f;
            const float2 xn = make_float2(sg * ci.node[2 * kp], sg * ci.node[2 * kp + 1]);
            BlkRaw nx;   // step tid of the next tile
            nx.load(a, m, mbase, lB + tid, r, lB + tid <= L);
            for (int t = 0; t < T; t++) {
                const uint32_t gt = t;
                const int buf = gt & 1, slot = gt & (BLK_SLOTS - 1);
                float2 *s_cf = reinterpret_cast<float2 *>(smem + S::OFF_CF);
                float4 *s_al = reinterpret_cast<float4 *>(smem + S::OFF_AL);
                {
                    // a warp stages the 32 steps of its own two blocks, alm of 32 steps (two blocks) scaled by one power of two
                    const float4 pc = nx.c, pd = nx.cd(m, tid);
                    const unsigned mx = __reduce_max_sync(0xffffffffu, __float_as_uint(
                        fmaxf(fmaxf(fabsf(pd.x), fabsf(pd.y)), fmaxf(fabsf(pd.z), fabsf(pd.w)))));
                    const float inv = blk_down(mx), rs = (tid & 1) ? -1.f : 1.f, ri = rs * inv;
                    const int o = blk_coff(tid >> 4, tid & 15);
                    s_cf[o] = make_float2(rs * pc.x, rs * pc.y);
                    s_al[o] = make_float4(pd.x * inv, pd.z * inv, pd.y * ri, pd.w * ri);
                    if ((tid & 15) == 15) s_ct[slot * BLK_NB + (tid >> 4)] = make_float4(-pc.x, -pc.y, blk_up(mx), 0.f);
                }
                __syncwarp();
                const int ln = lB + (t + 1) * BLK_TILE + tid;
                nx.load(a, m, mbase, ln, r, ln <= L);
                const float2 *cf = s_cf + blk_coff(pb, 0), *al = reinterpret_cast<const float2 *>(s_al + blk_coff(pb, 0)) + sp;
                BlkNode nd;
                nd.init(sg);
                float2 s0 = make_float2(0.f, 0.f), s1 = s0, s2 = s0, s3 = s0;
#pragma unroll
                for (int k = 0; k < BLK_K; k++) {
                    const float2 d = al[2 * k];
                    const float2 pk = (k & 1) ? nd.po : nd.p, qk = (k & 1) ? nd.qo : nd.q;
                    s0 = f2fma(make_float2(d.x, d.x), pk, s0);
                    s1 = f2fma(make_float2(d.y, d.y), pk, s1);
                    s2 = f2fma(make_float2(d.x, d.x), qk, s2);
                    s3 = f2fma(make_float2(d.y, d.y), qk, s3);
                    if (k < BLK_K - 1) nd.step(k, cf[k], xn);
                }
                nd.fix(sg);
                // the products of two tiles back have read this buffer
                if (gt > 1) ok &= blk_wait(a, &bars->bfree[buf], (gt >> 1) - 1);
                unsigned char *bh = smem + S::OFF_B + buf * 2 * S::BBUF, *bl = bh + S::BBUF;
                const int n0 = pb * 16 + sp;   // columns 2 j + spin of the block
                blk_put(bh, bl, blk_boff(n0 + 0, kp), nd.p);
                blk_put(bh, bl, blk_boff(n0 + 2, kp), nd.q);
                blk_put(bh, bl, blk_boff(n0 + 4, kp), nd.po);
                blk_put(bh, bl, blk_boff(n0 + 6, kp), nd.qo);
                blk_put(bh, bl, blk_boff(n0 + 8, kp), s0);
                blk_put(bh, bl, blk_boff(n0 + 10, kp), s1);
                blk_put(bh, bl, blk_boff(n0 + 12, kp), s2);
                blk_put(bh, bl, blk_boff(n0 + 14, kp), s3);
                tc::fence_async_smem();
                blk_warp_arrive(&bars->ready[buf]);
            }
        }
    } else if (!ringt) {
        if ((threadIdx.x & 31) == 0) {
            const int h = (threadIdx.x - BLK_NT - BLK_NN) >> 5;   // row tile
            const uint32_t va = tc::smem_u32(smem);
            const uint32_t idesc = tc::idesc_f16(128, 64, 0, 0);
            const uint64_t vh = tc::sdesc_f16(va + h * 8192, 128, 512), vl = tc::sdesc_f16(va + h * 8192 + 256, 128, 512);
            for (int t = 0; t < T; t++) {
                const uint32_t gt = t;
                ok &= blk_wait(a, &bars->ready[gt & 1], gt >> 1);
#pragma unroll
                for (int u = 0; u < 2; u++) {   // half tile: 4 blocks
                    const uint32_t bb = va + S::OFF_B + (gt & 1) * 2 * S::BBUF + u * 8 * BLK_BSBO, d = tmem + h * 128 + u * 64;
                    const uint64_t nh = tc::sdesc_f16(bb, BLK_BLBO, BLK_BSBO), nl = tc::sdesc_f16(bb + S::BBUF, BLK_BLBO, BLK_BSBO);
                    // the previous tile's values in these columns have been read
                    if (gt > 0) ok &= blk_wait(a, &bars->empty[h][u], gt - 1);
                    tc::fence_after();
                    tc::mma_f16(d, vl, nh, idesc, 0u);
                    tc::mma_f16(d, vh, nl, idesc, 1u);
                    tc::mma_f16(d, vh, nh, idesc, 1u);
                    tc::commit(&bars->full[h][u]);
                    tc::mbar_arrive(&bars->full[h][u]);   // the tile's hand-over values
                }
                tc::commit(&bars->bfree[gt & 1]);
            }
            ok &= blk_drain<false>(a, bars, T, h);
        }
    } else {
        float4 *s_al = reinterpret_cast<float4 *>(smem + S::OFF_PA);
        float2 *s_cf = reinterpret_cast<float2 *>(s_al + 64);
        const int warp_first = __reduce_min_sync(0xffffffffu, min(w[0].gs, w[1].gs));
        float2 aR[2], aI[2];   // (Σ c ξ+, Σ d ξ-), re and im
        aR[0] = aR[1] = aI[0] = aI[1] = make_float2(0.f, 0.f);
        // phase A: direct recurrence, 64 steps staged at a time (the next ones' loads in flight)
        const int lend = min(lB, L + 1);
        BlkRaw nx;
        nx.load(a, m, mbase, rg.first + tid, r, tid < 64 && rg.first < lend && rg.first + tid < lend);
        for (int lt = rg.first; lt < lend; lt += 64) {
            const int nl = min(64, lend - lt);
            blk_bar_rings();
            if (tid < 64) {
                const float rs = (tid & 1) ? -1.f : 1.f;
                s_cf[tid] = make_float2(rs * nx.c.x, rs * nx.c.y);
                s_al[tid] = nx.cd(m, tid);
            }
            blk_bar_rings();
            nx.load(a, m, mbase, lt + 64 + tid, r, tid < 64 && lt + 64 + tid < lend);
            blk_row_start(m, lt, w[0]);
            blk_row_start(m, lt, w[1]);
            if (warp_first > lt + nl - 1) continue;
            const bool all_live = __all_sync(0xffffffffu, (w[0].e == 0 || w[0].gs > lt) && (w[1].e == 0 || w[1].gs > lt));
#pragma unroll 1
            for (int i0 = 0; i0 < nl; i0 += 8) {
                // a ring whose state is still below the range contributes nothing over the 8 steps
                float2 tR[2], tI[2];
                tR[0] = tR[1] = tI[0] = tI[1] = make_float2(0.f, 0.f);
#pragma unroll
                for (int i = i0; i < i0 + 8; i += 2) {
                    const float4 c = *reinterpret_cast<const float4 *>(s_cf + i), d0 = s_al[i], d1 = s_al[i + 1];
#pragma unroll
                    for (int k = 0; k < 2; k++) {
                        const float2 X2 = make_float2(w[k].x, w[k].x);
                        tR[k] = f2fma(make_float2(d0.x, d0.y), w[k].V, tR[k]);
                        tI[k] = f2fma(make_float2(d0.z, d0.w), w[k].V, tI[k]);
                        w[k].VO = f2fma(f2fma(make_float2(c.x, c.x), X2, make_float2(c.y, -c.y)), w[k].V, w[k].VO);
                        tR[k] = f2fma(make_float2(d1.x, d1.y), w[k].VO, tR[k]);
                        tI[k] = f2fma(make_float2(d1.z, d1.w), w[k].VO, tI[k]);
                        w[k].V = f2fma(f2fma(make_float2(c.z, c.z), X2, make_float2(c.w, -c.w)), w[k].VO, w[k].V);
                    }
                }
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    if (all_live || w[k].e == 0) {
                        aR[k] = __fadd2_rn(aR[k], tR[k]);
                        aI[k] = __fadd2_rn(aI[k], tI[k]);
                    }
                    if (!all_live) blk_rescale(w[k]);
                }
            }
        }
        // phase B: jumps
        blk_unscale(w[0]);
        blk_unscale(w[1]);
        const uint32_t col = tmem + ((uint32_t)(tid & 96) << 16);
        for (int t = 0; t < T; t++) {
            const uint32_t gt = t;
            const float4 *ct = s_ct + (gt & (BLK_SLOTS - 1)) * BLK_NB;
#pragma unroll
            for (int u = 0; u < 2; u++) {
                ok &= blk_wait(a, &bars->full[0][u], gt);
                ok &= blk_wait(a, &bars->full[1][u], gt);
                tc::fence_after();
                // the two rings' values in turn: one is used while the other's load is in flight
                float g[2][16];
                tc::tmem_ld16(col + u * 64, g[0]);
#pragma unroll
                for (int b = 0; b < 4; b++) {
                    const float4 c = ct[4 * u + b];
#pragma unroll
                    for (int k = 0; k < 2; k++) {
                        tc::tmem_wait_ld(g[k]);
                        if (k == 0) tc::tmem_ld16(col + 128 + u * 64 + b * 16, g[1]);
                        else if (b < 3) tc::tmem_ld16(col + u * 64 + (b + 1) * 16, g[0]);
                        const float *gk = g[k];
                        const float2 Vc = __fmul2_rn(w[k].V, make_float2(c.z, c.z)), Oc = __fmul2_rn(w[k].VO, make_float2(c.z, c.z));
                        aR[k] = f2fma(make_float2(gk[12], gk[13]), Oc, f2fma(make_float2(gk[8], gk[9]), Vc, aR[k]));
                        aI[k] = f2fma(make_float2(gk[14], gk[15]), Oc, f2fma(make_float2(gk[10], gk[11]), Vc, aI[k]));
                        blk_jump(w[k], gk, c.x, c.y);
                    }
                }
                tc::fence_before();
                blk_warp_arrive2(&bars->empty[0][u], &bars->empty[1][u]);
            }
        }
#pragma unroll
        for (int k = 0; k < 2; k++) {
            if (w[k].ring < 0) continue;
            const size_t row = 2 * (size_t)L + 1;
            const long long pbound = (long long)a.R * a.nring * row;
            (void)pbound;
            const size_t pb = ((size_t)r * a.nring + w[k].ring) * row + L;   // Φ(ring, m = 0)
            a.phi[AKRA_IX(pb + m, pbound, kDbgPhiWrite)] = make_float2(aR[k].x, aI[k].x);
            if (m > 0) a.phi[AKRA_IX(pb - m, pbound, kDbgPhiWrite)] = make_float2(aR[k].y, -aI[k].y);
        }
    }
    if (!ok && a.err) atomicExch(a.err, 1);
    __syncthreads();
    return T;
}

// ---------------------------------------------------------------------------
// adjoint item: partial[chunk][r][idx(l, m)] = Σ_{rings of the chunk} (E-part, B-part) at every l, with
// a = Σ 2λ P, b = Σ (-2)λ Q, E-part = a + b, B-part = a - b (P = Φ'(m), Q = conj Φ'(-m) of the ring's row).
// Node threads: jump values of tile t, then the moments of tile t - 1 into its outputs.  Ring threads:
// products of the state with P and Q at each block's start (FP16 head and rest, the M x K operand of the
// moments), jump.
// ---------------------------------------------------------------------------
struct BlkAdjSmem {
    static constexpr int BBUF = 8 * BLK_BSBO;              // one part of a tile's jump values (64 columns)
    static constexpr int OFF_Y = BLK_VBYTES;               // products, M x K = (8 blocks x 8, 2 parts) x 256 rings
    static constexpr int YG = (BLK_RINGS / 8) * 128;         // bytes of one M group of 8
    static constexpr int OFF_B = OFF_Y + 16 * YG;          // [2 buffers][2 parts]
    static constexpr int ROWS = BLK_NB * BLK_CROW;
    static constexpr int OFF_CF = OFF_B + 4 * BBUF;        // [slots]
    static constexpr int OFF_SG = OFF_CF + BLK_SLOTS * ROWS * 8;       // [slots][128] output scales
    static constexpr int OFF_CT = OFF_SG + BLK_SLOTS * BLK_TILE * 4;   // [slots][8] {rA', rc'} of a block's last step
    static constexpr int OFF_MOM = OFF_CT + BLK_SLOTS * BLK_NB * 8, MROW = 20;
    static constexpr int BYTES = OFF_MOM + 128 * MROW * 4;
    static constexpr int NW = BLK_NT / 32;
    static constexpr int OFF_TR = OFF_Y, OFF_RED = OFF_Y + NW * 32 * 36 * 4, OFF_PA = OFF_RED + NW * 64 * 16;   // phase A
    static_assert(OFF_PA + 64 * 16 <= OFF_B, "");
    static_assert(2 * (BYTES + 2048) <= 227 * 1024 && 3 * (BYTES + 1024) > 228 * 1024, "2 blocks per SM, whose TMEM fits");
};

__device__ __forceinline__ int blk_adjoint_item(const LegArgs<float> &a, const int m, const int chunk, const int r,
                                                unsigned char *smem, BlkBars *bars, const uint32_t tmem)
{
    using S = BlkAdjSmem;
    const int L = a.L;
    const bool ringt = threadIdx.x < BLK_NT, nodet = !ringt && threadIdx.x < BLK_NT + BLK_NN;
    const int tid = ringt ? threadIdx.x : threadIdx.x - BLK_NT, lane = tid & 31, warp = tid >> 5;
    const int l0 = m > 2 ? m : 2;
    const long long mbase = (long long)m * (2 * L + 1 - m) / 2, ntri = a.ntri;
    float2 *s_ct = reinterpret_cast<float2 *>(smem + S::OFF_CT);
    float4 *part = reinterpret_cast<float4 *>(a.partial) + ((size_t)chunk * a.R + r) * ntri + mbase;
    const long long qbound = (long long)a.nchunks * a.R * ntri - (((long long)chunk * a.R + r) * ntri + mbase);
    (void)qbound;
    const BlkChunk &ci = a.blk_info[AKRA_IX(chunk, a.blk_chunks, kDbgUnits)];
    const uint32_t lane_base = tmem + ((uint32_t)(tid & 96) << 16);

    BlkRow w[2];
    float2 Xr[2], Xi[2];   // (P, Q): re and im
    Xr[0] = Xr[1] = Xi[0] = Xi[1] = make_float2(0.f, 0.f);
    if (ringt) {
#pragma unroll
        for (int k = 0; k < 2; k++) {
            blk_row_init(a, m, chunk, k, w[k]);
            if (w[k].ring < 0) continue;
            const size_t row = 2 * (size_t)L + 1;
            const long long pbound = (long long)a.R * a.nring * row;
            (void)pbound;
            const size_t pb = ((size_t)r * a.nring + w[k].ring) * row + L;   // Φ'(ring, m = 0)
            const float2 g = a.phi_in[AKRA_IX(pb + m, pbound, kDbgPhiRead)];
            const float2 h = a.phi_in[AKRA_IX(pb - m, pbound, kDbgPhiRead)];
            Xr[k] = make_float2(g.x, h.x);
            Xi[k] = make_float2(g.y, -h.y);
        }
    }
    const BlkRange rg = blk_range(w, ringt, __float_as_uint(fmaxf(fmaxf(blk_absmax(Xr[0]), blk_absmax(Xi[0])),
                                                                  fmaxf(blk_absmax(Xr[1]), blk_absmax(Xi[1])))));
    const int lB = rg.last == kNeverLive ? L + 1 : blk_switch(m, ci.zmax, min(rg.first, L + 1), rg.last);
    const int T = lB <= L ? (L - lB) / BLK_TILE + 1 : 0;
    const float xinv = blk_down(rg.xmax), xup = blk_up(rg.xmax);   // X is scaled to at most 2
    bool ok = true;

    if (nodet) {
        for (int i = tid; i < BLK_VBYTES / 16 && T > 0; i += BLK_NN)
            reinterpret_cast<uint4 *>(smem)[i] =
                a.blk_vtab[AKRA_IX((size_t)chunk * (BLK_VBYTES / 16) + i, (long long)a.blk_chunks * (BLK_VBYTES / 16), kDbgUnits)];
        const int kp = tid & 7, sp = (tid >> 3) & 1, pb = tid >> 4;   // node pair, spin, block
        const float sg = sp ? -1.f : 1.f;
        const float2 xn = make_float2(sg * ci.node[2 * kp], sg * ci.node[2 * kp + 1]);
        float *mom = reinterpret_cast<float *>(smem + S::OFF_MOM);
        float4 pc = make_float4(0.f, 0.f, 0.f, 0.f);
        if (T > 0 && lB + tid <= L) pc = a.coef[AKRA_IX(mbase + lB + tid, ntri, kDbgCoef)];
        // the moments lag two tiles, so that a tile's jump values are there before the ring threads need them
        for (int t = 0; t < T + 2 && T > 0; t++) {
            const uint32_t gt = t;
            if (t < T) {
                const int buf = gt & 1, slot = gt & (BLK_SLOTS - 1);
                float2 *s_cf = reinterpret_cast<float2 *>(smem + S::OFF_CF) + slot * S::ROWS;
                const float rs = (tid & 1) ? -1.f : 1.f;
                s_cf[blk_coff(tid >> 4, tid & 15)] = make_float2(rs * pc.x, rs * pc.y);
                if ((tid & 15) == 15) s_ct[slot * BLK_NB + (tid >> 4)] = make_float2(-pc.x, -pc.y);
                // the recurrence ran on ξ_l = s_l λ_l / σ_l, the sums on X scaled
                reinterpret_cast<float *>(smem + S::OFF_SG)[slot * 128 + tid] = pc.z * f2_sign(tid) * xup;
                __syncwarp();
                const int ln = lB + (t + 1) * BLK_TILE + tid;
                pc = make_float4(0.f, 0.f, 0.f, 0.f);
                if (ln <= L) pc = a.coef[AKRA_IX(mbase + ln, ntri, kDbgCoef)];
                BlkNode nd;
                nd.init(sg);
                const float2 *cf = s_cf + blk_coff(pb, 0);
#pragma unroll
                for (int k = 0; k < BLK_K - 1; k++) nd.step(k, cf[k], xn);
                nd.fix(sg);
                // the products of two tiles back have read this buffer
                if (gt > 1) ok &= blk_wait(a, &bars->bfree[buf], (gt >> 1) - 1);
                unsigned char *bh = smem + S::OFF_B + buf * 2 * S::BBUF, *bl = bh + S::BBUF;
                const int n0 = pb * 8 + sp;
                blk_put(bh, bl, blk_boff(n0 + 0, kp), nd.p);
                blk_put(bh, bl, blk_boff(n0 + 2, kp), nd.q);
                blk_put(bh, bl, blk_boff(n0 + 4, kp), nd.po);
                blk_put(bh, bl, blk_boff(n0 + 6, kp), nd.qo);
                tc::fence_async_smem();
                blk_warp_arrive(&bars->ready[buf]);
            }
            if (t > 1) {
                // moments: this warp's 32 TMEM rows = (part of Y, block of its two, product),
                // columns = (row tile, part of V, node)
                const uint32_t pt = gt - 2;
                const int buf = pt & 1, slot = pt & (BLK_SLOTS - 1);
                ok &= blk_wait(a, &bars->full2[buf], pt >> 1);
                tc::fence_after();
                {
                    float g0[16], g1[16];
                    tc::tmem_ld16(lane_base + 128 + buf * 64, g0);
                    tc::tmem_ld16(lane_base + 144 + buf * 64, g1);
                    tc::tmem_wait_ld(g0);
                    tc::tmem_wait_ld(g1);
#pragma unroll
                    for (int j = 0; j < 16; j++) g0[j] += g1[j];
                    tc::tmem_ld16(lane_base + 160 + buf * 64, g1);
                    tc::tmem_wait_ld(g1);
#pragma unroll
                    for (int j = 0; j < 16; j++) g0[j] += g1[j];
                    tc::tmem_ld16(lane_base + 176 + buf * 64, g1);
                    tc::tmem_wait_ld(g1);
                    float4 *dst = reinterpret_cast<float4 *>(mom + tid * S::MROW);
#pragma unroll
                    for (int j = 0; j < 4; j++)
                        dst[j] = make_float4(g0[4 * j] + g1[4 * j], g0[4 * j + 1] + g1[4 * j + 1],
                                             g0[4 * j + 2] + g1[4 * j + 2], g0[4 * j + 3] + g1[4 * j + 3]);
                }
                tc::fence_before();
                blk_warp_arrive(&bars->empty2[buf]);
                // Σ over rings at step k = p_k · (moments of ξ_l X) + q_k · (moments of ξ_{l-1} X) at every node: the
                // recurrence itself, started from the moments
                float2 M[4];
#pragma unroll
                for (int i = 0; i < 4; i++) {
                    const float *row = mom + ((pb >> 1) * 32 + (pb & 1) * 8 + 2 * i + sp) * S::MROW + 2 * kp;
                    const float2 u = *reinterpret_cast<const float2 *>(row);
                    const float2 v = *reinterpret_cast<const float2 *>(row + 16 * S::MROW);
                    M[i] = make_float2(u.x + v.x, u.y + v.y);
                }
                const float2 *cf = reinterpret_cast<const float2 *>(smem + S::OFF_CF) + slot * S::ROWS + blk_coff(pb, 0);
                float vr[16], vi[16];
                float2 re = M[0], im = M[1];
                float2 ro = __fmul2_rn(M[2], make_float2(sg, sg)), io = __fmul2_rn(M[3], make_float2(sg, sg));
#pragma unroll
                for (int k = 0; k < BLK_K; k++) {
                    const float2 rk = (k & 1) ? ro : re, ik = (k & 1) ? io : im;
                    vr[k] = rk.x + rk.y;   // (-1)^k of spin -: below
                    vi[k] = ik.x + ik.y;
                    if (k < BLK_K - 1) {
                        const float2 c = cf[k], tt = f2fma(make_float2(c.x, c.x), xn, make_float2(c.y, c.y));
                        if (k & 1) {
                            re = f2fma(tt, ro, re);
                            im = f2fma(tt, io, im);
                        } else {
                            ro = f2fma(tt, re, ro);
                            io = f2fma(tt, im, io);
                        }
                    }
                }
                // sum over the 8 node pairs, each lane keeping 2 of the 16 steps
#pragma unroll
                for (int w2 = 4; w2 > 0; w2 >>= 1) {
                    const bool up = (kp & w2) != 0;
#pragma unroll
                    for (int j = 0; j < 2 * w2; j++) {
                        const float sr = up ? vr[j] : vr[j + 2 * w2], si = up ? vi[j] : vi[j + 2 * w2];
                        vr[j] = (up ? vr[j + 2 * w2] : vr[j]) + __shfl_xor_sync(0xffffffffu, sr, w2);
                        vi[j] = (up ? vi[j + 2 * w2] : vi[j]) + __shfl_xor_sync(0xffffffffu, si, w2);
                    }
                }
                vr[1] *= sg;
                vi[1] *= sg;   // this lane's odd step
                // spin + holds a, spin - holds b: E = a + b from the first, B = a - b from the second
                const int i0 = pb * 16 + 2 * kp, l = lB + (t - 2) * BLK_TILE + i0;
                const float2 sc = *reinterpret_cast<const float2 *>(smem + S::OFF_SG + (slot * 128 + i0) * 4);
#pragma unroll
                for (int j = 0; j < 2; j++) {
                    const float orr = __shfl_xor_sync(0xffffffffu, vr[j], 8), oi = __shfl_xor_sync(0xffffffffu, vi[j], 8);
                    const float s = j == 0 ? sc.x : sc.y;
                    const float2 v = sp == 0 ? make_float2(s * (vr[j] + orr), s * (vi[j] + oi))
                                             : make_float2(s * (orr - vr[j]), s * (oi - vi[j]));
                    if (l + j <= L)
                        reinterpret_cast<float2 *>(part + AKRA_IX(l + j, qbound, kDbgPartialWrite))[sp] = v;
                }
                __syncwarp();   // the next tile's coefficients and moments take this tile's place
            }
        }
    } else if (!ringt) {
        if ((threadIdx.x & 31) == 0) {
            const int h = (threadIdx.x - BLK_NT - BLK_NN) >> 5;   // row tile
            const uint32_t va = tc::smem_u32(smem) + h * 8192, ya = tc::smem_u32(smem) + S::OFF_Y + h * 2048;
            const uint32_t id1 = tc::idesc_f16(128, 32, 0, 0), id2 = tc::idesc_f16(128, 32, 1, 1);
            const uint64_t vh = tc::sdesc_f16(va, 128, 512), vl = tc::sdesc_f16(va + 256, 128, 512);
            for (int t = 0; t <= T && T > 0; t++) {
                const uint32_t gt = t, pt = gt - 1;
                if (t < T) {
                    ok &= blk_wait(a, &bars->ready[gt & 1], gt >> 1);
                    const uint32_t bb = tc::smem_u32(smem) + S::OFF_B + (gt & 1) * 2 * S::BBUF;
#pragma unroll
                    for (int u = 0; u < 2; u++) {   // half tile: 4 blocks
                        const uint64_t nh = tc::sdesc_f16(bb + u * 4 * BLK_BSBO, BLK_BLBO, BLK_BSBO);
                        const uint64_t nl = tc::sdesc_f16(bb + S::BBUF + u * 4 * BLK_BSBO, BLK_BLBO, BLK_BSBO);
                        const uint32_t d = tmem + h * 64 + u * 32;
                        // the previous tile's jump values in these columns have been read
                        if (gt > 0) ok &= blk_wait(a, &bars->empty[h][u], gt - 1);
                        tc::fence_after();
                        tc::mma_f16(d, vl, nh, id1, 0u);
                        tc::mma_f16(d, vh, nl, id1, 1u);
                        tc::mma_f16(d, vh, nh, id1, 1u);
                        tc::commit(&bars->full[h][u]);
                        tc::mbar_arrive(&bars->full[h][u]);   // the tile's hand-over values
                    }
                    tc::commit(&bars->bfree[gt & 1]);
                }
                // the row tile's ring threads have stored the previous tile's products
                if (t > 0) ok &= blk_wait(a, &bars->yready[h], pt);
                if (t > 0) {
                    // the moments of two tiles before have been read
                    if (pt > 1) ok &= blk_wait(a, &bars->empty2[pt & 1], (pt - 2) >> 1);
                    tc::fence_after();
#pragma unroll
                    for (int ks = 0; ks < 8; ks++)   // 16 rings each
                        tc::mma_f16(tmem + 128 + (pt & 1) * 64 + h * 32, tc::sdesc_f16(ya + ks * 256, 128, S::YG),
                                    tc::sdesc_f16(va + ks * 1024, 512, 128), id2, ks > 0 ? 1u : 0u);
                    tc::commit(&bars->yfree[h]);
                    tc::commit(&bars->full2[pt & 1]);
                }
            }
            ok &= blk_drain<true>(a, bars, T, h);
        }
    } else {
#pragma unroll
        for (int k = 0; k < 2; k++) {
            Xr[k] = __fmul2_rn(Xr[k], make_float2(xinv, xinv));
            Xi[k] = __fmul2_rn(Xi[k], make_float2(xinv, xinv));
        }
        const int warp_first = __reduce_min_sync(0xffffffffu, min(w[0].gs, w[1].gs));
        // the l below the first start get zero partial sums
        for (int i = tid; i < min(rg.first, L + 1) - l0; i += BLK_NT)
            part[AKRA_IX(l0 + i, qbound, kDbgPartialWrite)] = make_float4(0.f, 0.f, 0.f, 0.f);
        // phase A: direct recurrence, the warp's lanes summed through a transpose buffer 8 steps at a time
        float2 *s_cf = reinterpret_cast<float2 *>(smem + S::OFF_PA);
        float (*tr)[36] = reinterpret_cast<float (*)[36]>(smem + S::OFF_TR + warp * 32 * 36 * 4);
        float (*red)[64][4] = reinterpret_cast<float (*)[64][4]>(smem + S::OFF_RED);
        const int lend = min(lB, L + 1);
        float4 pc = make_float4(0.f, 0.f, 0.f, 0.f);
        if (tid < 64 && rg.first < lend && rg.first + tid < lend) pc = a.coef[AKRA_IX(mbase + rg.first + tid, ntri, kDbgCoef)];
        for (int lt = rg.first; lt < lend; lt += 64) {
            const int nl = min(64, lend - lt);
            blk_bar_rings();
            const float rs = (tid & 1) ? -1.f : 1.f;
            if (tid < 64) s_cf[tid] = make_float2(rs * pc.x, rs * pc.y);
            const float sig = pc.z * f2_sign(tid) * xup;
            blk_bar_rings();
            pc = make_float4(0.f, 0.f, 0.f, 0.f);
            if (tid < 64 && lt + 64 + tid < lend) pc = a.coef[AKRA_IX(mbase + lt + 64 + tid, ntri, kDbgCoef)];
            blk_row_start(m, lt, w[0]);
            blk_row_start(m, lt, w[1]);
            if (warp_first > lt + nl - 1) {
                for (int i = lane; i < nl * 4; i += 32) red[warp][i >> 2][i & 3] = 0.f;
            } else {
                const bool all_live = __all_sync(0xffffffffu, (w[0].e == 0 || w[0].gs > lt) && (w[1].e == 0 || w[1].gs > lt));
#pragma unroll 1
                for (int i0 = 0; i0 < nl; i0 += 8) {
                    // a ring whose state is still below the range contributes nothing over the 8 steps
                    float2 Yr[2], Yi[2];
#pragma unroll
                    for (int k = 0; k < 2; k++) {
                        const bool live = all_live || w[k].e == 0;
                        Yr[k] = live ? Xr[k] : make_float2(0.f, 0.f);
                        Yi[k] = live ? Xi[k] : make_float2(0.f, 0.f);
                    }
#pragma unroll
                    for (int i = 0; i < 8; i += 2) {
                        const float4 c = *reinterpret_cast<const float4 *>(s_cf + i0 + i);
                        float2 fr = f2fma(w[1].V, Yr[1], __fmul2_rn(w[0].V, Yr[0]));
                        float2 fi = f2fma(w[1].V, Yi[1], __fmul2_rn(w[0].V, Yi[0]));
                        *reinterpret_cast<float4 *>(&tr[lane][4 * i]) = make_float4(fr.x, fr.y, fi.x, fi.y);
#pragma unroll
                        for (int k = 0; k < 2; k++)
                            w[k].VO = f2fma(f2fma(make_float2(c.x, c.x), make_float2(w[k].x, w[k].x), make_float2(c.y, -c.y)), w[k].V, w[k].VO);
                        fr = f2fma(w[1].VO, Yr[1], __fmul2_rn(w[0].VO, Yr[0]));
                        fi = f2fma(w[1].VO, Yi[1], __fmul2_rn(w[0].VO, Yi[0]));
                        *reinterpret_cast<float4 *>(&tr[lane][4 * i + 4]) = make_float4(fr.x, fr.y, fi.x, fi.y);
#pragma unroll
                        for (int k = 0; k < 2; k++)
                            w[k].V = f2fma(f2fma(make_float2(c.z, c.z), make_float2(w[k].x, w[k].x), make_float2(c.w, -c.w)), w[k].VO, w[k].V);
                    }
                    if (!all_live) {
                        blk_rescale(w[0]);
                        blk_rescale(w[1]);
                    }
                    __syncwarp();
                    const int h = lane >> 4, v = lane & 15;
                    const float2 *c2 = reinterpret_cast<const float2 *>(&tr[16 * h][0]) + v;
                    // 16 rows in four chains: the few warps of this phase wait on latency
                    float2 s4[4];
#pragma unroll
                    for (int t = 0; t < 4; t++) s4[t] = c2[t * 18];
#pragma unroll
                    for (int t = 4; t < 16; t++) s4[t & 3] = __fadd2_rn(s4[t & 3], c2[t * 18]);
                    float2 sm = __fadd2_rn(__fadd2_rn(s4[0], s4[1]), __fadd2_rn(s4[2], s4[3]));
                    sm.x += __shfl_xor_sync(0xffffffffu, sm.x, 16);
                    sm.y += __shfl_xor_sync(0xffffffffu, sm.y, 16);
                    __syncwarp();
                    red[warp][i0 + (v >> 1)][(v & 1) + 2 * h] = h == 0 ? sm.x + sm.y : sm.x - sm.y;
                }
            }
            blk_bar_rings();
            if (tid < nl) {
                float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
                for (int q = 0; q < S::NW; q++) {
                    const float4 t = *reinterpret_cast<const float4 *>(red[q][tid]);
                    s = make_float4(s.x + t.x, s.y + t.y, s.z + t.z, s.w + t.w);
                }
                part[AKRA_IX(lt + tid, qbound, kDbgPartialWrite)] = make_float4(s.x * sig, s.y * sig, s.z * sig, s.w * sig);
            }
        }
        blk_unscale(w[0]);
        blk_unscale(w[1]);
        blk_bar_rings();   // phase A's buffers become the products'
        unsigned char *yrow = smem + S::OFF_Y + (tid >> 3) * 128 + (tid & 7) * 16;   // row tile k: + 2048 k
        for (int t = 0; t < T; t++) {
            const uint32_t gt = t;
            const float2 *ct = s_ct + (gt & (BLK_SLOTS - 1)) * BLK_NB;
#pragma unroll
            for (int u = 0; u < 2; u++) {
                ok &= blk_wait(a, &bars->full[0][u], gt);
                ok &= blk_wait(a, &bars->full[1][u], gt);
                // the moments' products of the previous tile have read their operand
                if (u == 0 && t > 0) {
                    ok &= blk_wait(a, &bars->yfree[0], gt - 1);
                    ok &= blk_wait(a, &bars->yfree[1], gt - 1);
                }
                tc::fence_after();
                // two blocks of one ring, then of the other, whose load is in flight meanwhile
                float g[2][16];
                tc::tmem_ld16(lane_base + u * 32, g[0]);
#pragma unroll
                for (int v = 0; v < 2; v++) {
#pragma unroll
                    for (int k = 0; k < 2; k++) {
                        tc::tmem_wait_ld(g[k]);
                        if (k == 0) tc::tmem_ld16(lane_base + 64 + u * 32 + v * 16, g[1]);
                        else if (v == 0) tc::tmem_ld16(lane_base + u * 32 + 16, g[0]);
#pragma unroll
                        for (int q = 0; q < 2; q++) {
                            const int b = 4 * u + 2 * v + q;
                            const float2 y[4] = {__fmul2_rn(w[k].V, Xr[k]), __fmul2_rn(w[k].V, Xi[k]), __fmul2_rn(w[k].VO, Xr[k]),
                                                 __fmul2_rn(w[k].VO, Xi[k])};
                            union { __half2 h[4]; uint4 v; } hd, rs;
#pragma unroll
                            for (int j = 0; j < 4; j++) {
                                hd.h[j] = __float22half2_rn(y[j]);
                                const float2 f = __half22float2(hd.h[j]);
                                rs.h[j] = __float22half2_rn(make_float2(y[j].x - f.x, y[j].y - f.y));
                            }
                            unsigned char *yk = yrow + k * 2048 + ((b >> 1) * 4 + (b & 1)) * S::YG;
                            *reinterpret_cast<uint4 *>(yk) = hd.v;
                            *reinterpret_cast<uint4 *>(yk + 2 * S::YG) = rs.v;
                            const float2 c = ct[b];
                            blk_jump(w[k], g[k] + 8 * q, c.x, c.y);
                        }
                    }
                }
                tc::fence_before();
                blk_warp_arrive2(&bars->empty[0][u], &bars->empty[1][u]);
            }
            tc::fence_async_smem();
            blk_warp_arrive2(&bars->yready[0], &bars->yready[1]);
        }
    }
    if (!ok && a.err) atomicExch(a.err, 1);
    __syncthreads();
    return T;
}

}  // namespace akra
