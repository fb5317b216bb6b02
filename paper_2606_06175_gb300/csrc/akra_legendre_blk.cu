// akra_legendre_blk.cu -- kernels, tables and launchers of the block-jump FP32 Legendre stages
// (method: akra_legendre_blk.cuh).
#include "akra_legendre_blk.cuh"

namespace akra {

namespace {

// interpolation tables of one chunk per block: nodes (Chebyshev points of the chunk's x-interval, rounded
// to FP32) and V, the Lagrange basis on those nodes at every ring's FP64 x, split into two FP16 parts
__global__ void __launch_bounds__(BLK_RINGS)
k_blk_tables(int nrows, int nunit, int nring, const int *__restrict__ rows, const UnitInfo *__restrict__ uinfo,
             BlkChunk *info, unsigned char *vtab)
{
    __shared__ double s_node[16], s_w[16], s_lo, s_hi;
    const int c = blockIdx.x, tid = threadIdx.x, i = c * BLK_RINGS + blk_ring_of_row(tid);   // tid: MMA row
    double x = 0;
    if (i < nrows) {
        const int ring = rows[i];
        x = ring >= nunit ? -uinfo[nring - 1 - ring].x : uinfo[ring].x;
    }
    if (tid == 0) s_hi = x;                                   // rows ascend, x descends
    if (i < nrows && (i == nrows - 1 || i == (c + 1) * BLK_RINGS - 1)) s_lo = x;
    __syncthreads();
    // at least 4e-3 wide, so that the rounded nodes stay apart (a short last chunk)
    const double mid = 0.5 * (s_lo + s_hi), half = fmax(0.5 * (s_hi - s_lo), 2e-3);
    if (tid < 16) {
        const float nd = (float)(mid + half * cospi((2 * tid + 1) / 32.0));
        s_node[tid] = nd;
        info[c].node[tid] = nd;
    }
    if (tid == 0) info[c].zmax = (float)(fabs(mid) + half);
    __syncthreads();
    if (tid < 16) {
        double w = 1;
        for (int j = 0; j < 16; j++)
            if (j != tid) w *= s_node[tid] - s_node[j];
        s_w[tid] = 1.0 / w;
    }
    __syncthreads();
    for (int j = 0; j < 16; j++) {
        double v = s_w[j];
        for (int k = 0; k < 16; k++)
            if (k != j) v *= x - s_node[k];
        if (i >= nrows) v = 0;
        const __half h = __double2half(v);
        const __half g = __double2half(v - (double)__half2float(h));
        unsigned char *t = vtab + (size_t)c * BLK_VBYTES;
        *reinterpret_cast<__half *>(t + blk_voff(tid, j, 0)) = h;
        *reinterpret_cast<__half *>(t + blk_voff(tid, j, 1)) = g;
    }
}

// TMEM (256 columns) and the hand-over barriers of a block
__device__ __forceinline__ uint32_t blk_open(uint32_t *s_tmem, BlkBars *bars)
{
    if (threadIdx.x < 32) tc::tmem_alloc(s_tmem, 256);
    if (threadIdx.x == 0) {
        for (int h = 0; h < 2; h++) {
            tc::mbar_init(&bars->ready[h], 4);
            tc::mbar_init(&bars->bfree[h], 2);
            for (int u = 0; u < 2; u++) {
                tc::mbar_init(&bars->full[h][u], 2);
                tc::mbar_init(&bars->empty[h][u], 4);
            }
            tc::mbar_init(&bars->yready[h], 4);
            tc::mbar_init(&bars->yfree[h], 1);
            tc::mbar_init(&bars->full2[h], 2);
            tc::mbar_init(&bars->empty2[h], 4);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    return *s_tmem;
}

// the bounds-checked build also records a barrier whose last phase is still open when the block ends
template <bool ADJ>
__device__ __forceinline__ void blk_check_bars(BlkBars *bars, int T)
{
#ifdef AKRA_DEBUG
    if (threadIdx.x != 0) return;
    auto check = [](uint64_t *bar, int uses) {
        if (uses > 0 && !tc::mbar_test(bar, (uses - 1) & 1)) dbg_index(-1, 1, kDbgBarrier);
    };
    for (int h = 0; h < 2; h++) {
        const int nb = (T + 1 - h) / 2;   // uses of a barrier that alternates with the tiles
        check(&bars->ready[h], nb);
        check(&bars->bfree[h], nb);
        for (int u = 0; u < 2; u++) {
            check(&bars->full[h][u], T);
            check(&bars->empty[h][u], T);
        }
        if (!ADJ) continue;
        check(&bars->yready[h], T);
        check(&bars->yfree[h], T);
        check(&bars->full2[h], nb);
        check(&bars->empty2[h], nb);
    }
#else
    (void)bars;
    (void)T;
#endif
}

template <bool ADJ>
__device__ __forceinline__ void blk_close(uint32_t tmem, BlkBars *bars, int T)
{
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    blk_check_bars<ADJ>(bars, T);
    if (threadIdx.x < 32) tc::tmem_dealloc(tmem, 256);
}

__global__ void __launch_bounds__(BLK_THREADS, 2) k_leg_synth_blk(LegArgs<float> a)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ BlkBars bars;
    __shared__ uint32_t s_tmem;
    if (a.skip && *a.skip) return;
    const uint32_t tmem = blk_open(&s_tmem, &bars);
    const int m = blockIdx.x / a.blk_chunks;
    const int T = blk_synth_item(a, m, blockIdx.x - m * a.blk_chunks, blockIdx.y, smem, &bars, tmem);
    blk_close<false>(tmem, &bars, T);
}

__global__ void __launch_bounds__(BLK_THREADS, 2) k_leg_adjoint_blk(LegArgs<float> a)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    __shared__ BlkBars bars;
    __shared__ uint32_t s_tmem;
    if (a.skip && *a.skip) return;
    const uint32_t tmem = blk_open(&s_tmem, &bars);
    const int m = blockIdx.x / a.blk_chunks;
    const int T = blk_adjoint_item(a, m, blockIdx.x - m * a.blk_chunks, blockIdx.y, smem, &bars, tmem);
    blk_close<true>(tmem, &bars, T);
}

}  // namespace

void blk_tables_free(BlkTables &t)
{
    if (t.rows) cudaFree(t.rows);
    if (t.info) cudaFree(t.info);
    if (t.vtab) cudaFree(t.vtab);
    t = BlkTables();
}

// tables that hold any ring list of the plan (at plan creation, so that new weights allocate nothing)
akra_status blk_tables_alloc(akra_plan p, BlkTables &t)
{
    const size_t cap = p->nring, cch = (cap + BLK_RINGS - 1) / BLK_RINGS;
    const size_t bytes[3] = {sizeof(int) * cap, sizeof(BlkChunk) * cch, BLK_VBYTES * cch};
    if (cudaMalloc((void **)&t.rows, bytes[0]) != cudaSuccess || cudaMalloc((void **)&t.info, bytes[1]) != cudaSuccess ||
        cudaMalloc((void **)&t.vtab, bytes[2]) != cudaSuccess) {
        cudaGetLastError();
        blk_tables_free(t);
        set_error("plan table allocation failed");
        return AKRA_ENOMEM;
    }
    p->bytes_tables += bytes[0] + bytes[1] + bytes[2];
    return AKRA_OK;
}

akra_status blk_tables_build(akra_plan p, BlkTables &t, const std::vector<int> &rows, int npolar, cudaStream_t st)
{
    const int n = (int)rows.size(), nch = (n + BLK_RINGS - 1) / BLK_RINGS;
    t.nrows = n;
    t.nchunks = nch;
    t.npolar = npolar;
    if (n == 0) return AKRA_OK;
    AKRA_CUDA_TRY(cudaMemcpyAsync(t.rows, rows.data(), sizeof(int) * n, cudaMemcpyHostToDevice, st));
    AKRA_CUDA_TRY(cudaStreamSynchronize(st));   // the host list must outlive the copy
    k_blk_tables<<<nch, BLK_RINGS, 0, st>>>(n, p->nunit, p->nring, t.rows, p->d_units, t.info, (unsigned char *)t.vtab);
    AKRA_CUDA_TRY(cudaGetLastError());
    return AKRA_OK;
}

akra_status legendre_blk_prepare()
{
    AKRA_CUDA_TRY(cudaFuncSetAttribute(k_leg_synth_blk, cudaFuncAttributeMaxDynamicSharedMemorySize, BlkSynthSmem::BYTES));
    AKRA_CUDA_TRY(cudaFuncSetAttribute(k_leg_adjoint_blk, cudaFuncAttributeMaxDynamicSharedMemorySize, BlkAdjSmem::BYTES));
    return AKRA_OK;
}

akra_status legendre_synth_blk(akra_plan p, LegMode mode, const void *alm, void *phi, int R, const int *units,
                               cudaStream_t st)
{
    const BlkTables &t = blk_tables(p, units);
    if (t.nrows == 0) return AKRA_OK;
    LegArgs<float> a = leg_args<float>(p, LegShape{1, BLK_NT, 1}, mode, units, 0, R);
    a.alm = (const float2 *)alm;
    a.phi = (float2 *)phi;
    k_leg_synth_blk<<<dim3((unsigned)(p->lmax + 1) * t.nchunks, R), BLK_THREADS, BlkSynthSmem::BYTES, st>>>(a);
    AKRA_CUDA_TRY(cudaGetLastError());
    p->launches++;
    return AKRA_OK;
}

// partial sums of chunks 0 .. t.nchunks - 1 of an array of nchunks chunks
akra_status legendre_adjoint_blk(akra_plan p, const void *phi, void *partial, int R, const int *units, int nchunks,
                                 cudaStream_t st)
{
    const BlkTables &t = blk_tables(p, units);
    if (t.nrows == 0) return AKRA_OK;
    LegArgs<float> a = leg_args<float>(p, LegShape{1, BLK_NT, 1}, LegMode::Synth, units, 0, R);
    a.phi_in = (const float2 *)phi;
    a.partial = (float *)partial;
    a.nchunks = nchunks;
    k_leg_adjoint_blk<<<dim3((unsigned)(p->lmax + 1) * t.nchunks, R), BLK_THREADS, BlkAdjSmem::BYTES, st>>>(a);
    AKRA_CUDA_TRY(cudaGetLastError());
    p->launches++;
    return AKRA_OK;
}

AKRA_DEBUG_COLLECTOR(legendre_blk)

}  // namespace akra
