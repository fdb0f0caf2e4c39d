// Weight gradient of a 3 x 3 zero-padded convolution straight from the NHWC
// input and output gradient (included by nn_gemm.cu, whose barrier, TMA and
// tcgen05 helpers it uses):
//   dW[n][t cin + c] = sum_p X[p shifted by tap t][c] dY[p][n],  t = 3 ky + kx.
//
// The contraction runs over pixels, so both operands are used as they lie in
// memory, channels contiguous ("MN-major" shared-memory tiles): no transposed
// copies of X or dY are written.  A K block is bk = 64 (or 32) pixels of one
// image row; a TMA box brings the bk + 2 pixels of CB channels around it, and
// serves the three horizontal taps from it: a pixel is one row of CB * 2 bytes,
// so tap kx is a start address kx rows further (the swizzle works on address
// bits).  An MMA has 128 rows: CB = 64 channels at two neighbouring kx, or 32
// channels at four, whose blocks lie one pixel apart (the leading byte offset);
// the row block of kx = 3 is not used.  A CTA takes one slice of the pixels, one
// block of CB channels and of BN columns, and KYS = 3 vertical taps (a box of
// three image rows) or, where that leaves SMs idle, one; its accumulators
// stay in tensor memory for the whole slice.  The slices and the order of the
// pixels within one are those of the GEMM over transposed copies
// (wgrad3_bf16), whose results these are bit for bit.
//
// What bounds it: L2 gives each X pixel three times (the vertical taps); an MMA
// of 32 or 64 columns reads its 4 KB of A from shared memory in about twice the
// time its products take.  Before, three transposed copies of X and one of dY
// were written per layer and each tap's tile was loaded by itself: 4 x 512^2, 32 ->
// 32 channels, 105 us of gather and 214 of GEMM, now 35; the layers of a training
// step, 1980 us in all, now 700.  One CTA for the three vertical taps as columns of
// one MMA would issue a third of the MMAs, but the slices, fixed by the order of the
// sums, would then fill 60 to 101 of the SMs.
//
// Warp 0 loads, warp 1 issues the MMAs, warps 2-5 store the accumulators.
// Every wait is bounded, as in k_gemm_ws.

struct WgradGeo {
    int cin, N;              // rows kept per tap, columns
    int H, nx, bk;           // image rows, K blocks per row, pixels of a K block
    int blocks, per_split;   // K blocks in all and per slice
    int ncb, nnb;            // channel and column blocks
};

template <int CB, int KYS>
constexpr int wg_region() { return ((66 * KYS + 2) * CB * 2 + 1023) / 1024 * 1024; }  // bytes of one K block's X box
template <int KYS>
constexpr int wg_blocks() { return KYS == 1 ? 2 : 1; }  // K blocks per stage
template <int CB, int BN, int KYS>
constexpr int wg_stage() { return wg_blocks<KYS>() * (wg_region<CB, KYS>() + 64 * BN * 2); }
// KYS = 1: two CTAs share an SM
template <int CB, int BN, int KYS>
constexpr int wg_stages()
{
    constexpr int n = (KYS == 1 ? 100 : 200) * 1024 / wg_stage<CB, BN, KYS>();
    return n > 8 ? 8 : n;
}

// Descriptor of an MN-major tile: K rows of ROWB bytes (128 or 64, the swizzle
// width) holding ROWB / 2 values of M or N, 8-row groups contiguous; the next
// ROWB / 2 values lie lbo bytes on.  Low and high words.
__device__ __forceinline__ uint32_t mn_desc_lo(uint32_t saddr, uint32_t lbo) { return (saddr >> 4) | (lbo >> 4 << 16); }
template <int ROWB>
__device__ __forceinline__ constexpr uint32_t mn_desc_hi()
{
    return (8u * ROWB >> 4) | (1u << 14) | ((ROWB == 128 ? 2u : 4u) << 29);
}

template <int CB, int BN, int KYS>
__global__ void __launch_bounds__(kWsThreads, KYS == 1 ? 2 : 1)
    k_wgrad(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmY,
            float* __restrict__ part, const WgradGeo geo)
{
    constexpr int S = wg_stages<CB, BN, KYS>(), STAGE = wg_stage<CB, BN, KYS>(), KBS = wg_blocks<KYS>();
    constexpr int REGION = wg_region<CB, KYS>();
    constexpr int XB = CB * 2, YB = BN * 2;  // bytes of a pixel's row in the X and dY tiles
    constexpr int YTILE = 64 * YB;
    constexpr int MG = CB / 32, NACC = KYS * MG;
    constexpr uint32_t TMEM_COLS = NACC * BN <= 32    ? 32
                                   : NACC * BN <= 64  ? 64
                                   : NACC * BN <= 128 ? 128
                                   : NACC * BN <= 256 ? 256
                                                      : 512;
    static_assert(NACC * BN <= 512 && STAGE % 1024 == 0 && S >= 2, "tile sizes");
    // both operands MN-major
    constexpr uint32_t IDESC = idesc_bf16(kBM, BN) | (1u << 15) | (1u << 16);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full = (uint64_t*)(smem + S * STAGE);
    uint64_t* empty = full + S;
    uint64_t* done = empty + S;
    uint32_t* tmem_slot = (uint32_t*)(done + 1);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
    int* counts = (int*)(tmem_slot + 2);  // [0] loads issued, [1] stages consumed

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cb = blockIdx.x % geo.ncb, nb = (blockIdx.x / geo.ncb) % geo.nnb;
    const int ky0 = KYS == 1 ? blockIdx.x / (geo.ncb * geo.nnb) : 0;
    const int b0 = blockIdx.y * geo.per_split, nblk = min(geo.blocks - b0, geo.per_split);
    const int nk = (nblk + KBS - 1) / KBS;

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        *abort_flag = 0;
        counts[0] = counts[1] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    lbm::pdl_begin();  // after the tensor memory is taken, as in k_gemm_ws

    if (warp == 0) {  // ------------------------------------------- producer
        const uint32_t lead = elect_lane();
        if (lead) {
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmX) : "memory");
            asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&tmY) : "memory");
        }
        const uint32_t tx = (uint32_t)((geo.bk + 2) * KYS * XB + geo.bk * YB);  // bytes per K block
        int xb = b0 % geo.nx, y = (b0 / geo.nx) % geo.H, im = b0 / (geo.nx * geo.H);
        for (int it = 0; it < nk; ++it) {
            const int st = it % S, nb_it = min(KBS, nblk - it * KBS);
            if (it >= S && !mbar_wait_warp(&empty[st], (uint32_t)((it / S - 1) & 1), abort_flag)) break;
            uint8_t* a = smem + st * STAGE;
            if (lead) mbar_expect_tx(&full[st], tx * nb_it);
            for (int b = 0; b < nb_it; ++b) {
                if (lead) {
                    tma_load_4d(a + b * REGION, &tmX, cb * CB, xb * geo.bk - 1, y + ky0 - 1, im, &full[st]);
                    tma_load_4d(a + KBS * REGION + b * YTILE, &tmY, nb * BN, xb * geo.bk, y, im, &full[st]);
                }
                if (++xb == geo.nx) {
                    xb = 0;
                    if (++y == geo.H) {
                        y = 0;
                        ++im;
                    }
                }
            }
            if (lead) counts[0] = it + 1;
            __syncwarp();
        }
    } else if (warp == 1) {  // ------------------------------------------ MMA
        const uint32_t lead = elect_lane();
        const unsigned long long lim = g_operand_wait_ns;
        const int steps = geo.bk / 16;
        const uint32_t pitch = (uint32_t)((geo.bk + 2) * XB >> 4);  // an image row of the box, 16-byte units
        constexpr uint32_t XHI = mn_desc_hi<XB>(), YHI = mn_desc_hi<YB>();
        for (int it = 0; it < nk; ++it) {
            const int st = it % S, nb_it = min(KBS, nblk - it * KBS);
            if (!mbar_wait_warp(&full[st], (uint32_t)((it / S) & 1), abort_flag, lim)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a0 = smem_u32(smem + st * STAGE);
            for (int b = 0; b < nb_it; ++b) {
                uint32_t p = mn_desc_lo(a0 + b * REGION, XB), q = mn_desc_lo(a0 + KBS * REGION + b * YTILE, 0);
                for (int s = 0; s < steps; ++s) {
#pragma unroll
                    for (int ky = 0; ky < KYS; ++ky)
#pragma unroll
                        for (int g = 0; g < MG; ++g)
                            umma_lead(lead, tmem + (uint32_t)((ky * MG + g) * BN), p + ky * pitch + (2 * g * XB >> 4), XHI,
                                      q, YHI, IDESC, (it > 0 || b > 0 || s > 0) ? 1u : 0u);
                    p += 16 * XB >> 4;
                    q += 16 * YB >> 4;
                }
            }
            if (lead) {
                umma_commit(&empty[st]);
                counts[1] = it + 1;
            }
            __syncwarp();
        }
        if (lead) umma_commit(done);  // completes once every MMA issued has finished
        __syncwarp();
    } else if (mbar_wait_abort(done, 0, abort_flag) && !*abort_flag) {  // -- epilogue
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int q = warp & 3, m = q * 32 + lane;
        const int ci = cb * CB + m % CB;
        float* out = part + (size_t)blockIdx.y * 9 * geo.cin * geo.N;
#pragma unroll 1
        for (int a = 0; a < NACC; ++a) {
            const int ky = ky0 + a / MG, kx = 2 * (a % MG) + m / CB;
            const bool keep = kx < 3 && ci < geo.cin;
            float* row = out + ((size_t)(3 * ky + kx) * geo.cin + ci) * geo.N + nb * BN;
#pragma unroll 1
            for (int c = 0; c < BN; c += 32) {
                uint32_t r[32];
                tmem_ld32(r, tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(a * BN + c));
                tmem_wait32(r);
                if (!keep) continue;
#pragma unroll
                for (int j = 0; j < 32; j += 8)
                    if (nb * BN + c + j < geo.N) store32(row + c + j, r + j);  // N is a multiple of 8
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        // every issued MMA completes before TMEM is freed; on an abort also
        // every issued copy lands before the CTA's shared memory goes away
        const unsigned long long t0 = global_ns();
        bool fin = false;
        while (!(fin = (bool)mbar_try(done, 0)) && global_ns() - t0 < kWaitNs) {
        }
        if (!fin) atomicExch(&g_gemm_error, 1);
        if (*abort_flag)
            for (int it = counts[1]; it < counts[0]; ++it) mbar_wait(&full[it % S], (uint32_t)((it / S) & 1));
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
}

// Split-K GEMM over pixels from operands as they lie in memory: part[z][m][n] =
// sum over the slice's pixels p of A[p][m] B[p][n] (FP32, M x N), A [P][M] and
// B [P][N] BF16 contiguous: the up-convolutions' weight gradient without
// transposed copies.  128 x BN tiles, K blocks of 64 pixels; the slices and their
// order are those of k_gemm over the transposes, whose partial sums these are
// bit for bit.
template <int BN>
constexpr int tn_stage() { return 64 * (128 + BN) * 2; }
template <int BN>
constexpr int tn_stages()
{
    constexpr int n = (BN <= 64 ? 100 : 200) * 1024 / tn_stage<BN>();
    return n > 8 ? 8 : n;
}

template <int BN>
__global__ void __launch_bounds__(kWsThreads, BN <= 64 ? 2 : 1)
    k_gemm_tn(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
              float* __restrict__ part, int M, int N, int blocks, int per_split)
{
    constexpr int S = tn_stages<BN>(), STAGE = tn_stage<BN>();
    constexpr int NB = BN > 64 ? BN / 64 : 1, YB = BN > 32 ? 128 : 64;  // B boxes and bytes of their rows
    constexpr int ABOX = 64 * 128, BBOX = 64 * YB;
    constexpr uint32_t IDESC = idesc_bf16(kBM, BN) | (1u << 15) | (1u << 16);
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint64_t* full = (uint64_t*)(smem + S * STAGE);
    uint64_t* empty = full + S;
    uint64_t* done = empty + S;
    uint32_t* tmem_slot = (uint32_t*)(done + 1);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
    int* counts = (int*)(tmem_slot + 2);  // [0] loads issued, [1] stages consumed

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int m0 = blockIdx.x * kBM, n0 = blockIdx.y * BN;
    const int b0 = blockIdx.z * per_split, nk = min(blocks - b0, per_split);
    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(done, 1);
        *abort_flag = 0;
        counts[0] = counts[1] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"((uint32_t)BN)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    lbm::pdl_begin();  // after the tensor memory is taken, as in k_gemm_ws

    if (warp == 0) {
        const uint32_t lead = elect_lane();
        for (int it = 0; it < nk; ++it) {
            const int st = it % S, p0 = (b0 + it) * 64;
            if (it >= S && !mbar_wait_warp(&empty[st], (uint32_t)((it / S - 1) & 1), abort_flag)) break;
            uint8_t* a = smem + st * STAGE;
            if (lead) {
                mbar_expect_tx(&full[st], STAGE);
#pragma unroll
                for (int j = 0; j < 2; ++j) tma_load_2d(a + j * ABOX, &tmA, m0 + 64 * j, p0, &full[st]);
#pragma unroll
                for (int j = 0; j < NB; ++j) tma_load_2d(a + 2 * ABOX + j * BBOX, &tmB, n0 + 64 * j, p0, &full[st]);
                counts[0] = it + 1;
            }
            __syncwarp();
        }
    } else if (warp == 1) {
        const uint32_t lead = elect_lane();
        const unsigned long long lim = g_operand_wait_ns;
        constexpr uint32_t AHI = mn_desc_hi<128>(), BHI = mn_desc_hi<YB>();
        for (int it = 0; it < nk; ++it) {
            const int st = it % S;
            if (!mbar_wait_warp(&full[st], (uint32_t)((it / S) & 1), abort_flag, lim)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a0 = smem_u32(smem + st * STAGE);
            const uint32_t alo = mn_desc_lo(a0, ABOX), blo = mn_desc_lo(a0 + 2 * ABOX, BBOX);
#pragma unroll
            for (int s = 0; s < 4; ++s)
                umma_lead(lead, tmem, alo + (16 * 128 * s >> 4), AHI, blo + (16 * YB * s >> 4), BHI, IDESC,
                          (it > 0 || s > 0) ? 1u : 0u);
            if (lead) {
                umma_commit(&empty[st]);
                counts[1] = it + 1;
            }
            __syncwarp();
        }
        if (lead) umma_commit(done);
        __syncwarp();
    } else if (mbar_wait_abort(done, 0, abort_flag) && !*abort_flag) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int q = warp & 3, row = m0 + q * 32 + lane;
        float* out = part + ((size_t)blockIdx.z * M + row) * N + n0;
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
            uint32_t r[32];
            tmem_ld32(r, tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c);
            tmem_wait32(r);
            if (row >= M) continue;
#pragma unroll
            for (int j = 0; j < 32; j += 8)
                if (n0 + c + j < N) store32(out + c + j, r + j);  // N is a multiple of 8
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned long long t0 = global_ns();
        bool fin = false;
        while (!(fin = (bool)mbar_try(done, 0)) && global_ns() - t0 < kWaitNs) {
        }
        if (!fin) atomicExch(&g_gemm_error, 1);
        if (*abort_flag)
            for (int it = counts[1]; it < counts[0]; ++it) mbar_wait(&full[it % S], (uint32_t)((it / S) & 1));
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)BN) : "memory");
}
