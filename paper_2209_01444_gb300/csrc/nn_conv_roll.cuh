// Implicit 3 x 3 convolution that walks down columns of the image (included by
// nn_gemm.cu).  A CTA takes a run of rows of 128-pixel tiles, column by column, and
// keeps every weight tile in shared memory.  Each input row is multiplied once per
// horizontal tap by the weights of all three vertical taps side by side: 3 BN
// columns whose sums go to the accumulators of the three output rows around it,
// neighbours in a ring of tensor memory.  k_gemm_ws reads the same 128 x 16 operand
// from shared memory three times for BN columns each, 40 cycles an MMA whether 32
// or 8 columns, and its narrow tiles ran at that pace (32 -> 32 channels at 4 x
// 512^2: 774 cycles a tile).  An output still gets its products by input row, tap
// and channel, as there, so the results are the same bits.  k_gemm_ws against this,
// us at 4 x 512^2: 32 -> 32 channels 39 and 29, 64 -> 32 59 and 41, 32 -> 64 65 and 40;
// 64 -> 64 at 4 x 256^2 22.7 and 19.8, 128 -> 64 there 36.4 and 28.4 (CBL = 2: two channel
// blocks, whose products k_gemm_ws's row-reuse form adds in this order too).  What is left is about 8 us of launch, set-up
// and last drain, and 19 us of DRAM for the 32 channels in and out.
//
// Warp 0 loads RT input rows a stage, warp 1 issues the MMAs, the others drain the
// output rows that a stage completes in units of 128 pixels x 32 columns, with the
// ReLU mask loaded one stage ahead.  Waits are bounded as in k_gemm_ws.

// Input rows a stage: as many as the tensor memory's 512 columns allow (output rows
// in the ring: two unfinished and RT of each of three stages), and one where two
// channel blocks (CBL) of weights leave no room for more.
template <int BN, int BK, int CBL>
constexpr int roll_rows()
{
    return CBL == 2 ? 1 : BN == 32 && BK == 32 ? 4 : 2;
}
template <int BN, int BK, int CBL>
constexpr int roll_block_bytes()  // a channel block of a stage's rows
{
    return (roll_rows<BN, BK, CBL>() * (kBM + 2) * BK * 2 + 1023) / 1024 * 1024;
}
template <int BN, int BK, int CBL>
constexpr int roll_stages()
{
    constexpr int n = (224 * 1024 - 9 * CBL * BN * BK * 2) / (CBL * roll_block_bytes<BN, BK, CBL>());
    return n > 6 ? 6 : n;
}
constexpr int kRollEpi = 8;  // epilogue warps: two groups of one per lane quarter
constexpr int kRollThreads = 64 + 32 * kRollEpi;

// A value that is the same in every lane, in a uniform register.
__device__ __forceinline__ int uniform(int v) { return __reduce_max_sync(0xffffffffu, v); }

// total: rows of tiles, nx to an image row, H to a column, columns image by image.
template <int BN, bool OUT_BF16, int BK, int CBL>
__global__ void __launch_bounds__(kRollThreads, 1)
    k_conv_roll(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, void* __restrict__ D,
                const float* __restrict__ bias, int N, int ldd, int relu, int W, int H, int nx, int total, ShuffleGeo sh)
{
    constexpr int RT = roll_rows<BN, BK, CBL>(), S = roll_stages<BN, BK, CBL>();
    constexpr int BLK = roll_block_bytes<BN, BK, CBL>(), STAGE = CBL * BLK;
    constexpr int ROW = (kBM + 2) * BK * 2;  // bytes of an input row's channel block
    constexpr int B_BYTES = BN * BK * 2;
    constexpr int NS = 512 / BN;  // output rows in tensor memory
    constexpr int G = 4;          // stages whose outputs are under way
    static_assert(NS >= 2 + 3 * RT && S >= 2, "output rows of three stages");
    constexpr int KS = BK / 16;
    constexpr uint32_t HI = tile_desc_hi<BK>();
    constexpr int UN = BN / 32;                        // units per tile
    constexpr int MU = UN == 2 ? RT : (RT + 1) / 2;    // units a warp has of a stage
    extern __shared__ uint8_t smem_raw[];
    uint8_t* wts = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);  // [block][kx][2 - ky][BN][BK]
    uint8_t* rows = wts + 9 * CBL * B_BYTES;
    uint64_t* full = (uint64_t*)(rows + S * STAGE);
    uint64_t* empty = full + S;
    uint64_t* acc_full = empty + S;
    uint64_t* acc_empty = acc_full + G;
    uint64_t* wfull = acc_empty + G;
    uint64_t* done = wfull + 1;
    uint32_t* tmem_slot = (uint32_t*)(done + 1);
    volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
    int* counts = (int*)(tmem_slot + 2);  // [0] stages loaded, [1] stages waited for

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int r0 = (int)((long long)total * blockIdx.x / gridDim.x);
    const int r1 = (int)((long long)total * (blockIdx.x + 1) / gridDim.x);
    // a segment: the CTA's output rows r .. r + n - 1 of one column, input rows
    // i = 0 .. n + 1 of it, output j complete with input j + 2
    auto segment = [&](int r) { return min(H - r % H, r1 - r); };

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        for (int a = 0; a < G; ++a) {
            mbar_init(&acc_full[a], 1);
            mbar_init(&acc_empty[a], 32 * kRollEpi);
        }
        mbar_init(wfull, 1);
        mbar_init(done, 1);
        *abort_flag = 0;
        counts[0] = counts[1] = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *tmem_slot;
    // released before the wait: a CTA fills its SM, so nothing of the next kernel is
    // resident ahead, and its launch is out of the way (3 x 512 x 384, 64 -> 32 channels,
    // call after call, 24.6 us against 26.2)
    lbm::pdl_release();
    lbm::pdl_wait();

    if (warp == 0) {  // ------------------------------------------- producer
        const uint32_t lead = elect_lane();
        if (lead) {
            mbar_expect_tx(wfull, 9 * CBL * B_BYTES);
            for (int t = 0; t < 9 * CBL; ++t) {  // tap t / CBL, channel block t % CBL
                const int ky = t / (3 * CBL), kx = t / CBL - 3 * ky;
                tma_load_2d(wts + ((t % CBL * 3 + kx) * 3 + 2 - ky) * B_BYTES, &tmB, t * BK, 0, wfull);
            }
        }
        int it = 0;
        bool ok = true;
        for (int r = r0, n; r < r1 && ok; r += n) {
            const int ci = r / H, y = r - ci * H, b = ci / nx, x0 = (ci - b * nx) * kBM;
            n = segment(r);
            for (int i = 0; i < n + 2; i += RT, ++it) {  // input rows from y - 1 + i on, zeros outside the image
                const int st = it % S;
                if (it >= S && !(ok = mbar_wait_warp(&empty[st], (uint32_t)((it / S - 1) & 1), abort_flag))) break;
                if (!lead) continue;
                mbar_expect_tx(&full[st], CBL * RT * ROW);
                for (int cb = 0; cb < CBL; ++cb)
                    tma_load_4d(rows + st * STAGE + cb * BLK, &tmA, cb * BK, x0 - 1, y + i - 1, b, &full[st]);
                counts[0] = it + 1;
            }
        }
    } else if (warp == 1) {  // ------------------------------------------- MMA
        const uint32_t lead = elect_lane();
        const unsigned long long lim = g_operand_wait_ns;
        const int u0 = uniform(r0), u1 = uniform(r1);
        const uint32_t ut = uniform(tmem);
        const uint32_t w0 = uniform(tile_desc_lo<BK>(smem_u32(wts))), a0 = uniform(tile_desc_lo<BK>(smem_u32(rows)));
        int st = 0, ph = 0, g = 0;
        // nb blocks of BN columns from block b on, K step ks (channel block, tap kx, channels
        // 16 k ..), rows at a
        auto mma = [&](int slot, uint32_t a, int b, int nb, int ks, uint32_t acc) {
            const int cb = ks / (3 * KS), kx = ks / KS % 3, k = ks % KS;
            umma_lead(lead, ut + (uint32_t)(slot * BN), a + ((cb * BLK + kx * BK * 2 + k * 32) >> 4), HI,
                      w0 + ((((cb * 3 + kx) * 3 + b) * B_BYTES + k * 32) >> 4), HI, idesc_bf16(kBM, BN * nb), acc);
        };
        bool ok = mbar_wait_warp(wfull, 0, abort_flag, lim);
        for (int r = u0, n; r < u1 && ok; r += n) {
            n = uniform(min(H - r % H, u1 - r));
            for (int i0 = 0; i0 < n + 2; i0 += RT, ++g) {
                if (g >= G - 1 && !(ok = mbar_wait_warp(&acc_empty[(g - G + 1) % G],
                                                        (uint32_t)(((g - G + 1) / G) & 1), abort_flag)))
                    break;
                if (!(ok = mbar_wait_warp(&full[st], (uint32_t)ph, abort_flag, lim))) break;
                if (lead) counts[1] = g + 1;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int rr = 0; rr < RT; ++rr) {
                    const int i = i0 + rr;
                    if (i >= n + 2) break;
                    const uint32_t a = a0 + (uint32_t)(st * (STAGE >> 4) + rr * (ROW >> 4));
                    // blocks lo .. hi - 1 of output rows i - 2 + block; block 2's is new
                    const int lo = i < 2 ? 2 - i : 0, hi = i < n ? 3 : n + 2 - i;
                    const int s0 = (r - u0 + i - 2) & (NS - 1);
                    if (lo == 0 && hi == 3 && s0 <= NS - 3) {
                        mma(s0, a, 0, 2, 0, 1);
                        mma(s0 + 2, a, 2, 1, 0, 0);
#pragma unroll
                        for (int ks = 1; ks < 3 * KS * CBL; ++ks) mma(s0, a, 0, 3, ks, 1);
                    } else {
                        // the rows of a segment's ends, and where the ring wraps: block by block
#pragma unroll
                        for (int ks = 0; ks < 3 * KS * CBL; ++ks)
#pragma unroll
                            for (int b = 0; b < 3; ++b)
                                if (b >= lo && b < hi)
                                    mma((s0 + b) & (NS - 1), a, b, 1, ks, ks == 0 && b == 2 ? 0u : 1u);
                    }
                }
                if (lead) {
                    umma_commit(&acc_full[g % G]);
                    umma_commit(&empty[st]);
                }
                __syncwarp();
                if (++st == S) st = 0, ph ^= 1;
            }
        }
        if (lead) umma_commit(done);  // completes once every MMA issued has finished
        __syncwarp();
    } else {  // --------------------------------------------------- epilogue
        const int q = warp & 3, grp = (warp - 2) >> 2, px = q * 32 + lane;
        const bool vec = N % 32 == 0;  // whole units
        const int c = grp % UN * 32;   // this warp's columns
        float bv[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) bv[j] = (bias && c + j < N) ? bias[c + j] : 0.0f;
        // the stage under way: outputs j0 .. j1 - 1 of the segment at r, whose first
        // row's pixel is p0 (-1: outside the image)
        int r = r0, n = 0, i0 = 0, j0 = 0, j1 = 0;
        long long p0 = -1;
        auto enter = [&] {  // the segment at r
            const int ci = r / H, y = r - ci * H, b = ci / nx, x = (ci - b * nx) * kBM + px;
            n = segment(r);
            i0 = 0;
            p0 = x < W ? ((long long)b * H + y) * W + x : -1;
        };
        // this warp's units: tiles j0 + t of every second tile, or of every one
        Mask16 mk[MU][2] = {};
        long long p[MU];
        int slot[MU];
        auto plan = [&](Mask16(&m)[MU][2], long long (&pp)[MU], int (&ss)[MU]) {
            j0 = i0 < 2 ? 0 : i0 - 2;
            j1 = min(i0 + RT, n + 2) - 2;
#pragma unroll
            for (int t = 0; t < MU; ++t) {
                const int j = j0 + (UN == 2 ? t : 2 * t + grp);
                ss[t] = j < j1 ? (r - r0 + j) & (NS - 1) : -1;
                pp[t] = j < j1 && p0 >= 0 && c < N ? p0 + (long long)j * W : -1;
                if (pp[t] >= 0 && sh.mask && vec) {
                    const __nv_bfloat16* mp = sh.mask + pp[t] * sh.mpitch + c;
                    m[t][0] = load_relu_mask(mp, true);
                    m[t][1] = load_relu_mask(mp + 16, true);
                }
            }
        };
        enter();
        plan(mk, p, slot);
        for (int g = 0; r < r1; ++g) {
            // the next stage's masks are loaded before this one's outputs are waited for
            Mask16 mn[MU][2] = {};
            long long pn[MU] = {};
            int sn[MU] = {};
            i0 += RT;
            if (i0 >= n + 2) {
                r += n;
                if (r < r1) enter();
            }
            if (r < r1) plan(mn, pn, sn);
            if (!mbar_wait_abort(&acc_full[g % G], (uint32_t)((g / G) & 1), abort_flag)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
            for (int t = 0; t < MU; ++t) {
                if (slot[t] < 0) continue;
                uint32_t v32[32];
                tmem_ld32(v32, tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(slot[t] * BN + c));
                tmem_wait32(v32);
                if (p[t] >= 0) {
                    float v[32];
#pragma unroll
                    for (int j = 0; j < 32; ++j) {
                        const float x = __uint_as_float(v32[j]) + bv[j];
                        v[j] = relu ? fmaxf(x, 0.0f) : x;
                    }
                    store_unit<OUT_BF16>(v, mk[t], sh.mask ? sh.mask + p[t] * sh.mpitch + c : nullptr, vec, p[t], c, N,
                                         D, p[t] * ldd + c, p[t] * ldd + c + 16, sh);
                }
                __syncwarp();
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            mbar_arrive(&acc_empty[g % G]);
#pragma unroll
            for (int t = 0; t < MU; ++t) {
                p[t] = pn[t];
                slot[t] = sn[t];
                mk[t][0] = mn[t][0];
                mk[t][1] = mn[t][1];
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        // every issued MMA completes before TMEM is freed; on an abort also
        // every issued copy lands before the CTA's shared memory goes away
        unsigned long long t0 = global_ns();
        bool fin = false;
        while (!(fin = (bool)mbar_try(done, 0)) && global_ns() - t0 < kWaitNs) {
        }
        if (!fin) atomicExch(&g_gemm_error, 1);
        if (*abort_flag) {
            mbar_wait(wfull, 0);
            for (int it = counts[1]; it < counts[0]; ++it) mbar_wait(&full[it % S], (uint32_t)((it / S) & 1));
        }
    }
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (warp == 1)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}
