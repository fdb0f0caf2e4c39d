// Fused coupled step (phase field, solute, heat, flow), wall kernel and flow
// sub-step kernel for sm_103a.
//
// One coupled step n -> n+1 (Sec. 3, time-n macros for every model):
//   1. macros of Eqs. (15), (20), (23), (26) from the node's populations;
//   2. grad(phi) by the isotropic nine-point stencil on phi^n, which each CTA
//      builds in shared memory from the phi populations of its tile and a
//      one-node halo;
//   3. a_s and N of Eqs. (2)-(3) in the grain's crystal frame; Q of Eq. (5);
//      J_at of Eq. (7);
//   4. MRT collisions of the four models in moment space (Appendix B);
//   5. push streaming; phi uses the modified streaming of Eq. (13)/Remark 2,
//      f_i(x+c_i, t+1) = [f*_i(x) - (1 - a_s^2(x)) f_i(x+c_i, t)] / a_s^2(x),
//      whose f_i(x+c_i, t) is read from the same shared tile;
//   6. history (phi, Q, Cu, Hu at time n) is written in place for the
//      backward time differences of the next step.
// Periodic wrap is applied to every streaming destination; on non-periodic
// sides the wrapped values land on wall nodes, which the wall scheme then
// overwrites completely: the wall kernels after the step, or the next step of
// the same call as it loads them (coupled_tile).
#include <cuda_pipeline_primitives.h>
#include <cuda_runtime.h>
#include <stddef.h>

#include <type_traits>

#include "lbm_kernels.h"
#include "pdl.cuh"

namespace lbm {

namespace {

// The flow steps are launched as programmatic dependents (pdl.cuh).  The coupled
// steps are not: in a captured graph their launches cost little, and early CTAs
// took SM slots from the last wave (1024^2 0.7 % slower).

constexpr int kLocalGradIters = 2;  // fixed-point passes of the local grad(phi) scheme

__device__ __forceinline__ int mirror_or_wrap_local(int g, int n, int periodic, int local, int d)
{
    // Neighbour g = node + d seen from local index `local` of the node: a
    // periodic neighbour (or one inside the domain) is in the halo at
    // local + d; a non-periodic ghost is the mirror image at local - d.
    if (!periodic && (g < 0 || g >= n)) return local - d;
    return local + d;
}

#ifndef LBM_BATCH_WARPS
#define LBM_BATCH_WARPS 32  // resident warps per SM the batched kernel's register budget is sized for
#endif

#ifndef LBM_STEP_MIN_BLOCKS
#define LBM_STEP_MIN_BLOCKS 9  // resident CTAs of 128 threads per SM the register budget is sized for
                               // (56 registers; 36 warps hide more of the memory latency than 32)
#endif

// Non-equilibrium extrapolation (Guo et al.) on one side pair, applied to the
// freshly streamed buffer: pop(b) = pop^eq(boundary macros) + pop(f) -
// pop^eq(macros of f), f the first interior node.  `axis` 1: bottom/top rows
// over x in [xlo, xhi]; `axis` 0: left/right columns over every y.  The
// result depends on the interior node alone, so applying it twice changes
// nothing.
//
// Phase-field part: boundary populations fb from the interior populations ff,
// whose sum (node_macros' order) is p1f = phi_f + 1.
__device__ __forceinline__ void wall_phi(const StepParams& P, int type, const float (&ff)[5], float p1f,
                                         float (&fb)[5])
{
    const float p1b = type == 5 ? P.dir_phi + 1.0f : p1f;  // Dirichlet far field, else zero gradient
    float eb[5], ef[5];
    deq_phi(p1b, eb);
    deq_phi(p1f, ef);
#pragma unroll
    for (int i = 0; i < 5; ++i) fb[i] = eb[i] + ff[i] - ef[i];
}

// Flow, solute and heat parts from the interior node's macros m and
// populations n, g, h; the scalar parts only when !flow_only.
__device__ __forceinline__ void wall_rest(const StepParams& P, int axis, int type, const Macro& m,
                                          const float (&n)[5], const float (&g)[5], const float (&h)[9],
                                          float (&nb)[5], float (&gb)[5], float (&hb)[9], int flow_only)
{
    float ubx = 0.0f, uby = 0.0f, pb = m.p;
    if (type == 1) {  // inflow
        ubx = P.uin_x;
        uby = P.uin_y;
    } else if (type == 2) {  // outflow
        ubx = m.ux;
        uby = m.uy;
        pb = 0.0f;
    } else if (type == 3) {  // symmetry
        ubx = axis == 0 ? 0.0f : m.ux;
        uby = axis == 0 ? m.uy : 0.0f;
    }
    float eb[9], ef[9];
    deq_flow(pb, ubx, uby, eb);
    deq_flow(m.p, m.ux, m.uy, ef);
#pragma unroll
    for (int i = 0; i < 9; ++i) hb[i] = eb[i] + h[i] - ef[i];
    if (flow_only) return;

    float p1b = m.p1, dCb = m.dC, Ub = m.U, dthb = m.dth;
    if (type == 5) {  // Dirichlet far field
        p1b = P.dir_phi + 1.0f;
        Ub = P.dir_U;
        dCb = dC_of(Ub, p1b, P.k);
        dthb = P.dir_theta - P.theta_ref;
    }
    const float hp1b = h_plus_1(P.h_kind, p1b);
    const float Hb = (P.theta_ref + P.latent) + dthb - P.latent * hp1b;
    const float Cb = 1.0f + dCb, Cf = 1.0f + m.dC;
    const float sc = P.nsub;
    deq_C(dCb, (1.0f - 0.5f * p1b) * Ub, Cb * ubx * sc, Cb * uby * sc, eb);
    deq_C(m.dC, (1.0f - 0.5f * m.p1) * m.U, Cf * m.ux * sc, Cf * m.uy * sc, ef);
#pragma unroll
    for (int i = 0; i < 5; ++i) nb[i] = eb[i] + n[i] - ef[i];
    deq_H(dthb, P.latent * hp1b, Hb * ubx * sc, Hb * uby * sc, eb);
    deq_H(m.dth, P.latent * m.hp1, m.H * m.ux * sc, m.H * m.uy * sc, ef);
#pragma unroll
    for (int i = 0; i < 5; ++i) gb[i] = eb[i] + g[i] - ef[i];
}

// v as a store to plane q and a load would return it (16-bit storage rounds
// its planes; FP32 keeps v).
template <class Store>
__device__ __forceinline__ float stored(int q, float v)
{
    if constexpr (std::is_same<Store, StoreF32>::value) {
        return v;
    } else {
        if (Store::rest(q)) return v;
        return Conv<typename Store::T>::to(Conv<typename Store::T>::from(v * Store::scale(q))) * Store::inv_scale(q);
    }
}

// What the wall scheme gives the wall node (xw, yw) of a freshly streamed
// state whose wall passes (rows, then columns) have not run: its n, g and h in
// out[0..4], [5..9], [10..18], in the units the node update takes (rest
// populations unscaled).  A row node follows from its interior node; a column
// node from its interior node, which in a corner is itself a row node, as the
// row pass would store it.  Row nodes are rounded as the row pass stores them.
template <class Store>
__device__ __forceinline__ void wall_values(const StepParams& P, const void* __restrict__ src,
                                            const void* __restrict__ srcf, int xw, int yw, bool column, bool row,
                                            float* __restrict__ out)
{
    const int xi = !column ? xw : (xw == 0 ? 1 : P.nx - 2);
    const int yi = !row ? yw : (yw == 0 ? 1 : P.ny - 2);
    const long long oi = (long long)yi * P.pitch + xi;
    float f[5], n[5], g[5], h[9], fb[5], nb[5], gb[5], hb[9];
#pragma unroll
    for (int i = 0; i < 5; ++i) f[i] = Store::load(src, srcf, kF + i, oi, P);
#pragma unroll
    for (int i = 0; i < 5; ++i) n[i] = Store::load(src, srcf, kN + i, oi, P);
#pragma unroll
    for (int i = 0; i < 5; ++i) g[i] = Store::load(src, srcf, kG + i, oi, P);
#pragma unroll
    for (int i = 0; i < 9; ++i) h[i] = Store::load(src, srcf, kH + i, oi, P);
    // at most two extrapolations: the row's, then the column's
#pragma unroll 1
    for (int axis = row ? 1 : 0; axis >= (column ? 0 : 1); --axis) {
        const int side = axis ? (yw == 0 ? 2 : 3) : (xw == 0 ? 0 : 1);
        const Macro m = node_macros(f, n, g, h, P);
        wall_phi(P, P.bc[side], f, m.p1, fb);
        wall_rest(P, axis, P.bc[side], m, n, g, h, nb, gb, hb, 0);
#pragma unroll
        for (int i = 0; i < 5; ++i) f[i] = axis ? stored<Store>(kF + i, fb[i]) : fb[i];
#pragma unroll
        for (int i = 0; i < 5; ++i) n[i] = axis ? stored<Store>(kN + i, nb[i]) : nb[i];
#pragma unroll
        for (int i = 0; i < 5; ++i) g[i] = axis ? stored<Store>(kG + i, gb[i]) : gb[i];
#pragma unroll
        for (int i = 0; i < 9; ++i) h[i] = axis ? stored<Store>(kH + i, hb[i]) : hb[i];
    }
    out[0] = n[0];
    out[5] = g[0];
#pragma unroll
    for (int i = 1; i < 5; ++i) out[i] = n[i] * (float)Store::kSS;
#pragma unroll
    for (int i = 1; i < 5; ++i) out[5 + i] = g[i] * (float)Store::kSS;
#pragma unroll
    for (int i = 0; i < 9; ++i) out[10 + i] = h[i] * (float)Store::kSF;
}

// Per-node part of the coupled step for node (x, y) = tile-local (lx - 1, ly - 1):
// f, n, g, h are its populations at time n (n_1..n_4 and g_1..g_4 in units
// of 1/Store::kSS, h in units of 1/Store::kSF: the codec's push scales), the
// *_prev values its history;
// fs holds the tile's phi populations with a one-node halo, node (x, y) at
// column fx = lx - 1 + XO of rows of FW floats; ps holds phi on the tile and
// halo with node (x, y) at [ly][lx].  Collides, push-streams (the phase field
// by the modified streaming of Eq. 13) and writes the history.
template <class Store, bool GRAIN, bool WRITE_FB, int TYV, int FW, int XO>
__device__ __forceinline__ void coupled_node(const StepParams& P, void* __restrict__ dst, void* __restrict__ dstf,
                                             float* __restrict__ hist, float* __restrict__ fb, int x, int y,
                                             int lx, int ly, const float (&f)[5], const float (&n)[5],
                                             const float (&g)[5], const float (&h)[9], float phi_prev,
                                             float Q_prev, float Cux_prev, float Cuy_prev, float Hux_prev,
                                             float Huy_prev, bool grain_on, uint8_t gid,
                                             const float (&fs)[5][TYV + 2][FW],
                                             const float (&ps)[TYV + 2][TX + 2])
{
    const long long o = (long long)y * P.pitch + x;
    const int fx = lx - 1 + XO;

    constexpr int SS = Store::kSS, SF = Store::kSF;
    const Macro m = node_macros<SS, SF>(f, n, g, h, P);
    const float usx = m.ux * P.nsub, usy = m.uy * P.nsub;  // velocity of the scalar lattice

    float co = P.cos_o, so = P.sin_o;
    if (GRAIN && grain_on) {
        const float2 cs = P.grain_cs[gid];
        co = cs.x;
        so = cs.y;
    }
    float gx, gy;
    if (!P.grad_local) {
        // grad(phi): (1/cs^2) sum_i w_i c_i phi(x + c_i) over the D2Q9 neighbours
        const int xl = mirror_or_wrap_local(x - 1, P.nx, P.periodic_x, lx, -1);
        const int xr = mirror_or_wrap_local(x + 1, P.nx, P.periodic_x, lx, +1);
        const int yd = mirror_or_wrap_local(y - 1, P.ny, P.periodic_y, ly, -1);
        const int yu = mirror_or_wrap_local(y + 1, P.ny, P.periodic_y, ly, +1);
        const float pE = ps[ly][xr], pW = ps[ly][xl], pN = ps[yu][lx], pS = ps[yd][lx];
        const float pNE = ps[yu][xr], pNW = ps[yu][xl], pSE = ps[yd][xr], pSW = ps[yd][xl];
        // paired differences, so that mirror-symmetric neighbourhoods (a wall
        // ghost, a symmetric seed) give an exactly zero component
        gx = (pE - pW) * (1.0f / 3.0f) + ((pNE - pNW) + (pSE - pSW)) * (1.0f / 12.0f);
        gy = (pN - pS) * (1.0f / 3.0f) + ((pNE - pSE) + (pNW - pSW)) * (1.0f / 12.0f);
    } else {
        // local scheme of Sec. 3.1: grad(phi) = -(s1/cs^2)(sum_i c_i f_i + W0^2 N/tau0)
        // with s1 and N taken at grad(phi): two fixed-point passes from a_s = 1, N = 0
        const float jx = f[1] - f[3], jy = f[2] - f[4];
        const float k0 = P.kappa3 * (1.0f / 3.0f);
        float s1 = __fdividef(1.0f, P.kappa3 + 0.5f);
        gx = -3.0f * s1 * jx;
        gy = -3.0f * s1 * jy;
#pragma unroll
        for (int it = 0; it < kLocalGradIters; ++it) {
            float a1, nx_, ny_;
            anisotropy(gx, gy, P.eps, co, so, a1, nx_, ny_);
            s1 = __fdividef(1.0f, P.kappa3 * a1 * a1 + 0.5f);
            gx = -3.0f * s1 * (jx + k0 * nx_);
            gy = -3.0f * s1 * (jy + k0 * ny_);
        }
    }
    float as, Nx, Ny;
    anisotropy(gx, gy, P.eps, co, so, as, Nx, Ny);
    const float as2 = as * as;
    // 1/a_s^2 (a_s^2 within (1 - 3 eps)^2 .. (1 + eps)^2) and the phase-field
    // rate, by fast division (within 2 ulp; both denominators are O(1))
    const float ia = __fdividef(1.0f, as2);
    const float g2 = gx * gx + gy * gy;
    const float Q = coupling_Q(m.phi, P.theta_ref + m.dth, m.U, P);

    // ---- phase field: Eqs. (13)-(14), relaxation rate of Sec. 3.1
    float fo[5];
    {
        const float s1 = __fdividef(1.0f, P.kappa3 * as2 + 0.5f);
        const float S0 = (Q + 0.5f * as2 * (Q - Q_prev)) * P.inv_tau;
        const float ga = -(1.0f / 3.0f) * ia;
        collide_d2q5<1, SS>(f, m.p1, 0.0f, 0.0f, m.p1, s1, ga * Nx, ga * Ny, S0, fo);
    }
    // ---- solute: Eqs. (17)-(19) with J_at of Eq. (7)
    float no[5];
    {
        float Jx = 0.0f, Jy = 0.0f;
        if (!(g2 < kGradEps2)) {
            const float a = -0.35355339059327373f * P.W * (1.0f + (1.0f - P.k) * m.U) * (m.phi - phi_prev) *
                            rsqrtf(g2);
            Jx = a * gx;
            Jy = a * gy;
        }
        const float qt = 1.0f - 0.5f * m.p1;
        const float C = 1.0f + m.dC;
        const float Cux = C * usx, Cuy = C * usy;
        // sum_i c_i G_i = d_t(Cu) + cs^2 (U grad q~ + J_at/D), grad q~ = -grad(phi)/2
        const float Gx = (Cux - Cux_prev) + (1.0f / 3.0f) * (-0.5f * m.U * gx + Jx * P.inv_D);
        const float Gy = (Cuy - Cuy_prev) + (1.0f / 3.0f) * (-0.5f * m.U * gy + Jy * P.inv_D);
        collide_d2q5<SS, SS>(n, m.dC, Cux, Cuy, qt * m.U, P.s1C, Gx, Gy, 0.0f, no);
    }
    // ---- heat: Eqs. (21)-(23)
    float go[5];
    {
        const float Hux = m.H * usx, Huy = m.H * usy;
        collide_d2q5<SS, SS>(g, m.dH, Hux, Huy, m.dth, P.s1T, Hux - Hux_prev, Huy - Huy_prev, 0.0f, go);
    }
    // ---- flow: Eqs. (24)-(26)
    float ho[9];
    collide_flow<SF, SF>(h, m, P.s2u, ho);

    // ---- push streaming: the rest populations stay at o; every moving one
    // goes to the neighbour node (x + c_x, y + c_y), whose element index is a
    // row term plus a column term (three of each)
    const int xp = (x + 1 == P.nx) ? 0 : x + 1, xm = (x == 0) ? P.nx - 1 : x - 1;
    const int yp = (y + 1 == P.ny) ? 0 : y + 1, ym = (y == 0) ? P.ny - 1 : y - 1;
    {
        const long long rY = Store::mov_row(y, P), rP = Store::mov_row(yp, P), rM = Store::mov_row(ym, P);
        const int c0 = Store::mov_col(x), cP = Store::mov_col(xp), cM = Store::mov_col(xm);
        const long long d5[5] = {0, rY + cP, rP + c0, rY + cM, rM + c0};
        // modified streaming of the phase field: the destination's time-n
        // population sits in the shared tile (its halo is periodic-wrapped)
        const float ib = ia - 1.0f, ibs = ib * (float)SS;
        const float fd[5] = {fs[0][ly][fx], fs[1][ly][fx + 1], fs[2][ly + 1][fx], fs[3][ly][fx - 1],
                             fs[4][ly - 1][fx]};
        Store::store(dst, dstf, kF, o, fo[0] * ia - ib * fd[0], P);
        Store::store(dst, dstf, kN, o, no[0], P);
        Store::store(dst, dstf, kG, o, go[0], P);
#pragma unroll
        for (int i = 1; i < 5; ++i) Store::store_mov(dst, kF + i, d5[i], fo[i] * ia - ibs * fd[i]);
        // n_i and g_i go to the same neighbour (one word in 16-bit storage)
        const long long qY = Store::pair_row(y, P), qP = Store::pair_row(yp, P), qM = Store::pair_row(ym, P);
        const int p0 = Store::pair_col(x), pP = Store::pair_col(xp), pM = Store::pair_col(xm);
        const long long e5[5] = {0, qY + pP, qP + p0, qY + pM, qM + p0};
#pragma unroll
        for (int i = 1; i < 5; ++i) Store::store_pair(dst, i, e5[i], no[i], go[i]);
    }
    {
        const long long rY = Store::flow_row(y, P), rP = Store::flow_row(yp, P), rM = Store::flow_row(ym, P);
        const int c0 = Store::flow_col(x), cP = Store::flow_col(xp), cM = Store::flow_col(xm);
        const long long d9[9] = {rY + c0, rY + cP, rP + c0, rY + cM, rM + c0, rP + cP, rP + cM, rM + cM, rM + cP};
#pragma unroll
        for (int i = 0; i < 9; ++i) Store::store_flow(dstf, i, d9[i], ho[i]);
    }

    // ---- history of the backward differences
    hist_at(hist, 0, o) = m.phi;
    hist_at(hist, 1, o) = Q;
    hist_at(hist, 2, o) = (1.0f + m.dC) * usx;
    hist_at(hist, 3, o) = (1.0f + m.dC) * usy;
    hist_at(hist, 4, o) = m.H * usx;
    hist_at(hist, 5, o) = m.H * usy;
    if (WRITE_FB) fb[o] = m.Fy;
}


// One tile of the coupled step: the CTA (TX x TYV threads) updates the nodes
// [x0, x0 + TX) x [y0, y0 + TYV) of one domain.  GRAIN: the domain may carry a
// grain map (read when `grain` is not null).  All threads reach the barriers,
// so callers may loop over tiles.
//
// WALLS with wfix set: wall passes were left out after the previous step, and
// the tile applies their update to the wall cells it loads instead: kColumns,
// the left and right walls; kAllWalls, the bottom and top walls too (rows
// first: the corners belong to the columns).  Extrapolation depends on the first
// interior node alone, and the tile and its halo hold that node for every wall
// cell they hold, so the result is the passes' in FP32.  With 16-bit storage row
// values are rounded as the row pass stores them, column values (corners among them)
// are used as they are: the passes' but for that rounding.  (wall_node states the same
// update for the passes, wall_values and phi_cell for kAllWalls, the code under
// kColumns for the columns alone: what changes in one changes in all.)
enum Walls { kNoWalls, kColumns, kAllWalls };
template <class Store, bool GRAIN, bool WRITE_FB, int TYV, int WALLS = kNoWalls>
__device__ __forceinline__ void coupled_tile(const StepParams& P, const void* __restrict__ src,
                                             const void* __restrict__ srcf, void* __restrict__ dst,
                                             void* __restrict__ dstf, float* __restrict__ hist,
                                             const uint8_t* __restrict__ grain, float* __restrict__ fb, int x0,
                                             int y0, float (&fs)[5][TYV + 2][TX + 2], float (&ps)[TYV + 2][TX + 2],
                                             int wfix = 0)
{
    const int tx = threadIdx.x, ty = threadIdx.y;
    const int x = x0 + tx, y = y0 + ty;
    const bool active = x < P.nx && y < P.ny;
    // WALLS: C, H and flow populations of the tile's own wall nodes, computed
    // first, while no other values are held in registers
    const bool xwall_tile = WALLS && wfix && !P.periodic_x && (x0 == 0 || x0 + TX + 1 >= P.nx);
    const bool ywall_tile =
        WALLS == kAllWalls && wfix && !P.periodic_y && (y0 == 0 || y0 + TYV + 1 >= P.ny);
    constexpr bool ROWS = WALLS == kAllWalls;
    __shared__ float wcol[WALLS ? 2 : 1][WALLS ? TYV : 1][19];  // left and right columns
    __shared__ float wrow[ROWS ? 2 : 1][ROWS ? TX : 1][19];     // bottom and top rows, corners excepted
    if constexpr (WALLS) {
        static_assert(2 * TX + 2 * TYV <= TX * TYV && 2 * (TX + 2) <= TX * TYV && 2 * (TYV + 2) <= TX * TYV,
                      "wall thread ranges");
    }
    if constexpr (ROWS) {
        if (xwall_tile || ywall_tile) {
            const int tid = ty * TX + tx;
            if (ywall_tile && tid < 2 * TX) {
                const int side = tid / TX, yw = side ? P.ny - 1 : 0;
                if (yw >= y0 && yw < y0 + TYV && x < P.nx && (P.periodic_x || (x > 0 && x < P.nx - 1)))
                    wall_values<Store>(P, src, srcf, x, yw, false, true, wrow[side][tx]);
            }
            constexpr int T0 = 2 * TX;  // first of the columns' threads
            if (xwall_tile && tid >= T0 && tid < T0 + 2 * TYV) {
                const int side = (tid - T0) / TYV, r = (tid - T0) % TYV;
                const int xw = side ? P.nx - 1 : 0, yw = y0 + r;
                if (xw >= x0 && xw < x0 + TX && yw < P.ny)
                    wall_values<Store>(P, src, srcf, xw, yw, true, !P.periodic_y && (yw == 0 || yw == P.ny - 1),
                                       wcol[side][r]);
            }
            __syncthreads();  // keeps the loads below after the repair
        }
    }
    // (the columns alone in their own form: as a special case of the above, BF16
    // batches ran 0.6 to 2 % slower)
    if constexpr (WALLS == kColumns) {
        const int tid = ty * TX + tx;
        if (xwall_tile && tid < 2 * TYV) {
            const int side = tid / TYV, r = tid % TYV;
            const int xw = side == 0 ? 0 : P.nx - 1, xi = side == 0 ? 1 : P.nx - 2;
            const int yw = y0 + r;
            if (xw >= x0 && xw < x0 + TX && yw < P.ny) {
                const long long oi = (long long)yw * P.pitch + xi;
                float fi[5], ni[5], gi[5], hi[9], nbw[5], gbw[5], hbw[9];
#pragma unroll
                for (int i = 0; i < 5; ++i) fi[i] = Store::load(src, srcf, kF + i, oi, P);
#pragma unroll
                for (int i = 0; i < 5; ++i) ni[i] = Store::load(src, srcf, kN + i, oi, P);
#pragma unroll
                for (int i = 0; i < 5; ++i) gi[i] = Store::load(src, srcf, kG + i, oi, P);
#pragma unroll
                for (int i = 0; i < 9; ++i) hi[i] = Store::load(src, srcf, kH + i, oi, P);
                const Macro mi = node_macros(fi, ni, gi, hi, P);
                wall_rest(P, 0, P.bc[side], mi, ni, gi, hi, nbw, gbw, hbw, 0);
                // in the units the node update takes (rest populations unscaled)
                wcol[side][r][0] = nbw[0];
                wcol[side][r][5] = gbw[0];
#pragma unroll
                for (int i = 1; i < 5; ++i) wcol[side][r][i] = nbw[i] * (float)Store::kSS;
#pragma unroll
                for (int i = 1; i < 5; ++i) wcol[side][r][5 + i] = gbw[i] * (float)Store::kSS;
#pragma unroll
                for (int i = 0; i < 9; ++i) wcol[side][r][10 + i] = hbw[i] * (float)Store::kSF;
            }
        }
        if (xwall_tile) __syncthreads();  // keeps the loads below after the repair
    }
    // own-node loads first, so that they are in flight while the halo loads.
    // Every thread loads its own tile cell (x, y), wrapped into the grid when
    // the tile reaches past it (such cells serve as periodic neighbours of
    // the edge nodes); the first 2 (TX + 2) + 2 TYV threads load the halo ring.
    const long long o = active ? (long long)y * P.pitch + x : 0;
    int cx = x, cy = y;
    if (!active) {
        cx = cx >= P.nx ? wrap(cx, P.nx) : cx;
        cy = cy >= P.ny ? wrap(cy, P.ny) : cy;
    }
    const long long oc = active ? o : (long long)cy * P.pitch + cx;
    float f[5], n[5], g[5], h[9];
#pragma unroll
    for (int i = 0; i < 5; ++i) f[i] = Store::load(src, srcf, kF + i, oc, P);
    n[0] = Store::load(src, srcf, kN, o, P);
    g[0] = Store::load(src, srcf, kG, o, P);
#pragma unroll
    for (int i = 1; i < 5; ++i) Store::load_pair(src, i, o, n[i], g[i]);
#pragma unroll
    for (int i = 0; i < 9; ++i) h[i] = Store::load_flow(srcf, i, o);
    const float* hn = hist;
    const float phi_prev = hist_at(hn, 0, o);
    const float Q_prev = hist_at(hn, 1, o);
    const float Cux_prev = hist_at(hn, 2, o), Cuy_prev = hist_at(hn, 3, o);
    const float Hux_prev = hist_at(hn, 4, o), Huy_prev = hist_at(hn, 5, o);
    uint8_t gid = 0;
    if (GRAIN && grain) gid = grain[o];

    static_assert(2 * (TX + 2) + 2 * TYV <= TX * TYV, "halo ring thread range");
    const int tid = ty * TX + tx;
    if (tid < 2 * (TX + 2) + 2 * TYV) {
        int hx, hy;
        if (tid < 2 * (TX + 2)) {  // the rows below and above the tile, corners included
            hy = tid < TX + 2 ? 0 : TYV + 1;
            hx = tid < TX + 2 ? tid : tid - (TX + 2);
        } else {  // the columns left and right of it
            const int r = tid - 2 * (TX + 2);
            hx = r < TYV ? 0 : TX + 1;
            hy = 1 + (r < TYV ? r : r - TYV);
        }
        int gx = x0 - 1 + hx, gy = y0 - 1 + hy;
        gx = (gx < 0) ? gx + P.nx : (gx >= P.nx ? gx - P.nx : gx);
        gy = (gy < 0) ? gy + P.ny : (gy >= P.ny ? gy - P.ny : gy);
        if (gx >= P.nx) gx = wrap(gx, P.nx);  // domains narrower than a tile
        if (gy >= P.ny) gy = wrap(gy, P.ny);
        const long long oh = (long long)gy * P.pitch + gx;
        float sum = 0.0f;
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            const float v = Store::load(src, srcf, kF + i, oh, P);
            fs[i][hy][hx] = v;
            sum += v;
        }
        ps[hy][hx] = sum;
    }
    {
        float sum = 0.0f;
#pragma unroll
        for (int i = 0; i < 5; ++i) {
            fs[i][ty + 1][tx + 1] = f[i];
            sum += f[i];
        }
        ps[ty + 1][tx + 1] = sum;
    }
    __syncthreads();

    if constexpr (WALLS == kColumns) {
        if (xwall_tile) {
            // (side, row) of each wall column the tile holds: x = 0 (side 0)
            // at tile column 1 - x0, x = nx - 1 (side 1) at nx - x0
            const int tid = ty * TX + tx;
            if (tid < 2 * (TYV + 2)) {
                // phase-field populations and phi of a wall cell of the tile or its halo rows
                const int side = tid / (TYV + 2), hy = tid % (TYV + 2);
                const int hx = side == 0 ? 1 - x0 : P.nx - x0;
                if (hx >= 0 && hx <= TX + 1) {
                    const int hf = side == 0 ? hx + 1 : hx - 1;  // the interior node, never a wall (nx >= 4)
                    float ff[5], fbw[5];
#pragma unroll
                    for (int i = 0; i < 5; ++i) ff[i] = fs[i][hy][hf];
                    wall_phi(P, P.bc[side], ff, ff[0] + ff[1] + ff[2] + ff[3] + ff[4], fbw);
                    float sum = 0.0f;
#pragma unroll
                    for (int i = 0; i < 5; ++i) {
                        fs[i][hy][hx] = fbw[i];
                        sum += fbw[i];
                    }
                    ps[hy][hx] = sum;
                }
            }
            __syncthreads();
            if (active && (x == 0 || x == P.nx - 1)) {
                const int side = x == 0 ? 0 : 1;
#pragma unroll
                for (int i = 0; i < 5; ++i) f[i] = fs[i][ty + 1][tx + 1];  // as the repair left the tile
#pragma unroll
                for (int i = 0; i < 5; ++i) n[i] = wcol[side][ty][i];
#pragma unroll
                for (int i = 0; i < 5; ++i) g[i] = wcol[side][ty][5 + i];
#pragma unroll
                for (int i = 0; i < 9; ++i) h[i] = wcol[side][ty][10 + i];
            }
        }
    }
    if constexpr (ROWS) {
        // phase-field populations and phi of the wall cells of the tile and its
        // halo: rows (corners excepted), then columns
        const int tid = ty * TX + tx;
        auto phi_cell = [&](int side, int hy, int hx, int fy, int fx) {
            float ff[5], fbw[5];
#pragma unroll
            for (int i = 0; i < 5; ++i) ff[i] = fs[i][fy][fx];
            wall_phi(P, P.bc[side], ff, ff[0] + ff[1] + ff[2] + ff[3] + ff[4], fbw);
            float sum = 0.0f;
#pragma unroll
            for (int i = 0; i < 5; ++i) {
                const float v = side >= 2 ? stored<Store>(kF + i, fbw[i]) : fbw[i];
                fs[i][hy][hx] = v;
                sum += v;
            }
            ps[hy][hx] = sum;
        };
        if (ywall_tile) {
            if (tid < 2 * (TX + 2)) {
                const int side = tid / (TX + 2), hx = tid % (TX + 2);
                const int hy = side == 0 ? 1 - y0 : P.ny - y0;  // tile row of y = 0, y = ny - 1
                const int gx = x0 - 1 + hx;
                const bool corner = !P.periodic_x && (gx <= 0 || gx >= P.nx - 1);
                // the interior row is never a wall (ny >= 4)
                if (hy >= 0 && hy <= TYV + 1 && !corner) phi_cell(2 + side, hy, hx, side == 0 ? hy + 1 : hy - 1, hx);
            }
            __syncthreads();
        }
        if (xwall_tile) {
            if (tid < 2 * (TYV + 2)) {
                // x = 0 at tile column 1 - x0, x = nx - 1 at nx - x0
                const int side = tid / (TYV + 2), hy = tid % (TYV + 2);
                const int hx = side == 0 ? 1 - x0 : P.nx - x0;
                if (hx >= 0 && hx <= TX + 1) phi_cell(side, hy, hx, hy, side == 0 ? hx + 1 : hx - 1);
            }
            __syncthreads();
        }
        const bool on_col = xwall_tile && (x == 0 || x == P.nx - 1);
        const bool on_row = ywall_tile && (y == 0 || y == P.ny - 1);
        if (active && (on_col || on_row)) {
            const float* w = on_col ? wcol[x == 0 ? 0 : 1][ty] : wrow[y == 0 ? 0 : 1][tx];
#pragma unroll
            for (int i = 0; i < 5; ++i) f[i] = fs[i][ty + 1][tx + 1];  // as the repair left the tile
#pragma unroll
            for (int i = 0; i < 5; ++i) n[i] = w[i];
#pragma unroll
            for (int i = 0; i < 5; ++i) g[i] = w[5 + i];
#pragma unroll
            for (int i = 0; i < 9; ++i) h[i] = w[10 + i];
        }
    }

    if (!active) return;
    coupled_node<Store, GRAIN, WRITE_FB, TYV, TX + 2, 1>(P, dst, dstf, hist, fb, x, y, tx + 1, ty + 1, f, n, g, h,
                                                          phi_prev, Q_prev, Cux_prev, Cuy_prev, Hux_prev, Huy_prev,
                                                          grain != nullptr, gid, fs, ps);
}

// Resident CTAs per SM: see LBM_STEP_MIN_BLOCKS; kAllWalls with FP32 storage
// takes one less (64 registers), as its wall code spills at 56 (1024^2 forced
// flow 43.8 against 43.0 us per step; in 16-bit storage nine stay the faster).
template <class Store, bool GRAIN, bool WRITE_FB, int WALLS = kNoWalls>
__global__ void __launch_bounds__(TX* TY, LBM_STEP_MIN_BLOCKS -
                                              (WALLS == kAllWalls && std::is_same<Store, StoreF32>::value ? 1 : 0))
    k_coupled_step(const StepParams P, const void* __restrict__ src, const void* __restrict__ srcf,
                   void* __restrict__ dst, void* __restrict__ dstf, float* __restrict__ hist,
                   const uint8_t* __restrict__ grain, float* __restrict__ fb, int wfix = 0)
{
    __shared__ float fs[5][TY + 2][TX + 2];
    __shared__ float ps[TY + 2][TX + 2];
    coupled_tile<Store, GRAIN, WRITE_FB, TY, WALLS>(P, src, srcf, dst, dstf, hist, grain, fb, blockIdx.x * TX,
                                                    blockIdx.y * TY, fs, ps, wfix);
}

// Descriptors of the batch being stepped, in constant memory: the domain
// index is uniform across a CTA, so parameter reads are broadcast from the
// constant cache as in the single-domain kernel.  launch_batch_step copies the
// batch's table in before each step.
__constant__ DomainDesc c_batch_desc[kMaxBatchDomains];

// Batched coupled step: one persistent grid sweeps the tile table of every
// domain; each CTA takes a contiguous run of tiles, so consecutive tiles share
// the domain and their halos stay in L2.  A kernel boundary separates steps.
template <class Store, int TYV>
__global__ void __launch_bounds__(TX* TYV, (LBM_BATCH_WARPS / TYV > 0 ? LBM_BATCH_WARPS / TYV : 1))
    k_batch_step(const int4* __restrict__ tiles, int ntiles, int chunk, int parity, int wfix)
{
    __shared__ float fs[5][TYV + 2][TX + 2];
    __shared__ float ps[TYV + 2][TX + 2];
    const int t_end = min(ntiles, (blockIdx.x + 1) * chunk);
    for (int t = blockIdx.x * chunk; t < t_end; ++t) {
        const int4 tl = tiles[t];
        const DomainDesc& d = c_batch_desc[tl.x];
        coupled_tile<Store, true, false, TYV, kColumns>(d.P, d.sc[parity], d.fl[parity], d.sc[1 - parity],
                                                    d.fl[1 - parity], d.hist, d.grain, nullptr, tl.y, tl.z, fs, ps,
                                                    wfix);
        __syncthreads();  // the tile arrays are reused by the next tile
    }
}

// Flow populations the flow-only wall pass gives a wall node of `side` (axis
// 0: left/right columns, 1: bottom/top rows) from its interior node, whose flow
// populations are hi and whose phi + 1 and F_y (from its scalar populations)
// are sc.x and sc.y.
__device__ __forceinline__ void flow_wall_from(const StepParams& P, int axis, int side, float2 sc,
                                               const float (&hi)[9], float (&hb)[9])
{
    Macro m;
    m.p1 = sc.x;
    m.Fx = P.Fx;
    m.Fy = sc.y;
    flow_macros<1>(hi, m);
    const float none[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    float nb[5], gb[5];
    wall_rest(P, axis, P.bc[side], m, none, none, hi, nb, gb, hb, 1);
}

// phi + 1 and F_y of the node at offset o, from its scalar populations: node_macros'
// operations, each rounded as written (the compiler may contract those otherwise from
// kernel to kernel), so that every form of a flow step gives its walls the same bits.
template <class Store>
__device__ __forceinline__ float2 flow_wall_scalars(const StepParams& P, const void* __restrict__ sc, long long o)
{
    auto sum = [&](int q) {
        float v = Store::load(sc, nullptr, q, o, P);
#pragma unroll
        for (int i = 1; i < 5; ++i) v = __fadd_rn(v, Store::load(sc, nullptr, q + i, o, P));
        return v;
    };
    const float p1 = sum(kF), dC = sum(kN), dH = sum(kG);
    float hp1 = p1;
    if (P.h_kind == 1)  // h_plus_1
        hp1 = __fmul_rn(__fmul_rn(__fmul_rn(__fmul_rn(1.875f, p1), p1), p1),
                        __fmaf_rn(__fmul_rn(0.2f, p1), p1, __fsub_rn(4.0f / 3.0f, p1)));
    const float dth = __fmaf_rn(P.latent, hp1, dH);
    return make_float2(p1, __fmaf_rn(P.gbC, __fadd_rn(dC, P.dC_ref), __fmaf_rn(P.gbT, dth, P.Fy)));
}

// Collision of one flow step at a node: phi and the body force F_y frozen, h
// the node's populations; ho in units of 1/Store::kSF (as a store takes them).
template <class Store>
__device__ __forceinline__ void flow_collide(const StepParams& P, float phi, float fy, const float (&h)[9],
                                             float (&ho)[9])
{
    Macro m;
    m.phi = phi;
    m.p1 = m.phi + 1.0f;
    m.Fx = P.Fx;
    m.Fy = fy;
    flow_macros<1>(h, m);
    collide_flow<1, Store::kSF>(h, m, P.s2u, ho);
}

// The same with FP32 storage, with the sums that directions share taken once: of
// flow_macros and collide_flow 68 operations are left of 94.  F2: two nodes at once, in
// packed FP32 (one instruction for both; the packed form runs at half rate, so the FMA
// pipe, not the issue slots, sets the pace of a collision).  F1: one node, by the same
// operations in the same order, so that a step alone and several to a launch give the
// same bits.
struct F2 {
    float2 v;
    static __device__ __forceinline__ F2 of(float a) { return {make_float2(a, a)}; }
};
struct F1 {
    float v;
    static __device__ __forceinline__ F1 of(float a) { return {a}; }
};
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) { return {__ffma2_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ F2 operator+(F2 a, F2 b) { return {__fadd2_rn(a.v, b.v)}; }
__device__ __forceinline__ F2 operator-(F2 a, F2 b) { return fma2(b, F2::of(-1.0f), a); }
__device__ __forceinline__ F2 operator*(F2 a, F2 b) { return {__fmul2_rn(a.v, b.v)}; }
__device__ __forceinline__ F1 fma2(F1 a, F1 b, F1 c) { return {__fmaf_rn(a.v, b.v, c.v)}; }
__device__ __forceinline__ F1 operator+(F1 a, F1 b) { return {__fadd_rn(a.v, b.v)}; }
__device__ __forceinline__ F1 operator-(F1 a, F1 b) { return {__fsub_rn(a.v, b.v)}; }
__device__ __forceinline__ F1 operator*(F1 a, F1 b) { return {__fmul_rn(a.v, b.v)}; }

// nw: q~ - 1 = -(1 + phi)/2; hFy: half the body force along y.
template <class Store, class F>
__device__ __forceinline__ void flow_collide2(const StepParams& P, F nw, F hFy, const F (&h)[9], F (&out)[9])
{
    auto f2 = [](float a) { return F::of(a); };
    constexpr float SO = (float)Store::kSF;
    const F half = f2(0.5f), ns2 = f2(-P.s2u), hFx = f2(0.5f * P.Fx);
    const F a = h[5] - h[7], b = h[6] - h[8], e = h[5] + h[7], f = h[6] + h[8];
    const F s13 = h[1] + h[3], s24 = h[2] + h[4], d = e + f;
    const F usx = (h[1] - h[3]) + (a - b) + hFx, usy = (h[2] - h[4]) + (a + b) + hFy;  // u*
    const F mxx = s13 + d, myy = s24 + d, mxy = e - f, rest = mxx + s24;
    const F nt = nw * half;
    const F u = fma2(nt, usx, usx), v = fma2(nt, usy, usy);
    const F p = f2(0.6f) * fma2(f2(-(2.0f / 3.0f)), fma2(u, u, v * v), rest);
    // r1 = u + F'_x / 2 with F' = F + (1 - q~) f, f = -u*, and likewise r2
    const F r1 = u + fma2(nt, usx, hFx), r2 = v + fma2(nt, usy, hFy);
    const F pu = fma2(u, u, p);
    const F r3 = fma2(ns2, mxx - pu, mxx);
    const F r4 = fma2(ns2, myy - fma2(v, v, p), myy);
    const F r5 = fma2(ns2, fma2(u * f2(-1.0f), v, mxy), mxy);
    const F r8 = fma2(v, v, pu) * f2(1.0f / 3.0f);
    // (r1 - r7 along the axes, not its equal 2 r7: momentum is kept whatever the
    // rounding of 1/3)
    const F r6 = r2 * f2(1.0f / 3.0f), r7 = r1 * f2(1.0f / 3.0f);
    out[0] = f2(SO) * (r8 - (r3 + r4));
    const F hO = f2(0.5f * SO), ax = hO * (r3 - r8), ay = hO * (r4 - r8), bx = hO * (r1 - r7), by = hO * (r2 - r6);
    out[1] = ax + bx;
    out[3] = ax - bx;
    out[2] = ay + by;
    out[4] = ay - by;
    const F q = f2(0.25f * SO), s = q * (r6 + r7), t = q * (r6 - r7);
    const F c = q * (r8 + r5), g = q * (r8 - r5);
    out[5] = c + s;
    out[7] = c - s;
    out[6] = g + t;
    out[8] = g - t;
}

// The flow populations that the flow-only wall pass (rows, then columns) would have
// left at wall node (x, y) after the flow step before, which skipped it: a row node's
// from its interior node, a column node's from its interior node, which in a corner
// is itself a row node, as the row pass would store it.
template <class Store>
__device__ __forceinline__ void flow_wall_repair(const StepParams& P, const void* __restrict__ sc,
                                                 const void* __restrict__ src, int x, int y, bool column, bool row,
                                                 float (&h)[9])
{
    const int xi = !column ? x : (x == 0 ? 1 : P.nx - 2);
    const int yi = !row ? y : (y == 0 ? 1 : P.ny - 2);
    const long long oi = (long long)yi * P.pitch + xi;
    float hi[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) h[i] = Store::load(nullptr, src, kH + i, oi, P);
#pragma unroll 1
    for (int axis = row ? 1 : 0; axis >= (column ? 0 : 1); --axis) {
        // the column's own step reads the scalars of the node beside it
        const long long os = axis ? oi : (long long)y * P.pitch + xi;
#pragma unroll
        for (int i = 0; i < 9; ++i) hi[i] = h[i];
        flow_wall_from(P, axis, axis ? (y == 0 ? 2 : 3) : (x == 0 ? 0 : 1), flow_wall_scalars<Store>(P, sc, os), hi, h);
#pragma unroll
        for (int i = 0; i < 9; ++i) h[i] = stored<Store>(kH + i, h[i]);
    }
}

// One flow sub-step (two-time-scaling of Sec. 4): collide and stream h with phi
// and the force frozen at time n.
// phi: plane 0 of a node-block array of phi_np planes (the history, or the
// frozen phi of flow-only steps, phi_np = 1: a plain plane).  REPAIR: the flow step
// before left the flow-only wall pass out; wall nodes first take what it would have
// given them (sc: the newest scalar populations, whose macros it uses).
template <class Store, bool REPAIR>
__global__ void __launch_bounds__(256, 8) k_flow_substep(const StepParams P, const void* __restrict__ src,
                                                      void* __restrict__ dst, const float* __restrict__ phi,
                                                      int phi_np, const float* __restrict__ fb,
                                                      const void* __restrict__ sc)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    if (x >= P.nx || y >= P.ny) return;
    const long long o = (long long)y * P.pitch + x;
    float h[9], ho[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) h[i] = Store::load(nullptr, src, kH + i, o, P);
    if constexpr (REPAIR) {
        const bool column = !P.periodic_x && (x == 0 || x == P.nx - 1);
        const bool row = !P.periodic_y && (y == 0 || y == P.ny - 1);
        if (column || row) flow_wall_repair<Store>(P, sc, src, x, y, column, row, h);
    }
    const float ph = phi[block_index(o, phi_np)], fy = fb[o];
    if constexpr (std::is_same<Store, StoreF32>::value) {
        F1 h1[9], o1[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) h1[i].v = h[i];
        flow_collide2<Store>(P, F1{-0.5f * (ph + 1.0f)}, F1{0.5f * fy}, h1, o1);
#pragma unroll
        for (int i = 0; i < 9; ++i) ho[i] = o1[i].v;
    } else {
        flow_collide<Store>(P, ph, fy, h, ho);
    }
    const int xp = (x + 1 == P.nx) ? 0 : x + 1, xm = (x == 0) ? P.nx - 1 : x - 1;
    const int yp = (y + 1 == P.ny) ? 0 : y + 1, ym = (y == 0) ? P.ny - 1 : y - 1;
    const long long rY = Store::flow_row(y, P), rP = Store::flow_row(yp, P), rM = Store::flow_row(ym, P);
    const int c0 = Store::flow_col(x), cP = Store::flow_col(xp), cM = Store::flow_col(xm);
    const long long d9[9] = {rY + c0, rY + cP, rP + c0, rY + cM, rM + c0, rP + cP, rP + cM, rM + cM, rM + cP};
#pragma unroll
    for (int i = 0; i < 9; ++i) Store::store_flow(dst, i, d9[i], ho[i]);
}

// Several flow steps in one launch.  A step alone moves 80 bytes per node
// (FP32) for some 130 operations, so a step per launch is bound by L2 or HBM;
// here a CTA takes a region of kFmW x kFmH nodes and keeps its flow populations
// in shared memory for `ks` <= K steps.  The outermost nodes lose one ring per
// step (their neighbours are not in the region), so the CTA writes the inner
// (kFmW - 2 KX) x (kFmH - 2 K) nodes, which are exact (KX: K rounded up, so that
// regions start on a multiple of VW nodes).  Loads and stores of the populations
// move VW = 4 (K = 5: 2) nodes of a plane at a time, the loads straight into
// shared memory (cp.async): loading and storing took two thirds of a launch with
// a register and an instruction per value (1.12 M nodes, four steps: 46.5
// against 44 us; FP16 2.4 M nodes, 32 steps: 778 against 643 us, 697 with the
// single step's collision).
// Per step and node, each thread reads its own populations, collides (FP32: its rows
// in pairs, packed), and after a barrier pushes them to the neighbours'
// places, in the storage type (16-bit storage rounds at every step as a store
// to memory would).  Wall nodes take the values of the flow-only wall pass
// (rows, then columns) at the start of every step but the first (there when
// `repair` is set: the launch before left them out); the last step leaves them
// to the next launch or the pass.  more: another launch of the chain follows.
constexpr int kFmW = 64;   // region width: two warps
constexpr int kFmY = 8;    // rows of threads
constexpr int kFmR = 4;    // rows per thread
constexpr int kFmH = kFmY * kFmR;
constexpr int kFmB = 4;    // border columns left and right (groups of four stay aligned)
constexpr int kFmPW = kFmW + 2 * kFmB;
constexpr int fm_kx(int K) { return K == 5 ? 6 : (K + 3) / 4 * 4; }
template <int BYTES>
struct VecOf;
template <>
struct VecOf<4> { using V = uint32_t; };
template <>
struct VecOf<8> { using V = uint2; };
template <>
struct VecOf<16> { using V = uint4; };

// A flow population in shared memory: the storage type, in units of 1/kSF.
template <class Store>
__device__ __forceinline__ typename Store::T flow_enc(float vs)
{
    if constexpr (std::is_same<Store, StoreF32>::value)
        return vs;
    else
        return Conv<typename Store::T>::from(vs);
}
template <class Store>
__device__ __forceinline__ float flow_dec(typename Store::T v)
{
    if constexpr (std::is_same<Store, StoreF32>::value)
        return v;
    else
        return Conv<typename Store::T>::to(v) * (1.0f / Store::kSF);
}

// Region with its border, then two rows and two columns of wall scalars.
template <class Store>
constexpr int flow_multi_smem()
{
    return 9 * kFmPW * (kFmH + 2) * (int)sizeof(typename Store::T) + 2 * (kFmW + kFmH) * (int)sizeof(float2);
}

template <class Store, int K>
__global__ void __launch_bounds__(kFmW* kFmY, 2)
    k_flow_multi(const StepParams P, const void* __restrict__ src, void* __restrict__ dst,
                 const float* __restrict__ phi, int phi_np, const float* __restrict__ fb, const void* __restrict__ sc,
                 int ks, int repair, int more)
{
    static_assert(kFmR % 2 == 0, "rows in pairs");
    constexpr int KX = fm_kx(K);
    static_assert(kFmH > 2 * K && kFmW > 2 * KX, "region size");
    using T = typename Store::T;
    constexpr int NR = kFmR, RH = kFmH;
    // a border around the region takes what leaves it (never read), so that
    // every push is one store at a constant offset from the node
    constexpr int PW = kFmPW, PP = PW * (RH + 2), PJ = kFmY * PW;
    constexpr int kPush[9] = {0, 1, PW, -1, -PW, PW + 1, PW - 1, -PW - 1, -PW + 1};
    extern __shared__ float2 fm_smem[];
    float2* rowS = fm_smem;              // [2][kFmW] scalars of the row walls' interior nodes
    float2* colS = rowS + 2 * kFmW;      // [2][RH] and of the column walls'
    T* s = (T*)(colS + 2 * RH);          // [9][RH + 2][PW], node (lx, ly) at [ly + 1][lx + kFmB]

    const int lx = threadIdx.x, ty = threadIdx.y, t = ty * kFmW + lx;
    const int rx0 = blockIdx.x * (kFmW - 2 * KX) - KX, ry0 = blockIdx.y * (RH - 2 * K) - K;
    // node of this thread's column and rows; outside a wall there is none
    int gx = rx0 + lx;
    bool colx = true;
    if (P.periodic_x)
        gx = (gx < 0 || gx >= P.nx) ? wrap(gx, P.nx) : gx;
    else
        colx = gx >= 0 && gx < P.nx;
    const int margin = K - ks;  // rings the region has in excess
    T* const own = s + (ty + 1) * PW + lx + kFmB;  // row ty + kFmY j is PJ j further
    const bool walls = (!P.periodic_x && (rx0 <= 0 || rx0 + kFmW >= P.nx)) ||
                       (!P.periodic_y && (ry0 <= 0 || ry0 + RH >= P.ny));

    pdl_wait();
    if (more) pdl_release();  // the chain's next launch, of as many CTAs, at once; the wall pass at the end
    // FP32 collides two rows at once; with 16-bit storage each node does as in
    // k_flow_substep, to the bit: a rounding that falls the other way is 1e-4 of a field
    constexpr bool PACKED = std::is_same<Store, StoreF32>::value;
    float nw[NR], hfy[NR];  // PACKED: q~ - 1 and half the force; else phi and the force
    bool on[NR];
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        const int ly = ty + kFmY * j;
        int gy = ry0 + ly;
        bool rowy = true;
        if (P.periodic_y)
            gy = (gy < 0 || gy >= P.ny) ? wrap(gy, P.ny) : gy;
        else
            rowy = gy >= 0 && gy < P.ny;
        on[j] = colx && rowy && ly >= margin && ly < RH - margin;
        const long long o = on[j] ? (long long)gy * P.pitch + gx : 0;
        const float ph = phi[block_index(o, phi_np)], fy = fb[o];
        nw[j] = PACKED ? -0.5f * (ph + 1.0f) : ph;
        hfy[j] = PACKED ? 0.5f * fy : fy;
    }
    // the region's populations, groups of VW nodes of a row and plane; rx0 is a
    // multiple of VW, so a group inside the row lies in one node block
    constexpr int VW = KX % 4 == 0 ? 4 : 2, G = kFmW / VW, GB = VW * (int)sizeof(T);
    for (int q = t; q < G * RH; q += kFmW * kFmY) {
        const int ly = q / G, c = VW * (q % G);
        int y = ry0 + ly, x = rx0 + c;
        if (P.periodic_y)
            y = (y < 0 || y >= P.ny) ? wrap(y, P.ny) : y;
        else
            y = min(max(y, 0), P.ny - 1);  // (rows outside a wall are not used)
        T* d = s + (ly + 1) * PW + c + kFmB;
        if (!P.periodic_x) x = min(max(x, 0), P.pitch - VW);  // (nor are columns)
        if (!P.periodic_x || (x >= 0 && x + VW <= P.nx)) {
            const T* e = (const T*)src + block_index((long long)y * P.pitch + x, 9);
#pragma unroll
            for (int i = 0; i < 9; ++i) __pipeline_memcpy_async(d + i * PP, e + 32 * i, GB);
        } else {
            for (int k = 0; k < VW; ++k) {
                const T* e = (const T*)src + block_index((long long)y * P.pitch + wrap(x + k, P.nx), 9);
#pragma unroll
                for (int i = 0; i < 9; ++i) d[i * PP + k] = e[32 * i];
            }
        }
    }
    __pipeline_commit();
    // thread t's wall nodes in the wall pass: t < 2 kFmW a row wall's node in
    // this thread's column (the corners belong to the columns), the next 2 RH
    // threads a column wall's node
    int wrow = -1, wcol = -1;  // position of the node (row wall), of the node (column wall), or -1
    int wside = 0, win = 0;    // wall side; offset of the interior node
    if (walls) {
        if (!P.periodic_y && t < 2 * kFmW) {
            const int side = t / kFmW, ly = (side ? P.ny - 1 : 0) - ry0;
            if (ly >= 0 && ly < RH && colx && (P.periodic_x || (gx > 0 && gx < P.nx - 1))) {
                wrow = (ly + 1) * PW + lx + kFmB;
                wside = 2 + side;
                win = side ? -PW : PW;
                rowS[t] = flow_wall_scalars<Store>(P, sc, (long long)(side ? P.ny - 2 : 1) * P.pitch + gx);
            }
        }
        const int r = t - 2 * kFmW;
        if (!P.periodic_x && r >= 0 && r < 2 * RH) {
            const int side = r / RH, ly = r - side * RH, cx = (side ? P.nx - 1 : 0) - rx0;
            int yy = ry0 + ly;
            if (P.periodic_y) yy = wrap(yy, P.ny);
            if (cx >= 0 && cx < kFmW && yy >= 0 && yy < P.ny) {
                wcol = (ly + 1) * PW + cx + kFmB;
                wside = side;
                win = side ? -1 : 1;
                colS[r] = flow_wall_scalars<Store>(P, sc, (long long)yy * P.pitch + (side ? P.nx - 2 : 1));
            }
        }
    }
    auto wall_pass = [&](int w, int axis, float2 scal) {
        if (w < 0) return;
        float hi[9], hb[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) hi[i] = flow_dec<Store>(s[i * PP + w + win]);
        flow_wall_from(P, axis, wside, scal, hi, hb);
#pragma unroll
        for (int i = 0; i < 9; ++i) s[i * PP + w] = flow_enc<Store>(hb[i] * Store::kSF);
    };
    __pipeline_wait_prior(0);
    __syncthreads();

    for (int k = 0;; ++k) {
        if (walls && (k > 0 || repair)) {
            wall_pass(wrow, 1, wrow >= 0 ? rowS[t] : make_float2(0.0f, 0.0f));
            __syncthreads();
            wall_pass(wcol, 0, wcol >= 0 ? colS[t - 2 * kFmW] : make_float2(0.0f, 0.0f));
            __syncthreads();
        }
        F2 ho[NR / 2][9];
#pragma unroll
        for (int j = 0; j < NR; j += 2) {
            if constexpr (PACKED) {
                F2 h[9];
#pragma unroll
                for (int i = 0; i < 9; ++i) h[i].v = make_float2(own[i * PP + PJ * j], own[i * PP + PJ * (j + 1)]);
                flow_collide2<Store>(P, F2{make_float2(nw[j], nw[j + 1])}, F2{make_float2(hfy[j], hfy[j + 1])}, h,
                                     ho[j / 2]);
            } else {
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    float h[9], o9[9];
#pragma unroll
                    for (int i = 0; i < 9; ++i) h[i] = flow_dec<Store>(own[i * PP + PJ * (j + r)]);
                    flow_collide<Store>(P, nw[j + r], hfy[j + r], h, o9);
#pragma unroll
                    for (int i = 0; i < 9; ++i) (r ? ho[j / 2][i].v.y : ho[j / 2][i].v.x) = o9[i];
                }
            }
        }
        __syncthreads();
#pragma unroll
        for (int j = 0; j < NR; ++j) {
            // rows whose populations are exact at this step
            const int ly = ty + kFmY * j;
            if (!on[j] || ly < margin + k || ly >= RH - margin - k) continue;
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                const float2 v = ho[j / 2][i].v;
                own[i * PP + PJ * j + kPush[i]] = flow_enc<Store>(j & 1 ? v.y : v.x);
            }
        }
        __syncthreads();
        if (k + 1 == ks) break;
    }
    if (!more) pdl_release();
    using V = typename VecOf<GB>::V;
    constexpr int GO = (kFmW - 2 * KX) / VW, RO = RH - 2 * K;
    for (int q = t; q < GO * RO; q += kFmW * kFmY) {
        const int ly = K + q / GO, c = KX + VW * (q % GO), x = rx0 + c, y = ry0 + ly;
        if (x >= P.nx || y >= P.ny) continue;
        const T* e = s + (ly + 1) * PW + c + kFmB;
        T* d = (T*)dst + block_index((long long)y * P.pitch + x, 9);
        if (x + VW <= P.nx) {
#pragma unroll
            for (int i = 0; i < 9; ++i) *(V*)(d + 32 * i) = *(const V*)(e + i * PP);
        } else {
            for (int k = 0; x + k < P.nx; ++k)
#pragma unroll
                for (int i = 0; i < 9; ++i) d[32 * i + k] = e[i * PP + k];
        }
    }
}

template <class Store, int K>
cudaError_t launch_flow_multi(const StepParams& P, const void* src, void* dst, const float* phi, int phi_np,
                              const float* fb, const void* sc, int ks, int repair, int more, cudaStream_t s)
{
    constexpr int ow = kFmW - 2 * fm_kx(K), oh = kFmH - 2 * K, smem = flow_multi_smem<Store>();
    if (smem > 48 * 1024) {
        const cudaError_t e =
            cudaFuncSetAttribute(k_flow_multi<Store, K>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e != cudaSuccess) return e;
    }
    const dim3 grid((P.nx + ow - 1) / ow, (P.ny + oh - 1) / oh);
    return launch_pdl(k_flow_multi<Store, K>, grid, dim3(kFmW, kFmY), smem, s, P, src, dst, phi, phi_np, fb, sc, ks,
                      repair, more);
}

// Steps per launch for n >= 2 flow steps on an nx x ny grid, or 1 for node by node
// (the same bits).  In us: a launch of several steps costs about its steps plus 8 of
// them for loading, the walls' scalars and storing (5 where every region has an SM to itself),
// once for each wave of two CTAs per SM that the regions fill (15 flow steps at 1024^2:
// K = 4 fills 3 waves and K = 5 four, 818 and 834 us per four coupled steps; at 100^2,
// one wave, 222 and 205 us).
//
// Node by node a step costs its launch and about 3 for each 64 warps per SM.  In a
// replayed graph (`captured`) that launch is 1.6, and a step's wall repair 0.8 more with
// rows and 1.5 with columns: the faster on small grids with few steps (coupled steps of
// n_sub = 3 at 48^2, no walls, 6.3 us against 9.8 in regions, n_sub = 9 16.6 and 19.5).
// With walls on both axes it gains little (n_sub = 3 19.3 and 20.8, n_sub = 9 36 and 33)
// and an inflow's corners may round otherwise in the last bit.  Launched directly it is 4 (3 with
// 16-bit storage), which pays only on long strips, of which a region covers little more than half
// its nodes (14 steps of 262140 x 4 nodes, no walls: 190 us against 572 in regions, FP16
// 180 against 704); not on tall strips with walls at their sides, whose nodes
// a warp of a step finds one to a row (16 x 65536, FP32: 32 steps 1477 and 1086).
template <class Store>
int flow_multi_k(const StepParams& P, int n, bool captured)
{
    constexpr bool F32 = std::is_same<Store, StoreF32>::value;
    const int nx = P.nx, ny = P.ny;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int best = 2;
    long long least = 0, regions = 1;
    for (int K : {2, 4, 5}) {
        const int ow = kFmW - 2 * fm_kx(K), oh = kFmH - 2 * K;
        const long long tiles = (long long)((nx + ow - 1) / ow) * ((ny + oh - 1) / oh);
        const long long cost = (tiles + 2 * sms - 1) / (2 * sms) * (8 * ((n + K - 1) / K) + n);
        if (least == 0 || cost < least) {
            least = cost;
            best = K;
            regions = tiles;
        }
    }
    const double waves = (double)ny * ((nx + 31) / 32) / (64.0 * sms);
    if (captured && (P.periodic_x || P.periodic_y)) {
        const double cost = regions <= sms ? 5.2 * ((n + best - 1) / best) + 0.9 * n : (double)least;
        const double wall = !P.periodic_x ? 1.5 + 3e-4 * ny : !P.periodic_y ? 0.8 : 0.0;
        if (n * (1.6 + 3.0 * waves) + (n - 1) * wall < 1.1 * cost) return 1;
    } else if (regions > 2 * sms && 1.8 * nx * ny < (double)(regions * kFmW * kFmH) && (P.periodic_x || nx >= ny)) {
        if (n * ((F32 ? 4.0 : 3.0) + (F32 ? 3.2 : 2.8) * waves) < (double)least) return 1;
    }
    return best;
}

// n flow steps from buffer fl[*cf] (parity updated), the flow-only wall pass
// left out after the last.  A single step has no traffic to save and goes
// node by node; more are shared out evenly over the fewest launches.
template <class Store>
cudaError_t flow_chain(const StepParams& P, int n, const void* sc, void* const fl[2], int* cf, const float* phi,
                       int phi_np, const float* fb, cudaStream_t s)
{
    cudaError_t e = cudaSuccess;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (n > 1 && (e = cudaStreamIsCapturing(s, &cap)) != cudaSuccess) return e;
    const int K = n == 1 ? 1 : flow_multi_k<Store>(P, n, cap == cudaStreamCaptureStatusActive);
    if (K == 1) {
        const dim3 block(64, 4), grid((P.nx + 63) / 64, (P.ny + 3) / 4);
        for (int k = 0; k < n && e == cudaSuccess; ++k) {
            const auto step = k > 0 && !(P.periodic_x && P.periodic_y) ? k_flow_substep<Store, true> : k_flow_substep<Store, false>;
            step<<<grid, block, 0, s>>>(P, fl[*cf], fl[1 - *cf], phi, phi_np, fb, sc);
            *cf = 1 - *cf;
            e = cudaGetLastError();
        }
        return e;
    }
    int repair = 0;
    for (int left = (n + K - 1) / K; left > 0 && e == cudaSuccess; --left) {
        const int ks = (n + left - 1) / left;
        const auto launch = K == 2   ? launch_flow_multi<Store, 2>
                            : K == 4 ? launch_flow_multi<Store, 4>
                                     : launch_flow_multi<Store, 5>;
        e = launch(P, fl[*cf], fl[1 - *cf], phi, phi_np, fb, sc, ks, repair, left > 1, s);
        n -= ks;
        repair = 1;
        *cf = 1 - *cf;
    }
    return e;
}

template <class Store>
__device__ __forceinline__ void wall_node(const StepParams& P, void* __restrict__ pop, void* __restrict__ popf,
                                          int axis, int which, int j, int flow_only)
{
    const int side = axis == 0 ? which : 2 + which;
    if (P.bc[side] == 0) return;
    int xb, yb, xf, yf;
    if (axis == 0) {
        yb = yf = j;
        xb = which ? P.nx - 1 : 0;
        xf = which ? P.nx - 2 : 1;
    } else {
        xb = xf = j;
        yb = which ? P.ny - 1 : 0;
        yf = which ? P.ny - 2 : 1;
    }
    const long long ob = (long long)yb * P.pitch + xb, of = (long long)yf * P.pitch + xf;
    float f[5], n[5], g[5], h[9];
#pragma unroll
    for (int i = 0; i < 5; ++i) f[i] = Store::load(pop, popf, kF + i, of, P);
#pragma unroll
    for (int i = 0; i < 5; ++i) n[i] = Store::load(pop, popf, kN + i, of, P);
#pragma unroll
    for (int i = 0; i < 5; ++i) g[i] = Store::load(pop, popf, kG + i, of, P);
#pragma unroll
    for (int i = 0; i < 9; ++i) h[i] = Store::load(pop, popf, kH + i, of, P);
    const Macro m = node_macros(f, n, g, h, P);
    const int type = P.bc[side];
    float fb[5], nb[5], gb[5], hb[9];
    wall_rest(P, axis, type, m, n, g, h, nb, gb, hb, flow_only);
#pragma unroll
    for (int i = 0; i < 9; ++i) Store::store(pop, popf, kH + i, ob, hb[i], P);
    if (flow_only) return;
    wall_phi(P, type, f, m.p1, fb);
#pragma unroll
    for (int i = 0; i < 5; ++i) Store::store(pop, popf, kF + i, ob, fb[i], P);
#pragma unroll
    for (int i = 0; i < 5; ++i) Store::store(pop, popf, kN + i, ob, nb[i], P);
#pragma unroll
    for (int i = 0; i < 5; ++i) Store::store(pop, popf, kG + i, ob, gb[i], P);
}

template <class Store>
__global__ void k_walls(const StepParams P, void* __restrict__ pop, void* __restrict__ popf, int axis, int lo,
                        int count, int flow_only)
{
    pdl_begin();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 2 * count) return;
    const int which = t / count;           // 0: low side, 1: high side
    wall_node<Store>(P, pop, popf, axis, which, lo + (t - which * count), flow_only);
}

// Batched walls: one thread per entry {domain, axis, side, index} of a list
// holding one axis of every domain.
template <class Store>
__global__ void k_batch_walls(const DomainDesc* __restrict__ descs, const int4* __restrict__ nodes, int count,
                              int parity)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= count) return;
    const int4 e = nodes[t];
    const DomainDesc& d = descs[e.x];
    wall_node<Store>(d.P, d.sc[parity], d.fl[parity], e.y, e.z, e.w, 0);
}

// Rows (bottom/top walls, x in [1, nx - 2] when x is not periodic), then,
// with `columns`, the left/right columns over every y (corners included).
template <class Store>
cudaError_t walls(const StepParams& P, void* sc, void* fl, int flow_only, cudaStream_t s, bool columns = true)
{
    cudaError_t e = cudaSuccess;
    if (!P.periodic_y) {
        const int lo = P.periodic_x ? 0 : 1, hi = P.periodic_x ? P.nx - 1 : P.nx - 2;
        const int count = hi - lo + 1;
        e = launch_pdl(k_walls<Store>, (2 * count + 127) / 128, 128, 0, s, P, sc, fl, 1, lo, count, flow_only);
    }
    if (e == cudaSuccess && !P.periodic_x && columns) {
        e = launch_pdl(k_walls<Store>, (2 * P.ny + 127) / 128, 128, 0, s, P, sc, fl, 0, 0, P.ny, flow_only);
    }
    return e;
}

template <class Store>
cudaError_t flow_steps_t(const StepParams& P, int n, void* sc, void* const fl[2], int* cf, const float* phi,
                         const float* fy, cudaStream_t s)
{
    // wall pass after the last step only; each later step repairs the wall
    // nodes it loads instead
    if (n < 1) return cudaSuccess;
    cudaError_t e = flow_chain<Store>(P, n, sc, fl, cf, phi, 1, fy, s);
    if (e == cudaSuccess) e = walls<Store>(P, sc, fl[*cf], 1, s);
    return e;
}

constexpr long long kFoldNodes = 1 << 20;

template <class Store>
cudaError_t coupled_step(const StepParams& P, int n_sub, StepBuffers& B, cudaStream_t s, int repair, int skip_walls)
{
    const dim3 block(TX, TY), grid((P.nx + TX - 1) / TX, (P.ny + TY - 1) / TY);
    const void* src = B.sc[B.cs];
    const void* srcf = B.fl[B.cf];
    void* dst = B.sc[1 - B.cs];
    void* dstf = B.fl[1 - B.cf];
    const bool grain = B.grain != nullptr, wfb = n_sub > 1;
    if (B.ev_begin && !B.ev_substeps) cudaEventRecord(B.ev_begin, s);
    // walls: with skip_walls wall passes are left out and the next step,
    // launched with `repair`, updates the walls as it loads them
    // (coupled_tile); only steps with one flow step per coupled step do that:
    // flow sub-steps start from updated walls.  With walls at the bottom and top every
    // pass is left out up to kFoldNodes: two launches of few threads cost more than the
    // wall code in the step (100^2 forced flow 5.9 -> 4.4 us per step, 777 x 500 16.0 ->
    // 14.7); otherwise only the columns' strided pass.  The line is where FP16 stops
    // gaining: rows left to the step against the row pass, us per step with walls all round
    //          724^2              1024^2             1448^2             2048^2
    //   FP32   21.0 and 22.0      40.7 and 42.1      77.5 and 78.7      148.2 and 149.3
    //   FP16   17.5 and 17.8      35.1 and 35.6      65.8 and 65.4      122.6 and 120.2
    //   BF16   17.6 and 18.2      34.6 and 35.7      65.4 and 66.4      121.3 and 122.3
    // (at 4096^2 FP32 is 3.5 % slower with them).  Without walls at the bottom and top
    // there is no row pass to save, and the columns alone are the faster, 600 x 500 nodes
    // 10.4 us a step against 10.8.
    const bool all = !wfb && !P.periodic_y && (long long)P.nx * P.ny <= kFoldNodes;
    const bool columns = !wfb && !P.periodic_x && !all;
    const int wfix = all || columns ? repair : 0;
    if (all && grain)
        k_coupled_step<Store, true, false, kAllWalls>
            <<<grid, block, 0, s>>>(P, src, srcf, dst, dstf, B.hist, B.grain, B.fb, wfix);
    else if (all)
        k_coupled_step<Store, false, false, kAllWalls>
            <<<grid, block, 0, s>>>(P, src, srcf, dst, dstf, B.hist, B.grain, B.fb, wfix);
    else if (columns && grain)
        k_coupled_step<Store, true, false, kColumns>
            <<<grid, block, 0, s>>>(P, src, srcf, dst, dstf, B.hist, B.grain, B.fb, wfix);
    else if (columns)
        k_coupled_step<Store, false, false, kColumns>
            <<<grid, block, 0, s>>>(P, src, srcf, dst, dstf, B.hist, B.grain, B.fb, wfix);
    else if (grain && wfb)
        k_coupled_step<Store, true, true><<<grid, block, 0, s>>>(P, src, srcf, dst, dstf, B.hist, B.grain, B.fb);
    else if (grain)
        k_coupled_step<Store, true, false><<<grid, block, 0, s>>>(P, src, srcf, dst, dstf, B.hist, B.grain, B.fb);
    else if (wfb)
        k_coupled_step<Store, false, true><<<grid, block, 0, s>>>(P, src, srcf, dst, dstf, B.hist, B.grain, B.fb);
    else
        k_coupled_step<Store, false, false><<<grid, block, 0, s>>>(P, src, srcf, dst, dstf, B.hist, B.grain, B.fb);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (B.ev_end && !B.ev_substeps) cudaEventRecord(B.ev_end, s);
    if (!(all && skip_walls) && (e = walls<Store>(P, dst, dstf, 0, s, !(columns && skip_walls))) != cudaSuccess) return e;
    B.cs = 1 - B.cs;
    B.cf = 1 - B.cf;
    if (n_sub > 1) {
        // phi and the force of time n come from hist/fb; the wall scheme reads
        // the scalar macros of time n+1 from the newest scalar buffer.  The
        // flow-only wall pass runs after the last sub-step only: each later
        // sub-step repairs the wall nodes it loads instead.
        if (B.ev_begin && B.ev_substeps) cudaEventRecord(B.ev_begin, s);
        if ((e = flow_chain<Store>(P, n_sub - 1, B.sc[B.cs], B.fl, &B.cf, B.hist, kHist, B.fb, s)) != cudaSuccess)
            return e;
        if (B.ev_end && B.ev_substeps) cudaEventRecord(B.ev_end, s);
        if ((e = walls<Store>(P, B.sc[B.cs], B.fl[B.cf], 1, s)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// run: tiles per CTA; 0 makes the grid persistent (one contiguous run of
// tiles per resident CTA).
// repair / skip_walls: as for the single-domain step on a large grid (the
// columns); the column list holds the left/right walls of every domain that is
// not periodic in x.
template <class Store, int TYV>
cudaError_t batch_step_t(const BatchTables& T, int parity, int ctas, int run, cudaStream_t s, int repair,
                         int skip_walls)
{
    const int k = TYV == 4 ? 0 : TYV == 8 ? 1 : 2;
    const int chunk = run > 0 ? run : (T.ntiles[k] + ctas - 1) / ctas;
    const int grid = (T.ntiles[k] + chunk - 1) / chunk;
    if (T.ev_begin) cudaEventRecord(T.ev_begin, s);
    k_batch_step<Store, TYV><<<grid, dim3(TX, TYV), 0, s>>>(T.tiles[k], T.ntiles[k], chunk, parity, repair);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (T.ev_end) cudaEventRecord(T.ev_end, s);
    // the fused kernel wrote buffers 1 - parity; walls act on those (rows, then columns)
    if (T.nwall[0])
        k_batch_walls<Store><<<(T.nwall[0] + 127) / 128, 128, 0, s>>>(T.descs, T.walls[0], T.nwall[0], 1 - parity);
    if (T.nwall[1] && !skip_walls)
        k_batch_walls<Store><<<(T.nwall[1] + 127) / 128, 128, 0, s>>>(T.descs, T.walls[1], T.nwall[1], 1 - parity);
    return cudaGetLastError();
}

template <class Store>
cudaError_t batch_step_store(const BatchTables& T, int ty, int parity, int ctas, int run, cudaStream_t s,
                             int repair, int skip_walls)
{
    cudaError_t e = cudaMemcpyToSymbolAsync(c_batch_desc, T.descs, sizeof(DomainDesc) * T.ndomains, 0,
                                            cudaMemcpyDeviceToDevice, s);
    if (e != cudaSuccess) return e;
    switch (ty) {
    case 4: return batch_step_t<Store, 4>(T, parity, ctas, run, s, repair, skip_walls);
    case 16: return batch_step_t<Store, 16>(T, parity, ctas, run, s, repair, skip_walls);
    default: return batch_step_t<Store, 8>(T, parity, ctas, run, s, repair, skip_walls);
    }
}

template <class Store, int TYV>
int batch_ctas_t()
{
    int dev = 0, sms = 0, per = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_batch_step<Store, TYV>, TX * TYV, 0);
    return sms * (per > 0 ? per : 1);
}

}  // namespace

cudaError_t launch_batch_step(const BatchTables& T, int storage, int ty, int run, int parity, int ctas,
                              cudaStream_t s, int repair, int skip_walls)
{
    switch (storage) {
    case kStoreF16: return batch_step_store<StoreF16>(T, ty, parity, ctas, run, s, repair, skip_walls);
    case kStoreBF16: return batch_step_store<StoreBF16>(T, ty, parity, ctas, run, s, repair, skip_walls);
    default: return batch_step_store<StoreF32>(T, ty, parity, ctas, run, s, repair, skip_walls);
    }
}

int batch_resident_ctas(int storage, int ty)
{
    if (storage == kStoreF16) return ty == 4 ? batch_ctas_t<StoreF16, 4>() : ty == 16 ? batch_ctas_t<StoreF16, 16>() : batch_ctas_t<StoreF16, 8>();
    if (storage == kStoreBF16) return ty == 4 ? batch_ctas_t<StoreBF16, 4>() : ty == 16 ? batch_ctas_t<StoreBF16, 16>() : batch_ctas_t<StoreBF16, 8>();
    return ty == 4 ? batch_ctas_t<StoreF32, 4>() : ty == 16 ? batch_ctas_t<StoreF32, 16>() : batch_ctas_t<StoreF32, 8>();
}

cudaError_t flow_steps(const StepParams& P, int storage, int n, void* sc, void* const fl[2], int* cf, const float* phi,
                       const float* fy, cudaStream_t s)
{
    switch (storage) {
    case kStoreF16: return flow_steps_t<StoreF16>(P, n, sc, fl, cf, phi, fy, s);
    case kStoreBF16: return flow_steps_t<StoreBF16>(P, n, sc, fl, cf, phi, fy, s);
    default: return flow_steps_t<StoreF32>(P, n, sc, fl, cf, phi, fy, s);
    }
}

cudaError_t launch_coupled_step(const StepParams& P, int storage, int n_sub, StepBuffers& B, cudaStream_t s,
                                int repair, int skip_walls)
{
    switch (storage) {
    case kStoreF16: return coupled_step<StoreF16>(P, n_sub, B, s, repair, skip_walls);
    case kStoreBF16: return coupled_step<StoreBF16>(P, n_sub, B, s, repair, skip_walls);
    default: return coupled_step<StoreF32>(P, n_sub, B, s, repair, skip_walls);
    }
}

}  // namespace lbm
