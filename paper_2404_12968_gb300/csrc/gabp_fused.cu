// Fused GaBP iteration: one kernel computes the beliefs and every factor update of one
// synchronous iteration (Alg. 2, "Iterate MP Until Convergence": all new messages from the
// previous iteration's messages), so each message is read from HBM once and written once.
//
// Work unit: a TX x TY tile of cells.  The block
//   1. stages the 5 prior-message planes over the tile plus a 2-cell halo in shared memory
//      (the halo reads of neighbouring tiles hit L2, not HBM);
//   2. computes the compensated beliefs of the tile plus a 1-cell halo (every node a factor of
//      the tile touches), adding the observation messages that target those nodes;
//   3. updates the tile's cell factors (prior) and the observation factors whose base cell lies
//      in the tile, and writes the damped messages to the other ping-pong buffer.
// The arithmetic and the summation order are those of the split kernels, so both paths give
// bit-identical messages.
#include "gabp_device.cuh"
#include "gabp_internal.h"

namespace gabp {

namespace {

constexpr int FT = 256;   // threads per block

template <int TX, int TY> struct FusedLayout {
    static constexpr int RX = TX + 4, RY = TY + 4;   // staged message window (2-cell halo)
    static constexpr int BX = TX + 2, BY = TY + 2;   // belief window (1-cell halo)
    static constexpr size_t msg_bytes = sizeof(float2) * 5 * RX * RY;
    static constexpr size_t bel_bytes = sizeof(Belief<float>) * BX * BY;
    static constexpr size_t bytes = msg_bytes + bel_bytes + sizeof(int) * 2 * (TY + 1);
};

template <int TX, int TY>
__global__ void __launch_bounds__(FT) k_fused(DevProblem p, int src, float beta) {
    using LY = FusedLayout<TX, TY>;
    constexpr int RX = LY::RX, RY = LY::RY, BX = LY::BX, BY = LY::BY;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *sm = reinterpret_cast<float2 *>(smem_raw);                         // [5][RY][RX]
    Belief<float> *sb = reinterpret_cast<Belief<float> *>(smem_raw + LY::msg_bytes); // [BY][BX]
    int *rstart = reinterpret_cast<int *>(smem_raw + LY::msg_bytes + LY::bel_bytes);  // [TY+1]
    int *rpre = rstart + (TY + 1);                                                     // [TY+1]

    const int nx = p.nx, ny = p.ny;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const float2 *P = (const float2 *)p.P[src];
    float2 *Q = (float2 *)p.P[src ^ 1];
    const float *O = (const float *)p.O[src];
    float *OQ = (float *)p.O[src ^ 1];
    const int *optr = p.optr;

    // 1. stage the message window
    for (int q = threadIdx.x; q < 5 * RX * RY; q += FT) {
        const int d = q / (RX * RY);
        const int rem = q - d * (RX * RY);
        const int ly = rem / RX, lx = rem - ly * RX;
        const int gx = x0 - 2 + lx, gy = y0 - 2 + ly;
        float2 val;
        val.x = 0.f;
        val.y = 0.f;
        if (gx >= 0 && gx < nx && gy >= 0 && gy < ny) val = P[d * p.pn + (int64_t)gy * p.px + gx];
        sm[q] = val;
    }
    // observation ranges of the tile's base rows (cells [x0, x0+TX) of rows y0 .. y0+TY-1)
    if (p.m > 0 && threadIdx.x <= TY) {
        const int r = threadIdx.x;
        const int gy = y0 + r;
        int lo = 0, cnt = 0;
        if (r < TY && gy < ny) {
            const int xe = min(x0 + TX, nx);
            lo = optr[(int64_t)gy * nx + x0];
            cnt = optr[(int64_t)gy * nx + xe] - lo;
        }
        rstart[r] = lo;
        rpre[r] = cnt;   // prefix taken below
    }
    __syncthreads();
    if (p.m > 0 && threadIdx.x == 0) {
        int acc = 0;
        for (int r = 0; r < TY; ++r) {
            const int c = rpre[r];
            rpre[r] = acc;
            acc += c;
        }
        rpre[TY] = acc;
    }

    // 2. compensated beliefs over the tile plus a 1-cell halo
    for (int q = threadIdx.x; q < BX * BY; q += FT) {
        const int ly = q / BX, lx = q - ly * BX;
        const int gx = x0 - 1 + lx, gy = y0 - 1 + ly;
        if (gx < 0 || gx >= nx || gy < 0 || gy >= ny) continue;
        const int rx = lx + 1, ry = ly + 1;
        const int64_t v = (int64_t)gy * nx + gx;
        float2 m = sm[(DIR_C * RY + ry) * RX + rx];
        CompSum<float> se(m.x), sl(m.y);
        if (gx > 0) { m = sm[(DIR_E * RY + ry) * RX + rx - 1]; se.add(m.x); sl.add(m.y); }
        if (gx < nx - 1) { m = sm[(DIR_W * RY + ry) * RX + rx + 1]; se.add(m.x); sl.add(m.y); }
        if (gy > 0) { m = sm[(DIR_N * RY + ry - 1) * RX + rx]; se.add(m.x); sl.add(m.y); }
        if (gy < ny - 1) { m = sm[(DIR_S * RY + ry + 1) * RX + rx]; se.add(m.x); sl.add(m.y); }
        if (p.m > 0) {
            add_obs_pair(se, sl, O, gx > 0 ? optr[v - 1] : optr[v], optr[v], optr[v + 1], 1, 0);
            if (gy > 0)
                add_obs_pair(se, sl, O, gx > 0 ? optr[v - nx - 1] : optr[v - nx], optr[v - nx], optr[v - nx + 1], 3, 2);
        }
        se.finish();
        sl.finish();
        Belief<float> b;
        b.ehi = se.hi; b.elo = se.lo; b.lhi = sl.hi; b.llo = sl.lo;
        sb[q] = b;
    }
    __syncthreads();

    // 3a. prior cell factors of the tile
    const float var_prior = prior_var<float>(p);
    for (int q = threadIdx.x; q < TX * TY; q += FT) {
        const int ty = q / TX, tx = q - ty * TX;
        const int gx = x0 + tx, gy = y0 + ty;
        if (gx >= nx || gy >= ny) continue;
        const int64_t c = (int64_t)gy * nx + gx;
        const int deg = grid_degree(gy, gx, nx, ny);
        const float a[5] = {cell_coef<float>(p, deg), gx > 0 ? -1.f : 0.f, gx < nx - 1 ? -1.f : 0.f,
                        gy > 0 ? -1.f : 0.f, gy < ny - 1 ? -1.f : 0.f};
        // belief-window coordinates of the 5 nodes (C, W, E, S, N)
        const int bxs[5] = {tx + 1, tx, tx + 2, tx + 1, tx + 1};
        const int bys[5] = {ty + 1, ty + 1, ty + 1, ty, ty + 2};
        float2 own[5];
        float lam[5], eta[5];
#pragma unroll
        for (int u = 0; u < 5; ++u) {
            own[u] = sm[(u * RY + ty + 2) * RX + tx + 2];
            if (a[u] != 0.f) {
                cavity(sb[bys[u] * BX + bxs[u]], own[u].x, own[u].y, eta[u], lam[u]);
            } else {
                lam[u] = 1.f;
                eta[u] = 0.f;
            }
        }
        float L[5], E[5];
        const float r = p.ptgt ? ((const float *)p.ptgt)[c] : 0.f;
        factor_messages<float, 5>(a, var_prior, r, lam, eta, L, E);
#pragma unroll
        for (int u = 0; u < 5; ++u) {
            float2 out;
            if (a[u] != 0.f) {
                out.x = damp(own[u].x, E[u], beta);
                out.y = damp(own[u].y, L[u], beta);
            } else {
                out.x = 0.f;
                out.y = 0.f;
            }
            Q[u * p.pn + (int64_t)gy * p.px + gx] = out;
        }
    }

    // 3b. observation factors whose base cell lies in the tile
    if (p.m > 0) {
        const int total = rpre[TY];
        const float *W = (const float *)p.ow;
        const float *YV = (const float *)p.ovar;
        for (int q = threadIdx.x; q < total; q += FT) {
            int r = 0;
            while (r + 1 < TY && rpre[r + 1] <= q) ++r;
            const int64_t k = rstart[r] + (q - rpre[r]);
            const int b = p.obase[k];
            const int by = b / nx, bx = b - by * nx;
            const int lx = bx - x0 + 1, ly = by - y0 + 1;   // belief-window coordinates
            const int bidx[4] = {ly * BX + lx, ly * BX + lx + 1, (ly + 1) * BX + lx, (ly + 1) * BX + lx + 1};
            const float a[4] = {W[4 * k], W[4 * k + 1], W[4 * k + 2], W[4 * k + 3]};
            float oe[4], ol[4], lam[4], eta[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                oe[u] = O[8 * k + 2 * u];
                ol[u] = O[8 * k + 2 * u + 1];
                cavity(sb[bidx[u]], oe[u], ol[u], eta[u], lam[u]);
            }
            float L[4], E[4];
            factor_messages<float, 4>(a, YV[2 * k + 1], YV[2 * k], lam, eta, L, E);
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                OQ[8 * k + 2 * u] = damp(oe[u], E[u], beta);
                OQ[8 * k + 2 * u + 1] = damp(ol[u], L[u], beta);
            }
        }
    }
}

// ---- FP64 ----
// FP64 arithmetic bounds this kernel (GB300: two lanes per clock and SM; an iteration's bytes would
// take a twentieth of the time), so the work per cell is what it saves: no product by +-1 and no
// sum with an exact zero on interior cells (cell_update_interior), Fast2Sum, reciprocals without an
// FP64 operation (recip_fixed), comparisons and floors in the integer unit, and both observation ranges of a node
// in one loop, so that lanes with a term in either run together.  The messages are read straight
// from global memory (the second reading, in the factor update, hits L1): staging them cost a pass
// of index arithmetic and the shared memory that limited the resident blocks.  Tiles of TX columns
// and a height chosen per grid (fused_choose_shape_f64), NT threads.  Measured per iteration, with
// the staged kernel of 32 x 8 tiles, compensated sums of six additions and IEEE divisions before:
// 64^2 36 -> 13.5 us, 512^2 197 -> 91 us.
template <int TX, int NT>
__global__ void __launch_bounds__(NT) k_fused_f64(const __grid_constant__ DevProblem p, int TY, int src, double beta) {
    constexpr int BX = TX + 2;
    const int BY = TY + 2;   // belief window (1-cell halo)
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Belief<double> *sb = reinterpret_cast<Belief<double> *>(smem_raw);            // [BY][BX]
    int *rstart = reinterpret_cast<int *>(smem_raw + sizeof(Belief<double>) * BX * BY);   // [TY]
    int *rpre = rstart + TY;                                                              // [TY + 1]

    const int nx = p.nx, ny = p.ny, px = p.px;
    const int64_t pn = p.pn;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const double2 *P = (const double2 *)p.P[src];
    double2 *Q = (double2 *)p.P[src ^ 1];
    const double *O = (const double *)p.O[src];
    double *OQ = (double *)p.O[src ^ 1];
    const int *__restrict__ optr = p.optr;

    // observation ranges of the tile's base rows (the last warp; a prefix sum by shuffles)
    if (p.m > 0 && threadIdx.x >= NT - 32) {
        const int r = threadIdx.x - (NT - 32), gy = y0 + r;
        int lo = 0, cnt = 0;
        if (r < TY && gy < ny) {
            lo = optr[(int64_t)gy * nx + x0];
            cnt = optr[(int64_t)gy * nx + min(x0 + TX, nx)] - lo;
        }
        int inc = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (r >= o) inc += v;
        }
        if (r < TY) {
            rstart[r] = lo;
            rpre[r] = inc - cnt;
        }
        if (r == TY - 1) rpre[TY] = inc;
    }

    pdl_wait();   // the ranges above are static; the messages are the previous iteration's
    pdl_trigger();

    // 1. compensated beliefs over the tile plus a 1-cell halo
#pragma unroll 1
    for (int q = threadIdx.x; q < BX * BY; q += NT) {
        const int ly = q / BX, lx = q - ly * BX;
        const int gx = x0 - 1 + lx, gy = y0 - 1 + ly;
        if (gx < 0 || gx >= nx || gy < 0 || gy >= ny) continue;
        const int64_t v = (int64_t)gy * px + gx;
        const double2 zero = make_double2(0.0, 0.0);
        const double2 mC = P[DIR_C * pn + v];
        const double2 mE = gx > 0 ? P[DIR_E * pn + v - 1] : zero;
        const double2 mW = gx < nx - 1 ? P[DIR_W * pn + v + 1] : zero;
        const double2 mN = gy > 0 ? P[DIR_N * pn + v - px] : zero;
        const double2 mS = gy < ny - 1 ? P[DIR_S * pn + v + px] : zero;
        int lo1 = 0, mid1 = 0, hi1 = 0, lo2 = 0, mid2 = 0, hi2 = 0;
        if (p.m > 0) {
            const int *o = optr + (int64_t)gy * nx + gx;
            mid1 = o[0];
            hi1 = o[1];
            lo1 = gx > 0 ? o[-1] : mid1;
            if (gy > 0) {
                mid2 = o[-nx];
                hi2 = o[1 - nx];
                lo2 = gx > 0 ? o[-nx - 1] : mid2;
            }
        }
        CompSum<double> se(mC.x), sl(mC.y);   // a missing neighbour adds an exact zero
        se.second(mE.x); sl.second(mE.y);
        se.add(mW.x); sl.add(mW.y);
        se.add(mN.x); sl.add(mN.y);
        se.add(mS.x); sl.add(mS.y);
        // the observation messages of both ranges in their order, the next one loaded ahead
        const int n1 = hi1 - lo1, nt = n1 + hi2 - lo2;
        auto term = [&](int t) {
            const int k = t < n1 ? lo1 + t : lo2 + t - n1;
            const int cr = t < n1 ? (k < mid1 ? 1 : 0) : (k < mid2 ? 3 : 2);
            return *reinterpret_cast<const double2 *>(O + 8 * (int64_t)k + 2 * cr);
        };
        double2 nx_t = nt > 0 ? term(0) : zero;
        for (int t = 0; t < nt; ++t) {
            const double2 cu = nx_t;
            if (t + 1 < nt) nx_t = term(t + 1);
            se.add(cu.x);
            sl.add(cu.y);
        }
        se.finish();
        sl.finish();
        Belief<double> b;
        b.ehi = se.hi; b.elo = se.lo; b.lhi = sl.hi; b.llo = sl.lo;
        sb[q] = b;
    }
    __syncthreads();

    // 2. prior cell factors of the tile
    const double *__restrict__ tgt = (const double *)p.ptgt;
#pragma unroll 1
    for (int q = threadIdx.x; q < TX * TY; q += NT) {
        const int ty = q / TX, tx = q - ty * TX;
        const int gx = x0 + tx, gy = y0 + ty;
        if (gx >= nx || gy >= ny) continue;
        const int64_t c = (int64_t)gy * px + gx;
        double2 own[5], out[5];
#pragma unroll
        for (int u = 0; u < 5; ++u) own[u] = P[u * pn + c];
        const Belief<double> *w = sb + (ty + 1) * BX + tx + 1;
        const Belief<double> *const bs[5] = {w, w - 1, w + 1, w - BX, w + BX};
        cell_update_f64(p, gy, gx, tgt ? tgt[(int64_t)gy * nx + gx] : 0.0, bs, own, beta, out);
#pragma unroll
        for (int u = 0; u < 5; ++u) Q[u * pn + c] = out[u];
    }

    // 3. observation factors whose base cell lies in the tile, last threads first (the first ones
    // may still hold a cell of the loop above)
    if (p.m > 0) {
        const int total = rpre[TY];
        const double *W = (const double *)p.ow;
        const double *YV = (const double *)p.ovar;
        for (int q = NT - 1 - threadIdx.x; q < total; q += NT) {
            int r = 0;
            while (r + 1 < TY && rpre[r + 1] <= q) ++r;
            const int64_t k = rstart[r] + (q - rpre[r]);
            const int lx = p.obase[k] - (y0 + r) * nx - x0 + 1;   // belief-window column
            const Belief<double> *w = sb + (r + 1) * BX + lx;
            const Belief<double> *const bs[4] = {w, w + 1, w + BX, w + BX + 1};
            double a[4], lam[4], eta[4];
            double2 own[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                a[u] = W[4 * k + u];
                own[u] = *reinterpret_cast<const double2 *>(O + 8 * k + 2 * u);
                cavity(*bs[u], own[u].x, own[u].y, eta[u], lam[u]);
            }
            double L[4], E[4];
            factor_messages<double, 4>(a, YV[2 * k + 1], YV[2 * k], lam, eta, L, E);
#pragma unroll
            for (int u = 0; u < 4; ++u)
                *reinterpret_cast<double2 *>(OQ + 8 * k + 2 * u) =
                    make_double2(damp(own[u].x, E[u], beta), damp(own[u].y, L[u], beta));
        }
    }
}

// The same iteration for small grids, where a tile's chain of FP64 instructions is what takes the time
// (each holds its SM quarter for 64 cycles or more, however few lanes are active): the chain is cut by
// giving more warps a part of it.  Tiles of 8 x 4 cells, 8 warps:
//   beliefs: warps 0, 1 sum the window nodes' eta messages, warps 2, 3 their Lambda messages;
//   cell factors: warp u (0..4) owns slot u of the tile's 32 cells.  It forms the slot's terms
//     t_u = a_u^2 / lam_u and p_u = a_u eta_u / lam_u, the warps exchange them through shared memory,
//     and each adds the other four slots' in the order of factor_messages (21 FP64 instructions per
//     warp against 74 in one);
//   observation factors: warps 5..7, four lanes per factor, one per corner.
// Messages are bit-identical to the other kernels' (but for the sign of a zero at damping 0).
constexpr int WX = 8, WY = 4, WNT = 256, WBX = WX + 2, WNODES = WBX * (WY + 2);

__device__ __forceinline__ void bar_cells() { asm volatile("bar.sync 1, 160;" ::: "memory"); }   // warps 0..4

__global__ void __launch_bounds__(WNT) k_fused_f64_wide(const __grid_constant__ DevProblem p, int src, double beta) {
    __shared__ double sb[4][WNODES];        // eta_hi, eta_lo, lam_hi, lam_lo of the window's nodes
    __shared__ double2 stp[5][32];          // (t, p) of the cells' slots
    __shared__ int rstart[WY], rpre[WY + 1];
    const int nx = p.nx, ny = p.ny, px = p.px, tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const int64_t pn = p.pn;
    const int x0 = blockIdx.x * WX, y0 = blockIdx.y * WY;
    const double2 *P = (const double2 *)p.P[src];
    double2 *Q = (double2 *)p.P[src ^ 1];
    const double *O = (const double *)p.O[src];
    double *OQ = (double *)p.O[src ^ 1];
    const int *__restrict__ optr = p.optr;

    // observation ranges of the tile's base rows (one lane each)
    if (warp == 4 && p.m > 0) {
        const int gy = y0 + lane;
        int lo = 0, cnt = 0;
        if (lane < WY && gy < ny) {
            lo = optr[(int64_t)gy * nx + x0];
            cnt = optr[(int64_t)gy * nx + min(x0 + WX, nx)] - lo;
        }
        int inc = cnt;
#pragma unroll
        for (int o = 1; o < WY; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += v;
        }
        if (lane < WY) {
            rstart[lane] = lo;
            rpre[lane] = inc - cnt;
        }
        if (lane == WY - 1) rpre[WY] = inc;
    }
    // the window node of this thread and its observation ranges (static), then the messages
    const int node = (warp & 1) * 32 + lane, comp = warp >> 1;   // warps 0..3
    const int ly = node / WBX, lx = node - ly * WBX, gx = x0 - 1 + lx, gy = y0 - 1 + ly;
    const bool mine = warp < 4 && node < WNODES && gx >= 0 && gx < nx && gy >= 0 && gy < ny;
    int lo1 = 0, mid1 = 0, hi1 = 0, lo2 = 0, mid2 = 0, hi2 = 0;
    if (mine && p.m > 0) {
        const int *o = optr + (int64_t)gy * nx + gx;
        mid1 = o[0];
        hi1 = o[1];
        lo1 = gx > 0 ? o[-1] : mid1;
        if (gy > 0) {
            mid2 = o[-nx];
            hi2 = o[1 - nx];
            lo2 = gx > 0 ? o[-nx - 1] : mid2;
        }
    }
    pdl_wait();
    pdl_trigger();
    // the cell of this lane (warps 0..4): its own message on the warp's slot
    const int cty = lane / WX, ctx = lane - cty * WX, cx = x0 + ctx, cy = y0 + cty;
    const int u = warp;   // slot: C, W, E, S, N
    const bool cell = u < 5 && cx < nx && cy < ny;
    const bool has = cell && (u == 0 || (u == 1 && cx > 0) || (u == 2 && cx < nx - 1) || (u == 3 && cy > 0) ||
                              (u == 4 && cy < ny - 1));
    const int64_t pc = (int64_t)cy * px + cx;
    double2 own = make_double2(0.0, 0.0);
    if (has) own = P[u * pn + pc];

    // 1. compensated beliefs, one component per thread
    if (mine) {
        const int64_t v = (int64_t)gy * px + gx;
        auto at = [&](int d, int64_t i) { return reinterpret_cast<const double *>(P + d * pn + i)[comp]; };
        const double mC = at(DIR_C, v);
        const double mE = gx > 0 ? at(DIR_E, v - 1) : 0.0, mW = gx < nx - 1 ? at(DIR_W, v + 1) : 0.0;
        const double mN = gy > 0 ? at(DIR_N, v - px) : 0.0, mS = gy < ny - 1 ? at(DIR_S, v + px) : 0.0;
        const int n1 = hi1 - lo1, nt = n1 + hi2 - lo2;
        auto term = [&](int t) {   // the observation messages of both ranges in their order
            const int k = t < n1 ? lo1 + t : lo2 + t - n1;
            const int cr = t < n1 ? (k < mid1 ? 1 : 0) : (k < mid2 ? 3 : 2);
            return O[8 * (int64_t)k + 2 * cr + comp];
        };
        double next = nt > 0 ? term(0) : 0.0;
        CompSum<double> s(mC);
        s.second(mE);
        s.add(mW);
        s.add(mN);
        s.add(mS);
        for (int t = 0; t < nt; ++t) {
            const double cu = next;
            if (t + 1 < nt) next = term(t + 1);
            s.add(cu);
        }
        s.finish();
        sb[2 * comp][node] = s.hi;
        sb[2 * comp + 1][node] = s.lo;
    }
    __syncthreads();

    if (warp < 5) {
        // 2. cell factors: slot u of 32 cells
        const int w = (cty + 1) * WBX + ctx + 1 + (u == 1 ? -1 : u == 2 ? 1 : u == 3 ? -WBX : u == 4 ? WBX : 0);
        const double aC = cell ? p.aC[grid_degree(cy, cx, nx, ny)] : 1.0;
        const double a2 = u == 0 ? mul_rn(aC, aC) : 1.0;
        bool out = false;
        double2 tp = make_double2(0.0, 0.0);
        if (has) {
            const double lam = (sb[2][w] - own.y) + sb[3][w], eta = (sb[0][w] - own.x) + sb[1][w];
            double fl = lam_floor_rel<double>();
            if (u == 0) fl = floor_at(mul_rn(fl, a2), tiny_normal<double>());
            const double x = floor_at(lam, fl);
            double rl = recip_fixed(x, out);
            if (out) rl = 1.0 / x;
            tp.x = u == 0 ? mul_rn(a2, rl) : rl;
            tp.y = u == 0 ? mul_rn(aC, mul_rn(eta, rl)) : -mul_rn(eta, rl);
        }
        stp[u][lane] = tp;
        bar_cells();
        // the other slots' terms: those before u from the left, those after it from the right
        double V = p.var64, M = 0.0, sV = 0.0, sM = 0.0;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (q < u) {
                const double2 o = stp[q][lane];
                V = add_rn(V, o.x);
                M = q == 0 ? o.y : add_rn(M, o.y);
            }
#pragma unroll
        for (int q = 4; q > 0; --q)
            if (q > u) {
                const double2 o = stp[q][lane];
                sV = q == 4 ? o.x : add_rn(sV, o.x);
                sM = q == 4 ? o.y : add_rn(sM, o.y);
            }
        if (u < 4) {
            V = add_rn(V, sV);
            M = u == 0 ? sM : add_rn(M, sM);
        }
        if (p.ptgt && cell) M = add_rn(M, -((const double *)p.ptgt)[(int64_t)cy * nx + cx]);
        out = false;
        double rV = recip_fixed(V, out);
        if (out) rV = 1.0 / V;
        const double L = u == 0 ? mul_rn(a2, rV) : rV;
        const double E = u == 0 ? mul_rn(mul_rn(aC, -M), rV) : mul_rn(M, rV);
        if (cell) Q[u * pn + pc] = has ? make_double2(damp(own.x, E, beta), damp(own.y, L, beta)) : make_double2(0.0, 0.0);
    } else if (p.m > 0) {
        // 3. observation factors based in the tile: lane = (factor, corner)
        const int total = rpre[WY], c = lane & 3;
        const double *W = (const double *)p.ow;
        const double *YV = (const double *)p.ovar;
        for (int q0 = 8 * (warp - 5); q0 < total; q0 += 24) {
            const int q = q0 + (lane >> 2);
            const bool on = q < total;
            const int qq = on ? q : total - 1;
            int r = 0;
#pragma unroll
            for (int t = 1; t < WY; ++t)
                if (rpre[t] <= qq) r = t;
            const int64_t k = rstart[r] + (qq - rpre[r]);
            const int w = (r + 1 + (c >> 1)) * WBX + p.obase[k] - (y0 + r) * nx - x0 + 1 + (c & 1);
            const double a = W[4 * k + c], y = YV[2 * k], var = YV[2 * k + 1];
            const double2 o = *reinterpret_cast<const double2 *>(O + 8 * k + 2 * c);
            const double lam = (sb[2][w] - o.y) + sb[3][w], eta = (sb[0][w] - o.x) + sb[1][w];
            const double a2 = mul_rn(a, a);
            const double x = floor_at(lam, floor_at(mul_rn(lam_floor_rel<double>(), a2), tiny_normal<double>()));
            bool out = false;
            double rl = recip_fixed(x, out);
            if (out) rl = 1.0 / x;
            double t = mul_rn(a2, rl), pp = mul_rn(a, mul_rn(eta, rl));
            if (is_zero(a)) t = pp = 0.0;
            double V = var, M = 0.0, sV = 0.0, sM = 0.0;
#pragma unroll
            for (int j = 0; j < 4; ++j) {   // slots before this one, in order
                const double tj = __shfl_sync(0xffffffffu, t, j, 4), pj = __shfl_sync(0xffffffffu, pp, j, 4);
                if (j < 3) {
                    const double nV = add_rn(V, tj), nM = add_rn(M, pj);
                    if (j < c) V = nV, M = nM;
                }
            }
#pragma unroll
            for (int j = 3; j >= 0; --j) {   // slots after it, from the last
                const double tj = __shfl_sync(0xffffffffu, t, j, 4), pj = __shfl_sync(0xffffffffu, pp, j, 4);
                if (j > 0) {
                    const double nV = add_rn(sV, tj), nM = add_rn(sM, pj);
                    if (j > c) sV = nV, sM = nM;
                }
            }
            V = add_rn(V, sV);
            M = add_rn(M, sM);
            out = false;
            double rV = recip_fixed(V, out);
            if (out) rV = 1.0 / V;
            const double L = mul_rn(a2, rV), E = mul_rn(mul_rn(a, add_rn(y, -M)), rV);
            if (on) *reinterpret_cast<double2 *>(OQ + 8 * k + 2 * c) = make_double2(damp(o.x, E, beta), damp(o.y, L, beta));
        }
    }
}

// SMs of the current device (looked up once per device)
int sm_count() {
    static PerDevice<int> cache;
    int dev = 0, nsm = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cache.get(dev, nsm, [&](int &v) { return cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev); }) == cudaSuccess &&
        nsm > 0)
        return nsm;
    cudaGetLastError();
    return 152;
}

constexpr int F64_MAX_TY = 32;   // a warp holds the tile's row ranges

template <int TX, int NT>
cudaError_t launch_f64(const DevProblem &p, int ty, int src, double beta, cudaStream_t st) {
    static_assert(NT >= 32, "one warp at least");
    const size_t bytes = sizeof(Belief<double>) * (TX + 2) * (ty + 2) + sizeof(int) * (2 * ty + 1);
    if (ty < 1 || ty > F64_MAX_TY || bytes > 48 * 1024) return cudaErrorInvalidValue;
    const dim3 grid((unsigned)((p.nx + TX - 1) / TX), (unsigned)((p.ny + ty - 1) / ty));
    // overlapped launches for grids of at most one block per SM (64^2: 13.5 -> 12.8 us); with more, the
    // next launch's blocks fill the slots unevenly (256^2: 36 -> 38 us)
    return launch_pdl((int64_t)grid.x * grid.y <= sm_count(), k_fused_f64<TX, NT>, grid, NT, bytes, st, p, ty, src, beta);
}

template <int TX, int TY>
cudaError_t launch_shape(const DevProblem &p, int src, double beta, cudaStream_t st) {
    using LY = FusedLayout<TX, TY>;
    static PerDevice<bool> configured;   // per instantiation; the attribute is per function and device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    bool set = false;
    e = configured.get(dev, set, [](bool &v) {
        v = true;
        return cudaFuncSetAttribute(k_fused<TX, TY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)LY::bytes);
    });
    if (e != cudaSuccess) return e;
    dim3 grid((unsigned)((p.nx + TX - 1) / TX), (unsigned)((p.ny + TY - 1) / TY));
    k_fused<TX, TY><<<grid, FT, LY::bytes, st>>>(p, src, (float)beta);
    return cudaGetLastError();
}

cudaError_t dispatch_f32(const DevProblem &p, int src, double beta, FusedShape s, cudaStream_t st) {
#define GABP_SHAPE(X, Y) \
    if (s.tx == X && s.ty == Y) return launch_shape<X, Y>(p, src, beta, st);
    GABP_SHAPE(32, 8)
    GABP_SHAPE(32, 16)
    GABP_SHAPE(64, 8)
    GABP_SHAPE(64, 16)
    GABP_SHAPE(128, 8)
    GABP_SHAPE(32, 32)
#undef GABP_SHAPE
    return cudaErrorInvalidValue;
}

cudaError_t dispatch_f64(const DevProblem &p, int src, double beta, FusedShape s, cudaStream_t st) {
    switch (s.tx) {
        case 128: return launch_f64<128, 256>(p, s.ty, src, beta, st);
        case 64: return launch_f64<64, 256>(p, s.ty, src, beta, st);
        case 32: return launch_f64<32, 128>(p, s.ty, src, beta, st);
        case 8: {
            const dim3 grid((unsigned)((p.nx + WX - 1) / WX), (unsigned)((p.ny + WY - 1) / WY));
            return launch_pdl(s.ty == WY && grid.y <= 65535 ? (int64_t)grid.x * grid.y <= sm_count() : false, k_fused_f64_wide, grid,
                              WNT, 0, st, p, src, beta);
        }
        case 16: return launch_f64<16, 128>(p, s.ty, src, beta, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace

bool fused_shape_supported(int tx, int ty) {
    return (tx == 32 && (ty == 8 || ty == 16 || ty == 32)) || (tx == 64 && (ty == 8 || ty == 16)) ||
           (tx == 128 && ty == 8);
}

// Small grids: the 8 x 4 tiles of k_fused_f64_wide while an SM gets at most three of them (64^2 13.2 ->
// 6.8 us, 96^2 12.8 -> 11.1 us, 110^2 17.4 -> 14.6 us, 128^2 16.8 -> 17.2 us).  Else tiles of 16 columns,
// of 8, 16 and 32 the fastest or within 3 % of it up to 1024^2; their height is the shortest of 4, 8
// and 14 rows that gives an SM at most four tiles: short tiles spread a small grid over the chip
// (128^2: 16.3 us with 16 x 4 against 33.0 us with 16 x 14 tiles, 180^2: 24.8 against 29.6), tall ones
// recompute fewer halo beliefs (256^2: 37.7 against 36.1 us, 1024^2: 345 against 286 us).
FusedShape fused_choose_shape_f64(int nx, int ny) {
    const int nsm = sm_count();
    if ((int64_t)((nx + WX - 1) / WX) * ((ny + WY - 1) / WY) <= 3 * (int64_t)nsm) return {WX, WY};
    for (int ty : {4, 8})
        if ((int64_t)((nx + 15) / 16) * ((ny + ty - 1) / ty) <= 4 * (int64_t)nsm) return {16, ty};
    return {16, 14};
}

cudaError_t launch_fused_iteration(const DevProblem &p, int src, double beta, FusedShape shape,
                                   cudaStream_t st) {
    return p.prec ? dispatch_f64(p, src, beta, shape, st) : dispatch_f32(p, src, beta, shape, st);
}

}  // namespace gabp
