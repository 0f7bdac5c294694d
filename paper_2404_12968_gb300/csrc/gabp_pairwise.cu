// The paper's pairwise re-weighted Gaussian message passing (App. A, "Gaussian Setting" and
// "Re-weighted message updates"), as a second iteration family over the same posterior.
//
// Model: p(f) ~ exp(-f^T P f / 2 + h^T f) with P = gamma L^T L + H^T R^-1 H, h = H^T R^-1 y.
// One node factor per node and one pair factor per nonzero off-diagonal P_ij: the 13-point
// pattern of L^T L (offsets (0, +-1), (+-1, 0), (+-1, +-1), (0, +-2), (+-2, 0)); bilinear
// observations stay inside it.  Fractional messages with weight c (the information convention
// exp(-a f^2 / 2 + b f) throughout):
//   alpha_{j->i} = P_jj + c sum_{k != i} a_{kj} + (c - 1) a_{ij},
//   beta_{j->i}  = h_j  + c sum_{k != i} b_{kj} + (c - 1) b_{ij},
//   a_{ji} = -(P_ij / c)^2 / alpha_{j->i},   b_{ji} = -beta_{j->i} (P_ij / c) / alpha_{j->i},
// with (a_kj, b_kj) the pair factor (k, j)'s message to f_j.  The b update follows the integral
// that defines the message (the paper prints the opposite sign).  Damping with the paper's
// learning rate eta: m <- (1 - eta) m_old + eta m_new.  Marginal: mean (h_i + c sum_k b_ki) /
// (P_ii + c sum_k a_ki), precision P_ii + c sum_k a_ki.
//
// Layout: 12 "outgoing" planes of (a, b) pairs, ping-pong: plane d at node j holds the message of
// the pair factor (j, j + off_d) to f_{j + off_d}, computed by node j; slots without that
// neighbour hold (0, 0).  Node i reads its incoming messages from plane d at i - off_d, and
// the pair factor's message back to itself from plane opp(d) at i + off_d.  Coefficients per
// node: P_ii, h_i and P_{i, i + off_d}.
#include <algorithm>
#include <cmath>
#include <cstdlib>

#include "gabp_device.cuh"
#include "gabp_internal.h"

namespace gabp {

namespace {

constexpr int PW_TPB = 256;
constexpr int ND = 12;
// (dy, dx) of the 12 directions, ordered so that the opposite of direction d is d ^ 1; the
// first 8 are the nearest offsets (every corner pair of an observation cell)
__host__ __device__ constexpr int DY(int d) {
    return d == 2 || d == 4 || d == 6 ? -1 : d == 3 || d == 5 || d == 7 ? 1 : d == 10 ? -2 : d == 11 ? 2 : 0;
}
__host__ __device__ constexpr int DX(int d) {
    return d == 0 || d == 4 || d == 7 ? -1 : d == 1 || d == 5 || d == 6 ? 1 : d == 8 ? -2 : d == 9 ? 2 : 0;
}
__host__ __device__ constexpr int OPP(int d) { return d ^ 1; }

__device__ __forceinline__ int64_t gtid() { return blockIdx.x * (int64_t)blockDim.x + threadIdx.x; }
inline unsigned nblk(int64_t count) { return (unsigned)((count + PW_TPB - 1) / PW_TPB); }

// coefficient of node v in row c of L (zero-Neumann): kappa^2 + deg(c) on the diagonal, -1 for an
// existing 4-neighbour, 0 otherwise
__device__ __forceinline__ double L_coef(const DevProblem &p, int ci, int cj, int vi, int vj) {
    if (ci < 0 || ci >= p.ny || cj < 0 || cj >= p.nx) return 0.0;
    if (vi == ci && vj == cj) return p.aC[grid_degree(ci, cj, p.nx, p.ny)];
    const int d = abs(vi - ci) + abs(vj - cj);
    return d == 1 ? -1.0 : 0.0;
}

// Per node i: P_ii, h_i and P_{i, i + off_d} (FP64 sums, stored in T).  Prior: gamma sum over the
// cells c of the two nodes' stencils of L_ci L_cj; observations: s_k w_a w_b and s_k y_k w_a over
// the observations based in the four cells around i, in the order of the observation index.
template <typename T>
__global__ void k_pw_coef(DevProblem p, T *Pd, T *hv, T *Pn) {
    const int64_t v = gtid();
    if (v >= p.n) return;
    const int nx = p.nx, ny = p.ny;
    const int i = (int)(v / nx), j = (int)(v - (int64_t)i * nx);
    double diag = 0.0, off[ND];
    for (int d = 0; d < ND; ++d) off[d] = 0.0;
    // prior: cells c in {v} and its 4-neighbours
    const int cdy[5] = {0, 0, 0, -1, 1}, cdx[5] = {0, -1, 1, 0, 0};
    for (int q = 0; q < 5; ++q) {
        const int ci = i + cdy[q], cj = j + cdx[q];
        const double li = L_coef(p, ci, cj, i, j);
        if (li == 0.0) continue;
        diag += p.gamma * li * li;
        for (int d = 0; d < ND; ++d) {
            const int ti = i + DY(d), tj = j + DX(d);
            if (ti < 0 || ti >= ny || tj < 0 || tj >= nx) continue;
            off[d] += p.gamma * li * L_coef(p, ci, cj, ti, tj);
        }
    }
    // observations based in the cells (i, j), (i, j-1), (i-1, j), (i-1, j-1): node v is corner
    // 0, 1, 2, 3 of them respectively; corner c sits at (dy, dx) = (c >> 1, c & 1) from the base
    double hh = 0.0;
    if (p.m > 0) {
        const int *o = p.optr;
        for (int cc = 0; cc < 4; ++cc) {
            const int bi = i - (cc >> 1), bj = j - (cc & 1);
            if (bi < 0 || bj < 0 || bi > ny - 2 || bj > nx - 2) continue;
            const int64_t b = (int64_t)bi * nx + bj;
            for (int k = o[b]; k < o[b + 1]; ++k) {
                const double *w = p.ow64 + 4 * (int64_t)k;
                const double s = p.oys64[2 * (int64_t)k + 1], y = p.oys64[2 * (int64_t)k];
                diag += s * w[cc] * w[cc];
                hh += s * y * w[cc];
                for (int c2 = 0; c2 < 4; ++c2) {
                    if (c2 == cc) continue;
                    const int ddy = (c2 >> 1) - (cc >> 1), ddx = (c2 & 1) - (cc & 1);
                    for (int d = 0; d < 8; ++d)   // the 8 nearest offsets hold every corner pair
                        if (DY(d) == ddy && DX(d) == ddx) off[d] += s * w[cc] * w[c2];
                }
            }
        }
    }
    Pd[v] = T(diag);
    hv[v] = T(hh);
    for (int d = 0; d < ND; ++d) Pn[(int64_t)d * p.n + v] = T(off[d]);
}

template <typename T>
__global__ void k_pw_zero(T *m, int64_t count) {
    const int64_t q = gtid();
    if (q < count) m[q] = T(0);
}

// ---- one synchronous iteration ----
// Node j reads its 12 incoming messages, forms the leave-one-out sums by prefix and suffix sums,
// and writes its 12 damped outgoing messages.  Every operand (12 incoming and 12 own messages, 12
// coefficients) is copied to the thread's own shared-memory slots by cp.async first: all of a
// node's reads are in flight at once without a register each, and one latency is paid per node.
// (Loaded into registers, bounded to 40 for six resident blocks of 256 threads, the own messages and
// coefficients were read one direction after the other, and the spills missed L1.)  Slots
// are private to the thread, so no barrier is needed.  The order of the copies matters to DRAM:
// coefficients, incoming, own messages 0.70 ms at 4096^2; own before incoming messages 0.84 ms; own
// messages and coefficients in turn 0.88 ms.  Per iteration, before and after: 64^2 8.6 -> 3.4 us,
// 512^2 22.5 -> 11.3 us, 1024^2 71 -> 47 us, 4096^2 887 -> 703 us (5.9 TB/s); FP64 512^2 311 -> 206 us
// (bound by FP64 arithmetic; 247 us with blocks of 128).
template <typename T> struct PwSlots {
    static constexpr int NT = sizeof(T) == 4 ? 128 : 64;   // threads per block
    T2<T> in[ND][NT], old[ND][NT];
    T q[ND][NT];
};

template <int BYTES> __device__ __forceinline__ void copy_async(void *dst, const void *src) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src), "n"(BYTES)
                 : "memory");
}

// the new message of pair (j, i) from the leave-one-out sums: alpha, beta, q = P_ij / c, damped as
// new + (1 - eta)(old - new).  FP32: q = P_ij (1 / c) and the approximate reciprocal of the rank-1
// kernels.  (Scalar: in the packed two-lane form these products and sums came out fused.)
__device__ __forceinline__ float2 pw_message(float2 loo, float2 in, float2 node, float2 old, float P, float c, float inv_c,
                                             float cm1, float keep) {
    const float alpha = add_rn(add_rn(node.x, mul_rn(c, loo.x)), mul_rn(cm1, in.x));
    const float beta = add_rn(add_rn(node.y, mul_rn(c, loo.y)), mul_rn(cm1, in.y));
    const float q = mul_rn(P, inv_c), ra = recip(alpha);
    const float a = mul_rn(mul_rn(q, q), ra), b = mul_rn(mul_rn(beta, q), ra);   // minus the new message
    return make_float2(fma_rn(keep, add_rn(old.x, a), -a), fma_rn(keep, add_rn(old.y, b), -b));
}
// FP64: the reciprocal in the integer and FP32 units, the quotient P_ij / c by one correction
__device__ __forceinline__ double2 pw_message(double2 loo, double2 in, double2 node, double2 old, double P, double c, double inv_c,
                                              double cm1, double keep) {
    const double alpha = add_rn(add_rn(node.x, mul_rn(c, loo.x)), mul_rn(cm1, in.x));
    const double beta = add_rn(add_rn(node.y, mul_rn(c, loo.y)), mul_rn(cm1, in.y));
    const double q0 = mul_rn(P, inv_c), q = fma_rn(fma_rn(-q0, c, P), inv_c, q0);
    bool out = false;
    double ra = recip_fixed(alpha, out);
    if (out) ra = 1.0 / alpha;
    const double a = mul_rn(mul_rn(q, q), ra), b = mul_rn(mul_rn(beta, q), ra);
    return make_double2(fma_rn(keep, add_rn(old.x, a), -a), fma_rn(keep, add_rn(old.y, b), -b));
}
__device__ __forceinline__ float2 pair_add(float2 a, float2 b) { return make_float2(add_rn(a.x, b.x), add_rn(a.y, b.y)); }
__device__ __forceinline__ double2 pair_add(double2 a, double2 b) { return make_double2(add_rn(a.x, b.x), add_rn(a.y, b.y)); }

template <typename T>
__global__ void __launch_bounds__(PwSlots<T>::NT) k_pw_iter(int nx, int ny, int64_t n, const T *__restrict__ Pd, const T *__restrict__ hv,
                                                   const T *__restrict__ Pn, const T2<T> *src, T2<T> *dst,
                                                   T c, T inv_c, T eta) {
    extern __shared__ __align__(16) unsigned char pw_smem[];
    PwSlots<T> &S = *reinterpret_cast<PwSlots<T> *>(pw_smem);
    const int t = threadIdx.x;
    const int64_t v = blockIdx.x * (int64_t)PwSlots<T>::NT + t;
    if (v >= n) {
        pdl_wait();
        return;
    }
    const int i = (int)((unsigned)v / (unsigned)nx), j = (int)((unsigned)v - (unsigned)i * (unsigned)nx);   // n <= 2^30
    const bool interior = i >= 2 && i < ny - 2 && j >= 2 && j < nx - 2;
#pragma unroll
    for (int d = 0; d < ND; ++d) copy_async<sizeof(T)>(&S.q[d][t], Pn + (int64_t)d * n + v);
    const T2<T> node = {Pd[v], hv[v]};
    pdl_wait();   // the coefficients are static; the messages are the previous iteration's
    pdl_trigger();
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        // incoming from the neighbour at -off_d: plane d there
        const int si = i - DY(d), sj = j - DX(d);
        if (interior || (si >= 0 && si < ny && sj >= 0 && sj < nx))
            copy_async<sizeof(T2<T>)>(&S.in[d][t], src + (int64_t)d * n + v - ((int64_t)DY(d) * nx + DX(d)));
        else
            S.in[d][t] = T2<T>{T(0), T(0)};
    }
#pragma unroll
    for (int d = 0; d < ND; ++d) copy_async<sizeof(T2<T>)>(&S.old[d][t], src + (int64_t)d * n + v);
    const T cm1 = add_rn(c, T(-1)), keep = add_rn(T(1), -eta);
    asm volatile("cp.async.wait_all;" ::: "memory");
    // leave-one-out sums of the incoming messages, in direction order: suffix sums kept, the prefix
    // sum runs along
    T2<T> in[ND], suf[ND + 1];
#pragma unroll
    for (int d = 0; d < ND; ++d) in[d] = S.in[d][t];
    suf[ND] = T2<T>{T(0), T(0)};
#pragma unroll
    for (int d = ND - 1; d > 0; --d) suf[d] = pair_add(suf[d + 1], in[d]);
    T2<T> pre = {T(0), T(0)};
#pragma unroll
    for (int r = 0; r < ND; ++r) {
        // the message of pair (j, i = j + off_d) back to f_j arrives from direction r = opp(d)
        const int d = OPP(r);
        const int ti = i + DY(d), tj = j + DX(d);
        T2<T> out = {T(0), T(0)};
        if (interior || (ti >= 0 && ti < ny && tj >= 0 && tj < nx))
            out = pw_message(pair_add(pre, suf[r + 1]), in[r], node, S.old[d][t], S.q[d][t], c, inv_c, cm1, keep);
        __stcs(dst + (int64_t)d * n + v, out);
        pre = pair_add(pre, in[r]);
    }
}

// marginals (mean, precision) into mean / var arrays (FP64) or the residual's mean slot
template <typename T>
__global__ void k_pw_marg(DevProblem p, const T *Pd, const T *hv, const T2<T> *msg, T c, double *mean, double *var,
                          int to_residual) {
    const int64_t v = gtid();
    if (v >= p.n) return;
    const int nx = p.nx, ny = p.ny;
    const int64_t n = p.n;
    const int i = (int)(v / nx), j = (int)(v - (int64_t)i * nx);
    double sa = 0.0, sb = 0.0;
    for (int d = 0; d < ND; ++d) {
        const int si = i - DY(d), sj = j - DX(d);
        if (si < 0 || si >= ny || sj < 0 || sj >= nx) continue;
        const T2<T> m = msg[(int64_t)d * n + (int64_t)si * nx + sj];
        sa += (double)m.x;
        sb += (double)m.y;
    }
    const double prec = (double)Pd[v] + (double)c * sa;
    const double mu = ((double)hv[v] + (double)c * sb) / prec;
    if (to_residual) {
        if (p.prec == 0) {   // double-float pair for the FP32 contexts' residual kernels
            const float hi = __double2float_rn(mu);
            ((float2 *)p.mu64)[v] = make_float2(hi, __double2float_rn(mu - (double)hi));
        } else {
            p.mu64[v] = mu;
        }
    } else {
        mean[v] = mu;
        if (var) var[v] = 1.0 / prec;
    }
}

}  // namespace

cudaError_t pw_setup(const DevProblem &p, void *Pd, void *hv, void *Pn, cudaStream_t st) {
    if (p.prec) k_pw_coef<double><<<nblk(p.n), PW_TPB, 0, st>>>(p, (double *)Pd, (double *)hv, (double *)Pn);
    else k_pw_coef<float><<<nblk(p.n), PW_TPB, 0, st>>>(p, (float *)Pd, (float *)hv, (float *)Pn);
    return cudaGetLastError();
}

cudaError_t pw_zero(const DevProblem &p, void *msg, cudaStream_t st) {
    const int64_t count = 2 * ND * p.n;
    if (p.prec) k_pw_zero<double><<<nblk(count), PW_TPB, 0, st>>>((double *)msg, count);
    else k_pw_zero<float><<<nblk(count), PW_TPB, 0, st>>>((float *)msg, count);
    return cudaGetLastError();
}

namespace {
template <typename T>
cudaError_t pw_launch(const DevProblem &p, const void *Pd, const void *hv, const void *Pn, const void *src, void *dst, double c,
                      double eta, cudaStream_t st) {
    static PerDevice<bool> configured;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    bool set = false;
    e = configured.get(dev, set, [](bool &v) {
        v = true;
        return cudaFuncSetAttribute(k_pw_iter<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(PwSlots<T>));
    });
    if (e != cudaSuccess) return e;
    const unsigned blocks = (unsigned)((p.n + PwSlots<T>::NT - 1) / PwSlots<T>::NT);
    return launch_pdl(true, k_pw_iter<T>, dim3(blocks), PwSlots<T>::NT, sizeof(PwSlots<T>), st, p.nx, p.ny, p.n, (const T *)Pd, (const T *)hv,
                      (const T *)Pn, (const T2<T> *)src, (T2<T> *)dst, (T)c, (T)(1.0 / c), (T)eta);
}
}  // namespace

cudaError_t pw_iterate(const DevProblem &p, const void *Pd, const void *hv, const void *Pn, const void *src, void *dst,
                       double c, double eta, cudaStream_t st) {
    return p.prec ? pw_launch<double>(p, Pd, hv, Pn, src, dst, c, eta, st)
                  : pw_launch<float>(p, Pd, hv, Pn, src, dst, c, eta, st);
}

namespace {

// ---- Alg. 2 around the pairwise form: early stopping and upscaling ----

// Partial sums of |m_new - m_old| over both components of every stored message (slots without
// a neighbour hold (0, 0) in both buffers and add nothing), per-thread sums in T, block sums in
// FP64 in a fixed order; part[blockIdx.x] receives the block's sum.
template <typename T> __global__ void k_pw_change(int64_t count, const T *a, const T *b, double *part) {
    __shared__ double sh[PW_TPB];
    T acc = T(0);
    for (int64_t i = gtid(); i < count; i += (int64_t)gridDim.x * PW_TPB) acc += fabs(a[i] - b[i]);
    sh[threadIdx.x] = (double)acc;
    __syncthreads();
    for (int s2 = PW_TPB / 2; s2 > 0; s2 >>= 1) {
        if (threadIdx.x < s2) sh[threadIdx.x] += sh[threadIdx.x + s2];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

__global__ void k_pw_sum(const double *part, int count, double *out) {
    __shared__ double sh[PW_TPB];
    double acc = 0.0;
    for (int q = threadIdx.x; q < count; q += PW_TPB) acc += part[q];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int s2 = PW_TPB / 2; s2 > 0; s2 >>= 1) {
        if (threadIdx.x < s2) sh[threadIdx.x] += sh[threadIdx.x + s2];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sh[0];
}

// "Upscale Messages": fine plane d at node v = coarse plane d at v's parent (floor(i/2),
// floor(j/2)) when the fine node has that neighbour and the parent has it too, else (0, 0).
template <typename T>
__global__ void k_pw_upscale(int nxc, int nyc, int nxf, int nyf, const T2<T> *coarse, T2<T> *fine) {
    const int64_t v = gtid();
    const int64_t nf = (int64_t)nxf * nyf, nc = (int64_t)nxc * nyc;
    if (v >= nf) return;
    const int i = (int)(v / nxf), j = (int)(v - (int64_t)i * nxf);
    const int pi = min(i / 2, nyc - 1), pj = min(j / 2, nxc - 1);
#pragma unroll
    for (int d = 0; d < ND; ++d) {
        T2<T> m;
        m.x = T(0);
        m.y = T(0);
        const int ti = i + DY(d), tj = j + DX(d), ci = pi + DY(d), cj = pj + DX(d);
        if (ti >= 0 && ti < nyf && tj >= 0 && tj < nxf && ci >= 0 && ci < nyc && cj >= 0 && cj < nxc)
            m = coarse[(int64_t)d * nc + (int64_t)pi * nxc + pj];
        fine[(int64_t)d * nf + v] = m;
    }
}

}  // namespace

// directed edges of the pairwise form on an nx x ny grid (pairs within the 12 offsets)
int64_t pw_edge_count(int nx, int ny) {
    int64_t e = 0;
    for (int d = 0; d < ND; ++d) e += (int64_t)std::max(0, nx - std::abs(DX(d))) * std::max(0, ny - std::abs(DY(d)));
    return e;
}

cudaError_t pw_change(const DevProblem &p, const void *a, const void *b, double *part, int nparts, double *out,
                      cudaStream_t st) {
    const int64_t count = 2 * (int64_t)ND * p.n;
    if (p.prec) k_pw_change<double><<<nparts, PW_TPB, 0, st>>>(count, (const double *)a, (const double *)b, part);
    else k_pw_change<float><<<nparts, PW_TPB, 0, st>>>(count, (const float *)a, (const float *)b, part);
    k_pw_sum<<<1, PW_TPB, 0, st>>>(part, nparts, out);
    return cudaGetLastError();
}

cudaError_t pw_upscale(const DevProblem &fine, const DevProblem &coarse, const void *coarse_msg, void *fine_msg,
                       cudaStream_t st) {
    if (fine.prec != coarse.prec) return cudaErrorInvalidValue;
    if (fine.prec)
        k_pw_upscale<double><<<nblk(fine.n), PW_TPB, 0, st>>>(coarse.nx, coarse.ny, fine.nx, fine.ny,
                                                              (const double2 *)coarse_msg, (double2 *)fine_msg);
    else
        k_pw_upscale<float><<<nblk(fine.n), PW_TPB, 0, st>>>(coarse.nx, coarse.ny, fine.nx, fine.ny,
                                                             (const float2 *)coarse_msg, (float2 *)fine_msg);
    return cudaGetLastError();
}

cudaError_t pw_marginals(const DevProblem &p, const void *Pd, const void *hv, const void *msg, double c, double *mean,
                         double *var, int to_residual, cudaStream_t st) {
    if (p.prec)
        k_pw_marg<double><<<nblk(p.n), PW_TPB, 0, st>>>(p, (const double *)Pd, (const double *)hv, (const double2 *)msg,
                                                        c, mean, var, to_residual);
    else
        k_pw_marg<float><<<nblk(p.n), PW_TPB, 0, st>>>(p, (const float *)Pd, (const float *)hv, (const float2 *)msg,
                                                       (float)c, mean, var, to_residual);
    return cudaGetLastError();
}

}  // namespace gabp
