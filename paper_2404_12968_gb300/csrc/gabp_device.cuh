// Device-side arithmetic of one GaBP iteration, shared by the split and fused kernels.
//
// Message layout in HBM (both precisions, T = float or double):
//   prior messages: 5 planes of n (eta, Lambda) pairs, "outgoing" order: plane d at cell c
//     holds the message from the factor of cell c to node c + off_d, d = C, W, E, S, N
//     (off = 0, -1, +1, -nx, +nx).  Slots whose neighbour does not exist hold (0, 0).
//   observation messages: per observation (sorted by base cell), 8 values
//     eta_0..eta_3, Lambda_0..Lambda_3, one per bilinear corner.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace gabp {

// ---- back-to-back launches of the iteration kernels (programmatic dependent launch) ----
// An iteration kernel touches nothing that an earlier kernel writes or reads before pdl_wait() has
// returned: every kernel before it is complete then.  pdl_trigger() lets the next kernel's blocks
// start, so that launch latency and prologue overlap this one's tail; it follows the wait (with it
// first, several waiting kernels fill the SMs' slots unevenly: 256^2 5.4 -> 6.3 us).  Message
// pointers of such kernels carry no __restrict__ / __ldg (loads that the compiler may hoist).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
template <typename... P, typename... A>
inline cudaError_t launch_pdl(bool overlap, void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t st,
                              const A &...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = overlap ? 1 : 0;   // without it pdl_wait() returns at once
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

enum { DIR_C = 0, DIR_W = 1, DIR_E = 2, DIR_S = 3, DIR_N = 4 };

template <typename T> struct vec2;
template <> struct vec2<float> { using type = float2; };
template <> struct vec2<double> { using type = double2; };
template <typename T> using T2 = typename vec2<T>::type;

// Smallest normal number.
template <typename T> __device__ __forceinline__ T tiny_normal();
template <> __device__ __forceinline__ float tiny_normal<float>() { return 1.17549435e-38f; }
template <> __device__ __forceinline__ double tiny_normal<double>() { return 2.2250738585072014e-308; }

// Floor of a cavity precision relative to its slot's a^2 (see factor_messages).
template <typename T> __device__ __forceinline__ T lam_floor_rel();
template <> __device__ __forceinline__ float lam_floor_rel<float>() { return 1e-20f; }
template <> __device__ __forceinline__ double lam_floor_rel<double>() { return 1e-20; }

template <typename T> __device__ __forceinline__ T pos_inf();
template <> __device__ __forceinline__ float pos_inf<float>() { return __int_as_float(0x7f800000); }
template <> __device__ __forceinline__ double pos_inf<double>() {
    return __longlong_as_double(0x7ff0000000000000LL);
}

// Reciprocal.  FP32: the hardware approximation rcp.approx.ftz.f32, within 1 ulp over the
// range the callers use (they never pass 0, a denormal or an infinity: cavity precisions are
// floored at a normal number, and V is at least var > 0 and at most about 5e20).  FP64: below.
__device__ __forceinline__ float recip(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// FP64 reciprocal without an FP64 operation.  FP64 is the scarce unit of this GPU (measured: one
// warp instruction per 64 to 76 cycles and SM quarter, whatever its parallelism), while its integer
// and FP32 units are nearly idle in the FP64 kernels, so the quotient of the 53-bit significands is
// formed there, by Newton's method in mixed fixed point:
//   x = 2^E m, M = 2^52 m;  m = mh + ml with mh its 24-bit rounding;
//   r = the FP32 approximation of 1 / mh, e = 1 - m r (two exact-product FMAs, |e| <= 1.6 2^-23),
//   R0 = 2^53 (r + r (e + e^2)), an integer within 2^-46 of the quotient, relatively;
//   D = 2^105 - M R0, whose low 64 bits hold it (|D| <= 2^60);
//   R = R0 + round(R0 D / 2^105): within 0.5 + 2^-14 of 2^53 / m, the IEEE quotient but for near ties.
// 1 / x = 2^(-E - 53) R.  About 35 integer and FP32 instructions in the place of seven FP64 ones of
// IEEE sequence.  Exponents outside 2^+-1000 (zero, denormal, huge, infinite, NaN) set `out` and leave
// a meaningless value: the caller divides instead, once for all its reciprocals, so that several
// of them interleave without a branch (a branch in each made five of them take 1,250 cycles).
__device__ __forceinline__ double recip_fixed(double x, bool &out) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned ex = (hi >> 20) & 0x7ffu;
    out |= ex - 23u >= 2000u;
    const unsigned mhi = (hi & 0xfffffu) | 0x100000u;                 // M = mhi : lo
    const int tl = (int)(lo << 3) >> 3;                               // M's low 29 bits, signed: ml = 2^-52 tl
    const float mh = __uint_as_float(0x3f800000u + (((hi << 3) | (lo >> 29)) & 0x7fffffu) + ((lo >> 28) & 1u));
    const float r = recip(mh);
    const float e = __fmaf_rn(-0x1p-52f * __int2float_rn(tl), r, __fmaf_rn(-mh, r, 1.f));
    const unsigned ri = __float2uint_rn(r * 0x1p24f);                 // exact: r in [0.5, 1] has 24 bits
    const int ci = __float2int_rn(0x1p53f * r * __fmaf_rn(e, e, e));
    const unsigned long long R0 = ((unsigned long long)ri << 29) + (unsigned long long)(long long)ci;
    const unsigned rl = (unsigned)R0, rh = (unsigned)(R0 >> 32);
    // bits 32..63 of M R0; D's upper half is its complement (the dropped carry is 2^-20 of a unit)
    const int dh = (int)~(__umulhi(lo, rl) + lo * rh + mhi * rl);
    const long long R = (long long)R0 + __float2int_rn(0x1p-20f * r * __int2float_rn(dh));
    const unsigned long long bits = ((unsigned long long)(2044u - ex) << 52) + (unsigned long long)R;
    return __longlong_as_double((long long)(bits | ((unsigned long long)(hi & 0x80000000u) << 32)));
}

// The reciprocal in the message formulas: FP32 recip(); FP64 recip_fixed() (FAST) or the division.
template <bool FAST> __device__ __forceinline__ float recip_or(float x, bool &) { return recip(x); }
template <bool FAST> __device__ __forceinline__ double recip_or(double x, bool &out) {
    return FAST ? recip_fixed(x, out) : 1.0 / x;
}

// x == 0 and max(x, f) for f > 0 (f where x is NaN or negative).  FP64: on the bits, in the integer
// unit (a positive double orders as its bits do).
__device__ __forceinline__ bool is_zero(float x) { return x == 0.f; }
__device__ __forceinline__ bool is_zero(double x) { return (__double_as_longlong(x) << 1) == 0; }
__device__ __forceinline__ float floor_at(float x, float f) { return fmaxf(x, f); }
__device__ __forceinline__ double floor_at(double x, double f) {
    const long long b = __double_as_longlong(x);
    return b >= __double_as_longlong(f) && b <= 0x7ff0000000000000LL ? x : f;
}

// Explicitly rounded arithmetic for the message formulas: no multiply is contracted into a
// fused multiply-add unless written as one, so every kernel (scalar or packed two-lane FP32)
// evaluates them with the same roundings and produces the same bits.
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }

// Two-term compensated sum (TwoSum accumulation, Knuth TAOCP vol. 2 4.2.2): hi + lo carries
// the running sum to about twice the working precision.  Used for the belief sums so that
// the cavity (belief minus one message) keeps its relative accuracy even when that message
// dominates the belief.  FP64: the same exact error by Fast2Sum (Dekker 1971) on the operands
// ordered by exponent, three additions instead of six (the ordering runs in the integer unit), and
// no renormalisation, which the cavity (hi - own) + lo does not need: its error bound is the same.
template <typename T> struct CompSum {
    T hi, lo;
    // start from a first term: identical to adding it to an empty sum (TwoSum(0, x) = (x, 0))
    __device__ __forceinline__ explicit CompSum(T first) : hi(first), lo(T(0)) {}
    // hi += x; returns the rounding error
    __device__ __forceinline__ T step(T x) {
        const T t = hi + x;
        T e;
        if constexpr (sizeof(T) == 8) {
            const bool sw = (__double2hiint(x) & 0x7fffffff) > (__double2hiint(hi) & 0x7fffffff);
            const T big = sw ? x : hi, small = sw ? hi : x;
            e = small - (t - big);
        } else {
            const T z = t - hi;
            e = (hi - (t - z)) + (x - z);
        }
        hi = t;
        return e;
    }
    __device__ __forceinline__ void second(T x) { lo = step(x); }   // the second term: lo is still 0
    __device__ __forceinline__ void add(T x) { lo += step(x); }
    // renormalise so that hi = fl(hi + lo) (FP32)
    __device__ __forceinline__ void finish() {
        if constexpr (sizeof(T) == 4) {
            T t = hi + lo;
            lo = lo - (t - hi);
            hi = t;
        }
    }
};

// A compensated belief: (eta_hi, eta_lo, lam_hi, lam_lo).
template <typename T> struct Belief {
    T ehi, elo, lhi, llo;
};

// Adds the observation messages into node (x, y) that come from the base cells of one row:
// base (x-1, row) with corner cl for indices [lo, mid) and base (x, row) with corner cr for
// [mid, hi).  The two ranges are adjacent in the base-sorted observation array, so the terms
// are added in increasing observation index; every iteration kernel uses this order (corners
// 1, 0 from the node's row, then 3, 2 from the row below).  Four terms' loads are in flight together; the
// rest one by one, in a loop that is not unrolled: most nodes have a term or two, and code for more of
// them costs those.  Sweep kernel, 63^2 nodes with 0.1, 3 and 10 observations each: 103, 295 and 660 us per
// iteration; one loop as the compiler unrolls it 110, 301 and 655, by words 109, 294 and 667.
constexpr int OBS_LOADS = 4;
template <typename T>
__device__ __forceinline__ void add_obs_pair(CompSum<T> &se, CompSum<T> &sl, const T *O, int lo, int mid,
                                             int hi, int cl, int cr) {
    const T2<T> *Q = reinterpret_cast<const T2<T> *>(O) + 4u * (unsigned)lo;
    int l = mid - lo, n = hi - lo;
#pragma unroll 1
    for (; n >= OBS_LOADS; n -= OBS_LOADS, l -= OBS_LOADS, Q += 4 * OBS_LOADS) {
        T2<T> x[OBS_LOADS];
#pragma unroll
        for (int q = 0; q < OBS_LOADS; ++q) x[q] = Q[4 * q + (q < l ? cl : cr)];
#pragma unroll
        for (int q = 0; q < OBS_LOADS; ++q) {
            se.add(x[q].x);
            sl.add(x[q].y);
        }
    }
#pragma unroll 1
    for (; n > 0; --n, --l, Q += 4) {
        const T2<T> q = Q[l > 0 ? cl : cr];
        se.add(q.x);
        sl.add(q.y);
    }
}

// Cavity of one edge: the belief minus the edge's own incoming message, evaluated as
// (hi - own) + lo (App. A, variable-to-factor message).
template <typename T>
__device__ __forceinline__ void cavity(const Belief<T> &b, T own_eta, T own_lam, T &eta_c, T &lam_c) {
    lam_c = (b.lhi - own_lam) + b.llo;
    eta_c = (b.ehi - own_eta) + b.elo;
}

// Factor-to-variable messages of a rank-1 factor exp(-(1/(2 var)) (a . x - r)^2) with K slots
// (App. A factor-to-variable message generalised to K variables): for every slot v
//   V_v = var + sum_{u != v} a_u^2 / lam_u,   m_v = r - sum_{u != v} a_u eta_u / lam_u,
//   Lambda_v = a_v^2 / V_v,                   eta_v = a_v m_v / V_v.
// Leave-one-out sums come from prefix and suffix sums (no "total minus own" cancellation).
// Slots with a_u = 0 are skipped.  A cavity precision below 1e-20 a_u^2 (zero and negative
// included; in FP32 also below the smallest normal number) is raised to that floor.  Such a
// cavity is in the limit lam -> 0 with finite information, the linear potential exp(eta x):
// the messages to the other slots then equal that limit, (-a_v eta_u / a_u, 0), to a relative
// 1e-20 V, and nothing overflows.  (Far from the observations the precision recursion drives
// some cavity precisions far below the FP32 range while their information stays finite;
// treating them as carrying no information would drop that information.)
// FAST: returns false where a reciprocal was out of the fast form's range (FP64 only).
template <typename T, int K, bool FAST>
__device__ __forceinline__ bool factor_messages_as(const T (&a)[K], T var, T r, const T (&lam)[K], const T (&eta)[K],
                                                   T (&L)[K], T (&E)[K]) {
    bool out = false;
    T t[K], p[K];
#pragma unroll
    for (int u = 0; u < K; ++u) {
        if (is_zero(a[u])) {
            t[u] = T(0);
            p[u] = T(0);
        } else {
            const T a2 = mul_rn(a[u], a[u]);
            // a NaN cavity precision is floored
            const T fl = floor_at(mul_rn(lam_floor_rel<T>(), a2), tiny_normal<T>());
            const T rl = recip_or<FAST>(floor_at(lam[u], fl), out);
            t[u] = mul_rn(a2, rl);
            p[u] = mul_rn(a[u], mul_rn(eta[u], rl));
        }
    }
    T preV[K], preM[K];
    preV[0] = var;
    preM[0] = T(0);
#pragma unroll
    for (int v = 1; v < K; ++v) {
        preV[v] = add_rn(preV[v - 1], t[v - 1]);
        preM[v] = add_rn(preM[v - 1], p[v - 1]);
    }
    T sufV = T(0), sufM = T(0);
#pragma unroll
    for (int v = K - 1; v >= 0; --v) {
        const T V = add_rn(preV[v], sufV);
        const T M = add_rn(preM[v], sufM);
        const T rV = recip_or<FAST>(V, out);
        L[v] = mul_rn(mul_rn(a[v], a[v]), rV);
        E[v] = mul_rn(mul_rn(a[v], add_rn(r, -M)), rV);
        sufV = add_rn(sufV, t[v]);
        sufM = add_rn(sufM, p[v]);
    }
    return !out;
}
template <typename T, int K>
__device__ __forceinline__ void factor_messages(const T (&a)[K], T var, T r, const T (&lam)[K],
                                                const T (&eta)[K], T (&L)[K], T (&E)[K]) {
    if (!factor_messages_as<T, K, true>(a, var, r, lam, eta, L, E)) factor_messages_as<T, K, false>(a, var, r, lam, eta, L, E);
}

// Damped update m_t = beta m_{t-1} + (1 - beta) m_new, evaluated as the fused multiply-add
// m_new + beta (m_{t-1} - m_new).
template <typename T> __device__ __forceinline__ T damp(T old, T fresh, T beta) {
    return fma_rn(beta, add_rn(old, -fresh), fresh);
}

// Update of the factor of one cell with all four neighbours, FP64: the messages of
// factor_messages for a = (aC, -1, -1, -1, -1) with the products by -1 and 1 and the sums with an
// exact zero left out, then the damping.  a2 = aC^2 and flC = the floor of the centre's cavity
// precision are rounded on the host; b are the beliefs of the slots' nodes, own the cell's
// messages, out the damped new ones.  74 FP64 operations.  Returns false, out unset, where a
// reciprocal is out of recip_fixed()'s range: the general form serves those cells.
__device__ __forceinline__ bool cell_update_interior(double aC, double a2, double flC, double var, bool has_r, double r,
                                                     const Belief<double> *const (&b)[5], const double2 (&own)[5],
                                                     double beta, double2 (&out)[5]) {
    double t[5], p[5];
    bool oor = false;
#pragma unroll
    for (int u = 0; u < 5; ++u) {
        double eta, lam;
        cavity(*b[u], own[u].x, own[u].y, eta, lam);
        const double rl = recip_fixed(floor_at(lam, u == 0 ? flC : lam_floor_rel<double>()), oor);
        t[u] = u == 0 ? mul_rn(a2, rl) : rl;
        p[u] = u == 0 ? mul_rn(aC, mul_rn(eta, rl)) : -mul_rn(eta, rl);
    }
    double preV[5], preM[5];
    preV[0] = var;
    preV[1] = add_rn(var, t[0]);
    preM[0] = 0.0;
    preM[1] = p[0];
#pragma unroll
    for (int v = 2; v < 5; ++v) {
        preV[v] = add_rn(preV[v - 1], t[v - 1]);
        preM[v] = add_rn(preM[v - 1], p[v - 1]);
    }
    double sufV = 0.0, sufM = 0.0;
#pragma unroll
    for (int v = 4; v >= 0; --v) {
        const double V = v == 4 ? preV[4] : add_rn(preV[v], sufV);
        double M = v == 4 ? preM[4] : v == 0 ? sufM : add_rn(preM[v], sufM);
        if (has_r) M = add_rn(M, -r);
        const double rV = recip_fixed(V, oor);
        const double L = v == 0 ? mul_rn(a2, rV) : rV;
        const double E = v == 0 ? mul_rn(mul_rn(aC, -M), rV) : mul_rn(M, rV);
        out[v].x = fma_rn(beta, add_rn(own[v].x, -E), E);
        out[v].y = fma_rn(beta, add_rn(own[v].y, -L), L);
        if (v > 0) {
            sufV = v == 4 ? t[4] : add_rn(sufV, t[v]);
            sufM = v == 4 ? p[4] : add_rn(sufM, p[v]);
        }
    }
    return !oor;
}

// Number of existing 4-neighbours of node (i, j).
__device__ __forceinline__ int grid_degree(int i, int j, int nx, int ny) {
    return (j > 0) + (j < nx - 1) + (i > 0) + (i < ny - 1);
}

}  // namespace gabp
