// nu_periodic_search: Sect. 2.3-2.4 on the products of the linear search.
//
// For each trial period P every (duration d, phase j) cell gathers its single
// events at epochs T_k = T_ref + (j/n_phi + k) P, linearly interpolated in time
// between the bracketing grid epochs, and combines them with Eq. result using the
// biased estimates of Eq. sigma_delta:
//   pass 1:  S_inv = sum 1/s_k^2,  S_d = sum Delta_k / s_k^2,  S_L = sum gain_k
//            sigma^2 = 1/S_inv,    Delta = sigma^2 S_d
//   pass 2:  pen = sum [ln s_k^2 - ln(sigma^2 + s_k^2) + (Delta_k - Delta)^2/(s_k^2 + sigma^2)]
//            ln P = S_L - pen / 2
// The cell with the largest ln P (first in duration-major, phase order;
// Eq. phi0) gives Q(P) = Delta / sigma.
//
// Epoch arithmetic (T, the bracket, the weight) is FP64 in both precisions
// so that which epochs take part is decided exactly as in FP64; the event
// values and sums are FP64 (NU_FP64) or FP32 with compensated sums (NU_MIXED).
#include <algorithm>
#include <climits>
#include <cmath>
#include <mutex>
#include <string>
#include <vector>

#include "factor_core.cuh"
#include "filter.cuh"
#include "fold.cuh"
#include "nu_internal.cuh"

namespace nu {

// ------------------------------------------------------------------ helpers
// Reciprocals from the hardware approximation refined by Newton-Raphson
// (y <- y (2 - x y), each step doubling the correct bits); x > 0 finite.
__device__ __forceinline__ double rcp64(double x) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    double e = fma(-x, y, 1.0);
    y = fma(y, e, y);
    e = fma(-x, y, 1.0);
    return fma(y, e, y);
}
__device__ __forceinline__ float rcp32(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float rsqrt32(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lg2_32(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}


struct FoldGeom {
    const double* t0s;
    int64_t n_t0;
    double t_ref;
    double t_last;
    double dt;          // phase step
    double inv_dt;
    double gap_max;     // gap_factor * dt
    const int* bucket;  // bucket[b] = #{i : t0_i <= t_ref + b*dt}
    int64_t n_bucket;
};

__device__ __forceinline__ void fill_bucket(const double* __restrict__ t0s, int64_t n_t0,
                                            double t_ref, double dt, int64_t b,
                                            int* __restrict__ bucket) {
    const double edge = t_ref + (double)b * dt;
    int64_t lo = 0, hi = n_t0;          // count of t0 <= edge
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (t0s[mid] <= edge) lo = mid + 1; else hi = mid;
    }
    bucket[b] = (int)lo;
}

// Per-(duration, epoch) node records for the exact path.
template <typename T>
__device__ __forceinline__ T node_sigma(T d, T v, T l) {
    return (isfinite(d) && isfinite(v) && isfinite(l) && v > T(0)) ? sqrt(v) : T(NAN);
}

template <typename T>
__device__ __forceinline__ Node8<T> make_node8(const T* __restrict__ depth,
                                               const T* __restrict__ var,
                                               const T* __restrict__ gain,
                                               const double* __restrict__ t0, int64_t gid,
                                               int64_t i, int64_t n, double gap_max) {
    Node8<T> r;
    r.d = depth[gid];
    r.l = gain[gid];
    r.s = node_sigma<T>(r.d, var[gid], r.l);
    r.ig = T(NAN);
    r.dd = T(NAN);
    r.ds = T(NAN);
    r.dl = T(NAN);
    r.pad = T(0);
    if (i + 1 < n) {
        const double gap = t0[i + 1] - t0[i];
        if (gap <= gap_max && gap > 0.0) r.ig = (T)(1.0 / gap);
        const T d1 = depth[gid + 1], l1 = gain[gid + 1];
        const T s1 = node_sigma<T>(d1, var[gid + 1], l1);
        r.dd = d1 - r.d;
        r.ds = s1 - r.s;
        r.dl = l1 - r.l;
    }
    return r;
}

// Regular-grid test for the slot path: every epoch within 1e-3 slot of
// t_ref + s*dt with strictly increasing slots.  slot_of[i] = s.
__global__ void k_slots(const double* __restrict__ t0s, int64_t n_t0, double t_ref,
                        double inv_dt, int* __restrict__ slot_of, int* __restrict__ irregular) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n_t0) return;
    const double u = (t0s[i] - t_ref) * inv_dt;
    const double s = rint(u);
    bool bad = !(fabs(u - s) <= 1e-3) || !(s >= 0.0) || s > 2.0e9;
    if (i > 0) {
        const double up = rint((t0s[i - 1] - t_ref) * inv_dt);
        bad = bad || !(s > up);
    }
    slot_of[i] = bad ? -1 : (int)s;
    if (bad) atomicExch(irregular, 1);
}

__device__ __forceinline__ Node4<float> slot_record(const float* __restrict__ depth,
                                                    const float* __restrict__ var,
                                                    const float* __restrict__ gain,
                                                    int64_t gid) {
    const float d = depth[gid], v = var[gid], l = gain[gid];
    const bool ok = isfinite(d) && isfinite(v) && isfinite(l) && v > 0.f;
    return Node4<float>{d, ok ? sqrtf(v) : NAN, l, 0.f};
}

// Slot records (mixed path): node values placed at their slot, NaN sigma in
// empty slots.  One thread per (duration, epoch); slots were cleared to NaN.
// L (if given): the filters' gain table, rows of ns, cleared to 0: the largest
// gain on the interval that starts at the slot.
__global__ void k_slot_fill(const float* __restrict__ depth, const float* __restrict__ var,
                            const float* __restrict__ gain, const int* __restrict__ slot_of,
                            int64_t n_t0, int n_D, int64_t n_slots,
                            Node4<float>* __restrict__ rec, float* __restrict__ L, int64_t ns) {
    const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (gid >= n_t0 * (int64_t)n_D) return;
    const int64_t d = gid / n_t0, i = gid - d * n_t0;
    const int s = slot_of[i];
    if (s < 0 || s >= n_slots) return;
    const Node4<float> r = slot_record(depth, var, gain, gid);
    rec[d * n_slots + s] = r;
    if (L && i + 1 < n_t0 && slot_of[i + 1] == s + 1) {
        const Node4<float> q = slot_record(depth, var, gain, gid + 1);
        if (!isnan(r.s) && !isnan(q.s)) L[d * ns + s] = slot_gain(r, q);
    }
}

__global__ void k_fill_nan(Node4<float>* rec, int64_t n) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    rec[i] = Node4<float>{NAN, NAN, NAN, 0.f};
}

// Compensated FP32 and plain FP64 sums.  The products that enter the sums are
// written as the fused operations they are (add_prod, fma), so that every
// kernel that evaluates a cell rounds alike.
template <typename T> struct KSum {
    T s, c;
    __device__ __forceinline__ void init() { s = T(0); c = T(0); }
    __device__ __forceinline__ void add_y(T y) {
        const T t = __fadd_rn(s, y);
        c = __fsub_rn(__fsub_rn(t, s), y);
        s = t;
    }
    __device__ __forceinline__ void add(T x) { add_y(__fsub_rn(x, c)); }
    __device__ __forceinline__ void add_prod(T a, T b) { add_y(__fmaf_rn(a, b, -c)); }
};
template <> struct KSum<double> {
    double s;
    __device__ __forceinline__ void init() { s = 0.0; }
    __device__ __forceinline__ void add(double x) { s = __dadd_rn(s, x); }
    __device__ __forceinline__ void add_prod(double a, double b) { s = __fma_rn(a, b, s); }
};
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }

struct Best {
    double lnp;
    long long cell;
    double depth;
    double sigma;
};

__device__ __forceinline__ bool better(const Best& a, const Best& b) {
    // a beats b: larger ln P, ties to the smaller cell index
    if (a.lnp > b.lnp) return true;
    if (a.lnp < b.lnp) return false;
    return a.cell < b.cell;
}

__device__ __forceinline__ void write_best(const Best& b, int64_t p, int64_t n_phi, double t_ref,
                                           double P, double* Q_out, double* T0_out,
                                           int* Didx_out, double* dep_out, double* sig_out,
                                           double* lnp_out) {
    if (b.cell == LLONG_MAX) {
        Q_out[p] = 0.0;
        T0_out[p] = NAN;
        Didx_out[p] = -1;
        dep_out[p] = NAN;
        sig_out[p] = NAN;
        lnp_out[p] = -INFINITY;
    } else {
        const int d = (int)(b.cell / n_phi);
        const int64_t j = b.cell - (int64_t)d * n_phi;
        Q_out[p] = b.depth / b.sigma;
        T0_out[p] = __dadd_rn(t_ref, __dmul_rn((double)j / (double)n_phi, P));
        Didx_out[p] = d;
        dep_out[p] = b.depth;
        sig_out[p] = b.sigma;
        lnp_out[p] = b.lnp;
    }
}

// MAXT: the largest block size the caller is launched with
template <int MAXT = 256>
__device__ __forceinline__ Best block_argmax(Best best) {
    __shared__ Best sh[MAXT];
    sh[threadIdx.x] = best;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w && better(sh[threadIdx.x + w], sh[threadIdx.x]))
            sh[threadIdx.x] = sh[threadIdx.x + w];
        __syncthreads();
    }
    return sh[0];
}

// Bound used to skip the second pass of a cell that cannot be the argmax.
// With x_k = sigma^2 / s_k^2 (sum x_k = 1 by Eq. sigma_delta) the log terms of
// Eq. result contribute -1/2 sum ln(s_k^2/(sigma^2+s_k^2)) = 1/2 sum ln(1+x_k)
// <= 1/2 sum x_k = 1/2.  Because sigma^2 <= s_k^2, the depth terms satisfy
//   sum (Delta_k - Delta)^2 / (s_k^2 + sigma^2) >= 1/2 sum (Delta_k - Delta)^2 / s_k^2
//                                          = 1/2 (S_dd - S_d^2 / S_inv)
// with S_dd = sum Delta_k^2 / s_k^2 from the first pass.  Hence
//   ln P <= S_L + 1/2 - 1/4 (S_dd - S_d^2 / S_inv),
// and a cell whose bound is below the best ln P found so far cannot win:
// skipping its second pass changes no result.  The margins (on the bound and
// on the cancellation in S_dd - S_d^2/S_inv) are far above the rounding of
// each precision.
__device__ __forceinline__ bool cannot_win(double s_l, double s_inv, double s_d, double s_dd,
                                           double best) {
    const double q = fmax(0.0, s_dd - s_d * s_d / s_inv - 1e-9 * s_dd);
    const double ub = s_l + 0.5 - 0.25 * q;
    return ub + 1e-6 * fmax(1.0, fabs(ub)) < best;
}

__device__ __forceinline__ bool bad_period(double P, const FoldGeom& g) {
    // a period must be finite, > 0 and give at most 1e9 epochs and phases
    return !(P > 0.0) || !isfinite(P) || g.t_last - g.t_ref > 1.0e9 * P ||
           P / g.dt > 1.0e9;
}

__device__ __forceinline__ void write_bad(int64_t p, double* Q_out, double* T0_out,
                                          int* Didx_out, double* dep_out, double* sig_out,
                                          double* lnp_out) {
    Q_out[p] = NAN;
    T0_out[p] = NAN;
    Didx_out[p] = -1;
    dep_out[p] = NAN;
    sig_out[p] = NAN;
    lnp_out[p] = NAN;
}

// ------------------------------------------------ exact path (FP64 epochs)
// Order-preserving integer key of a non-NaN double (so comparisons of times
// run on the integer pipe; -0.0 never occurs among the epochs compared here).
__device__ __forceinline__ long long okey(double x) {
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}

// largest i with t0[i] <= T starting from a guess (exact)
__device__ __forceinline__ int64_t bracket_from(const FoldGeom& g, long long kT, int64_t i) {
    while (i + 1 < g.n_t0 && okey(g.t0s[i + 1]) <= kT) ++i;
    while (i > 0 && okey(g.t0s[i]) > kT) --i;
    return i;
}

__device__ __forceinline__ bool nan64(double x) {
    return (__double_as_longlong(x) & 0x7fffffffffffffffLL) > 0x7ff0000000000000LL;
}

__device__ __forceinline__ int64_t bracket_guess(const FoldGeom& g, double T) {
    int64_t b = (int64_t)((T - g.t_ref) * g.inv_dt);
    b = b < 0 ? 0 : (b >= g.n_bucket ? g.n_bucket - 1 : b);
    const int64_t i = (int64_t)g.bucket[b] - 1;
    return i < 0 ? 0 : i;
}

template <typename T> __device__ __forceinline__ T rcp_t(T x);
template <> __device__ __forceinline__ double rcp_t<double>(double x) { return rcp64(x); }
template <> __device__ __forceinline__ float rcp_t<float>(float x) { return rcp32(x); }

// One single event at epoch Tk: interpolated depth, sigma and gain.
template <typename T>
__device__ __forceinline__ bool event_exact(const FoldGeom& g, const Node8<T>* __restrict__ nd,
                                            double Tk, int64_t& i, T& dk, T& s, T& lk) {
    i = bracket_from(g, okey(Tk), i);
    const Node8<T> a = nd[i];
    const T w = (T)((Tk - g.t0s[i]) * (double)a.ig);   // NaN across a gap / at the end
    s = fma(w, a.ds, a.s);
    if (sizeof(T) == 8 ? nan64((double)s) : isnan(s)) return false;
    dk = fma(w, a.dd, a.d);
    lk = fma(w, a.dl, a.l);
    return true;
}

// Fixed-point (24.40) walk of the slot grid u = (T - t_ref)/dt used to guess
// brackets; the decisions themselves are FP64 comparisons with T.
struct SlotWalk {
    unsigned long long u0, ustep;
};
__device__ __forceinline__ SlotWalk slot_walk(double phi, double R) {
    const double SCALE = 1099511627776.0;   // 2^40
    SlotWalk w;
    const double a = phi * R * SCALE, b = R * SCALE;
    w.u0 = a < 4.0e18 ? (unsigned long long)llrint(a) : 4000000000000000000ull;
    w.ustep = b < 4.0e18 ? (unsigned long long)llrint(b) : 4000000000000000000ull;
    return w;
}
__device__ __forceinline__ int64_t guess_at(const FoldGeom& g, unsigned long long u) {
    int64_t b = (int64_t)(u >> 40);
    b = b >= g.n_bucket ? g.n_bucket - 1 : b;
    const int64_t i = (int64_t)g.bucket[b] - 1;
    return i < 0 ? 0 : i;
}

template <typename T>
struct ExactAcc {
    KSum<T> s_inv, s_d, s_l;
    T s_dd;                // sum Delta_k^2 / s_k^2 (bound only, plain sum)
    int K;
    __device__ __forceinline__ void init() {
        s_inv.init();
        s_d.init();
        s_l.init();
        s_dd = T(0);
        K = 0;
    }
    __device__ __forceinline__ void add(T dk, T s, T lk) {
        const T iv = rcp_t<T>(mul_rn(s, s));
        const T div = mul_rn(dk, iv);
        s_inv.add(iv);
        s_d.add(div);
        s_dd = fma(div, dk, s_dd);
        s_l.add(lk);
        ++K;
    }
    __device__ __forceinline__ bool cannot_win(double best) const {
        return nu::cannot_win((double)s_l.s, (double)s_inv.s, (double)s_d.s, (double)s_dd,
                              best);
    }
};

// second sum of Eq. result: ln s_k^2 - ln(sigma^2 + s_k^2) accumulated as the
// log of a product of ratios in [1/2, 1] (renormalised), plus
// (Delta_k - Delta)^2 / (s_k^2 + sigma^2)
template <typename T>
struct ExactPen {
    KSum<T> quad;
    double prod;
    int expo, cnt;
    float lsum;
    T s2, Dl;
    __device__ __forceinline__ void init(T s2_, T Dl_) {
        quad.init();
        prod = 1.0;
        expo = 0;
        cnt = 0;
        lsum = 0.f;
        s2 = s2_;
        Dl = Dl_;
    }
    __device__ __forceinline__ void add(T dk, T s) {
        const T sk2 = mul_rn(s, s);
        const T iden = rcp_t<T>(add_rn(sk2, s2));
        const T r = dk - Dl;
        quad.add_prod(mul_rn(r, r), iden);
        if (sizeof(T) == 8) {
            prod *= (double)mul_rn(sk2, iden);
            if ((++cnt & 255) == 0) {
                const int e = ((__double2hiint(prod) >> 20) & 0x7ff) - 1023;
                prod = __hiloint2double(__double2hiint(prod) - (e << 20), __double2loint(prod));
                expo += e;
            }
        } else {
            lsum += lg2_32((float)mul_rn(sk2, iden));
        }
    }
    // both sums of the penalty
    __device__ __forceinline__ double total() const {
        if (sizeof(T) == 8)
            return __dadd_rn(fma((double)expo, 0.69314718055994530942, log(prod)),
                             (double)quad.s);
        return fma((double)lsum, 0.69314718055994530942, (double)quad.s);
    }
};

// Order-preserving unsigned key of a non-NaN double, for a shared atomic max.
__device__ __forceinline__ unsigned long long max_key(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double from_max_key(unsigned long long k) {
    const unsigned long long b = (k >> 63) ? (k & 0x7fffffffffffffffull) : ~k;
    return __longlong_as_double((long long)b);
}

// A cell that survived the bound after its first pass, queued for the second.
template <typename T>
struct QCell {
    double phi;
    unsigned long long u0;
    long long cell;
    double s_l;
    T s2, Dl;
    int d;
    int kmax;
};

// Per-period constants of the exact evaluation of a cell.
struct CellCtx {
    double P, nphi_d, rphi;
    SlotWalk swp, swk;         // per-phase and per-epoch steps of the slot guess
    unsigned long long ulast;  // t_last on the same fixed-point scale
    float inv_ustep32;
    long long klast;           // order key of t_last
};

__device__ __forceinline__ CellCtx cell_ctx(const FoldGeom& g, double P, int64_t n_phi) {
    CellCtx c;
    c.P = P;
    const double R = P * g.inv_dt;
    c.swp = slot_walk(1.0 / (double)n_phi, R);
    c.swk = slot_walk(0.0, R);
    const double SCALE = 1099511627776.0;   // 2^40
    const double ulast_d = (g.t_last - g.t_ref) * g.inv_dt * SCALE;
    c.ulast = ulast_d < 4.0e18 ? (unsigned long long)llrint(ulast_d) : 4000000000000000000ull;
    c.inv_ustep32 = (float)(4294967296.0 / (double)c.swk.ustep);
    c.klast = okey(g.t_last);
    // phase j / n_phi: reciprocal plus one FMA correction of the quotient
    // (Markstein 1990), instead of a division per cell
    c.nphi_d = (double)n_phi;
    c.rphi = 1.0 / c.nphi_d;
    return c;
}

// The constants of one period that do not depend on the curve (phase count,
// fixed-point walk steps and their reciprocals), computed as screen_period
// and cell_ctx compute them.  The batched fold takes them from a table built
// once per call, so that its (curve, period) items, bound by the FP64 pipe
// when their cells are short, skip these divisions.
struct PeriodConst {
    int64_t n_phi;
    double R;                          // P / dt
    unsigned long long ustep, uph;     // screen steps (0 when R 2^40 >= 4e18)
    float c_inv_ustep32;
    SlotWalk swp, swk;
    double nphi_d, rphi;
};

// The table entry of period P (P must not be a bad period of the curves).
__device__ __forceinline__ PeriodConst period_const(double P, double dt, double inv_dt) {
    PeriodConst pc;
    const double SCALE = 1099511627776.0;   // 2^40
    pc.n_phi = (int64_t)ceil(P / dt);
    pc.R = P * inv_dt;
    if (pc.R * SCALE < 4.0e18) {
        pc.ustep = (unsigned long long)llrint(pc.R * SCALE);
        pc.uph = (unsigned long long)llrint(pc.R / (double)pc.n_phi * SCALE);
    } else {
        pc.ustep = pc.uph = 0;
    }
    pc.swp = slot_walk(1.0 / (double)pc.n_phi, pc.R);
    pc.swk = slot_walk(0.0, pc.R);
    pc.c_inv_ustep32 = (float)(4294967296.0 / (double)pc.swk.ustep);
    pc.nphi_d = (double)pc.n_phi;
    pc.rphi = 1.0 / pc.nphi_d;
    return pc;
}

// The position of a curve's last epoch for the exact paths' epoch counts.
static inline unsigned long long exact_uspan(double t_ref, double t_last, double dt) {
    const double u = (t_last - t_ref) * (1.0 / dt) * 1099511627776.0;
    return u < 4.0e18 ? (unsigned long long)llrint(u) : 4000000000000000000ull;
}
// cell_ctx from a table entry and the curve's last position (the same values,
// no FP64 arithmetic).
__device__ __forceinline__ CellCtx cell_ctx(const FoldGeom& g, double P, const PeriodConst& pc,
                                            unsigned long long uspan) {
    CellCtx c;
    c.P = P;
    c.swp = pc.swp;
    c.swk = pc.swk;
    c.ulast = uspan;
    c.inv_ustep32 = pc.c_inv_ustep32;
    c.klast = okey(g.t_last);
    c.nphi_d = pc.nphi_d;
    c.rphi = pc.rphi;
    return c;
}

// Table of period constants (invalid periods get placeholder entries; the
// folds test a period before they read its entry).
__device__ __forceinline__ void fill_period_const(const double* __restrict__ periods, int64_t i,
                                                  double dt, PeriodConst* __restrict__ out) {
    const double P = periods[i];
    if (!(P > 0.0) || !isfinite(P) || P / dt > 1.0e9) {
        out[i] = PeriodConst{1, 0.0, 0, 0, 0.f, {0, 0}, {0, 0}, 1.0, 1.0};
        return;
    }
    out[i] = period_const(P, dt, 1.0 / dt);
}

__global__ void k_period_consts(const double* __restrict__ periods, int64_t n_P, double dt,
                                PeriodConst* __restrict__ out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n_P) fill_period_const(periods, i, dt, out);
}

// Per-period constants of the slot path: phases, and the epoch and phase
// steps in 24.40 fixed point, in a table (k_slot_prep, k_slot_periods) or, where
// there is no room for one, per item by the same function.  bad marks a period
// that is not folded for any curve (the curve's own limit, a span of more
// than 1e9 periods, is tested per curve).
struct SlotPeriod {
    int64_t n_phi;
    unsigned long long ustep, uph;
    int bad;
};
// The position of a curve's last epoch (< 2^62 by the host's span check).
__host__ __device__ inline unsigned long long slot_ulast(double t_ref, double t_last, double dt) {
    return (unsigned long long)llrint((t_last - t_ref) / dt * 1099511627776.0);
}
__device__ __forceinline__ SlotPeriod slot_period(double P, double dt) {
    SlotPeriod sp{1, 0ull, 0ull, 1};
    if (!(P > 0.0) || !isfinite(P) || P / dt > 1.0e9) return sp;
    const double SCALE = 1099511627776.0;                      // 2^40
    const double R = P / dt;                                   // slots per period
    sp.n_phi = (int64_t)ceil(R);
    sp.ustep = R * SCALE < 4.0e18 ? (unsigned long long)llrint(R * SCALE)
                                  : 4000000000000000000ull;
    // phase j starts at j * (R / n_phi) slots; per-cell work stays integer
    sp.uph = (unsigned long long)llrint(R / (double)sp.n_phi * SCALE);
    sp.bad = 0;
    return sp;
}
__global__ void k_slot_periods(const double* __restrict__ periods, int64_t n_P, double dt,
                               SlotPeriod* __restrict__ out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n_P) out[i] = slot_period(periods[i], dt);
}

size_t period_const_bytes() {
    return sizeof(PeriodConst) > sizeof(SlotPeriod) ? sizeof(PeriodConst) : sizeof(SlotPeriod);
}

__device__ __forceinline__ double cell_phi(const CellCtx& c, int64_t j) {
    const double jd = (double)j;
    const double q0 = jd * c.rphi;
    return fma(fma(-q0, c.nphi_d, jd), c.rphi, q0);
}

__device__ __forceinline__ double epoch_time(const FoldGeom& g, const CellCtx& c, double phi,
                                             double kd) {
    return __dadd_rn(g.t_ref, __dmul_rn(__dadd_rn(phi, kd), c.P));
}

// number of epochs with T <= t_last: integer estimate, then the exact
// comparisons of the definition
__device__ __forceinline__ int64_t cell_kmax(const FoldGeom& g, const CellCtx& c, double phi,
                                             unsigned long long u0) {
    int64_t kk = u0 > c.ulast ? 0
                              : (int64_t)((float)(unsigned)((c.ulast - u0) >> 32) *
                                          c.inv_ustep32) + 1;
    while (kk > 0 && okey(epoch_time(g, c, phi, (double)(kk - 1))) > c.klast) --kk;
    while (okey(epoch_time(g, c, phi, (double)kk)) <= c.klast) ++kk;
    return kk;
}

// First and second sums of one cell over epochs k0, k0 + ks, ... < kmax.
template <typename T>
__device__ __forceinline__ void cell_pass1(const FoldGeom& g, const Node8<T>* __restrict__ nd,
                                           const CellCtx& c, double phi, unsigned long long u0,
                                           int64_t kmax, int k0, int ks, ExactAcc<T>& a1) {
    unsigned long long u = u0 + (unsigned long long)k0 * c.swk.ustep;
    const unsigned long long us = (unsigned long long)ks * c.swk.ustep;
    double kd = (double)k0;
    const double kds = (double)ks;
    for (int64_t k = k0; k < kmax; k += ks, u += us, kd += kds) {
        const double Tk = epoch_time(g, c, phi, kd);
        T dk, sk, lk;
        int64_t i = guess_at(g, u);
        if (event_exact<T>(g, nd, Tk, i, dk, sk, lk)) a1.add(dk, sk, lk);
    }
}
template <typename T>
__device__ __forceinline__ void cell_pass2(const FoldGeom& g, const Node8<T>* __restrict__ nd,
                                           const CellCtx& c, double phi, unsigned long long u0,
                                           int64_t kmax, int k0, int ks, ExactPen<T>& a2) {
    unsigned long long u = u0 + (unsigned long long)k0 * c.swk.ustep;
    const unsigned long long us = (unsigned long long)ks * c.swk.ustep;
    double kd = (double)k0;
    const double kds = (double)ks;
    for (int64_t k = k0; k < kmax; k += ks, u += us, kd += kds) {
        const double Tk = epoch_time(g, c, phi, kd);
        T dk, sk, lk;
        int64_t i = guess_at(g, u);
        if (event_exact<T>(g, nd, Tk, i, dk, sk, lk)) a2.add(dk, sk);
    }
}

// One period P of one light curve: every (duration, phase) cell, then the
// block argmax; results at index p of the outputs.  Called by all threads of
// the block.  Cells are processed in waves of blockDim: every thread runs the
// first pass of one cell, the cells whose bound can still beat the block's
// best are compacted into a shared queue, and the queue's second passes run
// densely (a warp instruction costs the same however many lanes are active).
template <typename T, int MAXT = 256>
__device__ __forceinline__ void fold_exact_one(const FoldGeom& g,
                                               const Node8<T>* __restrict__ nodes,
                                               int n_D, double P, int64_t p,
                                               double* __restrict__ Q_out,
                                               double* __restrict__ T0_out,
                                               int* __restrict__ Didx_out,
                                               double* __restrict__ dep_out,
                                               double* __restrict__ sig_out,
                                               double* __restrict__ lnp_out) {
    __shared__ QCell<T> sh_q[MAXT];
    __shared__ int sh_nq;
    __shared__ unsigned long long sh_best;
    if (bad_period(P, g)) {
        if (threadIdx.x == 0) write_bad(p, Q_out, T0_out, Didx_out, dep_out, sig_out, lnp_out);
        return;
    }
    const int64_t n_phi = (int64_t)ceil(P / g.dt);
    const int64_t n_cells = n_phi * n_D;
    const CellCtx c = cell_ctx(g, P, n_phi);
    double bl = -INFINITY;
    long long bc = LLONG_MAX;
    T bD = T(NAN), bs2 = T(NAN);
    if (threadIdx.x == 0) {
        sh_nq = 0;
        sh_best = max_key(-INFINITY);
    }
    __syncthreads();
    // cells walk (duration, phase) incrementally: no 64-bit division per cell
    int d = (int)(threadIdx.x / n_phi);
    int64_t j = (int64_t)threadIdx.x - (int64_t)d * n_phi;
    for (int64_t base = 0; base < n_cells; base += blockDim.x, j += blockDim.x) {
        while (j >= n_phi) {
            j -= n_phi;
            ++d;
        }
        const int64_t cell = base + threadIdx.x;
        if (cell < n_cells) {
            const double phi = cell_phi(c, j);
            const Node8<T>* nd = nodes + (int64_t)d * g.n_t0;
            const unsigned long long u0 = (unsigned long long)j * c.swp.u0;
            const int64_t kmax = cell_kmax(g, c, phi, u0);
            ExactAcc<T> a1;
            a1.init();
            cell_pass1<T>(g, nd, c, phi, u0, kmax, 0, 1, a1);
            const double best_now = fmax(bl, from_max_key(sh_best));
            if (a1.K > 0 && !a1.cannot_win(best_now)) {
                const T s2 = T(1) / a1.s_inv.s;
                const int q = atomicAdd(&sh_nq, 1);
                sh_q[q] = QCell<T>{phi, u0, (long long)cell, (double)a1.s_l.s, s2,
                                   s2 * a1.s_d.s, d, (int)kmax};
            }
        }
        __syncthreads();
        const int nq = sh_nq;
        for (int q = threadIdx.x; q < nq; q += blockDim.x) {
            const QCell<T> qc = sh_q[q];
            const Node8<T>* nd = nodes + (int64_t)qc.d * g.n_t0;
            ExactPen<T> a2;
            a2.init(qc.s2, qc.Dl);
            cell_pass2<T>(g, nd, c, qc.phi, qc.u0, qc.kmax, 0, 1, a2);
            const double lnp = qc.s_l - 0.5 * a2.total();
            if (!(lnp == lnp)) continue;   // NaN never selected
            if (lnp > bl || (lnp == bl && qc.cell < bc)) {
                bl = lnp;
                bc = qc.cell;
                bD = qc.Dl;
                bs2 = qc.s2;
            }
            atomicMax(&sh_best, max_key(lnp));
        }
        __syncthreads();
        if (threadIdx.x == 0) sh_nq = 0;
        __syncthreads();
    }
    Best best{-INFINITY, LLONG_MAX, NAN, NAN};
    if (bc != LLONG_MAX) best = Best{bl, bc, (double)bD, sqrt((double)bs2)};
    const Best b = block_argmax<MAXT>(best);
    if (threadIdx.x == 0)
        write_best(b, p, n_phi, g.t_ref, P, Q_out, T0_out, Didx_out, dep_out, sig_out, lnp_out);
}

// The period a block (or a batch item) folds.  Short periods hold few cells
// of many epochs each, and in the FP64 fold they are the longest blocks: a
// grid whose periods run downwards (uniform in frequency, say) is folded from
// its far end, so that those blocks start first (C2 FP64: 8.5 ms in
// ascending order, 13.8 ms descending).  Any order gives the same results.
__device__ __forceinline__ int64_t period_slot(int64_t b, const double* __restrict__ periods,
                                              int64_t n_P) {
    // (by integer keys: a NaN only changes the order)
    return okey(periods[n_P - 1]) < okey(periods[0]) ? n_P - 1 - b : b;
}

template <typename T>
__global__ void __launch_bounds__(256)
k_fold_exact(FoldGeom g, const Node8<T>* __restrict__ nodes, int n_D,
             const double* __restrict__ periods, int64_t n_P, double* __restrict__ Q_out,
             double* __restrict__ T0_out, int* __restrict__ Didx_out,
             double* __restrict__ dep_out, double* __restrict__ sig_out,
             double* __restrict__ lnp_out) {
    if ((int64_t)blockIdx.x >= n_P) return;
    const int64_t p = period_slot(blockIdx.x, periods, n_P);
    fold_exact_one<T>(g, nodes, n_D, periods[p], p, Q_out, T0_out, Didx_out, dep_out,
                          sig_out, lnp_out);
}

// ------------------------------ FP64 path: FP32 screen, exact survivors
// Every cell is first screened with FP32 events: an upper bound on its ln P
// (the bound of cannot_win, tightened below) computed from FP32 values with
// an error term that covers every rounding of the screen, on an epoch set
// that is provably the exact path's.  Only cells whose bound reaches the
// best ln P found so far are evaluated exactly (FP64 epochs and values, the
// same code as the exact path); a skipped cell cannot be the argmax, so the
// outputs are those of the exact evaluation of every cell.
//
// Tighter bound.  With x_k = sigma^2/s_k^2 and x_max = max_k x_k,
//   sum (Delta_k - Delta)^2/(s_k^2 + sigma^2) >= q / (1 + x_max),
//   q = sum (Delta_k - Delta)^2 / s_k^2 = S_dd - S_d^2/S_inv,
// so ln P <= S_L + 1/2 - q / (2 (1 + x_max)).
//
// Epoch set.  Epoch positions are walked in 24.40 fixed point of the slot
// grid (u = (T - t_ref)/dt), the epochs' own positions are stored on the same
// scale, and the interval of an event is the last epoch position <= u.  The
// walk differs from the FP64 epochs by at most e_pos (bounded per period
// from the fixed-point rounding and the FP64 rounding of T), so the interval
// is the exact path's whenever u is farther than delta >> e_pos from every
// epoch; within delta of an epoch (or of t_last, for the epoch count) the
// event's T is computed in FP64 exactly as the exact path does and the
// interval is taken by the same comparisons.  The screen's epoch set and
// intervals are therefore the exact path's.
//
// Error term.  An FP32 event value x (depth, sigma, gain) differs from the
// FP64 one by at most cv (|x_i| + |x_{i+1}|) (node and slope rounding,
// weight rounding and position error, the FMA; an event in the band of an
// epoch takes its exact interval and an FP32 weight within 5u of the exact
// one), with |x_i| + |x_{i+1}| <=
// 2|x| + |x_{i+1} - x_i| accumulated per cell.  Intervals whose end sigmas
// differ by more than a factor 3 (or outside the other limits of the
// screening record) are not screened, so |ds|/s <= 2 and the
// relative error of each 1/s_k^2 is at most gam = 2.2 cv (2 + 2) + 6u; sums
// of K positive terms carry at most (K + 2)u.  With these:
//   S_L     <= sl + (cv + (K+2)u) sum (2|l_k| + |dl_k|)
//   sqrt(q) >= sqrt(q_fp32_lo / (1 + gam + (K+2)u)) - cv sqrt(sum a_k^2/s_k^2)
//   x_max   <= min(1, ivmax/sinv (1 + 4 gam + 2(K+2)u))
// (triangle inequality in the 1/s^2-weighted norm for q).  Overflow or NaN
// anywhere makes the bound +inf or NaN, which never skips a cell.


struct ScreenGeom {
    const ScreenRec* rec;              // duration-major rows of n_t0 records
    const ulonglong2* vpair;           // (position of epoch i, of epoch i+1), 24.40
                                       // slots from t_ref; the last .y is 2^64 - 1
    const ScreenRec* srec;             // the same records placed at their epochs'
                                       // slots: duration-major rows of n_slots
    int64_t n_slots;
    const unsigned* reg;               // [0]: an epoch is off the slot grid,
                                       // [1]: max |offset from its slot| (float bits)
    int on;                            // screening allowed for this curve
    int f32;                           // the exact events are FP32 (mixed precision)
};

// Node sigma of one (duration, epoch) in FP64 (NaN when invalid).
template <typename T>
__device__ __forceinline__ double sigma_at(const T* depth, const T* var, const T* gain,
                                           int64_t o) {
    return (double)node_sigma<T>(depth[o], var[o], gain[o]);
}

// Slot of every epoch on the regular grid u = (t0 - t_ref)/dt and the largest
// offset from it; reg[0] is set when the slots are not strictly increasing
// or fall outside [0, n_slots).  reg must be zero on entry.
__device__ __forceinline__ void slot_offset(const double* __restrict__ t0, int64_t i,
                                            double inv_dt, int64_t n_slots,
                                            int* __restrict__ slot_of,
                                            unsigned* __restrict__ reg) {
    const double u = (t0[i] - t0[0]) * inv_dt;
    const double s = rint(u);
    bool bad = !(s >= 0.0) || !(s < (double)n_slots);
    if (i > 0) bad = bad || !(s > rint((t0[i - 1] - t0[0]) * inv_dt));
    slot_of[i] = bad ? -1 : (int)s;
    if (bad) atomicOr(&reg[0], 1u);
    atomicMax(&reg[1], __float_as_uint((float)fabs(u - s) * 1.0001f));
}

// Screening record of epoch i of a curve with n epochs (gid indexes the
// (duration, epoch) arrays; d is the duration), also placed at the epoch's
// slot, and for the first duration row the pair of epoch positions.
template <typename T>
__device__ __forceinline__ void make_screen(const T* __restrict__ depth,
                                            const T* __restrict__ var,
                                            const T* __restrict__ gain,
                                            const double* __restrict__ t0, int64_t gid,
                                            int64_t i, int64_t n, int64_t d, double gap_max,
                                            double dt, ScreenRec* __restrict__ out,
                                            ScreenRec* __restrict__ sout,
                                            int64_t n_slots, const int* __restrict__ slot_of,
                                            ulonglong2* __restrict__ vpair) {
    // an interval needs both ends valid and a gap in (0, gap_max]
    bool v0 = i + 1 < n;
    if (v0) {
        const double gap = t0[i + 1] - t0[i];
        v0 = gap > 0.0 && gap <= gap_max && !isnan(sigma_at<T>(depth, var, gain, gid)) &&
             !isnan(sigma_at<T>(depth, var, gain, gid + 1));
    }
    ScreenRec r;
    unsigned flags = 0u;
    const double d0 = (double)depth[gid], l0 = (double)gain[gid];
    r.d = (float)d0;
    r.l = (float)l0;
    if (v0) {
        const double s0 = sigma_at<T>(depth, var, gain, gid);
        const double s1 = sigma_at<T>(depth, var, gain, gid + 1);
        const double d1 = (double)depth[gid + 1], l1 = (double)gain[gid + 1];
        const double gap = t0[i + 1] - t0[i];
        r.s = (float)s0;
        r.dd = (float)(d1 - d0);
        r.ds = (float)(s1 - s0);
        r.dl = (float)(l1 - l0);
        r.wsc = (float)(2.384185791015625e-07 * dt / gap);   // 2^-22 dt / gap
        // outside the error model: very close epochs, or values whose FP32
        // sums could overflow
        const bool odd = gap < 0.25 * dt || !(s0 >= 1e-12 && s0 <= 1e12) ||
                         !(s1 >= 1e-12 && s1 <= 1e12) || !(s1 <= 3.0 * s0) ||
                         !(s0 <= 3.0 * s1) || !(fabs(d0) <= 1e8 * s0) ||
                         !(fabs(d1) <= 1e8 * s1) || !(fabs(l0) <= 1e20) || !(fabs(l1) <= 1e20);
        if (odd) {
            // sigma +inf marks the interval for the screen (flags for the
            // exact events)
            flags = 1u;
            r.s = INFINITY;
            r.ds = 0.f;
        }
    } else {
        r.s = NAN;
        r.dd = 0.f;
        r.ds = 0.f;
        r.dl = 0.f;
        r.wsc = 0.f;
    }
    r.flags = flags;
    out[gid] = r;
    if (sout) {
        const int sl = slot_of[i];
        if (sl >= 0 && sl < n_slots) sout[d * n_slots + sl] = r;
    }
    if (d == 0) {
        auto pos = [&](int64_t k) -> unsigned long long {
            const double v = (t0[k] - t0[0]) / dt * 1099511627776.0;
            return v < 9.0e18 ? (unsigned long long)llrint(v) : 9000000000000000000ull;
        };
        vpair[i] = make_ulonglong2(pos(i), i + 1 < n ? pos(i + 1) : ~0ull);
    }
}

// Slot records start as invalid intervals (slots without an epoch).
__device__ __forceinline__ ScreenRec no_interval() {
    return ScreenRec{0.f, NAN, 0.f, 0.f, 0.f, 0.f, 0.f, 0u};
}
__global__ void k_fill_screen(ScreenRec* __restrict__ rec, int64_t n) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    rec[i] = no_interval();
}

template <typename T>
__global__ void k_screen(const T* __restrict__ depth, const T* __restrict__ var,
                         const T* __restrict__ gain, const double* __restrict__ t0s,
                         int64_t n_t0, int n_D, double gap_max, double dt,
                         ScreenRec* __restrict__ rec, ScreenRec* __restrict__ srec,
                         int64_t n_slots, const int* __restrict__ slot_of,
                         ulonglong2* __restrict__ vpair) {
    const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (gid >= n_t0 * (int64_t)n_D) return;
    const int64_t d = gid / n_t0, i = gid - d * n_t0;
    make_screen<T>(depth, var, gain, t0s, gid, i, n_t0, d, gap_max, dt, rec, srec, n_slots,
                   slot_of, vpair);
}

// Per-period constants of the screen.
struct ScreenPeriod {
    unsigned long long uph, ustep, delta;
    unsigned long long uend;   // epochs walk while u < uend = (last epoch) + delta
    float wscale;   // 2^22 / dt (FP32): weight of an event in the band of an epoch
    float cv;       // error coefficient of an FP32 event value
    float hw;       // 1/2 - dw, dw the half-width of the band around an epoch as
                    // an interval weight: an event is in a band when |w - 1/2| > hw
    bool on;
    bool slots;     // regular grid: events from the slot records
};

// The curve-dependent constants of the screen (the walk's error bound, the
// band around epochs, the regular-grid test); sp holds the period's steps.
__device__ __forceinline__ ScreenPeriod screen_period_curve(const FoldGeom& g,
                                                            const ScreenGeom& sg, double P,
                                                            int64_t n_phi, double R,
                                                            double span, ScreenPeriod sp) {
    const double SCALE = 1099511627776.0;   // 2^40
    const unsigned long long ulast = sg.vpair[g.n_t0 - 1].x;
    // position error of the walk against the FP64 epochs, in 2^-40 slots:
    // half a unit per phase and epoch step, the rounding of T, t0 and vpos
    const double kb = span / R + 2.0;
    const double e_pos = 0.5 * ((double)n_phi + kb) + 4.0 +
                         8.881784197001252e-16 * (fabs(g.t_ref) + fabs(g.t_last) + P) *
                             g.inv_dt * SCALE;
    const double delta = 16.0 * e_pos + 1048576.0;          // + 2^-20 slot
    sp.on = delta < 1.6e10;                                  // below 2^-6 slot
    sp.delta = (unsigned long long)delta;
    sp.uend = ulast + sp.delta;
    // regular grid: every epoch within 2^-10 slot of its own slot.  The error
    // terms below grow with the largest offset; a phase step taken as the
    // median spacing of FP64 times carries a relative rounding of about
    // 1e-11, so on long curves (seven sectors: 1.2e-7 slot) the offsets are
    // well above the rounding of one sector's times.
    const float off = sg.srec ? __uint_as_float(sg.reg[1]) : 1.f;
    sp.slots = sg.srec && sg.reg[0] == 0u && off <= 9.765625e-04f;
    double e_w;
    float dw;
    if (sp.slots) {
        // the weight is the fraction of the slot: position error, the
        // epochs' offsets (3 x, both ends), 24-bit truncation
        dw = (float)(1.01 * (delta / SCALE + (double)off) + 2.4e-7);
        e_w = e_pos / SCALE + 3.0 * (double)off + 1.1920928955078125e-07;
    } else {
        // dt/gap <= 4 on a screened interval; 2^-22-slot truncation
        dw = (float)(4.04 * delta / SCALE + 2.0e-6);
        e_w = 4.0 * e_pos / SCALE + 9.5367431640625e-07;
    }
    // (the weight of an event in the band of an epoch, computed in FP32 by
    // screen_exact_event, is within 5u of the exact one: 3u more than the
    // smallest e_w)
    sp.cv = (float)(8.0 * 5.9604644775390625e-08 + 2.0 * (e_w + 3.0 * 5.9604644775390625e-08));
    // on a regular grid an event within one fraction unit of an epoch's slot
    // may take the epoch's values: off by at most ws times a slope, and for
    // sigma ws times 2 sigma (adjacent sigmas within a factor 3)
    if (sp.slots)
        sp.cv = fmaxf(sp.cv, (float)(2.02 * (1.1920928955078125e-07 + e_pos / SCALE + (double)off) +
                                     8.0 * 5.9604644775390625e-08));
    // mixed precision: the exact event itself is computed in FP32 (node
    // differences, weight and FMA: a few units of |x_i| + |x_{i+1}|)
    if (sg.f32) sp.cv += 8.0f * 5.9604645e-08f;
    sp.hw = 0.5f - dw;
    sp.wscale = (float)(4194304.0 * g.inv_dt);
    return sp;
}

__device__ __forceinline__ ScreenPeriod screen_period(const FoldGeom& g, const ScreenGeom& sg,
                                                      double P, const PeriodConst& pc) {
    ScreenPeriod sp;
    const double SCALE = 1099511627776.0;   // 2^40
    const double R = pc.R;
    const double span = (g.t_last - g.t_ref) * g.inv_dt;
    sp.on = sg.on != 0 && R * SCALE < 4.0e18 && span < 8388608.0;
    sp.slots = false;
    sp.uph = sp.ustep = sp.delta = sp.uend = 0;
    sp.wscale = 0.f;
    sp.cv = 0.f;
    sp.hw = 0.5f;
    if (!sp.on) return sp;
    sp.ustep = pc.ustep;
    sp.uph = pc.uph;
    return screen_period_curve(g, sg, P, pc.n_phi, R, span, sp);
}

// Sums of the screen (see above) and the bound they give.
// Integer-to-float conversions run on the FP64 pipe of this GPU, so the
// screen counts events in a float and builds weights from bit patterns.
struct ScreenAcc {
    float sinv, sd, sdd, sdd2, sl, sabs, ivmax, ivmin;
    float K;                 // number of events (exact in FP32 below 2^24)
    __device__ __forceinline__ void init() {
        sinv = sd = sdd = sdd2 = sl = sabs = ivmax = 0.f;
        ivmin = INFINITY;
        K = 0.f;
    }
    // event (depth dk, sigma s, gain lk) on an interval with depth and gain
    // differences dd, dl.  The error budget of the depths uses
    // (|Delta_i| + |Delta_{i+1}|)^2 <= (2|dk| + |dd|)^2 <= 8 dk^2 + 2 dd^2.
    __device__ __forceinline__ void add(float dk, float s, float lk, float dd, float dl) {
        const float iv = rcp32(s * s);
        const float div = dk * iv;
        sinv += iv;
        sd += div;
        sdd = fmaf(div, dk, sdd);
        sl += lk;
        sdd2 = fmaf(dd * dd, iv, sdd2);
        sabs += fmaf(2.f, fabsf(lk), fabsf(dl));
        ivmax = fmaxf(ivmax, iv);
        ivmin = fminf(ivmin, iv);
        K += 1.f;
    }
    // Hardware reciprocal / reciprocal square root (relative error below
    // 2^-21, counted as 8u per use) with every term rounded the safe way.
    // The q term only lowers the bound, so the cheaper S_L + 1/2 + margins
    // is returned when it already falls below the threshold bf.
    // *lb receives a lower bound on the cell's ln P (-inf when not computed):
    // the log terms are at least ln(1 + x_max) / (2 x_max) (ln(1 + x) is
    // concave and the x_k sum to 1), the depth terms at most q / (2 (1 + x_min)).
    __device__ __forceinline__ float bound(float cv, float bf, float* lb) const {
        if (K == 0.f) return -INFINITY;
        const float U = 5.9604645e-8f;                        // 2^-24
        const float sk = (K + 2.f) * U;
        const float e_l = 1.05f * (cv + sk) * sabs;
        const float ub0 = sl + e_l + 0.5f + 8.f * U * (sabs + 1.f);
        if (ub0 < bf) return ub0;
        // |ds|/s <= 2 on a screened interval (adjacent sigmas within a factor 3)
        const float gam = 2.2f * cv * 4.f + 6.f * U;
        const float r = rcp32(sinv);
        const float qc = fmaf(-sd * sd, r, sdd);
        const float qcl = qc - fmaf(4.f, K, 32.f) * U * sdd;
        float q_lo = 0.f;
        if (qcl > 0.f) {
            const float x1 = qcl * rcp32(1.f + gam + sk) * (1.f - 16.f * U);
            const float a = x1 * rsqrt32(x1) * (1.f - 16.f * U);
            const float y = fmaf(8.f, sdd, 2.f * sdd2) * (1.f + 2.f * gam + sk) * (1.f + 8.f * U);
            const float e = y > 0.f ? 1.05f * cv * (y * rsqrt32(y)) * (1.f + 16.f * U) : 0.f;
            if (a > e) q_lo = (a - e) * (a - e) * (1.f - 8.f * U);
        }
        const float x_hi = fminf(1.f, ivmax * r * (1.f + 4.f * gam + 2.f * sk + 24.f * U));
        {
            const float qch = fmaxf(qc + fmaf(4.f, K, 32.f) * U * sdd, 0.f);
            const float x1 = qch * (1.f + 4.f * gam + 2.f * sk + 16.f * U);
            const float y = fmaf(8.f, sdd, 2.f * sdd2) * (1.f + 2.f * gam + sk) * (1.f + 8.f * U);
            const float a = x1 > 0.f ? x1 * rsqrt32(x1) * (1.f + 16.f * U) : 0.f;
            const float e = y > 0.f ? 1.05f * cv * (y * rsqrt32(y)) * (1.f + 16.f * U) : 0.f;
            const float q_hi = (a + e) * (a + e) * (1.f + 8.f * U);
            const float x_lo = ivmin * r * (1.f - 4.f * gam - 2.f * sk - 24.f * U);
            const float lg = 0.69314718f * lg2_32(1.f + x_hi) * rcp32(x_hi);
            const float l = sl - e_l + 0.5f * lg - 0.5f * q_hi * rcp32(1.f + x_lo) -
                            (sabs + q_hi + 1.f) * 4e-6f;
            *lb = l == l ? l : -INFINITY;
        }
        return sl + e_l + 0.5f - 0.5f * q_lo * rcp32(1.f + x_hi) * (1.f - 16.f * U) +
               8.f * U * (sabs + q_lo + 1.f);
    }
};

// The event of epoch k whose walk position lies in the band of an epoch
// (or of t_last): T and its interval exactly as the exact path computes
// them (FP64 epoch, comparisons of the doubles' integer keys), then the
// weight (T - t_i)/gap in FP32 from the interval's screening record (within
// 5u of the exact path's weight, which the error coefficient covers) and the
// FP32 values as for any other event.  Returns 0 when there is no event, 1
// when the event was added, 2 when its interval is outside the error model.
__device__ __forceinline__ int screen_exact_event(const FoldGeom& g,
                                                  const ScreenRec* __restrict__ rd,
                                                  const CellCtx& c, double phi, int64_t k,
                                                  unsigned long long u, float wscale,
                                                  ScreenAcc& acc) {
    const double Tk = epoch_time(g, c, phi, (double)k);
    const long long kT = okey(Tk);
    if (kT > c.klast) return 0;                 // after the last epoch
    const int64_t i = bracket_from(g, kT, guess_at(g, u));
    const ScreenRec r = rd[i];
    if (r.flags) return 2;
    // wsc = 2^-22 dt/gap: (T - t_i) 2^22/dt wsc = (T - t_i)/gap
    const float w = (float)(Tk - g.t0s[i]) * wscale * r.wsc;
    const float s = fmaf(w, r.ds, r.s);
    if (isnan(s)) return 0;                     // the interval has no event
    acc.add(fmaf(w, r.dd, r.d), s, fmaf(w, r.dl, r.l), r.dd, r.dl);
    return 1;
}

// Upper bound on ln P of cell (j, duration rows rd / rs) whose first
// epoch is at u0 (see above): -inf when the cell has no event, +inf when an
// event falls on an interval outside the screen's error model; any value
// below bf when the cell is already known not to reach bf.  *lb: see
// ScreenAcc::bound (left as it is when the cell is not bounded).
__device__ __forceinline__ float screen_cell(const FoldGeom& g, const ScreenGeom& sg,
                                             const ScreenRec* __restrict__ rd,
                                             const ScreenRec* __restrict__ rs,
                                             const ScreenPeriod& sp, const CellCtx& c,
                                             int64_t j, unsigned long long u0, float bf,
                                             float* lb) {
    // epochs up to u < ulast + delta: those within delta of t_last (the last
    // epoch's position) fall in the band around it and take the exact event,
    // which drops T > t_last
    double phi = 0.0;
    bool have_phi = false;
    ScreenAcc acc;
    acc.init();
    unsigned long long u = u0;
    // the exact event of the epoch at u (rare: within the band of an epoch);
    // false when the cell must be evaluated exactly
    auto exact = [&]() -> bool {
        if (!have_phi) {
            phi = cell_phi(c, j);
            have_phi = true;
        }
        const int64_t k = (int64_t)((u - u0) / sp.ustep);
        return screen_exact_event(g, rd, c, phi, k, u, sp.wscale, acc) != 2;
    };
    if (sp.slots) {
        // regular grid: the interval is the slot's, the weight its fraction
        const unsigned ns1 = (unsigned)(sg.n_slots - 1);
        auto slot = [&](unsigned long long x) { return min((unsigned)(x >> 40), ns1); };
        auto visit = [&](const ScreenRec& r) -> bool {
            // fraction of the slot: its top 23 bits as the mantissa of a float in [1, 2)
            const float w =
                __uint_as_float(0x3f800000u | (unsigned)((u >> 17) & 0x7fffffu)) - 1.0f;
            if (fabsf(w - 0.5f) > sp.hw) {
                // in the band of an epoch.  A position within one unit of the
                // fraction of the epoch's slot m (every event of a period of
                // whole slots) takes the epoch's values when both intervals
                // at m are screened: the event lies on one of them, within
                // ws = 2^-23 + e_pos + off of m, so its values are the epoch's
                // within ws times either slope (the error coefficient covers
                // it, with the larger slope as the event's).  Otherwise the
                // exact event.
                if (w != 0.f && w < 0.99999988f) return exact();
                const unsigned sl = slot(u);
                const unsigned m = w < 0.5f ? sl : sl + 1u;
                if (m == 0u || m >= ns1) return exact();
                const ScreenRec L = m == sl ? rs[m - 1u] : r;
                const ScreenRec R = m == sl ? r : rs[m];
                if (!(L.s < INFINITY) || !(R.s < INFINITY)) return exact();
                acc.add(R.d, R.s, R.l, fmaxf(fabsf(L.dd), fabsf(R.dd)),
                        fmaxf(fabsf(L.dl), fabsf(R.dl)));
                return true;
            }
            const float s = fmaf(w, r.ds, r.s);
            if (!(s < INFINITY)) return s != s;   // NaN: no event; +inf: not screened
            acc.add(fmaf(w, r.dd, r.d), s, fmaf(w, r.dl, r.l), r.dd, r.dl);
            return true;
        };
        // two records in flight, alternating (no register moves)
        ScreenRec ra = rs[slot(u)], rb;
        while (u < sp.uend) {
            rb = rs[slot(u + sp.ustep)];
            if (!visit(ra)) return INFINITY;
            u += sp.ustep;
            if (!(u < sp.uend)) break;
            ra = rs[slot(u + sp.ustep)];
            if (!visit(rb)) return INFINITY;
            u += sp.ustep;
        }
        return acc.bound(sp.cv, bf, lb);
    }
    const int64_t nb1 = g.n_bucket - 1;
    int bnext = g.bucket[min((int64_t)(u >> 40), nb1)];
    for (; u < sp.uend; u += sp.ustep) {
        // interval guess from the bucket table (the next epoch's entry is
        // fetched one iteration ahead), verified against the stored positions
        int64_t i = bnext > 0 ? (int64_t)bnext - 1 : 0;
        bnext = g.bucket[min((int64_t)((u + sp.ustep) >> 40), nb1)];
        ulonglong2 v = sg.vpair[i];
        ScreenRec r = rd[i];
        if (u >= v.y || u < v.x) {
            while (u >= v.y) v = sg.vpair[++i];
            while (u < v.x) v = sg.vpair[--i];
            r = rd[i];
        }
        const long long sdu = (long long)(u - v.x);
        // position in units of 2^-22 slot (23 bits for du < 2 slots) as a float
        const float w = (__uint_as_float(0x4b000000u | ((unsigned)(sdu >> 18) & 0x7fffffu)) -
                         8388608.0f) * r.wsc;
        const float s = fmaf(w, r.ds, r.s);
        // within delta of either end (on a valid interval: w within dw of 0
        // or 1, dw >= 4 delta in slots as dt/gap <= 4): the exact event
        const bool near = isnan(s) ? ((unsigned long long)sdu < sp.delta || v.y - u < sp.delta)
                                   : fabsf(w - 0.5f) > sp.hw;
        if (near) {
            if (!exact()) return INFINITY;
            continue;
        }
        if (!(s < INFINITY)) {
            if (s != s) continue;                  // no event
            return INFINITY;                       // not screened
        }
        acc.add(fmaf(w, r.dd, r.d), s, fmaf(w, r.dl, r.l), r.dd, r.dl);
    }
    return acc.bound(sp.cv, bf, lb);
}

// ------------------------------------------------------- the cell kernels
// Both paths fold one (curve, period) item by one or two warps, or by the eight
// warps of a block where its cells are long or the items few: the filters
// (filter.cuh) over all cells, the FP32 screen (exact paths) or the first pass
// (slot path) of the cells they leave, then the evaluation of the few cells
// whose bound reaches the threshold.  The threshold is a lower bound of the
// best ln P: every screened cell gives a lower bound beside its upper bound,
// so no cell has to be evaluated to raise it.
//
// The exact evaluation is FP64 (64 cycles per warp instruction, whatever the
// number of active lanes), and an item leaves one to a few cells: evaluating
// them in place kept the FP64 pipe at 33 % on a sector's fold and at 74 % on
// short curves.  The cells that are left go to a list instead, which k_cand_eval
// evaluates with 32 cells of many items per warp and k_cand_best reduces, one
// thread per item.  An item that has more cells than its queues hold, or finds
// the list full, evaluates in place.
// What the screen needs of one (curve, period) item besides the period table:
// FP64 arithmetic done by k_item_consts for 32 items per warp instruction.
struct ItemConst {
    unsigned long long uend, delta;   // ScreenPeriod
    float cv, hw;
    float K;                          // span / P
    int flags;                        // 1: bad period, 2: screened, 4: slot records,
                                      // 8: cells of 32 or more epochs
};

// The items whose cells have heavy_k or more epochs: a block's eight warps fold
// each of them (their walks are long, and one warp would still be at it when
// the rest of a small grid is done: the first period of the sector grid, 0.2 d,
// ran 5.1 ms in one warp beside 2.6 ms for all others).  The others take one or
// two warps each, blocks of neighbouring periods together: neighbouring periods
// read the same table entries at nearly the same time, which the L1 serves
// (warps that took their items one by one from a counter: 3.8 ms on the
// sector's FP64 fold against 3.4 ms).
struct FoldLists {
    unsigned* block;       // item indices, appended by the preparation kernels
    unsigned* n;           // [0] their number, [1] taken
    float heavy_k;
    unsigned max;          // with more of them the warps keep them (list_max)
};
__device__ __forceinline__ bool list_taken(const FoldLists& l) {
    return l.block && l.n[0] <= l.max;
}
__device__ __forceinline__ void list_item(const FoldLists& l, bool heavy, unsigned o) {
    const int lane = threadIdx.x & 31;
    const unsigned m = __ballot_sync(0xffffffffu, heavy);
    if (!m) return;
    unsigned at = 0u;
    if (lane == __ffs(m) - 1) at = atomicAdd(l.n, (unsigned)__popc(m));
    at = __shfl_sync(0xffffffffu, at, __ffs(m) - 1);
    if (heavy) l.block[at + __popc(m & ((1u << lane) - 1u))] = o;
}

struct FoldJob {
    const FoldSeg* segs;   // the batch's curves, or nullptr: the one curve
    FoldSeg one;
    int n_seg, n_D;
    double dt, inv_dt, gap_max;
    const double* t;
    const void* nodes;
    const ScreenRec* screen;
    const ulonglong2* vpair;
    const ScreenRec* srec;
    const unsigned* reg;
    const unsigned long long* peak;
    const int* bucket;
    const Node4<float>* rec;
    FilterTab tab;
    const double* periods;
    const PeriodConst* ptab;     // nullptr: computed per item
    const SlotPeriod* stab;
    ItemConst* items;            // nullptr: computed by the item
    int64_t n_P;
    double *Q, *T0;
    int* Didx;
    double *dep, *sig, *lnp;
    FoldCand* cand;              // nullptr: evaluate in place
    unsigned long long* n_cand;
    unsigned long long cap;
    int2* range;                 // per item: first candidate, count (-1: written)
    SlotBest* sbest;             // nullptr: the item writes its result
    FoldLists list;              // block == nullptr: none
    unsigned* counters;          // the list's and (behind) the candidates', 32 bytes
};

__device__ __forceinline__ FoldGeom job_geom(const FoldJob& J, const FoldSeg& fs) {
    return FoldGeom{J.t + fs.s_off, fs.n_t0, fs.t_ref, fs.t_last, J.dt, J.inv_dt,
                    J.gap_max, J.bucket + fs.bucket_off, fs.n_bucket};
}
__device__ __forceinline__ ScreenGeom job_screen(const FoldJob& J, const FoldSeg& fs,
                                                 int64_t seg, bool f32) {
    return ScreenGeom{J.screen + fs.s_off * J.n_D, J.vpair + fs.s_off,
                      J.srec ? J.srec + fs.srec_off : nullptr, fs.n_slots, J.reg + 2 * seg,
                      fs.screen, f32 ? 1 : 0};
}
__device__ __forceinline__ ItemConst item_const(const FoldGeom& g, const ScreenGeom& sg, double P,
                                                const PeriodConst& pc) {
    ItemConst ic{0ull, 0ull, 0.f, 0.f, 0.f, 0};
    if (bad_period(P, g)) {
        ic.flags = 1;
        return ic;
    }
    const ScreenPeriod sp = screen_period(g, sg, P, pc);
    ic.uend = sp.uend;
    ic.delta = sp.delta;
    ic.cv = sp.cv;
    ic.hw = sp.hw;
    ic.K = (float)(unsigned)(sp.uend >> 32) / (float)max((unsigned)(sp.ustep >> 32), 1u);
    ic.flags = (sp.on ? 2 : 0) | (sp.slots ? 4 : 0) |
               (g.t_last - g.t_ref >= 32.0 * P ? 8 : 0);
    return ic;
}
__device__ __forceinline__ bool item_heavy(const FoldJob& J, const ItemConst& ic) {
    return J.list.block && (!(ic.K < J.list.heavy_k) || !(ic.flags & 2));
}
// One thread per item: its constants, and its place in the list.
__global__ void k_item_consts(const __grid_constant__ FoldJob J, int f32) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    bool in = i < (int64_t)J.n_seg * J.n_P, heavy = false;
    int64_t o = 0;
    if (in) {
        const int64_t seg = J.n_seg == 1 ? 0 : i / J.n_P;
        const int64_t p = period_slot(i - seg * J.n_P, J.periods, J.n_P);
        o = seg * J.n_P + p;
        const FoldSeg& fs = J.segs ? J.segs[seg] : J.one;
        if (fs.use_slots) {
            in = false;
        } else {
            const ItemConst ic = item_const(job_geom(J, fs), job_screen(J, fs, seg, f32 != 0),
                                            J.periods[p], J.ptab[p]);
            J.items[o] = ic;
            heavy = item_heavy(J, ic);
        }
    }
    if (J.list.block) list_item(J.list, in && heavy, (unsigned)o);
}

// What the screens compare with: an FP32 value below every ln P that an
// evaluated cell could lose by.  In FP64 the bound itself (its margins are far
// above FP64 rounding); in mixed precision the evaluated ln P carries FP32
// rounding (the events', the compensated sums', and up to 2^-21 per epoch
// from the logarithms), so the screens, which bound the real ln P, leave 2e-4
// relative and 5e-7 per epoch.
template <typename T>
__device__ __forceinline__ float screen_threshold(float lb, float K) {
    return sizeof(T) == 8 ? lb : lb - 2e-4f * (1.f + fabsf(lb)) - 5e-7f * K;
}

// Exact evaluation of a cell by one thread (the order of the sums over the
// epochs defines the result).
template <typename T>
__device__ __forceinline__ bool evaluate_cell(const FoldGeom& g, const Node8<T>* __restrict__ nd,
                                              const CellCtx& c, int64_t j, double& lnp, T& Dl,
                                              T& s2) {
    const double phi = cell_phi(c, j);
    const unsigned long long u0 = (unsigned long long)j * c.swp.u0;
    const int64_t kmax = cell_kmax(g, c, phi, u0);
    ExactAcc<T> a1;
    a1.init();
    cell_pass1<T>(g, nd, c, phi, u0, kmax, 0, 1, a1);
    if (a1.K == 0) return false;
    s2 = T(1) / a1.s_inv.s;
    Dl = s2 * a1.s_d.s;
    ExactPen<T> a2;
    a2.init(s2, Dl);
    cell_pass2<T>(g, nd, c, phi, u0, kmax, 0, 1, a2);
    lnp = (double)a1.s_l.s - 0.5 * a2.total();
    return lnp == lnp;                       // NaN never selected
}

// The same by a whole warp (lanes over epochs, fixed reduction order), called
// by all lanes with the same cell: the FP64 evaluation of every cell of a
// period whose cells have 32 or more epochs.
__device__ __forceinline__ bool evaluate_cell_warp(const FoldGeom& g,
                                                   const Node8<double>* __restrict__ nd,
                                                   const CellCtx& c, int64_t j, double& lnp,
                                                   double& Dl, double& s2) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const double phi = cell_phi(c, j);
    const unsigned long long u0 = (unsigned long long)j * c.swp.u0;
    const int64_t kmax = cell_kmax(g, c, phi, u0);
    ExactAcc<double> a1;
    a1.init();
    cell_pass1<double>(g, nd, c, phi, u0, kmax, lane, 32, a1);
    double s_inv = a1.s_inv.s, s_d = a1.s_d.s, s_l = a1.s_l.s;
    int K = a1.K;
    for (int o = 16; o > 0; o >>= 1) {
        s_inv += __shfl_xor_sync(FULL, s_inv, o);
        s_d += __shfl_xor_sync(FULL, s_d, o);
        s_l += __shfl_xor_sync(FULL, s_l, o);
        K += __shfl_xor_sync(FULL, K, o);
    }
    if (K == 0) return false;
    s2 = 1.0 / s_inv;
    Dl = s2 * s_d;
    ExactPen<double> a2;
    a2.init(s2, Dl);
    cell_pass2<double>(g, nd, c, phi, u0, kmax, lane, 32, a2);
    double pen = a2.total();
    for (int o = 16; o > 0; o >>= 1) pen += __shfl_xor_sync(FULL, pen, o);
    lnp = s_l - 0.5 * pen;
    return lnp == lnp;
}

// A large finite single-event gain of each curve, for the peak seed: key[g]
// = (order key of the gain rounded to FP32) << 32 | (2^32 - 1 - e), the
// maximum over the curve's grid entries e (duration-major, e < 2^32 - 1), so
// the largest rounded gain wins and ties go to the first entry.  key[g] must
// be zero on entry and stays zero when no gain is finite.  n_blocks blocks share
// a curve's entries (k_gain_peak: blockIdx.x is the curve of a batch).
template <typename T>
__device__ __forceinline__ void gain_peak(const T* __restrict__ row, int64_t n, unsigned block,
                                          unsigned n_blocks, unsigned long long* __restrict__ key) {
    if (n >= 0xffffffffLL) return;
    unsigned long long best = 0;
    for (int64_t e = block * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)n_blocks * blockDim.x) {
        const double v = (double)row[e];
        if (v > -INFINITY && v < INFINITY) {
            const unsigned long long k = ((unsigned long long)fkey((float)v) << 32) |
                                         (unsigned long long)(0xffffffffu - (unsigned)e);
            best = k > best ? k : best;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long k2 = __shfl_xor_sync(0xffffffffu, best, o);
        best = k2 > best ? k2 : best;
    }
    if ((threadIdx.x & 31) == 0 && best != 0) atomicMax(key, best);
}
template <typename T>
__global__ void k_gain_peak(const T* __restrict__ gain, const int64_t* __restrict__ s_off,
                            int n_D, unsigned long long* __restrict__ key) {
    const int g = blockIdx.x;
    const int64_t s0 = s_off[g];
    gain_peak<T>(gain + s0 * n_D, (s_off[g + 1] - s0) * n_D, blockIdx.y, gridDim.y, key + g);
}

// The tables of one curve's exact path that only read the inputs, in one
// launch: the blocks [end[i-1], end[i]) fill table i.  Six launches of 3 to 15
// us each ran one after the other; together they take the time of the longest
// (the call chain on 2 048 samples, 5 durations, 2 000 periods: 859 -> 837 us).
enum { PREP_BUCKETS, PREP_PEAK, PREP_PERIODS, PREP_OFFSETS, PREP_SLOTS, PREP_NODES, PREP_N };
template <typename T> struct FoldPrep {
    const T *depth, *var, *gain;
    const double* t0s;
    int64_t n_t0;
    int n_D;
    double t_ref, dt, gap_max;
    int64_t n_bucket;
    int* bucket;
    Node8<T>* nodes;
    int64_t n_slots;
    int* slot_of;
    unsigned* reg;
    ScreenRec* srec;
    const double* periods;
    int64_t n_P;
    PeriodConst* ptab;
    unsigned long long* peak;
    unsigned end[PREP_N];
};
// The same on the slot path: blocks [0, b_rec) clear the slot records and L, [b_rec,
// b_peak) find the largest gain, the rest fill the period table.
__global__ void __launch_bounds__(256)
k_slot_prep(Node4<float>* __restrict__ rec, int64_t n_rec, float* __restrict__ L, int64_t n_L,
            unsigned b_rec, const float* __restrict__ gain, int64_t n, unsigned b_peak,
            unsigned long long* __restrict__ peak, const double* __restrict__ periods,
            int64_t n_P, double dt, SlotPeriod* __restrict__ stab) {
    const unsigned b = blockIdx.x;
    if (b < b_rec) {
        const int64_t i = b * (int64_t)blockDim.x + threadIdx.x;
        if (i < n_rec) rec[i] = Node4<float>{NAN, NAN, NAN, 0.f};
        if (i < n_L) L[i] = 0.f;
    } else if (b < b_peak) {
        gain_peak<float>(gain, n, b - b_rec, b_peak - b_rec, peak);
    } else {
        const int64_t i = (b - b_peak) * (int64_t)blockDim.x + threadIdx.x;
        if (i < n_P) stab[i] = slot_period(periods[i], dt);
    }
}
template <typename T>
__global__ void __launch_bounds__(256) k_fold_prep(const __grid_constant__ FoldPrep<T> A) {
    int job = 0;
    unsigned first = 0;
    while (blockIdx.x >= A.end[job]) first = A.end[job++];
    const unsigned block = blockIdx.x - first;
    const int64_t i = block * (int64_t)blockDim.x + threadIdx.x;
    const int64_t ngrid = A.n_t0 * A.n_D;
    switch (job) {
    case PREP_BUCKETS:
        if (i < A.n_bucket) fill_bucket(A.t0s, A.n_t0, A.t_ref, A.dt, i, A.bucket);
        break;
    case PREP_PEAK:
        gain_peak<T>(A.gain, ngrid, block, A.end[job] - first, A.peak);
        break;
    case PREP_PERIODS:
        if (i < A.n_P) fill_period_const(A.periods, i, A.dt, A.ptab);
        break;
    case PREP_OFFSETS:
        if (i < A.n_t0) slot_offset(A.t0s, i, 1.0 / A.dt, A.n_slots, A.slot_of, A.reg);
        break;
    case PREP_SLOTS:
        if (i < A.n_slots * A.n_D) A.srec[i] = no_interval();
        break;
    default:
        if (i < ngrid)
            A.nodes[i] = make_node8<T>(A.depth, A.var, A.gain, A.t0s, i, i % A.n_t0, A.n_t0,
                                       A.gap_max);
    }
}

// The phases about an epoch at walk position u: the cells of one period that
// pass closest to it (the peak seed's).  Lane l < 8 gets phase l - 4 about the
// nearest.
__device__ __forceinline__ unsigned seed_phase(unsigned long long u, unsigned long long ustep,
                                               unsigned long long uph, int64_t n_phi, int l) {
    const unsigned long long r = u % ustep;
    int64_t j = (int64_t)(uph ? (r + (uph >> 1)) / uph : 0ull) + l - 4;
    j = j < 0 ? j + n_phi : (j >= n_phi ? j - n_phi : j);
    return (unsigned)(j < 0 ? 0 : (j >= n_phi ? n_phi - 1 : j));
}

// the warps of an item: one, or the block's
template <int NW>
__device__ __forceinline__ void item_sync() {
    if (NW == 1) __syncwarp(); else __syncthreads();
}
constexpr int FOLD_WARPS = 32;     // resident warps per SM (64 registers)
// Work item i of the job in the order of the fold (short periods first).
__device__ __forceinline__ bool ordered_item(const FoldJob& J, int64_t i, int64_t& item) {
    if (i >= (int64_t)J.n_seg * J.n_P) return false;
    const int64_t seg = J.n_seg == 1 ? 0 : i / J.n_P;
    item = seg * J.n_P + period_slot(i - seg * J.n_P, J.periods, J.n_P);
    return true;
}
// The k-th item of a block of the eight-warp kernels (*sh is the block's);
// false when no work is left.
__device__ __forceinline__ bool next_item(const FoldJob& J, int k_th, unsigned* sh,
                                          int64_t& item) {
    __syncthreads();
    if (J.list.block == nullptr)
        return ordered_item(J, blockIdx.x + (int64_t)k_th * gridDim.x, item);
    if (threadIdx.x == 0) *sh = atomicAdd(J.list.n + 1, 1u);
    __syncthreads();
    const unsigned k = *sh;
    if (k >= J.list.n[0] || !list_taken(J.list)) return false;
    item = J.list.block[k];
    return true;
}
// The item of a warp of the other kernels (blocks of 4 / NW items).
template <int NW>
__device__ __forceinline__ bool warp_item(const FoldJob& J, int64_t& item) {
    return ordered_item(J, NW == 1 ? (int64_t)blockIdx.x * 4 + (threadIdx.x >> 5) : blockIdx.x,
                        item);
}
__host__ __device__ constexpr int fold_threads(int nw) { return nw == 1 ? 128 : 32 * nw; }

// Per-warp shared state of the exact paths: survivors of the screen (their
// cells and bounds).
struct CellQueues {
    FilterQueues f;
    uint2 b[64];
    float bu[64];
    int nb;
};
struct CellItem {          // per-item shared state of the exact paths
    FilterCtx x;
    ScreenPeriod sp;
    CellCtx cc;
    FoldGeom g;
    ScreenGeom sg;
    int64_t item;
    int coop;              // cells evaluated by the warp's lanes
    int inl;               // some cell was evaluated in place
    unsigned cnt;
    long long start;
};

// The screen of the exact paths (filter.cuh) and what follows it.
template <typename T, bool LONE>
struct CellScreen {
    static constexpr bool lone = LONE;
    CellItem& it;
    CellQueues& q;
    const Node8<T>* nodes;
    Best& tb;              // the warp's best cell evaluated in place (shared)

    // drop the survivors that the threshold has overtaken
    __device__ __noinline__ void compact() {
        const int lane = threadIdx.x & 31;
        const float t = filter_thr(it.x);
        const int nb = q.nb;
        int n = 0;
        for (int h = 0; h < nb; h += 32) {
            const bool in = h + lane < nb;
            const uint2 cl = in ? q.b[h + lane] : make_uint2(0u, 0u);
            const float ub = in ? q.bu[h + lane] : 0.f;
            const bool keep = in && !(ub < t);
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            if (keep) {
                const int pos = n + __popc(m & ((1u << lane) - 1u));
                q.b[pos] = cl;
                q.bu[pos] = ub;
            }
            n += __popc(m);
            __syncwarp();
        }
        if (lane == 0) q.nb = n;
        __syncwarp();
    }

    // evaluation in place of the first n <= 32 survivors
    __device__ __noinline__ void evaluate(int n) {
        const unsigned FULL = 0xffffffffu;
        const int lane = threadIdx.x & 31;
        const FoldGeom& g = it.g;
        const CellCtx& c = it.cc;
        const int64_t n_phi = it.x.fp.n_phi;
        Best best{-INFINITY, LLONG_MAX, NAN, NAN};
        auto take = [&](const uint2& cl, double lnp, double Dl, double s2) {
            const Best cand{lnp, (long long)cl.y * n_phi + cl.x, Dl, s2};
            if (better(cand, best)) best = cand;
        };
        bool done = false;
        if constexpr (sizeof(T) == 8) {
            if (it.coop) {
                for (int e = 0; e < n; ++e) {
                    const uint2 cl = q.b[e];
                    double lnp, Dl, s2;
                    if (evaluate_cell_warp(g, nodes + (int64_t)cl.y * g.n_t0, c, cl.x, lnp, Dl,
                                           s2))
                        take(cl, lnp, Dl, s2);
                }
                done = true;
            }
        }
        if (!done && lane < n) {
            const uint2 cl = q.b[lane];
            double lnp;
            T Dl, s2;
            if (evaluate_cell<T>(g, nodes + (int64_t)cl.y * g.n_t0, c, cl.x, lnp, Dl, s2))
                take(cl, lnp, (double)Dl, (double)s2);
        }
        for (int s = 16; s > 0; s >>= 1) {
            const Best b{__shfl_xor_sync(FULL, best.lnp, s), __shfl_xor_sync(FULL, best.cell, s),
                         __shfl_xor_sync(FULL, best.depth, s),
                         __shfl_xor_sync(FULL, best.sigma, s)};
            if (better(b, best)) best = b;
        }
        if (lane == 0) {
            it.inl = 1;
            if (better(best, tb)) tb = best;
            if (best.cell != LLONG_MAX)
                filter_raise(it.x, fkey(screen_threshold<T>(__double2float_rd(best.lnp),
                                                            it.x.fp.K)));
        }
        __syncwarp();
    }

    __device__ __noinline__ void push(bool keep, const uint2& cl, float ub) {
        const int lane = threadIdx.x & 31;
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        const int nb = q.nb;
        if (keep) {
            const int pos = nb + __popc(m & ((1u << lane) - 1u));
            q.b[pos] = cl;
            q.bu[pos] = ub;
        }
        __syncwarp();
        if (lane == 0) q.nb = nb + __popc(m);
        __syncwarp();
        if (q.nb < 32) return;
        compact();
        const int n = q.nb;
        if (n < 32) return;
        evaluate(32);
        const float u2 = lane < n - 32 ? q.bu[32 + lane] : 0.f;
        filter_shift_queue(q.b, n, 32);
        if (lane < n - 32) q.bu[lane] = u2;
        if (lane == 0) q.nb = n - 32;
        __syncwarp();
    }

    // full screen of the queue's first cnt cells
    __device__ __noinline__ void operator()(int cnt) {
        const int lane = threadIdx.x & 31;
        float ub = -INFINITY, lb = -INFINITY;
        uint2 cl = make_uint2(0u, 0u);
        const ScreenGeom& sg = it.sg;
        if (lane < cnt) {
            cl = q.f.cell[lane];
            ub = screen_cell(it.g, sg, sg.rec + (int64_t)cl.y * it.g.n_t0,
                             sg.srec ? sg.srec + (int64_t)cl.y * sg.n_slots : nullptr, it.sp,
                             it.cc, (int64_t)cl.x, (unsigned long long)cl.x * it.sp.uph,
                             filter_thr(it.x), &lb);
        }
        const unsigned k =
            __reduce_max_sync(0xffffffffu, fkey(screen_threshold<T>(lb, it.x.fp.K)));
        if (lane == 0) filter_raise(it.x, k);
        __syncwarp();
        // a cell without events (bound -inf) is never the argmax; NaN survives
        push(lane < cnt && !(ub == -INFINITY) && !(ub < filter_thr(it.x)), cl, ub);
    }
};

// Shared state of an item, by one warp (an invalid period is written here).
__device__ __noinline__ void cell_item_setup(const FoldJob& J, const FoldSeg& fs, int64_t seg,
                                             int64_t p, int64_t o, bool f32, int nw,
                                             CellItem& it) {
    if ((threadIdx.x & 31) != 0) return;
    const double P = J.periods[p];
    const FoldGeom g = job_geom(J, fs);
    const ScreenGeom sg = job_screen(J, fs, seg, f32);
    PeriodConst tmp;
    const PeriodConst* pc = J.ptab ? J.ptab + p : &tmp;
    ItemConst ic;
    if (J.items) {
        ic = J.items[o];
    } else {
        tmp = bad_period(P, g) ? PeriodConst{1, 0.0, 0, 0, 0.f, {0, 0}, {0, 0}, 1.0, 1.0}
                               : period_const(P, J.dt, J.inv_dt);
        ic = item_const(g, sg, P, *pc);
    }
    it.item = o;
    if (ic.flags & 1) {
        write_bad(o, J.Q, J.T0, J.Didx, J.dep, J.sig, J.lnp);
        if (J.range) J.range[o] = make_int2(0, -1);
        it.item = -1;
        return;
    }
    it.g = g;
    it.sg = sg;
    it.cc = cell_ctx(g, P, *pc, fs.uspan);
    const bool on = ic.flags & 2;
    ScreenPeriod& sp = it.sp;
    sp.uph = on ? pc->uph : 0ull;
    sp.ustep = on ? pc->ustep : 0ull;
    sp.delta = ic.delta;
    sp.uend = ic.uend;
    sp.wscale = (float)(4194304.0 * J.inv_dt);
    sp.cv = ic.cv;
    sp.hw = ic.hw;
    sp.on = on;
    sp.slots = ic.flags & 4;
    FilterPeriod f;
    f.ustep = sp.ustep;
    f.uph = sp.uph;
    f.uend = sp.uend;
    f.n_phi = pc->n_phi;
    f.K = ic.K + 2.f;
    f.mode = on && sp.delta <= 8ull * FILTER_MARGIN
                 ? filter_mode(J.tab, sp.ustep, ic.K, f.n_phi * J.n_D, nw, sp.slots)
                 : FILTER_NONE;
    it.x.fp = f;
    it.x.f = filter_view(J.tab, fs);
    it.x.n_D = J.n_D;
    it.x.bfk = fkey(-INFINITY);
    // FP64 sums of long cells by the warp's lanes (one fixed order for every
    // cell of the period)
    it.coop = !f32 && on && (ic.flags & 8);
    it.inl = 0;
    it.cnt = 0u;
}

// One item of the exact paths by the nw warps that share it (w: this one).
template <typename T, int nw, bool LONE>
__device__ __forceinline__ void fold_cells_item(const FoldJob& J, int64_t o, int w, CellItem& it,
                                                CellQueues& q, Best* tbs) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t seg = J.n_seg == 1 ? 0 : o / J.n_P;
    const int64_t p = o - seg * J.n_P;
    const FoldSeg& fs = J.segs ? J.segs[seg] : J.one;
    if (fs.use_slots) return;
    if (nw < 8 && J.items && item_heavy(J, J.items[o]) && list_taken(J.list)) return;
    const int n_D = J.n_D;
    if (lane == 0) {
        q.f.ni = q.f.nq = q.f.nc = q.nb = 0;
        tbs[w] = Best{-INFINITY, LLONG_MAX, NAN, NAN};
    }
    if (w == 0) cell_item_setup(J, fs, seg, p, o, sizeof(T) == 4, nw, it);
    item_sync<nw>();
    if (it.item < 0) return;
    CellScreen<T, LONE> screen{it, q, (const Node8<T>*)J.nodes + fs.s_off * n_D, tbs[w]};
    if (it.x.fp.mode != FILTER_NONE) {
        // peak seed: the cells about the curve's largest single-event gain
        const unsigned long long pk = J.peak[seg];
        if (pk != 0 && w == 0) {
            const unsigned e = 0xffffffffu - (unsigned)(pk & 0xffffffffu);
            const unsigned pd = e / (unsigned)fs.n_t0;
            const unsigned long long u = it.sg.vpair[e - pd * (unsigned)fs.n_t0].x;
            if (lane < 8)
                q.f.cell[lane] = make_uint2(
                    seed_phase(u, it.x.fp.ustep, it.x.fp.uph, it.x.fp.n_phi, lane), pd);
            __syncwarp();
            screen(8);
            __syncwarp();
        }
        item_sync<nw>();
        filter_cells(it.x, w, nw, q.f, screen);
    } else {
        // every cell: to the screen, or (no screen) to the evaluation
        const int64_t n_phi = it.x.fp.n_phi, n_cells = n_phi * n_D;
        for (int64_t base = (int64_t)w * 32; base < n_cells; base += nw * 32) {
            const int64_t cell = base + lane;
            const bool in = cell < n_cells;
            const unsigned d = in ? (unsigned)(cell / n_phi) : 0u;
            const uint2 cl = make_uint2(in ? (unsigned)(cell - (int64_t)d * n_phi) : 0u, d);
            if (it.sp.on) {
                q.f.cell[lane] = cl;
                __syncwarp();
                screen((int)min((int64_t)32, n_cells - base));
                __syncwarp();
            } else {
                screen.push(in, cl, INFINITY);
            }
        }
    }
    item_sync<nw>();
    screen.compact();
    const int nb = q.nb;
    // hand the survivors on, unless some were evaluated here or the list is full
    if (J.cand != nullptr && it.inl == 0) {
        unsigned at = 0u;
        if (lane == 0) at = atomicAdd(&it.cnt, (unsigned)nb);
        item_sync<nw>();
        if (w == 0 && lane == 0) {
            const unsigned n = it.cnt;
            long long start = n ? (long long)atomicAdd(J.n_cand, (unsigned long long)n) : 0;
            if (n && (unsigned long long)start + n > J.cap) {
                for (unsigned long long i = start; i < J.cap && i < start + n; ++i)
                    J.cand[i].item = -1;
                start = -1;
            } else {
                J.range[o] = make_int2((int)start, (int)n);
            }
            it.start = start;
        }
        item_sync<nw>();
        if (it.start >= 0) {
            at = __shfl_sync(FULL, at, 0);
            if (lane < nb) {
                FoldCand& cd = J.cand[it.start + at + lane];
                cd.item = o;
                cd.j = q.b[lane].x;
                cd.d = (int)q.b[lane].y;
            }
            return;
        }
    }
    if (nb > 0) screen.evaluate(nb);
    item_sync<nw>();
    if (w == 0 && lane == 0) {
        Best tb = tbs[0];
        for (int i = 1; i < nw; ++i)
            if (better(tbs[i], tb)) tb = tbs[i];
        if (tb.cell != LLONG_MAX) tb.sigma = sqrt(tb.sigma);   // held sigma^2
        write_best(tb, o, it.x.fp.n_phi, it.g.t_ref, J.periods[p], J.Q, J.T0, J.Didx, J.dep,
                   J.sig, J.lnp);
        if (J.range) J.range[o] = make_int2(0, -1);
    }
}

// Exact paths (FP64 epochs; T: the type of the events).
template <typename T, int NW, bool LONE>
__global__ void __launch_bounds__(fold_threads(NW), FOLD_WARPS * 32 / fold_threads(NW))
k_fold_cells(const __grid_constant__ FoldJob J) {
    constexpr int W = fold_threads(NW) / 32;
    __shared__ CellQueues sh_q[W];
    __shared__ CellItem sh_i[W / NW];
    __shared__ Best sh_tb[W];
    const int wid = threadIdx.x >> 5;
    int64_t item = 0;
    if (NW == 8) {
        __shared__ unsigned sh_k;
        for (int k = 0; next_item(J, k, &sh_k, item); ++k)
            fold_cells_item<T, NW, LONE>(J, item, wid, sh_i[0], sh_q[wid], sh_tb);
    } else if (warp_item<NW>(J, item)) {
        fold_cells_item<T, NW, LONE>(J, item, wid % NW, sh_i[wid / NW], sh_q[wid],
                                     sh_tb + wid / NW * NW);
    }
}

// Exact evaluation of the listed cells, one per lane (or one per warp, see
// evaluate_cell_warp).
template <typename T>
__global__ void __launch_bounds__(64) k_cand_eval(const __grid_constant__ FoldJob J) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const unsigned long long n = min(*J.n_cand, J.cap);
    const unsigned long long groups = (n + 31) / 32;
    const unsigned long long n_warps = (unsigned long long)gridDim.x * blockDim.x / 32;
    const unsigned long long w0 =
        (blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x) / 32;
    // whether a candidate is one for a whole warp
    auto is_long = [&](const FoldCand& cd) {
        if (cd.item < 0) return false;
        const int64_t seg = J.n_seg == 1 ? 0 : cd.item / J.n_P;
        const double P = J.periods[cd.item - seg * J.n_P];
        const FoldSeg& fs = J.segs ? J.segs[seg] : J.one;
        return fs.t_last - fs.t_ref >= 32.0 * P;
    };
    for (unsigned long long w = w0; w < groups; w += n_warps) {
        const unsigned long long i = 32 * w + lane;
        if (i < n && J.cand[i].item >= 0) {
            FoldCand& cd = J.cand[i];
            const int64_t seg = J.n_seg == 1 ? 0 : cd.item / J.n_P;
            const int64_t p = cd.item - seg * J.n_P;
            if (sizeof(T) == 4 || !is_long(cd)) {
                const FoldSeg& fs = J.segs ? J.segs[seg] : J.one;
                const FoldGeom g = job_geom(J, fs);
                const CellCtx c = cell_ctx(g, J.periods[p], J.ptab[p], fs.uspan);
                const Node8<T>* nd =
                    (const Node8<T>*)J.nodes + fs.s_off * J.n_D + (int64_t)cd.d * g.n_t0;
                T D, s;
                double lnp;
                const bool ok = evaluate_cell<T>(g, nd, c, (int64_t)cd.j, lnp, D, s);
                cd.lnp = ok ? lnp : NAN;
                cd.Dl = (double)D;
                cd.s2 = (double)s;
            }
        }
        __syncwarp();
        // The long cells, lanes over epochs, one after the other.  They come in
        // runs (one item's, its neighbours'), so a warp takes every
        // groups-th candidate here: 32 of a run in one warp were most of the
        // kernel's 440 us on the sector fold (whole call 3.21 -> 2.93 ms).
        if constexpr (sizeof(T) == 8) {
            const unsigned long long k = w + lane * groups;
            const bool mine = k < n && is_long(J.cand[k]);
            for (unsigned m = __ballot_sync(FULL, mine); m; m &= m - 1u) {
                FoldCand& cd = J.cand[w + (__ffs(m) - 1) * groups];
                const int64_t seg = J.n_seg == 1 ? 0 : cd.item / J.n_P;
                const int64_t p = cd.item - seg * J.n_P;
                const FoldSeg& fs = J.segs ? J.segs[seg] : J.one;
                const FoldGeom g = job_geom(J, fs);
                const CellCtx c = cell_ctx(g, J.periods[p], J.ptab[p], fs.uspan);
                double l, D, s;
                const bool ok = evaluate_cell_warp(
                    g, (const Node8<double>*)J.nodes + fs.s_off * J.n_D + (int64_t)cd.d * g.n_t0,
                    c, (int64_t)cd.j, l, D, s);
                if (lane == 0) {
                    cd.lnp = ok ? l : NAN;
                    cd.Dl = D;
                    cd.s2 = s;
                }
            }
        }
    }
}
__global__ void k_cand_best(const __grid_constant__ FoldJob J) {
    const int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (o >= (int64_t)J.n_seg * J.n_P) return;
    const int64_t seg = J.n_seg == 1 ? 0 : o / J.n_P;
    const FoldSeg& fs = J.segs ? J.segs[seg] : J.one;
    const double P = J.periods[o - seg * J.n_P];
    if (fs.use_slots) return;
    const int2 r = J.range[o];
    if (r.y < 0) return;
    const int64_t n_phi = J.ptab[o - seg * J.n_P].n_phi;
    Best b{-INFINITY, LLONG_MAX, NAN, NAN};
    for (int i = 0; i < r.y; ++i) {
        const FoldCand& cd = J.cand[(unsigned)r.x + i];
        const double lnp = cd.lnp;
        if (!(lnp == lnp)) continue;
        const Best x{lnp, (long long)cd.d * n_phi + cd.j, cd.Dl, cd.s2};
        if (better(x, b)) b = x;
    }
    if (b.cell != LLONG_MAX) b.sigma = sqrt(b.sigma);
    write_best(b, o, n_phi, fs.t_ref, P, J.Q, J.T0, J.Didx, J.dep, J.sig, J.lnp);
}

// ---------------------------------------- slot path (mixed, regular grids)
struct SlotEvent {
    float d, s, l;
};
__device__ __forceinline__ SlotEvent slot_event(const Node4<float>* __restrict__ rd,
                                                unsigned long long u) {
    const int64_t s = (int64_t)(u >> 40);
    // weight = fractional slot position: its top 23 bits as the mantissa of a
    // float in [1, 2), minus 1 (no integer-to-float conversion)
    const float w =
        __uint_as_float(0x3f800000u | (unsigned)((u >> 17) & 0x7fffffu)) - 1.0f;
    const Node4<float> a = rd[s];
    const Node4<float> b = rd[s + 1];
    SlotEvent e;
    e.s = __fmaf_rn(w, b.s - a.s, a.s);
    e.d = __fmaf_rn(w, b.d - a.d, a.d);
    e.l = __fmaf_rn(w, b.l - a.l, a.l);
    return e;
}

struct SlotPass1 {
    KSum<float> s_inv, s_d, s_l;
    float s_dd;            // sum Delta_k^2 / s_k^2 (bound only)
    float ivmax, ivmin;    // max and min 1/s_k^2 (bounds only)
    int K;
    __device__ __forceinline__ void init() {
        s_inv.init();
        s_d.init();
        s_l.init();
        s_dd = 0.f;
        ivmax = 0.f;
        ivmin = INFINITY;
        K = 0;
    }
    // The bounds of ScreenAcc::bound on the sums; x_max, x_min = max and min
    // 1/s_k^2 over S_inv.  The reciprocals are the hardware approximation
    // (2^-21 relative, far inside the margins).
    __device__ __forceinline__ float upper() const {
        const float r = rcp32(s_inv.s);
        const float q = fmaxf(0.0f, s_dd - s_d.s * s_d.s * r - 1e-4f * s_dd);
        const float x = fminf(1.0f, ivmax * r * 1.001f);
        return s_l.s + 0.5f - 0.5f * q * rcp32(1.0f + x) * 0.9999f;
    }
    __device__ __forceinline__ float lower() const {
        const float r = rcp32(s_inv.s);
        const float q = fmaxf(0.0f, s_dd - s_d.s * s_d.s * r + 1e-4f * s_dd);
        const float xh = fminf(1.0f, ivmax * r * 1.001f), xl = ivmin * r * 0.999f;
        const float lb = s_l.s + 0.34657f * lg2_32(1.0f + xh) * rcp32(xh) -
                         0.5f * q * rcp32(1.0f + xl) * 1.0001f - 1e-4f;
        return lb == lb ? lb : -INFINITY;
    }
    __device__ __forceinline__ void add(const SlotEvent& e) {
        if (isnan(e.s)) return;
        const float iv = rcp32(__fmul_rn(e.s, e.s));
        const float div = __fmul_rn(e.d, iv);
        s_inv.add(iv);
        s_d.add(div);
        s_dd = fmaf(div, e.d, s_dd);
        ivmax = fmaxf(ivmax, iv);
        ivmin = fminf(ivmin, iv);
        s_l.add(e.l);
        ++K;
    }
};

struct SlotPass2 {
    KSum<float> quad;
    float lsum;
    float s2, Dl;
    __device__ __forceinline__ void init(float s2_, float Dl_) {
        quad.init();
        lsum = 0.f;
        s2 = s2_;
        Dl = Dl_;
    }
    __device__ __forceinline__ void add(float dk, float sg) {
        if (isnan(sg)) return;
        const float sk2 = __fmul_rn(sg, sg);
        const float iden = rcp32(__fadd_rn(sk2, s2));
        const float r = dk - Dl;
        quad.add_prod(__fmul_rn(r, r), iden);
        lsum += lg2_32(__fmul_rn(sk2, iden));
    }
};

__device__ __forceinline__ void write_slot_best(const SlotBest& sb, int64_t o, int64_t n_phi,
                                                double t_ref, double P, const FoldJob& J) {
    Best b{-INFINITY, LLONG_MAX, NAN, NAN};
    if (sb.d >= 0)
        b = Best{(double)sb.lnp, (long long)sb.d * n_phi + sb.j, (double)sb.Dl,
                 sqrt((double)sb.s2)};
    write_best(b, o, n_phi, t_ref, P, J.Q, J.T0, J.Didx, J.dep, J.sig, J.lnp);
}

// A cell of the slot path that passed the bound, queued for its second pass.
struct SCell {
    unsigned long long u0;
    unsigned j;
    int d, kmax;
    float s_l, s2, Dl, ub;
};

// Epochs walk the slot grid in 24.40 fixed point: u = (T - t_ref)/dt =
// (j/n_phi + k) P/dt.  The interval is (slot, slot+1) and the weight is the
// fractional part; on a grid whose epochs sit on the slots this is the
// interpolation between the bracketing epochs up to their offsets from the
// slot centres (checked to be below 1e-3 slot).
//
// Per item: the filters, whose tables hold the events of this walk; the first
// pass (FP32 compensated sums) of the cells they leave, with the bounds of
// SlotPass1, the lower one raising the threshold; and the second
// pass of the cells whose bound still reaches it, at the end or when 32 are
// queued.
struct SlotItem {
    FilterCtx x;
    int bad;
    SlotBest wb[8];
};
struct SlotQueues {
    FilterQueues f;
    SCell c[64];
    int n;
    float bl[32], bD[32], bs2[32];     // each lane's best cell
    unsigned bj[32];
    int bd[32];                        // -1: none
};

template <bool LONE>
struct SlotScreen {
    static constexpr bool lone = LONE;
    SlotItem& it;
    SlotQueues& q;
    const Node4<float>* rec;
    int64_t n_slots;
    unsigned long long ulast;

    // second pass of queued cell e, by one lane
    __device__ __forceinline__ void pass2(const SCell& e) {
        if (e.ub + 1e-4f * fmaxf(1.f, fabsf(e.ub)) < filter_thr(it.x)) return;   // overtaken
        const int lane = threadIdx.x & 31;
        const unsigned long long ustep = it.x.fp.ustep;
        const Node4<float>* rd = rec + (int64_t)e.d * n_slots;
        SlotPass2 p2;
        p2.init(e.s2, e.Dl);
        unsigned long long u = e.u0;
        for (int k = 0; k < e.kmax; ++k, u += ustep) {
            const SlotEvent ev = slot_event(rd, u);
            p2.add(ev.d, ev.s);
        }
        const float lnp = e.s_l - 0.5f * __fmaf_rn(p2.lsum, 0.693147180559945f, p2.quad.s);
        if (!(lnp == lnp)) return;
        const int bd = q.bd[lane];
        const float bl = q.bl[lane];
        if (bd < 0 || lnp > bl ||
            (lnp == bl && (e.d < bd || (e.d == bd && e.j < q.bj[lane])))) {
            q.bl[lane] = lnp;
            q.bD[lane] = p2.Dl;
            q.bs2[lane] = p2.s2;
            q.bj[lane] = e.j;
            q.bd[lane] = e.d;
        }
        filter_raise(it.x, fkey(screen_threshold<float>(lnp, it.x.fp.K)));
    }
    __device__ __forceinline__ void flush(int cnt) {
        const int lane = threadIdx.x & 31;
        if (lane < cnt) pass2(q.c[lane]);
        __syncwarp();
    }

    // first pass and bounds of the queue's first cnt cells
    __device__ __noinline__ void operator()(int cnt) {
        const unsigned FULL = 0xffffffffu;
        const int lane = threadIdx.x & 31;
        const unsigned long long ustep = it.x.fp.ustep;
        SCell e;
        bool keep = false;
        float lb = -INFINITY;
        if (lane < cnt) {
            const uint2 cl = q.f.cell[lane];
            const unsigned long long u0 = (unsigned long long)cl.x * it.x.fp.uph;
            const Node4<float>* rd = rec + (int64_t)cl.y * n_slots;
            SlotPass1 p1;
            p1.init();
            int kmax = 0;
            // two epochs' record loads in flight
#pragma unroll 2
            for (unsigned long long u = u0; u <= ulast; u += ustep, ++kmax)
                p1.add(slot_event(rd, u));
            if (p1.K > 0) {
                lb = p1.lower();
                e.ub = p1.upper();
                keep = !(e.ub + 1e-4f * fmaxf(1.f, fabsf(e.ub)) < filter_thr(it.x));
                e.s2 = 1.0f / p1.s_inv.s;
                e.Dl = e.s2 * p1.s_d.s;
                e.s_l = p1.s_l.s;
                e.u0 = u0;
                e.j = cl.x;
                e.d = (int)cl.y;
                e.kmax = kmax;
            }
        }
        const unsigned k = __reduce_max_sync(FULL, fkey(screen_threshold<float>(lb, it.x.fp.K)));
        if (lane == 0) filter_raise(it.x, k);
        const unsigned m = __ballot_sync(FULL, keep);
        int n = q.n;
        if (keep) q.c[n + __popc(m & ((1u << lane) - 1u))] = e;
        n += __popc(m);
        __syncwarp();
        if (n >= 32) {
            flush(32);
            n -= 32;
            SCell e2;
            if (lane < n) e2 = q.c[32 + lane];
            __syncwarp();
            if (lane < n) q.c[lane] = e2;
            __syncwarp();
        }
        if (lane == 0) q.n = n;
        __syncwarp();
    }
};

__device__ __forceinline__ float slot_K(const FoldSeg& fs, const SlotPeriod& sp) {
    return (float)(unsigned)(fs.ulast >> 32) / (float)max((unsigned)(sp.ustep >> 32), 1u);
}
// The slot path's list, as k_item_consts.
__global__ void k_slot_items(const __grid_constant__ FoldJob J) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    bool in = i < (int64_t)J.n_seg * J.n_P, heavy = false;
    int64_t o = 0;
    if (in) {
        const int64_t seg = J.n_seg == 1 ? 0 : i / J.n_P;
        const int64_t p = period_slot(i - seg * J.n_P, J.periods, J.n_P);
        o = seg * J.n_P + p;
        const FoldSeg& fs = J.segs ? J.segs[seg] : J.one;
        if (!fs.use_slots) {
            in = false;
        } else {
            heavy = !(slot_K(fs, J.stab[p]) < J.list.heavy_k);
        }
    }
    list_item(J.list, in && heavy, (unsigned)o);
}

// One item of the slot path by the nw warps that share it.
template <int nw, bool LONE>
__device__ __forceinline__ void fold_slots_item(const FoldJob& J, int64_t o, int w, SlotItem& it,
                                                SlotQueues& q) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int64_t seg = J.n_seg == 1 ? 0 : o / J.n_P;
    const int64_t p = o - seg * J.n_P;
    const FoldSeg& fs = J.segs ? J.segs[seg] : J.one;
    if (!fs.use_slots) return;
    if (nw < 8 && list_taken(J.list) && !(slot_K(fs, J.stab[p]) < J.list.heavy_k)) return;
    const int n_D = J.n_D;
    if (lane == 0) q.f.ni = q.f.nq = q.f.nc = q.n = 0;
    q.bd[lane] = -1;
    q.bl[lane] = -INFINITY;
    if (w == 0 && lane == 0) {
        const double P = J.periods[p];
        const SlotPeriod sp = J.stab ? J.stab[p] : slot_period(P, J.dt);
        it.bad = sp.bad || fs.t_last - fs.t_ref > 1.0e9 * P;
        FilterPeriod f;
        f.ustep = sp.ustep;
        f.uph = sp.uph;
        f.uend = fs.ulast + 1ull;
        f.n_phi = sp.n_phi;
        const float K = slot_K(fs, sp);
        f.K = K + 2.f;
        f.mode = filter_mode(J.tab, sp.ustep, K, f.n_phi * n_D, nw, true);
        it.x.fp = f;
        it.x.f = filter_view(J.tab, fs);
        it.x.n_D = n_D;
        it.x.bfk = fkey(-INFINITY);
    }
    item_sync<nw>();
    if (it.bad) {
        if (w == 0 && lane == 0) {
            write_bad(o, J.Q, J.T0, J.Didx, J.dep, J.sig, J.lnp);
            if (J.sbest) J.sbest[o].d = -2;
        }
        return;
    }
    SlotScreen<LONE> screen{it, q, J.rec + fs.rec_off, fs.n_slots, fs.ulast};
    if (it.x.fp.mode != FILTER_NONE) {
        const unsigned long long pk = J.peak[seg];
        if (pk != 0 && w == 0) {
            const unsigned e = 0xffffffffu - (unsigned)(pk & 0xffffffffu);
            const unsigned pd = e / (unsigned)fs.n_t0;
            const double x = (J.t[fs.s_off + (e - pd * (unsigned)fs.n_t0)] - fs.t_ref) * J.inv_dt;
            const unsigned long long u = (unsigned long long)llrint(fmax(x, 0.0)) << 40;
            if (lane < 8)
                q.f.cell[lane] = make_uint2(
                    seed_phase(u, it.x.fp.ustep, it.x.fp.uph, it.x.fp.n_phi, lane), pd);
            __syncwarp();
            screen(8);
            __syncwarp();
        }
        item_sync<nw>();
        filter_cells(it.x, w, nw, q.f, screen);
    } else {
        const int64_t n_phi = it.x.fp.n_phi, n_cells = n_phi * n_D;
        for (int64_t base = (int64_t)w * 32; base < n_cells; base += nw * 32) {
            const int64_t cell = min(base + lane, n_cells - 1);
            const unsigned d = (unsigned)(cell / n_phi);
            q.f.cell[lane] = make_uint2((unsigned)(cell - (int64_t)d * n_phi), d);
            __syncwarp();
            screen((int)min((int64_t)32, n_cells - base));
            __syncwarp();
        }
    }
    item_sync<nw>();
    screen.flush(q.n);
    // argmax in FP32 (larger ln P, ties to the smaller cell): the largest ln P,
    // then the smallest duration and phase among its lanes
    auto over = [](const SlotBest& a, const SlotBest& b) {   // a beats b
        if (a.d < 0) return false;
        if (b.d < 0 || a.lnp > b.lnp) return true;
        return a.lnp == b.lnp && (a.d < b.d || (a.d == b.d && a.j < b.j));
    };
    __syncwarp();
    const int bd = q.bd[lane];
    const unsigned key = bd >= 0 ? fkey(q.bl[lane] + 0.f) : 0u;   // (-0 ties with 0)
    const unsigned top = __reduce_max_sync(FULL, key);
    const bool lead = bd >= 0 && key == top;
    const unsigned d0 = __reduce_min_sync(FULL, lead ? (unsigned)bd : ~0u);
    const bool lead_d = lead && (unsigned)bd == d0;
    const unsigned j0 = __reduce_min_sync(FULL, lead_d ? q.bj[lane] : ~0u);
    const unsigned m = __ballot_sync(FULL, lead_d && q.bj[lane] == j0);
    SlotBest sb{-INFINITY, NAN, NAN, 0u, -1};
    if (m) {
        const int l = __ffs(m) - 1;
        sb = SlotBest{q.bl[l], q.bD[l], q.bs2[l], q.bj[l], q.bd[l]};
    }
    if (nw > 1) {
        if (lane == 0) it.wb[w] = sb;
        __syncthreads();
        if (w == 0 && lane == 0)
            for (int i = 1; i < nw; ++i)
                if (over(it.wb[i], sb)) sb = it.wb[i];
    }
    if (w == 0 && lane == 0) {
        if (J.sbest)
            J.sbest[o] = sb;                  // k_slot_best writes the outputs
        else
            write_slot_best(sb, o, it.x.fp.n_phi, fs.t_ref, J.periods[p], J);
    }
}

template <int NW, bool LONE>
__global__ void __launch_bounds__(fold_threads(NW), FOLD_WARPS * 32 / fold_threads(NW))
k_fold_slot_cells(const __grid_constant__ FoldJob J) {
    constexpr int W = fold_threads(NW) / 32;
    __shared__ SlotQueues sh_q[W];
    __shared__ SlotItem sh_i[W / NW];
    const int wid = threadIdx.x >> 5;
    int64_t item = 0;
    if (NW == 8) {
        __shared__ unsigned sh_k;
        for (int k = 0; next_item(J, k, &sh_k, item); ++k)
            fold_slots_item<NW, LONE>(J, item, wid, sh_i[0], sh_q[wid]);
    } else if (warp_item<NW>(J, item)) {
        fold_slots_item<NW, LONE>(J, item, wid % NW, sh_i[wid / NW], sh_q[wid]);
    }
}

// Outputs of the slot path, one thread per item: the FP64 divisions and roots
// of 32 items in one warp instruction.
__global__ void k_slot_best(const __grid_constant__ FoldJob J) {
    const int64_t o = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (o >= (int64_t)J.n_seg * J.n_P) return;
    const int64_t seg = J.n_seg == 1 ? 0 : o / J.n_P;
    const FoldSeg& fs = J.segs ? J.segs[seg] : J.one;
    if (!fs.use_slots) return;
    const SlotBest sb = J.sbest[o];
    if (sb.d == -2) return;
    const int64_t p = o - seg * J.n_P;
    write_slot_best(sb, o, J.stab[p].n_phi, fs.t_ref, J.periods[p], J);
}

// ------------------------------------------------------------ batch path

// Per-curve node records (exact path) and bucket tables; slot tables.
template <typename T>
__global__ void k_nodes_batch(const T* __restrict__ depth, const T* __restrict__ var,
                              const T* __restrict__ gain, const double* __restrict__ t,
                              const FoldSeg* __restrict__ segs, int n_seg,
                              const int64_t* __restrict__ s_off, int n_D, double gap_max,
                              Node8<T>* __restrict__ nodes) {
    const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (gid >= s_off[n_seg] * (int64_t)n_D) return;
    int lo = 0, hi = n_seg;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (s_off[mid] * (int64_t)n_D <= gid) lo = mid; else hi = mid;
    }
    const int64_t s0 = s_off[lo], ng = s_off[lo + 1] - s0;
    const int64_t i = (gid - s0 * n_D) % ng;
    nodes[gid] = make_node8<T>(depth, var, gain, t + s0, gid, i, ng, gap_max);
}

template <typename T>
__global__ void k_screen_batch(const T* __restrict__ depth, const T* __restrict__ var,
                               const T* __restrict__ gain, const double* __restrict__ t,
                               const FoldSeg* __restrict__ segs, int n_seg,
                               const int64_t* __restrict__ s_off, int n_D, double gap_max,
                               double dt, ScreenRec* __restrict__ rec,
                               ulonglong2* __restrict__ vpair, ScreenRec* __restrict__ srec,
                               const int* __restrict__ slot_of) {
    const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (gid >= s_off[n_seg] * (int64_t)n_D) return;
    int lo = 0, hi = n_seg;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (s_off[mid] * (int64_t)n_D <= gid) lo = mid; else hi = mid;
    }
    const FoldSeg fs = segs[lo];
    if (!fs.screen) return;
    const int64_t s0 = s_off[lo], ng = s_off[lo + 1] - s0;
    const int64_t w = gid - s0 * n_D;
    const int64_t d = w / ng, i = w - d * ng;
    make_screen<T>(depth, var, gain, t + s0, gid, i, ng, d, gap_max, dt, rec,
                   srec ? srec + fs.srec_off : nullptr, fs.n_slots,
                   slot_of + s0, vpair + s0);
}

// Slots of every sample of the screened curves (reg: two words per curve).
__global__ void k_slot_offsets_batch(const double* __restrict__ t,
                                     const FoldSeg* __restrict__ segs, int n_seg,
                                     const int64_t* __restrict__ s_off, double inv_dt,
                                     int* __restrict__ slot_of, unsigned* __restrict__ reg) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= s_off[n_seg]) return;
    int lo = 0, hi = n_seg;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (s_off[mid] <= i) lo = mid; else hi = mid;
    }
    const FoldSeg fs = segs[lo];
    if (!fs.screen) return;
    const int64_t s0 = s_off[lo];
    slot_offset(t + s0, i - s0, inv_dt, fs.n_slots, slot_of + s0, reg + 2 * lo);
}

__global__ void k_buckets_batch(const double* __restrict__ t, const FoldSeg* __restrict__ segs,
                                int n_seg, int64_t n_bucket_total, double dt,
                                int* __restrict__ bucket) {
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (b >= n_bucket_total) return;
    int lo = 0, hi = n_seg;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (segs[mid].bucket_off <= b) lo = mid; else hi = mid;
    }
    const FoldSeg fs = segs[lo];
    const double edge = fs.t_ref + (double)(b - fs.bucket_off) * dt;
    const double* t0 = t + fs.s_off;
    int64_t l = 0, h = fs.n_t0;
    while (l < h) {
        const int64_t mid = (l + h) >> 1;
        if (t0[mid] <= edge) l = mid + 1; else h = mid;
    }
    bucket[b] = (int)l;
}

__global__ void k_slot_fill_batch(const float* __restrict__ depth, const float* __restrict__ var,
                                  const float* __restrict__ gain, const double* __restrict__ t,
                                  const FoldSeg* __restrict__ segs, int n_seg,
                                  const int64_t* __restrict__ s_off, int n_D, double inv_dt,
                                  Node4<float>* __restrict__ rec) {
    const int64_t gid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (gid >= s_off[n_seg] * (int64_t)n_D) return;
    int lo = 0, hi = n_seg;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (s_off[mid] * (int64_t)n_D <= gid) lo = mid; else hi = mid;
    }
    const FoldSeg fs = segs[lo];
    if (!fs.use_slots) return;
    const int64_t s0 = s_off[lo], ng = s_off[lo + 1] - s0;
    const int64_t w = gid - s0 * n_D;
    const int64_t d = w / ng, i = w - d * ng;
    const int64_t s = (int64_t)rint((t[s0 + i] - fs.t_ref) * inv_dt);
    if (s < 0 || s >= fs.n_slots) return;
    const float dd = depth[gid], v = var[gid], l = gain[gid];
    Node4<float> r;
    r.d = dd;
    r.l = l;
    r.s = (isfinite(dd) && isfinite(v) && isfinite(l) && v > 0.f) ? sqrtf(v) : NAN;
    r.ig = 0.f;
    rec[fs.rec_off + d * fs.n_slots + s] = r;
}

// Regularity of each curve's epochs for the slot path (flag[g] = 1 if not).
__global__ void k_slots_batch(const double* __restrict__ t, const int64_t* __restrict__ s_off,
                              int n_seg, double inv_dt, int* __restrict__ irregular) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= s_off[n_seg]) return;
    int lo = 0, hi = n_seg;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (s_off[mid] <= i) lo = mid; else hi = mid;
    }
    const int64_t s0 = s_off[lo];
    const double tr = t[s0];
    const double u = (t[i] - tr) * inv_dt;
    const double sl = rint(u);
    bool bad = !(fabs(u - sl) <= 1e-3) || !(sl >= 0.0) || sl > 2.0e9;
    if (i > s0) bad = bad || !(sl > rint((t[i - 1] - tr) * inv_dt));
    if (bad) atomicExch(&irregular[lo], 1);
}

// Host side of the batch fold: per-curve layout and launches.

void plan_fold_batch(const std::vector<int64_t>& s_off, const std::vector<double>& t_first,
                     const std::vector<double>& t_last, const std::vector<int>& irregular,
                     bool fp64, double dt, double gap_factor, int n_D, int level,
                     FoldBatch& fb) {
    const int n_seg = (int)t_first.size();
    fb = FoldBatch{};
    fb.level = level;
    fb.segs.resize(n_seg);
    for (int g = 0; g < n_seg; ++g) {
        FoldSeg& f = fb.segs[g];
        f.s_off = s_off[g];
        f.n_t0 = s_off[g + 1] - s_off[g];
        f.t_ref = t_first[g];
        f.t_last = t_last[g];
        f.ulast = slot_ulast(f.t_ref, f.t_last, dt);
        f.uspan = exact_uspan(f.t_ref, f.t_last, dt);
        const double span = (t_last[g] - t_first[g]) / dt;
        f.n_bucket = (int64_t)span + 2;
        f.n_slots = f.n_bucket + 2;
        f.use_slots = (!fp64 && gap_factor > 1.0 && gap_factor < 2.0 && span < 4.0e6 &&
                       !irregular[g]) ? 1 : 0;
        f.screen = (!f.use_slots && gap_factor < 2.0 && span < 8.0e6 && (fp64 || level > 0)) ? 1
                                                                                             : 0;
        f.srec_off = fb.n_srec_total;
        fb.n_srec_total += fp64 && f.screen ? f.n_slots * n_D : 0;
        f.tab_off = fb.n_tab_total;
        f.g_off = fb.n_g_total;
        if (level == 2 && (f.screen || f.use_slots)) {
            const int64_t ns = filter_slots(f.n_slots);
            f.pair_off = fb.n_pair_total;
            fb.n_pair_total += ns * ((n_D + 1) / 2 * 2);
            fb.n_tab_total += ns * n_D;
            fb.n_g_total += ns * filter_cols(n_D);
        }
        f.bucket_off = fb.n_bucket_total;
        fb.n_bucket_total += f.use_slots ? 0 : f.n_bucket;
        f.rec_off = fb.n_rec_total;
        fb.n_rec_total += f.use_slots ? f.n_slots * n_D : 0;
        fb.any_slots = fb.any_slots || f.use_slots;
        fb.any_exact = fb.any_exact || !f.use_slots;
    }
}

size_t fold_scratch(const FoldBatch& fb, int64_t n_total, int n_lc, int n_D, int64_t n_P,
                    bool fp64, char* base, FoldScratch* fs) {
    size_t off = 0;
    auto take = [&](size_t bytes) {
        char* p = base ? base + off : nullptr;
        off += (bytes + 255) / 256 * 256;
        return p;
    };
    const bool lists = fb.level == 2;
    const int64_t items = std::min<int64_t>((int64_t)n_lc * n_P, BATCH_PASS);
    FoldScratch f{};
    f.pass = lists ? items : 0;
    f.nodes = take(fb.any_exact ? exact_layout(n_total, n_D, fp64, fp64 || fb.level > 0).total : 0);
    f.bucket = (int*)take((size_t)(fb.n_bucket_total + 1) * 4);
    f.rec = (Node4<float>*)take((size_t)(fb.n_rec_total + 1) * sizeof(Node4<float>));
    f.srec = (ScreenRec*)take((size_t)(fb.n_srec_total + 1) * sizeof(ScreenRec));
    f.slot_of = (int*)take(fp64 ? (size_t)n_total * sizeof(int) : 0);
    f.reg = (unsigned*)take((size_t)n_lc * 2 * sizeof(unsigned));
    f.peak = (unsigned long long*)take((size_t)n_lc * sizeof(unsigned long long));
    f.ptab = (PeriodConst*)take((size_t)n_P * period_const_bytes());
    if (lists) {
        const FilterLayout F = filter_layout(fb.n_tab_total, fb.n_pair_total, fb.n_g_total,
                                              (int64_t)n_lc * n_D);
        char* tab = take(F.total);
        if (base) f.tab = filter_tab(tab, F);
        f.n_list = (unsigned*)take(32);
        f.list = (unsigned*)take((size_t)items * sizeof(unsigned));
        if (fb.any_exact) {
            // one item leaves a few cells; an item that finds the list full
            // evaluates its own
            f.cap = (unsigned long long)(4 * items + 4096);
            f.cand = (FoldCand*)take((size_t)f.cap * sizeof(FoldCand));
            f.n_cand = (unsigned long long*)(f.n_list + 4);
            f.range = (int2*)take((size_t)items * sizeof(int2));
            f.items = (ItemConst*)take((size_t)items * sizeof(ItemConst));
        }
        if (fb.any_slots) f.sbest = (SlotBest*)take((size_t)items * sizeof(SlotBest));
    }
    if (fs) *fs = f;
    return off;
}

// The filter tables of every curve (the records they are built from are
// there).  Returns the first error of the memset.
static cudaError_t launch_filter_tables(const FoldSeg* segs, const FoldSeg& one, int n_seg,
                                        int n_D, int64_t n_entries, int64_t n_t0,
                                        const ScreenRec* screen, const ulonglong2* vpair,
                                        const int* bucket, const Node4<float>* rec,
                                        const FilterTab& tab, cudaStream_t st, int* launched) {
    if (n_entries == 0) return cudaSuccess;
    const int64_t rows = (int64_t)n_seg * n_D;
    if (tab.S) {
        const cudaError_t e = cudaMemsetAsync(tab.vmax, 0, (size_t)rows * sizeof(unsigned), st);
        if (e != cudaSuccess) return e;
        const unsigned gy = (unsigned)std::min<int64_t>(std::max<int64_t>(n_t0 / 512, 1), 64);
        k_filter_vmax<<<dim3((unsigned)rows, gy), 256, 0, st>>>(screen, rec, segs, one, n_D,
                                                                tab.vmax);
        ++*launched;
    }
    k_filter_slots<<<div_up(n_entries, 128), 128, 0, st>>>(screen, vpair, bucket, rec, segs, one,
                                                           n_seg, n_D, n_entries, tab);
    k_filter_groups<<<div_up(n_entries, 256), 256, 0, st>>>(segs, one, n_seg, n_D, n_entries, tab);
    *launched += 2;
    return cudaSuccess;
}

cudaError_t launch_fold_prep(const FoldBatch& fb, const FoldSeg* segs_dev,
                             const int64_t* s_off_dev, int n_seg, int64_t n_total, bool fp64,
                             const double* t, const void* depth, const void* var,
                             const void* gain, int n_D, double dt, double gap_factor,
                             const FoldScratch& fs, cudaStream_t st, int* n_launched) {
    int launched = 0;
    *n_launched = 0;
    const int64_t ngrid = n_total * (int64_t)n_D;
    const ExactLayout L = exact_layout(n_total, n_D, fp64, fp64 || fb.level > 0);
    ScreenRec* screen = (ScreenRec*)((char*)fs.nodes + L.off_screen);
    ulonglong2* vpair = (ulonglong2*)((char*)fs.nodes + L.off_vpos);
    cudaError_t e = cudaMemsetAsync(fs.peak, 0, (size_t)n_seg * sizeof(unsigned long long), st);
    if (e == cudaSuccess)
        e = cudaMemsetAsync(fs.reg, 0, (size_t)n_seg * 2 * sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    const dim3 peak_grid(n_seg, 1);
    if (fb.any_exact) {
        k_buckets_batch<<<div_up(fb.n_bucket_total, 256), 256, 0, st>>>(
            t, segs_dev, n_seg, fb.n_bucket_total, dt, fs.bucket);
        ++launched;
        if (fp64) {
            k_nodes_batch<double><<<div_up(ngrid, 256), 256, 0, st>>>(
                (const double*)depth, (const double*)var, (const double*)gain, t, segs_dev,
                n_seg, s_off_dev, n_D, gap_factor * dt, (Node8<double>*)fs.nodes);
            k_slot_offsets_batch<<<div_up(n_total, 256), 256, 0, st>>>(
                t, segs_dev, n_seg, s_off_dev, 1.0 / dt, fs.slot_of, fs.reg);
            k_fill_screen<<<div_up(fb.n_srec_total + 1, 256), 256, 0, st>>>(
                fs.srec, fb.n_srec_total);
            k_screen_batch<double><<<div_up(ngrid, 256), 256, 0, st>>>(
                (const double*)depth, (const double*)var, (const double*)gain, t, segs_dev,
                n_seg, s_off_dev, n_D, gap_factor * dt, dt, screen, vpair, fs.srec, fs.slot_of);
            launched += 4;
        } else {
            k_nodes_batch<float><<<div_up(ngrid, 256), 256, 0, st>>>(
                (const float*)depth, (const float*)var, (const float*)gain, t, segs_dev, n_seg,
                s_off_dev, n_D, gap_factor * dt, (Node8<float>*)fs.nodes);
            ++launched;
        }
        if (!fp64 && fb.level > 0) {
            k_screen_batch<float><<<div_up(ngrid, 256), 256, 0, st>>>(
                (const float*)depth, (const float*)var, (const float*)gain, t, segs_dev, n_seg,
                s_off_dev, n_D, gap_factor * dt, dt, screen, vpair, nullptr, nullptr);
            ++launched;
        }
    }
    if (fb.any_slots) {
        k_fill_nan<<<div_up(fb.n_rec_total, 256), 256, 0, st>>>(fs.rec, fb.n_rec_total);
        k_slot_fill_batch<<<div_up(ngrid, 256), 256, 0, st>>>(
            (const float*)depth, (const float*)var, (const float*)gain, t, segs_dev, n_seg,
            s_off_dev, n_D, 1.0 / dt, fs.rec);
        launched += 2;
    }
    if (fp64)
        k_gain_peak<double><<<peak_grid, 256, 0, st>>>((const double*)gain, s_off_dev, n_D,
                                                       fs.peak);
    else
        k_gain_peak<float><<<peak_grid, 256, 0, st>>>((const float*)gain, s_off_dev, n_D,
                                                      fs.peak);
    ++launched;
    if (fb.level == 2)
        e = launch_filter_tables(segs_dev, FoldSeg{}, n_seg, n_D, fb.n_tab_total,
                                 n_total / n_seg, screen, vpair, fs.bucket, fs.rec, fs.tab, st,
                                 &launched);
    *n_launched = launched;
    return e;
}

// Warps per item of n, each of `steps` slots x durations: eight where the items are
// few for their size, two (and eight for the long ones) from where they fill the
// GPU, one from 6 000 up by size, at the latest from 18 000 periods of one curve or
// 40 000 items of a batch.  One curve, FP64, us with eight / two / one: 2 000 periods
// of 2 000 epochs x 4 durations 307 / 281 / 358, 10 000 of them 717 / 471 / 400; 2 000
// of 8 000 x 4 475 / 531 / 637; 10 000 of 19 440 x 10 2 148 / 1 792 / 2 052, 18 000 two
// 2 630, one 2 400, 18 000 uniform in frequency 4 350, 5 170, 26 000 5 900, 5 970.  100
// curves of 2 000 x 8, 1 000 periods: two 8.4 ms, one 7.2; 64 of 18 000 x 10, 500
// periods, 15.4, 16.3.
static int fold_warps(int64_t n, double steps, bool batch) {
    if (n >= std::min(batch ? 40000.0 : 18000.0, 6000.0 + steps / 6.0)) return 1;
    return n >= std::min(6000.0, 1000.0 + steps / 32.0) ? 2 : 8;
}

// Epochs per cell of an item that takes a block of eight warps (45 beside one warp:
// 100 000 periods of 136 080 x 20, mixed, 95.9 -> 98.3 ms; 438 curves of 8 000-20 000 x
// 10 x 4 000, 241.9 -> 244.7).
constexpr float HEAVY_K = 22.f;
// How many of the n items may take blocks of eight: more fill the GPU either way,
// and one or two warps idle less at the ends of an item's rounds.  Beside two
// warps, periods uniform in frequency, with blocks / without: 10 000 of 19 440 x 10,
// mixed 3.28 / 2.50 ms, FP64 3.48 / 3.06; 14 curves of 12 000-18 000 x 7 durations x
// 969, mixed, 4.69 / 4.14 (one duration has few cells a period: 10 000 of 100 000 x
// 1, FP64, 3.93 / 4.44).  Beside one warp: 404 curves of 4 600-7 000 x 3 x 3 340, 23 %
// of the items long, FP64, 95.6 / 91.5; 438 of 8 000-20 000 x 10 x 4 000, 4 % long,
// mixed, 240 / 244.
static unsigned list_max(int nw, int n_D, int64_t n) {
    if (nw == 1) return (unsigned)std::min<int64_t>(n / 10, 0xffffffffll);
    return n_D > 1 ? 5000u : ~0u;
}

// The cell kernels of one job: the exact paths' items, then the slot path's.
// nw = 1 or 2 warps per item; with a list, its items run in eight-warp blocks on
// the side stream meanwhile.  nw = 8: every item in such a block.
static int launch_cells(const FoldJob& J, bool fp64, bool exact, bool slots, int nw,
                        cudaStream_t st, cudaStream_t side, cudaError_t* err) {
    const int64_t items = (int64_t)J.n_seg * J.n_P;
    int launched = 0;
    int dev = 0, n_sm = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    auto check = [&](cudaError_t e) {
        if (e != cudaSuccess && *err == cudaSuccess) *err = e;
    };
    if (nw == 2 && items > 0x7fffffffLL) nw = 1;          // the grid's limit
    const int g8 = (int)std::min<int64_t>(items, (int64_t)n_sm * (FOLD_WARPS / 8));
    // (the gains' tables alone: kernels of their own)
    const bool lone = J.tab.L && !J.tab.S;
#define NU_CELLS_AS(NW_, LONE_, GRID_, ST_)                                                \
    do {                                                                                   \
        const dim3 g_(GRID_), b_(fold_threads(NW_));                                       \
        if (path == 1) k_fold_slot_cells<NW_, LONE_><<<g_, b_, 0, ST_>>>(J);               \
        else if (fp64) k_fold_cells<double, NW_, LONE_><<<g_, b_, 0, ST_>>>(J);            \
        else k_fold_cells<float, NW_, LONE_><<<g_, b_, 0, ST_>>>(J);                       \
        ++launched;                                                                        \
    } while (0)
#define NU_CELLS(NW_, GRID_, ST_)                                                          \
    do {                                                                                   \
        if (lone) NU_CELLS_AS(NW_, true, GRID_, ST_);                                      \
        else NU_CELLS_AS(NW_, false, GRID_, ST_);                                          \
    } while (0)
    for (int path = 0; path < 2; ++path) {
        if (!(path == 0 ? exact : slots)) continue;
        // the list's counters and, behind them, the candidates'
        if (J.cand || J.list.block) check(cudaMemsetAsync(J.counters, 0, 32, st));
        if (path == 0 && J.items) {
            k_item_consts<<<div_up(items, 128), 128, 0, st>>>(J, fp64 ? 0 : 1);
            ++launched;
        }
        if (path == 1 && J.list.block) {
            k_slot_items<<<div_up(items, 128), 128, 0, st>>>(J);
            ++launched;
        }
        if (nw == 8) {
            NU_CELLS(8, g8, st);
        } else {
            cudaEvent_t fork = nullptr, join = nullptr;
            bool forked = false;
            if (J.list.block) {
                forked = side && side != st &&
                         cudaEventCreateWithFlags(&fork, cudaEventDisableTiming) == cudaSuccess &&
                         cudaEventCreateWithFlags(&join, cudaEventDisableTiming) == cudaSuccess &&
                         cudaEventRecord(fork, st) == cudaSuccess &&
                         cudaStreamWaitEvent(side, fork, 0) == cudaSuccess;
                const cudaStream_t hs = forked ? side : st;
                NU_CELLS(8, g8, hs);
                if (forked) check(cudaEventRecord(join, side));
            }
            if (nw == 2) NU_CELLS(2, (unsigned)items, st);
            else NU_CELLS(1, div_up(items, 4), st);
            if (forked) {
                const cudaError_t ej = cudaStreamWaitEvent(st, join, 0);
                check(ej);
                // not joined: the caller gives the scratch back in st's order
                if (ej != cudaSuccess) cudaStreamSynchronize(side);
            }
            if (fork) cudaEventDestroy(fork);
            if (join) cudaEventDestroy(join);
        }
        if (path == 0 && J.cand) {
            // a warp per 32 cells, enough warps that each takes few rounds
            const int eg = (int)std::min<int64_t>(div_up(items, 16), n_sm * 16);
            if (fp64) k_cand_eval<double><<<eg, 64, 0, st>>>(J);
            else k_cand_eval<float><<<eg, 64, 0, st>>>(J);
            k_cand_best<<<div_up(items, 128), 128, 0, st>>>(J);
            launched += 2;
        }
        if (path == 1 && J.sbest) {
            k_slot_best<<<div_up(items, 128), 128, 0, st>>>(J);
            ++launched;
        }
    }
#undef NU_CELLS
#undef NU_CELLS_AS
    return launched;
}

int launch_fold_batch(const FoldBatch& fb, const FoldSeg* segs_dev, int n_seg,
                      int64_t n_total, bool fp64, const double* t, const FoldScratch& fs,
                      int n_D, double dt, double gap_factor, const double* periods,
                      int64_t n_P, double* Q, double* T0, int* Didx, double* dep,
                      double* sig, double* lnp, cudaStream_t st, cudaStream_t side,
                      cudaError_t* err) {
    int launched = 0;
    const ExactLayout L = exact_layout(n_total, n_D, fp64, fp64 || fb.level > 0);
    FoldJob J{};
    J.segs = segs_dev;
    J.n_seg = n_seg;
    J.n_D = n_D;
    J.dt = dt;
    J.inv_dt = 1.0 / dt;
    J.gap_max = gap_factor * dt;
    J.t = t;
    J.nodes = fs.nodes;
    J.screen = (const ScreenRec*)((const char*)fs.nodes + L.off_screen);
    J.vpair = (const ulonglong2*)((const char*)fs.nodes + L.off_vpos);
    J.srec = fp64 ? fs.srec : nullptr;
    J.reg = fs.reg;
    J.peak = fs.peak;
    J.bucket = fs.bucket;
    J.rec = fs.rec;
    J.tab = fs.tab;
    J.periods = periods;
    J.ptab = fs.ptab;
    J.stab = reinterpret_cast<const SlotPeriod*>(fs.ptab);
    J.n_P = n_P;
    J.Q = Q;
    J.T0 = T0;
    J.Didx = Didx;
    J.dep = dep;
    J.sig = sig;
    J.lnp = lnp;
    J.cand = fs.cand;
    J.n_cand = fs.n_cand;
    J.cap = fs.cap;
    J.range = fs.range;
    J.items = fs.items;
    J.sbest = fs.sbest;
    J.counters = fs.n_list;
    int64_t slots = 0;
    for (int g = 0; g < n_seg; ++g) slots += fb.segs[g].n_bucket;
    const int nw = fold_warps((int64_t)n_seg * n_P, (double)slots / n_seg * n_D, true);
    // The passes: whole curves, or parts of one curve's periods.
    const int64_t pass = fs.pass ? fs.pass : (int64_t)n_seg * n_P;
    int64_t segs_pass = std::min<int64_t>(std::max<int64_t>(pass / n_P, 1), n_seg);
    segs_pass = div_up(n_seg, div_up(n_seg, segs_pass));
    const int64_t per_pass = std::min(n_P, pass);
    auto cells = [&](bool exact) {
        for (int64_t g = 0; g < n_seg; g += segs_pass)
            for (int64_t p = 0; p < n_P; p += per_pass) {
                FoldJob K = J;
                const int64_t o = g * n_P + p;
                K.segs += g;
                K.n_seg = (int)std::min<int64_t>(segs_pass, n_seg - g);
                K.reg += 2 * g;
                K.peak += g;
                K.periods += p;
                K.ptab += p;
                K.stab += p;
                K.n_P = std::min(per_pass, n_P - p);
                if (nw != 8 && fs.list)
                    K.list = FoldLists{fs.list, fs.n_list, HEAVY_K,
                                       list_max(nw, n_D, K.n_seg * K.n_P)};
                K.Q += o;
                K.T0 += o;
                K.Didx += o;
                K.dep += o;
                K.sig += o;
                K.lnp += o;
                launched += launch_cells(K, fp64, exact, !exact, nw, st, side, err);
            }
    };
    // (the two paths' period tables share a buffer)
    if (fb.any_exact) {
        k_period_consts<<<div_up(n_P, 256), 256, 0, st>>>(periods, n_P, dt, fs.ptab);
        ++launched;
        cells(true);
    }
    if (fb.any_slots) {
        k_slot_periods<<<div_up(n_P, 256), 256, 0, st>>>(periods, n_P, dt,
                                                         reinterpret_cast<SlotPeriod*>(fs.ptab));
        ++launched;
        cells(false);
    }
    return launched;
}

int launch_slots_test(const double* t, const int64_t* s_off_dev, int n_seg, int64_t n_total,
                      double dt, int* irregular, cudaStream_t st) {
    k_slots_batch<<<div_up(n_total, 256), 256, 0, st>>>(t, s_off_dev, n_seg, 1.0 / dt,
                                                       irregular);
    return 1;
}

}  // namespace nu

// ------------------------------------------------ single-curve host side
namespace nu {

// One call of the single-curve fold.
struct FoldCall {
    const char* who;
    const double* t0s;
    int64_t n_t0;
    int n_D;
    const void *depth, *var, *dlnl;
    bool fp64;
    const double* periods;
    int64_t n_P;
    double phase_step, gap_factor, t_ref, t_last;
    int64_t n_bucket;
    cudaStream_t st;
    bool fork;           // block items may run on a side stream (two events per pass
                         // with a list, and the stream with a thread's first such call)
    double *Q, *T0;
    int32_t* D_idx;
    double *dep, *sig, *lnP;

    double span_steps() const { return (t_last - t_ref) / phase_step; }
    int64_t n_slots() const { return n_bucket + 2; }      // slot records, NaN padded
    double item_steps() const { return span_steps() * n_D; }
    // the slot path needs a regular grid and a gap rule that only joins
    // neighbouring slots (1 < gap_factor < 2)
    bool may_use_slots() const {
        return !fp64 && gap_factor > 1.0 && gap_factor < 2.0 && span_steps() < 4.0e6;
    }
    // gap rules and spans that the screen does not cover: every cell is evaluated
    bool may_screen() const { return gap_factor < 2.0 && span_steps() < 8.0e6; }
    // Small calls: screening every cell costs less than the filters' tables and
    // rounds, and a few survivors per block less than the launches that pack
    // them.  FP64, us with filters -> without: 4 000 epochs x 4 durations x 1 200
    // periods (19 M steps) 365 -> 276, 1 100 x 12 x 300 (4 M) 285 -> 174; 2 000 x 12
    // x 1 200 (29 M) 325 -> 352; one duration, 8 000 x 4 000 (32 M) 472 -> 429.
    // On the slot path they bound by the gains that the records hold, which are
    // written with them (slots: 2 000 x 4 x 2 000, 17 M, 223 -> 186 us against
    // every cell; 1 100 x 4 x 12 000, 54 M, 344 -> 250 against all tables; items of
    // more steps go to the tables sooner: 4 000 x 20 x 1 000, 88 M, 330 with, 360
    // without).
    bool small(bool slots) const {
        const double work = item_steps() * (double)n_P;
        if (slots) return work < (item_steps() < 4.0e4 ? 6.0e7 : 2.4e7);
        return work < (n_D == 1 ? 4.0e7 : 2.4e7);
    }
    int warps(int64_t n) const { return fold_warps(n, item_steps(), false); }
};

// What a fold keeps in scratch beside the records of its events.
struct FoldPlan {
    bool slots;          // the mixed regular path's records, else the exact paths'
    bool screen;         // exact paths: the screen's records
    int tables;          // filter tables: 2 all, 1 the gains', 0 none; TABLES_SLOT: the
                         // slot path's L, written with its records
    int64_t pass;        // periods per pass, with their table and lists; 0: all in one
                         // pass without (survivors are evaluated in place)
};

constexpr int TABLES_SLOT = 3;
// The plans of a call, the best one first; the last needs the least.  Period
// tables and lists take 290 bytes per period, so that a long grid of periods goes
// through them in passes: 2^19 periods at most, and fewer where scratch is
// short, as the filters are worth more than one pass (19 440 epochs x 10
// durations x 20 000 periods, FP64: 2.9 ms in one pass, 4.2 in the passes that
// 32 MiB hold, 23.6 in one without filters).
constexpr int64_t PASS_MAX = 1ll << 19, PASS_MIN = 2048;
static std::vector<FoldPlan> fold_plans(const FoldCall& C, bool slots) {
    std::vector<FoldPlan> plans;
    const bool screen = !slots && C.may_screen();
    if (slots || screen) {
        for (int tables = !C.small(slots) ? 2 : (slots ? TABLES_SLOT : 0); tables >= 0;
             tables = tables == TABLES_SLOT ? 0 : tables - 1) {
            for (int64_t k = (C.n_P + PASS_MAX - 1) / PASS_MAX;; k += std::max<int64_t>(1, k / 4)) {
                const int64_t pass = (C.n_P + k - 1) / k;
                if (pass < PASS_MIN && pass < C.n_P) break;
                plans.push_back(FoldPlan{slots, screen, tables, pass});
                if (pass == 1) break;
            }
            plans.push_back(FoldPlan{slots, screen, tables, 0});
        }
    }
    if (!slots && !(screen && C.fp64)) plans.push_back(FoldPlan{false, false, 0, 0});
    return plans;
}

// Scratch layout of one plan.  The flags and the epochs' slots come first in
// all of them: which records a mixed call fills is known after its slot test.
struct SingleLayout {
    FoldPlan plan;
    ExactLayout el;
    FilterLayout fl;
    size_t flag, slot_of, records, bucket, srec, tab, ptab, cand, range, items, list, sbest, total;
    unsigned long long cap;
};
static SingleLayout single_layout(const FoldCall& C, const FoldPlan& plan) {
    SingleLayout L{};
    L.plan = plan;
    size_t end = 0;
    auto take = [&](size_t bytes) {
        const size_t at = end;
        end += (bytes + 255) / 256 * 256;
        return at;
    };
    const int64_t n_slots = C.n_slots();
    L.flag = take(256);
    L.slot_of = take((size_t)C.n_t0 * sizeof(int));
    if (plan.slots) {
        L.records = take((size_t)n_slots * C.n_D * sizeof(Node4<float>));
    } else {
        L.el = exact_layout(C.n_t0, C.n_D, C.fp64, plan.screen);
        L.records = take(L.el.total);
        L.bucket = take((size_t)C.n_bucket * sizeof(int));
        if (C.fp64 && plan.screen) L.srec = take((size_t)n_slots * C.n_D * sizeof(ScreenRec));
    }
    const int64_t ns = filter_slots(n_slots);
    if (plan.tables == TABLES_SLOT) {
        L.tab = take((size_t)ns * C.n_D * sizeof(float));
    } else if (plan.tables) {
        L.fl = filter_layout(ns * C.n_D, ns * ((C.n_D + 1) / 2 * 2),
                             ns * filter_cols(C.n_D), C.n_D,
                             plan.tables == 1);
        L.tab = take(L.fl.total);
    }
    if (plan.pass) {
        L.ptab = take((size_t)plan.pass * (plan.slots ? sizeof(SlotPeriod) : sizeof(PeriodConst)));
        L.list = take((size_t)plan.pass * sizeof(unsigned));
        if (plan.slots) {
            L.sbest = take((size_t)plan.pass * sizeof(SlotBest));
        } else {
            // (an item that finds the list full evaluates its cells in place)
            L.cap = (unsigned long long)(4 * plan.pass + 1024);
            L.cand = take((size_t)L.cap * sizeof(FoldCand));
            L.range = take((size_t)plan.pass * sizeof(int2));
            L.items = take((size_t)plan.pass * sizeof(ItemConst));
        }
    }
    L.total = end;
    return L;
}

// Enqueue the fold of one light curve with its scratch at `scratch`, laid out by
// Le, or by Ls (if given) when the mixed precision's slot test finds a regular
// grid; the test reads one flag back (one synchronisation of the stream).
static nu_status single_fold(const FoldCall& C, char* scratch, const SingleLayout* Ls,
                             const SingleLayout& Le) {
    const int64_t n_t0 = C.n_t0, n_P = C.n_P, n_bucket = C.n_bucket, n_slots = C.n_slots();
    const int n_D = C.n_D;
    const bool fp64 = C.fp64;
    const double phase_step = C.phase_step;
    const cudaStream_t st = C.st;
    const int64_t ngrid = n_t0 * (int64_t)n_D;
    int* slot_of = (int*)(scratch + Le.slot_of);
    int* flag = (int*)(scratch + Le.flag);
    int launched = 0;
    // one block of flags: [0] slot test, [1..2] regular-grid test, then the
    // peak key and the candidate counter
    cudaError_t e = cudaMemsetAsync(flag, 0, 256, st);
    const unsigned peak_grid = (unsigned)std::min<int64_t>(div_up(ngrid, 2048), 608);
    unsigned long long* peak = (unsigned long long*)(scratch + Le.flag + 16);
    bool use_slots = Ls != nullptr;
    if (use_slots) {
        int irregular = 0;
        k_slots<<<div_up(n_t0, 256), 256, 0, st>>>(C.t0s, n_t0, C.t_ref, 1.0 / phase_step,
                                                  slot_of, flag);
        // The tables of that path are filled before the test is read, so that
        // the host's next launch is the fold's (an irregular curve overwrites
        // them: 10 us on the GPU, hidden in part by the wait).
        const int64_t nrec = n_slots * n_D;
        Node4<float>* rec = (Node4<float>*)(scratch + Ls->records);
        const int64_t ns = filter_slots(n_slots);
        float* Lg = Ls->plan.tables == TABLES_SLOT ? (float*)(scratch + Ls->tab) : nullptr;
        const int64_t n_L = Lg ? ns * n_D : 0;
        const unsigned b_rec = (unsigned)div_up(std::max(nrec, n_L), 256);
        const unsigned b_peak = b_rec + peak_grid;
        const unsigned b_all = b_peak + (unsigned)div_up(Ls->plan.pass, 256);
        k_slot_prep<<<b_all, 256, 0, st>>>(rec, nrec, Lg, n_L, b_rec, (const float*)C.dlnl, ngrid,
                                           b_peak, peak, C.periods, Ls->plan.pass, phase_step,
                                           (SlotPeriod*)(scratch + Ls->ptab));
        k_slot_fill<<<div_up(ngrid, 256), 256, 0, st>>>(
            (const float*)C.depth, (const float*)C.var, (const float*)C.dlnl, slot_of,
            n_t0, n_D, n_slots, rec, Lg, ns);
        launched += 3;
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(&irregular, flag, sizeof(int), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        use_slots = irregular == 0;
    }
    if (e != cudaSuccess) {
        count_launches(launched);
        return cuda_fail(e, (std::string(C.who) + ": slot test").c_str());
    }
    const SingleLayout& L = use_slots ? *Ls : Le;
    FoldJob J{};
    J.n_seg = 1;
    J.n_D = n_D;
    J.dt = phase_step;
    J.inv_dt = 1.0 / phase_step;
    J.gap_max = C.gap_factor * phase_step;
    J.t = C.t0s;
    J.nodes = scratch + L.records;
    J.screen = (const ScreenRec*)(scratch + L.records + L.el.off_screen);
    J.vpair = (const ulonglong2*)(scratch + L.records + L.el.off_vpos);
    J.srec = fp64 && L.plan.screen ? (const ScreenRec*)(scratch + L.srec) : nullptr;
    J.reg = (const unsigned*)(flag + 1);
    J.peak = peak;
    J.bucket = (const int*)(scratch + L.bucket);
    J.rec = (const Node4<float>*)(scratch + L.records);
    FoldSeg& one = J.one;
    one.n_t0 = n_t0;
    one.t_ref = C.t_ref;
    one.t_last = C.t_last;
    one.n_bucket = n_bucket;
    one.n_slots = n_slots;
    one.use_slots = use_slots ? 1 : 0;
    one.screen = L.plan.screen ? 1 : 0;
    if (use_slots) one.ulast = slot_ulast(C.t_ref, C.t_last, phase_step);
    else one.uspan = exact_uspan(C.t_ref, C.t_last, phase_step);
    const int64_t pass = L.plan.pass ? L.plan.pass : n_P;
    if (L.plan.pass) {
        J.ptab = (const PeriodConst*)(scratch + L.ptab);
        J.stab = (const SlotPeriod*)(scratch + L.ptab);
    }
    if (L.plan.tables == TABLES_SLOT) J.tab.L = (float*)(scratch + L.tab);
    else if (L.plan.tables) J.tab = filter_tab(scratch + L.tab, L.fl, L.plan.tables == 1);
    if (!use_slots) {
        const double gap_max = J.gap_max;
        ScreenRec* screen = (ScreenRec*)J.screen;
        ulonglong2* vpair = (ulonglong2*)J.vpair;
        ScreenRec* srec = (ScreenRec*)J.srec;
        auto prep = [&](auto zero) {
            using T = decltype(zero);
            FoldPrep<T> A{(const T*)C.depth, (const T*)C.var, (const T*)C.dlnl, C.t0s,
                          n_t0, n_D, C.t_ref, phase_step, gap_max, n_bucket,
                          (int*)(scratch + L.bucket), (Node8<T>*)(scratch + L.records), n_slots,
                          slot_of, (unsigned*)(flag + 1), srec, C.periods, L.plan.pass,
                          J.ptab ? (PeriodConst*)(scratch + L.ptab) : nullptr, peak, {}};
            const unsigned blocks[PREP_N] = {
                (unsigned)div_up(n_bucket, 256), one.screen ? peak_grid : 0u,
                J.ptab ? (unsigned)div_up(L.plan.pass, 256) : 0u,
                srec ? (unsigned)div_up(n_t0, 256) : 0u,
                srec ? (unsigned)div_up(n_slots * n_D, 256) : 0u,
                (unsigned)div_up(ngrid, 256)};
            unsigned n = 0;
            for (int q = 0; q < PREP_N; ++q) A.end[q] = n += blocks[q];
            k_fold_prep<T><<<n, 256, 0, st>>>(A);
        };
        if (fp64) prep(0.0); else prep(0.0f);
        ++launched;
        if (!one.screen) {
            const FoldGeom g{C.t0s, n_t0, C.t_ref, C.t_last, phase_step, 1.0 / phase_step,
                             gap_max, (const int*)(scratch + L.bucket), n_bucket};
            if (fp64)
                k_fold_exact<double><<<(unsigned)n_P, 256, 0, st>>>(
                    g, (const Node8<double>*)J.nodes, n_D, C.periods, n_P, C.Q, C.T0, C.D_idx,
                    C.dep, C.sig, C.lnP);
            else
                k_fold_exact<float><<<(unsigned)n_P, 256, 0, st>>>(
                    g, (const Node8<float>*)J.nodes, n_D, C.periods, n_P, C.Q, C.T0, C.D_idx,
                    C.dep, C.sig, C.lnP);
            count_launches(launched + 1);
            e = cudaGetLastError();
            if (e != cudaSuccess) return cuda_fail(e, (std::string(C.who) + ": launch").c_str());
            return NU_OK;
        }
        if (fp64) {
            k_screen<double><<<div_up(ngrid, 256), 256, 0, st>>>(
                (const double*)C.depth, (const double*)C.var, (const double*)C.dlnl, C.t0s, n_t0,
                n_D, gap_max, phase_step, screen, srec, n_slots, slot_of, vpair);
        } else {
            k_screen<float><<<div_up(ngrid, 256), 256, 0, st>>>(
                (const float*)C.depth, (const float*)C.var, (const float*)C.dlnl, C.t0s, n_t0,
                n_D, gap_max, phase_step, screen, nullptr, n_slots, nullptr, vpair);
        }
        ++launched;
    }
    if (J.tab.G)
        e = launch_filter_tables(nullptr, one, 1, n_D, filter_slots(n_slots) * n_D, n_t0, J.screen,
                                 J.vpair, J.bucket, J.rec, J.tab, st, &launched);
    for (int64_t p0 = 0; p0 < n_P && e == cudaSuccess; p0 += pass) {
        const int64_t n = std::min(pass, n_P - p0);
        J.periods = C.periods + p0;
        J.n_P = n;
        J.Q = C.Q + p0;
        J.T0 = C.T0 + p0;
        J.Didx = C.D_idx + p0;
        J.dep = C.dep + p0;
        J.sig = C.sig + p0;
        J.lnp = C.lnP + p0;
        if (p0 > 0) {
            if (use_slots)
                k_slot_periods<<<div_up(n, 256), 256, 0, st>>>(J.periods, n, phase_step,
                                                               (SlotPeriod*)(scratch + L.ptab));
            else
                k_period_consts<<<div_up(n, 256), 256, 0, st>>>(J.periods, n, phase_step,
                                                                (PeriodConst*)(scratch + L.ptab));
            ++launched;
        }
        const int nw = C.warps(n);
        if (L.plan.pass && !(C.small(use_slots) && (nw == 8 || use_slots))) {
            J.counters = (unsigned*)(scratch + L.flag + 64);
            if (use_slots) {
                J.sbest = (SlotBest*)(scratch + L.sbest);
            } else {
                J.cand = (FoldCand*)(scratch + L.cand);
                J.n_cand = (unsigned long long*)(J.counters + 4);
                J.cap = L.cap;
                J.range = (int2*)(scratch + L.range);
                J.items = (ItemConst*)(scratch + L.items);
            }
            J.list = nw != 8 ? FoldLists{(unsigned*)(scratch + L.list), J.counters, HEAVY_K,
                                         list_max(nw, n_D, n)}
                             : FoldLists{};
        }
        const cudaStream_t side = C.fork && J.list.block ? thread_side_stream() : nullptr;
        launched += launch_cells(J, fp64, !use_slots, use_slots, nw, st, side, &e);
    }
    count_launches(launched);
    if (e == cudaSuccess) e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, (std::string(C.who) + ": launch").c_str());
    return NU_OK;
}

static nu_status check_args(const char* who, const double* t0s_dev, int64_t n_t0, int n_D,
                            const void* depth_dev, const void* var_dev, const void* dlnl_dev,
                            nu_precision prec, const double* periods_dev, int64_t n_P,
                            double gap_factor, double* Q_dev, double* T0_dev,
                            int32_t* D_idx_dev, double* depth_out_dev, double* sigma_out_dev,
                            double* lnP_dev) {
    if (!t0s_dev || !depth_dev || !var_dev || !dlnl_dev || !periods_dev || !Q_dev ||
        !T0_dev || !D_idx_dev || !depth_out_dev || !sigma_out_dev || !lnP_dev)
        return fail(NU_EINVAL, "%s: null array", who);
    if (n_t0 < 2 || n_D < 1 || n_P < 1)
        return fail(NU_EINVAL, "%s: need n_t0 >= 2, n_D >= 1, n_P >= 1", who);
    if (prec != NU_FP64 && prec != NU_MIXED) return fail(NU_EINVAL, "%s: unknown precision", who);
    if (!(gap_factor > 0.0)) return fail(NU_EINVAL, "%s: gap_factor <= 0", who);
    if (n_t0 > 2000000000LL) return fail(NU_EINVAL, "%s: n_t0 too large", who);
    if (n_P > 2147483647LL) return fail(NU_EINVAL, "%s: n_P too large", who);
    return NU_OK;
}

}  // namespace nu

using namespace nu;

extern "C" nu_status nu_periodic_search(const double* t0s_dev, int64_t n_t0,
                                        const double* Ds_host, int n_D,
                                        const void* depth_dev, const void* var_dev,
                                        const void* dlnl_dev, nu_precision prec,
                                        const double* periods_dev, int64_t n_P,
                                        double phase_step, double gap_factor, void* stream,
                                        double* Q_dev, double* T0_dev, int32_t* D_idx_dev,
                                        double* depth_out_dev, double* sigma_out_dev,
                                        double* lnP_dev) {
    const char* who = "nu_periodic_search";
    (void)Ds_host;
    nu_status s = check_args(who, t0s_dev, n_t0, n_D, depth_dev, var_dev, dlnl_dev, prec,
                             periods_dev, n_P, gap_factor, Q_dev, T0_dev, D_idx_dev,
                             depth_out_dev, sigma_out_dev, lnP_dev);
    if (s != NU_OK) return s;
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e;
    // grid end points (the step, when not given, is the median spacing of the
    // epochs)
    double ends[2];
    double t_ref, t_last;
    if (!(phase_step > 0.0)) {
        e = median_spacing(t0s_dev, n_t0, st, &phase_step, &t_ref, &t_last);
        if (e != cudaSuccess) return cuda_fail(e, "nu_periodic_search: median spacing");
    } else {
        e = cudaMemcpyAsync(&ends[0], t0s_dev, sizeof(double), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess)
            e = cudaMemcpyAsync(&ends[1], t0s_dev + n_t0 - 1, sizeof(double),
                                cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return cuda_fail(e, "nu_periodic_search: copy ends");
        t_ref = ends[0];
        t_last = ends[1];
    }
    if (!(phase_step > 0.0) || !std::isfinite(phase_step))
        return fail(NU_EINVAL, "nu_periodic_search: phase step must be > 0");
    if (!(t_last >= t_ref)) return fail(NU_EINVAL, "nu_periodic_search: t0s not sorted");
    const double span_steps = (t_last - t_ref) / phase_step;
    if (span_steps > 1.0e9) return fail(NU_EINVAL, "nu_periodic_search: phase grid too fine");
    const FoldCall C{who, t0s_dev, n_t0, n_D, depth_dev, var_dev, dlnl_dev, prec == NU_FP64,
                     periods_dev, n_P, phase_step, gap_factor, t_ref, t_last,
                     (int64_t)span_steps + 2, st, true, Q_dev, T0_dev, D_idx_dev, depth_out_dev,
                     sigma_out_dev, lnP_dev};
    // the best plan that there is memory for
    pool_keep_memory();
    const std::vector<FoldPlan> pe = fold_plans(C, false);
    const std::vector<FoldPlan> ps =
        C.may_use_slots() ? fold_plans(C, true) : std::vector<FoldPlan>{};
    char* scratch = nullptr;
    SingleLayout Le, Ls{};
    for (size_t i = 0; i < std::max(pe.size(), ps.size()); ++i) {
        Le = single_layout(C, pe[std::min(i, pe.size() - 1)]);
        if (!ps.empty()) Ls = single_layout(C, ps[std::min(i, ps.size() - 1)]);
        e = cudaMallocAsync((void**)&scratch, std::max(Le.total, Ls.total), st);
        if (e != cudaErrorMemoryAllocation) break;
        cudaGetLastError();
    }
    if (e != cudaSuccess) return cuda_fail(e, "nu_periodic_search: cudaMallocAsync");
    s = single_fold(C, scratch, ps.empty() ? nullptr : &Ls, Le);
    e = cudaFreeAsync(scratch, st);
    if (s != NU_OK) return s;
    if (e != cudaSuccess) return cuda_fail(e, "nu_periodic_search: cudaFreeAsync");
    return NU_OK;
}

// ------------------------------------------------ transit masking
// One thread per epoch: the distance to the nearest transit of (P, T0),
// each operation rounded once (no contraction), decides for all durations.
template <typename T>
__global__ void k_mask_transits(const double* __restrict__ t0s, int64_t n_t0, int n_D,
                                T* __restrict__ depth, T* __restrict__ var,
                                T* __restrict__ dlnl, double P, double T0, double hw) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n_t0) return;
    const double t = t0s[i];
    const double n = rint(__ddiv_rn(__dsub_rn(t, T0), P));
    const double dist = fabs(__dsub_rn(t, __dadd_rn(T0, __dmul_rn(n, P))));
    if (!(dist < hw)) return;
    for (int d = 0; d < n_D; ++d) {
        const int64_t o = (int64_t)d * n_t0 + i;
        depth[o] = T(NAN);
        var[o] = T(NAN);
        dlnl[o] = T(NAN);
    }
}

extern "C" nu_status nu_mask_transits(const double* t0s_dev, int64_t n_t0, int n_D,
                                      void* depth_dev, void* var_dev, void* dlnl_dev,
                                      nu_precision prec, double P, double T0,
                                      double half_width, void* stream) {
    if (!t0s_dev || !depth_dev || !var_dev || !dlnl_dev)
        return fail(NU_EINVAL, "nu_mask_transits: null array");
    if (n_t0 < 1 || n_D < 1) return fail(NU_EINVAL, "nu_mask_transits: need n_t0, n_D >= 1");
    if (prec != NU_FP64 && prec != NU_MIXED)
        return fail(NU_EINVAL, "nu_mask_transits: unknown precision");
    if (!(P > 0.0) || !std::isfinite(P) || !std::isfinite(T0) || !std::isfinite(half_width))
        return fail(NU_EINVAL, "nu_mask_transits: P must be finite and > 0, T0 and "
                               "half_width finite");
    cudaStream_t st = (cudaStream_t)stream;
    if (prec == NU_FP64)
        k_mask_transits<double><<<div_up(n_t0, 256), 256, 0, st>>>(
            t0s_dev, n_t0, n_D, (double*)depth_dev, (double*)var_dev, (double*)dlnl_dev, P, T0,
            half_width);
    else
        k_mask_transits<float><<<div_up(n_t0, 256), 256, 0, st>>>(
            t0s_dev, n_t0, n_D, (float*)depth_dev, (float*)var_dev, (float*)dlnl_dev, P, T0,
            half_width);
    count_launches(1);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "nu_mask_transits: launch");
    return NU_OK;
}

// ------------------------------------------------ rotation-alias periods
// One block walks the grid in tiles of its threads; a period is dropped when
// dP = P / P_star is within tol below its ceiling (or, symmetric, of its
// nearest integer), each operation rounded once; the kept periods are written
// in input order (warp ballots, then the warps' counts in shared memory).
__global__ void __launch_bounds__(1024)
k_alias_filter(const double* __restrict__ P, int64_t n_P, double P_star, double tol,
               int symmetric, double* __restrict__ kept, int64_t* __restrict__ n_kept) {
    __shared__ int warp_cnt[32];
    __shared__ int64_t base;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int n_warps = blockDim.x >> 5;
    if (threadIdx.x == 0) base = 0;
    __syncthreads();
    for (int64_t t0 = 0; t0 < n_P; t0 += blockDim.x) {
        const int64_t i = t0 + threadIdx.x;
        bool keep = false;
        double p = 0.0;
        if (i < n_P) {
            p = P[i];
            const double dP = __ddiv_rn(p, P_star);
            const double ref = symmetric ? rint(dP) : ceil(dP);
            keep = !(fabs(__dsub_rn(dP, ref)) < tol);
        }
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (lane == 0) warp_cnt[wid] = __popc(m);
        __syncthreads();
        int before = 0, total = 0;
        for (int w = 0; w < n_warps; ++w) {
            const int c = warp_cnt[w];
            if (w < wid) before += c;
            total += c;
        }
        if (keep) kept[base + before + __popc(m & ((1u << lane) - 1u))] = p;
        __syncthreads();
        if (threadIdx.x == 0) base += total;
        __syncthreads();
    }
    if (threadIdx.x == 0) *n_kept = base;
}

extern "C" nu_status nu_rotation_alias_filter(const double* periods_dev, int64_t n_P,
                                              double P_star, double tol, int symmetric,
                                              double* kept_dev, int64_t* n_kept_dev,
                                              void* stream) {
    if (!periods_dev || !kept_dev || !n_kept_dev)
        return fail(NU_EINVAL, "nu_rotation_alias_filter: null array");
    if (n_P < 1) return fail(NU_EINVAL, "nu_rotation_alias_filter: n_P must be >= 1");
    if (!(P_star > 0.0) || !std::isfinite(P_star) || !(tol >= 0.0) || !std::isfinite(tol))
        return fail(NU_EINVAL, "nu_rotation_alias_filter: P_star must be finite and > 0, "
                               "tol finite and >= 0");
    if (periods_dev == kept_dev)
        return fail(NU_EINVAL, "nu_rotation_alias_filter: kept must not alias periods");
    cudaStream_t st = (cudaStream_t)stream;
    k_alias_filter<<<1, 1024, 0, st>>>(periods_dev, n_P, P_star, tol, symmetric ? 1 : 0,
                                       kept_dev, n_kept_dev);
    count_launches(1);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "nu_rotation_alias_filter: launch");
    return NU_OK;
}

// ------------------------------------------------ allocation-free variant
// nu_periodic_search_noalloc runs the same kernels as nu_periodic_search but
// takes its scratch (epoch records, bucket table, slot table, flag) from the
// file-scope device array below instead of the stream-ordered pool, for
// callers that must not allocate device memory (it creates no stream and no
// event either: the block items run before the others, on the call's stream).
// The array is part of the
// library image: every GPU that loads the library holds it until the process
// exits.  Its address is looked up once per device (cudaGetSymbolAddress with
// that device current) on the first call made on the device.
#define NU_NOALLOC_SCRATCH_BYTES (32ull << 20)

static __device__ __align__(256) unsigned char g_fold_scratch[NU_NOALLOC_SCRATCH_BYTES];

namespace {
std::mutex g_scratch_mu;
void* g_scratch_ptr[64] = {};
}

// The scratch of the device that runs the call: the stream's device, which
// must be the current device (the symbol lookup and the launches use the
// current device) and must hold the epochs.
static nu_status noalloc_scratch(cudaStream_t st, const void* t0s_dev, void** out) {
    int dev = 0, sdev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return cuda_fail(e, "nu_periodic_search_noalloc: cudaGetDevice");
    e = cudaStreamGetDevice(st, &sdev);
    if (e != cudaSuccess) return cuda_fail(e, "nu_periodic_search_noalloc: cudaStreamGetDevice");
    if (sdev != dev)
        return fail(NU_EINVAL, "nu_periodic_search_noalloc: the stream belongs to device %d but "
                               "device %d is current; make the stream's device current", sdev,
                    dev);
    cudaPointerAttributes pa;
    e = cudaPointerGetAttributes(&pa, t0s_dev);
    if (e != cudaSuccess)
        return cuda_fail(e, "nu_periodic_search_noalloc: cudaPointerGetAttributes");
    if (pa.type == cudaMemoryTypeDevice && pa.device != dev)
        return fail(NU_EINVAL, "nu_periodic_search_noalloc: t0s is on device %d, the call runs "
                               "on device %d", pa.device, dev);
    if (dev < 0 || dev >= 64)
        return fail(NU_EINVAL, "nu_periodic_search_noalloc: device index %d out of range", dev);
    std::lock_guard<std::mutex> lock(g_scratch_mu);
    if (!g_scratch_ptr[dev]) {
        void* p = nullptr;
        e = cudaGetSymbolAddress(&p, g_fold_scratch);
        if (e != cudaSuccess || !p)
            return cuda_fail(e, "nu_periodic_search_noalloc: cudaGetSymbolAddress");
        g_scratch_ptr[dev] = p;
    }
    *out = g_scratch_ptr[dev];
    return NU_OK;
}

extern "C" uint64_t nu_periodic_search_noalloc_limit(void) { return NU_NOALLOC_SCRATCH_BYTES; }

extern "C" nu_status nu_periodic_search_noalloc(const double* t0s_dev, int64_t n_t0,
                                                const double* Ds_host, int n_D,
                                                const void* depth_dev, const void* var_dev,
                                                const void* dlnl_dev, nu_precision prec,
                                                const double* periods_dev, int64_t n_P,
                                                double phase_step, double gap_factor,
                                                void* stream, double* Q_dev, double* T0_dev,
                                                int32_t* D_idx_dev, double* depth_out_dev,
                                                double* sigma_out_dev, double* lnP_dev) {
    const char* who = "nu_periodic_search_noalloc";
    (void)Ds_host;
    nu_status s = check_args(who, t0s_dev, n_t0, n_D, depth_dev, var_dev, dlnl_dev, prec,
                             periods_dev, n_P, gap_factor, Q_dev, T0_dev, D_idx_dev,
                             depth_out_dev, sigma_out_dev, lnP_dev);
    if (s != NU_OK) return s;
    if (!(phase_step > 0.0) || !std::isfinite(phase_step))
        return fail(NU_EINVAL, "nu_periodic_search_noalloc: phase_step must be given (> 0)");
    cudaStream_t st = (cudaStream_t)stream;
    void* base = nullptr;
    s = noalloc_scratch(st, t0s_dev, &base);
    if (s != NU_OK) return s;
    double ends[2];
    cudaError_t e = cudaMemcpyAsync(&ends[0], t0s_dev, sizeof(double), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(&ends[1], t0s_dev + n_t0 - 1, sizeof(double), cudaMemcpyDeviceToHost,
                            st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return cuda_fail(e, "nu_periodic_search_noalloc: copy ends");
    const double t_ref = ends[0], t_last = ends[1];
    if (!(t_last >= t_ref)) return fail(NU_EINVAL, "nu_periodic_search_noalloc: t0s not sorted");
    const double span_steps = (t_last - t_ref) / phase_step;
    if (span_steps > 1.0e9)
        return fail(NU_EINVAL, "nu_periodic_search_noalloc: phase grid too fine");
    const FoldCall C{who, t0s_dev, n_t0, n_D, depth_dev, var_dev, dlnl_dev, prec == NU_FP64,
                     periods_dev, n_P, phase_step, gap_factor, t_ref, t_last,
                     (int64_t)span_steps + 2, st, false, Q_dev, T0_dev, D_idx_dev, depth_out_dev,
                     sigma_out_dev, lnP_dev};
    // the best plan that fits, of either kind of records
    auto fit = [&](bool slots) {
        SingleLayout L{};
        for (const FoldPlan& plan : fold_plans(C, slots)) {
            L = single_layout(C, plan);
            if (L.total <= NU_NOALLOC_SCRATCH_BYTES) break;
        }
        return L;
    };
    const SingleLayout Le = fit(false);
    const SingleLayout Ls = C.may_use_slots() ? fit(true) : SingleLayout{};
    const size_t need = std::max(Le.total, Ls.total);
    if (need > NU_NOALLOC_SCRATCH_BYTES)
        return fail(NU_EINVAL,
                    "nu_periodic_search_noalloc: this grid needs %zu bytes of scratch, more "
                    "than the fixed %llu bytes; use nu_periodic_search",
                    need, (unsigned long long)NU_NOALLOC_SCRATCH_BYTES);
    return single_fold(C, (char*)base, C.may_use_slots() ? &Ls : nullptr, Le);
}
