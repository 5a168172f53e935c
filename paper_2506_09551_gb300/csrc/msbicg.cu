// Multi-shifted BiCG on the device (App. C; Alg. 1 in corrected form).
//
// Systems (A - s_k I) x_k = b, A complex symmetric (A = H' - E_G - i Gamma
// - w_seed in the RIXS map).  One seed recurrence on A, shared by all shifts:
//
//   v = A p_m; mu = (p_m, v); alpha_m = rho_m / mu           (MVM, bilinear product)
//   zeta^k_{m+1} = (1 - alpha_m s_k) zeta^k_m
//                  + (alpha_m beta_m / alpha_{m-1}) (zeta^k_m - zeta^k_{m-1})        (Eq. 5, sign fixed)
//   r_{m+1} = r_m - alpha_m v; rho_{m+1} = (r_{m+1}, r_{m+1}); beta_{m+1} = rho_{m+1}/rho_m
//   p_{m+1} = r_{m+1} + beta_{m+1} p_m
//
// (.,.) is the bilinear product sum u_i v_i (App. A: the dual residual is
// conj(r), so the BiCG conditions need no conjugation).  beta_m is the
// coefficient that built p_m (App. C convention).
//
// Per shift (Eqs. 6-8), with the search direction stored rescaled as
// P^k_m = zeta^k_m p^k_m so that no 1/zeta multiply touches the vectors:
//   p^k_m = r_m / zeta^k_m + beta^k_m p^k_{m-1},  beta^k_m = (zeta^k_{m-1}/zeta^k_m)^2 beta_m
//     =>  P^k_m = r_m + gamma^k_m P^k_{m-1},      gamma^k_m = beta_m zeta^k_{m-1} / zeta^k_m
//   x^k_{m+1} = x^k_m + alpha^k_m p^k_m,           alpha^k_m = (zeta^k_m / zeta^k_{m+1}) alpha_m
//     =>  x^k_{m+1} = x^k_m + c^k_m P^k_m,         c^k_m = alpha_m / zeta^k_{m+1}
// A shift is frozen when ||r_{m+1}|| / |zeta^k_{m+1}| <= tol ||b|| (Eq. 4).
//
// Lagged fused update (the GB300 layout of Eqs. 7-8): the scalars gamma, c
// of a window of W consecutive iterations (56 in FP64, 32 in FP32) are kept per
// shift, the seed residuals r_{m0..m0+W-1} are kept in a ring, and one kernel then
// advances P^k and x^k over the window: one read and one write of each per-shift
// vector per W iterations.  FP32, and FP64 with few shifts: the recurrence in
// registers, its arithmetic and order exactly those of the per-iteration update.
// FP64 with more shifts: one contraction on the tensor cores (flush_tc.cuh).
//
// Exponent management.  The seed residual of a well-placed seed falls far
// faster than the residuals of distant shifts (1e-160 after ~1000 iterations
// at L = 8), so r_m and zeta^k_m leave the FP32 range long before the shifts
// converge, and the FP64 range on long runs.  Everything is linear, so the
// seed vectors r, p, v are stored as S_m times their true values (S_0 brings a right-hand side
// beyond 2^+-300 near one, so that rho, 1 / rho and the squares stay normal numbers) and each
// shift's (zeta_m, zeta_{m-1}) as g_k times theirs, with S_m and g_k powers of
// two (exact scaling: no rounding changes).  Only the scalars see the scales:
//   gamma~ = gamma * S_m / S_{m-1},   c~ = c / S_m = alpha 2^{E_k} / zeta~_{m+1},
//   ||r^k_m|| = ||r~_m|| 2^{E_k} / |zeta~_m|,      E_k = log2(g_k / S_m).
#include <chrono>
#include <cmath>
#include <memory>

#include "flush_tc.cuh"
#include "hubrows.cuh"
#include "kernels.cuh"
#include "msbicg_impl.cuh"
#include "profile.cuh"

namespace msb {

constexpr int kScalarThreads = 256;
constexpr int kVecThreads = 256;      // vector kernels of the iteration, three CTAs per SM

// ---------------------------------------------------------------------------
// Device state
// ---------------------------------------------------------------------------
struct SeedState {
    double2 rho;          // rho_m = (r_m, r_m)
    double2 alpha;        // alpha_m of the current iteration
    double2 beta;         // beta_m: built p_m (0 at m = 0)
    double2 beta_n, rho_n;   // beta_{m+1}, (r~_{m+1}, r~_{m+1}) before the rescale
    double rn2_n;         // ||r~_{m+1}||^2
    double2 irho;         // 1 / rho_m
    double2 boa;          // beta_m / alpha_{m-1}
    int f_n, bad_n;       // its rescale exponent; why beta could not be formed
    unsigned cnt_a, cnt_b;   // arrival counters of the two reductions
    unsigned bar_w, bar_a;   // k_window: arrivals of its workers, and of all its CTAs
    double2 alpha_w[2];      // k_window: alpha of even and odd iterations, from CTA 0
    int stop_at;             // k_window: iteration of the window at which the recurrence ended
    double rnorm;         // ||r_m||
    double bnorm;         // ||b||
    double ibnorm;        // 1 / ||b|| (0 for b = 0)
    double ir0;           // 1 / ||r~_0||
    int f0;               // log2 S_0: r~_0 = 2^f0 b
    double tol;
    int m;                // iteration count
    int m0;               // iteration at the start of the current block
    int j;                // iterations in the current block
    int jcur;             // j at the start of the iteration
    int slot0;            // ring slot holding r_{m0}
    int stop;             // the recurrence ended (set by k_update_p)
    int halted;           // copy of `stop` made by the product kernel, read by the two after it
    int bad;              // alpha could not be formed
    int status;           // msb_status of the recurrence
    int maxit;
    int nactive;
    int fexp;             // r~_m, p~_m were rescaled by 2^fexp after r_m was formed
    int sexp;             // log2 S_m (for reporting the true seed residual)
    int flush_J, flush_cnt, flush_first;   // work of the last fused update (profiling)
    int rexp[kTcWindow + 1];               // per ring slot: exponent of the stored ||r~||
};

// ---------------------------------------------------------------------------
// One iteration is three launches (four in the dual form), since the sums that alpha
// and beta need close over the whole vector:
//   the product      v = A p; its last CTA to finish: mu, alpha
//   k_seed_update    r_{m+1} = r_m - alpha v; its last CTA: rho, the norm, beta
//   k_update_p       p_{m+1} = r_{m+1} + beta p_m
// CTA 0 of the two vector kernels does the per-shift scalars meanwhile.  A kernel never
// writes a state field that its other CTAs read (`halted`, `jcur`, `beta_n` and the
// like are written one launch before they are read).  After the recurrence has ended
// all of them return at once.  FP64 scalar work is left to one thread or one warp: the
// FP64 pipe spends 16 cycles on a warp's instruction, so a division by every warp of
// every CTA costs more than the vectors (measured: alpha and beta formed by each CTA,
// 85 us for the two vector kernels at L = 12, as much as with separate scalar kernels).
// ---------------------------------------------------------------------------

// x 2^n, exact while the result is a normal number.
__device__ __forceinline__ double scale2(double x, int n) {
    return n > -1022 && n < 1023 ? x * __hiloint2double((1023 + n) << 20, 0) : ldexp(x, n);
}
__device__ __forceinline__ double2 scale2(double2 v, int n) { return make_double2(scale2(v.x, n), scale2(v.y, n)); }

// alpha_m = rho_m / mu; why it could not be formed, else MSB_OK.
__device__ __forceinline__ int form_alpha(double2 mu, double2 rho, double2& a) {
    a = make_double2(0.0, 0.0);
    if (!cfinite(mu)) return MSB_ENONFINITE;
    if (mu.x == 0.0 && mu.y == 0.0) return MSB_EBREAKDOWN;
    a = cdiv1(rho, mu);
    return cfinite(a) ? MSB_OK : MSB_ENONFINITE;
}

// beta_{m+1} = rho_{m+1} / rho_m and the exponent f of the rescale, from the sums (rho_{m+1},
// ||r_{m+1}||^2); why it could not be formed, else MSB_OK.  irho = 1 / rho_m was formed beside the
// vectors, off the chain (a division here: 2% of the L = 8 solve).
__device__ __forceinline__ int form_beta(const double (&v)[3], double2 irho, double ir0, double2& b, int& f) {
    b = make_double2(0.0, 0.0);
    f = 0;
    if (!isfinite(v[0]) || !isfinite(v[1]) || !isfinite(v[2])) return MSB_ENONFINITE;
    if (v[2] == 0.0) return MSB_OK;                         // exact solution: every shift converged
    if (v[0] == 0.0 && v[1] == 0.0) return MSB_EBREAKDOWN;  // (r, r) = 0 with r != 0
    b = cmul(make_double2(v[0], v[1]), irho);
    // bring ||r~|| back near ||r~_0|| once it drifts by more than 2^20
    const double ratio2 = v[2] * ir0 * ir0;
    if (ratio2 < 0x1p-40 || ratio2 > 0x1p40) f = -(ilogb(ratio2) >> 1);
    return MSB_OK;
}

// First thread block of the product kernel: the iteration's copy of `stop`.
__device__ __forceinline__ bool mvm_halted(SeedState* st) {
    const int h = st->stop;
    if (blockIdx.x == 0 && threadIdx.x == 0) st->halted = h;
    return h != 0;
}

// End of the product kernel: partial mu, and alpha_m from all of them in the last CTA.
// sm: 2 * blockDim.x doubles.
__device__ __forceinline__ void mvm_finish(double (&acc)[2], double* sm, double* part, SeedState* st) {
    block_sum_sm<2>(acc, sm);
    if (threadIdx.x == 0) {
        part[2 * int64_t(blockIdx.x)] = acc[0];
        part[2 * int64_t(blockIdx.x) + 1] = acc[1];
    }
    if (!last_cta(&st->cnt_a, gridDim.x)) return;
    double mu[2];
    sum_partials_cg<2>(part, gridDim.x, mu, sm);
    if (threadIdx.x == 0) {
        double2 a;
        const int bad = form_alpha(make_double2(mu[0], mu[1]), st->rho, a);
        if (bad) st->status = bad;
        st->bad = bad;
        st->alpha = a;
        st->jcur = st->j;
    }
}

// v = A p (A = op + c0), partial mu = (p, v).
// Dual form (pt != null, App. A): mu = <p~|v> (Hermitian) instead of (p, v).
template <class View, typename V>
__global__ void __launch_bounds__(256) k_mvm_dot(View op, const V* __restrict__ p, V* __restrict__ v,
                                                 int64_t n, double c0r, double c0i,
                                                 SeedState* __restrict__ st, double* part,
                                                 const V* __restrict__ pt) {
    if (mvm_halted(st)) return;
    __shared__ double sm[2 * 256];
    double acc[2] = {0.0, 0.0};
    DF4 df;
    for (int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; s < n;
         s += int64_t(gridDim.x) * blockDim.x) {
        const V ps = p[s];
        const V h = op.hx(s, p, ps);
        const V vs = vadd(h, cscale(c0r, c0i, ps));
        v[s] = vs;
        if (pt) {
            if constexpr (std::is_same<V, float2>::value) her_acc_df(pt[s], vs, df);
            else her_acc(pt[s], vs, acc[0], acc[1]);
        } else {
            if constexpr (std::is_same<V, float2>::value) bil_acc_df(ps, vs, df);
            else bil_acc(ps, vs, acc[0], acc[1]);
        }
    }
    if constexpr (std::is_same<V, float2>::value) {
        acc[0] = df_value(df.rh, df.rl);
        acc[1] = df_value(df.ih, df.il);
    }
    mvm_finish(acc, sm, part, st);
}

// The same as the epilogue of the row-tiled Hubbard product (hubrows.cuh).
template <typename V>
struct MvmEpi {
    V* v;
    SeedState* st;
    double* part;
    const V* pt;
    scalar_t<V> c0r, c0i;
    double acc[2];
    DF4 df;
    __device__ __forceinline__ bool stop() const { return mvm_halted(st); }
    __device__ __forceinline__ void begin(int) {}
    __device__ __forceinline__ void term(int64_t s, V ps, V vs) {
        if constexpr (std::is_same<V, float2>::value) {
            if (pt) her_acc_df(pt[s], vs, df);
            else bil_acc_df(ps, vs, df);
        } else {
            if (pt) her_acc(pt[s], vs, acc[0], acc[1]);
            else bil_acc(ps, vs, acc[0], acc[1]);
        }
    }
    template <typename S>
    __device__ __forceinline__ void operator()(int64_t s, V xs, V a, S dg, S mt, S shift) {
        const V h = hub_value(a, dg, mt, shift, c0r, c0i, xs);
        v[s] = h;
        term(s, xs, h);
    }
    __device__ __forceinline__ void pair(int64_t s, float2 xa, float2 xb, float2 a, float2 b, float da, float db,
                                         float mt, float shift) {
        const float2 p = hub_value(a, da, mt, shift, c0r, c0i, xa), q = hub_value(b, db, mt, shift, c0r, c0i, xb);
        *reinterpret_cast<float4*>(v + s) = make_float4(p.x, p.y, q.x, q.y);
        term(s, xa, p);
        term(s + 1, xb, q);
    }
    __device__ __forceinline__ void finish(double* sm) {
        if constexpr (std::is_same<V, float2>::value) {
            acc[0] = df_value(df.rh, df.rl);
            acc[1] = df_value(df.ih, df.il);
        }
        mvm_finish(acc, sm, part, st);
    }
};

// Dual-space product v~ = (A + c0*) p~ = (A + c0)^dagger p~ for Hermitian A (App. A).
template <class View, typename V>
__global__ void __launch_bounds__(256) k_dual_mvm(View op, const V* __restrict__ pt, V* __restrict__ vt, int64_t n,
                                                  double c0r, double c0i, const SeedState* __restrict__ st) {
    if (st->halted) return;
    for (int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; s < n; s += int64_t(gridDim.x) * blockDim.x) {
        const V ps = pt[s];
        vt[s] = vadd(op.hx(s, pt, ps), cscale(c0r, -c0i, ps));
    }
}

// Every active shift's zeta / gamma / c for block position j (one CTA).
template <typename C>
__device__ __forceinline__ void shift_scalars_a(SeedState* st, double2 alpha, const ShiftArrays& sh, int ns, int B) {
    if (threadIdx.x >= ns) return;
    const double2 beta = st->beta;
    const double2 ab_over = cmul(alpha, st->boa);                       // alpha_m beta_m / alpha_{m-1}
    const int j = st->j;
    const int fexp = st->fexp;
    for (int k = threadIdx.x; k < ns; k += blockDim.x) {
        if (!sh.active[k]) continue;
        const double2 z = sh.zeta[k], zp = sh.zeta_prev[k], s = sh.shift[k];
        const int ze = sh.zexp[k];
        // (1 - alpha s) z + (alpha beta / alpha_prev)(z - zp)
        const double2 one_m = make_double2(1.0 - (alpha.x * s.x - alpha.y * s.y), -(alpha.x * s.y + alpha.y * s.x));
        const double2 zn = cadd(cmul(one_m, z), cmul(ab_over, csub(z, zp)));
        if (!(zn.x != 0.0 || zn.y != 0.0) || !cfinite(zn)) {
            // shift breakdown: freeze it, not converged
            sh.active[k] = 0;
            sh.broken[k] = 1;
            continue;
        }
        // beta_m zeta_{m-1} / zeta_m, times S_m / S_{m-1}
        const double2 gamma = scale2(cmul(cmul(beta, zp), sh.izeta[k]), fexp);
        // alpha_m / zeta_{m+1} / S_m
        const double2 izn = cdiv1(make_double2(1.0, 0.0), zn);
        const double2 c = scale2(cmul(alpha, izn), ze);
        const int64_t o = int64_t(k) * B + j;
        sh.coef64[2 * o] = gamma;
        sh.coef64[2 * o + 1] = c;
        reinterpret_cast<C*>(sh.coefv)[2 * o] = from_d2<C>(gamma);
        reinterpret_cast<C*>(sh.coefv)[2 * o + 1] = from_d2<C>(c);
        sh.nblk[k] = j + 1;
        // keep zeta~ near 1: rescale the pair (zeta_{m+1}, zeta_m) by 2^q
        const double mag = fmax(fabs(zn.x), fabs(zn.y));
        int q = 0;
        if (mag < 0x1p-30 || mag > 0x1p30) q = -ilogb(mag);
        sh.zeta_prev[k] = scale2(z, q);
        sh.zeta[k] = scale2(zn, q);
        sh.izeta[k] = scale2(izn, -q);
        sh.zexp[k] = ze + q;
    }
}

// Sums over residual elements: rho = sum (x.x - y.y) + 2 i sum x.y and ||r||^2 = Re rho + 2 sum y.y,
// four products per element where rho and the norm separately take six.  Re rho is summed term by
// term: a difference of sum x.x and sum y.y would be rounded at the size of ||r||^2, which loses
// rho when the residual is close to isotropic.
struct ResSum {
    double re = 0.0, yy = 0.0, xy = 0.0;
    __device__ __forceinline__ void add(double2 r) {
        re = fma(r.x, r.x, fma(-r.y, r.y, re));
        yy = fma(r.y, r.y, yy);
        xy = fma(r.x, r.y, xy);
    }
    __device__ __forceinline__ void get(double (&a)[3]) const { a[0] = re; a[1] = 2.0 * xy; a[2] = fma(2.0, yy, re); }
};
struct ResSumF {
    float rh = 0.f, rl = 0.f, yh = 0.f, yl = 0.f, ch = 0.f, cl = 0.f;
    __device__ __forceinline__ void add(float2 r) {
        df_add_prod(rh, rl, r.x, r.x);
        df_add_prod(rh, rl, -r.y, r.y);
        df_add_prod(yh, yl, r.y, r.y);
        df_add_prod(ch, cl, r.x, r.y);
    }
    __device__ __forceinline__ void get(double (&a)[3]) const {
        a[0] = df_value(rh, rl);
        a[1] = 2.0 * df_value(ch, cl);
        a[2] = fma(2.0, df_value(yh, yl), a[0]);
    }
};
template <typename V> using res_sum_t = typename std::conditional<std::is_same<V, float2>::value, ResSumF, ResSum>::type;

// r + sg (c v), sg = +-1, the product rounded before it is added.
__device__ __forceinline__ float2 axpy_rn(float2 r, float2 c, float2 v, float sg) {
    const float2 t = cscale_rn(c.x, c.y, v);
    return make_float2(__fmaf_rn(sg, t.x, r.x), __fmaf_rn(sg, t.y, r.y));
}

// r_{m+1} = r_m - alpha v (into the next ring slot; slots ld elements apart, ld even);
// partials of rho and ||r||^2.  CTA 0: the per-shift scalars.
// Dual form (rt != null): also r~ <- r~ - conj(alpha) v~, and rho = <r~|r> (Hermitian).
// Bound by memory (three vectors; L2 while they fit); 16-byte accesses, two elements
// per access in FP32, two accesses in flight per vector.
template <typename V>
__global__ void __launch_bounds__(kVecThreads, 3) k_seed_update(V* ring, int64_t ld, const V* __restrict__ v, int64_t n,
                                                             int nslot, SeedState* __restrict__ st, double* part,
                                                             V* __restrict__ rt, const V* __restrict__ vt,
                                                             ShiftArrays sh, int ns, int B) {
    if (st->halted || st->bad) return;
    const double2 a = st->alpha;
    if (blockIdx.x == 0) {
        shift_scalars_a<V>(st, a, sh, ns, B);
        return;
    }
    __shared__ double sm[3 * kVecThreads];
    const int cur = (st->slot0 + st->jcur) % nslot, nxt = (cur + 1) % nslot;
    const V* __restrict__ r = ring + int64_t(cur) * ld;
    V* __restrict__ rn = ring + int64_t(nxt) * ld;
    const int64_t nth = int64_t(gridDim.x - 1) * blockDim.x, t0 = int64_t(blockIdx.x - 1) * blockDim.x + threadIdx.x;
    double acc[3] = {0.0, 0.0, 0.0};
    if (rt) {
        DF4 df;
        for (int64_t s = t0; s < n; s += nth) {
            const V x = vsub(r[s], cscale(a.x, a.y, v[s]));
            rn[s] = x;
            const V y = vsub(rt[s], cscale(a.x, -a.y, vt[s]));
            rt[s] = y;
            if constexpr (std::is_same<V, float2>::value) {
                her_acc_df(y, x, df);
                norm_acc_df(x, df);
            } else {
                her_acc(y, x, acc[0], acc[1]);
                acc[2] += norm2(x);
            }
        }
        if constexpr (std::is_same<V, float2>::value) {
            acc[0] = df_value(df.rh, df.rl);
            acc[1] = df_value(df.ih, df.il);
            acc[2] = df_value(df.nh, df.nl);
        }
    } else {
        res_sum_t<V> sum;
        if constexpr (std::is_same<V, float2>::value) {
            const int64_t h = n >> 1;
            const float2 af = from_d2<float2>(a);
            const float4* __restrict__ r4 = reinterpret_cast<const float4*>(r);
            const float4* __restrict__ v4 = reinterpret_cast<const float4*>(v);
            float4* __restrict__ o4 = reinterpret_cast<float4*>(rn);
            auto one = [&](int64_t i, float4 x, float4 w) {
                const float2 p = axpy_rn(make_float2(x.x, x.y), af, make_float2(w.x, w.y), -1.f);
                const float2 q = axpy_rn(make_float2(x.z, x.w), af, make_float2(w.z, w.w), -1.f);
                o4[i] = make_float4(p.x, p.y, q.x, q.y);
                sum.add(p);
                sum.add(q);
            };
            int64_t i = t0;
            for (; i + nth < h; i += 2 * nth) {
                const float4 x0 = r4[i], w0 = v4[i], x1 = r4[i + nth], w1 = v4[i + nth];
                one(i, x0, w0);
                one(i + nth, x1, w1);
            }
            if (i < h) one(i, r4[i], v4[i]);
            if ((n & 1) && t0 == 0) {
                const float2 x = axpy_rn(r[n - 1], af, v[n - 1], -1.f);
                rn[n - 1] = x;
                sum.add(x);
            }
        } else {
            const V na = make_double2(-a.x, -a.y);
            int64_t i = t0;
            for (; i + nth < n; i += 2 * nth) {
                const V x0 = r[i], w0 = v[i], x1 = r[i + nth], w1 = v[i + nth];
                const V y0 = cfma(na, w0, x0), y1 = cfma(na, w1, x1);
                rn[i] = y0;
                rn[i + nth] = y1;
                sum.add(y0);
                sum.add(y1);
            }
            if (i < n) {
                const V y0 = cfma(na, v[i], r[i]);
                rn[i] = y0;
                sum.add(y0);
            }
        }
        sum.get(acc);
    }
    block_sum_sm<3>(acc, sm);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int i = 0; i < 3; ++i) part[int64_t(blockIdx.x - 1) * 3 + i] = acc[i];
    }
    if (!last_cta(&st->cnt_b, gridDim.x - 1)) return;
    sum_partials_cg<3>(part, gridDim.x - 1, acc, sm);
    if (threadIdx.x == 0) {
        double2 b;
        int f;
        const int bad = form_beta(acc, st->irho, st->ir0, b, f);
        st->beta_n = b;
        st->rho_n = make_double2(acc[0], acc[1]);
        st->rn2_n = acc[2];
        st->f_n = f;
        st->bad_n = bad;
    }
}

// Convergence of every shift, iteration bookkeeping (one CTA).
// fz_coef is the factor from the stored r~_{m+1} (rescaled by 2^f) to each tested
// shift's recursive residual.
__device__ __forceinline__ void shift_scalars_b(SeedState* st, const ShiftArrays& sh, int ns, int nslot, int* s_still) {
    const int m = st->m + 1, f = st->f_n, bad = st->bad_n;
    const double rn = sqrt(st->rn2_n);
    if (threadIdx.x == 0) *s_still = 0;
    __syncthreads();
    if (threadIdx.x < ns) {
        const double thr = st->tol * st->bnorm, ib = st->ibnorm;
        int still = 0;
        for (int k = threadIdx.x; k < ns; k += blockDim.x) {
            if (!sh.active[k]) continue;
            // ||r^k_{m+1}|| = ||r~_{m+1}|| 2^{E_k} / |zeta~_{m+1}|
            const int ze = sh.zexp[k];
            const double2 iz = sh.izeta[k];
            const double rk = scale2(rn * sqrt(fma(iz.x, iz.x, iz.y * iz.y)), ze);
            sh.iters[k] = m;
            sh.resid[k] = rk * ib;
            sh.fz_coef[k] = scale2(iz, ze - f);
            sh.fz_iter[k] = m;
            sh.zexp[k] = ze - f;                           // S_{m+1} = S_m 2^f
            if (rk <= thr) { sh.active[k] = 0; sh.conv[k] = 1; }
            else ++still;
        }
        if (still) atomicAdd(s_still, still);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        st->m = m;
        st->j = st->jcur + 1;
        st->rexp[(st->slot0 + st->jcur + 1) % nslot] = rn > 0.0 && isfinite(rn) ? ilogb(rn) + f : 0;
        st->boa = cdiv1(st->beta_n, st->alpha);
        st->beta = st->beta_n;
        st->rnorm = scale2(rn, -st->sexp);
        st->fexp = f;
        st->sexp += f;
        st->nactive = *s_still;
        if (bad) st->status = bad;
        if (bad || *s_still == 0 || m >= st->maxit) st->stop = 1;
    } else if (threadIdx.x == 32) {
        // the divisions of the next iteration's scalars: off its critical path, beside each other
        const double2 rho = scale2(st->rho_n, 2 * f);
        st->irho = cdiv1(make_double2(1.0, 0.0), rho);
        st->rho = rho;
    }
}

// p = 2^f (r_{m+1} + beta p), r_{m+1} <- 2^f r_{m+1} (exact power-of-two rescale).
// CTA 0: the per-shift convergence tests.
// Dual form (rt != null): also p~ = 2^f (r~ + conj(beta) p~), r~ <- 2^f r~.
template <typename V>
__global__ void __launch_bounds__(kVecThreads, 3) k_update_p(V* ring, int64_t ld, V* __restrict__ p, int64_t n, int nslot,
                                                          SeedState* __restrict__ st, V* __restrict__ rt,
                                                          V* __restrict__ pt, ShiftArrays sh, int ns) {
    if (st->halted) return;
    if (blockIdx.x == 0) {
        __shared__ int s_still;
        if (st->bad) {
            if (threadIdx.x == 0) st->stop = 1;
        } else {
            shift_scalars_b(st, sh, ns, nslot, &s_still);
        }
        return;
    }
    if (st->bad || st->bad_n) return;
    const double2 b = st->beta_n;
    const int f = st->f_n;
    V* __restrict__ r = ring + int64_t((st->slot0 + st->jcur + 1) % nslot) * ld;
    const int64_t nth = int64_t(gridDim.x - 1) * blockDim.x, t0 = int64_t(blockIdx.x - 1) * blockDim.x + threadIdx.x;
    const V bv = from_d2<V>(b);
    if (f == 0 && !rt) {
        if constexpr (std::is_same<V, float2>::value) {
            const int64_t h = n >> 1;
            const float4* __restrict__ r4 = reinterpret_cast<const float4*>(r);
            float4* __restrict__ p4 = reinterpret_cast<float4*>(p);
            auto one = [&](float4 x, float4 q) {
                const float2 u = axpy_rn(make_float2(x.x, x.y), bv, make_float2(q.x, q.y), 1.f);
                const float2 w = axpy_rn(make_float2(x.z, x.w), bv, make_float2(q.z, q.w), 1.f);
                return make_float4(u.x, u.y, w.x, w.y);
            };
            int64_t i = t0;
            for (; i + nth < h; i += 2 * nth) {
                const float4 x0 = r4[i], q0 = p4[i], x1 = r4[i + nth], q1 = p4[i + nth];
                p4[i] = one(x0, q0);
                p4[i + nth] = one(x1, q1);
            }
            if (i < h) p4[i] = one(r4[i], p4[i]);
            if ((n & 1) && t0 == 0) p[n - 1] = axpy_rn(r[n - 1], bv, p[n - 1], 1.f);
        } else {
            int64_t i = t0;
            for (; i + nth < n; i += 2 * nth) {
                const V x0 = r[i], q0 = p[i], x1 = r[i + nth], q1 = p[i + nth];
                p[i] = cfma(bv, q0, x0);
                p[i + nth] = cfma(bv, q1, x1);
            }
            if (i < n) p[i] = cfma(bv, p[i], r[i]);
        }
    } else {
        const double sc = ldexp(1.0, f);
        for (int64_t s = t0; s < n; s += nth) {
            const V rs = r[s];
            p[s] = cscale(sc, 0.0, vadd(rs, cscale(b.x, b.y, p[s])));
            if (f != 0) r[s] = cscale(sc, 0.0, rs);
            if (rt) {
                const V ts = rt[s];
                pt[s] = cscale(sc, 0.0, vadd(ts, cscale(b.x, -b.y, pt[s])));
                if (f != 0) rt[s] = cscale(sc, 0.0, ts);
            }
        }
    }
}

// Start of a block of iterations: nothing pending for any shift.
__global__ void k_block_begin(SeedState* st, ShiftArrays sh, int ns, int nslot) {
    for (int k = threadIdx.x; k < ns; k += blockDim.x) sh.nblk[k] = 0;
    if (threadIdx.x == 0) {
        st->slot0 = (st->slot0 + st->j) % nslot;
        st->m0 = st->m;
        st->j = 0;
        st->bar_w = 0;
        st->bar_a = 0;
        st->stop_at = INT_MAX;
    }
}

// ---------------------------------------------------------------------------
// Short vectors: a whole window of iterations in one cooperative launch.
//
// With the vectors of an iteration in a few microseconds' reach of the chip, three dependent
// launches, their fences and the serial scalar work between them decide: 29 us per iteration
// on the L = 8 ring (n = 3,920), 14.5 here.  The CTAs of one launch keep r, p and v of their elements
// in registers for the whole window and meet at barriers in global memory (three per
// iteration): only p (for the gathers of the product, through L2), the residuals for the
// window's per-shift update and the partial sums leave the SM.  Every worker CTA forms alpha
// and beta from all partial sums itself.  The per-shift scalars, as long a chain as the vector
// work, run in a CTA of their own (the last) one iteration behind: after the barrier of
// iteration j it updates the shifts for j while the workers go on to j + 1.  If the recurrence
// ended at j, the workers' iteration j + 1 is not counted and nothing reads its vectors.
//
// Waits.  A worker arrives at and waits for bar_w after its part of mu and after its p;
// everybody does at bar_a after the part of rho, the scalar CTA once it has finished the
// iteration before.  Every worker takes every break from the same sums, or from stop_at < j,
// which the scalar CTA writes before its arrival for iteration stop_at + 1: all leave at the
// same iteration.  The launch is cooperative (all CTAs resident) and every wait is bounded.
// ---------------------------------------------------------------------------
constexpr int kWaitPolls = 1 << 24;       // about ten seconds

// Loads and stores that other SMs' barrier partners see (L2), never merged or moved by the compiler.
__device__ __forceinline__ double2 load_l2(const double2* p) {
    double2 v;
    asm volatile("ld.global.cg.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ float2 load_l2(const float2* p) {
    float2 v;
    asm volatile("ld.global.cg.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ double load_l2(const double* p) {
    double v;
    asm volatile("ld.global.cg.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ int load_l2(const int* p) {
    int v;
    asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void bar_arrive(unsigned* c) {
    __threadfence();
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" : : "l"(c) : "memory");
}
__device__ __forceinline__ bool bar_wait(const unsigned* c, unsigned target) {
    for (int i = 0; i < kWaitPolls; ++i) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(c) : "memory");
        if (v >= target) return true;
    }
    return false;
}

// ((A + c0) x)[s] with x read through L2, four hops in flight; rounded as in the launch-per-product
// form (hub_value, k_mvm_dot).
template <typename V>
__device__ __forceinline__ V gather_ax(const HubView& h, int64_t s, const V* x, V xs, double c0r, double c0i) {
    using S = scalar_t<V>;
    const uint32_t iu = uint32_t(s) / uint32_t(h.Ddn), id = uint32_t(s) - iu * uint32_t(h.Ddn);
    auto hops = [&](V acc, const int32_t* tab, int cnt, int64_t D, int64_t i, int64_t mul, const V* base) {
        for (int e = 0; e < cnt; e += 4) {
            int32_t t[4];
            V v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) t[q] = e + q < cnt ? __ldg(tab + int64_t(e + q) * D + i) : -1;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (t[q] >= 0) v[q] = load_l2(base + int64_t(t[q] >> 1) * mul);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (t[q] >= 0) acc = vhop(acc, t[q], v[q]);
        }
        return acc;
    };
    V acc = hops(vzero(xs), h.hup, __ldg(h.nup + iu), h.Dup, iu, h.Ddn, x + id);
    acc = hops(acc, h.hdn, __ldg(h.ndn + id), h.Ddn, id, 1, x + int64_t(iu) * h.Ddn);
    if (h.hup2) {
        V out = vaxpy(S(-h.t), acc, vscale(h.template diag<S>(iu, id), xs));
        acc = hops(vzero(xs), h.hup2, __ldg(h.nup2 + iu), h.Dup, iu, h.Ddn, x + id);
        acc = hops(acc, h.hdn2, __ldg(h.ndn2 + id), h.Ddn, id, 1, x + int64_t(iu) * h.Ddn);
        out = vaxpy(S(-h.t2), acc, out);
        return vadd(out, cscale(c0r, c0i, xs));
    }
    return hub_value(acc, h.template diag<S>(iu, id), S(-h.t), sizeof(S) == 8 ? S(c0r) : S(0), S(c0r), S(c0i), xs);
}
template <typename V>
__device__ __forceinline__ V gather_ax(const CsrView& m, int64_t s, const V* x, V xs, double c0r, double c0i) {
    using S = scalar_t<V>;
    V acc = vzero(xs);
    const int64_t b = __ldg(m.rowptr + s), e = __ldg(m.rowptr + s + 1);
    for (int64_t k = b; k < e; k += 4) {
        V v[4];
        S a[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            if (k + q >= e) continue;
            if constexpr (sizeof(S) == 8) a[q] = __ldg(m.val64 + k + q);
            else a[q] = __ldg(m.val32 + k + q);
            v[q] = load_l2(x + __ldg(m.col + k + q));
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (k + q < e) acc = vaxpy(a[q], v[q], acc);
    }
    return vadd(acc, cscale(c0r, c0i, xs));
}

// Sum of the G x NV partial sums of the workers, in a fixed order; every lane of one warp.
template <int NV>
__device__ __forceinline__ void window_sum(const double* part, int G, double (&v)[NV]) {
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = 0.0;
    for (int b = threadIdx.x & 31; b < G; b += 32) {
#pragma unroll
        for (int i = 0; i < NV; ++i) v[i] += load_l2(part + int64_t(b) * NV + i);
    }
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = warp_sum(v[i]);
}

// The scalar CTA's loop.
template <typename V>
__device__ void window_scalars(SeedState* st, const double* part, int G, const ShiftArrays& sh, int ns, int nslot, int W,
                               int iters) {
    __shared__ int s_still, s_end, s_stop;
    __shared__ double2 s_alpha;
    for (int j = 0; j < iters; ++j) {
        if (threadIdx.x < 32) {
            int end = 0;
            if (threadIdx.x == 0) {
                bar_arrive(&st->bar_a);
                if (!bar_wait(&st->bar_a, unsigned(j + 1) * unsigned(G + 1))) {
                    st->status = MSB_ETIMEOUT;
                    end = 1;
                } else if (const int bad = load_l2(&st->bad)) {
                    st->status = bad;
                    end = 1;
                }
            }
            end = __shfl_sync(0xffffffffu, end, 0);
            double v[3] = {0.0, 0.0, 0.0};
            if (!end) window_sum<3>(part + (2 + 3 * (j & 1)) * int64_t(G), G, v);
            if (threadIdx.x == 0) {
                s_end = end;
                if (!end) {
                    double2 b;
                    int f;
                    st->bad_n = form_beta(v, st->irho, st->ir0, b, f);
                    st->beta_n = b;
                    st->rho_n = make_double2(v[0], v[1]);
                    st->rn2_n = v[2];
                    st->f_n = f;
                    st->alpha = s_alpha = load_l2(&st->alpha_w[j & 1]);
                    st->jcur = st->j;
                } else {
                    st->stop = 1;
                }
            }
        }
        __syncthreads();
        if (s_end) return;
        shift_scalars_a<V>(st, s_alpha, sh, ns, W);
        __syncthreads();
        shift_scalars_b(st, sh, ns, nslot, &s_still);
        if (threadIdx.x == 0) {
            s_stop = st->stop;
            if (s_stop) {
                st->stop_at = j;
                bar_arrive(&st->bar_a);        // for iteration j + 1
            }
        }
        __syncthreads();
        if (s_stop) return;
    }
}

// part: 2 G doubles of mu, then twice 3 G of (rho, ||r||^2), for even and odd iterations.
template <class View, typename V, int NE>
__global__ void __launch_bounds__(256, 1) k_window(View op, V* ring, int64_t ld, V* p, int64_t n, double c0r, double c0i,
                                                   int nslot, SeedState* st, double* part, ShiftArrays sh, int ns, int W,
                                                   int iters) {
    if (st->stop) return;                      // set before this launch, or after every CTA has arrived
    constexpr bool f32 = std::is_same<V, float2>::value;
    const int G = gridDim.x - 1, b = blockIdx.x;
    if (b == G) {
        window_scalars<V>(st, part, G, sh, ns, nslot, W, iters);
        return;
    }
    __shared__ double sm[3 * 256];
    __shared__ double2 s_c;                    // alpha, then beta
    __shared__ int s_bad, s_f;
    const int tid = threadIdx.x;
    const int64_t nth = int64_t(G) * blockDim.x, t0 = int64_t(b) * blockDim.x + tid;
    const int slot0 = st->slot0;
    const double ir0 = st->ir0;
    double2 rho = st->rho, irho = st->irho;    // used by thread 0 only
    V r[NE], q[NE], v[NE];
#pragma unroll
    for (int i = 0; i < NE; ++i) {
        const int64_t s = t0 + i * nth;
        r[i] = s < n ? ring[int64_t(slot0) * ld + s] : vzero(V{});
        q[i] = s < n ? p[s] : vzero(V{});
    }
    unsigned bars = 0;                         // arrivals of the workers so far
    for (int j = 0; j < iters; ++j) {
        if (j > 0) {
            if (tid == 0) s_bad = bar_wait(&st->bar_w, bars) ? MSB_OK : MSB_ETIMEOUT;
            __syncthreads();
            if (s_bad) break;
        }
        double acc[2] = {0.0, 0.0};
        DF4 df;
#pragma unroll
        for (int i = 0; i < NE; ++i) {
            const int64_t s = t0 + i * nth;
            if (s >= n) break;
            v[i] = gather_ax(op, s, p, q[i], c0r, c0i);
            if constexpr (f32) bil_acc_df(q[i], v[i], df);
            else bil_acc(q[i], v[i], acc[0], acc[1]);
        }
        if constexpr (f32) {
            acc[0] = df_value(df.rh, df.rl);
            acc[1] = df_value(df.ih, df.il);
        }
        block_sum_sm<2>(acc, sm);
        bars += G;
        if (tid < 32) {
            bool ok = true;
            if (tid == 0) {
                part[2 * b] = acc[0];
                part[2 * b + 1] = acc[1];
                bar_arrive(&st->bar_w);
                ok = bar_wait(&st->bar_w, bars);
            }
            __syncwarp();
            double mu[2];
            window_sum<2>(part, G, mu);
            if (tid == 0) {
                double2 a;
                const int bad = ok ? form_alpha(make_double2(mu[0], mu[1]), rho, a) : int(MSB_ETIMEOUT);
                s_c = a;
                s_bad = bad;
                if (b == 0) {
                    st->alpha_w[j & 1] = a;
                    if (bad) st->bad = bad;
                }
            }
        }
        __syncthreads();
        const double2 a = s_c;
        const int bad = s_bad;
        double sums[3] = {0.0, 0.0, 0.0};
        if (!bad) {
            res_sum_t<V> rs;
            const V af = from_d2<V>(a);
#pragma unroll
            for (int i = 0; i < NE; ++i) {
                if (t0 + i * nth >= n) break;
                if constexpr (f32) r[i] = axpy_rn(r[i], af, v[i], -1.f);
                else r[i] = cfma(make_double2(-a.x, -a.y), v[i], r[i]);
                rs.add(r[i]);
            }
            rs.get(sums);
            block_sum_sm<3>(sums, sm);
        }
        if (tid < 32) {
            double* pr = part + (2 + 3 * (j & 1)) * int64_t(G);
            bool ok = true;
            if (tid == 0) {
                if (!bad) {
#pragma unroll
                    for (int i = 0; i < 3; ++i) pr[3 * int64_t(b) + i] = sums[i];
                }
                bar_arrive(&st->bar_a);
                ok = bad || bar_wait(&st->bar_a, unsigned(j + 1) * unsigned(G + 1));
            }
            __syncwarp();
            if (!bad) window_sum<3>(pr, G, sums);
            if (tid == 0) {
                double2 bt = make_double2(0.0, 0.0);
                int f = 0, e = bad;
                if (!e) e = !ok ? int(MSB_ETIMEOUT) : load_l2(&st->stop_at) < j ? int(MSB_EMAXITER) : form_beta(sums, irho, ir0, bt, f);
                s_c = bt;
                s_f = f;
                s_bad = e;
            }
        }
        __syncthreads();
        const int end = s_bad;                 // the same in every worker
        V* __restrict__ rn = ring + int64_t((slot0 + j + 1) % nslot) * ld;
        if (end) {
            // beta could not be formed: the iteration counts, and k_rrec reads its residual
            if (!bad && (end == MSB_EBREAKDOWN || end == MSB_ENONFINITE)) {
#pragma unroll
                for (int i = 0; i < NE; ++i)
                    if (t0 + i * nth < n) rn[t0 + i * nth] = r[i];
            }
            break;
        }
        const double2 beta = s_c;
        const int f = s_f;
        const V bv = from_d2<V>(beta);
        const double sc = scale2(1.0, f);
#pragma unroll
        for (int i = 0; i < NE; ++i) {
            const int64_t s = t0 + i * nth;
            if (s >= n) break;
            if constexpr (f32) q[i] = axpy_rn(r[i], bv, q[i], 1.f);
            else q[i] = cfma(bv, q[i], r[i]);
            if (f != 0) {
                q[i] = cscale(sc, 0.0, q[i]);
                r[i] = cscale(sc, 0.0, r[i]);
            }
            rn[s] = r[i];
            p[s] = q[i];
        }
        __syncthreads();
        bars += G;
        if (tid == 0 && j + 1 < iters) {
            bar_arrive(&st->bar_w);
            rho = scale2(make_double2(sums[0], sums[1]), 2 * f);
            irho = cdiv1(make_double2(1.0, 0.0), rho);
        }
    }
}

// Lagged fused per-shift update over the window's iterations (Eqs. 7-8):
// for every shift with pending iterations, P <- r_i + gamma_i P; x <- x + c_i P
// for i = 0 .. nblk[k]-1, r_i from the ring, BMAX iterations at a time with P and x in
// registers.  The order of the operations does not depend on the window.
// Optional row map: element e of the per-shift vectors is seed element
// rows[e / rowlen] * rowlen + e % rowlen (only the rows the caller needs).
// A thread carries NE elements: 2 NE FMAs per component pair share one coefficient load,
// and the NE chains cover each other's latency.  The next shift's P and x are loaded before
// the current one's arithmetic.
// FP32 (BMAX = 32: the whole window in one pass; NE = 2, the 64 residuals in registers at
// one CTA per SM): the FP32 pipe and DRAM are about balanced at 256 FMAs per 32 bytes of P
// and x.  48 shifts, n = 2.9 M, per 32 iterations: 3.4 ms as four windows of 8, 2.5 ms with
// NE = 1 (bound by the coefficient loads), 1.9 ms with NE = 2.
// Shorter windows (16 or 8 iterations, where the ring of residuals has less memory): NE = 1, two CTAs
// per SM.  Same update of 1,352 iterations: 80 ms (32), 100 ms (16), 164 ms (8).
// FP64 (BMAX = 8, NE = 1): bound by the FP64 pipe (8 FMAs per shift, element and
// iteration); windows with many shifts go to the tensor cores (flush_tc.cuh), and this
// kernel returns at once.
// (gamma, c) of one iteration, read in one access.
template <typename V>
struct __align__(16) CoefPair { V g, c; };

template <typename V, int BMAX, int NE>
__global__ void __launch_bounds__(256, NE == 1 ? 2 : 1) k_flush(const V* __restrict__ ring, int nslot, int64_t ld,
                                                                V* __restrict__ P, V* __restrict__ X, int64_t n_out,
                                                                const int32_t* __restrict__ rows, int64_t rowlen,
                                                                ShiftArrays sh, int ns, SeedState* __restrict__ st,
                                                                int W, const int* __restrict__ tc_cnt) {
    __shared__ int s_list[kMaxShifts];
    __shared__ unsigned char s_J[kMaxShifts];
    __shared__ int s_cnt;
    const bool tc = tc_cnt != nullptr && tc_use(*tc_cnt, st->bnorm);
    if (tc && blockIdx.x != 0) return;
    const int cnt = pending_list(sh.nblk, ns, 0, s_list, &s_cnt);
    const bool first = st->m0 == 0;
    const int slot0 = st->slot0, JW = st->j;                          // slot of r_{m0}
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        st->flush_J = JW;
        st->flush_cnt = cnt;
        st->flush_first = first;
    }
    if (tc || cnt == 0) return;
    for (int q = threadIdx.x; q < cnt; q += blockDim.x) s_J[q] = static_cast<unsigned char>(sh.nblk[s_list[q]]);
    __syncthreads();
    const CoefPair<V>* __restrict__ coef = reinterpret_cast<const CoefPair<V>*>(sh.coefv);
    // element u of a thread: e + u * blockDim.x (whole lines for any n_out)
    for (int64_t e = int64_t(blockIdx.x) * blockDim.x * NE + threadIdx.x; e < n_out;
         e += int64_t(gridDim.x) * blockDim.x * NE) {
        int64_t src[NE];
        bool on[NE];
#pragma unroll
        for (int u = 0; u < NE; ++u) {
            const int64_t eu = e + u * int64_t(blockDim.x);
            on[u] = eu < n_out;
            src[u] = on[u] ? eu : e;
            if (rows) {
                const int64_t row = src[u] / rowlen;
                src[u] = int64_t(__ldg(rows + row)) * rowlen + (src[u] - row * rowlen);
            }
        }
        for (int i0 = 0; i0 < JW; i0 += BMAX) {
            const bool fresh = first && i0 == 0;
            V r[NE][BMAX];
#pragma unroll
            for (int i = 0; i < BMAX; ++i) {
                const int sl = (slot0 + i0 + i) % nslot;
#pragma unroll
                for (int u = 0; u < NE; ++u) r[u][i] = (i0 + i < JW) ? ring[int64_t(sl) * ld + src[u]] : vzero(V{});
            }
            V np[NE], nx[NE];
            auto fetch = [&](int k) {
#pragma unroll
                for (int u = 0; u < NE; ++u) {
                    const int64_t o = int64_t(k) * n_out + e + u * int64_t(blockDim.x);
                    np[u] = !fresh && on[u] ? P[o] : vzero(V{});
                    nx[u] = !fresh && on[u] ? X[o] : vzero(V{});
                }
            };
            int k = s_list[0];
            fetch(k);
            for (int q = 0; q < cnt; ++q) {
                const int kc = k;
                V pk[NE], xk[NE];
#pragma unroll
                for (int u = 0; u < NE; ++u) {
                    pk[u] = np[u];
                    xk[u] = nx[u];
                }
                if (q + 1 < cnt) {
                    k = s_list[q + 1];
                    fetch(k);
                }
                const int J = s_J[q] - i0;
                if (J <= 0) continue;
                const CoefPair<V>* __restrict__ ck = coef + int64_t(kc) * W + i0;
                auto step = [&](int i) {
                    const CoefPair<V> gc = ck[i];
#pragma unroll
                    for (int u = 0; u < NE; ++u) {
                        pk[u] = cfma(gc.g, pk[u], r[u][i]);        // P = r_i + gamma_i P
                        xk[u] = cfma(gc.c, pk[u], xk[u]);          // x = x + c_i P
                    }
                };
                if (J >= BMAX) {
#pragma unroll
                    for (int i = 0; i < BMAX; ++i) step(i);
                } else {
#pragma unroll
                    for (int i = 0; i < BMAX; ++i) {
                        if (i >= J) break;
                        step(i);
                    }
                }
#pragma unroll
                for (int u = 0; u < NE; ++u) {
                    if (!on[u]) continue;
                    const int64_t o = int64_t(kc) * n_out + e + u * int64_t(blockDim.x);
                    P[o] = pk[u];
                    X[o] = xk[u];
                }
            }
        }
    }
}

// For a shift that froze in this window, or for every shift with pending iterations
// once the solve is done, its recursive residual at its last tested iteration,
// fz_coef[k] * r~_{fz_iter[k]} (r~ from the ring).  blockIdx.y: shift.
template <typename V>
__global__ void __launch_bounds__(256) k_rrec(const V* __restrict__ ring, int nslot, int64_t ld, V* __restrict__ rrec,
                                              int64_t n_out, const int32_t* __restrict__ rows, int64_t rowlen,
                                              ShiftArrays sh, const SeedState* __restrict__ st) {
    const int k = blockIdx.y;
    if (sh.nblk[k] == 0 || (sh.active[k] && !st->stop)) return;
    const int i = sh.fz_iter[k] - st->m0;                             // 1 .. j
    const V* __restrict__ r = ring + int64_t((st->slot0 + i) % nslot) * ld;
    const double2 cf = sh.fz_coef[k];
    for (int64_t e = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; e < n_out;
         e += int64_t(gridDim.x) * blockDim.x) {
        int64_t src = e;
        if (rows) {
            const int64_t row = e / rowlen;
            src = int64_t(__ldg(rows + row)) * rowlen + (e - row * rowlen);
        }
        rrec[int64_t(k) * n_out + e] = cscale(cf.x, cf.y, r[src]);
    }
}

// ---------------------------------------------------------------------------
// Initialisation: rho = (b,b), ||b||, r_0 = b in ring slot 0, p = b.
// ---------------------------------------------------------------------------
// Dual form (rt != null): r~_0 = p~_0 = b, rho = <b|b>.
template <typename V>
__global__ void __launch_bounds__(256) k_init_vectors(const V* __restrict__ b, V* __restrict__ ring,
                                                      V* __restrict__ p, int64_t n, double* part,
                                                      V* __restrict__ rt, V* __restrict__ pt) {
    __shared__ double sm[3 * 32];
    double acc[3] = {0.0, 0.0, 0.0};
    DF4 df;
    for (int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; s < n;
         s += int64_t(gridDim.x) * blockDim.x) {
        const V x = b[s];
        ring[s] = x;
        p[s] = x;
        if (rt) {
            rt[s] = x;
            pt[s] = x;
            if constexpr (std::is_same<V, float2>::value) {
                her_acc_df(x, x, df);
                norm_acc_df(x, df);
            } else {
                her_acc(x, x, acc[0], acc[1]);
                acc[2] += norm2(x);
            }
            continue;
        }
        if constexpr (std::is_same<V, float2>::value) {
            bil_acc_df(x, x, df);
            norm_acc_df(x, df);
        } else {
            bil_acc(x, x, acc[0], acc[1]);
            acc[2] += norm2(x);
        }
    }
    if constexpr (std::is_same<V, float2>::value) {
        acc[0] = df_value(df.rh, df.rl);
        acc[1] = df_value(df.ih, df.il);
        acc[2] = df_value(df.nh, df.nl);
    }
    store_partials<3>(acc, sm, part);
}

__global__ void __launch_bounds__(kScalarThreads) k_init_state(SeedState* st, const double* part, int nblk,
                                                               ShiftArrays sh, const double2* shifts, int ns,
                                                               double tol, int maxit) {
    __shared__ double sm[3 * 32];
    double v[3];
    reduce_partials<3>(part, nblk, v, sm);
    __shared__ double s_bn;
    __shared__ int s_f0;
    if (threadIdx.x == 0) {
        const double bn = sqrt(v[2]);
        const int f0 = bn > 0.0 && isfinite(bn) && !(bn > 0x1p-300 && bn < 0x1p300) ? -ilogb(bn) : 0;
        st->f0 = f0;
        st->rho = scale2(make_double2(v[0], v[1]), 2 * f0);
        st->alpha = make_double2(1.0, 0.0);
        st->boa = make_double2(0.0, 0.0);
        st->irho = cdiv1(make_double2(1.0, 0.0), st->rho);
        st->beta = make_double2(0.0, 0.0);
        st->rnorm = bn;
        st->bnorm = bn;
        st->ibnorm = bn > 0.0 ? 1.0 / bn : 0.0;
        st->ir0 = scale2(st->ibnorm, -f0);
        st->rexp[0] = bn > 0.0 && isfinite(bn) ? ilogb(bn) + f0 : 0;
        st->tol = tol;
        st->m = 0; st->m0 = 0; st->j = 0; st->jcur = 0; st->slot0 = 0;
        st->status = MSB_OK;
        st->maxit = maxit;
        st->halted = 0;
        st->bad = 0;
        st->bad_n = 0;
        st->cnt_a = 0;
        st->cnt_b = 0;
        st->bar_w = 0;
        st->bar_a = 0;
        st->stop_at = INT_MAX;
        st->stop = (bn == 0.0 || maxit <= 0) ? 1 : 0;
        if (bn != 0.0 && v[0] == 0.0 && v[1] == 0.0) { st->status = MSB_EBREAKDOWN; st->stop = 1; }
        st->nactive = bn == 0.0 ? 0 : ns;
        st->fexp = 0;
        st->sexp = f0;
        s_bn = bn;
        s_f0 = f0;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < ns; k += blockDim.x) {
        sh.shift[k] = shifts[k];
        sh.zeta[k] = make_double2(1.0, 0.0);
        sh.zeta_prev[k] = make_double2(1.0, 0.0);
        sh.izeta[k] = make_double2(1.0, 0.0);
        sh.active[k] = s_bn == 0.0 ? 0 : 1;
        sh.conv[k] = s_bn == 0.0 ? 1 : 0;
        sh.broken[k] = 0;
        sh.nblk[k] = 0;
        sh.iters[k] = 0;
        sh.resid[k] = 0.0;
        sh.zexp[k] = -s_f0;
        sh.fz_coef[k] = make_double2(1.0, 0.0);
        sh.fz_iter[k] = 0;
    }
}

// r~_0 = p_0 = 2^f0 b (dual form: the dual vectors too).
template <typename V>
__global__ void __launch_bounds__(256) k_init_scale(V* ring, V* p, int64_t n, const SeedState* __restrict__ st, V* rt, V* pt) {
    if (st->f0 == 0) return;
    const double sc = scale2(1.0, st->f0);
    for (int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; s < n; s += int64_t(gridDim.x) * blockDim.x) {
        ring[s] = cscale(sc, 0.0, ring[s]);
        p[s] = cscale(sc, 0.0, p[s]);
        if (rt) {
            rt[s] = cscale(sc, 0.0, rt[s]);
            pt[s] = cscale(sc, 0.0, pt[s]);
        }
    }
}

// Zero-fill of the per-shift solutions when the solve ends before any iteration.
template <typename V>
__global__ void k_zero(V* x, int64_t n) {
    for (int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; s < n; s += int64_t(gridDim.x) * blockDim.x)
        x[s] = vzero(V{});
}

// ---------------------------------------------------------------------------
// Host driver
// ---------------------------------------------------------------------------
thread_local SolverLimits g_solver_limits;

struct GraphOwner {
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    ~GraphOwner() {
        if (exec) cudaGraphExecDestroy(exec);
        if (graph) cudaGraphDestroy(graph);
    }
};

template <typename V>
struct SolverImpl {
    using C = V;
    const SolveProblem& pr;
    cudaStream_t st;
    int nslot, B, grid_vec, grid_flush, grid_mvm, grid_upd;
    // Window of the per-shift update: 32 iterations in FP32, 56 in FP64 (one contraction on
    // the tensor cores), whatever the block B of iterations per graph; 32, 16 or B when the ring
    // of residuals would take too much memory.
    int W = 0, grid_tc = 0;
    bool tc = false;
    TcCoef tcc{};
    DevBuf<int> tc_list, tc_cnt, tc_exp;
    DevBuf<double2> tc_mul;
    DevBuf<uint4> tc_frag;
    int64_t ld = 0;               // ring slot stride: n rounded up to even (16-byte FP32 pairs)
    RowPlan rows;                 // row-tiled seed product (Hubbard without a second amplitude or phases)
    const HubPart* rparts = nullptr;
    DevBuf<V> ring, p, v, Pbuf;
    DevBuf<V> rt, pt, vt;     // dual-space vectors (App. A), allocated only for the dual form
    DevBuf<double> part;
    DevBuf<SeedState> state;
    DevBuf<double2> zeta, zeta_prev, izeta, shift, coef64;
    DevBuf<C> coefv;
    DevBuf<int> active, conv, broken, nblk, iters, zexp, fz_iter;
    DevBuf<double2> fz_coef;
    DevBuf<double> resid;
    DevBuf<double2> shifts_dev;
    ShiftArrays sh{};
    int64_t launches = 0, flushes = 0;

    SolverImpl(const SolveProblem& p_, cudaStream_t s) : pr(p_), st(s) {}

    const msb_op* op = nullptr;
    size_t csz = sizeof(V);

    template <class View>
    void iteration(const View& view) {
        const int64_t n = pr.n;
        const double nb = double(n) * csz;
        {
            ProfScope ps("seed_mvm", st, 2 * nb + op->matrix_bytes(csz), op->hx_flops() + 16.0 * n);
            if (rows.ok)
                launch_hub_rows<V>(rows, rparts, p.p, n, 1, pr.c0.x,
                                   MvmEpi<V>{v.p, state.p, part.p, pt.p, scalar_t<V>(pr.c0.x), scalar_t<V>(pr.c0.y),
                                             {0.0, 0.0}, {}}, st);
            else
                k_mvm_dot<View, V><<<grid_vec, 256, 0, st>>>(view, p.p, v.p, n, pr.c0.x, pr.c0.y, state.p, part.p, pt.p);
        }
        if (pr.dual) {
            ProfScope ps("seed_mvm", st, 2 * nb + op->matrix_bytes(csz), op->hx_flops() + 8.0 * n);
            k_dual_mvm<View, V><<<grid_vec, 256, 0, st>>>(view, pt.p, vt.p, n, pr.c0.x, pr.c0.y, state.p);
        }
        {
            ProfScope ps("seed_update", st, (pr.dual ? 6 : 3) * nb, 20.0 * n);
            k_seed_update<V><<<grid_upd + 1, kVecThreads, 0, st>>>(ring.p, ld, v.p, n, nslot, state.p, part.p,
                                                                   rt.p, vt.p, sh, pr.ns, W);
        }
        {
            ProfScope ps("seed_p", st, 3 * nb, 8.0 * n);
            k_update_p<V><<<grid_upd + 1, kVecThreads, 0, st>>>(ring.p, ld, p.p, n, nslot, state.p, rt.p,
                                                                pt.p, sh, pr.ns);
        }
    }

    // A whole window of iterations in one launch (k_window), on the shape of coop_plan.  False: the
    // runtime refused it, since its CTAs do not fit the SMs at once (a context limited to part of
    // the SMs); nothing ran.
    int coop_t = 0, coop_ne = 0, coop_g = 0;
    template <class View>
    bool window(const View& view) {
        cudaError_t e = cudaErrorCooperativeLaunchTooLarge;
        if constexpr (!std::is_same<View, SumView>::value) {
            if (g_solver_limits.refuse_cooperative) return false;
            ProfScope ps("seed_window", st, 0, 0);
            auto go = [&](auto kern) {
                View vw = view;
                V *rg = ring.p, *pp = p.p;
                int64_t l = ld, n = pr.n;
                double cr = pr.c0.x, ci = pr.c0.y;
                int sl = nslot, ns = pr.ns, w = W;
                SeedState* s = state.p;
                double* pa = part.p;
                void* args[] = {&vw, &rg, &l, &pp, &n, &cr, &ci, &sl, &s, &pa, &sh, &ns, &w, &w};
                e = cudaLaunchCooperativeKernel((const void*)kern, dim3(coop_g + 1), dim3(coop_t), args, 0, st);
            };
            if (coop_ne == 1) go(k_window<View, V, 1>);
            else go(k_window<View, V, 2>);
        }
        if (e != cudaErrorCooperativeLaunchTooLarge && e != cudaErrorNotSupported) {
            MSB_CUDA(e);
            return true;
        }
        cudaGetLastError();
        return false;
    }

    // Launch shape of k_window, or none (coop_g = 0): up to 384 elements per worker (n = 57,984
    // on 152 SMs), the smallest CTAs that take one element per thread (the FP64 pipe of an SM
    // issues one warp at a time) and have a thread per shift.  Measured, us per iteration, graph of
    // launches -> k_window.  FP64: Hubbard sectors n = 36, 3,920, 15,876 and 52,920 with 41 shifts
    // 42 -> 28, 29.4 -> 17.9, 29.9 -> 20.2, 38.6 -> 32.2; random matrices n = 38,000 35.7 -> 25.3,
    // 60,001 40.1 -> 39.8, 100,003 (four elements per thread) 49 -> 85.  FP32: 28.5 -> 17.5 at
    // n = 3,920, 29.3 -> 23.6 at 52,920.
    void coop_plan(bool view_ok) {
        if (pr.dual || !view_ok) return;
        int dev = 0, ok = 0;
        MSB_CUDA(cudaGetDevice(&dev));
        MSB_CUDA(cudaDeviceGetAttribute(&ok, cudaDevAttrCooperativeLaunch, dev));
        const int most = sm_count() - 1;                          // one CTA per SM, one of them for the scalars
        if (!ok || most < 1) return;
        int t = 64;
        while (t < 256 && (pr.n > int64_t(t) * most || pr.ns > t)) t *= 2;
        if (pr.n > int64_t(384) * most) return;
        coop_ne = pr.n <= int64_t(t) * most ? 1 : 2;
        coop_t = t;
        coop_g = int((pr.n + int64_t(t) * coop_ne - 1) / (int64_t(t) * coop_ne));
    }

    // End of a window: the per-shift update of its iterations, then an empty window.
    void flush() {
        {
            ProfScope ps("shift_update", st, 0, 0);
            const int* cnt = tc ? tcc.cnt : nullptr;
            if (tc) {
                k_tc_coef<<<(pr.ns + 3) / 4, 128, 0, st>>>(nblk.p, coef64.p, pr.ns, W, nslot, &state.p->slot0,
                                                          &state.p->bnorm, tcc);
            }
            auto go = [&](auto kern) {
                kern<<<grid_flush, 256, 0, st>>>(ring.p, nslot, ld, Pbuf.p, (V*)pr.x, pr.n_out, pr.rows, pr.rowlen, sh, pr.ns,
                                                 state.p, W, cnt);
            };
            if constexpr (std::is_same<V, float2>::value) {
                if (W == 32) go(k_flush<V, 32, 2>);
                else if (W == 16) go(k_flush<V, 16, 1>);
                else go(k_flush<V, 8, 1>);
            } else {
                go(k_flush<V, 8, 1>);
            }
            if constexpr (std::is_same<V, double2>::value) {
                if (tc)
                    k_flush_tc<<<grid_tc, kTcThreads, kTcSmem, st>>>(ring.p, nslot, ld, Pbuf.p, (V*)pr.x, pr.n_out, pr.rows,
                                                                     pr.rowlen, &state.p->slot0, &state.p->j,
                                                                     &state.p->m0, &state.p->bnorm, tcc);
            }
            if (pr.rrec)
                k_rrec<V><<<dim3(grid_for(pr.n_out, 256, 2), pr.ns), 256, 0, st>>>(ring.p, nslot, ld, (V*)pr.rrec, pr.n_out,
                                                                                  pr.rows, pr.rowlen, sh, state.p);
        }
        launches += 1 + (tc ? 2 : 0) + (pr.rrec ? 1 : 0);
        ++flushes;
    }

    void window_begin() {
        ProfScope ps("shift_scalars", st, 0, 0);
        k_block_begin<<<1, kScalarThreads, 0, st>>>(state.p, sh, pr.ns, nslot);
        ++launches;
    }

    template <class View>
    void run(const msb_op* op_, const View& view, SolveResult& out) {
        op = op_;
        const int64_t n = pr.n, ns = pr.ns;
        // A window is whole blocks, and the same for every block the caller asks for (bitwise equal
        // results): FP64 graphs hold at most 8 iterations.
        static_assert(kTcWindow % 8 == 0, "whole blocks per window");
        B = std::min(pr.block, std::is_same<V, float2>::value ? 16 : 8);
        W = std::is_same<V, float2>::value ? 32 : kTcWindow;
        grid_vec = grid_for(n, 256, 8);
        constexpr bool f32 = std::is_same<V, float2>::value;
        rows = op->kind == 2 ? (f32 ? op->plan32 : op->plan64) : row_plan<V>(op, 1);
        if (op->kind == 2) rparts = f32 ? op->parts32.p : op->parts64.p;
        grid_mvm = rows.ok ? rows.grid : grid_vec;
        coop_plan(!std::is_same<View, SumView>::value);
        ld = (n + 1) / 2 * 2;
        grid_upd = std::min(grid_for((n * int64_t(sizeof(V)) + 15) / 16, kVecThreads, 3), 3 * sm_count() - 1);
        p.alloc(n);
        v.alloc(n);
        if (pr.dual) { rt.alloc(n); pt.alloc(n); vt.alloc(n); }
        Pbuf.alloc(size_t(ns) * pr.n_out);
        part.alloc(std::max(size_t(std::max(std::max(grid_vec, grid_mvm), grid_upd)) * 4, size_t(coop_g) * 8));
        state.alloc(1);
        zeta.alloc(ns); zeta_prev.alloc(ns); izeta.alloc(ns); shift.alloc(ns);
        coef64.alloc(size_t(ns) * W * 2);
        coefv.alloc(size_t(ns) * W * 2);
        active.alloc(ns); conv.alloc(ns); broken.alloc(ns); nblk.alloc(ns); iters.alloc(ns); zexp.alloc(ns);
        fz_iter.alloc(ns); fz_coef.alloc(ns);
        resid.alloc(ns);
        shifts_dev.alloc(ns);
        // The ring comes last.  A long one takes at most 16 GiB and a quarter of the memory that is
        // left, so that other threads' solves still find room: with less, the window is shorter,
        // and one block at the end, as small as it can be.  FP64 windows down to 16 iterations stay
        // on the tensor cores.  A window is not twice the iterations that the caller allows: five
        // iterations of the L = 14 seed in FP32 paid 0.6 ms of 4.3 for a ring of 32.
        const int longest = W;
        for (const int w : {longest, 32, 16, B}) {
            if (w > longest || w < B || (w > B && pr.maxit <= w / 2)) continue;
            const size_t bytes = size_t(w + 1) * ld * sizeof(V);
            if (w > B && bytes > g_solver_limits.ring_bytes) continue;
            if (w > B && bytes > (size_t(1) << 30)) {
                size_t free_b = 0, total_b = 0;
                MSB_CUDA(cudaMemGetInfo(&free_b, &total_b));
                if (bytes > free_b / 4) continue;
            }
            W = w;
            try {
                ring.alloc(size_t(w + 1) * ld);
                break;
            } catch (const Error& e) {
                if (e.status != MSB_ENOMEM || w == B) throw;
                cudaGetLastError();
            }
        }
        nslot = W + 1;
        tc = !f32 && W >= 16 && ns >= kTcMinShifts;
        // two elements per thread for a whole FP32 window only
        grid_flush = f32 && W == 32 ? grid_for((pr.n_out + 1) / 2, 256, 4) : grid_for(pr.n_out, 256, 8);
        if (tc) {
            tc_list.alloc(ns); tc_cnt.alloc(1); tc_exp.alloc(2 * ns); tc_mul.alloc(2 * ns);
            tc_frag.alloc(size_t((ns + 3) / 4) * kTcSteps * kTcDigits * 32);
            tcc = TcCoef{tc_list.p, tc_cnt.p, tc_mul.p, tc_exp.p, tc_frag.p, coef64.p, nblk.p, W, state.p->rexp};
            grid_tc = int(std::min<int64_t>((pr.n_out + kTcCols - 1) / kTcCols, 2 * sm_count()));
            raise_shared_limit((const void*)k_flush_tc, kTcSmem);
        }
        shifts_dev.upload(pr.shifts.data(), ns, st);
        sh = ShiftArrays{zeta.p, zeta_prev.p, izeta.p, shift.p, coef64.p, (void*)coefv.p,
                         active.p, conv.p, broken.p, nblk.p, iters.p, resid.p, zexp.p, fz_coef.p, fz_iter.p};

        {
            ProfScope ps("seed_init", st, 3.0 * n * csz, 12.0 * n);
            k_init_vectors<V><<<grid_vec, 256, 0, st>>>((const V*)pr.b, ring.p, p.p, n, part.p, rt.p, pt.p);
        }
        {
            ProfScope ps("shift_scalars", st, 0, 0);
            k_init_state<<<1, kScalarThreads, 0, st>>>(state.p, part.p, grid_vec, sh, shifts_dev.p, int(ns),
                                                        pr.tol, pr.maxit);
        }
        {
            ProfScope ps("shift_scalars", st, 0, 0);
            k_init_scale<V><<<grid_vec, 256, 0, st>>>(ring.p, p.p, n, state.p, rt.p, pt.p);
        }
        launches += 3;
        MSB_LAUNCH_CHECK();
        bool coop = false;
        int BB = 0;                                 // iterations per launch of a block
        int64_t per_block = 0, max_blocks = 0, blocks = 0;      // kernels per block
        auto form = [&](bool cooperative) {
            coop = cooperative;
            BB = coop ? W : B;
            per_block = coop ? 1 : (pr.dual ? 4 : 3) * int64_t(B);
            max_blocks = (int64_t(pr.maxit) + BB - 1) / BB + 1;
        };
        form(coop_g > 0);
        GraphOwner g;                               // one block of B iterations, captured at its first use
        auto launch_block = [&] {
            if (coop && !window(view)) {
                if (blocks > 0) fail(MSB_ECUDA, "a window of iterations was refused after others had run");
                form(false);
            }
            if (!coop && prof_on()) {
                for (int i = 0; i < B; ++i) iteration(view);
            } else if (!coop) {
                if (!g.exec) {
                    MSB_CUDA(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
                    for (int i = 0; i < B; ++i) iteration(view);
                    MSB_CUDA(cudaStreamEndCapture(st, &g.graph));
                    MSB_CUDA(cudaGraphInstantiate(&g.exec, g.graph, 0));
                }
                MSB_CUDA(cudaGraphLaunch(g.exec, st));
            }
            launches += per_block;
        };
        if (prof_on()) {
            // Profiled: direct launches, one sync per block, and one after each fused
            // update to attribute its work (shifts and iterations it carried).
            SeedState hs;
            auto look = [&] {
                MSB_CUDA(cudaMemcpyAsync(&hs, state.p, sizeof(SeedState), cudaMemcpyDeviceToHost, st));
                MSB_CUDA(cudaStreamSynchronize(st));
            };
            for (;;) {
                launch_block();
                ++blocks;
                look();
                if (coop)
                    prof_patch_last("seed_window", hs.j * (8.0 * n * csz + op->matrix_bytes(csz)),
                                    hs.j * (op->hx_flops() + 44.0 * n));
                const bool end = hs.stop || blocks > max_blocks + 2;
                if (end || blocks * BB % W == 0) {
                    flush();
                    look();
                    const double no = double(pr.n_out) * csz;
                    prof_patch_last("shift_update", hs.flush_J * no + hs.flush_cnt * (hs.flush_first ? 2.0 : 4.0) * no,
                                    16.0 * hs.flush_cnt * hs.flush_J * double(pr.n_out));
                    window_begin();
                }
                if (end) break;
            }
            prof_collect();
        } else {

        HostBuf<SeedState> hstate(2);
        cudaEvent_t ev[2];
        MSB_CUDA(cudaEventCreateWithFlags(&ev[0], cudaEventDisableTiming));
        MSB_CUDA(cudaEventCreateWithFlags(&ev[1], cudaEventDisableTiming));
        bool finished = false;
        // Two blocks in flight: launch block i, then look at the state copied
        // after block i-1.  Blocks launched after convergence return at once.
        while (!finished) {
            launch_block();
            if ((blocks + 1) * BB % W == 0) { flush(); window_begin(); }
            const int slot = int(blocks & 1);
            MSB_CUDA(cudaMemcpyAsync(&hstate.p[slot], state.p, sizeof(SeedState), cudaMemcpyDeviceToHost, st));
            MSB_CUDA(cudaEventRecord(ev[slot], st));
            if (blocks >= 1) {
                MSB_CUDA(cudaEventSynchronize(ev[slot ^ 1]));
                if (hstate.p[slot ^ 1].stop) finished = true;
            }
            ++blocks;
            if (blocks > max_blocks + 2) break;
        }
        flush();                                       // the last, partial window (nothing pending: no work)
        MSB_LAUNCH_CHECK();
        MSB_CUDA(cudaStreamSynchronize(st));
        cudaEventDestroy(ev[0]);
        cudaEventDestroy(ev[1]);
        }
        out.flushes = flushes;

        SeedState fs;
        MSB_CUDA(cudaMemcpyAsync(&fs, state.p, sizeof(SeedState), cudaMemcpyDeviceToHost, st));
        MSB_CUDA(cudaStreamSynchronize(st));
        if (fs.m == 0) {   // no iteration ran: solutions are zero
            k_zero<V><<<grid_for(ns * pr.n_out, 256, 8), 256, 0, st>>>((V*)pr.x, ns * pr.n_out);
            launches += 1;
        }
        out.iterations = fs.m;
        out.seed_residual = fs.bnorm > 0 ? fs.rnorm / fs.bnorm : 0.0;
        out.bnorm = fs.bnorm;
        out.iters.resize(ns);
        out.resid.resize(ns);
        out.conv.resize(ns);
        std::vector<int> brk(ns);
        MSB_CUDA(cudaMemcpyAsync(out.iters.data(), iters.p, ns * sizeof(int), cudaMemcpyDeviceToHost, st));
        MSB_CUDA(cudaMemcpyAsync(out.resid.data(), resid.p, ns * sizeof(double), cudaMemcpyDeviceToHost, st));
        MSB_CUDA(cudaMemcpyAsync(out.conv.data(), conv.p, ns * sizeof(int), cudaMemcpyDeviceToHost, st));
        MSB_CUDA(cudaMemcpyAsync(brk.data(), broken.p, ns * sizeof(int), cudaMemcpyDeviceToHost, st));
        MSB_CUDA(cudaStreamSynchronize(st));
        out.status = msb_status(fs.status);
        out.cooperative = coop;
        int nconv = 0;
        for (int k = 0; k < ns; ++k) nconv += out.conv[k];
        out.n_converged = nconv;
        bool any_broken = false;
        for (int k = 0; k < ns; ++k) any_broken |= brk[k] != 0;
        if (out.status == MSB_OK && any_broken) out.status = MSB_EBREAKDOWN;
        if (out.status == MSB_OK && nconv < ns) out.status = MSB_EMAXITER;
        out.launches = launches;
    }
};

void multishift_solve(msb_op* op, const SolveProblem& pr, SolveResult& out, cudaStream_t st) {
    MSB_REQUIRE(pr.ns >= 1 && pr.ns <= kMaxShifts, "n_shifts must be in 1..4096");
    MSB_REQUIRE(pr.dual || !op_has_flux(op),
                "the operator is complex Hermitian (Peierls phases), not complex symmetric: use the dual solver");
    if (pr.prec == MSB_FP64) {
        SolverImpl<double2> s(pr, st);
        if (op->kind == 0) s.run(op, op->hub, out);
        else if (op->kind == 1) s.run(op, op->csr, out);
        else s.run(op, op->sum, out);
    } else {
        SolverImpl<float2> s(pr, st);
        if (op->kind == 0) s.run(op, op->hub, out);
        else if (op->kind == 1) s.run(op, op->csr, out);
        else s.run(op, op->sum, out);
    }
}

int pick_block(int block, msb_precision prec, int64_t n, int ns) {
    if (block == 0) {
        const int t = n > 0 ? tuned_block(n, ns, prec) : 0;
        return t ? t : (prec == MSB_FP64 ? 4 : 8);
    }
    MSB_REQUIRE(block == 1 || block == 2 || block == 4 || block == 8 || block == 16,
                "block must be 0 (auto), 1, 2, 4, 8 or 16");
    return block;
}

}  // namespace msb

// ----------------------------------------------------------------------------
// C ABI
// ----------------------------------------------------------------------------
// For tests (not part of the header): the calling thread's limits of the solves that follow.
extern "C" void msb_test_solver_limits(int64_t ring_bytes, int refuse_cooperative) {
    msb::g_solver_limits.ring_bytes = ring_bytes > 0 ? size_t(ring_bytes) : msb::SolverLimits().ring_bytes;
    msb::g_solver_limits.refuse_cooperative = refuse_cooperative != 0;
}

static msb_status solve_entry(const char* fname, bool dual, msb_op* A, msb_complex c0, const void* b,
                              const msb_complex* shifts, int n_shifts, double tol, int maxit, int block,
                              msb_precision prec, void* x, int* iters, double* resid, int* converged,
                              msb_solve_info* info, void* stream) {
    msb_status result = MSB_OK;
    msb_status g = msb::guard(fname, [&] {
        msb::require_device();
        MSB_REQUIRE(A != nullptr && b != nullptr && x != nullptr && shifts != nullptr, "NULL argument");
        MSB_REQUIRE(prec == MSB_FP64 || prec == MSB_FP32_MIXED, "unknown precision");
        MSB_REQUIRE(tol >= 0.0, "tol must be >= 0");
        MSB_REQUIRE(maxit >= 0, "maxit must be >= 0");
        auto t0 = std::chrono::steady_clock::now();
        msb::g_alloc_bytes = 0;
        msb::SolveProblem pr;
        pr.n = A->dim;
        pr.ns = n_shifts;
        pr.b = b;
        pr.x = x;
        pr.n_out = A->dim;
        pr.c0 = make_double2(c0.re, c0.im);
        pr.tol = tol;
        pr.maxit = maxit;
        pr.block = msb::pick_block(block, prec, A->dim, n_shifts);
        pr.prec = prec;
        pr.dual = dual;
        pr.shifts.resize(n_shifts);
        for (int k = 0; k < n_shifts; ++k) pr.shifts[k] = make_double2(shifts[k].re, shifts[k].im);
        msb::SolveResult out;
        msb::StreamScope scope((cudaStream_t)stream);
        msb::multishift_solve(A, pr, out, scope.s);
        scope.finish();
        if (iters) for (int k = 0; k < n_shifts; ++k) iters[k] = out.iters[k];
        if (resid) for (int k = 0; k < n_shifts; ++k) resid[k] = out.resid[k];
        if (converged) for (int k = 0; k < n_shifts; ++k) converged[k] = out.conv[k];
        if (info) {
            *info = msb_solve_info{};
            info->iterations = out.iterations;
            info->n_converged = out.n_converged;
            info->matvecs = (dual ? 2 : 1) * int64_t(out.iterations);
            info->flushes = out.flushes;
            info->seed_residual = out.seed_residual;
            double mx = 0;
            for (double r : out.resid) mx = r > mx ? r : mx;
            info->max_shift_residual = mx;
            info->seconds_solve = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
            info->seconds_total = info->seconds_solve;
            info->device_bytes = msb::g_alloc_bytes;
            info->kernel_launches = out.launches;
        }
        result = out.status;
        if (result != MSB_OK)
            msb::set_error_message(std::string(fname) + ": recurrence ended with status " + std::to_string(int(result)));
    });
    return g != MSB_OK ? g : result;
}

extern "C" msb_status msb_multishift_bicg_solve(msb_op* A, msb_complex c0, const void* b,
                                                const msb_complex* shifts, int n_shifts, double tol,
                                                int maxit, int block, msb_precision prec, void* x,
                                                int* iters, double* resid, int* converged,
                                                msb_solve_info* info, void* stream) {
    return solve_entry("msb_multishift_bicg_solve", false, A, c0, b, shifts, n_shifts, tol, maxit, block, prec, x,
                       iters, resid, converged, info, stream);
}

extern "C" msb_status msb_multishift_bicg_dual_solve(msb_op* A, msb_complex c0, const void* b,
                                                     const msb_complex* shifts, int n_shifts, double tol,
                                                     int maxit, int block, msb_precision prec, void* x,
                                                     int* iters, double* resid, int* converged,
                                                     msb_solve_info* info, void* stream) {
    return solve_entry("msb_multishift_bicg_dual_solve", true, A, c0, b, shifts, n_shifts, tol, maxit, block, prec, x,
                       iters, resid, converged, info, stream);
}
