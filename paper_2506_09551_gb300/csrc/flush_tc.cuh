// The per-shift update of a whole window of iterations as one contraction on the tensor
// cores, in 64-bit fixed point (FP64 solves with many shifts).
//
// Over a window of J iterations the recurrence P <- r_i + gamma_i P, x <- x + c_i P of one
// shift is linear in P_0 and the seed residuals r_0 .. r_{J-1}:
//   x_J = x_0 + kappa P_0 + sum_i w_i r_i,   w_{J-1} = c_{J-1}, w_i = c_i + gamma_{i+1} w_{i+1},
//   P_J = G P_0 + sum_i g_i r_i,             g_{J-1} = 1,       g_i = gamma_{i+1} g_{i+1},
// kappa = gamma_0 w_0, G = gamma_0 g_0.  The sums of all shifts are a matrix product: rows
// (shift, x or P, re or im), depth (iteration, re or im), columns the elements.
//
// Why.  FP64 issues at 1/64 of the FP32 rate here, and the recurrence takes 8 FP64 FMAs per
// shift, element and iteration at 92% of that pipe.  As a contraction the FP64 work is 20
// operations per shift and element and window: the P_0 terms (8), and forming the integer
// sums and adding them to x and P (12).
//
// Split.  Each operand is an integer multiple of 2^-63 of the largest value it shares a scale
// with, cut into eight balanced 8-bit digits that bf16 holds exactly.  A product of two
// digits is at most 2^14, a sum over 112 depth entries and at most eight digit pairs of equal
// weight below 2^24, so the FP32 accumulators of the tensor core hold exact integers.  The
// 36 digit pairs of weight 2^0 .. 2^-56 are kept; the pairs of weight 2^-64 are dropped.
// Scales, all powers of two: e_i (of ||r_i||) per iteration, one per row of the coefficients
// (a shift's x or P), one per element (column), so that no element depends on its neighbours.
//
// Precision.  What is dropped and the rounding of the operands come to about 2^-60 of the
// product of the two scales.  An element that ends below 2^-16 of that product (its residuals
// are large where the coefficients are small, or the terms cancel), and whatever is not finite
// or near the ends of the exponent range, takes the recurrence instead, with its operations in
// its order.  So what the fixed point adds to an element is below 2^-44 of it in the worst case
// and below 2^-53 in the usual one.  Windows simulated against 64-bit mantissas (random matrix,
// L = 6 ring, diagonal and tridiagonal matrices with right-hand sides graded over 30 decades):
// error of x in the 2-norm 0.3 to 0.8 times the recurrence's, in the median over the elements
// 0.4 to 1.0 times.  (Seven digits, 28 pairs and one scale for 64 elements: 2 to 14 times in
// the 2-norm, and no correct digit in elements 1e-18 of a neighbour.)
//
// Measured (GB300): per-shift update of a whole solve, against the recurrence (k_flush in
// msbicg.cu): random symmetric matrix, n = 200,003, 128 shifts, 348 -> 35 ms (18 windows of
// 56 iterations); L = 12 intermediate sector, n = 731,808, 41 shifts, 399 -> 67 ms (31 windows;
// about 7 ms of it for the elements redone, nearly all in the first window).  Seven digits: 30
// and 52 ms.
#pragma once

#include <climits>

#include "kernels.cuh"
#include "msbicg_impl.cuh"

namespace msb {

constexpr int kTcWindow = 56;                 // iterations per window (112 KB of digits: two CTAs per SM)
constexpr int kTcSteps = kTcWindow / 8;       // depth steps of 16 = 8 iterations, re and im
constexpr int kTcCols = 64;                   // elements per column tile
constexpr int kTcDigits = 8;
constexpr int kTcThreads = 256;
constexpr int kTcLoss = 16;                   // bits below its scale at which an element is redone:
                                              // at 12 the L = 12 update takes 79 ms, at 14 70, at 16 67
constexpr int kTcMinShifts = 8;               // fewer pending shifts: the recurrence (k_flush)
constexpr size_t kTcSmem = size_t(kTcDigits) * kTcSteps * (kTcCols / 8) * 32 * 8;

// Per pending shift (in list order), x first, then P.
struct TcCoef {
    int* list;         // shift index
    int* cnt;          // number of pending shifts
    double2* mul;      // [2 * li + type]: kappa, G
    int* exp;          // [2 * li + type]: exponent of the row's scale, or kTcZero / kTcBad
    uint4* frag;       // [tile of 4 shifts][step][digit][lane]: A fragments
    const double2* coef;   // (gamma, c) of the window's iterations, W per shift
    const int* nblk;       // pending iterations of each shift
    int W;
    int* rexp;         // per ring slot: exponent of the stored ||r~||
};

// Exponents of a scale: every value is zero; the fixed point cannot hold the values.
constexpr int kTcZero = INT_MIN, kTcBad = INT_MAX;

// x 2^-e as eight balanced digits; |x 2^-e| <= 0.995.
__device__ __forceinline__ unsigned long long tc_fixed(double x, int e) {
    const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
    const int ex = int(b >> 52) & 0x7FF;
    const unsigned long long m = (b & 0x000FFFFFFFFFFFFFull) | (ex ? 0x0010000000000000ull : 0ull);
    const int s = max(ex, 1) - 1012 - e;                      // F = m 2^s
    unsigned long long f;
    if (s >= 0) f = m << min(s, 10);
    else if (s >= -54) f = (m + (1ull << (-s - 1))) >> -s;
    else f = 0;
    const unsigned long long sgn = static_cast<unsigned long long>(__double_as_longlong(x) >> 63);
    return ((f ^ sgn) - sgn) + 0x8080808080808080ull;
}
// Digit d (0 = most significant) as an exactly representable float.
__device__ __forceinline__ float tc_digit(unsigned long long u, int d) {
    const unsigned by = unsigned(u >> (56 - 8 * d)) & 0xFFu;
    return __uint_as_float(0x4B000000u | by) - 8388736.0f;    // 2^23 + 128
}
// Two floats that bf16 holds exactly, as a bf16 pair (lo in the low half).
__device__ __forceinline__ unsigned tc_pack(float lo, float hi) {
    return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}
// High word of the larger absolute value of two, 0 only if both are zero.
__device__ __forceinline__ int tc_high(double2 v) {
    const int h = max(__double2hiint(v.x) & 0x7FFFFFFF, __double2hiint(v.y) & 0x7FFFFFFF);
    return h ? h : (__double2loint(v.x) | __double2loint(v.y)) != 0;
}
// Exponent e with largest |value| 2^-e in [0.4975, 0.995] (below for subnormals), from the high
// word of the largest absolute value (its own exponent shifted by the caller).
__device__ __forceinline__ int tc_exponent(int key) { return (key >> 20) - 1022 + ((key & 0xFFFFF) > 0xFD000 ? 1 : 0); }

__device__ __forceinline__ double tc_pow2(int e) {
    return e > -1022 && e < 1023 ? __hiloint2double((1023 + e) << 20, 0) : ldexp(1.0, e);
}

// Shifts with pending iterations beyond i0, in order (warp 0; every thread calls).
__device__ __forceinline__ int pending_list(const int* __restrict__ nblk, int ns, int i0, int* list, int* s_cnt) {
    if (threadIdx.x < 32) {
        int c = 0;
        for (int b = 0; b < ns; b += 32) {
            const int k = b + threadIdx.x;
            const bool on = k < ns && nblk[k] > i0;
            const unsigned m = __ballot_sync(0xffffffffu, on);
            if (on) list[c + __popc(m & ((1u << threadIdx.x) - 1u))] = k;
            c += __popc(m);
        }
        if (threadIdx.x == 0) *s_cnt = c;
    }
    __syncthreads();
    return *s_cnt;
}

// Whether a window goes to the tensor cores: enough shifts to pay for cutting the residuals
// into digits, and a right-hand side whose residuals are normal numbers.
__device__ __forceinline__ bool tc_use(int cnt, double bnorm) {
    return cnt >= kTcMinShifts && bnorm > 0x1p-900 && bnorm < 0x1p900;
}

// Coefficients of the window: one CTA of four warps per tile of four shifts.
__global__ void __launch_bounds__(128) k_tc_coef(const int* __restrict__ nblk, const double2* __restrict__ coef64, int ns,
                                                 int W, int nslot, const int* __restrict__ p_slot0,
                                                 const double* __restrict__ p_bnorm, TcCoef tc) {
    __shared__ int s_list[kMaxShifts];
    __shared__ int s_cnt;
    __shared__ double2 s_g[4][kTcWindow];                       // gamma_i
    __shared__ double2 s_w[4][2][kTcWindow];                    // c_i, then w_i; g_i
    const int cnt = pending_list(nblk, ns, 0, s_list, &s_cnt);
    if (blockIdx.x == 0 && threadIdx.x == 0) *tc.cnt = cnt;
    if (!tc_use(cnt, *p_bnorm)) return;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int li = blockIdx.x * 4 + wid;
    if (int(blockIdx.x) * 4 >= cnt) return;
    const int k = li < cnt ? s_list[li] : -1;
    const int J = k >= 0 ? nblk[k] : 0;
    const double2* __restrict__ ck = coef64 + int64_t(k < 0 ? 0 : k) * W * 2;
    const int slot0 = *p_slot0;
    for (int i = lane; i < J; i += 32) {
        s_g[wid][i] = ck[2 * i];
        s_w[wid][0][i] = ck[2 * i + 1];
    }
    __syncwarp();
    // lane 0: w, lane 1: g (the same backward recurrence, without the c_i and from 1)
    if (lane < 2 && k >= 0) {
        double2 v = lane ? make_double2(1.0, 0.0) : s_w[wid][0][J - 1];
        s_w[wid][lane][J - 1] = v;
        for (int i = J - 2; i >= 0; --i) {
            v = cfma(s_g[wid][i + 1], v, lane ? make_double2(0.0, 0.0) : s_w[wid][0][i]);
            s_w[wid][lane][i] = v;
        }
        tc.mul[2 * li + lane] = cmul(s_g[wid][0], v);
        if (lane == 0) tc.list[li] = k;
    }
    __syncwarp();
    for (int type = 0; type < 2; ++type) {
        // scale of the row: the largest |w_i| 2^{e_i}
        int key = INT_MIN;
        for (int i = lane; i < J; i += 32) {
            const double2 w = s_w[wid][type][i];
            const int ei = tc.rexp[(slot0 + i) % nslot], h = tc_high(w);
            if ((h >> 20) + max(ei, 0) >= 2040) key = kTcBad;
            else if (h > 0) key = max(key, h + ei * 0x100000);
        }
        for (int o = 16; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
        const bool fixed = key != kTcZero && key != kTcBad;
        const int E = fixed ? tc_exponent(key) : 0;
        if (lane == 0 && k >= 0) tc.exp[2 * li + type] = fixed ? E : key;
        const int q = 2 * wid + type;                           // row of the real parts; + 8: imaginary parts
        for (int i = lane; i < kTcWindow; i += 32) {
            unsigned long long ur = 0x8080808080808080ull, ui = ur;      // zero
            if (i < J && fixed) {
                const double2 w = s_w[wid][type][i];
                const int e = E - tc.rexp[(slot0 + i) % nslot];
                ur = tc_fixed(w.x, e);
                ui = tc_fixed(w.y, e);
            }
            const int s = i >> 3, ii = i & 7;
            unsigned* __restrict__ f =
                reinterpret_cast<unsigned*>(tc.frag + (int64_t(blockIdx.x) * kTcSteps + s) * kTcDigits * 32);
            const int word = (q * 4 + (ii & 3)) * 4 + (ii < 4 ? 0 : 2);
#pragma unroll
            for (int d = 0; d < kTcDigits; ++d) {
                const float r = tc_digit(ur, d), m = tc_digit(ui, d);
                f[d * 128 + word] = tc_pack(r, -m);             // re row: (wr, -wi)
                f[d * 128 + word + 1] = tc_pack(m, r);          // im row: (wi, wr)
            }
        }
    }
}

__device__ __forceinline__ void tc_mma(float (&c)[4], const uint4& a, const uint2& b) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y));
}

// v + sc T, T = sum a[l] 2^(8 (7 - l)) of eight accumulators of equal-weight digit pairs.  T is the
// sum of two exact integers hi 2^32 + lo; 1.5 2^52 + lo has the integer in its low bits, and what
// that adds is taken off hi, so that one addition and one FMA give T rounded once.
__device__ __forceinline__ double tc_add(double v, const float (&a)[kTcDigits], double sc) {
    auto four = [](float p, float q, float r, float s) {
        return (static_cast<long long>(__float2int_rn(p)) << 24) + (static_cast<long long>(__float2int_rn(q)) << 16) +
               (__float2int_rn(r) * 256ll + __float2int_rn(s));
    };
    const double hi = __longlong_as_double(0x4338000000000000ll + four(a[0], a[1], a[2], a[3]));
    const double lo = __longlong_as_double(0x4338000000000000ll + four(a[4], a[5], a[6], a[7]));
    return fma(fma(hi - (6755399441055744.0 + 1572864.0), 4294967296.0, lo), sc, v);
}

// One CTA per tile of 64 elements (persistent): the window's residuals of the tile are cut
// into digits once and stay in shared memory (112 KB, two CTAs per SM) for all shifts; warp w
// takes columns 16 (w % 4) .. + 15 and every second tile of four shifts, coefficients from
// L2 / L1 in fragment order.  Rows 0..7 of a tile are the real parts of (shift, x or P), rows
// 8..15 the imaginary parts, so a thread ends with two whole complex elements of one vector
// and gets P_0 for an x row from the lane four over.
// Bound by the FP64 pipe (20 operations per shift, element and window), then by the legacy
// MMA rate and shared memory, about equal.
__global__ void __launch_bounds__(kTcThreads, 2) k_flush_tc(const double2* __restrict__ ring, int nslot, int64_t ld,
                                                            double2* __restrict__ P, double2* __restrict__ X,
                                                            int64_t n_out, const int32_t* __restrict__ rows,
                                                            int64_t rowlen, const int* __restrict__ p_slot0,
                                                            const int* __restrict__ p_j, const int* __restrict__ p_m0,
                                                            const double* __restrict__ p_bnorm, TcCoef tc) {
    const int cnt = *tc.cnt;
    if (!tc_use(cnt, *p_bnorm)) return;
    extern __shared__ __align__(16) uint2 s_b[];               // [digit][step][8 columns][lane]
    __shared__ int s_src[kTcCols];
    __shared__ int s_e[kTcWindow];
    __shared__ int s_slot[kTcWindow];
    __shared__ int s_te[kTcCols];                              // exponent of the column's scale
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int slot0 = *p_slot0, J = *p_j;
    const bool first = *p_m0 == 0;
    const int steps = (J + 7) >> 3;
    const int mt = (cnt + 3) >> 2;
    for (int i = tid; i < kTcWindow; i += kTcThreads) {
        const int sl = (slot0 + i) % nslot;
        s_slot[i] = sl;
        s_e[i] = tc.rexp[sl];
    }
    const int64_t tiles = (n_out + kTcCols - 1) / kTcCols;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        const int64_t c0 = tile * kTcCols;
        __syncthreads();
        if (tid < kTcCols) {
            const int64_t e = c0 + tid;
            int64_t src = -1;
            if (e < n_out) {
                src = e;
                if (rows) {
                    const int64_t row = e / rowlen;
                    src = int64_t(__ldg(rows + row)) * rowlen + (e - row * rowlen);
                }
            }
            s_src[tid] = int(src);
            s_te[tid] = kTcZero;
        }
        __syncthreads();
        const int col = tid & (kTcCols - 1), ig = tid / kTcCols;
        const int src = s_src[col];
        {
            int key = kTcZero;
            if (src >= 0)
                for (int i = ig; i < J; i += kTcThreads / kTcCols) {
                    const int h = tc_high(ring[int64_t(s_slot[i]) * ld + src]);
                    if (h >= 0x7FF00000) key = kTcBad;
                    else if (h > 0 && key != kTcBad) key = max(key, h - s_e[i] * 0x100000);
                }
            atomicMax(&s_te[col], key);
        }
        __syncthreads();
        if (tid < kTcCols && s_te[tid] != kTcZero && s_te[tid] != kTcBad) s_te[tid] = tc_exponent(s_te[tid]);
        __syncthreads();
        // digits: a warp takes eight columns and one depth step; lane: column lane % 8,
        // iterations lane / 8 and 4 more (whole 128-byte lines of r, conflict-free stores)
        for (int c = wid; c < steps * (kTcCols / 8); c += kTcThreads / 32) {
            const int s = c / (kTcCols / 8), nt = c % (kTcCols / 8), cl = lane & 7, ii = lane >> 3;
            const int sc = s_src[nt * 8 + cl], te = s_te[nt * 8 + cl];
            unsigned long long u[2][2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = s * 8 + ii + 4 * h;
                u[h][0] = u[h][1] = 0x8080808080808080ull;
                if (sc >= 0 && i < J && te != kTcZero && te != kTcBad) {
                    const double2 r = ring[int64_t(s_slot[i]) * ld + sc];
                    const int e = te + s_e[i];
                    u[h][0] = tc_fixed(r.x, e);
                    u[h][1] = tc_fixed(r.y, e);
                }
            }
            uint2* __restrict__ b = s_b + (s * (kTcCols / 8) + nt) * 32 + cl * 4 + ii;
#pragma unroll
            for (int d = 0; d < kTcDigits; ++d)
                b[d * (kTcSteps * (kTcCols / 8) * 32)] = make_uint2(tc_pack(tc_digit(u[0][0], d), tc_digit(u[0][1], d)),
                                                                   tc_pack(tc_digit(u[1][0], d), tc_digit(u[1][1], d)));
        }
        __syncthreads();
        const int nt0 = (wid & 3) * 2;
        const int q = lane >> 2, type = q & 1;
        for (int t = wid >> 2; t < mt; t += kTcThreads / 128) {
            float acc[kTcDigits][2][4];
#pragma unroll
            for (int d = 0; d < kTcDigits; ++d)
#pragma unroll
                for (int n = 0; n < 2; ++n)
#pragma unroll
                    for (int c = 0; c < 4; ++c) acc[d][n][c] = 0.f;
            const int li = t * 4 + (q >> 1);
            const bool on = li < cnt;
            const int k = on ? tc.list[li] : 0;
            double2* __restrict__ out = (type ? P : X) + int64_t(k) * n_out;
            const uint4* __restrict__ fa = tc.frag + int64_t(t) * kTcSteps * kTcDigits * 32 + lane;
            for (int s = 0; s < steps; ++s) {
                uint2 b[2][kTcDigits];
#pragma unroll
                for (int d = 0; d < kTcDigits; ++d)
#pragma unroll
                    for (int n = 0; n < 2; ++n) b[n][d] = s_b[((d * kTcSteps + s) * (kTcCols / 8) + nt0 + n) * 32 + lane];
#pragma unroll
                for (int d = 0; d < kTcDigits; ++d) {
                    const uint4 a = __ldg(fa + (s * kTcDigits + d) * 32);
#pragma unroll
                    for (int j = 0; j + d < kTcDigits; ++j)
#pragma unroll
                        for (int n = 0; n < 2; ++n) tc_mma(acc[d + j][n], a, b[n][j]);
                }
            }
            const double2 mul = on ? tc.mul[2 * li + type] : make_double2(0.0, 0.0);
            const int re = on ? tc.exp[2 * li + type] : kTcZero;
            double2 v[2][2];
            unsigned redo = 0;                                 // bit 2 n + c
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                const int64_t e = c0 + (nt0 + n) * 8 + (lane & 3) * 2;
                double2 own[2];
#pragma unroll
                for (int c = 0; c < 2; ++c)
                    own[c] = on && !first && e + c < n_out ? out[e + c] : make_double2(0.0, 0.0);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int te = s_te[(nt0 + n) * 8 + (lane & 3) * 2 + c];
                    // weight of the digit sums, and the high word below which an element is redone
                    int sch = 0, least = 0;
                    if (re == kTcBad || te == kTcBad) least = 0x7FF00000;
                    else if (re != kTcZero && te != kTcZero) {
                        const int x = re + te;
                        const bool in = x >= -880 && x <= 1000;
                        sch = in ? (1023 + x - 70) << 20 : 0;
                        least = in ? (1023 + x - kTcLoss) << 20 : 0x7FF00000;
                    }
                    double2 p0;
                    p0.x = __shfl_xor_sync(0xffffffffu, own[c].x, 4);
                    p0.y = __shfl_xor_sync(0xffffffffu, own[c].y, 4);
                    double2 w = own[c];
                    if (type) { p0 = own[c]; w = make_double2(0.0, 0.0); }
                    w.x = fma(mul.x, p0.x, fma(-mul.y, p0.y, w.x));
                    w.y = fma(mul.x, p0.y, fma(mul.y, p0.x, w.y));
                    float ar[kTcDigits], ai[kTcDigits];
#pragma unroll
                    for (int d = 0; d < kTcDigits; ++d) {
                        ar[d] = acc[d][n][c];
                        ai[d] = acc[d][n][2 + c];
                    }
                    const double sc = __hiloint2double(sch, 0);
                    w.x = tc_add(w.x, ar, sc);
                    w.y = tc_add(w.y, ai, sc);
                    v[n][c] = w;
                    const int h = tc_high(w);
                    if (on && e + c < n_out && (h < least || h >= 0x7FF00000)) redo |= 1u << (2 * n + c);
                }
            }
            // x and P of an element are redone together: x needs P_0
            const bool some = __any_sync(0xffffffffu, redo != 0);
            if (some) redo |= __shfl_xor_sync(0xffffffffu, redo, 4);
#pragma unroll
            for (int n = 0; n < 2; ++n)
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    const int64_t e = c0 + (nt0 + n) * 8 + (lane & 3) * 2 + c;
                    if (on && e < n_out && !(redo >> (2 * n + c) & 1u)) out[e] = v[n][c];
                }
            if (!some) continue;
            // the recurrence for the elements that the fixed point does not hold well enough; of a
            // thread and its partner (x and P of the same elements) each takes one of two columns
            while (redo & (5u << type)) {
                const int n = (redo >> type) & 1u ? 0 : 1, cc = (nt0 + n) * 8 + (lane & 3) * 2 + type;
                redo &= ~(1u << (2 * n + type));
                const int64_t o = int64_t(k) * n_out + c0 + cc;
                const double2* __restrict__ rs = ring + s_src[cc];
                const double2* __restrict__ ck = tc.coef + int64_t(k) * tc.W * 2;
                double2 p = first ? make_double2(0.0, 0.0) : P[o], x = first ? make_double2(0.0, 0.0) : X[o];
                const int Jk = tc.nblk[k];
                for (int i = 0; i < Jk; ++i) {
                    p = cfma(ck[2 * i], p, rs[int64_t(s_slot[i]) * ld]);
                    x = cfma(ck[2 * i + 1], p, x);
                }
                P[o] = p;
                X[o] = x;
            }
            __syncwarp();
        }
    }
}

}  // namespace msb
