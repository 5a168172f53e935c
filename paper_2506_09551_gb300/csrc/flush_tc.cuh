// The per-shift update of a whole window of iterations as one contraction on the tensor
// cores, in 56-bit fixed point (FP64 solves with many shifts).
//
// Over a window of J iterations the recurrence P <- r_i + gamma_i P, x <- x + c_i P of one
// shift is linear in P_0 and the seed residuals r_0 .. r_{J-1}:
//   x_J = x_0 + kappa P_0 + sum_i w_i r_i,   w_{J-1} = c_{J-1}, w_i = c_i + gamma_{i+1} w_{i+1},
//   P_J = G P_0 + sum_i g_i r_i,             g_{J-1} = 1,       g_i = gamma_{i+1} g_{i+1},
// kappa = gamma_0 w_0, G = gamma_0 g_0.  The sums of all shifts are a matrix product: rows
// (shift, x or P, re or im), depth (iteration, re or im), columns the elements.
//
// Why.  FP64 issues at 1/64 of the FP32 rate here, and the recurrence takes 8 FP64 FMAs per
// shift, element and iteration at 92% of that pipe.  As a contraction the FP64 work is 24
// operations per shift and element and window: the P_0 terms (8), and adding the integer
// sums to x and P (16).
//
// Split.  Each operand is an integer multiple of 2^-55 of the largest value it shares a scale
// with, cut into seven balanced 8-bit digits that bf16 holds exactly.  A product of two
// digits is below 2^14, a sum over 128 depth entries and at most seven digit pairs of equal
// weight below 2^24, so the FP32 accumulators of the tensor core hold exact integers.  The
// 28 digit pairs of weight 2^0 .. 2^-48 are kept; what is dropped and the rounding of the
// operands lie at 2^-53 of (largest w_i |r_i|) of the window.  Scales, all powers of two:
// e_i (of ||r_i||) per iteration, one per row of the coefficients, one per column tile.
// Each of x and P is then rounded a few times per window instead of per iteration.
//
// Measured (GB300): per-shift update of a whole solve, against the recurrence (k_flush in
// msbicg.cu): random symmetric matrix, n = 200,003, 128 shifts, 348 -> 30 ms (16 windows of
// 64 iterations, 1.9 ms each); L = 12 intermediate sector, n = 731,808, 41 shifts, 399 -> 52 ms.
#pragma once

#include <climits>

#include "kernels.cuh"
#include "msbicg_impl.cuh"

namespace msb {

constexpr int kTcWindow = 64;                 // iterations per window
constexpr int kTcSteps = kTcWindow / 8;       // depth steps of 16 = 8 iterations, re and im
constexpr int kTcCols = 64;                   // elements per column tile
constexpr int kTcDigits = 7;
constexpr int kTcThreads = 256;
constexpr int kTcMinShifts = 8;               // fewer pending shifts: the recurrence (k_flush)
constexpr size_t kTcSmem = size_t(kTcDigits) * kTcSteps * (kTcCols / 8) * 32 * 8;

// Per pending shift (in list order), x first, then P.
struct TcCoef {
    int* list;         // shift index
    int* cnt;          // number of pending shifts
    double2* mul;      // [2 * li + type]: kappa, G
    int* exp;          // [2 * li + type]: exponent of the row's scale
    uint4* frag;       // [tile of 4 shifts][step][digit][lane]: A fragments
    int* rexp;         // per ring slot: exponent of the stored ||r~||
};

// x 2^-e as seven balanced digits; |x 2^-e| <= 0.995.
__device__ __forceinline__ unsigned long long tc_fixed(double x, int e) {
    const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
    const int ex = int(b >> 52) & 0x7FF;
    const unsigned long long m = (b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
    const int s = ex - 1020 - e;                              // F = m 2^s
    unsigned long long f;
    if (s >= 0) f = m << min(s, 2);
    else if (s >= -54) f = (m + (1ull << (-s - 1))) >> -s;
    else f = 0;
    if (ex == 0) f = 0;                                       // zero (and subnormals)
    const unsigned long long sgn = static_cast<unsigned long long>(__double_as_longlong(x) >> 63);
    return ((f ^ sgn) - sgn) + 0x0080808080808080ull;
}
// Digit d (0 = most significant) as an exactly representable float.
__device__ __forceinline__ float tc_digit(unsigned long long u, int d) {
    const unsigned by = unsigned(u >> (48 - 8 * d)) & 0xFFu;
    return __uint_as_float(0x4B000000u | by) - 8388736.0f;    // 2^23 + 128
}
// Two floats that bf16 holds exactly, as a bf16 pair (lo in the low half).
__device__ __forceinline__ unsigned tc_pack(float lo, float hi) {
    return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}
// Exponent e with largest |value| 2^-e in [0.4975, 0.995], from the high word of the largest
// absolute value (its own exponent shifted by the caller).
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
            const int ei = tc.rexp[(slot0 + i) % nslot];
            const int h = max(__double2hiint(w.x) & 0x7FFFFFFF, __double2hiint(w.y) & 0x7FFFFFFF);
            if (h >= 0x100000) key = max(key, h + ei * 0x100000);
            if (h >= 0x7FF00000) key = INT_MAX;
        }
        for (int o = 16; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
        const bool none = key == INT_MIN, bad = key == INT_MAX;
        const int E = none || bad ? 0 : tc_exponent(key);
        if (lane == 0 && k >= 0) {
            tc.exp[2 * li + type] = bad ? INT_MAX : E;
        }
        const int q = 2 * wid + type;                           // row of the real parts; + 8: imaginary parts
        for (int i = lane; i < kTcWindow; i += 32) {
            unsigned long long ur = 0x0080808080808080ull, ui = ur;      // zero
            if (i < J && !none && !bad) {
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

// Seven accumulators of equal-weight digit pairs, added to v at the scale sc (weight of the
// last one): two exact integers, each converted with one FP64 addition.
__device__ __forceinline__ double tc_add(double v, float a0, float a1, float a2, float a3, float a4, float a5, float a6,
                                         double sc, double sch) {
    const long long hi = (static_cast<long long>(__float2int_rn(a0)) << 16) + __float2int_rn(a1) * 256ll + __float2int_rn(a2);
    const long long lo = (static_cast<long long>(__float2int_rn(a3)) << 24) +
                         (static_cast<long long>(__float2int_rn(a4)) << 16) + __float2int_rn(a5) * 256ll + __float2int_rn(a6);
    const double dh = __longlong_as_double(0x4338000000000000ll + hi) - 6755399441055744.0;   // 1.5 2^52
    const double dl = __longlong_as_double(0x4338000000000000ll + lo) - 6755399441055744.0;
    return fma(dh, sch, fma(dl, sc, v));
}

// One CTA per tile of 64 elements (persistent): the window's residuals of the tile are cut
// into digits once and stay in shared memory (112 KB, two CTAs per SM) for all shifts; warp w
// takes columns 16 (w % 4) .. + 15 and every second tile of four shifts, coefficients from
// L2 / L1 in fragment order.  Rows 0..7 of a tile are the real parts of (shift, x or P), rows
// 8..15 the imaginary parts, so a thread ends with two whole complex elements of one vector
// and gets P_0 for an x row from the lane four over.
// Bound by the FP64 pipe (24 operations per shift, element and window), then by the legacy
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
    __shared__ int s_key;
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
        }
        if (tid == 0) s_key = INT_MIN;
        __syncthreads();
        const int col = tid & (kTcCols - 1), ig = tid / kTcCols;
        const int src = s_src[col];
        {
            int key = INT_MIN;
            if (src >= 0)
                for (int i = ig; i < J; i += kTcThreads / kTcCols) {
                    const double2 r = ring[int64_t(s_slot[i]) * ld + src];
                    const int h = max(__double2hiint(r.x) & 0x7FFFFFFF, __double2hiint(r.y) & 0x7FFFFFFF);
                    if (h >= 0x7FF00000) key = INT_MAX;
                    else if (h >= 0x100000 && key != INT_MAX) key = max(key, h - s_e[i] * 0x100000);
                }
            for (int o = 16; o > 0; o >>= 1) key = max(key, __shfl_xor_sync(0xffffffffu, key, o));
            if (lane == 0) atomicMax(&s_key, key);
        }
        __syncthreads();
        const int tkey = s_key;
        const bool tbad = tkey == INT_MAX;
        const int te = tkey == INT_MIN || tbad ? 0 : tc_exponent(tkey);
        // digits: a warp takes eight columns and one depth step; lane: column lane % 8,
        // iterations lane / 8 and 4 more (whole 128-byte lines of r, conflict-free stores)
        for (int c = wid; c < steps * (kTcCols / 8); c += kTcThreads / 32) {
            const int s = c / (kTcCols / 8), nt = c % (kTcCols / 8), cl = lane & 7, ii = lane >> 3;
            const int sc = s_src[nt * 8 + cl];
            unsigned long long u[2][2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int i = s * 8 + ii + 4 * h;
                u[h][0] = u[h][1] = 0x0080808080808080ull;
                if (sc >= 0 && i < J && !tbad) {
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
        for (int t = wid >> 2; t < mt; t += 2) {
            float acc[kTcDigits][2][4];
#pragma unroll
            for (int d = 0; d < kTcDigits; ++d)
#pragma unroll
                for (int n = 0; n < 2; ++n)
#pragma unroll
                    for (int c = 0; c < 4; ++c) acc[d][n][c] = 0.f;
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
            const int li = t * 4 + (q >> 1);
            const bool on = li < cnt;
            const int k = on ? tc.list[li] : 0;
            const double2 mul = on ? tc.mul[2 * li + type] : make_double2(0.0, 0.0);
            const int re = on ? tc.exp[2 * li + type] : 0;
            double sc = 0.0, sch = 0.0;
            if (on) {
                sc = re == INT_MAX || tbad ? nan("") : tc_pow2(re + te - 62);
                sch = sc * 4294967296.0;
            }
            double2* __restrict__ out = (type ? P : X) + int64_t(k) * n_out;
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                const int64_t e = c0 + (nt0 + n) * 8 + (lane & 3) * 2;
                double2 own[2];
#pragma unroll
                for (int c = 0; c < 2; ++c)
                    own[c] = on && !first && e + c < n_out ? out[e + c] : make_double2(0.0, 0.0);
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    double2 p0;
                    p0.x = __shfl_xor_sync(0xffffffffu, own[c].x, 4);
                    p0.y = __shfl_xor_sync(0xffffffffu, own[c].y, 4);
                    double2 v = own[c];
                    if (type) { p0 = own[c]; v = make_double2(0.0, 0.0); }
                    v.x = fma(mul.x, p0.x, fma(-mul.y, p0.y, v.x));
                    v.y = fma(mul.x, p0.y, fma(mul.y, p0.x, v.y));
                    v.x = tc_add(v.x, acc[0][n][c], acc[1][n][c], acc[2][n][c], acc[3][n][c], acc[4][n][c],
                                 acc[5][n][c], acc[6][n][c], sc, sch);
                    v.y = tc_add(v.y, acc[0][n][2 + c], acc[1][n][2 + c], acc[2][n][2 + c], acc[3][n][2 + c],
                                 acc[4][n][2 + c], acc[5][n][2 + c], acc[6][n][2 + c], sc, sch);
                    if (on && e + c < n_out) out[e + c] = v;
                }
            }
        }
    }
}

}  // namespace msb
