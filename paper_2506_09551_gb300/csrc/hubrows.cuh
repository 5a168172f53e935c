// Row-tiled product with the Hubbard operator, y = H x per element with a fused
// epilogue: the plain apply, the seed product with its bilinear form and the
// Lanczos step share it.
//
// Layout.  A CTA takes R consecutive rows u of one vector (R = 1 once a row has as
// many elements as the CTA has threads; several short rows otherwise, so that tiny
// sectors still fill warps) or one of `split` equal parts of a single row, stages the
// rows in shared memory (one zero word past each row), and each thread forms whole
// elements: the up-spin hops read rows u' coalesced from global memory (L2), the
// down-spin hops gather from the staged row.  Row data that a thread per element
// would fetch again and again (offsets and signs of the up-spin hops, the up string,
// the diagonal's 3 (L + 1) values) sits in shared memory.
//
// What bounds it.  FP64: the FP64 pipe, which issues 1/64 of the FP32 rate here and
// is also held by predicated-off instructions.  A hop is therefore exactly one FMA
// per component with a multiplier +-1 built in the integer pipe (a sign select that
// compiles to predicated add and subtract costs two), the trip count of the down-spin
// loop is the warp's maximum with empty slots reading the zero word, and the diagonal
// is a table (an integer-to-double conversion runs in the FP64 pipe).  FP32: the L1 /
// shared pipe and L2 latency; two adjacent elements per thread when D_dn is even.
//
// Measured (GB300, per call, against a thread per element with both species' hops
// gathered from global memory): eight FP64 vectors on the L = 12 ring (D = 853,776)
// 1235 -> 535 us (the FP64 pipe alone needs about 410 us); one FP32 vector on the L = 14
// intermediate sector (D = 10,306,296) 246 -> 130 us; the L = 6 ring (300 states) 15 us
// either way.
#pragma once

#include <algorithm>

#include "kernels.cuh"

namespace msb {

// +-1 with the sign of a table entry's bit 0, without the FP64 pipe.
__device__ __forceinline__ double pm_one(double, uint32_t h) { return __hiloint2double(int(0x3FF00000u | (h << 31)), 0); }
__device__ __forceinline__ float pm_one(float, uint32_t h) { return __uint_as_float(0x3F800000u | (h << 31)); }

// acc += g v (g = +-1)
__device__ __forceinline__ void hop_add(double& a, double g, double v) { a = fma(g, v, a); }
__device__ __forceinline__ void hop_add(double2& a, double g, double2 v) { a.x = fma(g, v.x, a.x); a.y = fma(g, v.y, a.y); }
__device__ __forceinline__ void hop_add(float2& a, float g, float2 v) { a.x = fmaf(g, v.x, a.x); a.y = fmaf(g, v.y, a.y); }
__device__ __forceinline__ void hop_add(float4& a, float g, float4 v) {
    a.x = fmaf(g, v.x, a.x); a.y = fmaf(g, v.y, a.y); a.z = fmaf(g, v.z, a.z); a.w = fmaf(g, v.w, a.w);
}

// Epi: operator()(s, xs, acc, dg, mt, shift): element s of the column, x[s], the signed
// hop sum, the diagonal, -t and the block's shift (hub_value forms H x + c0 x from them);
// finish(): partial sums.
// PAIR (float2, even D_dn): two adjacent elements per thread.
template <typename V, bool Multi, bool PAIR, class Epi>
__global__ void __launch_bounds__(256) k_hub_rows(HubPart p0, const HubPart* __restrict__ parts, int np,
                                                  const V* __restrict__ x, int64_t ldx, int64_t tiles, double c0r,
                                                  double one, Epi epi) {
    using S = scalar_t<V>;
    if (epi.stop()) return;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    __shared__ double red[2 * 256];
    const int nt = blockDim.x;
    epi.begin(blockIdx.y);
    const V* __restrict__ xc = x + int64_t(blockIdx.y) * ldx;
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
        int q = 0;
        if constexpr (Multi) {
            while (q + 1 < np && tile >= parts[q + 1].tile0) ++q;
        }
        const HubPart& P = Multi ? parts[q] : p0;
        const HubView& h = P.v;
        const int Ddn = int(h.Ddn), L = h.L, W = h.Wup, R = P.R;
        const int tl = int(tile - P.tile0);
        const int u0 = (P.split > 1 ? tl / P.split : tl) * R;
        const int rows = min(R, int(h.Dup) - u0);
        const int chunk = P.split > 1 ? ((Ddn + 2 * P.split - 1) / (2 * P.split)) * 2 : rows * Ddn;
        const int e0 = P.split > 1 ? (tl % P.split) * chunk : 0;
        const int e1 = P.split > 1 ? min(e0 + chunk, Ddn) : rows * Ddn;
        const int64_t base = P.off + int64_t(u0) * Ddn;           // element of (u0, 0) in the column
        const int ldr = Ddn + 2;                                   // staged row and its zero word (16-byte pairs)
        V* row = reinterpret_cast<V*>(sm_raw);
        S* lut = reinterpret_cast<S*>(row + int64_t(R) * ldr);     // 3 (L + 1)
        S* s_sg = lut + 3 * (L + 1);                               // R x W
        int* s_off = reinterpret_cast<int*>(s_sg + R * W);         // R x W
        int* s_nu = s_off + R * W;                                 // R
        uint32_t* s_su = reinterpret_cast<uint32_t*>(s_nu + R);    // R
        const V* __restrict__ xp = xc + P.off;
        // stage the rows and their per-row data
        if constexpr (PAIR) {
            const int half = Ddn >> 1;
            const float4* __restrict__ src = reinterpret_cast<const float4*>(xc + base);
            if (R == 1) {
                for (int i = threadIdx.x; i < half; i += nt) reinterpret_cast<float4*>(row)[i] = src[i];
            } else {
                for (int i = threadIdx.x; i < rows * half; i += nt) {
                    const int r = i / half;
                    reinterpret_cast<float4*>(row)[r * (half + 1) + (i - r * half)] = src[i];
                }
            }
        } else {
            if (R == 1) {
                for (int i = threadIdx.x; i < Ddn; i += nt) row[i] = xc[base + i];
            } else {
                for (int i = threadIdx.x; i < rows * Ddn; i += nt) {
                    const int r = i / Ddn;
                    row[r * ldr + (i - r * Ddn)] = xc[base + i];
                }
            }
        }
        for (int r = threadIdx.x; r < rows; r += nt) {
            row[r * ldr + Ddn] = vzero(V{});
            row[r * ldr + Ddn + 1] = vzero(V{});
            s_nu[r] = __ldg(h.nup + u0 + r);
            s_su[r] = __ldg(h.sup + u0 + r);
        }
        for (int i = threadIdx.x; i < rows * W; i += nt) {
            const int r = i / W, e = i - r * W;
            const int32_t ent = __ldg(h.hup + int64_t(e) * h.Dup + u0 + r);    // -1 past the row's hops (not read)
            s_off[i] = (ent >> 1) * Ddn;
            s_sg[i] = (ent & 1) ? S(-1) : S(1);
        }
        for (int i = threadIdx.x; i < 3 * (L + 1); i += nt) {
            const int nb = i / (L + 1), pc = i - nb * (L + 1);
            if constexpr (sizeof(S) == 8) lut[i] = h.U * double(pc) - h.Uc * double(nb);
            else lut[i] = h.Uf * float(pc) - h.Ucf * float(nb);
        }
        __syncthreads();
        const int core = h.core;
        // FP64: the block's shift and the real part of c0 as one constant (c0 alone without a sum)
        const S mt = S(-h.t), shift = sizeof(S) == 8 ? S(P.shift + c0r) : S(P.shift);
        const S s1 = S(one);                                       // 1, opaque to the compiler: an FMA, not an add
        const uint16_t* __restrict__ t16 = h.hdnr16;
        constexpr int PE = PAIR ? 2 : 1;
        const int n = (e1 - e0) / PE;
        const int iters = (n + nt - 1) / nt;
        for (int it = 0; it < iters; ++it) {
            const int i = it * nt + threadIdx.x;
            const bool act = i < n;
            const int e = e0 + (act ? i : 0) * PE;
            const int r = R == 1 ? 0 : e / Ddn;
            const int d = e - r * Ddn;
            const int nu = s_nu[r];
            const int* __restrict__ uo = s_off + r * W;
            const S* __restrict__ us = s_sg + r * W;
            const V* __restrict__ xr = row + r * ldr;
            const uint32_t su = s_su[r];
            if constexpr (PAIR) {
                const float4* __restrict__ x4 = reinterpret_cast<const float4*>(xp);
                float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
                const int dh = d >> 1;
                int k = 0;
                for (; k + 4 <= nu; k += 4) {
                    const float4 v0 = x4[(uo[k] >> 1) + dh], v1 = x4[(uo[k + 1] >> 1) + dh];
                    const float4 v2 = x4[(uo[k + 2] >> 1) + dh], v3 = x4[(uo[k + 3] >> 1) + dh];
                    hop_add(a, us[k], v0); hop_add(a, us[k + 1], v1);
                    hop_add(a, us[k + 2], v2); hop_add(a, us[k + 3], v3);
                }
                if (k + 3 == nu) {
                    const float4 v0 = x4[(uo[k] >> 1) + dh], v1 = x4[(uo[k + 1] >> 1) + dh], v2 = x4[(uo[k + 2] >> 1) + dh];
                    hop_add(a, us[k], v0); hop_add(a, us[k + 1], v1); hop_add(a, us[k + 2], v2);
                } else if (k + 2 == nu) {
                    const float4 v0 = x4[(uo[k] >> 1) + dh], v1 = x4[(uo[k + 1] >> 1) + dh];
                    hop_add(a, us[k], v0); hop_add(a, us[k + 1], v1);
                } else if (k < nu) {
                    hop_add(a, us[k], x4[(uo[k] >> 1) + dh]);
                }
                const uint32_t nn = __ldg(reinterpret_cast<const uint16_t*>(h.ndn) + dh);
                const int nd = __reduce_max_sync(0xffffffffu, act ? max(nn & 0xFFu, nn >> 8) : 0u);
                const uint32_t* __restrict__ tp = reinterpret_cast<const uint32_t*>(t16) + dh;
                const int step = Ddn >> 1;
                k = 0;
                for (; k + 2 <= nd; k += 2, tp += 2 * step) {
                    const uint32_t ta = __ldg(tp), tb = __ldg(tp + step);
                    const float2 va = xr[(ta & 0xFFFFu) >> 1], vb = xr[ta >> 17];
                    const float2 vc = xr[(tb & 0xFFFFu) >> 1], vd = xr[tb >> 17];
                    const float ga = pm_one(0.f, ta), gb = pm_one(0.f, ta >> 16);
                    const float gc = pm_one(0.f, tb), gd = pm_one(0.f, tb >> 16);
                    a.x = fmaf(ga, va.x, a.x); a.y = fmaf(ga, va.y, a.y);
                    a.z = fmaf(gb, vb.x, a.z); a.w = fmaf(gb, vb.y, a.w);
                    a.x = fmaf(gc, vc.x, a.x); a.y = fmaf(gc, vc.y, a.y);
                    a.z = fmaf(gd, vd.x, a.z); a.w = fmaf(gd, vd.y, a.w);
                }
                if (k < nd) {
                    const uint32_t ta = __ldg(tp);
                    const float2 va = xr[(ta & 0xFFFFu) >> 1], vb = xr[ta >> 17];
                    const float ga = pm_one(0.f, ta), gb = pm_one(0.f, ta >> 16);
                    a.x = fmaf(ga, va.x, a.x); a.y = fmaf(ga, va.y, a.y);
                    a.z = fmaf(gb, vb.x, a.z); a.w = fmaf(gb, vb.y, a.w);
                }
                const uint32_t sa = __ldg(h.sdn + d), sb = __ldg(h.sdn + d + 1);
                const int ub = core >= 0 ? int((su >> core) & 1u) : 0;
                const int na = core >= 0 ? ub + int((sa >> core) & 1u) : 0;
                const int nb = core >= 0 ? ub + int((sb >> core) & 1u) : 0;
                const float da = lut[__popc(su & sa) + na * (L + 1)], db = lut[__popc(su & sb) + nb * (L + 1)];
                if (act) {
                    const float2 xa = xr[d], xb = xr[d + 1];
                    epi.pair(base + e, xa, xb, make_float2(a.x, a.y), make_float2(a.z, a.w), da, db, mt, shift);
                }
            } else {
                V a = vzero(V{});
                int k = 0;
                for (; k + 4 <= nu; k += 4) {
                    const V v0 = xp[uo[k] + d], v1 = xp[uo[k + 1] + d];
                    const V v2 = xp[uo[k + 2] + d], v3 = xp[uo[k + 3] + d];
                    hop_add(a, us[k], v0); hop_add(a, us[k + 1], v1);
                    hop_add(a, us[k + 2], v2); hop_add(a, us[k + 3], v3);
                }
                // the rest together, without FP64 work for missing hops
                if (k + 3 == nu) {
                    const V v0 = xp[uo[k] + d], v1 = xp[uo[k + 1] + d], v2 = xp[uo[k + 2] + d];
                    hop_add(a, us[k], v0); hop_add(a, us[k + 1], v1); hop_add(a, us[k + 2], v2);
                } else if (k + 2 == nu) {
                    const V v0 = xp[uo[k] + d], v1 = xp[uo[k + 1] + d];
                    hop_add(a, us[k], v0); hop_add(a, us[k + 1], v1);
                } else if (k < nu) {
                    hop_add(a, us[k], xp[uo[k] + d]);
                }
                const int nd = __reduce_max_sync(0xffffffffu, act ? unsigned(__ldg(h.ndn + d)) : 0u);
                const uint16_t* __restrict__ tp = t16 + d;
                k = 0;
                for (; k + 2 <= nd; k += 2, tp += 2 * Ddn) {
                    const uint32_t ta = __ldg(tp), tb = __ldg(tp + Ddn);
                    const V va = xr[ta >> 1], vb = xr[tb >> 1];
                    hop_add(a, h.dsign ? pm_one(S(0), ta) : s1, va);
                    hop_add(a, h.dsign ? pm_one(S(0), tb) : s1, vb);
                }
                if (k < nd) {
                    const uint32_t ta = __ldg(tp);
                    hop_add(a, h.dsign ? pm_one(S(0), ta) : s1, xr[ta >> 1]);
                }
                const uint32_t sd = __ldg(h.sdn + d);
                const int nb = core >= 0 ? int((su >> core) & 1u) + int((sd >> core) & 1u) : 0;
                const S dg = lut[__popc(su & sd) + nb * (L + 1)];
                if (act) epi(base + e, xr[d], a, dg, mt, shift);
            }
        }
        __syncthreads();                                           // the tile's shared memory is reused
    }
    epi.finish(red);
}

// H x + c0 x from the hop sum and the diagonal.  FP64: `shift` holds the real part of c0 too;
// it is not folded into the diagonal, whose sum with it would be rounded at the diagonal's
// size (13 hops and the c0 of a solve against exact arithmetic, error in the 2-norm: 7.0e-17 as
// here, 7.7e-17 element by element, 9.5e-17 folded).  FP32: in the order of the element-wise
// kernels.
__device__ __forceinline__ double2 hub_value(double2 acc, double dg, double mt, double shift, double, double c0i, double2 x) {
    return make_double2(fma(mt, acc.x, fma(dg, x.x, fma(shift, x.x, -c0i * x.y))),
                        fma(mt, acc.y, fma(dg, x.y, fma(shift, x.y, c0i * x.x))));
}
__device__ __forceinline__ float2 hub_value(float2 acc, float dg, float mt, float shift, float c0r, float c0i, float2 x) {
    float2 h = make_float2(__fmaf_rn(mt, acc.x, __fmul_rn(dg, x.x)), __fmaf_rn(mt, acc.y, __fmul_rn(dg, x.y)));
    if (shift != 0.f) h = vaxpy(shift, x, h);
    const float2 c = cscale_rn(c0r, c0i, x);
    return make_float2(__fadd_rn(h.x, c.x), __fadd_rn(h.y, c.y));
}

constexpr size_t kMaxRowBytes = 112 * 1024;      // two CTAs per SM

// Tiles of an operator's blocks and the launch shape for vectors of element V with
// `nvec` columns; ok = false: the element-wise kernels (a second hopping amplitude,
// Peierls phases, rows too long for shared memory).
template <typename V>
RowPlan row_plan(const msb_op* op, int nvec) {
    RowPlan p;
    if (op->kind != 0 && op->kind != 2) return p;
    const msb_op* const* ops = op->kind == 0 ? &op : op->parts.data();      // made for every apply: no heap
    const size_t nops = op->kind == 0 ? 1 : op->parts.size();
    int64_t maxD = 0;
    constexpr bool f32 = std::is_same<V, float2>::value;
    p.pair = f32;
    for (size_t i = 0; i < nops; ++i) {
        const HubView& h = ops[i]->hub;
        if (h.hdnr16 == nullptr || h.hup2 != nullptr || h.dirup != nullptr || h.Dup * h.Ddn >= (int64_t(1) << 31)) return p;
        maxD = std::max(maxD, h.Ddn);
        p.pair = p.pair && h.Ddn % 2 == 0;
    }
    const int pe = p.pair ? 2 : 1;
    p.threads = maxD >= 1024 * pe ? 256 : 128;
    int64_t t0 = 0;
    for (size_t i = 0; i < nops; ++i) {
        HubPart& q = i == 0 ? p.one : p.parts.emplace_back();
        q.v = ops[i]->hub;
        q.off = op->kind == 2 ? op->sum.off[i] : 0;
        q.shift = op->kind == 2 ? op->sum.shift[i] : 0.0;
        q.tile0 = int(t0);
        q.R = int(std::max<int64_t>(1, std::min<int64_t>(q.v.Dup, p.threads * pe / q.v.Ddn)));
        q.split = 1;
        // halve the rows' work while a column has fewer than ~12 tiles per SM and a part
        // still has two elements per thread
        while (q.R == 1 && q.split < 4 && q.v.Dup * q.split * int64_t(nops) * nvec < int64_t(sm_count()) * 12 &&
               q.v.Ddn / (2 * q.split) >= 2 * p.threads * pe)
            q.split *= 2;
        const size_t sm = size_t(q.R) * (q.v.Ddn + 2) * sizeof(V) + (3 * (q.v.L + 1) + q.R * q.v.Wup) * sizeof(scalar_t<V>) +
                          size_t(q.R) * (q.v.Wup + 2) * 4;
        p.smem = std::max(p.smem, sm);
        t0 += (q.v.Dup + q.R - 1) / q.R * q.split;
        if (i == 0 && op->kind == 2) {
            p.parts.reserve(nops);
            p.parts.push_back(q);
        }
    }
    p.tiles = t0;
    p.np = int(nops);
    const int64_t most = 4096;
    p.grid = int(t0 <= most ? t0 : (t0 + (t0 + most - 1) / most - 1) / ((t0 + most - 1) / most));
    p.ok = p.smem <= kMaxRowBytes && t0 < (int64_t(1) << 31);
    return p;
}

// Launch over `nvec` columns with stride ldx.  dparts: the plan's parts on the device
// (a direct sum), else null.
template <typename V, class Epi>
void launch_hub_rows(const RowPlan& p, const HubPart* dparts, const V* x, int64_t ldx, int nvec, double c0r, Epi epi,
                     cudaStream_t st) {
    auto go = [&](auto kern) {
        // dynamic and static shared memory (4 KB of an epilogue's block sum) together count
        // against the 48 KB that a launch gets without asking
        if (p.smem > 40 * 1024) raise_shared_limit((const void*)kern, kMaxRowBytes);
        kern<<<dim3(p.grid, nvec), p.threads, p.smem, st>>>(p.one, dparts, p.np, x, ldx, p.tiles, c0r, 1.0, epi);
    };
    if constexpr (std::is_same<V, float2>::value) {
        if (p.pair) {
            if (dparts) go(k_hub_rows<V, true, true, Epi>);
            else go(k_hub_rows<V, false, true, Epi>);
            return;
        }
    }
    if (dparts) go(k_hub_rows<V, true, false, Epi>);
    else go(k_hub_rows<V, false, false, Epi>);
}

}  // namespace msb
