// Per-keypoint preparation, shared by the kernels that prepare references and
// queries: a reference's FP32 record, sort key and level statistics; a
// query's FP32 record (a2, a3 of the path; bounds as geom.cu explains).
#pragma once

#include <math.h>

#include "egm_internal.cuh"

namespace egm {
namespace {

__device__ __forceinline__ void set_status(uint32_t *st, uint32_t bit) { atomicOr(st, bit); }

// The hardware conversion for the values d2f leaves to it (kept out of line,
// so that the common case issues no FP64-pipe instruction).
__device__ __noinline__ float d2f_other(double d) { return __double2float_rn(d); }

// double -> float rounded to nearest, ties to even, on the integer pipes (the
// IEEE 754 conversion: keep the sign, rebias the exponent, keep the top 23
// fraction bits and round on the 29 dropped ones; a carry out of the
// fraction moves into the exponent, and from the largest finite float to
// infinity, as rounding to nearest requires).  Only results that are normal
// floats before rounding take this path: zeros, subnormals, values above the
// float range and non-finite values take the hardware conversion.  GB300
// issues FP64-pipe instructions, conversions included, at a small fraction of
// its integer rate.
__device__ __forceinline__ float d2f(double d) {
    const uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
    const uint32_t e = (hi >> 20) & 0x7ffu;
    if (e - 897u > 253u) return d2f_other(d);  // float exponent field (e - 896) outside 1..254
    uint32_t f = (hi & 0x80000000u) | ((e - 896u) << 23) | ((hi & 0xfffffu) << 3) | (lo >> 29);
    const uint32_t rem = lo & 0x1fffffffu;
    f += (rem > 0x10000000u || (rem == 0x10000000u && (f & 1u))) ? 1u : 0u;
    return __uint_as_float(f);
}

// |(x, y)| within a few ulps: the square root of the FMA sum of squares
// where that sum is a normal float far from overflow (a component lost to
// underflow then changes the norm by far less than an ulp), hypotf elsewhere.
__device__ __forceinline__ float norm2f(float x, float y) {
    const float s = fmaf(x, x, y * y);
    if (s >= 1e-30f && s <= 1e30f) return sqrtf(s);
    return hypotf(x, y);
}

__device__ __forceinline__ float fold_atan2(float px, float py) {
    if (px < 0.0f || (px == 0.0f && py > 0.0f)) { px = -px; py = -py; }
    return atan2f(py, px);
}

// What the sort and the windows need of one reference.
struct RefRow {
    float4 rec;      // x - cx, y - cy, eps, index bits
    uint32_t key;    // level | quantised angle
    uint32_t s_bits, d_bits, t_bits;  // float bits: bounds of sin delta (above), distance (below), |p - c| (above)
};

// Reference j of pair P.
__device__ __forceinline__ RefRow prep_ref(const Launch &L, const PairView &P, const PairGeom &G, int64_t j) {
    const double x = P.xy2[2 * j], y = P.xy2[2 * j + 1];
    const double eps = P.eps2 ? P.eps2[j] : P.eps_scalar;
    if (!(finite64(x) && finite64(y) && finite64(eps))) set_status(L.status, kStNan);
    else if (!positive64(eps)) set_status(L.status, kStArg);
    const float epsf = d2f(eps);
    const float xf = d2f(x - G.cx), yf = d2f(y - G.cy);
    RefRow r;
    r.s_bits = 0u;
    r.d_bits = 0x7f800000u;
    // the reference's FP32 record, placed in its bucket by the sort
    r.rec = make_float4(xf, yf, epsf, __uint_as_float((uint32_t)j));
    int level;
    float key;
    if (G.mode == kModeAngular) {
        const float px = G.de + (G.ux * xf + G.uy * yf);
        const float py = (G.ux * yf - G.uy * xf) + G.kappa;
        key = fold_atan2(px, py);
        const float d = norm2f(px, py);
        // the level only groups references (its statistics come from
        // its members): an approximate quotient serves
        const float ratio = __fdividef(d, epsf);
        if (!(ratio >= 2.0f)) {
            level = 0;
        } else {
            level = ilogbf(ratio) - G.level_base;
            level = level < 1 ? 1 : (level > kLevels - 1 ? kLevels - 1 : level);
        }
        const float s = d > 0.0f ? epsf / d : INFINITY;
        r.s_bits = __float_as_uint(s * 1.000001f);
        r.d_bits = __float_as_uint(d * 0.999999f);
    } else {
        key = -G.uy * xf + G.ux * yf;
        level = ilogbf(epsf) - G.level_base;
        level = level < 1 ? 1 : (level > kLevels - 1 ? kLevels - 1 : level);
        r.s_bits = __float_as_uint(epsf * 1.000001f);
    }
    // |p - c| <= sqrt(2) max(|x|, |y|): it only scales FP32 rounding terms
    r.t_bits = __float_as_uint(fmaxf(fabsf(xf), fabsf(yf)) * 1.4142146f);
    if (!isfinite(key)) key = 0.0f;
    const uint32_t q = qmap(key, G.kmin, G.kscale);
    r.key = ((uint32_t)level << kQBits) | q;
    return r;
}

// Query gq (row gq - P.q_off of pair p): its record, also stored.
__device__ __forceinline__ QueryRec prep_query(const Launch &L, const PairView &P, const PairGeom &G, int p,
                                               int64_t gq) {
    const int64_t i = gq - P.q_off;
    const double x1 = P.xy1[2 * i], y1 = P.xy1[2 * i + 1];
    QueryRec r;
    r.flags = 0;
    r.pair = p;
    r.pad[0] = r.pad[1] = 0;
    if (gq % kStabQB == 0) L.blkpair[gq / kStabQB] = p;
    r.A = r.B = r.C = r.key = r.aux0 = r.aux1 = r.E0 = r.E1 = 0.0f;
    if (!(finite64(x1) && finite64(y1))) set_status(L.status, kStNan);
    const double *F = P.F;
    // the line with FMAs: within a few ulps of its terms of the exact line
    const double a = fma(F[0], x1, fma(F[1], y1, F[2]));
    const double b = fma(F[3], x1, fma(F[4], y1, F[5]));
    const double c = fma(F[6], x1, fma(F[7], y1, F[8]));
    const float x1f = fabsf(d2f(x1)), y1f = fabsf(d2f(y1));
    const float ta = fabsf(G.Ff[0]) * x1f + fabsf(G.Ff[1]) * y1f + fabsf(G.Ff[2]);
    const float tb = fabsf(G.Ff[3]) * x1f + fabsf(G.Ff[4]) * y1f + fabsf(G.Ff[5]);
    const float tc = fabsf(G.Ff[6]) * x1f + fabsf(G.Ff[7]) * y1f + fabsf(G.Ff[8]);
    const float af = d2f(a), bf = d2f(b);
    const float N = sqrtf(af * af + bf * bf);
    const bool usable = isfinite(N) && finite64(c) && N > 1e-6f * (ta + tb) && N > 1e-30f;
    if (!usable) {
        // tiny or overflowing line: decide degeneracy exactly as the
        // brute force (a^2 + b^2 == 0 in its evaluation order)
        double ea, eb, ec;
        exact_line(P.F, x1, y1, ea, eb, ec);
        if (exact_norm(ea, eb) == 0.0) r.flags = EGM_FLAG_DEGENERATE_LINE;
        else r.flags = kQExactOnly;
    } else {
        const float invN = 1.0f / N;
        const double Cn = fma(a, G.cx, fma(b, G.cy, c));
        float A = af * invN, B = bf * invN, C = d2f(Cn) * invN;
        // the oracle's line differs from (a, b, c) by at most ~2 ulps of the terms
        const float da = 8.9e-16f * ta, db = 8.9e-16f * tb, dc = 8.9e-16f * tc;
        r.E0 = (da * G.cxf + db * G.cyf + dc) * invN * 1.001f;
        r.E1 = (da + db) * invN * 1.001f;
        if (G.mode == kModeAngular) {
            // distance of the computed epipole from the line, bounded
            // above: the exact line there is p . v (|v_k| <= vb_k), and
            // the brute force's line is within a few ulps of its terms
            // of the exact one
            const float xe = fabsf(G.xef), ye = fabsf(G.yef);
            const float rerr = 2.0e-15f * (ta * xe + tb * ye + tc);
            const float rv = G.vb[0] * x1f + G.vb[1] * y1f + G.vb[2];
            r.aux0 = (rv + rerr) * invN * 1.00001f + 1e-12f;
            // line direction (B, -A) in the frame of u, reduced mod pi
            r.key = fold_atan2(B * G.ux - A * G.uy, -(G.ux * A + G.uy * B));
        } else {
            float cphi = -A * G.uy + B * G.ux;
            if (cphi < 0.0f) { A = -A; B = -B; C = -C; cphi = -cphi; }
            const float sphi = fabsf(A * G.ux + B * G.uy);
            r.aux0 = cphi * (1.0f - 1e-6f);
            r.aux1 = sphi * (1.0f + 1e-6f) + 1e-12f;
            r.key = cphi > 0.5f ? -C / cphi : 0.0f;
        }
        r.A = A;
        r.B = B;
        r.C = C;
        if (!isfinite(r.C) || !isfinite(r.key)) r.flags = kQExactOnly;
    }
    L.qrec[gq] = r;
    if (L.qbkt) {
        const uint32_t b = query_bucket(G, r);
        L.qbkt[gq] = (uint16_t)b;
        if (L.qhist) L.qrank[gq] = atomicAdd(L.qhist + (int64_t)p * kQBuckets + b, 1u);
    }
    return r;
}

// The extremes over a pair's queries of what their windows are padded by, from
// a converged warp's records (valid: the lane has one), warp-aggregated; the
// warp-per-query matching kernel's per-level windows cover every query with them.
__device__ __forceinline__ void query_extremes(const Launch &L, bool valid, int p, const QueryRec &r) {
    const int lane = threadIdx.x & 31;
    const bool use = valid && r.flags == 0u;
    const uint32_t qgroup = use ? (uint32_t)p : 0xffffffffu;
    const uint32_t qa0 = use ? __float_as_uint(r.aux0) : 0u, qa1 = use ? __float_as_uint(r.aux1) : 0u;
    const uint32_t qk = use ? __float_as_uint(fabsf(r.key)) : 0u;
    if (__any_sync(0xffffffffu, qgroup != 0xffffffffu)) {
        const uint32_t qpeers = __match_any_sync(0xffffffffu, qgroup);
        const uint32_t a0x = __reduce_max_sync(qpeers, qa0);
        const uint32_t a0n = __reduce_min_sync(qpeers, qgroup == 0xffffffffu ? 0x7f800000u : qa0);
        const uint32_t a1x = __reduce_max_sync(qpeers, qa1);
        const uint32_t kx = __reduce_max_sync(qpeers, qk);
        if (qgroup != 0xffffffffu && lane == __ffs(qpeers) - 1) {
            PairGeom &G = L.geom[qgroup];
            atomicMax(&G.qa0max, a0x);
            atomicMin(&G.qa0min, a0n);
            atomicMax(&G.qa1max, a1x);
            atomicMax(&G.qkabs, kx);
        }
    }
}

}  // namespace
}  // namespace egm
