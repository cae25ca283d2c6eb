// rowstat.cuh -- the statistics of a quantised row that the bound behind the
// reliability test needs, and the centred bf16 rows of the second screen.
#pragma once
#include <cuda_bf16.h>

#include "common.cuh"
#include "df.cuh"
#include "internal.h"

namespace km {

constexpr float kNormInflate = 1.0f + 1.0f / 4096.0f;
constexpr float kTinyNorm2 = 0x1p-100f;  // below this ||x||^2 the fp32 statistics are not trusted

// Two coordinates (scale 1, 16-bit formats) into the row's running sums, two
// per packed instruction: ||x||^2 as a pair of double-floats (exact product,
// two-sum), ||x~||^2 and ||x~ - x||^2 in fp32.
KM_DEV void row_sums2(float2 x, float2 q, float2& hi, float2& lo, float2& qq, float2& rr) {
    // (differences as fused products with -1: the packed operations take no sign)
    const float2 m1 = make_float2(-1.0f, -1.0f);
    const float2 nx = __fmul2_rn(x, m1), np = __fmul2_rn(nx, x);  // -x, -p with p = fl(x^2)
    const float2 pe = __ffma2_rn(x, x, np);
    const float2 s = __ffma2_rn(np, m1, hi);
    const float2 bb = __ffma2_rn(hi, m1, s);
    const float2 e1 = __ffma2_rn(__ffma2_rn(bb, m1, s), m1, hi);
    const float2 e = __ffma2_rn(__fadd2_rn(np, bb), m1, e1);
    hi = s;
    lo = __fadd2_rn(lo, __fadd2_rn(e, pe));
    qq = __ffma2_rn(q, q, qq);
    const float2 r = __fadd2_rn(q, nx);  // exact (Sterbenz)
    rr = __ffma2_rn(r, r, rr);
}

// Column maxima and minima of the centres' statistics (one block).
KM_DEV void colmax_block(const float4* cstat, int k, ColMax* out) {
    __shared__ float red[10][32];
    float a = 0, b = 0, c = 0, q = 0, c2 = 0;
    float an = INFINITY, bn = INFINITY, cn = INFINITY, qn = INFINITY, c2n = INFINITY;
    for (int j = threadIdx.x; j < k; j += blockDim.x) {
        const float4 s = __ldcg(cstat + j);  // (centred centres: written by other blocks of the launch)
        a = fmaxf(a, s.y);
        b = fmaxf(b, s.w);
        c = fmaxf(c, s.z);
        q = fmaxf(q, s.x);
        c2 = fmaxf(c2, s.z * s.z);
        an = fminf(an, s.y);
        bn = fminf(bn, s.w);
        cn = fminf(cn, s.z);
        qn = fminf(qn, s.x);
        c2n = fminf(c2n, s.z * s.z);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, off));
        b = fmaxf(b, __shfl_xor_sync(0xffffffffu, b, off));
        c = fmaxf(c, __shfl_xor_sync(0xffffffffu, c, off));
        q = fmaxf(q, __shfl_xor_sync(0xffffffffu, q, off));
        c2 = fmaxf(c2, __shfl_xor_sync(0xffffffffu, c2, off));
        an = fminf(an, __shfl_xor_sync(0xffffffffu, an, off));
        bn = fminf(bn, __shfl_xor_sync(0xffffffffu, bn, off));
        cn = fminf(cn, __shfl_xor_sync(0xffffffffu, cn, off));
        qn = fminf(qn, __shfl_xor_sync(0xffffffffu, qn, off));
        c2n = fminf(c2n, __shfl_xor_sync(0xffffffffu, c2n, off));
    }
    const int w = threadIdx.x >> 5, ln = threadIdx.x & 31;
    if (ln == 0) {
        red[0][w] = a; red[1][w] = b; red[2][w] = c; red[3][w] = q; red[4][w] = c2;
        red[5][w] = an; red[6][w] = bn; red[7][w] = cn; red[8][w] = qn; red[9][w] = c2n;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < (int)(blockDim.x / 32); i++) {
            a = fmaxf(a, red[0][i]); b = fmaxf(b, red[1][i]); c = fmaxf(c, red[2][i]);
            q = fmaxf(q, red[3][i]); c2 = fmaxf(c2, red[4][i]);
            an = fminf(an, red[5][i]); bn = fminf(bn, red[6][i]); cn = fminf(cn, red[7][i]);
            qn = fminf(qn, red[8][i]); c2n = fminf(c2n, red[9][i]);
        }
        ColMax o;
        o.nc = a; o.nrc = b; o.ncq = c; o.q = q; o.ncq2 = c2;
        o.pad[0] = o.pad[1] = o.pad[2] = 0.0f;
        o.nc_min = an; o.nrc_min = bn; o.ncq_min = cn; o.q_min = qn; o.ncq2_min = c2n;
        o.pad2[0] = o.pad2[1] = o.pad2[2] = 0.0f;
        *out = o;
    }
}

// ---- centred rows ----------------------------------------------------------
// Distances do not change when mu is taken from both sides, but the norms that
// the bound grows with do: rows that the plain screen cannot decide (data far
// from the origin, an 8-bit format on wide data, values past fp16's range) are
// screened again as bf16 copies of x - mu against c - mu.
//
// mu: the mean of up to 32 centres spread over C, the same bits wherever it is
// formed (any vector is a valid one).  All threads of the block take part;
// mu[l] = 0 for d <= l < ldq.
KM_DEV void centre_mean(const float* __restrict__ C, int k, int d, int ldq, float* mu) {
    const int m = k < 32 ? k : 32;
    const int64_t step = (int64_t)(k / m) * d;
    for (int l = threadIdx.x; l < ldq; l += blockDim.x) {
        float s = 0.0f;
        if (l < d) {
#pragma unroll 8
            for (int t = 0; t < m; t++) s = __fadd_rn(s, C[t * step + l]);
            s = __fdiv_rn(s, (float)m);
        }
        mu[l] = s;
    }
    __syncthreads();
}

// One centred row by eight lanes (sl of 8, gmask their lanes): y = fl(a - mu)
// in bf16 to dst (ldq entries, zero past d) and the statistics of y as in
// k_prep.cu.  y's own rounding (2^-24 relative per coordinate) moves a squared
// distance by at most 4 2^-24 (p + q): the caller's k_n covers it.
template <bool VEC>
KM_DEV void centred_row(const float* __restrict__ a, const float* mu, int d, int ldq, __nv_bfloat16* __restrict__ dst,
                        float4* __restrict__ stat, int sl, unsigned gmask) {
    float2 h2 = make_float2(0.f, 0.f), l2 = h2, qq2 = h2, rr2 = h2;
    bool nz = false;
    const int ldq4 = ldq >> 2;
    for (int c0 = sl; c0 < ldq4; c0 += 32) {
        float4 xs[4];  // four chunks' loads in flight
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int c = c0 + 8 * i;
            xs[i] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (VEC) {
                if (4 * c < d) xs[i] = reinterpret_cast<const float4*>(a)[c];
            } else {
                if (4 * c + 0 < d) xs[i].x = a[4 * c + 0];
                if (4 * c + 1 < d) xs[i].y = a[4 * c + 1];
                if (4 * c + 2 < d) xs[i].z = a[4 * c + 2];
                if (4 * c + 3 < d) xs[i].w = a[4 * c + 3];
            }
        }
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int c = c0 + 8 * i;
            if (c >= ldq4) break;
            const float4 x = xs[i], m4 = reinterpret_cast<const float4*>(mu)[c];
            const float2 u = fsub2(make_float2(x.x, x.y), make_float2(m4.x, m4.y));
            const float2 v = fsub2(make_float2(x.z, x.w), make_float2(m4.z, m4.w));
            nz |= (u.x != 0.0f) | (u.y != 0.0f) | (v.x != 0.0f) | (v.y != 0.0f);
            const __nv_bfloat162 hu = __float22bfloat162_rn(u), hv = __float22bfloat162_rn(v);
            uint2 w;
            w.x = *reinterpret_cast<const uint32_t*>(&hu);
            w.y = *reinterpret_cast<const uint32_t*>(&hv);
            reinterpret_cast<uint2*>(dst)[c] = w;
            row_sums2(u, __bfloat1622float2(hu), h2, l2, qq2, rr2);
            row_sums2(v, __bfloat1622float2(hv), h2, l2, qq2, rr2);
        }
    }
    float ph = h2.x, pl = l2.x;
    df_add(ph, pl, h2.y, l2.y);
    float q2 = qq2.x + qq2.y, r2 = rr2.x + rr2.y;
    const bool nzr = (__ballot_sync(gmask, nz) & gmask) != 0u;
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {
        const float oh = __shfl_xor_sync(gmask, ph, off), ol = __shfl_xor_sync(gmask, pl, off);
        df_add(ph, pl, oh, ol);
        q2 += __shfl_xor_sync(gmask, q2, off);
        r2 += __shfl_xor_sync(gmask, r2, off);
    }
    if (sl == 0) {
        const float p = ph + pl;
        float4 o = make_float4(p, sqrtf(p) * kNormInflate, sqrtf(q2) * kNormInflate, sqrtf(r2) * kNormInflate);
        if (!isfinite(o.z) || (nzr && !(p >= kTinyNorm2))) { o.z = INFINITY; o.w = INFINITY; }
        *stat = o;
    }
}

}  // namespace km
