// k_prep.cu -- input quantisation and row statistics (Section 4.3, Alg. 2
// line 1: x~ = fl_l(x)), and the norms the expanded formula reuses
// (Section 3.2: p_i = x_i^T x_i "precomputed and stored").
//
// A thread, eight lanes or a warp per row, by d, alignment and the number of rows
// (quant_kind).  Output per row: the quantised row (fp16 / bf16, or
// E4M3 scaled by a power of two), and stat = (p, ||x||, ||x~||, ||x~ - x||):
//   p is ||x||^2 accumulated as an fp32 double-float (error ~2^-44) and then
//   rounded to fp32 -- the same value as binary64 rounded to fp32 except in
//   ties below 2^-44;  ||x~|| and ||x~ - x|| are fp32 sums inflated by
//   (1 + 2^-12), which covers their own rounding (gamma_d(2^-24) < 2^-12 for
//   d <= 4096), so the bound B built from them stays rigorous.  A non-zero
//   row with ||x||^2 < 2^-100 (squares near binary32's underflow) gets
//   infinite ||x~|| and ||x~ - x||: the bound is then infinite and every pair
//   of the row goes to the direct formula, as for a row that overflowed the
//   low format.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "rowstat.cuh"

namespace km {

KM_DEV float quant_val(float v, int fmt) {
    if (fmt == 0) return __half2float(__float2half_rn(v));
    if (fmt == 1) return __bfloat162float(__float2bfloat16_rn(v));
    __nv_fp8_storage_t s = __nv_cvt_float_to_fp8(v, __NV_SATFINITE, __NV_E4M3);
    __half_raw hr = __nv_cvt_fp8_to_halfraw(s, __NV_E4M3);
    return __half2float(__half(hr));
}

// Row scale of E4M3 (the per-row power-of-two scaling read into Section 4.3's
// quantisation): the smallest power of two s with amax / s <= 448 (E4M3's
// largest finite value), so the row maximum lands in (224, 448]; s is kept a
// normal fp32 number (s >= 2^-126, so 1/s is finite and x / s exact), and an
// all-zero row takes s = 1.  Exact for every fp32 amax, subnormals included:
// amax = f 2^e with f in [0.5, 1) (frexpf is exact), and 448 = 0.875 2^9, so
// s = 2^(e - 9) when f <= 0.875, else 2^(e - 8).
KM_DEV float e4m3_row_scale(float amax) {
    if (!(amax > 0.0f)) return 1.0f;
    int e;
    const float f = frexpf(amax, &e);
    const int k = max(f <= 0.875f ? e - 9 : e - 8, -126);
    return __int_as_float((k + 127) << 23);
}

// Largest |a| seen by the block's threads, folded into *out with one atomic
// per block (non-negative floats order like their bit patterns).
KM_DEV void block_absmax(float v, unsigned* out) {
    __shared__ float wmax[32];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) wmax[w] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        float m = 0.0f;
        for (int i = 0; i < (int)(blockDim.x >> 5); i++) m = fmaxf(m, wmax[i]);
        atomicMax(out, __float_as_uint(m));
    }
}

// Column maxima of the bound terms, gathered by all blocks that quantise
// centres: maxima as bit patterns (non-negative floats order like integers;
// zero to start with), minima as the complement of theirs.
struct ColAcc {
    unsigned v[10];
};
KM_DEV unsigned col_bits(float x, bool least) { return x >= 0.0f ? (least ? ~__float_as_uint(x) : __float_as_uint(x)) : 0u; }

// Where a quantised row's statistics go: stat and (nullable) rscale, and for
// centres q_j, the scale and the block's column maxima as well.
struct RowOut {
    float4* stat;
    float* rscale;
    float* qpad;    // null: points
    float* spad;
    unsigned* acc;  // shared, 10 words
    KM_DEV void operator()(int64_t i, float4 o, float s) const {
        stat[i] = o;
        if (rscale) rscale[i] = s;
        if (qpad) {
            qpad[i] = o.x;
            spad[i] = s;
            const float m[5] = {o.y, o.w, o.z, o.x, o.z * o.z};
#pragma unroll
            for (int t = 0; t < 5; t++) {
                atomicMax(&acc[t], col_bits(m[t], false));
                atomicMax(&acc[5 + t], col_bits(m[t], true));
            }
        }
    }
};

// Any d and alignment: one warp per row.
KM_DEV void quantize_warp(const float* __restrict__ A, int64_t m, int d, int fmt, int ldq, void* Aq,
                          const RowOut& out, float& amx, unsigned block, unsigned nblocks) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)block * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)nblocks * blockDim.x) >> 5;
    for (int64_t i = warp; i < m; i += nw) {
        const float* a = A + i * d;
        float s = 1.0f;
        if (fmt == 2) {
            float amax = 0.0f;
            for (int l = lane; l < d; l += 32) amax = fmaxf(amax, fabsf(a[l]));
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
            s = e4m3_row_scale(amax);
        }
        const float inv = 1.0f / s;  // exact: s is a power of two
        float ph = 0.0f, pl = 0.0f, q2 = 0.0f, r2 = 0.0f;
        bool nz = false;
        for (int l = lane; l < ldq; l += 32) {
            float v = (l < d) ? a[l] : 0.0f;
            amx = fmaxf(amx, fabsf(v));
            nz |= v != 0.0f;
            float qv = quant_val(v * inv, fmt);  // quantised value of x / s
            if (l < d) {
                df_add_sq(v, ph, pl);
                float qs = qv * s;                // x~ = s fl_l(x / s), exact scaling
                q2 = fmaf(qs, qs, q2);
                float rr = qs - v;                // exact (Sterbenz): qs and v are within a factor 2
                r2 = fmaf(rr, rr, r2);
            }
            if (fmt == 0) {
                reinterpret_cast<__half*>(Aq)[i * ldq + l] = __float2half_rn(qv);
            } else if (fmt == 1) {
                reinterpret_cast<__nv_bfloat16*>(Aq)[i * ldq + l] = __float2bfloat16_rn(qv);
            } else {
                reinterpret_cast<__nv_fp8_storage_t*>(Aq)[i * ldq + l] =
                    __nv_cvt_float_to_fp8(v * inv, __NV_SATFINITE, __NV_E4M3);
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            float oh = __shfl_xor_sync(0xffffffffu, ph, off);
            float ol = __shfl_xor_sync(0xffffffffu, pl, off);
            df_add(ph, pl, oh, ol);
            q2 += __shfl_xor_sync(0xffffffffu, q2, off);
            r2 += __shfl_xor_sync(0xffffffffu, r2, off);
        }
        const bool nzr = __any_sync(0xffffffffu, nz);
        if (lane == 0) {
            float p = ph + pl;
            float4 o;
            o.x = p;
            o.y = sqrtf(p) * kNormInflate;
            o.z = sqrtf(q2) * kNormInflate;
            o.w = sqrtf(r2) * kNormInflate;
            // an element that overflowed the low format, or squares near the
            // underflow, make the row unusable for the expanded formula: an
            // infinite bound flags all its pairs
            if (!isfinite(o.z) || (nzr && !(p >= kTinyNorm2))) { o.z = INFINITY; o.w = INFINITY; }
            out(i, o, s);
        }
    }
}


// Group path (d % 4 == 0, padded width <= 256): 8 lanes per row, 4 rows per
// warp, so the row reductions take 3 shuffle levels and serve 4 rows at once.
// Lane l of a row's 8 holds float4 l, l + 8, ... (NV of them).  Bound by issue up
// to 64 coordinates (50 instructions a row, of which 20 were the row's reduction
// and square roots by itself): R rows' reductions together took 4e6 x 64 from 364
// to 311 us (1.6 GB; 0.76 of the copy rate), 1e6 x 128 runs at 0.83 of it.
template <int NV, bool FEW>
KM_DEV void quantize_g8(const float* __restrict__ A, int64_t m, int d, int fmt, int ldq, void* Aq,
                        const RowOut& out, float& amx, unsigned block, unsigned nblocks) {
    const int lane = threadIdx.x & 31, sl = lane & 7;
    const unsigned gmask = 0xFFu << (lane & ~7);
    const int64_t gid = (((int64_t)block * blockDim.x + threadIdx.x) >> 5) * 4 + (lane >> 3);
    const int64_t ngroups = (((int64_t)nblocks * blockDim.x) >> 5) * 4;
    const int d4 = d >> 2, ldq4 = ldq >> 2;
    // R rows per group and round, all their loads issued first: at least four
    // 16-byte loads in flight per lane (FEW: no group has a second row)
    constexpr int R = FEW || NV >= 4 ? 1 : 4 / NV;
    for (int64_t i0 = gid; i0 < m; i0 += ngroups * R) {
        float4 xr[R][NV];
#pragma unroll
        for (int r = 0; r < R; r++) {
            const int64_t ir = i0 + (int64_t)r * ngroups;
            const float4* a4 = reinterpret_cast<const float4*>(A + ir * d);
#pragma unroll
            for (int u = 0; u < NV; u++) {
                const int c = sl + 8 * u;
                xr[r][u] = (ir < m && c < d4) ? a4[c] : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        float vh[R], vl[R], vq[R], vr[R], vs[R];  // the lane's part of each row's sums, the row's scale
        unsigned nzm = 0;
#pragma unroll
        for (int r = 0; r < R; r++) {
        const int64_t i = i0 + (int64_t)r * ngroups;
        float4 x[NV];
        float amax = 0.0f;
#pragma unroll
        for (int u = 0; u < NV; u++) {
            x[u] = xr[r][u];
            amax = fmaxabs3(fmaxabs3(amax, x[u].x, x[u].y), x[u].z, x[u].w);
        }
        amx = fmaxf(amx, amax);
        // (a NaN alone leaves its row out here; its bound is infinite all the same)
        nzm |= (__ballot_sync(gmask, amax > 0.0f) & gmask) != 0u ? 1u << r : 0u;
        float s = 1.0f;
        if (fmt == 2) {
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(gmask, amax, off));
            s = e4m3_row_scale(amax);
        }
        vs[r] = s;
        if (r > 0 && i >= m) {  // past the last row (the same for the group's eight lanes)
            vh[r] = vl[r] = vq[r] = vr[r] = 0.0f;
            continue;
        }
        const float inv = 1.0f / s;
        float ph = 0.0f, pl = 0.0f, q2 = 0.0f, r2 = 0.0f;
        if (fmt != 2) {
            // 16-bit formats (scale 1): packed arithmetic, two coordinates at a time
            float2 h2 = make_float2(0.f, 0.f), l2 = h2, qq2 = h2, rr2 = h2;
#pragma unroll
            for (int u = 0; u < NV; u++) {
                const int c = sl + 8 * u;
                if (c >= ldq4) continue;
                const float2 a = make_float2(x[u].x, x[u].y), b = make_float2(x[u].z, x[u].w);
                float2 qa, qb;
                uint2 w;
                if (fmt == 0) {
                    const __half2 ha = __float22half2_rn(a), hb = __float22half2_rn(b);
                    qa = __half22float2(ha);
                    qb = __half22float2(hb);
                    w.x = *reinterpret_cast<const uint32_t*>(&ha);
                    w.y = *reinterpret_cast<const uint32_t*>(&hb);
                } else {
                    const __nv_bfloat162 ha = __float22bfloat162_rn(a), hb = __float22bfloat162_rn(b);
                    qa = __bfloat1622float2(ha);
                    qb = __bfloat1622float2(hb);
                    w.x = *reinterpret_cast<const uint32_t*>(&ha);
                    w.y = *reinterpret_cast<const uint32_t*>(&hb);
                }
                reinterpret_cast<uint2*>(Aq)[i * ldq4 + c] = w;
                row_sums2(a, qa, h2, l2, qq2, rr2);
                row_sums2(b, qb, h2, l2, qq2, rr2);
            }
            ph = h2.x;
            pl = l2.x;
            df_add(ph, pl, h2.y, l2.y);
            q2 = qq2.x + qq2.y;
            r2 = rr2.x + rr2.y;
        } else
#pragma unroll
        for (int u = 0; u < NV; u++) {
            const int c = sl + 8 * u;
            if (c >= ldq4) continue;
            const float xv[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
            float qv[4];
#pragma unroll
            for (int t = 0; t < 4; t++) {
                qv[t] = quant_val(xv[t] * inv, fmt);
                df_add_sq(xv[t], ph, pl);
                const float qs = qv[t] * s;
                q2 = fmaf(qs, qs, q2);
                const float rr = qs - xv[t];
                r2 = fmaf(rr, rr, r2);
            }
            uint32_t w = 0;
#pragma unroll
            for (int t = 0; t < 4; t++)
                w |= (uint32_t)__nv_cvt_float_to_fp8(xv[t] * inv, __NV_SATFINITE, __NV_E4M3) << (8 * t);
            reinterpret_cast<uint32_t*>(Aq)[i * ldq4 + c] = w;
        }
        vh[r] = ph;
        vl[r] = pl;
        vq[r] = q2;
        vr[r] = r2;
        }
        // The rows' sums over the eight lanes, the rows shared out on the way: at each
        // level with rows left, half of the lanes go on with one half of them and hand
        // over the other (the same additions as row by row, a third of the shuffles).
        int rr = 0, left = R;  // this lane's row
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) {
            if (left > 1) {
                left >>= 1;
                const bool up = (sl & off) != 0;
                rr += up ? left : 0;
#pragma unroll
                for (int r = 0; r < R / 2; r++) {
                    if (r >= left) break;
                    const float gh = up ? vh[r] : vh[r + left], gl = up ? vl[r] : vl[r + left];
                    const float gq = up ? vq[r] : vq[r + left], gr = up ? vr[r] : vr[r + left];
                    vh[r] = up ? vh[r + left] : vh[r];
                    vl[r] = up ? vl[r + left] : vl[r];
                    vq[r] = up ? vq[r + left] : vq[r];
                    vr[r] = up ? vr[r + left] : vr[r];
                    const float oh = __shfl_xor_sync(gmask, gh, off), ol = __shfl_xor_sync(gmask, gl, off);
                    df_add(vh[r], vl[r], oh, ol);
                    vq[r] += __shfl_xor_sync(gmask, gq, off);
                    vr[r] += __shfl_xor_sync(gmask, gr, off);
                }
            } else {
                const float oh = __shfl_xor_sync(gmask, vh[0], off), ol = __shfl_xor_sync(gmask, vl[0], off);
                df_add(vh[0], vl[0], oh, ol);
                vq[0] += __shfl_xor_sync(gmask, vq[0], off);
                vr[0] += __shfl_xor_sync(gmask, vr[0], off);
            }
        }
        const int64_t i = i0 + (int64_t)rr * ngroups;
        if ((sl & (8 / R - 1)) == 0 && i < m) {
            const float p = vh[0] + vl[0];
            float4 o;
            o.x = p;
            o.y = sqrtf(p) * kNormInflate;
            o.z = sqrtf(vq[0]) * kNormInflate;
            o.w = sqrtf(vr[0]) * kNormInflate;
            // an element that overflowed the low format, or squares near the
            // underflow, make the row unusable for the expanded formula: an
            // infinite bound flags all its pairs
            if (!isfinite(o.z) || (((nzm >> rr) & 1u) && !(p >= kTinyNorm2))) { o.z = INFINITY; o.w = INFINITY; }
            float s = vs[0];
#pragma unroll
            for (int r = 1; r < R; r++) s = rr == r ? vs[r] : s;
            out(i, o, s);
        }
    }
}

// Vector path (d % 4 == 0, 256 < d <= 512): one warp per row, each lane holds up to
// NV float4 of the row in registers (coalesced 16-byte loads).
KM_DEV void quantize_vec(const float* __restrict__ A, int64_t m, int d, int fmt, int ldq, void* Aq,
                         const RowOut& out, float& amx, unsigned block, unsigned nblocks) {
    constexpr int NV = 4;
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)block * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)nblocks * blockDim.x) >> 5;
    const int d4 = d >> 2, ldq4 = ldq >> 2;
    for (int64_t i = warp; i < m; i += nw) {
        const float4* a4 = reinterpret_cast<const float4*>(A + i * d);
        float4 x[NV];
        bool nz = false;
#pragma unroll
        for (int u = 0; u < NV; u++) {
            const int c = lane + 32 * u;
            x[u] = (c < d4) ? a4[c] : make_float4(0.f, 0.f, 0.f, 0.f);
            amx = fmaxf(amx, fmaxf(fmaxf(fabsf(x[u].x), fabsf(x[u].y)), fmaxf(fabsf(x[u].z), fabsf(x[u].w))));
            nz |= (x[u].x != 0.0f) | (x[u].y != 0.0f) | (x[u].z != 0.0f) | (x[u].w != 0.0f);
        }
        const bool nzr = __any_sync(0xffffffffu, nz);
        float s = 1.0f;
        if (fmt == 2) {
            float amax = 0.0f;
#pragma unroll
            for (int u = 0; u < NV; u++)
                amax = fmaxf(amax, fmaxf(fmaxf(fabsf(x[u].x), fabsf(x[u].y)), fmaxf(fabsf(x[u].z), fabsf(x[u].w))));
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
            s = e4m3_row_scale(amax);
        }
        const float inv = 1.0f / s;
        float ph = 0.0f, pl = 0.0f, q2 = 0.0f, r2 = 0.0f;
#pragma unroll
        for (int u = 0; u < NV; u++) {
            const int c = lane + 32 * u;
            if (c >= ldq4) continue;
            const float xv[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
            float qv[4];
#pragma unroll
            for (int t = 0; t < 4; t++) {
                qv[t] = quant_val(xv[t] * inv, fmt);
                df_add_sq(xv[t], ph, pl);
                const float qs = qv[t] * s;
                q2 = fmaf(qs, qs, q2);
                const float rr = qs - xv[t];
                r2 = fmaf(rr, rr, r2);
            }
            if (fmt == 0) {
                __half2 h0 = __floats2half2_rn(qv[0], qv[1]), h1 = __floats2half2_rn(qv[2], qv[3]);
                uint2 w;
                w.x = *reinterpret_cast<uint32_t*>(&h0);
                w.y = *reinterpret_cast<uint32_t*>(&h1);
                reinterpret_cast<uint2*>(Aq)[i * ldq4 + c] = w;
            } else if (fmt == 1) {
                __nv_bfloat162 h0 = __floats2bfloat162_rn(qv[0], qv[1]), h1 = __floats2bfloat162_rn(qv[2], qv[3]);
                uint2 w;
                w.x = *reinterpret_cast<uint32_t*>(&h0);
                w.y = *reinterpret_cast<uint32_t*>(&h1);
                reinterpret_cast<uint2*>(Aq)[i * ldq4 + c] = w;
            } else {
                uint32_t w = 0;
#pragma unroll
                for (int t = 0; t < 4; t++)
                    w |= (uint32_t)__nv_cvt_float_to_fp8(xv[t] * inv, __NV_SATFINITE, __NV_E4M3) << (8 * t);
                reinterpret_cast<uint32_t*>(Aq)[i * ldq4 + c] = w;
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            float oh = __shfl_xor_sync(0xffffffffu, ph, off);
            float ol = __shfl_xor_sync(0xffffffffu, pl, off);
            df_add(ph, pl, oh, ol);
            q2 += __shfl_xor_sync(0xffffffffu, q2, off);
            r2 += __shfl_xor_sync(0xffffffffu, r2, off);
        }
        if (lane == 0) {
            float p = ph + pl;
            float4 o;
            o.x = p;
            o.y = sqrtf(p) * kNormInflate;
            o.z = sqrtf(q2) * kNormInflate;
            o.w = sqrtf(r2) * kNormInflate;
            if (!isfinite(o.z) || (nzr && !(p >= kTinyNorm2))) { o.z = INFINITY; o.w = INFINITY; }
            out(i, o, s);
        }
    }
}

// Any alignment, rows of up to 32 NCH coordinates: eight lanes per row, each
// standing for four lanes of quantize_warp (lane l = sl + 8 i of 32: the same
// sums in the same tree, so the same statistics bit for bit), four rows per warp.  A warp
// per row spent its time on reductions of mostly idle lanes: 1e5 x 10 took 27 us
// (16.8 in this form, 6.9 in quantize_row's), 700,000 x 77 290 us (137 in this one).
template <int NCH>
KM_DEV void quantize_short(const float* __restrict__ A, int64_t m, int d, int fmt, int ldq, void* Aq,
                           const RowOut& out, float& amx, unsigned block, unsigned nblocks) {
    const int lane = threadIdx.x & 31, sl = lane & 7;
    const unsigned gmask = 0xFFu << (lane & ~7);
    const int64_t ng = (int64_t)nblocks * (blockDim.x / 8);
    for (int64_t i = (int64_t)block * (blockDim.x / 8) + threadIdx.x / 8; i < m; i += ng) {
        const float* a = A + i * d;
        constexpr int NT = 4 * NCH;
        float v[NT];  // coordinate sl + 8 t
#pragma unroll
        for (int t = 0; t < NT; t++) {
            v[t] = sl + 8 * t < d ? a[sl + 8 * t] : 0.0f;
            amx = fmaxf(amx, fabsf(v[t]));
        }
        float s = 1.0f;
        if (fmt == 2) {
            float amax = 0.0f;
#pragma unroll
            for (int t = 0; t < NT; t++) amax = fmaxf(amax, fabsf(v[t]));
#pragma unroll
            for (int off = 4; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(gmask, amax, off));
            s = e4m3_row_scale(amax);
        }
        const float inv = 1.0f / s;  // exact: s is a power of two
        float ph[4], pl[4], q2[4], r2[4];
        bool nz = false;
#pragma unroll
        for (int l = 0; l < 4; l++) ph[l] = pl[l] = q2[l] = r2[l] = 0.0f;
#pragma unroll
        for (int t = 0; t < NT; t++) {
            const int c = sl + 8 * t, l = t & 3;
            if (c < ldq) {
                const float qv = quant_val(v[t] * inv, fmt);
                nz |= v[t] != 0.0f;
                if (c < d) {
                    df_add_sq(v[t], ph[l], pl[l]);
                    const float qs = qv * s;
                    q2[l] = fmaf(qs, qs, q2[l]);
                    const float rr = qs - v[t];
                    r2[l] = fmaf(rr, rr, r2[l]);
                }
                if (fmt == 0) reinterpret_cast<__half*>(Aq)[i * ldq + c] = __float2half_rn(qv);
                else if (fmt == 1) reinterpret_cast<__nv_bfloat16*>(Aq)[i * ldq + c] = __float2bfloat16_rn(qv);
                else
                    reinterpret_cast<__nv_fp8_storage_t*>(Aq)[i * ldq + c] =
                        __nv_cvt_float_to_fp8(v[t] * inv, __NV_SATFINITE, __NV_E4M3);
            }
        }
        // levels 16 and 8 of the tree lie inside the lane
#pragma unroll
        for (int h = 2; h > 0; h >>= 1)
#pragma unroll
            for (int l = 0; l < h; l++) {
                df_add(ph[l], pl[l], ph[l + h], pl[l + h]);
                q2[l] += q2[l + h];
                r2[l] += r2[l + h];
            }
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) {
            const float oh = __shfl_xor_sync(gmask, ph[0], off);
            const float ol = __shfl_xor_sync(gmask, pl[0], off);
            df_add(ph[0], pl[0], oh, ol);
            q2[0] += __shfl_xor_sync(gmask, q2[0], off);
            r2[0] += __shfl_xor_sync(gmask, r2[0], off);
        }
        const bool nzr = (__ballot_sync(gmask, nz) & gmask) != 0u;
        if (sl == 0) {
            const float p = ph[0] + pl[0];
            float4 o = make_float4(p, sqrtf(p) * kNormInflate, sqrtf(q2[0]) * kNormInflate, sqrtf(r2[0]) * kNormInflate);
            if (!isfinite(o.z) || (nzr && !(p >= kTinyNorm2))) { o.z = INFINITY; o.w = INFINITY; }
            out(i, o, s);
        }
    }
}

// Rows of at most 16 coordinates, a thread each: no shuffles, a row's low-format
// copy leaves in one or two 16-byte stores.  The same sums in the same tree as
// quantize_g8's (VEC: aligned rows, a float4 per lane there) or quantize_short's
// (else), so the same statistics bit for bit.  Eight lanes a row, of which a
// short row fills two to four, took 16.8 us at 1e5 x 10 and 59 us at 930,486 x
// 16; this form 6.9 and 19.3.
template <bool VEC>
KM_DEV void quantize_row(const float* __restrict__ A, int64_t m, int d, int fmt, int ldq, void* Aq, const RowOut& out,
                         float& amx, unsigned block, unsigned nblocks) {
    for (int64_t i = (int64_t)block * blockDim.x + threadIdx.x; i < m; i += (int64_t)nblocks * blockDim.x) {
        float v[16];
        if constexpr (VEC) {
            const float4* a4 = reinterpret_cast<const float4*>(A + i * d);
#pragma unroll
            for (int f = 0; f < 4; f++) {
                const float4 t = 4 * f < d ? a4[f] : make_float4(0.f, 0.f, 0.f, 0.f);
                v[4 * f] = t.x; v[4 * f + 1] = t.y; v[4 * f + 2] = t.z; v[4 * f + 3] = t.w;
            }
        } else {
            const float* a = A + i * d;
#pragma unroll
            for (int c = 0; c < 16; c++) v[c] = c < d ? a[c] : 0.0f;
        }
        float amax = 0.0f;
#pragma unroll
        for (int c = 0; c < 16; c += 2) amax = fmaxabs3(amax, v[c], v[c + 1]);
        amx = fmaxf(amx, amax);
        const float s = fmt == 2 ? e4m3_row_scale(amax) : 1.0f, inv = 1.0f / s;
        // partial sums: per float4 (VEC), else per coordinate pair (c, c + 8)
        constexpr int NP = VEC ? 4 : 8;
        float ph[NP], pl[NP], q2[NP], r2[NP];
        uint32_t w[8];  // the row's low-format copy
        auto put = [&](int c, float lo, float hi) {  // coordinates c, c + 1 (quantised values, scaled)
            if (fmt == 0) {
                const __half2 h = __floats2half2_rn(lo, hi);
                w[c / 2] = *reinterpret_cast<const uint32_t*>(&h);
            } else if (fmt == 1) {
                const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);
                w[c / 2] = *reinterpret_cast<const uint32_t*>(&h);
            } else {
                const uint32_t b = (uint32_t)__nv_cvt_float_to_fp8(lo, __NV_SATFINITE, __NV_E4M3) |
                                   (uint32_t)__nv_cvt_float_to_fp8(hi, __NV_SATFINITE, __NV_E4M3) << 8;
                w[c / 4] = (c & 2) ? w[c / 4] | b << 16 : b;
            }
        };
#pragma unroll
        for (int c = 0; c < 16; c += 2) put(c, v[c] * inv, v[c + 1] * inv);
        if (VEC && fmt != 2) {
#pragma unroll
            for (int f = 0; f < 4; f++) {
                float2 h2 = make_float2(0.f, 0.f), l2 = h2, qq2 = h2, rr2 = h2;
#pragma unroll
                for (int t = 0; t < 2; t++) {
                    const uint32_t u = w[2 * f + t];
                    const float2 q = fmt == 0 ? __half22float2(*reinterpret_cast<const __half2*>(&u))
                                              : __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u));
                    row_sums2(make_float2(v[4 * f + 2 * t], v[4 * f + 2 * t + 1]), q, h2, l2, qq2, rr2);
                }
                ph[f % NP] = h2.x;
                pl[f % NP] = l2.x;
                df_add(ph[f % NP], pl[f % NP], h2.y, l2.y);
                q2[f % NP] = qq2.x + qq2.y;
                r2[f % NP] = rr2.x + rr2.y;
            }
        } else {
            auto term = [&](float x, float& h, float& l, float& qq, float& rr) {
                const float qs = quant_val(x * inv, fmt) * s;
                df_add_sq(x, h, l);
                qq = fmaf(qs, qs, qq);
                const float r = qs - x;
                rr = fmaf(r, r, rr);
            };
#pragma unroll
            for (int f = 0; f < NP; f++) {
                ph[f] = pl[f] = q2[f] = r2[f] = 0.0f;
                if constexpr (VEC) {
#pragma unroll
                    for (int t = 0; t < 4; t++) term(v[(4 * f + t) % 16], ph[f], pl[f], q2[f], r2[f]);
                } else {
                    float h = 0.0f, l = 0.0f, qq = 0.0f, rr = 0.0f;
                    term(v[f], ph[f], pl[f], q2[f], r2[f]);
                    term(v[f + 8], h, l, qq, rr);
                    df_add(ph[f], pl[f], h, l);
                    q2[f] += qq;
                    r2[f] += rr;
                }
            }
        }
#pragma unroll
        for (int off = NP / 2; off > 0; off >>= 1)
#pragma unroll
            for (int f = 0; f < off; f++) {
                df_add(ph[f], pl[f], ph[f + off], pl[f + off]);
                q2[f] += q2[f + off];
                r2[f] += r2[f + off];
            }
        const int esz = fmt == 2 ? 1 : 2;
        uint4* dst = reinterpret_cast<uint4*>(reinterpret_cast<char*>(Aq) + i * ldq * esz);
        dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
        if (ldq * esz > 16) dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
        const float p = ph[0] + pl[0];
        float4 o = make_float4(p, sqrtf(p) * kNormInflate, sqrtf(q2[0]) * kNormInflate, sqrtf(r2[0]) * kNormInflate);
        if (!isfinite(o.z) || (amax > 0.0f && !(p >= kTinyNorm2))) { o.z = INFINITY; o.w = INFINITY; }
        out(i, o, s);
    }
}

// The rows of a matrix, quantised (one side of a launch).
struct QuantSide {
    const float* A;
    int64_t m;
    void* Aq;
    float4* stat;
    float* rscale;
    unsigned* absmax;  // nullable: max |a| folded in
};
// What the screen needs of the centres beside their rows.
struct ColSide {
    ColMax* out;
    float* qpad;
    float* spad;
    int kpad;
    unsigned* ticket;
    unsigned* acc;  // 10 words, 0 before and after
};

// KIND: NV of quantize_g8 (1, 2, 4, 8; few rows: 9, 10), 16
// quantize_vec, 0 quantize_warp, -NCH of quantize_short (2, 4, 8), 32 and 33 quantize_row.  The first cblocks blocks take the centres
// and form their column data (q_j, +inf on the padding so padded columns never
// win; the E4M3 scales, 1 on the padding; the column maxima, written by the
// last of them to finish); the rest take the points.  One launch instead of three: the
// centres' part, 5 to 9 us of latency by itself, hides behind the points'.
constexpr int quant_blocks(int kind) { return kind == 0 ? 6 : (kind == 8 || kind == -8 ? 3 : 4); }  // per SM
template <int KIND>
__global__ void __launch_bounds__(256, quant_blocks(KIND)) k_quantize(const QuantSide x, const QuantSide c, const ColSide col, int d, int fmt,
                                                  int ldq, int cblocks, const ZeroWords zero) {
    chain_enter();
#pragma unroll
    for (int z = 0; z < 2; z++)
        for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < zero.n[z]; i += (int64_t)gridDim.x * blockDim.x)
            zero.p[z][i] = 0u;
    __shared__ bool last;
    __shared__ unsigned acc[10];
    const bool cs = (int)blockIdx.x < cblocks;
    const QuantSide& q = cs ? c : x;
    const unsigned block = cs ? blockIdx.x : blockIdx.x - cblocks, nblocks = cs ? cblocks : gridDim.x - cblocks;
    const bool cols = cs && col.out;
    if (cols) {
        if (threadIdx.x < 10) acc[threadIdx.x] = 0u;
        __syncthreads();
    }
    const RowOut out{q.stat, q.rscale, cols ? col.qpad : nullptr, col.spad, acc};
    float amx = 0.0f;  // largest |a| of this thread's elements
    if constexpr (KIND < 0) quantize_short<-KIND>(q.A, q.m, d, fmt, ldq, q.Aq, out, amx, block, nblocks);
    else if constexpr (KIND == 0) quantize_warp(q.A, q.m, d, fmt, ldq, q.Aq, out, amx, block, nblocks);
    else if constexpr (KIND < 16) quantize_g8<(KIND < 9 ? KIND : KIND - 8), (KIND > 8)>(q.A, q.m, d, fmt, ldq, q.Aq, out, amx, block, nblocks);
    else if constexpr (KIND == 16) quantize_vec(q.A, q.m, d, fmt, ldq, q.Aq, out, amx, block, nblocks);
    else quantize_row<KIND == 32>(q.A, q.m, d, fmt, ldq, q.Aq, out, amx, block, nblocks);
    if (q.absmax) block_absmax(amx, q.absmax);
    if (!cols) return;
    if (block == 0)
        for (int j = (int)c.m + threadIdx.x; j < col.kpad; j += blockDim.x) {
            col.qpad[j] = INFINITY;
            col.spad[j] = 1.0f;
        }
    __syncthreads();
    if (threadIdx.x < 10) atomicMax(&col.acc[threadIdx.x], acc[threadIdx.x]);
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicInc(col.ticket, cblocks - 1) == (unsigned)cblocks - 1;  // back to 0 for the next call
    __syncthreads();
    if (!last || threadIdx.x != 0) return;
    __threadfence();
    float m[10];
#pragma unroll
    for (int t = 0; t < 10; t++) {
        const unsigned u = atomicExch(&col.acc[t], 0u);
        m[t] = __uint_as_float(t < 5 ? u : (u ? ~u : 0x7f800000u));
    }
    ColMax o;
    o.nc = m[0]; o.nrc = m[1]; o.ncq = m[2]; o.q = m[3]; o.ncq2 = m[4];
    o.pad[0] = o.pad[1] = o.pad[2] = 0.0f;
    o.nc_min = m[5]; o.nrc_min = m[6]; o.ncq_min = m[7]; o.q_min = m[8]; o.ncq2_min = m[9];
    o.pad2[0] = o.pad2[1] = o.pad2[2] = 0.0f;
    *col.out = o;
}

// The kernel form for rows at A (k_quantize's KIND).
static int quant_kind(const float* A, const void* Aq, int d, int ldq, int64_t rows) {
    const bool vec = (d % 4 == 0) && (ldq % 4 == 0) && ((uintptr_t)A % 16 == 0) && ((uintptr_t)Aq % 16 == 0);
    const int nv8 = (ldq / 4 + 7) / 8;
    // a thread per short row once that makes a block for every SM: 6.9 against 16.8
    // us at 1e5 x 10, 5.8 against 5.2 at 1e4 x 16
    if (ldq <= 16 && (uintptr_t)Aq % 16 == 0 && rows >= 152 * 256) return vec ? 32 : 33;
    const bool few = rows <= 152 * 16 * 32;  // groups of one round (launch_quant)
    if (vec && nv8 <= 8) return nv8 <= 1 ? (few ? 9 : 1) : (nv8 <= 2 ? (few ? 10 : 2) : (nv8 <= 4 ? 4 : 8));
    if (vec && ldq <= 512) return 16;
    return ldq <= 64 ? -2 : (ldq <= 128 ? -4 : (ldq <= 256 ? -8 : 0));
}

static cudaError_t launch_quant(int kind, const QuantSide& x, const QuantSide& c, const ColSide& col, int d, int fmt,
                                int ldq, const ZeroWords& zero, cudaStream_t st) {
    // 8 lanes or a warp per row, enough warps in flight to cover the memory latency
    const int rows = kind >= 32 ? 256 : (kind == 0 || kind >= 16 ? 8 : 32);  // per block and round
    const int64_t most = kind >= 32 ? 152 * 8 : (kind == 0 || kind >= 16 ? 152 * 64 : 152 * 16);
    const int64_t xb = x.m ? std::min<int64_t>((x.m + rows - 1) / rows, most) : 0;
    const int64_t cb = c.m ? std::min<int64_t>((c.m + rows - 1) / rows, 152) : 0;
    switch (kind) {
#define KM_Q(K)                                                                                       \
    case K: klaunch(k_quantize<K>, (unsigned)(xb + cb), 256, 0, st, x, c, col, d, fmt, ldq, (int)cb, zero); break;
        KM_Q(-2) KM_Q(-4) KM_Q(-8) KM_Q(0) KM_Q(1) KM_Q(2) KM_Q(4) KM_Q(8) KM_Q(9) KM_Q(10) KM_Q(16) KM_Q(32) KM_Q(33)
#undef KM_Q
        default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

cudaError_t launch_quantize(const float* A, int64_t m, int d, int fmt, int ldq, void* Aq, float4* stat,
                            float* rscale, cudaStream_t st, unsigned* absmax_out) {
    return launch_quant(quant_kind(A, Aq, d, ldq, m), QuantSide{A, m, Aq, stat, rscale, absmax_out}, QuantSide{}, ColSide{}, d,
                        fmt, ldq, ZeroWords{}, st);
}

cudaError_t launch_prepare(const float* X, int64_t n, void* Xq, float4* xstat, float* xscale, unsigned* absmax_out,
                           const float* C, int k, void* Cq, float4* cstat, float* cscale, ColMax* colmax, float* qpad,
                           float* spad, int kpad, unsigned* ticket, unsigned* colacc, int d, int fmt, int ldq,
                           const ZeroWords& zero, cudaStream_t st, int* nlaunch) {
    const QuantSide x{X, X ? n : 0, Xq, xstat, xscale, absmax_out}, c{C, k, Cq, cstat, cscale, nullptr};
    const ColSide col{colmax, qpad, spad, kpad, ticket, colacc};
    const int64_t rows = X ? n : k;
    const int kc = quant_kind(C, Cq, d, ldq, rows), kx = X ? quant_kind(X, Xq, d, ldq, rows) : kc;
    *nlaunch = 1;
    if (kx == kc) return launch_quant(kc, x, c, col, d, fmt, ldq, zero, st);
    // points and centres aligned differently: each in its own form
    *nlaunch = 2;
    const cudaError_t e = launch_quant(kx, x, QuantSide{}, col, d, fmt, ldq, ZeroWords{}, st);
    return e != cudaSuccess ? e : launch_quant(kc, QuantSide{}, c, col, d, fmt, ldq, zero, st);
}

// ---- candidate-count prediction (the choice of the low format) ----------
// For a sample of rows: the fp32 direct distances to every centre, the row's
// certification window W = 2 B_max of the format (B_max from the row's
// quantisation statistics and the column maxima of the centres' ones, as the
// screening kernel forms it), and the number of centres within W of the
// row's minimum: the candidates the screen keeps for that row.  A row whose
// candidates exceed one epilogue group's list (TC_LIST entries) is counted
// as an overflow.  acc[0] += candidates, acc[1] += overflowing rows.
__global__ void __launch_bounds__(256) k_predict_candidates(const float* __restrict__ X, int64_t n, int d,
                                                            const float* __restrict__ C, int k, int fmt,
                                                            const ColMax* __restrict__ cmx, TestParams tp, int64_t stride,
                                                            int nsample, unsigned long long* acc) {
    chain_enter();
    extern __shared__ float xs[];
    __shared__ float red[8];
    __shared__ float sh_stat[4];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const ColMax cm = *cmx;
    for (int sidx = blockIdx.x; sidx < nsample; sidx += gridDim.x) {
        const int64_t i = (int64_t)sidx * stride;
        __syncthreads();
        for (int l = t; l < d; l += blockDim.x) xs[l] = X[i * d + l];
        __syncthreads();
        // the row's statistics in the format (warp 0): ||x||^2, ||x~||, ||x~ - x||
        if (w == 0) {
            float amax = 0.0f;
            for (int l = lane; l < d; l += 32) amax = fmaxf(amax, fabsf(xs[l]));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
            const float s = fmt == 2 ? e4m3_row_scale(amax) : 1.0f;
            float p = 0.0f, q2 = 0.0f, r2 = 0.0f;
            for (int l = lane; l < d; l += 32) {
                const float v = xs[l];
                const float qs = quant_val(v / s, fmt) * s;
                p = fmaf(v, v, p);
                q2 = fmaf(qs, qs, q2);
                r2 = fmaf(qs - v, qs - v, r2);
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                p += __shfl_xor_sync(0xffffffffu, p, o);
                q2 += __shfl_xor_sync(0xffffffffu, q2, o);
                r2 += __shfl_xor_sync(0xffffffffu, r2, o);
            }
            if (lane == 0) {
                sh_stat[0] = p;
                sh_stat[1] = sqrtf(q2) * kNormInflate;
                sh_stat[2] = sqrtf(r2) * kNormInflate;
            }
        }
        // fp32 direct distances: the row minimum first
        float mn = INFINITY;
        for (int j = t; j < k; j += blockDim.x) {
            const float* c = C + (int64_t)j * d;
            float acc2 = 0.0f;
            for (int l = 0; l < d; l++) {
                const float u = xs[l] - c[l];
                acc2 = fmaf(u, u, acc2);
            }
            mn = fminf(mn, acc2);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        if (lane == 0) red[w] = mn;
        __syncthreads();
        mn = red[0];
        for (int q = 1; q < (int)(blockDim.x >> 5); q++) mn = fminf(mn, red[q]);
        const float p = sh_stat[0], nxq = sh_stat[1], nrx = sh_stat[2];
        const float bmax = (2.0f * nrx * cm.nc + 2.0f * nxq * cm.nrc + tp.kacc * nxq * cm.ncq + tp.kn * (p + cm.q)) * tp.bsafe;
        const float lim = mn + 2.0f * bmax * 1.001f;
        unsigned cntc = 0;
        for (int j = t; j < k; j += blockDim.x) {
            const float* c = C + (int64_t)j * d;
            float acc2 = 0.0f;
            for (int l = 0; l < d; l++) {
                const float u = xs[l] - c[l];
                acc2 = fmaf(u, u, acc2);
            }
            cntc += acc2 <= lim ? 1u : 0u;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) cntc += __shfl_xor_sync(0xffffffffu, cntc, o);
        __syncthreads();
        if (lane == 0) reinterpret_cast<unsigned*>(red)[w] = cntc;
        __syncthreads();
        if (t == 0) {
            unsigned tot = 0;
            for (int q = 0; q < (int)(blockDim.x >> 5); q++) tot += reinterpret_cast<unsigned*>(red)[q];
            atomicAdd(&acc[0], (unsigned long long)tot);
            if (tot > (unsigned)TC_LIST) atomicAdd(&acc[1], 1ull);
        }
    }
}

cudaError_t launch_predict_candidates(const float* X, int64_t n, int d, const float* C, int k, int fmt,
                                      const ColMax* cmx, const TestParams& tp, int nsample,
                                      unsigned long long* acc, int num_sms, cudaStream_t st) {
    const int64_t stride = std::max<int64_t>(1, n / nsample);
    const int ns = (int)std::min<int64_t>(nsample, (n + stride - 1) / stride);
    const size_t sm = (size_t)d * sizeof(float);
    cudaError_t e = allow_max_smem(k_predict_candidates);
    if (e != cudaSuccess) return e;
    klaunch(k_predict_candidates, (unsigned)std::max(1, std::min(ns, num_sms * 4)), 256, sm, st, X, n, d, C, k, fmt, cmx, tp,
                                                                                           stride, ns, acc);
    return cudaGetLastError();
}

}  // namespace km
