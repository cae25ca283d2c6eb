// k_refine.cu -- recompute by the direct formula (Section 4.3: from the
// ORIGINAL data, Eq. (fallback-rule-mp)) and certified argmin.
//
// The screening kernel leaves, per row, lists of candidates, from which only
// the j with d^_j <= d^_min + 2 B_max can still be the nearest centre, where
// |d^_j - d_j| <= B_ij is the bound behind the reliability test (so no other
// centre can win).  One candidate is the argmin.  Of several, Eq.
// (dist-direct) in fp32 and Theorem 4.1, which puts each true value in
// [v (1 - g), v (1 + g)], g = gamma_{d+2}(2^-24): when exactly one interval
// can hold the minimum, that centre is the argmin; otherwise (near-ties) the
// open candidates are evaluated in binary64 (products and sums rounded
// separately, coordinates in order: the oracle's own arithmetic), lowest index
// on ties.  Rows whose list overflowed are listed for the centred screen
// (k_centre_rows prepares them) or the full-row kernel.
//
// Two forms with the same results:
//  * k_refine: one launch, 4, 8 or 32 rows per warp;
//  * more than 64 coordinates and n d > 2^25: k_cand_select (a flat list of
//    (row, j) pairs, each row's contiguous, from the rows' lists), k_pair_eval
//    (8 lanes per pair, 4 pairs per warp, no per-row bookkeeping), k_certify
//    (one thread per row) and k_amb_fp64.
// Measured, k_refine against the four launches (GPU time, without the gaps
// between launches): 1000 x 32 5.5 / 15.0 us, 1e4 x 16 5.6 / 16.3 us, 1e5 x 128
// 19.8 / 28.7 us, 4e6 x 64 206 / 260 us; 150,001 x 256 92 / 72 us, 1e6 x 128
// 293 / 219 us (x and two centres in registers leave three blocks per SM).

#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "rowstat.cuh"

namespace km {

// fp32 direct values of the candidate pairs.  NV float4 of a row per lane
// (lane l of a pair's 8 takes float4 l, l + 8, ...); NV == 0: scalar loads
// for any d and alignment.  A group of eight lanes takes two pairs per round
// (pi and pi + G, G the number of groups), all their loads issued first.
template <int NV>
KM_DEV float pair_value(const float* __restrict__ X, const float* __restrict__ C, int d, int2 pr, int sl) {
    float acc = 0.0f;
    if (NV > 0) {
        const int d4 = d >> 2;
        const float4* x4 = reinterpret_cast<const float4*>(X + (int64_t)pr.x * d);
        const float4* c4 = reinterpret_cast<const float4*>(C + (int64_t)pr.y * d);
#pragma unroll
        for (int u = 0; u < NV; u++) {
            const int c = sl + 8 * u;
            const float4 xv = (c < d4) ? x4[c] : make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 cv = (c < d4) ? c4[c] : make_float4(0.f, 0.f, 0.f, 0.f);
            const float t0 = xv.x - cv.x, t1 = xv.y - cv.y, t2 = xv.z - cv.z, t3 = xv.w - cv.w;
            acc = fmaf(t0, t0, acc);
            acc = fmaf(t1, t1, acc);
            acc = fmaf(t2, t2, acc);
            acc = fmaf(t3, t3, acc);
        }
    } else {
        const float* x = X + (int64_t)pr.x * d;
        const float* c = C + (int64_t)pr.y * d;
        for (int l = sl; l < d; l += 8) {
            const float t = x[l] - c[l];
            acc = fmaf(t, t, acc);
        }
    }
    return acc;
}

template <int NV>
__global__ void __launch_bounds__(256) k_pair_eval(const float* __restrict__ X, const float* __restrict__ C, int d,
                                                   const int2* __restrict__ pairs,
                                                   const unsigned long long* __restrict__ npairs, int64_t cap,
                                                   float* __restrict__ v32) {
    chain_enter();
    const int lane = threadIdx.x & 31, sl = lane & 7, gbase = lane & ~7;
    const unsigned gmask = 0xFFu << gbase;
    const int64_t gid = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 4 + (lane >> 3);
    const int64_t ngroups = (((int64_t)gridDim.x * blockDim.x) >> 5) * 4;
    const int64_t np = min((int64_t)*npairs, cap);
    for (int64_t pi = gid; pi < np; pi += 2 * ngroups) {
        const int64_t pj = pi + ngroups;
        const int2 pa = pairs[pi];
        const int2 pb = pj < np ? pairs[pj] : make_int2(-1, 0);
        // a slot of a row that did not fit is marked row -1 (the group's eight lanes alike)
        float va = pa.x >= 0 ? pair_value<NV>(X, C, d, pa, sl) : 0.0f;
        float vb = pb.x >= 0 ? pair_value<NV>(X, C, d, pb, sl) : 0.0f;
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) {
            va += __shfl_xor_sync(gmask, va, off);
            vb += __shfl_xor_sync(gmask, vb, off);
        }
        if (sl == 0) {
            if (pa.x >= 0) v32[pi] = va;
            if (pb.x >= 0) v32[pj] = vb;
        }
    }
}

// Candidate selection, one thread per row: the quad entries of every epilogue
// group's list inside the window of the row's final d^ minimum (the smallest
// of the groups' minima), each masked column written out as a (row, j) pair,
// contiguous per row, one atomic reservation per block.  Rows whose list
// overflowed, or that no longer fit in the pair buffer, get count -1
// (whole-row recompute).  A row with a single candidate is decided here: the
// window holds every centre that can be the nearest, so that one is; its
// label is written and its count is 0 (no evaluation: every caller refines
// the winner's distance afterwards, to binary64 accuracy).
__global__ void __launch_bounds__(256) k_cand_select(const int2* __restrict__ rowinfo, const float* __restrict__ roww,
                                                     const uint32_t* __restrict__ cand, int64_t n, int ng, int ebits,
                                                     int2* __restrict__ pairs, int64_t cap,
                                                     int2* __restrict__ rowpair, int32_t* __restrict__ labels,
                                                     DevCounters* cnt) {
    chain_enter();
    const int lane = threadIdx.x & 31;
    const uint32_t emask = (1u << ebits) - 1u;
    const float lscale = __uint_as_float((uint32_t)(127 + ebits - 23) << 23);  // 2^(ebits - 23)
    // rounds of blockDim rows per block, the same count in every warp (the
    // reservation synchronises the block)
    for (int64_t b0 = (int64_t)blockIdx.x * blockDim.x; b0 < n; b0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t row = b0 + threadIdx.x;
        const bool valid = row < n;
        int c = 0;
        bool full = false;
        int cnt_g[TC_GROUPS];
        float lim = 0.0f;
        // slot s of group g at cand[(g * TC_LIST + s) * n + row]: a warp reads 32 rows side by side
        const uint32_t* c0 = cand + row;
        unsigned msk[TC_GROUPS];  // entries inside the window, per group
        {
            float dmin = INFINITY;
            const float W = valid ? roww[row] : 0.0f;
#pragma unroll
            for (int g = 0; g < TC_GROUPS; g++) {
                const int2 ig = valid && g < ng ? rowinfo[(size_t)g * n + row] : make_int2(0, __float_as_int(INFINITY));
                full |= (ig.x & ROW_OVERFLOW) != 0;
                cnt_g[g] = ig.x & (ROW_OVERFLOW - 1);
                dmin = fminf(dmin, __int_as_float(ig.y));
            }
            lim = dmin + W;
            // an infinite window (or nothing comparable) takes in the columns' padding too: the whole row
            full |= !(lim < INFINITY);
        }
        // the first SPEC slots of every list in one round of loads, the rest (rare) after
        constexpr int SPEC = (16 / TC_GROUPS < TC_LIST) ? 16 / TC_GROUPS : TC_LIST;
#pragma unroll
        for (int g = 0; g < TC_GROUPS; g++) {
            const int cg_n = full ? 0 : cnt_g[g];
            const uint32_t* cg = c0 + (size_t)g * TC_LIST * n;
            uint32_t eg[SPEC];
#pragma unroll
            for (int s = 0; s < SPEC; s++) eg[s] = (s < cg_n) ? cg[(size_t)s * n] : 0u;
            unsigned m = 0;
#pragma unroll
            for (int s = 0; s < SPEC; s++) {
                const bool in = s < cg_n && cand_lower(eg[s], emask, lscale) <= lim;
                m |= in ? (1u << s) : 0u;
                c += in ? __popc(entry_mask(eg[s])) : 0;
            }
            for (int s = SPEC; s < cg_n; s++) {
                const uint32_t e = cg[(size_t)s * n];
                const bool in = cand_lower(e, emask, lscale) <= lim;
                m |= in ? (1u << s) : 0u;
                c += in ? __popc(entry_mask(e)) : 0;
            }
            msk[g] = m;
        }
        const bool single = valid && !full && c == 1;
        if (single) c = 0;  // decided: nothing to evaluate
        // one reservation per block: lane prefix sums, then warp totals through
        // shared memory (every warp of the block takes part in each round)
        int incl = c;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, incl, off);
            if (lane >= off) incl += o;
        }
        __shared__ int wtot[8];
        __shared__ unsigned long long bbase;
        const int wib = threadIdx.x >> 5;
        if (lane == 31) wtot[wib] = incl;
        __syncthreads();
        int wpre = 0, btot = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
            wpre += (w < wib) ? wtot[w] : 0;
            btot += wtot[w];
        }
        if (threadIdx.x == 0) bbase = btot ? atomicAdd(&cnt->npairs, (unsigned long long)btot) : 0ull;
        __syncthreads();
        const int64_t off0 = (int64_t)bbase + wpre + incl - c;
        const bool fits = off0 + c <= cap;
        if (single) {
#pragma unroll
            for (int g = 0; g < TC_GROUPS; g++) {
                if (msk[g]) {
                    const uint32_t e = c0[((size_t)g * TC_LIST + (__ffs(msk[g]) - 1)) * n];
                    labels[row] = 4 * entry_quad(e, emask) + __ffs(entry_mask(e)) - 1;
                }
            }
            rowpair[row] = make_int2(0, 0);
        } else if (valid) {
            if (!full && !fits) {
                // reserved but past the capacity: the part of the range below the
                // capacity is marked empty (row -1), so the evaluation skips it
                for (int64_t t = off0; t < off0 + c && t < cap; t++) pairs[t] = make_int2(-1, 0);
            }
            if (!full && fits) {
                int w = 0;
#pragma unroll
                for (int g = 0; g < TC_GROUPS; g++) {
                    const uint32_t* cg = c0 + (size_t)g * TC_LIST * n;
                    for (unsigned m = msk[g]; m; m &= m - 1) {
                        const uint32_t e = cg[(size_t)(__ffs(m) - 1) * n];
                        const int j0 = 4 * entry_quad(e, emask);
                        for (unsigned b = entry_mask(e); b; b &= b - 1) pairs[off0 + w++] = make_int2((int)row, j0 + __ffs(b) - 1);
                    }
                }
            }
            rowpair[row] = make_int2(fits ? (int)off0 : 0, (full || !fits) ? -1 : c);
        }
    }
}

// Certification, one thread per row, by Theorem 4.1's intervals: the winner's
// fp32 value and index; where more than one interval can hold the minimum,
// those candidates in binary64 (the oracle's arithmetic), lowest index on
// ties.  Rows with count -1 go on full_list for the full-row kernel.
__global__ void __launch_bounds__(256) k_certify(const int2* __restrict__ rowpair, int64_t n,
                                                 const int2* __restrict__ pairs, const float* __restrict__ v32,
                                                 const float* __restrict__ X, const float* __restrict__ C, int d,
                                                 float gamma32, int32_t* __restrict__ labels,
                                                 double* __restrict__ min_dist, int32_t* __restrict__ full_list,
                                                 int32_t* __restrict__ amb_list, DevCounters* cnt) {
    chain_enter();
    unsigned long long ev32 = 0, amb = 0, ovf_rows = 0;
    const float g = gamma32, tiny = direct_tiny(d);
    for (int64_t row = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; row < n;
         row += (int64_t)gridDim.x * blockDim.x) {
        const int2 rp = rowpair[row];
        if (rp.y == 0) continue;  // a single candidate: labelled by the selection
        if (rp.y < 0) {
            ovf_rows++;
            const int slot = atomicAdd(&cnt->ovf_count, 1);
            full_list[slot] = (int32_t)row;
            continue;
        }
        float up = INFINITY;
        for (int r = 0; r < rp.y; r++) up = fminf(up, direct_upper(v32[rp.x + r], g, tiny));
        int open = 0, bj = 0x7fffffff;
        float bv = INFINITY;
        for (int r = 0; r < rp.y; r++) {
            const float v = v32[rp.x + r];
            if (direct_lower(v, g) <= up) {
                open++;
                const int j = pairs[rp.x + r].y;
                if (v < bv || (v == bv && j < bj)) { bv = v; bj = j; }
            }
        }
        ev32 += (unsigned long long)rp.y;
        if (open == 1) {
            labels[row] = bj;
            min_dist[row] = (double)bv;
            continue;
        }
        amb++;
        const int slot = atomicAdd(&cnt->amb_count, 1);
        amb_list[slot] = (int32_t)row;
    }

#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        ev32 += __shfl_xor_sync(0xffffffffu, ev32, off);
        amb += __shfl_xor_sync(0xffffffffu, amb, off);
        ovf_rows += __shfl_xor_sync(0xffffffffu, ovf_rows, off);
    }
    if ((threadIdx.x & 31) == 0) {
        if (ev32) atomicAdd(&cnt->fp32_evals, ev32);
        if (amb) atomicAdd(&cnt->amb_rows, amb);
        if (ovf_rows) atomicAdd(&cnt->ovf_rows, ovf_rows);
    }
}

// Near-tie rows (listed by k_certify): one warp per row.  The candidates
// whose fp32 interval can still hold the minimum are taken AMB_B at a time:
// the warp stages x and their centre rows in shared memory and forms every
// binary64 product (x_l - c_l)^2 in parallel (each is one rounding, whatever
// the order); then one lane per candidate adds its products in coordinate
// order, one rounding per addition: the oracle's sequential sum.  The warp
// then takes the smallest value, lowest index on ties.
constexpr int AMB_B = 4;
__global__ void __launch_bounds__(256) k_amb_fp64(const int32_t* __restrict__ amb_list, const int* __restrict__ amb_count,
                                                  const int2* __restrict__ rowpair, const int2* __restrict__ pairs,
                                                  const float* __restrict__ v32, const float* __restrict__ X,
                                                  const float* __restrict__ C, int d, float gamma32,
                                                  int32_t* __restrict__ labels, double* __restrict__ min_dist,
                                                  DevCounters* cnt) {
    chain_enter();
    extern __shared__ double amb_sm[];  // per warp: AMB_B x d products
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    double* prod = amb_sm + (size_t)wib * AMB_B * d;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int na = *amb_count;
    const float g = gamma32, tiny = direct_tiny(d);
    unsigned long long ev64 = 0;
    for (int64_t t = w0; t < na; t += nw) {
        const int64_t row = amb_list[t];
        const int2 rp = rowpair[row];
        float up = INFINITY;
        for (int r = lane; r < rp.y; r += 32) up = fminf(up, direct_upper(v32[rp.x + r], g, tiny));
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) up = fminf(up, __shfl_xor_sync(0xffffffffu, up, off));
        const float* x = X + row * d;
        double best = INFINITY;
        int bj = 0x7fffffff;
        // the open candidates, AMB_B per batch (warp-uniform loop over the row's pairs)
        int r = 0;
        while (true) {
            int js[AMB_B] = {};
            int nb = 0;
            for (; r < rp.y && nb < AMB_B; r++)
                if (direct_lower(v32[rp.x + r], g) <= up) js[nb++] = pairs[rp.x + r].y;
            if (nb == 0) break;
            __syncwarp();
            // lanes over the coordinates (coalesced loads, no index division)
#pragma unroll
            for (int b = 0; b < AMB_B; b++) {
                if (b < nb) {
                    const float* c = C + (int64_t)js[b] * d;
                    for (int l = lane; l < d; l += 32) {
                        const double u = __dsub_rn((double)x[l], (double)c[l]);
                        prod[b * d + l] = __dmul_rn(u, u);
                    }
                }
            }
            __syncwarp();
            if (lane < nb) {
                const double* pp = prod + (size_t)lane * d;
                double sacc = 0.0;
                for (int l = 0; l < d; l++) sacc = __dadd_rn(sacc, pp[l]);
                int j = js[0];
#pragma unroll
                for (int q = 1; q < AMB_B; q++)
                    if (lane == q) j = js[q];
                ev64++;
                if (sacc < best || (sacc == best && j < bj)) { best = sacc; bj = j; }
            }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            const double ob = __shfl_xor_sync(0xffffffffu, best, off);
            const int oj = __shfl_xor_sync(0xffffffffu, bj, off);
            if (ob < best || (ob == best && oj < bj)) { best = ob; bj = oj; }
        }
        if (lane == 0) {
            labels[row] = bj != 0x7fffffff ? bj : pairs[rp.x].y;  // (not a number: a valid label all the same)
            min_dist[row] = best;
        }
        __syncwarp();
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) ev64 += __shfl_xor_sync(0xffffffffu, ev64, off);
    if (lane == 0 && ev64) atomicAdd(&cnt->fp64_evals, ev64);
}

// The candidates of a row that the fp32 values vs[0 .. total) leave open (their interval
// reaches up), in binary64 by a warp.  Returns the lane's evaluations.
KM_DEV unsigned refine_row_exact(const float* __restrict__ x, const float* __restrict__ C, int d, int total, float g, float up,
                                 int32_t* __restrict__ label, const int* js, const float* vs, double* prod) {
    const int lane = threadIdx.x & 31;
    unsigned ev64 = 0;
    // two candidates at a time: products by all lanes, a lane each adds one's
    double best = INFINITY;
    int bj = 0x7fffffff;
    for (int t = 0; t < total;) {
        int jc[2] = {0, 0}, nc = 0;
        for (; t < total && nc < 2; t++)
            if (direct_lower(vs[t], g) <= up) {
                jc[1] = js[t];
                if (nc++ == 0) jc[0] = jc[1];
            }
#pragma unroll
        for (int c = 0; c < 2; c++) {
            if (c >= nc) break;
            const float* cj = C + (int64_t)jc[c] * d;
            for (int l = lane; l < d; l += 32) {
                const double u = __dsub_rn((double)x[l], (double)cj[l]);
                prod[c * d + l] = __dmul_rn(u, u);
            }
        }
        __syncwarp();
        if (lane < nc) {
            const double* p = prod + lane * d;
            const int j = lane ? jc[1] : jc[0];
            double s = 0.0;
#pragma unroll 8
            for (int l = 0; l < d; l++) s = __dadd_rn(s, p[l]);
            ev64++;
            if (s < best || (s == best && j < bj)) { best = s; bj = j; }
        }
        __syncwarp();
    }
    const double ob = __shfl_xor_sync(0xffffffffu, best, 1);
    const int oj = __shfl_xor_sync(0xffffffffu, bj, 1);
    if (ob < best || (ob == best && oj < bj)) bj = oj;
    if (lane == 0) *label = bj != 0x7fffffff ? bj : js[0];  // (not a number: a valid label all the same)
    return ev64;
}

// Out of line where the rows' coordinates are in registers, for few rows come this far
// (4e6 x 64, k = 256, refinement with the winners' distances: bf16 497 us, 501 with the
// fp32 part out of line as well, 510 with nothing; e4m3, where more rows take the
// fp32 part, 908, 935 and 915), in line where they are not (500,000 x 50: 187 us, 203).
__device__ __noinline__ unsigned refine_row_exact_call(const float* __restrict__ x, const float* __restrict__ C, int d, int total,
                                                       float g, float up, int32_t* __restrict__ label, const int* js,
                                                       const float* vs, double* prod) {
    return refine_row_exact(x, C, d, total, g, up, label, js, vs, prod);
}

// One row by a warp: the candidates of its lists (cand: the row's column of them; n0,
// n1, n2 entries) inside rlim, `total` of them, in fp32, and in binary64 where their
// intervals overlap.  Returns the lane's binary64 evaluations, and 1 << 16 if any.
template <bool CALL>
KM_DEV unsigned refine_row_warp(const uint32_t* __restrict__ cand, int64_t n, int n0, int n1, int n2, float rlim, int total,
                                int row, const float* __restrict__ X, const float* __restrict__ C, int d, uint32_t emask,
                                float lscale, float g, int32_t* __restrict__ labels, int* js, float* vs, double* prod) {
    constexpr int NE = TC_GROUPS * TC_LIST;
    const int lane = threadIdx.x & 31, sl = lane & 7;
    const float tiny = direct_tiny(d);
    uint32_t e[2];
    unsigned m[2];
#pragma unroll
    for (int h = 0; h < 2; h++) {
        const int t = lane + 32 * h, gr = t / TC_LIST, slot = t % TC_LIST;
        const bool have = t < NE && slot < (gr == 0 ? n0 : (gr == 1 ? n1 : n2));
        e[h] = have ? cand[(size_t)t * n] : 0u;
        m[h] = have && cand_lower(e[h], emask, lscale) <= rlim ? entry_mask(e[h]) : 0u;
    }
    const int mine = __popc(m[0]) + __popc(m[1]);
    int incl = mine;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += o;
    }
    __syncwarp();
    int w = incl - mine;
#pragma unroll
    for (int h = 0; h < 2; h++)
        for (unsigned bb = m[h]; bb; bb &= bb - 1) js[w++] = 4 * entry_quad(e[h], emask) + __ffs(bb) - 1;
    __syncwarp();
    const float* x = X + (int64_t)row * d;
    for (int t0 = 0; t0 < total; t0 += 4) {
        const int t = t0 + (lane >> 3);
        float acc = t < total ? pair_value<0>(X, C, d, make_int2(row, js[t]), sl) : 0.0f;
#pragma unroll
        for (int off = 4; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (sl == 0 && t < total) vs[t] = acc;
    }
    __syncwarp();
    float up = INFINITY;
    for (int t = lane; t < total; t += 32) up = fminf(up, direct_upper(vs[t], g, tiny));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) up = fminf(up, __shfl_xor_sync(0xffffffffu, up, off));
    int open = 0, bj = 0x7fffffff;
    for (int t = lane; t < total; t += 32)
        if (direct_lower(vs[t], g) <= up) {
            open++;
            bj = js[t];  // (the only one, when open is 1 over the warp)
        }
    const unsigned who = __ballot_sync(0xffffffffu, open != 0);
    open = __reduce_add_sync(0xffffffffu, open);
    if (open == 1) {
        if (lane == __ffs(who) - 1) labels[row] = bj;
        return 0u;
    }
    if constexpr (CALL) return refine_row_exact_call(x, C, d, total, g, up, labels + row, js, vs, prod) | 1u << 16;
    else return refine_row_exact(x, C, d, total, g, up, labels + row, js, vs, prod) | 1u << 16;
}

// 32 rows per warp and round.  A lane per row reads the entries of the row's
// three lists (slot-major: 32 rows side by side) that lie inside the window of
// the row's final d^ minimum, the smallest of the groups' minima.  Rows with 2
// to RF_FEW candidates then take eight lanes each, four rows at a time: x in
// registers (NV float4 per lane; NV = 0: any d and alignment, x read again per
// candidate), two candidates' loads in flight.  Rows with more go with the
// overflowed ones where that is cheaper (many_to_list: a centred screen follows,
// or few centres: all of them in tiles take less than a row at a time; 89,201 x
// 173, k = 28, all pairs open: 340 us one by one, 138 in tiles), else, like those whose intervals
// overlap, they take the whole warp, which ends in binary64 (products in
// parallel, two candidates' sums at a time, each added in coordinate order by a lane).
// Labels only: every caller refines the winner's distance afterwards, to
// binary64 accuracy.
// LIST: the rows are list[0 .. *list_n) of X (r indexes the lists), else all n.
// Bound by the latency of a row's chain of loads (entries, then x and c).
// Evaluating the warp's pairs from one flat list in shared memory instead,
// eight at a time, was slower (1e6 x 128 listed rows 172 against 137 us,
// 4e6 x 64 249 against 196 us: 48 registers for five blocks per SM spill).
// (NV = 0 keeps 64 registers: given its own way the compiler took 48 and spilled,
// 300,000 x 77 134 us against 106.)
constexpr int RF_FEW = 12;
constexpr int RF_PROD_D = RF_FEW * 32 * (int)sizeof(int) / (2 * (int)sizeof(double));  // 2 d products in jl
template <int NV, bool LIST>
__global__ void __launch_bounds__(256, NV == 0 ? 4 : 0) k_refine(const int2* __restrict__ rowinfo, const float* __restrict__ roww, const uint32_t* __restrict__ cand,
                                                int64_t n, int ng, int ebits, const int32_t* __restrict__ list,
                                                const int* __restrict__ list_n, const float* __restrict__ X,
                                                const float* __restrict__ C, int d, float gamma32,
                                                int32_t* __restrict__ labels, int32_t* __restrict__ ovf_list,
                                                int* __restrict__ ovf_n, bool many_to_list, int rpw_all, DevCounters* cnt) {
    chain_enter();
    constexpr int NE = TC_GROUPS * TC_LIST;  // entries of a row's lists
    static_assert(NE <= 64 && TC_GROUPS == 3, "two entries per lane of three lists");
    extern __shared__ double rc_sm[];  // per warp: 2 d products, where jl has no room for them
    __shared__ int js_sh[8][4 * NE];
    __shared__ float vs_sh[8][4 * NE];
    __shared__ __align__(8) int jl_sh[8][RF_FEW * 32];
    __shared__ int ord_sh[8][32];
    const int64_t nrows = LIST ? (int64_t)*list_n : n;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, sl = lane & 7;
    int* js = js_sh[wib];
    float* vs = vs_sh[wib];
    int *jl = jl_sh[wib], *ord = ord_sh[wib];
    // (a row that takes the whole warp comes after the round's last use of jl; 8 KB a
    // block of their own, at d = 64, leave L1 that much less: 921 us for the 908 above)
    double* prod = d <= RF_PROD_D ? reinterpret_cast<double*>(jl) : rc_sm + (size_t)wib * 2 * d;
    const uint32_t emask = (1u << ebits) - 1u;
    const float lscale = __uint_as_float((uint32_t)(127 + ebits - 23) << 23);  // 2^(ebits - 23)
    const float g = gamma32, tiny = direct_tiny(d);
    const int d4 = d >> 2;
    unsigned ev32 = 0, ev64 = 0, amb = 0, ovf = 0;
    const int nwb = blockDim.x >> 5;
    // a list's rows, of unknown number, are spread evenly over the warps: a short
    // one of rows with many candidates each (taken one by one) took 74 us at 32 rows
    // per warp (1e5 x 128, k = 500), 9 now
    const int rpw = !LIST ? rpw_all : (int)max((int64_t)1, min((int64_t)32, (nrows + (int64_t)gridDim.x * nwb - 1) / ((int64_t)gridDim.x * nwb)));
    for (int64_t r0 = ((int64_t)blockIdx.x * nwb + wib) * rpw; r0 < nrows; r0 += (int64_t)gridDim.x * nwb * rpw) {
        const int64_t r = r0 + lane;
        const bool valid = lane < rpw && r < nrows;
        const int myrow = valid ? (LIST ? list[r] : (int)r) : 0;
        bool full = false;
        int cnt_g[TC_GROUPS];
        float lim = INFINITY;
        const float W = valid ? roww[r] : 0.0f;
#pragma unroll
        for (int q = 0; q < TC_GROUPS; q++) {
            const int2 ig = valid && q < ng ? rowinfo[(size_t)q * n + r] : make_int2(0, __float_as_int(INFINITY));
            full |= (ig.x & ROW_OVERFLOW) != 0;
            cnt_g[q] = ig.x & (ROW_OVERFLOW - 1);
            lim = fminf(lim, __int_as_float(ig.y));
        }
        lim += W;
        // an overflowed list, or an infinite window (which takes in the columns'
        // padding; nothing comparable counts as one): every centre
        full = valid && (full || !(lim < INFINITY));
        if (full) {
            ovf_list[atomicAdd(ovf_n, 1)] = myrow;
            ovf++;
        }
        int c = 0;
        // four slots' loads in flight
        auto take = [&](uint32_t e) {
            if (cand_lower(e, emask, lscale) <= lim)
                for (unsigned b = entry_mask(e); b; b &= b - 1, c++)
                    if (c < RF_FEW) jl[c * 32 + lane] = 4 * entry_quad(e, emask) + __ffs(b) - 1;
        };
#pragma unroll
        for (int q = 0; q < TC_GROUPS; q++) {
            if (!valid || full) cnt_g[q] = 0;
            const uint32_t* cg = cand + (size_t)q * TC_LIST * n + r;
            for (int s0 = 0; __any_sync(0xffffffffu, s0 < cnt_g[q]); s0 += 4) {
                uint32_t e[4];
#pragma unroll
                for (int s = 0; s < 4; s++) e[s] = s0 + s < cnt_g[q] ? cg[(size_t)(s0 + s) * n] : 0u;
#pragma unroll
                for (int s = 0; s < 4; s++)
                    if (s0 + s < cnt_g[q]) take(e[s]);
            }
        }
        if (c == 1) labels[myrow] = jl[lane];
        const bool few = c > 1 && c <= RF_FEW;
        const unsigned fm = __ballot_sync(0xffffffffu, few);
        if (few) ord[__popc(fm & ((1u << lane) - 1u))] = lane;
        __syncwarp();
        // rows of many candidates: up to four are taken here, one by one; more of them
        // leave for the next pass, whose launches (30 to 40 us once a row is listed)
        // a handful in all would not be worth (133,333 x 128 x 1024 uniform, 12 and more
        // candidates in one row of a thousand)
        unsigned slow = __ballot_sync(0xffffffffu, c > RF_FEW);
        if (many_to_list && __popc(slow) > 4) {
            if (c > RF_FEW) ovf_list[atomicAdd(ovf_n, 1)] = myrow;
            slow = 0;
        }
        const int nfew = __popc(fm);
        for (int i0 = 0; i0 < nfew; i0 += 4) {
            const int i = i0 + (lane >> 3);
            const int b = ord[min(i, nfew - 1)];
            const int cb = __shfl_sync(0xffffffffu, c, b), cc = i < nfew ? cb : 0;
            const int64_t row = __shfl_sync(0xffffffffu, myrow, b);
            const int most = __reduce_max_sync(0xffffffffu, cc);
            const float* x = X + row * d;
            float b1 = INFINITY, b2 = INFINITY;
            int j1 = 0;
            auto keep = [&](float v, int j, bool on) {
                if (on) {
                    if (v < b1) { b2 = b1; b1 = v; j1 = j; }
                    else b2 = fminf(b2, v);
                }
            };
            if constexpr (NV > 0) {
                constexpr int P = NV > 4 ? 1 : 2;  // candidates at once
                float4 xv[NV];
#pragma unroll
                for (int u = 0; u < NV; u++)
                    xv[u] = sl + 8 * u < d4 ? reinterpret_cast<const float4*>(x)[sl + 8 * u] : make_float4(0.f, 0.f, 0.f, 0.f);
                for (int t = 0; t < most; t += P) {
                    int j[P];
                    float acc[P];
                    float4 cv[P][NV];
#pragma unroll
                    for (int h = 0; h < P; h++) {
                        j[h] = jl[(t + h < cc ? t + h : 0) * 32 + b];
                        const float4* c4 = reinterpret_cast<const float4*>(C + (int64_t)j[h] * d);
#pragma unroll
                        for (int u = 0; u < NV; u++)
                            cv[h][u] = sl + 8 * u < d4 ? c4[sl + 8 * u] : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
#pragma unroll
                    for (int h = 0; h < P; h++) {
                        acc[h] = 0.0f;
#pragma unroll
                        for (int u = 0; u < NV; u++) {
                            const float u0 = xv[u].x - cv[h][u].x, u1 = xv[u].y - cv[h][u].y;
                            const float u2 = xv[u].z - cv[h][u].z, u3 = xv[u].w - cv[h][u].w;
                            acc[h] = fmaf(u0, u0, acc[h]);
                            acc[h] = fmaf(u1, u1, acc[h]);
                            acc[h] = fmaf(u2, u2, acc[h]);
                            acc[h] = fmaf(u3, u3, acc[h]);
                        }
                    }
#pragma unroll
                    for (int off = 4; off > 0; off >>= 1)
#pragma unroll
                        for (int h = 0; h < P; h++) acc[h] += __shfl_xor_sync(0xffffffffu, acc[h], off);
#pragma unroll
                    for (int h = 0; h < P; h++) keep(acc[h], j[h], t + h < cc);
                }
            } else {
                for (int t = 0; t < most; t++) {
                    const int j = jl[(t < cc ? t : 0) * 32 + b];
                    float acc = pair_value<0>(X, C, d, make_int2((int)row, j), sl);
#pragma unroll
                    for (int off = 4; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
                    keep(acc, j, t < cc);
                }
            }
            const bool sure = direct_lower(b2, g) > direct_upper(b1, g, tiny);  // false where nothing is comparable
            if (sl == 0 && cc) {
                ev32 += cc;
                if (sure) labels[row] = j1;
            }
            slow |= __reduce_or_sync(0xffffffffu, cc && !sure ? 1u << b : 0u);
        }
        // the others, the warp on one row at a time
        for (unsigned todo = slow; todo; todo &= todo - 1) {
            const int b = __ffs(todo) - 1;
            const int64_t row = __shfl_sync(0xffffffffu, myrow, b);
            const float rlim = __shfl_sync(0xffffffffu, lim, b);
            const int total = __shfl_sync(0xffffffffu, c, b);
            const int n0 = __shfl_sync(0xffffffffu, cnt_g[0], b), n1 = __shfl_sync(0xffffffffu, cnt_g[1], b);
            const int n2 = __shfl_sync(0xffffffffu, cnt_g[2], b);
            const unsigned r = refine_row_warp<(NV > 0)>(cand + r0 + b, n, n0, n1, n2, rlim, total, (int)row, X, C, d, emask,
                                                         lscale, g, labels, js, vs, prod);
            ev64 += r & 0xffffu;
            if (lane == 0) {
                amb += r >> 16;
                if (total > RF_FEW) ev32 += total;
            }
        }
        __syncwarp();
    }
    ev32 = __reduce_add_sync(0xffffffffu, ev32);
    if (ev64) atomicAdd(&cnt->fp64_evals, (unsigned long long)ev64);  // (lanes 0 and 1)
    ovf = __reduce_add_sync(0xffffffffu, ovf);
    if (lane == 0) {
        if (ev32) atomicAdd(&cnt->fp32_evals, (unsigned long long)ev32);
        if (amb) atomicAdd(&cnt->amb_rows, (unsigned long long)amb);
        if (ovf && !LIST) atomicAdd(&cnt->ovf_rows, (unsigned long long)ovf);
    }
}

bool refine_batched(int64_t n, int d) { return d > 64 && n * d > (int64_t)1 << 25; }

static cudaError_t launch_refine_batched(const float* X, const float* C, const TcArgs& a, int32_t* labels,
                                         double* min_dist, int32_t* full_list, int32_t* amb_list, int num_sms,
                                         cudaStream_t st, int* nlaunch) {
    // persistent grids: the resident blocks only
    int sel_per_sm = 1, cert_per_sm = 1;
    cudaError_t e0 = blocks_per_sm(k_cand_select, 256, 0, &sel_per_sm);
    if (e0 != cudaSuccess) return e0;
    e0 = blocks_per_sm(k_certify, 256, 0, &cert_per_sm);
    if (e0 != cudaSuccess) return e0;
    const int64_t rows_blocks = std::max<int64_t>(1, (a.n + 255) / 256);
    const int64_t rb = std::min<int64_t>(rows_blocks, (int64_t)num_sms * std::max(sel_per_sm, 1));
    const int64_t cb = std::min<int64_t>(rows_blocks, (int64_t)num_sms * std::max(cert_per_sm, 1));
    klaunch(k_cand_select, (unsigned)rb, 256, 0, st, a.rowinfo, a.roww, a.cand, a.n, tc_lists(a.k), a.ebits, a.pairs, a.pair_cap, a.rowpair, labels,
                                                a.cnt);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    *nlaunch = 4;
    // pair evaluation: a persistent grid of the resident blocks
    const bool vec = (a.d % 4 == 0) && a.d <= 256 && ((uintptr_t)X % 16 == 0) && ((uintptr_t)C % 16 == 0);
    const void* fn = !vec ? (const void*)k_pair_eval<0>
                          : (a.d <= 32 ? (const void*)k_pair_eval<1>
                                       : (a.d <= 128 ? (const void*)k_pair_eval<4> : (const void*)k_pair_eval<8>));
    int per_sm = 1;
    e = blocks_per_sm_of(fn, 256, 0, &per_sm);
    if (e != cudaSuccess) return e;
    const unsigned blocks = (unsigned)num_sms * (unsigned)std::max(per_sm, 1);
    const unsigned long long* np = &a.cnt->npairs;
    if (!vec) klaunch(k_pair_eval<0>, blocks, 256, 0, st, X, C, a.d, a.pairs, np, a.pair_cap, a.v32);
    else if (a.d <= 32) klaunch(k_pair_eval<1>, blocks, 256, 0, st, X, C, a.d, a.pairs, np, a.pair_cap, a.v32);
    else if (a.d <= 128) klaunch(k_pair_eval<4>, blocks, 256, 0, st, X, C, a.d, a.pairs, np, a.pair_cap, a.v32);
    else klaunch(k_pair_eval<8>, blocks, 256, 0, st, X, C, a.d, a.pairs, np, a.pair_cap, a.v32);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    klaunch(k_certify, (unsigned)cb, 256, 0, st, a.rowpair, a.n, a.pairs, a.v32, X, C, a.d, a.tp.gamma32, labels, min_dist,
                                             full_list, amb_list, a.cnt);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const size_t amb_smem = (size_t)8 * AMB_B * a.d * sizeof(double);  // 8 warps per block
    e = allow_max_smem(k_amb_fp64);
    if (e != cudaSuccess) return e;
    klaunch(k_amb_fp64, (unsigned)num_sms, 256, amb_smem, st, amb_list, &a.cnt->amb_count, a.rowpair, a.pairs, a.v32, X, C,
                                                          a.d, a.tp.gamma32, labels, min_dist, a.cnt);
    return cudaGetLastError();
}

template <int NV, bool LIST>
static cudaError_t launch_refine_nv(const float* X, const float* C, const TcArgs& a, const int32_t* list,
                                    const int* list_n, int32_t* labels, int32_t* ovf_list, int* ovf_n, bool many_to_list,
                                    int num_sms, cudaStream_t st) {
    auto fn = k_refine<NV, LIST>;
    // rows per warp: few rows are spread over the SMs in rounds of the four that
    // are evaluated together (a lane per row selects, so more rows want whole warps)
    const int rpw = !LIST && a.n <= (int64_t)num_sms * 128 ? 4 : (!LIST && a.n <= (int64_t)num_sms * 256 ? 8 : 32);
    const int64_t warps = (a.n + rpw - 1) / rpw;
    const int threads = LIST ? (a.n <= (int64_t)num_sms * 256 ? 32 : 256)
                             : 32 * (int)std::max<int64_t>(1, std::min<int64_t>(8, (warps + num_sms - 1) / num_sms));
    const int per_block = threads / 32 * rpw;
    const size_t sm = a.d <= RF_PROD_D ? 0 : (size_t)(threads / 32) * 2 * a.d * sizeof(double);
    cudaError_t e = allow_max_smem(fn);
    if (e != cudaSuccess) return e;
    int per_sm = 1;
    e = blocks_per_sm(fn, threads, sm, &per_sm);
    if (e != cudaSuccess) return e;
    const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((a.n + per_block - 1) / per_block, (int64_t)num_sms * std::max(per_sm, 1)));
    klaunch(fn, (unsigned)blocks, threads, sm, st, a.rowinfo, a.roww, a.cand, a.n, tc_lists(a.k), a.ebits, list, list_n, X, C, a.d, a.tp.gamma32,
                                              labels, ovf_list, ovf_n, many_to_list, rpw, a.cnt);
    return cudaGetLastError();
}

cudaError_t launch_refine(const float* X, const float* C, const TcArgs& a, const int32_t* list, const int* list_n,
                          int32_t* labels, double* min_dist, int32_t* ovf_list, int* ovf_n, int32_t* amb_list, bool centred_follows,
                          int num_sms, cudaStream_t st, int* nlaunch) {
    if (!list && refine_batched(a.n, a.d) && a.pairs)
        return launch_refine_batched(X, C, a, labels, min_dist, ovf_list, amb_list, num_sms, st, nlaunch);
    *nlaunch = 1;
    const bool many = centred_follows || (a.k <= 256 && a.d <= 256);
    const bool vec = a.d % 4 == 0 && a.d <= 256 && ((uintptr_t)X % 16 == 0) && ((uintptr_t)C % 16 == 0);
    const int nv = !vec ? 0 : (a.d <= 32 ? 1 : (a.d <= 64 ? 2 : (a.d <= 128 ? 4 : 8)));
#define KM_RF(NV)                                                                                            \
    if (nv == NV)                                                                                            \
        return list ? launch_refine_nv<NV, true>(X, C, a, list, list_n, labels, ovf_list, ovf_n, many, num_sms, st) \
                    : launch_refine_nv<NV, false>(X, C, a, list, list_n, labels, ovf_list, ovf_n, many, num_sms, st);
    KM_RF(0) KM_RF(1) KM_RF(2) KM_RF(4) KM_RF(8)
#undef KM_RF
    return cudaErrorInvalidValue;
}

// The centres and the listed rows, centred, for the second screen (eight lanes
// per row); the last block to finish forms the column maxima and q_j.  An
// empty list, the usual case, leaves at once.
__global__ void __launch_bounds__(256) k_centre_rows(const int32_t* __restrict__ list, const int* __restrict__ list_n,
                                                     const float* __restrict__ X, const float* __restrict__ C, int k,
                                                     int d, const Centred cen, unsigned* ticket) {
    chain_enter();
    const int nf = *list_n;
    if (nf == 0) return;
    __shared__ __align__(16) float mu[256];
    __shared__ bool last;
    centre_mean(C, k, d, cen.ldq, mu);
    const int lane = threadIdx.x & 31, sl = lane & 7;
    const unsigned gmask = 0xFFu << (lane & ~7);
    const bool vec = d % 4 == 0 && (((uintptr_t)X | (uintptr_t)C) & 15) == 0;
    const int64_t ng = (int64_t)gridDim.x * (blockDim.x / 8);
    for (int64_t r = (int64_t)blockIdx.x * (blockDim.x / 8) + threadIdx.x / 8; r < (int64_t)k + nf; r += ng) {
        const bool isc = r < k;
        const float* x = isc ? C + r * d : X + (int64_t)list[r - k] * d;
        __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(isc ? cen.Cq : cen.Xq) + (isc ? r : r - k) * cen.ldq;
        float4* stat = isc ? cen.cstat + r : cen.xstat + (r - k);
        if (vec) centred_row<true>(x, mu, d, cen.ldq, dst, stat, sl, gmask);
        else centred_row<false>(x, mu, d, cen.ldq, dst, stat, sl, gmask);
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    const int kpad = (k + 255) / 256 * 256;
    for (int j = threadIdx.x; j < kpad; j += blockDim.x) cen.qpad[j] = j < k ? __ldcg(cen.cstat + j).x : INFINITY;
    colmax_block(cen.cstat, k, cen.colmax);
}

cudaError_t launch_centre_rows(const int32_t* list, const int* list_n, const float* X, const float* C, int k, int d,
                               const Centred& cen, unsigned* ticket, int num_sms, cudaStream_t st) {
    klaunch(k_centre_rows, (unsigned)num_sms * 4, 256, 0, st, list, list_n, X, C, k, d, cen, ticket);
    return cudaGetLastError();
}

}  // namespace km
