// k_update.cu -- centre update, Eq. (center), with the accuracy Section 4.4
// asks of it.
//
// Section 4.4 (Lemma 4.4, Theorem 4.5, Corollary 4.7) shows the update needs
// more precision than the distances, increasingly so late in the iteration.
// Here the per-cluster coordinate sums are formed EXACTLY in 64-bit fixed
// point: every coordinate is scaled by 2^S (S chosen from max|x| and n so
// that no partial sum can exceed 2^62) and rounded once to an integer, after
// which integer addition is exact and associative.  The only error is that
// one rounding, <= 2^-(S+1) per coordinate, so |mu^ - mu| <= 2^-(S+1) before
// the final division (binary64) and the fp32 store -- below the binary64
// recursive-summation bound gamma_m a_bar of Lemma 4.4 for the data sizes
// here, and independent of the order in which threads add: results are
// bitwise reproducible run to run and alone or batched.
#include <algorithm>

#include "common.cuh"
#include "df.cuh"
#include "fixed.cuh"
#include "internal.h"

namespace km {

__global__ void k_absmax(const float* __restrict__ X, int64_t count, unsigned* out) {
    chain_enter();
    float m = 0.0f;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x)
        m = fmaxf(m, fabsf(X[e]));
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
    if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));  // non-negative floats order as uints
}

// Row-parallel accumulation with global atomics, for the shapes that neither
// the bucketed path nor shared memory takes (integer, so the result does not
// depend on the order of the adds).
__global__ void k_accumulate(const float* __restrict__ X, int64_t n, int d, const int32_t* __restrict__ labels,
                             int k, const unsigned* __restrict__ amax_bits, int64_t nscale, long long* __restrict__ sums,
                             long long* __restrict__ counts) {
    chain_enter();
    const FixedScale fx(fixed_shift(*amax_bits, nscale));
    // rows spread over the warps; within a row the lanes walk the coordinates
    // (for d < 32 a warp covers 32 / d rows at once)
    const int lane = threadIdx.x & 31;
    const int rpw = d < 32 ? 32 / d : 1;  // rows per warp step
    const int sub = lane / (d < 32 ? d : 32), l_in = lane % (d < 32 ? d : 32);
    const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t r = gw * rpw; r < n; r += nw * rpw) {
        const int64_t i = r + sub;
        if (sub >= rpw || i >= n) continue;
        const int j = labels[i];
        const float* x = X + i * d;
        for (int l = l_in; l < d; l += (d < 32 ? d : 32)) {
            const long long v = fx(x[l]);
            atomicAdd(reinterpret_cast<unsigned long long*>(&sums[(int64_t)j * d + l]), (unsigned long long)v);
        }
        if (l_in == 0) atomicAdd(reinterpret_cast<unsigned long long*>(&counts[j]), 1ull);
    }
}

// A warp's pass over STEP rows, each on LPR lanes of NV4 float4 as in
// k_winner_dist: the rows' labels (js, -1 past the end) and coordinates (xv);
// WD: each row's distance to its own centre (the same arithmetic, the same
// bits) from the same read of the row.
template <int NV4, int LPR, bool VEC, bool WD, int R>
KM_DEV void rows_pass(const float* __restrict__ X, int64_t n, int d, const int32_t* __restrict__ labels, int64_t base,
                      const float* __restrict__ C, double* __restrict__ md, int lane, int (&js)[R], float4 (&xv)[R][NV4]) {
    constexpr int G = 32 / LPR, STEP = R * G;
    const int sub = lane / LPR, cl = lane % LPR;
    const int d4 = (d + 3) >> 2;
    const int jl = (lane < STEP && base + lane < n) ? labels[base + lane] : 0;
    float4 cv[R][NV4];
#pragma unroll
    for (int b = 0; b < R; b++) {
        const int64_t row = base + b * G + sub;
        const int j = __shfl_sync(0xffffffffu, jl, b * G + sub);
        js[b] = row < n ? j : -1;
#pragma unroll
        for (int u = 0; u < NV4; u++) {
            const int cidx = cl + LPR * u;
            const bool ok = row < n && cidx < d4;
            xv[b][u] = cv[b][u] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (VEC) {
                if (ok) xv[b][u] = reinterpret_cast<const float4*>(X + row * d)[cidx];
                if (WD && ok) cv[b][u] = reinterpret_cast<const float4*>(C + (int64_t)j * d)[cidx];
            } else if (ok) {
                const float* x = X + row * d + 4 * cidx;
                const float* c = C + (int64_t)j * d + 4 * cidx;
                const int m = d - 4 * cidx;
                xv[b][u] = make_float4(x[0], m > 1 ? x[1] : 0.f, m > 2 ? x[2] : 0.f, m > 3 ? x[3] : 0.f);
                if (WD) cv[b][u] = make_float4(c[0], m > 1 ? c[1] : 0.f, m > 2 ? c[2] : 0.f, m > 3 ? c[3] : 0.f);
            }
        }
    }
    if (WD) {
        DF part[R];
#pragma unroll
        for (int b = 0; b < R; b++) part[b] = df_lane<NV4>(xv[b], cv[b]);
        int rs;
        const DF r = df_rows<R, LPR>(part, cl, rs);
        const int64_t row = base + rs * G + sub;
        if ((cl & (LPR / R - 1)) == 0 && row < n) md[row] = df_value(r);
    }
}

// k_accumulate in shared memory (the k d sums and k counts), with the winners'
// distances (WD, rows_pass), in one launch where the bucketed path takes four.
// Bound by the shared atomics: 1e5 x 10, k = 100 26 -> 19 us with the distances.
// Rows of one label take turns at its addresses, so a warp adds up several of
// them first: an update call with all rows in one of the 100 clusters took 64 us
// without that, 31 with (54 bucketed).
template <int NV4, int LPR, bool VEC, bool WD>
__global__ void __launch_bounds__(512) k_accum_rows(const float* __restrict__ X, int64_t n, int d,
                                                    const int32_t* __restrict__ labels, int k,
                                                    const unsigned* __restrict__ amax_bits, int64_t nscale,
                                                    long long* __restrict__ sums, long long* __restrict__ counts,
                                                    const float* __restrict__ C, double* __restrict__ md) {
    chain_enter();
    extern __shared__ unsigned long long acc_rows[];  // k d sums, k counts
    constexpr int G = 32 / LPR;
    constexpr int R = NV4 == 4 ? 2 : 4;
    constexpr int STEP = R * G;
    const FixedScale fx(fixed_shift(*amax_bits, nscale));
    const int kd = k * d;
    unsigned long long* const cacc = acc_rows + kd;
    for (int e = threadIdx.x; e < kd + k; e += blockDim.x) acc_rows[e] = 0ull;
    __syncthreads();
    const int lane = threadIdx.x & 31, cl = lane % LPR;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t base = w0 * STEP; base < n; base += nw * STEP) {
        float4 xv[R][NV4];
        int js[R];
        rows_pass<NV4, LPR, VEC, WD>(X, n, d, labels, base, C, md, lane, js, xv);
        // several rows of one label (the first row's, the last one's) are added up in
        // registers first: shared atomics on one address take turns
        const int lead[2] = {__shfl_sync(0xffffffffu, js[0], 0), __shfl_sync(0xffffffffu, js[R - 1], 31)};
        unsigned same = 0;  // the rows of either, 16 bits each
#pragma unroll
        for (int b = 0; b < R; b++) same += (js[b] == lead[0] ? 1u : 0u) + (js[b] == lead[1] ? 65536u : 0u);
        same = __reduce_add_sync(0xffffffffu, cl == 0 ? same : 0u);
        if ((same & 0xfffcfffcu) != 0u) {
#pragma unroll 1
            for (int h = 0; h < 2; h++) {
                const int j = lead[h];
                const unsigned m = h ? same >> 16 : same & 65535u;
                if (j < 0 || m < 4 || (h && j == lead[0])) continue;
#pragma unroll
                for (int u = 0; u < NV4; u++) {
                    unsigned long long v[4] = {};
#pragma unroll
                    for (int b = 0; b < R; b++) {
                        const float xe[4] = {xv[b][u].x, xv[b][u].y, xv[b][u].z, xv[b][u].w};
#pragma unroll
                        for (int t = 0; t < 4; t++) v[t] += js[b] == j ? (unsigned long long)fx(xe[t]) : 0ull;
                    }
#pragma unroll
                    for (int t = 0; t < 4; t++) {
#pragma unroll
                        for (int o = LPR; o < 32; o <<= 1) v[t] += __shfl_xor_sync(0xffffffffu, v[t], o);
                        const int l = 4 * (cl + LPR * u) + t;
                        if (lane < LPR && l < d && v[t]) atomicAdd(acc_rows + (int64_t)j * d + l, v[t]);
                    }
                }
                if (lane == 0) atomicAdd(cacc + j, (unsigned long long)m);
#pragma unroll
                for (int b = 0; b < R; b++) js[b] = js[b] == j ? -1 : js[b];
            }
        }
#pragma unroll
        for (int b = 0; b < R; b++)
            if (js[b] >= 0) {
                unsigned long long* a = acc_rows + (int64_t)js[b] * d;
#pragma unroll
                for (int u = 0; u < NV4; u++) {
                    const int l = 4 * (cl + LPR * u);
                    const float xe[4] = {xv[b][u].x, xv[b][u].y, xv[b][u].z, xv[b][u].w};
#pragma unroll
                    for (int t = 0; t < 4; t++)
                        if (l + t < d && xe[t] != 0.0f) atomicAdd(a + l + t, (unsigned long long)fx(xe[t]));
                }
                if (cl == 0) atomicAdd(cacc + js[b], 1ull);
            }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < kd; e += blockDim.x)
        if (acc_rows[e]) atomicAdd(reinterpret_cast<unsigned long long*>(sums) + e, acc_rows[e]);
    for (int e = threadIdx.x; e < k; e += blockDim.x)
        if (cacc[e]) atomicAdd(reinterpret_cast<unsigned long long*>(counts) + e, cacc[e]);
}

// The same straight to the sums in L2, whatever the labels: a block takes rb
// rows (a power of two, 16 to AO_ROWS) into shared
// memory, ranks them by label (each row against all) and sums them in that
// order, a thread per coordinate and slice of the order, so that a label costs
// one atomic per coordinate and block however many rows have it.  A run of one
// label that goes on from slice to slice is handed along through shared memory
// and added by the slice it ends in.
// Bound by latency, about four dependent stages, and for many rows of few
// coordinates by ranking and by the atomics.  An update call of 65,536 x 16 takes
// 31 us whether the rows spread over 1024 clusters or lie in one (53 and 58 in
// the four bucketed launches; atomics row by row, some 60 per ns on spread
// addresses but 2 on shared ones, took 31 and 671).  256 rows a block were
// slower (131,072 x 16, k = 4: 40 us against 34).
constexpr int AO_ROWS = 128;       // most rows per block
constexpr int AO_FLOATS = 8192;    // coordinates per block
template <int NV4, int LPR, bool VEC, bool WD>
__global__ void __launch_bounds__(256) k_accum_ordered(const float* __restrict__ X, int64_t n, int d,
                                                       const int32_t* __restrict__ labels, int rb,
                                                       const unsigned* __restrict__ amax_bits, int64_t nscale,
                                                       long long* __restrict__ sums, long long* __restrict__ counts,
                                                       const float* __restrict__ C, double* __restrict__ md) {
    chain_enter();
    extern __shared__ __align__(16) float ord_xs[];  // rb rows of ldx floats
    __shared__ __align__(16) int lab[AO_ROWS];
    __shared__ int order[AO_ROWS], slab[AO_ROWS];
    __shared__ unsigned long long part[256];
    constexpr int G = 32 / LPR;
    constexpr int R = NV4 == 4 ? 2 : 4;
    constexpr int STEP = R * G;
    const FixedScale fx(fixed_shift(*amax_bits, nscale));
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5, sub = lane / LPR, cl = lane % LPR;
    const int d4 = (d + 3) >> 2, ldx = 4 * d4;
    const int64_t r0 = (int64_t)blockIdx.x * rb;
    const int rows = (int)min((int64_t)rb, n - r0);
    if (t >= rows && t < AO_ROWS) lab[t] = 0x7fffffff;  // (past the last row: above every label)
    for (int base = wid * STEP; base < rows; base += 8 * STEP) {
        float4 xv[R][NV4];
        int js[R];
        rows_pass<NV4, LPR, VEC, WD>(X, r0 + rows, d, labels, r0 + base, C, md, lane, js, xv);
#pragma unroll
        for (int b = 0; b < R; b++)
            if (js[b] >= 0) {
                const int r = base + b * G + sub;
#pragma unroll
                for (int u = 0; u < NV4; u++)
                    if (cl + LPR * u < d4) reinterpret_cast<float4*>(ord_xs + r * ldx)[cl + LPR * u] = xv[b][u];
                if (cl == 0) lab[r] = js[b];
            }
    }
    __syncthreads();
    if (t < rows) {
        const int my = lab[t];
        int rank = 0, before = 0, same = 0;  // smaller labels, equal ones before this row, equal ones
        for (int q = 0; q < rows; q += 4) {
            const int4 o4 = *reinterpret_cast<const int4*>(lab + q);
            const int o[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
            for (int i = 0; i < 4; i++) {
                rank += o[i] < my ? 1 : 0;
                same += o[i] == my ? 1 : 0;
                before += o[i] == my && q + i < t ? 1 : 0;
            }
        }
        order[rank + before] = t;
        slab[rank + before] = my;
        if (before == 0) atomicAdd(reinterpret_cast<unsigned long long*>(counts) + my, (unsigned long long)same);
    }
    __syncthreads();
    const int ns = max(1, min(256 / d, (rows + 7) / 8)), per = (rows + ns - 1) / ns;  // slices, rows of a slice
    const int s = d <= 256 ? t / d : 0, p0 = s * per, p1 = min(rows, p0 + per);
    const bool work = s < ns && p0 < p1;
    auto flush = [&](int j, int l, unsigned long long v) {
        if (v) atomicAdd(reinterpret_cast<unsigned long long*>(sums) + (int64_t)j * d + l, v);
    };
    for (int l0 = 0; l0 < d; l0 += 256) {  // (one round up to 256 coordinates; one slice past them)
        const int l = d <= 256 ? t - s * d : l0 + t;
        const bool on = work && l < d;
        bool closes = false;     // a run from an earlier slice ends in this one
        unsigned long long acc = 0ull, first = 0ull;
        if (on) {
            int cur = slab[p0];
            bool joined = p0 > 0 && slab[p0 - 1] == cur;  // the current run came from an earlier slice
            for (int p = p0; p < p1; p++) {
                const int j = slab[p];
                if (j != cur) {
                    if (joined) {
                        first = acc;
                        closes = true;
                    } else {
                        flush(cur, l, acc);
                    }
                    joined = false;
                    cur = j;
                    acc = 0ull;
                }
                acc += (unsigned long long)fx(ord_xs[order[p] * ldx + l]);
            }
            if (p1 < rows && slab[p1] == cur) {
                part[t] = acc;  // goes on in the next slice
            } else if (joined) {
                first = acc;
                closes = true;
            } else {
                flush(cur, l, acc);
            }
        }
        if (ns > 1) __syncthreads();
        if (closes) {
            const int j = slab[p0];
            for (int q = s - 1; q >= 0; q--) {
                first += part[q * d + l];
                if (q == 0 || slab[q * per] != j || slab[q * per - 1] != j) break;
            }
            flush(j, l, first);
        }
    }
}

// ---- bucketed reduction: rows grouped by label, summed in registers ------
// Integer (fixed-point) addition is order-independent, so the row order
// inside a bucket (set by atomic cursors) does not change any bit of the
// result.
constexpr int SEG_MAX = 512;     // most rows per warp work item (the 32-bit part sums stay exact)
constexpr int SCAT_ROWS = 4096;  // rows per block of the histogram / scatter kernels

// Rows of a work item of a bucket of cnt rows: seg, but at least 64 where the
// bucket holds a quarter of all rows and more, whose items' sums all go to the
// same addresses (200,000 x 32 with all rows in one of 30 clusters: 159 us a call
// with items of 32 rows, 98 of 64; 150,001 x 256 with clusters of uneven size: 12
// us more in items of 64 for every cluster of 2048 rows).
// (big: a quarter of the rows where seg is below 64, else above all counts.)
KM_DEV int bucket_seg(int cnt, int big, int seg) { return cnt >= big ? 64 : seg; }
KM_DEV int bucket_items(int cnt, int big, int seg) {
    const int s = bucket_seg(cnt, big, seg);
    return (cnt + s - 1) / s;
}

// per-label counts (block histogram in shared memory, one global add per label)
__global__ void k_label_hist(const int32_t* __restrict__ labels, int64_t n, int k, int* __restrict__ cnt32) {
    chain_enter();
    extern __shared__ int h[];
    for (int j = threadIdx.x; j < k; j += blockDim.x) h[j] = 0;
    __syncthreads();
    const int64_t r0 = (int64_t)blockIdx.x * SCAT_ROWS, r1 = min(n, r0 + SCAT_ROWS);
    for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) atomicAdd(&h[labels[i]], 1);
    __syncthreads();
    for (int j = threadIdx.x; j < k; j += blockDim.x)
        if (h[j]) atomicAdd(&cnt32[j], h[j]);
}

// Exclusive scans (one block of 1024 threads): bucket offsets, cursors, and
// the offsets of each bucket's first work item; counts as int64.
__global__ void k_bucket_scan(const int* __restrict__ cnt32, int k, int seg, int big, int* __restrict__ off,
                              int* __restrict__ cursor, int* __restrict__ item_off, long long* __restrict__ counts) {
    chain_enter();
    __shared__ int sa[1024], sb[1024];
    const int t = threadIdx.x, T = blockDim.x;
    const int per = (k + T - 1) / T;
    const int j0 = min(k, t * per), j1 = min(k, j0 + per);
    int a = 0, b = 0;
    for (int j = j0; j < j1; j++) {
        a += cnt32[j];
        b += bucket_items(cnt32[j], big, seg);
    }
    sa[t] = a;
    sb[t] = b;
    __syncthreads();
    for (int st = 1; st < T; st <<= 1) {
        const int va = (t >= st) ? sa[t - st] : 0, vb = (t >= st) ? sb[t - st] : 0;
        __syncthreads();
        sa[t] += va;
        sb[t] += vb;
        __syncthreads();
    }
    int oa = sa[t] - a, ob = sb[t] - b;
    for (int j = j0; j < j1; j++) {
        off[j] = oa;
        cursor[j] = oa;
        item_off[j] = ob;
        counts[j] = cnt32[j];
        oa += cnt32[j];
        ob += bucket_items(cnt32[j], big, seg);
    }
    if (t == T - 1) {
        off[k] = sa[T - 1];
        item_off[k] = sb[T - 1];
    }
}

// Each block reserves one contiguous range per label (one global atomic per
// label present) and places its rows with shared-memory cursors.
__global__ void k_bucket_scatter(const int32_t* __restrict__ labels, int64_t n, int k, int* __restrict__ cursor,
                                 int32_t* __restrict__ perm) {
    chain_enter();
    extern __shared__ int sh[];
    int* h = sh;
    int* lc = sh + k;
    for (int j = threadIdx.x; j < k; j += blockDim.x) h[j] = 0;
    __syncthreads();
    const int64_t r0 = (int64_t)blockIdx.x * SCAT_ROWS, r1 = min(n, r0 + SCAT_ROWS);
    for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) atomicAdd(&h[labels[i]], 1);
    __syncthreads();
    for (int j = threadIdx.x; j < k; j += blockDim.x) lc[j] = h[j] ? atomicAdd(&cursor[j], h[j]) : 0;
    __syncthreads();
    for (int64_t i = r0 + threadIdx.x; i < r1; i += blockDim.x) perm[atomicAdd(&lc[labels[i]], 1)] = (int32_t)i;
}

KM_DEV int bucket_of(const int* __restrict__ item_off, int k, int64_t it) {
    int lo = 0, hi = k;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (item_off[mid] <= it) lo = mid; else hi = mid;
    }
    return lo;
}

// Coordinates 4c .. 4c + 3 of the row at `row` (zero past d).
template <bool VEC>
KM_DEV float4 load_chunk(const float* __restrict__ row, int d, int c) {
    if (VEC) return reinterpret_cast<const float4*>(row)[c];
    const float* x = row + 4 * c;
    const int m = d - 4 * c;
    return make_float4(x[0], m > 1 ? x[1] : 0.f, m > 2 ? x[2] : 0.f, m > 3 ? x[3] : 0.f);
}

// One warp per work item (bucket j, rows [c*CHUNK, (c+1)*CHUNK) of it); each
// row is spread over LPR lanes (NV4 float4 each, d % 4 == 0), so a warp reads
// 32 / LPR rows per load; exact sums in registers, folded across the row
// groups of the warp at the end, one atomic add per coordinate per item.
//
// WD: the same pass also gives each row's distance to its own centre c_j (the
// winner's ||x - c||^2, Eq. (dist-direct)) to binary64 accuracy (df.cuh: the
// rows' chunk partials reduced over the row's lanes, eight rows at a time), so
// the assignment's min_dist costs no second read of X.
// VEC: rows and centres are float4 (d % 4 == 0, aligned); else four loads each.
template <int NV4, int LPR, bool WD, bool VEC>
__global__ void __launch_bounds__(256, (NV4 == 1 && LPR == 32) ? 3 : (NV4 == 4 ? 1 : 2)) k_bucket_sum(const float* __restrict__ X, int d, int k, int seg, int big,
                                                       const int* __restrict__ off,
                             const int* __restrict__ item_off, const int32_t* __restrict__ perm,
                             const unsigned* __restrict__ amax_bits, int64_t nscale, long long* __restrict__ sums,
                             const float* __restrict__ C, double* __restrict__ md) {
    chain_enter();
    static_assert(LPR == 32 || NV4 == 1, "rows narrower than a warp take one float4 per lane");
    constexpr int G = 32 / LPR;                            // rows per warp load
    // loads in flight per lane: 8 at full-warp rows of one float4 (three blocks
    // per SM), else up to 16
    constexpr int RB = (NV4 == 1 && LPR == 32) ? 8 : ((16 / NV4) < (32 / G) ? 16 / NV4 : 32 / G);
    constexpr int STEP = RB * G;                           // rows per round (divides 32)
    const FixedScale fx(fixed_shift(*amax_bits, nscale));
    const int lane = threadIdx.x & 31, sub = lane / LPR, cl = lane % LPR;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int nitems = item_off[k];
    const int d4 = (d + 3) >> 2;
    for (int64_t it = w0; it < nitems; it += nw) {
        const int j = bucket_of(item_off, k, it);
        const int c = (int)(it - item_off[j]);
        const int sj = bucket_seg(off[j + 1] - off[j], big, seg);
        const int r0 = off[j] + c * sj, r1 = min(off[j + 1], r0 + sj);
        // the bucket's centre: this lane's chunks of c_j (WD)
        float4 cj[NV4];
        if (WD) {
#pragma unroll
            for (int u = 0; u < NV4; u++) {
                const int cidx = cl + LPR * u;
                cj[u] = (cidx < d4) ? load_chunk<VEC>(C + (int64_t)j * d, d, cidx) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
        }
        // biased parts of the fixed-point values, summed modulo 2^32 (SEG_MAX rows at most)
        unsigned a2[NV4][4], a1[NV4][4], a0[NV4][4];
#pragma unroll
        for (int u = 0; u < NV4; u++)
#pragma unroll
            for (int t = 0; t < 4; t++) a2[u][t] = a1[u][t] = a0[u][t] = 0u;
        unsigned rounds = 0;
        int64_t next_i = (r0 + lane < r1) ? (int64_t)perm[r0 + lane] : -1;
        for (int base = r0; base < r1; base += 32) {
            // the row indices of 32 rows in one coalesced load, then broadcast;
            // the following 32 rows' indices are loaded now and their data sent
            // to L2 once this round's loads are out
            const int64_t my_i = next_i;
            next_i = (base + 32 + lane < r1) ? (int64_t)perm[base + 32 + lane] : -1;
            bool pf = true;
#pragma unroll 1
            for (int b0 = 0; b0 < 32 && base + b0 < r1; b0 += STEP) {
                rounds++;
                float4 v[RB][NV4];
#pragma unroll
                for (int b = 0; b < RB; b++) {
                    const int64_t i = __shfl_sync(0xffffffffu, my_i, b0 + b * G + sub);
#pragma unroll
                    for (int u = 0; u < NV4; u++) {
                        const int cidx = cl + LPR * u;
                        v[b][u] = (i >= 0 && cidx < d4) ? load_chunk<VEC>(X + i * d, d, cidx) : make_float4(0.f, 0.f, 0.f, 0.f);
                    }
                }
                if (VEC && LPR < 32 && pf) {  // narrow rows (measured: a loss at 512-byte rows)
                    if (next_i >= 0) prefetch_l2_bulk(X + next_i * d, (uint32_t)d * 4u);
                    pf = false;
                }
#pragma unroll
                for (int b = 0; b < RB; b++)
#pragma unroll
                    for (int u = 0; u < NV4; u++) {
                        uint2 q2, q1, q0;
                        fx.split2(make_float2(v[b][u].x, v[b][u].y), q2, q1, q0);
                        a2[u][0] += q2.x; a2[u][1] += q2.y;
                        a1[u][0] += q1.x; a1[u][1] += q1.y;
                        a0[u][0] += q0.x; a0[u][1] += q0.y;
                        fx.split2(make_float2(v[b][u].z, v[b][u].w), q2, q1, q0);
                        a2[u][2] += q2.x; a2[u][3] += q2.y;
                        a1[u][2] += q1.x; a1[u][3] += q1.y;
                        a0[u][2] += q0.x; a0[u][3] += q0.y;
                    }
                if (WD) {
                    // the rows' distances to c_j, RW rows per multi-row butterfly
                    constexpr int RW = RB < 8 ? RB : 8;
#pragma unroll
                    for (int bb = 0; bb < RB; bb += RW) {
                        DF part[RW];
#pragma unroll
                        for (int b = 0; b < RW; b++) part[b] = df_lane<NV4>(v[bb + b], cj);
                        int rs;
                        const DF r = df_rows<RW, LPR>(part, cl, rs);
                        const int64_t i = __shfl_sync(0xffffffffu, my_i, b0 + (bb + rs) * G + sub);
                        if ((cl & (LPR / RW - 1)) == 0 && i >= 0) md[i] = df_value(r);
                    }
                }
            }
        }
        // the row groups' sums of the same coordinates (modulo 2^32 like the sums)
#pragma unroll
        for (int o = LPR; o < 32; o <<= 1)
#pragma unroll
            for (int u = 0; u < NV4; u++)
#pragma unroll
                for (int t = 0; t < 4; t++) {
                    a2[u][t] += __shfl_xor_sync(0xffffffffu, a2[u][t], o);
                    a1[u][t] += __shfl_xor_sync(0xffffffffu, a1[u][t], o);
                    a0[u][t] += __shfl_xor_sync(0xffffffffu, a0[u][t], o);
                }
        // every row slot of every round was split (absent rows and padding as 0.0f)
        const unsigned m = rounds * (unsigned)STEP;
#pragma unroll
        for (int u = 0; u < NV4; u++) {
            const int cidx = cl + LPR * u;
            if (sub == 0 && cidx < d4)
#pragma unroll
                for (int t = 0; t < 4; t++) {
                    const long long acc = FixedScale::combine(a2[u][t], a1[u][t], a0[u][t], m);
                    if (acc && (VEC || 4 * cidx + t < d))
                        atomicAdd(reinterpret_cast<unsigned long long*>(&sums[(int64_t)j * d + 4 * cidx + t]),
                                  (unsigned long long)acc);
                }
        }
    }
}

// d = 1, 2, 3 or 5: lanes over rows, each lane sums its rows' d coordinates,
// then a warp reduction.
template <int D>
__global__ void k_bucket_sum_small(const float* __restrict__ X, int k, int seg, int big, const int* __restrict__ off,
                                   const int* __restrict__ item_off, const int32_t* __restrict__ perm,
                                   const unsigned* __restrict__ amax_bits, int64_t nscale, long long* __restrict__ sums) {
    chain_enter();
    const FixedScale fx(fixed_shift(*amax_bits, nscale));
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int nitems = item_off[k];
    for (int64_t it = w0; it < nitems; it += nw) {
        const int j = bucket_of(item_off, k, it);
        const int c = (int)(it - item_off[j]);
        const int sj = bucket_seg(off[j + 1] - off[j], big, seg);
        const int r0 = off[j] + c * sj, r1 = min(off[j + 1], r0 + sj);
        long long acc[D];
#pragma unroll
        for (int l = 0; l < D; l++) acc[l] = 0;
        for (int r = r0 + lane; r < r1; r += 32) {
            const float* x = X + (int64_t)perm[r] * D;
#pragma unroll
            for (int l = 0; l < D; l++) acc[l] += fx(x[l]);
        }
#pragma unroll
        for (int l = 0; l < D; l++) {
            long long v = acc[l];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0 && v) atomicAdd(reinterpret_cast<unsigned long long*>(&sums[(int64_t)j * D + l]), (unsigned long long)v);
        }
    }
}

// Small d and small k * d: rows in their natural order, a warp per chunk of up
// to AS_CHUNK, 32 rows per step (one per lane, through a ring in shared memory
// filled by 16-byte asynchronous copies), each warp keeping the 32-bit parts of
// every cluster's fixed-point sum (and its count) in shared memory.
//  * A step whose rows all have one label (an image's pixels come in long runs)
//    adds each lane's parts to registers; they are folded over the warp when the
//    label changes or the chunk ends.
//  * Other steps: up to AS_FEW labels one after another by hardware reductions
//    over their lanes; more of them, in at most AS_RUNS runs, by a segmented
//    inclusive scan over the runs (five shuffle levels) that leaves each run's total
//    in its last lane, which adds it with a shared atomic; in no order, each row by
//    its own shared atomics.
// At the end of a chunk the block's eight accumulators are folded into the global
// int64 sums together, k d + k atomics on addresses that all blocks share: chunks
// as long as two blocks per SM allow.  Integer additions throughout: the order
// does not matter.
// NP: parts per value, 3, or 2 where the top one is always zero (from 2^22
// rows on).  WD: each row's distance to its own centre (binary64 accuracy,
// df.cuh) from the same read of the row, with C staged in shared memory.
// Bound by reads of X and the labels where runs are long, else by the steps'
// instructions; 16.8 M rows x 5, k = 16, image: 128 us (249 us with the scan in
// every step and D loads at a stride of D words).  An update call of 409,360 x 5,
// k = 19, labels in no order: 29 us (134 with a fold per warp and 32 rows, labels
// by reductions first; 57 with 1024 rows per warp), 1e6 x 5, k = 16 36 (121, 60).
constexpr int AS_CHUNK = 1024;   // rows per warp between folds (keeps each 32-bit part sum below 2^31)
constexpr int AS_MAX_KD = 512;   // k * d bound of this path
constexpr int AS_STAGES = 4;
constexpr int AS_FEW = 4;
constexpr int AS_RUNS = 8;
static size_t as_smem(int d, int k, bool wd) {
    const size_t parts = ((size_t)8 * (3 * (size_t)k * d + k) + 3) & ~(size_t)3;
    return parts * 4 + (size_t)8 * AS_STAGES * 32 * d * 4 + (wd ? (size_t)k * 32 : 0);
}
template <int D, bool WD, int NP>
__global__ void __launch_bounds__(256) k_accum_small(const float* __restrict__ X, int64_t n, int k, int chunk,
                                                     const int32_t* __restrict__ labels,
                                                     const unsigned* __restrict__ amax_bits, int64_t nscale,
                                                     long long* __restrict__ sums, long long* __restrict__ counts,
                                                     const float* __restrict__ C, double* __restrict__ md) {
    chain_enter();
    extern __shared__ __align__(16) unsigned acc_sm[];  // per warp: 3 k D parts, k counts; per warp: the ring; C (WD)
    const int S = fixed_shift(*amax_bits, nscale);
    if (FixedScale::two_parts(S, nscale) != (NP == 2)) return;  // (the other form's launch does the work)
    const FixedScale fx(S);
    const float f = __int_as_float((S + 127) << 23);
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int kd = k * D;
    unsigned* a = acc_sm + (size_t)wib * (3 * kd + k);
    unsigned* cntw = a + 3 * kd;
    const size_t parts = ((size_t)8 * (3 * kd + k) + 3) & ~(size_t)3;
    float* ring = reinterpret_cast<float*>(acc_sm + parts) + (size_t)wib * AS_STAGES * 32 * D;
    const uint32_t ring_s = smem_u32(ring);
    // C with rows of 8 floats (zero past D), 16-byte aligned: two vector reads per row
    float4* Cs = reinterpret_cast<float4*>(acc_sm + parts + (size_t)8 * AS_STAGES * 32 * D);
    if (WD) {
        for (int e = threadIdx.x; e < k * 8; e += blockDim.x) {
            const int j = e >> 3, l = e & 7;
            reinterpret_cast<float*>(Cs)[e] = l < D ? C[j * D + l] : 0.0f;
        }
        __syncthreads();
    }
    const bool staged = ((uintptr_t)X & 15) == 0;
    for (int64_t cb = (int64_t)blockIdx.x * 8 * chunk; cb < n; cb += (int64_t)gridDim.x * 8 * chunk) {
        for (int e = lane; e < 3 * kd + k; e += 32) a[e] = 0u;
        __syncwarp();
        const int64_t c0 = min(n, cb + wib * chunk), c1 = min(n, c0 + chunk);  // the warp's rows
        auto fetch = [&](int64_t base, int slot) {
            if (staged && base < c1) {
                const char* src = reinterpret_cast<const char*>(X + base * D);
                const int64_t left = (n - base) * D * 4;  // bytes
#pragma unroll
                for (int c = 0; c < (8 * D + 31) / 32; c++) {
                    const int q = lane + 32 * c;  // 16-byte piece
                    if (q < 8 * D) {
                        const int64_t rest = left - 16 * q;
                        const int bytes = rest >= 16 ? 16 : (rest > 0 ? (int)rest : 0);
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(
                                         ring_s + (uint32_t)(slot * 32 * D * 4 + 16 * q)),
                                     "l"(bytes ? src + 16 * q : reinterpret_cast<const char*>(X)), "r"(bytes)
                                     : "memory");
                    }
                }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        // parts of a run of whole steps with the label `cur`
        unsigned v[NP * D];
#pragma unroll
        for (int t = 0; t < NP * D; t++) v[t] = 0u;
        int cur = -1, steps = 0;
        auto flush = [&]() {
            if (steps) {
                unsigned mine = 0;
#pragma unroll
                for (int t = 0; t < NP * D; t++) {
                    const unsigned r = __reduce_add_sync(0xffffffffu, v[t] - (unsigned)steps * FixedScale::kBias);
                    if (lane == t) mine = r;
                    v[t] = 0u;
                }
                __syncwarp();
                // (lane t holds part NP - 1 - t % NP, the accumulators' order b2, b1, b0)
                if (lane < NP * D) a[3 * cur * D + 3 * (lane / NP) + (3 - NP) + lane % NP] += mine;
                if (lane == 0) cntw[cur] += 32u * (unsigned)steps;
                __syncwarp();
                steps = 0;
            }
        };
#pragma unroll
        for (int s = 0; s < AS_STAGES - 1; s++) fetch(c0 + 32 * s, s);
        int slot = 0;
        int jn = c0 + lane < c1 ? labels[c0 + lane] : -1;
        for (int64_t base = c0; base < c1; base += 32) {
            const int64_t i = base + lane;
            const bool valid = i < c1;
            const int j = jn;
            jn = i + 32 < c1 ? labels[i + 32] : -1;
            __syncwarp();
            fetch(base + 32 * (AS_STAGES - 1), slot == 0 ? AS_STAGES - 1 : slot - 1);
            asm volatile("cp.async.wait_group %0;" ::"n"(AS_STAGES - 1) : "memory");
            __syncwarp();
            float xr[D];
#pragma unroll
            for (int l = 0; l < D; l++) xr[l] = !valid ? 0.0f : (staged ? ring[(slot * 32 + lane) * D + l] : X[i * D + l]);
            slot = slot + 1 == AS_STAGES ? 0 : slot + 1;
            if (WD && valid) md[i] = df_value(df_small4<D>(xr, Cs[2 * j], D > 4 ? Cs[2 * j + 1] : make_float4(0.f, 0.f, 0.f, 0.f)));
            const int j0 = __shfl_sync(0xffffffffu, j, 0);
            const bool whole = __all_sync(0xffffffffu, valid && j == j0);
            unsigned u[NP * D];  // this row's parts (biased), b2 (NP = 3), b1, b0 per coordinate
#pragma unroll
            for (int l = 0; l < D; l += 2) {
                const float2 x2 = make_float2(xr[l], l + 1 < D ? xr[l + 1] : 0.0f);
                uint2 b2, b1, b0;
                if constexpr (NP == 2) fx.split2_low(x2, f, b1, b0);
                else fx.split2(x2, b2, b1, b0);
                if constexpr (NP == 3) u[NP * l] = b2.x;
                u[NP * l + NP - 2] = b1.x;
                u[NP * l + NP - 1] = b0.x;
                if (l + 1 < D) {
                    if constexpr (NP == 3) u[NP * (l + 1)] = b2.y;
                    u[NP * (l + 1) + NP - 2] = b1.y;
                    u[NP * (l + 1) + NP - 1] = b0.y;
                }
            }
            if (whole) {
                if (j0 != cur) {
                    flush();
                    cur = j0;
                }
#pragma unroll
                for (int t = 0; t < NP * D; t++) v[t] += u[t];
                steps++;
                continue;
            }
            // true (unbiased) parts modulo 2^32
#pragma unroll
            for (int t = 0; t < NP * D; t++) u[t] = u[t] - FixedScale::kBias;
            const unsigned vm = __ballot_sync(0xffffffffu, valid);
            const unsigned peers = __match_any_sync(0xffffffffu, j);
            const bool lead = valid && lane == __ffs(peers) - 1;
            unsigned rem = __ballot_sync(0xffffffffu, lead);  // each label's first lane
            if (__popc(rem) <= AS_FEW) {
                // one label after another, summed over its lanes by hardware reductions
                for (; rem; rem &= rem - 1) {
                    const int first = __ffs(rem) - 1;
                    const unsigned m = __shfl_sync(0xffffffffu, peers, first);
                    if ((m >> lane) & 1u) {
                        unsigned* aj = a + 3 * j * D;
#pragma unroll
                        for (int t = 0; t < NP * D; t++) {
                            const unsigned r = __reduce_add_sync(m, u[t]);
                            if (lane == first) aj[3 * (t / NP) + (3 - NP) + t % NP] += r;
                        }
                        if (lane == first) cntw[j] += (unsigned)__popc(m);
                    }
                    __syncwarp();
                }
                continue;
            }
            const int jp = __shfl_up_sync(0xffffffffu, j, 1);
            const bool head = lane == 0 || j != jp;
            if (__popc(__ballot_sync(0xffffffffu, head) & vm) > AS_RUNS) {  // each row by itself
                if (valid) {
                    unsigned* aj = a + 3 * j * D;
#pragma unroll
                    for (int t = 0; t < NP * D; t++) atomicAdd(&aj[3 * (t / NP) + (3 - NP) + t % NP], u[t]);
                    atomicAdd(&cntw[j], 1u);
                }
                __syncwarp();
                continue;
            }
            unsigned cnt = valid ? 1u : 0u;
#pragma unroll
            for (int t = 0; t < NP * D; t++) u[t] = valid ? u[t] : 0u;
            bool fl = head;  // segment flag of the scan
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
                const bool fu = __shfl_up_sync(0xffffffffu, fl, off);
                const bool take = lane >= off && !fl;
#pragma unroll
                for (int t = 0; t < NP * D; t++) {
                    const unsigned w = __shfl_up_sync(0xffffffffu, u[t], off);
                    if (take) u[t] += w;
                }
                const unsigned w = __shfl_up_sync(0xffffffffu, cnt, off);
                if (take) {
                    cnt += w;
                    fl = fu;
                }
            }
            const bool next_head = __shfl_down_sync(0xffffffffu, head, 1);
            const bool tail = lane == 31 || next_head;
            if (valid && tail) {
                unsigned* aj = a + 3 * j * D;
#pragma unroll
                for (int t = 0; t < NP * D; t++) atomicAdd(&aj[3 * (t / NP) + (3 - NP) + t % NP], u[t]);
                atomicAdd(&cntw[j], cnt);
            }
            __syncwarp();
        }
        flush();
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        // the eight warps' sums, one atomic each: the addresses are few
        for (int e = threadIdx.x; e < kd; e += blockDim.x) {
            long long s64 = 0;
            for (int w = 0; w < 8; w++) {
                const unsigned* aw = acc_sm + (size_t)w * (3 * kd + k) + 3 * e;
                s64 += FixedScale::combine(aw[0], aw[1], aw[2], 0u);
            }
            if (s64) atomicAdd(reinterpret_cast<unsigned long long*>(&sums[e]), (unsigned long long)s64);
        }
        for (int jj = threadIdx.x; jj < k; jj += blockDim.x) {
            unsigned c = 0;
            for (int w = 0; w < 8; w++) c += acc_sm[(size_t)w * (3 * kd + k) + 3 * kd + jj];
            if (c) atomicAdd(reinterpret_cast<unsigned long long*>(&counts[jj]), (unsigned long long)c);
        }
        __syncthreads();
    }
}

// ---- the winner's distance on its own (rows in natural order) ------------
// min_dist[i] = ||x_i - c_label(i)||^2 to binary64 accuracy, by the same
// arithmetic as the fused centre-sum passes above (df.cuh), so an assignment
// alone and an assignment followed by the centre update give the same bits.
// R rows per lane and pass (R <= LPR), G = 32 / LPR rows per load.
template <int NV4, int LPR, bool VEC>
__global__ void __launch_bounds__(256) k_winner_dist(const float* __restrict__ X, int64_t n, int d,
                                                     const float* __restrict__ C, const int32_t* __restrict__ labels,
                                                     double* __restrict__ md) {
    chain_enter();
    constexpr int G = 32 / LPR;
    constexpr int R = NV4 == 4 ? 2 : 4;  // 4 rows per pass: measured faster than 8 (occupancy)
    constexpr int STEP = R * G;
    static_assert(R <= LPR, "rows per lane exceed the lanes of a row");
    const int lane = threadIdx.x & 31, sub = lane / LPR, cl = lane % LPR;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int d4 = (d + 3) >> 2;
    for (int64_t base = w0 * STEP; base < n; base += nw * STEP) {
        const int jl = (lane < STEP && base + lane < n) ? labels[base + lane] : 0;
        float4 xv[R][NV4], cv[R][NV4];
#pragma unroll
        for (int b = 0; b < R; b++) {
            const int64_t row = base + b * G + sub;
            const int j = __shfl_sync(0xffffffffu, jl, b * G + sub);
#pragma unroll
            for (int u = 0; u < NV4; u++) {
                const int cidx = cl + LPR * u;
                const bool ok = row < n && cidx < d4;
                if (VEC) {
                    xv[b][u] = ok ? reinterpret_cast<const float4*>(X + row * d)[cidx] : make_float4(0.f, 0.f, 0.f, 0.f);
                    cv[b][u] = ok ? reinterpret_cast<const float4*>(C + (int64_t)j * d)[cidx]
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
                } else {
                    float xe[4], ce[4];
#pragma unroll
                    for (int t = 0; t < 4; t++) {
                        const int l = 4 * cidx + t;
                        xe[t] = (ok && l < d) ? X[row * d + l] : 0.0f;
                        ce[t] = (ok && l < d) ? C[(int64_t)j * d + l] : 0.0f;
                    }
                    xv[b][u] = make_float4(xe[0], xe[1], xe[2], xe[3]);
                    cv[b][u] = make_float4(ce[0], ce[1], ce[2], ce[3]);
                }
            }
        }
        DF part[R];
#pragma unroll
        for (int b = 0; b < R; b++) part[b] = df_lane<NV4>(xv[b], cv[b]);
        int rs;
        const DF r = df_rows<R, LPR>(part, cl, rs);
        const int64_t row = base + rs * G + sub;
        if ((cl & (LPR / R - 1)) == 0 && row < n) md[row] = df_value(r);
    }
}

// Rows of D <= 8 coordinates: one thread per row.
template <int D>
__global__ void __launch_bounds__(256) k_winner_small(const float* __restrict__ X, int64_t n,
                                                      const float* __restrict__ C, const int32_t* __restrict__ labels,
                                                      double* __restrict__ md) {
    chain_enter();
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int j = labels[i];
        float xr[D];
#pragma unroll
        for (int l = 0; l < D; l++) xr[l] = X[i * D + l];
        md[i] = df_value(df_small<D>(xr, C + (int64_t)j * D));
    }
}

cudaError_t launch_winner_dist(const float* X, int64_t n, int d, const float* C, const int32_t* labels, double* md,
                               int num_sms, cudaStream_t st) {
    if (n < 1) return cudaSuccess;
    if (d <= 8) {
        const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)num_sms * 8));
        switch (d) {
#define KM_WS(DD) \
    case DD: klaunch(k_winner_small<DD>, blocks, 256, 0, st, X, n, C, labels, md); break;
            KM_WS(1) KM_WS(2) KM_WS(3) KM_WS(4) KM_WS(5) KM_WS(6) KM_WS(7) KM_WS(8)
#undef KM_WS
        }
        return cudaGetLastError();
    }
    const bool vec = d % 4 == 0 && ((uintptr_t)X % 16) == 0 && ((uintptr_t)C % 16) == 0;
    const int lpr = df_lpr(d), nv4 = df_nv4(d);
    const void* fn = nullptr;
    void (*kern)(const float*, int64_t, int, const float*, const int32_t*, double*) = nullptr;
#define KM_WD(NV, L)                                                          \
    if (nv4 == NV && lpr == L) {                                              \
        if (vec) kern = k_winner_dist<NV, L, true>;                           \
        else kern = k_winner_dist<NV, L, false>;                              \
    }
    KM_WD(1, 8) KM_WD(1, 16) KM_WD(1, 32) KM_WD(2, 32) KM_WD(4, 32)
#undef KM_WD
    if (!kern) return cudaErrorInvalidValue;
    fn = (const void*)kern;
    int per_sm = 1;
    cudaError_t e = blocks_per_sm_of(fn, 256, 0, &per_sm);
    if (e != cudaSuccess) return e;
    const int rows_per_warp_pass = (nv4 == 4 ? 2 : 4) * (32 / lpr);
    const int64_t warps_needed = (n + rows_per_warp_pass - 1) / rows_per_warp_pass;
    const unsigned blocks = (unsigned)std::max<int64_t>(
        1, std::min<int64_t>((warps_needed + 7) / 8, (int64_t)num_sms * std::max(per_sm, 1)));
    klaunch(kern, blocks, 256, 0, st, X, n, d, C, labels, md);
    return cudaGetLastError();
}

// mean = sum 2^-S / m in binary64, stored in fp32 (the working precision);
// one warp per cluster.  shift_bits (nullable, zeroed): max_j ||c_new_j -
// c_old_j|| over the clusters with rows, as the bit pattern of a non-negative
// double (ordered like an integer, so the order does not matter); the reseeded
// clusters follow in k_empty_select, the kept ones do not move.
__global__ void __launch_bounds__(64) k_means(const long long* __restrict__ sums, const long long* __restrict__ counts,
                                               const unsigned* __restrict__ amax_bits, int64_t nscale, int k, int d,
                                               const float* __restrict__ C_old, float* __restrict__ C_new,
                                               int64_t* counts_out, unsigned long long* shift_bits) {
    chain_enter();
    const int S = fixed_shift(*amax_bits, nscale);
    const double unit = __hiloint2double((1023 - S) << 20, 0);  // 2^-S, S in [-98, 209]: the product is exact
    const int lane = threadIdx.x & 31;
    const int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t j = w0; j < k; j += nw) {
        const long long m = counts[j];
        double sq = 0.0;
        for (int l0 = lane; l0 < d; l0 += 128) {
            float old[4];
            long long sm[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int l = l0 + 32 * u;
                old[u] = l < d ? C_old[j * d + l] : 0.0f;
                sm[u] = l < d ? sums[j * d + l] : 0;
            }
            float c[4];
#pragma unroll
            for (int u = 0; u < 4; u++)  // int64 -> binary64 rounds once (2^-53 relative)
                c[u] = m > 0 && l0 - lane + 32 * u < d ? (float)((double)sm[u] * unit / (double)m) : old[u];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int l = l0 + 32 * u;
                if (l < d) C_new[j * d + l] = c[u];
                if (shift_bits && m > 0 && l0 - lane + 32 * u < d) {
                    const double df = (double)c[u] - (double)old[u];  // (0 past d)
                    sq = fma(df, df, sq);
                }
            }
        }
        if (lane == 0 && counts_out) counts_out[j] = m;
        if (shift_bits && m > 0) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
            if (lane == 0) atomicMax(shift_bits, (unsigned long long)__double_as_longlong(sqrt(sq)));
        }
    }
}

// ---- empty clusters: the rows with the largest min_dist ------------------
// KM_EMPTY_FARTHEST (reading of "automatic empty cluster reinitialisation",
// Section 6.2): the empty clusters, in ascending j, take the rows in
// decreasing order of min_dist, ties to the lowest row index, each row once.
// One cooperative launch over the resident blocks:
//   1. block 0 lists the empty clusters (E of them, ascending) and clears the
//      histograms; every block returns at once when E == 0;
//   2. radix select (up to eight passes of 8 bits, most significant first) of
//      T, the E-th largest min_dist bit pattern (non-negative doubles order
//      like their bits), and A, the number of rows above it; as soon as every
//      row of the digit picked is wanted, T is the digit's lowest pattern and
//      all rows from T on are the ones;
//   3. else, among the rows equal to T, radix select (four passes) of the
//      (E - A)-th smallest row index I;
//   4. the E rows {md > T} + {md == T, index <= I} are collected, ranked by
//      (md desc, index asc) and copied into the clusters in order.
// Work is O(n) per pass whatever E is; bound by the grid barriers, about 2 us
// each.  1e5 rows, a few empty clusters: 80 -> 10 us (the digits walked one L2
// read after another, and all twelve passes, before).  The blocks meet at a grid barrier
// whose every wait is bounded: on timeout the status word's timeout bit is
// set and the kernel winds down.
struct EmptySel {
    int nempty, ncollected;
    unsigned hist[12][256];       // 8 passes on the distance bits, 4 on the row index
};
size_t empty_select_bytes(int k) {
    return ((sizeof(EmptySel) + 255) & ~(size_t)255) + (size_t)k * (sizeof(int) + 16 + sizeof(int));
}

// bar: count and generation, both 0 at the launch
KM_DEV bool grid_barrier(unsigned* bar, unsigned nblocks, unsigned* status) {
    __shared__ int ok_sh;
    __syncthreads();
    if (threadIdx.x == 0) {
        int ok = 1;
        volatile unsigned* vgen = bar + 1;
        const unsigned g = *vgen;
        __threadfence();
        if (atomicAdd(bar, 1u) == nblocks - 1) {
            bar[0] = 0;
            __threadfence();
            atomicAdd(bar + 1, 1u);
        } else {
            const long long t0 = clock64();
            while (*vgen == g) {
                __nanosleep(64);
                if (clock64() - t0 > KM_WAIT_CYCLES) {
                    atomicOr(status, KM_DEVERR_TIMEOUT);
                    ok = 0;
                    break;
                }
            }
        }
        __threadfence();
        ok_sh = ok;
    }
    __syncthreads();
    return ok_sh != 0;
}

// From a pass's histogram: the digit holding the rank-th key (1-based) in the
// given direction (descending: from 255 down), the keys before that digit and
// in it.  All 256 threads take part: thread t holds the t-th digit in that
// direction, prefix sums over the warps, and the one that covers the rank
// tells the others (walked digit by digit, the L2 reads alone took 6 us a pass).
KM_DEV void radix_pick(const unsigned* hist, bool descending, unsigned rank, unsigned& digit, unsigned& before,
                       unsigned& in) {
    __shared__ unsigned wtot[8], pick[3];
    const int t = threadIdx.x, lane = t & 31;
    const unsigned dgt = descending ? 255u - t : (unsigned)t;
    const unsigned c = __ldcg(hist + dgt);  // written by other blocks' atomics
    unsigned incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
    }
    __syncthreads();  // (the previous call's readers are done)
    if (lane == 31) wtot[t >> 5] = incl;
    __syncthreads();
    for (int w = 0; w < (t >> 5); w++) incl += wtot[w];
    if (incl >= rank && incl - c < rank) {
        pick[0] = dgt;
        pick[1] = incl - c;
        pick[2] = c;
    }
    __syncthreads();
    digit = pick[0];
    before = pick[1];
    in = pick[2];
}

// fixed_e > 0: no cluster lists; the fixed_e rows of largest min_dist go, in
// that order, to rows_out / vals_out (a shard's candidates for the empty
// clusters of a row-sharded update).
__global__ void __launch_bounds__(256) k_empty_select(const long long* __restrict__ counts, int64_t n, int k, int d,
                                                      const float* __restrict__ X, const double* __restrict__ md,
                                                      const float* __restrict__ C_old, float* __restrict__ C_new,
                                                      unsigned long long* shift_bits, unsigned* bar, EmptySel* es,
                                                      int* __restrict__ empties, unsigned long long* __restrict__ keys,
                                                      int* __restrict__ rows, int* __restrict__ order,
                                                      unsigned* status, int fixed_e, long long* __restrict__ rows_out,
                                                      double* __restrict__ vals_out) {
    chain_enter();
    __shared__ unsigned sh[256];
    __shared__ int wsum[8];
    __shared__ int any_empty;
    const unsigned nb = gridDim.x;
    const int t = threadIdx.x;
    // 0. no empty cluster (the usual case): every block sees it in the counts
    //    and leaves at once, before any grid barrier
    if (fixed_e <= 0) {
        if (t == 0) any_empty = 0;
        __syncthreads();
        for (int j = t; j < k; j += blockDim.x)
            if (counts[j] == 0) any_empty = 1;
        __syncthreads();
        if (!any_empty) return;
    }
    // 1. the empty clusters in ascending j (block 0), histograms cleared
    if (blockIdx.x == 0) {
        for (int e = t; e < 12 * 256; e += blockDim.x) (&es->hist[0][0])[e] = 0u;
        int base = 0;
        if (fixed_e > 0) base = (int)min((int64_t)fixed_e, n);
        for (int j0 = 0; fixed_e <= 0 && j0 < k; j0 += blockDim.x) {
            const int j = j0 + t;
            const int e = (j < k && counts[j] == 0) ? 1 : 0;
            int incl = e;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, incl, o);
                if ((t & 31) >= o) incl += v;
            }
            if ((t & 31) == 31) wsum[t >> 5] = incl;
            __syncthreads();
            int pre = 0, tot = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); w++) {
                pre += (w < (t >> 5)) ? wsum[w] : 0;
                tot += wsum[w];
            }
            if (e) empties[base + pre + incl - 1] = j;
            base += tot;
            __syncthreads();
        }
        if (t == 0) {
            es->nempty = base;
            es->ncollected = 0;
        }
    }
    if (!grid_barrier(bar, nb, status)) return;
    const int E = *(volatile int*)&es->nempty;
    if (E == 0) return;
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + t, gstride = (int64_t)nb * blockDim.x;
    const unsigned long long* mdb = reinterpret_cast<const unsigned long long*>(md);
    // 2. T, the E-th largest distance pattern, and A, the rows above it
    unsigned long long prefix = 0, mask = 0;
    unsigned rank = (unsigned)E;
    bool whole = false;  // every row whose pattern starts with the prefix is wanted
    for (int pass = 0; pass < 8 && !whole; pass++) {
        const int shift = 56 - 8 * pass;
        sh[t] = 0;
        __syncthreads();
        for (int64_t i = gtid; i < n; i += gstride) {
            const unsigned long long key = mdb[i];
            if ((key & mask) == prefix) atomicAdd(&sh[(key >> shift) & 255u], 1u);
        }
        __syncthreads();
        if (sh[t]) atomicAdd(&es->hist[pass][t], sh[t]);
        if (!grid_barrier(bar, nb, status)) return;
        unsigned digit, before, in;
        radix_pick(es->hist[pass], true, rank, digit, before, in);
        rank -= before;
        whole = in == rank;
        prefix |= (unsigned long long)digit << shift;
        mask |= 255ull << shift;
    }
    const unsigned long long T = prefix;
    // 3. among the rows equal to T, the rank-th smallest index I (rank = E - A)
    unsigned iprefix = 0, imask = 0;
    for (int pass = 0; pass < 4 && !whole; pass++) {
        const int shift = 24 - 8 * pass;
        sh[t] = 0;
        __syncthreads();
        for (int64_t i = gtid; i < n; i += gstride) {
            if (mdb[i] == T && ((unsigned)i & imask) == iprefix) atomicAdd(&sh[((unsigned)i >> shift) & 255u], 1u);
        }
        __syncthreads();
        if (sh[t]) atomicAdd(&es->hist[8 + pass][t], sh[t]);
        if (!grid_barrier(bar, nb, status)) return;
        unsigned digit, before, in;
        radix_pick(es->hist[8 + pass], false, rank, digit, before, in);
        rank -= before;
        iprefix |= digit << shift;
        imask |= 255u << shift;
    }
    const unsigned I = whole ? 0xffffffffu : iprefix;
    // 4. collect the E rows, rank them, fill the clusters
    for (int64_t i = gtid; i < n; i += gstride) {
        const unsigned long long key = mdb[i];
        if (key > T || (key == T && (unsigned)i <= I)) {
            const int s = atomicAdd(&es->ncollected, 1);
            if (s < E) {
                keys[s] = key;
                rows[s] = (int)i;
            }
        }
    }
    if (!grid_barrier(bar, nb, status)) return;
    // (the lists were written by other blocks: read through L2)
    for (int64_t s = gtid; s < E; s += gstride) {
        const unsigned long long ks = __ldcg(keys + s);
        const int rs = __ldcg(rows + s);
        int r = 0;
        for (int q = 0; q < E; q++) {
            const unsigned long long kq = __ldcg(keys + q);
            r += (kq > ks || (kq == ks && __ldcg(rows + q) < rs)) ? 1 : 0;
        }
        order[r] = rs;
    }
    if (!grid_barrier(bar, nb, status)) return;
    if (fixed_e > 0) {
        for (int64_t r = gtid; r < E; r += gstride) {
            const int row = __ldcg(order + r);
            rows_out[r] = row;
            vals_out[r] = md[row];
        }
        return;
    }
    for (int64_t r = gtid >> 5; r < E; r += gstride >> 5) {  // a warp per cluster
        const int64_t j = __ldcg(empties + r), row = __ldcg(order + r);
        double sq = 0.0;
        for (int l = t & 31; l < d; l += 32) {
            const float c = X[row * d + l];
            C_new[j * d + l] = c;
            const double df = (double)c - (double)C_old[j * d + l];
            sq = fma(df, df, sq);
        }
        if (shift_bits) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
            if ((t & 31) == 0) atomicMax(shift_bits, (unsigned long long)__double_as_longlong(sqrt(sq)));
        }
    }
}

// Deterministic sum: a fixed partition into nparts chunks; a chunk is summed
// as 256 columns (column t adds rows t, t + 256, ... in order) folded by a
// halving tree; one warp adds the parts (lane l adds parts l, l + 32, ... in
// turn, then a butterfly).  The block that finishes last does that: one launch.
// WARP: a warp per part, eight columns per lane, the same tree (few rows per
// part: 1024 blocks of mostly idle threads took 7 us whatever n), else a
// block.  Bound by launch latency for few rows, by the FP64 pipe for many.
template <bool WARP>
__global__ void __launch_bounds__(256) k_sum(const double* __restrict__ v, int64_t n, int nparts, double* parts,
                                             double* __restrict__ out, unsigned* ticket) {
    chain_enter();
    __shared__ double red[256];
    __shared__ bool last;
    const int t = threadIdx.x, lane = t & 31;
    const int64_t chunk = (n + nparts - 1) / nparts;
    if (WARP) {
        const int part = blockIdx.x * 8 + (t >> 5);
        const int64_t b = part * chunk, e = min(n, b + chunk);
        double s[8];
#pragma unroll
        for (int i = 0; i < 8; i++) s[i] = 0.0;
        for (int64_t r = b + lane; r < e; r += 256)
#pragma unroll
            for (int i = 0; i < 8; i++)
                if (r + 32 * i < e) s[i] += v[r + 32 * i];
#pragma unroll
        for (int h = 4; h > 0; h >>= 1)
#pragma unroll
            for (int i = 0; i < h; i++) s[i] += s[i + h];
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s[0] += __shfl_down_sync(0xffffffffu, s[0], off);
        if (lane == 0 && part < nparts) parts[part] = s[0];
    } else {
        const int64_t b = (int64_t)blockIdx.x * chunk, e = min(n, b + chunk);
        double s = 0.0;
        for (int64_t i = b + t; i < e; i += 256) s += v[i];
        red[t] = s;
        __syncthreads();
        for (int st = 128; st > 0; st >>= 1) {
            if (t < st) red[t] += red[t + st];
            __syncthreads();
        }
        if (t == 0) parts[blockIdx.x] = red[0];
    }
    __threadfence();
    __syncthreads();
    if (t == 0) last = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;  // back to 0 for the next sum
    __syncthreads();
    if (!last || t >= 32) return;
    __threadfence();
    double s = 0.0;
#pragma unroll 8
    for (int i = lane; i < nparts; i += 32) s += __ldcg(parts + i);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane == 0) *out = s;
}

cudaError_t launch_absmax(const float* X, int64_t count, unsigned* out_bits, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(out_bits, 0, sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    int64_t blocks = min((int64_t)152 * 8, (count + 255) / 256);
    if (blocks < 1) blocks = 1;
    klaunch(k_absmax, (unsigned)blocks, 256, 0, st, X, count, out_bits);
    return cudaGetLastError();
}

cudaError_t launch_accumulate(const float* X, int64_t n, int d, const int32_t* labels, int k,
                              const unsigned* absmax_bits, long long* sums, long long* counts, int* iscratch,
                              int32_t* perm, int num_sms, cudaStream_t st, const float* C_wd, double* md_out,
                              int* nlaunch, int64_t nscale, bool zeroed) {
    if (nscale <= 0) nscale = n;  // the fixed-point scale of n rows (or of all shards' rows)
    // md_out: the rows' distances to their centres (C_wd) come out of the same
    // pass over X where the kernel has the row and its centre in hand, else
    // from the standalone kernel first (the same arithmetic either way)
    const bool want_wd = md_out != nullptr && C_wd != nullptr;
    int nl = 0;
    cudaError_t e = cudaSuccess;
    if (!zeroed) {
        e = cudaMemsetAsync(sums, 0, sizeof(long long) * (size_t)k * d, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(counts, 0, sizeof(long long) * (size_t)k, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(iscratch, 0, sizeof(int) * (size_t)k, st);
        if (e != cudaSuccess) return e;
    }
    // d <= 8: few rows of many clusters go to the general forms below
    const bool sparse = n <= 64 * (int64_t)k && n * d <= (int64_t)1 << 20;
    if (d <= 8 && (int64_t)k * d <= AS_MAX_KD && !sparse) {
        // small d: rows in order, per-warp shared accumulators (+ C for the distances)
        const size_t sm = as_smem(d, k, want_wd);
        // about two blocks per SM, so that few rows still reach all SMs while the folds,
        // k d + k atomics each on the same addresses, stay few
        const int chunk = (int)std::min<int64_t>(AS_CHUNK, std::max<int64_t>(32, (n / ((int64_t)num_sms * 16) + 31) / 32 * 32));
        const int64_t blocks = std::max<int64_t>(1, std::min<int64_t>((int64_t)num_sms * 8, (n + 8 * chunk - 1) / (8 * chunk)));
        typedef void (*SmallFn)(const float*, int64_t, int, int, const int32_t*, const unsigned*, int64_t, long long*,
                                long long*, const float*, double*);
        SmallFn three = nullptr, two = nullptr;
        switch (d) {
#define KM_ACC(DD)                                                                                             \
    case DD:                                                                                                   \
        three = want_wd ? (SmallFn)k_accum_small<DD, true, 3> : (SmallFn)k_accum_small<DD, false, 3>;          \
        two = want_wd ? (SmallFn)k_accum_small<DD, true, 2> : (SmallFn)k_accum_small<DD, false, 2>;            \
        break;
            KM_ACC(1) KM_ACC(2) KM_ACC(3) KM_ACC(4) KM_ACC(5) KM_ACC(6) KM_ACC(7) KM_ACC(8)
#undef KM_ACC
        }
        *nlaunch = 0;
        // two parts per value suffice from 2^22 rows on, whatever max |x| short of
        // the ends of the float range, where the three-part form still does the work
        int lgn = 0;
        while (((int64_t)1 << lgn) < nscale) lgn++;
        for (SmallFn fn : {61 - lgn <= 39 ? two : nullptr, three}) {
            if (!fn) continue;
            e = allow_max_smem(fn);
            if (e != cudaSuccess) return e;
            e = klaunch(fn, (unsigned)blocks, 256, sm, st, X, n, k, chunk, labels, absmax_bits, nscale, sums, counts,
                        want_wd ? C_wd : nullptr, want_wd ? md_out : nullptr);
            if (e != cudaSuccess) return e;
            ++*nlaunch;
        }
        return cudaSuccess;
    }
    const size_t hsm = sizeof(int) * (size_t)k;
    const bool vec = d % 4 == 0 && ((uintptr_t)X % 16) == 0;
    const bool can_bucket = 2 * hsm <= 200 * 1024 && d <= 512;
    const size_t smem = sizeof(long long) * ((size_t)k * d + k);
    typedef void (*RowsFn)(const float*, int64_t, int, const int32_t*, int, const unsigned*, int64_t, long long*, long long*,
                           const float*, double*);
    const bool v4 = vec && (!want_wd || ((uintptr_t)C_wd % 16) == 0);
    const int lpr = df_lpr(d), nv4 = df_nv4(d);
    // few coordinates per row, not too few clusters and many rows of each: shared sums,
    // folded once per block.  An update call of 100,000 x 10, k = 100 takes 32 us, 36 in the ordered
    // form below; 200,000 x 10, k = 200: 43 and 52.  With fewer clusters too many rows
    // share their addresses (131,072 x 16, k = 4: 46 and 34), with more the blocks'
    // folds weigh (131,072 x 16, k = 1000: 69 and 37).
    if (d <= 16 && k >= 32 && k * d <= 2048 && n > 64 * (int64_t)k && n * d <= (int64_t)1 << 21) {
        const RowsFn fn = v4 ? (want_wd ? (RowsFn)k_accum_rows<1, 8, true, true> : (RowsFn)k_accum_rows<1, 8, true, false>)
                             : (want_wd ? (RowsFn)k_accum_rows<1, 8, false, true> : (RowsFn)k_accum_rows<1, 8, false, false>);
        e = allow_max_smem(fn);
        if (e != cudaSuccess) return e;
        const int64_t blk = std::min<int64_t>(std::min<int64_t>((n + 255) / 256, num_sms), std::max<int64_t>(1, n / (4 * (int64_t)k)));
        *nlaunch = 1;
        return klaunch(fn, (unsigned)blk, 512, smem, st, X, n, d, labels, k, absmax_bits, nscale, sums, counts, C_wd, md_out);
    }
    // up to 2^21 coordinates, one launch of ordered sums in place of four bucketed
    // ones (16,384 x 64, k = 300: 30 against 47 us a call); up to 2^22 where the rows
    // are few (8000 x 512, k = 100: 45 and 54; 60,000 x 35, k = 4000: 47 and 63; but
    // 200,000 x 20, k = 200: 53 and 42; 400,000 x 10, k = 100: 89 and 53)
    if (d <= 512 && (n * d <= (int64_t)1 << 21 || (n * d <= (int64_t)1 << 22 && n <= (v4 ? 1 << 15 : 1 << 16)))) {
        RowsFn fn = nullptr;
#define KM_AO(NV, L)                                                                                                       \
    if (nv4 == NV && lpr == L)                                                                                             \
        fn = v4 ? (want_wd ? (RowsFn)k_accum_ordered<NV, L, true, true> : (RowsFn)k_accum_ordered<NV, L, true, false>)     \
                : (want_wd ? (RowsFn)k_accum_ordered<NV, L, false, true> : (RowsFn)k_accum_ordered<NV, L, false, false>);
        KM_AO(1, 8) KM_AO(1, 16) KM_AO(1, 32) KM_AO(2, 32) KM_AO(4, 32)
#undef KM_AO
        if (!fn) return cudaErrorInvalidValue;
        // as many rows per block as its shared memory takes, halved while the SMs
        // would not all have a block
        const int ldx = (d + 3) / 4 * 4;
        int rb = AO_ROWS;
        while (rb > 16 && (rb * ldx > AO_FLOATS || (n + rb - 1) / rb < num_sms)) rb >>= 1;
        *nlaunch = 1;
        return klaunch(fn, (unsigned)((n + rb - 1) / rb), 256, (size_t)rb * ldx * sizeof(float), st, X, n, d, labels, rb,
                       absmax_bits, nscale, sums, counts, C_wd, md_out);
    }
    const bool bucket = can_bucket;
    // the bucket kernels of rows wider than 5 coordinates take the distances along
    const bool wide = d > 5 || d == 4;
    const bool fused = want_wd && bucket && wide;
    const bool bvec = vec && (!fused || ((uintptr_t)C_wd % 16) == 0);
    if (want_wd && !fused) {
        e = launch_winner_dist(X, n, d, C_wd, labels, md_out, num_sms, st);
        if (e != cudaSuccess) return e;
        nl++;
    }
    if (bucket) {
        int* cnt32 = iscratch;            // k
        int* off = iscratch + k;          // k + 1
        int* cursor = off + k + 1;        // k
        int* item_off = cursor + k;       // k + 1
        const int64_t nblk = (n + SCAT_ROWS - 1) / SCAT_ROWS;
        e = allow_max_smem(k_label_hist);
        if (e != cudaSuccess) return e;
        klaunch(k_label_hist, (unsigned)nblk, 512, hsm, st, labels, n, k, cnt32);
        // persistent grid: every block resident at once (a partial second wave
        // would leave SMs idle), the items strided over the warps; work items of
        // `seg` rows, about four per resident warp (fewer, longer items mean
        // fewer atomic adds per centre coordinate)
        typedef void (*BucketFn)(const float*, int, int, int, int, const int*, const int*, const int32_t*,
                                 const unsigned*, int64_t, long long*, const float*, double*);
        BucketFn bfn = nullptr;
        if (wide) {
#define KM_BS(NV, L)                                                                                              \
    (fused ? (bvec ? (BucketFn)k_bucket_sum<NV, L, true, true> : (BucketFn)k_bucket_sum<NV, L, true, false>)      \
           : (bvec ? (BucketFn)k_bucket_sum<NV, L, false, true> : (BucketFn)k_bucket_sum<NV, L, false, false>))
            bfn = d <= 32 ? KM_BS(1, 8) : d <= 64 ? KM_BS(1, 16) : d <= 128 ? KM_BS(1, 32) : d <= 256 ? KM_BS(2, 32)
                                                                                                 : KM_BS(4, 32);
#undef KM_BS
        }
        int per_sm = 8;
        if (bfn) {
            e = blocks_per_sm_of((const void*)bfn, 256, 0, &per_sm);
            if (e != cudaSuccess) return e;
        }
        const int64_t resident_warps = (int64_t)num_sms * std::max(per_sm, 1) * 8;
        // (at least 64 rows where that still makes two items per warp: 500,000 x 12, k = 20
        // 83 us a call with items of 32 rows, 72 of 64; 100,000 x 128, k = 500 47 and 49)
        const int64_t least = n >= 128 * resident_warps ? 64 : 32;
        const int seg = (int)std::min<int64_t>(SEG_MAX, std::max<int64_t>(least, n / (resident_warps * 4) / 32 * 32));
        const int big = seg < 64 ? (int)std::max<int64_t>(1, n / 4) : INT32_MAX;
        klaunch(k_bucket_scan, 1, 1024, 0, st, cnt32, k, seg, big, off, cursor, item_off, counts);
        e = allow_max_smem(k_bucket_scatter);
        if (e != cudaSuccess) return e;
        klaunch(k_bucket_scatter, (unsigned)nblk, 512, 2 * hsm, st, labels, n, k, cursor, perm);
        const int64_t items = n / seg + k + 1;
        const unsigned blocks =
            (unsigned)std::max<int64_t>(1, std::min<int64_t>((items * 32 + 255) / 256, (int64_t)num_sms * std::max(per_sm, 1)));
        if (d == 1) klaunch(k_bucket_sum_small<1>, blocks, 256, 0, st, X, k, seg, big, off, item_off, perm, absmax_bits, nscale, sums);
        else if (d == 2) klaunch(k_bucket_sum_small<2>, blocks, 256, 0, st, X, k, seg, big, off, item_off, perm, absmax_bits, nscale, sums);
        else if (d == 3) klaunch(k_bucket_sum_small<3>, blocks, 256, 0, st, X, k, seg, big, off, item_off, perm, absmax_bits, nscale, sums);
        else if (d == 5) klaunch(k_bucket_sum_small<5>, blocks, 256, 0, st, X, k, seg, big, off, item_off, perm, absmax_bits, nscale, sums);
        else klaunch(bfn, blocks, 256, 0, st, X, d, k, seg, big, off, item_off, perm, absmax_bits, nscale, sums, C_wd, md_out);
        if (nlaunch) *nlaunch = nl + 4;
        return cudaGetLastError();
    }
    const int64_t blk = std::max<int64_t>(1, std::min<int64_t>((int64_t)num_sms * 8, (n * d + 511) / 512));
    if (nlaunch) *nlaunch = nl + 1;
    return klaunch(k_accumulate, (unsigned)blk, 512, 0, st, X, n, d, labels, k, absmax_bits, nscale, sums, counts);
}

cudaError_t launch_finalize(const long long* sums, const long long* counts, const unsigned* absmax_bits,
                            int64_t n, int k, int d, const float* C_old, int empty_policy, const float* X,
                            const double* min_dist, float* C_new, int64_t* counts_out, double* shift, unsigned* bar,
                            void* esel, unsigned* status, int num_sms, cudaStream_t st, int* nlaunch, int64_t nscale) {
    unsigned long long* shift_bits = reinterpret_cast<unsigned long long*>(shift);
    // (bound by the FP64 pipes: small blocks, so that few clusters reach all SMs)
    const int64_t blocks = std::min<int64_t>(((int64_t)k * 32 + 63) / 64, (int64_t)num_sms * 16);
    cudaError_t e = klaunch(k_means, (unsigned)blocks, 64, 0, st, sums, counts, absmax_bits, nscale > 0 ? nscale : n, k, d,
                            C_old, C_new, counts_out, shift_bits);
    if (e != cudaSuccess) return e;
    *nlaunch = 1;
    if (empty_policy == 1 && min_dist != nullptr) {
        EmptySel* es = reinterpret_cast<EmptySel*>(esel);
        char* tail = reinterpret_cast<char*>(esel) + ((sizeof(EmptySel) + 255) & ~(size_t)255);
        int* empties = reinterpret_cast<int*>(tail);
        unsigned long long* keys = reinterpret_cast<unsigned long long*>(empties + k + (k & 1));
        int* rows = reinterpret_cast<int*>(keys + k);
        int* order = rows + k;
        // one block per SM: every block resident at once (cooperative launch)
        int fixed_e = 0;
        long long* rows_out = nullptr;
        double* vals_out = nullptr;
        void* args[] = {(void*)&counts, (void*)&n,     (void*)&k,     (void*)&d,      (void*)&X,
                        (void*)&min_dist, (void*)&C_old, (void*)&C_new, (void*)&shift_bits, (void*)&bar, (void*)&es,
                        (void*)&empties, (void*)&keys, (void*)&rows,   (void*)&order, (void*)&status, (void*)&fixed_e,
                        (void*)&rows_out, (void*)&vals_out};
        e = cudaLaunchCooperativeKernel((const void*)k_empty_select, dim3((unsigned)num_sms), dim3(256), args, 0, st);
        if (e != cudaSuccess) return e;
        ++*nlaunch;
    }
    return cudaSuccess;
}

cudaError_t launch_farthest_rows(const double* min_dist, int64_t n, int e, long long* rows_out, double* vals_out,
                                 unsigned* bar, void* esel, unsigned* status, int num_sms, cudaStream_t st) {
    EmptySel* es = reinterpret_cast<EmptySel*>(esel);
    char* tail = reinterpret_cast<char*>(esel) + ((sizeof(EmptySel) + 255) & ~(size_t)255);
    int* empties = reinterpret_cast<int*>(tail);
    unsigned long long* keys = reinterpret_cast<unsigned long long*>(empties + e + (e & 1));
    int* rows = reinterpret_cast<int*>(keys + e);
    int* order = rows + e;
    const long long* counts = nullptr;
    int k = e, d = 0;
    const float *X = nullptr, *C_old = nullptr;
    float* C_new = nullptr;
    unsigned long long* shift_bits = nullptr;
    void* args[] = {(void*)&counts, (void*)&n,     (void*)&k,     (void*)&d,  (void*)&X,    (void*)&min_dist,
                    (void*)&C_old,  (void*)&C_new,  (void*)&shift_bits, (void*)&bar, (void*)&es,    (void*)&empties,
                    (void*)&keys, (void*)&rows, (void*)&order, (void*)&status, (void*)&e,     (void*)&rows_out,
                    (void*)&vals_out};
    return cudaLaunchCooperativeKernel((const void*)k_empty_select, dim3((unsigned)num_sms), dim3(256), args, 0, st);
}

cudaError_t launch_sum_f64(const double* v, int64_t n, double* partials, int nparts, double* out, unsigned* ticket,
                           cudaStream_t st) {
    // up to four rows per column of a part, a warp keeps up with the loads
    if (n <= (int64_t)nparts * 1024) klaunch(k_sum<true>, (nparts + 7) / 8, 256, 0, st, v, n, nparts, partials, out, ticket);
    else klaunch(k_sum<false>, nparts, 256, 0, st, v, n, nparts, partials, out, ticket);
    return cudaGetLastError();
}

}  // namespace km
