// k_direct.cu -- direct-formula assignment kernels, Eq. (dist-direct).
//
//  * k_direct_assign<double>: the plain FP64 path (every pair in binary64).
//  * k_direct_tiled, its general form k_direct_assign<float> and (d <= 8, few
//    centres) k_direct_small: fp32 direct distances for the fp32 path and for rows
//    whose tensor-core candidate list overflowed.  Theorem 4.1 bounds each value's
//    error (common.cuh); a row whose best and second-best intervals overlap is
//    not certified and its open centres are decided in binary64 by the same block
//    (resolve_row) or warp, lowest index on ties: products and sums rounded
//    separately (no FMA), equal to the CPU oracle's bit for bit.
//  * k_rows_full: the same for listed rows of more than 256 coordinates, a block
//    per row.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "df.cuh"
#include "internal.h"
#include "rowstat.cuh"

namespace km {

constexpr int DA_ROWS = 128;  // rows (threads) per block
constexpr int DA_TC = 32;     // centres per shared-memory tile

template <typename T>
__global__ void __launch_bounds__(DA_ROWS, 5) k_direct_assign(const float* __restrict__ X, int64_t n,
                                                         const float* __restrict__ C, int k, int d,
                                                         int32_t* __restrict__ labels, double* __restrict__ min_dist,
                                                         unsigned* __restrict__ absmax_out) {
    chain_enter();
    extern __shared__ __align__(16) unsigned char smem[];
    float amx = 0.0f;  // largest |x| this thread stages (absmax_out)
    const int ldx = d + 1;
    float* Xs = reinterpret_cast<float*>(smem);
    T* Cs = reinterpret_cast<T*>(smem + (((size_t)DA_ROWS * ldx * sizeof(float) + 15) & ~(size_t)15));
    const int tid = threadIdx.x;
    for (int64_t base = (int64_t)blockIdx.x * DA_ROWS; base < n; base += (int64_t)gridDim.x * DA_ROWS) {
        const int rows_here = (int)min((int64_t)DA_ROWS, n - base);
        for (int e = tid; e < rows_here * d; e += DA_ROWS) {
            const int r = e / d, l = e - r * d;
            const float xv = X[(base + r) * d + l];
            amx = fmaxf(amx, fabsf(xv));
            Xs[r * ldx + l] = xv;
        }
        T b1 = (T)INFINITY;
        int j1 = 0;
        for (int c0 = 0; c0 < k; c0 += DA_TC) {
            const int tc = min(DA_TC, k - c0);
            __syncthreads();
            for (int e = tid; e < tc * d; e += DA_ROWS) Cs[e] = (T)C[(int64_t)c0 * d + e];
            __syncthreads();
            if (tid < rows_here) {
                T acc[DA_TC];
#pragma unroll
                for (int c = 0; c < DA_TC; c++) acc[c] = (T)0;
                const float* xr = Xs + tid * ldx;
                for (int l = 0; l < d; l++) {
                    const T xl = (T)xr[l];
#pragma unroll
                    for (int c = 0; c < DA_TC; c++) {
                        if (c < tc) {
                            const T t = xl - Cs[c * d + l];
                            acc[c] = fma(t, t, acc[c]);
                        }
                    }
                }
#pragma unroll
                for (int c = 0; c < DA_TC; c++)
                    if (c < tc && acc[c] < b1) {
                        b1 = acc[c];
                        j1 = c0 + c;
                    }
            }
        }
        if (tid < rows_here) {
            labels[base + tid] = j1;
            min_dist[base + tid] = (double)b1;
        }
        __syncthreads();
    }
    if (absmax_out) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) amx = fmaxf(amx, __shfl_xor_sync(0xffffffffu, amx, off));
        if ((threadIdx.x & 31) == 0) atomicMax(absmax_out, __float_as_uint(amx));
    }
}

// Exact argmin of one row by a block of 256 threads: fp32 direct values of all
// centres (a warp per centre, four centres at a time: coalesced reads of C),
// Theorem 4.1's intervals, and binary64 (oracle arithmetic: products and sums
// rounded separately, coordinates in order) only for the centres whose
// interval can still hold the minimum.  Up to RF_OPEN of those take a warp
// each (products in parallel, one lane adds them in order); more take a thread
// each.
// Latency-bound: such rows are few.  440 rows x 1024 centres, d = 128: 742 us
// with binary64 values of every centre, 77 us with the fp32 values first.
constexpr int RF_OPEN = 64;
struct Top2 {
    float b1, b2;
    int j1;
};
KM_DEV Top2 top2_merge(Top2 A, Top2 B) {
    Top2 r;
    if (B.b1 < A.b1 || (B.b1 == A.b1 && B.j1 < A.j1)) {
        r.b1 = B.b1; r.j1 = B.j1; r.b2 = fminf(A.b1, B.b2);
    } else {
        r.b1 = A.b1; r.j1 = A.j1; r.b2 = fminf(A.b2, B.b1);
    }
    return r;
}

KM_DEV double direct64(const float* x, const float* c, int d) {
    double s = 0.0;
    for (int l = 0; l < d; l++) {
        const double t = __dsub_rn((double)x[l], (double)c[l]);
        s = __dadd_rn(s, __dmul_rn(t, t));
    }
    return s;
}

// fp32 direct values of centres j, j + 1, .., j + 3 (those below k): all lanes
// of the warp return the same four sums.
KM_DEV void warp_direct4(const float* xs, const float* __restrict__ C, int k, int d, int j, int lane, float (&v)[4]) {
#pragma unroll
    for (int q = 0; q < 4; q++) v[q] = 0.0f;
    // 16 loads in flight per lane
    for (int l0 = lane; l0 < d; l0 += 128) {
        float c[4][4], x[4];
#pragma unroll
        for (int u = 0; u < 4; u++) {
            const int l = l0 + 32 * u;
            x[u] = l < d ? xs[l] : 0.0f;
#pragma unroll
            for (int q = 0; q < 4; q++) c[u][q] = l < d && j + q < k ? C[(int64_t)(j + q) * d + l] : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < 4; u++)
#pragma unroll
            for (int q = 0; q < 4; q++) v[q] = fmaf(x[u] - c[u][q], x[u] - c[u][q], v[q]);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
#pragma unroll
        for (int q = 0; q < 4; q++) v[q] += __shfl_xor_sync(0xffffffffu, v[q], off);
}

// The bytes of scratch that a row of d coordinates takes; what is left of the
// scratch's `floats` after them holds the k fp32 values when they fit (else
// they are formed twice).
__host__ __device__ constexpr size_t resolve_bytes(int d) { return (size_t)d * (8 * sizeof(double) + sizeof(float)); }
// scratch: 16-byte aligned shared memory of `bytes` >= resolve_bytes(d).
// Returns true when binary64 was needed.
__device__ __noinline__ bool resolve_row(const float* __restrict__ X, const float* __restrict__ C, int k, int d,
                                         int64_t i, float gamma32, int32_t* __restrict__ labels,
                                         double* __restrict__ min_dist, void* scratch, size_t bytes,
                                         unsigned long long* ev64) {
    double* prod = reinterpret_cast<double*>(scratch);            // 8 x d products
    float* xs = reinterpret_cast<float*>(prod + (size_t)8 * d);   // d
    float* vs = xs + d;
    const bool keep_vals = bytes - resolve_bytes(d) >= (size_t)k * sizeof(float);
    __shared__ Top2 red[8];
    __shared__ double rv[8];
    __shared__ int rj[8];
    __shared__ int open_j[RF_OPEN], nopen;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    __syncthreads();
    for (int l = tid; l < d; l += 256) xs[l] = X[i * d + l];
    if (tid == 0) nopen = 0;
    __syncthreads();
    Top2 t{INFINITY, INFINITY, 0x7fffffff};
    for (int j = 4 * wid; j < k; j += 32) {
        float v[4];
        warp_direct4(xs, C, k, d, j, lane, v);
#pragma unroll
        for (int q = 0; q < 4; q++)
            if (j + q < k) {
                if (keep_vals && lane == 0) vs[j + q] = v[q];
                t = top2_merge(t, Top2{v[q], INFINITY, j + q});
            }
    }
    if (lane == 0) red[wid] = t;
    __syncthreads();
    t = red[0];
    for (int q = 1; q < 8; q++) t = top2_merge(t, red[q]);
    const float thr = direct_upper(t.b1, gamma32, direct_tiny(d));
    if (direct_lower(t.b2, gamma32) > thr) {
        if (tid == 0) {
            labels[i] = t.j1;
            min_dist[i] = (double)t.b1;
        }
        return false;
    }
    double best = INFINITY;
    int arg = 0x7fffffff;
    if (keep_vals) {
        for (int j = tid; j < k; j += 256)
            if (direct_lower(vs[j], gamma32) <= thr) {
                const int p = atomicAdd(&nopen, 1);
                if (p < RF_OPEN) open_j[p] = j;
            }
    } else {
        for (int j = 4 * wid; j < k; j += 32) {  // the same values as above
            float v[4];
            warp_direct4(xs, C, k, d, j, lane, v);
#pragma unroll
            for (int q = 0; q < 4; q++)
                if (lane == 0 && j + q < k && direct_lower(v[q], gamma32) <= thr) {
                    const int p = atomicAdd(&nopen, 1);
                    if (p < RF_OPEN) open_j[p] = j + q;
                }
        }
    }
    __syncthreads();
    const int no = nopen;
    if (no <= RF_OPEN) {
        double* pw = prod + (size_t)wid * d;
        for (int o = wid; o < no; o += 8) {
            const int j = open_j[o];
            const float* c = C + (int64_t)j * d;
            for (int l = lane; l < d; l += 32) {
                const double u = __dsub_rn((double)xs[l], (double)c[l]);
                pw[l] = __dmul_rn(u, u);
            }
            __syncwarp();
            if (lane == 0) {
                double s = 0.0;
#pragma unroll 8
                for (int l = 0; l < d; l++) s = __dadd_rn(s, pw[l]);
                if (s < best || (s == best && j < arg)) { best = s; arg = j; }
                ++*ev64;
            }
            __syncwarp();
        }
    } else {
        // (the open list did not fit: every centre it would have held)
        for (int j = tid; j < k; j += 256) {
            if (keep_vals && !(direct_lower(vs[j], gamma32) <= thr)) continue;
            const double s = direct64(xs, C + (int64_t)j * d, d);
            ++*ev64;
            if (s < best) { best = s; arg = j; }
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, off);
        const int oa = __shfl_xor_sync(0xffffffffu, arg, off);
        if (ob < best || (ob == best && oa < arg)) { best = ob; arg = oa; }
    }
    if (lane == 0) { rv[wid] = best; rj[wid] = arg; }
    __syncthreads();
    if (tid == 0) {
        best = rv[0];
        arg = rj[0];
        for (int q = 1; q < 8; q++)
            if (rv[q] < best || (rv[q] == best && rj[q] < arg)) { best = rv[q]; arg = rj[q]; }
        labels[i] = arg < k ? arg : 0;  // (no value to compare, NaN: a valid label all the same)
        min_dist[i] = best;
    }
    return true;
}

// The same by one warp for a row whose smallest fp32 value is known: thr =
// direct_upper of it.  Every centre whose interval reaches down to thr is evaluated
// in binary64, up to four at a time (their products by all lanes, a lane each adds
// one's in order).  scratch: the warp's `bytes` of shared memory, 16-byte aligned,
// at least rw_bytes(d, 1).
constexpr int RW_LIST = 32;  // candidates per evaluation
__host__ __device__ constexpr size_t rw_bytes(int d, int batch) {
    return (size_t)batch * d * sizeof(double) + ((size_t)d + RW_LIST) * sizeof(float);
}
__device__ __noinline__ void warp_resolve_row(const float* __restrict__ X, const float* __restrict__ C, int k, int d, int64_t i,
                                              float thr, float gamma32, int32_t* __restrict__ labels,
                                              double* __restrict__ min_dist, void* scratch, size_t bytes,
                                              unsigned long long* ev64) {
    const int lane = threadIdx.x & 31;
    const int batch = bytes >= rw_bytes(d, 4) ? 4 : (bytes >= rw_bytes(d, 2) ? 2 : 1);
    double* prod = reinterpret_cast<double*>(scratch);                  // batch x d products
    float* xs = reinterpret_cast<float*>(prod + (size_t)batch * d);     // d
    int* js = reinterpret_cast<int*>(xs + d);                           // RW_LIST
    __syncwarp();
    for (int l = lane; l < d; l += 32) xs[l] = X[i * d + l];
    __syncwarp();
    double best = INFINITY;
    int arg = 0x7fffffff, cnt = 0;
    auto evaluate = [&]() {
        __syncwarp();
        for (int b0 = 0; b0 < cnt; b0 += batch) {
            const int nb = min(batch, cnt - b0);
            for (int b = 0; b < nb; b++) {
                const float* c = C + (int64_t)js[b0 + b] * d;
                for (int l = lane; l < d; l += 32) {
                    const double u = __dsub_rn((double)xs[l], (double)c[l]);
                    prod[b * d + l] = __dmul_rn(u, u);
                }
            }
            __syncwarp();
            if (lane < nb) {
                const int j = js[b0 + lane];
                double t = 0.0;
#pragma unroll 8
                for (int l = 0; l < d; l++) t = __dadd_rn(t, prod[lane * d + l]);
                if (t < best || (t == best && j < arg)) { best = t; arg = j; }
                ++*ev64;
            }
            __syncwarp();
        }
        cnt = 0;
    };
    if (d < 32) {  // a centre per lane
        const bool vec = d % 4 == 0 && ((uintptr_t)C & 15) == 0;
        for (int j0 = 0; j0 < k; j0 += 32) {
            const int j = j0 + lane;
            float v = 0.0f;
            if (j < k && vec) {
                const float4* c4 = reinterpret_cast<const float4*>(C + (int64_t)j * d);
                for (int l = 0; l < d; l += 4) {
                    const float4 c = c4[l >> 2];
                    const float t0 = xs[l] - c.x, t1 = xs[l + 1] - c.y, t2 = xs[l + 2] - c.z, t3 = xs[l + 3] - c.w;
                    v = fmaf(t0, t0, v);
                    v = fmaf(t1, t1, v);
                    v = fmaf(t2, t2, v);
                    v = fmaf(t3, t3, v);
                }
            } else if (j < k) {
                for (int l = 0; l < d; l++) {
                    const float t = xs[l] - C[(int64_t)j * d + l];
                    v = fmaf(t, t, v);
                }
            }
            const unsigned m = __ballot_sync(0xffffffffu, j < k && direct_lower(v, gamma32) <= thr);
            if (!m) continue;
            if ((m >> lane) & 1u) js[__popc(m & ((1u << lane) - 1u))] = j;
            cnt = __popc(m);
            evaluate();
        }
    } else {
        for (int j0 = 0; j0 < k; j0 += 4) {
            float v[4];
            warp_direct4(xs, C, k, d, j0, lane, v);
#pragma unroll
            for (int q = 0; q < 4; q++)
                if (j0 + q < k && direct_lower(v[q], gamma32) <= thr) {
                    if (lane == 0) js[cnt] = j0 + q;
                    cnt++;
                }
            if (cnt > RW_LIST - 4) evaluate();
        }
        evaluate();
    }
#pragma unroll
    for (int off = 4; off > 0; off >>= 1) {  // (four lanes at most have evaluated)
        const double ob = __shfl_xor_sync(0xffffffffu, best, off);
        const int oa = __shfl_xor_sync(0xffffffffu, arg, off);
        if (ob < best || (ob == best && oa < arg)) { best = ob; arg = oa; }
    }
    if (lane == 0) {
        labels[i] = arg < k ? arg : 0;  // (no value to compare, NaN: a valid label all the same)
        min_dist[i] = best;
    }
}

// A block's open rows: a warp each, eight at a time; the block, quicker on a row by
// itself (its warps share the centres and the binary64 sums), takes a small rest in
// turn (146,112 x 256, k = 9, an open row in most blocks: 170 us so, 193 by a warp).
// scratch: resolve_bytes(d) at least, and 8 (rw_bytes(d, 1) + 16).
__device__ __noinline__ void resolve_open(const float* __restrict__ X, const float* __restrict__ C, int k, int d,
                                          const int* rows, const float* thr, int no, float gamma32,
                                          int32_t* __restrict__ labels, double* __restrict__ min_dist, void* scratch,
                                          size_t bytes, unsigned long long* ev64) {
    const int wid = threadIdx.x >> 5;
    const int byw = no % 8 > (k <= 64 ? 2 : 5) ? no : no & ~7;
    const size_t per = bytes / 8 & ~(size_t)15;
    for (int o = wid; o < byw; o += 8)
        warp_resolve_row(X, C, k, d, rows[o], thr[o], gamma32, labels, min_dist, static_cast<char*>(scratch) + wid * per, per, ev64);
    for (int o = byw; o < no; o++) resolve_row(X, C, k, d, rows[o], gamma32, labels, min_dist, scratch, bytes, ev64);
}

// Tiled fp32 direct distances, Eq. (dist-direct), any d (rows whose candidate
// list overflowed, the fp32 direct path, km_assign_static): 32 RPT rows per
// round resident in shared memory (zero-padded to a multiple of 4
// coordinates), the centres streamed through it in tiles of 64, DT_DK
// coordinates at a time (cp.async, two buffers).  Each thread holds RPT rows
// x 8 centres and takes two coordinates per packed instruction: the even and
// the odd coordinates are summed separately and then added, a summation order
// Theorem 4.1's bound covers like any other.  Per row the smallest and
// second-smallest value and the first index of the smallest (ties: lowest
// index), merged over the 8 threads of the row; rows that Theorem 4.1's
// intervals leave open are resolved by the block before its next round (a
// launch of its own for them cost every call 3 us).
// Bound by the FP32 pipe (two lane operations per pair and coordinate).
// Chunking the coordinates keeps the block at 111 KB or less, so two blocks
// share an SM and one computes while the other waits at a tile's barrier.
// Measured: 1e6 x 128 against 1024 centres 10.14 -> 9.67 ms (0.69 of the FP32
// pipe at its top clock; the block per SM before it had one 64 x d tile per
// barrier); 81,000 listed rows x 256, k = 389: 5.61 -> 0.81 ms and 60,013 x 50,
// k = 203: 0.197 -> 0.098 ms (a thread per row before, one to three blocks per SM).
constexpr int DT_C = 64;    // centres per tile
constexpr int DT_DK = 64;   // coordinates per streamed chunk

template <int BYTES>
KM_DEV void cp_async(uint32_t dst, const void* src) {
    if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(dst), "l"(src), "n"(BYTES) : "memory");
}
KM_DEV void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
KM_DEV void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Row stride (floats) of w staged coordinates (a multiple of 4): an odd number
// of 16-byte slots, so eight consecutive rows' reads fall on different banks.
__host__ __device__ constexpr int dt_stride(int w) { return (w / 4) % 2 ? w : w + 4; }
constexpr size_t dt_smem(int rpt, int d) {
    const int dp = (d + 3) & ~3, w = dp < DT_DK ? dp : DT_DK;
    return ((size_t)32 * rpt * dt_stride(dp) + (size_t)2 * DT_C * dt_stride(w)) * sizeof(float);
}

// VEC: floats per load (4, 2 or 1: what d and the pointers' alignment allow)
template <int RPT, int VEC>
KM_DEV void direct_tiled(const float* __restrict__ X, int64_t n, const float* __restrict__ C, int k, int d,
                         const int32_t* __restrict__ row_list, const int* __restrict__ row_count,
                         int32_t* __restrict__ labels, double* __restrict__ min_dist, DevCounters* cnt, float gamma32, unsigned* __restrict__ absmax_out) {
    extern __shared__ __align__(16) float dts[];
    constexpr int R = 32 * RPT;
    const int dp = (d + 3) & ~3, cw = min(dp, DT_DK);
    const int ldx = dt_stride(dp), ldc = dt_stride(cw);
    float* Xs = dts;
    float* Cs = dts + R * ldx;  // [2][DT_C][ldc]
    const uint32_t cs0 = smem_u32(Cs);
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3, lane = tid & 31, wid = tid >> 5;
    const int64_t nrows = row_list ? (int64_t)(*row_count) : n;
    const int ntile = (k + DT_C - 1) / DT_C, nck = (dp + DT_DK - 1) / DT_DK, nstep = ntile * nck;
    const float g = gamma32;
    __shared__ int open_rows[R], nopen;
    __shared__ float open_thr[R];
    float amx = 0.0f;
    unsigned long long local_amb = 0, ev64 = 0;
    if (tid == 0) nopen = 0;
    // the padding past d, at most 3 coordinates of a row: no load touches it
    if (dp != d)
        for (int e = tid; e < R * (dp - d); e += 256) Xs[(e / (dp - d)) * ldx + d + e % (dp - d)] = 0.0f;
    for (int64_t base = (int64_t)blockIdx.x * R; base < nrows; base += (int64_t)gridDim.x * R) {
        const int rows_here = (int)min((int64_t)R, nrows - base);
        __syncthreads();  // the previous round's readers are done with all buffers
        // few coordinates: the rows' floats one after another; else a warp per row, lanes
        // along it, coalesced without an index division (100,000 x 9, k = 10: 33 us
        // with nine of a warp's lanes, 27 so)
        if (d < 32 && !row_list) {
            const float* src = X + base * d;
            const int have = rows_here * d;
#pragma unroll 4
            for (int e = tid * VEC; e < R * d; e += 256 * VEC) {  // (VEC divides d)
                float v[VEC];
#pragma unroll
                for (int t = 0; t < VEC; t++) v[t] = 0.0f;
                if (e < have) {
                    if constexpr (VEC == 4) *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(src + e);
                    else if constexpr (VEC == 2) *reinterpret_cast<float2*>(v) = *reinterpret_cast<const float2*>(src + e);
                    else v[0] = src[e];
                }
                const int r = e / d;
#pragma unroll
                for (int t = 0; t < VEC; t++) {
                    amx = fmaxf(amx, fabsf(v[t]));
                    Xs[r * ldx + e - r * d + t] = v[t];
                }
            }
        } else
#pragma unroll 2
        for (int r = wid; r < R; r += 8) {
            const bool have = r < rows_here;
            const int64_t gi = !have ? 0 : (row_list ? (int64_t)row_list[base + r] : base + r);
            const float* src = X + gi * d;
#pragma unroll 4
            for (int l = lane * VEC; l < d; l += 32 * VEC) {
                float v[VEC];
#pragma unroll
                for (int t = 0; t < VEC; t++) v[t] = 0.0f;
                if (have) {
                    if constexpr (VEC == 4) *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(src + l);
                    else if constexpr (VEC == 2) *reinterpret_cast<float2*>(v) = *reinterpret_cast<const float2*>(src + l);
                    else v[0] = src[l];
                }
#pragma unroll
                for (int t = 0; t < VEC; t++) {
                    amx = fmaxf(amx, fabsf(v[t]));
                    Xs[r * ldx + l + t] = v[t];
                }
            }
        }
        // step s: coordinates [DT_DK (s % nck), ...) of the centres of tile s / nck
        auto load_step = [&](int s, int buf) {
            const int c0 = (s / nck) * DT_C, l0 = (s % nck) * DT_DK;
            const int w = min(DT_DK, d - l0);
            // LPC lanes per centre (a chunk is at most 64 coordinates)
            constexpr int LPC = 64 / VEC < 32 ? 64 / VEC : 32, CPW = 32 / LPC;
            const int cmax = min(DT_C, k - c0);  // (what lies past k stays from an earlier tile: its values are not used)
            for (int e = wid * CPW + lane / LPC; e < cmax * (64 / (LPC * VEC)); e += 8 * CPW) {
                const int c = e / (64 / (LPC * VEC)), l = (lane % LPC + LPC * (e % (64 / (LPC * VEC)))) * VEC;
                if (l >= w) continue;
                cp_async<4 * VEC>(cs0 + (uint32_t)(((buf * DT_C + c) * ldc + l) * 4), C + (int64_t)(c0 + c) * d + l0 + l);
            }
            if (w & 3)  // the last chunk's padding
                for (int c = tid; c < DT_C; c += 256)
                    for (int l = w; l < ((w + 3) & ~3); l++) Cs[(buf * DT_C + c) * ldc + l] = 0.0f;
            cp_async_commit();
        };
        load_step(0, 0);
        float b1[RPT], b2[RPT];
        int j1[RPT];
        float2 acc[RPT][8];
#pragma unroll
        for (int i = 0; i < RPT; i++) { b1[i] = INFINITY; b2[i] = INFINITY; j1[i] = 0; }
        int ck = 0, c0 = 0;
        for (int s = 0; s < nstep; s++) {
            const int buf = s & 1;
            cp_async_wait_all();
            __syncthreads();  // step s is in place; step s - 1's buffer is free
            if (s + 1 < nstep) load_step(s + 1, buf ^ 1);
            if (ck == 0) {
#pragma unroll
                for (int i = 0; i < RPT; i++)
#pragma unroll
                    for (int c = 0; c < 8; c++) acc[i][c] = make_float2(0.f, 0.f);
            }
            const float* xb = Xs + ty * ldx + ck * DT_DK;            // rows ty + 32 i
            const float* cb = Cs + (size_t)(buf * DT_C + tx) * ldc;  // centres tx + 8 c
            const int w = min(DT_DK, dp - ck * DT_DK), kleft = k - c0;
            auto chunk = [&](auto whole) {
#pragma unroll 1
                for (int l = 0; l < w; l += 4) {
                    float4 xv[RPT];
#pragma unroll
                    for (int i = 0; i < RPT; i++) xv[i] = *reinterpret_cast<const float4*>(xb + 32 * i * ldx + l);
#pragma unroll
                    for (int c = 0; c < 8; c++) {
                        if (!decltype(whole)::value && 8 * c >= kleft) break;  // (the last tile's missing centres)
                        const float4 cv = *reinterpret_cast<const float4*>(cb + 8 * c * ldc + l);
#pragma unroll
                        for (int i = 0; i < RPT; i++) {
                            const float2 t0 = fsub2(make_float2(xv[i].x, xv[i].y), make_float2(cv.x, cv.y));
                            acc[i][c] = __ffma2_rn(t0, t0, acc[i][c]);
                            const float2 t1 = fsub2(make_float2(xv[i].z, xv[i].w), make_float2(cv.z, cv.w));
                            acc[i][c] = __ffma2_rn(t1, t1, acc[i][c]);
                        }
                    }
                }
            };
            if (kleft > 56) chunk(std::true_type{});
            else chunk(std::false_type{});
            if (++ck < nck) continue;
            ck = 0;
#pragma unroll
            for (int c = 0; c < 8; c++) {
                const int j = c0 + tx + 8 * c;  // ascending in c: the first of equal values keeps its place
                if (j < k)
#pragma unroll
                    for (int i = 0; i < RPT; i++) {
                        const float v = acc[i][c].x + acc[i][c].y;
                        if (v < b1[i]) {
                            b2[i] = b1[i];
                            b1[i] = v;
                            j1[i] = j;
                        } else if (v < b2[i]) {
                            b2[i] = v;
                        }
                    }
            }
            c0 += DT_C;
        }
        // the 8 threads of each row: smallest (lowest index on ties) and second smallest
#pragma unroll
        for (int i = 0; i < RPT; i++)
#pragma unroll
            for (int off = 1; off < 8; off <<= 1) {
                const float ob1 = __shfl_xor_sync(0xffffffffu, b1[i], off);
                const float ob2 = __shfl_xor_sync(0xffffffffu, b2[i], off);
                const int oj = __shfl_xor_sync(0xffffffffu, j1[i], off);
                if (ob1 < b1[i] || (ob1 == b1[i] && oj < j1[i])) {
                    b2[i] = fminf(b1[i], ob2);
                    b1[i] = ob1;
                    j1[i] = oj;
                } else {
                    b2[i] = fminf(b2[i], ob1);
                }
            }
        if (tx == 0)
#pragma unroll
            for (int i = 0; i < RPT; i++) {
                const int r = ty + 32 * i;
                if (r < rows_here) {
                    const int64_t gi = row_list ? (int64_t)row_list[base + r] : base + r;
                    labels[gi] = j1[i];
                    min_dist[gi] = (double)b1[i];
                    const float thr = direct_upper(b1[i], g, direct_tiny(d));
                    if (!(direct_lower(b2[i], g) > thr)) {  // (Theorem 4.1)
                        const int o = atomicAdd(&nopen, 1);
                        open_rows[o] = (int)gi;
                        open_thr[o] = thr;
                        local_amb++;
                    }
                }
            }
        __syncthreads();
        if (const int no = nopen) {
            // (the centre buffers are free)
            resolve_open(X, C, k, d, open_rows, open_thr, no, g, labels, min_dist, Cs, (size_t)2 * DT_C * ldc * sizeof(float), &ev64);
            __syncthreads();
            if (tid == 0) {
                nopen = 0;
                atomicAdd(&cnt->fp32_evals, (unsigned long long)no * (unsigned long long)k);
            }
        }
        if (tid == 0) atomicAdd(&cnt->fp32_evals, (unsigned long long)rows_here * (unsigned long long)k);
    }
    cp_async_wait_all();
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) local_amb += __shfl_xor_sync(0xffffffffu, local_amb, off);
    if ((tid & 31) == 0 && local_amb) atomicAdd(&cnt->amb_rows, local_amb);
    if (ev64) atomicAdd(&cnt->fp64_evals, ev64);
    if (absmax_out) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) amx = fmaxf(amx, __shfl_xor_sync(0xffffffffu, amx, off));
        if ((tid & 31) == 0) atomicMax(absmax_out, __float_as_uint(amx));
    }
}

// 16 <= d <= 128, d % 4 == 0, 16-byte aligned rows
template <int RPT>
__global__ void __launch_bounds__(256, 2) k_direct_tiled(const float* __restrict__ X, int64_t n,
                                                         const float* __restrict__ C, int k, int d,
                                                         const int32_t* __restrict__ row_list,
                                                         const int* __restrict__ row_count,
                                                         int32_t* __restrict__ labels, double* __restrict__ min_dist,
                                                         DevCounters* cnt,
                                                         float gamma32, unsigned* __restrict__ absmax_out) {
    chain_enter();
    direct_tiled<RPT, 4>(X, n, C, k, d, row_list, row_count, labels, min_dist, cnt, gamma32, absmax_out);
}
// every other shape
template <typename T, int RPT, int VEC>
__global__ void __launch_bounds__(256, 2) k_direct_assign(const float* __restrict__ X, int64_t n,
                                                          const float* __restrict__ C, int k, int d,
                                                          const int32_t* __restrict__ row_list,
                                                          const int* __restrict__ row_count,
                                                          int32_t* __restrict__ labels, double* __restrict__ min_dist,
                                                          DevCounters* cnt,
                                                          float gamma32, unsigned* __restrict__ absmax_out) {
    chain_enter();
    static_assert(sizeof(T) == 4, "binary32 accumulation");
    direct_tiled<RPT, VEC>(X, n, C, k, d, row_list, row_count, labels, min_dist, cnt, gamma32, absmax_out);
}

template <int RPT, int VEC>
static cudaError_t launch_tiled(const float* X, int64_t n, const float* C, int k, int d, const int32_t* row_list,
                                const int* row_count, int32_t* labels, double* min_dist, DevCounters* cnt, float gamma32, int num_sms, cudaStream_t st, unsigned* absmax_out) {
    const size_t sm = dt_smem(RPT, d);
    void (*fn)(const float*, int64_t, const float*, int, int, const int32_t*, const int*, int32_t*, double*, DevCounters*, float, unsigned*) = k_direct_assign<float, RPT, VEC>;
    if constexpr (VEC == 4)
        if (d >= 16 && d <= 128) fn = k_direct_tiled<RPT>;
    cudaError_t e = allow_max_smem(fn);
    if (e != cudaSuccess) return e;
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((n + 32 * RPT - 1) / (32 * RPT), (int64_t)num_sms * 2));
    klaunch(fn, (unsigned)grid, 256, sm, st, X, n, C, k, d, row_list, row_count, labels, min_dist, cnt, gamma32,
                                        absmax_out);
    return cudaGetLastError();
}

// Small d (d <= 8) with C small enough to stay in shared memory for the whole
// launch.  Two passes over the centres, both in fp32 with a bound, decide a row
// when one centre alone can be the nearest:
//  * direct (d <= 2, and where the other decides too little): Eq. (dist-direct),
//    2 D operations a centre; every centre that can be the nearest has a value of
//    at most (1 + 3 g) times the smallest (Theorem 4.1, g = gamma_{D+2}(2^-24)).
//  * window: the expanded formula on centred data, x' = fl(x - mu), c' = fl(c -
//    mu), mu the mean of up to 32 centres,
//      e_j = q_j + sum_l x'_l (-2 c'_jl),  q_j = ||c'_j||^2   (D operations).
//    |e_j - (d_j - const)| <= gamma_D (q + 2 ||x'|| ||c'||) + gamma_D q + 2.1 u (||x'||
//    + ||c'||)^2, u = 2^-24 (the sums' rounding, q's, and that of the centring), so
//    every centre that can be the nearest lies within
//      W = (8 D + 20) u (||x'||^2 + max_j ||c'_j||^2)   (twice the bound, with slack)
//    of the smallest e.  W is absolute: it leaves most rows open when the centres
//    lie close together for their spread (k of them in 1-d: one row in seven at k =
//    256), or when one lies far away.
// A step whose rows the window leaves open in number is passed over directly, as
// are the next DS_SKIP steps of the warp; a few open rows take the warp each, lanes
// over the centres.  What the direct values leave open (near-ties) is decided in
// binary64.  min_dist is the winner's distance to binary64 accuracy (df.cuh), from
// the row in hand.
// A warp takes 64 rows per step, two per lane, the centres in pairs (packed
// arithmetic, each pair read once for both rows); the rows come through a ring in
// shared memory (16-byte asynchronous copies: D scalar loads per lane at a stride
// of D words cost D times the wavefronts) unless it would cost resident blocks.
// 16.8 M rows x 5, k = 16: 201 us with the winners' distances.  1e6 rows, uniform
// (in brackets: direct values of every centre for every row, without the distances,
// and a window for every row whose open rows one thread each took): d = 1, k = 1024
// 99 us (300, 733), d = 2, k = 1024 168 (364, 546), d = 3, k = 64 30 (50, 59), d = 8,
// k = 1024 414 (756, 1162), the same with one centre at 1e4 658 (756, 2900), d = 5, k
// = 16 on eight pairs of equal centres 116 (11,350, 692); 20,000 x 8, k = 1024 a
// latency of 55 (54, 136).
// Bound by dependent latencies at few centres or few rows, else by the FP32 pipe.
constexpr int DS_STAGES = 3;
constexpr int DS_SKIP = 8;  // steps without the window after one it was not worth
__host__ __device__ constexpr bool ds_window(int d) { return d > 2; }
// chunks of eight centres, coordinate by coordinate: the window's -2 c' and q, then c
__host__ __device__ constexpr size_t ds_window_floats(int d, int k) { return ds_window(d) ? (size_t)((k + 7) / 8 * 8) * (d + 1) : 0; }
__host__ __device__ constexpr size_t ds_centre_floats(int d, int k) { return ds_window_floats(d, k) + (size_t)((k + 7) / 8 * 8) * d; }
constexpr size_t ds_smem(int d, int k, int warps, bool staged) {
    return (ds_centre_floats(d, k) + (staged ? (size_t)warps * DS_STAGES * 64 * d : 0)) * sizeof(float);
}

// The values of a chunk's eight centres for NR rows, two per packed operation.
template <int D, bool DIRECT, int NR>
KM_DEV void ds_chunk(const float4* cp, const float2 (&u)[2][D], float2 (&e)[2][4], int r0 = 0) {
    if constexpr (!DIRECT) {
        const float4 qa = cp[2 * D], qb = cp[2 * D + 1];
#pragma unroll
        for (int r = 0; r < NR; r++) {
            e[r][0] = make_float2(qa.x, qa.y);
            e[r][1] = make_float2(qa.z, qa.w);
            e[r][2] = make_float2(qb.x, qb.y);
            e[r][3] = make_float2(qb.z, qb.w);
        }
    }
#pragma unroll
    for (int l = 0; l < D; l++) {
        const float4 ca = cp[2 * l], cb = cp[2 * l + 1];
        const float2 c[4] = {make_float2(ca.x, ca.y), make_float2(ca.z, ca.w), make_float2(cb.x, cb.y), make_float2(cb.z, cb.w)};
#pragma unroll
        for (int i = 0; i < 4; i++)
#pragma unroll
            for (int r = 0; r < NR; r++) {
                const float2 x = u[NR == 1 ? r0 : r][l];
                if constexpr (DIRECT) {
                    const float2 t = fsub2(x, c[i]);
                    e[r][i] = l == 0 ? __fmul2_rn(t, t) : __ffma2_rn(t, t, e[r][i]);
                } else {
                    e[r][i] = __ffma2_rn(x, c[i], e[r][i]);
                }
            }
    }
}
KM_DEV float ds_least(const float2 (&e)[4]) {
    return fmin3f(fmin3f(e[0].x, e[0].y, e[1].x), fmin3f(e[1].y, e[2].x, e[2].y), fminf(e[3].x, e[3].y));
}
// The signs of a chunk's values less thr as a mask (equality counts as outside:
// there is slack; so does what is not comparable).
KM_DEV unsigned ds_below(const float2 (&e)[4], float thr) {
    unsigned m = 0;
#pragma unroll
    for (int i = 3; i >= 0; i--) {
        const float2 t = fsub2(e[i], make_float2(thr, thr));
        m = __funnelshift_l(__float_as_uint(t.x), __funnelshift_l(__float_as_uint(t.y), m, 1), 1);
    }
    return m;
}

// A lane's two rows u (row 0, row 1) against all centres: for each row the only
// centre that can be the nearest, -1 when there are several; b1: their smallest
// values.  DIRECT: squared distances to the chunks at cs, those up to rel times the smallest (and W) count;
// else e, those within W of it.
// Few centres (ds_few): the chunks that hold a row's smallest value so far, or one
// near it, are looked at at once.  MANY: most chunks would be for one of the warp's
// 64 rows; the smallest value, its chunk and the smallest of the other chunks are
// kept, and that one chunk is formed again at the end (1e6 rows: d = 1, k = 64 24 ->
// 18 us, k = 1024 168 -> 100; d = 3, k = 1024 242 -> 195, but k = 64 31 -> 37; d = 7,
// k = 100 60 -> 84).
__host__ __device__ constexpr int ds_few(int d) { return d <= 2 ? 32 : 128; }
template <int D, bool DIRECT, bool MANY>
KM_DEV void ds_scan(const float* cs, int kp, const float2 (&u)[D], float2 W, float rel, int& ja, int& jb, float2& b1) {
    constexpr int L = DIRECT ? D : D + 1;
    float2 uu[2][D], e[2][4];
#pragma unroll
    for (int l = 0; l < D; l++) {
        uu[0][l] = make_float2(u[l].x, u[l].x);
        uu[1][l] = make_float2(u[l].y, u[l].y);
    }
    const float2 r2 = make_float2(rel, rel);
    auto upper = [&](float2 v) { return DIRECT ? __ffma2_rn(v, r2, W) : __fadd2_rn(v, W); };
    auto only = [](unsigned m) { return m != 0u && (m & (m - 1)) == 0u; };
    b1 = make_float2(INFINITY, INFINITY);
    ja = jb = -1;
    if constexpr (!MANY) {
        for (int j0 = 0; j0 < kp; j0 += 8) {
            const float4* cp = reinterpret_cast<const float4*>(cs + (size_t)j0 * L);
            ds_chunk<D, DIRECT, 2>(cp, uu, e);
            const float2 cm = make_float2(ds_least(e[0]), ds_least(e[1]));
            const float2 bw = upper(b1);
            const bool in0 = cm.x <= bw.x, in1 = cm.y <= bw.y;  // (false where nothing is comparable)
            if (!__any_sync(0xffffffffu, in0 || in1)) continue;
            const float2 cw = upper(cm);
            const unsigned m0 = ds_below(e[0], fminf(bw.x, cw.x)), m1 = ds_below(e[1], fminf(bw.y, cw.y));
            // strictly below what was found before and alone: the candidate; else several
            // lie in the window (a row with none here keeps what it had)
            if (in0) ja = cw.x < b1.x && only(m0) ? j0 + 31 - __clz(m0) : -1;
            if (in1) jb = cw.y < b1.y && only(m1) ? j0 + 31 - __clz(m1) : -1;
            b1 = make_float2(fminf(b1.x, cm.x), fminf(b1.y, cm.y));
        }
    } else {
        float2 b2 = b1;
        int c0 = 0, c1 = 0;
#pragma unroll(D <= 2 ? 2 : 1)
        for (int j0 = 0; j0 < kp; j0 += 8) {
            ds_chunk<D, DIRECT, 2>(reinterpret_cast<const float4*>(cs + (size_t)j0 * L), uu, e);
            const float2 cm = make_float2(ds_least(e[0]), ds_least(e[1]));
            // (nothing comparable in the chunk: the row stays open)
            b2 = make_float2(fminf(b2.x, fmaxf(b1.x, cm.x)), fminf(b2.y, fmaxf(b1.y, cm.y)));
            c0 = cm.x < b1.x ? j0 : c0;
            c1 = cm.y < b1.y ? j0 : c1;
            b1 = make_float2(fminf(b1.x, cm.x), fminf(b1.y, cm.y));
        }
        const float2 thr = upper(b1);
        ds_chunk<D, DIRECT, 1>(reinterpret_cast<const float4*>(cs + (size_t)c0 * L), uu, e, 0);
        const unsigned m0 = ds_below(e[0], thr.x);
        ds_chunk<D, DIRECT, 1>(reinterpret_cast<const float4*>(cs + (size_t)c1 * L), uu, e, 1);
        const unsigned m1 = ds_below(e[0], thr.y);
        if (!(b2.x < thr.x) && only(m0)) ja = c0 + 31 - __clz(m0);
        if (!(b2.y < thr.y) && only(m1)) jb = c1 + 31 - __clz(m1);
    }
}

// A row that the direct values leave open, by one thread: binary64 for every centre
// whose interval reaches down to thr.  live: the lanes that call.
template <int D>
__device__ __noinline__ int small_open_row(unsigned live, const float* __restrict__ X, int64_t i, const float* __restrict__ C,
                                           int k, float g, float thr, unsigned* ev64) {
    float x[D];
#pragma unroll
    for (int l = 0; l < D; l++) x[l] = X[i * D + l];
    auto value = [&](int j) {
        float acc = 0.0f;
#pragma unroll
        for (int l = 0; l < D; l++) {
            const float t = x[l] - C[j * D + l];
            acc = fmaf(t, t, acc);
        }
        return acc;
    };
    int j1 = 0;  // (no value to compare, NaN: a valid label all the same)
    // the candidates are listed first, all lanes at the same centre, then the lanes
    // evaluate theirs together (each when it comes to it, where almost every centre is
    // some lane's, 1e6 rows x 5 on eight pairs of equal centres took 750 us, 116 so)
    constexpr int LIST = 8;
    int cj[LIST], cnt = 0;
    double best = INFINITY;
    auto evaluate = [&]() {
        for (int t = 0; __any_sync(live, t < cnt); t++) {
            if (t >= cnt) continue;
            const int j = cj[t];
            const double s = direct64(x, C + j * D, D);
            ++*ev64;
            if (s < best) {
                best = s;
                j1 = j;
            }
        }
        cnt = 0;
    };
    for (int j = 0; j < k; j++) {
        if (direct_lower(value(j), g) <= thr) cj[cnt++] = j;
        if (__any_sync(live, cnt == LIST)) evaluate();
    }
    evaluate();
    return j1;
}

// The same by a warp, lanes over the centres.
template <int D>
__device__ __noinline__ int warp_open_row(const float* __restrict__ X, int64_t i, const float* __restrict__ C, int k, float g,
                                          unsigned* amb, unsigned* ev64) {
    const int lane = threadIdx.x & 31;
    float x[D];
#pragma unroll
    for (int l = 0; l < D; l++) x[l] = X[i * D + l];
    auto value = [&](int j) {
        float acc = 0.0f;
#pragma unroll
        for (int l = 0; l < D; l++) {
            const float t = x[l] - C[j * D + l];
            acc = fmaf(t, t, acc);
        }
        return acc;
    };
    Top2 t{INFINITY, INFINITY, 0x7fffffff};
    for (int j = lane; j < k; j += 32) t = top2_merge(t, Top2{value(j), INFINITY, j});
#pragma unroll
    for (int off = 16; off > 0; off >>= 1)
        t = top2_merge(t, Top2{__shfl_xor_sync(0xffffffffu, t.b1, off), __shfl_xor_sync(0xffffffffu, t.b2, off),
                               __shfl_xor_sync(0xffffffffu, t.j1, off)});
    const float thr = direct_upper(t.b1, g, direct_tiny(D));
    if (direct_lower(t.b2, g) > thr) return t.j1;
    *amb += lane == 0 ? 1u : 0u;
    double best = INFINITY;
    int arg = 0x7fffffff;
    for (int j = lane; j < k; j += 32) {
        if (!(direct_lower(value(j), g) <= thr)) continue;
        const double s = direct64(x, C + j * D, D);
        ++*ev64;
        if (s < best) { best = s; arg = j; }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const double ob = __shfl_xor_sync(0xffffffffu, best, off);
        const int oa = __shfl_xor_sync(0xffffffffu, arg, off);
        if (ob < best || (ob == best && oa < arg)) { best = ob; arg = oa; }
    }
    return arg < k ? arg : 0;  // (no value to compare, NaN: a valid label all the same)
}

template <int D, bool STAGED, bool MANY>
__global__ void __launch_bounds__(256, 3) k_direct_small(const float* __restrict__ X, int64_t n,
                                                      const float* __restrict__ C, int k,
                                                      const int32_t* __restrict__ row_list,
                                                      const int* __restrict__ row_count,
                                                      int32_t* __restrict__ labels, double* __restrict__ min_dist,
                                                      DevCounters* cnt, float gamma32,
                                                      unsigned* __restrict__ absmax_out) {
    chain_enter();
    extern __shared__ __align__(16) float dsm[];
    __shared__ float mu[8];
    __shared__ unsigned qmax_bits;
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nwb = blockDim.x >> 5;
    const int64_t nrows = row_list ? (int64_t)(*row_count) : n;
    if (nrows == 0) return;
    const int kp = (k + 7) / 8 * 8;
    float* const cdir = dsm + ds_window_floats(D, k);
    if (threadIdx.x == 0) qmax_bits = 0u;
    if (ds_window(D)) centre_mean(C, k, D, D, mu);
    for (int j = threadIdx.x; j < kp; j += blockDim.x) {
        float q = j < k ? 0.0f : INFINITY;  // (padding never wins)
        float* const cw = dsm + (size_t)(j & ~7) * (D + 1) + (j & 7);
#pragma unroll
        for (int l = 0; l < D; l++) {
            const float c0 = j < k ? C[j * D + l] : INFINITY;
            cdir[(size_t)(j & ~7) * D + 8 * l + (j & 7)] = c0;
            if (ds_window(D)) {
                const float c = j < k ? c0 - mu[l] : 0.0f;
                if (j < k) q = fmaf(c, c, q);
                cw[8 * l] = -2.0f * c;
            }
        }
        if (ds_window(D)) {
            cw[8 * D] = q;
            if (j < k) atomicMax(&qmax_bits, q >= 0.0f ? __float_as_uint(q) : 0x7f800000u);
        }
    }
    __syncthreads();
    const float qmax = __uint_as_float(qmax_bits);
    const float wscale = (float)(8 * D + 20) * 0x1p-24f * 1.02f;
    float m[D];
#pragma unroll
    for (int l = 0; l < D; l++) m[l] = ds_window(D) ? mu[l] : 0.0f;
    // the direct pass: (1 + g) / (1 - g) < 1 + 3 g with the rounding of the product
    const float rel = 1.0f + 3.0f * gamma32, wdir = 2.0f * direct_tiny(D);
    // open rows that cost less by the warp (instructions, about) than the direct pass
    const int few = (int)((unsigned)k * (2 * D + 6) / ((unsigned)(k >> 5) * (3 * D + 6) + 100u));
    int skip = 0;  // steps to take without the window
    constexpr int STEP = 64;
    float* ring = dsm + ds_centre_floats(D, k) + (size_t)wib * DS_STAGES * STEP * D;
    const uint32_t ring_s = smem_u32(ring);
    const int64_t w0 = (int64_t)blockIdx.x * nwb + wib, nw = (int64_t)gridDim.x * nwb;
    const int64_t nstep = (nrows + STEP - 1) / STEP;
    auto fetch = [&](int64_t st, int slot) {
        if (STAGED && st < nstep) {
            const char* src = reinterpret_cast<const char*>(X + st * STEP * D) + 16 * lane;
            const uint32_t dst = ring_s + (uint32_t)(slot * STEP * D * 4 + 16 * lane);
            const int left = (int)min((int64_t)STEP * D * 4, (nrows - st * STEP) * D * 4) - 16 * lane;  // bytes from src on
#pragma unroll
            for (int c = 0; c < (16 * D + 31) / 32; c++) {  // 16-byte pieces
                const int rest = left - 512 * c;
                if (rest > 0)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(dst + 512 * c), "l"(src + 512 * c),
                                 "r"(min(rest, 16))
                                 : "memory");
            }
        }
        cp_async_commit();
    };
    float amx = 0.0f;  // largest |x| of this thread's rows (absmax_out)
    unsigned rows_done = 0, local_amb = 0, ev64 = 0;
#pragma unroll
    for (int t = 0; t < DS_STAGES - 1; t++) fetch(w0 + t * nw, t);
    int slot = 0;
    for (int64_t st = w0; st < nstep; st += nw) {
        // (the slot fetched into was read in the step before: the warp is past it)
        __syncwarp();
        fetch(st + (DS_STAGES - 1) * nw, slot == 0 ? DS_STAGES - 1 : slot - 1);
        asm volatile("cp.async.wait_group %0;" ::"n"(DS_STAGES - 1) : "memory");
        __syncwarp();
        const int64_t r0 = st * STEP + lane;
        const bool valid0 = r0 < nrows, valid1 = r0 + 32 < nrows;
        const int64_t g0 = STAGED || !row_list ? r0 : (valid0 ? row_list[r0] : 0);
        const int64_t g1 = STAGED || !row_list ? r0 + 32 : (valid1 ? row_list[r0 + 32] : 0);
        float2 x[D];  // (row 0, row 1)
        const float* xs0 = ring + (slot * STEP + lane) * D;
#pragma unroll
        for (int l = 0; l < D; l++) {
            if (STAGED) {  // (rows past the end: whatever an earlier step left; nothing of them is kept)
                x[l] = make_float2(xs0[l], xs0[32 * D + l]);
                if (!valid1) x[l] = make_float2(valid0 ? x[l].x : 0.0f, 0.0f);
            } else {
                x[l] = make_float2(valid0 ? X[g0 * D + l] : 0.0f, valid1 ? X[g1 * D + l] : 0.0f);
            }
            amx = fmaxabs3(amx, x[l].x, x[l].y);
        }
        slot = slot + 1 == DS_STAGES ? 0 : slot + 1;
        int ja = -1, jb = -1;
        float2 b1;
        bool direct = !ds_window(D) || skip > 0;
        if constexpr (ds_window(D)) {
            if (!direct) {
                float2 y[D], p = make_float2(0.f, 0.f);
#pragma unroll
                for (int l = 0; l < D; l++) {
                    y[l] = fsub2(x[l], make_float2(m[l], m[l]));
                    p = __ffma2_rn(y[l], y[l], p);
                }
                const float2 W = __ffma2_rn(make_float2(wscale, wscale), __fadd2_rn(p, make_float2(qmax, qmax)),
                                            make_float2(0x1p-120f, 0x1p-120f));
                ds_scan<D, false, MANY>(dsm, kp, y, W, 0.0f, ja, jb, b1);
                const unsigned o0 = __ballot_sync(0xffffffffu, valid0 && ja < 0), o1 = __ballot_sync(0xffffffffu, valid1 && jb < 0);
                if (__popc(o0) + __popc(o1) > few) {
                    direct = true;
                    skip = DS_SKIP + 1;
                }
            }
        }
        if (direct) {
            ds_scan<D, true, MANY>(cdir, kp, x, make_float2(wdir, wdir), rel, ja, jb, b1);
            skip -= skip > 0 ? 1 : 0;
        }
        unsigned o0 = __ballot_sync(0xffffffffu, valid0 && ja < 0), o1 = __ballot_sync(0xffffffffu, valid1 && jb < 0);
        if (__popc(o0) + __popc(o1) > few) {
            // (only after the direct pass)
            if ((o0 >> lane) & 1u) ja = small_open_row<D>(o0, X, g0, C, k, gamma32, direct_upper(b1.x, gamma32, direct_tiny(D)), &ev64);
            if ((o1 >> lane) & 1u) jb = small_open_row<D>(o1, X, g1, C, k, gamma32, direct_upper(b1.y, gamma32, direct_tiny(D)), &ev64);
            local_amb += ((o0 >> lane) & 1u) + ((o1 >> lane) & 1u);
        } else {
            for (; o0 | o1; o0 ? o0 &= o0 - 1 : o1 &= o1 - 1) {
                const int b = __ffs(o0 ? o0 : o1) - 1;
                const int j = warp_open_row<D>(X, __shfl_sync(0xffffffffu, o0 ? g0 : g1, b), C, k, gamma32, &local_amb, &ev64);
                if (lane == b) (o0 ? ja : jb) = j;
            }
        }
        const float *ca = C + (int64_t)max(ja, 0) * D, *cb = C + (int64_t)max(jb, 0) * D;
        float2 c2[D];
#pragma unroll
        for (int l = 0; l < D; l++) c2[l] = make_float2(ca[l], cb[l]);
        const DF2 r = df2_small<D>(x, c2);
        if (valid0) {
            labels[g0] = ja;
            min_dist[g0] = df_value64(r.hi.x, r.lo.x);
        }
        if (valid1) {
            labels[g1] = jb;
            min_dist[g1] = df_value64(r.hi.y, r.lo.y);
        }
        rows_done += (valid0 ? 1 : 0) + (valid1 ? 1 : 0);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    rows_done = __reduce_add_sync(0xffffffffu, rows_done);
    local_amb = __reduce_add_sync(0xffffffffu, local_amb);
    ev64 = __reduce_add_sync(0xffffffffu, ev64);
    if (absmax_out) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) amx = fmaxf(amx, __shfl_xor_sync(0xffffffffu, amx, off));
    }
    if (lane == 0) {
        if (rows_done) atomicAdd(&cnt->fp32_evals, (unsigned long long)rows_done * (unsigned long long)k);
        if (local_amb) atomicAdd(&cnt->amb_rows, (unsigned long long)local_amb);
        if (ev64) atomicAdd(&cnt->fp64_evals, (unsigned long long)ev64);
        if (absmax_out) atomicMax(absmax_out, __float_as_uint(amx));
    }
}

// The small-d kernel where the centres' tables fit in shared memory (128 KB still
// beat the tiles with one block per SM: 1e6 x 4, k = 3600 733 us against 4495, 1e6 x
// 1, k = 10,000 912 against 16,520: tiles of 64 centres of so few coordinates wait
// for each other), but for few rows of seven or eight coordinates, where a warp's
// walk over all centres takes longer than the tiles (5000 x 8, k = 1032: 51 us
// against 34; 20,000 rows: 56 against 68).
bool direct_gives_winners(int64_t n, int d, int k) {
    if (d > 8 || ds_centre_floats(d, k) * sizeof(float) > (size_t)(ds_window(d) ? 128 : 200) * 1024) return false;
    return !(d >= 7 && k * d > 8192 && n <= 9728);
}

cudaError_t launch_direct_assign(bool acc64, const float* X, int64_t n, const float* C, int k, int d,
                                 const int32_t* row_list, const int* row_count, int32_t* labels,
                                 double* min_dist, DevCounters* cnt, float gamma32,
                                 int num_sms, cudaStream_t st, unsigned* absmax_out) {
    if (!acc64 && direct_gives_winners(n, d, k)) {
        // small d: C resident in shared memory, persistent grid; few rows in small
        // blocks, so that they spread over the SMs (but not too small for the table of
        // many centres that each block makes: 60,000 x 8, k = 1024: 114 us in blocks of
        // 64 threads, 71 of 128; 8192 x 1, k = 8192: 187 and 175)
        const int threads = n > (int64_t)num_sms * 512 ? 256 : (k * d <= 1024 ? 64 : 128);
        typedef void (*SmallFn)(const float*, int64_t, const float*, int, const int32_t*, const int*, int32_t*, double*,
                                DevCounters*, float, unsigned*);
        SmallFn ring = nullptr, plain = nullptr;
        switch (d) {
#define KM_SMALL(DD) \
    case DD:                                                                                  \
        ring = k > ds_few(DD) ? k_direct_small<DD, true, true> : k_direct_small<DD, true, false>;  \
        plain = k > ds_few(DD) ? k_direct_small<DD, false, true> : k_direct_small<DD, false, false>; \
        break;
            KM_SMALL(1) KM_SMALL(2) KM_SMALL(3) KM_SMALL(4) KM_SMALL(5) KM_SMALL(6) KM_SMALL(7) KM_SMALL(8)
#undef KM_SMALL
        }
        SmallFn fn = plain;
        size_t sm = ds_smem(d, k, threads / 32, false);
        cudaError_t e = allow_max_smem(fn);
        int per_sm = 1;
        if (e == cudaSuccess) e = blocks_per_sm(fn, threads, sm, &per_sm);
        if (e == cudaSuccess && !row_list && ((uintptr_t)X & 15) == 0) {
            const size_t sr = ds_smem(d, k, threads / 32, true);
            int pr = 1;
            e = allow_max_smem(ring);
            if (e == cudaSuccess) e = blocks_per_sm(ring, threads, sr, &pr);
            if (pr >= per_sm && sr <= (size_t)kMaxBlockSmem - 1024) {
                fn = ring;
                sm = sr;
                per_sm = pr;
            }
        }
        if (e != cudaSuccess) return e;
        const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((n + 2 * threads - 1) / (2 * threads), (int64_t)num_sms * per_sm));
        return klaunch(fn, (unsigned)grid, (unsigned)threads, sm, st, X, n, C, k, row_list, row_count, labels, min_dist, cnt,
                       gamma32, absmax_out);
    }
    if (!acc64) {
        // rows per block: 128, or 64 where 128 would leave one block per SM
        // (111 KB of dynamic shared memory, past d = 148) or too few blocks for two per
        // SM, or 32 where 64 would; a row list is taken for as long as the call's rows
        // (7265 x 128 x 436, most rows listed: 119 us with 128 rows per block, 66 with
        // 32; 37,638 x 128 x 44: 40 and 30 with 64)
        const bool a16 = ((uintptr_t)X % 16) == 0 && ((uintptr_t)C % 16) == 0;
        const bool a8 = ((uintptr_t)X % 8) == 0 && ((uintptr_t)C % 8) == 0;
        const int vec = d % 4 == 0 && a16 ? 4 : (d % 2 == 0 && a8 ? 2 : 1);
        int rpt = dt_smem(4, d) <= 111 * 1024 ? 4 : 2;
        while (rpt > 1 && (n + 32 * rpt - 1) / (32 * rpt) < 2 * num_sms) rpt >>= 1;
#define KM_DT(RP, VE)                                                                                              \
    if (rpt == RP && vec == VE)                                                                                    \
        return launch_tiled<RP, VE>(X, n, C, k, d, row_list, row_count, labels, min_dist, cnt, gamma32, \
                                    num_sms, st, absmax_out);
        KM_DT(4, 4) KM_DT(4, 2) KM_DT(4, 1) KM_DT(2, 4) KM_DT(2, 2) KM_DT(2, 1) KM_DT(1, 4) KM_DT(1, 2) KM_DT(1, 1)
#undef KM_DT
    }
    const size_t sm = ((((size_t)DA_ROWS * (d + 1) * sizeof(float)) + 15) & ~(size_t)15) + (size_t)DA_TC * d * 8;
    const int per_sm = std::min(8, (int)std::max<size_t>(1, (size_t)(200 * 1024) / sm));
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((n + DA_ROWS - 1) / DA_ROWS, (int64_t)num_sms * per_sm));
    void (*fn64)(const float*, int64_t, const float*, int, int, int32_t*, double*, unsigned*) = k_direct_assign<double>;
    cudaError_t e = allow_max_smem(fn64);
    if (e != cudaSuccess) return e;
    klaunch(fn64, (unsigned)grid, DA_ROWS, sm, st, X, n, C, k, d, labels, min_dist, absmax_out);
    return cudaGetLastError();
}

// Listed rows, a block each.
__global__ void __launch_bounds__(256) k_rows_full(const float* __restrict__ X, const float* __restrict__ C, int k,
                                                   int d, const int32_t* __restrict__ row_list,
                                                   const int* __restrict__ row_count, int32_t* __restrict__ labels,
                                                   double* __restrict__ min_dist, DevCounters* cnt, float gamma32,
                                                   size_t bytes) {
    chain_enter();
    extern __shared__ __align__(16) double shd[];
    const int64_t nrows = *row_count;
    unsigned long long ev32 = 0, ev64 = 0, open = 0;
    for (int64_t w = blockIdx.x; w < nrows; w += gridDim.x) {
        open += resolve_row(X, C, k, d, row_list[w], gamma32, labels, min_dist, shd, bytes, &ev64) ? 1 : 0;
        ev32 += (unsigned long long)k;
    }
    if (threadIdx.x == 0 && ev32) {
        atomicAdd(&cnt->fp32_evals, ev32);
        if (open) atomicAdd(&cnt->amb_rows, open);
    }
    if (ev64) atomicAdd(&cnt->fp64_evals, ev64);
}

cudaError_t launch_rows_full(const float* X, const float* C, int k, int d, const int32_t* row_list,
                             const int* row_count, int32_t* labels, double* min_dist, DevCounters* cnt,
                             float gamma32, int num_sms, cudaStream_t st) {
    cudaFuncAttributes fa;
    cudaError_t e = cudaFuncGetAttributes(&fa, (const void*)k_rows_full);
    if (e != cudaSuccess) return e;
    const size_t all = resolve_bytes(d) + (size_t)k * sizeof(float);
    const size_t bytes = all <= (size_t)kMaxBlockSmem - fa.sharedSizeBytes ? all : resolve_bytes(d);
    e = allow_max_smem(k_rows_full);
    if (e != cudaSuccess) return e;
    klaunch(k_rows_full, num_sms * 2, 256, bytes, st, X, C, k, d, row_list, row_count, labels, min_dist, cnt, gamma32, bytes);
    return cudaGetLastError();
}

}  // namespace km
