// k_direct.cu -- direct-formula assignment kernels, Eq. (dist-direct).
//
//  * k_direct_assign<double>: the plain FP64 path (every pair in binary64).
//  * k_direct_tiled, its general form k_direct_assign<float> and (d <= 8, few
//    centres) k_direct_small: fp32 direct distances for the fp32 path and for rows whose tensor-core candidate list
//    overflowed.  Theorem 4.1 bounds each value's relative error by
//    gamma_{d+2}(2^-24); a row whose best and second-best intervals overlap is
//    not certified and goes to
//  * k_rows_full: the exact argmin of one row over all centres (a block per
//    row), lowest index on ties; binary64 values with products and sums rounded
//    separately (no FMA), equal to the CPU oracle's bit for bit.
#include <algorithm>

#include "common.cuh"
#include "df.cuh"
#include "internal.h"

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
    if (t.b2 * (1.0f - gamma32) > t.b1 * (1.0f + gamma32)) {
        if (tid == 0) {
            labels[i] = t.j1;
            min_dist[i] = (double)t.b1;
        }
        return false;
    }
    // squares below binary32's range: each coordinate adds at most 2^-149 of absolute error
    const float thr = t.b1 * (1.0f + gamma32) + (float)(2 * d + 4) * 0x1p-149f;
    double best = INFINITY;
    int arg = 0x7fffffff;
    if (keep_vals) {
        for (int j = tid; j < k; j += 256)
            if (vs[j] * (1.0f - gamma32) <= thr) {
                const int p = atomicAdd(&nopen, 1);
                if (p < RF_OPEN) open_j[p] = j;
            }
    } else {
        for (int j = 4 * wid; j < k; j += 32) {  // the same values as above
            float v[4];
            warp_direct4(xs, C, k, d, j, lane, v);
#pragma unroll
            for (int q = 0; q < 4; q++)
                if (lane == 0 && j + q < k && v[q] * (1.0f - gamma32) <= thr) {
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
            if (keep_vals && !(vs[j] * (1.0f - gamma32) <= thr)) continue;
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
KM_DEV void cp_async(uint32_t dst, const void* src, bool full) {
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(full ? 16 : 0) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(BYTES), "r"(full ? BYTES : 0)
                     : "memory");
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
    const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
    const int64_t nrows = row_list ? (int64_t)(*row_count) : n;
    const int ntile = (k + DT_C - 1) / DT_C, nck = (dp + DT_DK - 1) / DT_DK, nstep = ntile * nck;
    const float g = gamma32;
    const int dv = d / VEC;  // loads per row
    __shared__ int open_rows[R], nopen;
    float amx = 0.0f;
    unsigned long long local_amb = 0, ev64 = 0;
    if (tid == 0) nopen = 0;
    // the padding past d, at most 3 coordinates of a row: no load touches it
    if (dp != d)
        for (int e = tid; e < R * (dp - d); e += 256) Xs[(e / (dp - d)) * ldx + d + e % (dp - d)] = 0.0f;
    for (int64_t base = (int64_t)blockIdx.x * R; base < nrows; base += (int64_t)gridDim.x * R) {
        const int rows_here = (int)min((int64_t)R, nrows - base);
        __syncthreads();  // the previous round's readers are done with all buffers
        for (int e = tid; e < R * dv; e += 256) {
            const int r = e / dv, l = (e - r * dv) * VEC;
            float v[VEC];
#pragma unroll
            for (int t = 0; t < VEC; t++) v[t] = 0.0f;
            if (r < rows_here) {
                const int64_t gi = row_list ? (int64_t)row_list[base + r] : base + r;
                const float* src = X + gi * d + l;
                if constexpr (VEC == 4) *reinterpret_cast<float4*>(v) = *reinterpret_cast<const float4*>(src);
                else if constexpr (VEC == 2) *reinterpret_cast<float2*>(v) = *reinterpret_cast<const float2*>(src);
                else v[0] = *src;
#pragma unroll
                for (int t = 0; t < VEC; t++) amx = fmaxf(amx, fabsf(v[t]));
            }
#pragma unroll
            for (int t = 0; t < VEC; t++) Xs[r * ldx + l + t] = v[t];
        }
        // step s: coordinates [DT_DK (s % nck), ...) of the centres of tile s / nck
        auto load_step = [&](int s, int buf) {
            const int c0 = (s / nck) * DT_C, l0 = (s % nck) * DT_DK;
            const int w = min(DT_DK, d - l0), wv = w / VEC;
            for (int e = tid; e < DT_C * wv; e += 256) {
                const int c = e / wv, l = (e - c * wv) * VEC;
                const bool ok = c0 + c < k;
                cp_async<4 * VEC>(cs0 + (uint32_t)(((buf * DT_C + c) * ldc + l) * 4),
                                  ok ? (const void*)(C + (int64_t)(c0 + c) * d + l0 + l) : (const void*)C, ok);
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
            const int w = min(DT_DK, dp - ck * DT_DK);
#pragma unroll 1
            for (int l = 0; l < w; l += 4) {
                float4 xv[RPT];
#pragma unroll
                for (int i = 0; i < RPT; i++) xv[i] = *reinterpret_cast<const float4*>(xb + 32 * i * ldx + l);
#pragma unroll
                for (int c = 0; c < 8; c++) {
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
                    // Theorem 4.1: true values lie in [v (1 - g), v (1 + g)]
                    if (!(b2[i] * (1.0f - g) > b1[i] * (1.0f + g))) {
                        open_rows[atomicAdd(&nopen, 1)] = (int)gi;
                        local_amb++;
                    }
                }
            }
        __syncthreads();
        if (const int no = nopen) {
            // (the centre buffers are free: 512 ldc bytes, resolve_bytes(d) at most 68 d of them)
            for (int o = 0; o < no; o++)
                resolve_row(X, C, k, d, open_rows[o], g, labels, min_dist, Cs, (size_t)2 * DT_C * ldc * sizeof(float), &ev64);
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

// Small d (d <= 8) with C small enough to stay in shared memory for the
// whole launch: one thread per row, the row in registers, every centre from
// shared memory (all lanes read the same centre: a broadcast).  The same
// fp32 operations, in the same order, and the same certificate as the tiled
// kernel above, so the two give the same results.
template <int D>
__global__ void __launch_bounds__(256) k_direct_small(const float* __restrict__ X, int64_t n,
                                                      const float* __restrict__ C, int k,
                                                      const int32_t* __restrict__ row_list,
                                                      const int* __restrict__ row_count,
                                                      int32_t* __restrict__ labels, double* __restrict__ min_dist,
                                                      DevCounters* cnt,
                                                      float gamma32, unsigned* __restrict__ absmax_out) {
    chain_enter();
    extern __shared__ __align__(16) float Csm[];
    float amx = 0.0f;  // largest |x| of this thread's rows (absmax_out)
    for (int e = threadIdx.x; e < k * D; e += blockDim.x) Csm[e] = C[e];
    __syncthreads();
    const int64_t nrows = row_list ? (int64_t)(*row_count) : n;
    const float g = gamma32;
    unsigned long long rows_done = 0, local_amb = 0, ev64 = 0;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nrows; r += (int64_t)gridDim.x * blockDim.x) {
        const int64_t gi = row_list ? (int64_t)row_list[r] : r;
        float x[D];
#pragma unroll
        for (int l = 0; l < D; l++) {
            x[l] = X[gi * D + l];
            amx = fmaxf(amx, fabsf(x[l]));
        }
        float b1 = INFINITY, b2 = INFINITY;
        int j1 = 0;
        for (int j = 0; j < k; j++) {
            float acc = 0.0f;
#pragma unroll
            for (int l = 0; l < D; l++) {
                const float t = x[l] - Csm[j * D + l];
                acc = fmaf(t, t, acc);
            }
            if (acc < b1) {
                b2 = b1;
                b1 = acc;
                j1 = j;
            } else if (acc < b2) {
                b2 = acc;
            }
        }
        labels[gi] = j1;
        min_dist[gi] = (double)b1;
        rows_done++;
        // Theorem 4.1: true values lie in [v (1 - g), v (1 + g)]; a row left open
        // takes binary64 values of the centres that can hold its minimum
        if (!(b2 * (1.0f - g) > b1 * (1.0f + g))) {
            local_amb++;
            // (squares below binary32's range: at most 2^-149 per coordinate)
            const float thr = b1 * (1.0f + g) + (float)(2 * D + 4) * 0x1p-149f;
            double best = INFINITY;
            for (int j = 0; j < k; j++) {
                float acc = 0.0f;
#pragma unroll
                for (int l = 0; l < D; l++) {
                    const float t = x[l] - Csm[j * D + l];
                    acc = fmaf(t, t, acc);
                }
                if (!(acc * (1.0f - g) <= thr)) continue;
                const double s = direct64(x, Csm + j * D, D);
                ev64++;
                if (s < best) {
                    best = s;
                    j1 = j;
                }
            }
            labels[gi] = j1;
            min_dist[gi] = best;
        }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        rows_done += __shfl_xor_sync(0xffffffffu, rows_done, off);
        local_amb += __shfl_xor_sync(0xffffffffu, local_amb, off);
        ev64 += __shfl_xor_sync(0xffffffffu, ev64, off);
    }
    if (absmax_out) {
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) amx = fmaxf(amx, __shfl_xor_sync(0xffffffffu, amx, off));
    }
    if ((threadIdx.x & 31) == 0) {
        if (rows_done) atomicAdd(&cnt->fp32_evals, rows_done * (unsigned long long)k);
        if (local_amb) atomicAdd(&cnt->amb_rows, local_amb);
        if (ev64) atomicAdd(&cnt->fp64_evals, ev64);
        if (absmax_out) atomicMax(absmax_out, __float_as_uint(amx));
    }
}

cudaError_t launch_direct_assign(bool acc64, const float* X, int64_t n, const float* C, int k, int d,
                                 const int32_t* row_list, const int* row_count, int32_t* labels,
                                 double* min_dist, DevCounters* cnt, float gamma32,
                                 int num_sms, cudaStream_t st, unsigned* absmax_out) {
    if (!acc64 && d <= 8 && (size_t)k * d * sizeof(float) <= 32 * 1024) {
        // small d: C resident in shared memory, one thread per row, persistent grid
        const size_t csm = (size_t)k * d * sizeof(float);
        int per_sm = 1;
        const void* fns[9] = {nullptr, (const void*)k_direct_small<1>, (const void*)k_direct_small<2>,
                              (const void*)k_direct_small<3>, (const void*)k_direct_small<4>,
                              (const void*)k_direct_small<5>, (const void*)k_direct_small<6>,
                              (const void*)k_direct_small<7>, (const void*)k_direct_small<8>};
        cudaError_t e = blocks_per_sm_of(fns[d], 256, csm, &per_sm);
        if (e != cudaSuccess) return e;
        const int64_t grid = std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)num_sms * std::max(per_sm, 1)));
        switch (d) {
#define KM_SMALL(DD)                                                                                                  \
    case DD:                                                                                                          \
        klaunch(k_direct_small<DD>, (unsigned)grid, 256, csm, st, X, n, C, k, row_list, row_count, labels, min_dist,      \
                                                              cnt, gamma32, absmax_out);                                \
        break;
            KM_SMALL(1) KM_SMALL(2) KM_SMALL(3) KM_SMALL(4) KM_SMALL(5) KM_SMALL(6) KM_SMALL(7) KM_SMALL(8)
#undef KM_SMALL
        }
        return cudaGetLastError();
    }
    if (!acc64) {
        // rows per block: 128, or 64 where 128 would leave one block per SM
        // (111 KB of dynamic shared memory, past d = 148) or too few blocks for two per
        // SM, or 32 where 64 would; a row list's length is not known here
        const bool a16 = ((uintptr_t)X % 16) == 0 && ((uintptr_t)C % 16) == 0;
        const bool a8 = ((uintptr_t)X % 8) == 0 && ((uintptr_t)C % 8) == 0;
        const int vec = d % 4 == 0 && a16 ? 4 : (d % 2 == 0 && a8 ? 2 : 1);
        int rpt = dt_smem(4, d) <= 111 * 1024 ? 4 : 2;
        while (rpt > 1 && !row_list && (n + 32 * rpt - 1) / (32 * rpt) < 2 * num_sms) rpt >>= 1;
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
