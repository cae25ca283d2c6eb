// k_seed.cu -- initial centres by D^2 sampling (k-means++): Section 2 names
// it beside uniformly drawn initial centres and leaves it outside the
// method.  The draws u_t in [0, 1) are inputs.
//   i_0 = min(floor(u_0 n), n - 1);
//   D^2_i = d(x_i, x_{i_0})^2 by the direct formula (Eq. (dist-direct)) to
//   binary64 accuracy (the double-float arithmetic of df.cuh);
//   for t = 1..k-1: T = sum_i D^2_i; i_t = the first row whose prefix sum
//   exceeds u_t T (the last row with D^2 > 0 when rounding leaves none;
//   min(floor(u_t n), n - 1) when T = 0), then D^2_i = min(D^2_i, d(x_i, x_{i_t})^2).
// One launch per pick.  Rows form chunks (a warp each) and eight chunks a group
// (a block): the pass over X updates D^2 and sums it by chunk and group in the
// registers that hold it, and the block that finishes last finds the group,
// the chunk and the row that hold the target.  Every sum is binary64 in an
// order fixed by n and d alone, so the result does not depend on the launch.
// A row whose fp32 distance already shows (Theorem 4.1) that the new centre is
// no closer keeps its D^2: the double-float distance is formed only for rows
// that may change, fewer with every pick.
// Bound by reads of X (L2 or HBM) and, at small n, by the pick's chain of
// dependent steps.  1e5 x 128: 53 us a pick in three launches, 22 us in one (the
// FP64 pipe's 16 cycles per warp instruction were half of that: additions are
// shared between lanes, comparisons done on the bits).
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "df.cuh"
#include "internal.h"
#include "seed.h"

namespace km {

constexpr int SD_WARPS = 8;             // chunks per group
constexpr int64_t SD_MAX_CHUNKS = 14336;  // with their groups they fit 16384 entries

// Chunks of one pass over X.
struct SeedPlan {
    int64_t rows;    // per chunk, a multiple of unit
    int64_t nc, ng;  // chunks, groups
};
static SeedPlan seed_plan(int64_t n, int d) {
    const int64_t unit = d <= 8 ? 32 : 16;  // a multiple of the rows of one warp pass
    SeedPlan p;
    p.rows = unit * std::max<int64_t>(1, (n + unit * SD_MAX_CHUNKS - 1) / (unit * SD_MAX_CHUNKS));
    p.nc = (n + p.rows - 1) / p.rows;
    p.ng = (p.nc + SD_WARPS - 1) / SD_WARPS;
    return p;
}
size_t seed_scratch_count(int64_t n, int d) {
    const SeedPlan p = seed_plan(n, d);
    return (size_t)(p.nc + p.ng + 1);
}

KM_DEV int64_t uniform_pick(double u, int64_t n) {
    const int64_t i = (int64_t)floor(u * (double)n);
    return i > n - 1 ? n - 1 : i;
}

// df_rows for one float per row.
template <int R, int L>
KM_DEV float f_rows(float (&v)[R], int cl) {
#pragma unroll
    for (int lev = 0; (L >> (lev + 1)) >= 1; lev++) {
        const int o = L >> (lev + 1);
        const int nr = (R >> lev) > 1 ? (R >> lev) : 1;
        if (nr > 1) {
            const int h = nr >> 1;
            const bool up = (cl & o) != 0;
#pragma unroll
            for (int r = 0; r < h; r++) {
                const float keep = up ? v[r + h] : v[r], send = up ? v[r] : v[r + h];
                v[r] = keep + __shfl_xor_sync(0xffffffffu, send, o);
            }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
        }
    }
    return v[0];
}

// The FP64 pipe takes 16 cycles per warp instruction for the whole SM: what is
// no addition is done on the bits (non-negative doubles order like integers).
KM_DEV double dmin_bits(double a, double b) {
    const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
    return __longlong_as_double(x < y ? x : y);
}
KM_DEV bool dpos(double a) { return __double_as_longlong(a) > 0; }
// A float at or above the non-negative double a (2^-100 at least, unless a is 0:
// there the fp32 distance's absolute roundings, 2^-150 each, are below its own).
KM_DEV float dround_up(double a) {
    const unsigned hi = (unsigned)__double2hiint(a), lo = (unsigned)__double2loint(a);
    const unsigned e = hi >> 20;
    if (e < 923u) return e == 0u && lo == 0u && hi == 0u ? 0.0f : 0x1p-100f;  // (below 2^-100)
    if (e > 1150u) return INFINITY;                                          // (2^128 or more, not a number)
    return __uint_as_float(((hi - (896u << 20)) << 3 | lo >> 29) + 1u);
}
// Whether a row's fp32 distance v (relative error at most g) may lie below old.
KM_DEV bool may_improve(float v, float g, double old) { return !(v * (1.0f - g) > dround_up(old)); }

// D^2 of rows [lo, hi) against c, min with the old values unless first; the
// lane's share of their sum (s) and its last row with D^2 > 0 (less lo).  The
// LPR / R lanes that hold the same row take turns at the passes' values, so one
// addition serves that many passes.
template <int NV4, int LPR, bool VEC>
KM_DEV void seed_rows(const float* __restrict__ X, int d, const float* __restrict__ c, const float4 (&cv)[NV4],
                      int64_t lo, int64_t hi, bool first, float g, double* D2, int lane, double& s, int& last) {
    constexpr int G = 32 / LPR;
    constexpr int R = NV4 == 4 ? 2 : 4;  // rows per lane and pass
    constexpr int STEP = R * G;
    static_assert(R <= LPR && 16 % STEP == 0, "a chunk is a whole number of passes");
    const int sub = lane / LPR, cl = lane % LPR;
    const int d4 = (d + 3) >> 2;
    int rs = 0;  // the row of a pass that this lane's reductions end in (f_rows, df_rows)
#pragma unroll
    for (int lev = 0; (R >> lev) > 1; lev++) rs += (cl & (LPR >> (lev + 1))) ? R >> (lev + 1) : 0;
    const bool owner = (cl & (LPR / R - 1)) == 0;
    auto load = [&](int64_t base, float4 (&xv)[R][NV4], double& old) {
#pragma unroll
        for (int b = 0; b < R; b++) {
            const int64_t row = base + b * G + sub;
#pragma unroll
            for (int u = 0; u < NV4; u++) {
                const int cidx = cl + LPR * u;
                // rows past the chunk repeat the centre: distance zero, dropped below
                const bool ok = row < hi && cidx < d4;
                if (VEC) {
                    xv[b][u] = ok ? reinterpret_cast<const float4*>(X + row * d)[cidx] : cv[u];
                } else {
                    const float* xr = X + row * d + 4 * cidx;
                    xv[b][u].x = ok && 4 * cidx + 0 < d ? xr[0] : cv[u].x;
                    xv[b][u].y = ok && 4 * cidx + 1 < d ? xr[1] : cv[u].y;
                    xv[b][u].z = ok && 4 * cidx + 2 < d ? xr[2] : cv[u].z;
                    xv[b][u].w = ok && 4 * cidx + 3 < d ? xr[3] : cv[u].w;
                }
            }
        }
        const int64_t row = base + rs * G + sub;
        old = !first && owner && row < hi ? D2[row] : 0.0;
    };
    // the next pass's rows are loaded while this one's are reduced
    float4 xn[R][NV4];
    double oldn = 0.0, turn = 0.0;
    constexpr int TURNS = LPR / R;
    int pass = 0;
    if (lo < hi) load(lo, xn, oldn);
    for (int64_t base = lo; base < hi; base += STEP) {
        float4 xv[R][NV4];
        const double old = oldn;
#pragma unroll
        for (int b = 0; b < R; b++)
#pragma unroll
            for (int u = 0; u < NV4; u++) xv[b][u] = xn[b][u];
        if (base + STEP < hi) load(base + STEP, xn, oldn);
        const int64_t row = base + rs * G + sub;
        const bool mine = owner && row < hi;
        double v = old;
        bool need = first;
        if (!first) {
            float part[R];
#pragma unroll
            for (int b = 0; b < R; b++) {
                part[b] = 0.0f;
#pragma unroll
                for (int u = 0; u < NV4; u++) {
                    const float t0 = xv[b][u].x - cv[u].x, t1 = xv[b][u].y - cv[u].y;
                    const float t2 = xv[b][u].z - cv[u].z, t3 = xv[b][u].w - cv[u].w;
                    part[b] = fmaf(t0, t0, part[b]);
                    part[b] = fmaf(t1, t1, part[b]);
                    part[b] = fmaf(t2, t2, part[b]);
                    part[b] = fmaf(t3, t3, part[b]);
                }
            }
            need = may_improve(f_rows<R, LPR>(part, cl), g, old);
        }
        if (__any_sync(0xffffffffu, mine && need)) {
            DF pd[R];
#pragma unroll
            for (int b = 0; b < R; b++) pd[b] = df_lane<NV4>(xv[b], cv);
            int rd;
            const DF r = df_rows<R, LPR>(pd, cl, rd);
            if (mine) {
                v = first ? df_value(r) : dmin_bits(old, df_value(r));
                D2[row] = v;
            }
        }
        if (mine && dpos(v)) last = (int)(row - lo);
        const double w = __shfl_sync(0xffffffffu, mine ? v : 0.0, lane & ~(TURNS - 1));
        if ((lane & (TURNS - 1)) == pass) turn = w;
        if (++pass == TURNS || base + STEP >= hi) {
            s += turn;
            turn = 0.0;
            pass = 0;
        }
    }
}

// D <= 8 coordinates: a lane per row.
template <int D>
KM_DEV void seed_rows_small(const float* __restrict__ X, const float* __restrict__ c, int64_t lo, int64_t hi, bool first,
                            double* D2, int lane, double& s, int& last) {
    for (int64_t i = lo + lane; i < hi; i += 32) {
        float xr[D];
#pragma unroll
        for (int l = 0; l < D; l++) xr[l] = X[i * D + l];
        double v = df_value(df_small<D>(xr, c));
        if (!first) v = dmin_bits(D2[i], v);
        D2[i] = v;
        s += v;
        if (dpos(v)) last = (int)(i - lo);
    }
}

// Inclusive prefix sums over the warp.
KM_DEV double warp_scan(double v, int lane) {
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const double o = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += o;
    }
    return v;
}

// The pick of step t.  The groups' sums go through shared memory; then one
// warp (the fewest FP64 instructions): lane p adds its groups [p GPL, (p + 1)
// GPL) in order and the lanes' totals give prefix sums and T.  The first lane,
// of its groups the first, of that group's chunks and of that chunk's rows the
// first whose prefix sum exceeds u_t T; when rounding leaves none, the last
// with D^2 > 0.
KM_DEV void seed_pick(const double* D2, int64_t n, const SeedPlan& pl, const double* csum, const int64_t* clast,
                      const double* gsum, double ut, int64_t* idx_t) {
    __shared__ double gs[SD_MAX_CHUNKS / SD_WARPS];
    const int tid = threadIdx.x, lane = tid & 31;
    const int ng = (int)pl.ng, gpl = (ng + 31) / 32;
#pragma unroll 7
    for (int j = tid; j < ng; j += 256) gs[j] = __ldcg(gsum + j);
    __syncthreads();
    if (tid >= 32) return;
    double A = 0.0;
#pragma unroll 4
    for (int j = lane * gpl; j < min(ng, (lane + 1) * gpl); j++) A += gs[j];
    const double incl = warp_scan(A, lane);
    const double T = __shfl_sync(0xffffffffu, incl, 31);
    int64_t pick = uniform_pick(ut, n);
    if (T > 0.0) {
        const double target = ut * T;
        // item of the warp's (value w, prefix sums in): the first live one whose
        // start + in exceeds the target, else the last live one; its start
        auto first_past = [&](double in, bool live, double& start) -> int {
            const unsigned lm = __ballot_sync(0xffffffffu, live);
            const unsigned past = __ballot_sync(0xffffffffu, live && target < start + in);
            if (!lm) return -1;
            const int hit = past ? __ffs(past) - 1 : 31 - __clz(lm);
            const double before = __shfl_sync(0xffffffffu, in, hit > 0 ? hit - 1 : 0);
            if (hit > 0) start += before;
            return hit;
        };
        double start = 0.0;
        const int p = first_past(incl, dpos(A), start);
        // the lane's groups, 32 at a time (GPL is at most 56)
        int grp = -1;
        double gstart = start;
        const int g0 = p * gpl, g1 = min(ng, g0 + gpl);
        for (int j = g0; j < g1; j += 32) {
            const double v = j + lane < g1 ? gs[j + lane] : 0.0, in = warp_scan(v, lane);
            double st = start;
            const int hit = first_past(in, dpos(v), st);
            const double tot = __shfl_sync(0xffffffffu, in, 31);
            if (hit >= 0) {
                grp = j + hit;
                gstart = st;
            }
            start += tot;
            if (target < start) break;
        }
        if (grp >= 0) {
            const int64_t c0 = (int64_t)grp * SD_WARPS, c = c0 + lane;
            const bool have = lane < SD_WARPS && c < pl.nc;
            const double cs = have ? __ldcg(csum + c) : 0.0;
            const long long cl = have ? __ldcg(reinterpret_cast<const long long*>(clast) + c) : -1;
            const double in = warp_scan(cs, lane);
            double acc = gstart;
            const int hit = first_past(in, cl >= 0, acc);
            if (hit >= 0) {
                pick = __shfl_sync(0xffffffffu, cl, hit);  // (the chunk's last row with D^2 > 0)
                const int64_t lo = (c0 + hit) * pl.rows, hi = lo + pl.rows < n ? lo + pl.rows : n;
                for (int64_t b = lo; b < hi; b += 32) {
                    const double v = b + lane < hi ? __ldcg(D2 + b + lane) : 0.0, sc = warp_scan(v, lane);
                    const unsigned over = __ballot_sync(0xffffffffu, dpos(v) && target < acc + sc);
                    if (over) {
                        pick = b + __ffs(over) - 1;
                        break;
                    }
                    acc += __shfl_sync(0xffffffffu, sc, 31);
                }
            }
        }
    }
    if (lane == 0) *idx_t = pick;
}

// Step t: D^2 against the pick of step t (step 0: the uniform one), then the
// pick of step t + 1.  SMALL: D = NV4 coordinates, a lane per row.
template <int NV4, int LPR, bool VEC, bool SMALL>
__global__ void __launch_bounds__(256, NV4 == 1 || SMALL ? 3 : 2) k_seed_step(const float* __restrict__ X, int64_t n, int d, const SeedPlan pl,
                                                   const double* __restrict__ u, int t, float g, double* D2, double* csum,
                                                   int64_t* clast, int64_t* idx, unsigned* ticket) {
    chain_enter();
    __shared__ double part_sh[SD_WARPS * 32];
    __shared__ int last_sh[SD_WARPS];
    __shared__ bool last_block;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const float* c = X + (t == 0 ? uniform_pick(u[0], n) : idx[t]) * d;
    float4 cv[SMALL ? 1 : NV4];
    if constexpr (!SMALL) {
        const int cl = lane % LPR;
#pragma unroll
        for (int q = 0; q < NV4; q++) {
            const int cidx = cl + LPR * q;
            if (VEC) {
                cv[q] = 4 * cidx < d ? reinterpret_cast<const float4*>(c)[cidx] : make_float4(0.f, 0.f, 0.f, 0.f);
            } else {
                float ce[4];
#pragma unroll
                for (int l = 0; l < 4; l++) ce[l] = (4 * cidx + l < d) ? c[4 * cidx + l] : 0.0f;
                cv[q] = make_float4(ce[0], ce[1], ce[2], ce[3]);
            }
        }
    }
    double* gsum = csum + pl.nc;
    for (int64_t grp = blockIdx.x; grp < pl.ng; grp += gridDim.x) {
        const int64_t chunk = grp * SD_WARPS + wid;
        const int64_t lo = chunk * pl.rows < n ? chunk * pl.rows : n, hi = lo + pl.rows < n ? lo + pl.rows : n;
        double s = 0.0;
        int last = -1;
        if constexpr (SMALL) seed_rows_small<NV4>(X, c, lo, hi, t == 0, D2, lane, s, last);
        else seed_rows<NV4, LPR, VEC>(X, d, c, cv, lo, hi, t == 0, g, D2, lane, s, last);
        last = __reduce_max_sync(0xffffffffu, last);
        __syncthreads();  // the previous group's sums have been read
        part_sh[threadIdx.x] = s;
        if (lane == 0) last_sh[wid] = last;
        __syncthreads();
        // the eight chunks' sums by one warp, four lanes each: eight lanes' shares
        // in order, then a tree; then the group's
        if (wid == 0) {
            const int q = lane >> 2;
            double a = 0.0;
#pragma unroll
            for (int l = 0; l < 8; l++) a += part_sh[q * 32 + (lane & 3) * 8 + l];
            a += __shfl_xor_sync(0xffffffffu, a, 1);
            a += __shfl_xor_sync(0xffffffffu, a, 2);
            if ((lane & 3) == 0 && grp * SD_WARPS + q < pl.nc) {
                csum[grp * SD_WARPS + q] = a;
                clast[grp * SD_WARPS + q] = last_sh[q] < 0 ? -1 : (grp * SD_WARPS + q) * pl.rows + last_sh[q];
            }
#pragma unroll
            for (int off = 4; off < 32; off <<= 1) a += __shfl_xor_sync(0xffffffffu, a, off);
            if (lane == 0) gsum[grp] = a;
        }
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last_block = atomicInc(ticket, gridDim.x - 1) == gridDim.x - 1;  // 0 again for the next step
    __syncthreads();
    if (!last_block) return;
    __threadfence();
    seed_pick(D2, n, pl, csum, clast, gsum, u[t + 1], idx + t + 1);
}

// The picked rows (and the first pick's index).
__global__ void k_seed_gather(const float* __restrict__ X, int64_t n, int d, const double* __restrict__ u, int64_t* idx,
                              int k, float* __restrict__ C) {
    chain_enter();
    const int64_t first = uniform_pick(u[0], n);
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < (int64_t)k * d;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t t = e / d;
        C[e] = X[(t == 0 ? first : idx[t]) * d + (e - t * d)];
        if (e == 0) idx[0] = first;
    }
}

cudaError_t launch_seed_pp(const float* X, int64_t n, int d, int k, const double* u_dev, double* D2, int64_t* idx,
                           double* csum, int64_t* clast, float* C_out, int num_sms, cudaStream_t st, int* nlaunch) {
    *nlaunch = 0;
    const SeedPlan pl = seed_plan(n, d);
    unsigned* ticket = reinterpret_cast<unsigned*>(clast + pl.nc + pl.ng);
    cudaError_t e = cudaMemsetAsync(ticket, 0, sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    const bool vec = d % 4 == 0 && ((uintptr_t)X % 16) == 0;
    const int lpr = df_lpr(d), nv4 = df_nv4(d);
    void (*kern)(const float*, int64_t, int, SeedPlan, const double*, int, float, double*, double*, int64_t*, int64_t*,
                 unsigned*) = nullptr;
    if (d <= 8) {
        switch (d) {
#define KM_SS(DD) \
    case DD: kern = k_seed_step<DD, 8, false, true>; break;
            KM_SS(1) KM_SS(2) KM_SS(3) KM_SS(4) KM_SS(5) KM_SS(6) KM_SS(7) KM_SS(8)
#undef KM_SS
        }
    } else {
#define KM_SD(NV, L)                                                        \
    if (nv4 == NV && lpr == L) {                                            \
        if (vec) kern = k_seed_step<NV, L, true, false>;                    \
        else kern = k_seed_step<NV, L, false, false>;                       \
    }
        KM_SD(1, 8) KM_SD(1, 16) KM_SD(1, 32) KM_SD(2, 32) KM_SD(4, 32)
#undef KM_SD
    }
    if (!kern) return cudaErrorInvalidValue;
    int per_sm = 1;
    e = blocks_per_sm(kern, 256, 0, &per_sm);
    if (e != cudaSuccess) return e;
    const unsigned blocks = (unsigned)std::min<int64_t>(pl.ng, (int64_t)num_sms * std::max(per_sm, 1));
    // Theorem 4.1's gamma_{d+2}(2^-24) with safety, and the double-float distance's own 2^-40
    const float g = (float)((d + 4) * std::ldexp(1.0, -24) * 1.01 + std::ldexp(1.0, -22));
    for (int t = 0; t + 1 < k; t++) {
        klaunch(kern, blocks, 256, 0, st, X, n, d, pl, u_dev, t, g, D2, csum, clast, idx, ticket);
        (*nlaunch)++;
    }
    const unsigned gb = (unsigned)std::max<int64_t>(1, std::min<int64_t>(((int64_t)k * d + 255) / 256, 4096));
    klaunch(k_seed_gather, gb, 256, 0, st, X, n, d, u_dev, idx, k, C_out);
    (*nlaunch)++;
    return cudaGetLastError();
}

}  // namespace km
