// Double-precision chunk sums for rows whose fp32 statistics were too close to a decision
// threshold.  Four warps per (listed row, chunk): sum of exp(l/T - max/T) over the chunk, exactly
// the terms of the definition.  The whole grid shares the work, so a handful of flagged rows
// costs microseconds; with an empty queue every CTA returns at once.
#pragma once
#include "common.cuh"

namespace picospec {

struct PreciseArgs {
    const void* logits;
    long long row_stride;
    int V, nch;
    int seq_rows;              // rows per sequence in the logits tensor (G or G+1)
    const float* temperature;  // [B]
    const int* rows;           // the rows whose exact chunk sums are wanted (indices into the logits tensor)
    const int* row_count;      // how many
    const float* row_max;      // [rows] exact row maxima from the fp32 pass
    double* dsum;              // [rows, pitch]
    int pitch = 0;             // chunk sums per row in dsum (0: nch)
};

// exp(x) for x <= 0 (-inf included) in double precision, to about one unit in the last place: x = (64 m + j) ln 2 / 64 + r
// with |r| <= ln 2 / 128, exp(x) = 2^m 2^(j/64) (1 + p(r)), p the Taylor polynomial of exp(r) - 1 of degree 5 (its
// remainder is below 2^-54).  The powers 2^(j/64) lie in shared memory.  ln 2 / 64 is taken off in two parts, the
// first of 34 bits, so that its product with 64 m + j is exact.  Below -700 the result is 0.
// 12 double-precision operations a term: 256 rows of the edge, 40 of them exact, 80.4 -> 76.4 us a pass against exp().
constexpr int EXP_STEPS = 64;
__device__ __forceinline__ void exp_table(double* table) {      // by the CTA's first threads (a barrier follows)
    if (threadIdx.x < EXP_STEPS) table[threadIdx.x] = exp2((double)(int)threadIdx.x / EXP_STEPS);
}
__device__ __forceinline__ double exp_by_table(double x, const double* table) {
    const double round = 6755399441055744.0;                    // 1.5 * 2^52: its last bits take the rounded product
    const double t = fma(x, 0x1.71547652b82fep+6, round);       // 64 / ln 2
    const int n = __double2loint(t);
    const double nd = t - round;
    const double r = fma(nd, -0x1.1cf79abc9e3b4p-42, fma(nd, -0x1.62e42fef80000p-7, x));
    const double q = fma(r, fma(r, fma(r, 1.0 / 120.0, 1.0 / 24.0), 1.0 / 6.0), 0.5);
    const double p = fma(r * r, q, r);
    const double w = table[n & (EXP_STEPS - 1)];
    const double y = fma(w, p, w);
    const double scaled = __hiloint2double(__double2hiint(y) + ((n >> 6) << 20), __double2loint(y));
    return (unsigned)__double2hiint(x) > 0xC085E000u ? 0.0 : scaled;        // x < -700
}

// A quarter of one item of the double-precision pass, held by a warp.  Item = (listed row, chunk).
constexpr int PRECISE_HELD = CHUNK / 4 / 32;
template <typename T> struct PreciseQuarter {
    int slot, row, c;           // the row's place in the list (-1: no such item), the row, the chunk
    float Tb, mx;
    float l[PRECISE_HELD];
    __device__ __forceinline__ void load(const PreciseArgs& a, long long item, long long total, int quarter, int lane) {
        slot = -1;
        if (item >= total) return;
        slot = (int)(item / a.nch);
        c = (int)(item - (long long)slot * a.nch);
        row = a.rows[slot] & 0x1FFFFFFF;    // (a list may keep flags above the index)
        Tb = a.temperature[row / a.seq_rows];
        mx = a.row_max[row];
        const T* p = reinterpret_cast<const T*>(a.logits) + (long long)row * a.row_stride;
        const int v0 = c * CHUNK + quarter * (CHUNK / 4) + lane;
#pragma unroll
        for (int x = 0; x < PRECISE_HELD; ++x) l[x] = v0 + x * 32 < a.V ? load_logit(p, v0 + x * 32) : -CUDART_INF_F;
    }
    // The sum of exp(l/T - mx/T).  x = l * (1/T) instead of l / T: one rounding of 2^-53 more per term, far below
    // every threshold this pass decides; four independent sums keep the exp pipeline busy.
    __device__ __forceinline__ double sum(const double* table) {
        const double rT = 1.0 / (double)Tb, m = (double)mx * rT;
        double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
#pragma unroll 1
        for (int x = 0; x < PRECISE_HELD; x += 4) {
            s0 += exp_by_table((double)l[0] * rT - m, table);
            s1 += exp_by_table((double)l[1] * rT - m, table);
            s2 += exp_by_table((double)l[2] * rT - m, table);
            s3 += exp_by_table((double)l[3] * rT - m, table);
#pragma unroll
            for (int y = 0; y + 4 < PRECISE_HELD; ++y) l[y] = l[y + 4];
        }
        return warp_sum((s0 + s1) + (s2 + s3));
    }
};
// where the sum of an item goes
template <typename T> __device__ __forceinline__ void precise_store(const PreciseArgs& a, const PreciseQuarter<T>& q, double sum) {
    a.dsum[(long long)q.row * (a.pitch > 0 ? a.pitch : a.nch) + q.c] = sum;
}

// A CTA takes two chunks at a time, four warps per chunk (a quarter of the chunk each, so that a handful of rows
// still spreads over the whole GPU); the four partial sums of a chunk are added in a fixed order.  Where a CTA
// takes several, the next one's logits are on the way while the exponentials of the one at hand are taken, so that
// three CTAs per SM do what took six (40 rows of 128256 entries: 17 us either way, 12 since the exponential goes by table,
// of which its operations are 3.3 at the nominal rate).  Few rows are bound by the launch: see precise_grid.
constexpr int PRECISE_CTAS = 3;     // per SM
template <typename T>
__global__ void __launch_bounds__(THREADS, PRECISE_CTAS) precise_chunk_sums_kernel(PreciseArgs a) {
    __shared__ double part[2][WARPS], table[EXP_STEPS];
    exp_table(table);
    grid_dependency_sync();
    const int nq = *a.row_count;
    if (nq == 0) return;
    __syncthreads();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sub = warp >> 2, quarter = warp & 3;
    const long long total = (long long)nq * a.nch;
    PreciseQuarter<T> next;
    next.load(a, 2ll * blockIdx.x + sub, total, quarter, lane);
    int copy = 0;
    for (long long pair = blockIdx.x; 2 * pair < total; pair += gridDim.x, copy ^= 1) {
        PreciseQuarter<T> q = next;
        next.load(a, 2 * (pair + gridDim.x) + sub, total, quarter, lane);
        const double s = q.slot >= 0 ? q.sum(table) : 0.0;
        if (lane == 0) part[copy][warp] = s;
        __syncthreads();        // (one barrier an item: the copies take turns)
        if (q.slot >= 0 && quarter == 0 && lane == 0)
            precise_store(a, q, (part[copy][warp] + part[copy][warp + 1]) + (part[copy][warp + 2] + part[copy][warp + 3]));
    }
}

}  // namespace picospec
