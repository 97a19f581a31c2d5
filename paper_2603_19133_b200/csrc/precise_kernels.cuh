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
    __device__ __forceinline__ double sum() {
        const double rT = 1.0 / (double)Tb, m = (double)mx * rT;
        double s0 = 0.0, s1 = 0.0, s2 = 0.0, s3 = 0.0;
#pragma unroll 1
        for (int x = 0; x < PRECISE_HELD; x += 4) {
            s0 += exp((double)l[0] * rT - m);
            s1 += exp((double)l[1] * rT - m);
            s2 += exp((double)l[2] * rT - m);
            s3 += exp((double)l[3] * rT - m);
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
// three CTAs per SM do what took six (40 rows of 128256 entries: 17 us either way, bound by the chain of one
// item).  Few rows are bound by the launch: see precise_grid.
constexpr int PRECISE_CTAS = 3;     // per SM
template <typename T>
__global__ void __launch_bounds__(THREADS, PRECISE_CTAS) precise_chunk_sums_kernel(PreciseArgs a) {
    grid_dependency_sync();
    const int nq = *a.row_count;
    if (nq == 0) return;
    __shared__ double part[2][WARPS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int sub = warp >> 2, quarter = warp & 3;
    const long long total = (long long)nq * a.nch;
    PreciseQuarter<T> next;
    next.load(a, 2ll * blockIdx.x + sub, total, quarter, lane);
    int copy = 0;
    for (long long pair = blockIdx.x; 2 * pair < total; pair += gridDim.x, copy ^= 1) {
        PreciseQuarter<T> q = next;
        next.load(a, 2 * (pair + gridDim.x) + sub, total, quarter, lane);
        const double s = q.slot >= 0 ? q.sum() : 0.0;
        if (lane == 0) part[copy][warp] = s;
        __syncthreads();        // (one barrier an item: the copies take turns)
        if (q.slot >= 0 && quarter == 0 && lane == 0)
            precise_store(a, q, (part[copy][warp] + part[copy][warp + 1]) + (part[copy][warp + 2] + part[copy][warp + 3]));
    }
}

}  // namespace picospec
