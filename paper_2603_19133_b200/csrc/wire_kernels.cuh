// Wire format of the sparse rows (Sec. 3.3: the verifier sends pairs of vocabulary id and
// probability -- under 100 bytes for K = 10 -- laid out so that the receiver can view the arrays in place).  One message:
//     0   u32  magic 0x31505350 ("PSP1")
//     4   u32  R, the number of rows
//     8   u16  K, the capacity of a dense row
//     10  u16  probability type: 0 = fp32, 1 = fp16 (round to nearest even)
//     12  u32  N = sum over rows of max(count, 0)
//     16  i16  count[R]   (-1 = invalid row), zero-padded to a multiple of 4 bytes
//     ..  i32  id[N]      rows in order, entries in stored order
//     ..  prob[N]         fp32 or fp16; the message is zero-padded to a multiple of 4 bytes
// Packing and unpacking are one kernel each: every CTA takes a block of consecutive rows, adds up all
// the counts for itself (they come from L2: 6 KB for 1536 rows) and moves its rows' entries.  Bound by
// latency and by the launch; with a scan by one CTA and the move as kernels of their own, and one warp
// per row, packing and unpacking took 25 us together for 27 rows of 925 entries.
#pragma once
#include <cuda_fp16.h>

#include "common.cuh"

namespace picospec {

constexpr unsigned WIRE_MAGIC = 0x31505350u;

struct WireArgs {
    int* q_idx;                 // [R, K]   (read by pack, written by unpack)
    float* q_prob;              // [R, K]
    int* q_count;               // [R]
    int R, K, prob_type;
    unsigned char* buf;         // the message
    long long capacity;         // bytes available at buf (pack) / bytes of the message (unpack)
    long long* bytes_out;       // pack: size of the message, or -1 if it does not fit
    unsigned* status;
};

__host__ __device__ __forceinline__ long long wire_pad4(long long n) { return (n + 3) / 4 * 4; }
__host__ __device__ __forceinline__ long long wire_bytes(long long rows, long long entries, int prob_type) {
    return 16 + wire_pad4(2 * rows) + 4 * entries + wire_pad4((prob_type == 0 ? 4 : 2) * entries);
}

// Threads that move one row: about four entries each, a warp at least, the CTA at most.
__host__ __device__ __forceinline__ int wire_row_threads(int K) {
    int t = 32;
    while (t < THREADS && 4 * t < K) t <<= 1;
    return t;
}

// CTA b: rows [b * per_cta, (b + 1) * per_cta).  Nothing of the message is written unless all of it fits
// the buffer (pack), nothing is taken from one that fails a check (unpack: every row comes back invalid).
template <bool PACK>
__global__ void __launch_bounds__(THREADS) wire_kernel(WireArgs a, int per_cta) {
    __shared__ int part[2][WARPS], offset[THREADS];
    grid_dependency_sync();
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int row0 = blockIdx.x * per_cta, row1 = min(a.R, row0 + per_cta);
    const short* wire_counts = reinterpret_cast<const short*>(a.buf + 16);
    unsigned h[4] = {0u, 0u, 0u, 0u};
    bool ok = true;
    if (!PACK) {
        // header: refuse a message for another shape, of another kind, or cut short
        ok = a.capacity >= 16;
        if (ok) {
#pragma unroll
            for (int x = 0; x < 4; ++x) h[x] = reinterpret_cast<const unsigned*>(a.buf)[x];
            const unsigned k = h[2] & 0xffffu, pt = h[2] >> 16;
            ok = h[0] == WIRE_MAGIC && h[1] == (unsigned)a.R && k == (unsigned)a.K && pt <= 1u &&
                 a.capacity >= wire_bytes(a.R, h[3], (int)pt);
        }
    }
    // a row's count; out of range: -1, and `bad` (pack: the row travels as invalid; unpack: the message is refused)
    auto count_of = [&](int r, bool& bad) {
        const int c = PACK ? a.q_count[r] : (int)wire_counts[r];
        if (c > a.K || c < -1) {
            bad = true;
            return -1;
        }
        return c;
    };
    // ---- entries in all rows, and in those before this CTA's
    int before = 0, total = 0;
    bool bad = false;
    if (ok) {
#pragma unroll 4
        for (int r = tid; r < a.R; r += THREADS) {
            const int n = max(count_of(r, bad), 0);
            total += n;
            if (r < row0) before += n;
        }
    }
    __syncwarp();
    before = __reduce_add_sync(0xffffffffu, before);
    total = __reduce_add_sync(0xffffffffu, total);
    if (lane == 0) {
        part[0][warp] = before;
        part[1][warp] = total;
    }
    bad = __syncthreads_or(bad);
    before = total = 0;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
        before += part[0][w];
        total += part[1][w];
    }
    const int ptype = PACK ? a.prob_type : (int)(h[2] >> 16);
    const long long need = wire_bytes(a.R, total, ptype);
    if (PACK) ok = need <= a.capacity;
    else ok = ok && !bad && (unsigned)total == h[3];
    if (blockIdx.x == 0 && tid == 0) {
        if (bad || !ok) atomicOr(a.status, ST_RANGE);
        if (PACK) {
            *a.bytes_out = ok ? need : -1;
            if (ok) {
                unsigned* out = reinterpret_cast<unsigned*>(a.buf);
                out[0] = WIRE_MAGIC;
                out[1] = (unsigned)a.R;
                out[2] = (unsigned)a.K | ((unsigned)a.prob_type << 16);
                out[3] = (unsigned)total;
                if (a.R & 1) reinterpret_cast<short*>(a.buf + 16)[a.R] = 0;      // padding of the counts
                if (a.prob_type == 1 && (total & 1))                              // padding of the message
                    *reinterpret_cast<unsigned short*>(a.buf + need - 2) = 0;
            }
        }
    }
    if (PACK && !ok) return;
    int* ids = reinterpret_cast<int*>(a.buf + 16 + wire_pad4(2ll * a.R));
    unsigned char* probs = reinterpret_cast<unsigned char*>(ids + (ok ? total : 0));
    const int tpr = wire_row_threads(a.K), sub = tid / tpr, t = tid - sub * tpr;
    for (int s0 = row0; s0 < row1; s0 += THREADS) {
        // ---- first entry of each of the next 256 rows
        const int r = s0 + tid;
        bool unused = false;
        const int n = ok && r < row1 ? max(count_of(r, unused), 0) : 0;
        int incl = n;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, d);
            incl += lane >= d ? y : 0;
        }
        __syncthreads();            // (the exchange areas of the step before are read)
        if (lane == 31) part[0][warp] = incl;
        __syncthreads();
        int base = before;
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
            if (w < warp) base += part[0][w];
            before += part[0][w];
        }
        offset[tid] = base + incl - n;
        __syncthreads();
        // ---- move
        for (int q = sub; q < THREADS && s0 + q < row1; q += THREADS / tpr) {
            const int rr = s0 + q, o = offset[q];
            const int c = ok ? count_of(rr, unused) : -1;
            const int m = max(c, 0);
            int* qi = a.q_idx + (long long)rr * a.K;
            float* qp = a.q_prob + (long long)rr * a.K;
            if (PACK) {
                if (t == 0) reinterpret_cast<short*>(a.buf + 16)[rr] = (short)c;
                for (int j0 = 0; j0 < m; j0 += 4 * tpr) {
                    int id[4];
                    float p[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int j = j0 + x * tpr + t;
                        id[x] = j < m ? qi[j] : 0;
                        p[x] = j < m ? qp[j] : 0.f;
                    }
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int j = j0 + x * tpr + t;
                        if (j < m) {
                            ids[o + j] = id[x];
                            if (ptype == 0) reinterpret_cast<float*>(probs)[o + j] = p[x];
                            else reinterpret_cast<__half*>(probs)[o + j] = __float2half_rn(p[x]);
                        }
                    }
                }
            } else {
                if (t == 0) a.q_count[rr] = c;
                for (int j0 = 0; j0 < a.K; j0 += 4 * tpr) {
                    int id[4];
                    float p[4];
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int j = j0 + x * tpr + t;
                        id[x] = -1;
                        p[x] = 0.f;
                        if (j < m) {
                            id[x] = ids[o + j];
                            p[x] = ptype == 0 ? reinterpret_cast<const float*>(probs)[o + j]
                                              : __half2float(reinterpret_cast<const __half*>(probs)[o + j]);
                        }
                    }
#pragma unroll
                    for (int x = 0; x < 4; ++x) {
                        const int j = j0 + x * tpr + t;
                        if (j < a.K) {
                            qi[j] = id[x];
                            qp[j] = p[x];
                        }
                    }
                }
            }
        }
    }
}

}  // namespace picospec
