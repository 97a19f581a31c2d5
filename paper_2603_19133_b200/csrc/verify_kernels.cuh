// Target-side kernels: streaming chunk statistics, per-sequence finish (accept test, scan,
// residual mass, two-level sampler) and the double-precision re-evaluation of flagged sequences.
#pragma once
#include "common.cuh"
#include "precise_kernels.cuh"
#include "stream_pipeline.cuh"

namespace picospec {

struct VerifyArgs {
    const void* logits;        // target logits [B, G+1, V]
    long long row_stride;      // elements
    int B, G, V, nch, k_max;
    int sample_only;           // 1: residual_sample entry point (row pos[b] only)
    // incremental verification: only the target rows [r0, r1) are read, for sequences that are
    // still undecided; the whole batch at once is r0 = 0, r1 = G + 1 with the pointers null
    int r0 = 0, r1 = -1;
    const int* gamma = nullptr;     // [B] drafted tokens per sequence (rows 0 .. gamma[b]); null: G
    const int* state_in = nullptr;  // [B] 1 = undecided so far, 0 = decided earlier (skipped); null: all 1
    int* state_out = nullptr;       // [B] or null
    const float* temperature;  // [B]
    const int* draft_tok;      // [B,G]
    const int* q_idx;          // [B,G,k_max]
    const float* q_prob;
    const int* q_count;        // [B,G]
    const float* u_accept;     // [B,G]
    const int* pos;            // [B] (sample_only)
    const float* u_resample;   // [B,2] or null
    int* accept_len;           // [B]
    float* p_draft;            // [B,G]
    float* resid_mass;         // [B,G]
    int* borderline;           // [1]
    int* token;                // [B] or null
    float* mass;               // [B] or null (sample_only)
    // Vocabulary-parallel verification (the logits are sharded along the vocabulary over several
    // ranks): the chunk records of all ranks lie rank after rank, [ranks, rows, chunks_per_rank], and
    // chunk c of the vocabulary is record c % chunks_per_rank of rank c / chunks_per_rank; one rank,
    // chunks_per_rank = nch is the plain layout.  entry_logits, if set, holds the target logits at the
    // stored entries (slots 0 .. k_max - 1) and at the drafted token (slot k_max) of every draft
    // position, gathered from the ranks that own them: the finish kernel then reads no logits itself
    // and hands the draw inside the picked chunk to that chunk's owner through `pick`.
    int chunks_per_rank = 0;        // 0: nch
    long long rank_stride = 0;      // records between two ranks' blocks
    int stats_pitch = 0;            // records per row written by the streaming pass (0: nch)
    const float* entry_logits = nullptr;   // [B*G, k_max + 1]
    bool cm_rows = false;           // the finish kernel keeps the chunk masses of every row it reads
    int* pick = nullptr;            // [B, 4]: sampled row, picked chunk (-1: none), flags, unused
    // workspace
    float2* stats;             // [B*(G+1), nch]: (chunk max logit, sum of 2^(l*c32 - max*c32))
    float* row_max;            // [B*(G+1)]
    double* dsum;              // [B*(G+1), nch]: exact chunk sums of flagged sequences
    int* queue;                // [B] flagged sequences
    unsigned long long* need_rows;  // [B] per flagged sequence: bit i = row i needs exact chunk sums
    int* queue_count;          // [1]
    int* rowq;                 // [B*(G+1)] rows (of the logits tensor) whose exact chunk sums are wanted
    int* rowq_count;           // [1]
    unsigned* status;          // sticky status word
    unsigned long long* slow_rows;  // cumulative rows re-evaluated in double precision
};

// Row r of the rows a verify call streams -> (sequence, row of the logits tensor); false: the row
// is not read (sequence decided earlier, or the row lies beyond the sequence's bonus row).
__device__ __forceinline__ bool streamed_row(const VerifyArgs& a, int r, int& b, int& src_row) {
    const int nr = a.r1 - a.r0;
    b = r / nr;
    const int i = a.r0 + (r - b * nr);
    src_row = b * (a.G + 1) + i;
    if (a.state_in && a.state_in[b] == 0) return false;
    if (a.gamma && i > a.gamma[b]) return false;
    return true;
}

// index of the record of (row, chunk c of the vocabulary) in stats / dsum
__device__ __forceinline__ long long record_index(const VerifyArgs& a, int row, int c) {
    if (a.chunks_per_rank == 0) return (long long)row * a.nch + c;      // one rank: the plain layout
    const int L = a.chunks_per_rank;
    const int r = c / L;
    return (long long)r * a.rank_stride + (long long)row * L + (c - r * L);
}
// flags of VerifyArgs::pick
constexpr int PICK_RESIDUAL = 1, PICK_FLAGGED = 2, PICK_DRAW_ONLY = 4, PICK_MASS_ONLY = 8;

// ---------------------------------------------------------------------------------------------
// Streaming pass through shared memory.  A tile is TILE_CHUNKS consecutive chunks of one row; CTA c takes tiles c, c + grid,
// c + 2 grid, ...  Warp 8 lane 0 is the producer: it keeps STAGES bulk copies in flight.  Each of
// the 8 consumer warps moves its chunk of a landed tile to registers, hands the stage back and
// then reduces the chunk to (maximum logit, fp32 sum of 2^((l - max) * log2e / T)).
// ---------------------------------------------------------------------------------------------
struct TileDesc {
    int src_row;   // row of the logits tensor
    int c0;        // first chunk of the tile
    float c32;     // log2(e) / T of the row's sequence
    int mis;       // elements between the row's first granule's start and the row (StagedRow)
    int valid;     // 0: bad temperature or position, or a row that is not read
};

template <typename T>
__global__ void __launch_bounds__(STREAM_THREADS, StreamCfg<T>::CTAS_PER_SM) chunk_stats_bulk_kernel(VerifyArgs a, int tiles_per_row,
                                                                             long long total_tiles,
                                                                             unsigned long long wait_limit_ns) {
    extern __shared__ __align__(1024) unsigned char stage_mem[];
    constexpr int STAGES = StreamCfg<T>::STAGES;
    constexpr int CPW = StreamCfg<T>::CPW;
    constexpr int TCH = TileGeom<T>::CHUNKS;
    constexpr int TILE_BYTES = TileGeom<T>::TILE_BYTES, STAGE_BYTES = TileGeom<T>::STAGE_BYTES;
    __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES];
    // Twice as many descriptors as stages: a warp uses the descriptor of a tile after it has handed the
    // stage back, and certainly no longer once it hands back the stage's next tile.
    __shared__ TileDesc desc[2][STAGES];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], WARPS);
        }
        mbar_init_fence();
    }
    grid_dependency_sync();
    if (tid == 0 && blockIdx.x == 0) {
        *a.queue_count = 0;
        *a.rowq_count = 0;
        if (a.borderline) *a.borderline = 0;
    }
    __syncthreads();

    if (warp == WARPS) {
        // ---- producer ---------------------------------------------------------------------
        if (lane != 0) return;
        const uint64_t pol = l2_evict_first_policy();
        // tile t = (streamed row r, tile tc of it); the next tile of this CTA is gridDim.x further on
        const int step_r = (int)gridDim.x / tiles_per_row, step_tc = (int)gridDim.x - step_r * tiles_per_row;
        int r = (int)blockIdx.x / tiles_per_row, tc = (int)blockIdx.x - r * tiles_per_row;
        uint32_t i = 0;
        for (long long t = blockIdx.x; t < total_tiles; ++i, t += gridDim.x) {
            const int s = (int)(i % STAGES);
            const uint32_t round = i / STAGES;
            TileDesc d;
            bool wanted = true;
            int b;
            if (a.sample_only) {
                b = r;
                const int j = a.pos[b];
                if (j < 0 || j > a.G) wanted = false;
                d.src_row = b * (a.G + 1) + (wanted ? j : 0);
            } else {
                wanted = streamed_row(a, r, b, d.src_row);
            }
            const StagedRow<T> sr(reinterpret_cast<const T*>(a.logits) + (long long)d.src_row * a.row_stride, a.V);
            if (round > 0) {
                const int wr = mbar_wait_twice(&empty[s], (round - 1) & 1, wait_limit_ns);
                if (wr != WAIT_OK) atomicOr(a.status, ST_INTERNAL);
                if (wr == WAIT_LOST) break;       // nothing more is issued
            }
            if (wanted) {
                constexpr int GRANULES = TILE_BYTES / 16;
                stage_tile<T>(stage_mem + s * STAGE_BYTES, sr, tc * GRANULES, GRANULES + (sr.mis ? 1 : 0), &full[s], pol);
            }
            // (looked up with the copy in flight; the copy of a row with a bad temperature is not used)
            const float Tb = a.temperature[b];
            d.valid = wanted && temp_ok(Tb);
            d.c32 = temp_scale(Tb);
            d.c0 = tc * TCH;
            d.mis = sr.mis;
            desc[round & 1][s] = d;
            mbar_arrive(&full[s]);
            r += step_r;
            tc += step_tc;
            if (tc >= tiles_per_row) {
                tc -= tiles_per_row;
                ++r;
            }
        }
        return;
    }

    // ---- consumers ------------------------------------------------------------------------
    long long t = blockIdx.x;
    bool late = false;      // a wait ran out: this warp computes no more, but keeps taking tiles
    for (uint32_t i = 0; t < total_tiles; ++i, t += gridDim.x) {
        const int s = (int)(i % STAGES);
        const uint32_t round = i / STAGES;
        const int wr = mbar_wait_twice(&full[s], round & 1, wait_limit_ns);
        if (wr != WAIT_OK) {
            late = true;
            if (lane == 0) atomicOr(a.status, ST_INTERNAL);
            if (wr == WAIT_LOST) break;
        }
        const TileDesc d = desc[round & 1][s];
#pragma unroll
        for (int q = 0; q < CPW; ++q) {
            const int c = d.c0 + warp * CPW + q;
            const bool work = d.valid && c < a.nch && !late;
            ChunkRegs<T> regs;
            if (work)
                load_staged_shifted(regs, stage_mem + s * STAGE_BYTES + (warp * CPW + q) * (CHUNK * (int)sizeof(T)), c * CHUNK,
                                    a.V + d.mis, d.mis, lane);
            // chunk maximum with NaN ignored; a NaN (or +inf) logit turns the exp-sum into NaN by
            // itself, which the finish kernel reports; a chunk of -inf only sums to zero
            const float cm = work ? warp_max_redux(regs.lane_max_plain()) : 0.f;
            if (q == CPW - 1) {
                // The stage is handed back only behind an instruction that needs every lane's entries: an
                // arrive may overtake shared-memory loads that are issued but still queued, and with
                // another kernel's gathers in the queue they were queued long enough for the next copy
                // to land first.
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty[s]);
            }
            if (work) {
                const float off = cm > -CUDART_INF_F ? __fmul_rn(cm, d.c32) : 0.f;
                const float sum = warp_sum(lane_exp_sum2(regs, d.c32, off));
                if (lane == 0) a.stats[(long long)d.src_row * (a.stats_pitch > 0 ? a.stats_pitch : a.nch) + c] = make_float2(cm, sum);
            }
        }
    }
}

// ---------------------------------------------------------------------------------------------
// Finish: one CTA per sequence.
// ---------------------------------------------------------------------------------------------
struct FinishShared {
    double Z[MAX_G1];     // normaliser on the scale of Weight<>
    double Zraw[MAX_G1];  // the same sum on the streaming pass's own scale (fast path)
    float mx[MAX_G1];
    int bad;
    int flag;
    unsigned char test[MAX_G1];   // per draft position: TEST_* bits
    double warp_tot[WARPS], warp_q[WARPS];
    int warp_first[WARPS], warp_last[WARPS];
    __align__(16) float qloc[CHUNK];
};

// queue entries of the verify path: the sequence, plus a flag
constexpr int QUEUE_SEQ_MASK = 0x1FFFFFFF, QUEUE_DRAW_ONLY = 0x40000000, QUEUE_MASS_ONLY = 0x20000000;

// outcome of a position's test: accepted, too close to call, borderline, small residual mass
constexpr int TEST_ACC = 1, TEST_AMB = 2, TEST_BORD = 4, TEST_SMALL = 8;

// bit i of a sequence's row mask (rows beyond 63 always count as set)
__device__ __forceinline__ bool row_needed(unsigned long long need, int i) { return i >= 64 || ((need >> i) & 1ull); }

// Combine the chunk statistics of one row (called by a full warp): the exact double-precision chunk sums
// if they were recomputed for this row, else the fp32 streaming statistics.  masses (or null): [nch]
// doubles of shared memory that receive the chunk masses, in units where the row sums to one.
template <typename T>
__device__ __forceinline__ void row_stats(const VerifyArgs& a, int src_row, float c32, int lane, bool exact, double& Z,
                                          double& Zraw, float& mx, bool& bad, double* masses = nullptr) {
    bad = false;
    Zraw = 0.0;
    double scale;
    if (exact) {
        mx = a.row_max[src_row];
        double s = 0.0;
        for (int c = lane; c < a.nch; c += 32) {
            const double e = a.dsum[record_index(a, src_row, c)];
            s += e;
            if (masses) masses[c] = e;
        }
        __syncwarp();
        Z = warp_sum(s);
        scale = 1.0 / Z;
    } else {
        constexpr int HELD = 8;         // records per lane that stay in registers: the first 256 chunks
        float2 held[HELD];
        float m = -CUDART_INF_F;
        bool nan = false;
#pragma unroll
        for (int u = 0; u < HELD; ++u) {
            const int c = u * 32 + lane;
            held[u] = c < a.nch ? a.stats[record_index(a, src_row, c)] : make_float2(-CUDART_INF_F, 0.f);
        }
#pragma unroll
        for (int u = 0; u < HELD; ++u) {
            m = fmaxf(m, held[u].x);
            nan |= held[u].y != held[u].y;
        }
        for (int c = HELD * 32 + lane; c < a.nch; c += 32) {
            const float2 v = a.stats[record_index(a, src_row, c)];
            m = fmaxf(m, v.x);
            nan |= v.y != v.y;
        }
        __syncwarp();
        m = warp_max_redux(m);
        nan = __any_sync(0xffffffffu, nan);
        mx = m;
        bad = nan || !(m > -CUDART_INF_F) || !(m < CUDART_INF_F);
        double s = 0.0;
        const double off = (double)__fmul_rn(m, c32);
        if (!bad) {
            // (one copy of the body, the records shifted through: see exp_call)
#pragma unroll 1
            for (int c0 = 0; c0 < a.nch; c0 += 32) {
                const int c = c0 + lane;
                float2 v = held[0];
#pragma unroll
                for (int u = 0; u + 1 < HELD; ++u) held[u] = held[u + 1];
                if (c0 >= HELD * 32) v = c < a.nch ? a.stats[record_index(a, src_row, c)] : make_float2(-CUDART_INF_F, 0.f);
                const double e = v.x > -CUDART_INF_F ? (double)v.y * exp2_call((double)__fmul_rn(v.x, c32) - off) : 0.0;
                s += e;
                if (masses && c < a.nch) masses[c] = e;
            }
        }
        __syncwarp();
        Zraw = warp_sum(s);
        if (!(Zraw > 0.0)) bad = true;
        Z = bad ? 0.0 : Zraw * stream_sum_scale(m, c32);
        scale = 1.0 / Zraw;
    }
    if (masses)
        for (int c = lane; c < a.nch; c += 32) masses[c] *= scale;      // (each lane its own)
    __syncwarp();
}

// Level 2 of the sampler, by the 256 threads of a CTA: the token inside chunk `cs` of a row whose
// logits start at `row` with vocabulary index `vbase` (0 for a whole row; the first index of the
// slice when the vocabulary is sharded).  Weights are max(0, p - q~) with the stored entries
// (idx, prob)[0 .. n) if use_resid, else p.  sh.qloc is zero on entry (and a barrier lies behind that).
// Sets sh.flag when the fast pass cannot call the draw.
template <typename T, bool PRECISE>
__device__ __forceinline__ int level2_draw(const VerifyArgs& a, const T* row, int vbase, int cs, const int* idx,
                                           const float* prob, int n, bool use_resid, const Weight<PRECISE>& wt,
                                           double invZ, float u2, FinishShared& sh) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // the 1024 entries of chunk cs, four consecutive entries per thread
    const int v0 = cs * CHUNK;
    float l[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int v = v0 + tid * 4 + e;
        l[e] = v < a.V ? load_logit(row, v - vbase) : -CUDART_INF_F;
    }
    if (use_resid) {
        for (int k = tid; k < n; k += THREADS) {
            const int v = idx[k];
            if (v >= v0 && v < v0 + CHUNK) sh.qloc[v - v0] = prob[k];
        }
        __syncthreads();
    }
    const float4 ql = *reinterpret_cast<const float4*>(&sh.qloc[tid * 4]);
    const float qv[4] = {ql.x, ql.y, ql.z, ql.w};
    double r[4], cum[4], qsum = 0.0, loc = 0.0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const double w = v0 + tid * 4 + e < a.V ? wt(l[e]) * invZ : 0.0;
        const double q = (double)qv[e];
        qsum += q;
        const double d = w - q;
        r[e] = d > 0.0 ? d : 0.0;
        loc += r[e];
        cum[e] = loc;
    }
    // running sum of the weights and total of the stored probabilities
    double incl = loc;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const double y = __shfl_up_sync(0xffffffffu, incl, d);
        incl += lane >= d ? y : 0.0;
    }
    qsum = use_resid ? warp_sum(qsum) : 0.0;
    if (lane == 31) {
        sh.warp_tot[warp] = incl;
        sh.warp_q[warp] = qsum;
    }
    __syncthreads();
    double M = 0.0, Q = 0.0, base = incl - loc;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
        const double t = sh.warp_tot[w];
        if (w < warp) base += t;
        M += t;
        Q += sh.warp_q[w];
    }
    const double thr2 = (double)u2 * M;
    int mine = 0x7fffffff, mylast = -1;
#pragma unroll
    for (int e = 3; e >= 0; --e) {
        if (base + cum[e] > thr2) mine = v0 + tid * 4 + e;
        if (r[e] > 0.0 && mylast < 0) mylast = v0 + tid * 4 + e;
    }
    const int wfirst = __reduce_min_sync(0xffffffffu, mine), wlast = __reduce_max_sync(0xffffffffu, mylast);
    if (lane == 0) {
        sh.warp_first[warp] = wfirst;
        sh.warp_last[warp] = wlast;
    }
    __syncthreads();
    int first = 0x7fffffff, last = -1;
#pragma unroll
    for (int w = 0; w < WARPS; ++w) {
        first = min(first, sh.warp_first[w]);
        last = max(last, sh.warp_last[w]);
    }
    const int token = first != 0x7fffffff ? first : last;
    if (!PRECISE && use_resid && Q > 0.0) {
        // with q~ present the thresholds depend on the normaliser: error <= GUARD_Z * Q
        const double E2 = 2.0 * GUARD_Z * Q;
        if (first == 0x7fffffff) {
            if (tid == 0) sh.flag = 1;
        } else if (mine == first) {
            const int e = mine - (v0 + tid * 4);
            double at = 0.0, re = 0.0;
#pragma unroll
            for (int x = 0; x < 4; ++x)
                if (x == e) {
                    at = base + cum[x];
                    re = r[x];
                }
            const double hi = at - thr2;
            const double lo = thr2 - (at - re);
            if (hi < E2 || lo < E2) sh.flag = 1;
        }
    }
    __syncthreads();
    return token;
}

__device__ __forceinline__ void zero_qloc(FinishShared& sh) {
    *reinterpret_cast<float4*>(&sh.qloc[threadIdx.x * 4]) = make_float4(0.f, 0.f, 0.f, 0.f);
}
// bits lo .. hi - 1
__device__ __forceinline__ unsigned long long bit_range(int lo, int hi) {
    const unsigned long long below_hi = hi >= 64 ? ~0ull : (1ull << hi) - 1ull;
    return lo >= 64 ? 0ull : below_hi & (~0ull << lo);
}

// Chunk masses of row j by the 256 threads of a CTA, into cm (a barrier follows); `entries`: with the stored
// entries' shares taken out.  For the calls whose rows' masses do not all fit shared memory, and for
// a residual that vanished.
template <typename T, bool PRECISE, bool SHARDED>
__device__ __noinline__ void chunk_masses(const VerifyArgs& a, FinishShared& sh, double* cm, int b, int j, bool exact,
                                          bool entries, int n) {
    const int G1 = a.G + 1, tid = threadIdx.x, rj = b * a.G + j;
    const float Tb = a.temperature[b];
    const float c32 = temp_scale(Tb);
    const double invZ = 1.0 / sh.Z[j];
    // at most 1024 entries, four per thread: their logits are under way while the masses form
    constexpr int PER = MAX_K / THREADS;
    const T* row = reinterpret_cast<const T*>(a.logits) + (long long)(b * G1 + j) * a.row_stride;
    int vv[PER];
    float qq[PER], ll[PER];
    if (!entries) n = 0;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const int k = tid + u * THREADS;
        vv[u] = k < n ? a.q_idx[(long long)rj * a.k_max + k] : -2;
        qq[u] = k < n ? a.q_prob[(long long)rj * a.k_max + k] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < PER; ++u) {
        const bool ok = vv[u] >= 0 && vv[u] < a.V;
        if (vv[u] != -2 && !ok) atomicOr(&sh.bad, (int)ST_RANGE);
        ll[u] = ok ? (SHARDED ? a.entry_logits[(long long)rj * (a.k_max + 1) + tid + u * THREADS] : load_logit(row, vv[u]))
                   : -CUDART_INF_F;
    }
    if (exact) {
        for (int c = tid; c < a.nch; c += THREADS) cm[c] = a.dsum[record_index(a, b * G1 + j, c)] * invZ;
    } else {
        const double off = (double)__fmul_rn(sh.mx[j], c32);
        const double scale = 1.0 / sh.Zraw[j];
        for (int c = tid; c < a.nch; c += THREADS) {
            const float2 v = a.stats[record_index(a, b * G1 + j, c)];
            cm[c] = v.x > -CUDART_INF_F ? (double)v.y * exp2_call((double)__fmul_rn(v.x, c32) - off) * scale : 0.0;
        }
    }
    __syncthreads();
    if (!entries) return;
    Weight<PRECISE> wt;
    wt.init(Tb, sh.mx[j]);
    double w[PER];
#pragma unroll
    for (int u = 0; u < PER; ++u) w[u] = wt.inlined(ll[u]);
#pragma unroll
    for (int u = 0; u < PER; ++u)
        if (vv[u] >= 0 && vv[u] < a.V) atomicAdd(&cm[vv[u] / CHUNK], -fmin(w[u] * invZ, (double)qq[u]));
    __syncthreads();
}

// One sequence (fast pass: sequence `slot`; double-precision pass: entry `slot` of the queue), by the
// 256 threads of a CTA.  cm: shared memory for the chunk masses: of every row that is read ([rows, nch]
// doubles) if a.cm_rows, else of the sampled row alone.
// SHARDED: vocabulary-parallel verification (a.entry_logits and a.pick are set).
//
// Bound by latency: a chain of loads, double-precision arithmetic and (since a CTA runs through the code
// once) instruction fetches.  Hence the order: all that does not depend on the streaming pass -- the
// stored entries and the logits at them -- is read before the kernel waits for that pass; a warp takes
// a row from its statistics through its test and leaves the row's chunk masses, with the entries'
// shares taken out, in shared memory, so that the draw starts from them whichever row it falls on.
// End to end after the streaming pass: 11.3 -> 8.0 us (8 sequences x 5, K = 64), 18.4 -> 11.3 (64 x 8,
// K = 128), 26 -> 13 (256 x 6, K = 256).  At K = 1024 (512 x 8: 197 -> 175 us) it is bound by the DRAM
// sectors of the gathers instead.  Without the reads before the wait 256 x 6 takes 24.6 us, with the
// streaming pass 5 us shorter for it.
// HELD: entries per lane that stay in registers (rows of at most 64 entries need two).
template <typename T, bool PRECISE, bool SHARDED, int HELD>
__device__ __forceinline__ void verify_finish_slot(const VerifyArgs& a, int slot, FinishShared& sh, double* cm) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int G = a.G, G1 = a.G + 1;
    {
        // a queue entry is the sequence, with QUEUE_DRAW_ONLY set when only the draw was too close to
        // call: then the accept decisions of the fast pass stand and only the sampled row is redone;
        // with QUEUE_MASS_ONLY every decision stands and only small residual masses are recomputed
        const int qe = PRECISE ? a.queue[slot] : slot;
        const int b = PRECISE ? (qe & QUEUE_SEQ_MASK) : slot;
        const bool draw_only = PRECISE && (qe & QUEUE_DRAW_ONLY) != 0;
        const bool mass_only = PRECISE && (qe & QUEUE_MASS_ONLY) != 0;
        const int alen_fast = draw_only ? a.accept_len[b] : 0;
        const unsigned long long need = PRECISE ? a.need_rows[b] : 0ull;   // rows with exact chunk sums
        if (!PRECISE && !a.sample_only && a.state_in && a.state_in[b] == 0) {
            // decided by an earlier call: nothing of this sequence is read or written
            // (the queue of the double-precision pass holds none of these; there state_in may be the
            // array in which the fast pass has just marked the sequence as decided by this call)
            grid_dependency_sync();
            if (tid == 0 && a.state_out) a.state_out[b] = 0;
            return;
        }
        const float Tb = a.temperature[b];
        const float c32 = temp_scale(Tb);
        const T* seq = reinterpret_cast<const T*>(a.logits) + (long long)b * G1 * a.row_stride;
        unsigned st_bits = 0;
        if (!temp_ok(Tb)) st_bits |= ST_TEMPERATURE;
        // the two uniforms of the draw, requested long before the chunk masses are ready
        const float u_chunk = a.u_resample ? a.u_resample[2 * b] : 0.f;
        const float u_entry = a.u_resample ? a.u_resample[2 * b + 1] : 0.f;
        // rows lo .. row_hi-1 are read, positions lo .. hi-1 are tested; g is the bonus row
        const int lo = a.sample_only ? 0 : a.r0;
        const int g = (!a.sample_only && a.gamma) ? a.gamma[b] : G;
        if (g < 0 || g > G || g < lo) st_bits |= ST_RANGE;
        const int hi = a.sample_only ? G : min(g, a.r1);
        const int row_hi = a.sample_only ? G1 : min(g + 1, a.r1);
        int jpos = -1;
        if (a.sample_only) {
            jpos = a.pos[b];
            if (jpos < 0 || jpos > G) st_bits |= ST_RANGE;
        }
        const int i_lo = a.sample_only ? jpos : lo, i_hi = a.sample_only ? jpos + 1 : row_hi;
        __syncthreads();        // (the sequence before is done with the shared state)
        if (tid == 0) {
            sh.bad = 0;
            sh.flag = 0;
        }
        if (!SHARDED) zero_qloc(sh);
        __syncthreads();

        // ---- 1. a warp per row: the normaliser; for a draft position p(x), q~(x), accept test,
        // ----    residual mass
        if (!st_bits) {
            for (int i = i_lo + warp; i < i_hi; i += WARPS) {
                if (draw_only && i != alen_fast) continue;
                if (mass_only && !row_needed(need, i)) continue;
                const bool tested = !a.sample_only && !draw_only && i < hi;
                const bool entries = tested || (a.cm_rows && (a.sample_only ? i < G : i < hi));
                const int ri = b * G + (entries ? i : 0);
                const int* idx = a.q_idx + (long long)ri * a.k_max;
                const float* prob = a.q_prob + (long long)ri * a.k_max;
                const T* row = seq + (long long)i * a.row_stride;
                const float* ent = SHARDED ? a.entry_logits + (long long)ri * (a.k_max + 1) : nullptr;
                // the first batch of stored entries is requested before the row's count is known
                // (every slot below k_max exists; slots at or beyond the count are dropped below)
                int vv[HELD], x = -1, n = 0;
                float qq[HELD], ll[HELD], ux = 0.f, lx = -CUDART_INF_F;
                bool range_bad = false;
                if (entries) {
                    n = a.q_count[ri];
                    if (tested) {
                        x = a.draft_tok[ri];
                        ux = a.u_accept[ri];
                    }
#pragma unroll
                    for (int u = 0; u < HELD; ++u) {
                        const int k = u * 32 + lane;
                        vv[u] = k < a.k_max ? idx[k] : -2;
                        qq[u] = k < a.k_max ? prob[k] : 0.f;
                    }
                    range_bad = n < 0 || n > a.k_max || (tested && (x < 0 || x >= a.V));
                    // p(x) on every lane (the same instructions as on one lane, and no divergent tail)
                    if (tested && !range_bad) lx = SHARDED ? ent[a.k_max] : load_logit(row, x);
#pragma unroll
                    for (int u = 0; u < HELD; ++u) {
                        const int k = u * 32 + lane;
                        if (k >= n || range_bad) vv[u] = -2;
                        const bool ok = vv[u] >= 0 && vv[u] < a.V;
                        ll[u] = ok ? (SHARDED ? ent[k] : load_logit(row, vv[u])) : -CUDART_INF_F;
                    }
                }
                grid_dependency_sync();
                double Z, Zraw;
                float mx;
                bool bad;
                double* masses = a.cm_rows ? cm + (long long)(i - i_lo) * a.nch : nullptr;
                row_stats<T>(a, b * G1 + i, c32, lane, PRECISE && row_needed(need, i), Z, Zraw, mx, bad, masses);
                if (lane == 0) {
                    sh.Z[i] = Z;
                    sh.Zraw[i] = Zraw;
                    sh.mx[i] = mx;
                    if (!PRECISE) a.row_max[b * G1 + i] = mx;
                    if (bad) atomicOr(&sh.bad, (int)ST_LOGIT);
                }
                if (!entries || bad) continue;
                Weight<PRECISE> wt;
                wt.init(Tb, mx);
                const double invZ = 1.0 / Z;     // the sums below take p = w * (1/Z): 2^-53 relative per term
                double smin = 0.0;
                float qx_mine = 0.f;
                int kx = 0x7fffffff;
                const int n_read = range_bad ? 0 : n;
                // entry k (v, q) with the logit l: its share of the residual; the weight w = exp(l/T - mx/T)
                auto take = [&](int k, int v, float q, double w) {
                    const bool ok = v >= 0 && v < a.V;
                    if (v != -2 && !ok) range_bad = true;
                    if (ok) {
                        const double d = fmin(w * invZ, (double)q);
                        smin += d;
                        if (masses) atomicAdd(&masses[v / CHUNK], -d);
                        if (v == x && k < kx) {
                            kx = k;
                            qx_mine = q;
                        }
                    }
                };
                if (HELD == 2 || n_read <= 64) {
                    // few entries: one copy of the body (see exp_call)
#pragma unroll 1
                    for (int k0 = 0; k0 < n_read; k0 += 32) {
                        take(k0 + lane, vv[0], qq[0], wt(ll[0]));
                        vv[0] = vv[1];
                        qq[0] = qq[1];
                        ll[0] = ll[1];
                        __syncwarp();
                    }
                } else if constexpr (HELD == 8) {
                    // many: four exponentials in flight
#pragma unroll 1
                    for (int k0 = 0; k0 < n_read; k0 += 128) {
                        if ((k0 & 255) == 0 && k0 > 0) {
                            // the next 256 entries, loads first
#pragma unroll
                            for (int u = 0; u < 8; ++u) {
                                const int k = k0 + u * 32 + lane;
                                vv[u] = k < n ? idx[k] : -2;
                                qq[u] = k < n ? prob[k] : 0.f;
                            }
#pragma unroll
                            for (int u = 0; u < 8; ++u) {
                                const bool ok = vv[u] >= 0 && vv[u] < a.V;
                                ll[u] = ok ? (SHARDED ? ent[k0 + u * 32 + lane] : load_logit(row, vv[u])) : -CUDART_INF_F;
                            }
                        }
                        double w[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u) w[u] = wt.inlined(ll[u]);
#pragma unroll
                        for (int u = 0; u < 4; ++u) take(k0 + u * 32 + lane, vv[u], qq[u], w[u]);
#pragma unroll
                        for (int u = 0; u < 4; ++u) {
                            vv[u] = vv[u + 4];
                            qq[u] = qq[u + 4];
                            ll[u] = ll[u + 4];
                        }
                        __syncwarp();
                    }
                }
                if (!tested) {
                    if (__any_sync(0xffffffffu, range_bad) && lane == 0) atomicOr(&sh.bad, (int)ST_RANGE);
                    continue;
                }
                const double px = wt(lx) / Z;
                range_bad = __any_sync(0xffffffffu, range_bad);
                smin = warp_sum(smin);
                kx = __reduce_min_sync(0xffffffffu, kx);
                // the stored probability of the first entry that names the draft token sits in lane kx % 32
                float qx = __shfl_sync(0xffffffffu, qx_mine, kx & 31);
                if (kx == 0x7fffffff) qx = 0.f;
                if (lane == 0) {
                    if (range_bad) {
                        atomicOr(&sh.bad, (int)ST_RANGE);
                    } else {
                        const double u = (double)ux;
                        bool acc = true, amb = false, bord = false;
                        if (qx > 0.f) {
                            const double ratio = px / (double)qx;
                            acc = u < fmin(1.0, ratio);
                            const double dist = fabs(ratio - u);
                            if (PRECISE)
                                bord = dist <= BORDER_REL * u;
                            else
                                amb = dist <= (BORDER_REL + GUARD_Z) * fmax(u, ratio);
                        }
                        double R = 1.0 - smin;
                        if (R < 0.0) R = 0.0;
                        // 1 - sum min(p, q~) inherits the absolute error of the fp32-accumulated
                        // normaliser: a small residual mass is reported from the exact sums instead
                        const bool small = !PRECISE && R < RESID_EXACT_BELOW;
                        sh.test[i] = (unsigned char)((acc ? TEST_ACC : 0) | (amb ? TEST_AMB : 0) | (bord ? TEST_BORD : 0) |
                                                     (small ? TEST_SMALL : 0));
                        a.p_draft[ri] = (float)px;
                        a.resid_mass[ri] = (float)R;
                    }
                }
            }
        }
        grid_dependency_sync();
        // (requested now, looked at when the outputs are written)
        const unsigned status_word = *(volatile unsigned*)a.status;
        __syncthreads();
        st_bits |= (unsigned)sh.bad;
        if (mass_only) return;          // (bad data was reported by the fast pass already)

        // ---- 2. first-rejection scan -----------------------------------------------------
        // A rejection inside the range decides the sequence; so does accepting every position
        // when the bonus row g is in the range.  Otherwise it waits for the next rows.
        int alen = lo, nborder = 0, first_amb = -1;
        bool flagged = false, rejected = false, decided = true;
        unsigned long long small_rows = 0ull;
        if (draw_only) {
            // (no accept test was ambiguous, so none is borderline either)
            alen = alen_fast;
            rejected = alen < hi;
        } else if (!st_bits && !a.sample_only) {
            const int t0 = lane >= lo && lane < hi ? sh.test[lane] : TEST_ACC;
            const int t1 = lane + 32 >= lo && lane + 32 < hi ? sh.test[lane + 32] : TEST_ACC;
            auto bits = [&](int which) {
                return (unsigned long long)__ballot_sync(0xffffffffu, t0 & which) |
                       (unsigned long long)__ballot_sync(0xffffffffu, t1 & which) << 32;
            };
            const unsigned long long refused = ~bits(TEST_ACC);
            rejected = refused != 0ull;
            alen = rejected ? __ffsll((long long)refused) - 1 : hi;
            decided = rejected || g < a.r1;
            const unsigned long long seen = bit_range(lo, rejected ? alen + 1 : hi);     // every decision that counts
            if (PRECISE) nborder = __popcll(bits(TEST_BORD) & seen);
            const unsigned long long amb = bits(TEST_AMB) & seen;
            if (amb) first_amb = __ffsll((long long)amb) - 1;
            small_rows = bits(TEST_SMALL);
            flagged = amb != 0ull || small_rows != 0ull;
        }

        // ---- 3. residual / bonus sample --------------------------------------------------
        int token = -1;
        int pick_row = 0, pick_chunk = -1;      // vocabulary-parallel: what the picked chunk's owner needs
        bool pick_resid = false;
        double Rtot = -1.0;
        const bool want_token = SHARDED || a.token != nullptr;
        if (!st_bits && want_token && decided) {
            const int j = a.sample_only ? jpos : alen;
            const int rj = b * G + j;
            int n = (a.sample_only ? j < G : rejected) ? a.q_count[rj] : 0;
            if (n < 0 || n > a.k_max) {
                n = 0;
                st_bits |= ST_RANGE;
            }
            const int* idx = a.q_idx + (long long)rj * a.k_max;
            const float* prob = a.q_prob + (long long)rj * a.k_max;
            const T* row = seq + (long long)j * a.row_stride;
            const bool exact = PRECISE && row_needed(need, j);
            bool use_resid = n > 0;
            int cstar = -1;
            double* mj = cm;
            if (a.cm_rows) mj = cm + (long long)(j - i_lo) * a.nch;
            else chunk_masses<T, PRECISE, SHARDED>(a, sh, cm, b, j, exact, use_resid, n);
            st_bits |= (unsigned)sh.bad;
            for (int pass = 0; pass < 2 && !st_bits; ++pass) {
                // level 1, by every warp for itself: lanes own contiguous blocks of chunks
                const int per = (a.nch + 31) / 32;
                const int c0 = lane * per;
                double s = 0.0;
#pragma unroll 1
                for (int c = c0; c < c0 + per; ++c)
                    if (c < a.nch) s += fmax(mj[c], 0.0);
                __syncwarp();
                double incl = s;
#pragma unroll
                for (int d = 1; d < 32; d <<= 1) {
                    const double y = __shfl_up_sync(0xffffffffu, incl, d);
                    incl += lane >= d ? y : 0.0;
                }
                Rtot = __shfl_sync(0xffffffffu, incl, 31);
                const double thr = (double)u_chunk * Rtot;
                double run = incl - s;
                int first = 0x7fffffff, lastpos = -1;
                bool close = false;
#pragma unroll 1
                for (int c = c0; c < c0 + per; ++c) {
                    if (c < a.nch) {
                        const double m = fmax(mj[c], 0.0);
                        run += m;
                        if (m > 0.0) lastpos = c;
                        if (run > thr) first = min(first, c);
                        // every prefix and the total carry an absolute error <= GUARD_Z
                        close |= fabs(run - thr) <= GUARD_Z;
                    }
                }
                __syncwarp();
                first = __reduce_min_sync(0xffffffffu, first);
                lastpos = __reduce_max_sync(0xffffffffu, lastpos);
                cstar = first != 0x7fffffff ? first : lastpos;
                if (!PRECISE && __any_sync(0xffffffffu, close) && tid == 0) sh.flag = 1;
                if (!use_resid) break;
                // the residual may vanish (q~ >= p everywhere): then the draw is from p itself
                const double tiny = PRECISE ? RESID_ZERO_BELOW : 4.0 * GUARD_Z;
                // (a reported mass this small would show the normaliser's error: exact sums instead)
                if (!PRECISE && a.mass && Rtot < RESID_EXACT_BELOW && tid == 0) sh.flag = 1;
                if (Rtot > tiny) break;
                if (!PRECISE) {
                    if (tid == 0) sh.flag = 1;   // too close to zero to call in fp32
                    break;
                }
                use_resid = false;  // precise: residual is zero, fall back to p
                __syncthreads();
                mj = cm;
                chunk_masses<T, PRECISE, SHARDED>(a, sh, cm, b, j, exact, false, 0);
            }
            pick_row = j;
            pick_chunk = cstar;
            pick_resid = use_resid;
            if (cstar >= 0 && !st_bits && !SHARDED) {
                Weight<PRECISE> wt;
                wt.init(Tb, sh.mx[j]);
                token = level2_draw<T, PRECISE>(a, row, 0, cstar, idx, prob, n, use_resid, wt, 1.0 / sh.Z[j], u_entry, sh);
            }
            flagged |= sh.flag != 0;
        }

        // ---- 4. outputs --------------------------------------------------------------------
        // a wait of the streaming pass ran out (now or in a call since the status word was last
        // cleared): its statistics are not complete, nothing of this call is valid
        if (status_word & ST_INTERNAL) st_bits |= ST_INTERNAL;
        if (tid == 0) {
            if (st_bits) {
                atomicOr(a.status, st_bits);
                if (!a.sample_only) {
                    a.accept_len[b] = -1;
                    for (int i = lo; i < hi && i < G; ++i) {
                        a.p_draft[b * G + i] = -1.f;
                        a.resid_mass[b * G + i] = -1.f;
                    }
                    if (a.state_out) a.state_out[b] = 0;
                }
                if (a.token) a.token[b] = -1;
                if (SHARDED) {
                    a.pick[4 * b + 0] = 0;
                    a.pick[4 * b + 1] = -1;
                    a.pick[4 * b + 2] = 0;
                }
                if (a.mass) a.mass[b] = -1.f;
            } else {
                if (!a.sample_only) {
                    a.accept_len[b] = decided ? alen : -2;
                    if (a.state_out) a.state_out[b] = decided ? 0 : 1;
                }
                if (a.token) a.token[b] = decided ? token : -2;
                if (a.mass) a.mass[b] = (float)Rtot;
                if (PRECISE) {
                    if (nborder && a.borderline) atomicAdd(a.borderline, nborder);
                    if (SHARDED) {
                        a.pick[4 * b + 0] = pick_row;
                        a.pick[4 * b + 1] = (decided && want_token) ? pick_chunk : -1;
                        a.pick[4 * b + 2] = pick_resid ? PICK_RESIDUAL : 0;
                    }
                } else if (flagged || SHARDED) {
                    // Which rows need exact sums: an ambiguous accept test can move the first
                    // rejection anywhere from its position on, so every row from there; an ambiguous
                    // draw needs the sampled row only; a small residual mass its own row.
                    unsigned long long nd = 0ull;
                    int nrows = 0;
                    bool draw_only_flag = false, mass_only_flag = false;
                    if (a.sample_only) {
                        nd = ~0ull;
                        nrows = 1;
                        a.rowq[atomicAdd(a.rowq_count, 1)] = b * G1 + jpos;
                    } else {
                        const bool any_small = small_rows != 0ull;
                        draw_only_flag = first_amb < 0 && !any_small;
                        mass_only_flag = first_amb < 0 && any_small && !sh.flag;
                        nd = small_rows;
                        if (first_amb >= 0) nd |= ~0ull << first_amb;
                        // (vocabulary-parallel: whether the draw inside the chunk is too close to call is
                        // only known to the chunk's owner later, so the sampled row is always listed)
                        if ((sh.flag || SHARDED) && want_token && decided && alen < 64) nd |= 1ull << alen;
                        nd &= bit_range(lo, row_hi);
                        const bool row64 = row_hi > 64;         // (row 64 has no bit: it always counts as listed)
                        nrows = __popcll(nd) + (row64 ? 1 : 0);
                        if (!SHARDED && nrows > 0) {
                            int at = atomicAdd(a.rowq_count, nrows);
                            for (unsigned long long left = nd; left; left &= left - 1ull)
                                a.rowq[at++] = b * G1 + __ffsll((long long)left) - 1;
                            if (row64) a.rowq[at] = b * G1 + 64;
                        }
                    }
                    a.need_rows[b] = nd;
                    if (SHARDED) {
                        // the queue is built once the owners' flags have been exchanged
                        a.pick[4 * b + 0] = pick_row;
                        a.pick[4 * b + 1] = (decided && want_token) ? pick_chunk : -1;
                        a.pick[4 * b + 2] = (pick_resid ? PICK_RESIDUAL : 0) | (flagged ? PICK_FLAGGED : 0) |
                                            (draw_only_flag ? PICK_DRAW_ONLY : 0) | (mass_only_flag ? PICK_MASS_ONLY : 0);
                        a.pick[4 * b + 3] = nrows;
                    } else {
                        const int q = atomicAdd(a.queue_count, 1);
                        a.queue[q] = b | (draw_only_flag ? QUEUE_DRAW_ONLY : 0) | (mass_only_flag ? QUEUE_MASS_ONLY : 0);
                        atomicAdd(a.slow_rows, (unsigned long long)nrows);
                    }
                }
            }
        }
    }
}

template <typename T, bool PRECISE, bool SHARDED = false, int HELD = 8>
__global__ void __launch_bounds__(THREADS, HELD == 2 ? 4 : 2) verify_finish_kernel(const __grid_constant__ VerifyArgs a) {
    extern __shared__ double cm[];  // chunk masses: of every row that is read (a.cm_rows), or of the sampled one
    __shared__ FinishShared sh;
    // Only the chunk statistics / exact sums come from the kernel before this one; whatever was written
    // before that kernel is visible as soon as this one runs, because that kernel let it start only after
    // its own wait.  (The sharded form follows an exchange and waits at once.)
    if (SHARDED) grid_dependency_wait();
    const int nloop = PRECISE ? *a.queue_count : a.B;
    for (int slot = blockIdx.x; slot < nloop; slot += gridDim.x) verify_finish_slot<T, PRECISE, SHARDED, HELD>(a, slot, sh, cm);
    grid_dependency_sync();
}

}  // namespace picospec
