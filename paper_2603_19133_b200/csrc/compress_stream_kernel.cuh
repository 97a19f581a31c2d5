// Draft-side compression, staged variant: rows that hold at least one full tile.  Two kernels.
//
// compress_filter_kernel streams the rows (one CTA per row at a time, in tiles of 8 chunks, one per
// warp, staged in shared memory by bulk async copies; the producer lanes run ahead into the next row)
// and keeps every element that can still be among the k largest:
//   - the CTA holds a running bound `thr` below which elements are dropped (how it is chosen, and which
//     chunks make a tile: bound_rank);
//   - per chunk a lane compares its 32 values with thr (packed compares for bf16) into a 32-bit
//     mask and appends the passing values (64-bit keys: logit, then lower index first; the value is
//     re-read from the staged tile) to the warp's own region of the candidate buffer;
//   - every stored candidate is counted in a two-level histogram whose bins count up from the
//     first tile's bound, one bin per 16-bit logit code (the top 16 bits of the orderable key: a
//     bf16 value, 2^-7 relative for fp32), magnitudes below 2^-10 sharing one bin on each side of
//     zero so that a window that crosses zero does not spend itself on tiny exponents; 4096 bins
//     reach 32 binades up, whatever lies beyond shares the last bin; thr is the lower edge of the
//     highest bin whose suffix count reaches the wanted rank.
//     One warp or another refreshes it, after ever more tiles;
//   - the first tile of a row gets its bound without the histogram: every warp finds a value that its
//     share of the wanted rank of small groups of its elements reach with their maximum; the smallest of
//     the eight values, or the third smallest with a larger share, is reached by the wanted rank of
//     elements (one CTA barrier, the only one of a row);
//   - a chunk of which too much passes goes a slower way (crowded_chunk);
//   - a row whose candidates do not fit (heavy ties), or whose bound rose past its k-th largest, is
//     handed to the direct kernel through a redo list;
//   - with top-p the same pass accumulates the softmax normaliser relative to the first tile's
//     maximum (a row whose later logits overflow that reference also goes to the redo list).
// At the end of a row every warp writes its candidates at or above thr to a per-row scratch area in global memory
// (thr was refreshed last after two thirds of the row or more: about 1.4 k of them), which gets the bound as it is
// when all have.
//
// compress_finish_kernel (a warp or a CTA per row) selects the k best of them and puts them in order
// with a counting sort over the 16-bit logit codes, then calls finish_row (top-p cut,
// renormalisation, emission, draft draw).
#pragma once
#include "compress_kernels.cuh"


#include "stream_pipeline.cuh"

namespace picospec {

// Two shapes of the filter kernel, both sized for three CTAs per SM on 16-bit rows (the kernel is
// bound by instruction issue, so resident warps count for more than tiles in flight: two stages
// measure the same as three, three CTAs 15 % faster than two).  Rows with k <= 512 need few live
// candidates: a small candidate buffer; larger k takes the big buffer.  32-bit rows have 32 KB tiles:
// two CTAs per SM in both shapes.  With spread tiles a region that is full empties itself into the scratch area, and
// the big buffer gives a quarter of its keys to a second histogram.  Without (k > 512: rows of at most two tiles) it
// keeps them, a row whose regions overflow being lost to the direct kernel: with 3072 keys all of 60 rows of 16384 entries
// (k = 1024, a third of them below index 1024) went there, with 4096 none.
constexpr int CS_CAP_SMALL = 2048, CS_CAP_LARGE = 4096, CS_CAP_LARGE_SPREAD = 3072;    // candidate keys held in shared memory
constexpr int CS_K_SMALL = 512;                            // largest k served by the small shape
constexpr int CS_BINS = 4096;        // histogram bins above the first tile's bound; the last one is open-ended
constexpr int CS_DEAD = 117 << 7;    // 16-bit magnitude codes below 2^-10: one bin on each side of zero
constexpr int CS_SUPER = CS_BINS / 32;
// Bin counts are 16 bits wide, two per word (super-bin counts are 32-bit).  A count can only wrap
// on rows that push tens of thousands of values into one bin; a wrap makes a sum too small (a
// lower, still valid bound) and its carry makes the neighbouring bin one too large, which can at
// worst leave fewer than k survivors: such a row goes to the redo list.
constexpr int CS_HIST_WORDS = CS_BINS / 2 + CS_SUPER;

// row flags written by the filter kernel
constexpr int CSF_TEMPERATURE = 1, CSF_LOGIT = 2, CSF_REDO = 4, CSF_ABORT = 8, CSF_RANGE = 16;

struct CsRowMeta {
    int count;        // survivors written for the row
    int flags;
    float ref_off;    // fp32(ref * c32): reference of the streamed normaliser
    unsigned thr_key; // the piece's last bound: every entry of it whose orderable logit is at least this is a survivor
    int top;          // bin coordinate of the largest survivor
    double z_stream;  // sum of 2^(l * c32 - ref_off) over the row (top-p only)
};

// capacity of a row's scratch area (keys) for a sparse-row capacity k_max: twice what a row leaves there on average
// (a bound refreshed last after 69 % of the row, as it is for 23 tiles, lets 1.45 k through)
__host__ __device__ __forceinline__ int cs_survivor_cap(int k_max) { return 3 * k_max > 512 ? 3 * k_max : 512; }

struct __align__(8) CsShared {
    unsigned thr_key;   // orderable form of the current lower bound on the k-th largest logit
    unsigned certain;   // counts are no longer capped (crowded_chunk): only k of them make a bound
    unsigned first_key[WARPS];  // the warps' own bounds of the first tile
    unsigned first_max[WARPS];  // the warps' largest orderable logits of the first tile (STATS)
    int g0;             // bin coordinate of the first tile's bound: origin of the histogram
    int area;           // scratch area of the piece
    int seen;           // chunks whose entries are counted, or are being counted
    int overflow;       // the scratch area ran out of room: the row goes to the redo list
    int nan;
    int m;              // survivors written
    unsigned top;       // 16-bit code of the largest of them
    int flags;          // CSF_TEMPERATURE / CSF_RANGE, known when the piece begins
    float ref_off;
    double wsum[WARPS];
};
// state of the CTA that outlives a piece
struct CsCta {
    int abort;          // a bounded wait ran out somewhere in the CTA
    int k, surv_cap, quota;     // as in FilterBound
    u64* surv_keys;
    int wcnt[WARPS];    // per warp: entries in its region (the slot counter its lanes draw from)
    int2 arg[WARPS];    // per warp: what crowded_chunk takes besides its arguments (chunk's offset, its first index)
};
// bf16: 2 stages x 16 KB, 66 KB SMALL, 74 KB LARGE (3 CTAs / SM).  fp32: 2 stages x 32 KB, 98 / 106 KB (2 CTAs / SM).
template <typename T, bool SMALL, bool SPREAD> struct CsGeom {
    static constexpr int CAP = SMALL ? CS_CAP_SMALL : SPREAD ? CS_CAP_LARGE_SPREAD : CS_CAP_LARGE;
    static constexpr int REGION = CAP / WARPS;             // each worker warp appends to its own region
    static constexpr int TIES = SMALL ? 128 : 256;         // of one code in a chunk (crowded_chunk): hopeless
    static constexpr int HISTS = SMALL || SPREAD ? 2 : 1;  // copies of the histogram
    static constexpr int STAGES = 2;
    static constexpr int CTAS = sizeof(T) == 2 ? 3 : 2;
    static constexpr int TILE_BYTES = TILE_CHUNKS * CHUNK * (int)sizeof(T);
    static constexpr int STAGE_BYTES = STAGES * TILE_BYTES;
    static constexpr int HIST_OFF = STAGE_BYTES + CAP * 8;
    static constexpr int SHARED_OFF = HIST_OFF + HISTS * CS_HIST_WORDS * 4;    // CsShared[2], CsCta
    static constexpr int SMEM_BYTES = SHARED_OFF + 2 * (int)sizeof(CsShared) + (int)sizeof(CsCta);
    __device__ static __forceinline__ unsigned* hist(unsigned char* dyn, int copy) {
        return reinterpret_cast<unsigned*>(dyn + HIST_OFF) + (HISTS == 2 ? copy * CS_HIST_WORDS : 0);
    }
};

__device__ __forceinline__ void cs_reset(CsShared& cs) {
    cs.thr_key = 0u;
    cs.certain = 0u;
    cs.seen = 0;
    cs.top = 0u;
    cs.overflow = 0;
    cs.nan = 0;
    cs.m = 0;
}

// ---- per-dtype pieces --------------------------------------------------------------------------

// 32-bit mask of the lane's values that are >= thr (NaN never passes).
//   bf16: bit k = low half of word k, bit 16 + k = high half of word k.  The packed threshold is
//         the smallest bf16 >= thr for every threshold this kernel produces (a bf16 value itself,
//         or the lower edge of a histogram bin: positive edges are bf16 values, negative edges
//         have all low bits set, so dropping them rounds towards zero, i.e. up).
//   fp32: bit k = value k.
__device__ __forceinline__ unsigned pass_mask(const ChunkRegs<__nv_bfloat16>& r, float thr) {
    const uint32_t h = __float_as_uint(thr) >> 16;
    const uint32_t t2 = h | (h << 16);
    const __nv_bfloat162 t = *reinterpret_cast<const __nv_bfloat162*>(&t2);
    unsigned mask = 0;
#pragma unroll
    for (int k = 0; k < 16; ++k)
        mask |= __hge2_mask(*reinterpret_cast<const __nv_bfloat162*>(&r.w[k]), t) & (0x00010001u << k);
    return mask;
}
__device__ __forceinline__ unsigned pass_mask(const ChunkRegs<float>& r, float thr) {
    unsigned mask = 0;
#pragma unroll
    for (int k = 0; k < 32; ++k) mask |= (r.f[k] >= thr ? 1u : 0u) << k;
    return mask;
}
// offset inside the chunk (in elements) of the value behind mask bit b of a lane
__device__ __forceinline__ int bit_offset(int b, int lane, const __nv_bfloat16*) {
    const int k = b & 15;
    return (k >> 2) * 256 + lane * 8 + (k & 3) * 2 + (b >> 4);
}
__device__ __forceinline__ int bit_offset(int b, int lane, const float*) { return (b >> 2) * 128 + lane * 4 + (b & 3); }
// value at an element offset of a staged chunk
__device__ __forceinline__ float staged_value(const unsigned char* chunk, int off, const __nv_bfloat16*) {
    return __uint_as_float((uint32_t)reinterpret_cast<const unsigned short*>(chunk)[off] << 16);
}
__device__ __forceinline__ float staged_value(const unsigned char* chunk, int off, const float*) {
    return reinterpret_cast<const float*>(chunk)[off];
}

// 16-bit orderable keys of the maxima of groups of 2 consecutive elements of the lane's chunk
// (NaN is ignored here).
__device__ __forceinline__ void pair_keys(const ChunkRegs<__nv_bfloat16>& r, unsigned (&key)[16]) {
#pragma unroll
    for (int k = 0; k < 16; ++k)
        key[k] = orderable(fmaxf(__uint_as_float(r.w[k] << 16), __uint_as_float(r.w[k] & 0xffff0000u))) >> 16;
}
__device__ __forceinline__ void pair_keys(const ChunkRegs<float>& r, unsigned (&key)[16]) {
#pragma unroll
    for (int k = 0; k < 16; ++k) key[k] = orderable(fmaxf(r.f[2 * k], r.f[2 * k + 1])) >> 16;
}

// Warp-wide search, two bits per step: the largest 16-bit key t such that at least `need` of the
// warp's G*32 group keys are >= t (the need-th largest key).  G in {4, 8, 16} keys per lane.
template <int G>
__device__ __forceinline__ unsigned warp_kth_key(const unsigned (&key)[16], int need) {
    unsigned prefix = 0;
#pragma unroll 1
    for (int bit = 14; bit >= 0; bit -= 2) {
        const unsigned t1 = prefix | (1u << bit), t2 = prefix | (2u << bit), t3 = prefix | (3u << bit);
        int c1 = 0, c2 = 0, c3 = 0;
#pragma unroll
        for (int x = 0; x < G; ++x) {
            c1 += key[x] >= t1 ? 1 : 0;
            c2 += key[x] >= t2 ? 1 : 0;
            c3 += key[x] >= t3 ? 1 : 0;
        }
        c1 = __reduce_add_sync(0xffffffffu, c1);
        c2 = __reduce_add_sync(0xffffffffu, c2);
        c3 = __reduce_add_sync(0xffffffffu, c3);
        prefix = c3 >= need ? t3 : c2 >= need ? t2 : c1 >= need ? t1 : prefix;
    }
    return prefix;
}

// First-tile bound of one warp: group size g (elements) in {2, 4, 8 (bf16 only)}.  (Inlined: an
// out-of-line call would force the chunk registers through local memory in every tile.)
template <typename T>
__device__ __forceinline__ unsigned first_tile_key(const ChunkRegs<T>& regs, int g, int need) {
    unsigned key[16];
    if (g == ChunkRegs<T>::VEC) {
        // groups = the lane's 16-byte vectors: their maxima come packed
        constexpr int NV = ChunkRegs<T>::NVEC;
#pragma unroll
        for (int j = 0; j < NV; ++j) key[j] = orderable(regs.vec_max(j)) >> 16;
        return warp_kth_key<NV>(key, need);
    }
    pair_keys(regs, key);
    if (g == 2) return warp_kth_key<16>(key, need);
#pragma unroll
    for (int x = 0; x < 8; ++x) key[x] = max(key[2 * x], key[2 * x + 1]);
    if (g == 4) return warp_kth_key<8>(key, need);
#pragma unroll
    for (int x = 0; x < 4; ++x) key[x] = max(key[2 * x], key[2 * x + 1]);
    return warp_kth_key<4>(key, need);
}

// two-level histogram update
// Bin coordinate of a 16-bit orderable code (monotone): the code itself with the magnitudes
// below 2^-10 squeezed onto 0x7FFF (negative side) and 0x8000 (positive side).
__device__ __forceinline__ int bin_coord(unsigned o16) {
    const bool pos = o16 >= 0x8000u;
    const int mag = pos ? (int)o16 - 0x8000 : 0x7FFF - (int)o16;
    const int c = max(mag - CS_DEAD, 0);
    return pos ? 0x8000 + c : 0x7FFF - c;
}
// smallest 16-bit code whose coordinate is at least G
__device__ __forceinline__ unsigned coord_code(int G) {
    if (G >= 0x8000) {
        const int c = G - 0x8000;
        return (unsigned)(c ? 0x8000 + c + CS_DEAD : 0x8000);
    }
    return (unsigned)(0x7FFF - ((0x7FFF - G) + CS_DEAD));
}
// bin of an orderable key at or above the bound whose coordinate is g0, the last one open-ended
__device__ __forceinline__ int hist_bin(unsigned okey, int g0) { return min(bin_coord(okey >> 16) - g0, CS_BINS - 1); }
__device__ __forceinline__ void hist_add(unsigned* hist, int bin) {
    atomicAdd(&hist[bin >> 1], (bin & 1) ? 0x10000u : 1u);
    atomicAdd(&hist[CS_BINS / 2 + (bin >> 5)], 1u);
}

// One warp: the highest bin whose suffix count (itself and every bin above it) reaches k, or -1 if
// fewer than k values have been counted.
__device__ __forceinline__ int kth_bin(const unsigned* hist, int k, int lane) {
    // level 1: lane l owns super-bins 4l .. 4l+3 (super-bin s covers bins 32 s .. 32 s + 31)
    const uint4 sv = *reinterpret_cast<const uint4*>(&hist[CS_BINS / 2 + 4 * lane]);
    const unsigned own = sv.x + sv.y + sv.z + sv.w;
    unsigned suf = own;             // inclusive suffix sum over lanes (higher lanes = higher bins)
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned y = __shfl_down_sync(0xffffffffu, suf, d);
        if (lane + d < 32) suf += y;
    }
    const unsigned hit = __ballot_sync(0xffffffffu, suf >= (unsigned)k);
    if (!hit) return -1;            // fewer than k counted so far
    const int L = 31 - __clz(hit);  // highest lane whose suffix reaches k
    unsigned above = __shfl_sync(0xffffffffu, suf - own, L);      // count strictly above lane L's super-bins
    const uint4 lv = make_uint4(__shfl_sync(0xffffffffu, sv.x, L), __shfl_sync(0xffffffffu, sv.y, L),
                                __shfl_sync(0xffffffffu, sv.z, L), __shfl_sync(0xffffffffu, sv.w, L));
    int s = 4 * L + 3;
    if (above + lv.w < (unsigned)k) {
        above += lv.w;
        s = 4 * L + 2;
        if (above + lv.z < (unsigned)k) {
            above += lv.z;
            s = 4 * L + 1;
            if (above + lv.y < (unsigned)k) {
                above += lv.y;
                s = 4 * L;
            }
        }
    }
    // level 2: the 32 bins of super-bin s, lane l reads bin 32 s + l
    unsigned bs = (hist[16 * s + (lane >> 1)] >> ((lane & 1) * 16)) & 0xffffu;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned y = __shfl_down_sync(0xffffffffu, bs, d);
        if (lane + d < 32) bs += y;
    }
    const unsigned hit2 = __ballot_sync(0xffffffffu, above + bs >= (unsigned)k);
    return hit2 ? 32 * s + (31 - __clz(hit2)) : 32 * s;
}

// One warp: raise thr to the lower edge of the highest bin whose suffix count reaches `rank` (or k, if
// counts that are not capped may be among those read: the flag is set before the first of them is added).
__device__ __forceinline__ void refresh_threshold(const unsigned* hist, CsShared& cs, int rank, int k, int lane) {
    int found = kth_bin(hist, rank, lane);
    if (rank < k) {
        __threadfence_block();
        if (__any_sync(0xffffffffu, *(volatile unsigned*)&cs.certain)) found = kth_bin(hist, k, lane);
    }
    if (found >= 0 && lane == 0) atomicMax(&cs.thr_key, coord_code(*(volatile int*)&cs.g0 + found) << 16);
}

// A candidate's low word is ~index, whose top bit is set; cleared, it marks an entry that is not counted yet.
constexpr u64 CS_COUNTED = 0x80000000ull;
// One warp: count the entries of its region that are not counted yet.
__device__ __forceinline__ void count_marked(unsigned* hist, u64* region, int n, int g0, int lane) {
    for (int x = lane; x < n; x += 32) {
        const u64 key = region[x];
        if (!(key & CS_COUNTED)) {
            region[x] = key | CS_COUNTED;
            hist_add(hist, hist_bin((unsigned)(key >> 32), g0));
        }
    }
    __syncwarp();
}

// Warp-local: drop the entries of this warp's region below thr (stable, in place).
__device__ __forceinline__ int compact_region(u64* region, int n, unsigned thr_key, int lane) {
    int out = 0;
    for (int base = 0; base < n; base += 32) {
        const int i = base + lane;
        const u64 key = i < n ? region[i] : 0ull;
        const bool keep = i < n && (unsigned)(key >> 32) >= thr_key;
        const unsigned m = __ballot_sync(0xffffffffu, keep);
        if (keep) region[out + __popc(m & ((1u << lane) - 1u))] = key;
        out += __popc(m);
    }
    __syncwarp();
    return out;
}

// The out-of-line functions find the shared state by its place in the dynamic shared memory (`copy`: which of
// the two of the per-piece state): every argument is a register that is live in the kernel's loop.
// Refresh the bound (one warp; out of line).
template <typename Geom> __device__ __noinline__ void refresh_bound(int copy, int rank, int k) {
    extern __shared__ __align__(1024) unsigned char dyn[];
    CsShared& cs = reinterpret_cast<CsShared*>(dyn + Geom::SHARED_OFF)[copy];
    refresh_threshold(Geom::hist(dyn, copy), cs, rank, k, threadIdx.x & 31);
}
// First tile of a piece: the bound is the NTH smallest of the warps' own (one warp, every warp with the same
// result; out of line).  Returns the largest orderable logit of the tile (STATS).
template <typename Geom, int NTH> __device__ __noinline__ unsigned first_bound(int copy, int area) {
    extern __shared__ __align__(1024) unsigned char dyn[];
    CsShared* cs = reinterpret_cast<CsShared*>(dyn + Geom::SHARED_OFF) + copy;
    const int lane = threadIdx.x & 31;
    // (the lane number makes the keys distinct)
    unsigned key = lane < WARPS ? *(volatile unsigned*)&cs->first_key[lane] | lane : 0xffffffffu;
    unsigned bound = __reduce_min_sync(0xffffffffu, key);
#pragma unroll
    for (int x = 1; x < NTH; ++x) {
        if (key == bound) key = 0xffffffffu;
        bound = __reduce_min_sync(0xffffffffu, key);
    }
    bound &= 0xffff0000u;
    if (lane == 0) {
        *(volatile int*)&cs->g0 = bin_coord(bound >> 16);
        *(volatile int*)&cs->area = area;
        atomicMax(&cs->thr_key, bound);
    }
    __syncwarp();
    return __reduce_max_sync(0xffffffffu, lane < WARPS ? *(volatile unsigned*)&cs->first_max[lane] : 0u);
}
// End of a piece, a warp: its entries at or above the bound go to the piece's scratch area (out of line).
template <typename Geom> __device__ __noinline__ void hand_over(int copy, int n) {
    extern __shared__ __align__(1024) unsigned char dyn[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    CsShared* cs = reinterpret_cast<CsShared*>(dyn + Geom::SHARED_OFF) + copy;
    const CsCta* cta = reinterpret_cast<const CsCta*>(dyn + Geom::SHARED_OFF + 2 * sizeof(CsShared));
    const u64* region = reinterpret_cast<const u64*>(dyn + Geom::STAGE_BYTES) + warp * Geom::REGION;
    const int surv_cap = cta->surv_cap;
    u64* dst = cta->surv_keys + (long long)*(volatile int*)&cs->area * surv_cap;
    const unsigned thr_key = __shfl_sync(0xffffffffu, *(volatile unsigned*)&cs->thr_key, 0);
    unsigned top = 0u;
    for (int x0 = 0; x0 < n; x0 += 32) {
        const u64 key = x0 + lane < n ? region[x0 + lane] : 0ull;
        const unsigned okey = (unsigned)(key >> 32);
        const unsigned keep = __ballot_sync(0xffffffffu, okey >= thr_key);      // (thr_key > 0: no empty slot)
        int base = 0;
        if (lane == 0) base = atomicAdd(&cs->m, __popc(keep));
        base = __shfl_sync(0xffffffffu, base, 0) + __popc(keep & ((1u << lane) - 1u));
        if (okey >= thr_key && base < surv_cap) dst[base] = key | CS_COUNTED;
        top = max(top, okey);
    }
    top = __reduce_max_sync(0xffffffffu, top) >> 16;
    if (lane == 0) atomicMax(&cs->top, top);
    __syncwarp();
}
// orderable form of a staged value (-0 becomes +0)
template <typename T> __device__ __forceinline__ uint32_t staged_key(const unsigned char* chunk, int off) {
    const uint32_t bits = __float_as_uint(staged_value(chunk, off, (const T*)nullptr) + 0.0f);
    return bits ^ ((uint32_t)((int32_t)bits >> 31) | 0x80000000u);
}
// A chunk of which more passes (`mask` per lane) than it may count with, or than the warp's region (n entries)
// has room for (one warp; out of line).
//   - If there is room, as many as the quota are counted, the others are marked.
//   - Else the bound is brought up to date and what falls below it is dropped.  With spread tiles all that
//     the warp holds is counted before, the chunk's values included, so that k of them make a bound that
//     is certain and as high as the counts allow; and if the rest still does not fit, the region is emptied
//     into the piece's scratch area, and the chunk's values follow if they are more than the region holds.
// Returns the entries in the region, or -1: the row goes to the direct kernel.
template <typename T, typename Geom, bool SPREAD>
__device__ __noinline__ int crowded_chunk(unsigned mask, int n, int copy) {
    extern __shared__ __align__(1024) unsigned char dyn[];
    constexpr int REGION = Geom::REGION;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    CsShared* cs = reinterpret_cast<CsShared*>(dyn + Geom::SHARED_OFF) + copy;
    CsCta* cta = reinterpret_cast<CsCta*>(dyn + Geom::SHARED_OFF + 2 * sizeof(CsShared));
    const unsigned char* chunk = dyn + cta->arg[warp].x;
    const int vchunk = cta->arg[warp].y;
    unsigned* hist = Geom::hist(dyn, copy);
    u64* region = reinterpret_cast<u64*>(dyn + Geom::STAGE_BYTES) + warp * REGION;
    u64* to = region;
    int* wcnt = &cta->wcnt[warp];
    const int g0 = *(volatile int*)&cs->g0, k = cta->k;
    int own = __popc(mask), added = __reduce_add_sync(0xffffffffu, own);
    int held = n;                   // slots taken at `to`
    int count = 0;                  // entries of the chunk that are counted below
    if (n + added <= REGION) {
        const bool certain = __any_sync(0xffffffffu, *(volatile unsigned*)&cs->certain);
        count = certain ? added : cta->quota;
    } else if (!SPREAD) {
        refresh_threshold(hist, *cs, k, k, lane);
        __syncwarp();
    } else {
        // Values that share the bound's own 16-bit code cannot be told apart by any bound: if, behind the first
        // tile, a chunk holds TIES of them, or if another warp has given up, so does this one.
        const unsigned code = *(volatile unsigned*)&cs->thr_key >> 16;
        int same = 0;
        for (unsigned m = mask; m; m &= m - 1u)
            same += staged_key<T>(chunk, bit_offset(__ffs(m) - 1, lane, (const T*)nullptr)) >> 16 == code ? 1 : 0;
        __syncwarp();
        same = __reduce_add_sync(0xffffffffu, same);
        if ((same > Geom::TIES && __any_sync(0xffffffffu, *(volatile int*)&cs->seen > WARPS)) ||
            __any_sync(0xffffffffu, *(volatile int*)&cs->overflow))
            return -1;
        if (lane == 0) *(volatile unsigned*)&cs->certain = 1u;
        __threadfence_block();
        __syncwarp();
        count_marked(hist, region, n, g0, lane);
        for (unsigned m = mask; m; m &= m - 1u)
            hist_add(hist, hist_bin(staged_key<T>(chunk, bit_offset(__ffs(m) - 1, lane, (const T*)nullptr)), g0));
        __syncwarp();
        refresh_threshold(hist, *cs, k, k, lane);
        __syncwarp();
    }
    if (n + added > REGION) {
        const unsigned thr_key = __shfl_sync(0xffffffffu, *(volatile unsigned*)&cs->thr_key, 0);
        held = n = compact_region(region, n, thr_key, lane);
        unsigned left = 0u;
        for (unsigned m = mask; m; m &= m - 1u)
            if (staged_key<T>(chunk, bit_offset(__ffs(m) - 1, lane, (const T*)nullptr)) >= thr_key) left |= m & (0u - m);
        __syncwarp();
        mask = left;
        own = __popc(mask);
        added = __reduce_add_sync(0xffffffffu, own);
        if (!SPREAD) count = added;
        if (n + added > REGION) {
            if (!SPREAD) return -1;
            const bool direct = added > REGION;
            const int spilled = n + (direct ? added : 0), surv_cap = cta->surv_cap;
            int base = 0;
            if (lane == 0) base = atomicAdd(&cs->m, spilled);
            base = __shfl_sync(0xffffffffu, base, 0);
            if (base + spilled > surv_cap) return -1;
            u64* dst = cta->surv_keys + (long long)cs->area * surv_cap + base;
            for (int x = lane; x < n; x += 32) dst[x] = region[x];
            held = direct ? n : 0;
            if (direct) to = dst;
        }
        __syncwarp();
        if (lane == 0) *wcnt = held;
        __syncwarp();
    }
    int pos = atomicAdd(wcnt, own);
    for (; mask; mask &= mask - 1u) {
        const int off = bit_offset(__ffs(mask) - 1, lane, (const T*)nullptr);
        const uint32_t okey = staged_key<T>(chunk, off);
        u64 key = ((u64)okey << 32) | (u64)(~(uint32_t)(vchunk + off));
        if (pos - held < count) hist_add(hist, hist_bin(okey, g0));
        else if (count) key &= ~CS_COUNTED;
        to[pos++] = key;
    }
    __syncwarp();
    if (to == region) return held + added;
    if (lane == 0) *wcnt = 0;
    __syncwarp();
    return 0;
}

// ---- how the rows of a call are dealt to the CTAs of the filter kernel ----------------------------
// With rows = q * grid + rem, CTA b first takes the q whole rows b, b + grid, ... (so that at any time
// the CTAs read one window of memory that moves forward, as a copy would).  The rem rows that
// are left would keep only some of the CTAs busy for a whole row's time, so each of them is cut into
// `split` pieces of consecutive tiles and the rem * split pieces are dealt round-robin: piece n goes
// to CTA n % grid.  A piece is filtered on its own, with the bound of its share of the row
// (bound_rank), and leaves its survivors in its own scratch area (whole row r: area r; tail piece n:
// area rows + n).  The finish kernel puts the pieces of a row together.
// No piece starts at a row's last tile when that tile is ragged (the first tile of a piece must be a
// full one, up to the few entries that a row's offset from a 16-byte boundary takes from it).
struct FilterPlan {
    int tiles_per_row;
    int ragged_last;        // the last tile of a row holds fewer than TILE_CHUNKS full chunks
    int grid;               // CTAs of the filter kernel
    int rows;
    int q;                  // whole rows per CTA
    int rem;                // rows dealt in pieces: rows q * grid .. rows - 1
    int split;              // pieces per such row
};
// first tile of piece p (0 .. split) of a split row
__host__ __device__ __forceinline__ int plan_piece_tile(const FilterPlan& p, int piece) {
    int c = p.tiles_per_row * piece / p.split;
    if (p.ragged_last && p.tiles_per_row > 1 && c < p.tiles_per_row && c == p.tiles_per_row - 1) --c;
    return c;
}
// The k-th unit of work of CTA b: a whole row or a piece of a tail row.  false: no more work.
struct FilterPiece {
    int row, tile0, tile1, area;
};
__host__ __device__ __forceinline__ bool plan_piece(const FilterPlan& p, int b, int k, FilterPiece& out) {
    if (k < p.q) {
        out.row = k * p.grid + b;      // the CTAs advance through memory side by side
        out.tile0 = 0;
        out.tile1 = p.tiles_per_row;
        out.area = out.row;
        return true;
    }
    const long long n = (long long)b + (long long)(k - p.q) * p.grid;
    if (n >= (long long)p.rem * p.split) return false;
    const int j = (int)(n / p.split), pc = (int)(n - (long long)j * p.split);
    out.row = p.q * p.grid + j;
    out.tile0 = plan_piece_tile(p, pc);
    out.tile1 = plan_piece_tile(p, pc + 1);
    out.area = p.rows + (int)n;
    return true;        // (tile0 == tile1: an empty piece, skipped by everyone)
}
// Host side: the plan for `rows` rows on `slots` resident CTAs.  Rows are cut only when a CTA gets at most
// one whole row (few rows per CTA: the remainder decides the kernel's length); the split is then the one
// that shortens the tail most among those that keep a piece at least two tiles long and the number of
// pieces within 2 * grid (the scratch areas are sized for that).
inline FilterPlan make_filter_plan(int rows, int tiles_per_row, bool ragged_last, long long slots) {
    FilterPlan p;
    p.tiles_per_row = tiles_per_row;
    p.ragged_last = ragged_last ? 1 : 0;
    p.rows = rows;
    long long g = slots < 1 ? 1 : slots;
    const long long most = (long long)rows * (tiles_per_row >= 2 ? tiles_per_row / 2 : 1);   // pieces of two tiles
    if (g > most) g = most;
    if (g < 1) g = 1;
    p.grid = (int)g;
    p.q = (int)(rows / g);
    p.rem = (int)(rows - (long long)p.q * g);
    p.split = 1;
    // Pieces pay the per-piece work (first-tile bound, hand-over) again; that is worth it only while
    // the remainder is a large part of what a CTA does.
    if (p.rem > 0 && p.q <= 1) {
        double best = 1e9;
        const int smax = tiles_per_row >= 2 ? tiles_per_row / 2 : 1;
        for (int sp = 1; sp <= 8 && sp <= smax && (long long)p.rem * sp <= 2 * g; ++sp) {
            const long long per_cta = ((long long)p.rem * sp + g - 1) / g;      // pieces the busiest CTA gets
            const double cost = (double)per_cta / sp;
            if (cost < best - 1e-9) {
                best = cost;
                p.split = sp;
            }
        }
    }
    return p;
}

// ---- how far a bound may reach ahead -------------------------------------------------------------
// A bound that k elements seen so far reach is certain, but while little of the row has been seen it
// lets k / (tiles seen) elements of every tile pass, k (1 + ln tiles) in all, and handling those was most
// of the kernel's instructions at large k.  The bound used is the value that
//     rank(f) = 1.5 k f + 5 sqrt(1.5 k f) + 12        (at most k)
// of the elements seen reach, f being the fraction of the row that has been seen: were the k largest spread
// evenly over the tiles, it would be lower than the k-th largest by a factor 1.5 and five standard
// deviations in the count.
// They are not: vocabularies have an order (frequent pieces first, languages and unused ids in blocks).
// A tile takes one chunk from each eighth of the row, so that each eighth is seen to the same fraction, and
//   - no chunk counts with more than a quarter of the first tile's rank and eight (chunk_quota; the entries
//     beyond it are marked and counted only if a region runs full): a crowded place cannot lift the bound above
//     what three quarters of the rank reach elsewhere, which is still 1.125 k f and more;
//   - the first tile's bound is the third smallest of the warps' own, a sixth of the rank each: it is neither
//     lifted by five crowded chunks nor dropped by two empty ones (an unused end of the vocabulary);
//   - eighth e is streamed by warp (e + tile) % 8, so that a crowded eighth does not fill one warp's region;
//   - a region that is too full makes the rest of the row go by certain bounds, and empties itself into
//     the row's scratch area if need be (crowded_chunk).
// It is not certain; it is checked: every element dropped was below the final bound, so the row is right if
// k survivors reach that, and goes to the direct kernel if not.  Against certain bounds throughout, compress
// takes 156 instead of 217 us for 1024 rows of 262144 entries (k = 1024) and 156 instead of 170 for 1536 rows
// of 128256 (top-p, k = 256) where the large logits lie evenly, 167 instead of 215 and 158 instead of 169 with a
// quarter of the k largest below index 1024.  (Without the precautions all rows of those two went to the
// direct kernel: 726 and 662 us.)
__host__ __device__ __forceinline__ int open_rank(int k, float f) {
    const float e = 1.5f * (float)k * f;
    return (int)(e + 5.0f * sqrtf(e)) + 12;
}
__host__ __device__ __forceinline__ int bound_rank(int k, float f) {
    const int r = open_rank(k, f);
    return r < k ? r : k;
}
// what one chunk may count with
__host__ __device__ __forceinline__ int chunk_quota(int k, float per_tile) { return (open_rank(k, per_tile) + 3) / 4 + 8; }
// Where one tile's rank is k already (small k) the tiles are contiguous instead: one copy of 16 KB a tile
// (4096 rows of 32000 entries, k = 8: 69 us against 75 us with eight copies of 2 KB).
// (Rows of two tiles: too few of the eighths may have a chunk in the first.)
__host__ __device__ __forceinline__ bool bound_spreads(int k, int tiles) { return tiles > 2 && bound_rank(k, 1.0f / (float)tiles) < k; }
// What the kernel needs of all this, worked out once per call (in the constant bank: no registers).
struct FilterBound {
    int k;                  // entries wanted of a row
    int surv_cap;           // keys in a scratch area
    bool spread;            // a tile takes a chunk from each eighth of the row (chunks [e, e + 1) * tiles), not eight consecutive
                            // ones; chunk `tile` of eighth e is streamed by warp (e + tile) % 8
    float per_tile, per_chunk;  // fractions of a row
    int need, group;        // first tile: elements that a warp's own bound is reached by, elements per group of its search
    int quota;              // chunk_quota
};
inline FilterBound make_filter_bound(int k, int k_max, int nch, int vec) {
    FilterBound f;
    f.k = k;
    f.surv_cap = cs_survivor_cap(k_max);
    // (the fewest tiles that a row of V entries takes: a fraction that is too large only makes a bound lower)
    const int tiles = (nch + TILE_CHUNKS - 1) / TILE_CHUNKS;
    f.per_tile = 1.0f / (float)tiles;
    f.per_chunk = f.per_tile / (float)TILE_CHUNKS;
    f.spread = bound_spreads(k, tiles);
    // First tile: up to 16 elements per warp from the lane maxima.  Beyond (a k that is large for the row)
    // the exact need-th largest maximum of groups of elements, at least 4 rank groups in the tile (cheaper
    // bounds from lane maxima or lane pairs let 10 to 25 % of a tile pass: the extra candidates cost
    // more than the search).
    const int rank1 = f.spread ? bound_rank(k, f.per_tile) : k;
    f.need = f.spread ? (rank1 + 5) / 6 : (rank1 + WARPS - 1) / WARPS;
    f.group = vec;
    while (f.group > 2 && (TILE_CHUNKS * CHUNK) / f.group < 4 * rank1) f.group >>= 1;
    f.quota = f.spread ? chunk_quota(k, f.per_tile) : CHUNK;
    return f;
}

// First-tile bound of one warp when it needs at most 16 elements: the need-th largest of its 32 lanes'
// maxima, as a 16-bit orderable code (rounded down).  (The smallest of the maxima of `need` groups of
// lanes is cheaper and also certain, but now and then so low that a fifth of the tile passes and a
// warp's region overflows: one row in five thousand at need = 15.)
__device__ __forceinline__ unsigned first_tile_key_lanes(float lane_max, int need) {
    const unsigned key = orderable(lane_max) >> 16;
    if (need == 1) return __reduce_max_sync(0xffffffffu, key);
    unsigned prefix = 0u;
#pragma unroll 4
    for (int bit = 15; bit >= 0; --bit) {
        const unsigned t = prefix | (1u << bit);
        if (__popc(__ballot_sync(0xffffffffu, key >= t)) >= need) prefix = t;
    }
    return prefix;
}

// SPREAD: bound_spreads for the call's rows
template <typename T, bool STATS, bool SMALL, bool SPREAD>
__global__ void __launch_bounds__(STREAM_THREADS, CsGeom<T, SMALL, SPREAD>::CTAS)
compress_filter_kernel(CompressArgs a, FilterPlan plan, FilterBound fb, unsigned long long wait_limit_ns) {
    extern __shared__ __align__(1024) unsigned char dyn[];
    typedef CsGeom<T, SMALL, SPREAD> Geom;
    constexpr int STAGES = Geom::STAGES;
    constexpr int TILE_BYTES = Geom::TILE_BYTES;
    constexpr int CS_CAND_CAP = Geom::CAP, CS_REGION = Geom::REGION;
    unsigned char* stage_mem = dyn;
    u64* cand = reinterpret_cast<u64*>(dyn + Geom::STAGE_BYTES);
    __shared__ __align__(8) uint64_t full[STAGES], empty[STAGES];
    // Two copies of the per-piece state and of the histogram, used in turn, so that a piece has one barrier, that
    // of its first tile: behind it every warp is done with the piece before, whose record is written and whose copies
    // are cleared there.  (With three barriers a piece, a last exact bound and one histogram the kernel took 70.8 us for
    // 4096 rows of 32000 entries at k = 8, 29.5 for 256 of 128256 at k = 10, 11.4 for 40 of 128256 at k = 64; now 67.8,
    // 27.6 and 10.6, and the finish behind it 6.6 instead of 10.3 at k = 8.  Long rows: no difference.)  A shape with one
    // histogram has a second barrier there, behind its clearing.
    CsShared* css = reinterpret_cast<CsShared*>(dyn + Geom::SHARED_OFF);
    CsCta& cta = *reinterpret_cast<CsCta*>(dyn + Geom::SHARED_OFF + 2 * sizeof(CsShared));

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], SPREAD ? WARPS : 1);
            mbar_init(&empty[s], WARPS);
        }
        mbar_init_fence();
        cs_reset(css[0]);
        cs_reset(css[1]);
        cta.abort = 0;
        cta.k = fb.k;
        cta.surv_cap = fb.surv_cap;
        cta.quota = fb.quota;
        cta.surv_keys = a.surv_keys;
    }
    if (tid < WARPS) cta.wcnt[tid] = 0;
    for (int i = tid; i < Geom::HISTS * CS_HIST_WORDS; i += STREAM_THREADS) Geom::hist(dyn, 0)[i] = 0u;
    grid_dependency_sync();
    if (tid == 0 && blockIdx.x == 0) *a.redo_count = 0;
    __syncthreads();

    if (warp == WARPS) {
        // ---- producer: every tile of every piece of this CTA, in order; a lane per copy of the tile ----
        if (lane >= (SPREAD ? WARPS : 1)) return;
        const uint64_t pol = l2_evict_first_policy();
        uint32_t i = 0;
        FilterPiece pc;
        for (int k = 0; plan_piece(plan, blockIdx.x, k, pc); ++k) {
            const long long srow = source_row(a, pc.row);
            // (a row with a bad temperature is copied for nothing: its workers look the temperature up)
            const StagedRow<T> sr(reinterpret_cast<const T*>(a.logits) + (srow < 0 ? 0 : srow) * a.row_stride, a.V);
            const int row_chunks = (sr.end + CHUNK - 1) / CHUNK;
            for (int ti = pc.tile0; ti < pc.tile1; ++ti, ++i) {
                const int s = (int)(i % STAGES);
                const uint32_t round = i / STAGES;
                if (round > 0) {
                    const int wr = mbar_wait_twice(&empty[s], (round - 1) & 1, wait_limit_ns);
                    if (wr != WAIT_OK) atomicOr(a.status, ST_INTERNAL);
                    if (wr == WAIT_LOST) return;      // nothing more is issued
                }
                constexpr int GRANULES = CHUNK * (int)sizeof(T) / 16;
                if (!SPREAD) {
                    if (srow >= 0)
                        stage_tile<T>(stage_mem + s * TILE_BYTES, sr, ti * (TILE_CHUNKS * GRANULES), TILE_CHUNKS * GRANULES, &full[s], pol);
                } else if (srow >= 0 && lane * plan.tiles_per_row + ti < row_chunks) {
                    // (a lane per eighth)
                    stage_tile<T>(stage_mem + s * TILE_BYTES + ((lane + ti) & (WARPS - 1)) * (GRANULES * 16), sr,
                                  (lane * plan.tiles_per_row + ti) * GRANULES, GRANULES, &full[s], pol);
                }
                mbar_arrive(&full[s]);
            }
        }
        return;
    }

    // ---- workers ------------------------------------------------------------------------------
    u64* region = cand + warp * CS_REGION;
    bool dead = false;      // a wait ran out: this warp computes no more, but takes every tile and joins every barrier
    bool lost = false;      // a wait did not complete at all: the warp stops waiting as well
    uint32_t i = 0;
    int parity = 0;         // which copy of the per-piece state this piece uses
    // the record of a piece that every warp has done its share of (one thread)
    auto write_record = [&](const CsShared& done) {
        const int m = done.m;
        int flags = done.flags;
        if (cta.abort) flags = CSF_ABORT;
        else if (flags == 0 && (done.overflow || m > fb.surv_cap)) flags = CSF_REDO;      // too many candidates, or ties at the bound
        else if (flags == 0 && done.nan) flags = CSF_LOGIT;
        double zs = 0.0;
        if (STATS)
            for (int w = 0; w < WARPS; ++w) zs += done.wsum[w];
        // a reference that later logits overflowed, or NaN / +inf data: the direct kernel sorts it out
        if (STATS && flags == 0 && !(zs > 0.0 && zs < CUDART_INF)) flags = CSF_REDO;
        CsRowMeta meta;
        meta.count = m;
        meta.flags = flags;
        meta.ref_off = done.ref_off;
        meta.thr_key = done.thr_key;
        meta.top = bin_coord(done.top);
        meta.z_stream = zs;
        a.surv_meta[done.area] = meta;
    };
    FilterPiece pc;
    for (int k = 0; plan_piece(plan, blockIdx.x, k, pc); ++k) {
        if (pc.tile0 >= pc.tile1) continue;
        CsShared& cs = css[parity];
        unsigned* hist = Geom::hist(dyn, parity);
        parity ^= 1;
        const int row = pc.row;
        const float Tb = a.temperature[row / a.G];
        const long long srow = source_row(a, row);
        const bool in_range = srow >= 0;
        // chunks are counted from the row's first granule here: which 1024 entries make one is no matter
        const StagedRow<T> sr(reinterpret_cast<const T*>(a.logits) + (in_range ? srow : 0) * a.row_stride, a.V);
        const int mis = sr.mis, end = sr.end;
        const bool valid = temp_ok(Tb) && in_range;
        // chunks of the row; 0 once nothing more of it is to be worked on
        int row_chunks = valid && !dead ? (unsigned)(end + CHUNK - 1) / CHUNK : 0;
        const float c32 = temp_scale(Tb);
        float ref_off = 0.f, acc = 0.f;
        int wcount = 0;             // candidates in this warp's region (cs.wcnt[warp] holds the same number)

        for (int ti = pc.tile0; ti < pc.tile1; ++ti, ++i) {
            const int s = (int)(i % STAGES);
            const uint32_t round = i / STAGES;
            if (!lost) {
                const int wr = mbar_wait_twice(&full[s], round & 1, wait_limit_ns);
                if (wr != WAIT_OK) {
                    dead = true;
                    row_chunks = 0;
                    lost = wr == WAIT_LOST;
                    if (lane == 0) {
                        cta.abort = 1;
                        atomicOr(a.status, ST_INTERNAL);
                    }
                }
            }
            // this warp's chunk of the tile
            const int c = SPREAD ? ((warp - ti) & (WARPS - 1)) * plan.tiles_per_row + ti : ti * TILE_CHUNKS + warp;
            const bool work = c < row_chunks;
            const unsigned char* chunk = stage_mem + s * TILE_BYTES + warp * (CHUNK * (int)sizeof(T));
            ChunkRegs<T> regs;
            if (work) load_staged(regs, chunk, c * CHUNK, end, lane);
            if (ti == pc.tile0) {
                // first tile of a piece: each warp's own bound (none without a chunk), then the smallest of them, or the
                // third smallest
                unsigned k16 = 0u, most = 0u;
                if (work) {
                    float wm = 0.f;
                    if (fb.need <= 16) {
                        const float lm = regs.lane_max_plain();
                        k16 = first_tile_key_lanes(lm, fb.need);
                        if (STATS) wm = warp_max_redux(lm);
                    } else {
                        k16 = first_tile_key(regs, fb.group, fb.need);
                        if (STATS) wm = warp_max_redux(regs.lane_max_plain());
                    }
                    if (STATS && wm == wm) most = orderable(wm);
                }
                if (lane == 0) {
                    cs.first_key[warp] = k16 << 16;
                    if (STATS) cs.first_max[warp] = most;
                }
                workers_sync();
                // the copies of the piece before
                if (tid == 0) {
                    if (i) write_record(css[parity]);
                    cs_reset(css[parity]);
                    cs.flags = !in_range ? CSF_RANGE : !valid ? CSF_TEMPERATURE : 0;
                }
                if (i)
                    for (int x = tid; x < CS_HIST_WORDS; x += THREADS) Geom::hist(dyn, parity)[x] = 0u;
                if (Geom::HISTS == 1) workers_sync();
                const unsigned first_top = first_bound<Geom, SPREAD ? 3 : 1>(parity ^ 1, pc.area);
                if (STATS) ref_off = __fmul_rn(from_orderable(first_top), c32);
                if (valid && __any_sync(0xffffffffu, *(volatile unsigned*)&cs.thr_key < 0x00800000u)) {
                    // no finite bound (rows of -inf): everything would pass, padding included
                    if (lane == 0) cs.overflow = 1;
                    row_chunks = 0;
                }
                __syncwarp();
            }
            int added = 0;          // what this chunk appends to the region
            if (work && row_chunks) {
                if (SPREAD && lane == 0) atomicAdd(&cs.seen, 1);
                unsigned mask = pass_mask(regs, from_orderable(*(volatile unsigned*)&cs.thr_key));
                const int n = __popc(mask);
                added = __reduce_add_sync(0xffffffffu, n);
                if (added) {
                    const int vchunk = c * CHUNK - mis;
                    if (added > (SPREAD ? min(fb.quota, CS_REGION - wcount) : CS_REGION - wcount)) {
                        if (lane == 0) cta.arg[warp] = make_int2((int)(chunk - dyn), vchunk);
                        __syncwarp();
                        wcount = crowded_chunk<T, Geom, SPREAD>(mask, wcount, parity ^ 1);
                        if (wcount < 0) {
                            if (lane == 0) cs.overflow = 1;
                            row_chunks = wcount = 0;
                        }
                        added = 0;
                    } else if (mask) {
                        // every lane appends its own passing values: its slots come from the warp's counter
                        int pos = atomicAdd(&cta.wcnt[warp], n);
                        do {
                            const int bit = __ffs(mask) - 1;
                            mask &= mask - 1u;
                            const int off = bit_offset(bit, lane, (const T*)nullptr);
                            region[pos++] = ((u64)staged_key<T>(chunk, off) << 32) | (u64)(~(uint32_t)(vchunk + off));
                        } while (mask);
                    }
                }
            }
            __syncwarp();
            if (lane == 0 && !lost) mbar_arrive(&empty[s]);     // the staged chunk is not read again
            if (work) {
                if (STATS) {
                    acc += lane_exp_sum2(regs, c32, ref_off);
                } else {
                    // without the exp-sum (which turns NaN by itself) a NaN has to be looked for
                    const float lm = regs.lane_max();
                    if (lm != lm) cs.nan = 1;
                }
                // count the new entries in the histogram (those of a crowded chunk are counted already)
                const int g0 = *(volatile int*)&cs.g0;
                for (int x = wcount + lane; x < wcount + added; x += 32) hist_add(hist, hist_bin((unsigned)(region[x] >> 32), g0));
                wcount += added;
                // The bound is refreshed after tiles 1, 2, 3, 4, 6, 8, 12, 16, 24, ..., by one warp or another.  (After
                // every tile it took 157 -> 162 us of compress for 1024 rows of 262144 entries, k = 1024.)
                // The rank goes by the chunks that all warps have counted: some are tiles ahead of this one.
                const int t = ti - pc.tile0 + 1;
                if (warp == ((t + (t >> 3)) & (WARPS - 1)) && ((t & (t - 1)) == 0 || (t & 7) == 0 || t == 3 || t == 6 || t == 12)) {
                    __syncwarp();
                    const int rank = SPREAD ? bound_rank(fb.k, fb.per_chunk * (float)*(volatile int*)&cs.seen) : fb.k;
                    refresh_bound<Geom>(parity ^ 1, rank, fb.k);
                }
            }
        }

        // ---- end of the piece: survivors and statistics to the piece's scratch area ------------------
        __syncwarp();
        if (STATS) {
            const double sw = (double)warp_sum(acc);
            if (lane == 0) cs.wsum[warp] = sw;
            if (tid == 0) cs.ref_off = ref_off;
        }
        if (valid && !__any_sync(0xffffffffu, *(volatile int*)&cs.overflow | *(volatile int*)&cta.abort)) hand_over<Geom>(parity ^ 1, wcount);
        if (lane == 0) cta.wcnt[warp] = 0;
        __syncwarp();
    }
    workers_sync();
    if (tid == 0 && i) write_record(css[parity ^ 1]);
}

// ---- finish: select, order, cut, emit ---------------------------------------------------------
constexpr int CS_MAX_PIECES = 8;    // most pieces a row is dealt in
// A group of TPR threads finishes a row: the CTA's 256 threads, or a warp (four rows per CTA).
//   CAP     keys at or above the boundary bin the group can hold (more: the direct kernel)
//   KCAP    largest k_eff
//   BINS    bins of the counting sort, counted up from the row's bound: one or more per 16-bit logit code
//           (bin_coord); BINS / 128 binades at least for values away from zero; the last one is open-ended
template <int TPR> struct FinishGeom;
template <> struct FinishGeom<32> {
    static constexpr int ROWS = 4, CAP = 512, KCAP = 128, BINS = 512, AHEAD = 4, HOLD = 4, CTAS = 7;
};
template <> struct FinishGeom<THREADS> {
    static constexpr int ROWS = 1, CAP = 2 * MAX_K, KCAP = MAX_K, BINS = 2048, AHEAD = 2, HOLD = 4, CTAS = 6;
};
template <int TPR> constexpr int finish_smem_bytes() {
    return FinishGeom<TPR>::ROWS * (FinishGeom<TPR>::CAP * 8 + FinishGeom<TPR>::KCAP * 8 + FinishGeom<TPR>::BINS * 4);
}

struct CsFinishShared {
    RowShared row;
    int scan[WARPS];    // bin counts per warp
    int kth;            // bin that holds the row's k-th largest key
    int overflow;       // more keys at or above that bin than the buffer holds
};

// A row's survivors lie in one scratch area, or in those of its pieces if it was dealt in pieces.  A
// survivor set holds all of a piece's elements at or above its final bound; the row's k best are among
// the survivors if k of them reach the largest of the pieces' bounds.  The k best are found and put in
// order by a counting sort over the 16-bit codes and as much of what orders the keys of one code as the
// bins have room for: count the keys per bin, sum from the top, move every key that is not below the
// bin of the k-th into its bin's stretch, then place each by its rank among the keys of its own stretch
// (all pairs: a few keys).  Bound by latency for few rows (meta, survivors, six
// short phases: about 9 K cycles) and by issue for many.  It replaces a trim and a bitonic network over
// the survivors, which was 32 of 51 K cycles of a row with k = 1024: 172 -> 78 us for 4096 rows with
// k = 1024, 22 -> 15.5 us for 1536 rows with k = 256, 41 -> 6.6 us for 4096 rows with k = 8 (a warp
// each), 16.4 -> 7.0 us for 40 rows in eight pieces with k = 64 (the pieces' records are read by one
// lane each instead of one after the other).
// With one bin per code, bf16 logits around 30 / 100 (k = 1024) took 95 / 267 us for 1536 rows; now 37 / 37, and
// 33 around 0.
//
// A group finishes a row: its part of the dynamic shared memory fin_mem is number `group`, its exchange area fs.
// Returns false if the row has to go through compress_row: a piece's candidates did not fit, or there are too
// many ties.
template <typename T, bool STATS, int TPR>
__device__ __forceinline__ bool finish_survivors(const CompressArgs& a, const FilterPlan& plan, int row, int k_eff, unsigned char* fin_mem,
                                                 int group, CsFinishShared& fs) {
    typedef FinishGeom<TPR> Geom;
    constexpr int AHEAD = Geom::AHEAD, HOLD = Geom::HOLD, PER = Geom::BINS / TPR;
    const int tid = group_tid<TPR>(), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    u64* stretch = reinterpret_cast<u64*>(fin_mem) + group * (Geom::CAP + Geom::KCAP);
    u64* keys = stretch + Geom::CAP;
    int* bins = reinterpret_cast<int*>(reinterpret_cast<u64*>(fin_mem) + Geom::ROWS * (Geom::CAP + Geom::KCAP)) + group * Geom::BINS;
    const int surv_cap = cs_survivor_cap(a.k_max);
    // the scratch areas that hold this row: its own, or those of its pieces if it was dealt in pieces
    const int whole_rows = plan.q * plan.grid;
    const bool split_row = row >= whole_rows;
    const int area0 = split_row ? plan.rows + (row - whole_rows) * plan.split : row;
    const int nareas = split_row ? plan.split : 1;
    for (int x = tid; x < Geom::BINS / 4; x += TPR) reinterpret_cast<int4*>(bins)[x] = make_int4(0, 0, 0, 0);
    if (tid == 0) fs.overflow = 0;
    grid_dependency_sync();
    if (row >= plan.rows) return true;  // (a warp beyond the last row)
    const u64* src = a.surv_keys + (long long)area0 * surv_cap;
    // the first area's first slots exist for every k_max: requested before their number is known
    u64 held[HOLD];
#pragma unroll
    for (int x = 0; x < AHEAD; ++x) held[x] = src[x * TPR + tid];
    const float Tb = a.temperature[row / a.G];
    // ---- the pieces, one per lane: flags, the row's bound, where each piece's survivors begin -------
    CsRowMeta meta;
    meta.count = 0; meta.flags = 0; meta.thr_key = 0u; meta.top = 0; meta.ref_off = 0.f; meta.z_stream = 0.0;
    if (lane < nareas && (!split_row || lane == 0 || plan_piece_tile(plan, lane + 1) > plan_piece_tile(plan, lane)))
        meta = a.surv_meta[area0 + lane];
    __syncwarp();
    const unsigned flags = __reduce_or_sync(0xffffffffu, (unsigned)meta.flags);
    const unsigned thr_key = __reduce_max_sync(0xffffffffu, meta.thr_key);
    if (flags & (CSF_ABORT | CSF_TEMPERATURE | CSF_LOGIT | CSF_RANGE)) {
        emit_invalid_row<TPR>(a, row);
        if (tid == 0 && !(flags & CSF_ABORT))
            atomicOr(a.status, (flags & CSF_TEMPERATURE) ? ST_TEMPERATURE : (flags & CSF_RANGE) ? ST_RANGE : ST_LOGIT);
        return true;
    }
    int begin[CS_MAX_PIECES], m = 0;        // begin[p]: flat number of piece p's first survivor
#pragma unroll
    for (int p = 0; p < CS_MAX_PIECES; ++p) {
        begin[p] = m;
        m += __shfl_sync(0xffffffffu, meta.count, p);
    }
    bool redo = (flags & CSF_REDO) != 0;
    if (!redo) {
        const int g0 = bin_coord(thr_key >> 16);
        auto key_at = [&](int i) -> u64 {       // survivor i of the row (i < m)
            if (nareas == 1) return src[i];
            int p = 0, b = 0;
#pragma unroll
            for (int x = 1; x < CS_MAX_PIECES; ++x)
                if (i >= begin[x]) {
                    p = x;
                    b = begin[x];
                }
            return src[(long long)p * surv_cap + (i - b)];
        };
        // As many bins per 16-bit code as the row's codes leave room for, by what orders the keys of one code: the
        // low half of the logit, and for 16-bit logits, where these are all equal, the index (squeezed codes
        // have one bin).
        const int span = max(__reduce_max_sync(0xffffffffu, meta.top), g0) - g0 + 1;
        const int lg = 31 - __clz(max(Geom::BINS / span, 1));
        const int drop = max(32 - __clz(a.V) - lg, 0);
        auto bin_of = [&](u64 key) {
            const int c = bin_coord((unsigned)(key >> 48));
            int sub = sizeof(T) == 2 ? (int)(((unsigned)(a.V - 1) - ~(unsigned)key) >> drop) : (int)(((unsigned)(key >> 32) & 0xffffu) << lg >> 16);
            if ((unsigned)(c - 0x7FFF) <= 1u) sub = 0;
            return min(((c - g0) << lg) + sub, Geom::BINS - 1);
        };
        // the first HOLD survivors of each thread stay in registers, those below the bound as zero
#pragma unroll
        for (int x = 0; x < HOLD; ++x) {
            const int i = x * TPR + tid;
            if (x >= AHEAD || nareas > 1) held[x] = i < m ? key_at(i) : 0ull;
            if (i >= m || (unsigned)(held[x] >> 32) < thr_key) held[x] = 0ull;
        }
        group_sync<TPR>();      // the bins are zero
        // ---- count ------------------------------------------------------------------------------
#pragma unroll
        for (int x = 0; x < HOLD; ++x)
            if (held[x]) atomicAdd(&bins[bin_of(held[x])], 1);
#pragma unroll 4
        for (int i = HOLD * TPR + tid; i < m; i += TPR) {
            const u64 key = key_at(i);
            if ((unsigned)(key >> 32) >= thr_key) atomicAdd(&bins[bin_of(key)], 1);
        }
        group_sync<TPR>();
        // ---- bins -> number of keys in higher bins (thread t owns PER bins, the highest first) ------
        int cnt[PER], own = 0;
        int4* mine = reinterpret_cast<int4*>(bins + Geom::BINS - (tid + 1) * PER);
#pragma unroll
        for (int x = 0; x < PER / 4; ++x) {
            const int4 v = mine[x];
            cnt[4 * x] = v.x; cnt[4 * x + 1] = v.y; cnt[4 * x + 2] = v.z; cnt[4 * x + 3] = v.w;
            own += v.x + v.y + v.z + v.w;
        }
        int run = own;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, run, d);
            run += lane >= d ? y : 0;
        }
        if (TPR != 32) {
            if (lane == 31) fs.scan[warp] = run;
            group_sync<TPR>();
#pragma unroll
            for (int w = 0; w < WARPS; ++w)
                if (w < warp) run += fs.scan[w];
        }
        const int live = run;                                         // (the last thread has counted all of them)
        const bool holds_kth = run - own < k_eff && run >= k_eff;     // one thread
        run -= own;
#pragma unroll
        for (int x = PER - 1; x >= 0; --x) {
            const int c = cnt[x];
            cnt[x] = run;
            run += c;
        }
        if (holds_kth) {
            int x = PER - 1;        // the k-th lies in the lowest of the thread's bins with fewer than k_eff keys above it
#pragma unroll
            for (int y = PER - 2; y >= 0; --y)
                if (cnt[y] < k_eff) x = y;
            int end = run;          // keys down to and including bin x
#pragma unroll
            for (int y = 1; y < PER; ++y)
                if (y == x) end = cnt[y - 1];
            fs.kth = Geom::BINS - (tid + 1) * PER + x;
            if (end > Geom::CAP) fs.overflow = 1;         // too many ties with the k-th
        }
        if (tid == TPR - 1 && live < k_eff) fs.overflow = 1;          // a piece's bound reached too far ahead
#pragma unroll
        for (int x = 0; x < PER / 4; ++x) mine[x] = make_int4(cnt[4 * x], cnt[4 * x + 1], cnt[4 * x + 2], cnt[4 * x + 3]);
        group_sync<TPR>();
        redo = fs.overflow != 0;
        if (!redo) {
            // ---- move: afterwards bins[b] is the end of bin b's stretch, which begins where bin b + 1's ends
            const int kth = fs.kth;
            auto move = [&](u64 key) {
                const int b = bin_of(key);
                if (b >= kth) stretch[atomicAdd(&bins[b], 1)] = key;
            };
#pragma unroll
            for (int x = 0; x < HOLD; ++x)
                if (held[x]) move(held[x]);
#pragma unroll 4
            for (int i = HOLD * TPR + tid; i < m; i += TPR) {
                const u64 key = key_at(i);
                if ((unsigned)(key >> 32) >= thr_key) move(key);
            }
            group_sync<TPR>();
            // ---- rank inside the stretch
            const int total = bins[kth];
            for (int i = tid; i < total; i += TPR) {
                const u64 key = stretch[i];
                const int b = bin_of(key);
                const int s0 = b + 1 < Geom::BINS ? bins[b + 1] : 0, s1 = bins[b];
                int rank = s0;
#pragma unroll 4
                for (int x = s0; x < s1; ++x) rank += stretch[x] > key ? 1 : 0;
                if (rank < k_eff) keys[rank] = key;         // keys are distinct: every rank is taken once
            }
            group_sync<TPR>();
        }
    }
    if (redo) return false;
    const float top = key_logit(keys[0]);
    double Z = 0.0;
    if (STATS) {
        // move every piece's streamed sum from its reference onto the scale of the weights exp(l/T - top/T)
        const float c32 = temp_scale(Tb);
        if (meta.count > 0) Z = meta.z_stream * exp2_call((double)meta.ref_off - (double)top * (double)c32);
        __syncwarp();
        Z = warp_sum(Z);
    }
    const bool bad = !(top > -CUDART_INF_F) || !(top < CUDART_INF_F) || (STATS && !(Z > 0.0));
    if (bad) {
        emit_invalid_row<TPR>(a, row);
        if (tid == 0) atomicOr(a.status, ST_LOGIT);
        return true;
    }
    finish_row<false, TPR>(a, row, keys, k_eff, Tb, Z, &fs.row);
    return true;
}

// Many rows: those that have to go through compress_row are listed for the kernel behind this one.
template <typename T, bool STATS, int TPR>
__global__ void __launch_bounds__(TPR * FinishGeom<TPR>::ROWS, FinishGeom<TPR>::CTAS)
compress_finish_kernel(CompressArgs a, FilterPlan plan) {
    extern __shared__ __align__(16) unsigned char fin_mem[];
    __shared__ CsFinishShared shared[FinishGeom<TPR>::ROWS];
    const int group = TPR == 32 ? threadIdx.x >> 5 : 0;
    const int row = blockIdx.x * FinishGeom<TPR>::ROWS + group;
    if (!finish_survivors<T, STATS, TPR>(a, plan, row, kept_entries(a), fin_mem, group, shared[group]) && group_tid<TPR>() == 0) {
        a.redo_rows[atomicAdd(a.redo_count, 1)] = row;
        atomicAdd(a.redo_total, 1ull);
    }
}

// Few rows (all of them resident at two CTAs per SM, so that a row that is read again takes no longer than in a kernel
// of its own): the CTA that finishes a row also takes it through compress_row if need be.  A kernel behind this one
// for listed rows is a launch of 0.9 to 1.3 us that normally finds an empty list.  With it the finish was 7.4 us (8 x 5,
// V = 128256, k = 64), 4.7 (1 x 4, V = 32000) and 9.3 (48 x 5, fp32, by warps); now 6.9, 4.3 and 6.6, and no launch behind it.
template <typename T, bool ALIGNED, bool STATS>
__global__ void __launch_bounds__(THREADS, 2)
compress_finish_few_kernel(const __grid_constant__ CompressArgs a, const __grid_constant__ FilterPlan plan) {
    extern __shared__ __align__(16) unsigned char fin_mem[];
    __shared__ CsFinishShared fs;
    __shared__ CompressShared sh;
    const int row = blockIdx.x, k_eff = kept_entries(a);
    if (!finish_survivors<T, STATS, THREADS>(a, plan, row, k_eff, fin_mem, 0, fs)) {
        if (threadIdx.x == 0) atomicAdd(a.redo_total, 1ull);
        u64* cand = reinterpret_cast<u64*>(fin_mem);
        compress_row<T, ALIGNED, STATS>(a, row, k_eff, cand, cand + CAND_CAP, sh);
    }
}

}  // namespace picospec
