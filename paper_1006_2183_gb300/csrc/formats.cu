// Format conversions: transpose (Section 2.4 transposes B once as a
// preprocessing step), CSC -> DCSC with the AUX column index (Section 2.3),
// and device-side validation of the CSC invariants.
#include <algorithm>

#include "internal.cuh"
#include "sortnet.cuh"

using namespace sg;

namespace {

constexpr int RS_BLOCK = 256;
constexpr int RS_ROUNDS = 8;
constexpr int RS_TILE = RS_BLOCK * RS_ROUNDS;
constexpr int RS_WARPS = RS_BLOCK / 32;

// ---------------------------------------------------------------- stable LSD radix sort
// (uint32 key, uint32 payload) pairs, 8-bit digits.  Tile order inside a CTA is
// element e = round * 256 + tid, ranks are assigned in that order, so each pass is
// stable and the passes compose into a stable sort.
__global__ void __launch_bounds__(RS_BLOCK) k_rs_hist(const uint32_t* __restrict__ keys, int64_t n, int shift,
                                                      int64_t ntiles, int64_t* __restrict__ hist) {
    __shared__ int cnt[256];
    cnt[threadIdx.x] = 0;
    __syncthreads();
    const int64_t t0 = (int64_t)blockIdx.x * RS_TILE;
    for (int r = 0; r < RS_ROUNDS; ++r) {
        int64_t e = t0 + r * RS_BLOCK + threadIdx.x;
        if (e < n) atomicAdd(&cnt[(keys[e] >> shift) & 255u], 1);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * ntiles + blockIdx.x] = cnt[threadIdx.x];
}

__global__ void __launch_bounds__(RS_BLOCK) k_rs_scatter(const uint32_t* __restrict__ kin,
                                                         const uint32_t* __restrict__ vin, int64_t n, int shift,
                                                         int64_t ntiles, const int64_t* __restrict__ off,
                                                         uint32_t* __restrict__ kout, uint32_t* __restrict__ vout) {
    __shared__ int run[256];
    __shared__ int wcnt[RS_WARPS][256];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    run[tid] = 0;
    const int64_t t0 = (int64_t)blockIdx.x * RS_TILE;
    for (int r = 0; r < RS_ROUNDS; ++r) {
        const int64_t e = t0 + r * RS_BLOCK + tid;
        const bool valid = e < n;
        uint32_t key = valid ? kin[e] : 0u;
        uint32_t val = valid ? vin[e] : 0u;
        int d = valid ? (int)((key >> shift) & 255u) : 256;
        unsigned mask = __match_any_sync(0xffffffffu, d);
        int rank = __popc(mask & ((1u << lane) - 1u));
        int leader = __ffs(mask) - 1;
#pragma unroll
        for (int ww = 0; ww < RS_WARPS; ++ww) wcnt[ww][tid] = 0;
        __syncthreads();
        if (valid && lane == leader) wcnt[w][d] = __popc(mask);
        __syncthreads();
        {
            int acc = run[tid];
#pragma unroll
            for (int ww = 0; ww < RS_WARPS; ++ww) {
                int c = wcnt[ww][tid];
                wcnt[ww][tid] = acc;
                acc += c;
            }
            run[tid] = acc;
        }
        __syncthreads();
        if (valid) {
            int64_t pos = off[(int64_t)d * ntiles + blockIdx.x] + wcnt[w][d] + rank;
            kout[pos] = key;
            vout[pos] = val;
        }
        __syncthreads();
    }
}

__global__ void k_iota_u32(uint32_t* p, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = (uint32_t)i;
}

// col[t] = the column of entry t, a tile of EX_TILE entries per CTA: the columns that start in
// the tile leave their number at their first entry (an empty column's is overwritten by the
// next one's, which is larger), and a running maximum carries it over the rest.  (Lanes
// walking one column each took as long as the longest column.)  A tile over more than EX_SPAN
// columns searches the column of every entry instead: a CTA that walks a long run of empty
// columns waits for a load per few hundred of them (transpose of 2,000 entries in 2^20 columns
// 908 -> 89 us, in 2^26 columns 126 -> 0.14 ms).  2^22 columns, walked against searched: 15 / 36
// us of this kernel at 8,192 columns per tile, 30 / 45 at 32,768.
constexpr int EX_BLOCK = 256;
constexpr int EX_ITEMS = 8;
constexpr int EX_TILE = EX_BLOCK * EX_ITEMS;
constexpr int64_t EX_SPAN = 32768;

// The last column of [lo, hi] that starts at or before entry t (column lo does), searched by a
// warp with 32 probes a step: 4 dependent loads for a million columns, where halving has 20.
__device__ __forceinline__ int64_t last_start(const int64_t* __restrict__ cp, int64_t lo, int64_t hi, int64_t t) {
    const int lane = threadIdx.x & 31;
    while (lo < hi) {
        const int64_t step = (hi - lo + 31) >> 5;
        const unsigned after = ~__ballot_sync(0xffffffffu, __ldg(cp + min(lo + step * (lane + 1), hi)) <= t);
        const int k = after ? __ffs(after) - 1 : 32;   // probes at or before t
        const int64_t below = k < 32 ? min(lo + step * (k + 1), hi) - 1 : hi;
        if (k > 0) lo = min(lo + step * k, hi);
        hi = max(lo, below);
    }
    return lo;
}

__global__ void __launch_bounds__(EX_BLOCK) k_expand_cols(const int64_t* __restrict__ cp, int64_t n, int64_t nnz,
                                                          int32_t* __restrict__ col) {
    __shared__ int s_col[EX_TILE];
    __shared__ int s_w[EX_BLOCK / 32];
    __shared__ int s_ends[2];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int64_t t0 = (int64_t)blockIdx.x * EX_TILE, t1 = min(t0 + EX_TILE, nnz);
    if (warp < 2) {   // the columns of the tile's first and last entry
        const int64_t c = last_start(cp, 0, n - 1, warp ? t1 - 1 : t0);
        if (lane == 0) s_ends[warp] = (int)c;
    }
    for (int i = tid; i < EX_TILE; i += EX_BLOCK) s_col[i] = 0;
    __syncthreads();
    const int64_t c0 = s_ends[0], c1 = s_ends[1];
    if (c1 - c0 > EX_SPAN) {
        for (int64_t t = t0 + tid; t < t1; t += EX_BLOCK) {
            int64_t lo = c0, hi = c1;
            while (lo < hi) {
                const int64_t mid = (lo + hi + 1) >> 1;
                if (__ldg(cp + mid) <= t) lo = mid;
                else hi = mid - 1;
            }
            col[t] = (int32_t)lo;
        }
        return;
    }
    for (int64_t j = c0 + 1 + tid; j <= c1; j += EX_BLOCK) {
        const int64_t at = __ldg(cp + j);
        if (at > t0 && at < t1) atomicMax(&s_col[at - t0], (int)(j - c0));   // always, in a valid operand
    }
    __syncthreads();
    int v[EX_ITEMS], m = 0;
#pragma unroll
    for (int i = 0; i < EX_ITEMS; ++i) {
        m = max(m, s_col[tid * EX_ITEMS + i]);
        v[i] = m;
    }
    int x = m;   // inclusive maximum over the lanes, then over the warps
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x = max(x, y);
    }
    if (lane == 31) s_w[warp] = x;
    int before = __shfl_up_sync(0xffffffffu, x, 1);
    if (lane == 0) before = 0;
    __syncthreads();
    for (int w = 0; w < warp; ++w) before = max(before, s_w[w]);
#pragma unroll
    for (int i = 0; i < EX_ITEMS; ++i) s_col[tid * EX_ITEMS + i] = max(before, v[i]);
    __syncthreads();
    for (int i = tid; i < (int)(t1 - t0); i += EX_BLOCK) col[t0 + i] = (int32_t)(c0 + s_col[i]);
}

__global__ void k_row_hist(const int32_t* __restrict__ ir, int64_t nnz, int64_t m, int64_t* __restrict__ cnt) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nnz; i += (int64_t)gridDim.x * blockDim.x)
        if (ir[i] >= 0 && ir[i] < m) atomicAdd(reinterpret_cast<unsigned long long*>(cnt + ir[i]), 1ull);
}

template <int W>
struct Word;
template <>
struct Word<1> { using T = uint8_t; };
template <>
struct Word<4> { using T = uint32_t; };
template <>
struct Word<8> { using T = uint64_t; };

template <int W>
__global__ void k_gather(const uint32_t* __restrict__ perm, const int32_t* __restrict__ colid,
                         const void* __restrict__ vin, int64_t nnz, int32_t* __restrict__ ir_out,
                         void* __restrict__ vout) {
    using T = typename Word<W>::T;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nnz; i += (int64_t)gridDim.x * blockDim.x) {
        uint32_t s = perm[i];
        ir_out[i] = colid[s];
        if (vin) reinterpret_cast<T*>(vout)[i] = reinterpret_cast<const T*>(vin)[s];
    }
}

template <int W>
__global__ void k_take_values(const uint32_t* __restrict__ at, const void* __restrict__ vin, int64_t nnz,
                              void* __restrict__ vout) {
    using T = typename Word<W>::T;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nnz; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t t = at[i];
        if (t < nnz)   // a malformed operand's conversion leaves entries out
            reinterpret_cast<T*>(vout)[i] = reinterpret_cast<const T*>(vin)[t];
    }
}

// ---------------------------------------------------------------- sort within columns
// Entries of every column put in ascending order of their (distinct) keys, for transpose and
// permutation, where only the order within a column is unknown: one read and one write of the
// entries instead of the stable radix passes over all of them (three for 18 bits of row and
// three for 18 of column): P A P^T, A^T and the DCSC form of R-MAT 18 with 4 million entries,
// all kernels 916 -> 550 us, 60 launches -> 25.
struct SegSort {
    const int64_t* in_cp;     // column c: entries [in_cp[c], in_cp[c+1]) of key and val
    int64_t n, nnz;
    const int64_t* out_cp;    // written from out_cp[out_col[c]] on (out_col null: c)
    const int32_t* out_col;
    const int32_t* key;
    const int32_t* relabel;   // key k counts as relabel[k] (null: k)
    const void* val;          // may be null
    int32_t* okey;
    void* oval;
    int64_t bound;            // keys are below bound < 2^23
    int32_t* list;            // long columns, *nlist of them
    int* nlist;
    // columns of more than split_len entries are split by their keys into nwin windows of
    // 2^wbits keys, in chunks of SEG_CHUNK entries
    int64_t split_len;
    int wbits, nwin;
    int32_t* split;           // the columns, *nsplit of them
    int2* chunk;              // place in `split` and number of every chunk, *nchunk of them
    uint32_t* win;            // per column: entries of its SEG_WIN windows
    uint32_t* off;            // per chunk: where its entries go in every window
    uint32_t* wkey;           // the entries by windows: key and place in the column (nnz each)
    uint32_t* widx;
    int *nsplit, *nchunk;
};
constexpr int SEG_SB = 9;                     // slots of a warp's column: at most 512 entries
constexpr int SEG_MAX = 1 << SEG_SB;
constexpr int64_t SEG_BOUND = (int64_t(1) << (32 - SEG_SB)) - 1;
constexpr int SEG_BLOCK = 128;
constexpr int SEGL_BLOCK = 512;
constexpr int64_t SEGL_ROWS = 1 << 20;        // keys ranked at a time in a long column
// A column of more entries than one CTA takes (SEG_SPLIT, fewer where it would read them once per
// SEGL_ROWS keys) is cut into at most SEG_WIN windows of keys: its chunks count their entries per
// window, then put them there, and a CTA ranks each window.  One CTA for the whole column took
// 25.7 ms for a row of 2^22 entries (2.9 now, all of it the row counters), 4.07 ms for the
// permutation of 8 columns of 2^20 (0.50).  The line: permutation of 8 columns of 32,768 entries
// 118 us split and 165 whole, of 256 such columns 341 and 331, of 512 columns of 16,384 entries
// 323 and 289.
constexpr int64_t SEG_SPLIT = 16384;
constexpr int64_t SEG_WHOLE = 65536;
constexpr int SEG_CHUNK = 8192;
constexpr int SEG_WIN = 256;
constexpr int SEG_WIN_KEYS = 1 << 15;         // 256 windows of it hold the 2^23 keys

__device__ __forceinline__ int32_t seg_row(const SegSort& S, int64_t t) {
    const int32_t x = __ldg(S.key + t);
    return S.relabel ? __ldg(S.relabel + x) : x;
}

__device__ __forceinline__ uint32_t seg_key(const SegSort& S, int64_t t, int slot) {
    return ((uint32_t)seg_row(S, t) << SEG_SB) | (uint32_t)slot;
}

// A column of at most G K entries per group of G lanes (len 0: none); whole warps call it.
// key_at(i) is entry i's key << SEG_SB | i, put(to, k) stores the entry of key k in place `to`.
template <int G, int K, class Key, class Put>
__device__ __forceinline__ void seg_sort_column(int len, uint32_t* stage, Key key_at, Put put) {
    const int lane = threadIdx.x & (G - 1);
    uint32_t key[K];
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const int i = r * G + lane;
        key[r] = i < len ? key_at(i) : 0xffffffffu;
    }
    sort_keys<G, K>(key, lane);
    if constexpr (K == 1) {
        if (lane < len) put(lane, key[0]);
        return;
    }
#pragma unroll
    for (int r = 0; r < K; ++r) stage[st_ph(K * lane + r)] = key[r];
    __syncwarp();
#pragma unroll
    for (int r = 0; r < K; ++r) {
        const int i = r * G + lane;
        if (i < len) put(i, stage[st_ph(i)]);
    }
    __syncwarp();
}

// The same for a warp and at most SEG_MAX entries.
template <class Key, class Put>
__device__ __forceinline__ void seg_sort_warp(int len, uint32_t* stage, Key key_at, Put put) {
    if (len <= 64) seg_sort_column<32, 2>(len, stage, key_at, put);
    else if (len <= 128) seg_sort_column<32, 4>(len, stage, key_at, put);
    else if (len <= 256) seg_sort_column<32, 8>(len, stage, key_at, put);
    else seg_sort_column<32, 16>(len, stage, key_at, put);
}

// Entry of key k (its slot in the low bits) of the column at s, stored at `to`.
template <int W>
__device__ __forceinline__ void seg_put(const SegSort& S, int64_t s, int64_t to, uint32_t k) {
    using T = typename Word<W>::T;
    S.okey[to] = (int32_t)(k >> SEG_SB);
    if (S.val) reinterpret_cast<T*>(S.oval)[to] = __ldg(reinterpret_cast<const T*>(S.val) + s + (k & (SEG_MAX - 1)));
}

// A column given up to the split: room for its windows and one record per chunk.
__device__ __forceinline__ void seg_split(const SegSort& S, int32_t c, int64_t len) {
    const int v = atomicAdd(S.nsplit, 1), nch = (int)((len + SEG_CHUNK - 1) / SEG_CHUNK);
    S.split[v] = c;
    for (int w = 0; w < SEG_WIN; ++w) S.win[(int64_t)v * SEG_WIN + w] = 0u;
    const int q = atomicAdd(S.nchunk, nch);
    for (int i = 0; i < nch; ++i) S.chunk[q + i] = make_int2(v, i);
}

// `per` columns per warp and round (32, or 4 where they are long enough to fill a warp's lanes
// one after another): up to 4 entries by the column's own lane, up to 32 by groups of 8 lanes,
// four columns at a time, up to SEG_MAX by the warp; longer columns are listed.
template <int W>
__global__ void __launch_bounds__(SEG_BLOCK) k_seg_sort(SegSort S, int per) {
    __shared__ uint32_t s_stage[SEG_BLOCK / 32][st_span<SEG_MAX>()];
    uint32_t* stage = s_stage[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31, grp = lane >> 3;
    const int64_t step = (int64_t)gridDim.x * (SEG_BLOCK / 32) * per;
    for (int64_t c0 = ((int64_t)blockIdx.x * (SEG_BLOCK / 32) + (threadIdx.x >> 5)) * per; c0 < S.n; c0 += step) {
        const int64_t c = c0 + lane;
        int64_t s = 0, o = 0, len = 0;
        if (lane < per && c < S.n) {
            s = __ldg(S.in_cp + c);
            len = __ldg(S.in_cp + c + 1) - s;
            if (len > 0) o = __ldg(S.out_cp + (S.out_col ? __ldg(S.out_col + c) : c));
        }
        if (len > S.split_len) {
            seg_split(S, (int32_t)c, len);
        } else if (len > SEG_MAX) {
            S.list[atomicAdd(S.nlist, 1)] = (int32_t)c;
        } else if (len > 0 && len <= 4) {
            uint32_t k[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) k[i] = i < len ? seg_key(S, s + i, i) : 0xffffffffu;
            auto order = [&](int i, int j) {
                const uint32_t x = min(k[i], k[j]), y = max(k[i], k[j]);
                k[i] = x;
                k[j] = y;
            };
            order(0, 1);
            order(2, 3);
            order(0, 2);
            order(1, 3);
            order(1, 2);
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < len) seg_put<W>(S, s, o + i, k[i]);
        }
        unsigned few = __ballot_sync(0xffffffffu, len > 4 && len <= 32);
        while (few) {
            int src = -1;   // the group's column: the grp-th of the remaining ones
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                if (i == grp && few) src = __ffs(few) - 1;
                few &= few - 1;
            }
            const int from = src < 0 ? 0 : src;
            const int64_t gs = __shfl_sync(0xffffffffu, s, from), go = __shfl_sync(0xffffffffu, o, from);
            const int gl = __shfl_sync(0xffffffffu, (int)len, from);
            seg_sort_column<8, 4>(src < 0 ? 0 : gl, stage + grp * 40, [&](int i) { return seg_key(S, gs + i, i); },
                                  [&](int to, uint32_t k) { seg_put<W>(S, gs, go + to, k); });
        }
        unsigned many = __ballot_sync(0xffffffffu, len > 32 && len <= SEG_MAX);
        while (many) {
            const int src = __ffs(many) - 1;
            many &= many - 1;
            const int64_t ws = __shfl_sync(0xffffffffu, s, src), wo = __shfl_sync(0xffffffffu, o, src);
            const int wl = __shfl_sync(0xffffffffu, (int)len, src);
            seg_sort_warp(wl, stage, [&](int i) { return seg_key(S, ws + i, i); },
                          [&](int to, uint32_t k) { seg_put<W>(S, ws, wo + to, k); });
        }
    }
}

// The entries of one column whose keys lie in [base, base + rows), among its `len` ones: marked
// in a bitmap in shared memory and written at their keys' ranks from `o` on.  key_at(i) is an
// entry's key, src_at(i) its place in the column.  Returns how many there were; ends with a
// barrier.
template <int W, int BLOCK, class Key, class Src>
__device__ __forceinline__ int seg_rank(const SegSort& S, int64_t s, int64_t len, int base, int rows, int64_t o,
                                        uint4* bits, int* pre, int* cc, Key key_at, Src src_at) {
    using T = typename Word<W>::T;
    __shared__ int s_total;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ng = (rows + 127) >> 7, nch = (ng + 31) >> 5;
    for (int g = tid; g < ng; g += BLOCK) bits[g] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    for (int64_t i = tid; i < len; i += BLOCK) {
        const int k = key_at(i) - base;
        if ((unsigned)k < (unsigned)rows) atomicOr(reinterpret_cast<uint32_t*>(bits) + (k >> 5), 1u << (k & 31));
    }
    __syncthreads();
    // keys before every 128 (pre, inside its chunk of 32 groups) and before every chunk (cc)
    for (int q = warp; q < nch; q += BLOCK / 32) {
        const int g = q * 32 + lane;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (g < ng) v = bits[g];
        const int k = __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w), inc = warp_incl_scan(k);
        if (g < ng) pre[g] = inc - k;
        if (lane == 31) cc[q] = inc;
    }
    __syncthreads();
    if (warp == 0) {
        int run = 0;
        for (int q0 = 0; q0 < nch; q0 += 32) {
            const int v = q0 + lane < nch ? cc[q0 + lane] : 0, inc = warp_incl_scan(v);
            if (q0 + lane < nch) cc[q0 + lane] = run + inc - v;
            run += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) s_total = run;
    }
    __syncthreads();
    for (int64_t i = tid; i < len; i += BLOCK) {
        const int k = key_at(i) - base;
        if ((unsigned)k >= (unsigned)rows) continue;
        const int g = k >> 7, y = (k >> 5) & 3;
        const uint4 v = bits[g];
        const uint32_t w = y == 0 ? v.x : y == 1 ? v.y : y == 2 ? v.z : v.w;
        const int rank = cc[g >> 5] + pre[g] + __popc(w & ((1u << (k & 31)) - 1u)) + (y > 0 ? __popc(v.x) : 0) +
                         (y > 1 ? __popc(v.y) : 0) + (y > 2 ? __popc(v.z) : 0);
        S.okey[o + rank] = k + base;
        if (S.val) reinterpret_cast<T*>(S.oval)[o + rank] = __ldg(reinterpret_cast<const T*>(S.val) + s + src_at(i));
    }
    const int total = s_total;
    __syncthreads();
    return total;
}

// entries [i0, i1) of a chunk, where they start in their column's arrays, and the column's place
// in the list of split columns
struct SegChunk {
    int v;
    int64_t c, s, i0, i1;
    __device__ SegChunk(const SegSort& S, int q) {
        const int2 e = S.chunk[q];
        v = e.x;
        c = S.split[v];
        s = __ldg(S.in_cp + c);
        const int64_t len = __ldg(S.in_cp + c + 1) - s;
        i0 = (int64_t)e.y * SEG_CHUNK;
        i1 = min(len, i0 + SEG_CHUNK);
    }
};

// A CTA per long column, SEGL_ROWS keys at a time, and per chunk of a split column: how many of
// its entries each window of keys gets, and where they go inside it.
template <int W>
__global__ void __launch_bounds__(SEGL_BLOCK) k_seg_long(SegSort S, int rows) {
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_win[SEG_WIN];
    const int ng = (rows + 127) >> 7;
    uint4* bits = reinterpret_cast<uint4*>(smem);
    int* pre = reinterpret_cast<int*>(bits + ng);
    int* cc = pre + ng;
    const int tid = threadIdx.x;
    const int n = *S.nlist, total = n + *S.nchunk;
    for (int l = blockIdx.x; l < total; l += gridDim.x) {
        if (l < n) {
            const int64_t c = S.list[l];
            const int64_t s = __ldg(S.in_cp + c), len = __ldg(S.in_cp + c + 1) - s;
            int64_t o = __ldg(S.out_cp + (S.out_col ? __ldg(S.out_col + c) : c));
            for (int64_t base = 0; base < S.bound; base += rows)
                o += seg_rank<W, SEGL_BLOCK>(S, s, len, (int)base, rows, o, bits, pre, cc,
                                             [&](int64_t i) { return seg_row(S, s + i); }, [](int64_t i) { return i; });
            continue;
        }
        const int q = l - n;
        const SegChunk ch(S, q);
        for (int w = tid; w < SEG_WIN; w += SEGL_BLOCK) s_win[w] = 0u;
        __syncthreads();
        for (int64_t i = ch.i0 + tid; i < ch.i1; i += SEGL_BLOCK) atomicAdd(&s_win[seg_row(S, ch.s + i) >> S.wbits], 1u);
        __syncthreads();
        for (int w = tid; w < SEG_WIN; w += SEGL_BLOCK) {
            const uint32_t k = s_win[w];
            S.off[(int64_t)q * SEG_WIN + w] = k ? atomicAdd(S.win + (int64_t)ch.v * SEG_WIN + w, k) : 0u;
        }
        __syncthreads();
    }
}

// Where the windows of split column v start inside it: s_at[w], from the windows' counts.  All
// threads of a CTA of at least SEG_WIN call it; ends with a barrier.
__device__ __forceinline__ void window_starts(const SegSort& S, int v, uint32_t* s_at, int* s_w) {
    const int tid = threadIdx.x, lane = tid & 31;
    int x = 0, inc = 0;
    if (tid < SEG_WIN) {
        x = (int)S.win[(int64_t)v * SEG_WIN + tid];
        inc = warp_incl_scan(x);
        if (lane == 31) s_w[tid >> 5] = inc;
    }
    __syncthreads();
    if (tid < SEG_WIN) {
        for (int w = 0; w < (tid >> 5); ++w) inc += s_w[w];
        s_at[tid] = (uint32_t)(inc - x);
    }
    __syncthreads();
}

// The entries of a chunk put into their windows, in any order inside them.
__global__ void __launch_bounds__(SEGL_BLOCK) k_seg_scatter(SegSort S) {
    __shared__ uint32_t s_at[SEG_WIN];
    __shared__ int s_w[SEG_WIN / 32];
    const int n = *S.nchunk;
    for (int q = blockIdx.x; q < n; q += gridDim.x) {
        const SegChunk ch(S, q);
        window_starts(S, ch.v, s_at, s_w);
        for (int w = threadIdx.x; w < SEG_WIN; w += SEGL_BLOCK) s_at[w] += S.off[(int64_t)q * SEG_WIN + w];
        __syncthreads();
        for (int64_t i = ch.i0 + threadIdx.x; i < ch.i1; i += SEGL_BLOCK) {
            const int k = seg_row(S, ch.s + i);
            const int64_t at = ch.s + atomicAdd(&s_at[k >> S.wbits], 1u);
            S.wkey[at] = (uint32_t)k;
            S.widx[at] = (uint32_t)i;
        }
        __syncthreads();
    }
}

// The windows of the split columns: those of at most SEG_MAX entries sorted by a warp each, eight
// of a column per CTA and round, then the longer ones ranked by a CTA each.
template <int W>
__global__ void __launch_bounds__(SEG_WIN, 4) k_seg_windows(SegSort S) {
    using T = typename Word<W>::T;
    constexpr int NG = SEG_WIN_KEYS / 128, NW = SEG_WIN / 32;
    __shared__ uint4 s_bits[NG];
    __shared__ int s_pre[NG], s_cc[(NG + 31) / 32], s_w[NW], s_big[SEG_WIN], s_nbig;
    __shared__ uint32_t s_at[SEG_WIN], s_stage[NW][st_span<SEG_MAX>()];
    const int tid = threadIdx.x, warp = tid >> 5;
    const int nsplit = *S.nsplit, per = (S.nwin + NW - 1) / NW;
    const T* __restrict__ val = reinterpret_cast<const T*>(S.val);
    int64_t s = 0, o = 0;   // of the column that s_at is for
    auto column = [&](int v) {
        window_starts(S, v, s_at, s_w);
        const int64_t c = S.split[v];
        s = __ldg(S.in_cp + c);
        o = __ldg(S.out_cp + (S.out_col ? __ldg(S.out_col + c) : c));
    };
    for (int l = blockIdx.x; l < nsplit * per; l += gridDim.x) {
        const int v = l / per, w = l % per * NW + warp;
        column(v);
        const uint32_t len = w < S.nwin ? S.win[(int64_t)v * SEG_WIN + w] : 0u;
        if (len > 0 && len <= SEG_MAX) {
            const int base = w << S.wbits;
            const int64_t at = s + s_at[w], to0 = o + s_at[w];
            seg_sort_warp((int)len, s_stage[warp], [&](int i) { return (S.wkey[at + i] - base) << SEG_SB | (uint32_t)i; },
                          [&](int to, uint32_t k) {
                              S.okey[to0 + to] = (int32_t)(k >> SEG_SB) + base;
                              if (val)
                                  reinterpret_cast<T*>(S.oval)[to0 + to] = __ldg(val + s + S.widx[at + (k & (SEG_MAX - 1))]);
                          });
        }
        __syncthreads();   // s_at is free for the next round
    }
    // the CTA's share of all windows, looked through by its threads at once
    const int64_t n = (int64_t)nsplit * S.nwin, step = gridDim.x;
    for (int64_t l0 = blockIdx.x; l0 < n; l0 += step * SEG_WIN) {
        if (tid == 0) s_nbig = 0;
        __syncthreads();
        const int64_t l = l0 + tid * step;
        if (l < n && S.win[l / S.nwin * SEG_WIN + l % S.nwin] > SEG_MAX) s_big[atomicAdd(&s_nbig, 1)] = (int)l;
        __syncthreads();
        const int nbig = s_nbig;
        for (int b = 0; b < nbig; ++b) {
            const int v = s_big[b] / S.nwin, w = s_big[b] % S.nwin;
            column(v);
            const int64_t len = S.win[(int64_t)v * SEG_WIN + w], at = s + s_at[w];
            seg_rank<W, SEG_WIN>(S, s, len, w << S.wbits, 1 << S.wbits, o + s_at[w], s_bits, s_pre, s_cc,
                                 [&](int64_t i) { return (int)S.wkey[at + i]; },
                                 [&](int64_t i) { return (int64_t)S.widx[at + i]; });
        }
        __syncthreads();
    }
}

// Transpose: where entry t goes inside its row, in any order (the rows are sorted afterwards).
// The additions to one counter queue at about one per nanosecond, so the rows that hold much of
// the matrix (about 0.8% of it and more: at least RP_HOT of RP_SAMPLES entries) are counted in
// shared memory, a tile of entries at a time, and take room for a tile's entries by one addition.
// Kernel times, transpose of a full 8 x 2^20 matrix: 1,071 -> 29 us; of one full row of 2^22
// entries beside a thousand of 4,200: 2,792 -> 208 us.  Every other row is counted entry by entry, in the order in which
// k_row_scatter writes the entries (the same grid): counting every row by tiles was faster here
// (R-MAT 18 72 -> 61 us), but a full 3000 x 3000 matrix then took 264 us to scatter, not 164.
constexpr int RP_BLOCK = 256;
constexpr int RP_ITEMS = 8;
constexpr int RP_TILE = RP_BLOCK * RP_ITEMS;
constexpr int RP_SAMPLES = 1024;
constexpr int RP_HOT = 8;
constexpr int RP_LOG = 11;                  // slots of the sampled rows: half of them stay free
constexpr int RP_HLOG = 7;                  // the rows counted in shared memory, four to a hash value
constexpr int RP_SLOTS = 4 << RP_HLOG;
constexpr int64_t RP_MIN = 1 << 18;         // no counter of fewer entries queues for long

// Zeroes n counters; CTA 0 looks for the rows to count in shared memory (nnz > 0): hot[slot], -1
// where there is none, and hot[RP_SLOTS] whether there is any.
__global__ void __launch_bounds__(RP_SAMPLES) k_row_begin(unsigned long long* __restrict__ cnt, int64_t n,
                                                          const int32_t* __restrict__ ir, int64_t nnz, int64_t m,
                                                          int32_t* __restrict__ hot) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) cnt[i] = 0ull;
    if (blockIdx.x > 0) return;
    __shared__ int s_row[1 << RP_LOG], s_hot[RP_SLOTS + 1];
    __shared__ int s_seen[1 << RP_LOG];
    const int tid = threadIdx.x;
    for (int i = tid; i < 1 << RP_LOG; i += RP_SAMPLES) {
        s_row[i] = -1;
        s_seen[i] = 0;
    }
    for (int i = tid; i < RP_SLOTS + 1; i += RP_SAMPLES) s_hot[i] = i < RP_SLOTS ? -1 : 0;
    __syncthreads();
    uint32_t x = (uint32_t)tid * 0x9E3779B1u;   // scattered: an even step could meet one row every time
    x ^= x >> 15;
    x *= 0x85EBCA6Bu;
    x ^= x >> 13;
    const int32_t r = ir[(int64_t)(((uint64_t)x * (uint64_t)nnz) >> 32)];
    if (r >= 0 && r < m) {
        uint32_t h = hash_row(r) >> (32 - RP_LOG);
        while (true) {
            const int held = atomicCAS(s_row + h, -1, r);
            if (held == -1 || held == r) break;
            h = (h + 1) & ((1 << RP_LOG) - 1);
        }
        if (atomicAdd(s_seen + h, 1) == RP_HOT - 1) {
            s_hot[RP_SLOTS] = 1;
            int* q = s_hot + 4 * (hash_row(r) >> (32 - RP_HLOG));
            for (int i = 0; i < 4 && atomicCAS(q + i, -1, r) != -1; ++i) {}   // a fifth is not counted there
        }
    }
    __syncthreads();
    for (int i = tid; i < RP_SLOTS + 1; i += RP_SAMPLES) hot[i] = s_hot[i];
}

__global__ void __launch_bounds__(RP_BLOCK) k_row_place(const int32_t* __restrict__ ir, int64_t nnz, int64_t m,
                                                        unsigned long long* __restrict__ cnt,
                                                        uint32_t* __restrict__ place, const int32_t* __restrict__ hot) {
    const int tid = threadIdx.x;
    if (!hot || !hot[RP_SLOTS]) {
        for (int64_t t = (int64_t)blockIdx.x * RP_BLOCK + tid; t < nnz; t += (int64_t)gridDim.x * RP_BLOCK) {
            const int32_t r = ir[t];
            if (r >= 0 && r < m) place[t] = (uint32_t)atomicAdd(cnt + r, 1ull);
        }
        return;
    }
    __shared__ __align__(16) int s_hot[RP_SLOTS];
    __shared__ uint32_t s_cnt[RP_SLOTS];   // entries of the tile, then where they start in the row
    for (int i = tid; i < RP_SLOTS; i += RP_BLOCK) {
        s_hot[i] = hot[i];
        s_cnt[i] = 0u;
    }
    __syncthreads();
    for (int64_t t0 = (int64_t)blockIdx.x * RP_TILE; t0 < nnz; t0 += (int64_t)gridDim.x * RP_TILE) {
        int row[RP_ITEMS], at[RP_ITEMS];   // at: slot and place among the tile's entries of the row, or -1
#pragma unroll
        for (int i = 0; i < RP_ITEMS; ++i) {
            const int64_t t = t0 + i * RP_BLOCK + tid;
            row[i] = t < nnz ? ir[t] : -1;
        }
#pragma unroll
        for (int i = 0; i < RP_ITEMS; ++i) {
            at[i] = -1;
            const int32_t r = row[i];
            if (r < 0 || r >= m) continue;   // malformed operand: left out
            const int h = (int)(hash_row(r) >> (32 - RP_HLOG));
            const int4 q = reinterpret_cast<const int4*>(s_hot)[h];
            const int slot = 4 * h + (q.y == r ? 1 : q.z == r ? 2 : q.w == r ? 3 : 0);
            if (q.x == r || slot > 4 * h) at[i] = slot * RP_TILE + (int)atomicAdd(s_cnt + slot, 1u);
            else place[t0 + i * RP_BLOCK + tid] = (uint32_t)atomicAdd(cnt + r, 1ull);
        }
        __syncthreads();
        for (int i = tid; i < RP_SLOTS; i += RP_BLOCK)
            if (s_cnt[i]) s_cnt[i] = (uint32_t)atomicAdd(cnt + s_hot[i], (unsigned long long)s_cnt[i]);
        __syncthreads();
#pragma unroll
        for (int i = 0; i < RP_ITEMS; ++i)
            if (at[i] >= 0) place[t0 + i * RP_BLOCK + tid] = s_cnt[at[i] / RP_TILE] + (uint32_t)(at[i] % RP_TILE);
        __syncthreads();
        for (int i = tid; i < RP_SLOTS; i += RP_BLOCK) s_cnt[i] = 0u;
        __syncthreads();
    }
}

template <int W>
__global__ void k_row_scatter(const int32_t* __restrict__ ir, const int32_t* __restrict__ colid,
                              const uint32_t* __restrict__ place, const void* __restrict__ num, int64_t nnz, int64_t m,
                              const int64_t* __restrict__ tcp, int32_t* __restrict__ key, void* __restrict__ val) {
    using T = typename Word<W>::T;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nnz; t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t r = ir[t];
        if (r < 0 || r >= m) continue;   // malformed operand: left out
        const int64_t at = __ldg(tcp + r) + place[t];
        key[at] = colid[t];
        if (num) reinterpret_cast<T*>(val)[at] = reinterpret_cast<const T*>(num)[t];
    }
}

// lengths of the permuted columns; with `zeroed` those of the nonempty ones alone
__global__ void k_perm_lens(const int64_t* __restrict__ cp, const int32_t* __restrict__ colp, int64_t n, bool zeroed,
                            int64_t* __restrict__ len) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        const int64_t l = cp[j + 1] - cp[j];
        if (l != 0 || !zeroed) len[colp ? colp[j] : j] = l;
    }
}

int grid_for(int64_t n, int block = 256) { return (int)std::max<int64_t>(1, std::min<int64_t>(ceil_div64(n, block), sm_count() * 32)); }

template <int W>
void run_seg_sort(cudaStream_t st, const SegSort& S) {
    // (R-MAT 18, 15 entries per column: 102 us with 4 columns per warp, 195 with 32, 126 with
    // one; a million columns of one entry: 20 us with 32, 464 with one)
    const int per = S.nnz >= 4 * S.n ? 4 : 32;
    const int grid = (int)std::min<int64_t>(ceil_div64(S.n, (SEG_BLOCK / 32) * per), (int64_t)sm_count() * 64);
    k_seg_sort<W><<<grid, SEG_BLOCK, 0, st>>>(S, per);
    const int rows = (int)std::min<int64_t>(S.bound, SEGL_ROWS);
    const size_t ng = (rows + 127) / 128;
    const size_t smem = ng * 20 + ((ng + 31) / 32) * 4;
    smem_at_least((const void*)k_seg_long<W>, smem);
    k_seg_long<W><<<sm_count() * 2, SEGL_BLOCK, smem, st>>>(S, rows);
    note_launch(2);
    if (S.nnz > S.split_len) {
        k_seg_scatter<<<(int)std::min<int64_t>(ceil_div64(S.nnz, SEG_CHUNK), sm_count() * 4), SEGL_BLOCK, 0, st>>>(S);
        k_seg_windows<W><<<sm_count() * 4, SEG_WIN, 0, st>>>(S);
        note_launch(2);
    }
}

// The scratch of a sort of n columns and nnz entries with keys below `bound`, laid out by
// take(bytes) -> offset; bind() sets S's pointers.  The counters are 16 bytes that the caller
// zeroes; wkey and widx are 4 nnz bytes each, the caller's too where they are given.
struct SegScratch {
    int64_t nnz, split_len;
    size_t o_list, o_split = 0, o_chunk = 0, o_win = 0, o_off = 0, o_wkey = 0, o_widx = 0;
    template <class Take>
    SegScratch(int64_t n, int64_t nz, int64_t bound, bool own_entries, Take take) : nnz(nz) {
        // a column holds no more entries than there are, nor than there are keys: up to SEG_WHOLE
        // of them none is split (a malformed one neither).  The two launches cost 6 us also
        // where no column needs them, of about 50 for a conversion of that size, and one CTA
        // takes 0.2 ms for a column of SEG_WHOLE entries.
        split_len = SEG_SPLIT / std::max<int64_t>(1, ceil_div64(bound, SEGL_ROWS));
        if (std::min(nnz, bound) <= SEG_WHOLE) split_len = INT64_MAX;
        o_list = take(4 * n);
        if (nnz <= split_len) return;
        const int64_t ns = nnz / split_len, nc = nnz / SEG_CHUNK + ns;
        o_split = take(4 * ns);
        o_chunk = take(8 * nc);
        o_win = take(4 * SEG_WIN * ns);
        o_off = take(4 * SEG_WIN * nc);
        if (own_entries) {
            o_wkey = take(4 * nnz);
            o_widx = take(4 * nnz);
        }
    }
    void bind(char* t, int* counters, uint32_t* wkey, uint32_t* widx, SegSort* S) const {
        S->list = (int32_t*)(t + o_list);
        S->nlist = counters;
        S->nsplit = counters + 1;
        S->nchunk = counters + 2;
        S->split_len = split_len;
        S->wbits = 10;
        while (S->bound > (int64_t)SEG_WIN << S->wbits) ++S->wbits;
        S->nwin = (int)ceil_div64(S->bound, int64_t(1) << S->wbits);
        S->split = (int32_t*)(t + o_split);
        S->chunk = (int2*)(t + o_chunk);
        S->win = (uint32_t*)(t + o_win);
        S->off = (uint32_t*)(t + o_off);
        S->wkey = wkey ? wkey : (uint32_t*)(t + o_wkey);
        S->widx = widx ? widx : (uint32_t*)(t + o_widx);
    }
};

void launch_seg_sort(cudaStream_t st, const SegSort& S, size_t w) {
    if (S.n <= 0) return;
    switch (w) {
    case 1: run_seg_sort<1>(st, S); break;
    case 4: run_seg_sort<4>(st, S); break;
    default: run_seg_sort<8>(st, S); break;
    }
}

// ---------------------------------------------------------------- DCSC
__global__ void k_nonempty(const int64_t* __restrict__ cp, int64_t n, int64_t* __restrict__ flag) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
        flag[j] = cp[j + 1] > cp[j] ? 1 : 0;
}

__global__ void k_dcsc_scatter(const int64_t* __restrict__ cp, int64_t n, const int64_t* __restrict__ pos,
                               int32_t* __restrict__ jc, int64_t* __restrict__ dcp) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        if (cp[j + 1] > cp[j]) {
            jc[pos[j]] = (int32_t)j;
            dcp[pos[j]] = cp[j];
        }
        if (j == n - 1) dcp[pos[n]] = cp[n];
    }
}

// AUX[t] = first JC position whose column id >= t * chunk; AUX[naux] = nzc
__global__ void k_aux(const int32_t* __restrict__ jc, int64_t nzc, int64_t chunk, int64_t naux,
                      int32_t* __restrict__ aux) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t <= naux; t += (int64_t)gridDim.x * blockDim.x) {
        if (t == naux) {
            aux[t] = (int32_t)nzc;
            continue;
        }
        int64_t v = t * chunk, lo = 0, hi = nzc;
        while (lo < hi) {
            int64_t mid = (lo + hi) >> 1;
            if ((int64_t)jc[mid] < v) lo = mid + 1;
            else hi = mid;
        }
        aux[t] = (int32_t)lo;
    }
}

// ---------------------------------------------------------------- validation
__global__ void k_validate(const int64_t* __restrict__ cp, const int32_t* __restrict__ ir, int64_t m, int64_t n,
                           int64_t nnz, int* __restrict__ bad) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
        int64_t s = cp[j], e = cp[j + 1];
        if (j == 0 && s != 0) { atomicMax(bad, 1); continue; }
        if (j == n - 1 && e != nnz) { atomicMax(bad, 2); continue; }
        if (e < s || s < 0 || e > nnz) { atomicMax(bad, 3); continue; }
        int32_t prev = -1;
        for (int64_t t = s; t < e; ++t) {
            int32_t r = ir[t];
            if (r < 0 || r >= m) { atomicMax(bad, 4); break; }
            if (r <= prev) { atomicMax(bad, 5); break; }
            prev = r;
        }
    }
}

// Format check of several stored CSC arrays at once: one warp per column of the
// concatenated column space (handle h owns columns [cbase[h], cbase[h+1])); the
// first lane checks the column's pointers, all lanes its rows.  bad[h] gets the
// largest violation code seen.
struct VDesc {
    const int64_t* cp;
    const int32_t* ir;
    int64_t m, n, nnz;
};
__global__ void k_validate_many(const VDesc* __restrict__ d, const int64_t* __restrict__ cbase, int nh,
                                int* __restrict__ bad) {
    const int lane = threadIdx.x & 31;
    const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t total = cbase[nh];
    for (int64_t c = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; c < total; c += nwarps) {
        int lo = 0, hi = nh - 1;   // the handle h with cbase[h] <= c < cbase[h+1]
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (cbase[mid] <= c) lo = mid;
            else hi = mid - 1;
        }
        const VDesc D = d[lo];
        const int64_t j = c - cbase[lo];
        const int64_t s = D.cp[j], e = D.cp[j + 1];
        int code = 0;
        if (j == 0 && s != 0) code = 1;
        else if (j == D.n - 1 && e != D.nnz) code = 2;
        else if (e < s || s < 0 || e > D.nnz) code = 3;
        if (code == 0) {
            for (int64_t t = s + lane; t < e; t += 32) {
                const int32_t r = D.ir[t];
                if (r < 0 || r >= D.m) code = code > 4 ? code : 4;
                else if (t > s && D.ir[t - 1] >= r) code = 5;
            }
        }
        if (code) atomicMax(bad + lo, code);
    }
}

}  // namespace

void launch_expand_cols(cudaStream_t st, const int64_t* cp, int64_t n, int64_t nnz, int32_t* col) {
    if (nnz <= 0) return;
    k_expand_cols<<<(unsigned)ceil_div64(nnz, EX_TILE), EX_BLOCK, 0, st>>>(cp, n, nnz, col);
    note_launch();
}

spgemm_status_t check_handles(spgemm_ctx* ctx, const std::vector<spgemm_mat*>& mats) {
    std::vector<spgemm_mat*> todo;
    for (spgemm_mat* M : mats)
        if (M && !M->checked && M->fmt != SPGEMM_FMT_DCSC && std::find(todo.begin(), todo.end(), M) == todo.end())
            todo.push_back(M);
    if (todo.empty()) return SPGEMM_OK;
    const int nh = (int)todo.size();
    std::vector<VDesc> hd(nh);
    std::vector<int64_t> hb(nh + 1, 0);
    for (int h = 0; h < nh; ++h) {
        spgemm_mat* M = todo[h];
        // stored arrays: CSC of (rows = stored m) x (cols = stored n)
        const int64_t sm = M->fmt == SPGEMM_FMT_CSR ? M->n : M->m;
        const int64_t sn = M->fmt == SPGEMM_FMT_CSR ? M->m : M->n;
        hd[h] = VDesc{M->cp, M->ir, sm, sn, M->nnz};
        hb[h + 1] = hb[h] + sn;
    }
    const size_t bytes = sizeof(VDesc) * nh + 8 * (nh + 1) + 4 * nh;
    auto buf = ctx_buf(ctx, bytes);
    if (!buf) return set_err(ctx, SPGEMM_ERR_OOM, "input check");
    VDesc* dd = (VDesc*)buf->p;
    int64_t* db = (int64_t*)(dd + nh);
    int* dbad = (int*)(db + nh + 1);
    cudaStream_t st = ctx->stream;
    SG_TRY(upload(ctx, dd, hd.data(), sizeof(VDesc) * nh));
    SG_TRY(upload(ctx, db, hb.data(), 8 * (nh + 1)));
    SG_CUDA(ctx, cudaMemsetAsync(dbad, 0, 4 * nh, st));
    std::vector<int> hbad(nh, 0);
    if (hb[nh] > 0) {
        k_validate_many<<<grid_for(hb[nh] * 32), 256, 0, st>>>(dd, db, nh, dbad);
        note_launch();
    }
    SG_TRY(read_back(ctx, hbad.data(), dbad, 4 * nh));
    // a matrix without columns: its (single) column pointer must be 0 and nnz 0
    std::vector<int64_t> c0(nh, 0);
    for (int h = 0; h < nh; ++h)
        if (hb[h + 1] == hb[h]) SG_TRY(read_back(ctx, &c0[h], todo[h]->cp, 8));
    SG_TRY(sync_ctx(ctx));
    static const char* why[] = {"", "colptr[0] != 0", "colptr[n] != nnz", "colptr not monotone",
                                "row index out of range", "rows not strictly ascending in a column"};
    for (int h = 0; h < nh; ++h) {
        int code = hbad[h];
        if (hb[h + 1] == hb[h] && (c0[h] != 0 || todo[h]->nnz != 0)) code = 1;
        if (code)
            return set_err(ctx, SPGEMM_ERR_BAD_FORMAT, "operand %d of this call (%lld x %lld): %s", h,
                           (long long)todo[h]->m, (long long)todo[h]->n, why[code < 6 ? code : 0]);
    }
    for (spgemm_mat* M : todo) M->checked = true;
    return SPGEMM_OK;
}

// Stable sort of (key, payload) pairs by the low `bits` bits of key, LSD with
// 8-bit digits.  Buffers (k0, v0) hold the input; the result ends in (k0, v0)
// or (k1, v1): *in_second tells which.  tmp needs radix_tmp_bytes(n).
size_t radix_tmp_bytes(int64_t n) {
    const int64_t ntiles = std::max<int64_t>(1, ceil_div64(n, RS_TILE));
    return 8 * (256 * ntiles + 1) * 2 + scan_tmp_bytes(256 * ntiles) + 256;
}

void radix_sort_pairs(cudaStream_t st, uint32_t* k0, uint32_t* v0, uint32_t* k1, uint32_t* v1, int64_t n, int bits,
                      void* tmp, bool* in_second) {
    *in_second = false;
    if (n <= 0 || bits <= 0) return;
    const int64_t ntiles = std::max<int64_t>(1, ceil_div64(n, RS_TILE));
    int64_t* hist = (int64_t*)tmp;
    int64_t* off = hist + (256 * ntiles + 1);
    void* stmp = off + (256 * ntiles + 1);
    for (int shift = 0; shift < bits; shift += 8) {
        k_rs_hist<<<(int)ntiles, RS_BLOCK, 0, st>>>(k0, n, shift, ntiles, hist);
        note_launch();
        launch_exclusive_scan(st, hist, 256 * ntiles, off, stmp);
        k_rs_scatter<<<(int)ntiles, RS_BLOCK, 0, st>>>(k0, v0, n, shift, ntiles, off, k1, v1);
        note_launch();
        std::swap(k0, k1);
        std::swap(v0, v1);
        *in_second = !*in_second;
    }
}

// CSC (m x n) -> CSC of the transpose (n x m), rows sorted.  `out` is filled in place.
spgemm_status_t transpose_csc(spgemm_ctx* ctx, int64_t m, int64_t n, int64_t nnz, const int64_t* cp,
                              const int32_t* ir, const void* num, size_t w, spgemm_mat_t out) {
    cudaStream_t st = ctx->stream;
    if (nnz > (int64_t)UINT32_MAX) return set_err(ctx, SPGEMM_ERR_INDEX_OVERFLOW, "transpose: nnz beyond 2^32");
    auto cpb = ctx_buf(ctx, 8 * (m + 1));
    auto irb = ctx_buf(ctx, 4 * std::max<int64_t>(nnz, 1));
    auto vb = ctx_buf(ctx, w * std::max<int64_t>(nnz, 1));
    if (nnz > 0 && n <= SEG_BOUND) {
        // rows counted, entries put into their rows in any order, then every row sorted; keys of
        // columns beyond 2^23 - 1 go through the radix passes below
        const int64_t nz = nnz;
        size_t off = 0;
        auto take = [&](size_t bytes) {
            const size_t o = off;
            off += (bytes + 255) / 256 * 256;
            return o;
        };
        const size_t o_cnt = take(8 * m + 16), o_sc = take(scan_tmp_bytes(m)), o_hot = take(4 * (RP_SLOTS + 1));
        const SegScratch scratch(m, nz, n, false, take);
        const size_t o_col = take(4 * nz), o_place = take(4 * nz), o_key = take(4 * nz), o_val = take(num ? w * nz : 0);
        auto tmp = ctx_buf(ctx, off);
        if (!cpb || !irb || !vb || !tmp) return set_err(ctx, SPGEMM_ERR_OOM, "transpose buffers");
        char* t = (char*)tmp->p;
        unsigned long long* cnt = (unsigned long long*)(t + o_cnt);   // m counts, then the sort's counters
        int32_t* colid = (int32_t*)(t + o_col);
        uint32_t* place = (uint32_t*)(t + o_place);
        int64_t* tcp = (int64_t*)cpb->p;
        int32_t* hot = nz >= RP_MIN ? (int32_t*)(t + o_hot) : nullptr;
        if (hot) {
            k_row_begin<<<grid_for(m + 2, RP_SAMPLES), RP_SAMPLES, 0, st>>>(cnt, m + 2, ir, nz, m, hot);
            note_launch();
        } else {
            SG_CUDA(ctx, cudaMemsetAsync(cnt, 0, 8 * m + 16, st));
        }
        k_row_place<<<grid_for(nz), RP_BLOCK, 0, st>>>(ir, nz, m, cnt, place, hot);
        note_launch();
        launch_expand_cols(st, cp, n, nz, colid);
        launch_exclusive_scan(st, (const int64_t*)cnt, m, tcp, t + o_sc);
        void* tv = num ? (void*)(t + o_val) : nullptr;
        switch (w) {
        case 1: k_row_scatter<1><<<grid_for(nz), 256, 0, st>>>(ir, colid, place, num, nz, m, tcp, (int32_t*)(t + o_key), tv); break;
        case 4: k_row_scatter<4><<<grid_for(nz), 256, 0, st>>>(ir, colid, place, num, nz, m, tcp, (int32_t*)(t + o_key), tv); break;
        default: k_row_scatter<8><<<grid_for(nz), 256, 0, st>>>(ir, colid, place, num, nz, m, tcp, (int32_t*)(t + o_key), tv); break;
        }
        note_launch();
        SegSort S{tcp, m, nz, tcp, nullptr, (const int32_t*)(t + o_key), nullptr, tv, (int32_t*)irb->p, vb->p, n};
        scratch.bind(t, (int*)(cnt + m), place, (uint32_t*)colid, &S);   // both are free by then
        launch_seg_sort(st, S, w);
        SG_CUDA(ctx, cudaGetLastError());
        out->ctx = ctx;
        out->fmt = SPGEMM_FMT_CSC;
        out->m = n;
        out->n = m;
        out->nnz = nnz;
        out->nzc = m;
        out->cp = tcp;
        out->ir = (const int32_t*)irb->p;
        out->num = num ? vb->p : nullptr;
        out->owned = {cpb, irb, vb};
        return SPGEMM_OK;
    }
    const int64_t ntiles = std::max<int64_t>(1, ceil_div64(nnz, RS_TILE));
    size_t tmp_bytes = 4 * 4 * std::max<int64_t>(nnz, 1) + 4 * std::max<int64_t>(nnz, 1) +
                       8 * (256 * ntiles + 1) * 2 + scan_tmp_bytes(std::max<int64_t>(256 * ntiles, m)) + 8 * (m + 1) +
                       1024;
    auto tmp = ctx_buf(ctx, tmp_bytes);
    if (!cpb || !irb || !vb || !tmp) return set_err(ctx, SPGEMM_ERR_OOM, "transpose buffers");
    char* t = (char*)tmp->p;
    const int64_t nz1 = std::max<int64_t>(nnz, 1);
    uint32_t* k0 = (uint32_t*)t; t += 4 * nz1;
    uint32_t* k1 = (uint32_t*)t; t += 4 * nz1;
    uint32_t* v0 = (uint32_t*)t; t += 4 * nz1;
    uint32_t* v1 = (uint32_t*)t; t += 4 * nz1;
    int32_t* colid = (int32_t*)t; t += 4 * nz1;
    t = (char*)(((uintptr_t)t + 255) / 256 * 256);
    int64_t* hist = (int64_t*)t; t += 8 * (256 * ntiles + 1);
    int64_t* off = (int64_t*)t; t += 8 * (256 * ntiles + 1);
    int64_t* rowcnt = (int64_t*)t; t += 8 * (m + 1);
    void* stmp = t;
    int64_t* tcp = (int64_t*)cpb->p;
    if (nnz > 0) {
        SG_CUDA(ctx, cudaMemcpyAsync(k0, ir, 4 * nnz, cudaMemcpyDeviceToDevice, st));
        k_iota_u32<<<grid_for(nnz), 256, 0, st>>>(v0, nnz);
        note_launch();
        launch_expand_cols(st, cp, n, nnz, colid);
        int bits = 0;
        while (bits < 32 && (int64_t(1) << bits) < m) ++bits;
        for (int shift = 0; shift < bits; shift += 8) {
            k_rs_hist<<<(int)ntiles, RS_BLOCK, 0, st>>>(k0, nnz, shift, ntiles, hist);
            note_launch();
            launch_exclusive_scan(st, hist, 256 * ntiles, off, stmp);
            k_rs_scatter<<<(int)ntiles, RS_BLOCK, 0, st>>>(k0, v0, nnz, shift, ntiles, off, k1, v1);
            note_launch();
            std::swap(k0, k1);
            std::swap(v0, v1);
        }
        SG_CUDA(ctx, cudaMemsetAsync(rowcnt, 0, 8 * m, st));
        k_row_hist<<<grid_for(nnz), 256, 0, st>>>(ir, nnz, m, rowcnt);
        note_launch();
        launch_exclusive_scan(st, rowcnt, m, tcp, stmp);
        note_launch();
        switch (w) {
        case 1: k_gather<1><<<grid_for(nnz), 256, 0, st>>>(v0, colid, num, nnz, (int32_t*)irb->p, vb->p); break;
        case 4: k_gather<4><<<grid_for(nnz), 256, 0, st>>>(v0, colid, num, nnz, (int32_t*)irb->p, vb->p); break;
        default: k_gather<8><<<grid_for(nnz), 256, 0, st>>>(v0, colid, num, nnz, (int32_t*)irb->p, vb->p); break;
        }
    } else {
        SG_CUDA(ctx, cudaMemsetAsync(tcp, 0, 8 * (m + 1), st));
    }
    SG_CUDA(ctx, cudaGetLastError());
    out->ctx = ctx;
    out->fmt = SPGEMM_FMT_CSC;
    out->m = n;
    out->n = m;
    out->nnz = nnz;
    out->nzc = m;
    out->cp = tcp;
    out->ir = (const int32_t*)irb->p;
    out->num = num ? vb->p : nullptr;
    out->owned = {cpb, irb, vb, tmp};
    // the temporaries are released with the handle's first owner release; drop them now
    out->owned.pop_back();
    return SPGEMM_OK;
}

spgemm_status_t csr_to_csc_refreshed(spgemm_ctx* ctx, spgemm_mat_t M, spgemm_mat_t* conv, ValueRefresh* r) {
    auto idx = ctx_buf(ctx, 4 * std::max<int64_t>(M->nnz, 1));
    auto val = ctx_buf(ctx, sr_size(M->sr) * std::max<int64_t>(M->nnz, 1));
    if (!idx || !val) return set_err(ctx, SPGEMM_ERR_OOM, "values of a CSR operand");
    if (M->nnz > 0) {
        k_iota_u32<<<grid_for(M->nnz), 256, 0, ctx->stream>>>((uint32_t*)idx->p, M->nnz);
        note_launch();
    }
    std::unique_ptr<spgemm_mat> T(new spgemm_mat());
    SG_TRY(transpose_csc(ctx, M->n, M->m, M->nnz, M->cp, M->ir, idx->p, 4, T.get()));
    T->sr = M->sr;
    *r = ValueRefresh{(const uint32_t*)T->num, M->num, val->p, M->nnz, sr_size(M->sr)};
    T->num = val->p;
    T->owned.push_back(val);
    *conv = T.release();
    return SPGEMM_OK;
}

void refresh_values(cudaStream_t st, const ValueRefresh& r) {
    if (r.nnz <= 0) return;
    switch (r.w) {
    case 1: k_take_values<1><<<grid_for(r.nnz), 256, 0, st>>>(r.at, r.from, r.nnz, r.to); break;
    case 4: k_take_values<4><<<grid_for(r.nnz), 256, 0, st>>>(r.at, r.from, r.nnz, r.to); break;
    default: k_take_values<8><<<grid_for(r.nnz), 256, 0, st>>>(r.at, r.from, r.nnz, r.to); break;
    }
    note_launch();
}

spgemm_status_t make_dcsc(spgemm_ctx* ctx, const spgemm_mat* M, bool with_aux, spgemm_mat* out) {
    cudaStream_t st = ctx->stream;
    const int64_t n = M->n;
    auto tmp = ctx_buf(ctx, 8 * (n + 1) * 2 + scan_tmp_bytes(n));
    if (!tmp) return set_err(ctx, SPGEMM_ERR_OOM, "dcsc temporaries");
    int64_t* flag = (int64_t*)tmp->p;
    int64_t* pos = flag + (n + 1);
    void* stmp = pos + (n + 1);
    int64_t nzc = 0;
    if (n > 0) {
        k_nonempty<<<grid_for(n), 256, 0, st>>>(M->cp, n, flag);
        note_launch();
        launch_exclusive_scan(st, flag, n, pos, stmp);
        SG_TRY(read_back(ctx, &nzc, pos + n, 8));
        SG_TRY(sync_ctx(ctx));
    }
    const int64_t chunk = n == 0 ? 1 : (nzc > 0 ? ceil_div64(n, nzc) : n);
    const int64_t naux = n == 0 ? 0 : ceil_div64(n, chunk);
    auto jcb = ctx_buf(ctx, 4 * std::max<int64_t>(nzc, 1));
    auto cpb = ctx_buf(ctx, 8 * (nzc + 1));
    std::shared_ptr<DevBuf> auxb;
    if (with_aux) auxb = ctx_buf(ctx, 4 * (naux + 1));
    if (!jcb || !cpb || (with_aux && !auxb)) return set_err(ctx, SPGEMM_ERR_OOM, "dcsc arrays");
    if (n > 0) {
        k_dcsc_scatter<<<grid_for(n), 256, 0, st>>>(M->cp, n, pos, (int32_t*)jcb->p, (int64_t*)cpb->p);
        note_launch();
    } else {
        SG_CUDA(ctx, cudaMemsetAsync(cpb->p, 0, 8, st));
    }
    if (with_aux) {
        k_aux<<<grid_for(naux + 1), 256, 0, st>>>((int32_t*)jcb->p, nzc, chunk, naux, (int32_t*)auxb->p);
        note_launch();
    }
    SG_CUDA(ctx, cudaGetLastError());
    out->ctx = ctx;
    out->fmt = SPGEMM_FMT_DCSC;
    out->sr = M->sr;
    out->m = M->m;
    out->n = n;
    out->nnz = M->nnz;
    out->nzc = nzc;
    out->cp = (const int64_t*)cpb->p;
    out->jc = (const int32_t*)jcb->p;
    out->aux = with_aux ? (const int32_t*)auxb->p : nullptr;
    out->naux = with_aux ? naux : 0;
    out->chunk = chunk;
    out->ir = M->ir;
    out->num = M->num;
    out->owned = M->owned;   // share the source's arrays if it owns them
    out->owned.push_back(jcb);
    out->owned.push_back(cpb);
    if (auxb) out->owned.push_back(auxb);
    return SPGEMM_OK;
}

// ------------------------------------------------------------------ permutation
// B = P A Q^T, B(p[i], q[j]) = A(i, j): the relabelling behind the random symmetric
// permutation of Section 5.3.3 (C' = (PAP^T)(PBP^T) = PCP^T) used to balance the 2D grid.

// counts[v]++ for every permutation entry; entries outside [0, n) raise the flag
__global__ void k_perm_count(const int32_t* __restrict__ perm, int64_t n, int32_t* __restrict__ cnt, int* bad) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t v = perm[i];
        if (v < 0 || v >= n) atomicExch(bad, 1);
        else atomicAdd(cnt + v, 1);
    }
}

// a permutation hits every value exactly once
__global__ void k_perm_check(const int32_t* __restrict__ cnt, int64_t n, int* bad) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        if (cnt[i] != 1) atomicExch(bad, 1);
}

// first sort key: the new row p[ir[t]] of every entry, and the entry index
__global__ void k_perm_rows(const int32_t* __restrict__ ir, const int32_t* __restrict__ rowp, int64_t nnz,
                            uint32_t* __restrict__ key, uint32_t* __restrict__ idx) {
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nnz; t += (int64_t)gridDim.x * blockDim.x) {
        const int32_t r = ir[t];
        key[t] = (uint32_t)(rowp ? rowp[r] : r);
        idx[t] = (uint32_t)t;
    }
}

// second sort key: the new column q[col(t)] of the entries in their row-sorted order
__global__ void k_perm_cols(const uint32_t* __restrict__ idx, const int32_t* __restrict__ colid,
                            const int32_t* __restrict__ colp, int64_t nnz, uint32_t* __restrict__ key,
                            int64_t* __restrict__ colcnt) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nnz; i += (int64_t)gridDim.x * blockDim.x) {
        const int32_t c = colid[idx[i]];
        const uint32_t nc = (uint32_t)(colp ? colp[c] : c);
        key[i] = nc;
        atomicAdd(reinterpret_cast<unsigned long long*>(colcnt + nc), 1ull);
    }
}

template <int W>
__global__ void k_perm_gather(const uint32_t* __restrict__ idx, const int32_t* __restrict__ ir,
                              const int32_t* __restrict__ rowp, const void* __restrict__ vin, int64_t nnz,
                              int32_t* __restrict__ ir_out, void* __restrict__ vout) {
    using T = typename Word<W>::T;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nnz; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t t = idx[i];
        const int32_t r = ir[t];
        ir_out[i] = rowp ? rowp[r] : r;
        if (vin) reinterpret_cast<T*>(vout)[i] = reinterpret_cast<const T*>(vin)[t];
    }
}

static int bits_for(int64_t n) {
    int b = 0;
    while (b < 32 && (int64_t(1) << b) < n) ++b;
    return b;
}

// Checks that row_perm and col_perm (null: identity) are permutations of 0..m-1 and 0..n-1, at
// one synchronisation.
static spgemm_status_t check_perms(spgemm_ctx* ctx, const int32_t* row_perm, int64_t m, const int32_t* col_perm,
                                   int64_t n) {
    const int32_t* perm[2] = {row_perm, col_perm};
    const int64_t len[2] = {m, n};
    static const char* what[] = {"row_perm", "col_perm"};
    cudaStream_t st = ctx->stream;
    std::shared_ptr<DevBuf> b[2];
    int h[2] = {0, 0};
    for (int i = 0; i < 2; ++i) {
        if (!perm[i] || len[i] == 0) continue;
        if (i == 1 && perm[1] == perm[0] && n == m) continue;   // the same array
        b[i] = ctx_buf(ctx, 4 * len[i] + 16);
        if (!b[i]) return set_err(ctx, SPGEMM_ERR_OOM, "permutation check");
        int32_t* cnt = (int32_t*)b[i]->p;
        int* bad = (int*)(cnt + len[i]);
        SG_CUDA(ctx, cudaMemsetAsync(cnt, 0, 4 * len[i] + 16, st));
        k_perm_count<<<grid_for(len[i]), 256, 0, st>>>(perm[i], len[i], cnt, bad);
        k_perm_check<<<grid_for(len[i]), 256, 0, st>>>(cnt, len[i], bad);
        note_launch(2);
        SG_TRY(read_back(ctx, &h[i], bad, sizeof(int)));
    }
    if (!b[0] && !b[1]) return SPGEMM_OK;
    SG_TRY(sync_ctx(ctx));
    for (int i = 0; i < 2; ++i)
        if (h[i])
            return set_err(ctx, SPGEMM_ERR_INVALID_ARG, "%s is not a permutation of 0..%lld", what[i],
                           (long long)(len[i] - 1));
    return SPGEMM_OK;
}

static spgemm_status_t permute_csc(spgemm_ctx* ctx, int64_t m, int64_t n, int64_t nnz, const int64_t* cp,
                                   const int32_t* ir, const void* num, size_t w, const int32_t* rowp,
                                   const int32_t* colp, spgemm_mat* out) {
    cudaStream_t st = ctx->stream;
    if (nnz > (int64_t)UINT32_MAX) return set_err(ctx, SPGEMM_ERR_INDEX_OVERFLOW, "permute: nnz beyond 2^32");
    const int64_t nz1 = std::max<int64_t>(nnz, 1);
    auto cpb = ctx_buf(ctx, 8 * (n + 1));
    auto irb = ctx_buf(ctx, 4 * nz1);
    auto vb = ctx_buf(ctx, w * nz1);
    if (n > 0 && m <= SEG_BOUND) {
        // the columns move whole, each sorted by its new rows; rows beyond 2^23 - 1 go through
        // the radix passes below
        size_t off = 0;
        auto take = [&](size_t bytes) {
            const size_t o = off;
            off += (bytes + 255) / 256 * 256;
            return o;
        };
        const size_t o_len = take(8 * n + 16), o_sc = take(scan_tmp_bytes(n));
        const SegScratch scratch(n, nnz, m, true, take);
        auto tmp = ctx_buf(ctx, off);
        if (!cpb || !irb || !vb || !tmp) return set_err(ctx, SPGEMM_ERR_OOM, "permute buffers");
        char* t = (char*)tmp->p;
        int64_t* len = (int64_t*)(t + o_len);   // n lengths, then the sort's counters
        int64_t* ocp = (int64_t*)cpb->p;
        // mostly empty columns: zeroes in order cost less than a scattered store per column
        // (2^26 columns of 2,000 entries: 2.53 ms of 5.4)
        const bool few = colp && nnz < n / 2;
        if (few) SG_CUDA(ctx, cudaMemsetAsync(len, 0, 8 * n + 16, st));
        else SG_CUDA(ctx, cudaMemsetAsync(len + n, 0, 16, st));
        k_perm_lens<<<grid_for(n), 256, 0, st>>>(cp, colp, n, few, len);
        note_launch();
        launch_exclusive_scan(st, len, n, ocp, t + o_sc);
        SegSort S{cp, n, nnz, ocp, colp, ir, rowp, num, (int32_t*)irb->p, vb->p, m};
        scratch.bind(t, (int*)(len + n), nullptr, nullptr, &S);
        launch_seg_sort(st, S, w);
        SG_CUDA(ctx, cudaGetLastError());
        out->ctx = ctx;
        out->fmt = SPGEMM_FMT_CSC;
        out->m = m;
        out->n = n;
        out->nnz = nnz;
        out->nzc = n;
        out->cp = ocp;
        out->ir = (const int32_t*)irb->p;
        out->num = num ? vb->p : nullptr;
        out->owned = {cpb, irb, vb};
        return sync_ctx(ctx);   // permute returns with its result complete
    }
    const size_t rs = radix_tmp_bytes(nnz);
    auto tmp = ctx_buf(ctx, 5 * 4 * nz1 + 8 * (n + 1) + rs + scan_tmp_bytes(std::max<int64_t>(n, 1)) + 1024);
    if (!cpb || !irb || !vb || !tmp) return set_err(ctx, SPGEMM_ERR_OOM, "permute buffers");
    char* t = (char*)tmp->p;
    uint32_t* k0 = (uint32_t*)t; t += 4 * nz1;
    uint32_t* k1 = (uint32_t*)t; t += 4 * nz1;
    uint32_t* v0 = (uint32_t*)t; t += 4 * nz1;
    uint32_t* v1 = (uint32_t*)t; t += 4 * nz1;
    int32_t* colid = (int32_t*)t; t += 4 * nz1;
    t = (char*)(((uintptr_t)t + 255) / 256 * 256);
    int64_t* colcnt = (int64_t*)t; t += 8 * (n + 1);
    t = (char*)(((uintptr_t)t + 255) / 256 * 256);
    void* rtmp = t; t += rs;
    t = (char*)(((uintptr_t)t + 255) / 256 * 256);
    void* stmp = t;
    int64_t* ocp = (int64_t*)cpb->p;
    SG_CUDA(ctx, cudaMemsetAsync(colcnt, 0, 8 * (n + 1), st));
    if (nnz > 0) {
        // LSD order: by new row, then stably by new column
        k_perm_rows<<<grid_for(nnz), 256, 0, st>>>(ir, rowp, nnz, k0, v0);
        note_launch();
        launch_expand_cols(st, cp, n, nnz, colid);
        bool second = false;
        radix_sort_pairs(st, k0, v0, k1, v1, nnz, bits_for(m), rtmp, &second);
        uint32_t* vr = second ? v1 : v0;   // entry indices in new-row order
        uint32_t* kA = second ? k0 : k1;   // free key buffer
        uint32_t* kB = second ? k1 : k0;   // the row keys, no longer needed
        uint32_t* vB = second ? v0 : v1;   // free value buffer
        k_perm_cols<<<grid_for(nnz), 256, 0, st>>>(vr, colid, colp, nnz, kA, colcnt);
        note_launch();
        bool second2 = false;
        radix_sort_pairs(st, kA, vr, kB, vB, nnz, bits_for(n), rtmp, &second2);
        const uint32_t* fin = second2 ? vB : vr;
        switch (w) {
        case 1: k_perm_gather<1><<<grid_for(nnz), 256, 0, st>>>(fin, ir, rowp, num, nnz, (int32_t*)irb->p, vb->p); break;
        case 4: k_perm_gather<4><<<grid_for(nnz), 256, 0, st>>>(fin, ir, rowp, num, nnz, (int32_t*)irb->p, vb->p); break;
        default: k_perm_gather<8><<<grid_for(nnz), 256, 0, st>>>(fin, ir, rowp, num, nnz, (int32_t*)irb->p, vb->p); break;
        }
        note_launch();
    }
    launch_exclusive_scan(st, colcnt, n, ocp, stmp);
    SG_CUDA(ctx, cudaGetLastError());
    out->ctx = ctx;
    out->fmt = SPGEMM_FMT_CSC;
    out->m = m;
    out->n = n;
    out->nnz = nnz;
    out->nzc = n;
    out->cp = ocp;
    out->ir = (const int32_t*)irb->p;
    out->num = num ? vb->p : nullptr;
    out->owned = {cpb, irb, vb};
    SG_TRY(sync_ctx(ctx));   // the temporaries are released when this call returns
    return SPGEMM_OK;
}

extern "C" {

spgemm_status_t spgemm_mat_permute(spgemm_ctx_t ctx, spgemm_mat_t a, const int32_t* row_perm,
                                   const int32_t* col_perm, spgemm_mat_t* out) {
    if (!ctx || !a || !out) return SPGEMM_ERR_INVALID_ARG;
    if (a->fmt == SPGEMM_FMT_DCSC) return set_err(ctx, SPGEMM_ERR_UNSUPPORTED, "permute of a DCSC handle");
    SG_TRY(check_perms(ctx, row_perm, a->m, col_perm, a->n));
    SG_TRY(check_handles(ctx, {a}));
    spgemm_mat_t conv = nullptr;
    DMat d;
    SG_TRY(to_csc_operand(ctx, a, &conv, &d));
    std::unique_ptr<spgemm_mat> hold(conv);
    auto* P = new spgemm_mat();
    spgemm_status_t s = permute_csc(ctx, d.m, d.n, d.nnz, d.cp, d.ir, d.num, sr_size(a->sr), row_perm, col_perm, P);
    if (s != SPGEMM_OK) {
        delete P;
        return s;
    }
    P->sr = a->sr;
    P->checked = true;
    *out = P;
    return SPGEMM_OK;
}

spgemm_status_t spgemm_mat_transpose(spgemm_ctx_t ctx, spgemm_mat_t a, spgemm_mat_t* out) {
    if (!ctx || !a || !out) return SPGEMM_ERR_INVALID_ARG;
    if (a->fmt == SPGEMM_FMT_DCSC) return set_err(ctx, SPGEMM_ERR_UNSUPPORTED, "transpose of a DCSC handle");
    SG_TRY(check_handles(ctx, {a}));
    auto* T = new spgemm_mat();
    T->checked = true;
    spgemm_status_t s;
    if (a->fmt == SPGEMM_FMT_CSR) {
        // CSR(A) stores CSC(A^T): its arrays already are A^T in CSC; copy nothing, borrow
        T->ctx = ctx;
        T->fmt = SPGEMM_FMT_CSC;
        T->m = a->n;
        T->n = a->m;
        T->nnz = a->nnz;
        T->nzc = a->m;
        T->cp = a->cp;
        T->ir = a->ir;
        T->num = a->num;
        T->owned = a->owned;
        s = SPGEMM_OK;
    } else {
        s = transpose_csc(ctx, a->m, a->n, a->nnz, a->cp, a->ir, a->num, sr_size(a->sr), T);
    }
    if (s != SPGEMM_OK) {
        delete T;
        return s;
    }
    T->sr = a->sr;
    *out = T;
    return SPGEMM_OK;
}

spgemm_status_t spgemm_mat_to_dcsc(spgemm_ctx_t ctx, spgemm_mat_t csc, int build_aux, spgemm_mat_t* out) {
    if (!ctx || !csc || !out) return SPGEMM_ERR_INVALID_ARG;
    if (csc->fmt != SPGEMM_FMT_CSC) return set_err(ctx, SPGEMM_ERR_INVALID_ARG, "to_dcsc expects a CSC handle");
    SG_TRY(check_handles(ctx, {csc}));
    auto* D = new spgemm_mat();
    D->checked = true;
    spgemm_status_t s = make_dcsc(ctx, csc, build_aux != 0, D);
    if (s != SPGEMM_OK) {
        delete D;
        return s;
    }
    *out = D;
    return SPGEMM_OK;
}

spgemm_status_t spgemm_mat_validate(spgemm_mat_t M) {
    if (!M) return SPGEMM_ERR_INVALID_ARG;
    spgemm_ctx* ctx = M->ctx;
    if (M->fmt == SPGEMM_FMT_DCSC) return set_err(ctx, SPGEMM_ERR_UNSUPPORTED, "validate of DCSC");
    // stored arrays: CSC with (rows = stored m) x (cols = stored n)
    const int64_t sm = M->fmt == SPGEMM_FMT_CSR ? M->n : M->m;
    const int64_t sn = M->fmt == SPGEMM_FMT_CSR ? M->m : M->n;
    auto flag = ctx_buf(ctx, 16);
    if (!flag) return set_err(ctx, SPGEMM_ERR_OOM, "validate flag");
    SG_CUDA(ctx, cudaMemsetAsync(flag->p, 0, 4, ctx->stream));
    int h = 0;
    if (sn > 0) {
        k_validate<<<grid_for(sn), 256, 0, ctx->stream>>>(M->cp, M->ir, sm, sn, M->nnz, (int*)flag->p);
        note_launch();
    } else {
        int64_t c0 = -1;
        SG_TRY(read_back(ctx, &c0, M->cp, 8));
        SG_TRY(sync_ctx(ctx));
        if (c0 != 0 || M->nnz != 0) h = 1;
    }
    if (sn > 0) {
        SG_TRY(read_back(ctx, &h, flag->p, 4));
        SG_TRY(sync_ctx(ctx));
    }
    static const char* why[] = {"", "colptr[0] != 0", "colptr[n] != nnz", "colptr not monotone",
                                "row index out of range", "rows not strictly ascending in a column"};
    if (h) return set_err(ctx, SPGEMM_ERR_BAD_FORMAT, "%s", why[h < 6 ? h : 0]);
    M->checked = true;
    return SPGEMM_OK;
}

}  // extern "C"
