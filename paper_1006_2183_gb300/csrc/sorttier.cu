// Sort tier: columns of at most 1024 products (TierCfg::sort_max), whatever the number
// of rows that the keys hold.  A group of G lanes takes one output column
// C(:,j) = (+)_{k in B(:,j)} A(:,k) (x) B(k,j) (Section 2.1), N = G K products at most:
//   1. product p goes to lane p mod G as the key (row << log2 N) | p, its value to slot
//      p of shared memory;
//   2. a bitonic network sorts the keys, element i = K lane + r in register r of its
//      lane: the steps at distances below K stay inside a lane, so a network over N
//      elements takes log2 G (log2 G + 1) / 2 shuffled steps (6 for 64 products on 8
//      lanes, where one register per lane on 32 lanes and 2 per lane would take 15);
//   3. equal rows are adjacent: a lane adds its runs up in ascending k, runs that cross
//      lanes go through a segmented scan, which is skipped where no run does (FP64
//      additions are the slow pipe of this part, about two lanes per SM clock);
//   4. rows and values are put in order in shared memory and stored coalesced.
// No atomics, no tables to fill and empty, and several columns per warp share the
// latency of the loads that a column starts with.  The counting form sorts rows alone.
// Bound by instruction issue and the FP64 pipe, not by memory: what the registers and the
// slots leave resident decides (the caps below).  Against one warp per column with 32-lane
// networks and, for operands of many rows, shared-memory hash tables whose entries were
// then sorted: R*(A*P) on 128^3 FP64, 262,144 columns of 50 to 60 products and as many of
// about 32, 736 -> 265 us (counting 294 -> 155 us); 20 int64 pairs, columns of up to 1024
// products, 1.35 -> 0.40 ms (counting 0.30 -> 0.27 ms); the columns of 513 to 1024 products
// of a scale-20 R-MAT square FP64, 1456 -> 361 us (counting 230 -> 218 us).
#include <algorithm>

#include "internal.cuh"
#include "sortnet.cuh"

namespace sg {
namespace {

// threads per CTA: 8 warps, fewer where a column's slots take 7 or 14 KB
constexpr int st_block(int K) { return K == 32 ? 64 : K == 16 ? 128 : 256; }
// CTAs per SM that the registers are held to: the most that the slots leave room for
// (numeric; at K = 8 one less, where a sixth spills: 693 -> 675 us for the 8-lane network
// of that product and two merges) or that the keys of the counting network allow
constexpr int st_min_blocks(int K, bool num) {
    if (num) return K >= 16 ? 8 : K == 8 ? 5 : 6;
    return K == 32 ? 12 : K == 16 ? 8 : 5;
}

template <int G, class V>
__device__ __forceinline__ V shflg(V x, int src) {
    if constexpr (sizeof(V) == 1) return (V)__shfl_sync(0xffffffffu, (int)x, src, G);
    else return __shfl_sync(0xffffffffu, x, src, G);
}

// NUM: rows and values to C (Coff as for launch_block_tier); otherwise counts to nnz_item.
template <class SR, int G, int K, bool NUM>
__global__ void __launch_bounds__(st_block(K), st_min_blocks(K, NUM))
k_sort(Items it, const int2* __restrict__ list, int64_t count, int64_t* __restrict__ nnz_item,
       const int64_t* __restrict__ Coff, int32_t* __restrict__ Cir, typename SR::T* __restrict__ Cv,
       const int* __restrict__ vals_zero) {
    using T = typename SR::T;
    using Acc = typename SR::Acc;
    constexpr int N = G * K, SB = ilog2(N), NG = st_block(K) / G, SPAN = st_span<N>();
    constexpr uint32_t NONE = 0xffffffffu;
    constexpr uint32_t NOROW = NONE >> SB;   // no stored row (the host bounds the rows)
    __shared__ Acc s_val[NUM ? NG * SPAN : 1];
    __shared__ uint32_t s_key[NG * SPAN];
    const int lane = threadIdx.x & (G - 1), grp = threadIdx.x / G;
    Acc* sv = s_val + (NUM ? grp * SPAN : 0);
    uint32_t* sk = s_key + grp * SPAN;
    // boolean products whose operands hold no false value: every output value is true
    const bool walk = NUM && (SR::id != SPGEMM_OR_AND_BOOL || vals_zero == nullptr || *vals_zero != 0);
    // the groups of a warp go round together (their shuffles name the whole warp)
    const int64_t step = (int64_t)gridDim.x * NG;
    for (int64_t w0 = (int64_t)blockIdx.x * NG + (grp & ~(32 / G - 1)); w0 < count; w0 += step) {
        const int64_t w = w0 + (grp & (32 / G - 1));
        const bool act = w < count;
        int2 e = make_int2(0, 0);
        if (act) e = __ldg(list + w);
        const Prod* pr = it.prods + e.x;
        const int64_t u = __ldg(it.item_base + e.x) + e.y;
        int64_t bs = 0, be = 0;
        if (act) {
            bs = __ldg(pr->B.cp + e.y);
            be = __ldg(pr->B.cp + e.y + 1);
        }
        const uint32_t m = (uint32_t)pr->A.m;
        const bool b_one = __all_sync(0xffffffffu, pr->B.num == nullptr);   // of every group of the warp
        // 1. products: the entries of B(:,j) G at a time (the bin bounds their products by N),
        //    U products per lane in flight; product p to slot p (however many entries they come
        //    from: keys kept in registers made every G entries pay for all K slots, 499 us
        //    for the 361 above)
        constexpr int U = K == 2 ? 1 : K <= 8 ? 2 : 4;
        int base = 0;
        for (int64_t b0 = bs; __any_sync(0xffffffffu, b0 < be && base < N); b0 += G) {
            const int64_t t = b0 + lane;
            int len = 0;
            int64_t a0 = 0;
            T bv = T(0);
            if (t < be) {
                const int32_t k = __ldg(pr->B.ir + t);
                int64_t sa, ea;
                a_col(it, pr, t, k, sa, ea);
                a0 = sa;
                len = (int)(ea - sa);
                if (walk) bv = load_val<SR>(pr->B, t);
            }
            const int inc = scan_g<G>(len, lane);
            const int tot = min(__shfl_sync(0xffffffffu, inc, G - 1, G), N - base);
            a0 -= inc - len;   // product q of the chunk is at a0 + q of its entry
            for (int q0 = lane; __any_sync(0xffffffffu, q0 < tot); q0 += G * U) {
                int32_t row[U];
                T av[U], bvs[U];
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    const int q = q0 + i * G;
                    int src = 0;                         // entries that end at or before product q
#pragma unroll
                    for (int st = G / 2; st > 0; st >>= 1)
                        if (__shfl_sync(0xffffffffu, inc, src + st - 1, G) <= q) src += st;
                    const int64_t as = __shfl_sync(0xffffffffu, a0, src, G);
                    bvs[i] = T(0);
                    av[i] = T(0);
                    if constexpr (NUM) bvs[i] = shflg<G>(bv, src);
                    row[i] = -1;
                    if (q < tot) {
                        row[i] = __ldg(pr->A.ir + as + q);
                        if (walk) av[i] = load_val<SR>(pr->A, as + q);
                    }
                }
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    const int q = q0 + i * G;
                    if (q < tot) {
                        const int slot = base + q;
                        // a row outside A is malformed input: skipped
                        sk[st_ph(slot)] = (uint32_t)row[i] < m ? ((uint32_t)row[i] << SB) | (uint32_t)slot : NONE;
                        if constexpr (NUM) sv[st_ph(slot)] = walk ? mul_by<SR>(av[i], bvs[i], b_one) : SR::one();
                    }
                }
            }
            base += tot;
        }
        __syncwarp();
        uint32_t key[K];
#pragma unroll
        for (int r = 0; r < K; ++r) {
            const int i = r * G + lane;
            key[r] = i < base ? sk[st_ph(i)] : NONE;
        }
        // 2. order
        sort_keys<G, K>(key, lane);
        // 3. runs of equal rows: the last element of a run holds its sum
        const uint32_t first = key[0] >> SB, last = key[K - 1] >> SB;
        uint32_t before = __shfl_up_sync(0xffffffffu, last, 1, G), after = __shfl_down_sync(0xffffffffu, first, 1, G);
        if (lane == 0) before = NOROW;
        if (lane == G - 1) after = NOROW;
        uint32_t end = 0;   // bit r: element r is the last of its run
#pragma unroll
        for (int r = 0; r < K; ++r) {
            const uint32_t nx = r + 1 < K ? key[r + 1 < K ? r + 1 : r] >> SB : after;
            if (key[r] != NONE && nx != (key[r] >> SB)) end |= 1u << r;
        }
        const int c = __popc(end);
        const int inc = scan_g<G>(c, lane);
        const int cnt = __shfl_sync(0xffffffffu, inc, G - 1, G);
        if constexpr (!NUM) {
            if (act && lane == 0) nnz_item[u] = cnt;
            __syncwarp();   // the slots are free for the next column
        } else {
            __syncwarp();
            // a run's sum goes to the slot of its last element, which no other lane touches
            Acc acc = SR::zero();
            uint32_t head = NONE;   // the last element of the lane's first run, if it ends here
#pragma unroll
            for (int r = 0; r < K; ++r) {
                Acc* slot = sv + st_ph((int)(key[r] & (N - 1)));
                const Acc x = key[r] != NONE ? *slot : SR::zero();
                bool same = false;
                if (r > 0) same = key[r] != NONE && (key[r] >> SB) == (key[r > 0 ? r - 1 : 0] >> SB);
                if (r > 0 && __any_sync(0xffffffffu, same)) acc = same ? SR::add(acc, x) : x;
                else acc = x;
                if ((end >> r) & 1u) {
                    *slot = acc;
                    if ((key[r] >> SB) == first) head = key[r];
                }
            }
            // a run that continues the lane before's last one takes that lane's sum
            const bool cont = key[0] != NONE && before == first;
            if (__any_sync(0xffffffffu, cont)) {
                Acc s = acc;
                int through = cont && last == first && key[K - 1] != NONE;   // one run, from the lane before's
#pragma unroll
                for (int d = 1; d < G; d <<= 1) {
                    const Acc sp = shflg<G>(s, lane >= d ? lane - d : lane);
                    const int tp = __shfl_up_sync(0xffffffffu, through, d, G);
                    if (lane >= d && through) {
                        s = SR::add(sp, s);
                        through = tp;
                    }
                }
                const Acc carry = shflg<G>(s, lane > 0 ? lane - 1 : 0);
                if (cont && head != NONE) {
                    Acc* slot = sv + st_ph((int)(head & (N - 1)));
                    *slot = SR::add(carry, *slot);
                }
            }
            // 4. the last elements of the runs in order, then coalesced stores
            int pos = inc - c;
#pragma unroll
            for (int r = 0; r < K; ++r)
                if ((end >> r) & 1u) sk[st_ph(pos++)] = key[r];
            __syncwarp();
            if (act) {
                const int64_t out0 = __ldg(Coff + u);
                const int64_t capn = __ldg(Coff + u + 1) - out0;
                if (nnz_item && lane == 0) nnz_item[u] = cnt;
                // exact offsets always fit; with nnz_item a column that does not fit its
                // slots is only counted
                if (cnt <= capn) {
                    const int32_t rb = out_row_base(pr, e.y);
                    for (int i = lane; i < cnt; i += G) {
                        const uint32_t k = sk[st_ph(i)];
                        __stcs(Cir + out0 + i, (int32_t)(k >> SB) + rb);
                        Cv[out0 + i] = SR::out(sv[st_ph((int)(k & (N - 1)))]);
                    }
                }
            }
            __syncwarp();   // the slots are free for the next column
        }
    }
}

template <class SR, int G, int K, bool NUM>
void run(const Lanes& st, const Items& it, const int2* list, int64_t count, int64_t* nnz_item, const int64_t* Coff,
         int32_t* Cir, typename SR::T* Cv, const int* vals_zero) {
    if (count <= 0) return;
    const int grid = (int)std::min<int64_t>(ceil_div64(count, st_block(K) / G), (int64_t)sm_count() * 32);
    k_sort<SR, G, K, NUM><<<grid, st_block(K), 0, st.next()>>>(it, list, count, nnz_item, Coff, Cir, Cv, vals_zero);
    note_launch();
}

template <class SR, bool NUM>
void run_bins(const Lanes& st, const Items& it, const int2* list, const int64_t* off, const int64_t* cnt,
              int64_t* nnz_item, const int64_t* Coff, int32_t* Cir, typename SR::T* Cv, const int* vz) {
    constexpr int S = BIN_SORT0;
    run<SR, 8, 2, NUM>(st, it, list + off[S], cnt[S], nnz_item, Coff, Cir, Cv, vz);
    run<SR, 8, 4, NUM>(st, it, list + off[S + 1], cnt[S + 1], nnz_item, Coff, Cir, Cv, vz);
    run<SR, 8, 8, NUM>(st, it, list + off[S + 2], cnt[S + 2], nnz_item, Coff, Cir, Cv, vz);
    run<SR, 16, 8, NUM>(st, it, list + off[S + 3], cnt[S + 3], nnz_item, Coff, Cir, Cv, vz);
    run<SR, 32, 8, NUM>(st, it, list + off[S + 4], cnt[S + 4], nnz_item, Coff, Cir, Cv, vz);
    run<SR, 32, 16, NUM>(st, it, list + off[S + 5], cnt[S + 5], nnz_item, Coff, Cir, Cv, vz);
    run<SR, 32, 32, NUM>(st, it, list + off[S + 6], cnt[S + 6], nnz_item, Coff, Cir, Cv, vz);
}

}  // namespace

template <class SR>
void launch_sort_tier(const Lanes& st, const Items& it, const int2* list, const int64_t* bin_off,
                      const int64_t* bin_cnt, int64_t* nnz_item, const int64_t* Coff, int32_t* Cir,
                      typename SR::T* Cv, const int* vals_zero) {
    run_bins<SR, true>(st, it, list, bin_off, bin_cnt, nnz_item, Coff, Cir, Cv, vals_zero);
}

void launch_sort_count(const Lanes& st, const Items& it, const int2* list, const int64_t* bin_off,
                       const int64_t* bin_cnt, int64_t* nnz_item) {
    run_bins<MP32, false>(st, it, list, bin_off, bin_cnt, nnz_item, nullptr, nullptr, nullptr, nullptr);
}

#define SG_INST(SR)                                                                                             \
    template void launch_sort_tier<SR>(const Lanes&, const Items&, const int2*, const int64_t*, const int64_t*, \
                                       int64_t*, const int64_t*, int32_t*, typename SR::T*, const int*);
SG_INST(PT64)
SG_INST(MP32)
SG_INST(BOOL8)
SG_INST(PTI64)
#undef SG_INST

}  // namespace sg
