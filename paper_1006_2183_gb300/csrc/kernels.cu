// Batched column-wise SpGEMM kernels (Gustavson's column-by-column
// formulation, Section 2.1; accumulation in the spirit of the sparse
// accumulator of Section 3.3), organised in accumulator tiers chosen per
// output column from cap = min(flops, m):
//   * up to 1024 products: sorted in the registers of 8 to 32 lanes (sorttier.cu),
//   * warp-wide shared-memory hash tables (short columns of many products),
//   * CTA-wide shared-memory hash tables (medium columns),
//   * the slab tier (long columns): row slabs, each counted through a row bitmap in
//     shared memory and accumulated at its rows' ranks.
// The symbolic pass counts nnz per output column; the numeric pass fills rows
// and values, in ascending row order without a sort wherever a row bitmap fits
// in shared memory.  Every kernel works on items (product, stored column of B).
#include <algorithm>
#include <atomic>
#include <climits>
#include <map>
#include <mutex>
#include <utility>

#include "kernels.cuh"

namespace sg {

static std::atomic<int64_t> g_launches{0};
void note_launch(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
int64_t launches() { return g_launches.load(std::memory_order_relaxed); }

int sm_count() {
    static std::mutex mu;
    static std::map<int, int> cache;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    auto f = cache.find(dev);
    if (f != cache.end()) return f->second;
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
        cudaGetLastError();
        return 1;   // not cached: asked again next time
    }
    cache[dev] = n;
    return n;
}

bool LanePool::init() {
    if (ready || failed) return ready;
    failed = cudaEventCreateWithFlags(&start, cudaEventDisableTiming) != cudaSuccess;
    for (int i = 0; i < NSIDE && !failed; ++i)
        failed = cudaStreamCreateWithFlags(&side[i], cudaStreamNonBlocking) != cudaSuccess ||
                 cudaEventCreateWithFlags(&done[i], cudaEventDisableTiming) != cudaSuccess;
    if (failed) {
        cudaGetLastError();   // passes then stay on one stream
        destroy();
        failed = true;
    }
    ready = !failed;
    return ready;
}

void LanePool::destroy() {
    if (start) cudaEventDestroy(start);
    for (int i = 0; i < NSIDE; ++i) {
        if (done[i]) cudaEventDestroy(done[i]);
        if (side[i]) cudaStreamDestroy(side[i]);
        done[i] = nullptr;
        side[i] = nullptr;
    }
    start = nullptr;
    ready = failed = false;
}

Lanes::Lanes(cudaStream_t main, LanePool* pool) : main_(main) {
    if (pool && pool->init() && cudaEventRecord(pool->start, main) == cudaSuccess) pool_ = pool;
}

cudaStream_t Lanes::next() const {
    const int t = turn_++ % (LanePool::NSIDE + 1);
    if (!pool_ || t == 0) return main_;
    const int i = t - 1;
    if (!used_[i]) {
        if (cudaStreamWaitEvent(pool_->side[i], pool_->start, 0) != cudaSuccess) return main_;
        used_[i] = true;
    }
    return pool_->side[i];
}

Lanes::~Lanes() {
    for (int i = 0; i < LanePool::NSIDE; ++i)
        if (used_[i]) {
            // should the join fail, the host waits instead: later work must not start early
            if (cudaEventRecord(pool_->done[i], pool_->side[i]) != cudaSuccess ||
                cudaStreamWaitEvent(main_, pool_->done[i], 0) != cudaSuccess)
                cudaStreamSynchronize(pool_->side[i]);
        }
}

// Raises a kernel's dynamic shared-memory limit on the current device to at least
// `bytes`; never lowers it (the limit belongs to the kernel, whichever launcher
// asks).  A refused request is not remembered, so the launch reports the error.
void smem_at_least(const void* fn, size_t bytes) {
    static std::mutex mu;
    static std::map<std::pair<int, const void*>, size_t> limit;
    int dev = 0;
    cudaGetDevice(&dev);
    std::lock_guard<std::mutex> lk(mu);
    size_t& cur = limit[{dev, fn}];
    if (cur < bytes && cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess)
        cur = bytes;
}

constexpr int WARP_BLOCK = 256;   // 8 warp groups per CTA

__host__ __device__ __forceinline__ int bin_of(int64_t flops, int64_t cap, int warp_max, int block_max,
                                              int sort_max) {
    if (cap <= 0) return 0;
    if (flops <= TINY_MAX) return BIN_SORT0;
    if (flops <= sort_max && cap <= block_max) {   // block_max is no smaller than warp_max
        int b = BIN_SORT0 + 1;
        for (int64_t t = 2 * TINY_MAX; t < flops; t <<= 1) ++b;
        return b;
    }
    if (cap <= warp_max) {
        int64_t t = WARP_TBL0;
        int b = BIN_WARP0;
        while (t < 2 * cap) { t <<= 1; ++b; }
        return b;
    }
    if (cap <= block_max) {
        int64_t t = BLK_TBL0;
        int b = BIN_BLK0;
        while (t < 2 * cap) { t <<= 1; ++b; }
        return b;
    }
    return BIN_DENSE;
}

__device__ __forceinline__ int find_prod(const int64_t* __restrict__ base, int64_t nprod, int64_t u) {
    // last product i with base[i] <= u
    int64_t lo = 0, hi = nprod - 1;
    while (lo < hi) {
        int64_t mid = (lo + hi + 1) >> 1;
        if (__ldg(base + mid) <= u) lo = mid;
        else hi = mid - 1;
    }
    return (int)lo;
}

__device__ __forceinline__ int64_t out_col(const DMat& B, int64_t p) { return B.jc ? __ldg(B.jc + p) : p; }

// ------------------------------------------------------------------ analysis
// Groups of LPI lanes per item (8; 1 where B columns are short, as in the block
// products; 32 where they hold 32 entries and more on average): flops = sum_k nnz(A(:,k)) (Section 1's flops), the tier bin,
// the product id, and optionally the predictor inputs.
// A lookup is a chain of dependent loads (B's row, A's column pointers), so a hub column
// of B on its 8 lanes was the whole kernel's time (23,356 entries at R-MAT scale 20: a
// chain of 2,900 lookups).  Columns longer than ANALYZE_LONG entries are walked by the
// whole CTA, four lookups in flight per thread: R-MAT 20 flat 1.73 -> 0.29 ms, R-MAT of
// 300,007 vertices 0.67 -> 0.16 ms.  Shorter ones stay on their lanes: up to 32 rounds of
// 8 lanes cost less than a pass of the CTA of their own.  Items strided over the CTAs (the
// hubs of an R-MAT graph sit side by side) took 0.42 ms at R-MAT 20: their pointers and
// results no longer share sectors.
constexpr int ANALYZE_LONG = 256;

// lookup of A(:,k) for entry t of B(:,j): its length, stored in the A-column cache if there is one
__device__ __forceinline__ long long analyze_entry(const Items& it, const DMat& A, int32_t k, int64_t cache_at) {
    int64_t cs, ce;
    col_range(A, k, cs, ce);
    if (it.acs) {
        it.acs[cache_at] = cs;
        it.acl[cache_at] = (int32_t)(ce - cs);
    }
    return ce - cs;
}

template <int LPI>
__global__ void __launch_bounds__(256) k_analyze(Items it, TierCfg cfg, int64_t* __restrict__ flops,
                                                 uint8_t* __restrict__ bin, int32_t* __restrict__ item_prod,
                                                 unsigned long long* bin_count, unsigned long long* flops_total,
                                                 const uint64_t* __restrict__ sketch,
                                                 const int64_t* __restrict__ sketch_base, float* __restrict__ feat,
                                                 int64_t* __restrict__ maxlen, int64_t* __restrict__ nnz_item) {
    constexpr int GRP = 256 / LPI;   // items of this CTA
    __shared__ unsigned long long s_cnt[NBIN];
    __shared__ unsigned long long s_fl, s_sort2;
    __shared__ int s_nlong;
    __shared__ int s_long[GRP];                                              // groups with a long column
    __shared__ unsigned long long s_lf[GRP], s_lmx[GRP], s_lsk[GRP];         // their totals
    if (threadIdx.x < NBIN) s_cnt[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        s_fl = s_sort2 = 0;
        s_nlong = 0;
    }
    __syncthreads();
    const int sub = threadIdx.x & (LPI - 1), grp = threadIdx.x / LPI;
    const int64_t u = (int64_t)blockIdx.x * GRP + grp;
    long long f = 0, mx = 0;
    unsigned long long sk = 0;
    int64_t bs = 0, be = 0, am = 0;
    int prod = 0;
    bool is_long = false;
    if (u < it.nitems) {
        prod = it.nprod == 1 ? 0 : __ldg(item_prod + u);   // filled per product beforehand
        const Prod* pr = it.prods + prod;
        const int64_t p = u - __ldg(it.item_base + prod);
        bs = __ldg(pr->B.cp + p);
        be = __ldg(pr->B.cp + p + 1);
        am = pr->A.m;
        const uint64_t* skp = sketch ? sketch + sketch_base[prod] : nullptr;
        const int64_t b0 = it.acs ? pr->bnz_base - __ldg(pr->B.cp) : 0;
        is_long = be - bs > ANALYZE_LONG;
        if (is_long) {
            if (sub == 0) {
                s_lf[grp] = s_lmx[grp] = s_lsk[grp] = 0;
                s_long[atomicAdd(&s_nlong, 1)] = grp;
            }
        } else if constexpr (LPI == 1) {
            // two entries of B(:,j) at a time, each step of their A-column lookups issued
            // for both before either is used (a lookup is a chain of dependent loads: B's
            // row, then AUX, then JC, then CP)
            const DMat& A = pr->A;
            for (int64_t t0 = bs; t0 < be; t0 += 2) {
                int32_t k[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) k[i] = t0 + i < be ? __ldg(pr->B.ir + t0 + i) : -1;
                int64_t cs[2], ce[2];
                col_range2(A, k, cs, ce);
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    if (t0 + i >= be) break;
                    const long long len = ce[i] - cs[i];
                    if (it.acs) {   // fill the A-column cache for the later passes
                        it.acs[b0 + t0 + i] = cs[i];
                        it.acl[b0 + t0 + i] = (int32_t)len;
                    }
                    f += len;
                    mx = len > mx ? len : mx;
                    if (skp && k[i] >= 0 && k[i] < A.n) sk |= __ldg(skp + k[i]);
                }
            }
        } else {
            for (int64_t t = bs + sub; t < be; t += LPI) {
                const int32_t k = __ldg(pr->B.ir + t);
                const long long len = analyze_entry(it, pr->A, k, b0 + t);
                f += len;
                mx = len > mx ? len : mx;
                if (skp && k >= 0 && k < pr->A.n) sk |= __ldg(skp + k);
            }
        }
    }
    __syncthreads();
    const int nlong = s_nlong;
    for (int l = 0; l < nlong; ++l) {   // the CTA's long columns, one after another
        const int g = s_long[l];
        const int64_t ul = (int64_t)blockIdx.x * GRP + g;
        const int lp = it.nprod == 1 ? 0 : __ldg(item_prod + ul);
        const Prod* pr = it.prods + lp;
        const int64_t p = ul - __ldg(it.item_base + lp);
        const int64_t s0 = __ldg(pr->B.cp + p), e0 = __ldg(pr->B.cp + p + 1);
        const uint64_t* skp = sketch ? sketch + sketch_base[lp] : nullptr;
        const int64_t b0 = it.acs ? pr->bnz_base - __ldg(pr->B.cp) : 0;
        long long lf = 0, lmx = 0;
        unsigned long long lsk = 0;
        constexpr int U = 4;
        for (int64_t t0 = s0 + threadIdx.x; t0 < e0; t0 += 256 * U) {
            int32_t k[U];
            long long len[U];
#pragma unroll
            for (int i = 0; i < U; ++i) k[i] = t0 + 256 * i < e0 ? __ldg(pr->B.ir + t0 + 256 * i) : -1;
#pragma unroll
            for (int i = 0; i < U; ++i)
                len[i] = t0 + 256 * i < e0 ? analyze_entry(it, pr->A, k[i], b0 + t0 + 256 * i) : 0;
#pragma unroll
            for (int i = 0; i < U; ++i) {
                lf += len[i];
                lmx = len[i] > lmx ? len[i] : lmx;
                if (skp && k[i] >= 0 && k[i] < pr->A.n) lsk |= __ldg(skp + k[i]);
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            lf += __shfl_xor_sync(0xffffffffu, lf, o);
            const long long om = __shfl_xor_sync(0xffffffffu, lmx, o);
            lmx = om > lmx ? om : lmx;
            lsk |= __shfl_xor_sync(0xffffffffu, lsk, o);
        }
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&s_lf[g], (unsigned long long)lf);
            atomicMax(&s_lmx[g], (unsigned long long)lmx);   // lengths are not negative
            if (lsk) atomicOr(&s_lsk[g], lsk);
        }
    }
    if (nlong > 0) __syncthreads();
    if (is_long && sub == 0) {
        f = (long long)s_lf[grp];
        mx = (long long)s_lmx[grp];
        sk = s_lsk[grp];
    }
#pragma unroll
    for (int o = LPI / 2; o > 0; o >>= 1) {
        f += __shfl_xor_sync(0xffffffffu, f, o, LPI);
        long long om = __shfl_xor_sync(0xffffffffu, mx, o, LPI);
        mx = om > mx ? om : mx;
        sk |= __shfl_xor_sync(0xffffffffu, sk, o, LPI);
    }
    const bool has = u < it.nitems && sub == 0;
    const int64_t cap = f < am ? f : am;
    const int b = has ? bin_of(f, cap, cfg.warp_max, cfg.block_max, cfg.sort_max) : -1;
    {
        // per-bin counts and total flops, one shared atomic per bin per warp (every
        // item of a CTA adding to the same few counters serialises on them)
        const unsigned peers = __match_any_sync(0xffffffffu, b);
        const int lane = threadIdx.x & 31;
        if (has && lane == __ffs(peers) - 1) atomicAdd(&s_cnt[b], (unsigned long long)__popc(peers));
        const unsigned over = __ballot_sync(0xffffffffu, b > BIN_SORT0 && b < BIN_WARP0 && cap > cfg.warp_max);
        if (lane == 0 && over) atomicAdd(&s_sort2, (unsigned long long)__popc(over));
        unsigned long long fs = has ? (unsigned long long)f : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) fs += __shfl_xor_sync(0xffffffffu, fs, o);
        if (lane == 0 && fs) atomicAdd(&s_fl, fs);
    }
    if (has) {
        flops[u] = f;
        if (it.nprod == 1) item_prod[u] = 0;
        bin[u] = (uint8_t)b;
        nnz_item[u] = 0;   // of the empty columns; the counting passes write the others
        if (maxlen) maxlen[u] = mx;
        if (feat) {
            // predictor inputs (definitions in predictor.cu)
            float d = (float)(be - bs);
            int pc = __popcll(sk);
            float pcf = fminf((float)pc, 63.5f);
            float lc = 64.0f * logf(64.0f / (64.0f - pcf));
            float* x = feat + u * 8;
            x[0] = log1pf(d);
            x[1] = log1pf((float)f);
            x[2] = log1pf((float)mx);
            x[3] = log1pf((float)am);
            x[4] = log1pf(lc);
            x[5] = log1pf((float)cap);
            x[6] = log1pf((float)(f - mx));
            x[7] = (float)pc * (1.0f / 64.0f);
        }
    }
    __syncthreads();
    // the counters are kept in CTR_REP copies on lines of their own (32,768 CTAs adding to
    // one line would queue in one L2 slice)
    const int rep = (blockIdx.x & (CTR_REP - 1)) * CTR_STRIDE;
    if (threadIdx.x < NBIN && s_cnt[threadIdx.x]) atomicAdd(bin_count + rep + threadIdx.x, s_cnt[threadIdx.x]);
    if (threadIdx.x == 0 && flops_total) atomicAdd(flops_total + rep, s_fl);
    if (threadIdx.x == 32 && s_sort2) atomicAdd(bin_count + rep + CTR_SORT2, s_sort2);
}

// item_prod[u] = the product of item u: one CTA per product over its contiguous items.
__global__ void k_item_prod(Items it, int32_t* __restrict__ item_prod) {
    const int64_t p = blockIdx.x;
    const int64_t u0 = __ldg(it.item_base + p), u1 = __ldg(it.item_base + p + 1);
    for (int64_t u = u0 + threadIdx.x; u < u1; u += blockDim.x) item_prod[u] = (int32_t)p;
}

void launch_analyze(cudaStream_t st, const Items& it, TierCfg cfg, int64_t* flops, uint8_t* bin, int32_t* item_prod,
                    unsigned long long* bin_count, unsigned long long* flops_total, const uint64_t* sketch,
                    const int64_t* sketch_base, float* feat, int64_t* maxlen, int64_t* nnz_item) {
    if (it.nitems == 0) return;
    if (it.nprod > 1) {
        k_item_prod<<<(unsigned)it.nprod, 256, 0, st>>>(it, item_prod);
        note_launch();
    }
    if (it.total_bnz < 4 * it.nitems) {   // about one B entry per item: one lane each
        int grid = (int)ceil_div64(it.nitems, 256);
        k_analyze<1><<<grid, 256, 0, st>>>(it, cfg, flops, bin, item_prod, bin_count, flops_total, sketch,
                                           sketch_base, feat, maxlen, nnz_item);
    } else if (it.total_bnz >= 32 * it.nitems) {
        int grid = (int)ceil_div64(it.nitems * 32, 256);
        k_analyze<32><<<grid, 256, 0, st>>>(it, cfg, flops, bin, item_prod, bin_count, flops_total, sketch,
                                            sketch_base, feat, maxlen, nnz_item);
    } else {
        int grid = (int)ceil_div64(it.nitems * 8, 256);
        k_analyze<8><<<grid, 256, 0, st>>>(it, cfg, flops, bin, item_prod, bin_count, flops_total, sketch,
                                           sketch_base, feat, maxlen, nnz_item);
    }
    note_launch();
}

// sketch(A(:,k)) = OR over rows i of 2^(bits 31..26 of i * 0x9E3779B1)
__global__ void k_row_sketch(DMat A, uint64_t* __restrict__ sk) {
    int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3;
    int sub = threadIdx.x & 7;
    unsigned long long v = 0;
    if (p < A.nzc) {
        int64_t s = __ldg(A.cp + p), e = A.ce ? __ldg(A.ce + p) : __ldg(A.cp + p + 1);
        for (int64_t t = s + sub; t < e; t += 8) {
            uint32_t h = (uint32_t)__ldg(A.ir + t) * 0x9E3779B1u;
            v |= 1ull << (h >> 26);
        }
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v |= __shfl_xor_sync(0xffffffffu, v, o, 8);
    if (p < A.nzc && sub == 0) sk[A.jc ? __ldg(A.jc + p) : p] = v;
}

void launch_row_sketch(cudaStream_t st, const DMat& A, uint64_t* sketch) {
    if (A.jc) cudaMemsetAsync(sketch, 0, sizeof(uint64_t) * std::max<int64_t>(A.n, 1), st);
    if (A.nzc == 0) return;
    k_row_sketch<<<(int)ceil_div64(A.nzc * 8, 256), 256, 0, st>>>(A, sketch);
    note_launch();
}

// Where every bin's list starts (s_off, NBIN entries) from the bins' counts, kept in `rep`
// copies CTR_STRIDE apart.  Called by all threads of a CTA; ends with a barrier.
__device__ __forceinline__ void bin_offsets(const unsigned long long* cnt, int rep, int64_t* s_off) {
    if (threadIdx.x < 32) {
        const int b = threadIdx.x;
        long long c = 0;
        if (b < NBIN)
            for (int r = 0; r < rep; ++r) c += (long long)__ldcg(cnt + r * CTR_STRIDE + b);
        const long long inc = warp_incl_scan64(c);
        if (b < NBIN) s_off[b] = inc - c;
    }
    __syncthreads();
}

// Where one thread's entry of bin b (<= 0: not listed) goes among the CTA's entries of that
// bin, which s_n counts.  Whole warps call it.
__device__ __forceinline__ int bin_rank(int b, int* s_n) {
    const unsigned peers = __match_any_sync(0xffffffffu, b);
    const int lane = threadIdx.x & 31, leader = __ffs(peers) - 1;
    int at = 0;
    if (b > 0 && lane == leader) at = atomicAdd(&s_n[b], __popc(peers));
    return __shfl_sync(0xffffffffu, at, leader) + __popc(peers & ((1u << lane) - 1));
}

// Where the CTA's entries of every bin start in the lists: one global addition per bin.  All
// threads call it, after a barrier; ends with one.
__device__ __forceinline__ void bin_bases(unsigned long long* cursor, const int64_t* s_off, const int* s_n,
                                          int64_t* s_base) {
    if (threadIdx.x < NBIN && threadIdx.x > 0 && s_n[threadIdx.x] > 0)
        s_base[threadIdx.x] = s_off[threadIdx.x] +
                              (int64_t)atomicAdd(cursor + threadIdx.x, (unsigned long long)s_n[threadIdx.x]);
    __syncthreads();
}

// One bin per thread (b <= 0: not listed): its place in the list of bin b, whose entries
// before this CTA's come from one global addition per bin.  All threads call it.
__device__ __forceinline__ int64_t list_place(int b, unsigned long long* cursor, const int64_t* s_off, int* s_n,
                                              int64_t* s_base) {
    if (threadIdx.x < NBIN) s_n[threadIdx.x] = 0;
    __syncthreads();
    const int at = bin_rank(b, s_n);
    __syncthreads();
    bin_bases(cursor, s_off, s_n, s_base);
    return b > 0 ? s_base[b] + at : 0;
}

// Scatter of items into per-bin lists, whose offsets every CTA makes from the counts (and
// CTA 0 leaves in off_out), so that the launch waits for no host.
__global__ void __launch_bounds__(256) k_bin_scatter(Items it, const uint8_t* __restrict__ bin,
                                                     const int32_t* __restrict__ item_prod,
                                                     const unsigned long long* __restrict__ cnt, int rep,
                                                     unsigned long long* cursor, int64_t* __restrict__ off_out,
                                                     int2* __restrict__ list) {
    __shared__ int64_t s_off[NBIN], s_base[NBIN];
    __shared__ int s_n[NBIN];
    bin_offsets(cnt, rep, s_off);
    if (blockIdx.x == 0 && threadIdx.x < NBIN) off_out[threadIdx.x] = s_off[threadIdx.x];
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int b = u < it.nitems ? bin[u] : -1;
    const int64_t at = list_place(b, cursor, s_off, s_n, s_base);
    if (b > 0) {
        const int prod = item_prod[u];
        list[at] = make_int2(prod, (int)(u - __ldg(it.item_base + prod)));
    }
}

void launch_bin_scatter(cudaStream_t st, const Items& it, const uint8_t* bin, const int32_t* item_prod,
                        const unsigned long long* cnt, int rep, unsigned long long* cursor, int64_t* off_out,
                        int2* list) {
    if (it.nitems == 0) return;
    k_bin_scatter<<<(int)ceil_div64(it.nitems, 256), 256, 0, st>>>(it, bin, item_prod, cnt, rep, cursor, off_out, list);
    note_launch();
}

// ------------------------------------------------------------------ hash tiers
template <class SR, int GS, int TBL, bool NUM>
struct HashLayout {
    using T = typename SR::T;
    using Acc = typename SR::Acc;
    static constexpr size_t keys = (size_t)TBL * 4;
    static constexpr size_t vals = NUM ? (size_t)TBL * sizeof(Acc) : 0;
    static constexpr size_t incl = (size_t)GS * 4;
    static constexpr size_t a0 = (size_t)GS * 8;
    static constexpr size_t bv = NUM ? (size_t)GS * 8 : 0;
    static constexpr size_t scan = 33 * 4 + 4;
    static constexpr size_t group = (keys + vals + incl + a0 + bv + scan + 15) / 16 * 16;
};

template <int GS, class Acc>
__device__ __forceinline__ void bitonic_sort(int32_t* keys, Acc* vals, int P) {
    using G = Group<GS>;
    const int lane = G::lane();
    for (int k = 2; k <= P; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            for (int t = lane; t < (P >> 1); t += GS) {
                int i = ((t & ~(j - 1)) << 1) | (t & (j - 1));
                int l = i + j;
                bool asc = (i & k) == 0;
                int32_t ki = keys[i], kl = keys[l];
                if ((ki > kl) == asc) {
                    keys[i] = kl;
                    keys[l] = ki;
                    Acc vi = vals[i];
                    vals[i] = vals[l];
                    vals[l] = vi;
                }
            }
            G::sync();
        }
    }
}

// Writes a group's table in row order: the rank of row r among the marked rows of
// `bitmap` (nw words) is the number of bits below it, from per-member prefix counts
// of groups of gw words plus the popcounts inside r's group, so every occupied slot
// writes its entry at its rank directly (no sort, no probing).  Empties the table
// and the bitmap.  Called by all GS members; returns the number of entries.  With
// `pred`, nothing is written when the count exceeds capn.
template <class SR, int TBL, int GS>
__device__ __forceinline__ int rank_emit(uint32_t* bitmap, uint16_t* wp, int nw, int32_t* keys,
                                         typename SR::Acc* vals, int* gp, int* scratch, bool pred, int64_t capn,
                                         int64_t out0, int32_t rb, int32_t* __restrict__ Cir,
                                         typename SR::T* __restrict__ Cv) {
    using G = Group<GS>;
    const int lane = G::lane();
    int lgw = 0;   // words per member: a power of two with GS members covering nw words
    while ((GS << lgw) < nw) ++lgw;
    const int gw = 1 << lgw;
    // wp[x]: set bits before word x within its member's words (< 2^16: gw <= 2^11)
    int c = 0;
    for (int x = lane * gw; x < (lane + 1) * gw && x < nw; ++x) {
        wp[x] = (uint16_t)c;
        c += __popc(bitmap[x]);
    }
    int total;
    const int incl = group_incl_scan<GS>(c, scratch, total);
    gp[lane] = incl - c;
    G::sync();
    const bool write = !pred || total <= capn;
    for (int s = lane; s < TBL; s += GS) {
        const int32_t kr = keys[s];
        if (kr < 0) continue;
        const int wd = kr >> 5;
        if (wd < nw && write) {   // rows past the bitmap occur only on malformed input
            const int rank = gp[wd >> lgw] + wp[wd] + __popc(bitmap[wd] & ((1u << (kr & 31)) - 1u));
            Cir[out0 + rank] = kr + rb;
            Cv[out0 + rank] = SR::out(vals[s]);
        }
        keys[s] = -1;
        vals[s] = SR::zero();
    }
    G::sync();
    for (int x = lane; x < nw; x += GS) bitmap[x] = 0u;
    G::sync();
    return total;
}

// The hash tables are latency-bound: registers are capped so that they never admit
// fewer CTAs per SM than shared memory does (48 warps for warp tables, tables of 2
// or 4 warps and 2048-slot CTA tables; 4 CTAs of 4096 slots; 2 CTAs of 512 threads).
constexpr int hash_min_blocks(int block, int tbl) {
    return block <= 128 ? 1536 / block : block == 256 ? (tbl <= 2048 ? 6 : 4) : 2;
}

template <class SR, int GS, int TBL, bool NUM, int BLOCK>
__global__ void __launch_bounds__(BLOCK, hash_min_blocks(BLOCK, TBL)) k_hash(Items it, const int2* __restrict__ list, int64_t count,
                                                int64_t* __restrict__ nnz_item, const int64_t* __restrict__ Coff,
                                                int32_t* __restrict__ Cir, typename SR::T* __restrict__ Cv,
                                                int bm_words) {
    using T = typename SR::T;
    using Acc = typename SR::Acc;
    using L = HashLayout<SR, GS, TBL, NUM>;
    using G = Group<GS>;
    constexpr int NG = BLOCK / GS;
    constexpr int LOG2 = __builtin_ctz(TBL);
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = G::lane();
    const int g = G::gid();
    unsigned char* base = smem + (size_t)g * L::group;
    int32_t* keys = reinterpret_cast<int32_t*>(base);
    Acc* vals = reinterpret_cast<Acc*>(base + L::keys);
    int* s_incl = reinterpret_cast<int*>(base + L::keys + L::vals);
    int64_t* s_a0 = reinterpret_cast<int64_t*>(base + L::keys + L::vals + L::incl);
    T* s_bv = reinterpret_cast<T*>(base + L::keys + L::vals + L::incl + L::a0);
    int* s_scan = reinterpret_cast<int*>(base + L::keys + L::vals + L::incl + L::a0 + L::bv);
    int* s_cnt = s_scan + 33;
    volatile int32_t* vkeys = keys;
    // Numeric tables order their output through a row bitmap (one per group) when
    // the rows fit; otherwise they compact and sort.
    uint32_t* bitmap = reinterpret_cast<uint32_t*>(smem + (size_t)NG * L::group) + (size_t)g * bm_words;
    // per-word prefixes of the bitmap, after the bitmaps of all groups
    uint16_t* wp = reinterpret_cast<uint16_t*>(smem + (size_t)NG * L::group + (size_t)NG * bm_words * 4) +
                   (size_t)g * bm_words;
    constexpr bool CAN_BM = NUM && (GS == BLOCK || (GS == 32 && TBL >= BM_WARP_MIN_TBL));
    if constexpr (CAN_BM) {
        for (int x = lane; x < bm_words; x += GS) bitmap[x] = 0u;
    }
    // Numeric tables start empty and every column leaves its table empty again (the
    // bitmap emit resets the slots it reads; the sorting path clears the table).
    if constexpr (NUM) {
        for (int s = lane; s < TBL; s += GS) {
            keys[s] = -1;
            vals[s] = SR::zero();
        }
    }
    G::sync();

    for (int64_t w = (int64_t)blockIdx.x * NG + g; w < count; w += (int64_t)gridDim.x * NG) {
        const int2 e = __ldg(list + w);
        const Prod* pr = it.prods + e.x;
        const int64_t u = __ldg(it.item_base + e.x) + e.y;
        const int64_t bs = __ldg(pr->B.cp + e.y), be = __ldg(pr->B.cp + e.y + 1);
        if constexpr (!NUM) {
            for (int s = lane; s < TBL; s += GS) keys[s] = -1;
            if (lane == 0) *s_cnt = 0;
            G::sync();
        }
        int mycnt = 0;
        // numeric columns whose rows fit the bitmap mark a row when they claim its slot
        int mark_nw = 0;
        if constexpr (CAN_BM) {
            const int64_t mw = (pr->A.m + 31) >> 5;
            mark_nw = mw <= bm_words ? (int)mw : 0;
        }
        for (int64_t b0 = bs; b0 < be; b0 += GS) {
            const int64_t t = b0 + lane;
            int len = 0;
            int64_t a0 = 0;
            T bv = T(0);
            if (t < be) {
                int32_t k = __ldg(pr->B.ir + t);
                int64_t s, en;
                a_col(it, pr, t, k, s, en);
                a0 = s;
                len = (int)(en - s);
                if constexpr (NUM) bv = load_val<SR>(pr->B, t);
            }
            // Every member finished the previous chunk's expansion before the scan's
            // barrier (or the warp's shuffles), so the chunk arrays can be rewritten
            // after it without a closing barrier.
            int total;
            int ns = GS;   // segments in s_incl / s_a0 / s_bv
            if constexpr (GS == 32) {
                const int incl = group_incl_scan_open<GS>(len, s_scan, total);
                s_incl[lane] = incl;
                s_a0[lane] = a0;
                if constexpr (NUM) s_bv[lane] = bv;
            } else {
                // several warps: keep the nonempty segments only (their ends are then
                // distinct), so that a warp finds its products' segments by windows
                long long tot64;
                const long long inc64 = group_incl_scan64_open<GS>(len > 0 ? ((1ll << 32) | len) : 0ll,
                                                                   reinterpret_cast<long long*>(s_scan), tot64);
                if (len > 0) {
                    const int p = (int)(inc64 >> 32) - 1;
                    s_incl[p] = (int)(inc64 & 0xffffffffll);
                    s_a0[p] = a0;
                    if constexpr (NUM) s_bv[p] = bv;
                }
                ns = (int)(tot64 >> 32);
                total = (int)(tot64 & 0xffffffffll);
            }
            G::sync();
            const int32_t* __restrict__ air = pr->A.ir;
            // U products per lane per round: their loads are all issued before the first insert
            constexpr int U = 4;
            // several warps: each takes a contiguous slice of the products, in windows of 32
            int q0 = 0, qend = total, o0 = 0;
            constexpr int QSTEP = GS == 32 ? GS * U : 32 * U;
            if constexpr (GS > 32) {
                constexpr int NWG = GS / 32;
                const int wg = (threadIdx.x % GS) >> 5;
                const int C = (total + NWG * 32 - 1) / (NWG * 32) * 32;
                q0 = wg * C;
                qend = min(total, q0 + C);
                int lo = 0, hi = ns;   // segments ending at or before the slice start
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (s_incl[mid] <= q0) lo = mid + 1;
                    else hi = mid;
                }
                o0 = lo;
            }
            for (; q0 < qend; q0 += QSTEP) {
                int32_t row[U];
                T av[U];
                int seg[U];
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    row[i] = -1;
                    if constexpr (GS == 32) {
                        const int q = q0 + i * GS + lane;
                        if (q < total) {
                            int lo = 0, hi = GS - 1;
                            while (lo < hi) {
                                int mid = (lo + hi) >> 1;
                                if (s_incl[mid] > q) hi = mid;
                                else lo = mid + 1;
                            }
                            const int64_t idx = s_a0[lo] + (q - (lo ? s_incl[lo - 1] : 0));
                            row[i] = __ldg(air + idx);
                            if constexpr (NUM) av[i] = load_val<SR>(pr->A, idx);
                            seg[i] = lo;
                        }
                    } else {
                        const int xw = q0 + 32 * i;
                        const int oi = warp_window_segment(s_incl, ns, xw, o0);
                        const int q = xw + (threadIdx.x & 31);   // this warp's lane, not the group's
                        if (q < qend) {
                            const int64_t idx = s_a0[oi] + (q - (oi ? s_incl[oi - 1] : 0));
                            row[i] = __ldg(air + idx);
                            if constexpr (NUM) av[i] = load_val<SR>(pr->A, idx);
                            seg[i] = oi;
                        }
                    }
                }
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    if (row[i] < 0) continue;
                    const int32_t r = row[i];
                    uint32_t h = hash_row(r) >> (32 - LOG2);
                    while (true) {
                        int32_t cur = vkeys[h];
                        if (cur == r) break;
                        if (cur == -1) {
                            int32_t prev = atomicCAS(&keys[h], -1, r);
                            if (prev == -1) {
                                ++mycnt;
                                if constexpr (CAN_BM)
                                    if ((r >> 5) < mark_nw) atomicOr(&bitmap[r >> 5], 1u << (r & 31));
                                break;
                            }
                            if (prev == r) break;
                        }
                        h = (h + 1) & (TBL - 1);
                    }
                    if constexpr (NUM) SR::atomic_add(&vals[h], SR::mul(av[i], s_bv[seg[i]]));
                }
            }
            if constexpr (GS == 32) __syncwarp();
        }
        G::sync();
        if constexpr (!NUM) {
            int c = warp_sum(mycnt);
            if constexpr (GS == 32) {
                if (lane == 0) nnz_item[u] = c;
            } else {
                if ((threadIdx.x & 31) == 0) atomicAdd(s_cnt, c);
                __syncthreads();
                if (lane == 0) nnz_item[u] = *s_cnt;
            }
            G::sync();
        } else {
            // exact mode: Coff holds exact offsets.  Predicted mode (nnz_item != nullptr): Coff holds
            // capacity offsets; the exact count is recorded and the column is written only if it fits.
            const int64_t out0 = __ldg(Coff + u);
            const int64_t capn = __ldg(Coff + u + 1) - out0;
            const int32_t rb = out_row_base(pr, e.y);
            if constexpr (CAN_BM) {
                // a warp prefers the bitmap once sorting the entries would cost more than scanning it
                bool use_bm = mark_nw > 0;
                if constexpr (GS == 32) use_bm = use_bm && mark_nw <= 8 * warp_sum(mycnt);
                if (use_bm) {
                    const int total = rank_emit<SR, TBL, GS>(bitmap, wp, mark_nw, keys, vals, s_incl, s_scan,
                                                             nnz_item != nullptr, capn, out0, rb, Cir, Cv);
                    if (nnz_item && lane == 0) nnz_item[u] = total;
                    continue;
                }
                // sorting instead: drop the marks
                for (int x = lane; x < mark_nw; x += GS) bitmap[x] = 0u;
            }
            // in-place compaction toward the front: the i-th occupied slot moves to i <= its slot.
            // Each lane holds a contiguous run of S slots in registers; rounds go up the table, and
            // every destination lies below the slots of later rounds, so nothing unread is overwritten.
            constexpr int S = (TBL / GS) < 8 ? (TBL / GS) : 8;
            int pos = 0;
            for (int r0 = 0; r0 < TBL; r0 += GS * S) {
                const int base_s = r0 + lane * S;
                int32_t kk[S];
                Acc vv[S];
                int occ = 0;
#pragma unroll
                for (int i = 0; i < S; ++i) {
                    kk[i] = keys[base_s + i];
                    vv[i] = vals[base_s + i];
                    occ += kk[i] != -1;
                }
                int total;
                int o = pos + group_incl_scan<GS>(occ, s_scan, total) - occ;
                G::sync();
#pragma unroll
                for (int i = 0; i < S; ++i) {
                    if (kk[i] != -1) {
                        keys[o] = kk[i];
                        vals[o] = vv[i];
                        ++o;
                    }
                }
                pos += total;
                G::sync();
            }
            const int nnz = nnz_item ? pos : (int)capn;
            if (nnz_item) {
                if (lane == 0) nnz_item[u] = pos;
                if (pos > capn) {   // overflow: recomputed into its exact place afterwards
                    for (int s = lane; s < TBL; s += GS) {
                        keys[s] = -1;
                        vals[s] = SR::zero();
                    }
                    G::sync();
                    continue;
                }
            }
            int P = 1;
            while (P < nnz) P <<= 1;
            for (int s = nnz + lane; s < P; s += GS) keys[s] = INT_MAX;
            G::sync();
            bitonic_sort<GS>(keys, vals, P);
            for (int s = lane; s < nnz; s += GS) {
                Cir[out0 + s] = keys[s] + rb;
                Cv[out0 + s] = SR::out(vals[s]);
            }
            G::sync();
            for (int s = lane; s < TBL; s += GS) {
                keys[s] = -1;
                vals[s] = SR::zero();
            }
            G::sync();
        }
    }
}

template <class SR, int GS, int TBL, bool NUM, int BLOCK>
static void run_hash(const Lanes& st, const Items& it, const int2* list, int64_t count, int64_t* nnz_item,
                     const int64_t* Coff, int32_t* Cir, typename SR::T* Cv) {
    if (count <= 0) return;
    using L = HashLayout<SR, GS, TBL, NUM>;
    constexpr int NG = BLOCK / GS;
    constexpr bool CAN_BM = NUM && (GS == BLOCK || (GS == 32 && TBL >= BM_WARP_MIN_TBL));
    // small groups keep the bitmap to the rows a warp would (its scan is per column)
    constexpr int64_t bm_rows = GS < 256 ? BM_WARP_MAX_ROWS : BM_MAX_ROWS;
    const int bm_words = CAN_BM && it.max_m > 0 && it.max_m <= bm_rows ? (int)((it.max_m + 31) / 32) : 0;
    size_t smem = L::group * NG + (size_t)bm_words * 6 * NG;   // bitmap words and their 16-bit prefixes
    auto kern = k_hash<SR, GS, TBL, NUM, BLOCK>;
    smem_at_least((const void*)kern, smem);
    int64_t want = ceil_div64(count, NG);
    int grid = (int)std::min<int64_t>(want, sm_count() * 32);
    kern<<<grid, BLOCK, smem, st.next()>>>(it, list, count, nnz_item, Coff, Cir, Cv, bm_words);
    note_launch();
}

// Symbolic count of columns whose rows fit a per-group bitmap (every A_i has at
// most BM_COUNT_MAX_ROWS rows, as the SUMMA merge columns): each product sets its
// row's bit and nnz is the popcount; no keys, no probing, no table to clear.
constexpr int64_t BM_COUNT_MAX_ROWS = 32768;
// shared memory of one counting group before the bitmaps: a0, incl, scan (34), l1 (32)
template <int GS>
constexpr size_t bitcount_group_bytes() { return ((size_t)GS * 12 + 34 * 4 + 32 * 4 + 15) / 16 * 16; }
template <int GS, int BLOCK>
__global__ void __launch_bounds__(BLOCK, 2048 / BLOCK) k_bitcount(Items it, const int2* __restrict__ list,
                                                                  int64_t count, int64_t* __restrict__ nnz_item,
                                                                  int bm_words) {
    using G = Group<GS>;
    constexpr int NG = BLOCK / GS;
    constexpr size_t GROUP = bitcount_group_bytes<GS>();
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = G::lane(), g = G::gid();
    unsigned char* base = smem + (size_t)g * GROUP;
    int64_t* s_a0 = reinterpret_cast<int64_t*>(base);
    int* s_incl = reinterpret_cast<int*>(base + (size_t)GS * 8);
    int* s_scan = s_incl + GS;
    uint32_t* l1 = reinterpret_cast<uint32_t*>(s_scan + 34);   // nonempty bitmap words (bm_words <= 1024)
    uint32_t* bitmap = reinterpret_cast<uint32_t*>(smem + (size_t)NG * GROUP) + (size_t)g * bm_words;
    for (int x = lane; x < bm_words; x += GS) bitmap[x] = 0u;
    for (int x = lane; x < 32; x += GS) l1[x] = 0u;
    G::sync();
    for (int64_t w = (int64_t)blockIdx.x * NG + g; w < count; w += (int64_t)gridDim.x * NG) {
        const int2 e = __ldg(list + w);
        const Prod* pr = it.prods + e.x;
        const int64_t u = __ldg(it.item_base + e.x) + e.y;
        const int64_t bs = __ldg(pr->B.cp + e.y), be = __ldg(pr->B.cp + e.y + 1);
        const uint32_t mrows = (uint32_t)(pr->A.m < (int64_t)bm_words * 32 ? pr->A.m : (int64_t)bm_words * 32);
        const int32_t* __restrict__ air = pr->A.ir;
        int c = 0;   // rows this lane marked first
        for (int64_t b0 = bs; b0 < be; b0 += GS) {
            const int64_t t = b0 + lane;
            int len = 0;
            int64_t a0 = 0;
            if (t < be) {
                int64_t s, en;
                a_col(it, pr, t, __ldg(pr->B.ir + t), s, en);
                a0 = s;
                len = (int)(en - s);
            }
            int total;
            int ns = GS;
            if constexpr (GS == 32) {
                const int incl = group_incl_scan_open<GS>(len, s_scan, total);
                s_incl[lane] = incl;
                s_a0[lane] = a0;
            } else {   // nonempty segments only, for the windowed walk below
                long long tot64;
                const long long inc64 = group_incl_scan64_open<GS>(len > 0 ? ((1ll << 32) | len) : 0ll,
                                                                   reinterpret_cast<long long*>(s_scan), tot64);
                if (len > 0) {
                    const int p = (int)(inc64 >> 32) - 1;
                    s_incl[p] = (int)(inc64 & 0xffffffffll);
                    s_a0[p] = a0;
                }
                ns = (int)(tot64 >> 32);
                total = (int)(tot64 & 0xffffffffll);
            }
            G::sync();
            constexpr int U = 4;
            int q0 = 0, qend = total, o0 = 0;
            constexpr int QSTEP = GS == 32 ? GS * U : 32 * U;
            if constexpr (GS > 32) {   // a contiguous slice of the products per warp
                constexpr int NWG = GS / 32;
                const int wg = (threadIdx.x % GS) >> 5;
                const int C = (total + NWG * 32 - 1) / (NWG * 32) * 32;
                q0 = wg * C;
                qend = min(total, q0 + C);
                int lo = 0, hi = ns;
                while (lo < hi) {
                    const int mid = (lo + hi) >> 1;
                    if (s_incl[mid] <= q0) lo = mid + 1;
                    else hi = mid;
                }
                o0 = lo;
            }
            for (; q0 < qend; q0 += QSTEP) {
                int32_t row[U];
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    row[i] = -1;
                    if constexpr (GS == 32) {
                        const int q = q0 + i * GS + lane;
                        if (q < total) {
                            int lo = 0, hi = GS - 1;
                            while (lo < hi) {
                                const int mid = (lo + hi) >> 1;
                                if (s_incl[mid] > q) hi = mid;
                                else lo = mid + 1;
                            }
                            row[i] = __ldg(air + s_a0[lo] + (q - (lo ? s_incl[lo - 1] : 0)));
                        }
                    } else {
                        const int xw = q0 + 32 * i;
                        const int oi = warp_window_segment(s_incl, ns, xw, o0);
                        const int q = xw + (threadIdx.x & 31);   // this warp's lane, not the group's
                        if (q < qend) row[i] = __ldg(air + s_a0[oi] + (q - (oi ? s_incl[oi - 1] : 0)));
                    }
                }
            // the atomic's return value says whether the row is new; a word that becomes
            // nonempty is marked in l1, so only touched words are cleared afterwards
#pragma unroll
                for (int i = 0; i < U; ++i) {
                    if ((uint32_t)row[i] >= mrows) continue;
                    const int wd = row[i] >> 5;
                    const uint32_t bit = 1u << (row[i] & 31);
                    const uint32_t old = atomicOr(&bitmap[wd], bit);
                    c += (old & bit) == 0u;
                    if (old == 0u) atomicOr(&l1[wd >> 5], 1u << (wd & 31));
                }
            }
            if constexpr (GS == 32) __syncwarp();
        }
        G::sync();
        int tot;
        group_incl_scan<GS>(c, s_scan, tot);
        if (lane == 0) nnz_item[u] = tot;
        // empty the words this column touched (through the first-level bitmap)
        for (int x = lane; x < 32; x += GS) {
            uint32_t bits = l1[x];
            while (bits) {
                bitmap[x * 32 + __ffs(bits) - 1] = 0u;
                bits &= bits - 1;
            }
            l1[x] = 0u;
        }
        G::sync();
    }
}

template <int GS, int BLOCK>
static void run_bitcount(const Lanes& st, const Items& it, const int2* list, int64_t count, int64_t* nnz_item) {
    if (count <= 0) return;
    constexpr int NG = BLOCK / GS;
    constexpr size_t GROUP = bitcount_group_bytes<GS>();
    const int bm_words = (int)((it.max_m + 31) / 32);
    const size_t smem = (GROUP + (size_t)bm_words * 4) * NG;
    auto kern = k_bitcount<GS, BLOCK>;
    smem_at_least((const void*)kern, smem);
    const int grid = (int)std::min<int64_t>(ceil_div64(count, NG), sm_count() * 32);
    kern<<<grid, BLOCK, smem, st.next()>>>(it, list, count, nnz_item, bm_words);
    note_launch();
}

// Tiny columns (flops <= TINY_MAX): one thread gathers the products in
// registers, insertion-sorts them by row (stable, so equal rows keep ascending
// k order), sums duplicates and writes the column.  No table, no barrier.
template <class SR, bool NUM>
__global__ void __launch_bounds__(256) k_tiny(Items it, const int2* __restrict__ list, int64_t count,
                                              int64_t* __restrict__ nnz_item, const int64_t* __restrict__ Coff,
                                              int32_t* __restrict__ Cir, typename SR::T* __restrict__ Cv) {
    using Acc = typename SR::Acc;
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < count; w += (int64_t)gridDim.x * blockDim.x) {
        const int2 e = __ldg(list + w);
        const Prod* pr = it.prods + e.x;
        const int64_t u = __ldg(it.item_base + e.x) + e.y;
        const int64_t bs = __ldg(pr->B.cp + e.y), be = __ldg(pr->B.cp + e.y + 1);
        int32_t r[TINY_MAX];
        Acc v[TINY_MAX];
        int n = 0;
        for (int64_t t = bs; t < be; ++t) {
            const int32_t k = __ldg(pr->B.ir + t);
            int64_t s0, en;
            a_col(it, pr, t, k, s0, en);
            typename SR::T bv = typename SR::T(0);
            if constexpr (NUM) bv = load_val<SR>(pr->B, t);
            for (int64_t q = s0; q < en && n < TINY_MAX; ++q) {
                r[n] = __ldg(pr->A.ir + q);
                if constexpr (NUM) v[n] = SR::mul(load_val<SR>(pr->A, q), bv);
                ++n;
            }
        }
        for (int i = 1; i < n; ++i) {
            const int32_t key = r[i];
            Acc val = NUM ? v[i] : Acc(0);
            int j = i - 1;
            while (j >= 0 && r[j] > key) {
                r[j + 1] = r[j];
                if constexpr (NUM) v[j + 1] = v[j];
                --j;
            }
            r[j + 1] = key;
            if constexpr (NUM) v[j + 1] = val;
        }
        int m = 0;
        for (int i = 0; i < n; ++i) {
            if (m > 0 && r[m - 1] == r[i]) {
                if constexpr (NUM) v[m - 1] = SR::add(v[m - 1], v[i]);
            } else {
                r[m] = r[i];
                if constexpr (NUM) v[m] = v[i];
                ++m;
            }
        }
        if constexpr (!NUM) {
            nnz_item[u] = m;
        } else {
            // exact mode: Coff are exact offsets; predicted mode (nnz_item set): capacity offsets
            const int64_t out0 = __ldg(Coff + u);
            if (nnz_item) nnz_item[u] = m;
            // overflow (predicted mode): redone in its exact place; in exact mode the counts
            // agree, and the check keeps an inconsistent input inside its column
            if (m > __ldg(Coff + u + 1) - out0) continue;
            const int32_t rb = out_row_base(pr, e.y);
            for (int i = 0; i < m; ++i) {
                Cir[out0 + i] = r[i] + rb;
                Cv[out0 + i] = SR::out(v[i]);
            }
        }
    }
}

template <class SR, bool NUM>
static void run_tiny(const Lanes& st, const Items& it, const int2* list, int64_t count, int64_t* nnz_item,
                     const int64_t* Coff, int32_t* Cir, typename SR::T* Cv) {
    if (count <= 0) return;
    const int grid = (int)std::min<int64_t>(ceil_div64(count, 256), sm_count() * 16);
    k_tiny<SR, NUM><<<grid, 256, 0, st.next()>>>(it, list, count, nnz_item, Coff, Cir, Cv);
    note_launch();
}

// every A_i has at most BLOCK_TIER_MAX_ROWS rows: numeric passes run in the block tier
static bool block_mode(const Items& it) { return it.max_m > 0 && it.max_m <= BLOCK_TIER_MAX_ROWS; }

// Columns of few products, counting or numeric: the sort tier, or, where not even 16
// products fit its keys (2^28 rows and more), a thread per column of at most 16.
template <class SR, bool NUM>
static void run_short(const Lanes& st, const Items& it, const int2* list, const int64_t* off, const int64_t* cnt,
                      int64_t* nnz_item, const int64_t* Coff, int32_t* Cir, typename SR::T* Cv, const int* vals_zero) {
    if (sort_max_products(it.max_m) == 0)
        run_tiny<SR, NUM>(st, it, list + off[BIN_SORT0], cnt[BIN_SORT0], nnz_item, Coff, Cir, Cv);
    else if constexpr (NUM) launch_sort_tier<SR>(st, it, list, off, cnt, nnz_item, Coff, Cir, Cv, vals_zero);
    else launch_sort_count(st, it, list, off, cnt, nnz_item);
}

template <class SR, bool NUM>
static void run_hash_bins(const Lanes& st, const Items& it, const int2* list, const int64_t* off, const int64_t* cnt,
                          int64_t* nnz_item, const int64_t* Coff, int32_t* Cir, typename SR::T* Cv,
                          const int* vals_zero = nullptr) {
    constexpr int W0 = BIN_WARP0, B0 = BIN_BLK0;
    run_short<SR, NUM>(st, it, list, off, cnt, nnz_item, Coff, Cir, Cv, vals_zero);
    run_hash<SR, 32, 64, NUM, WARP_BLOCK>(st, it, list + off[W0], cnt[W0], nnz_item, Coff, Cir, Cv);
    run_hash<SR, 32, 128, NUM, WARP_BLOCK>(st, it, list + off[W0 + 1], cnt[W0 + 1], nnz_item, Coff, Cir, Cv);
    if constexpr (!NUM) {
        if (it.max_m > 0 && it.max_m <= BM_COUNT_MAX_ROWS) {
            // rows fit a small bitmap: count the longer columns by bits (64 and 128
            // slots hold so few rows that clearing a bitmap would cost more)
            // one warp per column for the CTA-table bins too: a column of a few thousand
            // products has no barrier chain to wait on, and its bitmap is the same size
            run_bitcount<32, WARP_BLOCK>(st, it, list + off[W0 + 2],
                                         cnt[W0 + 2] + cnt[W0 + 3] + cnt[W0 + 4] + cnt[B0] + cnt[B0 + 1] + cnt[B0 + 2],
                                         nnz_item);
            return;
        }
    }
    run_hash<SR, 32, 256, NUM, WARP_BLOCK>(st, it, list + off[W0 + 2], cnt[W0 + 2], nnz_item, Coff, Cir, Cv);
    if constexpr (NUM) {
        // numeric tables of 512 and 1024 slots: one table per 2 or 4 warps, so that
        // shared memory admits more warps per SM (a warp each left a quarter of them)
        run_hash<SR, 64, 512, NUM, 64>(st, it, list + off[W0 + 3], cnt[W0 + 3], nnz_item, Coff, Cir, Cv);
        run_hash<SR, 128, 1024, NUM, 128>(st, it, list + off[W0 + 4], cnt[W0 + 4], nnz_item, Coff, Cir, Cv);
    } else {
        run_hash<SR, 32, 512, NUM, WARP_BLOCK>(st, it, list + off[W0 + 3], cnt[W0 + 3], nnz_item, Coff, Cir, Cv);
        run_hash<SR, 32, 1024, NUM, 128>(st, it, list + off[W0 + 4], cnt[W0 + 4], nnz_item, Coff, Cir, Cv);
    }
    run_hash<SR, 256, 2048, NUM, 256>(st, it, list + off[B0], cnt[B0], nnz_item, Coff, Cir, Cv);
    // 4096-slot tables: 256 threads per column when the row bitmap is small (more columns
    // in flight per SM), 512 when a large bitmap already limits the CTAs per SM
    if (it.max_m <= 65536)
        run_hash<SR, 256, 4096, NUM, 256>(st, it, list + off[B0 + 1], cnt[B0 + 1], nnz_item, Coff, Cir, Cv);
    else
        run_hash<SR, 512, 4096, NUM, 512>(st, it, list + off[B0 + 1], cnt[B0 + 1], nnz_item, Coff, Cir, Cv);
    run_hash<SR, 512, 8192, NUM, 512>(st, it, list + off[B0 + 2], cnt[B0 + 2], nnz_item, Coff, Cir, Cv);
}

// ------------------------------------------------------------------ slab tier (long columns)
// A long output column is split into P row slabs of at most RB rows (balanced by
// flops, at most MAX_PARTS, fewer where B(:,j) is long: every slab repeats two
// binary searches per entry of B(:,j)).  The symbolic kernel marks the rows of a
// slab in a shared-memory bitmap with one flattened walk over the slab's products,
// counts them and stores the slab's row set for the numeric pass: its bitmap words
// when the slab holds at least one row per word, else its rows in ascending order,
// whichever is smaller.  The numeric kernel reloads the row set into a
// shared-memory bitmap, ranks rows by per-group prefix counts (4 words = 128 rows
// per group), writes C's rows for the slab, sets the slab's values to the
// semiring zero and walks the products again, adding each one into C at its row's
// rank with an L2 reduction.  There is no shared-memory accumulator (FP64 shared
// atomics are the slow path on this part), no hashing and no sort, and a slab's
// products are spread evenly over the CTA's warps.
constexpr int RT_BLOCK = 512;
constexpr int RT_WARPS = RT_BLOCK / 32;

__device__ __forceinline__ int32_t lower_bound_rows(const int32_t* __restrict__ r, int64_t len, int64_t v) {
    int64_t lo = 0, hi = len;
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if ((int64_t)__ldg(r + mid) < v) lo = mid + 1;
        else hi = mid;
    }
    return (int32_t)lo;
}

// rows [R0, R1) of slab q of P over m rows (32-aligned cuts)
__host__ __device__ __forceinline__ void slab_rows(int64_t m, int q, int P, int64_t& R0, int64_t& R1) {
    R0 = ((int64_t)q * m / P) & ~int64_t(31);
    R1 = q == P - 1 ? m : (((int64_t)(q + 1) * m / P) & ~int64_t(31));
}

// the most rows any of the P slabs over m rows holds
__host__ __device__ __forceinline__ int64_t slab_max_rows(int64_t m, int P) {
    int64_t mx = 0;
    for (int q = 0; q < P; ++q) {
        int64_t R0, R1;
        slab_rows(m, q, P, R0, R1);
        mx = R1 - R0 > mx ? R1 - R0 : mx;
    }
    return mx;
}

// the quad walk applies to a product whose A is a CSC (no DCSC index, no gaps) of fewer than
// 2^31 entries with 16-byte aligned row and value arrays
__host__ __device__ __forceinline__ bool quads_ok(const Prod* pr) {
    return pr->A.jc == nullptr && pr->A.ce == nullptr && pr->A.nnz < INT_MAX - 8 && ((uintptr_t)pr->A.ir & 15) == 0 &&
           ((uintptr_t)pr->A.num & 15) == 0;
}

// Slabs of the long columns: P per column, items[sbase[d] + q] = (d, q); the
// storage bound of the slab row sets, sum over columns of min(flops, words),
// accumulates in *store_bound (a slab stores min(words, rows) 4-byte entries and
// rows <= flops).  The three global counters take one addition per warp (a column each
// queued on one L2 line), and nothing here walks a column's slabs with 64-bit divisions:
// R-MAT 20 flat 751 -> 27 us, R-MAT of 300,007 vertices 203 -> 10 us.
__global__ void k_dense_items(Items it, const int2* __restrict__ dlist, int64_t nd, const int64_t* __restrict__ flops,
                              int part_flops, int RB, int2* items, unsigned long long* nitems, int8_t* nparts,
                              int32_t* sbase, unsigned long long* store_bound, int64_t* bbase,
                              unsigned long long* bnd_total, unsigned long long* kinds) {
    const int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int lane = threadIdx.x & 31;
    const bool ok = d < nd;
    long long P = 0, bound = 0, bnd = 0;
    unsigned kind = 0;
    if (ok) {
        const int2 e = dlist[d];
        const Prod* pr = it.prods + e.x;
        const int64_t f = flops[__ldg(it.item_base + e.x) + e.y];
        const int64_t deg = __ldg(pr->B.cp + e.y + 1) - __ldg(pr->B.cp + e.y);
        const int64_t m = pr->A.m;
        // slab rows stay <= RB: the fewest slabs whose 32-aligned cuts all fit (the host
        // sized RB so that MAX_PARTS slabs always do); a cut moves a slab's ends by at
        // most 31 rows
        int64_t pmin = m <= RB ? 1 : ceil_div64(m, (int64_t)RB);
        while (pmin > 1 && pmin < MAX_PARTS && ceil_div64(m, pmin) + 31 > RB && slab_max_rows(m, (int)pmin) > RB) ++pmin;
        P = ceil_div64(f, part_flops);
        const int64_t pdeg = f / (32 * (deg > 0 ? deg : 1));   // about 32 products per (slab, B entry) at least
        P = P < pdeg ? P : pdeg;
        P = P < pmin ? pmin : P;
        P = P > MAX_PARTS ? MAX_PARTS : P;
        P = P < 1 ? 1 : P;
        const int64_t words = (m + 31) >> 5;   // of all its slabs: every inner cut is a multiple of 32
        bound = f < words ? f : words;
        // boundary table: P + 1 rows of deg positions (where each slab starts in every A(:,k)),
        // then two rows with where every A(:,k) starts (low and high 32 bits)
        bnd = (P + 3) * deg;
        if (kinds) kind = quads_ok(pr) ? 1u : 2u;
    }
    if (kinds) kind = __reduce_or_sync(0xffffffffu, kind);
    const long long ip = warp_incl_scan64(P), ib = warp_incl_scan64(bnd), sb = warp_sum(bound);
    unsigned long long bp = 0, bb = 0;
    if (lane == 31) {
        bp = atomicAdd(nitems, (unsigned long long)ip);
        bb = atomicAdd(bnd_total, (unsigned long long)ib);
        atomicAdd(store_bound, (unsigned long long)sb);
        if (kinds) atomicOr(kinds, (unsigned long long)kind);
    }
    bp = __shfl_sync(0xffffffffu, bp, 31);
    bb = __shfl_sync(0xffffffffu, bb, 31);
    if (!ok) return;
    const int64_t base = (int64_t)bp + ip - P;
    nparts[d] = (int8_t)P;
    bbase[d] = (int64_t)bb + ib - bnd;
    sbase[d] = (int32_t)base;
    for (int q = 0; q < P; ++q) items[base + q] = make_int2((int)d, q);
}

void launch_dense_items(cudaStream_t st, const Items& it, const int2* dense_list, int64_t ndense, const int64_t* flops,
                        int part_flops, int RB, int2* items, unsigned long long* nitems, int8_t* nparts,
                        int32_t* sbase, unsigned long long* store_bound, int64_t* bbase,
                        unsigned long long* bnd_total, unsigned long long* kinds) {
    if (ndense == 0) return;
    k_dense_items<<<(int)ceil_div64(ndense, 256), 256, 0, st>>>(it, dense_list, ndense, flops, part_flops, RB, items,
                                                               nitems, nparts, sbase, store_bound, bbase, bnd_total,
                                                               kinds);
    note_launch();
}

// Slab boundaries, once for both passes: row q of column d's table holds, for every
// entry t of B(:,j), where slab q starts inside A(:,k) (relative to the column's
// start); row P holds A(:,k)'s length.  One CTA per slab, every search of the slab
// in flight at once (the passes that read them no longer wait on search chains at
// their barriers).  Where most columns are cut, most slabs search, and a search is one chain
// of loads whatever the slab's entries: with up to 64 of them on average, CTAs of half as many
// threads put twice as many slabs in flight.  256 against 128 threads: R-MAT 20 (four slabs per
// column, 35 entries) 3.7 / 2.3 ms, R-MAT 19 (two, 39) 0.82 / 0.71 ms, A S^T of pairs at R-MAT 20
// (four, 2) 25 / 16 us.  Columns of one slab search nothing, and their time is that of the longest
// ones: R-MAT 18 (36 entries) 182 / 197 us, R-MAT 16 (31) 50 / 71 us, S (A S^T) (1,600) 91 / 172 us.
__global__ void __launch_bounds__(256) k_slab_bounds(Items it, DenseWork dw) {
    const int64_t nsym = (int64_t)*dw.nitems;
    for (int64_t w = blockIdx.x; w < nsym; w += gridDim.x) {
        const int2 itm = dw.items[w];
        const int d = itm.x, q = itm.y;
        const int2 e = __ldg(dw.dlist + d);
        const Prod* pr = it.prods + e.x;
        const int P = dw.nparts[d];
        const int64_t m = pr->A.m;
        int64_t R0, R1;
        slab_rows(m, q, P, R0, R1);
        const int64_t bs = __ldg(pr->B.cp + e.y), be = __ldg(pr->B.cp + e.y + 1);
        const int64_t deg = be - bs;
        int32_t* __restrict__ row = dw.bnd + dw.bbase[d] + (int64_t)q * deg;
        const int32_t* __restrict__ air = pr->A.ir;
        if (threadIdx.x == 0) {
            SlabRec r;
            r.prod = e.x;
            r.col = e.y;
            r.r0 = (int32_t)R0;
            r.r1 = (int32_t)R1;
            r.rb = out_row_base(pr, e.y);
            r.cnt = 0;
            r.bs = bs;
            r.be = be;
            r.bnd = dw.bbase[d] + (int64_t)q * deg;
            r.u = __ldg(it.item_base + e.x) + e.y;
            r.ob = 0;
            r.soff = -1;
            r.sab = dw.bbase[d] + (int64_t)(P + 1) * deg;
            dw.rec[w] = r;
        }
        for (int64_t t = threadIdx.x; t < deg; t += blockDim.x) {
            const int32_t k = __ldg(pr->B.ir + bs + t);
            int64_t s, en;
            a_col(it, pr, bs + t, k, s, en);
            row[t] = q == 0 ? 0 : lower_bound_rows(air + s, en - s, R0);
            if (q == P - 1) row[t + deg] = (int32_t)(en - s);
            if (q == 0) {   // where A(:,k) starts, for the passes' segment arithmetic
                int32_t* sr = dw.bnd + dw.bbase[d] + (int64_t)(P + 1) * deg;
                sr[t] = (int32_t)(uint32_t)s;
                sr[t + deg] = (int32_t)(s >> 32);
            }
        }
    }
}

// Any zero byte in v[0, n), 16 at a time between the aligned ends, the work spread over
// `stride` threads of which this is thread t0.  (A byte per load took 115 us for the 16 MB
// of an R-MAT scale 20 graph.)
__device__ __forceinline__ bool any_zero_byte(const uint8_t* __restrict__ v, int64_t n, int64_t t0, int64_t stride) {
    int64_t head = (int64_t)((16 - ((uintptr_t)v & 15)) & 15);
    head = head < n ? head : n;
    const int64_t nq = (n - head) >> 4;
    const uint4* __restrict__ q = reinterpret_cast<const uint4*>(v + head);
    bool f = false;
    auto zero = [](uint32_t x) { return ((x - 0x01010101u) & ~x & 0x80808080u) != 0u; };
    for (int64_t i = t0; i < nq; i += stride) {
        const uint4 x = __ldg(q + i);
        f |= zero(x.x) || zero(x.y) || zero(x.z) || zero(x.w);
    }
    for (int64_t i = t0; i < head; i += stride) f |= __ldg(v + i) == 0;
    for (int64_t i = head + 16 * nq + t0; i < n; i += stride) f |= __ldg(v + i) == 0;
    return f;
}

// flag = 1 when some stored value of an operand is false (boolean semiring): then
// the numeric pass must evaluate the products; else every output value is true.
__global__ void k_false_values(Items it, int* flag) {
    for (int64_t p = blockIdx.y; p < it.nprod; p += gridDim.y) {
        const Prod* pr = it.prods + p;
        for (int side = 0; side < 2; ++side) {
            const DMat& M = side ? pr->B : pr->A;
            if (M.num == nullptr || M.nzc <= 0) continue;
            const uint8_t* __restrict__ v = reinterpret_cast<const uint8_t*>(M.num);
            const int64_t stride = (int64_t)gridDim.x * blockDim.x;
            const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
            bool f = false;
            if (M.ce) {   // a CSC with gaps: only the stored part of every column
                for (int64_t c = t0; c < M.nzc; c += stride)
                    for (int64_t i = __ldg(M.cp + c); i < __ldg(M.ce + c); ++i) f |= __ldg(v + i) == 0;
            } else {
                const int64_t s = __ldg(M.cp), e = __ldg(M.cp + M.nzc);
                f = any_zero_byte(v + s, e - s, t0, stride);
            }
            if (f) *flag = 1;
        }
    }
}

__global__ void k_any_false(const uint8_t* __restrict__ v, int64_t n, int* flag) {
    if (any_zero_byte(v, n, (int64_t)blockIdx.x * blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x)) *flag = 1;
}

void launch_any_false(cudaStream_t st, const void* vals, int64_t n, int* flag) {
    if (!vals || n <= 0) return;
    k_any_false<<<(int)std::min<int64_t>(ceil_div64(n, 16 * 256), sm_count() * 8), 256, 0, st>>>((const uint8_t*)vals, n,
                                                                                          flag);
    note_launch();
}

void launch_false_values(cudaStream_t st, const Items& it, int64_t most, int* flag) {
    if (it.nprod <= 0) return;
    const int gy = (int)std::min<int64_t>(it.nprod, 65535);
    // no more CTAs than four 16-byte loads per thread need: it is queued before every numeric
    // pass, a replayed one's too
    const int gx = (int)std::max<int64_t>(1, std::min<int64_t>({(int64_t)sm_count() * 4, 4096 / gy, ceil_div64(most, 256 * 64)}));
    k_false_values<<<dim3(gx, gy), 256, 0, st>>>(it, flag);
    note_launch();
}

// The segments of one batch of RT_BLOCK entries of B(:,j), the nonempty ones in order: part a
// .. b of the arrays of A, and where it ends in the batch's flattened products (QUADS: in
// aligned quads of A's arrays, so that quad x of the batch is quad q + x of the array).
struct SegSmem {
    union {
        int4 seg[RT_BLOCK];       // QUADS: q, a, b
        int64_t start[RT_BLOCK];  // otherwise: a minus the products before the segment
    };
    int64_t bv[RT_BLOCK];     // B value bits (read back as SR::T)
    int end[RT_BLOCK];
    int2 tot[RT_WARPS];       // per warp: segments and products of its entries
};
// shared-memory offset of what follows a SegSmem (16-byte aligned for vector access)
constexpr size_t RS_BYTES = (sizeof(SegSmem) + 15) / 16 * 16;

// Where A(:,k) starts for entry i of B(:,j) (deg entries): two int32 rows of the
// column's boundary table, low and high 32 bits, written by the boundary pre-pass.
__device__ __forceinline__ int64_t seg_start(const int32_t* __restrict__ sab, int64_t i, int64_t deg) {
    return (int64_t)(uint32_t)__ldg(sab + i) | ((int64_t)__ldg(sab + deg + i) << 32);
}

// The segments of entries [b0, b0 + RT_BLOCK) of B(:,j) inside rows [R0, R1): brow0 / brow1 are
// the boundary rows of R0 and R1.  With VALS also B's values.  Returns the number of segments
// and of products (quads).  A warp without entries only meets the two barriers, the second of
// which publishes the segments.
template <class SR, bool VALS, bool QUADS>
__device__ __forceinline__ void slab_segments(const Prod* pr, int64_t b0, int64_t bs, int64_t be,
                                              const int32_t* __restrict__ brow0, const int32_t* __restrict__ brow1,
                                              const int32_t* __restrict__ sab, SegSmem* sc, int& ns, int& T) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t t = b0 + threadIdx.x;
    int len = 0, inc = 0, rank = 0;
    int64_t a = 0, b = 0, bvbits = 0;
    if (b0 + warp * 32 < be) {
        if (t < be) {
            const int64_t s = seg_start(sab, t - bs, be - bs);
            a = s + __ldg(brow0 + (t - bs));
            b = s + __ldg(brow1 + (t - bs));
            if constexpr (QUADS) len = b > a ? (int)(((b - 1) >> 2) - (a >> 2) + 1) : 0;
            else len = (int)(b - a);
            if constexpr (VALS) *reinterpret_cast<typename SR::T*>(&bvbits) = load_val<SR>(pr->B, t);
        }
        inc = warp_incl_scan(len);
        const unsigned some = __ballot_sync(0xffffffffu, len > 0);
        rank = __popc(some & ((1u << lane) - 1u));
        if (lane == 31) sc->tot[warp] = make_int2(__popc(some), inc);
    } else if (lane == 31) {
        sc->tot[warp] = make_int2(0, 0);
    }
    __syncthreads();
    const int2 w = lane < RT_WARPS ? sc->tot[lane] : make_int2(0, 0);
    ns = __reduce_add_sync(0xffffffffu, w.x);
    T = __reduce_add_sync(0xffffffffu, w.y);
    if (b0 + warp * 32 < be) {
        const int i = rank + __reduce_add_sync(0xffffffffu, lane < warp ? w.x : 0);
        const int e = inc + __reduce_add_sync(0xffffffffu, lane < warp ? w.y : 0);
        if (len > 0) {
            sc->end[i] = e;
            if constexpr (QUADS) sc->seg[i] = make_int4((int)(a >> 2) - (e - len), (int)a, (int)b, 0);
            else sc->start[i] = a - (e - len);
            if constexpr (VALS) sc->bv[i] = bvbits;
        }
    }
    __syncthreads();
}

// Four consecutive values of A at an aligned position p (16-byte loads: one for
// 4- and 1-byte types, two for 8-byte types).
template <class T>
__device__ __forceinline__ void load4(const T* __restrict__ p, T v[4]) {
    if constexpr (sizeof(T) == 8) {
        const ulonglong2 x = __ldg(reinterpret_cast<const ulonglong2*>(p));
        const ulonglong2 y = __ldg(reinterpret_cast<const ulonglong2*>(p) + 1);
        const unsigned long long w[4] = {x.x, x.y, y.x, y.y};
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = *reinterpret_cast<const T*>(&w[j]);
    } else if constexpr (sizeof(T) == 4) {
        const uint4 x = __ldg(reinterpret_cast<const uint4*>(p));
        const unsigned w[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = *reinterpret_cast<const T*>(&w[j]);
    } else {
        const unsigned x = __ldg(reinterpret_cast<const unsigned*>(p));
#pragma unroll
        for (int j = 0; j < 4; ++j) v[j] = (T)((x >> (8 * j)) & 0xffu);
    }
}

// Positions p0 .. p0 + 3 of A (an aligned quad): rows, and values with NUM.  A quad past the
// arrays' end (nnz_end entries) is read one by one.
template <class SR, bool NUM>
__device__ __forceinline__ void load_quad(const Prod* pr, int p0, int nnz_end, int32_t (&row)[4],
                                          typename SR::T (&av)[4]) {
    using V = typename SR::T;
    const int32_t* __restrict__ air = pr->A.ir;
    const V* __restrict__ anum = reinterpret_cast<const V*>(pr->A.num);
    if (p0 + 4 <= nnz_end) {
        const int4 r4 = __ldg(reinterpret_cast<const int4*>(air + p0));
        row[0] = r4.x;
        row[1] = r4.y;
        row[2] = r4.z;
        row[3] = r4.w;
        if constexpr (NUM) {
            if (anum) load4<V>(anum + p0, av);
            else av[0] = av[1] = av[2] = av[3] = (V)SR::one();
        }
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (p0 + j < nnz_end) {
                row[j] = __ldg(air + p0 + j);
                if constexpr (NUM) av[j] = load_val<SR>(pr->A, p0 + j);
            }
    }
}

// bit j: position p0 + j lies in [a, b), which meets the quad
__device__ __forceinline__ unsigned quad_mask(int p0, int a, int b) {
    return (0xfu << max(a - p0, 0)) & (0xfu >> (4 - min(b - p0, 4)));
}

// Walk over the products of the batch in sc: each warp takes a contiguous slice, U windows of
// 32 per step with every load issued before the updates.  With QUADS a lane takes an aligned
// quad per window (rows by one 16-byte load, values by one or two); positions are 32-bit and
// A.ir and A.num 16-byte aligned.  f(row, a, b) is called for every product of the lane (a and
// b, the A and B values, only with NUM).  A window inside one segment needs no search for its
// segments, and a window of whole quads no masks.  One quad per lane and step: the passes are
// bound by instructions and their latency, so registers go to warps (four CTAs of 512 threads
// per SM at 32 registers, where two at 64 kept two quads in flight).  Counting pass, R-MAT 18
// 3.2 -> 2.3 ms, 300,007 vertices 3.6 -> 2.6 ms, R-MAT 20 (slabs of 2^18 rows) 32.7 -> 25.4 ms;
// numeric pass, boolean 3.0 -> 2.7 ms, int64 623 -> 532 us, FP64 at R-MAT 20 52.4 -> 51.1 ms.
template <class SR, bool NUM, bool QUADS, class F>
__device__ __forceinline__ void slab_walk(const Prod* pr, const SegSmem* sc, int ns, int T, F&& f) {
    using V = typename SR::T;
    constexpr int U = QUADS ? 1 : 4, J = QUADS ? 4 : 1;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int C = (T + RT_BLOCK - 1) / RT_BLOCK * 32;
    const int xb = warp * C, xe = min(T, xb + C);
    if (xb >= xe) return;
    int lo = 0, hi = xb > 0 ? ns : 0;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (sc->end[mid] <= xb) lo = mid + 1;
        else hi = mid;
    }
    int o0 = lo, cend = sc->end[lo];   // the segment that the next window starts in
    [[maybe_unused]] const int nnz_end = QUADS ? (int)pr->A.nnz : 0;
    [[maybe_unused]] const int32_t* __restrict__ air = pr->A.ir;
    for (int x0 = xb; x0 < xe; x0 += 32 * U) {
        int32_t row[U][J];
        V av[U][J];
        V bv[U];
        unsigned vm[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int xw = x0 + 32 * u, x = xw + lane;
            int oi = o0;
            if (xw + 32 >= cend) {
                oi = warp_window_segment(sc->end, ns, xw, o0);
                cend = o0 < ns ? sc->end[o0] : INT_MAX;
            }
            vm[u] = 0u;
            bv[u] = V(0);
            if (x < xe) {
                if constexpr (NUM) bv[u] = *reinterpret_cast<const V*>(&sc->bv[oi]);
                if constexpr (QUADS) {
                    const int4 sg = sc->seg[oi];
                    const int p0 = (sg.x + x) << 2;
                    vm[u] = quad_mask(p0, sg.y, sg.z);
                    load_quad<SR, NUM>(pr, p0, nnz_end, row[u], av[u]);
                } else {
                    const int64_t p = sc->start[oi] + x;
                    vm[u] = 1u;
                    row[u][0] = __ldg(air + p);
                    if constexpr (NUM) av[u][0] = load_val<SR>(pr->A, p);
                }
            }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (QUADS && __all_sync(0xffffffffu, vm[u] == 0xfu)) {
#pragma unroll
                for (int j = 0; j < J; ++j) f(row[u][j], av[u][j], bv[u]);
            } else {
#pragma unroll
                for (int j = 0; j < J; ++j)
                    if ((vm[u] >> j) & 1u) f(row[u][j], av[u][j], bv[u]);
            }
        }
    }
}

// The products of column B(:,j) inside the slab, batch after batch; ends with a CTA barrier.
template <class SR, bool NUM, bool QUADS, class F>
__device__ __forceinline__ void slab_products(const Prod* pr, int64_t bs, int64_t be, const int32_t* __restrict__ brow0,
                                              const int32_t* __restrict__ brow1, const int32_t* __restrict__ sab,
                                              SegSmem* sc, F&& f) {
    for (int64_t b0 = bs; b0 < be; b0 += RT_BLOCK) {
        int ns, T;
        slab_segments<SR, NUM, QUADS>(pr, b0, bs, be, brow0, brow1, sab, sc, ns, T);
        slab_walk<SR, NUM, QUADS>(pr, sc, ns, T, f);
        __syncthreads();
    }
}

// the semiring whose slabs add up in shared memory
constexpr bool slab_local(int sr) { return sr == SPGEMM_MIN_PLUS_F32; }
// shared memory of the numeric pass before its accumulators
__host__ __device__ constexpr size_t slab_num_bytes(int RB) { return (RS_BYTES + (size_t)(RB / 128 + 1) * 20 + 15) / 16 * 16; }
// accumulators that leave room for two CTAs per SM beside slabs of RB rows
constexpr size_t SLAB_SMEM = 113152;

int slab_acc_entries(int sr, int RB) {
    if (!slab_local(sr) || slab_num_bytes(RB) >= SLAB_SMEM) return 0;
    return (int)((SLAB_SMEM - slab_num_bytes(RB)) / sizeof(MP32::Acc));
}

// Symbolic slab kernel: mark, count, store the row set.  `mixed`: only the products that QUADS is
// for; a launch of the other form takes the rest.
template <bool QUADS>
__global__ void __launch_bounds__(RT_BLOCK, 4) k_slab_sym(Items it, DenseWork dw, bool mixed) {
    extern __shared__ __align__(16) unsigned char smem[];
    SegSmem* sc = reinterpret_cast<SegSmem*>(smem);
    uint32_t* bitmap = reinterpret_cast<uint32_t*>(smem + RS_BYTES);
    int* s_scan = reinterpret_cast<int*>(sc->tot);
    __shared__ long long s_off;
    __shared__ SlabRec s_rec[2];   // this slab's record and the next one's, in flight
    constexpr int RC = sizeof(SlabRec) / 16;
    const int tid = threadIdx.x;
    const int64_t nsym = (int64_t)*dw.nitems;
    if (tid < RC && (int64_t)blockIdx.x < nsym)
        cp_async16(reinterpret_cast<int4*>(&s_rec[0]) + tid, reinterpret_cast<const int4*>(dw.rec + blockIdx.x) + tid);
    int k = 0;
    for (int64_t w = blockIdx.x; w < nsym; w += gridDim.x, k ^= 1) {
        if (tid < RC) cp_async_wait_all();
        __syncthreads();   // s_rec[k] is slab w's record; s_rec[k ^ 1] is free
        if (tid < RC && w + gridDim.x < nsym)
            cp_async16(reinterpret_cast<int4*>(&s_rec[k ^ 1]) + tid,
                       reinterpret_cast<const int4*>(dw.rec + w + gridDim.x) + tid);
        const SlabRec& rc = s_rec[k];
        const Prod* pr = it.prods + rc.prod;
        if (mixed && quads_ok(pr) != QUADS) continue;
        const int64_t R0 = rc.r0, R1 = rc.r1;
        const int nw = (int)((R1 - R0 + 31) >> 5);
        const int ng = (nw + 3) >> 2;   // groups of 4 words (the bitmap is padded to whole groups)
        const int64_t bs = rc.bs, be = rc.be;
        for (int g = tid; g < ng; g += RT_BLOCK) reinterpret_cast<uint4*>(bitmap)[g] = make_uint4(0u, 0u, 0u, 0u);
        __syncthreads();
        const int span = (int)(R1 - R0);
        const int32_t r0 = (int32_t)R0;
        // one shared atomic per product: R-MAT rows of one window mostly fall in different
        // words, so folding lanes per word first (shuffles) measured slower
        auto mark = [&](int32_t row, uint8_t, uint8_t) {
            const int lr = row - r0;
            if ((unsigned)lr < (unsigned)span) atomicOr(&bitmap[lr >> 5], 1u << (lr & 31));
        };
        const int32_t* brow0 = dw.bnd + rc.bnd;
        const int32_t* brow1 = brow0 + (be - bs);
        const int32_t* sab = dw.bnd + rc.sab;
        slab_products<BOOL8, false, QUADS>(pr, bs, be, brow0, brow1, sab, sc, mark);
        // count per chunk of 32 groups (lane l reads group 32 c + l with one 16-byte load:
        // no bank conflicts); a thread owns cpt consecutive chunks for the CTA scan
        constexpr int NWARP = RT_BLOCK / 32;
        const int lane = tid & 31, warp = tid >> 5;
        const int nch = (ng + 31) >> 5;
        const uint4* __restrict__ grp4 = reinterpret_cast<const uint4*>(bitmap);
        int* s_cc = reinterpret_cast<int*>(sc->seg);   // the walk's segment arrays are free now
        for (int cc = warp; cc < nch; cc += NWARP) {
            const int g = cc * 32 + lane;
            int c = 0;
            if (g < ng) {
                const uint4 v = grp4[g];
                c = __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
            }
            c = __reduce_add_sync(0xffffffffu, c);
            if (lane == 0) s_cc[cc] = c;
        }
        __syncthreads();
        const int cpt = (nch + RT_BLOCK - 1) / RT_BLOCK;
        const int c0 = min(tid * cpt, nch), c1 = min(c0 + cpt, nch);
        int cnt = 0;
        for (int cc = c0; cc < c1; ++cc) cnt += s_cc[cc];
        int total;
        int excl = group_incl_scan<RT_BLOCK>(cnt, s_scan, total) - cnt;
        for (int cc = c0; cc < c1; ++cc) {
            const int c = s_cc[cc];
            s_cc[cc] = excl;   // rows before chunk cc
            excl += c;
        }
        const bool dense = total >= nw;
        const int64_t size = dense ? nw : total;
        if (tid == 0) {
            long long off = size > 0 ? (long long)atomicAdd(dw.store_ctr, (unsigned long long)size) : 0;
            if (off + size > dw.store_cap) {
                atomicExch(dw.err, 3);
                off = -1;
            }
            dw.soff[w] = off;
            dw.scount[w] = total;
            dw.rec[w].soff = off;
            dw.rec[w].cnt = total;
            s_off = off;
        }
        __syncthreads();
        const long long off = s_off;
        if (off >= 0 && size > 0) {
            uint32_t* __restrict__ out = dw.store + off;
            if (dense) {
                for (int x = tid; x < nw; x += RT_BLOCK) __stcs(out + x, bitmap[x]);
            } else {
                // a warp per chunk: lanes write their group's rows at warp-scanned offsets,
                // so the lanes of one store hit neighbouring addresses
                for (int cc = warp; cc < nch; cc += NWARP) {
                    const int g = cc * 32 + lane;
                    uint4 v = make_uint4(0u, 0u, 0u, 0u);
                    if (g < ng) v = grp4[g];
                    const int c = __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
                    int r = s_cc[cc] + warp_incl_scan(c) - c;
                    if (__ballot_sync(0xffffffffu, c != 0) == 0u) continue;
                    const uint32_t wv[4] = {v.x, v.y, v.z, v.w};
                    const uint32_t base = (uint32_t)(R0 + (int64_t)g * 128);
#pragma unroll
                    for (int y = 0; y < 4; ++y) {
                        uint32_t bits = wv[y];
                        while (bits) {
                            __stcs(out + r++, base + 32 * y + __ffs(bits) - 1);
                            bits &= bits - 1;
                        }
                    }
                }
            }
        }
        __syncthreads();
    }
}

// Numeric slab kernel: row set -> ranks -> C's rows, zero values, products added at their
// ranks.  Min-plus slabs of at most acc_cap entries add up in shared memory, whose 32-bit
// atomics are native (the L2 takes 2.1e11 random reductions a second whatever their width),
// and store their values once: R-MAT 18 7.0 -> 6.0 ms.  Longer ones and the other semirings
// add into C by L2 reductions: a shared FP64 addition is a compare-and-swap loop (three
// times slower than the L2 at R-MAT 20), an int64 one two atomics (20 pairs 623 -> 726 us).
// Min-plus keeps 64 registers and two CTAs per SM, the others 32 (FP64 and int64 spill 28 bytes,
// boolean 20) and four, or three where a CTA takes more than 55 KB of shared memory (slabs beyond
// about 273,000 rows).
template <class SR, bool QUADS>
__global__ void __launch_bounds__(RT_BLOCK, slab_local(SR::id) ? 2 : 4) k_slab_num(Items it, DenseWork dw, const int64_t* __restrict__ Coff,
                                                          int32_t* __restrict__ Cir, typename SR::T* __restrict__ Cv,
                                                          int acc_cap) {
    using T = typename SR::T;
    using Acc = typename SR::Acc;
    constexpr bool LOCAL = slab_local(SR::id);
    extern __shared__ __align__(16) unsigned char smem[];
    SegSmem* sc = reinterpret_cast<SegSmem*>(smem);
    uint32_t* bitmap = reinterpret_cast<uint32_t*>(smem + RS_BYTES);              // groups * 4 words
    int* gp = reinterpret_cast<int*>(bitmap + (size_t)(dw.RB / 128 + 1) * 4);    // rows before each group
    Acc* acc = reinterpret_cast<Acc*>(smem + slab_num_bytes(dw.RB));
    const int tid = threadIdx.x;
    // boolean products whose operands hold no false value: every output is true
    const bool walk = SR::id != SPGEMM_OR_AND_BOOL || dw.vals_zero == nullptr || *dw.vals_zero != 0;
    const T init = walk ? SR::out(SR::zero()) : T(1);
    const int64_t nsym = (int64_t)*dw.nitems;
    __shared__ SlabRec s_rec[2];   // this slab's record and the next one's, in flight
    constexpr int RC = sizeof(SlabRec) / 16;
    if (tid < RC && (int64_t)blockIdx.x < nsym)
        cp_async16(reinterpret_cast<int4*>(&s_rec[0]) + tid, reinterpret_cast<const int4*>(dw.rec + blockIdx.x) + tid);
    int kb = 0;
    for (int64_t w = blockIdx.x; w < nsym; w += gridDim.x, kb ^= 1) {
        if (tid < RC) cp_async_wait_all();
        __syncthreads();   // s_rec[kb] is slab w's record; s_rec[kb ^ 1] is free
        if (tid < RC && w + gridDim.x < nsym)
            cp_async16(reinterpret_cast<int4*>(&s_rec[kb ^ 1]) + tid,
                       reinterpret_cast<const int4*>(dw.rec + w + gridDim.x) + tid);
        const SlabRec& rc = s_rec[kb];
        const int cnt = rc.cnt;
        // the same for every thread of the CTA; a row set that found no room (possible
        // only with malformed input, reported by the symbolic pass) is skipped, and so is
        // one that a launch of the other form takes (k_slab_fin)
        if (cnt == 0 || rc.soff < 0) continue;
        const Prod* pr = it.prods + rc.prod;
        const int64_t R0 = rc.r0, R1 = rc.r1;
        const int nw = (int)((R1 - R0 + 31) >> 5);
        const int ng = (nw + 3) >> 2;
        const int32_t rb = rc.rb;
        const int64_t ob = rc.ob;
        const uint32_t* __restrict__ rs = dw.store + rc.soff;
        const bool dense = cnt >= nw;
        // Streaming data (the stored row sets, read once; C's rows, written once) use
        // evict-first loads and stores, so that the slab's value region, zeroed below and
        // then reduced into, stays in L2 instead of coming back from DRAM.
        // 1. the slab's row bitmap (padded to whole groups)
        if (dense) {
            for (int x = tid; x < ng * 4; x += RT_BLOCK) bitmap[x] = x < nw ? __ldcs(rs + x) : 0u;
        } else {
            for (int x = tid; x < ng * 4; x += RT_BLOCK) bitmap[x] = 0u;
            __syncthreads();
            // four rows per thread in flight: the list comes from DRAM, and one load at a
            // time left this loop waiting for it (R-MAT 20 flat FP64: 55.0 -> 51.6 ms)
            constexpr int U = 4;
            for (int i0 = tid; i0 < cnt; i0 += RT_BLOCK * U) {
                int32_t r[U];
#pragma unroll
                for (int x = 0; x < U; ++x)
                    r[x] = i0 + x * RT_BLOCK < cnt ? (int32_t)__ldcs(rs + i0 + x * RT_BLOCK) : -1;
#pragma unroll
                for (int x = 0; x < U; ++x) {
                    if (i0 + x * RT_BLOCK >= cnt) break;
                    const int lr = (int)(r[x] - R0);
                    __stcs(Cir + ob + i0 + x * RT_BLOCK, r[x] + rb);    // C's rows: the row list itself
                    atomicOr(&bitmap[lr >> 5], 1u << (lr & 31));
                }
            }
        }
        __syncthreads();
        // 2. rows before every group: chunk totals (a warp per chunk of 32 groups, lane l reads
        //    group 32 c + l: no bank conflicts), their scan by one warp, then every group's
        const int lane = tid & 31, warp = tid >> 5;
        const int nch = (ng + 31) >> 5;
        int* s_cc = reinterpret_cast<int*>(sc->seg);   // free until the walk
        for (int cc = warp; cc < nch; cc += RT_WARPS) {
            const int g = cc * 32 + lane;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (g < ng) v = reinterpret_cast<const uint4*>(bitmap)[g];
            const int c = __reduce_add_sync(0xffffffffu, __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w));
            if (lane == 0) s_cc[cc] = c;
        }
        __syncthreads();
        if (warp == 0) {
            int run = 0;
            for (int c0 = 0; c0 < nch; c0 += 32) {
                const int v = c0 + lane < nch ? s_cc[c0 + lane] : 0, inc = warp_incl_scan(v);
                if (c0 + lane < nch) s_cc[c0 + lane] = run + inc - v;
                run += __shfl_sync(0xffffffffu, inc, 31);
            }
        }
        __syncthreads();
        for (int cc = warp; cc < nch; cc += RT_WARPS) {
            const int g = cc * 32 + lane;
            uint4 v = make_uint4(0u, 0u, 0u, 0u);
            if (g < ng) v = reinterpret_cast<const uint4*>(bitmap)[g];
            const int c = __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
            const int r = s_cc[cc] + warp_incl_scan(c) - c;
            if (g < ng) gp[g] = r;
        }
        __syncthreads();
        // 3. C's rows of a bitmap slab: a warp per chunk of 32 groups; lanes write their
        //    group's rows from its rank base, or, for chunks of at least 16 rows a word,
        //    the warp writes one word at a time (lane l: bit l), so that every store
        //    covers neighbouring addresses
        if (dense) {
            const uint4* __restrict__ grp4 = reinterpret_cast<const uint4*>(bitmap);
            for (int cc = warp; cc < nch; cc += RT_WARPS) {
                const int g = cc * 32 + lane;
                uint4 v = make_uint4(0u, 0u, 0u, 0u);
                if (g < ng) v = grp4[g];
                const int c = __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
                const int tot = __reduce_add_sync(0xffffffffu, c);
                if (tot == 0) continue;
                int r = g < ng ? gp[g] : 0;
                const int32_t base = (int32_t)(R0 + (int64_t)g * 128) + rb;
                const uint32_t wv[4] = {v.x, v.y, v.z, v.w};
                if (tot >= 2048) {
                    for (int src = 0; src < 32; ++src) {
                        int ry = __shfl_sync(0xffffffffu, r, src);
                        const int32_t by = __shfl_sync(0xffffffffu, base, src);
#pragma unroll
                        for (int y = 0; y < 4; ++y) {
                            const uint32_t wy = __shfl_sync(0xffffffffu, wv[y], src);
                            if ((wy >> lane) & 1u)
                                __stcs(Cir + ob + ry + __popc(wy & ((1u << lane) - 1u)), by + 32 * y + lane);
                            ry += __popc(wy);
                        }
                    }
                } else {
#pragma unroll
                    for (int y = 0; y < 4; ++y) {
                        uint32_t bits = wv[y];
                        while (bits) {
                            __stcs(Cir + ob + r++, base + 32 * y + __ffs(bits) - 1);
                            bits &= bits - 1;
                        }
                    }
                }
            }
        }
        // 4. values: the semiring zero (all true for the boolean shortcut)
        const bool local = LOCAL && cnt <= acc_cap;
        if (local)
            for (int i = tid; i < cnt; i += RT_BLOCK) acc[i] = SR::zero();
        else
            for (int i = tid; i < cnt; i += RT_BLOCK) Cv[ob + i] = init;
        __syncthreads();   // the stores above come before this CTA's additions
        // 5. every product, added at its row's rank
        if (walk) {
            const int span = (int)(R1 - R0);
            const int32_t r0 = (int32_t)R0;
            // rank of a row in the slab's set; -1 for rows outside it (malformed input only)
            auto rank_of = [&](int32_t row) {
                const int lr = row - r0;
                if ((unsigned)lr >= (unsigned)span) return -1;
                const int wd = lr >> 5, g = wd >> 2, y = wd & 3;
                const uint4 grp = reinterpret_cast<const uint4*>(bitmap)[g];
                const uint32_t wv = y == 0 ? grp.x : y == 1 ? grp.y : y == 2 ? grp.z : grp.w;
                const uint32_t bit = 1u << (lr & 31);
                if (!(wv & bit)) return -1;
                return gp[g] + __popc(wv & (bit - 1u)) + (y > 0 ? __popc(grp.x) : 0) + (y > 1 ? __popc(grp.y) : 0) +
                       (y > 2 ? __popc(grp.z) : 0);
            };
            const int64_t bs = rc.bs, be = rc.be;
            const int32_t* brow0 = dw.bnd + rc.bnd;
            const int32_t* brow1 = brow0 + (be - bs);
            const int32_t* sab = dw.bnd + rc.sab;
            if (LOCAL && local) {
                slab_products<SR, true, QUADS>(pr, bs, be, brow0, brow1, sab, sc, [&](int32_t row, T a, T b) {
                    const int rank = rank_of(row);
                    if (rank >= 0 && rank < cnt) SR::atomic_add(acc + rank, SR::mul(a, b));
                });
                for (int i = tid; i < cnt; i += RT_BLOCK) __stcs(Cv + ob + i, SR::out(acc[i]));
            } else {
                slab_products<SR, true, QUADS>(pr, bs, be, brow0, brow1, sab, sc, [&](int32_t row, T a, T b) {
                    const int rank = rank_of(row);
                    if (rank >= 0) red_out<SR>(Cv, ob + rank, SR::mul(a, b));
                });
            }
        } else {
            __syncthreads();
        }
    }
}

// Completes the slab records for the numeric pass: where each slab's rows start in C.  With both
// kinds of products (only_quads 0 or 1, else -1) the records of the other kind lose their row set
// for the launch that follows.
__global__ void k_slab_fin(Items it, DenseWork dw, const int64_t* __restrict__ Coff, int only_quads) {
    const int64_t nsym = (int64_t)*dw.nitems;
    for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < nsym; w += (int64_t)gridDim.x * blockDim.x) {
        dw.rec[w].ob = __ldg(Coff + dw.rec[w].u) + dw.spref[w];
        if (only_quads >= 0)
            dw.rec[w].soff = quads_ok(it.prods + dw.rec[w].prod) == (only_quads != 0) ? dw.soff[w] : -1;
    }
}

bool slab_quads(const Prod& pr) { return quads_ok(&pr); }

// CTAs per SM the kernel can keep resident with `smem` bytes, times the SM count
static int resident_grid(const void* fn, int block, size_t smem) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, block, smem) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    return per_sm * sm_count();
}

template <class SR>
static void run_slabs(const Lanes& lanes, const Items& it, const DenseWork& dw, bool numeric, const int64_t* Coff,
                      int32_t* Cir, typename SR::T* Cv) {
    if (dw.ndense <= 0) return;
    const cudaStream_t st = lanes.next();
    const int64_t nslab_max = dw.nslabs > 0 ? dw.nslabs : dw.ndense * MAX_PARTS;
    if (!numeric) {
        const int bnd_block = dw.many_short ? 128 : 256;
        k_slab_bounds<<<(int)std::min<int64_t>(nslab_max, sm_count() * (2048 / bnd_block)), bnd_block, 0, st>>>(it, dw);
        note_launch();
        const size_t smem = RS_BYTES + (size_t)(dw.RB / 128 + 1) * 16;
        for (int kind = 0; kind < 2; ++kind) {
            if (!((dw.kinds >> kind) & 1)) continue;
            auto kern = kind == 0 ? k_slab_sym<true> : k_slab_sym<false>;
            smem_at_least((const void*)kern, smem);
            const int grid = (int)std::min<int64_t>(nslab_max, resident_grid((const void*)kern, RT_BLOCK, smem));
            kern<<<grid, RT_BLOCK, smem, st>>>(it, dw, dw.kinds == 3);
            note_launch();
        }
    } else {
        const int acc_cap = slab_acc_entries(SR::id, dw.RB);
        const size_t smem = slab_num_bytes(dw.RB) + (size_t)acc_cap * sizeof(typename SR::Acc);
        for (int kind = 0; kind < 2; ++kind) {
            if (!((dw.kinds >> kind) & 1)) continue;
            k_slab_fin<<<(int)std::min<int64_t>(ceil_div64(nslab_max, 256), sm_count() * 8), 256, 0, st>>>(
                it, dw, Coff, dw.kinds == 3 ? kind == 0 : -1);
            note_launch();
            auto kern = kind == 0 ? k_slab_num<SR, true> : k_slab_num<SR, false>;
            smem_at_least((const void*)kern, smem);
            const int grid = (int)std::min<int64_t>(nslab_max, resident_grid((const void*)kern, RT_BLOCK, smem));
            kern<<<grid, RT_BLOCK, smem, st>>>(it, dw, Coff, Cir, Cv, acc_cap);
            note_launch();
        }
    }
}

template <class SR>
void launch_numeric_predicted(const Lanes& st, const Items& it, const int2* list, const int64_t* bin_off,
                              const int64_t* bin_cnt, const DenseWork& dw, const int64_t* cap_off, int64_t* nnz_item,
                              int32_t* Cir, typename SR::T* Cv) {
    if (block_mode(it)) {
        run_short<SR, true>(st, it, list, bin_off, bin_cnt, nnz_item, cap_off, Cir, Cv, dw.vals_zero);
        launch_block_tier<SR>(st, it, list, bin_off, bin_cnt, dw, nnz_item, cap_off, Cir, Cv, 1);
        return;
    }
    run_hash_bins<SR, true>(st, it, list, bin_off, bin_cnt, nnz_item, cap_off, Cir, Cv, dw.vals_zero);
}

template <class SR>
void launch_symbolic(const Lanes& st, const Items& it, TierCfg cfg, const int2* list, const int64_t* bin_off,
                     const int64_t* bin_cnt, const DenseWork& dw, int64_t* nnz_item, int which) {
    (void)cfg;
    if (which & 2) {   // the longest launches first
        if (dw.dcol) run_bitcount<256, 256>(st, it, dw.dlist, dw.ndense, nnz_item);   // rows fit the bitmap
        else run_slabs<SR>(st, it, dw, false, nullptr, nullptr, nullptr);
    }
    if (which & 1) run_hash_bins<SR, false>(st, it, list, bin_off, bin_cnt, nnz_item, nullptr, nullptr, nullptr);
}

template <class SR>
void launch_numeric(const Lanes& st, const Items& it, TierCfg cfg, const int2* list, const int64_t* bin_off,
                    const int64_t* bin_cnt, const DenseWork& dw, const int64_t* Coff, int32_t* Cir,
                    typename SR::T* Cv, int which) {
    (void)cfg;
    if (block_mode(it)) {
        if (which & 1) run_short<SR, true>(st, it, list, bin_off, bin_cnt, nullptr, Coff, Cir, Cv, dw.vals_zero);
        launch_block_tier<SR>(st, it, list, bin_off, bin_cnt, dw, nullptr, Coff, Cir, Cv, which);
        return;
    }
    if (which & 1) run_hash_bins<SR, true>(st, it, list, bin_off, bin_cnt, nullptr, Coff, Cir, Cv, dw.vals_zero);
    if (which & 2) run_slabs<SR>(st, it, dw, true, Coff, Cir, Cv);
}

#define SG_INST(SR)                                                                                              \
    template void launch_symbolic<SR>(const Lanes&, const Items&, TierCfg, const int2*, const int64_t*,          \
                                      const int64_t*, const DenseWork&, int64_t*, int);                          \
    template void launch_numeric<SR>(const Lanes&, const Items&, TierCfg, const int2*, const int64_t*,           \
                                     const int64_t*, const DenseWork&, const int64_t*, int32_t*, typename SR::T*, \
                                     int);                                                                       \
    template void launch_numeric_predicted<SR>(const Lanes&, const Items&, const int2*, const int64_t*,          \
                                               const int64_t*, const DenseWork&, const int64_t*, int64_t*, int32_t*, \
                                               typename SR::T*);
SG_INST(PT64)
SG_INST(MP32)
SG_INST(BOOL8)
SG_INST(PTI64)
#undef SG_INST


// ------------------------------------------------------------------ part sums, colptrs, stats
// nnz of a long column = the sum of its slab counts; spref[s] = rows of the
// column's earlier slabs (where slab s starts inside the column)
__global__ void k_sum_parts(Items it, DenseWork dw, int64_t* __restrict__ nnz_item) {
    const int64_t d = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= dw.ndense) return;
    const int P = dw.nparts[d];
    const int64_t s0 = dw.sbase[d];
    int32_t acc = 0;
    for (int q = 0; q < P; ++q) {
        dw.spref[s0 + q] = acc;
        acc += dw.scount[s0 + q];
    }
    const int2 e = dw.dlist[d];
    nnz_item[__ldg(it.item_base + e.x) + e.y] = acc;
}

void launch_sum_parts(cudaStream_t st, const Items& it, const DenseWork& dw, int64_t* nnz_item) {
    if (dw.ndense == 0 || dw.dcol) return;   // the dense-column mode counted directly
    k_sum_parts<<<(int)ceil_div64(dw.ndense, 256), 256, 0, st>>>(it, dw, nnz_item);
    note_launch();
}

// colptr_i[j] = offset of the first stored column of B_i with id >= j, relative to the product's start
__global__ void k_colptrs(Items it, const int64_t* __restrict__ colbase, int64_t total, const int64_t* __restrict__ Coff,
                          int64_t* __restrict__ out) {
    for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total; x += (int64_t)gridDim.x * blockDim.x) {
        int prod = it.nprod == 1 ? 0 : find_prod(colbase, it.nprod, x);
        const Prod* pr = it.prods + prod;
        const int64_t j = x - colbase[prod];
        const int64_t ib = __ldg(it.item_base + prod);
        const int64_t nzc = pr->B.nzc;
        int64_t p;
        if (pr->B.jc == nullptr) {
            p = j;
        } else {
            int64_t lo = 0, hi = nzc;
            while (lo < hi) {
                int64_t mid = (lo + hi) >> 1;
                if ((int64_t)__ldg(pr->B.jc + mid) < j) lo = mid + 1;
                else hi = mid;
            }
            p = lo;
        }
        out[x] = Coff[ib + p] - Coff[ib];
    }
}

__global__ void k_gather_offsets(const int64_t* __restrict__ Coff, const int64_t* __restrict__ item_base, int64_t np,
                                 int64_t* __restrict__ out) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= np; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = Coff[item_base[i]];
}

void launch_gather_offsets(cudaStream_t st, const int64_t* Coff, const int64_t* item_base, int64_t np, int64_t* out) {
    k_gather_offsets<<<(int)ceil_div64(np + 1, 256), 256, 0, st>>>(Coff, item_base, np, out);
    note_launch();
}

void launch_colptrs(cudaStream_t st, const Items& it, const int64_t* colbase, int64_t total_cols, const int64_t* Coff,
                    int64_t* out) {
    if (total_cols <= 0) return;
    int grid = (int)std::min<int64_t>(ceil_div64(total_cols, 256), sm_count() * 16);
    k_colptrs<<<grid, 256, 0, st>>>(it, colbase, total_cols, Coff, out);
    note_launch();
}

__global__ void k_fill_i64(int64_t* p, int64_t n, int64_t v) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        p[i] = v;
}

void launch_fill_i64(cudaStream_t st, int64_t* p, int64_t n, int64_t v) {
    if (n <= 0) return;
    int grid = (int)std::min<int64_t>(ceil_div64(n, 256), sm_count() * 16);
    k_fill_i64<<<grid, 256, 0, st>>>(p, n, v);
    note_launch();
}

__global__ void k_tier_stats(Items it, const uint8_t* __restrict__ bin, const int32_t* __restrict__ item_prod,
                             const int64_t* __restrict__ flops, const int64_t* __restrict__ nnz_item, int warp_max,
                             unsigned long long* out) {
    __shared__ unsigned long long s[16];
    if (threadIdx.x < 16) s[threadIdx.x] = 0;
    __syncthreads();
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < it.nitems;
         u += (int64_t)gridDim.x * blockDim.x) {
        int b = bin[u];
        int prod = item_prod[u];
        const Prod* pr = it.prods + prod;
        int t = tier_of_bin(b, min(flops[u], pr->A.m), warp_max);
        int64_t p = u - __ldg(it.item_base + prod);
        atomicAdd(&s[t], 1ull);
        atomicAdd(&s[4 + t], (unsigned long long)flops[u]);
        atomicAdd(&s[8 + t], (unsigned long long)nnz_item[u]);
        atomicAdd(&s[12 + t], (unsigned long long)(pr->B.cp[p + 1] - pr->B.cp[p]));
    }
    __syncthreads();
    if (threadIdx.x < 16 && s[threadIdx.x]) atomicAdd(out + threadIdx.x, s[threadIdx.x]);
}

void launch_tier_stats(cudaStream_t st, const Items& it, const uint8_t* bin, const int32_t* item_prod,
                       const int64_t* flops, const int64_t* nnz_item, int warp_max, unsigned long long* out) {
    if (it.nitems <= 0) return;
    int grid = (int)std::min<int64_t>(ceil_div64(it.nitems, 256), sm_count() * 4);
    k_tier_stats<<<grid, 256, 0, st>>>(it, bin, item_prod, flops, nnz_item, warp_max, out);
    note_launch();
}

// ------------------------------------------------------------------ device-wide exclusive scan
constexpr int SCAN_BLOCK = 1024;
constexpr int SCAN_ITEMS = 4;
constexpr int SCAN_TILE = SCAN_BLOCK * SCAN_ITEMS;
// up to this many tiles every CTA of the second pass adds the earlier tiles' sums itself
// (two 8-byte loads per thread at most); more tiles take a launch of their own for that
constexpr int64_t SCAN_SELF_TILES = 2 * SCAN_BLOCK;

__device__ __forceinline__ long long block_excl_scan64(long long v, long long* ws, long long& total) {
    long long x = warp_incl_scan64(v);
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 31) ws[w] = x;
    __syncthreads();
    if (w == 0) {
        long long s = ws[lane];
        s = warp_incl_scan64(s);
        ws[lane] = s;
    }
    __syncthreads();
    long long add = w > 0 ? ws[w - 1] : 0;
    total = ws[31];
    __syncthreads();
    return x + add - v;
}

// The end of the counting pass was five launches, two uploads and a memset: three scan
// launches, the bins from the counts (every thread adding to the same shared counters, 15 us
// for 4,096 columns), their offsets through the host, and the lists.  It is one launch up to
// 4,096 columns (9.5 us) and two up to 8 million: ER 4096^2 flat, a whole call, 137 -> 95 us.
// The lists take one round for a thread's four items, whose places in a warp stay close
// together: four rounds, one item each, took 11.2 us there and put every fourth column of a
// tile after one another (R*(A*P) on 128^3, a whole call, 646 against 626 us).
// What the scan of the exact counts does besides: the numeric bin of every item (hash tables
// need only 2 nnz slots, not 2 min(flops, m); slab-tier and empty items get bin 0, not
// listed), the bins' counts, and their lists.
struct CountBins {
    Items it;
    TierCfg cfg;
    const uint8_t* bin;
    const int64_t* flops;
    const int32_t* item_prod;
    uint8_t* nbin;
    unsigned long long* cnt;      // NBIN counts (zeroed by the caller)
    unsigned long long* cursor;   // NBIN cursors (zeroed by the caller)
    int2* list;
};

__device__ __forceinline__ int numeric_bin(const CountBins& nb, int64_t u, int64_t nnz) {
    const int b = nb.bin[u];
    if (b < BIN_SORT0 || b >= BIN_DENSE) return 0;
    return bin_of(nb.flops[u], nnz, nb.cfg.warp_max, nb.cfg.block_max, nb.cfg.sort_max);
}

// adds one thread's bin (b <= 0: none) to the CTA's counts; whole warps call it
__device__ __forceinline__ void count_bin(int b, int* s_n) {
    const unsigned peers = __match_any_sync(0xffffffffu, b);
    if (b > 0 && (int)(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&s_n[b], __popc(peers));
}

// First pass: the sum of every tile, and with BINS the numeric bins and their counts.
template <bool BINS>
__global__ void __launch_bounds__(SCAN_BLOCK) k_scan_reduce(const int64_t* __restrict__ in, int64_t n,
                                                             long long* __restrict__ sums, CountBins nb) {
    __shared__ long long ws[32];
    __shared__ int s_n[NBIN];
    if constexpr (BINS) {
        if (threadIdx.x < NBIN) s_n[threadIdx.x] = 0;
        __syncthreads();
    }
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
    long long s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        const int64_t u = base + i * SCAN_BLOCK + threadIdx.x;
        const long long v = u < n ? in[u] : 0;
        s += v;
        if constexpr (BINS) {
            const int b = u < n ? numeric_bin(nb, u, v) : 0;
            if (u < n) nb.nbin[u] = (uint8_t)b;
            count_bin(b, s_n);
        }
    }
    long long total;
    block_excl_scan64(s, ws, total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
    if constexpr (BINS) {
        if (threadIdx.x < NBIN && s_n[threadIdx.x])
            atomicAdd(nb.cnt + threadIdx.x, (unsigned long long)s_n[threadIdx.x]);
    }
}

__global__ void __launch_bounds__(SCAN_BLOCK) k_scan_sums(long long* sums, int64_t nb) {
    __shared__ long long ws[32];
    long long carry = 0;
    for (int64_t b0 = 0; b0 < nb; b0 += SCAN_BLOCK) {
        int64_t i = b0 + threadIdx.x;
        long long v = i < nb ? sums[i] : 0;
        long long total;
        long long ex = block_excl_scan64(v, ws, total);
        if (i < nb) sums[i] = carry + ex;
        carry += total;
    }
}

// Second pass: out[u + 1] for the CTA's tile, after the earlier tiles (`summed`: sums already
// holds their exclusive scan).  With BINS also the numeric lists; a single tile makes its own
// bins and counts first, so that the whole step is this one launch.
template <bool BINS>
__global__ void __launch_bounds__(SCAN_BLOCK) k_scan_apply(const int64_t* __restrict__ in, int64_t n,
                                                            const long long* __restrict__ sums, bool summed,
                                                            int64_t* __restrict__ out, CountBins nb) {
    __shared__ long long ws[32];
    __shared__ int64_t s_off[NBIN], s_base[NBIN];
    __shared__ int s_n[NBIN];
    long long before = 0;
    if (summed) {
        before = sums[blockIdx.x];
    } else if (blockIdx.x > 0) {
        long long s = 0;
        for (int64_t t = threadIdx.x; t < blockIdx.x; t += SCAN_BLOCK) s += sums[t];
        block_excl_scan64(s, ws, before);
    }
    const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_ITEMS;
    long long v[SCAN_ITEMS];
    long long s = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        v[i] = base + i < n ? in[base + i] : 0;
        s += v[i];
    }
    long long total;
    long long ex = block_excl_scan64(s, ws, total) + before;
    if (blockIdx.x == 0 && threadIdx.x == 0) out[0] = 0;
#pragma unroll
    for (int i = 0; i < SCAN_ITEMS; ++i) {
        ex += v[i];
        if (base + i < n) out[base + i + 1] = ex;
    }
    if constexpr (BINS) {
        const bool single = gridDim.x == 1;
        int b[SCAN_ITEMS], at[SCAN_ITEMS];
        if (threadIdx.x < NBIN) s_n[threadIdx.x] = 0;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < SCAN_ITEMS; ++i) {
            const int64_t u = base + i;
            b[i] = u >= n ? 0 : single ? numeric_bin(nb, u, v[i]) : nb.nbin[u];
            if (single && u < n) nb.nbin[u] = (uint8_t)b[i];
            at[i] = bin_rank(b[i], s_n);
        }
        __syncthreads();
        if (single) {   // the CTA's counts are the counts
            if (threadIdx.x < 32) {
                const int t = threadIdx.x, c = t < NBIN ? s_n[t] : 0;
                const long long inc = warp_incl_scan64(c);
                if (t < NBIN) {
                    nb.cnt[t] = (unsigned long long)c;
                    s_base[t] = inc - c;
                }
            }
            __syncthreads();
        } else {
            bin_offsets(nb.cnt, 1, s_off);
            bin_bases(nb.cursor, s_off, s_n, s_base);
        }
#pragma unroll
        for (int i = 0; i < SCAN_ITEMS; ++i) {
            if (b[i] > 0) {
                const int prod = nb.item_prod[base + i];
                nb.list[s_base[b[i]] + at[i]] = make_int2(prod, (int)(base + i - __ldg(nb.it.item_base + prod)));
            }
        }
    }
}

size_t scan_tmp_bytes(int64_t n) { return (size_t)(ceil_div64(std::max<int64_t>(n, 1), SCAN_TILE) + 1) * 8; }

template <bool BINS>
static void run_scan(cudaStream_t st, const int64_t* in, int64_t n, int64_t* out, void* tmp, const CountBins& nb) {
    const int64_t nt = ceil_div64(n, SCAN_TILE);
    long long* sums = reinterpret_cast<long long*>(tmp);
    const bool summed = nt > SCAN_SELF_TILES;
    if (nt > 1) {
        k_scan_reduce<BINS><<<(int)nt, SCAN_BLOCK, 0, st>>>(in, n, sums, nb);
        note_launch();
    }
    if (summed) {
        k_scan_sums<<<1, SCAN_BLOCK, 0, st>>>(sums, nt);
        note_launch();
    }
    k_scan_apply<BINS><<<(int)nt, SCAN_BLOCK, 0, st>>>(in, n, sums, summed, out, nb);
    note_launch();
}

void launch_exclusive_scan(cudaStream_t st, const int64_t* in, int64_t n, int64_t* out, void* tmp) {
    if (n <= 0) {
        cudaMemsetAsync(out, 0, sizeof(int64_t), st);
        return;
    }
    run_scan<false>(st, in, n, out, tmp, CountBins());
}

void launch_count_scan(cudaStream_t st, const Items& it, TierCfg cfg, const uint8_t* bin, const int64_t* flops,
                       const int32_t* item_prod, const int64_t* nnz_item, int64_t* out, void* tmp, uint8_t* nbin,
                       unsigned long long* cnt, int2* list) {
    if (it.nitems <= 0) {
        cudaMemsetAsync(out, 0, sizeof(int64_t), st);
        return;
    }
    run_scan<true>(st, nnz_item, it.nitems, out, tmp, CountBins{it, cfg, bin, flops, item_prod, nbin, cnt, cnt + NBIN, list});
}

}  // namespace sg
