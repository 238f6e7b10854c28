// Truncation of Eq. 11 and the ordering of sparse vectors.
//
// top-k: the k entries with the largest |c|, ties to the smaller rank, exact
// zeros excluded, decided exactly on bit patterns.  Each entry maps to a
// 127-bit composite X = (0x7fff...f - bits(|c|)) : rank, so the wanted entries
// are the k smallest X (for non-negative doubles the bit pattern orders like
// the value).  A radix select walks X from the top in 12-bit digits (the last
// digit has 7 bits): each pass histograms the digit of the entries whose
// higher digits equal the prefix found so far, and the block that finishes its
// part last picks the bin that holds the k-th smallest.  All state stays on the
// device; a pass that finds its bin exactly full ends the search early.  A last
// pass gathers every entry whose prefix is <= the threshold prefix.  Up to
// kSmall items one CTA does all passes in shared memory.
//
// sort: stable LSD radix sort of (uint64 key, double val) pairs with 8-bit
// digits over the significant key bits only (ceil(log2(dim)) bits): one pass
// counts every digit of every key (digits that all keys share are skipped),
// then per digit a histogram per tile, one scan per digit value over the
// tiles, and a stable scatter ranked per warp with __match_any_sync.  Up to
// kSmall pairs one CTA sorts in shared memory.
//
// What bounds it: at 3e6 items (48 MB) launches and the chain of passes, not
// bandwidth; the 2e5 largest of 3e6, sorted: 554 us with one-block scans over
// all counters and a pick launch per pass, 379 us so.  Where the capacity is
// far above the count, the kernels follow the count: an unsorted sigma of 2.2e7
// entries 60.2 ms when sorting over the capacity, 27.3 ms so.  A step on the
// whole 4900-determinant space: 1066 us with 30 launches a sort, 839 us so.
// With a pass of up to 256 tiles in one launch and only the partial sums that are
// there added: 379 -> 324 us, that step 599 -> 538 us.
#include <algorithm>

#include "sfci_internal.cuh"

namespace sfci {
namespace {

constexpr int kT = 256;
constexpr int kBins = 4096;
constexpr int kPasses = 11;  // 10 x 12 bits + 7 bits = 127
constexpr int kRedBlocks = 304;
// one CTA's shared memory holds this many pairs and its counters; below it a launch
// costs more than the work (10 to 30 launches of 2 to 5 us against one of 20 to 40 us)
constexpr int kSmall = 8192;
constexpr int kSmallT = 1024;

__host__ __device__ inline int pass_width(int p) { return p < 10 ? 12 : 7; }
__host__ __device__ inline int pass_low(int p) { return 127 - 12 * p - pass_width(p); }

struct SelState {
    unsigned long long pfx_hi, pfx_lo, mask_hi, mask_lo;
    unsigned long long need, total;
    int done, all, pass;
    unsigned ticket;  // blocks that have finished the pass's histogram
    double sumsq;
};

struct SelLayout {
    size_t state, hist, n_gather, result, bytes;
};

inline size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

SelLayout sel_layout() {
    SelLayout L{};
    size_t o = 0;
    L.state = o, o = a256(o + sizeof(SelState));
    L.hist = o, o = a256(o + sizeof(unsigned long long) * kBins);
    L.n_gather = o, o = a256(o + sizeof(unsigned long long));
    L.result = o, o = a256(o + sizeof(SplitResult));
    L.bytes = o;
    return L;
}

__device__ __forceinline__ bool item_valid(unsigned long long key, unsigned long long vbits) {
    return key != kEmpty && (vbits & 0x7fffffffffffffffull) != 0ull;
}

__device__ __forceinline__ unsigned digit_of(unsigned long long hi, unsigned long long lo, int p,
                                             int w) {
    unsigned long long v;
    if (p >= 64) v = hi >> (p - 64);
    else if (p + w <= 64) v = lo >> p;
    else v = (lo >> p) | (hi << (64 - p));
    return (unsigned)(v & ((1ull << w) - 1ull));
}

__global__ void sel_init_kernel(SelState *s, unsigned long long k, unsigned long long *hist,
                                unsigned long long *n_gather) {
    if (threadIdx.x == 0) {
        s->pfx_hi = s->pfx_lo = s->mask_hi = s->mask_lo = 0ull;
        s->need = k;
        s->total = 0;
        s->done = (k == 0);
        s->all = 0;
        s->pass = 0;
        s->ticket = 0;
        s->sumsq = 0.0;
        *n_gather = 0;
    }
    for (int b = threadIdx.x; b < kBins; b += blockDim.x) hist[b] = 0;
}

// the prefix and mask extended by digit b of the pass
__device__ __forceinline__ void sel_extend(SelState *s, unsigned b, int pass) {
    const int w = pass_width(pass), p = pass_low(pass);
    const unsigned long long dm = (1ull << w) - 1ull;
    // set digit b at bits [p, p+w) of the composite prefix and mask
    if (p >= 64) {
        s->pfx_hi |= (unsigned long long)b << (p - 64);
        s->mask_hi |= dm << (p - 64);
    } else if (p + w <= 64) {
        s->pfx_lo |= (unsigned long long)b << p;
        s->mask_lo |= dm << p;
    } else {
        s->pfx_lo |= (unsigned long long)b << p;
        s->mask_lo |= dm << p;
        s->pfx_hi |= (unsigned long long)b >> (64 - p);
        s->mask_hi |= dm >> (64 - p);
    }
}

// One block: choose the bin holding the need-th smallest.  Each thread owns kBins / T
// consecutive bins; a warp scan and a scan of the warps' sums find the thread.
template <int T>
__device__ void sel_pick(SelState *s, const unsigned long long *hist, int pass) {
    __shared__ unsigned long long wsum[T / 32];
    __shared__ int found_bin;
    __shared__ unsigned long long found_before, found_count;
    constexpr int per = kBins / T;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned long long need = s->need;
    if (pass == 0 && __ldcg(&s->total) <= need) {
        __syncthreads();
        if (tid == 0) s->all = 1, s->done = 1;
        return;
    }
    unsigned long long mine = 0;
    for (int q = 0; q < per; ++q) mine += __ldcg(&hist[tid * per + q]);
    unsigned long long x = mine;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    if (tid == 0) found_bin = -1;
    __syncthreads();
    unsigned long long before = x - mine;
    for (int w = 0; w < warp; ++w) before += wsum[w];
    if (before < need && before + mine >= need) {
        unsigned long long run = before;
        for (int q = 0; q < per; ++q) {
            const unsigned long long c = __ldcg(&hist[tid * per + q]);
            if (run + c >= need) {
                found_bin = tid * per + q;
                found_before = run;
                found_count = c;
                break;
            }
            run += c;
        }
    }
    __syncthreads();
    if (tid == 0) {
        // found_bin < 0 cannot happen for need <= total; stop instead of looping on
        sel_extend(s, found_bin < 0 ? 0u : (unsigned)found_bin, pass);
        s->need = need - (found_bin < 0 ? 0ull : found_before);
        if (found_bin < 0 || found_count == s->need || pass == kPasses - 1) s->done = 1;
        s->pass = pass + 1;
    }
}

// want_sq: also the sum of squares (a float64 add per item: 12 us for 3e6 items)
__global__ void sel_hist_kernel(Items it, SelState *s, unsigned long long *hist, int pass, int want_sq) {
    __shared__ unsigned sh[kBins];
    __shared__ double ssq[kT / 32];
    __shared__ unsigned long long scount[kT / 32];
    __shared__ bool last;
    if (s->done) return;
    for (int b = threadIdx.x; b < kBins; b += blockDim.x) sh[b] = 0;
    __syncthreads();
    const unsigned long long ph = s->pfx_hi, pl = s->pfx_lo, mh = s->mask_hi, ml = s->mask_lo;
    const int w = pass_width(pass), p = pass_low(pass);
    double sq = 0.0;
    unsigned long long cnt = 0;
    // four items in flight per thread (one: 20 us for 3e6 values that lie in L2)
    constexpr int U = 4;
    const long long step = (long long)gridDim.x * blockDim.x;
    for (long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x; i0 < it.n; i0 += U * step) {
        unsigned long long vb[U], key[U];
        bool fits[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const long long i = i0 + u * step;
            vb[u] = i < it.n ? (unsigned long long)__double_as_longlong(it.val[(size_t)i * it.stride]) : 0ull;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {  // (the key is read only where the value's prefix fits)
            const unsigned long long hi = 0x7fffffffffffffffull - (vb[u] & 0x7fffffffffffffffull);
            fits[u] = i0 + u * step < it.n && !(pass > 0 && (hi & mh) != ph);
            key[u] = fits[u] ? it.key[(size_t)(i0 + u * step) * it.stride] : 0ull;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (!fits[u] || !item_valid(key[u], vb[u])) continue;
            const unsigned long long hi = 0x7fffffffffffffffull - (vb[u] & 0x7fffffffffffffffull);
            if (pass == 0) {
                cnt += 1;
                if (want_sq) {
                    const double v = __longlong_as_double((long long)vb[u]);
                    sq += v * v;
                }
            }
            if ((key[u] & ml) != pl) continue;
            atomicAdd(&sh[digit_of(hi, key[u], p, w)], 1u);
        }
    }
    if (pass == 0) {
        for (int o = 16; o > 0; o >>= 1) {
            sq += __shfl_xor_sync(kFull, sq, o);
            cnt += __shfl_xor_sync(kFull, cnt, o);
        }
        if ((threadIdx.x & 31) == 0) ssq[threadIdx.x >> 5] = sq, scount[threadIdx.x >> 5] = cnt;
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kBins; b += blockDim.x)
        if (sh[b]) atomicAdd(&hist[b], (unsigned long long)sh[b]);
    if (pass == 0 && threadIdx.x == 0) {
        double a = 0.0;
        unsigned long long c = 0;
        for (int q = 0; q < kT / 32; ++q) a += ssq[q], c += scount[q];
        if (want_sq) atomicAdd(&s->sumsq, a);
        atomicAdd(&s->total, c);
    }
    // the last block to get here picks the bin and clears the histogram
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&s->ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    sel_pick<kT>(s, hist, pass);
    __syncthreads();
    for (int q = threadIdx.x; q < kBins; q += blockDim.x) hist[q] = 0;
    if (threadIdx.x == 0) s->ticket = 0;
}

// The whole selection of up to kSmall items by one CTA, the items in shared memory:
// the passes over 12-bit digits, then the chosen ones in order.
__global__ void __launch_bounds__(kSmallT)
sel_small_kernel(Items it, unsigned long long k, unsigned long long *out_key, double *out_val,
                 unsigned long long *n_out, double *sumsq_out, unsigned long long *total_out) {
    extern __shared__ __align__(16) unsigned char sm[];
    unsigned long long *key = reinterpret_cast<unsigned long long *>(sm);
    unsigned long long *vb = key + kSmall;
    unsigned *hist = reinterpret_cast<unsigned *>(vb + kSmall);
    __shared__ unsigned long long ph, pl, mh, ml, need;
    __shared__ int done, all, found;
    __shared__ unsigned wsum[kSmallT / 32], found_before;
    __shared__ double ssq[kSmallT / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = (int)it.n;
    double sq = 0.0;
    unsigned cnt = 0;
    for (int i = tid; i < n; i += kSmallT) {
        const unsigned long long kk = it.key[(size_t)i * it.stride];
        unsigned long long v = (unsigned long long)__double_as_longlong(it.val[(size_t)i * it.stride]);
        if (!item_valid(kk, v)) v = 0ull;  // (a zero value marks an item that does not count)
        else {
            ++cnt;
            if (sumsq_out) sq += __longlong_as_double((long long)v) * __longlong_as_double((long long)v);
        }
        key[i] = kk, vb[i] = v;
    }
    cnt = __reduce_add_sync(kFull, cnt);
    if (sumsq_out)
        for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(kFull, sq, o);
    if (lane == 0) ssq[warp] = sq, wsum[warp] = cnt;
    __syncthreads();
    if (tid == 0) {
        double a = 0.0;
        unsigned long long c = 0;
        for (int w = 0; w < kSmallT / 32; ++w) {
            c += wsum[w];
            if (sumsq_out) a += ssq[w];
        }
        need = k, ph = pl = mh = ml = 0ull;
        all = c <= k, done = all || k == 0;
        if (sumsq_out) *sumsq_out = a;
        if (total_out) *total_out = c;
    }
    __syncthreads();
    constexpr int per = kBins / kSmallT;
    for (int pass = 0; pass < kPasses && !done; ++pass) {
        const int w = pass_width(pass), p = pass_low(pass);
        for (int q = 0; q < per; ++q) hist[tid * per + q] = 0u;
        if (tid == 0) found = -1;
        __syncthreads();
        for (int i = tid; i < n; i += kSmallT) {
            const unsigned long long v = vb[i], hi = 0x7fffffffffffffffull - (v & 0x7fffffffffffffffull);
            if ((v << 1) != 0ull && (hi & mh) == ph && (key[i] & ml) == pl) atomicAdd(&hist[digit_of(hi, key[i], p, w)], 1u);
        }
        __syncthreads();
        unsigned mine = 0;
        for (int q = 0; q < per; ++q) mine += hist[tid * per + q];
        unsigned x = mine;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(kFull, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        unsigned before = x - mine;
        for (int q = 0; q < warp; ++q) before += wsum[q];
        if (before < need && before + mine >= need) {
            for (int q = 0; q < per; ++q) {
                const unsigned c = hist[tid * per + q];
                if (before + c >= need) {
                    found = tid * per + q, found_before = before;
                    break;
                }
                before += c;
            }
        }
        __syncthreads();
        if (tid == 0) {
            SelState t{};
            t.pfx_hi = ph, t.pfx_lo = pl, t.mask_hi = mh, t.mask_lo = ml;
            sel_extend(&t, found < 0 ? 0u : (unsigned)found, pass);
            ph = t.pfx_hi, pl = t.pfx_lo, mh = t.mask_hi, ml = t.mask_lo;
            if (found >= 0) need -= found_before;
            if (found < 0 || hist[found] == need || pass == kPasses - 1) done = 1;
        }
        __syncthreads();
    }
    // the chosen items, in their order
    unsigned base = 0;
    const bool none = k == 0 && !all;
    for (int i0 = 0; i0 < n; i0 += kSmallT) {
        const int i = i0 + tid;
        bool ok = false;
        unsigned long long v = 0ull;
        if (i < n) {
            v = vb[i];
            const unsigned long long hi = (0x7fffffffffffffffull - (v & 0x7fffffffffffffffull)) & mh;
            ok = (v << 1) != 0ull && !none && (all || hi < ph || (hi == ph && (key[i] & ml) <= pl));
        }
        const unsigned bal = __ballot_sync(kFull, ok);
        if (lane == 0) wsum[warp] = __popc(bal);
        __syncthreads();
        unsigned pos = base, tot = 0;
        for (int q = 0; q < kSmallT / 32; ++q) {
            if (q < warp) pos += wsum[q];
            tot += wsum[q];
        }
        pos += __popc(bal & ((1u << lane) - 1u));
        if (ok && (unsigned long long)pos < k) out_key[pos] = key[i], out_val[pos] = __longlong_as_double((long long)v);
        base += tot;
        __syncthreads();
    }
    if (tid == 0) *n_out = base;
}

__global__ void sel_gather_kernel(Items it, const SelState *s, unsigned long long *out_key,
                                  double *out_val, long long cap, unsigned long long *n_out) {
    __shared__ unsigned wt[kT / 32];
    __shared__ unsigned long long base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned long long ph = s->pfx_hi, pl = s->pfx_lo, mh = s->mask_hi, ml = s->mask_lo;
    const bool all = s->all;
    const bool none = (s->need == 0 && !all && mh == 0 && ml == 0);  // k == 0
    for (long long i0 = (long long)blockIdx.x * blockDim.x; i0 < it.n;
         i0 += (long long)gridDim.x * blockDim.x) {
        const long long i = i0 + threadIdx.x;
        bool ok = false;
        unsigned long long key = 0, vb = 0;
        if (i < it.n && !none) {
            key = it.key[(size_t)i * it.stride];
            vb = (unsigned long long)__double_as_longlong(it.val[(size_t)i * it.stride]);
            if (item_valid(key, vb)) {
                if (all) ok = true;
                else {
                    const unsigned long long hi = (0x7fffffffffffffffull - (vb & 0x7fffffffffffffffull)) & mh;
                    const unsigned long long lo = key & ml;
                    ok = (hi < ph) || (hi == ph && lo <= pl);
                }
            }
        }
        const unsigned bal = __ballot_sync(kFull, ok);
        if (lane == 0) wt[warp] = __popc(bal);
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned tot = 0;
            for (int w = 0; w < kT / 32; ++w) {
                unsigned c = wt[w];
                wt[w] = tot;
                tot += c;
            }
            base = tot ? atomicAdd(n_out, (unsigned long long)tot) : 0ull;
        }
        __syncthreads();
        if (ok) {
            const unsigned long long pos = base + wt[warp] + __popc(bal & ((1u << lane) - 1u));
            if ((long long)pos < cap) {
                out_key[pos] = key;
                out_val[pos] = __longlong_as_double((long long)vb);
            }
        }
        __syncthreads();
    }
}

__global__ void sel_stats_kernel(const SelState *s, double *sumsq_out, unsigned long long *total_out) {
    if (threadIdx.x == 0) {
        if (sumsq_out) *sumsq_out = s->sumsq;
        if (total_out) *total_out = s->total;
    }
}

// one pass: items of a smaller first digit than the picked bin -> out; of the
// picked bin -> cand (or out, when the bin is taken whole)
__global__ void sel_split_kernel(Items it, const SelState *s, unsigned long long *out_key,
                                 double *out_val, long long out_cap, unsigned long long *n_out,
                                 unsigned long long *cand_key, double *cand_val, long long cand_cap,
                                 unsigned long long *cand_n) {
    const int lane = threadIdx.x & 31;
    const bool all = s->all, done = s->done;
    const bool none = !all && s->mask_hi == 0;  // k == 0
    const unsigned b0 = (unsigned)(s->pfx_hi >> 51);
    for (long long i0 = (long long)blockIdx.x * blockDim.x; i0 < it.n;
         i0 += (long long)gridDim.x * blockDim.x) {
        const long long i = i0 + threadIdx.x;
        int dest = 0;  // 0 none, 1 out, 2 cand
        unsigned long long key = 0, vb = 0;
        if (i < it.n && !none) {
            key = it.key[(size_t)i * it.stride];
            vb = (unsigned long long)__double_as_longlong(it.val[(size_t)i * it.stride]);
            if (item_valid(key, vb)) {
                const unsigned d0 = (unsigned)((0x7fffffffffffffffull - (vb & 0x7fffffffffffffffull)) >> 51);
                if (all || d0 < b0 || (done && d0 == b0)) dest = 1;
                else if (d0 == b0) dest = 2;
            }
        }
        const unsigned bo = __ballot_sync(kFull, dest == 1), bc = __ballot_sync(kFull, dest == 2);
        unsigned long long base_o = 0, base_c = 0;
        if (lane == 0) {
            if (bo) base_o = atomicAdd(n_out, (unsigned long long)__popc(bo));
            if (bc) base_c = atomicAdd(cand_n, (unsigned long long)__popc(bc));
        }
        base_o = __shfl_sync(kFull, base_o, 0);
        base_c = __shfl_sync(kFull, base_c, 0);
        const unsigned lt = (1u << lane) - 1u;
        if (dest == 1) {
            const unsigned long long pos = base_o + __popc(bo & lt);
            if ((long long)pos < out_cap) out_key[pos] = key, out_val[pos] = __longlong_as_double((long long)vb);
        } else if (dest == 2) {
            const unsigned long long pos = base_c + __popc(bc & lt);
            if ((long long)pos < cand_cap) cand_key[pos] = key, cand_val[pos] = __longlong_as_double((long long)vb);
        }
    }
}

__global__ void sel_split_result_kernel(const SelState *s, const unsigned long long *n_out,
                                        const unsigned long long *cand_n, SplitResult *r) {
    if (threadIdx.x == 0) {
        r->n_out = *n_out;
        r->n_cand = *cand_n;
        r->need = s->need;
        r->total = s->total;
        r->all = s->all;
        r->done = s->done;
    }
}

int sms() {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

unsigned grid_for(long long n, int per_sm) {
    long long g = (n + kT - 1) / kT;
    long long c = (long long)sms() * per_sm;
    if (g > c) g = c;
    if (g < 1) g = 1;
    return (unsigned)g;
}

// ------------------------------------------------------------- radix sort

constexpr int kSortItems = 8;
constexpr int kTile = kT * kSortItems;  // 2048
constexpr int kRadix = 256;

constexpr int kDigits = 8;

// shared by a sort's kernels: how often each digit value occurs, and one of the keys
// (a digit whose value in that key is every key's needs no pass)
struct SortState {
    unsigned digit[kDigits][kRadix];
    unsigned long long key0;
};

__device__ __forceinline__ bool rs_skip(const SortState *s, unsigned n, int p) {
    return s->digit[p][(s->key0 >> (8 * p)) & 0xff] == n;
}

// which of the two buffers holds the pairs before pass p
__device__ __forceinline__ int rs_buffer(const SortState *s, unsigned n, int p) {
    int c = 0;
    for (int q = 0; q < p; ++q) c ^= !rs_skip(s, n, q);
    return c;
}

__device__ __forceinline__ long long rs_count(const unsigned long long *n_dev, long long cap) {
    const long long n = (long long)*n_dev;
    return n < cap ? n : cap;
}

__global__ void rs_digits_kernel(const unsigned long long *key, long long cap, const unsigned long long *n_dev,
                                 int passes, SortState *s) {
    __shared__ unsigned h[kDigits][kRadix];
    for (int b = threadIdx.x; b < kDigits * kRadix; b += blockDim.x) (&h[0][0])[b] = 0;
    __syncthreads();
    const long long n = rs_count(n_dev, cap);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const unsigned long long k = key[i];
        for (int p = 0; p < passes; ++p) atomicAdd(&h[p][(k >> (8 * p)) & 0xff], 1u);
        if (i == 0) s->key0 = k;
    }
    __syncthreads();
    for (int b = threadIdx.x; b < passes * kRadix; b += blockDim.x)
        if ((&h[0][0])[b]) atomicAdd(&(&s->digit[0][0])[b], (&h[0][0])[b]);
}

// Up to kFusedTiles tiles a pass is one launch: each tile's block adds up the counts of the
// tiles before it, and while it places its pairs it counts, for the tile each one lands in,
// the digit of the next pass that is not skipped.  counts: three buffers of [tile][value],
// taken in turn (read, filled, cleared).  Three launches a pass took 20 us each pass at
// 2e4 to 2e5 pairs, mostly launch gaps; above kFusedTiles the scan over all tiles is shared.
constexpr int kFusedTiles = 256;

__device__ __forceinline__ int rs_next(const SortState *s, unsigned n, int p, int passes) {
    while (++p < passes && rs_skip(s, n, p)) {}
    return p;
}

__device__ __forceinline__ int rs_done(const SortState *s, unsigned n, int p) {  // passes run before p
    int c = 0;
    for (int q = 0; q < p; ++q) c += !rs_skip(s, n, q);
    return c;
}

__global__ void rs_first_kernel(const unsigned long long *key, long long cap, const unsigned long long *n_dev, int passes,
                                const SortState *s, unsigned *counts) {
    __shared__ unsigned h[kRadix];
    const long long n = rs_count(n_dev, cap), t0 = (long long)blockIdx.x * kTile;
    const int p = rs_next(s, (unsigned)n, -1, passes);
    if (p >= passes || t0 >= n) return;
    h[threadIdx.x] = 0;  // kT == kRadix
    __syncthreads();
    for (int q = 0; q < kSortItems; ++q) {
        const long long i = t0 + (long long)q * kT + threadIdx.x;
        if (i < n) atomicAdd(&h[(key[i] >> (8 * p)) & 0xff], 1u);
    }
    __syncthreads();
    counts[(size_t)blockIdx.x * kRadix + threadIdx.x] = h[threadIdx.x];
}

// the pairs of a tile (kSortItems rounds of each warp's 32): their places among the pairs of
// their digit value in the tile; wc[warp][value]: the warp's count
__device__ __forceinline__ void rs_rank(const unsigned long long *key, long long w0, long long n, int shift, int warp,
                                        int lane, unsigned (*wc)[kRadix], unsigned *loc) {
#pragma unroll
    for (int q = 0; q < kSortItems; ++q) {
        const bool valid = w0 + (long long)q * 32 + lane < n;
        const unsigned d = valid ? (unsigned)((key[q] >> shift) & 0xff) : (0x1000u | lane);
        const unsigned peers = __match_any_sync(kFull, d);
        const unsigned before = __popc(peers & ((1u << lane) - 1u));
        const unsigned base = valid ? wc[warp][d] : 0u;
        __syncwarp();
        if (valid && (peers >> lane) == 1u) wc[warp][d] = base + __popc(peers);  // highest peer
        __syncwarp();
        loc[q] = base + before;
    }
}

__global__ void rs_pass_kernel(unsigned long long *ka, double *va, unsigned long long *kb, double *vb, long long cap,
                               const unsigned long long *n_dev, int p, int passes, const SortState *s, unsigned *counts,
                               size_t stride) {
    __shared__ unsigned wc[kT / 32][kRadix], wsum[kT / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, shift = 8 * p;
    const long long n = rs_count(n_dev, cap), t0 = (long long)blockIdx.x * kTile;
    if (t0 >= n || rs_skip(s, (unsigned)n, p)) return;
    const int done = rs_done(s, (unsigned)n, p), next = rs_next(s, (unsigned)n, p, passes);
    const unsigned *now = counts + (size_t)(done % 3) * stride;
    unsigned *then = counts + (size_t)((done + 1) % 3) * stride;
    counts[(size_t)((done + 2) % 3) * stride + (size_t)blockIdx.x * kRadix + tid] = 0u;
    const unsigned long long *kin = done & 1 ? kb : ka;
    const double *vin = done & 1 ? vb : va;
    unsigned long long *kout = done & 1 ? ka : kb;
    double *vout = done & 1 ? va : vb;
    const long long w0 = t0 + (long long)warp * (32 * kSortItems);
    unsigned long long key[kSortItems];
    double val[kSortItems];
#pragma unroll
    for (int q = 0; q < kSortItems; ++q) {
        const long long i = w0 + (long long)q * 32 + lane;
        key[q] = 0ull, val[q] = 0.0;
        if (i < n) key[q] = kin[i], val[q] = vin[i];
    }
    // where this tile's pairs of digit value tid begin
    unsigned before = 0, total = s->digit[p][tid], x = total;
    for (unsigned t = 0; t < blockIdx.x; ++t) before += now[(size_t)t * kRadix + tid];
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    for (int b = tid; b < (kT / 32) * kRadix; b += kT) (&wc[0][0])[b] = 0;
    __syncthreads();
    before += x - total;
    for (int w = 0; w < warp; ++w) before += wsum[w];
    unsigned loc[kSortItems];
    rs_rank(key, w0, n, shift, warp, lane, wc, loc);
    __syncthreads();
    for (int w = 0; w < kT / 32; ++w) {
        const unsigned c = wc[w][tid];
        wc[w][tid] = before;
        before += c;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kSortItems; ++q) {
        const long long i = w0 + (long long)q * 32 + lane;
        if (i < n) {
            const unsigned pos = wc[warp][(key[q] >> shift) & 0xff] + loc[q];
            kout[pos] = key[q];
            vout[pos] = val[q];
            if (next < passes) atomicAdd(&then[(size_t)(pos / kTile) * kRadix + ((key[q] >> (8 * next)) & 0xff)], 1u);
        }
    }
}

// per tile and digit value: the keys that have it; counts[value * tiles + tile]
__global__ void rs_hist_kernel(const unsigned long long *ka, const unsigned long long *kb, long long cap,
                               const unsigned long long *n_dev, int p, const SortState *s, unsigned *counts) {
    __shared__ unsigned h[kRadix];
    const long long n = rs_count(n_dev, cap);
    if (rs_skip(s, (unsigned)n, p)) return;
    const unsigned long long *key = rs_buffer(s, (unsigned)n, p) ? kb : ka;
    const int tiles = (int)((n + kTile - 1) / kTile);
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        h[threadIdx.x] = 0;  // kT == kRadix
        __syncthreads();
        const long long t0 = (long long)t * kTile;
        for (int q = 0; q < kSortItems; ++q) {
            const long long i = t0 + (long long)q * kT + threadIdx.x;
            if (i < n) atomicAdd(&h[(key[i] >> (8 * p)) & 0xff], 1u);
        }
        __syncthreads();
        counts[(size_t)threadIdx.x * tiles + t] = h[threadIdx.x];
        __syncthreads();
    }
}

// block v: exclusive scan over the tiles of digit value v, from the keys of smaller values on
__global__ void rs_scan_kernel(unsigned *counts, long long cap, const unsigned long long *n_dev, int p,
                               const SortState *s) {
    __shared__ unsigned wsum[32];
    const long long n = rs_count(n_dev, cap);
    if (rs_skip(s, (unsigned)n, p)) return;
    const int tiles = (int)((n + kTile - 1) / kTile), lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    unsigned *c = counts + (size_t)blockIdx.x * tiles;
    unsigned carry = 0;
    {
        unsigned v = threadIdx.x < blockIdx.x ? s->digit[p][threadIdx.x] : 0u;  // (kRadix <= threads)
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        if (lane == 0) wsum[warp] = v;
        __syncthreads();
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) carry += wsum[w];
        __syncthreads();
    }
    for (int b0 = 0; b0 < tiles; b0 += blockDim.x) {
        const int i = b0 + threadIdx.x;
        const unsigned v = i < tiles ? c[i] : 0u;
        unsigned x = v;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(kFull, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        unsigned before = carry, tot = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            if (w < warp) before += wsum[w];
            tot += wsum[w];
        }
        if (i < tiles) c[i] = before + x - v;
        carry += tot;
        __syncthreads();
    }
}

// A tile's pairs are put in order in shared memory first and leave in runs of one digit
// value: written from where they lay, each was a sector write of its own (540 us a pass for
// 2.2e7 pairs).
__global__ void rs_scatter_kernel(unsigned long long *ka, double *va, unsigned long long *kb, double *vb,
                                  long long cap, const unsigned long long *n_dev, int p, const SortState *s,
                                  const unsigned *offsets) {
    __shared__ unsigned wc[kT / 32][kRadix], to[kRadix], wsum[kT / 32];
    __shared__ unsigned long long sk[kTile];
    __shared__ double sv[kTile];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, shift = 8 * p;
    const long long n = rs_count(n_dev, cap);
    if (rs_skip(s, (unsigned)n, p)) return;
    const bool from_b = rs_buffer(s, (unsigned)n, p) != 0;
    const unsigned long long *kin = from_b ? kb : ka;
    const double *vin = from_b ? vb : va;
    unsigned long long *kout = from_b ? ka : kb;
    double *vout = from_b ? va : vb;
    const int tiles = (int)((n + kTile - 1) / kTile);
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        for (int b = tid; b < (kT / 32) * kRadix; b += kT) (&wc[0][0])[b] = 0;
        __syncthreads();
        const long long t0 = (long long)t * kTile, w0 = t0 + (long long)warp * (32 * kSortItems);
        unsigned loc[kSortItems];
        unsigned long long key[kSortItems];
        double val[kSortItems];
#pragma unroll
        for (int q = 0; q < kSortItems; ++q) {
            const long long i = w0 + (long long)q * 32 + lane;
            key[q] = 0ull, val[q] = 0.0;
            if (i < n) key[q] = kin[i], val[q] = vin[i];
        }
        const unsigned off = offsets[(size_t)tid * tiles + t];  // kT == kRadix
        rs_rank(key, w0, n, shift, warp, lane, wc, loc);
        __syncthreads();
        unsigned total = 0;
        for (int w = 0; w < kT / 32; ++w) total += wc[w][tid];
        unsigned x = total;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(kFull, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) wsum[warp] = x;
        __syncthreads();
        unsigned run = x - total;  // the value's first place in the tile
        for (int w = 0; w < warp; ++w) run += wsum[w];
        to[tid] = off - run;
        for (int w = 0; w < kT / 32; ++w) {
            const unsigned c = wc[w][tid];
            wc[w][tid] = run;
            run += c;
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kSortItems; ++q)
            if (w0 + (long long)q * 32 + lane < n) {
                const unsigned at = wc[warp][(key[q] >> shift) & 0xff] + loc[q];
                sk[at] = key[q], sv[at] = val[q];
            }
        __syncthreads();
        const int m = (int)(n - t0 < kTile ? n - t0 : kTile);
#pragma unroll
        for (int q = 0; q < kSortItems; ++q) {
            const int i = q * kT + tid;
            if (i < m) {
                const unsigned long long k = sk[i];
                const unsigned pos = to[(k >> shift) & 0xff] + i;
                kout[pos] = k;
                vout[pos] = sv[i];
            }
        }
        __syncthreads();
    }
}

// The sum over the partial sums in their order (thread 0's value; every thread of the block
// calls it): fetched together, then added.  Only the blocks that had entries are added (the
// others' sums are zero): all 304 take 12 us of float64 latency, 2e4 entries make 79.  (A tree
// is faster yet, but moves the last bit of the norm, and with it the sign that the cycle end's
// eigenvector comes out with.)
__device__ __forceinline__ double ordered_sum(const double *partial, int np, double *sh) {
    for (int k = threadIdx.x; k < np; k += blockDim.x) sh[k] = partial[k];
    __syncthreads();
    double s = 0.0;
    if (threadIdx.x == 0)
        for (int k = 0; k < np; ++k) s += sh[k];
    return s;
}

// Up to kSmall pairs sorted by one CTA in shared memory; digits that all keys share are
// skipped.  (Dividing by the norm here too was slower than its two launches: one SM's
// float64 units take 25 us for 4900 entries.)
__global__ void __launch_bounds__(kSmallT)
small_sort_kernel(unsigned long long *key, double *val, long long cap, const unsigned long long *n_dev, int bits) {
    extern __shared__ __align__(16) unsigned char sm[];
    unsigned long long *sk = reinterpret_cast<unsigned long long *>(sm);
    double *sv = reinterpret_cast<double *>(sk + kSmall);
    unsigned *wc = reinterpret_cast<unsigned *>(sv + kSmall);  // [warps][kRadix]
    __shared__ unsigned dsum[kRadix / 32];
    __shared__ unsigned differ[2];  // bits in which some key differs from the first
    constexpr int W = kSmallT / 32, kItems = kSmall / kSmallT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = (int)rs_count(n_dev, cap), per = (n + kSmallT - 1) / kSmallT;  // rounds of 32 per warp
    unsigned long long k[kItems];
    double v[kItems];
    const int w0 = warp * 32 * per + lane;
    const unsigned long long key0 = n > 0 ? key[0] : 0ull;
    unsigned long long diff = 0ull;
    if (tid < 2) differ[tid] = 0u;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kItems; ++q) {
        const int i = w0 + q * 32;
        k[q] = 0ull, v[q] = 0.0;
        if (q < per && i < n) k[q] = key[i], v[q] = val[i], diff |= k[q] ^ key0;
    }
    {
        const unsigned lo = __reduce_or_sync(kFull, (unsigned)diff), hi = __reduce_or_sync(kFull, (unsigned)(diff >> 32));
        if (lane == 0) atomicOr(&differ[0], lo), atomicOr(&differ[1], hi);
    }
    __syncthreads();
    diff = differ[0] | (unsigned long long)differ[1] << 32;
    for (int shift = 0; shift < bits; shift += 8) {
        if (((diff >> shift) & 0xffull) == 0ull) continue;
        for (int b = tid; b < W * kRadix; b += kSmallT) wc[b] = 0u;
        __syncthreads();
        unsigned loc[kItems];
#pragma unroll
        for (int q = 0; q < kItems; ++q) {
            loc[q] = 0u;
            if (q >= per) continue;
            const bool valid = w0 + q * 32 < n;
            const unsigned d = valid ? (unsigned)((k[q] >> shift) & 0xff) : (0x1000u | lane);
            const unsigned peers = __match_any_sync(kFull, d);
            const unsigned base = valid ? wc[warp * kRadix + d] : 0u;
            __syncwarp();
            if (valid && (peers >> lane) == 1u) wc[warp * kRadix + d] = base + __popc(peers);  // highest peer
            __syncwarp();
            loc[q] = base + __popc(peers & ((1u << lane) - 1u));
        }
        __syncthreads();
        unsigned tot = 0, x = 0;
        if (tid < kRadix) {
            for (int w = 0; w < W; ++w) tot += wc[w * kRadix + tid];
            x = tot;
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(kFull, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) dsum[warp] = x;
        }
        __syncthreads();
        if (tid < kRadix) {
            unsigned run = x - tot;
            for (int w = 0; w < warp; ++w) run += dsum[w];
            for (int w = 0; w < W; ++w) {
                const unsigned c = wc[w * kRadix + tid];
                wc[w * kRadix + tid] = run;
                run += c;
            }
        }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kItems; ++q)
            if (q < per && w0 + q * 32 < n) {
                const unsigned pos = wc[warp * kRadix + ((k[q] >> shift) & 0xff)] + loc[q];
                sk[pos] = k[q], sv[pos] = v[q];
            }
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kItems; ++q)
            if (q < per && w0 + q * 32 < n) k[q] = sk[w0 + q * 32], v[q] = sv[w0 + q * 32];
    }
#pragma unroll
    for (int q = 0; q < kItems; ++q)
        if (q < per && w0 + q * 32 < n) key[w0 + q * 32] = k[q], val[w0 + q * 32] = v[q];
}

// back into the caller's arrays when an odd number of passes ran
__global__ void copy_pairs_kernel(const unsigned long long *ks, const double *vs, unsigned long long *kd, double *vd,
                                  long long cap, const unsigned long long *n_dev, int passes, const SortState *s) {
    const long long n = rs_count(n_dev, cap);
    if (!rs_buffer(s, (unsigned)n, passes)) return;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        kd[i] = ks[i];
        vd[i] = vs[i];
    }
}

// ------------------------------------------------------------- normalisation

__global__ void sumsq_kernel(const double *v, long long cap, const unsigned long long *n_dev,
                             double *partial) {
    __shared__ double sh[kT / 32];
    long long n = (long long)*n_dev;
    if (n > cap) n = cap;
    double a = 0.0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        a = __fma_rn(v[i], v[i], a);
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(kFull, a, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        double r = 0.0;
        for (int w = 0; w < kT / 32; ++w) r += sh[w];
        partial[blockIdx.x] = r;
    }
}

__global__ void scale_kernel(double *v, long long cap, const unsigned long long *n_dev,
                             const double *partial, int nparts) {
    __shared__ double norm, sh[kRedBlocks];
    long long n = (long long)*n_dev;
    if (n > cap) n = cap;
    const long long used = (n + kT - 1) / kT;
    const double s = ordered_sum(partial, (int)(used < nparts ? used : nparts), sh);
    if (threadIdx.x == 0) norm = sqrt(s);
    __syncthreads();
    const double d = norm;
    if (!(d > 0.0)) return;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (long long)gridDim.x * blockDim.x)
        v[i] = __ddiv_rn(v[i], d);
}

}  // namespace

size_t select_workspace_bytes(long long, long long) { return sel_layout().bytes; }

cudaError_t select_topk(Items it, long long k, unsigned long long *out_key, double *out_val,
                        unsigned long long *n_out_dev, double *sumsq_dev,
                        unsigned long long *total_dev, void *ws, size_t ws_bytes, cudaStream_t st) {
    const SelLayout L = sel_layout();
    if (ws_bytes < L.bytes) return cudaErrorInvalidValue;
    if (it.n <= kSmall) {
        const size_t smem = size_t(kSmall) * 16 + kBins * 4;
        cudaError_t e = allow_max_smem(sel_small_kernel, smem);
        if (e != cudaSuccess) return e;
        count_launch();
        sel_small_kernel<<<1, kSmallT, smem, st>>>(it, (unsigned long long)(k < 0 ? 0 : k), out_key, out_val, n_out_dev,
                                                   sumsq_dev, total_dev);
        return cudaGetLastError();
    }
    char *base = static_cast<char *>(ws);
    SelState *s = reinterpret_cast<SelState *>(base + L.state);
    unsigned long long *hist = reinterpret_cast<unsigned long long *>(base + L.hist);
    count_launch();
    sel_init_kernel<<<1, kT, 0, st>>>(s, (unsigned long long)(k < 0 ? 0 : k), hist, n_out_dev);
    const unsigned g = grid_for(it.n, 4);
    for (int p = 0; p < kPasses; ++p) {
        count_launch();
        sel_hist_kernel<<<g, kT, 0, st>>>(it, s, hist, p, sumsq_dev != nullptr);
    }
    count_launch();
    sel_gather_kernel<<<grid_for(it.n, 8), kT, 0, st>>>(it, s, out_key, out_val, k, n_out_dev);
    if (sumsq_dev || total_dev) {
        count_launch();
        sel_stats_kernel<<<1, 32, 0, st>>>(s, sumsq_dev, total_dev);
    }
    return cudaGetLastError();
}

cudaError_t select_split(Items it, long long k,
                         unsigned long long *out_key, double *out_val, unsigned long long *n_out_dev,
                         unsigned long long *cand_key, double *cand_val, long long cand_cap,
                         unsigned long long *cand_n, void *ws, size_t ws_bytes, SplitResult *res_host,
                         cudaStream_t st) {
    const SelLayout L = sel_layout();
    if (ws_bytes < L.bytes) return cudaErrorInvalidValue;
    char *base = static_cast<char *>(ws);
    SelState *s = reinterpret_cast<SelState *>(base + L.state);
    unsigned long long *hist = reinterpret_cast<unsigned long long *>(base + L.hist);
    SplitResult *r = reinterpret_cast<SplitResult *>(base + L.result);
    count_launch();
    sel_init_kernel<<<1, kT, 0, st>>>(s, (unsigned long long)(k < 0 ? 0 : k), hist, n_out_dev);
    cudaError_t e = cudaMemsetAsync(cand_n, 0, 8, st);
    if (e != cudaSuccess) return e;
    count_launch();
    sel_hist_kernel<<<grid_for(it.n, 4), kT, 0, st>>>(it, s, hist, 0, 0);
    count_launch();
    sel_split_kernel<<<grid_for(it.n, 8), kT, 0, st>>>(it, s, out_key, out_val, k, n_out_dev,
                                                       cand_key, cand_val, cand_cap, cand_n);
    count_launch();
    sel_split_result_kernel<<<1, 32, 0, st>>>(s, n_out_dev, cand_n, r);
    e = cudaMemcpyAsync(res_host, r, sizeof(SplitResult), cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return e;
    return cudaStreamSynchronize(st);
}

namespace {
// Counters of up to ntiles tiles: three buffers for a pass of up to kFusedTiles tiles in one
// launch, one beyond.  Never less for more tiles: a caller may sort fewer pairs than its
// workspace was sized for, and 257 tiles alone need a third of what 256 do.
size_t sort_counts_bytes(long long ntiles) {
    const long long fused = std::min<long long>(std::max<long long>(ntiles, 1), kFusedTiles);
    return a256(size_t(std::max(3 * fused, ntiles)) * kRadix * 4);
}
}  // namespace

// (grows with cap: sfci_sigma sizes it for out_cap and sorts the entries it found)
size_t sort_pairs_bytes(long long cap) {
    const long long ntiles = (cap + kTile - 1) / kTile;
    return a256(size_t(cap) * 8) * 2 + sort_counts_bytes(ntiles) + a256(sizeof(SortState));
}

namespace {
cudaError_t small_sort(unsigned long long *key, double *val, long long cap, const unsigned long long *n_dev, int bits,
                       cudaStream_t st) {
    const size_t smem = size_t(kSmall) * 16 + size_t(kSmallT / 32) * kRadix * 4;
    cudaError_t e = allow_max_smem(small_sort_kernel, smem);
    if (e != cudaSuccess) return e;
    count_launch();
    small_sort_kernel<<<1, kSmallT, smem, st>>>(key, val, cap, n_dev, bits);
    return cudaGetLastError();
}
}  // namespace

cudaError_t sort_pairs(unsigned long long *key, double *val, long long cap,
                       const unsigned long long *n_dev, int bits, void *ws, cudaStream_t st) {
    if (cap <= 0) return cudaSuccess;
    if (cap <= kSmall) return small_sort(key, val, cap, n_dev, bits, st);
    const long long ntiles = (cap + kTile - 1) / kTile;
    char *b = static_cast<char *>(ws);
    unsigned long long *k2 = reinterpret_cast<unsigned long long *>(b);
    double *v2 = reinterpret_cast<double *>(b + a256(size_t(cap) * 8));
    unsigned *counts = reinterpret_cast<unsigned *>(b + 2 * a256(size_t(cap) * 8));
    SortState *s = reinterpret_cast<SortState *>(b + 2 * a256(size_t(cap) * 8) + sort_counts_bytes(ntiles));
    const int passes = (bits + 7) / 8;
    cudaError_t e = cudaMemsetAsync(s, 0, sizeof(SortState), st);
    if (e != cudaSuccess) return e;
    count_launch();
    rs_digits_kernel<<<grid_for(cap, 4), kT, 0, st>>>(key, cap, n_dev, passes, s);
    if (ntiles <= kFusedTiles) {
        const size_t stride = size_t(ntiles) * kRadix;
        e = cudaMemsetAsync(counts, 0, stride * 12, st);
        if (e != cudaSuccess) return e;
        count_launch();
        rs_first_kernel<<<(unsigned)ntiles, kT, 0, st>>>(key, cap, n_dev, passes, s, counts);
        for (int p = 0; p < passes; ++p) {
            count_launch();
            rs_pass_kernel<<<(unsigned)ntiles, kT, 0, st>>>(key, val, k2, v2, cap, n_dev, p, passes, s, counts, stride);
        }
        count_launch();
        copy_pairs_kernel<<<grid_for(cap, 8), kT, 0, st>>>(k2, v2, key, val, cap, n_dev, passes, s);
        return cudaGetLastError();
    }
    const unsigned g = (unsigned)(ntiles < (long long)sms() * 8 ? ntiles : (long long)sms() * 8);
    for (int p = 0; p < passes; ++p) {
        count_launch();
        rs_hist_kernel<<<g, kT, 0, st>>>(key, k2, cap, n_dev, p, s, counts);
        count_launch();
        rs_scan_kernel<<<kRadix, ntiles > 2048 ? 1024 : 256, 0, st>>>(counts, cap, n_dev, p, s);
        count_launch();
        rs_scatter_kernel<<<g, kT, 0, st>>>(key, val, k2, v2, cap, n_dev, p, s, counts);
    }
    count_launch();
    copy_pairs_kernel<<<grid_for(cap, 8), kT, 0, st>>>(k2, v2, key, val, cap, n_dev, passes, s);
    return cudaGetLastError();
}

cudaError_t sort_normalize(unsigned long long *key, double *val, long long cap, const unsigned long long *n_dev,
                           int bits, void *sort_ws, void *norm_ws, cudaStream_t st) {
    const cudaError_t e = sort_pairs(key, val, cap, n_dev, bits, sort_ws, st);
    return e == cudaSuccess ? normalize_vec(val, cap, n_dev, norm_ws, st) : e;
}

size_t normalize_ws_bytes(long long) { return a256(sizeof(double) * kRedBlocks); }

cudaError_t normalize_vec(double *val, long long cap, const unsigned long long *n_dev, void *ws,
                          cudaStream_t st) {
    double *partial = static_cast<double *>(ws);
    count_launch();
    sumsq_kernel<<<kRedBlocks, kT, 0, st>>>(val, cap, n_dev, partial);
    count_launch();
    scale_kernel<<<kRedBlocks, kT, 0, st>>>(val, cap, n_dev, partial, kRedBlocks);
    return cudaGetLastError();
}

}  // namespace sfci
