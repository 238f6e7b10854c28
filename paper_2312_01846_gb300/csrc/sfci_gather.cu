// sigma = H psi by target rows, without intermediate records: every target
// alpha string ("row", the paper's bucket on the spin-up string, Sec. 3)
// gathers its elements from the sources that reach it and sums them in a
// shared-memory table at once.
//
// The bucketed path (sfci_emit.cu, sfci_merge.cu) writes each intermediate
// element as a 16-byte record and reads it back: at N_d = 1e5 on 28 orbitals it
// spends 43 ms appending (reservations, row map, scattered stores) and 42 ms
// merging, neither near the memory rate.  Here nearly all elements (the
// opposite-spin and beta-beta doubles) go straight from their integral into
// their sum.  What makes that possible:
//
//  * The single and double excitations of each distinct beta string are
//    tabulated once (t1, t2): every row that a source reaches reads the same
//    table.  A row is then a list of its sources one alpha hop away (ab: beta
//    string, integral row, c_D), the sources it holds itself, and a short list
//    of ready elements (rec: alpha-alpha doubles, singles, diagonal; 15 % of
//    the elements at 28 orbitals).  All three lie in row order, so a group of
//    rows is one contiguous range of each and a CTA's warps share it evenly.
//  * Alpha strings that differ by one or two hops share an (n_alpha - 1)- or
//    (n_alpha - 2)-electron substring K, and a double shares exactly one.  The
//    sources' alpha strings are listed under their substrings (ent1, ent2), so
//    a row finds the strings that reach it by reading the lists of its own
//    n_alpha + C(n_alpha, 2) substrings: about one list entry per element
//    instead of C(n_alpha,2) C(n-n_alpha,2) candidates.  The sign of a
//    double is s_K(i,j) s_K(a,b) with s_K the parity of K's electrons below the
//    two orbitals, and its integral W[ab][ij] = (ai|bj) - (aj|bi) sits in a
//    row of a small table.
//  * A row's sums are keyed by pi(beta'), a bijection on ceil(log2 C(n, n_beta))
//    bits: 32-bit keys (native shared-memory compare-and-swap), no hashing per
//    element.  A row with more distinct entries than the table is processed
//    in classes, ranges of pi; the tables are ordered by the top bits of pi,
//    so a class reads its own segments.  A class that still outgrows the
//    table splits in two and runs again (its results have not left the CTA).
//    Light rows share a table, the row's number in the key's upper bits.
//
// Elements, their products with c_D and the exact 128-bit sums are those of the
// bucketed path bit for bit; the sums do not depend on the order of the adds.
#include <algorithm>
#include <cmath>

#include "sfci_stream.cuh"

namespace sfci {
namespace {

constexpr int kGT = 512;          // gather CTA threads
constexpr int kGW = kGT / 32;
constexpr int kGLog = 12;         // log2 table slots: 4096 x 20 B, two CTAs per SM
constexpr int kGSlots = 1 << kGLog;
constexpr unsigned kNoKey = 0xffffffffu;
constexpr int kMaxE = kGatherMaxElectrons;
constexpr int kLT = 256;          // list CTA threads
constexpr unsigned kMaxParts = 512;
constexpr int kMaxClassLog = 11;  // log2 of the most classes a row is planned in
constexpr unsigned long long kSeenEnough = 1000;  // entries from which a weight's statistics count

// ------------------------------------------------------------- helpers

__device__ __forceinline__ unsigned bperm(const GatherShape &p, unsigned x) {
    x ^= x >> p.bs;
    x = (x * p.m1) & p.bmask;
    x ^= x >> p.bs;
    x = (x * p.m2) & p.bmask;
    return x ^ (x >> p.bs);
}

__device__ __forceinline__ unsigned bperm_inv(const GatherShape &p, unsigned x) {
    x ^= x >> p.bs;
    x = (x * p.i2) & p.bmask;
    x ^= x >> p.bs;
    x = (x * p.i1) & p.bmask;
    return x ^ (x >> p.bs);
}

__device__ __forceinline__ double flip_d(double x, unsigned s) {
    return __longlong_as_double(__double_as_longlong(x) ^ ((long long)s << 63));
}

// inverse of Eq. 12, one thread: orbital c is occupied when C(c, i) <= r with i electrons
// left (the lanes of a warp walk the orbitals together)
__device__ unsigned long long unrank_one(unsigned long long r, int n, int m, const unsigned long long *bt, int ks) {
    unsigned long long s = 0;
    int i = m;
    for (int c = n - 1; c >= 0; --c) {
        const unsigned long long x = bt[c * ks + i];
        if (i && x <= r) r -= x, s |= 1ull << c, --i;
    }
    return s;
}

// the next string of the same electron count (Eq. 12's index plus one): Gosper's step
__device__ __forceinline__ unsigned long long next_string(unsigned long long x) {
    if (!x) return x;
    const int t = __ffsll((long long)x) - 1;
    const unsigned long long r = x + (1ull << t);
    return r | (t >= 62 ? 0ull : (r ^ x) >> (t + 2));
}

// single element of the hop i -> a of the spin whose string is `same`, with the
// source's strings: the term order of the emit kernel (h, Coulomb over alpha
// then beta, exchange), each sum rounded on its own
__device__ __noinline__ double single_of(const SysDev &d, int i, int a, unsigned long long alpha,
                                         unsigned long long beta, unsigned long long same) {
    const int n = d.n;
    const size_t at = size_t(a * n + i) * 2 * n;
    if (d.gf) {
        const float *gai = d.sgf + at;
        float v = __ldg(&d.hf[a * n + i]);
        for (unsigned long long s = alpha; s; s &= s - 1ull) v = __fadd_rn(v, __ldg(&gai[__ffsll((long long)s) - 1]));
        for (unsigned long long s = beta; s; s &= s - 1ull) v = __fadd_rn(v, __ldg(&gai[__ffsll((long long)s) - 1]));
        for (unsigned long long s = same; s; s &= s - 1ull) v = __fsub_rn(v, __ldg(&gai[n + __ffsll((long long)s) - 1]));
        return (double)v;
    }
    const double *gai = d.sg + at;
    double v = __ldg(&d.h[a * n + i]);
    for (unsigned long long s = alpha; s; s &= s - 1ull) v = __dadd_rn(v, __ldg(&gai[__ffsll((long long)s) - 1]));
    for (unsigned long long s = beta; s; s &= s - 1ull) v = __dadd_rn(v, __ldg(&gai[__ffsll((long long)s) - 1]));
    for (unsigned long long s = same; s; s &= s - 1ull) v = __dsub_rn(v, __ldg(&gai[n + __ffsll((long long)s) - 1]));
    return v;
}

// <D|H|D>, the emit kernel's term order
// (J + p stride: (pp|kk) over k, then (pk|kp); hd: the diagonal of h, hstride apart)
__device__ double diagonal_of(const SysDev &d, const double *J, int stride, const double *hd, int hstride,
                              unsigned long long alpha, unsigned long long beta) {
    const int n = d.n;
    double one = 0.0, coul = 0.0, exch = 0.0;
    unsigned long long str[2] = {alpha, beta};
    for (int s = 0; s < 2; ++s)
        for (unsigned long long x = str[s]; x; x &= x - 1ull)
            one = __dadd_rn(one, hd[(__ffsll((long long)x) - 1) * hstride]);
    for (int s = 0; s < 2; ++s)
        for (unsigned long long x = str[s]; x; x &= x - 1ull) {
            const int p = __ffsll((long long)x) - 1;
            const double *gpp = J + size_t(p) * stride;
            for (int t = 0; t < 2; ++t)
                for (unsigned long long y = str[t]; y; y &= y - 1ull)
                    coul = __dadd_rn(coul, gpp[__ffsll((long long)y) - 1]);
        }
    for (int s = 0; s < 2; ++s)
        for (unsigned long long x = str[s]; x; x &= x - 1ull) {
            const int p = __ffsll((long long)x) - 1;
            const double *gpq = J + size_t(p) * stride + n;
            for (unsigned long long y = str[s]; y; y &= y - 1ull)
                exch = __dadd_rn(exch, gpq[__ffsll((long long)y) - 1]);
        }
    return __dsub_rn(__dadd_rn(__dadd_rn(d.e_core, one), __dmul_rn(0.5, coul)), __dmul_rn(0.5, exch));
}

// ------------------------------------------------------------- preparation

__device__ __forceinline__ void load_binom(const SysDev &d, unsigned long long *bt) {
    for (int i = threadIdx.x; i < (d.n + 1) * d.ks; i += blockDim.x) bt[i] = d.binom[i];
    __syncthreads();
}

// W[ab][ij] = (ai|bj) - (aj|bi) over orbital pairs a < b, i < j (index b(b-1)/2 + a),
// 0 for pairs that share an orbital (no double: a list entry that is none drops out)
__global__ void pair_integrals_kernel(const SysDev d, int np, double *W) {
    const long long m = (long long)np * np;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < m; t += (long long)gridDim.x * blockDim.x) {
        const int p = (int)(t / np), q = (int)(t - (long long)p * np);
        int b = 1, j = 1;
        while ((b + 1) * b / 2 <= p) ++b;
        while ((j + 1) * j / 2 <= q) ++j;
        const int a = p - b * (b - 1) / 2, i = q - j * (j - 1) / 2, n = d.n;
        const size_t x1 = (size_t(a * n + i) * n + b) * n + j, x2 = (size_t(a * n + j) * n + b) * n + i;
        W[t] = a == i || a == j || b == i || b == j ? 0.0
               : d.gf ? (double)__fsub_rn(d.gf[x1], d.gf[x2]) : __dsub_rn(d.g[x1], d.g[x2]);
    }
}

__global__ void hop_integrals_kernel(const SysDev d, double *sg, float *sgf) {
    const int n = d.n;
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n * n * n; t += gridDim.x * blockDim.x) {
        const int ai = t / n, k = t - ai * n, a = ai / n, i = ai - a * n;
        const size_t x = size_t(ai) * n * n + size_t(k) * (n + 1), y = (size_t(a * n + k) * n + k) * n + i;
        const size_t o = size_t(ai) * 2 * n + k;
        sg[o] = d.g[x], sg[o + n] = d.g[y];
        if (sgf) sgf[o] = d.gf[x], sgf[o + n] = d.gf[y];
    }
}

// rp[r] = first entry of the (ascending) vector at or after row r, rp[ca] = n
__global__ void row_pointers_kernel(const unsigned long long *rank, long long n, unsigned long long ca,
                                    unsigned long long cb, unsigned *rp) {
    for (unsigned long long r = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; r <= ca;
         r += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long key = r * cb;
        long long lo = 0, hi = n;
        while (lo < hi) {
            const long long m = (lo + hi) >> 1;
            if (rank[m] < key) lo = m + 1;
            else hi = m;
        }
        rp[r] = (unsigned)lo;
    }
}

// (row << bb | pi(beta), c) of each source; beta strings seen; *runs = rows with sources
__global__ void sources_kernel(const GatherShape p, const unsigned long long *rank, const double *coef, long long n,
                               unsigned long long cb, unsigned long long *skey, double *sc, unsigned *bflag,
                               unsigned long long *runs, unsigned long long *seen) {
    unsigned c = 0;
    if (blockIdx.x == 0)  // what earlier sigmas saw counts an eighth
        for (int i = threadIdx.x; i < 2 * kSeenBins; i += blockDim.x) seen[i] >>= 3;
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n; s += (long long)gridDim.x * blockDim.x) {
        const unsigned long long r = rank[s], ha = r / cb;
        const unsigned hb = (unsigned)(r - ha * cb);
        skey[s] = (ha << p.bb) | bperm(p, hb);
        sc[s] = coef[s];
        bflag[hb] = 1u;
        c += s == 0 || rank[s - 1] / cb != ha;
    }
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(kFull, c, o);
    if ((threadIdx.x & 31) == 0 && c) atomicAdd(runs, (unsigned long long)c);
}

// per source (in run order): pi(beta), number of its beta string, <D|H|D>.  The diagonal is a
// chain of some hundred adds: its integrals are staged in shared memory (up to kStageN
// orbitals), since the first thread to need one waits for L2 (45 us for 2e4 sources).
constexpr int kStageN = 48;
__global__ void source_fields_kernel(const SysDev d, const GatherShape p, const unsigned long long *skey, long long n,
                                     const unsigned long long *bid, unsigned *spi, unsigned *sb, double *diag,
                                     unsigned long long *bstr) {
    extern __shared__ unsigned long long bt[];
    const int no = d.n;
    const double *J = d.sg, *hd = d.h;
    int stride = (no + 1) * 2 * no, hstride = no + 1;
    if (no <= kStageN) {
        double *sj = reinterpret_cast<double *>(bt + (no + 1) * d.ks), *sh = sj + 2 * no * no;
        for (int i = threadIdx.x; i < 2 * no * no; i += blockDim.x) sj[i] = __ldg(&d.sg[size_t(i / (2 * no)) * stride + i % (2 * no)]);
        for (int i = threadIdx.x; i < no; i += blockDim.x) sh[i] = __ldg(&d.h[i * hstride]);
        J = sj, hd = sh, stride = 2 * no, hstride = 1;
    }
    load_binom(d, bt);
    for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < n; s += (long long)gridDim.x * blockDim.x) {
        const unsigned long long k = skey[s];
        const unsigned pi = (unsigned)k & p.bmask, hb = bperm_inv(p, pi), id = (unsigned)bid[hb];
        const unsigned long long alpha = unrank_one(k >> p.bb, d.n, d.na, bt, d.ks);
        const unsigned long long beta = unrank_one(hb, d.n, d.nb, bt, d.ks);
        spi[s] = pi;
        sb[s] = id;
        bstr[id] = beta;  // every source of this beta string writes the same
        diag[s] = diagonal_of(d, J, stride, hd, hstride, alpha, beta);
    }
}

// shared memory of beta_tables_kernel: binomials, the prefix sums of each occupied
// pair's remainder, the virtual pairs' orbitals, and (kKeep) every double's pi and
// integral index between the two passes
__host__ __device__ inline size_t beta_smem(const SysDev &d, bool keep) {
    const size_t m = d.nb > 1 ? d.nb - 1 : 1;
    return size_t(d.n + 1) * d.ks * 8 + ((size_t(d.po_b) * 3 * m * 4 + size_t(d.pv_b) * 2 + 15) & ~size_t(15)) +
           (keep ? size_t(d.po_b) * d.pv_b * 10 : 0);
}

// Tables of the distinct beta strings, one CTA per string: its single
// excitations {pi(beta'), b n + j | sign << 31} ordered by the top kb1 bits of
// pi, its double excitations pi(beta') and signed element ordered by the top
// kb2 bits, and where each bin starts.  Two passes (count the bins, then place);
// a warp takes an occupied pair at a time and its lanes the virtual pairs, and
// the first pass keeps what the second needs when it fits (kKeep), so that the
// table leaves in order, in full sectors: 88000 strings of 4410 doubles took 6.8 ms
// with both passes computed and every double stored where its bin had room.
template <bool kKeep>
__global__ void __launch_bounds__(256)
beta_tables_kernel(const SysDev d, const GatherShape p, const unsigned long long *bstr, unsigned nd, const double *W,
                   uint2 *t1, unsigned short *idx1, unsigned *t2p, double *t2e, unsigned *idx2) {
    extern __shared__ unsigned long long bt[];
    load_binom(d, bt);
    const int n = d.n, ks = d.ks, m = d.nb, M = m - 2;
    const int stride = 3 * (m > 1 ? m - 1 : 1);
    unsigned *pre = reinterpret_cast<unsigned *>(bt + (n + 1) * ks);  // [po_b][3][m - 1] prefix sums of the remainder
    unsigned short *vp = reinterpret_cast<unsigned short *>(pre + d.po_b * stride);  // virtual pairs: a | b << 8
    uint2 *kept = reinterpret_cast<uint2 *>(reinterpret_cast<unsigned char *>(bt) + beta_smem(d, false));
    unsigned short *perm = reinterpret_cast<unsigned short *>(kept + p.nd2);  // the doubles in the order of their bins
    __shared__ unsigned h1[128], h2[512];
    __shared__ unsigned char occ[64], vir[64];
    const int nb1 = 1 << p.kb1, nb2 = 1 << p.kb2, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned char *po = d.pairs + 2 * d.pair_off[2], *pv = d.pairs + 2 * d.pair_off[3];
    for (unsigned id = blockIdx.x; id < nd; id += gridDim.x) {
        const unsigned long long beta = bstr[id];
        for (int i = tid; i < nb1; i += blockDim.x) h1[i] = 0;
        for (int i = tid; i < nb2; i += blockDim.x) h2[i] = 0;
        if (tid < n) {
            const unsigned long long below = beta & ((1ull << tid) - 1ull);
            if ((beta >> tid) & 1ull) occ[__popcll(below)] = (unsigned char)tid;
            else vir[tid - __popcll(below)] = (unsigned char)tid;
        }
        __syncthreads();
        for (int v = tid; v < d.pv_b; v += blockDim.x)
            vp[v] = (unsigned short)(vir[__ldg(&pv[2 * v])] | vir[__ldg(&pv[2 * v + 1])] << 8);
        for (int q = tid; q < d.po_b; q += blockDim.x) {
            const int x = po[2 * q], y = po[2 * q + 1];
            unsigned *A0 = pre + q * stride, *A1 = A0 + m - 1, *A2 = A1 + m - 1;
            A0[0] = A1[0] = A2[0] = 0;
            for (int t = 0; t < M; ++t) {
                int e = t;
                if (e >= x) ++e;
                if (e >= y) ++e;
                const int o = occ[e];
                A0[t + 1] = A0[t] + (unsigned)bt[o * ks + t + 1];
                A1[t + 1] = A1[t] + (unsigned)bt[o * ks + t + 2];
                A2[t + 1] = A2[t] + (unsigned)bt[o * ks + t + 3];
            }
        }
        __syncthreads();
        auto single = [&](int y, unsigned &pi, unsigned &x) {
            const int jo = y / d.vb, j = occ[jo], b = vir[y - jo * d.vb];
            pi = bperm(p, (unsigned)string_rank(beta ^ (1ull << j) ^ (1ull << b), bt, ks));
            x = (unsigned)(b * n + j) | ((unsigned)parity64(beta & between_mask(j, b)) << 31);
        };
        // every double as f(number, pi, index of its integral in W | sign << 31)
        auto doubles = [&](auto &&f) {
            for (int q = warp; q < d.po_b; q += 8) {
                const int x = __ldg(&po[2 * q]), y = __ldg(&po[2 * q + 1]), i = occ[x], j = occ[y];
                const unsigned long long rem = beta ^ (1ull << i) ^ (1ull << j);
                const unsigned rlo = (unsigned)rem, rhi = (unsigned)(rem >> 32), nlo = __popc(rlo);
                const unsigned *A0 = pre + q * stride, *A1 = A0 + m - 1, *A2 = A1 + m - 1;
                const unsigned ij = (unsigned)(j * (j - 1) / 2 + i), a2m = A2[M], sxy = (unsigned)(x + y - 1);
                auto below = [&](int o) {  // electrons of the remainder below orbital o
                    return o < 32 ? __popc(rlo & ((1u << o) - 1u)) : nlo + __popc(rhi & ((1u << (o - 32)) - 1u));
                };
                for (int v = lane; v < d.pv_b; v += 32) {
                    const int a = vp[v] & 0xff, b = vp[v] >> 8;
                    const unsigned q1 = below(a), q2 = below(b);
                    const unsigned r = A0[q1] + (unsigned)bt[a * ks + q1 + 1] + A1[q2] - A1[q1] +
                                       (unsigned)bt[b * ks + q2 + 2] + a2m - A2[q2];
                    f(q * d.pv_b + v, bperm(p, r),
                      ((unsigned)(b * (b - 1) / 2 + a) * p.npair + ij) | ((sxy + q1 + q2) & 1u) << 31);
                }
            }
        };
        const int s1 = p.bb - p.kb1, s2 = p.bb - p.kb2;
        for (int y = tid; y < d.sb; y += blockDim.x) {
            unsigned pi, x;
            single(y, pi, x);
            atomicAdd(&h1[pi >> s1], 1u);
        }
        doubles([&](int e, unsigned pi, unsigned w) {
            atomicAdd(&h2[pi >> s2], 1u);
            if (kKeep) kept[e] = make_uint2(pi, w);
        });
        __syncthreads();
        if (tid < 64) {  // warp 0: singles' bins, warp 1: doubles' bins
            unsigned *h = tid < 32 ? h1 : h2;
            const int nbin = tid < 32 ? nb1 : nb2;
            unsigned run = 0;
            for (int b0 = 0; b0 < nbin; b0 += 32) {
                const unsigned v = b0 + lane < nbin ? h[b0 + lane] : 0u;
                unsigned x = v;
                for (int o = 1; o < 32; o <<= 1) {
                    const unsigned u = __shfl_up_sync(kFull, x, o);
                    if (lane >= o) x += u;
                }
                if (b0 + lane < nbin) {
                    h[b0 + lane] = run + x - v;
                    if (tid < 32) idx1[(size_t)id * (nb1 + 1) + b0 + lane] = (unsigned short)(run + x - v);
                    else idx2[(size_t)id * (nb2 + 1) + b0 + lane] = run + x - v;
                }
                run += __shfl_sync(kFull, x, 31);
            }
            if (lane == 0) {
                if (tid < 32) idx1[(size_t)id * (nb1 + 1) + nb1] = (unsigned short)run;
                else idx2[(size_t)id * (nb2 + 1) + nb2] = run;
            }
        }
        __syncthreads();
        for (int y = tid; y < d.sb; y += blockDim.x) {
            unsigned pi, x;
            single(y, pi, x);
            t1[(size_t)id * d.sb + atomicAdd(&h1[pi >> s1], 1u)] = make_uint2(pi, x);
        }
        auto place = [&](unsigned pi, unsigned w) {
            const size_t o = (size_t)id * p.nd2 + atomicAdd(&h2[pi >> s2], 1u);
            t2p[o] = pi;
            t2e[o] = flip_d(__ldg(&W[w & 0x7fffffffu]), w >> 31);
        };
        if (kKeep) {
            for (int e = tid; e < p.nd2; e += blockDim.x) perm[atomicAdd(&h2[kept[e].x >> s2], 1u)] = (unsigned short)e;
            __syncthreads();
            for (int o = tid; o < p.nd2; o += blockDim.x) {
                const uint2 k = kept[perm[o]];
                t2p[(size_t)id * p.nd2 + o] = k.x;
                t2e[(size_t)id * p.nd2 + o] = flip_d(__ldg(&W[k.y & 0x7fffffffu]), k.y >> 31);
            }
        } else {
            doubles([&](int, unsigned pi, unsigned w) { place(pi, w); });
        }
        __syncthreads();
    }
}

// index (Eq. 12) of the string with electrons x and y removed (y >= m: x alone)
// from prefix sums P0, P1, P2 of C(e_t, t + 1), C(e_t, t), C(e_t, t - 1)
__device__ __forceinline__ unsigned rank_without(const unsigned *P0, const unsigned *P1, const unsigned *P2, int m,
                                                 int x, int y) {
    return y >= m ? P0[x] + P1[m] - P1[x + 1] : P0[x] + P1[y] - P1[x + 1] + P2[m] - P2[y + 1];
}

__device__ __forceinline__ void string_prefix(unsigned long long s, const unsigned long long *bt, int ks, unsigned *P0,
                                              unsigned *P1, unsigned *P2, unsigned char *e) {
    int t = 0;
    P0[0] = P1[0] = P2[0] = 0;
    for (; s; s &= s - 1ull, ++t) {
        const int o = __ffsll((long long)s) - 1;
        e[t] = (unsigned char)o;
        P0[t + 1] = P0[t] + (unsigned)bt[o * ks + t + 1];
        P1[t + 1] = P1[t] + (unsigned)bt[o * ks + t];
        P2[t + 1] = P2[t] + (t > 0 ? (unsigned)bt[o * ks + t - 1] : 0u);
    }
}

// The sources under the (n_alpha - 1)- and (n_alpha - 2)-electron substrings of their
// alpha strings: counted when ent2 is null, else written to off[K] + their turn.  An
// entry holds what a row needs of it, so that reading a list is one coalesced stream:
//   ent1 {pi(beta), beta string's number | i << 25 | s_K(i) << 31, c}
//   ent2 {pi(beta), pair (i, j) | s_K(i, j) << 31, c}
// with i (i, j) the orbitals the substring lacks.  Bound by the counters' atomics: sources
// lie by alpha string, so whole warps meet at the same substrings, and one lane counts for
// all that share a string; blockIdx.y is the first electron taken out (2e4 sources of 924
// strings: 161 us for both passes with an atomic per source and substring).
__global__ void substring_lists_kernel(const SysDev d, const GatherShape p, const unsigned long long *skey,
                                       const double *sc, const unsigned *sb, long long n, unsigned *cnt1, unsigned *cnt2,
                                       const unsigned long long *off1, const unsigned long long *off2, uint4 *ent1,
                                       uint4 *ent2) {
    extern __shared__ unsigned long long bt[];
    load_binom(d, bt);
    const int m = d.na, x = blockIdx.y, lane = threadIdx.x & 31;
    unsigned P0[kMaxE + 1], P1[kMaxE + 1], P2[kMaxE + 1];
    unsigned char e[kMaxE];
    for (long long s0 = blockIdx.x * (long long)blockDim.x + (threadIdx.x & ~31); s0 < n; s0 += (long long)gridDim.x * blockDim.x) {
        const long long s = s0 + lane;
        const bool in = s < n;
        const unsigned long long key = skey[in ? s : n - 1];
        const unsigned row = (unsigned)(key >> p.bb);
        string_prefix(unrank_one(row, d.n, m, bt, d.ks), bt, d.ks, P0, P1, P2, e);
        const unsigned pi = (unsigned)key & p.bmask, id = ent2 && in ? sb[s] : 0u;
        const double c = in ? sc[s] : 0.0;
        const unsigned clo = (unsigned)__double2loint(c), chi = (unsigned)__double2hiint(c);
        // the lanes of one alpha string take their places together
        const unsigned peers = __match_any_sync(kFull, in ? row : kNoKey);
        const int lead = __ffs((int)peers) - 1;
        const unsigned many = __popc(peers), mine = __popc(peers & ((1u << lane) - 1u));
        auto place = [&](unsigned *cnt, unsigned K) {
            unsigned base = 0u;
            if (in && lane == lead) {
                if (!ent2) atomicAdd(&cnt[K], many);
                else base = atomicSub(&cnt[K], many) - many;
            }
            return ent2 ? __shfl_sync(kFull, base, lead) + mine : 0u;
        };
        {
            const unsigned K = rank_without(P0, P1, P2, m, x, m), at = place(cnt1, K);
            if (ent2 && in)
                ent1[off1[K] + at] = make_uint4(pi, id | (unsigned)e[x] << 25 | (unsigned)(x & 1) << 31, clo, chi);
        }
        for (int y = x + 1; y < m; ++y) {
            const unsigned K = rank_without(P0, P1, P2, m, x, y), at = place(cnt2, K);
            if (ent2 && in)
                ent2[off2[K] + at] = make_uint4(
                    pi, (unsigned)(e[y] * (e[y] - 1) / 2 + e[x]) | (unsigned)((x + y - 1) & 1) << 31, clo, chi);
        }
    }
}

constexpr int kRowChunk = 8;  // consecutive rows per thread (one unrank, then successors)

// per row: s1 the sources one alpha hop away and s2 the sources listed under its
// (n_alpha - 2)-electron substrings (those two hops away once, the nearer ones
// several times: their entries drop out), from the source totals of the
// substrings; act = 1 for a row that any source reaches
__global__ void row_sources_kernel(const SysDev d, const unsigned *rp, const unsigned long long *off1,
                                   const unsigned long long *off2, unsigned *s1, unsigned *s2, unsigned *act) {
    extern __shared__ unsigned long long bt[];
    load_binom(d, bt);
    const int m = d.na;
    unsigned P0[kMaxE + 1], P1[kMaxE + 1], P2[kMaxE + 1];
    unsigned char e[kMaxE];
    const unsigned long long chunks = (d.ca + kRowChunk - 1) / kRowChunk;
    for (unsigned long long c = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; c < chunks;
         c += (unsigned long long)gridDim.x * blockDim.x) {
        unsigned long long s = unrank_one(c * kRowChunk, d.n, m, bt, d.ks);
        for (unsigned long long r = c * kRowChunk; r < d.ca && r < (c + 1) * kRowChunk; ++r, s = next_string(s)) {
            string_prefix(s, bt, d.ks, P0, P1, P2, e);
            unsigned long long S1 = 0, S2 = 0;
            const unsigned long long L = rp[r + 1] - rp[r];
            for (int x = 0; x < m; ++x) {
                const unsigned K1 = rank_without(P0, P1, P2, m, x, m);
                S1 += __ldg(&off1[K1 + 1]) - __ldg(&off1[K1]);
                for (int y = x + 1; y < m; ++y) {
                    const unsigned K2 = rank_without(P0, P1, P2, m, x, y);
                    S2 += __ldg(&off2[K2 + 1]) - __ldg(&off2[K2]);
                }
            }
            S1 -= m * L;
            s1[r] = (unsigned)S1;
            s2[r] = d.ss_any ? (unsigned)S2 : 0u;
            act[r] = L + S1 + S2 != 0ull;
        }
    }
}

// the rows with elements, in order: row, string, records (alpha-alpha doubles,
// alpha singles, and per own source the diagonal and the beta singles), one-hop
// sources, weight (elements and the fixed cost of a row), parts of its lists
__global__ void active_rows_kernel(const SysDev d, const GatherShape p, const unsigned *rp, const unsigned *s1,
                                   const unsigned *s2, const unsigned *act, const unsigned long long *pos,
                                   unsigned w_fixed, unsigned part_work, unsigned *row, unsigned long long *str, unsigned long long *aw,
                                   unsigned *nrec, unsigned *nab, unsigned *np) {
    extern __shared__ unsigned long long bt[];
    load_binom(d, bt);
    const unsigned long long chunks = (d.ca + kRowChunk - 1) / kRowChunk;
    for (unsigned long long c = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; c < chunks;
         c += (unsigned long long)gridDim.x * blockDim.x) {
        unsigned long long s = unrank_one(c * kRowChunk, d.n, d.na, bt, d.ks);
        for (unsigned long long r = c * kRowChunk; r < d.ca && r < (c + 1) * kRowChunk; ++r, s = next_string(s))
            if (act[r]) {
                const unsigned long long k = pos[r];
                const unsigned L = rp[r + 1] - rp[r];
                const unsigned rec = s2[r] + s1[r] + L * (1u + d.sb), ab = d.ab_any ? s1[r] : 0u;
                row[k] = (unsigned)r;
                str[k] = s;
                nrec[k] = rec;
                nab[k] = ab;
                aw[k] = rec + (unsigned long long)ab * d.sb + (unsigned long long)L * (d.ss_any ? p.nd2 : 0) + w_fixed;
                np[k] = min((rec + ab + part_work - 1) / part_work + (rec + ab == 0u), kMaxParts);
            }
    }
}

struct RowPlan {
    unsigned long long half;  // light rows: weight at most half a group
    double fill;              // distinct entries a table should hold
    double cb;
    int bb;
    const unsigned long long *seen;  // per weight bin: elements and distinct entries of the rows done so far
};

__device__ __forceinline__ int weight_bin(unsigned long long w) {  // half octaves
    const int l = 63 - __clzll((long long)(w | 1ull));
    return 2 * l + (l > 0 ? (int)((w >> (l - 1)) & 1ull) : 0);
}

__device__ __forceinline__ unsigned class_count(const RowPlan &r, double entries) {
    const unsigned n = (unsigned)ceil(entries / r.fill), most = r.bb > kGLog ? 1u << min(r.bb - kGLog, kMaxClassLog) : 1u;
    return n < 1u ? 1u : n < most ? n : most;
}

// Classes of a heavy row, from the distinct entries expected of it: elements over 1.6
// (w / 1024)^(1/4), moved towards what the rows of its weight had in the last sigmas (what truncated Lanczos vectors of 28 orbitals show: 1.6 at
// 1e3 elements, 3.6 at 1.6e4, 6.5 at 3e5, 16 at 4e6).  Only a plan: a class that
// turns out too full is split on the way.
__device__ __forceinline__ unsigned row_classes(const RowPlan &r, unsigned long long w) {
    const int b = weight_bin(w);
    const unsigned long long e = r.seen[2 * b], x = r.seen[2 * b + 1];
    double est = (double)w / (1.6 * sqrt(sqrt((double)w / 1024.0)));
    if (x > kSeenEnough) {
        const double was = (double)w * ((double)x / (double)e);
        est = was > est ? was : sqrt(was * est);
    }
    return class_count(r, est > r.cb ? r.cb : est);
}

// per active row: units it opens (a heavy row one per class, a light row one if
// it is the first of its group: the light rows whose weight prefix starts in
// one window of half a group)
// visits: sources that its classes read, summed over the heavy rows; own ones count four
// times (their segments are longer).
// The guess of row_classes is for vectors like Lanczos', whose sources share beta strings.  Where
// they do not (scattered), and no sigma has shown yet what the rows hold, a row's elements count as
// scattered over all strings: planned by the other guess its classes split again and again (3e5
// determinants drawn from 2e4 rows of 28 orbitals: the first sigma 825 ms, 532 so, by buckets 627).
// That is the most a row can hold, so a quarter more than a class should hold is left in one (two
// took 2 % of a sigma of 73 determinants; with every class 18 % fuller they overflow: 30000 of 28
// orbitals, 1 + 7 electrons 23.9 and 37.7 ms), and its visits count 23 / 32.
__global__ void row_units_kernel(RowPlan rp, const unsigned long long *aw, const unsigned long long *wpre,
                                 const unsigned long long *n_act, const unsigned *nab, const unsigned *row,
                                 const unsigned *src, unsigned *nu, bool scattered, unsigned long long *visits) {
    const unsigned long long A = *n_act;
    unsigned long long sum = 0ull;
    for (unsigned long long k = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; k < A;
         k += (unsigned long long)gridDim.x * blockDim.x) {
        const unsigned long long w = aw[k];
        if (w > rp.half && rp.bb <= kGLog) {
            nu[k] = 1u;  // (one table holds all strings)
        } else if (w > rp.half) {
            unsigned n;
            if (scattered) {
                const double most = -rp.cb * expm1(-(double)w / rp.cb);
                n = most <= 1.25 * rp.fill ? 1u : class_count(rp, most);
            } else {
                n = row_classes(rp, w);
            }
            nu[k] = n;
            const unsigned long long v = nab[k] + 4ull * (src[row[k] + 1] - src[row[k]]);
            if (n > 1u) sum += scattered ? n * v * 23ull / 32ull : n * v;
        } else nu[k] = k == 0 || aw[k - 1] > rp.half || wpre[k - 1] / rp.half != wpre[k] / rp.half;
    }
    if (rp.bb <= kGLog) return;
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(kFull, sum, o);
    if ((threadIdx.x & 31) == 0 && sum) atomicAdd(visits, sum);
}

__global__ void write_units_kernel(RowPlan rp, const unsigned long long *aw, const unsigned long long *wpre,
                                   unsigned long long A, const unsigned *nu, const unsigned *np,
                                   const unsigned long long *uoff, const unsigned long long *poff,
                                   const unsigned long long *rec_off, const unsigned long long *ab_off,
                                   const unsigned *row, const unsigned *src, GatherUnit *units, unsigned *part_k,
                                   unsigned *split_rows, unsigned long long *n_split) {
    for (unsigned long long k = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; k < A;
         k += (unsigned long long)gridDim.x * blockDim.x) {
        for (unsigned q = 0; q < np[k]; ++q) part_k[poff[k] + q] = (unsigned)k;
        const unsigned long long w = aw[k];
        const unsigned r = row[k];
        const bool heavy = w > rp.half;
        const unsigned n = heavy ? nu[k] : 1u;
        if (n > 1u) split_rows[atomicAdd(n_split, 1ull)] = (unsigned)k;
        const unsigned long long t = wpre[k] / rp.half;
        const bool first = heavy || nu[k];
        const bool last = heavy || k + 1 == A || aw[k + 1] > rp.half || wpre[k + 1] / rp.half != t;
        for (unsigned c = 0; c < n; ++c) {
            GatherUnit *u = units + (heavy ? uoff[k] + c : uoff[k] + nu[k] - 1);
            if (first) {
                u->rec0 = rec_off[k], u->ab0 = (unsigned)ab_off[k], u->src0 = src[r];
                u->k0 = (unsigned)k;
                // pi * n >> bb == c for lo <= pi < hi
                u->lo = (unsigned)((((unsigned long long)c << rp.bb) + n - 1) / n);
                u->hi = (unsigned)((((unsigned long long)(c + 1) << rp.bb) + n - 1) / n);
                u->bin = heavy ? (unsigned)weight_bin(w) : 0u, u->n_cls = n;
            }
            if (last) u->rec1 = rec_off[k + 1], u->ab1 = (unsigned)ab_off[k + 1], u->src1 = src[r + 1], u->k1 = (unsigned)k + 1;
        }
    }
}

// ------------------------------------------------------------- row lists

// which of the segments starting at cs (ascending over the lanes, ~0 past the
// last) holds element e0 + lane (every lane calls it)
__device__ __forceinline__ int segment_of(unsigned cs, unsigned e0, int lane) {
    const unsigned before = __popc(__ballot_sync(kFull, cs <= e0));
    const unsigned rel = cs - e0;
    const unsigned mask = __reduce_or_sync(kFull, cs > e0 && rel < 32u ? 1u << rel : 0u);
    return (int)(before + __popc(mask & ((2u << lane) - 1u))) - 1;
}

__device__ __forceinline__ unsigned warp_scan(unsigned x, int lane) {  // inclusive
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

struct ListArea {
    unsigned P0[kMaxE + 1], P1[kMaxE + 1], P2[kMaxE + 1];
    unsigned char own[32], occ[kMaxE];
};

// start (over the lanes) of the non-empty segments in order, ~0 past the last;
// own[m] = lane of the m-th
__device__ __forceinline__ unsigned pack_segments(ListArea &wa, unsigned len, unsigned start, int lane) {
    const unsigned nb = __ballot_sync(kFull, len != 0u);
    __syncwarp();
    if (len) wa.own[__popc(nb & ((1u << lane) - 1u))] = (unsigned char)lane;
    __syncwarp();
    const unsigned cs = __shfl_sync(kFull, start, lane < __popc(nb) ? wa.own[lane] : 0);
    return lane < __popc(nb) ? cs : ~0u;
}

// The rows' lists.  A warp takes a part (1/nq of the items) of a row:
//   records: [rec_off, + s2) the sources listed under its substrings (alpha-alpha
//   doubles; 0 for the nearer ones), then S1 alpha singles, then per own source the diagonal and the beta singles;
//   ab: the S1 one-hop sources {beta string, integral row | row in group << 24 |
//   sign << 31, c_D}.
// Record keys carry the row's number in its group.  Bound by the list entries'
// and integrals' load latency: one thread per entry, 48 warps an SM (40 registers: 7 %
// less time for the lists and tables than 32 warps with 64).
__global__ void __launch_bounds__(kLT, 6)
row_lists_kernel(const __grid_constant__ ListArgs A) {
    extern __shared__ unsigned long long bt[];
    __shared__ ListArea areas[kLT / 32];
    const SysDev &d = A.d;
    const GatherShape &gs = A.gs;
    load_binom(d, bt);
    const int tid = threadIdx.x, lane = tid & 31;
    const int n = d.n, ks = d.ks, na = d.na, bb = gs.bb;
    ListArea &wa = areas[tid >> 5];
    for (unsigned part = blockIdx.x * (kLT / 32) + (tid >> 5); part < A.n_parts; part += gridDim.x * (kLT / 32)) {
        const unsigned k = __ldg(&A.part_k[part]);
        const unsigned q = part - (unsigned)__ldg(&A.poff[k]), nq = (unsigned)(__ldg(&A.poff[k + 1]) - __ldg(&A.poff[k]));
        const unsigned row = __ldg(&A.act_row[k]);
        const unsigned long long str = __ldg(&A.act_str[k]);
        const unsigned uo = (unsigned)__ldg(&A.uoff[k]) + __ldg(&A.nu[k]);
        const GatherUnit *un = A.units + (uo - 1);
        const unsigned rl = k - __ldg(&un->k0), kb = rl << bb;
        const unsigned long long rec = __ldg(&A.rec_off[k]);
        const unsigned long long ab = __ldg(&A.ab_off[k]);
        const unsigned s1 = __ldg(&A.s1[row]), s2 = __ldg(&A.s2[row]);
        // electrons and prefix sums of the row's string
        __syncwarp();
        for (int half = 0; half < 2; ++half) {
            const int o = lane + 32 * half;
            if (o < n && ((str >> o) & 1ull)) wa.occ[__popcll(str & ((1ull << o) - 1ull))] = (unsigned char)o;
        }
        __syncwarp();
        {
            unsigned c0 = 0, c1 = 0, c2 = 0;
            if (lane < na) {
                const unsigned long long *b = bt + wa.occ[lane] * ks + lane;
                c0 = (unsigned)b[1], c1 = (unsigned)b[0], c2 = lane > 0 ? (unsigned)b[-1] : 0u;
            }
            c0 = warp_scan(c0, lane), c1 = warp_scan(c1, lane), c2 = warp_scan(c2, lane);
            if (lane < na) wa.P0[lane + 1] = c0, wa.P1[lane + 1] = c1, wa.P2[lane + 1] = c2;
            if (lane == 0) wa.P0[0] = wa.P1[0] = wa.P2[0] = 0u;
        }
        __syncwarp();
        // ---- alpha-alpha doubles: the lists of the (n_alpha - 2)-electron substrings, end to end
        unsigned before = 0;  // entries of the lists before this block of 32
        for (int p0 = 0; p0 < (s2 ? d.po_a : 0); p0 += 32) {
            const int p = p0 + lane;
            unsigned off = 0, len = 0, info = 0;
            if (p < d.po_a) {
                const int x = __ldg(&d.pairs[2 * p]), y = __ldg(&d.pairs[2 * p + 1]);
                const unsigned K = rank_without(wa.P0, wa.P1, wa.P2, na, x, y);
                off = (unsigned)__ldg(&A.off2[K]);
                len = (unsigned)__ldg(&A.off2[K + 1]) - off;
                const unsigned a = wa.occ[x], b = wa.occ[y];
                info = (b * (b - 1) / 2 + a) * gs.npair | (unsigned)((x + y - 1) & 1) << 31;
            }
            const unsigned inc = warp_scan(len, lane), total = __shfl_sync(kFull, inc, 31), start = inc - len;
            const unsigned cs = pack_segments(wa, len, start, lane);
#pragma unroll 2
            for (unsigned e0 = 32 * q; e0 < total; e0 += 32 * nq) {
                const int ol = wa.own[segment_of(cs, e0, lane)];
                const unsigned eo = __shfl_sync(kFull, off - start, ol) + e0 + lane, inf = __shfl_sync(kFull, info, ol);
                if (e0 + lane < total) {
                    const uint4 en = __ldg(&A.ent2[eo]);
                    const double ev = flip_d(__ldg(&A.W[(inf & 0x7fffffffu) + (en.y & 0x7fffffffu)]), (en.y ^ inf) >> 31);
                    const unsigned long long r = rec + before + e0 + lane;
                    __stcs(&A.rkey[r], kb | en.x);
                    __stcs(&A.rval[r], __dmul_rn(ev, __hiloint2double((int)en.w, (int)en.z)));
                }
            }
            before += total;
        }
        const unsigned s_own = __ldg(&A.rp[row]), L_own = __ldg(&A.rp[row + 1]) - s_own;
        // ---- one alpha hop: the lists of the (n_alpha - 1)-electron substrings (each holds
        // the row's own sources too: a row that has some counts the others with a cursor)
        if (s1) {
            unsigned off = 0, len = 0;
            if (lane < na) {
                const unsigned K = rank_without(wa.P0, wa.P1, wa.P2, na, lane, na);
                off = (unsigned)__ldg(&A.off1[K]);
                len = (unsigned)__ldg(&A.off1[K + 1]) - off;
            }
            const unsigned inc = warp_scan(len, lane), total = __shfl_sync(kFull, inc, 31), start = inc - len;
            const unsigned cs = pack_segments(wa, len, start, lane);
            for (unsigned e0 = 32 * q; e0 < total; e0 += 32 * nq) {
                const int x = wa.own[segment_of(cs, e0, lane)];
                const unsigned eo = __shfl_sync(kFull, off - start, x) + e0 + lane, a = wa.occ[x];
                uint4 en = make_uint4(0u, a << 25, 0u, 0u);
                if (e0 + lane < total) en = __ldg(&A.ent1[eo]);
                const unsigned i = (en.y >> 25) & 0x3fu, id = en.y & 0x1ffffffu;
                const bool hop = i != a;
                unsigned pos = e0 + lane;
                if (L_own) {
                    const unsigned bal = __ballot_sync(kFull, hop);
                    unsigned base = 0;
                    if (lane == 0 && bal) base = atomicAdd(&A.cursor[k], (unsigned)__popc(bal));
                    pos = __shfl_sync(kFull, base, 0) + __popc(bal & ((1u << lane) - 1u));
                }
                if (hop) {
                    const unsigned sg = (en.y >> 31) ^ ((unsigned)x & 1u);
                    const double c = __hiloint2double((int)en.w, (int)en.z);
                    const unsigned long long al = str ^ (1ull << a) ^ (1ull << i);
                    A.rkey[rec + s2 + pos] = kb | en.x;
                    A.rval[rec + s2 + pos] =
                        __dmul_rn(flip_d(single_of(d, (int)i, (int)a, al, __ldg(&A.bstr[id]), al), sg), c);
                    if (d.ab_any)
                        A.ab[ab + pos] = make_uint4(id, (a * n + i) * (unsigned)(n * n) | rl << 24 | sg << 31, en.z, en.w);
                }
            }
        }
        // ---- the row's own sources: diagonal and beta singles
        {
            const unsigned per = 1u + (unsigned)d.sb;
            for (unsigned t = 32 * q + lane; t < L_own * per; t += 32 * nq) {
                const unsigned s = s_own + t / per, y = t % per;
                const unsigned id = __ldg(&A.s_b[s]);
                const double c = __ldg(&A.s_c[s]);
                unsigned pi;
                double v;
                if (y == 0u) {
                    pi = __ldg(&A.s_pi[s]);
                    v = __dmul_rn(__ldg(&A.s_diag[s]), c);
                } else {
                    const uint2 y1 = __ldg(&A.t1[id * (unsigned)d.sb + y - 1u]);
                    const unsigned bj = y1.y & 0x7fffffffu;
                    const int bo = (int)(bj / (unsigned)n), jo = (int)(bj - (unsigned)bo * n);
                    const unsigned long long be = __ldg(&A.bstr[id]);
                    pi = y1.x;
                    v = __dmul_rn(flip_d(single_of(d, jo, bo, str, be, be), y1.y >> 31), c);
                }
                A.rkey[rec + s2 + s1 + t] = kb | pi;
                A.rval[rec + s2 + s1 + t] = v;
                if (y == 0u) A.s_kb[s] = kb;
            }
        }
    }
}

// The records of each row that is summed in classes, in the order of their class (a
// class would otherwise read all of its row's records: ten times those it keeps in the
// heaviest rows); each class's unit gets its range.  One CTA per row, two passes.
__global__ void __launch_bounds__(512)
class_order_kernel(const GatherShape gs, const unsigned *split_rows, const unsigned long long *n_split,
                   const unsigned *nu, const unsigned long long *uoff, const unsigned long long *rec_off,
                   const unsigned *rkey, const double *rval, unsigned *okey, double *oval, GatherUnit *units) {
    __shared__ unsigned h[1 << kMaxClassLog];
    __shared__ unsigned wt[16];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned long long n = *n_split;
    for (unsigned long long t = blockIdx.x; t < n; t += gridDim.x) {
        const unsigned k = split_rows[t], nc = nu[k];
        const unsigned long long r0 = rec_off[k];
        const unsigned cnt = (unsigned)(rec_off[k + 1] - r0);
        GatherUnit *u = units + uoff[k];
        for (unsigned c = tid; c < nc; c += 512) h[c] = 0u;
        __syncthreads();
        for (unsigned i = tid; i < cnt; i += 512)
            atomicAdd(&h[(unsigned)(((unsigned long long)rkey[r0 + i] * nc) >> gs.bb)], 1u);
        __syncthreads();
        unsigned carry = 0;
        for (unsigned c0 = 0; c0 < nc; c0 += 512) {
            const unsigned c = c0 + tid, v = c < nc ? h[c] : 0u;
            const unsigned x = warp_scan(v, lane);
            if (lane == 31) wt[warp] = x;
            __syncthreads();
            const unsigned ws = warp_scan(lane < 16 ? wt[lane] : 0u, lane);
            const unsigned ex = carry + x - v + (warp > 0 ? __shfl_sync(kFull, ws, warp - 1) : 0u);
            carry += __shfl_sync(kFull, ws, 15);
            if (c < nc) {
                h[c] = ex;
                u[c].rec0 = r0 + ex, u[c].rec1 = r0 + ex + v;
            }
            __syncthreads();
        }
        for (unsigned i0 = 0; i0 < cnt; i0 += 2048) {  // four in flight per thread
            unsigned key[4], at[4];
            double v[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const unsigned i = i0 + j * 512 + tid;
                if (i < cnt) key[j] = __ldcs(&rkey[r0 + i]), v[j] = __ldcs(&rval[r0 + i]);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (i0 + j * 512 + tid < cnt) at[j] = atomicAdd(&h[(unsigned)(((unsigned long long)key[j] * nc) >> gs.bb)], 1u);
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (i0 + j * 512 + tid < cnt) okey[r0 + at[j]] = key[j], oval[r0 + at[j]] = v[j];
        }
        __syncthreads();
    }
}

// ------------------------------------------------------------- gather

constexpr int kQueue = 64;  // elements of a warp waiting for a full round

struct WarpArea {
    union {
        struct {
            double v[kQueue];
            unsigned k[kQueue];
        } q;                                 // queued elements
        unsigned short list[kGSlots / kGW];  // occupied slots of the warp's share
    };
};

// The sources whose doubles the CTA is summing, up to one per thread: where each
// one's segment of its string's table begins (less its first element's number),
// what it carries, and its first element's number.
struct alignas(16) SourceBatch {
    uint4 st[kGT];
    unsigned start[kGT + 1];
    unsigned warp_tot[kGW];
};

// One element on its way into the table.
struct Element {
    unsigned key, slot;
    double v;
    bool ok;
};

// The CTA's table: 32-bit keys, each sum as four 32-bit limbs (their own arrays:
// 32 lanes hit 32 banks), exact in units of 2^-S.
struct TableView {
    unsigned *keys, *limb;
    unsigned max_probe;
    int S;
    volatile int *over;
};

// Adds v to the entry `key`, looked for from `slot` on (triangular steps: every slot once);
// called by every lane of the warp.  kAll: to the end; else at most two places are tried
// (a warp that probes to the end waits for its slowest lane, about eight places: the few
// elements that need more come back together).  False: not added.
// The value is placed as three 32-bit words at limb sh / 32 (the limbs below would receive
// 0) and each limb's carry goes up with the next add; lanes without an element add 0, so
// that the adds need no branches.
template <bool kAll>
__device__ __forceinline__ bool add_element(const TableView &t, const Element &el, bool &range_ok) {
    unsigned h = el.slot & (kGSlots - 1);
    unsigned old = el.ok ? atomicCAS(&t.keys[h], kNoKey, el.key) : kNoKey;
    bool hit = old == kNoKey || old == el.key;
    if (kAll) {
        for (unsigned probe = 0; !hit;) {
            h = (h + ++probe) & (kGSlots - 1);
            if (probe >= t.max_probe) {
                *t.over = 1;
                break;
            }
            old = atomicCAS(&t.keys[h], kNoKey, el.key);
            hit = old == kNoKey || old == el.key;
        }
    } else if (!hit) {
        h = (h + 1u) & (kGSlots - 1);
        old = atomicCAS(&t.keys[h], kNoKey, el.key);
        hit = old == kNoKey || old == el.key;
    }
    const bool ok = el.ok && hit;
    const unsigned hi = (unsigned)__double2hiint(el.v), lo = (unsigned)__double2loint(el.v);
    const unsigned ex = (hi >> 20) & 0x7ffu;
    const unsigned mh = (hi & 0xfffffu) | (ex ? 0x100000u : 0u);
    const int sh = (int)(ex ? ex : 1u) - 1075 + t.S;
    const unsigned r = (unsigned)sh & 31u;
    unsigned x0 = lo << r, x1 = __funnelshift_l(lo, mh, r), x2 = __funnelshift_l(mh, 0u, r);
    unsigned q = min((unsigned)sh >> 5, 3u);
    range_ok = range_ok && !(ok && sh > 74);  // would not fit in 127 bits
    if (__any_sync(kFull, ok && sh < 0)) {
        if (ok && sh < 0) {  // below the unit: nearest, ties away from zero
            const unsigned long long m = ((unsigned long long)mh << 32) | lo;
            const unsigned rr = (unsigned)(-sh);
            const unsigned long long y = shr64(m, rr) + (shr64(m, rr - 1u) & 1ull);
            x0 = (unsigned)y, x1 = (unsigned)(y >> 32), x2 = 0u, q = 0u;
        }
    }
    const unsigned neg = (unsigned)((int)hi >> 31), one = neg & 1u;
    unsigned x3;
    asm("{\n\t"
        "add.cc.u32 %0, %4, %8;\n\t"
        "addc.cc.u32 %1, %5, 0;\n\t"
        "addc.cc.u32 %2, %6, 0;\n\t"
        "addc.u32 %3, %7, 0;\n\t}"
        : "=r"(x0), "=r"(x1), "=r"(x2), "=r"(x3)
        : "r"(x0 ^ neg), "r"(x1 ^ neg), "r"(x2 ^ neg), "r"(neg), "r"(one));
    if (!ok) x0 = x1 = x2 = x3 = 0u;
    unsigned *l = t.limb + h;
    unsigned o = atomicAdd(l + q * kGSlots, x0);
    unsigned c = (o + x0) < o;
    unsigned x = q < 3u ? x1 + c : 0u;  // (no limb above the top one: its carry is the sign's)
    unsigned w = x < c;
    o = atomicAdd(l + min(q + 1u, 3u) * kGSlots, x);
    c = w | ((o + x) < o);
    x = q < 2u ? x2 + c : 0u;
    w = q < 2u && x < c;
    o = atomicAdd(l + min(q + 2u, 3u) * kGSlots, x);
    c = w | ((o + x) < o);
    if (__any_sync(kFull, q == 0u && ok)) {
        x = q < 1u ? x3 + c : 0u;
        atomicAdd(l + 3 * kGSlots, x);
    }
    return hit;
}

__host__ __device__ inline size_t gather_smem() {
    return size_t(kGSlots) * 20 + kGSlots / 8 + size_t(kGW) * sizeof(WarpArea) + sizeof(SourceBatch);
}

__device__ __forceinline__ unsigned row_salt(unsigned rl) { return (rl * 0x9E3779B1u) >> 13; }

__device__ __forceinline__ double read_sum(const unsigned *limb, unsigned h, int S) {
    return from_fixed(limb[h] | (unsigned long long)limb[h + kGSlots] << 32,
                      limb[h + 2 * kGSlots] | (unsigned long long)limb[h + 3 * kGSlots] << 32, S);
}

// Sums unit after unit (a group of light rows or a class of a heavy one): its doubles
// and ready elements into the table, sigma at the basis vectors' entries out of it,
// then the entries that can reach the truncation.  Bound by instruction issue (57 % of
// the slots at N_d = 2e4: about 260 warp instructions to place 32 elements, 90 to make
// them, 130 per 32 entries streamed) with 32 warps per SM, the most that 64 registers
// allow; DRAM is idle (2.5 GB read in 12 ms).  28 orbitals, sources of one to some
// thousand per string: 615e6 elements 12.4 ms (emit + merge 19), 3.07e9 53 to 61 ms
// (89), 3.07e10 510 to 730 ms (960, three passes); the lists and tables before it 4, 13
// and 100 to 145 ms (inside emit before).  Measured and left: 8192 slots in one CTA of
// 1024 threads (the same within 6 % either way), 2048 in four of 256 (up to 30 % slower:
// more classes), two or four rounds of elements at once (2 to 40 % slower), groups of
// four slots read at once (more instructions than the probes they save), a warp's probes
// run to the end (20 % slower: eight places for the slowest lane).
__global__ void __launch_bounds__(kGT, 1024 / kGT)
gather_kernel(const __grid_constant__ GatherArgs A) {
    extern __shared__ __align__(16) unsigned char gsm[];
    SourceBatch &sbatch = *reinterpret_cast<SourceBatch *>(gsm);
    WarpArea *areas = reinterpret_cast<WarpArea *>(gsm + sizeof(SourceBatch));
    unsigned *keys = reinterpret_cast<unsigned *>(areas + kGW);
    unsigned *limb = keys + kGSlots;
    unsigned *flag = limb + 4 * kGSlots;
    __shared__ __align__(16) GatherUnit s_units[2];
    __shared__ int s_over, s_raise, s_bin;
    __shared__ unsigned s_steps;
    const GatherShape &gs = A.gs;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const unsigned lt = (1u << lane) - 1u;
    const int bb = gs.bb;
    const unsigned bmask = gs.bmask;
    const bool f32 = A.gf != nullptr, screen = A.eps > 0.0;
    const unsigned long long eps_bits = abs_bits(A.eps);
    WarpArea &wa = areas[warp];
    for (int i = tid; i < kGSlots; i += kGT) {
        keys[i] = kNoKey;
        limb[i] = limb[i + kGSlots] = limb[i + 2 * kGSlots] = limb[i + 3 * kGSlots] = 0u;
    }
    for (int i = tid; i < kGSlots / 32; i += kGT) flag[i] = 0u;
    if (tid == 0) s_over = 0;
    TableView tab{keys, limb, 0u, A.fix_shift, &s_over};
    bool range_ok = true;
    double sq = 0.0;
    unsigned n_live = 0, n_nonzero = 0;
    unsigned long long n_read = 0;
    // the next unit is taken while this one runs: lanes 0..3 of warp 0 hold 16 bytes of it each
    uint4 next = make_uint4(0u, 0u, 0u, 0u);
    unsigned steps = 1u;
    unsigned long long streamed = 0ull, mark = ~0ull;
    auto take = [&]() {
        unsigned u = 0;
        if (lane == 0) u = atomicAdd(A.queue, 1u);
        u = __shfl_sync(kFull, u, 0);
        next = make_uint4(0u, 0u, 0u, 0u);  // (k1 = 0: no unit left)
        if (lane < 4 && u < A.n_units) next = __ldg(reinterpret_cast<const uint4 *>(A.units + u) + lane);
        // what other classes of its row had to split into (read once for the whole CTA)
        const unsigned k = __shfl_sync(kFull, next.x, 2), n_cls = __shfl_sync(kFull, next.y, 3);
        steps = n_cls > 1u ? *(volatile unsigned *)&A.split[k] : 1u;
        streamed = *(volatile unsigned long long *)A.out_n;
        mark = *(volatile unsigned long long *)A.mark;
    };
    if (warp == 0) take();
    for (unsigned turn = 0;; turn ^= 1u) {
        GatherUnit &s_unit = s_units[turn];  // (warps still in the unit before read the other one)
        if (warp == 0) {
            if (lane < 4) reinterpret_cast<uint4 *>(&s_unit)[lane] = next;
            if (lane == 0) {
                s_steps = steps;
                // raise the threshold once the stream has passed the mark (one CTA at a time)
                s_raise = streamed >= mark && atomicCAS(A.lock, 0, 1) == 0;
            }
        }
        __syncthreads();
        if (s_raise) {  // (the batch is idle here: its memory holds the partial sums)
            if (tid == 0) s_bin = -1;
            __syncthreads();
            raise_threshold<kGT>(A, tid, &s_bin, reinterpret_cast<unsigned long long *>(gsm));
        }
        const unsigned k0 = s_unit.k0, k1 = s_unit.k1;
        if (k1 == 0u) break;
        if (warp == 0) take();
        unsigned found = 0;  // entries of this unit in the warp's share of the table
        unsigned ka = k0, kz = k1, klen = k1 - k0;                              // rows and range of pi in the
        unsigned la = s_unit.lo, lz = s_unit.hi, llen = lz - la;                // table now; their step
        if (s_steps > 1u) llen = (llen + s_steps - 1u) / s_steps, lz = la + llen;
        unsigned long long rec0 = s_unit.rec0, rec1 = s_unit.rec1;
        unsigned ab0 = s_unit.ab0, ab1 = s_unit.ab1, src0 = s_unit.src0, src1 = s_unit.src1;
        for (;;) {
            // ---- sums
            unsigned n_try = 0;  // non-zero elements added in this attempt
            const bool part = lz - la <= bmask;  // a class: some of pi
            const unsigned n_ab = ab1 - ab0, n_src = A.nd2 ? src1 - src0 : 0u, n_rec = (unsigned)(rec1 - rec0);
            // the table holds every entry: few elements, or one row's range of at most its size
            const bool sure = lz - la <= (unsigned)kGSlots && kz - ka == 1u ? true
                              : n_rec + (unsigned long long)n_ab * A.sb + (unsigned long long)n_src * A.nd2 <= kGSlots;
            tab.max_probe = sure ? (unsigned)kGSlots : 64u;
            unsigned have = 0;  // elements in the warp's queue
            auto drain = [&](unsigned cnt) {  // the first cnt of them
                Element el;
                __syncwarp();
                el.ok = (unsigned)lane < cnt;
                el.key = el.ok ? wa.q.k[lane] : 0u;
                el.v = el.ok ? wa.q.v[lane] : 0.0;
                el.slot = (el.key & bmask) + row_salt(el.key >> bb);
                add_element<true>(tab, el, range_ok);
            };
            auto queue = [&](bool w, unsigned key, double v) {
                const unsigned bal = __ballot_sync(kFull, w);
                if (!bal) return;
                if (w) {
                    const unsigned p = have + __popc(bal & lt);
                    wa.q.k[p] = key, wa.q.v[p] = v;
                }
                have += __popc(bal);
                if (have < 32u) return;
                drain(32u);
                have -= 32u;
                __syncwarp();
                unsigned mk = 0u;
                double mv = 0.0;
                if ((unsigned)lane < have) mk = wa.q.k[32 + lane], mv = wa.q.v[32 + lane];
                __syncwarp();
                if ((unsigned)lane < have) wa.q.k[lane] = mk, wa.q.v[lane] = mv;
            };
            auto put = [&](const Element &el) {
                n_try += el.ok;
                queue(!add_element<false>(tab, el, range_ok), el.key, el.v);
            };
            // The doubles: own sources (beta-beta), then one-hop sources (opposite spin).  A
            // batch's segments are laid end to end and the warps take even shares of the
            // rounds of 32 elements.
            const unsigned n_all = n_src + n_ab;
            for (unsigned b0 = 0; b0 < n_all; b0 += kGT) {
                const unsigned s = b0 + tid;
                unsigned base = 0, len = 0, g = 0;
                uint4 e = make_uint4(0u, 0u, 0u, 0u);
                if (s < n_src) {
                    const unsigned id = __ldg(&A.s_b[src0 + s]);
                    const double c = __ldg(&A.s_c[src0 + s]);
                    e.z = (unsigned)__double2loint(c), e.w = (unsigned)__double2hiint(c);
                    g = id | __ldg(&A.s_kb[src0 + s]) >> bb << 25;
                    len = A.nd2;
                    if (part) {
                        const unsigned *iy = A.idx2 + (size_t)id * ((1 << gs.kb2) + 1);
                        base = __ldg(&iy[la >> (bb - gs.kb2)]);
                        len = __ldg(&iy[((lz - 1u) >> (bb - gs.kb2)) + 1u]) - base;
                    }
                } else if (s < n_all) {
                    e = __ldg(&A.ab[(size_t)ab0 + (s - n_src)]);
                    g = e.y;
                    base = e.x * A.sb, len = A.sb;
                    if (part) {
                        const unsigned short *ix = A.idx1 + (size_t)e.x * ((1 << gs.kb1) + 1);
                        const unsigned lo = __ldg(&ix[la >> (bb - gs.kb1)]);
                        len = __ldg(&ix[((lz - 1u) >> (bb - gs.kb1)) + 1u]) - lo;
                        base += lo;
                    }
                }
                unsigned inc = warp_scan(len, lane);
                if (lane == 31) sbatch.warp_tot[warp] = inc;
                __syncthreads();
                const unsigned wt = warp_scan(lane < kGW ? sbatch.warp_tot[lane] : 0u, lane);
                inc += warp > 0 ? __shfl_sync(kFull, wt, warp - 1) : 0u;
                const unsigned tot = __shfl_sync(kFull, wt, kGW - 1);
                sbatch.st[tid] = make_uint4(base - (inc - len), g, e.z, e.w);
                sbatch.start[tid] = inc - len;
                if (tid == 0) sbatch.start[kGT] = tot;
                __syncthreads();
                const unsigned n_own = n_src > b0 ? n_src - b0 : 0u;  // sources of the batch below it are own ones
                const unsigned rounds = (tot + 31u) >> 5, e1 = rounds * (warp + 1u) / kGW << 5;
                unsigned e0 = rounds * warp / kGW << 5, o = 0;
                const bool sparse = tot < 16u * kGT && tot < 16u * (n_all - b0);  // short segments
                for (bool search = true; e0 < e1; e0 += 32u, search = sparse) {
                    const unsigned at = min(e0 + lane, tot - 1u);
                    if (search) {
                        o = 0;
                        for (unsigned step = kGT / 2; step; step >>= 1)
                            if (sbatch.start[o + step] <= at) o += step;
                    } else {
                        while (sbatch.start[o + 1] <= at) ++o;
                    }
                    const uint4 p = sbatch.st[o];
                    const double c = __hiloint2double((int)p.w, (int)p.z);
                    Element el;
                    unsigned pi, rl;
                    if (o < n_own) {
                        const size_t t = (size_t)(p.y & 0x1ffffffu) * A.nd2 + (p.x + at);
                        pi = __ldg(&A.t2p[t]), rl = p.y >> 25;
                        el.v = __dmul_rn(__ldg(&A.t2e[t]), c);
                    } else {
                        const uint2 y = __ldg(&A.t1[p.x + at]);
                        const unsigned gi = (p.y & 0xffffffu) + (y.y & 0x7fffffffu);
                        const double gv = f32 ? (double)__ldg(&A.gf[gi]) : __ldg(&A.g[gi]);
                        pi = y.x, rl = (p.y >> 24) & 0x7fu;
                        el.v = __dmul_rn(flip_d(gv, (p.y ^ y.y) >> 31), c);
                    }
                    el.key = rl << bb | pi, el.slot = pi + row_salt(rl);
                    el.ok = e0 + lane < tot && abs_bits(el.v) >= A.min_bits && pi - la < lz - la;
                    put(el);
                    if (__any_sync(kFull, *tab.over)) break;
                }
                if (b0 + kGT < n_all) __syncthreads();  // (the next batch takes the place of this one)
            }
            // ready elements
            {
                const unsigned *rkey = s_unit.n_cls > 1u ? A.okey : A.rkey;
                const double *rval = s_unit.n_cls > 1u ? A.oval : A.rval;
                const unsigned rounds = (n_rec + 31u) >> 5, e1 = rounds * (kGW - warp) / kGW << 5;
                for (unsigned i = rounds * (kGW - 1 - warp) / kGW << 5; i < e1; i += 32u) {
                    Element el;
                    const unsigned long long r = rec0 + i + lane;
                    el.key = i + lane < n_rec ? __ldcs(&rkey[r]) : kNoKey;
                    el.v = 0.0;
                    if (el.key != kNoKey && (el.key & bmask) - la < lz - la) el.v = __ldcs(&rval[r]);
                    el.ok = abs_bits(el.v) >= A.min_bits;
                    el.slot = (el.key & bmask) + row_salt(el.key >> bb);
                    put(el);
                    if (__any_sync(kFull, *tab.over)) break;
                }
            }
            if (have) drain(have);
            __syncthreads();
            if (*tab.over) {  // too many distinct entries: clear, and half of the rows or of the range
                __syncthreads();
                for (int i = tid; i < kGSlots; i += kGT) {
                    keys[i] = kNoKey;
                    limb[i] = limb[i + kGSlots] = limb[i + 2 * kGSlots] = limb[i + 3 * kGSlots] = 0u;
                }
                if (kz - ka > 1u) {
                    klen = (kz - ka + 1u) / 2u;
                    kz = ka + klen;
                    rec1 = __ldg(&A.rec_off[kz]), ab1 = (unsigned)__ldg(&A.ab_off[kz]);
                    src1 = __ldg(&A.rp[__ldg(&A.act_row[kz - 1u]) + 1u]);
                } else {
                    llen = (lz - la + 1u) / 2u;
                    lz = la + llen;
                    // the row's other classes start with as many steps
                    if (tid == 0 && s_unit.n_cls > 1u) atomicMax(&A.split[k0], (s_unit.hi - s_unit.lo + llen - 1u) / llen);
                }
                if (tid == 0) s_over = 0;
                __syncthreads();
                continue;
            }
            n_read += n_try;
            const unsigned long long tau_bits = *(volatile unsigned long long *)A.tau_bits;  // (used below)
            // ---- sigma at the basis vectors' entries: one row: a warp per vector, its
            // lanes along the row's entries; several: a thread per (row, vector)
            {
                const bool one = kz - ka == 1u;
                const unsigned pairs = (kz - ka) * (unsigned)A.nvec;
                for (unsigned t = one ? (unsigned)warp : (unsigned)tid; t < pairs; t += one ? (unsigned)kGW : (unsigned)kGT) {
                    const unsigned k = ka + t / (unsigned)A.nvec, j = t % (unsigned)A.nvec;
                    const unsigned row = __ldg(&A.act_row[k]);
                    const unsigned long long rbase = (unsigned long long)row * A.cb;
                    const unsigned e1 = __ldg(&A.vrp[j][row + 1]), rl = k - k0;
                    for (unsigned e = __ldg(&A.vrp[j][row]) + (one ? lane : 0); e < e1; e += one ? 32 : 1) {
                        const unsigned pi = bperm(gs, (unsigned)(__ldg(&A.vrank[j][e]) - rbase));
                        if (pi - la >= lz - la) continue;
                        const unsigned key = (rl << bb) | pi;
                        unsigned h = (pi + row_salt(rl)) & (kGSlots - 1);
                        double sv = 0.0;
                        for (unsigned probe = 0; probe < (unsigned)kGSlots;) {
                            const unsigned c = keys[h];
                            if (c == key) {
                                sv = read_sum(limb, h, A.fix_shift);
                                if ((int)j == A.ja || (int)j == A.jb) atomicOr(&flag[h >> 5], 1u << (h & 31));
                                break;
                            }
                            if (c == kNoKey) break;
                            h = (h + ++probe) & (kGSlots - 1);
                        }
                        if (screen && abs_bits(sv) < eps_bits) sv = 0.0;  // screened entries count as absent
                        A.sigw[j][e] = sv;
                    }
                }
            }
            __syncthreads();
            // ---- entries with |u| >= tau leave (u = sigma off w_i, w_{i-1}); the table is
            // cleared.  Each warp lists the occupied slots of its share, then takes them
            // 32 at a time.
            {
                unsigned occ = 0;
                for (int h = warp * (kGSlots / kGW) + lane; h < (warp + 1) * (kGSlots / kGW); h += 32) {
                    const bool o = keys[h] != kNoKey;
                    const unsigned bal = __ballot_sync(kFull, o);
                    if (o) wa.list[occ + __popc(bal & lt)] = (unsigned short)h;
                    occ += __popc(bal);
                }
                __syncwarp();
                for (unsigned t0 = 0; t0 < occ; t0 += 32) {
                    unsigned key = 0u, hb = 0x80000000u | (unsigned)lane;
                    double v = 0.0;
                    bool w = false;
                    if (t0 + lane < occ) {
                        const unsigned h = wa.list[t0 + lane];
                        key = keys[h];
                        v = read_sum(limb, h, A.fix_shift);
                        const unsigned long long ab = abs_bits(v);
                        const bool live = !(screen && ab < eps_bits);
                        const bool nz = live && !((flag[h >> 5] >> (h & 31)) & 1u) && ab != 0ull;
                        n_live += live;
                        if (nz) {
                            ++n_nonzero;
                            sq = __fma_rn(v, v, sq);
                        }
                        w = A.all ? live : nz && !(ab < tau_bits);
                        keys[h] = kNoKey;
                        limb[h] = limb[h + kGSlots] = limb[h + 2 * kGSlots] = limb[h + 3 * kGSlots] = 0u;
                        if (w) hb = (unsigned)(ab >> kHistShift);
                    }
                    const unsigned bal = __ballot_sync(kFull, w);
                    if (bal) {
                        // histogram of the streamed entries (lanes sharing a bin add once)
                        if (!A.all) {
                            const unsigned peers = __match_any_sync(kFull, hb);
                            if (w && (peers & lt) == 0) atomicAdd(&A.hist[hb], (unsigned long long)__popc(peers));
                        }
                        unsigned long long base = 0;
                        if (lane == 0) base = atomicAdd(A.out_n, (unsigned long long)__popc(bal));
                        base = __shfl_sync(kFull, base, 0);
                        if (w) {
                            const unsigned long long pos = base + __popc(bal & lt);
                            if ((long long)pos < A.out_cap) {
                                A.out_key[pos] = (unsigned long long)__ldg(&A.act_row[k0 + (key >> bb)]) * A.cb +
                                                 bperm_inv(gs, key & bmask);
                                A.out_val[pos] = v;
                            } else {
                                atomicOr(A.status, 8);
                            }
                        }
                    }
                }
                __syncwarp();
                if (lane < kGSlots / kGW / 32) flag[warp * (kGSlots / kGW / 32) + lane] = 0u;
                found += occ;
            }
            // what a split left for later: the rest of the range, then of the rows
            if (lz < s_unit.hi) {
                la = lz, lz = min(s_unit.hi, la + llen);
            } else if (kz < k1) {
                la = s_unit.lo, lz = s_unit.hi;
                ka = kz, kz = min(k1, ka + klen);
                rec0 = rec1, ab0 = ab1;
                src0 = __ldg(&A.rp[__ldg(&A.act_row[ka])]), src1 = __ldg(&A.rp[__ldg(&A.act_row[kz - 1u]) + 1u]);
                rec1 = __ldg(&A.rec_off[kz]), ab1 = (unsigned)__ldg(&A.ab_off[kz]);
            } else {
                break;
            }
            __syncthreads();
        }
        // entries found in rows of this weight (bin 0: light rows): the next plan's estimate
        if (lane == 0 && found) atomicAdd(&A.seen[2 * s_unit.bin + 1], (unsigned long long)found);
        if (tid == 0) {
            const unsigned long long w = (s_unit.rec1 - s_unit.rec0) + (unsigned long long)(s_unit.ab1 - s_unit.ab0) * A.sb +
                                         (unsigned long long)(s_unit.src1 - s_unit.src0) * A.nd2;
            atomicAdd(&A.seen[2 * s_unit.bin], w / s_unit.n_cls);
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        sq += __shfl_xor_sync(kFull, sq, o);
        n_live += __shfl_xor_sync(kFull, n_live, o);
        n_nonzero += __shfl_xor_sync(kFull, n_nonzero, o);
        n_read += __shfl_xor_sync(kFull, n_read, o);
    }
    if (lane == 0) {
        atomicAdd(A.sumsq, sq);
        atomicAdd(A.n_live, (unsigned long long)n_live);
        atomicAdd(A.n_nonzero, (unsigned long long)n_nonzero);
        atomicAdd(A.n_read, n_read);
    }
    if (!range_ok) atomicOr(A.status, 32);
}

unsigned grid_for(unsigned long long work, unsigned per) {
    const unsigned long long g = (work + per - 1) / per;
    return (unsigned)(g < 1 ? 1 : g > 4096 ? 4096 : g);
}

unsigned inverse_odd(unsigned m) {  // modulo 2^32, Newton's iteration
    unsigned x = m;
    for (int i = 0; i < 5; ++i) x *= 2u - m * x;
    return x;
}

}  // namespace

namespace {
RowPlan row_plan(const SysDev &d, const GatherShape &p, const GatherBufs &b, const RowPlanArgs &ra) {
    return RowPlan{ra.half, ra.fill, (double)d.cb, p.bb, b.seen};
}
}  // namespace

bool gather_shape(const SysDev &d, GatherShape *p) {
    auto C = [](int n, int k) {
        double r = 1.0;
        for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;
        return k < 0 || k > n ? 0.0 : r;
    };
    if (d.na > kMaxE || d.nb > kMaxE || d.ca > (1ull << 26) || d.cb > (1ull << 26)) return false;
    const double k1 = C(d.n, d.na - 1), k2 = C(d.n, d.na - 2);
    if (k1 > 1e8 || k2 > 1e8) return false;
    int bb = 1;
    while ((1ull << bb) < d.cb) ++bb;
    p->bb = bb;
    p->bs = (bb + 1) / 2;
    p->bmask = (1u << bb) - 1u;
    p->m1 = 0x9E3779B1u, p->m2 = 0x85EBCA6Bu;
    p->i1 = inverse_odd(p->m1), p->i2 = inverse_odd(p->m2);
    p->kb1 = std::min(bb, 7);
    p->kb2 = std::min(bb, 9);
    p->nd2 = d.po_b * d.pv_b;
    p->nk1 = (unsigned)std::llround(k1);
    p->nk2 = (unsigned)std::llround(k2);
    p->npair = (unsigned)(d.n * (d.n - 1) / 2);
    return d.sb < 65536;
}

namespace {
// in the order of GatherCounts: one copy to the host instead of five
__global__ void pack_counts_kernel(const unsigned long long *a, const unsigned long long *b, const unsigned long long *c,
                                   const unsigned long long *d, const unsigned long long *e, unsigned long long *out) {
    const unsigned long long *const p[5] = {a, b, c, d, e};
    if (threadIdx.x == 0)
        for (int k = 0; k < 5; ++k) out[k] = *p[k];
}

// Memory one buffer hands out in 256-byte pieces (no base: sizes only)
struct Arena {
    char *base = nullptr;
    size_t off = 0;
    template <class T>
    T *take(size_t n) {
        T *p = base ? reinterpret_cast<T *>(base + off) : nullptr;
        off += (n * sizeof(T) + 255) & ~size_t(255);
        return p;
    }
};
}  // namespace

size_t gather_place_sources(char *base, GatherBufs &b, const SysDev &d, const GatherShape &p, long long n) {
    Arena a{base};
    const size_t ca = size_t(d.ca), cb = size_t(d.cb);
    b.words = a.take<unsigned long long>(16);
    b.skey = a.take<unsigned long long>(n);
    b.sc = a.take<double>(n);
    b.sort_ws = a.take<char>(p.bb > kGLog ? sort_pairs_bytes(n) : 0);
    b.scan_ws = a.take<char>(4 * scan_ws_bytes((long long)std::max({ca, cb, size_t(p.nk1), size_t(p.nk2)}) + 1));
    b.bflag = a.take<unsigned>(cb);
    b.bid = a.take<unsigned long long>(cb + 1);
    b.s_pi = a.take<unsigned>(n);
    b.s_b = a.take<unsigned>(n);
    b.s_kb = a.take<unsigned>(n);
    b.s_diag = a.take<double>(n);
    b.cnt1 = a.take<unsigned>(size_t(p.nk1) + p.nk2);
    b.cnt2 = b.cnt1 + p.nk1;
    b.off1 = a.take<unsigned long long>(size_t(p.nk1) + 1);
    b.off2 = a.take<unsigned long long>(size_t(p.nk2) + 1);
    b.s1 = a.take<unsigned>(ca);
    b.s2 = a.take<unsigned>(ca);
    b.act = a.take<unsigned>(ca);
    b.apos = a.take<unsigned long long>(ca + 1);
    b.act_row = a.take<unsigned>(ca);
    b.act_str = a.take<unsigned long long>(ca);
    b.wpre = a.take<unsigned long long>(ca + 1);
    b.aw = a.take<unsigned long long>(3 * ca);
    b.nrec = reinterpret_cast<unsigned *>(b.aw + ca), b.nab = b.nrec + ca, b.np = b.nab + ca, b.nu = b.np + ca;
    b.uoff = a.take<unsigned long long>(ca + 1);
    b.poff = a.take<unsigned long long>(ca + 1);
    b.rec_off = a.take<unsigned long long>(ca + 1);
    b.ab_off = a.take<unsigned long long>(ca + 1);
    return a.off;
}

size_t gather_place_tables(char *base, GatherBufs &b, const SysDev &d, const GatherShape &p, size_t nd, long long n) {
    Arena a{base};
    b.bstr = a.take<unsigned long long>(nd);
    b.t1 = a.take<uint2>(nd * d.sb);
    b.idx1 = a.take<unsigned short>(nd * ((1 << p.kb1) + 1));
    b.t2p = a.take<unsigned>(nd * p.nd2);
    b.t2e = a.take<double>(nd * p.nd2);
    b.idx2 = a.take<unsigned>(nd * ((1 << p.kb2) + 1));
    b.ent1 = a.take<uint4>(size_t(n) * d.na);
    b.ent2 = a.take<uint4>(size_t(n) * d.po_a);
    return a.off;
}

size_t gather_place_lists(char *base, GatherBufs &b, const GatherShape &p, const GatherCounts &n) {
    Arena a{base};
    b.units = a.take<GatherUnit>(n.units);
    b.part_k = a.take<unsigned>(n.parts);
    b.cursor = a.take<unsigned>(2 * n.act);
    b.split = b.cursor + n.act;
    b.split_rows = a.take<unsigned>(n.act);
    b.rkey = a.take<unsigned>(n.rec);
    b.rval = a.take<double>(n.rec);
    const size_t n_ord = p.bb > kGLog ? n.rec : 0;
    b.okey = a.take<unsigned>(n_ord);
    b.oval = a.take<double>(n_ord);
    b.ab = a.take<uint4>(n.ab);
    return a.off;
}

// 32-bit positions in the singles' table, the lists and one row's records (the sources listed
// under its substrings, those one hop away, the diagonal and beta singles of its own, which are
// as many as there are beta strings at most), 25 bits for a beta string's number
bool gather_numbers(const SysDev &d, long long n, unsigned long long nd) {
    constexpr double k32 = 4294967296.0;
    return n < (1ll << 31) && nd < (1ull << 25) && (double)nd * std::max(d.sb, 1) < k32 &&
           (double)n * std::max(d.po_a, d.na) < k32 &&
           (double)n * (d.po_a + 1.0) + std::min((double)n, (double)nd) * (d.sb + 1.0) < k32;
}

// A chip that a few units leave idle: 3.5 ns per element of a unit (30 rows of 9e5 elements: 3.8 ms,
// buckets 3.1).
bool enough_units(double units, double elements) { return units >= 152.0 || elements <= 5e5 * units; }

// Sigma by target rows against the buckets (330 systems of 8 to 64 orbitals with random and with
// level-like vectors, 10 to 3e5 determinants, both ways timed).  Besides its elements, 16 ps each
// against 31 to 39, the row path pays for
//  * every row of the space, 70 + 3.65 ps per substring of its string (the buckets: 62), and 0.25 ns
//    per row that a source reaches; it saves about 1.2 ms of the buckets' launches and read-backs.
//    28 orbitals with 12 + 12 electrons (3e7 rows): 30 determinants 11.9 ms by rows, 3.9 by buckets,
//    1e4 35 and 24, 1e5 100 and 98; with 7 + 7 (1.2e6 rows) rows win from one determinant on (0.8 and 1.9).
//    Without opposite-spin elements (no singles of one spin) all are records or own doubles, and
//    the buckets win from 1e7 elements on (28 orbitals, 7 electrons: 1.70 ms and 2.58).
//    Beside other solvers of a batch their work hides most of these, all of them with one spin.  Six
//    steps of batches of 24 orbitals: 8 systems of 7 + 0 electrons, 500 determinants 17.7 ms by rows,
//    10.3 by buckets; 4 of 10 + 10, 50 determinants 18.0 and 13.9; but 8 of 8 + 8, 8 determinants 12.5
//    and 17.3, 16 of 7 + 7, 300 determinants 34.8 and 47.2.
bool gather_pays(const SysDev &d, long long n, bool beside) {
    const double ca = (double)d.ca, subs = d.na + d.po_a, hops = 1.0 + d.sa + (double)d.po_a * d.pv_a;
    const double elements = (double)n * (double)(d.n_conn + 1);
    if ((d.sa == 0 || d.sb == 0) && (beside || elements > 1e7)) return false;
    if (d.cb <= kGSlots && !enough_units(ca, elements)) return false;  // (no row has classes)
    return ca * (8.0 + 3.65 * subs) + 250.0 * std::min(ca, n * hops) <= (beside ? 0.3e9 : 1.2e9) + 4.0 * elements;
}

//  * every class of a heavy row that a source is read for, 12 to 44 ps: where few rows hold most
//    sources, classes outnumber the excitations of a string and most visits find nothing.  Up to
//    0.65 visits per element.  Truncated Lanczos vectors of 28 orbitals, 7 + 7 electrons, 1e5 to 1e6
//    determinants 0.06 to 0.38, rows 0.68 to 0.81 of the buckets' time (1e6: 680 to 770 ms and 980);
//    22 orbitals, 3 + 9 0.43 to 0.53, 0.68; 28 orbitals, 3 + 8 0.96 to 1.5, 1.7 to 2.2; 2 + 9 1.2 to
//    2.2, 2.4 to 3.8; scattered vectors of 29 orbitals, 1 + 10 electrons 3.1 to 4.4, 7 to 11.
bool gather_pays(const SysDev &d, long long n, const GatherCounts &c) {
    const double elements = (double)n * (double)(d.n_conn + 1);
    return (double)c.visits <= 0.65 * elements && enough_units((double)c.units, elements);
}

// The standalone sigma's hash table has no preparation, but a warp per source (0.13 us an element in
// turn: 1.9 ms for 30 sources of 7876, by rows 0.5) and slots to clear and read (32 bytes each).  It
// is left to
//  * few elements a source and few slots: 28 orbitals, 1 + 1 electrons, 30 determinants 0.22 ms, by
//    rows 0.29; 20 orbitals, 5 electrons of one spin, 85 determinants 0.28 and 0.39; but 12
//    orbitals, 6 + 6 (1817 excitations), 20 determinants 0.50 and 0.39;
//  * elements of one spin alone (records or own doubles, no table of singles to share), until the
//    slots cost more: 28 orbitals, 7 electrons, 872 determinants (2^23 slots) 0.98 and 2.13, 8636
//    (2^22) 1.41 and 1.84, but (2^26) 4.03 and 3.48; 24 orbitals, 12 electrons, 300 determinants
//    (2^22) 1.02 and 0.77, 2000 1.28 and 1.80.
bool gather_beats_table(const SysDev &d, long long n, unsigned long long slots) {
    if (d.n_conn <= 1150 && slots <= 1ull << 20) return false;
    return (d.sa > 0 && d.sb > 0) || slots > 1ull << 23 || (double)n * (double)(d.n_conn + 1) < 2e6;
}

// and to heavy rows whose classes visit sources more than twice as often as there are elements (the
// plan, about 0.7 ms, is made for nothing then).  28 orbitals, 1 + 9 electrons: 1.3 visits an element
// (5000 determinants) 8.9 ms by rows, 12.4 by the table, 2.3 (1e4) 20.9 and 20.1, 3.6 (2e4) 52 and 34; 29
// orbitals, 1 + 10: 2.1 (8000) 21.4 and 22.1, 3.1 (25000) 115 and 57.
bool gather_beats_table(const SysDev &d, long long n, const GatherCounts &c) {
    return (double)c.visits <= 2.2 * (double)n * (double)(d.n_conn + 1);
}

// What the lists take at least, whatever the rows: a source is listed under C(n_alpha, 2) substrings
// of C(n - n_alpha + 2, 2) rows each, is one hop away from s_a rows, and has its own records.
size_t gather_lists_least(const SysDev &d, const GatherShape &p, long long n) {
    const double rows2 = 0.5 * (d.n - d.na + 2) * (d.n - d.na + 1);
    const double rec = (double)n * ((d.ss_any ? d.po_a * rows2 : 0.0) + d.sa + d.sb + 1.0);
    return (size_t)(rec * (p.bb > kGLog ? 24.0 : 12.0) + (d.ab_any ? 16.0 * (double)n * d.sa : 0.0));
}

RowPlanArgs row_plan_args(const SysDev &d, const GatherShape &p, long long n) {
    RowPlanArgs ra{};
    // a warp makes 128 to 1024 list items: as many warps as the chip holds twice, where there are enough
    const double items = (double)n * (1.0 + d.sb + 2.0 * d.sa + (d.ss_any ? (double)d.po_a * (d.pv_a + d.sa + d.po_a) : 0.0));
    ra.part_work = std::min(1024u, std::max(128u, (unsigned)std::min(items / 10000.0, 4096.0) & ~31u));
    // light rows repeat entries about 1.45 times (1.3 to 2): a group fills about 0.55 of its table
    ra.half = (unsigned long long)(0.55 * 1.45 * kGSlots);
    ra.fill = 0.65 * kGSlots;
    // at most 120 rows in a group (7 bits), and fewer than its key bits can number
    ra.w_fixed = std::max(32u, (unsigned)(2 * ra.half / std::min(120ull, (1ull << (32 - p.bb)) - 2ull) + 1));
    return ra;
}

cudaError_t gather_counts(const SysDev &d, const GatherBufs &b, GatherCounts *n, cudaStream_t st) {
    static_assert(sizeof(GatherCounts) == 48, "five words behind words[3], then the visits");
    count_launch();
    pack_counts_kernel<<<1, 32, 0, st>>>(b.apos + d.ca, b.uoff + d.ca, b.poff + d.ca, b.rec_off + d.ca, b.ab_off + d.ca,
                                         b.words + 3);
    const cudaError_t e = cudaMemcpyAsync(n, b.words + 3, sizeof(*n), cudaMemcpyDeviceToHost, st);
    return e == cudaSuccess ? cudaStreamSynchronize(st) : e;
}

void gather_inputs(GatherArgs &A, const SysDev &d, const GatherShape &p, const GatherBufs &b, const GatherCounts &n,
                   const unsigned *rp) {
    A.gs = p, A.cb = d.cb, A.g = d.g, A.gf = d.gf;
    A.sb = (unsigned)d.sb, A.nd2 = d.ss_any ? (unsigned)p.nd2 : 0u;
    A.units = b.units, A.n_units = (unsigned)n.units, A.act_row = b.act_row;
    A.rkey = b.rkey, A.rval = b.rval, A.okey = b.okey, A.oval = b.oval, A.split = b.split, A.ab = b.ab;
    A.rec_off = b.rec_off, A.ab_off = b.ab_off, A.rp = rp;
    A.s_b = b.s_b, A.s_kb = b.s_kb, A.s_c = b.sc;
    A.t1 = b.t1, A.idx1 = b.idx1, A.t2p = b.t2p, A.t2e = b.t2e, A.idx2 = b.idx2;
    A.seen = b.seen;
    A.min_bits = 1ull;
}

cudaError_t launch_pair_integrals(const SysDev &d, double *W, cudaStream_t st) {
    const int np = d.n * (d.n - 1) / 2;
    if (np <= 0) return cudaSuccess;
    count_launch();
    pair_integrals_kernel<<<grid_for((unsigned long long)np * np, 256), 256, 0, st>>>(d, np, W);
    return cudaGetLastError();
}

cudaError_t launch_hop_integrals(const SysDev &d, double *sg, float *sgf, cudaStream_t st) {
    count_launch();
    hop_integrals_kernel<<<grid_for((long long)d.n * d.n * d.n, 256), 256, 0, st>>>(d, sg, sgf);
    return cudaGetLastError();
}

cudaError_t launch_row_pointers(const SysDev &d, const unsigned long long *rank, long long n, unsigned *rp,
                                cudaStream_t st) {
    count_launch();
    row_pointers_kernel<<<grid_for(d.ca + 1, 256), 256, 0, st>>>(rank, n, d.ca, d.cb, rp);
    return cudaGetLastError();
}

cudaError_t gather_sources(const SysDev &d, const GatherShape &p, const unsigned long long *rank, const double *coef,
                           long long n, const GatherBufs &b, cudaStream_t st) {
    cudaError_t e = cudaMemsetAsync(b.bflag, 0, size_t(d.cb) * 4, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(b.words, 0, 128, st);
    if (e != cudaSuccess) return e;
    count_launch();
    sources_kernel<<<grid_for(n, 256), 256, 0, st>>>(p, rank, coef, n, d.cb, b.skey, b.sc, b.bflag, b.words, b.seen);
    e = exclusive_scan(static_cast<const unsigned *>(b.bflag), (long long)d.cb, b.bid, b.scan_ws, st);
    if (e != cudaSuccess) return e;
    if (p.bb <= kGLog) return cudaSuccess;  // no row is split: any order within a run will do
    // runs in the order of pi (the classes of a split row are contiguous in each run)
    int bits = p.bb;
    while ((1ull << (bits - p.bb)) < d.ca) ++bits;
    e = cudaMemcpyAsync(b.words + 1, &n, 8, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    return sort_pairs(b.skey, b.sc, n, b.words + 1, bits, b.sort_ws, st);
}

cudaError_t gather_tables(const SysDev &d, const GatherShape &p, long long n, unsigned nd, const double *W,
                          const unsigned *rp, const GatherBufs &b, const RowPlanArgs &ra, bool fresh, cudaStream_t st) {
    const size_t bts = size_t(d.n + 1) * d.ks * 8;
    count_launch();
    const size_t fields_smem = bts + (d.n <= kStageN ? size_t(2 * d.n + 1) * d.n * 8 : 0);
    source_fields_kernel<<<grid_for(n, 128), 128, fields_smem, st>>>(d, p, b.skey, n, b.bid, b.s_pi, b.s_b, b.s_diag, b.bstr);
    const bool keep = beta_smem(d, true) <= 100 * 1024;
    const size_t smem = beta_smem(d, keep);
    auto tables = keep ? beta_tables_kernel<true> : beta_tables_kernel<false>;
    cudaError_t e = allow_max_smem(tables, smem);
    if (e != cudaSuccess) return e;
    count_launch();
    tables<<<std::min(nd, 152u * 64u), 256, smem, st>>>(d, p, b.bstr, nd, W, b.t1, b.idx1, b.t2p, b.t2e, b.idx2);
    e = cudaMemsetAsync(b.cnt1, 0, (size_t(p.nk1) + p.nk2) * 4, st);  // cnt1 | cnt2
    if (e != cudaSuccess) return e;
    const dim3 sub_grid(grid_for(n, 128), (unsigned)d.na);
    if (d.na) count_launch(), substring_lists_kernel<<<sub_grid, 128, bts, st>>>(d, p, b.skey, b.sc, b.s_b, n, b.cnt1, b.cnt2, nullptr,
                                                              nullptr, nullptr, nullptr);
    e = exclusive_scan(static_cast<const unsigned *>(b.cnt1), p.nk1, b.off1, b.scan_ws, st);
    if (e == cudaSuccess) e = exclusive_scan(static_cast<const unsigned *>(b.cnt2), p.nk2, b.off2, b.scan_ws, st);
    if (e != cudaSuccess) return e;
    if (d.na) count_launch(), substring_lists_kernel<<<sub_grid, 128, bts, st>>>(d, p, b.skey, b.sc, b.s_b, n, b.cnt1, b.cnt2, b.off1,
                                                              b.off2, b.ent1, b.ent2);
    const unsigned long long chunks = (d.ca + kRowChunk - 1) / kRowChunk;
    count_launch();
    row_sources_kernel<<<grid_for(chunks, 128), 128, bts, st>>>(d, rp, b.off1, b.off2, b.s1, b.s2, b.act);
    e = exclusive_scan(static_cast<const unsigned *>(b.act), (long long)d.ca, b.apos, b.scan_ws, st);
    // (past the last active row: weight 0, no unit, no part)
    if (e == cudaSuccess) e = cudaMemsetAsync(b.aw, 0, size_t(d.ca) * 24, st);  // aw | nrec | nab | np | nu
    if (e != cudaSuccess) return e;
    count_launch();
    active_rows_kernel<<<grid_for(chunks, 128), 128, bts, st>>>(d, p, rp, b.s1, b.s2, b.act, b.apos, ra.w_fixed, ra.part_work,
                                                               b.act_row, b.act_str, b.aw, b.nrec, b.nab, b.np);
    e = exclusive_scan(static_cast<const unsigned long long *>(b.aw), (long long)d.ca, b.wpre, b.scan_ws, st);
    if (e != cudaSuccess) return e;
    // (drawn at random, n sources have cb (1 - exp(-n / cb)) beta strings; a vector of many more
    // than cb has them all, whatever it is)
    const double cb = (double)d.cb, drawn = -cb * std::expm1(-(double)n / cb);
    const bool scattered = fresh && (double)nd > 0.75 * drawn && (double)n < 1.5 * cb;
    count_launch();
    row_units_kernel<<<grid_for(d.ca, 256), 256, 0, st>>>(row_plan(d, p, b, ra), b.aw, b.wpre, b.apos + d.ca, b.nab,
                                                          b.act_row, rp, b.nu, scattered, b.words + 8);
    unsigned long long *const out[4] = {b.rec_off, b.ab_off, b.poff, b.uoff};  // nrec | nab | np | nu
    return exclusive_scan4(b.nrec, (long long)d.ca, out, b.scan_ws, st);
}

cudaError_t gather_lists(const SysDev &d, const GatherShape &p, unsigned long long n_act, unsigned long long n_parts,
                         const double *W, const unsigned *rp, const GatherBufs &b, const RowPlanArgs &ra,
                         cudaStream_t st) {
    count_launch();
    write_units_kernel<<<grid_for(n_act, 256), 256, 0, st>>>(row_plan(d, p, b, ra), b.aw, b.wpre, n_act, b.nu, b.np,
                                                            b.uoff, b.poff, b.rec_off, b.ab_off, b.act_row, rp, b.units,
                                                            b.part_k, b.split_rows, b.words + 2);
    cudaError_t e = cudaMemsetAsync(b.cursor, 0, size_t(n_act) * 8, st);  // cursor | split
    if (e != cudaSuccess) return e;
    ListArgs A{};
    A.d = d, A.gs = p, A.W = W;
    A.act_row = b.act_row, A.act_str = b.act_str, A.part_k = b.part_k, A.n_parts = (unsigned)n_parts;
    A.nu = b.nu, A.poff = b.poff, A.uoff = b.uoff, A.rec_off = b.rec_off, A.ab_off = b.ab_off;
    A.units = b.units, A.s1 = b.s1, A.s2 = b.s2, A.rp = rp;
    A.off1 = b.off1, A.off2 = b.off2, A.ent1 = b.ent1, A.ent2 = b.ent2;
    A.s_pi = b.s_pi, A.s_b = b.s_b, A.s_c = b.sc, A.s_diag = b.s_diag, A.bstr = b.bstr, A.t1 = b.t1;
    A.cursor = b.cursor, A.rkey = b.rkey, A.rval = b.rval, A.ab = b.ab, A.s_kb = b.s_kb;
    const size_t bts = size_t(d.n + 1) * d.ks * 8;
    count_launch();
    row_lists_kernel<<<(unsigned)std::min<unsigned long long>((n_parts + 7) / 8, 152ull * 8 * 16), kLT, bts, st>>>(A);
    if (p.bb <= kGLog) return cudaGetLastError();  // (no row has classes)
    count_launch();
    class_order_kernel<<<152 * 4, 512, 0, st>>>(p, b.split_rows, b.words + 2, b.nu, b.uoff, b.rec_off, b.rkey, b.rval,
                                                b.okey, b.oval, b.units);
    return cudaGetLastError();
}

cudaError_t launch_gather(const GatherArgs &A, cudaStream_t st) {
    const size_t smem = gather_smem();
    cudaError_t e = allow_max_smem(gather_kernel, smem);
    if (e != cudaSuccess) return e;
    int per_sm = 0, dev = 0, sms = 1;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, gather_kernel, kGT, smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    e = cudaMemsetAsync(A.queue, 0, 4, st);
    if (e != cudaSuccess) return e;
    const unsigned grid = std::min<unsigned>((unsigned)(sms * per_sm), std::max(A.n_units, 1u));
    count_launch();
    gather_kernel<<<grid, kGT, smem, st>>>(A);
    return cudaGetLastError();
}

}  // namespace sfci
