// One- and two-particle density matrices of a sparse vector, produced by the
// same excitation generator as sigma (sfci_emit.cu): for every determinant D of
// psi and every D' in {D} and the single and double excitations of D, the
// coefficient c_D' is looked up in a hash table built from psi; each hit adds
// c_D' c_D <D'| a+_p a+_r a_s a_q |D> into the spin-summed
//   gamma[p,q]      = sum_s   <psi| a+_ps a_qs |psi>
//   Gamma[p,q,r,s]  = sum_st  <psi| a+_ps a+_rt a_st a_qs |psi>
// (not normalised).  The operator strings that connect D to D' are:
//   D' = D:        n_ps n_rt for distinct spin orbitals (p,s) != (r,t), minus the
//                  exchange n_ps n_rs (same spin) on Gamma[p,r,r,p];
//   single i->a:   gamma[a,i]; Gamma[a,i,k,k], Gamma[k,k,a,i] for every other
//                  occupied k, minus Gamma[a,k,k,i], Gamma[k,i,a,k] for k of the
//                  hop's spin;
//   double:        Gamma[a,i,b,j] + Gamma[b,j,a,i], and for same spin
//                  - Gamma[a,j,b,i] - Gamma[b,i,a,j]
// with the sign of the excitation (hop 1 then hop 2, as in sigma).  These give
// E = e_core <psi|psi> + sum h gamma + 1/2 sum (pq|rs) Gamma = <psi|H|psi>,
// so dE/dh = gamma / <psi|psi> and dE/d(pq|rs) = Gamma / (2 <psi|psi>) for a
// fixed psi.
//
// Two ways to find the pairs (D, D') that are both in psi:
//  * by rows (rdm_rows_kernel; a row: the determinants of one alpha string).
//    Each unordered pair is met once and adds to one of its images; a last pass
//    sums Gamma over the images (p,q,r,s), (r,s,p,q), (q,p,s,r), (s,r,q,p).
//  * by lookups (rdm_kernel): every excitation of every determinant, in a global
//    hash table; for vectors and systems outside the limits of the former.
#include <algorithm>
#include <type_traits>

#include "sfci_internal.cuh"

namespace sfci {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

__host__ __device__ inline size_t al16(size_t x) { return (x + 15) & ~size_t(15); }

__host__ __device__ inline size_t rdm_block_smem(const SysDev &d) {
    return al16(size_t(d.n + 1) * d.ks * 8) + al16(size_t(d.n_pairs) * 2);
}

__host__ __device__ inline size_t rdm_warp_smem(const SysDev &d) {
    return al16(size_t(d.sa + d.sb) * 12 + 256);
}

__device__ __forceinline__ void acc(double *a, size_t i, double v) { atomicAdd(a + i, v); }

__global__ void __launch_bounds__(kThreads)
rdm_kernel(const SysDev d, const unsigned long long *__restrict__ rank,
           const double *__restrict__ coef, long long m, Table psi, double *__restrict__ g1,
           double *__restrict__ g2) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int n = d.n, ks = d.ks;
    unsigned long long *bt = reinterpret_cast<unsigned long long *>(sm);
    unsigned char *pairs = sm + al16(size_t(n + 1) * ks * 8);
    for (int i = threadIdx.x; i < (n + 1) * ks; i += blockDim.x) bt[i] = d.binom[i];
    for (int i = threadIdx.x; i < 2 * d.n_pairs; i += blockDim.x) pairs[i] = d.pairs[i];
    __syncthreads();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char *wb = sm + rdm_block_smem(d) + size_t(warp) * rdm_warp_smem(d);
    unsigned long long *rankA1 = reinterpret_cast<unsigned long long *>(wb);
    unsigned long long *rankB1 = rankA1 + d.sa;
    unsigned *hopA = reinterpret_cast<unsigned *>(rankB1 + d.sb);  // i | a << 8 | sign << 16
    unsigned *hopB = hopA + d.sa;
    unsigned char *occA = reinterpret_cast<unsigned char *>(hopB + d.sb);
    unsigned char *virA = occA + 64, *occB = occA + 128, *virB = occA + 192;
    const unsigned char *pOA = pairs + 2 * d.pair_off[0], *pVA = pairs + 2 * d.pair_off[1];
    const unsigned char *pOB = pairs + 2 * d.pair_off[2], *pVB = pairs + 2 * d.pair_off[3];
    const unsigned long long cb = d.cb;
    const size_t N1 = size_t(n), N2 = N1 * n, N3 = N2 * n;
#define G2(p, q, r, s) (size_t(p) * N3 + size_t(q) * N2 + size_t(r) * N1 + size_t(s))

    const long long gw = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long s = gw; s < m; s += nw) {
        const unsigned long long r = rank[s];
        const double c = coef[s];
        const unsigned long long hA = r / cb, hB = r - hA * cb;
        const unsigned long long alpha = string_unrank_warp(hA, n, d.na, bt, ks);
        const unsigned long long beta = string_unrank_warp(hB, n, d.nb, bt, ks);
        build_lists(alpha, beta, n, occA, virA, occB, virB);
        __syncwarp();
        for (int x = lane; x < d.sa; x += 32) {
            const int io = x / d.va, iv = x - io * d.va;
            const int i = occA[io], a = virA[iv];
            rankA1[x] = string_rank(alpha ^ (1ull << i) ^ (1ull << a), bt, ks);
            hopA[x] = unsigned(i) | (unsigned(a) << 8) | (unsigned(parity64(alpha & between_mask(i, a))) << 16);
        }
        for (int y = lane; y < d.sb; y += 32) {
            const int jo = y / d.vb, jv = y - jo * d.vb;
            const int j = occB[jo], b = virB[jv];
            rankB1[y] = string_rank(beta ^ (1ull << j) ^ (1ull << b), bt, ks);
            hopB[y] = unsigned(j) | (unsigned(b) << 8) | (unsigned(parity64(beta & between_mask(j, b))) << 16);
        }
        __syncwarp();
        if (c == 0.0) continue;
        // D' = D
        {
            const double v = c * c;
            const int NE = d.na + d.nb;
            for (int k = lane; k < NE; k += 32) {
                const int p = k < d.na ? occA[k] : occB[k - d.na];
                acc(g1, size_t(p) * n + p, v);
            }
            for (int e = lane; e < NE * NE; e += 32) {
                const int k = e / NE, l = e - k * NE;
                if (k == l) continue;
                const int p = k < d.na ? occA[k] : occB[k - d.na];
                const int q = l < d.na ? occA[l] : occB[l - d.na];
                acc(g2, G2(p, p, q, q), v);
                if ((k < d.na) == (l < d.na)) acc(g2, G2(p, q, q, p), -v);
            }
        }
        // singles
        for (int spin = 0; spin < 2; ++spin) {
            const int ns = spin ? d.sb : d.sa;
            const unsigned long long *rk = spin ? rankB1 : rankA1;
            const unsigned *hop = spin ? hopB : hopA;
            const unsigned char *same = spin ? occB : occA, *other = spin ? occA : occB;
            const int nsame = spin ? d.nb : d.na, nother = spin ? d.na : d.nb;
            for (int x = lane; x < ns; x += 32) {
                const unsigned long long tg = spin ? hA * cb + rk[x] : rk[x] * cb + hB;
                const long long f = table_find(psi, tg);
                if (f < 0) continue;
                const unsigned hp = hop[x];
                const int i = hp & 0xff, a = (hp >> 8) & 0xff;
                double v = __ldcg(&psi.slots[f].val) * c;
                if (hp >> 16) v = -v;
                acc(g1, size_t(a) * n + i, v);
                for (int q = 0; q < nsame; ++q) {
                    const int k = same[q];
                    if (k == i) continue;
                    acc(g2, G2(a, i, k, k), v);
                    acc(g2, G2(k, k, a, i), v);
                    acc(g2, G2(a, k, k, i), -v);
                    acc(g2, G2(k, i, a, k), -v);
                }
                for (int q = 0; q < nother; ++q) {
                    const int k = other[q];
                    acc(g2, G2(a, i, k, k), v);
                    acc(g2, G2(k, k, a, i), v);
                }
            }
        }
        // same-spin doubles
        for (int spin = 0; spin < 2; ++spin) {
            const unsigned long long str = spin ? beta : alpha;
            const unsigned char *occ = spin ? occB : occA, *vir = spin ? virB : virA;
            const unsigned char *po = spin ? pOB : pOA, *pv = spin ? pVB : pVA;
            const int npo = spin ? d.po_b : d.po_a, npv = spin ? d.pv_b : d.pv_a;
            for (int p = 0; p < npo; ++p) {
                const int i = occ[po[2 * p]], j = occ[po[2 * p + 1]];
                for (int q = lane; q < npv; q += 32) {
                    const int a = vir[pv[2 * q]], b = vir[pv[2 * q + 1]];
                    const int s1 = parity64(str & between_mask(i, a));
                    const unsigned long long s1s = str ^ (1ull << i) ^ (1ull << a);
                    const int s2 = parity64(s1s & between_mask(j, b));
                    const unsigned long long h2 = string_rank(s1s ^ (1ull << j) ^ (1ull << b), bt, ks);
                    const unsigned long long tg = spin ? hA * cb + h2 : h2 * cb + hB;
                    const long long f = table_find(psi, tg);
                    if (f < 0) continue;
                    double v = __ldcg(&psi.slots[f].val) * c;
                    if (s1 ^ s2) v = -v;
                    acc(g2, G2(a, i, b, j), v);
                    acc(g2, G2(b, j, a, i), v);
                    acc(g2, G2(a, j, b, i), -v);
                    acc(g2, G2(b, i, a, j), -v);
                }
            }
        }
        // opposite-spin doubles
        for (int x = 0; x < d.sa; ++x) {
            const unsigned long long ra = rankA1[x] * cb;
            const unsigned ha = hopA[x];
            const int i = ha & 0xff, a = (ha >> 8) & 0xff;
            for (int y = lane; y < d.sb; y += 32) {
                const long long f = table_find(psi, ra + rankB1[y]);
                if (f < 0) continue;
                const unsigned hb = hopB[y];
                const int j = hb & 0xff, b = (hb >> 8) & 0xff;
                double v = __ldcg(&psi.slots[f].val) * c;
                if ((ha >> 16) ^ (hb >> 16)) v = -v;
                acc(g2, G2(a, i, b, j), v);
                acc(g2, G2(b, j, a, i), v);
            }
        }
        __syncwarp();
    }
#undef G2
}

__global__ void norm2_kernel(const double *c, long long m, double *partial) {
    __shared__ double sh[kWarps];
    double a = 0.0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < m;
         i += (long long)gridDim.x * blockDim.x)
        a = __fma_rn(c[i], c[i], a);
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(kFull, a, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kWarps; ++w) t += sh[w];
        partial[blockIdx.x] = t;
    }
}

// the sum of np partial sums, by one warp
__device__ __forceinline__ double warp_total(const double *partial, int np) {
    double t = 0.0;
    for (int k = threadIdx.x; k < np; k += 32) t += partial[k];
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
    return t;
}

__global__ void norm2_finish(const double *partial, int np, double *out) {
    const double t = warp_total(partial, np);
    if (threadIdx.x == 0) *out = t;
}

constexpr int kNormBlocks = 152;

// partial[b] = sum over block b's share of k of x[k] y[k], fixed grid and order:
// h.gamma (blockIdx.y 0), g.Gamma (1)
__global__ void contract_kernel(const double *h, const double *g1, long long n2, const double *g, const double *g2,
                                long long n4, double *partial) {
    __shared__ double sh[kWarps];
    const double *x = blockIdx.y ? g : h, *y = blockIdx.y ? g2 : g1;
    const long long m = blockIdx.y ? n4 : n2;
    double a = 0.0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < m;
         i += (long long)gridDim.x * blockDim.x)
        a = __fma_rn(x[i], y[i], a);
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(kFull, a, o);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = a;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < kWarps; ++w) t += sh[w];
        partial[blockIdx.y * gridDim.x + blockIdx.x] = t;
    }
}

// E = e_core + (sum h gamma + 1/2 sum g Gamma) / norm2 from the two halves of partial
__global__ void energy_finish(const double *partial, int np, double e_core, double norm2, double *out) {
    const double one = warp_total(partial, np), two = warp_total(partial + np, np);
    if (threadIdx.x == 0) {
        out[0] = e_core + (one + 0.5 * two) / norm2;
        out[1] = one;
        out[2] = two;
    }
}

// ------------------------------------------------------------- pairs by rows
//
// The lookups of rdm_kernel (7876 a determinant at 20 orbitals, 1e9 at 3e5
// determinants counted once per pair) are bound by the L2 sectors of the hash
// table: 30 ms.  Here a CTA holds a row A' in a shared-memory table (beta index ->
// position) and looks up
//   opposite spin: the beta hops (tabulated once per beta string) of the
//       determinants of the rows one alpha hop away,
//   alpha singles and alpha-alpha doubles: the determinants of the rows one and
//       two hops away themselves,
// of each pair of rows the longer one in the table, so the shorter one is walked.
// Pairs within a row (beta singles, beta-beta doubles) come from comparing all its
// strings: m / 2 comparisons a determinant against sb + C(nb,2) C(vb,2) lookups.
// Pairs found wait in a queue per warp until 32 are there, and the diagonal's sums stay
// with the CTA: 3e5 determinants of 20 orbitals 30.4 ms by lookups, 5.9 ms with each pair
// worked on where it was found, 4.5 ms so (opposite spin 2.3, alpha 0.8, within rows 0.5),
// 3.3 ms with short rows compared string by string (up to 64 determinants 3.9, 256 3.3);
// 128 threads a CTA and four CTAs an SM instead of five were slower.

constexpr int kT = 256;
constexpr unsigned kChunk = 2048;       // determinants of a row in the table at once
constexpr unsigned kSlots = 4096;
constexpr unsigned kNone = 0xffffffffu;

struct RowArgs {
    SysDev d;
    const unsigned long long *rank;
    const double *coef;
    unsigned n;
    const int *flag;        // set: the ranks are not valid, nothing runs
    unsigned *first;        // [n] 1: starts a row
    unsigned long long *run_of;   // [n + 1] rows before
    unsigned *run_off;      // [n + 1] first determinant
    unsigned *run_row;      // [n]
    unsigned long long *run_str;  // [n] alpha string
    unsigned long long *units, *uoff;  // [n], [n + 1]
    unsigned *row_run;      // [ca] row -> run
    unsigned *b_seen;       // [cb]
    unsigned long long *b_id;     // [cb + 1]
    unsigned *s_b, *s_id;   // [n] beta index, number of the beta string
    unsigned *id_b;         // [distinct] its beta index
    unsigned long long *bstr;     // [distinct]
    uint2 *hops;            // [distinct * sb] beta index of the hop, b n + j | sign << 31
    unsigned long long *queue;    // and behind it the pairs of determinants that share a row, the units
    int count;                    // both are wanted
    double *g1, *g2;
};

struct RowUnits {  // of a row of m determinants
    unsigned long long n1, n2, n3;
    unsigned p1, p2, nb1, nb2, nf;
};

__device__ __forceinline__ RowUnits row_units(const SysDev &d, unsigned m) {
    RowUnits u;
    const unsigned nt = (m + kChunk - 1) / kChunk, tiles = (m + kT - 1) / kT;
    u.nb1 = d.sb > 0 ? (d.sa + kT - 1) / kT : 0u;
    u.nb2 = (d.sa + d.po_a * d.pv_a + kT - 1) / kT;
    u.p1 = (m + 31) / 32, u.p2 = (m + kT - 1) / kT;
    u.nf = (tiles + 3) / 4;
    u.n1 = (unsigned long long)u.nb1 * u.p1 * nt;
    u.n2 = (unsigned long long)u.nb2 * u.p2 * nt;
    u.n3 = (unsigned long long)tiles * u.nf;
    return u;
}

__global__ void rows_mark_kernel(RowArgs A) {
    if (*A.flag) return;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < A.n; i += gridDim.x * blockDim.x) {
        const unsigned long long r = A.rank[i], row = r / A.d.cb;
        const unsigned b = (unsigned)(r - row * A.d.cb);
        A.first[i] = i == 0 || A.rank[i - 1] / A.d.cb != row;
        A.s_b[i] = b;
        A.b_seen[b] = 1u;
    }
}

__global__ void rows_place_kernel(RowArgs A) {
    if (*A.flag) return;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < A.n; i += gridDim.x * blockDim.x) {
        const unsigned b = A.s_b[i], id = (unsigned)A.b_id[b];
        A.s_id[i] = id;
        A.id_b[id] = b;
        A.units[i] = 0ull;
        if (A.first[i]) {
            const unsigned run = (unsigned)A.run_of[i], row = (unsigned)(A.rank[i] / A.d.cb);
            A.run_off[run] = i;
            A.run_row[run] = row;
            A.row_run[row] = run;
        }
        if (i == A.n - 1) A.run_off[A.run_of[A.n]] = A.n;
    }
}

// a warp per distinct beta string: the string and its hops; then per row: its string, its units
__global__ void __launch_bounds__(kT) rows_strings_kernel(RowArgs A) {
    extern __shared__ __align__(16) unsigned char sm[];
    if (*A.flag) return;
    const SysDev &d = A.d;
    unsigned long long *bt = reinterpret_cast<unsigned long long *>(sm);
    for (int i = threadIdx.x; i < (d.n + 1) * d.ks; i += blockDim.x) bt[i] = d.binom[i];
    __syncthreads();
    __shared__ unsigned char lists[kT / 32][128];
    const int lane = threadIdx.x & 31;
    unsigned char *occ = lists[threadIdx.x >> 5], *vir = occ + 64;
    const unsigned nd = (unsigned)A.b_id[d.cb], runs = (unsigned)A.run_of[A.n];
    unsigned long long pairs = 0ull, units = 0ull;  // (lane 0's)
    for (unsigned w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nd + runs; w += (gridDim.x * blockDim.x) >> 5) {
        if (w >= nd) {
            const unsigned run = w - nd;
            const unsigned long long str = string_unrank_warp(A.run_row[run], d.n, d.na, bt, d.ks);
            if (lane == 0) {
                const unsigned m = A.run_off[run + 1] - A.run_off[run];
                const RowUnits u = row_units(d, m);
                pairs += (unsigned long long)m * (m - 1u) / 2ull;
                units += u.n1 + u.n2 + u.n3;
                A.run_str[run] = str;
                A.units[run] = u.n1 + u.n2 + u.n3;
            }
            continue;
        }
        const unsigned long long str = string_unrank_warp(A.id_b[w], d.n, d.nb, bt, d.ks);
        if (lane == 0) A.bstr[w] = str;
        __syncwarp();
        for (int p = lane; p < d.n; p += 32) {
            const int below = __popcll(str & ((1ull << p) - 1ull));
            if ((str >> p) & 1ull) occ[below] = (unsigned char)p;
            else vir[p - below] = (unsigned char)p;
        }
        __syncwarp();
        for (int x = lane; x < d.sb; x += 32) {
            const int j = occ[x / d.vb], b = vir[x % d.vb];
            const unsigned sg = parity64(str & between_mask(j, b));
            A.hops[(size_t)w * d.sb + x] =
                make_uint2((unsigned)string_rank(str ^ (1ull << j) ^ (1ull << b), bt, d.ks), (unsigned)(b * d.n + j) | sg << 31);
        }
    }
    if (A.count && units) {
        if (pairs) atomicAdd(A.queue + 1, pairs);
        atomicAdd(A.queue + 2, units);
    }
}

// D (string `from`) and D' (`to`) differ in this spin by one or two electrons, the other
// spin's string is `other`; v = c_D c_D' without the sign
__device__ __noinline__ void same_spin_pair(double *g1, double *g2, int n, unsigned long long from, unsigned long long to,
                                            unsigned long long other, double v) {
    const size_t N1 = size_t(n), N2 = N1 * n, N3 = N2 * n;
    unsigned long long out = from & ~to, in = to & ~from;
    const int i = __ffsll((long long)out) - 1, a = __ffsll((long long)in) - 1;
    int s = parity64(from & between_mask(i, a));
    out &= out - 1ull, in &= in - 1ull;
    if (out) {
        const int j = __ffsll((long long)out) - 1, b = __ffsll((long long)in) - 1;
        s ^= parity64((from ^ (1ull << i) ^ (1ull << a)) & between_mask(j, b));
        if (s) v = -v;
        acc(g2, a * N3 + i * N2 + b * N1 + j, v);
        acc(g2, a * N3 + j * N2 + b * N1 + i, -v);
        return;
    }
    if (s) v = -v;
    acc(g1, size_t(a) * n + i, v);
    for (unsigned long long k = from & to; k; k &= k - 1ull) {
        const int p = __ffsll((long long)k) - 1;
        acc(g2, a * N3 + i * N2 + p * N1 + p, v);
        acc(g2, a * N3 + p * N2 + p * N1 + i, -v);
    }
    for (unsigned long long k = other; k; k &= k - 1ull) {
        const int p = __ffsll((long long)k) - 1;
        acc(g2, a * N3 + i * N2 + p * N1 + p, v);
    }
}

// Opposite spin: a row of up to so many determinants is compared string by string (16 warp
// instructions per 32 pairs) instead of looking up every hop of the other row's (sb of them,
// 25 per 32 lookups); most rows of a sparse vector hold a few determinants.
constexpr unsigned kFew = 128;

struct RowShared {
    unsigned keys[kSlots];
    unsigned short pos[kSlots];  // (pairs within a row: strings and coefficients in place of both)
    unsigned start[kT + 1], off[kT], hop[kT];
    unsigned wsum[kT / 32];
    unsigned long long queue[kT / 32][64];  // pairs found, each warp's
    unsigned long long str[kFew];           // the strings of a row that is compared, not looked up in
    unsigned char occ[64], vir[64];
    unsigned long long u0;
    unsigned run;
};
// up to so many orbitals the diagonal's sums stay in shared memory until the kernel ends
constexpr int kDiagN = 32;
constexpr unsigned kTileF = 4 * kT;  // strings compared with a tile of 256 at a time
static_assert(kTileF * 16 <= kSlots * 4 && kT * 16 <= kSlots * 2, "a row's strings lie in the table's memory");

__device__ __forceinline__ int row_find(const unsigned *keys, unsigned mask, int shift, unsigned key) {
    unsigned h = (key * 0x9E3779B1u) >> shift;
    for (;;) {  // (at most half of the slots are taken)
        const unsigned k = keys[h];
        if (k == key) return (int)h;
        if (k == kNone) return -1;
        h = (h + 1u) & mask;
    }
}

__global__ void __launch_bounds__(kT, 5) rdm_rows_kernel(const __grid_constant__ RowArgs A) {
    extern __shared__ __align__(16) unsigned char sm[];
    if (*A.flag) return;
    RowShared &S = *reinterpret_cast<RowShared *>(sm);
    unsigned long long *bt = reinterpret_cast<unsigned long long *>(sm + al16(sizeof(RowShared)));
    const SysDev &d = A.d;
    const int n = d.n, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const size_t N1 = size_t(n), N2 = N1 * n, N3 = N2 * n;
    for (int i = tid; i < (n + 1) * d.ks; i += kT) bt[i] = d.binom[i];
    const unsigned runs = (unsigned)A.run_of[A.n];
    const unsigned long long total = A.uoff[A.n];
    unsigned have_run = kNone, have_t = 0u;  // what the table holds
    unsigned mask = 0u;
    int shift = 0;
    // D' = D: sums of c^2 by orbitals occupied together (each place has one thread that adds):
    // [p n + r] beta p < r, [p n + p] beta p, then [i n + j] alpha i < j, [i n + i] alpha i, then
    // [i n + p] alpha i and beta p
    double *diag = reinterpret_cast<double *>(bt + (n + 1) * d.ks);
    const bool staged = n <= kDiagN;
    if (staged)
        for (int x = tid; x < 3 * n * n; x += kT) diag[x] = 0.0;
    auto same = [&](int p, int r, double w) {  // a pair of one spin
        acc(A.g2, p * N3 + p * N2 + r * N1 + r, 0.5 * w);
        acc(A.g2, p * N3 + r * N2 + r * N1 + p, -0.5 * w);
    };
    // pairs found by the warp are worked on 32 at a time (one by one they left 26 lanes idle)
    unsigned have = 0;
    unsigned long long *found = S.queue[warp];
    const unsigned lt = (1u << lane) - 1u;
    auto push = [&](bool hit, unsigned long long item, auto &&work) {
        const unsigned bal = __ballot_sync(kFull, hit);
        if (!bal) return;
        if (hit) found[have + __popc(bal & lt)] = item;
        have += __popc(bal);
        __syncwarp();
        if (have < 32u) return;
        work(found[lane]);
        have -= 32u;
        unsigned long long left = 0ull;
        if ((unsigned)lane < have) left = found[32 + lane];
        __syncwarp();
        if ((unsigned)lane < have) found[lane] = left;
        __syncwarp();
    };
    auto finish = [&](auto &&work) {
        if ((unsigned)lane < have) work(found[lane]);
        have = 0u;
        __syncwarp();
    };
    for (;;) {
        __syncthreads();  // (the unit before is done with the shared memory)
        if (warp == 0) {  // (one unit at a time: four take 0.7 ms more at 3e5 determinants)
            unsigned long long u = 0ull;
            if (lane == 0) u = atomicAdd(A.queue, 1ull);
            u = __shfl_sync(kFull, u, 0);
            unsigned lo = 0, hi = runs;  // the last run whose units start at or before u
            while (u < total && hi - lo > 1u) {
                const unsigned step = (hi - lo + 31u) / 32u, at = lo + (lane + 1u) * step;
                const unsigned k = __popc(__ballot_sync(kFull, at < hi && __ldg(&A.uoff[at]) <= u));
                lo += k * step;
                hi = min(hi, lo + step);
            }
            if (lane == 0) S.u0 = u, S.run = lo;
        }
        __syncthreads();
        const unsigned long long u = S.u0;
        if (u >= total) break;
        const unsigned run = S.run;
        const unsigned base = __ldg(&A.run_off[run]), m = __ldg(&A.run_off[run + 1]) - base;
        const unsigned long long str = __ldg(&A.run_str[run]);
        const RowUnits U = row_units(d, m);
        unsigned long long q = u - __ldg(&A.uoff[run]);
        if (q >= U.n1 + U.n2) {
            // ---- pairs within the row: tile e against the strings f < e of four tiles
            q -= U.n1 + U.n2;
            const unsigned te = (unsigned)(q / U.nf), f0 = (unsigned)(q % U.nf) * kTileF;
            if (f0 > te * kT) continue;
            have_run = kNone;
            unsigned long long *fs = reinterpret_cast<unsigned long long *>(S.keys);
            double *fc = reinterpret_cast<double *>(fs + kTileF);
            unsigned long long *es = reinterpret_cast<unsigned long long *>(S.pos);
            double *ec = reinterpret_cast<double *>(es + kT);
            const unsigned e = te * kT + tid, nf = min(kTileF, m - f0), ne = min((unsigned)kT, m - te * kT);
            for (unsigned f = tid; f < nf; f += kT) {
                fs[f] = __ldg(&A.bstr[__ldg(&A.s_id[base + f0 + f])]);
                fc[f] = __ldg(&A.coef[base + f0 + f]);
            }
            if (e < m) {
                es[tid] = __ldg(&A.bstr[__ldg(&A.s_id[base + e])]);
                ec[tid] = __ldg(&A.coef[base + e]);
            }
            __syncthreads();
            {
                const unsigned long long be = e < m ? es[tid] : 0ull;
                const unsigned fe = e < m ? min(nf, e > f0 ? e - f0 : 0u) : 0u;
                const unsigned all = __reduce_max_sync(kFull, fe);
                const unsigned local = (unsigned)tid << 16;
                auto pair = [&](unsigned long long x) {
                    const unsigned le = (unsigned)x >> 16, lf = (unsigned)x & 0xffffu;
                    const double ce = ec[le], cf = fc[lf];
                    if (ce != 0.0 && cf != 0.0) same_spin_pair(A.g1, A.g2, n, es[le], fs[lf], str, ce * cf);
                };
                if (n <= 32)
                    for (unsigned f = 0; f < all; ++f)
                        push(f < fe && __popc((unsigned)be ^ (unsigned)fs[f]) <= 4, local | f, pair);
                else
                    for (unsigned f = 0; f < all; ++f) push(f < fe && __popcll(be ^ fs[f]) <= 4, local | f, pair);
                finish(pair);
            }
            if (f0 == 0u) {
                // D' = D: a thread per pair of beta orbitals (p < q: both occupied; p = q:
                // one) and one for the row's weight, along the tile
                for (int x = tid; x <= n * n; x += kT) {
                    const int p = x / n, r = x - p * n;
                    if (x < n * n && r < p) continue;
                    const unsigned long long both = x < n * n ? (1ull << p | 1ull << r) : 0ull;
                    double w = 0.0;
                    for (unsigned f = 0; f < ne; ++f)
                        if ((es[f] & both) == both && ec[f] != 0.0) w = __fma_rn(ec[f], ec[f], w);
                    if (w == 0.0) continue;
                    if (x == n * n) {
                        for (unsigned long long k = str; k; k &= k - 1ull) {
                            const int i = __ffsll((long long)k) - 1;
                            if (staged) diag[n * n + i * n + i] += w;
                            else acc(A.g1, size_t(i) * n + i, w);
                            for (unsigned long long l = k & (k - 1ull); l; l &= l - 1ull) {
                                const int j = __ffsll((long long)l) - 1;
                                if (staged) diag[n * n + i * n + j] += w;
                                else same(i, j, w);
                            }
                        }
                    } else if (p == r) {
                        if (staged) diag[x] += w;
                        else acc(A.g1, size_t(p) * n + p, w);
                        for (unsigned long long k = str; k; k &= k - 1ull) {
                            const int i = __ffsll((long long)k) - 1;
                            if (staged) diag[2 * n * n + i * n + p] += w;
                            else acc(A.g2, i * N3 + i * N2 + p * N1 + p, 0.5 * w);
                        }
                    } else {
                        if (staged) diag[x] += w;
                        else same(p, r, w);
                    }
                }
            }
            continue;
        }
        const bool opposite = q < U.n1;
        if (!opposite) q -= U.n1;
        const unsigned parts = opposite ? U.p1 : U.p2, nbat = opposite ? U.nb1 : U.nb2;
        const unsigned t = (unsigned)(q / ((unsigned long long)parts * nbat));
        const unsigned rem = (unsigned)(q - (unsigned long long)t * parts * nbat), batch = rem / parts, part = rem % parts;
        const unsigned t0 = t * kChunk, mc = min(kChunk, m - t0);
        // ---- the row's table and orbital lists
        if (have_run != run || have_t != t) {
            have_run = run, have_t = t;
            unsigned size = 256u;
            while (size < 4u * mc && size < kSlots) size *= 2u;
            mask = size - 1u;
            shift = 33 - __ffs((int)size);
            for (unsigned h = tid; h < size; h += kT) S.keys[h] = kNone;
            if (tid < n) {
                const int below = __popcll(str & ((1ull << tid) - 1ull));
                if ((str >> tid) & 1ull) S.occ[below] = (unsigned char)tid;
                else S.vir[tid - below] = (unsigned char)tid;
            }
            __syncthreads();
            for (unsigned f = tid; f < mc; f += kT) {
                const unsigned key = __ldg(&A.s_b[base + t0 + f]);
                unsigned h = (key * 0x9E3779B1u) >> shift;
                while (atomicCAS(&S.keys[h], kNone, key) != kNone) h = (h + 1u) & mask;
                S.pos[h] = (unsigned short)f;
                if (m <= kFew) S.str[f] = __ldg(&A.bstr[__ldg(&A.s_id[base + f])]);
            }
        }
        // ---- a batch of rows one or two hops away: hop from them to this row
        const unsigned x = batch * kT + tid, n_hops = opposite ? d.sa : d.sa + d.po_a * d.pv_a;
        unsigned cnt = 0, off = 0, hop = 0;
        unsigned long long from = 0ull;
        if (x < n_hops) {
            int i1, a1, i2 = 0, a2 = 0;
            const bool one = x < (unsigned)d.sa;
            if (one) {
                a1 = S.occ[x / d.va], i1 = S.vir[x % d.va];
                from = str ^ (1ull << a1) ^ (1ull << i1);
            } else {
                const unsigned y = x - d.sa;
                const unsigned char *po = d.pairs + 2 * (d.pair_off[0] + y / d.pv_a), *pv = d.pairs + 2 * (d.pair_off[1] + y % d.pv_a);
                a1 = S.occ[po[0]], a2 = S.occ[po[1]], i1 = S.vir[pv[0]], i2 = S.vir[pv[1]];
                from = str ^ (1ull << a1) ^ (1ull << i1) ^ (1ull << a2) ^ (1ull << i2);
            }
            const unsigned o = __ldg(&A.row_run[string_rank(from, bt, d.ks)]);
            if (o != kNone) {
                off = __ldg(&A.run_off[o]);
                const unsigned mo = __ldg(&A.run_off[o + 1]) - off;
                if (mo < m || (mo == m && o < run)) cnt = mo;
            }
            hop = (unsigned)(a1 * n + i1) | (unsigned)parity64(from & between_mask(i1, a1)) << 31;
        }
        unsigned inc = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const unsigned y = __shfl_up_sync(kFull, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) S.wsum[warp] = inc;
        __syncthreads();
        for (int w = 0; w < warp; ++w) inc += S.wsum[w];
        S.start[tid] = inc - cnt;
        S.off[tid] = off - (inc - cnt);
        S.hop[tid] = opposite ? hop : x;
        if (tid == kT - 1) S.start[kT] = inc;
        __syncthreads();
        const unsigned tot = S.start[kT];
        const unsigned lo = (unsigned)((unsigned long long)tot * part / parts), hi = (unsigned)((unsigned long long)tot * (part + 1) / parts);
        if (lo == hi) continue;
        auto segment = [&](unsigned at) {
            unsigned o = 0;
            for (unsigned step = kT / 2; step; step >>= 1)
                if (S.start[o + step] <= at) o += step;
            return o;
        };
        if (opposite && m <= kFew && m < 2u * d.sb) {
            auto pair = [&](unsigned long long x) {
                const unsigned s = (unsigned)(x >> 32), hp = S.hop[(unsigned)x >> 16 & 0xffffu], f = (unsigned)x & 0xffffu;
                const double c1 = __ldg(&A.coef[s]), c2 = __ldg(&A.coef[base + f]);
                if (c1 == 0.0 || c2 == 0.0) return;
                const unsigned long long b1 = __ldg(&A.bstr[__ldg(&A.s_id[s])]), b2 = S.str[f];
                const int j = __ffsll((long long)(b1 & ~b2)) - 1, b = __ffsll((long long)(b2 & ~b1)) - 1;
                const double v = c1 * c2;
                acc(A.g2, size_t(hp & 0x7fffffffu) * N2 + b * n + j,
                    (hp >> 31 ^ (unsigned)parity64(b1 & between_mask(j, b))) ? -v : v);
            };
            // a warp takes up to 32 determinants and runs through the row for each, end to end
            const unsigned per = min(32u, (hi - lo + kT / 32 - 1u) / (kT / 32));
            for (unsigned p0 = lo + warp * per; p0 < hi; p0 += per * (kT / 32)) {
                const unsigned k = min(per, hi - p0);
                unsigned o = 0, s = 0;
                unsigned long long bs = 0ull;
                if ((unsigned)lane < k) {
                    o = segment(p0 + lane), s = S.off[o] + p0 + lane;
                    bs = __ldg(&A.bstr[__ldg(&A.s_id[s])]);
                }
                unsigned l = (unsigned)lane / m, y = (unsigned)lane % m;
                const unsigned dl = 32u / m, dy = 32u % m;
                for (unsigned r = 0; r < k * m; r += 32u) {
                    const unsigned src = l < k ? l : 0u;
                    const unsigned long long b1 = __shfl_sync(kFull, bs, src);
                    const unsigned s1 = __shfl_sync(kFull, s, src), o1 = __shfl_sync(kFull, o, src);
                    push(l < k && __popcll(b1 ^ S.str[y]) == 2, (unsigned long long)s1 << 32 | o1 << 16 | y, pair);
                    l += dl, y += dy;
                    if (y >= m) y -= m, ++l;
                }
            }
            finish(pair);
        } else if (opposite) {
            // a warp takes up to 32 determinants and runs through their hops end to end
            const unsigned per = min(32u, (hi - lo + kT / 32 - 1u) / (kT / 32));
            for (unsigned p0 = lo + warp * per; p0 < hi; p0 += per * (kT / 32)) {
                const unsigned k = min(per, hi - p0);
                unsigned id = 0, hp = 0;
                double c = 0.0;
                if ((unsigned)lane < k) {
                    const unsigned o = segment(p0 + lane), s = S.off[o] + p0 + lane;
                    id = __ldg(&A.s_id[s]) * (unsigned)d.sb, hp = S.hop[o];
                    c = __ldg(&A.coef[s]);
                }
                unsigned l = (unsigned)lane / d.sb, y = (unsigned)lane % d.sb;
                const unsigned dl = 32u / d.sb, dy = 32u % d.sb;
                for (unsigned r = 0; r < k * d.sb; r += 32u) {
                    const bool in = l < k;
                    const unsigned src = in ? l : 0u;
                    const unsigned id1 = __shfl_sync(kFull, id, src), hp1 = __shfl_sync(kFull, hp, src);
                    const double c1 = __shfl_sync(kFull, c, src);
                    if (in) {
                        const uint2 e = __ldg(&A.hops[(size_t)id1 + y]);
                        const int f = row_find(S.keys, mask, shift, e.x);
                        if (f >= 0) {
                            const double c2 = __ldg(&A.coef[base + t0 + S.pos[f]]);
                            if (c1 != 0.0 && c2 != 0.0) {
                                const double v = c1 * c2;
                                acc(A.g2, size_t(hp1 & 0x7fffffffu) * N2 + (e.y & 0x7fffffffu), (hp1 ^ e.y) >> 31 ? -v : v);
                            }
                        }
                    }
                    l += dl, y += dy;
                    if (y >= (unsigned)d.sb) y -= d.sb, ++l;
                }
            }
        } else {
            // a pair: source in the upper half, its hop and its place in the table in the lower
            auto pair = [&](unsigned long long x) {
                const unsigned s = (unsigned)(x >> 32), y = S.hop[(unsigned)x >> 16 & 0xffffu], f = (unsigned)x & 0xffffu;
                const double c1 = __ldg(&A.coef[s]), c2 = __ldg(&A.coef[base + t0 + f]);
                if (c1 == 0.0 || c2 == 0.0) return;
                unsigned long long a = str;
                if (y < (unsigned)d.sa) {
                    a ^= (1ull << S.occ[y / d.va]) ^ (1ull << S.vir[y % d.va]);
                } else {
                    const unsigned z = y - d.sa;
                    const unsigned char *po = d.pairs + 2 * (d.pair_off[0] + z / d.pv_a), *pv = d.pairs + 2 * (d.pair_off[1] + z % d.pv_a);
                    a ^= (1ull << S.occ[po[0]]) ^ (1ull << S.occ[po[1]]) ^ (1ull << S.vir[pv[0]]) ^ (1ull << S.vir[pv[1]]);
                }
                same_spin_pair(A.g1, A.g2, n, a, str, __ldg(&A.bstr[__ldg(&A.s_id[s])]), c1 * c2);
            };
            for (unsigned i0 = lo + warp * 32; i0 < hi; i0 += kT) {
                const unsigned it = i0 + lane;
                unsigned o = 0, s = 0;
                int f = -1;
                if (it < hi) {
                    o = segment(it), s = S.off[o] + it;
                    f = row_find(S.keys, mask, shift, __ldg(&A.s_b[s]));
                }
                push(f >= 0, (unsigned long long)s << 32 | o << 16 | (f >= 0 ? S.pos[f] : 0), pair);
            }
            finish(pair);
        }
    }
    if (!staged) return;
    for (int x = tid; x < n * n; x += kT) {  // (every thread has left the units)
        const int p = x / n, r = x - p * n;
        const double b = diag[x], a = diag[n * n + x], ab = diag[2 * n * n + x];
        if (ab != 0.0) acc(A.g2, p * N3 + p * N2 + r * N1 + r, 0.5 * ab);
        if (p == r) {
            if (a + b != 0.0) acc(A.g1, x, a + b);
        } else if (a + b != 0.0) {
            same(p, r, a + b);
        }
    }
}

// each pair added to one image of its elements: the others, in place (an orbit per thread)
__global__ void rows_images_kernel(int n, const int *flag, double *g1, double *g2) {
    if (*flag) return;
    const unsigned n2 = n * n, n4 = n2 * n2;
    for (unsigned x = blockIdx.x * blockDim.x + threadIdx.x; x < n4; x += gridDim.x * blockDim.x) {
        const unsigned pq = x / n2, rs = x - pq * n2;
        const unsigned qp = pq % n * n + pq / n, sr = rs % n * n + rs / n;
        const unsigned x1 = rs * n2 + pq, x2 = qp * n2 + sr, x3 = sr * n2 + qp;
        if (x > x1 || x > x2 || x > x3) continue;
        const double v = (g2[x] + g2[x1]) + (g2[x2] + g2[x3]);
        g2[x] = g2[x1] = g2[x2] = g2[x3] = v;
    }
    for (unsigned x = blockIdx.x * blockDim.x + threadIdx.x; x < n2; x += gridDim.x * blockDim.x) {
        const unsigned p = x / n, q = x - p * n;
        if (p < q) {
            const double v = g1[x] + g1[q * n + p];
            g1[x] = g1[q * n + p] = v;
        }
    }
}

inline size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

unsigned long long rdm_slots(long long m) {
    unsigned long long want = 2ull * (unsigned long long)(m > 0 ? m : 1), p = 1024;
    while (p < want) p <<= 1;
    return p;
}

struct RdmLayout {
    unsigned long long slots;
    size_t table, status, count, partial, norm, bytes;
};

RdmLayout rdm_layout(long long m) {
    RdmLayout L{};
    L.slots = rdm_slots(m);
    size_t o = 0;
    L.table = o, o = a256(o + L.slots * sizeof(Slot));
    L.status = o, o = a256(o + sizeof(int));
    L.count = o, o = a256(o + 8);
    L.partial = o, o = a256(o + 8 * kNormBlocks);
    L.norm = o, o = a256(o + 8);
    L.bytes = o;
    return L;
}

// the row path's buffers in the workspace (base null: sizes only)
size_t rows_place(char *base, RowArgs &A, size_t &scan_ws, size_t &partial, const SysDev &d, long long n) {
    size_t o = 0;
    auto take = [&](auto *&p, size_t count) {
        p = base ? reinterpret_cast<std::remove_reference_t<decltype(p)>>(base + o) : nullptr;
        o = a256(o + count * sizeof(*p));
    };
    const size_t nn = size_t(n), ca = size_t(d.ca), cb = size_t(d.cb), nd = std::min(nn, cb);
    take(A.queue, 3);        // (the queue, the counts behind it and b_seen are cleared together)
    take(A.b_seen, cb);
    take(A.row_run, ca);
    take(A.b_id, cb + 1);
    take(A.first, nn);
    take(A.run_of, nn + 1);
    take(A.run_off, nn + 1);
    take(A.run_row, nn);
    take(A.run_str, nn);
    take(A.units, nn);
    take(A.uoff, nn + 1);
    take(A.s_b, nn);
    take(A.s_id, nn);
    take(A.id_b, nd);
    take(A.bstr, nd);
    take(A.hops, nd * size_t(d.sb));
    scan_ws = o, o = a256(o + scan_ws_bytes((long long)std::max(nn, cb) + 1));
    partial = o, o = a256(o + 8 * (kNormBlocks + 2));
    return o;
}

// Up to so many pairs within rows, and whether n determinants may have more: 26 per beta excitation
// of each determinant is where one row of 28 orbitals breaks even.  28 orbitals, 7 beta electrons:
// 5.8e5 determinants on one row 106 ms by rows and 43 by lookups, on four rows (with 7 alpha
// electrons) 57 and 143, on 1e5 rows 21 and 140; 1e5 on one row 3.8 and 9.4.
double row_pairs_limit(const SysDev &d, long long n) {
    return (2048.0 + 26.0 * ((double)d.sb + (double)d.po_b * d.pv_b)) * (double)n;
}
bool row_pairs_may_exceed(const SysDev &d, long long n) {
    return 0.5 * std::min((double)n, (double)d.cb) * (double)n > row_pairs_limit(d, n);
}

// Up to so many units, and whether n determinants may have more.  A unit takes some 9 ns of the chip
// even where it finds nothing (more with more beta electrons on the diagonal), and a row of one
// determinant has a unit per 256 alpha excitations; a lookup takes 10.5 ps, a determinant's other
// work there 45 ns (23 without beta hops), and no call less than one warp's lookups in turn, 50 ns
// each.  Where the opposite-spin lookups are few, the rows lose: 28 orbitals, 7 alpha electrons, 1e5
// determinants on as many rows and none, 1, 2, 3 beta electrons: 20.9, 19.9, 18.9, 18.8 ms by rows,
// 9.4, 11.1, 15.0, 18.1 by lookups; 20 to a row 1.2 (1 to 3 electrons) and 10.5, 14.8, 18.1.
double row_units_limit(const SysDev &d, long long n) {
    const double exc = (double)d.sa + d.sb + (double)d.po_a * d.pv_a + (double)d.po_b * d.pv_b + (double)d.sa * d.sb;
    return ((double)n * ((d.sb == 0 ? 23.0 : 45.0) + 0.0105 * exc) + 50.0 * exc) / (9.2 + 0.08 * d.nb);
}
bool row_units_may_exceed(const SysDev &d, long long n) {  // (as many where there is one beta string)
    const double hops = (double)d.sa + (double)d.po_a * d.pv_a;
    return (double)n * (1.0 + std::ceil(hops / kT) + (d.sb ? std::ceil((double)d.sa / kT) : 0.0)) > row_units_limit(d, n);
}

// A call whose rows are few or small waits for its slowest unit: a thread steps through the row's
// strings (up to 1024 of them) and through the tile for each of its places on the diagonal, 0.25 us a
// step, after 45 us more of launches than the lookups need; these wait for one warp's lookups in
// turn, 0.1 us each.  How uneven the rows are is not known: three times their mean.  One row of 1190
// determinants of 17 orbitals, 4 electrons 429 us by rows, 88 by lookups; 4427 of 23 orbitals, 4
// electrons 566 and 174.  (6463 systems of 8 to 34 orbitals: rows slower by a tenth or more in 467
// without this line, in 154 with it.)
bool rows_wait(const SysDev &d, long long n) {
    const double exc = (double)d.sa + d.sb + (double)d.po_a * d.pv_a + (double)d.po_b * d.pv_b + (double)d.sa * d.sb;
    const double m = std::min({(double)n, (double)d.cb, std::ceil(3.0 * (double)n / (double)d.ca)});
    const double steps = std::ceil((d.n * d.n + 1.0) / kT) * std::min(m, (double)kT) + std::min(m, (double)kTileF);
    return 90.0 + 0.25 * steps > 45.0 + 0.1 * exc + (double)n * (0.025 + 1.05e-5 * exc);
}

// Pairs by rows: strings are numbered in 26 bits, their hops in 32.  A determinant is compared
// with all of its row, 0.6 to 1.2 ps a pair, where the lookups take 7 to 16 ps for each of its
// excitations (28 orbitals, 7 + 7 electrons, level-like vectors: 3e5 determinants 20.5 ms and
// 78 by lookups, 5.8e5 34 and 145; up to 587 000 strings by the last line).
bool rows_taken(const SysDev &d, long long n) {
    const double exc = (double)d.sb + (double)d.po_b * d.pv_b;
    return n > 0 && n < (1ll << 31) && d.ca <= (1ull << 26) && d.cb <= (1ull << 26) &&
           std::min((double)n, (double)d.cb) * std::max(d.sb, 1) < 4294967296.0 &&
           (double)d.sa + (double)d.po_a * d.pv_a < 2147483648.0 &&
           std::min((double)n, (double)d.cb) <= 4096.0 + 128.0 * exc && !(d.cb == 1 && row_units_may_exceed(d, n)) &&
           !rows_wait(d, n);
}

int sms() {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return n > 0 ? n : 1;
}

}  // namespace
}  // namespace sfci

using namespace sfci;

extern "C" {

sfci_status sfci_rdm12_workspace_bytes(const sfci_system *s, int64_t n, size_t *bytes) {
    if (!s || !bytes || n < 0) {
        set_error("bad arguments");
        return SFCI_E_INVALID;
    }
    *bytes = rdm_layout(n).bytes;
    if (rows_taken(s->d, n)) {
        RowArgs A{};
        size_t scan_ws, partial;
        *bytes = std::max(*bytes, rows_place(nullptr, A, scan_ws, partial, s->d, n));
    }
    return SFCI_OK;
}

sfci_status sfci_rdm12(const sfci_system *s, const uint64_t *rank, const double *coef, int64_t n,
                       double *rdm1, double *rdm2, double *norm2, void *workspace,
                       size_t ws_bytes, void *stream) {
    if (!s || n < 0 || !rdm1 || !rdm2 || (n > 0 && (!rank || !coef))) {
        set_error("bad arguments");
        return SFCI_E_INVALID;
    }
    const RdmLayout L = rdm_layout(n);
    if (!workspace || ws_bytes < L.bytes) {
        set_error("workspace smaller than sfci_rdm12_workspace_bytes");
        return SFCI_E_CAPACITY;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const SysDev &d = s->d;
    const size_t n2 = size_t(d.n) * d.n;
    char *w = static_cast<char *>(workspace);
    SFCI_CUDA(cudaMemsetAsync(rdm1, 0, n2 * 8, st));
    SFCI_CUDA(cudaMemsetAsync(rdm2, 0, n2 * n2 * 8, st));
    const unsigned long long *r = reinterpret_cast<const unsigned long long *>(rank);
    RowArgs A{};
    size_t scan_ws = 0, part_at = L.partial;
    bool by_rows = rows_taken(d, n) && rows_place(nullptr, A, scan_ws, part_at, d, n) <= ws_bytes;
    double *nrm = nullptr;
    int *flag = nullptr;
    const auto norm_and_check = [&]() -> sfci_status {
        double *partial = reinterpret_cast<double *>(w + (by_rows ? part_at : L.partial));
        // the norm and, behind it, the flag of invalid ranks: read back together
        nrm = by_rows ? partial + kNormBlocks : reinterpret_cast<double *>(w + L.norm);
        flag = reinterpret_cast<int *>(nrm + 1);
        SFCI_CUDA(cudaMemsetAsync(nrm, 0, 16, st));
        SFCI_CUDA(validate_sorted(r, n, d.dim, flag, st));
        count_launch();
        norm2_kernel<<<kNormBlocks, kThreads, 0, st>>>(coef, n, partial);
        count_launch();
        norm2_finish<<<1, 32, 0, st>>>(partial, kNormBlocks, nrm);
        SFCI_CUDA(cudaGetLastError());
        return SFCI_OK;
    };
    sfci_status e = norm_and_check();
    if (e != SFCI_OK) return e;
    if (by_rows) {
        size_t ignore;
        rows_place(w, A, ignore, ignore, d, n);
        A.d = d, A.rank = r, A.coef = coef, A.n = (unsigned)n, A.flag = flag, A.g1 = rdm1, A.g2 = rdm2;
        A.count = row_pairs_may_exceed(d, n) || row_units_may_exceed(d, n);
        SFCI_CUDA(cudaMemsetAsync(A.queue, 0, size_t((char *)A.row_run - (char *)A.queue), st));
        SFCI_CUDA(cudaMemsetAsync(A.row_run, 0xff, size_t(d.ca) * 4, st));
        const unsigned g = (unsigned)std::min<long long>((n + kT - 1) / kT, sms() * 8ll);
        count_launch();
        rows_mark_kernel<<<g, kT, 0, st>>>(A);
        SFCI_CUDA(exclusive_scan(A.first, n, A.run_of, w + scan_ws, st));
        SFCI_CUDA(exclusive_scan(A.b_seen, (long long)d.cb, A.b_id, w + scan_ws, st));
        count_launch();
        rows_place_kernel<<<g, kT, 0, st>>>(A);
        const size_t bts = size_t(d.n + 1) * d.ks * 8;
        count_launch();
        rows_strings_kernel<<<(unsigned)std::min<long long>((n + kT / 64 - 1) / (kT / 64), sms() * 8ll), kT, bts, st>>>(A);
        if (A.count) {
            unsigned long long has[2] = {0, 0};  // pairs, units
            SFCI_CUDA(cudaMemcpyAsync(has, A.queue + 1, 16, cudaMemcpyDeviceToHost, st));
            SFCI_CUDA(cudaStreamSynchronize(st));
            // (the table takes the rows' place in the workspace)
            if ((double)has[0] > row_pairs_limit(d, n) || (double)has[1] > row_units_limit(d, n)) {
                by_rows = false;
                if ((e = norm_and_check()) != SFCI_OK) return e;
            }
        }
    }
    if (by_rows) {
        const size_t bts = size_t(d.n + 1) * d.ks * 8;
        SFCI_CUDA(exclusive_scan(A.units, n, A.uoff, w + scan_ws, st));
        const size_t smem = al16(sizeof(RowShared)) + bts + (d.n <= kDiagN ? size_t(3) * d.n * d.n * 8 : 0);
        SFCI_CUDA(allow_max_smem(rdm_rows_kernel, smem));
        int per_sm = 0;
        SFCI_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, rdm_rows_kernel, kT, smem));
        if (per_sm < 1) {
            set_error("rdm kernel does not fit on an SM for this system");
            return SFCI_E_CAPACITY;
        }
        count_launch();
        rdm_rows_kernel<<<sms() * per_sm, kT, smem, st>>>(A);
        count_launch();
        rows_images_kernel<<<(unsigned)std::min<size_t>((n2 * n2 + kT - 1) / kT, size_t(sms()) * 8), kT, 0, st>>>(d.n, flag, rdm1, rdm2);
        SFCI_CUDA(cudaGetLastError());
    } else {
        Table t;
        t.slots = reinterpret_cast<Slot *>(w + L.table);
        t.mask = L.slots - 1;
        t.shift = 64 - __builtin_ctzll(L.slots);
        t.status = reinterpret_cast<int *>(w + L.status);
        t.count = reinterpret_cast<unsigned long long *>(w + L.count);
        SFCI_CUDA(table_clear(t, st));
        SFCI_CUDA(table_axpy(t, r, coef, n, nullptr, 1.0, 1.0, st));
        if (n > 0) {
            const size_t smem = rdm_block_smem(d) + kWarps * rdm_warp_smem(d);
            SFCI_CUDA(allow_max_smem(rdm_kernel, smem));
            int per_sm = 0;
            SFCI_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, rdm_kernel, kThreads, smem));
            if (per_sm < 1) {
                set_error("rdm kernel does not fit on an SM for this system");
                return SFCI_E_CAPACITY;
            }
            long long grid = (long long)sms() * per_sm, want = (n + kWarps - 1) / kWarps;
            if (want < grid) grid = want;
            count_launch();
            rdm_kernel<<<(unsigned)grid, kThreads, smem, st>>>(d, r, coef, n, t, rdm1, rdm2);
            SFCI_CUDA(cudaGetLastError());
        }
    }
    struct {
        double norm;
        int flag, pad;
    } host{};
    SFCI_CUDA(cudaMemcpyAsync(&host, nrm, 16, cudaMemcpyDeviceToHost, st));
    SFCI_CUDA(cudaStreamSynchronize(st));
    if (host.flag) {
        set_error("input ranks must be strictly ascending and below dim");
        return SFCI_E_INVALID;
    }
    if (norm2) *norm2 = host.norm;
    return SFCI_OK;
}

sfci_status sfci_rdm_energy(int n_orb, const double *rdm1, const double *rdm2, double norm2,
                            const double *h, const double *g, double e_core, double *energy,
                            void *workspace, size_t ws_bytes, void *stream) {
    if (n_orb < 1 || n_orb > 64 || !rdm1 || !rdm2 || !h || !g || !energy || !(norm2 > 0.0)) {
        set_error("need 1 <= n_orb <= 64, device rdm1, rdm2, h, g, a host energy and norm2 > 0");
        return SFCI_E_INVALID;
    }
    if (!workspace || ws_bytes < size_t(2 * kNormBlocks + 3) * 8) {
        set_error("workspace below sfci_rdm_energy's 2456 bytes");
        return SFCI_E_CAPACITY;
    }
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    double *partial = static_cast<double *>(workspace);
    double *out = partial + 2 * kNormBlocks;
    const long long n2 = (long long)n_orb * n_orb;
    count_launch();
    contract_kernel<<<dim3(kNormBlocks, 2), kThreads, 0, st>>>(h, rdm1, n2, g, rdm2, n2 * n2, partial);
    count_launch();
    energy_finish<<<1, 32, 0, st>>>(partial, kNormBlocks, e_core, norm2, out);
    SFCI_CUDA(cudaGetLastError());
    SFCI_CUDA(cudaMemcpyAsync(energy, out, 8, cudaMemcpyDeviceToHost, st));
    SFCI_CUDA(cudaStreamSynchronize(st));
    return SFCI_OK;
}

}  // extern "C"
