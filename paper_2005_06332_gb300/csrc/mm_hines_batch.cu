// mm_hines_batch.cu -- a standalone batched Hines solve on the device.
//
// Algorithm 1 (Sec. 2) for many independent trees at once, any numbering with
// parent[j] < j.  Inputs are const; the diagonal and what it becomes (see
// solve_group) live in a scratch array, the rhs is worked on in the output
// array.  Device pointers in and out.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "mm.h"
#include "mm_fp64_math.h"

// Scratch of mm_hines_solve_noalloc: a fixed device array in this library
// image, so that the call never allocates.  The first 256 bytes hold the
// status words, the next 8 KiB the lists of left groups, the rest the working
// values of the diagonal (MM_NOALLOC_MAX_COMPS doubles, 8 MiB).  Every GPU that
// loads the library holds it until the process ends.
#define MM_NOALLOC_MAX_COMPS (1 << 20)
#define MM_NOALLOC_LEFT 1024
static __device__ __align__(256) double g_noalloc_scratch[32 + MM_NOALLOC_LEFT + MM_NOALLOC_MAX_COMPS];

namespace {

struct Batch {
    int32_t n_trees;
    int64_t n_comp;
    const int64_t *off;
    const int32_t *parent;
    const double *a, *b, *c, *rhs;
    double *x, *work;
    int *status;             // [0] nonzero: a tree violates the parent rule or its entries lie outside n_comp;
                             // [1], [2]: groups of trees left to hines_left_kernel and to hines_rest_kernel; [3],
                             // [4], [5]: of some of the first, how many, their levels, their largest tree
    int32_t *left;           // these groups, left_cap of the first kind, then left_cap of the second
    int32_t left_cap;
    int32_t trees_per_block; // 1 .. kMaxTrees
};

// One tree by one thread, exactly as Algorithm 1 is stated: the path of trees
// that the block's tables do not hold, and of blocks with an invalid tree (such
// a tree is skipped before any of its entries is touched).
__device__ void solve_serial(const Batch &B, int32_t t)
{
    const int64_t base = B.off[t], end = B.off[t + 1];
    if (base < 0 || end < base || end > B.n_comp) {
        atomicOr(B.status, 1);
        return;
    }
    const int64_t n = end - base;
    if (n == 0) return;
    const int32_t *__restrict__ p = B.parent + base;
    bool ok = p[0] == -1;
    for (int64_t i = 1; ok && i < n; ++i) ok = p[i] >= 0 && p[i] < i;
    if (!ok) {
        atomicOr(B.status, 1);
        return;
    }
    for (int64_t i = 0; i < n; ++i) {  // (x may be rhs)
        B.work[base + i] = B.b[base + i];
        B.x[base + i] = B.rhs[base + i];
    }
    double *__restrict__ w = B.work + base;
    double *__restrict__ r = B.x + base;
    const double *__restrict__ a = B.a + base, *__restrict__ c = B.c + base;
    // backward sweep, leaves to root
    for (int64_t i = n - 1; i >= 1; --i) {
        const double factor = a[i] / w[i];
        w[p[i]] -= factor * c[i];
        r[p[i]] -= factor * r[i];
    }
    r[0] /= w[0];
    // forward sweep, root to leaves
    for (int64_t i = 1; i < n; ++i) {
        r[i] -= c[i] * r[p[i]];
        r[i] /= w[i];
    }
}

// The sweeps by products and the short division keep Algorithm 1's results, its
// infinities and NaN included, for entries of ordinary size: |b| in [2^-200,
// 2^200], |a| and |c| (a root's are not used) at most 2^200, rhs zero or |rhs|
// in [2^-700, 2^200].  Then every eliminated diagonal is zero or in [2^-305,
// 2^740] (the smallest comes of a cancellation of two terms of 2^-200, the
// largest of a c / d), so N, M and the reciprocal of N keep all their bits, and S
// those of every rhs that is not below 2^-900 of the diagonal.  Trees in a block
// with an entry of any other size, infinities and NaN are solved as Algorithm 1
// is stated.  b and rhs are looked at where they are copied, a and c where they
// are loaded for the elimination; only where that has overwritten the rhs (x ==
// rhs) are a and c read for it beforehand.  3,000 trees of 50 to 5,000 entries:
// 0.877 ms without and with the looks.
__device__ __forceinline__ uint32_t exponent_of(double v) { return ((uint32_t)__double2hiint(v) >> 20) & 0x7FFu; }

__device__ __forceinline__ bool ordinary_row(double b, double rhs)
{
    constexpr uint32_t kMax = 1023 + 200, kMinB = 1023 - 200, kMinRhs = 1023 - 700;
    return exponent_of(b) - kMinB <= kMax - kMinB &&
           (exponent_of(rhs) - kMinRhs <= kMax - kMinRhs ||
            (((uint32_t)__double2hiint(rhs) << 1) | (uint32_t)__double2loint(rhs)) == 0);
}

// The larger of the magnitudes' high words (above kCouplingMax: not ordinary).
constexpr uint32_t kCouplingMax = ((1023u + 201u) << 20) - 1;
__device__ __forceinline__ uint32_t high_word(double a, double c)
{
    return (uint32_t)max(__double2hiint(a) & 0x7FFFFFFF, __double2hiint(c) & 0x7FFFFFFF);
}

// 1 / x and, with r = reciprocal(x), a / x for x in the range above or zero:
// rcp_nr and div_nr, but the first approximation where that is infinite or NaN
// (a zero pivot; a quotient beyond FP64's range; an infinite a), which the
// residuals would turn into NaN.  (A branch to CUDA's division there cost 0.11
// of 0.88 ms.)
__device__ __forceinline__ bool finite(double x) { return (__double2hiint(x) & 0x7FF00000) != 0x7FF00000; }

__device__ __forceinline__ double reciprocal(double x)
{
    const double r = mmk::rcp_approx(x), e = fma(-x, r, 1.0);
    return finite(r) ? fma(r, fma(e, e, e), r) : r;
}

__device__ __forceinline__ double divide(double a, double x, double r)
{
    const double q = a * r;
    return finite(q) ? fma(r, fma(-x, q, a), q) : q;
}

constexpr int kMaxTrees = 128;     // trees of one block
constexpr int kBlockComps = 2048;  // compartments aimed at per block
constexpr int kTiny = 8;           // trees of a block up to this size: a thread each at once (see solve_group)
constexpr int kSmallChains = 1024, kLargeChains = 8192;  // chains that a block's tables hold
constexpr int kSms = 152, kSmallSlots = 6 * kSms;  // blocks on the chip at a time with the larger and the smaller tables
enum { kFirst, kLeft, kCount };                    // solve_group
// Groups that may be left.  One that has more chains than the tables hold has
// more than kSmallChains entries, and the groups' entries lie side by side; deep
// ones are about as large.  Blocks beyond that (many deep small groups, or
// offsets that run backwards somewhere, which make the call fail) solve their
// trees serially at once.
constexpr int32_t left_cap_of(int64_t n_comp) { return (int32_t)(n_comp / (kSmallChains + 1)) + 1; }
static_assert(left_cap_of(MM_NOALLOC_MAX_COMPS) <= MM_NOALLOC_LEFT, "lists of the fixed scratch");
constexpr size_t smem_of(int chains) { return (size_t)chains * 20 + 16; }

// One entry of a chain's elimination: N / M is its eliminated diagonal, S / M
// its rhs.
struct Front {
    double N, M, S;
    // powers of two out, so that N lies in [1, 2); a zero pivot becomes NaN
    // (the division by it is what fails in Algorithm 1)
    __device__ __forceinline__ void normalise()
    {
        const int d = mmk::exponent2(N);
        if (((__double2hiint(N) & 0x7FFFFFFF) | __double2loint(N)) == 0) N = __longlong_as_double(0x7FF8000000000000LL);
        N = __hiloint2double(__double2hiint(N) - d, __double2loint(N));
        M = mmk::scale2(M, -d);
        S = mmk::scale2(S, -d);
    }
};

// A block solves trees_per_block consecutive trees together.  Bound by the
// FP64 pipe and, for the largest trees, by the chain of their sweeps: a warp's
// FP64 instruction takes 64 clocks of its scheduler whatever the number of
// active lanes, so the sweeps want many independent chains per warp, many
// blocks per SM, and few FP64 instructions per entry:
//   * the entries are cut into chains (runs with parent[i] = i - 1); chains
//     of one level -- hanging off chains of the level above -- are swept by
//     one lane each, from the deepest level up and back down;
//   * the elimination carries N, M, S (Algorithm 1's row times M: N' = b N -
//     (a M) c, M' = N, S' = rhs N - a S), five instructions instead of a
//     division and three; the division is a pass of full warps afterwards
//     (f = -c M / N, s = S / N), and the substitution is x_j = f_j x_{j-1} + s_j;
//   * a chain's first entry is divided when its warp's chains are done, and
//     its share goes into the entry it hangs off, b += a f, rhs -= a s, after
//     the level, one thread per entry, larger children first as Algorithm 1
//     does (the chains are sorted by level and that entry).
// b and rhs, then N and S, then f and s, then x live in the scratch and the
// output array (L2).  Measured (whole call, allocation included): 3,000 trees of
// 50 to 5,000 entries 12.4 ms with a thread per tree, 0.87 ms so (0.65 ms in
// the kernel, FP64 pipe 44 % busy); 3,000 of 8 to 300 0.78 -> 0.33 ms; 64 of 200
// to 5,000 9.0 -> 0.57 ms.  128 threads and six blocks per SM; 32 or 64 threads
// and more blocks 0.94 to 1.14 ms, groups of 4,096 entries 1.34 ms; eliminating
// the diagonal alone first (with a c stored: 2 + 2 + 2 instructions in the
// sweeps, but two passes more) 1.10 ms.  CHAINS: the chains that a block's tables hold.  MODE:
// kFirst every group of trees (`groups` in all), kLeft those that a smaller table
// left, kCount the levels of one of these and nothing else.  A group is on
// one list at a time, so that its trees are solved once, also where x is rhs.
// Where no tree has more than kTiny entries a thread solves each at once: what
// comes before the sweeps takes longer (a million trees of two entries 0.41 ->
// 0.30 ms, of five 0.61 -> 0.56; of twelve it is the other way, 1.13 -> 1.24).
template <int CHAINS, int NT, int MODE>
__device__ __forceinline__ void solve_group(const Batch &B, int group, int groups)
{
    constexpr int kChunk = 2;  // entries per step of a sweep (operands loaded one step ahead)
    constexpr int kSub = 8;    // the same of the substitution
    constexpr int kLook = 4;   // entries that a thread takes together in the passes over all entries
    extern __shared__ __align__(16) unsigned char smem[];
    unsigned long long *key = (unsigned long long *)smem;  // chains by (level, entry they hang off, chain)
    int *head = (int *)(key + CHAINS);                     // first entry of each chain, then the end
    int *up = head + CHAINS + 1;                           // chain above (pointer jumping)
    int *lev = up + CHAINS;                                // level; then where each level begins in key
    __shared__ int64_t s_off[kMaxTrees + 1];
    __shared__ int s_warp[kLook * NT / 32], s_bad, s_K, s_go, s_lev, s_long;
    static_assert(kMaxTrees < NT + 1 && (CHAINS & (CHAINS - 1)) == 0 && CHAINS <= 8192, "table sizes");
    constexpr unsigned long long kChain = 0x1FFF;  // a key: level << 43 | entry << 13 | chain
    const int tid = threadIdx.x, lane = tid & 31;
    const int32_t t0 = group * B.trees_per_block, t1 = min(t0 + B.trees_per_block, B.n_trees);
    const int nt = t1 - t0;
    if (tid == 0) s_bad = s_K = s_lev = s_long = 0;
    if (tid <= nt) s_off[tid] = B.off[t0 + tid];
    if (tid == 0 && nt == NT) s_off[nt] = B.off[t1];
    __syncthreads();
    if (tid < nt) {
        if (s_off[tid] < 0 || s_off[tid + 1] < s_off[tid] || s_off[tid + 1] > B.n_comp) s_bad = 1;
        else atomicMax(&s_long, (int)min(s_off[tid + 1] - s_off[tid], (int64_t)0x7FFFFFFF));
    }
    __syncthreads();
    const int64_t base = s_off[0];
    const int64_t total = s_off[nt] - base;
    if (MODE == kCount && (s_bad || total > 0x3FFFFFFF)) return;
    if (s_bad || total > 0x3FFFFFFF || s_long <= kTiny) {
        if (tid < nt) solve_serial(B, t0 + tid);
        return;
    }
    const int n = (int)total;
    if (n == 0) return;
    const int32_t *parent = B.parent + base;
    const double *a = B.a + base, *b = B.b + base, *c = B.c + base, *rhs = B.rhs + base;
    double *x = B.x + base, *work = B.work + base;

    // the first entry of entry i's tree, relative to the block's
    auto tree_base = [&](int i) {
        int lo = 0, hi = nt;  // last tree with s_off <= i (empty trees end where they begin)
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (s_off[mid] - base <= i) lo = mid; else hi = mid;
        }
        return (int)(s_off[lo] - base);
    };
    // 1. the parent rule, and the chains' first entries in order
    int stop = 0;  // 1: an invalid tree, 2: more chains than the tables hold
    for (int i0 = 0; i0 < n && !stop; i0 += kLook * NT) {
        int p[kLook];
#pragma unroll
        for (int u = 0; u < kLook; ++u) p[u] = i0 + u * NT + tid < n ? parent[i0 + u * NT + tid] : 0;
        bool first[kLook], bad = false;
        unsigned m[kLook];
#pragma unroll
        for (int u = 0; u < kLook; ++u) {
            const int i = i0 + u * NT + tid;
            first[u] = false;
            if (i < n) {
                const int tb = tree_base(i);
                bad |= i == tb ? p[u] != -1 : p[u] < 0 || p[u] >= i - tb;
                first[u] = i == tb || tb + p[u] != i - 1;
            }
            m[u] = __ballot_sync(0xFFFFFFFFu, first[u]);
            if (lane == 0) s_warp[u * (NT / 32) + (tid >> 5)] = __popc(m[u]);
        }
        __syncthreads();
        int k = s_K;
        int last = 0;
        for (int u = 0, w = 0; u < kLook; ++u) {
            for (; w < u * (NT / 32) + (tid >> 5); ++w) k += s_warp[w];
            last = k + __popc(m[u] & ((1u << lane) - 1u));
            if (first[u] && last < CHAINS) head[last] = i0 + u * NT + tid;
            last += first[u] ? 1 : 0;
        }
        __syncthreads();
        if (tid == NT - 1) s_K = last;
        if (__syncthreads_or(bad)) stop = 1;
        else if (s_K > CHAINS) stop = 2;
    }
    if (MODE == kCount && stop) return;
    if (stop == 1) {
        if (tid < nt) solve_serial(B, t0 + tid);
        return;
    }
    // leaves the group to hines_left_kernel (1) or hines_rest_kernel (2)
    auto leave = [&](int list) {
        if (tid == 0) {
            const int q = atomicAdd(B.status + list, 1);
            s_go = q < B.left_cap;
            if (s_go) B.left[(list - 1) * B.left_cap + q] = group;
        }
        __syncthreads();
        if (!s_go && tid < nt) solve_serial(B, t0 + tid);
    };
    if (stop == 2) {  // more chains than the tables hold
        leave(MODE == kFirst ? 1 : 2);
        return;
    }
    const int K = s_K;
    if (tid == 0) head[K] = n;
    __syncthreads();
    // 2. the entry each chain hangs off, the chain it belongs to, and levels
    //    by pointer jumping over these
    int P2 = 32;
    while (P2 < K) P2 <<= 1;
    for (int k = tid; k < P2; k += NT) {
        unsigned long long v = ~0ull;
        if (k < K) {
            const int i = head[k], p = parent[i];
            int u = -1, q = 0;
            if (p >= 0) {
                q = tree_base(i) + p;
                int lo = 0, hi = k;
                while (hi - lo > 1) {
                    const int mid = (lo + hi) >> 1;
                    if (head[mid] <= q) lo = mid; else hi = mid;
                }
                u = lo;
            }
            up[k] = u;
            lev[k] = u >= 0;
            v = ((unsigned long long)q << 13) | (unsigned)k;
        }
        key[k] = v;
    }
    for (;;) {
        __syncthreads();
        if (tid == 0) s_go = 0;
        __syncthreads();
        // rounds of NT chains read before they write; a chain's value counts
        // the levels up to its `up`, whichever round that came from
        for (int k0 = 0; k0 < K; k0 += NT) {
            const int k = k0 + tid;
            int u = -1, l = 0;
            const bool act = k < K && up[k] >= 0;
            if (act) {
                l = lev[k] + lev[up[k]];
                u = up[up[k]];
            }
            __syncthreads();
            if (act) {
                lev[k] = l;
                up[k] = u;
                if (u >= 0) s_go = 1;
            }
            __syncthreads();
        }
        if (!s_go) break;
    }
    int deepest = 0;
    for (int k = tid; k < K; k += NT) deepest = max(deepest, lev[k]);
    deepest = __reduce_max_sync(0xFFFFFFFFu, deepest);
    if (lane == 0) atomicMax(&s_lev, deepest);
    __syncthreads();
    const int levels = s_lev + 1;
    if (MODE == kCount) {
        if (tid == 0) {
            atomicAdd(B.status + 3, 1);
            atomicAdd(B.status + 4, levels);
            atomicMax(B.status + 5, s_long);
        }
        return;
    }
    // Deep trees of many groups are left to a thread each (see deep_batch; here
    // with six blocks on an SM).  Trees of under 64 levels, or of more than 16
    // entries to a level, are never that slow: without these two conditions the
    // small ones of 3,000 trees of 50 to 5,000 went there too, 1.24 ms instead
    // of 0.89.  3,000 combs of 1,000 entries and 500 levels 3.15 -> 2.75 ms,
    // 20,000 of 200 1.38 -> 0.86 ms.
    if (MODE == kFirst && levels >= 64 && 16LL * levels >= s_long &&
        8LL * max(groups, kSmallSlots) * (levels + 30) > 6LL * kSmallSlots * s_long) {
        leave(2);
        return;
    }
    // (x may be rhs: the copy leaves it as it is, for solve_serial)
    bool other = false;    // rows that the sweeps are not for
    uint32_t largest = 0;  // high_word of the couplings
    for (int i0 = tid; i0 < n; i0 += kLook * NT) {
        double bv[kLook], rv[kLook];
#pragma unroll
        for (int u = 0; u < kLook; ++u) {
            const int i = min(i0 + u * NT, n - 1);
            bv[u] = b[i];
            rv[u] = rhs[i];
            other |= !ordinary_row(bv[u], rv[u]);
            if (B.x == B.rhs && parent[i] >= 0) largest = max(largest, high_word(a[i], c[i]));
        }
#pragma unroll
        for (int u = 0; u < kLook; ++u) {
            const int i = i0 + u * NT;
            if (i < n) {
                work[i] = bv[u];
                x[i] = rv[u];
            }
        }
    }
    if (__syncthreads_or(other || largest > kCouplingMax)) {
        if (tid < nt) solve_serial(B, t0 + tid);
        return;
    }
    // 3. the chains by level and the entry they hang off (bitonic), and where
    //    each level begins
    for (int k = tid; k < K; k += NT) key[k] |= (unsigned long long)lev[k] << 43;
    for (int size = 2; size <= P2; size <<= 1)
        for (int stride = size >> 1; stride > 0; stride >>= 1) {
            __syncthreads();
            for (int q = tid; q < P2 / 2; q += NT) {
                const int i = 2 * q - (q & (stride - 1)), j = i + stride;
                const unsigned long long u = key[i], v = key[j];
                if ((u > v) == ((i & size) == 0)) {
                    key[i] = v;
                    key[j] = u;
                }
            }
        }
    __syncthreads();
    const int nlev = (int)(key[K - 1] >> 43) + 1;
    int *lbeg = lev;
    for (int q = tid; q < K; q += NT) {
        const int l = (int)(key[q] >> 43);
        if (q == 0 || (int)(key[q - 1] >> 43) != l) lbeg[l] = q;
    }
    __syncthreads();
    auto level_end = [&](int l) { return l + 1 < nlev ? lbeg[l + 1] : K; };

    // 4. elimination, deepest level first
    for (int l = nlev - 1; l >= 0; --l) {
        const int q0 = lbeg[l], q1 = level_end(l);
        for (int w0 = q0 + (tid & ~31); w0 < q1; w0 += NT) {
            // whole warps, to the longest chain's end (lanes without a chain
            // sweep none), so that the division below is done once
            const bool has = w0 + lane < q1;
            const int k = has ? (int)(key[w0 + lane] & kChain) : 0, h = head[k];
            int j = has ? head[k + 1] - 1 : h - 1;
            const int steps = __reduce_max_sync(0xFFFFFFFFu, j - h + 1);
            double an[kChunk], cn[kChunk], bn[kChunk], rn[kChunk];
            auto load = [&](int jj) {
#pragma unroll
                for (int z = 0; z < kChunk; ++z) {
                    const int i = max(jj - z, h);
                    an[z] = __ldg(a + i);
                    cn[z] = __ldg(c + i);
                    bn[z] = work[i];
                    rn[z] = x[i];
                }
            };
            if (has) load(j);
            Front F{1.0, 0.0, 0.0};     // below the leaf: N = b, S = rhs
            double ab = 0.0, cb = 0.0;  // a and c of the entry below
            double N = 0.0, S = 0.0, M = 0.0;
            for (int t = 0; t < steps; t += kChunk, j -= kChunk) {
                double av[kChunk], cv[kChunk], bv[kChunk], rv[kChunk];
#pragma unroll
                for (int z = 0; z < kChunk; ++z) {
                    av[z] = an[z];
                    cv[z] = cn[z];
                    bv[z] = bn[z];
                    rv[z] = rn[z];
                }
                if (j - kChunk >= h) load(j - kChunk);
#pragma unroll
                for (int z = 0; z < kChunk; ++z) {
                    const int i = j - z;
                    if (i >= h) {
                        N = fma(bv[z], F.N, -((ab * F.M) * cb));
                        S = fma(rv[z], F.N, -(ab * F.S));
                        M = F.N;
                        ab = av[z];
                        cb = cv[z];
                        if (l > 0 || i > h) largest = max(largest, high_word(ab, cb));
                        if (i > h) {
                            work[i] = N;
                            x[i] = S;
                        }
                        F = Front{N, M, S};
                        F.normalise();
                    }
                }
            }
            if (has) {
                const double inv = reciprocal(N);
                work[h] = -divide(cb * M, N, inv);
                x[h] = divide(S, N, inv);
            }
        }
        __syncthreads();
        if (l == 0) break;
        for (int q = q0 + tid; q < q1; q += NT) {
            const unsigned long long run = key[q] >> 13;  // level and entry
            if (q + 1 < q1 && (key[q + 1] >> 13) == run) continue;  // not the last of its run
            const int p = (int)(run & 0x3FFFFFFF);
            double bp = work[p], rp = x[p];
            for (int z = q; z >= q0 && (key[z] >> 13) == run; --z) {
                const int h = head[key[z] & kChain];
                const double ah = __ldg(a + h);
                bp = fma(ah, work[h], bp);
                rp = fma(-ah, x[h], rp);
            }
            work[p] = bp;
            x[p] = rp;
        }
        __syncthreads();
    }
    if (B.x != B.rhs && __syncthreads_or(largest > kCouplingMax)) {
        if (tid < nt) solve_serial(B, t0 + tid);
        return;
    }
    // 5. the division of every entry that is not a chain's first
    for (int i0 = 0; i0 < n; i0 += kLook * NT) {
        bool todo[kLook];
        double N[kLook], M[kLook], S[kLook], cc[kLook];
#pragma unroll
        for (int u = 0; u < kLook; ++u) {
            const int i = i0 + u * NT + tid;
            todo[u] = false;
            if (i < n) {
                const int tb = tree_base(i);
                todo[u] = i != tb && tb + parent[i] == i - 1;
                N[u] = work[i];
                S[u] = x[i];
                cc[u] = __ldg(c + i);
                M[u] = i + 1 < n && parent[i + 1] >= 0 && tb + parent[i + 1] == i ? mmk::mantissa(work[i + 1]) : 1.0;
            }
        }
        __syncthreads();  // the entry above has read this one's N
#pragma unroll
        for (int u = 0; u < kLook; ++u) {
            const int i = i0 + u * NT + tid;
            if (todo[u]) {
                const double inv = reciprocal(N[u]);
                work[i] = -divide(cc[u] * M[u], N[u], inv);
                x[i] = divide(S[u], N[u], inv);
            }
        }
    }
    __syncthreads();
    // 6. substitution, roots first
    for (int l = 0; l < nlev; ++l) {
        const int q1 = level_end(l);
        for (int q = lbeg[l] + tid; q < q1; q += NT) {
            const int k = (int)(key[q] & kChain), h = head[k], e = head[k + 1];
            double xv = x[h];
            if (l > 0) {
                xv = fma(work[h], x[(key[q] >> 13) & 0x3FFFFFFF], xv);
                x[h] = xv;
            }
            double fn[kSub], sn[kSub];
            auto load = [&](int jj) {
#pragma unroll
                for (int z = 0; z < kSub; ++z) {
                    const int i = min(jj + z, e - 1);
                    fn[z] = work[i];
                    sn[z] = x[i];
                }
            };
            int j = h + 1;
            if (j < e) load(j);
            for (; j < e; j += kSub) {
                double fv[kSub], sv[kSub];
#pragma unroll
                for (int z = 0; z < kSub; ++z) {
                    fv[z] = fn[z];
                    sv[z] = sn[z];
                }
                if (j + kSub < e) load(j + kSub);
#pragma unroll
                for (int z = 0; z < kSub; ++z) {
                    if (j + z < e) {
                        xv = fma(fv[z], xv, sv[z]);
                        x[j + z] = xv;
                    }
                }
            }
        }
        __syncthreads();
    }
}

template <int CHAINS, int NT, int BLOCKS>
__global__ void __launch_bounds__(NT, BLOCKS) hines_batch_kernel(Batch B)
{
    solve_group<CHAINS, NT, kFirst>(B, blockIdx.x, gridDim.x);
}

// The groups of trees that hines_batch_kernel left, with a larger table.
template <int CHAINS, int NT>
__global__ void __launch_bounds__(NT, 1) hines_left_kernel(Batch B)
{
    const int left = min(B.status[1], B.left_cap);
    for (int q = blockIdx.x; q < left; q += gridDim.x) {
        solve_group<CHAINS, NT, kLeft>(B, B.left[q], left);
        __syncthreads();
    }
}

// The levels of some of the groups left (a block each, evenly over the list).
template <int CHAINS, int NT>
__global__ void __launch_bounds__(NT, 1) hines_look_kernel(Batch B)
{
    const int left = min(B.status[1], B.left_cap);
    solve_group<CHAINS, NT, kCount>(B, B.left[(int64_t)blockIdx.x * left / gridDim.x], left);
}

// The trees of one of the lists, a thread for each tree, so that all of them run
// side by side: 40 trees of 20,000 entries before 60,000 of 50, which fall into
// two groups, 892 ms with a thread per group, 46 ms so.  lanes: a power of two,
// threads for each group.
__global__ void __launch_bounds__(128) hines_rest_kernel(Batch B, int list, int lanes)
{
    const int left = min(B.status[list], B.left_cap);
    for (int64_t i = blockIdx.x * 128LL + threadIdx.x; i < (int64_t)left * lanes; i += gridDim.x * 128LL) {
        const int64_t t0 = (int64_t)B.left[(list - 1) * B.left_cap + i / lanes] * B.trees_per_block;
        const int64_t t1 = min(t0 + B.trees_per_block, (int64_t)B.n_trees);
        for (int64_t t = t0 + i % lanes; t < t1; t += lanes) solve_serial(B, (int32_t)t);
    }
}

// Whether `left` groups, of which `some` have `levels` levels together and no
// tree of more than `longest` entries, are solved sooner by a thread per tree than
// one to an SM with the larger tables.  A level costs a block 1.7 us of barriers
// and dependent loads whatever it holds, what comes before and after the sweeps
// about 30 levels; a thread costs 2 us an entry, but all trees of the batch run
// at once.  One answer for all of them: where only some go to a thread, the
// others take their time besides (3,000 trees of 1,500 entries numbered breadth
// first, some 120 levels: 5.3 ms all with tables, 4.9 all with threads, 7.2
// mixed).  3,000 combs of 3,000 entries and 1,500 levels: 48 ms with tables, 7.9
// with threads, 7.8 so; 2,000 stars of 4,000, two levels, 10.3 and 12.3.
bool deep_batch(int left, int some, int levels, int longest)
{
    return some > 0 && 1.7 * ((double)levels / some + 30.0) * left / kSms > 2.0 * longest;
}

// The status words, once what was queued on the stream is done.
mm_status read_status(const Batch &B, cudaStream_t s, int h[6])
{
    if (cudaMemcpyAsync(h, B.status, 6 * sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess) return MM_ECUDA;
    return cudaStreamSynchronize(s) == cudaSuccess ? MM_OK : MM_ECUDA;
}

mm_status run_batch(Batch B, cudaStream_t s)
{
    int h[6] = {};
    if (cudaMemsetAsync(B.status, 0, 6 * sizeof(int), s) != cudaSuccess) return MM_ECUDA;
    if (B.n_trees > 0 && B.n_comp > 0) {
        // trees per block: about kBlockComps entries, fewer where the batch
        // would not fill the chip's slots otherwise, at least one tree.  The
        // tables of 1,024 chains leave room for six blocks per SM; groups with
        // more chains are taken up by a second launch with one block per SM, and
        // the rest by a third, which the host makes only where a group was left
        // (it waits for the solve in any case: 12 us of every other call)
        constexpr auto small = hines_batch_kernel<kSmallChains, 128, 6>;
        constexpr auto large = hines_left_kernel<kLargeChains, 256>;
        const int64_t mean = std::max<int64_t>(1, B.n_comp / B.n_trees);
        const int64_t trees = std::min<int64_t>(kBlockComps, B.n_comp / kSmallSlots) / mean;
        B.trees_per_block = (int32_t)std::min<int64_t>(kMaxTrees, std::max<int64_t>(1, trees));
        const int64_t blocks = ((int64_t)B.n_trees + B.trees_per_block - 1) / B.trees_per_block;
        small<<<(unsigned)blocks, 128, smem_of(kSmallChains), s>>>(B);
        if (cudaGetLastError() != cudaSuccess) return MM_ECUDA;
        mm_status st = read_status(B, s, h);
        if (st != MM_OK) return st;
        if (h[1] > 0 || h[2] > 0) {
            constexpr auto look = hines_look_kernel<kLargeChains, 256>;
            if (cudaFuncSetAttribute(large, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of(kLargeChains)) !=
                    cudaSuccess ||
                cudaFuncSetAttribute(look, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_of(kLargeChains)) !=
                    cudaSuccess)
                return MM_ECUDA;
            const int left = std::min(h[1], B.left_cap);
            bool deep = false;  // never with two groups to an SM or fewer: levels are at most half the entries
            if (left > 2 * kSms) {
                look<<<kSms, 256, smem_of(kLargeChains), s>>>(B);
                if (cudaGetLastError() != cudaSuccess) return MM_ECUDA;
                if ((st = read_status(B, s, h)) != MM_OK) return st;
                deep = deep_batch(left, h[3], h[4], h[5]);
            }
            if (left > 0 && !deep) large<<<(unsigned)std::min(left, kSms), 256, smem_of(kLargeChains), s>>>(B);
            int lanes = 1;
            while (lanes < B.trees_per_block) lanes *= 2;
            const int64_t rest = (int64_t)B.left_cap * lanes;
            const unsigned rest_blocks = (unsigned)std::min<int64_t>((rest + 127) / 128, kSms * 16);
            if (deep) hines_rest_kernel<<<rest_blocks, 128, 0, s>>>(B, 1, lanes);
            hines_rest_kernel<<<rest_blocks, 128, 0, s>>>(B, 2, lanes);
            if (cudaGetLastError() != cudaSuccess) return MM_ECUDA;
            if ((st = read_status(B, s, h)) != MM_OK) return st;
        }
    }
    return h[0] ? MM_EINVAL : MM_OK;
}

bool args_ok(int32_t n_trees, int64_t n_comp, const int64_t *off, const int32_t *parent, const double *a,
             const double *b, const double *c, const double *rhs, double *x)
{
    if (n_trees < 0 || n_comp < 0) return false;
    if (n_trees > 0 && !off) return false;
    if (n_comp > 0 && (!parent || !a || !b || !c || !rhs || !x)) return false;
    return true;
}

}  // namespace

extern "C" mm_status mm_hines_solve(int32_t n_trees, int64_t n_comp, const int64_t *tree_offset,
                                    const int32_t *parent, const double *a, const double *b, const double *c,
                                    const double *rhs, double *x, void *cuda_stream)
{
    if (!args_ok(n_trees, n_comp, tree_offset, parent, a, b, c, rhs, x)) return MM_EINVAL;
    cudaStream_t s = (cudaStream_t)cuda_stream;
    // scratch: the working values of the diagonal, the status words, the lists
    const size_t values = (size_t)(n_comp > 0 ? n_comp : 1) * sizeof(double);
    const int32_t cap = left_cap_of(n_comp);
    const size_t bytes = values + 256 + 2 * (size_t)cap * sizeof(int32_t);
    void *scratch = nullptr;
    if (cudaMalloc(&scratch, bytes) != cudaSuccess) {
        cudaGetLastError();
        return MM_ENOMEM;
    }
    double *work = (double *)scratch;
    int *status = (int *)((char *)scratch + values);
    const mm_status st =
        run_batch({n_trees, n_comp, tree_offset, parent, a, b, c, rhs, x, work, status, status + 64, cap, 1}, s);
    cudaFree(scratch);
    return st;
}

// The device address of g_noalloc_scratch is looked up on every call, with
// the caller's device current: in host code the array's name is only a
// host-side stand-in, and a cached address could outlive the module it
// points into (a cudaDeviceReset reloads it).  The lookup allocates nothing.
extern "C" mm_status mm_hines_solve_noalloc(int32_t n_trees, int64_t n_comp, const int64_t *tree_offset,
                                            const int32_t *parent, const double *a, const double *b,
                                            const double *c, const double *rhs, double *x, void *cuda_stream)
{
    if (!args_ok(n_trees, n_comp, tree_offset, parent, a, b, c, rhs, x)) return MM_EINVAL;
    if (n_comp > MM_NOALLOC_MAX_COMPS) return MM_EINVAL;
    void *base = nullptr;
    if (cudaGetSymbolAddress(&base, g_noalloc_scratch) != cudaSuccess || !base) {
        cudaGetLastError();
        return MM_ECUDA;
    }
    int *status = (int *)base;                                     // cleared by run_batch before the kernels
    double *work = (double *)base + 32 + MM_NOALLOC_LEFT;          // written before it is read, as the lists are
    return run_batch({n_trees, n_comp, tree_offset, parent, a, b, c, rhs, x, work, status, status + 64,
                      left_cap_of(n_comp), 1},
                     (cudaStream_t)cuda_stream);
}
