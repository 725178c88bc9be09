// k_variation.cu -- InitializePopulation and the offspring map of Alg. 1:
// topology-aware crossover (Sec. 4.3.1, Alg. 2) and topology-aware mutation
// (Sec. 4.3.2), for all N_p children of a generation at once.
//
// Both kernels work on node-major rows: a warp owns node v; lane q owns the
// four children 4q..4q+3, which share one Philox call per stage because the
// stream counter of (child i, node v) is (v, i / 4, g, stage), word i % 4.
#include <limits.h>

#include <utility>

#include "mocd_check.cuh"
#include "mocd_internal.h"
#include "philox.cuh"

namespace mocd {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// ---------------------------------------------------------------------------
// InitializePopulation: label of (individual i, node v) = pick(u, n), u the
// INIT word of (v, i) at generation 0.
// ---------------------------------------------------------------------------
__global__ void init_population_kernel(int n, int W, int np, uint32_t k0, uint32_t k1,
                                       int32_t *__restrict__ dst)
{
    const int nq = W >> 2;
    const long long total = (long long)n * nq;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const int v = (int)(t / nq);
        const int q = (int)(t % nq);
        const uint4 r = philox4x32_10(make_uint4((uint32_t)v, (uint32_t)q, 0u, kStageInit), k0, k1);
        int4 o;
        o.x = 4 * q + 0 < np ? (int)pick_index(r.x, (uint32_t)n) : 0;
        o.y = 4 * q + 1 < np ? (int)pick_index(r.y, (uint32_t)n) : 0;
        o.z = 4 * q + 2 < np ? (int)pick_index(r.z, (uint32_t)n) : 0;
        o.w = 4 * q + 3 < np ? (int)pick_index(r.w, (uint32_t)n) : 0;
        reinterpret_cast<int4 *>(dst)[t] = o;
    }
}

// ---------------------------------------------------------------------------
// Hybrid initialisation (init_mode 1): every node starts as its own community
// and then takes one synchronous neighbour-majority step at full rate, the tie
// broken by the INIT word of (v, i). In a singleton partition the labels of
// v's neighbours are their ids, all distinct because the uploaded adjacency
// has no repeats, so every neighbour ties at count 1 and the tied labels in
// ascending order are the adjacency row itself (it is stored sorted). The
// step therefore reads entry pick(u, deg v) of the row; a node of degree 0
// keeps label v.
// ---------------------------------------------------------------------------
__global__ void init_sweep_kernel(int n, int W, int np, uint32_t k0, uint32_t k1,
                                  const int32_t *__restrict__ row_ptr,
                                  const int32_t *__restrict__ col_idx, int32_t *__restrict__ dst)
{
    const int nq = W >> 2;
    const long long total = (long long)n * nq;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const int v = (int)(t / nq);
        const int q = (int)(t % nq);
        const int beg = __ldg(row_ptr + v);
        const uint32_t d = (uint32_t)(__ldg(row_ptr + v + 1) - beg);
        int4 o = make_int4(v, v, v, v);
        if (d > 0) {
            const uint4 r = philox4x32_10(make_uint4((uint32_t)v, (uint32_t)q, 0u, kStageInit), k0, k1);
            o.x = __ldg(col_idx + beg + pick_index(r.x, d));
            o.y = __ldg(col_idx + beg + pick_index(r.y, d));
            o.z = __ldg(col_idx + beg + pick_index(r.z, d));
            o.w = __ldg(col_idx + beg + pick_index(r.w, d));
        }
        if (4 * q + 0 >= np) o.x = 0;
        if (4 * q + 1 >= np) o.y = 0;
        if (4 * q + 2 >= np) o.z = 0;
        if (4 * q + 3 >= np) o.w = 0;
        reinterpret_cast<int4 *>(dst)[t] = o;
    }
}

// ---------------------------------------------------------------------------
// Crossover. Row v of R = (P half | Q) is staged in shared memory; the next P
// (environmental selection's keep list) is compacted into the other P half,
// and child i of the generation gets
//   copy_r[i] >= 0 : R_v[copy_r[i]]                    (x > C_P: random parent)
//   otherwise      : majority of R_v[par_r[i][j]], j < E_S, the tie among the t
//                    most frequent labels broken by the XTIE word: the
//                    pick(u, t)-th smallest of them (Eq. arg_max).
// ---------------------------------------------------------------------------

// Count of the maximal label and number t of distinct labels reaching it.
template <int EMAX>
__device__ __forceinline__ int mode_ties(const int (&x)[EMAX], int E, int &best)
{
    int cnt[EMAX];
#pragma unroll
    for (int a = 0; a < EMAX; ++a) {
        cnt[a] = 0;
#pragma unroll
        for (int b = 0; b < EMAX; ++b)
            if (a < E && b < E && x[b] == x[a]) cnt[a] += 1;
    }
    best = 0;
#pragma unroll
    for (int a = 0; a < EMAX; ++a)
        if (a < E && cnt[a] > best) best = cnt[a];
    int t = 0;
#pragma unroll
    for (int a = 0; a < EMAX; ++a) {
        bool first = a < E && cnt[a] == best;
#pragma unroll
        for (int b = 0; b < EMAX; ++b)
            if (b < a && x[b] == x[a]) first = false;
        t += first ? 1 : 0;
    }
    // Distinct maximal labels: a label's first occurrence is counted once.
    return t;
}

// The k-th smallest distinct label among those of count `best`.
template <int EMAX>
__device__ __forceinline__ int kth_tied(const int (&x)[EMAX], int E, int best, int k)
{
    int res = x[0];
#pragma unroll
    for (int a = 0; a < EMAX; ++a) {
        if (a >= E) continue;
        int c = 0;
        bool first = true;
#pragma unroll
        for (int b = 0; b < EMAX; ++b) {
            if (b >= E) continue;
            c += x[b] == x[a];
            if (b < a && x[b] == x[a]) first = false;
        }
        if (!first || c != best) continue;
        // rank of x[a] among the distinct tied labels
        int rank = 0;
#pragma unroll
        for (int b = 0; b < EMAX; ++b) {
            if (b >= E) continue;
            int cb = 0;
            bool fb = true;
#pragma unroll
            for (int e = 0; e < EMAX; ++e) {
                if (e >= E) continue;
                cb += x[e] == x[b];
                if (e < b && x[e] == x[b]) fb = false;
            }
            if (fb && cb == best && x[b] < x[a]) rank += 1;
        }
        if (rank == k) res = x[a];
    }
    return res;
}

template <int EMAX>
__device__ __forceinline__ void crossover_body(const GenParams gp, const int32_t *buf0, const int32_t *buf1,
                                               int32_t *out0, int32_t *out1, const int32_t *__restrict__ q,
                                               int32_t *__restrict__ child, const int32_t *__restrict__ keep,
                                               const int32_t *__restrict__ par_r, const int32_t *__restrict__ copy_r,
                                               const uint32_t *__restrict__ gen_ptr, int *__restrict__ dcount,
                                               int vblock, int vgrid)
{
    // The mutation kernel that follows appends deferred pairs from zero, and
    // counts the own label first if that settled at least half of the last
    // generation's sampled pairs.
    if (vblock == 0 && threadIdx.x == 0) {
        const int pairs = dcount[kDcountPairs], ok = dcount[kDcountOk];
        dcount[kDcountFast] = pairs > 0 && 2 * ok >= pairs ? 1 : 0;
        for (int k = 0; k <= kDcountOk; ++k) dcount[k] = 0;
    }
    extern __shared__ int smem[];
    const int W = gp.W, np = gp.np, E = gp.es;
    const int nq = W >> 2;
    // Per-child tables, stored so that lane q reading child 4q + k hits bank q:
    // entry (k, q) of a table lives at [k * 32 + q] (and [(j * 4 + k) * 32 + q]
    // for parent j).
    int *s_keep = smem;                    // row position of P position i
    int *s_copy = s_keep + kMaxPop;        // row position copied, or -1
    int *s_par = s_copy + kMaxPop;         // row positions of parents
    int *s_rows = s_par + kMaxPop * EMAX;  // per warp: [2W] staged row of R

    const uint32_t g = *gen_ptr;
    // R index r -> position in the staged row (P half at [0, W), Q at [W, 2W)).
    for (int t = threadIdx.x; t < np; t += blockDim.x) {
        const int slot = (t & 3) * 32 + (t >> 2);
        int r = keep[t];
        if (!MOCD_CHECK(r >= 0 && r < 2 * np, kCheckRIndex, t)) r = 0;
        s_keep[slot] = r < np ? r : W + (r - np);
        int c = copy_r[t];
        if (!MOCD_CHECK(c >= -1 && c < 2 * np, kCheckRIndex, t)) c = 0;
        s_copy[slot] = c < 0 ? -1 : (c < np ? c : W + (c - np));
        for (int j = 0; j < E; ++j) {
            int p = par_r[t * kMaxParents + j];
            if (!MOCD_CHECK(p >= 0 && p < 2 * np, kCheckRIndex, t)) p = 0;
            s_par[(j * 4 + (t & 3)) * 32 + (t >> 2)] = p < np ? p : W + (p - np);
        }
    }
    __syncthreads();

    // Generation g reads the P half buf[g & 1] and writes the compacted P
    // into the other half (the two never alias within one launch).
    const int4 *P4 = reinterpret_cast<const int4 *>((g & 1u) ? buf1 : buf0);
    int4 *D4 = reinterpret_cast<int4 *>((g & 1u) ? out0 : out1);
    const int4 *__restrict__ Q4 = reinterpret_cast<const int4 *>(q);
    int4 *__restrict__ C4 = reinterpret_cast<int4 *>(child);

    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    int *row = s_rows + wib * 2 * W;
    const int warp = (vblock * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (vgrid * blockDim.x) >> 5;
    const bool active = lane < nq;

    // Software pipeline: the next node's rows are requested before the
    // current node is processed.
    int4 cur_p = make_int4(0, 0, 0, 0), cur_q = make_int4(0, 0, 0, 0);
    if (active && warp < gp.n) {
        cur_p = P4[(size_t)warp * nq + lane];
        cur_q = Q4[(size_t)warp * nq + lane];
    }
    for (int v = warp; v < gp.n; v += nwarps) {
        const int vn = v + nwarps;
        int4 nxt_p = make_int4(0, 0, 0, 0), nxt_q = make_int4(0, 0, 0, 0);
        if (active && vn < gp.n) {
            nxt_p = P4[(size_t)vn * nq + lane];
            nxt_q = Q4[(size_t)vn * nq + lane];
        }
        if (active) {
            reinterpret_cast<int4 *>(row)[lane] = cur_p;
            reinterpret_cast<int4 *>(row + W)[lane] = cur_q;
        }
        cur_p = nxt_p;
        cur_q = nxt_q;
        __syncwarp();
        if (active && EMAX == 4 && E == 4) {
            // Sort each child's four votes (5 comparators); the run pattern of
            // the sorted values gives the maximal labels in ascending order:
            // t = 4 (all distinct), t = 2 (two pairs) or a unique maximum. All
            // four children are classified first so that the lane's tie word
            // (one Philox call for its four children) is computed at most once.
            int o[4], srt[4][4], tk[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = 4 * lane + k;
                o[k] = i < np ? row[s_keep[k * 32 + lane]] : 0;
                const int cp = i < np ? s_copy[k * 32 + lane] : 0;
                // Children past N_p (padding of the last quad) have no parent table.
                const bool real = i < np;
                int s0 = row[real ? s_par[(0 * 4 + k) * 32 + lane] : 0];
                int s1 = row[real ? s_par[(1 * 4 + k) * 32 + lane] : 0];
                int s2 = row[real ? s_par[(2 * 4 + k) * 32 + lane] : 0];
                int s3 = row[real ? s_par[(3 * 4 + k) * 32 + lane] : 0];
                int lo, hi;
                lo = min(s0, s1); hi = max(s0, s1); s0 = lo; s1 = hi;
                lo = min(s2, s3); hi = max(s2, s3); s2 = lo; s3 = hi;
                lo = min(s0, s2); hi = max(s0, s2); s0 = lo; s2 = hi;
                lo = min(s1, s3); hi = max(s1, s3); s1 = lo; s3 = hi;
                lo = min(s1, s2); hi = max(s1, s2); s1 = lo; s2 = hi;
                const bool e01 = s0 == s1, e12 = s1 == s2, e23 = s2 == s3;
                int t = (!e01 && !e12 && !e23) ? 4 : ((e01 && e23 && !e12) ? 2 : 1);
                int uniq = e01 ? s0 : (e12 ? s1 : s2);
                if (i >= np) {
                    t = 1;
                    uniq = 0;
                } else if (cp >= 0) {
                    t = 1;
                    uniq = row[cp];
                }
                srt[k][0] = t == 1 ? uniq : s0;
                srt[k][1] = s1;
                srt[k][2] = s2;
                srt[k][3] = s3;
                tk[k] = t;
            }
            uint4 u = make_uint4(0, 0, 0, 0);
            if (tk[0] > 1 || tk[1] > 1 || tk[2] > 1 || tk[3] > 1)
                u = philox4x32_10(make_uint4((uint32_t)v, (uint32_t)lane, g, kStageCrossTie), gp.key0, gp.key1);
            int r[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const uint32_t w = word_of(u, k);
                if (tk[k] == 4) {
                    const uint32_t kk = pick_index(w, 4u);
                    r[k] = kk == 0 ? srt[k][0] : kk == 1 ? srt[k][1] : kk == 2 ? srt[k][2] : srt[k][3];
                } else if (tk[k] == 2) {
                    r[k] = pick_index(w, 2u) == 0 ? srt[k][0] : srt[k][2];
                } else {
                    r[k] = srt[k][0];
                }
            }
            D4[(size_t)v * nq + lane] = make_int4(o[0], o[1], o[2], o[3]);
            C4[(size_t)v * nq + lane] = make_int4(r[0], r[1], r[2], r[3]);
        } else if (active) {
            int o[4];
            int r[4];
            bool have_u = false;
            uint4 u = make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const int i = 4 * lane + k;
                o[k] = i < np ? row[s_keep[k * 32 + lane]] : 0;
                r[k] = 0;
                if (i >= np) continue;
                const int cp = s_copy[k * 32 + lane];
                if (cp >= 0) {
                    r[k] = row[cp];
                    continue;
                }
                int x[EMAX];
#pragma unroll
                for (int j = 0; j < EMAX; ++j) x[j] = j < E ? row[s_par[(j * 4 + k) * 32 + lane]] : 0;
                int best;
                const int t = mode_ties<EMAX>(x, E, best);
                int kk = 0;
                if (t > 1) {
                    if (!have_u) {
                        u = philox4x32_10(make_uint4((uint32_t)v, (uint32_t)lane, g, kStageCrossTie),
                                          gp.key0, gp.key1);
                        have_u = true;
                    }
                    kk = (int)pick_index(word_of(u, k), (uint32_t)t);
                }
                r[k] = kth_tied<EMAX>(x, E, best, kk);
            }
            D4[(size_t)v * nq + lane] = make_int4(o[0], o[1], o[2], o[3]);
            C4[(size_t)v * nq + lane] = make_int4(r[0], r[1], r[2], r[3]);
        }
        __syncwarp();
    }
}

template <int EMAX>
__global__ void __launch_bounds__(kBlock)
crossover_kernel(GenParams gp, const int32_t *buf0, const int32_t *buf1, int32_t *out0, int32_t *out1,
                 const int32_t *__restrict__ q, int32_t *__restrict__ child,
                 const int32_t *__restrict__ keep, const int32_t *__restrict__ par_r,
                 const int32_t *__restrict__ copy_r, const uint32_t *__restrict__ gen_ptr,
                 int *__restrict__ dcount)
{
    crossover_body<EMAX>(gp, buf0, buf1, out0, out1, q, child, keep, par_r, copy_r, gen_ptr, dcount, blockIdx.x,
                         gridDim.x);
}

// The member of a multi-member launch that block blockIdx.x belongs to:
// members own consecutive block ranges, starts[k] .. starts[k + 1] - 1
// (empty for a member with nothing to do).
__device__ __forceinline__ int member_of_block(const int *__restrict__ starts, int count)
{
    const int b = (int)blockIdx.x;
    int lo = 0, hi = count;  // starts[lo] <= b < starts[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(starts + mid) <= b) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Crossover of every member of a batch in one launch.
template <int EMAX>
__global__ void __launch_bounds__(kBlock)
crossover_multi_kernel(const BatchMember *__restrict__ members, const int *__restrict__ starts, int count)
{
    const int k = member_of_block(starts, count);
    const BatchMember &mb = members[k];
    const PopState &ps = mb.ps;
    const int b0 = __ldg(starts + k);
    crossover_body<EMAX>(mb.gp, ps.buf[0], ps.buf[1], ps.buf[0], ps.buf[1], ps.q, ps.c, ps.keep, ps.par_r,
                         ps.copy_r, ps.gen, ps.dcount, (int)blockIdx.x - b0, __ldg(starts + k + 1) - b0);
}

// ---------------------------------------------------------------------------
// Mutation (Sec. 4.3.2). Node v of child i mutates iff its MCOIN word is
// below thr_m and deg(v) > 0; it then takes the most frequent label among its
// neighbours in the post-crossover child (synchronous: all reads come from
// `child`), the tie among the t most frequent labels broken by the MTIE word
// (the pick(u, t)-th smallest).
//
// A pair is a (node, selected child). A warp takes a batch of nodes, copies
// their rows to Q, and lists the batch's pairs; then every lane works on a
// pair of its own, so that the lanes stay full whatever number of children a
// node has selected (about 20 of 100 at M_P 0.2). In a settled population the
// result is nearly always the label the node already has, and counting the
// neighbours that hold it proves that: when it is on more than half of them
// it is the unique mode. The pairs this leaves open take the exact vote, by
// degree:
//   up to 32     in the same warp, a pair per lane: the labels are gathered
//                into registers, sorted by a merge-exchange network of 8, 12,
//                .., 28 or 32 entries (the smallest that holds the degree) and
//                the tied labels read off the runs
//   33..128      listed for mutation_vote_kernel, a pair per thread
//   129..512     a warp per pair: count table in shared memory (the node's
//                pairs are split over kWideParts warps)
//   above 512    listed for mutation_hub_kernel, a block per pair
// Whether the count of the own label is worth its pass over the neighbours is
// read from the last generation: the share of the pairs it settled (or would
// have settled), for degree <= 32 over a sample of all pairs, above per node.
//
// The neighbours come from the mutation's own adjacency: rows in processing
// order (degree descending), padded to four entries with the id n, whose
// child row holds a value above every label, so that four neighbours are one
// 16-byte load and padding needs no test.
// ---------------------------------------------------------------------------

// MTIE word of child i at node v.
__device__ __forceinline__ uint32_t tie_word(const GenParams &gp, int v, int i, uint32_t g)
{
    const uint4 r = philox4x32_10(make_uint4((uint32_t)v, (uint32_t)(i >> 2), g, kStageMutTie), gp.key0, gp.key1);
    return word_of(r, i & 3);
}

// A neighbour id read from the adjacency; in the debug build an id outside
// [0, n] is recorded and replaced by n (the padding row), so that the access
// it feeds stays in bounds.
__device__ __forceinline__ int checked_node(int u, int n)
{
    return MOCD_CHECK(u >= 0 && u <= n, kCheckNode, u) ? u : n;
}

__device__ __forceinline__ uint32_t hash_slot(int x, int hbits)
{
    return ((uint32_t)x * 2654435761u) >> (32 - hbits);
}

// Start of deferred-vote class c in the list: the classes are stored one
// after the other (written with selects: indexing the kernel parameter array
// at run time would copy it to local memory).
__device__ __forceinline__ int defer_offset(const GenParams &gp, int c)
{
    return c == 0 ? 0 : c == 1 ? gp.defer_cap[0] : gp.defer_cap[0] + gp.defer_cap[1];
}
__device__ __forceinline__ int defer_capacity(const GenParams &gp, int c)
{
    return c == 0 ? gp.defer_cap[0] : c == 1 ? gp.defer_cap[1] : gp.defer_cap[2];
}
constexpr int kLaneMax = 32;     // largest degree of the per-lane vote
constexpr int kMutBlock = 128;   // mutation threads per block
constexpr int kHubBlock = 256;   // threads per block of the hub kernel
constexpr int kBatch = 8;        // most nodes of a warp's batch

// Sorting networks for any N: Batcher's merge exchange in the form of
// Knuth, TAOCP vol. 3, Sec. 5.2.2, Algorithm M (for a power of two it is
// Batcher's odd-even merge sort: 19, 63, 191, 543 comparators for 8, 16, 32,
// 64 entries; 41, 97, 127, 161 for 12, 20, 24, 28). The comparator list is
// generated at compile time and unrolled, so every index is a constant and
// the array stays in registers.
template <int A, int B>
__device__ __forceinline__ void cmp_exchange(int *x)
{
    const int lo = min(x[A], x[B]);
    const int hi = max(x[A], x[B]);
    x[A] = lo;
    x[B] = hi;
}

template <int N>
struct MergeExchange {
    // Calls f(i, i + d) for every comparator in order (Algorithm M, steps
    // M1..M5: p = 2^(t-1), 2^(t-2), ..., 1; for each p the passes d = p,
    // q - p, ... with r = 0 then p).
    template <class F>
    static constexpr void each(F f)
    {
        int t = 0;
        while ((1 << t) < N) ++t;
        for (int p = t > 0 ? 1 << (t - 1) : 0; p > 0; p >>= 1) {
            int q = 1 << (t - 1), r = 0, d = p;
            while (d > 0) {
                for (int i = 0; i < N - d; ++i)
                    if ((i & p) == r) f(i, i + d);
                d = q - p;
                q >>= 1;
                r = p;
            }
        }
    }
    static constexpr int count()
    {
        int c = 0;
        each([&](int, int) { ++c; });
        return c;
    }
    static constexpr int C = count();
    struct List {
        int a[C > 0 ? C : 1];
        int b[C > 0 ? C : 1];
    };
    static constexpr List make()
    {
        List l{};
        int k = 0;
        each([&](int i, int j) {
            l.a[k] = i;
            l.b[k] = j;
            ++k;
        });
        return l;
    }
    static constexpr List P = make();
};

template <int N, std::size_t... K>
__device__ __forceinline__ void apply_network(int (&x)[N], std::index_sequence<K...>)
{
    (cmp_exchange<MergeExchange<N>::P.a[K], MergeExchange<N>::P.b[K]>(x), ...);
}

template <int N>
__device__ __forceinline__ void sort_network(int (&x)[N])
{
    apply_network<N>(x, std::make_index_sequence<MergeExchange<N>::C>{});
}

// x[pos] for a run-time pos < N without indexing the register array: a
// tree of selects on the bits of pos, one level per bit (LEN live entries).
template <int N, int LEN, int B>
__device__ __forceinline__ void select_level(int (&y)[N], int pos)
{
    if constexpr (LEN > 1) {
        const bool hi = (pos >> B) & 1;
#pragma unroll
        for (int k = 0; k < (LEN + 1) / 2; ++k) y[k] = (2 * k + 1 < LEN && hi) ? y[2 * k + 1] : y[2 * k];
        select_level<N, (LEN + 1) / 2, B + 1>(y, pos);
    }
}

template <int N>
__device__ __forceinline__ int select_at(const int (&x)[N], int pos)
{
    int y[N];
#pragma unroll
    for (int j = 0; j < N; ++j) y[j] = x[j];
    select_level<N, N, 0>(y, pos);
    return y[0];
}

// The first entries of the longest runs of equal values among the deg sorted
// entries behind e (bit j of e: entries j and j + 1 are equal, both < deg):
// a run of L values is L - 1 consecutive set bits; each step m &= m >> 1
// shortens every run of set bits by one, and the last non-zero m has one bit
// per longest run, at its first entry (all entries when no two are equal).
// best: the length of those runs.
__device__ __forceinline__ unsigned longest_runs(unsigned e, int deg, int &best)
{
    e &= deg >= 2 ? 0xffffffffu >> (33 - deg) : 0u;  // pairs (j, j + 1) with j + 1 < deg
    unsigned starts = deg >= 32 ? 0xffffffffu : (1u << deg) - 1u;
    best = 1;
    for (unsigned m = e; m != 0u; m &= m >> 1) {
        starts = m;
        ++best;
    }
    return starts;
}

// Position of the k-th set bit of m (k < popc(m)), halving the window.
__device__ __forceinline__ int kth_bit(unsigned m, unsigned k)
{
    int pos = 0;
#pragma unroll
    for (int w = 16; w >= 1; w >>= 1) {
        const unsigned low = m & ((1u << w) - 1u);
        const unsigned c = (unsigned)__popc(low);
        if (k >= c) {
            k -= c;
            m >>= w;
            pos += w;
        } else {
            m = low;
        }
    }
    return pos;
}

// Exact neighbour-majority of one pair by its own lane (deg <= N <= 32; 0
// for a lane without a pair): the labels are gathered into registers (the
// padding and the entries past it sort last), sorted, and the tied labels are
// the longest runs in ascending order. All lanes of the warp call together.
template <int N>
__device__ __forceinline__ int lane_vote(const GenParams &gp, const int4 *__restrict__ adj,
                                         const int32_t *__restrict__ child, int v, int i, int beg, int deg, uint32_t g,
                                         int &best)
{
    const int32_t *col = child + i;
    int x[N];
#pragma unroll
    for (int j = 0; j < N; j += 4) {
        const bool in = j < deg;
        const int4 u = in ? __ldg(adj + beg + j / 4) : make_int4(0, 0, 0, 0);
        x[j + 0] = in ? col[(size_t)checked_node(u.x, gp.n) * gp.W] : INT_MAX;
        x[j + 1] = in ? col[(size_t)checked_node(u.y, gp.n) * gp.W] : INT_MAX;
        x[j + 2] = in ? col[(size_t)checked_node(u.z, gp.n) * gp.W] : INT_MAX;
        x[j + 3] = in ? col[(size_t)checked_node(u.w, gp.n) * gp.W] : INT_MAX;
    }
    sort_network<N>(x);
    unsigned e = 0;
#pragma unroll
    for (int j = 0; j + 1 < N; ++j) e |= (x[j] == x[j + 1] ? 1u : 0u) << j;
    const unsigned starts = longest_runs(e, deg, best);
    const int t = __popc(starts);
    unsigned kk = 0;
    if (__any_sync(kFull, t > 1)) kk = t > 1 ? pick_index(tie_word(gp, v, i, g), (uint32_t)t) : 0u;
    return select_at<N>(x, kth_bit(starts, kk));
}

// Exact neighbour-majority of one pair of a node with degree kDeferMax + 1 ..
// kSharedTableMax by the whole warp: an open-addressing count table in shared
// memory, sized to the node (the smallest power of two with at least 2 deg
// slots), filled with one insert per distinct label of each 32-neighbour chunk
// (__match_any_sync gives the multiplicity). The labels reaching the largest
// count are then compacted (one slot per distinct label) and the pick(u, t)-th
// smallest of them is found either by stepping up through the minima (shallow
// ranks) or bit by bit from the top (deep ranks).
__device__ __forceinline__ int warp_mode_table(const GenParams &gp, const int32_t *__restrict__ child,
                                               const int *__restrict__ nbr, int deg, int v, int i, int *hkey,
                                               int *hcnt, uint32_t g, unsigned &best_count)
{
    const int lane = threadIdx.x & 31;
    const int W = gp.W;
    // 2 deg <= the per-warp capacity (gp.hash_size), so the table fits.
    int hbits = 8;
    while ((1 << hbits) < 2 * deg) ++hbits;
    const int HS = 1 << hbits;
    const int per_lane = HS >> 5;  // 8 .. 32
    for (int e = lane; e < HS; e += 32) {
        hkey[e] = -1;
        hcnt[e] = 0;
    }
    __syncwarp();
    for (int e0 = 0; e0 < deg; e0 += 32) {
        const bool in = e0 + lane < deg;
        int x = (int)(0x80000000u | lane);
        if (in) x = child[(size_t)checked_node(__ldg(nbr + e0 + lane), gp.n) * W + i];
        // One insert per distinct label of the chunk, with its multiplicity.
        const unsigned peers = __match_any_sync(kFull, x);
        if (in && (peers & ((1u << lane) - 1u)) == 0) {
            uint32_t h = hash_slot(x, hbits);
            // The table holds at most deg <= HS / 2 distinct labels, so an empty
            // or matching slot is always found.
            for (int probe = 0; probe < HS; ++probe) {
                const int prev = atomicCAS(hkey + h, -1, x);
                if (prev == -1 || prev == x) {
                    atomicAdd(hcnt + h, __popc(peers));
                    break;
                }
                h = (h + 1) & (uint32_t)(HS - 1);
            }
        }
    }
    __syncwarp();
    unsigned mx_l = 0;
    for (int s = 0; s < per_lane; ++s) mx_l = max(mx_l, (unsigned)hcnt[lane + 32 * s]);
    const unsigned mx = __reduce_max_sync(kFull, mx_l);
    best_count = mx;
    unsigned act = 0;
    for (int s = 0; s < per_lane; ++s)
        if ((unsigned)hcnt[lane + 32 * s] == mx) act |= 1u << s;
    // Compact the tied labels into hcnt[0, t) (the counts are no longer needed).
    const unsigned mine = (unsigned)__popc(act);
    unsigned incl = mine;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned y = __shfl_up_sync(kFull, incl, d);
        if (lane >= d) incl += y;
    }
    const int t = (int)__shfl_sync(kFull, incl, 31);
    int at = (int)(incl - mine);
    __syncwarp();
    for (int s = 0; s < per_lane; ++s)
        if ((act >> s) & 1u) hcnt[at++] = hkey[lane + 32 * s];
    __syncwarp();
    const unsigned kk = t > 1 ? pick_index(tie_word(gp, v, i, g), (uint32_t)t) : 0u;
    int res;
    if (kk > (unsigned)gp.label_bits) {
        // Deep rank: at bit b (from the top), count the tied labels that agree
        // with the bits chosen so far and have a 0 there; the rank falls among
        // them or, past them, among those with a 1. Labels are below
        // 2^label_bits.
        unsigned prefix = 0, rank = kk;
        for (int b = gp.label_bits - 1; b >= 0; --b) {
            const unsigned above = ~((2u << b) - 1u);  // the bits above b
            unsigned c = 0;
            for (int e = lane; e < t; e += 32) {
                const unsigned key = (unsigned)hcnt[e];
                c += ((key & above) == prefix && ((key >> b) & 1u) == 0u) ? 1u : 0u;
            }
            const unsigned cnt = __reduce_add_sync(kFull, c);
            if (rank >= cnt) {
                rank -= cnt;
                prefix |= 1u << b;
            }
        }
        res = (int)prefix;
    } else {
        // Shallow rank: the smallest tied label, then kk times the smallest
        // one above the previous (the tied labels are distinct, >= 0).
        int last = -1;
        for (unsigned s = 0; s <= kk; ++s) {
            unsigned my = 0xffffffffu;
            for (int e = lane; e < t; e += 32) {
                const int key = hcnt[e];
                if (key > last) my = min(my, (unsigned)key);
            }
            last = (int)__reduce_min_sync(kFull, my);
        }
        res = last;
    }
    __syncwarp();
    return res;
}

// D of the evaluation's degree histogram: child i's final label of a node of
// degree d (label-major cell label * W + i). The old value is not needed, so
// this is a reduction that does not stall.
__device__ __forceinline__ void add_degree(const GenParams &gp, uint32_t *__restrict__ hist, int label, int i, int d)
{
    if (MOCD_CHECK(label >= 0 && label < gp.n, kCheckLabel, label))
        atomicAdd(hist + (size_t)label * gp.W + i, (unsigned)d);
}

// Bit k set: child 4 * lane + k of node v mutates.
__device__ __forceinline__ unsigned selected(const GenParams &gp, int v, int lane, uint32_t g)
{
    const uint4 r = philox4x32_10(make_uint4((uint32_t)v, (uint32_t)lane, g, kStageMutCoin), gp.key0, gp.key1);
    const int i0 = 4 * lane;
    return ((i0 + 0 < gp.np && (unsigned long long)r.x < gp.thr_m) ? 1u : 0u) |
           ((i0 + 1 < gp.np && (unsigned long long)r.y < gp.thr_m) ? 2u : 0u) |
           ((i0 + 2 < gp.np && (unsigned long long)r.z < gp.thr_m) ? 4u : 0u) |
           ((i0 + 3 < gp.np && (unsigned long long)r.w < gp.thr_m) ? 8u : 0u);
}

// Node row of a warp: Q gets the children's own labels, the histogram the
// unselected ones (mutating pairs add theirs once decided), and the selected
// children go to list[total ..] tagged with `tag`. Returns their number.
__device__ __forceinline__ int take_row(const GenParams &gp, int v, int deg, bool active, const int4 &out, int lane,
                                        uint32_t g, int4 *__restrict__ Q4, uint32_t *__restrict__ hist,
                                        unsigned short *list, int total, int tag)
{
    unsigned sel = 0;
    if (active && deg > 0) sel = selected(gp, v, lane, g);
    if (active) {
        Q4[(size_t)v * (gp.W >> 2) + lane] = out;
        if (deg > 0) {
            const int i0 = 4 * lane;
            if (i0 + 0 < gp.np && !(sel & 1u)) add_degree(gp, hist, out.x, i0 + 0, deg);
            if (i0 + 1 < gp.np && !(sel & 2u)) add_degree(gp, hist, out.y, i0 + 1, deg);
            if (i0 + 2 < gp.np && !(sel & 4u)) add_degree(gp, hist, out.z, i0 + 2, deg);
            if (i0 + 3 < gp.np && !(sel & 8u)) add_degree(gp, hist, out.w, i0 + 3, deg);
        }
    }
    // Place of the lane's selected children: its count (0 .. 4) by bits.
    const unsigned lt = (1u << lane) - 1u;
    const int mine = __popc(sel);
    const unsigned b0 = __ballot_sync(kFull, mine & 1), b1 = __ballot_sync(kFull, mine & 2),
                   b2 = __ballot_sync(kFull, mine & 4);
    int at = total + __popc(b0 & lt) + 2 * __popc(b1 & lt) + 4 * __popc(b2 & lt);
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if ((sel >> k) & 1u) list[at++] = (unsigned short)(tag | (4 * lane + k));
    return __popc(b0) + 2 * __popc(b1) + 4 * __popc(b2);
}

// Deferred pairs of one class, appended by the lanes of `who` (warp-uniform).
// The capacity is the class's nodes x N_p, every pair a generation can defer:
// the check only keeps a corrupted count in bounds.
__device__ __forceinline__ void defer_pairs(const GenParams &gp, int cls, unsigned who, int node, int i, int lane,
                                            int2 *__restrict__ dlist, int *__restrict__ dcount)
{
    int first = 0;
    if (lane == 0) first = atomicAdd(dcount + cls, __popc(who));
    first = __shfl_sync(kFull, first, 0);
    if ((who >> lane) & 1u) {
        const int at = first + __popc(who & ((1u << lane) - 1u));
        if (at < defer_capacity(gp, cls)) dlist[defer_offset(gp, cls) + at] = make_int2(node, i);
    }
}

// hint of a node (or part): (pairs << 16) | pairs whose own label was on more
// than half of the neighbours, last generation; 0: no history.
__device__ __forceinline__ bool own_label_pays(uint32_t h)
{
    return h != 0u && 2u * (h & 0xffffu) >= (h >> 16);
}

// One item of the nodes above kDeferMax: a hub (idx < gp.n_hub), whose pairs
// are all listed for mutation_hub_kernel, or part `part` of a node of degree
// kDeferMax + 1 .. kSharedTableMax: the quads q with q % kWideParts == part.
__device__ __noinline__ void wide_item(const GenParams &gp, int item, const int4 *__restrict__ nodes,
                                       const int4 *__restrict__ adj, const int32_t *__restrict__ child,
                                       int32_t *__restrict__ q, uint32_t *__restrict__ hist,
                                       uint32_t *__restrict__ hint, int2 *__restrict__ dlist, int *__restrict__ dcount,
                                       unsigned short *list, int *hkey, int *hcnt, uint32_t g)
{
    const int lane = threadIdx.x & 31;
    const int nq = gp.W >> 2;
    const bool hub = item < gp.n_hub;
    const int idx = hub ? item : gp.n_hub + (item - gp.n_hub) / kWideParts;
    const int part = hub ? 0 : (item - gp.n_hub) % kWideParts;
    const int4 rec = __ldg(nodes + idx);
    const int v = rec.x, deg = rec.z;
    const bool active = lane < nq && (hub || lane % kWideParts == part);
    const int4 out = active ? reinterpret_cast<const int4 *>(child)[(size_t)v * nq + lane] : make_int4(0, 0, 0, 0);
    const int total = take_row(gp, v, deg, active, out, lane, g, reinterpret_cast<int4 *>(q), hist, list, 0, 0);
    uint32_t *h = hint + (hub ? idx : gp.n + (idx - gp.n_hub) * kWideParts + part);
    const bool fast = own_label_pays(*h);
    __syncwarp();
    if (hub) {
        // The flag travels with the pair: the hub kernel rewrites the hint.
        for (int base = 0; base < total; base += 32) {
            const bool has = base + lane < total;
            defer_pairs(gp, 2, __ballot_sync(kFull, has), idx | (fast ? kHubFast : 0), has ? list[base + lane] : 0, lane,
                        dlist, dcount);
        }
        if (lane == 0) *h = (uint32_t)total << 16;
        return;
    }
    int ok = 0;
    const int *nbr = reinterpret_cast<const int *>(adj + rec.y);
    for (int k = 0; k < total; ++k) {
        const int i = list[k];
        const int own = child[(size_t)v * gp.W + i];
        bool settled = false;
        if (fast) {
            int c = 0;
#pragma unroll 4
            for (int e = lane; e < deg; e += 32) c += child[(size_t)checked_node(__ldg(nbr + e), gp.n) * gp.W + i] == own;
            settled = 2 * __reduce_add_sync(kFull, c) > deg;
        }
        int lab = own;
        if (!settled) {
            unsigned mx = 0;
            lab = warp_mode_table(gp, child, nbr, deg, v, i, hkey, hcnt, g, mx);
            settled = !fast && lab == own && 2 * (int)mx > deg;
            if (lane == 0 && lab != own) q[(size_t)v * gp.W + i] = lab;
        }
        ok += settled ? 1 : 0;
        if (lane == 0) add_degree(gp, hist, lab, i, deg);
    }
    if (lane == 0) *h = ((uint32_t)total << 16) | (uint32_t)ok;
}

// WIDE: the graph has degrees above kDeferMax. batch: nodes a warp takes at a
// time (<= kBatch).
template <bool WIDE>
__global__ void __launch_bounds__(kMutBlock, 6)
mutation_kernel(const __grid_constant__ GenParams gp, const int4 *__restrict__ nodes, const int4 *__restrict__ adj,
                const int32_t *__restrict__ child, int32_t *__restrict__ q, const uint32_t *__restrict__ gen_ptr,
                uint32_t *__restrict__ hist, unsigned long long *__restrict__ acc, uint32_t *__restrict__ hint,
                int2 *__restrict__ dlist, int *__restrict__ dcount, int batch)
{
    __shared__ unsigned short s_list[kMutBlock / 32][kBatch * kMaxPop];
    __shared__ int4 s_rec[kMutBlock / 32][kBatch];
    __shared__ int s_ok[kMutBlock / 32][kBatch];
    extern __shared__ int s_table[];  // WIDE: per warp, keys and counts
    const int W = gp.W;
    const int nq = W >> 2;
    const uint32_t g = *gen_ptr;
    const bool lane_fast = dcount[kDcountFast] != 0;
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    unsigned short *list = s_list[wib];
    int4 *recs = s_rec[wib];
    int *oks = s_ok[wib];
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const bool active = lane < nq;
    const unsigned lt = (1u << lane) - 1u;
    const int4 *__restrict__ C4 = reinterpret_cast<const int4 *>(child);
    int4 *__restrict__ Q4 = reinterpret_cast<int4 *>(q);

    // The evaluation that follows accumulates into acc: clear it here. The
    // histogram is zero on entry (the previous evaluation's square sweep
    // cleared it) and receives D below.
    if (blockIdx.x == 0)
        for (int t = threadIdx.x; t < 2 * kMaxPop; t += blockDim.x) acc[t] = 0;

    // Nodes in degree-descending order: every warp starts with one of the
    // costliest batches, which balances the grid-stride loop.
    const int wide = WIDE ? gp.n_hub + gp.n_wide * kWideParts : 0;
    const int first = WIDE ? gp.n_hub + gp.n_wide : 0;
    const int items = wide + (gp.n - first + batch - 1) / batch;
    for (int item = warp; item < items; item += nwarps) {
        if (WIDE && item < wide) {
            wide_item(gp, item, nodes, adj, child, q, hist, hint, dlist, dcount, list,
                      s_table + wib * 2 * gp.hash_size, s_table + wib * 2 * gp.hash_size + gp.hash_size, g);
            __syncwarp();
            continue;
        }
        const int idx0 = first + (item - wide) * batch;
        const int nb = min(batch, gp.n - idx0);
        int4 rec = make_int4(0, 0, 0, 0);
        if (lane < nb) {
            rec = __ldg(nodes + idx0 + lane);
            const bool fast = rec.z <= kLaneMax ? lane_fast : own_label_pays(hint[idx0 + lane]);
            recs[lane] = make_int4(rec.x, rec.y, rec.z, fast ? rec.z : 0);  // .w: degree if the count pays
            oks[lane] = 0;
        }
        int total = 0, nsel = 0;
        int v = __shfl_sync(kFull, rec.x, 0);
        int4 nxt = active ? C4[(size_t)v * nq + lane] : make_int4(0, 0, 0, 0);
        for (int k = 0; k < nb; ++k) {
            const int deg = __shfl_sync(kFull, rec.z, k);
            const int4 out = nxt;
            const int cur = v;
            if (k + 1 < nb) {  // the next row is requested before this one is processed
                v = __shfl_sync(kFull, rec.x, k + 1);
                if (active) nxt = C4[(size_t)v * nq + lane];
            }
            const int c = take_row(gp, cur, deg, active, out, lane, g, Q4, hist, list, total, k << 7);
            nsel = lane == k ? c : nsel;
            total += c;
        }
        __syncwarp();

        // The own label's count; open pairs are compacted to the list's front.
        int open = 0, settled32 = 0;
        const bool any_fast = __any_sync(kFull, lane < nb && recs[lane < nb ? lane : 0].w != 0);
        if (!any_fast) open = total;
        for (int base = 0; any_fast && base < total; base += 32) {
            const bool has = base + lane < total;
            const int e = has ? list[base + lane] : 0;
            const int i = e & 127;
            const int4 r = recs[e >> 7];
            const int32_t *col = child + i;
            const int own = has ? col[(size_t)r.x * W] : 0;
            const int n4 = has ? (r.w + 3) >> 2 : 0;  // groups of four neighbours to count
            const int n4_max = __reduce_max_sync(kFull, n4);
            int c = 0;
            for (int j = 0; j < n4_max; j += 2) {
                const bool p0 = j < n4, p1 = j + 1 < n4;
                const int4 u0 = p0 ? __ldg(adj + r.y + j) : make_int4(0, 0, 0, 0);
                const int4 u1 = p1 ? __ldg(adj + r.y + j + 1) : make_int4(0, 0, 0, 0);
                int x[8];
                x[0] = p0 ? col[(size_t)checked_node(u0.x, gp.n) * W] : -1;
                x[1] = p0 ? col[(size_t)checked_node(u0.y, gp.n) * W] : -1;
                x[2] = p0 ? col[(size_t)checked_node(u0.z, gp.n) * W] : -1;
                x[3] = p0 ? col[(size_t)checked_node(u0.w, gp.n) * W] : -1;
                x[4] = p1 ? col[(size_t)checked_node(u1.x, gp.n) * W] : -1;
                x[5] = p1 ? col[(size_t)checked_node(u1.y, gp.n) * W] : -1;
                x[6] = p1 ? col[(size_t)checked_node(u1.z, gp.n) * W] : -1;
                x[7] = p1 ? col[(size_t)checked_node(u1.w, gp.n) * W] : -1;
#pragma unroll
                for (int t = 0; t < 8; ++t) c += x[t] == own;
            }
            const bool ok = has && 2 * c > r.z;
            if (ok) {
                add_degree(gp, hist, own, i, r.z);
                if (r.z > kLaneMax) atomicAdd(oks + (e >> 7), 1);
            }
            settled32 += __popc(__ballot_sync(kFull, ok && r.z <= kLaneMax));
            const unsigned rest = __ballot_sync(kFull, has && !ok);
            __syncwarp();
            if (has && !ok) list[open + __popc(rest & lt)] = (unsigned short)e;
            open += __popc(rest);
        }
        __syncwarp();

        // The exact votes of the open pairs (degrees still descending).
        int pairs32 = settled32;
        for (int base = 0; base < open; base += 32) {
            const bool has = base + lane < open;
            const int e = has ? list[base + lane] : 0;
            const int i = e & 127;
            int4 r = recs[e >> 7];
            const unsigned big = __ballot_sync(kFull, has && r.z > kLaneMax);
            if (big) {
                const unsigned far = __ballot_sync(kFull, has && r.z > 2 * kLaneMax);
                if (far) defer_pairs(gp, 1, far, idx0 + (e >> 7), i, lane, dlist, dcount);
                if (big & ~far) defer_pairs(gp, 0, big & ~far, idx0 + (e >> 7), i, lane, dlist, dcount);
            }
            const bool mine = has && r.z <= kLaneMax;
            const int deg = mine ? r.z : 0;
            const int top = __reduce_max_sync(kFull, deg);
            if (top == 0) continue;
            int res, best;
            if (top <= 8) res = lane_vote<8>(gp, adj, child, r.x, i, r.y, deg, g, best);
            else if (top <= 12) res = lane_vote<12>(gp, adj, child, r.x, i, r.y, deg, g, best);
            else if (top <= 16) res = lane_vote<16>(gp, adj, child, r.x, i, r.y, deg, g, best);
            else if (top <= 20) res = lane_vote<20>(gp, adj, child, r.x, i, r.y, deg, g, best);
            else if (top <= 24) res = lane_vote<24>(gp, adj, child, r.x, i, r.y, deg, g, best);
            else if (top <= 28) res = lane_vote<28>(gp, adj, child, r.x, i, r.y, deg, g, best);
            else res = lane_vote<32>(gp, adj, child, r.x, i, r.y, deg, g, best);
            bool same = false;
            if (mine) {
                const size_t cell = (size_t)r.x * W + i;
                same = res == child[cell];
                if (!same) q[cell] = res;
                add_degree(gp, hist, res, i, deg);
            }
            pairs32 += __popc(__ballot_sync(kFull, mine));
            settled32 += __popc(__ballot_sync(kFull, mine && same && r.w == 0 && 2 * best > deg));
        }
        // The history: per node above kLaneMax, a sample of the batches below
        // (the deferred pairs add theirs in mutation_vote_kernel).
        if (lane < nb && rec.z > kLaneMax) hint[idx0 + lane] = ((uint32_t)nsel << 16) | (uint32_t)oks[lane];
        if (((item - wide) & 7) == 0 && lane == 0 && pairs32 > 0) {
            atomicAdd(dcount + kDcountPairs, pairs32);
            atomicAdd(dcount + kDcountOk, settled32);
        }
        __syncwarp();
    }
}

// The exact neighbour-majority of one deferred pair (node of degree
// kLaneMax + 1 .. N) per thread: the pair's labels are gathered into
// registers, sorted by the merge-exchange network, and the pick(u, t)-th of
// the t longest runs is the result, u the MTIE word. The thread writes the
// label into Q, adds deg(v) to the degree histogram and, when the own label is
// on more than half of the neighbours, counts the pair in the node's hint.
template <int N>
__device__ __forceinline__ void mutation_vote_body(const GenParams &gp, int cls, const int4 *__restrict__ nodes,
                                                   const int4 *__restrict__ adj, const int32_t *__restrict__ child,
                                                   int32_t *__restrict__ q, const uint32_t *__restrict__ gen_ptr,
                                                   uint32_t *__restrict__ hist, uint32_t *__restrict__ hint,
                                                   const int2 *__restrict__ dlist, const int *__restrict__ dcount,
                                                   int vblock, int vgrid)
{
    constexpr int NW = (N + 63) / 64;
    const uint32_t g = *gen_ptr;
    const int W = gp.W;
    const int total = min(dcount[cls], defer_capacity(gp, cls));
    const int2 *list = dlist + defer_offset(gp, cls);
    for (int t = vblock * blockDim.x + threadIdx.x; t < total; t += vgrid * blockDim.x) {
        const int2 e = list[t];
        const int i = e.y;
        if (!MOCD_CHECK(e.x >= 0 && e.x < gp.n && i >= 0 && i < gp.np, kCheckNode, t)) continue;
        const int4 rec = __ldg(nodes + e.x);
        const int v = rec.x, deg = min(rec.z, N);
        const int32_t *col = child + i;
        int x[N];
#pragma unroll
        for (int j = 0; j < N; j += 4) {
            const bool in = j < deg;
            const int4 u = in ? __ldg(adj + rec.y + j / 4) : make_int4(0, 0, 0, 0);
            x[j + 0] = in ? col[(size_t)checked_node(u.x, gp.n) * W] : INT_MAX;
            x[j + 1] = in ? col[(size_t)checked_node(u.y, gp.n) * W] : INT_MAX;
            x[j + 2] = in ? col[(size_t)checked_node(u.z, gp.n) * W] : INT_MAX;
            x[j + 3] = in ? col[(size_t)checked_node(u.w, gp.n) * W] : INT_MAX;
        }
        sort_network<N>(x);
        // Runs of equal labels as in longest_runs, over NW 64-bit words: bit j
        // of eq is set when entries j and j + 1 (< deg) are equal; each step
        // m &= m >> 1 (across words) shortens every run of set bits by one,
        // and the last non-zero m marks the first entry of each longest run.
        unsigned long long eq[NW], starts[NW], m[NW];
#pragma unroll
        for (int w = 0; w < NW; ++w) eq[w] = 0ull;
#pragma unroll
        for (int j = 0; j + 1 < N; ++j) eq[j >> 6] |= (x[j] == x[j + 1] ? 1ull : 0ull) << (j & 63);
        bool any = false;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const int pairs = deg - 1 - 64 * w;  // valid bits of word w
            const int ents = deg - 64 * w;
            eq[w] &= pairs >= 64 ? ~0ull : pairs <= 0 ? 0ull : (1ull << pairs) - 1ull;
            starts[w] = ents >= 64 ? ~0ull : ents <= 0 ? 0ull : (1ull << ents) - 1ull;
            m[w] = eq[w];
            any |= eq[w] != 0ull;
        }
        int best = 1;
        while (any) {
            any = false;
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                starts[w] = m[w];
                const unsigned long long carry = w + 1 < NW ? m[w + 1 < NW ? w + 1 : w] << 63 : 0ull;
                m[w] &= (m[w] >> 1) | carry;
                any |= m[w] != 0ull;
            }
            ++best;
        }
        int tcount = 0;
#pragma unroll
        for (int w = 0; w < NW; ++w) tcount += __popcll(starts[w]);
        unsigned kk = 0;
        if (tcount > 1) kk = pick_index(tie_word(gp, v, i, g), (uint32_t)tcount);
        // Position of the kk-th set bit of the starts mask.
        int pos = 0;
        unsigned k = kk;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            const unsigned c = (unsigned)__popcll(starts[w]);
            if (k >= c) {
                k -= c;
                continue;
            }
            unsigned long long mm = starts[w];
            int p = 64 * w;
#pragma unroll
            for (int width = 32; width >= 1; width >>= 1) {
                const unsigned long long low = mm & ((1ull << width) - 1ull);
                const unsigned lc = (unsigned)__popcll(low);
                if (k >= lc) {
                    k -= lc;
                    mm >>= width;
                    p += width;
                } else {
                    mm = low;
                }
            }
            pos = p;
            break;
        }
        const int res = select_at<N>(x, pos);
        const size_t cell = (size_t)v * W + i;
        q[cell] = res;
        add_degree(gp, hist, res, i, deg);
        if (2 * best > deg && res == child[cell]) atomicAdd(hint + e.x, 1u);
    }
}

template <int N>
__global__ void __launch_bounds__(kMutBlock)
mutation_vote_kernel(const __grid_constant__ GenParams gp, int cls, const int4 *__restrict__ nodes,
                     const int4 *__restrict__ adj, const int32_t *__restrict__ child, int32_t *__restrict__ q,
                     const uint32_t *__restrict__ gen_ptr, uint32_t *__restrict__ hist, uint32_t *__restrict__ hint,
                     const int2 *__restrict__ dlist, const int *__restrict__ dcount)
{
    mutation_vote_body<N>(gp, cls, nodes, adj, child, q, gen_ptr, hist, hint, dlist, dcount, blockIdx.x, gridDim.x);
}

// The deferred votes of one degree class of every member of a batch.
// (Register cap: the single-member kernel's occupancy, 5 blocks of 128
// threads for 64 entries; 2 for 128, whose registers do not fit 3 here.)
template <int N>
__global__ void __launch_bounds__(kMutBlock, N <= 64 ? 5 : 2)
mutation_vote_multi_kernel(const BatchMember *__restrict__ members, const int *__restrict__ starts, int count,
                           int cls)
{
    const int k = member_of_block(starts, count);
    const BatchMember &mb = members[k];
    const PopState &ps = mb.ps;
    const GenParams gp = mb.gp;
    const int b0 = __ldg(starts + k);
    mutation_vote_body<N>(gp, cls, mb.nodes, mb.adj, ps.c, ps.q, ps.gen, ps.hist, ps.hint, ps.dlist, ps.dcount,
                          (int)blockIdx.x - b0, __ldg(starts + k + 1) - b0);
}

// Sum (or maximum) over the hub block; every thread gets it. s_red holds one
// word per warp; the trailing barrier frees it for the next call.
template <bool MAX>
__device__ __forceinline__ unsigned hub_reduce(unsigned x, unsigned *s_red)
{
    x = MAX ? __reduce_max_sync(kFull, x) : __reduce_add_sync(kFull, x);
    if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = x;
    __syncthreads();
    unsigned r = 0;
#pragma unroll
    for (int w = 0; w < kHubBlock / 32; ++w) r = MAX ? max(r, s_red[w]) : r + s_red[w];
    __syncthreads();
    return r;
}

// The listed pairs of hubs above kSharedTableMax, a block each: the own
// label's count if the node's history says it pays, else (or if it leaves the
// pair open) the exact vote with a count table of the smallest power of two
// >= 2 deg slots, in shared memory if it fits there (gp.hub_smem_hs), else in
// the block's slice of global scratch (2 gp.hub_hs ints). Writes the label
// into Q, adds deg(v) to the histogram and counts the pair in the hub's hint
// when its own label is on more than half of the neighbours. A block per pair
// keeps a hub of thousands of neighbours off the critical path: one warp per
// pair is a chain of deg / 32 dependent table inserts.
__global__ void __launch_bounds__(kHubBlock)
mutation_hub_kernel(const __grid_constant__ GenParams gp, const int4 *__restrict__ nodes,
                    const int4 *__restrict__ adj, const int32_t *__restrict__ child, int32_t *__restrict__ q,
                    const uint32_t *__restrict__ gen_ptr, uint32_t *__restrict__ hist, uint32_t *__restrict__ hint,
                    const int2 *__restrict__ dlist, const int *__restrict__ dcount, int *__restrict__ hub_table)
{
    extern __shared__ int s_table[];  // [2 gp.hub_smem_hs]
    __shared__ unsigned s_red[kHubBlock / 32];
    __shared__ int s_tied, s_res;
    const uint32_t g = *gen_ptr;
    const int lane = threadIdx.x & 31;
    const int total = min(dcount[2], defer_capacity(gp, 2));
    const int2 *list = dlist + defer_offset(gp, 2);
    for (int t = blockIdx.x; t < total; t += gridDim.x) {
        const int2 e = list[t];
        const int idx = e.x & ~kHubFast, i = e.y;
        if (!MOCD_CHECK(idx >= 0 && idx < gp.n && i >= 0 && i < gp.np, kCheckNode, t)) continue;  // (block-uniform)
        const int4 rec = __ldg(nodes + idx);
        const int v = rec.x, deg = min(rec.z, gp.hub_hs / 2);
        const int *nbr = reinterpret_cast<const int *>(adj + rec.y);
        const int32_t *col = child + i;
        const size_t cell = (size_t)v * gp.W + i;
        const int own = child[cell];
        if (e.x & kHubFast) {
            unsigned c = 0;
#pragma unroll 4
            for (int j = threadIdx.x; j < deg; j += kHubBlock)
                c += col[(size_t)checked_node(__ldg(nbr + j), gp.n) * gp.W] == own ? 1u : 0u;
            if (2 * (int)hub_reduce<false>(c, s_red) > deg) {  // (Q holds the own label already)
                if (threadIdx.x == 0) {
                    add_degree(gp, hist, own, i, deg);
                    atomicAdd(hint + idx, 1u);
                }
                continue;
            }
        }
        int hbits = 11;
        while ((1 << hbits) < 2 * deg) ++hbits;
        const int HS = 1 << hbits;
        int *hkey = HS <= gp.hub_smem_hs ? s_table : hub_table + (size_t)blockIdx.x * 2 * gp.hub_hs;
        int *hcnt = hkey + HS;
        for (int s = threadIdx.x; s < HS; s += kHubBlock) {
            hkey[s] = -1;
            hcnt[s] = 0;
        }
        if (threadIdx.x == 0) s_tied = 0;
        __syncthreads();
        for (int j0 = 0; j0 < deg; j0 += kHubBlock) {
            const int j = j0 + threadIdx.x;
            const bool in = j < deg;
            const int x = in ? col[(size_t)checked_node(__ldg(nbr + j), gp.n) * gp.W] : (int)(0x80000000u | lane);
            // One insert per distinct label of the warp's neighbours.
            const unsigned peers = __match_any_sync(kFull, x);
            if (in && (peers & ((1u << lane) - 1u)) == 0) {
                uint32_t h = hash_slot(x, hbits);
                for (int probe = 0; probe < HS; ++probe) {  // (at most HS / 2 distinct labels: a slot is found)
                    const int prev = atomicCAS(hkey + h, -1, x);
                    if (prev == -1 || prev == x) {
                        atomicAdd(hcnt + h, __popc(peers));
                        break;
                    }
                    h = (h + 1) & (uint32_t)(HS - 1);
                }
            }
        }
        __syncthreads();
        unsigned my = 0;
        for (int s = threadIdx.x; s < HS; s += kHubBlock) my = max(my, (unsigned)hcnt[s]);
        const unsigned mx = hub_reduce<true>(my, s_red);
        // The tied labels, compacted to hcnt[0, tied) once every thread has
        // read its slots' counts.
        for (int s = threadIdx.x; s < HS; s += kHubBlock)
            if ((unsigned)hcnt[s] != mx) hkey[s] = -1;
        __syncthreads();
        for (int s = threadIdx.x; s < HS; s += kHubBlock) {  // (HS is a multiple of the block: warps stay whole)
            const int key = hkey[s];
            const unsigned who = __ballot_sync(kFull, key >= 0);
            int at = 0;
            if (lane == 0 && who) at = atomicAdd(&s_tied, __popc(who));
            at = __shfl_sync(kFull, at, 0);
            if (key >= 0) hcnt[at + __popc(who & ((1u << lane) - 1u))] = key;
        }
        __syncthreads();
        const int tied = s_tied;
        if (tied == 1) {
            if (threadIdx.x == 0) s_res = hcnt[0];
        } else {
            // Bit by bit from the top, as in warp_mode_table.
            unsigned prefix = 0, rank = pick_index(tie_word(gp, v, i, g), (uint32_t)tied);
            for (int b = gp.label_bits - 1; b >= 0; --b) {
                const unsigned above = ~((2u << b) - 1u);  // the bits above b
                unsigned c = 0;
                for (int s = threadIdx.x; s < tied; s += kHubBlock) {
                    const unsigned key = (unsigned)hcnt[s];
                    c += ((key & above) == prefix && ((key >> b) & 1u) == 0u) ? 1u : 0u;
                }
                const unsigned cnt = hub_reduce<false>(c, s_red);
                if (rank >= cnt) {
                    rank -= cnt;
                    prefix |= 1u << b;
                }
            }
            if (threadIdx.x == 0) s_res = (int)prefix;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            const int lab = s_res;
            q[cell] = lab;
            add_degree(gp, hist, lab, i, deg);
            if (lab == own && 2 * (int)mx > deg) atomicAdd(hint + idx, 1u);
        }
        __syncthreads();
    }
}

template <int EMAX>
size_t crossover_smem()
{
    return sizeof(int) * (2 * kMaxPop + kMaxPop * EMAX + (kBlock / 32) * 2 * kMaxPop);
}

}  // namespace

cudaError_t launch_init_population(const GenParams &gp, int init_mode, const int32_t *row_ptr,
                                   const int32_t *col_idx, int32_t *dst, cudaStream_t s)
{
    const long long total = (long long)gp.n * (gp.W >> 2);
    long long blocks = (total + kBlock - 1) / kBlock;
    if (blocks > 65535LL * 16) blocks = 65535LL * 16;
    if (init_mode == 1)
        init_sweep_kernel<<<(int)blocks, kBlock, 0, s>>>(gp.n, gp.W, gp.np, gp.key0, gp.key1, row_ptr,
                                                         col_idx, dst);
    else
        init_population_kernel<<<(int)blocks, kBlock, 0, s>>>(gp.n, gp.W, gp.np, gp.key0, gp.key1, dst);
    return cudaGetLastError();
}

int grid_for_crossover(int sms, int es)
{
    int per_sm = 0;
    if (es <= 4)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, crossover_kernel<4>, kBlock, crossover_smem<4>());
    else if (es <= 8)
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, crossover_kernel<8>, kBlock, crossover_smem<8>());
    else
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, crossover_kernel<16>, kBlock, crossover_smem<16>());
    if (per_sm < 1) per_sm = 1;
    return sms * per_sm;
}

cudaError_t launch_crossover(const GenParams &gp, const PopState &ps, int grid, cudaStream_t s)
{
    if (gp.es <= 4)
        crossover_kernel<4><<<grid, kBlock, crossover_smem<4>(), s>>>(
            gp, ps.buf[0], ps.buf[1], ps.buf[0], ps.buf[1], ps.q, ps.c, ps.keep, ps.par_r, ps.copy_r, ps.gen,
            ps.dcount);
    else if (gp.es <= 8)
        crossover_kernel<8><<<grid, kBlock, crossover_smem<8>(), s>>>(
            gp, ps.buf[0], ps.buf[1], ps.buf[0], ps.buf[1], ps.q, ps.c, ps.keep, ps.par_r, ps.copy_r, ps.gen,
            ps.dcount);
    else
        crossover_kernel<16><<<grid, kBlock, crossover_smem<16>(), s>>>(
            gp, ps.buf[0], ps.buf[1], ps.buf[0], ps.buf[1], ps.q, ps.c, ps.keep, ps.par_r, ps.copy_r, ps.gen,
            ps.dcount);
    return cudaGetLastError();
}

cudaError_t launch_crossover_multi(const BatchMember *members, const int *starts, int count, int blocks, int es_max,
                                   cudaStream_t s)
{
    if (blocks <= 0) return cudaSuccess;
    if (es_max <= 4)
        crossover_multi_kernel<4><<<blocks, kBlock, crossover_smem<4>(), s>>>(members, starts, count);
    else if (es_max <= 8)
        crossover_multi_kernel<8><<<blocks, kBlock, crossover_smem<8>(), s>>>(members, starts, count);
    else
        crossover_multi_kernel<16><<<blocks, kBlock, crossover_smem<16>(), s>>>(members, starts, count);
    return cudaGetLastError();
}

cudaError_t launch_vote_multi(const BatchMember *members, const int *starts, int count, int blocks, int cls,
                              cudaStream_t s)
{
    if (blocks <= 0) return cudaSuccess;
    if (cls == 0)
        mutation_vote_multi_kernel<2 * kLaneMax><<<blocks, kMutBlock, 0, s>>>(members, starts, count, 0);
    else
        mutation_vote_multi_kernel<kDeferMax><<<blocks, kMutBlock, 0, s>>>(members, starts, count, 1);
    return cudaGetLastError();
}

int mutation_smem(int hash_size)
{
    return (kMutBlock / 32) * 2 * hash_size * (int)sizeof(int);
}

int mutation_warps_per_block()
{
    return kMutBlock / 32;
}

int grid_for_mutation(int sms, int hash_size)
{
    const int smem = mutation_smem(hash_size);
    int per_sm = 0;
    if (hash_size > 0) {
        cudaFuncSetAttribute(mutation_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mutation_kernel<true>, kMutBlock, smem);
    } else {
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mutation_kernel<false>, kMutBlock, 0);
    }
    return sms * (per_sm < 1 ? 1 : per_sm);
}

// Blocks of the hub kernel: as many as its shared table lets be resident.
int grid_for_hubs(int sms, int smem_hs)
{
    const int smem = 2 * smem_hs * (int)sizeof(int);
    cudaFuncSetAttribute(mutation_hub_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mutation_hub_kernel, kHubBlock, smem);
    return sms * (per_sm < 1 ? 1 : per_sm);
}

void grid_for_votes(int sms, int vote_n0, int *grid64, int *grid128)
{
    int a = 0, b = 0;
    switch (vote_n0) {
    case 40: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, mutation_vote_kernel<40>, kMutBlock, 0); break;
    case 48: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, mutation_vote_kernel<48>, kMutBlock, 0); break;
    case 56: cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, mutation_vote_kernel<56>, kMutBlock, 0); break;
    default:
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, mutation_vote_kernel<2 * kLaneMax>, kMutBlock, 0);
    }
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, mutation_vote_kernel<kDeferMax>, kMutBlock, 0);
    *grid64 = sms * (a < 1 ? 1 : a);
    *grid128 = sms * (b < 1 ? 1 : b);
}

namespace {

template <int N>
void launch_vote(const GenParams &gp, const PopState &ps, int cls, const int4 *nodes, const int4 *adj, int grid,
                 cudaStream_t s)
{
    mutation_vote_kernel<N><<<grid, kMutBlock, 0, s>>>(gp, cls, nodes, adj, ps.c, ps.q, ps.gen, ps.hist, ps.hint,
                                                       ps.dlist, ps.dcount);
}

}  // namespace

cudaError_t launch_mutation(const GenParams &gp, const PopState &ps, const int4 *nodes, const int4 *adj, int batch,
                            int grid, int grid64, int grid128, cudaStream_t s, bool with_votes)
{
    if (gp.hash_size > 0)
        mutation_kernel<true><<<grid, kMutBlock, mutation_smem(gp.hash_size), s>>>(
            gp, nodes, adj, ps.c, ps.q, ps.gen, ps.hist, ps.acc, ps.hint, ps.dlist, ps.dcount, batch);
    else
        mutation_kernel<false><<<grid, kMutBlock, 0, s>>>(gp, nodes, adj, ps.c, ps.q, ps.gen, ps.hist, ps.acc, ps.hint,
                                                          ps.dlist, ps.dcount, batch);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (with_votes && gp.defer_cap[0] > 0) {
        // The class's network holds the graph's largest degree in it.
        switch (gp.vote_n0) {
        case 40: launch_vote<40>(gp, ps, 0, nodes, adj, grid64, s); break;
        case 48: launch_vote<48>(gp, ps, 0, nodes, adj, grid64, s); break;
        case 56: launch_vote<56>(gp, ps, 0, nodes, adj, grid64, s); break;
        default: launch_vote<2 * kLaneMax>(gp, ps, 0, nodes, adj, grid64, s);
        }
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (with_votes && gp.defer_cap[1] > 0) {
        launch_vote<kDeferMax>(gp, ps, 1, nodes, adj, grid128, s);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    if (gp.defer_cap[2] > 0) {
        mutation_hub_kernel<<<gp.hub_blocks, kHubBlock, 2 * gp.hub_smem_hs * sizeof(int), s>>>(
            gp, nodes, adj, ps.c, ps.q, ps.gen, ps.hist, ps.hint, ps.dlist, ps.dcount, ps.hub_table);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace mocd

namespace mocd {
cudaError_t check_record_variation(unsigned long long *out, bool reset)
{
    return check_record(out, reset);
}
}  // namespace mocd
