// k_variation.cu -- InitializePopulation and the offspring map of Alg. 1:
// topology-aware crossover (Sec. 4.3.1, Alg. 2) and topology-aware mutation
// (Sec. 4.3.2), for all N_p children of a generation at once.
//
// Both kernels work on node-major rows, in quads: the four children 4q..4q+3
// of a node are one lane's, and share one Philox call per stage because the
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

// ---------------------------------------------------------------------------
// Crossover. Row v of R = (P half | Q) is staged in shared memory; the next P
// (environmental selection's keep list) is compacted into the other P half,
// and child i of the generation gets
//   copy_r[i] >= 0 : R_v[copy_r[i]]                    (x > C_P: random parent)
//   otherwise      : majority of R_v[par_r[i][j]], j < E_S, the tie among the t
//                    most frequent labels broken by the XTIE word: the
//                    pick(u, t)-th smallest of them (Eq. arg_max).
// A lane owns a quad of children; a warp takes as many nodes at a time as its
// lanes hold quads. The parents of a copied child are E_S times the copied
// member, those of a child past N_p (padding of the last quad) a cell that
// holds 0, so neither needs a case of its own.
// Up to four parents (the default), a lane keeps the row positions of its four
// children's parents and kept members in registers for the whole kernel: per
// node it loads 20 labels from shared memory and sorts four of them per child
// (5 comparators). Bound by the half-rate integer pipe and by the bank
// conflicts of the label reads. More parents: the positions stay in shared
// memory and a network of 8 or 16 entries sorts the labels. Measured a launch,
// N_p 100, E_S 4: n = 40,000 25.0 -> 21.4 us, n = 10^6 478 -> 388 us; E_S 3,
// N_p 50, n = 30,011 42 -> 11.8 us; E_S 6, N_p 128, n = 4,001 34 -> 10.1 us (against
// positions in shared memory, a node a warp, and pairwise counts of the votes
// for every E_S but 4).
// ---------------------------------------------------------------------------

constexpr int kRowPad = 4;  // cells after a staged row: two above every label, one 0

// Row position of member r of R.
__device__ __forceinline__ int row_position(const GenParams &gp, int r, int t)
{
    if (!MOCD_CHECK(r >= 0 && r < 2 * gp.np, kCheckRIndex, t)) r = 0;
    return r < gp.np ? r : gp.W + (r - gp.np);
}

// The pick(u, t)-th of the t most frequent of the E sorted values x (entries
// at E and above sort last): the longest runs, from a bit mask of equal
// neighbours (see lane_vote). word() is called only when t > 1.
template <int N, class F>
__device__ __forceinline__ int sorted_mode(const int (&x)[N], int E, F word)
{
    unsigned m = 0;
#pragma unroll
    for (int j = 0; j + 1 < N; ++j) m |= (x[j] == x[j + 1] ? 1u : 0u) << j;
    m &= (1u << (E - 1)) - 1u;
    unsigned starts = (1u << E) - 1u;
    while (m) {
        starts = m;
        m &= m >> 1;
    }
    const int t = __popc(starts);
    const unsigned k = t > 1 ? pick_index(word(), (uint32_t)t) : 0u;
    return select_at<N>(x, kth_bit(starts, k));
}

template <int EMAX>
__device__ __forceinline__ void crossover_body(const GenParams gp, const int32_t *buf0, const int32_t *buf1,
                                               int32_t *out0, int32_t *out1, const int32_t *__restrict__ q,
                                               int32_t *__restrict__ child, const int32_t *__restrict__ keep,
                                               const int32_t *__restrict__ par_r, const int32_t *__restrict__ copy_r,
                                               const uint32_t *__restrict__ gen_ptr, int vblock, int vgrid)
{
    extern __shared__ int smem[];
    const int W = gp.W, np = gp.np, E = gp.es;
    const int nq = W >> 2;
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    const int per_warp = 32 / nq;  // nodes a warp takes at a time (nq <= 32)
    const int sub = lane / nq, quad = lane - sub * nq;
    const bool active = sub < per_warp;
    const int row_words = 2 * W + kRowPad;
    // EMAX > 4: the parents' row positions, [EMAX][4][32], then the rows.
    constexpr int kTable = EMAX > 4 ? EMAX * kMaxPop : 0;
    int *row = smem + kTable + (wib * per_warp + (active ? sub : 0)) * row_words;
    const uint32_t g = *gen_ptr;

    // Row positions of child 4 quad + k's kept member and parents.
    const int zero = 2 * W + 2;
    int kept[4], par[4][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const int i = 4 * quad + k;
        const bool real = active && i < np;
        kept[k] = real ? row_position(gp, keep[i], i) : zero;
        if (EMAX == 4) {
            const int c = real ? copy_r[i] : -1;
            if (!real || c >= 0) {
                const int at = real ? row_position(gp, c, i) : zero;
#pragma unroll
                for (int j = 0; j < 4; ++j) par[k][j] = at;
            } else {
                const int4 p = *reinterpret_cast<const int4 *>(par_r + i * kMaxParents);
                par[k][0] = row_position(gp, p.x, i);
                // Fewer than four: values above every label, which sort last
                // and differ; one parent: four times the same.
                par[k][1] = E > 1 ? row_position(gp, p.y, i) : par[k][0];
                par[k][2] = E > 2 ? row_position(gp, p.z, i) : E == 2 ? 2 * W : par[k][0];
                par[k][3] = E > 3 ? row_position(gp, p.w, i) : E > 1 ? 2 * W + 1 : par[k][0];
            }
        }
    }
    if (EMAX > 4) {
        for (int t = threadIdx.x; t < kMaxPop; t += blockDim.x) {
            const int c = t < np ? copy_r[t] : -1;
            for (int j = 0; j < EMAX; ++j) {
                int at = zero;
                if (t < np) at = j >= E ? 2 * W + 1 : row_position(gp, c >= 0 ? c : par_r[t * kMaxParents + j], t);
                else if (j >= E) at = 2 * W + 1;
                smem[(j * 4 + (t & 3)) * 32 + (t >> 2)] = at;
            }
        }
        __syncthreads();
    }
    if (active && quad == 0) {
        row[2 * W] = INT_MAX - 1;
        row[2 * W + 1] = INT_MAX;
        row[2 * W + 2] = 0;
    }

    // Generation g reads the P half buf[g & 1] and writes the compacted P
    // into the other half (the two never alias within one launch).
    const int4 *P4 = reinterpret_cast<const int4 *>((g & 1u) ? buf1 : buf0);
    int4 *D4 = reinterpret_cast<int4 *>((g & 1u) ? out0 : out1);
    const int4 *__restrict__ Q4 = reinterpret_cast<const int4 *>(q);
    int4 *__restrict__ C4 = reinterpret_cast<int4 *>(child);

    const int warp = (vblock * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (vgrid * blockDim.x) >> 5;

    // Software pipeline: the next node's rows are requested before the
    // current node is processed.
    int4 cur_p = make_int4(0, 0, 0, 0), cur_q = make_int4(0, 0, 0, 0);
    if (active && warp * per_warp + sub < gp.n) {
        cur_p = P4[(size_t)(warp * per_warp + sub) * nq + quad];
        cur_q = Q4[(size_t)(warp * per_warp + sub) * nq + quad];
    }
    for (long long v0 = (long long)warp * per_warp; v0 < gp.n; v0 += (long long)nwarps * per_warp) {
        const long long v = v0 + sub, vn = v + (long long)nwarps * per_warp;
        const bool mine = active && v < gp.n;
        int4 nxt_p = make_int4(0, 0, 0, 0), nxt_q = make_int4(0, 0, 0, 0);
        if (active && vn < gp.n) {
            nxt_p = P4[(size_t)vn * nq + quad];
            nxt_q = Q4[(size_t)vn * nq + quad];
        }
        if (mine) {
            reinterpret_cast<int4 *>(row)[quad] = cur_p;
            reinterpret_cast<int4 *>(row + W)[quad] = cur_q;
        }
        cur_p = nxt_p;
        cur_q = nxt_q;
        __syncwarp();
        if (mine) {
            int o[4], r[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) o[k] = row[kept[k]];
            if (EMAX == 4) {
                // Sort each child's votes; the run pattern of the sorted values
                // gives the maximal labels in ascending order: all distinct
                // (t = E), two pairs (t = 2) or a unique maximum. All four
                // children are classified first so that the lane's tie word
                // (one Philox call for its four children) is computed at most
                // once.
                int srt[4][4];
                bool none[4], two[4];
                bool tie = false;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) srt[k][j] = row[par[k][j]];
                }
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    sort_network<4>(srt[k]);
                    const bool e01 = srt[k][0] == srt[k][1], e12 = srt[k][1] == srt[k][2], e23 = srt[k][2] == srt[k][3];
                    none[k] = !e01 && !e12 && !e23;
                    two[k] = e01 && e23 && !e12;
                    r[k] = e01 ? srt[k][0] : e12 ? srt[k][1] : srt[k][2];
                    tie |= none[k] || two[k];
                }
                if (tie) {
                    const uint4 u =
                        philox4x32_10(make_uint4((uint32_t)v, (uint32_t)quad, g, kStageCrossTie), gp.key0, gp.key1);
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const uint32_t w = word_of(u, k);
                        const uint32_t kk = pick_index(w, (uint32_t)E);
                        const int low = (kk & 1u) ? srt[k][1] : srt[k][0];
                        const int high = (kk & 1u) ? srt[k][3] : srt[k][2];
                        if (none[k]) r[k] = (kk & 2u) ? high : low;
                        else if (two[k] && (w >> 31)) r[k] = srt[k][2];
                    }
                }
            } else {
                bool have_u = false;
                uint4 u = make_uint4(0, 0, 0, 0);
                for (int k = 0; k < 4; ++k) {
                    int x[EMAX];
#pragma unroll
                    for (int j = 0; j < EMAX; ++j) x[j] = row[smem[(j * 4 + k) * 32 + quad]];
                    sort_network<EMAX>(x);
                    const int res = sorted_mode<EMAX>(x, E, [&]() {
                        if (!have_u) {
                            u = philox4x32_10(make_uint4((uint32_t)v, (uint32_t)quad, g, kStageCrossTie), gp.key0,
                                              gp.key1);
                            have_u = true;
                        }
                        return word_of(u, k);
                    });
                    r[0] = k == 0 ? res : r[0];
                    r[1] = k == 1 ? res : r[1];
                    r[2] = k == 2 ? res : r[2];
                    r[3] = k == 3 ? res : r[3];
                }
            }
            D4[(size_t)v * nq + quad] = make_int4(o[0], o[1], o[2], o[3]);
            C4[(size_t)v * nq + quad] = make_int4(r[0], r[1], r[2], r[3]);
        }
        __syncwarp();
    }
}

template <int EMAX>
__global__ void __launch_bounds__(kBlock, 2)
crossover_kernel(const __grid_constant__ GenParams gp, const int32_t *buf0, const int32_t *buf1, int32_t *out0,
                 int32_t *out1, const int32_t *__restrict__ q, int32_t *__restrict__ child,
                 const int32_t *__restrict__ keep, const int32_t *__restrict__ par_r,
                 const int32_t *__restrict__ copy_r, const uint32_t *__restrict__ gen_ptr)
{
    crossover_body<EMAX>(gp, buf0, buf1, out0, out1, q, child, keep, par_r, copy_r, gen_ptr, blockIdx.x, gridDim.x);
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
__global__ void __launch_bounds__(kBlock, 2)
crossover_multi_kernel(const BatchMember *__restrict__ members, const int *__restrict__ starts, int count)
{
    const int k = member_of_block(starts, count);
    const BatchMember &mb = members[k];
    const PopState &ps = mb.ps;
    const int b0 = __ldg(starts + k);
    crossover_body<EMAX>(mb.gp, ps.buf[0], ps.buf[1], ps.buf[0], ps.buf[1], ps.q, ps.c, ps.keep, ps.par_r,
                         ps.copy_r, ps.gen, (int)blockIdx.x - b0, __ldg(starts + k + 1) - b0);
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
// node has selected (about 20 of 100 at M_P 0.2). By degree:
//   up to 128    mutation_kernel, a pair per lane: the labels are gathered into
//                registers, sorted by a merge-exchange network and the tied
//                labels read off the runs. One launch for degrees up to 32
//                (networks of 8, 12, .., 28 or 32 entries, the smallest that
//                holds the lanes' degrees), one each for 33..64 (40, 48, 56 or
//                64 entries, the smallest that holds the graph's largest
//                degree there) and 65..128, so that no launch pays for the
//                registers of a larger network than its own
//   129..512     a warp per pair: count table in shared memory (the node's
//                pairs are split over gp.wide_parts warps), in the first launch
//   above 512    mutation_hub_kernel, a block per pair
// The launches touch different rows of Q and only add to the histogram, so
// they run side by side.
//
// A count table costs several passes over the neighbours' labels, and in a
// settled population the result is often the label the node already has:
// counting the neighbours that hold it proves that when it is on more than
// half of them (it is then the unique mode). Above degree 128 that count goes
// first when the node's last generation says it pays (own_label_pays). The
// vote in registers needs one pass, and a front keeps so many fragmented
// members that the count settles at most 0.45 of the pairs (n = 40,000 and
// 10^6, mu 0.3): trying it first there was slower at every threshold (n =
// 10^6: 2.59 ms a generation's mutation with it from half settled on, 2.50
// without).
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

constexpr int kLaneMax = 32;     // largest degree of the per-lane vote
constexpr int kMutBlock = 128;   // mutation threads per block
constexpr int kHubBlock = 256;   // threads per block of the hub kernel
static_assert(kMutBatchMax * kMaxPop <= 65536, "a pair is listed in 16 bits");

// Exact neighbour-majority of one pair by its own lane (deg <= N; 0 for a
// lane without a pair). The labels are gathered into registers (the padding
// and the entries past it sort last) and sorted; equal labels then form runs,
// the longest runs are the tied labels in ascending order, and the
// pick(u, t)-th of them is the result. Bit j of eq is set when entries j and
// j + 1 (< deg) are equal, so a run of L labels is L - 1 consecutive set bits;
// each step m &= m >> 1 (across words) shortens every run of set bits by one,
// and the last non-zero m has one bit per longest run, at its first entry (all
// entries when no two are equal). All lanes of the warp call together.
template <int N>
__device__ __forceinline__ int lane_vote(const GenParams &gp, const int4 *__restrict__ adj,
                                         const int32_t *__restrict__ child, int v, int i, int beg, int deg, uint32_t g)
{
    constexpr int NW = (N + 31) / 32;
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
    unsigned m[NW], starts[NW];
#pragma unroll
    for (int w = 0; w < NW; ++w) m[w] = 0u;
#pragma unroll
    for (int j = 0; j + 1 < N; ++j) m[j >> 5] |= (x[j] == x[j + 1] ? 1u : 0u) << (j & 31);
    bool any = false;
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        const int pairs = deg - 1 - 32 * w, ents = deg - 32 * w;  // valid bits of the word
        m[w] &= pairs >= 32 ? ~0u : pairs <= 0 ? 0u : (1u << pairs) - 1u;
        starts[w] = ents >= 32 ? ~0u : ents <= 0 ? 0u : (1u << ents) - 1u;
        any |= m[w] != 0u;
    }
    while (any) {
        any = false;
#pragma unroll
        for (int w = 0; w < NW; ++w) {
            starts[w] = m[w];
            m[w] &= __funnelshift_r(m[w], w + 1 < NW ? m[w + 1 < NW ? w + 1 : w] : 0u, 1);
            any |= m[w] != 0u;
        }
    }
    int t = 0;
#pragma unroll
    for (int w = 0; w < NW; ++w) t += __popc(starts[w]);
    unsigned k = 0;
    if (__any_sync(kFull, t > 1)) k = t > 1 ? pick_index(tie_word(gp, v, i, g), (uint32_t)t) : 0u;
    // The word that holds the k-th start, then its position there.
    int base = 0;
    unsigned word = starts[0];
#pragma unroll
    for (int w = 1; w < NW; ++w) {
        const unsigned c = (unsigned)__popc(word);
        if (base == 32 * (w - 1) && k >= c) {
            k -= c;
            word = starts[w];
            base = 32 * w;
        }
    }
    return select_at<N>(x, base + kth_bit(word, k));
}

// Adds the labels of the first 32 CHUNKS of the deg neighbours nbr to the
// warp's count table.
template <int CHUNKS>
__device__ __forceinline__ void table_insert(const GenParams &gp, const int32_t *__restrict__ col,
                                             const int *__restrict__ nbr, int deg, int *hkey, int *hcnt, int hbits)
{
    const int lane = threadIdx.x & 31;
    int x[CHUNKS];
#pragma unroll
    for (int k = 0; k < CHUNKS; ++k) {
        const int e = 32 * k + lane;
        x[k] = e < deg ? col[(size_t)checked_node(__ldg(nbr + e), gp.n) * gp.W] : (int)(0x80000000u | lane);
    }
#pragma unroll
    for (int k = 0; k < CHUNKS; ++k) {
        if (32 * k >= deg) break;  // (warp-uniform)
        // One insert per distinct label of the chunk, with its multiplicity.
        const unsigned peers = __match_any_sync(kFull, x[k]);
        if (x[k] >= 0 && (peers & ((1u << lane) - 1u)) == 0) {
            uint32_t h = hash_slot(x[k], hbits);
            // The table holds at most deg <= HS / 2 distinct labels, so an empty
            // or matching slot is always found.
            for (int probe = 0; probe < (1 << hbits); ++probe) {
                const int prev = atomicCAS(hkey + h, -1, x[k]);
                if (prev == -1 || prev == x[k]) {
                    atomicAdd(hcnt + h, __popc(peers));
                    break;
                }
                h = (h + 1) & (uint32_t)((1 << hbits) - 1);
            }
        }
    }
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
    // 2 deg <= the per-warp capacity (gp.hash_size), so the table fits.
    int hbits = 8;
    while ((1 << hbits) < 2 * deg) ++hbits;
    const int HS = 1 << hbits;
    int4 *key4 = reinterpret_cast<int4 *>(hkey), *cnt4 = reinterpret_cast<int4 *>(hcnt);
    for (int e = lane; e < HS / 4; e += 32) {
        key4[e] = make_int4(-1, -1, -1, -1);
        cnt4[e] = make_int4(0, 0, 0, 0);
    }
    __syncwarp();
    // Four labels a lane in flight, then their inserts (eight or sixteen spill
    // under the kernel's register cap: n = 10^6 2.91 -> 3.00 ms a generation).
    for (int e0 = 0; e0 < deg; e0 += 128) table_insert<4>(gp, child + i, nbr + e0, deg - e0, hkey, hcnt, hbits);
    __syncwarp();
    // Lane's slots: 4 (lane + 32 s) .. + 3, s < HS / 128 (2 .. 8).
    unsigned mx_l = 0;
    for (int s = 0; s < HS / 128; ++s) {
        const int4 c = cnt4[lane + 32 * s];
        mx_l = max(mx_l, (unsigned)max(max(c.x, c.y), max(c.z, c.w)));
    }
    const unsigned mx = __reduce_max_sync(kFull, mx_l);
    best_count = mx;
    unsigned act = 0;
    for (int s = 0; s < HS / 128; ++s) {
        const int4 c = cnt4[lane + 32 * s];
        act |= (((unsigned)c.x == mx ? 1u : 0u) | ((unsigned)c.y == mx ? 2u : 0u) | ((unsigned)c.z == mx ? 4u : 0u) |
                ((unsigned)c.w == mx ? 8u : 0u))
               << (4 * s);
    }
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
    for (unsigned m = act; m != 0u; m &= m - 1u) {
        const int s = __ffs((int)m) - 1;
        hcnt[at++] = hkey[4 * (lane + 32 * (s >> 2)) + (s & 3)];
    }
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

// Quad `lane_quad` of node v's row: Q gets the children's own labels and the
// histogram the unselected ones (mutating pairs add theirs once decided).
// Returns the selected children of the quad.
__device__ __forceinline__ unsigned take_quad(const GenParams &gp, int v, int deg, int quad, const int4 &out,
                                              uint32_t g, int4 *__restrict__ Q4, uint32_t *__restrict__ hist)
{
    const unsigned sel = deg > 0 ? selected(gp, v, quad, g) : 0u;
    Q4[(size_t)v * (gp.W >> 2) + quad] = out;
    if (deg > 0) {
        const int i0 = 4 * quad;
        if (i0 + 0 < gp.np && !(sel & 1u)) add_degree(gp, hist, out.x, i0 + 0, deg);
        if (i0 + 1 < gp.np && !(sel & 2u)) add_degree(gp, hist, out.y, i0 + 1, deg);
        if (i0 + 2 < gp.np && !(sel & 4u)) add_degree(gp, hist, out.z, i0 + 2, deg);
        if (i0 + 3 < gp.np && !(sel & 8u)) add_degree(gp, hist, out.w, i0 + 3, deg);
    }
    return sel;
}

// Appends each lane's selected children (bits of sel), tagged, to list[total
// ..]; returns their number. A lane's place: its count (0 .. 4) by bits.
__device__ __forceinline__ int list_selected(unsigned short *list, int total, unsigned sel, int tag)
{
    const unsigned lt = (1u << (threadIdx.x & 31)) - 1u;
    const int mine = __popc(sel);
    const unsigned b0 = __ballot_sync(kFull, mine & 1), b1 = __ballot_sync(kFull, mine & 2),
                   b2 = __ballot_sync(kFull, mine & 4);
    int at = total + __popc(b0 & lt) + 2 * __popc(b1 & lt) + 4 * __popc(b2 & lt);
#pragma unroll
    for (int k = 0; k < 4; ++k)
        if ((sel >> k) & 1u) list[at++] = (unsigned short)(tag + k);
    return __popc(b0) + 2 * __popc(b1) + 4 * __popc(b2);
}

// hint of a part of a node above degree 128: (pairs << 16) | pairs whose
// own label was on more than half of the neighbours, last generation; 0: no
// history. A quarter settled pays for the count.
__device__ __forceinline__ bool own_label_pays(uint32_t h)
{
    return h != 0u && 4u * (h & 0xffffu) >= (h >> 16);
}

// Part `part` of a node of degree kDeferMax + 1 .. kSharedTableMax (position
// idx): the quads q with q % gp.wide_parts == part, a warp per pair.
__device__ __noinline__ void wide_item(const GenParams &gp, int idx, int part, const int4 *__restrict__ nodes,
                                       const int4 *__restrict__ adj, const int32_t *__restrict__ child,
                                       int32_t *__restrict__ q, uint32_t *__restrict__ hist,
                                       uint32_t *__restrict__ hint, unsigned short *list, int *hkey, int *hcnt,
                                       uint32_t g)
{
    const int lane = threadIdx.x & 31;
    const int nq = gp.W >> 2;
    const int4 rec = __ldg(nodes + idx);
    const int v = rec.x, deg = rec.z;
    unsigned sel = 0;
    if (lane < nq && lane % gp.wide_parts == part) {
        const int4 out = reinterpret_cast<const int4 *>(child)[(size_t)v * nq + lane];
        sel = take_quad(gp, v, deg, lane, out, g, reinterpret_cast<int4 *>(q), hist);
    }
    const int total = list_selected(list, 0, sel, 4 * lane);
    uint32_t *h = hint + (idx - gp.n_hub) * gp.wide_parts + part;
    const bool fast = own_label_pays(*h);
    __syncwarp();
    int ok = 0;
    const int *nbr = reinterpret_cast<const int *>(adj + rec.y);
    for (int k = 0; k < total; ++k) {
        const int i = list[k];
        const int own = child[(size_t)v * gp.W + i];
        bool settled = false;
        if (fast) {
            int c = 0;
#pragma unroll 4
            for (int e = lane; e < deg; e += 32)
                c += child[(size_t)checked_node(__ldg(nbr + e), gp.n) * gp.W + i] == own;
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

// 16-byte words of a warp's shared memory in mutation_kernel.
__host__ __device__ __forceinline__ int mutation_warp_words(int np, int batch, int hash_size)
{
    return batch + (batch * np * 2 + 15) / 16 + hash_size / 2;
}

// The nodes at positions [first, last) of the order, of degree <= N.
//
// Bound by the half-rate integer pipe (58% of its peak at n = 40,000, the sorting
// networks) with waits for gathered labels between, so four-node batches in many
// blocks and 28 warps an SM; at n = 10^6 by DRAM and the L2's atomic rate (the
// histogram additions are 0.7 of 2.4 ms). Sizes of networks in steps of two, or
// 32 to 40 warps with fewer registers, are slower (instruction cache, spills).
// The launch for degrees up to 32, against one node a warp, staged labels and
// deferred votes of the higher degrees in launches behind it: n = 40,000 66.7 us
// + 12.7 -> 44.6, n = 170,001 270 us + 86 -> 205, n = 10^6 (tenth generation)
// 3.38 ms + 0.53 -> 2.0.
//
// The 128-entry network (1,471 comparators, for every degree of 65..128) keeps
// three blocks an SM at 168 registers and spills 268 bytes for it. Without the
// spills it is two blocks of 239: n = 5,000 of degree 100 94 -> 101 us a
// generation, n = 20,000 248 -> 245, n = 400,000 of degrees to 200 1.162 -> 1.152
// ms; not better, and slower where few blocks run.
//
// WIDE: the launch also takes the nodes of degree kDeferMax + 1 ..
// kSharedTableMax (positions n_hub .. n_hub + n_wide - 1). batch: nodes a warp
// takes at a time (<= kMutBatchMax).
template <int N, bool WIDE>
__global__ void __launch_bounds__(kMutBlock, N <= kLaneMax ? (WIDE ? 8 : 7) : N <= 40 ? 6 : N <= 64 ? 5 : 3)
mutation_kernel(const __grid_constant__ GenParams gp, int first, int last, const int4 *__restrict__ nodes,
                const int4 *__restrict__ adj, const int32_t *__restrict__ child, int32_t *__restrict__ q,
                const uint32_t *__restrict__ gen_ptr, uint32_t *__restrict__ hist, unsigned long long *__restrict__ acc,
                uint32_t *__restrict__ hint, int batch)
{
    // Per warp: the batch's node records, the pair list (two bytes a pair; sized
    // to the batch, so that the rest of the memory is L1 cache) and, WIDE, a
    // count table.
    extern __shared__ int4 s_warp[];
    cudaGridDependencySynchronize();  // (see overlap_next)
    const int W = gp.W;
    const int nq = W >> 2;
    const uint32_t g = *gen_ptr;
    const int lane = threadIdx.x & 31;
    const int wib = threadIdx.x >> 5;
    int4 *recs = s_warp + wib * mutation_warp_words(gp.np, batch, WIDE ? gp.hash_size : 0);
    unsigned short *list = reinterpret_cast<unsigned short *>(recs + batch);
    const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int4 *__restrict__ C4 = reinterpret_cast<const int4 *>(child);
    int4 *__restrict__ Q4 = reinterpret_cast<int4 *>(q);

    // The evaluation that follows accumulates into acc: clear it here. The
    // histogram is zero on entry (the previous evaluation's square sweep
    // cleared it) and receives D below.
    if (N <= kLaneMax && blockIdx.x == 0)
        for (int t = threadIdx.x; t < 2 * kMaxPop; t += blockDim.x) acc[t] = 0;

    // Nodes in degree-descending order: every warp starts with one of the
    // costliest batches, which balances the grid-stride loop.
    const int wide = WIDE ? gp.n_wide * gp.wide_parts : 0;
    const int items = wide + (last - first + batch - 1) / batch;
    const unsigned inv_nq = (65536u + (unsigned)nq - 1u) / (unsigned)nq;  // t / nq = t * inv_nq >> 16, t < 2^10
    for (int item = warp; item < items; item += nwarps) {
        if (WIDE && item < wide) {
            int *table = reinterpret_cast<int *>(recs + mutation_warp_words(gp.np, batch, 0));
            wide_item(gp, gp.n_hub + item / gp.wide_parts, item % gp.wide_parts, nodes, adj, child, q, hist, hint, list,
                      table, table + gp.hash_size, g);
            __syncwarp();
            continue;
        }
        const int idx0 = first + (item - wide) * batch;
        const int nb = min(batch, last - idx0);
        if (lane < nb) recs[lane] = __ldg(nodes + idx0 + lane);
        __syncwarp();
        // The batch's rows, a quad per lane; the next quad is requested before
        // this one is processed.
        const int quads = nb * nq;
        auto quad_of = [&](int t, int &k) {
            k = (int)(((unsigned)t * inv_nq) >> 16);
            return t - k * nq;
        };
        int total = 0;
        int k = 0, quad = 0, v = 0, deg = 0;
        int4 row = make_int4(0, 0, 0, 0);
        if (lane < quads) {
            quad = quad_of(lane, k);
            v = recs[k].x;
            deg = recs[k].z;
            row = C4[(size_t)v * nq + quad];
        }
        for (int t = lane; t - lane < quads; t += 32) {
            const int4 out = row;
            const int cur_k = k, cur_quad = quad, cur_v = v, cur_deg = deg;
            if (t + 32 < quads) {
                quad = quad_of(t + 32, k);
                v = recs[k].x;
                deg = recs[k].z;
                row = C4[(size_t)v * nq + quad];
            }
            unsigned sel = 0;
            if (t < quads) sel = take_quad(gp, cur_v, cur_deg, cur_quad, out, g, Q4, hist);
            total += list_selected(list, total, sel, cur_k * kMaxPop + 4 * cur_quad);
        }
        __syncwarp();

        // The votes (the list's degrees descend).
        for (int base = 0; base < total; base += 32) {
            const bool has = base + lane < total;
            const int e = has ? list[base + lane] : 0;
            const int i = e % kMaxPop;
            const int4 r = recs[e / kMaxPop];
            const int deg = has ? r.z : 0;
            int res;
            if constexpr (N > kLaneMax) {
                res = lane_vote<N>(gp, adj, child, r.x, i, r.y, deg, g);
            } else {
                const int top = __reduce_max_sync(kFull, deg);
                if (top <= 8) res = lane_vote<8>(gp, adj, child, r.x, i, r.y, deg, g);
                else if (top <= 12) res = lane_vote<12>(gp, adj, child, r.x, i, r.y, deg, g);
                else if (top <= 16) res = lane_vote<16>(gp, adj, child, r.x, i, r.y, deg, g);
                else if (top <= 20) res = lane_vote<20>(gp, adj, child, r.x, i, r.y, deg, g);
                else if (top <= 24) res = lane_vote<24>(gp, adj, child, r.x, i, r.y, deg, g);
                else if (top <= 28) res = lane_vote<28>(gp, adj, child, r.x, i, r.y, deg, g);
                else res = lane_vote<32>(gp, adj, child, r.x, i, r.y, deg, g);
            }
            if (has) {
                q[(size_t)r.x * W + i] = res;
                add_degree(gp, hist, res, i, deg);
            }
        }
        __syncwarp();
    }
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

// Exact neighbour-majority of one pair by the whole block: a count table of
// the smallest power of two >= 2 deg slots (at least 2048). Returns the label
// to every thread; the tables are free on return.
__device__ __forceinline__ int block_mode_table(const GenParams &gp, const int32_t *__restrict__ col,
                                                const int *__restrict__ nbr, int deg, int v, int i, int *hkey,
                                                int hbits, unsigned *s_red, int *s_tied, uint32_t g, unsigned &mx)
{
    const int lane = threadIdx.x & 31;
    const int HS = 1 << hbits;
    int *hcnt = hkey + HS;
    for (int s = threadIdx.x; s < HS; s += kHubBlock) {
        hkey[s] = -1;
        hcnt[s] = 0;
    }
    if (threadIdx.x == 0) *s_tied = 0;
    __syncthreads();
    for (int j0 = 0; j0 < deg; j0 += 4 * kHubBlock) {
        int x[4];  // four labels in flight per thread
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int j = j0 + k * kHubBlock + (int)threadIdx.x;
            x[k] = j < deg ? col[(size_t)checked_node(__ldg(nbr + j), gp.n) * gp.W] : (int)(0x80000000u | lane);
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            // One insert per distinct label of the warp's neighbours.
            const unsigned peers = __match_any_sync(kFull, x[k]);
            if (x[k] >= 0 && (peers & ((1u << lane) - 1u)) == 0) {
                uint32_t h = hash_slot(x[k], hbits);
                for (int probe = 0; probe < HS; ++probe) {  // (at most HS / 2 distinct labels: a slot is found)
                    const int prev = atomicCAS(hkey + h, -1, x[k]);
                    if (prev == -1 || prev == x[k]) {
                        atomicAdd(hcnt + h, __popc(peers));
                        break;
                    }
                    h = (h + 1) & (uint32_t)(HS - 1);
                }
            }
        }
    }
    __syncthreads();
    unsigned my = 0;
    for (int s = threadIdx.x; s < HS; s += kHubBlock) my = max(my, (unsigned)hcnt[s]);
    mx = hub_reduce<true>(my, s_red);
    // The tied labels, compacted to hcnt[0, tied) once every thread has read
    // its slots' counts.
    for (int s = threadIdx.x; s < HS; s += kHubBlock)
        if ((unsigned)hcnt[s] != mx) hkey[s] = -1;
    __syncthreads();
    for (int s = threadIdx.x; s < HS; s += kHubBlock) {  // (HS is a multiple of the block: warps stay whole)
        const int key = hkey[s];
        const unsigned who = __ballot_sync(kFull, key >= 0);
        int at = 0;
        if (lane == 0 && who) at = atomicAdd(s_tied, __popc(who));
        at = __shfl_sync(kFull, at, 0);
        if (key >= 0) hcnt[at + __popc(who & ((1u << lane) - 1u))] = key;
    }
    __syncthreads();
    const int tied = *s_tied;
    int res = hcnt[0];
    if (tied > 1) {
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
        res = (int)prefix;
    }
    __syncthreads();
    return res;
}

// The hubs, degree above kSharedTableMax (positions 0 .. n_hub - 1): a block
// per hub and quad of children, about one pair. The own label's count if the
// last generation says it pays, else (or if it leaves the pair open) the exact
// vote with a count table in shared memory if it fits there
// (gp.hub_smem_hs), else in the block's slice of global scratch (2 gp.hub_hs
// ints). A block per pair keeps a hub of thousands of neighbours off the
// critical path: one warp per pair is a chain of deg / 32 dependent inserts.
// The hint slot of (hub, quad) is that block's alone.
__global__ void __launch_bounds__(kHubBlock)
mutation_hub_kernel(const __grid_constant__ GenParams gp, const int4 *__restrict__ nodes,
                    const int4 *__restrict__ adj, const int32_t *__restrict__ child, int32_t *__restrict__ q,
                    const uint32_t *__restrict__ gen_ptr, uint32_t *__restrict__ hist, uint32_t *__restrict__ hint,
                    int *__restrict__ hub_table)
{
    extern __shared__ int s_table[];  // [2 gp.hub_smem_hs]
    __shared__ unsigned s_red[kHubBlock / 32];
    __shared__ int s_tied;
    cudaGridDependencySynchronize();  // (see overlap_next)
    const uint32_t g = *gen_ptr;
    const int nq = gp.W >> 2;
    for (int t = blockIdx.x; t < gp.n_hub * nq; t += gridDim.x) {
        const int idx = t / nq, quad = t % nq;
        const int4 rec = __ldg(nodes + idx);
        const int v = rec.x, deg = min(rec.z, gp.hub_hs / 2);
        const int *nbr = reinterpret_cast<const int *>(adj + rec.y);
        uint32_t *h = hint + gp.n_wide * gp.wide_parts + t;
        const bool fast = own_label_pays(*h);
        const int4 own4 = reinterpret_cast<const int4 *>(child)[(size_t)v * nq + quad];
        unsigned sel;
        if (threadIdx.x == 0)
            sel = take_quad(gp, v, deg, quad, own4, g, reinterpret_cast<int4 *>(q), hist);
        else
            sel = selected(gp, v, quad, g);
        int hbits = 11;
        while ((1 << hbits) < 2 * deg) ++hbits;
        int *hkey = (1 << hbits) <= gp.hub_smem_hs ? s_table : hub_table + (size_t)blockIdx.x * 2 * gp.hub_hs;
        const int pairs = __popc(sel);
        int ok = 0;
        __syncthreads();  // (every thread has read the hint)
        for (int k = 0; k < 4; ++k) {
            if (!((sel >> k) & 1u)) continue;  // (block-uniform)
            const int i = 4 * quad + k;
            const int own = k == 0 ? own4.x : k == 1 ? own4.y : k == 2 ? own4.z : own4.w;
            const int32_t *col = child + i;
            bool settled = false;
            if (fast) {
                unsigned c = 0;
#pragma unroll 4
                for (int j = threadIdx.x; j < deg; j += kHubBlock)
                    c += col[(size_t)checked_node(__ldg(nbr + j), gp.n) * gp.W] == own ? 1u : 0u;
                settled = 2 * (int)hub_reduce<false>(c, s_red) > deg;
            }
            int lab = own;
            if (!settled) {
                unsigned mx = 0;
                lab = block_mode_table(gp, col, nbr, deg, v, i, hkey, hbits, s_red, &s_tied, g, mx);
                settled = !fast && lab == own && 2 * (int)mx > deg;
            }
            ok += settled ? 1 : 0;
            if (threadIdx.x == 0) {
                if (lab != own) q[(size_t)v * gp.W + i] = lab;
                add_degree(gp, hist, lab, i, deg);
            }
        }
        if (threadIdx.x == 0) *h = ((uint32_t)pairs << 16) | (uint32_t)ok;
    }
}

template <int EMAX>
size_t crossover_smem(int W)
{
    const int per_warp = 32 / (W >> 2);
    return sizeof(int) * ((EMAX > 4 ? EMAX * kMaxPop : 0) + (kBlock / 32) * per_warp * (2 * W + kRowPad));
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

namespace {

template <int EMAX>
int crossover_occupancy(int W)
{
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, crossover_kernel<EMAX>, kBlock, crossover_smem<EMAX>(W));
    return per_sm < 1 ? 1 : per_sm;
}

template <int EMAX>
void crossover_launch(const GenParams &gp, const PopState &ps, int grid, cudaStream_t s)
{
    crossover_kernel<EMAX><<<grid, kBlock, crossover_smem<EMAX>(gp.W), s>>>(
        gp, ps.buf[0], ps.buf[1], ps.buf[0], ps.buf[1], ps.q, ps.c, ps.keep, ps.par_r, ps.copy_r, ps.gen);
}

}  // namespace

int grid_for_crossover(int sms, int es, int W)
{
    const int per_sm = es <= 4   ? crossover_occupancy<4>(W)
                       : es <= 8 ? crossover_occupancy<8>(W)
                                 : crossover_occupancy<16>(W);
    return sms * per_sm;
}

cudaError_t launch_crossover(const GenParams &gp, const PopState &ps, int grid, cudaStream_t s)
{
    if (gp.es <= 4) crossover_launch<4>(gp, ps, grid, s);
    else if (gp.es <= 8) crossover_launch<8>(gp, ps, grid, s);
    else crossover_launch<16>(gp, ps, grid, s);
    return cudaGetLastError();
}

cudaError_t launch_crossover_multi(const BatchMember *members, const int *starts, int count, int blocks, int es_max,
                                   int rows_max, cudaStream_t s)
{
    if (blocks <= 0) return cudaSuccess;
    // rows_max: the largest member's words of staged rows per warp.
    const size_t rows = sizeof(int) * (kBlock / 32) * (size_t)rows_max;
    if (es_max <= 4)
        crossover_multi_kernel<4><<<blocks, kBlock, rows, s>>>(members, starts, count);
    else if (es_max <= 8)
        crossover_multi_kernel<8><<<blocks, kBlock, rows + sizeof(int) * 8 * kMaxPop, s>>>(members, starts, count);
    else
        crossover_multi_kernel<16><<<blocks, kBlock, rows + sizeof(int) * 16 * kMaxPop, s>>>(members, starts, count);
    return cudaGetLastError();
}

int crossover_row_words(int W)
{
    return 32 / (W >> 2) * (2 * W + kRowPad);
}

int mutation_warps_per_block()
{
    return kMutBlock / 32;
}

namespace {

// Class c: 0: degree <= 32 (and the wide nodes), 1: 33..64, 2: 65..128.
using MutationFn = void (*)(GenParams, int, int, const int4 *, const int4 *, const int32_t *, int32_t *,
                            const uint32_t *, uint32_t *, unsigned long long *, uint32_t *, int);

MutationFn mutation_fn(int cls, int vote_n0, bool wide)
{
    if (cls == 0) return wide ? mutation_kernel<kLaneMax, true> : mutation_kernel<kLaneMax, false>;
    if (cls == 2) return mutation_kernel<kDeferMax, false>;
    // The class's network holds the graph's largest degree in it.
    switch (vote_n0) {
    case 40: return mutation_kernel<40, false>;
    case 48: return mutation_kernel<48, false>;
    case 56: return mutation_kernel<56, false>;
    default: return mutation_kernel<2 * kLaneMax, false>;
    }
}

}  // namespace

namespace {

size_t mutation_smem(int np, int batch, int cls, int hash_size)
{
    return (size_t)(kMutBlock / 32) * mutation_warp_words(np, batch, cls == 0 ? hash_size : 0) * sizeof(int4);
}

}  // namespace

int grid_for_mutation(int sms, int cls, int vote_n0, int hash_size, int np, int batch)
{
    const MutationFn fn = mutation_fn(cls, vote_n0, hash_size > 0);
    const size_t smem = mutation_smem(np, batch, cls, hash_size);
    cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kMutBlock, smem);
    return sms * (per_sm < 1 ? 1 : per_sm);
}

// Blocks of the hub kernel: as many as its shared table lets be resident.
int grid_for_hubs(int sms, int smem_hs)
{
    const int smem = 2 * smem_hs * (int)sizeof(int);
    // (The limit is the function's, for every context: always the largest table.)
    cudaFuncSetAttribute(mutation_hub_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         2 * kHubSmemSlots * (int)sizeof(int));
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, mutation_hub_kernel, kHubBlock, smem);
    return sms * (per_sm < 1 ? 1 : per_sm);
}

cudaError_t launch_mutation(const GenParams &gp, const PopState &ps, const int4 *nodes, const int4 *adj,
                            const MutationShape &shape, cudaStream_t s)
{
    // The launches are independent of each other: on a capturing stream they
    // become parallel branches, the longest votes first.
    Branches br(s, gp.n_hub > 0 || gp.n_vote[0] > 0 || gp.n_vote[1] > 0);
    cudaError_t o = cudaSuccess;
    if (gp.n_hub > 0) {
        o = overlap_next(s);
        mutation_hub_kernel<<<shape.hub_blocks, kHubBlock, 2 * gp.hub_smem_hs * sizeof(int), s>>>(
            gp, nodes, adj, ps.c, ps.q, ps.gen, ps.hist, ps.hint, ps.hub_table);
        br.next();
    }
    int first = gp.n_hub + gp.n_wide;
    for (int cls = 2; cls >= 0; --cls) {
        const int last = cls == 0 ? gp.n : first + gp.n_vote[cls - 1];
        if (cls == 0 || last > first) {
            if (o == cudaSuccess) o = overlap_next(s);
            mutation_fn(cls, gp.vote_n0, gp.hash_size > 0)<<<shape.grid[cls], kMutBlock,
                                                             mutation_smem(gp.np, shape.batch[cls], cls, gp.hash_size),
                                                             s>>>(
                gp, first, last, nodes, adj, ps.c, ps.q, ps.gen, ps.hist, ps.acc, ps.hint, shape.batch[cls]);
            br.next();
        }
        first = last;
    }
    const cudaError_t e = cudaGetLastError();
    return e != cudaSuccess ? e : o != cudaSuccess ? o : br.join();
}

}  // namespace mocd

namespace mocd {
cudaError_t check_record_variation(unsigned long long *out, bool reset)
{
    return check_record(out, reset);
}
}  // namespace mocd
