// k_eval.cu -- objective evaluation of a whole population (Eq. objectives,
// Sec. 4.1; Alg. 1 EvaluateIndividual, run for every individual at once).
//
// For each individual i the kernel accumulates
//   intra_i = #{{v, u} in E : L_i(v) = L_i(u)}   (= sum_c |E(c)|)
//   S_i     = sum_c D_c^2,  D_c = sum_{v : L_i(v) = c} deg v
// exactly in integers. Each undirected edge is counted once, from one
// endpoint. A context (its generations, its initial population, mocd_evaluate)
// walks an oriented adjacency that lists every edge once, at its endpoint of
// lower (degree, id), so the rows it reads are the higher-degree endpoints' --
// fewer distinct rows, each read more often, which keeps more of them in L2.
// mocd_evaluate_noalloc has only the caller's full adjacency, of which a warp
// reads the label rows of the neighbours u > v.
//
// Layout is node-major: lane q of the lanes that hold node v has the int4 of
// labels of individuals 4q..4q+3, so each neighbour u costs one coalesced row
// read of all individuals' labels instead of N_p scattered 4-byte gathers, and
// the adjacency is streamed once per population, not once per individual. With
// the oriented adjacency a warp takes as many nodes at a time as its lanes hold
// rows, with the full one a node.
//
// S without a sweep over the histogram D: when node v adds deg(v) to D_c, the
// atomic returns the old total o, and (o + d)^2 - o^2 = 2 o d + d^2. Summed
// over every addition these increments telescope to D_c^2 whatever the order
// of the atomics, so S is exact and deterministic. (Reductions and a sweep
// afterwards took 20 us more at n = 51,300, count 81.) Histogram layout: with
// the oriented adjacency (contexts) label-major, D of (individual i, label c) at
// c * W + i, as the generations have it: one atomic instruction of a warp (25
// individuals of node v) lands in few cache lines whenever individuals share
// v's label. With the full adjacency (mocd_evaluate_noalloc) individual-major,
// i * n + c: cells of different individuals then do not share sectors, which
// additions take turns on (n = 60,000, 69 labellings: of one community each
// 1,224 us label-major and 140 so, of some 500 communities 62 and 64).
//
// Inside a generation the D histogram is not built here: the mutation kernel,
// which writes every child's final label of node v, adds deg(v) to the
// label-major cell of that label as it goes (fire-and-forget reductions that
// overlap its own latency-bound work). The evaluation of the offspring then
// counts intra (ADD = false) and, in the same launch once a warp's nodes are
// done, forms S = sum_c D_c^2 in a coalesced sweep of the histogram rows,
// zeroing them for the next generation. While the labels are still nearly all
// distinct, the N_p n histogram additions land on different sectors, which at n
// = 10^6 (a 400 MB histogram) cost a DRAM read and write-back each; done by the
// mutation kernel, that traffic overlaps with its own work instead of stalling
// the evaluation's row stream.
//
// Labellings given from outside, up to 40,960 nodes: the histogram of each is one
// block's shared memory (hist_block_kernel), beside the edge count.
#include <algorithm>

#include "mocd_check.cuh"
#include "mocd_internal.h"

namespace mocd {

namespace {

// Blocks of the edge count that an SM holds, by their registers (48 and 62).
constexpr int kFullBlocks = 5;
constexpr int kOrientedBlocks = 4;

// FULL: row_ptr / col_idx hold both directions of every edge, rows by node id;
// else each edge once, lists by position in the order (the oriented adjacency).
// ADD: the degrees (from deg_ptr) go into the histogram; otherwise a histogram
// (if given) is complete: square and clear it.
template <bool FULL, bool ADD>
__device__ __forceinline__ void evaluate_body(int n, int W, int count,
                                              const int32_t *__restrict__ deg_ptr,
                                              const int32_t *__restrict__ row_ptr,
                                              const int32_t *__restrict__ col_idx,
                                              const int32_t *__restrict__ labels, uint32_t *__restrict__ hist,
                                              unsigned long long *__restrict__ intra,
                                              unsigned long long *__restrict__ sumsq,
                                              const int32_t *__restrict__ order, int vblock, int vgrid,
                                              bool beside = false)
{
    // The block's sums: the edge count (at most m < 2^30), then S in limbs of 22
    // bits, 256 of which fit a word. 64-bit additions in shared memory are loops
    // of compare and swap, in which the lanes that hold one quad for different
    // nodes take turns (n = 500, N_p 4: 30 us a launch with them, 8 with these).
    constexpr int kLimbBits = 22;
    constexpr uint32_t kLimb = (1u << kLimbBits) - 1u;
    static_assert(kBlock <= 1 << (32 - kLimbBits), "a limb's sum fits a word");
    __shared__ uint32_t s_sum[4][kMaxPop];  // [..][individual % 4][quad]
    __shared__ int s_nb[FULL ? kBlock : 1];  // FULL, per warp: the chunk's neighbours u > v
    for (int t = threadIdx.x; t < 4 * kMaxPop; t += blockDim.x) s_sum[0][t] = 0;
    __syncthreads();

    const int nq = W >> 2;
    const int wlane = threadIdx.x & 31;
    // A warp takes as many nodes at a time as its lanes hold rows (FULL: one).
    const int per_warp = FULL ? 1 : 32 / nq;
    const int sub = FULL ? 0 : wlane / nq;
    const int lane = wlane - sub * nq;  // the quad of individuals
    const bool active = sub < per_warp && lane < nq;
    const int first = ((vblock * blockDim.x + threadIdx.x) >> 5) * per_warp + sub;
    const int nodes = ((vgrid * blockDim.x) >> 5) * per_warp;  // taken at a time by all warps
    const int4 *__restrict__ L4 = reinterpret_cast<const int4 *>(labels);
    const int i0 = 4 * lane;

    uint32_t c0 = 0, c1 = 0, c2 = 0, c3 = 0;
    unsigned long long q0 = 0, q1 = 0, q2 = 0, q3 = 0;

    // Counts, per individual, the rows u (-1: none) that agree with `own`: four
    // independent row loads in flight per lane.
    auto count4 = [&](const int (&u)[4], const int4 &own) {
        int4 a[4];
#pragma unroll
        for (int t = 0; t < 4; ++t)
            a[t] = active && u[t] >= 0 ? L4[(size_t)u[t] * nq + lane] : make_int4(-1, -1, -1, -1);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            c0 += a[t].x == own.x;
            c1 += a[t].y == own.y;
            c2 += a[t].z == own.z;
            c3 += a[t].w == own.w;
        }
    };
    // Adds degree d of node v to the histogram cells of its labels.
    auto add = [&](int v, const int4 &own, unsigned d) {
        if (!active || d == 0) return;
        const unsigned long long d2 = (unsigned long long)d * d, dd = 2ull * d;
        auto cell = [&](int k, int c) {
            return FULL ? hist + (size_t)(i0 + k) * n + c : hist + (size_t)c * W + i0 + k;
        };
        if (i0 + 0 < count && MOCD_CHECK((unsigned)own.x < (unsigned)n, kCheckLabel, v))
            q0 += dd * atomicAdd(cell(0, own.x), d) + d2;
        if (i0 + 1 < count && MOCD_CHECK((unsigned)own.y < (unsigned)n, kCheckLabel, v))
            q1 += dd * atomicAdd(cell(1, own.y), d) + d2;
        if (i0 + 2 < count && MOCD_CHECK((unsigned)own.z < (unsigned)n, kCheckLabel, v))
            q2 += dd * atomicAdd(cell(2, own.z), d) + d2;
        if (i0 + 3 < count && MOCD_CHECK((unsigned)own.w < (unsigned)n, kCheckLabel, v))
            q3 += dd * atomicAdd(cell(3, own.w), d) + d2;
    };
    if constexpr (FULL) {
        int *nb = s_nb + (threadIdx.x & ~31);
        for (int v = first; v < n; v += nodes) {
            const int beg = __ldg(row_ptr + v);
            const int end = __ldg(row_ptr + v + 1);
            if (!MOCD_CHECK(end >= beg, kCheckRowPtr, v)) continue;  // (warp-uniform)
            const int4 own = active ? L4[(size_t)v * nq + lane] : make_int4(0, 0, 0, 0);
            for (int e0 = beg; e0 < end; e0 += 32) {
                const int cnt = min(32, end - e0);
                const int my_u = wlane < cnt ? __ldg(col_idx + e0 + wlane) : 0;
                // Keep the neighbours u > v, compacted.
                const bool up = wlane < cnt && my_u > v && MOCD_CHECK(my_u < n, kCheckNode, v);
                const unsigned upm = __ballot_sync(0xffffffffu, up);
                const int cu = __popc(upm);
                if (up) nb[__popc(upm & ((1u << wlane) - 1u))] = my_u;
                __syncwarp();
                for (int j0 = 0; j0 < cu; j0 += 4) {
                    int u[4];
#pragma unroll
                    for (int t = 0; t < 4; ++t) u[t] = j0 + t < cu ? nb[j0 + t] : -1;
                    count4(u, own);
                }
                __syncwarp();
            }
            if (ADD) add(v, own, (unsigned)(end - beg));
        }
    } else {
        // A node takes a chain of dependent loads (position -> id and list -> own row
        // and entries -> rows) and has ten entries or so: the kernel is bound by
        // that chain unless the next nodes' loads are under way. While a node's
        // rows are compared, the next one's own row and first entries and the
        // one after's id and list bounds are requested.
        auto entries = [&](int e, int end, int (&u)[4]) {
#pragma unroll
            for (int t = 0; t < 4; ++t) {
                u[t] = e + t < end ? __ldg(col_idx + e + t) : -1;
                if (!MOCD_CHECK(u[t] < n, kCheckNode, e)) u[t] = -1;
            }
        };
        auto head = [&](long long idx, int &v, int &beg, int &end) {
            const bool in = active && idx < n;
            v = in ? __ldg(order + idx) : 0;
            beg = in ? __ldg(row_ptr + idx) : 0;
            end = in ? __ldg(row_ptr + idx + 1) : 0;
            if (!MOCD_CHECK(end >= beg, kCheckRowPtr, v)) end = beg;
        };
        int v, beg, end, v1, beg1, end1, u[4];
        head(first, v, beg, end);
        head((long long)first + nodes, v1, beg1, end1);
        int4 own = active && first < n ? L4[(size_t)v * nq + lane] : make_int4(0, 0, 0, 0);
        entries(beg, end, u);
        for (long long idx = first; active && idx < n; idx += nodes) {
            int v2, beg2, end2, u1[4];
            const int4 own1 = L4[(size_t)v1 * nq + lane];
            entries(beg1, end1, u1);
            head(idx + 2ll * nodes, v2, beg2, end2);
            for (int e = beg; e < end; e += 4) {
                const int cur[4] = {u[0], u[1], u[2], u[3]};
                entries(e + 4, end, u);
                count4(cur, own);
            }
            if (ADD) add(v, own, (unsigned)(__ldg(deg_ptr + v + 1) - __ldg(deg_ptr + v)));
            v = v1;
            beg = beg1;
            end = end1;
            own = own1;
            v1 = v2;
            beg1 = beg2;
            end1 = end2;
#pragma unroll
            for (int t = 0; t < 4; ++t) u[t] = u1[t];
        }
    }

    if (!ADD && active && hist) {
        // S from the histogram [n][W] that the mutation kernel built: a warp
        // per row, lane q the int4 of individuals 4q..4q+3; every non-zero
        // cell is squared and cleared. D_c^2 < 2^62 and S <= (2m)^2, so the
        // 64-bit sums are exact.
        uint4 *__restrict__ H4 = reinterpret_cast<uint4 *>(hist);
        // Four rows in flight per lane.
        for (long long c0 = first; c0 < n; c0 += 4ll * nodes) {
            uint4 x[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const long long c = c0 + (long long)k * nodes;
                x[k] = c < n ? H4[(size_t)c * nq + lane] : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const long long c = c0 + (long long)k * nodes;
                if (x[k].x | x[k].y | x[k].z | x[k].w) {
                    q0 += (unsigned long long)x[k].x * x[k].x;
                    q1 += (unsigned long long)x[k].y * x[k].y;
                    q2 += (unsigned long long)x[k].z * x[k].z;
                    q3 += (unsigned long long)x[k].w * x[k].w;
                    H4[(size_t)c * nq + lane] = make_uint4(0, 0, 0, 0);
                }
            }
        }
    }
    if (active) {
        auto put = [&](int k, uint32_t c, unsigned long long q) {
            if (i0 + k >= count) return;
            uint32_t *at = &s_sum[0][k * (kMaxPop / 4) + lane];
            atomicAdd(at, c);
            atomicAdd(at + kMaxPop, (uint32_t)q & kLimb);
            atomicAdd(at + 2 * kMaxPop, (uint32_t)(q >> kLimbBits) & kLimb);
            atomicAdd(at + 3 * kMaxPop, (uint32_t)(q >> (2 * kLimbBits)));
        };
        put(0, c0, q0);
        put(1, c1, q1);
        put(2, c2, q2);
        put(3, c3, q3);
    }
    __syncthreads();
    if (beside) cudaGridDependencySynchronize();  // (it cleared intra)
    for (int t = threadIdx.x; t < count; t += blockDim.x) {
        const uint32_t *at = &s_sum[0][(t & 3) * (kMaxPop / 4) + (t >> 2)];
        const unsigned long long q = at[kMaxPop] + ((unsigned long long)at[2 * kMaxPop] << kLimbBits) +
                                     ((unsigned long long)at[3 * kMaxPop] << (2 * kLimbBits));
        if (at[0]) atomicAdd(intra + t, (unsigned long long)at[0]);
        if (q) atomicAdd(sumsq + t, q);
    }
}

// beside: the launch before this one on the stream (hist_block_kernel) runs
// beside it, until the sums are added to intra, which that launch cleared.
template <bool FULL, bool ADD>
__global__ void __launch_bounds__(kBlock, FULL ? kFullBlocks : kOrientedBlocks)
evaluate_kernel(int n, int W, int count, const int32_t *__restrict__ deg_ptr,
                const int32_t *__restrict__ row_ptr,
                const int32_t *__restrict__ col_idx, const int32_t *__restrict__ labels,
                uint32_t *__restrict__ hist, unsigned long long *__restrict__ intra,
                unsigned long long *__restrict__ sumsq, const int32_t *__restrict__ order, bool beside)
{
    // (see overlap_next) The selection that follows is one block: it may come in
    // as soon as every block here runs.
    if (!beside) cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
    evaluate_body<FULL, ADD>(n, W, count, deg_ptr, row_ptr, col_idx, labels, hist, intra, sumsq, order,
                             blockIdx.x, gridDim.x, beside);
}

// S of individual blockIdx.x with its histogram in shared memory (n words): no
// global atomics, nothing to clear. The block reads one label a row, an eighth
// of each sector, which costs less than n additions at the L2's atomic rate
// do. out: S of each individual; intra: 0 for each.
constexpr int kHistThreads = 1024;
constexpr size_t kPlainSharedBytes = 47 * 1024;  // dynamic shared memory a launch gets unasked, beside the static
__global__ void __launch_bounds__(kHistThreads)
hist_block_kernel(int n, int W, const int32_t *__restrict__ deg_ptr, const int32_t *__restrict__ labels,
                  unsigned long long *__restrict__ out, unsigned long long *__restrict__ intra)
{
    cudaTriggerProgrammaticLaunchCompletion();  // the edge count runs beside this
    extern __shared__ uint32_t s_hist[];
    __shared__ unsigned long long s_sum[kHistThreads / 32];
    for (int c = threadIdx.x; c < n; c += kHistThreads) s_hist[c] = 0;
    __syncthreads();
    const int32_t *col = labels + blockIdx.x;
    for (int v0 = threadIdx.x; v0 < n; v0 += 8 * kHistThreads) {
        int lab[8], d[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const int v = v0 + u * kHistThreads;
            lab[u] = v < n ? col[(size_t)v * W] : 0;
            d[u] = v < n ? __ldg(deg_ptr + v + 1) - __ldg(deg_ptr + v) : 0;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u)
            if (d[u] > 0 && MOCD_CHECK((unsigned)lab[u] < (unsigned)n, kCheckLabel, v0))
                atomicAdd(s_hist + lab[u], (unsigned)d[u]);
    }
    __syncthreads();
    unsigned long long q = 0;
    for (int c = threadIdx.x; c < n; c += kHistThreads) q += (unsigned long long)s_hist[c] * s_hist[c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_down_sync(0xffffffffu, q, o);
    if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = q;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    q = s_sum[threadIdx.x];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) q += __shfl_down_sync(0xffffffffu, q, o);
    if (threadIdx.x == 0) {
        out[blockIdx.x] = q;
        intra[blockIdx.x] = 0;
    }
}

// The offspring evaluation of every member of a batch in one launch: members
// own consecutive block ranges (starts[k] .. starts[k + 1] - 1).
__global__ void __launch_bounds__(kBlock, 4)
evaluate_multi_kernel(const BatchMember *__restrict__ members, const int *__restrict__ starts, int count)
{
    const int bk = (int)blockIdx.x;
    int lo = 0, hi = count;  // starts[lo] <= bk < starts[hi]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(starts + mid) <= bk) lo = mid;
        else hi = mid;
    }
    const BatchMember &mb = members[lo];
    const int b0 = __ldg(starts + lo);
    evaluate_body<false, false>(mb.gp.n, mb.gp.W, mb.gp.np, nullptr, mb.eptr, mb.eidx, mb.ps.q, mb.ps.hist, mb.ps.acc,
                         mb.ps.acc + kMaxPop, mb.order, bk - b0, __ldg(starts + lo + 1) - b0);
}

}  // namespace

int grid_for_eval_intra(int sms)
{
    int per_sm = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, evaluate_kernel<false, false>, kBlock, 0);
    if (per_sm < 1) per_sm = 1;
    return sms * per_sm;
}

// A histogram block takes a time of its own, however few labellings there are
// (it reads a sector a node), and longer where a row is 128 or 256 bytes; the
// histogram in global memory takes longer the more there are. With the full
// adjacency, whose launch has no other work to hide either, global memory is
// the faster one in a band of few labellings of many nodes (us a call, full
// adjacency of mean degree 16, blocks / global): n = 27,000, 32 labellings 35.7
// / 35.2, 48 34.3 / 43.0; n = 34,000, 32 47.5 / 36.1, 56 41.7 / 48.6, 100 44.6 /
// 61.1; n = 40,960, 20 39.1 / 39.4, 36 46.8 / 41.3, 64 56.2 / 54.4, 100 52.7 /
// 71.9. With the oriented adjacency the blocks are no slower up to their limit,
// and several times faster where the labels are few.
bool evaluate_needs_histogram(int64_t n, int W, bool full)
{
    if (n * (int64_t)sizeof(uint32_t) > kHistBlockBytes) return true;
    return full && ((n > 27000 && (W == 32 || W == 64)) || (n > 30000 && W > 24 && W <= 48));
}

cudaError_t launch_evaluate(int n, int W, int count, bool full, const int32_t *deg_ptr,
                            const int32_t *row_ptr, const int32_t *col_idx, const int32_t *labels, uint32_t *hist,
                            unsigned long long *intra, unsigned long long *sumsq, int sms, cudaStream_t s,
                            const int32_t *order)
{
    const bool add = evaluate_needs_histogram(n, W, full);
    const auto kernel = full ? (add ? evaluate_kernel<true, true> : evaluate_kernel<true, false>)
                             : (add ? evaluate_kernel<false, true> : evaluate_kernel<false, false>);
    const long long blocks = std::min<long long>((long long)sms * (full ? kFullBlocks : kOrientedBlocks),
                                                 ((long long)n + kBlock / 32 - 1) / (kBlock / 32));
    if (!add) {
        // A histogram block fills one SM's shared memory on `count` of them; the
        // edge count takes the rest of the GPU at the same time.
        // (If it cannot be had, nothing would write sumsq and clear intra.)
        const size_t bytes = n * sizeof(uint32_t);
        cudaError_t e = cudaSuccess;
        if (bytes > kPlainSharedBytes) {
            e = cudaFuncSetAttribute(hist_block_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kHistBlockBytes);
            if (e != cudaSuccess) return e;
        }
        hist_block_kernel<<<count, kHistThreads, bytes, s>>>(n, W, deg_ptr, labels, sumsq, intra);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        cudaLaunchAttribute attr = {};
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3((unsigned)blocks);
        cfg.blockDim = dim3(kBlock);
        cfg.stream = s;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        return cudaLaunchKernelEx(&cfg, kernel, n, W, count, deg_ptr, row_ptr, col_idx, labels,
                                  static_cast<uint32_t *>(nullptr), intra, sumsq, order, true);
    }
    kernel<<<(int)blocks, kBlock, 0, s>>>(n, W, count, deg_ptr, row_ptr, col_idx, labels, hist, intra, sumsq,
                                          order, false);
    return cudaGetLastError();
}

cudaError_t launch_evaluate_multi(const BatchMember *members, const int *starts, int count, int blocks,
                                  cudaStream_t s)
{
    if (blocks > 0) evaluate_multi_kernel<<<blocks, kBlock, 0, s>>>(members, starts, count);
    return cudaGetLastError();
}

cudaError_t launch_evaluate_offspring(int n, int W, int count, const int32_t *eptr, const int32_t *eidx,
                                      const int32_t *labels, uint32_t *hist, unsigned long long *acc,
                                      int grid, cudaStream_t s, const int32_t *order)
{
    evaluate_kernel<false, false><<<grid, kBlock, 0, s>>>(n, W, count, nullptr, eptr, eidx, labels, hist, acc,
                                                        acc + kMaxPop, order, false);
    return cudaGetLastError();
}

}  // namespace mocd

namespace mocd {
cudaError_t check_record_eval(unsigned long long *out, bool reset)
{
    return check_record(out, reset);
}
}  // namespace mocd
