// k_select.cu -- the NSGA-II bookkeeping of Alg. 1 on one thread block:
// FastNonDominatedSort, CrowdingDistanceAssignment, SortByRankAndDistance,
// TournamentSelection(P, E_S, k = 2) and EnvironmentalSelection(P u Q, N_p),
// plus Pareto-front extraction with SelectSolution (Alg. 3) and the layout
// conversions used by the host API.
//
// All ranking works on the exact integer keys (k1 = m - intra, k2 = S), so
// dominance (Sec. 2.2) is exact. Crowding distance follows Deb et al. 2002 on
// the integer keys: per front and objective, members ordered by (key,
// position); both ends +inf; an interior member adds
// (double)(k[next] - k[prev]) / (double)(k_max - k_min), objective 1 first,
// then objective 2; a zero range adds nothing; fronts of one or two members
// are all +inf. This file is built with -fmad=false; each floating-point
// operation is one correctly rounded IEEE operation.
#include <limits.h>
#include <math.h>

#include <algorithm>

#include "mocd_internal.h"
#include "philox.cuh"
#include "ratio.cuh"

namespace mocd {

namespace {

constexpr int kMaxPoints = 2 * kMaxPop;     // members of R = P u Q
constexpr int kSelThreads = 1024;
constexpr int kOwn = 4;                                      // points a thread counts for
constexpr int kSubR = kSelThreads * kOwn / kMaxPoints;       // threads that share them: R
constexpr int kSubP = kSelThreads * kOwn / kMaxPop;          // and P
constexpr unsigned kFull = 0xffffffffu;
constexpr unsigned long long kInfBits = 0x7ff0000000000000ull;  // +inf

// How the step is laid out. One population is at most 256 points, so what
// costs is not work but the length of the dependent chain: a bitonic sort of
// 256 keys is 36 dependent exchanges, 11 of them through a barrier. Every
// order here is found by counting instead: a thread holds four points, reads
// a sixteenth of the others' keys (broadcast reads, bound by the 128 bytes a
// cycle of shared memory, hence four points per read) and counts the smaller
// ones by the borrows of multi-word subtractions; the sum over the threads
// that share the points is their place. Only the peeling of the fronts is
// sequential; one warp does it, eight points a lane, with no barrier inside,
// and stops once the fronts found hold the next population. Bound by the
// half-rate integer pipe in the counting passes and by latency elsewhere:
// 13.0-13.5 us a selection at N_p = 100 (R of 200 points), against 18.2-19.9
// us for four unrolled bitonic sorts with block-wide scans.
struct SelShared {
    uint4 key[kMaxPoints];             // by point: k1, low and high word of k2
    float4 keyf[kMaxPoints];           // m < 2^23: k1, high and low 24 bits of k2 (exact)
    float ck[kMaxPoints];              // by point: rank of k1 << 16 | rank of k2 << 8 | point (exact)
    uint4 row[kMaxPoints];             // by place: tie index, inverted crowding distance (low, high), front
    int q[kMaxPoints];                 // by point: rank of k2 << 8 | rank of k1 (equal iff the keys are)
    int rank[kMaxPoints];              // by point: front, 1-based
    int gs[kMaxPoints];                // by point: place of the first point with the same keys
    int cid[kMaxPoints];               // point at each place of the (rank, k1, k2, index) order
    int tie[kMaxPoints];               // its index in the ordered set (R index or P position)
    __align__(16) unsigned short sq[kMaxPoints];  // by place in (k1, k2, index) order: q
    __align__(8) unsigned char sid[kMaxPoints];   // and the point
    unsigned heads[kMaxPoints / 32];   // places that start a group of identical keys
    int fstart[kMaxPoints + 2];        // first place of each front; one past the last front: the places taken
    int placed;                        // places taken (the fronts that hold the next population)
    int order[kMaxPoints];             // (rank, crowding desc, index) order
    int keep[kMaxPop];
    float pkey[kMaxPop];               // by P position: gs << 8 | position (exact)
    unsigned char minpos[kMaxPop * kMaxParents];  // tournament winners: places of P's order
    unsigned char skip[kMaxPop];       // parent copied when crossover is skipped, else 255
};

// c -= 1 if x < y (one, two or four words, least significant first): the
// borrow of x - y.
__device__ __forceinline__ void count_below(unsigned &c, unsigned x, unsigned y)
{
    asm("{\n\t.reg .u32 t;\n\tsub.cc.u32 t, %1, %2;\n\tsubc.u32 %0, %0, 0;\n\t}" : "+r"(c) : "r"(x), "r"(y));
}
__device__ __forceinline__ void count_below(unsigned &c, unsigned x0, unsigned x1, unsigned y0, unsigned y1)
{
    asm("{\n\t.reg .u32 t;\n\tsub.cc.u32 t, %1, %3;\n\tsubc.cc.u32 t, %2, %4;\n\tsubc.u32 %0, %0, 0;\n\t}"
        : "+r"(c)
        : "r"(x0), "r"(x1), "r"(y0), "r"(y1));
}
__device__ __forceinline__ void count_below(unsigned &c, const uint4 &x, const uint4 &y)
{
    asm("{\n\t.reg .u32 t;\n\t"
        "sub.cc.u32 t, %1, %5;\n\t"
        "subc.cc.u32 t, %2, %6;\n\t"
        "subc.cc.u32 t, %3, %7;\n\t"
        "subc.cc.u32 t, %4, %8;\n\t"
        "subc.u32 %0, %0, 0;\n\t}"
        : "+r"(c)
        : "r"(x.x), "r"(x.y), "r"(x.z), "r"(x.w), "r"(y.x), "r"(y.y), "r"(y.z), "r"(y.w));
}

// c += 1 if x < y, for integers of at most 24 bits held in floats: the
// difference is exact and saturates to 0 or 1. This and the next run in the FMA
// pipe, at twice the rate of the integer pipe's subtractions.
__device__ __forceinline__ void count_below(float &c, float x, float y)
{
    c = __fadd_rn(c, __saturatef(__fsub_rn(y, x)));
}
// The same for (xh, xl) < (yh, yl), integers of at most 24 bits each: a
// difference of the high parts outweighs any of the low parts, and the fused
// multiply-add keeps the sign and a magnitude of at least 1.
__device__ __forceinline__ void count_below(float &c, float xh, float xl, float yh, float yl)
{
    c = __fadd_rn(c, __saturatef(__fmaf_rn(__fsub_rn(yh, xh), 33554432.0f, __fsub_rn(yl, xl))));
}

// The four (negative) counts of a thread summed over the SUBS lanes that
// share its points; lane sub returns the count of point sub % 4. Counts stay
// below 2^16, so two travel in one word.
template <int SUBS>
__device__ __forceinline__ int sum_shared(const unsigned (&c)[kOwn], int sub)
{
    unsigned a = (0u - c[0]) | ((0u - c[1]) << 16), b = (0u - c[2]) | ((0u - c[3]) << 16);
#pragma unroll
    for (int d = 1; d < SUBS; d <<= 1) {
        a += __shfl_xor_sync(kFull, a, d);
        b += __shfl_xor_sync(kFull, b, d);
    }
    const unsigned w = (sub & 2) ? b : a;
    return (int)((sub & 1) ? w >> 16 : w & 0xffffu);
}

template <int SUBS>
__device__ __forceinline__ int sum_shared(const float (&c)[kOwn], int sub)
{
    unsigned w[kOwn];
#pragma unroll
    for (int k = 0; k < kOwn; ++k) w[k] = 0u - (unsigned)c[k];
    return sum_shared<SUBS>(w, sub);
}

// The place of each of n distinct keys below 2^24, held in floats: lane sub <
// 4 of a group returns that of its group's point sub.
template <int SUBS>
__device__ __forceinline__ int place_of(const float *keys, int n)
{
    const int i0 = threadIdx.x / SUBS * kOwn, sub = threadIdx.x % SUBS;
    float mine[kOwn], c[kOwn] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int k = 0; k < kOwn; ++k) mine[k] = keys[i0 + k];
    if (i0 < n) {
#pragma unroll 2
        for (int j = sub; j < n; j += SUBS) {
            const float x = keys[j];
#pragma unroll
            for (int k = 0; k < kOwn; ++k) count_below(c[k], x, mine[k]);
        }
    }
    return sum_shared<SUBS>(c, sub);
}

// Fronts of the N points of S.key, first to last, until they hold `want`
// points: q, rank, fstart and the places cid of the fronts-contiguous
// (rank, k1, k2, index) order of those points. small: S.keyf is set (k1 below
// 2^24, k2 below 2^48).
__device__ void rank_points(SelShared &S, int N, int want, bool small)
{
    const int i0 = threadIdx.x / kSubR * kOwn, sub = threadIdx.x % kSubR;
    const int i = i0 + sub;  // the point whose sums this lane takes (sub < 4)
    {
        // Ranks of k1 and of k2 among the points.
        int r1, r2;
        if (small) {
            float4 mine[kOwn];
            float c1[kOwn] = {0.0f, 0.0f, 0.0f, 0.0f}, c2[kOwn] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int k = 0; k < kOwn; ++k) mine[k] = S.keyf[i0 + k];
            if (i0 < N) {
                for (int j = sub; j < N; j += kSubR) {
                    const float4 x = S.keyf[j];
#pragma unroll
                    for (int k = 0; k < kOwn; ++k) {
                        count_below(c1[k], x.x, mine[k].x);
                        count_below(c2[k], x.y, x.z, mine[k].y, mine[k].z);
                    }
                }
            }
            r1 = sum_shared<kSubR>(c1, sub);
            r2 = sum_shared<kSubR>(c2, sub);
        } else {
            uint4 mine[kOwn];
            unsigned c1[kOwn] = {0, 0, 0, 0}, c2[kOwn] = {0, 0, 0, 0};
#pragma unroll
            for (int k = 0; k < kOwn; ++k) mine[k] = S.key[i0 + k];
            if (i0 < N) {
                for (int j = sub; j < N; j += kSubR) {
                    const uint4 x = S.key[j];
#pragma unroll
                    for (int k = 0; k < kOwn; ++k) {
                        count_below(c1[k], x.x, mine[k].x);
                        count_below(c2[k], x.y, x.z, mine[k].y, mine[k].z);
                    }
                }
            }
            r1 = sum_shared<kSubR>(c1, sub);
            r2 = sum_shared<kSubR>(c2, sub);
        }
        if (sub < kOwn && i < N) {
            S.q[i] = (r2 << 8) | r1;
            S.ck[i] = (float)((r1 << 16) | (r2 << 8) | i);
        }
    }
    __syncthreads();
    {
        const int at = place_of<kSubR>(S.ck, N);  // in (k1, k2, index) order
        if (sub < kOwn && i < N) {
            S.sq[at] = (unsigned short)S.q[i];
            S.sid[at] = (unsigned char)i;
        }
    }
    __syncthreads();
    // A remaining point is dominated iff some remaining point at an earlier
    // place has smaller (k2, k1), i.e. smaller q: its k1 is not larger, its
    // k2 not larger, and the two differ (identical points share q). Each
    // front's members take the next places in this order; the scan of a
    // front's member counts runs beside the next front's scan of minima.
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        const uint4 qw = reinterpret_cast<const uint4 *>(S.sq)[lane];
        const uint2 iw = reinterpret_cast<const uint2 *>(S.sid)[lane];
        const unsigned qs[4] = {qw.x, qw.y, qw.z, qw.w};
        const unsigned is[2] = {iw.x, iw.y};
        int qk[8], place[8], front[8];  // qk: INT_MAX once the point is taken
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            qk[k] = 8 * lane + k < N ? (int)((qs[k >> 1] >> (16 * (k & 1))) & 0xffffu) : INT_MAX;
            place[k] = -1;
            front[k] = 0;
        }
        int placed = 0;     // places of the fronts before the previous one
        unsigned prev = 0;  // members of the previous front
        int r = 1;
        for (;; ++r) {
            int low = min(min(min(qk[0], qk[1]), min(qk[2], qk[3])), min(min(qk[4], qk[5]), min(qk[6], qk[7])));
            int run = __shfl_up_sync(kFull, low, 1);  // smallest remaining q of the earlier lanes
            if (lane == 0) run = INT_MAX;
            const int c = __popc(prev);
            int incl = c;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const int y = __shfl_up_sync(kFull, run, d);
                const int z = __shfl_up_sync(kFull, incl, d);
                if (lane >= d) {
                    run = min(run, y);
                    incl += z;
                }
            }
            int at = placed + incl - c;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const bool in = (prev >> k) & 1u;
                place[k] = in ? at : place[k];
                front[k] = in ? r - 1 : front[k];
                at += in ? 1 : 0;
            }
            placed += __shfl_sync(kFull, incl, 31);
            if (lane == 0) S.fstart[r] = placed;
            if (placed >= want) break;
            prev = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int x = qk[k];
                const bool in = x != INT_MAX && run >= x;
                prev |= (in ? 1u : 0u) << k;
                qk[k] = in ? INT_MAX : x;
                run = min(run, x);
            }
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            if (place[k] < 0) continue;
            const int id = (int)((is[k >> 2] >> (8 * (k & 3))) & 0xffu);
            S.cid[place[k]] = id;
            S.tie[place[k]] = id;
            S.rank[id] = front[k];
        }
        if (lane == 0) S.placed = placed;
    }
    __syncthreads();
}

// Crowding distance of the N points at places 0 .. N - 1 (fronts truncated to
// N places), written with each place's tie index and front into S.row; also
// S.gs of every point. Two threads share a place, one objective each.
__device__ __noinline__ void crowd_places(SelShared &S, int N)
{
    const int t = threadIdx.x >> 1, obj = threadIdx.x & 1;
    const bool has = t < N;
    int id = 0, fs = 0, fe = 1, front = 0;
    if (has) {
        id = S.cid[t];
        front = S.rank[id];
        fs = S.fstart[front];
        fe = min(S.fstart[front + 1], N);
    }
    // A ballot covers 16 places (a place's two threads vote alike).
    const bool head = has && (t == fs || S.q[S.cid[t - 1]] != S.q[id]);
    const unsigned bal = __ballot_sync(kFull, head);
    if ((threadIdx.x & 31) == 0 && threadIdx.x < 2 * kMaxPoints) {
        unsigned m = bal & 0x55555555u;  // every other bit, packed
        m = (m | (m >> 1)) & 0x33333333u;
        m = (m | (m >> 2)) & 0x0f0f0f0fu;
        m = (m | (m >> 4)) & 0x00ff00ffu;
        m = (m | (m >> 8)) & 0x0000ffffu;
        reinterpret_cast<unsigned short *>(S.heads)[threadIdx.x >> 5] = (unsigned short)m;
    }
    __syncthreads();
    if (threadIdx.x < 2 * ((N + 15) & ~15)) {  // (whole warps)
        int gs = 0, ge = fe;                   // t's group, [gs, ge)
        if (has) {
            int w = t >> 5;
            unsigned m = S.heads[w] & (0xffffffffu >> (31 - (t & 31)));
            while (!m) m = S.heads[--w];  // (place fs <= t starts a group)
            gs = 32 * w + 31 - __clz((int)m);
            w = t >> 5;
            m = S.heads[w] & (0xfffffffeu << (t & 31));
            while (!m && ++w < kMaxPoints / 32) m = S.heads[w];
            if (m) ge = min(ge, 32 * w + __ffs((int)m) - 1);
        }
        // The places whose keys are subtracted: neighbours of the place in
        // its objective's order, and the two ends of the front. Objective 2
        // takes the groups in reverse order, index order inside a group.
        const int F = fe - fs;
        const int pos = obj == 0 ? t - fs : (fe - ge) + (t - gs);
        const bool end = F <= 2 || pos == 0 || pos == F - 1;
        int hi = t, lo = t;
        if (!end) {
            hi = obj == 0 ? t + 1 : (t < ge - 1 ? t : gs - 1);
            lo = obj == 0 ? t - 1 : (t > gs ? t : ge);
        }
        auto value = [&](int place) -> long long {
            const uint4 x = S.key[S.cid[place]];
            return obj == 0 ? (long long)x.x : (long long)(((unsigned long long)x.z << 32) | x.y);
        };
        const int top = obj == 0 ? fe - 1 : fs, bottom = obj == 0 ? fs : fe - 1;
        long long range = 0, gap = 0;
        if (has && !end) {
            range = value(top) - value(bottom);
            gap = value(hi) - value(lo);
        }
        unsigned long long c = end ? kInfBits : 0ull;
        if (range > 0) c = ratio_bits(gap, range);
        // Objective 1 + objective 2 (the partner thread holds the same place).
        const unsigned long long o = __shfl_xor_sync(kFull, c, 1);
        if (has && obj == 0) {
            const unsigned long long sum =
                (unsigned long long)__double_as_longlong(__dadd_rn(__longlong_as_double((long long)c),
                                                                   __longlong_as_double((long long)o)));
            S.row[t] = make_uint4((unsigned)S.tie[t], (unsigned)~sum, (unsigned)(~sum >> 32), (unsigned)front);
            S.gs[id] = gs;
        }
    }
    __syncthreads();
}

// The (rank, crowding desc, index) order of the N points at places 0 .. N - 1:
// S.order[place] = tie index. A point moves only within its front, so a
// thread counts over the fronts of its four points. Crowding distances are
// non-negative or +inf, so their bit patterns order like the values.
template <int SUBS>
__device__ void order_places(SelShared &S, int N)
{
    const int t0 = threadIdx.x / SUBS * kOwn, sub = threadIdx.x % SUBS;
    uint4 mine[kOwn];
    unsigned c[kOwn] = {0, 0, 0, 0};
    int fs = 0;
    if (t0 < N) {
#pragma unroll
        for (int k = 0; k < kOwn; ++k) mine[k] = S.row[min(t0 + k, N - 1)];
        fs = S.fstart[mine[0].w];
        const int fe = min(S.fstart[mine[kOwn - 1].w + 1], N);
        for (int j = fs + sub; j < fe; j += SUBS) {
            const uint4 x = S.row[j];
#pragma unroll
            for (int k = 0; k < kOwn; ++k) count_below(c[k], x, mine[k]);
        }
    }
    const int at = sum_shared<SUBS>(c, sub);
    if (sub < kOwn && t0 + sub < N) S.order[fs + at] = (int)S.row[t0 + sub].x;
    __syncthreads();
}

// One block: selection of one population (mode 0: keys of a fresh P from
// acc, `base` generations run so far; mode 1: R = P u Q), then rank, crowding and order of P and the next
// tournament.
__device__ __forceinline__ void select_body(const GenParams &gp, const PopState &ps, int mode, uint32_t base,
                                            SelShared &S)
{
    const int p = threadIdx.x;
    const int np = gp.np, E = gp.es;
    const long long m = gp.m;
    const uint32_t g = mode == 0 ? base : *ps.gen;
    const uint32_t gn = g + 1u;
    const unsigned long long *acc = ps.acc;
    const int N = mode == 0 ? np : 2 * np;
    const bool small = m < (1ll << 23);  // k1 <= m, k2 <= (2 m)^2

    // TournamentSelection's draws for generation gn = g + 1 do not depend on
    // the keys, and the generation number is the last selection's, which every
    // launch since then followed: they come before the wait for the evaluation
    // (see overlap_next). Parent j of child i is the better of sorted positions a, b,
    // i.e. position min(a, b). A thread takes a Philox block (two parents).
    const int blocks = E / 2 + 1;  // (2 E + 2 words) / 4, rounded up
    for (int t = threadIdx.x; t < np * blocks; t += kSelThreads) {
        const int i = t / blocks, w4 = t % blocks;
        const uint4 u = philox4x32_10(make_uint4((uint32_t)w4, (uint32_t)i, gn, kStageSelect), gp.key0, gp.key1);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = 2 * w4 + h;
            const uint32_t x = h ? u.z : u.x, y = h ? u.w : u.y;
            if (j < E) {
                S.minpos[i * kMaxParents + j] =
                    (unsigned char)min(pick_index(x, (uint32_t)np), pick_index(y, (uint32_t)np));
            } else if (j == E) {
                // Words 2 E (the crossover coin) and 2 E + 1 (the parent copied).
                S.skip[i] = (unsigned long long)x <= gp.thr_c ? 255 : (unsigned char)pick_index(y, (uint32_t)E);
            }
        }
    }
    cudaGridDependencySynchronize();
    // Keys by point: P's (mode 1), then those of the evaluated labellings.
    if (p < N) {
        const int i = mode == 0 ? p : p - np;
        const long long k1 = i < 0 ? ps.pk[p] : m - (long long)acc[i];
        const long long k2 = i < 0 ? ps.pk[kMaxPop + p] : (long long)acc[kMaxPop + i];
        S.key[p] = make_uint4((unsigned)k1, (unsigned)k2, (unsigned)((unsigned long long)k2 >> 32), 0u);
        S.keyf[p] = make_float4((float)(unsigned)k1, (float)(unsigned)((unsigned long long)k2 >> 24),
                                (float)((unsigned)k2 & 0xffffffu), 0.0f);
        if (mode == 1) {
            ps.rk[p] = k1;
            ps.rk[2 * kMaxPop + p] = k2;
        }
    }
    __syncthreads();
    rank_points(S, N, np, small);
    crowd_places(S, S.placed);
    if (mode == 1) {
        order_places<kSubR>(S, S.placed);
        if (p < np) S.keep[p] = S.order[p];
    } else if (p < np) {
        S.keep[p] = p;
    }
    __syncthreads();
    // The kept members keep their fronts: P is R's first fronts plus part of
    // the next one, so every dominator of a member is kept too, and front r
    // of P starts where front r of R does. Members in (rank, k1, k2, P
    // position) order: identical points form one group, in P order inside.
    if (p < np) {
        const int id = S.keep[p];
        const uint4 x = S.key[id];
        ps.pk[p] = (int64_t)x.x;
        ps.pk[kMaxPop + p] = (int64_t)(((unsigned long long)x.z << 32) | x.y);
        ps.keep[p] = id;
        ps.prank[p] = S.rank[id];
        S.pkey[p] = (float)((S.gs[id] << 8) | p);
    }
    __syncthreads();
    {
        const int at = place_of<kSubP>(S.pkey, np);
        const int sub = threadIdx.x % kSubP, i = threadIdx.x / kSubP * kOwn + sub;
        if (sub < kOwn && i < np) {
            S.cid[at] = S.keep[i];
            S.tie[at] = i;
        }
    }
    __syncthreads();
    // Crowding recomputed on P (Alg. 1, start of the generation).
    crowd_places(S, np);
    order_places<kSubP>(S, np);
    for (int t = threadIdx.x; t < np * E; t += kSelThreads) {
        const int i = t / E, j = t % E;
        const int r = S.keep[S.order[S.minpos[i * kMaxParents + j]]];
        ps.par_r[i * kMaxParents + j] = r;
        if (S.skip[i] == j) ps.copy_r[i] = r;
        else if (j == 0 && S.skip[i] == 255) ps.copy_r[i] = -1;
    }
    if (p == 0) *ps.gen = gn;
}

__global__ void __launch_bounds__(kSelThreads)
select_kernel(GenParams gp, PopState ps, int mode, uint32_t base)
{
    __shared__ SelShared S;
    select_body(gp, ps, mode, base, S);
}

// The selections of several populations in one launch (a batch of
// instances): block b selects population b.
__global__ void __launch_bounds__(kSelThreads)
select_multi_kernel(const GenParams *__restrict__ gps, const PopState *__restrict__ pss, int mode)
{
    __shared__ SelShared S;
    const GenParams gp = gps[blockIdx.x];
    const PopState ps = pss[blockIdx.x];
    select_body(gp, ps, mode, 0u, S);
}

// F_1 of P in P order and SelectSolution: argmin of 4 m k1 + k2 (= argmax of
// Q = 1 - f1 - f2), first member on ties. Also each member's exact intra and
// S, and f1 = k1 / m, f2 = S / (4 m^2) as single IEEE divisions.
// One thread per member of P (a block of kMaxPop threads): 4 us at N_p = 100,
// against 75 us for one thread that divided for each member in turn.
__global__ void __launch_bounds__(kMaxPop) front_kernel(GenParams gp, PopState ps)
{
    __shared__ int s_count[kMaxPop / 32];
    __shared__ long long s_key[kMaxPop / 32];
    __shared__ int s_at[kMaxPop / 32];
    const int p = threadIdx.x, lane = p & 31, w = p >> 5;
    const long long m = gp.m;
    const bool in = p < gp.np && ps.prank[p] == 1;
    const unsigned bal = __ballot_sync(kFull, in);
    if (lane == 0) s_count[w] = __popc(bal);
    __syncthreads();
    int at = __popc(bal & ((1u << lane) - 1u)), count = 0;
#pragma unroll
    for (int k = 0; k < kMaxPop / 32; ++k) {
        at += k < w ? s_count[k] : 0;
        count += s_count[k];
    }
    long long K = LLONG_MAX;
    if (in) {
        const long long k1 = ps.pk[p], k2 = ps.pk[kMaxPop + p];
        K = 4ll * m * k1 + k2;
        ps.front[2 + at] = p;
        ps.fint[at] = m - k1;
        ps.fint[kMaxPop + at] = k2;
        ps.fval[at] = __ddiv_rn((double)k1, (double)m);
        ps.fval[kMaxPop + at] = __ddiv_rn((double)k2, (double)(4ll * m * m));
    }
    int best = in ? at : INT_MAX;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) {
        const long long ok = __shfl_xor_sync(kFull, K, d);
        const int ob = __shfl_xor_sync(kFull, best, d);
        if (ok < K || (ok == K && ob < best)) {
            K = ok;
            best = ob;
        }
    }
    if (lane == 0) {
        s_key[w] = K;
        s_at[w] = best;
    }
    __syncthreads();
    if (p != 0) return;
#pragma unroll
    for (int k = 1; k < kMaxPop / 32; ++k)
        if (s_key[k] < K || (s_key[k] == K && s_at[k] < best)) {
            K = s_key[k];
            best = s_at[k];
        }
    ps.front[0] = count;
    ps.front[1] = count ? best : -1;
}

// The layout conversions of the host API go through a shared tile of 32 nodes
// x 32 individuals, so that both sides are read and written in whole rows
// (individual-major: 128 bytes of consecutive nodes; node-major: 128 bytes of
// one node's individuals). A thread per node striding over the individuals
// touched 32 rows per load instead.
constexpr int kTile = 32;
constexpr int kTileThreads = 256;
constexpr int kTileStep = kTileThreads / 32;

// out[k][v] = R_v[idx[k]] for k < count (idx NULL: identity on P).
__global__ void __launch_bounds__(kTileThreads)
gather_individuals_kernel(int n, int W, int np, const int32_t *__restrict__ phalf, const int32_t *__restrict__ q,
                          const int32_t *__restrict__ idx, int count, int32_t *__restrict__ out)
{
    __shared__ int32_t tile[kTile][kTile + 1];
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const int k0 = blockIdx.y * kTile, k = k0 + lane;
    const int r = k < count ? (idx ? idx[k] : k) : 0;
    const int32_t *src = r < np ? phalf + r : q + (r - np);
    for (int v0 = blockIdx.x * kTile; v0 < n; v0 += gridDim.x * kTile) {
#pragma unroll
        for (int j = row; j < kTile; j += kTileStep)
            if (v0 + j < n && k < count) tile[j][lane] = src[(size_t)(v0 + j) * W];
        __syncthreads();
#pragma unroll
        for (int j = row; j < kTile; j += kTileStep)
            if (k0 + j < count && v0 + lane < n) out[(size_t)(k0 + j) * n + v0 + lane] = tile[lane][j];
        __syncthreads();
    }
}

// dst[v][k] = src[k][v] for k < count, zero for count <= k < W. A label
// outside [0, n) sets *bad and becomes 0, so that whatever follows stays in
// bounds (dst NULL: only the check).
__global__ void __launch_bounds__(kTileThreads)
to_node_major_kernel(int n, int W, int count, const int32_t *__restrict__ src, int32_t *__restrict__ dst,
                     int *__restrict__ bad)
{
    __shared__ int32_t tile[kTile][kTile + 1];
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const int k0 = blockIdx.y * kTile;
    bool wrong = false;
    for (int v0 = blockIdx.x * kTile; v0 < n; v0 += gridDim.x * kTile) {
#pragma unroll
        for (int j = row; j < kTile; j += kTileStep) {
            int32_t x = k0 + j < count && v0 + lane < n ? src[(size_t)(k0 + j) * n + v0 + lane] : 0;
            if ((uint32_t)x >= (uint32_t)n) {
                wrong = true;
                x = 0;
            }
            tile[j][lane] = x;
        }
        if (!dst) continue;
        __syncthreads();
#pragma unroll
        for (int j = row; j < kTile; j += kTileStep)
            if (v0 + j < n && k0 + lane < W) dst[(size_t)(v0 + j) * W + k0 + lane] = tile[lane][j];
        __syncthreads();
    }
    if (wrong) *bad = 1;
}

dim3 tiles_for(int n, int width)
{
    return dim3((unsigned)std::min((n + kTile - 1) / kTile, 4096), (unsigned)((width + kTile - 1) / kTile));
}

}  // namespace

cudaError_t launch_select(const GenParams &gp, const PopState &ps, int mode, cudaStream_t s, uint32_t base)
{
    select_kernel<<<1, kSelThreads, 0, s>>>(gp, ps, mode, base);
    return cudaGetLastError();
}

cudaError_t launch_select_multi(const GenParams *gps, const PopState *pss, int count, int mode, cudaStream_t s)
{
    select_multi_kernel<<<count, kSelThreads, 0, s>>>(gps, pss, mode);
    return cudaGetLastError();
}

cudaError_t launch_front(const GenParams &gp, const PopState &ps, cudaStream_t s)
{
    front_kernel<<<1, kMaxPop, 0, s>>>(gp, ps);
    return cudaGetLastError();
}

cudaError_t launch_gather_individuals(int n, int W, int np, const int32_t *phalf, const int32_t *q,
                                      const int32_t *idx, int count, int32_t *out, cudaStream_t s)
{
    if (count <= 0) return cudaSuccess;
    gather_individuals_kernel<<<tiles_for(n, count), kTileThreads, 0, s>>>(n, W, np, phalf, q, idx, count, out);
    return cudaGetLastError();
}

cudaError_t launch_to_node_major(int n, int W, int count, const int32_t *src, int32_t *dst, int *bad, cudaStream_t s)
{
    to_node_major_kernel<<<tiles_for(n, W), kTileThreads, 0, s>>>(n, W, count, src, dst, bad);
    return cudaGetLastError();
}

}  // namespace mocd
