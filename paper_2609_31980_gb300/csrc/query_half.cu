// query_half.cu — the grid scan for grids of half cells (EventHdr::half), the
// automatic grids of five or more dimensions.
//
// Method (Eq. 1, Sec. 1): as in query.cu, every reference in the cells within
// +-1 of the query's cell along each gridded axis is a candidate (complete by
// the grid's roundoff-safe construction, build.cu), its squared distance is
// computed under the fixed float32 contract and it is kept if <= fl(r*r).
//
// What half cells change.  Cells of about r need 3 look-ups per gridded axis
// and query: 81 neighbour rows with five axes, three rounds of the warp's
// lanes, most of them empty.  Storing two cells together along every axis but
// the fastest leaves 2 per axis (a query in a stored cell's low half cannot
// reach the stored cell above, and the other way round): with six axes 32
// neighbour rows, exactly one per lane, whose row offsets and grid-edge tests
// are a few operations on the lane's bits.  A sixth axis becomes affordable
// (22 x 11^5 = 3.5 M stored cells instead of 22^5 = 5.2 M for the 300k x 8
// event), so the candidates do not grow (a CPU model of that event: 10.7 M
// evaluated pairs against 12.6 M, 144 k look-up rounds against 352 k).
//
// Organisation:
//   * a persistent grid; a warp takes `per` (16, fewer for small sets)
//     consecutive cell-sorted query slots at a time from an atomic counter,
//     sorts them by (row of cells, half bits, cell along the fastest axis) and
//     groups runs of equal row and half bits whose cells are equal or adjacent;
//   * lane l looks up neighbour row l of a group (the next group's look-ups in
//     flight), the non-empty slot ranges form one candidate stream over all
//     the groups of the chunk;
//   * each lane takes one candidate per round (its row and original index
//     loaded from L2, the next round's in flight) and computes the contract's
//     squared distance to every query of its group; which range a lane's
//     stream position lies in follows from one load of the next range starts
//     and one warp-wide OR of the positions where ranges start;
//   * accepted (d2, original index) pairs are appended to the query's list in
//     shared memory (kListCap entries), with K > kLongK then to the warp's part
//     of a scratch array in global memory (kMoreCap more); longer lists go to
//     select.cu, which searches again;
//   * rows past the shared-memory list: one at a time by a network across the
//     lanes, two or four keys a lane; compact rows among them go to a pool
//     behind the 32-wide staging rows, so no row is searched twice (calls with
//     K > kLongK);
//   * row sort: lanes q and q + 16 hold half of query q's list each, as 32-bit
//     keys (the distance's bits with the low five cleared, then the entry's
//     place in the list), sort them in registers (an odd-even merge network,
//     every compare-exchange one min and one max) and merge the halves with
//     one exchange between the two lanes: 16 rows at once in a few hundred
//     instructions, where a network across the lanes takes about a hundred a
//     row.  Rows in which two truncated distances agree are put in (d2, index)
//     order by counting;
//   * the sorted rows go back to shared memory and are written with 16-byte
//     stores (row width a multiple of 4 and aligned outputs; else 4-byte).
//
// Grids of few cells (EventHdr::half 0; the build's rule is derive_params in
// build.cu).  Half cells reach 4 cells along an axis, all of one that has no
// more, where plain cells reach 3, and at radii of a fifth of the extent a query
// has thousands of candidates.  Such events get plain cells over four axes (27
// rows, one a lane) or five (walked in three rounds), and wide_stream screens
// the candidates against four queries a step in packed arithmetic.  Uniform
// points in the unit cube, build + query, row tasks or chunks of the axes that
// were the default before / half cells / now: 60k x 8, r = 0.26 1.51 / 3.79 /
// 0.82 ms; 60k x 12, r = 0.3 1.76 / 6.0 / 1.72; 200k x 16, r = 0.22 5.8 / 23.2 /
// 3.0; 20k x 10, r = 0.18 0.110 / 0.143 / 0.079.
//
// What bounds it: instruction issue (71 % of the slots, 80 M warp instructions
// at 300k x 8 where the chunk scan over five axes took 143 M) and the
// load/store pipe (70 %).  Kernel alone, 300k x 8, K = 64: 193 us (chunk scan)
// -> 129 (8 CTAs per SM, 64 registers, 100 B of spills, one shared-memory
// atomic per accepted pair) -> 111 (7 CTAs, 72 registers) -> 105 (places in the
// lists by ballots instead of atomics, whose same-address conflicts were a
// fifth of the load/store pipe, and 32-byte row loads) -> 99 (a single event's
// tasks in a loop of their own).  Build + query, chunk scan or four-axis row
// tasks / now: 300k x 8 242 / 133 us, 500k x 12 523 / 323, 20k x 8 66 / 38.
#include <algorithm>
#include <climits>
#include <type_traits>

#include "frnn_host.h"
#include "warp_sort.cuh"

namespace frnn {
namespace half {

constexpr int kWarps = 4;
constexpr int kListCap = 32;     // accepted entries a query keeps in the kernel
constexpr int kListStr = 36;     // list row stride: 16-byte aligned rows
constexpr int kRangeCap = 128;   // candidate ranges of one batch of groups
constexpr int kQ = kChunkQ;      // queries a warp serves at once, at most
static_assert(kQ == 16, "lanes q and q + 16 share query q's row");
static_assert(kListCap <= kCsrStageW, "a staged compact row holds a whole kernel row");
static_assert(kListCap + kMoreCap <= 128, "four keys a lane sort a long row");

template <int D>
struct Cfg {
    static constexpr int DP = padded_dim(D);
    static constexpr int MINB = DP <= 8 ? 7 : (DP <= 12 ? 5 : 4);
};

struct WarpSmem {
    float* Q;         // [kQ][DP] query coordinates
    float* Ld;        // [kQ][kListStr] squared distances
    int32_t* Li;      // [kQ][kListStr] original indices
    int32_t* rpre;    // [kRangeCap + 4] stream position of each range
    int32_t* rdel;    // [kRangeCap] slot - stream position
    uint16_t* rq;     // [kRangeCap] first and past-the-last query of the range's group
    int32_t* cnt;     // [kQ] accepted entries
    int32_t* qor;     // [kQ] original query index
};

template <int D>
__host__ __device__ constexpr size_t warp_bytes() {
    return ((size_t)kQ * Cfg<D>::DP * 4 + 2 * (size_t)kQ * kListStr * 4 + (size_t)(kRangeCap + 4) * 4 +
            (size_t)kRangeCap * 4 + (size_t)kRangeCap * 2 + 2 * (size_t)kQ * 4 + 127) / 128 * 128;
}

template <int D>
__device__ __forceinline__ WarpSmem carve(unsigned char* base) {
    WarpSmem w;
    w.Q = reinterpret_cast<float*>(base);
    w.Ld = w.Q + kQ * Cfg<D>::DP;
    w.Li = reinterpret_cast<int32_t*>(w.Ld + kQ * kListStr);
    w.rpre = w.Li + kQ * kListStr;
    w.rdel = w.rpre + kRangeCap + 4;
    w.cnt = w.rdel + kRangeCap;
    w.qor = w.cnt + kQ;
    w.rq = reinterpret_cast<uint16_t*>(w.qor + kQ);
    return w;
}

// One point row of DP floats (32-byte rows with one 32-byte load).
template <int DP>
__device__ __forceinline__ void load_row(const float* p, float (&v)[DP]) {
    static_assert(DP % 4 == 0, "rows are 16-byte multiples");
    if constexpr (DP % 8 == 0) {
#pragma unroll
        for (int k = 0; k < DP; k += 8)
            asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                : "=f"(v[k]), "=f"(v[k + 1]), "=f"(v[k + 2]), "=f"(v[k + 3]), "=f"(v[k + 4]), "=f"(v[k + 5]),
                  "=f"(v[k + 6]), "=f"(v[k + 7])
                : "l"(p + k));
    } else {
#pragma unroll
        for (int k = 0; k < DP; k += 4) {
            const float4 x = __ldg(reinterpret_cast<const float4*>(p + k));
            v[k] = x.x;
            v[k + 1] = x.y;
            v[k + 2] = x.z;
            v[k + 3] = x.w;
        }
    }
}

__device__ __forceinline__ int chunk_event(const EventHdr* qev, int E, int c) {
    int lo = 0, hi = E - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (qev[mid].qchunk0 <= c) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Sort every query's list (n entries of query lane % 16 on its two lanes, at
// most 2 P; warp-wide call) in place by (d2, original index); the places from
// n to 2 P get the padding.
template <int P>
__device__ __forceinline__ void sort_rows(const WarpSmem& w, int n) {
    const int lane = threadIdx.x & 31;
    const int q = lane & 15, hh = lane >> 4;
    float* ld = w.Ld + q * kListStr;
    int32_t* li = w.Li + q * kListStr;
    uint32_t k[P];
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const int e = hh * P + i;
        // empty places: above every distance, 32 apart
        const uint32_t v = __float_as_uint(ld[e]);
        k[i] = e < n ? (v & ~31u) | (uint32_t)e : 0x80000000u | (uint32_t)(e * 33);
    }
    const bool near = sort_pair<P>(k);
    const unsigned tied = __ballot_sync(kFull, near);
    // entries to their places
    {
        float v[P];
#pragma unroll
        for (int i = 0; i < P; ++i) v[i] = ld[k[i] & 31];
        __syncwarp();
#pragma unroll
        for (int i = 0; i < P; i += 4) {
            const int e = hh * P + i;
            *reinterpret_cast<float4*>(ld + e) =
                make_float4(e < n ? v[i] : INFINITY, e + 1 < n ? v[i + 1] : INFINITY,
                            e + 2 < n ? v[i + 2] : INFINITY, e + 3 < n ? v[i + 3] : INFINITY);
        }
    }
    {
        int32_t v[P];
#pragma unroll
        for (int i = 0; i < P; ++i) v[i] = li[k[i] & 31];
        __syncwarp();
#pragma unroll
        for (int i = 0; i < P; i += 4) {
            const int e = hh * P + i;
            *reinterpret_cast<int4*>(li + e) = make_int4(e < n ? v[i] : -1, e + 1 < n ? v[i + 1] : -1,
                                                         e + 2 < n ? v[i + 2] : -1, e + 3 < n ? v[i + 3] : -1);
        }
    }
    __syncwarp();
    // rows with ties among the truncated distances: each entry's place is the
    // number of smaller (d2, index) keys
    unsigned rows = (tied | (tied >> 16)) & 0xffffu;
    while (rows) {
        const int r = __ffs(rows) - 1;
        rows &= rows - 1u;
        const int nr = __shfl_sync(kFull, n, r);
        const float d = lane < nr ? w.Ld[r * kListStr + lane] : 0.f;
        const int32_t x = lane < nr ? w.Li[r * kListStr + lane] : 0;
        int rank = 0;
        for (int j = 0; j < nr; ++j) {
            const float dj = __shfl_sync(kFull, d, j);
            const int32_t xj = __shfl_sync(kFull, x, j);
            rank += (dj < d || (dj == d && xj < x)) ? 1 : 0;
        }
        __syncwarp();
        if (lane < nr) {
            w.Ld[r * kListStr + rank] = d;
            w.Li[r * kListStr + rank] = x;
        }
    }
    __syncwarp();
}

// Sort and write one row of more than kListCap entries (n of them: the list,
// then the query's part of the scratch) with the whole warp, 32 P >= n keys.
// width: entries written, those from n on padding.  Not inlined: the scan's
// registers and instruction cache are for the rows that fit the lists.
template <int P>
__device__ __noinline__ void write_long_row(const float* ld, const int32_t* li, const uint64_t* scr, int n,
                                            int width, int32_t* irow, float* drow) {
    const int lane = threadIdx.x & 31;
    uint64_t k[P];
    k[0] = make_key(ld[lane], li[lane]);
#pragma unroll
    for (int p = 1; p < P; ++p)
        k[p] = 32 * p + lane < n ? __ldcg(scr + 32 * (p - 1) + lane) : ~0ull;
    warp_sort<P>(k);
    const bool vec = (width & 3) == 0 &&
                     ((reinterpret_cast<uintptr_t>(irow) | reinterpret_cast<uintptr_t>(drow)) & 15) == 0;
    const int e0 = lane * P;
    int32_t vi[P];
    float vd[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        vi[p] = e0 + p < n ? (int32_t)(uint32_t)k[p] : -1;
        vd[p] = e0 + p < n ? __uint_as_float((uint32_t)(k[p] >> 32)) : INFINITY;
    }
    if (vec && P == 4) {
        if (e0 < width) {
            *reinterpret_cast<int4*>(irow + e0) = make_int4(vi[0], vi[1], vi[P - 2], vi[P - 1]);
            *reinterpret_cast<float4*>(drow + e0) = make_float4(vd[0], vd[1], vd[P - 2], vd[P - 1]);
        }
    } else if (vec) {
        if (e0 < width) {
            *reinterpret_cast<int2*>(irow + e0) = make_int2(vi[0], vi[1]);
            *reinterpret_cast<float2*>(drow + e0) = make_float2(vd[0], vd[1]);
        }
    } else {
#pragma unroll
        for (int p = 0; p < P; ++p) {
            if (e0 + p < width) {
                irow[e0 + p] = vi[p];
                drow[e0 + p] = vd[p];
            }
        }
    }
    for (int e = 32 * P + lane; e < width; e += 32) {
        irow[e] = -1;
        drow[e] = INFINITY;
    }
}

// Packed float32 pairs (query_rows.cu has the proof of the screen's bound).
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t d;
    asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
    return d;
}
__device__ __forceinline__ uint64_t screen2(uint64_t s, uint64_t q, uint64_t c) {
    uint64_t d, t;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(q), "l"(c));
    asm("fma.rn.f32x2 %0, %1, %1, %2;" : "=l"(t) : "l"(d), "l"(s));
    return t;
}
__device__ __forceinline__ float min2(uint64_t v) {
    float a, b;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
    return fminf(a, b);
}

// The candidates of one batch of groups (U of them in nr ranges) on a grid of
// plain cells: few, full cells, so whole chunks of queries against thousands of
// candidates, of which few are neighbours.  A lane takes one candidate a round;
// a step screens it against four queries, two to a packed instruction, and the
// rest of the dimensions is left out when no lane's partial sum is within the
// bound (sums of squares never decrease).  What passes is computed again by the
// contract.  The queries lie pair-interleaved in w.Q.
template <int D, bool LONG>
__device__ __forceinline__ void wide_stream(const WarpSmem& w, const QueryArgs& a, int nr, int U) {
    constexpr int DP = Cfg<D>::DP;
    // dimensions summed before each vote (the gridded ones come last)
    constexpr int VOTE1 = D <= 5 ? D : (D == 9 || D == 10 ? 6 : 4), VOTE2 = D <= 10 ? D : 8;
    const int lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    const unsigned le_mask = lt_mask | (1u << lane);
    const float r2 = a.r2, rs2 = a.r2_screen;
    int cur = -1;
    auto load_cand = [&](int k0, int& qq, int32_t& orig, float (&cv)[DP]) {
        const int ri = cur + 1 + lane;
        const int d = ri < nr ? w.rpre[ri] - k0 : 32;
        const unsigned starts = __reduce_or_sync(kFull, d < 32 ? 1u << d : 0u);
        const int i = cur + __popc(starts & le_mask);
        cur += __popc(starts);
        qq = 0;
        orig = -1;
#pragma unroll
        for (int k = 0; k < DP; ++k) cv[k] = 0.f;
        const int u = k0 + lane;
        if (u < U) {
            const int slot = u + w.rdel[i];
            qq = w.rq[i];
            orig = __ldg(a.rperm + slot);
            load_row<DP>(a.rpts + (int64_t)slot * DP, cv);
        }
    };
    int qq;
    int32_t orig;
    float cv[DP];
    load_cand(0, qq, orig, cv);
#pragma unroll 1
    for (int k0 = 0; k0 < U; k0 += 32) {
        int qq_n;
        int32_t orig_n;
        float cvn[DP];
        load_cand(k0 + 32, qq_n, orig_n, cvn);   // next round in flight
        const int qa = qq & 255, qb = qq >> 8;
        const int pa = qa >> 1, np = ((qb + 1) >> 1) - pa;   // pairs of queries (the first and last may be half)
        const int mx = __reduce_max_sync(kFull, (unsigned)np);
        const int qq_p = __shfl_up_sync(kFull, qq, 1);
        const unsigned firsts = __ballot_sync(kFull, lane == 0 || qq != qq_p);
        const unsigned g_lo = lt_mask & ~((1u << (31 - __clz(firsts & le_mask))) - 1u);
        const unsigned later = firsts & ~le_mask;
        const unsigned g_hi = ~le_mask & (later ? (later & (0u - later)) - 1u : kFull);
        uint64_t cc[D];
#pragma unroll
        for (int k = 0; k < D; ++k) cc[k] = pack2(cv[k], cv[k]);
#pragma unroll 1
        for (int j = 0; j < mx; j += 2) {
            const float* Q0 = w.Q + (j < np ? pa + j : 0) * 2 * DP;
            const float* Q1 = w.Q + (j + 1 < np ? pa + j + 1 : 0) * 2 * DP;
            uint64_t s0 = 0, s1 = 0;
            auto dims = [&](auto from, auto to) {
#pragma unroll
                for (int k = decltype(from)::value; k < decltype(to)::value; k += 2) {
                    const ulonglong2 x = *reinterpret_cast<const ulonglong2*>(Q0 + 2 * k);
                    const ulonglong2 y = *reinterpret_cast<const ulonglong2*>(Q1 + 2 * k);
                    s0 = screen2(s0, x.x, cc[k]);
                    s1 = screen2(s1, y.x, cc[k]);
                    if (k + 1 < D) {
                        s0 = screen2(s0, x.y, cc[k + 1 < D ? k + 1 : k]);
                        s1 = screen2(s1, y.y, cc[k + 1 < D ? k + 1 : k]);
                    }
                }
            };
            auto near = [&]() {
                return __any_sync(kFull, (j < np && min2(s0) <= rs2) || (j + 1 < np && min2(s1) <= rs2));
            };
            dims(std::integral_constant<int, 0>{}, std::integral_constant<int, VOTE1>{});
            if (!near()) continue;
            if constexpr (VOTE1 < D) {
                dims(std::integral_constant<int, VOTE1>{}, std::integral_constant<int, VOTE2>{});
                if (VOTE2 < D && !near()) continue;
                dims(std::integral_constant<int, VOTE2>{}, std::integral_constant<int, D>{});
            }
            // the step's queries 2 (pa + j) + b, b < 4: bit b if it passes
            unsigned pass = 0;
            {
                float v[4];
                asm("mov.b64 {%0, %1}, %2;" : "=f"(v[0]), "=f"(v[1]) : "l"(s0));
                asm("mov.b64 {%0, %1}, %2;" : "=f"(v[2]), "=f"(v[3]) : "l"(s1));
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const int q = 2 * (pa + j) + b;
                    if (q >= qa && q < qb && v[b] <= rs2) pass |= 1u << b;
                }
            }
            unsigned left = __reduce_or_sync(kFull, pass);
            while (left) {
                const int b = __ffs(left) - 1;
                left &= left - 1u;
                const bool on = (pass >> b) & 1u;
                const int q = on ? 2 * (pa + j) + b : 0;
                const int held = w.cnt[q];
                const float* qp = w.Q + (q >> 1) * 2 * DP + (q & 1);
                float s = 0.f;
#pragma unroll
                for (int k = 0; k < D; ++k) {
                    const float d = __fsub_rn(qp[2 * k], cv[k]);
                    s = __fadd_rn(s, __fmul_rn(d, d));
                }
                const bool acc = on && s <= r2 && !(a.self && orig == w.qor[q]);
                const unsigned am = __ballot_sync(kFull, acc);
                const int p = held + __popc(am & g_lo);
                if (acc && p < kListCap) {
                    w.Ld[q * kListStr + p] = s;
                    w.Li[q * kListStr + p] = orig;
                }
                if (acc && (am & g_hi) == 0) w.cnt[q] = p + 1;
                if (LONG && acc && p >= kListCap && p < a.list_cap)
                    (a.scratch + (size_t)(blockIdx.x * kWarps + (threadIdx.x >> 5)) * kScratchKeys +
                     q * kMoreCap)[p - kListCap] = make_key(s, orig);
                __syncwarp();
            }
        }
        qq = qq_n;
        orig = orig_n;
#pragma unroll
        for (int k = 0; k < DP; ++k) cv[k] = cvn[k];
    }
}

// LONG: rows past the shared-memory lists are kept (scratch, pool) and written
// here; else they go to select.cu.
// WIDE: a grid of plain cells (EventHdr::half 0).  Task t: the queries `part`
// x `per` of chunk c, of event e.
template <int D, bool LONG, bool WIDE>
__device__ __forceinline__ void do_task(const QueryArgs& a, const WarpSmem& w, int e, int c, int part, int per) {
    constexpr int DP = Cfg<D>::DP;
    const int lane = threadIdx.x & 31;
    const unsigned lt_mask = (1u << lane) - 1u;
    const unsigned le_mask = lt_mask | (1u << lane);
    const EventHdr& hq = a.qev[e];
    const EventHdr& h = a.ev[e];
    const float r2 = a.r2;
    const int K = a.K;
    // row width of the output (compact staging rows have no padding) and, for
    // the 16-byte stores, its quarter
    const int width = a.csr ? kCsrStageW : K;
    const int w4 = width >> 2;
    // this warp's part of the scratch (formed where it is used: long rows only)
    auto scratch = [&](int q) {
        return a.scratch + (size_t)(blockIdx.x * kWarps + (threadIdx.x >> 5)) * kScratchKeys + q * kMoreCap;
    };
    int32_t* counts = a.counts ? a.counts : h.counts;
    int32_t* oidx = a.counts ? a.idx : h.idx;
    float* od2 = a.counts ? a.dist2 : h.dist2;
    const int64_t q_end = hq.pt_off + hq.n;
    const int s0 = (int)(hq.pt_off + (int64_t)(c - hq.qchunk0) * kQ) + part * per;
    const int nqc = (int)min((int64_t)per, q_end - (int64_t)s0);
    if (nqc <= 0) return;   // past the event's last query
    const bool act = lane < nqc;
    const int qorig0 = act ? a.qperm[s0 + lane] : 0;
    if (!h.valid) {
        // grid built from non-finite input: empty rows (frnn_sync reports it)
        for (int ql = 0; ql < nqc && !a.csr; ++ql) {
            const int qo = __shfl_sync(kFull, qorig0, ql);
            for (int e2 = lane; e2 < K; e2 += 32) {
                oidx[(int64_t)qo * K + e2] = -1;
                od2[(int64_t)qo * K + e2] = INFINITY;
            }
        }
        if (act) counts[qorig0] = 0;
        if (act && a.degree) a.degree[qorig0] = 0;
        return;
    }
    const int naxes = h.naxes, dims0 = h.dims[0];
    const int32_t* cells = a.cstart + h.cell_off;

    // the chunk's queries by (row of cells, half bits, cell on the row)
    int x, row, src, pk;
    {
        const int key = act ? a.qcell[s0 + lane] : 0;
        const int id = WIDE ? key : key >> kHalfBits;
        row = div_mag(id, h.mag[0]);
        x = id - row * dims0;
        const int prev = __shfl_up_sync(kFull, row, 1);
        const int rr = __popc(__ballot_sync(kFull, act && (lane == 0 || row != prev)) & le_mask);
        uint32_t sk = act ? ((uint32_t)rr << 20) | ((uint32_t)(WIDE ? 0 : key & ((1 << kHalfBits) - 1)) << 15) |
                                ((uint32_t)x << 5) | (uint32_t)lane
                          : 0xffffffffu;
#pragma unroll
        for (int k2 = 2; k2 <= kQ; k2 <<= 1) {
#pragma unroll
            for (int j = k2 >> 1; j > 0; j >>= 1) {
                const uint32_t o = __shfl_xor_sync(kFull, sk, j);
                const bool take_min = ((lane & j) == 0) == ((lane & k2) == 0 || k2 == kQ);
                sk = take_min ? min(sk, o) : max(sk, o);
            }
        }
        src = (int)(sk & 31u);
        pk = (int)(sk >> 5);
        x = pk & 1023;
        row = __shfl_sync(kFull, row, src);
    }
    const int bits = (pk >> 10) & 31;
    const int qs = s0 + src;
    const int qorig = __shfl_sync(kFull, qorig0, src);
    if (act) {
        const float4* q4 = reinterpret_cast<const float4*>(a.qpts + (int64_t)qs * DP);
        float4* dst = reinterpret_cast<float4*>(w.Q + lane * DP);
        if constexpr (!WIDE) {
#pragma unroll
            for (int k4 = 0; k4 < DP / 4; ++k4) dst[k4] = q4[k4];
        }
        w.qor[lane] = qorig;
        w.cnt[lane] = 0;
    }
    if (WIDE && lane < kQ) {   // pair-interleaved; no query: never within the radius
        const float* p = a.qpts + (int64_t)qs * DP;
        float* dst = w.Q + (lane >> 1) * 2 * DP + (lane & 1);
#pragma unroll 1
        for (int k = 0; k < DP; ++k) dst[2 * k] = act ? p[k] : __int_as_float(0x7fc00000);
    }
    // per query: the moves (bits of a neighbour row's number; plain cells:
    // two bits an axis, down and up) that would leave the grid; per lane:
    // the moves its row makes, and the row offset its own bits move by
    int bad = 0, moves = lane & 31, mv[kHdrAxes - 1], back = 0;
    // plain cells: a lane has one of the 27 rows of four axes; a fifth axis is
    // walked group by group, its rows last_rs apart
    const int rounds = WIDE && naxes == 5 ? 3 : 1;
    int last_rs = 0;
    if constexpr (WIDE) {
        int v = row, rs = 1, l = lane;
        moves = 0;
#pragma unroll
        for (int ax = 1; ax < kHdrAxes; ++ax) mv[ax - 1] = 0;
#pragma unroll 1
        for (int ax = 1; ax < naxes; ++ax) {
            const int da = h.dims[ax];
            const int qv = div_mag(v, h.mag[ax]);
            const int ca = v - qv * da;
            v = qv;
            if (ca == 0) bad |= 1 << (2 * ax - 2);
            if (ca == da - 1) bad |= 2 << (2 * ax - 2);
            if (ax < 4) {
                const int d = l % 3 - 1;
                l /= 3;
                if (d != 0) moves |= (d < 0 ? 1 : 2) << (2 * ax - 2);
                back += d * rs;
            } else {
                last_rs = rs;
            }
            rs *= da;
        }
        if (l > 0) moves |= 1 << 8;   // (past the last neighbour row)
        bad |= 1 << 8;
    } else {
        int v = row, rs = 1;
#pragma unroll
        for (int ax = 1; ax < kHdrAxes; ++ax) {
            mv[ax - 1] = 0;
            if (ax < naxes) {
                const int da = h.dims[ax];
                const int qv = div_mag(v, h.mag[ax]);
                const int ca = v - qv * da;
                v = qv;
                if (((bits >> (ax - 1)) & 1) ? ca == da - 1 : ca == 0) bad |= 1 << (ax - 1);
                if ((lane >> (ax - 1)) & 1) mv[ax - 1] = rs;
                rs *= da;
            }
        }
    }
    if constexpr (!WIDE) back = -(mv[0] + mv[1] + mv[2] + mv[3] + mv[4]);
    const bool lane_row = WIDE || lane < (1 << (naxes - 1));
    const int gp = bits | (bad << 5) | (x << 14);
    // groups
    const int ppk = __shfl_up_sync(kFull, pk, 1);
    const bool head = act && (lane == 0 || (pk >> 10) != (ppk >> 10) || x > (ppk & 1023) + 1);
    const unsigned gmask = __ballot_sync(kFull, head);
    const int ng = __popc(gmask) * rounds;

    // slot range of the neighbour row of group g (first query hl, past its
    // last hn) on this lane
    int nlo = 0, nhi = 0;
    unsigned gleft = gmask;   // heads of the groups not fetched yet
    int f_hl = 0, f_hn = 0;   // queries of the fetched group
    int f_round = rounds - 1;
    auto fetch = [&]() {
        if (!WIDE || ++f_round == rounds) {
            f_hl = __ffs(gleft) - 1;
            gleft &= gleft - 1u;
            f_hn = gleft ? __ffs(gleft) - 1 : nqc;
            f_round = 0;
        }
        const int g = __shfl_sync(kFull, gp, f_hl);
        const int grow = __shfl_sync(kFull, row, f_hl);
        const int xl = __shfl_sync(kFull, x, f_hn - 1);
        const int x0 = max((g >> 14) - 1, 0), x1 = min(xl + 1, dims0 - 1) + 1;
        nlo = 0;
        nhi = 0;
        int need = moves, off = back;
        if (WIDE && rounds == 3) {
            need |= f_round == 0 ? 1 << 6 : (f_round == 2 ? 2 << 6 : 0);
            off += (f_round - 1) * last_rs;
        }
        if (lane_row && (need & (g >> 5) & 511) == 0) {
#pragma unroll
            for (int ax = 0; ax < kHdrAxes - 1; ++ax)
                if ((g >> ax) & 1) off += 2 * mv[ax];
            const int base = (grow + off) * dims0;
            nlo = __ldg(cells + base + x0);
            nhi = __ldg(cells + base + x1);
        }
    };
    fetch();
    __syncwarp();

    int gdone = 0;   // groups taken into a batch
    while (gdone < ng) {
        int nr = 0;
        for (;;) {
            const int n = nhi - nlo;
            const unsigned bal = __ballot_sync(kFull, n > 0);
            if (nr + __popc(bal) > kRangeCap) break;   // this group opens the next batch
            if (n > 0) {
                const int pos = nr + __popc(bal & lt_mask);
                w.rdel[pos] = nlo;
                w.rpre[pos] = n;   // a count until the batch's scan
                w.rq[pos] = (uint16_t)(f_hl | (f_hn << 8));
            }
            nr += __popc(bal);
            if (++gdone == ng) break;
            fetch();
        }
        // counts -> stream positions
        __syncwarp();
        int U = 0;
        for (int b0 = 0; b0 < nr; b0 += 32) {
            const int i = b0 + lane;
            const int v = i < nr ? w.rpre[i] : 0;
            int incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(kFull, incl, o);
                if (lane >= o) incl += y;
            }
            if (i < nr) {
                const int start = U + incl - v;
                w.rpre[i] = start;
                w.rdel[i] -= start;
            }
            U += __shfl_sync(kFull, incl, 31);
        }
        __syncwarp();

        if constexpr (WIDE) {
            wide_stream<D, LONG>(w, a, nr, U);
            __syncwarp();
            continue;
        }
        int cur = -1;   // last range that starts before the next round
        auto load_cand = [&](int k0, int& qq, int32_t& orig, float (&cv)[DP]) {
            const int ri = cur + 1 + lane;
            const int d = ri < nr ? w.rpre[ri] - k0 : 32;
            const unsigned starts = __reduce_or_sync(kFull, d < 32 ? 1u << d : 0u);
            const int i = cur + __popc(starts & le_mask);
            cur += __popc(starts);
            qq = 0;
            orig = -1;
#pragma unroll
            for (int k = 0; k < DP; ++k) cv[k] = 0.f;
            const int u = k0 + lane;
            if (u < U) {
                const int slot = u + w.rdel[i];
                qq = w.rq[i];
                orig = __ldg(a.rperm + slot);
                load_row<DP>(a.rpts + (int64_t)slot * DP, cv);
            }
        };
        int qq;
        int32_t orig;
        float cv[DP];
        load_cand(0, qq, orig, cv);
#pragma unroll 1
        for (int k0 = 0; k0 < U; k0 += 32) {
            int qq_n;
            int32_t orig_n;
            float cvn[DP];
            load_cand(k0 + 32, qq_n, orig_n, cvn);   // next round in flight
            const int qa = qq & 255;
            const int nq = (qq >> 8) - qa;
            const int mx = __reduce_max_sync(kFull, (unsigned)nq);
            // the lanes of this lane's group before and after it (a group's
            // lanes are consecutive)
            const int qq_p = __shfl_up_sync(kFull, qq, 1);
            const unsigned firsts = __ballot_sync(kFull, lane == 0 || qq != qq_p);
            const unsigned g_lo = lt_mask & ~((1u << (31 - __clz(firsts & le_mask))) - 1u);
            const unsigned later = firsts & ~le_mask;
            const unsigned g_hi = ~le_mask & (later ? (later & (0u - later)) - 1u : kFull);
            for (int j = 0; j < mx; ++j) {
                const bool on = j < nq;
                const int q = on ? qa + j : 0;
                const float4* qp = reinterpret_cast<const float4*>(w.Q + q * DP);
                const int held = w.cnt[q];
                float s = 0.f;
#pragma unroll
                for (int k4 = 0; k4 < DP / 4; ++k4) {
                    const float4 v = qp[k4];
                    const float qv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        if (4 * k4 + k < D) {
                            const float d = __fsub_rn(qv[k], cv[4 * k4 + k]);
                            s = __fadd_rn(s, __fmul_rn(d, d));
                        }
                    }
                }
                bool acc = on && s <= r2;
                if (acc && a.self) acc = orig != w.qor[q];
                // places in the list by counting the group's accepting
                // lanes; the last of them writes the new count (a query
                // belongs to one group, so no other lane does)
                const unsigned am = __ballot_sync(kFull, acc);
                const int p = held + __popc(am & g_lo);
                if (acc && p < kListCap) {
                    w.Ld[q * kListStr + p] = s;
                    w.Li[q * kListStr + p] = orig;
                }
                if (acc && (am & g_hi) == 0) w.cnt[q] = p + 1;
                if constexpr (LONG) {
                    const bool over = acc && p >= kListCap;
                    if (__any_sync(kFull, over)) {
                        if (over && p < a.list_cap) scratch(q)[p - kListCap] = make_key(s, orig);
                    }
                }
                __syncwarp();
            }
            qq = qq_n;
            orig = orig_n;
#pragma unroll
            for (int k = 0; k < DP; ++k) cv[k] = cvn[k];
        }
        __syncwarp();   // the batch's ranges are rewritten by the next batch
    }

    // per query: counts, degree, rows for the selection kernel
    const int kept = act ? w.cnt[lane] : 0;
    bool spill = kept > (LONG ? a.list_cap : kListCap);
    const bool is_long = LONG && kept > kListCap && !spill;
    int64_t pool_at = 0;   // compact output: a long row's place in the pool
    if (LONG && is_long && a.csr) {
        const int need = (min(kept, K) + 3) & ~3;
        pool_at = (int64_t)atomicAdd(a.pool_count, (unsigned long long)need);
        spill = pool_at + need > a.pool_cap;
    }
    if (act && !spill) counts[qorig] = min(kept, K) | (is_long && a.csr ? kCsrPool : 0);
    if (spill && a.csr) counts[qorig] = kCsrSpill;   // counted by the selection kernel
    if (act && !spill && a.degree) a.degree[qorig] = kept;
    if (spill) {
        const int pos = atomicAdd(a.ovf_count, 1);
        if (pos < a.ovf_cap) {
            a.ovf[pos].qslot = qs;
            a.ovf[pos].ev = e;
        } else {
            atomicOr(a.status, kStatusCapacity);
        }
    }
    // rows longer than the lists, one by one (before the lists are sorted)
    unsigned long_rows = LONG ? __ballot_sync(kFull, is_long && !spill) : 0u;
    while (long_rows) {
        const int q = __ffs(long_rows) - 1;
        long_rows &= long_rows - 1u;
        const int nl = __shfl_sync(kFull, kept, q);
        const int64_t row = __shfl_sync(kFull, qorig, q);
        const int64_t pool = a.pool0 + __shfl_sync(kFull, pool_at, q);
        const int64_t at = a.csr ? pool : row * K;
        const int wide = a.csr ? (min(nl, K) + 3) & ~3 : K;
        const float* ld = w.Ld + q * kListStr;
        const int32_t* li = w.Li + q * kListStr;
        if (nl <= 64) write_long_row<2>(ld, li, scratch(q), nl, wide, oidx + at, od2 + at);
        else write_long_row<4>(ld, li, scratch(q), nl, wide, oidx + at, od2 + at);
        if (a.csr && lane == 0) *reinterpret_cast<int64_t*>(oidx + row * kCsrStageW) = pool;
    }
    const unsigned rows = __ballot_sync(kFull, act && kept <= kListCap);   // the other rows written here
    const int n = __shfl_sync(kFull, kept > kListCap ? 0 : kept, lane & 15);
    const int most = __reduce_max_sync(kFull, (unsigned)n);
    int sorted = 32;   // places of the lists that hold the row or its padding
    if (most <= 8) {
        sort_rows<4>(w, n);
        sorted = 8;
    } else if (most <= 16) {
        sort_rows<8>(w, n);
        sorted = 16;
    } else {
        sort_rows<16>(w, n);
    }
    const bool vec = (width & 3) == 0 &&
                     ((reinterpret_cast<uintptr_t>(oidx) | reinterpret_cast<uintptr_t>(od2)) & 15) == 0;
    if (vec) {
        // quarter p of a row: its indices for p < w4, then its distances
        for (int p0 = 0; p0 < 2 * w4; p0 += 32) {
            const int p = p0 + lane;
            const bool dist = p >= w4;
            const int e0 = 4 * (dist ? p - w4 : p);
            const bool lane_on = p < 2 * w4;
            const bool listed = lane_on && e0 < sorted;   // else padding
            const int pad = dist ? 0x7f800000 : -1;
            const int32_t* src4 = (dist ? reinterpret_cast<const int32_t*>(w.Ld) : w.Li) + e0;
            int32_t* dst = (dist ? reinterpret_cast<int32_t*>(od2) : oidx) + e0;
            unsigned left = rows;
            while (left) {
                const int q = __ffs(left) - 1;
                left &= left - 1u;
                int4 v = make_int4(pad, pad, pad, pad);
                if (listed) v = *reinterpret_cast<const int4*>(src4 + q * kListStr);
                if (lane_on && (!a.csr || e0 < w.cnt[q]))
                    *reinterpret_cast<int4*>(dst + (int64_t)w.qor[q] * width) = v;
            }
        }
    } else {
        unsigned left = rows;
        while (left) {
            const int q = __ffs(left) - 1;
            left &= left - 1u;
            const int64_t at = (int64_t)w.qor[q] * width;
            const int stop = a.csr ? min(w.cnt[q], width) : width;
            for (int e2 = lane; e2 < stop; e2 += 32) {
                oidx[at + e2] = e2 < sorted ? w.Li[q * kListStr + e2] : -1;
                od2[at + e2] = e2 < sorted ? w.Ld[q * kListStr + e2] : INFINITY;
            }
        }
    }
    __syncwarp();
}

// Not inlined: the scan of the half cells keeps its registers and instruction
// cache to itself.
template <int D, bool LONG>
__device__ __noinline__ void wide_task(const QueryArgs& a, int e, int c, int part, int per) {
    extern __shared__ __align__(128) unsigned char smem[];
    const WarpSmem w = carve<D>(smem + (size_t)(threadIdx.x >> 5) * warp_bytes<D>());
    do_task<D, LONG, true>(a, w, e, c, part, per);
}

template <int D, bool LONG>
__global__ void __launch_bounds__(kWarps * 32, Cfg<D>::MINB)
    k_half_query(const __grid_constant__ QueryArgs a, int sub_shift) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(128) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const WarpSmem w = carve<D>(smem + (size_t)(threadIdx.x >> 5) * warp_bytes<D>());
    const int per = kQ >> sub_shift;
    const int ntasks = a.nchunks << sub_shift;
    auto next_task = [&]() {
        int t = 0;
        if (lane == 0) t = atomicAdd(a.task_counter, 1);
        return __shfl_sync(kFull, t, 0);
    };
    if (!LONG && a.nev == 1 && a.ev[0].half && (a.path_filter < 0 || a.ev[0].path == a.path_filter)) {
        // one event: no other kind of task in the loop (300k x 8 138 -> 132 us,
        // build included, 500k x 12 335 -> 323; long rows gain nothing from it)
        for (int t = next_task(); t < ntasks; t = next_task())
            do_task<D, LONG, false>(a, w, 0, t >> sub_shift, t & ((1 << sub_shift) - 1), per);
        return;
    }
    for (int t = next_task(); t < ntasks; t = next_task()) {
        const int c = t >> sub_shift, part = t & ((1 << sub_shift) - 1);
        const int e = a.nev > 1 ? chunk_event(a.qev, a.nev, c) : 0;
        if (a.path_filter >= 0 && a.ev[e].path != a.path_filter) continue;   // another launch's event
        if (a.ev[e].half) do_task<D, LONG, false>(a, w, e, c, part, per);
        else wide_task<D, LONG>(a, e, c, part, per);
    }
}

template <int D, bool LONG>
cudaError_t launch_l(const QueryArgs& a, int num_sms, cudaStream_t st) {
    auto kern = &k_half_query<D, LONG>;
    const size_t smem = (size_t)kWarps * warp_bytes<D>();
    cudaError_t ce = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (ce != cudaSuccess) return ce;
    int per_sm = 0;
    ce = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kWarps * 32, smem);
    if (ce != cudaSuccess) return ce;
    const int64_t blocks = (int64_t)num_sms * std::min(std::max(per_sm, 1), 28 / kWarps);   // the scratch's warps
    // sets too small to give every resident warp a chunk of 16 queries are cut
    // into chunks of 8 or 4 (a warp's chunk is a serial chain)
    int sub = 0;
    while (sub < 2 && ((int64_t)a.nchunks << sub) < blocks * kWarps) ++sub;
    const int64_t need = ceil_div((int64_t)a.nchunks << sub, kWarps);
    launch_pdl(kern, dim3((unsigned)std::min(blocks, std::max<int64_t>(need, 1))), dim3(kWarps * 32), smem, st,
               a, sub);
    return cudaGetLastError();
}

// Keeping long rows costs the scan's inner loop a vote per step (300k x 8 147
// -> 151 us, 500k x 12 346 -> 361, build + query, none of whose rows are long)
// and saves searching them again (271,663 x 12, compact, K = 1000, two rows in
// three long: 758 -> 430).  Calls that keep more than 128 neighbours expect
// such rows; the others leave the few they meet to the selection kernel.
template <int D>
cudaError_t launch(const QueryArgs& a, int num_sms, cudaStream_t st) {
    return a.K > kLongK && a.list_cap > kListCap ? launch_l<D, true>(a, num_sms, st)
                                                 : launch_l<D, false>(a, num_sms, st);
}

}  // namespace half

cudaError_t enqueue_half_query(const QueryArgs& a, int num_sms, cudaStream_t st) {
    if (a.nchunks <= 0) return cudaSuccess;
    switch (a.D) {
#define FRNN_CASE(d) case d: return half::launch<d>(a, num_sms, st);
        FRNN_CASE(5) FRNN_CASE(6) FRNN_CASE(7) FRNN_CASE(8) FRNN_CASE(9) FRNN_CASE(10)
        FRNN_CASE(11) FRNN_CASE(12) FRNN_CASE(13) FRNN_CASE(14) FRNN_CASE(15) FRNN_CASE(16)
#undef FRNN_CASE
    }
    return cudaErrorInvalidValue;
}

}  // namespace frnn
