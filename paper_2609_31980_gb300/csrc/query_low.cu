// query_low.cu — the grid scan for the automatic grids of up to four
// dimensions, where every coordinate is gridded.
//
// Method (Eq. 1, Sec. 1): as in query.cu, every reference in the cells within
// +-m of the query's cell along each gridded axis is a candidate (complete by
// the grid's roundoff-safe construction, build.cu), its squared distance is
// computed under the fixed float32 contract and it is kept if <= fl(r*r).
//
// Why one query per lane here.  A point row is 16 bytes, a query has a few
// dozen candidates in 3, 9 or 27 short slot ranges and a handful of
// neighbours, and the queries of a warp (consecutive cell-sorted slots) lie
// side by side in one or two rows of cells, so their ranges overlap and their
// loads hit the same lines.  Putting the candidates of one group of queries on
// the lanes instead (query.cu) left most lanes idle: 2 queries a group, 27
// candidates spread over 9 look-ups.
//
// Organisation:
//   * a persistent grid; a warp takes 32 query slots (two chunks) at a time
//     from an atomic counter; every lane carries its own event's parameters, so
//     a warp may straddle the events of a batch.  Sets too small to fill the
//     chip give each query G = 4 or 8 lanes, which share its neighbour rows,
//     every G-th to a lane (a query's search is a serial chain: 4096 x 4 points,
//     G = 1 53 us, build included);
//   * each lane looks up kRows neighbour rows at a time, all loads in flight,
//     and keeps the non-empty ranges in its column of a shared-memory table;
//     it then walks them back to back, two candidates a step, moving to its
//     next range on its own, so lanes stay busy whatever the ranges' lengths;
//   * an accepted candidate's slot goes to the lane's row of a list in shared
//     memory (at most kListCap; longer lists go to select.cu).  Its distance
//     is computed again, by the same contract, when the row is sorted: the
//     distances' rows then share their memory with the range table, which
//     lets 24 instead of 20 warps reside on an SM;
//   * each lane sorts its own list in registers on 32-bit keys (the distance's
//     bits with the low five cleared, then the place in the list) with an
//     odd-even merge network of the warp's longest list's width, and writes the
//     entries back in order; equal truncated distances are put in (d2, index)
//     order afterwards;
//   * rows are written by the whole warp with 16-byte stores (row width a
//     multiple of 4 and aligned outputs; else 4-byte).
//
// What bounds it: the load/store pipe (70 % of its wavefronts: 32 lanes' rows
// lie on about ten lines) and instruction issue (63 %), at 1 M x 3 with 4
// neighbours each.  Kernel alone 429 -> 136 us there, 222 -> 115 at 300,000 x 4
// with 9 neighbours.  Build + query: 1 M x 3 498 -> 219 us, 300,000 x 4 255 ->
// 152, 4096 x 3 38.7 -> 30.  More resident warps (shorter lists, 28 warps) lost
// to the spills of the wider sorts.
#include <algorithm>

#include "frnn_host.h"

namespace frnn {
namespace low {

constexpr int kWarps = 4;
constexpr uint32_t kFull = 0xffffffffu;
constexpr int kListCap = 32;    // accepted entries a query keeps in the kernel
constexpr int kListStr = 33;    // list row stride: lanes at equal places hit distinct banks
constexpr int kRows = 9;        // neighbour rows looked up at once
constexpr int kMinBlocks = 6;   // CTAs per SM (shared memory)
static_assert(kListCap <= kCsrStageW, "a staged compact row holds a whole kernel row");

struct WarpSmem {
    int32_t* Li;    // [32][kListStr] slots, then original indices
    float* Ld;      // [32][kListStr] squared distances (once the search is done)
    int2* rng;      // [kRows][32] slot ranges (before)
    int32_t* cnt;   // [32] list lengths (G > 1)
};
constexpr size_t kWarpBytes = 2 * 32 * kListStr * 4 + 32 * 4;
static_assert(kRows * 32 * 8 <= 32 * kListStr * 4, "the ranges fit the distances' rows");
static_assert(kWarpBytes % 16 == 0, "aligned warp areas");

// Two point rows of 4 floats, the first at an even slot.
__device__ __forceinline__ void load_pair(const float4* p, float (&v)[8]) {
    asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
        : "l"(p));
}

__device__ __forceinline__ int chunk_event(const EventHdr* qev, int E, int c) {
    int lo = 0, hi = E - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (qev[mid].qchunk0 <= c) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ void cswap(uint32_t& a, uint32_t& b) {
    const uint32_t lo = min(a, b), hi = max(a, b);
    a = lo;
    b = hi;
}

// Sort one lane's list (the n <= P slots in li, accepted for query q) by (d2,
// original index) into ld, li; the places from n to P get the padding.
template <int D, int P>
__device__ __forceinline__ void sort_row(float* ld, int32_t* li, int n, const float4 q, const float4* rpts,
                                         const int32_t* perm) {
    const float qv[4] = {q.x, q.y, q.z, q.w};
    uint32_t k[P];
#pragma unroll
    for (int e = 0; e < P; ++e) {
        // empty places: above every distance, 32 apart
        k[e] = 0x80000000u | (uint32_t)(e * 33);
        if (e < n) {
            const float4 u = __ldg(rpts + li[e]);
            const float cu[4] = {u.x, u.y, u.z, u.w};
            float s = 0.f;
#pragma unroll
            for (int kk = 0; kk < D; ++kk) {
                const float d = __fsub_rn(qv[kk], cu[kk]);
                s = __fadd_rn(s, __fmul_rn(d, d));
            }
            ld[e] = s;
            k[e] = (__float_as_uint(s) & ~31u) | (uint32_t)e;
        }
    }
#pragma unroll
    for (int p = 1; p < P; p <<= 1) {
#pragma unroll
        for (int q = p; q >= 1; q >>= 1) {
#pragma unroll
            for (int i = 0; i < P; ++i) {
                const int j = q % p;
                if (i >= j && (i - j) % (2 * q) < q && i + q < P && i / (2 * p) == (i + q) / (2 * p))
                    cswap(k[i], k[i + q]);
            }
        }
    }
    uint32_t near = 32u;
#pragma unroll
    for (int i = 0; i + 1 < P; ++i) near = min(near, k[i] ^ k[i + 1]);
    int32_t x[P];
#pragma unroll
    for (int i = 0; i < P; ++i) x[i] = i < n ? __ldg(perm + li[k[i] & 31]) : -1;
    {
        float v[P];
#pragma unroll
        for (int i = 0; i < P; ++i) v[i] = ld[k[i] & 31];
#pragma unroll
        for (int i = 0; i < P; ++i) ld[i] = i < n ? v[i] : INFINITY;
    }
#pragma unroll
    for (int i = 0; i < P; ++i) li[i] = x[i];
    if (near < 32u) {
        // entries whose truncated distances agree: insertion on the whole key
        for (int i = 1; i < n; ++i) {
            const float d = ld[i];
            const int32_t x = li[i];
            int j = i;
            while (j > 0 && (ld[j - 1] > d || (ld[j - 1] == d && li[j - 1] > x))) {
                ld[j] = ld[j - 1];
                li[j] = li[j - 1];
                --j;
            }
            ld[j] = d;
            li[j] = x;
        }
    }
}

template <int D, int G>
__global__ void __launch_bounds__(kWarps * 32, kMinBlocks) k_low_query(QueryArgs a) {
    pdl_trigger();
    pdl_wait();
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char* base = smem + (size_t)warp * kWarpBytes;
    const WarpSmem w{reinterpret_cast<int32_t*>(base), reinterpret_cast<float*>(base) + 32 * kListStr,
                     reinterpret_cast<int2*>(base + 32 * kListStr * 4),
                     reinterpret_cast<int32_t*>(base + 2 * 32 * kListStr * 4)};
    constexpr int kPer = 32 / G;   // queries of a warp
    // ranges of about three slots (D = 3): pairs save wavefronts of the load
    // pipe (1 M points, 9 neighbours each: 294 -> 275 us, build included);
    // with four coordinates the longer ranges' extra steps cost more (300,000
    // points: 152 -> 161), with two neither matters
    constexpr bool PAIRS = D == 3;
    const int sq = lane / G;       // the query this lane searches for
    int32_t* li = w.Li + sq * kListStr;
    int2* rng = w.rng + lane;
    const float4* rpts = reinterpret_cast<const float4*>(a.rpts);   // rows of 4 floats up to D = 4
    const float r2 = a.r2;
    const int K = a.K;
    const int width = a.csr ? kCsrStageW : K;
    const int w4 = width >> 2;
    const int ntasks = (int)(((int64_t)a.nchunks * kChunkQ + kPer - 1) / kPer);

    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(a.task_counter, 1);
        t = __shfl_sync(kFull, t, 0);
        if (t >= ntasks) break;
        const int64_t pos0 = (int64_t)t * kPer + sq;
        const int c = (int)(pos0 / kChunkQ);
        const int e = a.nev > 1 ? chunk_event(a.qev, a.nev, min(c, a.nchunks - 1)) : 0;
        const EventHdr& hq = a.qev[e];
        const EventHdr& h = a.ev[e];
        int qs = (int)(hq.pt_off + (int64_t)(c - hq.qchunk0) * kChunkQ) + (int)(pos0 % kChunkQ);
        bool act = c < a.nchunks && (int64_t)qs < hq.pt_off + hq.n &&
                         !(a.path_filter >= 0 && h.path != a.path_filter);   // else another launch's event
        const bool search = act && h.valid;   // non-finite input: empty rows (frnn_sync reports it)
        int qorig = act ? a.qperm[qs] : 0;
        int cnt = 0;
        if constexpr (G > 1) {
            w.cnt[lane] = 0;
            __syncwarp();
        }
        // next place in the query's list
        auto place = [&]() -> int {
            if constexpr (G > 1) return atomicAdd(w.cnt + sq, 1);
            return cnt++;
        };
        if (search) {
            const int naxes = h.naxes, m = h.m;
            const float4 q4 = reinterpret_cast<const float4*>(a.qpts)[qs];
            const float qv[4] = {q4.x, q4.y, q4.z, q4.w};
            const int32_t* cells = a.cstart + h.cell_off;
            const int dims0 = h.dims[0];
            int row = div_mag(a.qcell[qs], h.mag[0]);
            const int x = a.qcell[qs] - row * dims0;
            const int x0 = max(x - m, 0), x1 = min(x + m, dims0 - 1) + 1;
            // coordinates of the query's row and their strides, axes 1..3
            int cc[3], dm[3], rs[3], nrows = 1;
            {
                int v = row, st = 1;
#pragma unroll
                for (int ax = 0; ax < 3; ++ax) {
                    cc[ax] = 0;
                    dm[ax] = 1;
                    rs[ax] = 0;
                    if (ax + 1 < D && ax + 1 < naxes) {
                        dm[ax] = h.dims[ax + 1];
                        const int qd = div_mag(v, h.mag[ax + 1]);
                        cc[ax] = v - qd * dm[ax];
                        v = qd;
                        rs[ax] = st * dims0;
                        st *= dm[ax];
                        nrows *= 2 * m + 1;
                    }
                }
            }
            const int self_slot = a.self ? qs : -1;
            // the neighbour rows' offsets, counted like digits of base 2m + 1;
            // of a query's G lanes each takes every G-th row
            const int side = 2 * m + 1, first = G > 1 ? lane % G : 0;
            const int step0 = G % side, step1 = G / side;   // (below side: G <= 8)
            int d0 = (naxes > 1 ? -m : 0) + first % side;
            int d1 = (naxes > 2 ? -m : 0) + first / side % side;
            int d2 = (naxes > 3 ? -m : 0) + first / side / side;
            const int row0 = row * dims0;
            for (int l0 = first; l0 < nrows; l0 += kRows * G) {
                int k = 0;
                {
                    int lo[kRows], hi[kRows];
#pragma unroll
                    for (int j = 0; j < kRows; ++j) {
                        lo[j] = 0;
                        hi[j] = 0;
                        const bool ok = l0 + j * G < nrows && (unsigned)(cc[0] + d0) < (unsigned)dm[0] &&
                                        (unsigned)(cc[1] + d1) < (unsigned)dm[1] &&
                                        (unsigned)(cc[2] + d2) < (unsigned)dm[2];
                        if (ok) {
                            const int at = row0 + d0 * rs[0] + d1 * rs[1] + d2 * rs[2];
                            lo[j] = __ldg(cells + at + x0);
                            hi[j] = __ldg(cells + at + x1);
                        }
                        if constexpr (G == 1) {
                            if (++d0 > m) {
                                d0 = -m;
                                if (++d1 > m) {
                                    d1 = -m;
                                    ++d2;
                                }
                            }
                        } else {
                            d0 += step0;
                            d1 += step1;
                            if (d0 > m) {
                                d0 -= side;
                                ++d1;
                            }
                            if (d1 > m) {
                                d1 -= side;
                                ++d2;
                            }
                        }
                    }
#pragma unroll
                    for (int j = 0; j < kRows; ++j) {
                        if (hi[j] > lo[j]) {
                            rng[k * 32] = make_int2(lo[j], hi[j]);
                            ++k;
                        }
                    }
                }
                // the ranges back to back, two candidates a step, the next
                // step's rows in flight.  PAIRS: an aligned pair of slots with
                // one 32-byte load (either may lie outside its range: such a
                // slot is read, not used; the rows run on past the last slot);
                // else the next two slots of the range with one load each
                int p_n = 0, lo_n = 0, hi_n = 0, i = 0;
                float c_n[8];
                auto next = [&]() -> bool {
                    if (p_n >= hi_n) {
                        if (i == k) return false;
                        const int2 r = rng[i * 32];
                        lo_n = r.x;
                        hi_n = r.y;
                        p_n = PAIRS ? lo_n & ~1 : lo_n;
                        ++i;
                    }
                    if constexpr (PAIRS) {
                        load_pair(rpts + p_n, c_n);
                    } else {
                        const float4 u = __ldg(rpts + p_n), v = __ldg(rpts + min(p_n + 1, hi_n - 1));
                        c_n[0] = u.x;
                        c_n[1] = u.y;
                        c_n[2] = u.z;
                        c_n[3] = u.w;
                        c_n[4] = v.x;
                        c_n[5] = v.y;
                        c_n[6] = v.z;
                        c_n[7] = v.w;
                    }
                    return true;
                };
                bool more = next();
                while (more) {
                    const int p = p_n;
                    const bool one = !PAIRS || p >= lo_n, two = p + 1 < hi_n;
                    const float cu[4] = {c_n[0], c_n[1], c_n[2], c_n[3]};
                    const float cv[4] = {c_n[4], c_n[5], c_n[6], c_n[7]};
                    p_n += 2;
                    more = next();
                    float s = 0.f, s2 = 0.f;
#pragma unroll
                    for (int kk = 0; kk < D; ++kk) {
                        const float du = __fsub_rn(qv[kk], cu[kk]);
                        const float dv = __fsub_rn(qv[kk], cv[kk]);
                        s = __fadd_rn(s, __fmul_rn(du, du));
                        s2 = __fadd_rn(s2, __fmul_rn(dv, dv));
                    }
                    if (one && s <= r2 && p != self_slot) {
                        const int at = place();
                        if (at < kListCap) li[at] = p;
                    }
                    if (two && s2 <= r2 && p + 1 != self_slot) {
                        const int at = place();
                        if (at < kListCap) li[at] = p + 1;
                    }
                }
            }
        }
        __syncwarp();

        // from here lane l < kPer has query l
        int32_t* counts = a.counts ? a.counts : h.counts;
        int32_t* oidx = a.counts ? a.idx : h.idx;
        float* od2 = a.counts ? a.dist2 : h.dist2;
        int ev = e;
        float* rd = w.Ld + lane * kListStr;
        int32_t* ri = w.Li + lane * kListStr;
        if constexpr (G > 1) {
            const int from = (lane * G) & 31;
            cnt = lane < kPer ? w.cnt[lane] : 0;
            act = __shfl_sync(kFull, act ? 1 : 0, from) != 0 && lane < kPer;
            qorig = __shfl_sync(kFull, qorig, from);
            qs = __shfl_sync(kFull, qs, from);
            ev = __shfl_sync(kFull, e, from);
            counts = reinterpret_cast<int32_t*>(__shfl_sync(kFull, reinterpret_cast<uint64_t>(counts), from));
            oidx = reinterpret_cast<int32_t*>(__shfl_sync(kFull, reinterpret_cast<uint64_t>(oidx), from));
            od2 = reinterpret_cast<float*>(__shfl_sync(kFull, reinterpret_cast<uint64_t>(od2), from));
        }
        // counts, degree, rows for the selection kernel
        const bool spill = cnt > kListCap;
        if (act) {
            if (!spill) counts[qorig] = min(cnt, K);
            if (spill && a.csr) counts[qorig] = kCsrSpill;   // counted by the selection kernel
            if (!spill && a.degree) a.degree[qorig] = cnt;
        }
        if (spill) {
            const int pos = atomicAdd(a.ovf_count, 1);
            if (pos < a.ovf_cap) {
                a.ovf[pos].qslot = qs;
                a.ovf[pos].ev = ev;
            } else {
                atomicOr(a.status, kStatusCapacity);
            }
        }
        const unsigned rows = __ballot_sync(kFull, act && !spill);   // rows written here
        const int n = spill ? 0 : cnt;
        const float4 q = reinterpret_cast<const float4*>(a.qpts)[n > 0 ? qs : 0];
        const int most = __reduce_max_sync(kFull, (unsigned)n);
        int sorted = 32;   // places of the lists that hold the row or its padding
        if (most <= 4) {
            sort_row<D, 4>(rd, ri, n, q, rpts, a.rperm);
            sorted = 4;
        } else if (most <= 8) {
            sort_row<D, 8>(rd, ri, n, q, rpts, a.rperm);
            sorted = 8;
        } else if (most <= 12) {
            sort_row<D, 12>(rd, ri, n, q, rpts, a.rperm);
            sorted = 12;
        } else if (most <= 16) {
            sort_row<D, 16>(rd, ri, n, q, rpts, a.rperm);
            sorted = 16;
        } else if (most <= 24) {
            sort_row<D, 24>(rd, ri, n, q, rpts, a.rperm);
            sorted = 24;
        } else {
            sort_row<D, 32>(rd, ri, n, q, rpts, a.rperm);
        }
        __syncwarp();
        int32_t* irow = oidx + (int64_t)qorig * width;
        float* drow = od2 + (int64_t)qorig * width;
        const bool aligned =
            ((reinterpret_cast<uintptr_t>(irow) | reinterpret_cast<uintptr_t>(drow)) & 15) == 0;
        const bool vec = (width & 3) == 0 && __all_sync(kFull, aligned || !act);
        if (vec && w4 <= 16) {
            // 32 / (2 w4) rows at a time: quarter p of a row is its indices for
            // p < w4, then its distances
            const int per = 2 * w4, nrow = 32 / per;
            const int g = lane / per, p = lane - g * per;
            const bool dist = p >= w4;
            const int e0 = 4 * (dist ? p - w4 : p);
            const int pad = dist ? 0x7f800000 : -1;
            const int32_t* src = (dist ? reinterpret_cast<const int32_t*>(w.Ld) : w.Li) + e0;
            const bool listed = e0 < sorted;
            const int32_t* dst = (dist ? reinterpret_cast<int32_t*>(a.dist2) : a.idx) + e0;
            for (int q0 = 0; q0 < kPer; q0 += nrow) {
                const int q = q0 + g;
                const int qq = q & 31;
                const int nq = __shfl_sync(kFull, n, qq);
                uint64_t at;
                if (a.counts) {   // one event: the arguments' outputs
                    at = reinterpret_cast<uint64_t>(dst + (int64_t)__shfl_sync(kFull, qorig, qq) * width);
                } else {
                    const uint64_t ip = __shfl_sync(kFull, reinterpret_cast<uint64_t>(irow), qq);
                    const uint64_t dp = __shfl_sync(kFull, reinterpret_cast<uint64_t>(drow), qq);
                    at = (dist ? dp : ip) + (uint64_t)e0 * 4;
                }
                if (g < nrow && q < 32 && ((rows >> qq) & 1u) && (!a.csr || e0 < nq)) {
                    int4 v = make_int4(pad, pad, pad, pad);
                    if (listed) {
                        const int32_t* s = src + qq * kListStr;
                        v = make_int4(s[0], s[1], s[2], s[3]);
                    }
                    *reinterpret_cast<int4*>(at) = v;
                }
            }
        } else {
            unsigned left = rows;
            while (left) {
                const int q = __ffs(left) - 1;
                left &= left - 1u;
                int32_t* ip = reinterpret_cast<int32_t*>(__shfl_sync(kFull, reinterpret_cast<uint64_t>(irow), q));
                float* dp = reinterpret_cast<float*>(__shfl_sync(kFull, reinterpret_cast<uint64_t>(drow), q));
                const int nq = __shfl_sync(kFull, n, q);
                const int stop = a.csr ? min(nq, width) : width;
                if (vec) {
                    for (int p = lane; 4 * p < stop; p += 32) {
                        const int e0 = 4 * p;
                        const bool listed = e0 < sorted;
                        const int32_t* si = w.Li + q * kListStr + (listed ? e0 : 0);
                        const float* sd = w.Ld + q * kListStr + (listed ? e0 : 0);
                        *reinterpret_cast<int4*>(ip + e0) =
                            listed ? make_int4(si[0], si[1], si[2], si[3]) : make_int4(-1, -1, -1, -1);
                        *reinterpret_cast<float4*>(dp + e0) =
                            listed ? make_float4(sd[0], sd[1], sd[2], sd[3])
                                   : make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
                    }
                } else {
                    for (int e2 = lane; e2 < stop; e2 += 32) {
                        ip[e2] = e2 < sorted ? w.Li[q * kListStr + e2] : -1;
                        dp[e2] = e2 < sorted ? w.Ld[q * kListStr + e2] : INFINITY;
                    }
                }
            }
        }
        __syncwarp();
    }
}

template <int D, int G>
cudaError_t launch_g(const QueryArgs& a, int num_sms, cudaStream_t st) {
    auto kern = &k_low_query<D, G>;
    const size_t smem = kWarps * kWarpBytes;
    cudaError_t ce = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (ce != cudaSuccess) return ce;
    int per_sm = 0;
    ce = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kWarps * 32, smem);
    if (ce != cudaSuccess) return ce;
    const int64_t blocks = (int64_t)num_sms * std::max(per_sm, 1);
    const int64_t need = ceil_div(ceil_div((int64_t)a.nchunks * kChunkQ * G, 32), kWarps);
    launch_pdl(kern, dim3((unsigned)std::min(blocks, std::max<int64_t>(need, 1))), dim3(kWarps * 32), smem, st, a);
    return cudaGetLastError();
}

// lanes per query: one, more while that leaves resident warps without a task.
// Never two: half the rows a lane, but places in the lists from a counter
// (build + query, cells of r / r/2, us: 30,000 x 4 G = 1 50 / 77, G = 2 58 / 112,
// G = 4 46 / 89; 50,000 x 4 62 / 102, 68 / 140, 58 / 128; 20,000 x 4 -, 51 / 100,
// 38 / 78; 30,000 x 3 38 / 42, 38 / 50, 41 / 41).
template <int D>
cudaError_t launch(const QueryArgs& a, int num_sms, cudaStream_t st) {
    // (half the resident warps: 20,000 x 2 points 33.5 us with G = 4, 35 with 8)
    const int64_t warps = (int64_t)num_sms * kMinBlocks * kWarps / 2;
    const int64_t tasks = ceil_div(a.nchunks, 2);   // with one lane a query
    if (2 * tasks >= warps) return launch_g<D, 1>(a, num_sms, st);
    if (4 * tasks >= warps) return launch_g<D, 4>(a, num_sms, st);
    return launch_g<D, 8>(a, num_sms, st);
}

}  // namespace low

cudaError_t enqueue_low_query(const QueryArgs& a, int num_sms, cudaStream_t st) {
    if (a.nchunks <= 0) return cudaSuccess;
    switch (a.D) {
        case 1: return low::launch<1>(a, num_sms, st);
        case 2: return low::launch<2>(a, num_sms, st);
        case 3: return low::launch<3>(a, num_sms, st);
        case 4: return low::launch<4>(a, num_sms, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace frnn
