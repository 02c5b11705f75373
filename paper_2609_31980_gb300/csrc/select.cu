// select.cu — exact selection for the query rows that do not fit the scan
// kernels' in-kernel lists (more than 32 neighbours).
//
// One warp per row.  The lanes look the query's neighbour rows up 32 at a
// time, concatenate the non-empty slot ranges into one candidate stream (an
// exclusive scan of their lengths) and take 32 candidates of it per round,
// the next round's rows in flight while the current one is evaluated under
// the exact float32 contract.  Accepted (d2, slot) pairs are appended to a
// buffer in shared memory; at the end the slots become original indices and
// the keys (d2 bits << 32 | index) are sorted, the first K are the row.
// Whenever the buffer is nearly full it is sorted and cut to its K smallest
// keys, whose last becomes the acceptance threshold, so any degree is exact.
//
// What bounds it, and why this shape.  The work per row is a few hundred
// candidates, so it is bound by the latency of dependent loads and wants
// resident warps: the buffer of the first pass holds kSelKeys = 256 keys a
// warp (3 KB with the range table: 32 warps an SM), sorted in registers, up
// to eight keys a lane.  Rows that outgrow it when K does not leave room to
// cut (K > kSelMaxCut) are marked and finished by a second pass over the same
// list with 2K keys a warp in shared memory.  A launch with an empty list ends
// at once.  The kernel this replaces walked the neighbour rows one after
// another (27 to 81 dependent look-ups a row) and always sorted 2K keys in
// shared memory at 12 warps an SM.  Measured (build + query, 271,663 x 12
// clustered points, r = 0.12, mean degree 34, two rows in three selected): compact,
// K = 1000, 56.1 -> 1.24 ms (0.43 since the half-cell scan keeps these rows
// itself at K > 128); dense, K = 100, 0.51 ms; with no row to select, 4096 x 3:
// 41.9 -> 38.7 us.
#include <algorithm>

#include "frnn_host.h"
#include "warp_sort.cuh"

namespace frnn {
namespace sel {

constexpr int kWarps = 4;
constexpr int kSelKeys = 256;                 // buffer of the first pass (keys a warp)
constexpr int kSelMaxCut = kSelKeys - 64;     // largest K whose cut leaves two rounds of room
constexpr int kSelMostKeys = 2 * kMaxK;       // the second pass' buffer at the largest K

// Sort the first 32 P keys of buf (entries past n hold any value).
template <int P>
__device__ __forceinline__ void sort_buffer_p(uint64_t* buf, int n) {
    const int lane = threadIdx.x & 31;
    uint64_t k[P];
#pragma unroll
    for (int p = 0; p < P; ++p) {
        const int i = p * 32 + lane;   // any assignment of keys to places: the network sorts them
        k[p] = i < n ? buf[i] : ~0ull;
    }
    warp_sort<P>(k);
    __syncwarp();
#pragma unroll
    for (int p = 0; p < P; ++p) buf[lane * P + p] = k[p];
    __syncwarp();
}

__device__ __forceinline__ void sort_buffer(uint64_t* buf, int n) {
    if (n <= 32) sort_buffer_p<1>(buf, n);
    else if (n <= 64) sort_buffer_p<2>(buf, n);
    else if (n <= 128) sort_buffer_p<4>(buf, n);
    else sort_buffer_p<8>(buf, n);
}

// The second pass' buffer: a network in shared memory over the power of two
// at or above n (the places from n on are filled with the largest key).
__device__ void sort_buffer_smem(uint64_t* buf, int n) {
    const int lane = threadIdx.x & 31;
    int len = 32;
    while (len < n) len <<= 1;
    for (int i = n + lane; i < len; i += 32) buf[i] = ~0ull;
    for (int k = 2; k <= len; k <<= 1) {
        for (int j = k >> 1; j > 0; j >>= 1) {
            __syncwarp();
            for (int i = lane; i < len / 2; i += 32) {
                const int lo = ((i & ~(j - 1)) << 1) | (i & (j - 1));
                const int hi = lo + j;
                const bool up = (lo & k) == 0;
                const uint64_t x = buf[lo], y = buf[hi];
                if ((x > y) == up) {
                    buf[lo] = y;
                    buf[hi] = x;
                }
            }
        }
    }
    __syncwarp();
}

__host__ __device__ constexpr size_t warp_bytes(int cap) {
    return (size_t)cap * sizeof(uint64_t) + (size_t)(2 * kMaxNbrRows + 2) * sizeof(int32_t);
}

// BIG: the second pass (rows the first left unfinished; `cap` >= 2K keys).
template <int D, bool BIG>
__global__ void __launch_bounds__(kWarps * 32, BIG ? 1 : (D <= 8 ? 8 : (D <= 12 ? 7 : 6))) k_select(QueryArgs a, int cap) {
    pdl_trigger();
    pdl_wait();
    constexpr int DP = padded_dim(D);
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint64_t* buf = reinterpret_cast<uint64_t*>(smem + (size_t)warp * warp_bytes(cap));
    int32_t* rpre = reinterpret_cast<int32_t*>(buf + cap);   // [kMaxNbrRows + 1] stream start of each range
    int32_t* rdel = rpre + kMaxNbrRows + 1;                  // [kMaxNbrRows] slot - stream position
    const int nov = min(*a.ovf_count, a.ovf_cap);
    if (nov == 0) {
        // nothing to select; the chunk counter alone needs clearing (the
        // list is empty already), and no block of this launch reads it
        if (blockIdx.x == 0 && threadIdx.x == 0 && a.ovf_done) *a.task_counter = 0;
        return;
    }
    const int K = a.K;
    const bool count_only = a.ovf_mode == 1;
    const bool csr_rows = a.ovf_mode == 2;
    const unsigned lt_mask = (1u << lane) - 1u;
    // a warp has every stride-th row of the list; the second pass looks for the
    // marked ones 32 at a time (rows next to each other in the list, which come
    // from the same dense place, go to different warps: uniform 3000 x 3, K =
    // 300, degrees of 1,500, 0.35 ms, with 32 consecutive rows a warp 3.1)
    const int stride = gridDim.x * kWarps;
    int64_t w = (int64_t)blockIdx.x * kWarps + warp - (BIG ? 0 : stride);
    int64_t w_base = 0;
    unsigned marked = 0;
    for (;;) {
        if constexpr (BIG) {
            while (!marked && w < nov) {
                const int64_t i = w + (int64_t)lane * stride;
                marked = __ballot_sync(kFull, i < nov && a.ovf[i].ev < 0);
                w_base = w;
                w += (int64_t)stride * 32;
            }
            if (!marked) break;
        } else {
            w += stride;
            if (w >= nov) break;
        }
        int64_t at_entry = w;
        if constexpr (BIG) {
            at_entry = w_base + (int64_t)(__ffs(marked) - 1) * stride;
            marked &= marked - 1u;
        }
        const Overflow o = a.ovf[at_entry];
        const int ev = BIG ? ~o.ev : o.ev;
        if constexpr (BIG) {
            __syncwarp();   // every lane has read the entry
            if (lane == 0) a.ovf[at_entry].ev = ev;   // no mark outlives the query
        }
        const EventHdr& h = a.ev[ev];
        const int qs = o.qslot;
        const int qo = a.qperm[qs];
        float qv[DP];
        {
            const float4* q4 = reinterpret_cast<const float4*>(a.qpts + (int64_t)qs * DP);
#pragma unroll
            for (int k4 = 0; k4 < DP / 4; ++k4) {
                const float4 v = q4[k4];
                qv[4 * k4] = v.x;
                qv[4 * k4 + 1] = v.y;
                qv[4 * k4 + 2] = v.z;
                qv[4 * k4 + 3] = v.w;
            }
        }
        // the neighbour rows' slot ranges, compact, as one candidate stream
        int nr = 0, U = 0;
        {
            const int key = a.qcell[qs];
            const int qc = stored_cell(h, key);
            const int dims0 = h.dims[0], m = h.m;
            const bool half = h.half != 0;
            const int bits = key & ((1 << kHalfBits) - 1);
            const int x = qc % dims0, qrow = qc / dims0;
            const int x0 = max(x - m, 0), x1 = min(x + m, dims0 - 1);
            const int nrows = half ? 1 << (h.naxes - 1) : neighbour_rows(h);
            for (int l0 = 0; l0 < nrows; l0 += 32) {
                const int l = l0 + lane;
                int lo = 0, n = 0;
                int64_t rowbase;
                if (l < nrows && (half ? neighbour_row_half(h, qrow, bits, l, rowbase)
                                       : neighbour_row(h, qrow, l, rowbase))) {
                    lo = __ldg(a.cstart + rowbase + x0);
                    n = __ldg(a.cstart + rowbase + x1 + 1) - lo;
                }
                int incl = n;
#pragma unroll
                for (int s = 1; s < 32; s <<= 1) {
                    const int v = __shfl_up_sync(kFull, incl, s);
                    if (lane >= s) incl += v;
                }
                const unsigned bal = __ballot_sync(kFull, n > 0);
                if (n > 0) {
                    const int pos = nr + __popc(bal & lt_mask);
                    rpre[pos] = U + incl - n;
                    rdel[pos] = lo - (U + incl - n);
                }
                nr += __popc(bal);
                U += __shfl_sync(kFull, incl, 31);
            }
            __syncwarp();
        }
        int st0 = 1;   // first step of the range search: the largest power of two < nr
        while (2 * st0 < nr) st0 <<= 1;
        auto load_cand = [&](int u, int& slot, float (&cv)[DP]) {
            slot = -1;
#pragma unroll
            for (int k = 0; k < DP; ++k) cv[k] = 0.f;
            if (u < U) {
                int i = 0;
                for (int st = st0; st > 0; st >>= 1)
                    if (i + st < nr && rpre[i + st] <= u) i += st;
                slot = u + rdel[i];
                const float4* p = reinterpret_cast<const float4*>(a.rpts + (int64_t)slot * DP);
#pragma unroll
                for (int k4 = 0; k4 < DP / 4; ++k4) {
                    const float4 v = __ldg(p + k4);
                    cv[4 * k4] = v.x;
                    cv[4 * k4 + 1] = v.y;
                    cv[4 * k4 + 2] = v.z;
                    cv[4 * k4 + 3] = v.w;
                }
            }
        };
        const int self_slot = a.self ? qs : -1;
        int fill = 0, conv = 0;   // entries held; the first conv carry original indices
        int64_t deg = 0;
        float thr = a.r2;         // entries above it cannot be among the K smallest
        bool left = false;        // outgrew the buffer: the second pass takes the row
        // slots of the entries added since the last sort -> original indices
        auto resolve = [&]() {
            __syncwarp();
            for (int i = conv + lane; i < fill; i += 32) {
                const uint64_t v = buf[i];
                buf[i] = (v & 0xffffffff00000000ull) | (uint32_t)a.rperm[(uint32_t)v];
            }
            __syncwarp();
        };
        auto sort_now = [&]() {
            resolve();
            if constexpr (BIG) sort_buffer_smem(buf, fill);
            else sort_buffer(buf, fill);
        };
        int slot;
        float cv[DP];
        load_cand(lane, slot, cv);
#pragma unroll 1
        for (int k0 = 0; k0 < U; k0 += 32) {
            int slot_n;
            float cvn[DP];
            load_cand(k0 + 32 + lane, slot_n, cvn);   // next round in flight
            float s = 0.f;
#pragma unroll
            for (int k = 0; k < D; ++k) {
                const float d = __fsub_rn(qv[k], cv[k]);
                s = __fadd_rn(s, __fmul_rn(d, d));
            }
            const bool in = slot >= 0 && slot != self_slot && s <= a.r2;
            deg += in ? 1 : 0;
            if (!count_only) {
                const bool take = in && s <= thr;
                const unsigned bal = __ballot_sync(kFull, take);
                if (take) buf[fill + __popc(bal & lt_mask)] = make_key(s, slot);
                fill += __popc(bal);
                if (fill > cap - 32) {
                    if (!BIG && K > kSelMaxCut) {
                        left = true;
                        break;
                    }
                    // keep the K smallest; equal distances stay in (the
                    // index decides between them at the next sort)
                    sort_now();
                    fill = min(fill, K);
                    conv = fill;
                    if (fill == K) thr = __uint_as_float((uint32_t)(buf[K - 1] >> 32));
                    __syncwarp();
                }
            }
            slot = slot_n;
#pragma unroll
            for (int k = 0; k < DP; ++k) cv[k] = cvn[k];
        }
        if (left) {   // mark the entry for the second pass
            if (lane == 0) a.ovf[at_entry].ev = ~ev;
            __syncwarp();
            continue;
        }
        for (int s = 16; s > 0; s >>= 1) deg += __shfl_xor_sync(kFull, deg, s);
        const int32_t c = (int32_t)(deg < K ? deg : K);
        if (count_only) {
            // compact output, first pass: the row's count (marked) and degree
            if (lane == 0) {
                (a.counts ? a.counts : h.counts)[qo] = c | kCsrSpill;
                if (a.degree) a.degree[qo] = (int32_t)(deg < INT32_MAX ? deg : INT32_MAX);
            }
            __syncwarp();
            continue;
        }
        // a compact output too small for the rows (its caller fails the
        // call) is not written past its end
        if (csr_rows && a.row_off[qo] + c > a.row_cap) continue;
        sort_now();
        const int64_t at = csr_rows ? a.row_off[qo] : (int64_t)qo * K;
        int32_t* irow = (a.counts ? a.idx : h.idx) + at;
        float* drow = (a.counts ? a.dist2 : h.dist2) + at;
        for (int e = lane; e < (csr_rows ? c : K); e += 32) {
            const bool real = e < c;
            const uint64_t v = real ? buf[e] : 0;
            irow[e] = real ? (int32_t)(uint32_t)v : -1;
            drow[e] = real ? __uint_as_float((uint32_t)(v >> 32)) : INFINITY;
        }
        if (lane == 0 && !csr_rows) (a.counts ? a.counts : h.counts)[qo] = c;
        __syncwarp();
    }
    // the last block to finish clears the query's counters for the next launch
    __syncthreads();
    if (threadIdx.x == 0 && a.ovf_done) {
        __threadfence();
        if (atomicAdd(a.ovf_done, 1) == (int)gridDim.x - 1) {
            *a.task_counter = 0;
            if (a.reset_ovf) *a.ovf_count = 0;
            __threadfence();
            *a.ovf_done = 0;
        }
    }
}

template <int D, bool BIG>
cudaError_t launch(const QueryArgs& a, int cap, int num_sms, cudaStream_t st) {
    auto kern = &k_select<D, BIG>;
    const size_t smem = kWarps * warp_bytes(cap);
    // (the limit is the function's, shared by every thread's calls: always the
    // most any K needs, so that no call lowers it under another's launch)
    constexpr size_t most = kWarps * warp_bytes(BIG ? kSelMostKeys : kSelKeys);
    cudaError_t ce = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
    if (ce != cudaSuccess) return ce;
    int per_sm = 0;
    ce = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kWarps * 32, smem);
    if (ce != cudaSuccess) return ce;
    launch_pdl(kern, dim3(num_sms * std::max(per_sm, 1)), dim3(kWarps * 32), smem, st, a, cap);
    return cudaGetLastError();
}

template <int D>
cudaError_t launch_d(const QueryArgs& a, int num_sms, cudaStream_t st) {
    // rows of more than kSelMaxCut kept neighbours may need the second pass
    // (a pass that only counts needs no buffer)
    const bool two = a.K > kSelMaxCut && a.ovf_mode != 1;
    QueryArgs first = a;
    if (two) first.ovf_done = nullptr;   // the second pass clears the counters
    cudaError_t ce = launch<D, false>(first, kSelKeys, num_sms, st);
    if (ce != cudaSuccess || !two) return ce;
    int cap = 2 * kSelKeys;
    while (cap < 2 * a.K) cap <<= 1;
    return launch<D, true>(a, cap, num_sms, st);
}

}  // namespace sel

frnn_status enqueue_overflow(const QueryArgs& a, int num_sms, cudaStream_t st, std::string& err) {
    cudaError_t ce = cudaErrorInvalidValue;
    switch (a.D) {
#define FRNN_CASE(d) case d: ce = sel::launch_d<d>(a, num_sms, st); break;
        FRNN_CASE(1) FRNN_CASE(2) FRNN_CASE(3) FRNN_CASE(4) FRNN_CASE(5) FRNN_CASE(6)
        FRNN_CASE(7) FRNN_CASE(8) FRNN_CASE(9) FRNN_CASE(10) FRNN_CASE(11) FRNN_CASE(12)
        FRNN_CASE(13) FRNN_CASE(14) FRNN_CASE(15) FRNN_CASE(16)
#undef FRNN_CASE
    }
    if (ce != cudaSuccess) {
        err = std::string("selection kernel launch failed: ") + cudaGetErrorString(ce);
        return FRNN_ERR_CUDA;
    }
    return FRNN_OK;
}

}  // namespace frnn
