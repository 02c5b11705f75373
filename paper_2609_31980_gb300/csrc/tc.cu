// tc.cu — tensor-core path: a BF16 tcgen05 pre-filter over grid candidate
// tiles, followed by the exact float32 recheck of every survivor.
//
// The squared distance is written as n(x) + n(y) - 2 x.y, the dot products of
// a 128-query tile with a chunk of up to 128 candidates computed by one
// tcgen05.mma (kind::f16, BF16 operands, FP32 accumulator in tensor memory).
// The filter only has to be conservative: every pair the float32 contract
// accepts must pass it; each survivor is then recomputed with the exact
// contract, so results are bit-identical to the grid path and the oracle.
//
// Operands (per point, built once per grid by k_tc_prep):
//   x' = fl(x - c)             c = centre of the event's bounding box
//   hi = bf16(x'), lo = bf16(x' - hi)          (x' - hi is exact in float32)
//   query row  A = [hi, hi, lo, 1, 1, 0...]
//   candidate  B = [hi, lo, hi, m_hi, m_lo, 0...],  m = -n/2 split in two bf16,
//                  n = ||hi + lo||^2 in float32
// so acc = A.B ~= x'.y' - n(y)/2 and the pair passes when acc >= t(x) with
// t(x) = (n(x) - Theta)/2 rounded down.
//
// Margin (proof sketch; every factor below is a generous upper bound).  Let
// u = 2^-24, nu^2 the largest n over the event (queries and references).  The
// contract accepts => ||x - y||^2 <= R^2 = r2 (1 + 2^-18) (float32 partial
// sums of non-negative terms lose at most (1-u)^(2D+2) <= 1 - 2^-18 for
// D <= 16).  Centring moves a difference by <= u (|x'| + |y'|) per coordinate,
// the two-term split by <= 2^-16 |x'| (bf16 keeps 8 significant bits), so
// ||x^ - y^|| <= ||x - y|| + 2^-15 nu.  The GEMM drops lo.lo (<= 2^-16 nu^2),
// accumulates <= 3D + 2 exact bf16 products in float32 (<= 2^-17 (3 nu^2 + nu^2)
// with a 2x slack for the unspecified accumulation order), and the norms and
// m carry <= 2^-16 nu^2; all together |n(x) - 2 acc - ||x^ - y^||^2| <= 2^-13 nu^2.
// Theta = (R + 2^-14 nu)^2 + 2^-12 nu^2 therefore keeps every accepted pair.
// The margin is validated empirically by the parity tests (the tensor-core
// path's output must equal the oracle's bit for bit), and the tightest slack
// is what the false-candidate rate measures.
//
// Kernel organisation (persistent, two CTAs per SM of 10 warps and 256 TMEM
// columns each; a task is 128 query slots of one row of cells):
//   * a loading warp takes the next task, lists its chunks (up to 128
//     candidates each) and sends for the query tile and for the chunks'
//     operands with cp.async.bulk, into a ring up to eight deep, while the
//     other warps still work on the task before;
//   * an MMA warp issues K/16 instructions per chunk into one of two TMEM
//     accumulators of 128 columns;
//   * eight epilogue warps: warp w reads TMEM lanes 32 (w % 4).. of accumulator
//     w / 4, so every other chunk, with tcgen05.ld 32x32b.x32; it tests 32
//     pairs per thread with a 3-input max tree, looks closer only at the octets
//     of columns in which some lane's maximum reaches t(x), gives the
//     accumulator back and only then collects the survivors (a prefix sum over
//     the lanes) in a buffer; whenever 32 have come together, over groups and
//     chunks, its lanes recheck one each exactly, the candidate's float32 row
//     from L2;
//   * per-query survivor lists in shared memory are sorted by (d2, index) by
//     pairs of lanes (warp_sort.cuh), 16 rows a warp, and written as coalesced
//     rows.  Lists longer than the capacity go to select.cu.
// Every mbarrier wait is bounded; on a timeout the CTA records the status,
// stops, waits (bounded) for its copies and MMAs in flight and frees TMEM.
//
// What bounds it: latency.  500k x 12 on three axes (4,077 tasks of 31 chunks,
// 1.9 G pairs, 6.3 M survivors in 16 % of the groups): 770 us, issue 42 % of
// the slots with 19 warps an SM, tensor pipe 13 %; the lists and the operand
// ring fill shared memory at two CTAs.  The steps, build and query, K = 128:
// 1184 us with one warp for copies and MMAs, accumulators held during the
// rechecks and candidate coordinates staged (D = 16: 1985, one CTA per SM) ->
// 1105 (survivors rechecked 32 at a time from L2 rows, which 30 lanes idled
// through before; D = 16: 1061) -> 1037 (accumulators given back early, next
// task prepared during the last) -> 959 (loads and MMAs in two warps, 16-byte
// row stores) -> 863 (32-bit sorting keys in all warps, prefix-sum appends) ->
// 865 (a warp takes whole chunks instead of half of each: 50k x 12 210 -> 202;
// D = 8, 500k 876 -> 863).  Slower: sixteen epilogue warps of 56 registers
// (1542), both halves' TMEM loads in flight at once (1338, spills), 16 columns
// tested while the next 16 are on their way (892 against 856).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "frnn_host.h"
#include "warp_sort.cuh"

namespace frnn {

constexpr int kTcM = 128;        // queries per task = MMA M = TMEM lanes
constexpr int kTcN = 128;        // candidates per chunk = MMA N (multiple of 32)
constexpr int kTcAcc = 2;        // TMEM accumulators in flight (kTcAcc * kTcN = kTcCols)
constexpr int kTcEpi = 256;      // epilogue threads: warp w < 8 owns TMEM lanes 32 (w % 4)..
                                 // and accumulator w / 4
constexpr int kTcThreads = kTcEpi + 64;   // + a loading warp (tasks, bulk copies) + an MMA warp
constexpr int kTcLStr = kTcM + 1;         // list table: one column per query row
constexpr int kTcMaxChunks = 128;         // chunk table entries kept in shared memory
constexpr int kTcMaxRows = 256;           // neighbour rows per task (3^5 on a six-axis grid of half cells)
constexpr int kTcCols = 256;     // TMEM columns per CTA: two accumulators (2 CTAs / SM)
constexpr int kTcList = 30;      // per-query survivor list capacity (2 CTAs / SM)
static_assert(kTcList <= kCsrStageW, "a staged compact row holds a whole list");

__host__ __device__ constexpr int tc_k_for(int D) { return ((3 * D + 2) + 15) / 16 * 16; }

// shared memory outside the operand ring
__host__ __device__ constexpr size_t tc_smem_fixed(int K, int DP);
// operand ring depth: as deep as fits two CTAs per SM (<= 107 KB each beside
// the static part), 2..8
__host__ __device__ constexpr int tc_ring_for(int D);

constexpr int kTcSurvCap = 96;   // survivors a warp holds (it rechecks as soon as 32 have come together)

__host__ __device__ constexpr size_t tc_smem_fixed(int K, int DP) {
    return (size_t)kTcM * K * 2                                // A tile
           + (size_t)kTcList * kTcLStr * 8                     // per-query lists
           + (size_t)kTcM * DP * 4                             // query coordinates
           + (size_t)(kTcEpi / 32) * kTcSurvCap * 5;           // per-warp survivor buffers
}
__host__ __device__ constexpr size_t tc_slot_bytes(int K, int DP) {
    (void)DP;
    return (size_t)kTcN * K * 2;       // B tile
}
__host__ __device__ constexpr int tc_ring_for(int D) {
    int r = 8;
    while (r > 2 && tc_smem_fixed(tc_k_for(D), padded_dim(D)) +
                            (size_t)r * tc_slot_bytes(tc_k_for(D), padded_dim(D)) >
                        107 * 1024)
        --r;
    return r;
}
__host__ __device__ constexpr size_t tc_smem_bytes(int D) {
    return tc_smem_fixed(tc_k_for(D), padded_dim(D)) +
           (size_t)tc_ring_for(D) * tc_slot_bytes(tc_k_for(D), padded_dim(D));
}

// element offset of (row s, column k) in the core-matrix layout of rows of K
// bf16: groups of 8 rows, inside a group K/8 core matrices of 8 rows x 16 B
__device__ __forceinline__ int64_t cm_off(int64_t s, int k, int K) {
    return ((s >> 3) * (K >> 3) + (k >> 3)) * 64 + (s & 7) * 8 + (k & 7);
}

// ------------------------------------------------------------- operand prep

__device__ __forceinline__ int find_event_slot(const EventHdr* hdr, int E, int64_t s) {
    int lo = 0, hi = E - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (hdr[mid].pt_off <= s) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ uint16_t bf16_bits(__nv_bfloat16 v) {
    return *reinterpret_cast<uint16_t*>(&v);
}

// One thread per slot: centred split operands, norm, per-event max norm.
// own: headers of this point set; ctr: headers whose centres to use.
template <int D>
__global__ void k_tc_prep(const EventHdr* own, const EventHdr* ctr, int E, int64_t n_total,
                          const float* pts, uint16_t* tcA, uint16_t* tcB, float* tcn,
                          int32_t* tcnu) {
    constexpr int K = tc_k_for(D);
    constexpr int DP = padded_dim(D);
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_total) return;
    const int e = find_event_slot(own, E, s);
    const EventHdr& h = own[e];
    const bool real = s < h.pt_off + h.n && ctr[e].valid;
    uint16_t hi[D], lo[D];
    float n = 0.f;
#pragma unroll
    for (int k = 0; k < D; ++k) {
        hi[k] = 0;
        lo[k] = 0;
        if (real) {
            const float xc = __fsub_rn(pts[pt_index(s, k, DP)], ctr[e].ctr[k]);
            const __nv_bfloat16 bh = __float2bfloat16_rn(xc);
            const __nv_bfloat16 bl = __float2bfloat16_rn(__fsub_rn(xc, __bfloat162float(bh)));
            const float xh = __fadd_rn(__bfloat162float(bh), __bfloat162float(bl));
            n = __fmaf_rn(xh, xh, n);
            hi[k] = bf16_bits(bh);
            lo[k] = bf16_bits(bl);
        }
    }
    uint16_t one = 0, mh = 0, ml = 0;
    if (real) {
        const float mneg = -0.5f * n;
        const __nv_bfloat16 bmh = __float2bfloat16_rn(mneg);
        const __nv_bfloat16 bml = __float2bfloat16_rn(__fsub_rn(mneg, __bfloat162float(bmh)));
        one = bf16_bits(__float2bfloat16_rn(1.f));
        mh = bf16_bits(bmh);
        ml = bf16_bits(bml);
    }
    // A = [hi, hi, lo, 1, 1, 0...], B = [hi, lo, hi, m_hi, m_lo, 0...]
    auto a_el = [&](int j) -> uint32_t {
        return j < D ? hi[j] : j < 2 * D ? hi[j - D] : j < 3 * D ? lo[j - 2 * D]
               : (j == 3 * D || j == 3 * D + 1) ? one : 0;
    };
    auto b_el = [&](int j) -> uint32_t {
        return j < D ? hi[j] : j < 2 * D ? lo[j - D] : j < 3 * D ? hi[j - 2 * D]
               : j == 3 * D ? mh : j == 3 * D + 1 ? ml : 0;
    };
#pragma unroll
    for (int kg = 0; kg < K / 8; ++kg) {
        uint4 va, vb;
        va.x = a_el(8 * kg + 0) | (a_el(8 * kg + 1) << 16);
        va.y = a_el(8 * kg + 2) | (a_el(8 * kg + 3) << 16);
        va.z = a_el(8 * kg + 4) | (a_el(8 * kg + 5) << 16);
        va.w = a_el(8 * kg + 6) | (a_el(8 * kg + 7) << 16);
        vb.x = b_el(8 * kg + 0) | (b_el(8 * kg + 1) << 16);
        vb.y = b_el(8 * kg + 2) | (b_el(8 * kg + 3) << 16);
        vb.z = b_el(8 * kg + 4) | (b_el(8 * kg + 5) << 16);
        vb.w = b_el(8 * kg + 6) | (b_el(8 * kg + 7) << 16);
        const int64_t off = cm_off(s, 8 * kg, K);
        *reinterpret_cast<uint4*>(tcA + off) = va;
        *reinterpret_cast<uint4*>(tcB + off) = vb;
    }
    tcn[s] = n;
    // per-event maximum: reduce across the warp first when its lanes share an
    // event (almost always), one atomic per warp instead of one per point
    const int32_t on = real ? float_to_ordered(n) : INT32_MIN;
    const unsigned same = __match_any_sync(__activemask(), e);
    const int32_t wmax = __reduce_max_sync(same, on);
    if (real && (threadIdx.x & 31) == __ffs(same) - 1) atomicMax(tcnu + e, wmax);
}

// ------------------------------------------------------------- tcgen05 helpers

__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    uint64_t d = 0;
    d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
    d |= (uint64_t)1 << 46;   // descriptor version for tcgen05; no swizzle, base offset 0
    return d;
}

// kind::f16 instruction descriptor: FP32 accumulate, BF16 A and B, both
// K-major, M = 128, N = n
__device__ __forceinline__ uint32_t mma_idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
           ((uint32_t)(kTcM >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                         uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile(
        "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
            smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// tcgen05.ld of 32 columns without the wait (several loads share one wait)
__device__ __forceinline__ void tmem_ld32_nowait(uint32_t taddr, uint32_t (&r)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
        "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
          "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]),
          "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]),
          "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr));
}
// The wait for that load: its registers pass through, so that no use of them is
// moved above it.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[32]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
                   "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]),
                   "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]),
                   "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]),
                   "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]),
                   "+r"(r[31])
                 :
                 : "memory");
}

__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

struct TcArgs {
    const EventHdr* ev;       // reference grid headers
    const Task* tasks;        // 128-query tasks of the query set
    const int32_t* ntasks;
    const uint16_t* tcA;      // query-set operands
    const uint16_t* tcB;      // reference operands
    const float* qn;          // query norms
    const int32_t* nu_q;      // per-event max norms (ordered ints)
    const int32_t* nu_r;
    const float* qpts;
    const int32_t* qperm;
    const int32_t* qcell;
    const float* rpts;
    const int32_t* rperm;
    const int32_t* cstart;
    int32_t* counts;          // single-event outputs or NULL (per-event headers)
    int32_t* idx;
    float* dist2;
    float r2;
    int32_t K;
    int32_t self;
    int32_t D;
    int32_t* task_counter;
    int32_t* status;
    Overflow* ovf;
    int32_t* ovf_count;
    int32_t ovf_cap;
    int32_t path_filter;                  // -1: every event; else only events with this path
    unsigned long long* stat_survivors;   // pre-filter survivors (false-candidate rate)
    unsigned long long* stat_accepted;    // exact accepts
    int32_t csr;                          // compact output: staging rows (see QueryArgs)
    int32_t* degree;
};

// Sort 16 lists held as columns (entry e of list r at Ld[e * kTcLStr + r]) by
// (d2, original index), in place: lanes q and q + 16 share list r0 + q of n <=
// 2 P entries (n the same on both).  Keys as in the half-cell scan: the
// distance's bits with the low five cleared, then the entry's place; lists in
// which two truncated distances agree are ordered by counting.
template <int P>
__device__ __forceinline__ void sort_columns(float* Ld, int32_t* Li, int r0, int n) {
    const int lane = threadIdx.x & 31, hh = lane >> 4;
    float* ld = Ld + r0 + (lane & 15);
    int32_t* li = Li + r0 + (lane & 15);
    uint32_t k[P];
#pragma unroll
    for (int i = 0; i < P; ++i) {
        const int e = hh * P + i;
        // empty places: above every distance, 32 apart
        k[i] = e < n ? (__float_as_uint(ld[e * kTcLStr]) & ~31u) | (uint32_t)e : 0x80000000u | (uint32_t)(e * 33);
    }
    const unsigned tied = __ballot_sync(kFull, sort_pair<P>(k));
    {
        float v[P];
#pragma unroll
        for (int i = 0; i < P; ++i) v[i] = hh * P + i < n ? ld[(k[i] & 31) * kTcLStr] : 0.f;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < P; ++i)
            if (hh * P + i < n) ld[(hh * P + i) * kTcLStr] = v[i];
    }
    {
        int32_t v[P];
#pragma unroll
        for (int i = 0; i < P; ++i) v[i] = hh * P + i < n ? li[(k[i] & 31) * kTcLStr] : 0;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < P; ++i)
            if (hh * P + i < n) li[(hh * P + i) * kTcLStr] = v[i];
    }
    __syncwarp();
    unsigned rows = (tied | (tied >> 16)) & 0xffffu;
    while (rows) {
        const int r = __ffs(rows) - 1;
        rows &= rows - 1u;
        const int nr = __shfl_sync(kFull, n, r);
        const float d = lane < nr ? Ld[lane * kTcLStr + r0 + r] : 0.f;
        const int32_t x = lane < nr ? Li[lane * kTcLStr + r0 + r] : 0;
        int rank = 0;
        for (int j = 0; j < nr; ++j) {
            const float dj = __shfl_sync(kFull, d, j);
            const int32_t xj = __shfl_sync(kFull, x, j);
            rank += (dj < d || (dj == d && xj < x)) ? 1 : 0;
        }
        __syncwarp();
        if (lane < nr) {
            Ld[rank * kTcLStr + r0 + r] = d;
            Li[rank * kTcLStr + r0 + r] = x;
        }
    }
    __syncwarp();
}

// Chunk geometry of a task: neighbour row L covers slot range [rs, re); its
// operand rows start at b8 = rs rounded down to 8 and end at e8 = re rounded
// up to 8; chunks of up to kTcN rows (the MMA N, rounded up to 32).
struct ChunkTab {
    int rs[kTcMaxRows], re[kTcMaxRows], pref[kTcMaxRows + 1];
    int nrows;
    int4 chunk[kTcMaxChunks];   // (start, n, lo, hi) of the first chunks
};

__device__ __forceinline__ int4 chunk_info(const ChunkTab& t, int c) {
    if (c < kTcMaxChunks) return t.chunk[c];
    int L = 0;
    while (L + 1 < t.nrows && t.pref[L + 1] <= c) ++L;
    const int start = (t.rs[L] & ~7) + (c - t.pref[L]) * kTcN;
    const int e8 = (t.re[L] + 7) & ~7;
    // whole 32-column TMEM loads; extra rows are masked by [lo, hi)
    return make_int4(start, (min(kTcN, e8 - start) + 31) & ~31, t.rs[L], t.re[L]);
}

// A task the loading warp has prepared.
struct TcTask {
    Task t;
    int nch;        // chunks (0: nothing to compare, or an invalid event)
    int done;       // no more tasks
    float theta;    // the event's pre-filter radius, rounded up
};

template <int D>
__global__ void __launch_bounds__(kTcThreads, 2) k_tc_query(TcArgs a) {
    constexpr int K = tc_k_for(D);
    constexpr int KS = K / 16;
    constexpr int DP = padded_dim(D);
    constexpr int kTcRing = tc_ring_for(D);
    extern __shared__ __align__(1024) unsigned char smem[];
    uint16_t* As = reinterpret_cast<uint16_t*>(smem);
    uint16_t* Bs = As + kTcM * K;
    float* Ld = reinterpret_cast<float*>(Bs + kTcRing * kTcN * K);
    int32_t* Li = reinterpret_cast<int32_t*>(Ld + kTcList * kTcLStr);
    float* Qs = reinterpret_cast<float*>(Li + kTcList * kTcLStr);      // [128][DP]
    uint32_t* Sv = reinterpret_cast<uint32_t*>(Qs + kTcM * DP);        // [warps][kTcSurvCap] slots, then rows

    // bar_b: chunk operands landed; bar_mma: accumulator ready and s_chunk
    // written; bar_acc: epilogue has read an accumulator (and its s_chunk);
    // bar_slot: MMAs done with a ring slot
    __shared__ __align__(8) uint64_t bar_a, bar_b[kTcRing], bar_mma[kTcAcc], bar_acc[kTcAcc],
        bar_slot[kTcRing];
    __shared__ uint32_t s_taddr;
    __shared__ TcTask s_task[2];
    __shared__ int s_abort;
    __shared__ ChunkTab s_ct;            // the loading warp's own
    __shared__ int4 s_load[kTcRing];     // (start, n, lo, hi) of the chunk in each ring slot
    __shared__ int4 s_chunk[kTcAcc];     // and in each accumulator
    __shared__ int s_cnt[kTcM];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_u32(&s_taddr)), "n"(kTcCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    if (tid == 0) {
        mbar_init(&bar_a, 1);
        for (int i = 0; i < kTcRing; ++i) {
            mbar_init(&bar_b[i], 1);
            mbar_init(&bar_slot[i], 1);
        }
        for (int i = 0; i < kTcAcc; ++i) {
            mbar_init(&bar_mma[i], 2);        // the MMAs' commit and the MMA warp
            mbar_init(&bar_acc[i], kTcEpi / kTcAcc);   // its epilogue threads, every chunk
        }
        s_abort = 0;
        fence_mbar_init();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t taddr = s_taddr;

    auto abort_now = [&]() {
        atomicOr(a.status, kStatusTimeout);
        atomicExch(&s_abort, 1);
    };
    auto aborted = [&]() -> int { return *reinterpret_cast<volatile int*>(&s_abort); };

    uint32_t g0 = 0;          // global chunk counter at the start of the task

    if (warp == kTcEpi / 32) {
        // ------------------------------------------------------ loading warp
        const int ntasks = *a.ntasks;
        int theta_ev = -1;
        float theta = 0.f;
        uint32_t a_loads = 0, g_loads = 0;   // query tiles and chunks sent for so far
        // Take the next task and list its chunks, while the other warps still
        // work on the task before.
        auto prepare = [&](TcTask& out) -> int {
            int t;
            Task tk;
            for (;;) {
                t = 0;
                if (lane == 0) t = aborted() ? ntasks : atomicAdd(a.task_counter, 1);
                t = __shfl_sync(0xffffffffu, t, 0);
                if (t >= ntasks) break;
                tk = a.tasks[t];
                if (a.path_filter < 0 || a.ev[tk.ev].path == a.path_filter) break;   // (else another launch's event)
            }
            if (t >= ntasks) {
                if (lane == 0) out.done = 1;
                return -1;
            }
            const EventHdr& h = a.ev[tk.ev];
            int carry = 0;
            if (h.valid) {
                const int dims0 = h.dims[0], m = h.m;
                const int xa = stored_cell(h, a.qcell[tk.qslot]) % dims0;
                const int xb = stored_cell(h, a.qcell[tk.qslot + tk.nq - 1]) % dims0;
                // (2m+1)^(naxes-1) <= kTcMaxRows rows (the grid parameters ensure
                // it), 32 per round with a running chunk count
                const int nrows = neighbour_rows(h);
                for (int rr = 0; rr * 32 < nrows; ++rr) {
                    const int l = rr * 32 + lane;
                    int rs = 0, re = 0;
                    int64_t rowbase;
                    if (l < nrows && neighbour_row(h, tk.row, l, rowbase)) {
                        rs = a.cstart[rowbase + max(xa - m, 0)];
                        re = a.cstart[rowbase + min(xb + m, dims0 - 1) + 1];
                    }
                    const int b8 = rs & ~7;
                    const int e8 = (re + 7) & ~7;
                    const int nch = re > rs ? (e8 - b8 + kTcN - 1) / kTcN : 0;
                    int pre = nch;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int v = __shfl_up_sync(0xffffffffu, pre, o);
                        if (lane >= o) pre += v;
                    }
                    if (l < kTcMaxRows) {
                        s_ct.rs[l] = rs;
                        s_ct.re[l] = re;
                        s_ct.pref[l] = carry + pre - nch;
                    }
                    // this lane's row: its chunks' (start, n, lo, hi)
                    for (int j = 0; j < nch; ++j) {
                        const int c = carry + pre - nch + j;
                        if (c >= kTcMaxChunks) break;
                        const int start = b8 + j * kTcN;
                        s_ct.chunk[c] = make_int4(start, (min(kTcN, e8 - start) + 31) & ~31, rs, re);
                    }
                    carry += __shfl_sync(0xffffffffu, pre, 31);
                }
                if (lane == 0) s_ct.nrows = nrows;
                if (tk.ev != theta_ev) {
                    const double nu2 = fmax((double)ordered_to_float(a.nu_q[tk.ev]),
                                            (double)ordered_to_float(a.nu_r[tk.ev]));
                    const double nu = sqrt(fmax(nu2, 0.0));
                    const double R = sqrt((double)a.r2 * (1.0 + 0x1p-18));
                    theta = __double2float_ru((R + 0x1p-14 * nu) * (R + 0x1p-14 * nu) + 0x1p-12 * nu2);
                    theta_ev = tk.ev;
                }
            }
            if (lane == 0) {
                out.t = tk;
                out.nch = carry;
                out.done = 0;
                out.theta = theta;
            }
            __syncwarp();
            return carry;
        };
        // chunk c of the listed task into ring slot g % R, which is free once
        // the MMAs of chunk g - R are done
        auto load = [&](int c, uint32_t g) -> bool {
            const int slot = g % kTcRing;
            const int4 ci = chunk_info(s_ct, c);
            if (g >= (uint32_t)kTcRing &&
                !mbar_wait_bounded(&bar_slot[slot], ((g - kTcRing) / kTcRing) & 1u))
                return false;
            s_load[slot] = ci;
            const uint32_t bB = (uint32_t)ci.y * K * 2;
            mbar_arrive_expect_tx(&bar_b[slot], bB);
            bulk_g2s(Bs + (size_t)slot * kTcN * K, a.tcB + cm_off(ci.x, 0, K), bB, &bar_b[slot]);
            g_loads = g + 1;
            return true;
        };
        // its query tile and its first chunks; the MMAs of the task before are
        // done (they read the tile this overwrites)
        auto start_loads = [&](const TcTask& tt, int nch) -> int {
            if (lane != 0 || nch <= 0) return 0;
            const uint32_t bA = (uint32_t)kTcM * K * 2;
            mbar_arrive_expect_tx(&bar_a, bA);
            bulk_g2s(As, a.tcA + cm_off(tt.t.qslot & ~7, 0, K), bA, &bar_a);
            ++a_loads;
            int c = 0;
            for (; c < nch && c < kTcRing; ++c) {
                if (!load(c, g0 + c)) {
                    abort_now();
                    break;
                }
            }
            return c;
        };

        int nch = prepare(s_task[0]);
        int loaded = start_loads(s_task[0], nch);
        for (uint32_t par = 0;; par ^= 1u) {
            __syncthreads();   // this task is ready; the epilogue has finished the one before
            if (nch < 0) break;
            if (lane == 0) {
                for (; loaded < nch && !aborted(); ++loaded) {
                    if (!load(loaded, g0 + loaded)) {
                        abort_now();
                        break;
                    }
                }
            }
            __syncwarp();
            const uint32_t g_end = g0 + (uint32_t)nch;
            const int nch_next = prepare(s_task[par ^ 1u]);
            // the query tile is free when the task's last MMAs are done
            if (lane == 0 && nch > 0 && !aborted() &&
                !mbar_wait_bounded(&bar_slot[(g_end - 1) % kTcRing], ((g_end - 1) / kTcRing) & 1u))
                abort_now();
            __syncwarp();
            g0 = g_end;
            nch = nch_next;
            loaded = aborted() ? 0 : start_loads(s_task[par ^ 1u], nch);
        }
        // after a timeout: copies that no MMA waited for (chunk g's is the last
        // phase of its slot's barrier)
        if (lane == 0 && aborted()) {
            if (a_loads > 0) mbar_wait_bounded(&bar_a, (a_loads - 1) & 1u);
            for (uint32_t g = g_loads - min(g_loads, (uint32_t)kTcRing); g < g_loads; ++g)
                mbar_wait_bounded(&bar_b[g % kTcRing], (g / kTcRing) & 1u);
        }
        __syncwarp();
    } else if (warp == kTcEpi / 32 + 1) {
        // ---------------------------------------------------------- MMA warp
        const uint32_t lbo = 128, sbo = (uint32_t)K * 16;
        const uint64_t descA = smem_desc(smem_u32(As), lbo, sbo);
        const uint64_t descB = smem_desc(smem_u32(Bs), lbo, sbo);
        uint32_t a_tiles = 0;     // query tiles waited for so far
        for (uint32_t par = 0;; par ^= 1u) {
            __syncthreads();
            if (s_task[par].done) break;
            const int nch = s_task[par].nch;
            if (lane == 0 && nch > 0) {
                bool ok = !aborted() && mbar_wait_bounded(&bar_a, a_tiles & 1u);
                int issued = 0;
                for (int c = 0; ok && c < nch; ++c) {
                    const uint32_t g = g0 + c;
                    const int slot = g % kTcRing;
                    const uint32_t acc = g % kTcAcc;
                    // operands landed and the accumulator's previous chunk read
                    ok = !aborted() && mbar_wait_bounded(&bar_b[slot], (g / kTcRing) & 1u);
                    const int4 ci = s_load[slot];
                    const uint32_t idesc = mma_idesc(ci.y);
                    const uint64_t db = descB + (uint32_t)slot * (kTcN * K * 2 / 16);
                    if (ok && g >= (uint32_t)kTcAcc)
                        ok = mbar_wait_bounded(&bar_acc[acc], ((g - kTcAcc) / kTcAcc) & 1u);
                    if (!ok) break;
                    tc_fence_after();
#pragma unroll
                    for (int ks = 0; ks < KS; ++ks)
                        mma_bf16(taddr + acc * kTcN, descA + ks * 16, db + ks * 16, idesc,
                                 ks > 0 ? 1u : 0u);
                    mma_commit(&bar_mma[acc]);
                    mma_commit(&bar_slot[slot]);
                    s_chunk[acc] = ci;
                    mbar_arrive(&bar_mma[acc]);
                    issued = c + 1;
                }
                if (!ok) {
                    abort_now();
                    if (issued > 0) {   // the MMAs in flight
                        const uint32_t g = g0 + issued - 1;
                        mbar_wait_bounded(&bar_slot[g % kTcRing], (g / kTcRing) & 1u);
                    }
                }
                ++a_tiles;
            }
            __syncwarp();
            g0 += nch;
        }
    } else {
        // ---------------------------------------------------------- epilogue
        const int half = warp >> 2;                // accumulator: every other chunk
        const int row = 32 * (warp & 3) + lane;    // TMEM lane / query row
        const float r2 = a.r2;
        const int Kout = a.K;
        uint32_t* sv_slot = Sv + warp * kTcSurvCap;
        uint8_t* sv_row = reinterpret_cast<uint8_t*>(Sv + (kTcEpi / 32) * kTcSurvCap) + warp * kTcSurvCap;
        unsigned long long n_surv = 0, n_acc = 0;

        for (uint32_t par = 0;; par ^= 1u) {
            __syncthreads();   // the task is ready
            const TcTask& ct = s_task[par];
            if (ct.done) break;
            const Task tk = ct.t;
            const int nch = ct.nch;
            const EventHdr& h = a.ev[tk.ev];
            int32_t* counts = a.counts ? a.counts : h.counts;
            int32_t* oidx = a.counts ? a.idx : h.idx;
            float* od2 = a.counts ? a.dist2 : h.dist2;
            const int qs = (tk.qslot & ~7) + row;
            const bool active = qs >= tk.qslot && qs < tk.qslot + tk.nq;
            const int qorig = active ? a.qperm[qs] : 0;
            if (!h.valid) {
                // grid built from non-finite input: empty rows (frnn_sync reports it)
                if (active) {
                    for (int e = 0; e < Kout && !a.csr; ++e) {
                        oidx[(int64_t)qorig * Kout + e] = -1;
                        od2[(int64_t)qorig * Kout + e] = INFINITY;
                    }
                    counts[qorig] = 0;
                    if (a.degree) a.degree[qorig] = 0;
                }
                continue;
            }
            // this thread's query: float32 coordinates (shared: the recheck
            // reads them from any lane)
            if (half == 0) {
                const float4* q4 = reinterpret_cast<const float4*>(a.qpts + (int64_t)(active ? qs : 0) * DP);
#pragma unroll
                for (int k4 = 0; k4 < DP / 4; ++k4) reinterpret_cast<float4*>(Qs + row * DP)[k4] = __ldg(q4 + k4);
                s_cnt[row] = 0;
            }
            const float tx = active ? __fmul_rd(0.5f, __fsub_rd(a.qn[qs], ct.theta)) : INFINITY;
            asm volatile("bar.sync 1, %0;" ::"n"(kTcEpi) : "memory");

            const int self_slot = a.self ? qs : -1;
            int fill = 0;   // survivors waiting for the recheck
            // recheck m entries from place p on, one per lane: the exact contract
            // on the float32 rows (the candidate's from L2)
            auto recheck = [&](int p, int m) {
                __syncwarp();
                if (lane < m) {
                    const int r = sv_row[p + lane], cs = (int)sv_slot[p + lane];
                    const float4* f4 = reinterpret_cast<const float4*>(a.rpts + (int64_t)cs * DP);
                    const float* qv = Qs + r * DP;
                    float f[DP];
#pragma unroll
                    for (int k4 = 0; k4 < DP / 4; ++k4) {
                        const float4 x = __ldg(f4 + k4);
                        f[4 * k4] = x.x;
                        f[4 * k4 + 1] = x.y;
                        f[4 * k4 + 2] = x.z;
                        f[4 * k4 + 3] = x.w;
                    }
                    const int32_t orig = __ldg(a.rperm + cs);
                    float sd = 0.f;
#pragma unroll
                    for (int k = 0; k < D; ++k) {
                        const float d = __fsub_rn(qv[k], f[k]);
                        sd = __fadd_rn(sd, __fmul_rn(d, d));
                    }
                    if (sd <= r2) {
                        ++n_acc;
                        const int pos = atomicAdd(&s_cnt[r], 1);
                        if (pos < kTcList) {
                            Ld[pos * kTcLStr + r] = sd;
                            Li[pos * kTcLStr + r] = orig;
                        }
                    }
                }
                __syncwarp();
            };
            // survivors of 64 columns starting at slot c0: each
            // lane appends its own, behind those of the lanes before it
            auto collect = [&](uint64_t mask, int c0) {
                while (__any_sync(kFull, mask != 0)) {
                    const int mine = __popcll(mask);
                    int pos = mine;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int v = __shfl_up_sync(kFull, pos, o);
                        if (lane >= o) pos += v;
                    }
                    const int total = __shfl_sync(kFull, pos, 31);
                    pos += fill - mine;
                    // (what finds no place stays in the mask for the next round)
                    while (mask && pos < kTcSurvCap) {
                        const int j = __ffsll((long long)mask) - 1;
                        mask &= mask - 1u;
                        sv_slot[pos] = (uint32_t)(c0 + j);
                        sv_row[pos] = (uint8_t)row;
                        ++pos;
                    }
                    const int got = min(total, kTcSurvCap - fill);
                    fill += got;
                    n_surv += (lane == 0) ? got : 0;
                    while (fill >= 32) {
                        fill -= 32;
                        recheck(fill, 32);
                    }
                }
            };
            // this warp's chunks: those of its accumulator
            for (int c = (int)((g0 ^ (uint32_t)half) & 1u); c < nch; c += kTcAcc) {
                const uint32_t g = g0 + c;
                if (!aborted()) {
                    if (!mbar_wait_bounded(&bar_mma[half], (g / kTcAcc) & 1u)) abort_now();
                }
                __syncwarp();
                tc_fence_after();
                uint64_t masks[2] = {0, 0};
                int start = 0;
                if (!__shfl_sync(0xffffffffu, aborted(), 0)) {
                    const int4 ci = s_chunk[half];   // (start, n, lo, hi)
                    const uint32_t tbase =
                        taddr + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)half * kTcN;
                    start = ci.x;
#pragma unroll 4
                    for (int gr = 0; gr < kTcN / 32; ++gr) {
                        if (32 * gr < ci.y) {   // n: a multiple of 32
                            uint32_t rv[32];
                            __syncwarp();
                            tmem_ld32_nowait(tbase + 32 * gr, rv);
                            tmem_wait_ld(rv);
                            // maxima of the four octets of columns, then of all 32
                            float oct[4];
#pragma unroll
                            for (int o = 0; o < 4; ++o) {
                                const auto v = [&](int j) { return __uint_as_float(rv[8 * o + j]); };
                                oct[o] = fmax3(fmax3(v(0), v(1), v(2)), fmax3(v(3), v(4), v(5)),
                                               fmaxf(v(6), v(7)));
                            }
                            const float mx = fmaxf(fmax3(oct[0], oct[1], oct[2]), oct[3]);
                            if (__any_sync(0xffffffffu, mx >= tx)) {
                                // columns of this group inside the chunk's own row range
                                const int c0 = start + 32 * gr;
                                const int jlo = max(ci.z - c0, 0), jhi = min(ci.w - c0, 32);
                                uint32_t valid =
                                    jhi > jlo ? (((jhi - jlo) == 32 ? 0xffffffffu
                                                                    : ((1u << (jhi - jlo)) - 1u))
                                                 << jlo)
                                              : 0u;
                                if ((unsigned)(self_slot - c0) < 32u) valid &= ~(1u << (self_slot - c0));
                                uint32_t mask = 0;
#pragma unroll
                                for (int o = 0; o < 4; ++o) {
                                    // (most octets hold no survivor of any lane)
                                    if (__any_sync(0xffffffffu, oct[o] >= tx)) {
#pragma unroll
                                        for (int j = 0; j < 8; ++j)
                                            if (__uint_as_float(rv[8 * o + j]) >= tx) mask |= 1u << (8 * o + j);
                                    }
                                }
                                {
                                    const uint64_t mv = (uint64_t)(mask & valid) << (32 * (gr & 1));
                                    if (gr < 2) masks[0] |= mv; else masks[1] |= mv;
                                }
                            }
                        }
                    }
                }
                // the accumulator goes back before the survivors are looked at:
                // they lie close together (16 of 100 groups hold them, 16 each),
                // and a warp that has some no longer holds up the others
                tc_fence_before();
                mbar_arrive(&bar_acc[half]);
#pragma unroll 1
                for (int hf = 0; hf < 2; ++hf) collect(hf ? masks[1] : masks[0], start + 64 * hf);
            }
            recheck(0, fill);
            g0 += nch;
            asm volatile("bar.sync 1, %0;" ::"n"(kTcEpi) : "memory");   // lists complete

            const int cnt = s_cnt[row];
            const bool spill = active && cnt > kTcList;
            if (half == 0) {
                if (active && !spill) counts[qorig] = min(cnt, Kout);
                if (active && spill && a.csr) counts[qorig] = kCsrSpill;   // counted by the selection kernel
                if (active && !spill && a.degree) a.degree[qorig] = cnt;
                if (spill) {
                    // longer than the list: the exact selection kernel finishes this row
                    const int pos = atomicAdd(a.ovf_count, 1);
                    if (pos < a.ovf_cap) {
                        a.ovf[pos].qslot = qs;
                        a.ovf[pos].ev = tk.ev;
                    } else {
                        atomicOr(a.status, kStatusCapacity);
                    }
                }
            }
            // each epilogue warp sorts 16 of the 128 rows and writes them
            {
                const int n = __shfl_sync(kFull, active && !spill ? cnt : 0, 16 * half + (lane & 15));
                const unsigned most = __reduce_max_sync(kFull, (unsigned)n);
                const int r0 = 32 * (warp & 3) + 16 * half;
                if (most > 16) {
                    sort_columns<16>(Ld, Li, r0, n);
                } else if (most > 1) {
                    sort_columns<8>(Ld, Li, r0, n);
                }
            }
            const unsigned skip = __ballot_sync(0xffffffffu, !active || spill);   // rows 32(w%4)..
            const int rstride = a.csr ? kCsrStageW : Kout;   // compact: staging row, no padding
            // rows of whole, aligned 16-byte pieces (a compact row's last one
            // may run past its entries, not past its staging row)
            const bool vec = (rstride & 3) == 0 &&
                             ((reinterpret_cast<uintptr_t>(oidx) | reinterpret_cast<uintptr_t>(od2)) & 15) == 0;
            for (int qq = 0; qq < 16; ++qq) {
                const int ql = 16 * half + qq;                 // lane of this row in the warp
                if (skip & (1u << ql)) continue;
                const int r = 32 * (warp & 3) + ql;
                const int c = min(__shfl_sync(0xffffffffu, cnt, ql), Kout);
                const int qo = __shfl_sync(0xffffffffu, qorig, ql);
                const int w = a.csr ? c : Kout;
                int32_t* irow = oidx + (int64_t)qo * rstride;
                float* drow = od2 + (int64_t)qo * rstride;
                if (vec) {
                    for (int e = 4 * lane; e < w; e += 128) {
                        int4 iv = make_int4(-1, -1, -1, -1);
                        float4 dv = make_float4(INFINITY, INFINITY, INFINITY, INFINITY);
                        if (e < c) {
                            iv.x = Li[e * kTcLStr + r];
                            dv.x = Ld[e * kTcLStr + r];
                        }
                        if (e + 1 < c) {
                            iv.y = Li[(e + 1) * kTcLStr + r];
                            dv.y = Ld[(e + 1) * kTcLStr + r];
                        }
                        if (e + 2 < c) {
                            iv.z = Li[(e + 2) * kTcLStr + r];
                            dv.z = Ld[(e + 2) * kTcLStr + r];
                        }
                        if (e + 3 < c) {
                            iv.w = Li[(e + 3) * kTcLStr + r];
                            dv.w = Ld[(e + 3) * kTcLStr + r];
                        }
                        *reinterpret_cast<int4*>(irow + e) = iv;
                        *reinterpret_cast<float4*>(drow + e) = dv;
                    }
                } else {
                    for (int e = lane; e < w; e += 32) {
                        const bool real = e < c;
                        irow[e] = real ? Li[e * kTcLStr + r] : -1;
                        drow[e] = real ? Ld[e * kTcLStr + r] : INFINITY;
                    }
                }
            }
        }
        if (a.stat_survivors) {
            atomicAdd(a.stat_survivors, n_surv);
            atomicAdd(a.stat_accepted, n_acc);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr),
                     "n"(kTcCols)
                     : "memory");
    }
}

// ------------------------------------------------------------- host

void tc_free(GridBufs& g) {
    if (g.tc_base) cudaFree(g.tc_base);
    g.tc_base = nullptr;
    g.tc_bytes = 0;
    g.tc_cap_rows = g.tc_cap_tasks = g.tc_cap_E = g.tc_cap_L = 0;
    g.tc_rtask = nullptr;
    g.rtask = nullptr;
    g.tc_ready = false;
}

static size_t al256(size_t x) { return (x + 255) / 256 * 256; }

// Allocate (or keep) the operand buffers of a point set; enqueues nothing but
// the one-time zeroing of a fresh allocation (on the legacy default stream,
// synchronised, so it may run before a capture begins).
frnn_status tc_reserve(GridBufs& g, std::string& err) {
    const int K = tc_k_for(g.D);
    const int64_t rows = (g.n_total + 7) / 8 * 8 + kTcRowPad;
    // a tile never spans two rows of cells and only rows holding a point open
    // one: a row of c queries takes at most floor(c / 128) + 1 tiles, or + 2
    // when its start alignment (up to 7 slots) carries it past a multiple of
    // 128, which needs c >= 121; so per event at most n / 128 + rows + n / 121
    int64_t tcap = 0;
    for (int e = 0; e < g.E; ++e)
        tcap += g.h_hdr[e].n / kTcM + g.h_hdr[e].n / 64 +
                std::min<int64_t>(g.h_hdr[e].cell_cap, g.h_hdr[e].n) + 2;
    if (tcap >= INT32_MAX) {
        err = "too many tensor-core tiles for one call";
        return FRNN_ERR_INVALID_ARG;
    }
    if (g.tc_base && g.tc_K == K && g.tc_cap_rows >= rows && g.tc_cap_tasks >= tcap &&
        g.tc_cap_E >= g.E && g.tc_cap_L >= g.L) {
        g.rtask = g.tc_rtask;
        return FRNN_OK;
    }
    tc_free(g);
    const size_t bA = al256(sizeof(uint16_t) * rows * K);
    const size_t bn = al256(sizeof(float) * rows);
    const size_t bnu = al256(sizeof(int32_t) * std::max(g.E, 1));
    const size_t bt = al256(sizeof(Task) * tcap);
    const size_t brt = al256(sizeof(int32_t) * std::max<int64_t>(g.L, 1));
    void* base = nullptr;
    cudaError_t ce = cudaMalloc(&base, 2 * bA + bn + bnu + bt + brt + 256);
    if (ce != cudaSuccess) {
        cudaGetLastError();
        err = "cudaMalloc of tensor-core operands failed";
        return FRNN_ERR_OUT_OF_MEMORY;
    }
    char* b = static_cast<char*>(base);
    g.tc_base = base;
    g.tc_bytes = 2 * bA + bn + bnu + bt + brt + 256;
    g.tcA = reinterpret_cast<uint16_t*>(b);
    g.tcB = reinterpret_cast<uint16_t*>(b + bA);
    g.tcn = reinterpret_cast<float*>(b + 2 * bA);
    g.tcnu = reinterpret_cast<int32_t*>(b + 2 * bA + bn);
    g.tc_tasks = reinterpret_cast<Task*>(b + 2 * bA + bn + bnu);
    g.tc_rtask = reinterpret_cast<int32_t*>(b + 2 * bA + bn + bnu + bt);
    g.rtask = g.tc_rtask;   // scratch of the task builder (per row of cells)
    g.tc_cap_L = g.L;
    g.tc_cap_rows = rows;
    g.tc_cap_tasks = tcap;
    g.tc_cap_E = g.E;
    g.tc_K = K;
    // rows past the last slot stay zero (chunks may read them).  Waited for: the
    // call returns before the device has run it, and a context's stream that
    // does not synchronise with the default one would write the operands first
    ce = cudaMemset(base, 0, 2 * bA + bn);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(nullptr);
    if (ce != cudaSuccess) {
        cudaGetLastError();
        err = "zeroing tensor-core operands failed";
        return FRNN_ERR_CUDA;
    }
    return FRNN_OK;
}

frnn_status tc_prepare(GridBufs& g, const GridBufs& center_src, int32_t* d_status,
                       cudaStream_t st, std::string& err, int path_filter, int64_t i0,
                       int64_t i1) {
    frnn_status s0 = tc_reserve(g, err);
    if (s0 != FRNN_OK) return s0;
    const int K = tc_k_for(g.D);
    cudaMemsetAsync(g.tcnu, 0, sizeof(int32_t) * g.E, st);   // ordered(0.0f) == 0
    if (g.n_total > 0) {
        const unsigned nb = (unsigned)ceil_div(g.n_total, 128);
        switch (g.D) {
#define FRNN_PREP(d)                                                                         \
    case d:                                                                                  \
        k_tc_prep<d><<<nb, 128, 0, st>>>(g.hdr, center_src.hdr, g.E, g.n_total, g.pts, g.tcA, \
                                         g.tcB, g.tcn, g.tcnu);                              \
        break;
            FRNN_PREP(8) FRNN_PREP(9) FRNN_PREP(10) FRNN_PREP(11) FRNN_PREP(12)
            FRNN_PREP(13) FRNN_PREP(14) FRNN_PREP(15) FRNN_PREP(16)
#undef FRNN_PREP
            default:
                err = "tensor-core path needs 8 <= D <= 16";
                return FRNN_ERR_UNSUPPORTED;
        }
        (void)K;
    }
    enqueue_tasks(g, kTcM, 8, g.tc_tasks, g.tc_cap_tasks, g.scalars + kScTcTasks, d_status, st,
                  path_filter, i0, i1);
    cudaError_t ce = cudaGetLastError();
    if (ce != cudaSuccess) {
        err = std::string("tensor-core prep launch failed: ") + cudaGetErrorString(ce);
        return FRNN_ERR_CUDA;
    }
    g.tc_ready = true;
    return FRNN_OK;
}

frnn_status enqueue_tc_query(const QueryLaunch& q, cudaStream_t st, std::string& err) {
    const GridBufs& qs = *q.qset;
    const GridBufs& rs = *q.rset;
    const int D = rs.D;
    const int K = tc_k_for(D);
    TcArgs a{};
    a.ev = rs.hdr;
    a.tasks = qs.tc_tasks;
    a.ntasks = qs.scalars + kScTcTasks;
    a.tcA = qs.tcA;
    a.tcB = rs.tcB;
    a.qn = qs.tcn;
    a.nu_q = qs.tcnu;
    a.nu_r = rs.tcnu;
    a.qpts = qs.pts;
    a.qperm = qs.perm;
    a.qcell = qs.cell;
    a.rpts = rs.pts;
    a.rperm = rs.perm;
    a.cstart = rs.cstart;
    a.counts = q.counts;
    a.idx = q.idx;
    a.dist2 = q.dist2;
    a.r2 = q.r2;
    a.K = q.K;
    a.self = q.self;
    a.D = D;
    a.task_counter = qs.scalars + kScTcCounter;
    a.status = q.d_status;
    a.ovf = qs.ovf;
    a.ovf_count = qs.scalars + kScOvfCount;
    a.ovf_cap = (int32_t)std::max<int64_t>(qs.n_total, 1);
    a.path_filter = q.path_filter;
    a.stat_survivors = q.tc_stats;
    a.stat_accepted = q.tc_stats ? q.tc_stats + 1 : nullptr;
    a.csr = q.csr;
    a.degree = q.degree;
    cudaMemsetAsync(qs.scalars + kScOvfCount, 0, sizeof(int32_t), st);
    cudaMemsetAsync(qs.scalars + kScTcCounter, 0, sizeof(int32_t), st);
    if (q.kev[0]) cudaEventRecord(q.kev[0], st);
    cudaError_t ce = cudaSuccess;
    auto launch = [&](auto kern, size_t smem) {
        ce = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (ce == cudaSuccess) {
            kern<<<2 * q.num_sms, kTcThreads, smem, st>>>(a);
            ce = cudaGetLastError();
        }
    };
    switch (D) {
        case 8: launch(k_tc_query<8>, tc_smem_bytes(8)); break;
        case 9: launch(k_tc_query<9>, tc_smem_bytes(9)); break;
        case 10: launch(k_tc_query<10>, tc_smem_bytes(10)); break;
        case 11: launch(k_tc_query<11>, tc_smem_bytes(11)); break;
        case 12: launch(k_tc_query<12>, tc_smem_bytes(12)); break;
        case 13: launch(k_tc_query<13>, tc_smem_bytes(13)); break;
        case 14: launch(k_tc_query<14>, tc_smem_bytes(14)); break;
        case 15: launch(k_tc_query<15>, tc_smem_bytes(15)); break;
        case 16: launch(k_tc_query<16>, tc_smem_bytes(16)); break;
        default:
            err = "tensor-core path needs 8 <= D <= 16";
            return FRNN_ERR_UNSUPPORTED;
    }
    if (ce != cudaSuccess) {
        err = std::string("tensor-core query launch failed: ") + cudaGetErrorString(ce);
        return FRNN_ERR_CUDA;
    }
    if (q.kev[1]) cudaEventRecord(q.kev[1], st);
    // rows whose lists overflowed: exact selection kernel
    QueryArgs o{};
    o.ev = rs.hdr;
    o.qpts = qs.pts;
    o.qperm = qs.perm;
    o.qcell = qs.cell;
    o.rpts = rs.pts;
    o.rperm = rs.perm;
    o.cstart = rs.cstart;
    o.counts = q.counts;
    o.idx = q.idx;
    o.dist2 = q.dist2;
    o.r2 = q.r2;
    o.K = q.K;
    o.self = q.self;
    o.D = D;
    o.status = q.d_status;
    o.ovf = qs.ovf;
    o.ovf_count = qs.scalars + kScOvfCount;
    o.ovf_cap = a.ovf_cap;
    // the selection clears the list, as after a grid scan (a compact count
    // pass leaves it to the fill, or to the next query of this point set)
    o.ovf_done = qs.scalars + kScOvfDone;
    o.task_counter = qs.scalars + kScTcCounter;
    o.reset_ovf = q.ovf_mode == 1 ? 0 : 1;
    qs.ovf_stale = q.ovf_mode == 1;
    o.path_filter = -1;   // the list only holds rows this launch queued
    o.csr = q.csr;
    o.ovf_mode = q.ovf_mode;
    o.degree = q.degree;
    o.row_off = q.row_off;
    return enqueue_overflow(o, q.num_sms, st, err);
}

}  // namespace frnn
