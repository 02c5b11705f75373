// build.cu — uniform-grid build: bounding boxes, cell parameters, cell ids,
// counting sort into cell-sorted padded rows, and the warp-task list.
//
// The uniform grid / cell list is the method of the original FRNN the paper
// starts from (Sec. 2: uniform-grid kernel, spacing chosen so that r is an
// integer multiple of it).  Here at most six coordinates are gridded; the cell
// assignment is "roundoff-safe" (Table 1): it provably never separates two
// points the float32 contract accepts by more than m cells per axis (proof at
// event_params below).
//
// Steps, all on the device, no host synchronisation:
//   k_bbox      zero the cell counts; per-event per-axis min / max (+ non-finite
//               flag), float4 staged; the event's last block to finish writes the
//               tables of a one-event build (passed by value) and derives the
//               grid parameters: gridded axes, cell edge, cells per axis
//               (k_begin_foreign instead when the parameters are another grid's)
//   k_cellid    cell id of every point and its rank inside the cell (atomics)
//   k_cells_*   exclusive prefix scan of the used counts -> cell starts
//   k_scatter   slot -> original index, slot -> cell, and the point's row of
//               DP floats at its slot (cell-sorted coordinates)
// Sets of up to 32,768 points are built by one launch instead (k_build_small).
// (row tasks and tensor-core tiles are listed at query time: k_rowtasks, a
// scan, k_emit)
#include <cooperative_groups.h>

#include <algorithm>
#include <climits>
#include <cmath>

#include "frnn_host.h"

namespace frnn {

// ------------------------------------------------------------------ helpers

// An entry of a box copy before any point.
__device__ __forceinline__ int32_t empty_box_entry(int k) {
    return k < 16 ? INT_MAX : (k < 32 ? INT_MIN : 0);   // minima, maxima; flag, block counter
}

// The grid parameters of src, by a whole block (or more than kMaxD threads).
__device__ __forceinline__ void copy_params(EventHdr& dst, const EventHdr& src) {
    const int t = threadIdx.x;
    if (t == 0) {
        dst.naxes = src.naxes;
        dst.m = src.m;
        dst.valid = src.valid;
        dst.inv_h = src.inv_h;
        dst.ncells = src.ncells;
        dst.half = src.half;
    }
    if (t < kHdrAxes) {
        dst.axes[t] = src.axes[t];
        dst.dims[t] = src.dims[t];
        dst.fdims[t] = src.fdims[t];
        dst.mag[t] = src.mag[t];
        dst.lo[t] = src.lo[t];
        dst.hi[t] = src.hi[t];
    }
    if (t < kMaxD) dst.ctr[t] = src.ctr[t];
}

// Entry of each event's box copy 0 that counts its finished k_bbox blocks.
constexpr int kBBoxDone = 33;
static_assert(kBBoxDone >= 33 && kBBoxDone < kBBoxStride, "after the minima, maxima and flag");

// The tables of a one-event build (header, block starts, cell offsets), passed
// to the first kernel by value instead of being copied from the host.
struct OneEventTables {
    EventHdr hdr;
    int64_t cell_end;   // cell_off[1]
    int32_t nblk;       // blk_start[1]
    int32_t set;        // 0: the tables are already on the device
};

// A one-event build's input, passed by value to the kernels that stage it:
// they stage their block's points before waiting for the previous kernel of
// the chain (no kernel of the chain writes the caller's points, and the
// header that would locate them is written by k_bbox in this case).  The work
// that wrote the points is complete by then, although it may itself have let
// its successors start early: the chain's first kernel waits for it and only
// then triggers, so nothing later in the chain starts before.  (Triggering
// first and waiting in k_cellid instead: 0.5 to 1 us slower a chain.  Reading
// the points before any wait, which is wrong after such work, was 0.5 to 1 us
// faster a build: 300k x 8 138.7 against 139.7 us, 4096 x 3 20.4 against 21.)
struct EarlyPts {
    const float* refs;
    int64_t n;
    int32_t set;   // 0: locate the points through the tables, after the wait
};

// Stage this block's input rows before the wait when the build is one event.
__device__ __forceinline__ bool stage_early(float* sm, const EarlyPts& ep, int D, bool pad);

__device__ __forceinline__ int find_event(const int32_t* starts, int E, int b) {
    // largest e with starts[e] <= b
    int lo = 0, hi = E - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (starts[mid] <= b) lo = mid; else hi = mid - 1;
    }
    return lo;
}

__device__ __forceinline__ int find_event64(const int64_t* starts, int E, int64_t i) {
    int lo = 0, hi = E - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (starts[mid] <= i) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Staged point rows in shared memory: float j of the block's rows sits at
// j + j / 32 when D is a multiple of 4 (one padding word per 32), else at j,
// so that a warp reading coordinate k of 32 consecutive rows (stride D) hits
// distinct banks for D = 4, 8, 16 and at most two per bank otherwise.
__device__ __forceinline__ int stage_slot(int j, bool pad) { return pad ? j + (j >> 5) : j; }
__host__ __device__ constexpr size_t staged_floats(int D) {
    return (size_t)kBuildPtsPerBlock * D + (size_t)kBuildPtsPerBlock * D / 32 + 1;
}

// Row i of the staged rows, indexed by coordinate.
struct StagedRow {
    const float* sm;
    int j0;
    bool pad;
    __device__ __forceinline__ float operator[](int k) const { return sm[stage_slot(j0 + k, pad)]; }
};

// One cell-sorted row of DP floats (zero padding), written in 32-byte or
// 16-byte pieces.
__device__ __forceinline__ void write_row(float* dst, const StagedRow& src, int D, int DP) {
    auto at = [&](int k) { return k < D ? src[k] : 0.f; };
    if ((DP & 7) == 0) {
        for (int k = 0; k < DP; k += 8)
            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst + k), "f"(at(k)),
                         "f"(at(k + 1)), "f"(at(k + 2)), "f"(at(k + 3)), "f"(at(k + 4)), "f"(at(k + 5)),
                         "f"(at(k + 6)), "f"(at(k + 7))
                         : "memory");
    } else {
        for (int k = 0; k < DP; k += 4)
            *reinterpret_cast<float4*>(dst + k) = make_float4(at(k), at(k + 1), at(k + 2), at(k + 3));
    }
}

// Stage nf consecutive floats of a row-major point array into shared memory
// (at stage_slot), using 16-byte vector loads for the aligned body.
__device__ __forceinline__ void stage_floats(float* sm, const float* src, int nf, bool pad) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(src);
    int head = (int)(((16u - (uint32_t)(a & 15u)) & 15u) >> 2);
    if (a & 3u) head = nf;   // not even 4-byte aligned: scalar path (cannot happen for float*)
    head = min(head, nf);
    for (int i = threadIdx.x; i < head; i += blockDim.x) sm[stage_slot(i, pad)] = __ldg(src + i);
    const int n4 = (nf - head) >> 2;
    const float4* s4 = reinterpret_cast<const float4*>(src + head);
    constexpr int kAhead = 3;   // loads in flight per thread
    for (int i0 = threadIdx.x; i0 < n4; i0 += kAhead * blockDim.x) {
        float4 v[kAhead];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int i = i0 + u * blockDim.x;
            v[u] = i < n4 ? __ldg(s4 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int i = i0 + u * blockDim.x;
            const int j = head + 4 * i;
            if (i < n4) {
                sm[stage_slot(j, pad)] = v[u].x;
                sm[stage_slot(j + 1, pad)] = v[u].y;
                sm[stage_slot(j + 2, pad)] = v[u].z;
                sm[stage_slot(j + 3, pad)] = v[u].w;
            }
        }
    }
    for (int i = head + 4 * n4 + threadIdx.x; i < nf; i += blockDim.x)
        sm[stage_slot(i, pad)] = __ldg(src + i);
}

__device__ __forceinline__ bool stage_early(float* sm, const EarlyPts& ep, int D, bool pad) {
    if (!ep.set) return false;
    const int64_t p0 = (int64_t)blockIdx.x * kBuildPtsPerBlock;
    const int np = (int)min((int64_t)kBuildPtsPerBlock, ep.n - p0);
    if (np > 0) stage_floats(sm, ep.refs + p0 * D, np * D, pad);
    return true;
}

// Cell coordinate along one gridded axis: floor(fl(fl(x' - lo) * inv_h))
// clamped to [0, dim - 1], with x' = x clamped to [lo, hi].  Every kernel that
// bins points (references and queries) uses exactly this function.
__device__ __forceinline__ int cell_coord(float x, float lo, float hi, float inv_h, int dim) {
    float xc = fminf(fmaxf(x, lo), hi);
    float g = __fmul_rn(__fsub_rn(xc, lo), inv_h);
    int c = __float2int_rd(g);
    return min(max(c, 0), dim - 1);
}

// A point's `cell` entry: its cell id (of a grid of half cells: the stored
// cell id and the half bits).
template <class Row>
__device__ __forceinline__ int point_cell(const Row& p, const EventHdr& h) {
    int c = 0, stride = 1, bits = 0;
#pragma unroll
    for (int a = 0; a < kHdrAxes; ++a) {
        if (a < h.naxes) {
            int x = cell_coord(p[h.axes[a]], h.lo[a], h.hi[a], h.inv_h, h.fdims[a]);
            if (a > 0 && h.half) {
                bits |= (x & 1) << (a - 1);
                x >>= 1;
            }
            c += x * stride;
            stride *= h.dims[a];
        }
    }
    return h.half ? (c << kHalfBits) | bits : c;
}

// ------------------------------------------------------------------ kernels

// Zero the counters and this block's share of the cell array (n4 quads).
__device__ __forceinline__ void zero_share(int32_t* counts, int64_t n4, int32_t* scalars) {
    int4* c4 = reinterpret_cast<int4*>(counts);
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n4; j += (int64_t)gridDim.x * blockDim.x)
        c4[j] = make_int4(0, 0, 0, 0);
    if (blockIdx.x == 0 && threadIdx.x < kScalars) scalars[threadIdx.x] = 0;
}

// One header by a whole block, word by word.
__device__ __forceinline__ void copy_header(EventHdr* dst, const EventHdr& src) {
    for (int i = threadIdx.x; i < (int)(sizeof(EventHdr) / 4); i += blockDim.x)
        reinterpret_cast<int32_t*>(dst)[i] = reinterpret_cast<const int32_t*>(&src)[i];
}

// The boxes of E events before any point (new buffers; afterwards the
// parameter step leaves them like this).
__global__ void k_box_reset(int32_t* bbox, int E) {
    pdl_trigger();
    pdl_wait();
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < E * kBBoxCopies * kBBoxStride) bbox[j] = empty_box_entry(j % kBBoxStride);
}

__device__ void event_params(EventHdr* hdr, int e, int D, int32_t* bbox, float r, int m,
                             int axes_mode, int naxes_req);

// Per-event bounding boxes, and the zeroing of the cell counts.  One CTA takes
// `sub` build blocks (256 points each); the ones that belong to one event are
// one run of floats, read as 16-byte pieces, four in flight a thread.  The
// threads that read (box_threads(D) of 256) stride by a multiple of D, so a
// thread meets the same four coordinates every time and keeps their extremes
// in registers; once per event the CTA's extremes are merged into one of
// kBBoxCopies copies of the event's box (copy = block mod kBBoxCopies), so that
// no address takes more than a few atomics.  The event's last block to finish
// (a counter beside copy 0, taken after a memory fence) combines the copies and
// derives the grid parameters; the zeroing of the other blocks runs beside that
// chain.  `sub` build blocks a CTA: as many as make one wave of kBoxWave CTAs,
// at most eight (a wave of 608, 304 or 1216 CTAs, build + query at 300k x 8:
// 138.7, 140.8, 142.1 us).  What bounds it is the chain from the first load to
// the derived parameters and, from a million points on, memory.  With the rows
// staged in shared memory, build block by build block: 300k x 8 141.4 -> 138.7
// us, 1 M x 3 215.3 -> 206.8, 500k x 12 335 -> 328, 16 events x 8 1551 -> 1513.
constexpr int kBoxWave = 608;
constexpr int kBoxMost = 8;

// Threads of 256 that read a run of rows of D floats in 16-byte pieces: as many
// as make 4 x threads a multiple of D.
__host__ __device__ constexpr int box_threads(int D) {
    const int period = D % 4 == 0 ? D / 4 : (D % 2 == 0 ? D / 2 : D);
    return kBuildPtsPerBlock - kBuildPtsPerBlock % period;
}

__global__ void __launch_bounds__(kBuildPtsPerBlock, 4) k_bbox(EventHdr* hdr, int32_t* blk_start, int64_t* cell_off,
                                                            int E, int nblk, int sub, int D, int32_t* bbox,
                                                            int32_t* status, float r, int m, int axes_mode, int naxes_req,
                                                            int32_t* counts, int64_t L, int32_t* scalars,
                                                            OneEventTables t1) {
    // the first kernel of a chain: the caller's work on the stream may have let
    // it start early, and wrote the points (see EarlyPts)
    pdl_wait();
    pdl_trigger();
    __shared__ int32_t red_mn[4 * kBuildPtsPerBlock], red_mx[4 * kBuildPtsPerBlock];
    __shared__ int red_bad, s_last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int T = box_threads(D);
    bool zeroed = false;
    const int b1 = min((int)(blockIdx.x + 1) * sub, nblk);
    int b = blockIdx.x * sub;
    while (b < b1) {
        const int e = t1.set ? 0 : find_event(blk_start, E, b);
        const int b_end = t1.set || e == E - 1 ? b1 : min(b1, blk_start[e + 1]);
        const float* refs = t1.set ? t1.hdr.refs : hdr[e].refs;
        const int64_t n = t1.set ? t1.hdr.n : hdr[e].n;
        const int64_t p0 = (int64_t)(t1.set ? b : b - blk_start[e]) * kBuildPtsPerBlock;
        const int np = (int)max((int64_t)0, min((int64_t)(b_end - b) * kBuildPtsPerBlock, n - p0));
        // thread t < T: elements head + 4 (t + i T) + c of the run; the head
        // and tail short of 16 bytes (at most three each) go to threads 0.. and
        // 32.. one by one
        const float* src = refs + p0 * D;
        const int nf = np * D;
        const int head = min(nf, (int)((16u - (uint32_t)(reinterpret_cast<uintptr_t>(src) & 15u)) & 15u) >> 2);
        const int n4 = (nf - head) >> 2;
        int32_t mn[4], mx[4];   // ordered ints
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            mn[c] = INT_MAX;
            mx[c] = INT_MIN;
        }
        bool bad = false;
        if ((int)threadIdx.x < T) {
            const float4* s4 = reinterpret_cast<const float4*>(src + head);
            constexpr int kAhead = 4;   // loads in flight per thread
            for (int i0 = threadIdx.x; i0 < n4; i0 += kAhead * T) {
                float4 v[kAhead];
#pragma unroll
                for (int u = 0; u < kAhead; ++u)   // (past the end: the run's piece at i0 again)
                    v[u] = __ldg(s4 + (i0 + u * T < n4 ? i0 + u * T : i0));
#pragma unroll
                for (int u = 0; u < kAhead; ++u) {
                    const float f[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        bad |= !isfinite(f[c]);
                        const int32_t x = float_to_ordered(f[c]);
                        mn[c] = min(mn[c], x);
                        mx[c] = max(mx[c], x);
                    }
                }
            }
        }
        int odd_at = -1;
        if ((int)threadIdx.x < head) odd_at = threadIdx.x;
        if (threadIdx.x >= 32 && (int)threadIdx.x - 32 < nf - head - 4 * n4) odd_at = head + 4 * n4 + (int)threadIdx.x - 32;
        const float odd = odd_at >= 0 ? __ldg(src + odd_at) : 0.f;
        bad |= !isfinite(odd);
        if (!zeroed) zero_share(counts, L / 4, scalars);
        zeroed = true;
        // merge
        if (threadIdx.x == 0) red_bad = 0;
        *reinterpret_cast<int4*>(red_mn + 4 * threadIdx.x) = make_int4(mn[0], mn[1], mn[2], mn[3]);
        *reinterpret_cast<int4*>(red_mx + 4 * threadIdx.x) = make_int4(mx[0], mx[1], mx[2], mx[3]);
        __syncthreads();
        int32_t* bb = bbox + ((int64_t)e * kBBoxCopies + (blockIdx.x % kBBoxCopies)) * kBBoxStride;
        for (int k = warp; k < D; k += kBuildPtsPerBlock / 32) {
            // entry q of the tables is an element of coordinate (head + q) % D
            int32_t lo = INT_MAX, hi = INT_MIN;
            for (int q = (k + 4 * D - head) % D + lane * D; q < 4 * T; q += 32 * D) {
                lo = min(lo, red_mn[q]);
                hi = max(hi, red_mx[q]);
            }
            lo = __reduce_min_sync(0xffffffffu, lo);
            hi = __reduce_max_sync(0xffffffffu, hi);
            if (lane == 0) {
                atomicMin(bb + k, lo);
                atomicMax(bb + 16 + k, hi);
            }
        }
        if (odd_at >= 0) {
            atomicMin(bb + odd_at % D, float_to_ordered(odd));
            atomicMax(bb + 16 + odd_at % D, float_to_ordered(odd));
        }
        if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(&red_bad, 1);
        __threadfence();   // this block's box updates before its count
        __syncthreads();
        if (threadIdx.x == 0) {
            if (red_bad) {
                atomicOr(bb + 32, 1);
                atomicOr(status, kStatusNonFinite);
                __threadfence();
            }
            const int total = t1.set ? t1.nblk : blk_start[e + 1] - blk_start[e];
            int32_t* done = bbox + (int64_t)e * kBBoxCopies * kBBoxStride + kBBoxDone;
            s_last = atomicAdd(done, b_end - b) == total - (b_end - b);
        }
        __syncthreads();
        if (s_last) {
            __threadfence();   // every other block's updates before the reads
            if (t1.set) {
                copy_header(hdr, t1.hdr);
                if (threadIdx.x == 0) {
                    blk_start[0] = 0;
                    blk_start[1] = t1.nblk;
                    cell_off[0] = 0;
                    cell_off[1] = t1.cell_end;
                }
                __syncthreads();
            }
            event_params(hdr, e, D, bbox, r, m, axes_mode, naxes_req);
        }
        __syncthreads();   // (the tables and s_last are written again)
        b = b_end;
    }
    if (!zeroed) zero_share(counts, L / 4, scalars);
}

// The start of a build with foreign parameters (a cross-set query's points,
// binned by the reference grid's header src): tables, parameters, zeroed counts.
__global__ void k_begin_foreign(OneEventTables t1, const EventHdr* src, EventHdr* hdr, int32_t* blk_start,
                                int64_t* cell_off, int32_t* counts, int32_t* scalars) {
    pdl_wait();      // (first of its chain: see EarlyPts)
    pdl_trigger();
    if (blockIdx.x == 0) {
        copy_header(hdr, t1.hdr);
        __syncthreads();
        copy_params(*hdr, *src);
        if (threadIdx.x == 0) {
            blk_start[0] = 0;
            blk_start[1] = t1.nblk;
            cell_off[0] = 0;
            cell_off[1] = t1.cell_end;
        }
    }
    // (t1.hdr.rowsort: used_entries of the finished header)
    const int used = (t1.hdr.rowsort ? src->ncells / src->dims[0] : src->ncells) + 1;
    const int64_t scanned = (int64_t)(used + kCellChunk - 1) / kCellChunk * kCellChunk;
    zero_share(counts, min(scanned, cell_entries(t1.hdr.cell_cap)) / 4, scalars);
}

// Grid parameters of one event (one CTA: its warps combine the box copies,
// then warp 0 derives the parameters, lane a handling gridded axis a).
//
// Roundoff-safe cell assignment (proof).  Let u = 2^-24.  If the contract
// accepts (x, y), every rounded square t_a = fl(fl(x_a - y_a)^2) is <= the
// final sum s (partial sums of non-negative terms never decrease under
// round-to-nearest) and s <= r2 = fl(r*r) <= r^2 (1 + u); with r2 normal this
// gives |fl(x_a - y_a)| <= r (1 + 2u) and |x_a - y_a| <= rho := r (1 + 2^-20).
// For lo <= x <= y <= hi the cell coordinate g(.) = fl(fl(. - lo) * inv_h) is
// monotone and g(y) - g(x) <= inv_h (rho + 2^-21 E) + 2^-148, E = hi - lo.  If
// that bound is < m, floor(g(y)) - floor(g(x)) <= m, and clamping to
// [0, dim-1] keeps it so; queries are clamped to [lo, hi] first, which only
// shrinks their distance to any reference.  So searching +-m cells per gridded
// axis finds every accepted pair.  The bound is evaluated in float32 with
// every operation rounded upward (rho, E and each step), which can only
// overestimate it: inv_h starts at fl_down(m / fl_up(r (1+2^-10))) and is
// lowered until the overestimate is below m - 2^-20, every axis has at most
// 1024 cells and the event's cell count fits its capacity.
static_assert(kBBoxCopies == 32, "one copy per lane when the copies are combined");

static_assert(kBuildPtsPerBlock == 256, "eight warps combine the box copies");
static_assert(kMaxD <= 32 && kHdrAxes <= 32, "one lane per coordinate");

// One candidate grid, held by warp 0: k gridded axes (the last k coordinates,
// or the k widest), cell multiple m, the cell edge fitted to the proof's
// condition, 1024 cells per axis and the event's cell budget, and the
// expected fraction of the event a query's neighbourhood covers if the
// points were spread evenly: the product over the gridded axes of
// min(1, (2m+1) cells / extent) (4 cells on the axes of a grid of half cells,
// whose budget counts stored cells).  The parameter step keeps the candidate
// with the smallest fraction; the choice never changes results.  Lane a < k
// holds gridded axis a (coordinate, cells, extremes); the other fields are
// the same on every lane.
struct GridFit {
    int naxes = 1, m = 1;
    int axis = 0, dim = 1, sdim = 1;   // sdim: stored cells
    float lo = 0.f, hi = 0.f;
    float inv_h = 0.f;
    int32_t ncells = 1;
    float frac = INFINITY;
    bool at_start = false;   // the starting cell edge fitted (no enlargement)
};

// lo_j, hi_j: the extremes of coordinate j on lane j < D.  once: no grid (an
// infinite fraction) where the starting cell edge does not fit.  Called by all
// lanes of a warp.
__device__ void grid_fit(GridFit& f, float lo_j, float hi_j, int D, int k, int m, int axes_mode,
                         float r, int64_t cap, bool valid, int max_rows, bool half, bool once = false) {
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const int la = lane & 7;   // the lane's axis (every eighth lane alike, for the products below)
    // product of an axis value over the axes, on every lane
    auto over_axes = [&](auto x) {
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) x *= __shfl_xor_sync(kAll, x, o);
        return x;
    };
    f.naxes = k;
    // neighbour rows, (2m+1)^(k-1): at most max_rows (the chunk kernel
    // enumerates kMaxNbrRows, 32 per round; the row-task kernel one per lane)
    int mm = max(m, 1);
    for (;;) {
        int rows = 1;
        for (int a = 1; a < k; ++a) rows *= 2 * mm + 1;
        if (rows <= max_rows || mm == 1) break;
        --mm;
    }
    f.m = mm;
    // the last k coordinates; a sixth axis (half cells) is the one before the
    // last five
    const int k5 = min(k, kMaxAxes);
    int ax = la < k5 ? D - k5 + la : (la < k ? D - 1 - la : 0);
    if (valid && axes_mode == 1 && D > k) {
        // the k widest coordinates (ties by lower index), in index order
        const float wj = __fsub_rn(hi_j, lo_j);
        int rank = 0;
        for (int i = 0; i < D; ++i) {
            const float wi = __shfl_sync(kAll, wj, i);
            if (wi > wj || (wi == wj && i < lane)) ++rank;
        }
        const unsigned sel = __ballot_sync(kAll, lane < D && rank < k);
        const int want_pos = k > kMaxAxes ? (la < kMaxAxes ? la + 1 : 0) : la;
        int cnt = 0;
        ax = 0;
        for (int j = 0; j < D; ++j) {
            if ((sel >> j) & 1u) {
                if (cnt == want_pos) ax = j;
                ++cnt;
            }
        }
    }
    const float lo = __shfl_sync(kAll, lo_j, ax);
    const float hi = __shfl_sync(kAll, hi_j, ax);
    f.axis = la < k ? ax : 0;
    f.lo = lo;
    f.hi = hi;
    if (!valid) {
        f.frac = 1.f;
        return;
    }
    // the cell coordinate of hi is floor(fl(ext * inv_h)): dim = that + 1
    const float ext = __fsub_rn(hi, lo);
    const float ext_up = __fsub_ru(hi, lo);
    const float rho_up = __fmul_ru(r, 1.0f + 0x1p-20f);
    const float need = (float)mm - 0x1p-20f;
    float ih = __fdiv_rd((float)mm, __fmul_ru(r, 1.0f + 0x1p-10f));
    int dim = 1, sdim = 1;
    int64_t cells = 1;
    bool fit = false;
    for (int it = 0; it < 4096; ++it) {
        bool ok = true;
        dim = 1;
        if (la < k) {
            const float c = floorf(__fmul_rn(ext, ih)) + 1.0f;
            if (!(c <= (float)kMaxDimsPerAxis)) ok = false;
            else dim = (int)c;
            const float bound =
                __fadd_ru(__fmul_ru(ih, __fadd_ru(rho_up, __fmul_ru(0x1p-21f, ext_up))), 0x1p-148f);
            if (!(bound < need)) ok = false;
        }
        sdim = half && la > 0 ? (dim + 1) >> 1 : dim;
        cells = over_axes((int64_t)sdim);   // (1 beyond the k axes; at most 1024^6)
        if (__all_sync(kAll, ok) && cells <= cap) {
            fit = true;
            f.at_start = it == 0;
            break;
        }
        if (once) return;   // (frac as it was: infinite)
        // too many cells: by the ratio the budget asks for (the dims' rounding
        // may need another step); a failed bound or axis limit: by a tenth
        float shrink = 0.9f;
        if (__all_sync(kAll, ok)) {
            shrink = exp2f(log2f((float)cap / (float)cells) / (float)k);
            shrink = fminf(fmaxf(shrink, 0.5f), 0.97f);
        }
        ih = __fmul_rd(ih, shrink);
        if (!(ih > 0.f)) break;
    }
    if (!fit) {   // one cell is always safe
        ih = 0.f;
        dim = 1;
        sdim = 1;
        cells = 1;
    }
    f.dim = la < k ? dim : 1;
    f.sdim = la < k ? sdim : 1;
    f.inv_h = ih;
    f.ncells = (int32_t)cells;
    float fr = 1.f;
    if (la < k && ext_up > 0.f) {
        const float cover = half && la > 0 ? 4.f : 2.f * (float)mm + 1.f;
        const float span = ih > 0.f ? cover / ih : INFINITY;
        fr = fminf(1.f, span / ext_up);
    }
    f.frac = over_axes(fr);
}

// ceil(2^36 / d) for 1 <= d <= 1024 (EventHdr::mag) in 32-bit divisions: with
// 2^32 = q d + rem, 0 < rem <= d, it is 16 q + ceil(16 rem / d).
__device__ __forceinline__ uint64_t division_multiplier(uint32_t d) {
    const uint32_t q = 0xffffffffu / d;
    const uint32_t rem = 0xffffffffu - q * d + 1u;
    return 16ull * q + (16u * rem + d - 1u) / d;
}

// The grid parameters of one event from its bounding box, by a whole block (at
// least kFitWarps warps): box[j], box[kMaxD + j] are the ordered-int extremes of
// coordinate j in shared memory, bad a non-finite input.  Warp w fits the
// candidate of k_hi - w axes; the best one's warp writes the parameters.
// H: the event's header (global or shared memory), everything else of it set.
// Half cells reach four cells along an axis where plain ones reach three, which
// is all of an axis of few cells: two more warps fit five and four axes of
// plain cells, taken (H.half = 0) where the expected candidates of a query, at
// kWideCost of a half cell's each (grids of few cells only: the starting edge
// must fit the budget) and with kWideMore5 or kWideMore4 for the
// look-ups (five axes: three times as many), are fewer.
constexpr int kFitWarps = 3;
constexpr int kWideWarps = 2;
constexpr float kWideCost = 0.45f;
constexpr float kWideMore5 = 350.f, kWideMore4 = 150.f;
__device__ void derive_params(EventHdr& H, const int32_t* box, bool bad, int D, float r, int m, int axes_mode,
                              int naxes_req) {
    __shared__ float s_frac[kFitWarps + kWideWarps];
    __shared__ int s_start[kFitWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n = H.n;
    // per-event presets (batched autotuning) win over the call's options; 0 =
    // automatic: the candidate with the smallest expected neighbourhood under
    // the cell budget among the widest count and one axis fewer (half cells:
    // six, five and four axes)
    const int want = H.naxes > 0 ? H.naxes : naxes_req;
    const int m_req = H.m > 0 ? H.m : m;
    const bool half = H.half != 0;
    const float lo_j = lane < D ? ordered_to_float(box[lane]) : 0.f;
    const float hi_j = lane < D ? ordered_to_float(box[kMaxD + lane]) : 0.f;
    const bool fin = lane >= D || (isfinite(lo_j) && isfinite(hi_j));
    const bool valid = __all_sync(0xffffffffu, fin) && !bad && n > 0;
    const int kmax = min(D, half ? kHdrAxes : kMaxAxes);
    const int k_hi = want > 0 ? min(D, min(want, kMaxAxes)) : kmax;
    const int k_lo = want > 0 ? k_hi : max(1, kmax - (half ? 2 : 1));
    const int64_t cap = half ? min((int64_t)H.cell_cap, kHalfMaxCells) : (int64_t)H.cell_cap;
    // grids requested with up to four axes are scanned by the row-task
    // kernel, whose lanes hold one neighbour row each
    const int max_rows = (want >= 1 && want <= 4) ? 32 : kMaxNbrRows;
    GridFit f;
    f.frac = INFINITY;
    if (warp < kFitWarps && k_hi - warp >= k_lo)
        grid_fit(f, lo_j, hi_j, D, k_hi - warp, half ? 1 : m_req, axes_mode, r, cap, valid, max_rows, half);
    if (warp >= kFitWarps && warp < kFitWarps + kWideWarps) {
        if (half) grid_fit(f, lo_j, hi_j, D, kMaxAxes - (warp - kFitWarps), 1, axes_mode, r, cap, valid, kMaxNbrRows, false, true);
        if (lane == 0) s_frac[warp] = f.frac;
    }
    if (warp < kFitWarps && lane == 0) {
        s_frac[warp] = f.frac;
        s_start[warp] = f.at_start ? 1 : 0;
    }
    __syncthreads();   // (also: every warp has read the header before it is written)
    // at the starting cell edge a grid over more axes covers at most the
    // fraction of one over fewer (one factor <= 1 more): those are not taken
    int best = 0;
    for (int w = 1; w < kFitWarps && k_hi - w >= k_lo && !s_start[w - 1]; ++w)
        if (s_frac[w] < s_frac[best]) best = w;
    float cost = (float)n * s_frac[best];
    for (int w = 0; w < kWideWarps && half && valid; ++w) {
        const float c = kWideCost * (float)n * s_frac[kFitWarps + w] + (w == 0 ? kWideMore5 : kWideMore4);
        if (c < cost) {
            cost = c;
            best = kFitWarps + w;
        }
    }
    if (warp != best) return;
    const int na = f.naxes;
    if (lane < kHdrAxes) {
        const bool gridded = lane < na;
        const int sd = gridded && valid ? f.sdim : 1;
        H.axes[lane] = gridded ? f.axis : 0;
        H.dims[lane] = sd;
        H.fdims[lane] = gridded && valid ? f.dim : 1;
        H.mag[lane] = division_multiplier((uint32_t)sd);
        H.lo[lane] = gridded && valid ? f.lo : 0.f;
        H.hi[lane] = gridded && valid ? f.hi : 0.f;
    }
    if (lane < kMaxD) {
        float c = 0.f;
        if (valid && lane < D) {
            c = __fadd_rn(lo_j, __fmul_rn(0.5f, __fsub_rn(hi_j, lo_j)));
            if (!isfinite(c)) c = 0.f;
        }
        H.ctr[lane] = c;
    }
    if (lane == 0) {
        if (best >= kFitWarps) H.half = 0;
        H.naxes = na;
        H.m = f.m;
        H.valid = valid ? 1 : 0;
        H.inv_h = valid ? f.inv_h : 0.f;
        H.ncells = valid ? f.ncells : 1;
    }
}

__device__ void event_params(EventHdr* hdr, int e, int D, int32_t* bbox, float r, int m,
                             int axes_mode, int naxes_req) {
    __shared__ int32_t bb[kBBoxStride];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // lane c holds copy c of entry k; a warp reduction combines them (all of a
    // warp's loads are issued before the first reduction)
    constexpr int kPer = (kBBoxStride + 7) / 8;
    int32_t v[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int k = warp + 8 * i;
        // L2 reads: the copies were updated by other blocks' atomics; they are
        // left empty for the next build
        int32_t* at = bbox + ((int64_t)e * kBBoxCopies + lane) * kBBoxStride + k;
        v[i] = k < kBBoxStride ? __ldcg(at) : 0;
        if (k < kBBoxStride) *at = empty_box_entry(k);
    }
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
        const int k = warp + 8 * i;
        const int32_t x = k < 16 ? __reduce_min_sync(0xffffffffu, v[i])
                                 : (k < 32 ? __reduce_max_sync(0xffffffffu, v[i])
                                           : (int32_t)__reduce_or_sync(0xffffffffu, (unsigned)v[i]));
        if (lane == 0 && k < kBBoxStride) bb[k] = x;
    }
    __syncthreads();
    derive_params(hdr[e], bb, bb[32] != 0, D, r, m, axes_mode, naxes_req);
}

// Non-finite check of a query set binned with foreign parameters (the bbox
// kernel does it for reference sets).
__global__ void __launch_bounds__(kBuildPtsPerBlock) k_cellid(const EventHdr* hdr,
                                                              const int32_t* blk_start, int E,
                                                              int D, int32_t* counts,
                                                              int32_t* cid, int32_t* rnk,
                                                              int check_finite, int32_t* status,
                                                              EarlyPts ep) {
    pdl_trigger();
    extern __shared__ float sm[];
    const bool pad = (D & 3) == 0;
    const bool staged = stage_early(sm, ep, D, pad);
    pdl_wait();
    const int e = find_event(blk_start, E, blockIdx.x);
    const EventHdr& h = hdr[e];
    const int64_t p0 = (int64_t)(blockIdx.x - blk_start[e]) * kBuildPtsPerBlock;
    const int np = (int)min((int64_t)kBuildPtsPerBlock, h.n - p0);
    if (!staged && np > 0) stage_floats(sm, h.refs + p0 * D, np * D, pad);
    __syncthreads();
    const int i = threadIdx.x;
    if (i >= np) return;
    const StagedRow p{sm, i * D, pad};
    int c = 0;
    if (check_finite) {
        bool bad = false;
        for (int k = 0; k < D; ++k) bad |= !isfinite(p[k]);
        if (bad) atomicOr(status, kStatusNonFinite);
    }
    if (h.valid) c = point_cell(p, h);
    const int64_t gi = h.pt_off + p0 + i;
    cid[gi] = c;
    rnk[gi] = atomicAdd(counts + h.cell_off + count_entry(h, c), 1);
}

// Slot maps and cell-sorted coordinates: each point's slot (its cell's start
// plus its rank), the slot's original index and cell, and the point's row of
// DP floats (zero padding) written with 16-byte stores (one 32-byte sector
// for D <= 8); the input rows are staged in shared memory with 16-byte loads.
// An odd event's padding slot gets NaN coordinates: never within any radius.
__global__ void __launch_bounds__(kBuildPtsPerBlock) k_scatter(const EventHdr* hdr,
                                                               const int32_t* blk_start, int E,
                                                               int D, int DP,
                                                               const int32_t* cstart,
                                                               const int32_t* cid,
                                                               const int32_t* rnk, float* pts,
                                                               int32_t* perm, int32_t* cell,
                                                               EarlyPts ep) {
    pdl_trigger();
    extern __shared__ float sm[];
    const bool pad = (D & 3) == 0;
    const bool staged = stage_early(sm, ep, D, pad);
    pdl_wait();
    const int e = find_event(blk_start, E, blockIdx.x);
    const EventHdr& h = hdr[e];
    const int64_t p0 = (int64_t)(blockIdx.x - blk_start[e]) * kBuildPtsPerBlock;
    const int np = (int)min((int64_t)kBuildPtsPerBlock, h.n - p0);
    if (p0 == 0 && threadIdx.x == 0 && (h.n & 1)) {
        const int64_t slot = h.pt_off + h.n;
        perm[slot] = -1;
        cell[slot] = 0;
        const float nan = __int_as_float(0x7fc00000);
        float4* dst = reinterpret_cast<float4*>(pts + slot * DP);
        for (int j = 0; j < DP / 4; ++j) dst[j] = make_float4(nan, nan, nan, nan);
    }
    if (!staged && np > 0) stage_floats(sm, h.refs + p0 * D, np * D, pad);
    __syncthreads();
    const int i = threadIdx.x;
    if (i >= np) return;
    const int64_t gi = h.pt_off + p0 + i;
    const int c = cid[gi];
    const int64_t slot = (int64_t)cstart[h.cell_off + count_entry(h, c)] + rnk[gi];
    perm[slot] = (int32_t)(p0 + i);
    cell[slot] = c;
    write_row(pts + slot * DP, StagedRow{sm, i * D, pad}, D, DP);
}

// Per row of cells (all gridded coordinates but the fastest fixed): number of
// query tasks.  A task is the intersection of the row's slot range with a
// window of W slots; windows start at the row's first slot rounded down to a
// multiple of A (A = 1 for the 16-query warp tasks of the grid path, A = 8 for
// the 128-query tensor-core tiles, whose operand rows come in groups of 8).
// Entry i of the cell arrays doubles as row slot i.
__device__ __forceinline__ void row_slots(const EventHdr& h, const int32_t* cstart, int64_t row,
                                          int32_t& base, int32_t& cnt) {
    if (h.valid) {
        const int64_t c0 = h.cell_off + row * h.dims[0];
        base = cstart[c0];
        cnt = cstart[c0 + h.dims[0]] - base;
    } else {
        // invalid event: all its queries in one row (they get empty rows)
        base = (int32_t)h.pt_off;
        cnt = row == 0 ? (int32_t)h.n : 0;
    }
}

__global__ void k_rowtasks(const EventHdr* hdr, const int64_t* cell_off, int E, int64_t i0,
                           int64_t i1, const int32_t* cstart, int32_t* rtask, int W, int A,
                           int path_filter) {
    pdl_trigger();
    pdl_wait();
    const int64_t i = i0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= i1) return;
    const int e = find_event64(cell_off, E, i);
    const EventHdr& h = hdr[e];
    const int64_t row = i - cell_off[e];
    int64_t nrows = 1;   // rows: every gridded coordinate but the fastest
    for (int a = 1; a < kHdrAxes && h.valid; ++a) nrows *= h.dims[a];
    int32_t nt = 0;
    // events another launch of a mixed batch queries get no tasks
    if (row < nrows && (path_filter < 0 || h.path == path_filter)) {
        int32_t base, cnt;
        row_slots(h, cstart, row, base, cnt);
        if (cnt > 0) {
            const int32_t w0 = base & ~(A - 1);
            nt = (base + cnt - w0 + W - 1) / W;
        }
    }
    rtask[i] = nt;
}

__global__ void k_emit(const EventHdr* hdr, const int64_t* cell_off, int E, int64_t i0,
                       int64_t i1, const int32_t* cstart, const int32_t* rtask_start,
                       const int32_t* rtask_count_src, Task* tasks, int64_t task_cap, int W,
                       int A, int32_t* status) {
    pdl_trigger();
    pdl_wait();
    const int64_t i = i0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= i1) return;
    const int e = find_event64(cell_off, E, i);
    const EventHdr& h = hdr[e];
    const int64_t row = i - cell_off[e];
    const int32_t t0 = rtask_start[i];
    const int32_t t1 = (i + 1 < i1) ? rtask_start[i + 1] : rtask_count_src[0];
    if (t1 <= t0) return;
    int32_t base, cnt;
    row_slots(h, cstart, row, base, cnt);
    const int32_t w0 = base & ~(A - 1);
    for (int32_t t = t0; t < t1; ++t) {
        if (t >= task_cap) {   // never with the tensor-core path's capacity; guarded all the same
            atomicOr(status, kStatusCapacity);
            return;
        }
        const int32_t ws = w0 + (t - t0) * W;
        const int32_t a = max(ws, base);
        const int32_t b = min(ws + W, base + cnt);
        Task tk;
        tk.qslot = a;
        tk.nq = b - a;
        tk.ev = e;
        tk.row = (int32_t)row;
        tasks[t] = tk;
    }
}

void enqueue_tasks(GridBufs& g, int W, int A, Task* out, int64_t out_cap, int32_t* count_out,
                   int32_t* d_status, cudaStream_t st, int path_filter, int64_t i0, int64_t i1) {
    if (i1 < 0) i1 = g.L;
    i0 = std::min(std::max<int64_t>(i0, 0), i1);
    const int64_t n = i1 - i0;
    const unsigned nb = (unsigned)std::max<int64_t>(1, ceil_div(n, 256));
    launch_pdl(k_rowtasks, dim3(nb), dim3(256), 0, st, g.hdr, g.cell_off, g.E, i0, i1, g.cstart,
               g.rtask, W, A, path_filter);
    // the scan of the range's task counts gives each row its first task
    enqueue_scan(g.rtask + i0, n, g.parts, count_out, st);
    launch_pdl(k_emit, dim3(nb), dim3(256), 0, st, g.hdr, g.cell_off, g.E, i0, i1, g.cstart, g.rtask,
               count_out, out, out_cap, W, A, d_status);
}

// ------------------------------------------------------------------ scan
// Exclusive prefix scan of int32 in place (three phases: per-block totals,
// scan of the totals, per-block scan with offset).  Inside a block each thread
// scans kScanItems consecutive values, then warp shuffles scan the thread
// totals and a second warp pass scans the warp totals.

constexpr int kScanThreads = 256;
constexpr int kScanItems = kScanChunk / kScanThreads;

__device__ __forceinline__ int32_t block_exclusive_scan(int32_t v, int32_t* warp_tot,
                                                        int32_t* block_total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) warp_tot[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int32_t w = lane < (kScanThreads / 32) ? warp_tot[lane] : 0;
        int32_t z = w;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int32_t y = __shfl_up_sync(0xffffffffu, z, o);
            if (lane >= o) z += y;
        }
        if (lane < kScanThreads / 32) warp_tot[lane] = z - w;
        if (lane == 31) *block_total = z;
    }
    __syncthreads();
    return x - v + warp_tot[warp];
}

__global__ void __launch_bounds__(kScanThreads) k_scan_reduce(const int32_t* data, int64_t n,
                                                              int32_t* parts) {
    pdl_trigger();
    pdl_wait();
    __shared__ int32_t red[kScanThreads / 32];
    const int64_t base = (int64_t)blockIdx.x * kScanChunk;
    int32_t s = 0;
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + (int64_t)k * kScanThreads + threadIdx.x;
        if (i < n) s += data[i];
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x < 32) {
        int32_t t = threadIdx.x < kScanThreads / 32 ? red[threadIdx.x] : 0;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) parts[blockIdx.x] = t;
    }
}

// Shared-memory slot of chunk entry i: one padding word per 32 entries, so
// that both the coalesced pass (entry k * 256 + t on thread t) and the
// per-thread pass (entries 8t .. 8t + 7 on thread t) touch 32 distinct banks
// per warp access.
__device__ __forceinline__ int scan_slot(int i) { return i + (i >> 5); }
constexpr int kScanSlots = kScanChunk + kScanChunk / 32;

// Scan one chunk of kScanChunk values in place with an added offset.
__device__ void scan_chunk(int32_t* data, int64_t n, int64_t base, int32_t offset,
                           int32_t* total_out) {
    __shared__ int32_t buf[kScanSlots];
    __shared__ int32_t warp_tot[kScanThreads / 32];
    __shared__ int32_t btot;
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + (int64_t)k * kScanThreads + threadIdx.x;
        buf[scan_slot(k * kScanThreads + threadIdx.x)] = i < n ? data[i] : 0;
    }
    __syncthreads();
    int32_t v[kScanItems];
    int32_t t = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        v[k] = buf[scan_slot(threadIdx.x * kScanItems + k)];
        t += v[k];
    }
    int32_t ex = block_exclusive_scan(t, warp_tot, &btot) + offset;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        buf[scan_slot(threadIdx.x * kScanItems + k)] = ex;
        ex += v[k];
    }
    __syncthreads();
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + (int64_t)k * kScanThreads + threadIdx.x;
        if (i < n) data[i] = buf[scan_slot(k * kScanThreads + threadIdx.x)];
    }
    if (total_out && threadIdx.x == 0) *total_out = btot + offset;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_single(int32_t* data, int64_t n,
                                                              int32_t* total) {
    pdl_trigger();
    pdl_wait();
    scan_chunk(data, n, 0, 0, total);
}

// Down pass.  summed == 0: block b first sums the partials of the blocks
// before it (used while there are at most kScanSumParts of them: at most 16
// L2 reads per thread, cheaper than a launch of the one-block partials scan),
// then scans its chunk with that offset; the last block also writes the
// total.  summed == 1: the partials were already scanned (k_scan_parts).
constexpr int kScanSumParts = 4096;

__global__ void __launch_bounds__(kScanThreads) k_scan_down(int32_t* data, int64_t n,
                                                            const int32_t* parts, int32_t* total,
                                                            int summed) {
    pdl_trigger();
    pdl_wait();
    if (summed) {
        scan_chunk(data, n, (int64_t)blockIdx.x * kScanChunk, parts[blockIdx.x], nullptr);
        return;
    }
    __shared__ int32_t red[kScanThreads / 32];
    __shared__ int32_t offset;
    int32_t v = 0;
    for (int j = threadIdx.x; j < (int)blockIdx.x; j += kScanThreads) v += parts[j];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        int32_t t = threadIdx.x < kScanThreads / 32 ? red[threadIdx.x] : 0;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (threadIdx.x == 0) offset = t;
    }
    __syncthreads();
    scan_chunk(data, n, (int64_t)blockIdx.x * kScanChunk, offset,
               blockIdx.x == gridDim.x - 1 ? total : nullptr);
}

// One CTA: exclusive scan of the nb partials in place, chunk after chunk with
// a running carry; writes the grand total.
__global__ void __launch_bounds__(kScanThreads) k_scan_parts(int32_t* parts, int64_t nb,
                                                             int32_t* total) {
    pdl_trigger();
    pdl_wait();
    __shared__ int32_t carry;
    if (threadIdx.x == 0) carry = 0;
    __syncthreads();
    for (int64_t base = 0; base < nb; base += kScanChunk) {
        const int32_t c = carry;
        __shared__ int32_t ctot;
        scan_chunk(parts, nb, base, c, &ctot);
        __syncthreads();
        if (threadIdx.x == 0) carry = ctot;
        __syncthreads();
    }
    if (threadIdx.x == 0) *total = carry;
}

int64_t scan_parts_needed(int64_t n) { return std::max<int64_t>(1, ceil_div(n, kScanChunk)); }

void enqueue_scan(int32_t* data, int64_t n, int32_t* parts, int32_t* total, cudaStream_t st) {
    const int64_t nb = scan_parts_needed(n);
    if (nb == 1) {
        launch_pdl(k_scan_single, dim3(1), dim3(kScanThreads), 0, st, data, n, total);
        return;
    }
    launch_pdl(k_scan_reduce, dim3((unsigned)nb), dim3(kScanThreads), 0, st, data, n, parts);
    if (nb <= kScanSumParts) {
        launch_pdl(k_scan_down, dim3((unsigned)nb), dim3(kScanThreads), 0, st, data, n, parts, total, 0);
    } else {
        launch_pdl(k_scan_parts, dim3(1), dim3(kScanThreads), 0, st, parts, nb, total);
        launch_pdl(k_scan_down, dim3((unsigned)nb), dim3(kScanThreads), 0, st, data, n, parts, total, 1);
    }
}

// ------------------------------------------------------------------ cell scan
// Exclusive scan of the cell counts, every event's on its own: an event's first
// slot is known, so events share nothing, and only the entries a grid uses are
// scanned.  Blocks of kCellChunk entries (an event's last one ends with its
// region), 16 entries a thread in four 16-byte loads; the down pass sums the totals of its
// event's blocks before it (beyond kCellSumParts of them a pass of one block per
// event scans the totals first).  300k x 8 (3.5 M cells), reduce + down: 5.0 +
// 9.6 us with 2,048-entry blocks and 4-byte accesses through shared memory.

constexpr int kCellThreads = 256;
constexpr int kCellSumParts = 4096;
static_assert(kCellChunk == 16 * kCellThreads, "four quads a thread");

// Event of a block, its first block, whether the block holds used entries, its
// own entries (from `at` on, in `quads` 16-byte pieces).
struct CellBlock {
    int e, first, quads;
    int64_t at;
    bool used;
    __device__ CellBlock(const EventHdr* hdr, int E) {
        int lo = 0, hi = E - 1;
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (hdr[mid].cblk0 <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
        }
        e = lo;
        const EventHdr& h = hdr[lo];
        first = h.cblk0;
        const int off = ((int)blockIdx.x - first) * kCellChunk;
        at = h.cell_off + off;
        quads = (int)min((int64_t)kCellChunk, cell_entries(h.cell_cap) - off) / 4;
        used = off < used_entries(h);
    }
};

__global__ void __launch_bounds__(kCellThreads) k_cells_reduce(const EventHdr* hdr, int E, const int32_t* counts,
                                                               int32_t* parts) {
    pdl_trigger();
    pdl_wait();
    __shared__ int32_t red[kCellThreads / 32];
    const CellBlock cb(hdr, E);
    if (!cb.used) return;
    const int4* c4 = reinterpret_cast<const int4*>(counts + cb.at) + threadIdx.x;
    int4 v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
        v[j] = (int)threadIdx.x + j * kCellThreads < cb.quads ? c4[j * kCellThreads] : make_int4(0, 0, 0, 0);
    int s = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) s += v[j].x + v[j].y + v[j].z + v[j].w;
    s = __reduce_add_sync(0xffffffffu, s);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        int t = 0;
        for (int w = 0; w < kCellThreads / 32; ++w) t += red[w];
        parts[blockIdx.x] = t;
    }
}

// Exclusive scan of one event's block totals in place.
__global__ void __launch_bounds__(1024) k_cells_parts(const EventHdr* hdr, int32_t* parts) {
    pdl_trigger();
    pdl_wait();
    __shared__ int32_t wt[32];
    const EventHdr& h = hdr[blockIdx.x];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nb = (used_entries(h) + kCellChunk - 1) / kCellChunk;
    int32_t* p = parts + h.cblk0;
    int carry = 0;
    for (int b0 = 0; b0 < nb; b0 += 1024) {
        const int i = b0 + threadIdx.x;
        const int v = i < nb ? p[i] : 0;
        int incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) wt[warp] = incl;
        __syncthreads();
        int below = 0, all = 0;
        for (int w = 0; w < 32; ++w) {
            below += w < warp ? wt[w] : 0;
            all += wt[w];
        }
        if (i < nb) p[i] = carry + below + incl - v;
        carry += all;
        __syncthreads();
    }
}

// scanned: the totals were scanned (k_cells_parts).
__global__ void __launch_bounds__(kCellThreads) k_cells_down(const EventHdr* hdr, int E, int32_t* counts,
                                                             const int32_t* parts, int scanned) {
    pdl_trigger();
    pdl_wait();
    constexpr int kW = kCellThreads / 32;
    __shared__ int32_t tot[4 * kW], red[kW];
    const CellBlock cb(hdr, E);
    if (!cb.used) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int4* c4 = reinterpret_cast<int4*>(counts + cb.at) + threadIdx.x;
    int4 v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
        v[j] = (int)threadIdx.x + j * kCellThreads < cb.quads ? c4[j * kCellThreads] : make_int4(0, 0, 0, 0);
    int before = 0;   // the event's entries before this block
    if (scanned) {
        if (threadIdx.x == 0) before = parts[blockIdx.x];
    } else {
        for (int j = cb.first + threadIdx.x; j < (int)blockIdx.x; j += kCellThreads) before += parts[j];
    }
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 0) red[warp] = before;
    int excl[4];   // of each quad within its warp's 128 entries
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int t = v[j].x + v[j].y + v[j].z + v[j].w;
        int incl = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        excl[j] = incl - t;
        if (lane == 31) tot[j * kW + warp] = incl;
    }
    __syncthreads();
    if (warp == 0) {
        static_assert(4 * kW == 32, "one total per lane");
        const int t = tot[lane];
        int incl = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const int base = (int)hdr[cb.e].pt_off + __reduce_add_sync(0xffffffffu, lane < kW ? red[lane] : 0);
        tot[lane] = base + incl - t;
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int x = tot[j * kW + warp] + excl[j];
        if ((int)threadIdx.x + j * kCellThreads < cb.quads)
            c4[j * kCellThreads] = make_int4(x, x + v[j].x, x + v[j].x + v[j].y, x + v[j].x + v[j].y + v[j].z);
    }
}

// ------------------------------------------------------------------ small sets
// The whole build of one small event in one launch: a cluster of kSmallCtas
// CTAs, cluster barriers where the chain above has kernel boundaries.  A set of
// a few thousand points leaves the six kernels of the chain nothing to do but
// launch, read the previous one's results from L2 and drain (about 3 us each);
// a cluster's SMs hold the points' cell ids and ranks in registers, and
// the barriers cost 0.5 us each.  All of the memory it shares across CTAs is
// read past L1 (ld.cg) after a cluster barrier.  Bound by the latency of its
// phases (4096 x 3: 10.4 us, 2.7 of them the grid parameters, 5.5 the cell
// counts' four round trips); sixteen SMs are enough up to 32,768 points, where
// the chain catches up.  Build + query, chain / cluster: 4096 x 3 30.8 / 21.1
// us, 5,000 x 8 40.5 / 24.4, 20,000 x 8 45.8 / 38.4, 32,000 x 8 52.2 / 49.9
// (eight CTAs without staged rows lost from 13,000 points on).
//   1 bounding box of the CTA's points, zeroing of the cell counts; boxes to
//     every CTA
//   2 grid parameters (one warp of every CTA, redundantly); cell ids, ranks
//   3 per-warp sums of the counts; CTA sums to every CTA
//   4 exclusive scan of the counts in place
//   5 slot maps and cell-sorted coordinates
// With `src` (cross-set queries) the parameters are those of src's grid.

constexpr int kSmallCtas = 16;
constexpr int kSmallThreads = 1024;
constexpr int kSmallPer = 2;    // points of a thread, at most
constexpr int kSmallQuads = 2;  // 128-entry steps of a warp's scan segment kept in registers
constexpr int64_t kSmallMax = (int64_t)kSmallCtas * kSmallThreads * kSmallPer;
constexpr int64_t kSmallCells = 16 * kSmallMax;   // cell-array entries

__host__ __device__ constexpr size_t small_stage_floats(int64_t per, int D) {
    return (size_t)per * D + (size_t)per * D / 32 + 1;
}
// The most any set needs: the shared-memory limit set before every launch (it
// is the function's, shared by every thread's calls, so no call may lower it).
constexpr size_t kSmallSmemMost = sizeof(float) * small_stage_floats(kSmallPer * kSmallThreads, kMaxD);

__global__ void __launch_bounds__(kSmallThreads, 1)
    k_build_small(OneEventTables t1, const EventHdr* src, int per, int D, int DP, float r, int m, int axes_mode,
                  int naxes_req, EventHdr* hdr, int32_t* blk_start, int64_t* cell_off, int32_t* counts,
                  int32_t* scalars, float* pts, int32_t* perm, int32_t* cell, int32_t* status) {
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    constexpr int kWarps = kSmallThreads / 32;
    constexpr unsigned kAll = 0xffffffffu;
    extern __shared__ float sm[];   // this CTA's input rows (staged_slot layout)
    __shared__ EventHdr sh;
    __shared__ int32_t s_mn[kMaxD], s_mx[kMaxD], s_bad;
    __shared__ int32_t s_box[kSmallCtas][2 * kMaxD + 1], s_all[2 * kMaxD];
    __shared__ int32_t s_wt[kWarps], s_tot[kSmallCtas];
    pdl_wait();      // (first of its chain: the points may have just been written)
    pdl_trigger();
    cluster.barrier_arrive();   // (every CTA must run before its shared memory is written)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int rank = (int)cluster.block_rank(), ctas = (int)cluster.num_blocks();
    const int n = (int)t1.hdr.n;
    const float* refs = t1.hdr.refs;
    const bool pad = (D & 3) == 0;
    // this CTA's points [p0, p0 + np); thread t has the t-th, t + 1024-th, ...
    const int p0 = min(rank * per, n), np = min(per, n - p0);
    const int first = rank * kSmallThreads + tid, step = ctas * kSmallThreads;
    if (tid < kMaxD) {
        s_mn[tid] = INT_MAX;
        s_mx[tid] = INT_MIN;
    }
    if (tid == 0) s_bad = 0;
    for (int i = tid; i < (int)(sizeof(EventHdr) / 4); i += kSmallThreads)
        reinterpret_cast<int32_t*>(&sh)[i] = reinterpret_cast<const int32_t*>(&t1.hdr)[i];
    stage_floats(sm, refs + (int64_t)p0 * D, np * D, pad);
    __syncthreads();
    {
        // warp w takes coordinate w % D of every (32 / D)-th run of 32 points
        const int runs = kWarps / D, k = warp % D, g = warp / D;
        if (g < runs) {
            bool bad = false;
            float mn = INFINITY, mx = -INFINITY;
#pragma unroll 4
            for (int i = g * 32 + lane; i < np; i += runs * 32) {
                const float v = sm[stage_slot(i * D + k, pad)];
                bad |= !isfinite(v);
                mn = fminf(mn, v);
                mx = fmaxf(mx, v);
            }
            const int32_t a = __reduce_min_sync(kAll, float_to_ordered(mn));
            const int32_t b = __reduce_max_sync(kAll, float_to_ordered(mx));
            const bool any_bad = __any_sync(kAll, bad);
            if (lane == 0) {
                atomicMin(s_mn + k, a);
                atomicMax(s_mx + k, b);
                if (any_bad) atomicOr(&s_bad, 1);
            }
        }
    }
    {
        // all of the cell array, or what the foreign parameters use of it
        const int L = src ? (t1.hdr.rowsort ? src->ncells / src->dims[0] : src->ncells) + 1 : t1.hdr.cell_cap + 1;
        int4* c4 = reinterpret_cast<int4*>(counts);
        for (int j = first; j < L / 4; j += step) c4[j] = make_int4(0, 0, 0, 0);
        for (int j = L / 4 * 4 + first; j < L; j += step) counts[j] = 0;
    }
    if (rank == 0 && tid < kScalars) scalars[tid] = 0;
    __syncthreads();
    cluster.barrier_wait();
    // this CTA's box to every CTA
    if (tid < ctas * 64) {
        const int to = tid >> 6, k = tid & 63;
        if (k <= 2 * kMaxD)
            *cluster.map_shared_rank(&s_box[rank][k], to) =
                k < kMaxD ? s_mn[k] : (k < 2 * kMaxD ? s_mx[k - kMaxD] : s_bad);
    }
    cluster.sync();
    int bad = 0;
    for (int c = 0; c < ctas; ++c) bad |= s_box[c][2 * kMaxD];
    if (rank == 0 && tid == 0 && bad) atomicOr(status, kStatusNonFinite);
    if (tid < 2 * kMaxD) {
        int32_t v = s_box[0][tid];
        for (int c = 1; c < ctas; ++c) v = tid < kMaxD ? min(v, s_box[c][tid]) : max(v, s_box[c][tid]);
        s_all[tid] = v;
    }
    __syncthreads();
    if (src) {
        copy_params(sh, *src);
    } else {
        derive_params(sh, s_all, bad != 0, D, r, m, axes_mode, naxes_req);
    }
    __syncthreads();
    if (rank == 0) {
        const int words = (int)(sizeof(EventHdr) / 4);
        for (int i = tid; i < words; i += kSmallThreads)
            reinterpret_cast<int32_t*>(hdr)[i] = reinterpret_cast<const int32_t*>(&sh)[i];
        if (tid == 0) {
            blk_start[0] = 0;
            blk_start[1] = t1.nblk;
            cell_off[0] = 0;
            cell_off[1] = t1.cell_end;
        }
    }
    // cell ids and ranks, kept in registers
    int32_t key[kSmallPer], rnk[kSmallPer];
#pragma unroll
    for (int j = 0; j < kSmallPer; ++j) {
        const int i = tid + j * kSmallThreads;
        key[j] = 0;
        rnk[j] = 0;
        if (i < np) {
            if (sh.valid) key[j] = point_cell(StagedRow{sm, i * D, pad}, sh);
            rnk[j] = atomicAdd(counts + count_entry(sh, key[j]), 1);
        }
    }
    cluster.sync();
    // exclusive scan of the used entries, the one past the last cell among
    // them: warp g of the cluster takes the g-th segment of `seg` entries
    const int used = used_entries(sh);
    const int seg = ((used + ctas * kWarps - 1) / (ctas * kWarps) + 127) / 128 * 128;
    const int s0 = (rank * kWarps + warp) * seg, s1 = min(s0 + seg, used);
    // four entries from i on (zero past the segment's end)
    auto quad = [&](int i) -> int4 {
        if (i + 4 <= s1) return __ldcg(reinterpret_cast<const int4*>(counts + i));
        int4 v = make_int4(0, 0, 0, 0);
        if (i < s1) v.x = __ldcg(counts + i);
        if (i + 1 < s1) v.y = __ldcg(counts + i + 1);
        if (i + 2 < s1) v.z = __ldcg(counts + i + 2);
        return v;
    };
    int4 held[kSmallQuads];   // the segment's first steps, for both passes
    int sum = 0;
#pragma unroll
    for (int j = 0; j < kSmallQuads; ++j) {
        const int o = s0 + 128 * j + 4 * lane;
        held[j] = o < s1 ? quad(o) : make_int4(0, 0, 0, 0);
    }
#pragma unroll
    for (int j = 0; j < kSmallQuads; ++j) sum += held[j].x + held[j].y + held[j].z + held[j].w;
#pragma unroll 4
    for (int o = s0 + 128 * kSmallQuads + 4 * lane; o < s1; o += 128) {
        const int4 v = quad(o);
        sum += v.x + v.y + v.z + v.w;
    }
    sum = __reduce_add_sync(kAll, sum);
    if (lane == 0) s_wt[warp] = sum;
    __syncthreads();
    if (warp == 0) {
        const int v = s_wt[lane];
        int incl = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kAll, incl, o);
            if (lane >= o) incl += y;
        }
        s_wt[lane] = incl - v;
        const int total = __shfl_sync(kAll, incl, 31);
        if (lane < ctas) *cluster.map_shared_rank(&s_tot[rank], lane) = total;
    }
    cluster.sync();
    int carry = s_wt[warp];
    for (int c = 0; c < rank; ++c) carry += s_tot[c];
    auto scan_step = [&](int b, const int4 v) {
        const int i = b + 4 * lane;
        const int t = v.x + v.y + v.z + v.w;
        int incl = t;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kAll, incl, o);
            if (lane >= o) incl += y;
        }
        const int x = carry + incl - t;
        const int4 w = make_int4(x, x + v.x, x + v.x + v.y, x + v.x + v.y + v.z);
        if (i + 4 <= s1) {
            *reinterpret_cast<int4*>(counts + i) = w;
        } else {
            if (i < s1) counts[i] = w.x;
            if (i + 1 < s1) counts[i + 1] = w.y;
            if (i + 2 < s1) counts[i + 2] = w.z;
        }
        carry += __shfl_sync(kAll, incl, 31);
    };
#pragma unroll
    for (int j = 0; j < kSmallQuads; ++j)
        if (s0 + 128 * j < s1) scan_step(s0 + 128 * j, held[j]);
    if (s0 + 128 * kSmallQuads < s1) {
        // (the next step's entries in flight)
        int4 next = quad(s0 + 128 * kSmallQuads + 4 * lane);
#pragma unroll 1
        for (int b = s0 + 128 * kSmallQuads; b < s1; b += 128) {
            const int4 v = next;
            next = quad(b + 128 + 4 * lane);
            scan_step(b, v);
        }
    }
    cluster.sync();
#pragma unroll
    for (int j = 0; j < kSmallPer; ++j) {
        const int i = tid + j * kSmallThreads;
        if (i < np) {
            const int slot = __ldcg(counts + count_entry(sh, key[j])) + rnk[j];
            perm[slot] = p0 + i;
            cell[slot] = key[j];
            write_row(pts + (int64_t)slot * DP, StagedRow{sm, i * D, pad}, D, DP);
        }
    }
    if (rank == 0 && tid == 0 && (n & 1)) {   // an odd event's padding slot
        perm[n] = -1;
        cell[n] = 0;
        const float nan = __int_as_float(0x7fc00000);
        float4* dst = reinterpret_cast<float4*>(pts + (int64_t)n * DP);
        for (int q = 0; q < DP / 4; ++q) dst[q] = make_float4(nan, nan, nan, nan);
    }
}

// ------------------------------------------------------------------ host

// The budget grows with n so that the cells stay near r on the sets the
// library is for, and not faster, since every build zeroes and scans it all;
// the parameter step falls back to fewer axes when it would make the cells too
// coarse.  Half cells: 12 n, just what six axes need for the 300k x 8
// tracking-like event (22 x 11^5 = 3.5 M; 6 n 171 us, 12 n 151, 18 n 156, 30 n
// 166, build + query), flat within 3 us for smaller sets.  Five axes of plain
// cells: 18 n (22^5 = 5.2 M there).  Up to four: 4 n (1 M x 3, two neighbours
// each: n / 2 269 us, n 236, 2 n 217, 4 n 219; 300k x 4: n 133, 2 n 119, 4 n
// 108) on automatic grids of up to four dimensions; requested axes as before
// (2 n for four, n / 2 for fewer: row tasks and tensor-core tiles want long
// rows of cells).
int64_t cell_cap_for(int64_t n, int naxes, CellKind kind) {
    if (kind == CellKind::kHalf) return std::min<int64_t>(std::max<int64_t>(16384, 12 * n), kHalfMaxCells);
    const int64_t per = naxes >= 5 ? 18 : (kind == CellKind::kLow ? 4 : (naxes == 4 ? 2 : 0));
    int64_t c = per ? per * n : n / 2 + 1;
    c = std::max<int64_t>(16384, c);
    return std::min<int64_t>(c, naxes >= 5 ? ((int64_t)1 << 27) : ((int64_t)1 << 24));
}

static size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

void grid_free(GridBufs& g) {
    tc_free(g);
    rows_free(g);
    if (g.base) cudaFree(g.base);
    if (g.h_pinned) cudaFreeHost(g.h_pinned);
    if (g.h_pinned_free) cudaEventDestroy(g.h_pinned_free);
    g = GridBufs();
}

frnn_status grid_alloc(GridBufs& g, int E, const int64_t* n, int D, std::string& err,
                       const int64_t* caps, int naxes) {
    const int DP = padded_dim(D);
    int64_t n_total = 0, L = 0, nblk = 0, nchunks = 0, ncblk = 0, cells = 0;
    g.h_hdr.assign(E, EventHdr{});
    g.h_blk_start.assign(E + 1, 0);
    g.h_cell_off.assign(E + 1, 0);
    for (int e = 0; e < E; ++e) {
        const int64_t cap = caps ? caps[e] : cell_cap_for(n[e], naxes);
        EventHdr& h = g.h_hdr[e];
        h.n = n[e];
        h.pt_off = n_total;
        h.cell_off = L;
        h.cell_cap = (int32_t)cap;
        h.qchunk0 = (int32_t)nchunks;
        nchunks += ceil_div(n[e], kChunkQ);
        g.h_blk_start[e] = (int32_t)nblk;
        g.h_cell_off[e] = L;
        h.cblk0 = (int32_t)ncblk;
        ncblk += cell_blocks(cap);
        cells += cap + 1;
        n_total += (n[e] + 1) & ~(int64_t)1;   // pair-aligned event regions
        L += cell_entries(cap);
        nblk += std::max<int64_t>(1, ceil_div(n[e], kBuildPtsPerBlock));
    }
    g.h_blk_start[E] = (int32_t)nblk;
    g.h_cell_off[E] = L;
    if (n_total >= INT32_MAX || cells >= ((int64_t)1 << 30) ||
        nblk >= INT32_MAX || nchunks >= INT32_MAX) {
        err = "problem too large for one call (points, cells or tasks exceed the limits)";
        return FRNN_ERR_INVALID_ARG;
    }
    g.E = E;
    g.D = D;
    g.DP = DP;
    g.n_total = n_total;
    g.L = L;
    g.ncblk = ncblk;
    g.nblk = nblk;
    g.nparts = std::max(scan_parts_needed(L), L / kCellChunk + E);   // (>= ncblk, and grows with L and E)
    g.nchunks = nchunks;
    // the buffers are reused only if every region is large enough, the
    // point rows included (a set of a higher dimension needs wider rows)
    const bool fits = g.base && g.cap_n >= n_total && g.cap_DP >= DP && g.cap_L >= L && g.cap_E >= E &&
                      g.cap_blk >= nblk;
    const int64_t cn = std::max<int64_t>(n_total, 1);
    if (!fits) {
        if (g.base) {
            cudaFree(g.base);
            g.base = nullptr;
        }
        size_t off = 0;
        auto take = [&](size_t bytes) {
            size_t o = off;
            off = align_up(off + bytes, 256);
            return o;
        };
        const size_t o_hdr = take(sizeof(EventHdr) * E);
        const size_t o_blk = take(sizeof(int32_t) * (E + 1));
        const size_t o_coff = take(sizeof(int64_t) * (E + 1));
        const size_t o_bbox = take(sizeof(int32_t) * kBBoxStride * kBBoxCopies * E);
        const size_t o_pts = take(sizeof(float) * DP * (cn + kTcRowPad));
        const size_t o_perm = take(sizeof(int32_t) * cn);
        const size_t o_cell = take(sizeof(int32_t) * cn);
        const size_t o_cid = take(sizeof(int32_t) * cn);
        const size_t o_rnk = take(sizeof(int32_t) * cn);
        const size_t o_cst = take(sizeof(int32_t) * L);
        const size_t o_ovf = take(sizeof(Overflow) * cn);
        const size_t o_sc = take(sizeof(int32_t) * kScalars);
        const size_t o_parts = take(sizeof(int32_t) * g.nparts);
        void* base = nullptr;
        cudaError_t ce = cudaMalloc(&base, off);
        if (ce != cudaSuccess) {
            cudaGetLastError();
            err = std::string("cudaMalloc of grid buffers failed: ") + cudaGetErrorString(ce);
            g.cap_n = g.cap_L = g.cap_E = g.cap_blk = g.clean_E = 0;
            g.cap_DP = 0;
            return FRNN_ERR_OUT_OF_MEMORY;
        }
        char* b = static_cast<char*>(base);
        g.base = base;
        g.bytes = off;
        g.hdr = reinterpret_cast<EventHdr*>(b + o_hdr);
        g.blk_start = reinterpret_cast<int32_t*>(b + o_blk);
        g.cell_off = reinterpret_cast<int64_t*>(b + o_coff);
        g.bbox = reinterpret_cast<int32_t*>(b + o_bbox);
        g.pts = reinterpret_cast<float*>(b + o_pts);
        g.perm = reinterpret_cast<int32_t*>(b + o_perm);
        g.cell = reinterpret_cast<int32_t*>(b + o_cell);
        g.cid = reinterpret_cast<int32_t*>(b + o_cid);
        g.rnk = reinterpret_cast<int32_t*>(b + o_rnk);
        g.cstart = reinterpret_cast<int32_t*>(b + o_cst);
        g.rtask = nullptr;   // the tensor-core operands carry the task builder's scratch
        g.ovf = reinterpret_cast<Overflow*>(b + o_ovf);
        g.scalars = reinterpret_cast<int32_t*>(b + o_sc);
        g.parts = reinterpret_cast<int32_t*>(b + o_parts);
        g.cap_n = n_total;
        g.cap_DP = DP;
        g.cap_L = L;
        g.cap_E = E;
        g.clean_E = 0;
        g.cap_blk = nblk;
    }
    // page-locked mirror for the per-event tables
    // (laid out like the device tables: header, block starts and cell offsets
    // at the same relative offsets, so one copy uploads all three)
    const size_t hbytes = (size_t)(reinterpret_cast<char*>(g.cell_off) -
                                   reinterpret_cast<char*>(g.hdr)) +
                          sizeof(int64_t) * (E + 1) + 64;
    if (g.h_pinned_bytes < hbytes) {
        if (g.h_pinned) {
            if (g.h_pinned_free) cudaEventSynchronize(g.h_pinned_free);
            cudaFreeHost(g.h_pinned);
            g.h_pinned = nullptr;
        }
        if (cudaMallocHost(&g.h_pinned, hbytes) != cudaSuccess) {
            cudaGetLastError();
            g.h_pinned_bytes = 0;
            err = "cudaMallocHost of grid tables failed";
            return FRNN_ERR_OUT_OF_MEMORY;
        }
        g.h_pinned_bytes = hbytes;
    }
    if (!g.h_pinned_free) cudaEventCreateWithFlags(&g.h_pinned_free, cudaEventDisableTiming);
    return FRNN_OK;
}

// k_begin_foreign's blocks: four per SM of the GB300's 152, all resident at once
constexpr unsigned kInitBlocks = 608;

static inline unsigned blocks_for(int64_t n, int t) {
    return (unsigned)std::max<int64_t>(1, ceil_div(n, t));
}

// Cell ids, the cell-start scan, slot maps, coordinates.
static void enqueue_sort(GridBufs& g, size_t smem_pts, int check_finite, int32_t* d_status,
                         cudaStream_t st, EarlyPts ep) {
    const int E = g.E, D = g.D;
    launch_pdl(k_cellid, dim3((unsigned)g.nblk), dim3(kBuildPtsPerBlock), smem_pts, st,
               g.hdr, g.blk_start, E, D, g.cstart, g.cid, g.rnk, check_finite, d_status, ep);
    const int64_t nb = g.ncblk;
    int64_t most = g.h_hdr.empty() ? nb : 0;   // blocks of the largest event (without host headers: the only one)
    for (const EventHdr& h : g.h_hdr) most = std::max(most, cell_blocks(h.cell_cap));
    launch_pdl(k_cells_reduce, dim3((unsigned)nb), dim3(kCellThreads), 0, st, g.hdr, E, g.cstart, g.parts);
    if (most > kCellSumParts)
        launch_pdl(k_cells_parts, dim3((unsigned)E), dim3(1024), 0, st, g.hdr, g.parts);
    launch_pdl(k_cells_down, dim3((unsigned)nb), dim3(kCellThreads), 0, st, g.hdr, E, g.cstart, g.parts,
               most > kCellSumParts ? 1 : 0);
    launch_pdl(k_scatter, dim3((unsigned)g.nblk), dim3(kBuildPtsPerBlock), smem_pts, st,
               g.hdr, g.blk_start, E, D, g.DP, g.cstart, g.cid, g.rnk, g.pts, g.perm, g.cell, ep);
    // no task list: the grid query takes chunks of kChunkQ slots in slot order
}

static int box_sub(int64_t nblk) {
    return (int)std::min<int64_t>(std::max<int64_t>(ceil_div(nblk, kBoxWave), 1), kBoxMost);
}

// Empty the boxes of buffers that no build has used yet.  Recorded into a
// caller's capture it has not run yet, so the next build does it again.
void grid_clean(GridBufs& g, cudaStream_t st) {
    if (g.clean_E >= g.E) return;
    launch_pdl(k_box_reset, dim3(blocks_for((int64_t)g.cap_E * kBBoxCopies * kBBoxStride, 256)), dim3(256), 0, st,
               g.bbox, (int)g.cap_E);
    if (!stream_capturing(st)) g.clean_E = g.cap_E;
}

frnn_status enqueue_build(GridBufs& g, const float* const* refs, const BuildOpts& o,
                          const GridBufs* params_from, int32_t* d_status, cudaStream_t st,
                          bool capturing, std::string& err) {
    const int E = g.E, D = g.D;
    for (int e = 0; e < E; ++e) {
        g.h_hdr[e].refs = refs[e];
        g.h_hdr[e].valid = 1;
    }
    // one event outside a capture: the first kernel writes the tables from its
    // arguments (no copy on the stream, so the chain stays one run of
    // programmatically dependent kernels)
    OneEventTables t1{};
    if (E == 1 && !capturing) {
        t1.hdr = g.h_hdr[0];
        t1.cell_end = g.h_cell_off[1];
        t1.nblk = g.h_blk_start[1];
        t1.set = 1;
    } else {
    // upload the per-event tables through the pinned mirror (wait until the
    // previous upload from it has been consumed)
    if (!capturing) cudaEventSynchronize(g.h_pinned_free);
    // the three tables are adjacent on the device: mirror that layout in the
    // pinned buffer and upload them with one copy
    char* hp = static_cast<char*>(g.h_pinned);
    const size_t s_hdr = sizeof(EventHdr) * E;
    const size_t s_blk = sizeof(int32_t) * (E + 1);
    const size_t s_coff = sizeof(int64_t) * (E + 1);
    const size_t o_blk = reinterpret_cast<char*>(g.blk_start) - reinterpret_cast<char*>(g.hdr);
    const size_t o_coff = reinterpret_cast<char*>(g.cell_off) - reinterpret_cast<char*>(g.hdr);
    memcpy(hp, g.h_hdr.data(), s_hdr);
    memcpy(hp + o_blk, g.h_blk_start.data(), s_blk);
    memcpy(hp + o_coff, g.h_cell_off.data(), s_coff);
    cudaMemcpyAsync(g.hdr, hp, o_coff + s_coff, cudaMemcpyHostToDevice, st);
    if (!capturing) cudaEventRecord(g.h_pinned_free, st);
    }

    // (a cross-set query's cells are its reference grid's: not a small set's)
    if (t1.set && t1.hdr.n > 0 && t1.hdr.n <= kSmallMax &&
        g.L <= (params_from && t1.hdr.rowsort ? 16 * kSmallCells : kSmallCells)) {
        const int per = (int)ceil_div(t1.hdr.n, kSmallCtas);   // at most kSmallPer * kSmallThreads
        const size_t smem = sizeof(float) * small_stage_floats(per, D);
        cudaError_t ce = cudaFuncSetAttribute(k_build_small, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (ce == cudaSuccess)
            ce = cudaFuncSetAttribute(k_build_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmemMost);
        if (ce == cudaSuccess)
            ce = launch_pdl_cluster(k_build_small, dim3(kSmallCtas), dim3(kSmallThreads), smem, st, kSmallCtas, t1,
                                    params_from ? (const EventHdr*)params_from->hdr : nullptr, per, D, g.DP, o.r, o.m,
                                    o.axes_mode, o.naxes, g.hdr, g.blk_start, g.cell_off, g.cstart, g.scalars, g.pts,
                                    g.perm, g.cell, d_status);
        if (ce == cudaSuccess) {
            g.tc_ready = false;
            g.rows_ready = false;
            return FRNN_OK;
        }
        // a cluster of this size is not portable: where it cannot be placed
        // the launch is refused, and the separate kernels build the set
        cudaGetLastError();
    }
    const size_t smem_pts = sizeof(float) * staged_floats(D);
    const EarlyPts ep{t1.hdr.refs, t1.hdr.n, t1.set};
    if (params_from) {
        if (!t1.set) {
            err = "foreign grid parameters need a one-event build";
            return FRNN_ERR_INVALID_ARG;
        }
        launch_pdl(k_begin_foreign, dim3(std::min<unsigned>(blocks_for(g.L / 4, 256), kInitBlocks)), dim3(256), 0, st,
                   t1, (const EventHdr*)params_from->hdr, g.hdr, g.blk_start, g.cell_off, g.cstart, g.scalars);
    } else {
        if (!capturing) grid_clean(g, st);
        const int sub = box_sub(g.nblk);
        launch_pdl(k_bbox, dim3((unsigned)ceil_div(g.nblk, sub)), dim3(kBuildPtsPerBlock), 0, st, g.hdr,
                   g.blk_start, g.cell_off, E, (int)g.nblk, sub, D, g.bbox, d_status, o.r, o.m, o.axes_mode, o.naxes,
                   g.cstart, g.L, g.scalars, t1);
    }
    enqueue_sort(g, smem_pts, params_from ? 1 : 0, d_status, st, ep);
    g.tc_ready = false;     // tensor-core operands describe the previous contents
    g.rows_ready = false;   // so do the row-task kernel's pair copy and tasks
    cudaError_t ce = cudaGetLastError();
    if (ce != cudaSuccess) {
        err = std::string("grid build launch failed: ") + cudaGetErrorString(ce);
        return FRNN_ERR_CUDA;
    }
    return FRNN_OK;
}

// The same build as enqueue_build, for a point set whose per-event tables
// (headers, block starts, cell offsets) some earlier work on the stream has
// already written on the device: nothing is copied from the host.
frnn_status enqueue_build_resident(GridBufs& g, const BuildOpts& o, int32_t* d_status,
                                   cudaStream_t st, std::string& err) {
    const int E = g.E, D = g.D;
    const size_t smem_pts = sizeof(float) * staged_floats(D);
    // (the array's contents are anybody's: its boxes are emptied first)
    launch_pdl(k_box_reset, dim3(blocks_for((int64_t)E * kBBoxCopies * kBBoxStride, 256)), dim3(256), 0, st, g.bbox, E);
    const int sub = box_sub(g.nblk);
    launch_pdl(k_bbox, dim3((unsigned)ceil_div(g.nblk, sub)), dim3(kBuildPtsPerBlock), 0, st, g.hdr,
               g.blk_start, g.cell_off, E, (int)g.nblk, sub, D, g.bbox, d_status, o.r, o.m, o.axes_mode, o.naxes, g.cstart,
               g.L, g.scalars, OneEventTables{});
    enqueue_sort(g, smem_pts, 0, d_status, st, EarlyPts{});
    g.tc_ready = false;
    g.rows_ready = false;
    cudaError_t ce = cudaGetLastError();
    if (ce != cudaSuccess) {
        err = std::string("grid build launch failed: ") + cudaGetErrorString(ce);
        return FRNN_ERR_CUDA;
    }
    return FRNN_OK;
}

// One thread per slot; an odd set's padding slot has no point.
__global__ void k_unsort(const float* pts, const int32_t* perm, int64_t n, int D, int DP, float* out) {
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n) return;
    float* dst = out + (int64_t)perm[s] * D;
    for (int k = 0; k < D; ++k) dst[k] = pts[pt_index(s, k, DP)];
}

cudaError_t enqueue_unsort(const GridBufs& g, float* out, cudaStream_t st) {
    const int64_t n = g.h_hdr[0].n;
    if (n > 0) k_unsort<<<blocks_for(n, 256), 256, 0, st>>>(g.pts, g.perm, n, g.D, g.DP, out);
    return cudaGetLastError();
}

}  // namespace frnn
