// pk_kernels.cu -- sm_103a kernels of the FFT power-spectrum path.
//
// Paint (Sec. 3.3.1 painting; Sec. 3.3.2 CIC / TSC / PCS B-spline windows and
// interlacing with a second mesh shifted by half a cell):
//   k_sort_count    wrap each object into the box, find its home tile (T^3
//                   cells) and its boundary class (per axis: near the low
//                   face, interior, near the high face -- 27 classes) and
//                   count objects per (tile, class) key (reductions whose
//                   result nobody waits for); sum w, w^2, |w| and max |w|.
//   k_wsum_reduce   weighted catalogs: the paint blocks' rows of weight sums
//                   added in a fixed order (run-to-run identical sums).
//   k_scan_*        exclusive scan of the key counts (uint32).
//   k_sort_scatter  write one float4 (x, y, z in the home tile's frame, w) per object
//                   at its key's cursor, advanced by the write (the scan
//                   leaves the offsets in the counts' place, too): the
//                   order inside a key is whatever order the cursors are
//                   served in, which the paint's integer deposits do not
//                   see.  No per-object rank array.
//   k_paint_tiles   one CTA per tile: gather the tile's own objects and the
//                   boundary classes of its 26 neighbours whose window reaches
//                   into it, deposit B-spline weights into shared memory as
//                   exact int64 fixed point held in two uint32 words per cell
//                   (the split point is chosen per tile so the low word can
//                   never carry; shared 32-bit atomics are ~5x faster than
//                   64-bit ones here), then write the tile once, coalesced,
//                   into the in-place r2c layout.  Where a 32-bit word holds
//                   every cell of the tile, one sweep over the candidates
//                   deposits both interlaced meshes, branch-free in sparse
//                   tiles; else one mesh per pass over staged candidates.
//                   Integer adds are order-free, and an FP32 cell is the same
//                   integers rounded once either way: the mesh is bit-identical
//                   run to run, for any object order, tile size of the plan's
//                   choice and batch.
//   k_paint_atomic  the variant without a sort: one thread per object adds
//                   each deposit with a 64-bit global atomic into a dense
//                   int64 accumulator per mesh (as order-free as the tiles);
//   k_acc_to_mesh   converts the accumulators into the r2c layout and clears
//                   them.  Cheaper than sorting for small meshes that stay in
//                   L2; the plan's paint_variant picks one of the two.
// Bin (Sec. 3.4.1, Eq. window-deconvolution):
//   k_bin           warps take whole rows of the stored half grid and visit
//                   only the binned l range; per mode: interlace combine,
//                   sinc^p compensation, |delta|^2, k bin (exact integer
//                   edges in m = |n|^2), mu bin (exact integer rule),
//                   Legendre L_2(mu) / L_4(mu) weights; runs of equal bins merged
//                   in registers, then per-CTA shared-memory histograms.
//   k_reduce_finalize  fixed-order FP64 sums of the per-CTA histograms, then
//                   normalization L^3 / (sum w)^2, shot noise, multipoles.
// Plan time (geometry only):
//   k_geom_*        exact mode counts per bin and mean k, mean mu from integer
//                   histograms over (m, mu bin), summed in FP64.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <type_traits>

#include "pk_internal.h"

namespace pk {

namespace {

constexpr int kCountThreads = 256;
constexpr unsigned kWsumBlocks = 2048;  // blocks per catalog of the passes that sum the weights
constexpr int kPaintThreads = 256;
constexpr int kBinThreads = 256;
constexpr int kBinVec = 4;            // consecutive modes per thread
// Up to this many blocks every block of the second scan pass adds up the totals
// before it itself (one load a thread at most), without a scan launch between.
constexpr int kScanDirect = 1024;
constexpr int kClasses = 27;          // boundary classes per tile
constexpr int kSegments = 75;         // (neighbour, class range) segments per tile
constexpr int kStage = 256;           // candidates staged in shared memory per batch (small: 6 CTAs / SM)
constexpr int kUploadChunk = 256;     // int64 values per parameter upload (2 KB)
// Sweep paint: tiles with at most this many candidates use branch-free
// deposits; denser tiles (e.g. uniform lattices, ~900 candidates per 16^3
// tile) were measured faster with deposits that skip cells outside the tile.
constexpr int kFlatMaxCand = 640;

// Objects [beg, end) of a catalog: off[item], off[item + 1], or [0, n) of the
// only one (off NULL: nothing to upload).
struct ItemRange {
    int64_t beg, end;
    __device__ __forceinline__ ItemRange(const int64_t *off, int64_t n, int item)
        : beg(off ? off[item] : 0), end(off ? off[item + 1] : n) {}
};

// Cell coordinate s = x * (N / L) wrapped periodically into [0, N).  Written
// with explicitly rounded intrinsics so that no FMA contraction can differ
// between the count and the scatter kernels: both must see the same s.
// FP32 positions: s is returned as s_hi + *e, where s_hi = fl(x * invH) and
// *e is the exact residual of that product plus x times the residual of
// invH = N / L; cells and tiles follow s_hi, and e is added back into the
// small tile-local coordinate (whose resolution is ~1e-6 cells), so large
// meshes do not lose the FP32 rounding of s (up to 1.2e-4 cells at N = 2048).
// Positions outside [0, L) are wrapped on s_hi with e = 0.
__device__ __forceinline__ float wrap_cells(float x, float invH, float invH_lo, int N, float *e) {
    const float n = (float)N;
    float s = __fmul_rn(x, invH);
    *e = __fadd_rn(__fmaf_rn(x, invH, -s), __fmul_rn(x, invH_lo));
    if (!(s >= 0.0f && s < n)) {
        *e = 0.0f;
        s = __fsub_rn(s, __fmul_rn(n, floorf(__fdiv_rn(s, n))));
        if (s < 0.0f) s = __fadd_rn(s, n);
        if (s >= n) s = __fsub_rn(s, n);
        if (!(s >= 0.0f && s < n)) s = 0.0f;            // NaN / inf positions
    }
    return s;
}
// The range tests compare the bit patterns of non-negative doubles as integers:
// this part runs FP64 at 1/64 of the FP32 rate, and the count and scatter of
// FP64 positions are bound by it (count and scatter of 1e6
// weighted objects 54 + 44 -> 47 + 33 us).
__device__ __forceinline__ double wrap_cells(double x, double invH, int N) {
    const double n = (double)N;
    double s = __dmul_rn(x, invH);
    // sign bit clear and s < n (NaN and infinities are not)
    if ((unsigned long long)__double_as_longlong(s) >= (unsigned long long)__double_as_longlong(n)) {
        s = __dsub_rn(s, __dmul_rn(n, floor(__ddiv_rn(s, n))));
        if (s < 0.0) s = __dadd_rn(s, n);
        if (s >= n) s = __dsub_rn(s, n);
        if (!(s >= 0.0 && s < n)) s = 0.0;
    }
    return s;
}

template <typename R>
struct Obj {
    R s[3];
    float e[3];       // residual of s (FP32 positions), 0 for FP64 positions
    float w;          // weight W (normalization: sum W)
    float a;          // painted amplitude W V (V: the painted value, 1 by default)
};

template <int DT>
struct PosReal { using type = float; };
template <>
struct PosReal<PK_F64> { using type = double; };

template <int DT>
__device__ __forceinline__ Obj<typename PosReal<DT>::type> load_obj(const void *pos, const float *w,
                                                                    const float *vals, int64_t i,
                                                                    const PaintGeom &g) {
    using R = typename PosReal<DT>::type;
    Obj<R> o;
    if (DT == PK_F32X4) {
        const float4 v = __ldg(reinterpret_cast<const float4 *>(pos) + i);
        o.s[0] = wrap_cells(v.x, g.invH, g.invH_lo, g.N, &o.e[0]);
        o.s[1] = wrap_cells(v.y, g.invH, g.invH_lo, g.N, &o.e[1]);
        o.s[2] = wrap_cells(v.z, g.invH, g.invH_lo, g.N, &o.e[2]);
        o.w = v.w;
    } else if (DT == PK_F32) {
        const float *p = reinterpret_cast<const float *>(pos) + 3 * i;
        o.s[0] = wrap_cells(__ldg(p + 0), g.invH, g.invH_lo, g.N, &o.e[0]);
        o.s[1] = wrap_cells(__ldg(p + 1), g.invH, g.invH_lo, g.N, &o.e[1]);
        o.s[2] = wrap_cells(__ldg(p + 2), g.invH, g.invH_lo, g.N, &o.e[2]);
        o.w = w ? __ldg(w + i) : 1.0f;
    } else {
        const double *p = reinterpret_cast<const double *>(pos) + 3 * i;
        o.s[0] = (R)wrap_cells(__ldg(p + 0), g.invHd, g.N);
        o.s[1] = (R)wrap_cells(__ldg(p + 1), g.invHd, g.N);
        o.s[2] = (R)wrap_cells(__ldg(p + 2), g.invHd, g.N);
        o.e[0] = o.e[1] = o.e[2] = 0.0f;
        o.w = w ? __ldg(w + i) : 1.0f;
    }
    o.a = vals ? o.w * __ldg(vals + i) : o.w;
    return o;
}

// Home tile and boundary class of one object.  Along each axis the class is
// 0 if the window reaches the tile below (c + lo < 0), 2 if it reaches the
// tile above (c + hi >= T), else 1; T >= hi - lo keeps these disjoint.
// u: the coordinate in the tile's frame (the tile, or the pair of tiles it is half
// of).  Halves, and what reaches across their seam, go by u, which the deposits are
// made of; what reaches into other frames goes by the cell of s, as with whole
// frames, so that both paint the same cells.
template <typename R, bool WANT_U>
__device__ __forceinline__ void home_key(const Obj<R> &o, const PaintGeom &g, int *tile3, float *u, int *cls) {
    int c = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const int F = g.T << g.flog;
        const int cell = min((int)o.s[a], g.N - 1);        // s >= 0: truncation is the floor
        int t = (int)(((unsigned)cell * g.inv_F) >> 20);            // cell / F (see PaintGeom)
        const int cl = cell - t * F;
        if (g.flog || WANT_U) u[a] = (float)(o.s[a] - (R)(t * F)) + o.e[a];
        bool below = cl < -g.lo, above = cl >= F - g.hi;
        if (g.flog) {
            const int cu = min(max(__float2int_rd(u[a]), 0), F - 1);
            t = 2 * t + (cu >= g.T);
            if (cu >= g.T) below = cu - g.T < -g.lo;
            else above = cu >= g.T - g.hi;
        }
        tile3[a] = t;
        c = c * 3 + (below ? 0 : above ? 2 : 1);
    }
    *cls = c;
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}

// Block reduction of the weight sums: sum W, sum (W V)^2, sum |W V| of the
// block's objects into its row wpart[(item * gridDim.x + block) * 3 + k]
// (summed over the blocks in a fixed order by k_wsum_reduce, so the sums do
// not depend on which block finishes first); wmax[item].x = max |W V| (float
// bits, order-free), with W the weight and W V the painted amplitude.
// .y = 1 if any W V is negative.  Unweighted: wsums[4 * item + {0,1,2}] += n,
// max = 1.
__device__ __forceinline__ void flush_wsums(double sw, double sw2, double swa, float mw, bool neg, bool weighted,
                                            int item, int64_t n_item, double *__restrict__ wsums,
                                            double *__restrict__ wpart, uint4 *__restrict__ wmax) {
    if (weighted) {
        __shared__ double red[3][kCountThreads / 32];
        __shared__ float redm[kCountThreads / 32];
        sw = warp_sum(sw);
        sw2 = warp_sum(sw2);
        swa = warp_sum(swa);
        mw = warp_max(mw);
        const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
        if (lane == 0) {
            red[0][wid] = sw;
            red[1][wid] = sw2;
            red[2][wid] = swa;
            redm[wid] = mw;
        }
        const int any_neg = __syncthreads_or(neg);
        if (threadIdx.x < 3) {
            double t = 0.0;
            for (int k = 0; k < kCountThreads / 32; ++k) t += red[threadIdx.x][k];
            wpart[((size_t)item * gridDim.x + blockIdx.x) * 3 + threadIdx.x] = t;
        } else if (threadIdx.x == 3) {
            float m = 0.0f;
            for (int k = 0; k < kCountThreads / 32; ++k) m = fmaxf(m, redm[k]);
            atomicMax(&wmax[item].x, __float_as_uint(m));
        } else if (threadIdx.x == 4 && any_neg) {
            atomicOr(&wmax[item].y, 1u);
        }
    } else if (blockIdx.x == 0 && threadIdx.x < 3) {
        atomicAdd(wsums + 4 * item + threadIdx.x, (double)n_item);   // exact below 2^53
        if (threadIdx.x == 0) atomicMax(&wmax[item].x, __float_as_uint(1.0f));
    }
}

// Fixed-order sum of the blocks' weight-sum rows of catalog blockIdx.x:
// thread t adds rows t, t + 256, ... in turn, then a fixed tree; the result
// is added to wsums[4 * item + k] (one writer per value).  wmax[item].z: the
// mean |W V| (float bits), from which the tile paint guesses a tile's sum.
__global__ void __launch_bounds__(256)
k_wsum_reduce(const double *wpart, int nblk, const int64_t *__restrict__ item_off, int64_t n_one,
              double *__restrict__ wsums, uint4 *__restrict__ wmax) {
    grid_wait(item_off);
    __shared__ double red[3][256];
    const int item = blockIdx.x, t = threadIdx.x;
    double a[3] = {0.0, 0.0, 0.0};
    for (int b = t; b < nblk; b += 256)
#pragma unroll
        for (int k = 0; k < 3; ++k) a[k] += wpart[((size_t)item * nblk + b) * 3 + k];
#pragma unroll
    for (int k = 0; k < 3; ++k) red[k][t] = a[k];
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if (t < h)
#pragma unroll
            for (int k = 0; k < 3; ++k) red[k][t] += red[k][t + h];
        __syncthreads();
    }
    if (t < 3) wsums[4 * item + t] += red[t][0];
    if (t == 3) {
        const ItemRange range(item_off, n_one, item);
        const float n = (float)(range.end - range.beg);
        // ten bits of it: the rounding of the sum, and so the order of the objects, is not seen
        wmax[item].z = __float_as_uint(n > 0.0f ? (float)red[2][0] / n : 0.0f) & 0xffffe000u;
    }
}

// Key of an object: (catalog, home tile, boundary class).
template <typename R, bool WANT_U>
__device__ __forceinline__ int64_t sort_key(const Obj<R> &o, const PaintGeom &g, int64_t kbase, float *u) {
    int t3[3], cls;
    home_key<R, WANT_U>(o, g, t3, u, &cls);
    return kbase + (((int64_t)t3[0] * g.ntx + t3[1]) * g.ntx + t3[2]) * kClasses + cls;
}

// Tile sort, pass 1: key counts, plus the weight sums.
template <int DT, bool WEIGHTED>
__global__ void __launch_bounds__(kCountThreads)
k_sort_count(const void *__restrict__ pos, const float *__restrict__ w, const float *__restrict__ vals,
             const int64_t *__restrict__ item_off, int64_t n_one, PaintGeom g, uint32_t *__restrict__ count,
             double *__restrict__ wsums, double *__restrict__ wpart, uint4 *__restrict__ wmax) {
    grid_wait(pos, w, vals, item_off);
    using R = typename PosReal<DT>::type;
    const int item = blockIdx.y;
    const ItemRange range(item_off, n_one, item);
    const int64_t beg = range.beg, end = range.end;
    const int64_t kbase = (int64_t)item * g.ntiles * kClasses;
    double sw = 0.0, sw2 = 0.0, swa = 0.0;
    float mw = 0.0f;
    bool neg = false;
    for (int64_t i = beg + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < end;
         i += (int64_t)gridDim.x * blockDim.x) {
        const Obj<R> o = load_obj<DT>(pos, w, vals, i, g);
        float u[3];
        atomicAdd(count + sort_key<R, false>(o, g, kbase, u), 1u);   // result unused: a reduction
        if (WEIGHTED) {
            const double ad = (double)o.a;
            sw += (double)o.w;
            sw2 += ad * ad;
            swa += fabs(ad);
            mw = fmaxf(mw, fabsf(o.a));
            neg |= o.a < 0.0f;
        }
    }
    flush_wsums(sw, sw2, swa, mw, neg, WEIGHTED, item, end - beg, wsums, wpart, wmax);
}

// Tile sort, pass 2: each object takes the slot at its key's cursor (the scan's
// offsets, copied over the counts) and advances it.  Two scattered accesses per
// object, the returning atomic and the 16-byte write: the L1 takes one 128-byte
// line of a scattered warp access per clock, and the offset and its successor
// read beside a decremented count were two more (1e7 objects at 512^3: 200 -> 176
// us; 1.3e8 at 1024^3: 4.66 -> 3.72 ms).  k_paint_tiles checks that every cursor
// ends at the next key's offset.  More objects per thread with every load and atomic
// issued before the first use ran slower (two, four, eight: 4, 10, 23 %).
template <int DT>
__global__ void __launch_bounds__(kCountThreads)
k_sort_scatter(const void *__restrict__ pos, const float *__restrict__ w, const float *__restrict__ vals,
               const int64_t *__restrict__ item_off, int64_t n_one, PaintGeom g, uint32_t *__restrict__ cursor,
               float4 *__restrict__ sorted, uint32_t ntot, int *__restrict__ err) {
    grid_wait(pos, w, vals, item_off);
    using R = typename PosReal<DT>::type;
    const int item = blockIdx.y;
    const ItemRange range(item_off, n_one, item);
    const int64_t beg = range.beg, end = range.end;
    const int64_t kbase = (int64_t)item * g.ntiles * kClasses;
    for (int64_t i = beg + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < end;
         i += (int64_t)gridDim.x * blockDim.x) {
        const Obj<R> o = load_obj<DT>(pos, w, vals, i, g);
        float u[3];
        const int64_t key = sort_key<R, true>(o, g, kbase, u);
        const uint32_t slot = atomicAdd(cursor + key, 1u);
        if (slot >= ntot) {                      // count and scatter disagree: never write
            atomicOr(err, 2);
            continue;
        }
        sorted[slot] = make_float4(u[0], u[1], u[2], o.a);
    }
}

// ---- exclusive scan of uint32 counts (totals < 2^32) or uint64 weights ----
// out and copy (COPY: a second place for the results) may alias in: every
// thread reads its own elements before writing them.
template <typename T, bool COPY>
__global__ void __launch_bounds__(kScanThreads)
k_scan_blocks(const T *in, int64_t n, T *out, T *bsum, T *copy) {
    grid_wait();
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanPer;
    T v[kScanPer];
    T s = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        v[k] = base + k < n ? in[base + k] : (T)0;
        s += v[k];
    }
    T total;
    T run = block_exclusive_scan<T>(s, &total);
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        if (base + k < n) {
            out[base + k] = run;
            if constexpr (COPY) copy[base + k] = run;
        }
        run += v[k];
    }
    if (threadIdx.x == 0) bsum[blockIdx.x] = total;
}

// DIRECT: bsum holds the blocks' totals (every block adds up those before it);
// else their exclusive scan with the total in bsum[nb].
template <typename T, bool COPY, bool DIRECT>
__global__ void __launch_bounds__(kScanThreads)
k_scan_add(T *__restrict__ out, int64_t n, const T *bsum, int nb, T *__restrict__ copy) {
    grid_wait();
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanPer;
    T add;
    if constexpr (DIRECT) {
        __shared__ T wsum[kScanThreads / 32];
        T t = (T)0;
        for (int k = threadIdx.x; k < (int)blockIdx.x; k += kScanThreads) t += bsum[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = t;
        __syncthreads();
        add = (T)0;
#pragma unroll
        for (int k = 0; k < kScanThreads / 32; ++k) add += wsum[k];
    } else {
        add = bsum[blockIdx.x];
    }
#pragma unroll
    for (int k = 0; k < kScanPer; ++k)
        if (base + k < n) {
            const T v = out[base + k] + add;
            out[base + k] = v;
            if constexpr (COPY) copy[base + k] = v;
        }
    if (DIRECT ? blockIdx.x == nb - 1 && threadIdx.x == 0 : blockIdx.x == 0 && threadIdx.x == 0)
        out[n] = DIRECT ? add + bsum[nb - 1] : bsum[nb];
}

// ---- tile paint ----
// Per-axis B-spline weights of order P at node-relative coordinate u (cells):
// nodes base .. base + P - 1.  Every multiply-add is written out: left to the
// compiler, 0.75 - g g was contracted in some instances of k_paint_tiles and not
// in others, so that an object's cells depended on the instance (weighted or
// not, one mesh or two, tile edge) that painted them.
template <int P>
__device__ __forceinline__ void spline_weights(float u, int &base, float *wt) {
    if (P == 2) {                       // CIC
        const float f0 = floorf(u);
        const float f = u - f0;
        base = (int)f0;
        wt[0] = 1.0f - f;
        wt[1] = f;
    } else if (P == 3) {                // TSC: nearest node base + 1
        const float f0 = floorf(u - 0.5f);
        const float g = u - (f0 + 1.0f);    // in [-1/2, 1/2)
        base = (int)f0;
        const float a = 0.5f - g, b = 0.5f + g;
        wt[0] = 0.5f * a * a;
        wt[1] = __fmaf_rn(-g, g, 0.75f);
        wt[2] = 0.5f * b * b;
    } else {                            // PCS
        const float f0 = floorf(u);
        const float f = u - f0, r = 1.0f - f;
        base = (int)f0 - 1;
        const float f2 = f * f, r2 = r * r;
        wt[0] = (1.0f / 6.0f) * r2 * r;
        wt[1] = (1.0f / 6.0f) * __fmaf_rn(3.0f * f2, f, __fmaf_rn(-6.0f, f2, 4.0f));
        wt[2] = (1.0f / 6.0f) * __fmaf_rn(3.0f * r2, r, __fmaf_rn(-6.0f, r2, 4.0f));
        wt[3] = (1.0f / 6.0f) * f2 * f;
    }
}

// Fixed-point split of one tile: deposit q = round(v) (v = w W 2^S) is held as
// hi * 2^B + lo with lo in [0, 2^B) (FP64 meshes: [0, 2^B]); the cell keeps sum(lo) and
// sum(hi) in two uint32 words.  With at most `ncand` deposits per cell, sum(lo) <=
// ncand 2^B < 2^32 and |sum(hi)| <= ncand (hmax + 1) < 2^31 by construction.
struct Split {
    int B;            // split bit (1 .. 30, FP64 meshes 1 .. 22)
    float twoB;       // 2^B
    unsigned twoB_u;  // 2^B as an integer
    float inv2B;      // 2^-B
    float hi_scale;   // 2^(B - S): weight units of one hi count
    int fast;         // 1: split when needed; 0: this tile uses 64-bit shared atomics instead
};

// round(vxy wz) as a two's complement word, the exact product rounded once, where
// fma_exact says so: one FMA against 2^23 (UNIT: [0, 2^23)) or 1.5 2^23 ([-2^22,
// 2^22)), whose bits hold the integer.
template <bool UNIT>
__device__ __forceinline__ unsigned quantize_fma(float vxy, float wz) {
    return __float_as_uint(fmaf(vxy, wz, UNIT ? 8388608.0f : 12582912.0f)) - (UNIT ? 0x4B000000u : 0x4B400000u);
}
template <bool UNIT>
__device__ __forceinline__ bool fma_exact(unsigned q) {
    return (UNIT ? q : q + (1u << 22)) < (1u << 23);
}
// Any |v| < 2^31 (UNIT: deposits known to be below 2^23): from 2^22 on the FP32 product
// holds two binary places at most and is converted (a product converted at any size
// was rounded twice).
template <bool UNIT>
__device__ __forceinline__ unsigned quantize(float vxy, float wz) {
    const unsigned q = quantize_fma<UNIT>(vxy, wz);
    return UNIT || fma_exact<UNIT>(q) ? q : (unsigned)__float2int_rn(vxy * wz);
}

// MODE 2: the tile's cells fit one word each (see the sweep in k_paint_tiles):
// one rounding and one 32-bit shared atomic per cell.  MODE 1: lo words with a
// split into hi * 2^B + lo for the rare large or negative deposit.  MODE 0:
// 64-bit shared atomics (dense tiles).  Meshes of M = float: the same integer in
// every mode, so that a cell does not depend on the way its tile is painted.
// (M = double has modes 0 and 1 only; the split rounds deposits from 2^B on to FP32
// first.)
template <int P, int MODE, int TC, bool UNIT, typename M>
__device__ __forceinline__ void deposit(unsigned *lo, unsigned *hi, unsigned long long *acc64,
                                        const Split &sp, int T, float x, float y, float z, float ws) {
    int bx, by, bz;
    float wx[P], wy[P], wz[P];
    spline_weights<P>(x, bx, wx);
    spline_weights<P>(y, by, wy);
    spline_weights<P>(z, bz, wz);
#pragma unroll
    for (int a = 0; a < P; ++a) {
        const int cx = bx + a;
        if ((unsigned)cx >= (unsigned)T) continue;
        const float vx = ws * wx[a];
#pragma unroll
        for (int b = 0; b < P; ++b) {
            const int cy = by + b;
            if ((unsigned)cy >= (unsigned)T) continue;
            const float vxy = vx * wy[b];
            const int row = (cx * T + cy) * T;
#pragma unroll
            for (int c = 0; c < P; ++c) {
                const int cz = bz + c;
                if ((unsigned)cz >= (unsigned)T) continue;
                if (MODE == 2) {
                    atomicAdd(lo + row + cz, quantize<UNIT>(vxy, wz[c]));
                } else if (MODE == 1 && sizeof(M) == 4) {
                    // lo and hi words of the integer (beyond 2^31, where FP32 products are
                    // multiples of 256, split as they are: exact for B <= 30)
                    unsigned q = quantize_fma<UNIT>(vxy, wz[c]);
                    int hf = 0;
                    if (__builtin_expect(!fma_exact<UNIT>(q), 0)) {
                        float v = vxy * wz[c];
                        if (fabsf(v) >= 2147483648.0f) {
                            const float h = floorf(v * sp.inv2B);
                            v = fmaf(-h, sp.twoB, v);
                            hf = (int)h;
                        }
                        q = (unsigned)__float2int_rn(v);
                    }
                    atomicAdd(lo + row + cz, q & (sp.twoB_u - 1u));
                    if (q >= sp.twoB_u || hf != 0) atomicAdd(hi + row + cz, (unsigned)(((int)q >> sp.B) + hf));
                } else if (MODE == 1) {
                    // 2^23 + round(v) in one FMA; its bits minus 0x4B000000 are
                    // round(v) whenever 0 <= round(v) < 2^B (B <= 22): the
                    // common case, one 32-bit shared atomic.
                    const unsigned q = __float_as_uint(fmaf(vxy, wz[c], 8388608.0f)) - 0x4B000000u;
                    if (q < sp.twoB_u) {
                        atomicAdd(lo + row + cz, q);
                    } else {              // large or negative deposit: split hi * 2^B + lo
                        const float v = vxy * wz[c];
                        const float hf = floorf(v * sp.inv2B);
                        const float lf = fmaf(-hf, sp.twoB, v);          // exact, in [0, 2^B)
                        const unsigned ql = __float_as_uint(lf + 8388608.0f) - 0x4B000000u;
                        atomicAdd(lo + row + cz, ql);
                        if (hf != 0.0f)
                            atomicAdd(hi + row + cz, (unsigned)(__float_as_int(hf + 12582912.0f) - 0x4B400000));
                    }
                } else {
                    const unsigned f = quantize_fma<UNIT>(vxy, wz[c]);
                    const long long q = sizeof(M) == 4 && fma_exact<UNIT>(f) ? (long long)(int)f : __float2ll_rn(vxy * wz[c]);
                    if (q) atomicAdd(acc64 + row + cz, (unsigned long long)q);
                }
            }
        }
    }
}

// MODE 2 deposit without branches: every one of the P^3 cells gets its
// atomic on sm[idx].  Per axis, an offset outside the tile is a large negative
// sentinel, so the index sum of a cell outside the tile is negative and
// min((unsigned)sum, trash) sends it to the lane's scratch word sm[trash]
// (never read); the lanes of a warp never split on tile bounds.  cell0: the
// first word of the mesh's cells in sm.
template <int P, int TC, bool UNIT>
__device__ __forceinline__ void deposit_flat(unsigned *sm, int cell0, unsigned trash, int T, float x, float y,
                                             float z, float ws) {
    int bx, by, bz;
    float wx[P], wy[P], wz[P];
    spline_weights<P>(x, bx, wx);
    spline_weights<P>(y, by, wy);
    spline_weights<P>(z, bz, wz);
    const int TT = TC > 0 ? TC : T;
    constexpr int kOut = -(1 << 24);
    int ox[P], oy[P], oz[P];
#pragma unroll
    for (int a = 0; a < P; ++a) {
        const int cx = bx + a, cy = by + a, cz = bz + a;
        ox[a] = (unsigned)cx < (unsigned)TT ? cell0 + cx * TT * TT : kOut;
        oy[a] = (unsigned)cy < (unsigned)TT ? cy * TT : kOut;
        oz[a] = (unsigned)cz < (unsigned)TT ? cz : kOut;
    }
#pragma unroll
    for (int a = 0; a < P; ++a) {
        // TSC: skip an x plane that lies wholly outside the tile (measured
        // faster for TSC, slower for PCS, whose lanes diverge more)
        if (P == 3 && ox[a] == kOut) continue;
        const float vxw = ws * wx[a];
#pragma unroll
        for (int b = 0; b < P; ++b) {
            const float vxy = vxw * wy[b];
            const int oab = ox[a] + oy[b];
#pragma unroll
            for (int c = 0; c < P; ++c) {
                atomicAdd(sm + min((unsigned)(oab + oz[c]), trash), quantize<UNIT>(vxy, wz[c]));
            }
        }
    }
}

// Blocks of a tile and its surroundings: 2^SH cells along each axis (twice that in
// tiles wider than 16), from one block below the tile on, at most NB per axis.  A
// cell's deposits come from an open interval of P cells per axis, so from SPAN
// neighbouring blocks at most.
template <int SH_, int NB_, int SPAN_, int SPAN_WIDE_>
struct Blocks {
    static constexpr int NB = NB_, Count = NB * NB * NB;
    __device__ static __forceinline__ int of(float x, float y, float z, bool wide) {
        const int sh = wide ? SH_ + 1 : SH_;
        const auto along = [&](float v) { return min(max(__float2int_rd(v) + (1 << sh), 0) >> sh, NB - 1); };
        return (along(x) * NB + along(y)) * NB + along(z);
    }
    // The largest sum of the counters that one cell's deposits come from, of this
    // thread's share of the cells.
    __device__ static __forceinline__ float most(const unsigned *blk, bool wide) {
        const int span = wide ? SPAN_WIDE_ : SPAN_, ends = NB - span + 1;
        float m = 0.0f;
        for (int c = threadIdx.x; c < ends * ends * ends; c += blockDim.x) {
            const unsigned *b = blk + (c / (ends * ends) * NB + c / ends % ends) * NB + c % ends;
            float n = 0.0f;
            for (int i = 0; i < span; ++i)
                for (int j = 0; j < span; ++j)
                    for (int k = 0; k < span; ++k) n += (float)b[(i * NB + j) * NB + k];
            m = fmaxf(m, n);
        }
        return m;
    }
};
// Counters that fit beside the cells without costing a CTA per SM (TSC blocks of 3 cells
// did: 816 -> 858 us for 2e7 objects at 512^3), and those that take the cells' place:
// 2 x 2 x 2 blocks are 64 cells (CIC) or 512, 3 x 3 x 3 are 216.  The smaller windows lie
// within the larger ones: what fits by the larger fits by the smaller.
template <int P>
using CoarseBlocks = typename std::conditional<P == 2, Blocks<1, 10, 2, 2>, Blocks<2, 6, 2, 2>>::type;
template <int P>
using FineBlocks = typename std::conditional<P == 2, Blocks<1, 10, 2, 2>, Blocks<1, 10, 3, 2>>::type;

// ---- one-sweep paint of 16^3 tiles into a padded layout (unit weights, TSC and PCS) ----
// Shared layout: cell (x, y, z) of the tile's mesh m at word
//   m * kWords + x * kXS + y * kYS + kZlo + z,
// where every row of z holds a halo [-kZlo, kYS - kZlo) wide enough for every
// deposit of every window that reaches the tile along z (objects of the tile
// and the boundary classes of its neighbours, both meshes), so a deposit
// needs no bounds test along z; a window wholly outside the tile along z (the
// other mesh of a boundary candidate) and a row outside the tile along x or
// y are skipped by predicates (a word shared by many lanes of one atomic
// instruction would serialize them).  Each deposit is then one FFMA, one
// IADD and one 32-bit shared atomic at an immediate offset from its row.
//
// The strides are odd: candidates arrive grouped by (tile, boundary class),
// and on a lattice-like catalog a warp's lanes share z offsets, so with even
// strides (plane 384 = 0 mod 32 words, rows 24) their deposits fell on a few
// banks (5.1 shared wavefronts per atomic instruction measured on a
// Zel'dovich lattice at 0.125 objects per cell); rows of 25 and planes of 401
// words spread them over all 32 banks (PCS + interlacing 1.93 -> 1.22 ms on
// that lattice at 512^3, 1.01 -> 0.92 ms on the log-normal catalog; TSC
// with rows of 21 and planes of 337: 1.02 -> 0.69 and 0.537 -> 0.526 ms).
template <int P>
struct SweepLayout {
    static constexpr int T = 16;
    static constexpr int Zlo = P == 4 ? 4 : P - 1;    // z halo below the tile
    static constexpr int YS = P == 4 ? 25 : (P == 3 ? 21 : 19);   // row stride
    static constexpr int XS = P == 4 ? 401 : (P == 3 ? 337 : 305);  // plane stride
    static constexpr int Words = T * XS;              // one mesh (a multiple of 4 words)
    // first nodes of the windows that reach the tile along z: any other
    // window lies wholly outside it and deposits nothing
    static constexpr int BzMin = -Zlo, BzMax = YS - Zlo - P;
    static_assert(Zlo >= P - 1 && BzMax >= T - 1, "the halo must hold every window that reaches the tile");
    static_assert(XS >= T * YS && Words % 4 == 0, "rows inside their plane; 16-byte zeroing");
};

// Deposits of one candidate (tile-frame coordinates x, y, z in cells, weight
// ws already scaled by 2^S) into the mesh whose first word is sm.  A first
// node bz outside [BzMin, BzMax] only occurs for a window lying wholly
// outside the tile along z: it deposits nothing.
template <int P, bool UNIT>
__device__ __forceinline__ void sweep_deposit(unsigned *sm, float x, float y, float z, float ws) {
    using Lay = SweepLayout<P>;
    constexpr int kOut = 1 << 20;                     // > Words: marks a row outside the tile
    int bx, by, bz;
    float wx[P], wy[P], wz[P];
    spline_weights<P>(x, bx, wx);
    spline_weights<P>(y, by, wy);
    spline_weights<P>(z, bz, wz);
    if (bz < Lay::BzMin || bz > Lay::BzMax) return;
    bz += Lay::Zlo;
    int ox[P], oy[P];
#pragma unroll
    for (int a = 0; a < P; ++a) {
        ox[a] = (unsigned)(bx + a) < (unsigned)Lay::T ? (bx + a) * Lay::XS : kOut;
        oy[a] = (unsigned)(by + a) < (unsigned)Lay::T ? (by + a) * Lay::YS + bz : kOut;
    }
#pragma unroll
    for (int a = 0; a < P; ++a) {
        const float vxw = ws * wx[a];
#pragma unroll
        for (int b = 0; b < P; ++b) {
            const float vxy = vxw * wy[b];
            const int ro = ox[a] + oy[b];
            if (ro < Lay::Words) {           // a row inside the tile (no deposit otherwise)
                unsigned *row = sm + ro;
#pragma unroll
                for (int c = 0; c < P; ++c)
                    atomicAdd(row + c, quantize<UNIT>(vxy, wz[c]));
            }
        }
    }
}

// Value of a one-word cell: two's complement where deposits can be negative.
template <typename M, bool UNIT>
__device__ __forceinline__ M word_value(unsigned w, bool sgn) {
    if constexpr (UNIT) return (M)w;
    else return sgn ? (M)(int)w : (M)w;
}

// Write mesh words of the padded layout (cells of the tile only) to the r2c
// mesh: two cells per thread and store, as flush_tile (two 32-bit loads: the
// odd strides leave a pair of cells 4-byte aligned only).
template <typename M, int P, bool UNIT>
__device__ __forceinline__ void sweep_flush(const unsigned *sm, bool sgn, float inv_scale, M *__restrict__ dst0, int N,
                                            long long pitch, int accumulate) {
    using Lay = SweepLayout<P>;
    using M2 = typename std::conditional<sizeof(M) == 4, float2, double2>::type;
    constexpr int T = Lay::T, hT = T / 2;
    constexpr int planes = kPaintThreads / (hT * T);          // x planes per pass
    static_assert(kPaintThreads % (hT * T) == 0 && T % planes == 0, "flush mapping");
    const int t = threadIdx.x;
    const int cz = 2 * (t % hT);
    const int cy = (t / hT) % T;
    const int cx0 = t / (hT * T);
    int w = cx0 * Lay::XS + cy * Lay::YS + Lay::Zlo + cz;
    M *dst = dst0 + ((long long)cx0 * N + cy) * pitch + cz;
    const long long gstep = (long long)planes * N * pitch;
#pragma unroll 2
    for (int k = 0; k < T / planes; ++k, w += planes * Lay::XS, dst += gstep) {
        M2 v;
        v.x = word_value<M, UNIT>(sm[w], sgn) * (M)inv_scale;
        v.y = word_value<M, UNIT>(sm[w + 1], sgn) * (M)inv_scale;
        M2 *d2 = reinterpret_cast<M2 *>(dst);
        if (accumulate) {
            const M2 o = *d2;
            v.x += o.x;
            v.y += o.y;
        }
        *d2 = v;
    }
}

// Correctly rounded int64 -> float without the 64-bit conversion instruction.
__device__ __forceinline__ float ll_to_float_rn(long long q) {
    if (q == (long long)(int)q) return (float)(int)q;
    const unsigned long long u = q < 0 ? 0ull - (unsigned long long)q : (unsigned long long)q;
    const int nb = 64 - __clzll((long long)u);
    float f;
    if (nb <= 24) {
        f = (float)(unsigned)u;
    } else {
        const int sh = nb - 24;
        unsigned long long m = u >> sh;
        const unsigned long long rem = u & ((1ull << sh) - 1ull);
        const unsigned long long half = 1ull << (sh - 1);
        if (rem > half || (rem == half && (m & 1ull))) ++m;
        f = (float)(unsigned)m * __uint_as_float((unsigned)(127 + sh) << 23);
    }
    return q < 0 ? -f : f;
}

// Cell value in weight units from its fixed-point words: the cell's integer rounded
// once, as in one-word cells (FP64: exact, it has far fewer than 53 bits).
template <typename M>
__device__ __forceinline__ M cell_value(unsigned lo, unsigned hi, unsigned long long a64, const Split &sp,
                                        float inv_scale);
template <>
__device__ __forceinline__ float cell_value<float>(unsigned lo, unsigned hi, unsigned long long a64,
                                                   const Split &sp, float inv_scale) {
    return ll_to_float_rn(sp.fast ? ((long long)(int)hi << sp.B) + (long long)lo : (long long)a64) * inv_scale;
}
// hi sh + lo sl for powers of two sl <= sh <= 2^52 sl, rounded once: 32-bit words
// put into the low half of the double 2^52 s become 2^52 s + word s without a
// conversion, and the sum of the offsets leaves again in the first of the two
// additions (exact).  Conversions and products took twice as many operations of
// the FP64 pipe, which bounds the write-out of FP64 meshes.
__device__ __forceinline__ double words_value(unsigned lo, int hi, float sl, float sh) {
    const int el = ((__float_as_int(sl) >> 23) + (1023 - 127 + 52)) << 20;
    const int eh = ((__float_as_int(sh) >> 23) + (1023 - 127 + 52)) << 20;
    const double off = __hiloint2double(eh, 0x80000000) + __hiloint2double(el, 0);
    return (__hiloint2double(eh, hi ^ 0x80000000) - off) + __hiloint2double(el, (int)lo);
}

template <>
__device__ __forceinline__ double cell_value<double>(unsigned lo, unsigned hi, unsigned long long a64,
                                                     const Split &sp, float inv_scale) {
    if (sp.fast) return words_value(lo, (int)hi, inv_scale, sp.hi_scale);
    return words_value((unsigned)a64, (int)(a64 >> 32), inv_scale, inv_scale * 4294967296.0f);
}

// 2^k for -126 <= k <= 127, exactly (the fixed-point scales: S <= 40, B <= 22).
__device__ __forceinline__ float pow2f(int k) { return __uint_as_float((unsigned)(127 + k) << 23); }

__device__ __forceinline__ int ceil_log2(unsigned x) {     // x >= 1
    return x <= 1u ? 0 : 32 - __clz(x - 1u);
}

// Neighbour offset (-1, 0, +1 per axis) of gather segment s: s = (ax * 5 + ay)
// * 3 + az with ax, ay over the 5 (offset, class) pairs -- offset -1, three
// classes at offset 0, offset +1 -- and az over the 3 z offsets.
__device__ __forceinline__ int seg_dx(int s) { const int ax = s / 15; return ax == 0 ? -1 : (ax == 4 ? 1 : 0); }
__device__ __forceinline__ int seg_dy(int s) { const int ay = (s / 3) % 5; return ay == 0 ? -1 : (ay == 4 ? 1 : 0); }
__device__ __forceinline__ int seg_dz(int s) { return s % 3 - 1; }

// Where a tile lies in its frame: the tile itself, or (half > 0) a pair of tiles along
// each axis, of which it is the lower or the upper one.  Coordinates of candidates, and
// their shifts to the second mesh, are rounded in the frame; at() then takes the frame
// coordinate to the tile's, exactly (in an upper half it is 5 or more).
template <int TC>
struct TileFrame {
    int T, bits;                                      // bits 0 .. 2: upper half along x, y, z; 3: halves
    __device__ __forceinline__ TileFrame(int T_, int flog, int tx, int ty, int tz)
        : T(T_), bits(flog ? 8 | (tx & 1) | (ty & 1) << 1 | (tz & 1) << 2 : 0) {}
    // Neighbour d's frame relative to this one, in cells.
    __device__ __forceinline__ float shift(int d, int axis) const {
        if (TC > 0) return (float)(d * TC);
        return (float)(bits & 8 ? (((bits >> axis & 1) + d) >> 1) * 2 * T : d * T);
    }
    __device__ __forceinline__ float at(float v, int axis) const {
        if (TC > 0) return v;
        return bits >> axis & 1 ? v - (float)T : v;
    }
};

// Candidate k of the tile (k < s_pre[kSegments]) in this tile's frame
// (segment shift added), weight scaled by 2^S.
template <int TC>
__device__ __forceinline__ float4 fetch_candidate(const float4 *sorted, const uint32_t *s_beg,
                                                  const uint32_t *s_pre, const TileFrame<TC> &fr, uint32_t k, float scale) {
    int lo_s = 0, hi_s = kSegments;                   // s_pre[lo_s] <= k < s_pre[hi_s]
    while (hi_s - lo_s > 1) {
        const int mid = (lo_s + hi_s) >> 1;
        if (s_pre[mid] <= k) lo_s = mid;
        else hi_s = mid;
    }
    const float4 v = sorted[s_beg[lo_s] + (k - s_pre[lo_s])];
    return make_float4(v.x + fr.shift(seg_dx(lo_s), 0), v.y + fr.shift(seg_dy(lo_s), 1), v.z + fr.shift(seg_dz(lo_s), 2),
                       v.w * scale);
}

// Copy candidates [k0, k0 + n) of the tile into shared memory.
template <int TC>
__device__ __forceinline__ void stage_candidates(const float4 *sorted, const uint32_t *s_beg,
                                                 const uint32_t *s_pre, const TileFrame<TC> &fr, uint32_t k0, uint32_t n,
                                                 float scale, float4 *cand) {
    for (uint32_t j = threadIdx.x; j < n; j += blockDim.x)
        cand[j] = fetch_candidate(sorted, s_beg, s_pre, fr, k0 + j, scale);
}

template <int P, int MODE, int TC, bool UNIT, typename M>
__device__ __forceinline__ void deposit_staged(const float4 *cand, uint32_t n, unsigned *lo, unsigned *hi,
                                               unsigned long long *acc64, const Split &sp, int T, const TileFrame<TC> &fr, float sh) {
    for (uint32_t j = threadIdx.x; j < n; j += blockDim.x) {
        const float4 v = cand[j];
        deposit<P, MODE, TC, UNIT, M>(lo, hi, acc64, sp, T, fr.at(v.x + sh, 0), fr.at(v.y + sh, 1), fr.at(v.z + sh, 2), v.w);
    }
}

template <int P, int TC, bool UNIT, typename M>
__device__ __forceinline__ void deposit_any(const float4 *cand, uint32_t n, unsigned *lo, unsigned *hi,
                                            unsigned long long *acc64, const Split &sp, int T, const TileFrame<TC> &fr, float sh) {
    if (sp.fast) deposit_staged<P, 1, TC, UNIT, M>(cand, n, lo, hi, acc64, sp, T, fr, sh);
    else deposit_staged<P, 0, TC, UNIT, M>(cand, n, lo, hi, acc64, sp, T, fr, sh);
}

// Write one tile's cells to the mesh (r2c layout, rows of T cells along z at
// the given pitch).  Sources: lo alone
// (one-word cells), lo + hi (split), or acc64 (64-bit cells).  Even T: two cells per thread with 8- (FP32) or 16-byte
// (FP64) stores; the row pitch and tile origin are even, so they are aligned.
template <typename M, int TC, bool UNIT>
__device__ __forceinline__ void flush_tile(const unsigned *lo, const unsigned *hi, const unsigned long long *acc64,
                                           const Split &sp, bool sgn, float inv_scale, M *__restrict__ mb, int T, int N,
                                           long long pitch, int accumulate) {
    using M2 = typename std::conditional<sizeof(M) == 4, float2, double2>::type;
    const auto cell = [&](int c) -> M {
        if (acc64) return cell_value<M>(0u, 0u, acc64[c], sp, inv_scale);
        if (hi) return cell_value<M>(lo[c], hi[c], 0ull, sp, inv_scale);
        return word_value<M, UNIT>(lo[c], sgn) * (M)inv_scale;
    };
    const auto pair = [&](int c) -> M2 {        // cells c, c + 1 (c even)
        M2 v;
        if (acc64) {
            v.x = cell_value<M>(0u, 0u, acc64[c], sp, inv_scale);
            v.y = cell_value<M>(0u, 0u, acc64[c + 1], sp, inv_scale);
        } else {
            const uint2 l2 = *reinterpret_cast<const uint2 *>(lo + c);
            if (hi) {
                const uint2 h2 = *reinterpret_cast<const uint2 *>(hi + c);
                v.x = cell_value<M>(l2.x, h2.x, 0ull, sp, inv_scale);
                v.y = cell_value<M>(l2.y, h2.y, 0ull, sp, inv_scale);
            } else {
                v.x = word_value<M, UNIT>(l2.x, sgn) * (M)inv_scale;
                v.y = word_value<M, UNIT>(l2.y, sgn) * (M)inv_scale;
            }
        }
        return v;
    };
    constexpr int kPlane = TC > 0 ? (TC / 2) * TC : 1;                 // cell pairs per x-plane
    constexpr bool kFixed = TC > 0 && TC % 2 == 0 && kPaintThreads % kPlane == 0 &&
                            TC % (kPaintThreads / kPlane) == 0;
    if constexpr (kFixed) {
        // each pass of the CTA covers whole x-planes: a thread keeps its
        // (cy, cz) and steps cx by a fixed stride, in shared and global memory
        constexpr int hT = TC > 0 ? TC / 2 : 1;
        constexpr int planes = kFixed ? kPaintThreads / kPlane : 1;
        const int t = threadIdx.x;
        const int cz = 2 * (t % hT);
        const int cy = (t / hT) % TC;
        const int cx0 = t / (hT * TC);
        int c = (cx0 * TC + cy) * TC + cz;
        M *dst = mb + ((long long)cx0 * N + cy) * pitch + cz;
        const long long gstep = (long long)planes * N * pitch;
#pragma unroll 2
        for (int k = 0; k < TC / planes; ++k, c += planes * TC * TC, dst += gstep) {
            M2 v = pair(c);
            M2 *d2 = reinterpret_cast<M2 *>(dst);
            if (accumulate) {
                const M2 o = *d2;
                v.x += o.x;
                v.y += o.y;
            }
            *d2 = v;
        }
    } else if ((T & 1) == 0) {
        const int hT = T >> 1;
        const int npairs = T * T * hT;
        for (int p = threadIdx.x; p < npairs; p += blockDim.x) {
            const int r = TC > 0 ? p / (TC / 2) : p / hT;           // row = cx T + cy
            const int cz = 2 * (p - r * hT);
            const int cx = TC > 0 ? r / TC : r / T;
            const int cy = r - cx * T;
            const int c = r * T + cz;
            M2 v = pair(c);
            M2 *dst = reinterpret_cast<M2 *>(mb + ((long long)cx * N + cy) * pitch + cz);
            if (accumulate) {
                const M2 o = *dst;
                v.x += o.x;
                v.y += o.y;
            }
            *dst = v;
        }
    } else {
        const int n = T * T * T;
        for (int c = threadIdx.x; c < n; c += blockDim.x) {
            const int r = c / T, cz = c - r * T;
            const int cx = r / T, cy = r - cx * T;
            const M val = cell(c);
            M *dst = mb + ((long long)cx * N + cy) * pitch + cz;
            if (accumulate) *dst += val;
            else *dst = val;
        }
    }
}

// Words of the cell area (two per cell), rounded up so that the float4 staging
// area behind it is 16-byte aligned for odd tile edges too (2 T^3 words are a
// multiple of 4 only when T is even).
__host__ __device__ constexpr int paint_cell_words(int T) { return (2 * T * T * T + 3) & ~3; }

// TC > 0: the tile edge is the compile-time constant TC (index math in shifts).
// CTAs per SM: as many as the shared memory of tiles of 16 lets in, and their registers;
// left to itself the compiler spilled for more (general path, weighted, 3e7 objects at
// 256^3, interlaced: TSC 3603 -> 3337 us, PCS 7103 -> 6214; 2048^3 lattice 74.3 -> 73.8 ms).
// Other tiles: its choice (asked for 5 or 6 CTAs, halves of tiles lost up to 35 %).
template <int P, int NM, int TC>
constexpr int kPaintCtas = TC != 16 ? 0 : NM == 1 || P == 2 ? 6 : P == 3 ? 5 : 4;
template <int P, int NM, typename M, int TC, bool UNIT>
__global__ void __launch_bounds__(kPaintThreads, kPaintCtas<P, NM, TC>)
k_paint_tiles(const float4 *sorted, const uint32_t *off, const uint32_t *cursor, int *__restrict__ err, PaintGeom g,
              int S, const uint4 *wmaxs, float wdep, M *__restrict__ mesh,
              long long item_stride, long long mesh_stride, int accumulate) {
    grid_wait();
    extern __shared__ __align__(16) unsigned smu[];   // lo[T^3], hi[T^3] or acc64[T^3]; cand[kStage]
    __shared__ uint32_t s_beg[kSegments];
    __shared__ uint32_t s_pre[kSegments + 1];
    const int T = TC > 0 ? TC : g.T, T3 = T * T * T;
    unsigned *lo = smu, *hi = smu + T3;
    unsigned long long *acc64 = reinterpret_cast<unsigned long long *>(smu);
    float4 *cand = reinterpret_cast<float4 *>(smu + paint_cell_words(T));

    // item * ntiles + tile (the launch keeps the block count below 2^31, so
    // 32-bit unsigned division suffices: 64-bit division is a long software
    // sequence that every thread of every tile would run)
    const unsigned gt = blockIdx.x;
    const unsigned ntiles = (unsigned)g.ntiles, ntx = (unsigned)g.ntx;
    const unsigned item = gt / ntiles;
    const unsigned t = gt - item * ntiles;
    const unsigned tq = t / ntx;
    const int tz = (int)(t - tq * ntx);
    const int tx = (int)(tq / ntx);
    const int ty = (int)(tq - (unsigned)tx * ntx);
    const TileFrame<TC> fr(T, g.flog, tx, ty, tz);
    const uint4 wm = wmaxs[item];

    // Segments: neighbour offset d (per axis -1, 0, +1) with the classes of
    // that neighbour whose window reaches this tile: d = -1 -> class 2,
    // d = 0 -> any class, d = +1 -> class 0.  Index s = (ax * 5 + ay) * 3 + az
    // with ax, ay over the 5 (d, class) pairs and az over the 3 z offsets
    // (whose class ranges are contiguous keys).
    if (threadIdx.x < kSegments) {
        const int s = threadIdx.x;
        const int ax = s / 15, ay = (s / 3) % 5, az = s % 3;
        const int dx = ax == 0 ? -1 : (ax == 4 ? 1 : 0), cx = ax == 0 ? 2 : (ax == 4 ? 0 : ax - 1);
        const int dy = ay == 0 ? -1 : (ay == 4 ? 1 : 0), cy = ay == 0 ? 2 : (ay == 4 ? 0 : ay - 1);
        const int dz = az - 1;
        const int cz0 = dz == -1 ? 2 : 0, cz1 = dz == 1 ? 0 : 2;
        const int n = g.ntx;
        const int wx = tx + dx < 0 ? tx + dx + n : (tx + dx >= n ? tx + dx - n : tx + dx);
        const int wy = ty + dy < 0 ? ty + dy + n : (ty + dy >= n ? ty + dy - n : ty + dy);
        const int wz = tz + dz < 0 ? tz + dz + n : (tz + dz >= n ? tz + dz - n : tz + dz);
        const int64_t nt = ((int64_t)wx * n + wy) * n + wz;
        const int64_t kb = ((int64_t)item * g.ntiles + nt) * kClasses + cx * 9 + cy * 3;
        const uint32_t b = off[kb + cz0], e = off[kb + cz1 + 1];
        s_beg[s] = b;
        s_pre[s + 1] = e - b;
    } else if (threadIdx.x >= 96 && threadIdx.x < 96 + kClasses) {
        // the scatter left every cursor of this tile's keys at the next key's offset
        const int64_t key = ((int64_t)item * g.ntiles + t) * kClasses + (threadIdx.x - 96);
        if (cursor[key] != off[key + 1]) atomicOr(err, 2);
    }
    __syncthreads();
    if (threadIdx.x < 32) {                          // warp scan of the 75 lengths
        const int lane = threadIdx.x;
        uint32_t v0 = 0, v1 = 0, v2 = 0;
        if (3 * lane < kSegments) v0 = s_pre[3 * lane + 1];
        if (3 * lane + 1 < kSegments) v1 = s_pre[3 * lane + 2];
        if (3 * lane + 2 < kSegments) v2 = s_pre[3 * lane + 3];
        uint32_t x = v0 + v1 + v2;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        const uint32_t before = x - (v0 + v1 + v2);
        __syncwarp();
        if (lane == 0) s_pre[0] = 0;
        if (3 * lane < kSegments) s_pre[3 * lane + 1] = before + v0;
        if (3 * lane + 1 < kSegments) s_pre[3 * lane + 2] = before + v0 + v1;
        if (3 * lane + 2 < kSegments) s_pre[3 * lane + 3] = before + v0 + v1 + v2;
    }
    __syncthreads();
    const uint32_t total = s_pre[kSegments];

    // Largest deposit of the tile's catalog in fixed-point units (wdep: the
    // window's largest weight).
    const float wmax = __uint_as_float(wm.x);
    const float scale = pow2f(S);
    const float inv_scale = pow2f(-S);
    const float dmax = wmax * wdep * scale;
    const long long pitch = 2LL * (g.N / 2 + 1);
    M *base = mesh + item * item_stride;
    const long long tile_off = ((long long)tx * T * g.N + (long long)ty * T) * pitch + (long long)tz * T;

    // Sweep: cells of one word.  The tile is painted in one pass over its
    // candidates, each read once straight from the sorted copy (nothing to
    // stage), both interlaced meshes together (lo: mesh 0, hi: mesh 1).
    // Unit weights: deposits below 2^23 whose sum cannot reach 2^32.  Other
    // weights: the sum of the candidates' |W V| bounds every cell; it is taken
    // during the sweep, and a tile whose cells might pass 2^31, or 2^32 where no
    // W V is negative (S = 22: sum |W V| above 1022 for CIC, 2424 for TSC, 3451
    // for PCS), is counted in blocks (below) and painted again, swept if those fit,
    // else the general way.  A tile that the catalog's mean |W V| says will not fit
    // skips the sweep.
    //
    // Weighted catalogs used to stage their candidates and take one pass per
    // mesh; unit weights needed deposits below the general path's 2^B, so at
    // most 1024 candidates, and CIC never qualified.  1e7 log-normal objects,
    // interlaced at 512^3, us: CIC 516 -> 444, weighted CIC 516 -> 438, TSC 985 ->
    // 535, PCS 2604 -> 948; 1.3e8 at 1024^3, ms: CIC 5.8 -> 3.8, TSC 6.5 -> 5.5,
    // PCS 20.9 -> 10.7, weighted CIC 5.7 -> 4.1, TSC 11.0 -> 5.7, PCS 29.4 -> 10.9.
    const float ncf = (float)total;
    bool sweep = UNIT ? dmax < 8388607.0f && ncf * (dmax + 1.0f) < 4.29e9f : dmax < 1.07e9f;
    const bool sgn = !UNIT && wm.y != 0u;
    const float cell_max = sgn ? 2.145e9f : 4.29e9f;      // 2^31, 2^32, less 1e-3 for rounding
    const float mean = UNIT ? (dmax + 1.0f) * ncf : ncf * __uint_as_float(wm.z) * wdep * scale;
    if (!UNIT && mean > 0.9f * cell_max) sweep = false;
    // FP64 meshes: only where every deposit is below the general path's 2^B, which
    // rounds no other way
    if (sizeof(M) == 8) sweep = sweep && UNIT && dmax < (float)(1u << max(min(22, 31 - ceil_log2(max(total, 1u))), 0)) - 1.0f;
    // A tile whose candidates in all pass that bound, but by no more than ten times, is
    // swept with its candidates counted per block (|W V| in steps of max |W V| / 1024,
    // rounded up): the blocks that a cell's deposits come from bound it.
    // Such tiles took the general path: 6.7e7 clustered objects at 512^3 (2000 a tile),
    // us: CIC 1133 -> 758, TSC interlaced 5255 -> 2197, weighted PCS interlaced 12363 ->
    // 5064; 1.3e5 at 64^3, TSC interlaced: 84 -> 27.
    // One candidate in eight tells first whether that would be in vain (not for CIC, whose
    // sweep costs little more); then, and where it was, all candidates are counted in
    // smaller blocks before anything is deposited.  Without that, crowded tiles were swept
    // in vain before they took the general path: fifty blobs of 2000 objects (0.6 cells
    // wide) at 64^3, interlaced, us a spectrum, general path alone, swept in vain, now: TSC
    // 320, 363, 315; PCS 440, 656, 458; 3e6 such objects at 128^3: 835, 894, 790; 1360, 1614,
    // 1356; 3e7 at 256^3: 4059, 3447, 2500; 7184, 4604, 3450.
    const bool dense = sizeof(M) == 4 && !sweep && mean < 10.0f * cell_max && ncf < 4.0e6f && dmax < (UNIT ? 8388607.0f : 1.07e9f);
    const float blk_scale = UNIT ? 1.0f : 1024.0f / (wmax * scale);
    const bool wide = T > 16;
    using Coarse = CoarseBlocks<P>;
    using Fine = FineBlocks<P>;
    static_assert(Fine::Count <= kStage * (int)(sizeof(float4) / sizeof(unsigned)), "counters in the smallest tile's memory");
    const auto blocks_fit = [&](float n) {               // n: largest count of a cell's blocks
        // every cell: sum of round(w W V 2^S) <= wdep sum |W V| 2^S + candidates
        return UNIT ? n * (dmax + 1.0f) < cell_max
                    : n * (wmax * scale * wdep * (1.0f / 1024.0f)) * 1.00001f + ncf < cell_max;
    };
    const auto steps = [&](float w) { return UNIT ? 1u : __float2uint_ru(fabsf(w) * blk_scale); };
    // Largest count of a cell's blocks B over candidates 0, stride, 2 stride, ..
    const auto count_blocks = [&](auto B, uint32_t stride) {
        for (int c = threadIdx.x; c < B.Count; c += blockDim.x) smu[c] = 0u;
        __syncthreads();
        for (uint32_t k = threadIdx.x * stride; k < total; k += blockDim.x * stride) {
            const float4 v = fetch_candidate(sorted, s_beg, s_pre, fr, k, scale);
            atomicAdd(smu + B.of(fr.at(v.x, 0), fr.at(v.y, 1), fr.at(v.z, 2), wide), steps(v.w));
        }
        __syncthreads();
        return B.most(smu, wide);
    };
    bool known = UNIT && sweep;                           // every cell is known to fit
    bool look = false;                                    // count in the smaller blocks first
    if (P > 2 && dense) look = __syncthreads_or(!blocks_fit(8.0f * count_blocks(Coarse{}, 8u)));
#pragma unroll 1
    while (sweep || dense) {
        if (look) {
            known = !__syncthreads_or(!blocks_fit(count_blocks(Fine{}, 1u)));
            if (!known) break;
        }
        const bool counted = dense && !known;
        // TSC and PCS sweeps of 16^3 tiles deposit into the padded layout
        // (SweepLayout); CIC keeps the compact one
        constexpr bool kPadded = TC == 16 && (P == 4 || P == 3);
        // block counters behind the cells (the staging area is unused here)
        unsigned *s_blk = smu + (kPadded ? NM * SweepLayout<P>::Words : paint_cell_words(T));
        {
            uint4 *z4 = reinterpret_cast<uint4 *>(smu);
            const int nw = kPadded ? NM * SweepLayout<P>::Words : (NM == 1 ? T3 : 2 * T3);
            const int n4 = nw / 4;
            for (int c = threadIdx.x; c < n4; c += blockDim.x) z4[c] = make_uint4(0u, 0u, 0u, 0u);
            for (int c = 4 * n4 + threadIdx.x; c < nw; c += blockDim.x) smu[c] = 0u;
            for (int c = threadIdx.x; counted && c < Coarse::Count; c += blockDim.x) s_blk[c] = 0u;
        }
        __syncthreads();
        // |W V| in units rounded up, as integers (NaN: far too much)
        unsigned long long sum_abs = 0ull;
        const auto account = [&](const float4 &v) {
            if (!UNIT) sum_abs += fabsf(v.w) < 4.29e9f ? (unsigned long long)__float2uint_ru(fabsf(v.w)) : 1ull << 40;
            if (counted) atomicAdd(s_blk + Coarse::of(fr.at(v.x, 0), fr.at(v.y, 1), fr.at(v.z, 2), wide), steps(v.w));
        };
        if (kPadded) {
            for (uint32_t k = threadIdx.x; k < total; k += blockDim.x) {
                const float4 v = fetch_candidate(sorted, s_beg, s_pre, fr, k, scale);
                account(v);
                sweep_deposit<P, UNIT>(smu, v.x, v.y, v.z, v.w);
                if (NM == 2)
                    sweep_deposit<P, UNIT>(smu + SweepLayout<P>::Words, v.x + 0.5f, v.y + 0.5f, v.z + 0.5f, v.w);
            }
        } else {
            // the first 32 words of the staging area are the lanes' scratch
            const unsigned trash = (unsigned)(2 * T3) + (threadIdx.x & 31);
            const bool flat = !dense && total <= (uint32_t)kFlatMaxCand;
            for (uint32_t k = threadIdx.x; k < total; k += blockDim.x) {
                const float4 v = fetch_candidate(sorted, s_beg, s_pre, fr, k, scale);
                account(v);
                const float x = fr.at(v.x, 0), y = fr.at(v.y, 1), z = fr.at(v.z, 2);
                const float x2 = fr.at(v.x + 0.5f, 0), y2 = fr.at(v.y + 0.5f, 1), z2 = fr.at(v.z + 0.5f, 2);
                if (flat) {
                    deposit_flat<P, TC, UNIT>(smu, 0, trash, T, x, y, z, v.w);
                    if (NM == 2) deposit_flat<P, TC, UNIT>(smu, T3, trash, T, x2, y2, z2, v.w);
                } else {
                    const Split none{};
                    deposit<P, 2, TC, UNIT, float>(lo, nullptr, nullptr, none, T, x, y, z, v.w);
                    if (NM == 2) deposit<P, 2, TC, UNIT, float>(hi, nullptr, nullptr, none, T, x2, y2, z2, v.w);
                }
            }
        }
        __syncthreads();
        if (known) {
        } else if (dense) {
            known = !__syncthreads_or(!blocks_fit(Coarse::most(s_blk, wide)));
        } else if constexpr (!UNIT) {
            __shared__ unsigned long long s_abs[kPaintThreads / 32];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sum_abs += __shfl_down_sync(0xffffffffu, sum_abs, o);
            if ((threadIdx.x & 31) == 0) s_abs[threadIdx.x >> 5] = sum_abs;
            __syncthreads();
            unsigned long long t = 0ull;
#pragma unroll
            for (int k = 0; k < kPaintThreads / 32; ++k) t += s_abs[k];
            __syncthreads();                              // read before a second sweep's sum
            // every cell: sum of round(w W V 2^S) <= wdep sum |W V| 2^S + candidates / 2
            known = (float)t * wdep + ncf < cell_max;
        }
        if (known) {
            const Split none{};
            if (kPadded) {
                sweep_flush<M, P, UNIT>(smu, sgn, inv_scale, base + tile_off, g.N, pitch, accumulate);
                if (NM == 2)
                    sweep_flush<M, P, UNIT>(smu + SweepLayout<P>::Words, sgn, inv_scale, base + mesh_stride + tile_off, g.N,
                                            pitch, accumulate);
            } else {
                flush_tile<M, TC, UNIT>(lo, nullptr, nullptr, none, sgn, inv_scale, base + tile_off, T, g.N, pitch,
                                        accumulate);
                if (NM == 2)
                    flush_tile<M, TC, UNIT>(hi, nullptr, nullptr, none, sgn, inv_scale, base + mesh_stride + tile_off, T,
                                            g.N, pitch, accumulate);
            }
            return;
        }
        if ((P == 2 && dense) || ncf >= 4.0e6f) break;    // the same blocks; beyond the counters' range
        look = true;
    }
    __syncthreads();                                      // the cells are zeroed again below

    // General path: one mesh per pass over staged candidates.
    Split sp;
    {
        const unsigned nc = total > 0u ? total : 1u;
        // FP32: sums of nc words below 2^B stay below 2^32; FP64: the split that its
        // rounding has always had
        sp.B = sizeof(M) == 4 ? min(30, 32 - ceil_log2(nc)) : min(22, 31 - ceil_log2(nc));
        sp.twoB = __uint_as_float((unsigned)(127 + max(sp.B, 0)) << 23);
        sp.twoB_u = 1u << max(sp.B, 0);
        sp.inv2B = __uint_as_float((unsigned)(127 - max(sp.B, 0)) << 23);
        sp.hi_scale = pow2f(sp.B - S);
        const float hmax = wmax * pow2f(S - sp.B);
        sp.fast = sp.B >= 1 && hmax < 4194304.0f && (float)nc * (hmax + 1.0f) < 2.0e9f;
    }
    const bool staged_once = total <= (uint32_t)kStage;
    if (staged_once) stage_candidates(sorted, s_beg, s_pre, fr, 0u, total, scale, cand);
#pragma unroll 1
    for (int m = 0; m < NM; ++m) {
        {
            uint4 *z4 = reinterpret_cast<uint4 *>(smu);
            const int nw = 2 * T3, n4 = nw / 4;
            for (int c = threadIdx.x; c < n4; c += blockDim.x) z4[c] = make_uint4(0u, 0u, 0u, 0u);
            for (int c = 4 * n4 + threadIdx.x; c < nw; c += blockDim.x) smu[c] = 0u;
        }
        __syncthreads();
        const float sh = m ? 0.5f : 0.0f;
        if (staged_once) {
            deposit_any<P, TC, UNIT, M>(cand, total, lo, hi, acc64, sp, T, fr, sh);
        } else {
            for (uint32_t k0 = 0; k0 < total; k0 += kStage) {     // dense tile: batches
                const uint32_t n = min((uint32_t)kStage, total - k0);
                __syncthreads();                                  // previous batch consumed
                stage_candidates(sorted, s_beg, s_pre, fr, k0, n, scale, cand);
                __syncthreads();
                deposit_any<P, TC, UNIT, M>(cand, n, lo, hi, acc64, sp, T, fr, sh);
            }
        }
        __syncthreads();
        flush_tile<M, TC, UNIT>(sp.fast ? lo : nullptr, sp.fast ? hi : nullptr, sp.fast ? nullptr : acc64, sp, false,
                                inv_scale, base + m * mesh_stride + tile_off, T, g.N, pitch, accumulate);
        __syncthreads();
    }
}

// ---- direct atomic paint (the variant without a sort) ----
// Per object: the same wrapped cell coordinate as the sort path, cell
// c0 = floor(s) and offset u = (s - c0) + e along each axis; every deposit
// round(w 2^S W) is added with a 64-bit global atomic (RED) into a dense
// N^3 int64 accumulator per mesh.  Integer adds keep the accumulator
// independent of object order.  The accumulator is converted and cleared by
// k_acc_to_mesh.
template <int P>
__device__ __forceinline__ void deposit_global(unsigned long long *__restrict__ acc, int N,
                                               const int *c0, const float *u, float sh, float ws) {
    int bx, by, bz;
    float wx[P], wy[P], wz[P];
    spline_weights<P>(u[0] + sh, bx, wx);
    spline_weights<P>(u[1] + sh, by, wy);
    spline_weights<P>(u[2] + sh, bz, wz);
    int cz[P];
#pragma unroll
    for (int c = 0; c < P; ++c) {
        int v = c0[2] + bz + c;
        v = v < 0 ? v + N : (v >= N ? v - N : v);
        cz[c] = v;
    }
#pragma unroll
    for (int a = 0; a < P; ++a) {
        int cx = c0[0] + bx + a;
        cx = cx < 0 ? cx + N : (cx >= N ? cx - N : cx);
        const float vx = ws * wx[a];
#pragma unroll
        for (int b = 0; b < P; ++b) {
            int cy = c0[1] + by + b;
            cy = cy < 0 ? cy + N : (cy >= N ? cy - N : cy);
            const float vxy = vx * wy[b];
            unsigned long long *row = acc + ((long long)cx * N + cy) * N;
#pragma unroll
            for (int c = 0; c < P; ++c) {
                // round(v) in one FMA when 0 <= round(v) < 2^22, else the
                // rounded product converted to int64
                const float t = fmaf(vxy, wz[c], 8388608.0f);
                long long q;
                if (t >= 8388608.0f && t < 12582912.0f) q = (long long)(__float_as_uint(t) - 0x4B000000u);
                else q = __float2ll_rn(vxy * wz[c]);
                if (q) atomicAdd(row + cz[c], (unsigned long long)q);
            }
        }
    }
}

template <int DT, int P, int NM>
__global__ void __launch_bounds__(kCountThreads)
k_paint_atomic(const void *__restrict__ pos, const float *__restrict__ w, const float *__restrict__ vals,
               const int64_t *__restrict__ item_off, int64_t n_one, PaintGeom g, int S, bool weighted,
               unsigned long long *__restrict__ acc, double *__restrict__ wsums,
               double *__restrict__ wpart, uint4 *__restrict__ wmax) {
    using R = typename PosReal<DT>::type;
    const int item = blockIdx.y;
    const ItemRange range(item_off, n_one, item);
    const int64_t beg = range.beg, end = range.end;
    const long long n3 = (long long)g.N * g.N * g.N;
    unsigned long long *ab = acc + (long long)item * NM * n3;
    const float scale = ldexpf(1.0f, S);
    double sw = 0.0, sw2 = 0.0, swa = 0.0;
    float mw = 0.0f;
    bool neg = false;
    for (int64_t i = beg + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < end;
         i += (int64_t)gridDim.x * blockDim.x) {
        const Obj<R> o = load_obj<DT>(pos, w, vals, i, g);
        int c0[3];
        float u[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            c0[a] = min((int)floor(o.s[a]), g.N - 1);
            u[a] = (float)(o.s[a] - (R)c0[a]) + o.e[a];
        }
        const float ws = o.a * scale;
#pragma unroll
        for (int m = 0; m < NM; ++m) deposit_global<P>(ab + m * n3, g.N, c0, u, m ? 0.5f : 0.0f, ws);
        if (weighted) {
            const double ad = (double)o.a;
            sw += (double)o.w;
            sw2 += ad * ad;
            swa += fabs(ad);
            mw = fmaxf(mw, fabsf(o.a));
            neg |= o.a < 0.0f;
        }
    }
    flush_wsums(sw, sw2, swa, mw, neg, weighted, item, end - beg, wsums, wpart, wmax);
}

template <typename M>
__device__ __forceinline__ M acc_value(unsigned long long q, float inv_scale);
template <>
__device__ __forceinline__ float acc_value<float>(unsigned long long q, float inv_scale) {
    return ll_to_float_rn((long long)q) * inv_scale;
}
template <>
__device__ __forceinline__ double acc_value<double>(unsigned long long q, float inv_scale) {
    return __ll2double_rn((long long)q) * (double)inv_scale;
}

// Dense int64 accumulators (nitems x nm x N^3, z fastest) -> the r2c padded
// mesh layout, two cells per thread; each accumulator pair is cleared after
// it is read so the next paint starts from zero.
template <typename M>
__global__ void __launch_bounds__(256)
k_acc_to_mesh(ulonglong2 *__restrict__ acc, long long npairs, int N, int nm, float inv_scale,
              M *__restrict__ mesh, long long item_stride, long long mesh_stride, int accumulate) {
    using M2 = typename std::conditional<sizeof(M) == 4, float2, double2>::type;
    const long long n3 = (long long)N * N * N;
    const long long pitch = 2LL * (N / 2 + 1);
    for (long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x; j < npairs;
         j += (long long)gridDim.x * blockDim.x) {
        const long long cell = 2 * j;
        const long long im = cell / n3;
        const long long r = cell - im * n3;
        const long long row = r / N;
        const int cz = (int)(r - row * N);
        const long long item = im / nm;
        const int m = (int)(im - item * nm);
        const ulonglong2 q = acc[j];
        acc[j] = make_ulonglong2(0ull, 0ull);
        M *dst = mesh + item * item_stride + m * mesh_stride + row * pitch + cz;
        M2 v;
        v.x = acc_value<M>(q.x, inv_scale);
        v.y = acc_value<M>(q.y, inv_scale);
        if (accumulate) {
            const M2 o = *reinterpret_cast<const M2 *>(dst);
            v.x += o.x;
            v.y += o.y;
        }
        *reinterpret_cast<M2 *>(dst) = v;
    }
}

// ---- fused compensate + interlace + bin ----
template <typename C>
__device__ __forceinline__ C cmul(C a, C b) {
    C r;
    r.x = a.x * b.x - a.y * b.y;
    r.y = a.x * b.y + a.y * b.x;
    return r;
}

__host__ __device__ __forceinline__ size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

template <typename R, typename C, typename A>
struct BinSmem {
    // layout: hist[nh] (A), cw_l[Nh] (R), ph_l[Nh] (C), edge pairs[nk] (int2: m range of bin b)
    __host__ __device__ static size_t off_cw(const BinGeom &g) { return align_up((size_t)g.nh * sizeof(A), 16); }
    // the cw and ph tables hold Nh + Nh/4 + 1 entries: k_bin stores entry l at l + l/4
    __host__ __device__ static size_t tab(const BinGeom &g) { return (size_t)g.Nh + (size_t)(g.Nh >> 2) + 1; }
    __host__ __device__ static size_t off_ph(const BinGeom &g) { return align_up(off_cw(g) + tab(g) * sizeof(R), 16); }
    __host__ __device__ static size_t off_edge(const BinGeom &g) { return align_up(off_ph(g) + tab(g) * sizeof(C), 16); }
    __host__ __device__ static size_t bytes(const BinGeom &g) { return align_up(off_edge(g) + (size_t)g.nk * sizeof(int2), 16); }
};

// floor(sqrt(x)) for 0 <= x < 2^26, exact.
__device__ __forceinline__ int isqrt_floor(int x) {
    int s = (int)sqrtf((float)x);
    while (s > 0 && s * s > x) --s;
    while ((s + 1) * (s + 1) <= x) ++s;
    return s;
}

// Fused compensate + interlace + bin.  Rows are the unit of work: each warp
// takes whole rows (i, j) and visits only the l range whose modes fall in a k
// bin, mlo <= i'^2 + j'^2 + l^2 < mhi (and m != 0); each lane sums kBinVec
// consecutive modes of it in registers and flushes a run to the per-CTA
// shared histogram when its bin changes.  CROSS: the meshes of a second
// catalog at meshb; each mode contributes Re(delta_a conj(delta_b)) instead
// of |delta|^2.  MU32: the mu-bin test q^2 m <= nmu^2 l^2 fits in 32 bits.
template <bool IL, bool TWOD, bool POLES, bool CROSS, bool MU32>
__global__ void __launch_bounds__(kBinThreads, 5)
k_bin(const float2 *mesh, long long item_stride_c, long long mesh_stride_c, BinGeom g,
      const float *cw, const float2 *ph, const int *kedge, float *__restrict__ partial, const float2 *meshb) {
    grid_wait();
    using R = float;
    using C = float2;
    using A = float;
    using SM = BinSmem<R, C, A>;
    extern __shared__ __align__(16) unsigned char smraw[];
    A *hist = reinterpret_cast<A *>(smraw);
    R *scw = reinterpret_cast<R *>(smraw + SM::off_cw(g));
    C *sph = reinterpret_cast<C *>(smraw + SM::off_ph(g));
    int2 *sedge = reinterpret_cast<int2 *>(smraw + SM::off_edge(g));
    for (int k = threadIdx.x; k < g.nh; k += blockDim.x) hist[k] = (A)0;
    // entry l at l + l/4: lanes read l = l0 + 4 lane + v, which this skew
    // spreads over all banks (4-byte cw) or two wavefronts (8-byte ph)
    for (int k = threadIdx.x; k < g.Nh; k += blockDim.x) {
        scw[k + (k >> 2)] = cw[k];
        sph[k + (k >> 2)] = ph[k + g.N / 2];
    }
    for (int k = threadIdx.x; k < g.nk; k += blockDim.x) sedge[k] = make_int2(kedge[k], kedge[k + 1]);
    __syncthreads();

    const int item = blockIdx.y;
    const C *m1 = mesh + (long long)item * item_stride_c;
    const C *m2 = m1 + mesh_stride_c;
    const C *n1 = CROSS ? meshb : m1;
    const C *n2 = n1 + mesh_stride_c;
    const int half = g.N / 2, N = g.N, Nh = g.Nh;
    const int nk = g.nk, nmu = g.nmu, hbase = g.hbase;
    const float kscale = g.kscale, koff = g.koff;
    const int lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    const int rows = N * N;
    for (int row = blockIdx.x * wpb + (threadIdx.x >> 5); row < rows; row += gridDim.x * wpb) {
        const int i = row / N, j = row - i * N;
        const int ip = i < half ? i : i - N;
        const int jp = j < half ? j : j - N;
        const int r2 = ip * ip + jp * jp;
        if (r2 >= g.mhi) continue;
        const int lhi = min(Nh, isqrt_floor(g.mhi - 1 - r2) + 1);
        int llo = g.mlo > r2 ? isqrt_floor(g.mlo - r2 - 1) + 1 : 0;
        if (r2 == 0 && llo == 0) llo = 1;
        if (llo >= lhi) continue;
        R rowcw = cw[i] * cw[j];
        C rowph;
        rowph.x = (R)0;
        rowph.y = (R)0;
        if (IL) {
            rowcw *= (R)0.25;
            rowph = cmul(ph[ip + half], ph[jp + half]);
        }
        const long long base = (long long)row * Nh;
        for (int l0 = llo + kBinVec * lane; l0 < lhi; l0 += 32 * kBinVec) {
            const int cnt = lhi - l0;                   // modes of this run: min(cnt, kBinVec)
            C a[kBinVec], b2[kBinVec], ca[CROSS ? kBinVec : 1], cb2[CROSS && IL ? kBinVec : 1];
#pragma unroll
            for (int v = 0; v < kBinVec; ++v) {
                const long long at = base + l0 + min(v, cnt - 1);   // the tail re-reads the last mode
                a[v] = __ldcs(m1 + at);
                if (IL) b2[v] = __ldcs(m2 + at);
                if (CROSS) {
                    ca[CROSS ? v : 0] = __ldcs(n1 + at);
                    if (IL) cb2[CROSS && IL ? v : 0] = __ldcs(n2 + at);
                }
            }
            int cur2 = -1, cur1 = -1;                 // open register runs
            R run2 = (R)0, runm2 = (R)0, runm4 = (R)0;
#pragma unroll
            for (int v = 0; v < kBinVec; ++v) {
                const bool live = v < cnt;
                const int l = min(l0 + v, lhi - 1);
                const int m = r2 + l * l;
                // FP32 estimate of the k bin, then one exact step against the FP64
                // edges: the estimate's error (below 4e-7 kmax / dk + 0.1, the
                // plan requires kmax / dk < 2^20) puts it at most one bin off
                const float rsm = rsqrtf((float)m);
                int b = (int)((float)m * rsm * kscale - koff);
                b = min(max(b, 0), nk - 1);
                {
                    const int2 e = sedge[b];
                    b += (int)(m >= e.y) - (int)(m < e.x);
                }
                C z = a[v];
                C y;
                if (CROSS) y = ca[CROSS ? v : 0];
                if (IL) {
                    const C t = cmul(rowph, sph[l + (l >> 2)]);
                    z.x += b2[v].x * t.x - b2[v].y * t.y;
                    z.y += b2[v].x * t.y + b2[v].y * t.x;
                    if (CROSS) {
                        const C u = cb2[CROSS && IL ? v : 0];
                        y.x += u.x * t.x - u.y * t.y;
                        y.y += u.x * t.y + u.y * t.x;
                    }
                }
                R pw = (CROSS ? z.x * y.x + z.y * y.y : z.x * z.x + z.y * z.y) * rowcw * scw[l + (l >> 2)];
                pw *= !live ? (R)0 : (l != 0 && l != half) ? (R)2 : (R)1;
                int key = b;
                if (TWOD) {
                    // mu bin: FP32 estimate, then one exact integer step each way
                    int q = (int)((float)(nmu * l) * rsm);
                    q = min(max(q, 0), nmu - 1);
                    if (MU32) {
                        const unsigned rhs = (unsigned)(nmu * nmu) * (unsigned)(l * l);
                        q -= (int)(q > 0 && (unsigned)(q * q) * (unsigned)m > rhs);
                        q += (int)(q < nmu - 1 && (unsigned)((q + 1) * (q + 1)) * (unsigned)m <= rhs);
                    } else {
                        const long long rhs = (long long)nmu * nmu * l * l;
                        q -= (int)(q > 0 && (long long)q * q * m > rhs);
                        q += (int)(q < nmu - 1 && (long long)(q + 1) * (q + 1) * m <= rhs);
                    }
                    key = b * nmu + q;
                }
                // flush an open run when the key changes (predicated, no branch)
                const bool new2 = key != cur2;
                if (new2 && cur2 >= 0) atomicAdd(hist + cur2, (A)run2);
                run2 = new2 ? pw : run2 + pw;
                cur2 = key;
                if (POLES) {
                    // mu = l rsqrt(m) from the k-bin estimate (a few ulp).  The sums are
                    // of P L_2(mu) and P L_4(mu) themselves, not of P mu^2 and P mu^4:
                    // forming P_4 from mu moments (35 M4 - 30 M2 + 3 S0) would amplify
                    // the FP32 partial sums' rounding about forty-fold.
                    const float mu = (float)l * rsm;
                    const R mu2 = mu * mu;
                    const R t2 = pw * ((R)1.5 * mu2 - (R)0.5);
                    const R t4 = pw * (((R)4.375 * mu2 - (R)3.75) * mu2 + (R)0.375);
                    const bool new1 = b != cur1;
                    if (new1 && cur1 >= 0) {
                        atomicAdd(hist + hbase + cur1, (A)runm2);
                        atomicAdd(hist + hbase + nk + cur1, (A)runm4);
                    }
                    runm2 = new1 ? t2 : runm2 + t2;
                    runm4 = new1 ? t4 : runm4 + t4;
                    cur1 = b;
                }
            }
            atomicAdd(hist + cur2, (A)run2);
            if (POLES) {
                atomicAdd(hist + hbase + cur1, (A)runm2);
                atomicAdd(hist + hbase + nk + cur1, (A)runm4);
            }
        }
    }
    __syncthreads();
    A *out = partial + ((long long)item * gridDim.x + blockIdx.x) * g.nh;
    for (int k = threadIdx.x; k < g.nh; k += blockDim.x) out[k] = hist[k];
}

// An integer 0 <= v < 2^32 as a double by one addition (the conversion
// instruction has the FP64 pipe's rate as well, and a longer latency).
__device__ __forceinline__ double u32_to_double(unsigned v) {
    return __hiloint2double(0x43300000, (int)v) - 4503599627370496.0;
}
// A normal float as a double, by its bits.
__device__ __forceinline__ double float_bits_to_double(float f) {
    const unsigned b = __float_as_uint(f);
    return __hiloint2double((int)((b >> 3) + (896u << 20)), (int)(b << 29));
}

// The bin pass of FP64 meshes: as k_bin, laid out for the FP64 pipe (two
// operations per SM and clock), which bounds it (85 % of its rate):
//   * 19 FP64 operations per mode with interlacing and multipoles: the phase of
//     a mode is one table entry (its arguments add up: i' + j' + l, folded by
//     e^{i pi} = -1 and e^{-ix} = conj e^{ix} into 0 .. N/2, so that the tables take
//     k_bin's places), weights of 1 or 2 stand in the cw table, Legendre sums are
//     one FMA each, and l^2 / m comes from the FP32 reciprocal r by
//     r (1 + e + e^2), e = 1 - m r (the geometric series of 1 / (m r); e^3 <
//     2^-60).
//   * Runs of kBinVec modes of four rows are dealt to the lanes without gaps: with
//     a row per warp a third of the lanes idled at the rows' ends, and an FP64
//     instruction costs the same with half of its lanes off.
// Two interlaced meshes, multipoles (k_bin in FP64 before): 64^3 49 -> 18 us, 256^3
// 512 -> 311 us, 512^3 3.25 -> 1.86 ms.  Eight rows a turn: 31, 283 us, 1.87 ms, but
// 400^3 1.03 ms for 0.94.
template <bool IL, bool TWOD, bool POLES, bool CROSS, bool MU32>
__global__ void __launch_bounds__(kBinThreads, 2)
k_bin_f64(const double2 *mesh, long long item_stride_c, long long mesh_stride_c, BinGeom g,
          const double *cw, const double2 *ph, const int *kedge, double *__restrict__ partial, const double2 *meshb) {
    grid_wait();
    using SM = BinSmem<double, double2, double>;
    constexpr int kRows = 4;                          // rows per warp and turn
    extern __shared__ __align__(16) unsigned char smraw[];
    double *hist = reinterpret_cast<double *>(smraw);
    double *scw = reinterpret_cast<double *>(smraw + SM::off_cw(g));
    double2 *sph = reinterpret_cast<double2 *>(smraw + SM::off_ph(g));
    int2 *sedge = reinterpret_cast<int2 *>(smraw + SM::off_edge(g));
    const int half = g.N / 2, N = g.N, Nh = g.Nh;
    for (int k = threadIdx.x; k < g.nh; k += blockDim.x) hist[k] = 0.0;
    for (int k = threadIdx.x; k < Nh; k += blockDim.x) scw[k + (k >> 2)] = (k != 0 && k != half ? 2.0 : 1.0) * cw[k];
    for (int k = threadIdx.x; IL && k < Nh; k += blockDim.x) sph[k + (k >> 2)] = ph[k + half];
    for (int k = threadIdx.x; k < g.nk; k += blockDim.x) sedge[k] = make_int2(kedge[k], kedge[k + 1]);
    __syncthreads();

    const int item = blockIdx.y;
    const double2 *m1 = mesh + (long long)item * item_stride_c;
    const double2 *m2 = m1 + mesh_stride_c;
    const double2 *n1 = CROSS ? meshb : m1;
    const double2 *n2 = n1 + mesh_stride_c;
    const int nk = g.nk, nmu = g.nmu, hbase = g.hbase;
    const float kscale = g.kscale, koff = g.koff;
    const int lane = threadIdx.x & 31;
    const int wpb = blockDim.x >> 5;
    const int rows = N * N;
    // Turn k of W warps covers W groups of rows, shifted so that a warp moves on by
    // 5/8 of a plane per turn: W = 152 x 16 groups are whole planes for powers of
    // two, and it would meet the same ky, short rows or long ones, on every turn.
    const int W = gridDim.x * wpb, w0 = blockIdx.x * wpb + (threadIdx.x >> 5);
    const int gp = (N + kRows - 1) / kRows, shift = (5 * gp / 8 + gp - W % gp) % gp % W;
    for (int first = 0, w = w0; first * kRows < rows; first += W, w = w + shift < W ? w + shift : w + shift - W) {
        const int row0 = (first + w) * kRows;
        if (row0 >= rows) continue;
        // lane r < kRows: row row0 + r, its l range, runs and weight
        int r2 = 0, llo = 0, lhi = 0, s0 = 0;
        double rowcw = 0.0;
        if (lane < kRows && row0 + lane < rows) {
            const int i = (row0 + lane) / N, j = row0 + lane - i * N;
            const int ip = i < half ? i : i - N;
            const int jp = j < half ? j : j - N;
            r2 = ip * ip + jp * jp;
            s0 = ip + jp;
            if (r2 < g.mhi) {
                lhi = min(Nh, isqrt_floor(g.mhi - 1 - r2) + 1);
                llo = g.mlo > r2 ? isqrt_floor(g.mlo - r2 - 1) + 1 : 0;
                if (r2 == 0 && llo == 0) llo = 1;
                rowcw = cw[i] * cw[j] * (IL ? 0.25 : 1.0);
            }
        }
        int incl = max(lhi - llo + kBinVec - 1, 0) / kBinVec;      // runs of this and the lanes before it
#pragma unroll
        for (int d = 1; d < kRows; d <<= 1) {
            const int o = __shfl_up_sync(0xffffffffu, incl, d);
            if (lane >= d) incl += o;
        }
        const int total = __shfl_sync(0xffffffffu, incl, kRows - 1);
        for (int t0 = 0; t0 < total; t0 += 32) {
            const int t = t0 + lane;
            int r = 0;                                             // rows whose runs all lie before run t
#pragma unroll
            for (int d = kRows / 2; d; d >>= 1)
                if (t >= __shfl_sync(0xffffffffu, incl, r + d - 1)) r += d;
            const int before = __shfl_sync(0xffffffffu, incl, max(r - 1, 0));
            const int rr2 = __shfl_sync(0xffffffffu, r2, r), rs = __shfl_sync(0xffffffffu, s0, r);
            const int end = __shfl_sync(0xffffffffu, lhi, r);
            const int l0 = __shfl_sync(0xffffffffu, llo, r) + kBinVec * (t - (r ? before : 0));
            const double rcw = __shfl_sync(0xffffffffu, rowcw, r);
            if (t >= total) continue;
            const int cnt = end - l0;                              // modes of this run: min(cnt, kBinVec)
            const long long base = (long long)(row0 + r) * Nh + l0;
            double2 a[kBinVec], b2[kBinVec], ca[CROSS ? kBinVec : 1], cb2[CROSS && IL ? kBinVec : 1];
#pragma unroll
            for (int v = 0; v < kBinVec; ++v) {
                const long long at = base + min(v, cnt - 1);       // the tail re-reads the last mode
                a[v] = __ldcs(m1 + at);
                if (IL) b2[v] = __ldcs(m2 + at);
                if (CROSS) {
                    ca[CROSS ? v : 0] = __ldcs(n1 + at);
                    if (IL) cb2[CROSS && IL ? v : 0] = __ldcs(n2 + at);
                }
            }
            int cur2 = -1, cur1 = -1;                              // open register runs
            double run2 = 0.0, runm2 = 0.0, runm4 = 0.0;
#pragma unroll
            for (int v = 0; v < kBinVec; ++v) {
                const bool live = v < cnt;
                const int l = min(l0 + v, end - 1);
                const int m = rr2 + l * l;
                const float rsm = rsqrtf((float)m);                // bins: as k_bin
                int b = (int)((float)m * rsm * kscale - koff);
                b = min(max(b, 0), nk - 1);
                {
                    const int2 e = sedge[b];
                    b += (int)(m >= e.y) - (int)(m < e.x);
                }
                double2 z = a[v], y;
                if (CROSS) y = ca[CROSS ? v : 0];
                if (IL) {
                    int s = rs + l, flip = 0, conj = 0;            // -N <= s <= 3 N / 2
                    if (s > half) s -= N, flip ^= 0x80000000;
                    if (s > half) s -= N, flip ^= 0x80000000;
                    if (s < -half) s += N, flip ^= 0x80000000;
                    if (s < 0) s = -s, conj = 0x80000000;
                    double2 w = sph[s + (s >> 2)];
                    w.x = __hiloint2double(__double2hiint(w.x) ^ flip, __double2loint(w.x));
                    w.y = __hiloint2double(__double2hiint(w.y) ^ flip ^ conj, __double2loint(w.y));
                    z.x = fma(b2[v].x, w.x, fma(-b2[v].y, w.y, z.x));
                    z.y = fma(b2[v].x, w.y, fma(b2[v].y, w.x, z.y));
                    if (CROSS) {
                        const double2 u = cb2[CROSS && IL ? v : 0];
                        y.x = fma(u.x, w.x, fma(-u.y, w.y, y.x));
                        y.y = fma(u.x, w.y, fma(u.y, w.x, y.y));
                    }
                }
                const double p2 = CROSS ? fma(z.x, y.x, z.y * y.y) : fma(z.x, z.x, z.y * z.y);
                const double pw = live ? p2 * (rcw * scw[l + (l >> 2)]) : 0.0;
                int key = b;
                if (TWOD) {
                    int q = (int)((float)(nmu * l) * rsm);
                    q = min(max(q, 0), nmu - 1);
                    if (MU32) {
                        const unsigned rhs = (unsigned)(nmu * nmu) * (unsigned)(l * l);
                        q -= (int)(q > 0 && (unsigned)(q * q) * (unsigned)m > rhs);
                        q += (int)(q < nmu - 1 && (unsigned)((q + 1) * (q + 1)) * (unsigned)m <= rhs);
                    } else {
                        const long long rhs = (long long)nmu * nmu * l * l;
                        q -= (int)(q > 0 && (long long)q * q * m > rhs);
                        q += (int)(q < nmu - 1 && (long long)(q + 1) * (q + 1) * m <= rhs);
                    }
                    key = b * nmu + q;
                }
                const bool new2 = key != cur2;
                if (new2 && cur2 >= 0) atomicAdd(hist + cur2, run2);
                run2 = new2 ? pw : run2 + pw;
                cur2 = key;
                if (POLES) {
                    const double rc = float_bits_to_double(rsm * rsm);
                    const double e = fma(-u32_to_double((unsigned)m), rc, 1.0);
                    const double q = u32_to_double((unsigned)(l * l)) * rc;
                    const double mu2 = fma(q, fma(e, e, e), q);
                    const bool new1 = b != cur1;
                    if (new1 && cur1 >= 0) {
                        atomicAdd(hist + hbase + cur1, runm2);
                        atomicAdd(hist + hbase + nk + cur1, runm4);
                    }
                    runm2 = fma(pw, fma(1.5, mu2, -0.5), new1 ? 0.0 : runm2);
                    runm4 = fma(pw, fma(fma(4.375, mu2, -3.75), mu2, 0.375), new1 ? 0.0 : runm4);
                    cur1 = b;
                }
            }
            atomicAdd(hist + cur2, run2);
            if (POLES) {
                atomicAdd(hist + hbase + cur1, runm2);
                atomicAdd(hist + hbase + nk + cur1, runm4);
            }
        }
    }
    __syncthreads();
    double *out = partial + ((long long)item * gridDim.x + blockIdx.x) * g.nh;
    for (int k = threadIdx.x; k < g.nh; k += blockDim.x) out[k] = hist[k];
}

// k bins per block of k_reduce_finalize: about 8 histogram slots, so that the
// rows are summed by 32 threads per slot (with 32 slots per block the serial row
// sums took twice as long).
__host__ __device__ __forceinline__ int final_bins(const FinalGeom &f) {
    const int per = (f.twod ? f.nmu : 1) + (f.poles ? 2 : 0);
    return per >= 8 ? 1 : 8 / per;
}

// Sum of the per-CTA histograms and the results, one block per final_bins() k
// bins and catalog: the block's slots times as many groups of rows as its
// threads allow, each summed in row order, then the groups in order (FP64, a
// fixed order); then normalization, shot noise and multipoles of the block's
// bins, written straight into the result block in pinned host memory.  One
// launch in place of two reduce passes, a finalize and a copy: 27 -> 18 us
// at 512^3 with 10 mu bins, 20 -> 13 us at 64^3 (launches counted alone).
// Auto power of every catalog (cross_b < 0: blockIdx.y = catalog), or the cross
// power of catalogs cross_a and cross_b: normalization
// L^3 / (sum w_a sum w_b), no shot noise; the result block then carries
// sum w_a and sum w_b in its wsum and w2sum slots.
template <typename A>
__global__ void __launch_bounds__(256)
k_reduce_finalize(const A *partial, int G, const unsigned long long *__restrict__ modes1d,
                  const unsigned long long *__restrict__ modes2d, const double *wsums, const int *err, FinalGeom f, ResultLayout rl, double *__restrict__ res, int cross_a,
                  int cross_b) {
    grid_wait();
    extern __shared__ __align__(16) unsigned char smraw[];
    double *sum = reinterpret_cast<double *>(smraw);       // the block's slots
    __shared__ double red[256];
    const bool cross = cross_b >= 0;
    const int item = blockIdx.y;
    // the normalization first: its FP64 divisions overlap the loads below
    const int ia = cross ? cross_a : item, ib = cross ? cross_b : item;
    double *r = res + (long long)item * f.RL;
    const double wsum = wsums[4 * ia], wsum_b = wsums[4 * ib];
    const double w2sum = cross ? wsum_b : wsums[4 * ia + 1];
    const double norm = f.L3 / (wsum * wsum_b);
    const double shot = cross ? 0.0 : f.L3 * w2sum / (wsum * wsum);
    const double sub = f.subtract_shot ? shot : 0.0;
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    const int KB = final_bins(f), b0 = blockIdx.x * KB, nb = min(KB, f.nk - b0);
    const int per = f.twod ? f.nmu : 1, n0 = nb * per, ns = n0 + (f.poles ? 2 * nb : 0);
    // slot s of the block: its (k, mu) or k sums, then the two pole sums per bin
    const auto slot = [&](int s) {
        if (s < n0) return b0 * per + s;
        s -= n0;
        return s < nb ? f.hbase + b0 + s : f.hbase + f.nk + b0 + s - nb;
    };
    const A *p = partial + (long long)item * G * f.nh;
    const int parts = ns < 256 ? 256 / ns : 1;
    for (int s0 = 0; s0 < ns; s0 += 256) {                 // one turn unless a bin has more than 254 mu bins
        const int s = s0 + (int)threadIdx.x % min(ns, 256), part = threadIdx.x / min(ns, 256);
        double t = 0.0;
        if (s < ns && part < parts) {
            const A *q = p + slot(s);
#pragma unroll 8
            for (int c = part; c < G; c += parts) t += (double)q[(long long)c * f.nh];
        }
        red[threadIdx.x] = t;
        __syncthreads();
        if (part == 0 && s < ns) {
            for (int k = 1; k < parts; ++k) t += red[threadIdx.x + k * ns];
            sum[s] = t;
        }
        __syncthreads();
    }

    // one thread per bin and multipole
    for (int k3 = threadIdx.x; k3 < 3 * nb; k3 += blockDim.x) {
        const int row = k3 / nb, k = k3 - row * nb, b = b0 + k;
        const double cnt = (double)modes1d[b];
        double p = nan;
        if (cnt > 0.0) {
            if (row == 0) {
                double S0 = 0.0;
                for (int q = 0; q < per; ++q) S0 += sum[k * per + q];
                p = norm * S0 / cnt - sub;
            } else if (f.poles) {        // slots: sum h P L_2(mu), sum h P L_4(mu)
                p = (row == 1 ? 5.0 : 9.0) * norm * sum[n0 + (row - 1) * nb + k] / cnt;
            }
        }
        if (row == 0) r[rl.pk + b] = p;
        r[rl.poles + row * f.nk + b] = ((f.poles_mask >> row) & 1u) ? p : nan;
    }
    if (f.twod) {
        for (int k = threadIdx.x; k < n0; k += blockDim.x) {
            const double cnt = (double)modes2d[b0 * per + k];
            r[rl.pkmu + b0 * per + k] = cnt > 0.0 ? norm * sum[k] / cnt - sub : nan;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const double wabs = fmax(wsums[4 * ia + 2], wsums[4 * ib + 2]);
        r[rl.shot] = shot;
        r[rl.wsum] = wsum;
        r[rl.w2sum] = w2sum;
        r[rl.flags] = (double)(((wabs > f.headroom) ? 1 : 0) | (*err & 6));
    }
}

// ---- projected power (ProjectedFFTPower): one plane or line of the transform ----
// By the projection-slice theorem the d-dimensional transform of the field
// summed over the dropped axes is the 3D transform at index 0 along them, so
// the projected power needs only those modes.  Each mode of the plane: the
// usual interlacing combine and compensation, |delta|^2 (times the half-grid
// weight h when z is kept), exact k bin from the m-edge table, FP64 atomics
// into count / sum h k / sum h |F|^2 cw per bin.
template <typename R, typename C>
__global__ void k_plane_bin(const C *__restrict__ m1, const C *__restrict__ m2, int N, int keep_mask,
                            const R *__restrict__ cw, const C *__restrict__ ph, const int *__restrict__ kedge,
                            int nk, double kF, double *__restrict__ sums) {
    const int Nh = N / 2 + 1;
    const int nx = (keep_mask & 1) ? N : 1, ny = (keep_mask & 2) ? N : 1, nz = (keep_mask & 4) ? Nh : 1;
    const long long total = (long long)nx * ny * nz;
    const int half = N / 2;
    for (long long f = (long long)blockIdx.x * blockDim.x + threadIdx.x; f < total;
         f += (long long)gridDim.x * blockDim.x) {
        const int l = (int)(f % nz);
        const long long r = f / nz;
        const int j = (int)(r % ny);
        const int i = (int)(r / ny);
        const int ip = i < half ? i : i - N, jp = j < half ? j : j - N;
        const long long m = (long long)ip * ip + (long long)jp * jp + (long long)l * l;
        if (m == 0 || m < kedge[0] || m >= kedge[nk]) continue;
        int a = 0, b = nk;                               // kedge[a] <= m < kedge[b]
        while (b - a > 1) {
            const int mid = (a + b) >> 1;
            if (kedge[mid] <= m) a = mid;
            else b = mid;
        }
        const long long idx = ((long long)i * N + j) * Nh + l;
        double zr = (double)m1[idx].x, zi = (double)m1[idx].y;
        double wgt = (double)cw[i] * (double)cw[j] * (double)cw[l];
        if (m2) {
            // e^{+i pi (i' + j' + l) / N} as the product of the per-axis phase table entries
            const C pa = ph[ip + half], pb = ph[jp + half], pc = ph[l + half];
            const double tr = (double)pa.x * pb.x - (double)pa.y * pb.y;
            const double ti = (double)pa.x * pb.y + (double)pa.y * pb.x;
            const double er = tr * pc.x - ti * pc.y, ei = tr * pc.y + ti * pc.x;
            const double br = (double)m2[idx].x, bi = (double)m2[idx].y;
            zr += br * er - bi * ei;
            zi += br * ei + bi * er;
            wgt *= 0.25;
        }
        const double h = ((keep_mask & 4) && l != 0 && l != half) ? 2.0 : 1.0;
        atomicAdd(sums + 3 * a, h);
        atomicAdd(sums + 3 * a + 1, h * kF * sqrt((double)m));
        atomicAdd(sums + 3 * a + 2, h * (zr * zr + zi * zi) * wgt);
    }
}

// ---- plan-time geometry: integer histograms over (m, q) ----
__global__ void k_geom_hist(BinGeom g, unsigned long long *__restrict__ H,
                            unsigned long long *__restrict__ HL) {
    const int nq = g.nmu > 0 ? g.nmu : 1;
    const int half = g.N / 2;
    for (long long row = blockIdx.x; row < (long long)g.N * g.N; row += gridDim.x) {
        const int i = (int)(row / g.N), j = (int)(row % g.N);
        const int ip = i < half ? i : i - g.N, jp = j < half ? j : j - g.N;
        const int r2 = ip * ip + jp * jp;
        for (int l = threadIdx.x; l < g.Nh; l += blockDim.x) {
            const int m = r2 + l * l;
            if (m == 0 || m < g.mlo || m >= g.mhi) continue;
            int q = 0;
            if (g.nmu > 0) {
                const long long rhs = (long long)g.nmu * g.nmu * l * l;
                while (q + 1 <= g.nmu - 1 && (long long)(q + 1) * (q + 1) * m <= rhs) ++q;
            }
            const unsigned long long h = (l == 0 || l == half) ? 1ull : 2ull;
            atomicAdd(H + (long long)m * nq + q, h);
            atomicAdd(HL + (long long)m * nq + q, h * (unsigned long long)l);
        }
    }
}

__global__ void k_geom_finalize(BinGeom g, const int *__restrict__ kedge, double kF,
                                const unsigned long long *__restrict__ H,
                                const unsigned long long *__restrict__ HL,
                                unsigned long long *__restrict__ modes2d,
                                double *__restrict__ kmean2d, double *__restrict__ mumean2d) {
    const int nq = g.nmu > 0 ? g.nmu : 1;
    const int idx = blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= g.nk * nq) return;
    const int b = idx / nq, q = idx % nq;
    unsigned long long cnt = 0;
    double ks = 0.0, mus = 0.0;
    const int m0 = max(kedge[b], 1), m1 = kedge[b + 1];
    for (int m = m0; m < m1; ++m) {
        const unsigned long long c = H[(long long)m * nq + q];
        if (c == 0) continue;
        const double sm = sqrt((double)m);
        cnt += c;
        ks += (double)c * sm;
        mus += (double)HL[(long long)m * nq + q] / sm;
    }
    const double nan = __longlong_as_double(0x7ff8000000000000LL);
    modes2d[idx] = cnt;
    kmean2d[idx] = cnt ? kF * ks / (double)cnt : nan;
    mumean2d[idx] = cnt ? mus / (double)cnt : nan;
}

template <typename K>
// Raise a kernel's dynamic shared-memory limit when the launch may pass the
// 48 KB default together with the kernel's static shared arrays (a few KB at
// most here), so an exactly-48 KB dynamic request is covered too.
cudaError_t set_smem(K kernel, size_t bytes) {
    if (bytes <= 40 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

unsigned grid_for(int64_t n, int threads, unsigned cap) {
    int64_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > (int64_t)cap) b = cap;
    return (unsigned)b;
}

}  // namespace

ResultLayout result_layout(int nk, int nmu) {
    ResultLayout r;
    r.pk = 0;
    r.poles = nk;
    r.pkmu = 4 * nk;
    r.shot = 4 * nk + nk * nmu;
    r.wsum = r.shot + 1;
    r.w2sum = r.shot + 2;
    r.flags = r.shot + 3;
    r.total = r.shot + 4;
    return r;
}

int paint_classes() { return kClasses; }

cudaError_t launch_sort_count(const void *pos, int dtype, const float *w, const float *vals,
                              const int64_t *item_off, int nitems, int64_t max_n, const PaintGeom &g,
                              uint32_t *count, double *wsums, double *wpart, uint4 *wmax, cudaStream_t st) {
    const bool weighted = w != nullptr || vals != nullptr || dtype == PK_F32X4;
    dim3 grid(grid_for(max_n, kCountThreads, weighted ? kWsumBlocks : 1u << 20), nitems);
#define PK_COUNT(DT)                                                                                    \
    if (weighted) chained(k_sort_count<DT, true>, grid, kCountThreads, 0, st)(pos, w, vals, item_off, max_n, g, count, wsums, wpart, wmax); \
    else chained(k_sort_count<DT, false>, grid, kCountThreads, 0, st)(pos, w, vals, item_off, max_n, g, count, wsums, wpart, wmax);
    switch (dtype) {
    case PK_F32: PK_COUNT(PK_F32) break;
    case PK_F64: PK_COUNT(PK_F64) break;
    default: PK_COUNT(PK_F32X4) break;
    }
#undef PK_COUNT
    if (weighted) {
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        chained(k_wsum_reduce, nitems, 256, 0, st)(wpart, (int)grid.x, item_off, max_n, wsums, wmax);
    }
    return cudaGetLastError();
}

size_t wsum_partial_elems(int nitems) { return (size_t)nitems * kWsumBlocks * 3; }

cudaError_t launch_sort_scatter(const void *pos, int dtype, const float *w, const float *vals,
                                const int64_t *item_off, int nitems, int64_t max_n, const PaintGeom &g,
                                uint32_t *cursor, float4 *sorted, uint32_t ntot, int *err, cudaStream_t st) {
    dim3 grid(grid_for(max_n, kCountThreads, 1u << 20), nitems);
    switch (dtype) {
    case PK_F32: chained(k_sort_scatter<PK_F32>, grid, kCountThreads, 0, st)(pos, w, vals, item_off, max_n, g, cursor, sorted, ntot, err); break;
    case PK_F64: chained(k_sort_scatter<PK_F64>, grid, kCountThreads, 0, st)(pos, w, vals, item_off, max_n, g, cursor, sorted, ntot, err); break;
    default: chained(k_sort_scatter<PK_F32X4>, grid, kCountThreads, 0, st)(pos, w, vals, item_off, max_n, g, cursor, sorted, ntot, err); break;
    }
    return cudaGetLastError();
}

// Small host arrays travel as kernel parameters (copied at launch, so the
// host may reuse its array at once and a captured graph keeps the values).
struct I64Chunk {
    int64_t v[kUploadChunk];
};

__global__ void k_upload_i64(int64_t *__restrict__ dst, I64Chunk c, int n) {
    if ((int)threadIdx.x < n) dst[threadIdx.x] = c.v[threadIdx.x];
}

cudaError_t launch_upload_i64(int64_t *dst, const int64_t *src, int n, int *launches, cudaStream_t st) {
    for (int b = 0; b < n; b += kUploadChunk) {
        const int m = n - b < kUploadChunk ? n - b : kUploadChunk;
        I64Chunk c;
        for (int k = 0; k < m; ++k) c.v[k] = src[b + k];
        k_upload_i64<<<1, kUploadChunk, 0, st>>>(dst + b, c, m);
        *launches += 1;
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

size_t scan_tmp_elems(int64_t n) {
    size_t t = 0;
    while (n > 1) {
        const int64_t nb = (n + kScanTile - 1) / kScanTile;
        t += (size_t)nb + 1;
        n = nb;
    }
    return t + 2;
}

template <typename T, bool COPY>
static cudaError_t scan_impl(const T *in, int64_t n, T *out, T *tmp, T *copy, int *launches, cudaStream_t st) {
    const int64_t nb = (n + kScanTile - 1) / kScanTile;
    if (nb <= 1) {
        chained(k_scan_blocks<T, COPY>, 1, kScanThreads, 0, st)(in, n, out, out + n, copy);
        *launches += 1;
        return cudaGetLastError();
    }
    if (nb > 0x7fffffffLL) return cudaErrorInvalidValue;
    chained(k_scan_blocks<T, false>, (unsigned)nb, kScanThreads, 0, st)(in, n, out, tmp, nullptr);
    *launches += 1;
    if (nb <= kScanDirect) {
        chained(k_scan_add<T, COPY, true>, (unsigned)nb, kScanThreads, 0, st)(out, n, tmp, (int)nb, copy);
        *launches += 1;
        return cudaGetLastError();
    }
    cudaError_t e = scan_impl<T, false>(tmp, nb, tmp, tmp + nb + 1, nullptr, launches, st);
    if (e != cudaSuccess) return e;
    chained(k_scan_add<T, COPY, false>, (unsigned)nb, kScanThreads, 0, st)(out, n, tmp, (int)nb, copy);
    *launches += 1;
    return cudaGetLastError();
}

// out[0 .. n) = exclusive scan of in, out[n] = total; in[0 .. n) gets a copy of
// out[0 .. n).  tmp: scan_tmp_elems(n).
cudaError_t launch_scan(uint32_t *in, int64_t n, uint32_t *out, uint32_t *tmp, int *launches, cudaStream_t st) {
    return scan_impl<uint32_t, true>(in, n, out, tmp, in, launches, st);
}

cudaError_t launch_scan64(const unsigned long long *in, int64_t n, unsigned long long *out,
                          unsigned long long *tmp, int *launches, cudaStream_t st) {
    return scan_impl<unsigned long long, false>(in, n, out, tmp, nullptr, launches, st);
}

size_t paint_smem_bytes(int T, int window, int nmesh) {
    const size_t general = (size_t)paint_cell_words(T) * sizeof(unsigned) + (size_t)kStage * sizeof(float4);
    const size_t words = window == 4   ? (size_t)nmesh * SweepLayout<4>::Words
                         : window == 3 ? (size_t)nmesh * SweepLayout<3>::Words : 0;
    const size_t padded = T == 16 && words ? (words + CoarseBlocks<3>::Count) * sizeof(unsigned) : 0;
    return general > padded ? general : padded;
}

template <int P, int NM, typename M, bool UNIT>
static cudaError_t paint_inst(const float4 *sorted, const uint32_t *off, const uint32_t *cursor, int *err, int nitems,
                              const PaintGeom &g, int S, const uint4 *wmax, float wdep, void *mesh, long long item_stride, long long mesh_stride, int accumulate,
                              cudaStream_t st) {
    const size_t smem = paint_smem_bytes(g.T, P, NM);   // one padded mesh fits the general area
    const long long nblocks = (long long)nitems * g.ntiles;
    if (nblocks <= 0) return cudaSuccess;
    if (nblocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    auto kern = g.T == 16 ? k_paint_tiles<P, NM, M, 16, UNIT> : k_paint_tiles<P, NM, M, 0, UNIT>;
    cudaError_t e = set_smem(kern, smem);
    if (e != cudaSuccess) return e;
    chained(kern, (unsigned)nblocks, kPaintThreads, smem, st)(sorted, off, cursor, err, g, S, wmax, wdep,
                                                         reinterpret_cast<M *>(mesh), item_stride,
                                                         mesh_stride, accumulate);
    return cudaGetLastError();
}

cudaError_t launch_paint_tiles(const float4 *sorted, const uint32_t *off, const uint32_t *cursor, int *err,
                               int nitems, const PaintGeom &g, int window, int nmesh, int S, int f64,
                               const uint4 *wmax, int unit_weights, void *mesh, long long item_stride, long long mesh_stride,
                               int accumulate, cudaStream_t st) {
    // The window's largest weight: (largest per-axis weight)^3.
    const float wdep = window == 2 ? 1.0f : window == 3 ? 0.421875f : 0.2962963f;
#define PK_PAINT_INST(P, NM, M)                                                                                  \
    (unit_weights ? paint_inst<P, NM, M, true>(sorted, off, cursor, err, nitems, g, S, wmax, wdep, mesh, \
                                               item_stride, mesh_stride, accumulate, st)                          \
                  : paint_inst<P, NM, M, false>(sorted, off, cursor, err, nitems, g, S, wmax, wdep, mesh, \
                                                item_stride, mesh_stride, accumulate, st))
#define PK_PAINT_CASE(P)                                                                                         \
    if (window == P) {                                                                                           \
        if (f64) return nmesh == 2 ? PK_PAINT_INST(P, 2, double) : PK_PAINT_INST(P, 1, double);                  \
        return nmesh == 2 ? PK_PAINT_INST(P, 2, float) : PK_PAINT_INST(P, 1, float);                             \
    }
    PK_PAINT_CASE(2)
    PK_PAINT_CASE(3)
    PK_PAINT_CASE(4)
#undef PK_PAINT_CASE
#undef PK_PAINT_INST
    return cudaErrorInvalidValue;
}

template <int DT, int P, int NM>
static cudaError_t atomic_inst(const void *pos, const float *w, const float *vals, const int64_t *item_off, int nitems,
                               int64_t max_n, const PaintGeom &g, int S, bool weighted,
                               unsigned long long *acc, double *wsums, double *wpart, uint4 *wmax,
                               cudaStream_t st) {
    dim3 grid(grid_for(max_n, kCountThreads, weighted ? kWsumBlocks : 1u << 20), nitems);
    k_paint_atomic<DT, P, NM><<<grid, kCountThreads, 0, st>>>(pos, w, vals, item_off, max_n, g, S, weighted, acc,
                                                             wsums, wpart, wmax);
    if (weighted) {
        cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        chained(k_wsum_reduce, nitems, 256, 0, st)(wpart, (int)grid.x, item_off, max_n, wsums, wmax);
    }
    return cudaGetLastError();
}

template <int DT>
static cudaError_t atomic_dispatch(const void *pos, const float *w, const float *vals, const int64_t *item_off, int nitems,
                                   int64_t max_n, const PaintGeom &g, int window, int nmesh, int S,
                                   bool weighted, unsigned long long *acc, double *wsums, double *wpart,
                                   uint4 *wmax, cudaStream_t st) {
#define PK_ATOMIC_CASE(P)                                                                              \
    if (window == P)                                                                                   \
        return nmesh == 2 ? atomic_inst<DT, P, 2>(pos, w, vals, item_off, nitems, max_n, g, S, weighted, acc, \
                                                  wsums, wpart, wmax, st)                             \
                          : atomic_inst<DT, P, 1>(pos, w, vals, item_off, nitems, max_n, g, S, weighted, acc, \
                                                  wsums, wpart, wmax, st);
    PK_ATOMIC_CASE(2)
    PK_ATOMIC_CASE(3)
    PK_ATOMIC_CASE(4)
#undef PK_ATOMIC_CASE
    return cudaErrorInvalidValue;
}

cudaError_t launch_paint_atomic(const void *pos, int dtype, const float *w, const float *vals,
                                const int64_t *item_off, int nitems, int64_t max_n, const PaintGeom &g,
                                int window, int nmesh, int S, unsigned long long *acc, double *wsums,
                                double *wpart, uint4 *wmax, cudaStream_t st) {
    const bool weighted = w != nullptr || vals != nullptr || dtype == PK_F32X4;
    switch (dtype) {
    case PK_F32:
        return atomic_dispatch<PK_F32>(pos, w, vals, item_off, nitems, max_n, g, window, nmesh, S, weighted, acc,
                                       wsums, wpart, wmax, st);
    case PK_F64:
        return atomic_dispatch<PK_F64>(pos, w, vals, item_off, nitems, max_n, g, window, nmesh, S, weighted, acc,
                                       wsums, wpart, wmax, st);
    default:
        return atomic_dispatch<PK_F32X4>(pos, w, vals, item_off, nitems, max_n, g, window, nmesh, S, weighted,
                                         acc, wsums, wpart, wmax, st);
    }
}

cudaError_t launch_acc_to_mesh(unsigned long long *acc, int nitems, int nmesh, int N, int S, int f64,
                               void *mesh, long long item_stride, long long mesh_stride, int accumulate,
                               int nsm, cudaStream_t st) {
    const long long npairs = (long long)nitems * nmesh * N * N * N / 2;
    if (npairs <= 0) return cudaSuccess;
    const unsigned grid = grid_for(npairs, 256, (unsigned)(nsm > 0 ? nsm * 8 : 1024));
    const float inv_scale = ldexpf(1.0f, -S);
    ulonglong2 *a2 = reinterpret_cast<ulonglong2 *>(acc);
    if (f64)
        k_acc_to_mesh<double><<<grid, 256, 0, st>>>(a2, npairs, N, nmesh, inv_scale,
                                                    reinterpret_cast<double *>(mesh), item_stride,
                                                    mesh_stride, accumulate);
    else
        k_acc_to_mesh<float><<<grid, 256, 0, st>>>(a2, npairs, N, nmesh, inv_scale,
                                                   reinterpret_cast<float *>(mesh), item_stride,
                                                   mesh_stride, accumulate);
    return cudaGetLastError();
}

size_t bin_smem_bytes(const BinGeom &g, int f64) {
    return f64 ? BinSmem<double, double2, double>::bytes(g) : BinSmem<float, float2, float>::bytes(g);
}

int bin_threads() { return kBinThreads; }

// The pass of either form, chosen by the types.
template <bool IL, bool TWOD, bool POLES, typename R, typename C, bool CROSS, bool MU32>
static auto bin_kernel() {
    if constexpr (sizeof(R) == 4) return k_bin<IL, TWOD, POLES, CROSS, MU32>;
    else return k_bin_f64<IL, TWOD, POLES, CROSS, MU32>;
}

template <bool IL, bool TWOD, bool POLES, typename R, typename C, bool CROSS>
static cudaError_t bin_inst(const void *mesh, long long item_stride_c, long long mesh_stride_c,
                            int nitems, int G, const BinGeom &g, const void *cw, const void *ph,
                            const int *kedge, void *partial, const void *meshb, cudaStream_t st) {
    const size_t smem = bin_smem_bytes(g, sizeof(R) == 8);
    auto kern = (g.mu32 || !TWOD) ? bin_kernel<IL, TWOD, POLES, R, C, CROSS, true>()
                                  : bin_kernel<IL, TWOD, POLES, R, C, CROSS, false>();
    cudaError_t e = set_smem(kern, smem);
    if (e != cudaSuccess) return e;
    dim3 grid(G, nitems);
    chained(kern, grid, kBinThreads, smem, st)(reinterpret_cast<const C *>(mesh), item_stride_c,
                                          mesh_stride_c, g, reinterpret_cast<const R *>(cw),
                                          reinterpret_cast<const C *>(ph), kedge,
                                          reinterpret_cast<R *>(partial), reinterpret_cast<const C *>(meshb));
    return cudaGetLastError();
}

template <typename R, typename C, bool CROSS>
static cudaError_t bin_dispatch(const void *mesh, int il, long long is, long long ms, int nitems,
                                int G, const BinGeom &g, const void *cw, const void *ph,
                                const int *kedge, void *partial, const void *meshb, cudaStream_t st) {
    const int key = (il ? 4 : 0) | (g.twod ? 2 : 0) | (g.poles ? 1 : 0);
#define PK_BIN(a, b, c) bin_inst<a, b, c, R, C, CROSS>(mesh, is, ms, nitems, G, g, cw, ph, kedge, partial, meshb, st)
    switch (key) {
    case 0: return PK_BIN(false, false, false);
    case 1: return PK_BIN(false, false, true);
    case 2: return PK_BIN(false, true, false);
    case 3: return PK_BIN(false, true, true);
    case 4: return PK_BIN(true, false, false);
    case 5: return PK_BIN(true, false, true);
    case 6: return PK_BIN(true, true, false);
    default: return PK_BIN(true, true, true);
    }
#undef PK_BIN
}

cudaError_t launch_bin(const void *mesh, int f64, int interlaced, long long item_stride_c,
                       long long mesh_stride_c, int nitems, int ctas_per_item,
                       const BinGeom &g, const void *cw, const void *ph, const int *kedge,
                       void *partial, cudaStream_t st) {
    if (f64)
        return bin_dispatch<double, double2, false>(mesh, interlaced, item_stride_c, mesh_stride_c, nitems,
                                                    ctas_per_item, g, cw, ph, kedge, partial, nullptr, st);
    return bin_dispatch<float, float2, false>(mesh, interlaced, item_stride_c, mesh_stride_c, nitems,
                                              ctas_per_item, g, cw, ph, kedge, partial, nullptr, st);
}

cudaError_t launch_bin_cross(const void *mesh_a, const void *mesh_b, int f64, int interlaced,
                             long long mesh_stride_c, int ctas, const BinGeom &g, const void *cw,
                             const void *ph, const int *kedge, void *partial, cudaStream_t st) {
    if (f64)
        return bin_dispatch<double, double2, true>(mesh_a, interlaced, 0, mesh_stride_c, 1, ctas, g, cw, ph, kedge,
                                                   partial, mesh_b, st);
    return bin_dispatch<float, float2, true>(mesh_a, interlaced, 0, mesh_stride_c, 1, ctas, g, cw, ph, kedge,
                                             partial, mesh_b, st);
}

int bin_ctas_per_sm(const BinGeom &g, int f64) {
    int n = 0;
    const size_t smem = bin_smem_bytes(g, f64);
    cudaError_t e;
    if (f64) {
        auto k = k_bin_f64<true, true, true, false, true>;
        set_smem(k, smem);
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, kBinThreads, smem);
    } else {
        auto k = k_bin<true, true, true, false, true>;
        set_smem(k, smem);
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, kBinThreads, smem);
    }
    if (e != cudaSuccess || n < 1) n = 1;
    return n;
}

cudaError_t launch_reduce_finalize(const void *partial, int f64, int G, const unsigned long long *modes1d,
                                   const unsigned long long *modes2d, const double *wsums, const int *err,
                                   const FinalGeom &f, int nitems, double *res, int cross_a, int cross_b,
                                   cudaStream_t st) {
    const ResultLayout rl = result_layout(f.nk, f.nmu);
    const int KB = final_bins(f);
    const size_t smem = sizeof(double) * (size_t)KB * ((f.twod ? f.nmu : 1) + (f.poles ? 2 : 0));   // <= 8 KB
    const dim3 grid((f.nk + KB - 1) / KB, nitems);
    if (f64)
        chained(k_reduce_finalize<double>, grid, 256, smem, st)(reinterpret_cast<const double *>(partial), G, modes1d,
                                                           modes2d, wsums, err, f, rl, res, cross_a, cross_b);
    else
        chained(k_reduce_finalize<float>, grid, 256, smem, st)(reinterpret_cast<const float *>(partial), G, modes1d,
                                                          modes2d, wsums, err, f, rl, res, cross_a, cross_b);
    return cudaGetLastError();
}

cudaError_t launch_plane_bin(const void *m1, const void *m2, int f64, int N, int keep_mask, const void *cw,
                             const void *ph, const int *kedge, int nk, double kF, double *sums, int nsm,
                             cudaStream_t st) {
    const int Nh = N / 2 + 1;
    const long long total = (long long)((keep_mask & 1) ? N : 1) * ((keep_mask & 2) ? N : 1) * ((keep_mask & 4) ? Nh : 1);
    const unsigned grid = grid_for(total, 256, (unsigned)(nsm > 0 ? nsm * 8 : 1024));
    if (f64)
        k_plane_bin<double, double2><<<grid, 256, 0, st>>>(
            reinterpret_cast<const double2 *>(m1), reinterpret_cast<const double2 *>(m2), N, keep_mask,
            reinterpret_cast<const double *>(cw), reinterpret_cast<const double2 *>(ph), kedge, nk, kF, sums);
    else
        k_plane_bin<float, float2><<<grid, 256, 0, st>>>(
            reinterpret_cast<const float2 *>(m1), reinterpret_cast<const float2 *>(m2), N, keep_mask,
            reinterpret_cast<const float *>(cw), reinterpret_cast<const float2 *>(ph), kedge, nk, kF, sums);
    return cudaGetLastError();
}

cudaError_t launch_geom_hist(const BinGeom &g, unsigned long long *H, unsigned long long *HL,
                             cudaStream_t st) {
    const long long rows = (long long)g.N * g.N;
    const unsigned grid = (unsigned)(rows < 65536 ? rows : 65536);
    k_geom_hist<<<grid, 256, 0, st>>>(g, H, HL);
    return cudaGetLastError();
}

cudaError_t launch_geom_finalize(const BinGeom &g, const int *kedge, double kF,
                                 const unsigned long long *H, const unsigned long long *HL,
                                 unsigned long long *modes2d, double *kmean2d, double *mumean2d,
                                 cudaStream_t st) {
    const int nq = g.nmu > 0 ? g.nmu : 1;
    const int n = g.nk * nq;
    k_geom_finalize<<<(n + 127) / 128, 128, 0, st>>>(g, kedge, kF, H, HL, modes2d, kmean2d, mumean2d);
    return cudaGetLastError();
}

}  // namespace pk
