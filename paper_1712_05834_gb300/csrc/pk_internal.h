// pk_internal.h -- declarations shared by the translation units of libpk.so.  Not
// installed.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/pk.h"

namespace pk {

// Message of the last failed plan creation on this thread (pk_plan_error).
void set_plan_error(const char *msg);

// Geometry of the tile-sorted paint (Sec. 3.3.1 painting, Sec. 3.3.2 windows).
// The mesh is cut into cubic tiles of T^3 cells.  Each object is sorted by
// (home tile, boundary class); the paint CTA of a tile gathers its own objects
// and the boundary classes of its 26 neighbours.  Cells [floor(s)+lo,
// floor(s)+hi] along each axis cover the window support on both meshes.
struct PaintGeom {
    float invH;         // N / L in FP32
    float invH_lo;      // N / L - invH (the FP32 rounding residual)
    double invHd;       // N / L in FP64
    int N;              // cells per side
    int T;              // tile edge (divides N, T >= hi - lo)
    int flog;           // 1: tiles are halves (along each axis) of frames of 2 T cells, in
                        // which positions are held; 0: a tile is its own frame
    unsigned inv_F;     // ceil(2^20 / F), F = T << flog: cell / F = cell * inv_F >> 20 exactly
                        // for cell < 4096 (the excess, below 2^-8, is less than 1 / F)
    int ntx;            // tiles per side = N / T
    int lo, hi;         // reach of the window support relative to floor(s)
    long long ntiles;   // ntx^3 tiles per catalog
};

// Geometry of the fused compensate + interlace + bin pass (Sec. 3.4.1).
struct BinGeom {
    int N, Nh;              // Nh = N/2 + 1 stored z modes
    int nk, nmu;            // k bins, mu bins (nmu = 0: 1D only)
    int twod, poles;        // accumulate (k, mu) sums / mu^2, mu^4 sums
    int hbase;              // first pole slot in the per-CTA histogram
    int nh;                 // histogram length
    float kscale, koff;     // bin estimate: sqrt(m) * kscale - koff
    int mlo, mhi;           // binned modes have mlo <= m < mhi (and m != 0)
    int mu32;               // nmu^2 * max m < 2^32: mu-bin checks in 32 bits
};

struct FinalGeom {
    int nk, nmu, twod, poles, hbase, nh;
    unsigned poles_mask;
    int subtract_shot;
    double L3;              // L^3
    double headroom;        // 2^(62 - S): largest sum |w| with int64 cells safe
    int RL;                 // doubles per item in the result block
};

// Offsets inside one item's FP64 result block.
struct ResultLayout {
    int pk, poles, pkmu, shot, wsum, w2sum, flags, total;
};
ResultLayout result_layout(int nk, int nmu);

// ---- scans ----
constexpr int kScanThreads = 1024;
constexpr int kScanPer = 4;           // elements per thread in a scan block
constexpr int kScanTile = kScanThreads * kScanPer;

#ifdef __CUDACC__
// Launches whose overhead overlaps the kernel before (programmatic dependent launch):
// the kernel begins with grid_wait(), which returns when every kernel before it on the
// stream has ended and its writes can be seen.  Grids up to kChainedCtas; those up to
// kEarlyCtas also let the next kernel's CTAs in as soon as all of their own have
// started: a 64^3 catalog 86 -> 72 us, weighted 100^3 halos 121 -> 104, 2e6 objects at
// 256^3 241 -> 219 (231 with only those chained; early entry at every size: 246, and 1e7
// objects at 512^3 2.31 ms for 2.01).
constexpr unsigned kChainedCtas = 8192, kEarlyCtas = 1216;
template <typename... Args>
struct ChainedLaunch {
    void (*kernel)(Args...);
    dim3 grid, block;
    size_t smem;
    cudaStream_t st;
    void operator()(Args... args) const {
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = grid;
        cfg.blockDim = block;
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cfg.attrs = &attr;
        cfg.numAttrs = (unsigned long long)grid.x * grid.y <= kChainedCtas ? 1 : 0;
        cudaLaunchKernelEx(&cfg, kernel, args...);          // an error is left to cudaGetLastError
    }
};
template <typename... Args>
ChainedLaunch<Args...> chained(void (*kernel)(Args...), dim3 grid, dim3 block, size_t smem, cudaStream_t st) {
    return {kernel, grid, block, smem, st};
}
// Such a kernel begins before the kernel ahead of it has ended, so what a kernel of the
// same call wrote is not constant over its lifetime: it is read through plain pointers
// (const without __restrict__, no __ldg), not through the read-only path.
// p: pointers to the caller's data, constant from before the call on and read through
// that path; they get an offset (zero) that the compiler first knows after the wait, so
// that no load through them can move above it.
template <typename... P>
__device__ __forceinline__ void grid_wait(P &...p) {
    const unsigned long long ctas = (unsigned long long)gridDim.x * gridDim.y;
    if (ctas <= kChainedCtas) asm volatile("griddepcontrol.wait;" ::: "memory");
    if (ctas <= kEarlyCtas) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    int zero;
    asm volatile("mov.b32 %0, 0;" : "=r"(zero)::"memory");
    ((p = (P)((const char *)p + zero)), ...);
}

// Exclusive scan of one value per thread of a kScanThreads block.
template <typename T>
__device__ __forceinline__ T block_exclusive_scan(T v, T *total) {
    __shared__ T wsum[kScanThreads / 32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    T x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const T y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[wid] = x;
    __syncthreads();
    if (wid == 0) {
        T s = lane < kScanThreads / 32 ? wsum[lane] : (T)0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const T y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < kScanThreads / 32) wsum[lane] = s;
    }
    __syncthreads();
    const T before = (wid > 0 ? wsum[wid - 1] : (T)0) + x - v;
    *total = wsum[kScanThreads / 32 - 1];
    __syncthreads();
    return before;
}
#endif

// ---- launchers (pk_kernels.cu); all asynchronous on `st` ----
int paint_classes();                  // boundary classes per tile (27)
// dynamic shared memory of one tile-paint CTA painting nmesh meshes
size_t paint_smem_bytes(int T, int window, int nmesh = 2);
size_t scan_tmp_elems(int64_t n);
// dst[0 .. n) = src[0 .. n) for a host array src, through kernel parameters
// (the host array may be reused as soon as the call returns).
cudaError_t launch_upload_i64(int64_t *dst, const int64_t *src, int n, int *launches, cudaStream_t st);
// item_off: the catalogs' offsets on the device, or NULL for one catalog of max_n
// objects.  w: weights (normalization; NULL = 1), vals: painted values V (NULL = 1);
// each object deposits W V and the sums keep sum W, sum (W V)^2, sum |W V|.
cudaError_t launch_sort_count(const void *pos, int dtype, const float *w, const float *vals,
                              const int64_t *item_off, int nitems, int64_t max_n, const PaintGeom &g,
                              uint32_t *count, double *wsums, double *wpart, uint4 *wmax, cudaStream_t st);
// Doubles of the per-block weight-sum rows (wpart) for nitems catalogs.
size_t wsum_partial_elems(int nitems);
// exclusive scan into out (total in out[n]) and, in place of the counts, into in
cudaError_t launch_scan(uint32_t *in, int64_t n, uint32_t *out, uint32_t *tmp, int *launches,
                        cudaStream_t st);
cudaError_t launch_scan64(const unsigned long long *in, int64_t n, unsigned long long *out,
                          unsigned long long *tmp, int *launches, cudaStream_t st);
cudaError_t launch_sort_scatter(const void *pos, int dtype, const float *w, const float *vals,
                                const int64_t *item_off, int nitems, int64_t max_n, const PaintGeom &g,
                                uint32_t *cursor, float4 *sorted, uint32_t ntot, int *err, cudaStream_t st);
// off, cursor: the scan's offsets and their copy as the scatter left it (err: 2
// if a cursor is not at the next key's offset).
cudaError_t launch_paint_tiles(const float4 *sorted, const uint32_t *off, const uint32_t *cursor, int *err,
                               int nitems, const PaintGeom &g, int window, int nmesh, int S, int f64,
                               const uint4 *wmax, int unit_weights, void *mesh, long long item_stride, long long mesh_stride,
                               int accumulate, cudaStream_t st);

// Direct atomic paint into dense int64 accumulators (nitems x nmesh x N^3,
// zero on entry), then conversion into the r2c mesh layout (clears them).
cudaError_t launch_paint_atomic(const void *pos, int dtype, const float *w, const float *vals,
                                const int64_t *item_off, int nitems, int64_t max_n, const PaintGeom &g,
                                int window, int nmesh, int S, unsigned long long *acc, double *wsums,
                                double *wpart, uint4 *wmax, cudaStream_t st);
cudaError_t launch_acc_to_mesh(unsigned long long *acc, int nitems, int nmesh, int N, int S, int f64,
                               void *mesh, long long item_stride, long long mesh_stride, int accumulate,
                               int nsm, cudaStream_t st);

cudaError_t launch_bin(const void *mesh, int f64, int interlaced, long long item_stride_c,
                       long long mesh_stride_c, int nitems, int ctas_per_item,
                       const BinGeom &g, const void *cw, const void *ph, const int *kedge,
                       void *partial, cudaStream_t st);
// Cross power of two catalogs: mesh_a / mesh_b point at each catalog's first
// mesh (the interlaced one follows at mesh_stride_c); one item, `ctas` CTAs.
cudaError_t launch_bin_cross(const void *mesh_a, const void *mesh_b, int f64, int interlaced,
                             long long mesh_stride_c, int ctas, const BinGeom &g, const void *cw,
                             const void *ph, const int *kedge, void *partial, cudaStream_t st);
size_t bin_smem_bytes(const BinGeom &g, int f64);
int bin_ctas_per_sm(const BinGeom &g, int f64);
int bin_threads();
// Per-CTA histograms (G rows per catalog) -> result blocks in res (pinned host
// memory): every catalog's auto power (cross_b < 0), or one cross power.
cudaError_t launch_reduce_finalize(const void *partial, int f64, int G, const unsigned long long *modes1d,
                                   const unsigned long long *modes2d, const double *wsums, const int *err,
                                   const FinalGeom &f, int nitems, double *res, int cross_a, int cross_b,
                                   cudaStream_t st);

// Projected power: bin the plane / line of one catalog's transform that keeps
// the axes in keep_mask (bit a: axis a); sums[3 b + {0,1,2}] += h, h k, h |F|^2 cw.
cudaError_t launch_plane_bin(const void *m1, const void *m2, int f64, int N, int keep_mask, const void *cw,
                             const void *ph, const int *kedge, int nk, double kF, double *sums, int nsm,
                             cudaStream_t st);

// ---- own FFT path (pk_fft.cu), FP32 meshes with N in {128, 192, 256, 512} ----
// The meshes' z rows are read as N/2 complex values (packed real pairs).
bool own_fft_packed(int N);
void own_fft_twiddles(int N, float *tw);          // tw[2e], tw[2e+1] = W_N^e, e < N
// length-N FFTs along y, then along x, of nmesh packed meshes mesh_c complex apart;
// rows (kx, ky) with kx^2 + ky^2 >= mhi are not written by the x pass
cudaError_t launch_fft_xy(void *mesh, int nmesh, long long mesh_c, int N, int mhi, const void *tw, cudaStream_t st);
// z transform + r2c split + the bin pass of launch_bin (FP32 form), partial
// histograms as launch_bin writes them
cudaError_t launch_zbin(const void *mesh, int interlaced, long long item_stride_c, long long mesh_stride_c,
                        int nitems, int ctas_per_item, const BinGeom &g, const void *cw, const void *ph,
                        const void *tw, const int *kedge, void *partial, cudaStream_t st);
size_t zbin_smem_bytes(const BinGeom &g, int interlaced);
int zbin_ctas_per_sm(const BinGeom &g, int interlaced);
// z transform + r2c split written back in place (the meshes then hold the r2c transform)
cudaError_t launch_zfinish(void *mesh, int interlaced, long long item_stride_c, long long mesh_stride_c,
                           int nitems, int N, const void *tw, int nsm, cudaStream_t st);

// ---- own FFT path (pk_fft_zyx.cu): z and y axes in one pass, then x ----
// Rows of a survey field formed on the way into the z axis: (D - alpha R) Y_lm(x^).
struct SurveyRows {
    const void *D = nullptr, *R = nullptr;     // real meshes in the r2c row layout; R may be NULL
    const double *alpha = nullptr;             // device: the factor of R
    long long slot_c = 0;                      // complex elements between the slots' meshes
    int s0 = -1, nslot = 1;                    // Y_lm slots s0 .. s0 + nslot - 1 (-1: weight 1)
    float ox = 0, oy = 0, oz = 0, H = 0;       // node (i, j, k) at o + H (i, j, k), in any unit near the box edge
};
struct ZyxOps {
    virtual bool plan_default() const = 0;     // box spectra of this size use it
    // zy into mesh, the first of sv.nslot meshes, of the rows described by sv, nx x
    // planes each; sync: 1 + nx * nslot counters.
    virtual cudaError_t zy_survey(void *mesh, int nx, const SurveyRows &sv, int ncol, int mcut, const void *tw,
                                  unsigned *sync, int *err, int nsm, cudaStream_t st) const = 0;
    // Columns l of one x tile; tile lists hold
    // ky index * 65536 + column block for the tiles with a mode m < mhi.
    virtual int tile_columns() const = 0;
    // z and y axes of `planes` consecutive x planes; only columns l < ncol and
    // rows with ky^2 + l^2 below mcut are transformed.  sync: 1 + planes
    // counters, zero on entry, cleared by the next x.  err: 4 if a wait
    // gave up.
    virtual cudaError_t zy(void *mesh, int planes, int ncol, int mcut, const void *tw, unsigned *sync, int *err,
                           int nsm, cudaStream_t st) const = 0;
    // x axis of nmesh meshes in place (tiles: tile_columns() wide).
    virtual cudaError_t x(void *mesh, int nmesh, long long mesh_c, int ncol, int mcut, const int *tiles, int ntiles,
                          const void *tw, unsigned *sync, int nsync, cudaStream_t st) const = 0;

protected:
    ~ZyxOps() = default;
};
// The counters of the z / y pass before a launch of it: zero at first and again after
// every x axis pass; cleared here if the pass that should have done so was never launched
// (the z / y pass would find its last ticket given out and leave the mesh as it is).
// *used: set until the x axis pass is on the stream.
inline cudaError_t zyx_counters(unsigned *sync, int nsync, int *used, cudaStream_t st) {
    const cudaError_t e = *used ? cudaMemsetAsync(sync, 0, sizeof(unsigned) * nsync, st) : cudaSuccess;
    *used = 1;
    return e;
}
const ZyxOps *zyx_ops_group0(int N);
const ZyxOps *zyx_ops_group1(int N);
const ZyxOps *zyx_ops_group2(int N);
// The launchers of size N (static storage), or NULL.
inline const ZyxOps *zyx_ops(int N) {
    const ZyxOps *o = zyx_ops_group0(N);
    if (!o) o = zyx_ops_group1(N);
    if (!o) o = zyx_ops_group2(N);
    return o;
}

// ---- own FFT path of FP64 meshes (pk_fft64.cu) ----
struct Fft64 {
    int N, nsteps, lc;                // lc: log2 of the lines per tile
    unsigned char radix[12];
    const double2 *tw;                // device: W_N^e (e < N), then the same halved
    const unsigned short *pos;        // device: place of frequency f after the steps
};
bool fft64_plan(int N, Fft64 *f);     // false: no own transform of this size
void fft64_tables(const Fft64 &f, double *tw, unsigned short *pos);    // 4 N reals, N places
// r2c of nmesh meshes in place; modes with |n|^2 >= mhi need not be transformed
cudaError_t launch_fft64(double *mesh, int nmesh, long long mesh_reals, const Fft64 &f, int mhi, cudaStream_t st);

cudaError_t launch_geom_hist(const BinGeom &g, unsigned long long *H, unsigned long long *HL,
                             cudaStream_t st);
cudaError_t launch_geom_finalize(const BinGeom &g, const int *kedge, double kF,
                                 const unsigned long long *H, const unsigned long long *HL,
                                 unsigned long long *modes2d, double *kmean2d, double *mumean2d,
                                 cudaStream_t st);

}  // namespace pk
