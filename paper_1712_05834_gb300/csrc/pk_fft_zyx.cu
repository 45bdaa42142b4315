// pk_fft_zyx.cu -- the library's own 3D r2c transform of FP32 meshes for sizes
// where it beats both cuFFT and the packed transform of pk_fft.cu, with its
// last axis fused into the bin pass (the transform of Sec. 3.3.1; the binning
// of Sec. 3.4.1, Eq. window-deconvolution).  In place, in the padded r2c
// layout (rows of N/2 + 1 complex), two kernels per compute:
//
//   k_fft_zy     z and y axes in one pass over device memory.  Persistent CTAs
//                take work items in ticket order: "z" items read a block of
//                real rows of one x plane, transform them (length-N/2 complex
//                FFT of the pairs d[2n] + i d[2n+1] and the real-input split
//                  D[l] = (C[l] + conj C[M-l]) / 2
//                         - (i/2) W_N^l (C[l] - conj C[M-l]),  M = N/2)
//                and write them back; "y" items transform a tile of columns
//                of a plane whose z items are done.  A plane's y items follow
//                its z items Cfg::LAG planes later, so they read the rows from
//                L2 (129 MB) and overwrite them there: device memory sees one
//                read and one write for two axes (512^3: 2.1 GB counted, where
//                two passes move 4.3).
//   k_fft_x      the x axis, written back in place; k_bin then bins the modes.  A
//                pass that took x and binned from shared memory at 1024 and 2048
//                was faster (1024 interlaced 10.0 ms for 10.4, 2048 51.5 for 54.3,
//                with k_fft_zy) but less exact: a CTA's FP32 sums ran over more
//                modes, the rms error of P_2 on a lattice of 512^3 objects at 1024
//                was 1.7e-6 of P_0 for 3.2e-7, at 2048 1.1e-5 for 2.3e-6.
//
// Sizes: each is an instance to compile and to measure; 320 to 800 are those with factors
// 2, 3 and 5 that the workloads and tests here use.  Others (432, 576, 720, 864, 960, 1000,
// and all with a factor 7) have no instance and go to cuFFT, as do the smaller ones but
// 128, 192 and 256 (pk_fft.cu).
//
// Only modes with m = |n|^2 < mhi enter a bin: columns l with l^2 >= mhi are
// neither transformed along y nor read, the y pass does not write rows ky with
// ky^2 + l0^2 >= mhi, and the x pass reads only tiles below mhi (21 % less
// traffic for kmax = k_N).  What they leave in the mesh is never read.
//
// All transforms are forward (e^{-2 pi i jk/n}), unnormalized, decimation in
// frequency in the radix order of radix_of; twiddles come from one table
// W_N^e (e < N) computed in FP64 on the host.
//
// The file is compiled once per group of sizes (PK_ZYX_GROUP), so that the
// groups build in parallel.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "pk_internal.h"
#include "pk_ylm.h"

namespace pk {

namespace {

// Complex sums as one packed FP32x2 instruction each.
__device__ __forceinline__ float2 c_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 c_sub(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 c_mul(float2 a, float2 b) {
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ float2 c_mi(float2 a) { return make_float2(a.y, -a.x); }   // a * (-i)

// In-register DFT of R points: v[k] <- sum_j v[j] W_R^{jk}.
//
// Constants that FP32 rounds badly carry their rest as a second term: with sin(2 pi/5)
// 2.4e-8 off, the codelets of 5 and 10 raised the mean power of a field by 1.7e-8 and
// 2.8e-8 a step, 1.9e-7 in all at 400^3, which a uniform catalog's P(k) shows once the shot
// noise is subtracted.  For the same reason 6 and 10 are taken apart into coprime
// factors, which need no twiddles.  Mean power of white noise, off by (1e-7; before,
// now, cuFFT): 320 -1.1, -1.8, -3.7; 384 -2.5, -2.0, -4.9; 400 1.9, 0.5, 1.0; 480 -0.4,
// -0.4, -0.3; 500 1.9, 0.2, 2.0; 600 1.4, 0.3, 0.0; 640 -0.8, -1.6, -2.0; 768 -3.0, -2.5,
// -3.0; 800 1.5, 0.0, -1.0; 1024 -2.6, -2.6, -4.8.  Times within 1 % (480: 2 %).
template <int R>
__device__ __forceinline__ void dft(float2 *v);

template <>
__device__ __forceinline__ void dft<2>(float2 *v) {
    const float2 a = v[0];
    v[0] = c_add(a, v[1]);
    v[1] = c_sub(a, v[1]);
}

template <>
__device__ __forceinline__ void dft<4>(float2 *v) {
    const float2 a = c_add(v[0], v[2]), b = c_sub(v[0], v[2]);
    const float2 c = c_add(v[1], v[3]), d = c_sub(v[1], v[3]);
    v[0] = c_add(a, c);
    v[2] = c_sub(a, c);
    v[1] = make_float2(b.x + d.y, b.y - d.x);                  // b -+ i d
    v[3] = make_float2(b.x - d.y, b.y + d.x);
}

template <>
__device__ __forceinline__ void dft<3>(float2 *v) {
    const float h = 0.86602540378443865f, dh = 1.55436251e-08f;  // sqrt(3) / 2
    const float2 s = c_add(v[1], v[2]), d = c_sub(v[1], v[2]);
    const float2 m = make_float2(v[0].x - 0.5f * s.x, v[0].y - 0.5f * s.y);
    v[0] = c_add(v[0], s);
    // W_3 = -1/2 - i sqrt(3)/2
    v[1] = make_float2(fmaf(h, d.y, fmaf(dh, d.y, m.x)), fmaf(-h, d.x, fmaf(-dh, d.x, m.y)));
    v[2] = make_float2(fmaf(-h, d.y, fmaf(-dh, d.y, m.x)), fmaf(h, d.x, fmaf(dh, d.x, m.y)));
}

// c1, c2 = cos(2 pi/5), cos(4 pi/5); s1, s2 the sines: outputs k and 5 - k
// share the cosine sum and take +- the sine sum.
template <>
__device__ __forceinline__ void dft<5>(float2 *v) {
    const float c1 = 0.30901699437494742f, c2 = -0.80901699437494742f;
    const float s1 = 0.95105651629515357f, s2 = 0.58778525229247313f, ds1 = -2.37172060e-08f;
    const float2 p1 = c_add(v[1], v[4]), q1 = c_sub(v[1], v[4]);
    const float2 p2 = c_add(v[2], v[3]), q2 = c_sub(v[2], v[3]);
    const float2 a = make_float2(v[0].x + c1 * p1.x + c2 * p2.x, v[0].y + c1 * p1.y + c2 * p2.y);
    const float2 b = make_float2(v[0].x + c2 * p1.x + c1 * p2.x, v[0].y + c2 * p1.y + c1 * p2.y);
    const float2 s = make_float2(fmaf(s1, q1.x, fmaf(s2, q2.x, ds1 * q1.x)), fmaf(s1, q1.y, fmaf(s2, q2.y, ds1 * q1.y)));
    const float2 t = make_float2(fmaf(-s1, q2.x, fmaf(s2, q1.x, -ds1 * q2.x)), fmaf(-s1, q2.y, fmaf(s2, q1.y, -ds1 * q2.y)));
    v[0] = c_add(v[0], c_add(p1, p2));
    v[1] = make_float2(a.x + s.y, a.y - s.x);
    v[4] = make_float2(a.x - s.y, a.y + s.x);
    v[2] = make_float2(b.x + t.y, b.y - t.x);
    v[3] = make_float2(b.x - t.y, b.y + t.x);
}

// Split into the even and odd outputs: X[2k] = DFT4(v[j] + v[j+4]),
// X[2k+1] = DFT4((v[j] - v[j+4]) W_8^j).
template <>
__device__ __forceinline__ void dft<8>(float2 *v) {
    const float h = 0.70710678118654752f;
    float2 u[4], w[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        u[j] = c_add(v[j], v[j + 4]);
        w[j] = c_sub(v[j], v[j + 4]);
    }
    w[1] = make_float2(h * (w[1].x + w[1].y), h * (w[1].y - w[1].x));    // * W_8 = (1 - i)/sqrt 2
    w[2] = c_mi(w[2]);                                                   // * W_8^2 = -i
    w[3] = make_float2(h * (w[3].y - w[3].x), -h * (w[3].x + w[3].y));   // * W_8^3 = -(1 + i)/sqrt 2
    dft<4>(u);
    dft<4>(w);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        v[2 * k] = u[k];
        v[2 * k + 1] = w[k];
    }
}

// 4 x 4: X[k + 4 q] = sum_j W_4^{jq} W_16^{jk} (DFT4 over v[j], v[j+4], v[j+8], v[j+12])[k].
template <>
__device__ __forceinline__ void dft<16>(float2 *v) {
    const float h = 0.70710678118654752f, c = 0.92387953251128676f, s = 0.38268343236508977f;
    float2 u[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
        for (int q = 0; q < 4; ++q) u[j][q] = v[j + 4 * q];
        dft<4>(u[j]);
    }
    const auto w8 = [&](float2 a) { return make_float2(h * (a.x + a.y), h * (a.y - a.x)); };      // * W_16^2
    const auto w83 = [&](float2 a) { return make_float2(h * (a.y - a.x), -h * (a.x + a.y)); };    // * W_16^6
    u[1][1] = c_mul(u[1][1], make_float2(c, -s));
    u[1][2] = w8(u[1][2]);
    u[1][3] = c_mul(u[1][3], make_float2(s, -c));
    u[2][1] = w8(u[2][1]);
    u[2][2] = c_mi(u[2][2]);
    u[2][3] = w83(u[2][3]);
    u[3][1] = c_mul(u[3][1], make_float2(s, -c));
    u[3][2] = w83(u[3][2]);
    u[3][3] = c_mul(u[3][3], make_float2(-c, s));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        float2 t[4] = {u[0][k], u[1][k], u[2][k], u[3][k]};
        dft<4>(t);
#pragma unroll
        for (int q = 0; q < 4; ++q) v[k + 4 * q] = t[q];
    }
}

// Radix 2 H with H odd by coprime factors (Good 1958): inputs n = H a + 2 b, outputs
// k = ka mod 2 = kb mod H.
template <int H>
__device__ __forceinline__ void dft_2h(float2 *v) {
    float2 u[2][H];
#pragma unroll
    for (int b = 0; b < H; ++b) {
        const float2 x = v[2 * b % (2 * H)], y = v[(H + 2 * b) % (2 * H)];
        u[0][b] = c_add(x, y);
        u[1][b] = c_sub(x, y);
    }
    dft<H>(u[0]);
    dft<H>(u[1]);
#pragma unroll
    for (int k = 0; k < 2 * H; ++k) v[k] = u[k % 2][k % H];
}

template <>
__device__ __forceinline__ void dft<6>(float2 *v) { dft_2h<3>(v); }

template <>
__device__ __forceinline__ void dft<10>(float2 *v) { dft_2h<5>(v); }

// Radix of the decimation-in-frequency step over blocks of S points: 10 and 6
// take the factors 5 and 3 out first (20: 5, then 4; 12: 4, then 3), then 8 and
// 16 so that a power of two takes the fewest steps (1024: 16, 8, 8; 2048: 16,
// 16, 8; measured against 8, 8, 4, 4 and 8, 8, 8, 4: both kernels 6 % faster).
__host__ __device__ constexpr int radix_of(int S) {
    return S <= 6 || S == 10              ? S
           : S == 480                     ? 6         // 10 first: twiddles 2.3e-8 off in the mean power, for 0.7e-8
           : S == 12                      ? 4
           : S == 20                      ? 5
           : S % 10 == 0                  ? 10
           : S % 6 == 0                   ? 6
           : S % 5 == 0                   ? 5
           : S % 3 == 0                   ? 3
           : S == 16 ? 4
           : S == 128 || S == 1024 || S == 2048 || S == 256 ? 16
                                          : 8;
}

// Radix order of the z FFTs: as radix_of, but 4 for the blocks of 32 and 8 first
// for 256 (8, 4, 8: the last step pairs its butterflies, see zrow_last).
__host__ __device__ constexpr int zradix_of(int S) { return S == 32 ? 4 : (S == 256 ? 8 : radix_of(S)); }

// Frequency at position p (< S) after all steps over a block of S points:
// a step of radix R puts output k of the butterfly at n + (S/R) k, so the
// digits of p, most significant first, are the frequency's digits from the
// least significant up.
template <int S, int MUL, bool Z = false>
__device__ __forceinline__ int dif_freq(int p) {
    if constexpr (S == 1) {
        return 0;
    } else {
        constexpr int R = Z ? zradix_of(S) : radix_of(S), Q = S / R;
        return (p / Q) * MUL + dif_freq<Q, MUL * R, Z>(p % Q);
    }
}

// Shapes per mesh size (128, 192, 256 and 512 serve the survey transforms; box
// spectra of these sizes take the packed form of pk_fft.cu).  T threads of k_fft_zy (CTAS per SM, 64 registers a
// thread), NBY columns per y tile, TX threads of the x kernels (CTASX per SM), NX
// columns per x tile.  About 12 to 16 complex values per thread.  At N = 2048
// and 1024 the x tiles take 128 KB and one CTA of 1024 threads, since their runs
// along z come from device memory (32-byte runs at 1024: 5.7 against 3.8 ms
// interlaced).  The y tiles are read from L2 in runs of 64 bytes or more: at 2048
// that takes one 768-thread CTA per SM (k_fft_zy 29.2 ms; 32.3 with 32-byte runs
// and two 512-thread CTAs, 58.9 with 16-byte runs), at 1024 two CTAs (6.06 ms; 6.55
// with 128-byte runs and one).  LAG: planes between a plane's z and y items (1024
// interlaced: 6.05, 6.06 and 6.31 ms at 4, 6 and 10 planes; 2048: 29.8 and 30.4 at
// 1 and 2; at 512, 8 planes 1060 us, 24 774, 64 858; the other sizes are set between
// those, not swept).
template <int N>
struct Shape;
template <int T_, int CTAS_, int NBY_, int TX_, int CTASX_, int NX_, int LAG_>
struct ShapeOf {
    static constexpr int T = T_, CTAS = CTAS_, NBY = NBY_, TX = TX_, CTASX = CTASX_, NX = NX_, LAG = LAG_;
};
template <> struct Shape<128> : ShapeOf<256, 4, 32, 256, 4, 16, 32> {};
template <> struct Shape<192> : ShapeOf<384, 2, 16, 384, 2, 16, 32> {};
template <> struct Shape<256> : ShapeOf<512, 2, 32, 512, 2, 16, 32> {};
template <> struct Shape<512> : ShapeOf<512, 2, 16, 512, 2, 16, 24> {};
template <> struct Shape<320> : ShapeOf<256, 4, 8, 320, 2, 16, 32> {};
template <> struct Shape<384> : ShapeOf<384, 2, 8, 384, 2, 16, 32> {};
template <> struct Shape<400> : ShapeOf<320, 3, 8, 320, 3, 8, 32> {};
template <> struct Shape<480> : ShapeOf<384, 2, 8, 384, 2, 16, 24> {};
template <> struct Shape<500> : ShapeOf<416, 2, 8, 416, 2, 8, 24> {};
template <> struct Shape<600> : ShapeOf<480, 2, 8, 480, 2, 8, 16> {};
template <> struct Shape<640> : ShapeOf<512, 2, 8, 512, 2, 8, 16> {};
template <> struct Shape<768> : ShapeOf<512, 2, 8, 512, 2, 8, 10> {};
template <> struct Shape<800> : ShapeOf<512, 2, 8, 512, 2, 8, 10> {};
template <> struct Shape<1024> : ShapeOf<512, 2, 8, 1024, 1, 16, 6> {};
template <> struct Shape<2048> : ShapeOf<768, 1, 8, 1024, 1, 8, 1> {};

template <int N>
struct Cfg : Shape<N> {
    static constexpr int M = N / 2, Nh = M + 1;
    // z rows: NT threads share NR rows of M complex (about 16 per thread)
    static constexpr int NT = M >= 1024 ? 64 : 32;
    static constexpr int NR = M > 256 ? 1 : M > 128 ? 2 : M > 64 ? 4 : 8;
    static constexpr int GROUPS = Shape<N>::T / NT;              // row groups per CTA (named barriers 1 .. GROUPS)
    static constexpr int RPI = GROUPS * NR;                      // rows per z item
    static constexpr int ZI = (N + RPI - 1) / RPI;               // z items per plane
    static_assert(NT == 32 || GROUPS <= 15, "named barriers are 1 .. 15");
};

// ---------------------------------------------------------------------------
// Column FFTs: a tile of LEN rows x NC columns in shared memory, element (r, c)
// at slot(r, c).  The first step takes its inputs from ld(r, c), the last hands
// its outputs to st(frequency, c, value); the steps in between stay in place.
// NC threads cover one row.  Slots: rows of 16 columns are conflict-free as
// they are; rows of 8 are swapped in pairs so that butterflies 8 rows apart
// (the last step) and the bin pass's runs of 4 rows reach both halves of the
// banks.  IL tiles (two meshes side by side) swap the halves of a row instead.
template <int NC, bool IL>
struct Tile {
    __device__ static __forceinline__ int slot(int r, int c) {
        if constexpr (NC == 16) {
            return r * NC + (IL ? c ^ (((r >> 2) & 1) << 3) : c);
        } else if constexpr (NC == 8) {
            if constexpr (IL) return (r ^ ((r >> 3) & 1)) * NC + (c ^ (((r >> 2) & 1) << 2));
            else return (r ^ (((r >> 2) ^ (r >> 3)) & 1)) * NC + c;
        } else {
            return r * NC + c;
        }
    }
};

template <int LEN, int NC, int T, bool IL, int S, bool FIRST, bool TOSM, typename Ld, typename St>
__device__ __forceinline__ void col_step(float2 *buf, const float2 *tw, int c, int grp, const Ld &ld, const St &st) {
    constexpr int R = radix_of(S), Q = S / R;
    constexpr int NG = T / NC;                  // thread groups (one per butterfly)
    constexpr int NBF = LEN / R;
    constexpr int PER = (NBF + NG - 1) / NG;    // butterflies per thread
    constexpr bool EVEN = NBF % NG == 0;
    using Tl = Tile<NC, IL>;
    // all of a thread's inputs loaded before the first butterfly, unless that
    // takes more than half of the 64 registers (a butterfly then goes at a time:
    // it reads and writes the same places, except in a last step to shared
    // memory, whose reordered writes come after every read)
    constexpr bool REORDER = Q == 1 && TOSM;
    constexpr bool HOLD = PER * R <= 16 || REORDER;
    constexpr int NV = HOLD ? PER : 1;
    float2 v[NV][R];
    const auto load = [&](int s) {
        const int beta = grp + NG * s;
        if (EVEN || beta < NBF) {
            const int base = (beta / Q) * S + beta % Q;
#pragma unroll
            for (int j = 0; j < R; ++j)
                v[HOLD ? s : 0][j] = FIRST ? ld(base + Q * j, c) : buf[Tl::slot(base + Q * j, c)];
        }
    };
    if constexpr (HOLD) {
#pragma unroll
        for (int s = 0; s < PER; ++s) load(s);
    }
    if constexpr (REORDER) __syncthreads();
    const auto work = [&](int s) {
        float2 *w = v[HOLD ? s : 0];
        const int beta = grp + NG * s;
        if (EVEN || beta < NBF) {
            const int n = beta % Q, base = (beta / Q) * S + n;
            dft<R>(w);
            if constexpr (Q > 1) {
                constexpr int E = LEN / S;
                float2 ww[R];
                ww[1] = tw[n * E];
                if constexpr (R == 16) {
                    ww[2] = tw[2 * n * E];
                    ww[4] = tw[4 * n * E];
                    ww[8] = tw[8 * n * E];
                    ww[3] = c_mul(ww[2], ww[1]);
#pragma unroll
                    for (int k = 5; k < 8; ++k) ww[k] = c_mul(ww[4], ww[k - 4]);
#pragma unroll
                    for (int k = 9; k < 16; ++k) ww[k] = c_mul(ww[8], ww[k - 8]);
                } else if constexpr (R == 8) {
                    ww[4] = tw[4 * n * E];
                    ww[2] = c_mul(ww[1], ww[1]);
                    ww[3] = c_mul(ww[2], ww[1]);
                    ww[5] = c_mul(ww[4], ww[1]);
                    ww[6] = c_mul(ww[4], ww[2]);
                    ww[7] = c_mul(ww[4], ww[3]);
                } else {
#pragma unroll
                    for (int k = 2; k < R; ++k) ww[k] = tw[k * n * E];
                }
#pragma unroll
                for (int k = 1; k < R; ++k) w[k] = c_mul(w[k], ww[k]);
#pragma unroll
                for (int k = 0; k < R; ++k) buf[Tl::slot(base + Q * k, c)] = w[k];
            } else {
                const int f0 = dif_freq<LEN, 1>(base);
#pragma unroll
                for (int k = 0; k < R; ++k) st(f0 + k * (LEN / R), c, w[k]);
            }
        }
    };
    if constexpr (HOLD) {
#pragma unroll
        for (int s = 0; s < PER; ++s) work(s);
    } else {
#pragma unroll 1
        for (int s = 0; s < PER; ++s) {
            load(s);
            work(s);
        }
    }
    if constexpr (Q > 1) {
        __syncthreads();
        col_step<LEN, NC, T, IL, Q, false, TOSM>(buf, tw, c, grp, ld, st);
    }
}

// ---------------------------------------------------------------------------
// z rows.  NT threads transform NR rows; position p of a row sits in slot
// p ^ L((p >> t) & 15) (the low four bits change, so the eight-byte values of a
// half-warp spread over the 16 bank pairs).  t and L per length were chosen by
// counting the wavefronts of every access of the steps below: none beyond the
// minimum at 128, 256 and 512, 12 % more at 1024, 15 % at 192, 320 and 384,
// 25-90 % at the others (a slot p ^ ((p >> 2) & 15) took 1.6 to 5 times it).
template <int M>
struct ZSlot {
    static constexpr bool POW2 = (M & (M - 1)) == 0;
    static constexpr int t = M <= 64 || M == 128 ? 3 : M == 96 ? 4 : M % 64 != 0 ? 6 : M >= 384 ? 6 : 5;
    static constexpr bool X8 = M == 96 || (M > 128 && M % 64 == 0);    // L(d) = d ^ 8 (d & 1), else d
    static constexpr int PAD = M <= 64 ? 4 : (M == 96 || M == 128 ? 8 : 0);
    static constexpr int RS = (M + 15) / 16 * 16 + PAD;                // slots per row
    __host__ __device__ static constexpr int at(int p) {
        const int d = (p >> t) & 15;
        return p ^ (X8 ? d ^ ((d & 1) << 3) : d);
    }
    // Slot of position base + off, the two without a common bit (power-of-two
    // lengths): the map is linear over bits, so the slot of base is shifted by a
    // constant and its low four bits flipped by another.
    __device__ static __forceinline__ int at(int zbase, int base, int off) {
        if constexpr (POW2) return (zbase ^ (at(off) & 15)) + (off & ~15);
        else return at(base + off);
    }
};

// Twiddles of the z FFT steps, one table per step with block size S (from M
// down): entry (k - 1) Q + n = W_S^{nk} (Q = S/R, n < Q, 1 <= k < R), so the
// lanes of a step read consecutive or equal entries.
__host__ __device__ constexpr int ztw_offset(int M, int S) {
    int off = 0;
    for (int s = M; s > S; s /= zradix_of(s)) {
        const int q = s / zradix_of(s);
        off += q > 1 ? (zradix_of(s) - 1) * q : 0;
    }
    return off;
}

__device__ __forceinline__ void fill_ztw(float2 *ztw, const float2 *__restrict__ twg, int M) {
    for (int s = M; s > 1; s /= zradix_of(s)) {
        const int R = zradix_of(s), Q = s / R, off = ztw_offset(M, s);
        if (Q == 1) continue;
        for (int e = threadIdx.x; e < (R - 1) * Q; e += blockDim.x) {
            const int k = e / Q + 1, n = e % Q;
            ztw[off + e] = twg[2 * n * k * (M / s)];     // W_N^{2nk M/S} = W_S^{nk}
        }
    }
}

// Barrier of the NT threads that share rows: a warp, or the aligned pair of
// warps `grp` on named barrier 1 + grp (0 is __syncthreads').
template <int NT>
__device__ __forceinline__ void row_sync(int grp) {
    if constexpr (NT == 32) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(NT) : "memory");
}

// Position of the block of a last step of radix R whose output k has frequency
// f0 + k M / R (the inverse of dif_freq over the steps before it).
template <int M, int S>
__device__ __forceinline__ int block_of(int f0) {
    constexpr int R = zradix_of(S), Q = S / R;
    if constexpr (Q == 1) return 0;
    else return (f0 % R) * Q + block_of<M, Q>(f0 / R);
}

template <int S>
__host__ __device__ constexpr int zlast_radix() {
    constexpr int R = zradix_of(S);
    if constexpr (S == R) return R;
    else return zlast_radix<S / R>();
}

// One step over blocks of S points (all but the last step) of the FFTs of rows
// [0, nrow) (FIRST: values from ld(row, position)).
template <int M, int NR, int NT, int S, bool FIRST, typename Ld>
__device__ __forceinline__ void zrow_step(float2 *rows, const Ld &ld, int nrow, const float2 *ztw, int lane,
                                          int grp) {
    constexpr int R = zradix_of(S), Q = S / R;
    using Zs = ZSlot<M>;
    if constexpr (Q > 1) {
        constexpr int BPR = M / R;                    // butterflies per row
        constexpr int TOT = NR * BPR;
        constexpr int PER = (TOT + NT - 1) / NT;
        constexpr int TW = ztw_offset(M, S);
        constexpr bool HOLD = Zs::POW2 && PER * R <= 16;
        constexpr int NV = HOLD ? PER : 1;
        float2 v[NV][R];
        const auto load = [&](int s) {
            const int beta = lane + NT * s;
            const int r = beta / BPR, b = beta % BPR;
            if ((TOT % NT == 0 || beta < TOT) && r < nrow) {
                const int base = (b / Q) * S + b % Q;
#pragma unroll
                for (int j = 0; j < R; ++j) {
                    if (FIRST) v[HOLD ? s : 0][j] = ld(r, base + Q * j);
                    else v[HOLD ? s : 0][j] = rows[r * Zs::RS + Zs::at(Zs::at(base), base, Q * j)];
                }
            }
        };
        const auto work = [&](int s) {
            float2 *w = v[HOLD ? s : 0];
            const int beta = lane + NT * s;
            const int r = beta / BPR, b = beta % BPR;
            if ((TOT % NT == 0 || beta < TOT) && r < nrow) {
                const int n = b % Q, base = (b / Q) * S + n;
                dft<R>(w);
                const float2 *tk = ztw + TW + n - Q;      // tk[k Q] = W_S^{nk}
                if constexpr (R == 8 || R == 16) {
                    // four loads and products instead of fifteen loads (two and
                    // seven): shared memory is the busiest pipe here
                    float2 ww[R];
                    ww[1] = tk[Q];
                    ww[2] = R == 16 ? tk[2 * Q] : c_mul(ww[1], ww[1]);
                    ww[4] = tk[4 * Q];
                    ww[3] = c_mul(ww[2], ww[1]);
#pragma unroll
                    for (int k = 5; k < 8; ++k) ww[k] = c_mul(ww[4], ww[k - 4]);
                    if constexpr (R == 16) {
                        ww[8] = tk[8 * Q];
#pragma unroll
                        for (int k = 9; k < 16; ++k) ww[k] = c_mul(ww[8], ww[k - 8]);
                    }
#pragma unroll
                    for (int k = 1; k < R; ++k) w[k] = c_mul(w[k], ww[k]);
                } else {
#pragma unroll
                    for (int k = 1; k < R; ++k) w[k] = c_mul(w[k], tk[k * Q]);
                }
#pragma unroll
                for (int k = 0; k < R; ++k) rows[r * Zs::RS + Zs::at(Zs::at(base), base, Q * k)] = w[k];
            }
        };
        if constexpr (HOLD) {
#pragma unroll
            for (int s = 0; s < PER; ++s) load(s);
#pragma unroll
            for (int s = 0; s < PER; ++s) work(s);
        } else {
#pragma unroll 1
            for (int s = 0; s < PER; ++s) {
                load(s);
                work(s);
            }
        }
        row_sync<NT>(grp);
        zrow_step<M, NR, NT, Q, false>(rows, ld, nrow, ztw, lane, grp);
    }
}

// D[l] and D[M-l] from u = C[l], v = C[M-l] and w = W_N^l: with s = u + conj v
// and q = i w (u - conj v), D[l] = (s - q) / 2 and D[M-l] = conj(s + q) / 2.
__device__ __forceinline__ void split_real(float2 u, float2 v, float2 w, float2 *dl, float2 *dm) {
    const float2 s = make_float2(0.5f * (u.x + v.x), 0.5f * (u.y - v.y));
    const float ox = u.x - v.x, oy = u.y + v.y;
    const float qx = -(w.x * oy + w.y * ox), qy = w.x * ox - w.y * oy;
    *dl = make_float2(fmaf(-0.5f, qx, s.x), fmaf(-0.5f, qy, s.y));
    *dm = make_float2(fmaf(0.5f, qx, s.x), -fmaf(0.5f, qy, s.y));
}

// The last step of the rows' FFTs, the real-input split and the store of
// D[0 .. ncol).  Of the B = M / R butterflies of a row, whose outputs are the
// frequencies f0 + B k, one thread takes f0 and B - f0 (f0 = 0 with B / 2): the
// partner M - f of each of its outputs is among them, so the transform never
// goes back to shared memory and is written straight from registers (for one k
// the lanes write neighbouring l).
template <int M, int NR, int NT>
__device__ __forceinline__ void zrow_last(const float2 *rows, int nrow, float2 *d, long long ds, int ncol,
                                          const float2 *tw, int lane) {
    constexpr int R = zlast_radix<M>(), B = M / R, GP = B / 2, TOT = NR * GP;
    using Zs = ZSlot<M>;
    static_assert(B % 2 == 0, "butterflies pair up");
#pragma unroll 1
    for (int t = lane; t < TOT; t += NT) {
        const int r = t / GP, i = t % GP;
        if (r >= nrow) continue;
        const int fb0 = i ? B - i : GP;
        float2 va[R], vb[R];
        {
            const int pa = block_of<M, M>(i), pb = block_of<M, M>(fb0), za = Zs::at(pa), zb = Zs::at(pb);
#pragma unroll
            for (int j = 0; j < R; ++j) {
                va[j] = rows[r * Zs::RS + Zs::at(za, pa, j)];
                vb[j] = rows[r * Zs::RS + Zs::at(zb, pb, j)];
            }
        }
        dft<R>(va);
        dft<R>(vb);
        float2 *row = d + r * ds;
        const auto put = [&](float2 u, float2 v, int f) {        // u = C[f], v = C[M - f]
            float2 dl, dm;
            split_real(u, v, tw[f], &dl, &dm);
            if (f < ncol) row[f] = dl;
            if (M - f < ncol) row[M - f] = dm;
        };
#pragma unroll
        for (int k = 0; k < R; ++k) put(va[k], i ? vb[R - 1 - k] : va[(R - k) % R], i + B * k);
        if (i == 0) {
#pragma unroll
            for (int k = 0; k < (R + 1) / 2; ++k) put(vb[k], vb[R - 1 - k], GP + B * k);
        }
    }
}

// Waits of y items for their plane's z items.  A CTA holds its current item and
// the ticket of its next one.  The unfinished item with the lowest ticket is
// always some running CTA's current one (were it a next one, that CTA's
// current item would have a lower ticket), and it does not wait: z items never
// do, and a y item's z items have lower tickets.  So every wait ends; the limit
// (about a second) only bounds it if that were ever wrong.
constexpr int kMaxPolls = 1 << 20;

// Y_lm(x^) along a z row as a polynomial in z: Y = (c[0] + c[1] z + .. + c[4] z^4)
// / r^l with r^2 = x^2 + y^2 + z^2; slots 0..4: l = 2, m = slot - 2, 5..13: l = 4,
// m = slot - 9 (the polynomials of ylm_slot in pk_survey.cu, r^2 put in).
__device__ __forceinline__ void ylm_row(int slot, float x, float y, float *c) {
    const float x2 = x * x, y2 = y * y, rho = x2 + y2, d = x2 - y2, xy = x * y;
    c[0] = c[1] = c[2] = c[3] = c[4] = 0.0f;
    switch (slot) {
    case 0: c[0] = (float)kYa * xy; break;
    case 1: c[1] = (float)kYa * y; break;
    case 2: c[0] = -(float)kYb * rho; c[2] = 2.0f * (float)kYb; break;
    case 3: c[1] = (float)kYa * x; break;
    case 4: c[0] = (float)kYc * d; break;
    case 5: c[0] = (float)kYd * xy * d; break;
    case 6: c[1] = (float)kYe * y * (3.0f * x2 - y2); break;
    case 7: c[0] = -(float)kYf * xy * rho; c[2] = 6.0f * (float)kYf * xy; break;
    case 8: c[1] = -3.0f * (float)kYg * y * rho; c[3] = 4.0f * (float)kYg * y; break;
    case 9: c[0] = 3.0f * (float)kYh * rho * rho; c[2] = -24.0f * (float)kYh * rho; c[4] = 8.0f * (float)kYh; break;
    case 10: c[1] = -3.0f * (float)kYg * x * rho; c[3] = 4.0f * (float)kYg * x; break;
    case 11: c[0] = -(float)kYi * d * rho; c[2] = 6.0f * (float)kYi * d; break;
    case 12: c[1] = (float)kYe * x * (x2 - 3.0f * y2); break;
    case 13: c[0] = (float)kYj * (x2 * (x2 - 3.0f * y2) - y2 * (3.0f * x2 - y2)); break;
    }
}

// sync[0]: next ticket; sync[1 + p]: z items done in plane p.  Zero at launch;
// the kernel that takes the x axis clears them again.  err: 4 if a wait gave up.
// SURVEY: plane p is x plane p / nslot of slot s0 + p % nslot (so the slots
// of a plane read their source rows from L2), whose rows are formed on the way
// in: the field D - alpha R times Y_lm(x^) of the slot (slot -1: 1).
template <int N, bool SURVEY>
__global__ void __launch_bounds__(Cfg<N>::T, Cfg<N>::CTAS)
k_fft_zy(float2 *mesh, int planes, int ncol, int mcut, const float2 *__restrict__ twg, unsigned *__restrict__ sync,
         int *__restrict__ err, SurveyRows sv) {
    using K = Cfg<N>;
    constexpr int M = K::M, Nh = K::Nh, T = K::T, NBY = K::NBY, LAG = K::LAG;
    extern __shared__ __align__(16) unsigned char smraw[];
    __shared__ unsigned s_ticket;
    float2 *tw = reinterpret_cast<float2 *>(smraw);
    float2 *ztw = tw + N;
    float2 *buf = ztw + (ztw_offset(M, 1) + 1) / 2 * 2;
    for (int e = threadIdx.x; e < N; e += T) tw[e] = twg[e];
    fill_ztw(ztw, twg, M);
    const unsigned ytiles = (unsigned)(ncol + NBY - 1) / NBY;
    const unsigned per = K::ZI + ytiles;
    const unsigned total = (unsigned)(planes + LAG) * per;
    const long long plane_c = (long long)N * Nh;
    const float alpha = SURVEY && sv.R ? (float)sv.alpha[0] : 0.0f;
    const auto plane_at = [&](int p) -> float2 * {
        if constexpr (!SURVEY) return mesh + (long long)p * plane_c;
        const int i = p / sv.nslot;
        return mesh + (long long)(p - i * sv.nslot) * sv.slot_c + (long long)i * plane_c;
    };
    unsigned next = threadIdx.x == 0 ? atomicAdd(sync, 1u) : 0u;
    for (;;) {
        __syncthreads();                        // the previous item is done with buf and s_ticket
        if (threadIdx.x == 0) s_ticket = next;
        __syncthreads();
        const unsigned t = s_ticket;
        if (t >= total) return;
        if (threadIdx.x == 0) next = atomicAdd(sync, 1u);    // in flight during this item
        const int step = (int)(t / per);
        const unsigned idx = t - (unsigned)step * per;
        if (idx < K::ZI) {
            if (step >= planes) continue;
            const int lane = threadIdx.x % K::NT, grp = threadIdx.x / K::NT;
            const int row0 = (int)idx * K::RPI + grp * K::NR;
            const int nrow = grp < K::GROUPS ? min(K::NR, N - row0) : 0;
            float2 *g = plane_at(step) + (long long)row0 * Nh;
            if (nrow > 0) {
                float2 *rows = buf + (size_t)grp * K::NR * ZSlot<M>::RS;
                if constexpr (!SURVEY) {
                    const auto ld = [&](int r, int p) { return __ldcs(g + (long long)r * Nh + p); };
                    zrow_step<M, K::NR, K::NT, M, true>(rows, ld, nrow, ztw, lane, grp);
                } else {
                    const int i = step / sv.nslot, slot = sv.s0 + step - i * sv.nslot;
                    const long long at = (long long)i * plane_c + (long long)row0 * Nh;
                    const float2 *D = reinterpret_cast<const float2 *>(sv.D) + at;
                    const float2 *Rm = sv.R ? reinterpret_cast<const float2 *>(sv.R) + at : nullptr;
                    const float x = sv.ox + (float)i * sv.H;
                    float c[K::NR][5], rho[K::NR];
#pragma unroll
                    for (int r = 0; r < K::NR; ++r) {
                        const float y = sv.oy + (float)(row0 + r) * sv.H;
                        rho[r] = x * x + y * y;
                        ylm_row(slot, x, y, c[r]);
                    }
                    const auto weight = [&](int r, int k) {       // Y_lm at z node k of the row
                        const float z = sv.oz + (float)k * sv.H, r2 = rho[r] + z * z;
                        const float ir = r2 > 0.0f ? rsqrtf(r2) : 0.0f;   // 0: the observer's node
                        // r^-4 as two factors: a node 2e-10 box edges from the observer, who
                        // sits on it but for FP32 rounding, would have an infinite one
                        const float inv = ir * ir;
                        const float y = (c[r][0] + z * (c[r][1] + z * (c[r][2] + z * (c[r][3] + z * c[r][4])))) * inv;
                        return slot >= 5 ? y * inv : y;
                    };
                    const auto ld = [&](int r, int p) {
                        float2 f = __ldcg(D + (long long)r * Nh + p);
                        if (Rm) {
                            const float2 q = __ldcg(Rm + (long long)r * Nh + p);
                            f.x -= alpha * q.x;
                            f.y -= alpha * q.y;
                        }
                        if (slot >= 0) {
                            f.x *= weight(K::NR == 1 ? 0 : r, 2 * p);
                            f.y *= weight(K::NR == 1 ? 0 : r, 2 * p + 1);
                        }
                        return f;
                    };
                    zrow_step<M, K::NR, K::NT, M, true>(rows, ld, nrow, ztw, lane, grp);
                }
                zrow_last<M, K::NR, K::NT>(rows, nrow, g, Nh, ncol, tw, lane);
            }
            __syncthreads();
            if (threadIdx.x == 0) {             // the CTA's rows, seen through the barrier, then the count
                __threadfence();
                atomicAdd(sync + 1 + step, 1u);
            }
        } else {
            const int plane = step - LAG;
            if (plane < 0 || plane >= planes) continue;
            if (threadIdx.x == 0) {
                unsigned *flag = sync + 1 + plane, done;
                int polls = 0;
                do {
                    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(done) : "l"(flag) : "memory");
                    if (done >= K::ZI) break;
                    __nanosleep(64);
                } while (++polls < kMaxPolls);
                if (done < K::ZI) atomicOr(err, 4);
            }
            __syncthreads();
            const int c0 = (int)(idx - K::ZI) * NBY;
            float2 *g = plane_at(plane) + c0;
            const int nc = ncol - c0;           // valid columns of the tile
            const auto ld = [&](int r, int c) {
                return c < nc ? __ldcg(g + (long long)r * Nh + c) : make_float2(0.0f, 0.0f);
            };
            const int l2 = c0 * c0;
            const auto st = [&](int f, int c, float2 v) {
                const int jp = f < M ? f : f - N;
                if (c < nc && jp * jp + l2 < mcut) g[(long long)f * Nh + c] = v;
            };
            col_step<N, NBY, T, false, N, true, false>(buf, tw, threadIdx.x % NBY, threadIdx.x / NBY, ld, st);
        }
    }
}

// ---------------------------------------------------------------------------
// x axis.  tiles[t] = ky index * 65536 + column block (the tiles that hold a
// mode below mcut).

// Clear the z / y pass's tickets and counters for the next compute.
__device__ __forceinline__ void clear_sync(unsigned *sync, int n) {
    if (blockIdx.x == 0 && blockIdx.y == 0)
        for (int k = threadIdx.x; k < n; k += blockDim.x) sync[k] = 0u;
}

// A value of a run along z at an x line's point: the runs of a tile are 64 or 128
// bytes, planes apart, and the tiles beside it are in flight too, so the L2 is
// told to fetch 256 bytes around.
__device__ __forceinline__ float2 load_run(const float2 *p) {
    float2 v;
    asm volatile("ld.global.L2::256B.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}

template <int N>
__global__ void __launch_bounds__(Cfg<N>::TX, Cfg<N>::CTASX)
k_fft_x(float2 *__restrict__ mesh, long long mesh_c, int ncol, int mcut, const int *__restrict__ tiles,
        const float2 *__restrict__ twg, unsigned *__restrict__ sync, int nsync) {
    using K = Cfg<N>;
    constexpr int M = K::M, Nh = K::Nh, NX = K::NX;
    extern __shared__ __align__(16) unsigned char smraw[];
    float2 *tw = reinterpret_cast<float2 *>(smraw);
    float2 *buf = tw + N;
    for (int e = threadIdx.x; e < N; e += K::TX) tw[e] = twg[e];
    clear_sync(sync, nsync);
    __syncthreads();
    const int tile = tiles[blockIdx.x];
    const int j = tile >> 16, c0 = (tile & 0xffff) * NX;
    const int jp = j < M ? j : j - N, nc = ncol - c0, r2 = jp * jp + c0 * c0;
    float2 *g = mesh + (long long)blockIdx.y * mesh_c + (long long)j * Nh + c0;
    const long long ps = (long long)N * Nh;
    const auto ld = [&](int r, int c) { return c < nc ? load_run(g + r * ps + c) : make_float2(0.0f, 0.0f); };
    const auto st = [&](int f, int c, float2 v) {
        const int ip = f < M ? f : f - N;
        if (c < nc && ip * ip + r2 < mcut) g[f * ps + c] = v;
    };
    col_step<N, NX, K::TX, false, N, true, false>(buf, tw, threadIdx.x % NX, threadIdx.x / NX, ld, st);
}

// ---------------------------------------------------------------- host --

template <int N>
constexpr size_t zy_smem() {
    using K = Cfg<N>;
    const size_t z = (size_t)K::RPI * ZSlot<K::M>::RS, y = (size_t)N * K::NBY;
    return sizeof(float2) * (N + (ztw_offset(K::M, 1) + 1) / 2 * 2 + (z > y ? z : y));
}

template <typename F>
cudaError_t allow_smem(F kern, size_t bytes) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

template <int N, bool SURVEY>
cudaError_t zy_inst(float2 *mesh, int planes, int ncol, int mcut, const float2 *tw, unsigned *sync, int *err, int nsm,
                    const SurveyRows &sv, cudaStream_t st) {
    using K = Cfg<N>;
    constexpr size_t smem = zy_smem<N>();
    cudaError_t e = allow_smem(k_fft_zy<N, SURVEY>, smem);
    if (e != cudaSuccess) return e;
    const long long items = (long long)(planes + K::LAG) * (K::ZI + (ncol + K::NBY - 1) / K::NBY);
    if (items > 0x7fffffffLL) return cudaErrorInvalidValue;
    const unsigned grid = (unsigned)std::min<long long>((long long)nsm * K::CTAS, items);
    k_fft_zy<N, SURVEY><<<grid, K::T, smem, st>>>(mesh, planes, ncol, mcut, tw, sync, err, sv);
    return cudaGetLastError();
}

template <int N>
cudaError_t x_inst(float2 *mesh, int nmesh, long long mesh_c, int ncol, int mcut, const int *tiles, int ntiles,
                   const float2 *tw, unsigned *sync, int nsync, cudaStream_t st) {
    using K = Cfg<N>;
    const size_t smem = sizeof(float2) * (N + (size_t)N * K::NX);
    cudaError_t e = allow_smem(k_fft_x<N>, smem);
    if (e != cudaSuccess) return e;
    k_fft_x<N><<<dim3(ntiles, nmesh), K::TX, smem, st>>>(mesh, mesh_c, ncol, mcut, tiles, tw, sync, nsync);
    return cudaGetLastError();
}

// One size's launchers.
template <int N>
struct OpsOf final : ZyxOps {
    int tile_columns() const override { return Cfg<N>::NX; }
    cudaError_t zy(void *mesh, int planes, int ncol, int mcut, const void *tw, unsigned *sync, int *err, int nsm,
                   cudaStream_t st) const override {
        return zy_inst<N, false>(reinterpret_cast<float2 *>(mesh), planes, ncol, mcut,
                                 reinterpret_cast<const float2 *>(tw), sync, err, nsm, SurveyRows{}, st);
    }
    cudaError_t zy_survey(void *mesh, int nx, const SurveyRows &sv, int ncol, int mcut, const void *tw, unsigned *sync,
                          int *err, int nsm, cudaStream_t st) const override {
        return zy_inst<N, true>(reinterpret_cast<float2 *>(mesh), nx * sv.nslot, ncol, mcut,
                                reinterpret_cast<const float2 *>(tw), sync, err, nsm, sv, st);
    }
    bool plan_default() const override { return N != 128 && N != 192 && N != 256 && N != 512; }
    cudaError_t x(void *mesh, int nmesh, long long mesh_c, int ncol, int mcut, const int *tiles, int ntiles,
                  const void *tw, unsigned *sync, int nsync, cudaStream_t st) const override {
        return x_inst<N>(reinterpret_cast<float2 *>(mesh), nmesh, mesh_c, ncol, mcut, tiles, ntiles,
                         reinterpret_cast<const float2 *>(tw), sync, nsync, st);
    }
};

template <int N>
const ZyxOps *ops_of() {
    static const OpsOf<N> ops;
    return &ops;
}

}  // namespace

#ifndef PK_ZYX_GROUP
#error "compile with -DPK_ZYX_GROUP=0 .. 2"
#endif
#define PK_ZYX_NAME2(g) zyx_ops_group##g
#define PK_ZYX_NAME(g) PK_ZYX_NAME2(g)

const ZyxOps *PK_ZYX_NAME(PK_ZYX_GROUP)(int N) {
    switch (N) {
#if PK_ZYX_GROUP == 0
    case 320: return ops_of<320>();
    case 384: return ops_of<384>();
    case 400: return ops_of<400>();
    case 480: return ops_of<480>();
    case 500: return ops_of<500>();
    case 600: return ops_of<600>();
    case 640: return ops_of<640>();
    case 768: return ops_of<768>();
    case 800: return ops_of<800>();
#elif PK_ZYX_GROUP == 1
    case 128: return ops_of<128>();
    case 192: return ops_of<192>();
    case 256: return ops_of<256>();
    case 512: return ops_of<512>();
    case 1024: return ops_of<1024>();
#else
    case 2048: return ops_of<2048>();
#endif
    default: return nullptr;
    }
}

}  // namespace pk
