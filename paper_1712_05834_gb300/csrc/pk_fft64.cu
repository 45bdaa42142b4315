// pk_fft64.cu -- the library's own 3D r2c transform of FP64 meshes (the
// transform of Sec. 3.3.1 in the double precision form).  In place, in the
// padded r2c layout (rows of N/2 + 1 complex): z rows, then y and x columns
// (k_fft64_z, k_fft64_col).
//
// What bounds it: the FP64 pipe.  A GB300 issues two FP64 operations per SM and
// clock (some 0.59 T a second), so a 256^3 mesh needs 0.9 ms for the 5.2e8
// operations below while its bytes take 0.12 ms.  Everything else is therefore
// laid out for few FP64 operations, not for bytes:
//   * Large radices (16 x 16 at 256: one twiddle multiply between the steps),
//     butterflies written for FMA (DFT_16 in 144 operations: sqrt(1/2) and
//     cos(pi/8) are factored out of the twiddled inputs and come back in the
//     FMAs of the last sums), and twiddle-free prime-factor codelets for 6, 10,
//     12, 14 and 15 (Good 1958).
//   * Two real rows as one complex line: their spectra come apart by two
//     additions per output (the factor 1/2 rides on the first twiddles).
//   * Lines that hold no binned mode are left out along y and x: columns l with
//     l^2 >= mhi, and lines (ky, l) with ky^2 + l^2 >= mhi (21 % of the x lines
//     for kmax = k_N).  What they leave in the mesh is never read.
// Index arithmetic is free beside that (64 issue slots per FP64 instruction of
// a warp), so one kernel takes the radix sequence at run time and serves every
// even N from 32 to 2048 with prime factors up to 7.
//
// Two meshes, us, cuFFT D2Z and these kernels (84 % of the FP64 pipe's rate while they
// run): 64^3 57 and 53, 100^3 244 and 192, 128^3 432 and 266, 200^3 2496 and 1401, 256^3
// 3461 and 2040, 320^3 8438 and 5157, 512^3 30980 and 19453, 640^3 89049 and 41294; no
// size tried was slower, so every size they can take does.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "pk_internal.h"

namespace pk {

namespace {

constexpr int kT64 = 128;            // threads per CTA
constexpr int kMaxN64 = 2048, kMinN64 = 32;

__host__ __device__ __forceinline__ double2 z_add(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ double2 z_sub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
// a + s b, a - s b with real s, and with i s
__host__ __device__ __forceinline__ double2 z_fma(double2 a, double s, double2 b) {
    return make_double2(fma(s, b.x, a.x), fma(s, b.y, a.y));
}
__host__ __device__ __forceinline__ double2 z_mul(double2 a, double2 b) {
    return make_double2(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}

// In-register DFT of R points: v[k] <- sum_j v[j] W_R^{jk}, W_R = e^{-2 pi i / R}.
template <int R>
struct Dft {
    // R = A B with A, B coprime: inputs n = B a + A b, outputs k = ka mod A = kb mod B
    static constexpr int A = R == 6 || R == 10 || R == 14 ? 2 : R == 12 || R == 15 ? 3 : 1;
    static constexpr int B = R / A;
    __host__ __device__ static constexpr int crt(int a, int b) {
        int k = a;
        while (k % B != b) k += A;
        return k;
    }
    __host__ __device__ static __forceinline__ void run(double2 *v) {
        static_assert(A > 1, "no codelet");
        double2 u[A][B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            double2 t[A];
#pragma unroll
            for (int a = 0; a < A; ++a) t[a] = v[(B * a + A * b) % R];
            Dft<A>::run(t);
#pragma unroll
            for (int a = 0; a < A; ++a) u[a][b] = t[a];
        }
#pragma unroll
        for (int a = 0; a < A; ++a) {
            Dft<B>::run(u[a]);
#pragma unroll
            for (int b = 0; b < B; ++b) v[crt(a, b)] = u[a][b];
        }
    }
};

template <>
struct Dft<2> {
    __host__ __device__ static __forceinline__ void run(double2 *v) {
        const double2 a = v[0];
        v[0] = z_add(a, v[1]);
        v[1] = z_sub(a, v[1]);
    }
};

template <>
struct Dft<3> {
    __host__ __device__ static __forceinline__ void run(double2 *v) {
        const double h = 0.86602540378443864676;               // sqrt(3) / 2
        const double2 s = z_add(v[1], v[2]), d = z_sub(v[1], v[2]);
        const double2 m = z_fma(v[0], -0.5, s);
        v[0] = z_add(v[0], s);
        v[1] = make_double2(fma(h, d.y, m.x), fma(-h, d.x, m.y));
        v[2] = make_double2(fma(-h, d.y, m.x), fma(h, d.x, m.y));
    }
};

template <>
struct Dft<4> {
    __host__ __device__ static __forceinline__ void run(double2 *v) {
        const double2 a = z_add(v[0], v[2]), b = z_sub(v[0], v[2]);
        const double2 c = z_add(v[1], v[3]), d = z_sub(v[1], v[3]);
        v[0] = z_add(a, c);
        v[2] = z_sub(a, c);
        v[1] = make_double2(b.x + d.y, b.y - d.x);             // b -+ i d
        v[3] = make_double2(b.x - d.y, b.y + d.x);
    }
};

// Odd R: outputs k and R - k share the cosine sum of v[j] + v[R-j] and take +-
// the sine sum of v[j] - v[R-j].  cs, sn: cos and sin of 2 pi j / R, j <= R/2.
template <int R>
__host__ __device__ __forceinline__ void dft_odd(double2 *v, const double *cs, const double *sn) {
    constexpr int H = R / 2;
    double2 p[H + 1], q[H + 1];
    double2 s0 = v[0];
#pragma unroll
    for (int j = 1; j <= H; ++j) {
        p[j] = z_add(v[j], v[R - j]);
        q[j] = z_sub(v[j], v[R - j]);
        s0 = z_add(s0, p[j]);
    }
#pragma unroll
    for (int k = 1; k <= H; ++k) {
        double2 a = v[0], b = make_double2(0.0, 0.0);
#pragma unroll
        for (int j = 1; j <= H; ++j) {
            const int e = j * k % R;
            const double c = cs[e <= H ? e : R - e], s = e <= H ? sn[e] : -sn[R - e];
            a = z_fma(a, c, p[j]);
            b = j == 1 ? make_double2(s * q[1].x, s * q[1].y) : z_fma(b, s, q[j]);
        }
        v[k] = make_double2(a.x + b.y, a.y - b.x);
        v[R - k] = make_double2(a.x - b.y, a.y + b.x);
    }
    v[0] = s0;
}

template <>
struct Dft<5> {
    __host__ __device__ static __forceinline__ void run(double2 *v) {
        const double cs[3] = {1.0, 0.30901699437494742410, -0.80901699437494742410};
        const double sn[3] = {0.0, 0.95105651629515357212, 0.58778525229247312917};
        dft_odd<5>(v, cs, sn);
    }
};

template <>
struct Dft<7> {
    __host__ __device__ static __forceinline__ void run(double2 *v) {
        const double cs[4] = {1.0, 0.62348980185873353053, -0.22252093395631440429, -0.90096886790241912624};
        const double sn[4] = {0.0, 0.78183148246802980871, 0.97492791218182360702, 0.43388373911755812048};
        dft_odd<7>(v, cs, sn);
    }
};

// Even outputs: DFT_4 of v[j] + v[j+4]; odd ones: DFT_4 of (v[j] - v[j+4]) W_8^j,
// with sqrt(1/2) of W_8 and W_8^3 taken into the last sums.
template <>
struct Dft<8> {
    __host__ __device__ static __forceinline__ void run(double2 *v) {
        const double h = 0.70710678118654752440;
        double2 u[4], w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            u[j] = z_add(v[j], v[j + 4]);
            w[j] = z_sub(v[j], v[j + 4]);
        }
        Dft<4>::run(u);
        const double2 p = make_double2(w[1].x + w[1].y, w[1].y - w[1].x);           // W_8 w1 / h
        const double2 q = make_double2(w[3].y - w[3].x, -(w[3].x + w[3].y));        // W_8^3 w3 / h
        const double2 e = z_add(p, q), f = z_sub(p, q);
        const double2 a = make_double2(w[0].x + w[2].y, w[0].y - w[2].x);           // w0 - i w2
        const double2 b = make_double2(w[0].x - w[2].y, w[0].y + w[2].x);
        v[0] = u[0], v[2] = u[1], v[4] = u[2], v[6] = u[3];
        v[1] = z_fma(a, h, e);
        v[5] = z_fma(a, -h, e);
        v[3] = make_double2(fma(h, f.y, b.x), fma(-h, f.x, b.y));
        v[7] = make_double2(fma(-h, f.y, b.x), fma(h, f.x, b.y));
    }
};

// 4 x 4: X[k + 4 q] = sum_j W_4^{jq} W_16^{jk} u[j][k], u[j] = DFT_4 of v[j + 4 m].
// With c = cos(pi/8), t = tan(pi/8): W_16 = c (1 - i t), W_16^3 = c (t - i),
// W_16^9 = -c (1 - i t); their c and the h of W_8 are applied in the last sums.
template <>
struct Dft<16> {
    __host__ __device__ static __forceinline__ void last(double2 *v, int k, double2 a, double2 b, double s, double2 e,
                                                          double2 f) {
        v[k] = z_fma(a, s, e);
        v[k + 8] = z_fma(a, -s, e);
        v[k + 4] = make_double2(fma(s, f.y, b.x), fma(-s, f.x, b.y));
        v[k + 12] = make_double2(fma(-s, f.y, b.x), fma(s, f.x, b.y));
    }
    __host__ __device__ static __forceinline__ void run(double2 *v) {
        const double h = 0.70710678118654752440, c = 0.92387953251128675613, t = 0.41421356237309504880;
        double2 u[4][4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
#pragma unroll
            for (int m = 0; m < 4; ++m) u[j][m] = v[j + 4 * m];
            Dft<4>::run(u[j]);
        }
        {
            double2 x[4] = {u[0][0], u[1][0], u[2][0], u[3][0]};
            Dft<4>::run(x);
            v[0] = x[0], v[4] = x[1], v[8] = x[2], v[12] = x[3];
        }
        {   // k = 1: W_16 u1, W_8 u2, W_16^3 u3
            const double2 x1 = u[1][1], x2 = u[2][1], x3 = u[3][1];
            const double2 p = make_double2(fma(t, x1.y, x1.x), fma(-t, x1.x, x1.y));
            const double2 q = make_double2(fma(t, x3.x, x3.y), fma(t, x3.y, -x3.x));
            const double2 r = make_double2(x2.x + x2.y, x2.y - x2.x);
            last(v, 1, z_fma(u[0][1], h, r), z_fma(u[0][1], -h, r), c, z_add(p, q), z_sub(p, q));
        }
        {   // k = 2: W_8 u1, -i u2, W_8^3 u3
            const double2 x1 = u[1][2], x2 = u[2][2], x3 = u[3][2], x0 = u[0][2];
            const double2 p = make_double2(x1.x + x1.y, x1.y - x1.x);
            const double2 q = make_double2(x3.y - x3.x, -(x3.x + x3.y));
            last(v, 2, make_double2(x0.x + x2.y, x0.y - x2.x), make_double2(x0.x - x2.y, x0.y + x2.x), h, z_add(p, q),
                 z_sub(p, q));
        }
        {   // k = 3: W_16^3 u1, W_8^3 u2, W_16^9 u3
            const double2 x1 = u[1][3], x2 = u[2][3], x3 = u[3][3];
            const double2 p = make_double2(fma(t, x1.x, x1.y), fma(t, x1.y, -x1.x));
            const double2 q = make_double2(fma(t, x3.y, x3.x), fma(-t, x3.x, x3.y));   // -W_16^9 u3 / c
            const double2 r = make_double2(x2.y - x2.x, -(x2.x + x2.y));
            last(v, 3, z_fma(u[0][3], h, r), z_fma(u[0][3], -h, r), c, z_sub(p, q), z_add(p, q));
        }
    }
};

// One decimation-in-frequency step over the tile's lines (element (p, c) at
// p * pitch + c): butterflies of R elements S / R apart in blocks of S, each in
// its own places.  half: the outputs are scaled by 1/2 (tw holds W_N^e, e < N,
// then the same halved).
template <int R>
__device__ __forceinline__ void step64(double2 *buf, int pitch, int lc, int N, int S, const double2 *__restrict__ tw,
                                       bool half) {
    const int Q = S / R, nt = (N / R) << lc, stride = N / S;
    if (half) tw += N;
    for (int t = threadIdx.x; t < nt; t += kT64) {
        const int beta = t >> lc, blk = beta / Q, n = beta - blk * Q;
        double2 *b = buf + (blk * S + n) * pitch + (t & ((1 << lc) - 1));
        double2 v[R];
#pragma unroll
        for (int j = 0; j < R; ++j) v[j] = b[Q * j * pitch];
        Dft<R>::run(v);
        if (Q > 1) {
            const int e = n * stride;
#pragma unroll
            for (int k = 1; k < R; ++k) v[k] = z_mul(v[k], __ldg(tw + e * k));
            if (half) v[0] = make_double2(0.5 * v[0].x, 0.5 * v[0].y);
        }
#pragma unroll
        for (int k = 0; k < R; ++k) b[Q * k * pitch] = v[k];
    }
}

__device__ __forceinline__ void steps64(double2 *buf, int pitch, int lc, const Fft64 &f, bool half) {
    int S = f.N;
    for (int s = 0; s < f.nsteps; ++s) {
        const int R = f.radix[s];
        switch (R) {
            case 2: step64<2>(buf, pitch, lc, f.N, S, f.tw, half); break;
            case 3: step64<3>(buf, pitch, lc, f.N, S, f.tw, half); break;
            case 4: step64<4>(buf, pitch, lc, f.N, S, f.tw, half); break;
            case 5: step64<5>(buf, pitch, lc, f.N, S, f.tw, half); break;
            case 6: step64<6>(buf, pitch, lc, f.N, S, f.tw, half); break;
            case 7: step64<7>(buf, pitch, lc, f.N, S, f.tw, half); break;
            case 8: step64<8>(buf, pitch, lc, f.N, S, f.tw, half); break;
            case 10: step64<10>(buf, pitch, lc, f.N, S, f.tw, half); break;
            case 12: step64<12>(buf, pitch, lc, f.N, S, f.tw, half); break;
            case 14: step64<14>(buf, pitch, lc, f.N, S, f.tw, half); break;
            case 15: step64<15>(buf, pitch, lc, f.N, S, f.tw, half); break;
            default: step64<16>(buf, pitch, lc, f.N, S, f.tw, half); break;
        }
        S /= R;
        half = false;
        __syncthreads();
    }
}

// z: 2 << lc rows per CTA, two rows to a line (rows r and r + 1 of a mesh as the
// real and imaginary parts); columns l < ncol of their spectra are written.
__global__ void __launch_bounds__(kT64, 4)
k_fft64_z(double *__restrict__ mesh, long long mesh_reals, int blocks, int ncol, Fft64 f) {
    extern __shared__ __align__(16) double2 buf64[];
    const int N = f.N, lc = f.lc, pitch = (1 << lc) + 1, Nh = N / 2 + 1;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rows = min(2 << lc, N * N - (int)(blockIdx.x % blocks) * (2 << lc));       // even
    double2 *base = reinterpret_cast<double2 *>(mesh + (blockIdx.x / blocks) * mesh_reals) +
                    (long long)(blockIdx.x % blocks) * (2 << lc) * Nh;
    double *bd = reinterpret_cast<double *>(buf64);
    for (int r = warp; r < 2 << lc; r += kT64 / 32)
        for (int i = lane; i < N / 2; i += 32) {
            const double2 d = r < rows ? base[(long long)r * Nh + i] : make_double2(0.0, 0.0);
            double *p = bd + 2 * (2 * i * pitch + (r >> 1)) + (r & 1);
            p[0] = d.x;
            p[2 * pitch] = d.y;
        }
    __syncthreads();
    steps64(buf64, pitch, lc, f, true);
    for (int c = warp; c < rows >> 1; c += kT64 / 32) {
        double2 *g = base + (long long)(2 * c) * Nh;
        for (int k = lane; k < ncol; k += 32) {
            const double2 a = buf64[f.pos[k] * pitch + c], b = buf64[f.pos[k ? N - k : 0] * pitch + c];
            g[k] = make_double2(a.x + b.x, a.y - b.y);
            g[Nh + k] = make_double2(a.y + b.y, b.x - a.x);
        }
    }
}

// y (X = false): lines (x, l) over rows ky of stride Nh; x (X = true): lines
// (ky, l) over x of stride N Nh, left out where no binned mode lies on them.
// One CTA per tile of 1 << lc columns l.
template <bool X>
__global__ void __launch_bounds__(kT64, 4)
k_fft64_col(double *__restrict__ mesh, long long mesh_reals, int ncol, int mhi, Fft64 f) {
    extern __shared__ __align__(16) double2 buf64[];
    const int N = f.N, lc = f.lc, NC = 1 << lc, Nh = N / 2 + 1, tiles = (ncol + NC - 1) >> lc;
    const int tile = blockIdx.x % tiles, rest = blockIdx.x / tiles, o = rest % N, l0 = tile << lc;
    if (X) {
        const int op = o <= N / 2 ? o : N - o;
        if (op * op + l0 * l0 >= mhi) return;
    }
    const long long stride = X ? (long long)N * Nh : Nh;
    double2 *g = reinterpret_cast<double2 *>(mesh + (rest / N) * mesh_reals) + (long long)o * (X ? Nh : N * Nh) + l0;
    const int nc = min(NC, ncol - l0);
    for (int t = threadIdx.x; t < N << lc; t += kT64) {
        const int c = t & (NC - 1);
        if (c < nc) {
            asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                         :: "r"((unsigned)__cvta_generic_to_shared(buf64 + t)), "l"(g + (t >> lc) * stride + c)
                         : "memory");
        } else {
            buf64[t] = make_double2(0.0, 0.0);
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    steps64(buf64, NC, lc, f, false);
    for (int t = threadIdx.x; t < N << lc; t += kT64) {
        const int c = t & (NC - 1);
        if (c < nc) g[(t >> lc) * stride + c] = buf64[(f.pos[t >> lc] << lc) + c];
    }
}

// FP64 operations per point of a step: the codelet, and the twiddles after it.
double step_cost(int R, bool last) {
    const double dft = R == 2    ? 2.0
                       : R == 3  ? 4.0
                       : R == 4  ? 4.0
                       : R == 5  ? 7.2
                       : R == 6  ? 6.0
                       : R == 7  ? 9.4
                       : R == 8  ? 6.5
                       : R == 10 ? 9.2
                       : R == 12 ? 8.0
                       : R == 14 ? 11.4
                       : R == 15 ? 11.2
                                 : 9.0;
    return dft + (last ? 0.0 : 4.0 * (R - 1) / R);
}

// Cheapest sequence of radices (not increasing) with product n.
double cheapest(int n, int top, std::vector<int> &seq) {
    if (n == 1) return 0.0;
    double best = 1e30;
    for (int R : {16, 15, 14, 12, 10, 8, 7, 6, 5, 4, 3, 2}) {
        if (R > top || n % R) continue;
        std::vector<int> rest;
        const double c = step_cost(R, n == R) + cheapest(n / R, R, rest);
        if (c < best) {
            best = c;
            seq.assign(1, R);
            seq.insert(seq.end(), rest.begin(), rest.end());
        }
    }
    return best;
}

size_t smem64(const Fft64 &f) { return sizeof(double2) * (size_t)f.N * ((1 << f.lc) + 1); }

}  // namespace

bool fft64_plan(int N, Fft64 *f) {
    if (N < kMinN64 || N > kMaxN64 || N % 2) return false;
    std::vector<int> seq;
    if (cheapest(N, 16, seq) >= 1e30 || seq.size() < 2 || seq.size() > sizeof(f->radix)) return false;
    f->N = N;
    f->nsteps = (int)seq.size();
    for (size_t i = 0; i < seq.size(); ++i) f->radix[i] = (unsigned char)seq[i];
    f->lc = N <= 512 ? 3 : 2;       // 8 columns (128-byte runs) while four CTAs share an SM's memory at 320 and below
    f->tw = nullptr;
    f->pos = nullptr;
    return true;
}

// The frequency at position p: each step of radix R moved output k of a block
// of S to its sub-block k, so p's digits, most significant first, are the
// frequency's from the least significant up.
void fft64_tables(const Fft64 &f, double *tw, unsigned short *pos) {
    const long double pi = 3.14159265358979323846264338327950288L;
    for (int e = 0; e < f.N; ++e) {
        const long double a = 2.0L * pi * e / f.N;
        const double c = (double)cosl(a), s = 4 * e == f.N ? -1.0 : 2 * e == f.N ? 0.0 : -(double)sinl(a);
        tw[2 * e] = 4 * e == f.N || 4 * e == 3 * f.N ? 0.0 : c;
        tw[2 * e + 1] = 4 * e == 3 * f.N ? 1.0 : s;
        tw[2 * (f.N + e)] = 0.5 * tw[2 * e];
        tw[2 * (f.N + e) + 1] = 0.5 * tw[2 * e + 1];
    }
    for (int p = 0; p < f.N; ++p) {
        int S = f.N, q = p, mul = 1, freq = 0;
        for (int s = 0; s < f.nsteps; ++s) {
            const int Q = S / f.radix[s];
            freq += q / Q * mul;
            q %= Q;
            mul *= f.radix[s];
            S = Q;
        }
        pos[freq] = (unsigned short)p;
    }
}

cudaError_t launch_fft64(double *mesh, int nmesh, long long mesh_reals, const Fft64 &f, int mhi, cudaStream_t st) {
    const int N = f.N, Nh = N / 2 + 1, NC = 1 << f.lc;
    int ncol = Nh;
    while (ncol > 1 && (long long)(ncol - 1) * (ncol - 1) >= mhi) --ncol;
    const size_t smem = smem64(f);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_fft64_z, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_fft64_col<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_fft64_col<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const long long zb = ((long long)N * N + 2 * NC - 1) / (2 * NC), cb = (long long)N * ((ncol + NC - 1) / NC);
    const long long most = 0x7fffffff / std::max(zb, cb);        // meshes per launch
    for (long long at = 0; at < nmesh; at += most) {
        const long long m = std::min<long long>(most, nmesh - at);
        double *d = mesh + at * mesh_reals;
        k_fft64_z<<<(unsigned)(zb * m), kT64, smem, st>>>(d, mesh_reals, (int)zb, ncol, f);
        k_fft64_col<false><<<(unsigned)(cb * m), kT64, (size_t)N * NC * 16, st>>>(d, mesh_reals, ncol, mhi, f);
        k_fft64_col<true><<<(unsigned)(cb * m), kT64, (size_t)N * NC * 16, st>>>(d, mesh_reals, ncol, mhi, f);
    }
    return cudaGetLastError();
}

}  // namespace pk
