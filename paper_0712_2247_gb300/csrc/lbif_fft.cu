// Attractive mean-field tail through the convolution theorem.
//
// The tail force of a node (Sec. Conclusions: a mean-field attraction added
// to the hard-sphere force; Lennard-Jones form with the Barker-Henderson
// split, cut at rcut sigma) is F_att(r)/n0 = n0 m(r) T(r) with m = n/n0 (zero
// outside the fluid) and T(r) = sum_d K(d) m(r + d), K(d) = phi'(|d|) d/|d|
// over sigma <= |d| <= rcut sigma: a correlation of m with a fixed, odd,
// vector kernel. Split m = f + dn with f = 1 on fluid planes and 0 outside:
// the part of f is x,y-uniform, has a z component only,
//   w(z) = sum_dz kappa(dz) f(z + dz),  kappa(dz) = sum_{dx,dy} K_z(dx, dy, dz),
// and is tabulated in double once (it carries the wall attraction; the odd
// kernel cancels it exactly in a periodic box). The small part dn is done in
// the x-y Fourier modes, where the correlation is diagonal; along z it stays
// a short direct sum (walls need no padding):
//   M(k, z)  = FFT_xy[dn(., ., z) f(z)](k)
//   T^(k, z) = sum_dz conj(FFT_xy[K(., ., dz)](k)) M(k, z + dz)
//   T(r)     = IFFT_xy[T^](r) / (nx ny) + (0, 0, w(z))
// The fields are real, so two planes share a complex transform: the forward
// one takes P_j = m(2j) + i m(2j+1) (m = dn f), whose spectrum gives both
// planes' as M(k, 2j) = (P(k) + conj P(-k)) / 2, M(k, 2j+1) = (P(k) -
// conj P(-k)) / 2i; the inverse ones take T_x + i T_y of each plane and
// T_z(2j) + i T_z(2j+1) of each pair. The kernel's transform is computed once
// per handle with the same FFT kernels. The packing of the density rides on
// the first x pass and the product n0 m T on the last one. Cost per step:
// about four passes over a complex field of nx ny nz, instead of ~2 * 10^4
// neighbour reads per node.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <vector>

#include "lbif_internal.h"

namespace lbif {
namespace {

constexpr int FFT_THREADS = 256;
// lines x line length held by one CTA: 4096, or 1024 where those would be fewer
// than two CTAs per SM (the tail of 32 x 32 x 128 89 -> 45 us, of 64 x 128 x 100
// 101 -> 62 us)
constexpr int FFT_GL = 4096, FFT_GL_SMALL = 1024;

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b)
{
    return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// -i a
__device__ __forceinline__ float2 cmi(float2 a) { return make_float2(a.y, -a.x); }

__device__ __forceinline__ int padded(const Geom& g, int x, int y, int z)
{
    return ((z + g.hw) * g.py + (y + g.hw)) * g.px + (x + g.hw);
}

// Batched Stockham FFT (decimation in frequency, natural order in and out)
// of lines of length L = 2^logL <= 1024 held in shared memory, GL / L
// lines per CTA. A stage of radix r at stride st (the product of the radices
// before it) maps x_j = X[q + st (p + j M)], M = L / (r st), to
//   Y[q + st (r p + k)] = (sum_j x_j e^{-2 pi i j k / r}) e^{-2 pi i p k st / L};
// radix-4 stages, preceded by one radix-2 stage when logL is odd.
// Along x: line l holds elements l L .. l L + L - 1. Along y: line l = z nx + x
// holds elements z nx L + x + i nx (consecutive lines are consecutive x, so
// the loads and stores of a CTA are row segments of GL / L nodes).
// tw[j] = exp(-2 pi i j / L) for j < L/2 (copied to shared memory, extended
// by tw[j + L/2] = -tw[j]); inverse = 1 conjugates them (unnormalised).
// Fused ends of the x passes (lines l = j ny + y of a plane-pair field):
// IN reads m(x, y, 2j) + i m(x, y, 2j+1) from the padded density instead of
// `data`; OUT writes Ft = n0 m T of both planes (T_x, T_y from O1, T_z the
// real / imaginary part of the transformed pair) instead of `data`.
struct FftEnds {
    Params P;
    const float* dn;
    const float2* O1;
    const float* w;
    float4* Ft;
};

__device__ __forceinline__ float fluid_dn(const Params& P, const float* dn, int x, int y, int z)
{
    return z < P.g.nz && P.zslit[z] >= 0 ? dn[padded(P.g, x, y, z)] : 0.f;
}

// What the outputs of plane z share. Every load is unconditional (planes past
// the end read the last one) and read-only, so that a thread's outputs wait on
// memory together; only the store depends on the plane. (With a chain of
// dependent loads behind a test per output, the last pass took 51 us where the
// same transform without it takes 15; now 26 us, at 256 x 256 x 64.)
struct TailPlane {
    float rho, w;
    bool on;
    int z;
};
__device__ __forceinline__ TailPlane tail_plane(const FftEnds& e, int z)
{
    TailPlane t;
    t.z = min(z, e.P.g.nz - 1);
    const int s = __ldg(e.P.zslit + t.z), sc = max(s, 0);
    t.rho = __ldg(&e.P.sl[sc].rho0);
    t.w = __ldg(e.w + t.z);
    t.on = z < e.P.g.nz && s >= 0 && !__ldg(e.P.done + sc);
    return t;
}
__device__ __forceinline__ void tail_out(const FftEnds& e, const TailPlane& t, int x, int y, float tz)
{
    const Geom& g = e.P.g;
    const float inv = 1.f / ((float)g.nx * (float)g.ny);
    const long long idx = ((long long)t.z * g.ny + y) * g.nx + x;
    const float pre = t.rho * (1.f + __ldg(e.dn + padded(g, x, y, t.z)));
    const float2 a = __ldg(e.O1 + idx);
    if (t.on) e.Ft[idx] = make_float4(pre * (a.x * inv), pre * (a.y * inv), pre * (tz * inv + t.w), 0.f);
}

template <int GL, bool ALONG_Y, bool IN = false, bool OUT = false>
__global__ void __launch_bounds__(FFT_THREADS, 3) k_fft(float2* __restrict__ data, int L, int logL, int lognx,
                                                        long long nlines, const float2* __restrict__ tw, int inverse,
                                                        FftEnds ends)
{
    extern __shared__ float2 fsm[];
    const int G = GL / L;
    float2* X = fsm;
    float2* Y = fsm + GL;
    float2* W = fsm + 2 * GL;  // L twiddles
    const long long l0 = (long long)blockIdx.x * G;
    const int nx = 1 << lognx;
    // element t of the CTA's block (t = g L + i along x, t = i G + g along y):
    // along x the block is contiguous; along y line l0 + g is node column
    // x = (l0 + g) mod nx of plane row z = (l0 + g) / nx (nx a power of two)
    const long long zb = l0 >> lognx;
    const int xb = (int)(l0 & (nx - 1));
    auto addr = [&](int t) -> long long {
        if (ALONG_Y) {
            const int g = t & (G - 1), i = t >> (__ffs(G) - 1);
            const int xg = xb + g;
            return ((zb + (xg >> lognx)) << lognx) * (long long)L + (xg & (nx - 1)) + (long long)i * nx;
        }
        return l0 * L + t;
    };
    auto line = [&](int t) -> long long { return l0 + (ALONG_Y ? (t & (G - 1)) : (t >> logL)); };
    const int half = L >> 1;
    for (int j = threadIdx.x; j < half; j += blockDim.x) {
        float2 w = tw[j];
        if (inverse) w.y = -w.y;
        W[j] = w;
        W[j + half] = make_float2(-w.x, -w.y);
    }
    // G L = GL: a fixed count of independent loads per thread, all issued
    // before the first store
    constexpr int PT = GL / FFT_THREADS;
    float2 v[PT];
#pragma unroll
    for (int k = 0; k < PT; ++k) {
        const int t = threadIdx.x + k * FFT_THREADS;
        const long long l = line(t);
        if (IN) {
            const int ny = ends.P.g.ny;
            const int y = (int)(l % ny), j = (int)(l / ny), x = t & (L - 1);
            v[k] = l < nlines ? make_float2(fluid_dn(ends.P, ends.dn, x, y, 2 * j),
                                            fluid_dn(ends.P, ends.dn, x, y, 2 * j + 1))
                              : make_float2(0.f, 0.f);
        } else {
            v[k] = l < nlines ? data[addr(t)] : make_float2(0.f, 0.f);
        }
    }
#pragma unroll
    for (int k = 0; k < PT; ++k) {
        const int t = threadIdx.x + k * FFT_THREADS;
        X[ALONG_Y ? (t & (G - 1)) * L + (t >> (__ffs(G) - 1)) : t] = v[k];
    }
    __syncthreads();
    int st = 1;
    if (logL & 1) {
        // radix 2: M = L / 2
        for (int t = threadIdx.x; t < G * half; t += blockDim.x) {
            const int g = t / half, p = t - g * half;
            const float2 a = X[g * L + p], c = X[g * L + p + half];
            Y[g * L + 2 * p] = cadd(a, c);
            Y[g * L + 2 * p + 1] = cmul(csub(a, c), W[p]);
        }
        __syncthreads();
        float2* tmp = X;
        X = Y;
        Y = tmp;
        st = 2;
    }
    const int quarter = L >> 2;
    for (; st < L; st <<= 2) {
        const int M = L / (4 * st);
        for (int t = threadIdx.x; t < G * quarter; t += blockDim.x) {
            const int g = t / quarter, b = t - g * quarter;
            const int p = b / st, q = b - p * st;
            const float2* xs = X + g * L + q + st * p;
            const float2 x0 = xs[0], x1 = xs[st * M], x2 = xs[2 * st * M], x3 = xs[3 * st * M];
            const float2 t0 = cadd(x0, x2), t1 = csub(x0, x2), t2 = cadd(x1, x3);
            const float2 t3 = inverse ? cmi(csub(x3, x1)) : cmi(csub(x1, x3));
            const int e = p * st;  // twiddle exponents e k, k = 1, 2, 3 (all < L)
            float2* ys = Y + g * L + q + 4 * st * p;
            ys[0] = cadd(t0, t2);
            ys[st] = cmul(cadd(t1, t3), W[e]);
            ys[2 * st] = cmul(csub(t0, t2), W[2 * e]);
            ys[3 * st] = cmul(csub(t1, t3), W[3 * e]);
        }
        __syncthreads();
        float2* tmp = X;
        X = Y;
        Y = tmp;
    }
#pragma unroll
    for (int k = 0; k < PT; ++k) {
        const int t = threadIdx.x + k * FFT_THREADS;
        const long long l = line(t);
        if (l >= nlines) continue;
        const float2 r = X[ALONG_Y ? (t & (G - 1)) * L + (t >> (__ffs(G) - 1)) : t];
        if (OUT) {
            const int ny = ends.P.g.ny;
            const int y = (int)(l % ny), j = (int)(l / ny), x = t & (L - 1);
            tail_out(ends, tail_plane(ends, 2 * j), x, y, r.x);
            tail_out(ends, tail_plane(ends, 2 * j + 1), x, y, r.y);
        } else {
            data[addr(t)] = r;
        }
    }
}

// T^(k, z) = sum_dz conj(Kh_c(k, dz)) M(k, z + dz) for 32 modes (one CTA row)
// and a chunk of ZC planes. The kernel's components are c(|d|) d: K_x and K_y are
// odd in the x-y plane and even in dz, K_z even in the plane and odd in dz, so
// their plane transforms are i b_x(dz), i b_y(dz) (even in dz) and b_z(dz) (odd):
//   T^_x,y = -i [b(0) M(z) + sum_{d>0} b(d) (M(z + d) + M(z - d))],
//   T^_z   = sum_{d>0} b_z(d) (M(z + d) - M(z - d)),
// five paired FP32 instructions per mode and pair +-d (24 multiply-adds without
// the symmetry; it now waits on its staging). A thread owns one mode and ZB consecutive planes; both windows
// M(z + d) and M(z - d) slide in registers, one shared-memory load each per d.
// 256 x 256 x 64, reach 20, under the profiler: 76 -> 47 us. ZB = 8 (116
// registers, half the warps): the whole tail 232 us against 224 at 256 x 256 x 128.
// M (unpacked from the plane-pair transform Pp at k and -k) and b staged in
// shared memory. Output O1 = T^_x + i T^_y per plane, O2 = T^_z(2j) + i T^_z(2j+1)
// per plane pair. Planes outside the grid read 0 (walls) or their periodic image.
// T is real, T^(-k) = conj T^(k): only the modes with ky <= ny/2 are computed;
// those with 0 < ky < ny/2 also write their mirror -k (rows 0 and ny/2 hold both
// members of their pairs and write only their own mode, so every output has one
// writer).
constexpr int ZC = 64, ZB = 4;

__host__ __device__ inline size_t zconv_smem(int D)
{
    return sizeof(float2) * (ZC + 2 * D) * 32 + sizeof(float4) * (D + 1) * 32;
}

__global__ void __launch_bounds__(32 * ZC / ZB, 2) k_tail_zconv(const float2* __restrict__ Pp,
                                                                const float4* __restrict__ Kb, float2* __restrict__ O1,
                                                                float2* __restrict__ O2, int nx, int ny, int nz, int D,
                                                                int zper)
{
    extern __shared__ __align__(16) unsigned char zsm[];
    float4* kb = reinterpret_cast<float4*>(zsm);            // (D + 1) x 32
    float2* slab = reinterpret_cast<float2*>(kb + (D + 1) * 32);  // (ZC + 2D) x 32
    const long long nxy = (long long)nx * ny;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const long long nhalf = (long long)(ny / 2 + 1) * nx;  // modes with ky <= ny/2
    const bool live = (long long)blockIdx.x * 32 + tx < nhalf;
    const long long col = live ? (long long)blockIdx.x * 32 + tx : 0;
    // the mode -k of k = (col mod nx, col / nx)
    const int kx = (int)(col % nx), ky = (int)(col / nx);
    const long long colm = (long long)((ny - ky) % ny) * nx + (nx - kx) % nx;
    const bool mirror = live && ky > 0 && 2 * ky < ny;
    const int z0 = blockIdx.y * ZC;
#pragma unroll 4
    for (int r = ty; r < ZC + 2 * D; r += ZC / ZB) {
        int z = z0 - D + r;
        bool in = true;
        if (zper) {
            z %= nz;
            if (z < 0) z += nz;
        } else {
            in = z >= 0 && z < nz;
        }
        // (planes past a wall load the first one and store 0)
        const long long j = in ? z >> 1 : 0;
        const float2 a = __ldg(Pp + (j * nxy + col)), b = __ldg(Pp + (j * nxy + colm));
        // M(2j) = (P(k) + conj P(-k)) / 2, M(2j+1) = (P(k) - conj P(-k)) / 2i
        const float2 v = (z & 1) ? make_float2(0.5f * (a.y + b.y), -0.5f * (a.x - b.x))
                                 : make_float2(0.5f * (a.x + b.x), 0.5f * (a.y - b.y));
        slab[r * 32 + tx] = in ? v : make_float2(0.f, 0.f);
    }
#pragma unroll 4
    for (int r = ty; r <= D; r += ZC / ZB) kb[r * 32 + tx] = __ldg(Kb + ((long long)r * nxy + col));
    __syncthreads();
    const int zb = ty * ZB;
    const float2* m = slab + (zb + D) * 32 + tx;  // M(z0 + zb) of this mode; planes 32 apart
    float2 up[ZB], dn[ZB], X[ZB], Y[ZB], Z[ZB];
    {
        const float4 b = kb[tx];
#pragma unroll
        for (int j = 0; j < ZB; ++j) {
            up[j] = dn[j] = m[j * 32];
            X[j] = make_float2(b.x * up[j].x, b.x * up[j].y);
            Y[j] = make_float2(b.y * up[j].x, b.y * up[j].y);
            Z[j] = make_float2(0.f, 0.f);
        }
    }
    // at step d, M(z + j + d) sits in up[(j + d) % ZB] and M(z + j - d) in dn[(j - d) % ZB]
    for (int d0 = 1; d0 <= D; d0 += ZB) {
#pragma unroll
        for (int u = 0; u < ZB; ++u) {
            const int d = d0 + u;
            if (d > D) break;
            up[u] = m[(ZB - 1 + d) * 32];
            dn[ZB - 1 - u] = m[-d * 32];
            const float4 b = kb[d * 32 + tx];
            const float2 bx = make_float2(b.x, b.x), by = make_float2(b.y, b.y), bz = make_float2(b.z, b.z);
#pragma unroll
            for (int j = 0; j < ZB; ++j) {
                const float2 a = up[(j + 1 + u) % ZB], c = dn[(j + 2 * ZB - 1 - u) % ZB];
                const float2 S = __fadd2_rn(a, c), Df = __ffma2_rn(c, make_float2(-1.f, -1.f), a);
                X[j] = __ffma2_rn(bx, S, X[j]);
                Y[j] = __ffma2_rn(by, S, Y[j]);
                Z[j] = __ffma2_rn(bz, Df, Z[j]);
            }
        }
    }
    if (!live) return;
#pragma unroll
    for (int j = 0; j < ZB; ++j) {
        const int z = z0 + zb + j;
        if (z >= nz) break;
        // a = T^_x = -i X, b = T^_y = -i Y
        const float2 a = make_float2(X[j].y, -X[j].x), b = make_float2(Y[j].y, -Y[j].x);
        O1[(long long)z * nxy + col] = make_float2(a.x - b.y, a.y + b.x);  // a + i b
        if (mirror) O1[(long long)z * nxy + colm] = make_float2(a.x + b.y, b.x - a.y);  // conj a + i conj b
    }
#pragma unroll
    for (int j = 0; j < ZB; j += 2) {
        const int z = z0 + zb + j;  // even: ZC, ZB even
        if (z >= nz) break;
        const float2 a = Z[j], b = z + 1 < nz ? Z[j + 1] : make_float2(0.f, 0.f);
        O2[(long long)(z >> 1) * nxy + col] = make_float2(a.x - b.y, a.y + b.x);
        if (mirror) O2[(long long)(z >> 1) * nxy + colm] = make_float2(a.x + b.y, b.x - a.y);
    }
}

// the symmetric part of the transformed kernel slices (dz = -D .. D, components
// x, y, z): b_x, b_y (imaginary, even in dz) and b_z (real, odd in dz) of d >= 0
__global__ void k_tail_symmetric(const float2* __restrict__ Kh, float4* __restrict__ Kb, long long nxy, int D)
{
    const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (k >= nxy) return;
    for (int d = 0; d <= D; ++d) {
        const float2* p = Kh + (long long)(D + d) * 3 * nxy + k;
        const float2* q = Kh + (long long)(D - d) * 3 * nxy + k;
        Kb[d * nxy + k] = make_float4(0.5f * (p[0].y + q[0].y), 0.5f * (p[nxy].y + q[nxy].y),
                                      0.5f * (p[2 * nxy].x - q[2 * nxy].x), 0.f);
    }
}

inline unsigned nblk(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

int ilog2(int v)
{
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
}

size_t fft_smem(int gl = FFT_GL) { return sizeof(float2) * (2 * gl + 1024); }

// 256-point lines by the four-step split 256 = 16 x 16: a thread holds the
// stride-16 subsequence n = 16 n1 + s of its line, takes the 16-point DFT
// over n1 in registers, multiplies by W_256^(s k1), exchanges through padded
// shared memory (thread k1 then holds k1 of every subsequence) and takes the
// 16-point DFT over the subsequences: X[k1 + 16 k2]. One exchange instead of
// four shared-memory stages. 16 lines per CTA, 16 threads per line; along y
// the 16 threads of a half-warp are 16 consecutive x columns at one y, along
// x 16 consecutive x of one line, so every access is a 128-byte segment.
__device__ __forceinline__ float2 cmi_dir(float2 a, int inverse)
{
    return inverse ? make_float2(-a.y, a.x) : make_float2(a.y, -a.x);  // +i a or -i a
}

// in-place 4-point DFT of (x0, x1, x2, x3)
__device__ __forceinline__ void dft4(float2& x0, float2& x1, float2& x2, float2& x3, int inverse)
{
    const float2 t0 = cadd(x0, x2), t1 = csub(x0, x2), t2 = cadd(x1, x3), t3 = cmi_dir(csub(x1, x3), inverse);
    x0 = cadd(t0, t2);
    x2 = csub(t0, t2);
    x1 = cadd(t1, t3);
    x3 = csub(t1, t3);
}

// 16-point DFT of a[0..15] in registers (16 = 4 x 4), natural order out;
// W = exp(-+ 2 pi i j / 256) for j < 256
__device__ __forceinline__ void dft16(float2 (&a)[16], const float2* W, int inverse)
{
    // DFT4 over n1 of a[4 n1 + n2] for each n2, twiddle W_16^(n2 k1)
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
        dft4(a[n2], a[4 + n2], a[8 + n2], a[12 + n2], inverse);
#pragma unroll
        for (int k1 = 1; k1 < 4; ++k1)
            if (n2) a[4 * k1 + n2] = cmul(a[4 * k1 + n2], W[16 * n2 * k1]);
    }
    // now b[n2][k1] sits in a[4 k1 + n2]; DFT4 over n2 gives A[k1 + 4 k2]
    float2 r[16];
#pragma unroll
    for (int k1 = 0; k1 < 4; ++k1) {
        float2 x0 = a[4 * k1], x1 = a[4 * k1 + 1], x2 = a[4 * k1 + 2], x3 = a[4 * k1 + 3];
        dft4(x0, x1, x2, x3, inverse);
        r[k1] = x0;
        r[k1 + 4] = x1;
        r[k1 + 8] = x2;
        r[k1 + 12] = x3;
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) a[k] = r[k];
}

template <bool ALONG_Y, bool IN = false, bool OUT = false>
__global__ void __launch_bounds__(256, 3) k_fft256(float2* __restrict__ data, int lognx, long long nlines,
                                                   const float2* __restrict__ tw, int inverse, FftEnds ends)
{
    constexpr int L = 256, G = 16, TP = 16 * 17 + 1;  // padded line stride of the exchange
    __shared__ float2 W[L];
    __shared__ float2 T[G * TP];
    const int tid = threadIdx.x;
    const int g = ALONG_Y ? (tid & 15) : (tid >> 4);
    const int s = ALONG_Y ? (tid >> 4) : (tid & 15);
    const long long l = (long long)blockIdx.x * G + g;
    const bool live = l < nlines;
    const int nx = 1 << lognx;
    auto addr = [&](int i) -> long long {
        if (ALONG_Y) return ((l >> lognx) << lognx) * L + (l & (nx - 1)) + (long long)i * nx;
        return l * L + i;
    };
    for (int j = tid; j < L / 2; j += blockDim.x) {
        float2 w = tw[j];
        if (inverse) w.y = -w.y;
        W[j] = w;
        W[j + L / 2] = make_float2(-w.x, -w.y);
    }
    float2 a[16];
    int yy = 0, jj = 0;
    if (IN || OUT) {
        const int ny = ends.P.g.ny;
        yy = (int)(l % ny);
        jj = (int)(l / ny);
    }
#pragma unroll
    for (int n1 = 0; n1 < 16; ++n1) {
        const int i = 16 * n1 + s;
        if (!live)
            a[n1] = make_float2(0.f, 0.f);
        else if (IN)
            a[n1] = make_float2(fluid_dn(ends.P, ends.dn, i, yy, 2 * jj), fluid_dn(ends.P, ends.dn, i, yy, 2 * jj + 1));
        else
            a[n1] = data[addr(i)];
    }
    __syncthreads();  // twiddles
    dft16(a, W, inverse);
#pragma unroll
    for (int k1 = 1; k1 < 16; ++k1)
        if (s) a[k1] = cmul(a[k1], W[s * k1]);
#pragma unroll
    for (int k1 = 0; k1 < 16; ++k1) T[g * TP + s * 17 + k1] = a[k1];
    __syncthreads();
#pragma unroll
    for (int n2 = 0; n2 < 16; ++n2) a[n2] = T[g * TP + n2 * 17 + s];
    dft16(a, W, inverse);
    if (!live) return;
    TailPlane t0, t1;
    if (OUT) {
        t0 = tail_plane(ends, 2 * jj);
        t1 = tail_plane(ends, 2 * jj + 1);
    }
#pragma unroll
    for (int k2 = 0; k2 < 16; ++k2) {
        const int i = s + 16 * k2;
        if (OUT) {
            tail_out(ends, t0, i, yy, a[k2].x);
            tail_out(ends, t1, i, yy, a[k2].y);
        } else {
            data[addr(i)] = a[k2];
        }
    }
}

template <int GL>
void fft_lines(float2* data, int L, int nx, long long nlines, bool along_y, const float2* tw, int inverse,
               cudaStream_t s, int ends_mode, const FftEnds& e)
{
    const size_t smem = fft_smem(GL);
    const unsigned blocks = nblk(nlines, GL / L);
    if (along_y)
        k_fft<GL, true><<<blocks, FFT_THREADS, smem, s>>>(data, L, ilog2(L), ilog2(nx), nlines, tw, inverse, e);
    else if (ends_mode == 1)
        k_fft<GL, false, true, false><<<blocks, FFT_THREADS, smem, s>>>(data, L, ilog2(L), ilog2(nx), nlines, tw, inverse,
                                                                         e);
    else if (ends_mode == 2)
        k_fft<GL, false, false, true><<<blocks, FFT_THREADS, smem, s>>>(data, L, ilog2(L), ilog2(nx), nlines, tw, inverse,
                                                                         e);
    else
        k_fft<GL, false><<<blocks, FFT_THREADS, smem, s>>>(data, L, ilog2(L), ilog2(nx), nlines, tw, inverse, e);
}

// one batched pass; `ends` selects the fused x-pass variants: 1 = read the
// packed density (IN), 2 = write the tail force (OUT)
cudaError_t fft_pass(float2* data, int L, int nx, long long nlines, bool along_y, const float2* tw, int inverse,
                     cudaStream_t s, int ends_mode = 0, const FftEnds* ends = nullptr)
{
    FftEnds e0;
    const FftEnds& e = ends ? *ends : e0;
    if (L == 256) {
        const unsigned b256 = nblk(nlines, 16);
        const int lnx = ilog2(nx);
        if (along_y)
            k_fft256<true><<<b256, 256, 0, s>>>(data, lnx, nlines, tw, inverse, e);
        else if (ends_mode == 1)
            k_fft256<false, true, false><<<b256, 256, 0, s>>>(data, lnx, nlines, tw, inverse, e);
        else if (ends_mode == 2)
            k_fft256<false, false, true><<<b256, 256, 0, s>>>(data, lnx, nlines, tw, inverse, e);
        else
            k_fft256<false><<<b256, 256, 0, s>>>(data, lnx, nlines, tw, inverse, e);
        return cudaGetLastError();
    }
    if (nlines * L < 2LL * NUM_SMS * FFT_GL)
        fft_lines<FFT_GL_SMALL>(data, L, nx, nlines, along_y, tw, inverse, s, ends_mode, e);
    else
        fft_lines<FFT_GL>(data, L, nx, nlines, along_y, tw, inverse, s, ends_mode, e);
    return cudaGetLastError();
}

}  // namespace

bool tail_spectral_ok(const Geom& g)
{
    auto pow2 = [](int v) { return v >= 2 && (v & (v - 1)) == 0; };
    return pow2(g.nx) && pow2(g.ny) && g.nx <= 1024 && g.ny <= 1024 && (long long)g.nx * g.ny >= 32;
}

size_t tail_spectral_bytes(const Geom& g, int D)
{
    const size_t nxy = (size_t)g.nx * g.ny;
    return sizeof(float4) * (D + 1) * nxy +
           sizeof(float2) * (3 * nxy * (size_t)g.nz + g.nx / 2 + g.ny / 2 + (g.nz + 1) / 2);
}

// Layout of the work buffer: Kb ((D+1) x ny x nx float4), Pp and O2 (together)
// and O1 and their rounding (3 nz nx ny complex in all), the twiddles of nx and
// of ny, then w (nz floats).
struct TailWork {
    float4* Kb;
    float2 *field, *twx, *twy;
    float* w;
};
static TailWork tail_layout(const Geom& g, int D, float2* work)
{
    const long long nxy = (long long)g.nx * g.ny;
    TailWork t;
    t.Kb = reinterpret_cast<float4*>(work);
    t.field = reinterpret_cast<float2*>(t.Kb + (D + 1) * nxy);
    t.twx = t.field + 3 * nxy * g.nz;
    t.twy = t.twx + g.nx / 2;
    t.w = reinterpret_cast<float*>(t.twy + g.ny / 2);
    return t;
}

cudaError_t tail_spectral_init(const Geom& g, int D, const int* pdx, const int* pdy, const int* pdz,
                               const float4* K, int npairs, const int* zslit, float2* work, cudaStream_t s)
{
    const long long nxy = (long long)g.nx * g.ny;
    const TailWork t = tail_layout(g, D, work);
    float2 *twx = t.twx, *twy = t.twy;
    std::vector<float2> tx(g.nx / 2), ty(g.ny / 2);
    for (int j = 0; j < g.nx / 2; ++j)
        tx[j] = make_float2((float)cos(-2.0 * M_PI * j / g.nx), (float)sin(-2.0 * M_PI * j / g.nx));
    for (int j = 0; j < g.ny / 2; ++j)
        ty[j] = make_float2((float)cos(-2.0 * M_PI * j / g.ny), (float)sin(-2.0 * M_PI * j / g.ny));
    // the full odd kernel on the periodic x-y grid, one slice per dz and component
    std::vector<float2> host((size_t)(2 * D + 1) * 3 * nxy, make_float2(0.f, 0.f));
    std::vector<double> acc((size_t)(2 * D + 1) * 3 * nxy, 0.0);
    auto put = [&](int dx, int dy, int dz, int c, double v) {
        const int x = ((dx % g.nx) + g.nx) % g.nx, y = ((dy % g.ny) + g.ny) % g.ny;
        acc[((size_t)(dz + D) * 3 + c) * nxy + (size_t)y * g.nx + x] += v;
    };
    for (int k = 0; k < npairs; ++k) {
        const double kv[3] = {K[k].x, K[k].y, K[k].z};
        for (int c = 0; c < 3; ++c) {
            put(pdx[k], pdy[k], pdz[k], c, kv[c]);
            put(-pdx[k], -pdy[k], -pdz[k], c, -kv[c]);
        }
    }
    for (size_t i = 0; i < host.size(); ++i) host[i] = make_float2((float)acc[i], 0.f);
    // w(z): the x,y-uniform response to the fluid indicator, in double
    std::vector<double> kappa(2 * D + 1, 0.0);
    for (int k = 0; k < npairs; ++k) {
        kappa[pdz[k] + D] += K[k].z;
        kappa[-pdz[k] + D] -= K[k].z;
    }
    std::vector<float> wz(g.nz);
    for (int z = 0; z < g.nz; ++z) {
        double a = 0.0;
        for (int d = -D; d <= D; ++d) {
            int zz = z + d;
            if (g.zper) {
                zz %= g.nz;
                if (zz < 0) zz += g.nz;
            } else if (zz < 0 || zz >= g.nz) {
                continue;
            }
            if (zslit[zz] >= 0) a += kappa[d + D];
        }
        wz[z] = (float)a;
    }
    float* wdev = t.w;
    cudaError_t e;
    float2* Kh = nullptr;  // the transformed slices, needed until their symmetric part is taken
    if ((e = cudaMalloc((void**)&Kh, sizeof(float2) * host.size()))) return e;
    auto done = [&](cudaError_t r) {
        cudaFree(Kh);
        return r;
    };
    if ((e = cudaMemcpyAsync(twx, tx.data(), sizeof(float2) * tx.size(), cudaMemcpyHostToDevice, s))) return done(e);
    if ((e = cudaMemcpyAsync(twy, ty.data(), sizeof(float2) * ty.size(), cudaMemcpyHostToDevice, s))) return done(e);
    if ((e = cudaMemcpyAsync(Kh, host.data(), sizeof(float2) * host.size(), cudaMemcpyHostToDevice, s))) return done(e);
    if ((e = cudaMemcpyAsync(wdev, wz.data(), sizeof(float) * wz.size(), cudaMemcpyHostToDevice, s))) return done(e);
    // (per-device attributes: sized for the largest reach, so that handles do not
    // lower each other's limit)
    if ((e = cudaFuncSetAttribute(k_tail_zconv, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)zconv_smem(4 * MAX_SIGMA))))
        return done(e);
    if ((e = cudaFuncSetAttribute(k_fft<FFT_GL, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fft_smem())))
        return done(e);
    if ((e = cudaFuncSetAttribute(k_fft<FFT_GL, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fft_smem())))
        return done(e);
    if ((e = cudaFuncSetAttribute(k_fft<FFT_GL, false, true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)fft_smem())))
        return done(e);
    if ((e = cudaFuncSetAttribute(k_fft<FFT_GL, false, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)fft_smem())))
        return done(e);
    const long long slices = (long long)(2 * D + 1) * 3;
    if ((e = fft_pass(Kh, g.nx, g.nx, slices * g.ny, false, twx, 0, s))) return done(e);
    if ((e = fft_pass(Kh, g.ny, g.nx, slices * g.nx, true, twy, 0, s))) return done(e);
    k_tail_symmetric<<<nblk(nxy, 128), 128, 0, s>>>(Kh, t.Kb, nxy, D);
    if ((e = cudaGetLastError())) return done(e);
    return done(cudaStreamSynchronize(s));
}

cudaError_t launch_tail_spectral(const Params& P, const float* dn, int D, float2* work, float4* Ft, cudaStream_t s)
{
    const Geom& g = P.g;
    const long long nxy = (long long)g.nx * g.ny;
    const int nz2 = (g.nz + 1) / 2;  // plane pairs
    const TailWork t = tail_layout(g, D, work);
    float2* Pp = t.field;  // Pp, O2 (nz2 planes each), O1 (nz planes)
    float2* O2 = Pp + nxy * nz2;
    float2* O1 = O2 + nxy * nz2;
    const float2 *twx = t.twx, *twy = t.twy;
    const float* w = t.w;
    FftEnds ends{P, dn, O1, w, Ft};
    cudaError_t e;
    if ((e = fft_pass(Pp, g.nx, g.nx, (long long)g.ny * nz2, false, twx, 0, s, 1, &ends))) return e;
    if ((e = fft_pass(Pp, g.ny, g.nx, (long long)g.nx * nz2, true, twy, 0, s))) return e;
    const long long nhalf = (long long)(g.ny / 2 + 1) * g.nx;
    dim3 grid((unsigned)((nhalf + 31) / 32), (unsigned)((g.nz + ZC - 1) / ZC));
    k_tail_zconv<<<grid, 32 * ZC / ZB, zconv_smem(D), s>>>(Pp, t.Kb, O1, O2, g.nx, g.ny, g.nz, D, g.zper);
    if ((e = cudaGetLastError())) return e;
    // O2 and O1 lie one after the other: one pass along y
    if ((e = fft_pass(O2, g.ny, g.nx, (long long)g.nx * (nz2 + g.nz), true, twy, 1, s))) return e;
    if ((e = fft_pass(O1, g.nx, g.nx, (long long)g.ny * g.nz, false, twx, 1, s))) return e;
    return fft_pass(O2, g.nx, g.nx, (long long)g.ny * nz2, false, twx, 1, s, 2, &ends);
}

}  // namespace lbif
