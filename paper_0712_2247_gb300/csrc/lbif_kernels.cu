// Device kernels of the hard-sphere lattice Boltzmann step (sm_103a).
//
// Arithmetic is FP32 on small quantities only. Populations are stored
// relative to the node's reference density (see lbif_internal.h), every
// field entering the nonlocal force is a deviation from the uniform state
// (dn = n/n0 - 1, dG = g2 - g2(eta0)), and mirror-image quadrature points are
// combined before they are summed, so a uniform state gives an exactly zero
// force. FP64 appears only in the profile / mass reductions.
#include <math.h>

#include <atomic>
#include <utility>

#include "lbif_device.cuh"

namespace lbif {

// ---------------------------------------------------------------------------
// initialisation and reference-field plumbing
// ---------------------------------------------------------------------------
struct OutsidePlanes {
    float* p[12];
    float v[12];
    int n;
};

__global__ void k_fill_outside(Params P, OutsidePlanes op)
{
    // constant values beyond the walls: n = 0 (dn = -1), u = 0, g2 unused (0)
    const Geom& g = P.g;
    long long plane = (long long)g.px * g.py;
    long long total = plane * 2 * g.hw;
    long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (k >= total) return;
    long long zl = k / plane;
    long long rem = k - zl * plane;
    int zp = (int)(zl < g.hw ? zl : zl + g.nz);
    long long p = (long long)zp * plane + rem;
    for (int j = 0; j < op.n; ++j) op.p[j][p] = op.v[j];
}

__device__ __forceinline__ uint64_t splitmix64(uint64_t x)
{
    uint64_t z = x + 0x9E3779B97F4A7C15ULL;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
    return z ^ (z >> 31);
}

// Every initial state below is an equilibrium: its stored populations (the
// non-equilibrium parts, see the pull pass) are 0 (the host zeroes the
// population buffer) and its moments are the fields themselves, written with
// their periodic images.
__global__ void k_init_noise(Params P, float* dn, uint64_t seed, double amp, long long offset)
{
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= P.g.N) return;
    int x, y, z;
    decompose(P.g, idx, x, y, z);
    if (slit_of(P, z) < 0) return;
    uint64_t r = splitmix64(seed ^ (uint64_t)(offset + idx));
    double U = (double)(r >> 11) * (1.0 / 9007199254740992.0);
    // f_i = w_i n0 (1 + xi) = f_i^eq(n0 (1 + xi), 0); u stays 0
    float xi = (float)(amp * (2.0 * U - 1.0));
    for_images(P.g, x, y, z, [&](int p) { dn[p] = xi; });
}

// the equilibrium of given density and velocity fields (u NULL: at rest)
__global__ void k_init_fields(Params P, float* dn, float* ux, float* uy, float* uz, const float* rho, const float* u)
{
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= P.g.N) return;
    int x, y, z;
    decompose(P.g, idx, x, y, z);
    const int s = slit_of(P, z);
    if (s < 0) return;
    const float d = rho[idx] / P.sl[s].rho0 - 1.f;
    const float vx = u ? u[idx] : 0.f, vy = u ? u[P.g.N + idx] : 0.f, vz = u ? u[2 * P.g.N + idx] : 0.f;
    for_images(P.g, x, y, z, [&](int p) {
        dn[p] = d;
        ux[p] = vx;
        uy[p] = vy;
        uz[p] = vz;
    });
}

// x,y-uniform equilibria from per-slit profiles n(z), u_x(z) (row s of n_z,
// ux_z holds slit s, entry j its plane zlo + j)
__global__ void k_init_profiles(Params P, float* dn, float* ux, float* uy, float* uz, const float* n_z,
                                const float* ux_z, int hmax)
{
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= P.g.N) return;
    int x, y, z;
    decompose(P.g, idx, x, y, z);
    const int s = slit_of(P, z);
    if (s < 0) return;
    const int j = z - P.sl[s].zlo;
    const float d = n_z[(long long)s * hmax + j] / P.sl[s].rho0 - 1.f;
    const float vx = ux_z ? ux_z[(long long)s * hmax + j] : 0.f;
    for_images(P.g, x, y, z, [&](int p) {
        dn[p] = d;
        ux[p] = vx;
        uy[p] = 0.f;
        uz[p] = 0.f;
    });
}

__global__ void k_tick(Params P, int4* clk)
{
    step_begin(P);
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= P.nslits || frozen(P, s)) return;
    int4 c = clk[s];
    c.x = c.x + 1 == P.g.nx ? 0 : c.x + 1;
    c.y = c.y + 1 == P.g.ny ? 0 : c.y + 1;
    c.z = c.z + 1 == P.sl[s].R ? 0 : c.z + 1;
    clk[s] = c;
}

// direction i of the current state in node order (gap planes skipped):
// to_pop = 0 gathers it from the buffer into canon, 1 scatters canon into it
template <typename T>
__global__ void k_pop_canon(Params P, T* pop, int i, T* canon, int to_pop)
{
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= P.g.N) return;
    int x, y, z;
    decompose(P.g, idx, x, y, z);
    const int s = slit_of(P, z);
    if (s < 0) return;
    long long at = idx;
    if (P.inplace) {
        // f_i(r, t) sits at the slot of coordinates r - t c_i
        const SlitParam S = P.sl[s];
        const int4 c = P.clk[s];
        const int xx = kCx(i) > 0 ? wrap_lo(x - c.x, P.g.nx) : (kCx(i) < 0 ? wrap_hi(x + c.x, P.g.nx) : x);
        const int yy = kCy(i) > 0 ? wrap_lo(y - c.y, P.g.ny) : (kCy(i) < 0 ? wrap_hi(y + c.y, P.g.ny) : y);
        const int zr = z - S.zlo;
        const int zz = kCz(i) > 0 ? wrap_lo(zr - c.z, S.R) : (kCz(i) < 0 ? wrap_hi(zr + c.z, S.R) : zr);
        at = ((long long)(S.zb + zz) * P.g.ny + yy) * P.g.nx + xx;
    }
    T* q = pop + (long long)i * P.g.Npad + at;
    if (to_pop)
        *q = canon[idx];
    else
        canon[idx] = *q;
}

// moment fields dn, ux, uy, uz <-> four unpadded N-arrays (checkpoints)
__global__ void k_write_fields(Params P, const float* src, float* dn, float* ux, float* uy, float* uz)
{
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= P.g.N) return;
    int x, y, z;
    decompose(P.g, idx, x, y, z);
    if (slit_of(P, z) < 0) return;
    const long long N = P.g.N;
    const float a = src[idx], b = src[N + idx], c = src[2 * N + idx], d = src[3 * N + idx];
    for_images(P.g, x, y, z, [&](int p) {
        dn[p] = a;
        ux[p] = b;
        uy[p] = c;
        uz[p] = d;
    });
}

__global__ void k_read_fields(Params P, const float* dn, const float* ux, const float* uy, const float* uz,
                              float* out)
{
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= P.g.N) return;
    int x, y, z;
    decompose(P.g, idx, x, y, z);
    const int p = pidx(P.g, x, y, z);
    const long long N = P.g.N;
    out[idx] = dn[p];
    out[N + idx] = ux[p];
    out[2 * N + idx] = uy[p];
    out[3 * N + idx] = uz[p];
}

// ---------------------------------------------------------------------------
// step 2: coarse-grained density over the ball |d| <= sigma/2 and the contact
// value g2(etabar) (Sec. Methods, Fischer-Methfessel prescription)
// ---------------------------------------------------------------------------
__device__ __forceinline__ float g2_deviation(const Params& P, float e0, float dnb, bool& bad)
{
    // g2(eta0 (1 + dnb)) - g2(eta0) written so that every term carries
    // Delta = eta0 dnb: (dN D0 - N0 dD) / (D1 D0), D = (1 - eta)^3
    float d = e0 * dnb;
    float a = 1.f - e0 - d, b = 1.f - e0;
    float N0, dN;
    if (P.g2form == 1) {
        N0 = 1.f - 0.5f * e0;
        dN = -0.5f * d;
    } else {
        N0 = 1.f - 0.5f * e0 + 0.25f * e0 * e0;
        dN = d * (-0.5f + 0.25f * (2.f * e0 + d));
    }
    float dD = -d * (a * a + a * b + b * b);
    float D0 = b * b * b, D1 = a * a * a;
    bad = !(a > 0.f);
    return (dN * D0 - N0 * dD) / (D1 * D0);
}

// tile of the z-marching ball kernel: 32 x 16 nodes, 256 threads, each thread
// the columns of two x-adjacent nodes, whose disc sums one paired addition
// serves (sigma 12 on 512 x 512 x 192, 1216 CTAs: two y-adjacent nodes with scalar
// additions 0.554 ms, two x-adjacent ones paired 0.535 ms; 256 slits of 32 x 32,
// sigma 4, 0.115 -> 0.105 ms; CTAs of 4 / 8 / 16 warps ran 0.567 / 0.552 / 0.573 ms
// in the former form)
constexpr int BALL_TX = 32, BALL_TY = 16, BALL_THREADS = BALL_TX / 2 * BALL_TY;

// x halo of the staged plane tile: R rounded up to 4, so that tile rows and
// their global sources are float4-aligned
template <int R>
constexpr int ball_c4() { return (R + 3) / 4 * 4; }

template <int R>
constexpr int ball_smem_floats()
{
    return (BALL_TY + 2 * R) * (BALL_TX + 2 * ball_c4<R>()) + (R + 1) * (BALL_TY + 2 * R) * BALL_TX;
}

// Self-test of the bounded wait above: the CTA waits on an mbarrier that
// nothing arrives on (its first phase never completes), gives up after
// `polls` polls, records bit 4 of status as the tile kernels do, and returns.
__global__ void k_wait_selftest(long long polls, int* status)
{
    __shared__ __align__(8) uint64_t mbar;
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&mbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    long long spins = 0;
    bool ok;
    while (!(ok = mbar_wait_parity(&mbar, 0)) && ++spins < polls) {
    }
    if (!__syncthreads_and(ok) && threadIdx.x == 0) atomicOr(status, 4);
}

// does the row at dy = r - R enter a disc sum D_k with row half-width w?
__host__ __device__ constexpr bool ball_row_used(int R, int r, int w)
{
    for (int k = 0; k <= R; ++k) {
        const int rem = R * R - k * k - (r - R) * (r - R);
        if (rem >= 0 && cisqrt(rem) == w) return true;
    }
    return false;
}

// Compile-time expansion of the disc sums of one thread: for every row r (in
// increasing order) and half-width w that some D[k] uses, one shared-memory
// read of the two columns' row sums, added into exactly those D[k].
template <int R, int r, int w, int k>
__device__ __forceinline__ void ball_add_one(float2 v, float2 (&D)[R + 1])
{
    constexpr int dy = r - R, rem = R * R - k * k - dy * dy;
    if constexpr (rem >= 0 && cisqrt(rem) == w) D[k] = __fadd2_rn(D[k], v);
}

template <int R, int r, int w, int... K>
__device__ __forceinline__ void ball_add_row(float2 v, float2 (&D)[R + 1], std::integer_sequence<int, K...>)
{
    (ball_add_one<R, r, w, K>(v, D), ...);
}

template <int R, int N>
__device__ __forceinline__ void ball_disc_row(const float* __restrict__ RS, int off, float2 (&D)[R + 1])
{
    constexpr int r = N / (R + 1), w = N % (R + 1);
    constexpr int H = BALL_TY + 2 * R;
    if constexpr (ball_row_used(R, r, w)) {
        const float2 v = *reinterpret_cast<const float2*>(RS + (w * H + r) * BALL_TX + off);
        ball_add_row<R, r, w>(v, D, std::make_integer_sequence<int, R + 1>{});
    }
}

// the comma fold runs the rows in increasing order
template <int R, int... N>
__device__ __forceinline__ void ball_disc_rows(const float* __restrict__ RS, int off, float2 (&D)[R + 1],
                                               std::integer_sequence<int, N...>)
{
    (ball_disc_row<R, N>(RS, off, D), ...);
}

// Row sums of every half-width 0..R for four adjacent columns per thread,
// from a staged plane tile T (H x W, column C4 + c holds node column c): the
// window sits in registers, additions grow outwards from the centre column.
template <int R>
__device__ __forceinline__ void ball_rowsums(const float* __restrict__ T, float* __restrict__ RS)
{
    constexpr int TX = BALL_TX, TY = BALL_TY;
    constexpr int C4 = ball_c4<R>();
    constexpr int W = TX + 2 * C4, H = TY + 2 * R;
    constexpr int NF = (C4 + R + 7) / 4;  // float4s a 4-column row-sum group reads
    for (int k = threadIdx.x; k < H * (TX / 4); k += blockDim.x) {
        int row = k / (TX / 4), c = 4 * (k - row * (TX / 4));
        const float* tr = T + row * W + c;
        float t[4 * NF];
#pragma unroll
        for (int i = 0; i < NF; ++i) {
            float4 v = *reinterpret_cast<const float4*>(tr + 4 * i);
            t[4 * i] = v.x;
            t[4 * i + 1] = v.y;
            t[4 * i + 2] = v.z;
            t[4 * i + 3] = v.w;
        }
        float s[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) s[j] = t[C4 + j];
        *reinterpret_cast<float4*>(RS + row * TX + c) = make_float4(s[0], s[1], s[2], s[3]);
#pragma unroll
        for (int w = 1; w <= R; ++w) {
#pragma unroll
            for (int j = 0; j < 4; ++j) s[j] += t[C4 + j - w] + t[C4 + j + w];
            *reinterpret_cast<float4*>(RS + (w * H + row) * TX + c) = make_float4(s[0], s[1], s[2], s[3]);
        }
    }
}

// Disc sums of input plane zi for the thread's two nodes (x, x + 1; y), added
// into the register ring acc of the 2R+1 output planes they touch; the completed
// plane zi - R is written (g2 deviation, with its periodic images), the ring
// shifts.
template <int R>
__device__ __forceinline__ void ball_disc_out(const Params& P, const float* __restrict__ RS, float2 (&acc)[2 * R + 1],
                                              int zi, int z0, int x, int y, int off, float* __restrict__ dG,
                                              int* status, int skip_done)
{
    const Geom& g = P.g;
    // D[k] = sum over dy = -R..R (in that order) of the row sum of half-width
    // cisqrt(R^2 - k^2 - dy^2) at row y + dy
    float2 D[R + 1];
#pragma unroll
    for (int k = 0; k <= R; ++k) D[k] = make_float2(0.f, 0.f);
    ball_disc_rows<R>(RS, off, D, std::make_integer_sequence<int, (2 * R + 1) * (R + 1)>{});
#pragma unroll
    for (int k = 0; k <= R; ++k) {
        acc[R - k] = __fadd2_rn(acc[R - k], D[k]);
        if (k) acc[R + k] = __fadd2_rn(acc[R + k], D[k]);
    }
    const int zo = zi - R;
    const int so = zo >= z0 ? slit_of(P, zo) : -1;
    if (so >= 0 && x < g.nx && y < g.ny && !(skip_done && frozen(P, so))) {
        const float e0 = P.sl[so].eta0;
        bool bad0, bad1;
        const float2 v = make_float2(g2_deviation(P, e0, acc[0].x * P.ball_inv, bad0),
                                     g2_deviation(P, e0, acc[0].y * P.ball_inv, bad1));
        const bool two = x + 1 < g.nx;
        if (bad0 || (two && bad1)) atomicOr(status, 2);
        if (two && no_images(g, x, y, zo) && no_images(g, x + 1, y, zo)) {
            // x, hw and px even: 8-byte aligned
            *reinterpret_cast<float2*>(dG + pidx(g, x, y, zo)) = v;
        } else {
            for_images(g, x, y, zo, [&](int q) { dG[q] = v.x; });
            if (two) for_images(g, x + 1, y, zo, [&](int q) { dG[q] = v.y; });
        }
    }
#pragma unroll
    for (int j = 0; j < 2 * R; ++j) acc[j] = acc[j + 1];
    acc[2 * R] = make_float2(0.f, 0.f);
}

// One CTA = a 32 x 16 column of nodes marching up a z chunk. Per input plane:
// stage the plane (+R halo) in shared memory, build x-row sums of every
// half-width 0..R, form the disc sums D_k (disc of radius^2 R^2 - k^2; a
// thread reads each row sum it needs once for its two nodes) and add
// them into a register ring of the 2R+1 output planes they touch, emit the
// completed plane.
template <int R>
__global__ void __launch_bounds__(BALL_THREADS) k_ball(Params P, const float* dn,
                                              float* __restrict__ dG, int* status, int zchunk,
                                              int skip_done)
{
    step_begin(P);
    constexpr int TX = BALL_TX, TY = BALL_TY;
    constexpr int C4 = ball_c4<R>();
    constexpr int W = TX + 2 * C4, H = TY + 2 * R;
    extern __shared__ __align__(16) float sm[];
    float* T = sm;           // H x W plane tile
    float* RS = sm + H * W;  // (R+1) x H x TX row sums
    const Geom& g = P.g;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int z0 = blockIdx.z * zchunk;
    const int z1 = min(z0 + zchunk, g.nz);
    const int tx = 2 * (threadIdx.x % (TX / 2)), ty = threadIdx.x / (TX / 2);
    const int x = x0 + tx, y = y0 + ty, off = ty * TX + tx;
    float2 acc[2 * R + 1];
#pragma unroll
    for (int j = 0; j <= 2 * R; ++j) acc[j] = make_float2(0.f, 0.f);

    for (int zi = z0 - R; zi < z1 + R; ++zi) {
        const float* plane = dn + (long long)(zi + g.hw) * g.py * g.px;
        // stage the plane tile with float4 copies (padded rows are 16-byte
        // aligned and hw >= C4, so every source float4 lies inside its row or
        // entirely past its end)
        for (int k = threadIdx.x; k < H * (W / 4); k += blockDim.x) {
            int row = k / (W / 4), q = k - row * (W / 4);
            int xp = x0 - C4 + g.hw + 4 * q, yp = y0 - R + row + g.hw;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (xp + 3 < g.px && yp < g.py) v = ld4(plane + (long long)yp * g.px + xp);
            *reinterpret_cast<float4*>(T + row * W + 4 * q) = v;
        }
        __syncthreads();
        ball_rowsums<R>(T, RS);
        __syncthreads();
        ball_disc_out<R>(P, RS, acc, zi, z0, x, y, off, dG, status, skip_done);
        __syncthreads();
    }
}

// The same kernel with the plane tiles brought in by the tensor-memory
// accelerator: one cp.async.bulk.tensor copy per plane (a W x H x 1 box of
// the padded density field, out-of-range rows filled with zeros), issued by
// one thread two planes ahead into alternating buffers, completion counted
// in bytes on an mbarrier per buffer. The arithmetic is k_ball's.
template <int R>
__global__ void __launch_bounds__(BALL_THREADS) k_ball_tma(Params P, const __grid_constant__ CUtensorMap tmap,
                                                  float* __restrict__ dG, int* status, int zchunk,
                                                  int skip_done)
{
    step_begin(P);
    constexpr int TX = BALL_TX, TY = BALL_TY;
    constexpr int C4 = ball_c4<R>();
    constexpr int W = TX + 2 * C4, H = TY + 2 * R;
    constexpr int TB = (H * W * 4 + 127) / 128 * 128;  // bytes of one tile buffer
    extern __shared__ __align__(128) unsigned char bsm[];
    float* RS = reinterpret_cast<float*>(bsm + 2 * TB);                 // (R+1) x H x TX
    uint64_t* mbar = reinterpret_cast<uint64_t*>(RS + (R + 1) * H * TX);  // 2 barriers
    const Geom& g = P.g;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int z0 = blockIdx.z * zchunk;
    const int z1 = min(z0 + zchunk, g.nz);
    const int tx = 2 * (threadIdx.x % (TX / 2)), ty = threadIdx.x / (TX / 2);
    const int x = x0 + tx, y = y0 + ty, off = ty * TX + tx;
    const int np = (z1 + R) - (z0 - R);  // input planes of this chunk
    // box origin in padded coordinates; x0 - C4 + hw is a multiple of 4 (16 bytes)
    const int bx = x0 - C4 + g.hw, by = y0 - R + g.hw;
    if (threadIdx.x == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tmap)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(mbar)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(mbar + 1)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    auto issue = [&](int q) {  // plane z0 - R + q into buffer q & 1 (one thread)
        const int b = q & 1;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(mbar + b)),
                     "r"((uint32_t)(H * W * 4))
                     : "memory");
        asm volatile(
            "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], "
            "[%5];" ::"r"(smem_addr(bsm + b * TB)),
            "l"(reinterpret_cast<uint64_t>(&tmap)), "r"(bx), "r"(by), "r"(z0 - R + q + g.hw), "r"(smem_addr(mbar + b))
            : "memory");
    };
    if (threadIdx.x == 0) {
        // the density was written by ordinary stores of a kernel that step_begin
        // waited for, not by an earlier launch boundary: order the copies after them
        asm volatile("fence.proxy.async.global;" ::: "memory");
        issue(0);
        if (np > 1) issue(1);
    }
    float2 acc[2 * R + 1];
#pragma unroll
    for (int j = 0; j <= 2 * R; ++j) acc[j] = make_float2(0.f, 0.f);
    uint32_t pbits = 0u;  // bit b: phase parity expected next on buffer b
    for (int q = 0; q < np; ++q) {
        const int b = q & 1;
        long long spins = 0;
        bool ok;
        while (!(ok = mbar_wait_parity(mbar + b, (pbits >> b) & 1u)) && ++spins < BALL_WAIT_LIMIT) {
        }
        if (!__syncthreads_and(ok)) {
            // record the timeout and wait (bounded) for the copies in flight
            if (threadIdx.x == 0) atomicOr(status, 4);
            for (int k = 0; k < 2; ++k) {
                if (q + k >= np) break;
                const int bk = (q + k) & 1;
                spins = 0;
                while (!mbar_wait_parity(mbar + bk, (pbits >> bk) & 1u) && ++spins < BALL_WAIT_LIMIT) {
                }
            }
            return;
        }
        pbits ^= 1u << b;
        ball_rowsums<R>(reinterpret_cast<const float*>(bsm + b * TB), RS);
        __syncthreads();  // buffer b is read: refill it two planes ahead
        if (threadIdx.x == 0 && q + 2 < np) issue(q + 2);
        ball_disc_out<R>(P, RS, acc, z0 - R + q, z0, x, y, off, dG, status, skip_done);
        __syncthreads();
    }
}

// Narrow grids (a 32 x 16 tile would leave most lanes idle): one thread per
// node, reading the padded field directly. The additions run in the order of
// k_ball (row sums grown outwards from the centre, disc sums over y, then the
// planes in increasing z), so both kernels give bit-identical results. Radii up
// to 4 are unrolled, so that a node's loads (33 at R = 2, 257 at R = 4) go out
// together instead of one chain of a few at a time: at R = 2, 2048 slits of 4 x 4
// 57 -> 30 us, 16 x 16 x 32 13 -> 7.4 us. Larger ones run the loop, four dx at a time
// (15 x 200 x 150, sigma 10: 107 us, 113 as the compiler unrolls it by itself).
template <int R0>
__global__ void __launch_bounds__(256) k_ball_direct(Params P, const float* dn,
                                                     float* __restrict__ dG, int* status, int skip_done)
{
    step_begin(P);
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= P.g.N) return;
    int x, y, z;
    decompose(P.g, idx, x, y, z);
    const int so = slit_of(P, z);
    if (so < 0 || (skip_done && frozen(P, so))) return;
    const int p = pidx(P.g, x, y, z);
    const int sy = P.g.px, sz = P.g.px * P.g.py;
    float s = 0.f;
    if constexpr (R0 > 0) {
#pragma unroll
        for (int dz = -R0; dz <= R0; ++dz) {
            float D = 0.f;
#pragma unroll
            for (int dy = -R0; dy <= R0; ++dy) {
                const int rem = R0 * R0 - dy * dy - dz * dz;
                if (rem < 0) continue;
                const int w = cisqrt(rem);
                const float* row = dn + p + (dz * sz + dy * sy);
                float r = ldp(row);
#pragma unroll
                for (int dx = 1; dx <= R0; ++dx)
                    if (dx <= w) r += ldp(row - dx) + ldp(row + dx);
                D += r;
            }
            s += D;
        }
    } else {
        const int R = P.sigma / 2;
        for (int dz = -R; dz <= R; ++dz) {
            float D = 0.f;
            for (int dy = -R; dy <= R; ++dy) {
                const int rem = R * R - dy * dy - dz * dz;
                if (rem < 0) continue;
                const int w = cisqrt(rem);
                const float* row = dn + p + (dz * sz + dy * sy);
                float r = ldp(row);
#pragma unroll 4
                for (int dx = 1; dx <= w; ++dx) r += ldp(row - dx) + ldp(row + dx);
                D += r;
            }
            s += D;
        }
    }
    bool bad;
    float v = g2_deviation(P, P.sl[so].eta0, s * P.ball_inv, bad);
    if (bad) atomicOr(status, 2);
    for_images(P.g, x, y, z, [&](int q) { dG[q] = v; });
}

// ---------------------------------------------------------------------------
// step 4: mean-field attractive tail, F/n0 = n0 (1 + dn) sum_d dn(r+d) phi'(|d|) d/|d|,
// by direct summation (lateral extents without a spectral transform). The kernel
// is odd, so the sum runs over pairs +-d: with c(d) = phi'(|d|)/|d| and, for a row
// (dy, dz) of displacements,
//   A(dx) = dn(r + d) - dn(r - d),
//   sum over dx and -dx:  c (A(dx) + A(-dx)) (dy, dz)  and  c dx (A(dx) - A(-dx)) x^,
// two additions, two subtractions and two multiply-adds for two pairs. A thread
// owns four x nodes and slides register windows of both rows outwards four dx at
// a time (four 16-byte loads and 96 FP32 instructions per 32 node-pairs of
// displacements; the former kernel loaded two scalars for each). The rows of a
// tile of 128 nodes are dealt to the eight warps of its CTA, whose sums are
// added in order, so that small grids fill the chip. It is bound by issue (about
// 115 instructions per four dx, a third of whose coefficients are zero where a
// row ends inside them). 60 x 52 x 40, sigma 4 (1,960 pairs a node): 287 -> 83
// us; 100 x 100 x 60, sigma 8 (15,649 pairs): 8.31 -> 1.87 ms. Three CTAs per SM
// (80 registers) 101 us, 16 / 4 warps per tile 93 / 88 us, no unrolling 88 us.
// ---------------------------------------------------------------------------
constexpr int TAIL_WARPS = 8;

// The sums of one node over the terms of the shell alone, in the kernel's order. The
// kernel also multiplies the neighbours that its chunks of four dx reach outside the
// shell, by zero coefficients; a node whose sums are not finite takes them from
// here, so that an infinite density reaches only the nodes whose shell holds it.
__device__ __noinline__ void tail_shell_only(const float* p, const TailRow* rows, int nrows, const float4* coef,
                                             float t[3])
{
    for (int w = 0; w < TAIL_WARPS; ++w) {
        float s[3] = {0.f, 0.f, 0.f};
        for (int r = w; r < nrows; r += TAIL_WARPS) {
            const TailRow row = rows[r];
            float rs = 0.f, rd = 0.f;
            for (int j = 0; j < 4 * row.count; ++j) {
                const float* c = reinterpret_cast<const float*>(coef + row.coef + 2 * (j / 4)) + j % 4;
                if (c[0] == 0.f && c[4] == 0.f) continue;
                const int dx = 4 * row.first + j;
                const float a = p[row.off + dx] - p[-row.off - dx], b = p[row.off - dx] - p[dx - row.off];
                rs = fmaf(c[0], a + b, rs);
                rd = fmaf(c[4], a - b, rd);
            }
            s[0] += rd;
            s[1] = fmaf(row.dy, rs, s[1]);
            s[2] = fmaf(row.dz, rs, s[2]);
        }
        for (int c = 0; c < 3; ++c) t[c] = w ? t[c] + s[c] : s[c];
    }
}

__global__ void __launch_bounds__(32 * TAIL_WARPS, 2) k_tail(Params P, const float* __restrict__ dn,
                                                          const TailRow* __restrict__ rows, int nrows,
                                                          const float4* __restrict__ coef, float4* __restrict__ Ft)
{
    __shared__ float part[TAIL_WARPS][12][32];
    const Geom& g = P.g;
    const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
    const int xb = (g.nx + 3) / 4;
    const long long nb = (long long)xb * g.ny * g.nz;
    // the lane's block of four x nodes (past the last one: the last again)
    auto block_of = [&](int l, int& x, int& y, int& z) {
        long long b = blockIdx.x * 32LL + l;
        const bool live = b < nb;
        if (!live) b = nb - 1;
        const int r = (int)(b / xb);
        x = 4 * (int)(b - (long long)r * xb);
        z = r / g.ny;
        y = r - z * g.ny;
        return live;
    };
    int x, y, z;
    block_of(lane, x, y, z);
    const float* base = dn + pidx(g, x, y, z);
    float sx[4], sy[4], sz[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) sx[i] = sy[i] = sz[i] = 0.f;
    TailRow next;
    if (warp < nrows) next = rows[warp];
    // gap planes and frozen slits have no tail force (the eight warps hold the same
    // nodes, so the whole CTA leaves): 64 slits of 20 x 20 x 8..80, sigma 4 0.823 ->
    // 0.659 ms; after the first row's load, as before it the two dependent loads
    // cost 60 x 52 x 40 1.5 us
    const int sl = slit_of(P, z);
    if (!__any_sync(0xffffffffu, sl >= 0 && !frozen(P, sl))) return;
    for (int r = warp; r < nrows; r += TAIL_WARPS) {
        const TailRow row = next;
        if (r + TAIL_WARPS < nrows) next = rows[r + TAIL_WARPS];
        const float* p = base + row.off + 4 * row.first;   // r + d, dx = 4 first
        const float* q = base + row.off - 4 * row.first;   // r + d, dx = -4 first
        const float* m = base - row.off + 4 * row.first;   // the same of r - (0, dy, dz)
        const float* n = base - row.off - 4 * row.first;
        float rs[4], rd[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) rs[i] = rd[i] = 0.f;
        float4 p0 = ld4(p), q0 = ld4(q), m0 = ld4(m), n0 = ld4(n);
        const float4* c4 = coef + row.coef;
#pragma unroll 2
        for (int j = 0; j < row.count; ++j) {
            p += 4, m += 4, q -= 4, n -= 4;
            const float4 cs = __ldg(c4 + 2 * j), cd = __ldg(c4 + 2 * j + 1);
            const float4 p1 = ld4(p), q1 = ld4(q), m1 = ld4(m), n1 = ld4(n);
            const float pw[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
            const float mw[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
            const float qw[8] = {q1.x, q1.y, q1.z, q1.w, q0.x, q0.y, q0.z, q0.w};
            const float nw[8] = {n1.x, n1.y, n1.z, n1.w, n0.x, n0.y, n0.z, n0.w};
            const float ck[4] = {cs.x, cs.y, cs.z, cs.w}, dk[4] = {cd.x, cd.y, cd.z, cd.w};
#pragma unroll
            for (int k = 0; k < 4; ++k)
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const float a = pw[i + k] - nw[4 + i - k], b = qw[4 + i - k] - mw[i + k];
                    rs[i] = fmaf(ck[k], a + b, rs[i]);
                    rd[i] = fmaf(dk[k], a - b, rd[i]);
                }
            p0 = p1, q0 = q1, m0 = m1, n0 = n1;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            sx[i] += rd[i];
            sy[i] = fmaf(row.dy, rs[i], sy[i]);
            sz[i] = fmaf(row.dz, rs[i], sz[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        part[warp][3 * i][lane] = sx[i];
        part[warp][3 * i + 1][lane] = sy[i];
        part[warp][3 * i + 2][lane] = sz[i];
    }
    __syncthreads();
    if (warp >= 4) return;
    // warp w adds node w of every lane's block
    if (!block_of(lane, x, y, z) || x + warp >= g.nx) return;
    const int s = slit_of(P, z);
    if (s < 0 || frozen(P, s)) return;
    float t[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        t[c] = part[0][3 * warp + c][lane];
#pragma unroll
        for (int w = 1; w < TAIL_WARPS; ++w) t[c] += part[w][3 * warp + c][lane];
    }
    if (!isfinite(t[0] + t[1] + t[2])) tail_shell_only(base + warp, rows, nrows, coef, t);
    const float pre = P.sl[s].rho0 * (1.f + __ldg(base + warp));
    Ft[((long long)z * g.ny + y) * g.nx + x + warp] = make_float4(pre * t[0], pre * t[1], pre * t[2], 0.f);
}

// Shells of few pairs (a cut-off just above sigma): one node per thread, pair by
// pair, which needs no zero coefficients, no sums across warps and two loads a pair
// (tail_by_pairs says when).
__global__ void __launch_bounds__(256) k_tail_pairs(Params P, const float* __restrict__ dn, const int* __restrict__ off,
                                                    const float4* __restrict__ K, int npairs, float4* __restrict__ Ft)
{
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= P.g.N) return;
    int x, y, z;
    decompose(P.g, idx, x, y, z);
    const int s = slit_of(P, z);
    if (s < 0 || frozen(P, s)) return;
    const float* p = dn + pidx(P.g, x, y, z);
    float sx = 0.f, sy = 0.f, sz = 0.f;
    for (int k = 0; k < npairs; ++k) {
        const int o = __ldg(off + k);
        const float d = __ldg(p + o) - __ldg(p - o);
        const float4 c = __ldg(K + k);
        sx = fmaf(c.x, d, sx);
        sy = fmaf(c.y, d, sy);
        sz = fmaf(c.z, d, sz);
    }
    const float pre = P.sl[s].rho0 * (1.f + __ldg(p));
    Ft[idx] = make_float4(pre * sx, pre * sy, pre * sz, 0.f);
}

// ---------------------------------------------------------------------------
// outputs
// ---------------------------------------------------------------------------
__global__ void k_force_soa(Params P, const float4* __restrict__ F, float* __restrict__ out)
{
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= P.g.N) return;
    float4 v = F[idx];
    out[idx] = v.x;
    out[P.g.N + idx] = v.y;
    out[2 * P.g.N + idx] = v.z;
}

// sum over the 18 points of W_q A_q (A_q = G_q n_q / n0 - G0)
__device__ __forceinline__ float shell_A_sum(const Params& P, const Fields& fl, int p, float G0)
{
    float s = 0.f;
    for (int a = 0; a < 3; ++a)
        for (int sg = -1; sg <= 1; sg += 2) {
            float dq = __ldg(fl.dn + p + sg * P.sh.ax_nb[a]);
            float gq = __ldg(fl.dG + p + sg * P.sh.ax_md[a]);
            s += (1.f / 30.f) * shell_A(dq, gq, G0);
        }
    for (int pl = 0; pl < 3; ++pl)
        for (int m = 0; m < 4; ++m) {
            const int sa = (m & 1) ? -1 : 1, sb = (m & 2) ? -1 : 1;
            float dq = 0.f, gq = 0.f;
            for (int k = 0; k < 4; ++k) {
                dq += P.sh.nb_w[pl][k] * __ldg(fl.dn + p + sa * P.sh.nb_a[pl][k] + sb * P.sh.nb_b[pl][k]);
                gq += P.sh.md_w[pl][k] * __ldg(fl.dG + p + sa * P.sh.md_a[pl][k] + sb * P.sh.md_b[pl][k]);
            }
            s += (1.f / 15.f) * shell_A(dq, gq, G0);
        }
    return s;
}

// rho, u and p = kT n + (kT sigma^3/6) 4 pi n0^2 (1 + dn) sum_q W_q (G0 + A_q)
__global__ void k_moments_out(Params P, Fields fl, float* rho, float* u, float* pr)
{
    long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= P.g.N) return;
    int x, y, z;
    decompose(P.g, idx, x, y, z);
    const int sl = slit_of(P, z);
    if (sl < 0) {
        if (rho) rho[idx] = 0.f;
        if (u) u[idx] = u[P.g.N + idx] = u[2 * P.g.N + idx] = 0.f;
        if (pr) pr[idx] = 0.f;
        return;
    }
    const SlitParam S = P.sl[sl];
    int p = pidx(P.g, x, y, z);
    const float d = fl.dn[p];
    if (rho) rho[idx] = S.rho0 * (1.f + d);
    if (u) {
        u[idx] = fl.ux[p];
        u[P.g.N + idx] = fl.uy[p];
        u[2 * P.g.N + idx] = fl.uz[p];
    }
    if (pr) {
        float s = 0.f;
        if (P.hs) s = (S.G0 + shell_A_sum(P, fl, p, S.G0)) * S.p_pref * (1.f + d);
        pr[idx] = (1.f / 3.f) * S.rho0 * (1.f + d) + s;
    }
}

// Per z plane: sum dn, sum ux, sum (1+dn) u (FP64 results, fixed order): CTA
// (z, c) reduces rows [c rc, (c+1) rc) of plane z into part, then
// k_profiles_sum adds the chunks of a plane in order. Per node the work is
// FP32 only (FP64 runs at a small fraction of the FP32 rate on this GPU):
// each thread keeps every sum as an unevaluated pair hi + lo of FP32 numbers,
// updated by Knuth's two-sum, which yields the rounding error of each FP32
// addition exactly, so the pair carries about 48 bits; the products
// (1 + dn) u enter as u + p + e with p = fl(dn u) and e = dn u - p (exact, by
// a fused multiply-add). Each thread converts its pairs to FP64 once; the
// CTA adds them by a fixed FP64 tree. (Merging the threads' pairs in FP32 too
// takes 28 us at 256 x 192 x 96, but 48 bits are too few where a plane's average
// cancels to far below the flow's amplitude; 38 us with four x nodes a thread,
// whose other order of additions moves such an average by 1e-9 of itself.)
// A thread's loads go out for PROF_U nodes at a time: 66 -> 50 us.
constexpr int PROF_K = 5;

struct F32Pair {
    float hi, lo;
};

__device__ __forceinline__ void pair_add(F32Pair& a, float x)
{
    const float s = a.hi + x;
    const float bb = s - a.hi;
    a.lo += (a.hi - (s - bb)) + (x - bb);
    a.hi = s;
}

constexpr int PROF_U = 4;
__global__ void __launch_bounds__(256) k_profiles(Params P, Fields fl, double* part, int chunks)
{
    __shared__ double sh[PROF_K][256];
    const Geom& g = P.g;
    const int z = blockIdx.x, c = blockIdx.y;
    const int rc = (g.ny + chunks - 1) / chunks;
    const int y0 = min(g.ny, c * rc), y1 = min(g.ny, y0 + rc);
    F32Pair a[PROF_K];
#pragma unroll
    for (int j = 0; j < PROF_K; ++j) a[j].hi = a[j].lo = 0.f;
    const int n = (y1 - y0) * g.nx;
    int dy = threadIdx.x / g.nx, x = threadIdx.x - dy * g.nx;
    const int step_y = blockDim.x / g.nx, step_x = blockDim.x - step_y * g.nx;
    for (int k = threadIdx.x; k < n; k += PROF_U * blockDim.x) {
        float d[PROF_U], v[PROF_U][3];
#pragma unroll
        for (int u = 0; u < PROF_U; ++u) {
            const bool in = k + u * (int)blockDim.x < n;
            const int p = in ? pidx(g, x, y0 + dy, z) : pidx(g, 0, y0, z);
            d[u] = __ldg(fl.dn + p);
            v[u][0] = __ldg(fl.ux + p);
            v[u][1] = __ldg(fl.uy + p);
            v[u][2] = __ldg(fl.uz + p);
            // next node of this thread: blockDim.x further in row-major order
            x += step_x;
            dy += step_y;
            if (x >= g.nx) {
                x -= g.nx;
                ++dy;
            }
        }
#pragma unroll
        for (int u = 0; u < PROF_U; ++u) {
            if (k + u * (int)blockDim.x >= n) break;
            pair_add(a[0], d[u]);
            pair_add(a[1], v[u][0]);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const float pr = d[u] * v[u][j];
                const float e = fmaf(d[u], v[u][j], -pr);
                pair_add(a[2 + j], v[u][j]);
                pair_add(a[2 + j], pr);
                pair_add(a[2 + j], e);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < PROF_K; ++j) sh[j][threadIdx.x] = (double)a[j].hi + (double)a[j].lo;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            for (int j = 0; j < PROF_K; ++j) sh[j][threadIdx.x] += sh[j][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x < PROF_K) part[((long long)z * chunks + c) * PROF_K + threadIdx.x] = sh[threadIdx.x][0];
}

__global__ void k_profiles_sum(const double* __restrict__ part, int nz, int chunks, double* __restrict__ prof)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= (long long)nz * PROF_K) return;
    const long long z = i / PROF_K, j = i - z * PROF_K;
    double s = 0.0;
    for (int c = 0; c < chunks; ++c) s += part[(z * chunks + c) * PROF_K + j];
    prof[i] = s;
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
cudaError_t launch_fill_outside(const Params& P, float* const* planes, const float* values,
                                int nplanes, cudaStream_t s)
{
    long long total = (long long)P.g.px * P.g.py * 2 * P.g.hw;
    if (P.g.zper || total == 0) return cudaSuccess;
    if (nplanes > 12) return cudaErrorInvalidValue;
    OutsidePlanes op;
    op.n = nplanes;
    for (int j = 0; j < nplanes; ++j) {
        op.p[j] = planes[j];
        op.v[j] = values[j];
    }
    k_fill_outside<<<nblocks(total, 256), 256, 0, s>>>(P, op);
    return cudaGetLastError();
}

cudaError_t launch_init_noise(const Params& P, float* dn, uint64_t seed, double amp, long long offset,
                              cudaStream_t s)
{
    k_init_noise<<<nblocks(P.g.N, 256), 256, 0, s>>>(P, dn, seed, amp, offset);
    return cudaGetLastError();
}

cudaError_t launch_init_profiles(const Params& P, float* const f[4], const float* n_z, const float* ux_z,
                                 int hmax, cudaStream_t s)
{
    k_init_profiles<<<nblocks(P.g.N, 256), 256, 0, s>>>(P, f[0], f[1], f[2], f[3], n_z, ux_z, hmax);
    return cudaGetLastError();
}

cudaError_t launch_init_fields(const Params& P, float* const f[4], const float* rho, const float* u,
                               cudaStream_t s)
{
    k_init_fields<<<nblocks(P.g.N, 256), 256, 0, s>>>(P, f[0], f[1], f[2], f[3], rho, u);
    return cudaGetLastError();
}

cudaError_t launch_tick(const Params& P, int4* clk, cudaStream_t s)
{
    return launch_step(k_tick, nblocks(P.nslits, 128), 128, 0, s, P, clk);
}

cudaError_t launch_pop_canon(const Params& P, void* pop, int i, void* canon, int to_pop, cudaStream_t s)
{
    if (P.storage == LBIF_STORE_F16)
        k_pop_canon<__half><<<nblocks(P.g.N, 256), 256, 0, s>>>(P, (__half*)pop, i, (__half*)canon, to_pop);
    else
        k_pop_canon<float><<<nblocks(P.g.N, 256), 256, 0, s>>>(P, (float*)pop, i, (float*)canon, to_pop);
    return cudaGetLastError();
}

cudaError_t launch_write_fields(const Params& P, const float* src, float* const f[4], cudaStream_t s)
{
    k_write_fields<<<nblocks(P.g.N, 256), 256, 0, s>>>(P, src, f[0], f[1], f[2], f[3]);
    return cudaGetLastError();
}

cudaError_t launch_read_fields(const Params& P, const float* const f[4], float* out, cudaStream_t s)
{
    k_read_fields<<<nblocks(P.g.N, 256), 256, 0, s>>>(P, f[0], f[1], f[2], f[3], out);
    return cudaGetLastError();
}

// z planes per CTA of the ball kernel: more CTAs fill the SMs, but each reads 2 R
// planes beyond its own. The length is the one that minimises
//   (planes + 2 R + 5) (1 + b k),  k = CTAs per SM,  b = 0.05 + 0.015 R^1.5,
// 5 standing for a CTA's start and b for what a co-resident CTA adds to the time of a
// plane (it grows with the radius as the row and disc sums take over from the
// latencies); up to five, CTAs per SM count whole. Over 26 grids (R 1 to 12, 2 to
// 512 tiles, 8 to 11,000 planes, every length timed) it lies within 9 % of the best
// length, 2 % on average. Microseconds with 1216 CTAs of at least 2 R planes (R or R / 2
// where those are few) / so: 203 x 117 x 75, sigma 10 55.6 / 45.6, sigma 24 196 / 151,
// 400 x 300 x 20, sigma 12 73.4 / 65.2, 128^3, sigma 18 107 / 94, 64 x 64 x 128, sigma 8
// 20.6 / 20.5, 256 x 256 x 128, sigma 8 90.4 / 92.1, 512 x 512 x 192, sigma 12 531 / 537.
int ball_chunk(const Geom& g, int sigma)
{
    const int R = sigma / 2;
    const double b = 0.05 + 0.015 * R * sqrt((double)R);
    const long long tiles = (long long)((g.nx + BALL_TX - 1) / BALL_TX) * ((g.ny + BALL_TY - 1) / BALL_TY);
    int best = g.nz;
    double cost = 1e300;
    // up to 16 CTAs per SM, at most 48 numbers of chunks
    long long most = 16LL * NUM_SMS / tiles;
    if (most > g.nz) most = g.nz;
    if (most < 1) most = 1;
    const long long tries = most < 48 ? most : 48;
    for (long long i = 1; i <= tries; ++i) {
        const int chunks = (int)(most * i / tries), z = (g.nz + chunks - 1) / chunks;
        const double q = (double)(tiles * ((g.nz + z - 1) / z)) / NUM_SMS;
        const double c = (z + 2 * R + 5) * (1.0 + b * (q <= 5.0 ? ceil(q) : q));
        if (c < cost) {
            cost = c;
            best = z;
        }
    }
    return best;
}

int ball_ctas(const Params& P)
{
    const Geom& g = P.g;
    return (g.nx + BALL_TX - 1) / BALL_TX * ((g.ny + BALL_TY - 1) / BALL_TY) * ((g.nz + P.ball_z - 1) / P.ball_z);
}

template <int R>
static cudaError_t ball_r(const Params& P, const float* dn, float* dG, int* status, int want,
                         int skip_done, const CUtensorMap* tmap, cudaStream_t s)
{
    const Geom& g = P.g;
    constexpr int H = BALL_TY + 2 * R, W = BALL_TX + 2 * ball_c4<R>();
    const size_t smem = tmap ? (size_t)2 * ((H * W * 4 + 127) / 128 * 128) + sizeof(float) * (R + 1) * H * BALL_TX + 16
                             : sizeof(float) * ball_smem_floats<R>();
    // the shared-memory limit is a per-device function attribute: set it
    // once per device that launches the kernel
    static std::atomic<uint64_t> configured{0}, configured_tma{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = 1ull << (dev & 63);
    std::atomic<uint64_t>& flags = tmap ? configured_tma : configured;
    if (!(flags.load() & bit)) {
        e = tmap ? cudaFuncSetAttribute(k_ball_tma<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)
                 : cudaFuncSetAttribute(k_ball<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        flags.fetch_or(bit);
    }
    int gx = (g.nx + BALL_TX - 1) / BALL_TX, gy = (g.ny + BALL_TY - 1) / BALL_TY;
    int zchunk = P.ball_z;
    if (want > 0) {
        // asked for: that many CTAs, of at least 2 R planes each (or the default's number)
        const long long tiles = (long long)gx * gy;
        const long long most = max(g.nz / (2 * R), (g.nz + zchunk - 1) / zchunk);
        const long long n = min((want + tiles - 1) / tiles, most);
        zchunk = (int)((g.nz + n - 1) / n);
    }
    const int nchunk = (g.nz + zchunk - 1) / zchunk;
    dim3 grid(gx, gy, nchunk);
    if (tmap)
        return launch_step(k_ball_tma<R>, grid, BALL_THREADS, smem, s, P, *tmap, dG, status, zchunk, skip_done);
    else
        return launch_step(k_ball<R>, grid, BALL_THREADS, smem, s, P, dn, dG, status, zchunk, skip_done);
}

void ball_box(int sigma, int* W, int* H)
{
    const int R = sigma / 2;
    *W = BALL_TX + 2 * ((R + 3) / 4 * 4);
    *H = BALL_TY + 2 * R;
}

cudaError_t launch_ball(const Params& P, const float* dn, float* dG, int* status, int want,
                        int skip_done, cudaStream_t s, const CUtensorMap* tmap)
{
    // direct sums below half a tile, and for the two smallest radii below a whole
    // tile row (20 x 200 x 150, sigma 4: tiles 18, direct 14 us; 128 slits of 32 x 32:
    // tiles 58, direct 72 us)
    if (P.g.nx < (P.sigma <= 4 ? BALL_TX : BALL_TX / 2) || P.g.ny < BALL_TY / 2) {
        // small blocks on small grids, so that the SMs share them; not for the loop over
        // large radii, whose blocks share their many rows in L1 (2 x 75 x 29, sigma 24: 64
        // threads 401 us, 256 threads 341; 3 x 70 x 12, sigma 12: 70 and 59)
        const int nt = P.g.N < 256LL * NUM_SMS && P.sigma <= 8 ? 64 : 256;
        const unsigned nb = nblocks(P.g.N, nt);
        switch (P.sigma / 2) {
        case 1: return launch_step(k_ball_direct<1>, nb, nt, 0, s, P, dn, dG, status, skip_done);
        case 2: return launch_step(k_ball_direct<2>, nb, nt, 0, s, P, dn, dG, status, skip_done);
        case 3: return launch_step(k_ball_direct<3>, nb, nt, 0, s, P, dn, dG, status, skip_done);
        case 4: return launch_step(k_ball_direct<4>, nb, nt, 0, s, P, dn, dG, status, skip_done);
        default: return launch_step(k_ball_direct<0>, nb, nt, 0, s, P, dn, dG, status, skip_done);
        }
    }
    switch (P.sigma / 2) {
    case 1: return ball_r<1>(P, dn, dG, status, want, skip_done, tmap, s);
    case 2: return ball_r<2>(P, dn, dG, status, want, skip_done, tmap, s);
    case 3: return ball_r<3>(P, dn, dG, status, want, skip_done, tmap, s);
    case 4: return ball_r<4>(P, dn, dG, status, want, skip_done, tmap, s);
    case 5: return ball_r<5>(P, dn, dG, status, want, skip_done, tmap, s);
    case 6: return ball_r<6>(P, dn, dG, status, want, skip_done, tmap, s);
    case 7: return ball_r<7>(P, dn, dG, status, want, skip_done, tmap, s);
    case 8: return ball_r<8>(P, dn, dG, status, want, skip_done, tmap, s);
    case 9: return ball_r<9>(P, dn, dG, status, want, skip_done, tmap, s);
    case 10: return ball_r<10>(P, dn, dG, status, want, skip_done, tmap, s);
    case 11: return ball_r<11>(P, dn, dG, status, want, skip_done, tmap, s);
    case 12: return ball_r<12>(P, dn, dG, status, want, skip_done, tmap, s);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_tail(const Params& P, const float* dn, const TailRow* rows, int nrows, const float4* coef,
                        float4* Ft, cudaStream_t s)
{
    const long long nb = (long long)((P.g.nx + 3) / 4) * P.g.ny * P.g.nz;
    k_tail<<<nblocks(nb, 32), 32 * TAIL_WARPS, 0, s>>>(P, dn, rows, nrows, coef, Ft);
    return cudaGetLastError();
}

// The rows' kernel pays per chunk of four dx (two thirds or less of it terms), the
// pairs' per pair, and needs more nodes to fill the chip the more pairs there are.
// Microseconds by rows / by pairs on 37 x 271 x 22 and 27 x 20 x 40: 3 pairs (3 chunks) 15.6 /
// 7.9 and 7.7 / 6.7, 15 (9) 19.3 / 10.2 and 8.0 / 8.5, 48 (15) 22.0 / 16.6 and 8.0 / 11.9,
// 132 (45) 37.3 / 35.8 and 11.7 / 22.4, but 115 (26) 28.4 / 31.4, 337 (81) 50.8 / 79.7.
bool tail_by_pairs(const Geom& g, int pairs, int chunks) { return 2 * pairs <= 7 * chunks && g.N >= 1500LL * pairs; }

cudaError_t launch_tail_pairs(const Params& P, const float* dn, const int* off, const float4* K, int npairs, float4* Ft,
                              cudaStream_t s)
{
    k_tail_pairs<<<nblocks(P.g.N, 256), 256, 0, s>>>(P, dn, off, K, npairs, Ft);
    return cudaGetLastError();
}

cudaError_t launch_wait_selftest(long long polls, int* status, cudaStream_t s)
{
    k_wait_selftest<<<1, 128, 0, s>>>(polls, status);
    return cudaGetLastError();
}

cudaError_t launch_force_soa(const Params& P, const float4* F, float* out, cudaStream_t s)
{
    k_force_soa<<<nblocks(P.g.N, 256), 256, 0, s>>>(P, F, out);
    return cudaGetLastError();
}

cudaError_t launch_moments_out(const Params& P, const Fields& f, float* rho, float* u, float* p,
                               cudaStream_t s)
{
    if (p && launch_pressure4(P, f, p, s)) p = nullptr;
    if (rho || u || p) k_moments_out<<<nblocks(P.g.N, 256), 256, 0, s>>>(P, f, rho, u, p);
    return cudaGetLastError();
}

// chunks per plane: enough CTAs to fill the GPU several times over
static int profile_chunks(const Geom& g)
{
    int c = (1216 + g.nz - 1) / g.nz;
    if (c > 32) c = 32;
    if (c > g.ny) c = g.ny;
    return c < 1 ? 1 : c;
}

size_t profile_doubles(const Geom& g) { return (size_t)PROF_K * g.nz * (1 + profile_chunks(g)); }

cudaError_t launch_profiles(const Params& P, const Fields& f, double* prof, cudaStream_t s)
{
    const int chunks = profile_chunks(P.g);
    double* part = prof + (size_t)PROF_K * P.g.nz;
    k_profiles<<<dim3(P.g.nz, chunks), 256, 0, s>>>(P, f, part, chunks);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_profiles_sum<<<nblocks((long long)P.g.nz * PROF_K, 256), 256, 0, s>>>(part, P.g.nz, chunks, prof);
    return cudaGetLastError();
}

}  // namespace lbif
