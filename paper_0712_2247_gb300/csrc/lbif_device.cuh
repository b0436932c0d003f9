// Device helpers shared by the kernel files: the D3Q19 set, typed population
// loads and stores, the padded-grid index maps, block -> node mappings, paired
// FP32 arithmetic and the bounded mbarrier wait.
#pragma once
#include <string.h>

#include "lbif_internal.h"

namespace lbif {

// D3Q19, antipodes in consecutive pairs (1,2), (3,4), ..., (17,18). The
// components are returned by switches so that, inside unrolled loops, every
// product with a lattice velocity folds to an add, a subtract or nothing.
__device__ __forceinline__ constexpr int kCx(int i)
{
    return (i == 1 || i == 7 || i == 9 || i == 11 || i == 13) ? 1
         : (i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1 : 0;
}
__device__ __forceinline__ constexpr int kCy(int i)
{
    return (i == 3 || i == 7 || i == 10 || i == 15 || i == 17) ? 1
         : (i == 4 || i == 8 || i == 9 || i == 16 || i == 18) ? -1 : 0;
}
__device__ __forceinline__ constexpr int kCz(int i)
{
    return (i == 5 || i == 11 || i == 14 || i == 15 || i == 18) ? 1
         : (i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1 : 0;
}
// |c_i|^2 (0, 1 or 2 on D3Q19)
__device__ __forceinline__ constexpr int kC2(int i) { return kCx(i) * kCx(i) + kCy(i) * kCy(i) + kCz(i) * kCz(i); }
__device__ __forceinline__ constexpr int opp_of(int i) { return i == 0 ? 0 : ((i & 1) ? i + 1 : i - 1); }

// Loads of what the step's kernels write (fields, forces, populations, clocks).
// Ordinary ones: a kernel under programmatic launch (step_begin) runs while its
// predecessor still writes them, where a read-only load (__ldg, or one that the
// compiler makes of a const __restrict__ argument) has no defined value. __ldg is
// for the tables that no kernel of a step writes.
__device__ __forceinline__ float ldp(const float* p) { return *p; }
__device__ __forceinline__ float ldp(const __half* p) { return __half2float(*p); }
// RAW: a 16-bit population is kept as its bits in the float's register and
// converted at its first use (late_cvt), so that no instruction waits on the
// gather before the work that is meant to hide its latency
template <bool RAW>
__device__ __forceinline__ float ldq(const float* p) { return ldp(p); }
template <bool RAW>
__device__ __forceinline__ float ldq(const __half* p)
{
    if constexpr (RAW)
        return __int_as_float((int)__half_as_ushort(*p));
    else
        return ldp(p);
}
__device__ __forceinline__ float late_cvt(float bits)
{
    return __half2float(__ushort_as_half((unsigned short)__float_as_int(bits)));
}
__device__ __forceinline__ void stp(float* p, float v) { *p = v; }
__device__ __forceinline__ void stp(__half* p, float v) { *p = __float2half_rn(v); }
// Four of them, in program order: the force kernel then keeps more of its windows'
// loads in flight than as the compiler orders plain ones (512 x 512 x 192, sigma 12 1.84 ->
// 1.76 ms; 203 x 117 x 75, sigma 6 88 -> 86 us; 256 x 256 x 128, sigma 8 291 -> 299 us).
// For data that the reading kernel does not write.
__device__ __forceinline__ float4 ld4(const float* p)
{
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ int pidx(const Geom& g, int x, int y, int z)
{
    return ((z + g.hw) * g.py + (y + g.hw)) * g.px + (x + g.hw);
}

__device__ __forceinline__ void decompose(const Geom& g, long long idx, int& x, int& y, int& z)
{
    int a = (int)(idx / g.nx);
    x = (int)(idx - (long long)a * g.nx);
    z = a / g.ny;
    y = a - z * g.ny;
}

// smallest periodic image x - k n that is >= -hw
__device__ __forceinline__ int img_start(int x, int n, int hw) { return x - ((x + hw) / n) * n; }

// Visit every padded index holding node (x, y, z): itself and its periodic
// images inside the halo (several on grids smaller than the halo).
template <class Fn>
__device__ __forceinline__ void for_images(const Geom& g, int x, int y, int z, Fn fn)
{
    int z0 = g.zper ? img_start(z, g.nz, g.hw) : z;
    int z1 = g.zper ? g.nz + g.hw : z + 1;
    int y0 = img_start(y, g.ny, g.hw);
    int x0 = img_start(x, g.nx, g.hw);
    for (int zi = z0; zi < z1; zi += g.nz)
        for (int yi = y0; yi < g.ny + g.hw; yi += g.ny)
            for (int xi = x0; xi < g.nx + g.hw; xi += g.nx)
                fn(((zi + g.hw) * g.py + (yi + g.hw)) * g.px + (xi + g.hw));
}

// node (x, y, z) lies at least hw from every periodic edge: its padded
// field value has no image in the halo
__device__ __forceinline__ bool no_images(const Geom& g, int x, int y, int z)
{
    return x >= g.hw && x < g.nx - g.hw && y >= g.hw && y < g.ny - g.hw &&
           (!g.zper || (z >= g.hw && z < g.nz - g.hw));
}

// Block -> node mapping of the stencil kernels: a CTA covers a TX x TY (x, y)
// tile of one z plane; CTAs are ordered tile-in-group fastest, then z, then
// group, where a group spans about 128 x 128 nodes. The CTAs resident at any
// moment then cover a compact 128 x 128 x ~20 block whose +-sigma stencil
// footprint stays in L2 instead of spanning 2 sigma + 1 full planes.
struct TileMap {
    int tx, ty, tiles_x, tiles_y, gtx, gty, ngx;
    int flat;  // 1: narrow grid, threads run over (x block, y, z) in order
};

__device__ __forceinline__ bool tile_origin(const Geom& g, const TileMap& tm, int& tile_x,
                                            int& tile_y, int& z)
{
    const int per = tm.gtx * tm.gty;
    const int b = blockIdx.x;
    const int tig = b % per;
    const int rest = b / per;
    z = rest % g.nz;
    const int grp = rest / g.nz;
    tile_x = (grp % tm.ngx) * tm.gtx + tig % tm.gtx;
    tile_y = (grp / tm.ngx) * tm.gty + tig / tm.gtx;
    return tile_x < tm.tiles_x && tile_y < tm.tiles_y;
}

static inline TileMap make_tilemap(const Geom& g, int tx, int ty, int group, unsigned& blocks)
{
    TileMap tm;
    tm.tx = tx;
    tm.ty = ty;
    tm.tiles_x = (g.nx + tx - 1) / tx;
    tm.tiles_y = (g.ny + ty - 1) / ty;
    int want_x = (group + tx - 1) / tx, want_y = (group + ty - 1) / ty;
    tm.gtx = tm.tiles_x < want_x ? tm.tiles_x : want_x;
    tm.gty = tm.tiles_y < want_y ? tm.tiles_y : want_y;
    tm.ngx = (tm.tiles_x + tm.gtx - 1) / tm.gtx;
    int ngy = (tm.tiles_y + tm.gty - 1) / tm.gty;
    blocks = (unsigned)tm.gtx * tm.gty * g.nz * tm.ngx * ngy;
    tm.flat = 0;
    return tm;
}

// narrow grids (nx below one tile row): one thread per block of xw x-nodes,
// consecutive threads over x blocks, then y, then z
static inline TileMap make_flatmap(const Geom& g, int xw, int threads, unsigned& blocks)
{
    TileMap tm;
    memset(&tm, 0, sizeof(tm));
    tm.flat = 1;
    tm.tx = (g.nx + xw - 1) / xw;  // x blocks per row
    long long n = (long long)tm.tx * g.ny * g.nz;
    blocks = (unsigned)((n + threads - 1) / threads);
    return tm;
}

__device__ __forceinline__ bool flat_node(const Geom& g, const TileMap& tm, int xw, int& x, int& y, int& z)
{
    long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    long long rows = (long long)g.ny * g.nz;
    if (k >= rows * tm.tx) return false;
    int xb = (int)(k % tm.tx);
    long long r = k / tm.tx;
    y = (int)(r % g.ny);
    z = (int)(r / g.ny);
    x = xb * xw;
    return true;
}

// slit of plane z (-1 for a gap plane between stacked slits)
__device__ __forceinline__ int slit_of(const Params& P, int z) { return __ldg(P.zslit + z); }
__device__ __forceinline__ bool frozen(const Params& P, int s) { return __ldg(P.done + s) != 0; }

__host__ __device__ constexpr int cisqrt(int n)
{
    int w = 0;
    while ((w + 1) * (w + 1) <= n) ++w;
    return w;
}

// paired FP32 arithmetic: one instruction on two values (fma / add / mul
// .f32x2, sm_100 and later); each component rounds as the scalar operation
__device__ __forceinline__ float2 bc2(float s) { return make_float2(s, s); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
// a - b, rounded once (b (-1) is exact)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, bc2(-1.f), a); }

__device__ __forceinline__ float shell_A(float dq, float gq, float G0) { return G0 * dq + gq * (1.f + dq); }

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool mbar_wait_parity(uint64_t* mbar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_addr(mbar)), "r"(parity)
        : "memory");
    return ok != 0;
}

constexpr long long BALL_WAIT_LIMIT = 1LL << 22;  // try_wait polls; seconds at most

// ---- populations in place ---------------------------------------------
// One buffer. Direction i of node (x, y, z) of slit s, in the slit's step t,
// sits at storage node
//   ((zb + (z - zlo - t c_iz) mod R) ny + (y - t c_iy) mod ny) nx + (x - t c_ix) mod nx,
// R = the slit's planes plus one ghost plane beyond its walls (none with
// periodic z). The slot a node's pull reads for direction i (its source
// r - c_i at step t) is then the slot it writes (itself at step t + 1); a
// bounce-back reads the node's own slot of the opposite direction at step t,
// which no other node reads or writes in that step, and writes a slot that
// belongs to a ghost-plane node at step t (read by nobody). Every slot is
// therefore read and written by one thread per step. The slit's clock holds
// t mod (nx, ny, R) and advances after every pull pass (not while the slit
// is frozen, so a frozen slit's slots stay where they are).
__device__ __forceinline__ int wrap_lo(int a, int n) { return a < 0 ? a + n : a; }   // a in [-n, n)
__device__ __forceinline__ int wrap_hi(int a, int n) { return a >= n ? a - n : a; }  // a in [0, 2n)

struct IpSlots {
    int x, xm, xp, y, ym, yp, zr, zm, zp;  // the node's coordinates and c_a = +1 (m) / -1 (p) shifted by t + 1
    int tx, ty, tz;                        // t mod (nx, ny, R)
    int zb, R, nx, ny;
    // the slot of direction i of the node at step t + 1 (= of its source at step t)
    __device__ __forceinline__ int slot(int i) const
    {
        const int cx = kCx(i), cy = kCy(i), cz = kCz(i);
        const int xx = cx > 0 ? xm : (cx < 0 ? xp : x);
        const int yy = cy > 0 ? ym : (cy < 0 ? yp : y);
        const int zz = cz > 0 ? zm : (cz < 0 ? zp : zr);
        return ((zb + zz) * ny + yy) * nx + xx;
    }
    // the slot of the node's own direction opp(i) at step t (bounce-back of i)
    __device__ __forceinline__ int wall_slot(int i) const
    {
        const int cx = kCx(i), cy = kCy(i), cz = kCz(i);
        const int xx = cx > 0 ? wrap_hi(x + tx, nx) : (cx < 0 ? wrap_lo(x - tx, nx) : x);
        const int yy = cy > 0 ? wrap_hi(y + ty, ny) : (cy < 0 ? wrap_lo(y - ty, ny) : y);
        const int zz = cz > 0 ? wrap_hi(zr + tz, R) : (cz < 0 ? wrap_lo(zr - tz, R) : zr);
        return ((zb + zz) * ny + yy) * nx + xx;
    }
};

__device__ __forceinline__ IpSlots ip_slots(const Params& P, const SlitParam& S, int s, int x, int y, int z)
{
    const int4 c = P.clk[s];
    IpSlots q;
    q.nx = P.g.nx;
    q.ny = P.g.ny;
    q.zb = S.zb;
    q.R = S.R;
    q.tx = c.x;
    q.ty = c.y;
    q.tz = c.z;
    const int sx = wrap_hi(c.x + 1, q.nx), sy = wrap_hi(c.y + 1, q.ny), sz = wrap_hi(c.z + 1, q.R);
    q.x = x;
    q.xm = wrap_lo(x - sx, q.nx);
    q.xp = wrap_hi(x + sx, q.nx);
    q.y = y;
    q.ym = wrap_lo(y - sy, q.ny);
    q.yp = wrap_hi(y + sy, q.ny);
    q.zr = z - S.zlo;
    q.zm = wrap_lo(q.zr - sz, q.R);
    q.zp = wrap_hi(q.zr + sz, q.R);
    return q;
}

// Programmatic dependent launch of the step's kernels: on a small grid a step is
// mostly launch latency, which is hidden when each kernel comes onto the SMs while
// its predecessor still runs. Every thread of such a kernel calls step_begin()
// first: it waits for the predecessor's end (and so, every kernel of the chain
// doing the same, for all earlier work) before it reads or writes anything, then
// lets the successor come up. What it reads of its predecessors goes through
// ordinary loads (ldp).
//
// P.overlap says whether the attribute is given (step_overlap).
__device__ __forceinline__ void step_begin(const Params& P)
{
    if (!P.overlap) return;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... K, class... A>
static inline cudaError_t launch_step(void (*kernel)(Params, K...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                                      const Params& P, A... args)
{
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = P.overlap ? 1 : 0;
    return cudaLaunchKernelEx(&c, kernel, P, static_cast<K>(args)...);
}

static inline unsigned nblocks(long long n, int bs) { return (unsigned)((n + bs - 1) / bs); }

}  // namespace lbif
