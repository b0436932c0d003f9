// The pull pass: collision, streaming and the next step's moments in one pass
// over the populations, with its launchers.
#include <atomic>
#include <utility>

#include "lbif_device.cuh"

namespace lbif {

// ---------------------------------------------------------------------------
// steps 5-6 with step 1 of the next step, in pull form (Sec. Methods: the
// forward-Euler update with the first-order source towards the local
// equilibrium; half-way bounce-back at the walls). Every node gathers the
// populations that stream into it, applies to each the collision of its
// source node, and forms the new moments from the 19 values it holds, so the
// populations are read and written once per step.
//
// Stored populations. A node's populations are kept as
//   h_i = s_T (f_i - f_i^eq(n, u)) / (w_i n),
// the non-equilibrium part of f_i relative to the node's equilibrium weight
// w_i n, at the moments n, u of the step they belong to (the field buffers of
// that step hold those moments in FP32); s_T = 2^8 with FP16 storage (keeps
// the small parts of the bulk clear of the FP16 subnormal range) and 1 with
// FP32. The equilibrium part, which carries the flow, is never rounded to the
// storage type. In units of w_i n0, with dn = n/n0 - 1 and
// e_i = (1 + dn)(3 c.u + 9/2 (c.u)^2 - 3/2 u.u),
//   f_i / (w_i n0) - 1 = dn + e_i + (1 + dn) h_i / s_T.
// BGK towards f^eq(n, u) with omega = 1/tau, plus the source
// 3 c.F + (3/2) F.w (|c|^2 - 1) (F the force per n0, F.w the energy source
// when on), gives the post-collision value
//   f_i' / (w_i n0) - 1 = dn + T_i + m h_i,  m = (1 - omega)(1 + dn) / s_T,
//   T_i = e_i + 3 c.F + (3/2) F.w (|c|^2 - 1),
// and T splits by lattice-velocity class into
//   axis a, sign s:            s P_a + C_a
//   plane (a, b), signs sa sb: sa P_a + sb P_b + C_ab + sa sb X_ab
//   rest:                      C_0
// with q = 1 + dn, P = 3 (q u + F), B = -(3/2) q u.u, C_a = B + (9/2) q u_a^2,
// C_ab = B + (9/2) q (u_a^2 + u_b^2) + (3/2) F.w, X_ab = 9 q u_a u_b and
// C_0 = B - (3/2) F.w = (2 (C_x + C_y + C_z) - (C_xy + C_xz + C_yz)) / 3.
// The value reaching r from s = r - c_i, relative to dn(r), is
// v_i = T_i(s) + m(s) h_i(s) + (dn(s) - dn(r)); at a wall it is the node's own
// post-collision value of the opposite direction (c -> -c: the P terms change
// sign). The new moments are dn(r) + S, S = sum_i w_i v_i, and
// u = sum_i w_i c_i v_i / (1 + dn(r) + S); the new populations are stored as
// their non-equilibrium parts at those moments.
// ---------------------------------------------------------------------------
template <typename T>
__host__ __device__ constexpr float store_scale() { return sizeof(T) == 2 ? 256.f : 1.f; }

// staged quantities of a node: dn, P_x..z, C_x..z, C_xy C_xz C_yz, X_xy X_xz X_yz
constexpr int SQ_DN = 0, SQ_P = 1, SQ_CA = 4, SQ_CP = 7, SQ_X = 10, CSM_NF = 13;

// The staged quantities of a node from its moments and force; st(k, value)
// receives quantity k. Each quantity ends in a rounding intrinsic (never
// merged into a later multiply-add), so a kernel that uses them at once and
// one that stores them first compute identical values.
//
// shifted (velocity-shifted second-order forcing, the force F from the
// unshifted moments): BGK towards f^eq(n, u') with u' = u + F/(2 q), and the
// source k [3 (c - u').F + 9 (c.u')(c.F)], k = 1 - omega/2. T_i is then
// (1 - omega) e_i(u) + omega e_i(u') + that source, whose class split, with
// T = alpha + beta.c + c.gamma.c, is P_a = beta_a, C_a = alpha + gamma_aa,
// C_ab = alpha + gamma_aa + gamma_bb, X_ab = 2 gamma_ab:
//   alpha   = -(3/2) q ((1 - omega) u.u + omega u'.u') - 3 k u'.F
//   beta_a  = 3 q ((1 - omega) u_a + omega u'_a) + 3 k F_a
//   gamma_ab = (9/2) q ((1 - omega) u_a u_b + omega u'_a u'_b) + (9/2) k (u'_a F_b + u'_b F_a).
template <class St>
__device__ __forceinline__ void src_terms(float d, float ux, float uy, float uz, float4 f, float om, bool shifted,
                                          St st)
{
    const float q1 = 1.f + d;
    st(SQ_DN, d);
    if (shifted) {
        const float hq = 0.5f / q1;
        const float vx = fmaf(hq, f.x, ux), vy = fmaf(hq, f.y, uy), vz = fmaf(hq, f.z, uz);  // u'
        const float k = fmaf(-0.5f, om, 1.f), a1 = 1.f - om;
        const float uu = ux * ux + uy * uy + uz * uz, vv = vx * vx + vy * vy + vz * vz;
        const float vF = vx * f.x + vy * f.y + vz * f.z;
        const float alpha = fmaf(-1.5f * q1, fmaf(a1, uu, om * vv), -3.f * k * vF);
        const float u[3] = {ux, uy, uz}, v[3] = {vx, vy, vz}, F[3] = {f.x, f.y, f.z};
        auto gam = [&](int a, int b) {
            return fmaf(4.5f * q1, fmaf(a1, u[a] * u[b], om * (v[a] * v[b])), 4.5f * k * fmaf(v[a], F[b], v[b] * F[a]));
        };
        const float gxx = gam(0, 0), gyy = gam(1, 1), gzz = gam(2, 2);
#pragma unroll
        for (int a = 0; a < 3; ++a)
            st(SQ_P + a, __fmul_rn(3.f, fmaf(q1, fmaf(a1, u[a], om * v[a]), k * F[a])));
        st(SQ_CA + 0, __fadd_rn(alpha, gxx));
        st(SQ_CA + 1, __fadd_rn(alpha, gyy));
        st(SQ_CA + 2, __fadd_rn(alpha, gzz));
        st(SQ_CP + 0, __fadd_rn(alpha, gxx + gyy));
        st(SQ_CP + 1, __fadd_rn(alpha, gxx + gzz));
        st(SQ_CP + 2, __fadd_rn(alpha, gyy + gzz));
        st(SQ_X + 0, __fmul_rn(2.f, gam(0, 1)));
        st(SQ_X + 1, __fmul_rn(2.f, gam(0, 2)));
        st(SQ_X + 2, __fmul_rn(2.f, gam(1, 2)));
        return;
    }
    const float B = __fmul_rn(-1.5f * q1, ux * ux + uy * uy + uz * uz);
    const float a = 4.5f * q1, ax = a * ux * ux, ay = a * uy * uy, az = a * uz * uz;
    const float fw = 1.5f * f.w, b = 9.f * q1;
    st(SQ_P + 0, __fmul_rn(3.f, fmaf(q1, ux, f.x)));
    st(SQ_P + 1, __fmul_rn(3.f, fmaf(q1, uy, f.y)));
    st(SQ_P + 2, __fmul_rn(3.f, fmaf(q1, uz, f.z)));
    st(SQ_CA + 0, __fadd_rn(B, ax));
    st(SQ_CA + 1, __fadd_rn(B, ay));
    st(SQ_CA + 2, __fadd_rn(B, az));
    st(SQ_CP + 0, __fadd_rn(B + (ax + ay), fw));
    st(SQ_CP + 1, __fadd_rn(B + (ax + az), fw));
    st(SQ_CP + 2, __fadd_rn(B + (ay + az), fw));
    st(SQ_X + 0, __fmul_rn(b * ux, uy));
    st(SQ_X + 1, __fmul_rn(b * ux, uz));
    st(SQ_X + 2, __fmul_rn(b * uy, uz));
}

// v_i (see above) from the source's staged quantities sl (quantity k at
// sl[k * ST]) and its stored h; wall: sl is the node itself and the
// direction arrives reversed
template <int i, int ST>
__device__ __forceinline__ float arrive(const float* sl, float h, float om1s, float dnr, bool wall)
{
    constexpr int cx = kCx(i), cy = kCy(i), cz = kCz(i);
    const float sg = wall ? -1.f : 1.f;
    float t;
    if constexpr (i == 0) {
        t = (2.f * (sl[(SQ_CA + 0) * ST] + sl[(SQ_CA + 1) * ST] + sl[(SQ_CA + 2) * ST]) -
             (sl[(SQ_CP + 0) * ST] + sl[(SQ_CP + 1) * ST] + sl[(SQ_CP + 2) * ST])) *
            (1.f / 3.f);
    } else if constexpr (kC2(i) == 1) {
        constexpr int a = cx ? 0 : (cy ? 1 : 2);
        constexpr float ca = (float)(cx + cy + cz);
        t = fmaf(sg * ca, sl[(SQ_P + a) * ST], sl[(SQ_CA + a) * ST]);
    } else {
        constexpr int pl = cz == 0 ? 0 : (cy == 0 ? 1 : 2);
        constexpr int a = pl == 2 ? 1 : 0, b = pl == 0 ? 1 : 2;
        constexpr float ca = (float)(a == 0 ? cx : cy), cb = (float)(b == 1 ? cy : cz);
        t = sl[(SQ_CP + pl) * ST] + sg * (ca * sl[(SQ_P + a) * ST] + cb * sl[(SQ_P + b) * ST]) +
            (ca * cb) * sl[(SQ_X + pl) * ST];
    }
    const float ds = sl[SQ_DN * ST];
    return fmaf(fmaf(om1s, ds, om1s), h, t) + (ds - dnr);
}

// fn(std::integral_constant<int, i>) for i = 0 .. Q-1, unrolled at compile time
template <class Fn, int... I>
__device__ __forceinline__ void for_dirs_seq(Fn&& fn, std::integer_sequence<int, I...>)
{
    (fn(std::integral_constant<int, I>{}), ...);
}
template <class Fn>
__device__ __forceinline__ void for_dirs(Fn&& fn)
{
    for_dirs_seq(fn, std::make_integer_sequence<int, Q>{});
}

// Mirror pairs. The flow along x and y is a small signal next to the
// wall-normal velocity and force (u_z and F_z of O(0.1) where u_x ~ 1e-4), so
// the arriving values of directions that differ only in the sign of c_x (or
// c_y) share large parts. Their difference is therefore formed from the
// differences of the staged quantities of their two sources (which lie in
// the same plane, two nodes apart), and the x and y momenta are sums of those
// differences: a sum of separately rounded values of O(1) would carry the
// signal only to ~1e-7 of those values. Ten pairs (plus member first):
//   along x: (1,2) (7,10) (9,8) (11,14) (13,12); along y: (3,4) (7,9) (10,8) (15,18) (17,16).
// Directions 1 3 7 9 10 11 13 15 17 are derived: slot i holds v_i - v_b of
// its pair partner b (7 from 10, 10 from 8), the others ("base") hold v_i.
template <int i, int ip>
struct Mirror {
    static constexpr int A = kCx(i) != kCx(ip) ? 0 : 1;  // the component that changes sign
    static constexpr bool axis = kC2(i) == 1;
    // the shared nonzero component of a plane direction and its sign
    static constexpr int B = axis ? 0 : (A == 0 ? (kCy(i) != 0 ? 1 : 2) : (kCx(i) != 0 ? 0 : 2));
    static constexpr int PL = (A == 2 || B == 2) ? (A == 0 || B == 0 ? 1 : 2) : 0;
    static constexpr float CB = axis ? 0.f : (float)(B == 0 ? kCx(i) : (B == 1 ? kCy(i) : kCz(i)));
};

// v_i - v_ip of a mirror pair (staged quantities of the sources at s and sp,
// stride ST; the stored values h, hp of the two directions; wall: both
// arrive reversed from the node itself, s = sp)
template <int i, int ip, int ST>
__device__ __forceinline__ float mirror_diff(const float* s, const float* sp, float h, float hp, float om1s, bool wall)
{
    using M = Mirror<i, ip>;
    const float sg = wall ? -1.f : 1.f;
    float dt;
    if constexpr (M::axis) {
        dt = (s[(SQ_CA + M::A) * ST] - sp[(SQ_CA + M::A) * ST]) + sg * (s[(SQ_P + M::A) * ST] + sp[(SQ_P + M::A) * ST]);
    } else {
        dt = (s[(SQ_CP + M::PL) * ST] - sp[(SQ_CP + M::PL) * ST]) +
             sg * (s[(SQ_P + M::A) * ST] + sp[(SQ_P + M::A) * ST]) +
             (sg * M::CB) * (s[(SQ_P + M::B) * ST] - sp[(SQ_P + M::B) * ST]) +
             M::CB * (s[(SQ_X + M::PL) * ST] + sp[(SQ_X + M::PL) * ST]);
    }
    const float ds = s[SQ_DN * ST], dsp = sp[SQ_DN * ST];
    // m(s) h - m(sp) hp with m = om1s (1 + d)
    const float dm = om1s * fmaf(1.f + ds, h - hp, (ds - dsp) * hp);
    return (dt + dm) + (ds - dsp);
}

// element off of direction i's part of a population buffer
template <typename T>
__device__ __forceinline__ T* pop_at(T* p, const Params& P, int i, long long off)
{
    return p + (P.dbase[i] + off);
}
// the same in place, where every element offset fits 32 bits: one 32-bit add
// and one widening multiply-add per address
template <typename T>
__device__ __forceinline__ T* pop_at_ip(T* p, const Params& P, int i, int slot)
{
    return p + (P.dbase32[i] + (unsigned)slot);
}

// the new moments of a node from its arriving values (slots as above, d79 =
// v_7 - v_9), then its populations stored as non-equilibrium parts at those
// moments (at(i): where direction i goes): base directions directly, derived
// ones as their partner's stored value plus the difference (so the pairs'
// differences survive the rounding of the large common parts); returns dn
// and writes u
template <typename T, class Addr>
__device__ __forceinline__ float pull_finish(Addr at, const float* v, float d79, float dnr, float& ux, float& uy,
                                             float& uz)
{
    constexpr float w1 = 1.f / 18.f, w2 = 1.f / 36.f;
    // arriving values of the derived directions
    const float v1 = v[2] + v[1], v3 = v[4] + v[3], v9 = v[8] + v[9], v10 = v[8] + v[10];
    const float v7 = v10 + v[7], v11 = v[14] + v[11], v13 = v[12] + v[13], v15 = v[18] + v[15];
    const float v17 = v[16] + v[17];
    const float S = (1.f / 3.f) * v[0] +
                    w1 * (((v1 + v[2]) + (v3 + v[4])) + (v[5] + v[6])) +
                    w2 * ((((v7 + v[8]) + (v9 + v10)) + ((v11 + v[12]) + (v13 + v[14]))) +
                          ((v15 + v[16]) + (v17 + v[18])));
    const float Jz = w1 * (v[5] - v[6]) +
                     w2 * (((v11 - v[12]) - (v13 - v[14])) + ((v15 - v[16]) - (v17 - v[18])));
    const float Jx = w1 * v[1] + w2 * (((v[7] + v[9]) + (v[11] + v[13])));
    const float Jy = w1 * v[3] + w2 * ((d79 + v[10]) + (v[15] + v[17]));
    const float dn = dnr + S;
    const float inv = 1.f / (1.f + dn);
    ux = Jx * inv;
    uy = Jy * inv;
    uz = Jz * inv;
    const float uu = ux * ux + uy * uy + uz * uz;
    constexpr float sT = store_scale<T>();
    auto p_of = [&](int i) {  // f_i^eq / (w_i n) - 1
        const float cu = dot_c(i, ux, uy, uz);
        return fmaf(cu, fmaf(4.5f, cu, 3.f), -1.5f * uu);
    };
    auto base = [&](int i, float vi) { return (vi - S) * inv - p_of(i); };
    // p_i - p_ip of a pair that differs in component a: u_a (6 + 18 R),
    // R = the shared part of c.u
    auto dp = [&](float ua, float R) { return ua * fmaf(18.f, R, 6.f); };
    auto put = [&](int i, float h) { stp(at(i), sT * h); };
    put(0, base(0, v[0]));
    put(5, base(5, v[5]));
    put(6, base(6, v[6]));
    const float h2 = base(2, v[2]), h4 = base(4, v[4]), h8 = base(8, v[8]);
    put(2, h2);
    put(1, h2 + (v[1] * inv - dp(ux, 0.f)));
    put(4, h4);
    put(3, h4 + (v[3] * inv - dp(uy, 0.f)));
    put(8, h8);
    put(9, h8 + (v[9] * inv - dp(ux, -uy)));
    const float h10 = h8 + (v[10] * inv - dp(uy, -ux));
    put(10, h10);
    put(7, h10 + (v[7] * inv - dp(ux, uy)));
    const float h12 = base(12, v[12]), h14 = base(14, v[14]);
    put(12, h12);
    put(13, h12 + (v[13] * inv - dp(ux, -uz)));
    put(14, h14);
    put(11, h14 + (v[11] * inv - dp(ux, uz)));
    const float h16 = base(16, v[16]), h18 = base(18, v[18]);
    put(16, h16);
    put(17, h16 + (v[17] * inv - dp(uy, -uz)));
    put(18, h18);
    put(15, h18 + (v[15] * inv - dp(uy, uz)));
    return dn;
}

// moments of a node written to the next step's fields (with their images)
__device__ __forceinline__ void put_fields(const Params& P, const CsmIO& io, int x, int y, int z, float dn, float ux,
                                           float uy, float uz, int* status)
{
    if (!(1.f + dn > 0.f) || !isfinite(dn) || !isfinite(ux + uy + uz)) atomicOr(status, 1);
    auto put = [&](int p) {
        io.dnw[p] = dn;
        io.uxw[p] = ux;
        io.uyw[p] = uy;
        io.uzw[p] = uz;
    };
    if (no_images(P.g, x, y, z))
        put(pidx(P.g, x, y, z));
    else
        for_images(P.g, x, y, z, put);
}

// What a source node contributes is staged per node in shared memory: a CTA
// owns a 32 x 4 tile of x-y nodes, keeps three planes of it (plus a one-node
// halo) in a ring, and marches up a segment of z planes.
// 32 x 4 tiles of 128 threads, six CTAs per SM (measured at 512 x 512 x 192, sigma 12, same
// state: 32 x 4 / 128 threads / 6 CTAs 2.186 ms, 32 x 8 / 256 / 3 2.334 ms, 32 x 12 / 384 / 2
// 2.508 ms): more, smaller CTAs keep more population loads in flight across the two barriers
// of each plane
constexpr int CSM_TX = 32, CSM_TY = 4, CSM_THREADS = CSM_TX * CSM_TY;
constexpr int CSM_HX = CSM_TX + 2, CSM_HN = CSM_HX * (CSM_TY + 2);  // staged nodes per plane
constexpr int CSM_SLOT = CSM_NF * CSM_HN;  // floats per staged plane
size_t csm_smem_bytes() { return sizeof(float) * 3 * CSM_SLOT; }

__device__ __forceinline__ int csm_slot(int q) { return (q + 3) % 3; }

// The halo nodes a thread stages in every plane (NT threads: h = thread,
// thread + NT, ...; at most two): their in-plane padded offset (x, y halo
// images hold the periodic values) and the in-plane index of their periodic
// image in the unpadded force array, or -1 (past the last halo node or a partial
// tile: never gathered).
constexpr int CSM_KS = 2;
struct CsmStaged {
    int p[CSM_KS], n[CSM_KS];
};

template <int NT>
__device__ __forceinline__ CsmStaged csm_staged(const Geom& g, int x0, int y0)
{
    static_assert(NT * CSM_KS >= CSM_HN, "two staged nodes per thread at most");
    CsmStaged st;
#pragma unroll
    for (int k = 0; k < CSM_KS; ++k) {
        const int h = threadIdx.x + k * NT;
        const int X = x0 - 1 + h % CSM_HX, Y = y0 - 1 + h / CSM_HX;
        st.p[k] = st.n[k] = -1;
        if (h >= CSM_HN || X > g.nx || Y > g.ny) continue;
        const int xw = X < 0 ? X + g.nx : (X >= g.nx ? X - g.nx : X);
        const int yw = Y < 0 ? Y + g.ny : (Y >= g.ny ? Y - g.ny : Y);
        st.p[k] = (Y + g.hw) * g.px + (X + g.hw);
        st.n[k] = yw * g.nx + xw;
    }
    return st;
}

// stage plane q (-1 <= q <= nz) of the tile into `slot`
template <int NT>
__device__ __forceinline__ void csm_stage(const Params& P, const CsmIO& io, const float4* __restrict__ F,
                                          float* slot, const CsmStaged& st, int q)
{
    const Geom& g = P.g;
    int zq = q;
    if (g.zper)
        zq = q < 0 ? q + g.nz : (q >= g.nz ? q - g.nz : q);
    else if (q < 0 || q >= g.nz)
        return;  // beyond the walls: only reached through bounce-back
    const int sq = slit_of(P, zq);
    if (sq < 0 || frozen(P, sq)) return;
    const int pq = (q + g.hw) * g.py * g.px;
    const float4* Fq = F + (long long)zq * g.ny * g.nx;
    const float om = P.sl[sq].inv_tau;
    const bool shifted = P.shifted != 0;
#pragma unroll
    for (int k = 0; k < CSM_KS; ++k) {
        if (k * NT >= CSM_HN || st.p[k] < 0) continue;
        const int h = threadIdx.x + k * NT;
        const int p = pq + st.p[k];
        src_terms(__ldg(io.dn + p), __ldg(io.ux + p), __ldg(io.uy + p), __ldg(io.uz + p), __ldg(Fq + st.n[k]), om,
                  shifted, [&](int j, float val) { slot[j * CSM_HN + h] = val; });
    }
}

// CTAs per SM the register budget is sized for (5 / 6 / 7 at 96 / 80 / 72
// registers: 2.57 / 2.39 / 2.55 ms at 512 x 512 x 192, sigma 12, FP32), and
// z planes per CTA segment
#ifndef CSM_MINB
#define CSM_MINB 6
#endif
#ifndef CSM_LZ
#define CSM_LZ 16
#endif

// the stored populations of directions [I0, I1) that stream into node
// (x, y, z): v[i - I0]; bit i of bb marks a direction that arrives from a
// wall (bounce-back: the node's own opposite population). IP: in place
// (slots from q, see above).
template <int I0, int I1, bool IP, typename T, bool RAW = false>
__device__ __forceinline__ void csm_pull(const Params& P, const T* __restrict__ pin, long long idx, int x, int y,
                                         int z, int zlo, int zhi, float* v, unsigned& bb, const IpSlots& q)
{
    const Geom& g = P.g;
    if constexpr (IP) {
#pragma unroll
        for (int i = I0; i < I1; ++i) {
            const int sz = z - kCz(i);
            if (!g.zper && (sz < zlo || sz > zhi)) {
                bb |= 1u << i;
                v[i - I0] = ldq<RAW>(pop_at_ip(pin, P, opp_of(i), q.wall_slot(i)));
            } else {
                v[i - I0] = ldq<RAW>(pop_at_ip(pin, P, i, q.slot(i)));
            }
        }
        return;
    }
    if (x > 0 && x < g.nx - 1 && y > 0 && y < g.ny - 1 && z > zlo && z < zhi) {
#pragma unroll
        for (int i = I0; i < I1; ++i) v[i - I0] = ldq<RAW>(pin + (idx + P.doff[i]));
        return;
    }
#pragma unroll
    for (int i = I0; i < I1; ++i) {
        int sx = x - kCx(i), sy = y - kCy(i), sz = z - kCz(i);
        sx = sx < 0 ? sx + g.nx : (sx >= g.nx ? sx - g.nx : sx);
        sy = sy < 0 ? sy + g.ny : (sy >= g.ny ? sy - g.ny : sy);
        if (g.zper) {
            sz = sz < 0 ? sz + g.nz : (sz >= g.nz ? sz - g.nz : sz);
        } else if (sz < zlo || sz > zhi) {
            bb |= 1u << i;
            v[i - I0] = ldq<RAW>(pin + (P.dbase[opp_of(i)] + idx));
            continue;
        }
        v[i - I0] = ldq<RAW>(pin + (P.dbase[i] + (((long long)sz * g.ny + sy) * g.nx + sx)));
    }
}

// The arriving values of a node in the slots described at Mirror: the ten
// mirror differences first (from the stored values as loaded), then the ten
// base directions. src(i) is the source quantities of direction i (stride
// ST); wall directions arrive reversed from the node itself (own).
template <int ST, bool WALLS, class Src>
__device__ __forceinline__ void pull_gather_impl(Src src, const float* own, float om1s, float dnr, unsigned bb,
                                                 float* v, float& d79)
{
    auto wall = [&](int i) { return WALLS && ((bb >> i) & 1u) != 0u; };
    auto diff = [&](auto ic, auto ipc) {
        constexpr int i = decltype(ic)::value, ip = decltype(ipc)::value;
        const bool w = wall(i);
        return mirror_diff<i, ip, ST>(w ? own : src(ic), w ? own : src(ipc), v[i], v[ip], om1s, w);
    };
    using std::integral_constant;
    const float d7_10 = diff(integral_constant<int, 7>{}, integral_constant<int, 10>{});
    const float d9_8 = diff(integral_constant<int, 9>{}, integral_constant<int, 8>{});
    const float d10_8 = diff(integral_constant<int, 10>{}, integral_constant<int, 8>{});
    d79 = diff(integral_constant<int, 7>{}, integral_constant<int, 9>{});
    v[7] = d7_10;
    v[9] = d9_8;
    v[10] = d10_8;
    v[1] = diff(integral_constant<int, 1>{}, integral_constant<int, 2>{});
    v[3] = diff(integral_constant<int, 3>{}, integral_constant<int, 4>{});
    v[11] = diff(integral_constant<int, 11>{}, integral_constant<int, 14>{});
    v[13] = diff(integral_constant<int, 13>{}, integral_constant<int, 12>{});
    v[15] = diff(integral_constant<int, 15>{}, integral_constant<int, 18>{});
    v[17] = diff(integral_constant<int, 17>{}, integral_constant<int, 16>{});
    auto one = [&](auto ic) {
        constexpr int i = decltype(ic)::value;
        if constexpr (i == 0 || i == 2 || i == 4 || i == 5 || i == 6 || i == 8 || i == 12 || i == 14 || i == 16 ||
                      i == 18) {
            const bool w = i != 0 && wall(i);
            v[i] = arrive<i, ST>((i == 0 || w) ? own : src(ic), v[i], om1s, dnr, w);
        }
    };
    for_dirs(one);
}

// The arriving values of a node in the slots described at Mirror: the ten
// mirror differences first (from the stored values as loaded), then the ten
// base directions. src(i) is the source quantities of direction i (stride
// ST); wall directions arrive reversed from the node itself (own). Nodes
// with no wall direction (bb = 0, almost all) take a path without the wall
// selections.
template <int ST, class Src>
__device__ __forceinline__ void pull_gather(Src src, const float* own, float om1s, float dnr, unsigned bb, float* v,
                                            float& d79)
{
    if (bb == 0u)
        pull_gather_impl<ST, false>(src, own, om1s, dnr, bb, v, d79);
    else
        pull_gather_impl<ST, true>(src, own, om1s, dnr, bb, v, d79);
}

// the gather of a node staged at hc in the ring (planes below, own, above)
__device__ __forceinline__ void csm_collide(const float* own, const float* below, const float* above, int hc,
                                            float om1s, float dnr, unsigned bb, float* v, float& d79)
{
    auto src = [&](auto ic) -> const float* {
        constexpr int i = decltype(ic)::value;
        constexpr int cx = kCx(i), cy = kCy(i), cz = kCz(i);
        return (cz > 0 ? below : (cz < 0 ? above : own)) + hc - cx - cy * CSM_HX;
    };
    pull_gather<CSM_HN>(src, own + hc, om1s, dnr, bb, v, d79);
}

// one node per thread, a CTA per 32 x 4 tile and z segment (measured with the
// earlier storage: two threads per node, each gathering half of the
// directions and adding the partial moments through shared memory, ran
// slower at twice the warps). PF: the population gathers of the next plane
// are issued before the current plane is staged and collided, so they are in
// flight across both barriers (19 more live registers: five CTAs per SM).
// FP16 gathers stay raw until the collision (measured at 512 x 512 x 192,
// sigma 12: 2.71 -> 2.54 ms; on a 256-slit ensemble 0.388 -> 0.335 ms): the
// staging between the gathers and their use then hides their latency, as it
// does for FP32 values, which nothing touches before the collision
template <typename T>
constexpr bool F16_RAW = sizeof(T) == 2;
template <typename T, bool PF, bool IP>
__global__ void __launch_bounds__(CSM_THREADS, PF ? CSM_MINB - 1 : CSM_MINB)
    k_csm(Params P, const T* pin, T* pout, CsmIO io, const float4* __restrict__ F, int lz, int tiles_x, int tiles_y,
          int* status)
{
    constexpr int NT = CSM_THREADS;
    extern __shared__ float sm[];
    const Geom& g = P.g;
    const int tiles = tiles_x * tiles_y;
    const int tile = blockIdx.x % tiles, seg = blockIdx.x / tiles;
    const int x0 = (tile % tiles_x) * CSM_TX, y0 = (tile / tiles_x) * CSM_TY;
    const int t = threadIdx.x;
    const int x = x0 + t % CSM_TX, y = y0 + t / CSM_TX;
    const int hc = (t / CSM_TX + 1) * CSM_HX + t % CSM_TX + 1;
    const bool in_xy = x < g.nx && y < g.ny;
    const int zb = seg * lz, ze = min(zb + lz, g.nz);
    const CsmStaged st = csm_staged<NT>(g, x0, y0);
    // the population gathers of plane z (act: the node steps; om its 1/tau)
    // (in place, q returns the node's slots, which its stores reuse)
    auto gather = [&](int z, float* v, unsigned& bb, bool& act, float& om, IpSlots& q) {
        const int s = slit_of(P, z);
        act = in_xy && s >= 0 && !frozen(P, s);
        bb = 0;
        om = 0.f;
        if (act) {
            om = P.sl[s].inv_tau;
            if constexpr (IP) q = ip_slots(P, P.sl[s], s, x, y, z);
            csm_pull<0, Q, IP, T, F16_RAW<T>>(P, pin, ((long long)z * g.ny + y) * g.nx + x, x, y, z, P.sl[s].zlo,
                                              P.sl[s].zhi, v, bb, q);
        }
    };
    IpSlots qn, qz;
    float vn[Q];
    unsigned bbn = 0;
    bool actn = false;
    float omn = 0.f;
    if constexpr (PF) gather(zb, vn, bbn, actn, omn, qn);
    csm_stage<NT>(P, io, F, sm + csm_slot(zb - 1) * CSM_SLOT, st, zb - 1);
    csm_stage<NT>(P, io, F, sm + csm_slot(zb) * CSM_SLOT, st, zb);
    for (int z = zb; z < ze; ++z) {
        // issue the population loads first: they do not depend on the ring
        float v[Q];
        unsigned bb;
        bool act;
        float om;
        if constexpr (PF) {
#pragma unroll
            for (int i = 0; i < Q; ++i) v[i] = vn[i];
            bb = bbn;
            act = actn;
            om = omn;
            if (z + 1 < ze) gather(z + 1, vn, bbn, actn, omn, qn);
        } else {
            gather(z, v, bb, act, om, qz);
        }
        __syncthreads();  // the slot of plane z - 2 is free
        csm_stage<NT>(P, io, F, sm + csm_slot(z + 1) * CSM_SLOT, st, z + 1);
        __syncthreads();
        if (!act) continue;
        const long long idx = ((long long)z * g.ny + y) * g.nx + x;
        const float* own = sm + csm_slot(z) * CSM_SLOT;
        const float dnr = own[SQ_DN * CSM_HN + hc];
        float d79;
        if constexpr (F16_RAW<T>) {
#pragma unroll
            for (int k = 0; k < Q; ++k) v[k] = late_cvt(v[k]);
        }
        csm_collide(own, sm + csm_slot(z - 1) * CSM_SLOT, sm + csm_slot(z + 1) * CSM_SLOT, hc,
                    (1.f - om) / store_scale<T>(), dnr, bb, v, d79);
        float ux, uy, uz;
        float dn;
        if constexpr (IP) {
            // FP16: the stores reuse the gather's slots (2.64 -> 2.47 ms at
            // 512 x 512 x 192, sigma 12); FP32 recomputes them (holding them
            // across the collision spills there: 2.50 -> 2.57 ms)
            IpSlots q;
            if constexpr (PF || sizeof(T) == 4) {
                const int s = slit_of(P, z);
                q = ip_slots(P, P.sl[s], s, x, y, z);
            } else {
                q = qz;
            }
            dn = pull_finish<T>([&](int i) { return pop_at_ip(pout, P, i, q.slot(i)); }, v, d79, dnr, ux, uy, uz);
        } else {
            dn = pull_finish<T>([&](int i) { return pop_at(pout, P, i, idx); }, v, d79, dnr, ux, uy, uz);
        }
        put_fields(P, io, x, y, z, dn, ux, uy, uz, status);
    }
}

// The pull pass with its population gathers brought in by the tensor-memory
// accelerator (two-buffer layout). For every plane whose 19 sources lie
// inside the grid - interior tiles, no wall direction, away from the ends of
// a periodic z - one thread issues, one plane ahead, one copy per direction
// i of the tile's source box (the tile shifted by -c_i, widened in x to
// 16-byte boundaries: BW nodes from x0 - XM when c_ix = 1, else from x0;
// a 4-D tensor map: x, y, z, direction) into one of two shared-memory
// stages, completion counted in bytes on an mbarrier; the threads then read
// their 19 values from there. Other planes gather directly. The arithmetic
// is k_csm's (identical results).
template <typename T>
__host__ __device__ constexpr int tma_xm() { return sizeof(T) == 2 ? 8 : 4; }
template <typename T>
__host__ __device__ constexpr int tma_bw() { return CSM_TX + tma_xm<T>(); }
template <typename T>
__host__ __device__ constexpr int tma_box_bytes() { return tma_bw<T>() * CSM_TY * (int)sizeof(T); }
template <typename T>
__host__ __device__ constexpr int tma_box_pitch() { return (tma_box_bytes<T>() + 127) / 128 * 128; }
__host__ __device__ constexpr int csm_ring_bytes() { return (3 * CSM_SLOT * 4 + 127) / 128 * 128; }
template <typename T>
__host__ __device__ constexpr int csm_tma_smem_bytes() { return csm_ring_bytes() + 2 * Q * tma_box_pitch<T>() + 16; }

void pop_box(int storage, int* W, int* H)
{
    *W = storage == LBIF_STORE_F16 ? tma_bw<__half>() : tma_bw<float>();
    *H = CSM_TY;
}

template <typename T>
__global__ void __launch_bounds__(CSM_THREADS, 4)
    k_csm_tma(Params P, const __grid_constant__ CUtensorMap pmap, const T* pin, T* pout, CsmIO io,
              const float4* __restrict__ F, int lz, int tiles_x, int tiles_y, int* status)
{
    constexpr int NT = CSM_THREADS, XM = tma_xm<T>(), BW = tma_bw<T>(), BOX = tma_box_bytes<T>();
    constexpr int PB = tma_box_pitch<T>(), SB = Q * PB;
    extern __shared__ __align__(128) unsigned char smraw[];
    float* sm = reinterpret_cast<float*>(smraw);
    unsigned char* stg = smraw + csm_ring_bytes();
    uint64_t* mbar = reinterpret_cast<uint64_t*>(stg + 2 * SB);
    const Geom& g = P.g;
    const int tiles = tiles_x * tiles_y;
    const int tile = blockIdx.x % tiles, seg = blockIdx.x / tiles;
    const int x0 = (tile % tiles_x) * CSM_TX, y0 = (tile / tiles_x) * CSM_TY;
    const int t = threadIdx.x;
    const int tx = t % CSM_TX, ty = t / CSM_TX;
    const int x = x0 + tx, y = y0 + ty;
    const int hc = (ty + 1) * CSM_HX + tx + 1;
    const bool in_xy = x < g.nx && y < g.ny;
    const int zb = seg * lz, ze = min(zb + lz, g.nz);
    const bool interior = x0 >= 1 && x0 + CSM_TX <= g.nx - 1 && y0 >= 1 && y0 + CSM_TY <= g.ny - 1;
    // every source of plane z inside the grid and no wall direction (CTA-uniform)
    auto plane_tma = [&](int z) -> bool {
        if (!interior || z < 1 || z > g.nz - 2) return false;
        const int s = slit_of(P, z);
        if (s < 0 || frozen(P, s)) return false;
        return z > P.sl[s].zlo && z < P.sl[s].zhi;
    };
    if (t == 0) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&pmap)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(mbar)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(mbar + 1)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    auto issue = [&](int z) {  // one thread: the 19 boxes of plane z into stage z & 1
        const int b = z & 1;
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(mbar + b)),
                     "r"((uint32_t)(Q * BOX))
                     : "memory");
#pragma unroll
        for (int i = 0; i < Q; ++i)
            asm volatile(
                "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, "
                "%5}], [%6];" ::"r"(smem_addr(stg + b * SB + i * PB)),
                "l"(reinterpret_cast<uint64_t>(&pmap)), "r"(kCx(i) > 0 ? x0 - XM : x0), "r"(y0 - kCy(i)),
                "r"(z - kCz(i)), "r"(i), "r"(smem_addr(mbar + b))
                : "memory");
    };
    uint32_t pbits = 0u;  // bit b: the parity expected next on stage b
    uint32_t pend = 0u;  // bit b: stage b has copies in flight
    // bounded wait for stage b's copies; false if it ran out
    auto wait_stage = [&](int b) -> bool {
        long long spins = 0;
        bool ok;
        while (!(ok = mbar_wait_parity(mbar + b, (pbits >> b) & 1u)) && ++spins < BALL_WAIT_LIMIT) {
        }
        return ok;
    };
    const CsmStaged st = csm_staged<NT>(g, x0, y0);
    if (zb < ze && plane_tma(zb)) {
        if (t == 0) issue(zb);
        pend = 1u << (zb & 1);
    }
    csm_stage<NT>(P, io, F, sm + csm_slot(zb - 1) * CSM_SLOT, st, zb - 1);
    csm_stage<NT>(P, io, F, sm + csm_slot(zb) * CSM_SLOT, st, zb);
    for (int z = zb; z < ze; ++z) {
        const int s = slit_of(P, z);
        const bool act = in_xy && s >= 0 && !frozen(P, s);
        const bool tz = (pend >> (z & 1)) & 1u;
        float v[Q];
        unsigned bb = 0;
        const long long idx = ((long long)z * g.ny + y) * g.nx + x;
        const float om = act ? P.sl[s].inv_tau : 0.f;
        if (act && !tz) {
            IpSlots q;
            csm_pull<0, Q, false>(P, pin, idx, x, y, z, P.sl[s].zlo, P.sl[s].zhi, v, bb, q);
        }
        __syncthreads();  // ring slot of plane z - 2 and stage (z + 1) & 1 are free
        const bool tn = z + 1 < ze && plane_tma(z + 1);
        if (tn) {
            if (t == 0) issue(z + 1);
            pend |= 1u << ((z + 1) & 1);
        }
        csm_stage<NT>(P, io, F, sm + csm_slot(z + 1) * CSM_SLOT, st, z + 1);
        __syncthreads();
        if (tz) {
            const int b = z & 1;
            if (!__syncthreads_and(wait_stage(b))) {
                // record the timeout and wait (bounded) for the copies in flight
                if (t == 0) atomicOr(status, 4);
                if (tn) wait_stage((z + 1) & 1);
                return;
            }
            pbits ^= 1u << b;
            pend &= ~(1u << b);
            if (act) {
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const T* p = reinterpret_cast<const T*>(stg + b * SB + i * PB) + ty * BW +
                                 (tx - kCx(i) + (kCx(i) > 0 ? XM : 0));
                    if constexpr (sizeof(T) == 2)
                        v[i] = __half2float(*reinterpret_cast<const __half*>(p));
                    else
                        v[i] = *reinterpret_cast<const float*>(p);
                }
            }
        }
        if (!act) continue;
        const float* own = sm + csm_slot(z) * CSM_SLOT;
        const float dnr = own[SQ_DN * CSM_HN + hc];
        float d79;
        csm_collide(own, sm + csm_slot(z - 1) * CSM_SLOT, sm + csm_slot(z + 1) * CSM_SLOT, hc,
                    (1.f - om) / store_scale<T>(), dnr, bb, v, d79);
        float ux, uy, uz;
        const float dn = pull_finish<T>([&](int i) { return pop_at(pout, P, i, idx); }, v, d79, dnr, ux, uy, uz);
        put_fields(P, io, x, y, z, dn, ux, uy, uz, status);
    }
}

// Narrow grids (below one 32 x 4 tile): the same pass with one thread per
// node and no staging; every source's quantities are formed where they are
// used, by the same code as the staged ones, so both kernels give identical
// results.
template <typename T, bool IP>
__global__ void __launch_bounds__(128) k_pull_node(Params P, const T* pin, T* pout, CsmIO io,
                                                   const float4* __restrict__ F, int* status)
{
    const long long idx = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (idx >= P.g.N) return;
    const Geom& g = P.g;
    int x, y, z;
    decompose(g, idx, x, y, z);
    const int s = slit_of(P, z);
    if (s < 0 || frozen(P, s)) return;
    const int zlo = P.sl[s].zlo, zhi = P.sl[s].zhi;
    const float om = P.sl[s].inv_tau, om1s = (1.f - om) / store_scale<T>();
    const bool shifted = P.shifted != 0;
    float v[Q];
    unsigned bb = 0;
    IpSlots q;
    if constexpr (IP) q = ip_slots(P, P.sl[s], s, x, y, z);
    csm_pull<0, Q, IP>(P, pin, idx, x, y, z, zlo, zhi, v, bb, q);
    const int p = pidx(g, x, y, z);
    float own[CSM_NF];
    src_terms(__ldg(io.dn + p), __ldg(io.ux + p), __ldg(io.uy + p), __ldg(io.uz + p), __ldg(F + idx), om, shifted,
              [&](int j, float val) { own[j] = val; });
    const float dnr = own[SQ_DN];
    // the source quantities of direction i, formed where they are used
    // (padded fields through their periodic images, the force at its
    // wrapped node); walls never ask (they use own)
    auto terms = [&](auto ic, float* out) {
        constexpr int i = decltype(ic)::value;
        int sx = x - kCx(i), sy = y - kCy(i), sz = z - kCz(i);
        sx = sx < 0 ? sx + g.nx : (sx >= g.nx ? sx - g.nx : sx);
        sy = sy < 0 ? sy + g.ny : (sy >= g.ny ? sy - g.ny : sy);
        if (g.zper) sz = sz < 0 ? sz + g.nz : (sz >= g.nz ? sz - g.nz : sz);
        const int ps = p - P.nbr[i];
        src_terms(__ldg(io.dn + ps), __ldg(io.ux + ps), __ldg(io.uy + ps), __ldg(io.uz + ps),
                  __ldg(F + (((long long)sz * g.ny + sy) * g.nx + sx)), om, shifted,
                  [&](int j, float val) { out[j] = val; });
    };
    auto wall = [&](int i) { return ((bb >> i) & 1u) != 0u; };
    auto diff = [&](auto ic, auto ipc) {
        constexpr int i = decltype(ic)::value, ip = decltype(ipc)::value;
        if (wall(i)) return mirror_diff<i, ip, 1>(own, own, v[i], v[ip], om1s, true);
        float a[CSM_NF], b[CSM_NF];
        terms(ic, a);
        terms(ipc, b);
        return mirror_diff<i, ip, 1>(a, b, v[i], v[ip], om1s, false);
    };
    using std::integral_constant;
    const float d7_10 = diff(integral_constant<int, 7>{}, integral_constant<int, 10>{});
    const float d9_8 = diff(integral_constant<int, 9>{}, integral_constant<int, 8>{});
    const float d10_8 = diff(integral_constant<int, 10>{}, integral_constant<int, 8>{});
    const float d79 = diff(integral_constant<int, 7>{}, integral_constant<int, 9>{});
    v[7] = d7_10;
    v[9] = d9_8;
    v[10] = d10_8;
    v[1] = diff(integral_constant<int, 1>{}, integral_constant<int, 2>{});
    v[3] = diff(integral_constant<int, 3>{}, integral_constant<int, 4>{});
    v[11] = diff(integral_constant<int, 11>{}, integral_constant<int, 14>{});
    v[13] = diff(integral_constant<int, 13>{}, integral_constant<int, 12>{});
    v[15] = diff(integral_constant<int, 15>{}, integral_constant<int, 18>{});
    v[17] = diff(integral_constant<int, 17>{}, integral_constant<int, 16>{});
    auto one = [&](auto ic) {
        constexpr int i = decltype(ic)::value;
        if constexpr (i == 0 || i == 2 || i == 4 || i == 5 || i == 6 || i == 8 || i == 12 || i == 14 || i == 16 ||
                      i == 18) {
            const bool w = i != 0 && wall(i);
            if (i == 0 || w) {
                v[i] = arrive<i, 1>(own, v[i], om1s, dnr, w);
            } else {
                float sv[CSM_NF];
                terms(ic, sv);
                v[i] = arrive<i, 1>(sv, v[i], om1s, dnr, false);
            }
        }
    };
    for_dirs(one);
    float ux, uy, uz;
    const float dn = IP ? pull_finish<T>([&](int i) { return pop_at_ip(pout, P, i, q.slot(i)); }, v, d79, dnr, ux,
                                         uy, uz)
                        : pull_finish<T>([&](int i) { return pop_at(pout, P, i, idx); }, v, d79, dnr, ux, uy, uz);
    put_fields(P, io, x, y, z, dn, ux, uy, uz, status);
}

bool csm_ok(const Geom& g) { return g.nx >= CSM_TX && g.ny >= CSM_TY; }

template <typename T, bool PF, bool IP>
static cudaError_t csm_tiled(const Params& P, const void* pin, void* pout, const CsmIO& io, const float4* F,
                             int* status, int lz, cudaStream_t s)
{
    const Geom& g = P.g;
    const int tx = (g.nx + CSM_TX - 1) / CSM_TX, ty = (g.ny + CSM_TY - 1) / CSM_TY;
    const int segs = (g.nz + lz - 1) / lz;
    const long long blocks = (long long)tx * ty * segs;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    const size_t smem = csm_smem_bytes();
    // the shared-memory limit is a per-device function attribute
    static std::atomic<uint64_t> configured{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = 1ull << (dev & 63);
    if (!(configured.load() & bit)) {
        e = cudaFuncSetAttribute(k_csm<T, PF, IP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    k_csm<T, PF, IP><<<(unsigned)blocks, CSM_THREADS, smem, s>>>(P, (const T*)pin, (T*)pout, io, F, lz, tx, ty, status);
    return cudaGetLastError();
}

template <typename T>
static cudaError_t csm_tma(const Params& P, const CUtensorMap* pmap, const void* pin, void* pout, const CsmIO& io,
                           const float4* F, int* status, int lz, cudaStream_t s)
{
    const Geom& g = P.g;
    const int tx = (g.nx + CSM_TX - 1) / CSM_TX, ty = (g.ny + CSM_TY - 1) / CSM_TY;
    const int segs = (g.nz + lz - 1) / lz;
    const long long blocks = (long long)tx * ty * segs;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    const size_t smem = csm_tma_smem_bytes<T>();
    static std::atomic<uint64_t> configured{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = 1ull << (dev & 63);
    if (!(configured.load() & bit)) {
        e = cudaFuncSetAttribute(k_csm_tma<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    k_csm_tma<T><<<(unsigned)blocks, CSM_THREADS, smem, s>>>(P, *pmap, (const T*)pin, (T*)pout, io, F, lz, tx, ty,
                                                            status);
    return cudaGetLastError();
}

cudaError_t launch_csm(const Params& P, const void* pin, void* pout, const CsmIO& io, const float4* F,
                       int* status, int lz, int prefetch, cudaStream_t s, const CUtensorMap* pmap)
{
    const Geom& g = P.g;
    const bool ip = P.inplace != 0, h16 = P.storage == LBIF_STORE_F16;
    if (prefetch == 2 && pmap && !ip && csm_ok(g)) {
        if (lz <= 0) lz = CSM_LZ;
        return h16 ? csm_tma<__half>(P, pmap, pin, pout, io, F, status, lz, s)
                   : csm_tma<float>(P, pmap, pin, pout, io, F, status, lz, s);
    }
    if (!csm_ok(g)) {
        const unsigned nb = nblocks(g.N, 128);
        if (h16 && ip) k_pull_node<__half, true><<<nb, 128, 0, s>>>(P, (const __half*)pin, (__half*)pout, io, F, status);
        if (h16 && !ip) k_pull_node<__half, false><<<nb, 128, 0, s>>>(P, (const __half*)pin, (__half*)pout, io, F, status);
        if (!h16 && ip) k_pull_node<float, true><<<nb, 128, 0, s>>>(P, (const float*)pin, (float*)pout, io, F, status);
        if (!h16 && !ip) k_pull_node<float, false><<<nb, 128, 0, s>>>(P, (const float*)pin, (float*)pout, io, F, status);
        return cudaGetLastError();
    }
    if (lz <= 0) lz = CSM_LZ;
    if (h16) {
        if (ip)
            return prefetch ? csm_tiled<__half, true, true>(P, pin, pout, io, F, status, lz, s)
                            : csm_tiled<__half, false, true>(P, pin, pout, io, F, status, lz, s);
        return prefetch ? csm_tiled<__half, true, false>(P, pin, pout, io, F, status, lz, s)
                        : csm_tiled<__half, false, false>(P, pin, pout, io, F, status, lz, s);
    }
    if (ip)
        return prefetch ? csm_tiled<float, true, true>(P, pin, pout, io, F, status, lz, s)
                        : csm_tiled<float, false, true>(P, pin, pout, io, F, status, lz, s);
    return prefetch ? csm_tiled<float, true, false>(P, pin, pout, io, F, status, lz, s)
                    : csm_tiled<float, false, false>(P, pin, pout, io, F, status, lz, s);
}

}  // namespace lbif
