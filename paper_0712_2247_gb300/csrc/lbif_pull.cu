// The pull pass: collision, streaming and the next step's moments in one pass
// over the populations, with its launchers.
#include <math.h>

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

// The pass's arithmetic, written once for one node (float) and for two nodes
// at a time (float2: one fma / add / mul .f32x2 instruction does both, each
// component rounding as the scalar operation). Every operation is explicit, so
// all kernels of the pass give identical results. The compiler merges a paired
// product into a paired addition that takes it (the scalar intrinsics it
// leaves alone): a product that feeds an addition is therefore written as one
// vfma, or rounded by itself as vfma(a, b, 0) (vprod).
__device__ __forceinline__ float vfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float vadd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float vsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float vmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float vneg(float a) { return -a; }
__device__ __forceinline__ float vrdiv(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return fma2(a, b, c); }
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return add2(a, b); }
__device__ __forceinline__ float2 vsub(float2 a, float2 b) { return sub2(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return mul2(a, b); }
__device__ __forceinline__ float2 vneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 vrdiv(float a, float2 b) { return make_float2(__fdiv_rn(a, b.x), __fdiv_rn(a, b.y)); }
template <class V>
__device__ __forceinline__ V vset(float s);
template <>
__device__ __forceinline__ float vset<float>(float s) { return s; }
template <>
__device__ __forceinline__ float2 vset<float2>(float s) { return bc2(s); }

template <class V>
__device__ __forceinline__ V vprod(V a, V b) { return vfma(a, b, vset<V>(0.f)); }

// staged quantities of a node: dn, P_x..z, C_x..z, C_xy C_xz C_yz, X_xy X_xz X_yz
constexpr int SQ_DN = 0, SQ_P = 1, SQ_CA = 4, SQ_CP = 7, SQ_X = 10, CSM_NF = 13;

// The staged quantities of a node from its moments and force; st(k, value)
// receives quantity k; om = 1/tau is used by the shifted form only.
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
template <class V, class St>
__device__ __forceinline__ void src_terms(V d, V ux, V uy, V uz, V fx, V fy, V fz, V fw, V om, bool shifted, St st)
{
    const V q1 = vadd(vset<V>(1.f), d);
    st(SQ_DN, d);
    if (shifted) {
        const V hq = vrdiv(0.5f, q1);
        const V u[3] = {ux, uy, uz}, F[3] = {fx, fy, fz};
        const V v[3] = {vfma(hq, fx, ux), vfma(hq, fy, uy), vfma(hq, fz, uz)};  // u'
        const V k = vfma(vset<V>(-0.5f), om, vset<V>(1.f)), a1 = vsub(vset<V>(1.f), om);
        auto dot = [](const V* a, const V* b) { return vfma(a[2], b[2], vfma(a[1], b[1], vmul(a[0], b[0]))); };
        const V k3 = vmul(vset<V>(3.f), k), k45 = vmul(vset<V>(4.5f), k), q45 = vmul(vset<V>(4.5f), q1);
        const V alpha = vfma(vmul(vset<V>(-1.5f), q1), vfma(a1, dot(u, u), vmul(om, dot(v, v))),
                             vmul(vset<V>(-1.f), vmul(k3, dot(v, F))));
        auto gam = [&](int a, int b) {
            return vfma(q45, vfma(a1, vmul(u[a], u[b]), vmul(om, vmul(v[a], v[b]))),
                        vmul(k45, vfma(v[a], F[b], vmul(v[b], F[a]))));
        };
        const V gxx = gam(0, 0), gyy = gam(1, 1), gzz = gam(2, 2);
#pragma unroll
        for (int a = 0; a < 3; ++a)
            st(SQ_P + a, vmul(vset<V>(3.f), vfma(q1, vfma(a1, u[a], vmul(om, v[a])), vmul(k, F[a]))));
        st(SQ_CA + 0, vadd(alpha, gxx));
        st(SQ_CA + 1, vadd(alpha, gyy));
        st(SQ_CA + 2, vadd(alpha, gzz));
        st(SQ_CP + 0, vadd(alpha, vadd(gxx, gyy)));
        st(SQ_CP + 1, vadd(alpha, vadd(gxx, gzz)));
        st(SQ_CP + 2, vadd(alpha, vadd(gyy, gzz)));
        st(SQ_X + 0, vmul(vset<V>(2.f), gam(0, 1)));
        st(SQ_X + 1, vmul(vset<V>(2.f), gam(0, 2)));
        st(SQ_X + 2, vmul(vset<V>(2.f), gam(1, 2)));
        return;
    }
    const V uu = vfma(uz, uz, vfma(uy, uy, vmul(ux, ux)));
    const V B = vmul(vmul(vset<V>(-1.5f), q1), uu);
    const V a = vmul(vset<V>(4.5f), q1), aux = vmul(a, ux), auy = vmul(a, uy), auz = vmul(a, uz);
    const V Cx = vfma(aux, ux, B), Cy = vfma(auy, uy, B), Cz = vfma(auz, uz, B), f15 = vset<V>(1.5f);
    st(SQ_P + 0, vmul(vset<V>(3.f), vfma(q1, ux, fx)));
    st(SQ_P + 1, vmul(vset<V>(3.f), vfma(q1, uy, fy)));
    st(SQ_P + 2, vmul(vset<V>(3.f), vfma(q1, uz, fz)));
    st(SQ_CA + 0, Cx);
    st(SQ_CA + 1, Cy);
    st(SQ_CA + 2, Cz);
    st(SQ_CP + 0, vfma(f15, fw, vfma(auy, uy, Cx)));
    st(SQ_CP + 1, vfma(f15, fw, vfma(auz, uz, Cx)));
    st(SQ_CP + 2, vfma(f15, fw, vfma(auz, uz, Cy)));
    const V bx = vmul(vset<V>(2.f), aux), by = vmul(vset<V>(2.f), auy);  // 9 q u_x, 9 q u_y
    st(SQ_X + 0, vmul(bx, uy));
    st(SQ_X + 1, vmul(bx, uz));
    st(SQ_X + 2, vmul(by, uz));
}

// C_0 of a node from its staged quantities (see above)
template <class V>
__device__ __forceinline__ V rest_term(V cx, V cy, V cz, V cxy, V cxz, V cyz)
{
    const V s = vadd(vadd(cx, cy), cz), d = vadd(vadd(cxy, cxz), cyz);
    return vmul(vsub(vadd(s, s), d), vset<V>(1.f / 3.f));
}

// a node's staged quantities at p, quantity k at p[k ST]
template <int ST>
struct Strided {
    const float* p;
    template <int K>
    __device__ __forceinline__ float get() const
    {
        return p[K * ST];
    }
    __device__ __forceinline__ float c0() const
    {
        return rest_term(get<SQ_CA>(), get<SQ_CA + 1>(), get<SQ_CA + 2>(), get<SQ_CP>(), get<SQ_CP + 1>(),
                         get<SQ_CP + 2>());
    }
};

// v_i (see above) from the source's staged quantities s and its stored h;
// wall: s is the node itself and the direction arrives reversed
template <int i, class V, class Src>
__device__ __forceinline__ V arrive(const Src& s, V h, float om1s, V dnr, bool wall)
{
    constexpr int cx = kCx(i), cy = kCy(i), cz = kCz(i);
    const V o = vset<V>(om1s), ds = s.template get<SQ_DN>(), m = vfma(o, ds, o);
    if constexpr (i == 0) {
        return vfma(m, h, s.c0());
    } else {
        V p, t;
        if constexpr (kC2(i) == 1) {
            constexpr int a = cx ? 0 : (cy ? 1 : 2);
            p = s.template get<SQ_P + a>();
            t = s.template get<SQ_CA + a>();
            t = (cx + cy + cz > 0) != wall ? vadd(t, p) : vsub(t, p);
        } else {
            constexpr int pl = cz == 0 ? 0 : (cy == 0 ? 1 : 2);
            constexpr int a = pl == 2 ? 1 : 0, b = pl == 0 ? 1 : 2;
            constexpr bool pa = (a == 0 ? cx : cy) > 0, same = pa == ((b == 1 ? cy : cz) > 0);
            const V A = s.template get<SQ_P + a>(), B = s.template get<SQ_P + b>();
            p = same ? vadd(A, B) : vsub(A, B);
            t = s.template get<SQ_CP + pl>();
            t = pa != wall ? vadd(t, p) : vsub(t, p);
            const V X = s.template get<SQ_X + pl>();
            t = same ? vadd(t, X) : vsub(t, X);
        }
        return vadd(vfma(m, h, t), vsub(ds, dnr));
    }
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

// v_i - v_ip of a mirror pair (staged quantities of the sources s and sp; the
// stored values h, hp of the two directions; wall: both arrive reversed from
// the node itself, s = sp)
template <int i, int ip, class V, class Src>
__device__ __forceinline__ V mirror_diff(const Src& s, const Src& sp, V h, V hp, float om1s, bool wall)
{
    using M = Mirror<i, ip>;
    const V pa = vadd(s.template get<SQ_P + M::A>(), sp.template get<SQ_P + M::A>());
    V dt;
    if constexpr (M::axis) {
        dt = vsub(s.template get<SQ_CA + M::A>(), sp.template get<SQ_CA + M::A>());
        dt = wall ? vsub(dt, pa) : vadd(dt, pa);
    } else {
        dt = vsub(s.template get<SQ_CP + M::PL>(), sp.template get<SQ_CP + M::PL>());
        dt = wall ? vsub(dt, pa) : vadd(dt, pa);
        const V pb = vsub(s.template get<SQ_P + M::B>(), sp.template get<SQ_P + M::B>());
        dt = (M::CB > 0.f) != wall ? vadd(dt, pb) : vsub(dt, pb);
        const V X = vadd(s.template get<SQ_X + M::PL>(), sp.template get<SQ_X + M::PL>());
        dt = M::CB > 0.f ? vadd(dt, X) : vsub(dt, X);
    }
    const V ds = s.template get<SQ_DN>(), dd = vsub(ds, sp.template get<SQ_DN>());
    // m(s) h - m(sp) hp with m = om1s (1 + d)
    const V dm = vfma(vadd(vset<V>(1.f), ds), vsub(h, hp), vmul(dd, hp));
    return vadd(vfma(vset<V>(om1s), dm, dt), dd);
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
// moments (put(i, h)): base directions directly, derived ones as their
// partner's stored value plus the difference (so the pairs' differences
// survive the rounding of the large common parts); returns dn and writes u
template <typename T, class V, class Put>
__device__ __forceinline__ V pull_finish(Put put, const V* v, V d79, V dnr, V& ux, V& uy, V& uz)
{
    const V w1 = vset<V>(1.f / 18.f), w2 = vset<V>(1.f / 36.f);
    // arriving values of the derived directions
    const V v1 = vadd(v[2], v[1]), v3 = vadd(v[4], v[3]), v9 = vadd(v[8], v[9]), v10 = vadd(v[8], v[10]);
    const V v7 = vadd(v10, v[7]), v11 = vadd(v[14], v[11]), v13 = vadd(v[12], v[13]), v15 = vadd(v[18], v[15]);
    const V v17 = vadd(v[16], v[17]);
    const V sa = vadd(vadd(vadd(v1, v[2]), vadd(v3, v[4])), vadd(v[5], v[6]));
    const V sd = vadd(vadd(vadd(vadd(v7, v[8]), vadd(v9, v10)), vadd(vadd(v11, v[12]), vadd(v13, v[14]))),
                      vadd(vadd(v15, v[16]), vadd(v17, v[18])));
    const V S = vfma(w2, sd, vfma(w1, sa, vmul(vset<V>(1.f / 3.f), v[0])));
    const V jz = vadd(vsub(vsub(v11, v[12]), vsub(v13, v[14])), vsub(vsub(v15, v[16]), vsub(v17, v[18])));
    const V Jz = vfma(w2, jz, vmul(w1, vsub(v[5], v[6])));
    const V Jx = vfma(w2, vadd(vadd(v[7], v[9]), vadd(v[11], v[13])), vmul(w1, v[1]));
    const V Jy = vfma(w2, vadd(vadd(d79, v[10]), vadd(v[15], v[17])), vmul(w1, v[3]));
    const V dn = vadd(dnr, S);
    const V inv = vrdiv(1.f, vadd(vset<V>(1.f), dn));
    ux = vprod(Jx, inv);
    uy = vprod(Jy, inv);
    uz = vprod(Jz, inv);
    const V u15 = vmul(vset<V>(1.5f), vfma(uz, uz, vfma(uy, uy, vmul(ux, ux))));
    const V sT = vset<V>(store_scale<T>());
    auto store = [&](int i, V h) { put(i, sizeof(T) == 2 ? vmul(sT, h) : h); };
    // (v_i - S) / (1 + dn) - p_i with p_i = f_i^eq / (w_i n) - 1 =
    // c.u (3 + 9/2 c.u) - 3/2 u.u, of a base direction with cm = -c.u
    auto base = [&](V vi, V cm) {
        return vfma(vsub(vi, S), inv, vfma(cm, vfma(vset<V>(-4.5f), cm, vset<V>(3.f)), u15));
    };
    // v inv - (p_i - p_ip) of a pair that differs in component a:
    // p_i - p_ip = u_a (6 + 18 R), R = the shared part of c.u (Rm = -R)
    auto diff = [&](V vi, V ua, V Rm) { return vfma(vi, inv, vmul(ua, vfma(vset<V>(18.f), Rm, vset<V>(-6.f)))); };
    const V six = vset<V>(-6.f);
    store(0, vfma(vsub(v[0], S), inv, u15));
    store(5, base(v[5], vneg(uz)));
    store(6, base(v[6], uz));
    const V h2 = base(v[2], ux), h4 = base(v[4], uy), h8 = base(v[8], vadd(ux, uy));
    store(2, h2);
    store(1, vadd(h2, vfma(v[1], inv, vmul(ux, six))));
    store(4, h4);
    store(3, vadd(h4, vfma(v[3], inv, vmul(uy, six))));
    store(8, h8);
    store(9, vadd(h8, diff(v[9], ux, uy)));
    const V h10 = vadd(h8, diff(v[10], uy, ux));
    store(10, h10);
    store(7, vadd(h10, diff(v[7], ux, vneg(uy))));
    const V h12 = base(v[12], vadd(ux, uz)), h14 = base(v[14], vsub(ux, uz));
    store(12, h12);
    store(13, vadd(h12, diff(v[13], ux, uz)));
    store(14, h14);
    store(11, vadd(h14, diff(v[11], ux, vneg(uz))));
    const V h16 = base(v[16], vadd(uy, uz)), h18 = base(v[18], vsub(uy, uz));
    store(16, h16);
    store(17, vadd(h16, diff(v[17], uy, uz)));
    store(18, h18);
    store(15, vadd(h18, diff(v[15], uy, vneg(uz))));
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
// owns a 32 x 4 tile of x-y nodes (more, smaller CTAs keep more population
// loads in flight across the two barriers of a round: 32 x 8 and 32 x 12 tiles
// ran 7 % and 15 % slower) and marches it up a segment of z planes. Three
// forms: two planes per round (the default, k_pull_pair below), and one plane
// per round (k_csm), with the next plane's gathers issued early or copied by
// the tensor-memory accelerator (k_csm_tma), whose ring holds three planes.
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

template <int NT, int TX = CSM_TX>
__device__ __forceinline__ CsmStaged csm_staged(const Geom& g, int x0, int y0)
{
    constexpr int HX = TX + 2, HN = HX * (CSM_THREADS / TX + 2);
    static_assert(NT * CSM_KS >= HN && HN <= CSM_HN, "two staged nodes per thread at most");
    CsmStaged st;
#pragma unroll
    for (int k = 0; k < CSM_KS; ++k) {
        const int h = threadIdx.x + k * NT;
        const int X = x0 - 1 + h % HX, Y = y0 - 1 + h / HX;
        st.p[k] = st.n[k] = -1;
        if (h >= HN || X > g.nx || Y > g.ny) continue;
        const int xw = X < 0 ? X + g.nx : (X >= g.nx ? X - g.nx : X);
        const int yw = Y < 0 ? Y + g.ny : (Y >= g.ny ? Y - g.ny : Y);
        st.p[k] = (Y + g.hw) * g.px + (X + g.hw);
        st.n[k] = yw * g.nx + xw;
    }
    return st;
}

// stage plane q (-1 <= q <= nz) of the tile into `slot`
template <int NT>
__device__ __forceinline__ void csm_stage(const Params& P, const CsmIO& io, const float4* F,
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
        const float4 f = Fq[st.n[k]];
        src_terms(ldp(io.dn + p), ldp(io.ux + p), ldp(io.uy + p), ldp(io.uz + p), f.x, f.y, f.z, f.w, om,
                  shifted, [&](int j, float val) { slot[j * CSM_HN + h] = val; });
    }
}

// CTAs per SM the register budget of the one-plane form is sized for (with and
// without prefetching), and the z planes per CTA segment of the one-plane forms
constexpr int CSM_MINB = 5, CSM_MINB_PLAIN = 6;
constexpr int CSM_LZ = 16;

// the stored populations of directions [I0, I1) that stream into node
// (x, y, z): v[i - I0]; bit i of bb marks a direction that arrives from a
// wall (bounce-back: the node's own opposite population). IP: in place
// (slots from q, see above).
template <int I0, int I1, bool IP, typename T, bool RAW = false>
__device__ __forceinline__ void csm_pull(const Params& P, const T* pin, long long idx, int x, int y,
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

// The arriving values of a node (or a pair of nodes) in the slots described
// at Mirror: the ten mirror differences first (from the stored values as
// loaded), then the ten base directions. src(i) is the source quantities of
// direction i; wall directions (bit i of bb) arrive reversed from the node
// itself (own).
template <bool WALLS, class V, class SrcOf, class Own>
__device__ __forceinline__ void pull_gather_impl(SrcOf src, const Own& own, float om1s, V dnr, unsigned bb, V* v,
                                                 V& d79)
{
    auto wall = [&](int i) { return WALLS && ((bb >> i) & 1u) != 0u; };
    auto diff = [&](auto ic, auto ipc) -> V {
        constexpr int i = decltype(ic)::value, ip = decltype(ipc)::value;
        if constexpr (WALLS && kCz(i) != 0) {
            if (wall(i)) return mirror_diff<i, ip, V>(own, own, v[i], v[ip], om1s, true);
        }
        return mirror_diff<i, ip, V>(src(ic), src(ipc), v[i], v[ip], om1s, false);
    };
    using std::integral_constant;
    const V d7_10 = diff(integral_constant<int, 7>{}, integral_constant<int, 10>{});
    const V d9_8 = diff(integral_constant<int, 9>{}, integral_constant<int, 8>{});
    const V d10_8 = diff(integral_constant<int, 10>{}, integral_constant<int, 8>{});
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
        if constexpr (i == 0) {
            v[i] = arrive<i, V>(own, v[i], om1s, dnr, false);
        } else if constexpr (i == 2 || i == 4 || i == 5 || i == 6 || i == 8 || i == 12 || i == 14 || i == 16 ||
                             i == 18) {
            if constexpr (WALLS && kCz(i) != 0) {
                if (wall(i)) {
                    v[i] = arrive<i, V>(own, v[i], om1s, dnr, true);
                    return;
                }
            }
            v[i] = arrive<i, V>(src(ic), v[i], om1s, dnr, false);
        }
    };
    for_dirs(one);
}

// the same; nodes with no wall direction (bb = 0, almost all) take a path
// without the wall selections
template <class V, class SrcOf, class Own>
__device__ __forceinline__ void pull_gather(SrcOf src, const Own& own, float om1s, V dnr, unsigned bb, V* v, V& d79)
{
    if (bb == 0u)
        pull_gather_impl<false, V>(src, own, om1s, dnr, bb, v, d79);
    else
        pull_gather_impl<true, V>(src, own, om1s, dnr, bb, v, d79);
}

// the gather of a node staged at hc in the ring (planes below, own, above)
__device__ __forceinline__ void csm_collide(const float* own, const float* below, const float* above, int hc,
                                            float om1s, float dnr, unsigned bb, float* v, float& d79)
{
    using Src = Strided<CSM_HN>;
    auto src = [&](auto ic) {
        constexpr int i = decltype(ic)::value;
        constexpr int cx = kCx(i), cy = kCy(i), cz = kCz(i);
        return Src{(cz > 0 ? below : (cz < 0 ? above : own)) + hc - cx - cy * CSM_HX};
    };
    pull_gather(src, Src{own + hc}, om1s, dnr, bb, v, d79);
}

// One node per thread and plane. PF, the prefetched form: the population gathers of
// the next plane issued before the current plane is staged and collided, so they
// are in flight across both barriers (96 registers, five CTAs per SM). FP16 gathers
// stay raw until the collision, so that the staging hides their latency. Without it
// (80 registers, six CTAs) the form of wide slits of few planes (low_slit).
template <typename T>
constexpr bool F16_RAW = sizeof(T) == 2;
template <typename T, bool IP, bool PF>
__global__ void __launch_bounds__(CSM_THREADS, PF ? CSM_MINB : CSM_MINB_PLAIN)
    k_csm(Params P, const T* pin, T* pout, CsmIO io, const float4* F, int lz, int tiles_x, int tiles_y,
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
    auto gather = [&](int z, float* v, unsigned& bb, bool& act, float& om) {
        const int s = slit_of(P, z);
        act = in_xy && s >= 0 && !frozen(P, s);
        bb = 0;
        om = 0.f;
        if (act) {
            om = P.sl[s].inv_tau;
            IpSlots q;
            if constexpr (IP) q = ip_slots(P, P.sl[s], s, x, y, z);
            csm_pull<0, Q, IP, T, F16_RAW<T>>(P, pin, ((long long)z * g.ny + y) * g.nx + x, x, y, z, P.sl[s].zlo,
                                              P.sl[s].zhi, v, bb, q);
        }
    };
    float vn[Q];
    unsigned bbn;
    bool actn;
    float omn;
    if constexpr (PF) gather(zb, vn, bbn, actn, omn);
    csm_stage<NT>(P, io, F, sm + csm_slot(zb - 1) * CSM_SLOT, st, zb - 1);
    csm_stage<NT>(P, io, F, sm + csm_slot(zb) * CSM_SLOT, st, zb);
    for (int z = zb; z < ze; ++z) {
        if constexpr (!PF) gather(z, vn, bbn, actn, omn);
        float v[Q];
#pragma unroll
        for (int i = 0; i < Q; ++i) v[i] = vn[i];
        const unsigned bb = bbn;
        const bool act = actn;
        const float om = omn;
        if (PF && z + 1 < ze) gather(z + 1, vn, bbn, actn, omn);
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
            const int s = slit_of(P, z);
            const IpSlots q = ip_slots(P, P.sl[s], s, x, y, z);
            dn = pull_finish<T>([&](int i, float h) { stp(pop_at_ip(pout, P, i, q.slot(i)), h); }, v, d79, dnr, ux, uy,
                                uz);
        } else {
            dn = pull_finish<T>([&](int i, float h) { stp(pop_at(pout, P, i, idx), h); }, v, d79, dnr, ux, uy, uz);
        }
        put_fields(P, io, x, y, z, dn, ux, uy, uz, status);
    }
}

// ---- two planes at a time ------------------------------------------------
// The default form: a thread owns the nodes (x, y, z) and (x, y, z + 1) and a
// CTA marches its tile of 128 nodes (TX x 128 / TX, 32 x 4 on all but narrow
// grids) up two planes per round. The pair's arithmetic
// is paired FP32 (one instruction for both nodes), one shared-memory load
// brings a staged quantity of both nodes, their wrapped x-y offsets are
// computed once, and a round of two planes costs two barriers. Populations
// stay scalar loads (one per node and direction), so the form has no
// alignment condition and serves both storage layouts. Against one plane per
// round and thread (the former default): 705 instructions per node for 1261,
// and at 512 x 512 x 192, sigma 12, 2.39 -> 2.19 ms FP32 (0.66 of the copy
// bandwidth at 196 B/node), 2.54 -> 1.90 ms FP16, 2.50 -> 2.34 ms FP32 in
// place; 256 stacked slits FP16 in place 0.68 -> 0.59 ms. It waits on load
// latency (14 warps per SM, 39 % issue): four CTAs per SM by registers (128)
// and shared memory. Tried and slower: three CTAs with the next round's
// gathers held in registers (2.32 ms), five CTAs at 96 registers (3.0 ms),
// prefetching the next round's rows to L2 (2.11-2.27 ms FP32 by what it
// spills, 1.93-2.13 ms FP16).
//
// Staged pairs (float2 per node of the halo tile). Of a round's planes
// z - 1 .. z + 2 the populations with c_z = +1 come from (z - 1, z), those
// with c_z = -1 from (z + 1, z + 2) and the others from (z, z + 1):
//   AB[2]  nine quantities of the pairs (z - 1, z) and (z + 1, z + 2), the
//          latter being the next round's former
//   OW[2]  five quantities of the pair (z, z + 1) that only c_z = 0 asks for
//          (C_x, C_y, C_xy, X_xy, C_0); its dn, P_x, P_y are read from AB
// A round stages planes z + 1 and z + 2: the pair into AB, plane z + 1 as the
// second half of this round's OW and plane z + 2 as the first half of the
// next round's.
constexpr int AB_DN = 0, AB_P = 1, AB_CZ = 4, AB_CP = 5, AB_X = 7, AB_NF = 9;  // P x y z; CP, X of xz, yz
constexpr int OW_C = 0, OW_CP = 2, OW_X = 3, OW_C0 = 4, OW_NF = 5;
constexpr int PAIR_FLOATS = 2 * CSM_HN * 2 * (AB_NF + OW_NF);
constexpr int PAIR_MINB = 4;  // CTAs per SM

__host__ __device__ constexpr int ab_of(int k)
{
    return k == SQ_DN ? AB_DN
         : k < SQ_CA ? AB_P + (k - SQ_P)
         : k == SQ_CA + 2 ? AB_CZ
         : k < SQ_X ? AB_CP + (k - SQ_CP - 1) : AB_X + (k - SQ_X - 1);
}
__host__ __device__ constexpr bool in_ow(int k) { return k == SQ_CA || k == SQ_CA + 1 || k == SQ_CP || k == SQ_X; }
__host__ __device__ constexpr int ow_of(int k) { return k == SQ_CP ? OW_CP : (k == SQ_X ? OW_X : OW_C + (k - SQ_CA)); }

// the staged pair of a round at one halo node, for the directions with c_z != 0
struct SideSrc {
    const float2* ab;
    template <int K>
    __device__ __forceinline__ float2 get() const
    {
        return ab[ab_of(K) * CSM_HN];
    }
};
// and for those with c_z = 0: lo, hi = AB of (z - 1, z) and (z + 1, z + 2)
struct LevelSrc {
    const float2* ow;
    const float2* lo;
    const float2* hi;
    template <int K>
    __device__ __forceinline__ float2 get() const
    {
        if constexpr (in_ow(K))
            return ow[ow_of(K) * CSM_HN];
        else
            return make_float2(lo[ab_of(K) * CSM_HN].y, hi[ab_of(K) * CSM_HN].x);
    }
    __device__ __forceinline__ float2 c0() const { return ow[OW_C0 * CSM_HN]; }
};
// one node j of the round's pair (the rounds that touch a wall, or where only
// one of the two planes steps): sources beside it, below or above it, and itself
struct LoneSrc {
    const float* ow;   // component j of OW
    const float* own;  // its plane in AB (z: second half of lo; z + 1: first half of hi)
    const float* side; // the plane asked for (own, or the one below / above)
    template <int K>
    __device__ __forceinline__ float get() const
    {
        return in_ow(K) ? ow[2 * ow_of(K) * CSM_HN] : side[2 * ab_of(K) * CSM_HN];
    }
    __device__ __forceinline__ float c0() const { return ow[2 * OW_C0 * CSM_HN]; }
};

// the staging loads of planes q and q + 1 for one halo node, and what they become
struct PairStage {
    float2 d, ux, uy, uz;
    float4 f0, f1;
};

// where direction i's populations are read from and written to, as pointers a
// 32-bit node offset is added to (two buffers: src folds in -c_z planes)
struct PullPtrs {
    const void* src[Q];
    void* dst[Q];
};

template <typename T, bool IP, int TX>
__global__ void __launch_bounds__(CSM_THREADS, PAIR_MINB)
    k_pull_pair(Params P, PullPtrs pp, CsmIO io, const float4* F, int lz, int tiles_x, int tiles_y,
                int* status)
{
    step_begin(P);
    constexpr int NT = CSM_THREADS, TY = NT / TX, HX = TX + 2;
    constexpr bool RAW = F16_RAW<T>;
    extern __shared__ __align__(16) float2 psm[];
    float2* const AB = psm;
    float2* const OW = psm + 2 * AB_NF * CSM_HN;
    const Geom& g = P.g;
    const int nx = g.nx, ny = g.ny, nz = g.nz, nxy = nx * ny;
    const int tiles = tiles_x * tiles_y;
    const int tile = blockIdx.x % tiles, seg = blockIdx.x / tiles;
    const int x0 = (tile % tiles_x) * TX, y0 = (tile / tiles_x) * TY;
    const int t = threadIdx.x;
    const int x = x0 + t % TX, y = y0 + t / TX;
    const int hc = (t / TX + 1) * HX + t % TX + 1;
    const bool in_xy = x < nx && y < ny;
    const int zb = seg * lz, ze = min(zb + lz, nz);
    const CsmStaged st = csm_staged<NT, TX>(g, x0, y0);
    const int pplane = g.py * g.px;
    const bool shifted = P.shifted != 0;

    // plane q as stored (periodic image), -1 where nothing is staged
    auto plane_of = [&](int q) -> int {
        if (g.zper) q = q < 0 ? q + nz : (q >= nz ? q - nz : q);
        if (q < 0 || q >= nz) return -1;
        const int s = slit_of(P, q);
        return s < 0 || frozen(P, s) ? -1 : q;
    };
    auto stage_load = [&](int q, int k, PairStage& a) {
        a.d = a.ux = a.uy = a.uz = make_float2(0.f, 0.f);
        a.f0 = a.f1 = make_float4(0.f, 0.f, 0.f, 0.f);
        if (st.p[k] < 0) return;
        const int p = (q + g.hw) * pplane + st.p[k];
        const int q0 = plane_of(q), q1 = plane_of(q + 1);
        if (q0 >= 0) {
            a.d.x = ldp(io.dn + p);
            a.ux.x = ldp(io.ux + p);
            a.uy.x = ldp(io.uy + p);
            a.uz.x = ldp(io.uz + p);
            a.f0 = F[(unsigned)(q0 * nxy + st.n[k])];
        }
        if (q1 >= 0) {
            a.d.y = ldp(io.dn + p + pplane);
            a.ux.y = ldp(io.ux + p + pplane);
            a.uy.y = ldp(io.uy + p + pplane);
            a.uz.y = ldp(io.uz + p + pplane);
            a.f1 = F[(unsigned)(q1 * nxy + st.n[k])];
        }
    };
    // planes (q, q + 1) into pair slot ab; plane q completes own slot ow, plane
    // q + 1 begins the other
    auto stage_store = [&](int q, int k, const PairStage& a, int ab, int ow) {
        if (st.p[k] < 0) return;
        const int h = t + k * NT;
        float2 om = make_float2(0.f, 0.f);
        if (shifted) {
            const int q0 = plane_of(q), q1 = plane_of(q + 1);
            if (q0 >= 0) om.x = P.sl[slit_of(P, q0)].inv_tau;
            if (q1 >= 0) om.y = P.sl[slit_of(P, q1)].inv_tau;
        }
        float2* A = AB + ab * AB_NF * CSM_HN + h;
        float2* O0 = OW + ow * OW_NF * CSM_HN + h;
        float2* O1 = OW + (ow ^ 1) * OW_NF * CSM_HN + h;
        float2 C[6];
        src_terms(a.d, a.ux, a.uy, a.uz, make_float2(a.f0.x, a.f1.x), make_float2(a.f0.y, a.f1.y),
                  make_float2(a.f0.z, a.f1.z), make_float2(a.f0.w, a.f1.w), om, shifted, [&](int j, float2 v) {
                      if (j >= SQ_CA && j < SQ_X) C[j - SQ_CA] = v;
                      if (in_ow(j)) {
                          O0[ow_of(j) * CSM_HN].y = v.x;
                          O1[ow_of(j) * CSM_HN].x = v.y;
                      } else {
                          A[ab_of(j) * CSM_HN] = v;
                      }
                  });
        const float2 c0 = rest_term(C[0], C[1], C[2], C[3], C[4], C[5]);
        O0[OW_C0 * CSM_HN].y = c0.x;
        O1[OW_C0 * CSM_HN].x = c0.y;
    };
    {
        PairStage a;
        stage_load(zb - 1, 0, a);
        stage_store(zb - 1, 0, a, 0, 1);
        stage_load(zb - 1, 1, a);
        stage_store(zb - 1, 1, a, 0, 1);
    }
    int xo[3], yo[3];  // x and y nx of the nodes' sources with c = 0, +1, -1 (two buffers: fixed)
    if constexpr (!IP) {
        xo[0] = x;
        xo[1] = x > 0 ? x - 1 : nx - 1;
        xo[2] = x < nx - 1 ? x + 1 : 0;
        yo[0] = y * nx;
        yo[1] = (y > 0 ? y - 1 : ny - 1) * nx;
        yo[2] = (y < ny - 1 ? y + 1 : 0) * nx;
    }
    for (int z = zb; z < ze; z += 2) {
        const int r = ((z - zb) >> 1) & 1;
        const int s0 = slit_of(P, z), s1 = z + 1 < ze ? slit_of(P, z + 1) : -1;
        const bool on0 = s0 >= 0 && !frozen(P, s0), on1 = s1 >= 0 && !frozen(P, s1);
        const bool act0 = in_xy && on0, act1 = in_xy && on1;
        // both nodes step and none of their sources lies beyond a wall (the
        // same for the whole CTA)
        bool both = on0 && on1 && s0 == s1;
        bool wrap = false;
        if (both) {
            const bool inner = z > P.sl[s0].zlo && z + 1 < P.sl[s0].zhi;
            both = inner || g.zper;
            wrap = !inner;
        }
        PairStage a0, a1;
        stage_load(z + 1, 0, a0);
        stage_load(z + 1, 1, a1);
        float2 v[Q];
        unsigned bb0 = 0, bb1 = 0;
        int zo[3][2];  // in place: z offsets of the slots, c_z = 0, +1, -1, of both nodes
        if (both && (IP || !wrap)) {
            if (in_xy) {
                if constexpr (IP) {
                    const IpSlots q0 = ip_slots(P, P.sl[s0], s0, x, y, z), q1 = ip_slots(P, P.sl[s0], s0, x, y, z + 1);
                    xo[0] = q0.x, xo[1] = q0.xm, xo[2] = q0.xp;
                    yo[0] = q0.y * nx, yo[1] = q0.ym * nx, yo[2] = q0.yp * nx;
                    zo[0][0] = (q0.zb + q0.zr) * nxy, zo[1][0] = (q0.zb + q0.zm) * nxy, zo[2][0] = (q0.zb + q0.zp) * nxy;
                    zo[0][1] = (q1.zb + q1.zr) * nxy, zo[1][1] = (q1.zb + q1.zm) * nxy, zo[2][1] = (q1.zb + q1.zp) * nxy;
                }
#pragma unroll
                for (int i = 0; i < Q; ++i) {
                    const int cx = kCx(i), cy = kCy(i), cz = kCz(i);
                    const int o = xo[cx > 0 ? 1 : (cx < 0 ? 2 : 0)] + yo[cy > 0 ? 1 : (cy < 0 ? 2 : 0)];
                    const T* p = static_cast<const T*>(pp.src[i]);
                    if constexpr (IP) {
                        const int k = cz > 0 ? 1 : (cz < 0 ? 2 : 0);
                        v[i].x = ldq<RAW>(p + (unsigned)(o + zo[k][0]));
                        v[i].y = ldq<RAW>(p + (unsigned)(o + zo[k][1]));
                    } else {
                        v[i].x = ldq<RAW>(p + (unsigned)(o + z * nxy));
                        v[i].y = ldq<RAW>(p + (unsigned)(o + (z + 1) * nxy));
                    }
                }
            }
        } else {
            // the general gathers, one node after the other
            const T* pin = static_cast<const T*>(pp.src[0]);
            float w[Q];
            IpSlots q;
            if (act0) {
                if constexpr (IP) q = ip_slots(P, P.sl[s0], s0, x, y, z);
                csm_pull<0, Q, IP, T, RAW>(P, pin, (long long)z * nxy + y * nx + x, x, y, z, P.sl[s0].zlo, P.sl[s0].zhi,
                                           w, bb0, q);
#pragma unroll
                for (int i = 0; i < Q; ++i) v[i].x = w[i];
            }
            if (act1) {
                if constexpr (IP) q = ip_slots(P, P.sl[s1], s1, x, y, z + 1);
                csm_pull<0, Q, IP, T, RAW>(P, pin, (long long)(z + 1) * nxy + y * nx + x, x, y, z + 1, P.sl[s1].zlo,
                                           P.sl[s1].zhi, w, bb1, q);
#pragma unroll
                for (int i = 0; i < Q; ++i) v[i].y = w[i];
            }
        }
        __syncthreads();  // the previous round's pairs are read
        stage_store(z + 1, 0, a0, r ^ 1, r);
        stage_store(z + 1, 1, a1, r ^ 1, r);
        __syncthreads();
        const float2* lo = AB + r * AB_NF * CSM_HN + hc;
        const float2* hi = AB + (r ^ 1) * AB_NF * CSM_HN + hc;
        const float2* ow = OW + r * OW_NF * CSM_HN + hc;
        if (both) {
            if (!in_xy) continue;
            if constexpr (RAW) {
#pragma unroll
                for (int i = 0; i < Q; ++i) v[i] = make_float2(late_cvt(v[i].x), late_cvt(v[i].y));
            }
            const float2 dnr = make_float2(lo[AB_DN * CSM_HN].y, hi[AB_DN * CSM_HN].x);
            auto src = [&](auto ic) {
                constexpr int i = decltype(ic)::value;
                constexpr int o = -kCx(i) - kCy(i) * HX, cz = kCz(i);
                if constexpr (cz != 0)
                    return SideSrc{(cz > 0 ? lo : hi) + o};
                else
                    return LevelSrc{ow + o, lo + o, hi + o};
            };
            float2 d79, ux, uy, uz;
            pull_gather_impl<false>(src, LevelSrc{ow, lo, hi}, (1.f - P.sl[s0].inv_tau) / store_scale<T>(), dnr, 0u, v,
                                    d79);
            const int o0 = z * nxy + y * nx + x;
            auto put = [&](int i, float2 h) {
                T* p = static_cast<T*>(pp.dst[i]);
                if constexpr (IP) {
                    const int cx = kCx(i), cy = kCy(i), cz = kCz(i);
                    const int o = xo[cx > 0 ? 1 : (cx < 0 ? 2 : 0)] + yo[cy > 0 ? 1 : (cy < 0 ? 2 : 0)];
                    const int k = cz > 0 ? 1 : (cz < 0 ? 2 : 0);
                    stp(p + (unsigned)(o + zo[k][0]), h.x);
                    stp(p + (unsigned)(o + zo[k][1]), h.y);
                } else {
                    stp(p + (unsigned)o0, h.x);
                    stp(p + (unsigned)(o0 + nxy), h.y);
                }
            };
            const float2 dn = pull_finish<T>(put, v, d79, dnr, ux, uy, uz);
            put_fields(P, io, x, y, z, dn.x, ux.x, uy.x, uz.x, status);
            put_fields(P, io, x, y, z + 1, dn.y, ux.y, uy.y, uz.y, status);
            continue;
        }
#pragma unroll 1
        for (int j = 0; j < 2; ++j) {
            if (!(j ? act1 : act0)) continue;
            float w[Q];
#pragma unroll
            for (int i = 0; i < Q; ++i) {
                w[i] = j ? v[i].y : v[i].x;
                if constexpr (RAW) w[i] = late_cvt(w[i]);
            }
            const float* fl = reinterpret_cast<const float*>(lo);
            const float* fh = reinterpret_cast<const float*>(hi);
            const float* fo = reinterpret_cast<const float*>(ow) + j;
            const float* own = j ? fh : fl + 1;
            const float* below = fl + j;
            const float* above = fh + j;
            auto src = [&](auto ic) {
                constexpr int i = decltype(ic)::value;
                constexpr int o = 2 * (-kCx(i) - kCy(i) * HX), cz = kCz(i);
                return LoneSrc{fo + o, own + o, (cz > 0 ? below : (cz < 0 ? above : own)) + o};
            };
            const int s = j ? s1 : s0;
            const float dnr = own[2 * AB_DN * CSM_HN];
            float d79, ux, uy, uz;
            pull_gather_impl<true>(src, LoneSrc{fo, own, own}, (1.f - P.sl[s].inv_tau) / store_scale<T>(), dnr,
                                   j ? bb1 : bb0, w, d79);
            IpSlots q;
            if constexpr (IP) q = ip_slots(P, P.sl[s], s, x, y, z + j);
            const int o0 = (z + j) * nxy + y * nx + x;
            const float dn = pull_finish<T>(
                [&](int i, float h) { stp(static_cast<T*>(pp.dst[i]) + (unsigned)(IP ? q.slot(i) : o0), h); }, w, d79,
                dnr, ux, uy, uz);
            put_fields(P, io, x, y, z + j, dn, ux, uy, uz, status);
        }
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
              const float4* F, int lz, int tiles_x, int tiles_y, int* status)
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
        const float dn =
            pull_finish<T>([&](int i, float h) { stp(pop_at(pout, P, i, idx), h); }, v, d79, dnr, ux, uy, uz);
        put_fields(P, io, x, y, z, dn, ux, uy, uz, status);
    }
}

// Thin grids (cross-sections of at most BLOCK_A nodes, such as the 4 x 4 slits
// that generate training profiles): a marched tile would leave most threads
// idle, so a CTA takes all nodes of tz whole planes, one per thread, with the
// planes' staged quantities (and one plane below and above) in shared memory,
// where the periodic neighbours in x and y are found by wrapping. The same code
// forms and uses the quantities as in the marched forms (identical results).
// 2048 slits of 4 x 4 x H: one node per thread without staging, each forming
// its ~35 sources' quantities itself, 339 us; so 225 us (130 with the shorter
// padded rows of later).
// Cross-sections of up to BLOCK_A_MAX nodes run so too where the marched tiles
// would be less than two thirds full. Microseconds in tiles / whole planes: 65 x 1 x
// 1600 28.9 / 17.4 (25.3 without staging), 33 x 2 x 1500 28.8 / 16.5, 13 x 6 x 20000
// 133 / 124, 11 x 11 x 20000 216 / 180, but 25 x 4 x 20000 156 / 164 and
// 16 x 8 x 20000 141 / 166.
// (Writing the new moments through shared memory as whole padded planes, images
// and all, instead of node by node: 217 us at 4 x 4, but 445 us against 372 at
// 8 x 8; not kept.)
constexpr int BLOCK_A = 64, BLOCK_A_MAX = 128, BLOCK_NT = 256;

template <typename T, bool IP, int AMAX>
__global__ void __launch_bounds__(BLOCK_NT) k_pull_block(Params P, const T* pin, T* pout, CsmIO io,
                                                         const float4* F, int tz, int* status)
{
    step_begin(P);
    constexpr int NS = BLOCK_NT + 2 * AMAX;  // staged nodes
    __shared__ float st[CSM_NF * NS];
    constexpr bool RAW = F16_RAW<T>;
    const Geom& g = P.g;
    const int nx = g.nx, ny = g.ny, A = nx * ny, z0 = blockIdx.x * tz;
    const bool shifted = P.shifted != 0;
    const int zl = threadIdx.x / A, xy = threadIdx.x - zl * A, y = xy / nx, x = xy - y * nx, z = z0 + zl;
    const int s = zl < tz && z < g.nz ? slit_of(P, z) : -1;
    const bool act = s >= 0 && !frozen(P, s);
    const long long idx = (long long)z * A + xy;
    float v[Q];
    unsigned bb = 0;
    IpSlots q;
    if (act) {
        if constexpr (IP) q = ip_slots(P, P.sl[s], s, x, y, z);
        csm_pull<0, Q, IP, T, RAW>(P, pin, idx, x, y, z, P.sl[s].zlo, P.sl[s].zhi, v, bb, q);
    }
    for (int k = threadIdx.x; k < (tz + 2) * A; k += blockDim.x) {
        const int kz = k / A, kxy = k - kz * A, ky = kxy / nx, kx = kxy - ky * nx;
        const int r = z0 - 1 + kz;  // plane; beyond a periodic end its image, beyond a wall nothing
        const int w = g.zper ? (r < 0 ? r + g.nz : (r >= g.nz ? r - g.nz : r)) : r;
        if (w < 0 || w >= g.nz || r > g.nz) continue;  // (the last CTA reaches past the grid)
        const int ks = slit_of(P, w);
        if (ks < 0 || frozen(P, ks)) continue;
        const int p = pidx(g, kx, ky, r);
        const float4 f = F[(long long)w * A + kxy];
        src_terms(ldp(io.dn + p), ldp(io.ux + p), ldp(io.uy + p), ldp(io.uz + p), f.x, f.y, f.z, f.w,
                  P.sl[ks].inv_tau, shifted, [&](int j, float val) { st[j * NS + k] = val; });
    }
    __syncthreads();
    if (!act) return;
    if constexpr (RAW) {
#pragma unroll
        for (int i = 0; i < Q; ++i) v[i] = late_cvt(v[i]);
    }
    const int xo[3] = {x, x > 0 ? x - 1 : nx - 1, x < nx - 1 ? x + 1 : 0};  // sources with c_x = 0, 1, -1
    const int yo[3] = {y * nx, (y > 0 ? y - 1 : ny - 1) * nx, (y < ny - 1 ? y + 1 : 0) * nx};
    using Src = Strided<NS>;
    auto src = [&](auto ic) {
        constexpr int i = decltype(ic)::value;
        constexpr int cx = kCx(i), cy = kCy(i), cz = kCz(i);
        return Src{st + (zl + 1 - cz) * A + yo[cy > 0 ? 1 : (cy < 0 ? 2 : 0)] + xo[cx > 0 ? 1 : (cx < 0 ? 2 : 0)]};
    };
    const Src own{st + (zl + 1) * A + xy};
    const float dnr = own.template get<SQ_DN>();
    float d79, ux, uy, uz;
    pull_gather(src, own, (1.f - P.sl[s].inv_tau) / store_scale<T>(), dnr, bb, v, d79);
    const float dn =
        pull_finish<T>([&](int i, float h) { stp(IP ? pop_at_ip(pout, P, i, q.slot(i)) : pop_at(pout, P, i, idx), h); },
                       v, d79, dnr, ux, uy, uz);
    put_fields(P, io, x, y, z, dn, ux, uy, uz, status);
}

template <typename T, bool IP>
static cudaError_t pull_block(const Params& P, const void* pin, void* pout, const CsmIO& io, const float4* F,
                              int* status, cudaStream_t s)
{
    const Geom& g = P.g;
    const int A = g.nx * g.ny;
    // planes per CTA: a full CTA, fewer on small grids so that the SMs share them
    int tz = BLOCK_NT / A;
    const int share = (g.nz + 2 * NUM_SMS - 1) / (2 * NUM_SMS);
    if (tz > share) tz = share;
    const int threads = (tz * A + 31) / 32 * 32;
    const auto kernel = A <= BLOCK_A ? k_pull_block<T, IP, BLOCK_A> : k_pull_block<T, IP, BLOCK_A_MAX>;
    return launch_step(kernel, (g.nz + tz - 1) / tz, threads, 0, s, P, (const T*)pin, (T*)pout, io, F, tz, status);
}

bool csm_ok(const Geom& g) { return g.nx >= CSM_TX && g.ny >= CSM_TY; }

// z planes per segment when the caller leaves them to the library: the even
// length that minimises (waves of the NUM_SMS PAIR_MINB resident CTAs) x
// (planes + 3), the 3 standing for a segment's first two staged planes and its
// start. Large grids get 32 (512 x 512 x 192: 8 / 16 / 32 / 64 planes 2.27 /
// 2.20 / 2.19 / 2.23 ms), small ones shorter segments so that every SM has
// work (64 x 64 x 128: 4 / 8 / 16 / 32 planes 42 / 40 / 53 / 81 us). Many
// waves overlap, so above four their count is not rounded up.
static int pair_segment(long long tiles, int nz)
{
    int best = 2;
    double cost = 1e300;
    for (int lz : {2, 4, 6, 8, 12, 16, 24, 32}) {
        const double w = (double)(tiles * ((nz + lz - 1) / lz)) / (NUM_SMS * PAIR_MINB);
        const double c = (w <= 4.0 ? ceil(w) : w) * (lz + 3);
        if (c <= cost) {
            cost = c;
            best = lz;
        }
    }
    return best;
}

template <typename T, bool IP, int TX>
static cudaError_t pull_pair(const Params& P, const void* pin, void* pout, const CsmIO& io, const float4* F,
                             int* status, int lz, cudaStream_t s)
{
    const Geom& g = P.g;
    constexpr int TY = CSM_THREADS / TX;
    const int tx = (g.nx + TX - 1) / TX, ty = (g.ny + TY - 1) / TY;
    if (lz <= 0) lz = pair_segment((long long)tx * ty, g.nz);
    lz += lz & 1;  // two planes per round
    const int segs = (g.nz + lz - 1) / lz;
    const long long blocks = (long long)tx * ty * segs;
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidValue;
    const size_t smem = sizeof(float) * PAIR_FLOATS;
    // the shared-memory limit is a per-device function attribute
    static std::atomic<uint64_t> configured{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const uint64_t bit = 1ull << (dev & 63);
    if (!(configured.load() & bit)) {
        e = cudaFuncSetAttribute(k_pull_pair<T, IP, TX>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    PullPtrs pp;
    for (int i = 0; i < Q; ++i) {
        const int cz = i == 5 || i == 11 || i == 14 || i == 15 || i == 18 ? 1
                       : (i == 6 || i == 12 || i == 13 || i == 16 || i == 17 ? -1 : 0);
        const long long back = IP ? 0 : -(long long)cz * g.nx * g.ny;
        pp.src[i] = static_cast<const T*>(pin) + P.dbase[i] + back;
        pp.dst[i] = static_cast<T*>(pout) + P.dbase[i];
    }
    return launch_step(k_pull_pair<T, IP, TX>, (unsigned)blocks, CSM_THREADS, smem, s, P, pp, io, F, lz, tx, ty, status);
}

// The marched tiles' width: the one that covers the cross-section with the least work,
// a tile of 16 or 8 columns counted 1.15 and 1.4 times one of 32 (its rows are
// 64 or 32 bytes a warp load). With 32 / 16 / 8 columns: 203 x 117 x 75 112 / 121
// / 154 us, a stack of 100 slits of 33 x 35 485 / 424 / 489 us, 7 x 300 x 100 50 /
// 31 / 25 us, 100 slits of 48 x 24 (FP16 in place) 332 / 264 / 368 us.
struct PairTiles {
    int width;
    long long nodes;  // that the tiles hold per plane
};
static PairTiles pair_tiles(const Geom& g)
{
    const int w[] = {32, 16, 8};
    const double f[] = {1.0, 1.15, 1.4};
    PairTiles best{32, 0};
    double cost = 1e300;
    for (int k = 0; k < 3; ++k) {
        const int ty = CSM_THREADS / w[k];
        const long long n = (long long)((g.nx + w[k] - 1) / w[k]) * ((g.ny + ty - 1) / ty);
        if (f[k] * n < cost) {
            cost = f[k] * n;
            best = PairTiles{w[k], n * CSM_THREADS};
        }
    }
    return best;
}

template <typename T, bool IP>
static cudaError_t pull_any(const Params& P, const void* pin, void* pout, const CsmIO& io, const float4* F,
                            int* status, int lz, cudaStream_t s)
{
    const long long A = (long long)P.g.nx * P.g.ny;
    const PairTiles tiles = pair_tiles(P.g);
    if (A <= BLOCK_A || (A <= BLOCK_A_MAX && 2 * tiles.nodes > 3 * A))
        return pull_block<T, IP>(P, pin, pout, io, F, status, s);
    switch (tiles.width) {
    case 32: return pull_pair<T, IP, 32>(P, pin, pout, io, F, status, lz, s);
    case 16: return pull_pair<T, IP, 16>(P, pin, pout, io, F, status, lz, s);
    default: return pull_pair<T, IP, 8>(P, pin, pout, io, F, status, lz, s);
    }
}

template <typename T, bool IP, bool PF>
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
        e = cudaFuncSetAttribute(k_csm<T, IP, PF>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        configured.fetch_or(bit);
    }
    k_csm<T, IP, PF><<<(unsigned)blocks, CSM_THREADS, smem, s>>>(P, (const T*)pin, (T*)pout, io, F, lz, tx, ty, status);
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

// Wide slits of few planes: most of their rounds of two planes touch a wall, where the
// pair form steps one node after the other, and one plane a round is faster (not
// with FP16 in two buffers, whose gathers cost that form more): prefetched, or (2)
// plain on the widest with FP32 in two buffers. Microseconds with pairs / prefetched /
// plain, FP32: 1000 x 1000 x 4 273 / 253 / 236, x 8 478 / 456 / 432, x 16 849 / 872 / 830,
// 300 x 300 x 4 38.7 / 29.1 / 31.1, x 8 57 / 58 / 61; 64 x 64 x 4 14 / 21. In place: 1000 x 1000 x 8
// FP32 480 / 420, FP16 472 / 431, x 16 861 / 830, 836 / 830. FP16 in two buffers x 8
// 463 / 482 / 528.
enum { LOW_NONE = 0, LOW_PREFETCHED = 1, LOW_PLAIN = 2 };
static int low_slit(const Params& P)
{
    const Geom& g = P.g;
    if (!csm_ok(g) || P.nslits > 1 || (P.storage == LBIF_STORE_F16 && !P.inplace)) return LOW_NONE;
    const long long tiles = (long long)((g.nx + CSM_TX - 1) / CSM_TX) * ((g.ny + CSM_TY - 1) / CSM_TY);
    if (tiles >= 4096) return g.nz > 16 ? LOW_NONE : (P.inplace ? LOW_PREFETCHED : LOW_PLAIN);
    return tiles >= 512 && g.nz <= 6 ? LOW_PREFETCHED : LOW_NONE;
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
    const int low = prefetch == 1 ? LOW_NONE : low_slit(P);
    if ((prefetch == 1 && csm_ok(g)) || low != LOW_NONE) {
        if (lz <= 0) lz = CSM_LZ;
        if (h16)
            return ip ? csm_tiled<__half, true, true>(P, pin, pout, io, F, status, lz, s)
                      : csm_tiled<__half, false, true>(P, pin, pout, io, F, status, lz, s);
        if (ip) return csm_tiled<float, true, true>(P, pin, pout, io, F, status, lz, s);
        return low == LOW_PLAIN ? csm_tiled<float, false, false>(P, pin, pout, io, F, status, lz, s)
                                : csm_tiled<float, false, true>(P, pin, pout, io, F, status, lz, s);
    }
    if (h16)
        return ip ? pull_any<__half, true>(P, pin, pout, io, F, status, lz, s)
                  : pull_any<__half, false>(P, pin, pout, io, F, status, lz, s);
    return ip ? pull_any<float, true>(P, pin, pout, io, F, status, lz, s)
              : pull_any<float, false>(P, pin, pout, io, F, status, lz, s);
}

}  // namespace lbif
