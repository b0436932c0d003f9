// Hard-sphere shell force (Eq. LBHS): the per-node kernel for any even sigma and
// the vectorised one, with their launcher.
#include <utility>

#include "lbif_device.cuh"

namespace lbif {

// ---------------------------------------------------------------------------
// step 3: hard-sphere shell force, Eq. LBHS at constant T, 18-point rule.
//   T_q = A_q - (G0 + A_q) lk s_q.(u_q - u),  A_q = G_q n_q / n0 - G0
//       = G0 dq + gq (1 + dq);  the coupling product is split by axis,
//   T_q = A_q - Pa_q - Pb_q, so that parts that cancel between mirror points
//   cancel exactly before they meet the small remainder.
// ---------------------------------------------------------------------------
template <int A>
__device__ __forceinline__ const float* ufield(const Fields& f)
{
    return A == 0 ? f.ux : (A == 1 ? f.uy : f.uz);
}

// generic path: one node per thread, scalar loads (any even sigma). The x and
// y components are formed from accurate mirror differences as in the
// vectorised path below (see there).
template <int A>
__device__ __forceinline__ void axis_pair(const Params& P, const Fields& fl, int p, const float u0[3],
                                          float G0, float lk, float f[3], float* cc)
{
    const int o = P.sh.ax_nb[A], om = P.sh.ax_md[A];
    const float* uf = ufield<A>(fl);
    float dp = ldp(fl.dn + p + o), dm = ldp(fl.dn + p - o);
    float up = ldp(uf + p + o), um = ldp(uf + p - o);
    float gp = ldp(fl.dG + p + om), gm = ldp(fl.dG + p - om);
    float Ap = shell_A(dp, gp, G0), Am = shell_A(dm, gm, G0);
    const float DA = A == 2 ? Ap - Am : fmaf(G0, dp - dm, fmaf(gp - gm, 1.f + dp, gm * (dp - dm)));
    f[A] += (1.f / 30.f) * (DA - lk * ((G0 + Ap) * (up - u0[A]) - (G0 + Am) * (u0[A] - um)));
    // Eq. C2eq: sum_q W_q (G_q n_q / n0) s_q.(u_q - u)
    if (cc) *cc += (1.f / 30.f) * ((G0 + Ap) * (up - u0[A]) + (G0 + Am) * (u0[A] - um));
}

template <int PL>
__device__ __forceinline__ void diag_quartet(const Params& P, const Fields& fl, int p, const float u0[3],
                                             float G0, float lk, float f[3], float* cc)
{
    constexpr int a = PL == 2 ? 1 : 0;
    constexpr int b = PL == 0 ? 1 : 2;
    constexpr float h = 0.70710678118654752f;
    const float* fa = a == 0 ? fl.ux : fl.uy;
    const float* fb = b == 1 ? fl.uy : fl.uz;
    // corner values of member m (sa = (m & 1) ? -1 : 1, sb = (m & 2) ? -1 : 1)
    auto nb = [&](int m, int k) { return p + ((m & 1) ? -1 : 1) * P.sh.nb_a[PL][k] + ((m & 2) ? -1 : 1) * P.sh.nb_b[PL][k]; };
    auto md = [&](int m, int k) { return p + ((m & 1) ? -1 : 1) * P.sh.md_a[PL][k] + ((m & 2) ? -1 : 1) * P.sh.md_b[PL][k]; };
    if constexpr (PL == 0) {
        // relative to the node's own n and g2: every member a small deviation
        const float d0 = ldp(fl.dn + p), g0 = ldp(fl.dG + p);
        const float Aref = fmaf(G0, d0, g0 * (1.f + d0));
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const float sa = (m & 1) ? -1.f : 1.f, sb = (m & 2) ? -1.f : 1.f;
            float dl = 0.f, gl = 0.f, ua = 0.f, ub = 0.f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float w = P.sh.nb_w[PL][k], wm = P.sh.md_w[PL][k];
                dl = fmaf(w, ldp(fl.dn + nb(m, k)) - d0, dl);
                ua = fmaf(w, ldp(fa + nb(m, k)), ua);
                ub = fmaf(w, ldp(fb + nb(m, k)), ub);
                gl = fmaf(wm, ldp(fl.dG + md(m, k)) - g0, gl);
            }
            const float av = fmaf(G0 + g0, dl, gl * ((1.f + d0) + dl));
            const float GA = G0 + (Aref + av);
            const float S = fmaf(sa, ua - u0[a], sb * (ub - u0[b]));
            const float tau = av - GA * lk * h * S;
            f[a] = fmaf(sa * (h / 15.f), tau, f[a]);
            f[b] = fmaf(sb * (h / 15.f), tau, f[b]);
            if (cc) *cc += (1.f / 15.f) * (GA * h * S);
        }
        return;
    }
    // planes (x, z), (y, z): the + and - members (in-plane sign) of each z
    // side, their in-plane difference from corner differences
    float da = 0.f, db = 0.f;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const float sb = side ? -1.f : 1.f;
        const int m = 2 * side, mp = 2 * side + 1;  // in-plane sign +, -
        float dm = 0.f, dpp = 0.f, Dd = 0.f, gm = 0.f, gp = 0.f, Dg = 0.f;
        float am = 0.f, ap = 0.f, bm = 0.f, bp = 0.f, Db = 0.f;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const float w = P.sh.nb_w[PL][k], wm = P.sh.md_w[PL][k];
            const float n1 = ldp(fl.dn + nb(m, k)), n2 = ldp(fl.dn + nb(mp, k));
            const float b1 = ldp(fb + nb(m, k)), b2 = ldp(fb + nb(mp, k));
            const float g1 = ldp(fl.dG + md(m, k)), g2 = ldp(fl.dG + md(mp, k));
            dm = fmaf(w, n1, dm);
            dpp = fmaf(w, n2, dpp);
            Dd = fmaf(w, n1 - n2, Dd);
            bm = fmaf(w, b1, bm);
            bp = fmaf(w, b2, bp);
            Db = fmaf(w, b1 - b2, Db);
            gm = fmaf(wm, g1, gm);
            gp = fmaf(wm, g2, gp);
            Dg = fmaf(wm, g1 - g2, Dg);
            am = fmaf(w, ldp(fa + nb(m, k)), am);
            ap = fmaf(w, ldp(fa + nb(mp, k)), ap);
        }
        const float Am = shell_A(dm, gm, G0), Ap = shell_A(dpp, gp, G0);
        const float DA = fmaf(G0, Dd, fmaf(Dg, 1.f + dm, gp * Dd));
        const float c1 = (G0 + Am) * lk * h, c2 = (G0 + Ap) * lk * h, Dc = DA * lk * h;
        const float xm = am - u0[a], xp = ap - u0[a], zm = bm - u0[b], zp = bp - u0[b];
        da += DA - fmaf(c1, xm, c2 * xp) - sb * fmaf(c1, Db, Dc * zp);
        db += sb * ((Am + Ap) - fmaf(c1, xm, -c2 * xp) - sb * fmaf(c1, zm, c2 * zp));
        if (cc) *cc += (1.f / 15.f) * h * ((G0 + Am) * (xm + sb * zm) + (G0 + Ap) * (-xp + sb * zp));
    }
    f[a] += (h / 15.f) * da;
    f[b] += (h / 15.f) * db;
}

__device__ __forceinline__ float coupling_factor(const Params& P, const SlitParam& S, int z)
{
    if (!P.coupling) return 0.f;
    float lam = 1.f;
    if (P.regularize && !P.g.zper) {
        float dw = fminf(z - S.zlo + 0.5f, S.zhi + 0.5f - z);
        lam = 1.f - expf(-dw * P.inv_sigma);
    }
    return lam * P.kappa;
}

// total force F / n0 at a node (body + hard sphere + tail), and the energy
// source of Eq. C2eq over n0 when it is on (0 otherwise)
__device__ __forceinline__ void node_force(const Params& P, const SlitParam& S, const Fields& fl,
                                           const float4* Ft, long long idx, int z,
                                           int p, float& fx, float& fy, float& fz, float& c2)
{
    const float d0 = ldp(fl.dn + p);
    const float u0[3] = {ldp(fl.ux + p), ldp(fl.uy + p), ldp(fl.uz + p)};
    float opd = 1.f + d0;
    fx = opd * S.body[0];
    fy = opd * S.body[1];
    fz = opd * S.body[2];
    c2 = 0.f;
    if (P.hs) {
        const float lk = coupling_factor(P, S, z);
        const float G0 = S.G0;
        float f[3] = {0.f, 0.f, 0.f};
        float cc = 0.f;
        float* pc = P.c2 ? &cc : nullptr;
        axis_pair<0>(P, fl, p, u0, G0, lk, f, pc);
        axis_pair<1>(P, fl, p, u0, G0, lk, f, pc);
        axis_pair<2>(P, fl, p, u0, G0, lk, f, pc);
        diag_quartet<0>(P, fl, p, u0, G0, lk, f, pc);
        diag_quartet<1>(P, fl, p, u0, G0, lk, f, pc);
        diag_quartet<2>(P, fl, p, u0, G0, lk, f, pc);
        float pre = S.hs_pref * opd;
        fx += pre * f[0];
        fy += pre * f[1];
        fz += pre * f[2];
        // C2 / n0 = -(kT sigma^2 4 pi n0 / 2) (1 + dn) sum_q W_q (G_q n_q / n0) s_q.(u_q - u)
        if (P.c2) c2 = 0.5f * pre * cc;
    }
    if (P.tail) {
        float4 t = Ft[idx];
        fx += t.x;
        fy += t.y;
        fz += t.z;
    }
}

// Four CTAs per SM (64 registers, no spills): 128^3 at sigma 18 144 -> 131 us, and without
// the hard spheres 337 x 24 x 211 27.4 -> 23.0, against 76 registers; five (48, spills) 150.
__global__ void __launch_bounds__(256, 4) k_force(Params P, TileMap tm, Fields fl,
                                                  const float4* Ft, float4* __restrict__ F)
{
    step_begin(P);
    const Geom& g = P.g;
    int x, y, z;
    if (tm.flat) {
        if (!flat_node(g, tm, 1, x, y, z)) return;
    } else {
        int tx, ty;
        if (!tile_origin(g, tm, tx, ty, z)) return;
        x = tx * tm.tx + threadIdx.x % 32;
        y = ty * tm.ty + threadIdx.x / 32;
        if (x >= g.nx || y >= g.ny) return;
    }
    const int s = slit_of(P, z);
    if (s < 0 || frozen(P, s)) return;
    const long long idx = ((long long)z * g.ny + y) * g.nx + x;
    const SlitParam S = P.sl[s];
    float fx, fy, fz, c2;
    node_force(P, S, fl, Ft, idx, z, pidx(g, x, y, z), fx, fy, fz, c2);
    F[idx] = make_float4(fx, fy, fz, c2);
}

// ---- vectorised path: four consecutive x nodes per thread, float4 loads ----
// (sigma a template parameter, so the x offsets and the window alignments are
// compile-time constants; the y / z strides are runtime)
typedef float v4[4];

__host__ __device__ constexpr int floor4(int d) { return d >= 0 ? (d / 4) * 4 : -(((-d) + 3) / 4) * 4; }

__device__ __forceinline__ void set4(v4 r, float4 a)
{
    r[0] = a.x;
    r[1] = a.y;
    r[2] = a.z;
    r[3] = a.w;
}

// Paired FP32 arithmetic on nodes (j, j + 1) of a v4: one instruction does
// both nodes (fma / add / mul .f32x2, sm_100 and later); each component
// rounds as the scalar operation does.
__device__ __forceinline__ float2 p2(const v4 r, int j) { return make_float2(r[j], r[j + 1]); }
__device__ __forceinline__ void put2(v4 r, int j, float2 v)
{
    r[j] = v.x;
    r[j + 1] = v.y;
}
// shell_A of a pair: G0 dq + gq (1 + dq)
__device__ __forceinline__ float2 shell_A2(float2 dq, float2 gq, float G0)
{
    return fma2(bc2(G0), dq, mul2(gq, add2(bc2(1.f), dq)));
}

// values at x offsets D..D+3 of a float4-aligned base
template <int D>
__device__ __forceinline__ void win(const float* f, int b, v4 r)
{
    constexpr int B4 = floor4(D), RR = D - B4;
    if constexpr (RR == 0) {
        set4(r, ld4(f + b + B4));
    } else {
        const float4 A = ld4(f + b + B4), C = ld4(f + b + B4 + 4);
        const float t[8] = {A.x, A.y, A.z, A.w, C.x, C.y, C.z, C.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) r[j] = t[RR + j];
    }
}

// Lanes of a warp in the tiled mapping: the warp is one y row, lane l holds
// the 4-node block at x0 + 4 l, so the value just past (before) a lane's float4
// is the next (previous) lane's first (last) one. hi / lo: this lane loads it
// itself (the last live lane of the row / the first lane).
struct Lanes {
    bool hi, lo;
};

// windows at x offsets D and D + 1 (the two corners along x), sharing loads.
// With LN the fifth value comes from the neighbouring lane by a shuffle, so a
// window costs the float4's wavefronts only (a strided scalar load costs as
// many again).
template <int D, bool LN>
__device__ __forceinline__ void win2(const float* f, int b, v4 w0, v4 w1, Lanes ln)
{
    constexpr int RR = D - floor4(D);
    if constexpr (RR == 0) {
        const float4 A = ld4(f + b + D);
        float s = 0.f;
        if constexpr (LN) s = __shfl_down_sync(0xffffffffu, A.x, 1);
        if (!LN || ln.hi) s = ldp(f + b + D + 4);
        set4(w0, A);
        w1[0] = A.y;
        w1[1] = A.z;
        w1[2] = A.w;
        w1[3] = s;
    } else if constexpr (RR == 3) {
        const float4 C = ld4(f + b + D + 1);
        float s = 0.f;
        if constexpr (LN) s = __shfl_up_sync(0xffffffffu, C.w, 1);
        if (!LN || ln.lo) s = ldp(f + b + D);
        w0[0] = s;
        w0[1] = C.x;
        w0[2] = C.y;
        w0[3] = C.z;
        set4(w1, C);
    } else {
        const float4 A = ld4(f + b + D - RR), C = ld4(f + b + D - RR + 4);
        const float t[8] = {A.x, A.y, A.z, A.w, C.x, C.y, C.z, C.w};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            w0[j] = t[RR + j];
            w1[j] = t[RR + 1 + j];
        }
    }
}

// x offsets of the two corners of a member with x sign SA: SA > 0: (LO, LO+1),
// SA < 0: (-LO, -LO-1); returns the windows in corner order (ka = 0, 1)
template <int LO, int SA, bool LN>
__device__ __forceinline__ void corners_x(const float* f, int b, v4 c0, v4 c1, Lanes ln)
{
    if constexpr (SA > 0)
        win2<LO, LN>(f, b, c0, c1, ln);
    else
        win2<-LO - 1, LN>(f, b, c1, c0, ln);
}

// Mirror images along x (and y) of the shell points carry the x (y) force as
// a small difference of large values next to a wall (density layering, wall-
// normal velocity u_z ~ 0.1), so those differences are formed before any
// large value is rounded: the points of the (x, y) plane are interpolated
// relative to the node's own n and g2 values (all members then are small
// in-plane deviations), the pairs of the (x, z) and (y, z) planes that share
// the z offset as corner-by-corner differences, and the x and y axis pairs as
// differences of the loaded values. With A = G0 dq + gq (1 + dq):
//   A - A' = G0 (dq - dq') + (gq - gq') (1 + dq) + gq' (dq - dq').

// interpolants of member M of plane PL (0: (x, y), 1: (x, z); a = x) from
// its x-window corners; REF: n and g2 relative to the node's own values
template <int SIG, int PL, int M, bool LN, bool REF>
__device__ __forceinline__ void member_x(const Params& P, const Fields& fl, int pb, const v4 d0, const v4 g0, v4 dq,
                                         v4 ua, v4 ub, v4 gq, Lanes ln)
{
    constexpr int LO = cisqrt(SIG * SIG / 2), LOM = cisqrt((SIG / 2) * (SIG / 2) / 2);
    constexpr int SA = (M & 1) ? -1 : 1, SB = (M & 2) ? -1 : 1;
    const int sbs = PL == 0 ? P.g.px : P.g.px * P.g.py;
    const float* fb = PL == 0 ? fl.uy : fl.uz;
#pragma unroll
    for (int kb = 0; kb < 2; ++kb) {
        const int row = pb + SB * (LO + kb) * sbs;
        const float w0 = P.sh.nb_w[PL][2 * kb], w1 = P.sh.nb_w[PL][2 * kb + 1];
        v4 c0, c1;
        // acc += w0 (c0 - r) + w1 (c1 - r), r the reference (REF) or 0
        auto interp = [&](float a0, float a1, const v4 r, v4 acc) {
#pragma unroll
            for (int j = 0; j < 4; j += 2) {
                float2 e0 = p2(c0, j), e1 = p2(c1, j);
                if (REF && r) {
                    e0 = sub2(e0, p2(r, j));
                    e1 = sub2(e1, p2(r, j));
                }
                put2(acc, j, fma2(bc2(a1), e1, fma2(bc2(a0), e0, p2(acc, j))));
            }
        };
        corners_x<LO, SA, LN>(fl.dn, row, c0, c1, ln);
        interp(w0, w1, d0, dq);
        corners_x<LO, SA, LN>(fl.ux, row, c0, c1, ln);
        interp(w0, w1, nullptr, ua);
        corners_x<LO, SA, LN>(fb, row, c0, c1, ln);
        interp(w0, w1, nullptr, ub);
        const int mrow = pb + SB * (LOM + kb) * sbs;
        const float v0 = P.sh.md_w[PL][2 * kb], v1 = P.sh.md_w[PL][2 * kb + 1];
        corners_x<LOM, SA, LN>(fl.dG, mrow, c0, c1, ln);
        interp(v0, v1, g0, gq);
    }
}

// plane (x, y): the four members relative to the node's own n and g2 (d0,
// g0); their terms tau = T - T_ref share one reference, so both force
// components are sums of small accurate values
template <int SIG, bool C2, bool LN>
__device__ __forceinline__ void quartet_xy(const Params& P, const Fields& fl, int pb, const v4 d0, const v4 g0,
                                           const v4 u0[3], float G0, float lk, v4 f[3], v4 cc, Lanes ln)
{
    constexpr float h = 0.70710678118654752f, c = h / 15.f;
    auto one = [&](auto mc) {
        constexpr int M = decltype(mc)::value;
        constexpr float sa = (M & 1) ? -1.f : 1.f, sb = (M & 2) ? -1.f : 1.f;
        v4 dl, ua, ub, gl;
#pragma unroll
        for (int j = 0; j < 4; ++j) dl[j] = ua[j] = ub[j] = gl[j] = 0.f;
        member_x<SIG, 0, M, LN, true>(P, fl, pb, d0, g0, dl, ua, ub, gl, ln);
#pragma unroll
        for (int j = 0; j < 4; j += 2) {
            const float2 d = p2(d0, j), gg = p2(g0, j), dlj = p2(dl, j), opd = add2(bc2(1.f), d);
            const float2 Aref = fma2(bc2(G0), d, mul2(gg, opd));
            const float2 a = fma2(add2(bc2(G0), gg), dlj, mul2(p2(gl, j), add2(opd, dlj)));
            const float2 GA = add2(bc2(G0), add2(Aref, a));
            const float2 S = fma2(bc2(sa), sub2(p2(ua, j), p2(u0[0], j)), mul2(bc2(sb), sub2(p2(ub, j), p2(u0[1], j))));
            const float2 tau = fma2(mul2(GA, bc2(-lk * h)), S, a);
            put2(f[0], j, fma2(bc2(sa * c), tau, p2(f[0], j)));
            put2(f[1], j, fma2(bc2(sb * c), tau, p2(f[1], j)));
            if constexpr (C2) put2(cc, j, fma2(bc2(h / 15.f), mul2(GA, S), p2(cc, j)));
        }
    };
    one(std::integral_constant<int, 0>{});
    one(std::integral_constant<int, 1>{});
    one(std::integral_constant<int, 2>{});
    one(std::integral_constant<int, 3>{});
}

// plane (x, z) (PL 1) or (y, z) (PL 2): the two members with z offset sign SB
// and opposite in-plane sign: their interpolants d, g, ua, ub (m: +, p: -)
// and the corner-by-corner differences of d, g and ub
template <int SIG, int PL, int SB, bool LN>
__device__ __forceinline__ void pair_interp(const Params& P, const Fields& fl, int pb, v4 dm, v4 dp, v4 Dd, v4 gm,
                                            v4 gp, v4 Dg, v4 am, v4 ap, v4 bm, v4 bp, v4 Db, Lanes ln)
{
    constexpr int LO = cisqrt(SIG * SIG / 2), LOM = cisqrt((SIG / 2) * (SIG / 2) / 2);
    const float* fa = PL == 1 ? fl.ux : fl.uy;
    const int sz = P.g.px * P.g.py;
    // corner values of the + and - members of one field (accumulated with weight w)
    auto acc = [&](const float* f, const v4 cp, const v4 cm, float w, v4 im, v4 ip, v4 D) {
#pragma unroll
        for (int j = 0; j < 4; j += 2) {
            const float2 a = p2(cp, j), b = p2(cm, j), W = bc2(w);
            put2(im, j, fma2(W, a, p2(im, j)));
            put2(ip, j, fma2(W, b, p2(ip, j)));
            if (D) put2(D, j, fma2(W, sub2(a, b), p2(D, j)));
        }
    };
    if constexpr (PL == 1) {
#pragma unroll
        for (int kb = 0; kb < 2; ++kb) {
            const int row = pb + SB * (LO + kb) * sz;
            const float w0 = P.sh.nb_w[1][2 * kb], w1 = P.sh.nb_w[1][2 * kb + 1];
            v4 c0, c1, e0, e1;
            corners_x<LO, 1, LN>(fl.dn, row, c0, c1, ln);
            corners_x<LO, -1, LN>(fl.dn, row, e0, e1, ln);
            acc(fl.dn, c0, e0, w0, dm, dp, Dd);
            acc(fl.dn, c1, e1, w1, dm, dp, Dd);
            corners_x<LO, 1, LN>(fa, row, c0, c1, ln);
            corners_x<LO, -1, LN>(fa, row, e0, e1, ln);
            acc(fa, c0, e0, w0, am, ap, nullptr);
            acc(fa, c1, e1, w1, am, ap, nullptr);
            corners_x<LO, 1, LN>(fl.uz, row, c0, c1, ln);
            corners_x<LO, -1, LN>(fl.uz, row, e0, e1, ln);
            acc(fl.uz, c0, e0, w0, bm, bp, Db);
            acc(fl.uz, c1, e1, w1, bm, bp, Db);
            const int mrow = pb + SB * (LOM + kb) * sz;
            const float v0 = P.sh.md_w[1][2 * kb], v1 = P.sh.md_w[1][2 * kb + 1];
            corners_x<LOM, 1, LN>(fl.dG, mrow, c0, c1, ln);
            corners_x<LOM, -1, LN>(fl.dG, mrow, e0, e1, ln);
            acc(fl.dG, c0, e0, v0, gm, gp, Dg);
            acc(fl.dG, c1, e1, v1, gm, gp, Dg);
        }
    } else {
        const int sy = P.g.px;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int ka = k & 1, kb = k >> 1;
            const int o = pb + (LO + ka) * sy + SB * (LO + kb) * sz;
            const int om = pb - (LO + ka) * sy + SB * (LO + kb) * sz;
            const int q = pb + (LOM + ka) * sy + SB * (LOM + kb) * sz;
            const int qm = pb - (LOM + ka) * sy + SB * (LOM + kb) * sz;
            const float w = P.sh.nb_w[2][k], wm = P.sh.md_w[2][k];
            v4 c, e;
            set4(c, ld4(fl.dn + o));
            set4(e, ld4(fl.dn + om));
            acc(fl.dn, c, e, w, dm, dp, Dd);
            set4(c, ld4(fa + o));
            set4(e, ld4(fa + om));
            acc(fa, c, e, w, am, ap, nullptr);
            set4(c, ld4(fl.uz + o));
            set4(e, ld4(fl.uz + om));
            acc(fl.uz, c, e, w, bm, bp, Db);
            set4(c, ld4(fl.dG + q));
            set4(e, ld4(fl.dG + qm));
            acc(fl.dG, c, e, wm, gm, gp, Dg);
        }
    }
}

// one z side (sign SB) of plane (x, z) or (y, z): T_+ - T_- (the in-plane
// force) from the differences, SB (T_+ + T_-) (the z force) directly
template <int SIG, int PL, int SB, bool C2, bool LN>
__device__ __forceinline__ void pair_terms(const Params& P, const Fields& fl, int pb, const v4 u0[3], float G0,
                                           float lk, v4 da, v4 db, v4 cc, Lanes ln)
{
    constexpr int a = PL == 1 ? 0 : 1;
    constexpr float h = 0.70710678118654752f, sb = (float)SB;
    v4 dm, dp, Dd, gm, gp, Dg, am, ap, bm, bp, Db;
#pragma unroll
    for (int j = 0; j < 4; ++j) dm[j] = dp[j] = Dd[j] = gm[j] = gp[j] = Dg[j] = am[j] = ap[j] = bm[j] = bp[j] = Db[j] = 0.f;
    pair_interp<SIG, PL, SB, LN>(P, fl, pb, dm, dp, Dd, gm, gp, Dg, am, ap, bm, bp, Db, ln);
    const float2 one = bc2(1.f), g0 = bc2(G0), lkh = bc2(lk * h), SB2 = bc2(sb);
#pragma unroll
    for (int j = 0; j < 4; j += 2) {
        const float2 dmj = p2(dm, j), dpj = p2(dp, j), Ddj = p2(Dd, j);
        const float2 Am = shell_A2(dmj, p2(gm, j), G0), Ap = shell_A2(dpj, p2(gp, j), G0);
        const float2 DA = fma2(g0, Ddj, fma2(p2(Dg, j), add2(one, dmj), mul2(p2(gp, j), Ddj)));
        const float2 Gm = add2(g0, Am), Gp = add2(g0, Ap);
        const float2 cm = mul2(Gm, lkh), cp = mul2(Gp, lkh), Dc = mul2(DA, lkh);
        const float2 xm = sub2(p2(am, j), p2(u0[a], j)), xp = sub2(p2(ap, j), p2(u0[a], j));  // in-plane offsets
        const float2 zm = sub2(p2(bm, j), p2(u0[2], j)), zp = sub2(p2(bp, j), p2(u0[2], j));  // wall-normal offsets
        // T = A - c (s_a (u_a - u0_a) + s_b (u_z - u0_z)), s_a = +1 for m, -1 for p
        const float2 ta = sub2(sub2(DA, fma2(cm, xm, mul2(cp, xp))), mul2(SB2, fma2(cm, p2(Db, j), mul2(Dc, zp))));
        put2(da, j, add2(p2(da, j), ta));
        const float2 tb = sub2(sub2(add2(Am, Ap), sub2(mul2(cm, xm), mul2(cp, xp))),
                               mul2(SB2, fma2(cm, zm, mul2(cp, zp))));
        put2(db, j, fma2(SB2, tb, p2(db, j)));
        if constexpr (C2)
            put2(cc, j, fma2(bc2(h / 15.f), fma2(Gm, fma2(SB2, zm, xm), mul2(Gp, fma2(SB2, zp, mul2(bc2(-1.f), xp)))),
                             p2(cc, j)));
    }
}

template <int SIG, int PL, bool C2, bool LN>
__device__ __forceinline__ void quartet_z(const Params& P, const Fields& fl, int pb, const v4 u0[3], float G0,
                                          float lk, v4 f[3], v4 cc, Lanes ln)
{
    constexpr int a = PL == 1 ? 0 : 1;
    constexpr float c = 0.70710678118654752f / 15.f;
    v4 da, db;
#pragma unroll
    for (int j = 0; j < 4; ++j) da[j] = db[j] = 0.f;
    pair_terms<SIG, PL, 1, C2, LN>(P, fl, pb, u0, G0, lk, da, db, cc, ln);
    pair_terms<SIG, PL, -1, C2, LN>(P, fl, pb, u0, G0, lk, da, db, cc, ln);
#pragma unroll
    for (int j = 0; j < 4; j += 2) {
        put2(f[a], j, fma2(bc2(c), p2(da, j), p2(f[a], j)));
        put2(f[2], j, fma2(bc2(c), p2(db, j), p2(f[2], j)));
    }
}

template <int SIG, int A, bool C2>
__device__ __forceinline__ void axis4(const Params& P, const Fields& fl, int pb, const v4 u0[3], float G0, float lk,
                                      v4 f[3], v4 cc)
{
    const float* uf = ufield<A>(fl);
    v4 dp, dm, up, um, gp, gm;
    if constexpr (A == 0) {
        win<SIG>(fl.dn, pb, dp);
        win<-SIG>(fl.dn, pb, dm);
        win<SIG>(uf, pb, up);
        win<-SIG>(uf, pb, um);
        win<SIG / 2>(fl.dG, pb, gp);
        win<-SIG / 2>(fl.dG, pb, gm);
    } else {
        const int st = A == 1 ? P.g.px : P.g.px * P.g.py;
        set4(dp, ld4(fl.dn + pb + SIG * st));
        set4(dm, ld4(fl.dn + pb - SIG * st));
        set4(up, ld4(uf + pb + SIG * st));
        set4(um, ld4(uf + pb - SIG * st));
        set4(gp, ld4(fl.dG + pb + (SIG / 2) * st));
        set4(gm, ld4(fl.dG + pb - (SIG / 2) * st));
    }
#pragma unroll
    for (int j = 0; j < 4; j += 2) {
        const float2 dpj = p2(dp, j), dmj = p2(dm, j), gpj = p2(gp, j), gmj = p2(gm, j), u0j = p2(u0[A], j);
        const float2 Ap = shell_A2(dpj, gpj, G0), Am = shell_A2(dmj, gmj, G0);
        // A_+ - A_-: from the differences of the loaded values along x and y
        float2 DA;
        if constexpr (A == 2) {
            DA = sub2(Ap, Am);
        } else {
            const float2 dd = sub2(dpj, dmj);
            DA = fma2(bc2(G0), dd, fma2(sub2(gpj, gmj), add2(bc2(1.f), dpj), mul2(gmj, dd)));
        }
        const float2 wp = mul2(add2(bc2(G0), Ap), sub2(p2(up, j), u0j));
        const float2 wm = mul2(add2(bc2(G0), Am), sub2(u0j, p2(um, j)));
        put2(f[A], j, fma2(bc2(1.f / 30.f), fma2(bc2(-lk), sub2(wp, wm), DA), p2(f[A], j)));
        if constexpr (C2) put2(cc, j, fma2(bc2(1.f / 30.f), add2(wp, wm), p2(cc, j)));
    }
}

// At most 128 registers, so that 16 warps share an SM: the kernel waits on
// L1 far more than it computes, and the extra warps hide that latency
// (measured: 146 registers / 12 warps is 6 % slower). CTAs of two warps (a
// 128 x 2 tile), eight per SM (measured at sigma 12 on 512 x 512 x 192:
// 32 / 64 / 128 / 256 / 512 threads 1.658 / 1.610 / 1.631 / 1.705 / 1.820 ms).
// LN: tiled mapping with lane shuffles (every exit above the node's own
// x test is taken by whole warps; lanes past the grid's edge stay, on the
// row's first block, until the stores)
constexpr int FORCE_NT = 64;
#ifndef FORCE_MINB
#define FORCE_MINB (512 / FORCE_NT)
#endif
template <int SIG, bool C2, bool LN>
__global__ void __launch_bounds__(FORCE_NT, FORCE_MINB) k_force4(Params P, TileMap tm, Fields fl,
                                                const float4* Ft, float4* __restrict__ F)
{
    step_begin(P);
    const Geom& g = P.g;
    int x, y, z;
    bool live = true;
    Lanes ln{false, false};
    if (!LN) {
        if (!flat_node(g, tm, 4, x, y, z)) return;
    } else {
        int tx, ty;
        if (!tile_origin(g, tm, tx, ty, z)) return;
        const int x0 = tx * 128, lane = threadIdx.x % 32;
        x = x0 + 4 * lane;
        y = ty * tm.ty + threadIdx.x / 32;
        if (x0 >= g.nx || y >= g.ny) return;  // whole warp
        live = x < g.nx;
        if (!live) x = x0;
        ln.hi = lane == 31 || x + 4 >= g.nx;
        ln.lo = lane == 0;
    }
    const int s = slit_of(P, z);
    if (s < 0 || frozen(P, s)) return;  // whole warp (one z plane)
    const SlitParam S = P.sl[s];
    const int pb = pidx(g, x, y, z);  // 16-byte aligned: x, hw, px multiples of 4
    v4 d0, g0, u0[3];
    set4(d0, ld4(fl.dn + pb));
    set4(g0, ld4(fl.dG + pb));
    set4(u0[0], ld4(fl.ux + pb));
    set4(u0[1], ld4(fl.uy + pb));
    set4(u0[2], ld4(fl.uz + pb));
    v4 f[3], cc;
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int j = 0; j < 4; ++j) f[a][j] = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) cc[j] = 0.f;
    if (P.hs) {
        const float lk = coupling_factor(P, S, z);
        axis4<SIG, 0, C2>(P, fl, pb, u0, S.G0, lk, f, cc);
        axis4<SIG, 1, C2>(P, fl, pb, u0, S.G0, lk, f, cc);
        axis4<SIG, 2, C2>(P, fl, pb, u0, S.G0, lk, f, cc);
        quartet_xy<SIG, C2, LN>(P, fl, pb, d0, g0, u0, S.G0, lk, f, cc, ln);
        quartet_z<SIG, 1, C2, LN>(P, fl, pb, u0, S.G0, lk, f, cc, ln);
        quartet_z<SIG, 2, C2, LN>(P, fl, pb, u0, S.G0, lk, f, cc, ln);
    }
    if (!live) return;
    const long long idx0 = ((long long)z * g.ny + y) * g.nx + x;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (x + j >= g.nx) break;
        const float opd = 1.f + d0[j];
        const float pre = S.hs_pref * opd;
        float fx = opd * S.body[0] + pre * f[0][j];
        float fy = opd * S.body[1] + pre * f[1][j];
        float fz = opd * S.body[2] + pre * f[2][j];
        if (P.tail) {
            float4 t = Ft[idx0 + j];
            fx += t.x;
            fy += t.y;
            fz += t.z;
        }
        // energy source of Eq. C2eq over n0 (when on)
        const float c2 = C2 && P.hs ? 0.5f * pre * cc[j] : 0.f;
        F[idx0 + j] = make_float4(fx, fy, fz, c2);
    }
}

// ---------------------------------------------------------------------------
// Local pressure p = kT n + (kT sigma^3/6) 4 pi n0^2 (1 + dn) sum_q W_q (G0 + A_q),
// four consecutive x nodes per thread with the windows of the force kernel (n and
// g2 only: half of its loads). 256 x 192 x 96, sigma 8: one node per thread with
// scalar loads 159 us, so 74 us.
// ---------------------------------------------------------------------------
// acc += w0 c0 + w1 c1
__device__ __forceinline__ void lerp4(float w0, float w1, const v4 c0, const v4 c1, v4 acc)
{
#pragma unroll
    for (int j = 0; j < 4; j += 2) put2(acc, j, fma2(bc2(w1), p2(c1, j), fma2(bc2(w0), p2(c0, j), p2(acc, j))));
}
// s += W (G0 dq + gq (1 + dq))
__device__ __forceinline__ void add_A(float W, const v4 dq, const v4 gq, float G0, v4 s)
{
#pragma unroll
    for (int j = 0; j < 4; j += 2) put2(s, j, fma2(bc2(W), shell_A2(p2(dq, j), p2(gq, j), G0), p2(s, j)));
}

template <int SIG, bool LN>
__global__ void __launch_bounds__(FORCE_NT) k_pressure4(Params P, TileMap tm, Fields fl, float* __restrict__ pr)
{
    const Geom& g = P.g;
    int x, y, z;
    bool live = true;
    Lanes ln{false, false};
    if (!LN) {
        if (!flat_node(g, tm, 4, x, y, z)) return;
    } else {
        int tx, ty;
        if (!tile_origin(g, tm, tx, ty, z)) return;
        const int x0 = tx * 128, lane = threadIdx.x % 32;
        x = x0 + 4 * lane;
        y = ty * tm.ty + threadIdx.x / 32;
        if (x0 >= g.nx || y >= g.ny) return;  // whole warp
        live = x < g.nx;
        if (!live) x = x0;
        ln.hi = lane == 31 || x + 4 >= g.nx;
        ln.lo = lane == 0;
    }
    const long long idx0 = ((long long)z * g.ny + y) * g.nx + x;
    const int sl = slit_of(P, z);
    if (sl < 0) {  // whole warp in the tiled mapping (one z plane)
        if (live)
            for (int j = 0; j < 4 && x + j < g.nx; ++j) pr[idx0 + j] = 0.f;
        return;
    }
    const SlitParam S = P.sl[sl];
    const int pb = pidx(g, x, y, z), sy = g.px, sz = g.px * g.py;
    v4 d0, s;
    set4(d0, ld4(fl.dn + pb));
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] = 0.f;
    if (P.hs) {
        constexpr int LO = cisqrt(SIG * SIG / 2), LOM = cisqrt((SIG / 2) * (SIG / 2) / 2);
        v4 d, q;
        win<SIG>(fl.dn, pb, d);
        win<SIG / 2>(fl.dG, pb, q);
        add_A(1.f / 30.f, d, q, S.G0, s);
        win<-SIG>(fl.dn, pb, d);
        win<-SIG / 2>(fl.dG, pb, q);
        add_A(1.f / 30.f, d, q, S.G0, s);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int st = ((k & 1) ? -1 : 1) * ((k & 2) ? sz : sy);
            set4(d, ld4(fl.dn + pb + SIG * st));
            set4(q, ld4(fl.dG + pb + SIG / 2 * st));
            add_A(1.f / 30.f, d, q, S.G0, s);
        }
        // planes (x, y) and (x, z): corners along x from the windows
        auto member = [&](auto plc, auto sac, int sb) {
            constexpr int PL = decltype(plc)::value, SA = decltype(sac)::value;
            const int st = sb * (PL == 0 ? sy : sz);
            v4 dq, gq, c0, c1;
#pragma unroll
            for (int j = 0; j < 4; ++j) dq[j] = gq[j] = 0.f;
#pragma unroll
            for (int kb = 0; kb < 2; ++kb) {
                corners_x<LO, SA, LN>(fl.dn, pb + (LO + kb) * st, c0, c1, ln);
                lerp4(P.sh.nb_w[PL][2 * kb], P.sh.nb_w[PL][2 * kb + 1], c0, c1, dq);
                corners_x<LOM, SA, LN>(fl.dG, pb + (LOM + kb) * st, c0, c1, ln);
                lerp4(P.sh.md_w[PL][2 * kb], P.sh.md_w[PL][2 * kb + 1], c0, c1, gq);
            }
            add_A(1.f / 15.f, dq, gq, S.G0, s);
        };
        using std::integral_constant;
#pragma unroll
        for (int sb = -1; sb <= 1; sb += 2) {
            member(integral_constant<int, 0>{}, integral_constant<int, 1>{}, sb);
            member(integral_constant<int, 0>{}, integral_constant<int, -1>{}, sb);
            member(integral_constant<int, 1>{}, integral_constant<int, 1>{}, sb);
            member(integral_constant<int, 1>{}, integral_constant<int, -1>{}, sb);
        }
        // plane (y, z): whole rows
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int ty = (m & 1) ? -sy : sy, tz = (m & 2) ? -sz : sz;
            v4 dq, gq, c0, c1;
#pragma unroll
            for (int j = 0; j < 4; ++j) dq[j] = gq[j] = 0.f;
#pragma unroll
            for (int kb = 0; kb < 2; ++kb) {
                set4(c0, ld4(fl.dn + pb + LO * ty + (LO + kb) * tz));
                set4(c1, ld4(fl.dn + pb + (LO + 1) * ty + (LO + kb) * tz));
                lerp4(P.sh.nb_w[2][2 * kb], P.sh.nb_w[2][2 * kb + 1], c0, c1, dq);
                set4(c0, ld4(fl.dG + pb + LOM * ty + (LOM + kb) * tz));
                set4(c1, ld4(fl.dG + pb + (LOM + 1) * ty + (LOM + kb) * tz));
                lerp4(P.sh.md_w[2][2 * kb], P.sh.md_w[2][2 * kb + 1], c0, c1, gq);
            }
            add_A(1.f / 15.f, dq, gq, S.G0, s);
        }
    }
    if (!live) return;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (x + j >= g.nx) break;
        const float q1 = 1.f + d0[j];
        pr[idx0 + j] = (1.f / 3.f) * S.rho0 * q1 + (P.hs ? (S.G0 + s[j]) * S.p_pref * q1 : 0.f);
    }
}

template <int SIG>
static void pressure4_sigma(const Params& P, const Fields& f, float* pr, cudaStream_t s)
{
    unsigned blocks;
    if (P.g.nx < 128) {
        const TileMap tm = make_flatmap(P.g, 4, FORCE_NT, blocks);
        k_pressure4<SIG, false><<<blocks, FORCE_NT, 0, s>>>(P, tm, f, pr);
    } else {
        const TileMap tm = make_tilemap(P.g, 128, FORCE_NT / 32, 128, blocks);
        k_pressure4<SIG, true><<<blocks, FORCE_NT, 0, s>>>(P, tm, f, pr);
    }
}

// Below 1024 nodes per SM the per-node kernel is the faster one: a thread's chain of
// loads is a quarter as long, and there are enough SMs for all. Microseconds per node /
// vectorised at sigma 4 and 12 on 64 x 64 x n: 10,000 nodes 7.7 / 8.5 and 8.4 / 11.5, 80,000
// 7.5 / 7.6 and 7.7 / 9.8, 160,000 11.1 / 7.8 and 11.1 / 10.0, 640,000 26.0 / 14.3 and 26.8 / 15.3.
bool launch_pressure4(const Params& P, const Fields& f, float* pr, cudaStream_t s)
{
    if (P.g.N < 1024LL * NUM_SMS) return false;
    switch (P.sigma) {
    case 4: pressure4_sigma<4>(P, f, pr, s); break;
    case 6: pressure4_sigma<6>(P, f, pr, s); break;
    case 8: pressure4_sigma<8>(P, f, pr, s); break;
    case 10: pressure4_sigma<10>(P, f, pr, s); break;
    case 12: pressure4_sigma<12>(P, f, pr, s); break;
    default: return false;
    }
    return true;
}

template <int SIG, bool LN>
static cudaError_t force4_launch(const Params& P, const TileMap& tm, const Fields& f, const float4* Ft, float4* F,
                          unsigned blocks, cudaStream_t s)
{
    return launch_step(P.c2 ? k_force4<SIG, true, LN> : k_force4<SIG, false, LN>, blocks, FORCE_NT, 0, s, P, tm, f, Ft,
                       F);
}

template <int SIG>
static cudaError_t force4_sigma(const Params& P, const Fields& f, const float4* Ft, float4* F, int group, cudaStream_t s)
{
    unsigned blocks;
    if (P.g.nx < 128) {
        const TileMap tm = make_flatmap(P.g, 4, FORCE_NT, blocks);
        return force4_launch<SIG, false>(P, tm, f, Ft, F, blocks, s);
    } else {
        const TileMap tm = make_tilemap(P.g, 128, FORCE_NT / 32, group, blocks);
        return force4_launch<SIG, true>(P, tm, f, Ft, F, blocks, s);
    }
}

// Even diameters from 4 to 12 have the vectorised kernel (an instance each, so
// that x offsets and window alignments are compile-time constants); the others
// run the per-node one. sigma 6 on 203 x 117 x 75: per node 134 us, vectorised
// 86 us.
cudaError_t launch_force(const Params& P, const Fields& f, const float4* Ft, float4* F, int group,
                         cudaStream_t s)
{
    if (group <= 0) group = 128;
    switch (P.sigma) {
    case 4: return force4_sigma<4>(P, f, Ft, F, group, s);
    case 6: return force4_sigma<6>(P, f, Ft, F, group, s);
    case 8: return force4_sigma<8>(P, f, Ft, F, group, s);
    case 10: return force4_sigma<10>(P, f, Ft, F, group, s);
    case 12: return force4_sigma<12>(P, f, Ft, F, group, s);
    default: {
        unsigned blocks;
        const TileMap tm = P.g.nx < 32 ? make_flatmap(P.g, 1, 256, blocks) : make_tilemap(P.g, 32, 8, group, blocks);
        return launch_step(k_force, blocks, 256, 0, s, P, tm, f, Ft, F);
    }
    }
}

}  // namespace lbif
