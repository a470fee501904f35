// elbm_adjoint.cuh -- reverse-mode derivative (vector-Jacobian product) of one
// node's collision f* = f + alpha(f) beta (f^eq(f) - f) (Eq. fstar_def), with
// alpha from the closed form of Sec. III / Appendix C-D differentiated through
// every intermediate: the sign-split sums, alpha_Lower, the bound h, the
// coefficient a, and the positivity clamp.
//
// The paper defines no adjoint; this is the chain rule written out by hand.
// Membership in Omega+ / Omega- is held fixed (each restricted term is O(x^3),
// so the sums are twice differentiable across x = 0); the cutoff and the clamp
// are branches, differentiated on the side the forward pass took.
//
// node_vjp is the general form (FP64, and FP32 nodes whose |x|max is beyond the power
// series); node_vjp_series the FP32 form of all other nodes, which is what a flow has.
#pragma once

#include "elbm_device.cuh"

namespace eelbm {

// Positive root R(a, b, c) = 2c / (b + sqrt(b^2 - 4ac)) and its partials.
template <class T>
struct RootGrad {
    T r, ra, rb, rc;
};

template <class T>
__device__ __forceinline__ RootGrad<T> root_grad(T a, T b, T c)
{
    const T Dsc = sqrt(b * b - T(4) * a * c); // >= b > 0 because a <= 0 <= c
    const T den = b + Dsc;
    const T id = T(1) / den;
    RootGrad<T> g;
    g.r = T(2) * c * id;
    g.rc = T(2) * id + T(4) * a * c * id * id / Dsc;
    g.rb = -T(2) * c * id * id * (T(1) + b / Dsc);
    g.ra = T(4) * c * c * id * id / Dsc;
    return g;
}

// h = J^T g for the collision at one node (pre-collision populations F).
// With kForce the node map is C(F) + Phi(C(F)), Phi the body-force term of
// add_force (f^eq(rho, u + F_b/rho) - f^eq(rho, u)); the incoming adjoint passes
// through Phi first, and dforce[a] receives this node's d<g, C + Phi>/dF_b,a.
template <int D, class T, bool kForce = false>
__device__ void node_vjp(const T (&F)[Lattice<D>::Q], const T (&gin0)[Lattice<D>::Q], const CollideParams &p,
                         T (&h)[Lattice<D>::Q], T *dforce = nullptr)
{
    constexpr int Q = Lattice<D>::Q;
    const T beta = beta_of<T>(p);

    // ---- forward: moments and the equilibrium (Sec. I), in the forms the step uses ----
    // Deviations from k_i T(W) (exact), drho corrected for the rest of W, r = rho W in two
    // parts, and per axis eps(c) = -t, 2t +- 3u with t = s - 1 = 3u^2/(1+s): then
    // f^eq_i = k_i r (1 + E_i) and f^eq_i - F_i = (k_i r) E_i + (k_i r - F_i) with one
    // rounding.  The same care matters here as in the step: a VJP of f^eq built on
    // rounded weights maps the conserved adjoint modes (g_i = a + c_i . m) to (1 + e)
    // times themselves, and e ~ 1e-8 per step grows over a long reverse sweep.
    T dev[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) dev[i] = F[i] - T(weight_k(D, i)) * T(weight_unit(D));
    T drho = T(0), j[D];
#pragma unroll
    for (int a = 0; a < D; ++a) j[a] = T(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        drho += dev[i];
#pragma unroll
        for (int a = 0; a < D; ++a) j[a] += T(vel(D, i, a)) * dev[i];
    }
    drho -= T(double(Q == 9 ? 36 : 216) * double(weight_unit_lo<D, T>()));
    const T rho = T(1) + drho;
    const T irho = T(1) / rho;
    const T rW = fma(rho, T(weight_unit(D)), rho * weight_unit_lo<D, T>());
    // eps[a][c+1] and its derivative d eps / d u_a: 6u/s - 3, -3u/s, 6u/s + 3
    T u[D], eps[D][3], deps[D][3];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        u[a] = j[a] * irho;
        const T sq = sqrt(T(1) + T(3) * u[a] * u[a]);
        const T t = T(3) * u[a] * u[a] / (T(1) + sq);
        eps[a][0] = T(2) * t - T(3) * u[a];
        eps[a][1] = -t;
        eps[a][2] = T(2) * t + T(3) * u[a];
        const T v = T(3) * u[a] / sq;
        deps[a][0] = T(2) * v - T(3);
        deps[a][1] = -v;
        deps[a][2] = T(2) * v + T(3);
    }
    // E without axis `skip` (skip = D: all axes): prod (1 + eps) - 1, never rounding 1 + eps
    auto E_excl_at = [&](const T (&ep)[D][3], int i, int skip) -> T {
        T e = T(0);
#pragma unroll
        for (int a = 0; a < D; ++a)
            if (a != skip) {
                const T ea = ep[a][vel(D, i, a) + 1];
                e = e + ea + e * ea;
            }
        return e;
    };
    auto E_excl = [&](int i, int skip) -> T { return E_excl_at(eps, i, skip); };
    T feq[Q], x[Q], delta[Q];
    T xabs = T(0), xmin = T(0);
    int imin = 0;
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        const T kr = T(weight_k(D, i)) * rW;
        const T E = E_excl(i, D);
        delta[i] = fma(kr, E, kr - F[i]);
        feq[i] = F[i] + delta[i];
        x[i] = delta[i] / F[i];
        xabs = fmax(xabs, fabs(x[i]));
        if (x[i] < xmin) {
            xmin = x[i];
            imin = i;
        }
    }

    // ---- forward: the path length with its intermediates (Appendix D order) ----
    T alpha = T(2);
    int br = kBranchCutoff;
    T B1 = 0, C1 = 0, Cc = 0, S3 = 0, S4 = 0, S5 = 0, S6 = 0, aL = 0, kk = 0, Bp = 0, b = 0, a2 = 0, hh = 0, A = 0;
    if (p.mode != kModeLBGK && !(p.cutoff && xabs < T(kCutoff))) {
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const T xi = x[i], fx2 = F[i] * xi * xi;
            B1 += fx2;
            C1 += fx2 / (T(2) + xi);
            Cc += fx2 * (T(60) + xi * (T(60) + T(11) * xi)) / (T(60) + xi * (T(90) + xi * (T(36) + T(3) * xi)));
            if (xi < T(0)) {
                const T fx3 = fx2 * xi;
                S3 += fx3;
                S4 += fx3 * xi;
                S5 += fx3 * xi * xi;
                S6 += fx3 * xi * xi * xi;
            }
        }
        B1 *= T(0.5);
        C1 *= T(2);
        if (B1 > T(0)) {
            aL = root_grad(T(0.5) * S3, B1, C1).r;
            if (p.mode == kModeLower) {
                alpha = aL;
            } else {
                kk = p.b_variant ? aL : aL * beta;
#pragma unroll
                for (int i = 0; i < Q; ++i)
                    if (x[i] >= T(0)) {
                        const T t = kk * x[i];
                        Bp += F[i] * x[i] * x[i] * x[i] * (T(80) + t * (T(80) + T(19) * t)) /
                              (T(64) + t * (T(96) + t * (T(44) + T(6) * t)));
                    }
                b = B1 - T(2.0 / 15.0) * aL * beta * beta * Bp;
                a2 = beta * beta * S3 / T(6);
                hh = root_grad(a2, b, Cc).r;
                const T hb = hh * beta;
                A = beta * beta * (S3 / T(6) - hb * S4 / T(12) + hb * hb * S5 / T(20) - hb * hb * hb * S6 / T(5));
                alpha = root_grad(A, b, Cc).r;
            }
            br = kBranchSolved;
        }
    }
    bool clamped = false;
    if (p.mode != kModeLBGK && xmin < T(0) && alpha * beta * (-xmin) > T(1)) {
        const T amax = T(-1) / (beta * xmin);
        alpha = T(0.5) * (T(1) + amax);
        if (alpha > amax) alpha = T(0.5) * amax;
        clamped = true;
    }

    // ---- reverse: d alpha / d F into Fb (via x: xb) ----
    T Fb[Q], xb[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) Fb[i] = xb[i] = T(0);
    if (clamped) {
        // alpha = (1 + alpha_max)/2 or alpha_max/2: both carry half of d alpha_max / d x_min
        xb[imin] = T(0.5) / (beta * xmin * xmin);
    } else if (br == kBranchSolved) {
        T B1b = 0, C1b = 0, Ccb = 0, S3b = 0, S4b = 0, S5b = 0, S6b = 0, aLb = 0, Bpb = 0;
        if (p.mode == kModeLower) {
            aLb = T(1);
        } else {
            const RootGrad<T> ra = root_grad(A, b, Cc);
            const T Ab = ra.ra;
            T bb = ra.rb;
            Ccb = ra.rc;
            const T hb = hh * beta;
            const T dAdh = beta * beta * (-beta * S4 / T(12) + T(2) * hh * beta * beta * S5 / T(20) -
                                          T(3) * hh * hh * beta * beta * beta * S6 / T(5));
            const T hbar = Ab * dAdh;
            S3b += Ab * beta * beta / T(6);
            S4b += -Ab * beta * beta * hb / T(12);
            S5b += Ab * beta * beta * hb * hb / T(20);
            S6b += -Ab * beta * beta * hb * hb * hb / T(5);
            const RootGrad<T> rh = root_grad(a2, b, Cc);
            bb += hbar * rh.rb;
            Ccb += hbar * rh.rc;
            S3b += hbar * rh.ra * beta * beta / T(6);
            B1b += bb;
            aLb += -bb * T(2.0 / 15.0) * beta * beta * Bp;
            Bpb = -bb * T(2.0 / 15.0) * aL * beta * beta;
            // Omega+ Boole term: d/dF, d/dx, and through k = alpha_L beta (or alpha_L)
            T kb = T(0);
#pragma unroll
            for (int i = 0; i < Q; ++i)
                if (x[i] >= T(0)) {
                    const T xi = x[i], t = kk * xi;
                    const T N = T(80) + t * (T(80) + T(19) * t), Np = T(80) + T(38) * t;
                    const T M = T(64) + t * (T(96) + t * (T(44) + T(6) * t));
                    const T Mp = T(96) + t * (T(88) + T(18) * t);
                    const T Bv = N / M, Bd = (Np * M - N * Mp) / (M * M);
                    const T x3 = xi * xi * xi;
                    Fb[i] += Bpb * x3 * Bv;
                    xb[i] += Bpb * F[i] * (T(3) * xi * xi * Bv + x3 * Bd * kk);
                    kb += Bpb * F[i] * x3 * Bd * xi;
                }
            aLb += kb * (p.b_variant ? T(1) : beta);
        }
        // alpha_Lower = R(S3/2, B1, C1)
        const RootGrad<T> rl = root_grad(T(0.5) * S3, B1, C1);
        S3b += aLb * rl.ra * T(0.5);
        B1b += aLb * rl.rb;
        C1b = aLb * rl.rc;
        // the sums: B1 = 1/2 <F,x^2>, C1 = 2 <F, x^2/(2+x)>, Cc = <F, x^2 P/Q>, S_k = <F, x^k>_-
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const T xi = x[i], Fi = F[i], x2 = xi * xi;
            const T P = T(60) + xi * (T(60) + T(11) * xi), Pp = T(60) + T(22) * xi;
            const T Qx = T(60) + xi * (T(90) + xi * (T(36) + T(3) * xi)), Qp = T(90) + xi * (T(72) + T(9) * xi);
            const T r = x2 * P / Qx;
            const T rp = (T(2) * xi * P + x2 * Pp) / Qx - x2 * P * Qp / (Qx * Qx);
            const T q = T(2) + xi;
            Fb[i] += B1b * T(0.5) * x2 + C1b * T(2) * x2 / q + Ccb * r;
            xb[i] += B1b * Fi * xi + C1b * Fi * (T(8) * xi + T(2) * x2) / (q * q) + Ccb * Fi * rp;
            if (xi < T(0)) {
                const T x3 = x2 * xi;
                Fb[i] += S3b * x3 + S4b * x3 * xi + S5b * x3 * x2 + S6b * x3 * x2 * xi;
                xb[i] += Fi * (T(3) * S3b * x2 + T(4) * S4b * x3 + T(5) * S5b * x3 * xi + T(6) * S6b * x3 * x2);
            }
        }
    }
    // x_i = f^eq_i / F_i - 1 and the equilibrium's dependence on F through (rho, u)
    T lam[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        Fb[i] += -xb[i] * feq[i] / (F[i] * F[i]);
        lam[i] = xb[i] / F[i];
    }
    // VJP of f^eq = rho W k_i prod_a (1 + eps_a(c_ia; v)) at a velocity v = (j + F_b)/rho
    // (F_b = 0: v = u):
    //   sum_i l_i d feq_i / d F_j = G_rho + sum_a G_a (c_ja - v_a) / rho,
    //   G_rho = sum_i l_i feq_i / rho,
    //   G_a = sum_i l_i (k_i r) eps_a'(c_ia) prod_{b != a} (1 + eps_b(c_ib)).
    auto feq_vjp_at = [&](const T (&l)[Q], T (&out)[Q], const T (&ep)[D][3], const T (&dep)[D][3],
                          const T (&vv)[D], const T (&fq)[Q], T (&Ga)[D]) {
        T Gr = T(0);
#pragma unroll
        for (int a = 0; a < D; ++a) Ga[a] = T(0);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            Gr += l[i] * fq[i];
            const T lk = l[i] * (T(weight_k(D, i)) * rW);
#pragma unroll
            for (int a = 0; a < D; ++a) {
                const T q = lk * dep[a][vel(D, i, a) + 1];
                Ga[a] += fma(q, E_excl_at(ep, i, a), q);
            }
        }
        Gr *= irho;
        T base = Gr;
#pragma unroll
        for (int a = 0; a < D; ++a) base -= Ga[a] * vv[a] * irho;
#pragma unroll
        for (int jj = 0; jj < Q; ++jj) {
            T v = base;
#pragma unroll
            for (int a = 0; a < D; ++a) v += Ga[a] * T(vel(D, jj, a)) * irho;
            out[jj] = v;
        }
    };
    auto feq_vjp = [&](const T (&l)[Q], T (&out)[Q]) {
        T Ga[D];
        feq_vjp_at(l, out, eps, deps, u, feq, Ga);
    };
    T V[Q];
    feq_vjp(lam, V);
#pragma unroll
    for (int i = 0; i < Q; ++i) Fb[i] += V[i]; // Fb = d alpha / d F

    // ---- the body-force term: gin = (I + dPhi/df*)^T gin0, and d/dF_b ----
    T gin[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) gin[i] = gin0[i];
    if constexpr (kForce) {
        T v[D], epv[D][3], depv[D][3], feqv[Q], Gv[D], Gu[D], Vv[Q], Vu[Q];
#pragma unroll
        for (int a = 0; a < D; ++a) {
            v[a] = u[a] + T(p.force[a]) * irho;
            const T sq = sqrt(T(1) + T(3) * v[a] * v[a]);
            const T t = T(3) * v[a] * v[a] / (T(1) + sq);
            epv[a][0] = T(2) * t - T(3) * v[a];
            epv[a][1] = -t;
            epv[a][2] = T(2) * t + T(3) * v[a];
            const T dv = T(3) * v[a] / sq;
            depv[a][0] = T(2) * dv - T(3);
            depv[a][1] = -dv;
            depv[a][2] = T(2) * dv + T(3);
        }
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            const T kr = T(weight_k(D, i)) * rW;
            feqv[i] = fma(kr, E_excl_at(epv, i, D), kr);
        }
        feq_vjp_at(gin0, Vv, epv, depv, v, feqv, Gv);
        feq_vjp_at(gin0, Vu, eps, deps, u, feq, Gu);
#pragma unroll
        for (int i = 0; i < Q; ++i) gin[i] += Vv[i] - Vu[i];
        if (dforce) {
#pragma unroll
            for (int a = 0; a < D; ++a) dforce[a] += Gv[a] * irho; // d v_a / d F_b,a = 1/rho
        }
    }

    // ---- the collision's VJP: h_j = g_j + beta (s dalpha/dF_j + alpha (feq_vjp(g)_j - g_j)) ----
    T s = T(0);
#pragma unroll
    for (int i = 0; i < Q; ++i) s += gin[i] * delta[i];
    feq_vjp(gin, V);
#pragma unroll
    for (int i = 0; i < Q; ++i) h[i] = gin[i] + beta * (s * Fb[i] + alpha * (V[i] - gin[i]));
}

// ---------------------------------------------------------------------------
// FP32 vector-Jacobian product of one node's collision where |x|max < kSeriesX.
//
// There alpha depends on the populations through the power sums M_k = <f, x^k> and, over
// Omega-, S_k alone (node_collide_pairs), so with the adjoints m_k and s_k of the sums
//   P(x) = sum_k m_k x^k + [x < 0] sum_k s_k x^k,   d alpha / d f_i = P(x_i) + f_i P'(x_i) dx_i/df_i + ...,
// and as x_i = feq_i / f_i - 1 the derivative with respect to f_i at fixed feq is
//   q_i = P(x_i) - (1 + x_i) P'(x_i),
// and that with respect to feq_i is P'(x_i): no division per population.  The VJP of feq is
// linear, so the whole product needs it once, applied to l_i = s P'(x_i) + alpha g_i with
// s = <g, feq - f>:
//   h_j = g_j + beta (s q_j - alpha g_j + V(l)_j).
// V is separable: per axis a line (l_-, l_0, l_+) with d = l_+ - l_-, w = 2 (l_+ + l_-) - 4 l_0
// contracts with 1 + eps to (l_+ + l_- + 4 l_0) + 3u d + t w, and with d eps / du to
// 3 d + (3u/s) w (eps = -t, 2t -+ 3u; the weights' 4 for the rest component included), so that
// 1 + eps is never rounded, and
//   V_j = 6^-D (C_0 + sum_a C_a (c_ja - u_a)),
// C_0 the full contraction and C_a the one with axis a differentiated: 160 operations where
// the products written out per population take over 1000.
// ---------------------------------------------------------------------------
struct AxisVjp {
    float u, t, v; // velocity, t = sqrt(1 + 3u^2) - 1, v = 3u / sqrt(1 + 3u^2)
};
__device__ __forceinline__ AxisVjp axis_vjp(float u)
{
    const float uu3 = 3.0f * u * u, s = sqrt_(1.0f + uu3);
    return {u, div_(uu3, 1.0f + s), 3.0f * u * rcp_(s)};
}
// One line along an axis against 1 + eps (returned) and against d eps / du (*du, may be null).
__device__ __forceinline__ float line_vjp(float lm, float l0, float lp, const AxisVjp &a, float *du)
{
    const float c0 = 4.0f * l0, d = lp - lm, sg = lp + lm, w = fmaf(2.0f, sg, -c0);
    if (du) *du = fmaf(3.0f, d, a.v * w);
    return (sg + c0) + fmaf(3.0f * a.u, d, a.t * w);
}
// C[0] = sum_i l_i k_i prod (1 + eps), C[1 + a] with axis a differentiated.
template <int D>
__device__ __forceinline__ void feq_contract(const float (&l)[Lattice<D>::Q], const AxisVjp (&ax)[D], float (&C)[D + 1])
{
    constexpr int P = Lattice<D>::Q / 3;
    float A[P], Ad[P]; // contracted along the last axis
#pragma unroll
    for (int k = 0; k < P; ++k) A[k] = line_vjp(l[3 * k], l[3 * k + 1], l[3 * k + 2], ax[D - 1], &Ad[k]);
    if constexpr (D == 2) {
        C[0] = line_vjp(A[0], A[1], A[2], ax[0], &C[1]);
        C[2] = line_vjp(Ad[0], Ad[1], Ad[2], ax[0], nullptr);
    } else {
        float B[3], By[3], Bz[3];
#pragma unroll
        for (int x = 0; x < 3; ++x) {
            B[x] = line_vjp(A[3 * x], A[3 * x + 1], A[3 * x + 2], ax[1], &By[x]);
            Bz[x] = line_vjp(Ad[3 * x], Ad[3 * x + 1], Ad[3 * x + 2], ax[1], nullptr);
        }
        C[0] = line_vjp(B[0], B[1], B[2], ax[0], &C[1]);
        C[2] = line_vjp(By[0], By[1], By[2], ax[0], nullptr);
        C[D] = line_vjp(Bz[0], Bz[1], Bz[2], ax[0], nullptr);
    }
}
// V_j = base + sum_a c_ja step_a of the contraction C (6^-D in two parts).
template <int D>
__device__ __forceinline__ void feq_vjp_terms(const float (&C)[D + 1], const AxisVjp (&ax)[D], float &base, float (&step)[D])
{
    constexpr float W = float(weight_unit(D)), Wl = weight_unit_lo<D, float>();
    base = fmaf(C[0], W, C[0] * Wl);
#pragma unroll
    for (int a = 0; a < D; ++a) {
        step[a] = fmaf(C[1 + a], W, C[1 + a] * Wl);
        base = fmaf(-step[a], ax[a].u, base);
    }
}
// The positive root of quad_root with its partial derivatives, scaled by b alike.
__device__ __forceinline__ RootGrad<float> root_grad_scaled(float a, float b, float c)
{
    const float rb = rcp_(b), q = c * rb, p = a * rb;
    const float w = sqrt_(fmaf(-4.0f * p, q, 1.0f)), rd = rcp_(1.0f + w), k = 4.0f * q * rd * rd * rcp_(w);
    const float dq = fmaf(k, p, 2.0f * rd), dp = k * q;
    return {2.0f * q * rd, dp * rb, -(q * dq + p * dp) * rb, dq * rb};
}

// F: populations, g: dL/df*; h receives dL/dF.  Returns false (h untouched) where the node
// needs node_vjp.  kForce as in node_vjp.
template <int D, bool kForce = false>
__device__ __forceinline__ bool node_vjp_series(const float (&F)[Lattice<D>::Q], float (&g)[Lattice<D>::Q],
                                                const CollideParams &p, float (&h)[Lattice<D>::Q], float *dforce = nullptr)
{
    constexpr int Q = Lattice<D>::Q, NP = Pairs<D>::NP;
    const float beta = p.beta_f;
    // moments from the deviations F_i - k_i W (as node_collide)
    float drho, j[D];
    {
        float s0[Q / 3], s1[Q / 3];
#pragma unroll
        for (int k = 0; k < Q / 3; ++k) {
            float d[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) d[c] = F[3 * k + c] - float(weight_k(D, 3 * k + c)) * float(weight_unit(D));
            s0[k] = (d[0] + d[2]) + d[1];
            s1[k] = d[2] - d[0];
        }
        if constexpr (D == 2) {
            drho = s0[0] + s0[1] + s0[2];
            j[0] = s0[2] - s0[0];
            j[1] = s1[0] + s1[1] + s1[2];
        } else {
            float t[3], ty[3], tz[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                t[a] = s0[3 * a] + s0[3 * a + 1] + s0[3 * a + 2];
                ty[a] = s0[3 * a + 2] - s0[3 * a];
                tz[a] = s1[3 * a] + s1[3 * a + 1] + s1[3 * a + 2];
            }
            drho = t[0] + t[1] + t[2];
            j[0] = t[2] - t[0];
            j[1] = ty[0] + ty[1] + ty[2];
            j[D - 1] = tz[0] + tz[1] + tz[2];
        }
    }
    drho -= float(double(Q == 9 ? 36 : 216) * double(weight_unit_lo<D, float>()));
    const float rho = 1.0f + drho, irho = rcp_nr(rho);
    const float r = fmaf(rho, float(weight_unit(D)), rho * weight_unit_lo<D, float>());
    AxisVjp ax[D];
    float eps[D][3];
#pragma unroll
    for (int a = 0; a < D; ++a) {
        ax[a] = axis_vjp(j[a] * irho);
        eps[a][0] = fmaf(-3.0f, ax[a].u, 2.0f * ax[a].t);
        eps[a][1] = -ax[a].t;
        eps[a][2] = fmaf(3.0f, ax[a].u, 2.0f * ax[a].t);
    }
    // departures, in pairs (node_collide_pairs)
    float2 f[NP], x[NP];
    float xabs = 0.0f;
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int m = pair_axis(D, k), i0 = pair_pop(D, k, 0), i1 = pair_pop(D, k, 1);
        f[k] = f2(F[i0], i1 >= 0 ? F[i1] : 1.0f);
        float G = 0.0f;
        bool first = true;
#pragma unroll
        for (int a = 0; a < D; ++a) {
            if (a == m) continue;
            const float e = eps[a][vel(D, i0, a) + 1];
            G = first ? e : G + e + G * e;
            first = false;
        }
        float2 E = f2(G, 0.0f);
        if (m >= 0) {
            const float2 em = f2(eps[m][0], eps[m][2]);
            E = pfma(f2(G), em, padd(f2(G), em));
        }
        const float2 kr = pmul(f2(kpair<D>(k, 0), kpair<D>(k, 1)), f2(r));
        float2 delta = pfma(kr, E, psub(kr, f[k]));
        if (m < 0) delta.y = 0.0f; // padding lane
        x[k] = pmul(delta, prcp(f[k]));
        xabs = fmaxf(xabs, fmaxf(fabsf(x[k].x), fabsf(x[k].y)));
    }
    const bool lbgk = p.mode == kModeLBGK;
    if (!lbgk && !(xabs < kSeriesX)) return false;
    if (lbgk) { // alpha is constant: no departure enters, however small a population is next to f^eq
#pragma unroll
        for (int k = 0; k < NP; ++k) x[k] = f2(0.0f);
    }

    if constexpr (kForce) {
        // g <- (I + dPhi/df*)^T g, Phi the body-force term, and d<g, C + Phi>/dF_b
        AxisVjp av[D];
#pragma unroll
        for (int a = 0; a < D; ++a) av[a] = axis_vjp(fmaf(float(p.force[a]), irho, ax[a].u));
        float Cu[D + 1], Cv[D + 1], bu, bv, su[D], sv[D];
        feq_contract<D>(g, ax, Cu);
        feq_contract<D>(g, av, Cv);
        feq_vjp_terms<D>(Cu, ax, bu, su);
        feq_vjp_terms<D>(Cv, av, bv, sv);
#pragma unroll
        for (int i = 0; i < Q; ++i) {
            float d = bv - bu;
#pragma unroll
            for (int a = 0; a < D; ++a) d += float(vel(D, i, a)) * (sv[a] - su[a]);
            g[i] += d;
        }
        if (dforce) {
#pragma unroll
            for (int a = 0; a < D; ++a) dforce[a] += sv[a]; // G_a / rho: d v_a / d F_b,a = 1 / rho
        }
    }

    // alpha and the adjoints m_k, s_k of the power sums
    float alpha = 2.0f, m2 = 0.0f, m3 = 0.0f, m4 = 0.0f, m5 = 0.0f, m6 = 0.0f, s3 = 0.0f, s4 = 0.0f, s5 = 0.0f, s6 = 0.0f;
    if (!lbgk && !(p.cutoff && xabs < float(kCutoff))) {
        PowerSums sums;
#pragma unroll
        for (int k = 0; k < NP; ++k) sums.add(f[k], x[k]);
        const float S2 = sums.M2.x + sums.M2.y, T3 = sums.M3.x + sums.M3.y, T4 = sums.M4.x + sums.M4.y;
        const float T5 = sums.M5.x + sums.M5.y, T6 = sums.M6.x + sums.M6.y;
        const float S3 = sums.S3.x + sums.S3.y, S4 = sums.S4.x + sums.S4.y;
        const float S5 = sums.S5.x + sums.S5.y, S6 = sums.S6.x + sums.S6.y;
        const float b1 = 0.5f * S2;
        const float c1 = S2 + fmaf(T3, -0.5f, fmaf(T4, 0.25f, fmaf(T5, -0.125f, T6 * 0.0625f)));
        const float c = S2 + fmaf(T3, -0.5f, fmaf(T4, 1.0f / 3.0f, fmaf(T5, -0.25f, T6 * 0.2f)));
        if (b1 > 0.0f) {
            const RootGrad<float> rl = root_grad_scaled(0.5f * S3, b1, c1); // alpha_Lower
            float aLb = 1.0f, b1b = 0.0f, cb = 0.0f, Pb = 0.0f, kk = 0.0f;
            alpha = rl.r;
            if (p.mode != kModeLower) {
                const float bb2 = beta * beta, kap = (2.0f / 15.0f) * bb2;
                kk = p.b_variant ? rl.r : rl.r * beta;
                const float P3 = T3 - S3, P4 = T4 - S4, P5 = T5 - S5, P6 = T6 - S6;
                const float bsum = fmaf(kk, fmaf(kk, fmaf(kk, -0.25f * P6, 0.375f * P5), -0.625f * P4), 1.25f * P3);
                const float b = fmaf(-kap * rl.r, bsum, b1);
                const RootGrad<float> rh = root_grad_scaled(bb2 * (1.0f / 6.0f) * S3, b, c); // h
                const float hb = rh.r * beta;
                const float A = bb2 * fmaf(hb, fmaf(hb, fmaf(hb, -0.2f * S6, 0.05f * S5), (-1.0f / 12.0f) * S4),
                                           (1.0f / 6.0f) * S3);
                const RootGrad<float> ra = root_grad_scaled(A, b, c); // alpha_Higher
                alpha = ra.r;
                const float Ab = ra.ra * bb2;
                const float hbar = Ab * beta * fmaf(hb, fmaf(hb, -0.6f * S6, 0.1f * S5), (-1.0f / 12.0f) * S4);
                s3 = Ab * (1.0f / 6.0f) + hbar * rh.ra * bb2 * (1.0f / 6.0f);
                s4 = Ab * hb * (-1.0f / 12.0f);
                s5 = Ab * hb * hb * 0.05f;
                s6 = Ab * hb * hb * hb * -0.2f;
                const float bbar = fmaf(hbar, rh.rb, ra.rb);
                cb = fmaf(hbar, rh.rc, ra.rc);
                b1b = bbar;
                Pb = -bbar * kap * rl.r; // adjoint of bsum
                const float kb = Pb * fmaf(kk, fmaf(kk, -0.75f * P6, 0.75f * P5), -0.625f * P4);
                aLb = fmaf(-bbar * kap, bsum, kb * (p.b_variant ? 1.0f : beta));
            }
            s3 = fmaf(aLb * 0.5f, rl.ra, s3);
            b1b = fmaf(aLb, rl.rb, b1b);
            const float c1b = aLb * rl.rc;
            const float P3b = 1.25f * Pb, P4b = -0.625f * kk * Pb, P5b = 0.375f * kk * kk * Pb, P6b = -0.25f * kk * kk * kk * Pb;
            m2 = 0.5f * b1b + c1b + cb;
            m3 = P3b - 0.5f * (c1b + cb);
            m4 = P4b + 0.25f * c1b + (1.0f / 3.0f) * cb;
            m5 = P5b - 0.125f * c1b - 0.25f * cb;
            m6 = P6b + 0.0625f * c1b + 0.2f * cb;
            s3 -= P3b, s4 -= P4b, s5 -= P5b, s6 -= P6b;
        }
    }
    // s = <g, feq - f>; then l = s P'(x) + alpha g, and q in the place of x
    float2 sp = f2(0.0f);
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int i0 = pair_pop(D, k, 0), i1 = pair_pop(D, k, 1);
        sp = pfma(f2(g[i0], i1 >= 0 ? g[i1] : 0.0f), pmul(x[k], f[k]), sp);
    }
    const float s = sp.x + sp.y;
    float l[Q];
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int i0 = pair_pop(D, k, 0), i1 = pair_pop(D, k, 1);
        const float2 xk = x[k], xm = f2(fminf(xk.x, 0.0f), fminf(xk.y, 0.0f));
        const float2 x2 = pmul(xk, xk), xm2 = pmul(xm, xm);
        const float2 pm = pfma(pfma(pfma(pfma(f2(m6), xk, f2(m5)), xk, f2(m4)), xk, f2(m3)), xk, f2(m2));
        const float2 ps = pfma(pfma(pfma(f2(s6), xm, f2(s5)), xm, f2(s4)), xm, f2(s3));
        const float2 P = pfma(x2, pm, pmul(pmul(xm2, xm), ps));
        const float2 dm = pfma(pfma(pfma(pfma(f2(6.0f * m6), xk, f2(5.0f * m5)), xk, f2(4.0f * m4)), xk, f2(3.0f * m3)), xk,
                               f2(2.0f * m2));
        const float2 ds = pfma(pfma(pfma(f2(6.0f * s6), xm, f2(5.0f * s5)), xm, f2(4.0f * s4)), xm, f2(3.0f * s3));
        const float2 lam = pfma(xk, dm, pmul(xm2, ds));
        x[k] = pfma(lam, psub(f2(-1.0f), xk), P); // q
        const float2 lk = pfma(f2(s), lam, pmul(f2(alpha), f2(g[i0], i1 >= 0 ? g[i1] : 0.0f)));
        l[i0] = lk.x;
        if (i1 >= 0) l[i1] = lk.y;
    }
    float C[D + 1], base, step[D];
    feq_contract<D>(l, ax, C);
    feq_vjp_terms<D>(C, ax, base, step);
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        float V = base;
#pragma unroll
        for (int a = 0; a < D; ++a)
            if (vel(D, i, a)) V = vel(D, i, a) > 0 ? V + step[a] : V - step[a];
        const int sl = pair_slot(D, i);
        const float q = (sl & 1) ? x[sl >> 1].y : x[sl >> 1].x;
        h[i] = fmaf(beta, fmaf(s, q, fmaf(-alpha, g[i], V)), g[i]);
    }
    return true;
}

} // namespace eelbm
