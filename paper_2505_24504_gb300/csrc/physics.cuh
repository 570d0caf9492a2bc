// Device model of Sec. 4 (eq. compressible-euler) in (rho, rho u, rho w, rho theta):
// theta-form EOS, convective flux, HLLC numerical flux, viscous flux
// F_v = mu rho (0, grad u, grad w, grad theta).  Templated on the scalar type
// (D64 for the FP64 operator, TL32 for the FP32 tangent-linear operator).
#pragma once

#include "numeric.cuh"

struct PhysC {
    double gamma, R, p0, g, mu;
    double R_over_p0;   // R / p0
    float gammaf, p0f, R_over_p0f, muf;   // float copies for the FP32 tangent
};

// p = p0 (R rho theta / p0)^gamma  (the EOS implied by eq. add-perturbation)
JF_D D64 pressure(D64 E, const PhysC &, const PowTab *pt) { return D64{eos_pow(E.x, pt)}; }
JF_D TL32 pressure(TL32 E, const PhysC &P, const PowTab *) {
    const float x = P.R_over_p0f * E.v;
    const float p = P.p0f * __powf(x, P.gammaf);
    return TL32{p, P.gammaf * p * frcp(E.v) * E.d};
}

template <class T>
JF_D T sel(bool c, T a, T b) { return c ? a : b; }

// Convective fluxes F_c(U) . e_x and F_c(U) . e_z at a node from u = U_1 / rho,
// w = U_2 / rho and p.  The mass components are U_1 and U_2 themselves; rho u w appears
// in both directions and is formed once.
template <class T>
JF_D void flux_xz(const T U[4], T u, T w, T p, T Fx[4], T Fz[4]) {
    Fx[0] = U[1];
    Fx[1] = jfma(U[1], u, p);
    Fx[2] = U[2] * u;
    Fx[3] = U[3] * u;
    Fz[0] = U[2];
    Fz[1] = Fx[2];
    Fz[2] = jfma(U[2], w, p);
    Fz[3] = U[3] * w;
}

// One side of a face: the conserved state and the quantities every face of that
// cell needs, 1/rho, p and the sound speed c = sqrt(gamma p / rho).  Cell-based
// kernels compute them once per cell instead of once per face.
template <class T>
struct Side {
    T U[4];
    T ir, p, c;
};

template <class T>
JF_D void side_of(const T U[4], const PhysC &P, const PowTab *pt, Side<T> &S) {
    const auto gam = mkc(P.gamma, P.gammaf, T{});
#pragma unroll
    for (int v = 0; v < 4; ++v) S.U[v] = U[v];
    S.ir = jrcp(U[0]);
    S.p = pressure(U[3], P, pt);
    S.c = jsqrt(gam * S.p * S.ir);
}

// slip-wall ghost of a side: normal momentum reversed, rho, p and c unchanged
template <class T, int D>
JF_D void mirror_side(const Side<T> &A, Side<T> &G) {
    G = A;
    G.U[1 + D] = -A.U[1 + D];
}

// Does S_L = u_L - c_L (S_R = u_L + c_L) hold of the Davis speeds?  FP64 compares the
// differences it has; the FP32 tangent, whose derivative jumps where the two speeds
// agree, compares the speeds themselves (a rounding of 3e-5 m/s decides either way, and
// the same way for the same states).
JF_D bool slower(D64, D64 cL, D64, D64, D64 x) { return le(-cL, x); }
JF_D bool faster(D64, D64, D64, D64 cR, D64 y) { return le(cR, y); }
JF_D bool slower(TL32 uL, TL32 cL, TL32 uR, TL32 cR, TL32) { return le(uL - cL, uR - cR); }
JF_D bool faster(TL32 uL, TL32 cL, TL32 uR, TL32 cR, TL32) { return le(uR + cR, uL + cL); }

// HLLC flux in direction e_D, normal from L to R.  Davis wave speeds
// S_L = min(u_L - c_L, u_R - c_R), S_R = max(u_L + c_L, u_R + c_R), c^2 = gamma p / rho;
// contact speed S*; star states rho*_K = rho_K (S_K - u_K)/(S_K - S*) with normal
// velocity S*, tangential velocity and theta of side K; F*_K = F_K + S_K (U*_K - U_K).
// Branches 0 <= S_L: F_L; 0 <= S*: F*_L; 0 <= S_R: F*_R; else F_R.  Only the side
// the branch selects is evaluated.
// With q_K = rho_K (S_K - u_K) the star flux is, identically, the flux of the star state
// through the contact: mass M = rho* S*, normal momentum M S* + p_K + q_K (S* - u_K),
// tangential momentum M v_t, M theta.  All speeds are taken relative to the sides, with
// d = u_R - u_L: S_L - u_L = min(-c_L, d - c_R), S_R - u_R = max(c_L - d, c_R),
// S* - u_L = ((p_R - p_L) - d q_R) / (q_L - q_R).  In this form nothing large cancels
// (F_K and S_K (U*_K - U_K) do in the textbook one), and the whole flux takes about 51
// FP64 instructions instead of 119.
// With the quotients, roots and powers of numeric.cuh the faces of the FP64 residual, then
// a launch of their own, fell from 48.6 to 28.0 us on 103,360 Q3 face points, from 46.9 to
// 26.0 us on the 50,016 viscous Q2 ones, and from 26 to 15 us where one SM's latency chain
// sets the time (20 x 10 elements, Q2).  (Faces and nodes in one launch: k_dg_flux.)
template <class T, int D>
JF_D void hllc_s(const Side<T> &L, const Side<T> &R, T H[4]) {
    constexpr int iN = 1 + D, iT = 2 - D;
    const T uL = L.U[iN] * L.ir, uR = R.U[iN] * R.ir;
    const T d = uR - uL;
    const T x = d - R.c, y = L.c - d;
    const T dL = sel(slower(uL, L.c, uR, R.c, x), -L.c, x);   // S_L - u_L
    const T dR = sel(faster(uL, L.c, uR, R.c, y), y, R.c);    // S_R - u_R
    const T qL = L.U[0] * dL, qR = R.U[0] * dR;
    const T sL = jfma(-d, qR, R.p - L.p) / (qL - qR);   // S* - u_L
    const T Sst = uL + sL;
    const bool sl = le(-dL, uL);              // 0 <= S_L
    const bool left = nonneg(Sst) || sl;
    const bool pure = sl || (!left && !le(-dR, uR));
    const T ir = sel(left, L.ir, R.ir), p = sel(left, L.p, R.p);
    const T Ut = sel(left, L.U[iT], R.U[iT]), U3 = sel(left, L.U[3], R.U[3]);
    if (pure) {
        const T Un = sel(left, L.U[iN], R.U[iN]), un = sel(left, uL, uR);
        H[0] = Un;
        H[iN] = jfma(Un, un, p);
        H[iT] = Ut * un;
        H[3] = U3 * un;
        return;
    }
    const T q = sel(left, qL, qR), s = sel(left, sL, sL - d);   // s = S* - u_K
    const T M = q / (sel(left, dL, dR) - s) * Sst;
    const T Mi = M * ir;
    H[0] = M;
    H[iN] = jfma(M, Sst, jfma(q, s, p));
    H[iT] = Mi * Ut;
    H[3] = Mi * U3;
}

template <class T, int D>
JF_D void hllc(const T UL[4], const T UR[4], const PhysC &P, const PowTab *pt, T H[4]) {
    Side<T> L, R;
    side_of(UL, P, pt, L);
    side_of(UR, P, pt, R);
    hllc_s<T, D>(L, R, H);
}

// Slip-wall ghost: normal momentum reversed.
template <class T, int D>
JF_D void mirror(const T U[4], T G[4]) {
    G[0] = U[0];
    G[1] = U[1];
    G[2] = U[2];
    G[3] = U[3];
    G[1 + D] = -U[1 + D];
}
// At a slip wall the outer state becomes the mirrored inner one (both faces' states are
// then evaluated alike: one flux evaluation serves walls and inner faces).
template <class T, int D>
JF_D void wall_states(T UL[4], T UR[4], bool wallL, bool wallR) {
    if (wallL) mirror<T, D>(UR, UL);
    if (wallR) mirror<T, D>(UL, UR);
}

// A(U) dU / mu with A = mu [[0,0,0,0],[-u,1,0,0],[-w,0,1,0],[-theta,0,0,1]]:
// rho (0, d u, d w, d theta) for dU the derivative of U along one direction; component
// v = 1, 2, 3 from phi = U_v / rho.
template <class T>
JF_D T visc_c(T phi, T dU0, T dUv) { return jfma(-phi, dU0, dUv); }

// Viscous part V of a face's term Phi = H - V, component v: the mean of the two sides'
// viscous fluxes (hmu = mu / 2, phi = U_v / rho, g the normal derivatives) less the
// interior penalty eta {A(U)} [U] on the jumps of u, w, theta (sL, sR = 1/2 A(U_side) [U]).
template <class T, class C, class E>
JF_D T visc_face(C hmu, E eta, T pL, T pR, const T gL[4], const T gR[4], int v, T sL, T sR) {
    return hmu * (visc_c(pL, gL[0], gL[v]) + visc_c(pR, gR[0], gR[v])) - eta * (sL + sR);
}

// |v . e_D| + c for pseudo-time step sizes (plain double, not on the residual path).
JF_D double wave_speed(const double U[4], int D, const PhysC &P, const PowTab *pt) {
    const double ir = 1.0 / U[0];
    const double p = eos_pow(U[3], pt);
    return fabs(U[1 + D] * ir) + sqrt(P.gamma * p * ir);
}
