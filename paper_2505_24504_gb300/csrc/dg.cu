// DG operator f = M^-1 L_h(U') on the GPU (Sec. 2.1; well-balanced form of Sec. 4).
//
// Two launches per evaluation:
//  k_dg_flux the first blocks take the face points, one thread each: traces of U' from
//            both sides (and the normal-gradient traces for the viscous terms),
//            HLLC^pert = HLLC(U'+Ubar) - HLLC(Ubar), symmetric interior penalty terms,
//            slip walls by a mirrored ghost.  Every face flux is computed once and
//            stored: Phi = H - {F_v.n} + eta [U] for the lift with l_a(+-1), and the two
//            symmetry terms 1/2 A(U_side) [U] for the lift with l_a'(+-1).  The other
//            blocks hold some elements each, one thread per node: fluxes F_c^pert - F_v,
//            the weak-form derivative by sum factorisation over the (k+1) nodes of the
//            row / column (tables in shared memory), gravity source.
//  k_dg_lift adds the lifts of the stored face terms and runs the mode's epilogue
//            (residual, FD product, Newton residual G or a pseudo-time smoothing step).
// The same kernels run on D64 (FP64 residual and finite-difference products)
// and on TL32 (FP32 tangent-linear products for the FP32 preconditioner).
#include <vector>

#include "internal.h"

namespace {

// the 1D tables the operator kernels read
struct TabK {
    int np1;
    double lp[5], lm[5], dlp[5], dlm[5], Dn[5][5];
};
struct DGK {
    int nx, nz, n_el, periodic;
    double two_hx, two_hz, g, mu, eta_x, eta_z;
    float two_hxf, two_hzf, gf, eta_xf, eta_zf;   // float copies for the FP32 tangent
    float tlp[5], tlm[5], tdlp[5], tdlm[5];       // trace tables l_a(+-1), l_a'(+-1) in float
    // volume tables with the 2/h factors folded in, built on the host in both
    // precisions: Dx = (2/hx) Dw, Dz = (2/hz) Dw, lift[0..3] x-lifts, lift[4..7] z-lifts
    double Dx[5][5], Dz[5][5], lift[8][5];
    float Dxf[5][5], Dzf[5][5], Dnf[5][5], liftf[8][5];
    PhysC pc;
    const PowTab *pt;
    const double *ubv, *dubv, *fbx, *fbz, *hbx, *hbxw, *ubh, *dubh, *hbz;
    const float *ubvf, *dubvf, *ubhf, *dubhf;
    TabK tab;
};

template <class T> struct OutT;
template <> struct OutT<D64> { typedef double type; };
template <> struct OutT<TL32> { typedef float type; };
JF_D double outv(D64 a) { return a.x; }
JF_D float outv(TL32 a) { return a.d; }

// Input of the perturbation state at global index i:
// IN 0: U'; IN 1: U' + eps y (FP64); IN 2: TL32 (U', y32)
template <class T, int IN> struct Loader;
template <> struct Loader<D64, 0> {
    const double *U;
    JF_D void prepare() {}
    JF_D D64 operator()(size_t i) const { return D64{U[i]}; }
};
template <> struct Loader<D64, 1> {
    const double *U, *y, *epsp;   // eps: a device scalar written by a reduction, or given
    double eps;
    JF_D void prepare() {
        if (epsp) eps = *epsp;
    }
    JF_D D64 operator()(size_t i) const { return D64{__fma_rn(eps, y[i], U[i])}; }
};
template <> struct Loader<TL32, 2> {
    const float *U;
    const float *y;
    JF_D void prepare() {}
    JF_D TL32 operator()(size_t i) const { return TL32{U[i], y[i]}; }
};

// background values: FP64 tables for D64, FP32 copies for TL32
JF_D D64 bgs(const double *d, const float *, size_t i, D64) { return D64{d[i]}; }
JF_D TLc bgs(const double *, const float *f, size_t i, TL32) { return TLc{f[i]}; }
template <class T>
JF_D T bg(const double *a, size_t i) { return mk(a[i], T{}); }

// ---------------------------------------------------------------------------
// Value and (viscous) derivative traces along a line of NP1 nodes i0 + q st with
// the end-point tables (pa: l_q(+-1), pd: l_q'(+-1)).
template <class T, int IN, int NP1, bool VISC>
JF_D void line_trace(const Loader<T, IN> &ld, size_t i0, size_t st, const double *pa, const float *paf,
                     const double *pd, const float *pdf, T &a, T &d) {
    a = mk(0.0, T{});
    d = mk(0.0, T{});
#pragma unroll
    for (int q = 0; q < NP1; ++q) {
        const T u = ld(i0 + q * st);
        a = jfma(mkc(pa[q], paf[q], T{}), u, a);
        if (VISC) d = jfma(mkc(pd[q], pdf[q], T{}), u, d);
    }
}
template <class T>
JF_D void swap_d(bool c, T &a, T &b) {
    const T t = a;
    a = sel(c, b, a);
    b = sel(c, t, b);
}

// Face terms of block `blk` of one operator evaluation, one thread per face point; K is
// the launch parameter (single operator) or a member's descriptor in global memory
// (grouped launch over ensemble members).  Vertical and horizontal faces run the same
// code: the momentum components are exchanged for the latter (the same arithmetic,
// component for component, in half the instructions and without a divergent block).
template <class T, int IN, int NP1, bool VISC>
__device__ __forceinline__ void faces_body(const DGK &K, const Loader<T, IN> &ld0, typename OutT<T>::type *phix,
                                           typename OutT<T>::type *symx, typename OutT<T>::type *phiz,
                                           typename OutT<T>::type *symz, unsigned blk, const LinPtr &lin) {
    typedef typename OutT<T>::type O;
    Loader<T, IN> ld = ld0;
    ld.prepare();
    constexpr int NP = NP1 * NP1;
    const int nx = K.nx, nz = K.nz;
    const size_t N1 = (size_t)K.n_el * NP;
    const long long nvert = (long long)nz * (nx + 1) * NP1, nfp = nvert + (long long)(nz + 1) * nx * NP1;
    const long long t = (long long)blk * blockDim.x + threadIdx.x;
    if (t >= nfp) return;
    const bool zf = t >= nvert;
    const int u = (int)(zf ? t - nvert : t);
    const int s = u % NP1, c = u / NP1;
    int eL, eR, ib;              // elements of the two sides (L: west / below), background index
    bool wallL, wallR;
    if (!zf) {
        const int fx = c % (nx + 1), ez = c / (nx + 1);
        wallL = fx == 0 && !K.periodic;
        wallR = fx == nx && !K.periodic;
        eL = ez * nx + (fx == 0 ? (K.periodic ? nx - 1 : 0) : fx - 1);
        eR = ez * nx + (fx == nx ? (K.periodic ? 0 : nx - 1) : fx);
        ib = ez * NP1 + s;
    } else {
        const int ex = c % nx, fz = c / nx;
        wallL = fz == 0;
        wallR = fz == nz;
        eL = (wallL ? 0 : fz - 1) * nx + ex;
        eR = (wallR ? nz - 1 : fz) * nx + ex;
        ib = fz;
    }
    const int nb = zf ? nz + 1 : nz * NP1;   // stride of the background tables
    const double *ub = zf ? K.ubh : K.ubv;
    const float *ubf = zf ? K.ubhf : K.ubvf;
    const int st = zf ? NP1 : 1, i0 = zf ? s : s * NP1;
    const auto two_h = mkc(zf ? K.two_hz : K.two_hx, zf ? K.two_hzf : K.two_hxf, T{});
    T UL[4], UR[4], gL[4], gR[4], J[4];   // states, normal derivatives and jumps
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        T aL, aR, dL, dR;
        line_trace<T, IN, NP1, VISC>(ld, v * N1 + (size_t)eL * NP + i0, st, K.tab.lp, K.tlp, K.tab.dlp, K.tdlp, aL, dL);
        line_trace<T, IN, NP1, VISC>(ld, v * N1 + (size_t)eR * NP + i0, st, K.tab.lm, K.tlm, K.tab.dlm, K.tdlm, aR, dR);
        UL[v] = aL + bgs(ub, ubf, (size_t)v * nb + ib, T{});
        UR[v] = aR + bgs(ub, ubf, (size_t)v * nb + ib, T{});
        if (VISC) {
            gL[v] = two_h * dL;
            gR[v] = two_h * dR;
            if (zf) {   // the background varies with z only
                gL[v] = gL[v] + bgs(K.dubh, K.dubhf, (size_t)v * nb + ib, T{});
                gR[v] = gR[v] + bgs(K.dubh, K.dubhf, (size_t)v * nb + ib, T{});
            }
            J[v] = aL - aR;
        }
    }
    if constexpr (IN == 0) {
        if (lin.tr) {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                lin.tr[(2 * v) * nfp + t] = outv(UL[v]);
                lin.tr[(2 * v + 1) * nfp + t] = outv(UR[v]);
                if (VISC) {
                    lin.tr[(8 + 2 * v) * nfp + t] = outv(gL[v]);
                    lin.tr[(9 + 2 * v) * nfp + t] = outv(gR[v]);
                    lin.tr[(16 + v) * nfp + t] = outv(J[v]);
                }
            }
        }
    }
    swap_d(zf, UL[1], UL[2]);
    swap_d(zf, UR[1], UR[2]);
    wall_states<T, 0>(UL, UR, wallL, wallR);
    Side<T> L, R;
    side_of(UL, K.pc, K.pt, L);
    side_of(UR, K.pc, K.pt, R);
    T H[4];
    hllc_s<T, 0>(L, R, H);
    swap_d(zf, H[1], H[2]);
    if constexpr (IN == 0) {
        if (lin.tr) {
#pragma unroll
            for (int v = 0; v < 4; ++v) lin.H[v * nfp + t] = outv(H[v]);
        }
    }
    const double *hb = zf ? K.hbz : (wallL ? K.hbxw : (wallR ? K.hbxw + 4 * (size_t)nb : K.hbx));
#pragma unroll
    for (int v = 0; v < 4; ++v)
        if (IN != 2) H[v] = H[v] - bg<T>(hb, (size_t)v * nb + ib);
    O *phi = zf ? phiz : phix;
    const size_t fs = zf ? (size_t)(nfp - nvert) : (size_t)nvert;
    if (VISC) {
        O *sym = zf ? symz : symx;
        if (wallL || wallR) {
#pragma unroll
            for (int q = 0; q < 6; ++q) sym[(size_t)q * fs + u] = 0;
        } else {
            swap_d(zf, L.U[1], L.U[2]);   // back to (u, w)
            swap_d(zf, R.U[1], R.U[2]);
            const auto eta = mkc(zf ? K.eta_z : K.eta_x, zf ? K.eta_zf : K.eta_xf, T{});
            const auto hmu = mkc(0.5 * K.mu, 0.5f * K.pc.muf, T{});
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int v = q + 1;
                const T pL = L.U[v] * L.ir, pR = R.U[v] * R.ir;
                const T sL = hmu * visc_c(pL, J[0], J[v]), sR = hmu * visc_c(pR, J[0], J[v]);
                const T V = visc_face(hmu, eta, pL, pR, gL, gR, v, sL, sR);
                H[v] = H[v] - V;
                if constexpr (IN == 0) {
                    if (lin.tr) {
                        lin.H[(4 + q) * nfp + t] = outv(V);
                        lin.H[(7 + q) * nfp + t] = outv(sL);
                        lin.H[(10 + q) * nfp + t] = outv(sR);
                    }
                }
                sym[(size_t)q * fs + u] = (O)outv(sL);
                sym[(size_t)(3 + q) * fs + u] = (O)outv(sR);
            }
        }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) phi[v * fs + u] = (O)outv(H[v]);
}

// ---------------------------------------------------------------------------
// Node fluxes and their weak-form derivatives with the gravity source: the operator
// without the lifted face terms, into `part` ([4][nodes]).  blockDim.x / NP elements per
// block (at most 128 threads), one thread per node.
template <class T, int IN, int NP1, bool VISC>
__device__ __forceinline__ void nodes_body(const DGK &K, const Loader<T, IN> &ld0, typename OutT<T>::type *part,
                                           unsigned blk, const LinPtr &lin) {
    typedef typename OutT<T>::type O;
    constexpr int NP = NP1 * NP1;
    constexpr int EPB = 128 / NP;
    __shared__ O sg[2][EPB][4][NP];
    __shared__ T su[VISC ? EPB : 1][4][VISC ? NP : 1];
    // weak-form derivative tables with the 2/h factors folded in: sDx = (2/hx) Dw, sDz = (2/hz) Dw
    __shared__ O sDx[NP1][NP1], sDz[NP1][NP1];
    __shared__ O sDn[NP1][NP1];
    Loader<T, IN> ld = ld0;
    ld.prepare();
    for (int i = threadIdx.x; i < NP; i += blockDim.x) {
        const int r = i / NP1, q = i % NP1;
        sDx[r][q] = pick<O>(K.Dx[r][q], K.Dxf[r][q]);
        sDz[r][q] = pick<O>(K.Dz[r][q], K.Dzf[r][q]);
        sDn[r][q] = pick<O>(K.tab.Dn[r][q], K.Dnf[r][q]);
    }
    const int le = threadIdx.x / NP;
    const int node = threadIdx.x % NP;
    const int a = node % NP1, b = node / NP1;
    const int epb = blockDim.x / NP;
    const int e = (int)blk * epb + le;
    const bool active = (le < epb) && (e < K.n_el);
    const int nx = K.nx, nz = K.nz;
    const int ez = active ? e / nx : 0;
    const size_t N1 = (size_t)K.n_el * NP;
    const size_t nrow = (size_t)nz * NP1;
    const int J = ez * NP1 + b;
    T Up[4], U[4];
    if (active) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            Up[v] = ld((size_t)v * N1 + (size_t)e * NP + node);
            U[v] = Up[v] + bgs(K.ubv, K.ubvf, v * nrow + J, T{});
            if (VISC) su[le][v][node] = Up[v];
        }
    }
    if (VISC) __syncthreads();
    if (active) {
        const T ir = jrcp(U[0]);
        const T p = pressure(U[3], K.pc, K.pt);
        const T u = U[1] * ir, w = U[2] * ir;
        T Fx[4], Fz[4];
        flux_xz(U, u, w, p, Fx, Fz);
        const size_t gl = (size_t)e * NP + node;
        if constexpr (IN == 0) {
            if (lin.tr) {
#pragma unroll
                for (int v = 0; v < 4; ++v) lin.U[v * N1 + gl] = outv(U[v]);
#pragma unroll
                for (int v = 1; v < 4; ++v) lin.F[(v - 1) * N1 + gl] = outv(Fx[v]);
                lin.F[3 * N1 + gl] = outv(Fz[2]);
                lin.F[4 * N1 + gl] = outv(Fz[3]);
            }
        }
        if (IN != 2) {   // minus the background's fluxes; the mass fluxes are linear
            Fx[0] = Up[1];
            Fz[0] = Up[2];
#pragma unroll
            for (int v = 1; v < 4; ++v) {
                Fx[v] = Fx[v] - bg<T>(K.fbx, v * nrow + J);
                Fz[v] = Fz[v] - bg<T>(K.fbz, v * nrow + J);
            }
        }
        if (VISC) {
            T dx[4], dz[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                T sx = mk(0.0, T{}), sz = mk(0.0, T{});
#pragma unroll
                for (int q = 0; q < NP1; ++q) {
                    sx = jfma(mkc((double)sDn[a][q], (float)sDn[a][q], T{}), su[le][v][b * NP1 + q], sx);
                    sz = jfma(mkc((double)sDn[b][q], (float)sDn[b][q], T{}), su[le][v][q * NP1 + a], sz);
                }
                dx[v] = mkc(K.two_hx, K.two_hxf, T{}) * sx;
                dz[v] = mkc(K.two_hz, K.two_hzf, T{}) * sz + bgs(K.dubv, K.dubvf, v * nrow + J, T{});
            }
            const auto mu = mkc(K.mu, K.pc.muf, T{});
            const T phi[4] = {u, u, w, U[3] * ir};
#pragma unroll
            for (int v = 1; v < 4; ++v) {
                const T gx = mu * visc_c(phi[v], dx[0], dx[v]), gz = mu * visc_c(phi[v], dz[0], dz[v]);
                Fx[v] = Fx[v] - gx;
                Fz[v] = Fz[v] - gz;
                if constexpr (IN == 0) {
                    if (lin.tr) {
                        lin.F[(12 + v) * N1 + gl] = outv(gx);
                        lin.F[(15 + v) * N1 + gl] = outv(gz);
                    }
                }
            }
            if constexpr (IN == 0) {
                if (lin.tr) {
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        lin.F[(5 + v) * N1 + gl] = outv(dx[v]);
                        lin.F[(9 + v) * N1 + gl] = outv(dz[v]);
                    }
                }
            }
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            sg[0][le][v][node] = (O)outv(Fx[v]);
            sg[1][le][v][node] = (O)outv(Fz[v]);
        }
    }
    __syncthreads();
    if (!active) return;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        O f = 0;
#pragma unroll
        for (int q = 0; q < NP1; ++q) {
            f = fma(sDx[a][q], sg[0][le][v][b * NP1 + q], f);
            f = fma(sDz[b][q], sg[1][le][v][q * NP1 + a], f);
        }
        if (v == 2) f = fma(-pick<O>(K.g, K.gf), (O)outv(Up[0]), f);
        part[(size_t)v * N1 + (size_t)e * NP + node] = f;
    }
}

// Both in one launch: the first `nface` blocks take the face points, the others the
// nodes; neither needs the other (the lift below adds them).  Bound by the FP64 pipe:
// 95 instructions a face point and 57 a Q3 node take 40.5 of the 48.1 us of Q3 160 x 80
// (Q4 320 x 160: 257 of 264).  As a face launch and a volume launch with the lifts the
// pair took 28.0 + 34.3 us against 48.1 + 12.6 now; the gain is on small grids, where each
// launch pays a latency chain of some thousand clocks (Q2 20 x 10: 14.4 us a residual
// then, 11.5 now, most of it the host's).
template <class T, int IN, int NP1, bool VISC>
struct k_dg_flux_b {
    static constexpr int TPB = 128, MINB = VISC ? 4 : 7;
    static constexpr bool GROUP = !VISC && std::is_same<T, D64>::value;   // a grouped twin is built (lock-step ensembles)
    static __device__ __forceinline__ void run(unsigned jf_bid, unsigned jf_nblk, JfArg<DGK> K, JfArg<unsigned> nface,
                                               JfArg<Loader<T, IN>> ld0, JfArg<typename OutT<T>::type *> part,
                                               JfArg<typename OutT<T>::type *> phix,
                                               JfArg<typename OutT<T>::type *> symx,
                                               JfArg<typename OutT<T>::type *> phiz,
                                               JfArg<typename OutT<T>::type *> symz, JfArg<LinPtr> lin) {
        jf_pdl_enter();
        if (jf_bid < nface) faces_body<T, IN, NP1, VISC>(K, ld0, phix, symx, phiz, symz, jf_bid, lin);
        else nodes_body<T, IN, NP1, VISC>(K, ld0, part, jf_bid - nface, lin);
    }
};
template <class T, int IN, int NP1, bool VISC>
__global__ void __launch_bounds__(128, VISC ? 4 : 7)
    k_dg_flux(DGK K, unsigned nface, Loader<T, IN> ld0, typename OutT<T>::type *part, typename OutT<T>::type *phix,
              typename OutT<T>::type *symx, typename OutT<T>::type *phiz, typename OutT<T>::type *symz, LinPtr lin) {
    k_dg_flux_b<T, IN, NP1, VISC>::run(blockIdx.x, gridDim.x, K, nface, ld0, part, phix, symx, phiz, symz, lin);
}

// Adds the lifts of the face terms to `part` and runs the mode's epilogue, one thread
// per node.
template <class T, int MODE, int NP1, bool VISC>
__device__ __forceinline__ void lift_body(const DGK &K, const DGArgs &A, const typename OutT<T>::type *part,
                                          const typename OutT<T>::type *phix, const typename OutT<T>::type *symx,
                                          const typename OutT<T>::type *phiz, const typename OutT<T>::type *symz,
                                          unsigned blk) {
    typedef typename OutT<T>::type O;
    constexpr int NP = NP1 * NP1;
    constexpr bool FD = MODE == DG_JV || MODE == DG_SMOOTH64;
    __shared__ O sl[8][NP1];    // sl[0..3] x-lifts, sl[4..7] z-lifts
    __shared__ double sce[2];   // eps and adt / eps of the FD modes: one quotient per block
    for (int i = threadIdx.x; i < 8 * NP1; i += blockDim.x)
        sl[i / NP1][i % NP1] = pick<O>(K.lift[i / NP1][i % NP1], K.liftf[i / NP1][i % NP1]);
    if (FD && threadIdx.x == 0) {
        const double e0 = A.eps ? *A.eps : A.eps_val;
        sce[0] = e0;
        sce[1] = e0 != 0.0 ? div64(A.adt, e0) : 0.0;
    }
    const int N1 = K.n_el * NP, n = (int)blk * (int)blockDim.x + (int)threadIdx.x;
    __syncthreads();
    if (n >= N1) return;
    const int e = n / NP, node = n % NP, a = node % NP1, b = node / NP1;
    const int nx = K.nx, nz = K.nz, ez = e / nx, ex = e - ez * nx;
    const int fsx = nz * (nx + 1) * NP1, fsz = (nz + 1) * nx * NP1;
    const int iL = (ez * (nx + 1) + ex) * NP1 + b, iR = iL + NP1;
    const int iB = (ez * nx + ex) * NP1 + a, iT = iB + nx * NP1;
    const double eps = FD ? sce[0] : 0.0, ceps = FD ? sce[1] : 0.0;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const size_t gi = (size_t)v * N1 + n;
        O f = part[gi];
        f = fma(sl[0][a], phix[(size_t)v * fsx + iL], f);
        f = fma(-sl[1][a], phix[(size_t)v * fsx + iR], f);
        f = fma(sl[4][b], phiz[(size_t)v * fsz + iB], f);
        f = fma(-sl[5][b], phiz[(size_t)v * fsz + iT], f);
        if (VISC && v > 0) {
            const int c = v - 1;
            f = fma(sl[2][a], symx[(size_t)(3 + c) * fsx + iL], f);
            f = fma(sl[3][a], symx[(size_t)c * fsx + iR], f);
            f = fma(sl[6][b], symz[(size_t)(3 + c) * fsz + iB], f);
            f = fma(sl[7][b], symz[(size_t)c * fsz + iT], f);
        }
        if (MODE == DG_RES) {
            ((double *)A.out0)[gi] = (double)f;
        } else if (MODE == DG_JV) {
            const double y = A.y[gi];
            ((double *)A.out0)[gi] = (eps == 0.0) ? y : fma(-ceps, (double)f - A.fU[gi], y);
        } else if (MODE == DG_G) {
            A.out1[gi] = (double)f;
            ((double *)A.out0)[gi] = A.U[gi] - A.adt * (double)f - A.Ubs[gi];
        } else if (MODE == DG_SMOOTH64) {
            const double z = A.y[gi];
            const double Jz = (eps == 0.0) ? z : fma(-ceps, (double)f - A.fU[gi], z);
            if (A.z0mode == 0) {
                ((double *)A.out0)[gi] = z + A.dtau[e] * (A.r[gi] - Jz);
            } else {
                const double st = (A.alpha * A.dtau[e]) * (A.r[gi] - Jz);
                ((double *)A.out0)[gi] = A.z0mode == 1 ? ((const double *)A.z0)[gi] + st : st;
            }
        } else if (MODE == DG_TLJV) {
            const float z = A.yf[gi];
            const float jz = z - A.adtf * (float)f;
            ((float *)A.out0)[gi] = A.rf ? A.rf[gi] - jz : jz;   // with r given: the defect r - G'z
        } else {  // DG_TLSMOOTH
            const float z = A.yf[gi];
            const float Jz = z - A.adtf * (float)f;
            if (A.z0mode == 0) {
                ((float *)A.out0)[gi] = z + A.dtauf[e] * (A.rf[gi] - Jz);
            } else {
                const float st = (A.alphaf * A.dtauf[e]) * (A.rf[gi] - Jz);
                ((float *)A.out0)[gi] = A.z0mode == 1 ? ((const float *)A.z0)[gi] + st : st;
            }
        }
    }
}
template <class T, int MODE, int NP1, bool VISC>
struct k_dg_lift_b {
    static constexpr int TPB = 128, MINB = 8;
    static constexpr bool GROUP = !VISC && std::is_same<T, D64>::value && MODE != DG_SMOOTH64;   // a grouped twin is built (lock-step ensembles)
    static __device__ __forceinline__ void run(unsigned jf_bid, unsigned jf_nblk, JfArg<DGK> K, JfArg<DGArgs> A,
                                               JfArg<const typename OutT<T>::type *> part,
                                               JfArg<const typename OutT<T>::type *> phix,
                                               JfArg<const typename OutT<T>::type *> symx,
                                               JfArg<const typename OutT<T>::type *> phiz,
                                               JfArg<const typename OutT<T>::type *> symz) {
        jf_pdl_enter();
        lift_body<T, MODE, NP1, VISC>(K, A, part, phix, symx, phiz, symz, jf_bid);
    }
};
template <class T, int MODE, int NP1, bool VISC>
__global__ void __launch_bounds__(128, 8)
    k_dg_lift(DGK K, DGArgs A, const typename OutT<T>::type *part, const typename OutT<T>::type *phix,
              const typename OutT<T>::type *symx, const typename OutT<T>::type *phiz, const typename OutT<T>::type *symz) {
    k_dg_lift_b<T, MODE, NP1, VISC>::run(blockIdx.x, gridDim.x, K, A, part, phix, symx, phiz, symz);
}

// ---------------------------------------------------------------------------
// FP32 tangent product in ONE launch (the preconditioner's DG smoothing steps
// and defect).  A block owns a strip of E elements of one element row, one
// thread per node.  The strip's states go to shared memory; every face point
// of the strip's elements is evaluated there (x faces between the strip's
// elements once, the strip's two end faces and the z faces with the neighbour
// trace read from global memory), then the volume term, the lift of the
// shared face terms and the mode's epilogue run as in the two-kernel form.  In
// FP32 the duplicated z faces (each is evaluated by the strips above and below)
// cost less than a second launch and the face buffers' round trip.
// FIRST = 1 (defect mode): the direction is the first pseudo-time step from zero,
// z = dtau_E r, formed on the fly; the epilogue also writes that z to out1f.

// Padding of an element's staged values [variable][node] in shared memory, in elements of
// `words` 32-bit words: with the plain stride 4 (k+1)^2 the face points of a strip's
// elements read the same banks (6 ways on Q3, 8 on Q1); these paddings minimise the
// conflicts over the face points of a block (1.4 to 1.8 ways, counted on the host for
// every padding below 33).
constexpr int strip_pad(int np1, int words) {
    return words == 1 ? (np1 == 2 ? 2 : np1 == 4 ? 9 : np1 == 5 ? 3 : 0) : (np1 == 2 ? 2 : 5);
}

// T^mf of the strip's defect (in sd) to the finest FV level: the 1D transfer matrix along
// x, then along z (through the scratch st), the mass fix (mean of the subcell values
// against the modified Newton-Cotes quadrature, both tensor products, so they follow the
// two sweeps: row sums smf, then their sum), written to b and, when x0 is given, x0 = dtau b.
// All threads of the block call it.
template <int NP1, int E>
__device__ __forceinline__ void dgtl_transfer(const TransferOut &TR, float (*sd)[4][NP1 * NP1],
                                              float (*smf)[4][2][NP1], float (*st)[4][NP1 * NP1], int le, int node,
                                              int ez, int ex, bool active) {
    constexpr int NP = NP1 * NP1;
    const int i = node % NP1, j = node / NP1;
    __syncthreads();   // sd complete; sg (scratch st) no longer read
    if (active) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {   // t1(i, b) = sum_a V[i][a] d(a, b), at [b][i]
            float acc = 0.0f;
#pragma unroll
            for (int a = 0; a < NP1; ++a) acc = fmaf(TR.V[i][a], sd[le][q][j * NP1 + a], acc);
            st[le][q][j * NP1 + i] = acc;
        }
    }
    __syncthreads();
    // row sums of t1: lane (q, j) of an element's first 4 NP1 threads, or in turn
    if (active)
        for (int r = node; r < 4 * NP1; r += NP) {
            const int q = r / NP1, row = r % NP1;
            float m = 0.0f, w = 0.0f;
#pragma unroll
            for (int k = 0; k < NP1; ++k) {
                const float x = st[le][q][row * NP1 + k];
                m += x;
                w = fmaf(TR.om[k], x, w);
            }
            smf[le][q][0][row] = m;
            smf[le][q][1][row] = w;
        }
    float Tu[4] = {0.f, 0.f, 0.f, 0.f};
    if (active) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            float acc = 0.0f;
#pragma unroll
            for (int b = 0; b < NP1; ++b) acc = fmaf(TR.V[j][b], st[le][q][b * NP1 + i], acc);
            Tu[q] = acc;
        }
    }
    __syncthreads();
    if (!active) return;
    const size_t I = (size_t)ex * NP1 + i, Jr = (size_t)ez * NP1 + j;
    const size_t cell = Jr * TR.NX + I, ncell = (size_t)TR.NX * TR.NZ;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        float shift = 0.0f;
        if (TR.massfix) {
#pragma unroll
            for (int b = 0; b < NP1; ++b) shift = fmaf(TR.vm[b], smf[le][q][0][b], shift);
#pragma unroll
            for (int b = 0; b < NP1; ++b) shift = fmaf(-TR.vo[b], smf[le][q][1][b], shift);
        }
        const float val = Tu[q] - shift;
        const size_t gi = (size_t)q * ncell + cell;
        TR.b[gi] = val;
        if (TR.x0) TR.x0[gi] = TR.dtau0[cell] * val;   // first pseudo-time step from zero
    }
}

// Sum of a block's per-thread sums of squares to *out: FP32 within a thread (a node's four
// values), FP64 from there on, so that neither the range nor the digits of the norm depend
// on the size of a block.  Seven dependent FP64 adds at the end of the block: an Arnoldi
// step of Q3 80 x 3 takes 0.8 us longer than with a sum in FP32 (1 % of the step).
// n threads (97 to 128) hold one; all of them call it.
__device__ __forceinline__ void block_squares(float sq, int n, double *out) {
    __shared__ float ssq[128];
    ssq[threadIdx.x] = sq;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    const float *q = ssq + threadIdx.x;
    double r = ((double)q[0] + (double)q[32]) + ((double)q[64] + (double)((int)threadIdx.x + 96 < n ? q[96] : 0.0f));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
    if (threadIdx.x == 0) *out = r;
}

template <int NP1, int MODE, int FIRST>
struct k_dgtl_b {
    static constexpr int TPB = 128, MINB = 5;
    static constexpr bool GROUP = false;   // (lock-step members of viscous ensembles replay one at a time)
    static __device__ __forceinline__ void run(unsigned jf_bid, unsigned jf_nblk, JfArg<DGK> K, JfArg<DGArgs> A,
                                               JfArg<float *> out1f, JfArg<TransferOut> TR) {
        jf_pdl_enter();
        constexpr int NP = NP1 * NP1;
        constexpr int E = strip_elems(NP1, true);
        // U' (value, tangent) of the strip's elements [1], of the elements below [0] and
        // above [2] them, and of the strip's west [0] and east [1] neighbours: every
        // trace the faces need comes from shared memory, loaded coalesced up front
        // (an element's values [variable][node], padded: see strip_pad)
        constexpr int S = 4 * NP + strip_pad(NP1, 2);
        __shared__ TL32 sn[3][E][S];
        __shared__ TL32 se[2][S];
        __shared__ float sg[2][E][4][NP];              // volume fluxes (tangent part)
        __shared__ float sPx[E + 1][4][NP1];           // x-face terms Phi (face f west of strip element f)
        __shared__ float sPz[2][E][4][NP1];            // z-face terms: [0] bottom, [1] top of element le
        __shared__ float sSx[E + 1][6][NP1];   // viscous symmetry terms (L side 0..2, R side 3..5)
        __shared__ float sSz[2][E][6][NP1];
        __shared__ float sDx[NP1][NP1], sDz[NP1][NP1], sDn[NP1][NP1], sl[8][NP1];
        __shared__ float sdf[FIRST ? E : 1][4][NP];    // the defect, for the transfer (FIRST)
        __shared__ float smf[FIRST ? E : 1][4][2][NP1];   // row sums of the mass fix
        const int nx = K.nx, nz = K.nz;
        const int nstrip = (nx + E - 1) / E;
        const int ez = (int)jf_bid / nstrip, ex0 = ((int)jf_bid % nstrip) * E;
        const int Ev = min(E, nx - ex0);
        const size_t N1 = (size_t)K.n_el * NP;
        const size_t nrow = (size_t)nz * NP1;
        if (threadIdx.x < NP) {
            const int r = threadIdx.x / NP1, q = threadIdx.x % NP1;
            sDx[r][q] = K.Dxf[r][q];
            sDz[r][q] = K.Dzf[r][q];
            sDn[r][q] = K.Dnf[r][q];
        }
        if (threadIdx.x < NP1) {
    #pragma unroll
            for (int r = 0; r < 8; ++r) sl[r][threadIdx.x] = K.liftf[r][threadIdx.x];
        }
        const int le = threadIdx.x / NP, node = threadIdx.x % NP;
        const int a = node % NP1, b = node / NP1;
        const bool active = le < Ev;
        const int e = ez * nx + ex0 + le;
        // direction at a node: y (or dtau_E r for the first step from zero)
        auto dir = [&](int el, size_t i) -> float { return FIRST ? A.dtauf[el] * A.rf[i] : A.yf[i]; };
        auto load = [&](int el, TL32 *dst) {
    #pragma unroll
            for (int v = 0; v < 4; ++v) {
                const size_t gi = (size_t)v * N1 + (size_t)el * NP + node;
                dst[v * NP + node] = TL32{A.Uf[gi], dir(el, gi)};
            }
        };
        float ef[4] = {0.f, 0.f, 0.f, 0.f}, edt = 0.0f;
        if (active) {
            load(e, sn[1][le]);
            if (ez > 0) load(e - nx, sn[0][le]);
            if (ez < nz - 1) load(e + nx, sn[2][le]);
    #pragma unroll
            for (int v = 0; v < 4; ++v) {
                const size_t gi = (size_t)v * N1 + (size_t)e * NP + node;
                if (MODE == DG_TLSMOOTH || (MODE == DG_TLJV && A.rf)) ef[v] = A.rf[gi];
            }
            if (MODE == DG_TLSMOOTH) edt = A.dtauf[e];
        }
        const bool has_w = ex0 > 0 || K.periodic, has_e = ex0 + Ev < nx || K.periodic;
        if (le == 0 && has_w) load(ez * nx + (ex0 - 1 + nx) % nx, se[0]);
        if (le == 1 && has_e) load(ez * nx + (ex0 + Ev) % nx, se[1]);
        __syncthreads();
        // ---- volume fluxes (independent of the faces below) -----------------------
        TL32 Up[4];
        if (active) {
            const int J = ez * NP1 + b;
            TL32 U[4];
    #pragma unroll
            for (int v = 0; v < 4; ++v) {
                Up[v] = sn[1][le][v * NP + node];
                U[v] = Up[v] + TLc{K.ubvf[v * nrow + J]};
            }
            const TL32 ir = jrcp(U[0]);
            const TL32 p = pressure(U[3], K.pc, nullptr);
            const TL32 u = U[1] * ir, w = U[2] * ir;
            TL32 Fx[4], Fz[4];
            flux_xz(U, u, w, p, Fx, Fz);
            TL32 dx[4], dz[4];
    #pragma unroll
            for (int v = 0; v < 4; ++v) {
                TL32 sx = mk(0.0, TL32{}), sz = mk(0.0, TL32{});
    #pragma unroll
                for (int q = 0; q < NP1; ++q) {
                    sx = jfma(TLc{sDn[a][q]}, sn[1][le][v * NP + b * NP1 + q], sx);
                    sz = jfma(TLc{sDn[b][q]}, sn[1][le][v * NP + q * NP1 + a], sz);
                }
                dx[v] = TLc{K.two_hxf} * sx;
                dz[v] = TLc{K.two_hzf} * sz + TLc{K.dubvf[v * nrow + J]};
            }
            const TLc mu = TLc{K.pc.muf};
            const TL32 phi[4] = {u, u, w, U[3] * ir};
    #pragma unroll
            for (int v = 1; v < 4; ++v) {
                Fx[v] = Fx[v] - mu * visc_c(phi[v], dx[0], dx[v]);
                Fz[v] = Fz[v] - mu * visc_c(phi[v], dz[0], dz[v]);
            }
    #pragma unroll
            for (int v = 0; v < 4; ++v) {
                sg[0][le][v][node] = Fx[v].d;
                sg[1][le][v][node] = Fz[v].d;
            }
        }
        // ---- faces ------------------------------------------------------------
        // value and derivative traces of variable v along NP1 nodes i0 + q st of one
        // element's staged nodes, in the order of line_trace
        auto trace = [&](const TL32 *src, int v, int i0, int st, const float *pa, const float *pd, TL32 &tv,
                         TL32 &td) {
            tv = mk(0.0, TL32{});
            td = mk(0.0, TL32{});
    #pragma unroll
            for (int q = 0; q < NP1; ++q) {
                const TL32 u = src[v * NP + i0 + q * st];
                tv = jfma(TLc{pa[q]}, u, tv);
                td = jfma(TLc{pd[q]}, u, td);
            }
        };
        const int nxf = (Ev + 1) * NP1, nzf = 2 * Ev * NP1;
        for (int t = threadIdx.x; t < nxf + nzf; t += blockDim.x) {
            TL32 trL[4], trR[4], gL[4], gR[4], UL[4], UR[4], H[4], Phi[4], sLv[3], sRv[3];
            if (t < nxf) {
                const int f = t / NP1, sp = t % NP1;      // face f lies west of strip element f
                const bool wallL = f == 0 && !has_w, wallR = f == Ev && !has_e;
                const TL32 *srcL = f > 0 ? sn[1][f - 1] : se[0];
                const TL32 *srcR = f < Ev ? sn[1][f] : se[1];
                const int J = ez * NP1 + sp;
    #pragma unroll
                for (int v = 0; v < 4; ++v) {
                    TL32 aL, aR, dL, dR;
                    if (!wallR) trace(srcR, v, sp * NP1, 1, K.tlm, K.tdlm, aR, dR);
                    if (!wallL) trace(srcL, v, sp * NP1, 1, K.tlp, K.tdlp, aL, dL);
                    if (wallL) { aL = aR; dL = dR; }
                    if (wallR) { aR = aL; dR = dL; }
                    trL[v] = aL;
                    trR[v] = aR;
                    gL[v] = TLc{K.two_hxf} * dL;
                    gR[v] = TLc{K.two_hxf} * dR;
                    UL[v] = aL + TLc{K.ubvf[v * nrow + J]};
                    UR[v] = aR + TLc{K.ubvf[v * nrow + J]};
                }
                wall_states<TL32, 0>(UL, UR, wallL, wallR);
                Side<TL32> SL, SR;
                side_of(UL, K.pc, nullptr, SL);
                side_of(UR, K.pc, nullptr, SR);
                hllc_s<TL32, 0>(SL, SR, H);
    #pragma unroll
                for (int v = 0; v < 4; ++v) Phi[v] = H[v];
                if (!wallL && !wallR) {
                    const TLc hmu = TLc{0.5f * K.pc.muf};
                    const TL32 J0 = trL[0] - trR[0];
    #pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        const int v = q + 1;
                        const TL32 pL = UL[v] * SL.ir, pR = UR[v] * SR.ir;
                        const TL32 Jv = trL[v] - trR[v];
                        sLv[q] = hmu * visc_c(pL, J0, Jv);
                        sRv[q] = hmu * visc_c(pR, J0, Jv);
                        Phi[v] = Phi[v] - visc_face(hmu, TLc{K.eta_xf}, pL, pR, gL, gR, v, sLv[q], sRv[q]);
                    }
                } else {
    #pragma unroll
                    for (int q = 0; q < 3; ++q) sLv[q] = sRv[q] = mk(0.0, TL32{});
                }
    #pragma unroll
                for (int v = 0; v < 4; ++v) sPx[f][v][sp] = Phi[v].d;
    #pragma unroll
                for (int q = 0; q < 3; ++q) {
                    sSx[f][q][sp] = sLv[q].d;
                    sSx[f][3 + q][sp] = sRv[q].d;
                }
            } else {
                const int u = t - nxf;
                const int top = u / (Ev * NP1), l = (u / NP1) % Ev, sp = u % NP1;   // column a = sp
                const int fz = ez + top;                 // global horizontal face 0..nz
                const bool wallB = fz == 0, wallT = fz == nz;
                TL32 gB[4], gT[4];
    #pragma unroll
                for (int v = 0; v < 4; ++v) {
                    TL32 aB, aT, dB, dT;
                    if (top) {   // own element below (trace at eta = +1), element ez+1 above
                        trace(sn[1][l], v, sp, NP1, K.tlp, K.tdlp, aB, dB);
                        if (!wallT) trace(sn[2][l], v, sp, NP1, K.tlm, K.tdlm, aT, dT);
                        else { aT = aB; dT = dB; }
                    } else {     // element ez-1 below, own element above (trace at eta = -1)
                        trace(sn[1][l], v, sp, NP1, K.tlm, K.tdlm, aT, dT);
                        if (!wallB) trace(sn[0][l], v, sp, NP1, K.tlp, K.tdlp, aB, dB);
                        else { aB = aT; dB = dT; }
                    }
                    trL[v] = aB;
                    trR[v] = aT;
                    const TLc dub = TLc{K.dubhf[(size_t)v * (nz + 1) + fz]};
                    gB[v] = TLc{K.two_hzf} * dB + dub;
                    gT[v] = TLc{K.two_hzf} * dT + dub;
                    UL[v] = aB + TLc{K.ubhf[(size_t)v * (nz + 1) + fz]};
                    UR[v] = aT + TLc{K.ubhf[(size_t)v * (nz + 1) + fz]};
                }
                wall_states<TL32, 1>(UL, UR, wallB, wallT);
                Side<TL32> SL, SR;
                side_of(UL, K.pc, nullptr, SL);
                side_of(UR, K.pc, nullptr, SR);
                hllc_s<TL32, 1>(SL, SR, H);
    #pragma unroll
                for (int v = 0; v < 4; ++v) Phi[v] = H[v];
                if (!wallB && !wallT) {
                    const TLc hmu = TLc{0.5f * K.pc.muf};
                    const TL32 J0 = trL[0] - trR[0];
    #pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        const int v = q + 1;
                        const TL32 pL = UL[v] * SL.ir, pR = UR[v] * SR.ir;
                        const TL32 Jv = trL[v] - trR[v];
                        sLv[q] = hmu * visc_c(pL, J0, Jv);
                        sRv[q] = hmu * visc_c(pR, J0, Jv);
                        Phi[v] = Phi[v] - visc_face(hmu, TLc{K.eta_zf}, pL, pR, gB, gT, v, sLv[q], sRv[q]);
                    }
                } else {
    #pragma unroll
                    for (int q = 0; q < 3; ++q) sLv[q] = sRv[q] = mk(0.0, TL32{});
                }
    #pragma unroll
                for (int v = 0; v < 4; ++v) sPz[top][l][v][sp] = Phi[v].d;
    #pragma unroll
                for (int q = 0; q < 3; ++q) {
                    sSz[top][l][q][sp] = sLv[q].d;
                    sSz[top][l][3 + q][sp] = sRv[q].d;
                }
            }
        }
        __syncthreads();
        if (!active && !(FIRST && TR.b) && !(MODE == DG_TLSMOOTH && A.npart)) return;
        float sq = 0.0f;   // sum of squares of the new z
        const float lmxa = sl[0][a], lpxa = sl[1][a], dlmxa = sl[2][a], dlpxa = sl[3][a];
        const float lmzb = sl[4][b], lpzb = sl[5][b], dlmzb = sl[6][b], dlpzb = sl[7][b];
        const float adtf = A.adtf;
    #pragma unroll
        for (int v = 0; v < 4 && active; ++v) {
            float f = 0.0f;
    #pragma unroll
            for (int q = 0; q < NP1; ++q) {
                f = fmaf(sDx[a][q], sg[0][le][v][b * NP1 + q], f);
                f = fmaf(sDz[b][q], sg[1][le][v][q * NP1 + a], f);
            }
            if (v == 2) f = fmaf(-K.gf, Up[0].d, f);
            f = fmaf(lmxa, sPx[le][v][b], f);
            f = fmaf(-lpxa, sPx[le + 1][v][b], f);
            f = fmaf(lmzb, sPz[0][le][v][a], f);
            f = fmaf(-lpzb, sPz[1][le][v][a], f);
            if (v > 0) {
                const int q = v - 1;
                f = fmaf(dlmxa, sSx[le][3 + q][b], f);
                f = fmaf(dlpxa, sSx[le + 1][q][b], f);
                f = fmaf(dlmzb, sSz[0][le][3 + q][a], f);
                f = fmaf(dlpzb, sSz[1][le][q][a], f);
            }
            const size_t gi = (size_t)v * N1 + (size_t)e * NP + node;
            const float z = Up[v].d;
            const float jz = z - adtf * f;
            if (MODE == DG_TLJV) {
                const float dv = A.rf ? ef[v] - jz : jz;   // with r given: the defect r - G'z
                if (FIRST && TR.b) sdf[le][v][node] = dv;
                else ((float *)A.out0)[gi] = dv;
                if (FIRST) out1f[gi] = z;
            } else {  // DG_TLSMOOTH
                if (A.z0mode == 0) {
                    const float zn = z + edt * (ef[v] - jz);
                    ((float *)A.out0)[gi] = zn;
                    sq = fmaf(zn, zn, sq);
                } else {
                    const float st = (A.alphaf * edt) * (ef[v] - jz);
                    ((float *)A.out0)[gi] = A.z0mode == 1 ? ((const float *)A.z0)[gi] + st : st;
                }
            }
        }
        if (MODE == DG_TLSMOOTH && A.npart) {
            static_assert(E * NP > 96 && E * NP <= 128, "block_squares");
            block_squares(sq, E * NP, A.npart + jf_bid);
        }
        if (FIRST && TR.b) dgtl_transfer<NP1, E>(TR, sdf, smf, sg[0], le, node, ez, ex0 + le, active);
    }
};
template <int NP1, int MODE, int FIRST>
__global__ void __launch_bounds__(128, 5) k_dgtl(DGK K, DGArgs A, float *out1f, TransferOut TR) {
    k_dgtl_b<NP1, MODE, FIRST>::run(blockIdx.x, gridDim.x, K, A, out1f, TR);
}

// ---------------------------------------------------------------------------
// FP32 tangent product about a stored linearisation (inviscid).  Every product of one
// Newton iterate differentiates the same fluxes, so the linearisation keeps, per face
// point, the 4 x 4 derivatives of the HLLC flux with respect to both states (FP32, eight
// float4 in structure-of-arrays order) and, per node, u, w, theta and dp/d(rho theta),
// from which the flux derivatives follow.  A product is then traces, two 4 x 4 products a
// face point, a dozen FMAs a node and the operator's sums: a fifth of the instructions of
// the tangent evaluation (k_dgtl, which the viscous operator keeps).
// What bounds it: the chain load - traces - sums of a block and L2 traffic (128 bytes a
// face point).  Each thread therefore fetches its face point's derivatives into registers
// first of all; they arrive while the block stages the direction.  Its arithmetic is
// written in explicit FMAs so that the grouped twin rounds alike.
// Measured on GB300 (events around a product): Q3 160 x 80 elements 13.7 us against 16.7
// for the tangent evaluation (17.0 without the padding of the staged values: half of L1's
// cycles were bank conflicts), Q4 320 x 160 52 against 61, Q1 200 x 100 10.8 against 13.4,
// Q2 20 x 10 7.4 against 8.5; the derivatives take 11.7 us once per Newton iterate.
template <int NP1>
struct k_dgjac_b {
    static constexpr int TPB = 128, MINB = 0;
    static constexpr bool GROUP = false;   // a few launches a Newton iterate: members one at a time
    static __device__ __forceinline__ void run(unsigned jf_bid, unsigned jf_nblk, JfArg<DGK> K, JfArg<const float *> Uf,
                                               JfArg<float4 *> J, JfArg<float4 *> Jn) {
        jf_pdl_enter();
        constexpr int NP = NP1 * NP1;
        const int nx = K.nx, nz = K.nz;
        const size_t N1 = (size_t)K.n_el * NP;
        const long long nvert = (long long)nz * (nx + 1) * NP1, nfp = nvert + (long long)(nz + 1) * nx * NP1;
        const long long t = (long long)jf_bid * blockDim.x + threadIdx.x;
        if (t >= nfp + (long long)N1) return;
        if (t >= nfp) {   // a node
            const size_t n = (size_t)(t - nfp);
            const int J0 = (int)(n / NP) / nx * NP1 + (int)(n % NP) / NP1;
            float U[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) U[v] = Uf[v * N1 + n] + K.ubvf[(size_t)v * nz * NP1 + J0];
            const float ir = frcp(U[0]);
            const TL32 p = pressure(TL32{U[3], 1.0f}, K.pc, nullptr);
            Jn[n] = make_float4(U[1] * ir, U[2] * ir, U[3] * ir, p.d);
            return;
        }
        const bool zf = t >= nvert;
        const int u = (int)(zf ? t - nvert : t);
        const int s = u % NP1, c = u / NP1;
        int eL, eR, ib;
        bool wallL, wallR;
        if (!zf) {
            const int fx = c % (nx + 1), ez = c / (nx + 1);
            wallL = fx == 0 && !K.periodic;
            wallR = fx == nx && !K.periodic;
            eL = ez * nx + (fx == 0 ? (K.periodic ? nx - 1 : 0) : fx - 1);
            eR = ez * nx + (fx == nx ? (K.periodic ? 0 : nx - 1) : fx);
            ib = ez * NP1 + s;
        } else {
            const int ex = c % nx, fz = c / nx;
            wallL = fz == 0;
            wallR = fz == nz;
            eL = (wallL ? 0 : fz - 1) * nx + ex;
            eR = (wallR ? nz - 1 : fz) * nx + ex;
            ib = fz;
        }
        const int nb = zf ? nz + 1 : nz * NP1;
        const float *ubf = zf ? K.ubhf : K.ubvf;
        const int st = zf ? NP1 : 1, i0 = zf ? s : s * NP1;
        float UL[4], UR[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            float a = 0.0f, b = 0.0f;
#pragma unroll
            for (int q = 0; q < NP1; ++q) {
                a = fmaf(K.tlp[q], Uf[v * N1 + (size_t)eL * NP + i0 + q * st], a);
                b = fmaf(K.tlm[q], Uf[v * N1 + (size_t)eR * NP + i0 + q * st], b);
            }
            UL[v] = a + ubf[(size_t)v * nb + ib];
            UR[v] = b + ubf[(size_t)v * nb + ib];
        }
        auto swapf = [&](float &a, float &b) {
            const float x = a;
            a = zf ? b : a;
            b = zf ? x : b;
        };
        swapf(UL[1], UL[2]);
        swapf(UR[1], UR[2]);
        float A[8][4];   // A[4 side + input][output], in the face's frame
#pragma unroll
        for (int d = 0; d < 8; ++d) {
            TL32 L[4], R[4], H[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                L[v] = TL32{UL[v], d == v ? 1.0f : 0.0f};
                R[v] = TL32{UR[v], d == 4 + v ? 1.0f : 0.0f};
            }
            wall_states<TL32, 0>(L, R, wallL, wallR);
            Side<TL32> SL, SR;
            side_of(L, K.pc, nullptr, SL);
            side_of(R, K.pc, nullptr, SR);
            hllc_s<TL32, 0>(SL, SR, H);
#pragma unroll
            for (int v = 0; v < 4; ++v) A[d][v] = H[v].d;
        }
        // to (rho, rho u, rho w, rho theta) order: exchange inputs and outputs 1, 2
#pragma unroll
        for (int q = 0; q < 2; ++q) {
#pragma unroll
            for (int v = 0; v < 4; ++v) swapf(A[4 * q + 1][v], A[4 * q + 2][v]);
#pragma unroll
            for (int i = 0; i < 4; ++i) swapf(A[4 * q + i][1], A[4 * q + i][2]);
#pragma unroll
            for (int v = 0; v < 4; ++v)   // row v: output v against the side's four inputs
                J[(size_t)(4 * q + v) * nfp + t] = make_float4(A[4 * q][v], A[4 * q + 1][v], A[4 * q + 2][v], A[4 * q + 3][v]);
        }
    }
};
template <int NP1>
__global__ void __launch_bounds__(128) k_dgjac(DGK K, const float *Uf, float4 *J, float4 *Jn) {
    k_dgjac_b<NP1>::run(blockIdx.x, gridDim.x, K, Uf, J, Jn);
}

JF_D float dot4(float4 a, const float x[4], float s) {
    return fmaf(a.w, x[3], fmaf(a.z, x[2], fmaf(a.y, x[1], fmaf(a.x, x[0], s))));
}

// A block of 128 threads owns a strip of E elements of one element row, (3 E + 1) NP1 <=
// 128 face points, as k_dgtl does.  MODE, FIRST and the transfer: as k_dgtl.
template <int NP1, int MODE, int FIRST>
struct k_dgjl_b {
    static constexpr int TPB = 128, MINB = 7;
    static __device__ __forceinline__ void run(unsigned jf_bid, unsigned jf_nblk, JfArg<DGK> K, JfArg<DGArgs> A,
                                               JfArg<const float4 *> J, JfArg<const float4 *> Jn, JfArg<float *> out1f,
                                               JfArg<TransferOut> TR) {
        jf_pdl_enter();
        constexpr int NP = NP1 * NP1;
        constexpr int E = strip_elems(NP1, false);
        constexpr int S = 4 * NP + strip_pad(NP1, 1);
        __shared__ float sz[3][E][S];                  // direction: rows below, own, above
        __shared__ float se[2][S];                     // west and east neighbours
        __shared__ float sg[2][E][4][NP];              // node flux derivatives
        __shared__ float sPx[E + 1][4][NP1], sPz[2][E][4][NP1];
        __shared__ float sDx[NP1][NP1], sDz[NP1][NP1], sl[4][NP1], st[2][NP1];
        __shared__ float sdf[FIRST ? E : 1][4][NP];
        __shared__ float smf[FIRST ? E : 1][4][2][NP1];   // row sums of the mass fix
        const int nx = K.nx, nz = K.nz;
        const int nstrip = (nx + E - 1) / E;
        const int ez = (int)jf_bid / nstrip, ex0 = ((int)jf_bid % nstrip) * E;
        const int Ev = min(E, nx - ex0);
        const size_t N1 = (size_t)K.n_el * NP;
        const size_t nvert = (size_t)nz * (nx + 1) * NP1, nfp = nvert + (size_t)(nz + 1) * nx * NP1;
        const int tid = threadIdx.x;
        // the face point of this thread and its derivatives
        const int nxf = (Ev + 1) * NP1, nzf = 2 * Ev * NP1;
        const bool isx = tid < nxf, face = tid < nxf + nzf;
        const int fu = isx ? tid : tid - nxf;
        const int sp = fu % NP1;
        const int f = fu / NP1;                                  // x: face west of strip element f
        const int top = isx ? 0 : f / Ev, l = isx ? 0 : f % Ev;  // z: bottom / top face of element l
        float4 JL[4], JR[4];
        if (face) {
            const size_t t = isx ? ((size_t)ez * (nx + 1) + ex0 + f) * NP1 + sp
                                 : nvert + ((size_t)(ez + top) * nx + ex0 + l) * NP1 + sp;
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                JL[v] = J[(size_t)v * nfp + t];
                JR[v] = J[(size_t)(4 + v) * nfp + t];
            }
        }
        const int le = tid / NP, node = tid % NP;
        const int a = node % NP1, b = node / NP1;
        const bool active = le < Ev;
        const int e = ez * nx + ex0 + le;
        auto dir = [&](int el, size_t i) -> float { return FIRST ? A.dtauf[el] * A.rf[i] : A.yf[i]; };
        auto load = [&](int el, float *dst) {
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const size_t gi = (size_t)v * N1 + (size_t)el * NP + node;
                dst[v * NP + node] = dir(el, gi);
            }
        };
        float ef[4] = {0.f, 0.f, 0.f, 0.f}, edt = 0.0f;
        float4 jn = make_float4(0.f, 0.f, 0.f, 0.f);
        if (active) {
            load(e, sz[1][le]);
            if (ez > 0) load(e - nx, sz[0][le]);
            if (ez < nz - 1) load(e + nx, sz[2][le]);
            jn = Jn[(size_t)e * NP + node];
#pragma unroll
            for (int v = 0; v < 4; ++v)
                if (MODE == DG_TLSMOOTH || A.rf) ef[v] = A.rf[(size_t)v * N1 + (size_t)e * NP + node];
            if (MODE == DG_TLSMOOTH) edt = A.dtauf[e];
        }
        const bool has_w = ex0 > 0 || K.periodic, has_e = ex0 + Ev < nx || K.periodic;
        if (le == 0 && has_w) load(ez * nx + (ex0 - 1 + nx) % nx, se[0]);
        if (le == 1 && has_e) load(ez * nx + (ex0 + Ev) % nx, se[1]);
        if (tid < NP) {
            const int r = tid / NP1, q = tid % NP1;
            sDx[r][q] = K.Dxf[r][q];
            sDz[r][q] = K.Dzf[r][q];
        }
        if (tid < NP1) {
            sl[0][tid] = K.liftf[0][tid];
            sl[1][tid] = K.liftf[1][tid];
            sl[2][tid] = K.liftf[4][tid];
            sl[3][tid] = K.liftf[5][tid];
            st[0][tid] = K.tlm[tid];
            st[1][tid] = K.tlp[tid];
        }
        __syncthreads();
        float z[4] = {0.f, 0.f, 0.f, 0.f};
        if (active) {
#pragma unroll
            for (int v = 0; v < 4; ++v) z[v] = sz[1][le][v * NP + node];
            const float u = jn.x, w = jn.y, th = jn.z, pd = jn.w * z[3];
            const float du = fmaf(-u, z[0], z[1]), dw = fmaf(-w, z[0], z[2]);   // rho du, rho dw
            const float uw = fmaf(w, du, u * z[2]);                            // d(rho u w) = w rho du + u d(rho w)
            sg[0][le][0][node] = z[1];
            sg[0][le][1][node] = fmaf(u, z[1] + du, pd);
            sg[0][le][2][node] = uw;
            sg[0][le][3][node] = fmaf(th, du, u * z[3]);
            sg[1][le][0][node] = z[2];
            sg[1][le][1][node] = uw;
            sg[1][le][2][node] = fmaf(w, z[2] + dw, pd);
            sg[1][le][3][node] = fmaf(th, dw, w * z[3]);
        }
        if (face) {
            // the lines of the two sides; at a wall the outer one only has to be finite (its
            // derivatives are zero)
            const float *sL, *sR;
            if (isx) {
                sL = f > 0 ? sz[1][f - 1] : (has_w ? se[0] : sz[1][0]);
                sR = f < Ev ? sz[1][f] : (has_e ? se[1] : sz[1][Ev - 1]);
            } else {
                sL = top ? sz[1][l] : (ez > 0 ? sz[0][l] : sz[1][l]);
                sR = top ? (ez < nz - 1 ? sz[2][l] : sz[1][l]) : sz[1][l];
            }
            const int i0 = isx ? sp * NP1 : sp, s1 = isx ? 1 : NP1;
            float dL[4], dR[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                dL[v] = dR[v] = 0.0f;
#pragma unroll
                for (int q = 0; q < NP1; ++q) {
                    dL[v] = fmaf(st[1][q], sL[v * NP + i0 + q * s1], dL[v]);
                    dR[v] = fmaf(st[0][q], sR[v * NP + i0 + q * s1], dR[v]);
                }
            }
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                const float H = dot4(JR[v], dR, dot4(JL[v], dL, 0.0f));
                if (isx) sPx[f][v][sp] = H;
                else sPz[top][l][v][sp] = H;
            }
        }
        __syncthreads();
        if (!active && !(FIRST && TR.b) && !(MODE == DG_TLSMOOTH && A.npart)) return;
        float sq = 0.0f;   // sum of squares of the new z
#pragma unroll
        for (int v = 0; v < 4 && active; ++v) {
            float r = 0.0f;
#pragma unroll
            for (int q = 0; q < NP1; ++q) {
                r = fmaf(sDx[a][q], sg[0][le][v][b * NP1 + q], r);
                r = fmaf(sDz[b][q], sg[1][le][v][q * NP1 + a], r);
            }
            if (v == 2) r = fmaf(-K.gf, z[0], r);
            r = fmaf(sl[0][a], sPx[le][v][b], r);
            r = fmaf(-sl[1][a], sPx[le + 1][v][b], r);
            r = fmaf(sl[2][b], sPz[0][le][v][a], r);
            r = fmaf(-sl[3][b], sPz[1][le][v][a], r);
            const size_t gi = (size_t)v * N1 + (size_t)e * NP + node;
            const float jz = fmaf(-A.adtf, r, z[v]);
            if (MODE == DG_TLJV) {
                const float dv = A.rf ? ef[v] - jz : jz;   // with r given: the defect r - G'z
                if (FIRST && TR.b) sdf[le][v][node] = dv;
                else ((float *)A.out0)[gi] = dv;
                if (FIRST) out1f[gi] = z[v];
            } else if (A.z0mode == 0) {
                const float zn = fmaf(edt, ef[v] - jz, z[v]);
                ((float *)A.out0)[gi] = zn;
                sq = fmaf(zn, zn, sq);
            } else {
                const float stp = __fmul_rn(A.alphaf * edt, ef[v] - jz);
                ((float *)A.out0)[gi] = A.z0mode == 1 ? ((const float *)A.z0)[gi] + stp : stp;
            }
        }
        if (MODE == DG_TLSMOOTH && A.npart) {
            block_squares(sq, 128, A.npart + jf_bid);
        }
        if (FIRST && TR.b) dgtl_transfer<NP1, E>(TR, sdf, smf, sg[0], le, node, ez, ex0 + le, active);
    }
};
template <int NP1, int MODE, int FIRST>
__global__ void __launch_bounds__(128, 7)
    k_dgjl(DGK K, DGArgs A, const float4 *J, const float4 *Jn, float *out1f, TransferOut TR) {
    k_dgjl_b<NP1, MODE, FIRST>::run(blockIdx.x, gridDim.x, K, A, J, Jn, out1f, TR);
}

// background fluxes at node rows and horizontal faces, with the residual's own
// D64 functions so that U' = 0 cancels bit for bit
__global__ void k_bg_dg(DGK K, double *fbx, double *fbz, double *hbx, double *hbxw, double *hbz) {
    jf_pdl_enter();
    const int nrow = K.nz * K.tab.np1;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < nrow) {
        D64 U[4], G[4], Fx[4], Fz[4], H[4];
        for (int v = 0; v < 4; ++v) U[v] = D64{K.ubv[v * nrow + i]};
        const D64 ir = jrcp(U[0]);
        flux_xz(U, U[1] * ir, U[2] * ir, pressure(U[3], K.pc, K.pt), Fx, Fz);
        for (int v = 0; v < 4; ++v) {
            fbx[v * nrow + i] = Fx[v].x;
            fbz[v * nrow + i] = Fz[v].x;
        }
        hllc<D64, 0>(U, U, K.pc, K.pt, H);
        for (int v = 0; v < 4; ++v) hbx[v * nrow + i] = H[v].x;
        mirror<D64, 0>(U, G);
        hllc<D64, 0>(G, U, K.pc, K.pt, H);
        for (int v = 0; v < 4; ++v) hbxw[v * nrow + i] = H[v].x;
        hllc<D64, 0>(U, G, K.pc, K.pt, H);
        for (int v = 0; v < 4; ++v) hbxw[(4 + v) * nrow + i] = H[v].x;
    } else if (i < nrow + K.nz + 1) {
        const int j = i - nrow;
        const int nf = K.nz + 1;
        D64 U[4], G[4], H[4];
        for (int v = 0; v < 4; ++v) U[v] = D64{K.ubh[v * nf + j]};
        mirror<D64, 1>(U, G);
        if (j == 0)
            hllc<D64, 1>(G, U, K.pc, K.pt, H);
        else if (j == K.nz)
            hllc<D64, 1>(U, G, K.pc, K.pt, H);
        else
            hllc<D64, 1>(U, U, K.pc, K.pt, H);
        for (int v = 0; v < 4; ++v) hbz[v * nf + j] = H[v].x;
    }
}

DGK make_K(jfnk_ctx *c) {
    DGK K;
    K.nx = c->grid.nx;
    K.nz = c->grid.nz;
    K.n_el = c->n_el;
    K.periodic = c->grid.periodic_x;
    K.two_hx = 2.0 / c->hx;
    K.two_hz = 2.0 / c->hz;
    K.g = c->phys.g;
    K.mu = c->phys.mu;
    K.gf = (float)K.g;
    const double n1 = c->np1;
    // interior-penalty factor C_IP (k+1)^2 / h; the viscosity enters through A(U)
    K.eta_x = c->opts.c_ip * n1 * n1 / c->hx;
    K.eta_z = c->opts.c_ip * n1 * n1 / c->hz;
    K.pc = c->pc;
    K.pt = c->powtab;
    K.ubv = c->ubv;
    K.dubv = c->dubv;
    K.fbx = c->fbx;
    K.fbz = c->fbz;
    K.hbx = c->hbx;
    K.hbxw = c->hbxw;
    K.ubh = c->ubh;
    K.dubh = c->dubh;
    K.hbz = c->hbz;
    K.ubvf = c->ubvf;
    K.dubvf = c->dubvf;
    K.ubhf = c->ubhf;
    K.dubhf = c->dubhf;
    K.tab.np1 = c->np1;
    for (int q = 0; q < 5; ++q) {
        K.tab.lp[q] = c->tab.lp[q];
        K.tab.lm[q] = c->tab.lm[q];
        K.tab.dlp[q] = c->tab.dlp[q];
        K.tab.dlm[q] = c->tab.dlm[q];
        for (int r = 0; r < 5; ++r) K.tab.Dn[r][q] = c->tab.Dn[r][q];
    }
    K.two_hxf = (float)K.two_hx;
    K.two_hzf = (float)K.two_hz;
    K.eta_xf = (float)K.eta_x;
    K.eta_zf = (float)K.eta_z;
    for (int r = 0; r < 5; ++r)
        for (int q = 0; q < 5; ++q) {
            K.Dx[r][q] = K.two_hx * c->tab.Dw[r][q];
            K.Dz[r][q] = K.two_hz * c->tab.Dw[r][q];
            K.Dxf[r][q] = (float)K.Dx[r][q];
            K.Dzf[r][q] = (float)K.Dz[r][q];
            K.Dnf[r][q] = (float)K.tab.Dn[r][q];
        }
    for (int q = 0; q < 5; ++q) {
        K.lift[0][q] = K.two_hx * c->tab.lmw[q];
        K.lift[1][q] = K.two_hx * c->tab.lpw[q];
        K.lift[2][q] = K.two_hx * K.two_hx * c->tab.dlmw[q];
        K.lift[3][q] = K.two_hx * K.two_hx * c->tab.dlpw[q];
        K.lift[4][q] = K.two_hz * c->tab.lmw[q];
        K.lift[5][q] = K.two_hz * c->tab.lpw[q];
        K.lift[6][q] = K.two_hz * K.two_hz * c->tab.dlmw[q];
        K.lift[7][q] = K.two_hz * K.two_hz * c->tab.dlpw[q];
        for (int r = 0; r < 8; ++r) K.liftf[r][q] = (float)K.lift[r][q];
    }
    for (int a = 0; a < 5; ++a) {
        K.tlp[a] = (float)K.tab.lp[a];
        K.tlm[a] = (float)K.tab.lm[a];
        K.tdlp[a] = (float)K.tab.dlp[a];
        K.tdlm[a] = (float)K.tab.dlm[a];
    }
    return K;
}

// adds the two launches' times of a timed evaluation (jfnk_time_operator)
int timing_close(jfnk_ctx *c, cudaStream_t s) {
    if (!c->timing) return JFNK_OK;
    JF_CK(cudaEventRecord(c->tev[2], s));
    JF_CK(cudaEventSynchronize(c->tev[2]));
    float m0 = 0.f, m1 = 0.f;
    JF_CK(cudaEventElapsedTime(&m0, c->tev[0], c->tev[1]));
    JF_CK(cudaEventElapsedTime(&m1, c->tev[1], c->tev[2]));
    c->t_faces_ms += m0;
    c->t_volume_ms += m1;
    return JFNK_OK;
}

#include "dg_fd.cuh"

template <class T, int IN, int MODE, int NP1, bool VISC>
int launch(jfnk_ctx *c, const DGK &K, const Loader<T, IN> &ld, const DGArgs &a, cudaStream_t s) {
    typedef typename OutT<T>::type O;
    O *phix, *symx, *phiz, *symz;
    if (IN == 2) {
        phix = (O *)c->phixf;
        symx = (O *)c->symxf;
        phiz = (O *)c->phizf;
        symz = (O *)c->symzf;
    } else {
        phix = (O *)c->phix;
        symx = (O *)c->symx;
        phiz = (O *)c->phiz;
        symz = (O *)c->symz;
    }
    const long long nf = (long long)K.nz * (K.nx + 1) * NP1 + (long long)(K.nz + 1) * K.nx * NP1;
    if (c->timing) JF_CK(cudaEventRecord(c->tev[0], s));
    const LinPtr lin = IN == 0 && a.lin_out ? c->lin : LinPtr{};
    const int epb = spread_elements<NP1>(c->opts.tile_volume, K.n_el, c->n_sm), tb = epb * NP1 * NP1;
    const unsigned nface = (unsigned)((nf + tb - 1) / tb), nnode = (unsigned)((K.n_el + epb - 1) / epb);
    // the operator without its lifts, closed in place
    O *part = MODE == DG_G ? (O *)a.out1 : (O *)a.out0;
    jf_launch<k_dg_flux_b<T, IN, NP1, VISC>>(k_dg_flux<T, IN, NP1, VISC>, nface + nnode, tb, 0, s, K, nface, ld, part, phix, symx, phiz, symz,
              lin);
    jf_launched();
    if (c->timing) JF_CK(cudaEventRecord(c->tev[1], s));
    const int tl = spread_threads(128, c->npt, c->n_sm);
    jf_launch<k_dg_lift_b<T, MODE, NP1, VISC>>(k_dg_lift<T, MODE, NP1, VISC>, (unsigned)((c->npt + tl - 1) / tl), tl, 0, s, K, a, (const O *)part,
              (const O *)phix, (const O *)symx, (const O *)phiz, (const O *)symz);
    jf_launched();
    JF_CK(cudaGetLastError());
    return timing_close(c, s);
}

// FP32 tangent modes: one fused launch (k_dgtl); a.first1 selects the defect at
// the first pseudo-time step from zero, whose z = dtau r is also written to a.out1f
template <int NP1, bool VISC, int MODE>
int launch_tl(jfnk_ctx *c, const DGK &K, const DGArgs &a, cudaStream_t s) {
    constexpr int E = strip_elems(NP1, VISC);
    const unsigned nb = (unsigned)(K.nz * ((K.nx + E - 1) / E));
    if (c->timing) JF_CK(cudaEventRecord(c->tev[0], s));
    if constexpr (VISC) {
        const int threads = E * NP1 * NP1;
        if (MODE == DG_TLJV && a.out1f)
            jf_launch<k_dgtl_b<NP1, MODE, 1>>(k_dgtl<NP1, MODE, 1>, nb, threads, 0, s, K, a, a.out1f,
                      a.tro ? *a.tro : TransferOut{});
        else
            jf_launch<k_dgtl_b<NP1, MODE, 0>>(k_dgtl<NP1, MODE, 0>, nb, threads, 0, s, K, a, (float *)nullptr, TransferOut{});
    } else {
        const float4 *J = (const float4 *)c->jac, *Jn = (const float4 *)c->jacn;
        if (MODE == DG_TLJV && a.out1f)
            jf_launch<k_dgjl_b<NP1, MODE, 1>>(k_dgjl<NP1, MODE, 1>, nb, 128, 0, s, K, a, J, Jn, a.out1f,
                      a.tro ? *a.tro : TransferOut{});
        else
            jf_launch<k_dgjl_b<NP1, MODE, 0>>(k_dgjl<NP1, MODE, 0>, nb, 128, 0, s, K, a, J, Jn, (float *)nullptr, TransferOut{});
    }
    jf_launched();
    JF_CK(cudaGetLastError());
    if (c->timing) {
        JF_CK(cudaEventRecord(c->tev[1], s));
        JF_CK(cudaEventSynchronize(c->tev[1]));
        float m0 = 0.f;
        JF_CK(cudaEventElapsedTime(&m0, c->tev[0], c->tev[1]));
        c->t_faces_ms += m0;   // the whole fused product; the volume share reads 0
    }
    return JFNK_OK;
}

template <int NP1, bool VISC>
int dispatch_mode(jfnk_ctx *c, int mode, const DGArgs &a, cudaStream_t s) {
    DGK K = make_K(c);
    switch (mode) {
        case DG_RES: return launch<D64, 0, DG_RES, NP1, VISC>(c, K, Loader<D64, 0>{a.U}, a, s);
        case DG_G: return launch<D64, 0, DG_G, NP1, VISC>(c, K, Loader<D64, 0>{a.U}, a, s);
        case DG_JV:
            if (a.lin && a.yf) return launch_fd<float, DG_JV, NP1, VISC>(c, a, a.yf, s);
            if (a.lin) return launch_fd<double, DG_JV, NP1, VISC>(c, a, a.y, s);
            return launch<D64, 1, DG_JV, NP1, VISC>(c, K, Loader<D64, 1>{a.U, a.y, a.eps, a.eps_val}, a, s);
        case DG_SMOOTH64:
            if (a.lin) return launch_fd<double, DG_SMOOTH64, NP1, VISC>(c, a, a.y, s);
            return launch<D64, 1, DG_SMOOTH64, NP1, VISC>(c, K, Loader<D64, 1>{a.U, a.y, a.eps, a.eps_val}, a, s);
        case DG_TLLIN:   // the stored linearisation of the fused FP32 products at Uf
            if constexpr (!VISC) {
                const long long nt = (long long)K.nz * (K.nx + 1) * NP1 + (long long)(K.nz + 1) * K.nx * NP1 + (long long)c->npt;
                jf_launch<k_dgjac_b<NP1>>(k_dgjac<NP1>, (unsigned)((nt + 127) / 128), 128, 0, s, K, a.Uf, (float4 *)c->jac, (float4 *)c->jacn);
                jf_launched();
                JF_CK(cudaGetLastError());
            }
            return JFNK_OK;
        case DG_TLJV:
            if (c->opts.dg_fused == 2 && !a.out1f)
                return launch<TL32, 2, DG_TLJV, NP1, VISC>(c, K, Loader<TL32, 2>{a.Uf, a.yf}, a, s);
            return launch_tl<NP1, VISC, DG_TLJV>(c, K, a, s);
        case DG_TLSMOOTH:
            if (c->opts.dg_fused == 2)
                return launch<TL32, 2, DG_TLSMOOTH, NP1, VISC>(c, K, Loader<TL32, 2>{a.Uf, a.yf}, a, s);
            return launch_tl<NP1, VISC, DG_TLSMOOTH>(c, K, a, s);
    }
    return JFNK_EINVAL;
}

// ---- one launch per operator across ensemble members ---------------------
// A member's share of a grouped residual launch: its operator constants, state,
// output and face buffers, its face block count and the first flux / lift block of the
// launch that belongs to it.
struct DGMember {
    DGK K;
    Loader<D64, 0> ld;
    DGArgs A;
    double *phix, *symx, *phiz, *symz;
    unsigned nface, fb0, lb0;
};
// flux and lift blocks of one member (128-thread blocks, 128 / NP elements each)
inline void group_blocks(const DGK &K, unsigned &nface, unsigned &nflux, unsigned &nlift) {
    const int n1 = K.tab.np1, np = n1 * n1, epb = 128 / np, tb = epb * np;
    const long long nf = (long long)K.nz * (K.nx + 1) * n1 + (long long)(K.nz + 1) * K.nx * n1;
    nface = (unsigned)((nf + tb - 1) / tb);
    nflux = nface + (unsigned)((K.n_el + epb - 1) / epb);
    nlift = (unsigned)(((long long)K.n_el * np + 127) / 128);
}

template <int NP1, bool VISC>
__global__ void __launch_bounds__(128, VISC ? 4 : 7) k_flux_grp(const DGMember *mem, int nm) {
    jf_pdl_enter();
    int m = 0;
    while (m + 1 < nm && blockIdx.x >= mem[m + 1].fb0) ++m;   // members in block order
    const DGMember &M = mem[m];
    const unsigned bid = blockIdx.x - M.fb0;
    if (bid < M.nface) faces_body<D64, 0, NP1, VISC>(M.K, M.ld, M.phix, M.symx, M.phiz, M.symz, bid, LinPtr{});
    else nodes_body<D64, 0, NP1, VISC>(M.K, M.ld, (double *)M.A.out0, bid - M.nface, LinPtr{});
}

template <int NP1, bool VISC>
__global__ void __launch_bounds__(128, 8) k_lift_grp(const DGMember *mem, int nm) {
    jf_pdl_enter();
    int m = 0;
    while (m + 1 < nm && blockIdx.x >= mem[m + 1].lb0) ++m;
    const DGMember &M = mem[m];
    lift_body<D64, DG_RES, NP1, VISC>(M.K, M.A, (const double *)M.A.out0, M.phix, M.symx, M.phiz, M.symz, blockIdx.x - M.lb0);
}

template <int NP1, bool VISC>
void launch_grp(const DGMember *dmem, const std::vector<DGMember> &h, int first, int cnt, cudaStream_t s) {
    const DGMember &last = h[first + cnt - 1];
    unsigned nface, nflux, nlift;
    group_blocks(last.K, nface, nflux, nlift);
    jf_launch_now(k_flux_grp<NP1, VISC>, last.fb0 + nflux, 128 / (NP1 * NP1) * (NP1 * NP1), 0, s, dmem + first, cnt);
    jf_launch_now(k_lift_grp<NP1, VISC>, last.lb0 + nlift, 128, 0, s, dmem + first, cnt);
    jf_launched(2);
}

}  // namespace

// The operator kernels of one order k = NP1 - 1.  The library compiles this
// file once per order (JF_DG_NP1 = 2..5, in parallel); the order-independent
// functions below come with the first.  Compiled without JF_DG_NP1, one unit
// holds every order.
template <int NP1>
int dg_dispatch(jfnk_ctx *c, int mode, const DGArgs &a, cudaStream_t s);
#if !defined(JF_DG_NP1)
#define JF_DG_ORDERS(X) X(2) X(3) X(4) X(5)
#else
#define JF_DG_ORDERS(X) X(JF_DG_NP1)
#endif
#define JF_DG_DEFINE(n)                                                                              \
    template <>                                                                                     \
    int dg_dispatch<n>(jfnk_ctx * c, int mode, const DGArgs &a, cudaStream_t s) {                   \
        return c->phys.mu != 0.0 ? dispatch_mode<n, true>(c, mode, a, s) : dispatch_mode<n, false>(c, mode, a, s); \
    }
JF_DG_ORDERS(JF_DG_DEFINE)

#if !defined(JF_DG_NP1) || JF_DG_NP1 == 2
#if defined(JF_DG_NP1)
template <> int dg_dispatch<3>(jfnk_ctx *c, int mode, const DGArgs &a, cudaStream_t s);
template <> int dg_dispatch<4>(jfnk_ctx *c, int mode, const DGArgs &a, cudaStream_t s);
template <> int dg_dispatch<5>(jfnk_ctx *c, int mode, const DGArgs &a, cudaStream_t s);
#endif

int dg_setup_background(jfnk_ctx *c, cudaStream_t s) {
    DGK K = make_K(c);
    const int n = c->grid.nz * c->np1 + c->grid.nz + 1;
    k_bg_dg<<<(n + 127) / 128, 128, 0, s>>>(K, c->fbx, c->fbz, c->hbx, c->hbxw, c->hbz); jf_launched();
    JF_CK(cudaGetLastError());
    return JFNK_OK;
}

int dg_apply(jfnk_ctx *c, int mode, const DGArgs &a_in, cudaStream_t s) {
    DGArgs a = a_in;
    a.adtf = (float)a.adt;
    a.alphaf = (float)a.alpha;
    if (mode != DG_TLLIN) c->dg_calls++;
    // the linearisation belongs to the cached f(U): any other writer of the cache drops it
    if (a.out0 == c->fU || a.out1 == c->fU) c->lin_valid = a.lin_out;
    if (a.lin && !c->lin_valid) return JFNK_EINVAL;
    switch (c->np1) {
        case 2: return dg_dispatch<2>(c, mode, a, s);
        case 3: return dg_dispatch<3>(c, mode, a, s);
        case 4: return dg_dispatch<4>(c, mode, a, s);
        case 5: return dg_dispatch<5>(c, mode, a, s);
    }
    return JFNK_EINVAL;
}

size_t dg_member_bytes() { return sizeof(DGMember); }

// f_m = M^-1 L_h(U_m) for every member, grouped by (order, viscous): one face
// and one volume launch per group.  dmem: device room for n descriptors.
int dg_residual_grouped(jfnk_ctx *const *ctx, int n, const double *const *U, double *const *f, void *dmem,
                        cudaStream_t s) {
    if (!ctx || !U || !f || !dmem || n < 1) return JFNK_EINVAL;
    std::vector<int> order;
    for (int np1 = 2; np1 <= 5; ++np1)
        for (int visc = 0; visc < 2; ++visc)
            for (int i = 0; i < n; ++i) {
                if (!ctx[i] || !U[i] || !f[i] || U[i] == f[i]) return JFNK_EINVAL;
                if (ctx[i]->np1 == np1 && (ctx[i]->phys.mu != 0.0) == (visc != 0)) order.push_back(i);
            }
    if ((int)order.size() != n) return JFNK_EINVAL;
    std::vector<DGMember> h(n);
    std::vector<int> gstart;
    unsigned fb = 0, lb = 0;
    for (int q = 0; q < n; ++q) {
        jfnk_ctx *c = ctx[order[q]];
        if (q == 0 || c->np1 != ctx[order[q - 1]]->np1 ||
            (c->phys.mu != 0.0) != (ctx[order[q - 1]]->phys.mu != 0.0)) {
            gstart.push_back(q);
            fb = lb = 0;
        }
        DGMember &M = h[q];
        M.K = make_K(c);
        M.ld = Loader<D64, 0>{U[order[q]]};
        M.A = DGArgs{};
        M.A.U = U[order[q]];
        M.A.out0 = f[order[q]];
        M.phix = (double *)c->phix;
        M.symx = (double *)c->symx;
        M.phiz = (double *)c->phiz;
        M.symz = (double *)c->symz;
        M.fb0 = fb;
        M.lb0 = lb;
        unsigned nflux, nlift;
        group_blocks(M.K, M.nface, nflux, nlift);
        fb += nflux;
        lb += nlift;
        c->dg_calls++;
    }
    JF_CK(cudaMemcpyAsync(dmem, h.data(), sizeof(DGMember) * (size_t)n, cudaMemcpyHostToDevice, s));
    const DGMember *dm = (const DGMember *)dmem;
    gstart.push_back(n);
    for (size_t gi = 0; gi + 1 < gstart.size(); ++gi) {
        const int a = gstart[gi], cnt = gstart[gi + 1] - a;
        const bool visc = h[a].K.mu != 0.0;
        switch (h[a].K.tab.np1) {
            case 2: visc ? launch_grp<2, true>(dm, h, a, cnt, s) : launch_grp<2, false>(dm, h, a, cnt, s); break;
            case 3: visc ? launch_grp<3, true>(dm, h, a, cnt, s) : launch_grp<3, false>(dm, h, a, cnt, s); break;
            case 4: visc ? launch_grp<4, true>(dm, h, a, cnt, s) : launch_grp<4, false>(dm, h, a, cnt, s); break;
            case 5: visc ? launch_grp<5, true>(dm, h, a, cnt, s) : launch_grp<5, false>(dm, h, a, cnt, s); break;
            default: return JFNK_EINVAL;
        }
    }
    JF_CK(cudaGetLastError());
    return JFNK_OK;
}
#endif  // order-independent part
