// Finite-difference product of Sec. 3.1 about a stored linearisation (included by dg.cu).
//
//   G'(U) y ~ y - alpha dt (f(U + eps y) - f(U)) / eps
//
// f is linear in its numerical and node fluxes, f = L(F), so f(U + eps y) - f(U) =
// L(F(U + eps y) - F(U)).  The residual at U keeps what does not depend on y: the states
// and (viscous) gradients at the face points and nodes, and the fluxes there.  A product
// then evaluates the fluxes at U + eps y in FP64, subtracts the stored ones (one rounding;
// none where the two are within a factor of two of each other, as they are except near
// zero), and applies L, the traces and the gradients of y in two-float arithmetic (an
// unevaluated sum of two floats, about 46 bits; products by FMA, sums by Knuth's TwoSum)
// on the FP32 pipe.
// What bounds it: FP64 instructions, as in the general form (19 clocks of an SM each per
// warp, where an FP32 one takes 0.25).  Per Q3 face point 63 of them against 103, per
// node 25 against 85.  Accuracy: the differences are formed before anything is summed, so
// the sums' rounding is relative to the difference and not to the fluxes, which are
// about 1/eps larger; 46 bits are far below the noise of the fluxes themselves.  The
// form holds for eps = sqrt(eps_mach)/|y| (the differences keep 2^-26 of U at most); a
// caller's own, larger eps takes the general form.
// Measured on GB300 (events around the launches; FP32 directions): Q3 160 x 80 elements
// 32.3 + 11.9 us, the general form as a face and a volume launch 33.0 + 40.7 (and
// 48.8 + 47.4 before the primitives of numeric.cuh); viscous Q2 256 x 32 31.6 + 9.1 against
// 49.0 + 30.9, Q4 320 x 160 151 + 37 against 191 + 267.  FP64 directions are scaled and
// split: 35.7, 34.8 and 178 us for the flux launch.  The 103,360 face points and 204,800
// nodes take 21.5 us of FP64 issue.

// Direction entries as two floats.  FP32 vectors are exact in the first part.  FP64 ones
// are scaled by the power of two that brings |y| (from eps = sqrt(eps_mach)/|y|) to about
// one, so that a direction of any magnitude keeps its 48 bits; `es` is eps scaled back.
template <class Y> struct Dir;
template <> struct Dir<float> {
    double es;
    JF_D explicit Dir(double eps) : es(eps) {}
    JF_D F2 operator()(float y) const { return F2{y, 0.0f}; }
};
template <> struct Dir<double> {
    double es;
    int k;
    JF_D explicit Dir(double eps) {
        const int hi = __double2hiint(eps), f = (hi >> 20) & 0x7ff;
        k = f - 997;   // binary exponent of eps, plus 26
        es = f ? __hiloint2double(hi - (k << 20), __double2loint(eps)) : eps * __hiloint2double(2020 << 20, 0);
    }
    JF_D F2 operator()(double y) const {
        const int hi = __double2hiint(y), f = (hi >> 20) & 0x7ff;
        if (f == 0x7ff) return split2(y);           // infinity, NaN
        if (f == 0 || f + k <= 0) return F2{0.0f, 0.0f};
        return split2(__hiloint2double(hi + (k << 20), __double2loint(y)));
    }
};
JF_D double y64(float y) { return f2d_normal(y); }
JF_D double y64(double y) { return y; }
JF_D double y64_any(float y) { return f2d_conv(y); }   // any input (NaN, infinity, subnormal)
JF_D double y64_any(double y) { return y; }

// ---- constants of a product ---------------------------------------------------
struct DGF {
    int nx, nz, n_el, periodic;
    double mu, eta_x, eta_z;
    float2 g;                       // gravity
    float2 lp[5], lm[5];            // l_q(+-1)
    float2 dl[2][2][5];             // [direction][end -1, +1]: (2/h) l_q'
    float2 D[2][5][5];              // weak-form derivative, 2/h folded in
    float2 Dn[2][5][5];             // (2/h) l_q'(xi_a): gradients at the nodes (viscous)
    float2 lift[8][5];              // as DGK::lift
    PhysC pc;
    const PowTab *pt;
    LinPtr lin;
};

constexpr int FD_MINB = 7;   // 72 registers: 28 warps an SM, no spills
constexpr int FD_MINV = 6;   // viscous, 80 registers: 31.3 us on Q2 256 x 32, 36.4 with 118 and no spills
// Difference of the face terms at U + eps y and U, one thread per face point (the linear
// index of the residual's face kernel).  Vertical and horizontal faces run the same code:
// the momentum components are exchanged for the latter.
template <class Y, int NP1, bool VISC>
JF_D void fd_faces(const DGF &K, const Y *y, double eps, float2 *phix, float2 *symx, float2 *phiz, float2 *symz,
                   unsigned blk) {
    constexpr int NP = NP1 * NP1;
    const Dir<Y> dir(eps);
    const int nx = K.nx, nz = K.nz;
    const size_t N1 = (size_t)K.n_el * NP;
    const long long nvert = (long long)nz * (nx + 1) * NP1, nf = nvert + (long long)(nz + 1) * nx * NP1;
    const long long t = (long long)blk * blockDim.x + threadIdx.x;
    if (t >= nf) return;
    const bool zf = t >= nvert;
    const int u = (int)(zf ? t - nvert : t);
    const int s = u % NP1, c = u / NP1;
    int eL, eR, iL, iR;          // elements of the two sides, first node of the lines there
    bool wallL, wallR;
    if (!zf) {
        const int fx = c % (nx + 1), ez = c / (nx + 1);
        wallL = fx == 0 && !K.periodic;
        wallR = fx == nx && !K.periodic;
        eL = ez * nx + (fx == 0 ? (K.periodic ? nx - 1 : 0) : fx - 1);
        eR = ez * nx + (fx == nx ? (K.periodic ? 0 : nx - 1) : fx);
        iL = iR = s * NP1;
    } else {
        const int ex = c % nx, fz = c / nx;
        wallL = fz == 0;
        wallR = fz == nz;
        eL = (wallL ? 0 : fz - 1) * nx + ex;
        eR = (wallR ? nz - 1 : fz) * nx + ex;
        iL = iR = s;
    }
    const int st = zf ? NP1 : 1;
    const size_t bL = (size_t)eL * NP + iL, bR = (size_t)eR * NP + iR;
    D64 UL[4], UR[4], gL[4], gR[4];
    D64 J[4];   // jump of the state (viscous), from the jump of U and that of y
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        F2 aL{0.f, 0.f}, aR{0.f, 0.f}, dL{0.f, 0.f}, dR{0.f, 0.f};
#pragma unroll
        for (int q = 0; q < NP1; ++q) {
            const F2 yl = dir(y[v * N1 + bL + q * st]), yr = dir(y[v * N1 + bR + q * st]);
            f2_fma(aL, f2(K.lp[q]), yl);
            f2_fma(aR, f2(K.lm[q]), yr);
            if (VISC) {
                f2_fma(dL, f2(K.dl[zf][1][q]), yl);
                f2_fma(dR, f2(K.dl[zf][0][q]), yr);
            }
        }
        const double tL = K.lin.tr[(2 * v) * nf + t], tR = K.lin.tr[(2 * v + 1) * nf + t];
        const double yL = join(aL), yR = join(aR);
        UL[v] = D64{__fma_rn(dir.es, yL, tL)};
        UR[v] = D64{__fma_rn(dir.es, yR, tR)};
        if (VISC) {
            gL[v] = D64{__fma_rn(dir.es, join(dL), K.lin.tr[(8 + 2 * v) * nf + t])};
            gR[v] = D64{__fma_rn(dir.es, join(dR), K.lin.tr[(9 + 2 * v) * nf + t])};
            J[v] = D64{__fma_rn(dir.es, __dsub_rn(yL, yR), K.lin.tr[(16 + v) * nf + t])};
        }
    }
    swap_d(zf, UL[1], UL[2]);
    swap_d(zf, UR[1], UR[2]);
    wall_states<D64, 0>(UL, UR, wallL, wallR);
    Side<D64> L, R;
    side_of(UL, K.pc, K.pt, L);
    side_of(UR, K.pc, K.pt, R);
    D64 H[4];
    hllc_s<D64, 0>(L, R, H);
    swap_d(zf, H[1], H[2]);
    float2 *phi = zf ? phiz : phix;
    const size_t fs = zf ? (size_t)(nf - nvert) : (size_t)nvert;
    double dP[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) dP[v] = __dsub_rn(H[v].x, K.lin.H[v * nf + t]);
    if (VISC) {
        float2 *sym = zf ? symz : symx;
        if (wallL || wallR) {
#pragma unroll
            for (int q = 0; q < 6; ++q) sym[(size_t)q * fs + u] = make_float2(0.f, 0.f);
        } else {
            swap_d(zf, L.U[1], L.U[2]);   // back to (u, w)
            swap_d(zf, R.U[1], R.U[2]);
            const D64 eta = D64{zf ? K.eta_z : K.eta_x}, hmu = D64{0.5 * K.mu};
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int v = q + 1;
                const D64 pL = L.U[v] * L.ir, pR = R.U[v] * R.ir;
                const D64 sL = hmu * visc_c(pL, J[0], J[v]), sR = hmu * visc_c(pR, J[0], J[v]);
                const D64 V = visc_face(hmu, eta, pL, pR, gL, gR, v, sL, sR);
                dP[v] = __dsub_rn(dP[v], __dsub_rn(V.x, K.lin.H[(4 + q) * nf + t]));
                sym[(size_t)q * fs + u] = f2v(split2(__dsub_rn(sL.x, K.lin.H[(7 + q) * nf + t])));
                sym[(size_t)(3 + q) * fs + u] = f2v(split2(__dsub_rn(sR.x, K.lin.H[(10 + q) * nf + t])));
            }
        }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) phi[v * fs + u] = f2v(split2(dP[v]));
}

// Differences of the node fluxes and their weak-form derivatives, blockDim.x / NP
// elements per block, one thread per node; the sums go to `part` (two-float, [4][nodes]).
template <class Y, int NP1, bool VISC>
JF_D void fd_nodes(const DGF &K, const Y *y, double eps, float2 *part, unsigned blk) {
    constexpr int NP = NP1 * NP1, EPB = 128 / NP;
    __shared__ float2 sF[2][EPB][4][NP];              // flux differences
    __shared__ float2 sy[VISC ? EPB : 1][4][VISC ? NP : 1];
    __shared__ float2 sD[2][NP1][NP1], sDn[VISC ? 2 : 1][NP1][NP1];
    const Dir<Y> dir(eps);
    const int epb = blockDim.x / NP;
    const int le = threadIdx.x / NP, node = threadIdx.x % NP;
    const int a = node % NP1, b = node / NP1;
    const int e = (int)blk * epb + le;
    const bool active = le < epb && e < K.n_el;
    const size_t N1 = (size_t)K.n_el * NP, gi0 = (size_t)e * NP + node;
    for (int i = threadIdx.x; i < 2 * NP; i += blockDim.x) {
        const int d = i / NP, r = (i % NP) / NP1, q = i % NP1;
        sD[d][r][q] = K.D[d][r][q];
        if (VISC) sDn[d][r][q] = K.Dn[d][r][q];
    }
    Y yv[4];
    if (active) {
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            yv[v] = y[v * N1 + gi0];
            if (VISC) sy[le][v][node] = f2v(dir(yv[v]));
        }
    }
    if (VISC) __syncthreads();
    const F2 e2 = split2(dir.es);
    if (active) {
        D64 U[4];
#pragma unroll
        for (int v = 0; v < 4; ++v) U[v] = D64{__fma_rn(eps, y64(yv[v]), K.lin.U[v * N1 + gi0])};
        const D64 ir = jrcp(U[0]);
        const D64 p = pressure(U[3], K.pc, K.pt);
        const D64 vu = U[1] * ir, vw = U[2] * ir;
        D64 Fx[4], Fz[4];
        flux_xz(U, vu, vw, p, Fx, Fz);
        sF[0][le][0][node] = f2v(f2_mul(e2, dir(yv[1])));   // the mass fluxes are linear
        sF[1][le][0][node] = f2v(f2_mul(e2, dir(yv[2])));
        if (VISC) {
            D64 dx[4], dz[4];
#pragma unroll
            for (int v = 0; v < 4; ++v) {
                F2 sx{0.f, 0.f}, sz{0.f, 0.f};
#pragma unroll
                for (int q = 0; q < NP1; ++q) {
                    f2_fma(sx, f2(sDn[0][a][q]), f2(sy[le][v][b * NP1 + q]));
                    f2_fma(sz, f2(sDn[VISC ? 1 : 0][b][q]), f2(sy[le][v][q * NP1 + a]));
                }
                dx[v] = D64{__fma_rn(dir.es, join(sx), K.lin.F[(5 + v) * N1 + gi0])};
                dz[v] = D64{__fma_rn(dir.es, join(sz), K.lin.F[(9 + v) * N1 + gi0])};
            }
            const D64 phi[4] = {vu, vu, vw, U[3] * ir};
            const D64 mu = D64{K.mu};
#pragma unroll
            for (int v = 1; v < 4; ++v) {
                const double gx = (mu * visc_c(phi[v], dx[0], dx[v])).x, gz = (mu * visc_c(phi[v], dz[0], dz[v])).x;
                // convective and viscous differences each against their stored values
                const int fz = v == 1 ? 1 : v + 1;   // F: x1, x2 = z1, x3, z2, z3
                sF[0][le][v][node] = f2v(split2(__dsub_rn(__dsub_rn(Fx[v].x, K.lin.F[(v - 1) * N1 + gi0]),
                                                          __dsub_rn(gx, K.lin.F[(12 + v) * N1 + gi0]))));
                sF[1][le][v][node] = f2v(split2(__dsub_rn(__dsub_rn(Fz[v].x, K.lin.F[fz * N1 + gi0]),
                                                          __dsub_rn(gz, K.lin.F[(15 + v) * N1 + gi0]))));
            }
        } else {
            const float2 d2 = f2v(split2(__dsub_rn(Fx[2].x, K.lin.F[1 * N1 + gi0])));
            sF[0][le][1][node] = f2v(split2(__dsub_rn(Fx[1].x, K.lin.F[0 * N1 + gi0])));
            sF[0][le][2][node] = d2;
            sF[0][le][3][node] = f2v(split2(__dsub_rn(Fx[3].x, K.lin.F[2 * N1 + gi0])));
            sF[1][le][1][node] = d2;
            sF[1][le][2][node] = f2v(split2(__dsub_rn(Fz[2].x, K.lin.F[3 * N1 + gi0])));
            sF[1][le][3][node] = f2v(split2(__dsub_rn(Fz[3].x, K.lin.F[4 * N1 + gi0])));
        }
    }
    __syncthreads();
    if (!active) return;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        F2 f{0.f, 0.f};
#pragma unroll
        for (int q = 0; q < NP1; ++q) {
            f2_fma(f, f2(sD[0][a][q]), f2(sF[0][le][v][b * NP1 + q]));
            f2_fma(f, f2(sD[1][b][q]), f2(sF[1][le][v][q * NP1 + a]));
        }
        if (v == 2) f2_fma(f, f2_neg(f2(K.g)), f2_mul(e2, dir(yv[0])));
        part[v * N1 + gi0] = f2v(f);
    }
}

// Both in one launch; neither needs the other (the lift below adds them).  The face
// blocks, FP64 work from end to end, come first, so that the shorter node blocks, part
// two-float sums, fill the last wave: 31.8 us on Q3 160 x 80, 34.7 with the face blocks
// dealt evenly among the node blocks, 52 as two launches with the lift in the second.
// The first block also leaves alpha dt / eps for the lift.
template <class Y, int NP1, bool VISC>
struct k_fd_flux_b {
    static constexpr int TPB = 128, MINB = VISC ? FD_MINV : FD_MINB;
    static constexpr bool GROUP = !VISC;   // a grouped twin is built (lock-step ensembles)
    static __device__ __forceinline__ void run(unsigned jf_bid, unsigned jf_nblk, JfArg<DGF> K, JfArg<unsigned> nface,
                                               JfArg<const Y *> y, JfArg<const double *> epsp, JfArg<double> adt,
                                               JfArg<double *> cepsp, JfArg<float2 *> part, JfArg<float2 *> phix,
                                               JfArg<float2 *> symx, JfArg<float2 *> phiz, JfArg<float2 *> symz) {
        jf_pdl_enter();
        const double eps = *epsp;
        if (jf_bid == 0 && threadIdx.x == 0) *cepsp = eps != 0.0 ? adt / eps : 0.0;
        if (jf_bid < nface) fd_faces<Y, NP1, VISC>(K, y, eps, phix, symx, phiz, symz, jf_bid);
        else fd_nodes<Y, NP1, VISC>(K, y, eps, part, jf_bid - nface);
    }
};
template <class Y, int NP1, bool VISC>
__global__ void __launch_bounds__(128, VISC ? FD_MINV : FD_MINB)
    k_fd_flux(DGF K, unsigned nface, const Y *y, const double *epsp, double adt, double *cepsp, float2 *part,
              float2 *phix, float2 *symx, float2 *phiz, float2 *symz) {
    k_fd_flux_b<Y, NP1, VISC>::run(blockIdx.x, gridDim.x, K, nface, y, epsp, adt, cepsp, part, phix, symx, phiz, symz);
}

// Adds the lifts of the face terms to the node sums, one thread per node, and closes: the
// product (MODE DG_JV) or a pseudo-time step of the FP64 preconditioner (DG_SMOOTH64).
template <class Y, int MODE, int NP1, bool VISC>
struct k_fd_lift_b {
    static constexpr int TPB = 256, MINB = VISC ? 4 : 5;
    static constexpr bool GROUP = !VISC && MODE == DG_JV;   // a grouped twin is built (lock-step ensembles)
    static __device__ __forceinline__ void run(unsigned jf_bid, unsigned jf_nblk, JfArg<DGF> K, JfArg<DGArgs> A,
                                               JfArg<const Y *> y, JfArg<const double *> cepsp,
                                               JfArg<const float2 *> part, JfArg<const float2 *> phix,
                                               JfArg<const float2 *> symx, JfArg<const float2 *> phiz,
                                               JfArg<const float2 *> symz) {
        jf_pdl_enter();
        constexpr int NP = NP1 * NP1;
        __shared__ float2 sl[8][NP1];
        for (int i = threadIdx.x; i < 8 * NP1; i += blockDim.x) sl[i / NP1][i % NP1] = K.lift[i / NP1][i % NP1];
        const int N1 = K.n_el * NP, n = (int)jf_bid * (int)blockDim.x + (int)threadIdx.x;
        const double ceps = *cepsp;
        const bool eps0 = (__double_as_longlong(*A.eps) << 1) == 0;
        __syncthreads();
        if (n >= N1) return;
        const int e = n / NP, node = n % NP, a = node % NP1, b = node / NP1;
        const int nx = K.nx, nz = K.nz, ez = e / nx, ex = e - ez * nx;
        const int fsx = nz * (nx + 1) * NP1, fsz = (nz + 1) * nx * NP1;
        const float2 *pL = phix + (ez * (nx + 1) + ex) * NP1 + b, *pB = phiz + (ez * nx + ex) * NP1 + a;
        const int dT = nx * NP1;
#pragma unroll
        for (int v = 0; v < 4; ++v) {
            const size_t gi = (size_t)v * N1 + n;
            const Y yv = y[gi];
            F2 f = f2(part[gi]);
            f2_fma(f, f2(sl[0][a]), f2(pL[(size_t)v * fsx]));
            f2_fma(f, f2_neg(f2(sl[1][a])), f2(pL[(size_t)v * fsx + NP1]));
            f2_fma(f, f2(sl[4][b]), f2(pB[(size_t)v * fsz]));
            f2_fma(f, f2_neg(f2(sl[5][b])), f2(pB[(size_t)v * fsz + dT]));
            if (VISC && v > 0) {
                const int q = v - 1;
                const float2 *sL = symx + (pL - phix), *sB = symz + (pB - phiz);
                f2_fma(f, f2(sl[2][a]), f2(sL[(size_t)(3 + q) * fsx]));
                f2_fma(f, f2(sl[3][a]), f2(sL[(size_t)q * fsx + NP1]));
                f2_fma(f, f2(sl[6][b]), f2(sB[(size_t)(3 + q) * fsz]));
                f2_fma(f, f2(sl[7][b]), f2(sB[(size_t)q * fsz + dT]));
            }
            // eps = 0: y = 0, or |y| not finite -- the product is y
            const double Jz = eps0 ? y64_any(yv) : __fma_rn(-ceps, join(f), y64(yv));
            if (MODE == DG_JV) {
                ((double *)A.out0)[gi] = Jz;
            } else {
                const double z = y64(yv);
                if (A.z0mode == 0) {
                    ((double *)A.out0)[gi] = z + A.dtau[e] * (A.r[gi] - Jz);
                } else {
                    const double stp = (A.alpha * A.dtau[e]) * (A.r[gi] - Jz);
                    ((double *)A.out0)[gi] = A.z0mode == 1 ? ((const double *)A.z0)[gi] + stp : stp;
                }
            }
        }
    }
};
template <class Y, int MODE, int NP1, bool VISC>
__global__ void __launch_bounds__(256, VISC ? 4 : 5)
    k_fd_lift(DGF K, DGArgs A, const Y *y, const double *cepsp, const float2 *part, const float2 *phix,
              const float2 *symx, const float2 *phiz, const float2 *symz) {
    k_fd_lift_b<Y, MODE, NP1, VISC>::run(blockIdx.x, gridDim.x, K, A, y, cepsp, part, phix, symx, phiz, symz);
}

inline float2 split_host(double d) {
    const float h = (float)d;
    return make_float2(h, (float)(d - (double)h));
}
inline DGF make_F(jfnk_ctx *c) {
    DGF F = {};
    const DGTab &T = c->tab;
    F.nx = c->grid.nx;
    F.nz = c->grid.nz;
    F.n_el = c->n_el;
    F.periodic = c->grid.periodic_x;
    F.mu = c->phys.mu;
    const double n1 = c->np1, s[2] = {2.0 / c->hx, 2.0 / c->hz};
    F.eta_x = c->opts.c_ip * n1 * n1 / c->hx;
    F.eta_z = c->opts.c_ip * n1 * n1 / c->hz;
    F.g = split_host(c->phys.g);
    for (int q = 0; q < 5; ++q) {
        F.lp[q] = split_host(T.lp[q]);
        F.lm[q] = split_host(T.lm[q]);
        for (int d = 0; d < 2; ++d) {
            F.dl[d][0][q] = split_host(s[d] * T.dlm[q]);
            F.dl[d][1][q] = split_host(s[d] * T.dlp[q]);
            F.lift[4 * d][q] = split_host(s[d] * T.lmw[q]);
            F.lift[4 * d + 1][q] = split_host(s[d] * T.lpw[q]);
            F.lift[4 * d + 2][q] = split_host(s[d] * s[d] * T.dlmw[q]);
            F.lift[4 * d + 3][q] = split_host(s[d] * s[d] * T.dlpw[q]);
            for (int r = 0; r < 5; ++r) {
                F.D[d][r][q] = split_host(s[d] * T.Dw[r][q]);
                F.Dn[d][r][q] = split_host(s[d] * T.Dn[r][q]);
            }
        }
    }
    F.pc = c->pc;
    F.pt = c->powtab;
    F.lin = c->lin;
    return F;
}

// The product (or smoothing step) about the context's linearisation; a.yf: FP32
// direction, else a.y.
template <class Y, int MODE, int NP1, bool VISC>
int launch_fd(jfnk_ctx *c, const DGArgs &a, const Y *y, cudaStream_t s) {
    const DGF K = make_F(c);
    float2 *phix = (float2 *)c->phix, *symx = (float2 *)c->symx, *phiz = (float2 *)c->phiz, *symz = (float2 *)c->symz;
    const long long nf = (long long)K.nz * (K.nx + 1) * NP1 + (long long)(K.nz + 1) * K.nx * NP1;
    if (c->timing) JF_CK(cudaEventRecord(c->tev[0], s));
    const int epb = spread_elements<NP1>(c->opts.tile_volume, K.n_el, c->n_sm), tb = epb * NP1 * NP1;
    const unsigned nface = (unsigned)((nf + tb - 1) / tb), nnode = (unsigned)((K.n_el + epb - 1) / epb);
    float2 *part = (float2 *)a.out0;   // the node sums, until the lift closes them in place
    double *cepsp = c->scal + S_CEPS;
    jf_launch<k_fd_flux_b<Y, NP1, VISC>>(k_fd_flux<Y, NP1, VISC>, nface + nnode, tb, 0, s, K, nface, y, a.eps, a.adt, cepsp,
                                         part, phix, symx, phiz, symz);
    jf_launched();
    if (c->timing) JF_CK(cudaEventRecord(c->tev[1], s));
    const int tl = spread_threads(256, c->npt, c->n_sm);
    jf_launch<k_fd_lift_b<Y, MODE, NP1, VISC>>(k_fd_lift<Y, MODE, NP1, VISC>, (unsigned)((c->npt + tl - 1) / tl), tl, 0, s,
                                               K, a, y, (const double *)cepsp, (const float2 *)part, (const float2 *)phix,
                                               (const float2 *)symx, (const float2 *)phiz, (const float2 *)symz);
    jf_launched();
    JF_CK(cudaGetLastError());
    return timing_close(c, s);
}
