// FP64 Runge-Kutta stage on a Cartesian-product grid x(i), y(j), z(k) with
// positive spacings (the box meshes of the jet runs): the same method as the
// four kernels of les_stage.cu with the zeros of its diagonal metric left out.
//
// Why.  GB300 issues two FP64 operations per clock and SM, so the FP64 stage
// costs what it counts: the general kernels issue 558 FP64 instructions per
// point and stage, and on such a grid most of them multiply or add the six
// cofactors that are exact zeros.  With h_a the spacing along axis a, the
// cofactor of axis a is the face area S_a = h_b h_d, the interface J^-1 is
// S_a hb (hb the mean of the two spacings along a), and d/dx_a =
// (1/h_a) d/dxi_a.  The stage then works on interface fluxes divided by the
// face area and doubled, G_a = 2 H_a / S_a,
//   G = F_L + F_R - sc [eps2 dW - eps4 d3W] - viscous,   sc = hb (lb_L + lb_R),
// with F the Cartesian point fluxes (nine products, rho u_i u_j is symmetric),
// and the update multiplies each flux difference by S_a / 2 once.
// FP64 instructions per point: point 69, gradients 66, interfaces 162, update 34 =
// 332.  Measured on the 384x256x144 jet, us per launch, general -> this form:
// point 2740 -> 1805, gradients 2710 -> 1703, interfaces 8385 -> 4201 (FP64 pipe
// 85-88 % busy in each), update 952 -> 897.
// Tangential derivatives reach the interface as c_ai = (1/2) du_a/dx_i and the
// divergence as the third s_a = (1/3) sum_{i != a} du_i/dx_i of each point, so
// that the sums over the two points need no factor.
// Everything that is not FP64 arithmetic (index arithmetic, maxima of
// non-negative numbers as integers, loads) is nearly free beside it.
// Blocks of 64 threads: on a small grid the last wave is what counts (48x32x32
// has 192 blocks of 256 threads for 152 SMs: 40 SMs work twice as long).
#include <cmath>

#include "les_fp64.cuh"
#include "les_internal.cuh"

namespace les {

namespace {

constexpr int PB = PROD_BLOCK;

__constant__ double c_alpha_p[5] = {0.25, 1.0 / 6.0, 0.375, 0.5, 1.0};

// Point fields (in the scratch of the general form's point fields)
enum {
    R_RHO = 0, R_U, R_V, R_W, R_T, R_RU, R_RV, R_RW, R_RH, R_P, R_MU, R_LB, // + a
    R_M = R_LB + 3, // rho u_i u_j (+ p on the diagonal): xx xy xz yy yz zz
    R_E = R_M + 6,  // rho H u_a
    R_COUNT = R_E + 3
};
static_assert(R_COUNT <= NPRIM, "point scratch");
// Derivative fields
enum { D_NU = 0, D_MUE = 3, D_KAP, D_S, /* + a */ D_C = D_S + 3 /* + 2 a + (rank of i) */, D_COUNT = D_C + 6 };
static_assert(D_COUNT <= NGRAD, "derivative scratch");

// index of (i, j) in the symmetric M
__host__ __device__ constexpr int sym(int i, int j) { return i > j ? sym(j, i) : (i == 0 ? j : (i == 1 ? 2 + j : 5)); }

// Spacing tables (see PROD_TABS) of one axis
struct Tab {
    const double *t;
    int n;
    __device__ __forceinline__ double operator()(int which, int q) const { return __ldg(t + which * n + q); }
};

// Point of block vb, thread threadIdx.x: jet, padded index, indices; false
// for padding.  32-bit arithmetic: an FP64 jet of 2^31 padded points would
// need 2.5 TB.
struct Pt {
    int lp, q[3];
};
__device__ __forceinline__ bool point_at(const JetDev<double> &J, int b, Pt &p)
{
    p.lp = b * PB + (int)threadIdx.x;
    const int r = p.lp / J.pitch;
    p.q[0] = p.lp - r * J.pitch;
    p.q[2] = r / J.n[1];
    p.q[1] = r - p.q[2] * J.n[1];
    return p.lp < J.npts_pad && p.q[0] < J.n[0];
}
// The point's index with its index along axis a replaced by `to`.
template <int a> __device__ __forceinline__ int moved(const JetDev<double> &J, const Pt &p, int to)
{
#if defined(LES_BOUNDS_CHECK) && defined(__CUDA_ARCH__)
    int r[3] = {p.q[0], p.q[1], p.q[2]};
    r[a] = to;
    return (int)lidx(J, r[0], r[1], r[2]);
#else
    const int st = a == 0 ? 1 : (a == 1 ? J.pitch : J.pitch * J.n[1]);
    return p.lp + (to - p.q[a]) * st;
#endif
}
// Neighbour index along a: wrapped on a periodic axis.
__device__ __forceinline__ int up1(int q, int n, int per) { return per && q + 1 == n ? 0 : q + 1; }
__device__ __forceinline__ int dn1(int q, int n, int per) { return per && q == 0 ? n - 1 : q - 1; }

} // namespace

__global__ void __launch_bounds__(PB) k_point_prod(const JetDev<double> *__restrict__ jets, BlockMap bm, int src)
{
    for (int vb = blockIdx.x; vb < bm.total; vb += gridDim.x) {
        const int jet = find_jet(bm, vb);
        const JetDev<double> &J = jets[jet];
        Pt pt;
        if (!point_at(J, vb - bm.start[jet], pt)) continue;
        const long long fs = J.fs;
        const double *__restrict__ Q = J.q[src] + pt.lp;
        double *__restrict__ P = J.prim + pt.lp;
        const double rj = J.met[MET_J * fs + pt.lp];
        const double rho = Q[0] * rj;
        const double m[3] = {Q[fs] * rj, Q[2 * fs] * rj, Q[3 * fs] * rj};
        const double e = Q[4 * fs] * rj;
        const double rr = rcp64(rho);
        const double u[3] = {m[0] * rr, m[1] * rr, m[2] * rr};
        const double ke2 = fma(m[2], u[2], fma(m[1], u[1], m[0] * u[0]));
        const double p = J.gm1 * fma(-0.5, ke2, e);
        const double T = J.gamma * p * rr;
        const double c = sqrt64(T); // speed of sound: c^2 = gamma p / rho = T in jet units
        P[R_MU * fs] = T * c * J.suth1 * rcp64_1(T + J.suth_S);
        const double rH = e + p;
        P[R_RHO * fs] = rho;
        P[R_T * fs] = T;
        P[R_P * fs] = p;
        P[R_RH * fs] = rH;
        double s[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            P[(R_U + a) * fs] = u[a];
            P[(R_RU + a) * fs] = m[a];
            P[(R_E + a) * fs] = rH * u[a];
#pragma unroll
            for (int i = a; i < 3; ++i)
                P[(R_M + sym(a, i)) * fs] = i == a ? fma(m[a], u[a], p) : m[a] * u[i];
            s[a] = sqrt64((fabs(u[a]) + c) * Tab{J.ptab[a], J.n[a]}(PT_RH, pt.q[a]));
        }
        // lambda-bar_a = s_a (s_a + s_b + s_d), s = lambda^1/2
        const double ss = s[0] + s[1] + s[2];
#pragma unroll
        for (int a = 0; a < 3; ++a) P[(R_LB + a) * fs] = s[a] * ss;
    }
}

// d[i] = the doubled central difference along a of u_i (one-sided three-point
// at the ends of a non-periodic axis), nu = the pressure sensor (the interior
// neighbour's at an end).
template <int a>
__device__ __forceinline__ void axis_diff(const JetDev<double> &J, const Pt &pt, double d[3], double &nu)
{
    const long long fs = J.fs;
    const double *__restrict__ P = J.prim;
    const int q = pt.q[a], n = J.n[a], per = J.per[a];
    const bool end = !per && (q == 0 || q == n - 1);
    // central: the two neighbours; at an end the points one and two inside
    const int t = q == 0 ? 1 : -1;
    const int o1 = moved<a>(J, pt, end ? q + t : dn1(q, n, per)), o2 = moved<a>(J, pt, end ? q + 2 * t : up1(q, n, per));
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const double *F = P + (R_U + i) * fs;
        d[i] = F[o2] - F[o1];
    }
    // a vote, so that this stays a branch: as predicated instructions the
    // one-sided form cost every point a third of the pass (93 instead of 63
    // FP64 instructions, 2444 instead of 1682 us on the 384x256x144 jet)
    if (__ballot_sync(__activemask(), end)) {
        if (end) {
            const double td = t > 0 ? 1.0 : -1.0;
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const double *F = P + (R_U + i) * fs;
                d[i] = td * fma(-3.0, F[pt.lp], fma(3.0, F[o1], -d[i])); // t (4 f1 - 3 f0 - f2)
            }
        }
    }
    const double *F = P + R_P * fs;
    const double p0 = F[pt.lp], p1 = F[o1], p2 = F[o2];
    const double pc = end ? p1 : p0;
    const double s = p2 + (end ? p0 : p1);
    nu = fabs(fma(-2.0, pc, s)) * rcp64_1(fma(2.0, pc, s));
}

__global__ void __launch_bounds__(PB) k_grads_prod(const JetDev<double> *__restrict__ jets, BlockMap bm)
{
    for (int vb = blockIdx.x; vb < bm.total; vb += gridDim.x) {
        const int jet = find_jet(bm, vb);
        const JetDev<double> &J = jets[jet];
        Pt pt;
        if (!point_at(J, vb - bm.start[jet], pt)) continue;
        const long long fs = J.fs;
        const double *__restrict__ P = J.prim + pt.lp;
        double *__restrict__ G = J.grad + pt.lp;
        double d[3][3], nu[3]; // d[a][i]
        axis_diff<0>(J, pt, d[0], nu[0]);
        axis_diff<1>(J, pt, d[1], nu[1]);
        axis_diff<2>(J, pt, d[2], nu[2]);
        double c[3][3]; // c[i][a]: du_i/dx_a, halved off the diagonal, a third of it on the diagonal
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const Tab t{J.ptab[a], J.n[a]};
            const double r4 = t(PT_RH4, pt.q[a]);
#pragma unroll
            for (int i = 0; i < 3; ++i) c[i][a] = d[a][i] * (i == a ? t(PT_RH6, pt.q[a]) : r4);
            G[(D_NU + a) * fs] = nu[a] * J.k2;
        }
        // 2 S_ij S_ij = 2 sum (3 c_ii)^2 + sum_{i<j} (2 (c_ij + c_ji))^2 = 4 (4.5 sd + so)
        const double a01 = c[0][1] + c[1][0], a02 = c[0][2] + c[2][0], a12 = c[1][2] + c[2][1];
        const double sd = fma(c[2][2], c[2][2], fma(c[1][1], c[1][1], c[0][0] * c[0][0]));
        const double so = fma(a12, a12, fma(a02, a02, a01 * a01));
        // Smagorinsky: mu_sgs = rho (Cs Delta)^2 (2 S_ij S_ij)^1/2
        const double mus = P[R_RHO * fs] * J.met[MET_CSD2 * fs + pt.lp] * twice_sqrt64(fma(4.5, sd, so));
        const double mu = P[R_MU * fs];
        G[D_MUE * fs] = fma(mu, J.inv_Re, mus);
        G[D_KAP * fs] = fma(mu, J.kap_mol, mus * J.kap_sgs);
        G[(D_S + 0) * fs] = c[1][1] + c[2][2];
        G[(D_S + 1) * fs] = c[0][0] + c[2][2];
        G[(D_S + 2) * fs] = c[0][0] + c[1][1];
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int k = 0; k < 2; ++k) G[(D_C + 2 * a + k) * fs] = c[a][k == 0 ? (a == 0 ? 1 : 0) : (a == 2 ? 1 : 2)];
    }
}

// G_a of the interface between the point and its +a neighbour.
template <int a> __device__ __forceinline__ void iface_prod(const JetDev<double> &J, const Pt &pt, double *__restrict__ H)
{
    const long long fs = J.fs;
    const double *__restrict__ P = J.prim;
    const double *__restrict__ G = J.grad;
    const int q = pt.q[a], n = J.n[a], per = J.per[a];
    const int qR = up1(q, n, per);
    const int L = pt.lp, R = moved<a>(J, pt, qR);
    // mirrored differences at a non-periodic end: W(L-1) = W(R), W(R+1) = W(L)
    const int Lm = !per && q == 0 ? R : moved<a>(J, pt, dn1(q, n, per));
    const int Rp = !per && qR == n - 1 ? L : moved<a>(J, pt, up1(qR, n, per));
    const Tab tab{J.ptab[a], n};
    // Turkel-Vatsa coefficients (the stored sensors carry k2)
    const double eps2 = max_nn(G[(D_NU + a) * fs + L], G[(D_NU + a) * fs + R]);
    const double eps4 = clamp0(J.k4 - eps2);
    const double sc = tab(PT_HB, q) * (P[(R_LB + a) * fs + L] + P[(R_LB + a) * fs + R]);
    const double se4 = sc * eps4;
    const double c2 = sc * fma(3.0, eps4, eps2);
    double h[5];
#pragma unroll
    for (int f = 0; f < 5; ++f) {
        const double *W = P + (f == 0 ? R_RHO : (f < 4 ? R_RU + f - 1 : R_RH)) * fs;
        const double *F = P + (f == 0 ? R_RU + a : (f < 4 ? R_M + sym(a, f - 1) : R_E + a)) * fs;
        h[f] = fma(c2, W[L] - W[R], fma(se4, W[Rp] - W[Lm], F[L] + F[R]));
    }
    // viscous + SGS: 2 tau_ai = (mu_L + mu_R) g_i with g_i = du_i/dx_a + du_a/dx_i
    // (i != a) and g_a = (4/3) du_a/dx_a - (2/3) sum_{i != a} du_i/dx_i
    const double rhb = tab(PT_RHB, q), c43 = tab(PT_RHB43, q);
    const double mu = G[D_MUE * fs + L] + G[D_MUE * fs + R];
    double su = 0.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const double *U = P + (R_U + i) * fs;
        const double uL = U[L], uR = U[R];
        double g;
        if (i == a) {
            const double *S = G + (D_S + a) * fs;
            g = fma(c43, uR - uL, -(S[L] + S[R]));
        } else {
            const double *C = G + (D_C + 2 * a + (i > a ? i - 1 : i)) * fs;
            g = fma(rhb, uR - uL, C[L] + C[R]);
        }
        h[1 + i] = fma(-mu, g, h[1 + i]);
        su = i == 0 ? (uL + uR) * g : fma(uL + uR, g, su);
    }
    // energy: 2 tau . u_interface + 2 kappa dT/dx_a
    const double *T = P + R_T * fs;
    const double dT = (T[R] - T[L]) * rhb;
    h[4] = fma(-0.5 * mu, su, h[4]);
    h[4] = fma(-(G[D_KAP * fs + L] + G[D_KAP * fs + R]), dT, h[4]);
#pragma unroll
    for (int f = 0; f < 5; ++f) H[f * fs] = h[f];
}

__global__ void __launch_bounds__(PB) k_iface_prod(const JetDev<double> *__restrict__ jets, BlockMap bm)
{
    for (int vb = blockIdx.x; vb < bm.total; vb += gridDim.x) {
        const int jet = find_jet(bm, vb);
        const JetDev<double> &J = jets[jet];
        Pt pt;
        if (!point_at(J, vb - bm.start[jet], pt)) continue;
        // an interface is used when the point is not an end of the two other
        // axes; there is none beyond the last point of a non-periodic axis
        bool in[3], last[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            last[a] = !J.per[a] && pt.q[a] == J.n[a] - 1;
            in[a] = J.per[a] || (pt.q[a] > 0 && !last[a]);
        }
        double *H = J.hflux + pt.lp;
        if (in[1] && in[2] && !last[0]) iface_prod<0>(J, pt, H);
        if (in[0] && in[2] && !last[1]) iface_prod<1>(J, pt, H + 5 * J.fs);
        if (in[0] && in[1] && !last[2]) iface_prod<2>(J, pt, H + 10 * J.fs);
    }
}

__global__ void __launch_bounds__(PB) k_update_prod(const JetDev<double> *__restrict__ jets, BlockMap bm, int dst,
                                                    int stage, const double *__restrict__ dt, int rhs_only)
{
    for (int vb = blockIdx.x; vb < bm.total; vb += gridDim.x) {
        const int jet = find_jet(bm, vb);
        const JetDev<double> &J = jets[jet];
        Pt pt;
        if (!point_at(J, vb - bm.start[jet], pt)) continue;
        const long long fs = J.fs;
        if (!interior(J, pt.q)) {
            if (rhs_only)
                for (int f = 0; f < NF; ++f) J.rhs[f * fs + pt.lp] = 0.0;
            continue;
        }
        const int back[3] = {moved<0>(J, pt, dn1(pt.q[0], J.n[0], J.per[0])),
                             moved<1>(J, pt, dn1(pt.q[1], J.n[1], J.per[1])),
                             moved<2>(J, pt, dn1(pt.q[2], J.n[2], J.per[2]))};
        // S_a / 2 times the flux differences' sum over a: the first axis's half area
        // s outside, the other two areas as ratios to it, so that the state is
        // rounded once.  (Three multiply-adds onto Q(0), as many operations, rounded
        // it three times: error against 64-bit torch after ten steps 4.3e-16 on
        // 48x32x32 and after four 2.3e-16 on 384x256x144, so 3.8e-16 and 1.9e-16.)
        const Tab X{J.ptab[0], J.n[0]}, Y{J.ptab[1], J.n[1]}, Z{J.ptab[2], J.n[2]};
        const double hx = X(PT_H, pt.q[0]);
        const double r1 = hx * Y(PT_RH, pt.q[1]), r2 = hx * Z(PT_RH, pt.q[2]);
        const double half = rhs_only ? 0.5 : -0.5 * (c_alpha_p[stage] * dt[jet]);
        const double s = Y(PT_H, pt.q[1]) * Z(PT_H, pt.q[2]) * half;
        const double *__restrict__ H = J.hflux;
        const double *Q0 = J.q[0];
        double *D = rhs_only ? J.rhs : J.q[dst];
#pragma unroll
        for (int f = 0; f < NF; ++f) {
            double d[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const double *Ha = H + (5 * a + f) * fs;
                d[a] = Ha[pt.lp] - Ha[back[a]];
            }
            const double sum = fma(r2, d[2], fma(r1, d[1], d[0]));
            D[f * fs + pt.lp] = fma(s, sum, rhs_only ? 0.0 : Q0[f * fs + pt.lp]);
        }
    }
}

void launch_stage_prod(const JetDev<double> *jets, BlockMap bm, int part, int src, int dst, int stage,
                       const double *dt, int rhs_only, int grid, cudaStream_t st)
{
    switch (part) {
    case 0: k_point_prod<<<grid, PB, 0, st>>>(jets, bm, src); break;
    case 1: k_grads_prod<<<grid, PB, 0, st>>>(jets, bm); break;
    case 2: k_iface_prod<<<grid, PB, 0, st>>>(jets, bm); break;
    default: k_update_prod<<<grid, PB, 0, st>>>(jets, bm, dst, stage, dt, rhs_only); break;
    }
}

} // namespace les
