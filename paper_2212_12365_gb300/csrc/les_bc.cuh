// Boundary conditions (Sec. "Boundary Conditions") at a face point, in the
// arithmetic of the storage precision.
#pragma once

#include "les_fp64.cuh"
#include "les_internal.cuh"
#include "les_pair.cuh"

namespace les {

// Products that a sum takes up are written as fma here, so that every
// compilation of this code gives the same bits (the pass exists for single jets
// and for batches).
template <typename T> __device__ __forceinline__ T dot3(const T *a, const T *b)
{
    return fma(a[2], b[2], fma(a[1], b[1], a[0] * b[0]));
}
__device__ __forceinline__ double sum_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float sum_rn(float a, float b) { return __fadd_rn(a, b); }

// Constants of the FP64 boundary arithmetic: gamma, gamma - 1, 1/(gamma-1),
// 1/gamma, 2/(gamma-1), ambient density and speed of sound.
struct BcD {
    double g, gm1, g1, rg, e2, TR, cinf;
};

__device__ __forceinline__ void cons_d(double rho, const double u[3], double p, const BcD &k, double Q[5])
{
    Q[0] = rho;
    Q[1] = rho * u[0];
    Q[2] = rho * u[1];
    Q[3] = rho * u[2];
    Q[4] = fma(p, k.g1, 0.5 * rho * dot3(u, u));
}

// Far field (Sec. "Far Field Boundary"): Riemann invariants along the unit
// outward normal n; R- from the ambient at rest, R+ from the interior point.
// With R+- = q_n +- 2c/(gamma-1): q_n,f = q_n,e/2 + (c_e - c_inf)/(gamma-1),
// c_f = (gamma-1) q_n,e/4 + (c_e + c_inf)/2, and the isentropic density
// (rho_e^gamma c_f^2 / (gamma p_e))^(1/(gamma-1)) is rho_e (c_f/c_e)^(2/(gamma-1))
// since gamma p_e = rho_e c_e^2 (on inflow the same with the ambient state):
// one exp and one log in place of two powers.
__device__ __forceinline__ void bc_farfield(const BcD &k, const double Qe[5], const double n[3], double Qf[5])
{
    const double rr = rcp64(Qe[0]);
    const double u[3] = {Qe[1] * rr, Qe[2] * rr, Qe[3] * rr};
    const double pe = k.gm1 * fma(-0.5, dot3(Qe + 1, u), Qe[4]);
    const double ce = sqrt64(k.g * pe * rr), rce = rcp64(ce);
    const double qne = dot3(u, n);
    const double mn = qne * rce;
    if (mn >= 1.0) {
        for (int t = 0; t < 5; ++t) Qf[t] = Qe[t];
        return;
    }
    if (mn <= -1.0) {
        const double z[3] = {0.0, 0.0, 0.0};
        cons_d(k.TR, z, k.rg, k, Qf);
        return;
    }
    const double qnf = fma(ce - k.cinf, k.g1, 0.5 * qne);
    const double cf = fma(0.25 * k.gm1, qne, 0.5 * (ce + k.cinf));
    // subsonic outflow, and |M_n| <= 1e-8 (q_n = 0 up to the rounding of weak
    // waves, which the paper's ranges leave open): entropy and tangential
    // velocity from inside; subsonic inflow: from the ambient (q_n,inf = 0,
    // gamma p_inf = 1)
    const bool out = mn >= -1e-8;
    const double dq = out ? qnf - qne : qnf;
    double uf[3];
    for (int c = 0; c < 3; ++c) uf[c] = out ? fma(dq, n[c], u[c]) : dq * n[c];
    const double x = out ? cf * rce : cf / k.cinf;
    const double rho = (out ? Qe[0] : k.TR) * exp(k.e2 * log(x));
    cons_d(rho, uf, rho * cf * cf * k.rg, k, Qf);
}

// Exit (Sec. "Exit Boundary Condition").
__device__ __forceinline__ void bc_exit(const BcD &k, const double Qe[5], const double n[3], double Qf[5])
{
    const double rr = rcp64(Qe[0]);
    const double u[3] = {Qe[1] * rr, Qe[2] * rr, Qe[3] * rr};
    const double pe = k.gm1 * fma(-0.5, dot3(Qe + 1, u), Qe[4]);
    if (dot3(u, n) * rsqrt64(k.g * pe * rr) >= 1.0) {
        for (int t = 0; t < 5; ++t) Qf[t] = Qe[t];
        return;
    }
    // p_f = p_inf = 1/gamma with the interior internal energy e_i = p/((gamma-1) rho)
    const double ei = pe * k.g1 * rr;
    const double rho = Qe[0] * rcp64(k.g * pe);
    Qf[0] = rho;
    Qf[1] = rho * u[0];
    Qf[2] = rho * u[1];
    Qf[3] = rho * u[2];
    Qf[4] = rho * fma(0.5, dot3(u, u), ei);
}

// FP32 storage: the boundary arithmetic runs in FP32 except the interior
// pressure and the temperature difference T_e - T_inf = c_e^2 - c_inf^2, which
// are formed from the stored values in pairs of floats (les_pair.cuh).  The
// far-field face state differs from the interior (or ambient) one by small
// amounts: the normal velocity by (c_e - c_inf)/(gamma - 1) - q_n,e/2, the
// density and pressure by factors (c_f/c)^m close to 1.  Each of these is
// computed as a difference that is accurate relative to itself (c_e - c_inf from
// T_e - T_inf; the factors as 1 + expm1(m log1p(x)) with x = c_f/c - 1 formed
// from small terms), so that FP32 rounding does not seed pressure or transverse
// momentum noise on the faces.  In FP64 those few operations and the conversions
// around them were 62 FP64 instructions per point and the pass's bound (55 % of
// the FP64 pipe).
__device__ __forceinline__ void cons_f(float rho, const float u[3], float p, const BcConst &k, float Q[5])
{
    Q[0] = rho;
    Q[1] = rho * u[0];
    Q[2] = rho * u[1];
    Q[3] = rho * u[2];
    Q[4] = fmaf(p, k.g1, 0.5f * rho * dot3(u, u));
}

// 1/rho, and the internal energy e - rho |u|^2 / 2 of the conserved Q, as pairs
__device__ __forceinline__ void energy_pair(const float Q[5], FloatPair &rr, FloatPair &ei)
{
    typedef Num<float> A;
    const float r0 = __fdividef(1.0f, Q[0]);
    rr = {r0, __fmul_rn(r0, __fmaf_rn(-Q[0], r0, 1.0f))};
    FloatPair m2 = A::mul(Q[1], FloatPair{Q[1], 0.0f});
    m2 = A::add(m2, A::mul(Q[2], FloatPair{Q[2], 0.0f}));
    m2 = A::add(m2, A::mul(Q[3], FloatPair{Q[3], 0.0f}));
    const FloatPair k = A::mulp(m2, rr);
    ei = A::add(FloatPair{Q[4], 0.0f}, FloatPair{-0.5f * k.h, -0.5f * k.l});
}

// Far field (Sec. "Far Field Boundary") for FP32 storage.  With
// R+- = q_n +- 2c/(gamma-1) (R- of the ambient at rest, R+ of the interior):
// q_n,f = (R+ + R-)/2 = q_n,e/2 + (c_e - c_inf)/(gamma-1) and
// c_f = (gamma-1)(R+ - R-)/4 = (gamma-1) q_n,e/4 + (c_e + c_inf)/2.  The
// isentropic density rho_e^gamma c_f^2 / (gamma p_e), raised to 1/(gamma-1),
// is rho_e (c_f/c_e)^(2/(gamma-1)) since gamma p_e = rho_e c_e^2, and the face
// pressure rho_f c_f^2 / gamma is p_e (c_f/c_e)^(2 gamma/(gamma-1)); on inflow
// the same with the ambient state (rho_inf c_inf^2 = gamma p_inf = 1).
__device__ __forceinline__ void bc_farfield_f32(const BcConst &k, const float Qe[5], const float n[3], float Qf[5])
{
    typedef Num<float> A;
    FloatPair rrp, ei;
    energy_pair(Qe, rrp, ei);
    const FloatPair Tp = A::mulp(A::mulp(ei, FloatPair{k.ggm1h, k.ggm1l}), rrp);
    const float dT = A::out(A::sub(Tp, FloatPair{k.Tinfh, k.Tinfl})); // T_e - T_inf
    const float p_e = A::out(A::mulp(ei, FloatPair{k.gm1h, k.gm1l}));
    const float rr = A::out(rrp);
    const float u[3] = {Qe[1] * rr, Qe[2] * rr, Qe[3] * rr};
    const float ce = sqrtf(A::out(Tp));
    const float dc = dT / (ce + k.cinf); // c_e - c_inf
    const float qne = dot3(u, n);
    const float mn = qne / ce;
    if (mn >= 1.0f) { // supersonic outflow: all from inside
        for (int t = 0; t < 5; ++t) Qf[t] = Qe[t];
        return;
    }
    if (mn <= -1.0f) { // supersonic inflow: the ambient at rest
        const float z[3] = {0.0f, 0.0f, 0.0f};
        cons_f(k.TR, z, k.rg, k, Qf);
        return;
    }
    const float qv = 0.25f * (k.g - 1.0f) * qne; // c_f = qv + (c_e + c_inf)/2
    // subsonic outflow, and |M_n| <= 1e-8 (as in the FP64 form): entropy and
    // tangential velocity from inside; subsonic inflow: from the ambient
    // (q_n,inf = 0)
    const bool out = mn >= -1e-8f;
    const float dq = fmaf(k.g1, dc, out ? -0.5f * qne : 0.5f * qne); // q_n,f - q_n,e; q_n,f
    float uf[3];
    for (int c = 0; c < 3; ++c) uf[c] = fmaf(dq, n[c], out ? u[c] : 0.0f);
    // log(c_f/c), c of the side the entropy comes from
    const float L = log1pf(fmaf(out ? -0.5f : 0.5f, dc, qv) / (out ? ce : k.cinf));
    const float r0 = out ? Qe[0] : k.TR, p0 = out ? p_e : k.rg;
    cons_f(fmaf(r0, expm1f(k.e2 * L), r0), uf, fmaf(p0, expm1f(k.e2g * L), p0), k, Qf);
}

// Exit (Sec. "Exit Boundary Condition") for FP32 storage.
__device__ __forceinline__ void bc_exit_f32(const BcConst &k, const float Qe[5], const float n[3], float Qf[5])
{
    typedef Num<float> A;
    FloatPair rrp, eip;
    energy_pair(Qe, rrp, eip);
    const float rr = A::out(rrp);
    const float u[3] = {Qe[1] * rr, Qe[2] * rr, Qe[3] * rr};
    const float q2 = dot3(u, u);
    const float p = A::out(A::mulp(eip, FloatPair{k.gm1h, k.gm1l}));
    if (dot3(u, n) * rsqrtf(k.g * p * rr) >= 1.0f) {
        for (int t = 0; t < 5; ++t) Qf[t] = Qe[t];
        return;
    }
    // p_f = p_inf = 1/gamma with the interior internal energy p/((gamma-1) rho)
    const float ei = p * k.g1 * rr;
    const float rho = Qe[0] / (k.g * p);
    Qf[0] = rho;
    Qf[1] = rho * u[0];
    Qf[2] = rho * u[1];
    Qf[3] = rho * u[2];
    Qf[4] = rho * fmaf(0.5f, q2, ei);
}

// SplitMix64: output number n of the generator seeded with `seed`.
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long seed,
                                                         unsigned long long n)
{
    unsigned long long z = seed + (n + 1ull) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Inflow noise of velocity component c at face point (jj, kk) for the step
// that `level` counts (level > 0): A U_j (2h - 1), h in [0, 1) the top 53 bits
// of SplitMix64 output number ((level - 1) nk + kk) nj + jj) * 3 + c.
template <typename real>
__device__ __forceinline__ double inflow_noise(const JetDev<real> &J, long long level, int kk, int jj, int c)
{
    const unsigned long long ctr =
        ((((unsigned long long)(level - 1) * (unsigned long long)J.n[2] + (unsigned long long)kk) *
              (unsigned long long)J.n[1] +
          (unsigned long long)jj) * 3ull) + (unsigned long long)c;
    const double h = (double)(splitmix64(J.seed, ctr) >> 11) * (1.0 / 9007199254740992.0);
    return J.noise_amp * J.mach * fma(2.0, h, -1.0);
}

// The jet entrance (Sec. "Entrance Boundary") at face point (jj, kk) with
// profile value ut >= 0.01: primitive state from the profile, the interior
// state Qe (subsonic entrance) and the noise of the level.
template <typename real, typename T>
__device__ __forceinline__ void inflow_state(const JetDev<real> &J, T ut, T g, T g1, T rg, T TR, const T Qe[5],
                                             long long level, int kk, int jj, T &rho, T u[3], T &p)
{
    const T M = (T)J.mach;
    if (M < T(1)) {
        // subsonic entrance: u fixed (profile and the u noise of the level), v
        // and w from the interior point, T from the jet's total temperature
        // 1 + (gamma-1) M^2/2 with the face velocity in units of a_j, p =
        // T^(gamma/(gamma-1))/gamma
        u[0] = M * ut;
        if (level > 0) u[0] = sum_rn(u[0], (T)inflow_noise(J, level, kk, jj, 0));
        const T rre = T(1) / Qe[0];
        u[1] = Qe[2] * rre;
        u[2] = Qe[3] * rre;
        const T hg = T(0.5) * (g - T(1)), Ttot = fma(hg * M, M, T(1));
        const T Ts = Ttot / fma(hg, dot3(u, u), T(1));
        p = pow(Ts, g * g1) * rg;
        rho = g * p / Ts;
    } else {
        const T Tt = fma(T(0.5) * (g - T(1)) * M * M * ut, T(1) - ut, fma(T(1) / TR, T(1) - ut, ut));
        p = rg;
        rho = T(1) / Tt; // gamma p / T
        u[0] = M * ut;
        u[1] = u[2] = T(0);
        if (level > 0)
            for (int c = 0; c < 3; ++c) u[c] = sum_rn(u[c], (T)inflow_noise(J, level, kk, jj, c));
    }
}

// Boundary state Qf at face point q of `axis` and `side`, metric row n, from the
// unscaled state Qe of its inner neighbour.
template <typename real, typename T>
__device__ __forceinline__ void face_state(const JetDev<real> &J, int axis, int side, T n[3], const int q[3],
                                           long long level, const T Qe[5], T Qf[5])
{
    const int type = J.bc[2 * axis + side];
    // unit outward normal from the face point's metric row n
    T nn = T(0);
    const T sg = side ? T(1) : T(-1);
    for (int c = 0; c < 3; ++c) {
        n[c] *= sg;
        nn = fma(n[c], n[c], nn);
    }
    const bool inflow = type == LES_BC_INFLOW_JET;
    const T ut = inflow ? (T)J.inflow_ut[(long long)q[2] * J.n[1] + q[1]] : T(0);
    if constexpr (sizeof(T) == sizeof(float)) {
        const BcConst &k = J.bcf;
        const float rn = rsqrtf(nn);
        for (int c = 0; c < 3; ++c) n[c] *= rn;
        // the branch on the profile takes its FP64 value
        const bool far = type == LES_BC_FARFIELD ||
                         (inflow && J.inflow_ut[(long long)q[2] * J.n[1] + q[1]] < 0.01);
        if (far) {
            bc_farfield_f32(k, Qe, n, Qf);
        } else if (!inflow) {
            bc_exit_f32(k, Qe, n, Qf);
        } else {
            float rho, u[3], p;
            inflow_state<real, float>(J, ut, k.g, k.g1, k.rg, k.TR, Qe, level, q[2], q[1], rho, u, p);
            cons_f(rho, u, p, k, Qf);
        }
    } else {
        const BcD k{J.gamma, J.gm1, J.bc_g1, J.bc_rg, 2.0 * J.bc_g1, J.TR, J.bc_cinf};
        const double rn = rsqrt64(nn);
        for (int c = 0; c < 3; ++c) n[c] *= rn;
        if (type == LES_BC_FARFIELD || (inflow && ut < 0.01)) {
            bc_farfield(k, Qe, n, Qf);
        } else if (!inflow) {
            bc_exit(k, Qe, n, Qf);
        } else {
            double rho, u[3], p;
            inflow_state<real, double>(J, ut, k.g, k.g1, k.rg, k.TR, Qe, level, q[2], q[1], rho, u, p);
            cons_d(rho, u, p, k, Qf);
        }
    }
}

// All boundary faces of a time level in one pass.  The conditions apply in
// the order faces y, z, x, a later face reading what an earlier one wrote on a
// shared edge; here the thread of a face point (an edge belongs to the last of
// its faces in that order) applies the conditions of every face the point lies
// on in turn, starting from the interior point inside all of them, so that no
// thread reads what another one writes.  What it replaces: three launches per
// stage whose 256-thread blocks left a small face on a dozen SMs, bound by the
// FP64 issue of those SMs; blocks of 64 spread every face over the chip.
// Measured per stage: FP64 48x32x32 95 -> 21 us (a traced launch costs 6 of
// them), 384x256x144 242 -> 131 us; FP32 192x128x72 37 -> 12 us.
constexpr int BC_BLOCK = 64;
// (32-bit face indices: a face has fewer points than a jet, and those fit.)
// Thread t of a jet's boundary pass: false if it has no point; else F, the
// padded index of its face point, and Q, the stored boundary state there, from
// the interior points of buffer Qs.
template <typename real>
__device__ __forceinline__ bool bc_point(const JetDev<real> &J, int t, long long level, const real *Qs,
                                         long long &F, real Q[5])
{
    using T = real;
    // the face the thread stands for: x, z, y faces in turn, both sides of an
    // axis, the lower tangential axis fastest across threads
    int axis = -1, q[3];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const int a = s == 0 ? 0 : 3 - s;
        if (J.per[a] || axis >= 0) continue;
        const int b = a == 0 ? 1 : 0, d = a == 2 ? 1 : 2;
        const int nface = J.n[b] * J.n[d];
        if (t < 2 * nface) {
            axis = a;
            const int side = t >= nface;
            const int r = t - side * nface;
            const int id = r / J.n[b];
            q[a] = side ? J.n[a] - 1 : 0;
            q[b] = r - id * J.n[b];
            q[d] = id;
        } else {
            t -= 2 * nface;
        }
    }
    if (axis < 0) return false;
    // faces of the point; the centerline face is not one of them (its axis
    // state is in place)
    bool on[3];
    int cur[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const bool lo = q[a] == 0, hi = q[a] == J.n[a] - 1;
        on[a] = !J.per[a] && ((lo && J.bc[2 * a] != LES_BC_CENTERLINE) || hi);
        cur[a] = on[a] ? (lo ? 1 : q[a] - 1) : q[a];
    }
    if (!on[axis] || (axis != 0 && on[0]) || (axis == 1 && on[2])) return false;
    const long long fs = J.fs;
    // In FP32 everything the chain reads is fetched before it, the metric rows of
    // the faces the point lies on too: one memory latency instead of one per face
    // (48x32x32 9.5 -> 8.3 us, 192x128x72 13.8 -> 11.9 us).  In FP64 the rows are
    // read face by face: nine more doubles held cost warps
    // (384x256x144 131 -> 137 us).
    constexpr bool AHEAD = sizeof(real) == sizeof(float);
    T nr[3][3];
    if (AHEAD) {
        int at[3] = {cur[0], cur[1], cur[2]};
#pragma unroll
        for (int s = 1; s < 4; ++s) {
            const int a = s == 3 ? 0 : s;
            if (!on[a]) continue;
            at[a] = q[a];
            const long long o = lidx(J, at[0], at[1], at[2]);
#pragma unroll
            for (int c = 0; c < 3; ++c) nr[a][c] = J.met[(3 * a + c) * fs + o];
        }
    }
    {
        const long long E = lidx(J, cur[0], cur[1], cur[2]);
        const T rs = sizeof(real) == sizeof(float) ? T(1) : (T)J.met[MET_J * fs + E];
        for (int f = 0; f < 5; ++f) Q[f] = Qs[f * fs + E] * rs;
    }
#pragma unroll 1
    for (int s = 1; s < 4; ++s) { // y, z, x
        const int a = s == 3 ? 0 : s;
        if (!(s == 1 ? on[1] : (s == 2 ? on[2] : on[0]))) continue;
        const int qa = s == 1 ? q[1] : (s == 2 ? q[2] : q[0]);
        T n[3], Qf[5];
        if (AHEAD) {
            for (int c = 0; c < 3; ++c) n[c] = s == 1 ? nr[1][c] : (s == 2 ? nr[2][c] : nr[0][c]);
        } else {
            if (s == 1) cur[1] = qa;
            else if (s == 2) cur[2] = qa;
            else cur[0] = qa;
            const long long o = lidx(J, cur[0], cur[1], cur[2]);
            for (int c = 0; c < 3; ++c) n[c] = J.met[(3 * a + c) * fs + o];
        }
        face_state<real, T>(J, a, qa != 0, n, q, level, Q, Qf);
        for (int f = 0; f < 5; ++f) Q[f] = Qf[f];
    }
    F = lidx(J, q[0], q[1], q[2]);
    const T sc = (T)stored_scale<real>(J.jinv64[F]);
    for (int f = 0; f < 5; ++f) Q[f] = sc * Q[f];
    return true;
}

} // namespace les
