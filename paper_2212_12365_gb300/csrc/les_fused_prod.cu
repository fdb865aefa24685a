// Fused single-pass Runge-Kutta stage in FP32 on a Cartesian-product grid x(i),
// y(j), z(k): what les_fused.cu does for general metrics, with the diagonal
// metric's zeros left out and the work cut anew for it.
//
// What bounded the previous form of this kernel (the general kernel with the
// metric made diagonal): 858 thread instructions per point at 8 warps per SM,
// issue 40 % busy, of which 265 were paired FP32; the rest was table traffic
// for quantities a diagonal metric does not use, index arithmetic, and moves
// that shifted row pairs by one row.  This kernel drops those tables and moves
// and runs 12 warps per SM (TY = 24).  Measured, 384x256x144, ms per stage:
// general metrics 0.951, diagonal before 0.700, this kernel 0.537; general metrics
// -> this kernel: 64 jets 11.55 -> 6.76 ms a step, 192x128x72 0.142 -> 0.090 ms a
// stage.  What bounds it: latency with 3 warps per scheduler (384x192x96, TY = 24:
// issue 42 % busy, shared-memory wavefronts 56 % and FMA pipe 33 % of peak; stalls
// per issue on shared-memory and MUFU results 1.6, on fixed-latency chains 1.4, on
// the memory queue 0.8, at barriers 0.5).
//
// Fluxes.  As in les_stage_prod.cu the interface flux is divided by the face
// area S_a and doubled, G_a = 2 H_a / S_a = F_L + F_R - hb (lb_L + lb_R) [eps2
// dW - eps4 d3W] - viscous, with F the Cartesian point flux, hb the mean spacing
// along a; the stored state is unscaled, so the stage is
//   Q(l) = Q(0) - alpha dt sum_a (1/(2 h_a)) (G_a(+1/2) - G_a(-1/2)).
// The viscous part needs du_i/dx_a and du_a/dx_i per flux direction a and the
// sum of the other two diagonal derivatives; temperature derivatives only as the
// interface difference.  Derivatives are kept as d/h with d = f(+1) - f(-1)
// (twice the derivative); the transport coefficients carry the 1/4 that the sum
// of two such values wants.  Pressure is stored less the ambient pressure (a
// constant pressure has no flux divergence; leaving it in adds FP32 rounding
// of O(1) terms to small momentum residuals).
//
// Split row pairs.  A CTA of 32 x TR threads (TR = TY/2) owns a tile of 32
// columns x TY rows (region R1) and updates its 30 x (TY-2) inner points; thread
// (tx, tr) owns rows tr and tr + TR of its column, the two lanes of its paired
// FP32 arithmetic.  The neighbours of such a pair in y are again whole pairs,
// (tr +- 1, tr + TR +- 1), so no value moves between lanes; the pairs that
// straddle the middle of the tile are stored once more (pair rows -2, -1 and TR,
// TR + 1 of the point ring; pair row TR of the tables).
//
// Per loaded plane kL, between barriers A and B:
//   primitives(kL) | A | gradients, closures(kL-1); zeta flux (kL-2 | kL-1);
//   update(kL-2); tables(kL-1) | B | xi and eta fluxes of plane kL-1
// The zeta flux uses the thread's own values of two planes, so its tables never
// go to shared memory; the eta flux of a thread is read by the row above after
// the next barrier A, and the flux differences of a plane are carried in
// registers until its update one plane later.  Point data: a ring of four
// planes over R2 = R1 plus one column each side and two rows above and below;
// cells outside a non-periodic axis hold the mirror image (W(-1) = W(1)), the
// paper's boundary fourth difference.
#include <algorithm>
#include <cmath>

#include "les_fused.cuh"

namespace les {

namespace {

// rows of the staging box and spacing rows of a tile: TY + 4
template <int TY> struct PGeo {
    static constexpr int TR = TY / 2;
    static constexpr int NT = FX * TR;
    static constexpr int C2 = FX + 2;   // R2 columns -1 .. FX
    static constexpr int P2 = TR + 4;   // R2 pair rows -2 .. TR + 1
    static constexpr int N2 = C2 * P2;
    static constexpr int NC = (N2 + NT - 1) / NT; // cells a thread loads
    static constexpr int N1 = FX * (TR + 1);      // table cells, pair rows 0 .. TR
    static constexpr int BR = tma_box_rows(TY);
    static constexpr size_t O_A = 0;                      // [4][N2] float4 (u, v)
    static constexpr size_t O_B = O_A + 16ull * 4 * N2;   // (w, p - p_inf)
    static constexpr size_t O_C = O_B + 16ull * 4 * N2;   // (rho, rho H)
    static constexpr size_t O_T = O_C + 16ull * 4 * N2;   // float2 T
    static constexpr size_t O_TB = O_T + 8ull * 4 * N2;   // [6][N1] float4, see TabXY
    static constexpr size_t O_HG = O_TB + 16ull * 6 * N1; // [5][NT] float2: eta fluxes
    static constexpr size_t O_QZ = O_HG + 8ull * 5 * NT;  // [10][NT] float: Q(0) of the updated points
    static constexpr size_t O_HX = O_QZ + 4ull * 10 * NT; // [C2] float4 (h, 1/h, h^(2/3), 0)
    static constexpr size_t O_HY = O_HX + 16ull * C2;     // [BR]
    static constexpr size_t O_HZ = O_HY + 16ull * BR;     // [4], slot k & 3
    static constexpr size_t O_QG = (O_HZ + 64 + 127) / 128 * 128; // staging box
    static constexpr unsigned BOX_BYTES = 4u * 5 * BR * TMA_BOX_X;
    static constexpr size_t O_MBAR = O_QG + BOX_BYTES;
    static constexpr size_t O_FPS = O_MBAR + 8;
    static constexpr size_t BYTES = O_FPS + 64;
    static_assert(BOX_BYTES % 16 == 0 && BYTES <= 227 * 1024, "shared memory of one CTA");
};

template <int TY> struct PSm {
    float4 *A, *B, *C;
    float2 *T;
    float4 *TB;
    float2 *HG;
    float *QZ;
    float4 *HX, *HY, *HZ;
    float *QG;
    unsigned long long *MBAR;
    float *FPS;
    __device__ __forceinline__ explicit PSm(unsigned char *b)
        : A((float4 *)(b + PGeo<TY>::O_A)), B((float4 *)(b + PGeo<TY>::O_B)), C((float4 *)(b + PGeo<TY>::O_C)),
          T((float2 *)(b + PGeo<TY>::O_T)), TB((float4 *)(b + PGeo<TY>::O_TB)), HG((float2 *)(b + PGeo<TY>::O_HG)),
          QZ((float *)(b + PGeo<TY>::O_QZ)), HX((float4 *)(b + PGeo<TY>::O_HX)), HY((float4 *)(b + PGeo<TY>::O_HY)),
          HZ((float4 *)(b + PGeo<TY>::O_HZ)), QG((float *)(b + PGeo<TY>::O_QG)),
          MBAR((unsigned long long *)(b + PGeo<TY>::O_MBAR)), FPS((float *)(b + PGeo<TY>::O_FPS))
    {
    }
};

// One point pair: velocity, p - p_inf, density, rho H, T, and rho u.
struct PP {
    float2 u[3], p, rho, rH, T, m[3];
};
// Transport data of a pair along one axis: coefficients / 4, k2 sensor,
// lambda-bar, the two cross derivatives du_a/dx_i (i ascending) and 2/3 of the
// other two diagonal derivatives' sum.
struct Tr {
    float2 mue, kap, nu, lb, c[2], s;
};

__device__ __forceinline__ void wvec(const PP &q, float2 W[5])
{
    W[0] = q.rho;
    W[1] = q.m[0];
    W[2] = q.m[1];
    W[3] = q.m[2];
    W[4] = q.rH;
}

// G_a of the interfaces between the pairs L and their +a neighbours R.
template <int a>
__device__ __forceinline__ void flux(float k4, const PP &L, const PP &R, const float2 Wm[5], const float2 Wp[5],
                                     const Tr &tL, const Tr &tR, float2 hb, float2 rhb4, float2 c43, float2 G[5])
{
    // Turkel-Vatsa coefficients
    const float2 eps2 = max2(tL.nu, tR.nu);
    const float2 eps4 = max2(bc(0.0f), sub2(bc(k4), eps2));
    const float2 sc = mul2(hb, add2(tL.lb, tR.lb));
    const float2 se4 = mul2(sc, eps4);
    const float2 c2 = mul2(sc, fma2(bc(3.0f), eps4, eps2));
    float2 WL[5], WR[5];
    wvec(L, WL);
    wvec(R, WR);
    G[0] = add2(L.m[a], R.m[a]);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        G[1 + i] = i == a ? fma2(L.m[a], L.u[i], add2(L.p, R.p)) : mul2(L.m[a], L.u[i]);
        G[1 + i] = fma2(R.m[a], R.u[i], G[1 + i]);
    }
    G[4] = fma2(R.rH, R.u[a], mul2(L.rH, L.u[a]));
#pragma unroll
    for (int f = 0; f < 5; ++f) G[f] = fma2(c2, sub2(WL[f], WR[f]), fma2(se4, sub2(Wp[f], Wm[f]), G[f]));
    const float2 mu = add2(tL.mue, tR.mue);
    float2 su = bc(0.0f);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float2 du = sub2(R.u[i], L.u[i]);
        float2 g;
        if (i == a) {
            g = sub2(mul2(c43, du), add2(tL.s, tR.s));
        } else {
            const int c = i > a ? i - 1 : i;
            g = fma2(rhb4, du, add2(tL.c[c], tR.c[c]));
        }
        const float2 sv = mul2(mu, g);
        G[1 + i] = sub2(G[1 + i], sv);
        const float2 us = add2(L.u[i], R.u[i]);
        su = i == 0 ? mul2(us, sv) : fma2(us, sv, su);
    }
    const float2 q = mul2(rhb4, sub2(R.T, L.T));
    G[4] = fma2(bc(-0.5f), su, G[4]);
    G[4] = sub2(G[4], mul2(add2(tL.kap, tR.kap), q));
}

} // namespace

// Index checks of a LES_BOUNDS_CHECK build (see les_fused.cu)
#define CK_G(site, x, n) LES_BOUNDS(J.oob, (site), (x), (n))
#define CK_RING(x) ((int)LES_BOUNDS(J.oob, 5, (x), 4 * N2))
#define CK_TAB(x, n) ((int)LES_BOUNDS(J.oob, 6, (x), (n)))
#define CK_SH(x) ((int)LES_BOUNDS(J.oob, 7, (x), 5 * NT))

template <int TY, bool ONE>
__global__ void __launch_bounds__(FX *TY / 2, 1)
    k_fused_prod(const JetDev<float> *__restrict__ jets, const FusedJet *__restrict__ fj, int njets, int total_items,
                 int total_tiles, int src, int dst, int stage, const double *__restrict__ dt, int rhs_only,
                 int balanced, int wait_limit, const __grid_constant__ JetDev<float> j1,
                 const __grid_constant__ FusedJet f1)
{
    using G_ = PGeo<TY>;
    constexpr int TR = G_::TR, NT = G_::NT, C2 = G_::C2, N2 = G_::N2, N1 = G_::N1, BR = G_::BR, NC = G_::NC;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const PSm<TY> S(smem_raw);
    const int tx = threadIdx.x, tr = threadIdx.y;
    const int tid = tr * FX + tx;
    const int c2 = (tr + 2) * C2 + (tx + 1); // own R2 pair cell (within a plane)

    // staging state, as in les_fused.cu: a wait that gives up is recorded (site
    // 8) and the CTA reads the state from global memory from then on
    const bool tma_smem_ok = (smem_u32(S.QG) & 127u) == 0;
    unsigned tpar = 0;
    bool tma_off = false, pend = false;
    if (tid == 0) mbar_init(S.MBAR);
    __syncthreads();

    Cursor<ONE> cur(fj, f1, njets, total_items, total_tiles, balanced);
    int key, jet;
    while (cur.next(key, jet)) {
        const JetDev<float> &J = jet_entry<ONE>(j1, jets, jet);
        const FusedJet &F = jet_entry<ONE>(f1, fj, jet);
        if constexpr (!ONE) {
            constexpr int NFP = sizeof(FusedParams) / 4;
            if (tid >= NT - NFP) S.FPS[tid - (NT - NFP)] = reinterpret_cast<const float *>(&F.fp)[tid - (NT - NFP)];
        }
        const FusedParams &FP = jet_params<ONE>(F.fp, S.FPS);
        const int ni = J.n[0], nj = J.n[1], nk = J.n[2];
        const int pi = J.per[0], pj = J.per[1], pk = J.per[2];
        const int ilo = pi ? 0 : 1, ihi = pi ? ni : ni - 1;
        const int jlo = pj ? 0 : 1, jhi = pj ? nj : nj - 1;
        const int klo = pk ? 0 : 1, khi = pk ? nk : nk - 1;
        int bx, by, k0, k1;
        cur.take(key, F, klo, khi, bx, by, k0, k1);
        // grid column / row of the tile's first R1 cell
        const int ib = ilo + bx * (FX - 2) - 1, jb = jlo + by * (TY - 2) - 1;
        const int fs = (int)J.fs; // 32-bit offsets: creation limits an FP32 jet
        const int plane = nj * J.pitch;
        const float *__restrict__ Qs = J.q[src];
        const float adt = rhs_only ? 0.0f : 0.5f * (c_alpha_f[stage] * (float)dt[jet]);

        // ---- per-item setup ----
        const int rA = tr, rB = tr + TR;
        const int gi = map_idx(ib + tx, ni, pi);
        const int gjA = map_idx(jb + rA, nj, pj), gjB = map_idx(jb + rB, nj, pj);
        // one-sided in-plane stencils (+-1) at a non-periodic end
        const int ti = (!pi && ib + tx == 0) ? 1 : ((!pi && ib + tx == ni - 1) ? -1 : 0);
        const int tjA = (!pj && jb + rA == 0) ? 1 : ((!pj && jb + rA == nj - 1) ? -1 : 0);
        const int tjB = (!pj && jb + rB == 0) ? 1 : ((!pj && jb + rB == nj - 1) ? -1 : 0);
        // outputs: columns 1..30, rows 1..TY-2 of R1 inside the output range
        const bool col_out = tx >= 1 && tx <= FX - 2 && (ib + tx) < ihi;
        const bool outA = col_out && rA >= 1 && (jb + rA) < jhi;
        const bool outB = col_out && rB <= TY - 2 && (jb + rB) < jhi;
        const int ocolA = gjA * J.pitch + gi, ocolB = gjB * J.pitch + gi;
        const CUtensorMap *tmap = nullptr;
        int tx0 = 0;
        if (F.tmap && tma_smem_ok && !pi && !pj && !tma_off) {
            tmap = F.tmap + (TY == 8 ? 0 : (TY == 16 ? 3 : 6)) + src;
            tx0 = (ib - 1) & ~3;
        }
        // the R2 pair cells this thread loads and, per row, the offset of the
        // source point in the staging box and in a plane
        int bo[NC][2], go[NC][2];
#pragma unroll
        for (int t = 0; t < NC; ++t) {
            const int c = min(tid + t * NT, N2 - 1);
            const int cc = c % C2, pr = c / C2;
            const int gc = map_idx(ib - 1 + cc, ni, pi);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int gr = map_idx(jb + pr - 2 + h * TR, nj, pj);
                go[t][h] = gr * J.pitch + gc;
                const int rr = min(max(gr - (jb - 2), 0), BR - 1), cl = min(max(gc - tx0, 0), TMA_BOX_X - 1);
                bo[t][h] = rr * TMA_BOX_X + cl;
            }
        }
        // 1-D spacings of the tile's columns and rows (the previous item's last
        // reads precede its last barrier)
        for (int t = tid; t < C2 + BR; t += NT) {
            if (t < C2) S.HX[t] = F.h1[0][map_idx(ib - 1 + t, ni, pi)];
            else S.HY[t - C2] = F.h1[1][map_idx(jb - 2 + (t - C2), nj, pj)];
        }
        __syncthreads(); // spacings written; shared memory of the previous item is free
        // spacing factors of the own points along xi (both rows alike) and eta
        const float4 hx0 = S.HX[tx + 1], hx1 = S.HX[tx + 2];
        const float4 hyA0 = S.HY[rA + 2], hyA1 = S.HY[rA + 3], hyB0 = S.HY[rB + 2], hyB1 = S.HY[rB + 3];
        const float2 rhx = bc(hx0.y), rhy = f2(hyA0.y, hyB0.y);
        const float hbx_ = __fmul_rn(0.5f, __fadd_rn(hx0.x, hx1.x)), rhbx_ = __fmul_rn(4.0f, rcpa(hbx_));
        const float2 hbx = bc(hbx_), rhbx = bc(rhbx_), c43x = bc(__fmul_rn(4.0f / 3.0f, rhbx_));
        const float2 hby = mul2(bc(0.5f), add2(f2(hyA0.x, hyB0.x), f2(hyA1.x, hyB1.x)));
        const float2 rhby = mul2(bc(4.0f), rcp2(hby)), c43y = mul2(bc(4.0f / 3.0f), rhby);
        // (Cs Delta)^2 / 4 less its k factor (the 1/4 of the coefficients)
        const float2 csxy = mul2(bc(__fmul_rn(__fmul_rn(0.25f, FP.cs2), hx0.z)), f2(hyA0.z, hyB0.z));

        auto stage_box = [&](int kq) {
            if (tid != 0) return;
            tma_box_load(S.QG, tmap, tx0, jb - 2, map_idx(kq, nk, pk), S.MBAR, G_::BOX_BYTES);
        };
        const int kfirst = k0 - 2, klast = k1 + 1;
        int gkU = map_idx(kfirst - 2, nk, pk), gkG = map_idx(kfirst - 1, nk, pk), gkL = map_idx(kfirst, nk, pk);
        if (tmap) stage_box(kfirst);

        // ---- shared-memory accessors ----
        struct V4 {
            float2 u[3], p;
        };
        auto ldv = [&](int cell, V4 &v) {
            const float4 a = S.A[cell], b = S.B[cell];
            v.u[0] = lo2(a);
            v.u[1] = hi2(a);
            v.u[2] = lo2(b);
            v.p = hi2(b);
        };
        auto ldp = [&](int cell, PP &q) {
            const float4 a = S.A[cell], b = S.B[cell], c = S.C[cell];
            q.u[0] = lo2(a);
            q.u[1] = hi2(a);
            q.u[2] = lo2(b);
            q.p = hi2(b);
            q.rho = lo2(c);
            q.rH = hi2(c);
            q.T = S.T[cell];
#pragma unroll
            for (int i = 0; i < 3; ++i) q.m[i] = mul2(q.rho, q.u[i]);
        };
        auto ldw = [&](int cell, float2 W[5]) {
            const float4 a = S.A[cell], b = S.B[cell], c = S.C[cell];
            W[0] = lo2(c);
            W[1] = mul2(W[0], lo2(a));
            W[2] = mul2(W[0], hi2(a));
            W[3] = mul2(W[0], lo2(b));
            W[4] = hi2(c);
        };
        const float pinf4 = 4.0f * FP.pinf;
        auto sensor = [&](float2 pm, float2 pc, float2 pp) { // of p - p_inf
            const float2 s = add2(pm, pp);
            const float2 num = fma2(pc, bc(-2.0f), s), den = fma2(pc, bc(2.0f), add2(s, bc(pinf4)));
            const float2 r = rcp2(den);
            return mul2(bc(FP.k2), f2(__fmul_rn(fabsf(num.x), r.x), __fmul_rn(fabsf(num.y), r.y)));
        };
        // one-sided at an end: cells c (own), c1, c2 one and two inside, t = +-1
        auto one_sided = [&](const V4 &o, int q1, int q2, int t, float2 d[3], float2 &nu) {
            V4 a, b;
            ldv(q1, a);
            ldv(q2, b);
            const float2 w0 = bc(-3.0f * t), w1 = bc(4.0f * t), w2 = bc(-1.0f * t);
#pragma unroll
            for (int i = 0; i < 3; ++i) d[i] = fma2(w2, b.u[i], fma2(w1, a.u[i], mul2(w0, o.u[i])));
            nu = sensor(o.p, a.p, b.p);
        };

        // carried from plane to plane: the xi flux difference of plane kU over h,
        // the zeta flux below it, and its zeta transport data.  (Every difference
        // is taken before the division by h: the fluxes are much larger than
        // their differences.)
        float2 acc[5], gzm[5];
        Tr tz;
#pragma unroll
        for (int f = 0; f < 5; ++f) acc[f] = gzm[f] = bc(0.0f);
        tz.mue = tz.kap = tz.nu = tz.lb = tz.s = tz.c[0] = tz.c[1] = bc(0.0f);

        for (int kL = kfirst; kL <= klast; ++kL) {
            const int kG = kL - 1, kU = kL - 2;
            // plane bases of the ring
            const int bL = (kL & 3) * N2, bG = (kG & 3) * N2, bU = (kU & 3) * N2, bM = ((kU - 1) & 3) * N2;
            // the mirror plane beyond the last plane of a non-periodic k axis is
            // not loaded (its slot holds a plane the last gradients need)
            const bool ghost_hi = !pk && kL == nk;
            // ---- load + primitives of plane kL on R2 ----
            if (!ghost_hi) {
                bool from_box = false;
                if (tmap) {
                    if (mbar_wait(S.MBAR, tpar, wait_limit)) {
                        from_box = true;
                        tpar ^= 1u;
                    } else {
                        if (J.oob) atomicCAS(J.oob, 0ull, 8ull << 48);
                        tma_off = true;
                        pend = true;
                    }
                }
                const int pofs = gkL * plane;
#pragma unroll
                for (int t = 0; t < NC; ++t) {
                    if (tid + t * NT >= N2) continue;
                    float q[2][5];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (from_box) {
#pragma unroll
                            for (int f = 0; f < 5; ++f)
                                q[h][f] = S.QG[CK_TAB(f * (BR * TMA_BOX_X) + bo[t][h], 5 * BR * TMA_BOX_X)];
                        } else {
                            const int o = CK_G(2, pofs + go[t][h], J.npts_pad);
#pragma unroll
                            for (int f = 0; f < 5; ++f) q[h][f] = Qs[f * fs + o];
                        }
                    }
                    const float2 rho = f2(q[0][0], q[1][0]), e = f2(q[0][4], q[1][4]);
                    const float2 m[3] = {f2(q[0][1], q[1][1]), f2(q[0][2], q[1][2]), f2(q[0][3], q[1][3])};
                    const float2 rr = rcp2(rho);
                    const float2 u = mul2(m[0], rr), v = mul2(m[1], rr), w = mul2(m[2], rr);
                    const float2 ke2 = fma2(m[2], w, fma2(m[1], v, mul2(m[0], u)));
                    // p rounded before p_inf is taken off, as in the general form: the
                    // far-field branches of weak waves (normal velocities at rounding
                    // level) then fall as there
                    const float2 p = mul2(bc(FP.gm1), fma2(ke2, bc(-0.5f), e));
                    const int cell = CK_RING(bL + tid + t * NT);
                    S.A[cell] = cat4(u, v);
                    S.B[cell] = cat4(w, sub2(p, bc(FP.pinf)));
                    S.C[cell] = cat4(rho, add2(e, p));
                    S.T[cell] = mul2(mul2(bc(FP.gam), p), rr);
                }
            }
            // thread 0's spacing copy of plane kL - 1 (two iterations ago) has landed
            if (tid == 0) cp_async_wait_prev();
            tma_off = __syncthreads_or(tma_off) != 0; // barrier A
            if (tma_off) tmap = nullptr;
            if (tmap && kL < klast && !(!pk && kL + 1 == nk)) stage_box(kL + 1);
            // the spacings of plane kL + 1 (slot of plane kL - 3), and Q(0) of
            // this iteration's updated points: one copy group per iteration
            if (tid == 0) cp_async16(S.HZ + ((kL + 1) & 3), F.h1[2] + map_idx(kL + 1, nk, pk));
            const bool do_upd = kU >= k0; // (kU <= k1 - 1 always)
            if (!rhs_only && do_upd) {
                const int pU = gkU * plane;
                const float *Q0 = J.q[0];
                if (outA) {
                    const int o = CK_G(4, pU + ocolA, J.npts_pad);
#pragma unroll
                    for (int f = 0; f < 5; ++f) cp_async4(S.QZ + (2 * f) * NT + tid, Q0 + f * fs + o);
                }
                if (outB) {
                    const int o = CK_G(4, pU + ocolB, J.npts_pad);
#pragma unroll
                    for (int f = 0; f < 5; ++f) cp_async4(S.QZ + (2 * f + 1) * NT + tid, Q0 + f * fs + o);
                }
            }
            cp_async_commit();

            if (kG >= k0 - 1 && !(!pk && kG == 0)) {
                // ---- gradients and closures of plane kG; those of the first plane of
                // a non-periodic k axis (which need planes 0..2) one plane late ----
                Tr X, Y, Z; // of the own pair along the three axes
                PP O;
#pragma unroll 1
                for (int g = (!pk && kG == 1 && k0 == 1) ? 0 : kG;; ++g) {
                    const int b0 = (g & 3) * N2 + c2, bm = ((g - 1) & 3) * N2 + c2, bp = ((g + 1) & 3) * N2 + c2;
                    ldp(CK_RING(b0), O);
                    V4 o;
                    o.u[0] = O.u[0];
                    o.u[1] = O.u[1];
                    o.u[2] = O.u[2];
                    o.p = O.p;
                    const float4 hz = S.HZ[g & 3];
                    float2 d[3][3], nu[3]; // d[a][i]: f(+1) - f(-1) of u_i along a
                    auto central = [&](int cm, int cp, float2 dd[3], float2 &nn) {
                        V4 a, b;
                        ldv(CK_RING(cm), a);
                        ldv(CK_RING(cp), b);
#pragma unroll
                        for (int i = 0; i < 3; ++i) dd[i] = sub2(b.u[i], a.u[i]);
                        nn = sensor(a.p, o.p, b.p);
                    };
                    central(b0 - 1, b0 + 1, d[0], nu[0]);
                    if (ti != 0) one_sided(o, CK_RING(b0 + ti), CK_RING(b0 + 2 * ti), ti, d[0], nu[0]);
                    central(b0 - C2, b0 + C2, d[1], nu[1]);
                    if (tjA != 0 || tjB != 0) {
                        float2 e[3], n;
                        if (tjA != 0) {
                            one_sided(o, CK_RING(b0 + tjA * C2), CK_RING(b0 + 2 * tjA * C2), tjA, e, n);
#pragma unroll
                            for (int i = 0; i < 3; ++i) d[1][i].x = e[i].x;
                            nu[1].x = n.x;
                        }
                        if (tjB != 0) {
                            one_sided(o, CK_RING(b0 + tjB * C2), CK_RING(b0 + 2 * tjB * C2), tjB, e, n);
#pragma unroll
                            for (int i = 0; i < 3; ++i) d[1][i].y = e[i].y;
                            nu[1].y = n.y;
                        }
                    }
                    const bool klo_end = !pk && g == 0, khi_end = !pk && g == nk - 1;
                    if (klo_end || khi_end) {
                        const int t = klo_end ? 1 : -1;
                        one_sided(o, CK_RING(((g + t) & 3) * N2 + c2), CK_RING(((g + 2 * t) & 3) * N2 + c2), t, d[2], nu[2]);
                    } else {
                        central(bm, bp, d[2], nu[2]);
                    }
                    // twice the physical derivatives: D[a][i] = 2 du_i/dx_a
                    const float2 rh[3] = {rhx, rhy, bc(hz.y)};
                    float2 D[3][3];
#pragma unroll
                    for (int a = 0; a < 3; ++a)
#pragma unroll
                        for (int i = 0; i < 3; ++i) D[a][i] = mul2(d[a][i], rh[a]);
                    const float2 a01 = add2(D[0][1], D[1][0]), a02 = add2(D[0][2], D[2][0]), a12 = add2(D[1][2], D[2][1]);
                    const float2 sd = fma2(D[2][2], D[2][2], fma2(D[1][1], D[1][1], mul2(D[0][0], D[0][0])));
                    const float2 so = fma2(a12, a12, fma2(a02, a02, mul2(a01, a01)));
                    // mu_sgs / 4 = rho (Cs Delta)^2 / 4 (2 S_ij S_ij)^1/2
                    const float2 mus = mul2(mul2(O.rho, mul2(csxy, bc(hz.z))), sqrt2(fma2(so, bc(0.25f), mul2(sd, bc(0.5f)))));
                    const float2 sT = sqrtp2(O.T); // speed of sound
                    const float2 mu4 = mul2(mul2(O.T, sT), mul2(bc(__fmul_rn(0.25f, FP.suth1)), rcp2(add2(O.T, bc(FP.suthS)))));
                    X.mue = fma2(mu4, bc(FP.inv_Re), mus);
                    X.kap = fma2(mu4, bc(FP.kap_mol), mul2(mus, bc(FP.kap_sgs)));
                    // lambda_a = (|u_a| + c) / |h_a|; lambda-bar_a = s_a (s_a + s_b + s_d)
                    float2 sq[3];
#pragma unroll
                    for (int a = 0; a < 3; ++a)
                        sq[a] = sqrtp2(f2(__fmul_rn(__fadd_rn(fabsf(O.u[a].x), sT.x), fabsf(rh[a].x)),
                                         __fmul_rn(__fadd_rn(fabsf(O.u[a].y), sT.y), fabsf(rh[a].y))));
                    const float2 ss = add2(add2(sq[0], sq[1]), sq[2]);
                    Y.mue = Z.mue = X.mue;
                    Y.kap = Z.kap = X.kap;
                    X.nu = nu[0];
                    Y.nu = nu[1];
                    Z.nu = nu[2];
                    X.lb = mul2(sq[0], ss);
                    Y.lb = mul2(sq[1], ss);
                    Z.lb = mul2(sq[2], ss);
                    X.c[0] = D[1][0];
                    X.c[1] = D[2][0];
                    Y.c[0] = D[0][1];
                    Y.c[1] = D[2][1];
                    Z.c[0] = D[0][2];
                    Z.c[1] = D[1][2];
                    const float2 t23 = bc(2.0f / 3.0f);
                    X.s = mul2(t23, add2(D[1][1], D[2][2]));
                    Y.s = mul2(t23, add2(D[0][0], D[2][2]));
                    Z.s = mul2(t23, add2(D[0][0], D[1][1]));
                    if (g == kG) break;
                    tz = Z;
                }
                // ---- zeta flux between planes kU and kG; update of plane kU ----
                float2 gz[5];
                if (kG >= k0) {
                    const float4 z0 = S.HZ[kU & 3], z1 = S.HZ[kG & 3];
                    const float hbz = __fmul_rn(0.5f, __fadd_rn(z0.x, z1.x)), rz = __fmul_rn(4.0f, rcpa(hbz));
                    PP L;
                    ldp(CK_RING(bU + c2), L);
                    float2 Wm[5], Wp[5];
                    ldw(CK_RING(bM + c2), Wm);
                    if (ghost_hi) wvec(L, Wp); // W(nk) = W(nk - 2)
                    else ldw(CK_RING(bL + c2), Wp);
                    flux<2>(FP.k4, L, O, Wm, Wp, tz, Z, bc(hbz), bc(rz), bc(__fmul_rn(4.0f / 3.0f, rz)), gz);
                    if (do_upd && (outA || outB)) {
                        cp_async_wait_all(); // this thread's Q(0) copies
                        // flux differences of plane kU: + zeta above, - eta below (the
                        // first thread row's upper lane lies above the last row's lower lane)
                        const int ib_ = tr > 0 ? tid - FX : (TR - 1) * FX + tx;
                        const float2 rhzU = bc(z0.y);
                        float2 R[5];
#pragma unroll
                        for (int f = 0; f < 5; ++f) {
                            float2 gb = S.HG[CK_SH(f * NT + ib_)];
                            if (tr == 0) gb.y = gb.x;
                            R[f] = fma2(rhzU, sub2(gz[f], gzm[f]), acc[f]);
                            R[f] = fma2(rhy, sub2(S.HG[CK_SH(f * NT + tid)], gb), R[f]);
                        }
                        const int pU = gkU * plane;
                        const int oA = CK_G(4, pU + ocolA, J.npts_pad), oB = CK_G(4, pU + ocolB, J.npts_pad);
                        float2 q[5];
                        float *out;
                        if (rhs_only) {
                            // RHS = J^-1 times the sum of flux differences over 2 h
                            const float2 jv = mul2(f2(hyA0.x, hyB0.x), bc(__fmul_rn(__fmul_rn(0.5f, hx0.x), z0.x)));
#pragma unroll
                            for (int f = 0; f < 5; ++f) q[f] = mul2(jv, R[f]);
                            out = J.rhs;
                        } else {
#pragma unroll
                            for (int f = 0; f < 5; ++f)
                                q[f] = fma2(bc(-adt), R[f], f2(S.QZ[(2 * f) * NT + tid], S.QZ[(2 * f + 1) * NT + tid]));
                            out = J.q[dst];
                        }
                        if (outA) {
#pragma unroll
                            for (int f = 0; f < 5; ++f) out[f * fs + oA] = q[f].x;
                        }
                        if (outB) {
#pragma unroll
                            for (int f = 0; f < 5; ++f) out[f * fs + oB] = q[f].y;
                        }
                    }
#pragma unroll
                    for (int f = 0; f < 5; ++f) gzm[f] = gz[f];
                }
                tz = Z;
                if (kG >= k0 && kG < k1) {
                    // ---- xi and eta tables of plane kG (pair row TR: the middle pair
                    // with the upper lane's values below) ----
                    const int c1 = tid;
                    const float4 tb[6] = {cat4(X.mue, X.kap), cat4(X.nu, X.lb), cat4(X.c[0], X.c[1]),
                                          cat4(Y.nu, Y.lb), cat4(Y.c[0], Y.c[1]), cat4(X.s, Y.s)};
#pragma unroll
                    for (int q = 0; q < 6; ++q) S.TB[CK_TAB(q * N1 + c1, 6 * N1)] = tb[q];
                    if (tr == 0) { // as the row above thread row TR - 1: (row TR, unused)
#pragma unroll
                        for (int q = 0; q < 6; ++q)
                            S.TB[CK_TAB(q * N1 + TR * FX + tx, 6 * N1)] = make_float4(tb[q].y, tb[q].y, tb[q].w, tb[q].w);
                    }
                    __syncthreads(); // barrier B
                    // ---- xi and eta fluxes of plane kG ----
                    auto ldt = [&](int cell, Tr &t, int y) {
                        const float4 m = S.TB[CK_TAB(cell, 6 * N1)], n = S.TB[CK_TAB((y ? 3 : 1) * N1 + cell, 6 * N1)],
                                     c = S.TB[CK_TAB((y ? 4 : 2) * N1 + cell, 6 * N1)],
                                     s = S.TB[CK_TAB(5 * N1 + cell, 6 * N1)];
                        t.mue = lo2(m);
                        t.kap = hi2(m);
                        t.nu = lo2(n);
                        t.lb = hi2(n);
                        t.c[0] = lo2(c);
                        t.c[1] = hi2(c);
                        t.s = y ? hi2(s) : lo2(s);
                    };
                    const int b0 = bG + c2;
                    float2 Wm[5], Wp[5], g[5];
                    PP R;
                    Tr tR;
                    // eta: the row above; the top pair's upper flux is not used
                    ldp(CK_RING(b0 + C2), R);
                    ldw(CK_RING(b0 - C2), Wm);
                    ldw(CK_RING(b0 + 2 * C2), Wp);
                    ldt(c1 + FX, tR, 1);
                    flux<1>(FP.k4, O, R, Wm, Wp, Y, tR, hby, rhby, c43y, g);
#pragma unroll
                    for (int f = 0; f < 5; ++f) S.HG[CK_SH(f * NT + tid)] = g[f];
                    // xi: the next column; lane 31 pairs with its own tables (an
                    // unused result), so that every lane runs the same code
                    ldp(CK_RING(b0 + 1), R);
                    ldw(CK_RING(b0 - 1), Wm);
                    ldw(CK_RING(b0 + 2), Wp);
                    ldt(tx <= FX - 2 ? c1 + 1 : c1, tR, 0);
                    flux<0>(FP.k4, O, R, Wm, Wp, X, tR, hbx, rhbx, c43x, g);
#pragma unroll
                    for (int f = 0; f < 5; ++f) {
                        const float2 gm = f2(__shfl_up_sync(0xffffffffu, g[f].x, 1), __shfl_up_sync(0xffffffffu, g[f].y, 1));
                        acc[f] = mul2(rhx, sub2(g[f], gm));
                    }
                }
            }
            gkU = gkG;
            gkG = gkL;
            gkL = map_idx(kL + 1, nk, pk);
        }
        cp_async_wait_all(); // spacing copies past the last plane
        __syncthreads();     // the last update's reads of shared memory
    }
    cp_async_wait_all();
    // a copy whose wait gave up: see les_fused.cu
    if (pend && tid == 0 && !mbar_wait(S.MBAR, tpar, MBAR_WAIT_LIMIT)) {
        const JetDev<float> &J0 = jet_entry<ONE>(j1, jets, 0);
        if (J0.oob) atomicMax(J0.oob, 9ull << 48);
    }
}

#undef CK_G
#undef CK_RING
#undef CK_TAB
#undef CK_SH

template <int TY> static int prepare_one()
{
    int rc = (int)cudaFuncSetAttribute(k_fused_prod<TY, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)PGeo<TY>::BYTES);
    if (!rc) rc = (int)cudaFuncSetAttribute(k_fused_prod<TY, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)PGeo<TY>::BYTES);
    return rc;
}
int fused_prod_prepare()
{
    int rc = prepare_one<8>();
    if (!rc) rc = prepare_one<16>();
    if (!rc) rc = prepare_one<24>();
    return rc;
}

template <int TY> static int ctas_one()
{
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_fused_prod<TY, true>, FX * TY / 2, PGeo<TY>::BYTES) !=
        cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return n > 0 ? n : 1;
}
int fused_prod_ctas_per_sm(int ty) { return ty == 8 ? ctas_one<8>() : (ty == 16 ? ctas_one<16>() : ctas_one<24>()); }

template <int TY>
static void launch_one(const FusedLaunch &a, int grid, const JetDev<float> &ja, const FusedJet &fa, bool one, cudaStream_t st)
{
    const dim3 block(FX, TY / 2);
    const int lim = a.wait_limit < 0 ? MBAR_WAIT_LIMIT : a.wait_limit;
    if (one)
        k_fused_prod<TY, true><<<grid, block, PGeo<TY>::BYTES, st>>>(a.jets, a.fj, a.njets, a.items, a.tiles, a.src, a.dst,
                                                                    a.stage, a.dt, a.rhs_only, a.balanced, lim, ja, fa);
    else
        k_fused_prod<TY, false><<<grid, block, PGeo<TY>::BYTES, st>>>(a.jets, a.fj, a.njets, a.items, a.tiles, a.src, a.dst,
                                                                     a.stage, a.dt, a.rhs_only, a.balanced, lim, ja, fa);
}
void launch_fused_prod(int ty, const FusedLaunch &a, int grid, const JetDev<float> *j1, const FusedJet *f1, cudaStream_t st)
{
    const bool one = a.njets == 1 && j1 && f1;
    static const JetDev<float> jz{};
    static const FusedJet fz{};
    const JetDev<float> &ja = one ? *j1 : jz;
    const FusedJet &fa = one ? *f1 : fz;
    if (ty == 8) launch_one<8>(a, grid, ja, fa, one, st);
    else if (ty == 16) launch_one<16>(a, grid, ja, fa, one, st);
    else launch_one<24>(a, grid, ja, fa, one, st);
}

} // namespace les
