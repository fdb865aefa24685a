// Fused single-pass Runge-Kutta stage for FP32 storage and arithmetic, general
// metrics (jets on a product grid take les_fused_prod.cu).
//
// One kernel does what k_point, k_grads, k_iface and k_update do for the FP64
// path (Secs. "Numerical Formulation", "Time Marching Method"), with the
// intermediate per-point and per-interface quantities in shared memory and
// registers instead of HBM: per stage a point's state, Q(0) and static metrics
// are read and its new state written once.
//
// Row pairs and paired arithmetic.  A CTA of 32 x TY/2 threads owns a tile of
// 32 columns x TY rows (region R1) and updates its 30 x (TY-2) inner points.
// Thread (tx, tr) owns the two points of column tx in rows 2tr and 2tr+1 and
// evaluates everything of the two points together: each quantity is a float2
// whose lanes are the two rows, and the arithmetic runs as paired FP32
// instructions (add/mul/fma .f32x2, two results per issue).  Shared-memory
// records interleave the two rows the same way, so one 16-byte load yields two
// quantities of both points in register pairs.  The interfaces to the +xi and
// +zeta neighbours pair up row by row; the two +eta interfaces of a thread
// (rows 2tr|2tr+1 and 2tr+1|2tr+2) take their right-hand points from its own
// second row and the next thread row's first.
//
// Halo.  Point data (primitives and rho H) live in a ring of 3 planes over
// R2 = R1 plus one column on each side and two rows above and below; cells
// outside a non-periodic axis hold the mirror image of the point one beyond
// the boundary point (W(-1) = W(1), W(n) = W(n-2)), which is the paper's
// boundary fourth difference, so the interface arithmetic has no end cases.
// Derivatives, transport coefficients, sensors, lambda-bar and metric
// cofactors of R1 are kept for two planes.  Per loaded plane kL:
// primitives(kL) | gradients(kL-1) | interfaces + update(kL-2).  The
// gradients of the first plane of a non-periodic k axis, which need planes
// 0..2, are formed one plane late, together with plane 1.
//
// Work list.  Items (jet, tile x, tile y, k-chunk) are walked by a persistent
// grid in a fixed order; results do not depend on the item order, the chunk
// length or the grid size: every point is computed by the same instruction
// sequence whichever tile, lane or chunk it falls in.
#include <algorithm>
#include <cmath>

#include "les_fused.cuh"

namespace les {

namespace {

// ---------------------------------------------------------------------------
// Shared-memory map (byte offsets; 16-byte records first)
//   ring (3 planes) over R2 pair cells:  PA (rho, u)  PB (v, w)  PC (p, T)
//                                         float4 each; PH (rho H) float2
//   R1 tables (2 planes) over R1 pair cells:
//     GD [3 axes][2]  float4: 2 d/d xi^a of (u, v) and (w, T)
//     GC [4]          float4: (mu_eff, kappa), (nu_a, lambda-bar_a) a = 0..2
//   MA [3 planes][5] float4 over R1 pair cells: cofactors (m0 m1) (m2 m3)
//                             (m4 m5) (m6 m7) (m8 J^-1), streamed in by
//                             cp.async one plane ahead
//   SH [5][NT] float          eta flux of each thread's second row
//   QZ [5][TY-2][30] float    Q(0) of the tile's updated points, copied in
//                             by cp.async during the plane's iteration
//   QG [5][TY+4][40] float    the next plane's state box (TMA), 128-aligned,
//                             then its mbarrier
// A "pair cell" is one column of two rows (2p, 2p+1); its float4 records
// interleave the two rows: (q1(2p), q1(2p+1), q2(2p), q2(2p+1)).
// ---------------------------------------------------------------------------
template <int TY> struct Geo {
    static constexpr int TR = TY / 2;              // thread rows
    static constexpr int NT = FX * TR;             // threads
    static constexpr int C2 = FX + 2;              // R2 columns -1 .. FX
    static constexpr int P2 = TR + 2;              // R2 pair rows -1 .. TR (rows -2 .. TY+1)
    static constexpr int N2 = C2 * P2;             // R2 pair cells
    static constexpr int N1 = NT;                  // R1 pair cells
    static constexpr int BR = tma_box_rows(TY);    // rows of the staging box
    static constexpr int NR = 3;                   // planes of the point ring
    static constexpr size_t O_PA = 0;
    static constexpr size_t O_PB = O_PA + 16ull * NR * N2;
    static constexpr size_t O_PC = O_PB + 16ull * NR * N2;
    static constexpr size_t O_PH = O_PC + 16ull * NR * N2;
    static constexpr size_t O_GD = O_PH + 8ull * NR * N2;
    static constexpr size_t O_GC = O_GD + 16ull * 2 * 6 * N1;
    static constexpr size_t O_MA = O_GC + 16ull * 2 * 4 * N1;
    static constexpr size_t O_SH = O_MA + 16ull * 3 * 5 * N1;
    static constexpr int QZN = (TY - 2) * (FX - 2); // updated points of a tile plane
    static constexpr size_t O_QZ = (O_SH + 4ull * 5 * NT + 15) / 16 * 16;
    static constexpr size_t O_QG = (O_QZ + 4ull * 5 * QZN + 127) / 128 * 128;
    static constexpr unsigned BOX_BYTES = 4u * 5 * BR * TMA_BOX_X;
    static_assert(BOX_BYTES % 16 == 0, "box size");
    static constexpr size_t O_MBAR = O_QG + BOX_BYTES;
    static constexpr size_t O_FPS = O_MBAR + 8;
    static constexpr size_t BYTES = O_FPS + 64;
    static_assert(BYTES <= 227 * 1024, "shared memory of one CTA");
};

template <int TY> struct Sm {
    float4 *PA, *PB, *PC;
    float2 *PH;
    float4 *GD, *GC, *MA;
    float *SH, *QZ;
    float *QG;
    unsigned long long *MBAR;
    float *FPS; // a batch jet's constants (FusedParams) for the item
    __device__ __forceinline__ explicit Sm(unsigned char *b)
        : PA((float4 *)(b + Geo<TY>::O_PA)), PB((float4 *)(b + Geo<TY>::O_PB)),
          PC((float4 *)(b + Geo<TY>::O_PC)), PH((float2 *)(b + Geo<TY>::O_PH)),
          GD((float4 *)(b + Geo<TY>::O_GD)), GC((float4 *)(b + Geo<TY>::O_GC)),
          MA((float4 *)(b + Geo<TY>::O_MA)), SH((float *)(b + Geo<TY>::O_SH)),
          QZ((float *)(b + Geo<TY>::O_QZ)),
          QG((float *)(b + Geo<TY>::O_QG)), MBAR((unsigned long long *)(b + Geo<TY>::O_MBAR)),
          FPS((float *)(b + Geo<TY>::O_FPS))
    {
    }
};

// Slot of plane k (k >= -6) in the three-plane rings.
__device__ __forceinline__ int r3(int k) { return (k + 6) % 3; }

// Point data of one side of an interface: two points (the two lanes).
struct Pts {
    float2 rho, u, v, w, p, T, rH; // rH = rho H = e + p
};
__device__ __forceinline__ Pts odd_pts(const Pts &a, const Pts &b)
{
    Pts r;
    r.rho = odd2(a.rho, b.rho);
    r.u = odd2(a.u, b.u);
    r.v = odd2(a.v, b.v);
    r.w = odd2(a.w, b.w);
    r.p = odd2(a.p, b.p);
    r.T = odd2(a.T, b.T);
    r.rH = odd2(a.rH, b.rH);
    return r;
}
// Dissipation vector W = [rho, rho u, rho v, rho w, e + p] (Eq. W_dissip,
// with the unscaled conserved variables)
__device__ __forceinline__ void wvec(const Pts &q, float2 W[5])
{
    W[0] = q.rho;
    W[1] = mul2(q.rho, q.u);
    W[2] = mul2(q.rho, q.v);
    W[3] = mul2(q.rho, q.w);
    W[4] = q.rH;
}

// Transport data of one side: coefficients, sensor and lambda-bar along the
// interface axis, and the doubled derivatives 2 d/d xi^b of (u, v, w, T)
// along the two tangential axes b (ascending).
struct Side {
    float2 mue, kap, nu, lb;
    float2 d[2][4];
};

// Flux through the interfaces between the points L and their +A neighbours R
// (Eqs. spatial_discret, inv_flux_vec, dissip_term, eps_2/4_dissip; the
// compact viscous + SGS flux of the interface): the centred inviscid flux
// minus J^-1 d minus the viscous flux, general metric cofactors.  WLm, WRp:
// W of the outer points of the dissipation stencil.
template <int A>
__device__ __forceinline__ void iface(const FusedParams &FP, const Pts &L, const float2 WL[5], const float2 mL[9],
                                      float2 jL, const Pts &R, const float2 WR[5], const float2 mR[9], float2 jR,
                                      const float2 WLm[5], const float2 WRp[5], const Side &SL, const Side &SR,
                                      float2 H[5])
{
    const float2 half = bc(0.5f);
    // centred inviscid flux: J^-1 U = m_A . u; the ambient pressure is taken
    // out of the pressure terms (a constant pressure has no flux divergence,
    // and leaving it in adds FP32 rounding of O(1) terms to small momentum
    // residuals)
    const float2 hJL = mul2(half, fma2(mL[3 * A + 2], L.w, fma2(mL[3 * A + 1], L.v, mul2(mL[3 * A], L.u))));
    const float2 hJR = mul2(half, fma2(mR[3 * A + 2], R.w, fma2(mR[3 * A + 1], R.v, mul2(mR[3 * A], R.u))));
    const float2 hpinf = bc(-0.5f * FP.pinf);
    const float2 pl = fma2(L.p, half, hpinf), pr = fma2(R.p, half, hpinf);
    H[0] = fma2(WR[0], hJR, mul2(WL[0], hJL));
#pragma unroll
    for (int c = 0; c < 3; ++c)
        H[1 + c] = fma2(pr, mR[3 * A + c], fma2(pl, mL[3 * A + c], fma2(WR[1 + c], hJR, mul2(WL[1 + c], hJL))));
    H[4] = fma2(WR[4], hJR, mul2(WL[4], hJL));
    // Turkel-Vatsa dissipation: F += se4 (W(R+1) - W(L-1)) - (se2 + 3 se4)(W(R) - W(L))
    const float2 Js = add2(jL, jR); // 2 x interface J^-1
    {
        const float2 eps2 = mul2(bc(FP.k2), max2(SL.nu, SR.nu));
        const float2 eps4 = max2(bc(0.0f), sub2(bc(FP.k4), eps2));
        const float2 sc = mul2(mul2(bc(0.25f), Js), add2(SL.lb, SR.lb));
        const float2 se4 = mul2(sc, eps4);
        const float2 c2 = fma2(se4, bc(3.0f), mul2(sc, eps2));
#pragma unroll
        for (int f = 0; f < 5; ++f) H[f] = fma2(c2, sub2(WL[f], WR[f]), fma2(se4, sub2(WRp[f], WLm[f]), H[f]));
    }
    // compact viscous + SGS flux.  With Ms = m_L + m_R (twice the interface
    // cofactors) and D = 4 x the computational derivatives at the interface
    // (normal: 4 (phi_R - phi_L); tangential: the sum of the two points'
    // doubled central differences), G_fc = sum_b Ms_bc D_fb = 4 Js d phi_f / d x_c.
    // Only row A of the stress tensor is needed:
    //   s_i = coef/(16 Js) (X_i + Y_i - 2/3 Ms_Ai div),  coef = mu_eff,L + mu_eff,R
    //   X_f = sum_c Ms_Ac G_fc = sum_b K_b D_fb,  K_b = sum_c Ms_Ac Ms_bc
    //   Y_i = sum_c Ms_Ac G_ci = sum_b Ms_bi w_b,  w_b = sum_c Ms_Ac D_cb
    //   div = sum_i G_ii
    // and the energy flux is s . u_interface + (kappa_L + kappa_R) X_T / (16 Js).
    // The factor 4 of the normal derivatives sits in K_A and w_A, the part b = A
    // of the divergence is w_A, and coef and kappa enter negated, so that the flux
    // takes them up by FMAs: 10 paired instructions of a flux less than term by
    // term (with the cube root of rcbrt2, polar 400x150x60 265 -> 259 us a stage).
    {
        constexpr int B1 = A == 0 ? 1 : 0, B2 = A == 2 ? 1 : 2;
        float2 Ms[9];
#pragma unroll
        for (int t = 0; t < 9; ++t) Ms[t] = add2(mL[t], mR[t]);
        float2 D[4][3]; // D[f][A] without its 4
        D[0][A] = sub2(R.u, L.u);
        D[1][A] = sub2(R.v, L.v);
        D[2][A] = sub2(R.w, L.w);
        D[3][A] = sub2(R.T, L.T);
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            D[f][B1] = add2(SL.d[0][f], SR.d[0][f]);
            D[f][B2] = add2(SL.d[1][f], SR.d[1][f]);
        }
        float2 K[3], wv[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            K[b] = fma2(Ms[3 * A + 2], Ms[3 * b + 2], fma2(Ms[3 * A + 1], Ms[3 * b + 1], mul2(Ms[3 * A], Ms[3 * b])));
            wv[b] = fma2(Ms[3 * A + 2], D[2][b], fma2(Ms[3 * A + 1], D[1][b], mul2(Ms[3 * A], D[0][b])));
        }
        K[A] = mul2(K[A], bc(4.0f));
        wv[A] = mul2(wv[A], bc(4.0f));
        float2 X[4];
#pragma unroll
        for (int f = 0; f < 4; ++f) X[f] = fma2(K[2], D[f][2], fma2(K[1], D[f][1], mul2(K[0], D[f][0])));
        float2 dv = wv[A], dw = mul2(Ms[3 * B2], D[0][B2]);
        dv = fma2(Ms[3 * B1], D[0][B1], dv);
        dw = fma2(Ms[3 * B2 + 1], D[1][B2], dw);
        dv = fma2(Ms[3 * B1 + 1], D[1][B1], dv);
        dw = fma2(Ms[3 * B2 + 2], D[2][B2], dw);
        dv = fma2(Ms[3 * B1 + 2], D[2][B1], dv);
        dv = add2(dv, dw);
        const float2 rJ = mul2(rcp2(Js), bc(-1.0f / 16.0f));
        const float2 f1 = mul2(add2(SL.mue, SR.mue), rJ);
        const float2 ntd = mul2(mul2(f1, bc(-2.0f / 3.0f)), dv);
        float2 s[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const float2 Y = fma2(Ms[6 + i], wv[2], fma2(Ms[3 + i], wv[1], fma2(Ms[i], wv[0], X[i])));
            s[i] = fma2(Ms[3 * A + i], ntd, mul2(f1, Y));
            H[1 + i] = add2(H[1 + i], s[i]);
        }
        const float2 kh = mul2(add2(SL.kap, SR.kap), rJ);
        const float2 e = fma2(s[2], add2(L.w, R.w), fma2(s[1], add2(L.v, R.v), mul2(s[0], add2(L.u, R.u))));
        H[4] = fma2(kh, X[3], fma2(half, e, H[4]));
    }
}

} // namespace

// Index checks of a LES_BOUNDS_CHECK build (nothing otherwise): global
// offsets against their arrays (site 2 state, 3 static records, 4 update),
// shared-memory slots against their tables (5 point ring, 6 R1 tables and
// the staging box, 7 eta-flux rows).
#define CK_G(site, x, n) LES_BOUNDS(J.oob, (site), (x), (n))
#define CK_RING(x) ((int)LES_BOUNDS(J.oob, 5, (x), G_::NR * N2))
#define CK_TAB(x, n) ((int)LES_BOUNDS(J.oob, 6, (x), (n)))
#define CK_SH(x) ((int)LES_BOUNDS(J.oob, 7, (x), 5 * NT))

template <int TY, bool ONE>
__global__ void __launch_bounds__(FX * TY / 2, 1)
    k_fused(const JetDev<float> *__restrict__ jets, const FusedJet *__restrict__ fj, int njets,
            int total_items, int total_tiles, int src, int dst, int stage, const double *__restrict__ dt,
            int rhs_only, int balanced, int wait_limit, const __grid_constant__ JetDev<float> j1,
            const __grid_constant__ FusedJet f1)
{
    using G_ = Geo<TY>;
    constexpr int TR = G_::TR, NT = G_::NT, C2 = G_::C2, N2 = G_::N2, N1 = G_::N1, BR = G_::BR;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const Sm<TY> S(smem_raw);
    const int tx = threadIdx.x, tr = threadIdx.y;
    const int tid = tr * FX + tx;
    const int c1 = tid;                       // own R1 pair cell
    const int c2 = (tr + 1) * C2 + (tx + 1);  // own R2 pair cell

    // general form: the TMA staging buffer must be 128-byte aligned (the
    // dynamic shared memory starts the window, so it is; checked anyway)
    const bool tma_smem_ok = (smem_u32(S.QG) & 127u) == 0;
    unsigned tpar = 0; // parity of the next staging phase
    // A staging wait that gives up (wait_limit polls) is recorded in the
    // jet's error word (site 8); from the next barrier on the whole CTA reads
    // the state directly from global memory for the rest of the launch, and
    // thread 0, which issued the outstanding copy, waits for it (bounded)
    // before the CTA exits.
    bool tma_off = false, pend = false;
    if (tid == 0) mbar_init(S.MBAR);
    __syncthreads();

    Cursor<ONE> cur(fj, f1, njets, total_items, total_tiles, balanced);
    int key, jet;
    while (cur.next(key, jet)) {
        const JetDev<float> &J = jet_entry<ONE>(j1, jets, jet);
        const FusedJet &F = jet_entry<ONE>(f1, fj, jet);
        if constexpr (!ONE) {
            // staged for the item (the previous item's last reads of FPS
            // precede its closing barrier; the item barrier below publishes it)
            constexpr int NFP = sizeof(FusedParams) / 4;
            if (tid >= NT - NFP) S.FPS[tid - (NT - NFP)] = reinterpret_cast<const float *>(&F.fp)[tid - (NT - NFP)];
        }
        const FusedParams &FP = jet_params<ONE>(F.fp, S.FPS);
        const int ni = J.n[0], nj = J.n[1], nk = J.n[2];
        const int pi = J.per[0], pj = J.per[1], pk = J.per[2];
        // output ranges; on a periodic j axis the tiles start at row 1 (so that
        // their row pairs start on even rows) and the last one wraps to row 0
        const int ilo = pi ? 0 : 1, ihi = pi ? ni : ni - 1;
        const int jlo = 1, jhi = pj ? nj + 1 : nj - 1;
        const int klo = pk ? 0 : 1, khi = pk ? nk : nk - 1;
        int bx, by, k0, k1;
        cur.take(key, F, klo, khi, bx, by, k0, k1);
        const int i0 = ilo + bx * (FX - 2), j0 = jlo + by * (TY - 2);
        const int ib = i0 - 1, jb = j0 - 1; // grid column / row of the tile's first R1 cell (jb even)
        // 32-bit offsets: creation limits an FP32 jet to 5 fields x fs and its
        // static records to fewer than 2^31 elements
        const int fs = (int)J.fs;
        const int plane = nj * J.pitch;
        const float *__restrict__ Qs = J.q[src];
        float *__restrict__ Qd = J.q[dst];
        const float adt = rhs_only ? 0.0f : c_alpha_f[stage] * (float)dt[jet];
        const float4 *__restrict__ mp = F.mp;
        const long long nrec = (long long)nk * F.njp * 5 * J.pitch;
        (void)nrec; // bound of the static-record checks of a LES_BOUNDS_CHECK build

        // ---- per-item setup ----
        // own column and rows (R1); static-record column and row pair
        const int gi = map_idx(ib + tx, ni, pi);
        const int rA = 2 * tr, rB = 2 * tr + 1;
        const int gjA = map_idx(jb + rA, nj, pj), gjB = map_idx(jb + rB, nj, pj);
        // the two rows share one paired static record (pair jpA) unless a
        // periodic j axis of odd length wraps between them; rows beyond a
        // non-periodic grid read the last record (their values feed no result)
        const bool rec_split = pj && (nj & 1);
        const int jpA = min((pj ? gjA : jb + rA) >> 1, F.njp - 1);
        // in-plane derivative stencils (0: central; +-1: one-sided at a
        // non-periodic end), per column and per row
        const int ti = (!pi && ib + tx == 0) ? 1 : ((!pi && ib + tx == ni - 1) ? -1 : 0);
        const int tjA = (!pj && jb + rA == 0) ? 1 : ((!pj && jb + rA == nj - 1) ? -1 : 0);
        const int tjB = (!pj && jb + rB == nj - 1) ? -1 : 0; // jb even: row 0 is never a second row
        // outputs: columns 1..30, rows 1..TY-2 of R1 inside the output range
        const bool col_out = tx >= 1 && tx <= FX - 2 && (ib + tx) < ihi;
        const bool outA = col_out && rA >= 1 && rA <= TY - 2 && (jb + rA) < jhi;
        const bool outB = col_out && rB >= 1 && rB <= TY - 2 && (jb + rB) < jhi;
        const int ocolA = gjA * J.pitch + gi, ocolB = gjB * J.pitch + gi;
        // slots of the two rows' Q(0) values in QZ (outputs only)
        const int zA = (rA - 1) * (FX - 2) + (tx - 1), zB = (rB - 1) * (FX - 2) + (tx - 1);
        // the R2 pair cells this thread loads (at most two) and, per row, the
        // offset of its source point in the staging box and in a plane
        int lc[2];
        int bo[2][2];
        int go[2][2];
        const CUtensorMap *tmap = nullptr;
        int tx0 = 0;
        if (F.tmap && tma_smem_ok && !pi && !pj && !tma_off) {
            tmap = F.tmap + (TY == 16 ? 3 : 0) + src;
            tx0 = (ib - 1) & ~3;
        }
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            const int c = tid + t * NT;
            lc[t] = c < N2 ? c : -1;
            const int cc = (c < N2 ? c : 0) % C2, pr = (c < N2 ? c : 0) / C2;
            const int gc = map_idx(ib - 1 + cc, ni, pi);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int gr = map_idx(jb + 2 * (pr - 1) + h, nj, pj);
                go[t][h] = gr * J.pitch + gc;
                int rr = gr - (jb - 2), cl = gc - tx0;
                rr = rr < 0 ? 0 : (rr > BR - 1 ? BR - 1 : rr);
                cl = cl < 0 ? 0 : (cl > TMA_BOX_X - 1 ? TMA_BOX_X - 1 : cl);
                bo[t][h] = rr * TMA_BOX_X + cl;
            }
        }
        // carried from plane to plane: the zeta flux below, W of the own
        // column one plane below the interface plane, J of the next update
        float2 hz_prev[5], Wc[5];
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            hz_prev[f] = bc(0.0f);
            Wc[f] = bc(0.0f);
        }
        float2 rjU = bc(0.0f), rjG = bc(0.0f);
        __syncthreads(); // shared memory of the previous item is free

        // thread 0 issues the box of plane kq once every thread is done with
        // the previous one (after a barrier)
        auto stage_box = [&](int kq) {
            if (tid != 0) return;
            const int gk = map_idx(kq, nk, pk);
            tma_box_load(S.QG, tmap, tx0, jb - 2, gk, S.MBAR, G_::BOX_BYTES);
        };
        const int kfirst = k0 - 2, klast = k1 + 1;
        // carried per iteration: grid planes of kL - 2, kL - 1, kL and the
        // three-plane ring slot of kL
        int gkUc = map_idx(kfirst - 2, nk, pk), gkGc = map_idx(kfirst - 1, nk, pk), gkLc = map_idx(kfirst, nk, pk);
        int q3c = r3(kfirst);
        if (tmap) stage_box(kfirst);

        // ---- metric cofactors and J^-1 of grid plane gk for the own row pair
        //      (general form) into MA slot q3: asynchronous copies, waited for one
        //      plane later; where the two rows come from two records, plain loads ----
        auto fetch_met = [&](int gk, int q3) {
            float4 *dst = S.MA + CK_TAB((q3 * 5) * N1 + c1, 15 * N1);
            const int rp = J.pitch;
            if (!rec_split) {
                const int r0 = (gk * F.njp + jpA) * 5 * rp + gi;
                const float4 *p = mp + CK_G(3, r0, nrec);
                (void)CK_G(3, r0 + 4 * rp, nrec);
#pragma unroll
                for (int q = 0; q < 5; ++q) cp_async16(dst + q * N1, p + q * rp);
            } else {
                // rows from two records: take each row's lane
                const int ra = (gk * F.njp + (gjA >> 1)) * 5 * rp + gi;
                const int rb = (gk * F.njp + (gjB >> 1)) * 5 * rp + gi;
                const float4 *pa = mp + CK_G(3, ra, nrec);
                const float4 *pb = mp + CK_G(3, rb, nrec);
                (void)CK_G(3, ra + 4 * rp, nrec);
                (void)CK_G(3, rb + 4 * rp, nrec);
                const bool sa = gjA & 1, sb = gjB & 1;
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    const float4 a = pa[q * rp], b = pb[q * rp];
                    dst[q * N1] = make_float4(sa ? a.y : a.x, sb ? b.y : b.x, sa ? a.w : a.z, sb ? b.w : b.z);
                }
            }
        };

        // ---- gradients, closures, sensors, lambda-bar of plane kg (grid plane gk;
        //      three-plane ring slots q3, q3m, q3p of planes kg, kg - 1, kg + 1) ----
        auto grad = [&](int kg, int gk, int q3, int q3m, int q3p) {
            // ring slots of planes kg, kg - 1 (= kg + 2), kg + 1 (= kg - 2)
            const int slm = q3m, slp = q3p, slm2 = q3p, slp2 = q3m;
            const int s0 = q3 * N2;
            const int slot = kg & 1;
            const int own = CK_RING(s0 + c2);
            const float4 a0 = S.PA[own], b0 = S.PB[own], q0 = S.PC[own];
            const float2 rho = lo2(a0), p0 = lo2(q0), T0 = hi2(q0);
            const float2 U0[3] = {hi2(a0), lo2(b0), hi2(b0)};
            float2 d[3][4]; // 2 x d/d xi^a of (u, v, w, T)
            float2 nu[3];
            auto sensor = [&](float2 pm, float2 pc, float2 pp) {
                const float2 s = add2(pm, pp);
                const float2 num = fma2(pc, bc(-2.0f), s), den = fma2(pc, bc(2.0f), s);
                const float2 r = rcp2(den);
                return make_float2(fabsf(num.x) * r.x, fabsf(num.y) * r.y);
            };
            // along xi: central, or one-sided over the cells c, c+t, c+2t at a
            // non-periodic end (the sensor of an end point is its interior
            // neighbour's: same three points)
            if (ti == 0) {
                const int om = CK_RING(s0 + c2 - 1), op = CK_RING(s0 + c2 + 1);
                const float4 am = S.PA[om], bm = S.PB[om], qm = S.PC[om];
                const float4 ap = S.PA[op], bp = S.PB[op], qp = S.PC[op];
                d[0][0] = sub2(hi2(ap), hi2(am));
                d[0][1] = sub2(lo2(bp), lo2(bm));
                d[0][2] = sub2(hi2(bp), hi2(bm));
                d[0][3] = sub2(hi2(qp), hi2(qm));
                nu[0] = sensor(lo2(qm), p0, lo2(qp));
            } else {
                const int o1 = CK_RING(s0 + c2 + ti), o2 = CK_RING(s0 + c2 + 2 * ti);
                const float4 a1 = S.PA[o1], b1 = S.PB[o1], q1 = S.PC[o1];
                const float4 a2 = S.PA[o2], b2 = S.PB[o2], q2 = S.PC[o2];
                const float2 w0 = bc(-3.0f * ti), w1 = bc(4.0f * ti), w2 = bc(-1.0f * ti);
                d[0][0] = fma2(w2, hi2(a2), fma2(w1, hi2(a1), mul2(w0, U0[0])));
                d[0][1] = fma2(w2, lo2(b2), fma2(w1, lo2(b1), mul2(w0, U0[1])));
                d[0][2] = fma2(w2, hi2(b2), fma2(w1, hi2(b1), mul2(w0, U0[2])));
                d[0][3] = fma2(w2, hi2(q2), fma2(w1, hi2(q1), mul2(w0, T0)));
                nu[0] = sensor(p0, lo2(q1), lo2(q2));
            }
            // along eta: rows 2tr-2 .. 2tr+3 from the pair cells below, own, above
            {
                const int om = CK_RING(s0 + c2 - C2), op = CK_RING(s0 + c2 + C2);
                const float4 am = S.PA[om], bm = S.PB[om], qm = S.PC[om];
                const float4 ap = S.PA[op], bp = S.PB[op], qp = S.PC[op];
                // per field u, v, w, T, p: rows [2tr-2, 2tr-1 | 2tr, 2tr+1 | 2tr+2, 2tr+3]
                const float2 fm[5] = {hi2(am), lo2(bm), hi2(bm), hi2(qm), lo2(qm)};
                const float2 fo[5] = {U0[0], U0[1], U0[2], T0, p0};
                const float2 fp[5] = {hi2(ap), lo2(bp), hi2(bp), hi2(qp), lo2(qp)};
                if (tjA == 0 && tjB == 0) {
#pragma unroll
                    for (int f = 0; f < 4; ++f) d[1][f] = make_float2(fo[f].y - fm[f].y, fp[f].x - fo[f].x);
                    nu[1] = sensor(odd2(fm[4], fo[4]), p0, odd2(fo[4], fp[4]));
                } else {
                    // one row (or both) at an end of a non-periodic j axis:
                    // per row, from the values of rows r-2 .. r+2
                    float v[5][6];
#pragma unroll
                    for (int f = 0; f < 5; ++f) {
                        v[f][0] = fm[f].x; v[f][1] = fm[f].y; v[f][2] = fo[f].x;
                        v[f][3] = fo[f].y; v[f][4] = fp[f].x; v[f][5] = fp[f].y;
                    }
                    float dA[4], dB[4], nA, nB;
                    auto row = [&](int r0, int t, float dd[4], float &nn) {
                        if (t == 0) {
#pragma unroll
                            for (int f = 0; f < 4; ++f) dd[f] = v[f][r0 + 1] - v[f][r0 - 1];
                            const float s = v[4][r0 + 1] + v[4][r0 - 1];
                            nn = fabsf(fmaf(v[4][r0], -2.0f, s)) * __fdividef(1.0f, fmaf(v[4][r0], 2.0f, s));
                        } else {
                            const float w0 = -3.0f * t, w1 = 4.0f * t, w2 = -1.0f * t;
#pragma unroll
                            for (int f = 0; f < 4; ++f)
                                dd[f] = fmaf(w2, v[f][r0 + 2 * t], fmaf(w1, v[f][r0 + t], w0 * v[f][r0]));
                            const float s = v[4][r0] + v[4][r0 + 2 * t];
                            nn = fabsf(fmaf(v[4][r0 + t], -2.0f, s)) * __fdividef(1.0f, fmaf(v[4][r0 + t], 2.0f, s));
                        }
                    };
                    row(2, tjA, dA, nA);
                    row(3, tjB, dB, nB);
#pragma unroll
                    for (int f = 0; f < 4; ++f) d[1][f] = make_float2(dA[f], dB[f]);
                    nu[1] = make_float2(nA, nB);
                }
            }
            // along zeta: the own column one plane below / above, or one-sided
            // at an end of a non-periodic k axis
            {
                const int tk = (!pk && gk == 0) ? 1 : ((!pk && gk == nk - 1) ? -1 : 0);
                if (tk == 0) {
                    const int om = CK_RING(slm * N2 + c2), op = CK_RING(slp * N2 + c2);
                    const float4 am = S.PA[om], bm = S.PB[om], qm = S.PC[om];
                    const float4 ap = S.PA[op], bp = S.PB[op], qp = S.PC[op];
                    d[2][0] = sub2(hi2(ap), hi2(am));
                    d[2][1] = sub2(lo2(bp), lo2(bm));
                    d[2][2] = sub2(hi2(bp), hi2(bm));
                    d[2][3] = sub2(hi2(qp), hi2(qm));
                    nu[2] = sensor(lo2(qm), p0, lo2(qp));
                } else {
                    const int o1 = CK_RING((tk > 0 ? slp : slm) * N2 + c2), o2 = CK_RING((tk > 0 ? slp2 : slm2) * N2 + c2);
                    const float4 a1 = S.PA[o1], b1 = S.PB[o1], q1 = S.PC[o1];
                    const float4 a2 = S.PA[o2], b2 = S.PB[o2], q2 = S.PC[o2];
                    const float2 w0 = bc(-3.0f * tk), w1 = bc(4.0f * tk), w2 = bc(-1.0f * tk);
                    d[2][0] = fma2(w2, hi2(a2), fma2(w1, hi2(a1), mul2(w0, U0[0])));
                    d[2][1] = fma2(w2, lo2(b2), fma2(w1, lo2(b1), mul2(w0, U0[1])));
                    d[2][2] = fma2(w2, hi2(b2), fma2(w1, hi2(b1), mul2(w0, U0[2])));
                    d[2][3] = fma2(w2, hi2(q2), fma2(w1, hi2(q1), mul2(w0, T0)));
                    nu[2] = sensor(p0, lo2(q1), lo2(q2));
                }
            }
            // metrics: cofactors m (rows of d xi^a / d x times J^-1), J,
            // (Cs Delta)^2 J, row norms
            float2 m[9], rj, csdJ, nrm[3];
            {
                float4 u[5];
#pragma unroll
                for (int q = 0; q < 5; ++q) u[q] = S.MA[CK_TAB((q3 * 5 + q) * N1 + c1, 15 * N1)];
                m[0] = lo2(u[0]); m[1] = hi2(u[0]); m[2] = lo2(u[1]); m[3] = hi2(u[1]);
                m[4] = lo2(u[2]); m[5] = hi2(u[2]); m[6] = lo2(u[3]); m[7] = hi2(u[3]);
                m[8] = lo2(u[4]);
                // J, (Cs Delta)^2 J = Cs^2 (J^-1)^(-1/3) with Delta = (J^-1)^(1/3), and
                // the row norms |grad xi^a| / J; on the degenerate axis of a polar
                // mesh (J^-1 = 0) J = 1 and the filter width is zero
                const float2 jv = hi2(u[4]);
                rj = f2(jv.x > 0.0f ? rcpa(jv.x) : 1.0f, jv.y > 0.0f ? rcpa(jv.y) : 1.0f);
                const float2 rc = rcbrt2(jv);
                csdJ = f2(jv.x > 0.0f ? FP.cs2 * rc.x : 0.0f, jv.y > 0.0f ? FP.cs2 * rc.y : 0.0f);
#pragma unroll
                for (int a = 0; a < 3; ++a) {
                    nrm[a] = sqrt2(fma2(m[3 * a + 2], m[3 * a + 2], fma2(m[3 * a + 1], m[3 * a + 1], mul2(m[3 * a], m[3 * a]))));
                }
            }
            // doubled physical velocity gradient g' = 2 J^-1 du_i/dx_c, strain norm,
            // Smagorinsky
            float2 g[3][3];
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int cc = 0; cc < 3; ++cc)
                    g[i][cc] = fma2(m[6 + cc], d[2][i], fma2(m[3 + cc], d[1][i], mul2(m[cc], d[0][i])));
            const float2 a01 = add2(g[0][1], g[1][0]), a02 = add2(g[0][2], g[2][0]), a12 = add2(g[1][2], g[2][1]);
            const float2 sd = fma2(g[2][2], g[2][2], fma2(g[1][1], g[1][1], mul2(g[0][0], g[0][0])));
            const float2 so = fma2(a12, a12, fma2(a02, a02, mul2(a01, a01)));
            // |S| = (2 S_ij S_ij)^1/2 = J sqrt(sd/2 + so/4) in terms of g'
            const float2 mus = mul2(mul2(rho, csdJ), sqrt2(fma2(so, bc(0.25f), mul2(sd, bc(0.5f)))));
            // Sutherland mu(T), speed of sound c = T^1/2
            const float2 sT = sqrtp2(T0);
            const float2 mu = mul2(mul2(T0, sT), mul2(bc(FP.suth1), rcp2(add2(T0, bc(FP.suthS)))));
            const float2 mue = fma2(mu, bc(FP.inv_Re), mus);
            const float2 kap = fma2(mu, bc(FP.kap_mol), mul2(mus, bc(FP.kap_sgs)));
            // spectral radii lambda_a = |U_a| + c |grad xi^a|, lambda-bar_a =
            // s_a (s_a + s_b + s_d) with s = lambda^1/2
            float2 sq[3];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                const float2 JU = fma2(m[3 * a + 2], U0[2], fma2(m[3 * a + 1], U0[1], mul2(m[3 * a], U0[0])));
                const float2 lam =
                    mul2(make_float2(fmaf(sT.x, nrm[a].x, fabsf(JU.x)), fmaf(sT.y, nrm[a].y, fabsf(JU.y))), rj);
                sq[a] = sqrt2(lam);
            }
            const float2 ssum = add2(add2(sq[0], sq[1]), sq[2]);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                S.GD[CK_TAB((slot * 6 + 2 * a) * N1 + c1, 12 * N1)] = cat4(d[a][0], d[a][1]);
                S.GD[CK_TAB((slot * 6 + 2 * a + 1) * N1 + c1, 12 * N1)] = cat4(d[a][2], d[a][3]);
            }
            S.GC[CK_TAB((slot * 4) * N1 + c1, 8 * N1)] = cat4(mue, kap);
#pragma unroll
            for (int a = 0; a < 3; ++a)
                S.GC[CK_TAB((slot * 4 + 1 + a) * N1 + c1, 8 * N1)] = cat4(nu[a], mul2(sq[a], ssum));
            rjG = rj;
        };

        // ---- shared-memory accessors of the interface phase ----
        auto pts = [&](int cell) {
            Pts P;
            const float4 a = S.PA[cell], b = S.PB[cell], q = S.PC[cell];
            P.rho = lo2(a); P.u = hi2(a); P.v = lo2(b); P.w = hi2(b); P.p = lo2(q); P.T = hi2(q);
            P.rH = S.PH[cell];
            return P;
        };
        auto wof = [&](int cell, float2 W[5]) {
            const float4 a = S.PA[cell], b = S.PB[cell];
            const float2 rho = lo2(a);
            W[0] = rho;
            W[1] = mul2(rho, hi2(a));
            W[2] = mul2(rho, lo2(b));
            W[3] = mul2(rho, hi2(b));
            W[4] = S.PH[cell];
        };
        auto mets = [&](int slot, int cell, float2 m[9], float2 &jv) {
            float4 u[5];
#pragma unroll
            for (int q = 0; q < 5; ++q) u[q] = S.MA[CK_TAB((slot * 5 + q) * N1 + cell, 15 * N1)];
            m[0] = lo2(u[0]); m[1] = hi2(u[0]); m[2] = lo2(u[1]); m[3] = hi2(u[1]);
            m[4] = lo2(u[2]); m[5] = hi2(u[2]); m[6] = lo2(u[3]); m[7] = hi2(u[3]);
            m[8] = lo2(u[4]);
            jv = hi2(u[4]);
        };
        // transport data along axis A: coefficients, (nu_A, lb_A), and
        // the doubled derivatives along the two other axes
        auto side = [&](int A, int slot, int cell, Side &Sd) {
            const float4 c0 = S.GC[CK_TAB((slot * 4) * N1 + cell, 8 * N1)];
            const float4 ca = S.GC[CK_TAB((slot * 4 + 1 + A) * N1 + cell, 8 * N1)];
            Sd.mue = lo2(c0); Sd.kap = hi2(c0); Sd.nu = lo2(ca); Sd.lb = hi2(ca);
            const int b1 = A == 0 ? 1 : 0, b2 = A == 2 ? 1 : 2;
            const float4 e0 = S.GD[CK_TAB((slot * 6 + 2 * b1) * N1 + cell, 12 * N1)];
            const float4 e1 = S.GD[CK_TAB((slot * 6 + 2 * b1 + 1) * N1 + cell, 12 * N1)];
            const float4 f0 = S.GD[CK_TAB((slot * 6 + 2 * b2) * N1 + cell, 12 * N1)];
            const float4 f1v = S.GD[CK_TAB((slot * 6 + 2 * b2 + 1) * N1 + cell, 12 * N1)];
            Sd.d[0][0] = lo2(e0); Sd.d[0][1] = hi2(e0); Sd.d[0][2] = lo2(e1); Sd.d[0][3] = hi2(e1);
            Sd.d[1][0] = lo2(f0); Sd.d[1][1] = hi2(f0); Sd.d[1][2] = lo2(f1v); Sd.d[1][3] = hi2(f1v);
        };
        for (int kL = kfirst; kL <= klast; ++kL) {
            const int kG = kL - 1, kU = kL - 2;
            // slots of planes kL, kG, kU in the three-plane rings, and their
            // grid planes
            const int q3L = q3c, q3G = q3L == 0 ? 2 : q3L - 1, q3U = q3L == 2 ? 0 : q3L + 1;
            const int gkLm = gkLc, gkGm = gkGc, gkUm = gkUc;
            const int sLr = q3L, sGr = q3G, sUr = q3U;
            const bool do_grad = kG >= k0 - 1 && kG <= k1 && !(!pk && kG == 0);
            // the first plane of a non-periodic k axis: formed with plane 1
            const bool do_grad0 = !pk && kG == 1 && k0 == 1;
            // the mirror plane beyond the last plane of a non-periodic k axis is
            // not loaded (its slot still holds a plane the last gradients need);
            // the last interface takes the mirror from its own plane
            const bool ghost_hi = !pk && kL == nk;
            // ---- load + primitives of plane kL on R2 ----
            if (!ghost_hi) {
                const int gkL = gkLm;
                bool from_box = false;
                if (tmap) {
                    // the box of this plane (issued one iteration earlier); a
                    // wait that gives up is recorded (site 8) instead of
                    // hanging, and this thread reads the plane from global memory
                    if (mbar_wait(S.MBAR, tpar, wait_limit)) {
                        from_box = true;
                        tpar ^= 1u;
                    } else {
                        if (J.oob) atomicCAS(J.oob, 0ull, 8ull << 48);
                        tma_off = true;
                        pend = true;
                    }
                }
                const int sb = sLr * N2;
                const int pofs = gkL * plane;
#pragma unroll
                for (int t = 0; t < 2; ++t) {
                    if (lc[t] < 0) continue;
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
                    const float2 rho = f2(q[0][0], q[1][0]);
                    const float2 rr = rcp2(rho);
                    const float2 u = mul2(f2(q[0][1], q[1][1]), rr), v = mul2(f2(q[0][2], q[1][2]), rr),
                                 ww = mul2(f2(q[0][3], q[1][3]), rr);
                    const float2 e = f2(q[0][4], q[1][4]);
                    const float2 q2 = fma2(ww, ww, fma2(v, v, mul2(u, u)));
                    const float2 p = mul2(bc(FP.gm1), fma2(mul2(rho, q2), bc(-0.5f), e));
                    const int cell = CK_RING(sb + lc[t]);
                    S.PA[cell] = cat4(rho, u);
                    S.PB[cell] = cat4(v, ww);
                    S.PC[cell] = cat4(p, mul2(mul2(bc(FP.gam), p), rr));
                    S.PH[cell] = add2(e, p);
                }
            }
            // (a thread whose staging wait gave up turns staging off for the
            // whole CTA here)
            tma_off = __syncthreads_or(tma_off) != 0;
            if (tma_off) tmap = nullptr;
            // the next plane's box, in flight during the rest of this iteration
            if (tmap && kL < klast && !(!pk && kL + 1 == nk)) stage_box(kL + 1);
            // one copy group per iteration: the metrics of the next gradient
            // plane (kL), waited for in the next iteration, and Q(0) of this
            // iteration's updated points (plane kL - 2), waited for before
            // the update; each thread copies, and later reads, its own values
            if (kL >= k0 - 1 && kL <= k1) fetch_met(gkLm, q3L);
            if (!rhs_only && kL - 2 >= k0 && kL - 2 <= k1 - 1) {
                const int pU = gkUm * plane;
                const float *Q0 = J.q[0];
                if (outA) {
                    const int oA = CK_G(4, pU + ocolA, J.npts_pad);
#pragma unroll
                    for (int f = 0; f < 5; ++f) cp_async4(S.QZ + CK_TAB(f * G_::QZN + zA, 5 * G_::QZN), Q0 + f * fs + oA);
                }
                if (outB) {
                    const int oB = CK_G(4, pU + ocolB, J.npts_pad);
#pragma unroll
                    for (int f = 0; f < 5; ++f) cp_async4(S.QZ + CK_TAB(f * G_::QZN + zB, 5 * G_::QZN), Q0 + f * fs + oB);
                }
            }
            cp_async_commit();
            // W of the own column at plane k0 - 2: the outer point of the
            // chunk's first zeta interface
            if (kL == k0) wof(CK_RING(sUr * N2 + c2), Wc);
            // ---- gradients of plane kG (and of plane 0, late) ----
            if (do_grad || do_grad0) cp_async_wait_prev();
            if (do_grad0) grad(0, map_idx(0, nk, pk), r3(0), r3(-1), r3(1));
            if (do_grad) grad(kG, gkGm, q3G, q3U, q3L);
            // ---- interfaces and update of plane kU ----
            if (kU >= k0 - 1 && kU <= k1 - 1) {
                const bool first = kU == k0 - 1; // only the -1/2 zeta flux of the chunk
                const int gkU = gkUm;
                const int sU = sUr * N2, sUp = sGr * N2, sUpp = sLr * N2;
                const int rU = (kU & 1), rP = ((kU + 1) & 1); // R1 tables
                const int mU = q3U, mP = q3G;       // metric tables
                // own points at plane kU
                const Pts L = pts(CK_RING(sU + c2));
                float2 WL[5];
                wvec(L, WL);
                float2 mL[9], jL = bc(0.0f);
                mets(mU, c1, mL, jL);
                float2 hx[5], hy[5], hz[5];
#pragma unroll
                for (int f = 0; f < 5; ++f) {
                    hx[f] = bc(0.0f);
                    hy[f] = bc(0.0f);
                    hz[f] = bc(0.0f);
                }
                const bool updA = !first && outA && kU >= k0, updB = !first && outB && kU >= k0;
                const int pU = gkU * plane;
                const int oA = CK_G(4, pU + ocolA, J.npts_pad), oB = CK_G(4, pU + ocolB, J.npts_pad);
                // zeta: R = the own column one plane up; R + 1 two planes up;
                // L - 1 one plane down (carried, or read on the first plane).
                // General form: evaluated between the eta and the xi flux in one
                // block (independent work for the scheduler to interleave; of the
                // orders measured, eta-zeta-xi ran fastest)
                auto zeta = [&]() {
                    const Pts R = pts(CK_RING(sUp + c2));
                    float2 WR[5], WRp[5];
                    wvec(R, WR);
                    if (ghost_hi) {
#pragma unroll
                        for (int f = 0; f < 5; ++f) WRp[f] = WL[f]; // W(nk) = W(nk - 2)
                    } else {
                        wof(CK_RING(sUpp + c2), WRp);
                    }
                    Side SL, SR;
                    side(2, rU, c1, SL);
                    side(2, rP, c1, SR);
                    float2 mR[9], jR;
                    mets(mP, c1, mR, jR);
                    iface<2>(FP, L, WL, mL, jL, R, WR, mR, jR, Wc, WRp, SL, SR, hz);
                };
                if (!first) {
                    // eta: R = (own second row, first row of the pair cell
                    // above); R + 1 = the pair cell above; L - 1 = (second row
                    // of the pair cell below, own first row)
                    {
                        const int up = tr + 1 < TR ? c1 + FX : c1; // the top thread row's second flux is not used
                        const Pts P1 = pts(CK_RING(sU + c2 + C2));
                        const Pts R = odd_pts(L, P1);
                        float2 WP1[5], WR[5], WLm[5], Wm[5];
                        wvec(P1, WP1);
                        wof(CK_RING(sU + c2 - C2), Wm);
#pragma unroll
                        for (int f = 0; f < 5; ++f) {
                            WR[f] = odd2(WL[f], WP1[f]);
                            WLm[f] = odd2(Wm[f], WL[f]);
                        }
                        Side SL, SU, SR;
                        side(1, rU, c1, SL);
                        side(1, rU, up, SU);
                        SR.mue = odd2(SL.mue, SU.mue);
                        SR.kap = odd2(SL.kap, SU.kap);
                        SR.nu = odd2(SL.nu, SU.nu);
                        SR.lb = odd2(SL.lb, SU.lb);
#pragma unroll
                        for (int b = 0; b < 2; ++b)
#pragma unroll
                            for (int f = 0; f < 4; ++f) SR.d[b][f] = odd2(SL.d[b][f], SU.d[b][f]);
                        float2 mA[9], jA, mR[9];
                        mets(mU, up, mA, jA);
#pragma unroll
                        for (int t = 0; t < 9; ++t) mR[t] = odd2(mL[t], mA[t]);
                        iface<1>(FP, L, WL, mL, jL, R, WR, mR, odd2(jL, jA), WLm, WP1, SL, SR, hy);
                    }
                    zeta();
                    // xi: R = the next column.  Lane 31's R has no R1 data: it pairs
                    // with its own R1 cell (an unused result), so that every lane
                    // runs the xi flux without a branch and the scheduler can
                    // interleave it with the eta flux
                    {
                        const int cR = tx <= FX - 2 ? c1 + 1 : c1;
                        const Pts R = pts(CK_RING(sU + c2 + 1));
                        float2 WR[5], WRp[5], WLm[5];
                        wvec(R, WR);
                        wof(CK_RING(sU + c2 + 2), WRp);
                        wof(CK_RING(sU + c2 - 1), WLm);
                        Side SL, SR;
                        side(0, rU, c1, SL);
                        side(0, rU, cR, SR);
                        float2 mR[9], jR;
                        mets(mU, cR, mR, jR);
                        iface<0>(FP, L, WL, mL, jL, R, WR, mR, jR, WLm, WRp, SL, SR, hx);
                    }
#pragma unroll
                    for (int f = 0; f < 5; ++f) S.SH[CK_SH(f * NT + tid)] = hy[f].y;
                } else {
                    zeta();
                }
                // the -1/2 xi flux from the lane below (all lanes of the warp
                // take part in the shuffle; the CTA-uniform `first` guards it)
                float2 hxm[5];
#pragma unroll
                for (int f = 0; f < 5; ++f) hxm[f] = bc(0.0f);
                if (!first) {
#pragma unroll
                    for (int f = 0; f < 5; ++f)
                        hxm[f] = f2(__shfl_up_sync(0xffffffffu, hx[f].x, 1), __shfl_up_sync(0xffffffffu, hx[f].y, 1));
                }
                __syncthreads(); // eta fluxes of the row below; the first plane's read of W below
                if (updA || updB) {
                    cp_async_wait_all(); // this thread's Q(0) copies
                    // residual R = sum over axes of flux(+1/2) - flux(-1/2); the
                    // -1/2 zeta flux from the previous plane, the -1/2 eta flux
                    // of the first row from the thread row below and of the
                    // second row from the own first
                    float2 Rs[5];
#pragma unroll
                    for (int f = 0; f < 5; ++f) {
                        const float hyb = tr > 0 ? S.SH[CK_SH(f * NT + tid - FX)] : 0.0f;
                        const float2 hym = f2(hyb, hy[f].x);
                        Rs[f] = add2(add2(sub2(hx[f], hxm[f]), sub2(hy[f], hym)), sub2(hz[f], hz_prev[f]));
                    }
                    if (rhs_only) {
                        if (updA) {
#pragma unroll
                            for (int f = 0; f < 5; ++f) J.rhs[f * fs + oA] = Rs[f].x;
                        }
                        if (updB) {
#pragma unroll
                            for (int f = 0; f < 5; ++f) J.rhs[f * fs + oB] = Rs[f].y;
                        }
                    } else {
                        // the stored state is unscaled: Q(l) = Q(0) - alpha dt J RHS
                        const float2 adtj = mul2(bc(adt), rjU);
                        if (updA) {
#pragma unroll
                            for (int f = 0; f < 5; ++f)
                                Qd[f * fs + oA] = fmaf(-adtj.x, Rs[f].x, S.QZ[CK_TAB(f * G_::QZN + zA, 5 * G_::QZN)]);
                        }
                        if (updB) {
#pragma unroll
                            for (int f = 0; f < 5; ++f)
                                Qd[f * fs + oB] = fmaf(-adtj.y, Rs[f].y, S.QZ[CK_TAB(f * G_::QZN + zB, 5 * G_::QZN)]);
                        }
                    }
                }
#pragma unroll
                for (int f = 0; f < 5; ++f) {
                    hz_prev[f] = hz[f];
                    Wc[f] = WL[f];
                }
            } else {
                __syncthreads(); // as in the branch above: this iteration's ring reads
                                 // precede the next iteration's loads into the freed slot
            }
            rjU = rjG; // plane kG is the next iteration's kU
            gkUc = gkGc;
            gkGc = gkLc;
            gkLc = map_idx(kL + 1, nk, pk);
            q3c = q3U;
        }
    }
    cp_async_wait_all();
    // a copy whose wait gave up may still be in flight into this CTA's
    // shared memory: its issuer waits for it (bounded) before exiting; if
    // that wait gives up too, the copy may land in the shared memory of the
    // next CTA on this SM, which is recorded as site 9 (it outranks site 8:
    // the state can no longer be trusted)
    if (pend && tid == 0 && !mbar_wait(S.MBAR, tpar, MBAR_WAIT_LIMIT)) {
        const JetDev<float> &J0 = jet_entry<ONE>(j1, jets, 0);
        if (J0.oob) atomicMax(J0.oob, 9ull << 48);
    }
}

#undef CK_G
#undef CK_RING
#undef CK_TAB
#undef CK_SH

// Paired static records of the general FP32 form (see FusedJet::mp).  The
// padding row of an odd nj is zero.
__global__ void __launch_bounds__(BLOCK) k_pack_pairs(const float *__restrict__ met, long long fs, int pitch,
                                                      int nj, int nk, float4 *__restrict__ mp)
{
    const int njp = (nj + 1) / 2;
    const long long total = (long long)nk * njp * pitch;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(t % pitch);
        const long long r = t / pitch;
        const int jp = (int)(r % njp), k = (int)(r / njp);
        float v[2][10];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = 2 * jp + h;
#pragma unroll
            for (int c = 0; c < 10; ++c) v[h][c] = 0.0f;
            if (j >= nj) continue;
            const float *m = met + ((long long)k * nj + j) * pitch + i;
#pragma unroll
            for (int c = 0; c < 9; ++c) v[h][c] = m[c * fs];
            v[h][9] = m[MET_JINV * fs];
        }
        float4 *out = mp + (r * 5) * pitch + i;
#pragma unroll
        for (int q = 0; q < 5; ++q)
            out[q * pitch] = make_float4(v[0][2 * q], v[1][2 * q], v[0][2 * q + 1], v[1][2 * q + 1]);
    }
}

void launch_pack_pairs(const float *met, long long fs, int pitch, int nj, int nk, float4 *mp, cudaStream_t st)
{
    const long long total = (long long)nk * ((nj + 1) / 2) * pitch;
    k_pack_pairs<<<(int)std::min<long long>((total + BLOCK - 1) / BLOCK, 65535LL * 4), BLOCK, 0, st>>>(
        met, fs, pitch, nj, nk, mp);
}

template <int TY> int fused_prepare()
{
    int rc = (int)cudaFuncSetAttribute(k_fused<TY, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)Geo<TY>::BYTES);
    if (!rc) rc = (int)cudaFuncSetAttribute(k_fused<TY, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)Geo<TY>::BYTES);
    return rc;
}

int fused_ctas_per_sm(int ty)
{
    int n = 0;
    const cudaError_t e =
        ty == 16 ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_fused<16, true>, FX * 8, Geo<16>::BYTES)
                 : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_fused<8, true>, FX * 4, Geo<8>::BYTES);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    return n > 0 ? n : 1;
}

template <int TY>
static void launch_one(const FusedLaunch &a, int grid, const JetDev<float> &ja, const FusedJet &fa, bool one, cudaStream_t st)
{
    const dim3 block(FX, TY / 2);
    const int lim = a.wait_limit < 0 ? MBAR_WAIT_LIMIT : a.wait_limit;
    if (one)
        k_fused<TY, true><<<grid, block, Geo<TY>::BYTES, st>>>(a.jets, a.fj, a.njets, a.items, a.tiles, a.src, a.dst,
                                                              a.stage, a.dt, a.rhs_only, a.balanced, lim, ja, fa);
    else
        k_fused<TY, false><<<grid, block, Geo<TY>::BYTES, st>>>(a.jets, a.fj, a.njets, a.items, a.tiles, a.src, a.dst,
                                                               a.stage, a.dt, a.rhs_only, a.balanced, lim, ja, fa);
}
void launch_fused(int ty, const FusedLaunch &a, int grid, const JetDev<float> *j1, const FusedJet *f1, cudaStream_t st)
{
    const bool one = a.njets == 1 && j1 && f1;
    static const JetDev<float> jz{};
    static const FusedJet fz{};
    const JetDev<float> &ja = one ? *j1 : jz;
    const FusedJet &fa = one ? *f1 : fz;
    if (ty == 16) launch_one<16>(a, grid, ja, fa, one, st);
    else launch_one<8>(a, grid, ja, fa, one, st);
}

template int fused_prepare<16>();
template int fused_prepare<8>();

} // namespace les
