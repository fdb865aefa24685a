// CUDA kernels of libles.so (sm_103a).
//
// Grid setup (metrics and static fields), boundary conditions, state
// conversion, time step, diagnostics, debug export and probe kernels.  The
// Runge-Kutta stage kernels are in les_stage.cu.
//   k_bc : all boundary faces (Sec. "Boundary Conditions"), after every stage
// All per-point kernels are persistent grid-stride loops over a block map that
// spans one or many jets (batched form); the per-point arithmetic does not
// depend on the map, so a jet gives the same bits alone or in a batch.
#include <cmath>
#include <algorithm>
#include <cstdint>

#include "les_bc.cuh"
#include "les_fp64.cuh"
#include "les_internal.cuh"
#include "les_sums.cuh"

namespace les {

// ---------------------------------------------------------------------------
// Small helpers
// ---------------------------------------------------------------------------

__device__ __forceinline__ int floordiv_i(int a, int n)
{
    int q = a / n;
    return (a % n != 0 && a < 0) ? q - 1 : q;
}

// ---------------------------------------------------------------------------
// Metric terms (FP64), Sec. "Transformation of Coordinates"
// ---------------------------------------------------------------------------

struct CoordGrid {
    const double *X[3];
    int n[3];
    int per[3];
    double shift[9];
};

// Coordinate c at lattice point q; on periodic axes q may be outside [0,n) and
// each crossed period adds the period shift (periodic extension of the grid).
__device__ double coord_at(const CoordGrid &G, int c, int q0, int q1, int q2)
{
    int q[3] = {q0, q1, q2};
    double off = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (G.per[a]) {
            int w = floordiv_i(q[a], G.n[a]);
            q[a] -= w * G.n[a];
            off += w * G.shift[3 * a + c];
        }
    }
    return G.X[c][((long long)q[2] * G.n[1] + q[1]) * G.n[0] + q[0]] + off;
}

// The metric stencils use explicitly rounded products and sums (no FMA
// contraction): on a Cartesian-product grid the cross terms are then exact
// zeros, as they are mathematically.  The boundary conditions branch on the
// sign of the normal velocity, and an edge point whose interior neighbour
// carries zero normal velocity must not see round-off residue there.

// d x_c / d xi^a at lattice point q.
__device__ double dcoord(const CoordGrid &G, int c, int a, const int q[3])
{
    // one-sided stencils are chosen from the wrapped index on periodic axes
    Stencil s = deriv_stencil(q[a], G.n[a], G.per[a]);
    double acc = 0.0;
    for (int t = 0; t < s.n; ++t) {
        int r[3] = {q[0], q[1], q[2]};
        r[a] += s.off[t];
        acc = __dadd_rn(acc, __dmul_rn(s.wgt[t], coord_at(G, c, r[0], r[1], r[2])));
    }
    return acc;
}

// D_outer [ x_c1 * D_inner x_c2 ] at lattice point q.
__device__ double dprod(const CoordGrid &G, int c1, int c2, int inner, int outer, const int q[3])
{
    Stencil s = deriv_stencil(q[outer], G.n[outer], G.per[outer]);
    double acc = 0.0;
    for (int t = 0; t < s.n; ++t) {
        int r[3] = {q[0], q[1], q[2]};
        r[outer] += s.off[t];
        double prod = __dmul_rn(coord_at(G, c1, r[0], r[1], r[2]), dcoord(G, c2, inner, r));
        acc = __dadd_rn(acc, __dmul_rn(s.wgt[t], prod));
    }
    return acc;
}

__global__ void __launch_bounds__(BLOCK) k_metrics(CoordGrid G, double *met, long long fs,
                                                   int pitch, double Cs)
{
    long long total = (long long)G.n[0] * G.n[1] * G.n[2];
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < total;
         p += (long long)gridDim.x * blockDim.x) {
        int q[3];
        q[0] = (int)(p % G.n[0]);
        q[1] = (int)((p / G.n[0]) % G.n[1]);
        q[2] = (int)(p / ((long long)G.n[0] * G.n[1]));
        long long o = ((long long)q[2] * G.n[1] + q[1]) * pitch + q[0];
        // conservative cofactors: J^-1 d xi^a / d x_c =
        //   D_b( x_c1 D_d x_c2 ) - D_d( x_c1 D_b x_c2 ),  (a,b,d), (c,c1,c2) cyclic
        for (int a = 0; a < 3; ++a) {
            int b = (a + 1) % 3, d = (a + 2) % 3;
            for (int c = 0; c < 3; ++c) {
                int c1 = (c + 1) % 3, c2 = (c + 2) % 3;
                met[(3 * a + c) * fs + o] = __dsub_rn(dprod(G, c1, c2, d, b, q), dprod(G, c1, c2, b, d, q));
            }
        }
        double t[3][3];
        for (int c = 0; c < 3; ++c)
            for (int a = 0; a < 3; ++a) t[c][a] = dcoord(G, c, a, q);
        // determinant of d(x,y,z)/d(xi,eta,zeta), as printed for 1/J
        double m0 = __dsub_rn(__dmul_rn(t[1][1], t[2][2]), __dmul_rn(t[1][2], t[2][1]));
        double m1 = __dsub_rn(__dmul_rn(t[1][0], t[2][2]), __dmul_rn(t[1][2], t[2][0]));
        double m2 = __dsub_rn(__dmul_rn(t[1][0], t[2][1]), __dmul_rn(t[1][1], t[2][0]));
        double jinv = __dadd_rn(__dsub_rn(__dmul_rn(t[0][0], m0), __dmul_rn(t[0][1], m1)),
                                __dmul_rn(t[0][2], m2));
        met[MET_JINV * fs + o] = jinv;
        double delta = cbrt(jinv); // filter width: cube root of the cell volume
        met[MET_CSD2 * fs + o] = (Cs * delta) * (Cs * delta);
    }
}

// General FP32 form: the 15 static fields the fused stage reads per point,
// packed into four consecutive float4 records so that the load phase fetches
// them with four vector loads from one array instead of fifteen.
// Separable form on a Cartesian-product grid: the spacing h_a(q) = d x_a /
// d xi^a along each axis, by the same FP64 stencils as the metrics (on such a
// grid the cofactors are products of these), stored with 1/h_a and h_a^(2/3)
// in FP32 for the fused stage.
__global__ void __launch_bounds__(BLOCK) k_sep_metrics(CoordGrid G, float4 *h1x, float4 *h1y, float4 *h1z)
{
    const int tot = G.n[0] + G.n[1] + G.n[2];
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < tot; t += gridDim.x * blockDim.x) {
        const int a = t < G.n[0] ? 0 : (t < G.n[0] + G.n[1] ? 1 : 2);
        const int qa = a == 0 ? t : (a == 1 ? t - G.n[0] : t - G.n[0] - G.n[1]);
        int q[3] = {0, 0, 0};
        q[a] = qa;
        const double h = dcoord(G, a, a, q);
        const double c = cbrt(h);
        float4 *out = a == 0 ? h1x : (a == 1 ? h1y : h1z);
        out[qa] = make_float4((float)h, (float)(1.0 / h), (float)(c * c), 0.0f);
    }
}

void launch_sep_metrics(const double *x, const double *y, const double *z, const int n[3], const int per[3],
                        const double shift[9], float4 *h1x, float4 *h1y, float4 *h1z, cudaStream_t st)
{
    CoordGrid G;
    G.X[0] = x;
    G.X[1] = y;
    G.X[2] = z;
    for (int a = 0; a < 3; ++a) {
        G.n[a] = n[a];
        G.per[a] = per[a];
    }
    for (int t = 0; t < 9; ++t) G.shift[t] = shift[t];
    const int tot = n[0] + n[1] + n[2];
    k_sep_metrics<<<(tot + BLOCK - 1) / BLOCK, BLOCK, 0, st>>>(G, h1x, h1y, h1z);
}

// Spacing tables of the product-grid FP64 stage (PROD_TABS per axis).
__global__ void __launch_bounds__(BLOCK) k_prod_tables(CoordGrid G, double *t0, double *t1, double *t2)
{
    const int tot = G.n[0] + G.n[1] + G.n[2];
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < tot; t += gridDim.x * blockDim.x) {
        const int a = t < G.n[0] ? 0 : (t < G.n[0] + G.n[1] ? 1 : 2);
        const int n = G.n[a], i = a == 0 ? t : (a == 1 ? t - G.n[0] : t - G.n[0] - G.n[1]);
        int q[3] = {0, 0, 0};
        q[a] = i;
        const double h = dcoord(G, a, a, q);
        q[a] = i + 1 < n ? i + 1 : (G.per[a] ? 0 : i);
        const double hb = 0.5 * (h + dcoord(G, a, a, q));
        double *o = (a == 0 ? t0 : (a == 1 ? t1 : t2)) + i;
        o[PT_H * n] = h;
        o[PT_RH * n] = 1.0 / h;
        o[PT_RH4 * n] = 0.25 / h;
        o[PT_RH6 * n] = 1.0 / (6.0 * h);
        o[PT_HB * n] = hb;
        o[PT_RHB * n] = 1.0 / hb;
        o[PT_RHB43 * n] = 4.0 / (3.0 * hb);
    }
}

void launch_prod_tables(const double *x, const double *y, const double *z, const int n[3], const int per[3],
                        const double shift[9], double *const tab[3], cudaStream_t st)
{
    CoordGrid G;
    G.X[0] = x;
    G.X[1] = y;
    G.X[2] = z;
    for (int a = 0; a < 3; ++a) {
        G.n[a] = n[a];
        G.per[a] = per[a];
    }
    for (int t = 0; t < 9; ++t) G.shift[t] = shift[t];
    const int tot = n[0] + n[1] + n[2];
    k_prod_tables<<<(tot + BLOCK - 1) / BLOCK, BLOCK, 0, st>>>(G, tab[0], tab[1], tab[2]);
}

// Static per-point fields derived from the metrics (FP64): J = 1/J^-1; per
// axis a the interface average of J^-1 towards the +a neighbour, its
// reciprocal, and the norm of metric row a.
__global__ void __launch_bounds__(BLOCK) k_static_fields(double *met, long long fs, int pitch, int ni,
                                                         int nj, int nk, int p0, int p1, int p2,
                                                         int iface_tables)
{
    const int n[3] = {ni, nj, nk};
    const int per[3] = {p0, p1, p2};
    const long long total = (long long)ni * nj * nk;
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < total;
         p += (long long)gridDim.x * blockDim.x) {
        int q[3];
        q[0] = (int)(p % ni);
        q[1] = (int)((p / ni) % nj);
        q[2] = (int)(p / ((long long)ni * nj));
        const long long o = ((long long)q[2] * nj + q[1]) * pitch + q[0];
        const double jinv = met[MET_JINV * fs + o];
        met[MET_J * fs + o] = 1.0 / state_scale(jinv);
        for (int a = 0; a < 3; ++a) {
            int r[3] = {q[0], q[1], q[2]};
            if (per[a]) r[a] = (q[a] + 1) % n[a];
            else if (q[a] + 1 < n[a]) r[a] = q[a] + 1;
            const long long oR = ((long long)r[2] * nj + r[1]) * pitch + r[0];
            const double jb = 0.5 * (jinv + met[MET_JINV * fs + oR]);
            // stored halved: the interface flux wants 1/2 (sum of the two
            // points' coefficients) times J^-1, so the 1/2 is taken here once
            met[(MET_JB + a) * fs + o] = 0.5 * jb;
            // an interface along the degenerate axis has no volume: zero weights
            met[(MET_RJB + a) * fs + o] = jb > 0.0 ? 1.0 / jb : 0.0;
            const double mx = met[(3 * a) * fs + o], my = met[(3 * a + 1) * fs + o],
                         mz = met[(3 * a + 2) * fs + o];
            met[(MET_NORM + a) * fs + o] = sqrt(mx * mx + my * my + mz * mz);
            if (iface_tables) {
                const double rjb = jb > 0.0 ? 1.0 / jb : 0.0;
                double A[9];
                for (int b = 0; b < 3; ++b)
                    for (int c = 0; c < 3; ++c) {
                        const double mc = 0.5 * (met[(3 * b + c) * fs + o] + met[(3 * b + c) * fs + oR]);
                        A[3 * b + c] = mc * rjb * (b == a ? 1.0 : 0.25);
                        met[(MET_A0 + 9 * a + 3 * b + c) * fs + o] = A[3 * b + c];
                    }
                for (int b = 0; b < 3; ++b)
                    met[(MET_K0 + 3 * a + b) * fs + o] =
                        A[3 * a] * A[3 * b] + A[3 * a + 1] * A[3 * b + 1] + A[3 * a + 2] * A[3 * b + 2];
            }
        }
    }
}

template <typename real>
__global__ void __launch_bounds__(BLOCK) k_convert_metrics(const double *met64, long long fs64,
                                                           real *met, long long fs, long long npad)
{
    for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < npad;
         p += (long long)gridDim.x * blockDim.x)
        for (int f = 0; f < NMET; ++f) met[f * fs + p] = (real)met64[f * fs64 + p];
}

// ---------------------------------------------------------------------------
// Boundary conditions (FP64 arithmetic on the stored state)
// ---------------------------------------------------------------------------

struct Prim64 {
    double rho, u[3], p;
};

__device__ __forceinline__ void cons_of(const Prim64 &s, double g, double Q[5])
{
    Q[0] = s.rho;
    Q[1] = s.rho * s.u[0];
    Q[2] = s.rho * s.u[1];
    Q[3] = s.rho * s.u[2];
    Q[4] = s.p / (g - 1.0) + 0.5 * s.rho * (s.u[0] * s.u[0] + s.u[1] * s.u[1] + s.u[2] * s.u[2]);
}

__device__ __forceinline__ Prim64 prim_of(const double Q[5], double g)
{
    Prim64 s;
    s.rho = Q[0];
    for (int c = 0; c < 3; ++c) s.u[c] = Q[1 + c] / Q[0];
    s.p = (g - 1.0) * (Q[4] - 0.5 * Q[0] * (s.u[0] * s.u[0] + s.u[1] * s.u[1] + s.u[2] * s.u[2]));
    return s;
}

// Centerline (Sec. "Centerline Boundary Condition") of a jet whose j- face is
// the axis: per (axial station i, conserved variable f) the mean over k of the
// unscaled ring j = 1, written, unscaled (state scale 1), to all azimuthal
// copies of the axis point (i, 0, k).  A block takes 32 stations of one
// variable (whole rows) and splits the ring over eight thread rows, whose
// partial sums are added in row order: the same order on every run.
constexpr int CL_ROWS = 8;
template <typename real>
__global__ void __launch_bounds__(32 * CL_ROWS) k_centerline(const JetDev<real> *__restrict__ jets, int dst)
{
    __shared__ double sh[CL_ROWS][32];
    const JetDev<real> &J = jets[blockIdx.z];
    if (J.bc[2] != LES_BC_CENTERLINE) return;
    const int i = blockIdx.x * 32 + threadIdx.x;
    const bool in = i < J.n[0];
    real *Q = J.q[dst] + blockIdx.y * J.fs;
    double sum = 0.0;
    for (int k = threadIdx.y; in && k < J.n[2]; k += CL_ROWS) {
        const long long o = lidx(J, i, 1, k);
        const double q = (double)Q[o];
        sum += sizeof(real) == sizeof(float) ? q : q * (double)J.met[MET_J * J.fs + o];
    }
    sh[threadIdx.y][threadIdx.x] = sum;
    __syncthreads();
    sum = 0.0;
    for (int r = 0; r < CL_ROWS; ++r) sum += sh[r][threadIdx.x];
    const real avg = (real)(sum / (double)J.n[2]);
    for (int k = threadIdx.y; in && k < J.n[2]; k += CL_ROWS) Q[lidx(J, i, 0, k)] = avg;
}

// All boundary faces of a time level (les_bc.cuh).
template <typename real, bool ONE>
__global__ void __launch_bounds__(BC_BLOCK) k_bc(const JetDev<real> *__restrict__ jets, BlockMap bm, int dst,
                                                 const long long *__restrict__ level_p,
                                                 const __grid_constant__ JetDev<real> j1)
{
    const int jet = ONE ? 0 : find_jet(bm, blockIdx.x);
    const JetDev<real> &J = ONE ? j1 : jets[jet];
    const int b0 = ONE ? 0 : bm.start[jet];
    long long F;
    real Q[5];
    if (!bc_point(J, (int)(blockIdx.x - b0) * BC_BLOCK + (int)threadIdx.x, *level_p, J.q[dst], F, Q)) return;
    for (int f = 0; f < 5; ++f) J.q[dst][f * J.fs + F] = Q[f];
}

// ---------------------------------------------------------------------------
// State conversion (host dense FP64 <-> device padded Qhat)
// ---------------------------------------------------------------------------

template <typename real>
__global__ void __launch_bounds__(BLOCK) k_set_state(const JetDev<real> *__restrict__ jets, int jet,
                                                     const double *__restrict__ in, int kind)
{
    const JetDev<real> &J = jets[jet];
    const long long N = (long long)J.n[0] * J.n[1] * J.n[2];
    for (long long lp = blockIdx.x * (long long)blockDim.x + threadIdx.x; lp < J.npts_pad;
         lp += (long long)gridDim.x * blockDim.x) {
        int q[3];
        if (!point_of(J, lp, q)) continue;
        long long dense = ((long long)q[2] * J.n[1] + q[1]) * J.n[0] + q[0];
        double v[5];
        for (int f = 0; f < 5; ++f) v[f] = in[f * N + dense];
        real *Q = J.q[0];
        if (kind == LES_STATE_RAW) {
            for (int f = 0; f < 5; ++f) Q[f * J.fs + lp] = (real)v[f];
            continue;
        }
        double Qc[5];
        if (kind == LES_STATE_PRIMITIVE) {
            Prim64 s;
            s.rho = v[0];
            s.u[0] = v[1];
            s.u[1] = v[2];
            s.u[2] = v[3];
            s.p = v[4];
            cons_of(s, J.gamma, Qc);
        } else {
            for (int f = 0; f < 5; ++f) Qc[f] = v[f];
        }
        const double jinv = stored_scale<real>(J.jinv64[lp]);
        for (int f = 0; f < 5; ++f) Q[f * J.fs + lp] = (real)(jinv * Qc[f]);
    }
}

template <typename real>
__global__ void __launch_bounds__(BLOCK) k_get_state(const JetDev<real> *__restrict__ jets, int jet,
                                                     double *__restrict__ out, int kind)
{
    const JetDev<real> &J = jets[jet];
    const long long N = (long long)J.n[0] * J.n[1] * J.n[2];
    for (long long lp = blockIdx.x * (long long)blockDim.x + threadIdx.x; lp < J.npts_pad;
         lp += (long long)gridDim.x * blockDim.x) {
        int q[3];
        if (!point_of(J, lp, q)) continue;
        long long dense = ((long long)q[2] * J.n[1] + q[1]) * J.n[0] + q[0];
        const real *Q = J.q[0];
        double v[5];
        for (int f = 0; f < 5; ++f) v[f] = (double)Q[f * J.fs + lp];
        if (kind != LES_STATE_RAW) {
            const double jinv = stored_scale<real>(J.jinv64[lp]);
            for (int f = 0; f < 5; ++f) v[f] /= jinv;
            if (kind == LES_STATE_PRIMITIVE) {
                Prim64 s = prim_of(v, J.gamma);
                v[0] = s.rho;
                v[1] = s.u[0];
                v[2] = s.u[1];
                v[3] = s.u[2];
                v[4] = s.p;
            }
        }
        for (int f = 0; f < 5; ++f) out[f * N + dense] = v[f];
    }
}

// ---------------------------------------------------------------------------
// Time step: max over points of lambda_xi + lambda_eta + lambda_zeta
// ---------------------------------------------------------------------------

template <typename real>
__global__ void __launch_bounds__(BLOCK) k_dt_max(const JetDev<real> *__restrict__ jets, BlockMap bm,
                                                  unsigned long long *maxbits)
{
    __shared__ double red[BLOCK];
    for (int vb = blockIdx.x; vb < bm.total; vb += gridDim.x) {
        int jet = find_jet(bm, vb);
        const JetDev<real> &J = jets[jet];
        long long lp = (long long)(vb - bm.start[jet]) * BLOCK + threadIdx.x;
        double val = 0.0;
        int q[3];
        if (lp < J.npts_pad && point_of(J, lp, q)) {
            const long long fs = J.fs;
            double rj = 1.0 / state_scale((double)J.met[MET_JINV * fs + lp]);
            double u = J.prim[P_U * fs + lp], v = J.prim[P_V * fs + lp], w = J.prim[P_W * fs + lp];
            double c = sqrt((double)J.prim[P_T * fs + lp]);
            for (int a = 0; a < 3; ++a) {
                double mx = J.met[(3 * a) * fs + lp], my = J.met[(3 * a + 1) * fs + lp],
                       mz = J.met[(3 * a + 2) * fs + lp];
                val += fabs((mx * u + my * v + mz * w) * rj) + c * sqrt(mx * mx + my * my + mz * mz) * rj;
            }
        }
        red[threadIdx.x] = val;
        __syncthreads();
        for (int s = BLOCK / 2; s > 0; s >>= 1) {
            if (threadIdx.x < s) red[threadIdx.x] = fmax(red[threadIdx.x], red[threadIdx.x + s]);
            __syncthreads();
        }
        if (threadIdx.x == 0)
            atomicMax(maxbits + jet, (unsigned long long)__double_as_longlong(red[0]));
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// Diagnostics: per-block partials in a fixed order, then one block combines
// (les_sums.cuh)
// ---------------------------------------------------------------------------

template <typename real>
__global__ void __launch_bounds__(SUM_BLOCK, SUM_BLOCKS_PER_SM) k_diag_partials(const JetDev<real> *__restrict__ jets,
                                                                int jet, double *part)
{
    const JetDev<real> &J = jets[jet];
    const long long n = J.npts_pad, fs = J.fs;
    const long long stride = (long long)gridDim.x * SUM_BLOCK;
    const long long p0 = blockIdx.x * (long long)SUM_BLOCK + threadIdx.x;
    const int pitch = J.pitch, ni = J.n[0];
    const real *Q = J.q[0], *R = J.rhs;
    const double *jinv = J.jinv64;
    // column of the thread's point, carried from point to point
    int i = (int)(p0 % pitch);
    const int di = (int)(stride % pitch);
    sum_block((n + stride - 1) / stride,
              [&](long long t, double q[5], double r[5]) {
                  const long long p = p0 + t * stride;
                  const bool in = p < n && i < ni; // padding columns hold nothing
                  i += di;
                  if (i >= pitch) i -= pitch;
                  // the Qhat the FP64 store holds (unscaled on a polar axis) from an
                  // unscaled FP32 store
                  const double qs = sizeof(real) == sizeof(float) && in ? state_scale(jinv[p]) : 1.0;
#pragma unroll
                  for (int f = 0; f < 5; ++f) {
                      q[f] = in ? (double)Q[f * fs + p] * qs : 0.0;
                      r[f] = in ? (double)R[f * fs + p] : 0.0;
                  }
              },
              part);
}

__global__ void __launch_bounds__(SUM_FINAL_THREADS) k_diag_final(const double *part, int nblocks, double *out)
{
    sum_final(part, nblocks, out);
}

// ---------------------------------------------------------------------------
// Debug point fields
// ---------------------------------------------------------------------------

template <typename real>
__global__ void __launch_bounds__(BLOCK) k_debug_field(const JetDev<real> *__restrict__ jets, int jet,
                                                       int field, double *out)
{
    const JetDev<real> &J = jets[jet];
    const long long N = (long long)J.n[0] * J.n[1] * J.n[2];
    for (long long lp = blockIdx.x * (long long)blockDim.x + threadIdx.x; lp < J.npts_pad;
         lp += (long long)gridDim.x * blockDim.x) {
        int q[3];
        if (!point_of(J, lp, q)) continue;
        long long dense = ((long long)q[2] * J.n[1] + q[1]) * J.n[0] + q[0];
        const long long fs = J.fs;
        switch (field) {
        case LES_FIELD_MU_SGS: out[dense] = J.grad[G_MUSGS * fs + lp]; break;
        case LES_FIELD_MU: out[dense] = J.prim[P_MU * fs + lp]; break;
        case LES_FIELD_P: out[dense] = J.prim[P_P * fs + lp]; break;
        case LES_FIELD_T: out[dense] = J.prim[P_T * fs + lp]; break;
        case LES_FIELD_LAMBDA_XI: out[dense] = J.prim[P_LXI * fs + lp]; break;
        case LES_FIELD_LAMBDA_ETA: out[dense] = J.prim[P_LETA * fs + lp]; break;
        case LES_FIELD_LAMBDA_ZETA: out[dense] = J.prim[P_LZETA * fs + lp]; break;
        case DBG_RHS:
            for (int f = 0; f < NF; ++f) out[f * N + dense] = J.rhs[f * fs + lp];
            break;
        default:
            if (field >= DBG_MET0 && field < DBG_MET0 + 9) out[dense] = J.met[(field - DBG_MET0) * fs + lp];
            else if (field == DBG_MET0 + 9) out[dense] = J.jinv64[lp];
            break;
        }
    }
}

// ---------------------------------------------------------------------------
// Surface probe: trilinear interpolation of rho, u, v, w, p
// ---------------------------------------------------------------------------

template <typename real>
__global__ void __launch_bounds__(BLOCK) k_probe(const JetDev<real> *__restrict__ jets,
                                                 const int *__restrict__ cell,
                                                 const double *__restrict__ wts, int npts, int every,
                                                 const long long *__restrict__ level_p,
                                                 const long long *__restrict__ base_p, real *out,
                                                 int capacity)
{
    const long long level = *level_p;
    if (level % every != 0) return;
    const long long frame = level / every - *base_p - 1;
    if (frame < 0) return;
    const JetDev<real> &J = jets[0];
    const long long fs = J.fs;
    real *o = out + (frame % capacity) * 5LL * npts;
    const double g = J.gamma;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < npts; s += gridDim.x * blockDim.x) {
        int lo[3] = {cell[3 * s], cell[3 * s + 1], cell[3 * s + 2]};
        double t[3] = {wts[3 * s], wts[3 * s + 1], wts[3 * s + 2]};
        double acc[5] = {0, 0, 0, 0, 0};
        for (int c = 0; c < 8; ++c) {
            int r[3];
            double wgt = 1.0;
            for (int a = 0; a < 3; ++a) {
                int up = (c >> a) & 1;
                r[a] = lo[a] + up;
                wgt *= up ? t[a] : 1.0 - t[a];
            }
            long long p = lidx(J, r[0], r[1], r[2]);
            double jinv = stored_scale<real>(J.jinv64[p]);
            double Q[5];
            for (int f = 0; f < 5; ++f) Q[f] = (double)J.q[0][f * fs + p] / jinv;
            Prim64 pr = prim_of(Q, g);
            acc[0] += wgt * pr.rho;
            acc[1] += wgt * pr.u[0];
            acc[2] += wgt * pr.u[1];
            acc[3] += wgt * pr.u[2];
            acc[4] += wgt * pr.p;
        }
        for (int f = 0; f < 5; ++f) o[(long long)f * npts + s] = (real)acc[f];
    }
}

__global__ void k_step_advance(long long *level) { *level += 1; }

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------

static int grid_for(long long work, int cap = 152 * 16)
{
    long long g = (work + BLOCK - 1) / BLOCK;
    if (g < 1) g = 1;
    if (g > cap) g = cap;
    return (int)g;
}

template <typename real>
void Launch<real>::metrics(const double *x, const double *y, const double *z, int ni, int nj, int nk,
                           const int per[3], const double shift[9], double *met64, long long fs64,
                           int pitch, double Cs, cudaStream_t st)
{
    CoordGrid G;
    G.X[0] = x;
    G.X[1] = y;
    G.X[2] = z;
    G.n[0] = ni;
    G.n[1] = nj;
    G.n[2] = nk;
    for (int a = 0; a < 3; ++a) G.per[a] = per[a];
    for (int t = 0; t < 9; ++t) G.shift[t] = shift[t];
    k_metrics<<<grid_for((long long)ni * nj * nk), BLOCK, 0, st>>>(G, met64, fs64, pitch, Cs);
}

template <typename real>
void Launch<real>::static_fields(double *met64, long long fs64, int pitch, const int n[3],
                                 const int per[3], int iface_tables, cudaStream_t st)
{
    k_static_fields<<<grid_for((long long)n[0] * n[1] * n[2]), BLOCK, 0, st>>>(
        met64, fs64, pitch, n[0], n[1], n[2], per[0], per[1], per[2], iface_tables);
}

template <typename real>
void Launch<real>::convert_metrics(const double *met64, long long fs64, real *met, long long fs,
                                   long long npad, cudaStream_t st)
{
    k_convert_metrics<real><<<grid_for(npad), BLOCK, 0, st>>>(met64, fs64, met, fs, npad);
}

template <typename real>
void launch_centerline(const JetDev<real> *jets, int njets, int max_ni, int dst, cudaStream_t st)
{
    k_centerline<real><<<dim3((max_ni + 31) / 32, 5, njets), dim3(32, CL_ROWS), 0, st>>>(jets, dst);
}
template void launch_centerline<float>(const JetDev<float> *, int, int, int, cudaStream_t);
template void launch_centerline<double>(const JetDev<double> *, int, int, int, cudaStream_t);

int bc_blocks(const int n[3], const int per[3])
{
    long long pts = 0;
    for (int a = 0; a < 3; ++a)
        if (!per[a]) pts += 2LL * n[(a + 1) % 3] * n[(a + 2) % 3];
    return (int)((pts + BC_BLOCK - 1) / BC_BLOCK);
}

template <typename real>
void Launch<real>::bc(const JetDev<real> *jets, BlockMap bm, int dst, const long long *level, const JetDev<real> *j1,
                      cudaStream_t st)
{
    if (bm.total <= 0) return;
    if (j1) k_bc<real, true><<<bm.total, BC_BLOCK, 0, st>>>(jets, bm, dst, level, *j1);
    else k_bc<real, false><<<bm.total, BC_BLOCK, 0, st>>>(jets, bm, dst, level, JetDev<real>{});
}

template <typename real>
void Launch<real>::set_state(const JetDev<real> *jets, int jet, const double *in, int kind,
                             long long npad, cudaStream_t st)
{
    k_set_state<real><<<grid_for(npad), BLOCK, 0, st>>>(jets, jet, in, kind);
}

template <typename real>
void Launch<real>::get_state(const JetDev<real> *jets, int jet, double *out, int kind,
                             long long npad, cudaStream_t st)
{
    k_get_state<real><<<grid_for(npad), BLOCK, 0, st>>>(jets, jet, out, kind);
}

template <typename real>
void Launch<real>::dt_max(const JetDev<real> *jets, BlockMap bm, unsigned long long *maxbits,
                          int grid, cudaStream_t st)
{
    k_dt_max<real><<<grid, BLOCK, 0, st>>>(jets, bm, maxbits);
}

template <typename real>
void Launch<real>::diag_partials(const JetDev<real> *jets, int jet, double *partials, int nblocks,
                                 cudaStream_t st)
{
    k_diag_partials<real><<<nblocks, SUM_BLOCK, 0, st>>>(jets, jet, partials);
}

template <typename real>
void Launch<real>::debug_field(const JetDev<real> *jets, int jet, int field, double *out,
                               long long npad, cudaStream_t st)
{
    k_debug_field<real><<<grid_for(npad), BLOCK, 0, st>>>(jets, jet, field, out);
}

template <typename real>
void Launch<real>::probe(const JetDev<real> *jets, const int *cell, const double *wts, int npts,
                         int every, const long long *level, const long long *base, real *out,
                         int capacity, cudaStream_t st)
{
    k_probe<real><<<grid_for(npts, 1024), BLOCK, 0, st>>>(jets, cell, wts, npts, every, level, base,
                                                          out, capacity);
}

void launch_diag_final(const double *partials, int nblocks, double *out, cudaStream_t st)
{
    k_diag_final<<<1, SUM_FINAL_THREADS, 0, st>>>(partials, nblocks, out);
}

void launch_step_advance(long long *level, cudaStream_t st) { k_step_advance<<<1, 1, 0, st>>>(level); }

template struct Launch<float>;
template struct Launch<double>;

} // namespace les
