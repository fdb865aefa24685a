// les_fwh: far-field acoustic pressure from the probe surface's frames by the
// Ffowcs Williams-Hawkings equation, the acoustic post-processing the paper's
// probe surface feeds (its Introduction and Concluding Remarks name FW-H for
// the far field but give no formulation).  Adopted formulation: Farassat's
// Formulation 1A (NASA TM-2007-214853) with the permeable-surface source
// terms of di Francescantonio (J. Sound Vib. 202, 1997), for a surface at rest
// in a medium at rest:
//     Q = rho u.n,   L_i = (p - p0) n_i + rho u_i u.n,
//     4 pi p'(x, t) = sum_panels A [ dQ/dtau / r + (dL_r/dtau) / (c0 r) + L_r / r^2 ]
// at the retarded time tau = t - r / c0, r = |x - y|, L_r = L.(x - y)/r.
// Discretisation: d/dtau by second-order central differences between frames
// (one-sided three-point at the first and last frame), retarded values by
// linear interpolation between the two frames around tau.
//
// Kernels, run over batches of panels whose source records, and whose records per
// microphone, take at most 256 MB each (1024 panels' source records if those take
// more):
//   k_fwh_check : distances' range per microphone and the largest spread over
//                 a microphone group (the input checks and the window length)
//   k_fwh_src   : per panel and frame L, dQ/dtau and dL/dtau as two float4,
//                 panel-major
//   k_fwh_geo   : per panel and microphone the weights and the emission-time
//                 offset
//   k_fwh_obs_win (staged) or k_fwh_obs (direct, when a window of frames would
//                 not fit): partial sums per (panel chunk, microphone, time)
//   k_fwh_sum   : the chunks added in chunk order
// Every sum has a fixed order, so the result is the same on every run.
#include <cmath>
#include <string>
#include <vector>

#include "les_fp64.cuh"
#include "les_fwh_plan.h"
#include "les_internal.cuh"
#include "les_pair.cuh"

namespace les {

namespace {

constexpr int FWH_SUB = 256; // panels per shared-memory sub-chunk

// 32-byte store (16-byte halves a, b) to a 32-byte aligned address
__device__ __forceinline__ void store8(float4 *p, const float4 &a, const float4 &b)
{
    asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(a.x), "f"(a.y), "f"(a.z),
                 "f"(a.w), "f"(b.x), "f"(b.y), "f"(b.z), "f"(b.w)
                 : "memory");
}

// Q and L of a panel at one frame, and their combinations over frames, in the
// arithmetic of the ring's precision: FP64 for a double ring; for a float ring
// pairs of floats (an unevaluated sum h + l, the error-free transformations of
// Knuth and Dekker), which carry about 48 bits.  The results are rounded to
// FP32, so both give the same records up to rare ties, and the pairs run on the
// FP32 pipe, 64 times as wide as the FP64 pipe that bounded this pass (98,304
// panels x 1024 frames: 7.6 -> 1.3 ms; now 3.7 TB/s of reads and writes).
// Per (panel j of the batch, frame m): src[(j*N + m)*2] = (L_x, L_y, L_z,
// dQ/dtau), src[(j*N + m)*2 + 1] = (dL_x/dtau, dL_y/dtau, dL_z/dtau, 0).  One
// thread per panel and segment of SEG frames marches its frames with the
// values of three consecutive frames in registers, so each is formed once
// (twice at the segment's ends).  Reads are whole rows of panels; a record is
// one 32-byte store, and a thread's consecutive records fill lines in L2.
constexpr int FWH_SEG = 64;
template <typename real>
__global__ void __launch_bounds__(128) k_fwh_src(const real *__restrict__ ring, int first, int cap, int npts, int j0,
                                                 int nb, int N, const double *__restrict__ nrm, double p0, double rdt2,
                                                 float4 *__restrict__ src)
{
    typedef Num<real> A;
    typedef typename A::T T;
    // blocks: panels fastest, then segments (a grid's x alone holds any number)
    const int pb = (nb + blockDim.x - 1) / blockDim.x, seg = blockIdx.x / pb;
    const int jl = (blockIdx.x - seg * pb) * blockDim.x + threadIdx.x;
    if (jl >= nb) return;
    const int j = j0 + jl;
    const T n[3] = {A::of(nrm[j]), A::of(nrm[npts + j]), A::of(nrm[2 * npts + j])};
    const T mp0 = A::of(-p0), r2 = A::of(rdt2);
    const int m0 = seg * FWH_SEG, m1 = min(N, m0 + FWH_SEG);
    float4 *o = src + (long long)jl * N * 2;
    struct F {
        T v[4]; // L_x, L_y, L_z, Q
    };
    auto frame = [&](int m) {
        int slot = first + m;
        slot -= slot >= cap ? cap : 0;
        const real *w = ring + (long long)slot * 5 * npts + j;
        const real rho = w[0], u[3] = {w[npts], w[2LL * npts], w[3LL * npts]}, p = w[4LL * npts];
        T one;
        if constexpr (sizeof(real) == sizeof(float)) one = T{p, 0.0f};
        else one = p;
        const T dp = A::add(one, mp0);
        const T un = A::add(A::add(A::mul(u[0], n[0]), A::mul(u[1], n[1])), A::mul(u[2], n[2]));
        F f;
        f.v[3] = A::mul(rho, un);
        for (int i = 0; i < 3; ++i) f.v[i] = A::add(A::mulp(dp, n[i]), A::mul(u[i], f.v[3]));
        return f;
    };
    auto put = [&](int m, const F &at, const T d[4]) {
        store8(o + 2 * m,
               make_float4(A::out(at.v[0]), A::out(at.v[1]), A::out(at.v[2]), A::out(A::mulp(d[3], r2))),
               make_float4(A::out(A::mulp(d[0], r2)), A::out(A::mulp(d[1], r2)), A::out(A::mulp(d[2], r2)), 0.0f));
    };
    // one-sided three-point differences at the first and last frame:
    // +-(-3 a + 4 b - c) for the frames a, b, c from the end inwards
    auto put_end = [&](int m, const F &a, const F &b, const F &c, real sign) {
        T d[4];
        for (int i = 0; i < 4; ++i)
            d[i] = A::add(A::add(A::mul(real(-3) * sign, a.v[i]), A::mul(real(4) * sign, b.v[i])),
                          A::mul(-sign, c.v[i]));
        put(m, a, d);
    };
    F a = frame(max(m0 - 1, 0)), b = frame(m0), c;
    if (m0 == 0) {
        b = frame(1);
        c = frame(2);
        put_end(0, a, b, c, real(1));
    } else {
        c = frame(min(m0 + 1, N - 1));
    }
    for (int m = max(m0, 1); m < m1 && m < N - 1; ++m) { // a, b, c: frames m - 1, m, m + 1
        T d[4];
        for (int i = 0; i < 4; ++i) d[i] = A::sub(c.v[i], a.v[i]);
        put(m, b, d);
        a = b;
        b = c;
        if (m + 2 < N && m + 1 < m1) c = frame(m + 2);
    }
    if (m1 == N) put_end(N - 1, frame(N - 1), frame(N - 2), frame(N - 3), real(-1));
}

// Order-preserving bits of a non-negative double for the atomic minima / maxima
__device__ __forceinline__ unsigned long long ubits(double v) { return (unsigned long long)__double_as_longlong(v); }

// (On the host, one core took 15 ms for the 6.3 M distances of 98,304 panels
// and 64 microphones; here 0.04 ms.)
// Squared distances: minimum and maximum per microphone (lim[o], lim[nobs +
// o]), and the largest spread of a panel's distances over a group of MG
// microphones (lim[2 nobs]), as bits of non-negative doubles.
__global__ void __launch_bounds__(256) k_fwh_check(int npts, const double *__restrict__ xyz,
                                                   const double *__restrict__ obs, int nobs, int MG,
                                                   unsigned long long *__restrict__ lim)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int jc = min(j, npts - 1); // the last panel again: changes no extremum
    const double x = xyz[jc], y = xyz[npts + jc], z = xyz[2 * npts + jc];
    double spread = 0.0;
    for (int o0 = 0; o0 < nobs; o0 += MG) {
        unsigned long long gmin = ~0ull, gmax = 0;
        for (int o = o0; o < min(nobs, o0 + MG); ++o) {
            const double dx = obs[o] - x, dy = obs[nobs + o] - y, dz = obs[2 * nobs + o] - z;
            const unsigned long long r2 = ubits(dx * dx + dy * dy + dz * dz);
            gmin = min(gmin, r2);
            gmax = max(gmax, r2);
            unsigned long long lo = r2, hi = r2;
#pragma unroll
            for (int s = 16; s > 0; s >>= 1) {
                lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, s));
                hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, s));
            }
            if ((threadIdx.x & 31) == 0) {
                atomicMin(lim + o, lo);
                atomicMax(lim + nobs + o, hi);
            }
        }
        spread = fmax(spread, sqrt(__longlong_as_double((long long)gmax)) - sqrt(__longlong_as_double((long long)gmin)));
    }
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) spread = fmax(spread, __shfl_xor_sync(0xffffffffu, spread, s));
    if ((threadIdx.x & 31) == 0) atomicMax(lim + 2 * nobs, ubits(spread));
}

// Per (panel j of the batch, microphone o) two float4: A/(4 pi r^2) times the
// unit direction to the microphone, A/(4 pi r); r/c0, the fraction and
// the integer part of the emission-frame offset B0 - r/(c0 dtau).
__global__ void __launch_bounds__(256) k_fwh_geo(int npts, int j0, int nb, const double *__restrict__ xyz,
                                                 const double *__restrict__ area, const double *__restrict__ obs,
                                                 int nobs, double B0, double rc0, double rdtau,
                                                 float4 *__restrict__ geo)
{
    const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (t >= (long long)nb * nobs) return;
    const int jl = (int)(t / nobs), o = (int)(t - (long long)jl * nobs), j = j0 + jl;
    const double dx = obs[o] - xyz[j], dy = obs[nobs + o] - xyz[npts + j], dz = obs[2 * nobs + o] - xyz[2 * npts + j];
    const double r2 = dx * dx + dy * dy + dz * dz, ir = rsqrt64(r2), r = r2 * ir;
    const double gw = area[j] * (1.0 / (4.0 * M_PI)) * ir, gl = gw * ir * ir;
    const double e = B0 - r * rc0 * rdtau, ef = floor(e);
    geo[2 * t] = make_float4((float)(gl * dx), (float)(gl * dy), (float)(gl * dz), (float)gw);
    geo[2 * t + 1] = make_float4((float)(r * rc0), (float)(e - ef), __int_as_float((int)ef), 0.0f);
}

__global__ void __launch_bounds__(FWH_T) k_fwh_obs(const float4 *__restrict__ src, int npts, int N,
                                                   const double *__restrict__ xyz, const double *__restrict__ area,
                                                   const double *__restrict__ obs, int nobs, double t0, double dt_obs,
                                                   int nt, double dtau, double c0, int chunk, int j00, int nb,
                                                   double *__restrict__ part)
{
    __shared__ float4 geo[FWH_SUB]; // unit direction to the observer, A/(4 pi r)
    __shared__ float fr[FWH_SUB];   // fractional part of the panel's frame offset
    __shared__ float irs[FWH_SUB];  // 1/r
    __shared__ int mb[FWH_SUB];     // integer part of the panel's frame offset
    const int k = blockIdx.x * FWH_T + threadIdx.x;
    const int o = blockIdx.y, c = blockIdx.z;
    const double ox = obs[o], oy = obs[nobs + o], oz = obs[2 * nobs + o];
    // The emission time of observer time t_k at distance r, in frames, is
    // s = t_k / dtau - r / (c0 dtau).  Split exactly in FP64 into a CTA base B
    // (an integer), the thread's small offset t_k/dtau - B (FP32) and the
    // panel's offset B - r/(c0 dtau) = M + f (integer M, fraction f in FP32),
    // so that the per-panel work of a thread is FP32 and integer arithmetic.
    const double B = floor((t0 + (double)(blockIdx.x * FWH_T) * dt_obs) / dtau);
    const float skl = (float)((t0 + (double)k * dt_obs) / dtau - B);
    const float rc0 = (float)(1.0 / c0);
    const int j0 = c * chunk, j1 = min(nb, j0 + chunk);
    double acc = 0.0;
    for (int jb = j0; jb < j1; jb += FWH_SUB) {
        const int nsub = min(FWH_SUB, j1 - jb);
        __syncthreads(); // the previous sub-chunk's geometry is no longer read
        if (threadIdx.x < nsub) {
            const int j = j00 + jb + threadIdx.x;
            const double dx = ox - xyz[j], dy = oy - xyz[npts + j], dz = oz - xyz[2 * npts + j];
            const double r = sqrt(dx * dx + dy * dy + dz * dz), ir = 1.0 / r;
            geo[threadIdx.x] = make_float4((float)(dx * ir), (float)(dy * ir), (float)(dz * ir),
                                           (float)(area[j] * ir / (4.0 * M_PI)));
            const double e = B - r / (c0 * dtau);
            const double ef = floor(e);
            mb[threadIdx.x] = (int)ef;
            fr[threadIdx.x] = (float)(e - ef);
            irs[threadIdx.x] = (float)ir;
        }
        __syncthreads();
        if (k < nt) {
            float sum = 0.0f, comp = 0.0f; // compensated sum over the sub-chunk
            for (int q = 0; q < nsub; ++q) {
                const float4 g = geo[q];
                const float s = skl + fr[q];
                const float fl = floorf(s);
                int m = mb[q] + (int)fl;
                m = m < 0 ? 0 : (m > N - 2 ? N - 2 : m);
                const float w = s - fl;
                const float4 *p = src + ((long long)(jb + q) * N + m) * 2;
                const float4 a0 = p[0], b0 = p[1], a1 = p[2], b1 = p[3];
                const float Lx = fmaf(w, a1.x - a0.x, a0.x), Ly = fmaf(w, a1.y - a0.y, a0.y),
                            Lz = fmaf(w, a1.z - a0.z, a0.z), dQ = fmaf(w, a1.w - a0.w, a0.w);
                const float dLx = fmaf(w, b1.x - b0.x, b0.x), dLy = fmaf(w, b1.y - b0.y, b0.y),
                            dLz = fmaf(w, b1.z - b0.z, b0.z);
                const float Lr = fmaf(Lx, g.x, fmaf(Ly, g.y, Lz * g.z));
                const float dLr = fmaf(dLx, g.x, fmaf(dLy, g.y, dLz * g.z));
                // A/(4 pi r) [dQ + dL_r / c0 + L_r / r]
                const float v = g.w * fmaf(Lr, irs[q], fmaf(dLr, rc0, dQ));
                const float y = v - comp;
                const float tsum = sum + y;
                comp = (tsum - sum) - y;
                sum = tsum;
            }
            acc += (double)sum;
        }
    }
    if (k < nt) {
        double *p = part + ((long long)c * nobs + o) * nt + k;
        *p = j00 > 0 ? *p + acc : acc; // batches in order
    }
}

// Observer pass, staged.  A CTA takes a group of up to 16 microphones, a block
// of T observer times and a panel chunk; thread t stands for the two times t
// and t + half, whose arithmetic runs as paired FP32.  The integrand is linear
// in the source record, so it is formed once per (panel, microphone, frame)
// and interpolated afterwards: per panel the CTA
//   1. projects the window of frames that its times and microphones need:
//      V[o][m] = gl.(L + (r/c0) dL/dtau) + gw dQ/dtau, seven multiply-adds per
//      frame and microphone (microphones in pairs), a frame's record read once
//      from global memory for all sixteen, V in shared memory;
//   2. interpolates V at each time's emission frame and adds it to the
//      compensated sum of its microphone, in registers over the whole chunk.
// V is double buffered: one barrier per panel; the next panel's records arrive
// by cp.async during the interpolation.  When every evaluation read its two
// frames (64 bytes) from shared memory and projected both, the pass ran at the
// shared-memory wavefront limit (66 %); now an evaluation reads 8 bytes and the
// pass is bound by issue and barriers at 16 warps per SM (issue 48 %, shared
// memory 54 %).  98,304 panels, 64 microphones, 512 times: 11.4 -> 4.7 ms.
__device__ __forceinline__ float2 fadd2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 fsub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a); }
__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 dup2(float v) { return make_float2(v, v); }
__device__ __forceinline__ void fwh_cp16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

// Staged geometry of a panel.
struct FwhGeo {
    float4 pair[FWH_MG / 2][3]; // microphones 2p, 2p+1: (glx, glx', gly, gly') (glz, glz', gw, gw') (q, q', -, -)
    float4 off[FWH_MG];         // fraction (twice), offset in the window (int bits), -
    unsigned mask[32];          // microphone pairs that read the window's entries 32 w .. 32 w + 31
    int base, pad[3];           // frame of the window's first entry
};
static_assert(sizeof(FwhGeo) == FWH_GEO_BYTES, "fwh_win_smem counts it");

// FULL: every group has sixteen microphones.
template <int NTH, bool FULL>
__global__ void __launch_bounds__(NTH, 512 / NTH) k_fwh_obs_win(const float4 *__restrict__ src, int nb, int N,
                                                      const float4 *__restrict__ geo, int nobs, int MG, double t0,
                                                      double dt_obs, int nt, int T, double dtau, int chunk, int W,
                                                      int span, int add, double *__restrict__ part)
{
    extern __shared__ __align__(16) float fwh_sm[];
    const int rows = FULL ? FWH_MG : (MG + 1) / 2 * 2; // fwh_rows
    float *V = fwh_sm;                             // [2][rows][W]
    float4 *RA = (float4 *)(V + 2 * rows * W);     // [W] records of the next panel: (L, dQ/dtau)
    float4 *RB = RA + W;                           // [W]: dL/dtau
    FwhGeo *G = (FwhGeo *)(RB + W);                // [FWH_PB]
    const int tid = threadIdx.x;
    // blocks: microphone groups fastest, then time blocks; panel chunks along y
    const int ng = (nobs + MG - 1) / MG, tb = blockIdx.x / ng;
    const int o0 = (blockIdx.x - tb * ng) * MG, mgt = FULL ? FWH_MG : min(MG, nobs - o0);
    const int k0 = tb * T, half = (min(T, nt - k0) + 1) / 2;
    const int c = blockIdx.y;
    // s(k) = t_k/dtau - B with B = floor of the block's first, an integer; split
    // into an integer and a fraction (a float of the whole offset would be good
    // to 3e-5 frames only)
    const double B0 = floor(t0 / dtau), B = floor((t0 + (double)k0 * dt_obs) / dtau);
    const int dB = (int)(B - B0);
    const double sx = (t0 + (double)(k0 + tid) * dt_obs) / dtau - B, sy = (t0 + (double)(k0 + tid + half) * dt_obs) / dtau - B;
    const int kx = (int)floor(sx) - 0x4B400000, ky = (int)floor(sy) - 0x4B400000; // less the bits of 1.5 2^23
    const float2 skl = make_float2((float)(sx - floor(sx)), (float)(sy - floor(sy)));
    float2 sum[FWH_MG], cmp[FWH_MG]; // cmp: the compensation, added
#pragma unroll
    for (int o = 0; o < FWH_MG; ++o) sum[o] = cmp[o] = dup2(0.0f);
    const int j0 = c * chunk, j1 = min(nb, j0 + chunk);
    // start the copies of a panel's records; a thread copies the entries it projects
    auto fetch = [&](int j, int fb) {
        const float4 *sp = src + (long long)j * N * 2;
        for (int fi = tid; fi < W; fi += NTH) {
            const int m = min(max(fb + fi, 0), N - 1);
            fwh_cp16(RA + fi, sp + 2 * m);
            fwh_cp16(RB + fi, sp + 2 * m + 1);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    float *Vb = V, *Vn = V + rows * W;
    for (int jb = j0; jb < j1; jb += FWH_PB) {
        const int np = min(FWH_PB, j1 - jb);
        __syncthreads(); // the previous panels' geometry is no longer read
        for (int i = tid; i < np * FWH_MG; i += NTH) {
            const int g = i / FWH_MG, o = i % FWH_MG;
            // an absent microphone of a group repeats the last one (unused)
            const float4 *r = geo + 2 * ((long long)(jb + g) * nobs + o0 + min(o, mgt - 1));
            const float4 a = r[0], b = r[1];
            float *q = (float *)G[g].pair[o / 2] + (o & 1);
            q[0] = a.x;
            q[2] = a.y;
            q[4] = a.z;
            q[6] = a.w;
            q[8] = b.x;
            G[g].off[o] = make_float4(b.y, b.y, b.z, 0.0f);
        }
        __syncthreads();
        for (int g = tid >> 5; g < np; g += NTH / 32) { // a warp per panel: window base, offsets, masks
            const int l = tid & 31;
            const int m = l < FWH_MG ? __float_as_int(G[g].off[l].z) : 0x7fffffff;
            const int lo = __reduce_min_sync(0xffffffffu, m);
            const int off = m - lo + 1;
            if (l < FWH_MG) G[g].off[l].z = __int_as_float(off);
            if (l == 0) G[g].base = lo + dB - 1;
            // microphone l reads the entries off - 1 .. off + span; lane l stands for entries 32 l .. 32 l + 31
            unsigned mk = 0;
#pragma unroll
            for (int o = 0; o < FWH_MG; ++o) {
                const int f = __shfl_sync(0xffffffffu, off, o);
                if (32 * l + 31 >= f - 1 && 32 * l <= f + span) mk |= 1u << (o / 2);
            }
            G[g].mask[l] = mk;
        }
        __syncthreads();
        fetch(jb, G[0].base);
        for (int g = 0; g < np; ++g) {
            asm volatile("cp.async.wait_all;\n" ::: "memory"); // own entries
            for (int fi = tid; fi < W; fi += NTH) {
                const float4 a = RA[fi], b = RB[fi];
                const unsigned mk = G[g].mask[fi >> 5];
                const float2 Lx = dup2(a.x), Ly = dup2(a.y), Lz = dup2(a.z), dQ = dup2(a.w);
                const float2 dx = dup2(b.x), dy = dup2(b.y), dz = dup2(b.z);
#pragma unroll
                for (int p = 0; p < FWH_MG / 2; ++p) {
                    if (!FULL && 2 * p >= mgt) break;
                    if (!((mk >> p) & 1u)) continue;
                    const float4 *r = G[g].pair[p];
                    const float4 r0 = r[0], r1 = r[1];
                    const float2 q = *(const float2 *)(r + 2);
                    float2 v = __fmul2_rn(make_float2(r1.z, r1.w), dQ);
                    v = ffma2(make_float2(r0.x, r0.y), ffma2(q, dx, Lx), v);
                    v = ffma2(make_float2(r0.z, r0.w), ffma2(q, dy, Ly), v);
                    v = ffma2(make_float2(r1.x, r1.y), ffma2(q, dz, Lz), v);
                    Vb[2 * p * W + fi] = v.x;
                    Vb[(2 * p + 1) * W + fi] = v.y;
                }
            }
            if (g + 1 < np) fetch(jb + g + 1, G[g + 1].base); // in flight during the interpolation
            __syncthreads();
            if (tid < half) {
                // r = 1.5 2^23 + floor(s), by an addition rounded down
                const float2 magic = dup2(12582912.0f), unmagic = dup2(-12582912.0f);
                const unsigned last = (unsigned)(W - 2);
#pragma unroll
                for (int o = 0; o < FWH_MG; ++o) {
                    if (!FULL && o >= mgt) break;
                    const float4 gd = G[g].off[o];
                    const float2 s = fadd2(skl, make_float2(gd.x, gd.y));
                    const float2 r = __fadd2_rd(s, magic);
                    const float2 w = fsub2(s, fadd2(r, unmagic));
                    const int off = __float_as_int(gd.z);
                    const unsigned ix = min((unsigned)(__float_as_int(r.x) + off + kx), last);
                    const unsigned iy = min((unsigned)(__float_as_int(r.y) + off + ky), last);
                    const float *Vo = Vb + o * W;
                    const float2 v0 = make_float2(Vo[ix], Vo[iy]), v1 = make_float2(Vo[ix + 1], Vo[iy + 1]);
                    const float2 v = ffma2(w, fsub2(v1, v0), v0);
                    const float2 y = fadd2(v, cmp[o]);
                    const float2 t = fadd2(sum[o], y);
                    cmp[o] = fsub2(y, fsub2(t, sum[o]));
                    sum[o] = t;
                }
            }
            float *sw = Vb;
            Vb = Vn;
            Vn = sw;
        }
    }
    if (tid < half) {
#pragma unroll
        for (int o = 0; o < FWH_MG; ++o) {
            if (o >= mgt) break;
            double *p = part + ((long long)c * nobs + o0 + o) * nt + k0 + tid;
            const double a = (double)sum[o].x + (double)cmp[o].x, b = (double)sum[o].y + (double)cmp[o].y;
            *p = add ? *p + a : a; // batches in order
            if (k0 + tid + half < min(nt, k0 + T)) p[half] = add ? p[half] + b : b;
        }
    }
}

template <int NTH, bool FULL>
static int launch_obs_win(dim3 grid, size_t smem, cudaStream_t st, const float4 *src, int nb, int N, const float4 *geo,
                          int nobs, int MG, double t0, double dt_obs, int nt, int T, double dtau, int chunk, int W,
                          int span, int add, double *part)
{
    // always the same limit: it belongs to the kernel, and calls from other host
    // threads may need another size between this line and the launch
    if (cudaFuncSetAttribute(k_fwh_obs_win<NTH, FULL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)FWH_WIN_SMEM) != cudaSuccess)
        return 1;
    k_fwh_obs_win<NTH, FULL><<<grid, NTH, smem, st>>>(src, nb, N, geo, nobs, MG, t0, dt_obs, nt, T, dtau, chunk, W,
                                                      span, add, part);
    return 0;
}

__global__ void k_fwh_sum(const double *__restrict__ part, int nchunk, long long n, double *__restrict__ out)
{
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    double s = 0.0;
    for (int c = 0; c < nchunk; ++c) s += part[(long long)c * n + i];
    out[i] = s;
}

} // namespace

} // namespace les

using namespace les;

extern "C" int les_fwh(const void *ring, int precision, int capacity, int64_t frames_written, int npts,
                       const double *xyz, const double *nrm, const double *area, double dtau, double p0, double c0,
                       int nobs, const double *obs, double t0, double dt_obs, int nt, double *p_out, void *stream,
                       double *ms_out)
{
    auto bad = [](const char *msg) {
        set_call_error(msg);
        return LES_ERR_ARG;
    };
    set_call_error("");
    if (!ring || !xyz || !nrm || !area || !obs || !p_out) return bad("null pointer");
    if (precision != LES_FP64 && precision != LES_FP32 && precision != LES_FP32_SEPARABLE)
        return bad("unknown precision");
    if (npts < 1 || nobs < 1 || nt < 1 || capacity < 1) return bad("npts, nobs, nt and capacity must be >= 1");
    const int N = (int)std::min<int64_t>(frames_written, capacity);
    if (frames_written < 3 || N < 3) return bad("at least three frames are needed");
    if (!(dtau > 0) || !(c0 > 0) || !(dt_obs >= 0)) return bad("dtau and c0 must be > 0, dt_obs >= 0");
    const int first = (int)((frames_written - N) % capacity);
    cudaStream_t st = (cudaStream_t)stream;
    int dev = 0, nsm = 152;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return LES_ERR_CUDA;
    const int MG = fwh_group(nobs);
    const size_t n_out = (size_t)nobs * nt;
    double *d_geo = nullptr;   // panel geometry, microphones, distance limits
    char *d_work = nullptr;    // batch records, partial sums, result
    auto release = [&]() {
        if (d_geo) cudaFree(d_geo);
        if (d_work) cudaFree(d_work);
    };
    auto oom = [&]() {
        cudaGetLastError();
        release();
        set_call_error("device allocation failed");
        return LES_ERR_OOM;
    };
    auto cuda_failed = [&]() {
        cudaGetLastError();
        release();
        set_call_error("CUDA failure in the FW-H evaluation");
        return LES_ERR_CUDA;
    };
    const size_t geo_doubles = (size_t)npts * 7 + (size_t)nobs * 3, lim_n = 2 * (size_t)nobs + 1;
    if (cudaMalloc(&d_geo, (geo_doubles + lim_n) * sizeof(double)) != cudaSuccess) return oom();
    double *d_xyz = d_geo, *d_nrm = d_geo + 3 * (size_t)npts, *d_area = d_geo + 6 * (size_t)npts,
           *d_obs = d_geo + 7 * (size_t)npts;
    unsigned long long *d_lim = (unsigned long long *)(d_geo + geo_doubles);
    std::vector<double> lim(lim_n);
    if (cudaMemcpyAsync(d_xyz, xyz, 3 * (size_t)npts * 8, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(d_nrm, nrm, 3 * (size_t)npts * 8, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(d_area, area, (size_t)npts * 8, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemcpyAsync(d_obs, obs, 3 * (size_t)nobs * 8, cudaMemcpyHostToDevice, st) != cudaSuccess ||
        cudaMemsetAsync(d_lim, 0xff, (size_t)nobs * 8, st) != cudaSuccess ||
        cudaMemsetAsync(d_lim + nobs, 0, ((size_t)nobs + 1) * 8, st) != cudaSuccess)
        return cuda_failed();
    k_fwh_check<<<(npts + 255) / 256, 256, 0, st>>>(npts, d_xyz, d_obs, nobs, MG, d_lim);
    if (cudaGetLastError() != cudaSuccess ||
        cudaMemcpyAsync(lim.data(), d_lim, lim_n * 8, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return cuda_failed();
    // every emission time of every panel must lie within the frames
    const double tau_max = (N - 1) * dtau, t1 = t0 + (nt - 1) * dt_obs;
    for (int o = 0; o < nobs; ++o) {
        const double rmin = std::sqrt(lim[o]), rmax = std::sqrt(lim[nobs + o]);
        const char *msg = nullptr;
        if (!(rmin > 0) || !(rmax > 0)) msg = "an observer coincides with a panel";
        else if (t0 - rmax / c0 < 0.0 || t1 - rmin / c0 > tau_max)
            msg = "an emission time t - r/c0 falls outside the frames: need t0 >= r_max/c0 and "
                  "t0 + (nt-1) dt_obs - r_min/c0 <= (frames - 1) dtau";
        if (msg) {
            release();
            return bad(msg);
        }
    }
    const FwhPlan P = fwh_plan(npts, N, nobs, nt, dt_obs, dtau, c0, lim[2 * nobs], nsm);
    const int NB = P.NB, nchunk = P.nchunk;
    if (cudaMalloc(&d_work, P.scratch()) != cudaSuccess) return oom();
    float4 *d_src = (float4 *)d_work, *d_rec = (float4 *)(d_work + P.b_src);
    double *d_part = (double *)(d_work + P.b_src + P.b_rec), *d_out = d_part + n_out * nchunk;
    cudaEvent_t ev[3] = {nullptr, nullptr, nullptr};
    int rc = LES_OK;
    if (ms_out) {
        ms_out[0] = ms_out[1] = 0.0;
        for (auto &e : ev)
            if (cudaEventCreate(&e) != cudaSuccess) rc = LES_ERR_CUDA;
    }
    const double rdt2 = 1.0 / (2.0 * dtau);
    for (int j0 = 0; j0 < npts && rc == LES_OK; j0 += NB) {
        const int nb = std::min(NB, npts - j0);
        // the same chunk count in every batch; a short last batch has shorter chunks
        const int chunk = (nb + nchunk - 1) / nchunk;
        if (ms_out) cudaEventRecord(ev[0], st);
        const int gs = (nb + 127) / 128 * ((N + FWH_SEG - 1) / FWH_SEG);
        if (precision == LES_FP64)
            k_fwh_src<double><<<gs, 128, 0, st>>>((const double *)ring, first, capacity, npts, j0, nb, N, d_nrm, p0,
                                                  rdt2, d_src);
        else
            k_fwh_src<float><<<gs, 128, 0, st>>>((const float *)ring, first, capacity, npts, j0, nb, N, d_nrm, p0, rdt2,
                                                 d_src);
        if (ms_out) cudaEventRecord(ev[1], st);
        if (P.staged) {
            k_fwh_geo<<<(int)(((long long)nb * nobs + 255) / 256), 256, 0, st>>>(
                npts, j0, nb, d_xyz, d_area, d_obs, nobs, std::floor(t0 / dtau), 1.0 / c0, 1.0 / dtau, d_rec);
            const dim3 go(P.ngroups * P.tblocks, nchunk);
            const bool full = P.MG == FWH_MG && nobs % FWH_MG == 0;
            const auto launch = P.nth == 64    ? (full ? launch_obs_win<64, true> : launch_obs_win<64, false>)
                                : P.nth == 128 ? (full ? launch_obs_win<128, true> : launch_obs_win<128, false>)
                                               : (full ? launch_obs_win<256, true> : launch_obs_win<256, false>);
            const int bad_attr = launch(go, fwh_win_smem(P.W, fwh_rows(P.MG)), st, d_src, nb, N, d_rec, nobs, P.MG, t0,
                                        dt_obs, nt, P.T, dtau, chunk, P.W, P.span, j0 > 0, d_part);
            if (bad_attr) rc = LES_ERR_CUDA;
        } else {
            k_fwh_obs<<<dim3(P.tblocks, nobs, nchunk), FWH_T, 0, st>>>(d_src, npts, N, d_xyz, d_area, d_obs, nobs, t0,
                                                                      dt_obs, nt, dtau, c0, chunk, j0, nb, d_part);
        }
        if (cudaGetLastError() != cudaSuccess) rc = LES_ERR_CUDA;
        if (ms_out && rc == LES_OK) {
            cudaEventRecord(ev[2], st);
            float a = 0.0f, b = 0.0f;
            if (cudaEventSynchronize(ev[2]) != cudaSuccess) rc = LES_ERR_CUDA;
            cudaEventElapsedTime(&a, ev[0], ev[1]);
            cudaEventElapsedTime(&b, ev[1], ev[2]);
            ms_out[0] += a;
            ms_out[1] += b;
        }
    }
    if (rc == LES_OK) {
        k_fwh_sum<<<(int)((n_out + 255) / 256), 256, 0, st>>>(d_part, nchunk, (long long)n_out, d_out);
        if (cudaGetLastError() != cudaSuccess ||
            cudaMemcpyAsync(p_out, d_out, n_out * 8, cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            rc = LES_ERR_CUDA;
    }
    for (auto &e : ev)
        if (e) cudaEventDestroy(e);
    if (rc != LES_OK) {
        cudaGetLastError();
        set_call_error("CUDA failure in the FW-H evaluation");
    }
    release();
    return rc;
}
