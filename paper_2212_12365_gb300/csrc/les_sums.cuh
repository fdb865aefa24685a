// Residual / conservation sums of a state: per block, then over the blocks.
// Shared by les_get_diagnostics (les_kernels.cu) and les_diag_sums_noalloc
// (les_noalloc.cu), which differ only in how a point's values are read.
//
// What bounds it.  A point is 10 values (80 bytes FP64), so memory sets the
// floor: 170 us for 14.2 M points at 6.66 TB/s.  A Neumaier sum per value is
// six FP64 operations, and GB300's FP64 pipe (2 lanes per clock and SM) takes
// 1.4 ms for five of them per point: the pipe, not memory, bounded the sums.
// So the conservation sums run on the integer pipe: every lane keeps a 128-bit
// fixed-point sum (SumFx) whose least bit sits 2^-52 below the last bit of the
// largest value its warp has met; the additions are exact above that bit, and
// what reaches below it is kept in a double of its own, so that large values may
// cancel without a trace (a test holds the sums to the exactly rounded ones).
// The sums of squares stay in FP64 (one multiply-add per value).
// Measured: 14,155,776 points 2098 -> 219 us (5.2 TB/s), 1,000,000 908 -> 49, one
// point 27 -> 22; les_get_diagnostics of a 192x128x72 FP32 jet about 1.0 ms less
// per call (most of it the final pass).
#pragma once

#include "les_internal.cuh"

namespace les {

constexpr int SUM_PART = 17;      // partial results per block, field-major [f][block]:
                                  // 0 max |RHS_rho|, 1..5 sum RHS^2, 6..10 sum Qhat,
                                  // 11..15 its compensation, 16 non-finite count
constexpr int SUM_BLOCK = 256;    // threads per block
// One wave: two blocks on each of 152 SMs, whose threads keep the next point's
// ten values in flight in registers (123 of them).  Four blocks without that
// read-ahead took 319 us at 14,155,776 points, three with it 287 (spills), two 250.
constexpr int SUM_BLOCKS_PER_SM = 2;
constexpr int SUM_MAX_BLOCKS = 152 * SUM_BLOCKS_PER_SM;

__device__ __forceinline__ void neumaier_add(double &s, double &c, double v)
{
    const double t = s + v;
    if (fabs(s) >= fabs(v)) c += (s - t) + v;
    else c += (v - t) + s;
    s = t;
}

// x 2^k for any k the sums meet (|k| < 2100): two exact halves
__device__ __forceinline__ double scale2(double x, int k)
{
    const int h = k >> 1;
    return ldexp(ldexp(x, h), k - h);
}

// Fixed-point sum of doubles: value = (hi 2^64 + lo) 2^(base - 1075) + the
// lane's tail, the base (a biased exponent) the same for all lanes of a warp.
// Bits below the base go to the tail, a double: its terms are below one unit of
// the base each, so that its rounding is some 2^-150 of the largest value.
struct SumFx {
    long long hi = 0;
    unsigned long long lo = 0;
    int base = -4096; // below every exponent: the first value sets it

    static constexpr int GUARD = 52; // bits kept below the largest value's last bit
    static constexpr int TOP = 55;   // largest shift: 53 + 55 bits, 19 bits left for the count and sign

    // Add a finite v; every lane of the warp calls it together.
    __device__ __forceinline__ void add(double v, double *tail)
    {
        const long long b = __double_as_longlong(v);
        const int ef = (int)((unsigned long long)b >> 52) & 0x7ff;
        int e = max(ef, 1); // subnormals have no hidden bit and exponent 1
        long long m = (b & 0xFFFFFFFFFFFFFll) | (ef ? 1ll << 52 : 0ll);
        // a value above the window, or reaching below it (seldom: within 2^-52 of
        // the largest value so far there is none)
        if (__any_sync(0xffffffffu, m != 0 && (unsigned)(e - base) > (unsigned)TOP)) {
            const int top = __reduce_max_sync(0xffffffffu, m != 0 ? e : -4096);
            if (top - base > TOP) rebase(top - GUARD, tail);
            const int d = base - e;
            if (m != 0 && d > 0) { // the lowest d bits
                const long long low = d > 52 ? ~0ll : (1ll << d) - 1;
                *tail += v - (d > 52 ? 0.0 : __longlong_as_double(b & ~low));
                m = d > 52 ? 0 : m >> d;
                e = base;
            }
        }
        m = b < 0 ? -m : m;
        const int l = (e - base) & 63;
        const unsigned long long al = (unsigned long long)m << l;
        const long long ah = (m >> 1) >> (63 - l);
        lo += al;
        hi += ah + (lo < al ? 1 : 0);
    }
    // Move the least bit up; what falls off goes to the tail.
    __device__ __forceinline__ void rebase(int nb, double *tail)
    {
        const int d = nb - base;
        if ((hi | (long long)lo) != 0) {
            const int u = base - 1075;
            if (d >= 120) { // less than a few units of the new base
                *tail += scale2((double)hi, u + 64) + scale2((double)lo, u);
                hi = 0;
                lo = 0;
            } else if (d >= 64) {
                *tail += scale2((double)(hi & ((1ll << (d - 64)) - 1)), u + 64) + scale2((double)lo, u);
                lo = (unsigned long long)(hi >> (d - 64));
                hi >>= 63;
            } else {
                *tail += scale2((double)(lo & ((1ull << d) - 1)), u);
                lo = (lo >> d) | ((unsigned long long)hi << (64 - d));
                hi >>= d;
            }
        }
        base = nb;
    }
    // Sum of the warp's lanes, in every lane.
    __device__ __forceinline__ void warp_reduce()
    {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const long long h = __shfl_xor_sync(0xffffffffu, hi, o);
            const unsigned long long l = __shfl_xor_sync(0xffffffffu, lo, o);
            lo += l;
            hi += h + (lo < l ? 1 : 0);
        }
    }
    // The sum as s + c: three 43-bit pieces, each a double exactly.
    __device__ __forceinline__ void value(double &s, double &c) const
    {
        const long long p2 = hi >> 22;
        const long long p1 = ((hi & 0x3FFFFFll) << 21) | (long long)(lo >> 43);
        const long long p0 = (long long)(lo & 0x7FFFFFFFFFFull);
        s = c = 0.0;
        neumaier_add(s, c, scale2((double)p2, base - 1075 + 86));
        neumaier_add(s, c, scale2((double)p1, base - 1075 + 43));
        neumaier_add(s, c, scale2((double)p0, base - 1075));
    }
};

// Partial sums of one block over `steps` strided points per thread.  load(t,
// q, r) fills the point's Qhat and residual values (zeros beyond the end);
// t counts points per thread, the same number for every lane of a warp.
template <typename Load> __device__ __forceinline__ void sum_block(long long steps, const Load &load, double *part)
{
    SumFx fx[5];
    // the lanes' tails: in shared memory, since they are seldom touched and the
    // registers hold the next point
    __shared__ double tails[5][SUM_BLOCK];
#pragma unroll
    for (int f = 0; f < 5; ++f) tails[f][threadIdx.x] = 0.0;
    double l2[5] = {0, 0, 0, 0, 0};
    long long mxb = 0; // |RHS_rho| as its bits, which order as integers (NaN ignored, as fmax does)
    int bad = 0;
    unsigned nf = 0; // fields that met a non-finite value: their sum is NaN
    double qn[5], rn[5];
    load(0, qn, rn);
    for (long long t = 0; t < steps; ++t) {
        double q[5], r[5];
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            q[f] = qn[f];
            r[f] = rn[f];
        }
        if (t + 1 < steps) load(t + 1, qn, rn); // in flight while this point is added
        const long long ab = __double_as_longlong(r[0]) & 0x7fffffffffffffffll;
        mxb = max(mxb, ab > 0x7ff0000000000000ll ? 0ll : ab);
#pragma unroll
        for (int f = 0; f < 5; ++f) {
            const bool vf = (((unsigned)__double2hiint(q[f]) >> 20) & 0x7ffu) != 0x7ffu;
            const bool rf = (((unsigned)__double2hiint(r[f]) >> 20) & 0x7ffu) != 0x7ffu;
            bad += !(vf && rf);
            if (!vf) nf |= 1u << f;
            l2[f] = fma(r[f], r[f], l2[f]);
            fx[f].add(vf ? q[f] : 0.0, &tails[f][threadIdx.x]);
        }
    }
    __shared__ double sh[SUM_PART][SUM_BLOCK / 32];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double mx = __longlong_as_double(mxb);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
#pragma unroll
        for (int f = 0; f < 5; ++f) l2[f] += __shfl_xor_sync(0xffffffffu, l2[f], o);
    }
    bad = __reduce_add_sync(0xffffffffu, bad);
    nf = __reduce_or_sync(0xffffffffu, nf);
    // lane f takes field f, so that the five conversions run at once (one after the
    // other, each in its own lane, they took 11 us of every call: one point 33 us)
    SumFx own;
    double l2o = 0.0, tail = 0.0;
#pragma unroll
    for (int f = 0; f < 5; ++f) {
        fx[f].warp_reduce();
        double t = tails[f][threadIdx.x];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == f) {
            own = fx[f];
            l2o = l2[f];
            tail = t;
        }
    }
    if (lane < 5) {
        double s, c;
        own.value(s, c);
        sh[1 + lane][w] = l2o;
        sh[6 + lane][w] = (nf >> lane) & 1 ? __longlong_as_double(0x7ff8000000000000ll) : s;
        sh[11 + lane][w] = c + tail;
    }
    if (lane == 0) {
        sh[0][w] = mx;
        sh[16][w] = (double)bad;
    }
    __syncthreads();
    const int f = threadIdx.x;
    const long long nb = gridDim.x;
    if (f < 6 || f == 16) {
        double a = sh[f][0];
        for (int i = 1; i < SUM_BLOCK / 32; ++i) a = f == 0 ? fmax(a, sh[f][i]) : a + sh[f][i];
        part[f * nb + blockIdx.x] = a;
    } else if (f < 11) {
        double s = sh[f][0], c = sh[f + 5][0];
        for (int i = 1; i < SUM_BLOCK / 32; ++i) {
            neumaier_add(s, c, sh[f][i]);
            c += sh[f + 5][i];
        }
        part[f * nb + blockIdx.x] = s;
        part[(f + 5) * nb + blockIdx.x] = c;
    }
}

// Blocks of a reduction over n points: four points per thread at least.
inline int sum_blocks(long long n)
{
    const long long b = (n + 4 * SUM_BLOCK - 1) / (4 * SUM_BLOCK);
    return (int)(b < 1 ? 1 : (b > SUM_MAX_BLOCKS ? SUM_MAX_BLOCKS : b));
}

// Combine nb blocks' partials into out[12] (see les_diag_sums_noalloc); a
// warp per result, lanes over the blocks, then a fixed shuffle tree.  (One
// thread walking 17 x 608 values in turn took 0.25 ms.)
constexpr int SUM_FINAL_THREADS = 12 * 32;
__device__ __forceinline__ void sum_final(const double *__restrict__ part, int nb, double *out)
{
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool pair = w >= 6 && w < 11;
    const double *p = part + (long long)(w == 11 ? 16 : w) * nb;
    double a = 0.0, c = 0.0;
    for (int b = lane; b < nb; b += 32) {
        if (w == 0) a = fmax(a, p[b]);
        else if (pair) {
            neumaier_add(a, c, p[b]);
            c += p[5LL * nb + b];
        } else a += p[b];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double a2 = __shfl_xor_sync(0xffffffffu, a, o), c2 = __shfl_xor_sync(0xffffffffu, c, o);
        if (w == 0) a = fmax(a, a2);
        else if (pair) {
            neumaier_add(a, c, a2);
            c += c2;
        } else a += a2;
    }
    if (lane == 0) out[w] = w >= 1 && w <= 5 ? sqrt(a) : (pair ? a + c : a);
}

} // namespace les
