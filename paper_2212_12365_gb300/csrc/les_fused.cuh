// Pieces shared by the two fused FP32 stage kernels (les_fused.cu, the general
// form; les_fused_prod.cu, the product-grid form): paired arithmetic,
// asynchronous copies, the bounded staging wait, and the work cursor.
#pragma once

#include "les_internal.cuh"

namespace les {

namespace {

constexpr int FX = 32; // threads (grid columns) along i

__constant__ float c_alpha_f[5] = {0.25f, 1.0f / 6.0f, 0.375f, 0.5f, 1.0f};

// ---------------------------------------------------------------------------
// Paired FP32 arithmetic (two rows per register pair)
// ---------------------------------------------------------------------------

__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }
__device__ __forceinline__ float2 bc(float s) { return make_float2(s, s); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b (one instruction; a multiply-add with -1 needs that constant in a register pair)
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;"
        : "=l"(r)
        : "l"(*reinterpret_cast<unsigned long long *>(&a)), "l"(*reinterpret_cast<unsigned long long *>(&b)));
    return *reinterpret_cast<float2 *>(&r);
}
__device__ __forceinline__ float2 lo2(const float4 &v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4 &v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float4 cat4(float2 a, float2 b) { return make_float4(a.x, a.y, b.x, b.y); }
// the pair (second lane of a, first lane of b): the +eta neighbours of a
// thread's two rows
__device__ __forceinline__ float2 odd2(float2 a, float2 b) { return make_float2(a.y, b.x); }
__device__ __forceinline__ float2 max2(float2 a, float2 b) { return make_float2(fmaxf(a.x, b.x), fmaxf(a.y, b.y)); }
// Hardware reciprocal and reciprocal square root (within 1.5 and 2.5 ulp;
// arguments normal numbers): the plain instructions, which flush subnormal
// numbers.  17 pairs per thread and plane in the general kernel: polar 400x150x60
// 276.6 us per stage with the calls that keep them, 265.1 with these.
__device__ __forceinline__ float rcpa(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqa(float x)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float2 rcp2(float2 a) { return f2(rcpa(a.x), rcpa(a.y)); }
// x^(-1/3), x > 0: 2^(-log2(x)/3) by the hardware functions (about 2^-20) and one
// Newton step of y^-3 = x, y + y (1 - x y^3)/3, in FP32 with FMAs (below 2 ulp)
__device__ __forceinline__ float2 rcbrt2(float2 x)
{
    float2 l, y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l.x) : "f"(x.x));
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(l.y) : "f"(x.y));
    l = mul2(l, bc(-1.0f / 3.0f));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(l.x));
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(l.y));
    const float2 r = fma2(mul2(mul2(y, y), y), mul2(x, bc(-1.0f)), bc(1.0f));
    return fma2(mul2(y, bc(1.0f / 3.0f)), r, y);
}
// x^1/2 = x rsqrt(x) for x > 0, and for x >= 0 (0 -> 0: no strain; a spectral
// radius vanishes on the axis of a polar mesh)
__device__ __forceinline__ float2 sqrtp2(float2 x) { return mul2(x, f2(rsqa(x.x), rsqa(x.y))); }
__device__ __forceinline__ float2 sqrt2(float2 x)
{
    return mul2(x, f2(rsqa(fmaxf(x.x, 1.17549435e-38f)), rsqa(fmaxf(x.y, 1.17549435e-38f))));
}

// Asynchronous 16-byte global -> shared copy, not kept in L1 (completes
// without the issuing thread waiting; cp_async_wait_prev() waits for all of
// this thread's groups but the most recent one).
__device__ __forceinline__ unsigned smem_u32_(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32_(dst)), "l"(src) : "memory");
}
// 4-byte variant (scattered Q(0) values)
__device__ __forceinline__ void cp_async4(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_u32_(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_prev() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Index of a tile cell along an axis: wrapped on a periodic axis; on a
// non-periodic one the mirror image about the end point (-g, 2(n-1) - g),
// clamped into the axis for cells further out (those feed no result).
__device__ __forceinline__ int map_idx(int g, int n, int per)
{
    if (per) {
        const int h = g < 0 ? g + n : (g >= n ? g - n : g);
        return (unsigned)h < (unsigned)n ? h : wrapi(g, n);
    }
    const int m = g < 0 ? -g : (g > n - 1 ? 2 * (n - 1) - g : g);
    return m < 0 ? 0 : (m > n - 1 ? n - 1 : m);
}

// TMA staging: an mbarrier with one arrival (the issuing thread's, carrying
// the expected byte count) completed by the copy.
__device__ __forceinline__ unsigned smem_u32(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(unsigned long long *bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(bar)) : "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); // visible to the copy engine
}
// 4-D tiled copy (x, y, z, field) of the tensor map's box into shared memory;
// x must be a multiple of 4 elements (16 bytes); other coordinates may lie
// outside the tensor (zero fill).
__device__ __forceinline__ void tma_box_load(float *dst, const CUtensorMap *map, int x, int y, int z,
                                             unsigned long long *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                 " [%0], [%1, {%2, %3, %4, %5}], [%6];\n" ::"r"(smem_u32(dst)),
                 "l"(reinterpret_cast<unsigned long long>(map)), "r"(x), "r"(y), "r"(z), "r"(0), "r"(smem_u32(bar))
                 : "memory");
}
// Wait for the phase of the given parity, polling at most `limit` times
// (false: gave up).
constexpr int MBAR_WAIT_LIMIT = 1 << 22;
__device__ __forceinline__ bool mbar_wait(unsigned long long *bar, unsigned parity, int limit)
{
    for (int it = 0; it < limit; ++it) {
        unsigned done;
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                     " selp.u32 %0, 1, 0, p;\n}\n"
                     : "=r"(done)
                     : "r"(smem_u32(bar)), "r"(parity)
                     : "memory");
        if (done) return true;
    }
    return false;
}

// The jet's table entries: in the single-jet form (ONE) the kernel
// parameters, whose fields the compiler reads from the parameter bank
// (warp-uniform operands, no memory loads in the plane loop); else the
// device tables.
template <bool ONE, typename T> __device__ __forceinline__ const T &jet_entry(const T &one, const T *tab, int j)
{
    if constexpr (ONE) return one;
    else return tab[j];
}

// The jet's constants: the kernel parameter (ONE), else the item's copy in
// shared memory (read with broadcast loads instead of global loads).
template <bool ONE>
__device__ __forceinline__ const FusedParams &jet_params(const FusedParams &param, const float *staged)
{
    if constexpr (ONE) return param;
    else return *reinterpret_cast<const FusedParams *>(staged);
}
static_assert(sizeof(FusedParams) % 4 == 0 && sizeof(FusedParams) <= 64, "FusedParams staging");

// Work cursor: items (jet, tile, k-chunk) strided over the grid (balanced =
// 0), or the CTA's contiguous, equal share of all tile-planes (jet-major, tile,
// then plane), cut into one column piece per tile it touches (balanced = 1).
// balanced = 2 (lockstep) first runs total_tiles / gridDim.x waves of whole
// columns (tile blockIdx.x + wave * gridDim.x: the CTAs march k together, so
// neighbouring tiles read their shared halo planes within a short window,
// mostly from L2) and shares out the remaining tile-planes the same way.  A
// piece starting mid-column recomputes its first zeta flux, so the result does
// not depend on where the cuts fall.
template <bool ONE> struct Cursor {
    const FusedJet *__restrict__ fj;
    const FusedJet &f1;
    int njets, total_items, total_tiles, balanced;
    int item, w, wend, wave, nwave;

    __device__ __forceinline__ Cursor(const FusedJet *fj_, const FusedJet &f1_, int nj, int items, int tiles, int bal)
        : fj(fj_), f1(f1_), njets(nj), total_items(items), total_tiles(tiles), balanced(bal), item(blockIdx.x), w(0),
          wend(0), wave(0), nwave(bal == 2 ? tiles / (int)gridDim.x : 0)
    {
    }
    // jet of a tile (KEY 0) or of an item (KEY 1); jets without items are passed over
    template <int KEY> __device__ __forceinline__ int jet_of(int t) const
    {
        if constexpr (ONE) return 0;
        int lo = 0, hi = njets;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if ((KEY ? fj[mid].item0 : fj[mid].tile0) <= t) lo = mid; else hi = mid;
        }
        return lo;
    }
    __device__ __forceinline__ bool next_range()
    {
        while (wave <= nwave) {
            if (wave < nwave) {
                const int t = blockIdx.x + wave * gridDim.x;
                const FusedJet &Fw = jet_entry<ONE>(f1, fj, jet_of<0>(t));
                w = Fw.item0 + (t - Fw.tile0) * Fw.nkc;
                wend = w + Fw.nkc;
            } else {
                const int t1 = nwave * gridDim.x;
                int i1 = total_items;
                if (t1 < total_tiles) {
                    const FusedJet &Fw = jet_entry<ONE>(f1, fj, jet_of<0>(t1));
                    i1 = Fw.item0 + (t1 - Fw.tile0) * Fw.nkc;
                }
                const long long rem = total_items - i1;
                w = i1 + (int)((rem * blockIdx.x) / gridDim.x);
                wend = i1 + (int)((rem * (blockIdx.x + 1)) / gridDim.x);
            }
            ++wave;
            if (w < wend) return true;
        }
        return false;
    }
    // the next item's key and jet; false at the end
    __device__ __forceinline__ bool next(int &key, int &jet)
    {
        if (balanced ? !(w < wend || next_range()) : item >= total_items) return false;
        key = balanced ? w : item;
        jet = jet_of<1>(key);
        return true;
    }
    // tile (bx, by) and planes [k0, k1) of the item, of output planes [klo, khi); moves on
    __device__ __forceinline__ void take(int key, const FusedJet &F, int klo, int khi, int &bx, int &by, int &k0, int &k1)
    {
        int r = key - F.item0;
        if (balanced) {
            const int np = khi - klo; // planes per column (F.nkc)
            const int tile = r / np, pl = r - tile * np;
            bx = tile % F.nbx;
            by = tile / F.nbx;
            k0 = klo + pl;
            k1 = klo + min(np, pl + (wend - w));
            w += k1 - k0;
        } else {
            bx = r % F.nbx;
            r /= F.nbx;
            by = r % F.nby;
            const int kc = r / F.nby;
            k0 = klo + kc * F.kc;
            k1 = min(k0 + F.kc, khi);
            item += gridDim.x;
        }
    }
};

} // namespace

} // namespace les
