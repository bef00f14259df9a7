// vk_common.cuh -- device building blocks of libvlasov (sm_103a).
//
//  * PTX wrappers: mbarrier, TMA tensor copies (cp.async.bulk.tensor), bulk
//    async groups, proxy fences, the global timer used by bounded waits.
//  * SL-MPP5 (Sec. 4.2 of Yoshikawa, Tanaka & Yoshida, SC'21): the
//    conservative semi-Lagrangian fractional flux, the Suresh-Huynh
//    monotonicity-preserving constraint and the positivity clamp, and the
//    march of one line in shared memory.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "vk_kernels.h"

namespace vk {

// A bounded wait gives up after this much wall time or this many polls.
constexpr uint64_t kWaitLimitNs = 2000000000ull;
constexpr unsigned kWaitLimitPolls = 1u << 26;
// How long one poll may keep the warp asleep (it wakes when the phase completes): warps that
// wait poll seldom and leave the issue slots to those that work.
constexpr unsigned kPollNs = 20000;

// ----------------------------------------------------------------------------
// PTX wrappers
// ----------------------------------------------------------------------------

__device__ __forceinline__ unsigned smem_u32(const void *p)
{
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t globaltimer()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}

__device__ __forceinline__ void fence_barrier_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(kPollNs)
        : "memory");
    return ok != 0;
}

// Non-blocking probe: has the phase with this parity completed?
__device__ __forceinline__ bool mbar_test_wait(uint64_t *bar, unsigned parity)
{
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for the phase of `bar` with the given parity; false if the wait ran out.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, unsigned parity)
{
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer();
    for (unsigned it = 1; it < kWaitLimitPolls; ++it) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 63u) == 0 && globaltimer() - t0 > kWaitLimitNs) return false;
    }
    return false;
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0,
                                            int c1)
{
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tma_load_3d(void *dst, const CUtensorMap *map, uint64_t *bar, int c0,
                                            int c1, int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, const void *src, int c0, int c1)
{
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(smem_u32(src)), "r"(c0), "r"(c1)
                 : "memory");
}

__device__ __forceinline__ void tma_store_3d(const CUtensorMap *map, const void *src, int c0, int c1,
                                             int c2)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(
            reinterpret_cast<uint64_t>(map)),
        "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }

__device__ __forceinline__ void bulk_wait_read_all()
{
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

// wait until at most n (0..7) of the most recent bulk groups are still reading shared memory
__device__ __forceinline__ void bulk_wait_read_at_most(unsigned n)
{
    switch (n) {
    case 0: asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); break;
    case 1: asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); break;
    case 2: asm volatile("cp.async.bulk.wait_group.read 2;" ::: "memory"); break;
    case 3: asm volatile("cp.async.bulk.wait_group.read 3;" ::: "memory"); break;
    case 4: asm volatile("cp.async.bulk.wait_group.read 4;" ::: "memory"); break;
    case 5: asm volatile("cp.async.bulk.wait_group.read 5;" ::: "memory"); break;
    case 6: asm volatile("cp.async.bulk.wait_group.read 6;" ::: "memory"); break;
    default: asm volatile("cp.async.bulk.wait_group.read 7;" ::: "memory"); break;
    }
}

// barrier among the consumer warps only (named barrier 1)
__device__ __forceinline__ void consumer_sync(int nthreads)
{
    asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
}

// ----------------------------------------------------------------------------
// chained launches
// ----------------------------------------------------------------------------
// A step is a chain of 10 to 15 kernels, each of which reads what the one before wrote; on a
// small grid the gaps between them are a third of it (8^3 x 16^3 cells: a step of 113 us, 80 with
// launches chained).  A kernel launched chained may start while the kernel before it on the
// stream still runs: it calls chain_enter() before its first access to global memory, which
// lets the next kernel start in turn and waits until the one before has ended and its writes
// are visible.  So the launch, the blocks' start-up and the set-up of barriers and tables are
// hidden, and nothing else changes: every kernel of a chain waits, so a kernel two behind has
// ended too.  Only kernels over at most kChainCells cells are launched so: on long ones the
// waiting blocks cost more than the gap they hide (steps of 16^3 x 16^3 cells 271 -> 265 us, of
// 20^3 x 16^3 481 -> 543, of 24^3 x 16^3 725 -> 805).
constexpr long long kChainCells = 1ll << 24;
__device__ __forceinline__ void chain_enter()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

struct ChainedLaunch {
    cudaLaunchAttribute attr;
    cudaLaunchConfig_t cfg;
    ChainedLaunch(long long cells, dim3 grid, dim3 block, size_t smem, cudaStream_t st) : attr{}, cfg{}
    {
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = cells <= kChainCells;
        cfg.gridDim = grid;
        cfg.blockDim = block;
        cfg.dynamicSmemBytes = smem;
        cfg.stream = st;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
    }
};
// cells: how many the kernel goes over (FP64: times 16, the ratio of their times)
inline cudaError_t launch_chained(long long cells, const void *k, dim3 grid, dim3 block, size_t smem, cudaStream_t st, void **params)
{
    ChainedLaunch l(cells, grid, block, smem, st);
    return cudaLaunchKernelExC(&l.cfg, k, params);
}
template <typename... P, typename... A>
cudaError_t launch_chained_t(long long cells, void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A &&...args)
{
    ChainedLaunch l(cells, grid, block, smem, st);
    return cudaLaunchKernelEx(&l.cfg, k, static_cast<P>(args)...);
}

// ----------------------------------------------------------------------------
// storage <-> compute conversions
// ----------------------------------------------------------------------------

template <typename T> struct Compute { using type = float; };
template <> struct Compute<double> { using type = double; };

__device__ __forceinline__ float to_c(float v) { return v; }
__device__ __forceinline__ double to_c(double v) { return v; }
__device__ __forceinline__ float to_c(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float to_c(__half v) { return __half2float(v); }

template <typename T> __device__ __forceinline__ T from_c(typename Compute<T>::type v);
template <> __device__ __forceinline__ float from_c<float>(float v) { return v; }
template <> __device__ __forceinline__ double from_c<double>(double v) { return v; }
template <> __device__ __forceinline__ __nv_bfloat16 from_c<__nv_bfloat16>(float v)
{
    return __float2bfloat16_rn(v);
}
template <> __device__ __forceinline__ __half from_c<__half>(float v) { return __float2half_rn(v); }

// ----------------------------------------------------------------------------
// min / max with three inputs (one instruction for f32 on sm_100+)
// ----------------------------------------------------------------------------

__device__ __forceinline__ float mn3(float a, float b, float c)
{
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ float mx3(float a, float b, float c)
{
    float d;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}
__device__ __forceinline__ double mn3(double a, double b, double c) { return fmin(a, fmin(b, c)); }
__device__ __forceinline__ double mx3(double a, double b, double c) { return fmax(a, fmax(b, c)); }
__device__ __forceinline__ float mn2(float a, float b) { return fminf(a, b); }
__device__ __forceinline__ float mx2(float a, float b) { return fmaxf(a, b); }
__device__ __forceinline__ double mn2(double a, double b) { return fmin(a, b); }
__device__ __forceinline__ double mx2(double a, double b) { return fmax(a, b); }

// ----------------------------------------------------------------------------
// 16-bit storage codec: stochastic rounding to BF16 / FP16
// ----------------------------------------------------------------------------
// Re-encoding f after every sweep with round-to-nearest drops or biases the
// small per-sweep updates; stochastic rounding keeps each encode unbiased in
// expectation.  Random bits: the 32-bit finalizer of MurmurHash3 (Appleby)
// seeds one stream per line of the march from the element index and a
// per-sweep seed; the stream then advances with the 32-bit linear congruential
// generator of Numerical Recipes (a = 1664525, c = 1013904223), whose upper 16
// bits feed one value each.  A run is reproducible.

__device__ __forceinline__ unsigned fmix32(unsigned h)
{
    h ^= h >> 16;
    h *= 0x85ebca6bu;
    h ^= h >> 13;
    h *= 0xc2b2ae35u;
    h ^= h >> 16;
    return h;
}

__device__ __forceinline__ unsigned sr_bits(unsigned long long elem, unsigned seed)
{
    return fmix32(unsigned(elem) ^ unsigned(elem >> 32) * 0x9e3779b9u ^ seed * 0x85ebca6bu);
}

__device__ __forceinline__ unsigned lcg_next(unsigned &x)
{
    constexpr Lcg step = kLcg;
    x = step(x);
    return x;
}

// Two non-negative FP32 values -> packed bf16x2 with stochastic rounding: 16 random bits (of
// two LCG steps) are added below the BF16 mantissa of x and of y, and one byte permute packs
// the two upper halves.
__device__ __forceinline__ unsigned sr_pack_bf16x2(float x, float y, unsigned r1, unsigned r2)
{
    return __byte_perm(__float_as_uint(x) + r1, __float_as_uint(y) + r2, 0x7632);
}
__device__ __forceinline__ unsigned sr_pack_bf16x2(float x, float y, unsigned &rng)
{
    const unsigned r1 = lcg_next(rng) >> 16, r2 = lcg_next(rng) >> 16;
    return sr_pack_bf16x2(x, y, r1, r2);
}

// Line scales of the 16-bit codec.  coded_scale: the scale a refresh stores for a line
// whose largest value is m; BF16 keeps at least 2^-64, so that a line left empty can
// still take in mass from the sweeps that keep the scale (BF16 carries 8 significant
// bits at any exponent: codes up to 2^64 x its largest value stay finite, and values
// down to 2^-190 stay representable); FP16 has 5 exponent bits and keeps m itself.
// inv_scale: 1 / s for encoding, 0 for s = 0 and for a subnormal s, whose reciprocal
// would overflow (such a line holds nothing above 2^-126; its values encode as 0).
template <typename T> __device__ __forceinline__ float coded_scale(float m) { return m; }
template <> __device__ __forceinline__ float coded_scale<__nv_bfloat16>(float m) { return fmaxf(m, 0x1p-64f); }
__device__ __forceinline__ float inv_scale(float s) { return s >= 0x1p-126f ? __fdividef(1.f, s) : 0.f; }

// Two non-negative FP32 values -> packed f16x2 with stochastic rounding: 13 of the upper
// 16 bits of two LCG steps are added below the FP16 mantissa (13 bits below FP32's), and
// one round-toward-zero conversion packs both (x in the lower half).
__device__ __forceinline__ unsigned sr_pack_f16x2(float x, float y, unsigned r1, unsigned r2)
{
    const float xr = __uint_as_float(__float_as_uint(x) + (r1 & 0x1fffu)), yr = __uint_as_float(__float_as_uint(y) + (r2 & 0x1fffu));
    unsigned out;
    asm("cvt.rz.f16x2.f32 %0, %1, %2;" : "=r"(out) : "f"(yr), "f"(xr));
    return out;
}
__device__ __forceinline__ unsigned sr_pack_f16x2(float x, float y, unsigned &rng)
{
    const unsigned r1 = lcg_next(rng) >> 16, r2 = lcg_next(rng) >> 16;
    return sr_pack_f16x2(x, y, r1, r2);
}

// ----------------------------------------------------------------------------
// arithmetic on float, double and float2 (two independent lines in packed FP32:
// add / sub / mul / fma use the f32x2 instructions of sm_100+, min / max / select
// act per component)
// ----------------------------------------------------------------------------

#define VK_F2_BINOP(name, op)                                                                        \
    __device__ __forceinline__ float2 name(float2 a, float2 b)                                        \
    {                                                                                                 \
        float2 d;                                                                                     \
        asm("{.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t" op     \
            " rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;}"                                                    \
            : "=f"(d.x), "=f"(d.y)                                                                    \
            : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));                                                \
        return d;                                                                                     \
    }
VK_F2_BINOP(vadd, "add.rn.f32x2")
VK_F2_BINOP(vsub, "sub.rn.f32x2")
VK_F2_BINOP(vmul, "mul.rn.f32x2")
#undef VK_F2_BINOP

// a * b + c
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("{.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
        "mov.b64 rc, {%6, %7};\n\tfma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;}"
        : "=f"(d.x), "=f"(d.y)
        : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
    return d;
}
__device__ __forceinline__ float vadd(float a, float b) { return a + b; }
__device__ __forceinline__ float vsub(float a, float b) { return a - b; }
__device__ __forceinline__ float vmul(float a, float b) { return a * b; }
__device__ __forceinline__ float vfma(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double vadd(double a, double b) { return a + b; }
__device__ __forceinline__ double vsub(double a, double b) { return a - b; }
__device__ __forceinline__ double vmul(double a, double b) { return a * b; }
__device__ __forceinline__ double vfma(double a, double b, double c) { return fma(a, b, c); }

__device__ __forceinline__ float2 mn2(float2 a, float2 b) { return make_float2(fminf(a.x, b.x), fminf(a.y, b.y)); }
__device__ __forceinline__ float2 mx2(float2 a, float2 b) { return make_float2(fmaxf(a.x, b.x), fmaxf(a.y, b.y)); }
__device__ __forceinline__ float2 mn3(float2 a, float2 b, float2 c)
{
    return make_float2(mn3(a.x, b.x, c.x), mn3(a.y, b.y, c.y));
}
__device__ __forceinline__ float2 mx3(float2 a, float2 b, float2 c)
{
    return make_float2(mx3(a.x, b.x, c.x), mx3(a.y, b.y, c.y));
}

template <typename X> __device__ __forceinline__ X splat(double v);
template <> __device__ __forceinline__ float splat<float>(double v) { return float(v); }
template <> __device__ __forceinline__ double splat<double>(double v) { return v; }
template <> __device__ __forceinline__ float2 splat<float2>(double v) { return make_float2(float(v), float(v)); }

// ----------------------------------------------------------------------------
// SL-MPP5 line coefficients
// ----------------------------------------------------------------------------

// v[0..3]: weights of fbar - c_0 on the four differences delta_{-2} .. delta_{1} of the
// stencil (the five weights of fbar sum to 1)
template <typename X> struct Lim {
    X v0, v1, v2, v3, s, alpha;
};

template <typename C> __device__ __forceinline__ Lim<C> to_lim(const LineCoefT<C> &k)
{
    return Lim<C>{-k.w[0], -(k.w[0] + k.w[1]), k.w[3] + k.w[4], k.w[4], k.s, k.alpha};
}

// two lines in one packed pair
__device__ __forceinline__ Lim<float2> to_lim2(const Lim<float> &a, const Lim<float> &b)
{
    return Lim<float2>{make_float2(a.v0, b.v0), make_float2(a.v1, b.v1), make_float2(a.v2, b.v2),
                       make_float2(a.v3, b.v3), make_float2(a.s, b.s), make_float2(a.alpha, b.alpha)};
}
__device__ __forceinline__ Lim<float2> to_lim2(const LineCoefT<float> &a, const LineCoefT<float> &b)
{
    return to_lim2(to_lim(a), to_lim(b));
}

// ----------------------------------------------------------------------------
// the flux of one face, in differences of neighbouring cells
// ----------------------------------------------------------------------------
// Everything the limiter compares is written relative to the donor c_0, as combinations of
// the differences delta_k = c_{k+1} - c_k, of which each face forms one and takes the rest
// from the faces before it:
//   fbar - c_0  = v0 delta_{-2} + v1 delta_{-1} + v2 delta_0 + v3 delta_1
//   f_MD - c_0  = delta_0 / 2 - dm4_{+1/2} / 2        f_UL - c_0 = alpha delta_{-1}
//   f_LC - c_0  = delta_{-1} / 2 + 4/3 dm4_{-1/2}     curvature d_k = delta_k - delta_{k-1}
// What bounds a march: on this part a min or max (two or three inputs) occupies the ALU
// pipe for two cycles per warp, an FP32 add / multiply / fma the FMA pipe for one, and a
// packed pair of them (f32x2) one issue slot.  Per face 20 FMA-pipe operations and 11 ALU
// operations (22 cycles), against 20 and 14 (28 cycles) when the same limiter is written
// in the cells themselves (34 instructions); FP64 arithmetic runs at 2 lanes per SM and
// cycle, so the FP64 form keeps to 17 FP64 operations and compares as integers.

// Limited curvature at the face between two cells of curvatures d0, d1: FP32 returns
// 2 dm4, dm4 = minmod(4 d0 - d1, 4 d1 - d0, d0, d1).  With S = d0 + d1, t = d0 - d1,
// e = |S| - |t| (twice the smaller magnitude when the signs agree, else <= 0) the four
// arguments' least magnitude is e / 2 or, once the larger exceeds 3 times the smaller,
// (3 e - 2 |t|) / 2; below 0 the minmod is 0; its sign is S's.  Three ALU operations
// instead of six.  FP64 returns dm4 itself.
__device__ __forceinline__ float limited_curv(float d0, float d1)
{
    const float S = d0 + d1, t = fabsf(d0 - d1);
    const float e = fabsf(S) - t;
    const float w = fmaf(2.f, e - t, e);
    return copysignf(fmaxf(fminf(e, w), 0.f), S);
}
__device__ __forceinline__ float2 limited_curv(float2 d0, float2 d1)
{
    const float2 S = vadd(d0, d1), t = vsub(d0, d1);
    const float2 e = make_float2(fabsf(S.x) - fabsf(t.x), fabsf(S.y) - fabsf(t.y));
    const float2 u = make_float2(e.x - fabsf(t.x), e.y - fabsf(t.y));
    const float2 w = vfma(make_float2(2.f, 2.f), u, e);
    return make_float2(copysignf(fmaxf(fminf(e.x, w.x), 0.f), S.x), copysignf(fmaxf(fminf(e.y, w.y), 0.f), S.y));
}

// FP64 values as integers in the same order (negative ones with their lower 63 bits
// flipped): min and max run on the integer pipe, 8 times the rate of FP64 comparisons
__device__ __forceinline__ long long order_key(double x)
{
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}
__device__ __forceinline__ double order_value(long long k)
{
    return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffll));
}
__device__ __forceinline__ long long kmin(long long a, long long b) { return a < b ? a : b; }
__device__ __forceinline__ long long kmax(long long a, long long b) { return a > b ? a : b; }

__device__ __forceinline__ double limited_curv(double d0, double d1)
{
    const long long a = order_key(fma(4.0, d0, -d1)), b = order_key(fma(4.0, d1, -d0)), p = order_key(d0),
                    q = order_key(d1);
    // minmod = median(lo, 0, hi) with lo / hi the smallest / largest argument
    return order_value(kmin(kmax(kmin(kmin(a, b), kmin(p, q)), 0ll), kmax(kmax(a, b), kmax(p, q))));
}
// what multiplies limited_curv's result in f_MD and f_LC
template <typename X> struct CurvScale {
    static constexpr double md = -0.25, lc = 2.0 / 3.0;
};
template <> struct CurvScale<double> {
    static constexpr double md = -0.5, lc = 4.0 / 3.0;
};

// clamp(phi, fmin, fmax) relative to the donor, fmin = max(A, B), fmax = min(C, D),
// A / C = min / max(0, dp, md), B / D = min / max(0, ul, lc): by associativity of max and
// min, min(max(phi, A, B), C, D).
//
// Suresh & Huynh keep fbar when it lies between c0 and the MP bound
// f_MP = c0 + minmod(cp1 - c0, alpha (c0 - cm1)) and otherwise take
// median(fbar, fmin, fmax).  f_MP is the median of (c0, cp1, f_UL), and every
// one of the sets bounding fmin and fmax contains c0 together with cp1 or f_UL,
// so [c0, f_MP] lies inside [fmin, fmax] (both are pure selections, exactly so
// in floating point): the constraint is the clamp of fbar to [fmin, fmax].
__device__ __forceinline__ float mp_clamp(float phi, float dp, float md, float ul, float lc)
{
    return mn3(mx3(phi, mn3(0.f, dp, md), mn3(0.f, ul, lc)), mx3(0.f, dp, md), mx3(0.f, ul, lc));
}
__device__ __forceinline__ float2 mp_clamp(float2 phi, float2 dp, float2 md, float2 ul, float2 lc)
{
    return make_float2(mp_clamp(phi.x, dp.x, md.x, ul.x, lc.x), mp_clamp(phi.y, dp.y, md.y, ul.y, lc.y));
}
__device__ __forceinline__ double mp_clamp(double phi, double dp, double md, double ul, double lc)
{
    const long long p = order_key(dp), m = order_key(md), u = order_key(ul), l = order_key(lc);
    const long long A = kmin(0ll, kmin(p, m)), C = kmax(0ll, kmax(p, m));
    const long long B = kmin(0ll, kmin(u, l)), D = kmax(0ll, kmax(u, l));
    return order_value(kmin(kmin(kmax(kmax(order_key(phi), A), B), C), D));
}
// positivity: F clamped to [0, donor]
template <typename X> __device__ __forceinline__ X flux_clamp(X F, X c0) { return mn2(mx2(F, splat<X>(0.0)), c0); }
__device__ __forceinline__ double flux_clamp(double F, double c0)
{
    return order_value(kmin(kmax(order_key(F), 0ll), order_key(c0)));
}

// Fractional flux through the downwind face of the donor c0 (local frame, flow toward
// +index): dmm, dm, dp, dpp = delta_{-2} .. delta_1 around it, hm, hp = dm / 2, dp / 2, qm /
// qp the limited curvatures (limited_curv) at its upwind / downwind faces.
// SPLIT (packed pairs): operations on the cells themselves act on the two lines one by one,
// for cells that do not sit in aligned register pairs.
__device__ __forceinline__ float2 two(float a, float b) { return make_float2(a, b); }
template <bool SPLIT, typename X> __device__ __forceinline__ X cell_sub(X a, X b)
{
    if constexpr (SPLIT) return two(a.x - b.x, a.y - b.y);
    else return vsub(a, b);
}
template <bool SPLIT, typename X> __device__ __forceinline__ X cell_add(X a, X b)
{
    if constexpr (SPLIT) return two(a.x + b.x, a.y + b.y);
    else return vadd(a, b);
}
template <bool SPLIT, typename X> __device__ __forceinline__ X cell_mul(X a, X b)
{
    if constexpr (SPLIT) return two(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y));
    else return vmul(a, b);
}

template <bool SPLIT = false, typename X>
__device__ __forceinline__ X sl_mpp5_flux(const Lim<X> &k, X c0, X dmm, X dm, X dp, X dpp, X hm, X hp, X qm, X qp)
{
    const X phi = vfma(k.v3, dpp, vfma(k.v2, dp, vfma(k.v1, dm, vmul(k.v0, dmm))));
    const X md = vfma(splat<X>(CurvScale<X>::md), qp, hp);
    const X lc = vfma(splat<X>(CurvScale<X>::lc), qm, hm);
    const X v = mp_clamp(phi, dp, md, vmul(k.alpha, dm), lc);
    return flux_clamp(vfma(k.s, v, cell_mul<SPLIT>(k.s, c0)), c0);
}

// ----------------------------------------------------------------------------
// the march of one line (local frame: flow toward +index), cell after cell:
// c_i <- c_i - (F_{i+1/2} - F_{i-1/2})
// ----------------------------------------------------------------------------
// The window around the next cell i: start_periodic / start_zero set it up from the first
// cells, face(cp2) takes cell i + 2, returns the new value of cell i and moves on; last()
// is the last cell of a zero-flux line (nothing crosses its outer face).  sum: of the new
// values (for the NaN / sign check).
template <typename X, bool SPLIT = false> struct March {
    const Lim<X> &k;
    X c0, cp1, dmm, dm, dp, hm, hp, d0, qm, Fm, sum;

    __device__ __forceinline__ explicit March(const Lim<X> &k_) : k(k_) {}

    // cells -3 .. 1 (the last three of the line, then the first two)
    __device__ __forceinline__ void start_periodic(X m3, X m2, X m1, X s0, X s1)
    {
        const X half = splat<X>(0.5);
        const X e3 = vsub(m2, m3), e2 = vsub(m1, m2), e1 = vsub(s0, m1), e0 = vsub(s1, s0);
        const X dmm_ = vsub(e2, e3), dm_ = vsub(e1, e2);
        d0 = vsub(e0, e1);
        qm = limited_curv(dm_, d0);
        hm = vmul(half, e1);
        hp = vmul(half, e0);
        Fm = sl_mpp5_flux(k, m1, e3, e2, e1, e0, vmul(half, e2), hm, limited_curv(dmm_, dm_), qm); // face -1/2
        begin(s0, s1, e2, e1, e0);
    }
    // ghost cells hold 0 and nothing crosses face -1/2
    __device__ __forceinline__ void start_zero(X s0, X s1)
    {
        const X half = splat<X>(0.5);
        const X e0 = vsub(s1, s0); // delta_{-1} = s0 - 0, curvature of the ghost cell -1: s0
        d0 = vsub(e0, s0);
        qm = limited_curv(s0, d0);
        hm = vmul(half, s0);
        hp = vmul(half, e0);
        Fm = splat<X>(0.0);
        begin(s0, s1, splat<X>(0.0), s0, e0);
    }
    __device__ __forceinline__ X face(X cp2)
    {
        const X dpp = cell_sub<SPLIT>(cp2, cp1);
        const X dn = vsub(dpp, dp); // curvature of cell i + 1
        const X qp = limited_curv(d0, dn);
        const X F = sl_mpp5_flux<SPLIT>(k, c0, dmm, dm, dp, dpp, hm, hp, qm, qp);
        const X out = cell_add<SPLIT>(c0, vsub(Fm, F));
        sum = cell_add<SPLIT>(sum, out);
        c0 = cp1;
        cp1 = cp2;
        dmm = dm;
        dm = dp;
        dp = dpp;
        hm = hp;
        hp = vmul(splat<X>(0.5), dpp);
        d0 = dn;
        qm = qp;
        Fm = F;
        return out;
    }
    __device__ __forceinline__ X last()
    {
        const X out = vadd(c0, Fm);
        sum = vadd(sum, out);
        return out;
    }

  private:
    __device__ __forceinline__ void begin(X s0, X s1, X a, X b, X c)
    {
        c0 = s0;
        cp1 = s1;
        dmm = a;
        dm = b;
        dp = c;
        sum = splat<X>(0.0);
    }
};

// ----------------------------------------------------------------------------
// one line in shared memory
// ----------------------------------------------------------------------------

// Advance the line p[0], p[step], ..., p[(L-1) step] (local frame: flow toward
// +index) by the fractional part of the Courant number, in place.  PERIODIC selects the
// position-space seam; otherwise ghost cells are 0 and both outer faces carry no flux.
// Returns the sum of the new values (used for the NaN / sign check).
// Requires L >= 4.
template <typename T, bool PERIODIC, typename C>
__device__ __forceinline__ C march_line(T *p, long step, int L, const Lim<C> &k)
{
    const C s0 = to_c(p[0]);
    const C s1 = to_c(p[step]);
    March<C> m(k);
    if (PERIODIC)
        m.start_periodic(to_c(p[(long)(L - 3) * step]), to_c(p[(long)(L - 2) * step]), to_c(p[(long)(L - 1) * step]),
                         s0, s1);
    else m.start_zero(s0, s1);
#pragma unroll 4
    for (int i = 0; i < L - 2; ++i) {
        const C out = m.face(to_c(p[(long)(i + 2) * step]));
        p[(long)i * step] = from_c<T>(out);
    }
    p[(long)(L - 2) * step] = from_c<T>(m.face(PERIODIC ? s0 : C(0)));
    p[(long)(L - 1) * step] = from_c<T>(PERIODIC ? m.face(s1) : m.last());
    return m.sum;
}

// rotate the line right by r positions (0 <= r < L): q[i] <- q[i - r]
template <typename T> __device__ __forceinline__ void rotate_line(T *p, long step, int L, int r)
{
    auto rev = [&](int a, int b) { // reverse [a, b)
        for (int i = a, j = b - 1; i < j; ++i, --j) {
            const T t = p[(long)i * step];
            p[(long)i * step] = p[(long)j * step];
            p[(long)j * step] = t;
        }
    };
    if (r == 0) return;
    rev(0, L - r);
    rev(L - r, L);
    rev(0, L);
}

} // namespace vk
