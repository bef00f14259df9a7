// plane_tail.cu -- the tail D_uz D_uy of a kick (Eq. 4 for i = 2, 3) in one pass over f: for
// velocity cubes too large for one CTA (n_uy = n_uz = 48, FP32 and 16-bit storage, sizes fixed at
// compile time), and on FP32 grids of other sizes, where D_uy or D_uz alone may also run here (the
// second half of this file).
//
// A (cell, j_x) plane of the velocity cube holds n_uy rows (j_y) of n_uz cells (j_z),
// contiguous in f (Listing 1: u_z innermost), and both sweeps stay inside it.  A
// block stages four planes of one spatial cell in shared memory, sweeps them along u_y, then
// along u_z, and writes them back: f is read and written once for the two sweeps.
//
// The pass is bound by the marches, not by DRAM, so a
// thread marches two lines at once, sums and products as f32x2 pairs (vk_common.cuh), through
// a window of a few cells, reading each cell once and writing it back in place: D_uy two
// adjacent columns (one 8-byte access per row), D_uz rows l and l + n_uy / 2 in 16-byte
// chunks.  Rows are padded to n_uz + 4 floats, an odd number of 16-byte units: eight rows
// read at one chunk fall on different banks.  FP32 rows come in by 16-byte asynchronous
// copies (a bulk copy per row costs more instructions: one thread of a warp at a time issues
// it).  Faces in blocks of 8 (D_uy) and 4 (D_uz): blocks of 23 and 20 faces missed in the
// instruction cache (3.6 fetch stalls per issue, 20 % slower).  The arithmetic is march_regs' in
// the same order: FP32 results equal the separate sweeps bit for bit.
// 24^3 x 48^3 cells, per kick tail: FP32 4.84 ms with one line per thread, 3.2 ms here (52
// instructions per face pair, issue 61 % and ALU pipe 56 % busy; DRAM alone 1.8 ms), FP16
// 4.90 -> 3.5 ms.
// 16-bit storage: the planes are decoded into FP32 as they are staged; D_uy's result
// stays FP32 and each row is encoded once, after D_uz, with a refreshed line scale (the
// rounding points of the fused tail of smaller cubes, not of the separate sweeps).
#include "vk_lines.cuh"

namespace vk {

namespace {

constexpr int kPlanesPerBlock = 4;

template <int NU> struct PlaneGeom {
    static constexpr int pitch = NU + 4;     // floats per row
    static constexpr int half = NU / 2;      // line pairs per plane
    static constexpr int threads = kPlanesPerBlock * half;
    static constexpr size_t smem = size_t(kPlanesPerBlock) * NU * pitch * sizeof(float);
    static_assert((pitch / 4) % 2 == 1 && NU % 8 == 0, "an odd number of 16-byte units per row");
};

// 16 bytes from global to shared memory without a register
__device__ __forceinline__ void copy16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}

// D_uy on the adjacent columns at p (row 0): p[r * pitch], p[r * pitch + 1]
template <int NU, bool NEG> __device__ __forceinline__ float2 plane_uy(float *p, const Lim<float2> &lim)
{
    constexpr int ST = NEG ? -PlaneGeom<NU>::pitch : PlaneGeom<NU>::pitch;
    if (NEG) p += (NU - 1) * PlaneGeom<NU>::pitch;
    auto cell = [&](int i) -> float2 & { return *reinterpret_cast<float2 *>(p + i * ST); };
    March<float2> m(lim);
    m.start_zero(cell(0), cell(1));
    constexpr int B = 8, R = (NU - 2) % B;
#pragma unroll 1
    for (int b = 0; b < (NU - 2) / B; ++b, p += B * ST)
#pragma unroll
        for (int q = 0; q < B; ++q) cell(q) = m.face(cell(q + 2));
#pragma unroll
    for (int q = 0; q < R; ++q) cell(q) = m.face(cell(q + 2));
    cell(R) = m.face(make_float2(0.f, 0.f));
    cell(R + 1) = m.last();
    return m.sum;
}

// D_uz on the rows at p and p + NU / 2 rows
template <int NU, bool NEG> __device__ __forceinline__ float2 plane_uz(float *p, const Lim<float2> &lim)
{
    constexpr int OTHER = (NU / 2) * PlaneGeom<NU>::pitch, C = NU / 4, ST = NEG ? -4 : 4;
    if (NEG) p += NU - 4;
    auto at = [&](int row, int j) -> float4 & { return *reinterpret_cast<float4 *>(p + row + j * ST); };
    auto pick = [](const float4 &a, const float4 &b, int i) { // cell i of a chunk in march order
        const int s = NEG ? 3 - i : i;
        return make_float2((&a.x)[s], (&b.x)[s]);
    };
    auto set = [](float4 &a, float4 &b, int i, float2 v) {
        const int s = NEG ? 3 - i : i;
        (&a.x)[s] = v.x;
        (&b.x)[s] = v.y;
    };
    March<float2, true> m(lim);
    float4 a = at(0, 0), b = at(OTHER, 0), oa, ob;
    float4 na = at(0, 1), nb = at(OTHER, 1); // read one chunk ahead of their use
    m.start_zero(pick(a, b, 0), pick(a, b, 1));
    set(oa, ob, 0, m.face(pick(a, b, 2)));
    set(oa, ob, 1, m.face(pick(a, b, 3)));
#pragma unroll 1
    for (int j = 1; j < C; ++j, p += ST) { // chunk j; the outputs of chunk j - 1 are at chunk 0 of p
        a = na;
        b = nb;
        if (j + 1 < C) {
            na = at(0, 2);
            nb = at(OTHER, 2);
        }
        set(oa, ob, 2, m.face(pick(a, b, 0)));
        set(oa, ob, 3, m.face(pick(a, b, 1)));
        at(0, 0) = oa;
        at(OTHER, 0) = ob;
        set(oa, ob, 0, m.face(pick(a, b, 2)));
        set(oa, ob, 1, m.face(pick(a, b, 3)));
    }
    set(oa, ob, 2, m.face(make_float2(0.f, 0.f)));
    set(oa, ob, 3, m.last());
    at(0, 0) = oa;
    at(OTHER, 0) = ob;
    return m.sum;
}

template <int NU, typename T>
__global__ void __launch_bounds__(PlaneGeom<NU>::threads, 5)
    plane_tail_kernel(T *__restrict__ f, const __grid_constant__ PlaneTailArgs a)
{
    using G = PlaneGeom<NU>;
    constexpr bool CODED = sizeof(T) == 2;
    constexpr int P = G::pitch, PER = 16 / int(sizeof(T));
    constexpr int ROWS = kPlanesPerBlock * NU;
    // thread t takes chunk t % CH of rows t / CH, t / CH + RP, ...
    constexpr int CH = NU / PER, RP = G::threads / CH;
    static_assert(NU % PER == 0 && G::threads % CH == 0 && ROWS % RP == 0, "whole passes of whole rows");
    extern __shared__ __align__(16) float plane_s[];
    // the block's planes belong to one spatial cell (the host checks n_ux % 4 == 0)
    const long long p0 = a.plane0 + blockIdx.x * (long long)kPlanesPerBlock;
    const long long cell = a.plane0 / a.nux + (long long)((blockIdx.x * unsigned(kPlanesPerBlock)) / unsigned(a.nux));
    const int row0 = threadIdx.x / CH, col0 = PER * (threadIdx.x - row0 * CH);
    T *g = f + p0 * NU * NU + row0 * NU + col0;
    float *sg = plane_s + row0 * P + col0;
    chain_enter();
#pragma unroll
    for (int k = 0; k < ROWS / RP; ++k) {
        if constexpr (CODED) { // decoded with their row's scale
            float v[PER];
            Chunk<T>::get(reinterpret_cast<const unsigned char *>(g + k * RP * NU), a.scale[p0 * NU + row0 + k * RP], v);
            float4 *s = reinterpret_cast<float4 *>(sg + k * RP * P);
            s[0] = make_float4(v[0], v[1], v[2], v[3]);
            s[1] = make_float4(v[4], v[5], v[6], v[7]);
        } else {
            copy16(sg + k * RP * P, g + k * RP * NU);
        }
    }
    const LineCoefT<float> ky = a.coef_y[cell], kz = a.coef_z[cell];
    if constexpr (!CODED) asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    const int q = threadIdx.x / G::half, l = threadIdx.x - q * G::half;
    float *plane = plane_s + q * NU * P;
    bool bad = false;
    auto check = [&](float2 s) { bad |= !(s.x >= 0.f) || !(s.y >= 0.f) || isinf(s.x) || isinf(s.y); };
    if (ky.nd >= 0) { // one Courant number per cell: block-uniform
        const Lim<float2> lim = to_lim2(ky, ky);
        check((ky.nd & 1) ? plane_uy<NU, true>(plane + 2 * l, lim) : plane_uy<NU, false>(plane + 2 * l, lim));
    }
    __syncthreads();
    if (kz.nd >= 0) {
        const Lim<float2> lim = to_lim2(kz, kz);
        check((kz.nd & 1) ? plane_uz<NU, true>(plane + l * P, lim) : plane_uz<NU, false>(plane + l * P, lim));
    }
    if constexpr (CODED) {
        __syncthreads();
        // a thread encodes whole rows (u_z lines) as the u_z sweep does: the new scale is the
        // row's largest value; stochastic rounding with the stream that sweep draws for the
        // line.  Planes that neither sweep touched keep their codes.
        if (ky.nd >= 0 || kz.nd >= 0) {
#pragma unroll 1
            for (int r = threadIdx.x; r < ROWS; r += G::threads) {
                const long long line = p0 * NU + r;
                const float4 *s = reinterpret_cast<const float4 *>(plane_s + r * P);
                float m = 0.f;
#pragma unroll
                for (int c = 0; c < NU / 4; ++c) m = mx3(mx3(m, s[c].x, s[c].y), s[c].z, s[c].w);
                m = coded_scale<T>(m);
                a.scale[line] = m;
                const float inv = inv_scale(m);
                unsigned rng = sr_bits((unsigned long long)line * NU, a.seed);
                unsigned char *dst = reinterpret_cast<unsigned char *>(f + line * NU);
#pragma unroll
                for (int c = 0; c < NU / PER; ++c) {
                    const float4 x = s[2 * c], y = s[2 * c + 1];
                    const float e[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
                    Chunk<T>::put(dst + 16 * c, inv, e, rng);
                }
            }
        }
    } else {
        __syncthreads();
#pragma unroll
        for (int k = 0; k < ROWS / RP; ++k)
            *reinterpret_cast<float4 *>(g + k * RP * NU) = *reinterpret_cast<const float4 *>(sg + k * RP * P);
    }
    if (bad) atomicOr(a.err, ERR_NAN);
}

// ----------------------------------------------------------------------------
// planes of any size (FP32): D_uy, D_uz or both in one pass, in place or src -> dst
// ----------------------------------------------------------------------------
// The same marches with the sizes at run time, for the velocity grids that the kernels of
// fixed sizes do not take (both sweeps in one pass up to n_uy = 4 n_uz).  A block stages as many whole planes as give its 128 threads a
// pair of lines each (of whatever cells: each pair looks up its own Courant number); the
// rows' pitch is an odd number of 16-byte units.  Bodies of four faces, whose look-ahead
// cells are read before the first of their writes.
// 21 x 26 x 19 x 24 x 20 x 28 cells (1.4e8), per call: D_uy streamed 0.28 ms and D_uz through a
// shared-memory transpose 0.54 ms; 0.250 and 0.270 ms here, both in one pass
// 0.378 ms (24^3 x 24^3: a kick 1.23 -> 0.87 ms; DRAM alone 0.165 ms a pass).
constexpr int kAnyThreads = 128;

__device__ __forceinline__ float2 any_uy(float *p, int st, int n, const Lim<float2> &lim)
{
    auto cell = [&](int i) -> float2 & { return *reinterpret_cast<float2 *>(p + i * st); };
    March<float2> m(lim);
    m.start_zero(cell(0), cell(1));
#pragma unroll 1
    for (int left = n - 4; left > 0; left -= 4, p += 4 * st) { // n is a multiple of 4
        float2 c[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) c[q] = cell(q + 2);
#pragma unroll
        for (int q = 0; q < 4; ++q) cell(q) = m.face(c[q]);
    }
    const float2 a = cell(2), b = cell(3);
    cell(0) = m.face(a);
    cell(1) = m.face(b);
    cell(2) = m.face(make_float2(0.f, 0.f));
    cell(3) = m.last();
    return m.sum;
}

// rows at p and p + other floats, C chunks of four cells
template <bool NEG> __device__ __forceinline__ float2 any_uz(float *p, int other, int C, const Lim<float2> &lim)
{
    constexpr int ST = NEG ? -4 : 4;
    if (NEG) p += 4 * (C - 1);
    auto at = [&](int row, int j) -> float4 & { return *reinterpret_cast<float4 *>(p + row + j * ST); };
    auto pick = [](const float4 &a, const float4 &b, int i) {
        const int s = NEG ? 3 - i : i;
        return make_float2((&a.x)[s], (&b.x)[s]);
    };
    auto set = [](float4 &a, float4 &b, int i, float2 v) {
        const int s = NEG ? 3 - i : i;
        (&a.x)[s] = v.x;
        (&b.x)[s] = v.y;
    };
    March<float2, true> m(lim);
    float4 a = at(0, 0), b = at(other, 0), oa, ob, na = a, nb = b;
    if (C > 1) {
        na = at(0, 1);
        nb = at(other, 1);
    }
    m.start_zero(pick(a, b, 0), pick(a, b, 1));
    set(oa, ob, 0, m.face(pick(a, b, 2)));
    set(oa, ob, 1, m.face(pick(a, b, 3)));
#pragma unroll 1
    for (int j = 1; j < C; ++j, p += ST) { // chunk j enters; the outputs of chunk j - 1 go to chunk 0 of p
        a = na;
        b = nb;
        if (j + 1 < C) {
            na = at(0, 2);
            nb = at(other, 2);
        }
        set(oa, ob, 2, m.face(pick(a, b, 0)));
        set(oa, ob, 3, m.face(pick(a, b, 1)));
        at(0, 0) = oa;
        at(other, 0) = ob;
        set(oa, ob, 0, m.face(pick(a, b, 2)));
        set(oa, ob, 1, m.face(pick(a, b, 3)));
    }
    set(oa, ob, 2, m.face(make_float2(0.f, 0.f)));
    set(oa, ob, 3, m.last());
    at(0, 0) = oa;
    at(other, 0) = ob;
    return m.sum;
}

__global__ void __launch_bounds__(kAnyThreads, 5)
    plane_any_kernel(const float *src, float *dst, const __grid_constant__ PlaneAnyArgs a)
{
    extern __shared__ __align__(16) float any_s[];
    const int ny = a.nuy, nz = a.nuz, pitch = a.pitch, u = nz / 4; // u: 16-byte chunks of a row
    const long long p0 = a.plane0 + (long long)blockIdx.x * a.per_block, pend = a.plane0 + a.nplanes;
    const int planes = pend - p0 < a.per_block ? int(pend - p0) : a.per_block;
    const long long e0 = p0 * ny * nz;
    const int chunks = planes * ny * u;
    chain_enter();
    for (int k = threadIdx.x; k < chunks; k += kAnyThreads) {
        const int row = int(fdiv(unsigned(k), a.div_u)), col = k - row * u;
        copy16(any_s + row * pitch + 4 * col, src + e0 + 4ll * k);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    bool bad = false;
    auto check = [&](float2 s) { bad |= !(s.x >= 0.f) || !(s.y >= 0.f) || isinf(s.x) || isinf(s.y); };
    if (a.coef_y) {
        const int half = nz / 2; // column pairs of a plane
        for (int k = threadIdx.x; k < planes * half; k += kAnyThreads) {
            const int q = int(fdiv(unsigned(k), a.div_hz)), c = k - q * half;
            const LineCoefT<float> ky = a.coef_y[fdiv(unsigned(p0 + q), a.div_nux)];
            if (ky.nd < 0) continue;
            const bool neg = ky.nd & 1;
            const Lim<float2> lim = to_lim2(ky, ky);
            check(any_uy(any_s + (q * ny + (neg ? ny - 1 : 0)) * pitch + 2 * c, neg ? -pitch : pitch, ny, lim));
        }
        __syncthreads();
    }
    if (a.coef_z) {
        const int half = ny / 2; // row pairs of a plane: l, l + half
        for (int k = threadIdx.x; k < planes * half; k += kAnyThreads) {
            const int q = int(fdiv(unsigned(k), a.div_hy)), l = k - q * half;
            const LineCoefT<float> kz = a.coef_z[fdiv(unsigned(p0 + q), a.div_nux)];
            if (kz.nd < 0) continue;
            const Lim<float2> lim = to_lim2(kz, kz);
            float *row = any_s + (q * ny + l) * pitch;
            check((kz.nd & 1) ? any_uz<true>(row, half * pitch, u, lim) : any_uz<false>(row, half * pitch, u, lim));
        }
        __syncthreads();
    }
    for (int k = threadIdx.x; k < chunks; k += kAnyThreads) {
        const int row = int(fdiv(unsigned(k), a.div_u)), col = k - row * u;
        *reinterpret_cast<float4 *>(dst + e0 + 4ll * k) = *reinterpret_cast<const float4 *>(any_s + row * pitch + 4 * col);
    }
    if (bad) atomicOr(a.err, ERR_NAN);
}

} // namespace

bool plane_tail_supported(int nuy, int nuz, int nux, int dtype)
{
    return dtype >= 1 && dtype <= 3 && nuy == nuz && nuz == 48 && nux % kPlanesPerBlock == 0;
}

template <typename T> static cudaError_t launch_plane_tail_t(T *f, const PlaneTailArgs &a, long long blocks, cudaStream_t st)
{
    const cudaError_t e = allow_smem((const void *)plane_tail_kernel<48, T>, PlaneGeom<48>::smem);
    if (e != cudaSuccess) return e;
    return launch_chained_t(a.nplanes * 48 * 48, plane_tail_kernel<48, T>, dim3(unsigned(blocks)), dim3(PlaneGeom<48>::threads), PlaneGeom<48>::smem,
                            st, f, a);
}

cudaError_t launch_plane_tail(void *f, const PlaneTailArgs &a, int nu, int dtype, cudaStream_t st)
{
    if (a.nplanes <= 0) return cudaSuccess;
    if (nu != 48 || a.plane0 % kPlanesPerBlock || a.nplanes % kPlanesPerBlock) return cudaErrorInvalidValue;
    if (dtype != 1 && !a.scale) return cudaErrorInvalidValue;
    const long long blocks = a.nplanes / kPlanesPerBlock;
    if (blocks > 0x7fffffffll) return cudaErrorInvalidValue;
    switch (dtype) {
    case 1: return launch_plane_tail_t(static_cast<float *>(f), a, blocks, st);
    case 2: return launch_plane_tail_t(static_cast<__nv_bfloat16 *>(f), a, blocks, st);
    case 3: return launch_plane_tail_t(static_cast<__half *>(f), a, blocks, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_plane_any(const float *src, float *dst, const PlaneAnyArgs &args, cudaStream_t st)
{
    if (args.nplanes <= 0) return cudaSuccess;
    // plane indices stay below 2^31 (u_z lines do, checked at init)
    if (args.nux < 1 || args.nuy < 4 || args.nuy % 4 || args.nuz < 4 || args.nuz % 4 || args.plane0 + args.nplanes > 0x7fffffffll)
        return cudaErrorInvalidValue;
    PlaneAnyArgs a = args;
    a.pitch = 4 * ((a.nuz / 4) | 1);
    const size_t plane = size_t(a.nuy) * a.pitch * sizeof(float);
    // a pair of lines per thread, within 48 KB where that holds at least a warp's pairs
    const int most = a.nuy > a.nuz ? a.nuy : a.nuz;
    a.per_block = 2 * kAnyThreads / most > 1 ? 2 * kAnyThreads / most : 1;
    while (a.per_block > 1 && a.per_block * plane > 48 * 1024 && (a.per_block - 1) * most >= 64) --a.per_block;
    if (a.nplanes < a.per_block) a.per_block = int(a.nplanes);
    a.div_u = make_fastdiv(unsigned(a.nuz / 4));
    a.div_hz = make_fastdiv(unsigned(a.nuz / 2));
    a.div_hy = make_fastdiv(unsigned(a.nuy / 2));
    a.div_nux = make_fastdiv(unsigned(a.nux));
    const size_t smem = a.per_block * plane;
    const cudaError_t e = allow_smem((const void *)plane_any_kernel, smem);
    if (e != cudaSuccess) return e;
    const long long blocks = (a.nplanes + a.per_block - 1) / a.per_block;
    return launch_chained_t(a.nplanes * a.nuy * a.nuz, plane_any_kernel, dim3(unsigned(blocks)), dim3(kAnyThreads), smem, st, src, dst, a);
}

} // namespace vk
