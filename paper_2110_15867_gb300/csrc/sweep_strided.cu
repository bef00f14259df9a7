// sweep_strided.cu -- SL-MPP5 sweeps along a strided axis (x, y, z, u_x, u_y).
//
// Eq. (3) (position advection, periodic) and Eq. (4) (velocity advection,
// zero-flux faces) of Yoshikawa, Tanaka & Yoshida, SC'21, one directional
// sweep at a time as in the split step of Eq. (5).
//
// f is viewed as a 3D tensor [O][L][I]: the swept axis (length L, stride I
// elements) between all slower axes (O) and all faster axes (I).  The GPU
// analogue of the paper's "SIMD over the second innermost loop" (Sec. 4.3):
// threads run over the contiguous inner index, each marching one whole line
// held in shared memory.
//
// Pipeline (one persistent CTA per SM slot):
//   warp 0, lane 0 (producer): TMA-loads box {W, L, P} tiles into a ring of
//     `stages` shared-memory buffers (mbarrier full[s] with transaction
//     bytes), and TMA-stores each finished tile back in place once the
//     consumers release it (mbarrier done[s]); a buffer is reloaded only after
//     the store has read it out.
//   warps 1..8 (consumers): one column each, sliding-window SL-MPP5 update in
//     shared memory, in place.
// Every wait is bounded: on expiry the kernel raises ERR_TIMEOUT in the error
// word and returns.
#include "vk_common.cuh"

namespace vk {

// The FP32 march of this kernel, with the flux written in the cells themselves (34
// operations a face) where every other kernel takes differences (31): over a drift of
// whole-cell shifts the two forms' roundings, both right to 7e-8 of the 2-norm, were driven
// apart in single cells by the limiter (3e-5 of the rms after six sweeps), more than these
// sweeps' results may change, for 4 % of their time (32 x 24 x 32 x 16 x 16 x 32 cells: 1.665
// against 1.597 ms, three sweeps).
__device__ __forceinline__ float minmod_curv(float d0, float d1)
{
    const float a = 4.f * d0 - d1, b = 4.f * d1 - d0;
    return mn2(mx2(mn2(mn3(a, b, d0), d1), 0.f), mx2(mx3(a, b, d0), d1));
}
__device__ __forceinline__ float cell_flux(const LineCoefT<float> &k, float cm2, float cm1, float c0, float cp1,
                                           float cp2, float dm4m, float dm4p)
{
    const float fbar = fmaf(k.w[4], cp2, fmaf(k.w[3], cp1, fmaf(k.w[2], c0, fmaf(k.w[1], cm1, k.w[0] * cm2))));
    const float dlm = c0 - cm1, ful = fmaf(k.alpha, dlm, c0), fmd = 0.5f * ((c0 + cp1) - dm4p);
    const float flc = fmaf(4.f / 3.f, dm4m, fmaf(0.5f, dlm, c0));
    const float v = mn3(mx3(fbar, mn3(c0, cp1, fmd), mn3(c0, ful, flc)), mx3(c0, cp1, fmd), mx3(c0, ful, flc));
    return flux_clamp(__fmul_rn(k.s, v), c0);
}
template <bool PERIODIC>
__device__ __forceinline__ float march_shift(float *p, long step, int L, const LineCoefT<float> &k)
{
    auto curv = [](float a, float b, float c) { return fmaf(-2.f, b, a) + c; };
    const float s0 = p[0], s1 = p[step];
    float cm2 = 0.f, cm1 = 0.f, c0 = s0, cp1 = s1, d = curv(0.f, s0, s1), q = minmod_curv(s0, d), Fm = 0.f, sum = 0.f;
    if (PERIODIC) {
        const float a = p[(long)(L - 3) * step];
        cm2 = p[(long)(L - 2) * step];
        cm1 = p[(long)(L - 1) * step];
        const float dm = curv(cm2, cm1, s0);
        d = curv(cm1, s0, s1);
        q = minmod_curv(dm, d);
        Fm = cell_flux(k, a, cm2, cm1, s0, s1, minmod_curv(curv(a, cm2, cm1), dm), q); // face -1/2, donor c_{-1}
    }
    auto face = [&](int i, float cp2, bool outer) {
        const float dn = curv(c0, cp1, cp2), qp = minmod_curv(d, dn);
        const float F = outer ? 0.f : cell_flux(k, cm2, cm1, c0, cp1, cp2, q, qp);
        const float out = c0 + (Fm - F);
        p[(long)i * step] = out;
        sum += out;
        cm2 = cm1;
        cm1 = c0;
        c0 = cp1;
        cp1 = cp2;
        d = dn;
        q = qp;
        Fm = F;
    };
#pragma unroll 4
    for (int i = 0; i < L - 2; ++i) face(i, p[(long)(i + 2) * step], false);
    face(L - 2, PERIODIC ? s0 : 0.f, false);
    face(L - 1, PERIODIC ? s1 : 0.f, !PERIODIC);
    return sum;
}
// The same on a periodic line, walked from its last cell down, with every new value written N
// cells on (0 <= N <= kStash, N < L): each row is read once and written once, where marching
// in place and rotating the line afterwards (three reversals) read and wrote it three times.
// Row i + N has been read when cell i is done; the N values that wrap around to the first
// rows, still to be read, wait in `held`, and the last three cells, overwritten before the
// first ones need them, in registers.  The values are march_shift's, face by face.  With tiles
// small enough for three CTAs per SM: 32 x 24 x 32 x 16 x 16 x 32 cells, x, y, z 0.600, 0.430, 0.643 ->
// 0.39 ms each (DRAM alone 0.238).
constexpr int kStash = 8;
__device__ __forceinline__ float march_shift_down(float *p, int step, int L, int N, const LineCoefT<float> &k)
{
    auto curv = [](float a, float b, float c) { return fmaf(-2.f, b, a) + c; };
    const float e3 = p[(L - 3) * step], e2 = p[(L - 2) * step], e1 = p[(L - 1) * step];
    const float s0 = p[0], s1 = p[step];
    float held[kStash], sum = 0.f;
    // face i + 1/2 from its upper side: donor c0 = cell i, cm1 = i - 1, ... ; start at i = L - 1
    float cp1 = s0, c0 = e1, cm1 = e2, cm2 = e3;
    float d = curv(cm1, c0, cp1), dm = curv(cm2, cm1, c0); // curvatures of cells i, i - 1
    float q = minmod_curv(dm, d);                          // at face i - 1/2
    float Fp = cell_flux(k, cm2, cm1, c0, cp1, s1, q, minmod_curv(d, curv(c0, cp1, s1)));
    auto cell = [&](float cm3) { // the next cell i down, with cell i - 3
        const float dmm = curv(cm3, cm2, cm1), qm = minmod_curv(dmm, dm);
        const float F = cell_flux(k, cm3, cm2, cm1, c0, cp1, qm, q); // face i - 1/2, donor cell i - 1
        const float out = c0 + (F - Fp);
        sum += out;
        cp1 = c0;
        c0 = cm1;
        cm1 = cm2;
        cm2 = cm3;
        dm = dmm;
        q = qm;
        Fp = F;
        return out;
    };
    int to = L - 1 + N; // where cell i goes; past the end of the line it wraps to row to - L
    auto put = [&](float v) {
        if (to < L) p[to * step] = v;
        else held[to - L] = v;
        --to;
    };
    const float *below = p + (L - 4) * step; // cell i - 3
#pragma unroll 4
    for (int i = L - 1; i >= 3; --i, below -= step) put(cell(*below));
    put(cell(e1));
    put(cell(e2));
    put(cell(e3));
    for (int j = 0; j < N; ++j) p[j * step] = held[j];
    return sum;
}

template <bool PERIODIC>
__device__ __forceinline__ double march_shift(double *p, long step, int L, const LineCoefT<double> &k)
{
    return march_line<double, PERIODIC, double>(p, step, L, to_lim(k));
}

template <typename T, bool PERIODIC>
__global__ void __launch_bounds__(kConsumers + kProducer)
    strided_sweep_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap dmap,
                         const __grid_constant__ StridedArgs<typename Compute<T>::type> args)
{
    using C = typename Compute<T>::type;
    extern __shared__ __align__(128) unsigned char smem[];
    const int S = args.stages;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem);
    uint64_t *done = full + S;
    LineCoefT<C> *tab = reinterpret_cast<LineCoefT<C> *>(smem + 128);
    const size_t tab_bytes = (args.coef_mode == 0) ? ((sizeof(LineCoefT<C>) * args.nvel + 127) & ~size_t(127)) : 0;
    T *stage0 = reinterpret_cast<T *>(smem + 128 + tab_bytes);
    const int L = args.L, W = args.W, P = args.P;
    const int tile_elems = W * L * P;
    const unsigned tile_bytes = unsigned(tile_elems * sizeof(T));
    // stage pitch in elements: each stage starts on a 128-byte boundary
    const size_t stage_elems = ((size_t(tile_bytes) + 127) & ~size_t(127)) / sizeof(T);

    if (threadIdx.x == 0) {
        for (int s = 0; s < S; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&done[s], kConsumers);
        }
        fence_barrier_init();
    }
    if (args.coef_mode == 0)
        for (int j = threadIdx.x; j < args.nvel; j += blockDim.x) tab[j] = args.table[j];
    __syncthreads();

    const long long G = gridDim.x, b = blockIdx.x;
    const long long n_my = (args.num_tiles > b) ? (args.num_tiles - b + G - 1) / G : 0;
    auto tile_coords = [&](long long t, int &ci, int &co) {
        const long long ti = t % args.tiles_inner;
        const long long to = t / args.tiles_inner;
        ci = int(ti * W);
        co = int(to * P);
    };

    if (threadIdx.x < kProducer) {
        if (threadIdx.x != 0) return;
        bool ok = true;
        long long issued = 0;
        for (long long k = 0; k < n_my; ++k) {
            const int st = int(k % S);
            if (k >= S) {
                const long long kp = k - S;
                if (!mbar_wait_bounded(&done[st], unsigned((kp / S) & 1))) { ok = false; break; }
                int ci, co;
                tile_coords(b + kp * G, ci, co);
                tma_store_3d(&dmap, stage0 + size_t(st) * stage_elems, ci, 0, co);
                bulk_commit();
                bulk_wait_read_all();
            }
            int ci, co;
            tile_coords(b + k * G, ci, co);
            mbar_arrive_expect_tx(&full[st], tile_bytes);
            tma_load_3d(stage0 + size_t(st) * stage_elems, &map, &full[st], ci, 0, co);
            ++issued;
        }
        if (ok) {
            for (long long kp = (n_my > S ? n_my - S : 0); kp < n_my; ++kp) {
                const int st = int(kp % S);
                if (!mbar_wait_bounded(&done[st], unsigned((kp / S) & 1))) { ok = false; break; }
                int ci, co;
                tile_coords(b + kp * G, ci, co);
                tma_store_3d(&dmap, stage0 + size_t(st) * stage_elems, ci, 0, co);
                bulk_commit();
            }
        }
        bulk_wait_all();
        if (!ok) {
            atomicOr(args.err, ERR_TIMEOUT);
            // let the loads still in flight land before the CTA's shared memory goes away
            for (long long t = (issued > S ? issued - S : 0); t < issued; ++t)
                mbar_wait_bounded(&full[t % S], unsigned((t / S) & 1));
        }
        return;
    }

    // consumers
    const int tid = threadIdx.x - kProducer;
    const int w = tid % W, p = tid / W;
    const bool has_col = tid < W * P;
    for (long long k = 0; k < n_my; ++k) {
        const int st = int(k % S);
        if (!mbar_wait_bounded(&full[st], unsigned((k / S) & 1))) {
            atomicOr(args.err, ERR_TIMEOUT);
            break;
        }
        const long long t = b + k * G;
        const long long inner = (t % args.tiles_inner) * W + w;
        const long long outer = (t / args.tiles_inner) * P + p;
        if (has_col && inner < args.n_inner && outer < args.n_outer) {
            LineCoefT<C> kc;
            if (args.coef_mode == 0)
                kc = tab[(inner / args.vstride) % args.nvel];
            else
                kc = args.cell_coef[outer / args.outer_per_cell];
            if (kc.nd >= 0) {
                const int N = kc.nd >> 1;
                const bool neg = kc.nd & 1;
                T *col = stage0 + size_t(st) * stage_elems + size_t(p) * L * W + w;
                T *base = neg ? col + size_t(L - 1) * W : col;
                const long step = neg ? -long(W) : long(W);
                C sum;
                if constexpr (PERIODIC && sizeof(T) == 4) {
                    if (N % L <= kStash && N % L < L) {
                        sum = march_shift_down(base, int(step), L, N % L, kc);
                    } else {
                        sum = march_shift<PERIODIC>(base, step, L, kc);
                        rotate_line(base, step, L, N % L);
                    }
                } else {
                    sum = march_shift<PERIODIC>(base, step, L, kc);
                    if (PERIODIC && N != 0) rotate_line(base, step, L, N % L);
                }
                if (!(sum >= C(0)) || isinf(sum)) atomicOr(args.err, ERR_NAN);
            }
        }
        fence_proxy_async();
        mbar_arrive(&done[st]);
    }
}

template <typename T>
static cudaError_t launch_strided_t(const CUtensorMap &map, const CUtensorMap &dmap, const StridedArgs<typename Compute<T>::type> &a,
                                    int grid, size_t smem, cudaStream_t st)
{
    auto kern = a.periodic ? strided_sweep_kernel<T, true> : strided_sweep_kernel<T, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    kern<<<grid, kConsumers + kProducer, smem, st>>>(map, dmap, a);
    return cudaGetLastError();
}

cudaError_t launch_strided_f32(const CUtensorMap &map, const CUtensorMap &dmap, const StridedArgs<float> &a, int grid, size_t smem,
                               cudaStream_t st)
{
    return launch_strided_t<float>(map, dmap, a, grid, smem, st);
}

cudaError_t launch_strided_f64(const CUtensorMap &map, const CUtensorMap &dmap, const StridedArgs<double> &a, int grid, size_t smem,
                               cudaStream_t st)
{
    return launch_strided_t<double>(map, dmap, a, grid, smem, st);
}

int occupancy_strided(int dtype, int periodic, size_t smem)
{
    const void *k;
    if (dtype == 0)
        k = periodic ? (const void *)strided_sweep_kernel<double, true> : (const void *)strided_sweep_kernel<double, false>;
    else
        k = periodic ? (const void *)strided_sweep_kernel<float, true> : (const void *)strided_sweep_kernel<float, false>;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess) return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, kConsumers + kProducer, smem) != cudaSuccess) return 0;
    return n;
}

} // namespace vk
