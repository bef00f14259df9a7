// sweep_shift32.cu -- position sweeps of Eq. (3) that shift whole cells (|nu| >= 1 on some line)
// on FP32 storage, whole lines staged in shared memory, two lines per thread.
//
// The tiles, the ring and its producer are those of sweep_pair32.cu (tiles of 128 columns, a
// group of threads per tile); each thread marches two adjacent lines down and writes every cell
// in its shifted place (march_shift_down, vk_shift.cuh), so lines may shift by different numbers
// of cells.  When some line shifts by more cells than a thread can hold back, all lines of the sweep are
// marched in place and rotated (whole_cell_rotate).
//
// Against one line per thread in three CTAs of 8 warps an SM (sweep_strided.cu with tiles of 36 KB, whose
// warps wait for each other at every tile, and 64-bit divisions per line): 32 x 24 x 32 x 16 x 16 x 32 cells
// (DRAM alone 0.238 ms a sweep) x, y, z 0.386, 0.412, 0.389 -> 0.335, 0.355, 0.340 ms, 16^3 x 32^3
// 0.311 -> 0.268 (0.159); one line per thread in this ring 0.352, 0.375, 0.355 and 0.286.  Bound by
// the marches: the flux in the cells themselves takes 28 ALU cycles a line and face.
#include "vk_shift.cuh"
#include "vk_tiles.cuh"

namespace vk {

namespace {

constexpr int kCols = 128, kRow = kCols * 4; // columns of a tile, bytes of a row
constexpr int kGroup = kCols / 2;            // threads of a group
constexpr int kMaxGroups = 8, kMaxSlots = 24; // (11 groups, 80 registers: 0.347-0.350 ms, 16^3 x 32^3 0.257)
constexpr int kHead = ((3 * kMaxSlots * 8 + 127) & ~127) + int(kMaxVel * sizeof(LineCoefT<float>));

// ROT: lines marched in place one by one and rotated (Pair32Args::rotate)
template <bool ROT>
__global__ void __launch_bounds__(kMaxGroups *kGroup + kProducer, 1)
    shift32_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap dmap,
                  const __grid_constant__ Pair32Args a)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int L = a.L, S = a.slots, NT = a.groups * kGroup;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem); // 2S: the slot holds its tile (full_bar)
    uint64_t *done = full + 2 * S;                       // S: the tile's group is done with it
    LineCoefT<float> *tab = reinterpret_cast<LineCoefT<float> *>(smem + ((3 * kMaxSlots * 8 + 127) & ~127));
    unsigned char *ring = smem + kHead + ((128u - ((smem_u32(smem) + unsigned(kHead)) & 127u)) & 127u);
    auto slot = [&](unsigned k) { return ring + size_t(L) * kRow * (k % S); };

    if (threadIdx.x == 0) {
        for (int q = 0; q < 2 * S; ++q) mbar_init(&full[q], 1);
        for (int q = 0; q < S; ++q) mbar_init(&done[q], kGroup);
        fence_barrier_init();
    }
    for (int j = threadIdx.x; j < a.nvel; j += blockDim.x) tab[j] = a.table[j];
    __syncthreads();
    chain_enter();

    const unsigned G = gridDim.x, b = blockIdx.x; // every tile and column index fits 32 bits (host)
    const unsigned n_my = a.num_tiles > b ? (a.num_tiles - b + G - 1) / G : 0;
    auto coords = [&](unsigned k, unsigned &ti, unsigned &o) {
        const unsigned t = b + k * G;
        o = fdiv(t, a.div_tiles);
        ti = t - o * a.tiles_inner;
    };

    if (threadIdx.x >= unsigned(NT)) {
        if (threadIdx.x != unsigned(NT)) return;
        auto load = [&](unsigned k) {
            unsigned ti, o;
            coords(k, ti, o);
            uint64_t *bar = full_bar(full, k, S);
            mbar_arrive_expect_tx(bar, unsigned(L) * kRow); // the whole box, clipped or not
            tma_load_3d(slot(k), &map, bar, int(ti * kCols), 0, int(o));
        };
        unsigned loaded = 0;
        for (; loaded < unsigned(S) && loaded < n_my; ++loaded) load(loaded);
        bool ok = true;
        for (unsigned k = 0; k < n_my; ++k) {
            if (!mbar_wait_bounded(&done[k % S], (k / S) & 1u)) {
                ok = false;
                break;
            }
            unsigned ti, o;
            coords(k, ti, o);
            tma_store_3d(&dmap, slot(k), int(ti * kCols), 0, int(o));
            bulk_commit();
            // reload the slot of tile k - lag: `lag` later stores may still be reading theirs
            if (k >= unsigned(a.lag) && loaded < n_my) {
                bulk_wait_read_at_most(a.lag);
                load(loaded++);
            }
        }
        bulk_wait_all();
        if (!ok) {
            atomicOr(a.err, ERR_TIMEOUT);
            // let the loads in flight (the last S at most) land before the CTA exits
            for (unsigned k = loaded > unsigned(S) ? loaded - S : 0; k < loaded; ++k) wait_tile(full, k, S);
        }
        return;
    }

    const int grp = threadIdx.x / kGroup, tid = threadIdx.x % kGroup;
    bool bad = false;
    for (unsigned k = grp; k < n_my; k += a.groups) {
        if (!__all_sync(0xffffffffu, wait_tile(full, k, S))) {
            atomicOr(a.err, ERR_TIMEOUT);
            return;
        }
        unsigned ti, o;
        coords(k, ti, o);
        const unsigned inner = ti * kCols + 2u * tid; // the thread's first column
        const unsigned qa = fdiv(inner, a.div_vstride), qb = fdiv(inner + 1, a.div_vstride); // (inner / vstride) % nvel
        const LineCoefT<float> ka = tab[qa - fdiv(qa, a.div_nvel) * unsigned(a.nvel)];
        const LineCoefT<float> kb = tab[qb - fdiv(qb, a.div_nvel) * unsigned(a.nvel)];
        if (ka.nd >= 0) {
            // a negative Courant number is the mirror image: march the line from its far end
            const bool neg = ka.nd & 1;
            auto shift = [&](int N) { return N < L ? N : N % L; };
            const int Na = shift(ka.nd >> 1), Nb = shift(kb.nd >> 1), step = neg ? -kGroup : kGroup; // rows in pairs
            float2 *p = reinterpret_cast<float2 *>(slot(k)) + tid + (neg ? (L - 1) * kGroup : 0);
            float2 sum;
            // (columns past the end of a row hold zeros: marched, never stored)
            if constexpr (ROT) {
                auto line = [&](float *q, int N, const LineCoefT<float> &kc) {
                    const float s = march_shift(q, long(2 * step), L, kc);
                    rotate_line(q, long(2 * step), L, N);
                    return s;
                };
                sum.x = line(&p->x, Na, ka);
                sum.y = line(&p->y, Nb, kb);
            } else {
                sum = march_shift_down(p, step, L, Na, Nb, ka, kb);
            }
            bad |= !(sum.x >= 0.f) || !(sum.y >= 0.f) || isinf(sum.x) || isinf(sum.y);
        }
        fence_proxy_async();
        mbar_arrive(&done[k % S]);
    }
    if (bad) atomicOr(a.err, ERR_NAN);
}

} // namespace

cudaError_t launch_shift32(const CUtensorMap &map, const CUtensorMap &dmap, const Pair32Args &args, int grid, cudaStream_t st)
{
    if (args.num_tiles == 0 || grid <= 0) return cudaSuccess;
    Pair32Args a = args; // slots and lag are pair32_geometry's: the ring is the same
    a.groups = a.slots - (a.slots >= 12 ? a.slots / 3 : 1);
    if (a.groups > kMaxGroups) a.groups = kMaxGroups;
    if (a.groups < 1 || a.slots > kMaxSlots || a.nvel <= 0 || a.nvel > kMaxVel ||
        a.vstride <= 0 || a.vstride * a.nvel % 4)
        return cudaErrorInvalidValue;
    a.div_tiles = make_fastdiv(a.tiles_inner);
    a.div_vstride = make_fastdiv(unsigned(a.vstride));
    a.div_nvel = make_fastdiv(unsigned(a.nvel));
    const size_t smem = kHead + 128 + size_t(a.slots) * a.L * kRow;
    const void *kern = a.rotate ? (const void *)shift32_kernel<true> : (const void *)shift32_kernel<false>;
    const cudaError_t e = allow_smem(kern, smem);
    if (e != cudaSuccess) return e;
    void *params[] = {const_cast<CUtensorMap *>(&map), const_cast<CUtensorMap *>(&dmap), &a};
    return launch_chained((long long)a.num_tiles * kCols * a.L, kern, dim3(grid),
                          dim3(a.groups * kGroup + kProducer), smem, st, params);
}

} // namespace vk
