// sweep_pair32.cu -- position sweeps D_x, D_y, D_z of Eq. (3) (|nu| < 1) and the u_x sweep of
// Eq. (4) on FP32 storage for lines of any length (from 9 cells; shorter ones mostly stream),
// whole lines staged in shared memory, two lines per thread.
//
// f is viewed as [O][L][I] (slower axes, the swept axis, the faster axes; for u_x: cells,
// j_x, j_y j_z) and I cut into tiles of 128 contiguous columns, the last one of a row partial
// (TMA fills and clips it): a tile is every cell of 128 lines, one TMA box {128, L}.  Groups
// of 64 threads march different tiles of a ring that one producer thread keeps full; a
// thread takes two adjacent columns, which always share the sign of their Courant number
// (it changes at multiples of n_uz / 2, an even number), by one 8-byte access a row, the march's
// sums and products in f32x2 pairs (March<float2>).  Sizes are run-time values; bodies of 4,
// 2 and 1 faces stay small, and the cells of a body are read ahead of its first write (the
// compiler cannot tell a row read from a row written).
//
// Against the streamed sweep, whose blocks walk a line in chunks of four rows, a line's cells
// are in flight at once and no thread waits between its rows: 21 x 26 x 19 x 24 x 20 x 28 cells
// (DRAM alone 0.165 ms a sweep) x, y, z 0.262, 0.306, 0.299 -> 0.209, 0.192, 0.228 ms, u_x 0.299
// -> 0.221; 32^3 x 32^3 y, z 1.44 (one line per thread, sweep_tile.cu) -> 1.31 ms.
#include <type_traits>

#include "vk_tiles.cuh"

namespace vk {

namespace {

constexpr int kCols = 128, kRow = kCols * 4; // columns of a tile, bytes of a row
constexpr int kGroup = kCols / 2;            // threads of a group
constexpr int kMaxGroups = 8, kMaxSlots = 24;
constexpr int kHead = ((3 * kMaxSlots * 8 + 127) & ~127) + int(kMaxVel * sizeof(LineCoefT<float>));

// March the two lines whose row r holds its cells at p + r st (bytes).  DIR = +1 / -1: rows
// walked forward / backward, the stride fixed at compile time; 0: taken at run time.  ZF:
// zero-flux lines, else periodic.  L >= 4.  Returns the sums of the new values.
template <bool ZF, int DIR>
__device__ __forceinline__ float2 march_pair(unsigned char *p, int st_rt, int L, const Lim<float2> &lim)
{
    const int st = DIR ? DIR * kRow : st_rt;
    auto cell = [&](int r) -> float2 & { return *reinterpret_cast<float2 *>(p + r * st); };
    const float2 s0 = cell(0), s1 = cell(1);
    March<float2> m(lim);
    if (ZF) m.start_zero(s0, s1);
    else m.start_periodic(cell(L - 3), cell(L - 2), cell(L - 1), s0, s1);
    auto block = [&](auto width) { // faces whose look-ahead cells lie on the line
        constexpr int B = decltype(width)::value;
        float2 c[B];
#pragma unroll
        for (int q = 0; q < B; ++q) c[q] = cell(q + 2);
#pragma unroll
        for (int q = 0; q < B; ++q) cell(q) = m.face(c[q]);
        p += B * st;
    };
    int left = L - 2;
#pragma unroll 1
    for (; left >= 4; left -= 4) block(std::integral_constant<int, 4>());
    if (left & 2) block(std::integral_constant<int, 2>());
    if (left & 1) block(std::integral_constant<int, 1>());
    cell(0) = m.face(ZF ? make_float2(0.f, 0.f) : s0);
    cell(1) = ZF ? m.last() : m.face(s1);
    return m.sum;
}

template <bool ZF>
__global__ void __launch_bounds__(kMaxGroups *kGroup + kProducer, 1)
    pair32_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap dmap,
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
        const unsigned t = a.tile0 + b + k * G;
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
        LineCoefT<float> ka, kb;
        if constexpr (ZF) {
            ka = kb = a.cell_coef[o];
        } else {
            // columns inner, inner + 1: (inner / vstride) % nvel
            const unsigned qa = fdiv(inner, a.div_vstride), qb = fdiv(inner + 1, a.div_vstride);
            ka = tab[qa - fdiv(qa, a.div_nvel) * unsigned(a.nvel)];
            kb = tab[qb - fdiv(qb, a.div_nvel) * unsigned(a.nvel)];
        }
        if (ka.nd >= 0) {
            const Lim<float2> lim = to_lim2(ka, kb);
            // a negative Courant number is the mirror image: march the line from its far end
            const bool neg = ka.nd & 1;
            unsigned char *p = slot(k) + 8 * tid + (neg ? (L - 1) * kRow : 0);
            float2 sum;
            // (columns past the end of a row hold zeros: marched, never stored)
            if (__all_sync(0xffffffffu, !neg)) sum = march_pair<ZF, 1>(p, 0, L, lim);
            else if (__all_sync(0xffffffffu, neg)) sum = march_pair<ZF, -1>(p, 0, L, lim);
            else sum = march_pair<ZF, 0>(p, neg ? -kRow : kRow, L, lim);
            bad |= !(sum.x >= 0.f) || !(sum.y >= 0.f) || isinf(sum.x) || isinf(sum.y);
        }
        fence_proxy_async();
        mbar_arrive(&done[k % S]);
    }
    if (bad) atomicOr(a.err, ERR_NAN);
}

const void *pair32(bool zf) { return zf ? (const void *)pair32_kernel<true> : (const void *)pair32_kernel<false>; }

size_t pair32_smem(const Pair32Args &a) { return kHead + 128 + size_t(a.slots) * a.L * kRow; }

} // namespace

int pair32_columns() { return kCols; }

// a ring of at least four slots has to fit: lines of up to about 110 cells
bool pair32_geometry(int L, long long n_inner, long long n_outer, Pair32Args &a)
{
    const long long tiles = (n_inner + kCols - 1) / kCols;
    if (L < 4 || L > 256 || n_inner < 4 || n_inner % 4 || n_inner > 0x7fffff00ll || n_outer * tiles > 0x7fffffffll) return false;
    a.L = L;
    a.tiles_inner = unsigned(tiles);
    const int fit = int((227 * 1024 - kHead - 128) / (L * kRow));
    a.slots = fit < kMaxSlots ? fit : kMaxSlots;
    if (a.slots < 4) return false;
    // a ring slot or more ahead of the groups, a third of the ring for long rings
    a.groups = a.slots - (a.slots >= 12 ? a.slots / 3 : 1);
    if (a.groups > kMaxGroups) a.groups = kMaxGroups;
    a.lag = a.slots >= 12 ? 3 : 0; // short tiles: the producer does not wait for each store
    return true;
}

int occupancy_pair32(const Pair32Args &a, bool zf)
{
    const size_t smem = pair32_smem(a);
    if (allow_smem(pair32(zf), smem) != cudaSuccess) return 0;
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, pair32(zf), a.groups * kGroup + kProducer, smem) != cudaSuccess) return 0;
    return n;
}

cudaError_t launch_pair32(const CUtensorMap &map, const CUtensorMap &dmap, const Pair32Args &args, int grid, cudaStream_t st)
{
    if (args.num_tiles == 0 || grid <= 0) return cudaSuccess;
    const bool zf = args.cell_coef != nullptr;
    // two adjacent columns share their line's direction: the sign of u changes at whole pairs
    if (args.groups < 1 || args.slots < args.groups || args.lag < 0 || args.lag >= args.slots ||
        (!zf && (args.nvel <= 0 || args.nvel > kMaxVel || args.vstride <= 0 || args.vstride * args.nvel % 4)))
        return cudaErrorInvalidValue;
    Pair32Args a = args;
    a.div_tiles = make_fastdiv(a.tiles_inner);
    a.div_vstride = make_fastdiv(unsigned(a.vstride > 0 ? a.vstride : 1));
    a.div_nvel = make_fastdiv(unsigned(a.nvel > 0 ? a.nvel : 1));
    const size_t smem = pair32_smem(a);
    cudaError_t e = allow_smem(pair32(zf), smem);
    if (e != cudaSuccess) return e;
    void *params[] = {const_cast<CUtensorMap *>(&map), const_cast<CUtensorMap *>(&dmap), &a};
    return launch_chained((long long)a.num_tiles * kCols * a.L, pair32(zf), dim3(grid), dim3(a.groups * kGroup + kProducer), smem, st, params);
}

} // namespace vk
