// sweep_tile16.cu -- position sweeps D_x, D_y, D_z of Eq. (3) (|nu| < 1) and the u_x sweep of
// Eq. (4) on 16-bit storage (BF16 / FP16 codes, one FP32 scale per u_z line), whole lines
// staged in shared memory, two lines per thread.
//
// f is viewed as [O][L][I] (slower axes, the swept axis, the faster axes; for u_x: cells,
// j_x, j_y j_z) and I cut into tiles of 256 contiguous columns: a tile is every cell of 256
// lines, one TMA box {32, 8, L} of codes (512-byte rows) plus the box of the scales of its
// u_z lines.  These sweeps keep every scale: a value is decoded as code x scale (a rounded
// product), its line marched in FP32 and the result encoded with stochastic rounding.
//
// They are bound by the marches and the codec, not by DRAM (4 bytes a cell and pass).  A thread takes two adjacent columns, which always share their u_z line and the
// sign of their Courant number: one 4-byte access, one scale and one inverse scale serve
// two cells, and the march's sums and products run as f32x2 pairs (March<float2>).  Groups
// of 128 threads march different tiles of a ring that one producer thread keeps full.  The
// length of the lines and the length of a u_z line are run-time values: bodies of 4, 2
// and 1 faces serve every shape and stay small (unrolled bodies that grow past the
// instruction cache cost far more than the loop).  The codes and scales of a body are read
// ahead of its marches, since the compiler cannot tell a row read from a row written.
// Measured: BF16 32^3 x 32^3, one sweep 1.80-2.20 ms with one line per thread in unrolled
// bodies, 1.60 with pairs and run-time strides, 1.44-1.49 here (77 instructions per face pair,
// issue 70 % busy; DRAM alone 0.67 ms); bodies of 8 faces for both directions missed in the
// instruction cache (1.77).  FP16 24^3 x 48^3: 5.0-8.1 ms streamed, 2.26-2.33 here.
// Scale and inverse scale of every u_z line and row a warp needs are put side by side in
// shared memory once per warp and tile.
#include <type_traits>

#include "vk_tiles.cuh"

namespace vk {

namespace {

constexpr int kPairGroup = 128; // threads of a group: the pairs of a tile
constexpr int kPairGroups = 4;

// The draws of two columns, 16 bits a value: the upper halves of two states, a step on per row.
struct PairDraws {
    unsigned x, y;
    Lcg step;
    __device__ void next()
    {
        x = step(x);
        y = step(y);
    }
};

template <typename T> struct PairCodec;
template <> struct PairCodec<__nv_bfloat16> {
    __device__ static float2 get(unsigned u, float s) // a bf16 is the upper half of an FP32
    {
        return vmul(make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u)), make_float2(s, s));
    }
    __device__ static unsigned put(float2 v, float inv, PairDraws &r)
    {
        const float2 c = vmul(v, make_float2(inv, inv));
        const unsigned u = sr_pack_bf16x2(c.x, c.y, r.x >> 16, r.y >> 16);
        r.next();
        return u;
    }
};
template <> struct PairCodec<__half> {
    __device__ static float2 get(unsigned u, float s)
    {
        return vmul(__half22float2(*reinterpret_cast<const __half2 *>(&u)), make_float2(s, s));
    }
    __device__ static unsigned put(float2 v, float inv, PairDraws &r)
    {
        const float2 c = vmul(v, make_float2(inv, inv));
        const unsigned u = sr_pack_f16x2(c.x, c.y, r.x >> 16, r.y >> 16);
        r.next();
        return u;
    }
};

// March the two lines whose row r holds codes at p + r st (bytes) and (scale, inverse scale)
// at sp + r sd.  DIR = +1 / -1: consecutive rows walked forward / backward, strides fixed at
// compile time; 0: taken at run time (st, sd).  ZF: zero-flux lines, else periodic.  L >= 4.
// Returns the sums of the new values.
template <typename T, bool ZF, int DIR>
__device__ __forceinline__ float2 march_pair16(unsigned char *p, int st_rt, const float2 *sp, int sd_rt, int L,
                                               const Lim<float2> &lim, PairDraws rng)
{
    const int st = DIR ? DIR * 512 : st_rt, sd = DIR ? DIR : sd_rt;
    auto code = [&](int r) -> unsigned & { return *reinterpret_cast<unsigned *>(p + r * st); };
    auto get = [&](int r) { return PairCodec<T>::get(code(r), sp[r * sd].x); };
    const float2 s0 = get(0), s1 = get(1);
    March<float2> m(lim);
    if (ZF) m.start_zero(s0, s1);
    else m.start_periodic(get(L - 3), get(L - 2), get(L - 1), s0, s1);
    // B faces whose look-ahead cells lie on the line: read them all, then march
    auto block = [&](auto width) {
        constexpr int B = decltype(width)::value;
        unsigned c[B];
        float2 s[B + 2]; // of rows 0 .. B + 1
#pragma unroll
        for (int q = 0; q < B + 2; ++q) s[q] = sp[q * sd];
#pragma unroll
        for (int q = 0; q < B; ++q) c[q] = code(q + 2);
#pragma unroll
        for (int q = 0; q < B; ++q) code(q) = PairCodec<T>::put(m.face(PairCodec<T>::get(c[q], s[q + 2].x)), s[q].y, rng);
        p += B * st;
        sp += B * sd;
    };
    int left = L - 2;
#pragma unroll 1
    for (; left >= 4; left -= 4) block(std::integral_constant<int, 4>());
    // a rolled single face spends more on moving the window than on the face
    if (left & 2) block(std::integral_constant<int, 2>());
    if (left & 1) block(std::integral_constant<int, 1>());
    code(0) = PairCodec<T>::put(m.face(ZF ? make_float2(0.f, 0.f) : s0), sp[0].y, rng);
    code(1) = PairCodec<T>::put(ZF ? m.last() : m.face(s1), sp[sd].y, rng);
    return m.sum;
}

template <typename T, bool ZF>
__global__ void __launch_bounds__(kPairGroups *kPairGroup + kProducer, 1)
    tile_pair16_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap smap,
                       const __grid_constant__ Tile16Args a)
{
    extern __shared__ __align__(128) unsigned char smem[];
    const int L = a.L, S = a.slots, NT = a.groups * kPairGroup, SX = a.scale_lines;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem); // 2S: the slot holds its tile (full_bar)
    uint64_t *done = full + 2 * S;                       // S: the tile's group is done with it
    LineCoefT<float> *tab = reinterpret_cast<LineCoefT<float> *>(smem + kTileBars);
    static_assert(3 * kTileSlots * 8 <= kTileBars, "barriers fit ahead of the table");
    unsigned char *ring = smem + kTileHeader + ((1024u - ((smem_u32(smem) + unsigned(kTileHeader)) & 1023u)) & 1023u);
    auto slot = [&](unsigned k) { return ring + size_t(a.slot_bytes) * (k % S); };
    auto sslot = [&](unsigned k) { return reinterpret_cast<float *>(slot(k) + unsigned(L) * 512u); };
    float2 *wscale = reinterpret_cast<float2 *>(ring + size_t(a.slot_bytes) * S);

    if (threadIdx.x == 0) {
        for (int q = 0; q < 2 * S; ++q) mbar_init(&full[q], 1);
        for (int q = 0; q < S; ++q) mbar_init(&done[q], kPairGroup);
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
    // first u_z line of the tile's scale box: a multiple of 4 (the 16-byte rule of TMA)
    auto line0 = [&](unsigned ti) { return fdiv(256u * ti, a.div_nuz) & ~3u; };

    if (threadIdx.x >= unsigned(NT)) {
        if (threadIdx.x != unsigned(NT)) return;
        auto load = [&](unsigned k) {
            unsigned ti, o;
            coords(k, ti, o);
            uint64_t *bar = full_bar(full, k, S);
            mbar_arrive_expect_tx(bar, unsigned(L) * 512u + unsigned(L) * 4u * unsigned(SX));
            tma_load_4d(slot(k), &map, bar, 0, int(8 * ti), 0, int(o));
            tma_load_3d(sslot(k), &smap, bar, int(line0(ti)), 0, int(o));
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
            tma_store_4d(&map, slot(k), 0, int(8 * ti), 0, int(o)); // the scales stay as they are
            bulk_commit();
            if (loaded < n_my) {
                bulk_wait_read_all(); // the slot is free once the store has read it
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

    const int grp = threadIdx.x / kPairGroup, tid = threadIdx.x % kPairGroup, w = tid >> 5, lane = tid & 31;
    // this warp's scales and inverse scales, [line][row]
    float2 *ws = wscale + (grp * (kPairGroup / 32) + w) * a.warp_lines * L;
    // the thread's pair of the tile.  z sweep of u_z lines that divide a tile: warps 0, 1 take the
    // pairs with u_z < 0, warps 2, 3 those with u_z > 0, so that each walks in one direction
    int pair = tid, wcol = 64 * w; // and the first column of the warp's lines
    if (a.zperm) {
        const int half = a.nuz / 4, n = tid & 63; // pairs of one sign per line
        pair = (n / half) * (a.nuz / 2) + (w >> 1) * half + n % half;
        wcol = 128 * (w & 1);
    }
    bool bad = false;
    for (unsigned k = grp; k < n_my; k += a.groups) {
        if (!__all_sync(0xffffffffu, wait_tile(full, k, S))) {
            atomicOr(a.err, ERR_TIMEOUT);
            return;
        }
        unsigned ti, o;
        coords(k, ti, o);
        const unsigned inner = 256u * ti + 2u * pair, c0 = 256u * ti + wcol; // the thread's and the warp's first column
        const unsigned x0 = line0(ti), first = fdiv(c0, a.div_nuz), line = fdiv(inner, a.div_nuz);
        const int nlines = int(fdiv(c0 + (a.zperm ? 127u : 63u), a.div_nuz) - first) + 1;
        const float *sp = sslot(k) + int(first - x0);
        __syncwarp(); // every lane is done with the previous tile's scales
        for (int h = 0; h < nlines; ++h)
            for (int r = lane; r < L; r += 32) {
                const float s = sp[r * SX + h];
                ws[h * L + r] = make_float2(s, inv_scale(s));
            }
        __syncwarp();
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
            const int far = neg ? L - 1 : 0, dir = neg ? -1 : 1;
            // the streams, from the index of the first cell of the pair or of each column
            const unsigned long long e = (unsigned long long)o * L * a.n_inner + inner;
            const unsigned seed = sr_bits(e, a.seed);
            const unsigned seed2 = a.own ? sr_bits(e + 1, a.seed) : seed;
            // (a fixed index keeps the step in the constant bank)
            auto rng = [&](int d) { return PairDraws{a.draws[d].x(seed), a.draws[d].y(seed2), a.draws[d].step}; };
            unsigned char *p = slot(k) + 4 * pair + far * 512;
            const float2 *s = ws + int(line - first) * L + far;
            float2 sum;
            if (__all_sync(0xffffffffu, !neg)) sum = march_pair16<T, ZF, 1>(p, 0, s, 0, L, lim, rng(0));
            else if (__all_sync(0xffffffffu, neg)) sum = march_pair16<T, ZF, -1>(p, 0, s, 0, L, lim, rng(1));
            else sum = march_pair16<T, ZF, 0>(p, dir * 512, s, dir, L, lim, rng(neg));
            bad |= !(sum.x >= 0.f) || !(sum.y >= 0.f) || isinf(sum.x) || isinf(sum.y);
        }
        fence_proxy_async();
        mbar_arrive(&done[k % S]);
    }
    if (bad) atomicOr(a.err, ERR_NAN);
}

const void *pair16_kernel(int dtype, bool zf)
{
    if (dtype == 2)
        return zf ? (const void *)tile_pair16_kernel<__nv_bfloat16, true> : (const void *)tile_pair16_kernel<__nv_bfloat16, false>;
    if (dtype == 3) return zf ? (const void *)tile_pair16_kernel<__half, true> : (const void *)tile_pair16_kernel<__half, false>;
    return nullptr;
}

size_t pair16_smem(const Tile16Args &a)
{
    return kTileHeader + 1024 + size_t(a.slots) * a.slot_bytes +
           size_t(a.groups) * (kPairGroup / 32) * a.warp_lines * a.L * sizeof(float2);
}

} // namespace

// A ring of at least three slots has to fit: lines of up to about 100 cells.
bool tile16_geometry(int L, long long n_inner, long long n_outer, int nuz, bool z, Tile16Args &a)
{
    if (L < 4 || n_inner % 256 || nuz < 4 || nuz % 4 || n_inner % nuz || (n_inner / nuz) % 4) return false;
    if (n_inner > 0x7fffffffll || n_outer * (n_inner / 256) > 0x7fffffffll) return false;
    a.L = L;
    a.nuz = nuz;
    a.n_inner = n_inner;
    a.tiles_inner = unsigned(n_inner / 256);
    // a tile's u_z lines: exactly 256 / n_uz, or the most 256 columns can touch after the up
    // to three lines ahead of them that the alignment of the box brings
    a.scale_lines = 256 % nuz == 0 ? 256 / nuz : (((255 / nuz) + 2 + 3 + 3) & ~3);
    if (a.scale_lines % 4 || a.scale_lines > 256) return false;
    a.zperm = z && 128 % nuz == 0 && nuz >= 8;
    a.warp_lines = a.zperm ? 128 / nuz : 64 % nuz == 0 ? 64 / nuz : 63 / nuz + 2;
    a.slot_bytes = unsigned((L * (512 + 4 * a.scale_lines) + 127) & ~127);
    const size_t limit = 227 * 1024;
    for (a.groups = kPairGroups; a.groups >= 2; --a.groups) { // one slot more than the groups, at least
        a.slots = 0;
        const size_t rest = pair16_smem(a);
        const int s = rest < limit ? int((limit - rest) / a.slot_bytes) : 0;
        a.slots = s < kTileSlots ? s : kTileSlots;
        if (a.slots > a.groups) break;
    }
    return a.groups >= 2;
}

int occupancy_tile16(const Tile16Args &a, int dtype, bool zf)
{
    const void *k = pair16_kernel(dtype, zf);
    if (!k) return 0;
    const size_t smem = pair16_smem(a);
    if (allow_smem(k, smem) != cudaSuccess) return 0;
    int n = 0;
    const int threads = a.groups * kPairGroup + kProducer;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, smem) != cudaSuccess) return 0;
    return n;
}

// Which streams a shape draws: those it has always drawn, whichever kernel took it.  16-bit results
// then repeat but for the last bit of the FP32 march.
//   own, walk order: one stream per column, a draw per cell as the line is walked (position lines of
//     16 to 96 cells with n_uz = 32, lines of 48 with n_uz = 48);
//   own, memory order: the same from the line's first cell on (u_x lines of 48 with other n_uz, as
//     the register-line kernel);
//   pair, memory order: one stream per two columns (all others: the streamed sweep's bits).
// A line walked against memory order takes its draws backward.
static void set_draws(Tile16Args &a, bool zf)
{
    const int L = a.L;
    const bool walk = a.nuz == 48 ? L == 48 : !zf && a.nuz == 32 && (L == 16 || L == 24 || L == 32 || L == 48 || L == 64 || L == 96);
    a.own = walk || (zf && L == 48);
    const int n = a.own ? 1 : 2; // draws of a stream per row
    a.draws[0] = a.draws[1] = {kLcg, lcg_power(kLcg, n), lcg_power(kLcg, n)};
    if (!walk) a.draws[1] = {lcg_power(kLcg, n * (L - 1) + 1), lcg_power(kLcg, n * L), lcg_power(kLcgBack, n)};
}

cudaError_t launch_tile16(const CUtensorMap &map, const CUtensorMap &smap, const Tile16Args &args, int dtype, int grid,
                          cudaStream_t st)
{
    if (args.num_tiles == 0 || grid <= 0) return cudaSuccess;
    const bool zf = args.cell_coef != nullptr;
    const void *k = pair16_kernel(dtype, zf);
    // two adjacent columns share their line's direction: the sign of u changes at whole pairs
    if (!k || args.groups < 2 || args.slots <= args.groups ||
        (!zf && (args.nvel <= 0 || args.nvel > kMaxVel || args.vstride <= 0 || args.vstride * args.nvel % 4)))
        return cudaErrorInvalidValue;
    Tile16Args a = args;
    a.div_tiles = make_fastdiv(a.tiles_inner);
    a.div_nuz = make_fastdiv(unsigned(a.nuz));
    a.div_vstride = make_fastdiv(unsigned(a.vstride > 0 ? a.vstride : 1));
    a.div_nvel = make_fastdiv(unsigned(a.nvel > 0 ? a.nvel : 1));
    set_draws(a, zf);
    const size_t smem = pair16_smem(a);
    cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    void *params[] = {const_cast<CUtensorMap *>(&map), const_cast<CUtensorMap *>(&smap), &a};
    return launch_chained((long long)a.num_tiles * 256 * a.L, k, dim3(grid), dim3(a.groups * kPairGroup + kProducer), smem, st, params);
}

} // namespace vk
