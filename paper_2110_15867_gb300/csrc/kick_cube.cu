// kick_cube.cu -- one kick of Eq. (5), D_uz D_uy D_ux, in a single pass over f.
//
// Every spatial cell owns its whole velocity cube (Listing 1: u_z innermost) and a
// kick never leaves the cell (Sec. 4.1.3: the velocity sweeps need no exchange), so
// a CTA can take one cube of NU^3 cells (NU = n_ux = n_uy = n_uz = 16 or 32) into
// shared memory, run the three velocity sweeps of Eq. (4) on it, and write it back
// once: f is read and written once per kick instead of once per sweep.
//
// Rows (u_z lines) are stored with the TMA 32/64/128-byte swizzle, so the three access
// patterns are free of bank conflicts.  One producer thread drives the TMA engine (loads
// with transaction-count mbarriers, bulk stores); every wait is bounded.  The lines are
// marched by the same SL-MPP5 code (March) as the separate sweeps, so the result equals
// D_uz D_uy D_ux run as separate kernels, bit for bit.  FP32 storage: kick_pairs_kernel, two
// lines per thread.  16-bit storage: kick_cube_kernel, one line per thread in registers.
//
// 16-bit storage.  Shared memory holds three half-cube buffers (NU / 2 planes of constant
// j_x each) that rotate: while a cube sits in two of them, the third receives the first half
// of the next cube, and once the first half of the current cube has been swept and stored,
// its buffer receives the second half of the next cube.  Half-cube number j (two per cube,
// in the order the CTA takes its cubes) always lives in buffer j % 3.
//   D_ux: thread = line (j_y, j_z), walks j_x across both halves (one value per
//         row, lanes on consecutive j_z: one row segment per warp access);
//   D_uy: a warp owns whole planes of a half; lane = column j_z, walks j_y;
//   D_uz: the same warp, lane = row j_y, reads its row in 16-byte chunks.
// The rounding points are those of the separate path: D_ux encodes its result with the line
// scales it decoded with (one stochastic draw per value, the stream of the u_x register-line
// kernel), D_uy writes FP32 into a per-warp plane buffer, D_uz takes its rows from there,
// refreshes each row scale to the row's largest value and encodes with the stream of the u_z
// kernel.
#include "vk_lines.cuh"

namespace vk {

namespace {

template <int NU, typename T> struct Cube {
    static constexpr int es = int(sizeof(T));
    static constexpr bool coded = sizeof(T) == 2;
    static constexpr int rowbytes = NU * es;
    static constexpr int chunks = rowbytes / 16;
    static constexpr int per = 16 / es;
    static constexpr int half_rows = NU * NU / 2; // u_z lines of half a cube
    static constexpr unsigned half_bytes = unsigned(half_rows) * rowbytes;
    static constexpr int box_rows = half_rows < 256 ? half_rows : 256;
    static constexpr int boxes = half_rows / box_rows;
    static constexpr unsigned scale_bytes = coded ? unsigned(half_rows) * 4u : 0u;
    static constexpr int threads = NU * NU / 2; // consumer threads
    static constexpr int warps = threads / 32;
    static constexpr int planes_per_warp = 32 / NU; // of each half
    static constexpr int pitch = NU + 1;            // FP32 plane buffer: floats per row
    static constexpr int plane_floats = NU * pitch; // NU = 16: the two planes of a warp fall on complementary banks
    static constexpr unsigned plane_bytes = coded ? unsigned(warps * planes_per_warp * plane_floats) * 4u : 0u;
    // 16-bit: per warp, the inverse scales of the rows its D_ux lines cross (32)
    static constexpr unsigned inv_bytes = coded ? unsigned(warps) * 32u * 4u : 0u;
    static constexpr size_t smem = 128 + 1024 + 3 * size_t(half_bytes) + 3 * size_t(scale_bytes) + plane_bytes + inv_bytes;
    // swizzled byte offset of 16-byte chunk j of row r / of element c of row r
    __device__ static int off(int r, int j) { return r * rowbytes + 16 * (j ^ ((r * rowbytes >> 7) & (chunks - 1))); }
    __device__ static int eoff(int r, int c) { return off(r, c / per) + (c % per) * es; }
};

// D_ux on line (jy, jz) of the cube in halves h[0], h[1] (scales s[0], s[1]); e0 =
// index of the line's first element in f (16-bit stochastic-rounding stream).
// Returns true when the line sum is negative, NaN or infinite.
template <int NU, typename T, bool NEG>
__device__ __forceinline__ bool cube_ux(unsigned char *const (&h)[2], const float *const (&s)[2], const float *inv_jx,
                                        int jy, int jz, const Lim<float> &lim, unsigned long long e0, unsigned seed)
{
    using G = Cube<NU, T>;
    constexpr int HP = NU / 2; // planes per half
    float v[NU];
#pragma unroll
    for (int jx = 0; jx < NU; ++jx) {
        const int r = (jx % HP) * NU + jy;
        const T c = *reinterpret_cast<const T *>(h[jx / HP] + G::eoff(r, jz));
        v[NEG ? NU - 1 - jx : jx] = RegCodec<T>::get(c, s[jx / HP][r]);
    }
    const float sum = march_regs<NU, float>(v, lim);
    unsigned rng = sr_bits(e0, seed);
#pragma unroll
    for (int jx = 0; jx < NU; ++jx) { // u_x keeps the scales
        const int r = (jx % HP) * NU + jy;
        *reinterpret_cast<T *>(h[jx / HP] + G::eoff(r, jz)) =
            RegCodec<T>::put(v[NEG ? NU - 1 - jx : jx], inv_jx[jx], lcg_next(rng) >> 16);
    }
    return !(sum >= 0.f) || isinf(sum);
}

// D_uy on column jz of plane jxl (within half buffer hb, scales sb), decoded into the FP32
// plane buffer pl (row pitch Cube::pitch).
template <int NU, typename T, bool NEG>
__device__ __forceinline__ bool cube_uy(unsigned char *hb, const float *sb, float *pl, int jxl, int jz,
                                        const Lim<float> &lim)
{
    using G = Cube<NU, T>;
    float v[NU];
#pragma unroll
    for (int jy = 0; jy < NU; ++jy) {
        const int r = jxl * NU + jy;
        const T c = *reinterpret_cast<const T *>(hb + G::eoff(r, jz));
        v[NEG ? NU - 1 - jy : jy] = RegCodec<T>::get(c, sb[r]);
    }
    const float sum = march_regs<NU, float>(v, lim);
#pragma unroll
    for (int jy = 0; jy < NU; ++jy) pl[jy * G::pitch + jz] = v[NEG ? NU - 1 - jy : jy];
    return !(sum >= 0.f) || isinf(sum);
}

// D_uz on row jy of plane jxl, from the FP32 plane buffer; the row's scale is then refreshed
// and the row encoded.
template <int NU, typename T, bool NEG>
__device__ __forceinline__ bool cube_uz(unsigned char *hb, float *sb, const float *pl, int jxl, int jy,
                                        const Lim<float> &lim, unsigned long long e0, unsigned seed)
{
    using G = Cube<NU, T>;
    const int r = jxl * NU + jy;
    float v[NU];
#pragma unroll
    for (int jz = 0; jz < NU; ++jz) v[NEG ? NU - 1 - jz : jz] = pl[jy * G::pitch + jz];
    const float sum = march_regs<NU, float>(v, lim);
    float m = 0.f;
#pragma unroll
    for (int l = 0; l < NU; ++l) m = fmaxf(m, v[l]);
    m = coded_scale<T>(m);
    sb[r] = m;
    const float inv = inv_scale(m);
    unsigned rng = sr_bits(e0, seed);
#pragma unroll
    for (int j = 0; j < G::chunks; ++j) {
        float a[G::per];
#pragma unroll
        for (int q = 0; q < G::per; ++q) a[q] = v[NEG ? NU - 1 - (G::per * j + q) : G::per * j + q];
        Chunk<T>::put(hb + G::off(r, j), inv, a, rng);
    }
    return !(sum >= 0.f) || isinf(sum);
}

template <int NU, typename T>
__global__ void __launch_bounds__(Cube<NU, T>::threads + kProducer, NU == 32 ? 1 : 4)
    kick_cube_kernel(const __grid_constant__ CUtensorMap fmap, const __grid_constant__ CUtensorMap smap,
                     const __grid_constant__ KickArgs a)
{
    using G = Cube<NU, T>;
    constexpr int NT = G::threads;
    constexpr unsigned tx_bytes = G::half_bytes + G::scale_bytes;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem); // 3: a half-cube buffer holds its data
    uint64_t *done = full + 3;                           // 3: the consumers are done with a half
    uint64_t *uxd = done + 3;                            // D_ux of the current cube is complete
    unsigned char *bufs = smem + 128 + ((1024u - ((smem_u32(smem) + 128u) & 1023u)) & 1023u);
    auto hbuf = [&](unsigned j) { return bufs + size_t(G::half_bytes) * (j % 3); };
    auto sbuf = [&](unsigned j) {
        return reinterpret_cast<float *>(bufs + 3 * size_t(G::half_bytes) + size_t(G::scale_bytes) * (j % 3));
    };
    float *planes = reinterpret_cast<float *>(bufs + 3 * size_t(G::half_bytes) + 3 * size_t(G::scale_bytes));
    float *invs = reinterpret_cast<float *>(bufs + 3 * size_t(G::half_bytes) + 3 * size_t(G::scale_bytes) +
                                            G::plane_bytes); // 16-bit: 32 per warp

    if (threadIdx.x == 0) {
        for (int q = 0; q < 3; ++q) {
            mbar_init(&full[q], 1);
            mbar_init(&done[q], NT);
        }
        mbar_init(uxd, NT);
        fence_barrier_init();
    }
    __syncthreads();

    const long long Gd = gridDim.x, b = blockIdx.x;
    const unsigned n_my = unsigned(a.ncells > b ? (a.ncells - b + Gd - 1) / Gd : 0);
    const unsigned halves = 2 * n_my;
    auto first_row = [&](unsigned j) {
        const long long cube = a.cell0 + b + (long long)(j / 2) * Gd;
        return cube * (NU * NU) + (j % 2) * G::half_rows;
    };

    if (threadIdx.x >= NT) {
        // producer: one thread drives the TMA engine
        if (threadIdx.x != NT) return;
        auto load = [&](unsigned j) {
            uint64_t *bar = &full[j % 3];
            mbar_arrive_expect_tx(bar, tx_bytes);
            const long long r0 = first_row(j);
            for (int q = 0; q < G::boxes; ++q)
                tma_load_2d(hbuf(j) + q * G::box_rows * G::rowbytes, &fmap, bar, 0, int(r0 + q * G::box_rows));
            tma_load_2d(sbuf(j), &smap, bar, 0, int(r0 / NU));
        };
        unsigned loaded = 0;
        for (; loaded < 3 && loaded < halves; ++loaded) load(loaded);
        bool ok = true;
        for (unsigned j = 0; j < halves; ++j) {
            if (!mbar_wait_bounded(&done[j % 3], (j / 3) & 1u)) {
                ok = false;
                break;
            }
            const long long r0 = first_row(j);
            for (int q = 0; q < G::boxes; ++q)
                tma_store_2d(&fmap, hbuf(j) + q * G::box_rows * G::rowbytes, 0, int(r0 + q * G::box_rows));
            tma_store_2d(&smap, sbuf(j), 0, int(r0 / NU));
            bulk_commit();
            if (loaded < halves) {
                bulk_wait_read_all(); // the buffer of half j is free once the store has read it
                load(loaded++);
            }
        }
        bulk_wait_all();
        if (!ok) {
            atomicOr(a.err, ERR_TIMEOUT);
            // let the loads in flight (the last three at most) land before the CTA exits
            for (unsigned j = loaded > 3 ? loaded - 3 : 0; j < loaded; ++j) mbar_wait_bounded(&full[j % 3], (j / 3) & 1u);
        }
        return;
    }

    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    float *pl = planes + (w * G::planes_per_warp + lane / NU) * G::plane_floats; // 16-bit: this lane's plane
    bool bad = false;
    for (unsigned k = 0; k < n_my; ++k) {
        const unsigned j0 = 2 * k, j1 = 2 * k + 1;
        const bool got = mbar_wait_bounded(&full[j0 % 3], (j0 / 3) & 1u) && mbar_wait_bounded(&full[j1 % 3], (j1 / 3) & 1u);
        if (!__all_sync(0xffffffffu, got)) {
            atomicOr(a.err, ERR_TIMEOUT);
            return;
        }
        const long long cube = a.cell0 + b + (long long)k * Gd;
        unsigned char *const h[2] = {hbuf(j0), hbuf(j1)};
        float *const s[2] = {sbuf(j0), sbuf(j1)};
        const unsigned long long e_cube = (unsigned long long)cube * (NU * NU * NU);
        // one Courant number per cell and axis: every branch below is CTA-uniform
        const LineCoefT<float> kx = a.coef_x[cube];
        if (kx.nd >= 0) {
            const Lim<float> lim = to_lim(kx);
            const float *const sc[2] = {s[0], s[1]};
#pragma unroll 1
            for (int q = 0; q < 2; ++q) {
                const int line = q * NT + t, jy = line / NU, jz = line % NU;
                const unsigned long long e0 = e_cube + (unsigned long long)line;
                // 16-bit: the warp's lines cross NU rows per j_y (32 / NU values of j_y): each
                // lane forms the inverse scale of one of them once, for the whole warp
                float *wi = invs + w * 32;
                __syncwarp();
                const int jy_l = (q * NT + w * 32) / NU + lane / NU, jx = lane % NU;
                wi[lane] = inv_scale(sc[jx / (NU / 2)][(jx % (NU / 2)) * NU + jy_l]);
                __syncwarp();
                const float *inv_jx = wi + (lane / NU) * NU;
                bad |= (kx.nd & 1) ? cube_ux<NU, T, true>(h, sc, inv_jx, jy, jz, lim, e0, a.seed_x)
                                   : cube_ux<NU, T, false>(h, sc, inv_jx, jy, jz, lim, e0, a.seed_x);
            }
        }
        // every D_ux line crosses every plane: all of them finish before D_uy
        mbar_arrive(uxd);
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(uxd, k & 1u))) {
            atomicOr(a.err, ERR_TIMEOUT);
            return;
        }
        const LineCoefT<float> ky = a.coef_y[cube], kz = a.coef_z[cube];
        const int jxl = w * G::planes_per_warp + lane / NU, c = lane % NU;
#pragma unroll 1
        for (int hh = 0; hh < 2; ++hh) {
            unsigned char *const hb = hh ? h[1] : h[0]; // selects, not a dynamically indexed array
            float *const sb = hh ? s[1] : s[0];
            if (ky.nd >= 0) {
                const Lim<float> lim = to_lim(ky);
                bad |= (ky.nd & 1) ? cube_uy<NU, T, true>(hb, sb, pl, jxl, c, lim)
                                   : cube_uy<NU, T, false>(hb, sb, pl, jxl, c, lim);
            } else {
                // no D_uy: the plane buffer takes the decoded values as they are
#pragma unroll 4
                for (int jy = 0; jy < NU; ++jy) {
                    const int r = jxl * NU + jy;
                    pl[jy * G::pitch + c] = RegCodec<T>::get(*reinterpret_cast<const T *>(hb + G::eoff(r, c)), sb[r]);
                }
            }
            __syncwarp();
            const unsigned long long e0 = e_cube + (unsigned long long)((hh * (NU / 2) + jxl) * NU + c) * NU;
            if (kz.nd >= 0) {
                const Lim<float> lim = to_lim(kz);
                bad |= (kz.nd & 1) ? cube_uz<NU, T, true>(hb, sb, pl, jxl, c, lim, e0, a.seed_z)
                                   : cube_uz<NU, T, false>(hb, sb, pl, jxl, c, lim, e0, a.seed_z);
            } else if (ky.nd >= 0) {
                // D_uy changed the plane but D_uz does not run: encode it with the row's scale
                // refreshed as the u_z sweep would not; keep the stored scale, round to nearest
                const int r = jxl * NU + c;
                const float inv = inv_scale(sb[r]);
#pragma unroll 4
                for (int jz = 0; jz < NU; ++jz)
                    *reinterpret_cast<T *>(hb + G::eoff(r, jz)) = from_c<T>(pl[c * G::pitch + jz] * inv);
            }
            __syncwarp();
            fence_proxy_async();
            mbar_arrive(&done[(2 * k + hh) % 3]);
        }
    }
    if (bad) atomicOr(a.err, ERR_NAN);
}

// ----------------------------------------------------------------------------
// FP32 storage: two lines per thread as packed pairs, lines walked in shared memory
// ----------------------------------------------------------------------------
// 32^3 x 32^3 cells, per kick: 3.83 ms with one line per thread in registers, 3.42 with the
// flux in differences, 3.05 here (76 cycles per face pair and scheduler: 49 instructions, the
// ALU pipe 60 % and issue 65 % busy; the DRAM traffic alone would take 1.27 ms).  Read from
// global memory by every thread when they were needed, the coefficients cost 8 % of that;
// cells read no further ahead than the window, 3 %.
// The kick is bound by instruction issue and by the ALU pipe (min / max at half rate), not
// by DRAM.  A thread marches two lines at once, their sums and products as f32x2 (one issue
// slot for two), through a window of a few cells (vk_common.cuh, March), reading each cell
// once and writing it back in place, so that 512 threads cover all 1024 lines of a 32^3
// cube in one go at about 100 registers: 16 warps per SM keep both pipes busy.  (Whole pairs
// of lines in registers left 8 warps per SM and were slower than one line per thread.)
//
// Pieces.  A cube is four pieces of NU / 4 planes of constant j_x; a ring of seven pieces
// holds the current cube and three pieces of the next.  D_ux walks the planes in the order
// of its flow and waits for each piece as it comes to it, so the fourth piece of a cube,
// which can only be loaded once a piece of the previous cube has been stored, arrives while
// the first three are marched.  Piece j (four per cube, in march order) lives in slot j % 7.
//   D_ux: thread = columns (j_y, j_z), (j_y, j_z + 1), one 8-byte access per row;
//   D_uy: a warp owns 64 / NU planes; thread = two adjacent columns of one, walks j_y;
//   D_uz: the same warp; thread = rows j_y and j_y + NU / 2 of a plane, in 16-byte chunks
//         (cells of the two rows do not sit in register pairs: SPLIT).
// All accesses are free of bank conflicts under the TMA swizzle (NU = 16: D_uy two-way).
template <int NU> struct PairCube {
    using G = Cube<NU, float>;
    static constexpr int planes = NU / 4;                       // of a piece
    static constexpr int rows = planes * NU;                    // u_z lines of a piece
    static constexpr unsigned bytes = unsigned(rows) * G::rowbytes;
    static constexpr int slots = 7;
    static constexpr int threads = NU * NU / 2; // one per pair of lines
    static constexpr int warps = threads / 32;
    static constexpr int wplanes = 64 / NU;     // planes a warp owns
    static constexpr int per_piece = threads / 4; // threads whose planes lie in one piece
    // barriers (128 B), the coefficients of three cubes (u_x, u_y, u_z), alignment, the ring
    static constexpr int head = 128 + ((9 * int(sizeof(LineCoefT<float>)) + 127) & ~127);
    static constexpr size_t smem = head + 1024 + size_t(slots) * bytes;
    static_assert(rows <= 256, "one TMA box per piece");
};

// D_ux on the columns at byte offset `off` of every plane.  slot(m): the piece in march
// order m (waits for it; false: the wait ran out).
template <int NU, bool NEG, typename Slot>
__device__ __forceinline__ bool pair_ux(Slot slot, int off, const Lim<float2> &lim, bool &ok)
{
    using P = PairCube<NU>;
    constexpr int NP = P::planes, ST = NU * P::G::rowbytes; // bytes of a plane
    auto cell = [&](unsigned char *p, int i) -> float2 & { // plane i of the piece in march order
        return *reinterpret_cast<float2 *>(p + (NEG ? NP - 1 - i : i) * ST);
    };
    unsigned char *cur = slot(0, ok) + off;
    if (!ok) return false;
    March<float2> m(lim);
    m.start_zero(cell(cur, 0), cell(cur, 1));
#pragma unroll
    for (int i = 2; i < NP; ++i) cell(cur, i - 2) = m.face(cell(cur, i));
#pragma unroll 1
    for (int q = 1; q < 4; ++q) {
        unsigned char *prev = cur;
        cur = slot(q, ok) + off;
        if (!ok) return false;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
            const float2 out = m.face(cell(cur, i));
            if (i < 2) cell(prev, NP - 2 + i) = out;
            else cell(cur, i - 2) = out;
        }
    }
    cell(cur, NP - 2) = m.face(make_float2(0.f, 0.f));
    cell(cur, NP - 1) = m.last();
    return !(m.sum.x >= 0.f) || !(m.sum.y >= 0.f) || isinf(m.sum.x) || isinf(m.sum.y);
}

// D_uy on the adjacent columns jz, jz + 1 (jz even) of the plane at pl
template <int NU, bool NEG>
__device__ __forceinline__ bool pair_uy(unsigned char *pl, int jz, const Lim<float2> &lim)
{
    using G = Cube<NU, float>;
    auto cell = [&](int i) -> float2 & { return *reinterpret_cast<float2 *>(pl + G::eoff(NEG ? NU - 1 - i : i, jz)); };
    March<float2> m(lim);
    m.start_zero(cell(0), cell(1));
    // Blocks of 8 faces (the swizzle repeats every 8 rows), whose look-ahead cells are all read
    // first: a read stays behind the writes before it (the compiler cannot tell the swizzled
    // addresses apart), and so must not wait for a face.
    constexpr int B = 8, R = (NU - 2) % B, ST = NEG ? -B * G::rowbytes : B * G::rowbytes;
#pragma unroll 1
    for (int b = 0; b < (NU - 2) / B; ++b, pl += ST) {
        float2 c[B];
#pragma unroll
        for (int q = 0; q < B; ++q) c[q] = cell(q + 2);
#pragma unroll
        for (int q = 0; q < B; ++q) cell(q) = m.face(c[q]);
    }
    float2 c[R];
#pragma unroll
    for (int q = 0; q < R; ++q) c[q] = cell(q + 2);
#pragma unroll
    for (int q = 0; q < R; ++q) cell(q) = m.face(c[q]);
    cell(R) = m.face(make_float2(0.f, 0.f));
    cell(R + 1) = m.last();
    return !(m.sum.x >= 0.f) || !(m.sum.y >= 0.f) || isinf(m.sum.x) || isinf(m.sum.y);
}

// D_uz on the rows jy and jy + NU / 2 of the plane at pl
template <int NU, bool NEG>
__device__ __forceinline__ bool pair_uz(unsigned char *pl, int jy, const Lim<float2> &lim)
{
    using G = Cube<NU, float>;
    constexpr int C = G::chunks;
    auto at = [&](int row, int j) -> float4 & {
        return *reinterpret_cast<float4 *>(pl + G::off(row, NEG ? C - 1 - j : j));
    };
    March<float2, true> m(lim);
    auto pick = [](const float4 &a, const float4 &b, int q) {
        const int s = NEG ? 3 - q : q;
        return make_float2((&a.x)[s], (&b.x)[s]);
    };
    auto set = [](float4 &a, float4 &b, int q, float2 v) {
        const int s = NEG ? 3 - q : q;
        (&a.x)[s] = v.x;
        (&b.x)[s] = v.y;
    };
    float4 a = at(jy, 0), b = at(jy + NU / 2, 0), oa, ob;
    float4 na = at(jy, 1), nb = at(jy + NU / 2, 1); // read one chunk ahead of their use
    m.start_zero(pick(a, b, 0), pick(a, b, 1));
    set(oa, ob, 0, m.face(pick(a, b, 2)));
    set(oa, ob, 1, m.face(pick(a, b, 3)));
    // (rolled: 32^3 cubes 2.5 % slower; unrolled: 16^3 cubes 9 % slower, four CTAs per SM share
    // the instruction cache)
#pragma unroll(NU == 32 ? C - 1 : 1)
    for (int j = 1; j < C; ++j) {
        a = na;
        b = nb;
        if (j + 1 < C) {
            na = at(jy, j + 1);
            nb = at(jy + NU / 2, j + 1);
        }
        set(oa, ob, 2, m.face(pick(a, b, 0)));
        set(oa, ob, 3, m.face(pick(a, b, 1)));
        at(jy, j - 1) = oa;
        at(jy + NU / 2, j - 1) = ob;
        set(oa, ob, 0, m.face(pick(a, b, 2)));
        set(oa, ob, 1, m.face(pick(a, b, 3)));
    }
    set(oa, ob, 2, m.face(make_float2(0.f, 0.f)));
    set(oa, ob, 3, m.last());
    at(jy, C - 1) = oa;
    at(jy + NU / 2, C - 1) = ob;
    return !(m.sum.x >= 0.f) || !(m.sum.y >= 0.f) || isinf(m.sum.x) || isinf(m.sum.y);
}

template <int NU>
__global__ void __launch_bounds__(PairCube<NU>::threads + kProducer, NU == 32 ? 1 : 4)
    kick_pairs_kernel(const __grid_constant__ CUtensorMap fmap, const __grid_constant__ KickArgs a)
{
    using P = PairCube<NU>;
    using G = Cube<NU, float>;
    constexpr int NT = P::threads, S = P::slots;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem); // S: the slot holds its piece
    uint64_t *done = full + S;                           // S: the warps that own its planes are done
    uint64_t *uxd = done + S;                            // D_ux of the current cube is complete
    static_assert((2 * S + 1) * 8 <= 128, "barriers fit ahead of the ring");
    LineCoefT<float> *coefs = reinterpret_cast<LineCoefT<float> *>(smem + 128);
    unsigned char *ring = smem + P::head + ((1024u - ((smem_u32(smem) + unsigned(P::head)) & 1023u)) & 1023u);
    auto slot = [&](unsigned j) { return ring + size_t(P::bytes) * (j % S); };

    if (threadIdx.x == 0) {
        for (int q = 0; q < S; ++q) {
            mbar_init(&full[q], 1);
            mbar_init(&done[q], P::per_piece);
        }
        mbar_init(uxd, NT);
        fence_barrier_init();
    }
    __syncthreads();

    const long long Gd = gridDim.x, b = blockIdx.x;
    const unsigned n_my = unsigned(a.ncells > b ? (a.ncells - b + Gd - 1) / Gd : 0);
    const unsigned pieces = 4 * n_my;

    if (threadIdx.x >= NT) {
        // producer: one thread drives the TMA engine
        if (threadIdx.x != NT) return;
        // the coefficients of the cube of piece j (the ring holds pieces of two cubes, and the
        // third slot keeps those of the cube before for warps still on it)
        auto coef = [&](unsigned j) { return coefs + 3 * ((j / 4) % 3); };
        auto first_row = [&](unsigned j) { // of piece j: the quarters of a cube in the order D_ux walks them
            const long long cube = a.cell0 + b + (long long)(j / 4) * Gd;
            const int nd = coef(j)->nd;
            const int q = nd >= 0 && (nd & 1) ? 3 - int(j % 4) : int(j % 4);
            return int(cube * (NU * NU) + q * P::rows);
        };
        auto load = [&](unsigned j) {
            if (j % 4 == 0) {
                // read here, ahead of the consumers, who would wait for them three times per cube;
                // they see them once they have waited for the piece
                const long long cube = a.cell0 + b + (long long)(j / 4) * Gd;
                const LineCoefT<float> cx = a.coef_x[cube], cy = a.coef_y[cube], cz = a.coef_z[cube];
                coef(j)[0] = cx;
                coef(j)[1] = cy;
                coef(j)[2] = cz;
            }
            uint64_t *bar = &full[j % S];
            mbar_arrive_expect_tx(bar, P::bytes);
            tma_load_2d(slot(j), &fmap, bar, 0, first_row(j));
        };
        unsigned loaded = 0;
        for (; loaded < unsigned(S) && loaded < pieces; ++loaded) load(loaded);
        bool ok = true;
        for (unsigned j = 0; j < pieces; ++j) {
            if (!mbar_wait_bounded(&done[j % S], (j / S) & 1u)) {
                ok = false;
                break;
            }
            tma_store_2d(&fmap, slot(j), 0, first_row(j));
            bulk_commit();
            if (loaded < pieces) {
                bulk_wait_read_all(); // the slot of piece j is free once the store has read it
                load(loaded++);
            }
        }
        bulk_wait_all();
        if (!ok) {
            atomicOr(a.err, ERR_TIMEOUT);
            // let the loads in flight (the last S at most) land before the CTA exits
            for (unsigned j = loaded > unsigned(S) ? loaded - S : 0; j < loaded; ++j)
                mbar_wait_bounded(&full[j % S], (j / S) & 1u);
        }
        return;
    }

    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    // D_ux: the thread's columns; D_uy, D_uz: its plane (within the warp's), column pair, row
    const int ux_off = G::eoff(t / (NU / 2), 2 * (t % (NU / 2)));
    const int wp = lane / (NU / 2), lp = lane % (NU / 2);
    const int quarter = w / (P::warps / 4); // of the cube: where the warp's planes lie
    const int pl_off = ((w % (P::warps / 4)) * P::wplanes + wp) * NU * G::rowbytes;
    bool bad = false, ok = true;
    for (unsigned k = 0; k < n_my; ++k) {
        auto piece = [&](int m, bool &good) { // piece m of the cube, once it is loaded
            const unsigned j = 4 * k + m;
            good = __all_sync(0xffffffffu, mbar_wait_bounded(&full[j % S], (j / S) & 1u));
            return slot(j);
        };
        piece(0, ok);
        if (!ok) {
            atomicOr(a.err, ERR_TIMEOUT);
            return;
        }
        // one Courant number per cell and axis: every branch below is CTA-uniform
        const LineCoefT<float> *co = coefs + 3 * (k % 3);
        const LineCoefT<float> kx = co[0];
        const bool xneg = kx.nd >= 0 && (kx.nd & 1);
        if (kx.nd >= 0) {
            const Lim<float2> lim = to_lim2(kx, kx);
            bad |= xneg ? pair_ux<NU, true>(piece, ux_off, lim, ok) : pair_ux<NU, false>(piece, ux_off, lim, ok);
        } else {
            for (int m = 1; m < 4 && ok; ++m) piece(m, ok);
        }
        if (!ok) {
            atomicOr(a.err, ERR_TIMEOUT);
            return;
        }
        // every D_ux line crosses every plane: all of them finish before D_uy
        mbar_arrive(uxd);
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(uxd, k & 1u))) {
            atomicOr(a.err, ERR_TIMEOUT);
            return;
        }
        const LineCoefT<float> ky = co[1], kz = co[2];
        const unsigned j = 4 * k + (xneg ? 3 - quarter : quarter);
        unsigned char *pl = slot(j) + pl_off;
        if (ky.nd >= 0) {
            const Lim<float2> lim = to_lim2(ky, ky);
            bad |= (ky.nd & 1) ? pair_uy<NU, true>(pl, 2 * lp, lim) : pair_uy<NU, false>(pl, 2 * lp, lim);
        }
        __syncwarp();
        if (kz.nd >= 0) {
            const Lim<float2> lim = to_lim2(kz, kz);
            bad |= (kz.nd & 1) ? pair_uz<NU, true>(pl, lp, lim) : pair_uz<NU, false>(pl, lp, lim);
        }
        __syncwarp();
        fence_proxy_async();
        mbar_arrive(&done[j % S]);
    }
    if (bad) atomicOr(a.err, ERR_NAN);
}

template <int NU, typename T> const void *kick_kernel() { return (const void *)kick_cube_kernel<NU, T>; }

const void *kick_kernel_for(int nu, int dtype)
{
    switch (dtype) {
    case 1: return nu == 32 ? (const void *)kick_pairs_kernel<32> : (const void *)kick_pairs_kernel<16>;
    case 2: return nu == 32 ? kick_kernel<32, __nv_bfloat16>() : kick_kernel<16, __nv_bfloat16>();
    case 3: return nu == 32 ? kick_kernel<32, __half>() : kick_kernel<16, __half>();
    default: return nullptr;
    }
}

template <int NU> size_t smem_for(int dtype)
{
    return dtype == 1 ? PairCube<NU>::smem : Cube<NU, __nv_bfloat16>::smem;
}

template <int NU> int threads_for() { return Cube<NU, float>::threads + kProducer; }

} // namespace

bool kick_cube_supported(int nux, int nuy, int nuz, int dtype)
{
    return nux == nuy && nuy == nuz && (nuz == 16 || nuz == 32) && dtype >= 1 && dtype <= 3;
}

int kick_cube_box_rows(int nu, int dtype)
{
    if (dtype == 1) return nu * nu / 4; // a piece
    return nu * nu / 2 < 256 ? nu * nu / 2 : 256;
}

size_t kick_cube_smem(int nu, int dtype) { return nu == 32 ? smem_for<32>(dtype) : smem_for<16>(dtype); }

int occupancy_kick_cube(int nu, int dtype)
{
    const void *k = kick_kernel_for(nu, dtype);
    if (!k) return 0;
    const size_t smem = kick_cube_smem(nu, dtype);
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem)) != cudaSuccess) return 0;
    int n = 0;
    const int threads = nu == 32 ? threads_for<32>() : threads_for<16>();
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, smem) != cudaSuccess) return 0;
    return n;
}

cudaError_t launch_kick_cube(const CUtensorMap &fmap, const CUtensorMap &smap, const KickArgs &a, int nu, int dtype,
                             int grid, cudaStream_t st)
{
    if (a.ncells <= 0 || grid <= 0) return cudaSuccess;
    const void *k = kick_kernel_for(nu, dtype);
    if (!k || !a.coef_x || !a.coef_y || !a.coef_z) return cudaErrorInvalidValue;
    // row coordinates of the tensor maps are 32-bit
    if ((a.cell0 + a.ncells) * (long long)nu * nu > 0x7fffffffll) return cudaErrorInvalidValue;
    const size_t smem = kick_cube_smem(nu, dtype);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
    if (e != cudaSuccess) return e;
    KickArgs args = a;
    void *params_f32[] = {const_cast<CUtensorMap *>(&fmap), &args};
    void *params_coded[] = {const_cast<CUtensorMap *>(&fmap), const_cast<CUtensorMap *>(&smap), &args};
    void **params = dtype == 1 ? params_f32 : params_coded;
    const int threads = nu == 32 ? threads_for<32>() : threads_for<16>();
    return cudaLaunchKernel(k, dim3(grid), dim3(threads), params, smem, st);
}

} // namespace vk
