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
// D_uz D_uy D_ux run as separate kernels, bit for bit (16-bit storage: the rounding points and
// random streams of the separate u_x kernel and the fused u_y u_z tail).
#include "vk_lines.cuh"

namespace vk {

namespace {

// a cube's rows (u_z lines) of T in shared memory
template <int NU, typename T> struct Cube {
    static constexpr int es = int(sizeof(T));
    static constexpr int rowbytes = NU * es;
    static constexpr int chunks = rowbytes / 16;
    static constexpr int per = 16 / es;
    // swizzled byte offset of 16-byte chunk j of row r / of element c of row r
    __device__ static int off(int r, int j) { return r * rowbytes + 16 * (j ^ ((r * rowbytes >> 7) & (chunks - 1))); }
    __device__ static int eoff(int r, int c) { return off(r, c / per) + (c % per) * es; }
};

// ----------------------------------------------------------------------------
// FP32 storage: two lines per thread as packed pairs, lines walked in shared memory
// ----------------------------------------------------------------------------
// 32^3 x 32^3 cells, per kick: 3.83 ms with one line per thread in registers, 3.42 with the
// flux in differences, 3.05 here (76 cycles per face pair and scheduler: 49 instructions, the
// ALU pipe 60 % and issue 65 % busy; the DRAM traffic alone would take 1.27 ms).  Read from
// global memory by every thread when they were needed, the coefficients cost 8 % of that;
// cells read no further ahead than the window, 3 %.
// The kick is bound by its marches, not by DRAM; min / max run at half rate on the ALU pipe.  A thread marches two lines at once, their sums and products as f32x2 (one issue
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
    chain_enter();

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

// ----------------------------------------------------------------------------
// 16-bit storage: the same marches on a cube decoded into FP32
// ----------------------------------------------------------------------------
// The pieces of a cube (codes and line scales) pass through a ring of four: D_ux decodes them
// as it walks, encodes each result with the line scale it keeps (one stochastic draw per
// value, the stream of the u_x register-line kernel) and writes what that code decodes to
// into a cube of FP32, on which D_uy and D_uz run as for FP32 storage.  So a piece is free
// as soon as D_ux is through, and the next cube loads while D_uy and D_uz run.  Each warp
// then takes its 64 rows into registers, refreshes their scales to the largest value,
// encodes them with the streams of the u_z kernel, densely into the front half of the same
// shared memory, and stores them itself; the FP32 cube may be written again once every
// warp's store has read its part (barrier `freed`).
// 32^3 x 32^3 BF16, per kick: 4.48 ms with one line per thread in registers (its unrolled
// bodies at the edge of the instruction cache), 3.91 here (61 instructions per face pair, issue 63 %
// busy); 32^3 x 16^3 FP16 0.82 -> 0.59 ms.
template <int NU, typename T> struct PairCube16 {
    using G = Cube<NU, T>;
    using F = Cube<NU, float>;
    static constexpr int planes = NU / 4;                  // of a piece
    static constexpr int rows = planes * NU;               // u_z lines of a piece
    static constexpr unsigned code_bytes = unsigned(rows) * G::rowbytes;
    static constexpr unsigned bytes = code_bytes + rows * 4u; // codes, then scales
    static constexpr int slots = 4;
    static constexpr int threads = NU * NU / 2; // one per pair of lines
    static constexpr int warps = threads / 32;
    static constexpr int wrows = 64;            // rows a warp owns for D_uy, D_uz (a TMA box)
    static constexpr int wplanes = wrows / NU;
    static constexpr int warp_js = 64 / NU;     // j_y of a warp's D_ux lines
    static constexpr size_t cube_bytes = size_t(NU) * NU * F::rowbytes;
    // barriers (128 B), the coefficients of three cubes, alignment, the FP32 cube, the ring, (scale,
    // inverse scale) of the rows each warp's D_ux lines cross
    static constexpr int head = 128 + ((9 * int(sizeof(LineCoefT<float>)) + 127) & ~127);
    static constexpr size_t smem = head + 1024 + cube_bytes + size_t(slots) * bytes + size_t(warps) * 64 * sizeof(float2);
};

// The rounding stream of a line draws for its cells in memory order (j_x = 0 first), as the
// u_x register-line kernel does; a line walked from its far end takes the same draws
// backward: the generator x -> a x + c run in reverse, from the state after NU + 1 steps.
template <bool NEG> __device__ __forceinline__ unsigned draw16(unsigned &x)
{
    constexpr Lcg step = NEG ? kLcgBack : kLcg;
    x = step(x);
    return x >> 16;
}
template <int NU, bool NEG> __device__ __forceinline__ unsigned draw_start(unsigned seed)
{
    constexpr Lcg end = lcg_power(kLcg, NU + 1);
    return NEG ? end(seed) : seed;
}

// value pair -> what the codes it is stochastically rounded to (bx, by: 16 random bits) decode to
__device__ __forceinline__ float2 recode(float2 v, float2 s, unsigned bx, unsigned by, __nv_bfloat16)
{
    const float2 c = vmul(v, make_float2(s.y, s.y));
    const unsigned x = (__float_as_uint(c.x) + bx) & 0xffff0000u;
    const unsigned y = (__float_as_uint(c.y) + by) & 0xffff0000u;
    return vmul(make_float2(__uint_as_float(x), __uint_as_float(y)), make_float2(s.x, s.x));
}
__device__ __forceinline__ float2 recode(float2 v, float2 s, unsigned bx, unsigned by, __half)
{
    const float2 c = vmul(v, make_float2(s.y, s.y));
    const __half x = RegCodec<__half>::put(c.x, 1.f, bx), y = RegCodec<__half>::put(c.y, 1.f, by);
    return vmul(make_float2(__half2float(x), __half2float(y)), make_float2(s.x, s.x));
}
__device__ __forceinline__ float2 decode2(unsigned u, float s, __nv_bfloat16)
{
    return vmul(make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u)), make_float2(s, s));
}
__device__ __forceinline__ float2 decode2(unsigned u, float s, __half)
{
    return vmul(__half22float2(*reinterpret_cast<const __half2 *>(&u)), make_float2(s, s));
}

// D_ux on one pair of columns: piece(q) is the piece in march order (waits for it and leaves
// its scales in ws; false: a wait ran out); codes at byte `co` of every plane of it, the FP32
// cube's cells at fp + plane FST (plane 0 .. NU - 1 of the cube); ws[n js + jl]: (scale, inverse)
// of the n-th plane in march order.  writable(): the FP32 cube may be written.
template <int NU, typename T, bool NEG, typename Piece, typename Writable>
__device__ __forceinline__ bool pair16_ux(Piece piece, Writable writable, int co, unsigned char *fp, const float2 *ws, int jl,
                                          const Lim<float2> &lim, unsigned rx, unsigned ry, bool &ok)
{
    using P = PairCube16<NU, T>;
    constexpr int NP = P::planes, CST = NU * P::G::rowbytes, FST = NU * P::F::rowbytes, JS = P::warp_js;
    auto code = [&](const unsigned char *p, int i) { // plane i of the piece in march order
        return *reinterpret_cast<const unsigned *>(p + (NEG ? NP - 1 - i : i) * CST);
    };
    // cell n of the line in march order: its scales, and where its value goes
    if (NEG) fp += (NU - 1) * FST;
    const float2 *s = ws + jl;
    auto out = [&](int n, float2 v) {
        *reinterpret_cast<float2 *>(fp + (NEG ? -n : n) * FST) =
            recode(v, s[n * JS], draw16<NEG>(rx), draw16<NEG>(ry), T());
    };
    rx = draw_start<NU, NEG>(rx);
    ry = draw_start<NU, NEG>(ry);
    const unsigned char *cur = piece(0, ok) + co;
    if (!ok || !(ok = writable())) return false;
    March<float2> m(lim);
    m.start_zero(decode2(code(cur, 0), s[0].x, T()), decode2(code(cur, 1), s[JS].x, T()));
#pragma unroll
    for (int i = 2; i < NP; ++i) out(i - 2, m.face(decode2(code(cur, i), s[i * JS].x, T())));
#pragma unroll 1
    for (int q = 1; q < 4; ++q) {
        cur = piece(q, ok) + co;
        if (!ok) return false;
        fp += (NEG ? -NP : NP) * FST;
        s += NP * JS;
#pragma unroll
        for (int i = 0; i < NP; ++i) out(i - 2, m.face(decode2(code(cur, i), s[i * JS].x, T())));
    }
    out(NP - 2, m.face(make_float2(0.f, 0.f)));
    out(NP - 1, m.last());
    return !(m.sum.x >= 0.f) || !(m.sum.y >= 0.f) || isinf(m.sum.x) || isinf(m.sum.y);
}

template <int NU, typename T>
__global__ void __launch_bounds__(PairCube16<NU, T>::threads + kProducer, NU == 32 ? 1 : 4)
    kick_pairs16_kernel(const __grid_constant__ CUtensorMap fmap, const __grid_constant__ CUtensorMap smap,
                        const __grid_constant__ KickArgs a)
{
    using P = PairCube16<NU, T>;
    using G = typename P::G;
    using F = typename P::F;
    constexpr int NT = P::threads, S = P::slots, NP = P::planes, JS = P::warp_js;
    extern __shared__ __align__(128) unsigned char smem[];
    uint64_t *full = reinterpret_cast<uint64_t *>(smem); // S: the slot holds its piece
    uint64_t *uxd = full + S;                            // D_ux of the current cube is complete
    uint64_t *freed = uxd + 1;                           // every warp's part of the FP32 cube is stored
    LineCoefT<float> *coefs = reinterpret_cast<LineCoefT<float> *>(smem + 128);
    unsigned char *cubef = smem + P::head + ((1024u - ((smem_u32(smem) + unsigned(P::head)) & 1023u)) & 1023u);
    unsigned char *ring = cubef + P::cube_bytes;
    float2 *scales = reinterpret_cast<float2 *>(ring + size_t(S) * P::bytes);
    auto slot = [&](unsigned j) { return ring + size_t(P::bytes) * (j % S); };

    if (threadIdx.x == 0) {
        for (int q = 0; q < S; ++q) mbar_init(&full[q], 1);
        mbar_init(uxd, NT);
        mbar_init(freed, P::warps);
        fence_barrier_init();
    }
    __syncthreads();
    chain_enter();

    const long long Gd = gridDim.x, b = blockIdx.x;
    const unsigned n_my = unsigned(a.ncells > b ? (a.ncells - b + Gd - 1) / Gd : 0);

    if (threadIdx.x >= NT) {
        // producer: one thread loads the pieces of cube k + 1 once D_ux of cube k is complete
        if (threadIdx.x != NT) return;
        unsigned k = 0;
        bool ok = true;
        for (; k < n_my; ++k) {
            if (k > 0 && !mbar_wait_bounded(uxd, (k - 1) & 1u)) {
                ok = false;
                break;
            }
            const long long cube = a.cell0 + b + (long long)k * Gd;
            // (three sets: warps still on cube k - 1 read theirs, and none can be on k - 2)
            LineCoefT<float> *co = coefs + 3 * (k % 3);
            const LineCoefT<float> cx = a.coef_x[cube], cy = a.coef_y[cube], cz = a.coef_z[cube];
            co[0] = cx;
            co[1] = cy;
            co[2] = cz;
            const bool neg = cx.nd >= 0 && (cx.nd & 1);
            fence_proxy_async(); // the consumers' reads of the slots come before the loads
            for (int m = 0; m < 4; ++m) {
                const int q = neg ? 3 - m : m;
                uint64_t *bar = &full[m];
                unsigned char *dst = slot(m);
                mbar_arrive_expect_tx(bar, P::bytes);
                for (int x = 0; x < P::rows / P::wrows; ++x) {
                    const int plane = int(cube * NU) + q * NP + x * P::wplanes;
                    tma_load_2d(dst + x * P::wrows * G::rowbytes, &fmap, bar, 0, plane * NU);
                    tma_load_2d(dst + P::code_bytes + x * P::wrows * 4, &smap, bar, 0, plane);
                }
            }
        }
        if (!ok) {
            atomicOr(a.err, ERR_TIMEOUT);
            if (k > 0) // let the loads in flight land before the CTA exits
                for (int m = 0; m < 4; ++m) mbar_wait_bounded(&full[m], (k - 1) & 1u);
        }
        return;
    }

    const int t = threadIdx.x, w = t >> 5, lane = t & 31;
    // D_ux: the thread's columns; D_uy, D_uz: its plane (within the warp's), column pair, row
    const int ujy = t / (NU / 2), ujz = 2 * (t % (NU / 2));
    const int co_off = G::eoff(ujy, ujz);
    float2 *ws = scales + w * 64;
    const int wp = lane / (NU / 2), lp = lane % (NU / 2);
    unsigned char *mine = cubef + size_t(w) * P::wrows * F::rowbytes; // the warp's rows
    unsigned char *pl = mine + wp * NU * F::rowbytes;
    bool bad = false, ok = true;
    for (unsigned k = 0; k < n_my; ++k) {
        const long long cube = a.cell0 + b + (long long)k * Gd;
        const unsigned long long e_cube = (unsigned long long)cube * (NU * NU * NU);
        const LineCoefT<float> *co = coefs + 3 * (k % 3);
        bool xneg = false;
        auto piece = [&](int m, bool &good) -> unsigned char * { // piece m in march order, its scales into ws
            good = __all_sync(0xffffffffu, mbar_wait_bounded(&full[m], k & 1u));
            if (!good) return nullptr;
            if (m == 0) xneg = co[0].nd >= 0 && (co[0].nd & 1);
            if (lane < NP * JS) {
                const int i = lane / JS, jl = lane % JS;
                const float s = reinterpret_cast<const float *>(slot(m) + P::code_bytes)[(xneg ? NP - 1 - i : i) * NU + w * JS + jl];
                ws[(m * NP + i) * JS + jl] = make_float2(s, inv_scale(s));
            }
            __syncwarp();
            return slot(m);
        };
        auto writable = [&]() { return k == 0 || __all_sync(0xffffffffu, mbar_wait_bounded(freed, (k - 1) & 1u)); };
        unsigned char *first = piece(0, ok);
        if (ok) {
            // one Courant number per cell and axis: every branch below is CTA-uniform
            const LineCoefT<float> kx = co[0];
            auto again = [&](int m, bool &good) { // piece 0 is here
                good = true;
                return m == 0 ? first : piece(m, good);
            };
            if (kx.nd >= 0) {
                const Lim<float2> lim = to_lim2(kx, kx);
                const unsigned long long e0 = e_cube + (unsigned long long)(ujy * NU + ujz);
                const unsigned rx = sr_bits(e0, a.seed_x), ry = sr_bits(e0 + 1, a.seed_x);
                unsigned char *fp = cubef + F::eoff(ujy, ujz);
                bad |= xneg ? pair16_ux<NU, T, true>(again, writable, co_off, fp, ws, ujy % JS, lim, rx, ry, ok)
                            : pair16_ux<NU, T, false>(again, writable, co_off, fp, ws, ujy % JS, lim, rx, ry, ok);
            } else if ((ok = writable())) {
                // no D_ux: the FP32 cube takes the decoded values as they are
                for (int m = 0; m < 4 && ok; ++m) {
                    const unsigned char *p = again(m, ok);
                    if (!ok) break;
#pragma unroll 1
                    for (int i = 0; i < NP; ++i)
                        *reinterpret_cast<float2 *>(cubef + F::eoff((m * NP + i) * NU + ujy, ujz)) =
                            decode2(*reinterpret_cast<const unsigned *>(p + i * NU * G::rowbytes + co_off),
                                    ws[(m * NP + i) * JS + ujy % JS].x, T());
                }
            }
        }
        if (!ok) {
            atomicOr(a.err, ERR_TIMEOUT);
            break;
        }
        // every D_ux line crosses every plane: all of them finish before D_uy; the pieces are read
        mbar_arrive(uxd);
        if (!__all_sync(0xffffffffu, mbar_wait_bounded(uxd, k & 1u))) {
            atomicOr(a.err, ERR_TIMEOUT);
            break;
        }
        const bool ran_x = co[0].nd >= 0;
        const LineCoefT<float> ky = co[1], kz = co[2];
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
        if (ran_x || ky.nd >= 0 || kz.nd >= 0) { // (else every code stays as it is)
            // rows lane and lane + 32 of the warp's 64, into registers, then encoded over them
            float v[2][NU];
#pragma unroll
            for (int h = 0; h < 2; ++h)
#pragma unroll
                for (int j = 0; j < F::chunks; ++j) {
                    const float4 x = *reinterpret_cast<const float4 *>(mine + F::off(lane + 32 * h, j));
                    v[h][4 * j] = x.x; v[h][4 * j + 1] = x.y; v[h][4 * j + 2] = x.z; v[h][4 * j + 3] = x.w;
                }
            __syncwarp();
            float *sdst = reinterpret_cast<float *>(mine + P::wrows * G::rowbytes);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int r = lane + 32 * h;
                const long long row = cube * (NU * NU) + w * P::wrows + r;
                if (kz.nd >= 0) {
                    float s = 0.f;
#pragma unroll
                    for (int l = 0; l < NU; l += 2) s = mx3(s, v[h][l], v[h][l + 1]);
                    s = coded_scale<T>(s);
                    sdst[r] = s;
                    const float inv = inv_scale(s);
                    unsigned rng = sr_bits((unsigned long long)row * NU, a.seed_z);
#pragma unroll
                    for (int j = 0; j < G::chunks; ++j) {
                        float e[8];
#pragma unroll
                        for (int q = 0; q < 8; ++q) e[q] = v[h][8 * j + q];
                        Chunk<T>::put(mine + G::off(r, j), inv, e, rng);
                    }
                } else {
                    // D_uz did not run: its rows keep their scales and round to nearest (codes
                    // that D_ux left come back as they were)
                    const float s = a.scale[row], inv = inv_scale(s);
                    sdst[r] = s;
#pragma unroll
                    for (int l = 0; l < NU; ++l) *reinterpret_cast<T *>(mine + G::eoff(r, l)) = from_c<T>(v[h][l] * inv);
                }
            }
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) {
                const int plane = int(cube * NU) + w * P::wplanes;
                tma_store_2d(&fmap, mine, 0, plane * NU);
                tma_store_2d(&smap, sdst, 0, plane);
                bulk_commit();
                bulk_wait_read_all();
            }
            __syncwarp();
        }
        if (lane == 0) mbar_arrive(freed);
    }
    if (lane == 0) bulk_wait_all();
    if (bad) atomicOr(a.err, ERR_NAN);
}

const void *kick_kernel_for(int nu, int dtype)
{
    switch (dtype) {
    case 1: return nu == 32 ? (const void *)kick_pairs_kernel<32> : (const void *)kick_pairs_kernel<16>;
    case 2: return nu == 32 ? (const void *)kick_pairs16_kernel<32, __nv_bfloat16> : (const void *)kick_pairs16_kernel<16, __nv_bfloat16>;
    case 3: return nu == 32 ? (const void *)kick_pairs16_kernel<32, __half> : (const void *)kick_pairs16_kernel<16, __half>;
    default: return nullptr;
    }
}

template <int NU> size_t smem_for(int dtype) { return dtype == 1 ? PairCube<NU>::smem : PairCube16<NU, __nv_bfloat16>::smem; }

template <int NU> int threads_for() { return PairCube<NU>::threads + kProducer; }

} // namespace

bool kick_cube_supported(int nux, int nuy, int nuz, int dtype)
{
    return nux == nuy && nuy == nuz && (nuz == 16 || nuz == 32) && dtype >= 1 && dtype <= 3;
}

int kick_cube_box_rows(int nu, int dtype) { return dtype == 1 ? nu * nu / 4 : 64; } // FP32: a piece; 16-bit: a warp's rows

size_t kick_cube_smem(int nu, int dtype) { return nu == 32 ? smem_for<32>(dtype) : smem_for<16>(dtype); }

int occupancy_kick_cube(int nu, int dtype)
{
    const void *k = kick_kernel_for(nu, dtype);
    if (!k) return 0;
    const size_t smem = kick_cube_smem(nu, dtype);
    if (allow_smem(k, smem) != cudaSuccess) return 0;
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
    cudaError_t e = allow_smem(k, smem);
    if (e != cudaSuccess) return e;
    KickArgs args = a;
    void *params_f32[] = {const_cast<CUtensorMap *>(&fmap), &args};
    void *params_coded[] = {const_cast<CUtensorMap *>(&fmap), const_cast<CUtensorMap *>(&smap), &args};
    void **params = dtype == 1 ? params_f32 : params_coded;
    const int threads = nu == 32 ? threads_for<32>() : threads_for<16>();
    return launch_chained(a.ncells * nu * nu * nu, k, dim3(grid), dim3(threads), smem, st, params);
}

} // namespace vk
