// adjoint_tile.cu -- reverse mode of the position sweeps (the transpose of D_x, D_y, D_z, Eq. 3,
// at frozen limiter branches) on FP32 storage: whole lines of the sweep's input f and of lambda
// staged in shared memory, one line per thread.
//
// f and lambda are viewed as [O][L][I] and I cut into tiles of COLS contiguous columns (the last
// one of a row partial: TMA fills and clips it); a ring slot holds a tile of f and under it the
// tile of lambda, two TMA boxes {COLS, L}.  Groups of COLS threads march different slots, one
// producer thread keeps the ring full.  A cell of f that no later face reads gives its place to
// the new lambda, which leaves from there; lambda's own rows are only read, so a line whose
// Courant number exceeds 1 (lambda read that many cells on) needs no second array.
//
// The march is written in differences, as the forward flux is (vk_common.cuh): with
// delta_k = c_{k+1} - c_k the limited value is c_0 + r, r one of phi = sum v_i delta_i (the
// mean fbar), 0, delta_0, f_MD, f_UL, f_LC, so a face adds s gbar to its donor and its partials
// to the adjoints of four deltas; cell m's new lambda is lambda_m + (its donor term) +
// G_{m-1} - G_m, G_k the adjoint of delta_k.  A face whose limited value is phi or the donor
// and that has no adjoint pending on a limited curvature (most; neighbouring columns of a warp
// mostly agree) takes no more than that; the others find the source and scatter the
// curvature's partials in a branch.
//
// Bound by instruction issue: 66 thread instructions per update at 81 % issue where few faces
// take the branch, against 104 at 68 % when a line was marched in registers over the cells' own
// values, fully unrolled (lines of 16, 32, 64 cells; others walked global memory).  x sweep of
// 32^3 x 16^3 0.527 -> 0.300 ms (DRAM alone 0.238), of 24^3 x 16^3 0.389 -> 0.142 (0.100), of 20 x 22
// x 48 x 20 x 16 x 12 0.572 -> 0.196 (0.144).  Where many faces are limited the branch counts: the
// x sweep of a 24^3 x 16^3 run 0.190 with the minmod's partials found from its four arguments at
// every such face, 0.174 from the two magnitudes, 0.161 and only where an adjoint is pending.
#include <type_traits>

#include "vk_tiles.cuh"

namespace vk {

namespace {

constexpr int kMaxThreads = 768; // of all groups (80 registers a thread)
constexpr int kMaxSlots = 24;
constexpr int kHead = ((3 * kMaxSlots * 8 + 127) & ~127) + int(kMaxVel * sizeof(LineCoefT<float>));

struct AdjFaces {
    const Lim<float> &k;
    float c0, cp1, dmm, dm, dp; // donor j and the next cell; delta_{j-2} .. delta_j
    float hm, hp, d0, qm;       // halves of dm, dp; curvature of cell j; limited curvature at j - 1/2
    float gq;                   // adjoint of dm4 at j - 1/2 from face j - 1
    float gl, g0, g1, g2;       // adjoints of delta_{j-3} (complete) .. delta_j
    float b0, b1;               // lambda + donor term of cells j - 2, j - 1
    float l0;                   // lambda of cell j

    __device__ __forceinline__ AdjFaces(const Lim<float> &kk) : k(kk) {}

    // cells -2, -1, 0, 1 and lambda of cell 0
    __device__ __forceinline__ void start(float m2, float m1, float s0, float s1, float lam0)
    {
        c0 = s0;
        cp1 = s1;
        dmm = m1 - m2;
        dm = s0 - m1;
        dp = s1 - s0;
        hm = 0.5f * dm;
        hp = 0.5f * dp;
        d0 = dp - dm;
        qm = limited_curv(dm - dmm, d0);
        gq = gl = g0 = g1 = g2 = b0 = b1 = 0.f;
        l0 = lam0;
    }
    // adjoint x of dm4 at j - 1/2 = minmod(4 a - b, 4 b - a, a, b), a and b the curvatures of
    // cells j - 1 and j: the argument of least magnitude is 4 a - b where |b| >= 3 |a|, 4 b - a
    // where |a| >= 3 |b|, else the smaller of a and b; nothing where the minmod is 0
    __device__ __forceinline__ void scatter_curv(float x)
    {
        const float a = fabsf(dm - dmm), b = fabsf(d0);
        const bool ia = b >= 3.f * a, ib = a >= 3.f * b, i0 = a <= b;
        if (qm == 0.f) x = 0.f;
        const float xm = x * (ia ? 4.f : ib ? -1.f : i0 ? 1.f : 0.f), x0 = x * (ia ? -1.f : ib ? 4.f : i0 ? 0.f : 1.f);
        g0 -= xm;
        g1 += xm - x0;
        g2 += x0;
    }
    // face j + 1/2; cp2 = cell j + 2, l1 = lambda of cell j + 1.  Returns cell j - 2's lambda.
    __device__ __forceinline__ float face(float cp2, float l1)
    {
        const float dpp = cp2 - cp1, dn = dpp - dp;
        const float qp = limited_curv(d0, dn);
        const float phi = fmaf(k.v3, dpp, fmaf(k.v2, dp, fmaf(k.v1, dm, k.v0 * dmm)));
        const float md = fmaf(float(CurvScale<float>::md), qp, hp), lc = fmaf(float(CurvScale<float>::lc), qm, hm);
        const float ul = k.alpha * dm;
        const float r = mp_clamp(phi, dp, md, ul, lc);
        const float F = fmaf(k.s, r, k.s * c0); // before the clamp to [0, c0]
        const float gbar = l1 - l0;
        const bool over = F > c0;
        const float gv = F >= 0.f && !over ? k.s * gbar : 0.f; // adjoint of c0 + r
        const float b2 = l0 + (over ? gbar : gv);
        const bool isf = r == phi;
        const float gf = isf ? gv : 0.f;
        g0 = fmaf(gf, k.v0, g0);
        g1 = fmaf(gf, k.v1, g1);
        g2 = fmaf(gf, k.v2, g2);
        float gn = 0.f; // adjoint of dm4 at j + 1/2
        if ((!isf && r != 0.f) || gq != 0.f) {
            // the source of r, first match in the order phi, 0, delta_0, f_MD, f_UL, f_LC
            const float x = isf || r == 0.f ? 0.f : gv;
            const bool e1 = r == dp, em = !e1 && r == md, eu = !e1 && !em && r == ul, el = !e1 && !em && !eu;
            g2 = fmaf(x, e1 ? 1.f : em ? 0.5f : 0.f, g2);
            g1 = fmaf(x, eu ? k.alpha : el ? 0.5f : 0.f, g1);
            gn = em ? -0.5f * x : 0.f;
            const float y = el ? fmaf(4.f / 3.f, x, gq) : gq;
            if (y != 0.f) scatter_curv(y);
        }
        const float out = b0 + (gl - g0);
        gl = g0;
        g0 = g1;
        g1 = g2;
        g2 = gf * k.v3;
        gq = gn;
        b0 = b1;
        b1 = b2;
        l0 = l1;
        c0 = cp1;
        cp1 = cp2;
        dmm = dm;
        dm = dp;
        dp = dpp;
        hm = hp;
        hp = 0.5f * dpp;
        d0 = dn;
        qm = qp;
        return out;
    }
};

// One line: row r of f at p + r st (bytes), of lambda at q + r st, L >= 6 rows; new lambda over f.
// ROT: lambda read `shift` cells on.  Returns the sum of the new values.  One body for both
// directions: with one for each the instruction cache did not hold them (24^3 x 16^3 158 ->
// 140 us); folding the ends of the line into the loop as well cost more than it saved (147 us).
template <bool ROT>
__device__ __forceinline__ float adjoint_line(unsigned char *p, const unsigned char *q, int st, int L, int shift,
                                              const Lim<float> &lim)
{
    auto cell = [&](int r) -> float & { return *reinterpret_cast<float *>(p + r * st); };
    int lr = ROT ? shift : 0; // the next row of lambda
    if (ROT) q += shift * st;
    auto next_lam = [&]() {
        const float v = *reinterpret_cast<const float *>(q);
        q += st;
        if (ROT && ++lr == L) {
            lr = 0;
            q -= L * st;
        }
        return v;
    };
    const float lam0 = next_lam();
    if (lim.s == 0.f) { // an integer Courant number: no flux, lambda passes through
        float sum = lam0;
        cell(0) = lam0;
#pragma unroll 1
        for (int i = 1; i < L; ++i) {
            p += st;
            const float v = next_lam();
            cell(0) = v;
            sum += v;
        }
        return sum;
    }
    const float s0 = cell(0), s1 = cell(1);
    AdjFaces m(lim);
    m.start(cell(L - 2), cell(L - 1), s0, s1, lam0);
    // faces 0 .. 3: delta_{-2}, delta_{-1} and delta_0 also meet the last faces; cells 0 and 1 wait
    m.face(cell(2), next_lam());
    const float pa = m.gl; // G_{-2} so far
    m.face(cell(3), next_lam());
    const float pb = m.gl; // G_{-1} so far
    float o0 = m.face(cell(4), next_lam());
    float o1 = m.face(cell(5), next_lam());
    unsigned char *const first = p;
    p += 2 * st; // row j - 2 of the next face, j = 4
    float sum = 0.f;
    auto block = [&](auto width) {
        constexpr int B = decltype(width)::value;
        float c[B], l[B];
#pragma unroll
        for (int i = 0; i < B; ++i) {
            c[i] = cell(4 + i);
            l[i] = next_lam();
        }
#pragma unroll
        for (int i = 0; i < B; ++i) {
            const float v = m.face(c[i], l[i]);
            cell(i) = v;
            sum += v;
        }
        p += B * st;
    };
    int left = L - 6;
#pragma unroll 1
    for (; left >= 4; left -= 4) block(std::integral_constant<int, 4>());
#pragma unroll 1
    for (; left > 0; --left) block(std::integral_constant<int, 1>());
    const float e4 = m.face(s0, next_lam()); // face L - 2
    const float e3 = m.face(s1, lam0);       // face L - 1
    cell(0) = e4;
    cell(1) = e3;
    if (m.gq != 0.f) m.scatter_curv(m.gq); // dm4 at L - 1/2
    // m.g0, g1, g2 are now what the last faces add to G_{-2}, G_{-1} and G_0
    const float G2 = m.g0 + pa, G1 = m.g1 + pb;
    const float e2 = m.b0 + (m.gl - G2), e1 = m.b1 + (G2 - G1);
    o0 += m.g1 - m.g2;
    o1 += m.g2;
    cell(2) = e2;
    cell(3) = e1;
    *reinterpret_cast<float *>(first) = o0;
    *reinterpret_cast<float *>(first + st) = o1;
    return sum + ((e4 + e3) + (e2 + e1)) + (o0 + o1);
}

template <int COLS>
__global__ void __launch_bounds__(kMaxThreads + kProducer, 1)
    adjoint_tile_kernel(const __grid_constant__ CUtensorMap fmap, const __grid_constant__ CUtensorMap lmap,
                        const __grid_constant__ AdjTileArgs a)
{
    constexpr int kRow = COLS * 4;
    extern __shared__ __align__(128) unsigned char smem[];
    const int L = a.L, S = a.slots, NT = a.groups * COLS;
    uint64_t *full = reinterpret_cast<uint64_t *>(smem); // 2S: the slot holds its tiles (full_bar)
    uint64_t *done = full + 2 * S;                       // S: the tile's group is done with it
    LineCoefT<float> *tab = reinterpret_cast<LineCoefT<float> *>(smem + ((3 * kMaxSlots * 8 + 127) & ~127));
    unsigned char *ring = smem + kHead + ((128u - ((smem_u32(smem) + unsigned(kHead)) & 127u)) & 127u);
    const int half = L * kRow; // bytes of one tile
    auto slot = [&](unsigned k) { return ring + size_t(2 * half) * (k % S); };

    if (threadIdx.x == 0) {
        for (int q = 0; q < 2 * S; ++q) mbar_init(&full[q], 1);
        for (int q = 0; q < S; ++q) mbar_init(&done[q], COLS);
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
            mbar_arrive_expect_tx(bar, unsigned(2 * half)); // whole boxes, clipped or not
            tma_load_3d(slot(k), &fmap, bar, int(ti * COLS), 0, int(o));
            tma_load_3d(slot(k) + half, &lmap, bar, int(ti * COLS), 0, int(o));
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
            tma_store_3d(&lmap, slot(k), int(ti * COLS), 0, int(o));
            bulk_commit();
            if (loaded < n_my) {
                bulk_wait_read_at_most(0);
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

    const int grp = threadIdx.x / COLS, tid = threadIdx.x % COLS;
    bool bad = false;
    for (unsigned k = grp; k < n_my; k += a.groups) {
        if (!__all_sync(0xffffffffu, wait_tile(full, k, S))) {
            atomicOr(a.err, ERR_TIMEOUT);
            return;
        }
        unsigned ti, o;
        coords(k, ti, o);
        const unsigned col = fdiv(ti * COLS + tid, a.div_vstride);
        const LineCoefT<float> kc = tab[col - fdiv(col, a.div_nvel) * unsigned(a.nvel)];
        unsigned char *p = slot(k) + 4 * tid;
        const bool same = kc.nd < 0; // line left unchanged by the forward sweep: identity
        const bool neg = !same && (kc.nd & 1);
        Lim<float> lim = to_lim(kc);
        if (same) lim.s = 0.f;
        const int shift = same ? 0 : (kc.nd >> 1) % L;
        // a negative Courant number is the mirror image: the line walked from its far end
        if (neg) p += (L - 1) * kRow;
        float sum;
        // (columns past the end of a row hold zeros: marched, never stored)
        const int st = neg ? -kRow : kRow;
        if (__any_sync(0xffffffffu, shift != 0)) sum = adjoint_line<true>(p, p + half, st, L, shift, lim);
        else sum = adjoint_line<false>(p, p + half, st, L, 0, lim);
        bad |= !same && !isfinite(sum);
        fence_proxy_async();
        mbar_arrive(&done[k % S]);
    }
    if (bad) atomicOr(a.err, ERR_NAN);
}

const void *adjoint_tile(int cols) { return cols == 128 ? (const void *)adjoint_tile_kernel<128> : (const void *)adjoint_tile_kernel<64>; }

size_t adjoint_tile_smem(const AdjTileArgs &a) { return kHead + 128 + size_t(a.slots) * a.L * a.cols * 8; }

} // namespace

bool adjoint_tile_geometry(int L, long long n_inner, long long n_outer, AdjTileArgs &a)
{
    if (L < 6 || L > 256 || n_inner < 64 || n_inner % 4 || n_inner > 0x7fffff00ll) return false;
    auto fit = [&](int cols) { return int((227 * 1024 - kHead - 128) / (L * cols * 8)); };
    a.cols = n_inner >= 128 && fit(128) >= 6 ? 128 : 64;
    const long long tiles = (n_inner + a.cols - 1) / a.cols;
    if (n_outer * tiles > 0x7fffffffll) return false;
    a.L = L;
    a.tiles_inner = unsigned(tiles);
    a.num_tiles = unsigned(n_outer * tiles);
    a.slots = fit(a.cols) < kMaxSlots ? fit(a.cols) : kMaxSlots;
    if (a.slots < 4) return false;
    a.groups = a.slots - (a.slots >= 6 ? a.slots / 4 : 1);
    if (a.groups > kMaxThreads / a.cols) a.groups = kMaxThreads / a.cols;
    return true;
}

cudaError_t launch_adjoint_tile(const CUtensorMap &fmap, const CUtensorMap &lmap, const AdjTileArgs &args, int sms, cudaStream_t st)
{
    if (args.num_tiles == 0) return cudaSuccess;
    if ((args.cols != 128 && args.cols != 64) || args.groups < 1 || args.slots < args.groups || args.nvel <= 0 ||
        args.nvel > kMaxVel || args.vstride <= 0)
        return cudaErrorInvalidValue;
    AdjTileArgs a = args;
    a.div_tiles = make_fastdiv(a.tiles_inner);
    a.div_vstride = make_fastdiv(unsigned(a.vstride));
    a.div_nvel = make_fastdiv(unsigned(a.nvel));
    const size_t smem = adjoint_tile_smem(a);
    const cudaError_t e = allow_smem(adjoint_tile(a.cols), smem);
    if (e != cudaSuccess) return e;
    const unsigned grid = a.num_tiles < unsigned(sms) ? a.num_tiles : unsigned(sms);
    void *params[] = {const_cast<CUtensorMap *>(&fmap), const_cast<CUtensorMap *>(&lmap), &a};
    return launch_chained((long long)a.num_tiles * a.cols * a.L, adjoint_tile(a.cols), dim3(grid), dim3(a.groups * a.cols + kProducer),
                          smem, st, params);
}

} // namespace vk
