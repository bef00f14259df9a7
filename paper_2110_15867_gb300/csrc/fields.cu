// fields.cu -- the small spatial-grid kernels around the sweeps
// (Yoshikawa, Tanaka & Yoshida, SC'21):
//   * velocity-sweep coefficients: g_i = d phi / d x_i by the periodic
//     4th-order central difference (the "differentiating" of the PM potential,
//     Sec. 4.1.2) and the Courant number nu = -g_i dt / du of Eq. (4);
//   * the density moment rho_nu(x) = int f d^3u (Sec. 4.1.3: every spatial
//     cell holds its whole velocity cube, so the moment needs no exchange);
//   * the total mass (compensated FP64);
//   * the periodic Poisson solve of Eq. (2) by discrete Fourier transform
//     (the convolution method of Sec. 4.1.2 on one GPU).
#include <type_traits>

#include "vk_common.cuh"

namespace vk {

// ----------------------------------------------------------------------------
// velocity-sweep coefficients
// ----------------------------------------------------------------------------

// One thread per cell and axis (blockIdx.y): the FP64 chain of a cell (the gradient, the five
// weights, a division; FP64 runs at 2 lanes per SM and clock) is what a small grid waits
// for, so its axes run side by side and small grids take small blocks, which spread over
// more SMs.  8^3 cells: 25 us with one thread per cell walking the three axes in blocks of
// 256, 8 us here; 64 x 64 x 32: 83 -> 48 us.
struct CoefAxes {
    double scale[3]; // nu = scale (8 (phi_+1 - phi_-1) - (phi_+2 - phi_-2)): -dt / (12 h du)
    int axis[3];
};
template <typename C>
__global__ void velocity_coef_kernel(int nx, int ny, int nz, const float *__restrict__ phi, CoefAxes ax,
                                     LineCoefT<C> *cx, LineCoefT<C> *cy, LineCoefT<C> *cz, unsigned *err)
{
    const unsigned ncell = unsigned(nx) * ny * nz; // <= 2^24
    const unsigned c = blockIdx.x * blockDim.x + threadIdx.x;
    chain_enter();
    if (c >= ncell) return;
    const int d = ax.axis[blockIdx.y];
    const int st = d == 2 ? 1 : d == 1 ? nz : ny * nz, n = d == 2 ? nz : d == 1 ? ny : nx;
    const int i = int(c / unsigned(st) % unsigned(n));
    auto at = [&](int o) { // cell i + o of the periodic line, |o| <= 2 <= n
        const int q = i + o;
        return (double)phi[int(c) + (q < 0 ? o + n : q >= n ? o - n : o) * st];
    };
    const double nu = ax.scale[blockIdx.y] * (8.0 * (at(1) - at(-1)) - (at(2) - at(-2)));
    LineCoefT<C> k = make_line_coef<C>(nu);
    if (!(fabs(nu) < 1.0)) { // also catches NaN
        k.nd = -1;
        atomicOr(err, ERR_CFL);
    }
    (d == 0 ? cx : d == 1 ? cy : cz)[c] = k;
}

cudaError_t launch_velocity_coef(const GridDims &g, const float *phi, double dt, int mask, void *coef_x,
                                 void *coef_y, void *coef_z, int dtype, unsigned *err, cudaStream_t st)
{
    const long long ncell = (long long)g.n[0] * g.n[1] * g.n[2];
    CoefAxes ax{};
    int axes = 0;
    for (int d = 0; d < 3; ++d) {
        if (!(mask & (1 << d))) continue;
        const double h = g.L / g.n[d], du = 2.0 * g.V / g.nu[d];
        ax.scale[axes] = -dt / (12.0 * h * du);
        ax.axis[axes++] = d;
    }
    if (!axes) return cudaSuccess;
    const int threads = ncell >= 65536 ? 128 : 32;
    const dim3 grid(unsigned((ncell + threads - 1) / threads), unsigned(axes));
    const long long velocity = (long long)g.nu[0] * g.nu[1] * g.nu[2];
    auto launch = [&](auto kernel, auto *cx, auto *cy, auto *cz) {
        return launch_chained_t(ncell * velocity * (dtype == 0 ? 16 : 1), kernel, grid, dim3(threads), 0, st, g.n[0], g.n[1], g.n[2], phi, ax, cx, cy, cz, err);
    };
    if (dtype == 0)
        return launch(velocity_coef_kernel<double>, (LineCoefT<double> *)coef_x, (LineCoefT<double> *)coef_y,
                      (LineCoefT<double> *)coef_z);
    return launch(velocity_coef_kernel<float>, (LineCoefT<float> *)coef_x, (LineCoefT<float> *)coef_y,
                  (LineCoefT<float> *)coef_z);
}

// ----------------------------------------------------------------------------
// moment
// ----------------------------------------------------------------------------

// Neumaier step in the working precision: (s, c) accumulates x exactly up to
// the second-order term; s + c is formed only in FP64.
__device__ __forceinline__ void neumaier(float &s, float &c, float x)
{
    const float t = s + x;
    c += (fabsf(s) >= fabsf(x)) ? ((s - t) + x) : ((x - t) + s);
    s = t;
}

__device__ __forceinline__ double warp_sum_d(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// One CTA per spatial cell (grid-stride): FP32 compensated partial sums over
// 16-byte vectors, combined in FP64 across the CTA in a fixed order.
template <typename T>
__global__ void __launch_bounds__(256) moment_kernel(GridDims g, const T *__restrict__ f, double *rho)
{
    const long long ncell = (long long)g.n[0] * g.n[1] * g.n[2];
    const long long cube = (long long)g.nu[0] * g.nu[1] * g.nu[2];
    const double du3 = (2.0 * g.V / g.nu[0]) * (2.0 * g.V / g.nu[1]) * (2.0 * g.V / g.nu[2]);
    __shared__ double part[8];
    for (long long c = blockIdx.x; c < ncell; c += gridDim.x) {
        const T *q = f + c * cube;
        double tot;
        if (sizeof(T) == 8) {
            double s = 0.0, e = 0.0;
            for (long long k = threadIdx.x; k < cube; k += blockDim.x) {
                const double x = (double)q[k];
                const double t = s + x;
                e += (fabs(s) >= fabs(x)) ? ((s - t) + x) : ((x - t) + s);
                s = t;
            }
            tot = s + e;
        } else {
            float s = 0.f, e = 0.f;
            const float4 *q4 = reinterpret_cast<const float4 *>(q);
            const long long n4 = cube / 4;
            for (long long k = threadIdx.x; k < n4; k += blockDim.x) {
                const float4 v = q4[k];
                neumaier(s, e, v.x);
                neumaier(s, e, v.y);
                neumaier(s, e, v.z);
                neumaier(s, e, v.w);
            }
            tot = (double)s + (double)e;
        }
        tot = warp_sum_d(tot);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = tot;
        __syncthreads();
        if (threadIdx.x == 0) {
            double r = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += part[w];
            rho[c] = du3 * r;
        }
        __syncthreads();
    }
}

// 16-bit storage: value = code * scale of its u_z line; 16-byte vectors of 8
// codes never straddle a line (n_uz is a multiple of 8).
template <typename T>
__global__ void __launch_bounds__(256) moment_coded_kernel(GridDims g, const T *__restrict__ f,
                                                           const float *__restrict__ scale, double *rho)
{
    const long long ncell = (long long)g.n[0] * g.n[1] * g.n[2];
    const int nuz = g.nu[2];
    const long long lines = (long long)g.nu[0] * g.nu[1];
    const long long cube = lines * nuz;
    const double du3 = (2.0 * g.V / g.nu[0]) * (2.0 * g.V / g.nu[1]) * (2.0 * g.V / g.nu[2]);
    __shared__ double part[8];
    // 16-byte vectors per line: 2 or 4 (n_uz 16 or 32, a shift), else 3, 5 or 6 (n_uz 24, 40, 48)
    const int vpl = nuz / 8, vshift = nuz == 32 ? 2 : 1;
    const bool pow2 = nuz == 16 || nuz == 32;
    for (long long c = blockIdx.x; c < ncell; c += gridDim.x) {
        const uint4 *q = reinterpret_cast<const uint4 *>(f + c * cube);
        const float *sc = scale + c * lines;
        float s = 0.f, e = 0.f;
        for (int k = threadIdx.x; k < int(cube / 8); k += blockDim.x) {
            const uint4 v = q[k];
            const unsigned u[4] = {v.x, v.y, v.z, v.w};
            // eight codes of 8 (BF16) or 11 (FP16) significant bits: their FP32 sum is
            // exact or off by the last bit
            float t = 0.f;
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                float2 x;
                if (std::is_same<T, __nv_bfloat16>::value)
                    x = make_float2(__uint_as_float(u[j] << 16), __uint_as_float(u[j] & 0xffff0000u));
                else
                    x = __half22float2(*reinterpret_cast<const __half2 *>(&u[j]));
                t += x.x + x.y;
            }
            // the product and its rounding error (exact, by FMA) both enter the sum
            const float w = sc[pow2 ? k >> vshift : k / vpl];
            const float pr = t * w;
            neumaier(s, e, pr);
            e += fmaf(t, w, -pr);
        }
        double tot = warp_sum_d((double)s + (double)e);
        if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = tot;
        __syncthreads();
        if (threadIdx.x == 0) {
            double r = 0.0;
            for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += part[w];
            rho[c] = du3 * r;
        }
        __syncthreads();
    }
}

cudaError_t launch_moment_coded(const GridDims &g, const void *f, const float *scale, int dtype, double *rho,
                                cudaStream_t st, int sm_count)
{
    const long long ncell = (long long)g.n[0] * g.n[1] * g.n[2];
    const long long blocks = ncell < (long long)sm_count * 8 ? ncell : (long long)sm_count * 8;
    if (dtype == 2)
        moment_coded_kernel<__nv_bfloat16><<<int(blocks), 256, 0, st>>>(g, (const __nv_bfloat16 *)f, scale, rho);
    else
        moment_coded_kernel<__half><<<int(blocks), 256, 0, st>>>(g, (const __half *)f, scale, rho);
    return cudaGetLastError();
}

cudaError_t launch_moment(const GridDims &g, const void *f, int dtype, double *rho, cudaStream_t st,
                          int sm_count)
{
    const long long ncell = (long long)g.n[0] * g.n[1] * g.n[2];
    const long long blocks = ncell < (long long)sm_count * 8 ? ncell : (long long)sm_count * 8;
    if (dtype == 0)
        moment_kernel<double><<<int(blocks), 256, 0, st>>>(g, (const double *)f, rho);
    else
        moment_kernel<float><<<int(blocks), 256, 0, st>>>(g, (const float *)f, rho);
    return cudaGetLastError();
}

// The moment fused into the x sweep: the velocity cube of spatial cell
// x cells_per_row + c arrives as nparts partial sums (in the storage type) laid out
// [c][part][x]; rho = du^3 x their sum in FP64 in a fixed order.  One block per c:
// 4 groups of 64 threads (x) take every 4th part, then one group adds the 4 sums.
template <typename P>
__global__ void __launch_bounds__(256) moment_finish_kernel(const P *__restrict__ mpart, int nparts, int nx,
                                                            long long cells_per_row, double du3, double *rho)
{
    __shared__ double red[4][64];
    const int tx = threadIdx.x & 63, grp = threadIdx.x >> 6;
    chain_enter();
    for (long long c = blockIdx.x; c < cells_per_row; c += gridDim.x) {
        const P *q = mpart + c * nparts * (long long)nx;
        for (int x0 = 0; x0 < nx; x0 += 64) {
            const int x = x0 + tx;
            double s = 0.0;
            if (x < nx)
                for (int k = grp; k < nparts; k += 4) s += double(q[(long long)k * nx + x]);
            red[grp][tx] = s;
            __syncthreads();
            if (grp == 0 && x < nx) rho[x * cells_per_row + c] = du3 * (((red[0][tx] + red[1][tx]) + red[2][tx]) + red[3][tx]);
            __syncthreads();
        }
    }
}

cudaError_t launch_moment_finish(const void *mpart, int dtype, int nparts, int nx, long long cells_per_row, double du3,
                                 double *rho, cudaStream_t st, int sm_count)
{
    const long long blocks = cells_per_row < (long long)sm_count * 8 ? cells_per_row : (long long)sm_count * 8;
    if (dtype == 0)
        return launch_chained_t(cells_per_row * nx * nparts * 128 * 16, moment_finish_kernel<double>, dim3(unsigned(blocks)), dim3(256), 0, st, (const double *)mpart,
                                nparts, nx, cells_per_row, du3, rho);
    return launch_chained_t(cells_per_row * nx * nparts * 256, moment_finish_kernel<float>, dim3(unsigned(blocks)), dim3(256), 0, st, (const float *)mpart, nparts,
                            nx, cells_per_row, du3, rho);
}

// Adjoint of the moment: rho(x) = du^3 sum_u f(x, u), so dL/df(x, u) =
// du^3 dL/drho(x) for every u.  lam (+)= that, 16 bytes per thread and step.
template <typename T>
__global__ void __launch_bounds__(256) moment_adjoint_kernel(GridDims g, const double *__restrict__ dLdrho, T *lam,
                                                             int accumulate)
{
    constexpr int V = 16 / int(sizeof(T));
    const long long cube = (long long)g.nu[0] * g.nu[1] * g.nu[2];
    const long long nvec = (long long)g.n[0] * g.n[1] * g.n[2] * cube / V;
    const double du3 = (2.0 * g.V / g.nu[0]) * (2.0 * g.V / g.nu[1]) * (2.0 * g.V / g.nu[2]);
    uint4 *q = reinterpret_cast<uint4 *>(lam);
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < nvec; i += (long long)gridDim.x * blockDim.x) {
        const T v = T(du3 * dLdrho[(i * V) / cube]); // a 16-byte vector never straddles a cell (cube % 64 == 0)
        uint4 u = accumulate ? q[i] : make_uint4(0, 0, 0, 0);
        T *e = reinterpret_cast<T *>(&u);
#pragma unroll
        for (int k = 0; k < V; ++k) e[k] += v;
        q[i] = u;
    }
}

cudaError_t launch_moment_adjoint(const GridDims &g, const double *dLdrho, int dtype, void *lam, int accumulate,
                                  cudaStream_t st, int sm_count)
{
    const int threads = 256;
    const int blocks = sm_count * 8;
    if (dtype == 0)
        moment_adjoint_kernel<double><<<blocks, threads, 0, st>>>(g, dLdrho, (double *)lam, accumulate);
    else
        moment_adjoint_kernel<float><<<blocks, threads, 0, st>>>(g, dLdrho, (float *)lam, accumulate);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// velocity moments: density, mean velocity, velocity dispersion tensor
// ----------------------------------------------------------------------------
// Sec. 4.1.3 keeps each spatial cell's velocity cube in one place so that these
// need no communication.  Per cell: S0 = sum f, S1_i = sum u_i f, S2_ij = sum
// u_i u_j f over the velocity cell centres; rho = du^3 S0, umean_i = S1_i / S0,
// sigma2_ij = S2_ij / S0 - umean_i umean_j (0 where S0 = 0).

// 16 bytes of storage -> N values (x the row's scale for 16-bit codes)
template <typename T> struct Vec16;
template <> struct Vec16<float> {
    static constexpr int N = 4;
    __device__ static void get(const uint4 &u, float, float (&o)[4])
    {
        o[0] = __uint_as_float(u.x); o[1] = __uint_as_float(u.y);
        o[2] = __uint_as_float(u.z); o[3] = __uint_as_float(u.w);
    }
};
template <> struct Vec16<double> {
    static constexpr int N = 2;
    __device__ static void get(const uint4 &u, double, double (&o)[2])
    {
        o[0] = __hiloint2double(int(u.y), int(u.x));
        o[1] = __hiloint2double(int(u.w), int(u.z));
    }
};
template <> struct Vec16<__nv_bfloat16> {
    static constexpr int N = 8;
    __device__ static void get(const uint4 &u, float sc, float (&o)[8])
    {
        const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            o[2 * q] = __fmul_rn(__uint_as_float(w[q] << 16), sc);
            o[2 * q + 1] = __fmul_rn(__uint_as_float(w[q] & 0xffff0000u), sc);
        }
    }
};
template <> struct Vec16<__half> {
    static constexpr int N = 8;
    __device__ static void get(const uint4 &u, float sc, float (&o)[8])
    {
        const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const float2 h = __half22float2(*reinterpret_cast<const __half2 *>(&w[q]));
            o[2 * q] = __fmul_rn(h.x, sc);
            o[2 * q + 1] = __fmul_rn(h.y, sc);
        }
    }
};

// compensated accumulator in the working precision
template <typename C> struct NSum {
    C s, c;
    __device__ void add(C x)
    {
        const C t = s + x;
        c += (fabs(s) >= fabs(x)) ? ((s - t) + x) : ((x - t) + s);
        s = t;
    }
    __device__ double get() const { return (double)s + (double)c; }
};

// The sums over the warp of v[0] .. v[15]: at each step a lane keeps half of its sums and
// hands the other half to its partner, 16 FP64 additions instead of 5 per sum (FP64 runs at
// two lanes per SM and clock).  Lanes 2 k and 2 k + 1 end with sum k, in a fixed order.
__device__ __forceinline__ double warp_sums16(double (&v)[16], int lane)
{
#pragma unroll
    for (int o = 16, n = 8; o > 1; o >>= 1, n >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int k = 0; k < n; ++k) {
            const double give = up ? v[k] : v[k + n];
            v[k] = (up ? v[k + n] : v[k]) + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// One warp per spatial cell: each lane sums every 32nd 16-byte vector of the
// cube, then the ten sums are combined across the warp in FP64 in a fixed order
// (32 x 32 x 24 x 32^3 FP32 cells: 0.710 ms with ten separate warp sums, 0.546 here; 0.476 at
// the copy rate).
template <typename T>
__global__ void __launch_bounds__(256) moments_kernel(GridDims g, const T *__restrict__ f,
                                                      const float *__restrict__ scale, double *rho, double *umean,
                                                      double *sigma2)
{
    using C = typename Compute<T>::type;
    constexpr int N = Vec16<T>::N;
    const long long ncell = (long long)g.n[0] * g.n[1] * g.n[2];
    const int nux = g.nu[0], nuy = g.nu[1], nuz = g.nu[2];
    const int nvec = nux * nuy * nuz / N; // 16-byte vectors per cube
    const int vrow = nuz / N;             // per u_z line
    const double du3 = (2.0 * g.V / nux) * (2.0 * g.V / nuy) * (2.0 * g.V / nuz);
    // n / d as a multiply-high by floor((2^32 - 1) / d) + 1: exact while n d < 2^32
    // (here n < 2^21, d <= 128)
    const unsigned mv = 0xffffffffu / unsigned(vrow) + 1u, my = 0xffffffffu / unsigned(nuy) + 1u;
    auto div_vrow = [&](int n) { return vrow == 1 ? n : int(__umulhi(unsigned(n), mv)); };
    auto div_nuy = [&](int n) { return int(__umulhi(unsigned(n), my)); };
    __shared__ C su[3][kMaxVel]; // velocity cell centres, formed in FP64 and rounded once
    for (int j = threadIdx.x; j < kMaxVel; j += blockDim.x)
        for (int d = 0; d < 3; ++d) su[d][j] = j < g.nu[d] ? C(-g.V + (j + 0.5) * (2.0 * g.V / g.nu[d])) : C(0);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
    for (long long cell = blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5); cell < ncell; cell += warps) {
        const uint4 *q = reinterpret_cast<const uint4 *>(f + cell * (long long)nvec * N);
        const float *sc = scale ? scale + cell * nux * nuy : nullptr;
        // S0 compensated; the other nine sums in the working precision
        NSum<C> s0{C(0), C(0)};
        C acc[9];
#pragma unroll
        for (int k = 0; k < 9; ++k) acc[k] = C(0);
#pragma unroll 4
        for (int k = lane; k < nvec; k += 32) {
            const int row = div_vrow(k), jz0 = (k - row * vrow) * N;
            const int jx = div_nuy(row), jy = row - jx * nuy;
            C v[N];
            Vec16<T>::get(q[k], sc ? sc[row] : 1.f, v);
            const C ux = su[0][jx], uy = su[1][jy];
            C t0 = C(0), t1 = C(0), t2 = C(0);
#pragma unroll
            for (int e = 0; e < N; ++e) {
                const C uz = su[2][jz0 + e];
                const C w = uz * v[e];
                t0 += v[e];
                t1 += w;
                t2 += uz * w;
            }
            s0.add(t0);
            acc[0] += ux * t0;
            acc[1] += uy * t0;
            acc[2] += t1;
            acc[3] += ux * ux * t0;
            acc[4] += uy * uy * t0;
            acc[5] += t2;
            acc[6] += ux * uy * t0;
            acc[7] += ux * t1;
            acc[8] += uy * t1;
        }
        double v[16];
        v[0] = s0.get();
#pragma unroll
        for (int k = 1; k < 16; ++k) v[k] = k < 10 ? (double)acc[k - 1] : 0.0;
        const double mine = warp_sums16(v, lane); // sum k sits in lanes 2 k, 2 k + 1
        double S[10];
#pragma unroll
        for (int k = 0; k < 10; ++k) S[k] = __shfl_sync(0xffffffffu, mine, 2 * k);
        if (lane == 0) {
            const double S0 = S[0], inv = S0 != 0.0 ? 1.0 / S0 : 0.0;
            const double m[3] = {S[1] * inv, S[2] * inv, S[3] * inv};
            // S index of sigma2 component k (xx, yy, zz, xy, xz, yz) and its pair
            const int si[6] = {4, 5, 6, 7, 8, 9}, pi[6] = {0, 1, 2, 0, 0, 1}, pj[6] = {0, 1, 2, 1, 2, 2};
            if (rho) rho[cell] = du3 * S0;
            if (umean)
                for (int i = 0; i < 3; ++i) umean[i * ncell + cell] = m[i];
            if (sigma2)
                for (int k = 0; k < 6; ++k)
                    sigma2[k * ncell + cell] = S0 != 0.0 ? S[si[k]] * inv - m[pi[k]] * m[pj[k]] : 0.0;
        }
    }
}

cudaError_t launch_moments(const GridDims &g, const void *f, const float *scale, int dtype, double *rho,
                           double *umean, double *sigma2, cudaStream_t st, int sm_count)
{
    const long long ncell = (long long)g.n[0] * g.n[1] * g.n[2];
    const long long need = (ncell + 7) / 8; // 8 warps (cells) per block
    // one wave of resident blocks: each warp strides over the cells, so a second, partial
    // wave would leave most of the SMs idle for its whole length
    const void *kern = dtype == 0 ? (const void *)moments_kernel<double>
                       : dtype == 1 ? (const void *)moments_kernel<float>
                       : dtype == 2 ? (const void *)moments_kernel<__nv_bfloat16>
                                    : (const void *)moments_kernel<__half>;
    int per_sm = 0;
    const cudaError_t oe = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 256, 0);
    if (oe != cudaSuccess) return oe;
    if (per_sm < 1) per_sm = 1;
    const long long wave = (long long)sm_count * per_sm;
    const long long blocks = need < wave ? need : wave;
    switch (dtype) {
    case 0: moments_kernel<double><<<int(blocks), 256, 0, st>>>(g, (const double *)f, nullptr, rho, umean, sigma2); break;
    case 1: moments_kernel<float><<<int(blocks), 256, 0, st>>>(g, (const float *)f, nullptr, rho, umean, sigma2); break;
    case 2:
        moments_kernel<__nv_bfloat16><<<int(blocks), 256, 0, st>>>(g, (const __nv_bfloat16 *)f, scale, rho, umean, sigma2);
        break;
    default: moments_kernel<__half><<<int(blocks), 256, 0, st>>>(g, (const __half *)f, scale, rho, umean, sigma2); break;
    }
    return cudaGetLastError();
}

// y += x (FP64), or y = x when x_only
__global__ void axpy_kernel(long long n, const double *__restrict__ x, double *y, int assign)
{
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        y[i] = assign ? x[i] : y[i] + x[i];
}

cudaError_t launch_add(long long n, const double *x, double *y, bool assign, cudaStream_t st)
{
    const int threads = 256;
    const int blocks = int((n + threads - 1) / threads < 4096 ? (n + threads - 1) / threads : 4096);
    axpy_kernel<<<blocks, threads, 0, st>>>(n, x, y, assign ? 1 : 0);
    return cudaGetLastError();
}

// dx dy dz * sum rho, Neumaier in FP64 per thread, fixed-order combine
__global__ void __launch_bounds__(1024) mass_kernel(GridDims g, const double *__restrict__ rho, double *out)
{
    const long long ncell = (long long)g.n[0] * g.n[1] * g.n[2];
    double s = 0.0, e = 0.0;
    for (long long k = threadIdx.x; k < ncell; k += blockDim.x) {
        const double x = rho[k];
        const double t = s + x;
        e += (fabs(s) >= fabs(x)) ? ((s - t) + x) : ((x - t) + s);
        s = t;
    }
    __shared__ double ps[1024], pe[1024];
    ps[threadIdx.x] = s;
    pe[threadIdx.x] = e;
    __syncthreads();
    if (threadIdx.x == 0) {
        double S = 0.0, E = 0.0;
        for (unsigned i = 0; i < blockDim.x; ++i) {
            const double x = ps[i];
            const double t = S + x;
            E += (fabs(S) >= fabs(x)) ? ((S - t) + x) : ((x - t) + S);
            S = t;
            E += pe[i];
        }
        *out = (S + E) * (g.L / g.n[0]) * (g.L / g.n[1]) * (g.L / g.n[2]);
    }
}

cudaError_t launch_mass(const GridDims &g, const double *rho, double *out, cudaStream_t st)
{
    mass_kernel<<<1, 1024, 0, st>>>(g, rho, out);
    return cudaGetLastError();
}

// ----------------------------------------------------------------------------
// Poisson, Eq. (2)
// ----------------------------------------------------------------------------

// DFT along dimension d: out[.., k, ..] = sum_m in[.., m, ..] e^{sign 2 pi i k m / n_d},
// factored once (Cooley-Tukey) as n = n1 n2 with m = n2 m1 + m2 and k = k1 + n1 k2:
//   Y[k1][m2] = W_n^{m2 k1} sum_{m1} x[n2 m1 + m2] W_{n1}^{m1 k1},
//   X[k1 + n1 k2] = sum_{m2} Y[k1][m2] W_{n2}^{m2 k2},
// n (n1 + n2 + 1) complex products per line instead of n^2 (n1 = 1 for a prime n: the
// plain sum).  W_{n1} = W_n^{n2}, W_{n2} = W_n^{n1}: one twiddle table per axis.  A
// block holds `lines` lines of the axis in shared memory, n threads per line.
//
// The solve is five launches: z (reading rho + rho_bg), y, x forward with the division by k^2
// and x back on the same lines, y back, z back (writing phi).  Small grids are bound by the
// launches and by each one's chain of dependent FP64 operations and loads, so blocks are kept
// small there (more SMs) and the twiddles come through shared memory.  8^3: 67 us in nine
// launches, 38 us here; 64 x 64 x 32: 250 -> 226 us.
// One output per thread of the n-point transform of x (y: scratch); all threads of the block
// call it.  x must not be written again before the next barrier.
__device__ __forceinline__ double2 dft_point(const double2 *x, double2 *y, const double2 *tw, int n, int n1, int k, int sign,
                                             bool act)
{
    const int n2 = n / n1;
    __syncthreads();
    if (act) {
        // stage 1 for (k1, m2) = (k / n2, k % n2)
        const int k1 = k / n2, m2 = k % n2;
        double sr = 0.0, si = 0.0;
        int q = 0; // (n2 m1 k1) mod n
        for (int m1 = 0; m1 < n1; ++m1) {
            const double2 v = x[n2 * m1 + m2], w = tw[q];
            const double wi = sign * w.y;
            sr += v.x * w.x - v.y * wi;
            si += v.x * wi + v.y * w.x;
            q += n2 * k1; // < n
            if (q >= n) q -= n;
        }
        const double2 w = tw[(m2 * k1) % n];
        const double wi = sign * w.y;
        y[k] = make_double2(sr * w.x - si * wi, sr * wi + si * w.x); // Y[k1][m2] at k1 n2 + m2
    }
    __syncthreads();
    double sr = 0.0, si = 0.0;
    if (act) {
        // stage 2 for output k = k1 + n1 k2
        const int k1 = k % n1, k2 = k / n1;
        int q = 0; // (n1 m2 k2) mod n
        for (int m2 = 0; m2 < n2; ++m2) {
            const double2 v = y[k1 * n2 + m2], w = tw[q];
            const double wi = sign * w.y;
            sr += v.x * w.x - v.y * wi;
            si += v.x * wi + v.y * w.x;
            q += n1 * k2; // < n
            if (q >= n) q -= n;
        }
    }
    return make_double2(sr, si);
}

enum class Dft { first, plain, middle, last };
struct DftArgs {
    int n[3], d, sign, n1, lines;
    unsigned nlines;
    const double *rho, *bg; // first: the real input (bg may be null)
    const double2 *in, *tw;
    double2 *out;
    double fac, L;          // middle: forward, times -fac / k^2 (0 for k = 0), back
    float *phi;             // last: the real part / ncell, FP32 (the field the kicks read)
    double *phi64;          // or FP64 (the adjoint's dL/drho); either may be null
};

template <Dft M> __global__ void __launch_bounds__(256) dft_axis_kernel(const __grid_constant__ DftArgs a)
{
    extern __shared__ double2 dft_smem[];
    const int d = a.d, n = a.n[d];
    const int st = d == 2 ? 1 : d == 1 ? a.n[2] : a.n[1] * a.n[2];
    // the other two dimensions of a line, in memory order
    const int da = d == 0 ? 1 : 0, db = d == 2 ? 1 : 2;
    const int sa = da == 0 ? a.n[1] * a.n[2] : a.n[2], sb = db == 1 ? a.n[2] : 1;
    const int li = threadIdx.x / n, k = threadIdx.x - li * n; // this thread: line li of the block, index k
    double2 *tw = dft_smem, *x = tw + n + li * n, *y = tw + n + (a.lines + li) * n;
    for (int q = threadIdx.x; q < n; q += blockDim.x) tw[q] = a.tw[q]; // written at start-up: no kernel before writes it
    chain_enter();
    const unsigned line = blockIdx.x * unsigned(a.lines) + li;
    const bool act = line < a.nlines;
    const int ia = int(line / unsigned(a.n[db])), ib = int(line - unsigned(ia) * a.n[db]);
    const int e = ia * sa + ib * sb + k * st; // < 2^24
    if (act) x[k] = M == Dft::first ? make_double2(a.rho[e] + (a.bg ? a.bg[e] : 0.0), 0.0) : a.in[e];
    double2 v = dft_point(x, y, tw, n, a.n1, k, a.sign, act);
    if constexpr (M == Dft::middle) {
        const int id[3] = {k, ia, ib}; // d = 0
        double k2 = 0.0;
        for (int q = 0; q < 3; ++q) {
            const int w = id[q] < (a.n[q] + 1) / 2 ? id[q] : id[q] - a.n[q]; // integer wave number
            const double kq = 2.0 * M_PI * (double)w / a.L;
            k2 += kq * kq;
        }
        const double s = (k2 == 0.0) ? 0.0 : -a.fac / k2;
        __syncthreads();
        if (act) x[k] = make_double2(v.x * s, v.y * s);
        v = dft_point(x, y, tw, n, a.n1, k, -a.sign, act);
    }
    if (!act) return;
    if constexpr (M == Dft::last) {
        const double p = v.x * (1.0 / ((double)a.n[0] * a.n[1] * a.n[2]));
        if (a.phi) a.phi[e] = (float)p;
        if (a.phi64) a.phi64[e] = p;
    } else {
        a.out[e] = v;
    }
}
// the factor n1 of n used by dft_axis_kernel: its largest divisor <= sqrt(n)
static int dft_n1(int n)
{
    int best = 1;
    for (int f = 2; f * f <= n; ++f)
        if (n % f == 0) best = f;
    return best;
}

cudaError_t launch_poisson(const GridDims &g, const PoissonScratch &ps, const double *rho, const double *bg,
                           double a, double four_pi_G, float *phi, cudaStream_t st, double *phi64)
{
    const long long n = (long long)g.n[0] * g.n[1] * g.n[2];
    DftArgs A{};
    for (int d = 0; d < 3; ++d) A.n[d] = g.n[d];
    A.rho = rho;
    A.bg = bg;
    A.fac = four_pi_G * a * a;
    A.L = g.L;
    A.phi = phi;
    A.phi64 = phi64;
    cudaError_t err = cudaSuccess;
    // Chained only up to 2^12 spatial cells (and kChainCells in all): of more, the blocks of the next
    // launch sit on the SMs while FP64 sums still run.  Chained / not: steps of 8^3 x 16^3 cells 81 / 92
    // us, 16^3 x 8^3 99 / 108, 16^3 x 16^3 264 / 274, but 31 x 13 x 11 x 8^3 170 / 132, 20^3 x 8^3 172 / 146 (20^3
    // x 12^3 363 / 372); the solve alone 32^3 99 / 65, 31 x 37 x 43 531 / 188.
    const long long cells = n <= 4096 ? n * g.nu[0] * g.nu[1] * g.nu[2] : kChainCells + 1;
    auto dft = [&](auto kernel, int d, int sign, const double2 *in, double2 *out) {
        const int nd = g.n[d]; // <= 256
        A.nlines = unsigned(n / nd);
        // up to 256 threads a block, but blocks for every SM first (of a warp at least)
        const int most = 256 / nd, least = nd >= 32 ? 1 : 32 / nd;
        const int spread = int((A.nlines + 303) / 304);
        A.lines = spread < least ? least : spread > most ? most : spread;
        A.d = d;
        A.sign = sign;
        A.n1 = dft_n1(nd);
        A.in = in;
        A.out = out;
        A.tw = ps.tw[d];
        const cudaError_t e = launch_chained_t(cells, kernel, dim3((A.nlines + A.lines - 1) / A.lines), dim3(A.lines * nd),
                                               (2 * A.lines + 1) * nd * sizeof(double2), st, A);
        if (err == cudaSuccess) err = e;
    };
    dft(dft_axis_kernel<Dft::first>, 2, -1, nullptr, ps.z0);
    dft(dft_axis_kernel<Dft::plain>, 1, -1, ps.z0, ps.z1);
    dft(dft_axis_kernel<Dft::middle>, 0, -1, ps.z1, ps.z0);
    dft(dft_axis_kernel<Dft::plain>, 1, +1, ps.z0, ps.z1);
    dft(dft_axis_kernel<Dft::last>, 2, +1, ps.z1, nullptr);
    return err;
}

} // namespace vk
