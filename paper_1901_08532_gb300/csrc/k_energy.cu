// Energy and angular momentum of the current state (paper, section 3 item 3:
// both are evaluated on the device and checked periodically; Eq. 1 defines
// their relative errors).  FP64 throughout, deterministic: per-block sums in
// a fixed tree order, then one block adds the block sums in a fixed order.
//   E_kin = sum 1/2 m_i |v_i|^2
//   E_pot = -sum_{i<j} m_i m_j / sqrt(|r_ij|^2 + eps^2)
//   L     = sum m_i x_i cross v_i,  and sum m_i |x_i cross v_i|
#include <algorithm>

#include "nb_internal.cuh"

namespace {

constexpr int kT = 256;

template <int NV, int TH>
__device__ void block_sum(double (&v)[NV], double *out)
{
    __shared__ double s[NV][TH / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        double x = v[q];
        for (int off = 16; off > 0; off >>= 1)
            x += __shfl_xor_sync(0xffffffffu, x, off);
        if (lane == 0)
            s[q][warp] = x;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int q = 0; q < NV; ++q) {
            double x = 0.0;
            for (int w = 0; w < TH / 32; ++w)
                x += s[q][w];
            out[q] = x;
        }
    }
}

// 1 / sqrt(x): the refined FP32 estimate, the library functions for infinities
// and NaN (positions beyond 1e154).
__device__ __forceinline__ double inv_sqrt(double x)
{
    if (static_cast<unsigned>(__double2hiint(x)) >= 0x7ff00000u)
        return 1.0 / sqrt(x);
    return nbk::rsqrt_fp64(x);
}

// Every unordered pair once: the particles form T tiles of B, a block takes the
// pairs of tile b with the tiles b + d (mod T) for its k offsets d of
// 0 .. T/2 (for even T the last offset counts from the lower half of the tiles
// only; d = 0 is the tile with itself, in ordered pairs at half weight).  128
// threads: B = 128 gives each an i-particle, B = 32 each warp a quarter of
// the j-tile, for systems that would otherwise leave SMs idle.
// Bound by the FP64 pipe: 10 operations per pair (was sqrt and a division for
// every ordered pair, on n / 256 blocks).  nb_energy, 1000 particles 1603 -> 42 us,
// 8192 12.96 -> 0.66 ms, 131072 827 -> 153 ms.
constexpr int kET = 128;

template <int B>
__global__ void __launch_bounds__(kET) energy_kernel(const double *st, const double *m, int n, double eps2, int T,
                                                     int k, double *blocksums)
{
    constexpr int S = kET / B;  // threads that share an i-particle
    __shared__ double sx[B], sy[B], sz[B], sm[B];
    const size_t N = static_cast<size_t>(n);
    const int b = blockIdx.x, da = blockIdx.y * k, db = min(T / 2 + 1, da + k);
    const int i = b * B + threadIdx.x % B, part = threadIdx.x / B;
    const bool valid = i < n;
    const int ii = valid ? i : n - 1;
    const double *x = st + F_X * 3 * N, *v = st + F_V * 3 * N;
    const double xi = x[ii], yi = x[N + ii], zi = x[2 * N + ii];
    double phi = 0.0;
    for (int d = da; d < db; ++d) {
        if (2 * d == T && b >= T / 2)
            break;
        const int c = b + d < T ? b + d : b + d - T;
        __syncthreads();
        if (threadIdx.x < B) {
            const int j = c * B + threadIdx.x, jj = min(j, n - 1);
            sx[threadIdx.x] = x[jj];
            sy[threadIdx.x] = x[N + jj];
            sz[threadIdx.x] = x[2 * N + jj];
            sm[threadIdx.x] = j < n ? m[j] : 0.0;
        }
        __syncthreads();
        double s = 0.0;
#pragma unroll 4
        for (int q = part * (B / S); q < (part + 1) * (B / S); ++q) {
            const double dx = sx[q] - xi, dy = sy[q] - yi, dz = sz[q] - zi;
            const double r = inv_sqrt(fma(dx, dx, fma(dy, dy, fma(dz, dz, eps2))));
            s = (d == 0 && c * B + q == i) ? s : fma(sm[q], r, s);
        }
        phi += d == 0 ? 0.5 * s : s;
    }
    double w[2] = {0.0, 0.0};
    if (valid) {
        w[1] = -m[i] * phi;
        if (da == 0 && part == 0)
            w[0] = 0.5 * m[i] * fma(v[i], v[i], fma(v[N + i], v[N + i], v[2 * N + i] * v[2 * N + i]));
    }
    block_sum<2, kET>(w, blocksums + 2 * (static_cast<size_t>(blockIdx.y) * gridDim.x + blockIdx.x));
}

__global__ void __launch_bounds__(kT) angmom_kernel(const double *st, const double *m, int n,
                                                    double *blocksums)
{
    const size_t N = static_cast<size_t>(n);
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    double v[4] = {0.0, 0.0, 0.0, 0.0};
    if (i < n) {
        const double x = st[(F_X * 3 + 0) * N + i], y = st[(F_X * 3 + 1) * N + i],
                     z = st[(F_X * 3 + 2) * N + i];
        const double vx = st[(F_V * 3 + 0) * N + i], vy = st[(F_V * 3 + 1) * N + i],
                     vz = st[(F_V * 3 + 2) * N + i];
        const double lx = y * vz - z * vy, ly = z * vx - x * vz, lz = x * vy - y * vx;
        v[0] = m[i] * lx;
        v[1] = m[i] * ly;
        v[2] = m[i] * lz;
        v[3] = m[i] * sqrt(lx * lx + ly * ly + lz * lz);
    }
    block_sum<4, kT>(v, blocksums + 4 * blockIdx.x);
}

// Sum nv interleaved block sums in a fixed order (one block).
template <int NV>
__global__ void __launch_bounds__(kT) final_sum_kernel(const double *blocksums, int nblocks, double *out)
{
    double v[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q)
        v[q] = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += kT)
#pragma unroll
        for (int q = 0; q < NV; ++q)
            v[q] += blocksums[static_cast<size_t>(b) * NV + q];
    block_sum<NV, kT>(v, out);
}

cudaError_t ensure_red(nb_ctx *c, size_t doubles)
{
    if (doubles <= c->red_cap)
        return cudaSuccess;
    cudaFree(c->red);
    c->red = nullptr;
    c->red_cap = 0;
    cudaError_t e = cudaMalloc(&c->red, doubles * sizeof(double));
    if (e == cudaSuccess)
        c->red_cap = doubles;
    return e;
}

}  // namespace

// out_dev[0] = E_kin, out_dev[1] = E_pot (device memory, 2 doubles).
cudaError_t nb_launch_energy(nb_ctx *c, double *out_dev)
{
    const int n = static_cast<int>(c->n);
    // 32-particle tiles below 6144 particles (1024: 528 blocks instead of 36)
    const int B = n < 6144 ? 32 : kET;
    const int T = (n + B - 1) / B, D = T / 2 + 1;
    // offsets per block: about 16384 blocks at most
    const int groups = std::max(1, std::min(D, 16384 / T)), k = (D + groups - 1) / groups;
    const dim3 grid(T, (D + k - 1) / k);
    const int nb = static_cast<int>(grid.x * grid.y);
    cudaError_t e = ensure_red(c, static_cast<size_t>(2) * nb);
    if (e != cudaSuccess)
        return e;
    const double eps2 = c->eps * c->eps;
    if (B == 32) energy_kernel<32><<<grid, kET, 0, c->stream>>>(c->st, c->m, n, eps2, T, k, c->red);
    else energy_kernel<kET><<<grid, kET, 0, c->stream>>>(c->st, c->m, n, eps2, T, k, c->red);
    final_sum_kernel<2><<<1, kT, 0, c->stream>>>(c->red, nb, out_dev);
    c->launches += 2;
    return cudaGetLastError();
}

// out_dev[0..2] = L, out_dev[3] = sum m |x cross v|.
cudaError_t nb_launch_angmom(nb_ctx *c, double *out_dev)
{
    const int n = static_cast<int>(c->n);
    const int nb = (n + kT - 1) / kT;
    cudaError_t e = ensure_red(c, static_cast<size_t>(4) * nb);
    if (e != cudaSuccess)
        return e;
    angmom_kernel<<<nb, kT, 0, c->stream>>>(c->st, c->m, n, c->red);
    final_sum_kernel<4><<<1, kT, 0, c->stream>>>(c->red, nb, out_dev);
    c->launches += 2;
    return cudaGetLastError();
}
