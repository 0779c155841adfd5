// Evaluation of a complete active set (paper, section 3 item 4): every
// particle is active, so each unordered pair {i, j} is needed in both
// directions, and both come from one set of differences, powers of R, alpha
// and beta.  Swapping i and j negates r, v and a, keeps alpha and beta, and
// so negates u and w: the terms on j are (-m_i / m_j) times those on i.  Per
// unordered pair the mixed formula takes 63 FP32-pipe operations instead of
// 2 x 53 (FP64 60 instead of 100, EX 608 instead of 992; one product more with
// masses above 1).
//
// Work split.  The particles form T tiles of B; a job (b, d) is the pairs of
// tile b with tile (b + d) mod T, and d = 0 .. T/2 covers every unordered pair
// of tiles once (for even T the last offset is taken by the lower half of the
// tiles).  d = 0 is the tile with itself, evaluated in ordered pairs.  A block
// runs the jobs of one tile b and a few consecutive offsets, or the part h of H
// of a job's j-tile where there are few jobs.
//   * Each lane keeps its i-particles and their sums in registers and works
//     through 32 j-particles at a time, one per lane: at step s lane l pairs
//     its i-particles with j = (l + s) mod 32 and adds the terms on j to the
//     running sums of that j, which move on to the next lane (shuffle) with
//     every step, so that after 32 steps they are back in the lane of their j.
//     Every lane reads a j-record of its own, without bank conflicts.
//   * The warps of a block work on different 32-particle parts of the j-tile
//     at a time (a barrier between parts), so they add their j-sums into one
//     shared-memory array without conflicts, in a fixed order.
//   * i-sums and j-sums of each job go to partial-sum slots of their own, one
//     per offset (j) or group of offsets (i), and fold_kernel adds the slots
//     in a fixed order: no atomics, the result does not depend on scheduling.
//     The offsets are evaluated in batches that bound the slots' memory.
#include <algorithm>

#include "nb_device.cuh"
#include "nb_ff.cuh"
#include "nb_internal.cuh"
#include "nb_sym.cuh"

namespace {

using namespace nbk;

// cp.async of 4, 8 or 16 bytes; bytes = 0 writes zeros.
__device__ __forceinline__ void cp_async4(void *dst, const void *src, uint32_t bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async8(void *dst, const void *src, uint32_t bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// ----------------------------------------------------------------- mixed

constexpr int kMixedWarps = 4;
constexpr int kMixedThreads = 32 * kMixedWarps;
__host__ __device__ constexpr int mixed_tile(int kp) { return kMixedThreads * 2 * kp; }

// mu = m_j q^3 and nu = -m_i q^3.  q^3 by itself leaves the FP32 range from
// separations of 2^42 on (and the low word of a double word from 2^26 on); where
// no mass is above 1 (LIGHT), m q^3 is no larger than it and leaves the range with it or
// before, so it may be formed once for both.  Larger masses, such as G m in metres
// or centimetres, come in before the second power of q, as in the ordinary
// kernels: one product more, 3.6 % (mixed) and 1.6 % (EX) of the time (524288
// particles mixed 296 / 307 ms, 16384 EX 2.54 / 2.58 ms).
template <bool LIGHT>
__device__ __forceinline__ void mass_factors(float2 q, float2 q2, float2 mj, float2 nmi, float2 &mu, float2 &nu)
{
    if constexpr (LIGHT) {
        const float2 q3 = mul2(q, q2);
        mu = mul2(mj, q3);
        nu = mul2(nmi, q3);
    } else {
        mu = mul2(mul2(mj, q), q2);
        nu = mul2(mul2(nmi, q), q2);
    }
}
template <bool LIGHT>
__device__ __forceinline__ void mass_factors(const ff::FF<float2> &q, const ff::FF<float2> &q2,
                                             const ff::FF<float2> &mj, const ff::FF<float2> &nmi,
                                             ff::FF<float2> &mu, ff::FF<float2> &nu)
{
    if constexpr (LIGHT) {
        const ff::FF<float2> q3 = ff::mul(q, q2);
        mu = ff::mul(mj, q3);
        nu = ff::mul(nmi, q3);
    } else {
        mu = ff::mul(ff::mul(mj, q), q2);
        nu = ff::mul(ff::mul(nmi, q), q2);
    }
}

// Both directions of the pairs of two i-particles (the lanes of the packed
// values) with one j: pi += terms on i, pj += terms on j.  ni are the negated
// i-values, nmi the negated masses, c the 13 j-values.
template <bool LIGHT>
__device__ __forceinline__ void pair_mixed_sym(const float (&c)[NCF], const float2 (&ni)[12], float2 nmi,
                                               float2 eps2, float2 (&pi)[9], float2 (&pj)[9])
{
    const float2 dx = add2(add2(f2(c[0]), ni[0]), add2(f2(c[4]), ni[3]));
    const float2 dy = add2(add2(f2(c[1]), ni[1]), add2(f2(c[5]), ni[4]));
    const float2 dz = add2(add2(f2(c[2]), ni[2]), add2(f2(c[6]), ni[5]));
    const float2 dvx = add2(f2(c[7]), ni[6]), dvy = add2(f2(c[8]), ni[7]), dvz = add2(f2(c[9]), ni[8]);
    const float2 dax = add2(f2(c[10]), ni[9]), day = add2(f2(c[11]), ni[10]), daz = add2(f2(c[12]), ni[11]);
    const float2 r2 = fma2(dx, dx, fma2(dy, dy, fma2(dz, dz, eps2)));
    const float2 rv = fma2(dx, dvx, fma2(dy, dvy, mul2(dz, dvz)));
    const float2 sv = fma2(dx, dax, fma2(dy, day, fma2(dz, daz, fma2(dvx, dvx, fma2(dvy, dvy, mul2(dvz, dvz))))));
    const float2 q = make_float2(rsqrt_est(r2.x), rsqrt_est(r2.y));
    const float2 q2 = make_float2(rcp_est(r2.x), rcp_est(r2.y));
    float2 mu, nu;
    mass_factors<LIGHT>(q, q2, f2(c[3]), nmi, mu, nu);
    const float2 al = mul2(rv, q2);
    const float2 be = fma2(al, al, mul2(sv, q2));
    const float2 na3 = mul2(al, f2(-3.0f)), na6 = mul2(al, f2(-6.0f)), nb3 = mul2(be, f2(-3.0f));
    const float2 ux = fma2(na3, dx, dvx), uy = fma2(na3, dy, dvy), uz = fma2(na3, dz, dvz);
    const float2 wx = fma2(na6, ux, fma2(nb3, dx, dax));
    const float2 wy = fma2(na6, uy, fma2(nb3, dy, day));
    const float2 wz = fma2(na6, uz, fma2(nb3, dz, daz));
    const float2 t[9] = {dx, dy, dz, ux, uy, uz, wx, wy, wz};
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        pi[k] = fma2(mu, t[k], pi[k]);
        pj[k] = fma2(nu, t[k], pj[k]);
    }
}

__device__ __forceinline__ void load_tile_mixed(const SymArgs &a, float *dst, int j0)
{
    const float *jf = static_cast<const float *>(a.jb);
    const int j = j0 + threadIdx.x;
    const int jc = min(j, a.n - 1);  // beyond the end: the last particle without its mass
#pragma unroll
    for (int r = 0; r < NCF; ++r)
        cp_async4(dst + r * kMixedThreads + threadIdx.x, jf + r * a.np + jc, r == 3 && j >= a.n ? 0u : 4u);
    cp_async_commit();
}

// KP packed pairs of i-particles per thread.  Like the ordinary mixed kernel it
// is bound by the register file's operand bandwidth (about 160 64-bit operand
// reads for the 63 packed operations, so at most 79 % of the FMA pipe; 75 %
// reached).  KP = 3 (255 registers, no spills) spreads the 13 loads and 18
// shuffles of a step over three packed pairs: KP = 2 runs 6 % below it with two
// blocks per SM and 3 % below with three, eight warps a block 1 % above at
// twice the tile.  Loading the next step's j ahead (-3 %), and adding the
// halves of pj before the shuffles (no change) did not help.  FP32 sums run
// over 64 terms on the i-side and 16 KP in each half on the j-side before they
// go to the compensated sums (64 in each half in the ordinary kernel): over
// 128 and 32 KP terms the kernel was 1.8 % faster and its error 8-17 %
// larger; now the RMS error in units of sum_j |T_ij| is 0.97-1.0 of the
// ordinary kernel's at 16384 to 65536 particles.
//
// All particles, prediction not included, ordinary kernel -> this one:
// 4096 51 -> 39 us, 8192 150 -> 111, 20011 744 -> 500, 65536 7.26 -> 5.05 ms,
// 131072 28.6 -> 19.2 ms, 2^20 1.813 -> 1.178 s.  Below about 3500 particles the
// ordinary kernels are faster (3000: 34 us against 39).
template <int KP, bool LIGHT>
__global__ void __launch_bounds__(kMixedThreads, 2) sym_mixed_kernel(SymArgs a)
{
    constexpr int W = kMixedWarps, TH = kMixedThreads, B = mixed_tile(KP);
    extern __shared__ __align__(16) float sm[];
    float *tile = sm;                        // [2][NCF][TH]
    float *jacc = sm + 2 * NCF * TH;         // [18][TH]: hi of the 9 sums, then lo
    float *iacc = jacc + 18 * TH;            // [2 KP][18][TH]
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const SymJob<B, TH> job(a);
    const float *jf = static_cast<const float *>(a.jb);
    const float2 eps2 = f2(static_cast<float>(a.eps2));
    constexpr int kRow[12] = {0, 1, 2, 4, 5, 6, 7, 8, 9, 10, 11, 12};

    float2 ni[KP][12], nmi[KP], pi[KP][9];
#pragma unroll
    for (int p = 0; p < KP; ++p) {
        const int i = job.b * B + (w * KP + p) * 64 + 2 * lane;
        const int i0 = min(i, a.n - 1), i1 = min(i + 1, a.n - 1);
#pragma unroll
        for (int q = 0; q < 12; ++q)
            ni[p][q] = make_float2(-jf[kRow[q] * a.np + i0], -jf[kRow[q] * a.np + i1]);
        nmi[p] = make_float2(i < a.n ? -jf[3 * a.np + i0] : 0.0f, i + 1 < a.n ? -jf[3 * a.np + i1] : 0.0f);
#pragma unroll
        for (int q = 0; q < 9; ++q)
            pi[p][q] = f2(0.0f);
    }
    for (int q = 0; q < 36 * KP; ++q)
        iacc[q * TH + tid] = 0.0f;
    for (int q = 0; q < 18; ++q)
        jacc[q * TH + tid] = 0.0f;

    if (job.nit > 0)
        load_tile_mixed(a, tile, job.start(a, 0));
    for (int it = 0; it < job.nit; ++it) {
        cp_async_wait_all();
        __syncthreads();
        if (it + 1 < job.nit)
            load_tile_mixed(a, tile + ((it + 1) & 1) * NCF * TH, job.start(a, it + 1));
        const float *s = tile + (it & 1) * NCF * TH;
        for (int st = 0; st < W; ++st) {
            const int sub = ((st + w) & (W - 1)) * 32;
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                float2 pj[9];
#pragma unroll
                for (int q = 0; q < 9; ++q)
                    pj[q] = f2(0.0f);
#pragma unroll 2
                for (int step = 16 * half; step < 16 * half + 16; ++step) {
                    const float *sj = s + sub + ((lane + step) & 31);
                    float c[NCF];
#pragma unroll
                    for (int r = 0; r < NCF; ++r)
                        c[r] = sj[r * TH];
#pragma unroll
                    for (int p = 0; p < KP; ++p)
                        pair_mixed_sym<LIGHT>(c, ni[p], nmi[p], eps2, pi[p], pj);
#pragma unroll
                    for (int q = 0; q < 9; ++q) {
                        pj[q].x = __shfl_sync(0xffffffffu, pj[q].x, lane + 1);
                        pj[q].y = __shfl_sync(0xffffffffu, pj[q].y, lane + 1);
                    }
                }
                // the sums of 16 KP terms in each half, into the compensated
                // ones of the j they belong to
                const int jl = sub + ((lane + 16 * (half + 1)) & 31);
#pragma unroll
                for (int q = 0; q < 9; ++q) {
                    float hi = jacc[q * TH + jl], lo = jacc[(9 + q) * TH + jl];
                    two_sum_acc(hi, lo, __fadd_rn(pj[q].x, pj[q].y));
                    jacc[q * TH + jl] = hi;
                    jacc[(9 + q) * TH + jl] = lo;
                }
                __syncwarp();
            }
            // the i-sums of 64 terms
            if (st & 1)
#pragma unroll
                for (int p = 0; p < KP; ++p)
#pragma unroll
                    for (int q = 0; q < 9; ++q) {
                        float *ia = iacc + (p * 36 + q) * TH + tid;
                        float hi = ia[0], lo = ia[9 * TH];
                        two_sum_acc(hi, lo, pi[p][q].x);
                        ia[0] = hi;
                        ia[9 * TH] = lo;
                        hi = ia[18 * TH], lo = ia[27 * TH];
                        two_sum_acc(hi, lo, pi[p][q].y);
                        ia[18 * TH] = hi;
                        ia[27 * TH] = lo;
                        pi[p][q] = f2(0.0f);
                    }
            __syncthreads();
        }
        float2 *out = static_cast<float2 *>(a.pj) + job.jslot(a, it) + tid;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            if (job.offset(it) > 0)
                out[q * a.ns] = make_float2(jacc[q * TH + tid], jacc[(9 + q) * TH + tid]);
            jacc[q * TH + tid] = 0.0f;
            jacc[(9 + q) * TH + tid] = 0.0f;
        }
    }
    float2 *out = static_cast<float2 *>(a.pi) + job.islot(a);
#pragma unroll
    for (int p = 0; p < KP; ++p) {
        const int i = job.b * B + (w * KP + p) * 64 + 2 * lane;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const float *ia = iacc + (p * 36 + q) * TH + tid;
            *reinterpret_cast<float4 *>(&out[q * a.ns + i]) =
                make_float4(ia[0], ia[9 * TH], ia[18 * TH], ia[27 * TH]);
        }
    }
}

// -------------------------------------------------------------------- EX

// Warps per block (W) sets the tile: 64 W particles, two per thread in the
// lanes of the packed values.
__host__ __device__ constexpr int ex_tile(int w) { return 64 * w; }

// Both directions of the pairs of two i-particles with one j in double words
// (pair_ex with the powers of q shared): ni the negated i-values, nmi the
// negated masses.
template <bool LIGHT>
__device__ __forceinline__ void pair_ex_sym(const float2 (&c)[NCX], const ExI<float2> &ni,
                                            const ff::FF<float2> &nmi, const ff::FF<float2> &eps2,
                                            ff::FF<float2> (&pi)[9], ff::FF<float2> (&pj)[9])
{
    using F = ff::FF<float2>;
    F r[3], dv[3], da[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        r[k] = ff::add_accurate(F{c[k], c[3 + k]}, ni.x[k]);  // close pairs cancel
        dv[k] = ff::add(F{c[6 + k], c[9 + k]}, ni.v[k]);
        da[k] = ff::add(F{c[12 + k], c[15 + k]}, ni.a[k]);
    }
    const F R = ff::mad(r[0], r[0], ff::mad(r[1], r[1], ff::mad(r[2], r[2], eps2)));
    const F rv = ff::mad(r[0], dv[0], ff::mad(r[1], dv[1], ff::mul(r[2], dv[2])));
    const F sv = ff::mad(r[0], da[0], ff::mad(r[1], da[1], ff::mad(r[2], da[2],
                 ff::mad(dv[0], dv[0], ff::mad(dv[1], dv[1], ff::sqr(dv[2]))))));
    const F q = ff::rsqrt(R, rsqrt_est_v(R.h));
    const F q2 = ff::sqr(q);
    F mu, nu;
    mass_factors<LIGHT>(q, q2, F{c[18], c[19]}, nmi, mu, nu);
    const F al = ff::mul(rv, q2);
    const F be = ff::mad(al, al, ff::mul(sv, q2));
    const float2 m3 = f2(-3.0f), two = f2(2.0f);
    const F na3 = ff::mul(al, m3);
    const F na6 = {ff::mul(na3.h, two), ff::mul(na3.l, two)};  // exact doubling
    const F nb3 = ff::mul(be, m3);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const F u = ff::mad(na3, r[k], dv[k]);
        const F w = ff::mad(na6, u, ff::mad(nb3, r[k], da[k]));
        ff::accumulate_mul(pi[k], mu, r[k]);
        ff::accumulate_mul(pj[k], nu, r[k]);
        ff::accumulate_mul(pi[3 + k], mu, u);
        ff::accumulate_mul(pj[3 + k], nu, u);
        ff::accumulate_mul(pi[6 + k], mu, w);
        ff::accumulate_mul(pj[6 + k], nu, w);
    }
}

// Bound by the FP32 pipe like the ordinary EX kernel; eight warps of 238
// registers fill an SM, and the tile shrinks with W for small systems.
// Double-word sums run over at most 64 terms in each half of a packed value and
// go to FP64 after at most 512, as in the ordinary kernel; its RMS error is 0.95-1.0
// of that kernel's.
// All particles, ordinary kernel -> this one: 2000 81 -> 72 us, 4096 268 -> 207,
// 16384 3.84 -> 2.55 ms, 40000 23.7 -> 14.7 ms (1.08e11 interactions/s).  Below
// about 1800 particles the ordinary kernel is faster.
template <int W, bool LIGHT>
__global__ void __launch_bounds__(32 * W, 8 / W) sym_ex_kernel(SymArgs a)
{
    using F = ff::FF<float2>;
    constexpr int TH = 32 * W, B = ex_tile(W);
    extern __shared__ __align__(16) float sm[];
    float *tile = sm;                 // [2][NCX][TH]
    float *jacc = sm + 2 * NCX * TH;  // [18][TH]: high parts of the 9 sums, then low parts
    float *iacc = jacc + 18 * TH;     // [2][18][TH]
    double *itot = reinterpret_cast<double *>(iacc + 36 * TH);  // [2][9][TH]
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const SymJob<B, TH> job(a);
    const float *jf = static_cast<const float *>(a.jb);
    const float e2h = __double2float_rn(a.eps2);
    const F eps2 = {f2(e2h), f2(__double2float_rn(a.eps2 - static_cast<double>(e2h)))};

    const int i = job.b * B + w * 64 + 2 * lane;
    const int i0 = min(i, a.n - 1), i1 = min(i + 1, a.n - 1);
    auto neg = [&](int row) { return make_float2(-jf[row * a.np + i0], -jf[row * a.np + i1]); };
    ExI<float2> ni;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        ni.x[k] = {neg(k), neg(3 + k)};
        ni.v[k] = {neg(6 + k), neg(9 + k)};
        ni.a[k] = {neg(12 + k), neg(15 + k)};
    }
    F nmi = {neg(18), neg(19)};
    if (i >= a.n) nmi.h.x = nmi.l.x = 0.0f;
    if (i + 1 >= a.n) nmi.h.y = nmi.l.y = 0.0f;
    F pi[9];
#pragma unroll
    for (int q = 0; q < 9; ++q)
        pi[q] = {f2(0.0f), f2(0.0f)};
    for (int q = 0; q < 36; ++q)
        iacc[q * TH + tid] = 0.0f;
    for (int q = 0; q < 18; ++q) {
        jacc[q * TH + tid] = 0.0f;
        itot[q * TH + tid] = 0.0;
    }

    auto load = [&](int it) {
        float *dst = tile + (it & 1) * NCX * TH;
        const int j = job.start(a, it) + tid, jc = min(j, a.n - 1);  // beyond the end: no mass
#pragma unroll
        for (int r = 0; r < NCX; ++r)
            cp_async4(dst + r * TH + tid, jf + r * a.np + jc, r >= 18 && j >= a.n ? 0u : 4u);
        cp_async_commit();
    };
    // acc (h, l in shared memory, ld floats apart) += t
    auto into = [](float *h, int ld, float th, float tl) {
        ff::FF<float> s = {h[0], h[ld]};
        ff::accumulate(s, ff::FF<float>{th, tl});
        h[0] = s.h;
        h[ld] = s.l;
    };
    auto wide = [](const float *h, int ld) { return to_double(h[0]) + to_double(h[ld]); };
    if (job.nit > 0)
        load(0);
    for (int it = 0; it < job.nit; ++it) {
        cp_async_wait_all();
        __syncthreads();
        if (it + 1 < job.nit)
            load(it + 1);
        const float *s = tile + (it & 1) * NCX * TH;
        for (int st = 0; st < W; ++st) {
            const int sub = ((st + w) & (W - 1)) * 32;
            F pj[9];
#pragma unroll
            for (int q = 0; q < 9; ++q)
                pj[q] = {f2(0.0f), f2(0.0f)};
#pragma unroll 1
            for (int step = 0; step < 32; ++step) {
                const float *sj = s + sub + ((lane + step) & 31);
                float2 c[NCX];
#pragma unroll
                for (int r = 0; r < NCX; ++r)
                    c[r] = f2(sj[r * TH]);
                pair_ex_sym<LIGHT>(c, ni, nmi, eps2, pi, pj);
#pragma unroll
                for (int q = 0; q < 9; ++q) {
                    pj[q].h.x = __shfl_sync(0xffffffffu, pj[q].h.x, lane + 1);
                    pj[q].h.y = __shfl_sync(0xffffffffu, pj[q].h.y, lane + 1);
                    pj[q].l.x = __shfl_sync(0xffffffffu, pj[q].l.x, lane + 1);
                    pj[q].l.y = __shfl_sync(0xffffffffu, pj[q].l.y, lane + 1);
                }
            }
            // double-word sums of 32 terms on each half of the j-side ...
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                into(jacc + q * TH + sub + lane, 9 * TH, pj[q].h.x, pj[q].l.x);
                into(jacc + q * TH + sub + lane, 9 * TH, pj[q].h.y, pj[q].l.y);
            }
            // ... and of 64 on the i-side (32 in a one-warp block)
            if (W == 1 || (st & 1))
#pragma unroll
                for (int q = 0; q < 9; ++q) {
                    into(iacc + q * TH + tid, 9 * TH, pi[q].h.x, pi[q].l.x);
                    into(iacc + (18 + q) * TH + tid, 9 * TH, pi[q].h.y, pi[q].l.y);
                    pi[q] = {f2(0.0f), f2(0.0f)};
                }
            __syncthreads();
        }
        double *out = static_cast<double *>(a.pj) + job.jslot(a, it) + tid;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            if (job.offset(it) > 0)
                out[q * a.ns] = wide(jacc + q * TH + tid, 9 * TH);
            jacc[q * TH + tid] = 0.0f;
            jacc[(9 + q) * TH + tid] = 0.0f;
        }
        // i-sums over at most 512 j in double words, like the ordinary kernel's
        // tiles, then FP64
        if ((it + 1) % (512 / TH) == 0 || it + 1 == job.nit)
            for (int q = 0; q < 9; ++q)
#pragma unroll
                for (int p = 0; p < 2; ++p) {
                    float *ia = iacc + (18 * p + q) * TH + tid;
                    itot[(9 * p + q) * TH + tid] += wide(ia, 9 * TH);
                    ia[0] = ia[9 * TH] = 0.0f;
                }
    }
    double *out = static_cast<double *>(a.pi) + job.islot(a);
#pragma unroll
    for (int q = 0; q < 9; ++q)
        *reinterpret_cast<double2 *>(&out[q * a.ns + i]) = make_double2(itot[q * TH + tid], itot[(9 + q) * TH + tid]);
}

// ------------------------------------------------------------------ FP64

// One i-particle per thread; the j-tile is 5 rows of 16-byte records.
__device__ __forceinline__ void pair_fp64_sym(const double2 (&c)[5], const double (&xi)[9], double nmi, double eps2,
                                              double (&pi)[9], double (&pj)[9])
{
    const double dx = c[0].x - xi[0], dy = c[0].y - xi[1], dz = c[1].x - xi[2];
    const double dvx = c[2].x - xi[3], dvy = c[2].y - xi[4], dvz = c[3].x - xi[5];
    const double dax = c[3].y - xi[6], day = c[4].x - xi[7], daz = c[4].y - xi[8];
    const double r2 = fma(dx, dx, fma(dy, dy, fma(dz, dz, eps2)));
    const double rv = fma(dx, dvx, fma(dy, dvy, dz * dvz));
    const double sv = fma(dx, dax, fma(dy, day, fma(dz, daz, fma(dvx, dvx, fma(dvy, dvy, dvz * dvz)))));
    const double q = nbk::rsqrt_fp64(r2);
    const double q2 = q * q, q3 = q * q2;
    const double mu = c[1].y * q3, nu = nmi * q3;
    const double al = rv * q2;
    const double be = fma(al, al, sv * q2);
    const double a3 = 3.0 * al, a6 = twice(a3), b3 = 3.0 * be;
    const double ux = fma(-a3, dx, dvx), uy = fma(-a3, dy, dvy), uz = fma(-a3, dz, dvz);
    const double wx = fma(-a6, ux, fma(-b3, dx, dax));
    const double wy = fma(-a6, uy, fma(-b3, dy, day));
    const double wz = fma(-a6, uz, fma(-b3, dz, daz));
    const double t[9] = {dx, dy, dz, ux, uy, uz, wx, wy, wz};
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        pi[k] = fma(mu, t[k], pi[k]);
        pj[k] = fma(nu, t[k], pj[k]);
    }
}

// Bound by the FP64 pipe (93 % of 2 operations per clock and SM): 60 operations
// per unordered pair for 100, so loads and shuffles cost nothing.  One warp per
// scheduler fills the pipe; W = 1 and 2 give small systems enough blocks.
// All particles, ordinary kernel -> this one: 1000 112 -> 94 us, 2000
// 394 -> 266, 4096 1.54 -> 0.95 ms, 8191 6.10 -> 3.73, 30000 82.9 -> 48.4 ms (1.86e10
// interactions/s).  Below about 900 particles the ordinary kernel is
// faster.
template <int W>
__global__ void __launch_bounds__(32 * W) sym_fp64_kernel(SymArgs a)
{
    constexpr int TH = 32 * W;
    __shared__ __align__(16) double2 tile[2][5][TH];
    __shared__ double jacc[9][TH];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const SymJob<TH, TH> job(a);
    const double2 *jb = static_cast<const double2 *>(a.jb);
    const int i = job.b * TH + tid;
    double xi[9], nmi, acc[9], pi[9];
    {
        const int ic = min(i, a.n - 1);
        const double2 r0 = jb[ic], r1 = jb[a.np + ic], r2 = jb[2 * a.np + ic], r3 = jb[3 * a.np + ic],
                      r4 = jb[4 * a.np + ic];
        xi[0] = r0.x; xi[1] = r0.y; xi[2] = r1.x;
        xi[3] = r2.x; xi[4] = r2.y; xi[5] = r3.x;
        xi[6] = r3.y; xi[7] = r4.x; xi[8] = r4.y;
        nmi = i < a.n ? -r1.y : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        acc[q] = pi[q] = 0.0;
        jacc[q][tid] = 0.0;
    }
    auto load = [&](int it) {
        double2 (&dst)[5][TH] = tile[it & 1];
        const int j = job.start(a, it) + tid, jc = min(j, a.n - 1);
#pragma unroll
        for (int r = 0; r < 5; ++r)
            if (r != 1)
                cp_async16(&dst[r][tid], jb + r * a.np + jc);
        const double2 *zm = jb + a.np + jc;  // beyond the end: the last particle without its mass
        cp_async8(&dst[1][tid].x, &zm->x, 8u);
        cp_async8(&dst[1][tid].y, &zm->y, j >= a.n ? 0u : 8u);
        cp_async_commit();
    };
    if (job.nit > 0)
        load(0);
    for (int it = 0; it < job.nit; ++it) {
        cp_async_wait_all();
        __syncthreads();
        if (it + 1 < job.nit)
            load(it + 1);
        const double2 (&s)[5][TH] = tile[it & 1];
        for (int st = 0; st < W; ++st) {
            const int sub = ((st + w) & (W - 1)) * 32;
            double pj[9];
#pragma unroll
            for (int q = 0; q < 9; ++q)
                pj[q] = 0.0;
#pragma unroll 1
            for (int step = 0; step < 32; ++step) {
                const int e = sub + ((lane + step) & 31);
                const double2 c[5] = {s[0][e], s[1][e], s[2][e], s[3][e], s[4][e]};
                pair_fp64_sym(c, xi, nmi, a.eps2, pi, pj);
#pragma unroll
                for (int q = 0; q < 9; ++q)
                    pj[q] = __shfl_sync(0xffffffffu, pj[q], lane + 1);
            }
#pragma unroll
            for (int q = 0; q < 9; ++q)
                jacc[q][sub + lane] += pj[q];
            __syncthreads();
        }
        // two-level summation: the j-tile's sums, then the running totals
        double *out = static_cast<double *>(a.pj) + job.jslot(a, it) + tid;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            acc[q] += pi[q];
            pi[q] = 0.0;
            if (job.offset(it) > 0)
                out[q * a.ns] = jacc[q][tid];
            jacc[q][tid] = 0.0;
        }
    }
    double *out = static_cast<double *>(a.pi) + job.islot(a) + i;
#pragma unroll
    for (int q = 0; q < 9; ++q)
        out[q * a.ns] = acc[q];
}

// ------------------------------------------------------------------- fold

// One value of the partial sums and the running total over slots: mixed sums
// stay compensated FP32 pairs within a batch (as inside the kernels).
struct FoldFF {
    using Part = float2;
    float h = 0.0f, l = 0.0f;
    __device__ __forceinline__ void add(float2 v)
    {
        two_sum_acc(h, l, v.x);
        l = __fadd_rn(l, v.y);
    }
    __device__ __forceinline__ double total() const { return static_cast<double>(h) + static_cast<double>(l); }
};

// EX: FP64 sums.
struct FoldEx {
    using Part = double;
    double s = 0.0;
    __device__ __forceinline__ void add(double v) { s += v; }
    __device__ __forceinline__ double total() const { return s; }
};
// out[q][p] (+)= the slots of a batch of offsets.
template <class F>
__global__ void __launch_bounds__(256) fold_kernel(const typename F::Part *pi, int nslots, int upper,
                                                   const typename F::Part *pj, int d0, int d1, size_t ns,
                                                   int T, int B, int n, double *out, size_t ostride, int first)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n)
        return;
    const double s = fold_slots<F, 9>(pi, nslots, upper, pj, d0, d1, ns, T, B, blockIdx.y, p);
    double *o = out + blockIdx.y * ostride + p;
    *o = first ? s : *o + s;
}

constexpr size_t mixed_smem(int kp) { return sizeof(float) * kMixedThreads * (2 * NCF + 18 + 36 * kp); }
constexpr size_t ex_smem(int w) { return sizeof(float) * 32 * w * (2 * NCX + 18 + 36 + 36); }

struct SymKind {
    void (*light)(SymArgs), (*heavy)(SymArgs);  // no mass above 1; any masses
    size_t smem;
    SymShape shape;
};

const SymKind kKinds[] = {
    {sym_mixed_kernel<3, true>, sym_mixed_kernel<3, false>, mixed_smem(3), {mixed_tile(3), kMixedThreads, 72, 3170.0, 1.12}},
    {sym_mixed_kernel<2, true>, sym_mixed_kernel<2, false>, mixed_smem(2), {mixed_tile(2), kMixedThreads, 72, 2750.0, 1.12}},
    {sym_mixed_kernel<1, true>, sym_mixed_kernel<1, false>, mixed_smem(1), {mixed_tile(1), kMixedThreads, 72, 2200.0, 1.12}},
    {sym_ex_kernel<4, true>, sym_ex_kernel<4, false>, ex_smem(4), {ex_tile(4), 128, 72, 360.0, 1.3}},
    {sym_ex_kernel<2, true>, sym_ex_kernel<2, false>, ex_smem(2), {ex_tile(2), 64, 72, 355.0, 2.6}},
    {sym_ex_kernel<1, true>, sym_ex_kernel<1, false>, ex_smem(1), {ex_tile(1), 32, 72, 345.0, 5.2}},
    {sym_fp64_kernel<4>, sym_fp64_kernel<4>, 0, {128, 128, 72, 60.0, 1.05}},
    {sym_fp64_kernel<2>, sym_fp64_kernel<2>, 0, {64, 64, 72, 59.5, 2.1}},
    {sym_fp64_kernel<1>, sym_fp64_kernel<1>, 0, {32, 32, 72, 58.5, 4.2}},
};

// Kinds of a precision: [first, first + 3).
int first_kind(int precision) { return nb_fp32_eval(precision) ? 0 : precision == NB_EX ? 3 : 6; }

}  // namespace

// The estimate behind a plan: the SM with the most jobs works through them at
// the kernel's full rate (with fewer than `fill` jobs as long as with that
// many), plus a fixed part per job and launch and the traffic of the slots.
// Mixed: within 5 % of the measured times of the plans it chooses from 4096 to
// 524288 particles; the next best plans lie within 2 % there.
void nb_sym_plan_shape(const SymShape &kd, int kind, int64_t n, int sms, SymPlan &best,
                       size_t max_bytes)
{
    const int64_t T = (n + kd.tile - 1) / kd.tile, D = T / 2 + 1;
    const double slot = static_cast<double>(kd.bytes) * static_cast<double>(T * kd.tile);
    const double budget = std::min(kSymSlotBytes, std::max(kSymMinBytes, kSymSlots * slot));
    const int64_t slots = max_bytes ? static_cast<int64_t>(static_cast<double>(max_bytes) / slot)
                                    : std::max<int64_t>(2, static_cast<int64_t>(budget / slot));
    const int subs = kd.tile / kd.threads;
    for (const int k : {1, 2, 4, 8})
        for (int parts = 1; parts <= subs; ++parts) {
            if (subs % parts || (k > 1 && parts > 1) || k > D || 1 + parts > slots)
                continue;
            // nd offsets a launch: nd j-slots, ceil(nd / k) parts i-slots
            int64_t nd = std::min<int64_t>(D, std::max<int64_t>(1, slots * k / (k + parts)));
            while (nd > 1 && nd + (nd + k - 1) / k * parts > slots)
                --nd;
            const int64_t batches = (D + nd - 1) / nd;
            nd = (D + batches - 1) / batches;
            const int64_t groups = (nd + k - 1) / k;
            const int64_t jobs = (T * nd - (T % 2 == 0 && batches == 1 ? T / 2 : 0)) * parts / k;
            const double each = static_cast<double>((jobs + sms - 1) / sms) + (k > 1 ? 0.5 : 0.05);
            const double pairs = static_cast<double>(kd.tile) * kd.tile * std::min<int64_t>(k, nd) / parts;
            const double us = batches * (std::max(each, kd.fill) * (pairs / kd.rate + 1.0) + 5.0 +
                                         (nd + groups * parts) * slot * 2.0 / 6e6);
            if (us < best.us) {
                best.us = us;
                best.kind = kind;
                best.T = static_cast<int>(T);
                best.k = k;
                best.parts = parts;
                best.nd = static_cast<int>(nd);
                best.ns = static_cast<size_t>(T) * kd.tile;
                best.pi_slots = static_cast<size_t>(groups * parts);
                best.bytes = static_cast<size_t>((nd + groups * parts) * slot);
            }
        }
}

SymPlan nb_sym_plan(int precision, int64_t n, int sms, size_t max_bytes)
{
    SymPlan best;
    for (int q = 0; q < 3; ++q)
        nb_sym_plan_shape(kKinds[first_kind(precision) + q].shape, first_kind(precision) + q, n, sms, best,
                          max_bytes);
    return best;
}

cudaError_t nb_sym_smem_setup()
{
    for (const SymKind &kd : kKinds)
        for (auto kernel : {kd.light, kd.heavy}) {
            if (kd.smem == 0)
                continue;
            const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                       static_cast<int>(kd.smem));
            if (e != cudaSuccess)
                return e;
        }
    return cudaSuccess;
}

cudaError_t nb_launch_sym(int precision, const SymPlan &pl, const void *jb, size_t np, int n, double eps2,
                          bool light, void *work, double *out, size_t ostride, bool add, cudaStream_t stream,
                          int *launches)
{
    const SymKind &kind = kKinds[pl.kind];
    const SymShape &kd = kind.shape;
    SymArgs a;
    a.jb = jb;
    a.np = np;
    a.n = n;
    a.tiles = pl.T;
    a.k = pl.k;
    a.parts = pl.parts;
    a.eps2 = eps2;
    a.ns = pl.ns;
    a.pi = work;
    a.pj = static_cast<unsigned char *>(work) + pl.pi_slots * pl.ns * kd.bytes;
    const int D = pl.T / 2 + 1;
    for (int d0 = 0; d0 < D; d0 += pl.nd) {
        a.d0 = d0;
        a.d1 = std::min(D, d0 + pl.nd);
        const int64_t jobs = sym_jobs(pl.T, a.d0, a.d1, pl.k);
        const int groups = (a.d1 - a.d0 + pl.k - 1) / pl.k;
        const int upper = static_cast<int>(jobs / pl.T) * pl.parts;  // i-slots of the upper half of the tiles
        (light ? kind.light : kind.heavy)<<<static_cast<unsigned>(jobs * pl.parts), kd.threads, kind.smem, stream>>>(a);
        const dim3 grid((n + 255) / 256, 9);
        auto fold = [&](auto f) {
            using F = decltype(f);
            using P = typename F::Part;
            fold_kernel<F><<<grid, 256, 0, stream>>>(static_cast<const P *>(a.pi), groups * pl.parts, upper,
                                                     static_cast<const P *>(a.pj), a.d0, a.d1, a.ns, pl.T,
                                                     kd.tile, n, out, ostride, d0 == 0 && !add);
        };
        if (precision == NB_FP64)
            fold(Fold64{});
        else if (precision == NB_EX)
            fold(FoldEx{});
        else
            fold(FoldFF{});
        *launches += 2;
    }
    return cudaGetLastError();
}
