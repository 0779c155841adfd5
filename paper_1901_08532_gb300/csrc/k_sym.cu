// Evaluation of a complete active set (paper, section 3 item 4): every
// particle is active, so each unordered pair {i, j} is needed in both
// directions, and both come from one set of differences, powers of R, alpha
// and beta.  Swapping i and j negates r, v and a, keeps alpha and beta, and
// so negates u and w: the terms on j are (-m_i / m_j) times those on i.  Per
// unordered pair the mixed formula takes 63 FP32-pipe operations instead of
// 2 x 53 (FP64 63 instead of 106, EX 608 instead of 992).
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

namespace {

using namespace nbk;

struct SymArgs {
    const void *jb;  // predicted particles (the evaluation buffer's rows)
    size_t np;       // row stride
    int n;
    int tiles;       // T
    int d0, d1;      // offsets of this launch, [d0, d1)
    int k;           // offsets per block
    int parts;       // H, parts of a j-tile
    double eps2;
    void *pi, *pj;   // partial sums: [group * H + h][9][ns], [d - d0][9][ns]
    size_t ns;       // T * B
};

// cp.async of one 32-bit word; bytes = 0 writes a zero.
__device__ __forceinline__ void cp_async4(void *dst, const void *src, uint32_t bytes)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Is offset d evaluated from tile b (for even T the last offset only from the
// lower half)?
__host__ __device__ __forceinline__ bool sym_job(int T, int b, int d) { return 2 * d != T || b < T / 2; }

// ----------------------------------------------------------------- mixed

constexpr int kMixedWarps = 4;
constexpr int kMixedThreads = 32 * kMixedWarps;
__host__ __device__ constexpr int mixed_tile(int kp) { return kMixedThreads * 2 * kp; }

// Both directions of the pairs of two i-particles (the lanes of the packed
// values) with one j: pi += terms on i, pj += terms on j.  ni are the negated
// i-values, nmi the negated masses, c the 13 j-values.
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
    const float2 q3 = mul2(q, q2);
    const float2 mu = mul2(f2(c[3]), q3), nu = mul2(nmi, q3);
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
// 4096 51 -> 39 us, 8192 150 -> 111, 20011 744 -> 500, 65536 7.26 -> 4.80 ms,
// 131072 28.6 -> 18.7 ms, 2^20 1.813 -> 1.178 s.  Below about 3500 particles the ordinary kernels
// are faster (3000: 34 us against 39).
template <int KP>
__global__ void __launch_bounds__(kMixedThreads, 2) sym_mixed_kernel(SymArgs a)
{
    constexpr int W = kMixedWarps, TH = kMixedThreads, B = mixed_tile(KP);
    extern __shared__ __align__(16) float sm[];
    float *tile = sm;                        // [2][NCF][TH]
    float *jacc = sm + 2 * NCF * TH;         // [18][TH]: hi of the 9 sums, then lo
    float *iacc = jacc + 18 * TH;            // [2 KP][18][TH]
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    // block -> part h of the job (tile b, offsets of group g); the last group of
    // an even T may be launched for the lower half of the tiles only
    const int h = blockIdx.x % a.parts, b = blockIdx.x / a.parts % a.tiles, g = blockIdx.x / a.parts / a.tiles;
    const int da = a.d0 + g * a.k, db = min(a.d1, da + a.k);
    const int part = B / a.parts, subs = part / TH;  // j per job part, tiles of TH
    const float *jf = static_cast<const float *>(a.jb);
    const float2 eps2 = f2(static_cast<float>(a.eps2));
    constexpr int kRow[12] = {0, 1, 2, 4, 5, 6, 7, 8, 9, 10, 11, 12};

    float2 ni[KP][12], nmi[KP], pi[KP][9];
#pragma unroll
    for (int p = 0; p < KP; ++p) {
        const int i = b * B + (w * KP + p) * 64 + 2 * lane;
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

    // the sub-tiles of this block's jobs in order: it -> (offset, sub-tile)
    const int last = (db - 1 >= da && !sym_job(a.tiles, b, db - 1)) ? db - 1 : db;
    const int nit = max(0, last - da) * subs;
    auto tile_start = [&](int it) {
        int c = b + da + it / subs;
        if (c >= a.tiles)
            c -= a.tiles;
        return c * B + h * part + (it % subs) * TH;
    };
    if (nit > 0)
        load_tile_mixed(a, tile, tile_start(0));
    for (int it = 0; it < nit; ++it) {
        cp_async_wait_all();
        __syncthreads();
        if (it + 1 < nit)
            load_tile_mixed(a, tile + ((it + 1) & 1) * NCF * TH, tile_start(it + 1));
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
                        pair_mixed_sym(c, ni[p], nmi[p], eps2, pi[p], pj);
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
        const int d = da + it / subs;
        float2 *pj = static_cast<float2 *>(a.pj) + static_cast<size_t>(d - a.d0) * 9 * a.ns + tile_start(it) + tid;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            if (d > 0)
                pj[q * a.ns] = make_float2(jacc[q * TH + tid], jacc[(9 + q) * TH + tid]);
            jacc[q * TH + tid] = 0.0f;
            jacc[(9 + q) * TH + tid] = 0.0f;
        }
    }
    float2 *pi_out = static_cast<float2 *>(a.pi) + static_cast<size_t>(g * a.parts + h) * 9 * a.ns;
#pragma unroll
    for (int p = 0; p < KP; ++p) {
        const int i = b * B + (w * KP + p) * 64 + 2 * lane;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const float *ia = iacc + (p * 36 + q) * TH + tid;
            *reinterpret_cast<float4 *>(&pi_out[q * a.ns + i]) =
                make_float4(ia[0], ia[9 * TH], ia[18 * TH], ia[27 * TH]);
        }
    }
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

// out[q][p] (+)= the i-slots in order, then the j-slots in order of the offset.
template <class F>
__global__ void __launch_bounds__(256) fold_kernel(const typename F::Part *pi, int nslots, int upper,
                                                   const typename F::Part *pj, int d0, int d1, size_t ns,
                                                   int T, int B, int n, double *out, size_t ostride, int first)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const int q = blockIdx.y;
    if (p >= n)
        return;
    constexpr int U = 8;  // slots in flight
    F f;
    const size_t step = 9 * ns;
    const typename F::Part *src = pi + q * ns + p;
    // tile c takes j-sums at every offset but 0, and at d = T/2 only in the
    // upper half, which has `upper` i-slots
    const int c = p / B;
    if (c >= T / 2)
        nslots = upper;
    int s = 0;
    for (; s + U <= nslots; s += U) {
        typename F::Part v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            v[u] = src[(s + u) * step];
#pragma unroll
        for (int u = 0; u < U; ++u)
            f.add(v[u]);
    }
    for (; s < nslots; ++s)
        f.add(src[s * step]);
    const int da = max(d0, 1), db = (2 * (d1 - 1) == T && c < T / 2) ? d1 - 1 : d1;
    src = pj + q * ns + p;
    int d = da;
    for (; d + U <= db; d += U) {
        typename F::Part v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            v[u] = src[(d - d0 + u) * step];
#pragma unroll
        for (int u = 0; u < U; ++u)
            f.add(v[u]);
    }
    for (; d < db; ++d)
        f.add(src[(d - d0) * step]);
    double *o = out + q * ostride + p;
    *o = first ? f.total() : *o + f.total();
}

size_t mixed_smem(int kp) { return sizeof(float) * kMixedThreads * (2 * NCF + 18 + 36 * kp); }

}  // namespace

// ------------------------------------------------------------------- plan

// The kernels of a precision: particles per tile, threads, bytes of a partial
// sum, and the measured rate with the chip full in unordered pairs per
// microsecond and SM.
struct SymKind {
    int kp, tile, threads, bytes;
    double rate;
};

constexpr SymKind kMixedKinds[] = {{3, mixed_tile(3), kMixedThreads, 8, 3170.0},
                                   {2, mixed_tile(2), kMixedThreads, 8, 2750.0},
                                   {1, mixed_tile(1), kMixedThreads, 8, 2200.0}};

// Tiles x groups of the offsets [d0, d1), without the upper half of the tiles
// where the last group is the offset T / 2 alone.
static int64_t sym_jobs(int64_t T, int64_t d0, int64_t d1, int64_t k)
{
    const int64_t groups = (d1 - d0 + k - 1) / k;
    return T * groups - (2 * (d1 - 1) == T && (d1 - d0 - 1) % k == 0 ? T / 2 : 0);
}

// The estimate behind a plan: the SM with the most jobs works through them at
// the kernel's full rate (one block of four warps reaches 88 % of it), plus a
// fixed part per job and launch and the traffic of the slots.  Within 5 % of
// the measured times of the plans it chooses from 4096 to 524288 particles;
// the next best plans lie within 2 % there.
static void plan_kind(const SymKind &kd, int kind, int64_t n, int sms, SymPlan &best)
{
    const int64_t T = (n + kd.tile - 1) / kd.tile, D = T / 2 + 1;
    const double slot = 9.0 * kd.bytes * static_cast<double>(T * kd.tile);
    const int64_t slots = std::max<int64_t>(2, static_cast<int64_t>(kSymSlotBytes / slot));
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
            const int64_t each = (jobs + sms - 1) / sms;
            const double pairs = static_cast<double>(kd.tile) * kd.tile * std::min<int64_t>(k, nd) / parts;
            const double us = batches * ((each > 1 ? each + (k > 1 ? 0.5 : 0.05) : 1.12) * (pairs / kd.rate + 1.0) + 5.0 +
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

SymPlan nb_sym_plan(int precision, int64_t n, int sms)
{
    SymPlan best;
    if (nb_fp32_eval(precision))
        for (int q = 0; q < 3; ++q)
            plan_kind(kMixedKinds[q], q, n, sms, best);
    return best;
}

template <typename K>
static cudaError_t allow_smem(K kernel, size_t bytes)
{
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
}

cudaError_t nb_sym_smem_setup()
{
    cudaError_t e;
    if ((e = allow_smem(sym_mixed_kernel<1>, mixed_smem(1))) != cudaSuccess) return e;
    if ((e = allow_smem(sym_mixed_kernel<2>, mixed_smem(2))) != cudaSuccess) return e;
    return allow_smem(sym_mixed_kernel<3>, mixed_smem(3));
}

cudaError_t nb_launch_sym(int precision, const SymPlan &pl, const void *jb, size_t np, int n, double eps2,
                          void *work, double *out, size_t ostride, cudaStream_t stream, int *launches)
{
    const SymKind &kd = kMixedKinds[pl.kind];
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
    a.pj = static_cast<unsigned char *>(work) + pl.pi_slots * 9 * pl.ns * kd.bytes;
    const int D = pl.T / 2 + 1;
    for (int d0 = 0; d0 < D; d0 += pl.nd) {
        a.d0 = d0;
        a.d1 = std::min(D, d0 + pl.nd);
        const int groups = (a.d1 - a.d0 + pl.k - 1) / pl.k;
        const unsigned grid = static_cast<unsigned>(sym_jobs(pl.T, a.d0, a.d1, pl.k) * pl.parts);
        const size_t smem = mixed_smem(kd.kp);
        if (kd.kp == 3) sym_mixed_kernel<3><<<grid, kd.threads, smem, stream>>>(a);
        else if (kd.kp == 2) sym_mixed_kernel<2><<<grid, kd.threads, smem, stream>>>(a);
        else sym_mixed_kernel<1><<<grid, kd.threads, smem, stream>>>(a);
        fold_kernel<FoldFF><<<dim3((n + 255) / 256, 9), 256, 0, stream>>>(
            static_cast<const float2 *>(a.pi), groups * pl.parts,
            static_cast<int>(sym_jobs(pl.T, a.d0, a.d1, pl.k) / pl.T) * pl.parts,
            static_cast<const float2 *>(a.pj), a.d0, a.d1,
            a.ns, pl.T, kd.tile, n, out, ostride, d0 == 0);
        *launches += 2;
    }
    return cudaGetLastError();
}
