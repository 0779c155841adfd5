// Device-resident block stepping for one system (paper, section 3: block
// time steps, predictor / evaluation / corrector).
//
// Most block steps of a cluster integration have only a few active
// particles; driven from the host, each costs several launches and a host
// round trip for the size of the active set, more than its arithmetic.  This
// kernel runs such steps back to back in ONE cooperative launch whose blocks
// stay resident on every SM, separated by grid barriers:
//   schedule  every block scans its contiguous slice of the particles for
//             the earliest t_i + dt_i and lists the particles that reach it;
//             after a grid barrier all blocks read the same minima and counts
//             and take the same decision;
//   evaluate  every block predicts its slice and the active particles into
//             shared memory (chunk by chunk, the layout of the evaluation
//             buffer of the precision) and sums the active set against its
//             slice; partial sums go to global memory;
//   correct   after a second grid barrier the block that owns an active
//             particle adds the partial sums of all blocks in a fixed order
//             and applies the FP64 corrector and step selection (the same
//             device function as the corrector kernel).
// What bounds a step is latency: two barriers, the L2 round trips between
// them, and above all serial chains of FP64 instructions, each of which holds
// a scheduler's pipe for 64 clocks for a warp however few of its threads are
// active.  So FP64 work is spread over the block's four warps (prediction
// and corrector by component, sums over lanes and over blocks by value, each
// output a short chain of one thread), and comparisons use integers.  Time
// per step with about 13 active particles, before -> after: FP64 N = 1024
// 39.2 -> 18.1 us, EX N = 8192 46.1 -> 20.7 us, mixed N = 65536 58.0 -> 31.6 us.
// It returns to the host when the next active set holds more than
// kStepSmall particles (the host then runs that step with the tuned
// evaluation kernels), when the next block time passes t_end, or after an
// error flag.  Every block takes the same branch at every barrier (decisions
// come from the same global values), and no block waits on a flag.
#include <cooperative_groups.h>

#include <algorithm>

#include "nb_correct.cuh"
#include "nb_device.cuh"
#include "nb_ff.cuh"
#include "nb_internal.cuh"

namespace cg = cooperative_groups;

namespace {

using namespace nbk;

constexpr int kQ = 2;            // blocks of the grid per thread in the step decision
constexpr int kStepSmall = 128;  // active sets up to this size are stepped on the device
// Particles per block at least (small systems: fewer blocks), and the slice from
// which a block has 256 threads instead of 128: more warps predict a long
// slice, fewer make every sum over lanes and blocks shorter (us a step, 128 / 256
// threads: EX N = 8192 20.7 / 21.6, EX 20000 30.8 / 26.8, mixed 65536
// 38.5 / 31.6; FP64 N = 1024 with 8 and 16 particles per block 18.1 and 19.4).
constexpr int kSliceFp64 = 8, kSliceFp32 = 16, kSliceWide = 96;
constexpr int kChunkCap = 1024;  // j-records per shared-memory chunk

struct StepOut {
    int64_t steps;     // block steps taken by the launch
    int64_t act_sum;   // active particles summed over those steps
    int32_t reason;    // 0: next block time beyond t_end, 1: next active set too large, 2: error
    int32_t n_act;     // active count of the last step taken
    double t_last;     // time of the last step taken
};

struct StepArgs {
    int n;
    double *st, *t, *dt;
    const double *m;
    double eps2, eta, dt_min, dt_max, dt_shared, t_end, noise;
    int drop_lo;        // single-precision control: positions without their low part
    unsigned long long *bmin;  // [B] per-block earliest t_i + dt_i, as bits
    int *bcnt;          // [B] particles reaching it
    int *cand;          // [B][kStepSmall] their indices, ascending
    double *part;       // [kStepSmall][9][B] partial sums
    int32_t *act;       // active set of the last step taken
    nb_ctl *ctl;
    StepOut *out;
    double *log_t;      // per-step log (device), entries [log_base, log_cap)
    int64_t *log_n;
    int64_t log_cap, log_base;
};

// Bytes per j-record in shared memory: FP64 5 x 16, mixed 13 x 4, EX 20 x 4.
__host__ __device__ constexpr int rec_bytes(int pr) { return pr == 0 ? 80 : (pr == 1 ? NCF * 4 : NCX * 4); }

// Block minimum of 64-bit values (non-negative doubles order like their bits).
__device__ __forceinline__ unsigned long long block_min_u64(unsigned long long v, unsigned long long *red)
{
    for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long u = __shfl_xor_sync(0xffffffffu, v, o);
        v = u < v ? u : v;
    }
    __syncthreads();
    if ((threadIdx.x & 31) == 0)
        red[threadIdx.x >> 5] = v;
    __syncthreads();
    unsigned long long r = red[0];
    for (int q = 1; q < static_cast<int>(blockDim.x >> 5); ++q)
        r = red[q] < r ? red[q] : r;
    return r;
}

__device__ __forceinline__ int block_scan_excl(int v, int *red, int *total)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int incl = v;
    for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o)
            incl += u;
    }
    __syncthreads();
    if (lane == 31)
        red[w] = incl;
    __syncthreads();
    int base = 0, tot = 0;
    for (int q = 0; q < nw; ++q) {
        if (q < w)
            base += red[q];
        tot += red[q];
    }
    *total = tot;
    return base + incl - v;
}

// Component d of the predicted record of particle i at time tp, in rows of
// `stride` entries: FP64 10 rows x y z m vx vy vz ax ay az; mixed 13 FP32 rows
// (x_hi, m, x_lo, v, a; x_lo = 0 for the single-precision control); EX 20 FP32
// rows (hi then lo of x, v, a; m hi, lo).  d = 0 also stores the mass.
template <int PR>
__device__ __forceinline__ void predict_component(const StepArgs &a, int i, int d, double tp, void *rows, int stride)
{
    const size_t N = static_cast<size_t>(a.n), at = static_cast<size_t>(d) * N + i;
    const double dt = tp - a.t[i];
    const Taylor p = taylor(a.st[F_X * 3 * N + at], a.st[F_V * 3 * N + at], a.st[F_A * 3 * N + at],
                            a.st[F_J * 3 * N + at], a.st[F_S * 3 * N + at], a.st[F_C * 3 * N + at], dt);
    if constexpr (PR == 0) {
        double *r = static_cast<double *>(rows);
        r[d * stride] = p.x;
        r[(4 + d) * stride] = p.v;
        r[(7 + d) * stride] = p.a;
        if (d == 0)
            r[3 * stride] = a.m[i];
    } else if constexpr (PR == 1) {
        float *r = static_cast<float *>(rows);
        const float h = to_float(p.x);
        r[d * stride] = h;
        r[(4 + d) * stride] = a.drop_lo ? 0.0f : to_float(p.x - to_double(h));
        r[(7 + d) * stride] = to_float(p.v);
        r[(10 + d) * stride] = to_float(p.a);
        if (d == 0)
            r[3 * stride] = to_float(a.m[i]);
    } else {
        float *r = static_cast<float *>(rows);
        const double q[3] = {p.x, p.v, p.a};
#pragma unroll
        for (int g = 0; g < 3; ++g) {
            const float h = to_float(q[g]);
            r[(6 * g + d) * stride] = h;
            r[(6 * g + 3 + d) * stride] = to_float(q[g] - to_double(h));
        }
        if (d == 0) {
            const double mi = a.m[i];
            const float mh = to_float(mi);
            r[18 * stride] = mh;
            r[19 * stride] = to_float(mi - to_double(mh));
        }
    }
}

__host__ __device__ constexpr int rows_of(int pr) { return pr == 0 ? 10 : pr == 1 ? NCF : NCX; }
// Row entry size: double or float.
__host__ __device__ constexpr int word_of(int pr) { return pr == 0 ? 8 : 4; }

// v[0] + ... + v[n - 1] in four chains.
__device__ __forceinline__ double sum4(const double *v, int n)
{
    double s[4] = {0.0, 0.0, 0.0, 0.0};
    for (int e = 0; e < n; e += 4)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (e + c < n)
                s[c] += v[e + c];
    return (s[0] + s[1]) + (s[2] + s[3]);
}

// Sums of the K active particles (listed in act) over the j of [lo, hi), all
// predicted to tp, written to part[(k * 9 + q) * pstride].  L = T / K2 lanes per
// active particle (K2 the power of two >= K) take every L-th j (pair of j in
// the FP32 precisions); their sums meet in shared memory, where one thread per
// value adds them in lane order.  rec: rows of the active particles; red: 9 T
// 8-byte words.
template <int PR, int T>
__device__ void eval_slice(const StepArgs &a, int lo, int hi, double tp, int K, const int *act, void *rec,
                           double *part, int pstride, double *red, unsigned char *smem)
{
    const int tid = threadIdx.x;
    int K2 = 1;
    while (K2 < K)
        K2 <<= 1;
    const int L = T / K2;
    const int g = tid / L, lane = tid - g * L;
    const bool valid = g < K;
    const int gi = valid ? g : 0;
    constexpr int cap = kChunkCap;
    float *sf = reinterpret_cast<float *>(smem);
    double *sd = reinterpret_cast<double *>(smem);
    double acc[9];
    float2 ni[12], pm[9];
    float ah[9], al[9];
    ExI<float2> nie;
    ff::FF<float2> px[9];
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        acc[q] = 0.0;
        pm[q] = f2(0.0f);
        ah[q] = al[q] = 0.0f;
        px[q] = {f2(0.0f), f2(0.0f)};
    }
    const float2 eps2f = f2(__double2float_rn(a.eps2));
    const float e2h = __double2float_rn(a.eps2);
    const ff::FF<float2> eps2x = {f2(e2h), f2(__double2float_rn(a.eps2 - static_cast<double>(e2h)))};
    int cnt = 0;
    bool first = true, spilled = false;
    for (int b = lo; b < hi || first; b += cap) {
        const int len = max(0, min(cap, hi - b)), ka = first ? K : 0;
        // the slice and, with the first chunk, the active particles: few of
        // them by component, so that more warps share the FP64 chain; many
        // whole (the five step factors once instead of three times)
        const int m = len + ka, split = 2 * T >= 3 * m ? 3 : 1;
        for (int u = tid; u < split * m; u += T) {
            const int d0 = u / m, e = u - d0 * m;
            const int i = e < len ? b + e : act[e - len];
            unsigned char *rows = e < len ? smem + static_cast<size_t>(e) * word_of(PR)
                                          : static_cast<unsigned char *>(rec) + static_cast<size_t>(e - len) * word_of(PR);
            const int stride = e < len ? cap : kStepSmall;
            if (split == 3)
                predict_component<PR>(a, i, d0, tp, rows, stride);
            else
#pragma unroll
                for (int d = 0; d < 3; ++d)
                    predict_component<PR>(a, i, d, tp, rows, stride);
        }
        __syncthreads();
        if (first) {
            if (PR == 1) {
                const float *f = static_cast<const float *>(rec) + gi;
                constexpr int kRow[12] = {0, 1, 2, 4, 5, 6, 7, 8, 9, 10, 11, 12};
#pragma unroll
                for (int q = 0; q < 12; ++q)
                    ni[q] = f2(-f[kRow[q] * kStepSmall]);
            } else if (PR == 2) {
                const float *f = static_cast<const float *>(rec) + gi;
                auto neg = [&](int row) { return f2(-f[row * kStepSmall]); };
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    nie.x[k] = {neg(k), neg(3 + k)};
                    nie.v[k] = {neg(6 + k), neg(9 + k)};
                    nie.a[k] = {neg(12 + k), neg(15 + k)};
                }
            }
            first = false;
        }
        if constexpr (PR == 0) {
            const double *v = static_cast<const double *>(rec) + gi;
            auto iv = [&](int row) { return v[row * kStepSmall]; };
            for (int jj = lane; jj < len; jj += L) {
                auto c = [&](int row) { return sd[row * cap + jj]; };
                pair_fp64(make_double2(c(0), c(1)), make_double2(c(2), c(3)), make_double2(c(4), c(5)),
                          make_double2(c(6), c(7)), make_double2(c(8), c(9)), iv(0), iv(1), iv(2), iv(4), iv(5), iv(6),
                          iv(7), iv(8), iv(9), a.eps2, acc);
            }
        } else {
            constexpr int NR = PR == 1 ? NCF : NCX;
            constexpr int mrow = PR == 1 ? 3 : 18;  // first mass row
            for (int jj = 2 * lane; jj < len; jj += 2 * L) {
                float2 c[NR];
                if (jj + 1 < len) {
#pragma unroll
                    for (int r = 0; r < NR; ++r)
                        c[r] = *reinterpret_cast<const float2 *>(sf + r * cap + jj);
                } else {
                    // odd tail: the second half repeats the first j with no mass
#pragma unroll
                    for (int r = 0; r < NR; ++r) {
                        const float x0 = sf[r * cap + jj];
                        c[r] = make_float2(x0, r >= mrow ? 0.0f : x0);
                    }
                }
                if constexpr (PR == 1)
                    pair_mixed2(c, ni, eps2f, pm);
                else
                    pair_ex(c, nie, eps2x, px);
                if (++cnt == 32) {
#pragma unroll
                    for (int q = 0; q < 9; ++q) {
                        if (PR == 1) {
                            two_sum_acc(ah[q], al[q], __fadd_rn(pm[q].x, pm[q].y));
                            pm[q] = f2(0.0f);
                        } else {
                            acc[q] += (static_cast<double>(px[q].h.x) + static_cast<double>(px[q].l.x)) +
                                      (static_cast<double>(px[q].h.y) + static_cast<double>(px[q].l.y));
                            px[q] = {f2(0.0f), f2(0.0f)};
                        }
                    }
                    cnt = 0;
                    spilled = true;
                }
            }
        }
        __syncthreads();
    }
    // this thread's sums: doubles, or (hi, lo) words in the FP32 precisions
    // (EX: the two halves of the packed sums joined by a double-word sum, and
    // FP64 only where more than 32 iterations went to acc)
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        if (PR == 0) {
            red[tid * 9 + q] = acc[q];
        } else if (PR == 1) {
            two_sum_acc(ah[q], al[q], __fadd_rn(pm[q].x, pm[q].y));
            const int span = L < 32 ? L : 32;
            for (int o = span >> 1; o > 0; o >>= 1) {
                const float oh = __shfl_xor_sync(0xffffffffu, ah[q], o);
                const float ol = __shfl_xor_sync(0xffffffffu, al[q], o);
                two_sum_acc(ah[q], al[q], oh);
                al[q] = __fadd_rn(al[q], ol);
            }
            reinterpret_cast<float2 *>(red)[tid * 9 + q] = make_float2(ah[q], al[q]);
        } else {
            const ff::FF<float> x = {px[q].h.x, px[q].l.x}, y = {px[q].h.y, px[q].l.y};
            const ff::FF<float> s = ff::add_accurate(x, y);
            reinterpret_cast<float2 *>(red)[tid * 9 + q] = make_float2(s.h, s.l);
        }
    }
    __syncthreads();
    // the lanes' sums (mixed: one per warp or group): S threads per value take
    // every S-th lane, one adds their sums; four chains each (an FP64 addition
    // waits about a hundred clocks for the one before)
    const int stepl = PR == 1 ? (L < 32 ? L : 32) : 1, nl = L / stepl, nv = 9 * K;
    const int S = max(1, min(T / nv, nl / 4));
    auto lane_sum = [&](int v, int s0) {
        const int k = v / 9, q = v - 9 * k;
        double s[4] = {0.0, 0.0, 0.0, 0.0};
        for (int e = s0; e < nl; e += 4 * S)
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (e + c * S < nl) {
                    const int at = (k * L + (e + c * S) * stepl) * 9 + q;
                    if (PR == 0) {
                        s[c] += red[at];
                    } else {
                        const float2 w = reinterpret_cast<const float2 *>(red)[at];
                        s[c] += to_double(w.x) + to_double(w.y);
                    }
                }
        return (s[0] + s[1]) + (s[2] + s[3]);
    };
    if (S == 1) {
        for (int u = tid; u < nv; u += T)
            part[static_cast<size_t>(u) * pstride] = lane_sum(u, 0);
    } else {
        const double mine = tid < nv * S ? lane_sum(tid / S, tid % S) : 0.0;
        __syncthreads();
        red[tid] = mine;
        __syncthreads();
        if (tid < nv)
            part[static_cast<size_t>(tid) * pstride] = sum4(red + tid * S, S);
    }
    if (PR == 2 && __syncthreads_or(spilled)) {
        // long slices: the FP64 sums of the first iterations, added behind
        __syncthreads();
#pragma unroll
        for (int q = 0; q < 9; ++q)
            red[tid * 9 + q] = acc[q];
        __syncthreads();
        for (int u = tid; u < 9 * K; u += T) {
            const int k = u / 9, q = u - 9 * k;
            double s = part[static_cast<size_t>(u) * pstride];
            for (int e = 0; e < L; ++e)
                s += red[(k * L + e) * 9 + q];
            part[static_cast<size_t>(u) * pstride] = s;
        }
    }
    __syncthreads();
}

template <int PR, int T>
__global__ void __launch_bounds__(T) step_kernel(StepArgs a)
{
    cg::grid_group grid = cg::this_grid();
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ unsigned long long red_u[T / 32];
    __shared__ int red_i[T / 32];
    __shared__ int s_act[kStepSmall];
    __shared__ __align__(8) unsigned char s_rec[kStepSmall * rows_of(PR) * word_of(PR)];
    __shared__ double s_red[9 * T];  // sums of the lanes, then of the blocks
    __shared__ CorrectScratch s_cor;
    const int B = gridDim.x, bk = blockIdx.x, tid = threadIdx.x;
    const int per = (a.n + B - 1) / B;
    const int lo = min(a.n, bk * per), hi = min(a.n, lo + per);
    const int per_t = (hi - lo + T - 1) / T;
    const int c0 = min(hi, lo + tid * per_t), c1 = min(hi, c0 + per_t);
    int64_t steps = 0, act_sum = 0;
    int reason = 0, last_n = 0;
    double last_t = 0.0;
    for (;;) {
        // schedule: this block's earliest t_i + dt_i, the particles reaching it
        unsigned long long mt = ~0ull;
        int ct = 0;
        for (int i = c0; i < c1; ++i) {
            const unsigned long long tt = static_cast<unsigned long long>(__double_as_longlong(a.t[i] + a.dt[i]));
            if (tt < mt) {
                mt = tt;
                ct = 1;
            } else if (tt == mt) {
                ++ct;
            }
        }
        const unsigned long long mb = block_min_u64(mt, red_u);
        const int mine = (mt == mb && mb != ~0ull) ? ct : 0;
        int tot_b = 0;
        const int ex = block_scan_excl(mine, red_i, &tot_b);
        if (mine > 0 && tot_b <= kStepSmall) {
            int pos = ex;
            for (int i = c0; i < c1; ++i)
                if (static_cast<unsigned long long>(__double_as_longlong(a.t[i] + a.dt[i])) == mb)
                    a.cand[bk * kStepSmall + pos++] = i;
        }
        if (tid == 0) {
            a.bmin[bk] = mb;
            a.bcnt[bk] = tot_b;
        }
        grid.sync();
        // the same decision in every block: thread tid looks at the blocks
        // kQ tid .. kQ tid + kQ - 1
        unsigned long long bm[kQ], mn_bits = ~0ull;
        int bc[kQ];
#pragma unroll
        for (int e = 0; e < kQ; ++e) {
            const int q = tid * kQ + e;
            bm[e] = q < B ? __ldcg(&a.bmin[q]) : ~0ull;
            bc[e] = q < B ? __ldcg(&a.bcnt[q]) : 0;
            mn_bits = bm[e] < mn_bits ? bm[e] : mn_bits;
        }
        const int err = *reinterpret_cast<volatile int *>(&a.ctl->err);
        mn_bits = block_min_u64(mn_bits, red_u);
        const double mn = __longlong_as_double(static_cast<long long>(mn_bits));
        int c = 0;
#pragma unroll
        for (int e = 0; e < kQ; ++e)
            c += bm[e] == mn_bits ? min(bc[e], kStepSmall + 1) : 0;
        int total = 0;
        int pos = block_scan_excl(c, red_i, &total);
        if (err) {
            reason = 2;
            break;
        }
        if (mn > a.t_end) {
            reason = 0;
            break;
        }
        if (total > kStepSmall) {
            reason = 1;
            break;
        }
        // active list, ascending: blocks in order, each block's list in order
#pragma unroll
        for (int e = 0; e < kQ; ++e)
            if (bm[e] == mn_bits)
                for (int u = 0; u < bc[e]; ++u)
                    s_act[pos++] = (tid * kQ + e) * kStepSmall + u;
        __syncthreads();
        if (tid < total)
            s_act[tid] = __ldcg(&a.cand[s_act[tid]]);
        __syncthreads();
        eval_slice<PR, T>(a, lo, hi, mn, total, s_act, s_rec, a.part + bk, B, s_red, smem);
        grid.sync();
        // this block's active particles (they are consecutive in the list)
        int first_own = 0, own = 0;
        for (int k = 0; k < total; ++k) {
            const int i = s_act[k];
            if (i < lo)
                first_own = k + 1;
            else if (i < hi)
                ++own;
        }
        for (int o0 = 0; o0 < own; o0 += 32) {
            const int no = min(32, own - o0);
            // the partial sums of all blocks: S threads per value take every
            // S-th block, one adds their sums in order
            const int nv = 9 * no;
            const int S = nv <= T ? T / nv : 1;
            for (int u = tid; u < nv * S; u += T) {
                const int v = u / S, s = u - v * S;
                const double *pp = a.part + (static_cast<size_t>(first_own + o0) * 9 + v) * B;
                double sum[4] = {0.0, 0.0, 0.0, 0.0};
                constexpr int U = 12;  // loads in flight
                for (int q = s; q < B; q += U * S) {
                    double w[U];
#pragma unroll
                    for (int e = 0; e < U; ++e)
                        w[e] = q + e * S < B ? __ldcg(pp + q + e * S) : 0.0;
#pragma unroll
                    for (int e = 0; e < U; ++e)
                        if (q + e * S < B)
                            sum[e & 3] += w[e];
                }
                s_red[u] = (sum[0] + sum[1]) + (sum[2] + sum[3]);
            }
            __syncthreads();
            if (S > 1) {
                const double sum = tid < nv ? sum4(s_red + tid * S, S) : 0.0;
                __syncthreads();
                if (tid < nv)
                    s_red[tid] = sum;
                __syncthreads();
            }
            const int lane = tid & 31, d = tid >> 5;
            const bool valid = d < 3 && lane < no;
            double f[3] = {0.0, 0.0, 0.0};
            if (valid)
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    f[q] = s_red[lane * 9 + 3 * q + d];
            correct_group_fp64(a.st, a.t, a.dt, static_cast<size_t>(a.n), valid ? s_act[first_own + o0 + lane] : 0,
                               valid, mn, f, a.eta, a.dt_min, a.dt_max, a.dt_shared, a.ctl, a.noise, s_cor);
        }
        if (bk == 0) {
            for (int k = tid; k < total; k += T)
                a.act[k] = s_act[k];
            if (tid == 0) {
                const int64_t li = a.log_base + steps;
                if (li < a.log_cap) {
                    a.log_t[li] = mn;
                    a.log_n[li] = total;
                }
            }
        }
        ++steps;
        act_sum += total;
        last_t = mn;
        last_n = total;
        __syncthreads();
    }
    if (bk == 0 && tid == 0) {
        a.out->steps = steps;
        a.out->act_sum = act_sum;
        a.out->reason = reason;
        a.out->n_act = last_n;
        a.out->t_last = last_t;
    }
}

template <int PR, int T>
cudaError_t launch_stepper(nb_ctx *c, StepArgs &a, int grid)
{
    const size_t smem = static_cast<size_t>(kChunkCap) * rec_bytes(PR);
    cudaError_t e = cudaFuncSetAttribute(step_kernel<PR, T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         static_cast<int>(smem));
    if (e != cudaSuccess)
        return e;
    void *args[] = {&a};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(step_kernel<PR, T>), dim3(grid), dim3(T), args,
                                       smem, c->stream);
}

// One block per SM (with two, every barrier and sum over blocks grows: EX
// N = 8192 28.2 us a step), all of them resident.
template <int PR>
cudaError_t launch_stepper(nb_ctx *c, StepArgs &a, int grid_max)
{
    const int slice = PR == 0 ? kSliceFp64 : kSliceFp32;
    const int grid = std::min({c->sm_count, grid_max, kQ * 128,
                               std::max(1, static_cast<int>((c->n + slice - 1) / slice))});
    return c->n >= static_cast<int64_t>(grid) * kSliceWide ? launch_stepper<PR, 256>(c, a, grid)
                                                           : launch_stepper<PR, 128>(c, a, grid);
}

}  // namespace

int nb_stepper_small() { return kStepSmall; }

// One launch of the device-resident stepper; reports what it did in
// *steps, *act_sum, *reason, *n_act, *t_last (synchronises the stream).
cudaError_t nb_run_stepper(nb_ctx *c, double t_end, int64_t log_cap, int64_t log_base, int64_t *steps,
                           int64_t *act_sum, int *reason, int *n_act, double *t_last)
{
    // scratch sized for the largest grid this device can hold
    const int grid_max = c->sm_count * 16;
    if (!c->stp_bmin) {
        cudaError_t e;
        if ((e = cudaMalloc(&c->stp_bmin, grid_max * sizeof(double))) != cudaSuccess) return e;
        if ((e = cudaMalloc(&c->stp_bcnt, grid_max * sizeof(int))) != cudaSuccess) return e;
        if ((e = cudaMalloc(&c->stp_cand, static_cast<size_t>(grid_max) * kStepSmall * sizeof(int))) != cudaSuccess)
            return e;
        if ((e = cudaMalloc(&c->stp_part, static_cast<size_t>(grid_max) * kStepSmall * 9 * sizeof(double))) !=
            cudaSuccess)
            return e;
        if ((e = cudaMalloc(&c->stp_out, sizeof(StepOut))) != cudaSuccess) return e;
        if ((e = cudaMallocHost(&c->stp_out_h, sizeof(StepOut))) != cudaSuccess) return e;
    }
    StepArgs a;
    a.n = static_cast<int>(c->n);
    a.st = c->st;
    a.t = c->t;
    a.dt = c->dt;
    a.m = c->m;
    a.eps2 = c->eps * c->eps;
    a.eta = c->cfg.eta;
    a.noise = c->cfg.step_noise;
    a.dt_min = c->cfg.dt_min;
    a.dt_max = c->cfg.dt_max;
    a.dt_shared = c->cfg.dt_shared;
    a.t_end = t_end;
    a.drop_lo = c->cfg.precision == NB_SP ? 1 : 0;
    a.bmin = reinterpret_cast<unsigned long long *>(c->stp_bmin);
    a.bcnt = c->stp_bcnt;
    a.cand = c->stp_cand;
    a.part = c->stp_part;
    a.act = c->act;
    a.ctl = c->ctl;
    a.out = static_cast<StepOut *>(c->stp_out);
    a.log_t = c->stp_log_t;
    a.log_n = c->stp_log_n;
    a.log_cap = c->stp_log_t ? log_cap : 0;
    a.log_base = log_base;
    const int pr = c->cfg.precision == NB_EX ? 2 : (nb_fp32_eval(c->cfg.precision) ? 1 : 0);
    cudaError_t e = pr == 2 ? launch_stepper<2>(c, a, grid_max)
                            : (pr == 1 ? launch_stepper<1>(c, a, grid_max) : launch_stepper<0>(c, a, grid_max));
    if (e != cudaSuccess)
        return e;
    c->launches += 1;
    e = cudaMemcpyAsync(c->stp_out_h, c->stp_out, sizeof(StepOut), cudaMemcpyDeviceToHost, c->stream);
    if (e != cudaSuccess)
        return e;
    e = cudaStreamSynchronize(c->stream);
    if (e != cudaSuccess)
        return e;
    const StepOut *o = static_cast<const StepOut *>(c->stp_out_h);
    *steps = o->steps;
    *act_sum = o->act_sum;
    *reason = o->reason;
    *n_act = o->n_act;
    *t_last = o->t_last;
    return cudaSuccess;
}
