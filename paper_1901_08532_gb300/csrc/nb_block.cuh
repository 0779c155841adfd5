// A block's share of a block step with a small active set, for the device-
// resident stepper (k_stepper.cu) and the ensemble (k_ensemble.cu): prediction
// by component, and the sums of the active particles over the block's slice.
// Both are bound by latency; k_stepper.cu says how that shapes them.
#pragma once

#include "nb_device.cuh"
#include "nb_ff.cuh"

namespace nbk {

// State a block predicts from: rows st[(F * 3 + d) * n + i].
struct StateView {
    const double *st, *t, *m;
    size_t n;
    int drop_lo;  // single-precision control: positions without their low part
};

// Bytes per j-record in shared memory: FP64 5 x 16, mixed 13 x 4, EX 20 x 4.
__host__ __device__ constexpr int rec_bytes(int pr) { return pr == 0 ? 80 : (pr == 1 ? NCF * 4 : NCX * 4); }

// Block minimum of 64-bit values (times as time_key(), or as their bits where
// none is negative).
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
__device__ __forceinline__ void predict_component(const StateView &a, int i, int d, double tp, void *rows, int stride)
{
    const size_t N = a.n, at = static_cast<size_t>(d) * N + i;
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

// s[q] (+)= the halves of the packed double words p[q], joined in FP64: the words
// meet in exact FP32 sums, which leaves two FP64 additions of the three, and one
// test covers the conversions.
__device__ __forceinline__ void join_halves(const ff::FF<float2> (&p)[9], bool add, double (&s)[9])
{
    float w[9][3];
    bool normal = true;
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        const ff::FF<float> h = ff::two_sum(p[q].h.x, p[q].h.y), l = ff::two_sum(p[q].l.x, p[q].l.y);
        const ff::FF<float> m = ff::two_sum(h.l, l.h);
        w[q][0] = h.h;
        w[q][1] = m.h;
        w[q][2] = ff::add(m.l, l.l);
#pragma unroll
        for (int k = 0; k < 3; ++k)
            normal = normal && zero_or_normal(w[q][k]);
    }
    auto join = [&](auto wide) {
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const double v = wide(w[q][0]) + (wide(w[q][1]) + wide(w[q][2]));
            s[q] = add ? s[q] + v : v;
        }
    };
    if (normal)
        join([](float x) { return to_double_normal(x); });
    else
        join([](float x) { return static_cast<double>(x); });
}

// Sums of the K active particles (listed in act, at most kmax) over the j of
// [lo, hi), all predicted to tp, written to part[(k * 9 + q) * pstride].  The
// slice goes through shared memory in chunks of cap records.  L = T / K2 lanes
// per active particle (K2 the power of two >= K) take every L-th j (pair of j
// in the FP32 precisions); their sums meet in shared memory, where threads
// add them in a fixed order.  rec: rows of the active particles, stride kmax;
// red: 9 T 8-byte words (it may lie in smem).  Record(i, d, rows, stride)
// writes component d (d < 0: all) of particle i's predicted record.
template <int PR, class Record>
__device__ __forceinline__ void eval_slice(const Record &record, double eps2, int lo, int hi, int K, const int *act,
                                           void *rec, int kmax, double *part, int pstride, double *red,
                                           unsigned char *smem, int cap, int T)
{
    const int tid = threadIdx.x;
    int K2 = 1;
    while (K2 < K)
        K2 <<= 1;
    const int L = T / K2;
    const int g = tid / L, lane = tid - g * L;
    const bool valid = g < K;
    const int gi = valid ? g : 0;
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
    const float2 eps2f = f2(__double2float_rn(eps2));
    const float e2h = __double2float_rn(eps2);
    const ff::FF<float2> eps2x = {f2(e2h), f2(__double2float_rn(eps2 - static_cast<double>(e2h)))};
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
            const int stride = e < len ? cap : kmax;
            record(i, split == 3 ? d0 : -1, rows, stride);
        }
        __syncthreads();
        if (first) {
            if (PR == 1) {
                const float *f = static_cast<const float *>(rec) + gi;
                constexpr int kRow[12] = {0, 1, 2, 4, 5, 6, 7, 8, 9, 10, 11, 12};
#pragma unroll
                for (int q = 0; q < 12; ++q)
                    ni[q] = f2(-f[kRow[q] * kmax]);
            } else if (PR == 2) {
                const float *f = static_cast<const float *>(rec) + gi;
                auto neg = [&](int row) { return f2(-f[row * kmax]); };
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
            auto iv = [&](int row) { return v[row * kmax]; };
            for (int jj = lane; jj < len; jj += L) {
                auto c = [&](int row) { return sd[row * cap + jj]; };
                pair_fp64(make_double2(c(0), c(1)), make_double2(c(2), c(3)), make_double2(c(4), c(5)),
                          make_double2(c(6), c(7)), make_double2(c(8), c(9)), iv(0), iv(1), iv(2), iv(4), iv(5), iv(6),
                          iv(7), iv(8), iv(9), eps2, acc);
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
    // mixed: lanes joined by shuffles, in groups of a power of two of them
    const int span = min(32, L & -L);
    // this thread's sums: doubles, or (hi, lo) words in the mixed precision
    if (PR == 2)
        join_halves(px, spilled, acc);  // acc is zero in short slices
#pragma unroll
    for (int q = 0; q < 9; ++q) {
        if (PR != 1) {
            red[tid * 9 + q] = acc[q];
        } else {
            two_sum_acc(ah[q], al[q], __fadd_rn(pm[q].x, pm[q].y));
            for (int o = span >> 1; o > 0; o >>= 1) {
                const float oh = __shfl_xor_sync(0xffffffffu, ah[q], o);
                const float ol = __shfl_xor_sync(0xffffffffu, al[q], o);
                two_sum_acc(ah[q], al[q], oh);
                al[q] = __fadd_rn(al[q], ol);
            }
            reinterpret_cast<float2 *>(red)[tid * 9 + q] = make_float2(ah[q], al[q]);
        }
    }
    __syncthreads();
    // the lanes' sums (mixed: one per warp or group): S threads per value take
    // every S-th lane, one adds their sums; four chains each (an FP64 addition
    // waits about a hundred clocks for the one before)
    const int stepl = PR == 1 ? span : 1, nl = L / stepl, nv = 9 * K;
    const int S = max(1, min(T / nv, nl / 4));
    auto lane_sum = [&](int v, int s0) {
        const int k = v / 9, q = v - 9 * k;
        double s[4] = {0.0, 0.0, 0.0, 0.0};
        for (int e = s0; e < nl; e += 4 * S)
#pragma unroll
            for (int c = 0; c < 4; ++c)
                if (e + c * S < nl) {
                    const int at = (k * L + (e + c * S) * stepl) * 9 + q;
                    if (PR != 1) {
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
    __syncthreads();
}

// The FP64 prediction as eval_slice's Record.
template <int PR>
struct PredictedRecord {
    StateView v;
    double tp;
    __device__ __forceinline__ void operator()(int i, int d, void *rows, int stride) const
    {
        if (d >= 0)
            predict_component<PR>(v, i, d, tp, rows, stride);
        else
#pragma unroll
            for (int k = 0; k < 3; ++k)
                predict_component<PR>(v, i, k, tp, rows, stride);
    }
};

}  // namespace nbk
