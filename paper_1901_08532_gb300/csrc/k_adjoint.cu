// All-pairs evaluation and its hand-written adjoint, FP64, stateless (every
// particle active), for differentiating fixed-step Hermite trajectories.
//
// Forward: the caller's rows x, v, a [n][3] and m [n] are packed into the
// evaluation records and the FP64 evaluation kernel runs with every particle
// active (paper, section 3 item 4).
//
// Adjoint: for a pair term (i <- j) with r = x_j - x_i, v = v_j - v_i,
// a = a_j - a_i, R = r.r + eps^2, q = R^(-1/2), mu = m_j q^3,
// alpha = (r.v) q^2, beta = (v.v + r.a) q^2 + alpha^2, u = v - 3 alpha r,
// w = a - 6 alpha u - 3 beta r and A = mu r, J = mu u, S = mu w, the
// cotangents (Ab, Jb, Sb) of particle i give L = Ab.A + Jb.J + Sb.S = mu Phi,
//   Phi = Pr.r + (Jb - 6 alpha Sb).v + Sb.a,
//   Pr  = Ab - 3 alpha Jb + (18 alpha^2 - 3 beta) Sb.
// With Pa = dPhi/dalpha = -3 Jb.r - 6 Sb.v + 36 alpha Sb.r and
// Pb = dPhi/dbeta = -3 Sb.r (alpha and beta held fixed in Phi):
//   dL/dr = mu [Pr + q^2 ((Pa + 2 alpha Pb) v + Pb a
//                         - (3 Phi + 2 alpha Pa + 2 (beta + alpha^2) Pb) r)]
//   dL/dv = mu [Jb - 6 alpha Sb + q^2 ((Pa + 2 alpha Pb) r + 2 Pb v)]
//   dL/da = mu [Sb + q^2 Pb r]
//   dL/dm_j = q^3 Phi,
// from dmu/dr = -3 mu q^2 r, dalpha/dr = q^2 (v - 2 alpha r),
// dalpha/dv = q^2 r, dbeta/dr = q^2 (a + 2 alpha v - 2 (beta + alpha^2) r),
// dbeta/dv = 2 q^2 (v + alpha r), dbeta/da = q^2 r.
// Particle k receives -dL/d(r, v, a) of every pair where it is i (with its
// own cotangents) and +dL/d(r, v, a) and dL/dm of every pair where it is j
// (with the other particle's cotangents).  `lanes` consecutive threads own
// k and visit every l once between them (every lanes-th l of each tile);
// their sums are combined by a fixed-order butterfly of warp shuffles, so
// no atomics are needed and the result does not depend on scheduling.  The
// lanes keep small systems from leaving most SMs idle (one thread per k
// would give 64 blocks for 8192 particles).
#include <algorithm>

#include "nb_device.cuh"
#include "nb_internal.cuh"
#include "nb_sym.cuh"

namespace {

using namespace nbk;

constexpr int kAdjThreads = 128;
constexpr int kAdjTile = 64;

// -3 alpha, -6 alpha and -3 beta of a pair.
struct PairFactors {
    double na3, na6, nb3;
};

// The bracket B(g) of dL/d(r, v, a) = q^3 B(g) for a pair with unit source
// mass (mu = m_j q^3 factored out), linear in the cotangents g; phi = Phi(g).
// Doublings go by the exponent, off the FP64 pipe (twice).
__device__ __forceinline__ void bracket_from_phi(const double (&r)[3], const double (&v)[3], const double (&a)[3],
                                                 double q2, double al, double be, const PairFactors &k, double phi,
                                                 const double *g, double (&br)[3], double (&bv)[3], double (&ba)[3])
{
    const double *Ab = g, *Jb = g + 3, *Sb = g + 6;
    const double c18 = fma(k.na3, k.na6, k.nb3);  // 18 alpha^2 - 3 beta
    double sr = 0, sv = 0, jr = 0;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        sr = fma(Sb[d], r[d], sr);
        sv = fma(Sb[d], v[d], sv);
        jr = fma(Jb[d], r[d], jr);
    }
    const double Pa = -3.0 * (jr + twice(fma(k.na6, sr, sv)));
    const double Pb = -3.0 * sr, Pb2 = twice(Pb);
    const double cv = fma(k.na6, sr, Pa);
    const double ncr = -fma(3.0, phi, twice(fma(al, Pa, fma(al, al, be) * Pb)));
    const double qPb = q2 * Pb;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const double Pr = fma(c18, Sb[d], fma(k.na3, Jb[d], Ab[d]));
        br[d] = fma(q2, fma(cv, v[d], fma(Pb, a[d], ncr * r[d])), Pr);
        bv[d] = fma(q2, fma(cv, r[d], Pb2 * v[d]), fma(k.na6, Sb[d], Jb[d]));
        ba[d] = fma(qPb, r[d], Sb[d]);
    }
}

// For particle k and every l: the pair (i = k, j = l) with k's cotangents and
// source mass m_l, and the pair (i = l, j = k) with l's cotangents and source
// mass m_k.  Negating r, v, a negates u, w, Phi and the bracket's
// coefficients, so the second pair's gradient with respect to x_k equals the
// first pair's form evaluated at (r, v, a) with l's cotangents; by linearity
// both roles need one bracket with g* = m_k g_l - m_l g_k, times q^3.  The mass
// gradient of m_k is -q^3 Phi(g_l).  For l = k, g* and Phi are zero; the rounding of
// m_k g_k that the fused g* leaves must not meet q^3 = eps^-3.
__global__ void __launch_bounds__(kAdjThreads) adjoint_kernel(int n, int lanes, const double *__restrict__ m,
                                                              const double *__restrict__ x,
                                                              const double *__restrict__ v,
                                                              const double *__restrict__ a,
                                                              const double *__restrict__ gA,
                                                              const double *__restrict__ gJ,
                                                              const double *__restrict__ gS, double eps2,
                                                              double *__restrict__ gx, double *__restrict__ gv,
                                                              double *__restrict__ ga, double *__restrict__ gm)
{
    __shared__ double s_st[kAdjTile][10];  // x, v, a, m
    __shared__ double s_g[kAdjTile][9];    // cotangents
    const int slot = threadIdx.x / lanes, lj = threadIdx.x - slot * lanes;
    const int k = blockIdx.x * (blockDim.x / lanes) + slot;
    const bool valid = k < n;
    const int kk = valid ? k : 0;
    double xk[3], vk[3], ak[3], gk[9];
    for (int d = 0; d < 3; ++d) {
        xk[d] = x[3 * kk + d];
        vk[d] = v[3 * kk + d];
        ak[d] = a[3 * kk + d];
        gk[d] = gA[3 * kk + d];
        gk[3 + d] = gJ[3 * kk + d];
        gk[6 + d] = gS[3 * kk + d];
    }
    const double mk = m[kk];
    double ox[3] = {0, 0, 0}, ov[3] = {0, 0, 0}, oa[3] = {0, 0, 0}, om = 0.0;
    for (int l0 = 0; l0 < n; l0 += kAdjTile) {
        __syncthreads();
        for (int e = threadIdx.x; e < kAdjTile; e += blockDim.x) {
            const int l = l0 + e;
            const bool ok = l < n;
            const int ll = ok ? l : 0;
            for (int d = 0; d < 3; ++d) {
                s_st[e][d] = x[3 * ll + d];
                s_st[e][3 + d] = v[3 * ll + d];
                s_st[e][6 + d] = a[3 * ll + d];
                s_g[e][d] = ok ? gA[3 * ll + d] : 0.0;
                s_g[e][3 + d] = ok ? gJ[3 * ll + d] : 0.0;
                s_g[e][6 + d] = ok ? gS[3 * ll + d] : 0.0;
            }
            s_st[e][9] = ok ? m[ll] : 0.0;
        }
        __syncthreads();
        const int len = min(kAdjTile, n - l0);
        for (int e = lj; e < len; e += lanes) {
            double r[3], vr[3], ar[3];
            for (int d = 0; d < 3; ++d) {
                r[d] = s_st[e][d] - xk[d];
                vr[d] = s_st[e][3 + d] - vk[d];
                ar[d] = s_st[e][6 + d] - ak[d];
            }
            const double R = fma(r[0], r[0], fma(r[1], r[1], fma(r[2], r[2], eps2)));
            const double q = nbk::rsqrt_fp64(R);
            const double q2 = q * q, q3 = l0 + e == k ? 0.0 : q * q2;
            const double al = fma(r[0], vr[0], fma(r[1], vr[1], r[2] * vr[2])) * q2;
            const double be = fma(fma(vr[0], vr[0], fma(vr[1], vr[1], vr[2] * vr[2])) +
                                      fma(r[0], ar[0], fma(r[1], ar[1], r[2] * ar[2])),
                                  q2, al * al);
            const double na3 = -3.0 * al;
            const PairFactors f = {na3, twice(na3), -3.0 * be};
            double u[3], w[3];
            for (int d = 0; d < 3; ++d) {
                u[d] = fma(f.na3, r[d], vr[d]);
                w[d] = fma(f.na6, u[d], fma(f.nb3, r[d], ar[d]));
            }
            const double ml = s_st[e][9];
            double gs[9];
            double phil = 0.0;
            for (int q9 = 0; q9 < 9; ++q9)
                gs[q9] = fma(mk, s_g[e][q9], -ml * gk[q9]);
            for (int d = 0; d < 3; ++d)
                phil = fma(s_g[e][d], r[d], fma(s_g[e][3 + d], u[d], fma(s_g[e][6 + d], w[d], phil)));
            double br[3], bv[3], ba[3], phi = 0.0;
            for (int d = 0; d < 3; ++d)
                phi = fma(gs[d], r[d], fma(gs[3 + d], u[d], fma(gs[6 + d], w[d], phi)));
            bracket_from_phi(r, vr, ar, q2, al, be, f, phi, gs, br, bv, ba);
            for (int d = 0; d < 3; ++d) {
                ox[d] = fma(q3, br[d], ox[d]);
                ov[d] = fma(q3, bv[d], ov[d]);
                oa[d] = fma(q3, ba[d], oa[d]);
            }
            om = fma(-q3, phil, om);
        }
    }
    for (int off = lanes >> 1; off > 0; off >>= 1) {
        for (int d = 0; d < 3; ++d) {
            ox[d] += __shfl_xor_sync(0xffffffffu, ox[d], off);
            ov[d] += __shfl_xor_sync(0xffffffffu, ov[d], off);
            oa[d] += __shfl_xor_sync(0xffffffffu, oa[d], off);
        }
        om += __shfl_xor_sync(0xffffffffu, om, off);
    }
    if (valid && lj == 0) {
        for (int d = 0; d < 3; ++d) {
            gx[3 * k + d] = ox[d];
            gv[3 * k + d] = ov[d];
            ga[3 * k + d] = oa[d];
        }
        gm[k] = om;
    }
}

// The same gradients with each unordered pair {k, l} taken once (the scheme of
// k_sym.cu): the bracket of g* = m_k g_l - m_l g_k is the gradient with respect
// to x_k, v_k, a_k and, negated, that with respect to x_l, v_l, a_l (swapping the
// two negates g* and r, v, a, and the bracket with them), and Phi(g*) =
// m_k Phi(g_l) - m_l Phi(g_k) comes from the two forms that the mass gradients
// need.  About 150 FP64 operations per unordered pair instead of 2 x 140.
// Bound by the FP64 pipe (87 % of 2 operations per clock and SM); the tile
// shrinks with W for small systems.
// Ordered kernel -> this one: 1000 particles 326 -> 195 us,
// 4096 4.47 -> 2.37 ms, 8192 17.8 -> 9.35 ms.
template <int W>
__global__ void __launch_bounds__(32 * W) adjoint_sym_kernel(SymArgs a, const double *__restrict__ m,
                                                             const double *__restrict__ x,
                                                             const double *__restrict__ v,
                                                             const double *__restrict__ ac,
                                                             const double *__restrict__ gA,
                                                             const double *__restrict__ gJ,
                                                             const double *__restrict__ gS)
{
    constexpr int TH = 32 * W, NV = 10;
    __shared__ double tile[19][TH];  // x, v, a, m, cotangents
    __shared__ double jacc[NV][TH];  // gradients with respect to x, v, a, m
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const SymJob<TH, TH, NV> job(a);
    const int k = job.b * TH + tid;
    double st[9], gk[9], mk;
    auto fetch = [&](int l, double (&s)[9], double (&g)[9], double &ms) {
        const int c = min(l, a.n - 1);  // beyond the end: the last particle without mass and cotangents
        const bool ok = l < a.n;
        for (int d = 0; d < 3; ++d) {
            s[d] = x[3 * static_cast<size_t>(c) + d];
            s[3 + d] = v[3 * static_cast<size_t>(c) + d];
            s[6 + d] = ac[3 * static_cast<size_t>(c) + d];
            g[d] = ok ? gA[3 * static_cast<size_t>(c) + d] : 0.0;
            g[3 + d] = ok ? gJ[3 * static_cast<size_t>(c) + d] : 0.0;
            g[6 + d] = ok ? gS[3 * static_cast<size_t>(c) + d] : 0.0;
        }
        ms = ok ? m[c] : 0.0;
    };
    fetch(k, st, gk, mk);
    double acc[NV], ok[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        acc[q] = ok[q] = 0.0;
        jacc[q][tid] = 0.0;
    }
    for (int it = 0; it < job.nit; ++it) {
        const int j0 = job.start(a, it);
        const bool self = job.offset(it) == 0;  // the tile with itself: ordered pairs
        __syncthreads();
        {
            double ls[9], lg[9], lm;
            fetch(j0 + tid, ls, lg, lm);
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                tile[q][tid] = ls[q];
                tile[10 + q][tid] = lg[q];
            }
            tile[9][tid] = lm;
        }
        __syncthreads();
        for (int sg = 0; sg < W; ++sg) {
            const int sub = ((sg + w) & (W - 1)) * 32;
            double ol[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q)
                ol[q] = 0.0;
#pragma unroll 1
            for (int step = 0; step < 32; ++step) {
                const int e = sub + ((lane + step) & 31);
                double r[3], vr[3], ar[3];
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    r[d] = tile[d][e] - st[d];
                    vr[d] = tile[3 + d][e] - st[3 + d];
                    ar[d] = tile[6 + d][e] - st[6 + d];
                }
                const double R = fma(r[0], r[0], fma(r[1], r[1], fma(r[2], r[2], a.eps2)));
                const double q = nbk::rsqrt_fp64(R);
                const double q2 = q * q;
                const double q3 = self && j0 + e == k ? 0.0 : q * q2;
                const double al = fma(r[0], vr[0], fma(r[1], vr[1], r[2] * vr[2])) * q2;
                const double be = fma(fma(vr[0], vr[0], fma(vr[1], vr[1], vr[2] * vr[2])) +
                                          fma(r[0], ar[0], fma(r[1], ar[1], r[2] * ar[2])),
                                      q2, al * al);
                const double ml = tile[9][e];
                const double na3 = -3.0 * al;
                const PairFactors f = {na3, twice(na3), -3.0 * be};
                double u[3], ww[3], gs[9];
                double phil = 0.0, phik = 0.0;
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    u[d] = fma(f.na3, r[d], vr[d]);
                    ww[d] = fma(f.na6, u[d], fma(f.nb3, r[d], ar[d]));
                    const double g0 = tile[10 + d][e], g1 = tile[13 + d][e], g2 = tile[16 + d][e];
                    phil = fma(g0, r[d], fma(g1, u[d], fma(g2, ww[d], phil)));
                    phik = fma(gk[d], r[d], fma(gk[3 + d], u[d], fma(gk[6 + d], ww[d], phik)));
                    gs[d] = fma(mk, g0, -ml * gk[d]);
                    gs[3 + d] = fma(mk, g1, -ml * gk[3 + d]);
                    gs[6 + d] = fma(mk, g2, -ml * gk[6 + d]);
                }
                double br[3], bv[3], ba[3];
                bracket_from_phi(r, vr, ar, q2, al, be, f, fma(mk, phil, -ml * phik), gs, br, bv, ba);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    ok[d] = fma(q3, br[d], ok[d]);
                    ok[3 + d] = fma(q3, bv[d], ok[3 + d]);
                    ok[6 + d] = fma(q3, ba[d], ok[6 + d]);
                    ol[d] = fma(-q3, br[d], ol[d]);
                    ol[3 + d] = fma(-q3, bv[d], ol[3 + d]);
                    ol[6 + d] = fma(-q3, ba[d], ol[6 + d]);
                }
                ok[9] = fma(-q3, phil, ok[9]);
                ol[9] = fma(q3, phik, ol[9]);
#pragma unroll
                for (int c = 0; c < NV; ++c)
                    ol[c] = __shfl_sync(0xffffffffu, ol[c], lane + 1);
            }
#pragma unroll
            for (int c = 0; c < NV; ++c)
                jacc[c][sub + lane] += ol[c];
            __syncthreads();
        }
        double *out = static_cast<double *>(a.pj) + job.jslot(a, it) + tid;
#pragma unroll
        for (int c = 0; c < NV; ++c) {
            acc[c] += ok[c];
            ok[c] = 0.0;
            if (!self)
                out[c * a.ns] = jacc[c][tid];
            jacc[c][tid] = 0.0;
        }
    }
    double *out = static_cast<double *>(a.pi) + job.islot(a) + k;
#pragma unroll
    for (int c = 0; c < NV; ++c)
        out[c * a.ns] = acc[c];
}

// gx, gv, ga [n][3] and gm [n] (+)= the slots of a batch of offsets.
__global__ void __launch_bounds__(256) adjoint_fold_kernel(SymArgs a, int nslots, int upper, int B, double *gx,
                                                           double *gv, double *ga, double *gm, int first)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x, c = blockIdx.y;
    if (p >= a.n)
        return;
    const double s = fold_slots<Fold64, 10>(static_cast<const double *>(a.pi), nslots, upper,
                                            static_cast<const double *>(a.pj), a.d0, a.d1, a.ns, a.tiles, B, c, p);
    double *o = c == 9 ? gm + p : (c < 3 ? gx : c < 6 ? gv : ga) + 3 * static_cast<size_t>(p) + c % 3;
    *o = first ? s : *o + s;
}

constexpr SymShape kAdjShapes[] = {{128, 128, 80, 22.0, 1.05}, {64, 64, 80, 21.5, 2.1}, {32, 32, 80, 21.0, 4.2}};
// Number of SMs that the workspace sizes and plans of the stateless entry
// points assume, so that they depend on n alone (GB300).
constexpr int kPlanSms = 152;
constexpr int64_t kAdjSymMin = 700;

__global__ void pack_records(int n, const double *m, const double *x, const double *v, const double *a,
                             double2 *rec, int32_t *iota)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n)
        return;
    const size_t N = static_cast<size_t>(n);
    rec[i] = make_double2(x[3 * i], x[3 * i + 1]);
    rec[N + i] = make_double2(x[3 * i + 2], m[i]);
    rec[2 * N + i] = make_double2(v[3 * i], v[3 * i + 1]);
    rec[3 * N + i] = make_double2(v[3 * i + 2], a[3 * i]);
    rec[4 * N + i] = make_double2(a[3 * i + 1], a[3 * i + 2]);
    iota[i] = i;
}

__global__ void unpack_rows(int n, const double *sums, double *acc, double *jerk, double *snap)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= 3 * n)
        return;
    const int i = e / 3, d = e - 3 * i;
    const size_t N = static_cast<size_t>(n);
    acc[e] = sums[(0 + d) * N + i];
    jerk[e] = sums[(3 + d) * N + i];
    snap[e] = sums[(6 + d) * N + i];
}

size_t align256(size_t b) { return (b + 255) / 256 * 256; }

}  // namespace

// FP64 evaluation kernel entry for the stateless path (k_eval.cu).
cudaError_t nb_launch_eval_fp64_rows(const double2 *rec, int n, const int32_t *act, double *out,
                                     double eps2, nb_ctl *ctl, cudaStream_t stream, int sm_count);

extern "C" {

// Workspace of nb_pairs_fp64: the records, then the ordinary kernel's list, the
// sums and the control word, then the slots of the pairwise plan.
struct PairsWork {
    size_t list, sums, ctl, slots, bytes;
    SymPlan plan;
    bool sym;
};

static PairsWork pairs_work(int64_t n)
{
    const size_t N = static_cast<size_t>(n);
    PairsWork w;
    w.list = align256(5 * N * sizeof(double2));
    w.sums = w.list + align256(N * sizeof(int32_t));
    w.ctl = w.sums + align256(9 * N * sizeof(double));
    w.slots = w.ctl + align256(sizeof(nb_ctl));
    // from about 900 particles (k_sym.cu), as long as the slots stay within
    // what a plan may use
    if (n >= 900 && n <= (1LL << 26))
        w.plan = nb_sym_plan(NB_FP64, n, kPlanSms);
    w.sym = w.plan.bytes > 0 && static_cast<double>(w.plan.bytes) <= kSymSlotBytes;
    w.bytes = w.slots + (w.sym ? align256(w.plan.bytes) : 0);
    return w;
}

size_t nb_pairs_workspace_bytes(int64_t n)
{
    return n < 1 ? 0 : pairs_work(n).bytes;
}

nb_status nb_pairs_fp64(int64_t n, const double *m, const double *x, const double *v, const double *a,
                        double eps, double *acc, double *jerk, double *snap, void *work, void *stream)
{
    if (n < 1 || n > (1LL << 26) || !m || !x || !v || !a || !acc || !jerk || !snap || !work ||
        !(eps >= 0x1p-60) || !(eps <= 1e18)) {
        nb_set_thread_error("nb_pairs_fp64: invalid argument");
        return NB_EINVAL;
    }
    const int nn = static_cast<int>(n);
    const PairsWork pw = pairs_work(n);
    unsigned char *w = static_cast<unsigned char *>(work);
    double2 *rec = reinterpret_cast<double2 *>(w);
    int32_t *iota = reinterpret_cast<int32_t *>(w + pw.list);
    double *sums = reinterpret_cast<double *>(w + pw.sums);
    nb_ctl *ctl = reinterpret_cast<nb_ctl *>(w + pw.ctl);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int dev = 0, sms = 0, launches = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess && !pw.sym)
        e = cudaMemsetAsync(ctl, 0, sizeof(nb_ctl), s);
    if (e == cudaSuccess) {
        pack_records<<<(nn + 255) / 256, 256, 0, s>>>(nn, m, x, v, a, rec, iota);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess)
        e = pw.sym ? nb_launch_sym(NB_FP64, pw.plan, rec, static_cast<size_t>(nn), nn, eps * eps, false, w + pw.slots, sums,
                                   static_cast<size_t>(nn), false, s, &launches)
                   : nb_launch_eval_fp64_rows(rec, nn, iota, sums, eps * eps, ctl, s, sms);
    if (e == cudaSuccess) {
        unpack_rows<<<(3 * nn + 255) / 256, 256, 0, s>>>(nn, sums, acc, jerk, snap);
        e = cudaGetLastError();
    }
    if (e != cudaSuccess) {
        nb_set_thread_error(cudaGetErrorString(e));
        return NB_ECUDA;
    }
    return NB_OK;
}

// The pairwise plan of the adjoint; used from about 700 particles on and while
// its slots stay within what a plan may use.
static bool adjoint_plan(int64_t n, SymPlan &plan)
{
    plan = SymPlan();
    if (n < kAdjSymMin || n > (1LL << 26))
        return false;
    for (int q = 0; q < 3; ++q)
        nb_sym_plan_shape(kAdjShapes[q], q, n, kPlanSms, plan);
    return static_cast<double>(plan.bytes) <= kSymSlotBytes;
}

size_t nb_pairs_adjoint_workspace_bytes(int64_t n)
{
    SymPlan plan;
    return adjoint_plan(n, plan) ? align256(plan.bytes) : 0;
}

nb_status nb_pairs_fp64_adjoint_work(int64_t n, const double *m, const double *x, const double *v, const double *a,
                                     double eps, const double *gacc, const double *gjerk, const double *gsnap,
                                     double *gx, double *gv, double *ga, double *gm, void *work, void *stream)
{
    SymPlan pl;
    if (!work || !adjoint_plan(n, pl))
        return nb_pairs_fp64_adjoint(n, m, x, v, a, eps, gacc, gjerk, gsnap, gx, gv, ga, gm, stream);
    if (!m || !x || !v || !a || !gacc || !gjerk || !gsnap || !gx || !gv || !ga || !gm || !(eps >= 0x1p-60) ||
        !(eps <= 1e18)) {
        nb_set_thread_error("nb_pairs_fp64_adjoint_work: invalid argument");
        return NB_EINVAL;
    }
    const SymShape &kd = kAdjShapes[pl.kind];
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    SymArgs arg;
    arg.jb = nullptr;
    arg.np = 0;
    arg.n = static_cast<int>(n);
    arg.tiles = pl.T;
    arg.k = pl.k;
    arg.parts = pl.parts;
    arg.eps2 = eps * eps;
    arg.ns = pl.ns;
    arg.pi = work;
    arg.pj = static_cast<unsigned char *>(work) + pl.pi_slots * pl.ns * kd.bytes;
    const int D = pl.T / 2 + 1;
    for (int d0 = 0; d0 < D; d0 += pl.nd) {
        arg.d0 = d0;
        arg.d1 = std::min(D, d0 + pl.nd);
        const int64_t jobs = sym_jobs(pl.T, arg.d0, arg.d1, pl.k);
        const int groups = (arg.d1 - arg.d0 + pl.k - 1) / pl.k;
        auto run = [&](auto kernel) {
            kernel<<<static_cast<unsigned>(jobs), kd.threads, 0, s>>>(arg, m, x, v, a, gacc, gjerk, gsnap);
        };
        if (pl.kind == 0) run(adjoint_sym_kernel<4>);
        else if (pl.kind == 1) run(adjoint_sym_kernel<2>);
        else run(adjoint_sym_kernel<1>);
        adjoint_fold_kernel<<<dim3((arg.n + 255) / 256, 10), 256, 0, s>>>(
            arg, groups, static_cast<int>(jobs / pl.T), kd.tile, gx, gv, ga, gm, d0 == 0);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
        nb_set_thread_error(cudaGetErrorString(e));
        return NB_ECUDA;
    }
    return NB_OK;
}

nb_status nb_pairs_fp64_adjoint(int64_t n, const double *m, const double *x, const double *v,
                                const double *a, double eps, const double *gacc, const double *gjerk,
                                const double *gsnap, double *gx, double *gv, double *ga, double *gm,
                                void *stream)
{
    if (n < 1 || n > (1LL << 26) || !m || !x || !v || !a || !gacc || !gjerk || !gsnap || !gx || !gv ||
        !ga || !gm || !(eps >= 0x1p-60) || !(eps <= 1e18)) {
        nb_set_thread_error("nb_pairs_fp64_adjoint: invalid argument");
        return NB_EINVAL;
    }
    const int nn = static_cast<int>(n);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess)
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) {
        nb_set_thread_error(cudaGetErrorString(e));
        return NB_ECUDA;
    }
    // lanes per particle: the fewest that give every SM at least four blocks
    int lanes = 1;
    while (lanes < 32 && (static_cast<int64_t>(nn) * lanes + kAdjThreads - 1) / kAdjThreads < 4 * sms)
        lanes *= 2;
    const int per_block = kAdjThreads / lanes;
    adjoint_kernel<<<(nn + per_block - 1) / per_block, kAdjThreads, 0, s>>>(
        nn, lanes, m, x, v, a, gacc, gjerk, gsnap, eps * eps, gx, gv, ga, gm);
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        nb_set_thread_error(cudaGetErrorString(e));
        return NB_ECUDA;
    }
    return NB_OK;
}

}  // extern "C"
