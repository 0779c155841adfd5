// Internal declarations of libnb: the context, device helpers shared by the
// kernels (TMA bulk copies, bounded mbarrier waits, FP64 reciprocal square
// root, TwoSum), and the launch functions of each kernel file.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "nb.h"

// ------------------------------------------------------------------ layout
//
// State (FP64, structure of arrays, component-major, stride n):
//   st[(F * 3 + k) * n + i] for field F in {X, V, A, J, S, C}, component k.
// Evaluation buffers written by the predictor (stride n):
//   FP64:  jb64[c * n + i], c = 0..4: (x, y) (z, m) (vx, vy) (vz, ax) (ay, az)
//   mixed: jf32[c * npad + i], 13 float rows c = 0..12:
//          xh yh zh m xl yl zl vx vy vz ax ay az, with xh = fp32(x) and
//          xl = fp32(x - xh); npad = n rounded up to a multiple of 4, the
//          padding rows hold zero-mass particles (contribute exactly 0).
// Evaluation output (stride ostride): out[q * ostride + k], q = 0..8 for
//   acc x,y,z, jerk x,y,z, snap x,y,z of the k-th listed particle.
enum { F_X = 0, F_V = 1, F_A = 2, F_J = 3, F_S = 4, F_C = 5, NFIELD = 6 };

// Evaluations that use the FP32 row buffer and the packed FP32 kernel.
inline bool nb_fp32_eval(int precision) { return precision == NB_MIXED || precision == NB_SP; }
// FP32 rows per particle of the predicted j-buffer (0: FP64 records).
inline int nb_jrows(int precision)
{
    return precision == NB_EX ? 20 : (nb_fp32_eval(precision) ? 13 : 0);
}

struct nb_ctl {                      // small device control block
    unsigned long long tnext_key;    // min over i of (t_i + dt_i), as time_key()
    int32_t n_act;                   // active count from the scheduler
    int32_t err;                     // bit flags, see NB_ERR_*
    int64_t floor_hits;              // steps clamped at dt_min
};
#define NB_ERR_NONFINITE 1
#define NB_ERR_TIMEOUT 2

// Evaluation of a complete active set with each unordered pair once (k_sym.cu).
// Launch plan for n particles: the kernel (kind), T tiles, k offsets per block, j-tiles in
// `parts`, nd offsets per launch, row length ns and number of the i-slots,
// workspace bytes, estimated time.
struct SymPlan {
    double us = 1e300;
    int kind = 0, T = 0, k = 1, parts = 1, nd = 1;
    size_t ns = 0, pi_slots = 0, bytes = 0;
};
// Bytes of partial sums that a plan may use where it needs more than the two
// slots (72 B per particle each) of the smallest one: 24 slots, at least
// 256 MB, at most 1 GB.  Every context holds them, so a program with many middle-
// sized ones pays for them many times: at least 512 MB made mixed sums of 65536
// to 150000 particles 0-5 % faster (65536 4.84 ms with 418 MB, 5.06 with 209 MB) and
// those of 262144 3 % slower; 2 GB at most would gain 1 % from 131072 particles on.
constexpr double kSymSlotBytes = 1e9, kSymMinBytes = 256e6, kSymSlots = 24.0;

struct nb_ctx {
    int dev = 0;
    cudaStream_t stream = nullptr;
    nb_config cfg{};
    int64_t n = 0;
    double eps = 0;
    int sm_count = 0;

    double *m = nullptr;       // [n]
    double *st = nullptr;      // [18][n]
    double *t = nullptr;       // [n]
    double *dt = nullptr;      // [n]
    double2 *jb64 = nullptr;   // [5][n]
    float *jf32 = nullptr;     // [13][npad]
    int64_t npad = 0;
    int32_t *act = nullptr;    // [n] active set of the last step evaluated
    int32_t *act_next = nullptr;  // [n] active set found by the scheduler, swapped in by the step
    double *anew = nullptr;    // [9][n]
    double *stage = nullptr;   // [3][n][3] output staging
    double *part = nullptr;    // split-j partials
    size_t part_cap = 0;       // doubles
    unsigned *tile_cnt = nullptr;
    size_t tile_cnt_cap = 0;
    std::vector<void *> outgrown;  // earlier, smaller blocks of part and tile_cnt
    SymPlan sym_plan;          // evaluation of all particles, each pair once
    bool sym_use = false;
    bool light = false;        // no mass is above 1
    void *sym_work = nullptr;  // its partial sums
    int32_t *blk = nullptr;    // scheduler block counts
    double *red = nullptr;     // reduction scratch
    size_t red_cap = 0;        // doubles
    nb_ctl *ctl = nullptr;     // device
    nb_ctl *ctl_h = nullptr;   // pinned host mirror
    double *diag = nullptr;    // [8] device results of energy / angmom
    double *diag_h = nullptr;  // [8] pinned host mirror
    double *ring = nullptr;    // [ring_cap][8] diagnostics samples of nb_run_diag
    int64_t ring_cap = 0;
    // device-resident stepper (k_stepper.cu): per-block scratch, results, log
    double *stp_bmin = nullptr;
    int *stp_bcnt = nullptr, *stp_cand = nullptr;
    double *stp_part = nullptr;
    void *stp_out = nullptr, *stp_out_h = nullptr;
    double *stp_log_t = nullptr;
    int64_t *stp_log_n = nullptr;

    int64_t n_act = 0;         // size of the last evaluated set
    bool have_pred = false;
    double t_pred = 0;
    bool have_eval = false;
    double t_eval = 0;
    double t_sys = 0;          // min t_i after the last block step (host copy)
    int64_t launches = 0;
    double interactions = 0;
    int32_t inject = 0;        // one-shot fault injection for tests (nb_inject_fault)
    bool dead = false;
    std::string err;
};

// --------------------------------------------------------- device helpers

namespace nbk {

// Key of a time that orders, as an unsigned integer, like the time itself (the
// bits of a double alone do so from 0 on only; a state may hold negative
// times), on the integer pipe; one to one.  ~0 is the key of a NaN, behind
// every time.
__device__ __forceinline__ unsigned long long time_key(double t)
{
    const long long b = __double_as_longlong(t);
    return static_cast<unsigned long long>(b) ^ (static_cast<unsigned long long>(b >> 63) | 1ull << 63);
}
__host__ __device__ constexpr unsigned long long time_key_bits(unsigned long long key)
{
    return key ^ (key >> 63 ? 1ull << 63 : ~0ull);
}
__device__ __forceinline__ double time_of(unsigned long long key)
{
    return __longlong_as_double(static_cast<long long>(time_key_bits(key)));
}

__device__ __forceinline__ unsigned long long globaltimer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

// 1-D TMA bulk copy global -> shared, completion signalled on bar.
// dst, src 16-byte aligned; bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    asm volatile(
        "cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, "
        "p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

// Wait for phase `parity` of bar to complete, giving up after limit_ns of
// wall-clock time (globaltimer).  Returns false on timeout.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity,
                                                  unsigned long long limit_ns)
{
    if (mbar_test(bar, parity))
        return true;
    const unsigned long long t0 = globaltimer_ns();
    while (!mbar_test(bar, parity)) {
        if (globaltimer_ns() - t0 > limit_ns)
            return false;
    }
    return true;
}

constexpr unsigned long long kWaitLimitNs = 1000000000ull;  // 1 s

// Reciprocal square root of a positive normal double in three FP64 operations
// (the FP64 pipe runs at 1/64 of FP32 here; an FP32 seed alone takes five for a
// third-order step).  x = m 4^k with m in [1, 4); y = the FP32 hardware estimate
// of 1/sqrt(m); its residual r = 1 - m y^2 in FP32 (y^2 exactly as a pair, m as
// a pair) gives the correction y r / 2, added to y's bits as an integer and
// rounded to 26 bits: y0, within 2^-26.  Then y0^2 is exact (also where it is
// subnormal, x > 2^1022: y0 is a multiple of 2^-26 2^-k there), h = 1 - x y0^2
// rounds once, and y = y0 + (y0 / 2)(1 + 3 h / 4) h, the series of
// (1 - h)^(-1/2) to h^2 (what is left is below 2^-75), rounds once more: the
// factor 1 + 3 h / 4 goes into the bits of y0 / 2 as an integer too.
// Valid for all positive normal x; relative error within 1.0 x 2^-53, rms 0.43.
// Against the five-operation form: 8191 particles in FP64 3.87 -> 3.73 ms, the
// energy of 131072 186 -> 153 ms.
__device__ __forceinline__ double rsqrt_fp64(double x)
{
    const unsigned hi = static_cast<unsigned>(__double2hiint(x)), lo = static_cast<unsigned>(__double2loint(x));
    const unsigned odd = ~(hi >> 20) & 1u;  // of the unbiased exponent (bias 1023)
    // m = mh + ml, mh the leading 24 bits
    const float mh = __uint_as_float(((hi & 0xfffffu) << 3 | lo >> 29) + ((127u + odd) << 23));
    const float ml = static_cast<float>(lo & 0x1fffffffu) * (odd ? 0x1p-51f : 0x1p-52f);
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(mh));
    y = fmaxf(fminf(y, 0x1.fffffep-1f), 0.5f);  // one binade, [1/2, 1): units of 2^-24
    const float p = __fmul_rn(y, y), e = __fmaf_rn(y, y, -p);
    const float r = __fmaf_rn(-ml, p, __fmaf_rn(-mh, e, __fmaf_rn(-mh, p, 1.0f)));
    // y + y r / 2 in units of 2^-26: four per unit of y
    const int c = __float2int_rn(__fmul_rn(__fmul_rn(y, r), 0x1p25f));
    const unsigned yb = __float_as_uint(y);
    long long bits = (static_cast<long long>((yb >> 3) + (896u << 20)) << 32 | static_cast<long long>(yb << 29)) +
                     static_cast<long long>(c) * (1ll << 27);
    // exponent: y0 = y 2^-k, k = (E - odd) / 2 with E the unbiased exponent
    bits -= static_cast<long long>((static_cast<int>(hi >> 20) - 1023 - static_cast<int>(odd)) / 2) * (1ll << 52);
    const double y0 = __longlong_as_double(bits);
    const double h = fma(-x, y0 * y0, 1.0);
    // |h| 2^53 as a float from h's bits (0 where h is too small to matter)
    const int hh = __double2hiint(h);
    const unsigned sh = 1023u - ((static_cast<unsigned>(hh) >> 20) & 0x7ff);  // |h| = 1.f 2^-sh
    const float hm = __uint_as_float((static_cast<unsigned>(hh) & 0xfffffu) << 3 | 127u << 23);  // 1.f
    const float hs = sh < 64u ? __fmul_rn(hm, __uint_as_float((127u + 53u - sh) << 23)) : 0.0f;   // |h| 2^53
    const int d = __float2int_rn(__fmul_rn(__fmul_rn(y, 0.75f), hs));
    const double half = __longlong_as_double(bits - (1ll << 52) + (hh < 0 ? -d : d));
    return fma(half, h, y0);
}

// 2 x by the exponent, off the FP64 pipe.
__device__ __forceinline__ double twice(double x)
{
    const int hi = __double2hiint(x);
    if (static_cast<unsigned>((hi & 0x7ff00000) - 0x00100000) >= 0x7fd00000u)
        return x + x;  // zero, subnormal, the largest, infinite, NaN
    return __hiloint2double(hi + 0x00100000, __double2loint(x));
}

// TwoSum (Knuth): s + e == a + b exactly.  Accumulates the rounding error
// of hi + p into lo.
__device__ __forceinline__ void two_sum_acc(float &hi, float &lo, float p)
{
    const float s = __fadd_rn(hi, p);
    const float bp = __fsub_rn(s, hi);
    const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(p, bp));
    hi = s;
    lo = __fadd_rn(lo, e);
}

}  // namespace nbk

// ------------------------------------------------------- launch functions

struct EvalLaunch {
    const int32_t *act;  // device list of n_act indices
    int n_act;
    double *out;         // [9][ostride]
    int ostride;
    nb_tiles tiles;      // resolved
    int64_t j0 = 0, j1 = -1;  // j-range [j0, j1) of the evaluation buffer; j1 < 0: all of it
};

// k_eval.cu
cudaError_t nb_launch_eval(nb_ctx *c, const EvalLaunch &L);
// j_count: length of the j-range evaluated (0: the whole buffer)
// *us: the estimated time
nb_tiles nb_auto_tiles(const nb_ctx *c, int64_t n_act, const nb_tiles &req, int64_t j_count = 0,
                       double *us = nullptr);
cudaError_t nb_eval_smem_setup();
// k_sym.cu
// max_bytes: of partial sums that there are (0: as many as a context's own plan may use)
SymPlan nb_sym_plan(int precision, int64_t n, int sms, size_t max_bytes = 0);
cudaError_t nb_sym_smem_setup();
// jb, np: predicted particles and row stride; light: no mass is above 1 (FP64: of
// no effect); work: plan.bytes of device memory, 256-byte aligned; out
// [9][ostride], added to where `add`; *launches counts kernels.
cudaError_t nb_launch_sym(int precision, const SymPlan &plan, const void *jb, size_t np, int n, double eps2,
                          bool light, void *work, double *out, size_t ostride, bool add, cudaStream_t stream,
                          int *launches);
// k_predict.cu
cudaError_t nb_launch_predict(nb_ctx *c, double t);
// The same into active-first order: rows [0, n_act) are the particles of the
// ascending list act, the others follow in ascending order; rows[k] = k.
cudaError_t nb_launch_predict_front(nb_ctx *c, double t, const int32_t *act, int n_act, int32_t *rows);
// k_correct.cu
cudaError_t nb_launch_correct(nb_ctx *c, double t1, int n_act);
cudaError_t nb_launch_init_state(nb_ctx *c, int pass);
// anew rows q0 .. q0 + 2 -> dst [n_act][3]; all three sums where wanted (NULL: not)
cudaError_t nb_launch_transpose_out(nb_ctx *c, int n_act, int q0, double *dst);
cudaError_t nb_launch_outputs(nb_ctx *c, int n_act, double *acc, double *jerk, double *snap);
cudaError_t nb_launch_rows_to_soa(nb_ctx *c, const double *rows, int field);
cudaError_t nb_launch_soa_to_rows(nb_ctx *c, int field, double *rows);
// k_sched.cu
cudaError_t nb_launch_schedule(nb_ctx *c);
cudaError_t nb_launch_iota(nb_ctx *c, int n, int32_t *dst);
// nb_api.cu: message returned by nb_last_error(NULL) on this thread
void nb_set_thread_error(const char *msg);
// k_stepper.cu
struct StepperResult {
    int64_t steps, act_sum;  // block steps taken and the active particles summed over them
    int reason;              // 0: t_end reached, 1: next active set too large, 2: error flag
    int n_act;               // active count and time of the last step taken
    double t_last;
    double t_next;           // reason 1: time and active count of the next step
    int n_next;
};
cudaError_t nb_run_stepper(nb_ctx *c, double t_end, int64_t log_cap, int64_t log_base, StepperResult *r);

// k_energy.cu
cudaError_t nb_launch_energy(nb_ctx *c, double *ek_pe_dev);
cudaError_t nb_launch_angmom(nb_ctx *c, double *l4_dev);
// k_kappa.cu: condition numbers sum_j |A_ij|, |J_ij|, |S_ij| of the listed
// particles against the predicted j-buffer, out_dev [3][n_act].
cudaError_t nb_launch_kappa(nb_ctx *c, const int32_t *act_dev, int n_act, double *out_dev);
