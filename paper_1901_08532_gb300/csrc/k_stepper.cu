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
// 39.2 -> 18.1 us, EX N = 8192 46.1 -> 21.3 us, mixed N = 65536 58.0 -> 31.6 us.
// It returns to the host when the next active set holds more than
// kStepSmall particles, which it leaves listed (the host then runs that step
// with the tuned evaluation kernels and needs no scheduler pass, about 28 us),
// when the next block time passes t_end, or after an error flag.  Every block
// takes the same branch at every barrier (decisions come from the same global
// values), and no block waits on a flag.
#include <cooperative_groups.h>

#include <algorithm>

#include "nb_block.cuh"
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
// 38.5 / 31.6; FP64 N = 1024 with 8 and 16 particles per block 18.1 and 19.4; the
// EX figures without the lanes' FP64 join, 0.6 us).
constexpr int kSliceFp64 = 8, kSliceFp32 = 16, kSliceWide = 96;
constexpr int kChunkCap = 1024;  // j-records per shared-memory chunk

struct StepOut {
    int64_t steps;     // block steps taken by the launch
    int64_t act_sum;   // active particles summed over those steps
    int32_t reason;    // 0: next block time beyond t_end, 1: next active set too large, 2: error
    int32_t n_act;     // active count of the last step taken
    double t_last;     // time of the last step taken
    double t_next;     // reason 1: time of the next step and its active count
    int32_t n_next;
};

struct StepArgs {
    int n;
    double *st, *t, *dt;
    const double *m;
    double eps2, eta, dt_min, dt_max, dt_shared, t_end, noise;
    int drop_lo;        // single-precision control: positions without their low part
    unsigned long long *bmin;  // [B] per-block earliest t_i + dt_i, as time_key()
    int *bcnt;          // [B] particles reaching it
    int *cand;          // [B][kStepSmall] their indices, ascending
    double *part;       // [kStepSmall][9][B] partial sums
    int32_t *act;       // active set of the last step taken
    int32_t *act_next;  // reason 1: the next active set, ascending
    nb_ctl *ctl;
    StepOut *out;
    double *log_t;      // per-step log (device), entries [log_base, log_cap)
    int64_t *log_n;
    int64_t log_cap, log_base;
};

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
    int reason = 0, last_n = 0, next_n = 0;
    double last_t = 0.0, next_t = 0.0;
    for (;;) {
        // schedule: this block's earliest t_i + dt_i, the particles reaching it
        unsigned long long mt = ~0ull;
        int ct = 0;
        for (int i = c0; i < c1; ++i) {
            const unsigned long long tt = time_key(a.t[i] + a.dt[i]);
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
                if (time_key(a.t[i] + a.dt[i]) == mb)
                    a.cand[bk * kStepSmall + pos++] = i;
        }
        if (tid == 0) {
            a.bmin[bk] = mb;
            a.bcnt[bk] = tot_b;
        }
        grid.sync();
        // the same decision in every block: thread tid looks at the blocks
        // kQ tid .. kQ tid + kQ - 1
        unsigned long long bm[kQ], mn_key = ~0ull;
        int bc[kQ];
#pragma unroll
        for (int e = 0; e < kQ; ++e) {
            const int q = tid * kQ + e;
            bm[e] = q < B ? __ldcg(&a.bmin[q]) : ~0ull;
            bc[e] = q < B ? __ldcg(&a.bcnt[q]) : 0;
            mn_key = bm[e] < mn_key ? bm[e] : mn_key;
        }
        const int err = *reinterpret_cast<volatile int *>(&a.ctl->err);
        mn_key = block_min_u64(mn_key, red_u);
        const double mn = time_of(mn_key);
        int c = 0;
#pragma unroll
        for (int e = 0; e < kQ; ++e)
            c += bm[e] == mn_key ? bc[e] : 0;
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
            // too many for a step here: list them for the host's
            reason = 1;
            __syncthreads();  // red_i was read by the scan
#pragma unroll
            for (int e = 0, q = pos; e < kQ; ++e) {
                if (tid * kQ + e == bk)
                    red_i[0] = q;
                q += bm[e] == mn_key ? bc[e] : 0;
            }
            __syncthreads();
            if (mine > 0 && mb == mn_key) {
                int at = red_i[0] + ex;
                for (int i = c0; i < c1; ++i)
                    if (time_key(a.t[i] + a.dt[i]) == mb)
                        a.act_next[at++] = i;
            }
            next_t = mn;
            next_n = total;
            break;
        }
        // active list, ascending: blocks in order, each block's list in order
#pragma unroll
        for (int e = 0; e < kQ; ++e)
            if (bm[e] == mn_key)
                for (int u = 0; u < bc[e]; ++u)
                    s_act[pos++] = (tid * kQ + e) * kStepSmall + u;
        __syncthreads();
        if (tid < total)
            s_act[tid] = __ldcg(&a.cand[s_act[tid]]);
        __syncthreads();
        eval_slice<PR>(PredictedRecord<PR>{{a.st, a.t, a.m, static_cast<size_t>(a.n), a.drop_lo}, mn}, a.eps2, lo, hi, total,
                       s_act, s_rec, kStepSmall, a.part + bk, B, s_red, smem, kChunkCap, T);
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
        a.out->t_next = next_t;
        a.out->n_next = next_n;
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

// One launch of the device-resident stepper; reports what it did in *r
// (synchronises the stream).  reason 1 leaves the next active set in
// c->act_next.
cudaError_t nb_run_stepper(nb_ctx *c, double t_end, int64_t log_cap, int64_t log_base, StepperResult *r)
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
    a.act_next = c->act_next;
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
    *r = {o->steps, o->act_sum, o->reason, o->n_act, o->t_last, o->t_next, o->n_next};
    return cudaSuccess;
}
