// Evaluation by unordered pairs: the job split, the partial-sum slots and their
// fold, shared by the force kernels (k_sym.cu) and the pair adjoint
// (k_adjoint.cu).  The scheme is described in k_sym.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "nb_internal.cuh"

namespace nbk {

struct SymArgs {
    const void *jb;  // predicted particles (the evaluation buffer's rows)
    size_t np;       // row stride
    int n;
    int tiles;       // T
    int d0, d1;      // offsets of this launch, [d0, d1)
    int k;           // offsets per block
    int parts;       // H, parts of a j-tile
    double eps2;
    void *pi, *pj;   // partial sums: [group * H + h][NV][ns], [d - d0][NV][ns]
    size_t ns;       // T * B
};

// Is offset d evaluated from tile b (for even T the last offset only from the
// lower half)?
__host__ __device__ __forceinline__ bool sym_job(int T, int b, int d) { return 2 * d != T || b < T / 2; }

// What a block does: part h of the jobs (tile b, offsets of group g), as nit
// j-tiles of SUB particles, with NV sums per particle.  The last group of an even T may be launched for
// the lower half of the tiles only.
template <int B, int SUB, int NV = 9>
struct SymJob {
    int b, da, part, subs, nit;
    __device__ __forceinline__ explicit SymJob(const SymArgs &a)
    {
        b = blockIdx.x / a.parts % a.tiles;
        da = a.d0 + blockIdx.x / a.parts / a.tiles * a.k;
        const int db = min(a.d1, da + a.k);
        subs = B / SUB / a.parts;
        part = blockIdx.x % a.parts * subs * SUB;
        nit = max(0, (sym_job(a.tiles, b, db - 1) ? db : db - 1) - da) * subs;
    }
    __device__ __forceinline__ int offset(int it) const { return da + it / subs; }
    __device__ __forceinline__ int start(const SymArgs &a, int it) const  // first particle of j-tile it
    {
        const int c = b + offset(it);
        return (c >= a.tiles ? c - a.tiles : c) * B + part + it % subs * SUB;
    }
    __device__ __forceinline__ size_t jslot(const SymArgs &a, int it) const
    {
        return static_cast<size_t>(offset(it) - a.d0) * NV * a.ns + start(a, it);
    }
    __device__ __forceinline__ size_t islot(const SymArgs &a) const
    {
        return static_cast<size_t>(blockIdx.x / a.parts / a.tiles * a.parts + blockIdx.x % a.parts) * NV * a.ns;
    }
};

// FP64 slots enter a compensated total (the rounding errors of a plain chain over
// the T slots would exceed those of the ordinary kernel's sums: at 30000
// particles 2.3e-16 of sum_j |A_ij| RMS against 0.7e-16).
struct Fold64 {
    using Part = double;
    double s = 0.0, e = 0.0;
    __device__ __forceinline__ void add(double v)
    {
        const double t = s + v, b = t - s;
        e += (s - (t - b)) + (v - b);
        s = t;
    }
    __device__ __forceinline__ double total() const
    {
        const double r = s + e;
        return isnan(r) ? s : r;  // an infinite sum leaves no error term
    }
};

template <class F, int U>
__device__ __forceinline__ void add_all(F &f, const typename F::Part (&v)[U])
{
#pragma unroll
    for (int u = 0; u < U; ++u)
        f.add(v[u]);
}
template <int U>
__device__ __forceinline__ void add_all(Fold64 &f, const double (&v)[U])
{
    // pairwise among themselves, compensated into the total
    double t[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
        t[u] = v[u];
#pragma unroll
    for (int h = U / 2; h > 0; h /= 2)
#pragma unroll
        for (int u = 0; u < h; ++u)
            t[u] += t[u + h];
    f.add(t[0]);
}

// Total over slots of value q (of NV) of particle p: the i-slots in order, then
// the j-slots in order of the offset.
template <class F, int NV>
__device__ __forceinline__ double fold_slots(const typename F::Part *pi, int nslots, int upper,
                                             const typename F::Part *pj, int d0, int d1, size_t ns, int T, int B,
                                             int q, int p)
{
    constexpr int U = 8;  // slots in flight
    F f;
    const size_t step = NV * ns;
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
        add_all(f, v);
    }
    for (; s < nslots; ++s)
        f.add(src[s * step]);
    const int db = (2 * (d1 - 1) == T && c < T / 2) ? d1 - 1 : d1;
    src = pj + q * ns + p;
    int d = max(d0, 1);
    for (; d + U <= db; d += U) {
        typename F::Part v[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
            v[u] = src[(d - d0 + u) * step];
        add_all(f, v);
    }
    for (; d < db; ++d)
        f.add(src[(d - d0) * step]);
    return f.total();
}

// Tiles x groups of the offsets [d0, d1), without the upper half of the tiles
// where the last group is the offset T / 2 alone.
inline int64_t sym_jobs(int64_t T, int64_t d0, int64_t d1, int64_t k)
{
    const int64_t groups = (d1 - d0 + k - 1) / k;
    return T * groups - (2 * (d1 - 1) == T && (d1 - d0 - 1) % k == 0 ? T / 2 : 0);
}

}  // namespace nbk

// What a plan needs to know of a kernel: particles per tile, threads, bytes of
// a particle's partial sums, the measured rate with the chip full in
// unordered pairs per microsecond and SM, and the jobs an SM needs for it.
struct SymShape {
    int tile, threads, bytes;
    double rate, fill;
};

// k_sym.cu: best becomes the plan for this kernel where that is faster.
void nb_sym_plan_shape(const SymShape &kd, int kind, int64_t n, int sms, SymPlan &best, size_t max_bytes = 0);
