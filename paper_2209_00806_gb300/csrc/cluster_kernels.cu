// Cluster-resident time stepping for small samples (TBPM_VARIANT_CLUSTER).
//
// A small sample -- the 64 x 64 graphene DOS workload has 8192 rows -- fits, with
// psi0, psi and the two Clenshaw buffers, in the shared memory of one thread-block
// cluster of 16 blocks (8 where the device runs no larger one).  All time steps of
// the propagation then run in one launch, one cluster per state: each block holds a
// contiguous range of rows, gathers x from the owning block's shared memory
// (distributed shared memory across the cluster), and a cluster barrier separates
// the Clenshaw terms (Sec. 2.2, Eq. psi_t).  FP64 takes a row a thread, up to
// 16 x 1024 rows; FP32 up to eight rows a thread, 16 x 4096 rows with three slots a
// row and 16 x 1024 otherwise.  Real values, at most kClusterMaxW entries per row.
// The closing term's sums of <psi0|phi> and <phi|phi> are formed per block in a
// fixed tree after the block has arrived at the term's barrier (no later term
// needs them), and added over the blocks in a fixed tree by block 0 two barriers
// later (FP64 throughout, or float pairs up to the block; deterministic).  Per row
// the arithmetic and its order are those of the plain term kernel, so the states
// equal the per-term launches' bit for bit; the launch cost of 15 kernels per step
// is gone.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <string>
#include <vector>

#include "tbpm_internal.cuh"

namespace cg = cooperative_groups;

namespace tbpm {
namespace {

// Address of `p` (this block's shared memory) in the shared::cluster
// window of block `rank`, and a 16-byte load through that window.
__device__ __forceinline__ uint32_t cluster_addr(const void *p, int rank)
{
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}

__device__ __forceinline__ double2 ld_cluster(uint32_t addr)
{
    double2 v;
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(addr));
    return v;
}

constexpr uint32_t kNoEntry = 0xffffffffu;

// Sums of three values over a warp (lane l: v0, v1, v2 of row l) by a tree that
// halves the values held as it doubles the lanes summed: six FP64 adds a warp
// where a butterfly per value takes fifteen, each 64 cycles of the FP64 pipe.
// Lane 0 returns the sum of v0, lane 16 that of v1, lane 8 that of v2.
__device__ __forceinline__ double warp_sum3(double v0, double v1, double v2)
{
    const int l = threadIdx.x & 31;
    const bool hi = l & 16, q = l & 8;
    // lanes 0-15 keep (v0, v2), lanes 16-31 keep (v1, nothing)
    const double s0 = hi ? v0 : v1, s1 = hi ? v2 : 0.0;          // sent to lane ^ 16
    double a = (hi ? v1 : v0) + __shfl_xor_sync(0xffffffffu, s0, 16);
    double b = (hi ? 0.0 : v2) + __shfl_xor_sync(0xffffffffu, s1, 16);
    // of those, lanes with bit 3 clear keep a, the others b
    a = (q ? b : a) + __shfl_xor_sync(0xffffffffu, q ? a : b, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}
// the lane of value v in the result
__device__ __forceinline__ int sum3_lane(int v) { return v == 0 ? 0 : v == 1 ? 16 : 8; }

// MAXW: the widest row the launch allows (its gather addresses stay in
// registers): 3 when every row has three slots (graphene), else 4 or
// kClusterMaxW.  M: the matrix form.  What a form lacks is not in its kernel:
// a conditional FP64 operation costs its 64 cycles of the pipe executed or
// not, and the FP64 pipes of the cluster's SMs set the time.  64 x 64 graphene
// executed 14 FP64 instructions a row and term for 8, 15 more a row and
// step for the sums and 96 in sequence on one warp: 31.4 us a step, 22.0 now
// (25 with a diagonal, 31 with values per entry).
template <int MAXW, int MAXT, Vals M>
__global__ void __launch_bounds__(MAXT, 1) k_cluster_steps(ClusterArgs a)
{
    constexpr bool ONE = one_value(M);
    cg::cluster_group cl = cg::this_cluster();
    const int K = (int)cl.num_blocks();
    const int rank = (int)cl.block_rank();
    const ClusterState me = a.states[blockIdx.x / K];        // one cluster a state
    const int R = a.rows_per_cta;
    const int t = threadIdx.x;
    const int64_t r = (int64_t)rank * R + t;
    extern __shared__ __align__(16) unsigned char sm[];
    double2 *vec = reinterpret_cast<double2 *>(sm);                  // [4][R]
    int32_t *ent = reinterpret_cast<int32_t *>(vec + 4 * R);         // [W][R] owner << 16 | local
    double *sval = reinterpret_cast<double *>(ent + a.max_w * R);    // [W][R] (general values)
    __shared__ double part[2][3];
    __shared__ double red[32][3];
    __shared__ FusedTerm tab[3 * kClusterMaxTerms];

    for (int i = t; i < 3 * a.J; i += blockDim.x)
        tab[i] = a.terms[(i / a.J) * kMaxTerms + i % a.J];
    // this row's entries, as (owning block, local row) pairs
    int w;
    int64_t base;
    if (MAXW == 3 || a.fixed_width) {
        w = MAXW == 3 ? 3 : a.fixed_width;
        base = (r / kSliceRows) * (kSliceRows * (int64_t)w) + r % kSliceRows;
    } else {
        const int64_t q = r / kSliceRows;
        base = a.slice_ptr[q] + r % kSliceRows;
        w = (int)((a.slice_ptr[q + 1] - a.slice_ptr[q]) / kSliceRows);
    }
    for (int k = 0; k < w; ++k) {
        const int32_t c = a.col[base + (int64_t)k * kSliceRows];
        ent[k * R + t] = c == (int32_t)r && ONE ? -1 : ((c / R) << 16) | (c % R);
        if (!ONE) sval[k * R + t] = a.val[base + (int64_t)k * kSliceRows];
    }
    const double d = a.diag[r];
    const double d2 = d + d;                 // 2 d, exact: gamma d of the interior terms
    // gamma d of a step's first term (the same in the three tables)
    const double d_first = M == kOne ? a.terms[0].gamma * d : 0.0;
    vec[t] = reinterpret_cast<const double2 *>(me.psi0)[r * me.B];
    for (int b = 0; b < 3; ++b)
        vec[(1 + b) * R + t] = b == a.cur0 ? reinterpret_cast<const double2 *>(me.bufs[b])[r * me.B]
                                           : make_double2(0.0, 0.0);
    cl.sync();
    // gathered entries' shared::cluster addresses in x buffer 0 (a buffer
    // is R rows further on), fixed for the launch; kNoEntry for padding
    // (one-value form)
    uint32_t gsrc[MAXW];
#pragma unroll
    for (int k = 0; k < MAXW; ++k) {
        gsrc[k] = kNoEntry;
        if (MAXW == 3 || k < w) {
            const int32_t e = ent[k * R + t];
            if (e >= 0) gsrc[k] = cluster_addr(vec + (e & 0xffff), e >> 16);
        }
    }

    int cur = a.cur0;
    bool pending = false;                    // a cluster barrier arrived at, not yet waited on
    // a step whose block parts await block 0's sum, and the barrier waits
    // until they are all written: the closing term's own barrier completes
    // before the blocks write their parts, the next one after
    int sum_step = 0, sum_waits = 0;
    // block 0, warp 0: lane k loads block k's parts of step m, added in a fixed
    // tree; C_m, the norm and the drift checks
    auto cluster_sum = [&](int m) {
        double w0 = 0.0, w1 = 0.0, w2 = 0.0;
        if (t < K) {
            const double *pk = cl.map_shared_rank(&part[m & 1][0], t);
            w0 = pk[0];
            w1 = pk[1];
            w2 = pk[2];
        }
        const double v = warp_sum3(w0, w1, w2);
        const double sm0 = v, sm1 = __shfl_sync(0xffffffffu, v, sum3_lane(1));
        const double sm2 = __shfl_sync(0xffffffffu, v, sum3_lane(2));
        if (t == 0) {
            me.corr[m] = make_double2(sm0, sm1);
            me.norms[m] = sm2;
            const double ref = *me.norm_ref;
            const double drift = ref > 0.0 ? fabs(sm2 / ref - 1.0) : sm2;
            if (!(sm2 == sm2) || !(sm0 == sm0) || !(sm1 == sm1) || sm2 - sm2 != 0.0)
                atomicOr(a.err, 2);
            else if (drift > a.hard_bound)
                atomicOr(a.err, 1);
        }
    };
    for (int n = 1; n <= a.n_steps; ++n) {
        const FusedTerm *tt = tab + cur * a.J;
        for (int j = 0; j < a.J; ++j) {
            const FusedTerm tm = tt[j];
            const int xb = 1 + (tm.x < 0 ? cur : tm.x);
            // own-row operands (written only by this thread) before the wait
            const double2 p = vec[(1 + cur) * R + t];
            double2 zz = make_double2(0.0, 0.0);
            if (tm.z >= 0) zz = vec[(1 + tm.z) * R + t];
            const int xoff = xb * R;
            const uint32_t xoff_b = (uint32_t)xoff * (uint32_t)sizeof(double2);
            double2 o;
            // one-value form: its first product, fma(c, psi, z), needs nothing
            // of this term's x, so it runs before the barrier wait
            double re = 0.0, im = 0.0;
            if (ONE) {
                re = fma(tm.c_hi, p.x, zz.x);
                im = fma(tm.c_hi, p.y, zz.y);
            }
            if (pending) cl.barrier_wait();      // the gathered vector is complete
            pending = false;
            if (sum_waits > 0 && --sum_waits == 0 && rank == 0 && t < 32) cluster_sum(sum_step);
            if constexpr (ONE) {
                // the one-value form of the per-term kernels: neighbours summed
                // in stored order (padding only after a row's entries), then
                // fma(gh, s, fma(gd, x_r, fma(c, psi, z)))
                double2 sm = make_double2(0.0, 0.0);
                if (gsrc[0] != kNoEntry) sm = ld_cluster(gsrc[0] + xoff_b);
#pragma unroll
                for (int k = 1; k < MAXW; ++k) {
                    if ((MAXW == 3 || k < w) && gsrc[k] != kNoEntry) {
                        const double2 x = ld_cluster(gsrc[k] + xoff_b);
                        sm.x += x.x;
                        sm.y += x.y;
                    }
                }
                if constexpr (M == kOne) {
                    const double gd = tm.gd_sel == 2 ? xor_sign(d2, tm.gd_sign)
                                    : tm.gd_sel == 1 ? xor_sign(d, tm.gd_sign)
                                                     : d_first;
                    const double2 xo = vec[xoff + t];
                    re = fma(gd, xo.y, re);
                    im = fma(-gd, xo.x, im);
                }
                o.x = fma(tm.gh, sm.y, re);
                o.y = fma(-tm.gh, sm.x, im);
            } else {
                // y = H~ x in the plain kernel's order: diagonal, then the entries
                double2 y = vec[xoff + t];
                y.x *= d;
                y.y *= d;
#pragma unroll
                for (int k = 0; k < MAXW; ++k) {
                    if (MAXW == 3 || k < w) {
                        const double h = sval[k * R + t];
                        const double2 x = ld_cluster(gsrc[k] + xoff_b);
                        y.x = fma(h, x.x, y.x);
                        y.y = fma(h, x.y, y.y);
                    }
                }
                re = fma(tm.gamma, y.y, zz.x);
                im = fma(-tm.gamma, y.x, zz.y);
                o.x = fma(tm.c_hi, p.x, re);
                o.y = fma(tm.c_hi, p.y, im);
            }
            vec[(1 + tm.out) * R + t] = o;
            cl.barrier_arrive();                 // release this term's writes
            pending = true;
            if (tm.final_term) {
                // the step's sums, off the critical path: nothing of the next
                // terms needs them, so they are formed while the other blocks
                // reach the barrier; block 0 adds the blocks' parts two
                // barriers on (part is double-buffered by step parity)
                const double2 p0 = vec[t];
                double v0 = fma(p0.x, o.x, p0.y * o.y);
                double v1 = fma(p0.x, o.y, -(p0.y * o.x));
                double v2 = fma(o.x, o.x, o.y * o.y);
                const int lane = t % 32;
                const double v = warp_sum3(v0, v1, v2);
                if (lane % 8 == 0 && lane < 24) red[t / 32][lane == 0 ? 0 : lane == 16 ? 1 : 2] = v;
                __syncthreads();
                if (t < 32) {               // the warps' sums, in a fixed tree
                    const int nq = (R + 31) / 32;
                    double w0 = 0.0, w1 = 0.0, w2 = 0.0;
                    if (t < nq) {
                        w0 = red[t][0];
                        w1 = red[t][1];
                        w2 = red[t][2];
                    }
                    const double u = warp_sum3(w0, w1, w2);
                    if (t % 8 == 0 && t < 24) part[n & 1][t == 0 ? 0 : t == 16 ? 1 : 2] = u;
                }
                sum_step = n;
                sum_waits = 2;
            }
        }
        cur = a.next_cur[cur];
    }
    // the last step's parts: its closing barrier, one more, then block 0 adds them
    if (pending) {
        cl.barrier_wait();
        if (sum_waits > 0) --sum_waits;
    }
    pending = false;
    if (sum_waits > 0) {
        cl.sync();
        if (rank == 0 && t < 32) cluster_sum(sum_step);
    }
    reinterpret_cast<double2 *>(me.bufs[cur])[r * me.B] = vec[(1 + cur) * R + t];
    cl.sync();                                           // no block leaves while others read it
}

// ---- FP32 ----------------------------------------------------------------------
__device__ __forceinline__ float2 ld_cluster_f(uint32_t addr)
{
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr));
    return v;
}
__device__ __forceinline__ FF ff_shfl(FF v, int o)
{
    return FF{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
// warp_sum3 of float pairs
__device__ __forceinline__ FF warp_sum3(FF v0, FF v1, FF v2)
{
    const int l = threadIdx.x & 31;
    const bool hi = l & 16, q = l & 8;
    const FF zero = {0.f, 0.f};
    FF a = ff_add(hi ? v1 : v0, ff_shfl(hi ? v0 : v1, 16));
    const FF b = ff_add(hi ? zero : v2, ff_shfl(hi ? v2 : zero, 16));
    a = ff_add(q ? b : a, ff_shfl(q ? a : b, 8));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) a = ff_add(a, ff_shfl(a, o));
    return a;
}

// The FP32 form of the stepping: states and arithmetic those of the per-term
// FP32 kernels (bit-identical), RPT rows a thread (rows t, t + T, ...), the
// closing sums as float pairs up to the block and FP64 from there.  The
// norm carry: a state whose norm has drifted past the bound after step m starts
// step m + 1 rescaled, as with the per-term kernels.  Step m's sums are known
// while step m + 1 runs, so it is run once more from its start, which is still
// in its buffer, with the factor: one step more per rescaling (64 x 64 graphene
// drifts 8e-9 a step: one in 1,300 at the default bound).  A state that drifts
// past the bound in the step after a rescaling has a bound within a step's
// rounding and would run every step twice: the launch ends there with error bit
// 8, and the caller repeats the run with the per-term kernels.  4,096 steps at
// the default bound: 9.8 us a step at 64 x 64 and 25 us at 180 x 180 (repeated
// whole by the per-term kernels: 51 and 70 us).  Bound by the latency of a term
// (barrier, distributed shared-memory gathers): 64 x 64 graphene, one state, 10 us
// a step against 42 us of dependent launches; 180 x 180 25 against 47 us.
template <int MAXW, int RPT, Vals M>
__global__ void __launch_bounds__(512, 1) k_cluster_steps_f32(ClusterArgs a)
{
    cg::cluster_group cl = cg::this_cluster();
    const int K = (int)cl.num_blocks();
    const int rank = (int)cl.block_rank();
    const ClusterState me = a.states[blockIdx.x / K];
    const int R = a.rows_per_cta, T = blockDim.x, t = threadIdx.x;
    extern __shared__ __align__(16) unsigned char sm[];
    float2 *vec = reinterpret_cast<float2 *>(sm);                    // [4][R]
    float *sval = reinterpret_cast<float *>(vec + 4 * R);            // [W][R] (value per entry)
    __shared__ double part[2][3];
    __shared__ FF red[32][3];
    __shared__ FusedTerm tab[3 * kClusterMaxTerms];
    __shared__ float rescale;        // block 0 -> every block: factor, kStop, or 0
    __shared__ int start;            // buffer of the last step's starting state
    __shared__ int scaled;           // (block 0) the last step that called for a factor
    constexpr float kStop = -1.f;
    if (t == 0) {
        rescale = 0.f;
        scaled = -1;
    }
    for (int i = t; i < 3 * a.J; i += T) tab[i] = a.terms[(i / a.J) * kMaxTerms + i % a.J];

    uint32_t gsrc[RPT][MAXW];
    float d[RPT];
    int w[RPT];
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
        const int row = t + i * T;
        w[i] = 0;
        d[i] = 0.f;
#pragma unroll
        for (int k = 0; k < MAXW; ++k) gsrc[i][k] = kNoEntry;
        if (row >= R) continue;
        const int64_t r = (int64_t)rank * R + row;
        const int64_t q = r / kSliceRows;
        int64_t base;
        if (MAXW == 3) {
            w[i] = 3;
            base = q * (3 * kSliceRows) + r % kSliceRows;
        } else {
            base = a.slice_ptr[q] + r % kSliceRows;
            w[i] = (int)((a.slice_ptr[q + 1] - a.slice_ptr[q]) / kSliceRows);
        }
        d[i] = a.diag32[r];
#pragma unroll
        for (int k = 0; k < MAXW; ++k)
            if (k < w[i]) {
                const int32_t c = a.col[base + (int64_t)k * kSliceRows];
                // one value: padding (own row) adds nothing; else its value is zero
                if (M != kOne || c != (int32_t)r) gsrc[i][k] = cluster_addr(vec + c % R, c / R);
                if (M != kOne) sval[k * R + row] = a.val32[base + (int64_t)k * kSliceRows];
            }
        vec[row] = reinterpret_cast<const float2 *>(me.psi0)[r * me.B];
        for (int b = 0; b < 3; ++b)
            vec[(1 + b) * R + row] = b == a.cur0 ? reinterpret_cast<const float2 *>(me.bufs[b])[r * me.B]
                                                 : make_float2(0.f, 0.f);
    }
    cl.sync();

    int cur = a.cur0;
    bool pending = false;
    int sum_step = 0, sum_waits = 0;         // as in the FP64 kernel
    auto cluster_sum = [&](int m) {
        double w0 = 0.0, w1 = 0.0, w2 = 0.0;
        if (t < K) {
            const double *pk = cl.map_shared_rank(&part[m & 1][0], t);
            w0 = pk[0];
            w1 = pk[1];
            w2 = pk[2];
        }
        const double v = warp_sum3(w0, w1, w2);
        const double sm1 = __shfl_sync(0xffffffffu, v, sum3_lane(1));
        const double sm2 = __shfl_sync(0xffffffffu, v, sum3_lane(2));
        if (t == 0) {
            me.corr[m] = make_double2(v, sm1);
            me.norms[m] = sm2;
            const double ref = *me.norm_ref;
            const double drift = ref > 0.0 ? fabs(sm2 / ref - 1.0) : sm2;
            if (!(sm2 == sm2) || !(v == v) || !(sm1 == sm1) || sm2 - sm2 != 0.0) atomicOr(a.err, 2);
            else if (drift > a.hard_bound) atomicOr(a.err, 1);
            if (drift > a.renorm_bound && sm2 > 0.0 && ref > 0.0 && sm2 - sm2 == 0.0) {
                atomicAdd(a.renorm_count, 1ull);
                if (m < a.n_steps) {
                    const bool again = m == scaled + 1;
                    if (again) atomicOr(a.err, 8);
                    scaled = m;
                    const float f = again ? kStop : (float)sqrt(ref / sm2);
                    for (int k = 0; k < K; ++k) *cl.map_shared_rank(&rescale, k) = f;
                }
            }
        }
    };
    auto next_vector = [&]() {
        if (!pending) return;
        cl.barrier_wait();                   // the gathered vector is complete
        pending = false;
        if (sum_waits > 0 && --sum_waits == 0 && rank == 0 && t < 32) cluster_sum(sum_step);
    };
    for (int n = 1;; ++n) {
        if (pending) {                       // (the sums come a barrier later)
            cl.barrier_wait();
            pending = false;
            --sum_waits;
        }
        // step n - 2's factor, written before the barrier just passed: the same
        // for every thread of the cluster
        const float f = *(volatile float *)&rescale;
        if (f > 0.f) {                       // step n - 1 once more, from its rescaled start
            __syncthreads();
            if (t == 0) rescale = 0.f;
            cur = start;
            sum_waits = 0;                   // not the sums of its first run
            --n;
        }
        const float sc = f > 0.f ? f : 1.f;  // of this step's starting state
        if (f < 0.f || n > a.n_steps) break;
        const FusedTerm *tt = tab + cur * a.J;
        for (int j = 0; j < a.J; ++j) {
            const FusedTerm tm = tt[j];
            const int xoff = (1 + (tm.x < 0 ? cur : tm.x)) * R;
            const uint32_t xoff_b = (uint32_t)xoff * (uint32_t)sizeof(float2);
            // the factors without branches among the rows' loads and gathers, which would
            // cost their overlap.  Eight rows a thread are out of registers: with this
            // form, 180 x 180, one value and values per entry, 24.6 and 26.2 us a step
            // (24.3 and 26.2 without a norm carry), with that of fewer rows 25.0 and 26.5
            const float scx = (RPT < 8 ? tm.x < 0 : j == 0) ? sc : 1.f;
            float2 p[RPT], zz[RPT];          // own rows: written only by this thread
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const int row = min(t + i * T, R - 1);
                p[i] = vec[(1 + cur) * R + row];
                zz[i] = tm.z >= 0 ? vec[(1 + tm.z) * R + row] : make_float2(0.f, 0.f);
            }
            if (RPT < 8 || sc != 1.f)
#pragma unroll
                for (int i = 0; i < RPT; ++i) {
                    p[i].x *= sc;
                    p[i].y *= sc;
                }
            next_vector();
            FF v0 = {0.f, 0.f}, v1 = v0, v2 = v0;
#pragma unroll
            for (int i = 0; i < RPT; ++i) {
                const int row = min(t + i * T, R - 1);
                const bool in = t + i * T < R;
                float2 x[MAXW];
#pragma unroll
                for (int k = 0; k < MAXW; ++k)
                    if (gsrc[i][k] != kNoEntry) x[k] = ld_cluster_f(gsrc[i][k] + xoff_b);
                float2 y = vec[xoff + row];
                y.x *= d[i];
                y.y *= d[i];
#pragma unroll
                for (int k = 0; k < MAXW; ++k)
                    if (gsrc[i][k] != kNoEntry) {
                        const float h = M == kOne ? a.h_uniform_f : sval[k * R + row];
                        y.x = fmaf(h, x[k].x, y.x);
                        y.y = fmaf(h, x[k].y, y.y);
                    }
                y.x *= scx;
                y.y *= scx;
                float2 o;
                o.x = fmaf(tm.c_hi_f, p[i].x, fmaf(tm.c_lo_f, p[i].x, fmaf(tm.gamma_f, y.y, zz[i].x)));
                o.y = fmaf(tm.c_hi_f, p[i].y, fmaf(tm.c_lo_f, p[i].y, fmaf(-tm.gamma_f, y.x, zz[i].y)));
                if (in) vec[(1 + tm.out) * R + row] = o;
                if (tm.final_term && in) {
                    const float2 p0 = vec[row];
                    FF re, im, nr;
                    ff_dot3(p0.x, p0.y, o.x, o.y, re, im, nr);
                    v0 = ff_add(v0, re);
                    v1 = ff_add(v1, im);
                    v2 = ff_add(v2, nr);
                }
            }
            cl.barrier_arrive();             // release this term's writes
            pending = true;
            if (tm.final_term) {             // the sums, while the other blocks arrive
                const int lane = t % 32;
                const FF v = warp_sum3(v0, v1, v2);
                if (lane % 8 == 0 && lane < 24) red[t / 32][lane == 0 ? 0 : lane == 16 ? 1 : 2] = v;
                __syncthreads();
                if (t < 32) {
                    const FF zero = {0.f, 0.f};
                    const bool has = t < (T + 31) / 32;
                    const FF u = warp_sum3(has ? red[t][0] : zero, has ? red[t][1] : zero,
                                           has ? red[t][2] : zero);
                    if (t % 8 == 0 && t < 24)
                        part[n & 1][t == 0 ? 0 : t == 16 ? 1 : 2] = ff_to_double(u);
                }
                sum_step = n;
                sum_waits = 2;
            }
        }
        if (t == 0) start = cur;
        cur = a.next_cur[cur];
    }
    if (rescale < 0.f) {                     // the caller starts again
        cl.sync();
        return;
    }
    if (sum_waits > 0) {
        cl.sync();
        if (rank == 0 && t < 32) cluster_sum(sum_step);
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i)
        if (t + i * T < R)
            reinterpret_cast<float2 *>(me.bufs[cur])[((int64_t)rank * R + t + i * T) * me.B] =
                vec[(1 + cur) * R + t + i * T];
    cl.sync();                               // no block leaves while others read it
}

}  // namespace

namespace {
constexpr int kClusterSmem = 200 * 1024;     // dynamic shared memory of a block at most
// 16-block clusters (non-portable size) run on this device
bool cluster16()
{
    static const bool ok = [] {
        bool best16 = false;
        if (cudaFuncSetAttribute(k_cluster_steps<kClusterMaxW, 1024, kReal>,
                                 cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute at;
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = 16;
            at.val.clusterDim.y = 1;
            at.val.clusterDim.z = 1;
            cfg.gridDim = dim3(16);
            cfg.blockDim = dim3(512);
            cfg.dynamicSmemBytes = 64 * 1024;
            cfg.attrs = &at;
            cfg.numAttrs = 1;
            int n = 0;
            allow_shared<k_cluster_steps<kClusterMaxW, 1024, kReal>>(kClusterSmem);
            if (cudaOccupancyMaxActiveClusters(&n, k_cluster_steps<kClusterMaxW, 1024, kReal>, &cfg) ==
                    cudaSuccess &&
                n >= 1)
                best16 = true;
        }
        cudaGetLastError();
        return best16;
    }();
    return ok;
}
}  // namespace

int cluster_blocks_for(int64_t n_rows, int max_w, int uniform, int fp32, int fixed_width)
{
    const int rpt = fp32 && fixed_width == 3 ? 4 : 1;        // rows a thread at most
    if (n_rows <= 0 || n_rows > 16 * 1024 * rpt || max_w > kClusterMaxW) return 0;
    auto fits = [&](int K) {
        if (n_rows % K || n_rows / K > 1024 * rpt) return false;
        const int64_t R = n_rows / K;
        const int64_t smem = fp32 ? 4 * R * 8 + (int64_t)std::max(1, max_w) * R * (uniform ? 0 : 4)
                                  : 4 * R * 16 + (int64_t)std::max(1, max_w) * R * (uniform ? 4 : 12);
        return smem <= kClusterSmem;
    };
    // GB300's FP64 rate per SM makes more SMs pay; else 8
    if (cluster16() && fits(16)) return 16;
    return fits(8) ? 8 : 0;
}

// Estimated us a step of 15 products, both ways, fitted to sweeps of lattices of 3
// to 12 entries a row, 1,024 to 65,536 rows, 1 to 16 states, rows in lattice order,
// with the sublattices apart and in random order (the far lines cost 1.2 to
// 2 us a thousand and wave of seven clusters):
//                                      far lines   FP64, cluster / launches   FP32
//   3 entries, 8,192 rows, 1 state        512          27 /  43              12 / 44
//     the same, random order           22,419          52 /  45              47 / 45
//   3 entries, 65,536 rows, 1 state     2,048                                29 / 46
//     the same, sublattices apart      26,624                                66 / 47
//     the same, random order          183,884                               287 / 86
//   8 entries, 4,096 rows, 4 states       896          38 /  82              14 / 50
//     the same, random order           28,465          83 /  81              68 / 56
//     the same, 16 states              28,465         240 / 261             222 / 59
// The slower way is chosen in 20 of the 1,044 points, by 10 % on average (before, every
// point took the cluster: 35 % over all of them).
bool cluster_pays(const BuildOutput &H, int fp32, const std::vector<int> &widths)
{
    const int w = std::max(1, H.max_width);
    const double n = (double)H.n_rows, R = n / 16, far = H.far_lines / 1000.0;
    int S = 0;
    for (int B : widths) S += B;
    const int waves = (S + kClusterStates - 1) / kClusterStates;
    double cluster, launches = 0.0;
    if (fp32) {
        // blocks of fewer than 512 rows share an SM
        const double turns = R < 512 ? std::ceil(S * R / (kClusterStates * 512.0)) : waves;
        cluster = turns * (10.5 + n / 8192) + waves * (w <= 4 ? 1.5 : 1.95) * far;
        for (int B : widths) launches += 38 + 1.4 * w + 0.9 * std::min(B * n / 16384, 16.0);
    } else {
        // the FP64 pipe: more rows a block or states an SM take longer
        const double q = std::pow(R / 512, 1.5), each = S / (double)kClusterStates;
        const double turns = R > 256 ? waves : std::max(1.0, each * (0.2 + R / 270));
        cluster = turns * (w > 4 ? 24 + 44 * q : 16 + 17 * q) +
                  std::max(1.0, each) * (w <= 4 ? 1.15 : 1.55) * far;
        const int rounds = (w + 3) / 4;              // entries in rounds of four
        for (int B : widths) {
            const double x = std::max(0.0, B * n / 1000 - 10);
            launches += H.fixed_width == 3 ? 45 + 0.95 * x
                                           : 42 + 11 * rounds + (0.75 + 1.15 * rounds) * std::min(x, 23.0);
        }
    }
    return cluster <= launches;
}

template <auto k>
cudaError_t launch_cluster(const ClusterArgs &a, int K, int threads, size_t smem, cudaStream_t st)
{
    cudaError_t e = allow_shared<k>(kClusterSmem);
    if (e != cudaSuccess) return e;
    if (K > 8) {
        e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e != cudaSuccess) return e;
    }
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = K;
    at.val.clusterDim.y = 1;
    at.val.clusterDim.z = 1;
    cfg.gridDim = dim3(K * a.n_states);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k, a);
}

template <int MAXW, int MAXT, Vals M>
cudaError_t launch_cluster_t(const ClusterArgs &a, int K, size_t smem, cudaStream_t st)
{
    return launch_cluster<k_cluster_steps<MAXW, MAXT, M>>(a, K, a.rows_per_cta, smem, st);
}

template <int MAXW, int RPT>
cudaError_t launch_cluster_f(const ClusterArgs &a, int K, cudaStream_t st)
{
    const int R = a.rows_per_cta, threads = ((R + RPT - 1) / RPT + 31) / 32 * 32;
    const size_t smem = (size_t)4 * R * sizeof(float2) +
                        (a.uniform ? 0 : (size_t)a.max_w * R * sizeof(float));
    return a.uniform ? launch_cluster<k_cluster_steps_f32<MAXW, RPT, kOne>>(a, K, threads, smem, st)
                     : launch_cluster<k_cluster_steps_f32<MAXW, RPT, kReal>>(a, K, threads, smem, st);
}

template <int MAXW, int MAXT>
cudaError_t launch_cluster_m(const ClusterArgs &a, int K, size_t smem, cudaStream_t st)
{
    if (!a.uniform) return launch_cluster_t<MAXW, MAXT, kReal>(a, K, smem, st);
    return a.zero_diag ? launch_cluster_t<MAXW, MAXT, kOneNoDiag>(a, K, smem, st)
                       : launch_cluster_t<MAXW, MAXT, kOne>(a, K, smem, st);
}
template <int MAXT>
cudaError_t launch_cluster_w(const ClusterArgs &a, int K, size_t smem, cudaStream_t st)
{
    if (a.fixed_width == 3) return launch_cluster_m<3, MAXT>(a, K, smem, st);
    return a.max_w <= 4 ? launch_cluster_m<4, MAXT>(a, K, smem, st)
                        : launch_cluster_m<kClusterMaxW, MAXT>(a, K, smem, st);
}

cudaError_t launch_cluster_steps(const ClusterArgs &a, int fp32, int K, cudaStream_t st)
{
    const int R = a.rows_per_cta;
    if (fp32) {
        // at most 512 threads, 128 registers each, several rows a thread
        if (a.fixed_width != 3)
            return R <= 512 ? launch_cluster_f<kClusterMaxW, 1>(a, K, st)
                            : launch_cluster_f<kClusterMaxW, 2>(a, K, st);
        return R <= 512    ? launch_cluster_f<3, 1>(a, K, st)
               : R <= 1024 ? launch_cluster_f<3, 2>(a, K, st)
               : R <= 2048 ? launch_cluster_f<3, 4>(a, K, st)
                           : launch_cluster_f<3, 8>(a, K, st);
    }
    const size_t smem = (size_t)4 * R * sizeof(double2) + (size_t)a.max_w * R * sizeof(int32_t) +
                        (a.uniform ? 0 : (size_t)a.max_w * R * sizeof(double));
    // up to 512 rows per block: 128 registers a thread, else 64
    return R <= 512 ? launch_cluster_w<512>(a, K, smem, st) : launch_cluster_w<1024>(a, K, smem, st);
}

}  // namespace tbpm
