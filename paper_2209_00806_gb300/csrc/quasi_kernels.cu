// Quasi-eigenstates (Sec. 2.6, Eq. quasi): after every time step of the
// forward run and of the backward run (H -> -H), each state lane adds
// c_{n,k} psi(t_n) to the accumulator of every energy E_k, where
// c_{n,k} = (tau / 2 pi) w_n e^{i E_k t_n} comes from a host table (FP64 and
// FP32 copies) indexed by the step counter the reduction has just advanced
// (graph-safe).  Then the
// accumulators go to the caller's layout and are normalised per energy,
// state and sample.
#include <cuda_runtime.h>
#include <stdint.h>

#include "tbpm_internal.cuh"

namespace tbpm {
namespace {

template <typename V> struct QeC;
template <> struct QeC<double> {
    typedef double2 type;
    __device__ static const double *scale(const QeArgs &a) { return a.scale; }
    __device__ static const void *coef(const QeArgs &a) { return a.coef; }
};
template <> struct QeC<float> {
    typedef float2 type;
    __device__ static const float *scale(const QeArgs &a) { return a.scale_f; }
    __device__ static const void *coef(const QeArgs &a) { return a.coef_f; }
};

// acc is [K][n_rows][S] with this group's lanes at s0 .. s0 + B - 1, in the
// group's precision: FP32 accumulators in the FP32 form (GB300 runs FP64 at a
// small fraction of the FP32 rate; the sum of 2N + 1 windowed terms keeps the
// FP32 states' accuracy), FP64 in the FP64 form.  One thread per N adjacent
// lanes of a row: N = 2 moves 16 bytes an access in FP32 where the lanes and
// the accumulators pair up (even B, S and s0), N = 1 otherwise.  Bound by
// HBM, 2K + 1 accesses of the state: 819,200 rows x 4 FP32 states, K = 4,
// 236 MB, 48 us one lane a thread, 37 us two.
template <typename V, int N> struct alignas(N * 2 * sizeof(V)) QeLanes {
    typename QeC<V>::type c[N];
};
template <typename V, int N>
__global__ void __launch_bounds__(256) k_qe_acc(QeArgs a)
{
    typedef typename QeC<V>::type C;
    typedef QeLanes<V, N> Q;
    dep_launch();
    dep_wait();
    const int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * N;
    if (t >= a.n_rows * a.B) return;
    const int64_t r = t / a.B;
    const int l = (int)(t % a.B);
    const int smp = a.chunk_sample[r / kChunkRows];
    const int n = a.step[smp] - 1;
    Q v = *reinterpret_cast<const Q *>(reinterpret_cast<const C *>(a.psi) + t);
    if (a.scale) {
#pragma unroll
        for (int j = 0; j < N; ++j) {
            const V sc = (V)QeC<V>::scale(a)[(int64_t)smp * a.B + l + j];
            v.c[j].x *= sc;
            v.c[j].y *= sc;
        }
    }
    const C *cf = reinterpret_cast<const C *>(QeC<V>::coef(a)) + (int64_t)n * a.K;
    C *acc = reinterpret_cast<C *>(a.acc) + r * a.S + a.s0 + l;
    const int64_t stride = a.n_rows * a.S;
#pragma unroll 4
    for (int k = 0; k < a.K; ++k) {
        const C c = cf[k];
        Q *q = reinterpret_cast<Q *>(acc + k * stride);
        Q o = *q;
#pragma unroll
        for (int j = 0; j < N; ++j) {
            o.c[j].x = fma(c.x, v.c[j].x, fma(-c.y, v.c[j].y, o.c[j].x));
            o.c[j].y = fma(c.x, v.c[j].y, fma(c.y, v.c[j].x, o.c[j].y));
        }
        *q = o;
    }
}

// Squared norms of the accumulators, per 1024-row chunk (chunks do not
// straddle samples; padding rows are zero): block (chunk, k), thread (row
// part, state) sums rows part, part + P, ... in order, then the parts are
// added in order.  (One block per energy, state and sample left the device
// idle: 637 us at 820,000 rows, 4 x 4 vectors.)
constexpr int kQeThreads = 256;
template <typename V>
__global__ void __launch_bounds__(kQeThreads) k_qe_chunk_norms(const typename QeC<V>::type *acc,
                                                               int S, int64_t n_rows,
                                                               double *partial)
{
    const int P = kQeThreads / S;                  // S <= 64
    const int p = threadIdx.x % S, part = threadIdx.x / S;
    const int64_t chunk = blockIdx.x, k = blockIdx.y;
    const typename QeC<V>::type *v = acc + (k * n_rows + chunk * kChunkRows) * S;
    __shared__ double red[kQeThreads];
    double sum = 0.0;
    if (part < P) {
        for (int row = part; row < kChunkRows; row += P) {
            const typename QeC<V>::type x = v[(int64_t)row * S + p];
            const double re = x.x, im = x.y;       // squares in FP64: no FP32 underflow
            sum = fma(re, re, fma(im, im, sum));
        }
    }
    red[threadIdx.x] = sum;
    __syncthreads();
    if ((int)threadIdx.x < S) {
        double t = red[threadIdx.x];
        for (int q = 1; q < P; ++q) t += red[q * S + threadIdx.x];
        partial[(k * gridDim.x + chunk) * S + threadIdx.x] = t;
    }
}

// Norm of (k, p, sample s) from its chunks, strided per-thread sums then a
// shared-memory tree (fixed order), and the factor that normalises it (1 for
// a zero vector): formed once here, not by a division and a root per element.
__global__ void __launch_bounds__(kQeThreads) k_qe_norms(const double *partial, int S, int n_samples,
                                                         int64_t n_chunks,
                                                         const int64_t *chunk_off, double *norms,
                                                         double *factor)
{
    const int64_t kps = blockIdx.x;            // (k * S + p) * n_samples + s
    const int smp = (int)(kps % n_samples);
    const int64_t kp = kps / n_samples;
    const int p = (int)(kp % S);
    const int64_t k = kp / S;
    double acc = 0.0;
    for (int64_t c = chunk_off[smp] + threadIdx.x; c < chunk_off[smp + 1]; c += kQeThreads)
        acc += partial[(k * n_chunks + c) * S + p];
    __shared__ double red[kQeThreads];
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = kQeThreads / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        norms[kps] = red[0];
        factor[kps] = red[0] > 0.0 ? 1.0 / sqrt(red[0]) : 1.0;
    }
}

// out[k][p][i] = factor acc[k][row(i)][p]
template <typename C>
__global__ void k_qe_store(const C *acc, int K, int S, int64_t n_rows, int64_t n_orb,
                           const int32_t *user_to_row, const int32_t *orb_sample, int n_samples,
                           const double *factor, double2 *out)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n_orb) return;
    const int64_t row = user_to_row[i];
    const int smp = orb_sample[i];
    const int k = blockIdx.y;
    for (int p = 0; p < S; ++p) {
        const C v = acc[((int64_t)k * n_rows + row) * S + p];
        const int64_t kp = (int64_t)k * S + p;
        const double f = factor[kp * n_samples + smp];
        out[kp * n_orb + i] = make_double2(f * (double)v.x, f * (double)v.y);
    }
}

}  // namespace

cudaError_t launch_qe_acc(const QeArgs &a, int fp32, cudaStream_t st)
{
    const bool two = fp32 && a.B % 2 == 0 && a.S % 2 == 0 && a.s0 % 2 == 0;
    const int64_t n = a.n_rows * a.B / (two ? 2 : 1);
    const unsigned blocks = (unsigned)((n + 255) / 256);
    if (two) return launch_dependent(k_qe_acc<float, 2>, blocks, 256, 0, st, a);
    return fp32 ? launch_dependent(k_qe_acc<float, 1>, blocks, 256, 0, st, a)
                : launch_dependent(k_qe_acc<double, 1>, blocks, 256, 0, st, a);
}

cudaError_t launch_qe_finish(const void *acc, int fp32, int K, int S, int64_t n_rows, int64_t n_orb,
                             int n_samples, const int32_t *user_to_row, const int32_t *orb_sample,
                             const int64_t *chunk_off, double *partial, double2 *out, double *norms,
                             double *factor, cudaStream_t st)
{
    const int64_t n_chunks = n_rows / kChunkRows;
    const dim3 cg((unsigned)n_chunks, (unsigned)K);
    const dim3 sg((unsigned)((n_orb + 255) / 256), (unsigned)K);
    const float2 *af = reinterpret_cast<const float2 *>(acc);
    const double2 *ad = reinterpret_cast<const double2 *>(acc);
    if (fp32) k_qe_chunk_norms<float><<<cg, kQeThreads, 0, st>>>(af, S, n_rows, partial);
    else k_qe_chunk_norms<double><<<cg, kQeThreads, 0, st>>>(ad, S, n_rows, partial);
    k_qe_norms<<<(unsigned)((int64_t)K * S * n_samples), kQeThreads, 0, st>>>(
        partial, S, n_samples, n_chunks, chunk_off, norms, factor);
    if (fp32)
        k_qe_store<float2><<<sg, 256, 0, st>>>(af, K, S, n_rows, n_orb, user_to_row, orb_sample,
                                               n_samples, factor, out);
    else
        k_qe_store<double2><<<sg, 256, 0, st>>>(ad, K, S, n_rows, n_orb, user_to_row, orb_sample,
                                                n_samples, factor, out);
    return cudaGetLastError();
}

}  // namespace tbpm
