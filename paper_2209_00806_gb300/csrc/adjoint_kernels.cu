// a8: adjoint of the Chebyshev propagation (FP64).
//
// For a real loss L of the correlations C_n = <psi0|phi_n> the caller gives
// gbar_n = dL/dRe C_n + i dL/dIm C_n per sample and state.  The adjoint of
// the trajectory obeys Lambda_N = gbar_N psi0 and
// Lambda_n = gbar_n psi0 + P^dagger Lambda_{n+1}, with P the one-step
// propagator of the Chebyshev sum (Sec. 2.2).  H~ is Hermitian, so
// P^dagger = sum_m a_m T^_m(H~)^dagger is the same series with +i in place
// of -i: the backward pass reuses the Clenshaw schedule of the forward one
// with gamma -> -gamma.  Its intermediate vectors are exactly the adjoints
// mu_m of the forward polynomials T^_m, so the kernel that forms mu_m from
// the gathered mu_{m+1} also accumulates, for every stored entry (r, c),
//   G_rc += g_{m+1} Im(conj(mu_{m+1, c}) T^_{m, r}),
// the contribution of the transposed element to dL/dH~ (g = 2, or 1 for the
// closing term; G holds half of that sum).  A bond's gradient is the sum of its
// two stored entries;
// the diagonal entry gives dL/deps.  Entries of a row are owned by one
// thread, so the accumulation needs no atomics and is deterministic.
#include <cuda_runtime.h>
#include <stdint.h>

#include "tbpm_internal.cuh"

namespace tbpm {
namespace {

// One term of the forward or the conjugate series, SPL states a thread, L
// threads a row, with the row's matrix values already scaled by |gamma|:
//   out = [c psi] + z + sigma (-i) (H' x)                      (sigma = +-1)
//   out = [c psi] + fac sigma (-i) (H' x)                      (FAC: first term)
// and, GRAD, G_rc += w Im(conj(x_c) T_r) with w = 1, or gfac with FAC or the
// closing term (WFAC): the caller's G is half the gradient, since interior
// terms have weight 2.  Bound by the FP64 pipe, one 64-cycle slot per warp and
// instruction: every product lands in the output or in G by one FMA, started
// from z and from the stored G, so a state and row of E entries takes 4 + 2E
// operations (2 + 2E without c) and 2 + 2E for the gradients: 18 on graphene,
// against 36 with gamma and the weight multiplied in, entries in rounds of
// four and one thread per state (whose partial gradients had to be added by
// shuffles).  524,288 rows x 2 states: 36 us a gradient term (68 before; 45 us the
// first of a step, 52 us the closing one), 19 us a plain one (36 before), 23 us with
// the next state's share.
// ACC (polynomials): the term's share of the next state too, next += ca out
// (2: the first polynomial, next = c x + ca out); out may then be nullptr.
template <int L, int SPL, int W, bool HASC, bool FAC, bool GRAD, bool WFAC, int ACC = 0>
__global__ void __launch_bounds__(128) k_adj(AdjArgs a)
{
    constexpr int NS = W ? W : 4;
    dep_launch();
    const uint32_t t = blockIdx.x * 128u + threadIdx.x;
    // the grid covers exactly n_rows * L threads (n_rows is a multiple of
    // kChunkRows), so every warp is complete and shuffles below are safe
    const uint32_t r = t / L, l = t % L;
    const uint32_t q = r / kSliceRows, lr = r % kSliceRows;
    int64_t base;
    int w;
    if (W || a.fixed_width) {
        w = W ? W : a.fixed_width;
        base = (int64_t)q * (kSliceRows * w) + lr;
    } else {
        base = __ldg(a.slice_ptr + q);
        w = (int)((__ldg(a.slice_ptr + q + 1) - base) / kSliceRows);
        base += lr;
    }
    int32_t c[NS];
    double h[NS];
    auto entries = [&](int k) {
#pragma unroll
        for (int u = 0; u < NS; ++u) {
            const bool ok = W || k + u < w;
            c[u] = ok ? __ldg(a.col + base + (int64_t)(k + u) * kSliceRows) : (int32_t)r;
            h[u] = ok ? xor_sign(__ldg(a.val + base + (int64_t)(k + u) * kSliceRows), a.sign) : 0.0;
        }
    };
    entries(0);
    const double d = xor_sign(__ldg(a.diag + r), a.sign);
    dep_wait();
    const double2 *x = reinterpret_cast<const double2 *>(a.x);
    auto at = [&](uint32_t row) { return ((int64_t)row * L + l) * SPL; };
    double2 o[SPL], T[SPL], xr[SPL];
#pragma unroll
    for (int j = 0; j < SPL; ++j) {
        xr[j] = x[at(r) + j];
        o[j] = make_double2(0.0, 0.0);
        if (GRAD) T[j] = reinterpret_cast<const double2 *>(a.T_own)[at(r) + j];
        if (!FAC && a.z) o[j] = reinterpret_cast<const double2 *>(a.z)[at(r) + j];
    }
    double2 p[SPL];
    double2 nx[SPL];
    if (ACC == 1)
#pragma unroll
        for (int j = 0; j < SPL; ++j) nx[j] = reinterpret_cast<const double2 *>(a.next)[at(r) + j];
    if (HASC)
#pragma unroll
        for (int j = 0; j < SPL; ++j) p[j] = reinterpret_cast<const double2 *>(a.psi)[at(r) + j];
    if (GRAD && WFAC)
#pragma unroll
        for (int j = 0; j < SPL; ++j) {
            T[j].x *= a.gfac;
            T[j].y *= a.gfac;
        }
    // sum over this thread's states, and over the row's threads; g: the stored
    // value on the row's first thread, zero on the others
    auto grad = [&](const double2 (&xc)[SPL], double g) {
#pragma unroll
        for (int j = 0; j < SPL; ++j) {
            g = fma(xc[j].x, T[j].y, g);
            g = fma(-xc[j].y, T[j].x, g);
        }
#pragma unroll
        for (int off = 1; off < L; off <<= 1) g += __shfl_xor_sync(0xffffffffu, g, off);
        return g;
    };
    double gd = 0.0;
    if (GRAD && l == 0) gd = a.Gdiag[r];
#pragma unroll
    for (int j = 0; j < SPL; ++j) {
        o[j].x = fma(d, xr[j].y, o[j].x);
        o[j].y = fma(-d, xr[j].x, o[j].y);
    }
    if (GRAD) {
        gd = grad(xr, gd);
        if (l == 0) a.Gdiag[r] = gd;
    }
    for (int k = 0; W ? k < 1 : k < w; k += 4) {
        if (!W && k) entries(k);
        double2 xv[NS][SPL];
        double G[NS];
#pragma unroll
        for (int u = 0; u < NS; ++u) {
#pragma unroll
            for (int j = 0; j < SPL; ++j) xv[u][j] = x[at(c[u]) + j];
            G[u] = 0.0;
            if (GRAD && l == 0 && (W || k + u < w)) G[u] = a.G[base + (int64_t)(k + u) * kSliceRows];
        }
#pragma unroll
        for (int u = 0; u < NS; ++u) {
#pragma unroll
            for (int j = 0; j < SPL; ++j) {
                o[j].x = fma(h[u], xv[u][j].y, o[j].x);
                o[j].y = fma(-h[u], xv[u][j].x, o[j].y);
            }
            if (GRAD) {
                G[u] = grad(xv[u], G[u]);
                if (l == 0 && (W || k + u < w)) a.G[base + (int64_t)(k + u) * kSliceRows] = G[u];
            }
        }
    }
    double2 *out = reinterpret_cast<double2 *>(a.out);
#pragma unroll
    for (int j = 0; j < SPL; ++j) {
        if (FAC) {
            o[j].x *= a.fac;
            o[j].y *= a.fac;
        }
        if (HASC) {
            o[j].x = fma(a.c, p[j].x, o[j].x);
            o[j].y = fma(a.c, p[j].y, o[j].y);
        }
    }
    if (GRAD && WFAC && a.gbar) {   // + gbar_n psi0 (the adjoint source of step n)
        const int smp = a.chunk_sample[r / kChunkRows];
#pragma unroll
        for (int j = 0; j < SPL; ++j) {
            const double2 g = a.gbar[((int64_t)smp * a.n_states + a.state0 + l * SPL + j) *
                                         (a.n_steps + 1) + a.step];
            const double2 p0 = reinterpret_cast<const double2 *>(a.psi0)[at(r) + j];
            o[j].x += g.x * p0.x - g.y * p0.y;
            o[j].y += g.x * p0.y + g.y * p0.x;
        }
    }
    if (ACC) {
#pragma unroll
        for (int j = 0; j < SPL; ++j) {
            if (ACC == 2) nx[j] = make_double2(a.c * xr[j].x, a.c * xr[j].y);
            nx[j].x = fma(a.ca, o[j].x, nx[j].x);
            nx[j].y = fma(a.ca, o[j].y, nx[j].y);
            reinterpret_cast<double2 *>(a.next)[at(r) + j] = nx[j];
        }
        if (!out) return;
    }
#pragma unroll
    for (int j = 0; j < SPL; ++j) out[at(r) + j] = o[j];
}

// 2 H~: the values and the diagonal of the interior terms (exact)
__global__ void k_double(int64_t n, const double *src, double *dst)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) dst[i] = src[i] + src[i];
}

// out = gbar_N psi0 (the adjoint of the last state).
__global__ void k_source_init(int64_t n_rows, int B, const int32_t *chunk_sample,
                              const double2 *gbar, int n_states, int state0, int n_steps,
                              int step, const double2 *psi0, double2 *out)
{
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n_rows * B) return;
    const int64_t r = i / B;
    const int b = (int)(i % B);
    const int s = chunk_sample[r / kChunkRows];
    const double2 g = gbar[((int64_t)s * n_states + state0 + b) * (n_steps + 1) + step];
    const double2 p = psi0[i];
    out[i] = make_double2(g.x * p.x - g.y * p.y, g.x * p.y + g.y * p.x);
}

__device__ __forceinline__ double find_entry(const int64_t *slice_ptr, const int32_t *col,
                                             const double *G, int32_t r, int32_t c)
{
    const int64_t q = r / kSliceRows;
    const int lr = r % kSliceRows;
    const int64_t base = slice_ptr[q];
    const int w = (int)((slice_ptr[q + 1] - base) / kSliceRows);
    for (int k = 0; k < w; ++k) {
        const int64_t e = base + (int64_t)k * kSliceRows + lr;
        if (col[e] == c) return G[e];
    }
    return __longlong_as_double(0x7ff8000000000000LL);   // not stored: NaN flags it
}

__global__ void k_bond_grad(int64_t n_hop, const int32_t *bond_rows, const int64_t *slice_ptr,
                            const int32_t *col, const double *G, double two_inv_s, double *grad)
{
    const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (b >= n_hop) return;
    const int32_t ri = bond_rows[2 * b], rj = bond_rows[2 * b + 1];
    grad[b] = (find_entry(slice_ptr, col, G, ri, rj) + find_entry(slice_ptr, col, G, rj, ri)) *
              two_inv_s;
}

__global__ void k_onsite_grad(int64_t n_orb, const int32_t *user_to_row, const double *Gd,
                              double two_inv_s, double *grad)
{
    const int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (u < n_orb) grad[u] = Gd[user_to_row[u]] * two_inv_s;
}

}  // namespace

namespace {
template <int L, int SPL, int W>
cudaError_t launch_adj_w(const AdjArgs &a, AdjKind kind, cudaStream_t st)
{
    const unsigned blocks = (unsigned)(a.n_rows * L / 128);
    auto go = [&](void (*k)(AdjArgs)) { return launch_dependent(k, blocks, 128, 0, st, a); };
    switch (kind) {
    case kAdjPoly: return go(k_adj<L, SPL, W, false, false, false, false>);
    case kAdjPolyAcc: return go(k_adj<L, SPL, W, false, false, false, false, 1>);
    case kAdjPolyFirst: return go(k_adj<L, SPL, W, false, false, false, false, 2>);
    case kAdjStep: return go(k_adj<L, SPL, W, true, false, false, false>);
    case kAdjStepFirst: return go(k_adj<L, SPL, W, true, true, false, false>);
    case kAdjGrad: return go(k_adj<L, SPL, W, true, false, true, false>);
    case kAdjGradFirst: return go(k_adj<L, SPL, W, true, true, true, true>);
    case kAdjGradLast: return go(k_adj<L, SPL, W, true, false, true, true>);
    }
    return cudaErrorInvalidValue;
}
template <int L, int SPL>
cudaError_t launch_adj_t(const AdjArgs &a, AdjKind kind, cudaStream_t st)
{
    return a.fixed_width == 3 ? launch_adj_w<L, SPL, 3>(a, kind, st)
                              : launch_adj_w<L, SPL, 0>(a, kind, st);
}
}  // namespace

cudaError_t launch_adj(const AdjArgs &a, AdjKind kind, int B, cudaStream_t st)
{
    switch (B) {
    case 1: return launch_adj_t<1, 1>(a, kind, st);
    case 2: return launch_adj_t<1, 2>(a, kind, st);
    case 4: return launch_adj_t<2, 2>(a, kind, st);
    case 8: return launch_adj_t<4, 2>(a, kind, st);
    }
    return cudaErrorInvalidValue;
}

cudaError_t launch_double(int64_t n, const double *src, double *dst, cudaStream_t st)
{
    if (n > 0) k_double<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, src, dst);
    return cudaGetLastError();
}

cudaError_t launch_source_init(int64_t n_rows, int B, const int32_t *chunk_sample,
                               const double2 *gbar, int n_states, int state0, int n_steps,
                               int step, const void *psi0, void *out, cudaStream_t st)
{
    const int64_t n = n_rows * B;
    k_source_init<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(
        n_rows, B, chunk_sample, gbar, n_states, state0, n_steps, step,
        reinterpret_cast<const double2 *>(psi0), reinterpret_cast<double2 *>(out));
    return cudaGetLastError();
}

cudaError_t launch_param_grads(int64_t n_hop, const int32_t *bond_rows, const int64_t *slice_ptr,
                               const int32_t *col, const double *G, const double *Gd,
                               int64_t n_orb, const int32_t *user_to_row, double inv_s,
                               double *grad_hop, double *grad_onsite, cudaStream_t st)
{
    if (n_hop > 0)
        k_bond_grad<<<(unsigned)((n_hop + 255) / 256), 256, 0, st>>>(n_hop, bond_rows, slice_ptr,
                                                                     col, G, 2.0 * inv_s, grad_hop);
    k_onsite_grad<<<(unsigned)((n_orb + 255) / 256), 256, 0, st>>>(n_orb, user_to_row, Gd, 2.0 * inv_s,
                                                                   grad_onsite);
    return cudaGetLastError();
}

}  // namespace tbpm
