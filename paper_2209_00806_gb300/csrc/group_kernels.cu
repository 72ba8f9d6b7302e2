// Grouped staged-gather term (real FP32 values, long rows).  The one-stage
// staged kernel reads a neighbour's states from shared memory once per stored
// entry (64 bytes for eight states) and is bound by those reads.  Here four consecutive rows share one list of columns (build_groups):
// a thread holds a 16-byte lane of four rows, so one read of a neighbour and
// one of four values feed 16 FMAs.  The lists' zeros (1.84 slots a stored
// entry on the twisted bilayer) cost FMAs, which are not the limit, and HBM
// bytes (500 a row of values).  The values and positions run through a small
// ring of asynchronous copies per octet, sixteen entries ahead (read four
// ahead into registers they were waited for, 355 us a term at 1.1M rows, and
// took six L1 wavefronts an entry against two); stages of eight entries
// halve the loop's bookkeeping (230 -> 209 us against four).  Shared memory is
// mostly the halo, so four blocks share an SM.  1.1M rows, eight states, 68
// entries a row: 209 us a term against 300 us of the one-stage kernel; L1
// wavefronts, HBM (4.5 TB/s) and issue slots are each about 60-70 % busy.
// Each row's products keep their order, and an entry the row does not have
// adds 0 x: the states equal the plain kernel's.  (A non-finite state also reaches rows of its group
// that do not reference it; the call fails with NONFINITE either way.)
#include <cuda_runtime.h>
#include <stdint.h>

#include "tbpm_internal.cuh"

namespace tbpm {
namespace {

constexpr int kGroupStages = 3;                       // ring stages
constexpr int kGroupStageBytes = kGroupStep * (8 * 16 + 8 * 2);  // values, positions of an octet
constexpr int kGroupRing = 4 * kGroupStages * kGroupStageBytes;

template <int C>
__global__ void __launch_bounds__(32 * C, 16 / C) k_term_group(TermArgs a)
{
    constexpr int R = kGroupRows, OT = 8 * C, ST = kGroupStages;
    constexpr int VB = kGroupStep * 128;             // bytes of values a stage
    extern __shared__ __align__(16) unsigned char sm[];
    const int tid = threadIdx.x;
    const int l = tid % C, slot = tid / C, oct = slot / 8, s8 = slot % 8;
    const int64_t hb = block_of(a.reverse);
    dep_launch();
    const int64_t h0 = __ldg(a.halo_ptr + hb);
    const int H = (int)(__ldg(a.halo_ptr + hb + 1) - h0);
    const int g = __ldg(a.gperm + hb * 32 + slot);
    const int64_t k0 = __ldg(a.gptr + hb * 4 + oct);
    const int stages = (int)(__ldg(a.gptr + hb * 4 + oct + 1) - k0) / kGroupStep;
    // octets of a warp (two of sixteen lanes each for C = 2) run the longer
    // one's stages
    int run = stages;
    if (OT < 32) run = max(run, __shfl_xor_sync(0xffffffffu, run, 16));
    // ring of the octet: where the next stage goes, and what this lane copies
    unsigned char *ring = sm + oct * (ST * kGroupStageBytes);
    const int ol = tid % OT;                         // lane of the octet
    const unsigned char *vsrc = reinterpret_cast<const unsigned char *>(a.gval + k0 * 8) + ol * 16;
    const unsigned char *psrc = reinterpret_cast<const unsigned char *>(a.gpos + k0 * 8) + ol * 16;
    int wr = 0, left = stages;
    auto issue = [&]() {
        if (left > 0) {
            unsigned char *dst = ring + wr + ol * 16;
#pragma unroll
            for (int c = 0; c < VB / 16; c += OT) cp_async16(dst + c * 16, vsrc + c * 16);
            if (ol < kGroupStep) cp_async16(dst + VB, psrc);
            vsrc += VB;
            psrc += kGroupStep * 16;
        }
        --left;
        wr = wr == (ST - 1) * kGroupStageBytes ? 0 : wr + kGroupStageBytes;
        cp_async_commit();                           // an empty group keeps the count
    };
    for (int i = 0; i < ST - 1; ++i) issue();
    const uint32_t r0 = (uint32_t)(hb * kHaloRows) + g * R;
    float d[R];
    {
        const float4 dv = __ldg(reinterpret_cast<const float4 *>(a.H.diag) + r0 / 4);
        d[0] = dv.x; d[1] = dv.y; d[2] = dv.z; d[3] = dv.w;
    }
    constexpr int HB = 8;
    unsigned char *halo = sm + kGroupRing;
    const unsigned char *xg = reinterpret_cast<const unsigned char *>(a.x);
    for (int hr = 0; hr < H; hr += 32 * HB) {        // row numbers HB at a time, then the copies
        int32_t gr[HB];
#pragma unroll
        for (int k = 0; k < HB; ++k) {
            const int h = hr + k * 32 + slot;
            gr[k] = h < H ? __ldg(a.halo_rows + h0 + h) : 0;
        }
        if (hr == 0) dep_wait();
#pragma unroll
        for (int k = 0; k < HB; ++k) {
            const int h = hr + k * 32 + slot;
            if (h < H) cp_async16(halo + (h * C + l) * 16, xg + ((int64_t)gr[k] * C + l) * 16);
        }
    }
    cp_async_commit();
    float4 p[R], z[R];                               // in flight while the halo lands
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int64_t at = (int64_t)(r0 + i) * C + l;
        p[i] = reinterpret_cast<const float4 *>(a.psi)[at];
        z[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (a.z) z[i] = reinterpret_cast<const float4 *>(a.z)[at];
    }
    cp_async_wait_group<0>();
    __syncthreads();
    const unsigned char *xl = halo + l * 16;
    auto x_at = [&](int h) { return *reinterpret_cast<const float4 *>(xl + h * (C * 16)); };
    float4 y[R];
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const float4 x = x_at(g * R + i);
        y[i] = make_float4(x.x * d[i], x.y * d[i], x.z * d[i], x.w * d[i]);
    }
    const unsigned char *rd = ring + s8 * 16, *rd_end = rd + ST * kGroupStageBytes;
    for (int i = 0; i < run; ++i) {
        cp_async_wait_group<ST - 2>();               // stage i has landed (this lane's part)
        __syncwarp();                                // all lanes' parts; stage i - 1 is read
        issue();
        if (OT == 32 || i < stages) {
#pragma unroll
            for (int v = 0; v < kGroupStep / 4; ++v) {
                const uint2 pk = *reinterpret_cast<const uint2 *>(rd + VB + v * 64 - s8 * 8);
                const int hp[4] = {(int)(pk.x & 0xffff), (int)(pk.x >> 16), (int)(pk.y & 0xffff),
                                   (int)(pk.y >> 16)};
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const float4 x = x_at(hp[u]);
                    const float4 w = *reinterpret_cast<const float4 *>(rd + (v * 4 + u) * 128);
                    const float hv[R] = {w.x, w.y, w.z, w.w};
#pragma unroll
                    for (int j = 0; j < R; ++j) {
                        y[j].x = fmaf(hv[j], x.x, y[j].x);
                        y[j].y = fmaf(hv[j], x.y, y[j].y);
                        y[j].z = fmaf(hv[j], x.z, y[j].z);
                        y[j].w = fmaf(hv[j], x.w, y[j].w);
                    }
                }
            }
        }
        rd += kGroupStageBytes;
        if (rd == rd_end) rd -= ST * kGroupStageBytes;
    }
    cp_async_wait_group<0>();
    float4 s = make_float4(1.f, 1.f, 1.f, 1.f);          // (re, im) scales of the two states
    if (a.scale_f) {
        const float *sc = a.scale_f + (int64_t)a.chunk_sample[r0 / kChunkRows] * (C * 2) + l * 2;
        s = make_float4(sc[0], sc[0], sc[1], sc[1]);
    }
    const float gm = a.gamma_f, ch = a.c_hi_f, cl = a.c_lo_f;
#pragma unroll
    for (int i = 0; i < R; ++i) {
        const int64_t at = (int64_t)(r0 + i) * C + l;
        if (a.scale_f) {
            p[i].x *= s.x; p[i].y *= s.y; p[i].z *= s.z; p[i].w *= s.w;
            if (a.x_is_psi) { y[i].x *= s.x; y[i].y *= s.y; y[i].z *= s.z; y[i].w *= s.w; }
        }
        // + gamma (-i) y, then the coefficient's low and high part
        float4 o;
        o.x = fmaf(ch, p[i].x, fmaf(cl, p[i].x, fmaf(gm, y[i].y, z[i].x)));
        o.y = fmaf(ch, p[i].y, fmaf(cl, p[i].y, fmaf(-gm, y[i].x, z[i].y)));
        o.z = fmaf(ch, p[i].z, fmaf(cl, p[i].z, fmaf(gm, y[i].w, z[i].z)));
        o.w = fmaf(ch, p[i].w, fmaf(cl, p[i].w, fmaf(-gm, y[i].z, z[i].w)));
        reinterpret_cast<float4 *>(a.out)[at] = o;
    }
}

template <int C>
cudaError_t launch_group_t(const TermArgs &a, cudaStream_t st)
{
    const int smem = kGroupRing + a.halo_max * C * 16;
    const cudaError_t e = allow_shared<k_term_group<C>>(kGroupRing + (kHaloRows + kHaloMaxExt) * C * 16);
    if (e != cudaSuccess) return e;
    return launch_dependent(k_term_group<C>, (unsigned)(a.n_rows / kHaloRows), 32 * C, smem, st, a);
}

}  // namespace

cudaError_t launch_term_group(const TermArgs &a, int B, cudaStream_t st)
{
    return B == 4 ? launch_group_t<2>(a, st) : launch_group_t<4>(a, st);
}

}  // namespace tbpm
