// lbmhd_step.cu -- the fused pull-stream + collide kernel of one LB-MHD
// time step over a single lattice (Sec. 1.2 streaming, Sec. 3 MRT / SRT
// collisions).  The per-thread work is step_body (lbmhd_step_body.cuh): a
// warp covers 32*V consecutive nodes of one row, loads each of the 19
// planes once with aligned vector loads, takes the x-halo from the
// neighbouring lane by a shuffle and collides in registers.  All HBM
// traffic is the 19 plane reads and 19 plane writes per node.
#include "lbmhd_internal.h"
#include "lbmhd_pdl.cuh"
#include "lbmhd_step_body.cuh"

namespace lbmhd {

template <int P, int V>
__global__ void __launch_bounds__(256) step_kernel(const typename Fmt<P>::S* src,
                                                   typename Fmt<P>::S* dst, int nx,
                                                   int ny, long long ps, unsigned total,
                                                   unsigned total_pad,
                                                   Coll<typename Fmt<P>::R> c, float scale,
                                                   float inv_scale, int y0) {
    after_previous();
    const unsigned stride = gridDim.x * blockDim.x;
    for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < total_pad; t += stride)
        step_body<P, V>(src, dst, nx, ny, ps, t, total, c, scale, inv_scale, y0);
}

// Eight FP16 nodes per thread, held to 128 registers, 16 warps per SM (left to
// itself ptxas takes 143, 12 warps: 8192^2 933 us per step).
__global__ void __launch_bounds__(256, 2)
    step_kernel_h8(const unsigned short* src, unsigned short* dst, int nx,
                   int ny, long long ps, unsigned total, unsigned total_pad, Coll<float> c,
                   float scale, float inv_scale, int y0) {
    after_previous();
    const unsigned stride = gridDim.x * blockDim.x;
    for (unsigned t = blockIdx.x * blockDim.x + threadIdx.x; t < total_pad; t += stride)
        step_body<P_FP16_DEV, 8>(src, dst, nx, ny, ps, t, total, c, scale, inv_scale, y0);
}

template <int P, int V>
static cudaError_t launch_pv(int block, int max_blocks, const void* src, void* dst, const Geom& g,
                             const HostColl& hc, cudaStream_t st, int y0, int y1, bool whole) {
    using S = typename Fmt<P>::S;
    using R = typename Fmt<P>::R;
    const unsigned total = (unsigned)((long long)g.nx / V * (y1 - y0));
    const unsigned total_pad = (total + 31u) / 32u * 32u;
    long long blocks = ((long long)total_pad + block - 1) / block;
    if (max_blocks > 0 && blocks > max_blocks) blocks = max_blocks;
    auto k = step_kernel<P, V == 8 ? 1 : V>;
    if constexpr (V == 8) k = step_kernel_h8;
    // a range of rows may follow other work than a step: a plain launch
    if (!whole) {
        k<<<(unsigned)blocks, block, 0, st>>>((const S*)src, (S*)dst, g.nx, g.ny, g.ps, total, total_pad,
                                              coll_for_prec<R>(hc, P), hc.scale, hc.inv_scale, y0);
        return cudaGetLastError();
    }
    return launch_after(k, (unsigned)blocks, block, st, (const S*)src, (S*)dst, g.nx, g.ny, g.ps, total,
                        total_pad, coll_for_prec<R>(hc, P), hc.scale, hc.inv_scale, y0);
}

bool step_variant_ok(int prec, int vec, int nx) {
    if (prec < 0 || prec > 4) return false;
    if (vec != 1 && vec != 2 && vec != 4 && !(vec == 8 && prec == P_FP16_DEV)) return false;
    return nx % vec == 0;
}

cudaError_t launch_step(int prec, int vec, int block, int max_blocks, const void* src, void* dst,
                        const Geom& g, const HostColl& c, cudaStream_t st, int y0, int y1) {
    const bool whole = y1 < 0;
    if (whole) y1 = g.ny;
#define LBMHD_CASE(P)                                                                      \
    case P:                                                                                \
        switch (vec) {                                                                     \
            case 1: return launch_pv<P, 1>(block, max_blocks, src, dst, g, c, st, y0, y1, whole); \
            case 2: return launch_pv<P, 2>(block, max_blocks, src, dst, g, c, st, y0, y1, whole); \
            case 4: return launch_pv<P, 4>(block, max_blocks, src, dst, g, c, st, y0, y1, whole); \
        }                                                                                  \
        break;
    switch (prec) {
        LBMHD_CASE(P_FP64)
        LBMHD_CASE(P_FP32)
        LBMHD_CASE(P_FP32_DEV)
        LBMHD_CASE(P_FF)
        case P_FP16_DEV:
            switch (vec) {
                case 1: return launch_pv<P_FP16_DEV, 1>(block, max_blocks, src, dst, g, c, st, y0, y1, whole);
                case 2: return launch_pv<P_FP16_DEV, 2>(block, max_blocks, src, dst, g, c, st, y0, y1, whole);
                case 4: return launch_pv<P_FP16_DEV, 4>(block, max_blocks, src, dst, g, c, st, y0, y1, whole);
                case 8: return launch_pv<P_FP16_DEV, 8>(block, max_blocks, src, dst, g, c, st, y0, y1, whole);
            }
            break;
    }
#undef LBMHD_CASE
    return cudaErrorInvalidValue;
}

}  // namespace lbmhd
