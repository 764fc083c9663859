// lbmhd_step_pipe.cu -- S = 2, 3 or 4 LB-MHD time steps in one pass over the
// state, for the FP32 and FP16 storage forms with the local rates or no
// closure (les 0, 1): the values of S single steps (lbmhd_step.cu), bit for bit
// but for the sign of a zero (mul_, lbmhd_pair.cuh).
//
// Why: the one-step kernel moves 152 B per node update (FP32) at the copy
// bandwidth (1.03 of it at 8192^2), so only fewer passes over HBM make it
// faster.  A step is a 3 x 3 stencil, so S steps of a strip of columns need
// S rows of history and S halo columns on each side, nothing else.
//
// How: one warp owns a strip of 64 columns (two neighbouring ones per lane)
// and a segment of rows, and sweeps down it; no other warp is involved, so
// there is no barrier and nothing to wait for.  When the first step is at
// row r, the second is at row r - 1, the third at r - 2: a row that a step
// has just computed is streamed along x by one shuffle per plane with
// c_x != 0 and feeds the next step at once (planes with c_y < 0), one row
// later (c_y = 0, kept in shared memory, each lane its own values) or two
// rows later (c_y > 0, kept in registers).  The strip's outer S columns (the
// left side rounded up to an even number, so that every lane's pair is
// aligned) are computed from incomplete neighbours and not stored:
// neighbouring strips overlap by them, as segments do by 2 (S - 1) rows.
// Rows and columns wrap periodically at the loads, so nothing else knows of
// the edges of the lattice.
//
// The next row's 19 planes are fetched into shared memory by cp.async while
// the present one is computed (each lane copies what it reads itself, so its
// own wait orders it).  The two columns of a lane go through the collision
// together in packed two-wide FP32 instructions (lbmhd_pair.cuh).
//
// Bound: instruction issue and the FMA pipe with the latency of few warps: the
// history of S - 1 steps takes registers, two to four warps per scheduler.  ncu,
// 4096^2, S = 4: FP32 173 instructions per update and thread, 54% of the issue
// slots and 61% of the FMA pipe busy, 60% of DRAM, 1.1 cycles per instruction
// waiting for a fixed latency and none of the others above 0.4; FP16 194
// instructions, 63% and 65%, 31% of DRAM, 1.4 cycles waiting for the pipe.
// Measured on GB300, 8192^2, updates per second:
//   FP32  one-step 45.9 G;  S = 2 82.6 G;  S = 3 121.5 G;  S = 4 127.9 G
//   FP16  one-step 81.6 G;  S = 2 124 G;   S = 3 132 G;    S = 4 133.9 G
// and 1024^2 (FP32) 36.9 -> 93.0 G, 1999 x 1201 (odd rows) 34.3 -> 95.6 G.
// On the way (FP32, S = 3): scalar collision without the fetch ahead 91 G
// (61% issue, 1.7 of 4.4 cycles per instruction waiting for the row), with
// it 104 G, packed 108 G, and 120 G once shared memory held only the nine
// c_y = 0 planes -- L1 takes what shared memory leaves, and it holds the
// rows in flight; with the largest shared-memory carve-out S = 2 fell to
// 57 G, and any spilled register costs half the rate.
#include "lbmhd_batch_run.cuh"
#include "lbmhd_cp_async.cuh"
#include "lbmhd_internal.h"
#include "lbmhd_pair.cuh"
#include "lbmhd_pdl.cuh"
#include "lbmhd_pipe_plan.h"
#include "lbmhd_step_body.cuh"

namespace lbmhd {

namespace {

// A pair of neighbouring columns of one plane, as stored.
template <int P>
struct PairOf {
    using T = float2;
};
template <>
struct PairOf<P_FP16_DEV> {  // column x0 in the low half
    using T = unsigned;
};

// The pair that streams in along CX: the values of columns x - CX.  The
// outer lanes get a wrong value for the missing column: a halo column whose
// result is not used.
template <int CX>
__device__ __forceinline__ float2 stream1(float2 v) {
    if constexpr (CX == 0) return v;
    if constexpr (CX > 0) return make_float2(__shfl_up_sync(0xffffffffu, v.y, 1), v.x);
    return make_float2(v.y, __shfl_down_sync(0xffffffffu, v.x, 1));
}
template <int CX>
__device__ __forceinline__ unsigned stream1(unsigned v) {
    if constexpr (CX == 0) return v;
    if constexpr (CX > 0) return __byte_perm(__shfl_up_sync(0xffffffffu, v, 1), v, 0x5432);
    return __byte_perm(v, __shfl_down_sync(0xffffffffu, v, 1), 0x5432);
}

// A row's pairs from their stored form, and back.
template <int P>
__device__ __forceinline__ void unpack(const typename PairOf<P>::T (&z)[kPlanes], float2 (&d)[9], float2 (&g)[10]) {
#pragma unroll
    for (int p = 0; p < kPlanes; ++p) {
        float2 v;
        if constexpr (P == P_FP16_DEV) v = __half22float2(*reinterpret_cast<const __half2*>(&z[p]));
        else v = z[p];
        if (P == P_FP32 && p < 9) v = add_(v, dup<float2>(-plane_rest<float>(p)));
        if (p < 9) d[p] = v;
        else g[p - 9] = v;
    }
}
template <int P>
__device__ __forceinline__ void pack(const float2 (&d)[9], const float2 (&g)[10], typename PairOf<P>::T (&z)[kPlanes]) {
#pragma unroll
    for (int p = 0; p < kPlanes; ++p) {
        float2 v = p < 9 ? d[p] : g[p - 9];
        if (P == P_FP32 && p < 9) v = add_(v, dup<float2>(plane_rest<float>(p)));
        if constexpr (P == P_FP16_DEV) {
            const __half2 h = __float22half2_rn(v);
            z[p] = *reinterpret_cast<const unsigned*>(&h);
        } else {
            z[p] = v;
        }
    }
}

// Both columns of a pair through the collision, stored form to stored form.
template <int P>
__device__ __forceinline__ void collide_pair(typename PairOf<P>::T (&z)[kPlanes], const Coll<float>& c) {
    float2 d[9], g[10];
    unpack<P>(z, d, g);
    collide_r<float2, Fmt<P>::kScaled, P == P_FP32>(d, g, c);
    pack<P>(d, g, z);
}

// Place of plane p among the planes that do not move along y.
__host__ __device__ constexpr int keep_slot(int p) {
    int n = 0;
    for (int q = 0; q < p; ++q) n += plane_cy(q) == 0;
    return n;
}

// The populations that stream along y into row r0 of the lane's columns xa, xb
// (fetched ahead into pre by cp.async, or into z), and on to the next row.
template <int P, bool AL, int N>
__device__ __forceinline__ void fetch_row(const typename Fmt<P>::S* __restrict__ src, int nx, long long ps,
                                          int xa, int xb, int& rm, int& r0, int& rp, int ny,
                                          typename PairOf<P>::T (&pre)[N][32],
                                          typename PairOf<P>::T (&z)[kPlanes]) {
    using T = typename Fmt<P>::S;
    const int lane = threadIdx.x;
    const unsigned om = (unsigned)rm * (unsigned)nx, o0 = (unsigned)r0 * (unsigned)nx,
                   op = (unsigned)rp * (unsigned)nx;
#pragma unroll
    for (int p = 0; p < kPlanes; ++p) {
        const unsigned row = plane_cy(p) == 0 ? o0 : (plane_cy(p) > 0 ? om : op);
        const T* base = src + p * ps;
        if constexpr (AL) cp_async_small<2 * sizeof(T)>(&pre[p][lane], base + (row + xa));
        else if constexpr (P != P_FP16_DEV) {
            cp_async_small<4>(&pre[p][lane].x, base + (row + xa));
            cp_async_small<4>(&pre[p][lane].y, base + (row + xb));
        } else {
            z[p] = (unsigned)base[row + xa] | (unsigned)base[row + xb] << 16;
        }
    }
    if (AL || P != P_FP16_DEV) cp_async_commit();
    rm = r0;
    r0 = rp;
    rp = rp + 1 == ny ? 0 : rp + 1;
}

// A row streamed along x.
template <int P>
__device__ __forceinline__ void stream_row(typename PairOf<P>::T (&v)[kPlanes]) {
#pragma unroll
    for (int p = 0; p < kPlanes; ++p)
        v[p] = plane_cx(p) == 0 ? v[p] : (plane_cx(p) > 0 ? stream1<1>(v[p]) : stream1<-1>(v[p]));
}

template <int P, bool AL>
__device__ __forceinline__ void store_row(typename Fmt<P>::S* __restrict__ dst, long long ps, unsigned orow,
                                          bool outb, const typename PairOf<P>::T (&z)[kPlanes]) {
    using T = typename Fmt<P>::S;
#pragma unroll
    for (int p = 0; p < kPlanes; ++p) {
        T* o = dst + p * ps + orow;
        if constexpr (AL) {
            *reinterpret_cast<typename PairOf<P>::T*>(o) = z[p];
        } else if constexpr (P == P_FP16_DEV) {
            o[0] = (T)z[p];
            if (outb) o[1] = (T)(z[p] >> 16);
        } else {
            o[0] = z[p].x;
            if (outb) o[1] = z[p].y;
        }
    }
}

// The shared memory of one warp.
template <int P, int S, bool AL>
struct PipeShared {
    using Q = typename PairOf<P>::T;
    // cp.async moves 4 or 8 bytes: odd rows of FP16 are loaded directly
    static constexpr bool PF = AL || P != P_FP16_DEV;
    Q pre[PF ? kPlanes : 1][32];  // the fetched row
    Q keep[S - 1][9][32];         // each step's last row, c_y = 0
};

// One warp: S steps of rows [y0, y1) of one strip of a lattice.  AL: nx is
// even, so a lane's pair is one aligned word in every row.
template <int P, int S, bool AL>
__device__ __forceinline__ void pipe_body(const typename Fmt<P>::S* __restrict__ src,
                                          typename Fmt<P>::S* __restrict__ dst, int nx, int ny,
                                          long long ps, int strip, int y0, int y1,
                                          const Coll<float>& c, PipeShared<P, S, AL>& sh) {
    using T = typename Fmt<P>::S;
    using Q = typename PairOf<P>::T;
    constexpr int HL = pipe_halo(S), U = pipe_useful(S);
    constexpr bool PF = PipeShared<P, S, AL>::PF;
    auto& pre = sh.pre;
    auto& keep = sh.keep;
    const int lane = threadIdx.x;
    const int x = strip * U - HL + 2 * lane;  // this lane's first column, unwrapped
    int xa = x % nx;
    if (xa < 0) xa += nx;
    const int xb = xa + 1 == nx ? 0 : xa + 1;
    const bool outa = x >= strip * U && x < strip * U + U && x < nx;
    const bool outb = outa && x + 1 < nx;
    // rows r - 1, r, r + 1 of the row r that the first step is at
    int rm = (y0 - S) % ny, r0, rp;
    if (rm < 0) rm += ny;
    r0 = rm + 1 == ny ? 0 : rm + 1;
    rp = r0 + 1 == ny ? 0 : r0 + 1;

    auto fetch = [&](Q(&z)[kPlanes]) { fetch_row<P, AL>(src, nx, ps, xa, xb, rm, r0, rp, ny, pre, z); };
    auto stream = [&](Q(&v)[kPlanes]) { stream_row<P>(v); };

    Q h1[S - 1][kPlanes], h2[S - 1][kPlanes];  // c_y > 0: the last row and the one before
    const int n = y1 - y0 + 2 * (S - 1);
    unsigned orow = (unsigned)y0 * (unsigned)nx + (unsigned)x;
    Q z[kPlanes];
    if (PF) fetch(z);
#pragma unroll 1
    for (int it = 0; it < n; ++it) {
        if (PF) {
            cp_async_wait<0>();
#pragma unroll
            for (int p = 0; p < kPlanes; ++p) z[p] = pre[p][lane];
            stream(z);
            if (it + 1 < n) fetch(z);
        } else {
            fetch(z);
            stream(z);
        }
        collide_pair<P>(z, c);
        bool done = false;  // the next step's rows are not there yet
#pragma unroll
        for (int k = 1; k < S; ++k) {
            if (done) continue;
            stream(z);
            Q w[kPlanes];
#pragma unroll
            for (int p = 0; p < kPlanes; ++p) {
                if (plane_cy(p) < 0) w[p] = z[p];
                else if (plane_cy(p) == 0) {
                    w[p] = keep[k - 1][keep_slot(p)][lane];
                    keep[k - 1][keep_slot(p)][lane] = z[p];
                } else {
                    w[p] = h2[k - 1][p];
                    h2[k - 1][p] = h1[k - 1][p];
                    h1[k - 1][p] = z[p];
                }
            }
            if (it < 2 * k) {
                done = true;
                continue;
            }
            collide_pair<P>(w, c);
#pragma unroll
            for (int p = 0; p < kPlanes; ++p) z[p] = w[p];
        }
        if (done) continue;
        if (outa) store_row<P, AL>(dst, ps, orow, outb, z);
        orow += (unsigned)nx;
    }
}

// ---- two steps of a kinetic closure (les 2, 3) per pass ---------------------
// A step of these closures needs the conserved moments of the streamed
// populations at the four neighbours, so each of the two steps keeps its
// last streamed row (in shared memory) and the moments of its last two rows
// (in registers), and collides a row when the next one has been streamed:
// one more row of lag and one more halo column on each side per step than
// above.  Measured on GB300 (us per step, the one-step fused kernel / this):
// 8192^2 FP32 les 2 1735 / 1116, les 3 1737 / 1098; FP16 les 2 1521 / 1081, les 3
// 1517 / 955; 4096^2 FP32 les 2 448 / 293.  The one-step kernel ran at 0.87 of
// the copy bandwidth at 152 B per node; this one is bound by issue and
// latency at two warps per scheduler (ncu, 4096^2 FP32 les 2: 353 instructions
// per update and thread, 52% of the issue slots, 56% of the FMA pipe, 56% of
// DRAM).
template <int P, bool AL>
struct KinShared {
    using Q = typename PairOf<P>::T;
    static constexpr bool PF = AL || P != P_FP16_DEV;
    Q pre[PF ? kPlanes : 1][32];
    Q row[2][kPlanes][32];  // each step's last streamed row
    Q keep[9][32];          // the first step's last result, c_y = 0
};
constexpr int kKinHalo = 4, kKinUseful = 64 - 2 * kKinHalo;

__device__ __forceinline__ float2 west(float2 v) { return stream1<1>(v); }   // values at x - 1
__device__ __forceinline__ float2 east(float2 v) { return stream1<-1>(v); }  // at x + 1

// The closure's fields of a streamed row: rho, j, B (les 2) or u, B (les 3).
template <int P, int MODE>
__device__ __forceinline__ void kin_fields(const typename PairOf<P>::T (&z)[kPlanes], const Coll<float>& c,
                                           float2 (&m)[MODE == 2 ? 5 : 4]) {
    float2 d[9], g[10], a[5];
    unpack<P>(z, d, g);
    moments_r<float2, Fmt<P>::kScaled>(d, g, c.inv_s, a);
    if constexpr (MODE == 2) {
#pragma unroll
        for (int q = 0; q < 5; ++q) m[q] = a[q];
    } else {
        const float2 ir = recip_(a[0]);
        m[0] = mul_(a[1], ir);
        m[1] = mul_(a[2], ir);
        m[2] = a[3];
        m[3] = a[4];
    }
}

// A streamed row collided with the fields of the row below (lo), its own (at)
// and the row above (hi).
template <int P, int MODE>
__device__ __forceinline__ void kin_collide(typename PairOf<P>::T (&z)[kPlanes],
                                            const float2 (&lo)[MODE == 2 ? 5 : 4],
                                            const float2 (&at)[MODE == 2 ? 5 : 4],
                                            const float2 (&hi)[MODE == 2 ? 5 : 4], const Coll<float>& c) {
    constexpr int NF = MODE == 2 ? 5 : 4;
    constexpr bool SC = Fmt<P>::kScaled;
    float2 gx[NF], gy[NF];
#pragma unroll
    for (int q = 0; q < NF; ++q) {
        gx[q] = mul_(0.5f, sub_(east(at[q]), west(at[q])));
        gy[q] = mul_(0.5f, sub_(hi[q], lo[q]));
    }
    float2 d[9], g[10];
    if constexpr (MODE == 2) {
        float2 sh[4];
        filtered_shift_r<float2>(at, gx, gy, c.d2, sh);
        if (SC)
#pragma unroll
            for (int q = 0; q < 4; ++q) sh[q] = mul_(c.scl, sh[q]);
        unpack<P>(z, d, g);
        collide_kin_r<float2, SC, true>(d, g, c, sh);
    } else {
        const float2 gu[2][2] = {{gx[0], gy[0]}, {gx[1], gy[1]}}, gb[2][2] = {{gx[2], gy[2]}, {gx[3], gy[3]}};
        float2 taus[2];
        carati_taus_r<float2>(gu, gb, c, taus);
        unpack<P>(z, d, g);
        collide_kin_r<float2, SC, false>(d, g, c, taus);
    }
    pack<P>(d, g, z);
}

// Warps per scheduler: two for FP32 (222 registers; at 168 it spills, 1753 us
// per step), three for FP16.
constexpr int kin_pipe_warps(int prec) { return prec == P_FP16_DEV ? 3 : 2; }
template <int P, int MODE, bool AL>
__global__ void __launch_bounds__(32, 4 * kin_pipe_warps(P))
    kin_pipe_kernel(const typename Fmt<P>::S* src, typename Fmt<P>::S* dst,
                    int nx, int ny, long long ps, int strips, int seglen, Coll<float> c) {
    using T = typename Fmt<P>::S;
    using Q = typename PairOf<P>::T;
    constexpr int NF = MODE == 2 ? 5 : 4;
    constexpr bool PF = KinShared<P, AL>::PF;
    __shared__ KinShared<P, AL> sh;
    after_previous();
    const int strip = (int)(blockIdx.x % (unsigned)strips), seg = (int)(blockIdx.x / (unsigned)strips);
    const int y0 = seg * seglen, y1 = min(y0 + seglen, ny);
    const int lane = threadIdx.x;
    const int x = strip * kKinUseful - kKinHalo + 2 * lane;
    int xa = x % nx;
    if (xa < 0) xa += nx;
    const int xb = xa + 1 == nx ? 0 : xa + 1;
    const bool outa = x >= strip * kKinUseful && x < strip * kKinUseful + kKinUseful && x < nx;
    const bool outb = outa && x + 1 < nx;
    int rm = (y0 - 4) % ny, r0, rp;  // the first streamed row is y0 - 3
    if (rm < 0) rm += ny;
    r0 = rm + 1 == ny ? 0 : rm + 1;
    rp = r0 + 1 == ny ? 0 : r0 + 1;
    auto fetch = [&](Q(&z)[kPlanes]) { fetch_row<P, AL>(src, nx, ps, xa, xb, rm, r0, rp, ny, sh.pre, z); };

    Q h1[kPlanes], h2[kPlanes];           // the first step's results, c_y > 0
    float2 ma[2][NF], mb[2][NF], mc[NF];  // fields of each step's last two rows, and the new one
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
        for (int q = 0; q < NF; ++q) ma[k][q] = mb[k][q] = make_float2(1.0f, 1.0f);
    const int n = y1 - y0 + 6;
    unsigned orow = (unsigned)y0 * (unsigned)nx + (unsigned)x;
    Q z[kPlanes];
    if (PF) fetch(z);
#pragma unroll 1
    for (int it = 0; it < n; ++it) {
        if (PF) {
            cp_async_wait<0>();
#pragma unroll
            for (int p = 0; p < kPlanes; ++p) z[p] = sh.pre[p][lane];
            stream_row<P>(z);
            if (it + 1 < n) fetch(z);
        } else {
            fetch(z);
            stream_row<P>(z);
        }
        bool done = false;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            if (done) continue;
            if (k == 1) {  // the second step's streamed row from the first one's results
                stream_row<P>(z);
#pragma unroll
                for (int p = 0; p < kPlanes; ++p) {
                    const Q v = z[p];
                    if (plane_cy(p) == 0) {
                        z[p] = sh.keep[keep_slot(p)][lane];
                        sh.keep[keep_slot(p)][lane] = v;
                    } else if (plane_cy(p) > 0) {
                        z[p] = h2[p];
                        h2[p] = h1[p];
                        h1[p] = v;
                    }
                }
                if (it < 4) {
                    done = true;
                    continue;
                }
            }
            kin_fields<P, MODE>(z, c, mc);
#pragma unroll
            for (int p = 0; p < kPlanes; ++p) {  // the row before this one comes out
                const Q v = z[p];
                z[p] = sh.row[k][p][lane];
                sh.row[k][p][lane] = v;
            }
            if (it >= 4 * k + 2) kin_collide<P, MODE>(z, ma[k], mb[k], mc, c);
            else done = true;
#pragma unroll
            for (int q = 0; q < NF; ++q) {
                ma[k][q] = mb[k][q];
                mb[k][q] = mc[q];
            }
        }
        if (done) continue;
        if (outa) store_row<P, AL>(dst, ps, orow, outb, z);
        orow += (unsigned)nx;
    }
}

template <int P, int S, bool AL>
__global__ void __launch_bounds__(32, 4 * pipe_warps(sizeof(typename Fmt<P>::S), S))
    pipe_kernel(const typename Fmt<P>::S* src, typename Fmt<P>::S* dst,
                int nx, int ny, long long ps, int strips, int seglen, Coll<float> c) {
    __shared__ PipeShared<P, S, AL> sh;
    after_previous();
    const int strip = (int)(blockIdx.x % (unsigned)strips), seg = (int)(blockIdx.x / (unsigned)strips);
    const int y0 = seg * seglen;
    pipe_body<P, S, AL>(src, dst, nx, ny, ps, strip, y0, min(y0 + seglen, ny), c, sh);
}

// kPipeSteps steps of every run of an ensemble, a warp per strip-segment of a
// run, so every run gets the values of its own lattice.  Bound as above (ncu, 64
// runs of 512^2 FP32: 54% of the issue slots, 56% of the FMA pipe, 50% of DRAM).
template <int P, bool AL>
__global__ void __launch_bounds__(32, 4 * batch_pipe_warps(sizeof(typename Fmt<P>::S)))
    batch_pipe_kernel(const RunDev<float>* runs, const RunPass* pass,
                      const int* unit_run, const typename Fmt<P>::S* src,
                      typename Fmt<P>::S* dst) {
    __shared__ PipeShared<P, kPipeSteps, AL> sh;
    after_previous();
    const int r = unit_run[blockIdx.x];
    const RunDev<float>& rd = runs[r];
    const RunPass rp = pass[r];
    const int l = (int)(blockIdx.x - rp.unit0);
    const int strip = l % rp.strips, y0 = l / rp.strips * rp.seglen;
    const Coll<float> c = rd.c;
    pipe_body<P, kPipeSteps, AL>(src + rd.off, dst + rd.off, rd.nx, rd.ny, rd.ps, strip, y0,
                                 min(y0 + rp.seglen, rd.ny), c, sh);
}

template <int P, int S, bool AL>
cudaError_t launch_pipe_t(int seglen, const void* src, void* dst, const Geom& g, const HostColl& hc,
                          cudaStream_t st) {
    using T = typename Fmt<P>::S;
    const int strips = (g.nx + pipe_useful(S) - 1) / pipe_useful(S);
    const int nseg = (g.ny + seglen - 1) / seglen;
    return launch_after(pipe_kernel<P, S, AL>, (unsigned)strips * (unsigned)nseg, 32, st, (const T*)src,
                        (T*)dst, g.nx, g.ny, g.ps, strips, seglen, coll_for_prec<float>(hc, P));
}

template <int P>
cudaError_t launch_pipe_p(int steps, int seglen, const void* src, void* dst, const Geom& g,
                          const HostColl& c, cudaStream_t st) {
    const bool al = g.nx % 2 == 0;
    switch (steps) {
        case 2: return (al ? launch_pipe_t<P, 2, true> : launch_pipe_t<P, 2, false>)(seglen, src, dst, g, c, st);
        case 3: return (al ? launch_pipe_t<P, 3, true> : launch_pipe_t<P, 3, false>)(seglen, src, dst, g, c, st);
        case 4: return (al ? launch_pipe_t<P, 4, true> : launch_pipe_t<P, 4, false>)(seglen, src, dst, g, c, st);
    }
    return cudaErrorInvalidValue;
}

template <int P>
cudaError_t launch_kin_pipe_p(int seglen, const void* src, void* dst, const Geom& g, const HostColl& hc,
                              cudaStream_t st) {
    using T = typename Fmt<P>::S;
    const int strips = (g.nx + kKinUseful - 1) / kKinUseful;
    const bool al = g.nx % 2 == 0;
    auto k = hc.kin == 3 ? (al ? kin_pipe_kernel<P, 3, true> : kin_pipe_kernel<P, 3, false>)
                         : (al ? kin_pipe_kernel<P, 2, true> : kin_pipe_kernel<P, 2, false>);
    return launch_after(k, (unsigned)strips * (unsigned)((g.ny + seglen - 1) / seglen), 32, st,
                        (const T*)src, (T*)dst, g.nx, g.ny, g.ps, strips, seglen, coll_for_prec<float>(hc, P));
}

}  // namespace

cudaError_t launch_kin_pipe(int prec, int seglen, const void* src, void* dst, const Geom& g,
                            const HostColl& c, cudaStream_t st) {
    switch (prec) {
        case P_FP32: return launch_kin_pipe_p<P_FP32>(seglen, src, dst, g, c, st);
        case P_FP32_DEV: return launch_kin_pipe_p<P_FP32_DEV>(seglen, src, dst, g, c, st);
        case P_FP16_DEV: return launch_kin_pipe_p<P_FP16_DEV>(seglen, src, dst, g, c, st);
    }
    return cudaErrorInvalidValue;
}

static bool narrow(int prec) { return prec == P_FP32 || prec == P_FP32_DEV || prec == P_FP16_DEV; }
int pipe_steps(int prec, int nx, int ny, bool kin, int sm_count) {
    const int bytes = storage_bytes(prec);
    if (!narrow(prec)) return 0;
    if (kin) return kin_pipe_pays(bytes, nx, ny) ? kKinPipeSteps : 0;
    return pipe_pays(bytes, 1, &nx, &ny, false, sm_count) ? kPipeSteps : 0;
}
bool batch_pipe_pays(int prec, int nruns, const int* nx, const int* ny, int sm_count) {
    return narrow(prec) && pipe_pays(storage_bytes(prec), nruns, nx, ny, true, sm_count);
}

int pipe_seglen(int prec, int steps, int nx, int ny, bool kin, int sm_count) {
    const int bytes = storage_bytes(prec), useful = kin ? kKinUseful : pipe_useful(steps);
    const long long strips = (nx + useful - 1) / useful;
    // a kinetic closure: the rows around a segment and the time of a row are
    // about those of four steps
    return pipe_plan(kin ? kPipeSteps : steps, kin ? kin_pipe_warps(prec) : pipe_warps(bytes, steps), ny,
                     sm_count, [&](int len) { return strips * ((ny + len - 1) / len); })
        .seglen;
}

int batch_pipe_plan(int prec, int nruns, const int* nx, const int* ny, int sm_count, int* strips) {
    constexpr int U = pipe_useful(kPipeSteps);
    int most = 1;
    for (int r = 0; r < nruns; ++r) {
        strips[r] = (nx[r] + U - 1) / U;
        most = std::max(most, ny[r]);
    }
    return pipe_plan(kPipeSteps, batch_pipe_warps(storage_bytes(prec)), most, sm_count, [&](int len) {
        long long u = 0;
        for (int r = 0; r < nruns; ++r) u += (long long)strips[r] * ((ny[r] + len - 1) / len);
        return u;
    }).seglen;
}

cudaError_t launch_batch_pipe(int prec, bool even, const void* runs, const RunPass* pass, const int* unit_run,
                              unsigned nunits, const void* src, void* dst, cudaStream_t st) {
    const RunDev<float>* rd = (const RunDev<float>*)runs;
#define LBMHD_BP(P)                                                                           \
    case P:                                                                                   \
        return launch_after(even ? batch_pipe_kernel<P, true> : batch_pipe_kernel<P, false>, nunits, \
                            32, st, rd, pass, unit_run, (const Fmt<P>::S*)src, (Fmt<P>::S*)dst);
    switch (prec) {
        LBMHD_BP(P_FP32)
        LBMHD_BP(P_FP32_DEV)
        LBMHD_BP(P_FP16_DEV)
    }
#undef LBMHD_BP
    return cudaErrorInvalidValue;
}

cudaError_t launch_pipe(int prec, int steps, int seglen, const void* src, void* dst, const Geom& g,
                        const HostColl& c, cudaStream_t st) {
    switch (prec) {
        case P_FP32: return launch_pipe_p<P_FP32>(steps, seglen, src, dst, g, c, st);
        case P_FP32_DEV: return launch_pipe_p<P_FP32_DEV>(steps, seglen, src, dst, g, c, st);
        case P_FP16_DEV: return launch_pipe_p<P_FP16_DEV>(steps, seglen, src, dst, g, c, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace lbmhd
