// lb_kernels.cu -- the default two-pass timestep (phi pass, then the fused
// pull-collide-stream pass).
//
// Storage convention: the context keeps the post-collision, pre-streaming
// distributions A_i(x).  The post-streaming state of the model is the pull
// f_i(x, t) = A_i(x - c_i), so one timestep is "pull, collide at x, write
// A'_i(x)": every store is aligned to its own site and every load is a
// shifted, still coalesced read (targetDP Sec. III.B: SoA so consecutive
// sites are consecutive in memory).
#include <cuda_runtime.h>

#include <algorithm>

#include "d3q19.cuh"
#include "lb_internal.cuh"
#include "lb_pdl.cuh"
#include "lb_site.cuh"

namespace lbk {

// ------------------------------------------------------------------ two-pass step
// (both kernels launched with programmatic dependent launch, lb_pdl.cuh)

// phi = sum_i g_i(x - c_i) of V sites per thread (the paper's virtual vector
// length): the thread's sites are blockDim.x apart, their 19 V loads are
// issued before any sum.  A step that changes g by these passes takes back the
// moments flag (lb_ctx::moments, if any): a launch less than a memset
template <typename T, int V>
__global__ void __launch_bounds__(256) k_phi_pull(const T *__restrict__ ga, T *__restrict__ phi,
                                                  int *__restrict__ moments, int nx, int ny, int nz, long long S)
{
    pdl_wait_then_release();
    if (moments && blockIdx.x == 0 && threadIdx.x == 0) *moments = 0;
    const int N = nx * ny * nz;
    const int s0 = blockIdx.x * blockDim.x * V + threadIdx.x;
    T g[V][Q];
#pragma unroll
    for (int v = 0; v < V; v++) {
        const int s = s0 + v * (int)blockDim.x;
        if (s < N) {
            const Nbr n(s, nx, ny, nz);
#pragma unroll
            for (int i = 0; i < Q; i++) g[v][i] = ga[(size_t)i * S + n.src(i)];
        }
    }
#pragma unroll
    for (int v = 0; v < V; v++) {
        const int s = s0 + v * (int)blockDim.x;
        if (s < N) phi[s] = sum19(g[v]);
    }
}

// CTAs per SM the register budget of the collide/stream kernel must allow
// (measured: FP64 is bound by the FP64 pipe at 2 or 3; an allowance of 1
// lets ptxas spend 152 registers and loses 11 %; FP32 is DRAM-bound).
// Double-float with g unread (GEQ): without g's 38 words in flight 96
// registers do, in CTAs of 128 threads five to an SM -- 221 us a step at
// 144x120x100 against 255 with two CTAs of 256 and 240 with g read
// (arithmetic-bound either way: the 20 warps are what hides its latency).
// FP64 with tau = 1 too (FEQ), the gradient doubled (D2) and the edges of g
// from three products: 64^3, 50 steps with start and read-out 6.48 -> 5.87 ms.
#ifndef LBK_K2_MINB64
#define LBK_K2_MINB64 2
#endif
#ifndef LBK_K2_MINB32
#define LBK_K2_MINB32 3
#endif
#ifndef LBK_K2_MINBDF
#define LBK_K2_MINBDF 2
#endif
#ifndef LBK_K2_MINB32W
#define LBK_K2_MINB32W 3   // FP32 with the 19- / 27-point stencils
#endif
#ifndef LBK_K2_MINBDFG
#define LBK_K2_MINBDFG 5   // double-float, GEQ (of 128 threads)
#endif
#define LBK_K2_MAXT(T, GEQ) (is_df64<T>::value && (GEQ) ? 128 : 256)
#define LBK_K2_MINB(T, NP, GEQ)                                                                        \
    (is_df64<T>::value ? ((GEQ) ? LBK_K2_MINBDFG : LBK_K2_MINBDF) : sizeof(T) == 8 ? LBK_K2_MINB64   \
                                                                  : NP > 7 ? LBK_K2_MINB32W : LBK_K2_MINB32)

// GEQ: tau_g = 1, g is not read; FEQ: tau = 1 too (collide_site)
template <typename T, bool SH, int NP, bool GEQ, bool FEQ>
__global__ void __launch_bounds__(LBK_K2_MAXT(T, GEQ), LBK_K2_MINB(T, NP, GEQ)) k_collide_pull(const T *__restrict__ fa, const T *__restrict__ ga,
                                                      const T *__restrict__ phi,
                                                      T *__restrict__ fb, T *__restrict__ gb,
                                                      Coll<T> p, int nx, int ny, int nz, long long S)
{
    pdl_wait_then_release();
    const long long N = (long long)nx * ny * nz;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    const Nbr n(s, nx, ny, nz);
    collide_site<T, SH, NP, GEQ, FEQ>(fa, ga, phi, fb, gb, p, n, s, S);
}

// multiple-relaxation-time collision of f with a Guo body force (collide_mrt)
template <typename T, bool SH, int NP, bool GEQ>
__global__ void __launch_bounds__(LBK_K2_MAXT(T, GEQ), LBK_K2_MINB(T, NP, GEQ))
k_collide_pull_mrt(const T *__restrict__ fa, const T *__restrict__ ga, const T *__restrict__ phi,
                   T *__restrict__ fb, T *__restrict__ gb, Coll<T> p, Mrt<T> m, int nx, int ny, int nz,
                   long long S)
{
    pdl_wait_then_release();
    const long long N = (long long)nx * ny * nz;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    const Nbr n(s, nx, ny, nz);
    collide_site<T, SH, NP, GEQ>(fa, ga, phi, fb, gb, p, n, s, S, &m);
}

// ------------------------------------------------------------------ launchers

static inline unsigned grid_for(long long N, int tpb) { return (unsigned)((N + tpb - 1) / tpb); }

// Threads per CTA of both passes where the caller leaves them open; small
// lattices want small CTAs, which spread over the SMs.  Microseconds a step:
//   FP64 (bound by its instructions): 32 below 2^18 sites -- 16^3 19.8 at 256
//   threads, 10.8 at 32; 70x37x11 21.9 / 16.3 (tau, tau_g != 1 30.8 / 18.5);
//   32^3 23.2 / 17.8; 48^3 56.7 / 50.7; 56x52x60 84.9 / 74.0.  Above, 128 or
//   192, whichever leaves the busiest of the 152 SMs fewer sites: 64^3 114.5
//   at 256, 113.6 at 128, 109.8 at 192; 80^3 221.3, 213.6, 214.1; 100^3 407.1,
//   405.5, 409.2.
//   FP32: 128 below 2^20 sites -- 16^3 4.28 at 256 / 3.55, 64^3 12.97 / 12.23
//   (tau_g != 1 13.9 / 13.5), 80^3 26.6 / 26.0 (30.3 / 29.9) -- and 256 above,
//   where 128 lose up to 2 % (160^3 234.6 / 239.5); but where 152 SMs have one
//   or two CTAs of 128 each the uneven share shows: 32 from 3 x 2^13 to 3 x 2^14
//   sites -- 30^3 4.48 at 128 / 4.52 (tau_g != 1 4.92 / 4.55), 32^3 4.74 / 4.59
//   (5.22 / 4.79; 4.75 at 256), 34^3 5.57 / 4.97 (5.64 / 5.41), 36^3 5.73 / 5.09
//   (6.17 / 5.50) -- and from there to 2^17 160 where g is not read: 38^3 6.28 /
//   5.40, 40^3 6.75 / 5.68 (at 256, reading g, 6.36), 42^3 6.69 / 6.50, 46^3 8.17 /
//   7.73; 52^3 8.11 / 8.80 (with g read 42^3 6.27 / 7.49).
//   Double-float: 64 below 2^18 sites (16^3 to 56x52x60 3 to 8 % with tau_g
//   != 1, 1 % without), 256 above (128x128x64 152.3 / 155.4).
template <typename T>
static int default_threads(long long N, bool geq = false)
{
    const bool small = N < (1LL << 18);
    if (is_df64<T>::value) return small ? 64 : 256;
    if (sizeof(T) == 4) {
        if (N >= 3 << 13 && N < 3 << 14) return 32;
        if (geq && N >= 3 << 14 && N <= 1 << 17) return 160;
        return N < (1LL << 20) ? 128 : 256;
    }
    if (small) return 32;
    auto busiest = [&](int tpb) { return ((N + tpb - 1) / tpb + 151) / 152 * tpb; };
    return busiest(192) < busiest(128) ? 192 : 128;
}

int fp64_threads(long long N) { return default_threads<double>(N); }

// the phi pass with V sites per thread
template <typename T>
static cudaError_t launch_phi(lb_ctx *c, const T *ga, T *phi, int tpb, int vvl)
{
    const int nx = c->p.nx, ny = c->p.ny, nz = c->p.nz;
    const unsigned grid = grid_for(c->N, tpb * vvl);
    const auto kernel = vvl == 4 ? k_phi_pull<T, 4> : vvl == 2 ? k_phi_pull<T, 2> : k_phi_pull<T, 1>;
    return launch_pdl(kernel, grid, tpb, c->stream, ga, phi, c->moments, nx, ny, nz, c->S);
}

// the collide/stream pass from level fa, ga (and phi of the state) to fb, gb
template <typename T, bool SH, int NP, bool GEQ>
static cudaError_t launch_collide(lb_ctx *c, const T *fa, const T *ga, const T *phi, T *fb, T *gb, int tpb)
{
    const auto p = make_coll<T>(c->p);
    tpb = std::min(tpb, LBK_K2_MAXT(T, GEQ));
    const unsigned grid = grid_for(c->N, tpb);
    const int nx = c->p.nx, ny = c->p.ny, nz = c->p.nz;
    if (uses_mrt(c))
        return launch_pdl(k_collide_pull_mrt<T, SH, NP, GEQ && !is_df64<T>::value>, grid, tpb, c->stream, fa, ga, phi, fb, gb, p,
                          make_mrt<T>(c), nx, ny, nz, c->S);
    if constexpr (GEQ && sizeof(T) == 8)
        if (f_is_equilibrium(c->p))
            return launch_pdl(k_collide_pull<T, SH, NP, true, true>, grid, tpb, c->stream, fa, ga, phi, fb, gb, p, nx,
                              ny, nz, c->S);
    return launch_pdl(k_collide_pull<T, SH, NP, GEQ, false>, grid, tpb, c->stream, fa, ga, phi, fb, gb, p, nx, ny, nz,
                      c->S);
}

// tau_g = 1: the collide pass does not read g, except in double-float with the
// multiple relaxation times, whose collision does not fit the 96 registers
// that pay there (144x120x100 338 us a step against 321 with g read), and where
// the caller asks for more threads than that collision is compiled for (128 in
// double-float: 222.7 us a step; 240.4 with g read in CTAs of 256)
template <typename T>
static bool leaves_g_unread(const lb_ctx *c)
{
    return g_is_equilibrium(c->p) && !(is_df64<T>::value && uses_mrt(c)) && c->block_x <= LBK_K2_MAXT(T, true);
}

template <typename T, bool SH, int NP>
static int two_pass(lb_ctx *c, int nsteps)
{
    // launch shape: threads per CTA of both passes, sites per thread of the
    // phi pass (lb_set_kernel's block_x, block_y; 0 = default_threads, cut to
    // the collision's limit there, and 1)
    const int tpb = c->block_x ? c->block_x : default_threads<T>(c->N, leaves_g_unread<T>(c));
    const int vvl = c->block_y ? c->block_y : 1;
    for (int t = 0; t < nsteps; t++) {
        const int a = c->buf.cur, b = 1 - a;
        const T *fa = (const T *)c->buf.f[a], *ga = (const T *)c->buf.g[a], *phi = (const T *)c->phi;
        T *fb = (T *)c->buf.f[b], *gb = (T *)c->buf.g[b];
        cudaError_t e = launch_phi<T>(c, ga, (T *)c->phi, tpb, vvl);
        if (e == cudaSuccess)
            e = leaves_g_unread<T>(c) ? launch_collide<T, SH, NP, true>(c, fa, ga, phi, fb, gb, tpb)
                                      : launch_collide<T, SH, NP, false>(c, fa, ga, phi, fb, gb, tpb);
        int rc = e != cudaSuccess ? cuda_status(e) : check_launch();
        if (rc) return rc;
        c->buf.cur = b;
    }
    return LB_OK;
}

int launch_two_pass_fp64_raw(const lb_params &prm, const double *fa, const double *ga, double *phi, double *fb,
                             double *gb, long long S, cudaStream_t stream)
{
    const auto p = make_coll<double>(prm);
    const long long N = (long long)prm.nx * prm.ny * prm.nz;
    const int tpb = default_threads<double>(N);
    const unsigned grid = grid_for(N, tpb);
    k_phi_pull<double, 1><<<grid, tpb, 0, stream>>>(ga, phi, nullptr, prm.nx, prm.ny, prm.nz, S);
    const auto collide = !g_is_equilibrium(prm)  ? k_collide_pull<double, false, 7, false, false>
                         : f_is_equilibrium(prm) ? k_collide_pull<double, false, 7, true, true>
                                                 : k_collide_pull<double, false, 7, true, false>;
    collide<<<grid, tpb, 0, stream>>>(fa, ga, phi, fb, gb, p, prm.nx, prm.ny, prm.nz, S);
    return check_launch();
}

template <typename T, bool SH>
static int two_pass_t(lb_ctx *c, int nsteps)
{
    if (c->npts == 19) return two_pass<T, SH, 19>(c, nsteps);
    if (c->npts == 27) return two_pass<T, SH, 27>(c, nsteps);
    return two_pass<T, SH, 7>(c, nsteps);
}

int two_pass_validate(int block_x, int block_y, int z_chunk)
{
    if (block_x != 0 && (block_x % 32 != 0 || block_x < 32 || block_x > 256)) return LB_ERR_INVALID;
    if (block_y != 0 && block_y != 1 && block_y != 2 && block_y != 4) return LB_ERR_INVALID;
    return z_chunk == 0 ? LB_OK : LB_ERR_INVALID;
}

int launch_step_two_pass(lb_ctx *c, int nsteps)
{
    return by_precision(c, [&](auto P) { return two_pass_t<typename decltype(P)::T, decltype(P)::SH>(c, nsteps); });
}

}  // namespace lbk
