// lb_taug1.cu -- the timestep for tau_g = 1, keeping g as its moments.
//
// With tau_g = 1 the collision of g returns its equilibrium exactly,
// g*_i = geq_i(phi, mu, u), so after streaming g_i(x, t+1) = geq_i evaluated
// with (phi, mu, u) of site x - c_i at time t, and phi(x, t+1) is the sum of
// those 19 values.  The context then keeps, instead of 19 values of g, five
// per site in its g buffers:
//     level a: component 0      phi(t)  (the stencil's input)
//              components 1..4  the quad (gmh, u_x, u_y, u_z) of each site,
//                               interleaved (one 16 B / 32 B vector per
//                               site), gmh = 9/2 (Gamma mu - phi/3)
// With P = phi (1 - 3/2 u^2) the equilibrium is then
//     geq_i = w_i [P + gmh (c_i^2 - 1) + c_i.u (3 phi + 9/2 phi c_i.u)].
// One step is two passes:
//   k_t1_collide  pull f, 7-point stencil of phi(t), collide f; write f* and
//                 gmh(t), u(t) next to phi(t)        (19+1 r, 19+4 w words)
//   k_t1_phi      phi(x, t+1) = sum_i geq_i(moments at x - c_i) into the
//                 other level's component 0          (5 r, 1 w words)
// -- 49 words per site instead of the 97 of the general two-pass step.
// k_t1_phi streams along z so that each source site's moments are loaded and
// expanded about once: a warp covers 32 consecutive positions of the rows
// (with halo positions between them, t1_phi_tile) of which the 30 inner ones
// are outputs (the outer two only feed their neighbours); each
// lane walks a run of z planes for KY rows of its column, holding the
// partial sums of the three output planes a source plane reaches.  Sources
// in the lane's own column (c_x = 0) add to its own outputs; those with
// c_x = +-1 add to per-output partial sums that one shuffle each hands to
// lane +-1 once the output plane is complete.
// The per-site arithmetic is the general collision's (the g relaxation is
// simply not needed); results agree with the general step to rounding.
//
// Flag m_valid: (mu, u) of the previous step are present.  After lb_init or
// lb_set_state only phi(t) is known; g is then reported as the equilibrium at
// each site (exact after lb_init, which starts from that equilibrium).
#include <cuda_runtime.h>

#include <atomic>
#include <type_traits>
#include <utility>

#include "d3q19.cuh"
#include "lb_internal.cuh"
#include "lb_pdl.cuh"
#include "lb_site.cuh"
#include "lb_t1.cuh"

namespace lbk {

namespace {

constexpr int kT1Threads = 256;

template <typename T, bool SH, int NP>
__global__ void __launch_bounds__(kT1Threads, sizeof(T) == 8 ? 2 : 3)
k_t1_collide(const T *__restrict__ fa, const T *__restrict__ phi, T *__restrict__ quad, T *__restrict__ fb,
             Coll<T> p, int nx, int ny, int nz, long long S)
{
    pdl_wait_then_release();
    const long long N = (long long)nx * ny * nz;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    t1_collide_site<T, SH, NP>(fa, phi, quad, fb, p, nx, ny, nz, S, s);
}

// The same on a general state (run_geq).  With gb, a call's last step: g* = geq
// in full as well, phi in the phi buffer (keep, if it is not there) and the
// flag that quads and phi are at hand.  One kernel for a call's last step and
// the others, since two kernels' products and sums need not be contracted
// alike and a run's bits would depend on where its calls end.  MRT: the
// multiple relaxation times or a body force.
template <int NP, bool MRT>
__global__ void __launch_bounds__(kT1Threads, 3)
k_geq_collide(const float *__restrict__ fa, const float *__restrict__ phi, float *__restrict__ quad,
              float *__restrict__ fb, float *__restrict__ gb, float *__restrict__ keep, int *__restrict__ moments,
              Coll<float> p, Mrt<float> m, int nx, int ny, int nz, long long S)
{
    pdl_wait_then_release();
    const long long N = (long long)nx * ny * nz;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    t1_collide_site<float, true, NP>(fa, phi, quad, fb, p, nx, ny, nz, S, s, MRT ? &m : nullptr, gb);
    if (!gb) return;
    if (keep) keep[s] = phi[s];
    if (s == 0) *moments = 1;
}

constexpr int kPhiWarps = 4;      // default warps per block, stacked in y
constexpr int kPhiMaxWarps = 8;

template <typename T, int KY>
__global__ void __launch_bounds__(32 * kPhiMaxWarps) k_t1_phi(const T *__restrict__ phi,
                                                               const T *__restrict__ quad, T *__restrict__ phi_out,
                                                               int nx, int ny, int nz, int kzc)
{
    pdl_wait_then_release();
    t1_phi_tile<T, KY>(phi, quad, phi_out, nx, ny, nz, kzc, blockIdx.x, blockDim.y, threadIdx.y, blockIdx.y,
                       threadIdx.x);
}

// The phi pass on a general state (run_geq); one kernel for all of a run's, as
// k_geq_collide.  With ga, a call's first: phi and the quads may not be at hand
// (*moments), and phi is the sum of the stored g then.  phi_out may be row 0
// of ga, which only its own site reads (so neither is declared __restrict__).
// The bounds are the registers that k_t1_phi takes by itself, 64 and 80: with
// the sum beside it ptxas takes 54 for one row (80^3 20.0 instead of 19.6 us a
// step), and one CTA in place of 6 costs two rows 4 % (256^3 536 / 516).
template <int KY>
__global__ void __launch_bounds__(32 * kPhiWarps, KY == 1 ? 8 : 6)
k_geq_phi(const float *ga, const int *moments, const float *phi, const float *quad, float *phi_out, int nx, int ny,
          int nz, int kzc, long long S)
{
    pdl_wait_then_release();
    if (ga && !*moments) {
        const int N = nx * ny * nz, threads = 32 * blockDim.y;
        const long long stride = (long long)gridDim.x * gridDim.y * threads;
        for (long long s = (long long)(blockIdx.y * gridDim.x + blockIdx.x) * threads + threadIdx.y * 32 + threadIdx.x;
             s < N; s += stride)
            phi_out[s] = phi_site(ga, Nbr((int)s, nx, ny, nz), S);
        return;
    }
    t1_phi_tile<float, KY>(phi, quad, phi_out, nx, ny, nz, kzc, blockIdx.x, blockDim.y, threadIdx.y, blockIdx.y,
                           threadIdx.x);
}

// g state of the reduced form as post-streaming FP64 rows [i0, i1):
// streamed equilibria of the previous step's moments (m_valid), else the
// equilibrium at each site from phi(t), its stencil and u from f.
template <typename T, bool SH, int NP>
__global__ void __launch_bounds__(kT1Threads) k_t1_g_state(const T *__restrict__ fa, const T *__restrict__ gcur,
                                                            const T *__restrict__ gprev, int m_valid, Coll<T> p,
                                                            double *__restrict__ out, int i0, int i1, int nx,
                                                            int ny, int nz, long long S)
{
    const long long N = (long long)nx * ny * nz;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    const Nbr n(s, nx, ny, nz);
    if (m_valid) {
#pragma unroll
        for (int i = 0; i < Q; i++) {
            if (i < i0 || i >= i1) continue;
            out[(size_t)(i - i0) * N + s] = double(geq_eq(i, load_eq(gprev, S, n.src(i))));
        }
        return;
    }
    double f[Q];
#pragma unroll
    for (int i = 0; i < Q; i++) f[i] = double(fa[(size_t)i * S + n.src(i)]);
    double R, jx, jy, jz;
    density_moments(f, R, jx, jy, jz);
    const double rho = SH ? double(p.rho0) + R : R;
    const double ph = double(gcur[s]);
    double dx, dy, dz, lap;
    stencil_np<NP, double>(gcur, n, ph, dx, dy, dz, lap);
    const double mu = ph * (double(p.A) + double(p.B) * ph * ph) - double(p.kappa) * lap;
    const Eq<double> e = make_eq(ph, gmh_of(ph, mu, double(p.gamma)), jx / rho, jy / rho, jz / rho);
#pragma unroll
    for (int i = 0; i < Q; i++) {
        if (i < i0 || i >= i1) continue;
        out[(size_t)(i - i0) * N + s] = geq_eq(i, e);
    }
}

// phi(t) of a full-form state (pull sum of g) into component 0 of level b
template <typename T>
__global__ void __launch_bounds__(kT1Threads) k_t1_from_full(const T *__restrict__ ga, T *__restrict__ phi_out,
                                                              int nx, int ny, int nz, long long S)
{
    const long long N = (long long)nx * ny * nz;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    const Nbr n(s, nx, ny, nz);
    phi_out[s] = phi_site(ga, n, S);
}

// full-form g (post-collision storage) from the reduced form: A_i(x - c_i) =
// the g state at x.  gcur is phi(t) (a copy: gout is the current level)
template <typename T, bool SH, int NP>
__global__ void __launch_bounds__(kT1Threads) k_t1_to_full(const T *__restrict__ fa, const T *__restrict__ gcur,
                                                            const T *__restrict__ gprev, int m_valid, Coll<T> p,
                                                            T *__restrict__ gout, int nx, int ny, int nz, long long S)
{
    const long long N = (long long)nx * ny * nz;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    const Nbr n(s, nx, ny, nz);
    double f[Q];
#pragma unroll
    for (int i = 0; i < Q; i++) f[i] = double(fa[(size_t)i * S + n.src(i)]);
    double R, jx, jy, jz;
    density_moments(f, R, jx, jy, jz);
    const double rho = SH ? double(p.rho0) + R : R;
    const double ph = double(gcur[s]);
    double dx, dy, dz, lap;
    stencil_np<NP, double>(gcur, n, ph, dx, dy, dz, lap);
    const double mu = ph * (double(p.A) + double(p.B) * ph * ph) - double(p.kappa) * lap;
    const Eq<double> own = make_eq(ph, gmh_of(ph, mu, double(p.gamma)), jx / rho, jy / rho, jz / rho);
#pragma unroll
    for (int i = 0; i < Q; i++) {
        double v;
        if (m_valid)
            v = double(geq_eq(i, load_eq(gprev, S, n.src(i))));
        else
            v = geq_eq(i, own);
        gout[(size_t)i * S + n.src(i)] = T(v);
    }
}

template <typename T>
__global__ void __launch_bounds__(kT1Threads) k_t1_copy_phi(const T *__restrict__ phi_src, T *__restrict__ dst,
                                                            long long N)
{
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s < N) dst[s] = phi_src[s];
}

inline unsigned grid_of(long long N) { return (unsigned)((N + kT1Threads - 1) / kT1Threads); }

// resident CTAs per SM of a phi-pass kernel and block size
template <typename K>
int blocks_per_sm(K kernel, int threads, int smem, std::atomic<int> &cache, int *bps)
{
    int b = cache.load(std::memory_order_relaxed);
    if (!b) {
        const int rc = cuda_status(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, threads, smem));
        if (rc) return rc;
        b = b > 0 ? b : 1;
        cache.store(b, std::memory_order_relaxed);
    }
    *bps = b;
    return LB_OK;
}

// z run of the phi pass: the launch's choice, else by the resident blocks
// (phi_run_length)
int phi_z_run(lb_ctx *c, long long columns, int bps, int *kzc)
{
    int z = c->z_chunk;
    if (!z) {
        int dev = 0, sms = 0;
        int rc = cuda_status(cudaGetDevice(&dev));
        if (!rc) rc = cuda_status(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        if (rc) return rc;
        z = phi_run_length(columns, c->p.nz, (long long)sms * bps);
    }
    *kzc = z > c->p.nz ? c->p.nz : z;
    return LB_OK;
}

// launch shape of a phi pass: KY rows a lane, block_warps warps a CTA (0: the default)
template <int KY>
struct PhiLaunch {
    dim3 grid, block;
    int kzc = 0;

    template <typename K>
    int plan(lb_ctx *c, K kernel, int block_warps, std::atomic<int> (&cache)[kPhiMaxWarps + 1])
    {
        const int nx = c->p.nx, ny = c->p.ny, nz = c->p.nz;
        const int warps = block_warps ? block_warps : kPhiWarps;
        const int gxy = phi_blocks(nx, ny, KY, warps);
        int bps = 0;
        int rc = blocks_per_sm(kernel, 32 * warps, 0, cache[warps], &bps);
        if (!rc) rc = phi_z_run(c, gxy, bps, &kzc);
        grid = dim3(gxy, (nz + kzc - 1) / (kzc ? kzc : 1));
        block = dim3(32, warps);
        return rc;
    }
};

template <typename T, bool SH, int NP, int KY>
int run_t1(lb_ctx *c, int nsteps)
{
    static std::atomic<int> cache[kPhiMaxWarps + 1];
    PhiLaunch<KY> phi;
    int rc = phi.plan(c, k_t1_phi<T, KY>, c->block_y, cache);
    if (rc) return rc;
    const auto p = make_coll<T>(c->p);
    const int nx = c->p.nx, ny = c->p.ny, nz = c->p.nz;
    for (int t = 0; t < nsteps; t++) {
        const int a = c->buf.cur, b = 1 - a;
        T *ga = (T *)c->buf.g[a], *quad = quads(ga, c->S);   // phi in row 0
        cudaError_t e = launch_pdl(k_t1_collide<T, SH, NP>, grid_of(c->N), kT1Threads, c->stream,
                                   (const T *)c->buf.f[a], (const T *)ga, quad, (T *)c->buf.f[b], p, nx, ny, nz, c->S);
        if (e == cudaSuccess)
            e = launch_pdl(k_t1_phi<T, KY>, phi.grid, phi.block, c->stream, (const T *)ga, (const T *)quad,
                           (T *)c->buf.g[b], nx, ny, nz, phi.kzc);
        rc = e != cudaSuccess ? cuda_status(e) : check_launch();
        if (rc) return rc;
        c->buf.cur = b;
        c->m_valid = 1;
    }
    return LB_OK;
}

// y rows a lane of the phi pass in FP32: two from 2^20 sites on (us a step:
// 128^3 68.2 against 70.1, 256^3 513 / 529, 200x152x136 131.2 / 137.1; below,
// one: 129x97x65 31.5 / 31.0, 96^3 33.4 / 33.5), one where the lattice has
// fewer than four rows.
int phi_rows(const lb_ctx *c) { return c->N >= (1LL << 20) && c->p.ny >= 4 ? 2 : 1; }

template <typename T, bool SH, int NP>
int run_t1_ky(lb_ctx *c, int nsteps)
{
    const int rows = std::is_same<T, float>::value ? phi_rows(c) : PhiTile<T>::KY;
    switch (c->block_x ? c->block_x : rows) {
    case 1: return run_t1<T, SH, NP, 1>(c, nsteps);
    case 2: return run_t1<T, SH, NP, 2>(c, nsteps);
    case 4:
        if constexpr (is_df64<T>::value) return LB_ERR_INVALID;   // spills at four rows
        else return run_t1<T, SH, NP, 4>(c, nsteps);
    default: return LB_ERR_INVALID;
    }
}

}  // namespace

template <typename T, bool SH>
int run_t1_t(lb_ctx *c, int nsteps)
{
    if (c->npts == 19) return run_t1_ky<T, SH, 19>(c, nsteps);
    if (c->npts == 27) return run_t1_ky<T, SH, 27>(c, nsteps);
    return run_t1_ky<T, SH, 7>(c, nsteps);
}

template <typename T, bool SH, int NP>
void to_full(lb_ctx *c)
{
    const int cur = c->buf.cur, oth = 1 - cur;
    k_t1_copy_phi<T><<<grid_of(c->N), kT1Threads, 0, c->stream>>>((const T *)c->buf.g[cur], (T *)c->phi, c->N);
    k_t1_to_full<T, SH, NP><<<grid_of(c->N), kT1Threads, 0, c->stream>>>(
        (const T *)c->buf.f[cur], (const T *)c->phi, (const T *)c->buf.g[oth], c->m_valid,
        make_coll<T>(c->p), (T *)c->buf.g[cur], c->p.nx, c->p.ny, c->p.nz, c->S);
}

template <typename T, bool SH>
void to_full_t(lb_ctx *c)
{
    if (c->npts == 19)
        to_full<T, SH, 19>(c);
    else if (c->npts == 27)
        to_full<T, SH, 27>(c);
    else
        to_full<T, SH, 7>(c);
}

template <typename T, bool SH, int NP>
void g_rows(lb_ctx *c, int i0, int i1, double *out)
{
    const int cur = c->buf.cur, oth = 1 - cur;
    k_t1_g_state<T, SH, NP><<<grid_of(c->N), kT1Threads, 0, c->stream>>>(
        (const T *)c->buf.f[cur], (const T *)c->buf.g[cur], (const T *)c->buf.g[oth], c->m_valid,
        make_coll<T>(c->p), out, i0, i1, c->p.nx, c->p.ny, c->p.nz, c->S);
}

template <typename T, bool SH>
void g_rows_t(lb_ctx *c, int i0, int i1, double *out)
{
    if (c->npts == 19)
        g_rows<T, SH, 19>(c, i0, i1, out);
    else if (c->npts == 27)
        g_rows<T, SH, 27>(c, i0, i1, out);
    else
        g_rows<T, SH, 7>(c, i0, i1, out);
}

// FP32-shifted steps of a general (19-value) state with tau_g = 1.  Within
// one call g's 19 values are only wanted at its end: the steps are the reduced
// form's two passes on scratch in the g level that the call does not end in,
// and the last step's collision writes g* = geq in full too.  The stored state
// between calls stays the general one.
// The first phi is the sum of the stored g after a new start (init,
// set_state, steps of another kernel), else the phi pass over the last step's
// phi (kept in the phi buffer) and quads (in the spare g level), so that the
// bits of a run do not depend on how it is cut into calls.  Which it is stands
// in device memory (lb_ctx::moments, cleared on the stream by every call that
// writes the state), so that captured steps do not fix it.  n steps move
// 6 + 49 (n - 1) + 64 words a site (20 + 49 (n - 1) + 64 after a new start)
// instead of 76 n (the bulk kernel) or 97 n (two passes).
template <int NP, int KY>
static int run_geq(lb_ctx *c, int nsteps)
{
    static std::atomic<int> cache[kPhiMaxWarps + 1];
    PhiLaunch<KY> pass;
    int rc = pass.plan(c, k_geq_phi<KY>, 0, cache);
    if (rc) return rc;
    const auto collide = uses_mrt(c) ? k_geq_collide<NP, true> : k_geq_collide<NP, false>;
    const auto p = make_coll<float>(c->p);
    const auto m = make_mrt<float>(c);
    const int nx = c->p.nx, ny = c->p.ny, nz = c->p.nz;
    int a = c->buf.cur;
    const int last = (a + nsteps) & 1;
    float *kept = (float *)c->phi;
    float *scratch = (float *)c->buf.g[1 - last];   // g(t) itself where nsteps is odd, until its phi is summed
    float *quad = quads(scratch, c->S);
    // phi(t) stands in row 0 of scratch and in the phi buffer by turns
    float *phi = scratch, *next = kept;
    auto phi_pass = [&](const float *ga, const float *from, const float *q, float *to) {
        return launch_pdl(k_geq_phi<KY>, pass.grid, pass.block, c->stream, ga, (const int *)c->moments, from, q, to,
                          nx, ny, nz, pass.kzc, c->S);
    };
    cudaError_t e = phi_pass((const float *)c->buf.g[a], kept, quads((float *)c->buf.g[1 - a], c->S), phi);
    for (int t = 0; t < nsteps && e == cudaSuccess; t++, a = 1 - a) {
        const bool ends = t + 1 == nsteps;
        e = launch_pdl(collide, grid_of(c->N), kT1Threads, c->stream, (const float *)c->buf.f[a], (const float *)phi,
                       quad, (float *)c->buf.f[1 - a], ends ? (float *)c->buf.g[last] : nullptr,
                       phi == kept ? nullptr : kept, c->moments, p, m, nx, ny, nz, c->S);
        if (ends || e != cudaSuccess) break;
        e = phi_pass(nullptr, phi, quad, next);
        std::swap(phi, next);
    }
    rc = e != cudaSuccess ? cuda_status(e) : check_launch();
    if (rc) return rc;
    c->buf.cur = last;
    return LB_OK;
}

template <int KY>
static int run_geq_np(lb_ctx *c, int nsteps)
{
    if (c->npts == 19) return run_geq<19, KY>(c, nsteps);
    if (c->npts == 27) return run_geq<27, KY>(c, nsteps);
    return run_geq<7, KY>(c, nsteps);
}

// When the library default takes these steps.  The phi pass gains by the words
// that it saves and loses by its latency -- warps walk along z -- and by the
// lanes that write nothing: of the positions of a row nx of nx + 2 do, of the
// rows of a CTA's warps ny of a multiple of them.  Microseconds a step over 50
// steps and in calls of one, against two passes that leave g unread (78 words
// a site; with g read, the default until these steps were there, in brackets):
//   256^3 516 and 713 / 770 (904), 128^3 68.9 and 93.8 / 103 (121), 80^3 19.6
//   and 27.5 / 25.8 (30.4), 72^3 15.3 and 20.6 / 18.0 (21.5), 68^3 14.1 and 18.3
//   / 14.9 (17.8), 64^3 12.5 and 15.1 / 12.1 (13.8), 48^3 9.1 and 10.5 / 8.2;
//   rows of 2, 4, 8 sites (2^20 sites) 44.9, 40.9, 39.9 and 57.4, 53.5, 52.6 /
//   52.3 (61.4);  600x3x300 22.4 and 30.5 / 27.5 (32.0), 128x5x600 17.0 and 22.6
//   / 18.4 (21.9), 600x2x300 17.7 and 22.8 / 17.3 (20.7);
//   1024x1x1024 57.6 and 70.5 / 53.0 (61.0), 16x1x60000 75.6 and 87.6 / 48.0 (56);
//   one plane, read three times for one written: 600x600 17.3 and 22.1 / 17.3
//   (20.4), 1200x1200 67.8 and 84.6 / 72.5 (84.3), 2000x2000 173 and 219 / 193
//   (228), 12x99000 60.3 and 74.5 / 60.6 (69.7).
// FP64 and double-float steps are bound by arithmetic, of which the reduced
// form's phi pass has more; they take the two passes.
bool auto_uses_geq(const lb_ctx *c)
{
    if (c->p.precision != LB_FP32_SHIFTED || !g_is_equilibrium(c->p)) return false;
    const int rows = phi_rows(c) * kPhiWarps, nx = c->p.nx, ny = c->p.ny;
    const double writing = double(nx) / (nx + 2.0) * ny / (double(ny - 1 - (ny - 1) % rows) + rows);
    const bool plane = c->p.nz == 1;
    return writing >= (plane ? 0.9 : 0.45) && writing * c->N >= (plane ? 1 << 20 : 5 << 16);
}

int launch_step_geq(lb_ctx *c, int nsteps)
{
    return phi_rows(c) == 2 ? run_geq_np<2>(c, nsteps) : run_geq_np<1>(c, nsteps);
}

int taug1_validate(const lb_params &p, int block_x, int block_y, int z_chunk)
{
    if (p.tau_g != 1.0) return LB_ERR_INVALID;
    if (block_x != 0 && block_x != 1 && block_x != 2 && block_x != 4) return LB_ERR_INVALID;
    if (block_x == 4 && p.precision == LB_FP64_DF) return LB_ERR_INVALID;
    if (block_y < 0 || block_y > kPhiMaxWarps || z_chunk < 0) return LB_ERR_INVALID;
    return LB_OK;
}

int launch_step_taug1(lb_ctx *c, int nsteps)
{
    return by_precision(c, [&](auto P) { return run_t1_t<typename decltype(P)::T, decltype(P)::SH>(c, nsteps); });
}

// convert the stored state between the full and the reduced form
int taug1_convert(lb_ctx *c, int to_reduced)
{
    const int cur = c->buf.cur;
    const unsigned grid = grid_of(c->N);
    const int nx = c->p.nx, ny = c->p.ny, nz = c->p.nz;
    return by_precision(c, [&](auto P) {
        using T = typename decltype(P)::T;
        if (to_reduced) {
            // phi(t) into the phi scratch, then into component 0 of level cur
            k_t1_from_full<T><<<grid, kT1Threads, 0, c->stream>>>((const T *)c->buf.g[cur], (T *)c->phi, nx, ny, nz,
                                                                  c->S);
            k_t1_copy_phi<T><<<grid, kT1Threads, 0, c->stream>>>((const T *)c->phi, (T *)c->buf.g[cur], c->N);
            c->m_valid = 0;
        } else {
            // back to the full form: phi(t) into the phi scratch, then the 19
            // values of g rebuilt into the current level (the previous step's
            // moments are read from the other level)
            to_full_t<T, decltype(P)::SH>(c);
        }
        const int rc = check_launch();
        return rc ? rc : state_written(c);
    });
}

template <typename T>
__global__ void __launch_bounds__(kT1Threads) k_t1_phi_out(const T *__restrict__ phi, double *__restrict__ out,
                                                           long long N)
{
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s < N) out[s] = double(phi[s]);
}

int taug1_phi_out(lb_ctx *c, double *out)
{
    const unsigned grid = grid_of(c->N);
    const int cur = c->buf.cur;
    return by_precision(c, [&](auto P) {
        using T = typename decltype(P)::T;
        k_t1_phi_out<T><<<grid, kT1Threads, 0, c->stream>>>((const T *)c->buf.g[cur], out, c->N);
        return check_launch();
    });
}

int taug1_g_rows(lb_ctx *c, int i0, int i1, double *out)
{
    return by_precision(c, [&](auto P) {
        g_rows_t<typename decltype(P)::T, decltype(P)::SH>(c, i0, i1, out);
        return check_launch();
    });
}

}  // namespace lbk
