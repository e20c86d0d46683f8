// lb_adjoint.cu -- reverse mode of the FP64 timestep (a kernel pair) and of
// the initialisation, for gradients of a loss on phi_T.
//
// States are in the ABI (post-streaming) convention, so the forward
// quantities of F(t) are local to each site.  Per reverse step:
//   k_phi_local   phi(x) = sum_i g_i(x, t)
//   k_adj_collide at x: recompute rho, j, u, mu, the stress; gather the
//                 adjoint after streaming, fs_bar_i(x) = f_bar_i(x + c_i, t+1);
//                 apply the collision's vector-Jacobian product; write
//                 f_bar(x, t), the direct part of g_bar, and the adjoints of
//                 phi, grad phi and lap phi at x; per-CTA partial dJ/dkappa
//   k_adj_stencil phi_bar(x) = local part + transposed 7-point stencils;
//                 g_bar_i(x, t) += phi_bar(x); the sum of the partial dJ/dkappa
// (launched with programmatic dependent launch, lb_pdl.cuh).
// The equilibrium VJP sums each opposite pair (i+, i-) once: its even part
// feeds rho and the stress, its odd part the momentum.
#include <cuda_runtime.h>

#include <cmath>

#include "d3q19.cuh"
#include "lb_internal.cuh"
#include "lb_pdl.cuh"
#include "lb_site.cuh"

namespace lbk {

namespace {

// Model parameters, and the relaxation rate folded into the factors of the
// weight sums below (formed on the host): R = w/36, O = w/12 (3 w/36),
// T = w/8 (9/2 w/36), W = w/24 (3/2 w/36), w the rate of f or of g.  R and W in two
// parts: an adjoint that is the same for all velocities is multiplied by 36 R in
// every step and has no stress, 12 T = 36 W, and with each rounded by itself,
// 2^-54 off with the same sign, gradients drifted by 1.25e-16 a step (5e-19 now;
// four instructions more, 64^3 168.0 -> 169.6 us a reverse step).
struct AdjRate {
    double R, Rlo, O, T, W, Wlo;
};
struct AdjP {
    double rho0, gamma, A, B, B3, kappa, kappa2;   // B3 = 3 B, kappa2 = 2 kappa
    double keep_f, keep_g;                         // 1 - w: the part of f, g that a step keeps
    AdjRate f, g;
};

// Sums of a distribution's adjoint F over the velocities, weighted in units
// of 1/36 (36 w_i = 12, 2, 1): W = sum 36 w F, O = sum 36 w c F and
// T = sum 36 w c c F.  Opposite pairs enter by their sum and difference and
// every sum names the velocities that reach it: written as loops over c_i the
// products with its zeros stay (0 * x is not 0 for every x), and they were
// most of the FP64 instructions of this kernel.
struct WeightSums {
    double W, Ox, Oy, Oz, Txx, Tyy, Tzz, Txy, Txz, Tyz;
};

__device__ __forceinline__ WeightSums weight_sums(const double (&F)[Q])
{
    WeightSums m;
    {
        const double sx = F[1] + F[2], sy = F[3] + F[4], sz = F[5] + F[6];
        const double xy = F[7] + F[8], xy_ = F[9] + F[10];   // along (1, 1, 0) and (1, -1, 0)
        const double xz = F[11] + F[12], xz_ = F[13] + F[14];
        const double yz = F[15] + F[16], yz_ = F[17] + F[18];
        const double exy = xy + xy_, exz = xz + xz_, eyz = yz + yz_;
        const double ex = exy + exz;
        m.Txx = 2.0 * sx + ex;
        m.Tyy = 2.0 * sy + (exy + eyz);
        m.Tzz = 2.0 * sz + (exz + eyz);
        m.Txy = xy - xy_;
        m.Txz = xz - xz_;
        m.Tyz = yz - yz_;
        m.W = 12.0 * F[0] + (2.0 * ((sx + sy) + sz) + (ex + eyz));
    }
    {
        const double xy = F[7] - F[8], xy_ = F[9] - F[10];
        const double xz = F[11] - F[12], xz_ = F[13] - F[14];
        const double yz = F[15] - F[16], yz_ = F[17] - F[18];
        m.Ox = 2.0 * (F[1] - F[2]) + ((xy + xy_) + (xz + xz_));
        m.Oy = 2.0 * (F[3] - F[4]) + ((xy - xy_) + (yz + yz_));
        m.Oz = 2.0 * (F[5] - F[6]) + ((xz - xz_) + (yz - yz_));
    }
    return m;
}

// Adjoint of (rho, j, phi, d, lap, kappa) -> (w feq, w geq) at one site from
// the weight sums of the adjoints of f (mf) and g (mg), w in p's factors.
// INIT: rho and j are inputs (no adjoint flows into them).
template <bool INIT>
__device__ __forceinline__ void equilibrium_vjp(const AdjP &p, double rinv, const double (&u)[3], double phi,
                                                const double (&d)[3], double lap, const WeightSums &mf,
                                                const WeightSums &mg, double &rho_b, double (&j_b)[3], double &phi_b,
                                                double (&d_b)[3], double &lap_b, double &kap_b)
{
    const double third = 1.0 / 3.0;
    // feq_i = w_i [rho + 3 c.j + 9/2 c S c - 3/2 tr S],  S = pb I + kappa d d + j j / rho
    const double fw = fma(p.f.W, mf.W, p.f.Wlo * mf.W);
    const double S[3][3] = {{p.f.T * mf.Txx - fw, p.f.T * mf.Txy, p.f.T * mf.Txz},
                            {p.f.T * mf.Txy, p.f.T * mf.Tyy - fw, p.f.T * mf.Tyz},
                            {p.f.T * mf.Txz, p.f.T * mf.Tyz, p.f.T * mf.Tzz - fw}};
    const double pb_b = S[0][0] + S[1][1] + S[2][2];
    const double kpb = p.kappa * pb_b;
    double dSd = 0.0, uSu = 0.0, Su[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const double Sd = S[a][0] * d[0] + S[a][1] * d[1] + S[a][2] * d[2];
        dSd = a ? dSd + d[a] * Sd : d[a] * Sd;
        d_b[a] = p.kappa2 * Sd - kpb * d[a];
        if (!INIT) {
            Su[a] = S[a][0] * u[0] + S[a][1] * u[1] + S[a][2] * u[2];
            uSu = a ? uSu + u[a] * Su[a] : u[a] * Su[a];
        }
    }
    // geq_i = w_i [phi + 3 phi c.u + 9/2 c G c - 3/2 tr G],  G = (Gamma mu - phi/3) I + phi u u
    const double gw = fma(p.g.W, mg.W, p.g.Wlo * mg.W);
    const double G[3][3] = {{p.g.T * mg.Txx - gw, p.g.T * mg.Txy, p.g.T * mg.Txz},
                            {p.g.T * mg.Txy, p.g.T * mg.Tyy - gw, p.g.T * mg.Tyz},
                            {p.g.T * mg.Txz, p.g.T * mg.Tyz, p.g.T * mg.Tzz - gw}};
    const double trG = G[0][0] + G[1][1] + G[2][2];
    const double mu_b = p.gamma * trG;
    const double o[3] = {p.g.O * mg.Ox, p.g.O * mg.Oy, p.g.O * mg.Oz};
    double uo = 0.0, uGu = 0.0, Gu[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        Gu[a] = G[a][0] * u[0] + G[a][1] * u[1] + G[a][2] * u[2];
        uo = a ? uo + u[a] * o[a] : u[a] * o[a];
        uGu = a ? uGu + u[a] * Gu[a] : u[a] * Gu[a];
    }
    // pb = A/2 phi^2 + 3B/4 phi^4 - kappa phi lap - kappa/2 |d|^2;  mu = A phi + B phi^3 - kappa lap
    const double dmu = p.A + p.B3 * (phi * phi);
    phi_b = fma(p.g.R, mg.W, fma(p.g.Rlo, mg.W, uo)) + (uGu - third * trG) + pb_b * (phi * dmu - p.kappa * lap) + mu_b * dmu;
    lap_b = -(kpb * phi + p.kappa * mu_b);
    const double dd = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
    kap_b = dSd - pb_b * (phi * lap + 0.5 * dd) - lap * mu_b;
    if (!INIT) {
        // u = j / rho: with v = o + 2 G u, dJ/du = phi v (of g), dJ/dj = dJ/du / rho + 2 S u + direct
        const double pr = phi * rinv;
        const double fo[3] = {p.f.O * mf.Ox, p.f.O * mf.Oy, p.f.O * mf.Oz};
#pragma unroll
        for (int a = 0; a < 3; a++) j_b[a] = (fo[a] + 2.0 * Su[a]) + pr * (o[a] + 2.0 * Gu[a]);
        rho_b = fma(p.f.R, mf.W, fma(p.f.Rlo, mf.W, -uSu)) - pr * (uo + 2.0 * uGu);
    }
}

__device__ __forceinline__ double block_sum_d(double v, double *sh)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    __syncthreads();
    if (lane == 0) sh[wid] = v;
    __syncthreads();
    double r = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) r += sh[w];
    return r;
}

// At most: k_phi_local and k_adj_collide run fp64_threads(N), like the FP64
// step.  A reverse step at 256 threads and so: 12^3 28.4 -> 16.6 us, 32^3 31.6
// -> 27.2, 48x40x44 77.3 -> 66.7, 64^3 174.4 -> 168.4, 80^3 332 -> 322.
constexpr int kAdjThreads = 256;

// phi(x) = sum_i g_i(x) of a post-streaming state
__global__ void __launch_bounds__(kAdjThreads) k_phi_local(const double *__restrict__ g, double *__restrict__ phi,
                                                           long long N)
{
    pdl_wait_then_release();
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    double v[Q];
#pragma unroll
    for (int i = 0; i < Q; i++) v[i] = g[(size_t)i * N + s];
    phi[s] = sum19(v);
}

// Collision VJP per site.  INIT: the initial state (f_bar of the equilibria
// in af_in/ag_in, no streaming, phi given by phi0, j = rho0 u0).  KEEP_F,
// KEEP_G: tau, tau_g != 1, a step keeps a part of f, g; without it the values
// of f_bar (g_bar) are not held for the output, and g_bar is phi_bar alone,
// which k_adj_stencil writes.
//
// Bound by the FP64 pipe (2 lanes a clock per SM), so written for few FP64
// instructions: weight_sums, one reciprocal of rho instead of eleven
// divisions, rates folded into the factors.  64^3, tau = tau_g = 1: a reverse
// step 0.40 -> 0.17 ms (168 us at 192 threads, 175 at 256), the gradient
// through 200 steps 138.3 -> 92.6 ms.
// Two CTAs of 256 an SM: the FP64 pipe is full with 16 warps.
template <bool INIT, bool KEEP_F, bool KEEP_G>
__global__ void __launch_bounds__(kAdjThreads, 2) k_adj_collide(const double *__restrict__ f,
                                                                const double *__restrict__ phi,
                                                                const double *__restrict__ u0,
                                                                const double *__restrict__ af_in,
                                                                const double *__restrict__ ag_in,
                                                                double *__restrict__ af_out,
                                                                double *__restrict__ ag_out, double *__restrict__ aux,
                                                                double *__restrict__ kpart, AdjP p, int nx, int ny,
                                                                int nz)
{
    pdl_wait_then_release();
    __shared__ double sh[kAdjThreads / 32];
    const long long N = (long long)nx * ny * nz;
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    double kap_b = 0.0;
    if (s < N) {
        const Nbr n((int)s, nx, ny, nz);
        const double ph = phi[s];
        double d[3], lap;
        stencil(phi, n, ph, d[0], d[1], d[2], lap);
        double rinv = 0.0, u[3];
        if (INIT) {
#pragma unroll
            for (int a = 0; a < 3; a++) u[a] = u0 ? u0[a * N + s] : 0.0;
        } else {
            double fv[Q], rho, j[3];
#pragma unroll
            for (int i = 0; i < Q; i++) fv[i] = f[(size_t)i * N + s];
            density_moments(fv, rho, j[0], j[1], j[2]);
            rinv = 1.0 / rho;
#pragma unroll
            for (int a = 0; a < 3; a++) u[a] = j[a] * rinv;
        }
        // adjoint after the streaming transpose: value of (x + c_i) at t+1
        double fsb[Q], gsb[Q];
#pragma unroll
        for (int i = 0; i < Q; i++) fsb[i] = af_in[(size_t)i * N + (INIT ? s : n.at(cx(i), cy(i), cz(i)))];
        const WeightSums mf = weight_sums(fsb);
#pragma unroll
        for (int i = 0; i < Q; i++) gsb[i] = ag_in[(size_t)i * N + (INIT ? s : n.at(cx(i), cy(i), cz(i)))];
        const WeightSums mg = weight_sums(gsb);
        if (KEEP_G) {
#pragma unroll
            for (int i = 0; i < Q; i++) ag_out[(size_t)i * N + s] = p.keep_g * gsb[i];
        }
        double rho_b, j_b[3], phi_b, d_b[3], lap_b;
        equilibrium_vjp<INIT>(p, rinv, u, ph, d, lap, mf, mg, rho_b, j_b, phi_b, d_b, lap_b, kap_b);
        if (!INIT) {
            // f_bar_i = keep f_bar_i(x + c_i) + rho_b + c_i.j_b
            auto put = [&](int i, double v) { af_out[(size_t)i * N + s] = KEEP_F ? p.keep_f * fsb[i] + v : v; };
            auto put_pair = [&](int i, double cj) {
                put(i, rho_b + cj);
                put(i + 1, rho_b - cj);
            };
            put(0, rho_b);
            put_pair(1, j_b[0]);
            put_pair(3, j_b[1]);
            put_pair(5, j_b[2]);
            put_pair(7, j_b[0] + j_b[1]);
            put_pair(9, j_b[0] - j_b[1]);
            put_pair(11, j_b[0] + j_b[2]);
            put_pair(13, j_b[0] - j_b[2]);
            put_pair(15, j_b[1] + j_b[2]);
            put_pair(17, j_b[1] - j_b[2]);
        }
        aux[s] = phi_b;
        aux[N + s] = d_b[0];
        aux[2 * N + s] = d_b[1];
        aux[3 * N + s] = d_b[2];
        aux[4 * N + s] = lap_b;
    }
    const double tot = block_sum_d(kap_b, sh);
    if (threadIdx.x == 0) kpart[blockIdx.x] = tot;
}

// phi_bar = local part + transposed stencils; g_bar_i += phi_bar (KEEP_G) or,
// where nothing of g is kept, g_bar_i = phi_bar; for the initialisation
// phi0_bar = phi_bar.  The first CTA adds the per-CTA partials of dJ/dkappa
// (fixed order) to *dkappa.
template <bool INIT, bool KEEP_G>
__global__ void __launch_bounds__(kAdjThreads) k_adj_stencil(const double *__restrict__ aux, double *__restrict__ out,
                                                             const double *__restrict__ kpart, int nparts,
                                                             double *__restrict__ dkappa, int nx, int ny, int nz)
{
    pdl_wait_then_release();
    if (blockIdx.x == 0) {
        __shared__ double sh[kAdjThreads / 32];
        double v = 0.0;
        for (int b = threadIdx.x; b < nparts; b += blockDim.x) v += kpart[b];
        const double tot = block_sum_d(v, sh);
        if (threadIdx.x == 0) *dkappa += tot;
    }
    const long long N = (long long)nx * ny * nz;
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    const Nbr n((int)s, nx, ny, nz);
    const double *db0 = aux + N, *db1 = aux + 2 * N, *db2 = aux + 3 * N, *lb = aux + 4 * N;
    const int xp = n.at(1, 0, 0), xm = n.at(-1, 0, 0), yp = n.at(0, 1, 0), ym = n.at(0, -1, 0);
    const int zp = n.at(0, 0, 1), zm = n.at(0, 0, -1);
    const double pb = aux[s] + 0.5 * ((db0[xm] - db0[xp]) + (db1[ym] - db1[yp]) + (db2[zm] - db2[zp]))
                    + ((lb[xm] + lb[xp]) + (lb[ym] + lb[yp]) + (lb[zm] + lb[zp])) - 6.0 * lb[s];
    if (INIT) {
        out[s] = pb;
    } else {
#pragma unroll
        for (int i = 0; i < Q; i++) {
            const size_t o = (size_t)i * N + s;
            out[o] = KEEP_G ? out[o] + pb : pb;
        }
    }
}

// Adjoint of the read-out phi_T = sum_i g_i(T): f_bar = 0 and every
// g_bar_i = dJ/dphi_T at the same site
__global__ void __launch_bounds__(kAdjThreads) k_adj_seed(const double *__restrict__ phi_bar,
                                                          double *__restrict__ af, double *__restrict__ ag,
                                                          long long N)
{
    const long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    const double pb = phi_bar[s];
#pragma unroll
    for (int i = 0; i < Q; i++) {
        af[(size_t)i * N + s] = 0.0;
        ag[(size_t)i * N + s] = pb;
    }
}

// the factors of a rate, R and W as what T (rounded) makes them: 2/9 T and T/3,
// the second parts from the first's exact remainders
AdjRate adj_rate(double w)
{
    AdjRate a;
    a.O = w / 12.0;
    a.T = w / 8.0;
    a.R = 2.0 * a.T / 9.0;
    a.Rlo = std::fma(-9.0, a.R, 2.0 * a.T) / 9.0;
    a.W = a.T / 3.0;
    a.Wlo = std::fma(-3.0, a.W, a.T) / 3.0;
    return a;
}

// rates w, w_g: 1 for the equilibria of the initialisation
AdjP adj_params(const lb_params &q, double w, double wg)
{
    AdjP p;
    p.rho0 = q.rho0;
    p.gamma = q.gamma;
    p.A = q.A;
    p.B = q.B;
    p.B3 = 3.0 * q.B;
    p.kappa = q.kappa;
    p.kappa2 = 2.0 * q.kappa;
    p.keep_f = 1.0 - w;
    p.keep_g = 1.0 - wg;
    p.f = adj_rate(w);
    p.g = adj_rate(wg);
    return p;
}

int full_blocks(long long N) { return (int)((N + kAdjThreads - 1) / kAdjThreads); }

// the collision's and the stencils' kernels of a reverse step
template <bool KEEP_F, bool KEEP_G>
cudaError_t reverse_step(lb_ctx *c, const double *f, const double *phi, const double *af_in, const double *ag_in,
                         double *af_out, double *ag_out, double *dkappa, double *aux, double *kpart)
{
    const int nb = adjoint_blocks(c->N);
    const int nx = c->p.nx, ny = c->p.ny, nz = c->p.nz;
    const AdjP p = adj_params(c->p, 1.0 / c->p.tau, 1.0 / c->p.tau_g);
    cudaError_t e = launch_pdl(k_adj_collide<false, KEEP_F, KEEP_G>, nb, fp64_threads(c->N), c->stream, f, phi,
                               (const double *)nullptr, af_in, ag_in, af_out, ag_out, aux, kpart, p, nx, ny, nz);
    if (e == cudaSuccess)
        e = launch_pdl(k_adj_stencil<false, KEEP_G>, full_blocks(c->N), kAdjThreads, c->stream, (const double *)aux,
                       ag_out, (const double *)kpart, nb, dkappa, nx, ny, nz);
    return e;
}

}  // namespace

// CTAs of k_adj_collide, each with a partial dJ/dkappa
int adjoint_blocks(long long N)
{
    const int tpb = fp64_threads(N);
    return (int)((N + tpb - 1) / tpb);
}

int launch_adjoint_step(lb_ctx *c, const double *f, const double *g, const double *af_in, const double *ag_in,
                        double *af_out, double *ag_out, double *dkappa, double *aux, double *kpart)
{
    double *phi = aux + 5 * c->N;
    cudaError_t e =
        launch_pdl(k_phi_local, adjoint_blocks(c->N), fp64_threads(c->N), c->stream, g, phi, (long long)c->N);
    if (e == cudaSuccess) {
        const auto step = c->p.tau == 1.0 ? (c->p.tau_g == 1.0 ? reverse_step<false, false> : reverse_step<false, true>)
                                          : (c->p.tau_g == 1.0 ? reverse_step<true, false> : reverse_step<true, true>);
        e = step(c, f, phi, af_in, ag_in, af_out, ag_out, dkappa, aux, kpart);
    }
    return e != cudaSuccess ? cuda_status(e) : check_launch();
}

int launch_adjoint_seed(lb_ctx *c, const double *phi_bar, double *af, double *ag)
{
    k_adj_seed<<<full_blocks(c->N), kAdjThreads, 0, c->stream>>>(phi_bar, af, ag, c->N);
    return check_launch();
}

int launch_adjoint_init(lb_ctx *c, const double *phi0, const double *u0, const double *af0, const double *ag0,
                        double *phi0_bar, double *dkappa, double *aux, double *kpart)
{
    const int nb = adjoint_blocks(c->N);
    const int nx = c->p.nx, ny = c->p.ny, nz = c->p.nz;
    double *none = nullptr;
    cudaError_t e = launch_pdl(k_adj_collide<true, false, false>, nb, fp64_threads(c->N), c->stream,
                               (const double *)none, phi0, u0, af0, ag0, none, none, aux, kpart,
                               adj_params(c->p, 1.0, 1.0), nx, ny, nz);
    if (e == cudaSuccess)
        e = launch_pdl(k_adj_stencil<true, false>, full_blocks(c->N), kAdjThreads, c->stream, (const double *)aux,
                       phi0_bar, (const double *)kpart, nb, dkappa, nx, ny, nz);
    return e != cudaSuccess ? cuda_status(e) : check_launch();
}

}  // namespace lbk
