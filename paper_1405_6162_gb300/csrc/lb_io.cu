// lb_io.cu -- initialisation, moments, state I/O and the FP64 conservation
// reductions of a lattice (everything but the timestep itself).
//
// The context keeps the post-collision, pre-streaming distributions A_i(x);
// the post-streaming state is the pull f_i(x, t) = A_i(x - c_i), so every
// per-site quantity here gathers A_i from x - c_i.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "d3q19.cuh"
#include "df64.cuh"
#include "lb_internal.cuh"
#include "lb_moments.cuh"
#include "lb_site.cuh"

namespace lbk {

// ------------------------------------------------------------------ init

// A_i(x - c_i) = feq_i(x), so that the first pull yields the equilibrium of
// phi0 (its stencils taken in double) and u0.  Double storage evaluates the
// equilibria in double.  Float and double-float storage evaluate them in
// double-float arithmetic on the FP32 units (df64.cuh, ~48 bits; the double
// pipe runs at 1/64 of the float rate), with the inputs split on the integer
// units: double-float storage keeps the value, by direct sums, float storage the
// float nearest to it, the same float as rounding a double result except at a
// near tie.  Without u0 float and double storage do not form half of the sums
// (opposite values are equal).
// Float, 7 points: 256^3 592 us without u0 (380 is the copy rate over its
// bytes) and 1102 with it, bound by the FP32 units.  With the inputs converted on
// the FP64 pipe and direct sums 1657 and 1959.
__device__ __forceinline__ void init_store(float *a, size_t o, df64 v) { a[o] = __fadd_rn(v.hi, v.lo); }
template <typename T>
__device__ __forceinline__ void init_store(T *a, size_t o, T v)
{
    a[o] = v;
}
// The wide stencils in double by opposite pairs (their sums and differences),
// with fewer of the FP64 instructions that bound the start of float storage than
// stencil_np: 129x97x65, 27 points, 112 us without u0 and 119 with it, by single
// values 147 and 151; 19 points 75 and 93, 96 and 105.
template <int NP>
__device__ __forceinline__ void stencil_pairs(const double *__restrict__ phi, const Nbr &n, double ph, double (&d)[3],
                                              double &lap)
{
    static_assert(NP == 19 || NP == 27, "the 7-point differences are pairs already");
    // by class (faces, edges, corners), differences by axis too; the first term
    // of each is not added to a zero (0 + x is an instruction)
    double sum[3], dif[3][3];
    int terms[4][3] = {};
    auto add = [](double &to, int &n, double x) { to = n++ ? to + x : x; };
#pragma unroll
    for (int a = 0; a <= 1; a++)
#pragma unroll
        for (int b = -1; b <= 1; b++)
#pragma unroll
            for (int c = -1; c <= 1; c++) {
                // one of each pair: the first component that is not zero is 1
                if (a == 0 && (b < 0 || (b == 0 && c <= 0))) continue;
                const int k = a * a + b * b + c * c - 1;
                if (k == 2 && NP == 19) continue;
                const double vp = phi[n.at(a, b, c)], vm = phi[n.at(-a, -b, -c)];
                const double m = vp - vm;
                add(sum[k], terms[3][k], vp + vm);
                if (a) add(dif[0][k], terms[0][k], m);
                if (b) add(dif[1][k], terms[1][k], b > 0 ? m : -m);
                if (c) add(dif[2][k], terms[2][k], c > 0 ? m : -m);
            }
    constexpr double w1 = NP == 19 ? 1.0 / 18.0 : 2.0 / 27.0, w2 = NP == 19 ? 1.0 / 36.0 : 1.0 / 54.0;
    constexpr double w3 = NP == 19 ? 0.0 : 1.0 / 216.0;
    constexpr double out = 6.0 * (6.0 * w1 + 12.0 * w2 + 8.0 * w3);   // the weights of all neighbours
#pragma unroll
    for (int x = 0; x < 3; x++) {
        d[x] = 3.0 * w1 * dif[x][0] + 3.0 * w2 * dif[x][1];
        if constexpr (NP == 27) d[x] += 3.0 * w3 * dif[x][2];
    }
    lap = 6.0 * w1 * sum[0] + 6.0 * w2 * sum[1] - out * ph;
    if constexpr (NP == 27) lap += 6.0 * w3 * sum[2];
}

template <typename E>
__device__ __forceinline__ E init_arith(double v)
{
    if constexpr (is_df64<E>::value)
        return split_double(v);
    else
        return v;
}

// p in the arithmetic type E of the equilibria; FLOW: u0 is given
template <typename T, typename E, bool SH, int NP, bool FLOW>
__global__ void __launch_bounds__(256) k_init(const double *__restrict__ phi0,
                                              const double *__restrict__ u0,
                                              T *__restrict__ fa, T *__restrict__ ga, Coll<E> p, double rho0, int nx,
                                              int ny, int nz, long long S)
{
    const long long N = (long long)nx * ny * nz;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    const Nbr n(s, nx, ny, nz);
    const double ph = phi0[s];
    double d[3], lap;
    if constexpr (std::is_same<T, float>::value && NP != 7)
        stencil_pairs<NP>(phi0, n, ph, d, lap);
    else
        stencil_np<NP, double>(phi0, n, ph, d[0], d[1], d[2], lap);
    E v[3] = {E(0), E(0), E(0)};   // u, or rho0 u
    if (FLOW)
#pragma unroll
        for (int a = 0; a < 3; a++)
            v[a] = init_arith<E>(is_df64<T>::value ? rho0 * u0[a * N + s] : u0[a * N + s]);
    const E q = init_arith<E>(ph), gx = init_arith<E>(d[0]), gy = init_arith<E>(d[1]), gz = init_arith<E>(d[2]);
    const E l = init_arith<E>(lap);
    auto sink = [&](int i, E fe, E ge) {
        const size_t o = (size_t)i * S + n.src(i);
        init_store(fa, o, fe);
        init_store(ga, o, ge);
    };
    if constexpr (is_df64<T>::value)
        equilibria_direct<E, SH>(p, p.rho0, v[0], v[1], v[2], q, gx, gy, gz, l, sink);
    else
        equilibria<E, SH, FLOW>(p, v[0], v[1], v[2], q, gx, gy, gz, l, sink);
}

// ------------------------------------------------------------------ moments / state

template <typename T, bool SH>
__global__ void __launch_bounds__(256) k_moments(const T *__restrict__ fa, const T *__restrict__ ga,
                                                 double *__restrict__ rho, double *__restrict__ u,
                                                 double *__restrict__ phi, double rho0, double hFx,
                                                 double hFy, double hFz, int nx, int ny, int nz, long long S)
{
    const long long N = (long long)nx * ny * nz;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    const Nbr n(s, nx, ny, nz);
    if (rho || u) {
        double r, v[3];
        site_rho_u<T, SH>(fa, n, S, rho0, hFx, hFy, hFz, r, v);
        if (rho) rho[s] = r;
        if (u) {
            u[s] = v[0];
            u[N + s] = v[1];
            u[2 * N + s] = v[2];
        }
    }
    if (phi) phi[s] = site_phi(ga, n, S);
}

// out[(i - i0)*N + s] = A_i(x - c_i) + shift_i, for i in [i0, i1)
template <typename T>
__global__ void __launch_bounds__(256) k_get_state(const T *__restrict__ a, double *__restrict__ out,
                                                   int i0, int i1, double shift_rho0,
                                                   int nx, int ny, int nz, long long S)
{
    const long long N = (long long)nx * ny * nz;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    const Nbr n(s, nx, ny, nz);
#pragma unroll
    for (int i = 0; i < Q; i++) {
        if (i < i0 || i >= i1) continue;
        out[(size_t)(i - i0) * N + s] = double(a[(size_t)i * S + n.src(i)]) + weight(i) * shift_rho0;
    }
}

// A_i(x - c_i) = in[(i - i0)*N + s] - shift_i, for i in [i0, i1)
template <typename T>
__global__ void __launch_bounds__(256) k_set_state(T *__restrict__ a, const double *__restrict__ in,
                                                   int i0, int i1, double shift_rho0,
                                                   int nx, int ny, int nz, long long S)
{
    const long long N = (long long)nx * ny * nz;
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= N) return;
    const Nbr n(s, nx, ny, nz);
#pragma unroll
    for (int i = 0; i < Q; i++) {
        if (i < i0 || i >= i1) continue;
        a[(size_t)i * S + n.src(i)] = T(in[(size_t)(i - i0) * N + s] - weight(i) * shift_rho0);
    }
}

// ------------------------------------------------------------------ reductions
// Totals over all sites need no pull: sum_x f_i(x, t) = sum_x A_i(x - c_i)
// = sum_x A_i(x) on the periodic lattice.

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

template <int K>
__device__ __forceinline__ void block_sum(double (&acc)[K], double *out)
{
    __shared__ double sh[kReduceThreads / 32][K];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; k++) acc[k] = warp_sum(acc[k]);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < K; k++) sh[wid][k] = acc[k];
    __syncthreads();
    if (wid == 0) {
#pragma unroll
        for (int k = 0; k < K; k++) {
            double v = lane < kReduceThreads / 32 ? sh[lane][k] : 0.0;
            v = warp_sum(v);
            if (lane == 0) out[k] = v;
        }
    }
}

// s + e = a + b exactly (Knuth), s into a; e is returned
__device__ __forceinline__ float two_sum_into(float &a, float b)
{
    float s, e;
    dfops::two_sum(a, b, s, e);
    a = s;
    return e;
}

// The sum of a thread's values of one row.  double: a double.  float and
// double-float: a float sum, the sum of its (exact) rounding errors with the
// low parts, and that sum's rounding errors -- about 70 bits in all, more than
// a double keeps.
template <typename T>
struct RowSum {
    T s;
    __device__ __forceinline__ void zero() { s = 0.0; }
    __device__ __forceinline__ void add(T v) { s += v; }
    __device__ __forceinline__ bool finite() const { return true; }   // inf and NaN are the double sum's own
    __device__ __forceinline__ double total() const { return s; }
};
struct FloatRowSum {
    float s, e, d;
    __device__ __forceinline__ void zero() { s = e = d = 0.0f; }
    __device__ __forceinline__ void add(float v) { d += two_sum_into(e, two_sum_into(s, v)); }
    __device__ __forceinline__ void add(df64 v)
    {
        const float t = two_sum_into(s, v.hi);
        const float t1 = two_sum_into(e, t), t2 = two_sum_into(e, v.lo);
        d += t1 + t2;
    }
    __device__ __forceinline__ bool finite() const { return fabsf(s) <= 3.402823466e38f; }
    __device__ __forceinline__ double total() const { return widen(s) + (widen(e) + widen(d)); }
};
template <>
struct RowSum<float> : FloatRowSum {};
template <>
struct RowSum<df64> : FloatRowSum {};

// V consecutive values of a row in one load
template <typename T, int V>
struct Packed {
    T v[V];
};
template <>
struct __align__(8) Packed<float, 2> {
    float v[2];
};

// the values of V sites from s on added to the row sums (V = 2: s even, so
// that the loads are aligned, rows starting at multiples of 64 elements)
template <typename T, int G_ROWS, int GS, int V>
__device__ __forceinline__ void add_sites(const T *__restrict__ fa, const T *__restrict__ ga, long long S, long long s,
                                          RowSum<T> (&fs)[Q], RowSum<T> (&gs)[GS])
{
    using P = Packed<T, V>;
    P f[Q], g[G_ROWS];
#pragma unroll
    for (int i = 0; i < Q; i++) f[i] = *reinterpret_cast<const P *>(fa + (size_t)i * S + s);
#pragma unroll
    for (int i = 0; i < G_ROWS; i++) g[i] = *reinterpret_cast<const P *>(ga + (size_t)i * S + s);
#pragma unroll
    for (int i = 0; i < Q; i++)
#pragma unroll
        for (int v = 0; v < V; v++) fs[i].add(f[i].v[v]);
#pragma unroll
    for (int i = 0; i < G_ROWS; i++)
#pragma unroll
        for (int v = 0; v < V; v++) gs[i % GS].add(g[i].v[v]);
}

// sites of a thread's load
template <typename T>
constexpr int kReduceSites = std::is_same<T, float>::value ? 2 : 1;

// Per-block partial totals.  A thread sums each of the 19 f rows over its
// sites (sum_x A_i(x)), and the g rows (G rows: 19, or 1 in the tau_g = 1
// reduced form, whose row 0 holds phi) into a few partial sums, as only their
// total, sum phi, is wanted; R and j = sum_i c_i F_i are formed from the 19
// row totals once per thread.  GB300 adds about 2 doubles a clock per SM, and
// one FP64 addition per value bounded this kernel (256^3: 1.26 ms in FP32, two
// additions a value and 2.47 ms in double-float), so float values are summed
// on the FP32 units (RowSum) and reach FP64 once per thread: 0.44 and 0.77 ms,
// the copy rate over the stored words being 0.38 and 0.75 ms.  FP64 storage
// keeps its 38 additions a site (1.29 ms).  A thread whose float sums leave the
// float range sums its sites again in FP64.
// The CTA that finishes last (out.ticket counts them, and is left at zero)
// adds the partials of all and puts the totals and the flag of bounded waits
// (err) side by side, so that one kernel and one copy bring both to the host
// (70x37x11, a step and its totals: about 10 us less of 80).
// The order of every addition is fixed by the launch shape, so the totals are
// bitwise reproducible.
template <typename T, int G_ROWS>
__global__ void __launch_bounds__(kReduceThreads, 2) k_reduce(const T *__restrict__ fa, const T *__restrict__ ga,
                                                              long long N, long long S, double *partial,
                                                              double offset0, const unsigned int *err, ReduceOut *out)
{
    constexpr int GS = G_ROWS < 4 ? G_ROWS : 4;   // partial sums of g
    constexpr int V = kReduceSites<T>;
    const long long stride = (long long)gridDim.x * blockDim.x, first = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    RowSum<T> fs[Q], gs[GS];
#pragma unroll
    for (int i = 0; i < Q; i++) fs[i].zero();
#pragma unroll
    for (int i = 0; i < GS; i++) gs[i].zero();
#pragma unroll 1
    for (long long s = V * first; s + V <= N; s += V * stride) add_sites<T, G_ROWS, GS, V>(fa, ga, S, s, fs, gs);
    if (V > 1 && first < N % V) add_sites<T, G_ROWS, GS, 1>(fa, ga, S, N - N % V + first, fs, gs);
    bool ok = true;
#pragma unroll
    for (int i = 0; i < Q; i++) ok = ok && fs[i].finite();
#pragma unroll
    for (int i = 0; i < GS; i++) ok = ok && gs[i].finite();
    double F[Q], G[GS];
#pragma unroll
    for (int i = 0; i < Q; i++) F[i] = fs[i].total();
#pragma unroll
    for (int i = 0; i < GS; i++) G[i] = gs[i].total();
    if (!ok) {
#pragma unroll
        for (int i = 0; i < Q; i++) F[i] = 0.0;
#pragma unroll
        for (int i = 0; i < GS; i++) G[i] = 0.0;
        auto add_double = [&](long long s) {
#pragma unroll
            for (int i = 0; i < Q; i++) F[i] += widen(fa[(size_t)i * S + s]);
#pragma unroll
            for (int i = 0; i < G_ROWS; i++) G[i % GS] += widen(ga[(size_t)i * S + s]);
        };
#pragma unroll 1
        for (long long s = V * first; s + V <= N; s += V * stride)
#pragma unroll 1
            for (int v = 0; v < V; v++) add_double(s + v);
        if (V > 1 && first < N % V) add_double(N - N % V + first);
    }
    double acc[5];
    density_moments(F, acc[0], acc[1], acc[2], acc[3]);
    acc[4] = GS == 4 ? (G[0] + G[GS > 1 ? 1 : 0]) + (G[GS > 2 ? 2 : 0] + G[GS - 1]) : G[0];
    block_sum<5>(acc, partial + 5 * blockIdx.x);
    // the CTA's partials are written by its first thread
    __shared__ bool last;
    if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(&out->ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
#pragma unroll
    for (int k = 0; k < 5; k++) acc[k] = 0.0;
    for (int b = threadIdx.x; b < (int)gridDim.x; b += blockDim.x)
#pragma unroll
        for (int k = 0; k < 5; k++) acc[k] += __ldcg(partial + 5 * b + k);
    block_sum<5>(acc, out->totals);
    if (threadIdx.x == 0) {
        out->totals[0] += offset0;
        out->wait_failed = *err;
        out->ticket = 0;
    }
}

// ------------------------------------------------------------------ launchers

static inline unsigned grid_for(long long N, int tpb) { return (unsigned)((N + tpb - 1) / tpb); }

template <typename T, bool SH, int NP>
static void init_np(lb_ctx *c, const double *phi0_d, const double *u0_d)
{
    const int cur = c->buf.cur;
    using E = typename std::conditional<std::is_same<T, double>::value, double, df64>::type;
    const auto kernel = u0_d ? k_init<T, E, SH, NP, true> : k_init<T, E, SH, NP, false>;
    kernel<<<grid_for(c->N, 256), 256, 0, c->stream>>>(phi0_d, u0_d, (T *)c->buf.f[cur], (T *)c->buf.g[cur],
                                                       make_coll<E>(c->p), c->p.rho0, c->p.nx, c->p.ny, c->p.nz, c->S);
}

template <typename T, bool SH>
static void init_t(lb_ctx *c, const double *phi0_d, const double *u0_d)
{
    if (c->npts == 19)
        init_np<T, SH, 19>(c, phi0_d, u0_d);
    else if (c->npts == 27)
        init_np<T, SH, 27>(c, phi0_d, u0_d);
    else
        init_np<T, SH, 7>(c, phi0_d, u0_d);
}

int launch_init(lb_ctx *c, const double *phi0_d, const double *u0_d)
{
    return by_precision(c, [&](auto P) {
        init_t<typename decltype(P)::T, decltype(P)::SH>(c, phi0_d, u0_d);
        const int rc = check_launch();
        return rc ? rc : state_written(c);
    });
}

int launch_moments(lb_ctx *c, double *rho, double *u, double *phi)
{
    const int cur = c->buf.cur;
    const double hF[3] = {0.5 * c->force[0], 0.5 * c->force[1], 0.5 * c->force[2]};
    const unsigned grid = grid_for(c->N, 256);
    return by_precision(c, [&](auto P) {
        using T = typename decltype(P)::T;
        k_moments<T, decltype(P)::SH><<<grid, 256, 0, c->stream>>>((const T *)c->buf.f[cur], (const T *)c->buf.g[cur],
                                                                  rho, u, phi, c->p.rho0, hF[0], hF[1], hF[2],
                                                                  c->p.nx, c->p.ny, c->p.nz, c->S);
        return check_launch();
    });
}

// f or g, components [i0, i1), to out (i1 - i0 rows of N)
static int get_rows(lb_ctx *c, int which, int i0, int i1, double *out)
{
    const int cur = c->buf.cur;
    const unsigned grid = grid_for(c->N, 256);
    const double shift = (which == 0 && c->p.precision == LB_FP32_SHIFTED) ? c->p.rho0 : 0.0;
    const void *a = which == 0 ? c->buf.f[cur] : c->buf.g[cur];
    return by_precision(c, [&](auto P) {
        using T = typename decltype(P)::T;
        k_get_state<T><<<grid, 256, 0, c->stream>>>((const T *)a, out, i0, i1, shift, c->p.nx, c->p.ny, c->p.nz,
                                                     c->S);
        return check_launch();
    });
}

static int set_rows(lb_ctx *c, int which, int i0, int i1, const double *in)
{
    const int cur = c->buf.cur;
    const unsigned grid = grid_for(c->N, 256);
    const double shift = (which == 0 && c->p.precision == LB_FP32_SHIFTED) ? c->p.rho0 : 0.0;
    void *a = which == 0 ? c->buf.f[cur] : c->buf.g[cur];
    return by_precision(c, [&](auto P) {
        using T = typename decltype(P)::T;
        k_set_state<T><<<grid, 256, 0, c->stream>>>((T *)a, in, i0, i1, shift, c->p.nx, c->p.ny, c->p.nz, c->S);
        const int rc = check_launch();
        return rc ? rc : state_written(c);
    });
}

int launch_get_state(lb_ctx *c, double *f, double *g)
{
    int rc = LB_OK;
    if (f) rc = get_rows(c, 0, 0, Q, f);
    if (!rc && g) rc = get_rows(c, 1, 0, Q, g);
    return rc;
}

int launch_set_state(lb_ctx *c, const double *f, const double *g)
{
    int rc = LB_OK;
    if (f) rc = set_rows(c, 0, 0, Q, f);
    if (!rc && g) rc = set_rows(c, 1, 0, Q, g);
    return rc;
}

int launch_rows(lb_ctx *c, int which, int i0, int i1, double *buf, int dir)
{
    return dir == 0 ? get_rows(c, which, i0, i1, buf) : set_rows(c, which, i0, i1, buf);
}

int launch_reduce(lb_ctx *c)
{
    const int cur = c->buf.cur;
    const double off = c->p.precision == LB_FP32_SHIFTED ? double(c->N) * c->p.rho0 : 0.0;
    return by_precision(c, [&](auto P) {
        using T = typename decltype(P)::T;
        const T *fa = (const T *)c->buf.f[cur], *ga = (const T *)c->buf.g[cur];
        const auto kernel = c->reduced ? k_reduce<T, 1> : k_reduce<T, Q>;
        // no CTA without a site: forming and adding a thread's totals is some
        // 70 FP64 additions, which on small lattices are most of the work
        // (70x37x11 FP64, a step and its totals: 3 us less of 60
        // with its 112 CTAs than with 304)
        const long long per = kReduceThreads * kReduceSites<T>;
        const int grid = (int)std::min<long long>(kReduceBlocks, (c->N + per - 1) / per);
        kernel<<<grid, kReduceThreads, 0, c->stream>>>(fa, ga, c->N, c->S, c->partial, off, c->err_flag,
                                                                c->dev_out);
        return check_launch();
    });
}

}  // namespace lbk
