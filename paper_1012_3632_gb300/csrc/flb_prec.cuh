// flb_prec.cuh -- kernels and launchers instantiated once per (compute type R,
// storage type S): the fused step, the density gather, initial state,
// population exchange, observables and reduction partials.  Included by
// flb_fp64.cu, flb_fp32.cu and flb_bf16.cu only.
#pragma once

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "flb_internal.h"
#include "flb_kernels.cuh"

#include "flb_force.cuh"

namespace flb {

// ---------------------------------------------------------------------------
// Host -> kernel parameters
// ---------------------------------------------------------------------------
template <class L, class R>
Coll<R> make_coll(const HostModel& m, uint64_t step)
{
    Coll<R> c{};
    c.rho0 = R(m.rho0);
    // Eq. (lbe-mom) per non-conserved mode a = D + 1 + k, divided by N_a:
    // relaxation omega_a / N_a, forcing prefactor (1 - omega_a / 2) / N_a, and
    // Eq. (noise-lbe): variance rho kT (2 - w) w N_a / cs^2 added to m_a, so
    // the kernel adds ns * sqrt(rho) * z to m_a / N_a.
    const int nstress = L::D * (L::D + 1) / 2;
    for (int k = 0; k < L::NNC; ++k) {
        const int a = L::D + 1 + k;
        const double om = (k == 0) ? m.om_b : (k < nstress) ? m.om_s : m.om_g;
        const double Na = L::N(a);
        c.rel[k] = R(-om / Na);
        if (k < nstress) c.frc[k] = R((1.0 - 0.5 * om) / Na);
        c.ns[k] = R(std::sqrt(m.kT * (2.0 - om) * om * Na * 3.0) / Na);
    }
    c.sqrt_rho0 = R(std::sqrt(m.rho0));
    c.noise = m.kT > 0.0;
    c.noise_local = m.noise_local;
    c.key = philox_keys(m.seed);
    c.step = (uint32_t)step;
    c.replica = m.replica;
    return c;
}

template <class L, class R>
StepArgs<R> make_args(const HostModel& m, uint64_t step)
{
    StepArgs<R> a{};
    a.c = make_coll<L, R>(m, step);
    a.X = m.X;
    a.Y = m.Y;
    a.Z = m.Z;
    a.V = m.V;
    a.A = R(m.A);
    a.B = R(m.B);
    a.kappa = R(m.kappa);
    a.rho0_minus_rhoc = R(m.rho0 - m.rho_c);
    a.pgrad = R(m.nonideal && m.total ? 1 : 0);
    a.inv_v = R(1.0 / (double)m.V);
    a.inv_v_lo = R(1.0 / (double)m.V - (double)a.inv_v);
    return a;
}

inline dim3 grid_for(const HostModel& m, dim3 b)
{
    return dim3((m.X + b.x - 1) / b.x, (m.Y + b.y - 1) / b.y, (m.Z + b.z - 1) / b.z);
}

template <class L>
inline dim3 site_block()
{
    return L::D == 3 ? dim3(32, 4, 2) : dim3(32, 8, 1);
}

// ---------------------------------------------------------------------------
// Auxiliary kernels
// ---------------------------------------------------------------------------

// Initial state f^eq(rho, u) (+ thermal modes), written as post-collision data
// at r - c_i so that the next pull returns it at r.
template <class R>
struct ThermalAmp {
    R tn[19];  // sqrt(kT N_a / cs^2) / N_a per mode
};

template <class L, class R, class S>
__global__ void k_init(const StepArgs<R> a, S* __restrict__ dst, const double* __restrict__ rho_in,
                       const double* __restrict__ u_in, int thermal, const ThermalAmp<R> amp)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z * blockDim.z + threadIdx.z;
    if (x >= a.X || y >= a.Y || z >= a.Z) return;
    const long V = a.V;
    const int s = x + a.X * (y + a.Y * z);
    const R rho = rho_in ? R(rho_in[s]) : a.c.rho0;
    const R drho = rho_in ? R(rho_in[s] - (double)a.c.rho0) : R(0);
    R u[3] = {R(0), R(0), R(0)};
    if (u_in)
        for (int d = 0; d < L::D; ++d) u[d] = R(u_in[d * V + s]);
    R m[L::Q], g[L::Q];
    L::eq_moments(drho, rho, u[0], u[1], u[2], m);
#pragma unroll
    for (int q = 0; q < L::Q; ++q) m[q] *= R(1.0 / L::N(q));
    if (thermal) {
        // Eqs. (G-ideal), (mu-ideal): every mode a gets variance rho kT N_a / cs^2
        const R sr = a.c.noise_local ? sqrt(rho) : a.c.sqrt_rho0;
        R zz[4 * L::NCALL_ALL];
#pragma unroll
        for (int b = 0; b < L::NCALL_ALL; ++b)
            normals4(a.c.key, (uint32_t)s, 0u, (uint32_t)b | (1u << 8), a.c.replica, zz + 4 * b);
#pragma unroll
        for (int q = 0; q < L::Q; ++q) m[q] += amp.tn[q] * sr * zz[q];
    }
    L::from_moments(m, g);
    const Nbhd nb(x, y, z, a.X, a.Y, a.Z);
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
        store_s(dst + (long)i * V + nb.src(Vel<L>::cx(i), Vel<L>::cy(i), Vel<L>::cz(i)), g[i]);
}

template <class L, class R, class S>
__global__ void k_get_pop(const S* __restrict__ src, double* __restrict__ out, double rho0, int X, int Y, int Z)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z * blockDim.z + threadIdx.z;
    if (x >= X || y >= Y || z >= Z) return;
    const long V = (long)X * Y * Z;
    const int s = x + X * (y + Y * z);
    const Nbhd nb(x, y, z, X, Y, Z);
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
        out[(long)i * V + s] = Vel<L>::w(i) * rho0 +
                               (double)load_s<R>(src + (long)i * V + nb.src(Vel<L>::cx(i), Vel<L>::cy(i), Vel<L>::cz(i)));
}

// f_i(r_k) = w_i rho0 + g_i pulled from r_k - c_i, for a list of sites r_k.
template <class L, class R, class S>
__global__ void k_get_sites(const S* __restrict__ src, const long long* __restrict__ sites, int n,
                            double* __restrict__ out, double rho0, int X, int Y, int Z)
{
    const long V = (long)X * Y * Z;
    for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n; k += gridDim.x * blockDim.x) {
        const long s = sites[k];
        const int x = (int)(s % X), y = (int)((s / X) % Y), z = (int)(s / ((long)X * Y));
        const Nbhd nb(x, y, z, X, Y, Z);
#pragma unroll
        for (int i = 0; i < L::Q; ++i)
            out[(long)i * n + k] =
                Vel<L>::w(i) * rho0 +
                (double)load_s<R>(src + (long)i * V + nb.src(Vel<L>::cx(i), Vel<L>::cy(i), Vel<L>::cz(i)));
    }
}

template <class L, class R, class S>
__global__ void k_set_pop(const double* __restrict__ in, S* __restrict__ dst, double rho0, int X, int Y, int Z)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z * blockDim.z + threadIdx.z;
    if (x >= X || y >= Y || z >= Z) return;
    const long V = (long)X * Y * Z;
    const int s = x + X * (y + Y * z);
    const Nbhd nb(x, y, z, X, Y, Z);
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
        store_s(dst + (long)i * V + nb.src(Vel<L>::cx(i), Vel<L>::cy(i), Vel<L>::cz(i)),
                R(in[(long)i * V + s] - Vel<L>::w(i) * rho0));
}

// Pre-collision deviations in the storage type, [i][s] (pull of the stored
// post-collision buffer) and the inverse scatter.  Bound by DRAM.  A store holds
// back the loads behind it, so that a site's values go in batches, all loads of one
// before its stores: 256^3 pull / push in us, one by one FP32 646 / 648, BF16 527 /
// 550; batches of 10 375 / 398 and 269 / 247, of 7 394 / 401 and 255 / 245, of all
// 375 / 410 and 265 / 253.
template <class S>
constexpr int kStateBatch = sizeof(S) == 2 ? 7 : 10;
template <class L, class S>
__global__ void k_pull_state(const S* src, S* __restrict__ out, int X, int Y, int Z)
{
    pdl_wait();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z * blockDim.z + threadIdx.z;
    if (x >= X || y >= Y || z >= Z) return;
    const long V = (long)X * Y * Z;
    const int s = x + X * (y + Y * z);
    const Nbhd nb(x, y, z, X, Y, Z);
    constexpr int K = kStateBatch<S>;
    S g[K];
#pragma unroll
    for (int b = 0; b < L::Q; b += K) {
#pragma unroll
        for (int i = b; i < L::Q && i < b + K; ++i)
            g[i - b] = src[(long)i * V + nb.src(Vel<L>::cx(i), Vel<L>::cy(i), Vel<L>::cz(i))];
#pragma unroll
        for (int i = b; i < L::Q && i < b + K; ++i) out[(long)i * V + s] = g[i - b];
    }
}
template <class L, class S>
__global__ void k_push_state(const S* in, S* __restrict__ dst, int X, int Y, int Z)
{
    pdl_wait();
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z * blockDim.z + threadIdx.z;
    if (x >= X || y >= Y || z >= Z) return;
    const long V = (long)X * Y * Z;
    const int s = x + X * (y + Y * z);
    const Nbhd nb(x, y, z, X, Y, Z);
    constexpr int K = kStateBatch<S>;
    S g[K];
#pragma unroll
    for (int b = 0; b < L::Q; b += K) {
#pragma unroll
        for (int i = b; i < L::Q && i < b + K; ++i) g[i - b] = in[(long)i * V + s];
#pragma unroll
        for (int i = b; i < L::Q && i < b + K; ++i)
            dst[(long)i * V + nb.src(Vel<L>::cx(i), Vel<L>::cy(i), Vel<L>::cz(i))] = g[i - b];
    }
}

// which: 0 rho, 1 u = (j + F/2)/rho, 2 all moments (m_0 = rho).
template <class L, class R, class S>
__global__ void k_moments(const S* __restrict__ src, double* __restrict__ out, int which,
                          const R* __restrict__ F, double rho0, int X, int Y, int Z)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z * blockDim.z + threadIdx.z;
    if (x >= X || y >= Y || z >= Z) return;
    const long V = (long)X * Y * Z;
    const int s = x + X * (y + Y * z);
    const Nbhd nb(x, y, z, X, Y, Z);
    R g[L::Q], m[L::Q];
    pull<L>(src, V, nb, g);
    L::moments(g, m);
    const double rho = rho0 + (double)m[0];
    if (which == 0) {
        out[s] = rho;
    } else if (which == 1) {
        for (int d = 0; d < L::D; ++d) {
            const double Fd = F ? (double)F[d * V + s] : 0.0;
            out[d * V + s] = ((double)m[1 + d] + 0.5 * Fd) / rho;
        }
    } else {
#pragma unroll
        for (int q = 0; q < L::Q; ++q) out[(long)q * V + s] = (q == 0) ? rho : (double)m[q];
    }
}

// mu = psi'(rho) - kappa lap rho and F = -rho grad mu on the whole lattice
// (global-memory stencils; used for observables, not in the time step).
template <class L, class R>
__global__ void k_mu(const StepArgs<R> a, const R* __restrict__ drho, R* __restrict__ mu)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z * blockDim.z + threadIdx.z;
    if (x >= a.X || y >= a.Y || z >= a.Z) return;
    const int s = x + a.X * (y + a.Y * z);
    const Nbhd nb(x, y, z, a.X, a.Y, a.Z);
    const R r0 = drho[s];
    R lap = R(0);
#pragma unroll
    for (int i = 1; i < L::Q; ++i)
        lap += R(Vel<L>::w(i)) * (drho[nb.src(-Vel<L>::cx(i), -Vel<L>::cy(i), -Vel<L>::cz(i))] - r0);
    lap *= R(6);
    const R d = r0 + a.rho0_minus_rhoc;
    mu[s] = d * (a.A + a.B * d * d) - a.kappa * lap;
}

template <class L, class R>
__global__ void k_force(const StepArgs<R> a, const R* __restrict__ drho, const R* __restrict__ mu, R* __restrict__ F)
{
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    const int y = blockIdx.y * blockDim.y + threadIdx.y;
    const int z = blockIdx.z * blockDim.z + threadIdx.z;
    if (x >= a.X || y >= a.Y || z >= a.Z) return;
    const int s = x + a.X * (y + a.Y * z);
    const Nbhd nb(x, y, z, a.X, a.Y, a.Z);
    R gr[3] = {R(0), R(0), R(0)}, pr[3] = {R(0), R(0), R(0)};
#pragma unroll
    for (int i = 1; i < L::Q; ++i) {
        const int q = nb.src(-Vel<L>::cx(i), -Vel<L>::cy(i), -Vel<L>::cz(i));  // r + c_i
        const R wm = R(Vel<L>::w(i)) * mu[q], wr = R(Vel<L>::w(i)) * drho[q];
        gr[0] += R(Vel<L>::cx(i)) * wm;
        gr[1] += R(Vel<L>::cy(i)) * wm;
        gr[2] += R(Vel<L>::cz(i)) * wm;
        pr[0] += R(Vel<L>::cx(i)) * wr;
        pr[1] += R(Vel<L>::cy(i)) * wr;
        pr[2] += R(Vel<L>::cz(i)) * wr;
    }
    const R pre = R(-3) * (a.c.rho0 + drho[s]);
    for (int d = 0; d < 3; ++d) F[d * a.V + s] = pre * gr[d] + a.pgrad * pr[d];
}

// Block sum of NV values per thread into out[0..NV) (one row per block): warp
// sums in the values' own type (32 terms; FP32 values stay off GB300's slow
// FP64 pipe), FP64 across the warps and, in k_sum_columns, across blocks.
template <int NV, class V>
__device__ __forceinline__ void block_sum_row(V v[NV], double* __restrict__ row)
{
    __shared__ double red[32][NV];
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    const int nthr = blockDim.x * blockDim.y * blockDim.z;
    const int lane = tid & 31, warp = tid >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k)
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    if (lane == 0)
        for (int k = 0; k < NV; ++k) red[warp][k] = (double)v[k];
    __syncthreads();
    const int nw = (nthr + 31) / 32;
    for (int k = tid; k < NV; k += nthr) {
        double acc = 0.0;
        for (int w = 0; w < nw; ++w) acc += red[w][k];
        row[k] = acc;
    }
}

// Sums of m_a and m_a^2 of the pre-collision moments (m_0 = drho) over one or
// many lattices.  A warp takes groups of 32 sites along x and adds the 2 Q
// values of its lanes in the compute type by exchanging halves: at distance 16,
// 8, .. 1 a lane keeps half of its columns and adds what the other lane holds
// of them (39 exchanges for 38 columns; a shuffle tree per column takes 190).
// Two columns are left per lane, and only these go to FP64, once per group.
// Bound by DRAM (76 B/site): 128^3 FP32 148 -> 28 us; the trees and a
// conversion of every column per warp and block kept the FP64 pipe busy.
template <int N, int O, class R>
__device__ __forceinline__ void halve_columns(R* v)
{
    constexpr int H = (N + 1) / 2;
    const bool up = threadIdx.x & O;
#pragma unroll
    for (int k = 0; k < H; ++k) {
        const R hi = k + H < N ? v[k + H] : R(0);
        const R keep = up ? hi : v[k], send = up ? v[k] : hi;
        v[k] = keep + __shfl_xor_sync(0xffffffffu, send, O);
    }
    if constexpr (O > 1) halve_columns<H, O / 2>(v);
}
// Column of value k after halve_columns<N, 16>, or -1 for padding.
template <int N, int O>
__device__ __forceinline__ int halved_column(int k)
{
    constexpr int H = (N + 1) / 2;
    if constexpr (O > 1) k = halved_column<H, O / 2>(k);
    if (k < 0 || k >= H) return -1;
    k += (threadIdx.x & O) ? H : 0;
    return k < N ? k : -1;
}

constexpr int kModeWarps = 8;

template <class L, class R, class S>
__global__ void __launch_bounds__(32 * kModeWarps) k_mode_sums(const __grid_constant__ ModeSums a)
{
    constexpr int NC = 2 * L::Q, NK = 2;  // columns, columns left per lane
    static_assert(NC <= 64, "two columns per lane");
    __shared__ double red[kModeWarps][NC];
    pdl_wait();
    int lo = 0, hi = a.n;  // the lattice of this block
    while (hi - lo > 1) {
        const int mid = (lo + hi) / 2;
        if ((int)blockIdx.x >= a.lat[mid].first)
            lo = mid;
        else
            hi = mid;
    }
    const ModeLattice& q = a.lat[lo];
    const int X = q.X, Y = q.Y, Z = q.Z, nx = (X + 31) / 32;
    const long V = (long)X * Y * Z;
    const S* src = (const S*)q.src;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, wpb = blockDim.x >> 5;
    const int nb = a.lat[lo + 1].first - q.first;
    const long groups = (long)nx * Y * Z, stride = (long)nb * wpb;
    double acc[NK] = {0.0, 0.0};
    for (long g = ((int)blockIdx.x - q.first) * wpb + warp; g < groups; g += stride) {
        const long row = g / nx;
        const int x = (int)(g - row * nx) * 32 + lane, y = (int)(row % Y), z = (int)(row / Y);
        R v[NC + 1];
#pragma unroll
        for (int k = 0; k < NC + 1; ++k) v[k] = R(0);
        if (x < X) {
            const Nbhd nb3(x, y, z, X, Y, Z);
            R f[L::Q], m[L::Q];
            pull<L>(src, V, nb3, f);
            L::moments(f, m);
#pragma unroll
            for (int k = 0; k < L::Q; ++k) {
                v[k] = m[k];
                v[L::Q + k] = m[k] * m[k];
            }
        }
        halve_columns<NC, 16>(v);
#pragma unroll
        for (int k = 0; k < NK; ++k) acc[k] += (double)v[k];
    }
#pragma unroll
    for (int k = 0; k < NK; ++k) {
        const int c = halved_column<NC, 16>(k);
        if (c >= 0) red[warp][c] = acc[k];
    }
    __syncthreads();
    for (int c = threadIdx.x; c < NC; c += blockDim.x) {
        double t = 0.0;
        for (int w = 0; w < wpb; ++w) t += red[w][c];
        a.rows[(long)blockIdx.x * NC + c] = t;
    }
}

// Per block: sum of g and of g c over the stored buffer (a permutation of the
// pre-collision populations, so the totals are those of the state).  The grid
// depends on V alone, so the result is deterministic.
// Every thread walks the sites with a fixed stride; per velocity pair (c, -c) it
// keeps the sum of the two populations and that of their difference (which stays
// small, so that the momentum keeps its digits) and combines the pairs at the
// end.  FP64 storage: in FP64.  Single precision: in (hi, lo) pairs by Knuth's
// TwoSum, so the rounding error of each addition is kept in lo (the FP64 rate of
// the part is a small fraction of its FP32 rate).
// A sum per component instead, 49 additions per site of D3Q19 in four dependent
// chains, took longer than the loads.  What a step with sums takes longer than one
// without: ideal 256^3 FP32 246 -> 220 us (the loads alone 188), 128^3 54 -> 38,
// 32^3 10.2 -> 5.0; FP64 96^3 170 -> 78 us.  3 blocks of 256 per SM: 6 are 11 us
// slower at 64^3 and 128^3 (the ends of more threads), 2 with 20 % more registers 23.
__device__ __forceinline__ void two_sum_add(float& hi, float& lo, float b)
{
    const float s = hi + b;
    const float bb = s - hi;
    lo += (hi - (s - bb)) + (b - bb);
    hi = s;
}

// A sum in R: a double, or two floats.
template <class R>
struct Sum {
    double v = 0.0;
    __device__ __forceinline__ void add(double b) { v += b; }
    __device__ __forceinline__ void add_difference(double a, double b) { v += a - b; }
    __device__ __forceinline__ void add(const Sum& b, int sign) { v += sign * b.v; }
    __device__ __forceinline__ double value() const { return v; }
};
template <>
struct Sum<float> {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(float b) { two_sum_add(hi, lo, b); }
    __device__ __forceinline__ void add_difference(float a, float b)
    {
        two_sum_add(a, lo, -b);
        two_sum_add(hi, lo, a);
    }
    __device__ __forceinline__ void add(const Sum& b, int sign)
    {
        two_sum_add(hi, lo, sign * b.hi);
        lo += sign * b.lo;
    }
    __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};

// First velocity of pair k, and the opposite of a velocity (D2Q9: (1,3) (2,4)
// (5,7) (6,8); D3Q19: (2k + 1, 2k + 2)).
template <class L>
__host__ __device__ constexpr int pair_of(int k)
{
    return L::Q == 19 ? 2 * k + 1 : k < 2 ? k + 1 : k + 3;
}
template <class L>
__host__ __device__ constexpr int opposite(int i)
{
    return L::Q == 19 ? i + 1 : i + 2;
}

template <class L, class R, class S>
__global__ void __launch_bounds__(kConsThreads, sizeof(R) == 8 ? 2 : 3)
    k_cons_partials(const S* src, double* __restrict__ partials, long V)
{
    pdl_wait();
    constexpr int NP = (L::Q - 1) / 2;
    Sum<R> m[NP], d[NP], t[4];
    for (long s = blockIdx.x * (long)kConsThreads + threadIdx.x; s < V; s += (long)gridDim.x * kConsThreads) {
        R g[L::Q];
#pragma unroll
        for (int i = 0; i < L::Q; ++i) g[i] = load_s<R>(src + (long)i * V + s);
        t[0].add(g[0]);
#pragma unroll
        for (int k = 0; k < NP; ++k) {
            const R a = g[pair_of<L>(k)], b = g[opposite<L>(pair_of<L>(k))];
            m[k].add(a);
            m[k].add(b);
            d[k].add_difference(a, b);
        }
    }
#pragma unroll
    for (int k = 0; k < NP; ++k) {
        const int i = pair_of<L>(k);
        t[0].add(m[k], 1);
        if (Vel<L>::cx(i) != 0) t[1].add(d[k], Vel<L>::cx(i));
        if (Vel<L>::cy(i) != 0) t[2].add(d[k], Vel<L>::cy(i));
        if (Vel<L>::cz(i) != 0) t[3].add(d[k], Vel<L>::cz(i));
    }
    double v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = t[k].value();
    block_sum_row<4>(v, partials + (long)blockIdx.x * 4);
}

template <class L, class R, class S, class T>
__global__ void __launch_bounds__(kSitesThreads)
    k_mode_field(const S* src, int mode, T* __restrict__ out, int X, int Y, int Z, const Tiling t)
{
    pdl_wait();
    const int3 r = tile_site<1, L::D == 3 ? 2 : 1, false>(t, threadIdx.x);
    if (r.x >= X || r.y >= Y || r.z >= Z) return;
    const Nbhd nb(r.x, r.y, r.z, X, Y, Z);
    R g[L::Q], m[L::Q];
    pull<L>(src, (long)X * Y * Z, nb, g);
    L::moments(g, m);
    R v = m[0];
#pragma unroll
    for (int q = 1; q < L::Q; ++q)
        if (q == mode) v = m[q];
    if constexpr (std::is_same<T, double2>::value)
        out[r.x + X * (r.y + Y * r.z)] = make_double2(v, 0.0);
    else
        out[r.x + X * (r.y + Y * r.z)] = v;
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
template <class R, class S>
struct Prec {
    // FP32 arithmetic on FP32 or BF16 storage: the two-sites-per-thread kernels
    static constexpr bool kPackedStorage =
        std::is_same<R, float>::value && (std::is_same<S, float>::value || std::is_same<S, __nv_bfloat16>::value);
    // The packed kernels take every D3Q19 lattice in FP32 storage; in BF16 storage
    // those of even X without the total free energy.  (The others keep the
    // arithmetic of one site per lane: another order of the FP32 operations moves
    // populations across BF16 rounding boundaries, and the conserved totals with
    // them by 1e-8.)
    static bool packed(const HostModel& m)
    {
        return kPackedStorage && m.Q == 19 && (std::is_same<S, float>::value || (m.X % 2 == 0 && !m.total));
    }
    static cudaError_t density(const HostModel& m, const void* pop, void* drho, cudaStream_t st)
    {
        if constexpr (kPackedStorage) {
            if (packed(m)) return density_packed(m, pop, (float*)drho, nullptr, nullptr, st);
        }
        const Tiling t = make_tiling(m.X, m.Y, m.Z, 1, kSitesThreads, m.D == 3 ? 2 : 1);
        const auto k = m.Q == 19 ? k_density<D3Q19, R, S> : k_density<D2Q9, R, S>;
        return launch_chain(k, dim3(t.blocks()), dim3(kSitesThreads), st, (const S*)pop, (R*)drho, m.X, m.Y, m.Z, t);
    }

    // Blocks up to which a step's kernel draws its noise before it waits for the
    // kernel before it (EARLY), which then lets it start as soon as it has its own
    // input: two steps share the chip.  Measured, us per step, without / with:
    // ideal FP32 32^3 2.92 / 2.3, 48^3 (432 blocks) 4.80 / 4.01, 64^3 (1024) 7.85 /
    // 7.39, 96^3 (3456) 24.7 / 26.4, BF16 48^3 4.32 / 2.97; force model FP32 32^3
    // 7.1 / 6.6, 48^3 9.9 / 9.0, 56^3 (784) 12.6 / 12.0, 64^3 (1024) 13.8 / 14.1.
    static constexpr unsigned kEarlyIdealBlocks = 8 * 152, kEarlyForceBlocks = 6 * 152;

    // The step of one site per lane (k_sites).  FP64: small lattices are stepped
    // 32 sites per block, whose other warps draw the noise meanwhile; larger ones
    // fill the FP64 pipe either way.  Measured, us per step, 128 sites / 32 per
    // block: D2Q9 32^2 7.7 / 5.2, 160 x 128 12.1 / 7.7, 224 x 200 15.7 / 12.9,
    // 256^2 equal; D3Q19 force 16^3 22.9 / 17.4, 28^3 35.7 / 33.6, 36^3 48.8 / 51.7.
    static bool split_sites(const HostModel& m) { return m.V <= (m.D == 2 ? 65536 : 24576); }
    template <class L, bool FORCE, bool TOTAL>
    static cudaError_t step_sites(const HostModel& m, uint64_t step, const void* src, void* dst, const R* drho,
                                  cudaStream_t st)
    {
        const StepArgs<R> a = make_args<L, R>(m, step);
        const Planes<S> pl = make_planes<S>(src, dst, L::Q, m.V);
        const R* mu = (const R*)m.mu;
        if constexpr (std::is_same<R, double>::value) {
            if (split_sites(m)) {
                const Tiling t = make_tiling(m.X, m.Y, m.Z, 1, 32, 1);
                return launch_chain(k_sites<L, R, S, FORCE, TOTAL, true, true>, t.grid(), dim3(kSitesThreads), st, a,
                                    pl, drho, mu, t);
            }
        }
        const Tiling t = make_tiling(m.X, m.Y, m.Z, 1, kSitesThreads, L::D == 3 ? 2 : 1);
        const auto k = t.threads ? k_sites<L, R, S, FORCE, TOTAL, false, true>
                                 : k_sites<L, R, S, FORCE, TOTAL, false, false>;
        return launch_chain(k, t.grid(), dim3(kSitesThreads), st, a, pl, drho, mu, t);
    }
    // D3Q19 force model, one site per lane: density, mu and collision passes.
    static cudaError_t step_force_sites(const HostModel& m, uint64_t step, const void* src, void* dst, R* drho,
                                        cudaStream_t st)
    {
        cudaError_t e = density(m, src, drho, st);
        if (e != cudaSuccess) return e;
        const Tiling t = make_tiling(m.X, m.Y, m.Z, 1, kSitesThreads, 2);
        const R* rho = drho;
        e = launch_chain(k_mu_field<R>, dim3(t.blocks()), dim3(kSitesThreads), st, make_args<D3Q19, R>(m, step), rho,
                         (R*)m.mu, t);
        if (e != cudaSuccess) return e;
        return m.total ? step_sites<D3Q19, true, true>(m, step, src, dst, rho, st)
                       : step_sites<D3Q19, true, false>(m, step, src, dst, rho, st);
    }
    // The D3Q19 force model steps in passes over the context's density and mu
    // fields: packed storage by flb_force.cuh, the rest by k_sites.
    static int step_in_passes(const HostModel& m) { return m.Q == 19 && m.nonideal; }
    static int gather_width(const HostModel& m) { return m.X % 4 == 0 ? 4 : m.X % 2 == 0 ? 2 : 1; }
    // density: quads of sites per thread, or pairs
    static Tiling density_tiling(const HostModel& m)
    {
        return make_tiling(m.X, m.Y, m.Z, gather_width(m) == 4 ? 4 : 2, 128, 2);
    }
    // one row per warp; X even and the excess free energy, whose deviations are
    // small: FP32 sums over a warp's sites would lose digits on a stripe's
    static int step_row_count(const HostModel& m)
    {
        return packed(m) && m.nonideal && m.X % 2 == 0 && !m.total ? 4 * (int)density_tiling(m).blocks() : 0;
    }
    // rows (or NULL): step_row_count rows of mass deviation and momentum; state
    // (or NULL, FP32 without rows, 16-byte aligned): the pulled deviations
    static cudaError_t density_packed(const HostModel& m, const void* pop, float* rho, float* rows, void* state,
                                      cudaStream_t st)
    {
        const Planes<S> pl = make_planes<S>(pop, state, 19, m.V);
        const Tiling t = density_tiling(m);
        auto go = [&](auto G) {
            constexpr int GX = decltype(G)::value;
            auto k = GX != 1 && rows ? k_force_density<S, GX, GX != 1> : k_force_density<S, GX, false>;
            if constexpr (std::is_same<S, float>::value) {
                if (state) k = k_force_density<S, GX, false, true>;
            }
            return launch_chain(k, dim3(t.blocks()), dim3(128), st, pl, rho, rows, m.X, m.Y, m.Z, t);
        };
        const int gx = gather_width(m);
        return gx == 4   ? go(std::integral_constant<int, 4>{})
               : gx == 2 ? go(std::integral_constant<int, 2>{})
                         : go(std::integral_constant<int, 1>{});
    }
    static cudaError_t step_force(const HostModel& m, uint64_t step, const void* src, void* dst, float* rho,
                                  float* rows, void* state, cudaStream_t st)
    {
        const StepArgs<R> a = make_args<D3Q19, R>(m, step);
        const Planes<S> pl = make_planes<S>(src, dst, 19, m.V);
        const float* crho = rho;
        const float* mu = (const float*)m.mu;
        const int gx = gather_width(m);
        cudaError_t e = density_packed(m, src, rho, rows, state, st);
        if (e != cudaSuccess) return e;
        const Tiling tm = make_tiling(m.X, m.Y, (m.Z + 1) / 2, gx == 4 ? 4 : 2, 128, 2);  // two planes per thread
        const auto km = gx == 4 ? k_force_mu<4> : gx == 2 ? k_force_mu<2> : k_force_mu<1>;
        const Tiling tc = make_tiling(m.X, m.Y, m.Z, 2, 128, 2);  // site pairs
        const bool early = tc.blocks() <= kEarlyForceBlocks;
        e = launch_chain(km, dim3(tm.blocks()), dim3(128), st, a, crho, (float*)m.mu, tm, early);
        if (e != cudaSuccess) return e;
        auto pick = [&](auto E) {
            constexpr bool EARLY = decltype(E)::value;
            if (gx == 1)
                return m.total ? k_force_collide<S, false, true, EARLY, true>
                               : k_force_collide<S, false, false, EARLY, true>;
            if constexpr (!EARLY)
                if (!tc.threads)
                    return m.total ? k_force_collide<S, true, true, false, false>
                                   : k_force_collide<S, true, false, false, false>;
            return m.total ? k_force_collide<S, true, true, EARLY, true> : k_force_collide<S, true, false, EARLY, true>;
        };
        const auto kc = early ? pick(std::true_type{}) : pick(std::false_type{});
        return launch_chain(kc, tc.grid(), dim3(128), st, a, pl, crho, mu, tc);
    }
    // pull_state of src, then the step: one pass over src does both where the
    // step pulls the state for its density (FP32 force model).
    static cudaError_t step_state(const HostModel& m, uint64_t t, const void* src, void* dst, const void* drho,
                                  void* state, cudaStream_t st)
    {
        if constexpr (std::is_same<S, float>::value) {
            if (packed(m) && m.nonideal && ((uintptr_t)state & 15) == 0)
                return step_force(m, t, src, dst, (float*)const_cast<void*>(drho), nullptr, state, st);
        }
        const cudaError_t e = pull_state(m, src, state, st);
        return e != cudaSuccess ? e : step(m, t, src, dst, drho, st);
    }
    // The step; with rows (non-NULL) also the mass deviation and momentum of
    // the state it steps from, as step_row_count rows of 4 partial sums, where
    // the step kernels provide them (cudaErrorNotSupported elsewhere, before any
    // launch).
    static cudaError_t step(const HostModel& m, uint64_t t, const void* src, void* dst, const void* drho,
                            cudaStream_t st)
    {
        return step_rows(m, t, src, dst, drho, nullptr, st);
    }
    static cudaError_t step_rows(const HostModel& m, uint64_t step, const void* src, void* dst, const void* drho,
                                 float4* rows, cudaStream_t st)
    {
        if (rows && !step_row_count(m)) return cudaErrorNotSupported;
        // drho: the context's density field, scratch of the steps in passes
        if constexpr (kPackedStorage) {
            if (packed(m) && m.nonideal)
                return step_force(m, step, src, dst, (float*)const_cast<void*>(drho), (float*)rows, nullptr, st);
        }
        if (step_in_passes(m)) return step_force_sites(m, step, src, dst, (R*)const_cast<void*>(drho), st);
        if (m.Q == 9 && m.nonideal && m.model == 1) {
            const StepArgs<R> a = make_args<D2Q9, R>(m, step);
            const Planes<S> pl = make_planes<S>(src, dst, 9, m.V);
            const auto* xi = (const NoiseField<R>*)m.swift_xi;
            if constexpr (kPackedStorage) {
                const Tiling t = make_tiling(m.X, m.Y, 1, 2, 128, 1);
                const auto k = m.X % 2 == 0 ? k_step_swift2<S, true> : k_step_swift2<S, false>;
                return launch_chain(k, dim3(t.blocks()), dim3(128), st, a, pl, (const R*)drho, xi, t);
            } else {
                const dim3 b(32, 8, 1);
                return launch_chain(k_step_swift<R, S, 32, 8>, grid_for(m, b), b, st, a, pl, (const R*)drho, xi);
            }
        }
        if (m.Q == 9 && m.nonideal) {
            if constexpr (kPackedStorage) {
                constexpr int TX = 32, TY = 8;
                Tiling t{};
                t.ntx = (m.X + TX - 1) / TX;
                t.nty = (m.Y + TY - 1) / TY;
                t.ntz = 1;
                fast_div((uint32_t)t.ntx, t.mx, t.sx);
                const auto k = m.X % 2 == 0 ? (m.total ? k_step_gather2<S, true, true, TX, TY>
                                                       : k_step_gather2<S, true, false, TX, TY>)
                                            : (m.total ? k_step_gather2<S, false, true, TX, TY>
                                                       : k_step_gather2<S, false, false, TX, TY>);
                return launch_chain(k, dim3(t.blocks()), dim3(TX * TY / 2), st, make_args<D2Q9, R>(m, step),
                                    make_planes<S>(src, dst, 9, m.V), t);
            } else {
                const dim3 b(32, 8, 1);
                return launch_chain(k_step_gather<R, S, 32, 8>, grid_for(m, b), b, st, make_args<D2Q9, R>(m, step),
                                    make_planes<S>(src, dst, 9, m.V));
            }
        }
        if constexpr (kPackedStorage) {
            if (packed(m)) {
                // minimum resident blocks per SM: 5 with FP32 storage (96 registers, 48
                // bytes spilled: measured faster than 4 at 126), 4 with BF16 storage
                constexpr int MINB = sizeof(S) == 4 ? 5 : 4;
                const Tiling t = make_tiling(m.X, m.Y, m.Z, 2, 128, 2);
                const bool al = m.X % 2 == 0;
                const bool early = t.blocks() <= kEarlyIdealBlocks;
                const auto k = early ? (al ? k_step2<S, true, 3, true, true> : k_step2<S, false, 3, true, true>)
                               : !al ? k_step2<S, false, MINB, false, true>
                               : t.threads ? k_step2<S, true, MINB, false, true>
                                           : k_step2<S, true, MINB, false, false>;
                return launch_chain(k, t.grid(), dim3(128), st, make_args<D3Q19, R>(m, step),
                                    make_planes<S>(src, dst, 19, m.V), t);
            }
        }
        return m.Q == 19 ? step_sites<D3Q19, false, false>(m, step, src, dst, nullptr, st)
                         : step_sites<D2Q9, false, false>(m, step, src, dst, nullptr, st);
    }

    template <class L>
    static cudaError_t init_l(const HostModel& m, void* dst, const double* rho, const double* u, int thermal,
                              cudaStream_t st)
    {
        const StepArgs<R> a = make_args<L, R>(m, 0);
        ThermalAmp<R> amp{};
        for (int q = 0; q < L::Q; ++q) amp.tn[q] = R(std::sqrt(3.0 * m.kT / L::N(q)));
        const dim3 b = site_block<L>();
        k_init<L, R, S><<<grid_for(m, b), b, 0, st>>>(a, (S*)dst, rho, u, thermal, amp);
        return cudaGetLastError();
    }
    static cudaError_t init(const HostModel& m, void* dst, const double* rho, const double* u, int thermal,
                            cudaStream_t st)
    {
        return m.Q == 19 ? init_l<D3Q19>(m, dst, rho, u, thermal, st) : init_l<D2Q9>(m, dst, rho, u, thermal, st);
    }

    static cudaError_t get_pop(const HostModel& m, const void* src, double* out, cudaStream_t st)
    {
        if (m.Q == 19) {
            const dim3 b = site_block<D3Q19>();
            k_get_pop<D3Q19, R, S><<<grid_for(m, b), b, 0, st>>>((const S*)src, out, m.rho0, m.X, m.Y, m.Z);
        } else {
            const dim3 b = site_block<D2Q9>();
            k_get_pop<D2Q9, R, S><<<grid_for(m, b), b, 0, st>>>((const S*)src, out, m.rho0, m.X, m.Y, m.Z);
        }
        return cudaGetLastError();
    }
    static cudaError_t set_pop(const HostModel& m, const double* in, void* dst, cudaStream_t st)
    {
        if (m.Q == 19) {
            const dim3 b = site_block<D3Q19>();
            k_set_pop<D3Q19, R, S><<<grid_for(m, b), b, 0, st>>>(in, (S*)dst, m.rho0, m.X, m.Y, m.Z);
        } else {
            const dim3 b = site_block<D2Q9>();
            k_set_pop<D2Q9, R, S><<<grid_for(m, b), b, 0, st>>>(in, (S*)dst, m.rho0, m.X, m.Y, m.Z);
        }
        return cudaGetLastError();
    }
    static cudaError_t moments(const HostModel& m, const void* src, double* out, int which, const void* F,
                               cudaStream_t st)
    {
        if (m.Q == 19) {
            const dim3 b = site_block<D3Q19>();
            k_moments<D3Q19, R, S><<<grid_for(m, b), b, 0, st>>>((const S*)src, out, which, (const R*)F, m.rho0,
                                                                  m.X, m.Y, m.Z);
        } else {
            const dim3 b = site_block<D2Q9>();
            k_moments<D2Q9, R, S><<<grid_for(m, b), b, 0, st>>>((const S*)src, out, which, (const R*)F, m.rho0,
                                                                 m.X, m.Y, m.Z);
        }
        return cudaGetLastError();
    }
    template <class L>
    static cudaError_t mu_force_l(const HostModel& m, const void* drho, void* mu, void* F, cudaStream_t st)
    {
        const StepArgs<R> a = make_args<L, R>(m, 0);
        const dim3 b = site_block<L>();
        k_mu<L, R><<<grid_for(m, b), b, 0, st>>>(a, (const R*)drho, (R*)mu);
        k_force<L, R><<<grid_for(m, b), b, 0, st>>>(a, (const R*)drho, (const R*)mu, (R*)F);
        return cudaGetLastError();
    }
    static cudaError_t mu_force(const HostModel& m, const void* drho, void* mu, void* F, cudaStream_t st)
    {
        return m.Q == 19 ? mu_force_l<D3Q19>(m, drho, mu, F, st) : mu_force_l<D2Q9>(m, drho, mu, F, st);
    }
    // a density field written before the step: only the modified-equilibrium step
    // reads one (the force-model steps form their density themselves)
    static int needs_density(const HostModel& m) { return m.nonideal && m.Q == 9 && m.model == 1 ? 1 : 0; }
    static int site_blocks(const HostModel& m)
    {
        const dim3 b = m.Q == 19 ? site_block<D3Q19>() : site_block<D2Q9>();
        const dim3 g = grid_for(m, b);
        return (int)(g.x * g.y * g.z);
    }
    static int rows(const HostModel& m) { return std::max(site_blocks(m), kModeRowsMin); }
    // one launch over a.n lattices whose `first` and `rows` are set (mode_blocks)
    static cudaError_t mode_sums(const ModeSums& a, int Q, int warps, cudaStream_t st)
    {
        const dim3 g(a.lat[a.n].first), b(32 * warps);
        return Q == 19 ? launch_chain(k_mode_sums<D3Q19, R, S>, g, b, st, a)
                       : launch_chain(k_mode_sums<D2Q9, R, S>, g, b, st, a);
    }
    static cudaError_t cons_partials(const HostModel& m, const void* src, double* partials, cudaStream_t st)
    {
        const auto k = m.Q == 19 ? k_cons_partials<D3Q19, R, S> : k_cons_partials<D2Q9, R, S>;
        return launch_chain(k, dim3(cons_rows(m.V)), dim3(kConsThreads), st, (const S*)src, partials, m.V);
    }
    static cudaError_t mode_field(const HostModel& m, const void* src, int mode, void* out, cudaStream_t st)
    {
        if constexpr (kPackedStorage) {
            if (mode == 0 && packed(m) && ((uintptr_t)out & 15) == 0)
                return density_packed(m, src, (float*)out, nullptr, nullptr, st);  // the same sums, a quad per thread
        }
        using T = typename std::conditional<std::is_same<R, double>::value, double2, float>::type;
        const Tiling t = make_tiling(m.X, m.Y, m.Z, 1, kSitesThreads, m.D == 3 ? 2 : 1);
        const auto k = m.Q == 19 ? k_mode_field<D3Q19, R, S, T> : k_mode_field<D2Q9, R, S, T>;
        return launch_chain(k, dim3(t.blocks()), dim3(kSitesThreads), st, (const S*)src, mode, (T*)out, m.X, m.Y, m.Z,
                            t);
    }

    static cudaError_t pull_state(const HostModel& m, const void* src, void* out, cudaStream_t st)
    {
        const dim3 b = m.Q == 19 ? site_block<D3Q19>() : site_block<D2Q9>();
        if (m.Q == 19)
            return launch_chain(k_pull_state<D3Q19, S>, grid_for(m, b), b, st, (const S*)src, (S*)out, m.X, m.Y, m.Z);
        return launch_chain(k_pull_state<D2Q9, S>, grid_for(m, b), b, st, (const S*)src, (S*)out, m.X, m.Y, m.Z);
    }
    static cudaError_t push_state(const HostModel& m, const void* in, void* dst, cudaStream_t st)
    {
        const dim3 b = m.Q == 19 ? site_block<D3Q19>() : site_block<D2Q9>();
        if (m.Q == 19)
            return launch_chain(k_push_state<D3Q19, S>, grid_for(m, b), b, st, (const S*)in, (S*)dst, m.X, m.Y, m.Z);
        return launch_chain(k_push_state<D2Q9, S>, grid_for(m, b), b, st, (const S*)in, (S*)dst, m.X, m.Y, m.Z);
    }

    static cudaError_t get_sites(const HostModel& m, const void* src, const long long* sites, int n, double* out,
                                 cudaStream_t st)
    {
        if (n <= 0) return cudaSuccess;
        const int nb = std::min((n + 127) / 128, 152 * 4);
        if (m.Q == 19)
            k_get_sites<D3Q19, R, S><<<nb, 128, 0, st>>>((const S*)src, sites, n, out, m.rho0, m.X, m.Y, m.Z);
        else
            k_get_sites<D2Q9, R, S><<<nb, 128, 0, st>>>((const S*)src, sites, n, out, m.rho0, m.X, m.Y, m.Z);
        return cudaGetLastError();
    }

    static const PrecOps& ops()
    {
        static const PrecOps o = {(int)sizeof(S), (int)sizeof(R), density, step, init, get_pop, set_pop, moments,
                                  mu_force, mode_sums, cons_partials, mode_field, rows, needs_density, step_in_passes,
                                  pull_state, push_state, get_sites, step_row_count, step_rows, step_state};
        return o;
    }
};

}  // namespace flb
