// flb_adjoint.cu -- adjoint (reverse-mode derivative) of one fluctuating LB
// time step of D3Q19, ideal gas or force-based non-ideal fluid, with the
// identical Philox noise replayed.
//
// Forward map of one step, on pre-collision deviations g^n (layout [i][s]):
//   g^{n+1}_i(r + c_i) = C_i(g^n(r), F(r); theta),  F = -rho grad mu,
//   mu = psi'(rho) - kappa lap rho,  rho = rho0 + sum_i g^n_i,
// with C the moment-space collision of Eq. (lbe-mom) (noise included, its
// amplitude depending on the local density).  Given lam^{n+1} = dJ/dg^{n+1}
// the step computes lam^n = dJ/dg^n and adds dJ/dtheta for
// theta = (omega_shear, omega_bulk, omega_ghost, kappa, A, B).
//
// Kernels (all hand-written VJPs):
//   k_adj_density, k_force_mu / k_mu_field
//                  rho and mu of the states of up to kAdjBatch steps, a launch each;
//   k_adj_collide  per step: pull lam^{n+1}(r + c_i) (adjoint of streaming), replay
//                  the forward collision at r and propagate through it: the local
//                  part of lam^n, the force adjoint Fbar(r), the direct term
//                  -Fbar . grad mu of rho and the relaxation parameter gradients;
//   k_adj_mu       mubar(y) = -3 sum_i w_i c_i . rho(y - c_i) Fbar(y - c_i)
//                  (adjoint of F = -rho grad mu);
//   k_adj_rho      rhobar = psi''(rho) mubar - kappa lap(mubar) + direct term,
//                  added to every population (rho = sum_i g_i), and the
//                  kappa, A, B gradients;
//   k_sum_grads, k_add_grads
//                  the gradients' block sums of those steps into grad.
// At 64^3 a launch takes little more than its latency, so that fields which the
// states of several steps give at once are not a launch per step, neighbours are
// read once (30 values for mubar, not 90) and the launches are chained: a segment
// of 20 steps, recomputed and swept back, takes 0.94 ms; with density, mu, force
// and gradient launches per step and its states pulled apart it took 1.8 ms.
#include <cuda_runtime.h>

#include <cmath>
#include <string>

#include "../../include/flb.h"
#include "flb_internal.h"
#include "flb_prec.cuh"

namespace flb {

Coll<float> coll_fp32(const HostModel& m, uint64_t step);
Coll<double> coll_fp64(const HostModel& m, uint64_t step);

namespace {

using L = D3Q19;

// Adjoint parameters per launch.
template <class R>
struct AdjArgs {
    Coll<R> c;
    int X, Y, Z;
    long V;
    R A, B, kappa, rho0_minus_rhoc;
    // per class of modes (0 bulk: mode 0 of the non-conserved ones, 1 shear: 1-5,
    // 2 ghost: 6-14): 1 / omega, d ln(ns) / d omega
    R inv_om[3], dln_ns[3];
};

__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }

// sites per thread
template <class T>
constexpr int kSites = std::is_same<T, F2>::value ? 2 : 1;
__device__ __forceinline__ double value_sum(double v, bool) { return v; }
__device__ __forceinline__ float value_sum(F2 v, bool two) { return two ? v.v.x + v.v.y : v.v.x; }

// d_a = sum_i T_ai w_i l_i: L::moments of w l, the weights (axis pairs 1/18, edge
// pairs 1/36) taken out of the sums.  (w l first rounds every value once more, for a
// sum and a difference: error of a step back 7.3e-8, one site per thread 7.0e-8, so
// 6.4e-8.)
template <class T>
__device__ __forceinline__ void weighted_moments(const T l[19], T d[19])
{
    T s[10], e[10];
#pragma unroll
    for (int k = 1; k < 10; ++k) {
        s[k] = l[2 * k - 1] + l[2 * k];
        e[k] = l[2 * k - 1] - l[2 * k];
    }
    const T wa(1.0 / 18), we(1.0 / 36);
    const T sa = s[1] + s[2] + s[3], sxy = s[4] + s[5], sxz = s[6] + s[7], syz = s[8] + s[9], se = sxy + sxz + syz;
    const T jx = (e[4] + e[5]) + (e[6] + e[7]), jy = (e[4] - e[5]) + (e[8] + e[9]), jz = (e[6] - e[7]) + (e[8] - e[9]);
    d[0] = mad(T(1.0 / 3), l[0], mad(wa, sa, we * se));
    d[1] = mad(wa, e[1], we * jx);
    d[2] = mad(wa, e[2], we * jy);
    d[3] = mad(wa, e[3], we * jz);
    d[4] = mad(T(-1.0 / 3), l[0], we * se);
    d[5] = mad(wa, mad(T(2), s[1], T(-1) * (s[2] + s[3])), we * mad(T(-2), syz, sxy + sxz));
    d[6] = mad(wa, s[2] - s[3], we * (sxy - sxz));
    d[7] = we * (s[4] - s[5]);
    d[8] = we * (s[8] - s[9]);
    d[9] = we * (s[6] - s[7]);
    d[10] = mad(T(-1.0 / 27), e[1], T(1.0 / 108) * jx);
    d[11] = mad(T(-1.0 / 27), e[2], T(1.0 / 108) * jy);
    d[12] = mad(T(-1.0 / 27), e[3], T(1.0 / 108) * jz);
    d[13] = we * ((e[4] + e[5]) - (e[6] + e[7]));
    d[14] = we * ((e[5] - e[4]) + (e[8] + e[9]));
    d[15] = we * ((e[6] - e[7]) - (e[8] - e[9]));
    d[16] = mad(T(1.0 / 9), l[0], mad(T(-1.0 / 27), sa, T(1.0 / 108) * se));
    d[17] = mad(wa, mad(T(0.5), s[2] + s[3], T(-1) * s[1]), we * mad(T(0.5), sxy + sxz, T(-1) * syz));
    d[18] = mad(we, s[3] - s[2], T(1.0 / 72) * (sxy - sxz));
}

// lb_i += sum_a T_ai b_a, the transpose of L::moments
template <class T>
__device__ __forceinline__ void add_transposed(const T b[19], T lb[19])
{
    const T h17 = T(0.5) * b[17], h18 = T(0.5) * b[18];
    lb[0] += mad(T(1.0 / 3), b[16], b[0] - b[4]);
    const T Ea = mad(T(-2.0 / 3), b[16], b[0]), Ee = mad(T(1.0 / 3), b[16], b[0] + b[4]);
    const T s56 = b[5] + b[6], d56 = b[6] - b[5];
    const T E1 = Ea + mad(T(2), b[5], T(-1) * b[17]), O1 = mad(T(-2.0 / 3), b[10], b[1]);
    const T E2 = Ea + d56 + (h17 - h18), O2 = mad(T(-2.0 / 3), b[11], b[2]);
    const T E3 = Ea - s56 + (h17 + h18), O3 = mad(T(-2.0 / 3), b[12], b[3]);
    const T Exy = Ee + s56 + (h17 + h18), Exz = Ee - d56 + (h17 - h18), Eyz = Ee - mad(T(2), b[5], b[17]);
    const T jx = mad(T(1.0 / 3), b[10], b[1]), jy = mad(T(1.0 / 3), b[11], b[2]), jz = mad(T(1.0 / 3), b[12], b[3]);
    const T E[10] = {Ea, E1, E2, E3, Exy + b[7], Exy - b[7], Exz + b[9], Exz - b[9], Eyz + b[8], Eyz - b[8]};
    const T O[10] = {Ea, O1, O2, O3, jx + jy + (b[13] - b[14]), jx - jy + (b[13] + b[14]), jx + jz - (b[13] - b[15]),
                     jx - jz - (b[13] + b[15]), jy + jz + (b[14] - b[15]), jy - jz + (b[14] + b[15])};
#pragma unroll
    for (int k = 1; k < 10; ++k) {
        lb[2 * k - 1] += E[k] + O[k];
        lb[2 * k] += E[k] - O[k];
    }
}

// VJP of the collision of one site (two with T = F2).  m: moments of the
// pre-collision deviations; F: force; l: adjoint of the post-collision
// populations (pulled from step n+1), turned into the local part of the adjoint
// of the deviations.  Out: fb (force adjoint), gp[3] (gradients of omega_bulk,
// omega_shear, omega_ghost).
// The collision is D_k = rel_k (m_k - rho u.Q_k u) + frc_k 2 u.Q_k F + ns_k s z_k
// with 15 modes k, of which 0-5 have a quadratic form Q_k: all derivatives of
// those six in u, F and rho go through the two symmetric matrices
//   E = 2 sum_k e_k Q_k,  M = 2 sum_k f_k Q_k,  e_k = rel_k d_k, f_k = frc_k d_k,
// d = moments of w lb.
template <bool FORCE, class T, class R>
__device__ __forceinline__ void collide_vjp(const T m[19], const T F[3], T l[19], const AdjArgs<R>& a, uint32_t site,
                                            T fb[3], T gp[3])
{
    const Coll<R>& P = a.c;
    const T rho = P.rho0 + m[0];
    T ir;
    if constexpr (std::is_same<T, F2>::value)
        ir = F2(1.0f / rho.v.x, 1.0f / rho.v.y);
    else
        ir = T(1) / rho;
    T u[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) u[k] = (FORCE ? mad(T(0.5), F[k], m[1 + k]) : m[1 + k]) * ir;
    T d[19], b[19];
    weighted_moments(l, d);
    // noise: A_c = sum_k ns_k z_k d_k over the modes of class c
    T rb(0);
#pragma unroll
    for (int c = 0; c < 3; ++c) gp[c] = T(0);
    if (P.noise) {
        T z[16], A[3] = {T(0), T(0), T(0)};
        noise_normals<4>(P.key, site, P.step, P.replica, z);
#pragma unroll
        for (int k = 0; k < 15; ++k) {
            const int c = k == 0 ? 0 : k < 6 ? 1 : 2;
            A[c] = mad(P.ns[k] * d[4 + k], z[k], A[c]);
        }
        T sr;
        if constexpr (std::is_same<T, F2>::value)
            sr = P.noise_local ? F2(sqrtf(rho.v.x), sqrtf(rho.v.y)) : F2(P.sqrt_rho0);
        else
            sr = P.noise_local ? T(sqrt(rho)) : T(P.sqrt_rho0);
#pragma unroll
        for (int c = 0; c < 3; ++c) gp[c] = sr * (a.dln_ns[c] * A[c]);
        if (P.noise_local) rb = T(0.5) * (A[0] + A[1] + A[2]) * (sr * ir);  // d sqrt(rho) = sqrt(rho) / (2 rho)
    }
#pragma unroll
    for (int k = 0; k < 15; ++k) b[4 + k] = P.rel[k] * d[4 + k];
    auto symmetric = [](const T* e, const T v[3], T out[3]) {  // 2 sum_k e_k Q_k v
        const T e0 = T(2) * e[0], e1 = T(2) * e[1], e2 = T(2) * e[2];
        const T xx = mad(T(2), e1, e0), yy = e0 - e1 + e2, zz = e0 - e1 - e2;
        out[0] = mad(xx, v[0], mad(e[3], v[1], e[5] * v[2]));
        out[1] = mad(e[3], v[0], mad(yy, v[1], e[4] * v[2]));
        out[2] = mad(e[5], v[0], mad(e[4], v[1], zz * v[2]));
    };
    T Eu[3];
    symmetric(b + 4, u, Eu);
    const T uu = mad(u[0], u[0], mad(u[1], u[1], u[2] * u[2]));
    const T huEu = T(0.5) * mad(u[0], Eu[0], mad(u[1], Eu[1], u[2] * Eu[2]));  // sum_k e_k u.Q_k u
    // omega gradients: d rel = rel / omega, d frc = rel / (2 omega)
    T g0 = mad(T(-1) * rho, uu, m[4]), g1 = mad(b[4], uu, T(-1) * huEu), gm(0), g2(0);
#pragma unroll
    for (int k = 1; k < 6; ++k) gm = mad(b[4 + k], m[4 + k], gm);
    g1 = mad(rho, g1, gm);
#pragma unroll
    for (int k = 6; k < 15; ++k) g2 = mad(b[4 + k], m[4 + k], g2);
    rb = rb - huEu;
    T ub[3];
    if constexpr (FORCE) {
        const T uF = mad(u[0], F[0], mad(u[1], F[1], u[2] * F[2]));
        const T uEF = mad(F[0], Eu[0], mad(F[1], Eu[1], F[2] * Eu[2]));  // 2 sum_k e_k u.Q_k F
        g0 += uF;
        g1 += mad(T(0.5), uEF, T(-1) * (b[4] * uF));
        T f[6], Mu[3], MF[3];
#pragma unroll
        for (int k = 0; k < 6; ++k) f[k] = P.frc[k] * d[4 + k];
        symmetric(f, u, Mu);
        symmetric(f, F, MF);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            ub[k] = mad(T(-1) * rho, Eu[k], MF[k]) * ir;
            fb[k] = mad(T(0.5), ub[k], mad(T(3), d[1 + k], Mu[k]));
        }
    } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) ub[k] = T(-1) * Eu[k];
    }
    gp[0] = mad(a.inv_om[0], b[4] * g0, gp[0]);
    gp[1] = mad(a.inv_om[1], g1, gp[1]);
    gp[2] = mad(a.inv_om[2], g2, gp[2]);
    // u = (j + F/2) / rho
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        b[1 + k] = ub[k];
        rb = mad(T(-1) * ub[k], u[k], rb);
    }
    b[0] = rb;
    add_transposed(b, l);
}

// Block sums of NV per-thread values: warp sums in the compute type (32
// terms; FP64 arithmetic per thread would run on GB300's slow FP64 pipe),
// then FP64 across the warps of the block and, in sum_columns, across blocks.
template <int NV, class R>
__device__ __forceinline__ void block_rows(R v[NV], double* __restrict__ row)
{
    __shared__ double red[32][NV];
    const int tid = threadIdx.x + blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z);
    const int nthr = blockDim.x * blockDim.y * blockDim.z;
#pragma unroll
    for (int k = 0; k < NV; ++k)
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
    if ((tid & 31) == 0)
        for (int k = 0; k < NV; ++k) red[tid >> 5][k] = (double)v[k];
    __syncthreads();
    for (int k = tid; k < NV; k += nthr) {
        double acc = 0.0;
        for (int w = 0; w < (nthr + 31) / 32; ++w) acc += red[w][k];
        row[k] = acc;
    }
}

// densities of the states g^n (pre-collision deviations) blockIdx.y = 0, 1, ..
template <class R>
__global__ void __launch_bounds__(128) k_adj_density(const R* gn, R* __restrict__ drho, long V)
{
    pdl_wait();
    gn += (long)blockIdx.y * 19 * V;
    drho += (long)blockIdx.y * V;
    for (long s = blockIdx.x * (long)blockDim.x + threadIdx.x; s < V; s += (long)gridDim.x * blockDim.x) {
        R g[19], m[19];
#pragma unroll
        for (int i = 0; i < 19; ++i) g[i] = gn[(long)i * V + s];
        L::moments(g, m);
        drho[s] = m[0];
    }
}

// Loads of the kSites<T> values of a row from x on, one site or two: two at x
// by one load with AL (X even, rows aligned), single ones elsewhere.
template <class T, class R>
struct Row {
    int x, x1, xm, xe;  // the sites, their neighbours -1 and +1
    template <bool AL>
    __device__ __forceinline__ T at(const R* p, int c) const
    {
        if constexpr (kSites<T> == 1)
            return p[c == 0 ? x : c < 0 ? xm : xe];
        else if (c == 0)
            return AL ? mk2(*reinterpret_cast<const float2*>(p + x)) : F2(p[x], p[x1]);
        else
            return c < 0 ? F2(p[xm], p[x]) : F2(p[x1], p[xe]);
    }
};
template <class T, bool AL, class R>
__device__ __forceinline__ void put(R* p, T v, bool two)
{
    if constexpr (kSites<T> == 1) {
        *p = v;
    } else if constexpr (AL) {
        *reinterpret_cast<float2*>(p) = v.v;
    } else {
        p[0] = v.v.x;
        if (two) p[1] = v.v.y;
    }
}

// The VJP of the collision.  T = F2: two sites per thread (FP32), which halves
// the instructions: 64^3 23.0 -> 18.9 us, the 60 MB of states and adjoints in
// L2 and DRAM take 9.  3 blocks per SM: 168 registers; 4 (spilled) and 2 make a
// step back 1.5 and 2.7 us longer.  AL: X even and every pointer aligned to two values.
// rb_next (or NULL): the density part of lam_next kept apart by the previous
// adjoint step of a segment; lam_next + rb_next is the full adjoint state.
// W: rho Fbar (TOTAL: Fbar), three fields; rb1: -Fbar . grad mu.
template <class T, class R, bool AL, bool FORCE, bool TOTAL>
__global__ void __launch_bounds__(128, kSites<T> == 2 ? 3 : 2)
    k_adj_collide(const AdjArgs<R> a, const R* gn, const R* drho, const R* mu,
                  const R* lam_next, const R* rb_next, R* __restrict__ lam,
                  R* __restrict__ W, R* __restrict__ rb1, double* __restrict__ rows, const Tiling t)
{
    pdl_wait();
    const int3 r = tile_site<kSites<T>, 2, false>(t, threadIdx.x);
    const int x = r.x, y = r.y, z = r.z, X = a.X, Y = a.Y, Z = a.Z, XY = X * Y;
    R gs[3] = {R(0), R(0), R(0)};
    if (x < X && y < Y && z < Z) {
        const long V = a.V;
        const int x1 = x + 1 == X ? 0 : x + 1;
        const Row<T, R> row{x, x1, x == 0 ? X - 1 : x - 1, kSites<T> == 1 ? x1 : x1 + 1 == X ? 0 : x1 + 1};
        const int yo[3] = {X * wrap_once(y - 1, Y), X * y, X * wrap_once(y + 1, Y)};
        const int zo[3] = {XY * (z == 0 ? Z - 1 : z - 1), XY * z, XY * (z == Z - 1 ? 0 : z + 1)};
        const bool two = AL || x + 1 < X;
        T l[19], m[19], F[3], fb[3], gp[3], d[3];
        {
            T g[19];
#pragma unroll
            for (int i = 0; i < 19; ++i) g[i] = row.template at<AL>(gn + (i * V + yo[1] + zo[1]), 0);
            L::moments(g, m);
        }
#pragma unroll
        for (int i = 0; i < 19; ++i) {
            // streaming moved the post-collision population i from r to r + c_i
            const int o = yo[1 + Vel<L>::cy(i)] + zo[1 + Vel<L>::cz(i)];
            l[i] = row.template at<AL>(lam_next + (i * V + o), Vel<L>::cx(i));
            if (rb_next) l[i] += row.template at<AL>(rb_next + o, Vel<L>::cx(i));
        }
        // sum_i w_i c_i f(r + c_i) (a gradient / 3) from the differences f(c) - f(-c)
        // of the velocity pairs (2k-1, 2k): axis pairs weigh 1/18, edge pairs 1/36
        auto gradient = [&](const R* f, T out[3]) {
            T e[10];
#pragma unroll
            for (int k = 1; k <= 9; ++k) {
                const int cx = Vel<L>::cx(2 * k - 1), cy = Vel<L>::cy(2 * k - 1), cz = Vel<L>::cz(2 * k - 1);
                e[k] = row.template at<AL>(f + (yo[1 + cy] + zo[1 + cz]), cx) -
                       row.template at<AL>(f + (yo[1 - cy] + zo[1 - cz]), -cx);
            }
            out[0] = T(1.0 / 18) * e[1] + T(1.0 / 36) * ((e[4] + e[5]) + (e[6] + e[7]));
            out[1] = T(1.0 / 18) * e[2] + T(1.0 / 36) * ((e[4] - e[5]) + (e[8] + e[9]));
            out[2] = T(1.0 / 18) * e[3] + T(1.0 / 36) * ((e[6] - e[7]) + (e[8] - e[9]));
        };
        const T rho = a.c.rho0 + m[0];
        if constexpr (FORCE) {
            gradient(mu, d);
#pragma unroll
            for (int k = 0; k < 3; ++k) F[k] = T(-3) * rho * d[k];
            if constexpr (TOTAL) {
                T p[3];
                gradient(drho, p);
#pragma unroll
                for (int k = 0; k < 3; ++k) F[k] += p[k];
            }
        }
        const int s = x + yo[1] + zo[1];
        collide_vjp<FORCE>(m, F, l, a, (uint32_t)s, fb, gp);
#pragma unroll
        for (int i = 0; i < 19; ++i) put<T, AL>(lam + (i * V + s), l[i], two);
        if constexpr (FORCE) {
#pragma unroll
            for (int k = 0; k < 3; ++k) put<T, AL>(W + (k * V + s), TOTAL ? fb[k] : rho * fb[k], two);
            put<T, AL>(rb1 + s, T(-3) * (d[0] * fb[0] + d[1] * fb[1] + d[2] * fb[2]), two);
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) gs[c] = value_sum(gp[c], two);
    }
    block_rows<3>(gs, rows + 3 * (long)blockIdx.x);
}

// mubar(y) = -3 sum_i w_i c_i . rho(y - c_i) Fbar(y - c_i); TOTAL (F gains
// cs^2 grad rho): rb1 += sum_i w_i c_i . Fbar(y - c_i) as well.
template <class R, bool TOTAL>
__global__ void __launch_bounds__(128)
    k_adj_mu(const AdjArgs<R> a, const R* drho, const R* W, R* __restrict__ mubar,
             R* __restrict__ rb1, const Tiling t)
{
    pdl_wait();
    const int3 r = tile_site<1, 2, false>(t, threadIdx.x);
    if (r.x >= a.X || r.y >= a.Y || r.z >= a.Z) return;
    const long V = a.V;
    const int s = r.x + a.X * (r.y + a.Y * r.z);
    const Nbhd nb(r.x, r.y, r.z, a.X, a.Y, a.Z);
    R ax = R(0), ed = R(0), axp = R(0), edp = R(0);  // axis and edge velocities, weights 1/18 and 1/36
#pragma unroll
    for (int i = 1; i < 19; ++i) {
        const int cx = Vel<L>::cx(i), cy = Vel<L>::cy(i), cz = Vel<L>::cz(i);
        const int q = nb.src(cx, cy, cz);  // y - c_i
        R cf = R(0);
        if (cx) cf += R(cx) * W[q];
        if (cy) cf += R(cy) * W[V + q];
        if (cz) cf += R(cz) * W[2 * V + q];
        R rf = cf;
        if constexpr (TOTAL) {
            rf = mul_rn(a.c.rho0 + drho[q], cf);  // rounded: c and -c cancel where nothing varies
            if (i < 7)
                axp += cf;
            else
                edp += cf;
        }
        if (i < 7)
            ax += rf;
        else
            ed += rf;
    }
    mubar[s] = R(-3.0 / 18) * ax + R(-3.0 / 36) * ed;
    if constexpr (TOTAL) rb1[s] += R(1.0 / 18) * axp + R(1.0 / 36) * edp;
}

// rhobar = rb1 + psi''(rho) mubar - kappa lap(mubar), added to every population
// (or, with rb_out, stored for the next adjoint step of a segment to add);
// kappa, A, B gradients.  The kappa gradient -sum mubar lap(rho) is formed from the
// differences along each of the nine velocity pairs, 6 sum_k w_k (mubar(r + c_k) -
// mubar(r)) (rho(r + c_k) - rho(r)): the lattice Laplacian is symmetric, and no part
// of a field that is the same everywhere comes in.  (As -sum rho lap(mubar) the
// rounding of the Laplacian was multiplied by rho - rho0: a fluid at rho0 - 0.5 lost
// two to three digits.)
template <class R>
__global__ void __launch_bounds__(128)
    k_adj_rho(const AdjArgs<R> a, const R* drho, const R* mubar,
              const R* rb1, R* __restrict__ lam, R* __restrict__ rb_out, double* __restrict__ rows,
              const Tiling t)
{
    pdl_wait();
    const int3 r = tile_site<1, 2, false>(t, threadIdx.x);
    R gp[3] = {R(0), R(0), R(0)};
    if (r.x < a.X && r.y < a.Y && r.z < a.Z) {
        const long V = a.V;
        const int s = r.x + a.X * (r.y + a.Y * r.z);
        const Nbhd nb(r.x, r.y, r.z, a.X, a.Y, a.Z);
        const R mb = mubar[s], r0 = drho[s];
        R ax = R(0), ed = R(0), kax = R(0), ked = R(0);
#pragma unroll
        for (int i = 1; i < 19; ++i) {
            const int q = nb.src(-Vel<L>::cx(i), -Vel<L>::cy(i), -Vel<L>::cz(i));
            const R v = mubar[q] - mb;
            if (i < 7)
                ax += v;
            else
                ed += v;
            if (i & 1) {  // c of the pair (c, -c)
                if (i < 7)
                    kax += v * (drho[q] - r0);
                else
                    ked += v * (drho[q] - r0);
            }
        }
        const R lapm = R(1.0 / 3) * ax + R(1.0 / 6) * ed;  // 6 sum_i w_i (..)
        const R d = r0 + a.rho0_minus_rhoc;
        const R psi2 = a.A + R(3) * a.B * d * d;
        const R rb = rb1[s] + psi2 * mb - a.kappa * lapm;
        if (rb_out)
            rb_out[s] = rb;
        else
#pragma unroll
            for (int i = 0; i < 19; ++i) lam[(long)i * V + s] += rb;
        gp[0] = R(1.0 / 3) * kax + R(1.0 / 6) * ked;  // kappa
        gp[1] = mb * d;                               // A
        gp[2] = mb * d * d * d;                       // B
    }
    block_rows<3>(gp, rows + 3 * (long)blockIdx.x);
}

// lam += rb on every population: the deferred density part of the last step
template <class R>
__global__ void k_add_rb(R* __restrict__ lam, const R* rb, long V)
{
    pdl_wait();
    for (long s = blockIdx.x * (long)blockDim.x + threadIdx.x; s < V; s += (long)gridDim.x * blockDim.x) {
        const R r = rb[s];
#pragma unroll
        for (int i = 0; i < 19; ++i) lam[(long)i * V + s] += r;
    }
}

// Column blockIdx.x of the block rows of step blockIdx.y (nc rows of the
// collision's three columns, then nr of k_adj_rho's) summed into
// part[step * 6 + column].
__global__ void __launch_bounds__(256) k_sum_grads(const double* rows, int nc, int nr,
                                                   double* __restrict__ part)
{
    __shared__ double sh[256];
    pdl_wait();
    const int c = blockIdx.x, n = c < 3 ? nc : nr;
    const double* p = rows + 3 * ((long)blockIdx.y * (nc + nr) + (c < 3 ? 0 : nc)) + c % 3;
    double acc = 0.0;
    for (int r = threadIdx.x; r < n; r += blockDim.x) acc += p[(long)r * 3];
    sh[threadIdx.x] = acc;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.y * 6 + c] = sh[0];
}

// The steps' sums added to their parameters, the last step first: columns
// (bulk, shear, ghost, kappa, A, B) go to grad (omega_shear, omega_bulk,
// omega_ghost, kappa, A, B), the free-energy columns only for the non-ideal fluid.
__global__ void k_add_grads(const double* part, int n, double* __restrict__ grad, int nonideal)
{
    pdl_wait();
    const int c = threadIdx.x;
    if (c >= 6 || (c >= 3 && !nonideal)) return;
    double acc = grad[c == 0 ? 1 : c == 1 ? 0 : c];
    for (int k = n - 1; k >= 0; --k) acc += part[k * 6 + c];
    grad[c == 0 ? 1 : c == 1 ? 0 : c] = acc;
}

template <class R>
AdjArgs<R> make_adj(const HostModel& m, const Coll<R>& c)
{
    AdjArgs<R> a{};
    a.c = c;
    a.X = m.X;
    a.Y = m.Y;
    a.Z = m.Z;
    a.V = m.V;
    a.A = R(m.A);
    a.B = R(m.B);
    a.kappa = R(m.kappa);
    a.rho0_minus_rhoc = R(m.rho0 - m.rho_c);
    const double om[3] = {m.om_b, m.om_s, m.om_g};
    for (int c = 0; c < 3; ++c) {
        a.inv_om[c] = R(1.0 / om[c]);
        a.dln_ns[c] = R((1.0 - om[c]) / (om[c] * (2.0 - om[c])));
    }
    return a;
}

// rho and mu of `n` states, V values each, the states one after another.
template <class R>
cudaError_t adjoint_fields_t(const HostModel& m, const Coll<R>& c, const R* states, int n, R* rho, R* mu,
                             cudaStream_t st)
{
    const unsigned nb = (unsigned)std::min<long>((m.V + 127) / 128, 152 * 16);
    cudaError_t e = launch_chain(k_adj_density<R>, dim3(nb, n), dim3(128), st, states, rho, m.V);
    if (e != cudaSuccess) return e;
    const AdjArgs<R> a = make_adj<R>(m, c);
    StepArgs<R> sa{};
    sa.c = c;
    sa.X = m.X;
    sa.Y = m.Y;
    sa.Z = m.Z;
    sa.V = m.V;
    sa.A = a.A;
    sa.B = a.B;
    sa.kappa = a.kappa;
    sa.rho0_minus_rhoc = a.rho0_minus_rhoc;
    sa.pgrad = R(m.total ? 1 : 0);
    const R* crho = rho;
    if constexpr (std::is_same<R, float>::value) {
        const int gx = m.X % 4 == 0 && m.V % 4 == 0 ? 4 : m.X % 2 == 0 ? 2 : 1;
        const Tiling t = make_tiling(m.X, m.Y, (m.Z + 1) / 2, gx == 4 ? 4 : 2, 128, 2);
        const auto k = gx == 4 ? k_force_mu<4> : gx == 2 ? k_force_mu<2> : k_force_mu<1>;
        return launch_chain(k, dim3(t.blocks(), n), dim3(128), st, sa, crho, mu, t, false);
    } else {
        const Tiling t = make_tiling(m.X, m.Y, m.Z, 1, kSitesThreads, 2);
        return launch_chain(k_mu_field<R>, dim3(t.blocks(), n), dim3(kSitesThreads), st, sa, crho, mu, t);
    }
}

// the collision (two sites per thread in FP32) and k_adj_mu, k_adj_rho
Tiling collide_tiling(const HostModel& m, int prec)
{
    return make_tiling(m.X, m.Y, m.Z, prec == FLB_FP64 ? 1 : 2, 128, 2);
}
Tiling adjoint_tiling(const HostModel& m) { return make_tiling(m.X, m.Y, m.Z, 1, 128, 2); }

template <class T, class R, bool AL>
auto collide_kernel(const HostModel& m)
{
    return !m.nonideal ? k_adj_collide<T, R, AL, false, false>
           : m.total   ? k_adj_collide<T, R, AL, true, true>
                       : k_adj_collide<T, R, AL, true, false>;
}

template <class R>
cudaError_t adjoint_step_t(const HostModel& m, const Coll<R>& c, const R* gn, const R* rho, const R* mu,
                           const R* lam_next, const R* rb_next, R* lam, R* rb_out, R* work, double* rows,
                           cudaStream_t st)
{
    constexpr bool f32 = std::is_same<R, float>::value;
    using T = std::conditional_t<f32, F2, R>;
    const long V = m.V;
    R* W = work;
    R* mubar = work + 3 * V;
    R* rb1 = work + 4 * V;
    const AdjArgs<R> a = make_adj<R>(m, c);
    const Tiling tc = collide_tiling(m, f32 ? FLB_FP32 : FLB_FP64), t = adjoint_tiling(m);
    const dim3 b(128);
    // the caller's arrays may begin at any value
    const bool al = f32 && m.X % 2 == 0 && (((uintptr_t)gn | (uintptr_t)lam_next | (uintptr_t)lam) & 7) == 0;
    const auto k = al ? collide_kernel<T, R, f32>(m) : collide_kernel<T, R, false>(m);
    cudaError_t e = launch_chain(k, dim3(tc.blocks()), b, st, a, gn, rho, mu, lam_next, rb_next, lam, W, rb1, rows, tc);
    if (e != cudaSuccess || !m.nonideal) return e;
    const R* cW = W;
    const R* cmubar = mubar;
    const R* crb1 = rb1;
    const dim3 g(t.blocks());
    e = launch_chain(m.total ? k_adj_mu<R, true> : k_adj_mu<R, false>, g, b, st, a, rho, cW, mubar, rb1, t);
    if (e != cudaSuccess) return e;
    return launch_chain(k_adj_rho<R>, g, b, st, a, rho, cmubar, crb1, lam, rb_out, rows + 3 * (size_t)tc.blocks(), t);
}

}  // namespace

cudaError_t adjoint_fields(const HostModel& m, int prec, const void* states, int n, void* rho, void* mu,
                           cudaStream_t st)
{
    if (!m.nonideal) return cudaSuccess;
    if (prec == FLB_FP64)
        return adjoint_fields_t<double>(m, coll_fp64(m, 0), (const double*)states, n, (double*)rho, (double*)mu, st);
    return adjoint_fields_t<float>(m, coll_fp32(m, 0), (const float*)states, n, (float*)rho, (float*)mu, st);
}

cudaError_t adjoint_step(const HostModel& m, int prec, uint64_t step, const void* gn, const void* rho, const void* mu,
                         const void* lam_next, const void* rb_next, void* lam, void* rb_out, void* work, double* rows,
                         cudaStream_t st)
{
    if (prec == FLB_FP64)
        return adjoint_step_t<double>(m, coll_fp64(m, step), (const double*)gn, (const double*)rho,
                                      (const double*)mu, (const double*)lam_next, (const double*)rb_next, (double*)lam,
                                      (double*)rb_out, (double*)work, rows, st);
    return adjoint_step_t<float>(m, coll_fp32(m, step), (const float*)gn, (const float*)rho, (const float*)mu,
                                 (const float*)lam_next, (const float*)rb_next, (float*)lam, (float*)rb_out,
                                 (float*)work, rows, st);
}

cudaError_t adjoint_grads(const HostModel& m, int prec, const double* rows, int n, double* part, double* grad,
                          cudaStream_t st)
{
    const int nc = (int)collide_tiling(m, prec).blocks();
    cudaError_t e = launch_chain(k_sum_grads, dim3(m.nonideal ? 6 : 3, n), dim3(256), st, rows, nc,
                                 adjoint_rows(m, prec) - nc, part);
    if (e != cudaSuccess) return e;
    return launch_chain(k_add_grads, dim3(1), dim3(32), st, (const double*)part, n, grad, m.nonideal);
}

cudaError_t adjoint_add_rb(const HostModel& m, int prec, void* lam, const void* rb, cudaStream_t st)
{
    const dim3 nb((unsigned)std::min<long>((m.V + 255) / 256, 152 * 16)), b(256);
    if (prec == FLB_FP64) return launch_chain(k_add_rb<double>, nb, b, st, (double*)lam, (const double*)rb, m.V);
    return launch_chain(k_add_rb<float>, nb, b, st, (float*)lam, (const float*)rb, m.V);
}

int adjoint_rows(const HostModel& m, int prec)
{
    return (int)(collide_tiling(m, prec).blocks() + adjoint_tiling(m).blocks());
}

}  // namespace flb
