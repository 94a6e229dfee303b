// flb_force.cuh -- the non-ideal steps with FP32 or BF16 storage: D2Q9 in one
// launch (k_step_gather2, k_step_swift2, at the end), D3Q19 as three launches in
// packed FP32: density (pull and sum), mu = psi'(rho) - kappa lap rho, then
// pull + collide with F = -rho grad mu.
//
// Every site's density and mu are formed once, and each pass runs at the
// occupancy that suits it.  One launch that marched columns of sites through z
// with the densities in shared-memory rings formed them 1.9 and 1.3 times over
// (tile halos, ring fills), held 12 warps per SM at two barriers a plane and
// left the chip part empty below 256^3.  Measured, march -> passes, per step:
// 256^3 FP32 757 -> 698 us (with sums 790 -> 716), BF16 660 -> 597, 128^3 FP32
// 111 -> 91, 64^3 35 -> 14.6, 129x95x67 84 -> 67.
//
// What bounds them at 256^3 FP32: density 196 us, DRAM (80 B/site, 6.8 TB/s);
// mu 46 us, L1 wavefronts of the row loads; collision 474 us, DRAM (156 B/site,
// 5.3 TB/s) with issue slots 52 % and the FMA-heavy pipe (integer multiplies of
// the noise) near as busy; with BF16 storage the issue slots alone.
//
// The collision takes the planes in descending order, so that it starts on the
// lines the density pass read last and leaves the ones the next density pass
// reads first in L2: 91.0 against 94.8 us at 128^3, 699 against 707 at 256^3.
#pragma once

#include "flb_kernels.cuh"

namespace flb {

// A row of a field around the N sites x .. x+N-1: v[0] = f(x-1), v[1..N],
// v[N+1] = f(x+N) (periodic: xm, xe; x1 the periodic x+1 of unaligned pairs).
template <int N, bool AL>
__device__ __forceinline__ void load_row(const float* p, int x, int x1, int xm, int xe, bool ends, float v[N + 2])
{
    if constexpr (N == 4) {
        const float4 m = *reinterpret_cast<const float4*>(p + x);
        v[1] = m.x;
        v[2] = m.y;
        v[3] = m.z;
        v[4] = m.w;
    } else if constexpr (AL) {
        const float2 m = *reinterpret_cast<const float2*>(p + x);
        v[1] = m.x;
        v[2] = m.y;
    } else {
        v[1] = p[x];
        v[2] = p[x1];
    }
    if (ends) {
        v[0] = p[xm];
        v[N + 1] = p[xe];
    }
}

// Density: drho(r) = sum_i g*_i(r - c_i).  GX: X % 4 == 0 (4: a quad of sites
// per thread), X even (2: a pair) or any X (1: a pair by single loads).
// SUMS: every warp also writes the mass deviation and momentum of its sites
// (FP32 within the warp).  This pass waits for memory and has the issue slots
// for it; in the collision the same sums cost 9 % (474 -> 519 us at 256^3).  At
// least 7 blocks per SM: the sums would take 88 registers and with them the
// warps that hide the loads (a step with sums 716 us, at 6 blocks 727, 8: 740).
// STATE: the pulled deviations go to P.dst as well, the states that the adjoint
// keeps (FP32; 64^3 14.7 us, without them 8.3 and a pull of their own 9.5), at 5
// blocks per SM: they are held until the last load (20 steps of 64^3, forward and
// back, 1000 -> 943 us).
template <class S, int GX, bool SUMS, bool STATE = false>
__global__ void __launch_bounds__(128, STATE ? 5 : 7) k_force_density(const __grid_constant__ Planes<S> P, float* __restrict__ rho,
                                                       float* __restrict__ rows, int X, int Y, int Z, const Tiling t)
{
    using L = D3Q19;
    using A = Packed<S>;
    constexpr int N = GX == 4 ? 4 : 2;
    pdl_wait();
    const int3 r0 = tile_site<N, 2, false>(t, threadIdx.x);
    const int x = r0.x, y = r0.y, z = r0.z, XY = X * Y;
    const bool in = x < X && y < Y && z < Z;
    if (!SUMS && !in) return;
    float v4[4] = {0.f, 0.f, 0.f, 0.f};
    if (in) {
        const int zo[3] = {XY * (z == 0 ? Z - 1 : z - 1), XY * z, XY * (z == Z - 1 ? 0 : z + 1)};
        const int yo[3] = {X * wrap_once(y - 1, Y), X * y, X * wrap_once(y + 1, Y)};
        const int xm = x == 0 ? X - 1 : x - 1, x1 = x + 1 == X ? 0 : x + 1;
        const int xl = N == 4 ? x + 3 : x1, xe = xl + 1 == X ? 0 : xl + 1;
        float* out = rho + (XY * z + X * y + x);
        if constexpr (GX == 4) {
            F2 lo[L::Q], hi[L::Q], m[L::Q], n[L::Q];
#pragma unroll
            for (int i = 0; i < L::Q; ++i) {
                const S* r = P.src[i] + (yo[1 - Vel<L>::cy(i)] + zo[1 - Vel<L>::cz(i)]);
                const float4 v = A::keep4(r + x);
                const int cx = Vel<L>::cx(i);
                if (cx == 0) {
                    lo[i] = F2(v.x, v.y);
                    hi[i] = F2(v.z, v.w);
                } else if (cx > 0) {
                    lo[i] = F2(A::keep1(r + xm), v.x);
                    hi[i] = F2(v.y, v.z);
                } else {
                    lo[i] = F2(v.y, v.z);
                    hi[i] = F2(v.w, A::keep1(r + xe));
                }
            }
            if constexpr (STATE) {  // after the loads: a store would hold back the loads behind it
#pragma unroll
                for (int i = 0; i < L::Q; ++i)
                    *reinterpret_cast<float4*>(P.dst[i] + (XY * z + X * y + x)) =
                        make_float4(lo[i].v.x, lo[i].v.y, hi[i].v.x, hi[i].v.y);
            }
            L::moments(lo, m);
            L::moments(hi, n);
            *reinterpret_cast<float4*>(out) = make_float4(m[0].v.x, m[0].v.y, n[0].v.x, n[0].v.y);
            if constexpr (SUMS) {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const F2 c = m[k] + n[k];
                    v4[k] = c.v.x + c.v.y;
                }
            }
        } else {
            F2 g[L::Q], m[L::Q];
#pragma unroll
            for (int i = 0; i < L::Q; ++i) {
                const S* r = P.src[i] + (yo[1 - Vel<L>::cy(i)] + zo[1 - Vel<L>::cz(i)]);
                const int cx = Vel<L>::cx(i);
                if (cx == 0)
                    g[i] = GX == 2 ? mk2(A::plain2(r + x)) : F2(A::plain1(r + x), A::plain1(r + x1));
                else if (cx > 0)
                    g[i] = F2(A::plain1(r + xm), A::plain1(r + x));
                else
                    g[i] = F2(A::plain1(r + x1), A::plain1(r + xe));
            }
            if constexpr (STATE) {
#pragma unroll
                for (int i = 0; i < L::Q; ++i) {
                    S* o = P.dst[i] + (XY * z + X * y + x);
                    if constexpr (GX == 2) {
                        *reinterpret_cast<float2*>(o) = g[i].v;
                    } else {
                        o[0] = g[i].v.x;
                        if (x + 1 < X) o[1] = g[i].v.y;
                    }
                }
            }
            L::moments(g, m);
            if constexpr (GX == 2) {
                *reinterpret_cast<float2*>(out) = m[0].v;
            } else {
                out[0] = m[0].v.x;
                if (x + 1 < X) out[1] = m[0].v.y;
            }
            if constexpr (SUMS) {  // GX == 2: both sites exist
#pragma unroll
                for (int k = 0; k < 4; ++k) v4[k] = m[k].v.x + m[k].v.y;
            }
        }
    }
    if constexpr (SUMS) {
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        // the sums of four values over a warp in six exchanges: halves keep two, quarters one
        const bool h16 = lane & 16, h8 = lane & 8;
        float p = h16 ? v4[2] : v4[0], q = h16 ? v4[3] : v4[1];
        p += __shfl_xor_sync(0xffffffffu, h16 ? v4[0] : v4[2], 16);
        q += __shfl_xor_sync(0xffffffffu, h16 ? v4[1] : v4[3], 16);
        float c = h8 ? q : p;
        c += __shfl_xor_sync(0xffffffffu, h8 ? p : q, 8);
        for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
        if ((lane & 7) == 0) rows[4 * (4 * (long)blockIdx.x + warp) + (lane >> 3)] = c;
    }
}

// mu = psi'(rho) - kappa lap rho of the sites of two planes z, z + 1: the 12
// rows of four planes serve both (51 -> 46 us at 256^3 against a plane per
// thread with its 9 rows).
template <int GX>
__global__ void __launch_bounds__(128)
    k_force_mu(const StepArgs<float> a, const float* rho, float* __restrict__ mu, const Tiling t,
               bool trigger)
{
    using L = D3Q19;
    constexpr int N = GX == 4 ? 4 : 2;
    pdl_wait();
    if (trigger) pdl_trigger();  // the collision draws its noise meanwhile
    int3 r0 = tile_site<N, 2, true>(t, threadIdx.x);
    const int X = a.X, Y = a.Y, Z = a.Z, XY = X * Y;
    rho += (long)blockIdx.y * a.V;  // several fields in one launch (the adjoint's states)
    mu += (long)blockIdx.y * a.V;
    // the tiling's two planes are rows of threads: here each thread takes a pair of planes
    const int x = r0.x, y = r0.y, z = 2 * r0.z;
    if (x >= X || y >= Y || z >= Z) return;
    const int z1 = z + 1 == Z ? 0 : z + 1, z2 = z1 + 1 == Z ? 0 : z1 + 1;
    const int zo[4] = {XY * (z == 0 ? Z - 1 : z - 1), XY * z, XY * z1, XY * z2};
    const int yo[3] = {X * wrap_once(y - 1, Y), X * y, X * wrap_once(y + 1, Y)};
    const int xm = x == 0 ? X - 1 : x - 1, x1 = x + 1 == X ? 0 : x + 1;
    const int xl = N == 4 ? x + 3 : x1, xe = xl + 1 == X ? 0 : xl + 1;
    float r[4][3][N + 2];  // rows (plane, dy)
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
        for (int dy = 0; dy < 3; ++dy)
            load_row<N, GX != 1>(rho + (yo[dy] + zo[k]), x, x1, xm, xe, dy == 1 || k == 1 || k == 2, r[k][dy]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        float out[N];
#pragma unroll
        for (int k = 0; k < N; k += 2) {
            // sum_i w_i (rho_i - rho) = (1/18) (axis sum) + (1/36) (edge sum) - (2/3) rho
            // (the Laplacian is 6 times it)
            F2 sax(0.f), sed(0.f);
#pragma unroll
            for (int i = 1; i < L::Q; ++i) {
                const float* w = r[h + 1 + Vel<L>::cz(i)][1 + Vel<L>::cy(i)] + (k + 1 + Vel<L>::cx(i));
                if (i < 7)
                    sax += F2(w[0], w[1]);
                else
                    sed += F2(w[0], w[1]);
            }
            const F2 rc(r[h + 1][1][k + 1], r[h + 1][1][k + 2]);
            const F2 lap = (1.0f / 18.0f) * sax + (1.0f / 36.0f) * sed - (2.0f / 3.0f) * rc;
            const F2 d = rc + a.rho0_minus_rhoc;
            const F2 m = d * (a.A + a.B * (d * d)) - (6.0f * a.kappa) * lap;
            out[k] = m.v.x;
            out[k + 1] = m.v.y;
        }
        if (h == 1 && z + 1 == Z) return;
        float* o = mu + (zo[1 + h] + X * y + x);
        if constexpr (N == 4) {
            *reinterpret_cast<float4*>(o) = make_float4(out[0], out[1], out[2], out[3]);
        } else if constexpr (GX == 2) {
            *reinterpret_cast<float2*>(o) = make_float2(out[0], out[1]);
        } else {
            o[0] = out[0];
            if (x + 1 < X) o[1] = out[1];
        }
    }
}

// Pull, collide with F = -rho grad mu and store, a site pair per thread.  AL:
// X even.  TOTAL: psi is the total bulk free energy, F gains cs^2 grad rho
// (read from the density field).  EARLY: the noise is drawn before the wait for
// mu (k_force_mu's trigger).  4 blocks per SM: 128 registers; 5 (96, 72 bytes
// spilled) measured 474 -> 480 us at 256^3.
template <class S, bool AL, bool TOTAL, bool EARLY, bool LINE>
__global__ void __launch_bounds__(128, EARLY ? 3 : 4)
    k_force_collide(const StepArgs<float> a, const __grid_constant__ Planes<S> P, const float* rho,
                    const float* mu, const Tiling t)
{
    using L = D3Q19;
    using A = Packed<S>;
    if constexpr (!EARLY) pdl_wait();
    const int3 r0 = grid_tile<2, 2, true, LINE>(t, threadIdx.x);
    const int x = r0.x, y = r0.y, z = r0.z, X = a.X, Y = a.Y, Z = a.Z, XY = X * Y;
    F2 zn[EARLY ? 16 : 1];
    if constexpr (EARLY) {
        if (a.c.noise) noise_normals<4>(a.c.key, (uint32_t)(x + X * y + XY * z), a.c.step, a.c.replica, zn);
        pdl_wait();
    }
    if (x >= X || y >= Y || z >= Z) return;
    const int xm = x == 0 ? X - 1 : x - 1, x1 = x + 1 == X ? 0 : x + 1, xe = x1 + 1 == X ? 0 : x1 + 1;
    const int yo[3] = {X * wrap_once(y - 1, Y), X * y, X * wrap_once(y + 1, Y)};
    const int zo[3] = {XY * (z == 0 ? Z - 1 : z - 1), XY * z, XY * (z == Z - 1 ? 0 : z + 1)};
    F2 g[L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const S* r = P.src[i] + (yo[1 - Vel<L>::cy(i)] + zo[1 - Vel<L>::cz(i)]);
        const int cx = Vel<L>::cx(i);
        if (cx == 0)
            g[i] = AL ? mk2(A::stream2(r + x)) : F2(A::stream1(r + x), A::stream1(r + x1));
        else if (cx > 0)
            g[i] = F2(A::stream1(r + xm), A::stream1(r + x));
        else
            g[i] = F2(A::stream1(r + x1), A::stream1(r + xe));
    }
    // sum_i w_i c_i f_i (a gradient / 3) from the differences f(c) - f(-c) of
    // the nine velocity pairs (2p-1, 2p): axis pairs weigh 1/18, edge pairs
    // 1/36; pairs 4..9: (1,1,0) (1,-1,0) (1,0,1) (1,0,-1) (0,1,1) (0,1,-1)
    auto grad = [&](const float* f, F2& gx, F2& gy, F2& gz) {
        float r[3][3][4];
#pragma unroll
        for (int dz = 0; dz < 3; ++dz)
#pragma unroll
            for (int dy = 0; dy < 3; ++dy)
                load_row<2, AL>(f + (yo[dy] + zo[dz]), x, x1, xm, xe, dy == 1 || dz == 1, r[dz][dy]);
        F2 dp[10];
#pragma unroll
        for (int k = 1; k <= 9; ++k) {
            const int i = 2 * k - 1;
            const float* u = r[1 + Vel<L>::cz(i)][1 + Vel<L>::cy(i)] + (1 + Vel<L>::cx(i));
            const float* w = r[1 - Vel<L>::cz(i)][1 - Vel<L>::cy(i)] + (1 - Vel<L>::cx(i));
            dp[k] = F2(u[0], u[1]) - F2(w[0], w[1]);
        }
        gx = (1.0f / 18.0f) * dp[1] + (1.0f / 36.0f) * ((dp[4] + dp[5]) + (dp[6] + dp[7]));
        gy = (1.0f / 18.0f) * dp[2] + (1.0f / 36.0f) * ((dp[4] - dp[5]) + (dp[8] + dp[9]));
        gz = (1.0f / 18.0f) * dp[3] + (1.0f / 36.0f) * ((dp[6] - dp[7]) + (dp[8] - dp[9]));
    };
    F2 gx, gy, gz;
    grad(mu, gx, gy, gz);
    // the density of the pulled populations, as k_force_density sums it
    F2 m[L::Q];
    L::moments(g, m);
    const F2 pre = -3.0f * (a.c.rho0 + m[0]);
    F2 fx = pre * gx, fy = pre * gy, fz = pre * gz;
    if constexpr (TOTAL) {
        F2 px, py, pz;
        grad(rho, px, py, pz);
        fx += px;
        fy += py;
        fz += pz;
    }
    const int site = x + X * y + XY * z;
    const bool two = AL || x + 1 < X;
    if constexpr (EARLY)
        L::template collide_with<true>(g, fx, fy, fz, a.c, [&](F2* q) {
#pragma unroll
            for (int k = 0; k < 16; ++k) q[k] = zn[k];
        });
    else
        L::collide(g, fx, fy, fz, a.c, (uint32_t)site, a.c.step);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        if constexpr (AL) {
            A::store2(P.dst[i] + site, g[i].v);
        } else {
            A::store1(P.dst[i] + site, g[i].v.x);
            if (two) A::store1(P.dst[i] + site + 1, g[i].v.y);
        }
    }
}

// D2Q9 force model in one launch, a site pair per thread: a block pulls the
// pairs of its tile, which stay in registers, and those of a 2-site halo, whose
// densities go to shared memory with the tile's; mu is formed on the tile + 1
// (pairs of the same grid, so that 2 columns more are formed than used), then
// the pair collides with F = -rho grad mu.  AL: X even, the pairs of every row
// begin at even x.
// 1024 x 400 FP32 lies in L2 and is bound by the latency of its three phases and
// by issue slots: 14.4 -> 9.6 us a step (9.6 -> 5.1 million warp instructions)
// against one site per thread with the tile pulled twice; 129 x 97 6.2 -> 3.1.
// Tiles of 32 x 8: 32 x 16 10.2, 64 x 8 9.9, 64 x 16 14.7, 16 x 16 11.8 us.
template <class S, bool AL, bool TOTAL, int TX, int TY>
__global__ void __launch_bounds__(TX* TY / 2)
    k_step_gather2(const StepArgs<float> a, const __grid_constant__ Planes<S> P, const Tiling t)
{
    using L = D2Q9;
    using A = Packed<S>;
    constexpr int HX = TX / 2, RX = TX + 4, RP = RX / 2, RY = TY + 4, NT = HX * TY;
    constexpr int NHALO = RP * RY - NT;  // halo pairs: two rows below and above, then a column on each side
    __shared__ float2 rho_pad[RY * RP + 2], smu[RY * RP];  // a corner pair of mu reads one site past the field
    float2* const srho = rho_pad + 1;
    pdl_wait();
    const int X = a.X, Y = a.Y, tid = threadIdx.x;
    const uint32_t ry = fast_quot(blockIdx.x, t.mx, t.sx);
    const int bx = TX * (int)(blockIdx.x - ry * t.ntx), by = TY * (int)ry;
    auto pull = [&](int x, int y, F2 g[L::Q]) {  // x, y within a few tiles of the lattice
        const int xa = wrap_any(x, X), y0 = wrap_any(y, Y);
        const int xm = xa == 0 ? X - 1 : xa - 1, x1 = xa + 1 == X ? 0 : xa + 1, xe = x1 + 1 == X ? 0 : x1 + 1;
        const int yo[3] = {X * wrap_once(y0 - 1, Y), X * y0, X * wrap_once(y0 + 1, Y)};
#pragma unroll
        for (int i = 0; i < L::Q; ++i) {
            const S* r = P.src[i] + yo[1 - Vel<L>::cy(i)];
            const int cx = Vel<L>::cx(i);
            if (cx == 0)
                g[i] = AL ? mk2(A::plain2(r + xa)) : F2(A::plain1(r + xa), A::plain1(r + x1));
            else if (cx > 0)
                g[i] = F2(A::plain1(r + xm), A::plain1(r + xa));
            else
                g[i] = F2(A::plain1(r + x1), A::plain1(r + xe));
        }
    };
    const int px = tid % HX, py = tid / HX, x = bx + 2 * px, y = by + py;
    const int own = px + 1 + RP * (py + 2);
    F2 g[L::Q], m[L::Q];
    pull(x, y, g);
    L::moments(g, m);
    srho[own] = m[0].v;
    for (int e = tid; e < NHALO; e += NT) {
        int hx, hy;
        if (e < 4 * RP) {
            hx = e % RP;
            hy = e / RP;
            if (hy >= 2) hy += TY;
        } else {
            hx = (e & 1) * (RP - 1);
            hy = 2 + ((e - 4 * RP) >> 1);
        }
        F2 h[L::Q], n[L::Q];
        pull(bx - 2 + 2 * hx, by - 2 + hy, h);
        L::moments(h, n);
        srho[hx + RP * hy] = n[0].v;
    }
    __syncthreads();
    // the differences f(c) - f(-c) of the pair at index e of a shared field
    struct Rows {
        float v[3][4];
        __device__ __forceinline__ Rows(const float2* f, int e)
        {
            const float* p = reinterpret_cast<const float*>(f);
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int o = e + RP * (k - 1);
                v[k][0] = p[2 * o - 1];
                v[k][1] = f[o].x;
                v[k][2] = f[o].y;
                v[k][3] = p[2 * o + 2];
            }
        }
        __device__ __forceinline__ F2 at(int cx, int cy) const { return F2(v[1 + cy][1 + cx], v[1 + cy][2 + cx]); }
    };
    // mu = psi'(rho) - kappa lap rho; lap phi = 6 sum_i w_i (phi(r + c_i) - phi(r))
    for (int e = RP + tid; e < RP * (RY - 1); e += NT) {
        const Rows r(srho, e);
        const F2 rc = r.at(0, 0);
        F2 ax(0.f), ed(0.f);
#pragma unroll
        for (int i = 1; i < L::Q; ++i) (i < 5 ? ax : ed) += r.at(Vel<L>::cx(i), Vel<L>::cy(i)) - rc;
        const F2 lap = (6.0f / 9.0f) * ax + (6.0f / 36.0f) * ed;
        const F2 d = rc + a.rho0_minus_rhoc;
        smu[e] = (d * (a.A + a.B * (d * d)) - a.kappa * lap).v;
    }
    __syncthreads();
    if (x >= X || y >= Y) return;
    // sum_i w_i c_i f(r + c_i) (a gradient / 3)
    auto gradient = [&](const float2* f, F2& gx, F2& gy) {
        const Rows r(f, own);
        const F2 d1 = r.at(1, 0) - r.at(-1, 0), d2 = r.at(0, 1) - r.at(0, -1);
        const F2 d5 = r.at(1, 1) - r.at(-1, -1), d8 = r.at(1, -1) - r.at(-1, 1);
        gx = (1.0f / 9.0f) * d1 + (1.0f / 36.0f) * (d5 + d8);
        gy = (1.0f / 9.0f) * d2 + (1.0f / 36.0f) * (d5 - d8);
    };
    F2 gx, gy;
    gradient(smu, gx, gy);
    const F2 pre = -3.0f * (a.c.rho0 + m[0]);
    F2 fx = pre * gx, fy = pre * gy;
    if constexpr (TOTAL) {
        gradient(srho, gx, gy);
        fx += gx;
        fy += gy;
    }
    const int site = x + X * y;
    L::collide(g, fx, fy, a.c, (uint32_t)site, a.c.step);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        if constexpr (AL) {
            A::store2(P.dst[i] + site, g[i].v);
        } else {
            A::store1(P.dst[i] + site, g[i].v.x);
            if (x + 1 < X) A::store1(P.dst[i] + site + 1, g[i].v.y);
        }
    }
}

// Modified-equilibrium step of D2Q9 (k_step_swift), a site pair per thread with
// the density rows read from the field: no shared tile to wait for.
// 1024 x 400 FP32: a step with its noise passes 35.3 -> 31.5 us against one site per
// thread, by fewer instructions and no barrier; 31.0 with the differences of the
// pressure and the stresses as fused operations (mad), which also keeps the rounding
// of single values: error against 64 bits 1.06e-7 after 20 steps of 256 x 96, 1.21e-7
// with the products rounded before they were subtracted.
template <class S, bool AL>
__global__ void __launch_bounds__(128)
    k_step_swift2(const StepArgs<float> a, const __grid_constant__ Planes<S> P, const float* drho,
                  const float2* xi, const Tiling t)
{
    using L = D2Q9;
    using A = Packed<S>;
    pdl_wait();
    const int3 r0 = tile_site<2, 1, false>(t, threadIdx.x);
    const int x = r0.x, y = r0.y, X = a.X, Y = a.Y;
    if (x >= X || y >= Y) return;
    const int xm = x == 0 ? X - 1 : x - 1, x1 = x + 1 == X ? 0 : x + 1, xe = x1 + 1 == X ? 0 : x1 + 1;
    const int yo[3] = {X * wrap_once(y - 1, Y), X * y, X * wrap_once(y + 1, Y)};
    float r[3][4];
#pragma unroll
    for (int k = 0; k < 3; ++k) load_row<2, AL>(drho + yo[k], x, x1, xm, xe, true, r[k]);
    F2 g[L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const S* p = P.src[i] + yo[1 - Vel<L>::cy(i)];
        const int cx = Vel<L>::cx(i);
        if (cx == 0)
            g[i] = AL ? mk2(A::plain2(p + x)) : F2(A::plain1(p + x), A::plain1(p + x1));
        else if (cx > 0)
            g[i] = F2(A::plain1(p + xm), A::plain1(p + x));
        else
            g[i] = F2(A::plain1(p + x1), A::plain1(p + xe));
    }
    const int site = x + X * y;
    const bool two = AL || x + 1 < X;
    F2 ne(0.f), np(0.f);
    if (a.c.noise) {
        // v / V with 1 / V in two floats: rounded once, and off the FP64 pipe
        const float2 v = xi[site], w = two ? xi[site + 1] : v;
        ne = F2(fmaf(v.x, a.inv_v, v.x * a.inv_v_lo), fmaf(w.x, a.inv_v, w.x * a.inv_v_lo));
        np = F2(-fmaf(v.y, a.inv_v, v.y * a.inv_v_lo), -fmaf(w.y, a.inv_v, w.y * a.inv_v_lo));
    }
    auto at = [&](int cx, int cy) { return F2(r[1 + cy][1 + cx], r[1 + cy][2 + cx]); };
    const F2 rc = at(0, 0);
    F2 ax(0.f), ed(0.f);
#pragma unroll
    for (int i = 1; i < L::Q; ++i) (i < 5 ? ax : ed) += at(Vel<L>::cx(i), Vel<L>::cy(i)) - rc;
    const F2 lap = mad(6.0f / 36.0f, ed, (6.0f / 9.0f) * ax);  // 6 sum_i w_i (rho_i - rho)
    const F2 d5 = at(1, 1) - at(-1, -1), d8 = at(1, -1) - at(-1, 1);
    const F2 gx = mad(3.0f / 36.0f, d5 + d8, (3.0f / 9.0f) * (at(1, 0) - at(-1, 0)));
    const F2 gy = mad(3.0f / 36.0f, d5 - d8, (3.0f / 9.0f) * (at(0, 1) - at(0, -1)));
    const F2 rho = a.c.rho0 + rc, d = rc + a.rho0_minus_rhoc, dd = d * d;
    const F2 half = mad(0.25f * a.B, dd, F2(0.5f * a.A));  // psi = d^2 half
    const F2 psip = d * mad(a.B, dd, F2(a.A));
    const F2 pex = mad(rho, mad(-a.kappa, lap, F2(a.pgrad * (-1.0f / 3.0f))), mad(rho, psip, (-1.0f * dd) * half));
    L::collide_swift(g, pex, gx, gy, a.kappa, ne, np, a.c, (uint32_t)site, a.c.step);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        if constexpr (AL) {
            A::store2(P.dst[i] + site, g[i].v);
        } else {
            A::store1(P.dst[i] + site, g[i].v.x);
            if (two) A::store1(P.dst[i] + site + 1, g[i].v.y);
        }
    }
}

}  // namespace flb
