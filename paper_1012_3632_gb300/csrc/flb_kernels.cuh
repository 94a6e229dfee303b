// flb_kernels.cuh -- kernel templates of the fluctuating LB step.
//
// Storage: two structure-of-arrays buffers of deviations g_i = f_i - w_i rho0,
// layout [i][z][y][x].  A buffer holds the post-collision populations f* of
// the last completed step; the paper's pre-collision state is recovered by a
// pull, f^LB_i(r, t) = f*_i(r - c_i, t - 1) (streaming of Eq. (lbe-gen)).
//
// One step (Sec. V, Eq. (lbe-mom)) per site r, fused in one kernel:
//   pull g_i(r - c_i) -> moments -> relax, force, noise -> back-transform
//   -> write g*_i(r) into the other buffer.
// The non-ideal fluid (App. A) first needs rho on a neighbourhood, drho(r) =
// sum_i g*_i(r - c_i), and mu = psi'(rho) - kappa lap rho on a smaller one.  D3Q19:
// passes over the whole lattice write both fields before the collision reads them
// (k_density, k_mu_field here; flb_force.cuh for packed storage).  D2Q9 force model:
// density and mu of a tile with its halo in shared memory, one launch.  D2Q9
// modified equilibrium: the density field is written first, no mu.
#pragma once

#include <type_traits>

#include "flb_device.cuh"

namespace flb {

// Programmatic dependent launch.  A kernel launched with launch_chain may start
// while the last blocks of the kernel before it on the stream are ending:
// pdl_wait waits until everything before this kernel is complete and visible
// and comes before any access to memory.  The source has to fix that order: loads
// in inline PTX are asm volatile, which keep their place behind the wait, and a
// pointer that a kernel reads through is not __restrict__ (data that nothing
// writes while the kernel runs may be loaded at any point of it, and the kernel
// before may still run).  A kernel triggers its dependent
// before its blocks' end only where that one has work that needs no memory, the
// noise, and both fit the chip (EARLY), and only after its own wait, so that no
// more than two kernels are under way.  Elsewhere blocks that start while this
// kernel still computes are placed on the SMs that happen to have room, several
// on one, and wait there (a trigger at the start: 48^3 force model 15.7 instead
// of 9.7 us a step, 160 x 128 in FP64 30.9 instead of 12.1; a trigger before the
// stores: ideal step 256^3 420 instead of 417).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Indices of the 3x3x3 neighbourhood of (x, y, z) on a periodic X*Y*Z lattice:
// xv[1+dx] + rb[1+dy][1+dz] is the site index of (x+dx, y+dy, z+dz).
struct Nbhd {
    int xv[3];
    int rb[3][3];
    __device__ __forceinline__ Nbhd(int x, int y, int z, int X, int Y, int Z)
    {
        xv[0] = wrap_once(x - 1, X);
        xv[1] = x;
        xv[2] = wrap_once(x + 1, X);
        const int yv[3] = {wrap_once(y - 1, Y), y, wrap_once(y + 1, Y)};
        const int zv[3] = {wrap_once(z - 1, Z), z, wrap_once(z + 1, Z)};
#pragma unroll
        for (int a = 0; a < 3; ++a)
#pragma unroll
            for (int b = 0; b < 3; ++b) rb[a][b] = X * (yv[a] + Y * zv[b]);
    }
    // index of r - c for c = (cx, cy, cz)
    __device__ __forceinline__ int src(int cx, int cy, int cz) const { return xv[1 - cx] + rb[1 - cy][1 - cz]; }
};

// Tiles of threads over the lattice: rows of 2^lw threads (each N sites along
// x), 2^lh rows in y and one or two planes in z.  Tiles are numbered along one
// grid dimension, x fastest (no axis meets a grid limit of 65535).  Or (threads)
// no tiles: thread n of the grid takes the n-th N sites, row after row.
struct Tiling {
    int lw, lh;
    int ntx, nty, ntz;
    uint32_t mx, sx, my, sy;  // quotients by ntx and nty: (umulhi(n, m) + n) >> s, n < 2^31
    int threads;              // != 0: threads in line over rows of ntx, nty rows, ntz planes
    unsigned blocks() const
    {
        const long n = (long)ntx * nty * ntz;
        return (unsigned)(threads ? (n + threads - 1) / threads : n);
    }
    // a grid of three dimensions where its limits allow, for kernels that find their
    // tile by grid_tile
    dim3 grid() const { return threads || nty > 65535 || ntz > 65535 ? dim3(blocks()) : dim3(ntx, nty, ntz); }
};

inline void fast_div(uint32_t d, uint32_t& m, uint32_t& s)
{
    for (s = 0; (1u << s) < d; ++s) {
    }
    m = (uint32_t)(((1ull << 32) * ((1ull << s) - d)) / d + 1);
}
__device__ __forceinline__ uint32_t fast_quot(uint32_t n, uint32_t m, uint32_t s) { return (__umulhi(n, m) + n) >> s; }

// The row width that covers an X x Y plane at the least cost: the number of
// tiles, weighed by what the narrower rows lose on partial sectors (measured on
// the pair kernels at X = 36 to 129: rows of 64 sites and of 32 alike, 16 worth
// 1.2, 8 worth 1.6 tiles; 129 x 95 x 67 force model, rows of 64 / 32 / 16 / 8:
// 51.7, 46.8, 48.3, 65.9 us).
inline Tiling make_tiling(int X, int Y, int Z, int N, int threads, int planes)
{
    Tiling t{};
    int lt = 5;  // log2 of the threads per plane
    while ((1 << lt) * planes < threads) ++lt;
    double best = 0.0;
    for (int lw = 5; lw >= 2; --lw) {
        const int w = N << lw, lh = lt - lw, h = 1 << lh, nx = (X + w - 1) / w, ny = (Y + h - 1) / h;
        const double cost = (double)nx * ny * (w >= 64 ? 1.0 : w >= 32 ? 1.05 : w >= 16 ? 1.2 : w >= 8 ? 1.6 : 2.5);
        if (best > 0.0 && cost >= best) continue;
        best = cost;
        t.lw = lw;
        t.lh = lh;
        t.ntx = nx;
        t.nty = ny;
    }
    t.ntz = (Z + planes - 1) / planes;
    // Rows that fill no tile well: the threads in line over all rows.  Measured, us per
    // step, tiles / in line: ideal 73 x 55 x 77 13.6 / 10.6, 129 x 95 x 67 29.5 / 25.2,
    // 172 x 202 x 79 (tiles 10 % empty) 77.9 / 73.0, force model 129 x 95 x 67 47.2 /
    // 39.8, 39 x 152 x 148 52.1 / 42.7.
    const long p = (X + N - 1) / N;
    if (1.1 * (double)(p * Y) < best * (1 << lt) && p * Y * Z < (1l << 31)) {
        t.threads = threads;
        t.ntx = (int)p;
        t.nty = Y;
        t.ntz = Z;
    }
    fast_div((uint32_t)t.ntx, t.mx, t.sx);
    fast_div((uint32_t)t.nty, t.my, t.sy);
    return t;
}

// First site (x, y, z) of thread `tid` of tile b (this block's) of PLANES planes;
// REV: the z planes in descending order.  LINE: t may have its threads in line.
template <int N, int PLANES, bool REV, bool LINE = true>
__device__ __forceinline__ int3 tile_site(const Tiling& t, int tid, uint32_t b)
{
    if (LINE && t.threads) b = b * t.threads + tid;
    const uint32_t r = fast_quot(b, t.mx, t.sx), bx = b - r * t.ntx;
    const uint32_t rz = fast_quot(r, t.my, t.sy), by = r - rz * t.nty;
    const int bz = REV ? t.ntz - 1 - (int)rz : (int)rz;
    if (LINE && t.threads) return make_int3(N * (int)bx, (int)by, (int)rz < t.ntz ? bz : t.ntz);  // past the last row: outside
    const int tx = tid & ((1 << t.lw) - 1), row = tid >> t.lw;
    return make_int3(N * (((int)bx << t.lw) + tx), ((int)by << t.lh) + (row & ((1 << t.lh) - 1)),
                     PLANES * bz + (row >> t.lh));
}

template <int N, int PLANES, bool REV>
__device__ __forceinline__ int3 tile_site(const Tiling& t, int tid)
{
    return tile_site<N, PLANES, REV>(t, tid, blockIdx.x);
}

// The same for a grid of Tiling::grid(): ten instructions fewer where no quotient
// is needed, which the issue-bound steps notice (BF16 256^3 ideal 374.7 -> 372.1
// us, with the pulls' row offsets as sums of two 370.9); not LINE, where it need
// not look for threads in line (force model 8 steps 256^3 BF16 4867 -> 4768 us).
template <int N, int PLANES, bool REV, bool LINE>
__device__ __forceinline__ int3 grid_tile(const Tiling& t, int tid)
{
    if (gridDim.y * gridDim.z == 1) return tile_site<N, PLANES, REV, LINE>(t, tid, blockIdx.x);
    const int bz = REV ? t.ntz - 1 - (int)blockIdx.z : (int)blockIdx.z;
    const int tx = tid & ((1 << t.lw) - 1), row = tid >> t.lw;
    return make_int3(N * (((int)blockIdx.x << t.lw) + tx), ((int)blockIdx.y << t.lh) + (row & ((1 << t.lh) - 1)),
                     PLANES * bz + (row >> t.lh));
}

// Velocity tables for the pull / scatter addressing (same order as the API).
template <class L>
struct Vel;
template <>
struct Vel<D2Q9> {
    __device__ __forceinline__ static int cx(int i)
    {
        return (i == 1 || i == 5 || i == 8) ? 1 : (i == 3 || i == 6 || i == 7) ? -1 : 0;
    }
    __device__ __forceinline__ static int cy(int i)
    {
        return (i == 2 || i == 5 || i == 6) ? 1 : (i == 4 || i == 7 || i == 8) ? -1 : 0;
    }
    __device__ __forceinline__ static int cz(int) { return 0; }
    __device__ __forceinline__ static double w(int i) { return i == 0 ? 4.0 / 9 : i < 5 ? 1.0 / 9 : 1.0 / 36; }
};
template <>
struct Vel<D3Q19> {
    __device__ __forceinline__ static int cx(int i)
    {
        return (i == 1 || i == 7 || i == 9 || i == 11 || i == 13) ? 1
             : (i == 2 || i == 8 || i == 10 || i == 12 || i == 14) ? -1 : 0;
    }
    __device__ __forceinline__ static int cy(int i)
    {
        return (i == 3 || i == 7 || i == 10 || i == 15 || i == 17) ? 1
             : (i == 4 || i == 8 || i == 9 || i == 16 || i == 18) ? -1 : 0;
    }
    __device__ __forceinline__ static int cz(int i)
    {
        return (i == 5 || i == 11 || i == 14 || i == 15 || i == 18) ? 1
             : (i == 6 || i == 12 || i == 13 || i == 16 || i == 17) ? -1 : 0;
    }
    __device__ __forceinline__ static double w(int i) { return i == 0 ? 1.0 / 3 : i < 7 ? 1.0 / 18 : 1.0 / 36; }
};

// Pull g_i(r - c_i) for all i.
template <class L, class R, class S>
__device__ __forceinline__ void pull(const S* src, long V, const Nbhd& nb, R g[L::Q])
{
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
        g[i] = load_s<R>(src + (long)i * V + nb.src(Vel<L>::cx(i), Vel<L>::cy(i), Vel<L>::cz(i)));
}

// Base pointers of the Q population planes of the source and destination
// buffers (in the parameter bank): a population address is one 32-bit site
// offset from a per-direction base.
template <class S>
struct Planes {
    const S* src[19];
    S* dst[19];
};

template <class S>
Planes<S> make_planes(const void* src, void* dst, int Q, long V)
{
    Planes<S> p{};
    for (int i = 0; i < Q; ++i) {
        p.src[i] = (const S*)src + (long)i * V;
        p.dst[i] = (S*)dst + (long)i * V;
    }
    return p;
}

// Pull g_i(r - c_i) through the plane pointers.
template <class L, class R, class S>
__device__ __forceinline__ void pull_planes(const Planes<S>& P, const Nbhd& nb, R g[L::Q])
{
#pragma unroll
    for (int i = 0; i < L::Q; ++i)
        g[i] = load_s<R>(P.src[i] + nb.src(Vel<L>::cx(i), Vel<L>::cy(i), Vel<L>::cz(i)));
}

// Cache-hinted FP32 loads (PTX ld.global with an L1 eviction priority and an
// L2 prefetch size).  stream2/stream1: populations read once per kernel by the
// ideal step and the force collision -- not allocated in L1, the L2 fetches
// 256-byte sectors.  keep4/keep1: the quads of the force model's density pass,
// whose lines the loads of neighbouring sites (c_x = +-1) touch again -- kept in L1
// with the evict_last priority, 256-byte L2 fetches.
__device__ __forceinline__ float2 ld_stream2(const float* p)
{
    float2 v;
    asm volatile("ld.global.L1::no_allocate.L2::256B.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld_stream1(const float* p)
{
    float v;
    asm volatile("ld.global.L1::no_allocate.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float4 ld_keep4(const float* p)
{
    float4 v;
    asm volatile("ld.global.L1::evict_last.L2::256B.v4.f32 {%0, %1, %2, %3}, [%4];"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
        : "l"(p));
    return v;
}
__device__ __forceinline__ float ld_keep1(const float* p)
{
    float v;
    asm volatile("ld.global.L1::evict_last.L2::256B.f32 %0, [%1];" : "=f"(v) : "l"(p));
    return v;
}

// Storage access of the two-sites-per-thread kernels, FP32 in registers:
// S = float, or __nv_bfloat16 (a bf16 widens to FP32 exactly by a 16-bit
// shift; stores round to nearest even, as store_s does).  stream: the ideal
// step's hints above; keep: the density pass's; plain: no hint.
template <class S>
struct Packed;
template <>
struct Packed<float> {
    static __device__ __forceinline__ float2 stream2(const float* p) { return ld_stream2(p); }
    static __device__ __forceinline__ float stream1(const float* p) { return ld_stream1(p); }
    static __device__ __forceinline__ float4 keep4(const float* p) { return ld_keep4(p); }
    static __device__ __forceinline__ float keep1(const float* p) { return ld_keep1(p); }
    static __device__ __forceinline__ float2 plain2(const float* p) { return *reinterpret_cast<const float2*>(p); }
    static __device__ __forceinline__ float plain1(const float* p) { return *p; }
    static __device__ __forceinline__ void store2(float* p, float2 v) { __stcs(reinterpret_cast<float2*>(p), v); }
    static __device__ __forceinline__ void store1(float* p, float v) { __stcs(p, v); }
};
template <>
struct Packed<__nv_bfloat16> {
    using B = __nv_bfloat16;
    static __device__ __forceinline__ float lo(uint32_t u) { return __uint_as_float(u << 16); }
    static __device__ __forceinline__ float hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }
    static __device__ __forceinline__ float2 stream2(const B* p)
    {
        uint32_t u;
        asm volatile("ld.global.L1::no_allocate.L2::256B.b32 %0, [%1];" : "=r"(u) : "l"(p));
        return make_float2(lo(u), hi(u));
    }
    static __device__ __forceinline__ float stream1(const B* p)
    {
        unsigned short u;
        asm volatile("ld.global.L1::no_allocate.L2::256B.b16 %0, [%1];" : "=h"(u) : "l"(p));
        return lo(u);
    }
    static __device__ __forceinline__ float4 keep4(const B* p)
    {
        uint32_t a, b;
        asm volatile("ld.global.L1::evict_last.L2::256B.v2.b32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "l"(p));
        return make_float4(lo(a), hi(a), lo(b), hi(b));
    }
    static __device__ __forceinline__ float keep1(const B* p)
    {
        unsigned short u;
        asm volatile("ld.global.L1::evict_last.L2::256B.b16 %0, [%1];" : "=h"(u) : "l"(p));
        return lo(u);
    }
    static __device__ __forceinline__ float2 plain2(const B* p)
    {
        const uint32_t u = *reinterpret_cast<const uint32_t*>(p);
        return make_float2(lo(u), hi(u));
    }
    static __device__ __forceinline__ float plain1(const B* p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void store2(B* p, float2 v)
    {
        const __nv_bfloat162 b = __float22bfloat162_rn(v);
        __stcs(reinterpret_cast<unsigned int*>(p), *reinterpret_cast<const unsigned int*>(&b));
    }
    static __device__ __forceinline__ void store1(B* p, float v) { store_stream<float, B>(p, v); }
};

// ---------------------------------------------------------------------------
// Step parameters
// ---------------------------------------------------------------------------
template <class R>
struct StepArgs {
    Coll<R> c;
    int X, Y, Z;
    long V;
    // non-ideal fluid: psi'(rho) = A (rho - rho_c) + B (rho - rho_c)^3, with
    // rho - rho_c = drho + rho0_minus_rhoc; mu = psi' - kappa lap rho.
    // pgrad = 1 when psi is the total bulk free energy: F = -rho grad mu gains
    // cs^2 grad rho = sum_i w_i c_i rho(r + c_i), which cancels the LB's own
    // ideal-gas pressure gradient (Eq. (he-force)); pgrad = 0 otherwise.
    R A, B, kappa, rho0_minus_rhoc, pgrad;
    R inv_v, inv_v_lo;  // 1 / V and what its rounding left
};

// ---------------------------------------------------------------------------
// Density gather: drho(r) = sum_i g*_i(r - c_i), the density deviation the
// coming step sees (needed on a neighbourhood by the force).
// ---------------------------------------------------------------------------
constexpr int kSitesThreads = 128;

template <class L, class R, class S>
__global__ void __launch_bounds__(kSitesThreads)
    k_density(const S* src, R* __restrict__ drho, int X, int Y, int Z, const Tiling t)
{
    pdl_wait();
    const int3 r = tile_site<1, L::D == 3 ? 2 : 1, false>(t, threadIdx.x);
    if (r.x >= X || r.y >= Y || r.z >= Z) return;
    const Nbhd nb(r.x, r.y, r.z, X, Y, Z);
    R g[L::Q], m[L::Q];
    pull<L>(src, (long)X * Y * Z, nb, g);
    L::moments(g, m);
    drho[r.x + X * (r.y + Y * r.z)] = m[0];
}

// ---------------------------------------------------------------------------
// Fused pull + collide + store, one site per lane: FP64 storage, the D2Q9 ideal
// gas.  FORCE (D3Q19): F = -rho grad mu with mu written by k_mu_field before;
// TOTAL: psi is the total bulk free energy, F gains cs^2 grad rho.
// SPLIT (FP64, small lattices): a block of four warps steps 32 sites; the first
// pulls and collides, the others draw the normals meanwhile.
//
// LINE: t may have its threads in line (grid_tile).  Single precision is bound by
// issue slots: with the tile number along one dimension, and idle lanes sent to the
// first site before they return, BF16 2048 x 2048 took 62.3 us a step, now 54.2,
// 255^3 478, now 461 to 465.
//
// FP64: the FP64 pipe (16 cycles per warp instruction of an SM) where the
// lattice fills the chip, 64^3 force model 198 us a step (840 before: a column
// march on 64 blocks that formed densities and mu several times over, normals
// on the same pipe); below, the latency of one warp's chain of instructions,
// 32 x 32 5.2 us (15.1 on 4 blocks of 256).
// ---------------------------------------------------------------------------
template <class L, class R, class S, bool FORCE, bool TOTAL, bool SPLIT, bool LINE>
__global__ void __launch_bounds__(kSitesThreads)
    k_sites(const StepArgs<R> a, const __grid_constant__ Planes<S> P, const R* drho,
            const R* mu, const Tiling t)
{
    constexpr int PLANES = L::D == 3 && !SPLIT ? 2 : 1, NPAIR = (L::NNC + 1) / 2;
    __shared__ R zs[SPLIT ? 2 * NPAIR : 1][32];
    pdl_wait();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, X = a.X, Y = a.Y, Z = a.Z;
    const int3 r = grid_tile<1, PLANES, false, LINE>(t, SPLIT ? lane : (int)threadIdx.x);
    const bool in = r.x < X && r.y < Y && r.z < Z;
    if (!SPLIT && !in) return;
    const int x = in ? r.x : 0, y = in ? r.y : 0, z = in ? r.z : 0;  // idle lanes of SPLIT repeat the first site
    const int s = x + X * (y + Y * z);
    if constexpr (SPLIT) {
        if (warp > 0) {
            if (!a.c.noise) return;
            for (int p = warp - 1; p < NPAIR; p += 3)
                normal_pair(a.c.key, (uint32_t)s, a.c.step, p, a.c.replica, zs[2 * p][lane], zs[2 * p + 1][lane]);
            __syncthreads();
            return;
        }
    }
    const Nbhd nb(x, y, z, X, Y, Z);
    R g[L::Q];
    pull_planes<L>(P, nb, g);
    R F[3] = {R(0), R(0), R(0)};
    if constexpr (FORCE) {
        if constexpr (std::is_same<R, float>::value) {
            // grad = 3 sum_i w_i c_i mu(r + c_i); F = -rho grad mu (+ cs^2 grad rho)
            R gr[3] = {R(0), R(0), R(0)};
            auto add = [&](const R* f, R d[3]) {
#pragma unroll
                for (int i = 1; i < L::Q; ++i) {
                    const int cx = Vel<L>::cx(i), cy = Vel<L>::cy(i), cz = Vel<L>::cz(i);
                    const R wm = R(Vel<L>::w(i)) * f[nb.src(-cx, -cy, -cz)];
                    if (cx) d[0] += R(cx) * wm;
                    if (cy) d[1] += R(cy) * wm;
                    if (cz) d[2] += R(cz) * wm;
                }
            };
            add(mu, gr);
            const R pre = R(-3) * (a.c.rho0 + drho[s]);
            F[0] = pre * gr[0];
            F[1] = pre * gr[1];
            F[2] = pre * gr[2];
            if (a.pgrad != R(0)) add(drho, F);
        } else {
            // sum_i w_i c_i f(r + c_i) from the differences f(c) - f(-c) of the velocity
            // pairs (2k-1, 2k): axis pairs weigh 1/18, edge pairs 1/36
            auto grad = [&](const R* f, R d[3]) {
                R e[10];
#pragma unroll
                for (int k = 1; k <= 9; ++k) {
                    const int i = 2 * k - 1, cx = Vel<L>::cx(i), cy = Vel<L>::cy(i), cz = Vel<L>::cz(i);
                    e[k] = f[nb.src(-cx, -cy, -cz)] - f[nb.src(cx, cy, cz)];
                }
                d[0] = R(1.0 / 18) * e[1] + R(1.0 / 36) * ((e[4] + e[5]) + (e[6] + e[7]));
                d[1] = R(1.0 / 18) * e[2] + R(1.0 / 36) * ((e[4] - e[5]) + (e[8] + e[9]));
                d[2] = R(1.0 / 18) * e[3] + R(1.0 / 36) * ((e[6] - e[7]) + (e[8] - e[9]));
            };
            R d[3];
            grad(mu, d);
            const R pre = R(-3) * (a.c.rho0 + drho[s]);
            for (int k = 0; k < 3; ++k) F[k] = pre * d[k];
            if constexpr (TOTAL) {
                grad(drho, d);
                for (int k = 0; k < 3; ++k) F[k] += d[k];
            }
        }
    }
    auto normals = [&](R* q) {
        if constexpr (SPLIT) {
            __syncthreads();
#pragma unroll
            for (int k = 0; k < 2 * NPAIR; ++k) q[k] = zs[k][lane];
        } else {
            noise_normals<L::NCALL>(a.c.key, (uint32_t)s, a.c.step, a.c.replica, q);
        }
    };
    if constexpr (L::D == 3)
        L::template collide_with<FORCE>(g, F[0], F[1], F[2], a.c, normals);
    else
        L::collide_with(g, F[0], F[1], a.c, normals);
    if (!in) return;
#pragma unroll
    for (int i = 0; i < L::Q; ++i) store_stream(P.dst[i] + s, g[i]);
}

// mu = psi'(rho) - kappa lap rho of every site (D3Q19, one site per thread): the
// Laplacian is 6 sum_i w_i (rho_i - rho), in FP64 as (1/3) (axis sum) + (1/6)
// (edge sum) - 4 rho (fewer operations on the slow pipe).
template <class R>
__global__ void __launch_bounds__(kSitesThreads)
    k_mu_field(const StepArgs<R> a, const R* drho, R* __restrict__ mu, const Tiling t)
{
    using L = D3Q19;
    pdl_wait();
    const int3 r = tile_site<1, 2, false>(t, threadIdx.x);
    if (r.x >= a.X || r.y >= a.Y || r.z >= a.Z) return;
    drho += (long)blockIdx.y * a.V;  // several fields in one launch (the adjoint's states)
    mu += (long)blockIdx.y * a.V;
    const Nbhd nb(r.x, r.y, r.z, a.X, a.Y, a.Z);
    const int s = r.x + a.X * (r.y + a.Y * r.z);
    const R rc = drho[s];
    R lap = R(0), ed = R(0);
#pragma unroll
    for (int i = 1; i < L::Q; ++i) {
        const R v = drho[nb.src(-Vel<L>::cx(i), -Vel<L>::cy(i), -Vel<L>::cz(i))];
        if constexpr (std::is_same<R, float>::value)
            lap += R(Vel<L>::w(i)) * (v - rc);
        else if (i < 7)
            lap += v;
        else
            ed += v;
    }
    if constexpr (std::is_same<R, float>::value)
        lap *= R(6);
    else
        lap = R(1.0 / 3) * lap + R(1.0 / 6) * ed - R(4) * rc;
    const R d = rc + a.rho0_minus_rhoc;
    mu[s] = d * (a.A + a.B * d * d) - a.kappa * lap;
}

// ---------------------------------------------------------------------------
// D2Q9 force model with FP64 storage in one launch: a block's density tile (tile + 2-site halo)
// is gathered from the populations into shared memory, mu is formed on the tile
// + 1-site halo, then pull + collide with F = -rho grad mu + store.
// ---------------------------------------------------------------------------
template <class R, class S, int TX, int TY>
__global__ void __launch_bounds__(TX* TY)
    k_step_gather(const StepArgs<R> a, const __grid_constant__ Planes<S> P)
{
    using L = D2Q9;
    constexpr int RX = TX + 4, RY = TY + 4, MX = TX + 2, MY = TY + 2, NT = TX * TY;
    const int x = blockIdx.x * TX + threadIdx.x;
    const int y = blockIdx.y * TY + threadIdx.y;
    const int X = a.X, Y = a.Y;
    __shared__ R srho[RY * RX];
    __shared__ R smu[MY * MX];
    const int tid = threadIdx.x + TX * threadIdx.y;
    const int x0 = blockIdx.x * TX - 2, y0 = blockIdx.y * TY - 2;
    pdl_wait();
    for (int e = tid; e < RY * RX; e += NT) {
        const Nbhd nh(wrap_any(x0 + e % RX, X), wrap_any(y0 + e / RX, Y), 0, X, Y, 1);
        R g[L::Q], m[L::Q];
        pull_planes<L>(P, nh, g);
        L::moments(g, m);
        srho[e] = m[0];
    }
    __syncthreads();
    // mu = psi'(rho) - kappa lap rho on the tile + 1 halo;
    // lap phi = 6 sum_i w_i (phi(r + c_i) - phi(r))
    for (int e = tid; e < MY * MX; e += NT) {
        const int cidx = e % MX + 1 + RX * (e / MX + 1);
        const R r0 = srho[cidx];
        R lap = R(0);
#pragma unroll
        for (int i = 1; i < L::Q; ++i) {
            const int o = Vel<L>::cx(i) + RX * Vel<L>::cy(i);
            lap += R(Vel<L>::w(i)) * (srho[cidx + o] - r0);
        }
        lap *= R(6);
        const R d = r0 + a.rho0_minus_rhoc;
        smu[e] = d * (a.A + a.B * d * d) - a.kappa * lap;
    }
    __syncthreads();
    if (x >= X || y >= Y) return;
    // grad mu = 3 sum_i w_i c_i mu(r + c_i); F = -rho grad mu
    const int cm = threadIdx.x + 1 + MX * (threadIdx.y + 1);
    const int cr = threadIdx.x + 2 + RX * (threadIdx.y + 2);
    R gx = R(0), gy = R(0);
#pragma unroll
    for (int i = 1; i < L::Q; ++i) {
        const R wm = R(Vel<L>::w(i)) * smu[cm + Vel<L>::cx(i) + MX * Vel<L>::cy(i)];
        if (Vel<L>::cx(i)) gx += R(Vel<L>::cx(i)) * wm;
        if (Vel<L>::cy(i)) gy += R(Vel<L>::cy(i)) * wm;
    }
    const R pre = R(-3) * (a.c.rho0 + srho[cr]);
    R fx = pre * gx, fy = pre * gy;
    if (a.pgrad != R(0)) {
#pragma unroll
        for (int i = 1; i < L::Q; ++i) {
            const R wr = R(Vel<L>::w(i)) * srho[cr + Vel<L>::cx(i) + RX * Vel<L>::cy(i)];
            if (Vel<L>::cx(i)) fx += R(Vel<L>::cx(i)) * wr;
            if (Vel<L>::cy(i)) fy += R(Vel<L>::cy(i)) * wr;
        }
    }
    const Nbhd nb(x, y, 0, X, Y, 1);
    R g[L::Q];
    pull_planes<L>(P, nb, g);
    const int s = x + X * y;
    L::collide(g, fx, fy, a.c, (uint32_t)s, a.c.step);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) store_stream(P.dst[i] + s, g[i]);
}

// ---------------------------------------------------------------------------
// Modified-equilibrium model (Sec. IV.C), D2Q9 with FP64 storage (the others:
// k_step_swift2): the pressure p = p0(rho) - kappa rho lap rho and the
// square-gradient stress enter the equilibrium (D2Q9::collide_swift); no force.
// The density deviation is read from its field (tile + 1 halo in shared memory), the
// coloured e/eps noise comes from swift_noise: xi_e = Re(xi[s]) / V, xi_eps =
// -Im(xi[s]) / V.  p0 = rho psi' - psi (+ rho cs^2 when psi is the excess free
// energy, pgrad = 0).
// ---------------------------------------------------------------------------
template <class R>
using NoiseField = typename std::conditional<std::is_same<R, double>::value, double2, float2>::type;

template <class R, class S, int TX, int TY>
__global__ void __launch_bounds__(TX* TY)
    k_step_swift(const StepArgs<R> a, const __grid_constant__ Planes<S> P, const R* drho,
                 const NoiseField<R>* xi)
{
    using L = D2Q9;
    constexpr int RX = TX + 2, RY = TY + 2;
    __shared__ R srho[RY * RX];
    const int X = a.X, Y = a.Y;
    const int tid = threadIdx.x + TX * threadIdx.y;
    const int x0 = blockIdx.x * TX - 1, y0 = blockIdx.y * TY - 1;
    pdl_wait();
    for (int e = tid; e < RX * RY; e += TX * TY)
        srho[e] = drho[wrap_any(x0 + e % RX, X) + (long)X * wrap_any(y0 + e / RX, Y)];
    __syncthreads();
    const int x = blockIdx.x * TX + threadIdx.x, y = blockIdx.y * TY + threadIdx.y;
    if (x >= X || y >= Y) return;
    const int c = (threadIdx.x + 1) + RX * (threadIdx.y + 1);
    const R r0 = srho[c];
    R lap = R(0), gx = R(0), gy = R(0);
#pragma unroll
    for (int i = 1; i < L::Q; ++i) {
        const R v = srho[c + Vel<L>::cx(i) + RX * Vel<L>::cy(i)];
        lap += R(Vel<L>::w(i)) * (v - r0);
        if (Vel<L>::cx(i)) gx += R(Vel<L>::cx(i) * Vel<L>::w(i)) * v;
        if (Vel<L>::cy(i)) gy += R(Vel<L>::cy(i) * Vel<L>::w(i)) * v;
    }
    lap *= R(6);
    gx *= R(3);
    gy *= R(3);
    const R rho = a.c.rho0 + r0;
    const R d = r0 + a.rho0_minus_rhoc;
    const R psi = d * d * (R(0.5) * a.A + R(0.25) * a.B * d * d);
    const R psip = d * (a.A + a.B * d * d);
    const R pex = rho * psip - psi - a.pgrad * rho * R(1.0 / 3.0) - a.kappa * rho * lap;
    const int s = x + X * y;
    R xe = R(0), xp = R(0);
    if (a.c.noise) {
        const NoiseField<R> v = xi[s];
        xe = v.x * a.inv_v;
        xp = -v.y * a.inv_v;
    }
    const Nbhd nb(x, y, 0, X, Y, 1);
    R g[L::Q];
    pull_planes<L>(P, nb, g);
    L::collide_swift(g, pex, gx, gy, a.kappa, xe, xp, a.c, (uint32_t)s, a.c.step);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) store_stream(P.dst[i] + s, g[i]);
}

// ---------------------------------------------------------------------------
// D3Q19 ideal gas, FP32 or BF16 storage, two sites (x, x+1) per thread with
// packed FP32 arithmetic (F2).  AL: X even, a thread's pair never straddles a
// row and its populations at (x, x+1) are aligned to the pair's size: pulls
// along c_x = 0 are single loads of two, along c_x = +-1 the pair comes from
// (x-1, x) or (x+1, x+2).  Odd X: single loads, the last pair of a row is one
// site.
// EARLY: the normals are drawn before the wait for the step before (2.9 -> 2.3
// us at 32^3), in 32 registers more.
// Bound by DRAM at 256^3 (406 us, 152 B/site at 6.3 TB/s; 378 without the
// collision) and 128^3; small lattices by latency: chained launches 6.2 -> 2.9 us
// at 32^3, tiles that fit the row 32.6 -> 24 us at 96^3, pairs instead of single
// sites 34.9 -> 30.8 us at 129 x 95 x 67.
// ---------------------------------------------------------------------------
// FP32 storage, large lattices of whole lines (X % 32 == 0): each warp asks for
// the lines of its rows in the tile kPrefetchTiles further on, about a wave, so
// that DRAM has reads to serve while the warps compute: 417 -> 408 us at 256^3,
// 54.9 -> 53.5 at 128^3 (152 tiles 418, 304 413, 1520 416; bulk prefetches of
// whole rows 430).  Rows that share their lines with the next are better left
// alone (72^3 12.0 -> 13.3 us), and BF16 storage, whose step is bound by its
// instructions (374 -> 386).
constexpr uint32_t kPrefetchTiles = 4 * 152;
template <class S>
__device__ __forceinline__ void prefetch_rows(const S* src, const StepArgs<float>& a, const Tiling& t)
{
    const int lane = threadIdx.x & 31;
    if (a.X % 32 != 0 || t.threads || lane >= D3Q19::Q) return;
    const uint32_t b = blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z) + kPrefetchTiles;
    if (b >= gridDim.x * gridDim.y * gridDim.z) return;
    const int rows = 32 >> t.lw;  // of a warp
    for (int k = 0, row = (threadIdx.x >> 5) * rows; k < rows; ++k, ++row) {
        const int3 r = tile_site<2, 2, false, false>(t, row << t.lw, b);
        if (r.x >= a.X || r.y >= a.Y || r.z >= a.Z) continue;
        const char* p = reinterpret_cast<const char*>(src + lane * a.V + (r.x + a.X * (r.y + a.Y * r.z)));
        const int bytes = min(2 << t.lw, a.X - r.x) * (int)sizeof(S);
        for (int o = 0; o < bytes; o += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + o));
    }
}

template <class S, bool AL, int MINB, bool EARLY, bool LINE>
__global__ void __launch_bounds__(128, MINB)
    k_step2(const StepArgs<float> a, const __grid_constant__ Planes<S> P, const Tiling t)
{
    using L = D3Q19;
    using A = Packed<S>;
    if constexpr (!EARLY) pdl_wait();
    const int3 r0 = grid_tile<2, 2, false, LINE>(t, threadIdx.x);
    const int x = r0.x, y = r0.y, z = r0.z, X = a.X, Y = a.Y, Z = a.Z;
    const int s = x + X * (y + Y * z);
    F2 zn[EARLY ? 16 : 1];
    if constexpr (EARLY) {
        if (a.c.noise) noise_normals<4>(a.c.key, (uint32_t)s, a.c.step, a.c.replica, zn);
        pdl_wait();
        pdl_trigger();
    }
    if (x >= X || y >= Y || z >= Z) return;
    const int xm = x == 0 ? X - 1 : x - 1, x1 = AL ? x + 1 : x + 1 == X ? 0 : x + 1, x2 = x1 + 1 == X ? 0 : x1 + 1;
    const int XY = X * Y, yo[3] = {X * (y == 0 ? Y - 1 : y - 1), X * y, X * (y == Y - 1 ? 0 : y + 1)};
    const int zo[3] = {XY * (z == 0 ? Z - 1 : z - 1), XY * z, XY * (z == Z - 1 ? 0 : z + 1)};
    F2 g[L::Q];
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        const S* p = P.src[i] + (yo[1 - Vel<L>::cy(i)] + zo[1 - Vel<L>::cz(i)]);
        const int cx = Vel<L>::cx(i);
        if (cx == 0)
            g[i] = AL ? mk2(A::stream2(p + x)) : F2(A::stream1(p + x), A::stream1(p + x1));
        else if (cx > 0)
            g[i] = F2(A::stream1(p + xm), A::stream1(p + x));
        else
            g[i] = F2(A::stream1(p + x1), A::stream1(p + x2));
    }
    if constexpr (!EARLY && sizeof(S) == 4) prefetch_rows(P.src[0], a, t);
    if constexpr (EARLY)
        L::template collide_with<false>(g, F2(0.f), F2(0.f), F2(0.f), a.c, [&](F2* q) {
#pragma unroll
            for (int k = 0; k < 16; ++k) q[k] = zn[k];
        });
    else
        L::template collide<false>(g, F2(0.f), F2(0.f), F2(0.f), a.c, (uint32_t)s, a.c.step);
#pragma unroll
    for (int i = 0; i < L::Q; ++i) {
        if constexpr (AL) {
            A::store2(P.dst[i] + s, g[i].v);
        } else {
            A::store1(P.dst[i] + s, g[i].v.x);
            if (x + 1 < X) A::store1(P.dst[i] + s + 1, g[i].v.y);
        }
    }
}

}  // namespace flb
