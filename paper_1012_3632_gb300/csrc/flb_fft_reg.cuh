// flb_fft_reg.cuh -- FP32 transforms of lines, two radix passes at a time in
// registers: the kernels of a length, and the table of all lengths that have them.
#pragma once

#include <cstdint>

#include "flb_kernels.cuh"
#include "flb_swift.cuh"

namespace flb {

// Complex arithmetic on double2 (FP64 transforms) and float2 (FP32 transforms).
template <class T>
__device__ __forceinline__ T cmul(T a, T b)
{
    return T{a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <class T>
__device__ __forceinline__ T cadd(T a, T b)
{
    return T{a.x + b.x, a.y + b.y};
}
template <class T>
__device__ __forceinline__ T csub(T a, T b)
{
    return T{a.x - b.x, a.y - b.y};
}

// |a|^2 with the rounding fixed: the fused and the separate power spectrum agree
// to the bit.
__device__ __forceinline__ float norm2(float2 a) { return fmaf(a.y, a.y, __fmul_rn(a.x, a.x)); }

// Twiddle table tw[m] = exp(-2 pi i m / L), m < L, built by every block in shared
// memory: one FP32 sincospi per entry.
__device__ __forceinline__ void fill_twiddles(float2* tw, int L, float2*)
{
    for (int m = threadIdx.x; m < L; m += blockDim.x) {
        float s, c;
        sincospif(-2.0f * ((float)m / (float)L), &s, &c);
        tw[m] = make_float2(c, s);
    }
}

// Bound by latency and shared-memory passes: the radix-by-radix kernel of flb_fft.cu
// crosses shared memory once per radix and fetches a 2048-element block per
// 256 threads.  Here a thread takes Ra Rb elements q + (r0 Rb + r') L / (Ra Rb)
// of a line, which the radix-Ra butterflies j = q + r' L / (Ra Rb) and the
// radix-Rb butterflies of the next pass exchange among themselves alone, so that
// a length of up to 256 crosses shared memory once; strided lines load and
// store straight from registers, blocks keep their twiddle table for several
// groups of lines.  The arithmetic of every butterfly is that of the passes there.
// Structure factor of a 128^3 state 113 -> 59 us, 96^3 82 -> 22, 256^3 703 -> 408
// (density field and power spectrum included); 80^3 38 -> 19, 100^3 71 -> 39, 160^3
// 272 -> 118, 36^3 20 -> 11, 18^3 18 -> 10.
//
// Every length that fits has its kernels, compiled for it: three to six of the
// radices 4, 2, 3, 5 (in this order), two to a pass and the last alone where they
// are odd in number (rb = 1), at most 1024 elements (a block's lines and twiddles
// fit 48 KB); n = 0: none.  One kernel for all, with the length a number, was 1.3 to
// 1.8 times slower (64^3 21 us against 12: twice the instructions).
struct RegPlan {
    int n, ra[3], rb[3];
};
constexpr int kRegMax = 1024;
__host__ __device__ constexpr RegPlan reg_plan(int L)
{
    RegPlan p{};
    const int radices[4] = {4, 2, 3, 5};
    int k = 0, left = L;
    for (int r : radices)
        for (; left >= r && left % r == 0 && k < 7; left /= r, ++k)
            if (k < 6) (k % 2 ? p.rb : p.ra)[k / 2] = r;
    if (k % 2 && k < 6) p.rb[k / 2] = 1;
    p.n = L <= kRegMax && left == 1 && k >= 3 && k <= 6 ? (k + 1) / 2 : 0;
    return p;
}
// The lengths that have a plan, in ascending order: number and n-th of them.
constexpr int reg_index(int L)
{
    int n = 0;
    for (int l = 1; l < L; ++l) n += reg_plan(l).n != 0;
    return n;
}
constexpr int reg_length(int n)
{
    int l = 0;
    for (int k = -1; k < n;) k += reg_plan(++l).n != 0;
    return l;
}
constexpr int kRegLengths = reg_index(kRegMax + 1);

// The R-point DFT of butterfly(), on registers.
template <int R, class T>
__device__ __forceinline__ void dft(const T (&v)[R], T (&y)[R], const T* __restrict__ tw, int L)
{
    using E = decltype(T::x);
    if constexpr (R == 1) {
        y[0] = v[0];
    } else if constexpr (R == 2) {
        y[0] = cadd(v[0], v[1]);
        y[1] = csub(v[0], v[1]);
    } else if constexpr (R == 4) {
        const T a = cadd(v[0], v[2]), b = csub(v[0], v[2]);
        const T c = cadd(v[1], v[3]), d = csub(v[1], v[3]);
        y[0] = cadd(a, c);
        y[2] = csub(a, c);
        y[1] = T{b.x + d.y, b.y - d.x};  // b - i d
        y[3] = T{b.x - d.y, b.y + d.x};  // b + i d
    } else if constexpr (R == 3) {
        const E h = E(0.86602540378443864676);  // sqrt(3)/2
        const T t = cadd(v[1], v[2]), u = csub(v[1], v[2]);
        y[0] = cadd(v[0], t);
        const T m = T{v[0].x - E(0.5) * t.x, v[0].y - E(0.5) * t.y};
        y[1] = T{m.x + h * u.y, m.y - h * u.x};  // m - i h u
        y[2] = T{m.x - h * u.y, m.y + h * u.x};  // m + i h u
    } else {  // R == 5
        const int f = L / 5;
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            T acc = v[0];
#pragma unroll
            for (int r = 1; r < 5; ++r) acc = cadd(acc, cmul(v[r], tw[((q * r) % 5) * f]));
            y[q] = acc;
        }
    }
}

// Passes Ra and Rb (N0: product of the radices before) of the items w, w + TL,
// .. of a line: ld(i) its element i, st(i, v, n) the result, the thread's n-th.
// pre(i, n) announces a result before the butterflies (what st adds to it is
// loaded meanwhile).  sync stands between the last load and the first store.
constexpr int kRegSlots = 32;
template <int L, int N0, int Ra, int Rb, class T, class LD, class PR, class ST, class SY>
__device__ __forceinline__ void two_passes(const T* __restrict__ tw, int w, LD&& ld, PR&& pre, ST&& st, SY&& sync)
{
    constexpr int E = Ra * Rb, S = L / E, TL = (L + 15) / 16, IT = (S + TL - 1) / TL;
    static_assert(IT * E <= kRegSlots, "results of a thread");
    T v[IT][E];
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int q = w + it * TL;
        if (S % TL == 0 || q < S) {
#pragma unroll
            for (int e = 0; e < E; ++e) v[it][e] = ld(q + e * S);
        } else {
            // a value all the same, or that of the group of lines before would be kept
            // in its registers (L = 225: 732 bytes spilled, now 60)
#pragma unroll
            for (int e = 0; e < E; ++e) v[it][e] = T{0.f, 0.f};
        }
    }
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int q = w + it * TL, base = (q / N0) * (N0 * E) + q % N0;
        if (S % TL == 0 || q < S)
#pragma unroll
            for (int e = 0; e < E; ++e) pre(base + N0 * e, it * E + e);
    }
    sync();
#pragma unroll
    for (int it = 0; it < IT; ++it) {
        const int q = w + it * TL;
        if (S % TL != 0 && q >= S) continue;
        const int k = q % N0, A = q / N0;
        T y[Rb][Ra];
#pragma unroll
        for (int rb = 0; rb < Rb; ++rb) {
            T x[Ra];
            x[0] = v[it][rb];
#pragma unroll
            for (int r = 1; r < Ra; ++r) {
                x[r] = v[it][r * Rb + rb];
                if (N0 > 1) x[r] = cmul(x[r], tw[r * k * (L / (N0 * Ra))]);
            }
            dft<Ra>(x, y[rb], tw, L);
        }
        const int base = A * (N0 * E) + k;
#pragma unroll
        for (int r = 0; r < Ra; ++r) {
            T x[Rb], z[Rb];
            x[0] = y[0][r];
#pragma unroll
            for (int rb = 1; rb < Rb; ++rb) x[rb] = cmul(y[rb][r], tw[rb * (k + r * N0) * (L / (N0 * E))]);
            dft<Rb>(x, z, tw, L);
#pragma unroll
            for (int rb = 0; rb < Rb; ++rb) st(base + N0 * (r + rb * Ra), z[rb], it * E + r + rb * Ra);
        }
    }
}

// Lines per block: 128 threads or a little more, rows of 32 bytes or wider.
template <int L>
constexpr int kRegLines = L <= 32 ? 64 : L <= 64 ? 32 : L <= 192 ? 16 : L <= 512 ? 8 : 4;
template <int L>
constexpr int kRegThreads = kRegLines<L> * ((L + 15) / 16);

// Lines through shared memory: L elements of B lines at pitch P (element-major).
template <int L, class T, class LD, class PR, class ST>
__device__ __forceinline__ void reg_fft(const T* tw, T* sm, int P, int w, int l, LD&& ld, PR&& pre, ST&& st)
{
    constexpr RegPlan Pl = reg_plan(L);
    auto rd = [&](int i) { return sm[i * P + l]; };
    auto wr = [&](int i, T v, int) { sm[i * P + l] = v; };
    auto none = [](int, int) {};
    auto sync = [] { __syncthreads(); };
    constexpr int N1 = Pl.ra[0] * Pl.rb[0], N2 = N1 * Pl.ra[1] * Pl.rb[1];
    two_passes<L, 1, Pl.ra[0], Pl.rb[0]>(tw, w, ld, none, wr, sync);  // sync: ld may read sm
    __syncthreads();
    if constexpr (Pl.n == 2) {
        two_passes<L, N1, Pl.ra[1], Pl.rb[1]>(tw, w, rd, pre, st, sync);  // sync: st may write sm
    } else {
        two_passes<L, N1, Pl.ra[1], Pl.rb[1]>(tw, w, rd, none, wr, sync);
        __syncthreads();
        two_passes<L, N2, Pl.ra[2], Pl.rb[2]>(tw, w, rd, pre, st, sync);
    }
}

// What the last pass of a strided axis leaves: the transform in place, or its
// power spectrum.
struct PowerOut {
    double* acc;   // += p (or NULL)
    double* out;   // = p, or with acc = scale * (acc + p) (or NULL)
    double scale;
    float inv;     // 1 / V
};

// Input of the rows: complex numbers in place, real numbers, or the white e/eps
// normals of the modified equilibrium's noise.
enum RowInput { kInComplex, kInReal, kInWhite };
struct WhiteIn {
    PhiloxKeys key;
    uint32_t step, replica;
};

// The kernels leave room for 512 threads per SM (128 registers): the fastest of 256
// to 1024 at 96^3 to 256^3.

// n_lines consecutive rows.
template <int L>
__global__ void __launch_bounds__(kRegThreads<L>, 512 / kRegThreads<L>)
    k_fft_rows(float2* data, const float* real, int n_lines, const RowInput in, const __grid_constant__ WhiteIn white)
{
    constexpr int B = kRegLines<L>, T = kRegThreads<L>, P = B + 1;
    extern __shared__ __align__(16) unsigned char smraw[];
    float2* tw = reinterpret_cast<float2*>(smraw);
    float2* sm = tw + L;
    const int tid = threadIdx.x, l = tid % B, w = tid / B;
    fill_twiddles(tw, L, (float2*)nullptr);
    pdl_wait();
    __syncthreads();
    const int tasks = (n_lines + B - 1) / B;
    for (int task = blockIdx.x; task < tasks; task += gridDim.x) {
        const int r0 = task * B, nl = min(B, n_lines - r0), tot = nl * L;
        float2* p = data + (long)r0 * L;
        auto fetch = [&](auto value) {
#pragma unroll 4
            for (int e = tid; e < tot; e += T) {
                const int row = e / L, j = e - row * L;
                sm[j * P + row] = value(e);
            }
        };
        if (in == kInReal)
            fetch([&](int e) { return make_float2(real[(long)r0 * L + e], 0.f); });
        else if (in == kInWhite)
            fetch([&](int e) {
                return swift_white<float2>(white.key, (uint32_t)(r0 * L + e), white.step, white.replica);
            });
        else
            fetch([&](int e) { return p[e]; });
        __syncthreads();
        reg_fft<L>(tw, sm, P, w, l, [&](int i) { return sm[i * P + l]; }, [](int, int) {},
                   [&](int i, float2 v, int) { sm[i * P + l] = v; });
        __syncthreads();
#pragma unroll 4
        for (int e = tid; e < tot; e += T) {
            const int row = e / L, j = e - row * L;
            p[e] = sm[j * P + row];
        }
        __syncthreads();
    }
}

// Line (i0, i1) starts at i0 + i1 s_out, elements es apart, i0 < n_in, i1 < n_out.
template <int L, bool POWER>
__global__ void __launch_bounds__(kRegThreads<L>, 512 / kRegThreads<L>)
    k_fft_strided(float2* data, int es, int s_out, int n_in, int n_out, const PowerOut pw)
{
    constexpr int B = kRegLines<L>;
    extern __shared__ __align__(16) unsigned char smraw[];
    float2* tw = reinterpret_cast<float2*>(smraw);
    float2* sm = tw + L;
    const int l = threadIdx.x % B, w = threadIdx.x / B;
    fill_twiddles(tw, L, (float2*)nullptr);
    pdl_wait();
    __syncthreads();
    // element offsets fit 32 bits: the field has V < 2^31 sites
    const int groups = (n_in + B - 1) / B, tasks = n_out * groups;
    for (int task = blockIdx.x; task < tasks; task += gridDim.x) {
        const int i1 = task / groups, i0 = (task - i1 * groups) * B + l;
        const bool in = i0 < n_in;
        const int s0 = (in ? i0 : 0) + i1 * s_out;
        auto ld = [&](int i) { return data[s0 + i * es]; };
        if constexpr (POWER) {
            // the accumulator's values are loaded ahead: one load after another store
            // to it would wait for memory each (128^3: 28 us)
            double acc[kRegSlots] = {};
            reg_fft<L>(tw, sm, B, w, l, ld, [&](int i, int n) { acc[n] = pw.acc ? pw.acc[s0 + i * es] : 0.0; },
                       [&](int i, float2 v, int n) {
                           if (!in) return;
                           const int s = s0 + i * es;
                           double p = s == 0 ? 0.0 : (double)(norm2(v) * pw.inv);
                           if (pw.acc) {
                               p += acc[n];
                               pw.acc[s] = p;
                               p *= pw.scale;
                           }
                           if (pw.out) pw.out[s] = p;
                       });
        } else {
            reg_fft<L>(tw, sm, B, w, l, ld, [](int, int) {}, [&](int i, float2 v, int) {
                if (in) data[s0 + i * es] = v;
            });
        }
        __syncthreads();
    }
}

// Coloured noise of the modified equilibrium (flb_swift.cu has the method).
// The y transform of the columns nx and X - nx, the colouring of every
// (ny, nx), (-ny, -nx) pair between them, and the y transform of the result, in
// one pass over the field: H columns and their mirror images per block.  With
// the white noise drawn into the x transform's rows a step of 1024 x 400 makes
// three passes instead of six: 82 -> 35 us with the register transforms.
template <int L>
__global__ void __launch_bounds__(kRegThreads<L>, 512 / kRegThreads<L>)
    k_swift_columns(const float2* in, float2* __restrict__ out, const float* chol, int X)
{
    constexpr int B = kRegLines<L>, H = B / 2;
    extern __shared__ __align__(16) unsigned char smraw[];
    float2* tw = reinterpret_cast<float2*>(smraw);
    float2* sm = tw + L;
    const int l = threadIdx.x % B, w = threadIdx.x / B;
    fill_twiddles(tw, L, (float2*)nullptr);
    pdl_wait();
    __syncthreads();
    const int n0 = blockIdx.x * H + (l < H ? l : l - H);
    const bool valid = n0 <= X / 2;
    const int n = valid ? n0 : 0, nx = l < H ? n : (n == 0 ? 0 : X - n);  // this line's column
    const int partner = l < H ? l + H : l - H;
    reg_fft<L>(tw, sm, B, w, l, [&](int i) { return in[nx + X * i]; }, [](int, int) {},
               [&](int i, float2 v, int) { sm[i * B + l] = v; });
    __syncthreads();
    reg_fft<L>(
        tw, sm, B, w, l,
        [&](int i) {
            const float2 zk = sm[i * B + l], zm = sm[(i == 0 ? 0 : L - i) * B + partner];
            // E = (Z(k) + conj Z(-k)) / 2, P = (Z(k) - conj Z(-k)) / (2i)
            const float er = 0.5f * (zk.x + zm.x), ei = 0.5f * (zk.y - zm.y);
            const float pr = 0.5f * (zk.y + zm.y), pi = -0.5f * (zk.x - zm.x);
            const float* c = chol + 3 * (nx + X * i);
            const float c11 = c[0], c21 = c[1], c22 = c[2];
            // conjugate of E' + i P' = (Er - Pi) + i (Ei + Pr)
            return make_float2(c11 * er - (c21 * ei + c22 * pi), -(c11 * ei + (c21 * er + c22 * pr)));
        },
        [](int, int) {},
        [&](int i, float2 v, int) {
            if (valid) out[nx + X * i] = v;
        });
}


// The kernels of a length.  The lengths are spread over kRegParts translation
// units (flb_fft_reg.cu, FLB_REG_PART): the n-th is entry n / kRegParts of part
// n % kRegParts.
struct RegKernels {
    int L, lines, threads;
    void (*rows)(float2*, const float*, int, RowInput, WhiteIn);
    void (*strided)(float2*, int, int, int, int, PowerOut);
    void (*power)(float2*, int, int, int, int, PowerOut);
    void (*columns)(const float2*, float2*, const float*, int);
};
#define FLB_REG_PARTS(F) F(0) F(1) F(2) F(3) F(4) F(5) F(6) F(7) F(8) F(9) F(10) F(11)
constexpr int kRegParts = 12;
#define FLB_REG_DECLARE(K) const RegKernels* reg_part_##K();
FLB_REG_PARTS(FLB_REG_DECLARE)
#undef FLB_REG_DECLARE

}  // namespace flb
