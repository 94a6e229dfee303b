// flb_internal.h -- host-side interface between the C ABI (flb_api.cu) and the
// precision-specific kernel instantiations (flb_fp64.cu, flb_fp32.cu,
// flb_bf16.cu) and the precision-independent kernels (flb_fft.cu, flb_sums.cu).
#pragma once

#include <cstdint>
#include <string>

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include "../../include/flb.h"

namespace flb {

// Tracing: every C-ABI call that launches GPU work opens an NVTX range named
// after the call, so a profiler attributes each kernel to the call that issued
// it (e.g. ncu --nvtx --nvtx-include "flb_step/").  NVTX is header-only and
// costs a few nanoseconds per range when no profiler is attached.
struct NvtxRange {
    explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
    ~NvtxRange() { nvtxRangePop(); }
    NvtxRange(const NvtxRange&) = delete;
    NvtxRange& operator=(const NvtxRange&) = delete;
};
#define FLB_TRACE() ::flb::NvtxRange flb_trace_range_(__func__)

// flb_z_chunk's answer for contexts that set no z_chunk of their own (no step has one).
constexpr int kZChunkDefault = 16;

// Model parameters in double; each instantiation converts to its compute type.
struct HostModel {
    int Q, D, X, Y, Z;
    long V;
    double rho0;
    double om_s, om_b, om_g, kT;
    int nonideal;
    double A, B, rho_c, kappa;
    int total;  // psi is the total bulk free energy: F gains cs^2 grad rho
    int model;  // 0 force-based, 1 modified equilibrium (D2Q9)
    const void* swift_xi = nullptr;  // modified equilibrium: FFT of the coloured e/eps noise (double2 or float2)
    uint64_t seed;
    uint32_t replica;
    int noise_local;
    int zchunk = 0;  // flb_options.z_chunk
    void* mu = nullptr;  // force-model step in passes: the context's chemical potential field
};

// Lattices whose mode sums one launch forms; lattice r owns the blocks and rows
// lat[r].first .. lat[r + 1].first of 2 Q doubles.
struct ModeLattice {
    const void* src;
    int X, Y, Z, first;
};
struct ModeSums {
    int n;
    double* rows;
    ModeLattice lat[FLB_BATCH_MAX + 1];
};
constexpr int kModeRowsMin = 512;  // rows that a partial-sum buffer holds at least
// Append a lattice; returns its blocks.  Sixteen groups of 32 sites per warp and
// at most six blocks per SM: long enough that the block's own sums do not count.
// Lattices that give an SM fewer than eight groups go in small blocks, two per SM
// (mode_warps): a warp per SM left an FP64 one waiting for its own chain of
// operations, us of the whole call at 32^3 and 31 x 29 x 37, one warp 74 and 81, two
// 47 and 44, eight 44 and 57 (FP32 42, 34, 33).
inline int mode_warps(int X, int Y, int Z) { return (long)((X + 31) / 32) * Y * Z < 8 * 152 ? 2 : 8; }
inline int mode_blocks(ModeSums& a, const void* src, int X, int Y, int Z, int warps)
{
    const long groups = (long)((X + 31) / 32) * Y * Z, most = 6 * 152;
    long nb = (groups + 16 * warps - 1) / (16 * warps);
    const long least = warps == 8 ? 152 : 2 * 152, one = (groups + warps - 1) / warps;  // <= kModeRowsMin rows
    if (nb < least) nb = one < least ? one : least;
    if (nb > most) nb = most;
    ModeLattice& q = a.lat[a.n];
    q.src = src;
    q.X = X;
    q.Y = Y;
    q.Z = Z;
    a.lat[++a.n].first = q.first + (int)nb;
    return (int)nb;
}
// Column sums of each lattice's rows: out[r * ncol + c] (flb_sums.cu).
cudaError_t sum_lattices(const ModeSums& a, int ncol, double* out, cudaStream_t s);

// Kernels whose code depends on the compute/storage type.  Pointers are device
// pointers; `pop` buffers hold Q*V elements of the storage type, `field`
// buffers V (or 3V) elements of the compute type.
struct PrecOps {
    int elem_size;    // bytes per stored population
    int real_size;    // bytes per compute-type scalar (density/force fields)
    cudaError_t (*density)(const HostModel&, const void* pop, void* drho, cudaStream_t);
    cudaError_t (*step)(const HostModel&, uint64_t step, const void* src, void* dst, const void* drho,
                        cudaStream_t);
    cudaError_t (*init)(const HostModel&, void* dst, const double* rho, const double* u, int thermal,
                        cudaStream_t);
    cudaError_t (*get_pop)(const HostModel&, const void* src, double* out, cudaStream_t);
    cudaError_t (*set_pop)(const HostModel&, const double* in, void* dst, cudaStream_t);
    // which: 0 rho, 1 u (needs F or NULL for the ideal gas), 2 modes
    cudaError_t (*moments)(const HostModel&, const void* src, double* out, int which, const void* F,
                           cudaStream_t);
    cudaError_t (*mu_force)(const HostModel&, const void* drho, void* mu, void* F, cudaStream_t);
    // per-block sums of m_a and m_a^2, warps per block as mode_blocks returns
    cudaError_t (*mode_sums)(const ModeSums&, int Q, int warps, cudaStream_t);
    // cons_rows(V) rows of partial sums of mass deviation and momentum
    cudaError_t (*cons_partials)(const HostModel&, const void* src, double* partials, cudaStream_t);
    // mode a of the pre-collision state: double2 of an FP64 state, float (real)
    // of the others
    cudaError_t (*mode_field)(const HostModel&, const void* src, int mode, void* out, cudaStream_t);
    int (*partial_rows_max)(const HostModel&);
    int (*step_needs_density)(const HostModel&);
    int (*step_in_passes)(const HostModel&);  // the step uses the density and mu fields itself
    // pre-collision deviations in the storage type, [i][s], to / from a device buffer
    cudaError_t (*pull_state)(const HostModel&, const void* src, void* out, cudaStream_t);
    cudaError_t (*push_state)(const HostModel&, const void* in, void* dst, cudaStream_t);
    // pre-collision populations f_i at n sites (device list), out[i*n + k]
    cudaError_t (*get_sites)(const HostModel&, const void* src, const long long* sites, int n, double* out,
                             cudaStream_t);
    // float4 rows of mass deviation and momentum that step_rows writes (the sums
    // over warps of the state it steps from); 0: the step does not provide them
    int (*step_row_count)(const HostModel&);
    cudaError_t (*step_rows)(const HostModel&, uint64_t step, const void* src, void* dst, const void* drho,
                             float4* rows, cudaStream_t);
    // the step from src, whose pre-collision deviations go to state as well
    cudaError_t (*step_state)(const HostModel&, uint64_t step, const void* src, void* dst, const void* drho,
                              void* state, cudaStream_t);
};

const PrecOps& ops_fp64();
const PrecOps& ops_fp32();
const PrecOps& ops_bf16();

// Launch a kernel that begins with pdl_wait() on a stream: it may start while
// the kernel before it drains (programmatic dependent launch), which hides the
// launch latency between the kernels of a step.
template <class... P, class... A>
cudaError_t launch_chain_smem(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A... args)
{
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, kernel, P(args)...);
}
template <class... P, class... A>
cudaError_t launch_chain(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st, A... args)
{
    return launch_chain_smem(kernel, grid, block, 0, st, args...);
}

// Deterministic column sums of k arrays of nrows rows, one after another:
// out[i*ncol + c] = sum_r partials[(i*nrows + r)*ncol + c], plus add0 on the
// columns 0 (flb_sums.cu).
cudaError_t sum_columns(const double* partials, int nrows, int ncol, double* out, cudaStream_t s,
                        double add0 = 0.0, int k = 1);

// Rows of cons_partials, a block of kConsThreads each: at most the blocks of one
// site per thread, for which the buffer of partial sums has 2 Q columns.
constexpr int kConsThreads = 256, kConsBlocksMax = 152 * 3;
inline int cons_rows(long V)
{
    const long b = (V + kConsThreads - 1) / kConsThreads;
    return (int)(b < kConsBlocksMax ? b : kConsBlocksMax);
}

// Sums of k steps' warp rows (flb_sums.cu): rows holds k times nrows float4 rows
// (mass deviation and momentum); out[4 i ..] receives the sums of step i's, the
// mass with add0.  part: kSumBlocksMax k doubles x 4, ticks: k counters that are
// zero between launches.
cudaError_t sum_steps(const float4* rows, int nrows, int k, double* part, unsigned* ticks, double* out, double add0,
                      cudaStream_t s);
constexpr int kSumBlocksMax = 64;  // blocks per step
constexpr int kSumStepsMax = 16;   // steps summed by one launch

// True when an axis of length L is transformed by the in-place mixed-radix FFT
// (L a product of 2, 3 and 5, at most 4096); other lengths need `scratch`.
bool fft_length_in_place(int L);

// Record the calling thread's last error message (flb_last_error) and return code.
int set_error(int code, const std::string& msg);

// In-place forward DFT along every axis of length > 1 of a complex X*Y*Z field
// (FP64, and an FP32 form for fields whose precision needs no more).
cudaError_t fft3d(double2* data, int X, int Y, int Z, double2* scratch, cudaStream_t s);
cudaError_t fft3d(float2* data, int X, int Y, int Z, float2* scratch, cudaStream_t s);
// In-place forward DFT of n consecutive rows of length X (scratch: X n elements).
cudaError_t fft_rows(double2* data, int X, int n, double2* scratch, cudaStream_t s);

// Modified-equilibrium model (flb_swift.cu).  swift_table fills chol with
// (c11, c21, c22) per wavevector, the lower Cholesky factor of the lattice
// covariance of the e and eps noise; false (with a message) where it is not
// positive definite.  swift_noise draws the white e/eps normals of `step`,
// transforms them to Fourier space, colours them with chol (float when fp32,
// else double) and leaves in
// `out` a field whose real part times 1/V is xi_e and minus imaginary part
// times 1/V is xi_eps; `work` is scratch (both V complex numbers, float2 when
// fp32, else double2).
bool swift_table(const HostModel& m, double* chol, std::string& err);
cudaError_t swift_noise(const HostModel& m, uint64_t step, const void* chol, void* work, void* out, bool fp32,
                        cudaStream_t s);

// Interface heights of a stripe (flb_capillary.cu): drho is the density
// deviation field (real_size 4 or 8 bytes), h receives 2 X doubles.
cudaError_t interface_heights(const void* drho, int real_size, double rho0, int X, int Y,
                              const flb_interface_fit& f, double* h, cudaStream_t s);
// Height spectrum of the 2 X heights h: work and scratch hold 2 X complex
// doubles; accumulate: acc += p, else out = p (X doubles).
cudaError_t height_power(const double* h, int X, double2* work, double2* scratch, double* acc, double* out,
                         cudaStream_t s);

// Adjoint of D3Q19 steps (flb_adjoint.cu).  States and adjoints are [19][V]
// deviations in the storage type (FP64 or FP32).
// adjoint_fields: rho and mu (V values each, state after state) of n <= kAdjBatch
// consecutive states; nothing for the ideal gas.
// adjoint_step: the adjoint of one step at state gn with its rho and mu; work
// holds kAdjFields V values, rows adjoint_rows(m, prec) * 3 doubles of block sums of
// the parameter gradients.  Within a segment the density part of the adjoint
// (one scalar per site, added to every population) may be passed on instead of
// added: rb_out (V scalars or NULL) receives it and the next step takes it as
// rb_next (NULL: lam_next is complete); adjoint_add_rb adds the last one.
// adjoint_grads: the block sums of n steps (rows step after step, part: n * 6
// doubles) added to grad (6 doubles, device), the last step first.
constexpr int kAdjBatch = 8, kAdjFields = 5;
cudaError_t adjoint_fields(const HostModel& m, int prec, const void* states, int n, void* rho, void* mu,
                           cudaStream_t st);
cudaError_t adjoint_step(const HostModel& m, int prec, uint64_t step, const void* gn, const void* rho, const void* mu,
                         const void* lam_next, const void* rb_next, void* lam, void* rb_out, void* work, double* rows,
                         cudaStream_t st);
cudaError_t adjoint_grads(const HostModel& m, int prec, const double* rows, int n, double* part, double* grad, cudaStream_t st);
cudaError_t adjoint_add_rb(const HostModel& m, int prec, void* lam, const void* rb, cudaStream_t st);
int adjoint_rows(const HostModel& m, int prec);

// p = |data|^2 / V with p(0) = 0: acc += p and out = scale * acc (out may be
// NULL), or without acc out = p.
cudaError_t power_spectrum(const double2* data, long V, double* acc, double* out, cudaStream_t s, double scale = 1.0);
// The same of an FP32 field of real numbers: transform (data: work, V complex
// numbers, scratch as many) and power spectrum.
cudaError_t spectrum(float2* data, const float* real, int X, int Y, int Z, float2* scratch, double* acc, double* out,
                     double scale, cudaStream_t s);

}  // namespace flb
