// Internal declarations shared by the CUDA translation units of libpic.
#pragma once

#include <cstdint>
#include <vector>
#include <cuda_runtime.h>

#include "../../include/pic.h"
#include "per_device.h"

namespace pic {

// Division by a run-time constant d without an integer divide (Granlund-Montgomery):
// n / d = (t + ((n - t) >> 1)) >> (s - 1), t = umulhi(m, n), for all 32-bit n.
struct FastDiv {
    uint32_t d, m;
    int s;   // -1: d == 1
};

inline FastDiv make_fastdiv(uint32_t d) {
    FastDiv f{d, 0u, -1};
    if (d <= 1) return f;
    int l = 0;
    while ((1ull << l) < d) ++l;
    f.m = (uint32_t)((((1ull << 32) * ((1ull << l) - d)) / d) + 1);
    f.s = l;
    return f;
}

// Grid constants passed by value to every kernel.
struct GridP {
    int ndim;
    int nz, nx, ny;     // cells
    int nzg;            // nz + 2: z extent of the guarded particle cell index
    long long ncell;    // nz * nx * ny
    float dz, dx, dy, dt;
    int shape;          // 1 or 2
    FastDiv div_nzg, div_nx;   // filled by the particle launchers
};

// Axial stencil (Appendix C).  M = 1, C[0] = 1 is the Yee difference.  C: the E-side d+
// (Faraday's law, [k]_E1); Cm: the B-side d- (Ampere's and Gauss's laws, [k]_B1), equal to C
// unless the handle was created with separate B-side coefficients.
struct StencilP {
    int M;
    float C[PIC_MAX_M];
    float Cm[PIC_MAX_M];
    float2 C2[PIC_MAX_M], Cm2[PIC_MAX_M];   // each coefficient twice: operands of packed arithmetic
};

// Field-advance launch parameters.
struct FieldP {
    GridP g;
    StencilP st;
    const float* Ein;
    const float* Bin;
    const float* J1;     // current components (J1 may be the corrected copy)
    const float* J2;
    const float* J3;
    float* Eout;
    float* Bout;
    int shift;           // 1: write the result one cell towards -z, zero the front column
    int vec4;            // nz % 4 == 0 and every array 16-byte aligned (set by launch_field_advance)
};

// One species' particle arrays and per-species constants.
struct SpeciesP {
    int32_t* cell;
    float* off;          // [ndim][cap]
    float* u;            // [3][cap]
    int32_t* id;         // may be null
    int32_t* count;      // device live-slot extent
    long long cap;
    float eps;           // q dt / (2 m)   (Boris)
    float kz[2], kx[2], ky[2];   // dt/dz, dt/dx, dt/dy as float-float (hi, lo)
    float qv;            // q w / V        (charge density of one macro-particle per unit shape)
    double qv64;
    double wm;           // w m            (kinetic energy)
    int32_t* prev_cell;  // scratch for the unfused path
    float* prev_off;
};

// The species of a step whose deferred chunks one launch finishes (3D fused mode).
struct LeftoverP {
    int n;
    SpeciesP sp[PIC_MAX_SPECIES];
    int* defer[PIC_MAX_SPECIES];     // chunks for the general path (count in [0], chunks from [2])
    int* defer2[PIC_MAX_SPECIES];    // chunks beyond it
};

// One instance of a batched run: its grid, its (single) species, its two field buffers.
struct PartInst {
    GridP g;
    SpeciesP sp;
    const float* E[2];   // fields read at even / odd steps
    const float* B[2];
    float* J;
};

// Current correction of one instance (customised stencil).
struct CorrInst {
    GridP g;
    float h[2 * PIC_MAX_HLEN + 1];
    int hlen;
    float* J1;
};

// Current filter of one batched instance (all three components of J).
struct FiltInst {
    GridP g;
    float* J;
    int vec4;            // nz % 4 == 0 and J 16-byte aligned
};

// Device status word bits.
enum : int { STATUS_CAPACITY = 1, STATUS_TIMEOUT = 2 };
constexpr int WAIT_POLLS = 1 << 20;      // looks of a bounded device-side wait, of up to a microsecond each

#ifdef __CUDACC__
// ---- chained launches ----
// The kernels of a step follow one another on one stream.  Launched chained, a kernel is brought onto the
// device while the one before it still runs and waits there (chain_enter, first thing in every kernel
// that is launched so) until that one has completed and its writes are visible: 1 to 2 us less between
// two kernels, which is what steps of small grids consist of (256 x 128 cells, one particle: a step 24.2
// -> 11.8 us; the separate phases at 1024 x 256: 106 -> 96 us; the gradient of 500 steps there: 42.8 ->
// 36.8 ms).  Field and current kernels over more than CHAIN_CELLS cells, and 3D field kernels, are launched
// plainly: there the blocks of the early kernel settle where the other ends first instead of evenly (8192 x
// 2048, M = 16, four steps: 1166 us chained, 1148 us not; 2048 x 512 still gains, 2860 -> 2790 us for eight
// steps).
constexpr long long CHAIN_CELLS = 1 << 20;
__device__ __forceinline__ void chain_enter() {
    asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
    asm volatile("griddepcontrol.wait;\n" ::: "memory");
}
// A chained kernel starts with the split between shared memory and L1 that the one before it left, unless it asks
// for another, and where the split changes the device runs empty first.  So the kernels of a 2D step
// ask for one split, 164 KB of shared memory and 92 KB of L1: what the particle kernel's four CTAs need, with
// the L1 of its path for unsorted particles.  Left to the driver (field kernels 228 KB): 2048 x 512 with
// 1000 scattered particles 45 us a step, 34 now; 511 x 255 with 524288 sorted ones 37 and 32.  Only a kernel
// whose grid fits the device at once under that split asks (in_step): it loses nothing.
constexpr int STEP_CARVEOUT = 71;                    // percent of 228 KB, rounded down to the next split
constexpr size_t STEP_SHARED = 164 * 1024, CTA_RESERVED = 2 * 1024;
inline int in_step(dim3 grid, size_t smem) {
    const unsigned long long ctas = (unsigned long long)grid.x * grid.y * grid.z;
    return smem > 0 && ctas <= 152ull * (STEP_SHARED / (smem + CTA_RESERVED)) ? STEP_CARVEOUT : -1;
}
// Dynamic shared memory that spreads a grid of less than a wave evenly over the SMs: the CTAs of a chained kernel
// settle on the SMs that the kernel before it leaves first, as many as fit there (2048 x 512, 20000 scattered
// particles, quadratic: 61 us a step, 33 with one CTA per SM).
inline size_t spread_shared(unsigned ctas, size_t smem) {
    const size_t share = STEP_SHARED / ((ctas + 151) / 152) - CTA_RESERVED;
    return share > smem ? share : smem;
}
// carveout: percent of the shared memory that an SM can give; -1 asks for nothing
template <typename... P, typename... A>
cudaError_t launch_split(bool chain, int carveout, void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                         A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[2];
    if (chain) {
        attr[cfg.numAttrs].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[cfg.numAttrs++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (carveout >= 0) {
        attr[cfg.numAttrs].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
        attr[cfg.numAttrs++].val.sharedMemCarveout = (unsigned)carveout;
    }
    cfg.attrs = attr;
    return cudaLaunchKernelEx(&cfg, k, static_cast<A&&>(args)...);
}
template <typename... P, typename... A>
cudaError_t launch_chained_if(bool chain, void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
    return launch_split(chain, chain ? in_step(grid, smem) : -1, k, grid, block, smem, s, static_cast<A&&>(args)...);
}
template <typename... P, typename... A>
cudaError_t launch_chained(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
    return launch_chained_if(true, k, grid, block, smem, s, static_cast<A&&>(args)...);
}
inline int current_device() {
    int dev = -1;
    return cudaGetDevice(&dev) == cudaSuccess ? dev : -1;
}
// Allows k `bytes` of dynamic shared memory on the current device; granted: the launch's own static.
template <typename K>
cudaError_t allow_shared(PerDevice& granted, K k, size_t bytes) {
    return (cudaError_t)granted.grant(current_device(), (int)bytes, [&] {
        return (int)cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    });
}
inline bool few_cells(const GridP& g) { return g.ncell <= CHAIN_CELLS; }
#endif

// ---- launchers (return cudaGetLastError of the launch) ----
cudaError_t launch_field_advance(const FieldP& p, cudaStream_t s, int variant = 0);
// f = 0 (n floats); d0 = s0 and d1 = s1 (n floats each)
cudaError_t launch_zero(float* f, long long n, cudaStream_t s);
cudaError_t launch_copy2(float* d0, const float* s0, float* d1, const float* s1, long long n, cudaStream_t s);
int copy2_launches(long long n);     // 1 kernel, or 2 copies
int field_variants(int ndim);
int field_vec4(const FieldP& p);     // 1: its arrays can be moved in 16-byte groups
int default_field_variant(const GridP& g, int M);

// batched: instance tables live in device memory
cudaError_t launch_field_advance_batch(const FieldP* inst, const int4* work, int total_tiles, int ndim, int maxm,
                                       int parity, cudaStream_t s);
void batch_tiles(std::vector<int4>& work, int inst, int ndim, int nz, int nx, int ny);
// Batched 2D field advance with the x-marching segments: work[w] = (instance, z0 | cells << 16, first
// row, last row + 1).
constexpr int ROWS_BATCH_NT = 64;
std::vector<int4> rows_batch_work(int maxm, const std::vector<int>& nz, const std::vector<int>& nx);
// The same tile list as launch_field_advance_batch with register-blocked tiles.
cudaError_t launch_field_advance_rb_batch(const FieldP* inst, const int4* work, int total_tiles, int ndim, int maxm,
                                          int parity, cudaStream_t s);
cudaError_t launch_field_advance_rows_batch(const FieldP* inst, const int4* work, int nwork, int maxm, int parity,
                                            cudaStream_t s);
cudaError_t launch_correct_j1_batch(const CorrInst* inst, int ninst, int max_rows, int max_nz, cudaStream_t s);
cudaError_t launch_push_batch(const PartInst* inst, int ninst, int ndim, int shape, long long max_extent, int parity,
                              cudaStream_t s);
cudaError_t launch_zero_j_batch(const PartInst* inst, int ninst, long long max_ncell, cudaStream_t s);
// defer (3D fused mode): library scratch of two lists of defer_len(cap) ints each, their first two
// ints zero on first use: the chunks whose shared-memory boxes do not fit.  launch_push_leftover,
// after launch_push of every species, processes the lists of all of them and clears them.
constexpr long long defer_len(long long cap) { return 2 + (cap + 255) / 256; }
cudaError_t launch_push(const GridP& g, const SpeciesP& sp, const float* E, const float* B,
                        float* J, int shift, int mode, long long extent, int* defer, int* status, int polls, cudaStream_t s);
cudaError_t launch_push_leftover(const GridP& g, const SpeciesP* sp, int* const* defer, const long long* extent, int n,
                                 const float* E, const float* B, float* J, int shift, cudaStream_t s);
cudaError_t launch_deposit_unfused(const GridP& g, const SpeciesP& sp, float* J, long long extent,
                                   cudaStream_t s);
// Appends the new column's cold plasma (3D: at the count rounded up to 256, patch-ordered);
// *extent, the host's upper bound of the count, is advanced accordingly.
cudaError_t launch_inject(const GridP& g, const SpeciesP& sp, const int ppc[3], long long next_id,
                          int* status, long long* extent, cudaStream_t s);
long long sort_bins(const GridP& g);
cudaError_t launch_sort(const GridP& g, const SpeciesP& sp, long long extent, int32_t* hist,
                        int32_t* blocksums, int32_t* cell_alt, float* off_alt, float* u_alt,
                        int32_t* id_alt, cudaStream_t s);
cudaError_t launch_rho(const GridP& g, const SpeciesP& sp, int shift, double* rho, long long extent,
                       cudaStream_t s);
cudaError_t launch_gauss(const GridP& g, const StencilP& st, const float* E, const double* rho,
                         double rho_bg, double* G, cudaStream_t s);
cudaError_t launch_diag_reduce(const GridP& g, const StencilP& st, const float* E, const float* B,
                               const double* rho, double rho_bg, int margin, double* acc,
                               cudaStream_t s);
cudaError_t launch_kinetic(const GridP& g, const SpeciesP& sp, long long extent, double* acc,
                           cudaStream_t s);

// ---- current filter and Sec. 3 correction along z (current_kernels.cu) ----
cudaError_t launch_correct_j1(const GridP& g, const float* taps, int hlen, float* J1, cudaStream_t s);
// filter on J1, J2, J3 and the correction on J1 in one launch (J: the three components)
cudaError_t launch_filter_correct(const GridP& g, const float* taps, int hlen, float* J, cudaStream_t s);
bool filter_vec4_ok(const float* J, int nz);
cudaError_t launch_filter_current(const GridP& g, float* J, cudaStream_t s);
cudaError_t launch_filter_rho(const GridP& g, double* rho, cudaStream_t s);
cudaError_t launch_filter_current_batch(const FiltInst* inst, int ninst, long long max_rows3, cudaStream_t s);

// ---- adjoint (adjoint_kernels.cu) ----
struct TapsP {
    float h[2 * PIC_MAX_HLEN + 1];       // centred: h[m] at PIC_MAX_HLEN + m
};
// E^{n+1} of a step from its E, B, J: components 2 and 3 of out
cudaError_t launch_adjoint_enew(const GridP& g, const StencilP& st, const float* E, const float* B, const float* J,
                                float* out, cudaStream_t s);
// first and third stage (F: the step's E^{n+1} and E^n) and second stage of the adjoint step
cudaError_t launch_adjoint_ampere(const GridP& g, const StencilP& st, const float* F, const float* aB, float* aE,
                                  double* grad, cudaStream_t s);
cudaError_t launch_adjoint_faraday(const GridP& g, const StencilP& st, const float* E, const float* B, const float* J1,
                                   const float* aE, float* aB, const float* taps, int hlen, double* grad, cudaStream_t s);

// ---- host math (host_math.cpp) ----
int fit_coefficients(double kappa, int M, double wk, double n, double* C);
int fit_coefficients_b(double kappa, int M, double wk, double n, const double* CE, int ME, double* C);
int correction_taps(const double* C, int M, int hlen, double* h);
double cfl_dt(int ndim, double dz, double dx, double dy, const double* C, int M);
// with the E-side (CE) and B-side (CB) symbols: max of their product; -1 if the product is negative
double cfl_dt_split(int ndim, double dz, double dx, double dy, const double* CE, const double* CB, int M);
// k-space field advance (PIC_SOLVER_SPECTRAL, PIC_SOLVER_KT; kspace_kernels.cu).  Status codes:
// 0 ok, 1 error (message in err), 2 device memory.
struct KSpaceState;
bool kspace_available();
int kspace_create(const GridP& g, int solver, double dz, double dx, double dy, double dt, KSpaceState** out,
                  char* err, size_t nerr);
void kspace_destroy(KSpaceState* k);
long long kspace_modes(const KSpaceState* k);
int kspace_advance(KSpaceState* k, const float* Ein, const float* Bin, const float* J, float* Eout, float* Bout,
                   bool cont, bool keep, cudaStream_t s, char* err, size_t nerr);
// largest stable dt of the k-space solvers (kt = 0: spectral, 1: [k1]_t along z, 2: PSATD)
double kspace_cfl_dt(int ndim, int kt, double dz, double dx, double dy);

}  // namespace pic
