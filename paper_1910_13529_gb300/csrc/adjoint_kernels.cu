// Adjoint of the field advance (Eq. 1 leapfrog with the customised axial stencil of Sec. 3 /
// Appendix C) and of the Sec. 3 current correction, for gradients of a loss with respect to
// the axial coefficients C_l.
//
// Forward step (T = d+ x, S = d- x = T^T, h = dt/2):
//   B' = B - h T E;   E' = E + dt (S B' - J);   B'' = B' - h T E'
// Adjoint (l_E, l_B: adjoints of the step's outputs), with T_l, S_l the parts of T, S carried
// by coefficient l (axial taps l only):
//   g_l += -h <l_B, T_l E'>;  l_E <- l_E - h S l_B
//   g_l += dt <l_E, S_l B'>;  l_B <- l_B + dt T l_E;  l_J1 = -dt l_E1
//   g_l += -h <l_B, T_l E>;   l_E <- l_E - h S l_B
// Correction J1c = P^{-1} J1 (P symmetric, dP/dC_l = the box filter of half-width l-1):
//   g_l += -<P^{-1} l_J1, P_l J1c> = dt <P^{-1} l_E1, P_l J1c>.
//
// Three launches per step (four when E' has to be rebuilt from E, B, J): each of the three stages reads
// its rows once and does its field update and its gradient terms together; B' exists only in shared
// memory.  A CTA owns ADJ_SEG cells of one z row, four per thread; rows that are differentiated along z
// are staged with their halo, everything else is read at the cell.
//
// The gradient sums of FP32 fields are wide sums (wide_math.h: exact differences and products, sums kept to
// about 2^-72), which become FP64 at the warp totals.  FP64 arithmetic per cell was what the step waited for: this
// chip does 64 FP32 operations for one in FP64.  1024 x 256, M = 4: pic_adjoint_step 200 us with FP64 sums, 58 with
// these; the gradient of 500 steps 128 and 45 ms.  (Sums in pairs, 48 bits, took 42 us and 37 ms: too few bits.)
// A term costs 40 FP32 operations; half of the rest is launches and their latency.  Each warp scales its
// cells and its windows by powers of two to about 1, so that fields may be as small or large as FP32 holds; where
// the largest product of a warp is still below 1e-18 of what its largest cells could give, and for values that
// are not finite, the warp adds in FP64.
#include <cuda_runtime.h>

#include <type_traits>

#include "pic_internal.h"
#include "wide_math.h"

namespace pic {

namespace {

constexpr int ADJ_NT = 128, ADJ_SEG = 4 * ADJ_NT;
constexpr int HL = PIC_MAX_HLEN;

__device__ __forceinline__ int wrapm(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

constexpr int ADJ_W = ADJ_NT / 32;

// grad[l] += scale * the sum of part[l] over the warps, l < M (ends what the warps wrote to part)
template <int MP>
__device__ __forceinline__ void flush_grad(const double (&part)[MP][ADJ_W], int M, double scale, double* grad) {
    __syncthreads();
    if (threadIdx.x < M) {
        double v = 0.0;
        for (int q = 0; q < ADJ_W; ++q) v += part[threadIdx.x][q];
        if (v != 0.0) atomicAdd(grad + threadIdx.x, scale * v);
    }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// The largest |a| of a warp: its bits, and the power of two that brings it to about 1.
struct WarpScale {
    unsigned bits = 0u;
    template <int N>
    __device__ __forceinline__ void look(const float (&a)[N]) {
#pragma unroll
        for (int k = 0; k < N; ++k) bits = max(bits, __float_as_uint(fabsf(a[k])));
    }
    __device__ __forceinline__ void agree() { bits = __reduce_max_sync(0xffffffffu, bits); }
    __device__ __forceinline__ bool finite() const { return bits < 0x7f800000u; }
    __device__ __forceinline__ float factor() const {
        return __uint_as_float((unsigned)min(max(254 - (int)(bits >> 23), 1), 253) << 23);
    }
};
template <int N>
__device__ __forceinline__ void scale_by(float (&a)[N], float f) {
#pragma unroll
    for (int k = 0; k < N; ++k) a[k] *= f;
}
// The sums of a warp's scaled terms stand when the largest product (top) leaves its residuals in range.
__device__ __forceinline__ bool wide_enough(float top) {
    return __reduce_max_sync(0xffffffffu, __float_as_uint(top)) >= __float_as_uint(1e-18f);
}
// Sums of acc[0 .. N) over the lanes at distances O, O / 2, .., 1: a lane hands over half of its sums at each step
// until it has one left, in the end that of acc[lane MP / 32].  MP + 4 - log2(MP) additions where summing
// each over the warp takes 5 MP (M = 16: 16 and 80).
template <int N, int O, int MP>
__device__ __forceinline__ void fold_sums(WideSum (&acc)[MP]) {
    if constexpr (O > 0) {
        if constexpr (N == 1) {
            acc[0].add_lane(acc[0], O);
        } else {
            const bool up = threadIdx.x & O;
#pragma unroll
            for (int k = 0; k < N / 2; ++k) {
                const WideSum give = up ? acc[k] : acc[k + N / 2];
                if (up) acc[k] = acc[k + N / 2];
                acc[k].add_lane(give, O);
            }
        }
        fold_sums<(N > 1 ? N / 2 : 1), O / 2>(acc);
    }
}
// part[l] = the warp's sum of acc[l], unscaled; zero: nothing was added
template <int MP>
__device__ __forceinline__ void keep_sums(WideSum (&acc)[MP], bool zero, int M, float fa, float fb,
                                          double (&part)[MP][ADJ_W]) {
    if (!zero) fold_sums<MP, 16>(acc);
    const int l = (threadIdx.x & 31) * MP / 32;
    if ((threadIdx.x & (32 / MP - 1)) == 0 && l < M) part[l][threadIdx.x >> 5] = acc[0].value() / ((double)fa * (double)fb);
}

// Cells [zlo, zlo + n) of a row into s, zero outside 0 <= z < nz, asynchronously: a stage's rows are
// all in flight together (stage_wait, then a barrier); loads that wait for one another made the staging
// take longer than the arithmetic.
__device__ __forceinline__ void stage_cells(float* s, const float* __restrict__ row, int zlo, int n, int nz) {
    for (int k = threadIdx.x; k < n; k += ADJ_NT) {
        const int z = zlo + k;
        const bool in = (unsigned)z < (unsigned)nz;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(s + k)),
                     "l"(row + (in ? z : 0)), "r"(in ? 4 : 0)
                     : "memory");
    }
}
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// the thread's four cells of a row (zero beyond the grid)
__device__ __forceinline__ void cells4(float (&v)[4], const float* row, int zi, int nz) {
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = zi + j < nz ? row[zi + j] : 0.f;
}

// w[k] = s[k], k < N (s 16-byte aligned)
template <int N>
__device__ __forceinline__ void load_window(float (&w)[N], const float* s) {
    static_assert(N % 4 == 0, "whole groups");
#pragma unroll
    for (int q = 0; q < N / 4; ++q) {
        const float4 v = *reinterpret_cast<const float4*>(s + 4 * q);
        w[4 * q] = v.x;
        w[4 * q + 1] = v.y;
        w[4 * q + 2] = v.z;
        w[4 * q + 3] = v.w;
    }
}

// axial d+ (PLUS) or d- of the window w (cell j at w[MP + j]) times dz
template <int MP, bool PLUS>
__device__ __forceinline__ float axial(const StencilP& st, const float (&w)[2 * MP + 4], int j) {
    float s = 0.f;
#pragma unroll
    for (int l = 1; l <= MP; ++l) {
        if (l > st.M) break;
        s = fmaf(st.C[l - 1], PLUS ? w[MP + j + l] - w[MP + j - l + 1] : w[MP + j + l - 1] - w[MP + j - l], s);
    }
    return s;
}

// part[l - 1] = the warp's sum of l3 D_l f2 - l2 D_l f3 over its cells, D_l tap l of d+ (PLUS) or d-
// without its 1/dz.  L2, L3: the thread's four cells; F2, F3: its windows (cell 0 at F + MP); all staged,
// zero outside the grid.
template <int MP, bool PLUS>
__device__ __forceinline__ void grad_terms(double (&part)[MP][ADJ_W], int M, const float* L2, const float* L3,
                                           const float* F2, const float* F3) {
    float l2[4], l3[4], f2[2 * MP + 4], f3[2 * MP + 4];
    load_window(l2, L2);
    load_window(l3, L3);
    load_window(f2, F2);
    load_window(f3, F3);
    WarpScale ml, mf;
    ml.look(l2);
    ml.look(l3);
    mf.look(f2);
    mf.look(f3);
    ml.agree();
    mf.agree();
    bool wide = ml.finite() && mf.finite();
    if (wide) {
        const float a = ml.factor(), b = mf.factor();
        scale_by(l2, a);
        scale_by(l3, a);
        scale_by(f2, b);
        scale_by(f3, b);
        WideSum acc[MP];
        const bool zero = ml.bits == 0u || mf.bits == 0u;
        float top = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (zero || (l2[j] == 0.f && l3[j] == 0.f)) continue;
#pragma unroll
            for (int l = 1; l <= MP; ++l) {
                if (l > M) break;
                const int hi = PLUS ? MP + j + l : MP + j + l - 1, lo = PLUS ? MP + j - l + 1 : MP + j - l;
                float d, e;
                two_sum(f3[hi], -f3[lo], d, e);
                top = fmaxf(top, fabsf(acc[l - 1].fma(-l2[j], d, e)));
                two_sum(f2[hi], -f2[lo], d, e);
                top = fmaxf(top, fabsf(acc[l - 1].fma(l3[j], d, e)));
            }
        }
        wide = zero || wide_enough(top);
        if (wide) keep_sums(acc, zero, M, a, b, part);
    }
    if (!wide) {
#pragma unroll 1
        for (int l = 1; l <= M; ++l) {
            const int hi = PLUS ? MP + l : MP + l - 1, lo = PLUS ? MP - l + 1 : MP - l;
            double v = 0.0;
            for (int j = 0; j < 4; ++j) {
                const double a2 = L2[j], a3 = L3[j];
                if (a2 == 0.0 && a3 == 0.0) continue;
                v += -a2 * ((double)F3[j + hi] - (double)F3[j + lo]) + a3 * ((double)F2[j + hi] - (double)F2[j + lo]);
            }
            v = warp_sum(v);
            if ((threadIdx.x & 31) == 0) part[l - 1][threadIdx.x >> 5] = v;
        }
    }
}

// part[l - 1] = the warp's sum of v (sum of J1 over |m| < l), J: the thread's window (cell 0 at J + MP).
template <int MP>
__device__ __forceinline__ void correction_terms(double (&part)[MP][ADJ_W], int M, const float (&v)[4], const float* J) {
    float w[4], jw[2 * MP + 4];
#pragma unroll
    for (int j = 0; j < 4; ++j) w[j] = v[j];
    load_window(jw, J);
    WarpScale mv, mj;
    mv.look(w);
    mj.look(jw);
    mv.agree();
    mj.agree();
    bool wide = mv.finite() && mj.finite();
    if (wide) {
        const float a = mv.factor(), b = mj.factor();
        scale_by(w, a);
        scale_by(jw, b);
        WideSum acc[MP];
        const bool zero = mv.bits == 0u || mj.bits == 0u;
        float top = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (zero || w[j] == 0.f) continue;
            WideSum box;                                       // of J1 over |m| < l
            box.h = jw[MP + j];
            top = fmaxf(top, fabsf(acc[0].fma(w[j], box.h, 0.f)));
#pragma unroll
            for (int l = 2; l <= MP; ++l) {
                if (l > M) break;
                box.add(jw[MP + j - (l - 1)]);
                box.add(jw[MP + j + (l - 1)]);
                top = fmaxf(top, fabsf(acc[l - 1].fma(w[j], box.h, box.m, box.l)));
            }
        }
        wide = zero || wide_enough(top);
        if (wide) keep_sums(acc, zero, M, a, b, part);
    }
    if (!wide) {
#pragma unroll 1
        for (int l = 1; l <= M; ++l) {
            double s = 0.0;
            for (int j = 0; j < 4; ++j) {
                if (v[j] == 0.f) continue;
                double box = J[MP + j];
                for (int m = 1; m < l; ++m) box += (double)J[MP + j - m] + (double)J[MP + j + m];
                s += (double)v[j] * box;
            }
            s = warp_sum(s);
            if ((threadIdx.x & 31) == 0) part[l - 1][threadIdx.x >> 5] = s;
        }
    }
}

struct RowAt {
    long long row, xm, xp, ym, yp;    // z row offsets of (x, y) and its neighbours (y: itself in 2D)
};
__device__ __forceinline__ RowAt row_at(const GridP& g, int r) {
    const int j = r % g.nx, k = r / g.nx;
    auto at = [&](int jj, int kk) { return ((long long)kk * g.nx + jj) * g.nz; };
    RowAt q;
    q.row = at(j, k);
    q.xm = at(wrapm(j - 1, g.nx), k);
    q.xp = at(wrapm(j + 1, g.nx), k);
    q.ym = g.ndim == 3 ? at(j, wrapm(k - 1, g.ny)) : q.row;
    q.yp = g.ndim == 3 ? at(j, wrapm(k + 1, g.ny)) : q.row;
    return q;
}

// First and third stage: g_l += -h <l_B, T_l F> and l_E -= h S l_B, F (components 2 and 3) E' or E.
template <int MP>
__global__ void __launch_bounds__(ADJ_NT) adjoint_ampere_kernel(GridP g, StencilP st, const float* __restrict__ F,
                                                                const float* __restrict__ aB, float* aE, double* grad) {
    chain_enter();
    constexpr int W = ADJ_SEG + 2 * MP;
    __shared__ __align__(16) float sB[2][W], sF[2][W];
    __shared__ double part[MP][ADJ_W];
    const long long N = g.ncell;
    const RowAt q = row_at(g, blockIdx.x);
    const int z0 = blockIdx.y * ADJ_SEG, nz = g.nz;
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        stage_cells(sB[c], aB + (c + 1) * N + q.row, z0 - MP, W, nz);
        stage_cells(sF[c], F + (c + 1) * N + q.row, z0 - MP, W, nz);
    }
    const int t4 = 4 * threadIdx.x, zi = z0 + t4;
    const float h = 0.5f * g.dt, hz = -h * (1.f / g.dz), hx = -h * (1.f / g.dx), hy = -h * (1.f / g.dy);
    float e1[4], e2[4], e3[4], b1[4], x1[4], x3[4], y1[4], y2[4];
    cells4(e1, aE + q.row, zi, nz);
    cells4(e2, aE + N + q.row, zi, nz);
    cells4(e3, aE + 2 * N + q.row, zi, nz);
    cells4(b1, aB + q.row, zi, nz);
    cells4(x1, aB + q.xm, zi, nz);
    cells4(x3, aB + 2 * N + q.xm, zi, nz);
    if (g.ndim == 3) {
        cells4(y1, aB + q.ym, zi, nz);
        cells4(y2, aB + N + q.ym, zi, nz);
    }
    stage_wait();
    __syncthreads();
    float b2[2 * MP + 4], b3[2 * MP + 4];
    load_window(b2, sB[0] + t4);
    load_window(b3, sB[1] + t4);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (zi + j >= nz) break;
        float* o = aE + q.row + zi + j;
        float s1 = hx * (b3[MP + j] - x3[j]), s2 = -hz * axial<MP, false>(st, b3, j);
        if (g.ndim == 3) {
            s1 -= hy * (b2[MP + j] - y2[j]);
            s2 += hy * (b1[j] - y1[j]);
        }
        o[0] = e1[j] + s1;
        o[N] = e2[j] + s2;
        o[2 * N] = e3[j] + (hz * axial<MP, false>(st, b2, j) - hx * (b1[j] - x1[j]));
    }
    grad_terms<MP, true>(part, st.M, sB[0] + t4 + MP, sB[1] + t4 + MP, sF[0] + t4, sF[1] + t4);
    flush_grad<MP>(part, st.M, -(double)h / (double)g.dz, grad);
}

// rows of B' (components 2, 3) over [z0 - MP, z0 + ADJ_SEG + MP) into sH, by way of E2, E3 staged in sE
// over one more halo; ends with a barrier
template <int MP>
__device__ __forceinline__ void stage_b_half(const GridP& g, const StencilP& st, const float* __restrict__ E,
                                             const float* __restrict__ B, const RowAt& q, int z0,
                                             float (&sE)[2][ADJ_SEG + 4 * MP], float (&sH)[2][ADJ_SEG + 2 * MP]) {
    for (int c = 0; c < 2; ++c)
        stage_cells(sE[c], E + (c + 1) * g.ncell + q.row, z0 - 2 * MP, ADJ_SEG + 4 * MP, g.nz);
    stage_wait();
    __syncthreads();
    const long long N = g.ncell;
    const float h = 0.5f * g.dt, hz = h * (1.f / g.dz), hx = h * (1.f / g.dx), hy = h * (1.f / g.dy);
    for (int s = threadIdx.x; s < (ADJ_SEG + 2 * MP) / 4; s += ADJ_NT) {
        const int zi = z0 - MP + 4 * s;
        float w2[2 * MP + 4], w3[2 * MP + 4];
        load_window(w2, sE[0] + 4 * s);
        load_window(w3, sE[1] + 4 * s);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int z = zi + j;
            float v2 = 0.f, v3 = 0.f;
            if ((unsigned)z < (unsigned)g.nz) {
                const float e1 = __ldg(E + q.row + z);
                v2 = __ldg(B + N + q.row + z) + hz * axial<MP, true>(st, w3, j);
                v3 = __ldg(B + 2 * N + q.row + z) - (hz * axial<MP, true>(st, w2, j) - hx * (__ldg(E + q.xp + z) - e1));
                if (g.ndim == 3) v2 -= hy * (__ldg(E + q.yp + z) - e1);
            }
            sH[0][4 * s + j] = v2;
            sH[1][4 * s + j] = v3;
        }
    }
    __syncthreads();
}

// Second stage: g_l += dt <l_E, S_l B'>, the correction's g_l += dt <P^{-1} l_E1, P_l J1> (hlen > 0),
// and l_B += dt T l_E.  taps: h[m] at HL + m.
template <int MP>
__global__ void __launch_bounds__(ADJ_NT) adjoint_faraday_kernel(GridP g, StencilP st, const float* __restrict__ E,
                                                                 const float* __restrict__ B, const float* __restrict__ J1,
                                                                 const float* __restrict__ aE, float* aB, TapsP taps,
                                                                 int correct, double* grad) {
    chain_enter();
    constexpr int W = ADJ_SEG + 2 * MP, W1 = ADJ_SEG + 2 * HL;
    __shared__ __align__(16) float sE[2][ADJ_SEG + 4 * MP], sH[2][W], sA[2][W], sA1[W1], sJ[W];
    __shared__ double part[MP][ADJ_W];
    const long long N = g.ncell;
    const RowAt q = row_at(g, blockIdx.x);
    const int z0 = blockIdx.y * ADJ_SEG, nz = g.nz;
#pragma unroll
    for (int c = 0; c < 2; ++c) stage_cells(sA[c], aE + (c + 1) * N + q.row, z0 - MP, W, nz);
    if (correct) {
        stage_cells(sA1, aE + q.row, z0 - HL, W1, nz);
        stage_cells(sJ, J1 + q.row, z0 - MP, W, nz);
    }
    const int t4 = 4 * threadIdx.x, zi = z0 + t4;
    const float dt = g.dt, fz = dt * (1.f / g.dz), fx = dt * (1.f / g.dx), fy = dt * (1.f / g.dy);
    float b1[4], b2[4], b3[4], a1[4], x1[4], x3[4], y1[4], y2[4];
    cells4(b1, aB + q.row, zi, nz);
    cells4(b2, aB + N + q.row, zi, nz);
    cells4(b3, aB + 2 * N + q.row, zi, nz);
    cells4(a1, aE + q.row, zi, nz);
    cells4(x1, aE + q.xp, zi, nz);
    cells4(x3, aE + 2 * N + q.xp, zi, nz);
    if (g.ndim == 3) {
        cells4(y1, aE + q.yp, zi, nz);
        cells4(y2, aE + N + q.yp, zi, nz);
    }
    stage_b_half<MP>(g, st, E, B, q, z0, sE, sH);
    {
        float a2[2 * MP + 4], a3[2 * MP + 4];
        load_window(a2, sA[0] + t4);
        load_window(a3, sA[1] + t4);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            if (zi + j >= nz) break;
            float* o = aB + q.row + zi + j;
            float s1 = fx * (x3[j] - a3[MP + j]), s2 = -fz * axial<MP, true>(st, a3, j);
            if (g.ndim == 3) {
                s1 -= fy * (y2[j] - a2[MP + j]);
                s2 += fy * (y1[j] - a1[j]);
            }
            o[0] = b1[j] + s1;
            o[N] = b2[j] + s2;
            o[2 * N] = b3[j] + (fz * axial<MP, true>(st, a2, j) - fx * (x1[j] - a1[j]));
        }
    }
    grad_terms<MP, false>(part, st.M, sA[0] + t4 + MP, sA[1] + t4 + MP, sH[0] + t4, sH[1] + t4);
    // the correction's sum has another factor: flushed on its own
    flush_grad<MP>(part, st.M, (double)dt / (double)g.dz, grad);
    if (!correct) return;
    __syncthreads();
    float w[2 * HL + 4], v[4];
    load_window(w, sA1 + t4);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        v[j] = 0.f;                                            // P^{-1} l_E1
#pragma unroll
        for (int k = 0; k <= 2 * HL; ++k) v[j] = fmaf(taps.h[k], w[j + 2 * HL - k], v[j]);
        if (zi + j >= nz) v[j] = 0.f;
    }
    correction_terms<MP>(part, st.M, v, sJ + t4);
    flush_grad<MP>(part, st.M, (double)dt, grad);
}

// E' = E + dt (S B' - J), components 2 and 3, into out (component stride N, component 1 not written).
template <int MP>
__global__ void __launch_bounds__(ADJ_NT) adjoint_enew_kernel(GridP g, StencilP st, const float* __restrict__ E,
                                                              const float* __restrict__ B, const float* __restrict__ J,
                                                              float* __restrict__ out) {
    chain_enter();
    constexpr int W = ADJ_SEG + 2 * MP;
    __shared__ __align__(16) float sE[2][ADJ_SEG + 4 * MP], sH[2][W];
    const long long N = g.ncell;
    const RowAt q = row_at(g, blockIdx.x);
    const RowAt qm = row_at(g, (int)(q.xm / g.nz)), qy = row_at(g, (int)(q.ym / g.nz));
    const int z0 = blockIdx.y * ADJ_SEG, nz = g.nz;
    stage_b_half<MP>(g, st, E, B, q, z0, sE, sH);
    const int t4 = 4 * threadIdx.x, zi = z0 + t4;
    const float dt = g.dt, h = 0.5f * dt, hx = h * (1.f / g.dx), hy = g.ndim == 3 ? h * (1.f / g.dy) : 0.f;
    const float fz = dt * (1.f / g.dz), fx = dt * (1.f / g.dx), fy = g.ndim == 3 ? dt * (1.f / g.dy) : 0.f;
    float h2[2 * MP + 4], h3[2 * MP + 4];
    load_window(h2, sH[0] + t4);
    load_window(h3, sH[1] + t4);
    auto b1 = [&](const RowAt& r, int z) {                     // B'1 at row r
        const float e2 = __ldg(E + N + r.row + z), e3 = __ldg(E + 2 * N + r.row + z);
        return __ldg(B + r.row + z) - (hx * (__ldg(E + 2 * N + r.xp + z) - e3) - hy * (__ldg(E + N + r.yp + z) - e2));
    };
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int z = zi + j;
        if (z >= nz) break;
        const long long c = q.row + z;
        const float v = b1(q, z), dxB1 = v - b1(qm, z), dyB1 = g.ndim == 3 ? v - b1(qy, z) : 0.f;
        out[N + c] = __ldg(E + N + c) + (fy * dyB1 - fz * axial<MP, false>(st, h3, j)) - dt * __ldg(J + N + c);
        out[2 * N + c] = __ldg(E + 2 * N + c) + (fz * axial<MP, false>(st, h2, j) - fx * dxB1) - dt * __ldg(J + 2 * N + c);
    }
}

inline dim3 adj_grid(const GridP& g) {
    return dim3((unsigned)(g.nx * g.ny), (unsigned)((g.nz + ADJ_SEG - 1) / ADJ_SEG));
}

template <typename F>
cudaError_t by_width(int M, F&& f) {
    if (M <= 4) return f(std::integral_constant<int, 4>());
    if (M <= 8) return f(std::integral_constant<int, 8>());
    return f(std::integral_constant<int, 16>());
}

}  // namespace

cudaError_t launch_adjoint_enew(const GridP& g, const StencilP& st, const float* E, const float* B, const float* J,
                                float* out, cudaStream_t s) {
    return by_width(st.M, [&](auto m) {
        return launch_chained(adjoint_enew_kernel<decltype(m)::value>, adj_grid(g), ADJ_NT, 0, s, g, st, E, B, J, out);
    });
}

cudaError_t launch_adjoint_ampere(const GridP& g, const StencilP& st, const float* F, const float* aB, float* aE,
                                  double* grad, cudaStream_t s) {
    return by_width(st.M, [&](auto m) {
        return launch_chained(adjoint_ampere_kernel<decltype(m)::value>, adj_grid(g), ADJ_NT, 0, s, g, st, F, aB, aE, grad);
    });
}

cudaError_t launch_adjoint_faraday(const GridP& g, const StencilP& st, const float* E, const float* B, const float* J1,
                                   const float* aE, float* aB, const float* taps, int hlen, double* grad, cudaStream_t s) {
    TapsP t;
    for (int m = -HL; m <= HL; ++m) t.h[HL + m] = m >= -hlen && m <= hlen ? taps[m + hlen] : 0.f;
    return by_width(st.M, [&](auto m) {
        return launch_chained(adjoint_faraday_kernel<decltype(m)::value>, adj_grid(g), ADJ_NT, 0, s, g, st, E, B, J1, aE, aB,
                              t, hlen > 0 ? 1 : 0, grad);
    });
}

}  // namespace pic
