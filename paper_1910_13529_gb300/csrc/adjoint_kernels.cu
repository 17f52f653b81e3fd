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
// The gradient sums of FP32 fields are kept to about 48 bits in pairs of FP32 numbers (pair_math.h: exact
// differences, products and sums) and added up in FP64 from the warp
// totals on.  FP64 arithmetic per cell was what the step waited for: this chip does 64 FP32 operations
// for one in FP64, so that 1024 x 256 cells with M = 4 took 34 us per gradient kernel, 127 us of the
// 163 us of an adjoint step (now 26 us).  The pairs cost 17 FP32 operations per tap and component and the step is
// bound by its launches and their latency.
#include <cuda_runtime.h>

#include <type_traits>

#include "pair_math.h"
#include "pic_internal.h"

namespace pic {

namespace {

constexpr int ADJ_NT = 128, ADJ_SEG = 4 * ADJ_NT;
constexpr int HL = PIC_MAX_HLEN;

__device__ __forceinline__ int wrapm(int a, int n) { return a < 0 ? a + n : (a >= n ? a - n : a); }

// grad[l] += scale * the block's sum of acc[l], l < M
template <int MAXM>
__device__ __forceinline__ void flush_grad(PairSum (&acc)[MAXM], int M, double scale, double* grad) {
    __shared__ double part[MAXM][ADJ_NT / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int l = 0; l < MAXM; ++l) {
        if (l >= M) break;
        acc[l].warp_sum();
        if (lane == 0) part[l][w] = acc[l].value();
    }
    __syncthreads();
    if (threadIdx.x < M) {
        double v = 0.0;
        for (int q = 0; q < ADJ_NT / 32; ++q) v += part[threadIdx.x][q];
        if (v != 0.0) atomicAdd(grad + threadIdx.x, scale * v);
    }
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
    for (int l = 1; l <= MP; ++l)
        s = fmaf(st.C[l - 1], PLUS ? w[MP + j + l] - w[MP + j - l + 1] : w[MP + j + l - 1] - w[MP + j - l], s);
    return s;
}

// acc[l - 1] += sum_j l3[j] D_l f2 - l2[j] D_l f3 over the thread's four cells, D_l tap l of d+ (PLUS)
// or d- without its 1/dz
template <int MP, bool PLUS>
__device__ __forceinline__ void grad_terms(PairSum (&acc)[MP], const float (&l2)[4], const float (&l3)[4],
                                           const float (&f2)[2 * MP + 4], const float (&f3)[2 * MP + 4]) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (l2[j] == 0.f && l3[j] == 0.f) continue;
#pragma unroll
        for (int l = 1; l <= MP; ++l) {
            const int a = PLUS ? MP + j + l : MP + j + l - 1, b = PLUS ? MP + j - l + 1 : MP + j - l;
            float d, e;
            add2(f3[a], -f3[b], d, e);
            acc[l - 1].fma(-l2[j], d, e);
            add2(f2[a], -f2[b], d, e);
            acc[l - 1].fma(l3[j], d, e);
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
    PairSum acc[MP];
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
    {
        const float l2[4] = {b2[MP], b2[MP + 1], b2[MP + 2], b2[MP + 3]};
        const float l3[4] = {b3[MP], b3[MP + 1], b3[MP + 2], b3[MP + 3]};
        float f2[2 * MP + 4], f3[2 * MP + 4];
        load_window(f2, sF[0] + t4);
        load_window(f3, sF[1] + t4);
        grad_terms<MP, true>(acc, l2, l3, f2, f3);
    }
    flush_grad<MP>(acc, st.M, -(double)h / (double)g.dz, grad);
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
    PairSum acc[MP];
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
        const float l2[4] = {a2[MP], a2[MP + 1], a2[MP + 2], a2[MP + 3]};
        const float l3[4] = {a3[MP], a3[MP + 1], a3[MP + 2], a3[MP + 3]};
        float f2[2 * MP + 4], f3[2 * MP + 4];
        load_window(f2, sH[0] + t4);
        load_window(f3, sH[1] + t4);
        grad_terms<MP, false>(acc, l2, l3, f2, f3);
    }
    // the correction's sum has another factor: flushed on its own
    flush_grad<MP>(acc, st.M, (double)dt / (double)g.dz, grad);
    if (!correct) return;
    __syncthreads();
    PairSum cor[MP];
    float w[2 * HL + 4], jw[2 * MP + 4];
    load_window(w, sA1 + t4);
    load_window(jw, sJ + t4);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        float v = 0.f;                                         // P^{-1} l_E1
#pragma unroll
        for (int k = 0; k <= 2 * HL; ++k) v = fmaf(taps.h[k], w[j + 2 * HL - k], v);
        if (v == 0.f || zi + j >= nz) continue;
        float bh = jw[MP + j], bl = 0.f;                       // sum of J1 over |m| < l
        cor[0].fma(v, bh, 0.f);
#pragma unroll
        for (int l = 2; l <= MP; ++l) {
            float s, e;
            add2(bh, jw[MP + j - (l - 1)], s, e);
            bl += e;
            add2(s, jw[MP + j + (l - 1)], bh, e);
            bl += e;
            cor[l - 1].fma(v, bh, bl);
        }
    }
    flush_grad<MP>(cor, st.M, (double)dt, grad);
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
