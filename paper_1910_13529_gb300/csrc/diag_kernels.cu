// Diagnostics: Gauss residual d-.E - rho - rho_bg (Eq. Gauss of Sec. 2.1, with the same axial d- as Ampere's
// law), field and kinetic energy.  The divergence and each particle's gamma - 1 are wide sums of FP32 parts
// (wide_math.h, about 2^-70), which become FP64 where they meet rho and the sums; the rest is FP64
// throughout.  With FP64 from the first difference on, the FP64 pipe and its conversions were busy all the
// time: pic_gauss on 1024 x 256 nodes 39 us (M = 1) and 77 (M = 16), now 29 and 36; on 128 x 64 x 64 with 1e6
// particles 126 and 66.
#include <cuda_runtime.h>

#include <type_traits>

#include "pic_internal.h"
#include "wide_math.h"

namespace pic {

namespace {

constexpr int DG_NT = 128, DG_SEG = 4 * DG_NT;

// Cell sizes of the axes, their reciprocals in three parts, -rho_bg as well; plain: reciprocals of a size
// that FP32 products can take.
struct InvP {
    double h[3], bg;
    float z[3], x[3], y[3], back[3];
    bool plain;
};

// Nodes of one row segment [z0, z0 + DG_SEG): d-.E - rho_bg at the thread's four nodes.  sE: the E1 cells the
// windows need (staged here).  Differences are exact, and the sum of all axes is wide as long as its largest
// term lies where FP32 products leave exact residuals; outside (fields below about 1e-18 or above 1e30) and
// for values that are not finite the node takes FP64 from the first difference on.
template <int MP>
__device__ __forceinline__ void div_row(const GridP& g, const StencilP& st, const InvP& inv, const float* __restrict__ E,
                                        int row_index, int z0, float* sE, double (&out)[4]) {
    constexpr int W = DG_SEG + 2 * MP;
    const long long N = g.ncell;
    const int j = row_index % g.nx, k = row_index / g.nx;
    const long long row = (long long)row_index * g.nz;
    const long long rxm = ((long long)k * g.nx + (j == 0 ? g.nx - 1 : j - 1)) * g.nz;
    const long long rym = ((long long)(k == 0 ? g.ny - 1 : k - 1) * g.nx + j) * g.nz;
    for (int i = threadIdx.x; i < W; i += DG_NT) {
        const int z = z0 - MP + i;
        const bool in = (unsigned)z < (unsigned)g.nz;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"((unsigned)__cvta_generic_to_shared(sE + i)),
                     "l"(E + row + (in ? z : 0)), "r"(in ? 4 : 0)
                     : "memory");
    }
    const int zi = z0 + 4 * threadIdx.x;
    float x1[4], x0[4], y1[4], y0[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const bool in = zi + q < g.nz;
        x1[q] = in ? __ldg(E + N + row + zi + q) : 0.f;
        x0[q] = in ? __ldg(E + N + rxm + zi + q) : 0.f;
        y1[q] = in && g.ndim == 3 ? __ldg(E + 2 * N + row + zi + q) : 0.f;
        y0[q] = in && g.ndim == 3 ? __ldg(E + 2 * N + rym + zi + q) : 0.f;
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
    float w[2 * MP + 4];
#pragma unroll
    for (int q = 0; q < (2 * MP + 4) / 4; ++q) {
        const float4 v = *reinterpret_cast<const float4*>(sE + 4 * threadIdx.x + 4 * q);
        w[4 * q] = v.x;
        w[4 * q + 1] = v.y;
        w[4 * q + 2] = v.z;
        w[4 * q + 3] = v.w;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        out[q] = 0.0;
        if (zi + q >= g.nz) continue;
        WideSum s, t;
        float top = 0.f, range = 0.f;                 // largest term, largest difference
#pragma unroll
        for (int l = 1; l <= MP; ++l) {
            if (l > st.M) break;
            float d, e;
            two_sum(w[MP + q + l - 1], -w[MP + q - l], d, e);
            range = fmaxf(range, fabsf(d));
            top = fmaxf(top, fabsf(s.fma(st.Cm[l - 1], d, e)));      // the B-side d- of Ampere's law
        }
        s.scale(inv.z[0], inv.z[1], inv.z[2]);
        two_sum(x1[q], -x0[q], t.h, t.m);
        top = fmaxf(top, fabsf(t.h));
        range = fmaxf(range, fabsf(t.h));
        t.l = 0.f;
        t.scale(inv.x[0], inv.x[1], inv.x[2]);
        s.add(t.h, t.m, t.l);
        if (g.ndim == 3) {
            two_sum(y1[q], -y0[q], t.h, t.m);
            top = fmaxf(top, fabsf(t.h));
            range = fmaxf(range, fabsf(t.h));
            t.l = 0.f;
            t.scale(inv.y[0], inv.y[1], inv.y[2]);
            s.add(t.h, t.m, t.l);
        }
        s.add(inv.back[0], inv.back[1], inv.back[2]);
        if (inv.plain && fabsf(s.h) < 1e30f && (top > 1e-18f || range == 0.f)) {
            out[q] = s.value();
        } else {
            double dz = 0.0;
#pragma unroll 1
            for (int l = 1; l <= st.M; ++l) {
                const float* c = sE + 4 * threadIdx.x + MP + q;
                dz += (double)st.Cm[l - 1] * ((double)c[l - 1] - (double)c[-l]);
            }
            out[q] = dz / inv.h[0] + ((double)x1[q] - (double)x0[q]) / inv.h[1];
            if (g.ndim == 3) out[q] += ((double)y1[q] - (double)y0[q]) / inv.h[2];
            out[q] += inv.bg;
        }
    }
    __syncthreads();                                  // sE may be filled again
}

template <int MP>
__global__ void __launch_bounds__(DG_NT, 5) gauss_kernel(GridP g, StencilP st, InvP inv, const float* E, const double* rho,
                                                      double* G) {
    __shared__ __align__(16) float sE[DG_SEG + 2 * MP];
    const int z0 = blockIdx.y * DG_SEG;
    double d[4];
    div_row<MP>(g, st, inv, E, blockIdx.x, z0, sE, d);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int z = z0 + 4 * threadIdx.x + q;
        if (z >= g.nz) break;
        const long long c = (long long)blockIdx.x * g.nz + z;
        G[c] = d[q] - rho[c];
    }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// non-negative doubles order like their bit patterns
__device__ __forceinline__ void atomic_max_nonneg(double* a, double v) {
    atomicMax(reinterpret_cast<unsigned long long*>(a), (unsigned long long)__double_as_longlong(v));
}

// acc: [0] max|G| [1] sum G^2 [2] max|rho| [3] sum (E^2+B^2) [4] kinetic [5] interior nodes
//      [6] live particles
template <int MP>
__global__ void __launch_bounds__(DG_NT) diag_kernel(GridP g, StencilP st, InvP inv, const float* E, const float* B,
                                                     const double* rho, int margin, int segs, long long items, double* acc) {
    __shared__ __align__(16) float sE[DG_SEG + 2 * MP];
    __shared__ double sh[5][DG_NT / 32];
    const long long N = g.ncell;
    double gmax = 0.0, rmax = 0.0, g2 = 0.0, w = 0.0;
    int cnt = 0;
    for (long long it = blockIdx.x; it < items; it += gridDim.x) {
        const int r = (int)(it / segs), z0 = (int)(it - (long long)r * segs) * DG_SEG;
        double d[4];
        div_row<MP>(g, st, inv, E, r, z0, sE, d);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int z = z0 + 4 * threadIdx.x + q;
            if (z >= g.nz) break;
            const long long c = (long long)r * g.nz + z;
#pragma unroll
            for (int m = 0; m < 3; ++m) {
                const double e = __ldg(E + m * N + c), b = __ldg(B + m * N + c);
                w += e * e + b * b;
            }
            const double rv = rho[c];
            rmax = fmax(rmax, fabs(rv));
            if (z >= margin && z < g.nz - margin) {
                const double G = d[q] - rv;
                gmax = fmax(gmax, fabs(G));
                g2 += G * G;
                ++cnt;
            }
        }
    }
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    gmax = warp_max(gmax);
    rmax = warp_max(rmax);
    g2 = warp_sum(g2);
    w = warp_sum(w);
    cnt = __reduce_add_sync(0xffffffffu, cnt);
    if (lane == 0) {
        sh[0][wid] = gmax;
        sh[1][wid] = g2;
        sh[2][wid] = rmax;
        sh[3][wid] = w;
        sh[4][wid] = cnt;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double v[5] = {0, 0, 0, 0, 0};
        for (int q = 0; q < DG_NT / 32; ++q) {
            v[0] = fmax(v[0], sh[0][q]);
            v[1] += sh[1][q];
            v[2] = fmax(v[2], sh[2][q]);
            v[3] += sh[3][q];
            v[4] += sh[4][q];
        }
        atomic_max_nonneg(acc + 0, v[0]);
        atomicAdd(acc + 1, v[1]);
        atomic_max_nonneg(acc + 2, v[2]);
        atomicAdd(acc + 3, v[3]);
        atomicAdd(acc + 5, v[4]);
    }
}

__global__ void __launch_bounds__(256) kinetic_kernel(SpeciesP sp, double* acc) {
    WideSum e;
    double big = 0.0;                                 // momenta beyond the range of FP32 squares
    int alive = 0;
    const long long n = *sp.count;
    for (long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x; p < n;
         p += (long long)gridDim.x * blockDim.x) {
        if (sp.cell[p] < 0) continue;
        const float u0 = sp.u[p], u1 = sp.u[sp.cap + p], u2 = sp.u[2 * sp.cap + p];
        if (u0 * u0 + u1 * u1 + u2 * u2 < 1e30f) {
            const WideSum k = gamma_minus_one(u0, u1, u2);
            e.add(k.h, k.m, k.l);
        } else {
            const double a = u0, b = u1, c = u2;
            big += sqrt(1.0 + a * a + b * b + c * c) - 1.0;
        }
        ++alive;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e.add_lane(e, o);
    big = warp_sum(big);
    alive = __reduce_add_sync(0xffffffffu, alive);
    __shared__ double sh[2][8];
    if ((threadIdx.x & 31) == 0) {
        sh[0][threadIdx.x >> 5] = e.value() + big;
        sh[1][threadIdx.x >> 5] = alive;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0, c = 0;
        for (int q = 0; q < (int)(blockDim.x >> 5); ++q) {
            a += sh[0][q];
            c += sh[1][q];
        }
        atomicAdd(acc + 4, a * sp.wm);
        atomicAdd(acc + 6, c);
    }
}

InvP inverses(const GridP& g, double rho_bg) {
    InvP q;
    q.plain = true;
    // v + rest in three parts
    auto parts = [](double v, double rest, float* p) {
        p[0] = (float)v;
        p[1] = (float)(v - (double)p[0]);
        p[2] = (float)(v - (double)p[0] - (double)p[1] + rest);
    };
    float* const inv[3] = {q.z, q.x, q.y};
    const float h[3] = {g.dz, g.dx, g.dy};
    for (int a = 0; a < 3; ++a) {
        q.h[a] = h[a];
        const double r = 1.0 / q.h[a];
        parts(r, std::fma(-r, q.h[a], 1.0) * r, inv[a]);
        if (a < g.ndim) q.plain = q.plain && r > 1e-10 && r < 1e10;
    }
    q.bg = -rho_bg;
    parts(q.bg, 0.0, q.back);
    q.plain = q.plain && (rho_bg == 0.0 || (std::fabs(rho_bg) > 1e-18 && std::fabs(rho_bg) < 1e30));
    return q;
}

template <typename F>
cudaError_t by_width(int M, F&& f) {
    if (M <= 4) f(std::integral_constant<int, 4>());
    else if (M <= 8) f(std::integral_constant<int, 8>());
    else f(std::integral_constant<int, 16>());
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_gauss(const GridP& g, const StencilP& st, const float* E, const double* rho,
                         double rho_bg, double* G, cudaStream_t s) {
    const dim3 grid((unsigned)(g.nx * g.ny), (unsigned)((g.nz + DG_SEG - 1) / DG_SEG));
    return by_width(st.M, [&](auto m) {
        gauss_kernel<decltype(m)::value><<<grid, DG_NT, 0, s>>>(g, st, inverses(g, rho_bg), E, rho, G);
    });
}

cudaError_t launch_diag_reduce(const GridP& g, const StencilP& st, const float* E, const float* B,
                               const double* rho, double rho_bg, int margin, double* acc,
                               cudaStream_t s) {
    const int segs = (g.nz + DG_SEG - 1) / DG_SEG;
    const long long items = (long long)segs * g.nx * g.ny;
    const unsigned blocks = (unsigned)(items < 152 * 8 ? items : 152 * 8);
    return by_width(st.M, [&](auto m) {
        diag_kernel<decltype(m)::value>
            <<<blocks, DG_NT, 0, s>>>(g, st, inverses(g, rho_bg), E, B, rho, margin, segs, items, acc);
    });
}

cudaError_t launch_kinetic(const GridP& g, const SpeciesP& sp, long long extent, double* acc,
                           cudaStream_t s) {
    (void)g;
    if (extent <= 0) return cudaSuccess;
    long long want = (extent + 255) / 256;
    unsigned blocks = (unsigned)(want < 152 * 8 ? want : 152 * 8);
    kinetic_kernel<<<blocks, 256, 0, s>>>(sp, acc);
    return cudaGetLastError();
}

}  // namespace pic
