// Linearised disturbance ensembles about a frozen streamwise-mean base flow
// (paper, "Diagnostic utilities that benefit from vectorization" and "Growth
// functional and linearized adjoint equations of streamwise-mean flow
// dynamics").  A linear group holds one streamwise wavenumber kx != 0 and every
// kept kz; its members are disturbance vectors.  The y-derivative, forcing and
// implicit-apply stages are the DNS's own kernels (one kx column, no mean
// mode); this file holds what differs:
//
//   * the physical-space stage: for one interior plane of one member, the nine
//     fields u, v, w, d_y(u, v, w), d_z(u, v, w) are inverse-transformed along
//     z only (the x dependence is the single harmonic exp(i kx x), so d_x is a
//     factor i kx), multiplied with the base flow B = (U, V, W)(y, z) and its
//     derivatives, and the three products are transformed back and truncated:
//       forward  N_i = i kx U u_i + V d_y u_i + W d_z u_i + v d_y B_i + w d_z B_i
//                     ((B . grad) u' + (u' . grad) B),
//       adjoint  N_i = -(i kx U l_i + V d_y l_i + W d_z l_i) + sum_k l_k d_i B_k
//                     (-(B . grad) l + (grad B)^T l, no x-derivative of B),
//     the equations reading d/dt = -N - grad p + (1/Re) lap in both directions
//     (the adjoint runs in reversed time); the direction is read from device
//     memory at every launch, so a captured step graph serves both;
//   * modified Gram-Schmidt of the member set in the energy inner product
//     <a, b> = (1/4) sum_q sum_j w_j (conj(v_a) v_b + (conj(Dv_a) Dv_b +
//     conj(eta_a) eta_b) / k^2) over the interior nodes (w_j Clenshaw-Curtis
//     weights, Dv = D1 v with v = 0 at the walls), on contiguous copies of the
//     vectors: one launch per vector k projects x_k out of every later vector, a
//     thread-block cluster each.
#include "dns_internal.hpp"
#include "eo.cuh"
#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace dnsk {

constexpr int GS_THREADS = 256;

// threads of the plane stage for transforms of length MZ: one per butterfly of
// the widest stage over the nine lines (at most 320)
__host__ __device__ constexpr int lin_threads(int MZ) {
    int nb = 0;
    for (int s = 0; s < ct_stages(MZ); ++s) nb = MZ / ct_radix(MZ, s) > nb ? MZ / ct_radix(MZ, s) : nb;
    int t = 9 * nb;
    t = t > 320 ? 320 : t;
    return (t + 31) / 32 * 32;
}

template <typename T> struct LinTab;
template <> struct LinTab<double> {
    static __device__ __forceinline__ const double2* tw(const GroupView& g) { return g.twz; }
    static __device__ __forceinline__ const double* base(const GroupView& g) { return g.base; }
    static __device__ __forceinline__ const double* k2i(const GroupView& g) { return g.k2inv; }
    static __device__ __forceinline__ const double* kz(const GroupView& g) { return g.kzt; }
};
template <> struct LinTab<float> {
    static __device__ __forceinline__ const float2* tw(const GroupView& g) { return g.twzf; }
    static __device__ __forceinline__ const float* base(const GroupView& g) { return g.basef; }
    static __device__ __forceinline__ const float* k2i(const GroupView& g) { return g.k2invf; }
    static __device__ __forceinline__ const float* kz(const GroupView& g) { return g.kztf; }
};

template <typename T>
size_t lin_plane_smem_bytes(int mz) {
    return 2 * 9 * (size_t)mz * sizeof(typename C2<T>::type);
}

// i * (a x + b y) for complex x, y and real a, b
template <typename C, typename T>
__device__ __forceinline__ C i_lin2(T a, C x, T b, C y) {
    C r;
    r.x = -(a * x.y + b * y.y);
    r.y = a * x.x + b * y.x;
    return r;
}

template <typename C, typename T>
__device__ __forceinline__ C axpy3(T a, C x, T b, C y, T c, C z) {
    C r;
    r.x = a * x.x + b * y.x + c * z.x;
    r.y = a * x.y + b * y.y + c * z.y;
    return r;
}

template <typename T, int MZ>
__global__ void __launch_bounds__(lin_threads(MZ)) k_lin_plane(GroupView g) {
    typedef typename C2<T>::type C;
    extern __shared__ __align__(16) unsigned char sm[];
    const int y = blockIdx.x, e = blockIdx.y;
    constexpr int Mz = MZ;
    const int Ny = g.ny, E = g.E, NM = g.nmodes, Kz = g.kz;
    C* b0 = (C*)sm;
    C* b1 = b0 + 9 * Mz;
    const bool adjoint = *g.dir != 0;
    const size_t fs = (size_t)Ny * E * NM;
    const C* P = (const C*)g.P5 + ((size_t)y * E + e) * NM;
    const T kx = (T)g.kxt[0];
    const T* kzt = LinTab<T>::kz(g);
    const T* k2i = LinTab<T>::k2i(g);
    for (int i = threadIdx.x; i < 9 * Mz; i += blockDim.x) b0[i] = czero<C>();
    __syncthreads();
    // zero-padded spectral lines: u, v, w | d_y u, d_y v, d_y w | d_z u, d_z v, d_z w
    for (int q = threadIdx.x; q < NM; q += blockDim.x) {
        const int m = q - Kz, pos = m >= 0 ? m : m + Mz;
        const C v = P[q], dv = P[fs + q], d2v = P[2 * fs + q], et = P[3 * fs + q], de = P[4 * fs + q];
        const T kz = kzt[q], ki = k2i[q];
        // u = i (kx Dv - kz eta) / k^2, w = i (kz Dv + kx eta) / k^2
        const C u = cscale(i_lin2(kx, dv, -kz, et), ki);
        const C w = cscale(i_lin2(kz, dv, kx, et), ki);
        const C uy = cscale(i_lin2(kx, d2v, -kz, de), ki);
        const C wy = cscale(i_lin2(kz, d2v, kx, de), ki);
        b0[0 * Mz + pos] = u;
        b0[1 * Mz + pos] = v;
        b0[2 * Mz + pos] = w;
        b0[3 * Mz + pos] = uy;
        b0[4 * Mz + pos] = dv;
        b0[5 * Mz + pos] = wy;
        b0[6 * Mz + pos] = cscale(cmuli(u), kz);
        b0[7 * Mz + pos] = cscale(cmuli(v), kz);
        b0[8 * Mz + pos] = cscale(cmuli(w), kz);
    }
    __syncthreads();
    C* ph = fft_lines_ct<C, +1, MZ, 9>(b0, b1, LinTab<T>::tw(g));
    // products at every z (one thread reads the nine values at z and writes the
    // three results there)
    const T* B = LinTab<T>::base(g) + (size_t)y * Mz;
    const size_t bs = (size_t)Ny * Mz;
    for (int z = threadIdx.x; z < Mz; z += blockDim.x) {
        C a[9];
#pragma unroll
        for (int f = 0; f < 9; ++f) a[f] = ph[f * Mz + z];
        const T U = B[z], V = B[bs + z], W = B[2 * bs + z];
        const T By[3] = {B[3 * bs + z], B[4 * bs + z], B[5 * bs + z]};
        const T Bz[3] = {B[6 * bs + z], B[7 * bs + z], B[8 * bs + z]};
        C N[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            // (B . grad) a_i = i kx U a_i + V d_y a_i + W d_z a_i
            C adv = cscale(cmuli(a[i]), kx * U);
            adv.x += V * a[3 + i].x + W * a[6 + i].x;
            adv.y += V * a[3 + i].y + W * a[6 + i].y;
            if (!adjoint) {
                N[i].x = adv.x + a[1].x * By[i] + a[2].x * Bz[i];
                N[i].y = adv.y + a[1].y * By[i] + a[2].y * Bz[i];
            } else if (i == 0) {
                N[i].x = -adv.x;
                N[i].y = -adv.y;
            } else {
                const C t = (i == 1) ? axpy3(By[0], a[0], By[1], a[1], By[2], a[2])
                                     : axpy3(Bz[0], a[0], Bz[1], a[1], Bz[2], a[2]);
                N[i].x = t.x - adv.x;
                N[i].y = t.y - adv.y;
            }
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) ph[i * Mz + z] = N[i];
    }
    __syncthreads();
    C* out = fft_lines_ct<C, -1, MZ, 3>(ph, ph == b0 ? b1 : b0, LinTab<T>::tw(g));
    // keep |m| <= Kz; the forward transform carries 1/Mz
    const T sc = (T)(1.0 / (double)Mz);
    C* N3 = (C*)g.N3 + ((size_t)y * E + e) * NM;
    for (int i = threadIdx.x; i < 3 * NM; i += blockDim.x) {
        const int f = i / NM, q = i - f * NM, m = q - Kz, pos = m >= 0 ? m : m + Mz;
        N3[(size_t)f * fs + q] = cscale(out[f * Mz + pos], sc);
    }
}

template <typename T, int MZ>
void launch_lin_plane_t(const GroupView& g, cudaStream_t st) {
    k_lin_plane<T, MZ><<<dim3(g.ny, g.E), lin_threads(MZ), lin_plane_smem_bytes<T>(MZ), st>>>(g);
}

template <typename T>
void launch_lin_plane_p(const GroupView& g, cudaStream_t st) {
    switch (g.mz) {   // the spanwise sizes a group accepts
        case 16: launch_lin_plane_t<T, 16>(g, st); break;
        case 32: launch_lin_plane_t<T, 32>(g, st); break;
        case 48: launch_lin_plane_t<T, 48>(g, st); break;
        case 64: launch_lin_plane_t<T, 64>(g, st); break;
        default: launch_lin_plane_t<T, 128>(g, st); break;
    }
}

void launch_lin_plane(const GroupView& g, bool fp64, cudaStream_t st) {
    if (fp64) launch_lin_plane_p<double>(g, st);
    else launch_lin_plane_p<float>(g, st);
}

// ------------------------------------------------------------ Gram-Schmidt

// Why this form: a vector's elements lie E apart in the state, so one CTA per
// vector reading them there drew half of every sector for nothing and left the
// whole FP64 work of a vector (the pipe takes an SM about 16 cycles per warp
// instruction) to one SM.  The vectors are gathered once, contiguous and scaled
// to energy coordinates (sqrt of the weights), and a cluster of GS_CL CTAs
// shares each projection: 45 vectors of 61 x 43 modes, per group 2.5 -> 0.25 ms.

constexpr int GS_CL = 8;     // CTAs per vector
constexpr int GS_EC = 8;     // members of a gather CTA
constexpr int GS_B = 4;      // elements of a thread in flight

// The three parts of a vector in energy coordinates, each [member][q Ny + y]:
// v sqrt(w), Dv sqrt(w) / k, eta sqrt(w) / k.  They lie in arrays that a step
// writes before it reads them (the sub-step states and a combined forcing).
struct GsParts {
    double2* y[3];
};
__host__ __device__ inline GsParts gs_parts(const GroupView& g) { return {{g.v_s, g.e_s, g.Fv}}; }
// g.gsr: [3][E] norms, squared norms' reciprocals, squared norms
__device__ __forceinline__ double* gs_norm(const GroupView& g) { return g.gsr; }
__device__ __forceinline__ double* gs_inv(const GroupView& g) { return g.gsr + g.E; }
__device__ __forceinline__ double* gs_sq(const GroupView& g) { return g.gsr + 2 * g.E; }

__global__ void __launch_bounds__(GS_THREADS) k_gs_gather(GroupView g) {
    extern __shared__ __align__(16) unsigned char sm[];
    double2* X = (double2*)sm;                       // parity parts of v, then natural rows of v, eta [Ny][ec]
    const int Ny = g.ny, E = g.E, q = blockIdx.x, e0 = blockIdx.y * GS_EC, ec = min(GS_EC, E - e0);
    const int NE = (Ny + 1) / 2, NO = Ny / 2, RP = spc::eo_rp(Ny);
    double2* VN = X + Ny * ec;
    double2* HN = VN + Ny * ec;
    for (int i = threadIdx.x; i < NE * ec; i += blockDim.x) {
        const int p = i / ec, el = i - p * ec;
        const spc::EoRows R = spc::eo_rows(p, Ny);
        const size_t h0 = ((size_t)q * Ny + R.y0) * E + e0 + el, h1 = ((size_t)q * Ny + R.y1) * E + e0 + el;
        const double2 a = g.v_t[h0];
        VN[R.y0 * ec + el] = a;
        HN[R.y0 * ec + el] = g.e_t[h0];
        X[p * ec + el] = a;
        if (R.pair) {
            const double2 b = g.v_t[h1];
            VN[R.y1 * ec + el] = b;
            HN[R.y1 * ec + el] = g.e_t[h1];
            X[p * ec + el] = make_double2(a.x + b.x, a.y + b.y);
            X[(NE + p) * ec + el] = make_double2(a.x - b.x, a.y - b.y);
        }
    }
    __syncthreads();
    const double* D1e = g.D1EO64;                    // even output rows (contract the odd part), then the odd ones
    const double* D1o = D1e + (size_t)NO * RP;
    const GsParts Y = gs_parts(g);
    const size_t n = (size_t)g.nmodes * Ny;
    const double ik = sqrt(g.k2inv[q]);
    for (int i = threadIdx.x; i < NE * ec; i += blockDim.x) {
        const int el = i / NE, p = i - el * NE;      // consecutive threads: consecutive rows of a vector
        double2 de = make_double2(0.0, 0.0), dd = de;
#pragma unroll 4
        for (int k = 0; k < NO; ++k) {
            const double b = D1e[k * RP + p];
            const double2 x = X[(NE + k) * ec + el];
            de.x += b * x.x;
            de.y += b * x.y;
        }
#pragma unroll 4
        for (int k = 0; k < NE; ++k) {
            const double b = D1o[k * RP + p];
            const double2 x = X[k * ec + el];
            dd.x += b * x.x;
            dd.y += b * x.y;
        }
        const spc::EoRows R = spc::eo_rows(p, Ny);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (r && !R.pair) break;
            const int y = r ? R.y1 : R.y0;
            const double w = sqrt(g.ccw[y + 1]), wk = w * ik, h = R.pair ? 0.5 : 1.0, sg = !R.pair ? 0.0 : r ? -1.0 : 1.0;
            const size_t o = (size_t)(e0 + el) * n + (size_t)q * Ny + y;
            const double2 v = VN[y * ec + el], t = HN[y * ec + el];
            Y.y[0][o] = make_double2(v.x * w, v.y * w);
            Y.y[1][o] = make_double2(h * (de.x + sg * dd.x) * wk, h * (de.y + sg * dd.y) * wk);
            Y.y[2][o] = make_double2(t.x * wk, t.y * wk);
        }
    }
}

// Sum of the threads' values over the cluster, in a fixed order, times f; the
// result in every thread.  On the FP64 pipe an addition costs a warp 16 cycles
// of its SM, so one warp adds up the CTA and one thread the cluster.
struct GsShared {
    double2 lane[GS_THREADS];
    double2 part, sum;
};
__device__ __forceinline__ double2 cluster_sum(double2 v, double f, GsShared& sh) {
    cg::cluster_group cl = cg::this_cluster();
    sh.lane[threadIdx.x] = v;
    __syncthreads();
    if (threadIdx.x < 32) {
        double2 t = sh.lane[threadIdx.x];
#pragma unroll
        for (int i = 32; i < GS_THREADS; i += 32) {
            const double2 u = sh.lane[threadIdx.x + i];
            t.x += u.x;
            t.y += u.y;
        }
        for (int o = 16; o > 0; o >>= 1) {
            t.x += __shfl_xor_sync(0xffffffffu, t.x, o);
            t.y += __shfl_xor_sync(0xffffffffu, t.y, o);
        }
        if (threadIdx.x == 0) sh.part = t;
    }
    cl.sync();
    if (threadIdx.x == 0) {
        double2 t = make_double2(0.0, 0.0);
#pragma unroll
        for (int r = 0; r < GS_CL; ++r) {
            const double2 u = *cl.map_shared_rank(&sh.part, r);
            t.x += u.x;
            t.y += u.y;
        }
        sh.sum = make_double2(t.x * f, t.y * f);
    }
    cl.sync();       // the sum is there, and no peer reads this CTA's part any more
    return sh.sum;
}

// Launch k = -1: the squared norm of x_0.  Launch k >= 0: cluster b takes
// x_j -= (<x_k, x_j> / <x_k, x_k>) x_k for j = k + 1 + b; x_{k+1} then has all its
// projections, and its squared norm and its reciprocal are recorded.
__global__ void __cluster_dims__(GS_CL, 1, 1) __launch_bounds__(GS_THREADS, 3) k_gs_project(GroupView g, int k) {
    __shared__ GsShared sh;
    const int j = k + 1 + blockIdx.x / GS_CL, rank = blockIdx.x % GS_CL;
    const GsParts Y = gs_parts(g);
    const int n = g.nmodes * g.ny, n3 = 3 * n, step = GS_CL * GS_THREADS, i0 = rank * GS_THREADS + threadIdx.x;
    // element i of the three parts' concatenation, of vector m
    auto at = [&](int m, int i) -> double2* {
        const int f = (i >= n) + (i >= 2 * n);
        return (f == 0 ? Y.y[0] : f == 1 ? Y.y[1] : Y.y[2]) + (size_t)m * n + (i - f * n);
    };
    // GS_B elements of a thread at a time, their loads in flight together; the
    // first batch stays in registers between the product and the projection
    double2 a0[GS_B], b0[GS_B];
    auto load = [&](int i, double2* a, double2* b) {
#pragma unroll
        for (int u = 0; u < GS_B; ++u) {
            a[u] = b[u] = make_double2(0.0, 0.0);
            if (i + u * step < n3) {
                b[u] = *at(j, i + u * step);
                if (k >= 0) a[u] = *at(k, i + u * step);
            }
        }
    };
    load(i0, a0, b0);
    double2 c = make_double2(0.0, 0.0);
    if (k >= 0) {
        double2 s = make_double2(0.0, 0.0);
        auto dot = [&](const double2* a, const double2* b) {
#pragma unroll
            for (int u = 0; u < GS_B; ++u) {
                s.x = fma(a[u].x, b[u].x, fma(a[u].y, b[u].y, s.x));
                s.y = fma(a[u].x, b[u].y, fma(-a[u].y, b[u].x, s.y));
            }
        };
        dot(a0, b0);
        for (int i = i0 + GS_B * step; i < n3; i += GS_B * step) {
            double2 a[GS_B], b[GS_B];
            load(i, a, b);
            dot(a, b);
        }
        c = cluster_sum(s, gs_inv(g)[k], sh);
    }
    const bool norm = j == k + 1;
    double2 s = make_double2(0.0, 0.0);
    auto update = [&](int i, const double2* a, const double2* b) {
#pragma unroll
        for (int u = 0; u < GS_B; ++u) {
            double2 x = b[u];
            if (k >= 0 && i + u * step < n3) {
                x.x = fma(c.y, a[u].y, fma(-c.x, a[u].x, x.x));
                x.y = fma(-c.y, a[u].x, fma(-c.x, a[u].y, x.y));
                *at(j, i + u * step) = x;
            }
            if (norm) s.x = fma(x.x, x.x, fma(x.y, x.y, s.x));
        }
    };
    update(i0, a0, b0);
    for (int i = i0 + GS_B * step; i < n3; i += GS_B * step) {
        double2 a[GS_B], b[GS_B];
        load(i, a, b);
        update(i, a, b);
    }
    if (norm) {
        __syncthreads();
        s = cluster_sum(s, 1.0, sh);
        if (rank == 0 && threadIdx.x == 0) {
            gs_sq(g)[j] = s.x;
            gs_inv(g)[j] = 1.0 / s.x;
        }
    }
}

// Every vector normalised and back in the state, GS_EC members a CTA; the CTAs of
// mode 0 record the energy norms (the 1/4 included).
__global__ void __launch_bounds__(GS_THREADS) k_gs_scatter(GroupView g) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int Ny = g.ny, E = g.E, q = blockIdx.x, e0 = blockIdx.y * GS_EC, ec = min(GS_EC, E - e0);
    double* iw = (double*)sm;            // 1 / sqrt(w)
    double* ir = iw + Ny;                // 1 / norm
    for (int i = threadIdx.x; i < Ny + ec; i += blockDim.x) {
        if (i < Ny) iw[i] = 1.0 / sqrt(g.ccw[i + 1]);
        else {
            const double r = sqrt(0.25 * gs_sq(g)[e0 + i - Ny]);
            ir[i - Ny] = 1.0 / r;
            if (q == 0) gs_norm(g)[e0 + i - Ny] = r;
        }
    }
    __syncthreads();
    const GsParts Y = gs_parts(g);
    const size_t n = (size_t)g.nmodes * Ny;
    const double k1 = sqrt(1.0 / g.k2inv[q]);
    for (int i = threadIdx.x; i < Ny * ec; i += blockDim.x) {
        const int y = i / ec, el = i - y * ec;
        const double s = iw[y] * ir[el], t = s * k1;
        const size_t o = (size_t)(e0 + el) * n + (size_t)q * Ny + y, h = ((size_t)q * Ny + y) * E + e0 + el;
        const double2 a = Y.y[0][o], b = Y.y[2][o];
        g.v_t[h] = make_double2(a.x * s, a.y * s);
        g.e_t[h] = make_double2(b.x * t, b.y * t);
    }
}

int launch_lin_orthonormalize(const GroupView& g, cudaStream_t st) {
    const dim3 grid(g.nmodes, (g.E + GS_EC - 1) / GS_EC);
    k_gs_gather<<<grid, GS_THREADS, 3 * (size_t)g.ny * GS_EC * sizeof(double2), st>>>(g);
    for (int k = -1; k < g.E - 1; ++k) k_gs_project<<<GS_CL * (k < 0 ? 1 : g.E - 1 - k), GS_THREADS, 0, st>>>(g, k);
    k_gs_scatter<<<grid, GS_THREADS, (g.ny + GS_EC) * sizeof(double), st>>>(g);
    return g.E + 2;
}

void set_attributes_linear() {
    allow_max_dynamic_smem(k_gs_gather);
    // the plane stage needs at most 2 x 9 x 128 x 16 B = 36 KB, below the default limit
}

}  // namespace dnsk
