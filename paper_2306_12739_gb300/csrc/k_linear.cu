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
#include "dft.cuh"
#include "eo.cuh"
#include "pairs.cuh"
#include <cooperative_groups.h>

namespace cg = cooperative_groups;

namespace dnsk {

constexpr int GS_THREADS = 256;

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

using namespace prs;

// The plane stage: one CTA per interior plane and NV vectors, one warp per field
// (u, v, w, then their y- and z-derivatives), 32 / H = NV transforms of H lanes in
// a warp.  A transform of Mz = N1 N2 points is a four-step one inside its lanes (a
// lane does the residues 2 j and 2 j + 1 modulo N2 as a pair, then N2-point DFTs
// whose two halves are the rows p and p + Mz/2), so only the products between the
// inverse and the forward transforms need the CTA together.  61 planes x 45 vectors
// of 64 points: 16.6 us a launch alone with a Stockham transform of the nine lines of
// one vector per CTA, a barrier per radix-4 pass, 18.5 here; but a launch takes less of
// the chip, and groups run side by side: 3 x 45 vectors, 20 + 20 steps with
// Gram-Schmidt 10270 -> 9790 us.
template <int MZ> struct LinCfg {
    static constexpr int N1 = dft::Split<MZ>::N1, N2 = dft::Split<MZ>::N2, H = N2 / 2, HP = MZ / 2;
    static constexpr int NV = 32 / H;                         // vectors of a CTA
    static constexpr int NQ = (N1 + H - 1) / H;               // N2-point tasks per lane
    static constexpr int KZ = (MZ - 1) / 3;
    static constexpr int XS = H + 1;                          // rows of the exchange (complex pairs)
    // a transform's storage: its exchange, then its points; for H = 4 two transforms
    // share an eight-lane access and lie four 16-byte banks apart
    static constexpr int R0 = N1 * XS > HP ? N1 * XS : HP;
    static constexpr int RS = H == 4 ? R0 + ((4 - R0 % 8) + 8) % 8 : R0;
};
constexpr int LIN_THREADS = 9 * 32;

template <typename T, int MZ>
size_t lin_plane_smem_bytes() {
    typedef LinCfg<MZ> K;
    return sizeof(Pc<T>) * (9 * K::NV * K::RS + K::N1 * K::H);
}

template <typename T, int MZ>
__global__ void __launch_bounds__(LIN_THREADS, sizeof(T) == 4 ? 2 : 1) k_lin_plane(GroupView g) {
    typedef LinCfg<MZ> K;
    constexpr int N1 = K::N1, N2 = K::N2, H = K::H, HP = K::HP, NV = K::NV, KZ = K::KZ, XS = K::XS, RS = K::RS;
    struct Cv { T x, y; };
    extern __shared__ __align__(16) unsigned char sm[];
    Pc<T>* X = (Pc<T>*)sm;                                     // [field][vector][RS]
    Pc<T>* tw = X + 9 * NV * RS;                               // [k1][j]: the residue pair (2 j, 2 j + 1)
    const int y = blockIdx.x, e0 = blockIdx.y * NV, E = g.E, NM = g.nmodes;
    const int tid = threadIdx.x, lane = tid & 31, f = tid >> 5, j = lane % H, vec = lane / H;
    const bool live = e0 + vec < E;
    const size_t fs = (size_t)g.ny * E * NM;
    for (int i = tid; i < N1 * H; i += LIN_THREADS) {
        const int k1 = i / H, r = i - k1 * H;
        const auto a = LinTab<T>::tw(g)[2 * r * k1], b = LinTab<T>::tw(g)[(2 * r + 1) * k1];
        tw[i] = {pr((T)a.x, (T)b.x), pr((T)a.y, (T)b.y)};
    }
    const T kx = (T)g.kxt[0];
    Pc<T>* L = X + (f * NV + vec) * RS;

    // ---- field f = 3 kind + comp: u_comp, d_y u_comp (kind 1), d_z u_comp (2), with
    // u = i (kx Dv - kz eta) / k^2, w = i (kz Dv + kx eta) / k^2 (d_y: D2v, D eta)
    const int kind = f / 3, comp = f - 3 * kind;
    Pc<T> v[N1];
    {
        const Cv* P = (const Cv*)g.P5 + ((size_t)y * E + e0 + vec) * NM;
        const Cv* A = P + (comp == 1 ? (kind == 1 ? 1 : 0) : (kind == 1 ? 2 : 1)) * fs;
        const Cv* B = P + (kind == 1 ? 4 : 3) * fs;
        const T* kzt = LinTab<T>::kz(g);
        const T* k2i = LinTab<T>::k2i(g);
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) {
            v[n1] = {dup((T)0), dup((T)0)};
            const int z0 = N2 * n1;
            if (z0 > KZ && z0 + N2 - 1 < MZ - KZ) continue;      // wholly padding
            Cv c[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int z = z0 + 2 * j + r;
                const bool lo = z <= KZ;
                c[r] = {(T)0, (T)0};
                if (!live || !(lo || z >= MZ - KZ)) continue;
                const int q = lo ? z + KZ : z - MZ + KZ;
                const T kz = kzt[q];
                Cv a = A[q];
                if (comp != 1) {
                    const Cv b = B[q];
                    const T ki = k2i[q], ka = comp == 0 ? kx : kz, kb = comp == 0 ? -kz : kx;
                    a = {-((ka * a.y + kb * b.y) * ki), (ka * a.x + kb * b.x) * ki};
                }
                c[r] = kind == 2 ? Cv{-kz * a.y, kz * a.x} : a;
            }
            v[n1] = {pr(c[0].x, c[1].x), pr(c[0].y, c[1].y)};
        }
    }
    pdft_padded<N1, +1>(v);
    __syncthreads();                                             // the twiddles
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) stp(L + k1 * XS + j, k1 == 0 ? v[0] : pmul<true>(v[k1], ldp(tw + k1 * H + j)));
    __syncwarp();
    Pc<T> o[K::NQ][H];
#pragma unroll
    for (int q = 0; q < K::NQ; ++q) {
        const int k1 = j + H * q;
        if (K::NQ * H > N1 && k1 >= N1) continue;
#pragma unroll
        for (int i = 0; i < H; ++i) o[q][i] = ldp(L + k1 * XS + i);
        dft_dit<N2, +1>(o[q]);
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < K::NQ; ++q) {
        const int k1 = j + H * q;
        if (K::NQ * H > N1 && k1 >= N1) continue;
#pragma unroll
        for (int k = 0; k < H; ++k) stp(L + k1 + N1 * k, o[q][k]);
    }
    __syncthreads();

    // ---- products at the rows p and p + Mz/2, over the lines of u, v, w
    const bool adjoint = *g.dir != 0;
    const size_t bs = (size_t)g.ny * MZ;
    for (int i = tid; i < NV * HP; i += LIN_THREADS) {
        const int ve = i / HP, p = i - ve * HP;
        const T* B = LinTab<T>::base(g) + (size_t)y * MZ + p;
        Pc<T> a[9];
#pragma unroll
        for (int c = 0; c < 9; ++c) a[c] = ldp(X + (c * NV + ve) * RS + p);
        auto base = [&](int c) { return pr(B[c * bs], B[c * bs + HP]); };
        const Pr<T> U = base(0) * dup(kx), V = base(1), W = base(2);
        Pr<T> By[3], Bz[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) { By[c] = base(3 + c); Bz[c] = base(6 + c); }
        Pc<T> N[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            // (B . grad) a_c = i kx U a_c + V d_y a_c + W d_z a_c
            const Pc<T> adv = {pfma(V, a[3 + c].x, W * a[6 + c].x) - U * a[c].y,
                               pfma(V, a[3 + c].y, pfma(W, a[6 + c].y, U * a[c].x))};
            if (!adjoint) {
                N[c] = {pfma(a[1].x, By[c], pfma(a[2].x, Bz[c], adv.x)), pfma(a[1].y, By[c], pfma(a[2].y, Bz[c], adv.y))};
            } else if (c == 0) {
                N[c] = {pneg(adv.x), pneg(adv.y)};
            } else {
                const Pr<T>* G = c == 1 ? By : Bz;
                N[c] = {pfma(G[0], a[0].x, pfma(G[1], a[1].x, G[2] * a[2].x)) - adv.x,
                        pfma(G[0], a[0].y, pfma(G[1], a[1].y, G[2] * a[2].y)) - adv.y};
            }
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) stp(X + (c * NV + ve) * RS + p, N[c]);
    }
    __syncthreads();

    // ---- forward transforms, kept modes, 1 / Mz
    if (f >= 3) return;
#pragma unroll
    for (int q = 0; q < K::NQ; ++q) {
        const int k1 = j + H * q;
        if (K::NQ * H > N1 && k1 >= N1) continue;
#pragma unroll
        for (int k = 0; k < H; ++k) o[q][k] = ldp(L + k1 + N1 * k);
        dft_dif<N2, -1>(o[q]);
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < K::NQ; ++q) {
        const int k1 = j + H * q;
        if (K::NQ * H > N1 && k1 >= N1) continue;
#pragma unroll
        for (int i = 0; i < H; ++i) stp(L + k1 * XS + i, pmul<false>(o[q][i], ldp(tw + k1 * H + i)));
    }
    __syncwarp();
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) v[k1] = ldp(L + k1 * XS + j);
    Pdft<N1, -1, T>::run(v);
    if (!live) return;
    Cv* out = (Cv*)g.N3 + (size_t)f * fs + ((size_t)y * E + e0 + vec) * NM;
    const T sc = (T)(1.0 / (double)MZ);
#pragma unroll
    for (int k2 = 0; k2 < N1; ++k2)
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int m = 2 * j + r + N2 * k2, q = m <= KZ ? m + KZ : (m >= MZ - KZ ? m - MZ + KZ : -1);
            if (q >= 0) out[q] = {(r ? v[k2].x.b : v[k2].x.a) * sc, (r ? v[k2].y.b : v[k2].y.a) * sc};
        }
}

template <typename T, int MZ>
void launch_lin_plane_t(const GroupView& g, cudaStream_t st) {
    constexpr int NV = LinCfg<MZ>::NV;
    k_lin_plane<T, MZ><<<dim3(g.ny, (g.E + NV - 1) / NV), LIN_THREADS, lin_plane_smem_bytes<T, MZ>(), st>>>(g);
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

// Sum of the threads' values over the cluster, in a fixed order, divided by d; the
// result in every thread.  inv is 1 / d, infinite for a subnormal d (vectors of norms
// below 1e-154), which then divides.  On the FP64 pipe an addition costs a warp 16
// cycles of its SM, so one warp adds up the CTA and one thread the cluster.
struct GsShared {
    double2 lane[GS_THREADS];
    double2 part, sum;
};
__device__ __forceinline__ double2 cluster_sum(double2 v, double inv, double d, GsShared& sh) {
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
        sh.sum = isinf(inv) ? make_double2(t.x / d, t.y / d) : make_double2(t.x * inv, t.y * inv);
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
        c = cluster_sum(s, gs_inv(g)[k], gs_sq(g)[k], sh);
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
        s = cluster_sum(s, 1.0, 1.0, sh);
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
#define DNS_CASE(a) allow_max_dynamic_smem(k_lin_plane<float, a>); allow_max_dynamic_smem(k_lin_plane<double, a>);
    DNS_CASE(16) DNS_CASE(32) DNS_CASE(48) DNS_CASE(64) DNS_CASE(128)
#undef DNS_CASE
}

}  // namespace dnsk
