// Physical-space stage of one sub-step as three launches that hand the planes
// on through L2 / HBM instead of keeping one plane on one SM or cluster (paper
// Sec. 3.1-3.2; the same mathematics as k_plane_lines.cu, both precisions):
//   k_ps_zinv  the spectral fields of every plane (u_i, d_y u_i, d_z u_i, or u_i
//              and the vorticity), inverse transforms along z, into column
//              storage COL[plane][field][z][n], n <= Kx;
//   k_ps_x     per line pair (rows p and p + Mz/2 packed as one complex line):
//              the inverse x transforms of all its fields (d_x u_i is u_i's
//              columns times i kx), the products, the forward x transforms;
//              N_i's kept columns overwrite u_i's rows, which only this line
//              pair reads; partial sums of u v and w v;
//   k_ps_zfwd  forward transforms along z, truncation, the plane means.
//
// Why: a 128 x 128 plane does not fit one SM, and over a thread-block cluster
// every transform is a cluster barrier apart from the next.  Line pairs need
// nothing of one another between the z transforms, so after the hand-over
// there is no barrier at all (a line pair belongs to N2 / 2 lanes of one
// warp), and any number of CTAs fits an SM.  The hand-over costs 9 + 3 columns
// written and read once each, 1.06 MB a plane at 128 x 128 in single precision.
//
// Line layout.  A transform of N = N1 N2 points is a four-step one.  For the x
// lines a thread t < N2 / 2 owns the residues t and N2 - t (0 and N2 / 2 for t
// = 0) modulo N2: a kept coefficient k and its mirror N - k belong to the same
// thread, so each is loaded once, and the two real rows of a packed line
// separate in registers after the forward transform.
#include "dns_internal.hpp"
#include "dft.cuh"
#include "ff.cuh"
#include "pairs.cuh"
#include <type_traits>

namespace dnsk {

namespace psp {

using namespace prs;
using dft::Split;

// COL holds complex pairs: the rows p and p + Mz/2 of one column side by side
// (re p, re p + Mz/2, im p, im p + Mz/2), [plane][field][p][n], n fastest.
__host__ __device__ inline int col_row(int nkx) { return (nkx + 1) & ~1; }
__host__ __device__ inline int col_fields(int rot) { return rot ? 6 : 9; }

template <typename T> struct Tab;
template <> struct Tab<float> {
    static __device__ __forceinline__ const float* kx(const GroupView& g) { return g.kxtf; }
    static __device__ __forceinline__ const float* kz(const GroupView& g) { return g.kztf; }
    static __device__ __forceinline__ const float* k2inv(const GroupView& g) { return g.k2invf; }
    static __device__ __forceinline__ const float2* twx(const GroupView& g) { return g.twxf; }
    static __device__ __forceinline__ const float2* twz(const GroupView& g) { return g.twzf; }
};
template <> struct Tab<double> {
    static __device__ __forceinline__ const double* kx(const GroupView& g) { return g.kxt; }
    static __device__ __forceinline__ const double* kz(const GroupView& g) { return g.kzt; }
    static __device__ __forceinline__ const double* k2inv(const GroupView& g) { return g.k2inv; }
    static __device__ __forceinline__ const double2* twx(const GroupView& g) { return g.twx; }
    static __device__ __forceinline__ const double2* twz(const GroupView& g) { return g.twz; }
};
template <typename T> struct Cv { T x, y; };               // one complex value

// ------------------------------------------------------------- z transforms

// Mz = N1 N2.  A CTA holds TN columns, the column index fastest over its
// threads (global and shared accesses are contiguous), and H = N2 / 2 thread
// rows.  Inverse: row j does the N1-point DFTs of the residues 2 j and 2 j + 1
// modulo N2 as one pair, then (decimation in time over that pair) N2-point DFTs
// whose lanes are the rows p and p + Mz/2; forward is the reverse.
template <int MZ> struct ZCfg {
    static constexpr int N1 = Split<MZ>::N1, N2 = Split<MZ>::N2, H = N2 / 2;
    static constexpr int NQ = (N1 + H - 1) / H;                // N2-point tasks per thread
    static constexpr int KZ = (MZ - 1) / 3;
};
constexpr int ZTHREADS = 128;                                 // most threads of a CTA
// columns of a CTA: the tiles of a plane as equal as they come within ZTHREADS
__host__ __device__ constexpr int ztiles(int nkx, int h) { return (nkx * h + ZTHREADS - 1) / ZTHREADS; }
__host__ __device__ constexpr int ztile(int nkx, int h) { return (nkx + ztiles(nkx, h) - 1) / ztiles(nkx, h); }
// threads of a CTA: at least one whole warp (rows j >= H idle)
__host__ __device__ constexpr int zthreads(int tn, int h) { return tn * h < 32 ? 32 : tn * h; }
// stride of the k1 rows of the exchange, = TN modulo 8: two neighbouring rows
// then fall in the 16-byte banks as if contiguous
template <int MZ>
__host__ __device__ inline int zrow_stride(int tn) {
    const int a = ZCfg<MZ>::H * tn;
    return a + ((tn - a) % 8 + 8) % 8;
}
template <int MZ, typename T>
size_t zsmem(int nkx, int buffers) {
    return sizeof(Pc<T>) * ((size_t)buffers * ZCfg<MZ>::N1 * zrow_stride<MZ>(ztile(nkx, ZCfg<MZ>::H)) + ZCfg<MZ>::N1 * ZCfg<MZ>::H) + 64;
}
// twiddles of the residue pairs (2 j, 2 j + 1): exp(-2 pi i k1 n2 / Mz)
template <typename T, int MZ>
__device__ __forceinline__ void fill_ztw(const GroupView& g, Pc<T>* tw) {
    typedef ZCfg<MZ> K;
    for (int i = threadIdx.x; i < K::N1 * K::H; i += blockDim.x) {
        const int k1 = i / K::H, j = i - k1 * K::H;
        const auto a = Tab<T>::twz(g)[2 * j * k1], b = Tab<T>::twz(g)[(2 * j + 1) * k1];
        tw[i] = {pr((T)a.x, (T)b.x), pr((T)a.y, (T)b.y)};
    }
}

// The fields in three groups by the inputs they share (blockIdx.z): a thread
// loads its modes' inputs once, all loads in flight together, and transforms
// the group's fields from registers.  Advective: u, w, u_z, w_z from Dv, eta;
// v, v_z, v_y from v, Dv; u_y, w_y from D2v, Deta.  Rotational: u, w; v,
// omega_y = eta; omega_x = d_y w - d_z v, omega_z = d_x v - d_y u.
template <typename T, int MZ, bool ROT>
__global__ void __launch_bounds__(ZTHREADS, sizeof(T) == 4 ? 4 : 2)
k_ps_zinv(GroupView g, const double* __restrict__ Ucur, const double* __restrict__ Wcur) {
    typedef ZCfg<MZ> K;
    typedef Cv<T> C;
    constexpr int N1 = K::N1, N2 = K::N2, H = K::H, KZ = K::KZ, HP = MZ / 2;
    constexpr int NF = ROT ? 6 : 9;
    extern __shared__ __align__(16) unsigned char smem[];
    const int nkx = g.nkx, TN = ztile(nkx, H), KS = zrow_stride<MZ>(TN), NS = col_row(nkx);
    double* red = (double*)smem;
    Pc<T>* tw = (Pc<T>*)(smem + 64);
    Pc<T>* X = tw + N1 * H;                                     // two exchange buffers
    const int tid = threadIdx.x, j = tid / TN, nl = tid - j * TN;
    const int pe = blockIdx.x, y = pe / g.E, e = pe - y * g.E, n = blockIdx.y * TN + nl;
    const size_t fs = (size_t)g.ny * g.E * g.nmodes;
    const bool row = j < H, act = row && n < nkx;
    if (!DNS_CK(g.status, y < g.ny && MZ == g.mz, CK_PLANE_SPLIT, pe)) return;
    const C* __restrict__ P = (const C*)g.P5 + (size_t)pe * g.nmodes + (act ? n : 0);
    Pc<T>* __restrict__ col = (Pc<T>*)g.COL + (size_t)pe * NF * HP * NS + n;

    auto group = [&](auto gc) {
        constexpr int G = decltype(gc)::value;
        constexpr bool DY = G == 2;                             // needs the mean's y-derivatives
        constexpr int NI = ROT && G == 2 ? 3 : 2;
        constexpr int in0 = G == 0 ? 1 : G == 1 ? 0 : 2, in1 = G == 0 ? 3 : G == 1 ? (ROT ? 3 : 1) : 4;
        Pc<T> in[NI][N1];
        Pr<T> kz[N1], ki[N1];
        const T kx = act ? Tab<T>::kx(g)[n] : (T)0;
        const T* __restrict__ kzt = Tab<T>::kz(g);
        const T* __restrict__ k2i = Tab<T>::k2inv(g) + (act ? n : 0);
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) {
            const int z0 = N2 * n1;
            if (z0 > KZ && z0 + N2 - 1 < MZ - KZ) continue;      // wholly padding
            C p[NI][2];
            T kk[2], kv[2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int z = z0 + 2 * j + r;
                const bool lo = z <= KZ, keep = act && (lo || z >= MZ - KZ);
                const int mi = lo ? z + KZ : z - MZ + KZ;
                const size_t m = (size_t)mi * nkx;
#pragma unroll
                for (int i = 0; i < NI; ++i) p[i][r] = {(T)0, (T)0};
                kk[r] = kv[r] = (T)0;
                if (keep) {
                    p[0][r] = P[(size_t)in0 * fs + m];
                    p[1][r] = P[(size_t)in1 * fs + m];
                    if (NI == 3) p[NI - 1][r] = P[m];
                    kv[r] = kzt[mi];
                    if (G != 1) kk[r] = k2i[m];
                }
            }
#pragma unroll
            for (int i = 0; i < NI; ++i) in[i][n1] = {pr(p[i][0].x, p[i][1].x), pr(p[i][0].y, p[i][1].y)};
            kz[n1] = pr(kv[0], kv[1]);
            ki[n1] = pr(kk[0], kk[1]);
        }
        fill_ztw<T, MZ>(g, tw);
        T mu = 0, mw = 0;                                        // the (0, 0) mode of the u and w fields
        const bool mean = j == 0 && n == 0;
        if (G != 1 && blockIdx.y == 0) {
            const double *Ue = Ucur + (size_t)e * g.my, *We = Wcur + (size_t)e * g.my;
            if (DY) mean_dy_row(g.D1, Ue, We, g.my, y + 1, red);
            else { mu = (T)Ue[y + 1]; mw = (T)We[y + 1]; }
        }
        __syncthreads();
        if (DY && blockIdx.y == 0) { mu = (T)red[0]; mw = (T)red[1]; }
        const Pr<T> kxp = dup(kx);
        // u = i (kx a - kz b) / k^2, w = i (kz a + kx b) / k^2
        auto u_of = [&](int i, bool w) -> Pc<T> {
            const Pc<T> a = in[0][i], b = in[1][i];
            Pc<T> r;
            if (!w) r = {pfma(kz[i], b.y, pneg(kxp * a.y)) * ki[i], (kxp * a.x - kz[i] * b.x) * ki[i]};
            else r = {pneg(pfma(kz[i], a.y, kxp * b.y) * ki[i]), pfma(kz[i], a.x, kxp * b.x) * ki[i]};
            if (i == 0 && mean) { r.x.a = w ? mw : mu; r.y.a = (T)0; }
            return r;
        };
        auto ik = [&](Pr<T> k, Pc<T> r) -> Pc<T> { return {pneg(k * r.y), k * r.x}; };
        // field number c of the group: its place in COL and its value at slot i
        constexpr int NC = ROT ? 2 : G == 0 ? 4 : G == 1 ? 3 : 2;
        auto place = [&](int c) {
            if (ROT) return G == 0 ? 2 * c : G == 1 ? 1 + 3 * c : 3 + 2 * c;
            return G == 0 ? (c < 2 ? 2 * c : 2 * c + 2) : G == 1 ? (c == 0 ? 1 : c == 1 ? 7 : 4) : 3 + 2 * c;
        };
        auto value = [&](int c, int i) -> Pc<T> {
            if (G == 0) return c < 2 ? u_of(i, c == 1) : ik(kz[i], u_of(i, c == 3));
            if (G == 1) return c == 0 ? in[0][i] : ROT || c == 2 ? in[1][i] : ik(kz[i], in[0][i]);
            if (!ROT) return u_of(i, c == 1);
            return c == 0 ? u_of(i, true) - ik(kz[i], in[NI - 1][i]) : ik(kxp, in[NI - 1][i]) - u_of(i, false);
        };
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            Pc<T> v[N1];
#pragma unroll
            for (int i = 0; i < N1; ++i) {
                const int z0 = N2 * i;
                if (z0 > KZ && z0 + N2 - 1 < MZ - KZ) v[i] = {dup((T)0), dup((T)0)};
                else v[i] = value(c, i);
            }
            Pc<T>* Xb = X + (c & 1) * N1 * KS;
            Pc<T>* x = Xb + j * TN + nl;
            if (row) {
                pdft_padded<N1, +1>(v);
#pragma unroll
                for (int k1 = 0; k1 < N1; ++k1)
                    stp(x + k1 * KS, k1 == 0 ? v[0] : pmul<true>(v[k1], ldp(tw + k1 * H + j)));
            }
            __syncthreads();
#pragma unroll
            for (int q = 0; q < K::NQ; ++q) {
                const int k1 = j + H * q;
                if (!row || (K::NQ * H > N1 && k1 >= N1)) continue;
                const Pc<T>* xr = Xb + k1 * KS + nl;
                Pc<T> o[H];
#pragma unroll
                for (int i = 0; i < H; ++i) o[i] = ldp(xr + i * TN);
                dft_dit<N2, +1>(o);
                if (act) {
                    Pc<T>* t = col + ((size_t)place(c) * HP + k1) * NS;
#pragma unroll
                    for (int k = 0; k < H; ++k) stp(t + (size_t)(N1 * k) * NS, o[k]);
                }
            }
        }
    };
    if (blockIdx.z == 0) group(std::integral_constant<int, 0>());
    else if (blockIdx.z == 1) group(std::integral_constant<int, 1>());
    else group(std::integral_constant<int, 2>());
}

// One field (blockIdx.z) of one plane and column tile.
template <typename T, int MZ>
__global__ void __launch_bounds__(ZTHREADS)
k_ps_zfwd(GroupView g, int parts) {
    typedef ZCfg<MZ> K;
    constexpr int N1 = K::N1, N2 = K::N2, H = K::H, KZ = K::KZ, HP = MZ / 2;
    extern __shared__ __align__(16) unsigned char smem[];
    const int nkx = g.nkx, TN = ztile(nkx, H), KS = zrow_stride<MZ>(TN), NS = col_row(nkx);
    Pc<T>* tw = (Pc<T>*)(smem + 64);
    Pc<T>* X = tw + N1 * H;
    const int tid = threadIdx.x, j = tid / TN, nl = tid - j * TN;
    const int pe = blockIdx.x, n = blockIdx.y * TN + nl, f = blockIdx.z;
    const bool row = j < H, act = row && n < nkx;
    if (!DNS_CK(g.status, pe < g.ny * g.E && MZ == g.mz, CK_PLANE_SPLIT, pe)) return;
    if (f == 0 && blockIdx.y == 0 && tid == 0) {
        // plane means <uv>, <wv>: the line pairs' partial sums in a fixed order
        const double2* p = g.psum + (size_t)pe * parts;
        double a = 0.0, b = 0.0;
        for (int i = 0; i < parts; ++i) { a += p[i].x; b += p[i].y; }
        const int y = pe / g.E, e = pe - y * g.E;
        const double pts = (double)g.mx * MZ;
        g.uv[(size_t)e * g.my + y + 1] = a / pts;
        g.wv[(size_t)e * g.my + y + 1] = b / pts;
    }
    fill_ztw<T, MZ>(g, tw);
    const Pc<T>* __restrict__ col =
        (const Pc<T>*)g.COL + ((size_t)pe * col_fields(g.rot) + f) * HP * NS + (act ? n : 0);
    Pc<T> v[K::NQ][H];
#pragma unroll
    for (int q = 0; q < K::NQ; ++q) {
        const int k1 = j + H * q;
        if (!row || (K::NQ * H > N1 && k1 >= N1)) continue;
#pragma unroll
        for (int k = 0; k < H; ++k) v[q][k] = ldp(col + (size_t)(k1 + N1 * k) * NS);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < K::NQ; ++q) {
        const int k1 = j + H * q;
        if (!row || (K::NQ * H > N1 && k1 >= N1)) continue;
        dft_dif<N2, -1>(v[q]);
        Pc<T>* x = X + k1 * KS + nl;
#pragma unroll
        for (int i = 0; i < H; ++i) stp(x + i * TN, pmul<false>(v[q][i], ldp(tw + k1 * H + i)));
    }
    __syncthreads();
    if (!act) return;
    Pc<T> o[N1];
    const Pc<T>* x = X + j * TN + nl;
#pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) o[k1] = ldp(x + k1 * KS);
    Pdft<N1, -1, T>::run(o);
    Cv<T>* out = (Cv<T>*)g.N3 + (size_t)f * g.ny * g.E * g.nmodes + (size_t)pe * g.nmodes + n;
    const T sz = (T)1 / (T)MZ;
#pragma unroll
    for (int k2 = 0; k2 < N1; ++k2) {
        const int m0 = 2 * j + N2 * k2;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int m = m0 + r, mi = m <= KZ ? m + KZ : (m >= MZ - KZ ? m - MZ + KZ : -1);
            if (mi >= 0)
                out[(size_t)mi * nkx] = {(r ? o[k2].x.b : o[k2].x.a) * sz, (r ? o[k2].y.b : o[k2].y.a) * sz};
        }
    }
}

// ------------------------------------------------- x transforms and products

template <int MX> struct XCfg {
    static constexpr int N1 = Split<MX>::N1, N2 = Split<MX>::N2, H = N2 / 2;
    static constexpr int L = 32 / H;                          // line pairs per warp, H lanes each
    static constexpr int NQ = (N1 + H - 1) / H;               // N2-point tasks per lane
    static constexpr int KX = (MX - 1) / 3;
    static constexpr int NL = KX / N2 + 1;                    // kept coefficients per residue
    static constexpr int XS = H + 1, XF = N1 + 1;             // exchange row strides (complex pairs)
    // line stride: for H = 4 two lines share an eight-lane access and must lie
    // four 16-byte banks apart
    static constexpr int R0 = N1 * XS > H * XF ? N1 * XS : H * XF;
    static constexpr int RS = H == 4 ? R0 + ((4 - R0 % 8) + 8) % 8 : R0;
    static constexpr int PH = NQ * H;                         // point pairs per lane
    static constexpr bool RAGGED = H == 2;                    // a warp may hold more line pairs than a plane has
    static_assert(2 * NL <= N1, "kept coefficients and their mirrors fill distinct slots");
};
constexpr int XWARPS = 4;   // most warps of a CTA
// complex pairs of shared memory per warp: its exchange and its lanes' own
// copies of the fields the products need (u, v, w; rotational also omega_x, omega_y)
template <int MX> constexpr int xwarp_pairs(bool rot) {
    return XCfg<MX>::L * XCfg<MX>::RS + (rot ? 5 : 3) * XCfg<MX>::PH * 32;
}
template <int MX, typename T>
size_t xsmem(int warps, bool rot) {
    return sizeof(Pc<T>) * ((size_t)warps * xwarp_pairs<MX>(rot) + XCfg<MX>::N1 * XCfg<MX>::XS) + 512;
}

template <typename T, int MX, bool ROT>
__global__ void __launch_bounds__(32 * XWARPS, sizeof(T) == 4 ? 3 : 1)
k_ps_x(GroupView g) {
    typedef XCfg<MX> K;
    constexpr int N1 = K::N1, N2 = K::N2, H = K::H, NQ = K::NQ, KX = K::KX, NL = K::NL;
    constexpr int XS = K::XS, XF = K::XF, PH = K::PH;
    constexpr int NF = ROT ? 6 : 9;
    extern __shared__ __align__(16) unsigned char smem[];
    Pc<T>* tw = (Pc<T>*)(smem + 512);                          // [k1][t]: the residue pair (t, nb)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, t = lane & (H - 1);
    Pc<T>* VEL = tw + N1 * XS + warp * xwarp_pairs<MX>(ROT) + lane;   // this lane's points, stride 32
    Pc<T>* X = tw + N1 * XS + warp * xwarp_pairs<MX>(ROT) + (ROT ? 5 : 3) * PH * 32 + (lane / H) * K::RS;
    const int pe = blockIdx.x, HP = g.mz / 2, NS = col_row(K::KX + 1);
    const int p = (blockIdx.y * (blockDim.x >> 5) + warp) * K::L + lane / H;
    const bool act = !K::RAGGED || p < HP;
    if (!DNS_CK(g.status, pe < g.ny * g.E && (p < HP || K::RAGGED) && MX == g.mx, CK_PLANE_SPLIT, pe)) return;
    for (int i = tid; i < N1 * H; i += blockDim.x) {
        const int k1 = i / H, j = i - k1 * H;
        const auto a = Tab<T>::twx(g)[j * k1], b = Tab<T>::twx(g)[(j ? N2 - j : H) * k1];
        tw[k1 * XS + j] = {pr((T)a.x, (T)b.x), pr((T)a.y, (T)b.y)};
    }
    __syncthreads();
    const int nb = t ? N2 - t : H;                             // second residue of this lane
    Pc<T>* row0 = (Pc<T>*)g.COL + ((size_t)pe * NF * HP + p) * NS;
    const size_t fstr = (size_t)HP * NS;
    T kxa[NL], kxb[NL];
#pragma unroll
    for (int j = 0; j < NL; ++j) {
        const int ka = N2 * j + t, kb = N2 * j + nb;
        kxa[j] = ka <= KX ? Tab<T>::kx(g)[ka] : (T)0;
        kxb[j] = kb <= KX ? Tab<T>::kx(g)[kb] : (T)0;
    }
    // this lane's twiddles of the inverse transforms: in registers in single
    // precision, whose shared-memory bandwidth is what bounds this kernel
    constexpr bool TWREG = sizeof(T) == 4;
    Pc<T> wt[TWREG ? N1 : 1];
    if constexpr (TWREG) {
#pragma unroll
        for (int k1 = 1; k1 < N1; ++k1) wt[k1] = ldp(tw + k1 * XS + t);
    }
    // kept coefficients of the two rows at this lane's residues
    Pc<T> A[NL], B[NL];
    auto load = [&](int f) {
        const Pc<T>* r = row0 + f * fstr;
#pragma unroll
        for (int j = 0; j < NL; ++j) {
            const int ka = N2 * j + t, kb = N2 * j + nb;
            A[j] = B[j] = {dup((T)0), dup((T)0)};
            if (act && ka <= KX) A[j] = ldp(r + ka);
            if (act && kb <= KX) B[j] = ldp(r + kb);
        }
    };
    // the loaded line pair (times i kx for dx) inverse transformed: o[q H + m] holds
    // the points x = (t + H q) + N1 (2 m) and N1 further, row p in .x and row
    // p + Mz/2 in .y; the coefficients of field `next` are on their way meanwhile
    auto xinv = [&](bool dx, int next, Pc<T>* o) {
        if (dx) {
#pragma unroll
            for (int j = 0; j < NL; ++j) {
                A[j] = {A[j].y * dup(-kxa[j]), A[j].x * dup(kxa[j])};
                B[j] = {B[j].y * dup(-kxb[j]), B[j].x * dup(kxb[j])};
            }
        }
        Pc<T> v[N1];
#pragma unroll
        for (int n1 = 0; n1 < N1; ++n1) v[n1] = {dup((T)0), dup((T)0)};
#pragma unroll
        for (int j = 0; j < NL; ++j) {
            // rows a, b packed: a + i b at k, conj(a) + i conj(b) at N - k
            v[j].x = pr(A[j].x.a - A[j].y.b, B[j].x.a - B[j].y.b);
            v[j].y = pr(A[j].y.a + A[j].x.b, B[j].y.a + B[j].x.b);
            const T mxa = A[j].x.a + A[j].y.b, mya = A[j].x.b - A[j].y.a;
            const T mxb = B[j].x.a + B[j].y.b, myb = B[j].x.b - B[j].y.a;
            T mx0 = 0, my0 = 0;                                // residue 0: its own next coefficient's mirror
            if (j + 1 < NL) { mx0 = A[j + 1].x.a + A[j + 1].y.b; my0 = A[j + 1].x.b - A[j + 1].y.a; }
            v[N1 - 1 - j].x = pr(t ? mxb : mx0, t ? mxa : mxb);
            v[N1 - 1 - j].y = pr(t ? myb : my0, t ? mya : myb);
        }
        if (t == 0) { v[0].x.a = A[0].x.a; v[0].y.a = A[0].x.b; }   // k = 0: the Hermitian part
        if (next >= 0) load(next);
        pdft_padded<N1, +1>(v);
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1)
            stp(X + k1 * XS + t, k1 == 0 ? v[0] : pmul<true>(v[k1], TWREG ? wt[TWREG ? k1 : 0] : ldp(tw + k1 * XS + t)));
        __syncwarp();
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int k1 = t + H * q;
            Pc<T>* oq = o + q * H;
            if (NQ * H > N1 && k1 >= N1) {
#pragma unroll
                for (int m = 0; m < H; ++m) oq[m] = {dup((T)0), dup((T)0)};
                continue;
            }
            Pc<T> r[H];
#pragma unroll
            for (int i = 0; i < H; ++i) r[i] = ldp(X + k1 * XS + i);
            // residue pairs (i, N2 - i), (0, H)  ->  (i, i + H)
#pragma unroll
            for (int i = 0; i < H; ++i) {
                const Pc<T> c = r[(H - i) % H];
                oq[i] = {pr(r[i].x.a, c.x.b), pr(r[i].y.a, c.y.b)};
            }
            dft_dif<N2, +1>(oq);
        }
        __syncwarp();
    };
    // forward transform of the products acc (laid out as o), the two rows
    // separated, the kept columns over the rows of field i
    const T sx = (T)0.5 / (T)MX;
    auto xfwd = [&](int f, Pc<T>* acc) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
            const int k1 = t + H * q;
            if (NQ * H > N1 && k1 >= N1) continue;
            Pc<T>* a = acc + q * H;
            dft_dit<N2, -1>(a);
#pragma unroll
            for (int i = 0; i < H; ++i) {
                const Pc<T> c = a[(H - i) % H];
                const Pc<T> w = {pr(a[i].x.a, c.x.b), pr(a[i].y.a, c.y.b)};
                stp(X + i * XF + k1, pmul<false>(w, ldp(tw + k1 * XS + i)));
            }
        }
        __syncwarp();
        Pc<T> v[N1];
#pragma unroll
        for (int k1 = 0; k1 < N1; ++k1) v[k1] = ldp(X + t * XF + k1);
        Pdft<N1, -1, T>::run(v);
        Pc<T>* r = row0 + f * fstr;
#pragma unroll
        for (int j = 0; j < NL; ++j) {
            const int ka = N2 * j + t, kb = N2 * j + nb;
            const Pc<T> u = v[N1 - 1 - j], s = v[(N1 - j) % N1];
            const T wx = v[j].x.a, wy = v[j].y.a, cx = t ? u.x.b : s.x.a, cy = t ? u.y.b : s.y.a;
            if (act && ka <= KX) stp(r + ka, Pc<T>{pr((wx + cx) * sx, (wy + cy) * sx), pr((wy - cy) * sx, (cx - wx) * sx)});
            const T zx = v[j].x.b, zy = v[j].y.b, dx = t ? u.x.a : u.x.b, dy = t ? u.y.a : u.y.b;
            if (act && kb <= KX) stp(r + kb, Pc<T>{pr((zx + dx) * sx, (zy + dy) * sx), pr((zy - dy) * sx, (dx - zx) * sx)});
        }
        __syncwarp();
    };

    // sums of u v and w v over this lane's points (float-float in single precision)
    Pr<T> s1h = dup((T)0), s1l = s1h, s2h = s1h, s2l = s1h;
    auto add_prod = [&](Pr<T>& h, Pr<T>& l, Pr<T> a, Pr<T> b) {
        if constexpr (std::is_same<T, float>::value) {
            // ff_add_prod on both lanes
            const Pr<T> q = a * b, e0 = pfma(a, b, pneg(q));
            const Pr<T> s = h + q, z = s - h;
            const Pr<T> e = (h - (s - z)) + (q - z);
            h = s;
            l = l + (e + e0);
        } else {
            h = pfma(a, b, h);
        }
    };
    load(0);
    Pc<T> o[PH];
#pragma unroll 1
    for (int f = 0; f < 3; ++f) {
        xinv(false, f < 2 ? f + 1 : ROT ? 3 : 0, o);
#pragma unroll
        for (int m = 0; m < PH; ++m) {
            stp(VEL + (f * PH + m) * 32, o[m]);
            // the idle lanes' points of a ragged N1 are zero
            if (f == 1) {
                const Pc<T> u = ldp(VEL + m * 32);
                add_prod(s1h, s1l, u.x, o[m].x);
                add_prod(s1h, s1l, u.y, o[m].y);
            }
            if (f == 2) {
                const Pc<T> u = ldp(VEL + (PH + m) * 32);
                add_prod(s2h, s2l, o[m].x, u.x);
                add_prod(s2h, s2l, o[m].y, u.y);
            }
        }
    }
    if constexpr (!ROT) {
        // N_i = u d_x u_i + v d_y u_i + w d_z u_i
        Pc<T> acc[PH];
#pragma unroll 1
        for (int s = 0; s < 9; ++s) {
            const int i = s / 3, j = s - 3 * i;
            const int next = s == 8 ? -1 : j == 2 ? i + 1 : 3 * (j + 1) + i;
            xinv(j == 0, next, o);
            if (j == 0) {
#pragma unroll
                for (int m = 0; m < PH; ++m) acc[m] = {dup((T)0), dup((T)0)};
            }
#pragma unroll
            for (int m = 0; m < PH; ++m) {
                const Pc<T> u = ldp(VEL + (j * PH + m) * 32);
                acc[m] = {pfma(u.x, o[m].x, acc[m].x), pfma(u.y, o[m].y, acc[m].y)};
            }
            if (j == 2) xfwd(i, acc);
        }
    } else {
        // N = omega x u: omega_x, omega_y kept beside u, v, w; with omega_z the
        // products, over u, v, w
#pragma unroll 1
        for (int f = 3; f < 6; ++f) {
            xinv(false, f < 5 ? f + 1 : -1, o);
            if (f < 5) {
#pragma unroll
                for (int m = 0; m < PH; ++m) stp(VEL + (f * PH + m) * 32, o[m]);
            }
        }
#pragma unroll
        for (int m = 0; m < PH; ++m) {
            const Pc<T> u = ldp(VEL + m * 32), v = ldp(VEL + (PH + m) * 32), w = ldp(VEL + (2 * PH + m) * 32);
            const Pc<T> ox = ldp(VEL + (3 * PH + m) * 32), oy = ldp(VEL + (4 * PH + m) * 32), oz = o[m];
            stp(VEL + m * 32, Pc<T>{oy.x * w.x - oz.x * v.x, oy.y * w.y - oz.y * v.y});
            stp(VEL + (PH + m) * 32, Pc<T>{oz.x * u.x - ox.x * w.x, oz.y * u.y - ox.y * w.y});
            stp(VEL + (2 * PH + m) * 32, Pc<T>{ox.x * v.x - oy.x * u.x, ox.y * v.y - oy.y * u.y});
        }
#pragma unroll 1
        for (int i = 0; i < 3; ++i) {
#pragma unroll
            for (int m = 0; m < PH; ++m) o[m] = ldp(VEL + (i * PH + m) * 32);
            xfwd(i, o);
        }
    }
    double suv = 0.0, swv = 0.0;
    if constexpr (std::is_same<T, float>::value) {
        ff_add(s1h.a, s1l.a, s1h.b, s1l.b);
        ff_add(s2h.a, s2l.a, s2h.b, s2l.b);
        ff_block_sum2(s1h.a, s1l.a, s2h.a, s2l.a, (float*)smem, &suv, &swv);
    } else {
        suv = block_sum(s1h.a + s1h.b, (double*)smem);
        swv = block_sum(s2h.a + s2h.b, (double*)smem);
    }
    if (tid == 0) g.psum[(size_t)pe * gridDim.y + blockIdx.y] = make_double2(suv, swv);
}

// warps of a k_ps_x CTA: the most, up to XWARPS, that divide the plane's warps
// (0: line pairs the lanes of a warp do not divide)
template <int MX> constexpr int xplane_warps(int mz) {
    return (mz / 2 + XCfg<MX>::L - 1) / XCfg<MX>::L;
}
template <int MX>
int xwarps(int mz) {
    if (!XCfg<MX>::RAGGED && mz / 2 % XCfg<MX>::L) return 0;
    for (int w = XWARPS; w > 0; --w)
        if (xplane_warps<MX>(mz) % w == 0) return w;
    return 0;
}

template <typename T, int MX, bool ROT>
int launch_x(const GroupView& g, cudaStream_t st) {
    const int w = xwarps<MX>(g.mz), parts = xplane_warps<MX>(g.mz) / w;
    k_ps_x<T, MX, ROT><<<dim3(g.ny * g.E, parts), 32 * w, xsmem<MX, T>(w, ROT), st>>>(g);
    return parts;
}

template <typename T, int MZ>
void launch_zinv(const GroupView& g, const double* U, const double* W, cudaStream_t st) {
    const int tn = ztile(g.nkx, ZCfg<MZ>::H);
    const dim3 grid(g.ny * g.E, (g.nkx + tn - 1) / tn, 3);
    if (g.rot) k_ps_zinv<T, MZ, true><<<grid, zthreads(tn, ZCfg<MZ>::H), zsmem<MZ, T>(g.nkx, 2), st>>>(g, U, W);
    else k_ps_zinv<T, MZ, false><<<grid, zthreads(tn, ZCfg<MZ>::H), zsmem<MZ, T>(g.nkx, 2), st>>>(g, U, W);
}
template <typename T, int MZ>
void launch_zfwd(const GroupView& g, int parts, cudaStream_t st) {
    const int tn = ztile(g.nkx, ZCfg<MZ>::H);
    const dim3 grid(g.ny * g.E, (g.nkx + tn - 1) / tn, 3);
    k_ps_zfwd<T, MZ><<<grid, zthreads(tn, ZCfg<MZ>::H), zsmem<MZ, T>(g.nkx, 1), st>>>(g, parts);
}

}  // namespace psp

#define DNS_SPLIT_LENGTHS(X) X(16) X(32) X(48) X(64) X(128)

bool plane_split_supported(const GroupView& g) {
    if (g.lin || (g.rot && (g.mx == 128 || g.mz == 128))) return false;
    bool x = false, z = false;
#define DNS_CASE(a) if (g.mx == a) x = psp::xwarps<a>(g.mz) > 0; if (g.mz == a) z = true;
    DNS_SPLIT_LENGTHS(DNS_CASE)
#undef DNS_CASE
    return x && z;
}

size_t plane_split_col_bytes(const GroupView& g, bool fp64) {
    return (size_t)g.ny * g.E * psp::col_fields(g.rot) * (g.mz / 2) * psp::col_row(g.nkx) * (fp64 ? 32 : 16);
}
// one partial sum per line pair at most
size_t plane_split_psum_bytes(const GroupView& g) { return (size_t)g.ny * g.E * (g.mz / 2) * sizeof(double2); }

template <typename T>
static void launch_split_t(const GroupView& g, const double* U, const double* W, cudaStream_t st) {
    int parts = 0;
#define DNS_CASE(a) if (g.mz == a) psp::launch_zinv<T, a>(g, U, W, st);
    DNS_SPLIT_LENGTHS(DNS_CASE)
#undef DNS_CASE
#define DNS_CASE(a) \
    if (g.mx == a) parts = g.rot ? psp::launch_x<T, a, true>(g, st) : psp::launch_x<T, a, false>(g, st);
    DNS_SPLIT_LENGTHS(DNS_CASE)
#undef DNS_CASE
#define DNS_CASE(a) if (g.mz == a) psp::launch_zfwd<T, a>(g, parts, st);
    DNS_SPLIT_LENGTHS(DNS_CASE)
#undef DNS_CASE
}

void launch_plane_split(const GroupView& g, bool fp64, const double* U, const double* W, cudaStream_t st) {
    if (fp64) launch_split_t<double>(g, U, W, st);
    else launch_split_t<float>(g, U, W, st);
}

void set_attributes_plane_split() {
#define DNS_CASE(a)                                       \
    allow_max_dynamic_smem(psp::k_ps_x<float, a, false>); \
    allow_max_dynamic_smem(psp::k_ps_x<float, a, true>);  \
    allow_max_dynamic_smem(psp::k_ps_x<double, a, false>);\
    allow_max_dynamic_smem(psp::k_ps_x<double, a, true>); \
    allow_max_dynamic_smem(psp::k_ps_zinv<float, a, false>); \
    allow_max_dynamic_smem(psp::k_ps_zinv<float, a, true>);  \
    allow_max_dynamic_smem(psp::k_ps_zinv<double, a, false>);\
    allow_max_dynamic_smem(psp::k_ps_zinv<double, a, true>); \
    allow_max_dynamic_smem(psp::k_ps_zfwd<float, a>);     \
    allow_max_dynamic_smem(psp::k_ps_zfwd<double, a>);
    DNS_SPLIT_LENGTHS(DNS_CASE)
#undef DNS_CASE
}

}  // namespace dnsk
