// The per-wavenumber kernels of the FP64 path, every product in parity blocks
// (eo.cuh): k_yderiv64 (Dv, D2v, D eta and the H -> P relayout, Sec. 3.1),
// k_forcing64 (Eqs. Dv, eta and the RK3 combination) and k_helm64 (Eqs. CN1,
// CN2: M_h x_t + P_h F~ per wavenumber pair, with M_1 x_t computed once and
// reused by the third sub-step).
//
// What bounds them is the FP64 pipe: one warp instruction takes an SM about 16
// cycles, so operand loads hide behind it and what counts is the number of
// multiply-adds and that no SM is without work.  On the symmetric Chebyshev
// grid M, P and D2 map the even part of a column to the even part and the odd to
// the odd, D1 swaps them: half the multiply-adds of the full matrices, and
// half the operator bytes.  Column tiles shrink until the grid covers the chip
// twice (a member count that is no multiple of the tile costs nothing: the
// tile takes min(E, 4) members and fills up with modes).
// Microseconds a launch, full matrices -> here: 64x65x64 x 4 y-derivatives 203 ->
// 111, forcing 93 -> 55, apply 254 -> 112; 128x97x128 x 1 1701 -> 240, 651 -> 106,
// 1159 -> 241 (there the full matrices did not fit shared memory).
#include "dns_internal.hpp"
#include "eo.cuh"
#include "mbar.cuh"
#include "mean.cuh"

namespace dnsk {

namespace s64 {

using spc::eo_rows;
using spc::EoRows;

constexpr int THREADS = 256;

struct Tile {
    int QT, EBT, NC;   // QT modes x EBT members
};
__host__ __device__ inline Tile tile_of(int E, int nm) {
    Tile t;
    t.EBT = E < 4 ? E : 4;
    for (int cap = 16;; cap /= 2) {
        t.QT = cap / t.EBT > 0 ? cap / t.EBT : 1;
        t.NC = t.QT * t.EBT;
        const long long ctas = (long long)((nm + t.QT - 1) / t.QT) * ((E + t.EBT - 1) / t.EBT);
        if (cap <= 4 || ctas >= 2 * 152) return t;
    }
}

__device__ __forceinline__ double2 dadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 dsub(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ void dfma(double2& a, double b, double2 x) { a.x = fma(b, x.x, a.x); a.y = fma(b, x.y, a.y); }
// natural row from its pair-row's even and odd output parts (row 0: p, 1: Ny-1-p)
__device__ __forceinline__ double2 row_of(double2 e, double2 o, bool pair, int row) {
    if (!pair) return e;
    return row ? make_double2(0.5 * (e.x - o.x), 0.5 * (e.y - o.y)) : make_double2(0.5 * (e.x + o.x), 0.5 * (e.y + o.y));
}

__global__ void __launch_bounds__(THREADS) k_yderiv64(GroupView g, const double2* __restrict__ V,
                                                      const double2* __restrict__ H, double2* __restrict__ P,
                                                      int sprev) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int Ny = g.ny, E = g.E, NM = g.nmodes;
    const Tile T = tile_of(E, NM);
    if (mean_finish_rows(g, sprev, (E + T.EBT - 1) / T.EBT, sm)) return;
    const int NE = (Ny + 1) / 2, NO = Ny / 2, RP = spc::eo_rp(Ny), NC = T.NC;
    const int q0 = blockIdx.x * T.QT, e0 = blockIdx.y * T.EBT;
    double2* XV = (double2*)sm;              // parity parts of v [Ny][NC]
    double2* XE = XV + Ny * NC;              // of eta
    // the tile in H order [q][y][e]
    const int per = NE * T.EBT;
    for (int i = threadIdx.x; i < T.QT * per; i += THREADS) {
        const int qq = i / per, r = i - qq * per, p = r / T.EBT, el = r - p * T.EBT;
        const int q = q0 + qq, e = e0 + el, c = el * T.QT + qq;
        const EoRows R = eo_rows(p, Ny);
        double2 a[2], b[2];
        a[0] = a[1] = b[0] = b[1] = make_double2(0.0, 0.0);
        if (q < NM && e < E) {
            const size_t h0 = ((size_t)q * Ny + R.y0) * E + e, h1 = ((size_t)q * Ny + R.y1) * E + e;
            a[0] = V[h0];
            b[0] = H[h0];
            if (R.pair) { a[1] = V[h1]; b[1] = H[h1]; }
        }
        XV[p * NC + c] = dadd(a[0], a[1]);
        XE[p * NC + c] = dadd(b[0], b[1]);
        if (R.pair) {
            XV[(NE + p) * NC + c] = dsub(a[0], a[1]);
            XE[(NE + p) * NC + c] = dsub(b[0], b[1]);
        }
    }
    __syncthreads();
    const size_t fs = (size_t)Ny * E * NM;
    const double* __restrict__ D1e = g.D1EO64;                       // even output rows (contract the odd part)
    const double* __restrict__ D1o = D1e + (size_t)NO * RP;          // odd output rows
    const double* __restrict__ D2e = g.D2EO64;
    const double* __restrict__ D2o = D2e + (size_t)NE * RP;
    for (int m = threadIdx.x; m < NE * NC; m += THREADS) {
        const int p = m / NC, j = m - p * NC;                        // consecutive threads: consecutive q
        const int el = j / T.QT, q = q0 + j - el * T.QT, e = e0 + el;
        if (q >= NM || e >= E) continue;
        const double2 z = make_double2(0.0, 0.0);
        double2 ve = z, vo = z, we = z, wo = z, he = z, ho = z;      // Dv, D2v, D eta: even and odd rows
#pragma unroll 4
        for (int k = 0; k < NE; ++k) {
            const double b1 = D1o[k * RP + p], b2 = D2e[k * RP + p];
            const double2 x = XV[k * NC + j], h = XE[k * NC + j];
            dfma(vo, b1, x);
            dfma(we, b2, x);
            dfma(ho, b1, h);
        }
#pragma unroll 4
        for (int k = 0; k < NO; ++k) {
            const double b1 = D1e[k * RP + p], b2 = D2o[k * RP + p];
            const double2 x = XV[(NE + k) * NC + j], h = XE[(NE + k) * NC + j];
            dfma(ve, b1, x);
            dfma(wo, b2, x);
            dfma(he, b1, h);
        }
        const EoRows R = eo_rows(p, Ny);
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (r && !R.pair) break;
            const int y = r ? R.y1 : R.y0;
            const size_t o = ((size_t)y * E + e) * NM + q, h = ((size_t)q * Ny + y) * E + e;
            P[o] = V[h];
            P[fs + o] = row_of(ve, vo, R.pair, r);
            P[2 * fs + o] = row_of(we, wo, R.pair, r);
            P[3 * fs + o] = H[h];
            P[4 * fs + o] = row_of(he, ho, R.pair, r);
        }
    }
}

__global__ void __launch_bounds__(THREADS) k_forcing64(GroupView g, int s) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int Ny = g.ny, E = g.E, NM = g.nmodes, NKX = g.nkx;
    const Tile T = tile_of(E, NM);
    const int NE = (Ny + 1) / 2, NO = Ny / 2, RP = spc::eo_rp(Ny), NC = T.NC;
    const int q0 = blockIdx.x * T.QT, e0 = blockIdx.y * T.EBT;
    double2* PH = (double2*)sm;              // parity parts of phi = i kx Nu + i kz Nw [Ny][NC]
    double2* GG = PH + Ny * NC;              // i kz Nu - i kx Nw, natural rows
    double2* KV = GG + Ny * NC;              // -k^2 Nv, natural rows
    const size_t fs = (size_t)Ny * E * NM;
    const double2* N3 = (const double2*)g.N3;
    for (int i = threadIdx.x; i < NE * NC; i += THREADS) {
        const int p = i / NC, c = i - p * NC, el = c / T.QT, q = q0 + c - el * T.QT, e = e0 + el;
        const EoRows R = eo_rows(p, Ny);
        double2 ph[2];
        ph[0] = ph[1] = make_double2(0.0, 0.0);
        if (q < NM && e < E) {
            const int mi = q / NKX, n = q - mi * NKX;
            const double kx = g.kxt[n], kz = g.kzt[mi], k2 = g.k2t[q];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                if (r && !R.pair) break;
                const int y = r ? R.y1 : R.y0;
                const size_t o = ((size_t)y * E + e) * NM + q;
                const double2 nu = N3[o], nv = N3[fs + o], nw = N3[2 * fs + o];
                ph[r] = make_double2(-(kx * nu.y + kz * nw.y), kx * nu.x + kz * nw.x);
                GG[y * NC + c] = make_double2(-(kz * nu.y - kx * nw.y), kz * nu.x - kx * nw.x);
                KV[y * NC + c] = make_double2(-k2 * nv.x, -k2 * nv.y);
            }
        }
        PH[p * NC + c] = dadd(ph[0], ph[1]);
        if (R.pair) PH[(NE + p) * NC + c] = dsub(ph[0], ph[1]);
    }
    __syncthreads();
    const int q_mean = mean_mode(g);
    const double* __restrict__ D1e = g.D1EO64;
    const double* __restrict__ D1o = D1e + (size_t)NO * RP;
    const int per = NE * T.EBT;
    for (int m = threadIdx.x; m < T.QT * per; m += THREADS) {
        // consecutive threads: consecutive members, then rows (the H layout)
        const int qq = m / per, r0 = m - qq * per, p = r0 / T.EBT, el = r0 - p * T.EBT;
        const int q = q0 + qq, e = e0 + el, j = el * T.QT + qq;
        if (q >= NM || e >= E) continue;
        double2 ye = make_double2(0.0, 0.0), yo = ye;
#pragma unroll 4
        for (int k = 0; k < NO; ++k) dfma(ye, D1e[k * RP + p], PH[(NE + k) * NC + j]);
#pragma unroll 4
        for (int k = 0; k < NE; ++k) dfma(yo, D1o[k * RP + p], PH[k * NC + j]);
        const EoRows R = eo_rows(p, Ny);
        const int mi = q / NKX, n = q - mi * NKX;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            if (r && !R.pair) break;
            const int y = r ? R.y1 : R.y0;
            double2 F = dsub(KV[y * NC + j], row_of(ye, yo, R.pair, r)), G = GG[y * NC + j];
            if (q == q_mean) { F = make_double2(0.0, 0.0); G = F; }
            if (g.fn > 0 && n == g.fn) {   // stochastic forcing of the step
                const size_t o = ((size_t)mi * Ny + y) * E + e, half = (size_t)g.nkz * Ny * E;
                F = dadd(F, g.noise[o]);
                G = dadd(G, g.noise[half + o]);
            }
            const size_t h = ((size_t)q * Ny + y) * E + e;
            double2 Ft = F, Gt = G;
            if (s == 0) {
                g.Av[h] = F;
                g.Ae[h] = G;
            } else {
                const double2 a = g.Av[h], b = g.Ae[h];
                if (s == 1) {
                    Ft = make_double2(2.0 * F.x - a.x, 2.0 * F.y - a.y);
                    Gt = make_double2(2.0 * G.x - b.x, 2.0 * G.y - b.y);
                    g.Av[h] = make_double2((1.0 / 6.0) * a.x + (4.0 / 6.0) * F.x, (1.0 / 6.0) * a.y + (4.0 / 6.0) * F.y);
                    g.Ae[h] = make_double2((1.0 / 6.0) * b.x + (4.0 / 6.0) * G.x, (1.0 / 6.0) * b.y + (4.0 / 6.0) * G.y);
                } else {
                    Ft = make_double2(a.x + (1.0 / 6.0) * F.x, a.y + (1.0 / 6.0) * F.y);
                    Gt = make_double2(b.x + (1.0 / 6.0) * G.x, b.y + (1.0 / 6.0) * G.y);
                }
            }
            g.Fv[h] = Ft;
            g.Fe[h] = Gt;
        }
    }
}

// members of a k_helm64 CTA: two operators of up to 64 KB and both inputs of the
// pair's two modes fit its shared memory at every Ny
constexpr int HELM_EC = 8;
__host__ __device__ inline int helm_ec(const GroupView& g) {
    const int ec = helm_member_chunk(g);
    return ec < HELM_EC ? ec : HELM_EC;
}
__host__ __device__ inline int helm_chunks(const GroupView& g) { return (g.E + helm_ec(g) - 1) / helm_ec(g); }

// One CTA per (pair, field, member chunk) after the mean-flow row CTAs.
__global__ void __launch_bounds__(THREADS) k_helm64(GroupView g, int s) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int Ny = g.ny, E = g.E, NKX = g.nkx;
    const int nrow = mean_row_ctas(g);
    if ((int)blockIdx.x < nrow) {
        mean_rows(g, s, blockIdx.x % E, (blockIdx.x / E) * (THREADS / 32), sm);
        return;
    }
    const int b = blockIdx.x - nrow;
    const int pr = b % g.npairs, f = (b / g.npairs) & 1, ch = b / (2 * g.npairs);
    const int n = pr % NKX, am = pr / NKX;
    if (!g.lin && pr == 0) return;                        // the mean mode (DNS groups)
    const int e0 = ch * helm_ec(g), ec = min(helm_ec(g), E - e0), nq = am > 0 ? 2 : 1, NC = nq * ec;
    const int NE = (Ny + 1) / 2, NO = Ny / 2, RP = spc::eo_rp(Ny);
    const size_t MEO = spc::eo_mat(Ny);
    const bool needM = s != 2;
    double* MS = (double*)sm;                             // M, P in parity blocks
    double* PS = MS + MEO;
    double2* XS = (double2*)(PS + MEO);                   // parity parts of x_t, F~ [Ny][NC]
    double2* FS = XS + Ny * NC;
    unsigned long long* bar = (unsigned long long*)(FS + Ny * NC);
    const unsigned bar_a = su32(bar);
    if (threadIdx.x == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar_a) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        const double* src = g.ops64[s == 0 ? 0 : 1] + ((size_t)pr * 4 + 2 * f + (needM ? 0 : 1)) * MEO;
        const unsigned bytes = (unsigned)((needM ? 2 : 1) * MEO * sizeof(double));
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar_a), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                     ::"r"(su32(needM ? MS : PS)), "l"(src), "r"(bytes), "r"(bar_a) : "memory");
    }
    const int q1 = (g.kz + am) * NKX + n, q2 = (g.kz - am) * NKX + n;
    const double2* X = f == 0 ? g.v_t : g.e_t;
    const double2* F = f == 0 ? g.Fv : g.Fe;
    double2* M1 = f == 0 ? g.mx1_v : g.mx1_e;
    double2* O = s == 2 ? (f == 0 ? g.v_t : g.e_t) : (f == 0 ? g.v_s : g.e_s);
    const int per = NE * ec;
    for (int i = threadIdx.x; i < nq * per; i += THREADS) {
        const int which = i / per, r = i - which * per, p = r / ec, el = r - p * ec, c = which * ec + el;
        const EoRows R = eo_rows(p, Ny);
        const size_t q = which ? q2 : q1, h0 = (q * Ny + R.y0) * E + e0 + el, h1 = (q * Ny + R.y1) * E + e0 + el;
        const double2 z = make_double2(0.0, 0.0);
        const double2 f0 = F[h0], f1 = R.pair ? F[h1] : z;
        FS[p * NC + c] = dadd(f0, f1);
        if (R.pair) FS[(NE + p) * NC + c] = dsub(f0, f1);
        if (needM) {
            const double2 x0 = X[h0], x1 = R.pair ? X[h1] : z;
            XS[p * NC + c] = dadd(x0, x1);
            if (R.pair) XS[(NE + p) * NC + c] = dsub(x0, x1);
        }
    }
    __syncthreads();
    if (!mbar_wait(bar_a, 0)) {
        // the operator copy did not land: flag it, give the copy one more bounded
        // wait so no write into this CTA's shared memory is left in flight, leave
        if (threadIdx.x == 0) atomicExch(g.status, 1);
        mbar_wait(bar_a, 0);
        return;
    }
    const double* Mo = MS + (size_t)NE * RP;
    const double* Po = PS + (size_t)NE * RP;
    for (int i = threadIdx.x; i < nq * per; i += THREADS) {
        const int which = i / per, r = i - which * per, p = r / ec, el = r - p * ec, c = which * ec + el;
        const double2 z = make_double2(0.0, 0.0);
        double2 me = z, mo = z, pe = z, po = z;
        if (needM) {
#pragma unroll 4
            for (int k = 0; k < NE; ++k) {
                dfma(me, MS[k * RP + p], XS[k * NC + c]);
                dfma(pe, PS[k * RP + p], FS[k * NC + c]);
            }
#pragma unroll 4
            for (int k = 0; k < NO; ++k) {
                dfma(mo, Mo[k * RP + p], XS[(NE + k) * NC + c]);
                dfma(po, Po[k * RP + p], FS[(NE + k) * NC + c]);
            }
        } else {
#pragma unroll 4
            for (int k = 0; k < NE; ++k) dfma(pe, PS[k * RP + p], FS[k * NC + c]);
#pragma unroll 4
            for (int k = 0; k < NO; ++k) dfma(po, Po[k * RP + p], FS[(NE + k) * NC + c]);
        }
        const EoRows R = eo_rows(p, Ny);
#pragma unroll
        for (int r2 = 0; r2 < 2; ++r2) {
            if (r2 && !R.pair) break;
            const size_t h = ((size_t)(which ? q2 : q1) * Ny + (r2 ? R.y1 : R.y0)) * E + e0 + el;
            double2 mx;
            if (needM) {
                mx = row_of(me, mo, R.pair, r2);
                if (s == 1) M1[h] = mx;
            } else {
                mx = M1[h];
            }
            O[h] = dadd(mx, row_of(pe, po, R.pair, r2));
        }
    }
}

size_t tile_bytes(const GroupView& g, int vectors) {
    const size_t b = (size_t)vectors * g.ny * tile_of(g.E, g.nmodes).NC * sizeof(double2), m = mean_smem_bytes(g);
    return b > m ? b : m;
}

}  // namespace s64

void launch_yderiv64(const GroupView& g, const double2* v, const double2* e, double2* P5, cudaStream_t st, int sprev) {
    const s64::Tile t = s64::tile_of(g.E, g.nmodes);
    dim3 grid((g.nmodes + t.QT - 1) / t.QT, (g.E + t.EBT - 1) / t.EBT);
    grid.y += mean_finish_extra_rows(g, grid.x, sprev);
    s64::k_yderiv64<<<grid, s64::THREADS, s64::tile_bytes(g, 2), st>>>(g, v, e, P5, sprev);
}

void launch_forcing64(const GroupView& g, int s, cudaStream_t st) {
    const s64::Tile t = s64::tile_of(g.E, g.nmodes);
    const dim3 grid((g.nmodes + t.QT - 1) / t.QT, (g.E + t.EBT - 1) / t.EBT);
    s64::k_forcing64<<<grid, s64::THREADS, s64::tile_bytes(g, 3), st>>>(g, s);
}

void launch_helm64(const GroupView& g, int s, cudaStream_t st) {
    size_t b = 2 * spc::eo_mat(g.ny) * sizeof(double) + 2 * (size_t)g.ny * 2 * s64::helm_ec(g) * sizeof(double2) + 16;
    if (b < mean_smem_bytes(g)) b = mean_smem_bytes(g);
    s64::k_helm64<<<mean_row_ctas(g) + 2 * g.npairs * s64::helm_chunks(g), s64::THREADS, b, st>>>(g, s);
}

cudaError_t load_yderiv64() {
    cudaFuncAttributes a;
    return cudaFuncGetAttributes(&a, (const void*)s64::k_yderiv64);
}

void set_attributes_step64() {
    allow_max_dynamic_smem(s64::k_yderiv64);
    allow_max_dynamic_smem(s64::k_forcing64);
    allow_max_dynamic_smem(s64::k_helm64);
}

}  // namespace dnsk
