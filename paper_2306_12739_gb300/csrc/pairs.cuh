// Two transforms side by side: every value a pair of lanes (a, b), the two real
// numbers of two independent transforms.  In single precision a pair is one
// 64-bit register pair and an operation on it one packed instruction (two
// IEEE single-precision operations), so the arithmetic of two transforms costs
// the issue slots of one.  Complex pairs keep real and imaginary parts apart:
// a product by i is a renaming, and nothing is swapped between lanes.
#pragma once
#include <cuda_runtime.h>

namespace dnsk {
namespace prs {

template <typename T> struct Pr { T a, b; };
template <typename T> struct Pc { Pr<T> x, y; };          // two complex numbers

template <typename T> __device__ __forceinline__ Pr<T> pr(T a, T b) { Pr<T> r; r.a = a; r.b = b; return r; }
template <typename T> __device__ __forceinline__ Pr<T> dup(T a) { return pr(a, a); }

__device__ __forceinline__ float2 f2of(Pr<float> p) { return make_float2(p.a, p.b); }
__device__ __forceinline__ Pr<float> pof(float2 v) { return pr(v.x, v.y); }

__device__ __forceinline__ Pr<float> operator+(Pr<float> p, Pr<float> q) { return pof(__fadd2_rn(f2of(p), f2of(q))); }
// p - q = fma(q, -1, p): the product is exact, so this is the rounded difference
__device__ __forceinline__ Pr<float> operator-(Pr<float> p, Pr<float> q) {
    return pof(__ffma2_rn(f2of(q), make_float2(-1.f, -1.f), f2of(p)));
}
__device__ __forceinline__ Pr<float> operator*(Pr<float> p, Pr<float> q) { return pof(__fmul2_rn(f2of(p), f2of(q))); }
__device__ __forceinline__ Pr<float> pneg(Pr<float> p) { return pof(__fmul2_rn(f2of(p), make_float2(-1.f, -1.f))); }
__device__ __forceinline__ Pr<float> pfma(Pr<float> p, Pr<float> q, Pr<float> r) {
    return pof(__ffma2_rn(f2of(p), f2of(q), f2of(r)));
}
__device__ __forceinline__ Pr<double> operator+(Pr<double> p, Pr<double> q) { return pr(p.a + q.a, p.b + q.b); }
__device__ __forceinline__ Pr<double> operator-(Pr<double> p, Pr<double> q) { return pr(p.a - q.a, p.b - q.b); }
__device__ __forceinline__ Pr<double> operator*(Pr<double> p, Pr<double> q) { return pr(p.a * q.a, p.b * q.b); }
__device__ __forceinline__ Pr<double> pneg(Pr<double> p) { return pr(-p.a, -p.b); }
__device__ __forceinline__ Pr<double> pfma(Pr<double> p, Pr<double> q, Pr<double> r) {
    return pr(fma(p.a, q.a, r.a), fma(p.b, q.b, r.b));
}

template <typename T> __device__ __forceinline__ Pc<T> operator+(Pc<T> p, Pc<T> q) { return {p.x + q.x, p.y + q.y}; }
template <typename T> __device__ __forceinline__ Pc<T> operator-(Pc<T> p, Pc<T> q) { return {p.x - q.x, p.y - q.y}; }
// p + S i q, S = +1 or -1
template <int S, typename T> __device__ __forceinline__ Pc<T> add_i(Pc<T> p, Pc<T> q) {
    if (S > 0) return {p.x - q.y, p.y + q.x};
    return {p.x + q.y, p.y - q.x};
}
// p w (CONJ: p conj(w)), a twiddle factor of each lane
template <bool CONJ, typename T> __device__ __forceinline__ Pc<T> pmul(Pc<T> p, Pc<T> w) {
    if (CONJ) return {pfma(p.y, w.y, p.x * w.x), p.y * w.x - p.x * w.y};
    return {p.x * w.x - p.y * w.y, pfma(p.x, w.y, p.y * w.x)};
}

// In-register DFTs of R points, natural order in and out, kernel
// exp(S 2 pi i jk / R).  MID0: points 3 and 4 of 8 are zero (padding).
template <int R, int S, typename T> struct Pdft;
template <int S, typename T> struct Pdft<2, S, T> {
    __device__ __forceinline__ static void run(Pc<T>* v) {
        const Pc<T> a = v[0] + v[1];
        v[1] = v[0] - v[1];
        v[0] = a;
    }
};
template <int S, typename T> struct Pdft<3, S, T> {
    __device__ __forceinline__ static void run(Pc<T>* v) {
        const Pr<T> h = dup((T)0.86602540378443864676), m = dup((T)-0.5);
        const Pc<T> t1 = v[1] + v[2], t2 = v[1] - v[2];
        const Pc<T> c = {pfma(m, t1.x, v[0].x), pfma(m, t1.y, v[0].y)};
        const Pc<T> s = {h * t2.x, h * t2.y};
        v[0] = v[0] + t1;
        v[1] = add_i<S>(c, s);
        v[2] = add_i<-S>(c, s);
    }
};
template <int S, typename T> struct Pdft<4, S, T> {
    __device__ __forceinline__ static void run(Pc<T>* v) {
        const Pc<T> a = v[0] + v[2], b = v[0] - v[2], c = v[1] + v[3], d = v[1] - v[3];
        v[0] = a + c;
        v[2] = a - c;
        v[1] = add_i<S>(b, d);
        v[3] = add_i<-S>(b, d);
    }
};
template <int S, typename T> struct Pdft<6, S, T> {
    __device__ __forceinline__ static void run(Pc<T>* v) {
        Pc<T> e[3] = {v[0], v[2], v[4]}, o[3] = {v[1], v[3], v[5]};
        Pdft<3, S, T>::run(e);
        Pdft<3, S, T>::run(o);
        const Pr<T> h = dup((T)0.86602540378443864676), q = dup((T)0.5), m = dup((T)-0.5);
        const Pc<T> h1 = {h * o[1].x, h * o[1].y}, h2 = {h * o[2].x, h * o[2].y};
        const Pc<T> t1 = add_i<S>(Pc<T>{q * o[1].x, q * o[1].y}, h1);      // o1 (1/2 + S i h)
        const Pc<T> t2 = add_i<S>(Pc<T>{m * o[2].x, m * o[2].y}, h2);      // o2 (-1/2 + S i h)
        v[0] = e[0] + o[0]; v[3] = e[0] - o[0];
        v[1] = e[1] + t1; v[4] = e[1] - t1;
        v[2] = e[2] + t2; v[5] = e[2] - t2;
    }
};
template <int S, typename T> struct Pdft<8, S, T> {
    template <bool MID0 = false>
    __device__ __forceinline__ static void run(Pc<T>* v) {
        Pc<T> e[4], o[4];
        if (MID0) {
            const Pc<T> c = v[2] + v[6], d = v[2] - v[6], p = v[1] + v[5], q = v[1] - v[5];
            e[0] = v[0] + c; e[2] = v[0] - c; e[1] = add_i<S>(v[0], d); e[3] = add_i<-S>(v[0], d);
            o[0] = p + v[7]; o[2] = p - v[7]; o[1] = add_i<-S>(q, v[7]); o[3] = add_i<S>(q, v[7]);
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i) { e[i] = v[2 * i]; o[i] = v[2 * i + 1]; }
            Pdft<4, S, T>::run(e);
            Pdft<4, S, T>::run(o);
        }
        const T cc = (T)0.70710678118654752440;
        const Pr<T> c = dup(cc), n = dup(-cc);
        const Pc<T> t1 = add_i<S>(o[1], o[1]), t3 = add_i<-S>(o[3], o[3]);   // o1 (1 + S i), o3 (1 - S i)
        v[0] = e[0] + o[0]; v[4] = e[0] - o[0];
        v[1] = {pfma(c, t1.x, e[1].x), pfma(c, t1.y, e[1].y)};
        v[5] = {pfma(n, t1.x, e[1].x), pfma(n, t1.y, e[1].y)};
        v[2] = add_i<S>(e[2], o[2]); v[6] = add_i<-S>(e[2], o[2]);
        v[3] = {pfma(n, t3.x, e[3].x), pfma(n, t3.y, e[3].y)};
        v[7] = {pfma(c, t3.x, e[3].x), pfma(c, t3.y, e[3].y)};
    }
};
// first DFTs of a zero-padded transform: with eight points the middle two are padding
template <int R, int S, typename T> __device__ __forceinline__ void pdft_padded(Pc<T>* v) {
    if constexpr (R == 8) Pdft<8, S, T>::template run<true>(v);
    else Pdft<R, S, T>::run(v);
}

// (x, y) exp(S 2 pi i j / N), N = 4, 8 or 16, j < N / 2 a compile-time value after unrolling
template <int N, int S, typename T> __device__ __forceinline__ void rot_const(int j, T& x, T& y) {
    const T c1 = (T)0.92387953251128675613, s1 = (T)0.38268343236508977173, c2 = (T)0.70710678118654752440;
    const T cs[8] = {(T)1, c1, c2, s1, (T)0, -s1, -c2, -c1}, sn[8] = {(T)0, s1, c2, c1, (T)1, c1, c2, s1};
    const int i = j * (16 / N);
    if (i == 0) return;
    const T x0 = x, y0 = y;
    if (i == 4) { x = S > 0 ? -y0 : y0; y = S > 0 ? x0 : -x0; return; }
    const T c = cs[i], s = S > 0 ? sn[i] : -sn[i];
    x = x0 * c - y0 * s;
    y = y0 * c + x0 * s;
}

// One N-point DFT (N = 4, 8, 16) of a single transform, its halves as the two lanes.
// Decimation in time: lanes (2 m, 2 m + 1) in, (k, k + N / 2) out.
template <int N, int S, typename T> __device__ __forceinline__ void dft_dit(Pc<T>* v) {
    Pdft<N / 2, S, T>::run(v);
#pragma unroll
    for (int k = 0; k < N / 2; ++k) {
        T x = v[k].x.b, y = v[k].y.b;
        rot_const<N, S>(k, x, y);
        const T ex = v[k].x.a, ey = v[k].y.a;
        v[k] = {pr(ex + x, ex - x), pr(ey + y, ey - y)};
    }
}
// Decimation in frequency: lanes (j, j + N / 2) in, (2 m, 2 m + 1) out.
template <int N, int S, typename T> __device__ __forceinline__ void dft_dif(Pc<T>* v) {
#pragma unroll
    for (int j = 0; j < N / 2; ++j) {
        const T ax = v[j].x.a, ay = v[j].y.a, bx = v[j].x.b, by = v[j].y.b;
        T dx = ax - bx, dy = ay - by;
        rot_const<N, S>(j, dx, dy);
        v[j] = {pr(ax + bx, dx), pr(ay + by, dy)};
    }
    Pdft<N / 2, S, T>::run(v);
}

// A complex pair in memory: (x.a, x.b, y.a, y.b), 16-byte accesses.
__device__ __forceinline__ Pc<float> ldp(const Pc<float>* p) {
    const float4 q = *(const float4*)p;
    return {pr(q.x, q.y), pr(q.z, q.w)};
}
__device__ __forceinline__ void stp(Pc<float>* p, Pc<float> v) { *(float4*)p = make_float4(v.x.a, v.x.b, v.y.a, v.y.b); }
__device__ __forceinline__ Pc<double> ldp(const Pc<double>* p) {
    const double2 q = ((const double2*)p)[0], r = ((const double2*)p)[1];
    return {pr(q.x, q.y), pr(r.x, r.y)};
}
__device__ __forceinline__ void stp(Pc<double>* p, Pc<double> v) {
    ((double2*)p)[0] = make_double2(v.x.a, v.x.b);
    ((double2*)p)[1] = make_double2(v.y.a, v.y.b);
}

}  // namespace prs
}  // namespace dnsk
