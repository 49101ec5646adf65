// The fused per-wavenumber stage in parity blocks with its products on the warp
// level tensor instructions (the stage of k_spec.cu: forcing, RK3 combination,
// implicit apply, y-derivatives of the new state, mean flow).
//
// Why: the SIMT form of the stage spends its issue slots on operand loads from
// shared memory, one per two multiply-adds (20.9 M warp instructions for 4
// members of 64x65x64, of which 3.8 M are single-precision multiply-adds), and
// holds 40 KB of operators per CTA, so that three CTAs fill an SM and 484 CTAs
// take two waves.  Here a pair's operators come as matrix fragments in the order
// the instruction wants them, straight from L2 into registers, and a warp's
// product of two 16-row blocks with 4 complex columns is 24 instructions.
//
// Precision: every single-precision factor is written as three BF16 pieces (24
// significant bits) and the six products that reach 2^-24 of the leading one are
// accumulated in single precision, smallest first.  D2 v, whose rows cancel
// beyond single precision, is a product of signed 8-bit digits in parity blocks: eight
// (seven up to My = 34) of each factor, D2's against its row's largest entry, v's
// against its column's, the levels of digit products down to the last digit's, summed
// without error.  What that leaves out is below a float-float sum's error at every
// size (smooth columns, relative to max |D2 v|: 2.6e-13 against 8.8e-13 at My = 33,
// 7.5e-13 against 5.8e-12 at 65, 3.3e-12 against 1.2e-11 at 97, 7.6e-12 against 2.9e-11
// at 129), so that the rounding to single precision, 5e-8, is all that shows.
//
// One CTA per (pair (n, |m|), member chunk).  A warp has 16 pair-rows x 4 complex
// columns (8 real ones); a lane owns two pair-rows of one column (their even and
// odd output parts) in every phase, so the natural rows, the RK combination and
// the FP64 update stay in its registers.  Vectors cross the warps of a column tile
// in shared memory as BF16 pieces [column][even part | odd part]; the rows of a
// part are ordered so that a lane's two rows are neighbours (one 32-bit store),
// and the operators' columns are permuted to match.  Only the warps of one column
// tile (and field) meet at the barriers between phases.
//
// What bounds a CTA is the chain of its phases (operand loads from L2, products,
// epilogues).  The chains of v and eta are almost independent until D v, so on
// groups too small to fill the chip every tile gets two warps, one per field
// (TWO); on larger ones a warp does both, which holds half the warps for less than
// twice the time (sides measured at spec_mma_two).
#include "dns_internal.hpp"
#include "cvt.cuh"
#include "eo.cuh"
#include "ff.cuh"
#include "mean.cuh"
#include "mbar.cuh"
#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

namespace dnsk {

namespace smm {

using spc::eo_rows;
using spc::EoRows;
typedef unsigned short bf;

constexpr int EC_MAX = 8;      // members per CTA (two modes: 16 complex columns)
// members per CTA of the y-derivatives (one column tile each): one from three row
// tiles up, whose CTAs are then 6 or 8 warps and three fit an SM
__host__ __device__ constexpr int yd_ec(int kt) { return kt > 2 ? 1 : 2; }
__host__ __device__ constexpr int yd_regs(int kt) { return kt == 3 ? 112 : 128; }
constexpr int PIECES = 3;
// D2 v: signed digits of DBITS bits of either factor (at most 256 units, exact in
// BF16); the levels s + t < ndig of the digit products are summed.  Seven digits leave
// less than a float-float sum up to My = 34 (one row tile), eight at every size.
constexpr int DBITS = 8;
__host__ __device__ constexpr int ndig(int kt) { return kt == 1 ? 7 : 8; }

__host__ __device__ inline int tiles(int ny) { return ((ny + 1) / 2 + 15) / 16; }   // 16-row tiles of a parity block
// members per CTA: at most 512 threads
__host__ __device__ inline int chunk_members(const GroupView& g) {
    const int cap = tiles(g.ny) > 2 ? EC_MAX / 2 : EC_MAX;
    const int ec = (g.spec_ec > 0 && g.spec_ec <= cap) ? g.spec_ec : cap;
    return g.E < ec ? g.E : ec;
}
__host__ __device__ inline int chunks(const GroupView& g) { return (g.E + chunk_members(g) - 1) / chunk_members(g); }
__host__ __device__ inline int col_tiles(int ec) { return (2 * ec + 3) / 4; }        // of 4 complex columns
// fragments: [block][row tile][k tile][piece or digit][lane] of 16 bytes
__host__ __device__ constexpr int mat_frags(int kt, int n) { return 2 * kt * kt * n * 32; }

// shared memory: the stage 6 vectors of three pieces (phi / v+, G~, x_eta, x_v, F~, eta+;
// the digits of v+ then lie over G~, x_eta and x_v), the derivatives alone v, its
// digits and eta; column exponents
constexpr int STAGE_PIECES = 6 * PIECES;
__host__ __device__ constexpr int deriv_pieces(int kt) { return 2 * PIECES + ndig(kt); }
static_assert(ndig(4) <= 3 * PIECES, "the digits lie over three vectors");
struct Shape {
    int KT, NT, CS, VP;     // k tiles, column tiles, column stride and piece size (BF16 values)
};
__host__ __device__ inline Shape shape_of(int ny, int nt) {
    Shape s;
    s.KT = tiles(ny);
    s.NT = nt;
    s.CS = 32 * s.KT + 8;   // conflict-free: lanes' 8 columns are 4 (mod 8) banks apart
    s.VP = 8 * s.NT * s.CS;
    return s;
}
__host__ __device__ inline Shape shape_of(const GroupView& g) { return shape_of(g.ny, col_tiles(chunk_members(g))); }
inline size_t smem_bytes(const Shape& s, int pieces) {
    return (size_t)pieces * s.VP * sizeof(bf) + (size_t)s.KT * 8 * s.NT * sizeof(int);
}

__device__ __forceinline__ void mma(float (&d)[4], uint4 a, unsigned b0, unsigned b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldm4(unsigned (&r)[4], unsigned addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
// two values as BF16 (round to nearest even), lo in the low half
__device__ __forceinline__ unsigned bf2(float lo, float hi) {
    unsigned r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}

struct Cols {
    int p, n, am, q1, q2, e0, ec, C;
};
__device__ __forceinline__ Cols cols_of(const GroupView& g, int b) {
    Cols c;
    const int np1 = g.npairs - 1, ch = b / np1;        // pair 0 is the mean mode: no CTA
    c.p = 1 + b % np1;
    c.n = c.p % g.nkx;
    c.am = c.p / g.nkx;
    c.q1 = (g.kz + c.am) * g.nkx + c.n;
    c.q2 = (g.kz - c.am) * g.nkx + c.n;
    c.e0 = ch * chunk_members(g);
    c.ec = min(chunk_members(g), g.E - c.e0);
    c.C = (c.am > 0 ? 2 : 1) * c.ec;
    return c;
}
__device__ __forceinline__ bool in_range(const GroupView& g, int q, int y, int e) {
    return DNS_CK(g.status, (unsigned)q < (unsigned)g.nmodes && (unsigned)y < (unsigned)g.ny && (unsigned)e < (unsigned)g.E,
                  CK_SPEC, ((long long)q * g.ny + y) * g.E + e);
}

// A warp's place: row tile mt, column tile nt; the lane's pair-rows p(r) = 16 mt +
// lane / 4 + 8 r, r = 0, 1, and complex column j = 4 nt + lane % 4.
struct Place {
    int lane, mt, nt, j;
    __device__ __forceinline__ int p(int r) const { return 16 * mt + (lane >> 2) + 8 * r; }
};

// the three pieces of the lane's two rows of one part (0 even, 1 odd) of real
// column 2 j + c
__device__ __forceinline__ void put2(bf* vec, const Shape& S, const Place& w, int c, int part, float x0, float x1) {
    unsigned* o = (unsigned*)(vec + (2 * w.j + c) * S.CS + 16 * (S.KT * part + w.mt)) + (w.lane >> 2);
    const int vp = S.VP / 2;
#pragma unroll
    for (int i = 0; i < PIECES; ++i) {
        const unsigned h = bf2(x0, x1);
        o[i * vp] = h;
        x0 -= __uint_as_float(h << 16);
        x1 -= __uint_as_float(h & 0xFFFF0000u);
    }
}
// the parts of the lane's rows n[r][k2] of its complex column (rows without a
// mirror row: k2 = 1 holds zero, as do rows beyond the grid)
__device__ __forceinline__ void put_parts(bf* vec, const Shape& S, const Place& w, const bool (&pair)[2],
                                          const float2 (&n)[2][2]) {
    put2(vec, S, w, 0, 0, n[0][0].x + n[0][1].x, n[1][0].x + n[1][1].x);
    put2(vec, S, w, 1, 0, n[0][0].y + n[0][1].y, n[1][0].y + n[1][1].y);
    put2(vec, S, w, 0, 1, pair[0] ? n[0][0].x - n[0][1].x : 0.f, pair[1] ? n[1][0].x - n[1][1].x : 0.f);
    put2(vec, S, w, 1, 1, pair[0] ? n[0][0].y - n[0][1].y : 0.f, pair[1] ? n[1][0].y - n[1][1].y : 0.f);
}

// even and odd output rows of two pair-rows of one complex column
struct Out {
    float e[4], o[4];        // [2 r + c]
    // natural row k2 (0: p, 1: Ny - 1 - p) of pair-row r
    __device__ __forceinline__ float2 nat(int r, bool pair, int k2) const {
        if (!pair) return make_float2(e[2 * r], e[2 * r + 1]);
        if (k2) return make_float2(0.5f * (e[2 * r] - o[2 * r]), 0.5f * (e[2 * r + 1] - o[2 * r + 1]));
        return make_float2(0.5f * (e[2 * r] + o[2 * r]), 0.5f * (e[2 * r + 1] + o[2 * r + 1]));
    }
};

// The tensor cores cut a sum off towards zero.  What that takes on average, in units in
// the last place (emulated on the sums of this library's operators, My = 33 to 97, smooth
// and rough columns; the instruction itself was seen to do it on random sums): of the
// products of P 0.2 to 0.5, whose terms spread over many powers of two, of M - I 0.06 to
// 0.36, of D1 0.02 to 0.27, mostly below 0.1 (many of its sums need no cut).  Left alone
// it makes every increment a little too small, step after step: against 64 bits, after
// 20 to 50 steps, errors of the state up to 1.18 times the FP32 stage's (32x24x32
// rotational; 64x28x16 1.11, 48x36x32 1.04).  So P's leading sums get half a unit back
// (to the small products' accumulator), M - I's a quarter: 0.90, 0.88 and 0.89 times.
constexpr float CUT_P = 0x1p-24f, CUT_M = 0x1p-25f;     // of the sum's power of two

// the power of two of x's binary exponent, x's sign
__device__ __forceinline__ float power_of(float x) { return __uint_as_float(__float_as_uint(x) & 0xFF800000u); }

// out = matrix x vector for this warp's tile.  SWAP: an anti-centro-symmetric
// matrix (D1): its even rows contract the odd part, its odd rows the even part; its sums
// are left as they are, those of the others get cut.
template <int KT, bool SWAP>
__device__ __forceinline__ void product(const uint4* __restrict__ A, const bf* vec, const Shape& S, const Place& w,
                                        Out& out, float cut = 0.f) {
    // this lane's row address of the four 8 x 8 blocks of an ldmatrix: columns of
    // the tile, k halves, parts
    const unsigned at = su32(vec + (8 * w.nt + (w.lane & 7)) * S.CS + ((w.lane >> 3) & 1) * 8 + (w.lane >> 4) * 16 * KT);
    // The leading products of a k tile start from zero and are added up rounded to
    // nearest, the small ones have an accumulator of their own.
    float le[4] = {0.f, 0.f, 0.f, 0.f}, lo[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int kt = 0; kt < KT; ++kt) {
        uint4 ae[PIECES], ao[PIECES];
        unsigned b[PIECES][4];
        const uint4* fe = A + ((w.mt * KT + kt) * PIECES) * 32 + w.lane;
        const uint4* fo = fe + KT * KT * PIECES * 32;
#pragma unroll
        for (int i = 0; i < PIECES; ++i) { ae[i] = fe[i * 32]; ao[i] = fo[i * 32]; }
#pragma unroll
        for (int i = 0; i < PIECES; ++i) ldm4(b[i], at + 2 * (i * S.VP + 16 * kt));
        // pieces i + l = 2, 1: the smallest products first
#pragma unroll
        for (int l = PIECES - 1; l > 0; --l)
#pragma unroll
            for (int i = 0; i <= l; ++i) {
                mma(le, ae[l - i], b[i][SWAP ? 2 : 0], b[i][SWAP ? 3 : 1]);
                mma(lo, ao[l - i], b[i][SWAP ? 0 : 2], b[i][SWAP ? 1 : 3]);
            }
        float he[4] = {0.f, 0.f, 0.f, 0.f}, ho[4] = {0.f, 0.f, 0.f, 0.f};
        mma(he, ae[0], b[0][SWAP ? 2 : 0], b[0][SWAP ? 3 : 1]);
        mma(ho, ao[0], b[0][SWAP ? 0 : 2], b[0][SWAP ? 1 : 3]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            out.e[i] = kt == 0 ? he[i] : __fadd_rn(out.e[i], he[i]);
            out.o[i] = kt == 0 ? ho[i] : __fadd_rn(out.o[i], ho[i]);
            if (!SWAP) {
                le[i] = __fmaf_rn(power_of(he[i]), cut, le[i]);
                lo[i] = __fmaf_rn(power_of(ho[i]), cut, lo[i]);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        out.e[i] = __fadd_rn(out.e[i], le[i]);
        out.o[i] = __fadd_rn(out.o[i], lo[i]);
    }
}

// h + b, the rounding error added to l
__device__ __forceinline__ void two_sum(float& h, float& l, float b) {
    const float s = __fadd_rn(h, b), v = __fsub_rn(s, h);
    l = __fadd_rn(l, __fadd_rn(__fsub_rn(h, __fsub_rn(s, v)), __fsub_rn(b, v)));
    h = s;
}
// D2 v: digit products level by level.  A level's terms are multiples of one power of
// two and stay below 2^24 of it (64 columns, at most 8 products of a first digit up to
// 256 or others up to 130), so each level sums exactly; the levels add up by error-free
// transformations.  The last two levels share an accumulator: they weigh less than
// 2^-40 of the scale, and cutting that off at 24 bits stays below what is left out.
// up: the columns' powers of two.
template <int KT>
__device__ __forceinline__ void d2_product(const GroupView& g, const bf* dig, const Shape& S, const Place& w, float2 up,
                                           Out& out) {
    constexpr int NDIG = ndig(KT), NACC = NDIG - 1;
    const unsigned at = su32(dig + (8 * w.nt + (w.lane & 7)) * S.CS + ((w.lane >> 3) & 1) * 8 + (w.lane >> 4) * S.VP);
#pragma unroll 1
    for (int blk = 0; blk < 2; ++blk) {
        const uint4* A = (const uint4*)g.D2MM + (size_t)blk * KT * KT * NDIG * 32;
        float acc[NACC][4];
#pragma unroll
        for (int L = 0; L < NACC; ++L)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[L][i] = 0.f;
#pragma unroll
        for (int kt = 0; kt < KT; ++kt) {
            uint4 a[NDIG];
#pragma unroll
            for (int s = 0; s < NDIG; ++s) a[s] = A[((w.mt * KT + kt) * NDIG + s) * 32 + w.lane];
#pragma unroll
            for (int s = 0; s < NDIG; s += 2) {
                unsigned b[4];           // digits s, s + 1 (beyond the last: whatever follows it, unused)
                ldm4(b, at + 2 * (s * S.VP + 16 * KT * blk + 16 * kt));
#pragma unroll
                for (int L = s; L < NDIG; ++L) mma(acc[L < NACC ? L : NACC - 1], a[L - s], b[0], b[1]);
#pragma unroll
                for (int L = s + 1; L < NDIG; ++L) mma(acc[L < NACC ? L : NACC - 1], a[L - s - 1], b[2], b[3]);
            }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            float h = acc[0][i], l = 0.f;
#pragma unroll
            for (int L = 1; L < NACC - 1; ++L) two_sum(h, l, acc[L][i]);
            const float r = __fmul_rn(__fadd_rn(h, __fadd_rn(l, acc[NACC - 1][i])), i & 1 ? up.y : up.x);
            if (!blk) out.e[i] = r;
            else out.o[i] = r;
        }
    }
}

// v's even and odd parts as float-float pairs of the lane's two rows, [r][c]
struct NewV {
    float eh[2][2], el[2][2], oh[2][2], ol[2][2];
};
// biased exponent of |x| rounded up: |x| < 2^(result - 126)
__device__ __forceinline__ int fexp(float x) { return (int)((__float_as_uint(x) >> 23) & 0xFF); }

// v's parts (natural rows v[r][k2], zero where there is none): single-precision
// pieces for D v, and the columns' exponents
__device__ __forceinline__ void stage_v(const Shape& S, const Place& w, const bool (&pair)[2], const double2 (&v)[2][2],
                                        NewV& nv, bf* VV, int* cexp) {
    int mx[2] = {0, 0};
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            spc::eo_ff(c ? v[r][0].y : v[r][0].x, c ? v[r][1].y : v[r][1].x, nv.eh[r][c], nv.el[r][c], nv.oh[r][c],
                       nv.ol[r][c]);
            if (!pair[r]) nv.oh[r][c] = nv.ol[r][c] = 0.f;
            mx[c] = max(mx[c], max(fexp(nv.eh[r][c]), fexp(nv.oh[r][c])));
        }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        put2(VV, S, w, c, 0, nv.eh[0][c], nv.eh[1][c]);
        put2(VV, S, w, c, 1, nv.oh[0][c], nv.oh[1][c]);
#pragma unroll
        for (int o = 4; o < 32; o *= 2) mx[c] = max(mx[c], __shfl_xor_sync(0xffffffffu, mx[c], o));
        if (w.lane < 4) cexp[w.mt * 8 * S.NT + 2 * w.j + c] = mx[c];
    }
}
// After a barrier: the digits of v's parts, the column scaled by a power of two to
// below 1 (a column of any magnitude keeps all of them); the result is that power.
// Digit s is the multiple of 2^(-DBITS (s + 1)) nearest to what the digits before it
// leave (adding and subtracting 1.5 2^23 units rounds to whole units).  The pair's low
// part, below 2^-23, joins after the second digit as an error-free sum, whose error
// joins after the fourth.
template <int KT>
__device__ __forceinline__ float2 stage_digits(const Shape& S, const Place& w, const NewV& nv, bf* DG, const int* cexp) {
    float up[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        int be = 0;
        for (int m = 0; m < S.KT; ++m) be = max(be, cexp[m * 8 * S.NT + 2 * w.j + c]);
        be = min(be, 252);                       // (beyond it, and for Inf and NaN, D2 v overflows)
        up[c] = __uint_as_float((unsigned)(be + 1) << 23);                  // 2^f, f = be - 126
        const float down = __uint_as_float((unsigned)(253 - be) << 23);     // 2^-f
        unsigned* o = (unsigned*)(DG + (2 * w.j + c) * S.CS + 16 * w.mt) + (w.lane >> 2);
#pragma unroll
        for (int part = 0; part < 2; ++part) {
            float r0 = __fmul_rn(part ? nv.oh[0][c] : nv.eh[0][c], down), l0 = __fmul_rn(part ? nv.ol[0][c] : nv.el[0][c], down);
            float r1 = __fmul_rn(part ? nv.oh[1][c] : nv.eh[1][c], down), l1 = __fmul_rn(part ? nv.ol[1][c] : nv.el[1][c], down);
#pragma unroll
            for (int s = 0; s < ndig(KT); ++s) {
                const float m = __uint_as_float(((unsigned)(127 + 23 - DBITS * (s + 1)) << 23) | 0x400000u);
                const float d0 = __fsub_rn(__fadd_rn(r0, m), m), d1 = __fsub_rn(__fadd_rn(r1, m), m);
                o[s * (S.VP / 2) + 8 * S.KT * part] = __byte_perm(__float_as_uint(d0), __float_as_uint(d1), 0x7632);
                r0 = __fsub_rn(r0, d0);
                r1 = __fsub_rn(r1, d1);
                if (s == 1) {
                    float e0 = 0.f, e1 = 0.f;
                    two_sum(r0, e0, l0);
                    two_sum(r1, e1, l1);
                    l0 = e0;
                    l1 = e1;
                }
                if (s == 3) {
                    r0 = __fadd_rn(r0, l0);
                    r1 = __fadd_rn(r1, l1);
                }
            }
        }
    }
    return make_float2(up[0], up[1]);
}

// A CTA's view of its work: the lane's column and natural rows
template <int KT, bool TWO>
struct Lane {
    Shape S;
    Cols c;
    Place w;
    int Ny, E, NM, q, e;
    bool eta, tile;                   // TWO: this warp has eta, else v; it has columns
    bool pair[2], on[2][2];           // rows with a mirror row; rows that exist
    size_t fs5;
    __device__ __forceinline__ Lane(const GroupView& g, int b) : S(shape_of(g)), c(cols_of(g, b)) {
        place(g);
        tile = 4 * w.nt < c.C;
        const bool live = w.j < c.C, first = w.j < c.ec;
        q = first ? c.q1 : c.q2;
        e = c.e0 + (first ? w.j : w.j - c.ec);
        rows(g, live);
    }
    // the y-derivatives' columns: a column tile is 4 consecutive modes of one member
    __device__ __forceinline__ Lane(const GroupView& g, int q0, int e0) : S(shape_of(g.ny, yd_ec(KT))), c() {
        place(g);
        q = q0 + (w.lane & 3);
        e = e0 + w.nt;
        tile = e < g.E;
        rows(g, tile && q < g.nmodes);
    }
    __device__ __forceinline__ void place(const GroupView& g) {
        Ny = g.ny; E = g.E; NM = g.nmodes;
        fs5 = (size_t)Ny * E * NM;
        const int warp = threadIdx.x >> 5;
        w.lane = threadIdx.x & 31;
        eta = TWO && warp >= KT * S.NT;
        w.mt = warp % KT;
        w.nt = warp / KT - (eta ? S.NT : 0);
        w.j = 4 * w.nt + (w.lane & 3);
    }
    __device__ __forceinline__ void rows(const GroupView& g, bool live) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            pair[r] = w.p(r) < Ny / 2;
            on[r][0] = live && w.p(r) < (Ny + 1) / 2 && in_range(g, q, w.p(r), e);
            on[r][1] = live && pair[r] && in_range(g, q, Ny - 1 - w.p(r), e);
        }
    }
    __device__ __forceinline__ int y(int r, int k2) const { return k2 ? Ny - 1 - w.p(r) : w.p(r); }
    __device__ __forceinline__ size_t h(int r, int k2) const { return ((size_t)q * Ny + y(r, k2)) * E + e; }    // H layout
    __device__ __forceinline__ size_t o(int r, int k2) const { return ((size_t)y(r, k2) * E + e) * NM + q; }    // P layout
    // the warps of this column tile and field meet; of both fields
    __device__ __forceinline__ void sync() const {
        if (KT == 1) __syncwarp();
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + w.nt + (eta ? S.NT : 0)), "r"(32 * KT) : "memory");
    }
    __device__ __forceinline__ void sync_both() const {
        if (!TWO) sync();
        else asm volatile("bar.sync %0, %1;" ::"r"(1 + 2 * S.NT + w.nt), "r"(64 * KT) : "memory");
    }
    __device__ __forceinline__ void write(const GroupView& g, int f, const Out& d) const {
        float2* P5 = (float2*)g.P5 + f * fs5;
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k2 = 0; k2 < 2; ++k2)
                if (on[r][k2]) P5[o(r, k2)] = d.nat(r, pair[r], k2);
    }
};

// The end of the stage and of the derivatives of a newly set state, the new
// state's vectors staged: D eta and D v (eta's warps), D2 v (v's).
template <int KT, bool TWO>
__device__ __forceinline__ void derivatives(const GroupView& g, const Lane<KT, TWO>& l, const NewV& nv, const bf* VV,
                                            bf* DG, const bf* EN, const int* cexp) {
    Out d;
    if (!TWO || l.eta) {
        if (TWO) l.sync();
#pragma unroll 1
        for (int f = 4; f > 0; f -= 3) {        // D eta, then D v
            product<KT, true>((const uint4*)g.D1MM, f == 4 ? EN : VV, l.S, l.w, d);
            l.write(g, f, d);
            if (f == 4) l.sync_both();
        }
        if (TWO) return;
    } else {
        l.sync_both();
    }
    const float2 up = stage_digits<KT>(l.S, l.w, nv, DG, cexp);
    l.sync();
    d2_product<KT>(g, DG, l.S, l.w, up, d);
    l.write(g, 2, d);
}

// F (or G) of a row, its accumulator a: the sub-step's combination; a becomes the new
// accumulator.  (Sums of products are written out as fused multiply-adds here and
// below: a member's bits must not depend on the form its group runs.)
__device__ __forceinline__ float2 combine(int s, float2 F, float2& a) {
    float2 r = F;
    if (s == 0) {
        a = F;
    } else if (s == 1) {
        r = make_float2(2.f * F.x - a.x, 2.f * F.y - a.y);
        a = make_float2(__fmaf_rn(1.f / 6.f, a.x, __fmul_rn(4.f / 6.f, F.x)),
                        __fmaf_rn(1.f / 6.f, a.y, __fmul_rn(4.f / 6.f, F.y)));
    } else {
        r = make_float2(__fmaf_rn(1.f / 6.f, F.x, a.x), __fmaf_rn(1.f / 6.f, F.y, a.y));
    }
    return r;
}
__device__ __forceinline__ float sum2(float a, float x, float b, float y) { return __fmaf_rn(a, x, __fmul_rn(b, y)); }

// The lane's rows of one field
struct Rows {
    float2 f[2][2], acc[2][2];   // v: -k^2 Nv, eta: G (+ noise); the RK accumulator
    double2 x[2][2];             // x_t
    float2 m1[2][2];             // third sub-step: the stored (M - I) x_t
};

// One field's share of a CTA's work, its phases between the barriers
template <int KT, bool TWO>
struct Field {
    const GroupView& g;
    const Lane<KT, TWO>& l;
    const int s;
    const bool eta, needM;
    const uint4* ops;            // M - I, then P
    const double2* X;
    double2* O;
    float2 *M1, *A;
    __device__ __forceinline__ Field(const GroupView& g_, const Lane<KT, TWO>& l_, int s_, bool eta_)
        : g(g_), l(l_), s(s_), eta(eta_), needM(s_ != 2) {
        ops = (const uint4*)g.opsMM[s == 0 ? 0 : 1] + (size_t)(l.c.p * 4 + (eta ? 2 : 0)) * mat_frags(KT, PIECES);
        X = eta ? g.e_t : g.v_t;
        O = eta ? (s == 2 ? g.e_t : g.e_s) : (s == 2 ? g.v_t : g.v_s);
        M1 = (float2*)(eta ? g.mx1_e : g.mx1_v);
        A = (float2*)(eta ? g.Ae : g.Av);
    }
    __device__ __forceinline__ void load_x(Rows& R) const {
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k2 = 0; k2 < 2; ++k2) {
                R.x[r][k2] = make_double2(0.0, 0.0);
                if (l.on[r][k2]) R.x[r][k2] = X[l.h(r, k2)];
            }
    }
    __device__ __forceinline__ void store_acc(const Rows& R) const {
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k2 = 0; k2 < 2; ++k2)
                if (s != 2 && l.on[r][k2]) A[l.h(r, k2)] = R.acc[r][k2];
    }
    __device__ __forceinline__ void load_acc(Rows& R) const {
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k2 = 0; k2 < 2; ++k2) {
                R.acc[r][k2] = make_float2(0.f, 0.f);
                if (s != 0 && l.on[r][k2]) R.acc[r][k2] = A[l.h(r, k2)];
            }
    }
    __device__ __forceinline__ void load_m1(Rows& R) const {
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k2 = 0; k2 < 2; ++k2)
                if (s == 2 && l.on[r][k2]) R.m1[r][k2] = M1[l.h(r, k2)];
    }
    // Nu, Nw, the accumulator and (v) Nv of the lane's rows
    __device__ __forceinline__ void load(Rows& R, float2 (&nu)[2][2], float2 (&nw)[2][2]) const {
        const float2* N3 = (const float2*)g.N3;
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k2 = 0; k2 < 2; ++k2) {
                nu[r][k2] = nw[r][k2] = R.f[r][k2] = make_float2(0.f, 0.f);
                if (!l.on[r][k2]) continue;
                const size_t o = l.o(r, k2);
                nu[r][k2] = N3[o];
                nw[r][k2] = N3[2 * l.fs5 + o];
                if (!eta) R.f[r][k2] = N3[l.fs5 + o];
            }
        load_acc(R);
    }
    // v: t = phi = i kx Nu + i kz Nw, R.f = -k^2 Nv; eta: t = G~ combined from G = i kz Nu
    // - i kx Nw, the accumulator written back
    __device__ __forceinline__ void terms(Rows& R, const float2 (&nu)[2][2], const float2 (&nw)[2][2],
                                          float2 (&t)[2][2]) const {
        const float kx = g.kxtf[l.c.n];
        const int mz = l.w.j < l.c.ec ? g.kz + l.c.am : g.kz - l.c.am;
        const float kz = g.kztf[mz], k2n = sum2(kx, kx, kz, kz);
        const bool forced = g.fn > 0 && l.c.n == g.fn;
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k2 = 0; k2 < 2; ++k2) {
                const float2 u = nu[r][k2], v = nw[r][k2];
                float2 f = eta ? make_float2(-sum2(kz, u.y, -kx, v.y), sum2(kz, u.x, -kx, v.x))
                               : make_float2(-k2n * R.f[r][k2].x, -k2n * R.f[r][k2].y);
                if (forced && l.on[r][k2] && DNS_CK(g.status, mz < g.nkz, CK_SPEC, l.q)) {
                    const size_t o = ((size_t)mz * l.Ny + l.y(r, k2)) * l.E + l.e, half = (size_t)g.nkz * l.Ny * l.E;
                    const double2 nz = g.noise[eta ? half + o : o];
                    f.x = __fadd_rn(f.x, (float)nz.x);
                    f.y = __fadd_rn(f.y, (float)nz.y);
                }
                if (!eta) R.f[r][k2] = f;
                t[r][k2] = eta ? combine(s, f, R.acc[r][k2]) : make_float2(-sum2(kx, u.y, kz, v.y), sum2(kx, u.x, kz, v.x));
            }
        if (eta) store_acc(R);
    }
    __device__ __forceinline__ void put_x(const Rows& R, bf* XT) const {
        if (!needM) return;
        float2 t[2][2];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k2 = 0; k2 < 2; ++k2) t[r][k2] = make_float2(d2f(R.x[r][k2].x), d2f(R.x[r][k2].y));
        put_parts(XT, l.S, l.w, l.pair, t);
    }
    // the two-warp form's first phase: phi or G~ into N, x_t into XT
    __device__ __forceinline__ void begin(Rows& R, bf* N, bf* XT) const {
        float2 nu[2][2], nw[2][2], t[2][2];
        load(R, nu, nw);
        load_x(R);
        terms(R, nu, nw, t);
        put_parts(N, l.S, l.w, l.pair, t);
        put_x(R, XT);
    }
    // v: F~ from D1 phi into FT
    __device__ __forceinline__ void forcing(Rows& R, const bf* PH, bf* FT) const {
        Out d;
        product<KT, true>((const uint4*)g.D1MM, PH, l.S, l.w, d);
        float2 t[2][2];
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k2 = 0; k2 < 2; ++k2) {
                const float2 dd = d.nat(r, l.pair[r], k2);
                const float2 F = make_float2(__fsub_rn(R.f[r][k2].x, dd.x), __fsub_rn(R.f[r][k2].y, dd.y));
                t[r][k2] = l.on[r][k2] ? combine(s, F, R.acc[r][k2]) : make_float2(0.f, 0.f);
            }
        store_acc(R);
        put_parts(FT, l.S, l.w, l.pair, t);
    }
    __device__ __forceinline__ void increment(const bf* XT, Out& dm) const {
        if (needM) product<KT, false>(ops, XT, l.S, l.w, dm, CUT_M);
    }
    // x+ = x_t + ((M - I) x_t + P F~): into the state, the per-plane field and R.x; its
    // single-precision rows in xs
    __device__ __forceinline__ void apply(Rows& R, const Out& dm, const bf* F, float2 (&xs)[2][2]) const {
        Out dp;
        product<KT, false>(ops + mat_frags(KT, PIECES), F, l.S, l.w, dp, CUT_P);
        float2* P = (float2*)g.P5 + (eta ? 3 : 0) * l.fs5;
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int k2 = 0; k2 < 2; ++k2) {
                xs[r][k2] = make_float2(0.f, 0.f);
                if (!l.on[r][k2]) continue;
                const float2 m = s == 2 ? R.m1[r][k2] : dm.nat(r, l.pair[r], k2), pp = dp.nat(r, l.pair[r], k2);
                const size_t h = l.h(r, k2);
                if (s == 1) M1[h] = m;
                R.x[r][k2].x += (double)__fadd_rn(m.x, pp.x);
                R.x[r][k2].y += (double)__fadd_rn(m.y, pp.y);
                O[h] = R.x[r][k2];
                xs[r][k2] = make_float2(d2f(R.x[r][k2].x), d2f(R.x[r][k2].y));
                P[l.o(r, k2)] = xs[r][k2];
            }
    }
};

template <int KT, int REGS, bool TWO>
__global__ void __maxnreg__(REGS) k_spec_mma(GroupView g, int s) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int nrow = g.E * mean_ctas_per_member(g, blockDim.x);
    if ((int)blockIdx.x < nrow) {
        mean_cta(g, s, blockIdx.x, sm);
        return;
    }
    const Lane<KT, TWO> l(g, blockIdx.x - nrow);
    if (!l.tile) return;                        // only the warps of a column tile meet
    const int V = PIECES * l.S.VP;
    bf* VV = (bf*)sm;                           // phi, then v+
    bf* GT = VV + V;                            // G~; the digits of v+ start here
    bf* XE = GT + V;                            // eta_t
    bf* XV = XE + V;                            // v_t
    bf* FT = XV + V;                            // F~
    bf* EN = FT + V;                            // eta+
    int* cexp = (int*)(EN + V);
    float2 xs[2][2];
    NewV nv;
    Out dm;
    if (TWO) {
        const Field<KT, TWO> f(g, l, s, l.eta);
        Rows R;
        f.begin(R, l.eta ? GT : VV, l.eta ? XE : XV);
        l.sync();
        f.increment(l.eta ? XE : XV, dm);
        if (!l.eta) {
            f.forcing(R, VV, FT);
            l.sync();
        }
        f.load_m1(R);
        f.apply(R, dm, l.eta ? GT : FT, xs);
        if (l.eta) put_parts(EN, l.S, l.w, l.pair, xs);
        else stage_v(l.S, l.w, l.pair, R.x, nv, VV, cexp);
    } else {
        // every load of the first phase in flight together
        const Field<KT, TWO> fv(g, l, s, false), fe(g, l, s, true);
        Rows Rv, Re;
        float2 nu[2][2], nw[2][2];
        fv.load(Rv, nu, nw);
        fe.load_acc(Re);
        if (fv.needM) {
            fe.load_x(Re);
            fv.load_x(Rv);
        }
        fv.terms(Rv, nu, nw, xs);
        put_parts(VV, l.S, l.w, l.pair, xs);
        fe.terms(Re, nu, nw, xs);
        put_parts(GT, l.S, l.w, l.pair, xs);
        fe.put_x(Re, XE);
        fv.put_x(Rv, XV);
        l.sync();
        fv.forcing(Rv, VV, FT);
        // eta, then v: rolled, as is every other loop whose turns share their code (a
        // warp runs the kernel once, top to bottom, and instruction fetch is what it
        // waits for most)
#pragma unroll 1
        for (int eta = 1; eta >= 0; --eta) {
            const Field<KT, TWO> f(g, l, s, eta != 0);
            Rows R;
            f.load_x(R);
            f.load_m1(R);
            if (!eta) l.sync();
            f.increment(eta ? XE : XV, dm);
            f.apply(R, dm, eta ? GT : FT, xs);
            if (eta) put_parts(EN, l.S, l.w, l.pair, xs);
            else stage_v(l.S, l.w, l.pair, R.x, nv, VV, cexp);
        }
    }
    derivatives<KT, TWO>(g, l, nv, VV, GT, EN, cexp);
}

// v, Dv, D2v, eta, D eta of (V, H) in the per-plane layout: what the stage leaves for the
// state it produces (the same parts, products and order).
template <int KT>
__device__ __forceinline__ void state_derivatives(const GroupView& g, const Lane<KT, true>& l, const double2* __restrict__ V,
                                                  const double2* __restrict__ H, unsigned char* sm) {
    bf* VV = (bf*)sm;
    bf* DG = VV + PIECES * l.S.VP;
    bf* EN = DG + ndig(KT) * l.S.VP;
    int* cexp = (int*)(EN + PIECES * l.S.VP);
    const double2* X = l.eta ? H : V;
    float2* P = (float2*)g.P5 + (l.eta ? 3 : 0) * l.fs5;
    double2 x[2][2];
    float2 xs[2][2];
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int k2 = 0; k2 < 2; ++k2) {
            x[r][k2] = make_double2(0.0, 0.0);
            if (l.on[r][k2]) x[r][k2] = X[l.h(r, k2)];
        }
#pragma unroll
    for (int r = 0; r < 2; ++r)
#pragma unroll
        for (int k2 = 0; k2 < 2; ++k2) {
            xs[r][k2] = make_float2(d2f(x[r][k2].x), d2f(x[r][k2].y));
            if (l.on[r][k2]) P[l.o(r, k2)] = xs[r][k2];
        }
    NewV nv;
    if (l.eta) put_parts(EN, l.S, l.w, l.pair, xs);
    else stage_v(l.S, l.w, l.pair, x, nv, VV, cexp);
    derivatives<KT, true>(g, l, nv, VV, DG, EN, cexp);
}

// for a newly set state (one CTA per pair and member chunk, as the stage)
template <int KT>
__global__ void __maxnreg__(128) k_mma_derivs(GroupView g) {
    extern __shared__ __align__(16) unsigned char sm[];
    const Lane<KT, true> l(g, blockIdx.x);
    if (l.tile) state_derivatives<KT>(g, l, g.v_t, g.e_t, sm);
}

// The y-derivatives of the step-by-step stage: 4 consecutive modes x yd_ec members a
// CTA, so that the per-plane fields are written in whole sectors; the grid's rows
// beyond the members finish the previous sub-step's mean flow.
template <int KT>
__global__ void __maxnreg__(yd_regs(KT)) k_yderiv_mma(GroupView g, const double2* __restrict__ V, const double2* __restrict__ H,
                                              int sprev) {
    extern __shared__ __align__(16) unsigned char sm[];
    if (mean_finish_rows(g, sprev, (g.E + yd_ec(KT) - 1) / yd_ec(KT), sm)) return;
    const Lane<KT, true> l(g, 4 * blockIdx.x, yd_ec(KT) * blockIdx.y);
    if (l.tile) state_derivatives<KT>(g, l, V, H, sm);
}

}  // namespace smm

// ------------------------------------------------------------------- host

static uint16_t bf16_of(double x) {              // round to nearest even
    const float f = (float)x;
    uint32_t u;
    memcpy(&u, &f, 4);
    u += 0x7FFFu + ((u >> 16) & 1u);
    return (uint16_t)(u >> 16);
}
static double of_bf16(uint16_t h) {
    const uint32_t u = (uint32_t)h << 16;
    float f;
    memcpy(&f, &u, 4);
    return f;
}

// One matrix in parity blocks (spec_eo_image64: [KE][RP] of its even output rows,
// [KO][RP] of its odd ones) as A fragments.  piece(row value, n) -> BF16 of piece n
template <typename Piece>
static void fragments(const double* eo, int ny, bool anti, int npiece, uint16_t* out, Piece piece) {
    const int KT = smm::tiles(ny), NE = spc::eo_ne(ny), NO = ny / 2, RP = spc::eo_rp(ny);
    for (int blk = 0; blk < 2; ++blk) {
        const int rows = blk ? NO : NE, ks = (blk != 0) == anti ? NE : NO;
        const double* B = eo + (blk ? (size_t)(anti ? NO : NE) * RP : 0);
        for (int mt = 0; mt < KT; ++mt)
            for (int kt = 0; kt < KT; ++kt)
                for (int i = 0; i < npiece; ++i)
                    for (int lane = 0; lane < 32; ++lane)
                        for (int h = 0; h < 8; ++h) {
                            // registers a0..a3: rows g, g + 8, g, g + 8; k 2t.., 2t.., 2t + 8.., 2t + 8..
                            const int reg = h >> 1;
                            const int r = 16 * mt + (lane >> 2) + (reg & 1 ? 8 : 0);
                            // (place i of a k tile holds row i / 2 + 8 (i mod 2), see put2)
                            const int i16 = 2 * (lane & 3) + (h & 1) + (reg & 2 ? 8 : 0);
                            const int k = 16 * kt + (i16 >> 1) + 8 * (i16 & 1);
                            *out++ = r < rows && k < ks ? piece(B[(size_t)k * RP + r], blk, r, i) : (uint16_t)0;
                        }
    }
}

size_t spec_mma_mat_bytes(int ny) { return (size_t)smm::mat_frags(smm::tiles(ny), smm::PIECES) * 16; }
size_t spec_mma_d2_bytes(int ny) { return (size_t)smm::mat_frags(smm::tiles(ny), smm::ndig(smm::tiles(ny))) * 16; }

void spec_mma_image(const double* eo, int ny, bool anti, uint16_t* out) {
    fragments(eo, ny, anti, smm::PIECES, out, [](double v, int, int, int i) {
        uint16_t h = bf16_of(v);
        for (; i > 0; --i) {
            v -= of_bf16(h);
            h = bf16_of(v);
        }
        return h;
    });
}

// D2's digits: digit i of a parity row whose entries are below 2^e is the multiple
// of 2^(e - DBITS (i + 1)) nearest to what the digits before it leave
void spec_mma_d2_image(const double* eo, int ny, uint16_t* out) {
    const int KT = smm::tiles(ny), NE = spc::eo_ne(ny), NO = ny / 2, RP = spc::eo_rp(ny);
    std::vector<int> rexp(2 * 16 * KT, 0);
    for (int blk = 0; blk < 2; ++blk)
        for (int r = 0; r < (blk ? NO : NE); ++r) {
            double mx = 0.0;
            const double* B = eo + (blk ? (size_t)NE * RP : 0);
            for (int k = 0; k < (blk ? NO : NE); ++k) mx = std::fmax(mx, std::fabs(B[(size_t)k * RP + r]));
            if (mx > 0.0) std::frexp(mx, &rexp[blk * 16 * KT + r]);
        }
    fragments(eo, ny, false, smm::ndig(KT), out, [&](double v, int blk, int r, int i) {
        double d = 0.0;
        for (int s = 0; s <= i; ++s) {
            v -= d;
            const double u = std::ldexp(1.0, rexp[blk * 16 * KT + r] - smm::DBITS * (s + 1));
            d = std::nearbyint(v / u) * u;
        }
        return bf16_of(d);
    });
}

// The fused stage with tensor-instruction products: its operator fragments (both
// step lengths, 1.5 times the single-precision operators) must stay a fraction of
// L2, or streaming them costs more than the products save (128x97x128: 206 MB a
// step length).
bool spec_mma_supported(const GroupView& g) {
    return !g.lin && g.npairs > 1 && g.ny >= 3 && smm::smem_bytes(smm::shape_of(g), smm::STAGE_PIECES) + 1024 <= 227 * 1024 &&
           2 * (size_t)g.npairs * 4 * spec_mma_mat_bytes(g.ny) <= ((size_t)96 << 20);
}

size_t spec_mma_smem_bytes(const GroupView& g) {
    const size_t b = smm::smem_bytes(smm::shape_of(g), smm::STAGE_PIECES), m = mean_smem_bytes(g);
    return b > m ? b : m;
}

// Two warps per tile while the chip then still holds every one of them at once (16
// at 128 registers on each of 152 SMs): 16x33x16 x 1 12.5 us a launch against 16.2,
// 48x36x32 x 3 16.3 against 19.6; beyond it 64x65x64 x 4 34.2 against 31.5.
static bool spec_mma_two(const GroupView& g) {
    const long long warps = (long long)(g.npairs - 1) * smm::chunks(g) * smm::tiles(g.ny) *
                            smm::col_tiles(smm::chunk_members(g)) * g.nblk;
    return 2 * warps <= 16 * 152;
}

void launch_spec_mma(const GroupView& g, int s, cudaStream_t st) {
    const bool two = spec_mma_two(g);
    const int kt = smm::tiles(g.ny), threads = (two ? 64 : 32) * kt * smm::col_tiles(smm::chunk_members(g));
    const int ctas = g.E * mean_ctas_per_member(g, threads) + (g.npairs - 1) * smm::chunks(g);
    const size_t sm = spec_mma_smem_bytes(g);
#define DNS_GO(k, r)                                                                         \
    {                                                                                        \
        if (two) smm::k_spec_mma<k, r, true><<<ctas, threads, sm, st>>>(g, s);               \
        else smm::k_spec_mma<k, r, false><<<ctas, threads, sm, st>>>(g, s);                  \
    }
#define DNS_CASE(k)                                                                          \
    if (kt == k) {                                                                           \
        if (g.spec_minb == 3) DNS_GO(k, 96) else DNS_GO(k, 128)                              \
    }
    DNS_CASE(1) DNS_CASE(2) DNS_CASE(3) DNS_CASE(4)
#undef DNS_CASE
#undef DNS_GO
}

void launch_mma_derivs(const GroupView& g, cudaStream_t st) {
    const int kt = smm::tiles(g.ny), threads = 64 * kt * smm::col_tiles(smm::chunk_members(g));
    const int ctas = (g.npairs - 1) * smm::chunks(g);
    const size_t sm = spec_mma_smem_bytes(g);
#define DNS_CASE(k) if (kt == k) smm::k_mma_derivs<k><<<ctas, threads, sm, st>>>(g);
    DNS_CASE(1) DNS_CASE(2) DNS_CASE(3) DNS_CASE(4)
#undef DNS_CASE
}

void launch_yderiv_mma(const GroupView& g, const double2* v, const double2* e, cudaStream_t st, int sprev) {
    const int kt = smm::tiles(g.ny), ec = smm::yd_ec(kt), threads = 64 * kt * ec;
    dim3 grid((g.nmodes + 3) / 4, (g.E + ec - 1) / ec);
    grid.y += mean_finish_extra_rows(g, grid.x, sprev);
    size_t sm = smm::smem_bytes(smm::shape_of(g.ny, ec), smm::deriv_pieces(kt));
    if (sm < mean_smem_bytes(g)) sm = mean_smem_bytes(g);
#define DNS_CASE(k) if (kt == k) smm::k_yderiv_mma<k><<<grid, threads, sm, st>>>(g, v, e, sprev);
    DNS_CASE(1) DNS_CASE(2) DNS_CASE(3) DNS_CASE(4)
#undef DNS_CASE
}

void set_attributes_spec_mma() {
#define DNS_CASE(k)                                  \
    allow_max_dynamic_smem(smm::k_spec_mma<k, 96, false>);  \
    allow_max_dynamic_smem(smm::k_spec_mma<k, 128, false>); \
    allow_max_dynamic_smem(smm::k_spec_mma<k, 96, true>);   \
    allow_max_dynamic_smem(smm::k_spec_mma<k, 128, true>);  \
    allow_max_dynamic_smem(smm::k_mma_derivs<k>);           \
    allow_max_dynamic_smem(smm::k_yderiv_mma<k>);
    DNS_CASE(1) DNS_CASE(2) DNS_CASE(3) DNS_CASE(4)
#undef DNS_CASE
}

}  // namespace dnsk
