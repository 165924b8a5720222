// physics_exact.cuh -- FP64 RHS arithmetic in the reference operation order.
//
// The same stiffened-gas EOS (arXiv 2409.10729, Sec. II-A), WENO5-JS and
// HLLC (Sec. II-B) as physics.cuh, but every formula is evaluated in the
// textbook order the serial FP64 oracle uses, with one IEEE rounding per
// operation.  Compiled with -fmad=false (no contraction of a*b+c), the
// results are bit-identical to that order.  GB300's FP64 pipe retires two
// operations per SM and clock, so the quotients, the square roots, WENO5's
// products and products by small integers are formed from the IEEE 754 fields
// on the integer pipes -- correctly rounded, hence the same bits.  A division
// by a width given with its rounded reciprocal y = RN(1/b) takes one FMA
// correction (Markstein, "Computation of elementary functions on the IBM RISC
// System/6000", 1990):  q = RN(a y),  r = RN(a - b q) (exact),  RN(q + r y),
// which is a/b rounded for operands without overflow or underflow.
#pragma once
#include "physics.cuh"

namespace mfc5 {
namespace exact {

// Correctly rounded a/b given y = RN(1/b).
__device__ __forceinline__ double div_rcp(double a, double b, double y) {
    double q = __dmul_rn(a, y);
    double r = __fma_rn(-b, q, a);
    return __fma_rn(r, y, q);
}

// ---- correctly rounded quotients on the integer pipes ------------------------
// A quotient a/b of positive normal doubles from the significands alone:
// b = m 2^(e-1075), m in [2^52, 2^53).  rcp_i forms R, 1/(m 2^-53) scaled by
// 2^62 and low by at most 1.2 units: an FP32 seed I0 2^-23 of 24 bits (its
// relative error eps is below 2^-22), whose residual E = 2^76 - m I0 fits 55
// bits, so the low 64 bits of m I0 hold it exactly, and one cubic step
// R = I0 (1 + eps + eps^2).  quot_i multiplies the numerator's significand
// (doubled where it is the smaller one, so that the quotient starts at 2^52)
// by R, rounds the product to 53 bits -- never above the nearest integer q*,
// at most one below it, because R, the dropped partial product and the
// rounding constant (127/256 instead of 1/2) all err downwards by less than
// 1/50 unit together -- and takes q + 1 where the exact remainder says so:
// c 2^k - q m > m/2, read off the sign of c 2^k - q m - floor(m/2) - 1, which
// fits 64 bits.  A quotient of two 53-bit integers is never halfway between
// two 53-bit integers, so that is round-to-nearest: the IEEE bits.  About 20
// integer instructions for a quotient and 20 for a reciprocal shared by
// several, where the FP64 pipe (2 lanes per SM and clock) takes 48 and 80
// clocks per warp, and that pipe bounds these kernels: of the 104 FP64
// instructions per field and cell of WENO5, 61 were reciprocals and quotients.
// Measured on the 256^3 droplets: 0.80 -> 0.60 ns per cell, equation and RHS
// with WENO's quotients formed here, 0.557 with those of the EOS and of HLLC.
__device__ __forceinline__ unsigned lo32(unsigned long long v) { return (unsigned)v; }
__device__ __forceinline__ unsigned hi32(unsigned long long v) { return (unsigned)(v >> 32); }
__device__ __forceinline__ unsigned long long wide(unsigned a, unsigned b) { return (unsigned long long)a * b; }
// {ah, al} +- {bh, bl} on 32-bit words
__device__ __forceinline__ void add2(unsigned& h, unsigned& l, unsigned bh, unsigned bl) {
    asm("add.cc.u32 %1, %1, %3;\n\taddc.u32 %0, %0, %2;" : "+r"(h), "+r"(l) : "r"(bh), "r"(bl));
}
__device__ __forceinline__ void sub2(unsigned& h, unsigned& l, unsigned bh, unsigned bl) {
    asm("sub.cc.u32 %1, %1, %3;\n\tsubc.u32 %0, %0, %2;" : "+r"(h), "+r"(l) : "r"(bh), "r"(bl));
}

struct RcpI {
    unsigned r1, r0;   // R
    unsigned mh, ml;   // significand m of the divisor
    unsigned nh, nl;   // -m
    unsigned kh, kl;   // -floor(m/2) - 1
    unsigned e20;      // exponent field in place
};

__device__ __forceinline__ RcpI rcp_i(double b) {
    RcpI o;
    const unsigned h = (unsigned)__double2hiint(b), l = (unsigned)__double2loint(b);
    o.e20 = h & 0x7ff00000u;
    o.mh = (h & 0x000fffffu) | 0x00100000u;
    o.ml = l;
    // m 2^-53 to 24 bits; the last bit set keeps its reciprocal below 2
    const float x = __uint_as_float((__funnelshift_l(l, h & 0x000fffffu, 3)) | 0x3f000001u);
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    const unsigned I0 = (__float_as_uint(r) & 0x007fffffu) | 0x00800000u;
    const unsigned long long p = wide(l, I0);
    const unsigned ph = hi32(p) + o.mh * I0, pl = lo32(p);          // m I0 mod 2^64 = -E
    const unsigned long long sq = (unsigned long long)((long long)(int)ph * (int)ph);   // eps^2 2^88
    unsigned dh = hi32(sq) >> 12, dl = __funnelshift_r(lo32(sq), hi32(sq), 12);
    sub2(dh, dl, ph, pl);                                           // (eps + eps^2) 2^76
    const unsigned long long t =
        (unsigned long long)((long long)(int)I0 * (int)dh) + (unsigned long long)__umulhi(I0, dl);   // scale 2^67
    o.r0 = __funnelshift_r(lo32(t), hi32(t), 5);
    o.r1 = (I0 << 7) + (unsigned)((int)hi32(t) >> 5);
    o.nh = 0u;
    o.nl = 0u;
    sub2(o.nh, o.nl, o.mh, l);
    o.kh = ~(o.mh >> 1);
    o.kl = ~__funnelshift_r(l, o.mh, 1);
    return o;
}

// RN(a/b) for positive normal a and b whose quotient is normal; b as rcp_i(b)
__device__ __forceinline__ double quot_i(double a, const RcpI& b) {
    const unsigned h = (unsigned)__double2hiint(a), l = (unsigned)__double2loint(a);
    const unsigned ch = (h & 0x000fffffu) | 0x00100000u;
    const bool ge = ch > b.mh || (ch == b.mh && l >= b.ml);
    const unsigned s = ge ? 9u : 10u;
    const unsigned c1 = __funnelshift_l(l, ch, s), c0 = l << s;     // below 2^63
    const unsigned lowp = __umulhi(c0, b.r1) + (__umulhi(c1, b.r0) + 127u);
    const unsigned long long Q = wide(c1, b.r1) + lowp;             // quotient 2^60, 127/256 added
    const unsigned qh = hi32(Q) >> 8, ql = __funnelshift_r(lo32(Q), hi32(Q), 8);
    const unsigned long long t = wide(ql, b.nl) + (((unsigned long long)((c0 << 11) + b.kh) << 32) | b.kl);
    const unsigned th = hi32(t) + ql * b.nh + qh * b.nl;            // sign of c 2^k - q m - floor(m/2) - 1
    unsigned oh = (h & 0x7ff00000u) - b.e20 + (ge ? 1022u << 20 : 1021u << 20) + qh, ol = ql;
    add2(oh, ol, 0u, (~th) >> 31);
    return __hiloint2double((int)oh, (int)ol);
}

// Both operands' range: exponent field within 300 of 1.0's, positive (so every
// quotient of two such numbers, and of those by their sums, is normal)
__device__ __forceinline__ bool mid_range(double x) {
    return ((unsigned)__double2hiint(x) - (723u << 20)) < (600u << 20);
}

// a / b out of line, for the rare operands outside that range
static __device__ __noinline__ double div_any(double a, double b) { return a / b; }
static __device__ __noinline__ double sqrt_any(double a) { return sqrt(a); }

// ---- correctly rounded products on the integer pipes -------------------------
// The 106-bit product of two significands (words w3..w0, in [2^104, 2^106))
// rounded to 53 bits, ties to even: the low 32 + s bits are dropped, their
// first 32 in f with the rest or-ed into its last bit, and f + 2^31 - 1 + (last
// kept bit) carries exactly when the kept part has to go up.  e20: sum of the
// exponent fields less 1024, in place.
// A product costs about 35 integer instructions with its checks, where the FP64
// pipe takes 16 clocks a warp: it pays as long as that pipe is the bound and the
// code stays in the instruction caches.  WENO5's 14 products and squares and
// HLLC's square roots moved here: FP64 instructions per warp cell 547 -> 440,
// 256^3 0.464 -> 0.411 ns (the products with everything unrolled 0.454, their
// loops over indicators and faces kept rolled 0.421).  HLLC's fifty products as
// well brought 0.400 to 0.469, depending on the block size, and slowed small
// grids (32^3 0.454 -> 0.478 ms a step): the instruction caches; out of line
// 0.436.  They stay on the FP64 pipe.
__device__ __forceinline__ double round_product(unsigned w3, unsigned w2, unsigned w1, unsigned w0, unsigned e20) {
    const unsigned n = w3 >> 9, s = 20u + n;
    const unsigned ql = __funnelshift_r(w1, w2, s), qh = __funnelshift_r(w2, w3, s);
    const unsigned f = __funnelshift_r(w0, w1, s) | min(w0 << (12u - n), 1u);
    const unsigned up = 0x7fffffffu + (ql & 1u);
    const unsigned e = e20 + (n << 20);
    unsigned oh, ol;
    asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %3, %4;\n\taddc.cc.u32 %1, %2, 0;\n\taddc.u32 %0, %5, %6;\n\t}"
        : "=r"(oh), "=r"(ol)
        : "r"(ql), "r"(f), "r"(up), "r"(qh), "r"(e));
    return __hiloint2double((int)oh, (int)ol);
}

// |x| within 2^-R .. 2^R
template <unsigned R>
__device__ __forceinline__ bool in_range(double x) {
    return (((unsigned)__double2hiint(x) & 0x7fffffffu) - ((1023u - R) << 20)) < ((2u * R) << 20);
}

// Normal: neither zero, subnormal, infinite nor NaN; h: the number's high word
__device__ __forceinline__ bool normal_hi(unsigned h) { return (h & 0x7ff00000u) - 0x00100000u < 0x7fe00000u; }

// RN(x^2) for |x| within 2^-300 .. 2^300; smaller x give 0, larger ones and NaN
// clear ok.  (The squares of differences below 2^-300 are parts of smoothness
// indicators, added to eps.  They sum to less than 2^-598, under half a unit in
// the last place of any eps from 2^-538 up; the square of a smaller eps is zero,
// and the face values of such a cell are NaN with or without these parts.)
__device__ __forceinline__ double sq_i(double x, bool& ok) {
    const unsigned h = (unsigned)__double2hiint(x) & 0x7fffffffu, l = (unsigned)__double2loint(x);
    ok = ok && h < (1323u << 20);
    const unsigned m = (h & 0x000fffffu) | 0x00100000u;
    const unsigned long long t0 = wide(l, l), t1 = wide(l, m << 1) + hi32(t0), t2 = wide(m, m) + hi32(t1);
    const double r = round_product(hi32(t2), lo32(t2), lo32(t1), lo32(t0), 2u * (h & 0x7ff00000u) - (1024u << 20));
    return h < (723u << 20) ? 0.0 : r;
}

// RN(a b) for a positive and normal and b zero, or b and the product normal (else
// ok is cleared; a is the caller's to check)
__device__ __forceinline__ double mul_i(double a, double b, bool& ok) {
    const unsigned ha = (unsigned)__double2hiint(a), la = (unsigned)__double2loint(a);
    const unsigned hb = (unsigned)__double2hiint(b), lb = (unsigned)__double2loint(b);
    const bool zero = ((hb << 1) | lb) == 0u;
    const unsigned e20 = (ha & 0x7ff00000u) + (hb & 0x7ff00000u) - (1024u << 20);
    ok = ok && (zero || (normal_hi(hb) && e20 < (2044u << 20)));
    const unsigned ma = (ha & 0x000fffffu) | 0x00100000u, mb = (hb & 0x000fffffu) | 0x00100000u;
    const unsigned long long t0 = wide(la, lb), t1 = wide(la, mb) + hi32(t0), t2 = wide(ma, lb) + lo32(t1);
    const unsigned long long t3 = wide(ma, mb) + (hi32(t1) + hi32(t2));
    const double r = round_product(hi32(t3), lo32(t3), lo32(t2), lo32(t0), e20);
    const unsigned sign = hb & 0x80000000u;
    return __hiloint2double((int)((zero ? 0u : (unsigned)__double2hiint(r)) | sign),
                            (int)(zero ? 0u : (unsigned)__double2loint(r)));
}

// RN(a b) for a and b each zero, or both and the product normal (else ok is cleared)
__device__ __forceinline__ double mul_s(double a, double b, bool& ok) {
    const unsigned ha = (unsigned)__double2hiint(a), la = (unsigned)__double2loint(a);
    const bool zero = ((ha << 1) | la) == 0u;
    bool in = normal_hi(ha);
    const double r = mul_i(a, b, in);
    const unsigned hb = (unsigned)__double2hiint(b);
    ok = ok && (in || (zero && (hb & 0x7ff00000u) != 0x7ff00000u));
    // the sign from the operands: with a zero, r's high word means nothing
    const unsigned h = zero ? 0u : (unsigned)__double2hiint(r) & 0x7fffffffu;
    return __hiloint2double((int)(h | ((ha ^ hb) & 0x80000000u)), zero ? 0 : __double2loint(r));
}

// How the EOS functions below form their products: on the FP64 pipe, or on the
// integer pipes (the same bits; ok is cleared when an operand was out of range
// and the results do not count).
struct MulFp {
    __device__ __forceinline__ double operator()(double a, double b) const { return a * b; }
};
struct MulInt {
    bool& ok;
    __device__ __forceinline__ double operator()(double a, double b) const { return mul_s(a, b, ok); }
};

// RN(sqrt(a)) for a within 2^-300 .. 2^300.  a = m' 2^(2 k), m' in [2^52, 2^54):
// the square root's significand is q = RN(sqrt(m' 2^52)).  An FP32 seed I0 2^-23
// of 1/sqrt(x), x = m' 2^-54, whose residual eps = 1 - x I0^2 2^-46 (below
// 2^-20, taken from the 101-bit product m' I0^2 without its lowest 32 bits)
// gives 1/sqrt(x) = I0 (1 + eps/2 + 3/8 eps^2) to 2^-61, then sqrt(x) = x /
// sqrt(x) to 4 units of 2^-58, low; rounded to 53 bits with 15/32 it is q or
// q - 1, and N - q^2 - q - 1 >= 0 with N = m' 2^52 (64 bits hold its sign) says
// which.  A square root of 53-bit integers is never halfway between two.
__device__ __forceinline__ double sqrt_i(double a) {
    const unsigned h = (unsigned)__double2hiint(a), l = (unsigned)__double2loint(a);
    const unsigned odd = ~(h >> 20) & 1u;   // an even exponent field: m doubled
    const unsigned mh = (h & 0x000fffffu) | 0x00100000u;
    const unsigned Mh = __funnelshift_l(l, mh, odd), Ml = l << odd;
    const float x = __uint_as_float((odd ? 0x3f000004u : 0x3e800004u) | ((h & 0x000fffffu) << 3));
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    const unsigned I0 = (__float_as_uint(fmaxf(r, 1.0f)) & 0x007fffffu) | 0x00800000u;
    const unsigned long long S = wide(I0, I0);
    const unsigned long long t0 = wide(Ml, hi32(S)) + __umulhi(Ml, lo32(S));
    const unsigned long long t = wide(Mh, lo32(S)) + t0;
    unsigned eh = 0u, el = 0u;
    sub2(eh, el, hi32(t) + Mh * hi32(S), lo32(t));                    // eps 2^68
    const int em = (int)__funnelshift_r(el, eh, 18);
    const unsigned long long sq = (unsigned long long)((long long)em * em);   // eps^2 2^100
    const unsigned long long s3 = wide(hi32(sq), 3u);
    unsigned ch = (unsigned)((int)eh >> 1), cl = __funnelshift_r(el, eh, 1);
    add2(ch, cl, hi32(s3) >> 3, __funnelshift_r(lo32(s3), hi32(s3), 3));
    const unsigned long long T =
        (unsigned long long)((long long)(int)I0 * (int)ch) + (unsigned long long)__umulhi(I0, cl);
    const unsigned r0 = lo32(T), r1 = (I0 << 4) + hi32(T);            // 1/sqrt(x) 2^59
    const unsigned a1 = __funnelshift_l(Ml, Mh, 9), a0 = Ml << 9;
    const unsigned long long Q = wide(a1, r1) + (__umulhi(a1, r0) + __umulhi(a0, r1) + 15u);   // sqrt(x) 2^58
    const unsigned ql = __funnelshift_r(lo32(Q), hi32(Q), 5), qh = hi32(Q) >> 5;
    const unsigned long long q2 = wide(ql, ql) + ql;                  // q^2 + q, low 64 bits
    const unsigned q2h = hi32(q2) + 2u * (ql * qh) + qh;
    unsigned dh = Ml << 20, dl = 0u;
    sub2(dh, dl, q2h, lo32(q2));
    sub2(dh, dl, 0u, 1u);
    unsigned oh = ((((h >> 20) - 1075u - odd + 4096u) >> 1) - 2048u + 1048u) << 20, ol = ql;
    oh += qh;
    add2(oh, ol, 0u, (~dh) >> 31);
    return __hiloint2double((int)oh, (int)ol);
}

// RN(sqrt(a)) for any a
__device__ __forceinline__ double sqrt_p(double a) {
    const double r = sqrt_i(a);
    return __builtin_expect(in_range<300>(a) && gt0(a), 1) ? r : sqrt_any(a);
}

// RN(a/b) for any a and b, y = rcp_i(b): signs and a zero numerator are dealt
// with here, operands or quotients that are not normal take the FP64 division.
// (Disturbances run ahead of a front by many orders of magnitude a cell, so tiny
// normal numbers are common: while anything below 2^-300 took the FP64 path,
// here and in the squares and products, 256^3 droplets took 154 ms a step after
// twelve steps, 139 now, and 142 -> 134 at the start.)
__device__ __forceinline__ double quot(double a, double b, const RcpI& y) {
    const unsigned ha = (unsigned)__double2hiint(a), la = (unsigned)__double2loint(a);
    const unsigned hb = (unsigned)__double2hiint(b);
    const bool zero = ((ha << 1) | la) == 0u;
    const bool in = normal_hi(ha) && (ha & 0x7ff00000u) - y.e20 + (1021u << 20) < (2044u << 20);
    const double q = quot_i(a, y);
    const unsigned sign = (ha ^ hb) & 0x80000000u;
    double r = __hiloint2double((int)((zero ? 0u : (unsigned)__double2hiint(q)) | sign),
                                (int)(zero ? 0u : (unsigned)__double2loint(q)));
    if (__builtin_expect(!(normal_hi(hb) && (in || zero)), 0)) r = div_any(a, b);
    return r;
}
__device__ __forceinline__ double quot(double a, double b) { return quot(a, b, rcp_i(b)); }

__device__ __forceinline__ double sq(double x) { return x * x; }

// Gamma = sum_i alpha_i g_i, Pi = sum_i alpha_i P_i over the NF fluids, the
// carried fractions a[0..NF-2] first and alpha_N = 1 - a[0] - ... - a[NF-2]
// last (two fluids: a1 g1 + (1 - a1) g2).
template <int NF, typename M>
__device__ __forceinline__ void mixture(const M& mul, const Eos& e, const double* a, double& G, double& Pi) {
    double aN = 1.0 - a[0];
#pragma unroll
    for (int i = 1; i < NF - 1; ++i) aN = aN - a[i];
    double sg = mul(a[0], e.g[0]), sp = mul(a[0], e.P[0]);
#pragma unroll
    for (int i = 1; i < NF - 1; ++i) {
        sg = sg + mul(a[i], e.g[i]);
        sp = sp + mul(a[i], e.P[i]);
    }
    G = sg + mul(aN, e.g[NF - 1]);
    Pi = sp + mul(aN, e.P[NF - 1]);
}

template <int NF>
__device__ __forceinline__ double mix_rho(const double* q) {
    double rho = q[0] + q[1];
#pragma unroll
    for (int i = 2; i < NF; ++i) rho = rho + q[i];
    return rho;
}

// 0.5 rho |u|^2 in the oracle's order, whose sum starts from 0.0: 0.0 + u_0^2
// is u_0^2 itself (a square is never -0), so the sum starts there.
template <int NDIM, typename M>
__device__ __forceinline__ double kinetic(const M& mul, double rho, const double* u) {
    double s = mul(u[0], u[0]);
#pragma unroll
    for (int k = 1; k < NDIM; ++k) s = s + mul(u[k], u[k]);
    return mul(0.5 * rho, s);
}

// Conservative -> primitive (u_k = rho u_k / rho, p = (rho E - ke - Pi)/Gamma).
template <int NDIM, int NF = 2, typename M = MulFp>
__device__ __forceinline__ void cons_to_prim(const Eos& e, const double* q, double* w, const M& mul = M()) {
    using FL = Fields<NDIM, NF>;
    double rho = mix_rho<NF>(q);
    const RcpI y = rcp_i(rho);
    double u[NDIM];
#pragma unroll
    for (int k = 0; k < NDIM; ++k) u[k] = quot(q[FL::IU + k], rho, y);
    double ke = kinetic<NDIM>(mul, rho, u);
    double G, Pi;
    mixture<NF>(mul, e, q + FL::IA, G, Pi);
    double p = quot(q[FL::IE] - ke - Pi, G);
#pragma unroll
    for (int i = 0; i < NF; ++i) w[i] = q[i];
#pragma unroll
    for (int k = 0; k < NDIM; ++k) w[FL::IU + k] = u[k];
    w[FL::IE] = p;
#pragma unroll
    for (int i = 0; i < FL::NA; ++i) w[FL::IA + i] = q[FL::IA + i];
}

// Primitive -> conservative (rho E = Gamma p + Pi + ke).
template <int NDIM, int NF = 2, typename M = MulFp>
__device__ __forceinline__ void prim_to_cons(const Eos& e, const double* w, double* q, const M& mul = M()) {
    using FL = Fields<NDIM, NF>;
    double rho = mix_rho<NF>(w);
    double u[NDIM];
#pragma unroll
    for (int k = 0; k < NDIM; ++k) u[k] = w[FL::IU + k];
    double ke = kinetic<NDIM>(mul, rho, u);
    double G, Pi;
    mixture<NF>(mul, e, w + FL::IA, G, Pi);
#pragma unroll
    for (int i = 0; i < NF; ++i) q[i] = w[i];
#pragma unroll
    for (int k = 0; k < NDIM; ++k) q[FL::IU + k] = mul(rho, u[k]);
    q[FL::IE] = mul(G, w[FL::IE]) + Pi + ke;
#pragma unroll
    for (int i = 0; i < FL::NA; ++i) q[FL::IA + i] = w[FL::IA + i];
}

template <typename M>
__device__ __forceinline__ double sound2(const M& mul, double G, double Pi, double rho, double p) {
    return quot(mul(G + 1.0, p) + Pi, mul(G, rho));
}

// WENO5-JS: left-biased value at i+1/2 and right-biased value at i-1/2 from
// v0..v4 = v_{i-2}..v_{i+2}; weights a_k = d_k/(eps+beta_k)^2, omega_k = a_k/sum(a),
// candidate values (.)/6, face value sum omega_k p_k.
//
// Products by a power of two (2, 4, 1/4) are exact, so RN(RN(2 v) + x) equals
// the single fused RN(2 v + x): those sums are written as FMAs (fma2 below),
// which changes no result bit (barring a product in the subnormal range,
// below 2^-1022, that a scaling by 1/4 would round).
__device__ __forceinline__ double fma2(double k, double v, double x) { return __fma_rn(k, v, x); }

// Two correctly rounded operations of WENO5 computed from the IEEE 754
// binary64 fields on the integer pipes (GB300's FP64 pipe retires two
// operations per SM and clock): the product of v by a small odd integer K and
// the quotient x/6, both on 32-bit words (32-bit multiplies, multiply-highs,
// shifts and adds; no floating-point or 64-bit integer instruction).  Same bits as the FP64 operation for every input: zeros
// are returned directly, and subnormal, infinite or NaN operands and results
// near the exponent limits take the FP64 instruction.
//
// K v: with v = +-M 2^(e-1075), M in [2^52, 2^53), the product M K has 54 to
// 57 bits; it is rounded to 53 bits (ties to even) by adding 2^(s-1) - 1 plus
// the lowest kept bit before the shift by s.  The rounded significand (up to
// 2^53) is added onto the shifted exponent field, so a carry out of the
// significand raises the exponent.
template <unsigned K>
__device__ __forceinline__ double mul_small(double v) {
    static_assert(K % 2 == 1 && K >= 3 && K <= 15, "odd factor 3..15");
    constexpr unsigned S0 = K < 4 ? 1 : (K < 8 ? 2 : 3);   // M K in [2^(52+S0), 2^(54+S0))
    const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
    const unsigned e = (hi >> 20) & 0x7ffu;
    // subnormals, |v| >= 2^1019, infinities and NaNs
    if (__builtin_expect(e > 2041u || (e == 0u && ((hi << 1) | lo) != 0u), 0)) return (double)K * v;
    // P = M K in two 32-bit words (M = mh:lo): no 64-bit integer instruction
    const unsigned mh = (hi & 0x000fffffu) | 0x00100000u;
    const unsigned pl = lo * K;
    const unsigned ph = mh * K + __umulhi(lo, K);
    const unsigned s = S0 + ((ph >> (21 + S0)) & 1u);   // P >= 2^(53+S0): one more bit to drop
    const unsigned add = ((1u << (s - 1u)) - 1u) + ((pl >> s) & 1u);
    const unsigned nl = pl + add;
    const unsigned nh = ph + (nl < pl ? 1u : 0u);
    const unsigned rl = __funnelshift_r(nl, nh, s), rh = nh >> s;
    const bool zero = e == 0u;   // +-0: K 0 = 0 with the sign kept
    const unsigned oh = zero ? hi : (hi & 0x80000000u) + ((e + s - 1u) << 20) + rh;
    const unsigned ol = zero ? lo : rl;
    return __hiloint2double((int)oh, (int)ol);
}

// x/6: with x = +-M 2^(e-1075), x/6 = +-(M 2^k / 3) 2^(e-1076-k), where k = 2
// for M < 3 2^51 and k = 1 otherwise puts M 2^k / 3 in [2^52, 2^53).  A third
// of an integer is never halfway between two integers, so the round-to-nearest
// significand is floor((M 2^k + 1) / 3) and never reaches 2^53.
__device__ __forceinline__ double div6(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    const unsigned e = (hi >> 20) & 0x7ffu;
    if (__builtin_expect(e == 2047u || (e < 4u && ((hi << 1) | lo) != 0u), 0)) return x / 6.0;
    // N = M 2^k + 1 in two 32-bit words (M = mh:lo), then N / 3 word by word:
    // H = 3 q1 + r1, L = 3 qL + rL and 2^32 = 3 * 1431655765 + 1 give
    // N / 3 = q1 2^32 + r1 * 1431655765 + qL + (r1 + rL >= 3), whose low word never carries
    const unsigned mh = (hi & 0x000fffffu) | 0x00100000u;
    const unsigned k = mh < 0x00180000u ? 2u : 1u;
    const unsigned L = (lo << k) | 1u, H = __funnelshift_l(lo, mh, k);
    const unsigned q1 = __umulhi(H, 0xAAAAAAABu) >> 1, r1 = H - 3u * q1;
    const unsigned qL = __umulhi(L, 0xAAAAAAABu) >> 1, rL = L - 3u * qL;
    const unsigned q0 = r1 * 1431655765u + qL + (r1 + rL >= 3u ? 1u : 0u);
    const bool zero = e == 0u;   // +-0 (subnormals took the division)
    const unsigned oh = zero ? hi : (hi & 0x80000000u) + ((e - 2u - k) << 20) + q1;
    const unsigned ol = zero ? lo : q0;
    return __hiloint2double((int)oh, (int)ol);
}

// The curvature term of a Jiang-Shu smoothness indicator on the three cells
// a, b, c: 13/12 (a - 2 b + c)^2.  The stencil {i-1, i, i+1} gives beta_1 of
// cell i, beta_2 of cell i-1 and beta_0 of cell i+1 the same term, formed
// from the same three values in the same order -- the same bits -- so a sweep
// that slides along a pencil can form it once per cell and pass it on.
__device__ __forceinline__ double curv(double a, double b, double c) {
    const double c13 = 13.0 / 12.0;
    const double x = fma2(-2.0, b, a) + c;
    bool ok = true;
    double t = sq_i(x, ok);
    t = mul_i(c13, t, ok);
    if (__builtin_expect(!ok, 0)) t = c13 * sq(x);
    return t;
}

// Both faces' values of WENO5 from x_k, the odd parts' arguments of the three
// smoothness indicators (beta_k = 1/4 x_k^2 + t_k), and the candidates p (left
// face) and r (right face): weights a_k = d_k / (eps + beta_k)^2 with d = (0.1,
// 0.6, 0.3) and (0.3, 0.6, 0.1), omega_k = a_k / sum(a), face value
// sum omega_k p_k.  Plain FP64 for operands out of the integer forms' range.
static __device__ __noinline__ void weno5_faces_any(double eps, const double* x, const double* t, const double* p,
                                                    const double* r, double* out) {
    double s[3];
    for (int k = 0; k < 3; ++k) s[k] = sq(eps + fma2(0.25, sq(x[k]), t[k]));
    const double a0 = 0.1 / s[0], a1 = 0.6 / s[1], a2 = 0.3 / s[2], e0 = 0.3 / s[0], e2 = 0.1 / s[2];
    const double sm = a0 + a1 + a2, sp = e0 + a1 + e2;
    out[0] = a0 / sm * p[0] + a1 / sm * p[1] + a2 / sm * p[2];
    out[1] = e0 / sp * r[0] + a1 / sp * r[1] + e2 / sp * r[2];
}

__device__ __forceinline__ void weno5_faces(double eps, const double* x, const double* t, const double* p,
                                            const double* r, double& vm, double& vp) {
    bool ok = true;
    // d_k / s_k of both faces (d_1 is the same at both), one indicator a pass,
    // then the weighted sum, one face a pass: the loops are not unrolled, so
    // that the code of a reconstruction stays in the instruction caches
    double x0 = x[0], x1 = x[1], t0 = t[0], t1 = t[1], dm = 0.1, dp = 0.3;
    double m0 = 0.0, m1 = 0.0, m2 = 0.0, p0 = 0.0, p1 = 0.0, p2 = 0.0;
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        const double e = eps + fma2(0.25, sq_i(x0, ok), t0);
        ok = ok && in_range<150>(e);   // so that every quotient below is normal
        const RcpI y = rcp_i(sq_i(e, ok));
        m0 = m1;
        m1 = m2;
        m2 = quot_i(dm, y);
        p0 = p1;
        p1 = p2;
        p2 = quot_i(dp, y);
        x0 = x1;
        x1 = x[2];
        t0 = t1;
        t1 = t[2];
        dm = k == 0 ? 0.6 : 0.3;
        dp = k == 0 ? 0.6 : 0.1;
    }
    double q0 = p[0], q1 = p[1], q2 = p[2], v = 0.0;
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
        vm = v;
        const RcpI y = rcp_i(m0 + m1 + m2);
        v = mul_i(quot_i(m0, y), q0, ok) + mul_i(quot_i(m1, y), q1, ok) + mul_i(quot_i(m2, y), q2, ok);
        m0 = p0;
        m1 = p1;
        m2 = p2;
        q0 = r[0];
        q1 = r[1];
        q2 = r[2];
    }
    vp = v;
    if (__builtin_expect(!ok, 0)) {
        double out[2];
        weno5_faces_any(eps, x, t, p, r, out);
        vm = out[0];
        vp = out[1];
    }
}

// WENO5-JS of cell i from its window, given the curvature terms t0 = curv(v0,
// v1, v2), t1 = curv(v1, v2, v3) and t2 = curv(v2, v3, v4).  The right-face
// candidates of cell i, (-v_{i-2} + 5 v_{i-1} + 2 v_i)/6 and (2 v_{i-1} + 5 v_i
// - v_{i+1})/6, are the left-face candidates p1 and p2 of cell i-1, formed from
// the same values in the same order (the same bits): weno5_tc takes them as r0,
// r1 and returns this cell's p1, p2 for the next.
__device__ __forceinline__ void weno5_tc(double eps, double v0, double v1, double v2, double v3, double v4,
                                         double t0, double t1, double t2, double& r0, double& r1, double& vm,
                                         double& vp) {
    const double v2x3 = mul_small<3>(v2), v2x5 = mul_small<5>(v2), v2x11 = mul_small<11>(v2);
    const double x[3] = {fma2(-4.0, v1, v0) + v2x3, v1 - v3, fma2(-4.0, v3, v2x3) + v4};
    const double t[3] = {t0, t1, t2};
    const double p[3] = {div6(fma2(2.0, v0, -mul_small<7>(v1)) + v2x11),     // (2 v0 - 7 v1 + 11 v2)/6
                         div6(fma2(2.0, v3, -v1 + v2x5)),                    // (-v1 + 5 v2 + 2 v3)/6
                         div6(fma2(2.0, v2, mul_small<5>(v3)) - v4)};        // (2 v2 + 5 v3 - v4)/6
    const double r[3] = {r0, r1, div6(fma2(2.0, v4, v2x11 - mul_small<7>(v3)))};   // (11 v2 - 7 v3 + 2 v4)/6
    weno5_faces(eps, x, t, p, r, vm, vp);
    r0 = p[1];
    r1 = p[2];
}

// The right-face candidates r0, r1 of the cell whose window is v0..v3 (as in weno5_tc).
__device__ __forceinline__ void weno5_right01(double v0, double v1, double v2, double v3, double& r0, double& r1) {
    r0 = div6(fma2(2.0, v2, -v0 + mul_small<5>(v1)));
    r1 = div6(fma2(2.0, v1, mul_small<5>(v2)) - v3);
}

// WENO5-JS on a non-uniform grid from the cell's table T (kTabDoubles values, the
// same for every pencil): candidates q_k^+- = cp_k.v, cm_k.v, smoothness beta_k =
// (B_k.v)^2 + 13/3 (C_k.v)^2, linear weights dp, dm; weights in product form, one
// quotient for both faces.  The tables have their own rounding, so there is no
// reference order to keep: fused operations (128^3 with three refined
// directions 0.98 ns as sliding window, 0.58 here).
__device__ __forceinline__ void weno5_tab(const double* __restrict__ T, double v0, double v1, double v2, double v3,
                                          double v4, double eps, double& vm, double& vp) {
    const double v[5] = {v0, v1, v2, v3, v4};
    double qp[3], qm[3], s[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        auto dot = [&](int base) {
            const double* t = T + base + 3 * k;
            return __fma_rn(__ldg(t + 2), v[k + 2], __fma_rn(__ldg(t + 1), v[k + 1], __ldg(t) * v[k]));
        };
        qp[k] = dot(0);
        qm[k] = dot(9);
        const double c = dot(18), d = dot(27);
        const double e = eps + __fma_rn(c, c, 13.0 / 3.0 * (d * d));
        s[k] = e * e;
    }
    const double m0 = s[1] * s[2], m1 = s[0] * s[2], m2 = s[0] * s[1];
    const double ap0 = __ldg(T + 36) * m0, ap1 = __ldg(T + 37) * m1, ap2 = __ldg(T + 38) * m2;
    const double am0 = __ldg(T + 39) * m0, am1 = __ldg(T + 40) * m1, am2 = __ldg(T + 41) * m2;
    const double Dp = ap0 + ap1 + ap2, Dm = am0 + am1 + am2;
    const double r = quot(1.0, Dp * Dm);
    vm = __fma_rn(ap2, qp[2], __fma_rn(ap1, qp[1], ap0 * qp[0])) * Dm * r;
    vp = __fma_rn(am2, qm[2], __fma_rn(am1, qm[1], am0 * qm[0])) * Dp * r;
}

// WENO3-JS in the reference order: v1..v3 = v_{i-1}..v_{i+1}; weights
// a_k = d_k/(eps+beta_k)^2 with d = (1/3, 2/3) at i+1/2 and (2/3, 1/3) at
// i-1/2, omega_k = a_k/sum(a), candidates (.)/2 (an exact halving).
__device__ __forceinline__ void weno3(double eps, double v1, double v2, double v3, double& vm, double& vp) {
    const double c1 = 1.0 / 3.0, c2 = 2.0 / 3.0;
    double b0 = sq(v2 - v1), b1 = sq(v3 - v2);
    double s0 = sq(eps + b0), s1 = sq(eps + b1);
    const bool ok = mid_range(s0) && mid_range(s1);
    const RcpI y0 = rcp_i(s0), y1 = rcp_i(s1);
    double a0 = quot_i(c1, y0), a1 = quot_i(c2, y1), a2 = quot_i(c2, y0), a3 = quot_i(c1, y1);
    const RcpI ym = rcp_i(a0 + a1), yp = rcp_i(a2 + a3);
    double w0 = quot_i(a0, ym), w1 = quot_i(a1, ym), w2 = quot_i(a2, yp), w3 = quot_i(a3, yp);
    if (__builtin_expect(!ok, 0)) {
        a0 = div_any(c1, s0);
        a1 = div_any(c2, s1);
        a2 = div_any(c2, s0);
        a3 = div_any(c1, s1);
        const double sm = a0 + a1, sp = a2 + a3;
        w0 = div_any(a0, sm);
        w1 = div_any(a1, sm);
        w2 = div_any(a2, sp);
        w3 = div_any(a3, sp);
    }
    double p0 = (-v1 + 3.0 * v2) * 0.5;
    double p1 = (v2 + v3) * 0.5;
    vm = w0 * p0 + w1 * p1;
    p0 = (v1 + v2) * 0.5;
    p1 = (3.0 * v2 - v3) * 0.5;
    vp = w2 * p0 + w3 * p1;
}

struct Face {
    double rho, p, G, Pi, E;
};

// Physical flux of side K (primitives w, face state K) normal to DIR; the
// volume-fraction slots carry alpha_i,K u_n.
template <int NDIM, int DIR, int NF = 2>
__device__ __forceinline__ void phys_flux(const double* w, const Face& K, double* F) {
    using FL = Fields<NDIM, NF>;
    double un = w[FL::IU + DIR];
#pragma unroll
    for (int i = 0; i < NF; ++i) F[i] = w[i] * un;
#pragma unroll
    for (int k = 0; k < NDIM; ++k) F[FL::IU + k] = K.rho * w[FL::IU + k] * un;
    F[FL::IU + DIR] = F[FL::IU + DIR] + K.p;
    F[FL::IE] = (K.E + K.p) * un;
#pragma unroll
    for (int i = 0; i < FL::NA; ++i) F[FL::IA + i] = w[FL::IA + i] * un;
}

// HLLC flux through a face normal to DIR; regions 0<=S_L: F_L, S_L<0<=S*: F*_L,
// S*<0<=S_R: F*_R, else F_R; the alpha1 slot carries alpha1_K times the
// region velocity, returned in uf.  Returns true for a non-physical face state.
// The states are read from wL[f * fs] and wR[f * fs] (shared memory), first
// side by side for the wave speeds -- one pass of a loop each, so that the
// instruction caches hold one copy of a side's code -- then the selected side.
template <int NDIM, int DIR, int NF = 2>
__device__ __forceinline__ bool hllc(const Eos& e, const double* wL, const double* wR, int fs, double* F, double& uf) {
    using FL = Fields<NDIM, NF>;
    Face L{}, R{};
    double aL = 0.0, aR = 0.0, bL = 0.0, bR = 0.0, uL = 0.0, uR = 0.0;
    bool bad = false;
    const double* s = wL;
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
        L = R;
        aL = aR;
        bL = bR;
        uL = uR;
        double rho[NF], al[FL::NA];
#pragma unroll
        for (int i = 0; i < NF; ++i) rho[i] = s[i * fs];
#pragma unroll
        for (int i = 0; i < FL::NA; ++i) al[i] = s[(FL::IA + i) * fs];
        R.rho = mix_rho<NF>(rho);
        R.p = s[FL::IE * fs];
        mixture<NF>(MulFp(), e, al, R.G, R.Pi);
        const double c2 = sound2(MulFp(), R.G, R.Pi, R.rho, R.p);
        bad = bad || !gt0(R.rho) || !gt0(c2);
        const double c = sqrt_p(c2);
        uR = s[(FL::IU + DIR) * fs];
        aR = uR - c;
        bR = uR + c;
        s = wR;
    }
    double SL = less(aL, aR) ? aL : aR;
    double SR = less(bR, bL) ? bL : bR;
    double num = R.p - L.p + L.rho * uL * (SL - uL) - R.rho * uR * (SR - uR);
    double den = L.rho * (SL - uL) - R.rho * (SR - uR);
    double Ss = quot(num, den);
    const bool left = ge0(SL) || ge0(Ss);
    const bool star = left ? !ge0(SL) : ge0(SR);
    s = left ? wL : wR;
    double w[FL::NEQ];
#pragma unroll
    for (int f = 0; f < FL::NEQ; ++f) w[f] = s[f * fs];
    Face K;
    K.rho = left ? L.rho : R.rho;
    K.p = left ? L.p : R.p;
    K.G = left ? L.G : R.G;
    K.Pi = left ? L.Pi : R.Pi;
    K.E = K.G * K.p + K.Pi + kinetic<NDIM>(MulFp(), K.rho, w + FL::IU);   // of the selected side only
    double SK = left ? SL : SR;
    double un = w[FL::IU + DIR];
    phys_flux<NDIM, DIR, NF>(w, K, F);
    uf = un;
    if (star) {
        double chi = quot(SK - un, SK - Ss);
#pragma unroll
        for (int i = 0; i < NF; ++i) F[i] = F[i] + SK * (chi * w[i] - w[i]);
#pragma unroll
        for (int k = 0; k < NDIM; ++k) {
            double mstar = (k == DIR) ? chi * K.rho * Ss : chi * K.rho * w[FL::IU + k];
            F[FL::IU + k] = F[FL::IU + k] + SK * (mstar - K.rho * w[FL::IU + k]);
        }
        double Estar = chi * (K.E + (Ss - un) * (K.rho * Ss + quot(K.p, SK - un)));
        F[FL::IE] = F[FL::IE] + SK * (Estar - K.E);
#pragma unroll
        for (int i = 0; i < FL::NA; ++i) F[FL::IA + i] = w[FL::IA + i] * Ss;
        uf = Ss;
    }
    return bad;
}

// S contribution of one cell: sum_d (|u_d| + c)/dx_d, from the conservative state.
template <int NDIM, int NF = 2, typename M = MulFp>
__device__ __forceinline__ double cell_wavespeed(const Eos& e, const double* q, const double* dx,
                                                 const double* rdx, bool& bad, const M& mul = M()) {
    using FL = Fields<NDIM, NF>;
    double w[FL::NEQ];
    cons_to_prim<NDIM, NF>(e, q, w, mul);
    double rho = mix_rho<NF>(w);
    double G, Pi;
    mixture<NF>(mul, e, w + FL::IA, G, Pi);
    double c2 = sound2(mul, G, Pi, rho, w[FL::IE]);
    bad |= !gt0(mix_rho<NF>(q)) || !gt0(rho) || !gt0(c2);
    const double cs = sqrt_p(c2);
    double s = 0.0;
#pragma unroll
    for (int d = 0; d < NDIM; ++d) s = s + div_rcp(fabs(w[FL::IU + d]) + cs, dx[d], rdx[d]);
    bad |= !less(s, INFINITY);
    return s;
}

}  // namespace exact
}  // namespace mfc5
