// sweep_df.cuh -- the TRT collision of Sec. III, Eq. "lb", for FP64 storage,
// computed in double-float arithmetic: every quantity is an unevaluated sum
// h + l of two FP32 numbers, carried by error-free transformations (Knuth's
// two-sum for additions, Dekker's product through FMA for multiplications).
//
// Why: GB300 issues FP64 arithmetic at about 2 lanes per SM and cycle against
// 128 for FP32.  A TRT update in FP64 is about 130 FP64 instructions per cell,
// which caps the FP64 sweep near a fifth of its HBM roofline.  The same update
// in double-float takes about 900 FP32 operations, issued two at a time.
//
// Precision: FP64 storage holds the deviations g_i = f_i - w_i rho0, whose
// magnitude is that of the flow (|g| ~ 1e-3 here), not of f (~0.05 .. 1/3).
// The arithmetic carries about 47 significant bits of g, i.e. an absolute
// error near 2^-47 |g| per operation: below the rounding of f itself in FP64
// (ulp(1/3) / 2 = 2^-55), which is what the FP64 oracle carries.
//
// The conversions between an FP64 word and a pair run in integer arithmetic
// on the bit pattern (no FP64 instruction at all):
//   load:  h = the FP64 value truncated to 24 significant bits (exponent
//          rebiased 1023 -> 127), l = the remaining 29 mantissa bits, rounded
//          to 24 bits, with h's sign and exponent;
//   store: s = h + l rounded toward zero, e = (h + l) - s (same sign as s),
//          then the FP64 bits of s plus e counted in FP64 ulps of s.
// Magnitudes are clamped to [2^-126, 2^101) on load (deviations below 1e-38
// are zero for every purpose here); a cell whose density or momentum is not
// finite after that (NaN or Inf populations) stores NaN, so a diverged state
// stays visible to the mass sum and the body update.
#pragma once

#include <cstdint>

namespace lbsq {

// hi/lo parts of the collision's constants (DfK indices below), for DfK::h/l
enum DfIdx : int {
    DK_W18 = 0,  // 1/18
    DK_W3,       // 1/3
    DK_LW18,     // 3 lo / 18
    DK_LW36,     // 3 lo / 36
    DK_CH,       // (1 - lo) / 2
    DK_LE,       // le
    DK_LE3,      // le / 3
    DK_1MLE,     // 1 - le
    DK_CS,       // (1 - le) / 2
    DK_RHO0,     // rho0
    DK_IRHO0,    // 1 / rho0
    DK_N
};
struct DfK {
    float h[DK_N], l[DK_N];
    int le1;  // le == 1: the even part relaxes fully
};
__host__ __device__ inline void df_split(double v, float& h, float& l) {
    h = (float)v;
    l = (float)(v - (double)h);
}
__host__ __device__ inline DfK df_constants(double le, double lo, double rho0) {
    const double v[DK_N] = {1.0 / 18.0, 1.0 / 3.0, 3.0 * lo / 18.0, 3.0 * lo / 36.0, 0.5 * (1.0 - lo), le,
                            le / 3.0,   1.0 - le,  0.5 * (1.0 - le), rho0,            1.0 / rho0};
    DfK k;
    for (int i = 0; i < DK_N; ++i) df_split(v[i], k.h[i], k.l[i]);
    k.le1 = (1.0 - le) == 0.0;
    return k;
}

struct df {
    float h, l;
};

// ---- error-free transformations (every rounding explicit: no contraction)

// a + b = s + e exactly (Knuth), for any a, b
__device__ __forceinline__ df two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return {s, e};
}
// x + y: the exact sum of the high parts plus the low parts, left
// unnormalised (|l| grows by an ulp of the operands per addition)
__device__ __forceinline__ df dadd(df x, df y) {
    df s = two_sum(x.h, y.h);
    s.l = __fadd_rn(s.l, __fadd_rn(x.l, y.l));
    return s;
}
__device__ __forceinline__ df dneg(df x) { return {-x.h, -x.l}; }
__device__ __forceinline__ df dsub(df x, df y) { return dadd(x, dneg(y)); }
// x * y: the exact product of the high parts (Dekker, through FMA) plus the
// cross terms.  The product of the low parts is left out: with |l| within a
// few ulps of |h| it is below 2^-46 of |x y|, the size of the rounding of the
// low parts themselves.
__device__ __forceinline__ df dmul(df x, df y) {
    const float p = __fmul_rn(x.h, y.h);
    float e = __fmaf_rn(x.h, y.h, -p);
    e = __fmaf_rn(x.h, y.l, e);
    e = __fmaf_rn(x.l, y.h, e);
    return {p, e};
}
__device__ __forceinline__ df dsqr(df x) {
    const float p = __fmul_rn(x.h, x.h);
    const float t = __fadd_rn(x.h, x.h);
    float e = __fmaf_rn(x.h, x.h, -p);
    e = __fmaf_rn(t, x.l, e);
    return {p, e};
}
// x * c for an FP32 c
__device__ __forceinline__ df dmulf(df x, float c) {
    const float p = __fmul_rn(x.h, c);
    float e = __fmaf_rn(x.h, c, -p);
    e = __fmaf_rn(x.l, c, e);
    return {p, e};
}
// x * 2^k (exact)
__device__ __forceinline__ df dpow2(df x, float p2) { return {__fmul_rn(x.h, p2), __fmul_rn(x.l, p2)}; }
// |l| <= ulp(h) / 2 (Fast2Sum)
__device__ __forceinline__ df dnorm(df x) {
    const float s = __fadd_rn(x.h, x.l);
    return {s, __fsub_rn(x.l, __fsub_rn(s, x.h))};
}
// 1 / x for x near 1 (a density): FP32 estimate, one FP32 Newton step
// (relative error ~2^-24), then one step in double-float (error squared)
__device__ __forceinline__ df drcp(df x) {
    float r;
    asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x.h));
    r = __fmaf_rn(r, __fmaf_rn(-x.h, r, 1.0f), r);
    float e = __fmaf_rn(-x.h, r, 1.0f);  // 1 - x r, small: one rounding of itself
    e = __fmaf_rn(-x.l, r, e);
    return {r, __fmul_rn(r, e)};
}
__device__ __forceinline__ df dk(const DfK& K, int i) { return {K.h[i], K.l[i]}; }

// ---- FP64 word <-> double-float pair, in integer arithmetic

// (lo, hi) = the two 32-bit words of an FP64 value
__device__ __forceinline__ df df_from_bits(unsigned lo, unsigned hi) {
    const unsigned sign = hi & 0x80000000u;
    unsigned a = hi & 0x7fffffffu;
    a = umax(a, 897u << 20);                  // |g| >= 2^-126
    a = umin(a, (1124u << 20) - 1u);          // |g| < 2^101
    // exponent 1023 -> 127 and the top 23 mantissa bits: a truncated float
    const unsigned hb = __funnelshift_l(lo, a - (896u << 20), 3) | sign;
    // the remaining 29 bits weigh 2^(e - 52), e the unbiased exponent
    const float rem = __uint2float_rn(lo & 0x1fffffffu);
    const float pw = __uint_as_float(hb & 0xff800000u);  // +-2^e
    return {__uint_as_float(hb), __fmul_rn(__fmul_rn(rem, pw), 0x1p-52f)};
}
// FP64 bits of h + l (to ~2^-47 relative; |h + l| below 2^-75 may come out
// as any value of that size)
__device__ __forceinline__ uint2 df_to_bits(df x) {
    const float s = __fadd_rz(x.h, x.l);                  // |s| <= |h + l|
    const float e = __fsub_rn(x.l, __fsub_rn(s, x.h));    // (h + l) - s
    const unsigned sb = __float_as_uint(s), ab = sb & 0x7fffffffu;
    unsigned hi = ((ab >> 3) + (896u << 20)) | (sb & 0x80000000u);
    unsigned lo = sb << 29;
    // e in FP64 ulps of s, 2^(es - 127 - 52): fewer than 2^29 of them, so the
    // 52-bit mantissa cannot overflow.  For |s| < 2^-75 the scale's exponent
    // field wraps (or is Inf): the count is then garbage, an error below
    // 2^-75 in absolute value.
    const float pw = __uint_as_float((306u << 23) - (sb & 0x7f800000u));  // 2^(179 - es)
    const unsigned k = __float2uint_rn(__fmul_rn(fabsf(e), pw));
    asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(lo), "+r"(hi) : "r"(k));
    return make_uint2(lo, hi);
}

// ---- two double-float numbers at a time
//
// GB300 retires add/mul/fma.f32x2 (two FP32 operations per instruction), and
// with one operation per instruction the sweep was bound by instruction issue
// (76 % of the slots busy, FMA pipe 51 %), so the collision carries its
// direction pairs two by two; every half rounds as the scalar operation would.
// Whole sweeps on GB300, scalar -> in pairs: 256^3 891 -> 830 us (0.90 of the
// 6.8 TB/s copy rate), 128^3 107 -> 100 us.
struct df2 {
    unsigned long long h, l;
};
__device__ __forceinline__ unsigned long long f2_pack(float a, float b) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_unpack(unsigned long long v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ unsigned long long f2_add(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long f2_sub(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long f2_mul(unsigned long long a, unsigned long long b) {
    unsigned long long r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ unsigned long long f2_fma(unsigned long long a, unsigned long long b,
                                                     unsigned long long c) {
    unsigned long long r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ df2 pack(df a, df b) { return {f2_pack(a.h, b.h), f2_pack(a.l, b.l)}; }
__device__ __forceinline__ df2 splat(df a) { return pack(a, a); }
__device__ __forceinline__ void unpack(df2 v, df& a, df& b) {
    f2_unpack(v.h, a.h, b.h);
    f2_unpack(v.l, a.l, b.l);
}
__device__ __forceinline__ df2 dadd(df2 x, df2 y) {
    const unsigned long long s = f2_add(x.h, y.h);
    const unsigned long long bb = f2_sub(s, x.h);
    const unsigned long long e = f2_add(f2_sub(x.h, f2_sub(s, bb)), f2_sub(y.h, bb));
    return {s, f2_add(e, f2_add(x.l, y.l))};
}
__device__ __forceinline__ df2 dsub(df2 x, df2 y) {
    const unsigned long long s = f2_sub(x.h, y.h);
    const unsigned long long bb = f2_sub(s, x.h);
    const unsigned long long e = f2_sub(f2_sub(x.h, f2_sub(s, bb)), f2_add(y.h, bb));
    return {s, f2_add(e, f2_sub(x.l, y.l))};
}
__device__ __forceinline__ df2 dmul(df2 x, df2 y) {
    const unsigned long long p = f2_mul(x.h, y.h);
    unsigned long long e = f2_fma(x.h, y.h, p ^ 0x8000000080000000ull);
    e = f2_fma(x.h, y.l, e);
    e = f2_fma(x.l, y.h, e);
    return {p, e};
}
__device__ __forceinline__ df2 dsqr(df2 x) {
    const unsigned long long p = f2_mul(x.h, x.h);
    const unsigned long long t = f2_add(x.h, x.h);
    unsigned long long e = f2_fma(x.h, x.h, p ^ 0x8000000080000000ull);
    e = f2_fma(t, x.l, e);
    return {p, e};
}
__device__ __forceinline__ df2 dpow2(df2 x, float p2) {
    const unsigned long long q = f2_pack(p2, p2);
    return {f2_mul(x.h, q), f2_mul(x.l, q)};
}

// TRT collision (Sec. III) of one cell on deviations g_i = f_i - w_i rho0, in
// the pair form of collide_trt (sweep_body.cuh): with s = g_i + g_ib and
// d = g_i - g_ib for the nine pairs, sigma = sum g, rho = rho0 + sigma,
//   base = sigma - 3/2 |j|^2 / rho   (incompressible: / rho0),
//   ep   = w base + 9/2 w (c.j)^2 / rho,
//   g_0 += le (base / 3 - g_0),  g_i = q + h,  g_ib = q - h,
//   q = le ep + (1 - le)/2 s,  h = 3 lo w c.j + (1 - lo)/2 d
// (g_i + E + O with g_i = (s + d)/2 and the relaxations E = le (ep - s/2),
// O = 3 lo w c.j - lo/2 d).  le = 1: g_0 = base / 3, q = ep, and s is only
// summed.
// LE1: le == 1 (K.le1), the form taken.  Returns false when the cell's
// density or momentum is not finite.
//
// The nine direction pairs p (first members 2p - 1) are taken as x alone,
// (y, z), and the edges as (xy+, xz+), (xy-, xz-), (yz+, yz-): then the momentum
// and c.j of two pairs come from one operation each,
//   (jy, jz) = (d_y, d_z) + (d_xy+ - d_xy-, d_xz+ - d_xz-)
//              + (d_yz+ + d_yz-, d_yz+ - d_yz-),
//   c.j = jx +- (jy, jz) for the first two edge groups, jy +- jz for the third.
// first member's index in g of group q's pair k
__host__ __device__ constexpr int df_i(int q, int k) {
    return 2 * (q == 0 ? 2 + k : (q == 1 ? 4 + 2 * k : (q == 2 ? 5 + 2 * k : 8 + k))) - 1;
}
template <bool LE1>
__device__ __forceinline__ bool collide_trt_df(df g[Q], const DfK& K, int inc) {
    df2 s[4], d[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int a = df_i(q, 0), b = df_i(q, 1);
        const df2 u = pack(g[a], g[b]), v = pack(g[a + 1], g[b + 1]);
        s[q] = dadd(u, v);
        d[q] = dsub(u, v);
    }
    const df s1 = dadd(g[1], g[2]), d1 = dsub(g[1], g[2]);
    df sa, sb;
    unpack(dadd(dadd(s[0], s[1]), dadd(s[2], s[3])), sa, sb);
    const df sum = dnorm(dadd(dadd(g[0], s1), dadd(sa, sb)));
    df xp, xq, e8, e9, jy, jz;
    unpack(dadd(d[1], d[2]), xp, xq);  // d_xy+ + d_xy-, d_xz+ + d_xz-
    const df jx = dnorm(dadd(dadd(d1, xp), xq));
    unpack(d[3], e8, e9);
    unpack(dadd(dadd(d[0], dsub(d[1], d[2])), dadd(pack(e8, e8), pack(e9, dneg(e9)))), jy, jz);
    jy = dnorm(jy);
    jz = dnorm(jz);
    const df j2 = dadd(dadd(dsqr(jx), dsqr(jy)), dsqr(jz));
    const bool ok = fabsf(sum.h) < 0x1p60f && j2.h < 0x1p100f;
    const df inv = inc ? dk(K, DK_IRHO0) : drcp(dnorm(dadd(dk(K, DK_RHO0), sum)));
    const df ju = dmul(j2, inv);                       // rho u.u
    const df base = dnorm(dsub(sum, dmulf(ju, 1.5f)));  // sigma - 3/2 rho u.u
    const df wb18 = dmul(base, dk(K, DK_W18)), wb36 = dpow2(wb18, 0.5f);
    const df lw18 = dk(K, DK_LW18), lw36 = dk(K, DK_LW36);
    const df2 jyz = pack(jy, jz), jxx = splat(jx), inv2 = splat(inv);
    const df2 cj[4] = {jyz, dadd(jxx, jyz), dsub(jxx, jyz), dadd(splat(jy), pack(jz, dneg(jz)))};
    // ep = w base + 9/2 w (c.j)^2 / rho; 9/2 w = 1/4 (faces), 1/8 (edges)
    const df ep1 = dadd(dpow2(dmul(dsqr(jx), inv), 0.25f), wb18);
    if constexpr (LE1) g[0] = dmul(base, dk(K, DK_W3));
    else g[0] = dadd(dmul(dk(K, DK_LE3), base), dmul(dk(K, DK_1MLE), g[0]));
    const df ch = dk(K, DK_CH), le = dk(K, DK_LE), cs = dk(K, DK_CS);
    const df2 ch2 = splat(ch), lwf = splat(lw18), lwe = splat(lw36), wbf = splat(wb18), wbe = splat(wb36);
    const df h1 = dadd(dmul(lw18, jx), dmul(ch, d1));
    const df q1 = LE1 ? ep1 : dadd(dmul(le, ep1), dmul(cs, s1));
    g[1] = dadd(q1, h1);
    g[2] = dsub(q1, h1);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int a = df_i(q, 0), b = df_i(q, 1);
        df2 e = dadd(dpow2(dmul(dsqr(cj[q]), inv2), q == 0 ? 0.25f : 0.125f), q == 0 ? wbf : wbe);
        if constexpr (!LE1) e = dadd(dmul(splat(le), e), dmul(splat(cs), s[q]));
        const df2 h = dadd(dmul(q == 0 ? lwf : lwe, cj[q]), dmul(ch2, d[q]));
        unpack(dadd(e, h), g[a], g[b]);
        unpack(dsub(e, h), g[a + 1], g[b + 1]);
    }
    return ok;
}

}  // namespace lbsq
