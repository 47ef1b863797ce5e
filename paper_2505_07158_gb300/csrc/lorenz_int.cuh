// One RK4 step of Eq. (1) on the integer pipes, bit-identical to the binary64 step.
//
// Why.  A binary64 instruction holds its sub-partition's pipe for 64 cycles whatever the number of active
// lanes, and every rounded operation of the step waits for the one before: the step of chaos_dev.cuh is 27
// such instructions and four exchanges, ~2.1k cycles, with the integer pipes idle.  The same roundings on
// the integer pipes take ~20 cycles each.  Measured on GB300, the records of one 1080p frame (8,124 steps, one
// warp): 6.21 ms, 1,580 cycles a step with the binary64 redoes below, against 8.53 ms.  What bounds it now is one
// warp's issue: ~110 integer instructions a stage at two cycles each on a chain of ~235 cycles (exchange 50,
// A B 60, k 25, c k 60, tin 40).
//
// Representation.  The four lanes of a chain hold one variable each.  A variable, and every sum of the step
// (T1, T2, k, acc, tin), is a 64-bit two's complement integer on its lane's grid 2^-G (G = 62 for x, y, z
// and 60 for w), modulo 2^64: exact, since every rounded value of at least 2^(53-G) is a multiple of its own
// ulp >= 2^(1-G).  Binary64 rounding of such a sum is rounding to nearest even at bit p = e - 52 + G, with e
// the exponent of the sum; e comes from a float shadow of the sum, which is a few cycles ahead of it.  A
// product takes its factors as 53-bit integers N (value N 2^(e-52), N = n1 2^32 + n0 with a signed low
// digit), is formed exactly, rounded half up at bit 52 or 53 (the shadow says which) and shifted onto the
// grid.  The bits of a sum above its 64 come from the shadow too.  The z lane holds -z, so that every
// component is T1 = M1 a - own1 + T, T2 = M2 T1 - own2, k = T2 + A B with non-negative M1 and M2:
//   x: a = y, own1 = x, M2 = 10, A B = 1 w;   y: a = x, M1 = 28, own2 = y, A B = x (-z);
//   z (-z, k as it is, c negated): T = beta (-z), A B = x y;   w: T = gamma w, A B = y (-z).
//
// What makes it exact.  Each shadow has an error bound (IntStepTab, by interval arithmetic over the four
// stages for |x|, |y| < 32, |z| < 64, |w| < 256); a shadow within its bound of a power of two or of the
// smallest magnitude its grid carries, a variable outside those ranges, and a factor whose low 26 bits are
// zero (only then could a product be a tie) mark the step, and a marked step is done again in binary64.  On
// the attractor that is about 2 % of the steps at h = 0.01.  Three constants of the step (h/2, h, h/6) and gamma
// have to be in range for the shifts (IntStepTab::ok, int_gamma_ok); otherwise every step is binary64.
#pragma once
#include "common.cuh"

namespace fhd {
namespace {

constexpr int kGridXYZ = 62, kGridW = 60;
// Scale of a lane's shadows: 2^kappa with (exponent field of a shadow) mod 32 = the rounding bit p.
constexpr int kKappaXYZ = 11, kKappaW = 9;   // (G - 52 - 127) mod 32

struct IntLimbs {
    int n0, n1;   // N = n1 2^32 + n0
    float f;      // shadow: value 2^kappa
};

// A lane's variable: its fixed-point value and its limbs.
struct IntVar {
    uint32_t v0, v1;
    IntLimbs l;
};

// Constants of a lane.
struct IntLane {
    uint32_t M1, M2, own1, own2;       // own1, own2: -1 where the lane's own value is subtracted, else 0
    float fM1, fM2, fo1, fo2;
    int t0, t1;                        // limbs of the constant of T (0 on the x and y lanes)
    float tf;
    uint32_t t_half, t_place, q_half, q_place;   // shift amounts of the products, less the exponent fields
    float q_scale, above;              // scale of the shadow of A B; 2^-(64 - G + kappa)
    float d1, d2, dt, qA, qB;          // shadow error bounds
    int c0[3], c1[3];                  // limbs of h/2, h, h/6 (negated on the z lane)
    float cf[3];
    uint32_t c_half[3], c_place[3];
    float limit;                       // the variable's range, scaled
    uint32_t amask, aone1, aonef;      // A is 1.0 on the x lane
    int sa, sA, sB;                    // source lanes of a, A and B
    uint32_t expo;                     // 127 + kappa
    int grid;
    bool negated;
};

struct IntMarks {
    uint32_t m;      // exponent or sign bits that differ: a shadow near a power of two
    float least, most;
    bool few_bits;
};

struct IntProduct {
    uint32_t g0, g1, g2;
};

__device__ __forceinline__ uint32_t fbits(float f) { return __float_as_uint(f); }
__device__ __forceinline__ uint64_t pack64(uint32_t lo, uint32_t hi) { return ((uint64_t)hi << 32) | lo; }

// 53-bit significand with sign of a binary64 as signed digits, and its exponent; false for zero, subnormal,
// infinite and NaN.
__device__ __forceinline__ bool split_double(double d, bool negate, int &n0, int &n1, int &e) {
    const uint32_t h = (uint32_t)__double2hiint(d), l = (uint32_t)__double2loint(d);
    const uint32_t eb = (h >> 20) & 0x7ff;
    const long long a = (long long)pack64(l, (h & 0xfffff) | 0x100000);
    const long long N = ((h >> 31) != 0) != negate ? -a : a;
    n0 = (int)(uint32_t)N;
    n1 = (int)((N - (long long)n0) >> 32);
    e = (int)eb - 1023;
    return eb - 1 < 0x7fe;
}

// The product of two significands divided by 2^32, rounded half up at the bit of 2 half (bit 20 or 21) and
// with the bits below it cleared.
__device__ __forceinline__ IntProduct int_product(int a0, int a1, int b0, int b1, uint32_t half) {
    const int lh = __mulhi(a0, b0);
    const long long mid = (long long)a0 * b1 + (long long)a1 * b0;
    const long long Z = mid + ((long long)lh + (long long)half);
    const uint32_t z0 = (uint32_t)Z;
    const int z1 = (int)(Z >> 32);
    const long long hi = (long long)a1 * b1;
    IntProduct g;
    g.g0 = z0 & (0u - 2u * half);
    const long long H = hi + (long long)z1;
    g.g1 = (uint32_t)H;
    g.g2 = (uint32_t)(H >> 32);
    return g;
}

// Marks the step when |f| is within d of a power of two; returns |f| - d, the least magnitude it can have.
__device__ __forceinline__ float int_check(IntMarks &b, float f, float d) {
    const float a = fabsf(f), l = __fadd_rn(a, -d);
    b.m |= fbits(__fadd_rn(a, d)) ^ fbits(l);
    return l;
}
// The least magnitude that a grid carries is 4 in every lane's scale (checked once, in int_step).
__device__ __forceinline__ void int_least(IntMarks &b, float l) { b.least = fminf(b.least, l); }

__device__ __forceinline__ uint32_t low_mask(uint32_t x) {   // 2^(x mod 32) - 1
    uint32_t m;
    asm("bmsk.wrap.b32 %0, 0, %1;" : "=r"(m) : "r"(x));
    return m;
}

// Round to nearest even at bit x mod 32: add half a unit less one and the bit above it, clear the rest.
// Returns the low word before clearing (enough for a shift by x).
__device__ __forceinline__ uint32_t int_round(uint32_t &v0, uint32_t &v1, uint32_t x) {
    const uint32_t um = low_mask(x), t = __funnelshift_r(v0, 0, x) & 1;
    uint32_t a, b;
    asm("{.reg .u32 p; add.u32 p, %4, %5; add.cc.u32 %0, %2, p; addc.u32 %1, %3, 0;}"
        : "=&r"(a), "=&r"(b)
        : "r"(v0), "r"(v1), "r"(um >> 1), "r"(t));
    v0 = a & ~um;
    v1 = b;
    return a;
}
// The same carrying into the word above; sticky (0 or 1): nonzero bits below the grid.
__device__ __forceinline__ uint32_t int_round3(uint32_t &v0, uint32_t &v1, uint32_t &v2, uint32_t x, uint32_t sticky) {
    const uint32_t um = low_mask(x), t = (__funnelshift_r(v0, 0, x) & 1) | sticky;
    uint32_t a, b, c;
    asm("{.reg .u32 p; add.u32 p, %6, %7; add.cc.u32 %0, %3, p; addc.cc.u32 %1, %4, 0; addc.u32 %2, %5, 0;}"
        : "=&r"(a), "=&r"(b), "=&r"(c)
        : "r"(v0), "r"(v1), "r"(v2), "r"(um >> 1), "r"(t));
    v0 = a & ~um;
    v1 = b;
    v2 = c;
    return a;
}

// The word above a value known modulo 2^64, from its shadow: the whole number of 2^64 between them.
__device__ __forceinline__ uint32_t word_above(uint32_t v1, float f, float above) {
    const float y = __fmaf_rn(__int2float_rn((int)v1), -0x1p-32f, __fmul_rn(f, above));
    return fbits(__fadd_rn(y, 12582912.0f)) - 0x4B400000u + (uint32_t)((int)v1 >> 31);
}

// Shadow of a significand (hi:lo), with the exponent field of x: 24 bits and an odd last one, so that it never
// reaches the next binade; off by at most 2^-23 of the binade's end.
__device__ __forceinline__ float shadow_of(uint32_t lo, uint32_t hi, float x) {
    return __fmul_rn(__int2float_rn((int)(__funnelshift_l(lo, hi, 2) | 1u)),
                     __uint_as_float((fbits(x) & 0x7f800000u) - (22u << 23)));
}

// acc - (v1:v0) where m = -1, acc where m = 0, on the multiplier's pipe.
__device__ __forceinline__ uint64_t sub_masked(uint64_t acc, uint32_t v0, uint32_t v1, uint32_t m) {
    const uint64_t p = (uint64_t)v0 * m + acc;
    uint32_t hi = (uint32_t)(p >> 32);
    hi = v0 * m + hi;
    hi = v1 * m + hi;
    return pack64((uint32_t)p, hi);
}

// Stage ST of the step: from tin (t) to the next tin, or in the last stage to the next state.
template <int ST>
__device__ __forceinline__ void int_stage(const IntVar &s, IntVar &t, const IntLane &L, uint32_t &acc0, uint32_t &acc1,
                                          float &accf, float &accd, IntMarks &bad) {
    constexpr int kc = ST == 2 ? 1 : ST == 3 ? 2 : 0;
    constexpr unsigned kAll = 0xffffffffu;
    // the other variables of the chain
    IntLimbs B{__shfl_sync(kAll, t.l.n0, L.sB), __shfl_sync(kAll, t.l.n1, L.sB), __shfl_sync(kAll, t.l.f, L.sB)};
    IntLimbs A{__shfl_sync(kAll, t.l.n0, L.sA), __shfl_sync(kAll, t.l.n1, L.sA), __shfl_sync(kAll, t.l.f, L.sA)};
    const uint32_t a0 = __shfl_sync(kAll, t.v0, L.sa), a1 = __shfl_sync(kAll, t.v1, L.sa);
    const float af = __shfl_sync(kAll, t.l.f, L.sa);
    A.n0 &= (int)L.amask;
    A.n1 = (A.n1 & (int)L.amask) | (int)L.aone1;
    A.f = __uint_as_float((fbits(A.f) & L.amask) | L.aonef);
    // A B
    const uint32_t xab = (fbits(A.f) >> 23) + (fbits(B.f) >> 23);
    const float qf = __fmul_rn(__fmul_rn(A.f, L.q_scale), B.f);
    const float dq = __fmaf_rn(fabsf(A.f), L.qA, __fmul_rn(fabsf(B.f), L.qB));
    const float lq = int_check(bad, qf, dq);
    uint64_t q;
    {
        const IntProduct g = int_product(A.n0, A.n1, B.n0, B.n1, __funnelshift_l(0, 1, (fbits(qf) >> 23) - xab + L.q_half));
        const uint32_t r = L.q_place - xab;
        q = pack64(__funnelshift_r(g.g0, g.g1, r), __funnelshift_r(g.g1, g.g2, r));
    }
    // T and the own terms
    const uint32_t xo = fbits(t.l.f) >> 23;
    const float Tf = __fmul_rn(t.l.f, L.tf);
    uint64_t O1;
    {
        const IntProduct g = int_product(t.l.n0, t.l.n1, L.t0, L.t1, __funnelshift_l(0, 1, (fbits(Tf) >> 23) - xo + L.t_half));
        const uint32_t r = L.t_place - xo;
        O1 = sub_masked(pack64(__funnelshift_r(g.g0, g.g1, r), __funnelshift_r(g.g1, g.g2, r)), t.v0, t.v1, L.own1);
    }
    const uint64_t O2 = sub_masked(0, t.v0, t.v1, L.own2);
    // T1, T2, k.  The low words on their own first: the roundings' chain runs through them.
    uint64_t V = (uint64_t)a0 * L.M1 + O1;
    uint32_t w0 = a0 * L.M1 + (uint32_t)O1, w1 = (uint32_t)(V >> 32) + a1 * L.M1;
    const float T1f = __fmaf_rn(af, L.fM1, __fmaf_rn(t.l.f, L.fo1, Tf));
    const float l1 = int_check(bad, T1f, L.d1);
    int_round(w0, w1, fbits(T1f) >> 23);
    V = (uint64_t)w0 * L.M2 + O2;
    w1 = (uint32_t)(V >> 32) + w1 * L.M2;
    w0 = w0 * L.M2 + (uint32_t)O2;
    const float T2f = __fmaf_rn(T1f, L.fM2, __fmul_rn(t.l.f, L.fo2));
    int_least(bad, fminf(l1, int_check(bad, T2f, L.d2)));
    int_round(w0, w1, fbits(T2f) >> 23);
    V = pack64(w0, w1) + q;
    w0 = (uint32_t)V;
    w1 = (uint32_t)(V >> 32);
    const float kf = __fadd_rn(T2f, qf), dk = __fadd_rn(L.d2, dq);
    int_least(bad, fminf(lq, int_check(bad, kf, dk)));
    uint32_t up = 0, wk;
    if (ST < 3) {
        up = word_above(w1, kf, L.above);
        wk = int_round3(w0, w1, up, fbits(kf) >> 23, 0);
    } else {
        wk = int_round(w0, w1, fbits(kf) >> 23);
    }
    // acc: k1, acc + 2 k2, acc + 2 k3, acc + k4
    float xf = kf, dx = dk;
    if (ST == 0) {
        acc0 = w0;
        acc1 = w1;
        accf = kf;
        accd = dk;
    } else {
        const uint64_t k64 = pack64(w0, w1);
        V = pack64(acc0, acc1) + (ST < 3 ? 2 * k64 : k64);
        acc0 = (uint32_t)V;
        acc1 = (uint32_t)(V >> 32);
        accf = ST < 3 ? __fmaf_rn(kf, 2.0f, accf) : __fadd_rn(kf, accf);
        accd = ST < 3 ? __fmaf_rn(dk, 2.0f, accd) : __fadd_rn(dk, accd);
        int_least(bad, int_check(bad, accf, accd));
        if (ST == 3) {
            up = word_above(acc1, accf, L.above);
            wk = int_round3(acc0, acc1, up, fbits(accf) >> 23, 0);
            w1 = acc1;
            xf = accf;
            dx = accd;
        } else {
            int_round(acc0, acc1, fbits(accf) >> 23);
        }
    }
    // m = c k (c acc), with a word below the grid
    const uint32_t xk = fbits(xf) >> 23;
    const int k0 = (int)__funnelshift_r(wk, w1, xk);
    const int k1 = (int)(__funnelshift_r(w1, up, xk) + ((uint32_t)k0 >> 31));
    bad.few_bits = bad.few_bits || ((uint32_t)k0 << 6) == 0;
    const float mf = __fmul_rn(xf, L.cf[kc]);
    const float dm = __fmul_rn(dx, fabsf(L.cf[kc]));
    int_check(bad, mf, dm);
    const IntProduct g = int_product(k0, k1, L.c0[kc], L.c1[kc], __funnelshift_l(0, 1, (fbits(mf) >> 23) - xk + L.c_half[kc]));
    const uint32_t r = xk + L.c_place[kc];
    const uint32_t below = __funnelshift_l(0, g.g0, r);
    // the next tin
    V = pack64(s.v0, s.v1) + pack64(__funnelshift_l(g.g0, g.g1, r), __funnelshift_l(g.g1, g.g2, r));
    w0 = (uint32_t)V;
    w1 = (uint32_t)(V >> 32);
    const float tf = __fadd_rn(s.l.f, mf);
    int_least(bad, int_check(bad, tf, __fadd_rn(L.dt, dm)));
    bad.most = fmaxf(bad.most, fabsf(tf));
    const uint32_t xt = fbits(tf) >> 23;
    up = word_above(w1, tf, L.above);
    const uint32_t wt = int_round3(w0, w1, up, xt, min(below, 1u));
    const uint32_t hi = __funnelshift_r(w1, up, xt);
    t.v0 = w0;
    t.v1 = w1;
    t.l.n0 = (int)__funnelshift_r(wt, w1, xt);
    t.l.n1 = (int)(hi + ((uint32_t)t.l.n0 >> 31));
    t.l.f = tf;
    bad.few_bits = bad.few_bits || ((uint32_t)t.l.n0 << 6) == 0;
    if (ST == 3) {
        t.l.f = shadow_of((uint32_t)t.l.n0, hi, tf);
        bad.m |= fbits(t.l.f) ^ fbits(tf);
    }
}

// One step of every chain of the warp (lane 4 c + v: variable v of chain c); true on a lane whose step is
// marked (s is then garbage).  All 32 lanes call it together.
__device__ __forceinline__ bool int_step(IntVar &s, const IntLane &L) {
    IntMarks bad{0, 1e30f, 0.0f, false};
    IntVar t = s;
    uint32_t acc0, acc1;
    float accf, accd;
    int_stage<0>(s, t, L, acc0, acc1, accf, accd, bad);
    int_stage<1>(s, t, L, acc0, acc1, accf, accd, bad);
    int_stage<2>(s, t, L, acc0, acc1, accf, accd, bad);
    int_stage<3>(s, t, L, acc0, acc1, accf, accd, bad);
    s = t;
    return (bad.m & 0xff800000u) != 0 || !(bad.least >= 4.0f) || !(bad.most < L.limit) || bad.few_bits;
}

// |N| of a variable: the 53 bits of its binary64 significand.
__device__ __forceinline__ uint64_t int_significand(const IntVar &s) {
    const long long N = ((long long)s.l.n1 << 32) + (long long)s.l.n0;
    return (uint64_t)(N < 0 ? -N : N);
}

__device__ __forceinline__ double int_to_double(const IntVar &s, const IntLane &L) {
    const uint64_t a = int_significand(s);
    const uint32_t eb = ((fbits(s.l.f) >> 23) & 255) - L.expo + 1022;
    const uint32_t sign = ((fbits(s.l.f) >> 31) != 0) != L.negated ? 0x80000000u : 0u;
    return __hiloint2double((int)(((eb << 20) + (uint32_t)(a >> 32)) | sign), (int)(uint32_t)a);
}

// A value that the step cannot take (outside the grid's range, few bits) becomes a zero, which marks the step.
__device__ __forceinline__ void int_from_double(IntVar &s, double d, const IntLane &L) {
    int e;
    const bool normal = split_double(d, L.negated, s.l.n0, s.l.n1, e);
    const int p = e - 52 + L.grid;
    const bool ok = normal && p >= 1 && p < 32;
    const uint64_t N = (uint64_t)(((long long)s.l.n1 << 32) + (long long)s.l.n0), V = N << (ok ? p : 0);
    const float x = __uint_as_float((uint32_t)(e + (int)L.expo) << 23);
    s.v0 = (uint32_t)V;
    s.v1 = (uint32_t)(V >> 32);
    s.l.f = shadow_of((uint32_t)N, (uint32_t)(N >> 32), x);
    if (!ok || ((fbits(s.l.f) ^ fbits(x)) & 0x7f800000u) != 0 || !(fabsf(s.l.f) < L.limit) ||
        ((uint32_t)s.l.n0 << 6) == 0) {
        s.v0 = s.v1 = 0;
        s.l = IntLimbs{0, 0, 0.0f};
    }
}

// gamma as a factor: its exponent within the shifts' range and its low 26 bits not all zero.
__device__ __forceinline__ bool int_gamma_ok(double gamma) {
    int n0, n1, e;
    return split_double(gamma, false, n0, n1, e) && e >= -8 && e <= 0 && ((uint32_t)n0 << 6) != 0;
}

// Constants of this lane: v = its variable, base = the first lane of its chain.
__device__ IntLane int_lane(const IntStepTab &T, int lane, double gamma) {
    IntLane L;
    const int v = lane & 3, base = lane & ~3;
    const int kap = v == 3 ? kKappaW : kKappaXYZ;
    L.grid = v == 3 ? kGridW : kGridXYZ;
    L.expo = 127 + kap;
    L.negated = v == 2;
    L.M1 = v == 0 ? 1 : v == 1 ? 28 : 0;
    L.M2 = v == 0 ? 10 : 1;
    L.own1 = v == 0 ? ~0u : 0;
    L.own2 = v == 1 ? ~0u : 0;
    L.fM1 = (float)L.M1;
    L.fM2 = (float)L.M2;
    L.fo1 = v == 0 ? -1.0f : 0.0f;
    L.fo2 = v == 1 ? -1.0f : 0.0f;
    int e = 0;
    L.t0 = L.t1 = 0;
    L.tf = 0.0f;
    if (v >= 2) {
        const double c = v == 2 ? 8.0 / 3.0 : gamma;
        split_double(c, false, L.t0, L.t1, e);
        L.tf = __double2float_rn(c);
    }
    L.t_half = (uint32_t)(19 - e);
    L.t_place = (uint32_t)(72 - L.grid - e + (int)L.expo);
    // A: 1.0, x, x, y;  B: w, -z, y, -z
    L.sA = base + (v == 3 ? 1 : 0);
    L.sB = base + (v == 0 ? 3 : v == 2 ? 1 : 2);
    L.sa = base + (v == 0 ? 1 : 0);
    const int kB = v == 0 ? kKappaW : kKappaXYZ;
    L.amask = v == 0 ? 0u : ~0u;
    L.aone1 = v == 0 ? 1u << 20 : 0u;
    L.aonef = v == 0 ? (uint32_t)(127 + kKappaXYZ) << 23 : 0u;
    L.q_scale = __uint_as_float((uint32_t)(127 + kap - kKappaXYZ - kB) << 23);
    L.q_half = (uint32_t)(19 - kap - 127 + 127 + kKappaXYZ + 127 + kB);
    L.q_place = (uint32_t)(72 - L.grid + 127 + kKappaXYZ + 127 + kB);
    L.above = __uint_as_float((uint32_t)(127 - (64 - L.grid + kap)) << 23);
    L.d1 = T.d1[v];
    L.d2 = T.d2[v];
    L.dt = T.dt[v];
    L.qA = T.qA[v];
    L.qB = T.qB[v];
    L.limit = T.limit[v];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        split_double(T.c[k], v == 2, L.c0[k], L.c1[k], e);
        const float f = __double2float_rn(T.c[k]);
        L.cf[k] = v == 2 ? -f : f;
        L.c_half[k] = (uint32_t)(19 - e);
        L.c_place[k] = (uint32_t)(e + L.grid - 40 - (int)L.expo);
    }
    return L;
}

}  // namespace
}  // namespace fhd
