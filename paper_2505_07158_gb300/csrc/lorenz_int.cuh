// One RK4 step of Eq. (1) on the integer pipes, bit-identical to the binary64 step.
//
// Why.  A binary64 instruction holds its sub-partition's pipe for 64 cycles whatever the number of active
// lanes, and every rounded operation of the step waits for the one before: the step of chaos_dev.cuh is 27
// such instructions and four exchanges, ~2.1k cycles, with the integer pipes idle.  The same roundings on
// the integer pipes take ~20 cycles each.  Measured on GB300, the records of one 1080p frame (8,124 steps, one
// warp): 5.11 ms, 1,300 cycles a step with the binary64 redoes below, against 8.53 ms.  What bounds it now is one
// warp's latency and issue together: a stage's chain is ~260 cycles (exchange 50, A B 50, T 30, k 30, c k 50, tin
// 50) and its ~110 integer and ~40 float instructions take about as long to issue.
//
// Representation.  The four lanes of a chain hold one variable each.  A variable, and every sum of the step
// (T1, T2, k, acc, tin), is a 64-bit two's complement integer on its lane's grid 2^-G (G = 64 for x and z, 63 for
// y and w), modulo 2^64: exact, since every rounded value of at least 2^(53-G) is a multiple of its own
// ulp >= 2^(1-G).  Binary64 rounding of such a sum is rounding to nearest even at bit p = e - 52 + G, with e
// the exponent of the sum; e comes from a float shadow of the sum, which is a few cycles ahead of it.  A
// product takes its factors as 53-bit integers N (value N 2^(e-52), N = n1 2^32 + n0 with a signed low
// digit), is formed exactly, rounded half up at bit 52 or 53 (the shadow says which) and shifted onto the
// grid.  The bits of a sum above its 64 come from the shadow too.  The z lane holds -z, so that every
// component is T1 = M1 a - own1, T2 = M2 T1 - own2, k = T2 + T + A B with non-negative M1 and M2:
//   x: a = y, own1 = x, M2 = 10, A B = 1 w;   y: a = x, M1 = 28, own2 = y, A B = x (-z);
//   z (-z, k as it is, c negated): T = beta (-z), A B = x y;   w: T = gamma w, A B = y (-z).
// T has a lane of its own beside the chain, where the instructions that form A B form it (formed in the z and w
// lanes by a product of its own it cost 40 cycles a stage: 5.9 against 5.5 ms), and the constants 1, beta and gamma
// are lanes too, so that every factor comes by a shuffle.
//
// What makes it exact.  Each shadow has an error bound (IntStepTab, by interval arithmetic over the four
// stages for |x| < 28, |y| < 30, |z| < 50, |w| < 216); a shadow within its bound of a power of two or of the
// smallest magnitude its grid carries, a variable outside those ranges, and a factor whose low bits are all
// zero (only then could a product be a tie: 51 zero bits in both factors together) mark the step, and a marked step
// is done again in binary64.  On the attractor at h = 0.01 that is 2.2 to 2.8 % of the steps for gamma from -1.52 to
// -0.5, 3.2 % at -0.3 and 4.9 to 5.1 % at -0.1 and -0.06, where w comes near zero (800,000 steps each; at -0.9 1.5 % for
// h = 0.001, 3.7 % for 0.02, 7.3 % for 0.0399).  Three constants of the step (h/2, h, h/6) and gamma
// have to be in range for the shifts (IntStepTab::ok, int_gamma_ok); otherwise every step is binary64.
#pragma once
#include "common.cuh"

namespace fhd {
namespace {

// Grids of x, y, z, w: as fine as the shifts of their products allow (q_place in 0..31 over the ranges below).
__host__ __device__ constexpr int int_grid(int v) { return v == 0 || v == 2 ? 64 : 63; }
// Scale of a lane's shadows: 2^kappa with (exponent field of a shadow) mod 32 = the rounding bit p.
__host__ __device__ constexpr int int_kappa(int v) { return int_grid(v) - 51; }   // (G - 52 - 127) mod 32

// Lanes of a warp: variable v of chain c in lane 4 c + v, two chains; then the lanes that form the products T of
// the chains' z and w, and the lanes that hold the constants among a product's factors: 1, beta and gamma, as
// variables that the step leaves as they are.
constexpr int kIntChains = 2, kIntT = 4 * kIntChains, kIntOne = kIntT + 2 * kIntChains, kIntBeta = kIntOne + 1,
              kIntGamma = kIntOne + 2;

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
    uint32_t M1, M2, own1, own2, tmask;   // own1, own2: -1 where the lane's own value is subtracted, else 0;
                                          // tmask: -1 where T is added
    float fM1, fM2, fo1, fo2;             // fo1: the constant of T on the z and w lanes
    uint32_t q_half, q_place;             // shift amounts of the product, less the exponent fields
    float q_scale, above;                 // scale of the shadow of A B; 2^-(64 - G + kappa - 6)
    float d1, d2, dk, dt, qA, qB;         // shadow error bounds
    int c0[3], c1[3];                     // limbs of h/2, h, h/6 (negated on the z lane, 0 beyond the chains)
    float cf[3];
    uint32_t c_half[3], c_place[3];
    float limit;                          // the variable's range, scaled
    int sa, sA, sB, sT;                   // source lanes of a, A, B and T
    uint32_t expo;                        // 127 + kappa
    int grid;
    bool negated;
};

struct IntMarks {
    uint32_t m;      // exponent or sign bits that differ: a shadow near a power of two
    float least, most;
    uint32_t few;    // 0: a factor whose low bits are all zero
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
    const int lh = __mulhi(a0, b0) + (int)half;
    const long long Z = (long long)a1 * b0 + ((long long)a0 * b1 + (long long)lh);
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
__device__ __forceinline__ void int_least(IntMarks &b, float l1, float l2) {
    asm("min.f32 %0, %0, %1, %2;" : "+f"(b.least) : "f"(l1), "f"(l2));
}

__device__ __forceinline__ uint32_t low_mask(uint32_t x) {   // 2^(x mod 32) - 1
    uint32_t m;
    asm("bmsk.wrap.b32 %0, 0, %1;" : "=r"(m) : "r"(x));
    return m;
}

// Round to nearest even at bit x mod 32: add half a unit less one and the bit above it, clear the rest.  Bit 0 of
// a sum of rounded values is 0 (each is a multiple of 2), so the bit above goes there by a logic operation; where
// it is 1 (tin: part of the product below the grid), the sum is no tie from x = 2 on, and x = 1 marks the step.
// Returns the low word before clearing (enough for a shift by x).
__device__ __forceinline__ uint32_t int_round(uint32_t &v0, uint32_t &v1, uint32_t x) {
    const uint32_t um = low_mask(x), t = v0 | (__funnelshift_r(v0, 0, x) & 1);
    uint32_t a, b;
    asm("add.cc.u32 %0, %2, %4; addc.u32 %1, %3, 0;" : "=&r"(a), "=&r"(b) : "r"(t), "r"(v1), "r"(um >> 1));
    v0 = a & ~um;
    v1 = b;
    return a;
}
// The same carrying into the word above; sticky (0 or 1): nonzero bits below the grid.
__device__ __forceinline__ uint32_t int_round3(uint32_t &v0, uint32_t &v1, uint32_t &v2, uint32_t x, uint32_t sticky) {
    const uint32_t um = low_mask(x), t = v0 | (__funnelshift_r(v0, 0, x) & 1) | sticky;
    uint32_t a, b, c;
    asm("add.cc.u32 %0, %3, %6; addc.cc.u32 %1, %4, 0; addc.u32 %2, %5, 0;"
        : "=&r"(a), "=&r"(b), "=&r"(c)
        : "r"(t), "r"(v1), "r"(v2), "r"(um >> 1));
    v0 = a & ~um;
    v1 = b;
    v2 = c;
    return a;
}

// The word above a value known modulo 2^64, from its shadow (above: its scale to 2^-6 of that word, where the shadow
// is off by less than 2): the whole number of 2^64 between them.
__device__ __forceinline__ uint32_t word_above(uint32_t v1, float f, float above) {
    const uint32_t y = fbits(__fmaf_rn(f, above, 12582912.0f)) - (0x4B400000u - 32u);
    return (uint32_t)((int)(y - (v1 >> 26)) >> 6);
}

// Shadow of a significand (hi:lo), with the exponent field of x: 24 bits and an odd last one, so that it never
// reaches the next binade; off by at most 2^-23 of the binade's end.
__device__ __forceinline__ float shadow_of(uint32_t lo, uint32_t hi, float x) {
    return __fmul_rn(__int2float_rn((int)(__funnelshift_l(lo, hi, 2) | 1u)),
                     __uint_as_float((fbits(x) & 0x7f800000u) - (22u << 23)));
}

// The other variables of the chain that a stage reads.
struct IntOthers {
    IntLimbs A, B;
    uint32_t a0, a1;
    float af;
};
__device__ __forceinline__ IntOthers int_exchange(const IntVar &t, const IntLane &L) {
    constexpr unsigned kAll = 0xffffffffu;
    IntOthers o;
    o.a0 = __shfl_sync(kAll, t.v0, L.sa);
    o.af = __shfl_sync(kAll, t.l.f, L.sa);
    o.a1 = __shfl_sync(kAll, t.v1, L.sa);
    o.B.f = __shfl_sync(kAll, t.l.f, L.sB);
    o.A.f = __shfl_sync(kAll, t.l.f, L.sA);
    o.B.n0 = __shfl_sync(kAll, t.l.n0, L.sB);
    o.A.n0 = __shfl_sync(kAll, t.l.n0, L.sA);
    o.B.n1 = __shfl_sync(kAll, t.l.n1, L.sB);
    o.A.n1 = __shfl_sync(kAll, t.l.n1, L.sA);
    return o;
}

// Stage ST of the step: from tin (t) and the others' to the next tin, or in the last stage to the next state.
template <int ST>
__device__ __forceinline__ void int_stage(const IntVar &s, IntVar &t, const IntOthers &o, const IntLane &L, uint32_t &acc0,
                                          uint32_t &acc1, float &accf, float &accd, IntMarks &bad) {
    constexpr int kc = ST == 2 ? 1 : ST == 3 ? 2 : 0;
    constexpr unsigned kAll = 0xffffffffu;
    const IntLimbs &A = o.A, &B = o.B;
    const uint32_t a0 = o.a0, a1 = o.a1;
    const float af = o.af;
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
    // T of the z and w lanes, formed in another lane by the instructions of A B
    const uint64_t T = pack64(__shfl_sync(kAll, (uint32_t)q, L.sT) & L.tmask,
                              __shfl_sync(kAll, (uint32_t)(q >> 32), L.sT) & L.tmask);
    // the own terms
    const uint64_t neg = 0 - pack64(t.v0, t.v1);
    const uint64_t O1 = neg & pack64(L.own1, L.own1), O2 = neg & pack64(L.own2, L.own2);
    // T1, T2, k.  On the z and w lanes T1 = T2 = 0 and T joins in k; their shadows carry it from T1 on.
    uint64_t V = (uint64_t)a0 * L.M1 + O1;
    uint32_t w0 = (uint32_t)V, w1 = (uint32_t)(V >> 32) + a1 * L.M1;
    const float T1f = __fmaf_rn(af, L.fM1, __fmul_rn(t.l.f, L.fo1));
    const float l1 = int_check(bad, T1f, L.d1);
    int_round(w0, w1, fbits(T1f) >> 23);
    V = (uint64_t)w0 * L.M2 + O2;
    w1 = (uint32_t)(V >> 32) + w1 * L.M2;
    w0 = (uint32_t)V;
    const float T2f = __fmaf_rn(T1f, L.fM2, __fmul_rn(t.l.f, L.fo2));
    int_least(bad, l1, int_check(bad, T2f, L.d2));
    int_round(w0, w1, fbits(T2f) >> 23);
    {
        uint32_t x0, x1;
        asm("add.cc.u32 %0, %2, %4; addc.u32 %1, %3, %5;"
            : "=&r"(x0), "=&r"(x1)
            : "r"(w0), "r"(w1), "r"((uint32_t)q), "r"((uint32_t)(q >> 32)));
        asm("add.cc.u32 %0, %2, %4; addc.u32 %1, %3, %5;"
            : "=&r"(w0), "=&r"(w1)
            : "r"(x0), "r"(x1), "r"((uint32_t)T), "r"((uint32_t)(T >> 32)));
    }
    const float kf = __fadd_rn(T2f, qf), dk = __fadd_rn(L.dk, dq);
    int_least(bad, lq, int_check(bad, kf, dk));
    uint32_t up = 0, wk;
    if (ST < 3) {
        up = word_above(w1, kf, L.above);
        wk = int_round3(w0, w1, up, fbits(kf) >> 23, 0);
    } else {
        wk = int_round(w0, w1, fbits(kf) >> 23);
    }
    // acc: k1, acc + 2 k2, acc + 2 k3, acc + k4
    float xf = kf, dx = dk, la = 1e30f;
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
        la = int_check(bad, accf, accd);
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
    // twice the least magnitude: x = 2
    int_least(bad, la, 0.5f * int_check(bad, tf, __fadd_rn(L.dt, dm)));
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
    bad.few = __vimin3_u32(bad.few, (uint32_t)k0, (uint32_t)t.l.n0 << 6);
    if (ST == 3) {
        t.l.f = shadow_of((uint32_t)t.l.n0, hi, tf);
        bad.m |= fbits(t.l.f) ^ fbits(tf);
    }
}

// One step of every chain of the warp; o: the exchange of s.  True on a lane whose step is marked (s is then
// garbage).  All 32 lanes call it together.
__device__ __forceinline__ bool int_step(IntVar &s, const IntOthers &o, const IntLane &L) {
    IntMarks bad{0, 1e30f, 0.0f, ~0u};
    IntVar t = s;
    uint32_t acc0, acc1;
    float accf, accd;
    int_stage<0>(s, t, o, L, acc0, acc1, accf, accd, bad);
    int_stage<1>(s, t, int_exchange(t, L), L, acc0, acc1, accf, accd, bad);
    int_stage<2>(s, t, int_exchange(t, L), L, acc0, acc1, accf, accd, bad);
    int_stage<3>(s, t, int_exchange(t, L), L, acc0, acc1, accf, accd, bad);
    s = t;
    return (bad.m & 0xff800000u) != 0 || !(bad.least >= 4.0f) || !(bad.most < L.limit) || bad.few == 0;
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

// Exponent and limbs of d on this lane's grid; false where the grid does not carry it.
__device__ __forceinline__ bool int_place(IntVar &s, double d, const IntLane &L, float &x) {
    int e;
    const bool normal = split_double(d, L.negated, s.l.n0, s.l.n1, e);
    const int p = e - 52 + L.grid;
    const bool ok = normal && p >= 1 && p < 32;
    const uint64_t N = (uint64_t)(((long long)s.l.n1 << 32) + (long long)s.l.n0), V = N << (ok ? p : 0);
    x = __uint_as_float((uint32_t)(e + (int)L.expo) << 23);
    s.v0 = (uint32_t)V;
    s.v1 = (uint32_t)(V >> 32);
    s.l.f = shadow_of((uint32_t)N, (uint32_t)(N >> 32), x);
    return ok;
}

// A value that the step cannot take (outside the grid's range, few bits) becomes a zero, which marks the step.
__device__ __forceinline__ void int_from_double(IntVar &s, double d, const IntLane &L) {
    float x;
    const bool ok = int_place(s, d, L, x);
    if (!ok || ((fbits(s.l.f) ^ fbits(x)) & 0x7f800000u) != 0 || !(fabsf(s.l.f) < L.limit) ||
        ((uint32_t)s.l.n0 << 6) == 0) {
        s.v0 = s.v1 = 0;
        s.l = IntLimbs{0, 0, 0.0f};
    }
}

// The lanes beyond the chains, and the shadows of T's constants on the z and w lanes.  gamma: lane 0's, for the warp.
__device__ __forceinline__ void int_constants(IntVar &s, IntLane &L, int lane, double gamma) {
    float x;
    gamma = __shfl_sync(0xffffffffu, gamma, 0);
    if (lane >= 4 * kIntChains) int_place(s, lane == kIntBeta ? 8.0 / 3.0 : lane == kIntGamma ? gamma : 1.0, L, x);
    const float scale = __uint_as_float((uint32_t)(127 - int_kappa(3)) << 23);
    const float fb = __fmul_rn(__shfl_sync(0xffffffffu, s.l.f, kIntBeta), scale);
    const float fg = __fmul_rn(__shfl_sync(0xffffffffu, s.l.f, kIntGamma), scale);
    if (lane < 4 * kIntChains && (lane & 3) >= 2) L.fo1 = (lane & 3) == 2 ? fb : fg;
}

// gamma as a factor: its exponent within the shifts' range and its low 26 bits not all zero.  A positive gamma from 1/4 on
// is left to binary64: its chains leave the ranges before long (and overflow in the end), and every step is then marked,
// 2,048 steps at gamma = 0.9 3.80 ms against 2.11 (0.3: 2.35).
__device__ __forceinline__ bool int_gamma_ok(double gamma) {
    int n0, n1, e;
    return split_double(gamma, false, n0, n1, e) && e >= -8 && e <= (gamma > 0.0 ? -3 : 0) && ((uint32_t)n0 << 6) != 0;
}

// Constants of this lane.
__device__ IntLane int_lane(const IntStepTab &T, int lane) {
    IntLane L;
    const bool chain = lane < 4 * kIntChains, product = !chain && lane < kIntOne;
    // its variable (a product's lane: the one it is for; a constant's lane: the grid of w)
    const int v = chain ? lane & 3 : product ? 2 + (lane & 1) : 3;
    const int base = chain ? lane & ~3 : 4 * ((lane - kIntT) >> 1);
    L.grid = int_grid(v);
    L.expo = 127 + int_kappa(v);
    L.negated = chain && v == 2;
    L.M1 = v == 0 ? 2 : v == 1 ? 14 : 0;   // 1 and 28 between the grids of x and y
    L.M2 = v == 0 ? 10 : 1;
    L.own1 = v == 0 ? ~0u : 0;
    L.own2 = v == 1 ? ~0u : 0;
    L.tmask = v >= 2 ? ~0u : 0;
    L.fM1 = (float)L.M1;
    L.fM2 = (float)L.M2;
    L.fo1 = v == 0 ? -1.0f : 0.0f;
    L.fo2 = v == 1 ? -1.0f : 0.0f;
    L.sa = L.sA = L.sB = L.sT = lane;
    int kA = int_kappa(3), kB = kA;
    if (chain) {   // A: 1.0, x, x, y;  B: w, -z, y, -z
        L.sA = v == 0 ? kIntOne : base + (v == 3 ? 1 : 0);
        L.sB = base + (v == 0 ? 3 : v == 2 ? 1 : 2);
        L.sa = base + (v == 0 ? 1 : 0);
        L.sT = v < 2 ? lane : kIntT + 2 * (lane >> 2) + (v - 2);
        kA = int_kappa(v == 0 ? 3 : v == 3 ? 1 : 0);
        kB = int_kappa(v == 0 ? 3 : v == 2 ? 1 : 2);
    } else if (product) {
        L.sA = base + v;
        L.sB = v == 2 ? kIntBeta : kIntGamma;
        kA = int_kappa(v);
    }
    const int kap = int_kappa(v);
    L.q_scale = __uint_as_float((uint32_t)(127 + kap - kA - kB) << 23);
    L.q_half = (uint32_t)(19 - kap - 127 + 127 + kA + 127 + kB);
    L.q_place = (uint32_t)(72 - L.grid + 127 + kA + 127 + kB);
    L.above = __uint_as_float((uint32_t)(127 + 6 - (64 - L.grid + kap)) << 23);
    L.d1 = T.d1[v];
    L.d2 = T.d2[v];
    L.dk = T.dk[v];
    L.dt = T.dt[v];
    L.qA = T.qA[v];
    L.qB = T.qB[v];
    L.limit = T.limit[v];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int e;
        split_double(T.c[k], v == 2, L.c0[k], L.c1[k], e);
        const float f = __double2float_rn(T.c[k]);
        L.cf[k] = v == 2 ? -f : f;
        L.c_half[k] = (uint32_t)(19 - e);
        L.c_place[k] = (uint32_t)(e + L.grid - 40 - (int)L.expo);
        if (!chain) {
            L.c0[k] = L.c1[k] = 0;
            L.cf[k] = 0.0f;
        }
    }
    return L;
}

}  // namespace
}  // namespace fhd
