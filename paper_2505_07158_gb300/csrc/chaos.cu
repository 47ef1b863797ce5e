// K2a (master) and K2b (workers): the Lorenz hyperchaotic iterations.
//
// Eq. (1) of the paper with sigma = 10, rho = 28, beta = 8/3 and the stream's
// gamma, integrated by classical RK4 with step h (the paper names no
// integrator; this reading is fixed with the oracle):
//   k1 = f(s); k2 = f(s + (h/2) k1); k3 = f(s + (h/2) k2); k4 = f(s + h k3);
//   s' = s + (h/6) (((k1 + 2 k2) + 2 k3) + k4),
// every operation an explicit round-to-nearest binary64 intrinsic (no FMA
// contraction; the library is also built with -fmad=false), so the iterates
// are bit-identical to a plain C implementation.  The term acc + 2 k of the
// combination is one fma(k, 2, acc) (see below).
//
// GPU mapping.  On this GPU a binary64 instruction occupies the SM
// sub-partition's FP64 pipe for ~64 cycles whatever the number of active
// lanes, one after another (no overlap, dependent or not), and handing a
// binary64 result to another unit (shuffle, shared memory, integer select)
// costs ~15-40 more cycles per hand-off; every chain is strictly sequential.
// So the time per step is the binary64 instructions one warp issues per step
// plus its hand-offs.  A warp carries six chains, one variable per lane
// (lane = 4 chain + v, v = x, y, z, w), and every component of Eq. (1) is the
// same four fused multiply-adds with per-lane operands:
//   p = fma(Pa, Pb, -Pc); q = fma(Qa, Qb, -0); p2 = fma(p, B2, -P2); k = fma(q, kS, p2)
//   v = x: p = Y*1 - X, q = W*1, p2 = sigma p,     k = q + p2  = sigma (y - x) + w
//   v = y: p = X rho,   q = X Z, p2 = p*1 - Y,     k = p2 - q  = (rho x - y) - x z
//   v = z: p = Z beta,  q = X Y, p2 = -p,          k = q + p2  = x y - beta z
//   v = w: p = W gamma, q = Y Z, p2 = p,           k = p2 - q  = gamma w - y z
// Each fma rounds once, a product with addend -0 or a sum with a factor of
// +-1, so k is bit-identical to the dmul/dadd/dsub sequence of the plain
// definition.  The variable operands Pa, Pc, Qa, Qb, P2 arrive by five warp
// shuffles per stage; a constant operand (the 1 of v = x, the 0 addends) is
// shuffled from lane 24 (+0) or lane 25 (1.0), which stay fixed points of the
// update because their own k is +0.  No selects and no barriers remain: a
// step takes 27 binary64 instructions and ~2.0k cycles on GB300 (the earlier
// mapping, one warp per variable with a shared-memory exchange and one barrier
// per stage, took ~3.5k).  In the combination, acc + 2 k is one fma(k, 2, acc):
// 2 k is exact, so it equals the separate doubling and add whenever 2 k is
// finite (an overflowing 2 k makes the definition's state non-finite anyway).
//
// LHCS_m, the trajectory kernel and the one-pair worker kernel step on the integer pipes instead (Chains in
// chaos_dev.cuh, lorenz_int.cuh): ~1.3k cycles a step, bit-identical.  That costs issue slots, which a warp that
// has its sub-partition to itself does not miss; the worker-pair launches that fill the GPU with chains keep the
// binary64 steps above, six or eight chains to a warp.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "chaos_dev.cuh"

namespace fhd {
namespace {

// K2a: one warp per stream of the batch; the stream's frames in call order.
__global__ void __launch_bounds__(32, 1) master_kernel(const __grid_constant__ Batch b, StreamState *states,
                                                    unsigned *status) {
    __shared__ __align__(16) uint8_t H[32];
    if (blockIdx.x >= b.groups) return;
    master_stream(b, blockIdx.x, states, status, H, threadIdx.x, [](uint32_t) { return true; }, [](uint32_t) {});
}

// fhd_master: one warp, one state of 5 doubles (x, y, z, w, gamma).
__global__ void __launch_bounds__(32, 1) master_raw_kernel(double *state5, const uint8_t *Hg, uint32_t n, Rk4 c,
                                                        const __grid_constant__ IntStepTab tab, uint4 u4, double *IR,
                                                        unsigned *status) {
    __shared__ __align__(16) uint8_t H[32];
    const int lane = threadIdx.x;
    H[lane] = Hg[lane];
    __syncwarp();
    const uint32_t u[4] = {u4.x, u4.y, u4.z, u4.w};
    const double gamma = state5[4];
    Chains ch;
    ch.init(lane, lane < 4, gamma, c, tab);
    const bool use_int = Chains::usable(lane < 4, lane, gamma, tab);
    double s = lane_init(lane, lane < 4 ? state5[lane] : 0.0);
    master_frame(s, lane, ch, use_int, H, u, n, IR);
    if (lane < 4) {
        state5[lane] = s;
        if (!finite(s) && status) atomicOr(status, kStatusNonFinite);
    }
}

// K2b: one warp per kPairs worker pairs of one frame (three with the six-chain step, four with the
// eight-chain step); a CTA carries blockDim.x / 32 consecutive such warps (warps of one CTA are spread over
// the SM's sub-partitions).
// kMix (eight-chain step only): b.int_mix of every 8 consecutive warps step on the integer pipes instead of
// the binary64 pipe (the same bytes: rk4_step_lanes8_int).  A separate instantiation, so that the binary64-only
// kernel keeps its own register allocation.
template <int kPairs, bool kMix = false>
__global__ void __launch_bounds__(256) keystream_kernel(const __grid_constant__ Batch b) {
    const uint32_t wpf = (b.n + kPairs - 1) / kPairs;
    const uint32_t task = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const uint32_t f = task / wpf, pg = task % wpf;
    if (f >= b.count) return;
    const Rk4 c{b.hstep, b.hhalf, b.hsixth};
    if constexpr (kMix) {
        if ((task & 7) < b.int_mix) {
            keystream_warp<kPairs, true>(b.f[f], b.n, c, pg, threadIdx.x & 31);
            return;
        }
    }
    keystream_warp<kPairs>(b.f[f], b.n, c, pg, threadIdx.x & 31);
}

// ---- One-trajectory route (see traj_records in common.cuh; the warp and chunk bodies are in chaos_dev.cuh).

// Warps per CTA of the kernels whose chains step on the integer pipes: one to each of the SM's sub-partitions.
// With one-warp CTAs two chains may meet on a sub-partition while others are free, which costs a pipeline of many
// launches: the clip pipeline (720 trajectories in flight) 11.3k frames/s, 13.1k with four warps per CTA, and a
// single launch the same either way (measured with a step of 1,580 cycles; 13.9k with the present one).  Two frames
// to a warp, 4 % slower by themselves, were left: marked steps of either frame hold both up.
constexpr uint32_t kIntWarps = 4;

// One worker pair per one-warp CTA, its two chains on the integer pipes (lorenz_int.cuh).
__global__ void __launch_bounds__(32, 1) keystream_pair_kernel(const __grid_constant__ Batch b) {
    const uint32_t f = blockIdx.x / b.n, pg = blockIdx.x % b.n;
    if (f >= b.count) return;
    keystream_warp<1>(b.f[f], b.n, Rk4{b.hstep, b.hhalf, b.hsixth}, pg, threadIdx.x, &b.tab);
}
// Most worker pairs of a launch of it: one warp per sub-partition of the GPU (608 on 152 SMs).  Up to there a pair's
// latency is the launch's (32 pairs of a 720p frame: 2.91 ms against 4.23 ms for the binary64 kernel; four pairs
// per CTA took 3 % longer, with 608 pairs too); beyond, its one pair per warp would cost more issue slots than the
// binary64 kernel's three have pipe time.
uint32_t pair_launch() { return 4 * sm_count(); }
// Fewest steps of its longest slice, from nine pairs on: iterates from anywhere (Algorithm 2) need some steps to come to
// the attractor, and many a step on the way is marked; a launch takes as long as its unluckiest pair.  32 pairs and
// more of ~11, 21 and 43 steps: 23, 38, 56-59 us here, 19, 31, 56 in the binary64 kernel; one pair of 21 steps 33 and
// 42, eight 32 and 35.
constexpr uint64_t kPairSteps = 48, kFewPairs = 8;

// K2t: the records of one frame per warp, its chain in lanes 0..3.
__global__ void __launch_bounds__(32 * kIntWarps, 1) trajectory_kernel(const __grid_constant__ Batch b) {
    const int lane = threadIdx.x & 31;
    const uint32_t f = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (f >= b.count) return;
    trajectory_warp(lane < 4 ? &b.f[f] : nullptr, b.n, Rk4{b.hstep, b.hhalf, b.hsixth}, b.tab, lane);
}

// K2e: D and B of every frame from its records.  CTA (x, f) takes worker slice i = x / cps of frame f and
// part j = x % cps of it: part 0 also writes the slice's D bytes, and the parts split the slice's B bytes
// in runs of kEmitChunks x kEmitThreads 16-byte chunks of B.
constexpr int kEmitThreads = 256;
constexpr int kEmitChunks = 4;

__global__ void __launch_bounds__(kEmitThreads) emit_kernel(const __grid_constant__ Batch b, uint32_t cps) {
    const uint32_t f = blockIdx.y, i = blockIdx.x / cps, j = blockIdx.x % cps;
    if (f >= b.count || i >= b.n) return;
    const FrameDesc &fd = b.f[f];
    __shared__ WorkerSlice ws_s;
    if (threadIdx.x == 0) ws_s = worker_slice((uint64_t)fd.C * (fd.h + fd.w), fd.N, b.n, i);
    __syncthreads();
    const WorkerSlice ws = ws_s;
    if (j == 0) emit_d_slice(fd, b.n, i, ws, threadIdx.x, kEmitThreads);
    if (!ws.nb) return;
    const uint64_t per = 16ull * kEmitThreads * kEmitChunks;
    const uint64_t base = (ws.b0 >> 4) << 4;   // the slice's first chunk
    const uint64_t lo = base + j * per, hi = lo + per;
    const uint64_t a = lo > ws.b0 ? lo : ws.b0, e = hi < ws.b0 + ws.nb ? hi : ws.b0 + ws.nb;
    if (a < e) emit_b_part(fd, b.n, i, ws, a, e, threadIdx.x, kEmitThreads);
}

int g_ks_route = FHD_KS_ROUTE_TRAJECTORY;

}  // namespace

// Error bounds of the integer step's shadows (lorenz_int.cuh), unscaled, for |x| < 28, |y| < 30, |z| < 50, |w| < 216 (the
// ranges that every unmarked step keeps to) and |gamma| < 2: interval arithmetic over the stages with u = 2^-24 the rounding unit of a float.  A state's
// shadow is off by less than 2^-23 of its range; a stage's by that, plus c times the error of k, plus roundings.
// All bounds are taken over the four stages and widened by a quarter.
IntStepTab int_step_tab(double h) {
    IntStepTab t{};
    t.c[0] = h / 2.0;
    t.c[1] = h;
    t.c[2] = h / 6.0;
    // the step constants' shift range (c_place in 0..31 for every k and acc) and a one among their low 19 bits; beyond
    // h = 0.04 the bounds mark too many steps
    t.ok = h >= 0.0008 && h <= 0.04;
    for (double c : t.c) {
        unsigned long long bits;
        std::memcpy(&bits, &c, sizeof bits);
        if ((bits & 0x7ffffull) == 0) t.ok = 0;
    }
    if (!t.ok) return t;
    // ranges: just beyond the attractor's, each within the power of two that the shifts allow
    const double u = 0x1p-24, lim[4] = {28, 30, 50, 216}, end[4] = {32, 32, 64, 256}, g = 2.0, beta = 8.0 / 3.0;
    const double X = lim[0], Y = lim[1], Z = lim[2], W = lim[3];
    const double kmax[4] = {10 * (X + Y) + W, 28 * X + Y + X * Z, beta * Z + X * Y, g * W + Y * Z};
    double es[4], e[4], acc[4] = {}, amax[4] = {}, d1[4] = {}, d2[4] = {}, dk[4] = {}, et[4] = {};
    for (int v = 0; v < 4; ++v) es[v] = e[v] = end[v] * 0x1p-23;
    for (int st = 0; st < 4; ++st) {
        const double t1[4] = {e[0] + e[1] + u * (X + Y), 28 * (e[0] + u * X), beta * e[2] + (0x1p-21 + u * beta) * Z,
                              g * e[3] + (0x1p-22 + u * g) * W};
        const double t2[4] = {10 * t1[0] + 20 * u * (X + Y), t1[1] + e[1] + u * (56 * X + 2 * Y), t1[2], t1[3]};
        const double q[4] = {e[3] + (0x1p-22 + 3 * u) * W, X * e[2] + Z * e[0] + e[0] * e[2] + 2 * u * X * Z,
                             X * e[1] + Y * e[0] + e[0] * e[1] + 2 * u * X * Y,
                             Y * e[2] + Z * e[1] + e[1] * e[2] + 2 * u * Y * Z};
        const double f = st == 1 || st == 2 ? 2.0 : 1.0, c = st == 2 ? h : st == 3 ? h / 6.0 : h / 2.0;
        for (int v = 0; v < 4; ++v) {
            const double k = t2[v] + q[v] + u * kmax[v];
            d1[v] = std::max(d1[v], t1[v]);
            d2[v] = std::max(d2[v], t2[v]);
            // k's own rounding, a sixth of those of acc (14 u) and of c acc (12 u) and what is left of c k's
            dk[v] = std::max(dk[v], t2[v] + 5 * u * kmax[v] + 2 * u * kmax[v] / 6);
            amax[v] += f * kmax[v];
            acc[v] += f * k + u * amax[v];
            e[v] = es[v] + c * (st == 3 ? acc[v] : k) + 2 * u * c * (st == 3 ? amax[v] : kmax[v]) + u * lim[v];
            et[v] = std::max(et[v], e[v]);
        }
    }
    const int grid_kappa[4] = {int_kappa(0), int_kappa(1), int_kappa(2), int_kappa(3)};
    const int sA[4] = {-1, 0, 0, 1}, sB[4] = {3, 2, 1, 2};
    for (int v = 0; v < 4; ++v) {
        const double scale = 1.25 * std::ldexp(1.0, grid_kappa[v]);   // and the roundings of the bounds and checks
        t.d1[v] = (float)(scale * d1[v]);
        t.d2[v] = (float)(scale * d2[v]);
        t.dk[v] = (float)(scale * dk[v]);
        t.dt[v] = (float)(scale * (es[v] + 2 * u * lim[v] + 2 * u * h * kmax[v]));
        t.limit[v] = (float)std::ldexp(lim[v], grid_kappa[v]);
        // |A~| qA + |B~| qB in this lane's scale: A~, B~ carry their own lanes' scales
        const double eA = sA[v] < 0 ? 0x1p-22 : et[sA[v]], eB = et[sB[v]], lB = lim[sB[v]], lA = sA[v] < 0 ? 1.0 : lim[sA[v]];
        const int kA = sA[v] < 0 ? int_kappa(3) : grid_kappa[sA[v]], kB = grid_kappa[sB[v]];
        t.qA[v] = (float)(scale * (eB + eA * eB / lA + 2 * u * lB) / std::ldexp(1.0, kA));
        t.qB[v] = (float)(scale * (eA + 2 * u * lA) / std::ldexp(1.0, kB));
    }
    return t;
}

int set_keystream_route(int route) {
    if (route != FHD_KS_ROUTE_TRAJECTORY && route != FHD_KS_ROUTE_PAIRS) return -1;
    const int old = g_ks_route;
    g_ks_route = route;
    return old;
}

int keystream_route() { return g_ks_route; }

cudaError_t launch_trajectory_keystream(const Batch &b, cudaStream_t s) {
    if (!b.count) return cudaSuccess;
    uint64_t nb_max = 0;
    for (uint32_t k = 0; k < b.count; ++k) {
        const uint64_t nb = (b.f[k].N + b.n - 1) / b.n;
        nb_max = nb > nb_max ? nb : nb_max;
    }
    const uint32_t wpc = b.count < kIntWarps ? b.count : kIntWarps;
    trajectory_kernel<<<(b.count + wpc - 1) / wpc, 32 * wpc, 0, s>>>(b);
    note_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    const uint64_t chunks = nb_max / 16 + 2;   // chunks of B one slice meets
    const uint64_t per_cta = (uint64_t)kEmitThreads * kEmitChunks;
    const uint64_t cps = (chunks + per_cta - 1) / per_cta;
    const uint64_t gx = cps * b.n;
    if (gx > 0x7fffffffull) return cudaErrorInvalidConfiguration;
    emit_kernel<<<dim3((unsigned)gx, b.count), kEmitThreads, 0, s>>>(b, (uint32_t)cps);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_master(const Batch &b, StreamState *states, unsigned *status, cudaStream_t s) {
    if (!b.groups) return cudaSuccess;
    master_kernel<<<b.groups, 32, 0, s>>>(b, states, status);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_master_raw(double *state5, const uint8_t *H, uint32_t n, double hstep, const uint32_t u[4],
                              double *IR, unsigned *status, cudaStream_t s) {
    Rk4 c{hstep, hstep / 2.0, hstep / 6.0};   // host arithmetic: IEEE round-to-nearest
    master_raw_kernel<<<1, 32, 0, s>>>(state5, H, n, c, int_step_tab(hstep), make_uint4(u[0], u[1], u[2], u[3]), IR,
                                       status);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_keystream(const Batch &b, cudaStream_t s, bool dense, uint32_t warps_per_cta, uint32_t smem) {
    if (!b.count) return cudaSuccess;
    const uint32_t k = warps_per_cta ? warps_per_cta : 1;
    if (smem > 48 * 1024) {
        const void *fns[3] = {(const void *)keystream_kernel<4>, (const void *)keystream_kernel<4, true>,
                              (const void *)keystream_kernel<kPairsPerWarp>};
        for (const void *f : fns) {
            cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            if (e != cudaSuccess) return e;
        }
    }
    if (dense) {
        const uint32_t warps = b.count * ((b.n + 3) / 4);
        if (b.int_mix)
            keystream_kernel<4, true><<<(warps + k - 1) / k, 32 * k, smem, s>>>(b);
        else
            keystream_kernel<4><<<(warps + k - 1) / k, 32 * k, smem, s>>>(b);
        note_launch();
        return cudaGetLastError();
    }
    uint64_t steps = 0;
    for (uint32_t f = 0; f < b.count; ++f) {
        const FrameDesc &d = b.f[f];
        const uint64_t LD = (uint64_t)d.C * (d.h + d.w);
        steps = std::max(steps, (2 * ((LD + b.n - 1) / b.n) + (d.N + b.n - 1) / b.n + 23) / 24);
    }
    if (k == 1 && smem == 0 && b.count * b.n <= pair_launch() && (steps >= kPairSteps || b.count * b.n <= kFewPairs)) {
        keystream_pair_kernel<<<b.count * b.n, 32, 0, s>>>(b);
        note_launch();
        return cudaGetLastError();
    }
    const uint32_t warps = b.count * ((b.n + kPairsPerWarp - 1) / kPairsPerWarp);
    keystream_kernel<kPairsPerWarp><<<(warps + k - 1) / k, 32 * k, smem, s>>>(b);
    note_launch();
    return cudaGetLastError();
}

}  // namespace fhd

FHD_BOUNDS_TAKER(take_bounds_chaos)
