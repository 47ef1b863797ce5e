// Frame statistics of the paper's evaluation, batched over frames and
// channels: histogram variance and chi^2 (Sec. III-A, Eqs. (4)-(5)),
// adjacent-pixel correlation (Sec. III-B, Eqs. (6)-(9)), information entropy
// and local Shannon entropy (Sec. III-C, Eqs. (10)-(11)), NPCR and UACI
// (Sec. IV-B, Eqs. (14)-(15)).
//
// Frames are one contiguous batch [count][h][w][C] of uint8.  Counting work
// (histograms, changed pixels, |a - b|, the correlation sums) is exact
// integer arithmetic; only the final formula of each statistic rounds.
// GPU mapping: the histogram and NPCR/UACI passes stream the frames once with
// 16-byte loads (memory bound) in groups of 16 * C bytes, so that every byte's
// channel is a compile-time constant (C is a template parameter); per-warp
// shared-memory histograms, or per-thread channel sums built four bytes at a
// time with the SIMD byte instructions, are merged with one global atomic per
// counter and CTA, and a CTA per (frame, channel) finishes the statistic.  The correlation and local-entropy
// statistics read only the sampled pairs and blocks (a few kB per frame).
#include <cooperative_groups.h>

#include <algorithm>

#include "bounds.cuh"
#include "common.cuh"

namespace fhd {
namespace {

constexpr int kStatThreads = 256;
constexpr int kStatWarps = kStatThreads / 32;
// Threads of a histogram CTA, whose counters leave room for two in an SM at C = 3: 32 warps for the atomics'
// latency (30 frames of 1080p: 61 us a call, 71 with 256 threads, 61 with 1024).
constexpr int kHistThreads = 512;

__global__ void zero_kernel(unsigned long long *p, uint64_t n) {
    for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (uint64_t)gridDim.x * blockDim.x) p[k] = 0;
}

// The streaming passes cut each frame into `cuts` runs of whole 16 * C-byte groups (the last one with the rest);
// CTA b has run b % cuts of frame b / cuts, and so starts on channel 0.
struct Run {
    uint64_t begin, end;   // bytes of the batch
    uint32_t head;         // bytes before the first 16-byte boundary
};
template <int C>
__device__ __forceinline__ Run stat_run(const uint8_t *p, uint64_t frame_bytes, uint32_t cuts) {
    const uint64_t f = blockIdx.x / cuts, j = blockIdx.x % cuts, groups = frame_bytes / (16 * C);
    Run r;
    r.begin = f * frame_bytes + 16 * C * (groups * j / cuts);
    r.end = j + 1 == cuts ? (f + 1) * frame_bytes : f * frame_bytes + 16 * C * (groups * (j + 1) / cuts);
    r.head = (uint32_t)(-reinterpret_cast<uintptr_t>(p + r.begin)) & 15;
    return r;
}

// Runs per frame: as many as give the CTAs the GPU holds at once (`slots`) a run each, several rounds of them while a
// run is longer than `most` bytes, fewer where it would be shorter than `least`.
uint32_t stat_cuts(uint64_t frame_bytes, uint32_t count, uint32_t C, uint64_t slots, uint64_t least, uint64_t most) {
    const uint64_t total = frame_bytes * count, rounds = std::max<uint64_t>(1, (total + slots * most - 1) / (slots * most));
    uint64_t cuts = std::max<uint64_t>(1, slots * rounds / count);
    cuts = std::min(cuts, std::max<uint64_t>(1, frame_bytes / least));
    cuts = std::min(cuts, std::max<uint64_t>(1, 0x7fffffffull / count));   // the grid's limit
    return (uint32_t)std::min<uint64_t>(cuts, 1u << 20);
}

// Histogram pass.  A thread takes groups of 16 * C aligned bytes (C 16-byte
// loads) in which byte q belongs to channel (PH + q) mod C, PH the run's head
// mod C: the channel of every byte is a compile-time constant.  The CTA's counters are
// [channel][bin][lane]: each lane counts in its own bank, so the shared
// atomics of a warp never conflict on a bank; at the end the 32 lane copies
// are summed and added to the frame's global histogram.
//
// Bound by the shared atomics, one a byte.  The runs fill the two CTAs of 96 KB (C = 3) that an SM holds: cut at
// divisors of the frame near 512 KB, 30 frames of 1080p made 360 CTAs for 304 places, and a frame that has no
// such divisor one CTA, which read it byte by byte.  Those 30 frames: 71 -> 42 us.
template <int C, int PH>
__device__ __forceinline__ void hist_groups(const uint8_t *p, uint64_t groups, uint32_t *mine) {
    for (uint64_t k = threadIdx.x; k < groups; k += kHistThreads) {
        uint4 v[C];
#pragma unroll
        for (int m = 0; m < C; ++m) v[m] = __ldcs(reinterpret_cast<const uint4 *>(p + 16 * C * k) + m);
#pragma unroll
        for (int m = 0; m < C; ++m) {
            const uint32_t wd[4] = {v[m].x, v[m].y, v[m].z, v[m].w};
#pragma unroll
            for (int q = 0; q < 16; ++q)
                atomicAdd(&mine[(((PH + 16 * m + q) % C) * 256 + ((wd[q >> 2] >> (8 * (q & 3))) & 255)) * 32], 1u);
        }
    }
}

template <int C>
__global__ void __launch_bounds__(kHistThreads) hist_kernel(const uint8_t *frames, uint64_t total, uint64_t frame_bytes,
                                                            uint32_t cuts, unsigned long long *hist) {
    extern __shared__ uint32_t sh[];   // C * 256 * 32
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t k = threadIdx.x; k < C * 256 * 32; k += blockDim.x) sh[k] = 0;
    __syncthreads();
    const Run run = stat_run<C>(frames, frame_bytes, cuts);
    uint32_t *mine = sh + lane;
    const uint64_t length = run.end - run.begin, head = min((uint64_t)run.head, length);
    const uint64_t groups = FHD_IN(run.end, total + 1, kSiteStats) ? (length - head) / (16 * C) : 0;
    const uint8_t *p = frames + run.begin;
    if (groups) switch (head % C) {
        case 0: hist_groups<C, 0>(p + head, groups, mine); break;
        case 1: hist_groups<C, 1 % C>(p + head, groups, mine); break;
        case 2: hist_groups<C, 2 % C>(p + head, groups, mine); break;
        default: hist_groups<C, 3 % C>(p + head, groups, mine); break;
    }
    // the head and what the groups leave
    const uint64_t done = head + 16 * C * groups;
    for (uint64_t t = threadIdx.x; t < length - 16 * C * groups; t += kHistThreads) {
        const uint64_t at = t < head ? t : t - head + done;
        if (FHD_IN(run.begin + at, total, kSiteStats)) atomicAdd(&mine[((uint32_t)(at % C) * 256 + p[at]) * 32], 1u);
    }
    __syncthreads();
    const uint64_t f = run.begin / frame_bytes;
    for (uint32_t q = threadIdx.x; q < C * 256; q += blockDim.x) {
        const uint32_t *row = sh + q * 32;
        uint32_t s = 0;
#pragma unroll 8
        for (int l = 0; l < 32; ++l) s += row[(l + q) & 31];   // rotated start: the threads of a warp read 32 banks
        if (s) atomicAdd(&hist[f * C * 256 + q], (unsigned long long)s);
    }
}

// One CTA per (frame, channel): var(Z) (Eq. 4) = S2/256 - (S1/256)^2,
// chi^2 (Eq. 5) = (256 S2 - N^2) / N, H (Eq. 10) = log2 N - (sum z log2 z) / N.
// A thread per bin: its logarithm is ~30 binary64 instructions of 64 cycles, so
// eight of them in one lane were the kernel's time.  90 histograms: 27 -> 8 us.
__global__ void __launch_bounds__(256) hist_finish_kernel(const unsigned long long *hist, uint32_t *hist32, double *out) {
    __shared__ unsigned long long zs[256];
    __shared__ double term[256];
    const uint64_t item = blockIdx.x;
    const uint32_t t = threadIdx.x;
    const unsigned long long v = hist[item * 256 + t];
    zs[t] = v;
    term[t] = v ? (double)v * log2((double)v) : 0.0;
    if (hist32) hist32[item * 256 + t] = (uint32_t)v;
    __syncthreads();
    if (t >= 32) return;
    unsigned long long s1 = 0, s2 = 0;
    double zl = 0.0;
#pragma unroll
    for (uint32_t i = t; i < 256; i += 32) {
        s1 += zs[i];
        s2 += zs[i] * zs[i];
        zl += term[i];
    }
    for (int o = 16; o; o >>= 1) {
        s1 += __shfl_xor_sync(0xffffffffu, s1, o);
        s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        zl += __shfl_xor_sync(0xffffffffu, zl, o);
    }
    if (t == 0) {
        const double N = (double)s1;
        const double m1 = N / 256.0;
        out[3 * item + 0] = (double)s2 / 256.0 - m1 * m1;
        out[3 * item + 1] = (double)(long long)(256ull * s2 - s1 * s1) / N;
        out[3 * item + 2] = log2(N) - zl / N;
    }
}

// Bytes of 32-bit word m of a 16 * C-byte group that belong to channel c.
template <int C>
__host__ __device__ constexpr uint32_t chan_mask(int m, int c) {
    uint32_t r = 0;
    for (int t = 0; t < 4; ++t)
        if ((4 * m + t) % C == c) r |= 0xFFu << (8 * t);
    return r;
}

// NPCR / UACI pass: per CTA run and 16 * C-byte groups as in hist_kernel.
// Four bytes at a time: __vabsdiffu4 gives |a - b| per byte, __vcmpne4 marks
// the differing bytes, and a channel's bytes of the word are summed with
// __dp4a through a compile-time mask.
template <int C, int PH>
__device__ __forceinline__ void npcr_groups(const uint8_t *a, const uint8_t *b, uint64_t groups, uint32_t (&changed)[C],
                                            uint32_t (&diff)[C]) {
    for (uint64_t k = threadIdx.x; k < groups; k += kStatThreads) {
        uint4 va[C], vb[C];
#pragma unroll
        for (int m = 0; m < C; ++m) {
            va[m] = __ldcs(reinterpret_cast<const uint4 *>(a + 16 * C * k) + m);
            vb[m] = __ldcs(reinterpret_cast<const uint4 *>(b + 16 * C * k) + m);
        }
#pragma unroll
        for (int m = 0; m < 4 * C; ++m) {
            const uint32_t x = (&va[m >> 2].x)[m & 3], y = (&vb[m >> 2].x)[m & 3];
            const uint32_t d = __vabsdiffu4(x, y);
            const uint32_t ne = __vcmpne4(x, y) & 0x01010101u;
#pragma unroll
            for (int c = 0; c < C; ++c) {
                constexpr uint32_t ones = 0x01010101u;
                const uint32_t mk = chan_mask<C>(m, (c + C - PH) % C);
                diff[c] = __dp4a(d & mk, ones, diff[c]);
                changed[c] = __dp4a(ne & mk, ones, changed[c]);
            }
        }
    }
}

template <int C>
__global__ void __launch_bounds__(kStatThreads) npcr_kernel(const uint8_t *a, const uint8_t *b, uint64_t total,
                                                            uint64_t frame_bytes, uint32_t cuts,
                                                            unsigned long long *acc) {
    __shared__ unsigned long long sacc[4][2];
    if (threadIdx.x < 8) sacc[threadIdx.x >> 1][threadIdx.x & 1] = 0;
    __syncthreads();
    uint32_t changed[C], diff[C];
#pragma unroll
    for (int c = 0; c < C; ++c) changed[c] = diff[c] = 0;
    const Run run = stat_run<C>(a, frame_bytes, cuts);
    const uint64_t length = run.end - run.begin, head = min((uint64_t)run.head, length);
    const bool vec = ((reinterpret_cast<uintptr_t>(a) ^ reinterpret_cast<uintptr_t>(b)) & 15) == 0;
    const uint64_t groups = vec && FHD_IN(run.end, total + 1, kSiteStats) ? (length - head) / (16 * C) : 0;
    const uint8_t *pa = a + run.begin, *pb = b + run.begin;
    if (groups) switch (head % C) {
        case 0: npcr_groups<C, 0>(pa + head, pb + head, groups, changed, diff); break;
        case 1: npcr_groups<C, 1 % C>(pa + head, pb + head, groups, changed, diff); break;
        case 2: npcr_groups<C, 2 % C>(pa + head, pb + head, groups, changed, diff); break;
        default: npcr_groups<C, 3 % C>(pa + head, pb + head, groups, changed, diff); break;
    }
    const uint64_t done = head + 16 * C * groups;
    for (uint64_t t = threadIdx.x; t < length - 16 * C * groups; t += kStatThreads) {
        const uint64_t at = t < head ? t : t - head + done;
        if (!FHD_IN(run.begin + at, total, kSiteStats)) break;
        const uint32_t c = (uint32_t)(at % C);
        const int x = pa[at], y = pb[at];
#pragma unroll
        for (int cc = 0; cc < C; ++cc)
            if ((uint32_t)cc == c) {
                changed[cc] += x != y;
                diff[cc] += (uint32_t)abs(x - y);
            }
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
        unsigned long long x = changed[c], y = diff[c];
        for (int o = 16; o; o >>= 1) {
            x += __shfl_xor_sync(0xffffffffu, x, o);
            y += __shfl_xor_sync(0xffffffffu, y, o);
        }
        if ((threadIdx.x & 31) == 0) {
            atomicAdd(&sacc[c][0], x);
            atomicAdd(&sacc[c][1], y);
        }
    }
    __syncthreads();
    const uint64_t f = run.begin / frame_bytes;
    if (threadIdx.x < 2 * C) atomicAdd(&acc[(f * C + (threadIdx.x >> 1)) * 2 + (threadIdx.x & 1)], sacc[threadIdx.x >> 1][threadIdx.x & 1]);
}

__global__ void npcr_finish_kernel(const unsigned long long *acc, uint32_t items, uint64_t wh, double *out) {
    const uint32_t item = blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= items) return;
    out[2 * item + 0] = 100.0 * (double)acc[2 * item] / (double)wh;
    out[2 * item + 1] = 100.0 * (double)acc[2 * item + 1] / ((double)wh * 255.0);
}

// Correlation: one cluster per (frame, direction); pairs[(f * 3 + d) * npairs + k] = (i, j) of x; y is the
// neighbour (0, 1), (1, 0) or (1, 1).  Exact sums sx, sy, sxx, syy, sxy per channel, then
// r = (N sxy - sx sy) / sqrt((N sxx - sx^2)(N syy - sy^2)).
//
// A pair is a read of its place and two scattered reads behind it, so what counts is how many are in flight: one
// CTA per (frame, direction) walked 40 pairs a thread one after another on 90 of the 152 SMs.  The pairs are now
// shared by the CTAs of a cluster, kLoads a thread at a time, and the sums meet in its first CTA's hands through
// distributed shared memory, with no counters to clear and no second launch.  10,000 pairs in each direction of 30
// frames: 57 -> 27 us.  A thread has at most 2^22 / 256 pairs, whose sums of squares
// fit 32 bits.
template <int C>
__global__ void __launch_bounds__(kStatThreads) corr_kernel(const uint8_t *frames, uint32_t h, uint32_t w,
                                                            const uint32_t *pairs, uint32_t npairs, long long *sums,
                                                            double *out, unsigned *status) {
    constexpr int kLoads = 4;
    __shared__ unsigned long long red[kStatWarps][C][5];
    __shared__ long long part[C][5];
    namespace cg = cooperative_groups;
    const cg::cluster_group cluster = cg::this_cluster();
    const uint32_t parts = cluster.num_blocks(), rank = cluster.block_rank(), item = blockIdx.x / parts;
    const uint32_t f = item / 3, d = item % 3;
    const uint32_t di = d == 0 ? 0 : 1, dj = d == 1 ? 0 : 1;
    const uint8_t *F = frames + (uint64_t)f * h * w * C;
    const uint32_t *pp = pairs + 2 * ((uint64_t)item * npairs);
    uint32_t acc[C][5] = {};
    const uint32_t stride = parts * kStatThreads;
    for (uint32_t k0 = rank * kStatThreads + threadIdx.x; k0 < npairs; k0 += kLoads * stride) {
        uint64_t at[kLoads];
        bool use[kLoads];
        uint8_t x[kLoads][C], y[kLoads][C];
#pragma unroll
        for (int u = 0; u < kLoads; ++u) {
            const uint32_t k = k0 + u * stride;   // npairs <= 2^22
            use[u] = k < npairs;
            const uint32_t i = use[u] ? pp[2 * k] : 0, j = use[u] ? pp[2 * k + 1] : 0;
            if (use[u] && (i >= h - di || j >= w - dj)) {   // out of the frame: counted nowhere, reported
                atomicOr(status, 1u);
                use[u] = false;
            }
            at[u] = (uint64_t)i * w + j;
            if (use[u] && !FHD_IN((at[u] + (uint64_t)di * w + dj) * C + C - 1, (uint64_t)h * w * C, kSiteStats))
                use[u] = false;
        }
#pragma unroll
        for (int u = 0; u < kLoads; ++u)
#pragma unroll
            for (int c = 0; c < C; ++c) {
                x[u][c] = use[u] ? __ldg(F + at[u] * C + c) : 0;
                y[u][c] = use[u] ? __ldg(F + (at[u] + (uint64_t)di * w + dj) * C + c) : 0;
            }
#pragma unroll
        for (int u = 0; u < kLoads; ++u)
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const uint32_t a = x[u][c], b = y[u][c];
                acc[c][0] += a;
                acc[c][1] += b;
                acc[c][2] += a * a;
                acc[c][3] += b * b;
                acc[c][4] += a * b;
            }
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
        for (int m = 0; m < 5; ++m) {
            const unsigned long long lo = __reduce_add_sync(0xffffffffu, acc[c][m] & 0xffffu);
            const unsigned long long hi = __reduce_add_sync(0xffffffffu, acc[c][m] >> 16);
            if (lane == 0) red[warp][c][m] = lo + (hi << 16);
        }
    __syncthreads();
    if (threadIdx.x < 5 * C) {
        long long v = 0;
#pragma unroll
        for (int w8 = 0; w8 < kStatWarps; ++w8) v += (long long)(&red[w8][0][0])[threadIdx.x];
        (&part[0][0])[threadIdx.x] = v;
    }
    cluster.sync();
    if (rank == 0 && threadIdx.x < C) {
        const uint32_t c = threadIdx.x;
        long long s[5] = {0, 0, 0, 0, 0};
        for (uint32_t p = 0; p < parts; ++p) {
            const long long *q = cluster.map_shared_rank(&part[c][0], p);
#pragma unroll
            for (int m = 0; m < 5; ++m) s[m] += q[m];
        }
        const long long N = (long long)npairs;
        long long *so = sums + ((uint64_t)(f * C + c) * 3 + d) * 5;
        for (int m = 0; m < 5; ++m) so[m] = s[m];
        const double num = (double)(N * s[4] - s[0] * s[1]);
        const double vx = (double)(N * s[2] - s[0] * s[0]), vy = (double)(N * s[3] - s[1] * s[1]);
        out[(uint64_t)(f * C + c) * 3 + d] = num / sqrt(vx * vy);
    }
    cluster.sync();   // the first CTA has read the others' sums
}

template <int C>
cudaError_t corr_launch(const uint8_t *frames, uint32_t count, uint32_t h, uint32_t w, const uint32_t *pairs,
                        uint32_t npairs, long long *sums, double *out, unsigned *status, cudaStream_t s) {
    // CTAs to an item: twice as many while its pairs keep their threads in loads (1,024 pairs a CTA), and the items have no
    // more than three CTAs to an SM, or ten where a CTA keeps 3,500 pairs; a CTA more costs ~6 ns.  Eight throughout took
    // 176 us for 1,025 pairs of 1,000 frames, 33 with one; by this rule 10,000 pairs of 30, 60, 200 and 300 frames take
    // 27, 43, 87 and 64 us (eight: 31, 46, 110, 111; one: 41, 53, 122, 64).
    const uint64_t items = 3ull * count, sms = sm_count();
    uint32_t parts = 1;
    while (parts < 8 && npairs > 1024 * parts &&
           (items * 2 * parts <= 3 * sms || (items * 2 * parts <= 10 * sms && npairs / (2 * parts) >= 3500)))
        parts *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(count * 3 * parts);
    cfg.blockDim = dim3(kStatThreads);
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = parts;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, corr_kernel<C>, frames, h, w, pairs, npairs, sums, out, status);
}

// Local Shannon entropy: one CTA per (frame, block) builds the block's
// histograms in shared memory and writes each channel's entropy; a second
// kernel takes the mean over the k blocks in block order (a fixed summation
// order, so the result does not depend on scheduling).
//
// Read row by row, a block was 44 round trips to memory, and its 768 terms
// z log2 z, ~30 binary64 instructions each, held the binary64 pipes for most
// of the rest.  The bytes are now read kLoads to a thread at a time whatever
// the row, and a term is computed once for each count that occurs up to 256
// (the counts of a noise block of 44 x 44 are under 32, one warp's work; a flat
// block's one count is a warp's work too).  900 noise blocks of 44 x 44: 82 -> 22 us.
template <int C>
__global__ void __launch_bounds__(kStatThreads) block_entropy_kernel(const uint8_t *frames, uint32_t h, uint32_t w,
                                                                     const uint32_t *blocks, uint32_t k, uint32_t bs,
                                                                     double *ent, unsigned *status) {
    constexpr int kLoads = 8;
    __shared__ uint32_t hist[C][256];
    __shared__ double term[256];   // of count z in term[z - 1]
    __shared__ bool occurs[256];   // whether a bin has that count
    const uint32_t f = blockIdx.x / k, q = blockIdx.x % k;
    const uint8_t *F = frames + (uint64_t)f * h * w * C;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t r0 = blocks[2 * ((uint64_t)f * k + q)], c0 = blocks[2 * ((uint64_t)f * k + q) + 1];
    const bool inside = r0 <= h - bs && c0 <= w - bs;   // bs <= h, w
    for (uint32_t t = threadIdx.x; t < C * 256; t += kStatThreads) (&hist[0][0])[t] = 0;
    occurs[threadIdx.x] = false;
    __syncthreads();
    if (inside) {
        const uint32_t row = bs * C, down = kStatThreads / row, along = kStatThreads % row;
        uint32_t i = threadIdx.x / row, t = threadIdx.x % row;
        while (i < bs) {
            uint8_t v[kLoads];
            uint32_t c[kLoads];
#pragma unroll
            for (int u = 0; u < kLoads; ++u) {
                const uint64_t at = ((uint64_t)(r0 + i) * w + c0) * C + t;
                c[u] = C;
                if (i < bs && FHD_IN(at, (uint64_t)h * w * C, kSiteStats)) {
                    v[u] = __ldg(F + at);
                    c[u] = t % C;
                }
                i += down;
                t += along;
                if (t >= row) {
                    t -= row;
                    ++i;
                }
            }
#pragma unroll
            for (int u = 0; u < kLoads; ++u)
                if (c[u] < C) atomicAdd(&hist[c[u]][v[u]], 1u);
        }
    } else if (threadIdx.x == 0) {
        atomicOr(status, 1u);
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < C; ++c) {
        const uint32_t z = hist[c][threadIdx.x];
        if (z - 1 < 256) occurs[z - 1] = true;
    }
    __syncthreads();
    if (occurs[threadIdx.x]) term[threadIdx.x] = (double)(threadIdx.x + 1) * log2((double)(threadIdx.x + 1));
    __syncthreads();
    if (warp < C) {
        double e = 0.0;
        for (int i = lane; i < 256; i += 32) {
            const uint32_t z = hist[warp][i];
            if (z) e += z <= 256 ? term[z - 1] : (double)z * log2((double)z);
        }
        for (int o = 16; o; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
        const double T = (double)bs * (double)bs;
        if (lane == 0) ent[((uint64_t)f * k + q) * C + warp] = log2(T) - e / T;
    }
}

__global__ void block_entropy_mean_kernel(const double *ent, uint32_t count, uint32_t C, uint32_t k, double *out) {
    const uint32_t item = blockIdx.x * blockDim.x + threadIdx.x;
    if (item >= count * C) return;
    const uint32_t f = item / C, c = item % C;
    double acc = 0.0;
#pragma unroll 8
    for (uint32_t q = 0; q < k; ++q) acc += ent[((uint64_t)f * k + q) * C + c];
    out[item] = acc / (double)k;
}

unsigned zero_grid(uint64_t n) {
    const uint64_t g = (n + 255) / 256;
    return (unsigned)(g < 1024 ? (g ? g : 1) : 1024);
}

}  // namespace

cudaError_t launch_stats_histogram(const uint8_t *frames, uint32_t count, uint64_t frame_bytes, uint32_t C,
                                   unsigned long long *hist64, uint32_t *hist32, double *out, cudaStream_t s) {
    const uint64_t total = (uint64_t)count * frame_bytes;
    const uint64_t items = (uint64_t)count * C;
    zero_kernel<<<zero_grid(items * 256), 256, 0, s>>>(hist64, items * 256);
    note_launch();
    const size_t smem = (size_t)C * 256 * 32 * sizeof(uint32_t);
    cudaError_t e = cudaFuncSetAttribute(hist_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 131072);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(hist_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 131072);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(hist_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, 131072);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(hist_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 131072);
    if (e != cudaSuccess) return e;
    // CTAs of 32 C KB of counters and 512 threads, at most four of them to an SM; a run of 64 KB at least,
    // for the sum of the copies
    const uint32_t cuts = stat_cuts(frame_bytes, count, C, sm_count() * std::min(4u, 227u / (32 * C + 1)), 1u << 16, 1u << 20);
    const uint64_t ctas = (uint64_t)cuts * count;
    switch (C) {
        case 1: hist_kernel<1><<<(unsigned)ctas, kHistThreads, smem, s>>>(frames, total, frame_bytes, cuts, hist64); break;
        case 2: hist_kernel<2><<<(unsigned)ctas, kHistThreads, smem, s>>>(frames, total, frame_bytes, cuts, hist64); break;
        case 3: hist_kernel<3><<<(unsigned)ctas, kHistThreads, smem, s>>>(frames, total, frame_bytes, cuts, hist64); break;
        default: hist_kernel<4><<<(unsigned)ctas, kHistThreads, smem, s>>>(frames, total, frame_bytes, cuts, hist64); break;
    }
    note_launch();
    hist_finish_kernel<<<(unsigned)items, 256, 0, s>>>(hist64, hist32, out);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_stats_npcr(const uint8_t *a, const uint8_t *b, uint32_t count, uint64_t frame_bytes, uint32_t C,
                              uint64_t wh, unsigned long long *acc, double *out, cudaStream_t s) {
    const uint64_t total = (uint64_t)count * frame_bytes;
    const uint64_t items = (uint64_t)count * C;
    zero_kernel<<<zero_grid(items * 2), 256, 0, s>>>(acc, items * 2);
    note_launch();
    // eight CTAs of 256 threads to an SM; runs of 64 KB where there are more than a round of them
    const uint32_t cuts = stat_cuts(frame_bytes, count, C, sm_count() * 8, 1u << 13, 1u << 16);
    const unsigned grid = cuts * count;
    switch (C) {
        case 1: npcr_kernel<1><<<grid, kStatThreads, 0, s>>>(a, b, total, frame_bytes, cuts, acc); break;
        case 2: npcr_kernel<2><<<grid, kStatThreads, 0, s>>>(a, b, total, frame_bytes, cuts, acc); break;
        case 3: npcr_kernel<3><<<grid, kStatThreads, 0, s>>>(a, b, total, frame_bytes, cuts, acc); break;
        default: npcr_kernel<4><<<grid, kStatThreads, 0, s>>>(a, b, total, frame_bytes, cuts, acc); break;
    }
    note_launch();
    npcr_finish_kernel<<<(unsigned)((items + 255) / 256), 256, 0, s>>>(acc, (uint32_t)items, wh, out);
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_stats_correlation(const uint8_t *frames, uint32_t count, uint32_t h, uint32_t w, uint32_t C,
                                     const uint32_t *pairs, uint32_t npairs, long long *sums, double *out,
                                     unsigned *status, cudaStream_t s) {
    cudaError_t e;
    switch (C) {
        case 1: e = corr_launch<1>(frames, count, h, w, pairs, npairs, sums, out, status, s); break;
        case 2: e = corr_launch<2>(frames, count, h, w, pairs, npairs, sums, out, status, s); break;
        case 3: e = corr_launch<3>(frames, count, h, w, pairs, npairs, sums, out, status, s); break;
        default: e = corr_launch<4>(frames, count, h, w, pairs, npairs, sums, out, status, s); break;
    }
    if (e != cudaSuccess) return e;
    note_launch();
    return cudaGetLastError();
}

cudaError_t launch_stats_local_entropy(const uint8_t *frames, uint32_t count, uint32_t h, uint32_t w, uint32_t C,
                                       const uint32_t *blocks, uint32_t k, uint32_t bs, double *ent, double *out,
                                       unsigned *status, cudaStream_t s) {
    switch (C) {
        case 1: block_entropy_kernel<1><<<count * k, kStatThreads, 0, s>>>(frames, h, w, blocks, k, bs, ent, status); break;
        case 2: block_entropy_kernel<2><<<count * k, kStatThreads, 0, s>>>(frames, h, w, blocks, k, bs, ent, status); break;
        case 3: block_entropy_kernel<3><<<count * k, kStatThreads, 0, s>>>(frames, h, w, blocks, k, bs, ent, status); break;
        default: block_entropy_kernel<4><<<count * k, kStatThreads, 0, s>>>(frames, h, w, blocks, k, bs, ent, status); break;
    }
    note_launch();
    block_entropy_mean_kernel<<<(count * C + 127) / 128, 128, 0, s>>>(ent, count, C, k, out);
    note_launch();
    return cudaGetLastError();
}

}  // namespace fhd

FHD_BOUNDS_TAKER(take_bounds_stats)
