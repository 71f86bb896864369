// exa_reduce.h -- the reductions that follow an evaluation kernel: CSC values, dense gradient,
// augmented constraint rows and the objective, as independent jobs of one launch.  No atomics: every
// output element is written by one thread, from entries in an order fixed at creation.
//
// What bounds them: the gathers.  A job moves an index, a value and a result per entry (20 bytes),
// and on models that fit the L2 cache it takes a few microseconds, less than the gap between two
// dependent launches.  So all jobs of a step are blocks of one kernel, and that kernel is launched
// with programmatic stream serialization: its blocks become resident while the evaluation kernel
// drains (when its blocks have finished their tiles), load their indices (constant since creation) and
// only then wait for its results.
//
// Measured (GB300, whole exa_eval_all steps; before: one kernel per reduction on three streams, the
// multi-entry CSC segments added onto a first pass): this alone took a 1000-variable model from 25.4 to
// 15.4 us, a 30,000-bus network from 48.6 to 35.8, PDE 1000^2 from 94.6 to 80, PDE 2001^2 mixed from 307
// to 274, the 256-network batch from 795 to 790 (with the later changes to the step's graph, the FP64
// gradient and the FP64 compressed sums: 12.3, 33.2, 72.7, 273 and 774 us).  On the batch the kernel takes
// 0.33 ms for 52 M Jacobian gathers and those of the Hessian sums; on its first 96 networks 121 us, 672 MB of
// DRAM (5.6 TB/s, caches cold), 26.6 M sectors loaded, 66 % of the warps resident.  It gains from more gathers
// in flight only up to 48 warps x 8 per SM (64 warps: 808 us a step against 799; 40: 892; 4 or 16 gathers per
// thread at 48 warps: 825, 818).
#pragma once

#include <cuda_runtime.h>

namespace exa_red {

// Waits until the kernels this one depends on have completed and their writes are visible (no-op
// for an ordinary launch), and returns src: loads through the returned pointer cannot be moved ahead of
// the wait, whatever kind of load they are.
static __device__ __forceinline__ const double *wait_inputs(const double *src) {
    asm volatile("griddepcontrol.wait;" : "+l"(src) : : "memory");
    return src;
}

enum Kind {
    PERM = 0,  // dst[p] = src[perm[p]] for perm[p] >= 0; 0.0 for EMPTY; nothing for ELSEWHERE
    SEG,       // dst[row[s]] = the values src[perm[q]], q in [ptr[s], ptr[s+1]), added in ascending q
    WSEG,      // the same over q in [ptr[2 s], ptr[2 s + 1]) for longer segments: one warp each, lanes'
               // strided sums, then a tree
    BSEG,      // the same, one block each
    CHUNK,     // dst[c] = sum of src[perm[q]], q in [ptr[2 c], ptr[2 c + 1]) (a piece of a long segment)
    CSUM,      // dst[row[s]] = the pieces src[ptr[s] .. ptr[s+1]) of long segment s
    OBJ,       // dst[0] = sum of the objective partials src[0 .. n)
    FILL       // dst[p] = 0.0, p in [lo, n), where bit p of the mask is clear
};
constexpr int EMPTY = -1, ELSEWHERE = -2;  // codes in a PERM list

struct Job {
    int kind = PERM;
    int blk0 = 0;    // first block of the job
    int n = 0;       // positions, segments, pieces or partials
    int wide = 0;    // PERM: 8 positions per thread instead of 2; SEG: 64 segments per warp instead of 32
    int add = 0;     // SEG, WSEG, BSEG, CSUM: the segment is added onto dst[row[s]]
    int lo = 0;      // FILL: first position (n is the end)
    const int *ptr = nullptr, *perm = nullptr, *row = nullptr;  // FILL: ptr is the mask
    const double *src = nullptr;
    double *dst = nullptr;
};
constexpr int MAX_JOBS = 16;
struct Jobs {
    int nj = 0;
    int sums = 0;   // blocks of the sums, which come first in the list; the streaming jobs follow
    unsigned long long *stamp = nullptr;  // if set: device time (ns) at which the inputs were complete
    int every = 1;  // > 1: every `every`-th block of the launch is one of the sums (while they last)
    // k_reduce<true>, products of stored entries with a vector: entry e stands for src[e] * vec[other[e]];
    // e >= wrap for src[e - wrap] (the second mention of a symmetric entry)
    const double *vec = nullptr;
    const int *other = nullptr;
    int wrap = 0x7fffffff;
    Job j[MAX_JOBS];
};

constexpr int THREADS = 256;
constexpr int CHUNK_LEN = 4096;  // entries of a long segment per block
constexpr int SHORT_MAX = 32;    // longest segment a single lane adds up (any length in CSC sums: ascending COO order)
// Longest segment a single warp, a single block adds up: an iteration of either is a gather latency of
// about 1.2 us for 4 entries per thread.  One 2000-entry variable of 2000 took a warp 42 us, a block 8.
constexpr int WARP_MAX = 256, BLOCK_MAX = 8192;

// Blocks of a job; decides `wide`: enough work for two blocks per SM at the larger share per thread.
// In 64 bits: n reaches 2^31 - 1.
inline long long plan(Job &j, int sms) {
    const long long n = j.n, two = 2LL * sms;
    auto blocks = [n](long long per) { return (n + per - 1) / per; };
    switch (j.kind) {
    case PERM: j.wide = n >= two * 2048; return blocks(j.wide ? 2048 : 512);
    case SEG: j.wide = n >= two * 512; return blocks(j.wide ? 512 : 256);
    case WSEG: case CSUM: return blocks(8);
    case CHUNK: case BSEG: return n;
    case OBJ: return 1;
    default: return ((n + 31) / 32 - j.lo / 32 + 255) / 256;
    }
}

template <bool PROD>
static __device__ __forceinline__ double entry(const Jobs &J, const double *src, int e) {
    if (!PROD) return __ldcg(src + e);
    return __ldcg(src + (e >= J.wrap ? e - J.wrap : e)) * J.vec[__ldg(J.other + e)];
}

// PERM: a block covers ILP x 256 consecutive positions; thread t takes positions t, t + 256, ... so
// that the index loads and the stores stay coalesced, and its ILP gathers are in flight together.
template <int ILP, bool PROD>
static __device__ __forceinline__ void perm_job(const Jobs &J, const Job &j, int blk) {
    const unsigned i0 = (unsigned)blk * (THREADS * ILP) + threadIdx.x;
    const int left = (int)((unsigned)j.n - i0);  // may be negative
    int p[ILP];
    {
        const int *perm = j.perm + i0;
#pragma unroll
        for (int u = 0; u < ILP; u++) p[u] = THREADS * u < left ? __ldg(perm + THREADS * u) : ELSEWHERE;
    }
    const double *src = wait_inputs(j.src);
    double v[ILP];
#pragma unroll
    for (int u = 0; u < ILP; u++) v[u] = p[u] >= 0 ? entry<PROD>(J, src, p[u]) : 0.0;
    double *dst = j.dst + i0;
#pragma unroll
    for (int u = 0; u < ILP; u++)
        if (p[u] != ELSEWHERE) dst[THREADS * u] = v[u];
}

// SEG: one warp takes 32 x G consecutive segments, whose entries are one contiguous range of sorted
// positions: all lanes gather that range in pieces of 256 into shared memory (8 independent loads
// per lane), then every lane adds up its own G segments from there.
constexpr int PIECE = 256;
template <int G, bool PROD>
static __device__ __forceinline__ void seg_job(const Jobs &J, const Job &j, int blk, double *buf) {
    const int lane = threadIdx.x & 31;
    const unsigned s0 = ((unsigned)blk * (THREADS / 32) + (threadIdx.x >> 5)) * (32 * G);
    if (s0 >= (unsigned)j.n) {
        wait_inputs(j.src);
        return;
    }
    double *b = buf + (threadIdx.x >> 5) * PIECE;
    const int left = j.n - (int)s0 - lane;  // segment g of this lane exists where 32 g < left
    const int *ptr = j.ptr + s0;
    const int beg = __ldg(ptr), end = __ldg(ptr + min(j.n - (int)s0, 32 * G));
    int myb[G], mye[G], p[PIECE / 32];
#pragma unroll
    for (int g = 0; g < G; g++) {
        myb[g] = 32 * g < left ? __ldg(ptr + lane + 32 * g) : end;
        mye[g] = 32 * g < left ? __ldg(ptr + lane + 32 * g + 1) : end;
    }
#pragma unroll
    for (int u = 0; u < PIECE / 32; u++) p[u] = beg + lane + 32 * u < end ? __ldg(j.perm + beg + lane + 32 * u) : -1;
    const double *src = wait_inputs(j.src);
    double acc[G];
#pragma unroll
    for (int g = 0; g < G; g++) acc[g] = j.add && 32 * g < left ? j.dst[__ldg(j.row + s0 + lane + 32 * g)] : 0.0;
    for (int c0 = beg;;) {
#pragma unroll
        for (int u = 0; u < PIECE / 32; u++)
            if (p[u] >= 0) b[lane + 32 * u] = entry<PROD>(J, src, p[u]);
        __syncwarp();
        const int c1 = min(c0 + PIECE, end);
#pragma unroll
        for (int g = 0; g < G; g++) {
            int q = max(myb[g], c0);
            const int qe = min(mye[g], c1);
            if (!j.add && q == myb[g] && q < qe) acc[g] = b[q++ - c0];  // the first entry as it is
            for (; q < qe; q++) acc[g] += b[q - c0];
        }
        c0 = c1;
        if (c0 >= end) break;
        __syncwarp();
#pragma unroll
        for (int u = 0; u < PIECE / 32; u++) p[u] = c0 + lane + 32 * u < end ? __ldg(j.perm + c0 + lane + 32 * u) : -1;
    }
#pragma unroll
    for (int g = 0; g < G; g++)
        if (32 * g < left) j.dst[__ldg(j.row + s0 + lane + 32 * g)] = acc[g];
}

// Sum over [beg, end) of src[perm[q]] (perm null: src[q]) by `width` threads, this one being number t:
// strided partial sums with 8 independent gathers in flight per thread.
template <bool PROD = false>
static __device__ __forceinline__ double strided_sum(const double *src, const int *perm, int beg, int end, int t,
                                                     int width, const Jobs *J = nullptr) {
    double s = 0.0;
    for (unsigned q = beg + t; q < (unsigned)end; q += 8 * width) {  // end < 2^31: no wrap
        double v[8];
#pragma unroll
        for (int u = 0; u < 8; u++) {
            const unsigned e = q + u * width;
            v[u] = e >= (unsigned)end ? 0.0 : PROD ? entry<true>(*J, src, __ldg(perm + e)) : perm ? src[__ldg(perm + e)] : src[e];
        }
#pragma unroll
        for (int u = 0; u < 8; u++) s += v[u];
    }
    return s;
}
static __device__ __forceinline__ double warp_sum(double s) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    return s;
}
static __device__ __forceinline__ double block_sum(double s, double *buf) {
    s = warp_sum(s);
    if ((threadIdx.x & 31) == 0) buf[threadIdx.x >> 5] = s;
    __syncthreads();
    double t = 0.0;
    if (threadIdx.x == 0)
        for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += buf[w];
    return t;
}

template <bool PROD>
static __global__ void __launch_bounds__(THREADS, 6) k_reduce(const __grid_constant__ Jobs J) {
    __shared__ double buf[(THREADS / 32) * PIECE];
    if (J.stamp && blockIdx.x == 0 && threadIdx.x == 0) {
        wait_inputs(nullptr);
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(*J.stamp) : : "memory");
    }
    // block of the job list: as launched, or every `every`-th one a block of a sum
    int vb = (int)blockIdx.x;
    if (J.every > 1) {
        const int g = vb / J.every;
        if (g < J.sums) vb = vb == g * J.every ? g : J.sums + vb - g - 1;
    }
    int i = 0;
    while (i + 1 < J.nj && vb >= J.j[i + 1].blk0) i++;
    const Job &j = J.j[i];
    const int blk = vb - j.blk0;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    switch (j.kind) {
    case PERM:
        if (j.wide) perm_job<8, PROD>(J, j, blk);
        else perm_job<2, PROD>(J, j, blk);
        break;
    case SEG:
        if (j.wide) seg_job<2, PROD>(J, j, blk, buf);
        else seg_job<1, PROD>(J, j, blk, buf);
        break;
    case WSEG: case CSUM: {
        const int s = blk * (THREADS / 32) + w;
        const double *src = wait_inputs(j.src);
        if (s >= j.n) break;
        const int *r = j.kind == CSUM ? j.ptr + s : j.ptr + 2 * (long long)s;
        // (the pieces of a long segment are sums already: never in a k_reduce<true> launch)
        const double t = warp_sum(strided_sum<PROD>(src, j.kind == CSUM ? nullptr : j.perm, __ldg(r), __ldg(r + 1), lane, 32, &J));
        if (lane == 0) {
            double *d = j.dst + __ldg(j.row + s);
            *d = j.add ? *d + t : t;
        }
        break;
    }
    case CHUNK: case BSEG: {
        const double *src = wait_inputs(j.src);
        const double t = block_sum(strided_sum<PROD>(src, j.perm, __ldg(j.ptr + 2 * (long long)blk), __ldg(j.ptr + 2 * (long long)blk + 1), threadIdx.x, THREADS, &J), buf);
        if (threadIdx.x == 0) {
            double *d = j.dst + (j.kind == BSEG ? __ldg(j.row + blk) : blk);
            *d = j.add ? *d + t : t;
        }
        break;
    }
    case OBJ: {
        const double *src = wait_inputs(j.src);
        const double t = block_sum(strided_sum(src, nullptr, 0, j.n, threadIdx.x, THREADS), buf);
        if (threadIdx.x == 0) j.dst[0] = t;
        break;
    }
    default: {  // FILL: 32 positions per thread, one mask word
        const long long word = j.lo / 32 + (long long)blk * THREADS + threadIdx.x;
        unsigned keep = word * 32 < j.n ? __ldg((const unsigned *)j.ptr + word) : 0xffffffffu;
        wait_inputs(nullptr);
        // a warp writes its 1024 positions as 32 coalesced rows
        for (int r = 0; r < 32; r++) {
            const unsigned k = __shfl_sync(0xffffffffu, keep, r);
            const long long p = (word - lane + r) * 32 + lane;
            if (p >= j.lo && p < j.n && !((k >> lane) & 1u)) j.dst[p] = 0.0;
        }
        break;
    }
    }
}

// f[0] = the sum of n objective partials, one CTA (the whole launch of the objective callbacks).
static __global__ void __launch_bounds__(1024) k_obj_final(const double *part, int n, double *f) {
    __shared__ double buf[32];
    part = wait_inputs(part);
    const double t = block_sum(strided_sum(part, nullptr, 0, n, threadIdx.x, blockDim.x), buf);
    if (threadIdx.x == 0) f[0] = t;
}

}  // namespace exa_red
