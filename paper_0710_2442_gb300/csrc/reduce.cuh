// reduce.cuh -- deterministic FP64 global reductions fused into kernels.
//
// Every block sums its threads' FP64 values (block_sum: integers of a common
// scale, rounded once) and writes one partial.  Who adds the partials up:
//  - FIN_PARTIAL: the blocks of the kernel that uses the sum, all the same way
//    (sum_partials; the CG iterations, blas.cu);
//  - else a ticket from a global counter decides: the block that draws the last
//    one sums all partials in a fixed order (thread t adds partials t, t+B, ...;
//    then block_sum), runs the finisher that turns the sum into solver scalars,
//    and resets the counter for the next launch on the stream.
// No result depends on block scheduling, and no block ever waits for another one.
#pragma once

#include "common.cuh"

namespace wl {

enum FinOp {
    FIN_STORE = 0,     // result[0] = sum
    FIN_CG_BETA = 3,   // |r|^2: beta = |r|^2 / gam, gam = |r|^2
    FIN_ADD = 4,       // result[0] += sum
    FIN_CG_GAM = 5,    // |r|^2: gam = |r|^2 (start of a CG)
    FIN_PARTIAL = 6    // the blocks' partials stay where they are: the next kernel sums them
};

// Scalars of one CG solve, kept on the device so that iterations never wait
// for the host.
struct CGScalars {
    double gam;      // |r|^2 of the normal-equation residual r = Mhat^dag s
    double alpha;
    double beta;
    double pq;       // |Mhat p|^2
    double snorm2;   // |s|^2, recursively updated Schur residual
    double stop2;    // the inner iteration ends when snorm2 <= stop2
    int done;        // 1: converged (snorm2 <= stop2), 2: maxiter, 3: NaN/Inf, 4: finished earlier
    int iter;        // iterations completed since the counter was last reset
    int maxiter;     // iteration cap for this inner solve
    int iter2;       // iter and gam as the x, s update left them for the p update (blas.cu)
    double gam2;
};

// A reduction may have several independent slots (one per right-hand side):
// slot k uses partials[k * slot_cap ...], counter[k], result[k] and sc[k].
struct RedArgs {
    double* partials;       // slot_cap partials per slot (slot_cap >= blocks per slot)
    unsigned int* counter;  // one per slot: 0 before the launch; reset to 0 by the last block
    double* result;         // FIN_STORE / FIN_ADD targets (one per slot)
    CGScalars* sc;          // FIN_CG_* targets (one per slot)
    int op;
    int slot_cap;
};

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sum over the block by FP64 additions; valid in thread 0.
inline __device__ __noinline__ double block_sum_fp64(double v) {
    __shared__ double sm[32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = (blockDim.x + 31) >> 5;
    v = warp_sum(v);
    __syncthreads();  // protects sm against a previous use
    if (lane == 0) sm[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < nwarps ? sm[lane] : 0.0;
        v = warp_sum(v);
    }
    return v;
}

// A term of block_sum_of: the value >= 0 with words hi, lo in units of 2^(e - 1023 - 61), to nearest;
// e: the largest term's exponent field, 128 or more.  At most 2^62.
__host__ __device__ __forceinline__ unsigned long long sum_term(unsigned hi, unsigned lo, int e) {
    const unsigned mh = (hi & 0xFFFFFu) | (hi >> 20 ? 0x100000u : 0u);
    int t = 2 + e - (int)(hi >> 20);  // from the top of 64 bits
    t = t < 65 ? t : 65;
    const unsigned long long y = ((unsigned long long)mh << 32 | lo) << 10;  // half of that
    return ((y >> (t - 2)) + 1) >> 1;
}
// The bits of the double nearest to (s2 2^42 + s1 2^21 + s0) 2^(e - 1023 - 61), a sum of at
// most 2048 terms (s2 <= 2^31, s1 and s0 < 2^32) of which one is 2^61 or more.
__host__ __device__ __forceinline__ unsigned long long sum_bits(unsigned s2, unsigned s1, unsigned s0, int e) {
    const unsigned long long a = ((unsigned long long)s2 << 21) + s1 + (s0 >> 21);  // 2^40 .. 2^52
    const unsigned r = s0 & 0x1FFFFFu;                                             // the sum is a 2^21 + r
#ifdef __CUDA_ARCH__
    const int n = __clzll((long long)a);
#else
    const int n = __builtin_clzll(a);
#endif
    const bool more = n < 21 && (r & ((1u << (21 - n)) - 1));
    const unsigned long long m = a << n | ((unsigned long long)r << 43) >> (64 - n) | (more ? 1u : 0u);
    const unsigned long long q = m >> 11;  // 53 bits; the others round, to nearest even
    const unsigned up = ((unsigned)m & 0x7FFu) + ((unsigned)q & 1) > 0x400u;
    const int field = e + 23 - n;  // of the result, before the rounding
    if (field >= 2047) return 0x7FFULL << 52;
    return q + up + ((unsigned long long)(field - 1) << 52);  // q's leading bit adds 1 to the field
}

// Sum over the block of N values >= 0 a thread; valid in thread 0.  An FP64 addition
// takes the FP64 pipe 64 cycles, and a shuffle tree is ten of them in a row.
// Here the values become integers of 62 bits below the block's largest
// exponent, in three limbs that are added per thread and then by a warp with one
// instruction each (redux); the sum is rounded to FP64 once.  A term within 2^-9 of the
// largest one is exact, a smaller one is rounded to 2^-62 of the scale: a single value comes
// back as it is, and a sum of n terms is off by at most half a unit in its last place and
// n 2^-62 of its largest term (a tree of FP64 additions: half a unit at each of its levels).
// Zeros, tiny values, Inf and NaN take the FP64 additions.
// A limb's sum fits 32 bits: 21 bits, N blockDim <= 2048 values.
template <int N>
__device__ __forceinline__ double block_sum_of(const double (&v)[N]) {
    __shared__ unsigned smx[32];
    __shared__ unsigned sl[3][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int nwarps = (blockDim.x + 31) >> 5;
    unsigned m = 0;
#pragma unroll
    for (int i = 0; i < N; i++) m = max(m, (unsigned)__double2hiint(v[i]));
    m = __reduce_max_sync(0xffffffffu, m);  // a sign bit or a NaN comes out on top
    __syncthreads();  // protects the arrays against a previous use
    if (lane == 0) smx[warp] = m;
    __syncthreads();
    m = __reduce_max_sync(0xffffffffu, lane < nwarps ? smx[lane] : 0u);
    const int e = (int)(m >> 20);
    if (e < 128 || e >= 2047) {
        double a = v[0];
#pragma unroll
        for (int i = 1; i < N; i++) a += v[i];
        return block_sum_fp64(a);
    }
    unsigned l[3] = {0, 0, 0};
#pragma unroll
    for (int i = 0; i < N; i++) {
        const unsigned long long n = sum_term((unsigned)__double2hiint(v[i]), (unsigned)__double2loint(v[i]), e);
        l[0] += (unsigned)n & 0x1FFFFFu;
        l[1] += (unsigned)(n >> 21) & 0x1FFFFFu;
        l[2] += (unsigned)(n >> 42);
    }
#pragma unroll
    for (int k = 0; k < 3; k++) l[k] = __reduce_add_sync(0xffffffffu, l[k]);
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < 3; k++) sl[k][warp] = l[k];
    }
    __syncthreads();
    if (warp != 0) return 0.0;
#pragma unroll
    for (int k = 0; k < 3; k++) l[k] = __reduce_add_sync(0xffffffffu, lane < nwarps ? sl[k][lane] : 0u);
    return __longlong_as_double((long long)sum_bits(l[2], l[1], l[0], e));
}
__device__ inline double block_sum(double v) {
    const double one[1] = {v};
    return block_sum_of(one);
}

__device__ inline void run_finisher(const RedArgs& r, int slot, double sum) {
    CGScalars* sc = r.sc ? r.sc + slot : nullptr;
    switch (r.op) {
        case FIN_STORE: r.result[slot] = sum; break;
        case FIN_ADD: r.result[slot] += sum; break;
        case FIN_CG_GAM:
            sc->gam = sum;
            if (!isfinite(sum)) sc->done = 3;
            break;
        case FIN_CG_BETA:
            if (!isfinite(sum)) { sc->done = 3; sc->beta = 0.0; break; }
            sc->beta = sc->gam > 0.0 ? sum / sc->gam : 0.0;
            sc->gam = sum;
            break;
    }
}

// Called by all threads of every block that reduces into `slot` (uniformly):
// nblocks blocks contribute to the slot, this block is number bid of them.
__device__ inline void grid_reduce(double v, const RedArgs& r, int slot, unsigned int nblocks, unsigned int bid) {
    const double bs = block_sum(v);
    __shared__ int s_last;
    double* part = r.partials + (size_t)slot * r.slot_cap;
    if (r.op == FIN_PARTIAL) {
        if (threadIdx.x == 0) part[bid] = bs;
        return;
    }
    if (threadIdx.x == 0) {
        part[bid] = bs;
        __threadfence();
        const unsigned int ticket = atomicAdd(r.counter + slot, 1u);
        s_last = (ticket == nblocks - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    // Each thread adds its strided partials in index order; the loads are
    // issued eight at a time so that their L2 latencies overlap (the order of
    // the additions, and so the result, is that of the plain loop).
    double acc = 0.0;
    const unsigned int step = blockDim.x;
    unsigned int i = threadIdx.x;
    for (; i + 7 * step < nblocks; i += 8 * step) {
        double v[8];
#pragma unroll
        for (int k = 0; k < 8; k++) v[k] = __ldcg(part + i + k * step);
#pragma unroll
        for (int k = 0; k < 8; k++) acc += v[k];
    }
    for (; i < nblocks; i += step) acc += __ldcg(part + i);
    const double total = block_sum(acc);
    if (threadIdx.x == 0) {
        run_finisher(r, slot, total);
        r.counter[slot] = 0u;
        __threadfence();
    }
}

// The sum of a slot's n partials (FIN_PARTIAL, an earlier kernel), the same in every block
// that forms it (blocks of 256 threads, at most kMaxPartials of them); valid in thread 0.
constexpr int kMaxPartials = 2048;
__device__ inline double sum_partials(const RedArgs& r, int slot, int n) {
    const double* part = r.partials + (size_t)slot * r.slot_cap;
    if (n <= 512) {
        double v[2];
#pragma unroll
        for (int i = 0; i < 2; i++) v[i] = i * 256 + (int)threadIdx.x < n ? __ldcg(part + i * 256 + threadIdx.x) : 0.0;
        return block_sum_of(v);
    }
    double v[kMaxPartials / 256];
#pragma unroll
    for (int i = 0; i < kMaxPartials / 256; i++)
        v[i] = i * 256 + (int)threadIdx.x < n ? __ldcg(part + i * 256 + threadIdx.x) : 0.0;
    return block_sum_of(v);
}

// Single-slot form: every block of the grid contributes.
__device__ inline void grid_reduce(double v, const RedArgs& r) {
    grid_reduce(v, r, 0, gridDim.x * gridDim.y, blockIdx.x + gridDim.x * blockIdx.y);
}

}  // namespace wl
