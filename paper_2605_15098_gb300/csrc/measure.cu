// Read-out kernels: FP64 marginal probabilities, renormalisation, argmax and
// inverse-CDF sampling (the measured bitstring of Sec. IV-A, arxiv 2605.15098).
//
// All sums run in a fixed order, so a call returns the same bits every time:
//   1. partial[g][m] = sum of |amp|^2 over the g-th slice of the amplitudes
//      that map to outcome m, summed in increasing index order; slices of one
//      thread block that share an outcome are added in a fixed tree;
//   2. p[m] = sum over the partials in a fixed tree;
//   3. total = block sums in a fixed tree; p[m] /= total.
// Every read-out is one kernel over the state and at most one over the
// partials (plus the division of a large marginal): each thread block leaves
// its sum and its largest outcome, and the last block to finish combines them
// in block order.
// Sampling builds the inclusive CDF in blocks of 1024 outcomes (in-block
// running sums in index order, block totals accumulated in block order) and
// binary-searches the smallest i with C_i > u * C_last for each shot.
#include <algorithm>
#include <type_traits>

#include "common.h"

namespace sv {
namespace {

constexpr int kRedThreads = 256;
// Resident blocks per SM of the marginal kernels: 64 registers hold eight
// 16-byte loads per thread in flight (128 KiB per SM); a grid that walks the
// outcomes has exactly these blocks.
constexpr int kRedBlocks = 4;

struct MargArgs {
    int n;
    int m;                    // outcome bits
    uint64_t mask;            // physical bits of the outcome
    uint64_t rest;            // physical bits summed over (within n; RB: without bit 0)
    uint64_t upper;           // layout R: rest bits above the 5 lane bits
    int spos[34];             // outcome physical bits, ascending
    int out_bit[34];          // logical output bit of spos[k]
    uint64_t per_group;       // enumerated rest values (RB: pairs of them) per group
    int groups_log2;
    int in_order;             // the output order is the physical one
    uint64_t flush;           // values a thread sums before it adds them to its FP64 sum
};

__device__ __forceinline__ uint64_t pdep_mask(uint64_t v, uint64_t mask) {
    uint64_t r = 0;
    for (uint64_t b = 1; mask; b <<= 1) {
        uint64_t low = mask & (~mask + 1);
        if (v & b) r |= low;
        mask &= mask - 1;
    }
    return r;
}

// Running sum of |amp|^2.  complex128: FP64.  complex64: the squares of the
// FP32 components are formed exactly (product plus fmaf remainder) and added
// with error-free FP32 sums into a (hi, lo) pair, converted to FP64 once per
// thread: the result is the FP64-rounded exact sum to within about 2^-44
// relative, at FP32 instruction cost (GB300 issues FP64 at 1/64 of FP32).
template <typename R>
struct ProbAcc;

// Amplitude loads a reduction thread keeps in flight before accumulating
// them (in order): enough bytes in flight per SM to cover HBM latency.
constexpr int kLoadBatch = 8;

template <>
struct ProbAcc<double> {
    using V = double2;
    // one multiply-add per component (the FP64 pipe bounds this), into sums of
    // half the size each: fewer roundings than adding the squared modulus
    double re = 0.0, im = 0.0;
    __device__ static V load(const double *s, uint64_t x) {
        return reinterpret_cast<const double2 *>(s)[x];
    }
    __device__ void add(V v) {
        re = fma(v.x, v.x, re);
        im = fma(v.y, v.y, im);
    }
    __device__ void add(const double *s, uint64_t x) { add(load(s, x)); }
    __device__ double value() const { return re + im; }
};

template <>
struct ProbAcc<float> {
    float hi = 0.f, lo = 0.f;
    __device__ void two_sum(float b) {
        const float t = hi + b;
        const float bb = t - hi;
        lo += (hi - (t - bb)) + (b - bb);
        hi = t;
    }
    using V = float2;
    __device__ static V load(const float *s, uint64_t x) {
        return reinterpret_cast<const float2 *>(s)[x];
    }
    __device__ void add(V v) {
        const float pr = v.x * v.x, pi = v.y * v.y;
        lo += fmaf(v.x, v.x, -pr) + fmaf(v.y, v.y, -pi);
        two_sum(pr);
        two_sum(pi);
    }
    __device__ void add(const float *s, uint64_t x) { add(load(s, x)); }
    __device__ double value() const { return (double)hi + (double)lo; }
};

// complex64 sums without rounding errors down to FP64's: the remainders' sum
// keeps its own remainders.  Twice the pair's instructions, for a thread that
// sums a whole outcome, where the pair's error (rms 1.8e-15 after 32 amplitudes,
// against 2e-16) would show and FP64 additions in between cost more.
struct ExactAcc {
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
    __device__ static float two_sum(float &s, float b) {
        const float t = s + b, bb = t - s;
        const float e = (s - (t - bb)) + (b - bb);
        s = t;
        return e;
    }
    __device__ void square(float x) {
        const float p = __fmul_rn(x, x);  // not contracted into the sum
        const float e = two_sum(s1, two_sum(s0, p));
        s2 += e + two_sum(s1, fmaf(x, x, -p));
    }
    __device__ void add(float2 v) {
        square(v.x);
        square(v.y);
    }
    __device__ double value() const { return (double)s0 + ((double)s1 + (double)s2); }
};

// A load's amplitudes: two outcomes (PB = 1), or one or two of one outcome.
template <int PB, typename A>
__device__ __forceinline__ void add_vec(A &a, A &b, float4 v) {
    a.add(make_float2(v.x, v.y));
    if (PB) b.add(make_float2(v.z, v.w));
    else a.add(make_float2(v.z, v.w));
}
template <int PB, typename A>
__device__ __forceinline__ void add_vec(A &a, A &, float2 v) { a.add(v); }
template <int PB, typename A>
__device__ __forceinline__ void add_vec(A &a, A &, double2 v) { a.add(v); }

// What a read-out leaves besides the marginal itself.
struct ReadResult {
    double total;   // sum of the marginal
    double recip;   // 1 / total
    double best;    // its maximum divided by the total
    uint64_t idx;   // lowest output index of the maximum
};

// Scratch of a reduction over thread blocks, in the handle's 64 KiB area.
constexpr int kMaxStatBlocks = 2048;
struct Stats {
    double *sum, *best;
    uint64_t *idx;
    ReadResult *res;
    unsigned *done;  // zero between launches
};
constexpr size_t kStatRes = 3 * 8 * kMaxStatBlocks;
static_assert(kStatRes + sizeof(ReadResult) <= kSmallDone, "reduction scratch");

Stats stats_of(sv_state *h) {
    char *b = reinterpret_cast<char *>(h->small);
    Stats s;
    s.sum = reinterpret_cast<double *>(b);
    s.best = s.sum + kMaxStatBlocks;
    s.idx = reinterpret_cast<uint64_t *>(s.best + kMaxStatBlocks);
    s.res = reinterpret_cast<ReadResult *>(b + kStatRes);
    s.done = reinterpret_cast<unsigned *>(b + kSmallDone);
    return s;
}

// The larger value, the lower index among equals.  The values are sums of
// squares or the -1 of "none" (no NaN): their bit patterns compare like
// integers, without the FP64 pipe.
__device__ __forceinline__ void better(double &v, uint64_t &i, double v2, uint64_t i2) {
    const long long a = __double_as_longlong(v), b = __double_as_longlong(v2);
    if (b > a || (b == a && i2 < i)) {
        v = v2;
        i = i2;
    }
}

// Whether an entry (a sum of squares, or a NaN, which never wins) reaches the
// best so far.
__device__ __forceinline__ bool may_beat(double v, double best) {
    const long long b = __double_as_longlong(v);
    // (unsigned: a NaN of either sign is above infinity)
    return b >= __double_as_longlong(best) && (unsigned long long)b <= 0x7ff0000000000000ull;
}

// Output index of the entry at position i of a marginal ordered as p says.
__device__ __forceinline__ uint64_t output_index(uint64_t i, const OutPerm &p) {
    if (!p.m) return i;
    uint64_t r = 0;
    for (int k = 0; k < p.m; k++) r |= ((i >> k) & 1) << p.bit[k];
    return r;
}

// Sum and (with ARG) largest entry of a thread block's outcomes, by a fixed
// tree (lanes, then warps); the results are in thread 0.
template <bool ARG>
__device__ __forceinline__ void block_reduce(double &sum, double &v, uint64_t &i) {
    constexpr int kWarps = kRedThreads / 32;
    __shared__ double s_sum[kWarps], s_v[kWarps];
    __shared__ uint64_t s_i[kWarps];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto lanes = [&](int from) {
        for (int w = from; w; w >>= 1) {
            sum += __shfl_down_sync(0xffffffffu, sum, w);
            if (ARG) {
                const double v2 = __shfl_down_sync(0xffffffffu, v, w);
                const uint64_t i2 = __shfl_down_sync(0xffffffffu, (unsigned long long)i, w);
                better(v, i, v2, i2);
            }
        }
    };
    lanes(16);
    __syncthreads();  // earlier use of the arrays is over
    if (lane == 0) {
        s_sum[warp] = sum;
        s_v[warp] = v;
        s_i[warp] = i;
    }
    __syncthreads();
    if (warp == 0) {
        sum = lane < kWarps ? s_sum[lane] : 0.0;
        v = lane < kWarps ? s_v[lane] : -1.0;
        i = lane < kWarps ? s_i[lane] : ~UINT64_C(0);
        lanes(kWarps / 2);
    }
}

// Leave this block's sum and largest entry; the last block to arrive combines
// all of them in block order into the result.
template <bool ARG>
__device__ __forceinline__ void finish_stats(double sum, double v, uint64_t i, const Stats &st) {
    __shared__ bool s_last;
    block_reduce<ARG>(sum, v, i);
    if (gridDim.x == 1) {
        if (threadIdx.x == 0) *st.res = ReadResult{sum, 1.0 / sum, ARG ? v / sum : 0.0, i};
        return;
    }
    if (threadIdx.x == 0) {
        st.sum[blockIdx.x] = sum;
        if (ARG) {
            st.best[blockIdx.x] = v;
            st.idx[blockIdx.x] = i;
        }
        __threadfence();
        s_last = atomicAdd(st.done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double t = 0.0, bv = -1.0;
    uint64_t bi = ~UINT64_C(0);
    for (unsigned b = threadIdx.x; b < gridDim.x; b += kRedThreads) {
        t += __ldcg(st.sum + b);
        if (ARG) better(bv, bi, __ldcg(st.best + b), __ldcg(reinterpret_cast<const unsigned long long *>(st.idx) + b));
    }
    block_reduce<ARG>(t, bv, bi);
    if (threadIdx.x == 0) {
        *st.res = ReadResult{t, 1.0 / t, ARG ? bv / t : 0.0, bi};
        *st.done = 0;
    }
}

// What a marginal kernel does with its sums: keep them as partials of the
// slices (PART), write the marginal and total it (SUM), or only find its
// total and largest entry (ARG).
enum { MARG_PART = 0, MARG_SUM = 1, MARG_ARG = 2 };

// Layout M: consecutive threads take consecutive physical-order outcomes.
// PB = 1 (complex64 with physical bit 0 an outcome bit): the two outcomes that
// differ in it, whose amplitudes one 16-byte load covers.  RB (complex64 with
// bit 0 summed over): such a load covers two amplitudes of one outcome.  RB = 2:
// where a warp per outcome used to sum, with no larger error: exactly
// (ExactAcc), or in complex128 in shorter chains.
// With fewer outcomes than
// a block has threads, the block's slices of one outcome are added here, so
// that a marginal of a few qubits leaves a thousand partials per outcome
// instead of up to 2^18.  HBM bounds it: 512 MiB in 86 us (0.93 of the
// measured rate); QPE n = 28's argmax, 2 GiB, 376 us against 470 us for the
// marginal, its block sums and its argmax as kernels of their own.
template <typename R, int PB, int RB, int MODE>
__global__ void __launch_bounds__(kRedThreads, kRedBlocks)
k_marg_m(const R *__restrict__ s, MargArgs a, double *__restrict__ partial, const Stats st, const OutPerm perm) {
    constexpr bool kWide = sizeof(R) == 8;
    using V = typename std::conditional<!kWide && (PB || RB), float4, typename ProbAcc<R>::V>::type;
    using Acc = typename std::conditional<!kWide && RB == 2, ExactAcc, ProbAcc<R>>::type;
    constexpr int kShift = !kWide && (PB || RB) ? 1 : 0;
    // complex128 sums that a warp's lanes used to share: even and odd loads
    // apart, so that no addition has more before it than there
    constexpr int kAlt = kWide && RB == 2 ? 1 : 0;
    __shared__ double sh[MODE == MARG_PART ? 2 * kRedThreads : 1];
    const uint64_t outcomes = UINT64_C(1) << a.m;
    const uint64_t per = outcomes >> PB;  // threads per slice
    const uint64_t items = per << a.groups_log2;
    const V *sv_ = reinterpret_cast<const V *>(s);
    double tot = 0.0, best = -1.0;
    uint64_t bidx = ~UINT64_C(0);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    const uint64_t tid0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    // the thread's outcome as physical bits; the outcome `stride` further on
    // is an addition on those bits alone
    uint64_t xm = pdep_mask((tid0 & (per - 1)) << PB, a.mask);
    const uint64_t step = MODE == MARG_PART ? 0 : pdep_mask((stride & (per - 1)) << PB, a.mask);
    for (uint64_t tid = tid0;; tid += stride, xm = ((xm | ~a.mask) + step) & a.mask) {
        const bool in = tid < items;
        if (MODE != MARG_PART && !in) break;
        const uint64_t mp = (tid & (per - 1)) << PB;
        const uint64_t g = tid >> (a.m - PB);
        uint64_t ml = mp;
        if (MODE != MARG_ARG && !a.in_order) {
            ml = 0;
            for (int k = PB; k < a.m; k++) ml |= ((mp >> k) & 1) << a.out_bit[k];
        }
        const uint64_t ml1 = PB ? ml | (UINT64_C(1) << a.out_bit[0]) : ml;
        uint64_t xr = pdep_mask(g * a.per_group, a.rest);
        Acc acc0, acc1;
        double p0 = 0.0, p1 = 0.0;
        auto flush = [&](uint64_t done) {
            if (done & (a.flush - 1)) return;
            if (a.flush == a.per_group) {  // one sum: nothing to add it to
                p0 = kAlt ? acc0.value() + acc1.value() : acc0.value();
                if (PB) p1 = acc1.value();
                return;
            }
            p0 += kAlt ? acc0.value() + acc1.value() : acc0.value();
            acc0 = Acc();
            if (PB) p1 += acc1.value();
            if (PB || kAlt) acc1 = Acc();
        };
        uint64_t i = in ? 0 : a.per_group;
        // kLoadBatch loads in flight per thread, then accumulated in order
        for (; i + kLoadBatch <= a.per_group; i += kLoadBatch) {
            V v[kLoadBatch];
#pragma unroll
            for (int k = 0; k < kLoadBatch; k++) {
                v[k] = sv_[(xm | xr) >> kShift];
                xr = ((xr | ~a.rest) + 1) & a.rest;
            }
            if (a.flush >= kLoadBatch) {
#pragma unroll
                for (int k = 0; k < kLoadBatch; k++) add_vec<PB>(kAlt && (k & 1) ? acc1 : acc0, acc1, v[k]);
                flush(i + kLoadBatch);
            } else {
#pragma unroll
                for (int k = 0; k < kLoadBatch; k++) {
                    add_vec<PB>(acc0, acc1, v[k]);
                    flush(k + 1);
                }
            }
        }
        for (; i < a.per_group; i++) {
            const V v = sv_[(xm | xr) >> kShift];
            add_vec<PB>(acc0, acc1, v);
            flush(i + 1);
            xr = ((xr | ~a.rest) + 1) & a.rest;
        }
        if (MODE == MARG_PART) {
            uint64_t row = g;
            if (per < kRedThreads) {  // add the block's slices of each outcome
                sh[threadIdx.x] = p0;
                if (PB) sh[kRedThreads + threadIdx.x] = p1;
                __syncthreads();
                for (unsigned w = kRedThreads / 2; w >= per; w >>= 1) {
                    if (threadIdx.x < w) {
                        sh[threadIdx.x] += sh[threadIdx.x + w];
                        if (PB) sh[kRedThreads + threadIdx.x] += sh[kRedThreads + threadIdx.x + w];
                    }
                    __syncthreads();
                }
                if (threadIdx.x >= per) return;
                p0 = sh[threadIdx.x];
                p1 = sh[(PB ? kRedThreads : 0) + threadIdx.x];
                row = blockIdx.x;
            } else if (!in) {
                return;
            }
            partial[row * outcomes + ml] = p0;
            if (PB) partial[row * outcomes + ml1] = p1;
            return;  // one item per thread
        }
        if (MODE == MARG_SUM) {
            partial[ml] = p0;
            if (PB) partial[ml1] = p1;
        }
        tot += PB ? p0 + p1 : p0;
        if (MODE == MARG_ARG) {
            if (may_beat(p0, best)) better(best, bidx, p0, output_index(mp, perm));
            if (PB && may_beat(p1, best)) better(best, bidx, p1, output_index(mp | 1, perm));
        }
    }
    if constexpr (MODE != MARG_PART) finish_stats<MODE == MARG_ARG>(tot, best, bidx, st);
}

// Layout R: physical bit 0 is summed over; 2^J lanes per (group, outcome) take
// the J lowest rest bits (RB: above bit 0, which is inside a load).  J = 5 for
// few outcomes: with many, the five FP64 additions over the lanes and the
// start of each sum are most of the work (see marginal).
template <typename R, int J, int RB, int MODE>
__global__ void __launch_bounds__(kRedThreads, kRedBlocks)
k_marg_r(const R *__restrict__ s, MargArgs a, double *__restrict__ partial, const Stats st, const OutPerm perm) {
    using V = typename std::conditional<RB == 1, float4, typename ProbAcc<R>::V>::type;
    const V *sv_ = reinterpret_cast<const V *>(s);
    const uint64_t outcomes = UINT64_C(1) << a.m;
    const int sub = threadIdx.x & ((1 << J) - 1);
    const uint64_t xl = pdep_mask((uint64_t)sub, a.rest & ~a.upper);
    const uint64_t items = outcomes << a.groups_log2;
    double tot = 0.0, best = -1.0;
    uint64_t bidx = ~UINT64_C(0);
    // (items: a multiple of the warp's, so that its lanes leave together)
    for (uint64_t item = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) >> J; item < items;
         item += ((uint64_t)gridDim.x * blockDim.x) >> J) {
        const uint64_t mp = item & (outcomes - 1);
        const uint64_t g = item >> a.m;
        uint64_t xm = 0, ml = 0;
        for (int k = 0; k < a.m; k++) {
            if ((mp >> k) & 1) {
                xm |= UINT64_C(1) << a.spos[k];
                ml |= UINT64_C(1) << a.out_bit[k];
            }
        }
        uint64_t xo = pdep_mask(g * a.per_group, a.upper);
        ProbAcc<R> pa;
        double acc = 0.0;
        auto flush = [&](uint64_t done) {
            if (done & (a.flush - 1)) return;
            acc += pa.value();
            pa = ProbAcc<R>();
        };
        uint64_t i = 0;
        for (; i + kLoadBatch <= a.per_group; i += kLoadBatch) {
            V v[kLoadBatch];
#pragma unroll
            for (int k = 0; k < kLoadBatch; k++) {
                v[k] = sv_[(xm | xo | xl) >> RB];
                xo = ((xo | ~a.upper) + 1) & a.upper;
            }
            if (a.flush >= kLoadBatch) {
#pragma unroll
                for (int k = 0; k < kLoadBatch; k++) add_vec<0>(pa, pa, v[k]);
                flush(i + kLoadBatch);
            } else {
#pragma unroll
                for (int k = 0; k < kLoadBatch; k++) {
                    add_vec<0>(pa, pa, v[k]);
                    flush(k + 1);
                }
            }
        }
        for (; i < a.per_group; i++) {
            add_vec<0>(pa, pa, sv_[(xm | xo | xl) >> RB]);
            flush(i + 1);
            xo = ((xo | ~a.upper) + 1) & a.upper;
        }
#pragma unroll
        for (int off = 1 << (J - 1); off; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
        if (sub == 0) {
            if (MODE != MARG_ARG) partial[g * outcomes + ml] = acc;
            if (MODE != MARG_PART) tot += acc;
            if (MODE == MARG_ARG && may_beat(acc, best)) better(best, bidx, acc, output_index(mp, perm));
        }
    }
    if constexpr (MODE != MARG_PART) finish_stats<MODE == MARG_ARG>(tot, best, bidx, st);
}

// x / t for many x: r = 1 / t correctly rounded, and one correction of
// x * r by its exact remainder gives the correctly rounded quotient (P.
// Markstein, IBM J. Res. Dev. 34, 1990) in three FP64 operations instead of a
// division's dozens; outside the range where the remainder is exact, divide.
__device__ __forceinline__ double divide(double x, double t, double r, bool plain) {
    // (x >= 0: compared as integers, off the FP64 pipe)
    if (plain || __double_as_longlong(x) < __double_as_longlong(1e-280)) return x / t;
    const double q = x * r;
    return fma(fma(-q, t, x), r, q);
}
__device__ __forceinline__ bool divide_plain(double t) { return !(t > 1e-200 && t < 1e200); }

// The sum of rows first, first + step, ... of outcome m, eight at a time (an
// FP64 addition takes about 90 cycles).
__device__ __forceinline__ double sum_rows(const double *__restrict__ partial, uint64_t outcomes, uint64_t m,
                                           int first, int rows, int step) {
    double part[8] = {};
    int g = first;
    for (; g + 7 * step < rows; g += 8 * step) {
        double v[8];
#pragma unroll
        for (int k = 0; k < 8; k++) v[k] = partial[(uint64_t)(g + k * step) * outcomes + m];
#pragma unroll
        for (int k = 0; k < 8; k++) part[k] += v[k];
    }
    for (; g < rows; g += step) part[0] += partial[(uint64_t)g * outcomes + m];
    return ((part[0] + part[1]) + (part[2] + part[3])) + ((part[4] + part[5]) + (part[6] + part[7]));
}

// Thread t of a block holds outcome t % to and one of the block's 256 / to
// shares of the rows; the shares are added in a fixed tree, the sum of outcome
// o in thread o.
__device__ __forceinline__ double block_rows(const double *__restrict__ partial, uint64_t outcomes, uint64_t m0,
                                             int first, int rows, int step, int to) {
    __shared__ double sh[kRedThreads];
    const int o = threadIdx.x % to, sl = threadIdx.x / to, ns = kRedThreads / to;
    sh[threadIdx.x] = sum_rows(partial, outcomes, m0 + o, first + sl * step, rows, ns * step);
    __syncthreads();
    for (int w = kRedThreads / 2; w >= to; w >>= 1) {
        if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    return sh[threadIdx.x];
}

// kFoldRows rows from many: row y of the result adds rows y, y + kFoldRows, ...
// (three qubits of n = 26, 1024 rows: 4 us and 5 us for the last sums; one
// thread per outcome took 267 us for its 2048 rows).
constexpr int kFoldRows = 32;
__global__ void __launch_bounds__(kRedThreads)
k_fold_rows(const double *__restrict__ partial, uint64_t outcomes, int rows, int to, double *__restrict__ out) {
    const uint64_t m0 = (uint64_t)blockIdx.x * to;
    const double acc = block_rows(partial, outcomes, m0, blockIdx.y, rows, gridDim.y, to);
    if ((int)threadIdx.x < to) out[blockIdx.y * outcomes + m0 + threadIdx.x] = acc;
}

// p[m] = the sum of its partials; then as MODE says.  With `norm` and one
// block the marginal is divided by its total here.
template <int MODE>
__global__ void __launch_bounds__(kRedThreads)
k_sum_groups(const double *__restrict__ partial, uint64_t outcomes, int rows, int to, double *__restrict__ out,
             const Stats st, const OutPerm perm, bool norm) {
    const uint64_t m0 = (uint64_t)blockIdx.x * to, m = m0 + threadIdx.x;
    const bool mine = (int)threadIdx.x < to;
    double acc = block_rows(partial, outcomes, m0, 0, rows, 1, to);
    if (!mine) acc = 0.0;
    if (mine && MODE == MARG_SUM && !(norm && gridDim.x == 1)) out[m] = acc;
    const bool cand = mine && may_beat(acc, -1.0);
    finish_stats<MODE == MARG_ARG>(acc, cand ? acc : -1.0, cand ? output_index(m, perm) : ~UINT64_C(0), st);
    if (MODE == MARG_SUM && norm && gridDim.x == 1) {
        __syncthreads();
        if (mine) out[m] = divide(acc, st.res->total, st.res->recip, divide_plain(st.res->total));
    }
}

__global__ void __launch_bounds__(kRedThreads)
k_normalise(double *__restrict__ p, uint64_t len, const ReadResult *__restrict__ res) {
    const double t = res->total, r = res->recip;
    const bool plain = divide_plain(t);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    double2 *p2 = reinterpret_cast<double2 *>(p);
    const bool pairs = (reinterpret_cast<uintptr_t>(p) & 15) == 0;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < len / 2; i += stride) {
        double2 v = pairs ? p2[i] : make_double2(p[2 * i], p[2 * i + 1]);
        v.x = divide(v.x, t, r, plain);
        v.y = divide(v.y, t, r, plain);
        if (pairs) p2[i] = v;
        else {
            p[2 * i] = v.x;
            p[2 * i + 1] = v.y;
        }
    }
}

// Running FP64 sums of non-negative values in order, 32 at a time: lane k adds
// x to the sum of everything before it, every addition rounded to nearest as
// one addition after the other rounds it.  While the sum stays in one binade
// a value adds a whole number of the sum's last places, whatever the sum is,
// so the 32 steps are a prefix sum of integers on the sum's bit pattern.  The
// exceptions take an FP64 addition of their own, and the lanes after it start
// again from its result: a tie (its direction depends on the sum), a value
// above the sum's binade, a step out of the binade, a sum that is not a
// normal number.  Zeros change nothing and are never exceptions.
//
// An exception costs a prefix sum, about four additions' time.  Sums of similar
// values have about two per doubling of the sum, ten in their first 32 values,
// but all 32 of a step can be exceptions: a kernel that meets more than
// kRunMost of them in a step adds the rest of its values one after the other.
// 2^20 outcomes, k_cdf_blocks on Gaussian amplitudes 18.7 us without this and
// 19.0 with it, on sums of 16 of them 18.5 and 18.8; the call of sv_sample
// where every value is a tie 497 and 249, where the values grow by 2^2000 in
// all 521 and 255.  (Counted in here, step by step: 19.0 and 19.0, 18.4 of 17.7
// for 2^16 outcomes and 24.4 of 21.9 for 2^21, calls 234 and 248.)
//
// total: the sum so far, the same in every lane, on return the sum with all
// 32 values; returns the sum up to and including the lane's own value.
// rounds: the prefix sums it took.
constexpr int kRunMost = 16;
__device__ __forceinline__ double warp_run(double &total, double x, int lane, int &rounds) {
    uint64_t c = (uint64_t)__double_as_longlong(total), mine = c;
    const uint64_t xb = (uint64_t)__double_as_longlong(x);
    const int ex = (int)(xb >> 52);
    const uint64_t m = (xb & ((UINT64_C(1) << 52) - 1)) | (ex ? UINT64_C(1) << 52 : 0);
    rounds = 0;
    for (int pos = 0; pos < 32; rounds++) {
        const int e = (int)(c >> 52);
        const int de = e - (ex ? ex : 1);
        bool bad = false;
        uint64_t s = 0;
        if (lane >= pos && xb) {
            const int d = de < 0 ? 0 : de > 63 ? 63 : de;
            const uint64_t q = m >> d, rest = (m - (q << d)) << 1, one = UINT64_C(1) << d;
            bad = e < 1 || e > 0x7fe || de < 0 || rest == one;
            s = bad ? 0 : q + (rest > one);
        }
#pragma unroll
        for (int w = 1; w < 32; w <<= 1) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, s, w);
            if (lane >= w) s += y;
        }
        const uint64_t after = c + s;
        bad = bad || (lane >= pos && (int)(after >> 52) != e);
        const unsigned stop = __ballot_sync(0xffffffffu, bad);
        const int first = stop ? __ffs((int)stop) - 1 : 32;
        if (lane >= pos && lane < first) mine = after;
        // lanes below pos add nothing, so lane first - 1 has the sum before
        // the exception (c itself when that is the first lane of this round)
        const uint64_t last = __shfl_sync(0xffffffffu, after, first ? first - 1 : 0);
        c = first > pos ? last : c;
        if (first < 32) {
            const double xf = __shfl_sync(0xffffffffu, x, first);
            c = (uint64_t)__double_as_longlong(__dadd_rn(__longlong_as_double((long long)c), xf));
            if (lane == first) mine = c;
        }
        pos = first + 1;
    }
    total = __longlong_as_double((long long)c);
    return __longlong_as_double((long long)mine);
}

// CDF, step 1: running sums of blocks of 1024 outcomes in index order.  One
// warp takes a block, 32 consecutive outcomes at a time (warp_run), and keeps
// the running sum at every 32nd outcome (chk) and at the end (btot).  The
// latency of the shuffles bounds it, about 45 prefix sums per block: 18 us for
// 2^20 outcomes.  With one FP64 addition after the other (about 90 cycles
// each) a lane per block took 70 us.
constexpr int kCdfBlock = 1024, kCdfStep = 32, kCdfAhead = 4;
__global__ void __launch_bounds__(kRedThreads)
k_cdf_blocks(const double *__restrict__ p, uint64_t len, double *__restrict__ chk, double *__restrict__ btot) {
    constexpr int steps = kCdfBlock / kCdfStep;
    const int lane = threadIdx.x & 31;
    const uint64_t b = (uint64_t)blockIdx.x * (kRedThreads / 32) + (threadIdx.x >> 5);
    if (b * kCdfBlock >= len) return;  // the whole warp
    auto value = [&](int c) {
        const uint64_t i = b * kCdfBlock + c * kCdfStep + lane;
        return c < steps && i < len ? p[i] : 0.0;  // outcomes beyond len add nothing
    };
    double run = 0.0, nxt[kCdfAhead];
#pragma unroll
    for (int k = 0; k < kCdfAhead; k++) nxt[k] = value(k);
    int c = 0;
    for (bool go = true; go && c < steps; c += kCdfAhead) {
#pragma unroll
        for (int k = 0; k < kCdfAhead; k++) {
            const double x = nxt[k];
            nxt[k] = value(c + kCdfAhead + k);
            if (lane == 0) chk[b * steps + c + k] = run;
            int rounds;
            warp_run(run, x, lane, rounds);
            go = go && rounds <= kRunMost;
        }
    }
    for (; c < steps; c++) {
        const double x = value(c);
        if (lane == 0) chk[b * steps + c] = run;
#pragma unroll 8
        for (int k = 0; k < 32; k++) run = __dadd_rn(run, __shfl_sync(0xffffffffu, x, k));
    }
    if (lane == 0) btot[b] = run;
}

// CDF, step 2: before[b] = running total of the blocks before b, in block
// order; before[nb] = C_last: one warp, 32 blocks at a time: 15 us for 1024
// blocks, against 48 us with one addition after the other.
__global__ void __launch_bounds__(32)
k_cdf_scan(const double *__restrict__ btot, uint64_t nb, double *__restrict__ before) {
    const int lane = threadIdx.x;
    auto value = [&](uint64_t i) { return i + lane < nb ? btot[i + lane] : 0.0; };
    double run = 0.0, nxt[kCdfAhead];
    if (lane == 0) before[0] = 0.0;
#pragma unroll
    for (int k = 0; k < kCdfAhead; k++) nxt[k] = value(32 * k);
    uint64_t c = 0;
    for (bool go = true; go && c < nb; c += 32 * kCdfAhead) {
#pragma unroll
        for (int k = 0; k < kCdfAhead; k++) {
            const uint64_t i = c + 32 * k;
            const double x = nxt[k];
            nxt[k] = value(i + 32 * kCdfAhead);
            int rounds;
            const double after = warp_run(run, x, lane, rounds);
            if (i + lane < nb) before[i + lane + 1] = after;
            go = go && rounds <= kRunMost;
        }
    }
    for (; c < nb; c += 32) {
        const double x = value(c);
        double after = 0.0;
#pragma unroll 8
        for (int k = 0; k < 32; k++) {
            run = __dadd_rn(run, __shfl_sync(0xffffffffu, x, k));
            if (lane == k) after = run;
        }
        if (c + lane < nb) before[c + lane + 1] = after;
    }
}

// CDF, step 3: the smallest i with C_i > u * C_last, where C_i = (total before
// the block) + (running sum in the block): the block by its end, the step of
// 32 in it by the kept sums, then the outcomes of the step in order.  The CDF
// does not decrease, so this is what a search over all of it gives.
__global__ void k_sample(const double *__restrict__ p, uint64_t len, const double *__restrict__ before,
                         const double *__restrict__ chk, const double *__restrict__ u, uint64_t shots,
                         uint64_t *__restrict__ out) {
    const uint64_t s = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= shots) return;
    const uint64_t nb = (len + kCdfBlock - 1) / kCdfBlock;
    const double target = u[s] * before[nb];
    uint64_t lo = 0, hi = nb - 1;
    while (lo < hi) {
        const uint64_t mid = lo + (hi - lo) / 2;
        if (before[mid + 1] > target) hi = mid;
        else lo = mid + 1;
    }
    const double bb = before[lo];
    const double *ck = chk + lo * (kCdfBlock / kCdfStep);
    // the first step whose end exceeds the target (the last one if none of the
    // kept sums does)
    const uint64_t left = len - lo * kCdfBlock;
    const int steps = left >= (uint64_t)kCdfBlock ? kCdfBlock / kCdfStep : (int)((left + kCdfStep - 1) / kCdfStep);
    int a = 0, z = steps - 1;
    while (a < z) {
        const int mid = (a + z) / 2;
        if (bb + ck[mid + 1] > target) z = mid;
        else a = mid + 1;
    }
    const uint64_t i0 = lo * kCdfBlock + (uint64_t)a * kCdfStep;
    double run = ck[a];
    uint64_t i = i0;
    const uint64_t i1 = i0 + kCdfStep < len ? i0 + kCdfStep : len;
    for (; i < i1; i++) {
        run += p[i];
        if (bb + run > target) break;
    }
    out[s] = i < len ? i : len - 1;
}

unsigned blocks_for(uint64_t work, int threads) {
    uint64_t b = (work + threads - 1) / threads;
    return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(b, 0x7fffffffULL));
}

}  // namespace

sv_status ensure_scratch(sv_state *h, size_t bytes) {
    if (bytes <= h->scratch_cap) return SV_OK;
    if (h->scratch) {
        SV_CUDA(cudaStreamSynchronize(h->stream));
        cudaFree(h->scratch);
        h->scratch = nullptr;
        h->scratch_cap = 0;
    }
    size_t cap = std::max<size_t>(bytes, (size_t)1 << 20);
    if (dev_malloc(&h->scratch, cap) != cudaSuccess) {
        cudaGetLastError();
        h->scratch = nullptr;
        return fail(SV_ERR_OOM, "cannot allocate %zu bytes of device scratch", cap);
    }
    h->scratch_cap = cap;
    return SV_OK;
}

sv_status ensure_probs(sv_state *h, size_t bytes) {
    if (bytes <= h->probs_cap) return SV_OK;
    if (h->probs) {
        SV_CUDA(cudaStreamSynchronize(h->stream));
        cudaFree(h->probs);
        h->probs = nullptr;
        h->probs_cap = 0;
    }
    size_t cap = std::max<size_t>(bytes, (size_t)1 << 16);
    if (dev_malloc(&h->probs, cap) != cudaSuccess) {
        cudaGetLastError();
        h->probs = nullptr;
        return fail(SV_ERR_OOM, "cannot allocate %zu bytes for probabilities", cap);
    }
    h->probs_cap = cap;
    return SV_OK;
}

namespace {

template <int MODE>
void launch_marginal(sv_state *h, const MargArgs &a, int lanes_log2, bool pairs, bool rest_pairs, bool exact, unsigned grid,
                     double *partial, const Stats &st, const OutPerm &perm) {
    if (h->dt == SV_C128) {
        const double *s = reinterpret_cast<const double *>(h->amps);
        if (lanes_log2)
            k_marg_r<double, 5, 0, MODE><<<grid, kRedThreads, 0, h->stream>>>(s, a, partial, st, perm);
        else if (exact)
            k_marg_m<double, 0, 2, MODE><<<grid, kRedThreads, 0, h->stream>>>(s, a, partial, st, perm);
        else
            k_marg_m<double, 0, 0, MODE><<<grid, kRedThreads, 0, h->stream>>>(s, a, partial, st, perm);
    } else {
        const float *s = reinterpret_cast<const float *>(h->amps);
        if (lanes_log2 == 5)
            k_marg_r<float, 5, 0, MODE><<<grid, kRedThreads, 0, h->stream>>>(s, a, partial, st, perm);
        else if (lanes_log2)
            k_marg_r<float, 1, 1, MODE><<<grid, kRedThreads, 0, h->stream>>>(s, a, partial, st, perm);
        else if (pairs)
            k_marg_m<float, 1, 0, MODE><<<grid, kRedThreads, 0, h->stream>>>(s, a, partial, st, perm);
        else if (exact)
            k_marg_m<float, 0, 2, MODE><<<grid, kRedThreads, 0, h->stream>>>(s, a, partial, st, perm);
        else if (rest_pairs)
            k_marg_m<float, 0, 1, MODE><<<grid, kRedThreads, 0, h->stream>>>(s, a, partial, st, perm);
        else
            k_marg_m<float, 0, 0, MODE><<<grid, kRedThreads, 0, h->stream>>>(s, a, partial, st, perm);
    }
}

// Whether the handle has this much scratch, or can get it now: not while the
// stream is being captured, where an allocation would end the capture.
bool scratch_at_hand(sv_state *h, size_t bytes) {
    if (bytes <= h->scratch_cap) return true;
    cudaStreamCaptureStatus cs;
    if (cudaStreamIsCapturing(h->stream, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone) {
        cudaGetLastError();
        return false;
    }
    if (ensure_scratch(h, bytes) == SV_OK) return true;
    clear_error();
    return false;
}

// pos[j]: physical bit of output bit j.  MODE MARG_SUM: the marginal and its
// total, in dev_out; MARG_ARG: its total and largest entry only (dev_out may
// be NULL).  *divided: the marginal was divided by its total already.
// no_scratch: a marginal of 2^15 outcomes or more without partial sums.
template <int MODE>
sv_status marginal(sv_state *h, const int *pos, int m, double *dev_out, bool norm, bool *divided,
                   bool no_scratch = false) {
    SV_TRY(materialize(h));
    const int n = h->n;
    MargArgs a{};
    a.n = n;
    a.m = m;
    OutPerm perm{};
    // outcome bits sorted by physical position
    int order[34];
    for (int j = 0; j < m; j++) order[j] = j;
    std::sort(order, order + m, [&](int x, int y) { return pos[x] < pos[y]; });
    for (int k = 0; k < m; k++) {
        a.spos[k] = pos[order[k]];
        // the argmax keeps partials in physical order (coalesced whatever the
        // qubit map) and maps only its candidates
        a.out_bit[k] = MODE == MARG_ARG ? k : order[k];
        a.mask |= UINT64_C(1) << pos[order[k]];
    }
    a.in_order = 1;
    for (int k = 0; k < m; k++) a.in_order &= a.out_bit[k] == k;
    if (MODE == MARG_ARG) {
        perm.m = m;
        for (int k = 0; k < m; k++) perm.bit[k] = (int8_t)order[k];
    }
    const uint64_t all = (n == 64) ? ~UINT64_C(0) : ((UINT64_C(1) << n) - 1);
    a.rest = all & ~a.mask;
    const int rbits = n - m;
    const uint64_t outcomes = UINT64_C(1) << m;
    const bool bit0 = (a.mask & 1) != 0;
    // Where physical bit 0 is summed over, a warp per outcome below 2^15 of them
    // (layout R).  Above, the five FP64 additions over its lanes and the start
    // of each sum are most of the work: one thread per outcome (layout M), in
    // complex64 with exact sums (ExactAcc), or, where a lane of that warp would
    // hold 16 amplitudes or more, FP32 pairs of as many, and two lanes with 32
    // contiguous bytes if bit 1 is summed over too.  n = 26, complex64, the 2^m
    // outcomes of the highest qubits, a warp against this: m = 14 104 against
    // 107 us, m = 15 121 and 110, m = 17 197 and 105, m = 18 281 and 144, m = 20
    // 985 and 140; n = 22: m = 14 27 and 33, m = 15 60 and 25, m = 17 110 and 23.
    // complex128, where the sums themselves fill the FP64 pipe, keeps the warp
    // for 2^10 amplitudes or more per outcome, 2^9 from 2^18 outcomes up (a warp
    // against a thread: n = 25, m = 15 168 and 173, m = 16 179 and 175; n = 26,
    // m = 15 298 and 324, m = 16 308 and 326, m = 17 338 and 328; n = 27, m = 17
    // 593 and 627, m = 18 659 and 712), unless its lanes lie far apart: where
    // only two bits summed over are below bit 18 the warp takes 1.2 to 2.6 times
    // as long (n = 26, m = 16, the qubits from 1 up 629 and 324, from 2 up 414 and
    // 323; m = 15, with the third bit at 17, 301 and 324).
    uint64_t third = a.rest & (a.rest - 1);
    third &= third - 1;  // the bits summed over without the two lowest
    const bool far = !(third & ((UINT64_C(1) << 18) - 1));
    const bool many_rest =
        !no_scratch && !bit0 && rbits >= 5 && m >= 15 && (h->dt == SV_C64 || far || rbits < (m >= 18 ? 9 : 10));
    const bool exact = many_rest && (h->dt == SV_C128 || rbits < 9);
    const int lanes_log2 = bit0 || rbits < 5 ? 0 : !many_rest ? 5 : exact || (a.mask & 2) ? 0 : 1;
    const bool layout_r = lanes_log2 > 0;
    // complex64 with bit 0 summed over: two amplitudes per load where two share
    // an FP32 sum (a.flush below)
    const bool rest_pairs = lanes_log2 < 5 && !bit0 && h->dt == SV_C64 && n >= 20;
    if (rest_pairs) a.rest &= ~UINT64_C(1);
    const int bits = rbits - rest_pairs;
    // complex64 with physical bit 0 an outcome bit: two outcomes per thread
    const bool pairs = bit0 && h->dt == SV_C64;
    // slices per outcome: enough threads (layout M) or lanes (layout R) for the
    // device, but at least 16 (8) loads per thread, so that a marginal with
    // many outcomes, or a small state's, is one launch
    const int target_log2 = 18;
    int gl;
    if (layout_r) {
        uint64_t up = a.rest;
        for (int i = 0; i < lanes_log2; i++) up &= up - 1;  // drop the lanes' rest bits
        a.upper = up;
        int ubits = bits - lanes_log2;
        gl = std::max(0, std::min(ubits - 3, target_log2 - lanes_log2 - m));
        a.per_group = UINT64_C(1) << (ubits - gl);
    } else {
        gl = std::max(0, std::min(bits - 4, target_log2 - rest_pairs - m));
        a.per_group = UINT64_C(1) << (bits - gl);
    }
    a.groups_log2 = gl;
    // FP32 pairs carry about 2^-48 of their sum's size per addition: short
    // sums, added up in FP64, keep the marginal's error below 1e-15 on small
    // and mid-sized states, where the conversions cost nothing (2^19 of them
    // or one per amplitude, whichever is less)
    int short_log2 = std::max(0, rbits - lanes_log2 - std::max(0, 19 - lanes_log2 - m));
    if (many_rest) short_log2 = !exact ? rbits - 5 : rest_pairs ? rbits : 4;
    a.flush = std::min(a.per_group, UINT64_C(1) << (short_log2 - rest_pairs));
    const int pb = pairs ? 1 : 0;
    const Stats st = stats_of(h);
    const unsigned most = (unsigned)std::min(kMaxStatBlocks, h->sm_count * kRedBlocks);
    const uint64_t threads = layout_r ? (outcomes << gl) << lanes_log2 : (outcomes >> pb) << gl;
    const unsigned blocks = blocks_for(threads, kRedThreads);
    const bool fold = !layout_r && (outcomes >> pb) < kRedThreads;  // the block adds its slices
    *divided = false;
    if (gl == 0) {  // every thread (warp) holds whole outcomes
        // layout R's items are few and large: a block for each of them where
        // that is at most two waves of blocks (n = 26, m = 13: 105 against 116
        // us), with two lanes per outcome at all sizes
        const unsigned cap = lanes_log2 == 5 ? 2 * most : lanes_log2 ? (unsigned)kMaxStatBlocks : most;
        const unsigned grid = blocks <= cap ? blocks : most;
        launch_marginal<MODE>(h, a, lanes_log2, pairs, rest_pairs, exact, grid, dev_out, st, perm);
        SV_CUDA(cudaGetLastError());
        note_launch();
        return SV_OK;
    }
    uint64_t rows = fold ? blocks : UINT64_C(1) << gl;
    // many partials of few outcomes: one block would read them all (8
    // outcomes, 2048 rows: 18 us), so more blocks add most of them
    const bool fold_rows = rows > 4 * kFoldRows && outcomes * kFoldRows <= 8192;
    const size_t bytes = (rows + (fold_rows ? kFoldRows : 0)) * outcomes * sizeof(double);
    // (up to 2 MiB for 2^15 to 2^17 outcomes; the warp per outcome needs none)
    if (many_rest && !scratch_at_hand(h, bytes)) return marginal<MODE>(h, pos, m, dev_out, norm, divided, true);
    SV_TRY(ensure_scratch(h, bytes));
    double *partial = reinterpret_cast<double *>(h->scratch);
    launch_marginal<MARG_PART>(h, a, lanes_log2, pairs, rest_pairs, exact, blocks, partial, st, perm);
    SV_CUDA(cudaGetLastError());
    note_launch();
    if (fold_rows) {
        double *folded = partial + rows * outcomes;
        const int to = (int)std::min<uint64_t>(outcomes, 32);
        k_fold_rows<<<dim3((unsigned)(outcomes / to), kFoldRows), kRedThreads, 0, h->stream>>>(
            partial, outcomes, (int)rows, to, folded);
        SV_CUDA(cudaGetLastError());
        note_launch();
        partial = folded;
        rows = kFoldRows;
    }
    // outcomes per block: all its threads while that fills the device
    const int to = (int)std::min<uint64_t>(outcomes, rows <= 16 || outcomes > 32768 ? 256 : 32);
    const unsigned grid = (unsigned)(outcomes / to);
    k_sum_groups<MODE><<<grid, kRedThreads, 0, h->stream>>>(partial, outcomes, (int)rows, to, dev_out, st, perm, norm);
    SV_CUDA(cudaGetLastError());
    note_launch();
    *divided = norm && grid == 1;
    return SV_OK;
}

}  // namespace

sv_status marginal_device(sv_state *h, const int *pos, int m, double *dev_out) {
    bool divided;
    SV_TRY(marginal<MARG_SUM>(h, pos, m, dev_out, true, &divided));
    if (divided) return SV_OK;
    const uint64_t outcomes = UINT64_C(1) << m;
    const unsigned grid = std::min<unsigned>(blocks_for((outcomes + 1) / 2, kRedThreads), (unsigned)h->sm_count * 8);
    k_normalise<<<grid, kRedThreads, 0, h->stream>>>(dev_out, outcomes, stats_of(h).res);
    SV_CUDA(cudaGetLastError());
    note_launch();
    return SV_OK;
}

sv_status argmax_device(sv_state *h, const int *pos, int m, uint64_t *host_idx, double *host_p) {
    bool divided;
    SV_TRY(marginal<MARG_ARG>(h, pos, m, nullptr, false, &divided));
    ReadResult r;
    SV_CUDA(cudaMemcpyAsync(&r, stats_of(h).res, sizeof r, cudaMemcpyDeviceToHost, h->stream));
    SV_TRY(finish_sync(h));
    *host_idx = r.idx;
    if (host_p) *host_p = r.best;
    return SV_OK;
}

sv_status sample_device(sv_state *h, const double *dev_p, uint64_t len, const double *host_u,
                        size_t shots, uint64_t *host_out) {
    if (!shots) return finish_sync(h);
    const uint64_t nb = (len + kCdfBlock - 1) / kCdfBlock;
    const size_t off_bt = nb * (kCdfBlock / kCdfStep) * sizeof(double);
    const size_t off_be = off_bt + nb * sizeof(double);
    const size_t off_u = off_be + (nb + 1) * sizeof(double);
    const size_t off_o = off_u + shots * sizeof(double);
    SV_TRY(ensure_scratch(h, off_o + shots * sizeof(uint64_t)));
    char *base = reinterpret_cast<char *>(h->scratch);
    double *chk = reinterpret_cast<double *>(base);
    double *bt = reinterpret_cast<double *>(base + off_bt);
    double *before = reinterpret_cast<double *>(base + off_be);
    double *du = reinterpret_cast<double *>(base + off_u);
    uint64_t *dout = reinterpret_cast<uint64_t *>(base + off_o);
    k_cdf_blocks<<<blocks_for(nb, kRedThreads / 32), kRedThreads, 0, h->stream>>>(dev_p, len, chk, bt);
    SV_CUDA(cudaGetLastError());
    k_cdf_scan<<<1, 32, 0, h->stream>>>(bt, nb, before);
    SV_CUDA(cudaGetLastError());
    SV_CUDA(cudaMemcpyAsync(du, host_u, shots * sizeof(double), cudaMemcpyHostToDevice, h->stream));
    k_sample<<<blocks_for(shots, 64), 64, 0, h->stream>>>(dev_p, len, before, chk, du, shots, dout);
    SV_CUDA(cudaGetLastError());
    note_launch(3);
    SV_CUDA(cudaMemcpyAsync(host_out, dout, shots * sizeof(uint64_t), cudaMemcpyDeviceToHost, h->stream));
    return finish_sync(h);
}

}  // namespace sv
