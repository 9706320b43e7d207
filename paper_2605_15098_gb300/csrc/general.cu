// General gate set on the per-gate path: multi-controlled U (MCU), two-qubit
// unitaries (U2Q with its three row records) and projective measurement
// with collapse (MEASURE).  Gates arrive with PHYSICAL qubit positions.
//
// MCU is Algorithm 1 (Sec. III-A) with the control rule taken to a set of
// controls: the pair (x, x + 2^t) is updated only when every control bit of
// x is 1, so the kernel enumerates exactly those pairs (2^(n-1-k) of them).
// U2Q updates the four amplitudes that agree off its two qubits.  MEASURE
// sums |amp|^2 over each value of its qubit to FP64 accuracy (partials in a
// fixed tree, then the blocks in a fixed tree), picks the outcome on the
// device as the smallest i with C_i > u C_last for C = (p0, p0 + p1), and
// collapses the state: the other half is zeroed and the kept one divided by
// sqrt(p_i).  No host synchronisation: the outcome goes to a device array
// that sv_last_measurements reads.
//
// All of them are HBM (up to n = 23: L2) sweeps: threads keep several 16-byte
// vectors in flight, of two amplitudes in complex64 when no qubit of the gate
// is bit 0.  A dynamic circuit of n = 23 with 6 MCU, 6 U2Q and 2 measurements:
// 1074 us with one 8-byte amplitude at a time in MCU and U2Q, 1045 so.
#include <algorithm>
#include <cmath>

#include "common.h"

namespace sv {
namespace {

constexpr int kThreads = 256;
constexpr int kMeasBlocks = 1216;  // partial sums of a measurement (2 doubles each)

// Positions (ascending) where the enumeration inserts a bit.
struct Ins {
    int n;
    int8_t pos[40];
};

__device__ __forceinline__ uint64_t insert_zeros(uint64_t u, const Ins &in) {
    for (int i = 0; i < in.n; i++) {
        const int p = in.pos[i];
        u = ((u >> p) << (p + 1)) | (u & ((UINT64_C(1) << p) - 1));
    }
    return u;
}

template <typename R>
struct C2 {
    R re[4], im[4];
};
template <typename R>
struct C4 {
    R re[16], im[16];
};

// A vector of the state: VB = 1 two complex64 amplitudes, VB = 0 one
// amplitude.
template <typename R, int VB>
struct Vec;
template <>
struct Vec<float, 1> {
    using T = float4;
};
template <>
struct Vec<float, 0> {
    using T = float2;
};
template <>
struct Vec<double, 0> {
    using T = double2;
};

constexpr int kItems = 4;  // vectors (pairs, quadruples: half as many) a thread keeps in flight

template <typename R, int VB>
__global__ void __launch_bounds__(kThreads)
k_mcu(R *__restrict__ s, uint64_t units, Ins in, uint64_t ones, uint64_t tbit, C2<R> c) {
    using T = typename Vec<R, VB>::T;
    T *v = reinterpret_cast<T *>(s);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t u0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; u0 < units; u0 += stride * kItems) {
        T a[kItems], b[kItems];
        uint64_t x[kItems];
#pragma unroll
        for (int k = 0; k < kItems; k++) {
            const uint64_t u = u0 + k * stride;
            if (u >= units) break;
            x[k] = insert_zeros(u, in) | ones;
            a[k] = v[x[k]];
            b[k] = v[x[k] | tbit];
        }
#pragma unroll
        for (int k = 0; k < kItems; k++) {
            if (u0 + k * stride >= units) break;
            R *pa = reinterpret_cast<R *>(&a[k]), *pb = reinterpret_cast<R *>(&b[k]);
#pragma unroll
            for (int e = 0; e < (1 << VB); e++) {
                const R ar = pa[2 * e], ai = pa[2 * e + 1], br = pb[2 * e], bi = pb[2 * e + 1];
                pa[2 * e] = c.re[0] * ar - c.im[0] * ai + c.re[1] * br - c.im[1] * bi;
                pa[2 * e + 1] = c.re[0] * ai + c.im[0] * ar + c.re[1] * bi + c.im[1] * br;
                pb[2 * e] = c.re[2] * ar - c.im[2] * ai + c.re[3] * br - c.im[3] * bi;
                pb[2 * e + 1] = c.re[2] * ai + c.im[2] * ar + c.re[3] * bi + c.im[3] * br;
            }
            v[x[k]] = a[k];
            v[x[k] | tbit] = b[k];
        }
    }
}

template <typename R, int VB>
__global__ void __launch_bounds__(kThreads)
k_u2q(R *__restrict__ s, uint64_t units, Ins in, uint64_t ma, uint64_t mb, C4<R> m) {
    using T = typename Vec<R, VB>::T;
    constexpr int NI = kItems / 2;
    T *v = reinterpret_cast<T *>(s);
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t u0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; u0 < units; u0 += stride * NI) {
        T q[NI][4];
        uint64_t x[NI];
#pragma unroll
        for (int i = 0; i < NI; i++) {
            const uint64_t u = u0 + i * stride;
            if (u >= units) break;
            x[i] = insert_zeros(u, in);
            q[i][0] = v[x[i]];
            q[i][1] = v[x[i] | ma];
            q[i][2] = v[x[i] | mb];
            q[i][3] = v[x[i] | ma | mb];
        }
#pragma unroll
        for (int i = 0; i < NI; i++) {
            if (u0 + i * stride >= units) break;
            T y[4];
#pragma unroll
            for (int e = 0; e < (1 << VB); e++)
#pragma unroll
                for (int r = 0; r < 4; r++) {
                    R yr = 0, yi = 0;
#pragma unroll
                    for (int k = 0; k < 4; k++) {
                        const R vr = reinterpret_cast<const R *>(&q[i][k])[2 * e];
                        const R vi = reinterpret_cast<const R *>(&q[i][k])[2 * e + 1];
                        yr += m.re[4 * r + k] * vr - m.im[4 * r + k] * vi;
                        yi += m.re[4 * r + k] * vi + m.im[4 * r + k] * vr;
                    }
                    reinterpret_cast<R *>(&y[r])[2 * e] = yr;
                    reinterpret_cast<R *>(&y[r])[2 * e + 1] = yi;
                }
            v[x[i]] = y[0];
            v[x[i] | ma] = y[1];
            v[x[i] | mb] = y[2];
            v[x[i] | ma | mb] = y[3];
        }
    }
}

// Sum of squares of one value of the measured qubit.  complex128: FP64.
// complex64: summed in FP32 without error (exact squares as product and fmaf
// remainder; sums and their remainders as an unevaluated sum of three), which
// is good to the FP64 it becomes; FP64 issues at 1/64 of the FP32 rate, so
// that its conversions and additions are made once per thread.  Where the sum
// lies outside [2^-90, 2^120] this does not hold: a square's remainder goes
// below 2^-149, or a square above the FP32 range.  keep() then takes the last
// vectors out again and is false, and the caller adds them in FP64.
template <typename R>
struct Squares {
    double sr = 0.0, si = 0.0;
    __device__ void add(R re, R im) {
        sr = fma(re, re, sr);
        si = fma(im, im, si);
    }
    __device__ bool keep(const Squares &) { return true; }
    __device__ void add_wide(R, R) {}
    __device__ double value() const { return sr + si; }
};
template <>
struct Squares<float> {
    double wide = 0.0;
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
    // s <- fl(s + b); returns the rounding's remainder
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
    __device__ void add(float re, float im) {
        square(re);
        square(im);
    }
    // `before`: the sum before the vectors since the last call
    __device__ bool keep(const Squares &before) {
        if (s0 >= 0x1p-90f && s0 <= 0x1p120f) return true;
        *this = before;
        return false;
    }
    __device__ void add_wide(float re, float im) {
        wide = fma((double)re, (double)re, wide);
        wide = fma((double)im, (double)im, wide);
    }
    __device__ double value() const { return wide + ((double)s0 + ((double)s1 + (double)s2)); }
};

// The bits of an amplitude but for its signs: zero if it is zero.
__device__ __forceinline__ uint32_t magnitude(float re, float im) { return (__float_as_uint(re) | __float_as_uint(im)) << 1; }
__device__ __forceinline__ uint32_t magnitude(double, double) { return 0; }  // FP64 sums are always kept

// Sum over a block by a fixed tree; the result in thread 0.
__device__ __forceinline__ double block_sum(double x) {
    __shared__ double sh[kThreads / 32];
#pragma unroll
    for (int w = 16; w; w >>= 1) x += __shfl_down_sync(0xffffffffu, x, w);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x < 32) {
        x = threadIdx.x < kThreads / 32 ? sh[threadIdx.x] : 0.0;
#pragma unroll
        for (int w = kThreads / 64; w; w >>= 1) x += __shfl_down_sync(0xffffffffu, x, w);
    }
    return x;
}

// p0 and p1 of the measured qubit: each thread takes the vectors that differ
// in it (VB = 1 and the qubit bit 0: `intra`, both in one vector).  The last
// block to finish adds the blocks' sums in a fixed tree and decides: the
// outcome (smallest i with C_i > u C_last) and the kept half's scale.  As FP64
// sums of every amplitude and one thread over 1024 partials this took 216 us
// at n = 23 (64 MiB).
template <typename R, int VB>
__global__ void __launch_bounds__(kThreads, 4)
k_meas_decide(const R *__restrict__ s, uint64_t units, int pos, uint64_t tbit, bool intra, double *__restrict__ part,
              unsigned *__restrict__ done, double u, double *dec, uint8_t *outcome) {
    using T = typename Vec<R, VB>::T;
    __shared__ bool last;
    const T *v = reinterpret_cast<const T *>(s);
    auto at = [&](uint64_t i) { return intra ? i : ((i >> pos) << (pos + 1)) | (i & ((UINT64_C(1) << pos) - 1)); };
    Squares<R> s0, s1;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t u0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; u0 < units; u0 += stride * kItems) {
        T a[kItems], b[kItems];
#pragma unroll
        for (int k = 0; k < kItems; k++) {
            const uint64_t i = u0 + k * stride;
            a[k] = b[k] = T{};
            if (i >= units) continue;
            const uint64_t x = at(i);
            a[k] = v[x];
            if (!intra) b[k] = v[x | tbit];
        }
        const Squares<R> was0 = s0, was1 = s1;
        uint32_t any0 = 0, any1 = 0;  // zero if the vectors have zeros only
#pragma unroll
        for (int k = 0; k < kItems; k++) {
            const R *pa = reinterpret_cast<const R *>(&a[k]), *pb = reinterpret_cast<const R *>(&b[k]);
            if (intra) {
                s0.add(pa[0], pa[1]);
                any0 |= magnitude(pa[0], pa[1]);
                if (VB) {
                    s1.add(pa[VB * 2], pa[VB * 2 + 1]);
                    any1 |= magnitude(pa[VB * 2], pa[VB * 2 + 1]);
                }
            } else {
#pragma unroll
                for (int e = 0; e < (1 << VB); e++) {
                    s0.add(pa[2 * e], pa[2 * e + 1]);
                    s1.add(pb[2 * e], pb[2 * e + 1]);
                    any0 |= magnitude(pa[2 * e], pa[2 * e + 1]);
                    any1 |= magnitude(pb[2 * e], pb[2 * e + 1]);
                }
            }
        }
        // (zeros, in the half that an earlier measurement cleared, add nothing:
        // read again one by one they made the measurement of a qubit measured
        // before take 100 us instead of 44 at n = 23; the other vectors are read
        // again: kept, they cost a resident block)
        const bool ok0 = s0.keep(was0) || !any0, ok1 = s1.keep(was1) || !any1;
        if (ok0 && ok1) continue;
#pragma unroll 1
        for (int k = 0; k < kItems; k++) {
            const uint64_t i = u0 + k * stride;
            if (i >= units) break;
            const uint64_t x = at(i);
            const T wa = v[x], wb = intra ? T{} : v[x | tbit];
            const R *pa = reinterpret_cast<const R *>(&wa), *pb = reinterpret_cast<const R *>(&wb);
            if (intra) {
                if (!ok0) s0.add_wide(pa[0], pa[1]);
                if (VB && !ok1) s1.add_wide(pa[VB * 2], pa[VB * 2 + 1]);
                continue;
            }
#pragma unroll
            for (int e = 0; e < (1 << VB); e++) {
                if (!ok0) s0.add_wide(pa[2 * e], pa[2 * e + 1]);
                if (!ok1) s1.add_wide(pb[2 * e], pb[2 * e + 1]);
            }
        }
    }
    double p0 = block_sum(s0.value()), p1 = block_sum(s1.value());
    if (threadIdx.x == 0) {
        part[2 * blockIdx.x] = p0;
        part[2 * blockIdx.x + 1] = p1;
        __threadfence();
        last = atomicAdd(done, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    p0 = p1 = 0.0;
    for (unsigned b = threadIdx.x; b < gridDim.x; b += kThreads) {
        p0 += __ldcg(part + 2 * b);
        p1 += __ldcg(part + 2 * b + 1);
    }
    p0 = block_sum(p0);
    p1 = block_sum(p1);
    if (threadIdx.x == 0) {
        const double total = p0 + p1;
        const int out = (p0 > u * total) ? 0 : 1;
        const double keep = out ? p1 : p0;
        dec[0] = (double)out;
        dec[1] = keep > 0.0 ? 1.0 / sqrt(keep) : 0.0;
        *outcome = (uint8_t)out;
        *done = 0;
    }
}

// The kept half scaled, the other one zeroed (written without reading it).
template <typename R, int VB>
__global__ void __launch_bounds__(kThreads)
k_meas_collapse(R *__restrict__ s, uint64_t units, int pos, uint64_t tbit, bool intra, const double *__restrict__ dec) {
    using T = typename Vec<R, VB>::T;
    T *v = reinterpret_cast<T *>(s);
    const int out = (int)dec[0];
    const R sc = (R)dec[1];
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t u0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; u0 < units; u0 += stride * kItems) {
        T a[kItems];
        uint64_t x[kItems];
#pragma unroll
        for (int k = 0; k < kItems; k++) {
            const uint64_t i = u0 + k * stride;
            if (i >= units) break;
            x[k] = intra ? i : ((i >> pos) << (pos + 1)) | (i & ((UINT64_C(1) << pos) - 1));
            if (!intra && out) x[k] |= tbit;
            a[k] = v[x[k]];
        }
#pragma unroll
        for (int k = 0; k < kItems; k++) {
            if (u0 + k * stride >= units) break;
            R *pa = reinterpret_cast<R *>(&a[k]);
#pragma unroll
            for (int e = 0; e < (2 << VB); e++) pa[e] = intra && (e >> 1) != out ? R(0) : pa[e] * sc;
            v[x[k]] = a[k];
            if (!intra) v[x[k] ^ tbit] = T{};
        }
    }
}

unsigned grid_of(uint64_t units, int sm_count) {
    const uint64_t b = (units + kThreads - 1) / kThreads;
    return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>(b, (uint64_t)sm_count * 16));
}

// The bits of `fixed`, in vectors of 2^vb amplitudes.
Ins make_ins(uint64_t fixed, int vb) {
    Ins in{};
    for (int b = 0; b < 64; b++)
        if ((fixed >> b) & 1) in.pos[in.n++] = (int8_t)(b - vb);
    return in;
}

template <typename R>
sv_status launch_general(sv_state *h, const sv_gate *g, sv_launch_record &meta) {
    R *s = reinterpret_cast<R *>(h->amps);
    const int n = h->n;
    const uint64_t N = UINT64_C(1) << n;
    if (g[0].kind == SV_MCU) {
        const uint64_t cm = (uint64_t)g[0].num, tb = UINT64_C(1) << g[0].target;
        const int k = __builtin_popcountll(cm);
        const Mat2 m = gate_matrix(g[0]);
        C2<R> c;
        for (int e = 0; e < 4; e++) {
            c.re[e] = (R)m.re[e];
            c.im[e] = (R)m.im[e];
        }
        // complex64: two neighbouring amplitudes at a time unless bit 0 is
        // one of the gate's
        const int vb = sizeof(R) == 4 && !((cm | tb) & 1) ? 1 : 0;
        const uint64_t units = UINT64_C(1) << (n - 1 - k - vb);
        meta.bytes = 2.0 * std::ldexp(1.0, -k) * (double)state_bytes(h);
        const int slot = prof_begin(h);
        const unsigned grid = grid_of((units + kItems - 1) / kItems, h->sm_count);
        if (vb) {
            if constexpr (sizeof(R) == 4)
                k_mcu<R, 1><<<grid, kThreads, 0, h->stream>>>(s, units, make_ins(cm | tb, 1), cm >> 1, tb >> 1, c);
        } else {
            k_mcu<R, 0><<<grid, kThreads, 0, h->stream>>>(s, units, make_ins(cm | tb, 0), cm, tb, c);
        }
        SV_CUDA(cudaGetLastError());
        note_launch();
        prof_end(h, slot, meta);
    } else if (g[0].kind == SV_U2Q) {
        const uint64_t ma = UINT64_C(1) << g[0].target, mb = UINT64_C(1) << g[0].control;
        C4<R> m;
        for (int r = 0; r < 4; r++)
            for (int k = 0; k < 4; k++) {
                m.re[4 * r + k] = (R)g[r].p[2 * k];
                m.im[4 * r + k] = (R)g[r].p[2 * k + 1];
            }
        const int vb = sizeof(R) == 4 && !((ma | mb) & 1) ? 1 : 0;
        const uint64_t units = N >> (2 + vb);
        meta.bytes = 2.0 * (double)state_bytes(h);
        const int slot = prof_begin(h);
        const unsigned grid = grid_of((units + 1) / 2, h->sm_count);
        if (vb) {
            if constexpr (sizeof(R) == 4)
                k_u2q<R, 1><<<grid, kThreads, 0, h->stream>>>(s, units, make_ins(ma | mb, 1), ma >> 1, mb >> 1, m);
        } else {
            k_u2q<R, 0><<<grid, kThreads, 0, h->stream>>>(s, units, make_ins(ma | mb, 0), ma, mb, m);
        }
        SV_CUDA(cudaGetLastError());
        note_launch();
        prof_end(h, slot, meta);
    } else {  // SV_MEASURE
        SV_TRY(ensure_meas(h, h->nmeas + 1));
        double *part = reinterpret_cast<double *>(h->small);
        double *dec = part + 2 * kMeasBlocks;
        unsigned *done = reinterpret_cast<unsigned *>(static_cast<char *>(h->small) + kSmallDone);
        // complex64 vectors hold two amplitudes: a measurement of bit 0 finds
        // both halves in each vector
        constexpr int VB = sizeof(R) == 4 ? 1 : 0;
        const int q = g[0].target;
        const bool intra = VB && q == 0;
        const int pos = intra ? 0 : q - VB;
        const uint64_t units = intra ? N >> 1 : N >> (1 + VB);
        const uint64_t tb = intra ? 0 : UINT64_C(1) << pos;
        const unsigned grid = grid_of((units + kItems - 1) / kItems, h->sm_count);
        const unsigned nb = std::min<unsigned>(kMeasBlocks, grid);
        // one read to sum; one read of the kept half and one write to collapse
        meta.bytes = 2.5 * (double)state_bytes(h);
        const int slot = prof_begin(h);
        k_meas_decide<R, VB><<<nb, kThreads, 0, h->stream>>>(s, units, pos, tb, intra, part, done, g[0].p[0], dec,
                                                            h->meas_dev + h->nmeas);
        k_meas_collapse<R, VB><<<grid, kThreads, 0, h->stream>>>(s, units, pos, tb, intra, dec);
        SV_CUDA(cudaGetLastError());
        note_launch(2);
        prof_end(h, slot, meta);
        h->nmeas++;
    }
    h->stats.kernels++;
    return SV_OK;
}

}  // namespace

int general_records(int kind) { return kind == SV_U2Q ? 4 : 1; }

bool is_general_kind(int kind) { return kind == SV_MCU || kind == SV_U2Q || kind == SV_MEASURE; }

sv_status general_apply(sv_state *h, const sv_gate *g) {
    static_assert(2 * kMeasBlocks * sizeof(double) + 64 <= kSmallDone, "measurement scratch fits the small area");
    SV_TRY(materialize(h));
    SV_TRY(resolve_norm(h));
    SV_TRY(launch_check());
    sv_launch_record meta{};
    meta.kind = SV_KERNEL_PERGATE;
    meta.pass = h->launch_index++;
    meta.n = h->n;
    meta.nops = 1;
    meta.ngates = 1;
    meta.dtype = (int32_t)h->dt;
    meta.gate_kind = g[0].kind;
    meta.feat = UINT64_C(1) << g[0].target;
    if (g[0].kind == SV_MCU) meta.feat |= (uint64_t)g[0].num;
    if (g[0].kind == SV_U2Q) meta.feat |= UINT64_C(1) << g[0].control;
    const sv_status st = h->dt == SV_C128 ? launch_general<double>(h, g, meta)
                                          : launch_general<float>(h, g, meta);
    if (st != SV_OK) return st;
    h->stats.passes++;
    h->stats.touched_bytes += meta.bytes;
    return SV_OK;
}

sv_status ensure_meas(sv_state *h, size_t count) {
    if (count <= h->meas_cap) return SV_OK;
    const size_t cap = std::max<size_t>(2 * count, 256);
    uint8_t *p = nullptr;
    if (dev_malloc(&p, cap) != cudaSuccess) {
        cudaGetLastError();
        return fail(SV_ERR_OOM, "cannot allocate the measurement outcomes (%zu bytes)", cap);
    }
    if (h->meas_dev) {
        SV_CUDA(cudaMemcpyAsync(p, h->meas_dev, h->nmeas, cudaMemcpyDeviceToDevice, h->stream));
        SV_CUDA(cudaStreamSynchronize(h->stream));
        cudaFree(h->meas_dev);
    }
    h->meas_dev = p;
    h->meas_cap = cap;
    return SV_OK;
}

}  // namespace sv
