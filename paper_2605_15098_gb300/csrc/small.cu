// Resident kernel: a run of gates on a small state in one launch.
//
// A state of up to 2^15 amplitudes fits the shared memory of one cluster: each
// of its CTAs holds 2^10 amplitudes or more and the launch applies the whole
// run there (Algorithm 1 of arxiv 2605.15098 gate by gate, Sec. III-A, with
// its control rule), reading and writing global memory once.  One launch per
// gate costs about 2.6 us each at these sizes, whatever the kernel does.
//
// The gates are taken in order, in groups whose targets span at most three
// qubits (diagonal gates have none).  In a group every thread holds the eight
// amplitudes of one setting of the other qubits in registers, applies the
// group's gates to them and writes them back: one pass over shared memory and
// one barrier per group instead of one per gate.  Every amplitude sees the
// per-gate kernels' arithmetic in the same order (gateops.cuh), so the result
// has the same bits.
//
// The top qubits number the CTAs of the cluster.  A group that targets one of
// them reads and writes through distributed shared memory, between cluster
// barriers; the others need only a CTA barrier.  Latency and issue bound the
// kernel (complex64; complex128: the FP64 pipe), so it spreads over as many
// CTAs as a cluster holds: 2^10 amplitudes per CTA in up to 16 CTAs against
// 2^11 in up to 8 took 156 against 205 us for a random circuit of n = 15,
// depth 20 (440 gates; 1806 us one launch per gate), 117 against 150 us at
// n = 13; 2^9 per CTA is no faster.  QPE n = 11 to 15: 21 to 42 us.
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <vector>

#include "common.h"
#include "gateops.cuh"

namespace cg = cooperative_groups;

namespace sv {
namespace {

constexpr int kSliceLog = 10;      // amplitudes per CTA while CTAs are left
constexpr int kMaxClusterLog = 4;  // 16 CTAs where the device can place them, else 8

// log2 of the CTAs of an n-qubit state's cluster.
int cluster_log(int n, int most) { return std::max(0, std::min(most, n - kSliceLog)); }

struct SmallGroup {
    uint8_t p[3];  // target qubits, ascending
    uint8_t cross;  // a target is a cluster qubit
    uint16_t o0, o1;
};

// One gate of a group: acts on register bit j (and j2 for a SWAP) of the
// register indexes in rmask (those whose controls among the group's qubits
// are 1), on the threads whose other control qubits (tmask) are 1.
template <typename R>
struct SmallOp {
    uint8_t op, j, j2, rmask;
    uint32_t tmask;
    R pad[sizeof(R) == 4 ? 2 : 1];
    Coef<R> c;
};
static_assert(sizeof(SmallOp<float>) == 48 && sizeof(SmallOp<double>) == 80, "16-byte records");

// The launch parameter: the programme itself (no upload, nothing kept).
template <typename R, int NO>
struct SmallArgs {
    int n, nl;            // qubits; qubits inside a CTA
    int ngroups, nops;
    int gen;              // start from the product state H^{hq}|basis> of amplitude v
    uint32_t basis, hq;
    R v;
    SmallGroup group[NO];
    alignas(16) SmallOp<R> op[NO];
};

template <typename R>
struct AmpT;
template <>
struct AmpT<float> {
    using T = float2;
    static constexpr int W = 4;  // 16 amplitudes fill the 32 banks
};
template <>
struct AmpT<double> {
    using T = double2;
    static constexpr int W = 3;  // eight do
};

// Bank swizzle: the low W bits take the exclusive-or of the higher ones, W at
// a time; linear over GF(2).
template <int W>
__device__ __forceinline__ uint32_t swizzle(uint32_t i) {
    return i ^ (((i >> W) ^ (i >> (2 * W)) ^ (i >> (3 * W))) & ((1u << W) - 1));
}

__device__ __forceinline__ uint32_t insert0(uint32_t x, int p) {
    return ((x >> p) << (p + 1)) | (x & ((1u << p) - 1));
}

template <typename R, int OP, int J>
__device__ __forceinline__ void pairs(typename AmpT<R>::T (&x)[8], const Coef<R> &c, uint32_t rmask) {
    if (rmask == 0xffu) {  // no control among the group's qubits: no test per pair
#pragma unroll
        for (int i = 0; i < 4; i++) {
            const int a = ((i >> J) << (J + 1)) | (i & ((1 << J) - 1)), b = a | (1 << J);
            pair_update<R, OP>(x[a].x, x[a].y, x[b].x, x[b].y, c);
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < 4; i++) {
        const int a = ((i >> J) << (J + 1)) | (i & ((1 << J) - 1)), b = a | (1 << J);
        if ((rmask >> a) & 1) pair_update<R, OP>(x[a].x, x[a].y, x[b].x, x[b].y, c);
    }
}

template <typename R, int OP>
__device__ __forceinline__ void gate_on(int j, typename AmpT<R>::T (&x)[8], const Coef<R> &c, uint32_t rmask) {
    if (j == 0) pairs<R, OP, 0>(x, c, rmask);
    else if (j == 1) pairs<R, OP, 1>(x, c, rmask);
    else pairs<R, OP, 2>(x, c, rmask);
}

template <typename R>
__device__ __forceinline__ void apply_op(const SmallOp<R> &o, typename AmpT<R>::T (&x)[8]) {
    const uint32_t rmask = o.rmask;
    switch (o.op) {
        case OP_U: gate_on<R, OP_U>(o.j, x, o.c, rmask); break;
        case OP_H: gate_on<R, OP_H>(o.j, x, o.c, rmask); break;
        case OP_X: gate_on<R, OP_X>(o.j, x, o.c, rmask); break;
        case OP_PHASE:
#pragma unroll
            for (int r = 0; r < 8; r++)
                if ((rmask >> r) & 1) single_update<R, OP_PHASE>(x[r].x, x[r].y, o.c);
            break;
        case OP_NEG:
#pragma unroll
            for (int r = 0; r < 8; r++)
                if ((rmask >> r) & 1) single_update<R, OP_NEG>(x[r].x, x[r].y, o.c);
            break;
        default: {  // SWAP of register bits j < j2: the indexes with j set and j2 clear
            typename AmpT<R>::T t;
            if (o.j == 0 && o.j2 == 1) {
                t = x[1]; x[1] = x[2]; x[2] = t;
                t = x[5]; x[5] = x[6]; x[6] = t;
            } else if (o.j == 0) {
                t = x[1]; x[1] = x[4]; x[4] = t;
                t = x[3]; x[3] = x[6]; x[6] = t;
            } else {
                t = x[2]; x[2] = x[4]; x[4] = t;
                t = x[3]; x[3] = x[5]; x[5] = t;
            }
        }
    }
}

template <typename R, int NO>
__global__ void __launch_bounds__(512) k_small(R *__restrict__ state, const __grid_constant__ SmallArgs<R, NO> a) {
    using V = typename AmpT<R>::T;
    constexpr int W = AmpT<R>::W;
    extern __shared__ __align__(1024) unsigned char sm[];
    V *amps = reinterpret_cast<V *>(sm);
    const int nl = a.nl, tid = threadIdx.x, nt = blockDim.x;
    SmallGroup *groups = reinterpret_cast<SmallGroup *>(sm + (sizeof(V) << nl));
    SmallOp<R> *ops = reinterpret_cast<SmallOp<R> *>(sm + (sizeof(V) << nl) + sizeof(SmallGroup) * NO);
    cg::cluster_group cluster = cg::this_cluster();
    const bool single = a.n == nl;
    const uint32_t rank = single ? 0u : cluster.block_rank();
    // the programme, from the parameter block by 16-byte loads (each thread
    // its own; read in place every gate would cost a constant-cache miss)
    {
        const int4 *src = reinterpret_cast<const int4 *>(a.op);
        asm volatile("" : "+l"(src));
        int4 *dst = reinterpret_cast<int4 *>(ops);
        for (int i = tid; i < a.nops * (int)(sizeof(SmallOp<R>) / 16); i += nt) dst[i] = src[i];
        const uint64_t *gs = reinterpret_cast<const uint64_t *>(a.group);
        asm volatile("" : "+l"(gs));
        for (int i = tid; i < a.ngroups; i += nt) reinterpret_cast<uint64_t *>(groups)[i] = gs[i];
    }
    V *gstate = reinterpret_cast<V *>(state) + ((size_t)rank << nl);
    for (uint32_t i = tid; i < (1u << nl); i += nt) {
        V v;
        if (a.gen) {
            const uint32_t x = i | (rank << nl);
            v.x = ((x ^ a.basis) & ~a.hq) ? R(0) : ((__popc(x & a.basis & a.hq) & 1) ? -a.v : a.v);
            v.y = R(0);
        } else {
            v = gstate[i];
        }
        amps[swizzle<W>(i)] = v;
    }
    __syncthreads();
    const uint32_t lmask = (1u << nl) - 1;
    const uint32_t u = (uint32_t)tid;
    const bool active = u < (1u << (nl - 3));
    bool was_cross = false;
    for (int g = 0; g < a.ngroups; g++) {
        const SmallGroup G = groups[g];
        const int o0 = G.o0, o1 = G.o1;
        // the amplitudes of the previous group are in place (the first
        // group's: of the fill above)
        if (G.cross || was_cross) cluster.sync();
        else if (g) __syncthreads();
        was_cross = G.cross;
        if (!active) continue;
        uint32_t base = u | (rank << (nl - 3));
        base = insert0(insert0(insert0(base, G.p[0]), G.p[1]), G.p[2]);
        const uint32_t s0 = 1u << G.p[0], s1 = 1u << G.p[1], s2 = 1u << G.p[2];
        V *at[8];
        if (!G.cross) {
            const uint32_t b = swizzle<W>(base & lmask), w0 = swizzle<W>(s0), w1 = swizzle<W>(s1), w2 = swizzle<W>(s2);
#pragma unroll
            for (int r = 0; r < 8; r++)
                at[r] = amps + (b ^ ((r & 1) ? w0 : 0u) ^ ((r & 2) ? w1 : 0u) ^ ((r & 4) ? w2 : 0u));
        } else {
#pragma unroll
            for (int r = 0; r < 8; r++) {
                const uint32_t i = base | ((r & 1) ? s0 : 0u) | ((r & 2) ? s1 : 0u) | ((r & 4) ? s2 : 0u);
                at[r] = cluster.map_shared_rank(amps, i >> nl) + swizzle<W>(i & lmask);
            }
        }
        V x[8];
#pragma unroll
        for (int r = 0; r < 8; r++) x[r] = *at[r];
        for (int o = o0; o < o1; o++) {
            const SmallOp<R> &op = ops[o];
            if ((base & op.tmask) != op.tmask) continue;
            apply_op<R>(op, x);
        }
#pragma unroll
        for (int r = 0; r < 8; r++) *at[r] = x[r];
    }
    if (was_cross) cluster.sync();
    else __syncthreads();
    for (uint32_t i = tid; i < (1u << nl); i += nt) gstate[i] = amps[swizzle<W>(i)];
}

template <typename R, int NO>
sv_status launch_small(sv_state *h, int most, const std::vector<SmallGroup> &groups,
                       const std::vector<SmallOp<R>> &ops, const sv_launch_record &meta) {
    SV_TRY(launch_check());
    SmallArgs<R, NO> a;
    const int n = h->n;
    auto kern = k_small<R, NO>;
    const int cl = cluster_log(n, most);
    a.n = n;
    a.nl = n - cl;
    a.ngroups = (int)groups.size();
    a.nops = (int)ops.size();
    a.gen = h->basis >= 0;
    a.basis = (uint32_t)h->basis;
    a.hq = (uint32_t)h->basis_h;
    a.v = (R)std::pow(2.0, -0.5 * __builtin_popcountll(h->basis_h));
    std::copy(groups.begin(), groups.end(), a.group);
    std::copy(ops.begin(), ops.end(), a.op);
    const size_t smem = (2 * sizeof(R) << a.nl) + sizeof(SmallGroup) * NO + sizeof(SmallOp<R>) * ops.size();
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(1u << cl);
    cfg.blockDim = dim3(std::max(32, 1 << (a.nl - 3)));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = h->stream;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 1u << cl;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    const int slot = prof_begin(h);
    SV_CUDA(cudaLaunchKernelEx(&cfg, kern, reinterpret_cast<R *>(h->amps), a));
    note_launch();
    prof_end(h, slot, meta);
    h->stats.kernels++;
    if (a.gen) {
        h->basis = -1;
        h->basis_h = 0;
    }
    return SV_OK;
}

// Records a launch holds: the parameter block is at most 32,764 bytes.  Short
// lists take the small block, which is quicker to hand over.
template <typename R>
constexpr int kFewOps = 96;
template <typename R>
constexpr int kManyOps = sizeof(R) == 4 ? 512 : 320;
static_assert(sizeof(SmallArgs<float, kManyOps<float>>) <= 32000, "launch parameters");
static_assert(sizeof(SmallArgs<double, kManyOps<double>>) <= 32000, "launch parameters");

// Prepare the kernels for the current device (their attributes are the
// device's own) and return the log2 of the largest cluster it can place with
// these resources in *most.  Once per device: a second thread that comes at
// the same time sets the same.
template <typename R>
sv_status prepare_small(int device, int *most) {
    constexpr int kDevices = 64, kSmem = 128 * 1024;
    static std::atomic<int8_t> known[kDevices];  // 0: not yet
    if (device < kDevices && (*most = known[device].load(std::memory_order_acquire)) > 0) return SV_OK;
    auto prepare = [](auto kern) -> sv_status {
        SV_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
        SV_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        return SV_OK;
    };
    auto kern = k_small<R, kManyOps<R>>;
    SV_TRY(prepare(kern));
    SV_TRY(prepare(k_small<R, kFewOps<R>>));
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(1u << kMaxClusterLog);
    cfg.blockDim = dim3(512);
    cfg.dynamicSmemBytes = kSmem;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 1u << kMaxClusterLog;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int count = 0;
    const bool ok = cudaOccupancyMaxActiveClusters(&count, kern, &cfg) == cudaSuccess && count > 0;
    cudaGetLastError();
    *most = ok ? kMaxClusterLog : 3;
    if (device < kDevices) known[device].store((int8_t)*most, std::memory_order_release);
    return SV_OK;
}

template <typename R>
sv_status run_small(sv_state *h, const std::vector<sv_gate> &g) {
    const int n = h->n;
    int most = 0;
    SV_TRY(prepare_small<R>(h->device, &most));
    const int nl = n - cluster_log(n, most);
    size_t i = 0;
    std::vector<SmallGroup> groups;
    std::vector<SmallOp<R>> ops;
    std::vector<std::pair<int, int>> span;  // gates of each group
    while (i < g.size()) {
        groups.clear();
        ops.clear();
        const size_t first = i;
        uint64_t feat = 0;
        // groups until the launch is full
        while (i < g.size() && (int)ops.size() < kManyOps<R>) {
            int set[3], ns = 0;
            auto has = [&](int q) {
                for (int k = 0; k < ns; k++)
                    if (set[k] == q) return true;
                return false;
            };
            size_t e = i;
            for (; e < g.size() && ops.size() + (e - i) < (size_t)kManyOps<R>; e++) {
                if (is_diagonal_kind(g[e].kind)) continue;
                int want[2], nw = 0;
                if (!has(g[e].target)) want[nw++] = g[e].target;
                if (g[e].kind == SV_SWAP && !has(g[e].control)) want[nw++] = g[e].control;
                if (ns + nw > 3) break;
                for (int k = 0; k < nw; k++) set[ns++] = want[k];
            }
            // fill up with the highest qubits inside a CTA (their strides
            // spread over the banks)
            for (int q = nl - 1; q >= 0 && ns < 3; q--)
                if (!has(q)) set[ns++] = q;
            std::sort(set, set + 3);
            SmallGroup G{};
            for (int k = 0; k < 3; k++) G.p[k] = (uint8_t)set[k];
            G.cross = set[2] >= nl;
            G.o0 = (uint16_t)ops.size();
            auto reg = [&](int q) { return q == set[0] ? 0 : q == set[1] ? 1 : q == set[2] ? 2 : -1; };
            for (; i < e; i++) {
                const sv_gate &a = g[i];
                Mat2 m;
                SmallOp<R> o;
                std::memset(&o, 0, sizeof o);
                o.op = (uint8_t)gate_op(a, h->dt, &m);
                o.c = to_coef<R>(m);
                uint32_t need = 0;  // register bits that must be 1
                auto control = [&](int q) {
                    const int r = reg(q);
                    if (r >= 0) need |= 1u << r;
                    else o.tmask |= 1u << q;
                };
                feat |= UINT64_C(1) << a.target;
                if (a.kind == SV_SWAP) {
                    const int x = reg(a.target), y = reg(a.control);
                    o.j = (uint8_t)std::min(x, y);
                    o.j2 = (uint8_t)std::max(x, y);
                } else {
                    if (is_controlled_kind(a.kind)) control(a.control);
                    if (is_diagonal_kind(a.kind)) control(a.target);
                    else o.j = (uint8_t)reg(a.target);
                }
                for (uint32_t r = 0; r < 8; r++)
                    if ((r & need) == need) o.rmask |= (uint8_t)(1u << r);
                ops.push_back(o);
            }
            G.o1 = (uint16_t)ops.size();
            groups.push_back(G);
        }
        sv_launch_record meta{};
        meta.kind = SV_KERNEL_TILE;
        meta.pass = h->launch_index++;
        meta.n = meta.k = meta.c = n;
        meta.nops = (int)ops.size();
        meta.ngates = (int)(i - first);
        meta.dtype = (int32_t)h->dt;
        meta.gate_kind = -1;
        meta.generated = h->basis >= 0;
        meta.bytes = (meta.generated ? 1.0 : 2.0) * (double)state_bytes(h);
        meta.feat = feat;
        if (ops.size() <= (size_t)kFewOps<R>)
            SV_TRY((launch_small<R, kFewOps<R>>(h, most, groups, ops, meta)));
        else
            SV_TRY((launch_small<R, kManyOps<R>>(h, most, groups, ops, meta)));
        h->stats.passes++;
        h->stats.touched_bytes += meta.bytes;
    }
    return SV_OK;
}

}  // namespace

// complex64 up to n = 15, where SV_MODE_AUTO turns to the tile passes;
// complex128 up to n = 14: 16 SMs' FP64 pipes take 3.4 us for a U3 at n = 15
// (2.6 us for a launch over the whole chip), 1.9 us at n = 14.
bool small_fits(int n, sv_dtype dt) { return n >= 3 && n <= (dt == SV_C128 ? 14 : 15); }

sv_status small_apply(sv_state *h, const std::vector<sv_gate> &gates_phys) {
    return h->dt == SV_C128 ? run_small<double>(h, gates_phys) : run_small<float>(h, gates_phys);
}

}  // namespace sv
