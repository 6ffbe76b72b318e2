// k_whole.cu -- many gates on a small state in one launch: the state sits in one block's shared
// memory, and the gates run there one after another, each on its reduced iteration set (Section III-B
// of arXiv 2411.18354: the 2^(n-1-c) pairs whose controls hold, each index one bit deposit).
//
// Why not register groups (k_tile_pass): a state of one tile occupies one SM whatever the kernel does,
// and there the tile pass is bound by the latency of its per-gate chain (descriptor, decode, dispatch
// into one of some two hundred unrolled code variants, most of them instruction-cache misses): 0.6 us
// a gate with nothing else on the SM to hide it. Here a gate is a few dozen instructions that stay in
// the cache, its descriptor was read while the previous gate ran, and a gate with c controls touches 2^-c of the state; what is left is the shared-memory
// traffic (4096 amplitudes read and written: 512 clocks) and a barrier per gate.
// 200 gates with 0-3 controls, complex64: 12 qubits 129 -> 87 us, 10 qubits 110 -> 56; complex128, 10
// qubits: 705 -> 160.
#include <algorithm>
#include <cstring>

#include "k_gate.cuh"
#include "k_whole.cuh"

namespace qs {
namespace {

constexpr int kWholeChunk = 128;    // descriptors staged in shared memory at a time
constexpr int kWholeSeg = 7;        // free-bit segments of n <= 14 qubits
constexpr int kWholeThreads = 512;  // at most

template <typename Real> struct alignas(16) WholeGate {
    uint16_t mask[kWholeSeg];  // pair counter -> free bits (IndexMap)
    uint8_t op, nseg;
    uint8_t shift[kWholeSeg], pad0;
    uint32_t units;           // pairs (one-sided: amplitudes) the gate changes
    // byte offsets in shared memory:
    uint32_t at;              // of the control values (and of side 1 of a one-sided gate)
    uint32_t other;           // difference of a pair's two amplitudes
    uint32_t off[3];          // differences of the pairs 1, 2 and 4 block widths further on
    Real m[8];
    typename FxOf<Real>::T fx;
};

// Position of amplitude k: consecutive pairs of a gate differ in low bits except where its target and
// controls sit, so the low four bits are mixed with the higher ones. Linear over XOR.
__host__ __device__ __forceinline__ uint32_t whole_swz(uint32_t k) { return k ^ (((k >> 4) ^ (k >> 8) ^ (k >> 12)) & 15u); }

// The thread's R pairs of a gate: counters tid, tid + blockDim, ... have disjoint bits, so their
// positions differ by XOR constants and one bit deposit serves all of them.
template <int OP, int R, typename Real, typename T2>
__device__ __forceinline__ void run_pairs(T2 *sm, const WholeGate<Real> &g) {
    uint32_t k = (threadIdx.x << g.shift[0]) & g.mask[0];
    k |= (threadIdx.x << g.shift[1]) & g.mask[1];
    if (g.nseg > 2) {  // uniform: controls
#pragma unroll
        for (int s = 2; s < kWholeSeg; ++s) k |= (threadIdx.x << g.shift[s]) & g.mask[s];  // (0 past the last)
    }
    k = (whole_swz(k) * (uint32_t)sizeof(T2)) ^ g.at;
    unsigned char *const base = reinterpret_cast<unsigned char *>(sm);
    uint32_t p[R];
#pragma unroll
    for (int r = 0; r < R; ++r) p[r] = r == 0 ? k : p[r & (r - 1)] ^ g.off[r & 1 ? 0 : r & 2 ? 1 : 2];
    if (OP == OP_SIDE) {
        T2 x[R];
#pragma unroll
        for (int r = 0; r < R; ++r) x[r] = *reinterpret_cast<T2 *>(base + p[r]);
#pragma unroll
        for (int r = 0; r < R; ++r) {
            gate_side(x[r], g);
            *reinterpret_cast<T2 *>(base + p[r]) = x[r];
        }
    } else {
        T2 x[R], y[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            x[r] = *reinterpret_cast<T2 *>(base + p[r]);
            y[r] = *reinterpret_cast<T2 *>(base + (p[r] ^ g.other));
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            gate_pair<OP>(x[r], y[r], g);
            *reinterpret_cast<T2 *>(base + p[r]) = x[r];
            *reinterpret_cast<T2 *>(base + (p[r] ^ g.other)) = y[r];
        }
    }
}

template <int OP, typename Real, typename T2>
__device__ __forceinline__ void run_op(T2 *sm, const WholeGate<Real> &g) {
    if (g.units <= blockDim.x) {
        if (threadIdx.x < g.units) run_pairs<OP, 1, Real>(sm, g);
    } else if (g.units == 2 * blockDim.x) {
        run_pairs<OP, 2, Real>(sm, g);
    } else if (g.units == 4 * blockDim.x) {
        run_pairs<OP, 4, Real>(sm, g);
    } else {
        run_pairs<OP, 8, Real>(sm, g);
    }
}

template <typename Real, typename T2>
__device__ __forceinline__ void run_gate(T2 *sm, const WholeGate<Real> &g) {
    switch (g.op) {  // uniform
    case OP_GEN: run_op<OP_GEN, Real>(sm, g); break;
    case OP_GENP: if (sizeof(Real) == 8) run_op<OP_GENP, Real>(sm, g); break;
    case OP_REAL: run_op<OP_REAL, Real>(sm, g); break;
    case OP_SWAP: run_op<OP_SWAP, Real>(sm, g); break;
    case OP_DIAG: run_op<OP_DIAG, Real>(sm, g); break;
    default: run_op<OP_SIDE, Real>(sm, g); break;
    }
}

template <typename Real>
__global__ void __launch_bounds__(kWholeThreads) k_whole(typename CxT<Real>::T *__restrict__ psi, int n,
                                                const WholeGate<Real> *__restrict__ gates, int count) {
    using T2 = typename CxT<Real>::T;
    extern __shared__ __align__(16) unsigned char smem[];
    T2 *sm = reinterpret_cast<T2 *>(smem);
    WholeGate<Real> *sg = reinterpret_cast<WholeGate<Real> *>(smem + (sizeof(T2) << n));
    const uint32_t N = 1u << n;
    for (uint32_t k = threadIdx.x; k < N; k += blockDim.x)
        if (QS_DBG_OK(k, 1)) sm[whole_swz(k)] = psi[k];
    for (int g0 = 0; g0 < count; g0 += kWholeChunk) {
        const int chunk = min(kWholeChunk, count - g0);
        __syncthreads();  // the previous chunk has been read
        const uint4 *src = reinterpret_cast<const uint4 *>(gates + g0);
        for (int i = threadIdx.x; i < (int)(chunk * sizeof(WholeGate<Real>) / 16); i += blockDim.x)
            reinterpret_cast<uint4 *>(sg)[i] = src[i];
        __syncthreads();
        if (sizeof(Real) == 4) {
            WholeGate<Real> cur = sg[0];
            for (int i = 0; i < chunk; ++i) {
                const WholeGate<Real> g = cur;
                if (i + 1 < chunk) cur = sg[i + 1];
                run_gate<Real>(sm, g);
                __syncthreads();
            }
        } else {  // (a complex128 descriptor with its limbs does not fit in registers beside the work)
            for (int i = 0; i < chunk; ++i) {
                run_gate<Real>(sm, sg[i]);
                __syncthreads();
            }
        }
    }
    for (uint32_t k = threadIdx.x; k < N; k += blockDim.x)
        if (QS_DBG_OK(k, 1)) {
            psi[k] = sm[whole_swz(k)];
            QS_DBG_WRITE(k, 1);
        }
}

inline void set_fx(WholeGate<float> &, const GatePlan &) {}
inline void set_fx(WholeGate<double> &g, const GatePlan &p) {
    make_fx(p.U, p.op, &g.fx);
    if (p.op == OP_GEN && g.fx.form == FX_GENP) g.op = OP_GENP;
}

// Threads of the block. complex64: a gate is mostly issue (each thread's index and descriptor work, 16
// multiply-adds a pair), so a thread takes 4 or, from 11 qubits, 8 pairs of an uncontrolled gate (200
// gates with 0-3 controls, 12 qubits: 1024 threads of 2 201 us, 512 of 4 106, 256 of 8 87; 10 qubits:
// 57 with 4, 61 with 8). complex128: fixed-point arithmetic, as many threads as pairs up to 512 (9
// qubits: 125 us with one pair a thread, 195 with 4).
inline uint32_t whole_threads(int n, bool dbl) {
    if (dbl) return n <= 6 ? 32u : std::min(512u, 1u << (n - 1));
    return n <= 8 ? 32u : n <= 10 ? 1u << (n - 3) : 1u << (n - 4);
}

template <typename Real>
void pack(const GatePlan &p, void *dst) {
    WholeGate<Real> g{};
    // the map of single pairs (a GatePlan's units may be wider): insert target and controls
    int pos[64], m = 0;
    for (uint64_t all = p.ctrl_mask | p.tbit; all; all &= all - 1) pos[m++] = __builtin_ctzll(all);
    IndexMap map;
    build_map(p.n, pos, m, p.ctrl_vals, &map);
    g.nseg = (uint8_t)map.nseg;
    const uint32_t threads = whole_threads(p.n, sizeof(Real) == 8);
    uint32_t far[3] = {0, 0, 0};  // the free bits of counters 1, 2 and 4 times `threads`
    for (int s = 0; s < map.nseg; ++s) {
        g.mask[s] = (uint16_t)map.mask[s];
        g.shift[s] = (uint8_t)map.shift[s];
        for (int i = 0; i < 3; ++i) far[i] |= ((threads << i) << map.shift[s]) & (uint32_t)map.mask[s];
    }
    const uint32_t bytes = 2 * sizeof(Real);
    g.at = bytes * whole_swz((uint32_t)map.ins | (p.op == OP_SIDE && p.side ? (uint32_t)p.tbit : 0u));
    g.other = bytes * whole_swz((uint32_t)p.tbit);
    for (int i = 0; i < 3; ++i) g.off[i] = bytes * whole_swz(far[i]);
    g.units = 1u << (p.n - m);
    g.op = (uint8_t)p.op;
    for (int i = 0; i < 8; ++i) g.m[i] = (Real)p.U[i];
    set_fx(g, p);
    std::memcpy(dst, &g, sizeof(g));
}

template <typename Real>
cudaError_t go(void *psi, int n, const void *gates, int count, cudaStream_t st) {
    using T2 = typename CxT<Real>::T;
    const size_t smem = (sizeof(T2) << n) + kWholeChunk * sizeof(WholeGate<Real>);
    const cudaError_t e = allow_smem(reinterpret_cast<const void *>(k_whole<Real>), smem);
    if (e != cudaSuccess) return e;
    // a gate has at most 8 block widths of pairs (run_op)
    static_assert(1 << (kWholeBitsC64 - 4) <= kWholeThreads && 1 << (kWholeBitsC128 - 4) <= 512, "more pairs per thread");
    k_whole<Real><<<1, whole_threads(n, sizeof(Real) == 8), smem, st>>>(static_cast<T2 *>(psi), n, static_cast<const WholeGate<Real> *>(gates), count);
    return cudaGetLastError();
}

}  // namespace

size_t whole_gate_bytes(int dtype) { return dtype == QS_C64 ? sizeof(WholeGate<float>) : sizeof(WholeGate<double>); }

void pack_whole_gate(int dtype, const GatePlan &p, void *dst) {
    if (dtype == QS_C64) pack<float>(p, dst);
    else pack<double>(p, dst);
}

cudaError_t launch_whole(int dtype, void *psi, int n, const void *gates, int count, cudaStream_t st) {
    return dtype == QS_C64 ? go<float>(psi, n, gates, count, st) : go<double>(psi, n, gates, count, st);
}

}  // namespace qs
