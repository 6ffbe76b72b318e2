// k_adjoint.cu -- adjoint (reverse-sweep) gradient kernels.
//
// For E = <psi|O|psi>, psi = U_G ... U_1 |psi_in>, O = sum_i Z_i:
//   lambda = O psi;  for g = G .. 1:  if g has a parameter: grad += 2 Re <lambda| dU_g U_g^dagger psi>;
//                                     psi <- U_g^dagger psi;  lambda <- U_g^dagger lambda.
// No intermediate state is stored: un-applying a unitary gate recovers the state before
// it. One kernel does the three steps of one gate on the gate's reduced iteration set
// (the 2^(n-1-c) control-satisfied pairs, Section III-B of arXiv 2411.18354), reading
// and writing psi and lambda once. A parameterised gate is a rotation exp(-i theta P / 2) about
// P = Y or Z, so dU U^dagger = (-i / 2) P and the inner product is Im <lambda| P psi> / 2, taken from
// the pair before the un-apply: four products per pair. It is summed per thread in the state's
// precision, per warp and block in float64, and per block written to a fixed slot; a
// final pass adds the slots in a fixed order.
//
// complex128 un-applies in fixed point (k_fx.cuh): in float64 arithmetic a step took 28 operations
// per pair, 14 SM clocks against 5.4 of memory time and less from the L2. n = 20 (psi and lambda in
// the L2), 8-layer ansatz gradient with its 320 rotation steps: 16.6 -> 8.1 ms, with one-sided Z rotations 7.3.
#include <algorithm>

#include "k_gate_dispatch.cuh"
#include "qs_debug.cuh"

namespace qs {

constexpr int kAdjMaxBlocks = 1024;

namespace {

enum : int { PAULI_NONE = 0, PAULI_Y = 1, PAULI_Z = 2 };

template <typename Real, typename Idx, int NS, int LAY, int R, int OP, int PAULI>
__global__ void __launch_bounds__(kGateThreads)
k_adj_step(typename CxT<Real>::T *__restrict__ psi, typename CxT<Real>::T *__restrict__ lam,
           const DevGate<Real, Idx> g, Idx units, int side, double *__restrict__ part) {
    using T2 = typename CxT<Real>::T;
    constexpr int r = Log2<R>::v;
    constexpr int A = (LAY == LAY_ADJ) ? 2 * R : R;
    // programmatic dependent launch as in k_gate: nothing is touched before the previous kernel
    // on the stream has completed
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    Real acc = 0;
    const Idx step = (Idx)gridDim.x * kGateThreads;
    for (Idx u = (Idx)blockIdx.x * kGateThreads + threadIdx.x; u < units; u += step) {
        const Idx lo = deposit<Idx, NS>(u << r, g);
        if (OP == OP_SIDE) {  // the side that changes
            const Idx k = lo | (side ? g.tbit : (Idx)0);
            if (!QS_DBG_OK(k, R)) continue;
            T2 x[R], a[R];
            Vec<Real, R>::ld(psi + k, x);
            Vec<Real, R>::ld(lam + k, a);
#pragma unroll
            for (int i = 0; i < R; ++i) {
                if (PAULI == PAULI_Z) {  // Im(conj(a) x), doubled below
                    acc = fma(a[i].x, x[i].y, acc);
                    acc = fma(-a[i].y, x[i].x, acc);
                }
                gate_side<true>(x[i], g);
                gate_side<true>(a[i], g);
            }
            Vec<Real, R>::st(psi + k, x);
            Vec<Real, R>::st(lam + k, a);
            QS_DBG_WRITE(k, R);
            continue;
        }
        if (LAY == LAY_ADJ ? !QS_DBG_OK(lo, A) : (!QS_DBG_OK(lo, R) || !QS_DBG_OK(lo | g.tbit, R))) continue;
        T2 px[A], py[(LAY == LAY_SPLIT) ? R : 1], lx[A], ly[(LAY == LAY_SPLIT) ? R : 1];
        if (LAY == LAY_ADJ) {
            Vec<Real, A>::ld(psi + lo, px);
            Vec<Real, A>::ld(lam + lo, lx);
        } else {
            Vec<Real, R>::ld(psi + lo, px);
            Vec<Real, R>::ld(psi + (lo | g.tbit), py);
            Vec<Real, R>::ld(lam + lo, lx);
            Vec<Real, R>::ld(lam + (lo | g.tbit), ly);
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            T2 &x = (LAY == LAY_ADJ) ? px[2 * i] : px[i];
            T2 &y = (LAY == LAY_ADJ) ? px[2 * i + 1] : py[i];
            T2 &a = (LAY == LAY_ADJ) ? lx[2 * i] : lx[i];
            T2 &b = (LAY == LAY_ADJ) ? lx[2 * i + 1] : ly[i];
            if (PAULI == PAULI_Y) {  // Im <l|Y p> = (b . x) - (a . y), real dot products
                acc = fma(b.x, x.x, acc);
                acc = fma(b.y, x.y, acc);
                acc = fma(-a.x, y.x, acc);
                acc = fma(-a.y, y.y, acc);
            } else if (PAULI == PAULI_Z) {  // Im(conj(a) x) - Im(conj(b) y)
                acc = fma(a.x, x.y, acc);
                acc = fma(-a.y, x.x, acc);
                acc = fma(-b.x, y.y, acc);
                acc = fma(b.y, y.x, acc);
            }
            gate_pair<OP>(x, y, g);  // psi <- U^dagger psi
            gate_pair<OP>(a, b, g);  // lambda <- U^dagger lambda
        }
        if (LAY == LAY_ADJ) {
            Vec<Real, A>::st(psi + lo, px);
            Vec<Real, A>::st(lam + lo, lx);
            QS_DBG_WRITE(lo, A);
        } else {
            QS_DBG_WRITE(lo, R);
            QS_DBG_WRITE(lo | g.tbit, R);
            Vec<Real, R>::st(psi + lo, px);
            Vec<Real, R>::st(psi + (lo | g.tbit), py);
            Vec<Real, R>::st(lam + lo, lx);
            Vec<Real, R>::st(lam + (lo | g.tbit), ly);
        }
    }
    if (PAULI != PAULI_NONE) {
        __shared__ double wsum[kGateThreads / 32];
        double v = (double)acc;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = v;
        __syncthreads();
        if (threadIdx.x == 0) {
            double s = 0.0;
            for (int w = 0; w < kGateThreads / 32; ++w) s += wsum[w];
            // one side of a Z rotation stands for both (Im <lambda|psi> = 0); side 1 counts negative
            part[blockIdx.x] = OP == OP_SIDE ? (side ? -s : s) : 0.5 * s;
        }
    }
}

// Two consecutive steps on one qubit without controls: a one-sided Z rotation (matrix and side 1 of
// gz), then a Y rotation (g); one read and write of psi and lambda and one launch instead of two (an
// ansatz layer applies RY and RZ to every qubit). n = 20 complex128,
// 8-layer gradient: 7.27 -> 5.81 ms (with half of the real update's conversions on the integer pipe
// and two blocks per SM for the tile sweep); 5.94 with a scale of its own for every part of small phases.
// Bound by the FP64 pipe (77 % busy): six multiply-adds of the derivative products and the other conversions.
template <typename Real, typename Idx, int NS, int LAY, int R>
__global__ void __launch_bounds__(kGateThreads)
k_adj_step_zy(typename CxT<Real>::T *__restrict__ psi, typename CxT<Real>::T *__restrict__ lam,
              const DevGate<Real, Idx> g, const DevGate<Real, Idx> gz, Idx units, double *__restrict__ part_z,
              double *__restrict__ part_y) {
    using T2 = typename CxT<Real>::T;
    constexpr int r = Log2<R>::v;
    constexpr int A = (LAY == LAY_ADJ) ? 2 * R : R;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    Real az = 0, ay = 0;
    const Idx step = (Idx)gridDim.x * kGateThreads;
    for (Idx u = (Idx)blockIdx.x * kGateThreads + threadIdx.x; u < units; u += step) {
        const Idx lo = deposit<Idx, NS>(u << r, g);
        if (LAY == LAY_ADJ ? !QS_DBG_OK(lo, A) : (!QS_DBG_OK(lo, R) || !QS_DBG_OK(lo | g.tbit, R))) continue;
        T2 px[A], py[(LAY == LAY_SPLIT) ? R : 1], lx[A], ly[(LAY == LAY_SPLIT) ? R : 1];
        if (LAY == LAY_ADJ) {
            Vec<Real, A>::ld(psi + lo, px);
            Vec<Real, A>::ld(lam + lo, lx);
        } else {
            Vec<Real, R>::ld(psi + lo, px);
            Vec<Real, R>::ld(psi + (lo | g.tbit), py);
            Vec<Real, R>::ld(lam + lo, lx);
            Vec<Real, R>::ld(lam + (lo | g.tbit), ly);
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            T2 &x = (LAY == LAY_ADJ) ? px[2 * i] : px[i];
            T2 &y = (LAY == LAY_ADJ) ? px[2 * i + 1] : py[i];
            T2 &a = (LAY == LAY_ADJ) ? lx[2 * i] : lx[i];
            T2 &b = (LAY == LAY_ADJ) ? lx[2 * i + 1] : ly[i];
            az = fma(b.y, y.x, az);  // -Im(conj(b) y): side 1 of a Z rotation (k_adj_step)
            az = fma(-b.x, y.y, az);
            gate_side<true>(y, gz);
            gate_side<true>(b, gz);
            ay = fma(b.x, x.x, ay);
            ay = fma(b.y, x.y, ay);
            ay = fma(-a.x, y.x, ay);
            ay = fma(-a.y, y.y, ay);
            gate_pair<OP_REAL>(x, y, g);
            gate_pair<OP_REAL>(a, b, g);
        }
        if (LAY == LAY_ADJ) {
            Vec<Real, A>::st(psi + lo, px);
            Vec<Real, A>::st(lam + lo, lx);
            QS_DBG_WRITE(lo, A);
        } else {
            QS_DBG_WRITE(lo, R);
            QS_DBG_WRITE(lo | g.tbit, R);
            Vec<Real, R>::st(psi + lo, px);
            Vec<Real, R>::st(psi + (lo | g.tbit), py);
            Vec<Real, R>::st(lam + lo, lx);
            Vec<Real, R>::st(lam + (lo | g.tbit), ly);
        }
    }
    __shared__ double wsum[2][kGateThreads / 32];
    double v[2] = {(double)az, (double)ay};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
        if ((threadIdx.x & 31) == 0) wsum[q][threadIdx.x >> 5] = v[q];
    }
    __syncthreads();
    if (threadIdx.x < 2) {
        double s = 0.0;
        for (int w = 0; w < kGateThreads / 32; ++w) s += wsum[threadIdx.x][w];
        (threadIdx.x ? part_y : part_z)[blockIdx.x] = threadIdx.x ? 0.5 * s : s;
    }
}

// lambda_k = (n - 2 popcount(k)) psi_k : O = sum_i Z_i is diagonal with that eigenvalue (complex128).
__global__ void k_obs_sumz(const double2 *__restrict__ psi, double2 *__restrict__ lam, int n, uint64_t N) {
    const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N; k += step) {
        const double w = (double)(n - 2 * __popcll(k));
        double2 v = psi[k];
        v.x *= w;
        v.y *= w;
        lam[k] = v;
    }
}

__global__ void k_sum_vec(const double *__restrict__ z, int n, double *__restrict__ out) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double s = 0.0;
        for (int i = 0; i < n; ++i) s += z[i];
        *out = s;
    }
}

// lambda = O psi as above and the energy's partial sums in the same read: part[b] = this block's sum of
// (n - 2 popcount k) |psi_k|^2 (complex64: float32 over two amplitudes, a compensated running sum per
// thread, float64 across threads). One launch and one read of psi instead of the <Z_i> reduction, its
// final pass, their sum and lambda (complex128 keeps those: its reduction sums integers, k_reduce.cu).
__global__ void __launch_bounds__(256) k_obs_energy(const float2 *__restrict__ psi, float2 *__restrict__ lam, int n,
                                                    uint64_t N, double *__restrict__ part) {
    Acc<float> acc{};
    const uint64_t step = (uint64_t)gridDim.x * 256;
    for (uint64_t j = (uint64_t)blockIdx.x * 256 + threadIdx.x; j < N / 2; j += step) {
        float4 v = reinterpret_cast<const float4 *>(psi)[j];
        const float w0 = (float)(n - 2 * __popcll(2 * j)), w1 = w0 - 2.f;
        acc.add(fmaf(w0, fmaf(v.x, v.x, v.y * v.y), w1 * fmaf(v.z, v.z, v.w * v.w)));
        v.x *= w0;
        v.y *= w0;
        v.z *= w1;
        v.w *= w1;
        reinterpret_cast<float4 *>(lam)[j] = v;
    }
    __shared__ double wsum[8];
    double t = acc.value();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double e = 0.0;
        for (int w = 0; w < 8; ++w) e += wsum[w];
        part[blockIdx.x] = e;
    }
}

// Sums of the first `rows` slot rows, each into its first element: a warp per row.
__global__ void __launch_bounds__(256) k_slot_sums(double *__restrict__ part, int rows) {
    const int s = (int)((blockIdx.x * 256 + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (s >= rows) return;  // uniform over the warp
    double *row = part + (size_t)s * kAdjMaxBlocks;
    double v = 0.0;
    for (int b = lane; b < kAdjMaxBlocks; b += 32) v += row[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) row[0] = v;
}

// grad[p] = 2 * sum over the slots whose parameter is p, and over their blocks, of part[s][b]: a warp
// per parameter, lane l looking at slots l, l + 32, ... and adding blocks l, l + 32, ... of each hit
// (SUMMED: the hit's sum, which k_slot_sums left in its first element), then a fixed-order shuffle
// reduction. Warp nparams (energy != nullptr): the energy from slot row nslots. (A thread per parameter
// walking all slots, and the energy's own kernels, were two more launches; the walk took 55 us at 960 slots.)
template <bool SUMMED>
__global__ void __launch_bounds__(256) k_grad_final(const double *__restrict__ part, const int *__restrict__ slot_param,
                                                    int nslots, double *__restrict__ grad, int nparams,
                                                    double *__restrict__ energy) {
    const int p = (int)((blockIdx.x * 256 + threadIdx.x) >> 5);
    const int lane = threadIdx.x & 31;
    if (p > nparams || (p == nparams && !energy)) return;  // uniform over the warp
    double v = 0.0;
    auto add_row = [&](int s) {
        for (int b = lane; b < (SUMMED ? 1 : kAdjMaxBlocks); b += 32) v += part[(size_t)s * kAdjMaxBlocks + b];
    };
    if (p == nparams) {
        add_row(nslots);
    } else {
        for (int s0 = 0; s0 < nslots; s0 += 32) {
            const bool hit = s0 + lane < nslots && slot_param[s0 + lane] == p;
            if (SUMMED) {
                if (hit) v += part[(size_t)(s0 + lane) * kAdjMaxBlocks];
            } else {
                unsigned hits = __ballot_sync(0xffffffffu, hit);
                for (; hits; hits &= hits - 1) add_row(s0 + __ffs(hits) - 1);
            }
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) (p == nparams ? *energy : grad[p]) = p == nparams ? v : 2.0 * v;
}

template <typename K>
int occ_of(K kern) {
    int o = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, kGateThreads, 0) != cudaSuccess || o < 1) o = 1;
    return o;
}

template <typename Real, typename Idx, int NS, int LAY, int R, int OP, int PAULI>
cudaError_t go(void *psi, void *lam, const GatePlan &p, const FxMat &fx, double *part, cudaStream_t st) {
    auto kern = k_adj_step<Real, Idx, NS, LAY, R, OP, PAULI>;
    static const int occ = occ_of(kern);
    const uint64_t need = (p.units + kGateThreads - 1) / kGateThreads;
    const uint64_t cap = std::min<uint64_t>((uint64_t)device_sm_count() * occ, (uint64_t)kAdjMaxBlocks);
    const unsigned grid = (unsigned)std::max<uint64_t>(1, std::min(need, cap));
    DevGate<Real, Idx> g = gate_detail::make_dev<Real, Idx>(p, 0, 0);
    gate_detail::set_fx(g, fx);
    using T2 = typename CxT<Real>::T;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kGateThreads);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = (p.units << p.r) <= (uint64_t)grid << 15 ? 1 : 0;  // the rule of k_gate
    return cudaLaunchKernelEx(&cfg, kern, reinterpret_cast<T2 *>(psi), reinterpret_cast<T2 *>(lam), g, (Idx)p.units,
                              p.side, part);
}

template <typename Real, typename Idx, int LAY, int R>
cudaError_t go_zy(void *psi, void *lam, const GatePlan &z, const GatePlan &y, double *part_z, double *part_y,
                  cudaStream_t st) {
    auto kern = k_adj_step_zy<Real, Idx, 2, LAY, R>;  // no controls: at most two index segments
    static const int occ = occ_of(kern);
    const uint64_t need = (y.units + kGateThreads - 1) / kGateThreads;
    const uint64_t cap = std::min<uint64_t>((uint64_t)device_sm_count() * occ, (uint64_t)kAdjMaxBlocks);
    const unsigned grid = (unsigned)std::max<uint64_t>(1, std::min(need, cap));
    DevGate<Real, Idx> g = gate_detail::make_dev<Real, Idx>(y, 0, 0), gz = gate_detail::make_dev<Real, Idx>(z, 0, 0);
    FxMat fx;
    if (sizeof(Real) == 8) {
        make_fx(y.U, OP_REAL, &fx);
        gate_detail::set_fx(g, fx);
        make_fx(z.U, OP_SIDE, &fx);
        gate_detail::set_fx(gz, fx);
    }
    using T2 = typename CxT<Real>::T;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kGateThreads);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = (y.units << y.r) <= (uint64_t)grid << 15 ? 1 : 0;  // the rule of k_gate
    return cudaLaunchKernelEx(&cfg, kern, reinterpret_cast<T2 *>(psi), reinterpret_cast<T2 *>(lam), g, gz, (Idx)y.units,
                              part_z, part_y);
}

template <typename Real, typename Idx>
cudaError_t zy_by_shape(void *psi, void *lam, const GatePlan &z, const GatePlan &y, double *part_z, double *part_y,
                        cudaStream_t st) {
    if (y.layout == LAY_ADJ) return go_zy<Real, Idx, LAY_ADJ, 1>(psi, lam, z, y, part_z, part_y, st);
    if (sizeof(Real) == 4 && y.r == 1) return go_zy<Real, Idx, LAY_SPLIT, sizeof(Real) == 4 ? 2 : 1>(psi, lam, z, y, part_z, part_y, st);
    return go_zy<Real, Idx, LAY_SPLIT, 1>(psi, lam, z, y, part_z, part_y, st);
}

template <typename Real, typename Idx, int NS>
cudaError_t by_shape(void *psi, void *lam, const GatePlan &p, const FxMat &fx, double *part, cudaStream_t st) {
    constexpr bool F = sizeof(Real) == 4;
    int op = p.op;
    if (!F && op == OP_GEN && fx.form == FX_GENP) op = OP_GENP;
#define QS_ADJ_OPS(LAY, R)                                                                                     \
    if (part) {                                                                                                \
        if (op == OP_DIAG) return go<Real, Idx, NS, LAY, R, OP_DIAG, PAULI_Z>(psi, lam, p, fx, part, st);       \
        if (op == OP_REAL) return go<Real, Idx, NS, LAY, R, OP_REAL, PAULI_Y>(psi, lam, p, fx, part, st);       \
        if (op == OP_SIDE && LAY == LAY_SPLIT)                                                                 \
            return go<Real, Idx, NS, LAY_SPLIT, R, OP_SIDE, PAULI_Z>(psi, lam, p, fx, part, st);                \
    } else {                                                                                                   \
        if (op == OP_REAL) return go<Real, Idx, NS, LAY, R, OP_REAL, PAULI_NONE>(psi, lam, p, fx, part, st);    \
        if (op == OP_GEN) return go<Real, Idx, NS, LAY, R, OP_GEN, PAULI_NONE>(psi, lam, p, fx, part, st);      \
        if (op == OP_GENP) return go<Real, Idx, NS, LAY, R, F ? OP_GEN : OP_GENP, PAULI_NONE>(psi, lam, p, fx, part, st); \
        if (op == OP_DIAG) return go<Real, Idx, NS, LAY, R, OP_DIAG, PAULI_NONE>(psi, lam, p, fx, part, st);    \
        if (op == OP_SWAP) return go<Real, Idx, NS, LAY, R, OP_SWAP, PAULI_NONE>(psi, lam, p, fx, part, st);    \
        if (op == OP_SIDE && LAY == LAY_SPLIT)                                                                 \
            return go<Real, Idx, NS, LAY_SPLIT, R, OP_SIDE, PAULI_NONE>(psi, lam, p, fx, part, st);             \
    }
    if (p.layout == LAY_SPLIT) {
        if (p.r == 0) { QS_ADJ_OPS(LAY_SPLIT, 1) }
        else if (p.r == 1 && F) { QS_ADJ_OPS(LAY_SPLIT, 2) }
    } else if (p.r == 0) {
        QS_ADJ_OPS(LAY_ADJ, 1)
    }
#undef QS_ADJ_OPS
    return cudaErrorInvalidValue;
}

template <typename Real>
cudaError_t adj_step_impl(void *psi, void *lam, const GatePlan &p, double *part, cudaStream_t st) {
    if (p.units == 0) return cudaSuccess;
    const bool narrow = p.n <= 32;
    FxMat fx;
    if (sizeof(Real) == 8) make_fx(p.U, p.op, &fx);
    if (p.map.nseg <= 4)
        return narrow ? by_shape<Real, uint32_t, 4>(psi, lam, p, fx, part, st)
                      : by_shape<Real, uint64_t, 4>(psi, lam, p, fx, part, st);
    return narrow ? by_shape<Real, uint32_t, kMaxSeg>(psi, lam, p, fx, part, st)
                  : by_shape<Real, uint64_t, kMaxSeg>(psi, lam, p, fx, part, st);
}

}  // namespace

size_t adj_partials_per_slot() { return kAdjMaxBlocks; }

// part: the gradient slot of a parameterised gate (a rotation: OP_REAL about Y, OP_DIAG and OP_SIDE about Z).
cudaError_t launch_adj_step(int dtype, void *psi, void *lam, const GatePlan &p, double *part, cudaStream_t st) {
    return dtype == QS_C64 ? adj_step_impl<float>(psi, lam, p, part, st) : adj_step_impl<double>(psi, lam, p, part, st);
}

bool adj_steps_join(const GatePlan &z, const GatePlan &y) {
    return z.op == OP_SIDE && z.side == 1 && y.op == OP_REAL && z.t == y.t && z.ctrl_mask == 0 && y.ctrl_mask == 0;
}

cudaError_t launch_adj_step_zy(int dtype, void *psi, void *lam, const GatePlan &z, const GatePlan &y, double *part_z,
                               double *part_y, cudaStream_t st) {
    const bool narrow = y.n <= 32;
    if (dtype == QS_C64)
        return narrow ? zy_by_shape<float, uint32_t>(psi, lam, z, y, part_z, part_y, st)
                      : zy_by_shape<float, uint64_t>(psi, lam, z, y, part_z, part_y, st);
    return narrow ? zy_by_shape<double, uint32_t>(psi, lam, z, y, part_z, part_y, st)
                  : zy_by_shape<double, uint64_t>(psi, lam, z, y, part_z, part_y, st);
}

cudaError_t launch_obs_sumz(const void *psi, void *lam, int n, cudaStream_t st) {
    const uint64_t N = 1ull << n;
    const unsigned grid = (unsigned)std::min<uint64_t>((N + 255) / 256, (uint64_t)device_sm_count() * 8);
    k_obs_sumz<<<grid, 256, 0, st>>>(static_cast<const double2 *>(psi), static_cast<double2 *>(lam), n, N);
    return cudaGetLastError();
}

cudaError_t launch_sum_vec(const double *z, int n, double *out, cudaStream_t st) {
    k_sum_vec<<<1, 32, 0, st>>>(z, n, out);
    return cudaGetLastError();
}

// complex64, n >= 1: lambda = O psi and the energy's partial sums in part[0 .. adj_partials_per_slot())
// (zeroed by the caller).
cudaError_t launch_obs_energy(const void *psi, void *lam, int n, double *part, cudaStream_t st) {
    const uint64_t N = 1ull << n;
    const unsigned grid = (unsigned)std::max<uint64_t>(
        1, std::min<uint64_t>({(N / 2 + 255) / 256, (uint64_t)device_sm_count() * 6, (uint64_t)kAdjMaxBlocks}));
    k_obs_energy<<<grid, 256, 0, st>>>(static_cast<const float2 *>(psi), static_cast<float2 *>(lam), n, N, part);
    return cudaGetLastError();
}

int grad_final_launches(int most) { return most > 2 ? 2 : 1; }

// energy (may be null): written from the partial sums in row nslots of part. most: the most slots that
// one parameter has. Its warp reads a row of 1024 partial sums in 1.8 us, and rows follow one another (one
// parameter for all 320 slots of an n = 20 complex64 gradient: 1758 us, with the rows summed first 1188);
// a launch of its own for the rows' sums takes about as long as two rows.
cudaError_t launch_grad_final(double *part, int nslots, int most, const int *slot_param, double *grad, int nparams,
                              double *energy, cudaStream_t st) {
    if (nparams == 0 && !energy) return cudaSuccess;
    const unsigned grid = (unsigned)(((uint64_t)nparams + 1 + 7) / 8);
    if (grad_final_launches(most) > 1) {
        const int rows = nslots + (energy ? 1 : 0);
        k_slot_sums<<<(rows + 7) / 8, 256, 0, st>>>(part, rows);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        k_grad_final<true><<<grid, 256, 0, st>>>(part, slot_param, nslots, grad, nparams, energy);
    } else {
        k_grad_final<false><<<grid, 256, 0, st>>>(part, slot_param, nslots, grad, nparams, energy);
    }
    return cudaGetLastError();
}

}  // namespace qs
