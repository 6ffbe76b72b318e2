// k_gate_dispatch.cuh -- picks the k_gate instantiation for a GatePlan and launches it.
// Included once per precision (k_gate_c64.cu, k_gate_c128.cu) so the two instantiation
// sets compile in parallel.
#pragma once

#include <algorithm>

#include "k_gate.cuh"

namespace qs {
namespace gate_detail {

template <typename Real, typename Idx>
DevGate<Real, Idx> make_dev(const GatePlan &p, uint64_t cmask, uint64_t cvals) {
    DevGate<Real, Idx> g;
    for (int s = 0; s < kMaxSeg; ++s) {
        g.mask[s] = (Idx)(s < p.map.nseg ? p.map.mask[s] : 0);
        g.shift[s] = s < p.map.nseg ? p.map.shift[s] : 0;
    }
    g.ins = (Idx)p.map.ins;
    g.tbit = (Idx)p.tbit;
    g.cmask = (Idx)cmask;
    g.cvals = (Idx)cvals;
    for (int i = 0; i < 8; ++i) g.m[i] = (Real)p.U[i];
    return g;
}

inline void set_fx(DevGate<float, uint32_t> &, const FxMat &) {}
inline void set_fx(DevGate<float, uint64_t> &, const FxMat &) {}
template <typename Idx>
void set_fx(DevGate<double, Idx> &g, const FxMat &fx) {
    g.fx = fx;
}

template <typename K>
int occupancy_of(K kern) {
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, kGateThreads, 0) != cudaSuccess || occ < 1)
        occ = 1;
    return occ;
}

template <typename Real, typename Idx, int NS, int LAY, int R, int OP, bool MASKED>
cudaError_t go(void *psi, const GatePlan &p, const FxMat &fx, uint64_t cmask, uint64_t cvals, cudaStream_t st) {
    // units in flight per thread: complex64 2 with a vector on each side, 4 with one vector per unit.
    // Exchanges have no arithmetic, and with 2 units their loads and stores alternate at the memory: n = 29
    // complex64, target 14, 1 / 2 / 4 / 8 units 1.35 / 1.43 / 1.34 / 1.32 ms. Single amplitudes (an inserted
    // qubit 0: isolated 8 bytes) keep 2: X on q controlled by every lower qubit, q = 0..28, 1 / 2 / 4 units
    // 7.10 / 7.14 / 7.60 ms (q = 1 alone 1.52 / 1.46 / 1.53). complex128 exchanges take 1: n = 28, target 14,
    // 1 / 2 / 4 units 1.33 / 1.55 / 1.33 ms, X controlled by every lower qubit 5.56 / 5.86 / 5.64 (slower with 1
    // are targets 1 to 3 and 5 with a control: 0.69 / 0.67 / 0.67; adjacent pairs take 4).
    // complex128 arithmetic (one 16-byte vector per amplitude; n = 28, target 14, 1 / 2 / 4 units): general
    // 1.38 / 1.39 / 1.36 ms, real 1.40 / 1.39 / 1.35, parts of unlike size 1.97 / 1.90 / 1.94 (at five blocks
    // per SM; n = 20: 9.1 / 10.0 / 10.3 us), diagonal 1.39 / 1.41 / 1.40, one-sided 0.67 / 0.72 / 0.72.
    constexpr bool pair_unit = LAY == LAY_ADJ || OP == OP_SIDE;  // one vector per unit
    constexpr int UNR = sizeof(Real) == 4 ? (pair_unit || (OP == OP_SWAP && R == 2) ? 4 : 2)
                        : OP == OP_SWAP   ? (pair_unit ? 4 : 1)
                                          : (OP == OP_GEN || OP == OP_REAL ? 4 : 1);
    auto kern = k_gate<Real, Idx, NS, LAY, R, OP, MASKED, UNR>;
    static const int occ = occupancy_of(kern);
    const uint64_t per_block = (uint64_t)kGateThreads * UNR;
    const uint64_t need = (p.units + per_block - 1) / per_block;
    const uint64_t cap = (uint64_t)device_sm_count() * (uint64_t)occ;
    const unsigned grid = (unsigned)std::max<uint64_t>(1, std::min(need, cap));
    using T2 = typename CxT<Real>::T;
    // small gates (at most 2^15 pair counters per block of the grid: c >= 4 at n = 30) start as
    // programmatic dependents of the previous kernel, hiding their launch behind its tail; large
    // ones launch normally (their blocks would only wait on the SMs while the previous gate drains)
    const bool dependent = (p.units << p.r) <= (uint64_t)grid << 15;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kGateThreads);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = dependent ? 1 : 0;
    DevGate<Real, Idx> g = make_dev<Real, Idx>(p, cmask, cvals);
    set_fx(g, fx);
    return cudaLaunchKernelEx(&cfg, kern, reinterpret_cast<T2 *>(psi), g, (Idx)p.units, p.side);
}

template <typename Real, typename Idx, int NS, bool MASKED>
cudaError_t by_shape(void *psi, const GatePlan &p, const FxMat &fx, uint64_t cmask, uint64_t cvals, cudaStream_t st) {
    constexpr bool F = sizeof(Real) == 4;
    int op = MASKED ? (int)OP_GEN : p.op;
    if (!F && !MASKED && op == OP_GEN && fx.form == FX_GENP) op = OP_GENP;
#define QS_OPS(LAY, R)                                                                        \
    switch (op) {                                                                             \
        case OP_GEN: return go<Real, Idx, NS, LAY, R, OP_GEN, MASKED>(psi, p, fx, cmask, cvals, st); \
        case OP_GENP: if (!MASKED && !F) return go<Real, Idx, NS, LAY, R, F ? OP_GEN : OP_GENP, false>(psi, p, fx, cmask, cvals, st); break; \
        case OP_REAL: if (!MASKED) return go<Real, Idx, NS, LAY, R, OP_REAL, false>(psi, p, fx, cmask, cvals, st); break; \
        case OP_SWAP: if (!MASKED) return go<Real, Idx, NS, LAY, R, OP_SWAP, false>(psi, p, fx, cmask, cvals, st); break; \
        case OP_DIAG: if (!MASKED) return go<Real, Idx, NS, LAY, R, OP_DIAG, false>(psi, p, fx, cmask, cvals, st); break; \
        case OP_SIDE: if (!MASKED && LAY == LAY_SPLIT) return go<Real, Idx, NS, LAY_SPLIT, R, OP_SIDE, false>(psi, p, fx, cmask, cvals, st); break; \
        default: break;                                                                       \
    }
    if (p.layout == LAY_SPLIT) {
        if (p.r == 0) { QS_OPS(LAY_SPLIT, 1) }
        else if (p.r == 1 && F) { QS_OPS(LAY_SPLIT, 2) }
    } else if (p.r == 0) {
        QS_OPS(LAY_ADJ, 1)
    }
#undef QS_OPS
    return cudaErrorInvalidValue;
}

template <typename Real, typename Idx, bool MASKED>
cudaError_t by_nseg(void *psi, const GatePlan &p, const FxMat &fx, uint64_t cmask, uint64_t cvals, cudaStream_t st) {
    const int ns = p.map.nseg;
    if (ns <= 2) return by_shape<Real, Idx, 2, MASKED>(psi, p, fx, cmask, cvals, st);
    if (ns <= 4) return by_shape<Real, Idx, 4, MASKED>(psi, p, fx, cmask, cvals, st);
    if (ns <= 10) return by_shape<Real, Idx, 10, MASKED>(psi, p, fx, cmask, cvals, st);
    return by_shape<Real, Idx, kMaxSeg, MASKED>(psi, p, fx, cmask, cvals, st);
}

template <typename Real>
cudaError_t launch(void *psi, const GatePlan &p, bool masked, uint64_t cmask, uint64_t cvals,
                   cudaStream_t st) {
    if (p.units == 0) return cudaSuccess;
    const bool narrow = p.n <= 32;  // every amplitude index fits in 32 bits
    FxMat fx;
    GatePlan masked_plan;
    const GatePlan *pp = &p;
    if (sizeof(Real) == 8) {
        if (!masked) {
            make_fx(p.U, p.op, &fx);
        } else {
            // the comparator runs the arithmetic of the class its matrix has (k_fx.cuh)
            masked_plan = p;
            make_fx_full(p.U, &fx, &masked_plan.side);
            if (fx.form == FX_SIDE && masked_plan.side)  // the scalar where the kernel reads it
                for (int i = 0; i < 2; ++i) masked_plan.U[i] = p.U[6 + i];
            pp = &masked_plan;
        }
    }
    if (masked)
        return narrow ? by_nseg<Real, uint32_t, true>(psi, *pp, fx, cmask, cvals, st)
                      : by_nseg<Real, uint64_t, true>(psi, *pp, fx, cmask, cvals, st);
    return narrow ? by_nseg<Real, uint32_t, false>(psi, *pp, fx, cmask, cvals, st)
                  : by_nseg<Real, uint64_t, false>(psi, *pp, fx, cmask, cvals, st);
}

}  // namespace gate_detail
}  // namespace qs
