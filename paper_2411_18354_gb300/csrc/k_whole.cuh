// k_whole.cuh -- a run of gates on a state that fits one SM's shared memory (see k_whole.cu).
#pragma once

#include <vector>

#include "qs_internal.cuh"

namespace qs {

// Largest states that run this way (qubits): above, several tiles on several SMs are faster. With 12
// qubits complex64 only circuits whose gates select at most 0.7 of the pairs on average: register
// groups keep rows of several uncontrolled gates in registers (6-layer ansatz, 0.76: 72 us against
// 75; QFT, 0.36: 38 against 35; 0-3 controls, 0.47: 129 against 87).
constexpr int kWholeBitsC64 = 12;
constexpr int kWholeBitsC128 = 12;
inline int whole_bits(int dtype) { return dtype == QS_C64 ? kWholeBitsC64 : kWholeBitsC128; }

// Bytes of a packed gate, and packing (the state's precision).
size_t whole_gate_bytes(int dtype);
void pack_whole_gate(int dtype, const GatePlan &p, void *dst);

// `count` packed gates (device) in order on the 2^n amplitudes at psi, in one block.
cudaError_t launch_whole(int dtype, void *psi, int n, const void *gates, int count, cudaStream_t st);

}  // namespace qs
