// k_batch_major.cu -- helper kernels of the batch's pass-major path (qs_batch_run with
// QS_FLAG_JIT): the states of one batch program (same qubit count and gate list) live side by
// side in one buffer, and every pass of the program runs over all of them in one launch of a
// kernel compiled for that pass (qs_jit.cu). These kernels prepare the states and angles,
// form lambda = O psi with the energies, and sum the per-tile gradient partials.
#include "k_batch_major.cuh"
#include "k_gate.cuh"

namespace qs {
namespace {

constexpr int kBmThreads = 256;
constexpr uint32_t kObsChunk = 1u << 14;  // amplitudes per block of the energy pass

// psi_s = |0...0> for every state; cs[s][p] = (cos, sin) of theta / 2 for its parameters.
template <typename Real>
__global__ void __launch_bounds__(kBmThreads) k_bm_init(typename CxT<Real>::T *__restrict__ psi, int n, int S,
                                                       double *__restrict__ cs, int nparam,
                                                       const double *__restrict__ theta,
                                                       const uint64_t *__restrict__ param_off,
                                                       const int *__restrict__ gstate) {
    using T2 = typename CxT<Real>::T;
    const uint64_t N = 1ull << n, total = (uint64_t)S << n;
    const uint64_t step = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += step) {
        T2 v;
        v.x = (i & (N - 1)) == 0 ? (Real)1 : (Real)0;
        v.y = 0;
        psi[i] = v;
    }
    const uint64_t np = (uint64_t)S * nparam;
    for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < np; j += step) {
        const uint64_t s = j / nparam, p = j % nparam;
        double sn, c;
        sincos(0.5 * theta[param_off[gstate[s]] + p], &sn, &c);
        cs[2 * j] = c;
        cs[2 * j + 1] = sn;
    }
}

// One warp per (pass, state), a lane per gate: the matrices of the pass's parameterised gates for the
// state's angles, in the order they are applied. A divided rotation [c -s; s c] (the dagger in the
// sweep) holds {q, q, -q, -q, which} with the larger of c, s divided out; the next full one is
// multiplied by the product of what was divided out so far (a scan over the lanes, restarted after
// each full one), and each derivative product is scaled by its square. (A thread walking a pass's
// gates took 66 us for 70 states of 18 qubits.)
template <typename Real>
__global__ void __launch_bounds__(kBmThreads) k_bm_mats(const BatchMatPass *__restrict__ passes,
                                                       const BatchMatGate *__restrict__ gates, int S,
                                                       const double *__restrict__ cs, int nparam,
                                                       Real *__restrict__ mats) {
    const BatchMatPass P = passes[blockIdx.x];
    const int lane = threadIdx.x & 31;
    for (int s = blockIdx.y * (kBmThreads / 32) + (threadIdx.x >> 5); s < S; s += gridDim.y * (kBmThreads / 32)) {
        Real *rows = mats + P.off + (uint64_t)s * P.words;
        double carry = 1.0;  // divided out before this chunk of 32 gates
        for (int j0 = 0; j0 < P.count; j0 += 32) {
            const int j = j0 + lane;
            const bool on = j < P.count;
            BatchMatGate G{0, BM_RZ, 0};
            double c = 1.0, sn = 0.0;
            if (on) {
                G = gates[P.begin + j];
                const double *v = cs + 2 * ((uint64_t)s * nparam + G.pidx);
                c = v[0];
                sn = G.adjoint ? -v[1] : v[1];
            }
            const bool wide = fabs(sn) > fabs(c);
            const double d = wide ? sn : c;
            double prod = G.kind == BM_RY_DIVIDED ? d : 1.0;  // inclusive product since the last full gate
            int full = G.kind == BM_RY_FULL;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const double p = __shfl_up_sync(0xffffffffu, prod, o);
                const int f = __shfl_up_sync(0xffffffffu, full, o);
                if (lane >= o) {
                    if (!full) prod *= p;
                    full |= f;
                }
            }
            if (!full) prod *= carry;
            double pending = __shfl_up_sync(0xffffffffu, prod, 1);  // before this gate
            if (lane == 0) pending = carry;
            carry = __shfl_sync(0xffffffffu, prod, 31);
            if (!on) continue;
            if (G.adjoint) rows[8 * P.count + j] = (Real)(pending * pending);
            Real u[8] = {0, 0, 0, 0, 0, 0, 0, 0};
            if (G.kind == BM_RY_DIVIDED) {
                const double q = (wide ? c : sn) / d;
                u[0] = u[1] = (Real)q;
                u[2] = u[3] = (Real)-q;
                u[4] = wide ? (Real)1 : (Real)0;
            } else if (G.kind == BM_RY_FULL || G.kind == BM_RY_CONTROLLED) {
                const double f = G.kind == BM_RY_FULL ? pending : 1.0;
                u[0] = u[6] = (Real)(c * f);
                u[2] = (Real)(-sn * f);
                u[4] = (Real)(sn * f);
                if (sizeof(Real) == 4) {  // for packed multiply-adds
                    u[1] = u[0];
                    u[3] = u[2];
                    u[5] = u[4];
                    u[7] = u[6];
                }
            } else if (G.kind == BM_RZ_SIDE) {  // diag(1, e^{i theta}): the global phase is left out
                u[0] = (Real)(c * c - sn * sn);
                u[1] = (Real)(2.0 * c * sn);
            } else {
                u[0] = u[6] = (Real)c;
                u[1] = (Real)-sn;
                u[7] = (Real)sn;
            }
            using V = typename CxT<Real>::T;
#pragma unroll
            for (int i = 0; i < 8; i += 2) {
                V w;
                w.x = u[i];
                w.y = u[i + 1];
                *reinterpret_cast<V *>(rows + 8 * j + i) = w;
            }
        }
    }
}

// lambda = O psi with O = sum_i Z_i (weight n - 2 popcount(k) on amplitude k) and the
// partial sums of <psi|O|psi>, one block per chunk of a state: part[s * chunks + c].
template <typename Real>
__global__ void __launch_bounds__(kBmThreads) k_bm_obs(const typename CxT<Real>::T *__restrict__ psi,
                                                      typename CxT<Real>::T *__restrict__ lam, int n, uint32_t chunks,
                                                      double *__restrict__ part) {
    using T2 = typename CxT<Real>::T;
    __shared__ double red[kBmThreads / 32];
    const uint64_t s = blockIdx.x / chunks, c = blockIdx.x % chunks;
    const uint64_t N = 1ull << n;
    const uint64_t len = N / chunks;  // chunks divides N (both powers of two)
    const uint64_t k0 = c * len;
    const T2 *src = psi + s * N;
    T2 *dst = lam + s * N;
    Acc<Real> acc{};
    constexpr int U = 4;
    for (uint64_t k = threadIdx.x; k < len; k += (uint64_t)U * kBmThreads) {
        T2 v[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t kk = k + (uint64_t)u * kBmThreads;
            if (kk < len) v[u] = src[k0 + kk];
        }
        Real run = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const uint64_t kk = k + (uint64_t)u * kBmThreads;
            if (kk < len) {
                const Real w = (Real)(n - 2 * __popcll(k0 + kk));
                run += w * (v[u].x * v[u].x + v[u].y * v[u].y);
                v[u].x *= w;
                v[u].y *= w;
                dst[k0 + kk] = v[u];
            }
        }
        acc.add(run);
    }
    double t = acc.value();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
        double e = 0.0;
        for (int w = 0; w < kBmThreads / 32; ++w) e += red[w];
        part[blockIdx.x] = e;
    }
}

// energy of each state: its chunks' partials added in order.
__global__ void __launch_bounds__(kBmThreads) k_bm_energy(const double *__restrict__ part, int S, uint32_t chunks,
                                                         double *__restrict__ energy, const int *__restrict__ gstate) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < S; s += gridDim.x * blockDim.x) {
        double e = 0.0;
        for (uint32_t c = 0; c < chunks; ++c) e += part[(uint64_t)s * chunks + c];
        energy[gstate[s]] = e;
    }
}

// dE/dtheta_p = 2 sum over the gates p drives (in program order) of the per-tile partials of
// Re <lambda| dU psi>: block.x per state, `lanes` (a power of two <= 32) lanes per parameter, lane l
// adding tiles l, l + lanes, ..., then a fixed-order shuffle reduction (a thread per parameter and
// all its tiles took 39 us for 70 states of 128 tiles). items[csr_ptr[p] .. csr_ptr[p+1]) are the
// offsets of p's gates' partial blocks ([J][state][tile] of their sweep pass).
__global__ void __launch_bounds__(kBmThreads) k_bm_grad(const double *__restrict__ part, const int *__restrict__ csr_ptr,
                                                       const uint64_t *__restrict__ items, int nparam,
                                                       uint32_t tiles, int lanes, double *__restrict__ grad,
                                                       const uint64_t *__restrict__ param_off,
                                                       const int *__restrict__ gstate) {
    const int s = blockIdx.x, lane = threadIdx.x & (lanes - 1);
    const int p = (int)((blockIdx.y * kBmThreads + threadIdx.x) / lanes);
    double g = 0.0;
    if (p < nparam)
        for (int it = csr_ptr[p]; it < csr_ptr[p + 1]; ++it) {
            const double *q = part + items[it] + (uint64_t)s * tiles;
            for (uint32_t t = lane; t < tiles; t += lanes) g += q[t];
        }
    for (int o = lanes >> 1; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
    if (p < nparam && lane == 0) grad[param_off[gstate[s]] + p] = 2.0 * g;
}

template <typename Real>
cudaError_t init_impl(void *psi, int n, int S, double *cs, int nparam, const double *theta, const uint64_t *param_off,
                      const int *gstate, cudaStream_t st) {
    const uint64_t work = std::max<uint64_t>((uint64_t)S << n, (uint64_t)S * nparam);
    const unsigned grid = (unsigned)std::min<uint64_t>((work + kBmThreads - 1) / kBmThreads,
                                                       (uint64_t)device_sm_count() * 8);
    k_bm_init<Real><<<std::max(1u, grid), kBmThreads, 0, st>>>(static_cast<typename CxT<Real>::T *>(psi), n, S,
                                                                cs, nparam, theta, param_off,
                                                                gstate);
    return cudaGetLastError();
}

template <typename Real>
cudaError_t obs_impl(const void *psi, void *lam, int n, int S, double *part, double *energy, const int *gstate,
                     cudaStream_t st) {
    const uint64_t N = 1ull << n;
    const uint32_t chunks = (uint32_t)std::max<uint64_t>(1, N / kObsChunk);
    k_bm_obs<Real><<<(unsigned)((uint64_t)S * chunks), kBmThreads, 0, st>>>(
        static_cast<const typename CxT<Real>::T *>(psi), static_cast<typename CxT<Real>::T *>(lam), n, chunks, part);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_bm_energy<<<(S + kBmThreads - 1) / kBmThreads, kBmThreads, 0, st>>>(part, S, chunks, energy, gstate);
    return cudaGetLastError();
}

}  // namespace

size_t bm_obs_partials(int n, int S) {
    const uint64_t N = 1ull << n;
    return (size_t)S * (size_t)std::max<uint64_t>(1, N / kObsChunk);
}

cudaError_t launch_bm_init(int dtype, void *psi, int n, int S, double *cs, int nparam, const double *theta,
                           const uint64_t *param_off, const int *gstate, cudaStream_t st) {
    return dtype == QS_C64 ? init_impl<float>(psi, n, S, cs, nparam, theta, param_off, gstate, st)
                           : init_impl<double>(psi, n, S, cs, nparam, theta, param_off, gstate, st);
}

cudaError_t launch_bm_mats(int dtype, const BatchMatPass *passes, int npasses, const BatchMatGate *gates, int S,
                           const double *cs, int nparam, void *mats, cudaStream_t st) {
    if (npasses == 0 || S == 0) return cudaSuccess;
    const dim3 grid((unsigned)npasses, (unsigned)std::min(32768, (S + kBmThreads / 32 - 1) / (kBmThreads / 32)));
    if (dtype == QS_C64) k_bm_mats<float><<<grid, kBmThreads, 0, st>>>(passes, gates, S, cs, nparam, static_cast<float *>(mats));
    else k_bm_mats<double><<<grid, kBmThreads, 0, st>>>(passes, gates, S, cs, nparam, static_cast<double *>(mats));
    return cudaGetLastError();
}

cudaError_t launch_bm_obs(int dtype, const void *psi, void *lam, int n, int S, double *part, double *energy,
                          const int *gstate, cudaStream_t st) {
    return dtype == QS_C64 ? obs_impl<float>(psi, lam, n, S, part, energy, gstate, st)
                           : obs_impl<double>(psi, lam, n, S, part, energy, gstate, st);
}

cudaError_t launch_bm_grad(const double *part, const int *csr_ptr, const uint64_t *items, int nparam, int S,
                           uint32_t tiles, double *grad, const uint64_t *param_off, const int *gstate, cudaStream_t st) {
    if (nparam == 0) return cudaSuccess;
    int lanes = 1;
    while (lanes < 32 && (uint32_t)lanes < tiles) lanes *= 2;
    const dim3 blocks((unsigned)S, (unsigned)(((uint64_t)nparam * lanes + kBmThreads - 1) / kBmThreads));
    k_bm_grad<<<blocks, kBmThreads, 0, st>>>(part, csr_ptr, items, nparam, tiles, lanes, grad, param_off, gstate);
    return cudaGetLastError();
}

}  // namespace qs
