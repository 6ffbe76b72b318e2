// k_reduce.cu -- one-pass <Z_i> for every qubit and the squared norm.
//
// <Z_i> = sum_k |psi_k|^2 (1 - 2 bit_i(k)) = T - 2 S_i with T = sum_k |psi_k|^2 and
// S_i = sum over k with bit i set. One read of the state gives T and all S_i:
//  - a block works on tiles of 2^TB consecutive amplitudes; inside a tile the amplitude
//    offset is (j, thread, v) with v the element inside a 16-byte vector (complex64 only),
//    the thread index (lane bits, then warp bits) and the unrolled load index j (4 bits);
//  - each thread sums |psi|^2 over its 32 (complex64) or 16 (complex128) values, also per
//    v bit and per j bit (those bits are compile-time constants of the unrolled loop);
//  - warp shuffles reduce the per-thread sums and form the lane-bit sums;
//  - warp totals give the warp-bit sums; bits at or above TB are constant per tile and
//    take the tile total when set;
//  - thread b of the block owns output b and accumulates it over the block's tiles; a final
//    one-block pass adds the per-block results in float64 in a fixed order.
// Complex64: per-thread, per-warp and per-tile sums are float32 (at most 32, 1024 and 8192
// terms), the running sum over a block's tiles is a compensated (Kahan) float32 sum, and the
// sum over blocks is float64. Complex128: float64 everywhere. The result does not depend on
// scheduling (fixed tile-to-block assignment and fixed summation order).
//
// Complex128 in float64 arithmetic is bound by the FP64 pipe (2 operations per SM and clock; |psi|^2
// and the sums took ~5 per amplitude, 2.5 clocks against 0.7 of memory time). A thread's 16 values
// therefore share one power-of-two scale and are squared and added as 64-bit integers
// (k_expz_c128): 58-bit magnitudes, |x|^2 as xh^2 + yh^2 + (the cross and low products >> 30) in
// units of 2^-56 of the scale's square, below 2^57 each, so that the 16-value sums are exact. Five
// sums per 16 values become float64 and are added there. The warp-level sums are formed once per
// run of 2^m consecutive tiles (the low m tile bits have per-thread sums of their own). n = 28:
// 2.72 -> 0.80 ms (5.4 TB/s), error against exact arithmetic as before (1-2 units in the last place);
// a basis state, whose zeros add nothing, 2.74 -> 0.63. What is left in float64 keeps that pipe 61 % busy, with
// two blocks of 126 registers per SM.
#include <algorithm>

#include "k_gate.cuh"

namespace qs {
namespace {

constexpr int kRedThreads = 256;
constexpr int kRedMaxBlocks = 1024;
constexpr int kJ = 16;  // unrolled loads per thread per tile

template <typename Real> struct RedT;
template <> struct RedT<float> {
    using T2 = float2;
    static constexpr int TB = 13;  // log2(amplitudes per tile): 256 threads, 16 loads of 16 bytes
};
template <> struct RedT<double> {
    using T2 = double2;
    static constexpr int TB = 12;
};

template <typename A>
__device__ __forceinline__ A warp_sum(A v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__global__ void __launch_bounds__(kRedThreads)
k_expz_c64(const float2 *__restrict__ psi, int n, uint64_t ntiles, double *__restrict__ partials) {
    constexpr int TB = RedT<float>::TB;
    // per-warp values: [0] total, [1] element bit, [2..5] j bits, [6..10] lane bits
    __shared__ float wpart[kRedThreads / 32][11];
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    Acc<float> acc{};  // output `tid` of this block, over its tiles
    for (uint64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
        float tot = 0, sv = 0, sj[4] = {0, 0, 0, 0};
        const float4 *base = reinterpret_cast<const float4 *>(psi) + (tile << (TB - 1));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            float4 q[kJ / 2];
#pragma unroll
            for (int jj = 0; jj < kJ / 2; ++jj) q[jj] = base[(h * (kJ / 2) + jj) * kRedThreads + tid];
#pragma unroll
            for (int jj = 0; jj < kJ / 2; ++jj) {
                const int j = h * (kJ / 2) + jj;
                const float p0 = fmaf(q[jj].x, q[jj].x, q[jj].y * q[jj].y);
                const float p1 = fmaf(q[jj].z, q[jj].z, q[jj].w * q[jj].w);
                const float s = p0 + p1;
                tot += s;
                sv += p1;
#pragma unroll
                for (int b = 0; b < 4; ++b)
                    if ((j >> b) & 1) sj[b] += s;
            }
        }
        // lane-bit sums before the total is reduced
        float sl[5];
#pragma unroll
        for (int b = 0; b < 5; ++b) sl[b] = warp_sum<float>(((lane >> b) & 1) ? tot : 0.f);
        tot = warp_sum<float>(tot);
        sv = warp_sum<float>(sv);
#pragma unroll
        for (int b = 0; b < 4; ++b) sj[b] = warp_sum<float>(sj[b]);
        if (lane == 0) {
            wpart[warp][0] = tot;
            wpart[warp][1] = sv;
#pragma unroll
            for (int b = 0; b < 4; ++b) wpart[warp][2 + b] = sj[b];
#pragma unroll
            for (int b = 0; b < 5; ++b) wpart[warp][6 + b] = sl[b];
        }
        __syncthreads();
        if (tid <= n) {
            // output tid: tid == n -> total; else S_tid (sum over amplitudes with bit tid set)
            float v = 0;
            const int b = tid;
            if (b == n) {
                for (int w = 0; w < kRedThreads / 32; ++w) v += wpart[w][0];
            } else if (b < 1) {
                for (int w = 0; w < kRedThreads / 32; ++w) v += wpart[w][1];
            } else if (b < 6) {
                for (int w = 0; w < kRedThreads / 32; ++w) v += wpart[w][6 + (b - 1)];
            } else if (b < 9) {
                for (int w = 0; w < kRedThreads / 32; ++w)
                    if ((w >> (b - 6)) & 1) v += wpart[w][0];
            } else if (b < TB) {
                for (int w = 0; w < kRedThreads / 32; ++w) v += wpart[w][2 + (b - 9)];
            } else if ((tile >> (b - TB)) & 1ull) {
                for (int w = 0; w < kRedThreads / 32; ++w) v += wpart[w][0];
            }
            acc.add(v);
        }
        __syncthreads();
    }
    if (tid <= n) partials[(size_t)tid * gridDim.x + blockIdx.x] = acc.value();  // output-major
}

// A value of a thread's 16 as limbs of a 58-bit magnitude in units of 2^(E - 1080): the high 28 bits
// and twice the low 30.
__device__ __forceinline__ void magnitude(double v, int E, unsigned &h, unsigned &l2) {
    const int hi = fx::abs_hi(v);
    const int d = E - (hi >> 20);
    unsigned long long m = ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
    m <<= 7;
    asm("shr.b64 %0, %0, %1;" : "+l"(m) : "r"(d));  // (amounts above 63 give 0: zeros)
    h = (unsigned)(m >> 32);
    l2 = (unsigned)m >> 1;
}

// Sum of 16 values and the sums over the values with bit b of their index set, as a pairwise tree.
template <typename A>
__device__ __forceinline__ void tree16(const A *p, A &t, A *sj) {
    A a[8], b4[4];
#pragma unroll
    for (int i = 0; i < 8; ++i) a[i] = p[2 * i] + p[2 * i + 1];
#pragma unroll
    for (int i = 0; i < 4; ++i) b4[i] = a[2 * i] + a[2 * i + 1];
    const A c0 = b4[0] + b4[1], c1 = b4[2] + b4[3];
    t = c0 + c1;
    sj[3] = c1;
    sj[2] = b4[1] + b4[3];
    sj[1] = (a[1] + a[3]) + (a[5] + a[7]);
    sj[0] = ((p[1] + p[3]) + (p[5] + p[7])) + ((p[9] + p[11]) + (p[13] + p[15]));
}

constexpr int kRunBits = 4;            // at most: low tile bits with sums of their own
constexpr int kSqLow = 600;            // exponents whose squares the integer form takes
constexpr unsigned kSqSpan = 900;

// complex128: blocks take runs of 2^m consecutive tiles.
__global__ void __launch_bounds__(kRedThreads, 2)
k_expz_c128(const double2 *__restrict__ psi, int n, int m, uint64_t nruns, double *__restrict__ partials) {
    constexpr int TB = RedT<double>::TB;
    // per-warp values: [0] total, [1..4] j bits, [5..8] low tile bits, [9..13] lane bits
    __shared__ double wpart[kRedThreads / 32][14];
    const int tid = threadIdx.x;
    const int lane = tid & 31;
    const int warp = tid >> 5;
    double acc = 0;  // output `tid` of this block, over its runs
    for (uint64_t run = blockIdx.x; run < nruns; run += gridDim.x) {
        double tot = 0, s8[8] = {0, 0, 0, 0, 0, 0, 0, 0};  // j bits, then low tile bits
        for (int tl = 0; tl < (1 << m); ++tl) {
            const double2 *base = psi + (((run << m) | (uint64_t)tl) << TB);
            double2 q[kJ];
#pragma unroll
            for (int j = 0; j < kJ; ++j) q[j] = base[j * kRedThreads + tid];
            int top = 0;
#pragma unroll
            for (int j = 0; j < kJ; ++j) top = max(top, max(fx::abs_hi(q[j].x), fx::abs_hi(q[j].y)));
            const int E = top >> 20;
            double t, sj[4];
            if ((unsigned)(E - kSqLow) < kSqSpan) {
                unsigned long long p[kJ], ti, si[4];
#pragma unroll
                for (int j = 0; j < kJ; ++j) {
                    unsigned xh, xl, yh, yl;
                    magnitude(q[j].x, E, xh, xl);
                    magnitude(q[j].y, E, yh, yl);
                    const unsigned long long mid = (unsigned long long)xh * xl + (unsigned long long)yh * yl +
                                                   ((unsigned long long)__umulhi(xl, xl) + __umulhi(yl, yl));
                    p[j] = (unsigned long long)xh * xh + (unsigned long long)yh * yh + (mid >> 30);
                }
                tree16(p, ti, si);
                const int sc = 2 * E - 2100;
                t = fx::to_f64((long long)ti, sc);
#pragma unroll
                for (int b = 0; b < 4; ++b) sj[b] = fx::to_f64((long long)si[b], sc);
            } else if (top == 0) {  // zeros (a basis state, a register that is mostly |0>); subnormals square to 0
                t = 0;
#pragma unroll
                for (int b = 0; b < 4; ++b) sj[b] = 0;
            } else {  // infinities, NaN, or squares out of range
                double p[kJ];
#pragma unroll
                for (int j = 0; j < kJ; ++j) p[j] = fma(q[j].x, q[j].x, q[j].y * q[j].y);
                tree16(p, t, sj);
            }
            tot += t;
#pragma unroll
            for (int b = 0; b < 4; ++b) s8[b] += sj[b];
#pragma unroll
            for (int b = 0; b < kRunBits; ++b)
                if ((tl >> b) & 1) s8[4 + b] += t;
        }
        // butterfly over the lane bits: before step b, tot sums the 2^b lanes that differ from
        // this one below bit b; the half with bit b set is this lane's tot or its partner's
        double lb[5];
#pragma unroll
        for (int b = 0; b < 5; ++b) {
            const double pt = __shfl_xor_sync(0xffffffffu, tot, 1 << b);
#pragma unroll
            for (int c = 0; c < b; ++c) lb[c] += __shfl_xor_sync(0xffffffffu, lb[c], 1 << b);
            lb[b] = ((lane >> b) & 1) ? tot : pt;
            tot += pt;
        }
        // the eight other sums at once: each step trades half of them with the partner lane; sum i
        // ends in the lanes with lane / 4 == i
#pragma unroll
        for (int w = 4, of = 16; w > 0; w >>= 1, of >>= 1) {
            const bool up = lane & of;
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (i < w) s8[i] = (up ? s8[i + w] : s8[i]) + __shfl_xor_sync(0xffffffffu, up ? s8[i] : s8[i + w], of);
        }
        double v8 = s8[0];
        v8 += __shfl_xor_sync(0xffffffffu, v8, 2);
        v8 += __shfl_xor_sync(0xffffffffu, v8, 1);
        if (lane == 0) {
            wpart[warp][0] = tot;
#pragma unroll
            for (int b = 0; b < 5; ++b) wpart[warp][9 + b] = lb[b];
        }
        if ((lane & 3) == 0) wpart[warp][1 + (lane >> 2)] = v8;
        __syncthreads();
        if (tid <= n) {
            const int b = tid;
            double v = 0;
            if (b >= 5 && b < 8) {
                for (int w = 0; w < kRedThreads / 32; ++w)
                    if ((w >> (b - 5)) & 1) v += wpart[w][0];
            } else if (b == n || b < TB + m || ((run >> (b - TB - m)) & 1ull)) {
                const int at = b == n ? 0 : b < 5 ? 9 + b : b < TB ? 1 + (b - 8) : b < TB + m ? 5 + (b - TB) : 0;
                for (int w = 0; w < kRedThreads / 32; ++w) v += wpart[w][at];
            }
            acc += v;
        }
        __syncthreads();
    }
    if (tid <= n) partials[(size_t)tid * gridDim.x + blockIdx.x] = acc;  // output-major
}

// Fixed-order sum of the per-block partials (output-major: partials[b * nblocks + g]); one
// block, a warp per output: lane l adds blocks l, l + 32, ... and the warp combines its lanes
// in a fixed shuffle order.
__global__ void k_expz_final(const double *__restrict__ partials, int nblocks, int n,
                             double *__restrict__ out_z, double *__restrict__ out_norm2) {
    __shared__ double sums[kMaxQubits + 1];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int b = warp; b <= n; b += nw) {
        double v = 0.0;
        for (int g = lane; g < nblocks; g += 32) v += partials[(size_t)b * nblocks + g];
        v = warp_sum<double>(v);
        if (lane == 0) sums[b] = v;
    }
    __syncthreads();
    const int b = threadIdx.x;
    if (b < n && out_z) out_z[b] = sums[n] - 2.0 * sums[b];
    if (b == n && out_norm2) *out_norm2 = sums[n];
}

// Small states (fewer amplitudes than one tile): one block, float64 per amplitude.
template <typename Real>
__global__ void __launch_bounds__(kRedThreads)
k_expz_small(const typename RedT<Real>::T2 *__restrict__ psi, int n, double *__restrict__ out_z,
             double *__restrict__ out_norm2) {
    constexpr int kMaxSmallBits = 13;
    __shared__ double red[kRedThreads / 32][kMaxSmallBits + 1];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint64_t N = 1ull << n;
    double tot = 0.0, s[kMaxSmallBits];
#pragma unroll
    for (int b = 0; b < kMaxSmallBits; ++b) s[b] = 0.0;
    for (uint64_t k = tid; k < N; k += kRedThreads) {
        const double re = (double)psi[k].x, im = (double)psi[k].y;
        const double p = re * re + im * im;
        tot += p;
#pragma unroll
        for (int b = 0; b < kMaxSmallBits; ++b)
            if (b < n && ((k >> b) & 1ull)) s[b] += p;
    }
    tot = warp_sum<double>(tot);
#pragma unroll
    for (int b = 0; b < kMaxSmallBits; ++b) s[b] = warp_sum<double>(s[b]);
    if (lane == 0) {
        red[warp][kMaxSmallBits] = tot;
#pragma unroll
        for (int b = 0; b < kMaxSmallBits; ++b) red[warp][b] = s[b];
    }
    __syncthreads();
    if (tid == 0) {
        double T = 0.0;
        for (int w = 0; w < kRedThreads / 32; ++w) T += red[w][kMaxSmallBits];
        for (int b = 0; b < n; ++b) {
            double S = 0.0;
            for (int w = 0; w < kRedThreads / 32; ++w) S += red[w][b];
            if (out_z) out_z[b] = T - 2.0 * S;
        }
        if (out_norm2) *out_norm2 = T;
    }
}

template <typename Real>
cudaError_t expect_z_impl(const void *psi, int n, double *scratch, double *out_z, double *out_norm2,
                          cudaStream_t st) {
    using T2 = typename RedT<Real>::T2;
    constexpr int TB = RedT<Real>::TB;
    const T2 *p = reinterpret_cast<const T2 *>(psi);
    if (n < TB) {
        k_expz_small<Real><<<1, kRedThreads, 0, st>>>(p, n, out_z, out_norm2);
        return cudaGetLastError();
    }
    static const int occ = [] {
        int o = 0;
        cudaError_t e;
        if constexpr (sizeof(Real) == 8) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_expz_c128, kRedThreads, 0);
        else e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_expz_c64, kRedThreads, 0);
        return e != cudaSuccess || o < 1 ? 1 : o;
    }();
    // complex128: runs as long as at least 4096 are left to share out over the ~300 blocks
    const int m = sizeof(Real) == 8 ? std::min(kRunBits, std::max(0, n - TB - 12)) : 0;
    const uint64_t nruns = 1ull << (n - TB - m);
    const uint64_t cap = std::min<uint64_t>((uint64_t)kRedMaxBlocks, (uint64_t)device_sm_count() * occ);
    const int grid = (int)std::min<uint64_t>(nruns, cap);
    if constexpr (sizeof(Real) == 8) k_expz_c128<<<grid, kRedThreads, 0, st>>>(p, n, m, nruns, scratch);
    else k_expz_c64<<<grid, kRedThreads, 0, st>>>(p, n, nruns, scratch);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    k_expz_final<<<1, 1024, 0, st>>>(scratch, grid, n, out_z, out_norm2);
    return cudaGetLastError();
}

}  // namespace

size_t reduce_scratch_doubles(int n) { return (size_t)kRedMaxBlocks * (size_t)(n + 1); }

int expect_z_launches(int dtype, int n) { return n < (dtype == QS_C64 ? RedT<float>::TB : RedT<double>::TB) ? 1 : 2; }

cudaError_t launch_expect_z(int dtype, const void *psi, int n, double *scratch, double *out_z,
                            double *out_norm2, cudaStream_t st) {
    if (dtype == QS_Q30) return launch_expect_z_q30(psi, n, scratch, out_z, out_norm2, st);
    return dtype == QS_C64 ? expect_z_impl<float>(psi, n, scratch, out_z, out_norm2, st)
                           : expect_z_impl<double>(psi, n, scratch, out_z, out_norm2, st);
}

}  // namespace qs
