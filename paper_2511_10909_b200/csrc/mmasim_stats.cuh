// The deviations of model outputs from an FP64 reference, summed up (mmasim_error_stats, mmasim_deviation_stats).
#pragma once
#include <cuda_fp16.h>
#include "mmasim_internal.h"

namespace mmasim {
namespace stats {

constexpr int NSTAT = 8;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    return v;
}
__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
    return v;
}
template <bool ACC16>
__device__ __forceinline__ double output_value(const void* D, int64_t i) {
    return ACC16 ? double(__half2float(__ushort_as_half(static_cast<const unsigned short*>(D)[i]))) : double(__uint_as_float(static_cast<const uint32_t*>(D)[i]));
}

// A thread's share: count, sum, sum of magnitudes, of squares, negative, positive, largest magnitude, sum of relative magnitudes.
struct Deviations {
    double cnt = 0.0, sum = 0.0, sabs = 0.0, ssq = 0.0, nneg = 0.0, npos = 0.0, mx = 0.0, srel = 0.0;

    __device__ __forceinline__ void add(double d, double r) {
        const double delta = d - r;
        if (!(fabs(delta) <= 1.7976931348623157e308)) return;        // NaN or infinite on either side: not counted
        cnt += 1.0;
        sum += delta;
        sabs += fabs(delta);
        ssq += delta * delta;
        nneg += delta < 0.0 ? 1.0 : 0.0;
        npos += delta > 0.0 ? 1.0 : 0.0;
        mx = fmax(mx, fabs(delta));
        if (r != 0.0) srel += fabs(delta) / fabs(r);
    }
    // Over a CTA of WARPS warps, all of whose threads call it, into `stats` (one atomic per statistic, by the first eight threads).
    template <int WARPS>
    __device__ __forceinline__ void reduce_to(double* stats) const {
        const double v[NSTAT] = {warp_sum(cnt), warp_sum(sum), warp_sum(sabs), warp_sum(ssq), warp_sum(nneg), warp_sum(npos), warp_max(mx), warp_sum(srel)};
        __shared__ double part[NSTAT][WARPS];
        if ((threadIdx.x & 31) == 0) {
#pragma unroll
            for (int s = 0; s < NSTAT; ++s) part[s][threadIdx.x >> 5] = v[s];
        }
        __syncthreads();
        if (threadIdx.x < NSTAT) {
            const int s = threadIdx.x;
            double t = part[s][0];
#pragma unroll
            for (int w = 1; w < WARPS; ++w) t = s == 6 ? fmax(t, part[s][w]) : t + part[s][w];
            if (s == 6) atomicMax(reinterpret_cast<unsigned long long*>(stats + s), (unsigned long long)__double_as_longlong(t));   // non-negative doubles order like their bit patterns
            else atomicAdd(stats + s, t);
        }
    }
};

}  // namespace stats
}  // namespace mmasim
