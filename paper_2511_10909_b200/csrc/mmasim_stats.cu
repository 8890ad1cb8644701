// Error statistics of model outputs against an FP64 reference: the reduction behind the accuracy analysis of
// Section 6 (the deviations delta = D - D_real of Figure 3, their sign balance and size), and the widening of that
// reference's operands.  A grid-stride pass over the outputs, four in flight per thread, per-thread partial sums in FP64, reduced
// over the CTA, one atomic per CTA and statistic (one per warp, 9472 on each of eight addresses, took 85 of the 89 us
// of a 1024 x 1024 reduction).
#include <cstring>
#include "mmasim_stats.cuh"

namespace mmasim {
namespace {

template <bool ACC16>
__global__ void __launch_bounds__(256) stats_kernel(int64_t n, const void* D, const double* ref, double* out) {
    after_previous();
    stats::Deviations s;
#pragma unroll 4
    for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) s.add(stats::output_value<ACC16>(D, i), ref[i]);
    s.reduce_to<8>(out);
}

// An operand widened exactly to FP64, two elements per thread and step: 16-byte stores, consecutive threads side by side.
struct Widen {
    const void* src;
    double* dst;
    int64_t n;
    int fmt;
};
__device__ __forceinline__ double widen_one(int fmt, const void* p, int64_t i) {
    switch (fmt) {
        case EF_F16: return double(__half2float(__ushort_as_half(static_cast<const unsigned short*>(p)[i])));
        case EF_BF16: return double(__uint_as_float(uint32_t(static_cast<const uint16_t*>(p)[i]) << 16));
        case EF_TF32: return double(__uint_as_float(static_cast<const uint32_t*>(p)[i] & ~0x1FFFu));
        case EF_F32: return double(__uint_as_float(static_cast<const uint32_t*>(p)[i]));
        default: {
            const unsigned short x = static_cast<const uint8_t*>(p)[i];
            uint32_t h;
            if (fmt == EF_E5M2) asm("cvt.rn.f16x2.e5m2x2 %0, %1;" : "=r"(h) : "h"(x));
            else asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h) : "h"(x));
            return double(__half2float(__ushort_as_half((unsigned short)h)));
        }
    }
}
// (`zero`: NULL, or memory of that many bytes to be zeroed beside)
__global__ void __launch_bounds__(256) widen_kernel(Widen a, Widen b, Widen c, unsigned char* zero, int zero_bytes) {
    after_previous();
    if (zero && blockIdx.x == 0 && blockIdx.y == 0 && int(threadIdx.x) < zero_bytes) zero[threadIdx.x] = 0;
    const Widen w = blockIdx.y == 0 ? a : (blockIdx.y == 1 ? b : c);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const int64_t i = ((int64_t(blockIdx.x) * 4 + q) * 256 + threadIdx.x) * 2;
        if (i + 1 < w.n) *reinterpret_cast<double2*>(w.dst + i) = make_double2(widen_one(w.fmt, w.src, i), widen_one(w.fmt, w.src, i + 1));
        else if (i < w.n) w.dst[i] = widen_one(w.fmt, w.src, i);
    }
}

}  // namespace

int launch_error_stats(int acc, int64_t n, const void* D, const double* ref, double* stats, cudaStream_t stream) {
    if (acc != ACC_F32 && acc != ACC_F16) { set_error("mmasim_error_stats: the accumulator format must be FP32 or FP16"); return MMASIM_ERR_INVALID_ARG; }
    const int64_t want = (n + 255) / 256;
    const unsigned blocks = unsigned(want < 148 * 4 ? want : 148 * 4);
    const cudaError_t err = enqueue(acc == ACC_F16 ? stats_kernel<true> : stats_kernel<false>, blocks, 256, 0, stream, n, D, ref, stats);
    if (err != cudaSuccess) { set_error("mmasim_error_stats launch failed: %s", cudaGetErrorString(err)); return MMASIM_ERR_CUDA; }
    return MMASIM_OK;
}

// D_real = A x B^T + C in FP64 (Phi_FMA): the operands widened to scratch memory in one launch, then the FP64 kernel.
int launch_reference_fp64(int fmt, int acc, int64_t M, int64_t N, int64_t K, const void* A, const void* B, const void* C, double* ref, cudaStream_t stream) {
    cudaMemPool_t pool;
    double* scratch = nullptr;
    cudaError_t err = scratch_pool(&pool);
    const int64_t na = M * K, nb = N * K, nc = C ? M * N : 0, a_at = 0, b_at = (na + 1) / 2 * 2, c_at = b_at + (nb + 1) / 2 * 2;
    if (err == cudaSuccess) err = cudaMallocFromPoolAsync(reinterpret_cast<void**>(&scratch), size_t(c_at + nc) * 8, pool, stream);
    int st = MMASIM_OK;
    if (err == cudaSuccess) {
        const Widen wa = {A, scratch + a_at, na, fmt}, wb = {B, scratch + b_at, nb, fmt}, wc = {C, scratch + c_at, nc, acc == ACC_F16 ? EF_F16 : EF_F32};
        const int64_t most = na > nb ? (na > nc ? na : nc) : (nb > nc ? nb : nc);
        err = enqueue(widen_kernel, dim3(unsigned((most + 2047) / 2048), C ? 3 : 2), 256, 0, stream, wa, wb, wc, nullptr, 0);
    }
    if (err == cudaSuccess) {
        DevModel m;
        std::memset(&m, 0, sizeof(m));
        m.family = FAM_FMA;
        m.fmt_a = m.fmt_b = EF_F64;
        m.acc = ACC_F64;
        GemmArgs g;
        std::memset(&g, 0, sizeof(g));
        g.M = M; g.N = N; g.K = K;
        g.A = scratch + a_at; g.B = scratch + b_at; g.C = C ? scratch + c_at : nullptr; g.D = ref;
        g.lda = g.ldb = K;
        g.ldc = g.ldd = N;
        st = launch_fast_fp(m, g, stream);
    }
    if (scratch) cudaFreeAsync(scratch, stream);
    if (err != cudaSuccess) { set_error("mmasim_reference_fp64: %s", cudaGetErrorString(err)); return MMASIM_ERR_CUDA; }
    return st;
}

// The two ends of mmasim_deviation_stats.  Before the product: A and B widened, the sums zeroed.  Behind it: the FP64 kernel, whose CTAs
// compare their outputs with the model's and add up the deviations in place of storing a reference; the last one to finish writes the
// eight sums to `host`, mapped host memory.
size_t deviation_scratch(int64_t M, int64_t N, int64_t K) { return DEVIATION_SUMS + size_t((M * K + 1) / 2 * 2 + N * K) * 8; }
int launch_deviation_start(int fmt, int64_t M, int64_t N, int64_t K, const void* A, const void* B, void* scratch, cudaStream_t stream) {
    double* a = reinterpret_cast<double*>(static_cast<unsigned char*>(scratch) + DEVIATION_SUMS);
    const int64_t na = M * K, nb = N * K, most = na > nb ? na : nb;
    const Widen wa = {A, a, na, fmt}, wb = {B, a + (na + 1) / 2 * 2, nb, fmt};
    const cudaError_t err = enqueue(widen_kernel, dim3(unsigned((most + 2047) / 2048), 2), 256, 0, stream, wa, wb, wb, static_cast<unsigned char*>(scratch), int(DEVIATION_SUMS));
    if (err != cudaSuccess) { set_error("mmasim_deviation_stats: %s", cudaGetErrorString(err)); return MMASIM_ERR_CUDA; }
    return MMASIM_OK;
}
int launch_deviation_end(int acc, int64_t M, int64_t N, int64_t K, const void* C, const void* D, void* scratch, double* host, cudaStream_t stream) {
    const double* a = reinterpret_cast<const double*>(static_cast<unsigned char*>(scratch) + DEVIATION_SUMS);
    GemmArgs g;
    std::memset(&g, 0, sizeof(g));
    g.M = M; g.N = N; g.K = K;
    g.A = a; g.B = a + (M * K + 1) / 2 * 2; g.C = C;
    g.lda = g.ldb = K;
    g.ldc = g.ldd = N;
    DeviationArgs s;
    s.D = D;
    s.sums = static_cast<double*>(scratch);
    s.finished = reinterpret_cast<unsigned int*>(s.sums + stats::NSTAT);
    s.host = host;
    const cudaError_t err = launch_fma64_deviations(acc, g, s, stream);
    if (err != cudaSuccess) { set_error("mmasim_deviation_stats: %s", cudaGetErrorString(err)); return MMASIM_ERR_CUDA; }
    return MMASIM_OK;
}

}  // namespace mmasim
