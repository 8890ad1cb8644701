// Types shared by the host-side registry / API and the device kernels of libmmasim.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>
#include "../../include/mmasim.h"

namespace mmasim {

// Every kernel of a call is launched so that its CTAs may be set up while the kernel before it in the stream ends, and begins with
// after_previous(): it touches no memory before everything in front of it in the stream has finished and can be seen.  (A kernel that
// left without waiting would let the one behind it start before the one in front of it had finished.)  Launched plainly, a
// kernel starts on the next tick of 2.05 us after the one before it; this way 1.0 us after it: kernels of 0.5 / 2.5 / 4 / 7 us one after
// the other took 4.1 / 6.2 / 6.2 / 10.3 us each, and take 2.5 / 3.7 / 5.1 / 8.0.
#ifdef __CUDACC__
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
#endif
template <class... P, class... A>
cudaError_t enqueue(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t stream, const A&... args) {
    cudaLaunchAttribute early;
    early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    early.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = &early;
    cfg.numAttrs = 1;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kernel, P(args)...);
    if (err != cudaSuccess) cudaGetLastError();         // (it is the caller's now; left in the thread, the next launch of anybody would report it)
    return err;
}

// Element formats (device-side ids).  The order is private to the library.
enum ElemFmt : int {
    EF_F64 = 0, EF_F32, EF_TF32, EF_BF16, EF_F16, EF_E4M3, EF_E5M2, EF_E3M2, EF_E2M3, EF_E2M1, EF_E8M0, EF_UE4M3,
    EF_COUNT
};
enum Specials : int { SP_IEEE = 0, SP_FN, SP_NONE, SP_E8M0 };

struct FmtDesc {
    int ebits, mbits, bias, specials, is_signed, low_ignored, storage_bits;
};

// IEEE-754 binary64/32/16, BF16 and TF32 as truncated binary32, the OCP FP8 formats (E5M2 IEEE-like, E4M3 with
// no infinity and one NaN pattern), the OCP Microscaling element formats (no specials) and scale formats.
__host__ __device__ inline FmtDesc fmt_desc(int f) {
    switch (f) {
        case EF_F64: return {11, 52, 1023, SP_IEEE, 1, 0, 64};
        case EF_F32: return {8, 23, 127, SP_IEEE, 1, 0, 32};
        case EF_TF32: return {8, 10, 127, SP_IEEE, 1, 13, 32};
        case EF_BF16: return {8, 7, 127, SP_IEEE, 1, 0, 16};
        case EF_F16: return {5, 10, 15, SP_IEEE, 1, 0, 16};
        case EF_E4M3: return {4, 3, 7, SP_FN, 1, 0, 8};
        case EF_E5M2: return {5, 2, 15, SP_IEEE, 1, 0, 8};
        case EF_E3M2: return {3, 2, 3, SP_NONE, 1, 0, 8};
        case EF_E2M3: return {2, 3, 1, SP_NONE, 1, 0, 8};
        case EF_E2M1: return {2, 1, 1, SP_NONE, 1, 0, 8};
        case EF_E8M0: return {8, 0, 127, SP_E8M0, 0, 0, 8};
        default: return {4, 3, 7, SP_FN, 0, 0, 8};   // EF_UE4M3
    }
}

enum Family : int { FAM_FMA = 0, FAM_FTZ, FAM_E, FAM_T, FAM_ST, FAM_GST, FAM_TR, FAM_GTR };
enum Rho : int { RHO_NONE = 0, RHO_RZ_FP32, RHO_RZ_E8M13, RHO_RNE_FP32, RHO_RNE_FP16 };
enum Acc : int { ACC_F32 = 0, ACC_F16, ACC_F64 };

// Everything a kernel needs to know about a model; passed by value as a kernel argument.
struct DevModel {
    int family;
    int fmt_a, fmt_b;     // ElemFmt of A and B elements
    int acc;              // Acc
    int L, F, F2, rho;
    int P, G, k_block, scale_fmt;
    int frac;             // fractional bits of a product term (mbits_a + mbits_b; GST: 2 + 2 * scale mbits)
    int inner_round;      // 0: paper; 1: TR second stage in RZ
    int packed4;          // A and B hold two FP4 codes per byte
    int literal_emax;     // 1: the maximum exponent over every term, as Algorithms 7-11 print it (generic kernels only)
};

// Per-call arguments common to the GEMM-shaped kernels.
struct GemmArgs {
    int64_t M, N, K;
    const void* A;
    const void* B;
    const void* C;
    void* D;
    int64_t lda, ldb, ldc, ldd;   // in elements
    const uint8_t* sfa;
    const uint8_t* sfb;
    int64_t ld_sfa, ld_sfb;       // scale factors per row
    int64_t k_chunk;
    const float* row_scale;
    const float* col_scale;
    int dot_mode;                 // 1: n independent dots (row t of A with row t of B), N is ignored
    // one byte per redo_rows rows of A x 128 rows of B, redo_across of them per 128 rows of B, or NULL: the emulating kernels then leave
    // a tile alone unless it touches a set one (the matrix instruction has done the rest; see mmasim_umma.cu)
    const unsigned char* redo;
    int redo_rows, redo_across;
    unsigned int* copy_timeouts;  // device counter of CTAs whose bounded wait on a bulk copy ran out (may be NULL)
    void* scratch;                // memory for the call's scratch (see take_scratch), or NULL
    size_t scratch_bytes;
};

}  // namespace mmasim

struct mmasim_model {
    int arch, a_fmt, b_fmt, acc_fmt;   // public enums
    mmasim::DevModel dev;
    mmasim_info info;
};

namespace mmasim {
// mmasim_registry.cpp
bool registry_lookup(int arch, int a_fmt, int b_fmt, int acc_fmt, mmasim_model* out, const char** why);
// mmasim_generic.cu
int launch_generic(const DevModel& m, const GemmArgs& g, cudaStream_t stream);
// mmasim_tfdpa_fast.cu
bool fast_tfdpa_supported(const DevModel& m, const GemmArgs& g);
size_t fast_tfdpa_scratch(const DevModel& m, const GemmArgs& g);         // bytes that launch_fast_tfdpa takes at most
int launch_fast_tfdpa(const DevModel& m, const GemmArgs& g, cudaStream_t stream);
// the small-tile kernels (mmasim_direct.cuh): any K, any row stride; DIRECT_NONE: the large kernel is the better one
enum DirectSize : int { DIRECT_NONE = 0, DIRECT_8x16, DIRECT_16x16, DIRECT_32x32 };
DirectSize direct_size(const DevModel& m, const GemmArgs& g, double* us = nullptr);       // `us`: about what the emulation takes
DirectSize small_size(const DevModel& m, const GemmArgs& g);                                // the best of the small tiles (where they take the call)
bool panels_on_large_tiles(const DevModel& m, const GemmArgs& g, int64_t panels, int64_t last_rows);     // a product for which direct_size has none
int launch_direct(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t stream);
int launch_gemm_noalloc(const DevModel& m, const GemmArgs& g, cudaStream_t stream);   // status code; sets the error message
// mmasim_umma.cu: the rows that the B200's own matrix instruction computes
bool umma_supported(const DevModel& m, const GemmArgs& g);
int launch_umma(const DevModel& m, const GemmArgs& g, cudaStream_t stream);
size_t umma_scratch(const DevModel& m, const GemmArgs& g);              // bytes that launch_umma takes
// mmasim_warp_mma.cu: FP16 products of few rows (of those that umma_supported takes) on the warp-level instruction
bool warp_mma_supported(const DevModel& m, const GemmArgs& g);
cudaError_t launch_warp_mma(const DevModel& m, const GemmArgs& g, cudaStream_t stream);
// mmasim_fp_fast.cu
bool fast_fp_supported(const DevModel& m, const GemmArgs& g);
int launch_fast_fp(const DevModel& m, const GemmArgs& g, cudaStream_t stream);
struct DeviationArgs {
    const void* D;                      // the model's outputs, M x N
    double* sums;                       // eight, zeroed
    unsigned int* finished;             // zeroed
    double* host;                       // device address of mapped host memory
};
// Phi_FMA in FP64 with g.C in the model's accumulator type; nothing is stored but the sums of the deviations of s.D from it
cudaError_t launch_fma64_deviations(int acc, const GemmArgs& g, const DeviationArgs& s, cudaStream_t stream);
// mmasim_gst_fast.cu
bool fast_gst_supported(const DevModel& m, const GemmArgs& g);
int launch_fast_gst(const DevModel& m, const GemmArgs& g, cudaStream_t stream);
// mmasim_dot_stream.cu
bool dot_stream_supported(const DevModel& m, const GemmArgs& g);
int launch_dot_stream(const DevModel& m, const GemmArgs& g, cudaStream_t stream);
// mmasim_hw_mma.cu
int launch_hw_mma(int kind, int64_t M, int64_t K, const void* A, const void* B, const void* C, void* D, cudaStream_t stream);
// mmasim_hw_umma.cu
int launch_hw_umma(int kind, int64_t M, int64_t K, const void* A, const void* B, const void* C, void* D, const void* sfa,
                   const void* sfb, int32_t* status, cudaStream_t stream);
// mmasim_stats.cu
int launch_error_stats(int acc, int64_t n, const void* D, const double* ref, double* stats, cudaStream_t stream);
constexpr size_t DEVIATION_SUMS = 128;          // bytes in front of the widened operands: eight sums, the number of CTAs that have finished
size_t deviation_scratch(int64_t M, int64_t N, int64_t K);
int launch_deviation_start(int fmt, int64_t M, int64_t N, int64_t K, const void* A, const void* B, void* scratch, cudaStream_t stream);
int launch_deviation_end(int acc, int64_t M, int64_t N, int64_t K, const void* C, const void* D, void* scratch, double* host, cudaStream_t stream);
int launch_reference_fp64(int fmt, int acc, int64_t M, int64_t N, int64_t K, const void* A, const void* B, const void* C, double* ref, cudaStream_t stream);
// mmasim_peak.cu
int launch_int_peak(int kind, int64_t blocks, int64_t iters, void* sink, int32_t* ops_per_round, cudaStream_t stream);
// mmasim_api.cpp
unsigned int* copy_timeout_counter();          // the current device's counter (a device variable of the library; NULL on failure)
cudaError_t scratch_pool(cudaMemPool_t* out);   // the library's own memory pool of the current device (created on first use)
// Scratch of a call: g.scratch if it is large enough, else out of the pool in the order of the stream, and back behind the call's kernels.
cudaError_t take_scratch(const GemmArgs& g, size_t bytes, cudaStream_t stream, void** out);
cudaError_t give_scratch(const GemmArgs& g, void* scratch, cudaStream_t stream);
// The status of a call that came to `st` and whose kernels counted `count` given-up waits, which join the device's total.
int given_up_waits(int st, unsigned int count, int device, const char* call);
void set_error(const char* fmt, ...);
void set_kernel_name(const char* name, const char* variant);   // mmasim_last_kernel, mmasim_last_variant
}  // namespace mmasim
