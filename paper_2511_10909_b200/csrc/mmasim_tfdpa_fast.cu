// Dispatch to the tuned FDPA kernels (T-, ST-, TR-, GTR- and E-FDPA; see mmasim_tfdpa_fast.cuh for what they share).
#include "mmasim_tfdpa_fast.cuh"
#include <algorithm>
#include <mutex>

namespace mmasim {

namespace direct {      // mmasim_direct_*.cu
cudaError_t launch_lut8(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t stream);
cudaError_t launch_f16(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t stream);
cudaError_t launch_bf16(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t stream);
cudaError_t launch_tf32(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t stream);
cudaError_t launch_tr(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t stream);
cudaError_t launch_e(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t stream);
}  // namespace direct

namespace {

bool is8(int f) { return f == EF_E4M3 || f == EF_E5M2 || f == EF_E3M2 || f == EF_E2M3 || f == EF_E2M1; }

constexpr int KIND_TR = 100, KIND_E = 101;

// 0: no tuned kernel; KIND_TR: the TR-/GTR-FDPA kernel; KIND_E: the E-FDPA kernel; otherwise 1 + element kind of the
// T-FDPA kernel
int kind_of(const DevModel& m) {
    if (m.family == FAM_E) {
        const bool ok = m.fmt_a == m.fmt_b && m.acc == ACC_F32 && ((m.fmt_a == EF_F16 && m.L == 4) || (m.fmt_a == EF_BF16 && m.L == 2));
        return ok ? KIND_E : 0;
    }
    if (m.family == FAM_TR || m.family == FAM_GTR) {
        if (m.F != 24 || m.F2 != 31 || m.rho != RHO_RNE_FP32 || m.inner_round || m.acc != ACC_F32) return 0;
        if (m.family == FAM_GTR) return (is8(m.fmt_a) && is8(m.fmt_b) && m.L == 16) ? KIND_TR : 0;
        if (m.fmt_a != m.fmt_b) return 0;
        const bool ok = (m.fmt_a == EF_F16 && m.L == 8) || (m.fmt_a == EF_BF16 && m.L == 8) || (m.fmt_a == EF_TF32 && m.L == 4);
        return ok ? KIND_TR : 0;
    }
    if ((m.family != FAM_T && m.family != FAM_ST) || m.packed4) return 0;
    if (m.family == FAM_ST) {
        const bool ok = is8(m.fmt_a) && is8(m.fmt_b) && m.F == 25 && m.L == 32 && m.rho == RHO_RZ_FP32 && m.acc == ACC_F32 &&
                        m.k_block == 32 && m.scale_fmt == EF_E8M0;
        return ok ? 1 + fast::EK_LUT8 : 0;
    }
    const bool acc_ok = (m.rho == RHO_RNE_FP16) == (m.acc == ACC_F16) && m.acc != ACC_F64;
    if (!acc_ok) return 0;
    if (is8(m.fmt_a) && is8(m.fmt_b)) {
        const bool combo = (m.F == 13 && (m.L == 16 || m.L == 32) && (m.rho == RHO_RZ_E8M13 || m.rho == RHO_RNE_FP16)) ||
                           (m.F == 25 && m.L == 32 && (m.rho == RHO_RZ_FP32 || m.rho == RHO_RNE_FP16));
        return combo ? 1 + fast::EK_LUT8 : 0;
    }
    if (m.fmt_a != m.fmt_b) return 0;
    if (m.fmt_a == EF_F16) {
        const bool combo = ((m.F == 23 && m.L == 4) || (m.F == 24 && m.L == 8) || (m.F == 25 && m.L == 16)) &&
                           (m.rho == RHO_RZ_FP32 || m.rho == RHO_RNE_FP16);
        return combo ? 1 + fast::EK_F16 : 0;
    }
    if (m.fmt_a == EF_BF16) {
        const bool combo = ((m.F == 24 && m.L == 8) || (m.F == 25 && m.L == 16)) && m.rho == RHO_RZ_FP32;
        return combo ? 1 + fast::EK_BF16 : 0;
    }
    if (m.fmt_a == EF_TF32) {
        const bool combo = ((m.F == 24 && m.L == 4) || (m.F == 25 && m.L == 8)) && m.rho == RHO_RZ_FP32;
        return combo ? 1 + fast::EK_TF32 : 0;
    }
    return 0;
}

}  // namespace

bool fast_tfdpa_supported(const DevModel& m, const GemmArgs& g) {
    const int kind = kind_of(m);
    if (!kind || g.dot_mode || m.literal_emax) return false;
    const int bytes = fmt_desc(m.fmt_a).storage_bits / 8;
    if (g.K % fast::KC) return false;
    if (g.k_chunk % fast::KC) return false;
    if ((kind == KIND_TR || kind == KIND_E) && g.k_chunk) return false;
    if (((g.lda * bytes) % 16) || ((g.ldb * bytes) % 16)) return false;      // 16-byte row starts for the vector loads
    if (m.F == 13 && g.M > 65535ll * fast::BM) return false;                // grid.y
    if (g.N > 0x7FFFFFFFll - 128 || g.K > 0x7FFFFFFFll - 64) return false;   // 32-bit tile origins and k offsets in the kernels
    return true;
}

// Small tiles, or the large kernel?  What an SM does per chunk of 32 elements of K decides: CTAs on the fullest SM times the time
// of one, plus the latency of a chunk when there are few.  In units of a 16 x 16 tile's chunk (about 0.45 us), measured on one to
// eighteen CTAs per SM at K = 1024 and 256: 8 x 16 tiles 0.6, 32 x 32 tiles `mid`, tiles of the large kernel `large` (two to an SM;
// one that is alone takes 16 % longer) and 17 us for its decode pass and two more launches (F = 13: 7).  Small against large in us,
// on both sides of the line, K = 1024: Ampere FP16 512 x 512 75 / 124, 768 x 768 142 / 126, 1024 x 1536 370 / 297; CDNA3 FP16
// 768 x 768 150 / 166, 1024 x 1536 394 / 404, 2048 x 2048 - / 889; CDNA3 E4M3 768 x 768 188 / 161.
DirectSize direct_size(const DevModel& m, const GemmArgs& g, double* us) {
    const int kind = kind_of(m);
    if (!kind || g.dot_mode || m.literal_emax) return DIRECT_NONE;
    if ((kind == KIND_TR || kind == KIND_E) && g.k_chunk) return DIRECT_NONE;
    if (g.M > 65535ll * 8 || g.N > 0x7FFFFFFFll - 128) return DIRECT_NONE;                                 // grid.y, 32-bit columns
    // The kernels count the bytes left in a row, and the chunks, in 32 bits; TR-FDPA of the wide formats tags exponents with the chunk's
    // number in 21 bits.
    const int64_t row = g.K * (fmt_desc(m.fmt_a).storage_bits / 8);
    const bool tagged = m.family == FAM_TR && (m.fmt_a == EF_BF16 || m.fmt_a == EF_TF32);
    if (row > 0x7FFFFFFFll - 1024 || (tagged && g.K > (int64_t(1) << 21) * fast::KC - 256)) return DIRECT_NONE;
    constexpr int64_t SMS = 148;
    auto fullest = [&](int bm, int bn) { return double((((g.M + bm - 1) / bm) * ((g.N + bn - 1) / bn) + SMS - 1) / SMS); };
    const bool f13 = kind == 1 + fast::EK_LUT8 && m.F == 13, bits8 = kind == 1 + fast::EK_LUT8;
    const double mid = bits8 ? 2.1 : (kind == KIND_E ? 2.3 : (kind == KIND_TR ? (m.family == FAM_GTR ? 3.05 : 2.4) : (m.L <= 4 ? 3.2 : 2.3)));
    const double large = f13 ? 13.5 : (bits8 ? 5.0 : (kind == KIND_E ? 7.6 : (kind == KIND_TR ? (m.family == FAM_GTR ? 8.3 : 8.7) :
                         (m.L <= 4 ? 10.1 : (kind == 1 + fast::EK_F16 ? (m.acc == ACC_F16 ? 7.8 : 6.3) : 7.3)))));
    const double c8 = 0.5 + 0.6 * fullest(8, 16), c16 = 0.6 + fullest(16, 16), c32 = 0.6 + mid * fullest(32, 32);
    const double chunks = double((g.K + fast::KC - 1) / fast::KC);
    double big = 1e30;
    if (fast_tfdpa_supported(m, g)) {
        const double n = f13 ? fullest(fast::BM, m.acc != ACC_F16 && !g.k_chunk ? 128 : fast::BN) : fullest(64, 64);
        big = large * (f13 || int64_t(n) % 2 == 0 ? n : n + 0.16 / n) + (f13 ? 15.0 : 38.0) / chunks;
    }
    if (us) *us = 3.0 + 0.45 * chunks * std::min(std::min(c8, c16), std::min(c32, big));
    if (big <= c8 && big <= c16 && big <= c32) return DIRECT_NONE;
    return c8 <= c16 && c8 <= c32 ? DIRECT_8x16 : (c16 <= c32 ? DIRECT_16x16 : DIRECT_32x32);
}

int launch_direct(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t stream) {
    cudaError_t err = cudaErrorInvalidValue;
    const int kind = kind_of(m);
    if (kind == KIND_TR) {
        set_kernel_name(m.family == FAM_GTR ? "gtrfdpa" : "trfdpa", "small_tiles");
        err = direct::launch_tr(m, g, size, stream);
    } else if (kind == KIND_E) {
        set_kernel_name("efdpa", "small_tiles");
        err = direct::launch_e(m, g, size, stream);
    } else switch (kind - 1) {
        case fast::EK_LUT8: set_kernel_name("tfdpa_lut8", "small_tiles"); err = direct::launch_lut8(m, g, size, stream); break;
        case fast::EK_F16: set_kernel_name("tfdpa_f16", "small_tiles"); err = direct::launch_f16(m, g, size, stream); break;
        case fast::EK_BF16: set_kernel_name("tfdpa_bf16", "small_tiles"); err = direct::launch_bf16(m, g, size, stream); break;
        case fast::EK_TF32: set_kernel_name("tfdpa_tf32", "small_tiles"); err = direct::launch_tf32(m, g, size, stream); break;
        default: break;
    }
    if (err != cudaSuccess) {
        set_error("small-tile FDPA kernel launch failed: %s", cudaGetErrorString(err));
        return MMASIM_ERR_CUDA;
    }
    return MMASIM_OK;
}

// The counter of bulk-copy timeouts: one word per device in a device variable of the library (nothing is allocated).
namespace {
__device__ unsigned int g_copy_timeouts_word = 0u;
std::mutex g_counter_mutex;
unsigned int* g_counter_ptr[64] = {};
}  // namespace

unsigned int* copy_timeout_counter() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
    std::lock_guard<std::mutex> lock(g_counter_mutex);
    if (!g_counter_ptr[dev]) {
        void* p = nullptr;
        if (cudaGetSymbolAddress(&p, g_copy_timeouts_word) != cudaSuccess) return nullptr;
        g_counter_ptr[dev] = static_cast<unsigned int*>(p);
    }
    return g_counter_ptr[dev];
}

int launch_gemm_noalloc(const DevModel& m, const GemmArgs& g, cudaStream_t stream) {
    if (!fast::noalloc_supported(m) || !fast_tfdpa_supported(m, g)) {
        set_error("mmasim_gemm_noalloc serves the FP8 models with F = 13 (Ada and Hopper FP8 rows), K a multiple of 32 and "
                  "16-byte row strides; this call needs another kernel");
        return MMASIM_ERR_UNSUPPORTED;
    }
    const size_t need = fast::noalloc_need(m, g), cap = fast::noalloc_capacity();
    if (need > cap) {
        set_error("mmasim_gemm_noalloc: this problem needs %zu bytes of scratch, the fixed array holds %zu "
                  "(about (ceil(M/128) + ceil(N/128)) * K/32 * 27 KiB); use mmasim_gemm_ex", need, cap);
        return MMASIM_ERR_SHAPE;
    }
    set_kernel_name("tfdpa_lut8_noalloc", "large_tiles");
    const cudaError_t err = fast::launch_noalloc(m, g, stream);
    if (err != cudaSuccess) {
        set_error("mmasim_gemm_noalloc: %s", cudaGetErrorString(err));
        return MMASIM_ERR_CUDA;
    }
    return MMASIM_OK;
}

int launch_fast_tfdpa(const DevModel& m, const GemmArgs& g, cudaStream_t stream) {
    cudaError_t err = cudaErrorInvalidValue;
    if (kind_of(m) == KIND_TR) {
        set_kernel_name(m.family == FAM_GTR ? "gtrfdpa" : "trfdpa", "large_tiles");
        err = fast::launch_tr(m, g, stream);
    } else if (kind_of(m) == KIND_E) {
        set_kernel_name("efdpa", "large_tiles");
        err = fast::launch_e(m, g, stream);
    } else switch (kind_of(m) - 1) {
        case fast::EK_LUT8: set_kernel_name("tfdpa_lut8", "large_tiles"); err = fast::launch_lut8(m, g, stream); break;
        case fast::EK_F16: set_kernel_name("tfdpa_f16", "large_tiles"); err = fast::launch_f16(m, g, stream); break;
        case fast::EK_BF16: set_kernel_name("tfdpa_bf16", "large_tiles"); err = fast::launch_bf16(m, g, stream); break;
        case fast::EK_TF32: set_kernel_name("tfdpa_tf32", "large_tiles"); err = fast::launch_tf32(m, g, stream); break;
        default: break;
    }
    if (err != cudaSuccess) {
        set_error("tuned T-FDPA kernel launch failed: %s", cudaGetErrorString(err));
        return MMASIM_ERR_CUDA;
    }
    return MMASIM_OK;
}

}  // namespace mmasim
