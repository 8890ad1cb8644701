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

// Rows that are no whole number of chunks or start off 16 bytes.
static bool ragged(const DevModel& m, const GemmArgs& g) {
    const int bytes = fmt_desc(m.fmt_a).storage_bits / 8;
    return g.K % fast::KC || (g.lda * bytes) % 16 || (g.ldb * bytes) % 16;
}

// Whether the small-tile kernels take the call at all.
static bool direct_takes(const DevModel& m, const GemmArgs& g) {
    const int kind = kind_of(m);
    if (!kind || g.dot_mode || m.literal_emax) return false;
    if ((kind == KIND_TR || kind == KIND_E) && g.k_chunk) return false;
    if (g.M > 65535ll * 8 || g.N > 0x7FFFFFFFll - 128) return false;                                       // grid.y, 32-bit columns
    // The kernels count the bytes left in a row, and the chunks, in 32 bits; TR-FDPA of the wide formats tags exponents with the chunk's
    // number in 21 bits.
    const int64_t row = g.K * (fmt_desc(m.fmt_a).storage_bits / 8);
    const bool tagged = m.family == FAM_TR && (m.fmt_a == EF_BF16 || m.fmt_a == EF_TF32);
    return row <= 0x7FFFFFFFll - 1024 && !(tagged && g.K > (int64_t(1) << 21) * fast::KC - 256);
}

bool fast_tfdpa_supported(const DevModel& m, const GemmArgs& g) {
    const int kind = kind_of(m);
    if (!kind || g.dot_mode || m.literal_emax) return false;
    if (g.K % m.L || (m.family == FAM_ST && g.K % fast::KC)) return false;   // (ragged chunks are filled up with whole blocks of zeros)
    if (ragged(m, g) && !direct_takes(m, g)) return false;                  // (what they fall back on where there is no memory for scratch)
    if (g.k_chunk % fast::KC) return false;
    if ((kind == KIND_TR || kind == KIND_E) && g.k_chunk) return false;
    if (m.F == 13 && g.M > 65535ll * fast::BM) return false;                // grid.y
    if (g.N > 0x7FFFFFFFll - 128 || g.K > 0x7FFFFFFFll - 64) return false;   // 32-bit tile origins and k offsets in the kernels
    return true;
}

// Small tiles, or the large kernel?  What the fullest SM does decides.  In us, with `chunks` of 32 elements of K and n CTAs on that SM:
//     small tiles   4 + chain chunks + per_tile n (chunks + 1.2)        8 x 16 outputs: 0.65 of a 16 x 16 tile
//     large tiles   decode + large n (chunks + 0.5)                     (an odd n: the last tile has the SM to itself, 0.16 of one more)
// with the constants of the arithmetic, fitted to the times of all four at sizes from 16 x 64 to 1076 x 3218 and K = 64, 256 and 1024
// (within 10 %); those of the FP8 rows again after their staging and the F = 13 tiles had become faster.  Small / large in us on both
// sides of the line: Hopper E4M3 256 x 1024 x 1024 58 / 96, 768 x 768 x 256 35 / 33, Hopper E4M3 -> FP16 512 x 512 x 256 37 / 43, 256 x
// 1024 x 1024 130 / 133, Ampere FP16 768 x 768 x 256 36 / 38, 1024 x 1024 x 256 70 / 62, CDNA1 BF16 512 x 512 x 1024 129 / 211, 768 x
// 768 x 1024 258 / 215.
namespace {
struct TileCosts { double chain, t16, t32, large, decode; };
TileCosts tile_costs(const DevModel& m, int kind, bool promoted) {
    const bool h = m.acc == ACC_F16;
    if (kind == KIND_E) return m.fmt_a == EF_F16 ? TileCosts{0.26, 0.28, 0.89, 3.3, 15} : TileCosts{0.58, 0.50, 1.55, 5.3, 15};
    if (kind == KIND_TR) {
        if (m.family == FAM_GTR) return {0.19, 0.39, 1.17, 3.5, 15};
        if (m.fmt_a == EF_TF32) return {0.35, 0.46, 1.54, 5.8, 15};
        return {0.21, 0.35, 1.13, 3.85, 15};
    }
    if (kind == 1 + fast::EK_LUT8) {
        if (m.F != 13) return h ? TileCosts{0.37, 0.63, 1.96, 4.5, 15} : (m.family == FAM_ST ? TileCosts{0.26, 0.50, 1.15, 2.3, 15} : TileCosts{0.19, 0.44, 1.05, 2.2, 15});
        if (h) return m.L == 16 ? TileCosts{0.66, 0.56, 2.13, 5.5, 17} : TileCosts{0.37, 0.63, 1.96, 3.7, 17};
        // (large: times f13_chunk_us; promoted sums only have the smaller tiles)
        return m.L == 16 ? TileCosts{0.19, 0.32, 0.88, promoted ? 1.38 : 1.3, 22} : TileCosts{0.10, 0.38, 0.90, promoted ? 1.06 : 1.0, 22};
    }
    if (kind == 1 + fast::EK_F16 && h) return m.L == 4 ? TileCosts{0.46, 0.45, 1.83, 6.3, 15} : TileCosts{0.25, 0.36, 1.15, 3.75, 15};
    if (kind == 1 + fast::EK_TF32) return m.L == 4 ? TileCosts{0.27, 0.43, 1.32, 4.3, 15} : TileCosts{0.21, 0.35, 1.08, 3.1, 15};
    if (m.L == 4) return {0.28, 0.41, 1.29, 4.3, 15};
    if (m.L == 8) return kind == 1 + fast::EK_F16 ? TileCosts{0.18, 0.34, 1.01, 2.8, 15} : TileCosts{0.19, 0.34, 1.04, 3.2, 15};
    return {0.18, 0.32, 0.92, 2.3, 15};
}
}  // namespace

static DirectSize choose_size(const DevModel& m, const GemmArgs& g, bool large_too, double* us) {
    if (!direct_takes(m, g)) return DIRECT_NONE;
    const int kind = kind_of(m);
    constexpr int64_t SMS = 148;
    auto fullest = [&](int bm, int bn) { return double((((g.M + bm - 1) / bm) * ((g.N + bn - 1) / bn) + SMS - 1) / SMS); };
    const bool f13 = kind == 1 + fast::EK_LUT8 && m.F == 13;
    const TileCosts t = tile_costs(m, kind, g.k_chunk != 0);
    const double chunks = double((g.K + fast::KC - 1) / fast::KC), start = 4.0 + t.chain * chunks, each = chunks + 1.2;
    const double c8 = start + 0.65 * t.t16 * fullest(8, 16) * each, c16 = start + t.t16 * fullest(16, 16) * each, c32 = start + t.t32 * fullest(32, 32) * each;
    double big = 1e30;
    if (large_too && fast_tfdpa_supported(m, g)) {
        if (f13 && m.acc != ACC_F16) {
            const double low = fast::f13_chunk_us(g, 64), tall = fast::f13_chunk_us(g, 128);
            big = t.decode + t.large * (g.k_chunk || low < tall ? low : tall) * chunks;
        } else {
            const double n = f13 ? fullest(fast::BM, fast::BN) : fullest(64, 64);
            big = t.decode + t.large * (f13 || int64_t(n) % 2 == 0 ? n : n + 0.16 / n) * (f13 ? chunks : chunks + 0.5);
        }
    }
    if (us) *us = std::min(std::min(c8, c16), std::min(c32, big));
    if (big <= c8 && big <= c16 && big <= c32) return DIRECT_NONE;
    return c8 <= c16 && c8 <= c32 ? DIRECT_8x16 : (c16 <= c32 ? DIRECT_16x16 : DIRECT_32x32);
}

DirectSize direct_size(const DevModel& m, const GemmArgs& g, double* us) { return choose_size(m, g, true, us); }
DirectSize small_size(const DevModel& m, const GemmArgs& g) { return choose_size(m, g, false, nullptr); }

// Row panels whose copies and kernels overlap (mmasim_gemm_host) are not what the costs above were fitted to: large tiles end late where
// the last panel comes last, above all a short one, and where those of all panels do not fill the places for tiles (two on each of 148 SMs)
// some SMs get two and others none; and every panel decodes B.  So ragged products of the FP64 kernels, which the small tiles took before,
// have to gain by the costs: 1.15 times in several panels, 1.4 with a last one of less than two tiles or with places left, hardly in one
// panel or with one and a half times as many tiles as places.  (The F = 13 kernels were never slower than the costs say.)  Of 366 ragged
// products that the costs alone give to the large tiles 38 took over 3 % longer on them, by up to 1.32; of those that are left 13 do, by up to
// 1.21; and 12 of the others would have been over 3 % faster.  Large / small in us (ratio of the costs): Ampere FP16 1925 x 441 x 1576 (1.09)
// 584 / 448, Ampere BF16 1479 x 742 x 1800 (1.30, 288 tiles in three panels) 751 / 618, Ampere TF32 1998 x 454 x 1556 (1.09) 908 / 689; kept:
// CDNA3 E4M3 2471 x 880 x 688 (1.26, 546 tiles) 460 / 526, Ampere FP16 2138 x 2503 x 1016 (1360 tiles) 1246 / 1448.
bool panels_on_large_tiles(const DevModel& m, const GemmArgs& g, int64_t panels, int64_t last_rows) {
    if (!ragged(m, g) || m.F == 13) return true;
    double small = 0.0, large = 0.0;
    choose_size(m, g, false, &small);
    choose_size(m, g, true, &large);                   // (it chose the large ones)
    constexpr int64_t PLACES = 2 * 148;
    const int64_t tiles = ((g.M + 63) / 64) * ((g.N + 63) / 64);
    double gain = last_rows < 128 || tiles <= PLACES ? 1.4 : 1.15;
    if (panels == 1) gain = 1.02;
    if (2 * tiles > 3 * PLACES) gain = 1.04;
    return small > gain * large;
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
    if (!fast::noalloc_supported(m) || !fast_tfdpa_supported(m, g) || g.K % fast::KC || g.lda % 16 || g.ldb % 16) {
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

size_t fast_tfdpa_scratch(const DevModel& m, const GemmArgs& g) {
    auto tiles = [](int64_t rows, int64_t of) { return size_t((rows + of - 1) / of); };
    const size_t chunks = tiles(g.K, fast::KC);
    if (m.F != 13 || kind_of(m) != 1 + fast::EK_LUT8) return chunks * fast::BLK64_BYTES * (tiles(g.M, 64) + tiles(g.N, 64));
    return chunks * (tiles(g.M, fast::BM) * fast::blk_t_bytes(fast::BM) + std::max(tiles(g.N, 64) * fast::blk_t_bytes(64), tiles(g.N, 128) * fast::blk_t_bytes(128)));
}

// A stream whose work is being recorded into a graph.
static bool capturing(cudaStream_t stream) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(stream, &status) != cudaSuccess) { cudaGetLastError(); return false; }
    return status != cudaStreamCaptureStatusNone;
}

int launch_fast_tfdpa(const DevModel& m, const GemmArgs& g, cudaStream_t stream) {
    // Ragged rows run on the small tiles where the decoded operands get no memory, and in a graph: one with memory nodes in it cannot be
    // cloned, made part of another one or instantiated twice, and those of ragged calls never had any.  (Whole chunks on large tiles always did.)
    if (ragged(m, g) && capturing(stream)) return launch_direct(m, g, small_size(m, g), stream);
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
    if (err == cudaErrorMemoryAllocation && ragged(m, g)) {
        cudaGetLastError();
        return launch_direct(m, g, small_size(m, g), stream);
    }
    if (err != cudaSuccess) {
        set_error("tuned T-FDPA kernel launch failed: %s", cudaGetErrorString(err));
        return MMASIM_ERR_CUDA;
    }
    return MMASIM_OK;
}

}  // namespace mmasim
