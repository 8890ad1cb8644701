// C ABI of libmmasim: argument validation, model objects, dispatch to the kernels.
#include <atomic>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include "mmasim_internal.h"

namespace mmasim {

static thread_local char g_error[512] = "";
static thread_local const char *g_kernel = "", *g_variant = "";     // (string literals)

void set_error(const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_error, sizeof(g_error), fmt, ap);
    va_end(ap);
}
void set_kernel_name(const char* name, const char* variant) { g_kernel = name; g_variant = variant; }

namespace {

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

bool ranges_meet(const void* p, size_t p_bytes, const void* q, size_t q_bytes) {
    const uintptr_t a = reinterpret_cast<uintptr_t>(p), b = reinterpret_cast<uintptr_t>(q);
    return p_bytes && q_bytes && a < b + q_bytes && b < a + p_bytes;
}

// MMASIM_OK if p is device-accessible memory; ERR_INVALID_ARG for plain host memory; ERR_CUDA otherwise.
int check_device_ptr(const void* p, const char* name) {
    cudaPointerAttributes attr;
    const cudaError_t err = cudaPointerGetAttributes(&attr, p);
    if (err != cudaSuccess) {
        cudaGetLastError();
        set_error("cudaPointerGetAttributes(%s) failed: %s", name, cudaGetErrorString(err));
        return MMASIM_ERR_CUDA;
    }
    if (attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged) return MMASIM_OK;
    set_error("%s is not a device pointer", name);
    return MMASIM_ERR_INVALID_ARG;
}

// Shape rules shared by gemm and dot_batch.  Returns MMASIM_OK or an error status.
int check_k(const DevModel& m, int64_t K) {
    if (K < 1) { set_error("K must be >= 1"); return MMASIM_ERR_SHAPE; }
    if (m.family == FAM_FMA) return MMASIM_OK;
    if (m.family == FAM_FTZ) {
        if (K % m.P) { set_error("K = %lld is not a multiple of P = %d", (long long)K, m.P); return MMASIM_ERR_SHAPE; }
        return MMASIM_OK;
    }
    const int64_t L = K < m.L ? K : m.L;
    if (K % L) {
        set_error("K = %lld is not a multiple of L = min(K, L_max) = %lld", (long long)K, (long long)L);
        return MMASIM_ERR_SHAPE;
    }
    if (m.family == FAM_GST && (L % 32)) { set_error("GST-FDPA models need K to be a multiple of 32"); return MMASIM_ERR_SHAPE; }
    if (m.family == FAM_GTR && (L % 2)) { set_error("GTR-FDPA models need an even K"); return MMASIM_ERR_SHAPE; }
    if (m.family == FAM_ST && K > 32 && (K % 32)) { set_error("ST-FDPA models need K to be a multiple of 32"); return MMASIM_ERR_SHAPE; }
    return MMASIM_OK;
}

// `whole`: the product that g is a row panel of, if it is one: its size decides on the tiles (panels run beside each other).  `small`: on
// small tiles, whatever direct_size says.
int dispatch(const mmasim_model* model, const GemmArgs& g, int flags, cudaStream_t stream, const GemmArgs* whole, bool small) {
    const DevModel& m = model->dev;
    if (!(flags & MMASIM_GEMM_FORCE_GENERIC) && !m.literal_emax) {
        if (!(flags & MMASIM_GEMM_LARGE_TILES) && umma_supported(m, g)) return launch_umma(m, g, stream);
        if (small) return launch_direct(m, g, small_size(m, whole ? *whole : g), stream);
        const DirectSize size = (flags & MMASIM_GEMM_LARGE_TILES) && fast_tfdpa_supported(m, g) ? DIRECT_NONE : direct_size(m, whole ? *whole : g);
        if (size != DIRECT_NONE) return launch_direct(m, g, size, stream);
        if (fast_tfdpa_supported(m, g)) return launch_fast_tfdpa(m, g, stream);
        if (fast_fp_supported(m, g)) return launch_fast_fp(m, g, stream);
        if (fast_gst_supported(m, g)) return launch_fast_gst(m, g, stream);
    }
    set_kernel_name("generic", "generic");
    return launch_generic(m, g, stream);
}
int run_gemm(const mmasim_model* model, const GemmArgs& g, int flags, cudaStream_t stream, const GemmArgs* whole = nullptr, bool small = false) {
    const int st = dispatch(model, g, flags, stream, whole, small);
    if (st == MMASIM_ERR_CUDA) cudaGetLastError();      // (an allocation that failed is this call's error, not the next launch's)
    return st;
}

int build_args(const mmasim_model* model, int64_t M, int64_t N, int64_t K, const void* A, const void* B,
               const void* C, void* D, const mmasim_gemm_opts* opts, GemmArgs* out) {
    if (!model) { set_error("model is NULL"); return MMASIM_ERR_INVALID_ARG; }
    if (!A || !B || !D) { set_error("A, B and D must not be NULL"); return MMASIM_ERR_INVALID_ARG; }
    if (M < 1 || N < 1) { set_error("M and N must be >= 1"); return MMASIM_ERR_SHAPE; }
    const DevModel& m = model->dev;
    int st = check_k(m, K);
    if (st != MMASIM_OK) return st;
    GemmArgs g;
    std::memset(&g, 0, sizeof(g));
    g.M = M; g.N = N; g.K = K;
    g.A = A; g.B = B; g.C = C; g.D = D;
    g.lda = g.ldb = K;
    g.ldc = g.ldd = N;
    g.copy_timeouts = copy_timeout_counter();
    if (m.k_block) g.ld_sfa = g.ld_sfb = (K + m.k_block - 1) / m.k_block;
    if (opts) {
        if (opts->lda) g.lda = opts->lda;
        if (opts->ldb) g.ldb = opts->ldb;
        if (opts->ldc) g.ldc = opts->ldc;
        if (opts->ldd) g.ldd = opts->ldd;
        g.sfa = static_cast<const uint8_t*>(opts->sfa);
        g.sfb = static_cast<const uint8_t*>(opts->sfb);
        g.k_chunk = opts->k_chunk;
        g.row_scale = opts->row_scale;
        g.col_scale = opts->col_scale;
    }
    if (g.lda < K || g.ldb < K || g.ldc < N || g.ldd < N) { set_error("leading dimension smaller than the row length"); return MMASIM_ERR_SHAPE; }
    if (m.packed4 && ((g.lda | g.ldb | K) & 1)) { set_error("packed FP4 operands need even K and leading dimensions"); return MMASIM_ERR_SHAPE; }
    if (m.k_block && (!g.sfa || !g.sfb)) { set_error("this model needs scale factors (opts->sfa, opts->sfb)"); return MMASIM_ERR_INVALID_ARG; }
    if (!m.k_block && (g.sfa || g.sfb)) { set_error("this model takes no scale factors"); return MMASIM_ERR_INVALID_ARG; }
    const bool fdpa32 = m.family != FAM_FMA && m.family != FAM_FTZ && m.acc == ACC_F32;
    if (g.k_chunk) {
        if (!fdpa32) { set_error("k_chunk needs an FDPA model with an FP32 accumulator"); return MMASIM_ERR_UNSUPPORTED; }
        const int64_t L = K < m.L ? K : m.L;
        if (g.k_chunk < 0 || g.k_chunk % L || K % g.k_chunk) { set_error("k_chunk must be a multiple of L that divides K"); return MMASIM_ERR_SHAPE; }
    }
    if ((g.row_scale != nullptr) != (g.col_scale != nullptr)) { set_error("row_scale and col_scale must be given together"); return MMASIM_ERR_INVALID_ARG; }
    if (g.row_scale && !fdpa32) { set_error("dequantisation scales need an FDPA model with an FP32 accumulator"); return MMASIM_ERR_UNSUPPORTED; }
    *out = g;
    return MMASIM_OK;
}

}  // namespace

namespace {
// Device memory the library takes for itself (the staging buffers of mmasim_gemm_host, the decoded operand blocks of
// the tuned kernels): one memory pool per device, the library's own (the device's default pool and its attributes are
// the caller's and stay untouched), created on first use, keeping up to 1 GiB between calls.
constexpr int MAX_DEVICES = 64;
std::mutex g_pool_mutex;
cudaMemPool_t g_pools[MAX_DEVICES] = {};

}  // namespace

cudaError_t scratch_pool(cudaMemPool_t* out) {
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_pool_mutex);
    if (!g_pools[dev]) {
        cudaMemPoolProps props;
        std::memset(&props, 0, sizeof(props));
        props.allocType = cudaMemAllocationTypePinned;
        props.handleTypes = cudaMemHandleTypeNone;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t pool = nullptr;
        err = cudaMemPoolCreate(&pool, &props);
        if (err != cudaSuccess) return err;
        unsigned long long keep = 1ull << 30;
        err = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        // a buffer that another stream will free must not make this stream wait for it: row panels run beside each other
        int no = 0;
        if (err == cudaSuccess) err = cudaMemPoolSetAttribute(pool, cudaMemPoolReuseAllowInternalDependencies, &no);
        if (err != cudaSuccess) { cudaMemPoolDestroy(pool); return err; }
        g_pools[dev] = pool;
    }
    *out = g_pools[dev];
    return cudaSuccess;
}

cudaError_t take_scratch(const GemmArgs& g, size_t bytes, cudaStream_t stream, void** out) {
    *out = g.scratch;
    if (g.scratch && bytes <= g.scratch_bytes) return cudaSuccess;
    cudaMemPool_t pool = nullptr;
    const cudaError_t err = scratch_pool(&pool);
    return err != cudaSuccess ? err : cudaMallocFromPoolAsync(out, bytes, pool, stream);
}
cudaError_t give_scratch(const GemmArgs& g, void* scratch, cudaStream_t stream) {
    return scratch == g.scratch ? cudaSuccess : cudaFreeAsync(scratch, stream);
}

namespace {
// The streams and events of one mmasim_gemm_host call (mmasim_deviation_stats uses only the memory), and a word of mapped host memory
// that its kernels count given-up waits in (a copy of the device's counter before and after each call cost 15 us).  Creating them took about 100 us of every call, so up to
// LANES_KEPT sets per device wait for the next one; a call has its set to itself, and mmasim_host_release destroys those that wait.
struct HostLane {
    static constexpr int PANELS = 6;        // (with the streams of the copies eight: more would share the hardware's eight queues)
    int device = -1;
    cudaStream_t in = nullptr, out = nullptr, k[PANELS] = {};
    cudaEvent_t ev_in[PANELS] = {}, ev_k[PANELS] = {};
    unsigned int* gave_up = nullptr;        // host address
    unsigned int* gave_up_dev = nullptr;    // device address
    double* stats = nullptr;                // eight doubles behind it (mmasim_deviation_stats)
};
constexpr int LANES_KEPT = 4;
std::atomic<unsigned int> g_host_timeouts[MAX_DEVICES];     // what the words of finished calls held
std::mutex g_lane_mutex;
HostLane g_lanes[MAX_DEVICES][LANES_KEPT];       // the first g_lane_count of a device (plain arrays: nothing here may throw)
int g_lane_count[MAX_DEVICES] = {};

void destroy_lane(HostLane& l) {
    for (int p = 0; p < HostLane::PANELS; ++p) {
        if (l.ev_in[p]) cudaEventDestroy(l.ev_in[p]);
        if (l.ev_k[p]) cudaEventDestroy(l.ev_k[p]);
        if (l.k[p]) cudaStreamDestroy(l.k[p]);
    }
    if (l.in) cudaStreamDestroy(l.in);
    if (l.out) cudaStreamDestroy(l.out);
    if (l.gave_up) cudaFreeHost(l.gave_up);
    l = HostLane();
}
cudaError_t take_lane(HostLane* out) {
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(g_lane_mutex);
        if (g_lane_count[dev]) { *out = g_lanes[dev][--g_lane_count[dev]]; return cudaSuccess; }
    }
    HostLane l;
    l.device = dev;
    err = cudaHostAlloc(reinterpret_cast<void**>(&l.gave_up), 128, cudaHostAllocMapped);
    if (err == cudaSuccess) err = cudaHostGetDevicePointer(reinterpret_cast<void**>(&l.gave_up_dev), l.gave_up, 0);
    if (err == cudaSuccess) l.stats = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(l.gave_up) + 64);
    if (err == cudaSuccess) err = cudaStreamCreateWithFlags(&l.in, cudaStreamNonBlocking);
    if (err == cudaSuccess) err = cudaStreamCreateWithFlags(&l.out, cudaStreamNonBlocking);
    for (int p = 0; p < HostLane::PANELS && err == cudaSuccess; ++p) {
        err = cudaStreamCreateWithFlags(&l.k[p], cudaStreamNonBlocking);
        if (err == cudaSuccess) err = cudaEventCreateWithFlags(&l.ev_in[p], cudaEventDisableTiming);
        if (err == cudaSuccess) err = cudaEventCreateWithFlags(&l.ev_k[p], cudaEventDisableTiming);
    }
    if (err != cudaSuccess) destroy_lane(l);
    *out = l;
    return err;
}
void give_lane(HostLane& l, bool sound) {
    if (l.device < 0) return;
    if (sound) {
        std::lock_guard<std::mutex> lock(g_lane_mutex);
        if (g_lane_count[l.device] < LANES_KEPT) { g_lanes[l.device][g_lane_count[l.device]++] = l; return; }
    }
    destroy_lane(l);
}
}  // namespace

int given_up_waits(int st, unsigned int count, int device, const char* call) {
    if (count && device >= 0 && device < MAX_DEVICES) g_host_timeouts[device] += count;
    if (!count || st != MMASIM_OK) return st;
    set_error("%s: %u CTAs gave up waiting for a bulk copy and stored nothing", call, count);
    return MMASIM_ERR_TIMEOUT;
}

}  // namespace mmasim

using namespace mmasim;

extern "C" {

mmasim_model* mmasim_create_model_ex(int arch, int a_fmt, int b_fmt, int acc_fmt, const mmasim_overrides* ov) {
    mmasim_model tmp;
    const char* why = "";
    if (!registry_lookup(arch, a_fmt, b_fmt, acc_fmt, &tmp, &why)) {
        set_error("mmasim_create_model: %s (arch %d, input %d x %d, accumulator %d)", why, arch, a_fmt, b_fmt, acc_fmt);
        return nullptr;
    }
    if (ov) {
        DevModel& d = tmp.dev;
        const bool fdpa = d.family == FAM_T || d.family == FAM_ST || d.family == FAM_TR || d.family == FAM_GTR;
        if ((ov->l_max >= 0 || ov->F >= 0 || ov->F2 >= 0 || ov->rho >= 0 || ov->inner_round >= 0) && !fdpa) {
            set_error("overrides apply to T-, ST-, TR- and GTR-FDPA models only");
            return nullptr;
        }
        if (ov->l_max >= 0) {
            if (ov->l_max < 1 || ov->l_max > 64 || (d.family == FAM_GTR && (ov->l_max & 1)) || (d.family == FAM_ST && ov->l_max != 32)) {
                set_error("l_max override out of range"); return nullptr;
            }
            d.L = ov->l_max;
        }
        if (ov->F >= 0) { if (ov->F > 30 || ov->F < 1) { set_error("F override must be in 1..30"); return nullptr; } d.F = ov->F; }
        if (ov->F2 >= 0) { if (d.F2 == 0 || ov->F2 > 36) { set_error("F2 override not applicable"); return nullptr; } d.F2 = ov->F2; }
        if (d.F2 && d.F2 < d.F) { set_error("F2 must be >= F"); return nullptr; }
        if (ov->rho >= 0) {
            const bool fp16 = d.acc == ACC_F16;
            const bool ok = fp16 ? ov->rho == MMASIM_RNE_FP16 : (ov->rho >= MMASIM_RZ_FP32 && ov->rho <= MMASIM_RNE_FP32);
            if (!ok) { set_error("rho override does not match the accumulator type"); return nullptr; }
            d.rho = ov->rho;
        }
        if (ov->inner_round >= 0) {
            if (ov->inner_round > 1 || d.family != FAM_TR) { set_error("inner_round applies to TR-FDPA models only"); return nullptr; }
            d.inner_round = ov->inner_round;
        }
        if (ov->literal_emax > 0) {
            if (!fdpa && d.family != FAM_GST) { set_error("literal_emax applies to T-, ST-, GST-, TR- and GTR-FDPA models only"); return nullptr; }
            d.literal_emax = 1;
        }
        tmp.info.l_max = d.L; tmp.info.F = d.F; tmp.info.F2 = d.F2; tmp.info.rho = d.rho; tmp.info.inner_round = d.inner_round;
    }
    mmasim_model* m = new (std::nothrow) mmasim_model(tmp);
    if (!m) set_error("out of host memory");
    return m;
}

mmasim_model* mmasim_create_model(int arch, int in_fmt, int acc_fmt) {
    return mmasim_create_model_ex(arch, in_fmt, in_fmt, acc_fmt, nullptr);
}

void mmasim_destroy_model(mmasim_model* model) { delete model; }

int mmasim_model_info(const mmasim_model* model, mmasim_info* out) {
    if (!model || !out) { set_error("mmasim_model_info: NULL argument"); return MMASIM_ERR_INVALID_ARG; }
    *out = model->info;
    return MMASIM_OK;
}

int mmasim_gemm_ex(const mmasim_model* model, int64_t M, int64_t N, int64_t K, const void* A, const void* B,
                   const void* C, void* D, const mmasim_gemm_opts* opts, void* stream) {
    GemmArgs g;
    int st = build_args(model, M, N, K, A, B, C, D, opts, &g);
    if (st != MMASIM_OK) return st;
    if (!aligned16(A) || !aligned16(B) || !aligned16(D) || (C && !aligned16(C))) {
        set_error("A, B, C and D must be 16-byte aligned");
        return MMASIM_ERR_ALIGN;
    }
    if ((st = check_device_ptr(A, "A")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(B, "B")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(D, "D")) != MMASIM_OK) return st;
    if (C && (st = check_device_ptr(C, "C")) != MMASIM_OK) return st;
    if (g.sfa && (st = check_device_ptr(g.sfa, "opts->sfa")) != MMASIM_OK) return st;
    if (g.sfb && (st = check_device_ptr(g.sfb, "opts->sfb")) != MMASIM_OK) return st;
    if (g.row_scale && (st = check_device_ptr(g.row_scale, "opts->row_scale")) != MMASIM_OK) return st;
    if (g.col_scale && (st = check_device_ptr(g.col_scale, "opts->col_scale")) != MMASIM_OK) return st;
    return run_gemm(model, g, opts ? opts->flags : 0, static_cast<cudaStream_t>(stream));
}

int mmasim_gemm_noalloc(const mmasim_model* model, int64_t M, int64_t N, int64_t K, const void* A, const void* B,
                        const void* C, void* D, const mmasim_gemm_opts* opts, void* stream) {
    GemmArgs g;
    int st = build_args(model, M, N, K, A, B, C, D, opts, &g);
    if (st != MMASIM_OK) return st;
    if (!aligned16(A) || !aligned16(B) || !aligned16(D) || (C && !aligned16(C))) {
        set_error("A, B, C and D must be 16-byte aligned");
        return MMASIM_ERR_ALIGN;
    }
    if ((st = check_device_ptr(A, "A")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(B, "B")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(D, "D")) != MMASIM_OK) return st;
    if (C && (st = check_device_ptr(C, "C")) != MMASIM_OK) return st;
    if (g.row_scale && (st = check_device_ptr(g.row_scale, "opts->row_scale")) != MMASIM_OK) return st;
    if (g.col_scale && (st = check_device_ptr(g.col_scale, "opts->col_scale")) != MMASIM_OK) return st;
    return launch_gemm_noalloc(model->dev, g, static_cast<cudaStream_t>(stream));
}

int mmasim_gemm(const mmasim_model* model, int64_t M, int64_t N, int64_t K, const void* A, const void* B,
                const void* C, void* D, void* stream) {
    return mmasim_gemm_ex(model, M, N, K, A, B, C, D, nullptr, stream);
}

int mmasim_dot_batch(const mmasim_model* model, int64_t n, int64_t K, const void* A, const void* B,
                     const void* C, void* D, void* stream) {
    if (!model) { set_error("model is NULL"); return MMASIM_ERR_INVALID_ARG; }
    if (!A || !B || !D) { set_error("A, B and D must not be NULL"); return MMASIM_ERR_INVALID_ARG; }
    if (n < 1) { set_error("n must be >= 1"); return MMASIM_ERR_SHAPE; }
    const DevModel& m = model->dev;
    if (m.k_block) { set_error("mmasim_dot_batch supports unscaled models only"); return MMASIM_ERR_UNSUPPORTED; }
    int st = check_k(m, K);
    if (st != MMASIM_OK) return st;
    if (!aligned16(A) || !aligned16(B) || !aligned16(D) || (C && !aligned16(C))) {
        set_error("A, B, C and D must be 16-byte aligned");
        return MMASIM_ERR_ALIGN;
    }
    if ((st = check_device_ptr(A, "A")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(B, "B")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(D, "D")) != MMASIM_OK) return st;
    if (C && (st = check_device_ptr(C, "C")) != MMASIM_OK) return st;
    GemmArgs g;
    std::memset(&g, 0, sizeof(g));
    g.M = n; g.N = 1; g.K = K;
    g.A = A; g.B = B; g.C = C; g.D = D;
    g.lda = g.ldb = K;
    g.ldc = g.ldd = 1;
    g.dot_mode = 1;
    if (!m.literal_emax && dot_stream_supported(m, g)) return launch_dot_stream(m, g, static_cast<cudaStream_t>(stream));
    set_kernel_name("generic_dot", "generic");
    return launch_generic(m, g, static_cast<cudaStream_t>(stream));
}

int mmasim_gemm_host(const mmasim_model* model, int64_t M, int64_t N, int64_t K, const void* A, const void* B,
                     const void* C, void* D, const mmasim_gemm_opts* opts) {
    GemmArgs g;
    int st = build_args(model, M, N, K, A, B, C, D, opts, &g);
    if (st != MMASIM_OK) return st;
    const mmasim_info& info = model->info;
    const size_t a_bytes = size_t((M - 1) * g.lda + K) * info.a_bits / 8;
    const size_t b_bytes = size_t((N - 1) * g.ldb + K) * info.b_bits / 8;
    const size_t c_bytes = g.C ? size_t((M - 1) * g.ldc + N) * info.acc_bytes : 0;
    const size_t d_bytes = size_t((M - 1) * g.ldd + N) * info.acc_bytes;
    const size_t sfa_bytes = g.sfa ? size_t(M * g.ld_sfa) : 0, sfb_bytes = g.sfb ? size_t(N * g.ld_sfb) : 0;
    // Row panels of D (outputs are independent, Section 3.1 Step 1): B once, then per panel its rows of A and C in, the kernel, its rows
    // of D out, so that copies in, arithmetic and copies out run beside each other.  A panel is whole CTA tiles and, with its copies,
    // about 3 MB (55 us of the bus, against some 10 us that its calls cost), at most six; every panel has a stream of its own, because
    // one alone does not fill the SMs.  Large tiles want 512 rows: every one walks all of K, and the last panel's come last.
    // In us, one panel / several: Ampere BF16 1475 x 1214 x 1072 890 / 675, 1477 x 1229 x 144 283 / 256, 1216 x 1306 x 624 604 / 430,
    // Hopper E4M3 2048 x 2048 x 2048 1460 / 1130 (384 rows: 1215).
    const int flags = opts ? opts->flags : 0;
    const bool large_tiles = fast_tfdpa_supported(model->dev, g) && !umma_supported(model->dev, g) && direct_size(model->dev, g) == DIRECT_NONE;
    int panels = int((a_bytes + c_bytes + d_bytes) / (size_t(3) << 20));
    panels = panels < 1 || M < 512 ? 1 : (panels > HostLane::PANELS ? HostLane::PANELS : panels);
    // D over an operand that later panels still read: everything goes in before anything comes out.  (C in place is fine: a panel's rows of
    // D replace its own rows of C.)
    const bool in_place = g.C == g.D && g.ldc == g.ldd;
    if (ranges_meet(D, d_bytes, A, a_bytes) || ranges_meet(D, d_bytes, g.sfa, sfa_bytes) || (!in_place && ranges_meet(D, d_bytes, C, c_bytes))) panels = 1;
    const int64_t rows_by_bytes = panels > 1 ? ((M + panels - 1) / panels + 127) / 128 * 128 : M;
    int64_t panel_rows = large_tiles && panels > 1 && rows_by_bytes < 512 ? 512 : rows_by_bytes;
    bool small_tiles = false;
    if (large_tiles && !(flags & (MMASIM_GEMM_LARGE_TILES | MMASIM_GEMM_FORCE_GENERIC))) {
        const int64_t n = (M + panel_rows - 1) / panel_rows;
        small_tiles = !panels_on_large_tiles(model->dev, g, n, M - (n - 1) * panel_rows);
        if (small_tiles) panel_rows = rows_by_bytes;
    }
    panels = int((M + panel_rows - 1) / panel_rows);
    HostLane lane;
    cudaError_t err = take_lane(&lane);
    cudaMemPool_t pool = nullptr;
    if (err == cudaSuccess) err = scratch_pool(&pool);
    // One allocation, stream-ordered out of the library's own pool (which keeps up to 1 GiB between calls), the scratch of the panels in it:
    // blocks that went back on the panels' streams made every later allocation look at them (a call of 128 x 128 x 64 took 51 us, 68 behind a
    // product in six panels).
    auto up256 = [](size_t x) { return (x + 255) / 256 * 256; };
    const size_t sizes[8] = {a_bytes, b_bytes, c_bytes, d_bytes, sfa_bytes, sfb_bytes, g.row_scale ? size_t(M) * 4 : 0, g.col_scale ? size_t(N) * 4 : 0};
    size_t total = 0, scratch_at[HostLane::PANELS + 1];
    for (size_t x : sizes) total += up256(x);
    for (int p = 0; p <= panels; ++p) {
        scratch_at[p] = total;
        if (p == panels || (flags & MMASIM_GEMM_FORCE_GENERIC)) continue;
        GemmArgs q = g;
        q.M = p + 1 < panels ? panel_rows : M - p * panel_rows;
        if (!(flags & MMASIM_GEMM_LARGE_TILES) && umma_supported(model->dev, q)) total += up256(umma_scratch(model->dev, q));
        else if (large_tiles && !small_tiles) total += up256(fast_tfdpa_scratch(model->dev, q));
    }
    unsigned char* base = nullptr;
    if (err == cudaSuccess) {
        err = cudaMallocFromPoolAsync(reinterpret_cast<void**>(&base), total, pool, lane.in);
        if (err == cudaErrorMemoryAllocation && total > scratch_at[0]) {  // the panels see for themselves, one after the other
            cudaGetLastError();
            for (size_t& x : scratch_at) x = scratch_at[0];
            err = cudaMallocFromPoolAsync(reinterpret_cast<void**>(&base), scratch_at[0], pool, lane.in);
        }
    }
    unsigned char* at[8];
    size_t off = 0;
    for (int i = 0; i < 8; ++i) { at[i] = sizes[i] ? base + off : nullptr; off += up256(sizes[i]); }
    unsigned char *dA = at[0], *dB = at[1], *dC = at[2], *dD = at[3], *dSA = at[4], *dSB = at[5], *dRS = at[6], *dCS = at[7];
    auto h2d = [&](void* dst, const void* src, size_t at_byte, size_t bytes) {
        if (err != cudaSuccess || !src || !bytes) return;
        err = cudaMemcpyAsync(static_cast<unsigned char*>(dst) + at_byte, static_cast<const unsigned char*>(src) + at_byte, bytes, cudaMemcpyHostToDevice, lane.in);
    };
    if (err == cudaSuccess) { *lane.gave_up = 0u; g.copy_timeouts = lane.gave_up_dev; }
    h2d(dB, B, 0, b_bytes);
    h2d(dSB, g.sfb, 0, sfb_bytes);
    h2d(dRS, g.row_scale, 0, size_t(M) * 4);
    h2d(dCS, g.col_scale, 0, size_t(N) * 4);
    const GemmArgs host = g;
    // A copy into pageable memory holds the calling thread until it is done: those wait until every panel is queued.  (Behind each panel they
    // put the panels in a row, one alone on the GPU after the other: Hopper E4M3 2048 x 2048 x 2048 on numpy arrays 4.9 ms, now 2.7; in one
    // panel 3.7.  Ampere BF16 1475 x 1214 x 1088 2.4, now 1.4; in one panel 2.1.)
    cudaPointerAttributes d_attr;
    bool pinned_out = false;
    if (err == cudaSuccess) {
        if (cudaPointerGetAttributes(&d_attr, D) == cudaSuccess) pinned_out = d_attr.type != cudaMemoryTypeUnregistered;
        else cudaGetLastError();
    }
    auto copy_out = [&](int p) {
        const int64_t r0 = p * panel_rows, rows = (r0 + panel_rows <= M ? panel_rows : M - r0);
        const size_t off = size_t(r0 * host.ldd) * info.acc_bytes, pitch = size_t(host.ldd) * info.acc_bytes, width = size_t(N) * info.acc_bytes;
        const cudaStream_t so = panels > 1 ? lane.out : lane.in;
        if (panels > 1) err = cudaStreamWaitEvent(so, lane.ev_k[p], 0);
        if (err != cudaSuccess) return;
        // only the N words of every row go back: with ldd > N the words between the rows of the caller's D are not the library's
        if (host.ldd == N) err = cudaMemcpyAsync(static_cast<unsigned char*>(D) + off, dD + off, width * size_t(rows), cudaMemcpyDeviceToHost, so);
        else err = cudaMemcpy2DAsync(static_cast<unsigned char*>(D) + off, pitch, dD + off, pitch, width, size_t(rows), cudaMemcpyDeviceToHost, so);
    };
    for (int p = 0; p < panels && err == cudaSuccess && st == MMASIM_OK; ++p) {
        const int64_t r0 = p * panel_rows, rows = (r0 + panel_rows <= M ? panel_rows : M - r0);
        // byte ranges of the panel's rows (a row of packed 4-bit elements starts on a byte: leading dimensions are even)
        const size_t a_off = size_t(r0 * host.lda) * info.a_bits / 8, a_len = size_t((rows - 1) * host.lda + K) * info.a_bits / 8;
        const size_t c_off = size_t(r0 * host.ldc) * info.acc_bytes, c_len = size_t((rows - 1) * host.ldc + N) * info.acc_bytes;
        const size_t d_off = size_t(r0 * host.ldd) * info.acc_bytes;
        h2d(dA, A, a_off, a_len);
        h2d(dC, C, c_off, c_len);
        h2d(dSA, host.sfa, size_t(r0 * host.ld_sfa), host.sfa ? size_t(rows * host.ld_sfa) : 0);
        if (err != cudaSuccess) break;
        const cudaStream_t sk = panels > 1 ? lane.k[p] : lane.in;
        if (panels > 1) {
            err = cudaEventRecord(lane.ev_in[p], lane.in);
            if (err == cudaSuccess) err = cudaStreamWaitEvent(sk, lane.ev_in[p], 0);
            if (err != cudaSuccess) break;
        }
        GemmArgs q = host;
        q.M = rows;
        q.A = dA + a_off;
        q.B = dB;
        q.C = dC ? dC + c_off : nullptr;
        q.D = dD + d_off;
        q.sfa = dSA ? dSA + r0 * host.ld_sfa : nullptr;
        q.sfb = dSB;
        q.row_scale = dRS ? reinterpret_cast<const float*>(dRS) + r0 : nullptr;
        q.col_scale = reinterpret_cast<const float*>(dCS);
        q.scratch = scratch_at[p + 1] > scratch_at[p] ? base + scratch_at[p] : nullptr;
        q.scratch_bytes = scratch_at[p + 1] - scratch_at[p];
        st = run_gemm(model, q, flags, sk, &host, small_tiles);
        if (st != MMASIM_OK) break;
        if (panels > 1) {
            err = cudaEventRecord(lane.ev_k[p], sk);
            if (err != cudaSuccess) break;
        }
        if (pinned_out) copy_out(p);
    }
    for (int p = 0; p < panels && !pinned_out && err == cudaSuccess && st == MMASIM_OK; ++p) copy_out(p);
    // everything drains, then the buffers go back to the pool in the order of the stream they came from
    bool sound = err == cudaSuccess;
    if (lane.in) {
        for (int p = 0; p < panels && panels > 1; ++p) { const cudaError_t e = cudaStreamSynchronize(lane.k[p]); if (err == cudaSuccess) err = e; }
        if (panels > 1) { const cudaError_t e = cudaStreamSynchronize(lane.out); if (err == cudaSuccess) err = e; }
        if (base) cudaFreeAsync(base, lane.in);
        const cudaError_t e = cudaStreamSynchronize(lane.in);
        if (err == cudaSuccess) err = e;
    }
    const int device = lane.device;
    const unsigned int count = err == cudaSuccess ? *static_cast<volatile unsigned int*>(lane.gave_up) : 0u;
    give_lane(lane, sound && err == cudaSuccess);
    if (err != cudaSuccess) {
        cudaGetLastError();
        set_error("mmasim_gemm_host: %s", cudaGetErrorString(err));
        return MMASIM_ERR_CUDA;
    }
    return given_up_waits(st, count, device, "mmasim_gemm_host");
}

int mmasim_int_peak(int kind, int64_t blocks, int64_t iters, void* sink, int32_t* ops_per_round, void* stream) {
    if (!sink || !ops_per_round || blocks < 1 || iters < 1 || kind < 0) { set_error("mmasim_int_peak: bad argument"); return MMASIM_ERR_INVALID_ARG; }
    const int st = check_device_ptr(sink, "sink");
    if (st != MMASIM_OK) return st;
    return launch_int_peak(kind, blocks, iters, sink, ops_per_round, static_cast<cudaStream_t>(stream));
}

int mmasim_hw_mma(int kind, int64_t M, int64_t K, const void* A, const void* B, const void* C, void* D, void* stream) {
    if (!A || !B || !D) { set_error("mmasim_hw_mma: A, B and D must not be NULL"); return MMASIM_ERR_INVALID_ARG; }
    int st;
    if ((st = check_device_ptr(A, "A")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(B, "B")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(D, "D")) != MMASIM_OK) return st;
    if (C && (st = check_device_ptr(C, "C")) != MMASIM_OK) return st;
    return launch_hw_mma(kind, M, K, A, B, C, D, static_cast<cudaStream_t>(stream));
}

int mmasim_hw_umma(int kind, int64_t M, int64_t K, const void* A, const void* B, const void* C, void* D, const void* sfa,
                   const void* sfb, int32_t* status, void* stream) {
    if (!A || !B || !D || !status) { set_error("mmasim_hw_umma: A, B, D and status must not be NULL"); return MMASIM_ERR_INVALID_ARG; }
    int st;
    if ((st = check_device_ptr(A, "A")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(B, "B")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(D, "D")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(status, "status")) != MMASIM_OK) return st;
    if (C && (st = check_device_ptr(C, "C")) != MMASIM_OK) return st;
    if (sfa && (st = check_device_ptr(sfa, "sfa")) != MMASIM_OK) return st;
    if (sfb && (st = check_device_ptr(sfb, "sfb")) != MMASIM_OK) return st;
    if (!aligned16(A) || !aligned16(B)) { set_error("mmasim_hw_umma: A and B must be 16-byte aligned"); return MMASIM_ERR_ALIGN; }
    return launch_hw_umma(kind, M, K, A, B, C, D, sfa, sfb, status, static_cast<cudaStream_t>(stream));
}

int mmasim_error_stats(int acc_fmt, int64_t n, const void* D, const double* ref, double* stats, void* stream) {
    if (!D || !ref || !stats || n < 1) { set_error("mmasim_error_stats: bad argument"); return MMASIM_ERR_INVALID_ARG; }
    int st;
    if ((st = check_device_ptr(D, "D")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(ref, "ref")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(stats, "stats")) != MMASIM_OK) return st;
    return launch_error_stats(acc_fmt == MMASIM_ACC_F16 ? ACC_F16 : (acc_fmt == MMASIM_ACC_F32 ? ACC_F32 : -1), n, D, ref, stats,
                              static_cast<cudaStream_t>(stream));
}

namespace {
bool has_reference(const DevModel& m) {
    const int f = m.fmt_a;
    return f == m.fmt_b && (f == EF_F16 || f == EF_BF16 || f == EF_TF32 || f == EF_F32 || f == EF_E4M3 || f == EF_E5M2) && !m.k_block && m.acc != ACC_F64;
}
}  // namespace

// One call, kernels one behind the other and nothing else in the stream: the operands widened, the product, and the FP64 reference, which
// is compared where it is computed (see launch_deviation_end).  CDNA3 FP16, 1024 x 1024 x 256: 169 us as five calls from Python, 149 us
// as one of five kernels, a memset and a copy, now 138.
int mmasim_deviation_stats(const mmasim_model* model, int64_t M, int64_t N, int64_t K, const void* A, const void* B, const void* C,
                           double* stats, void* stream) {
    GemmArgs g;
    int st = build_args(model, M, N, K, A, B, C, stats, nullptr, &g);
    if (st != MMASIM_OK) return st;
    const DevModel& m = model->dev;
    if (!has_reference(m)) {
        set_error("mmasim_deviation_stats: unscaled models of FP32, TF32, BF16, FP16 and FP8 inputs of one type");
        return MMASIM_ERR_UNSUPPORTED;
    }
    if (!aligned16(A) || !aligned16(B) || (C && !aligned16(C))) { set_error("A, B and C must be 16-byte aligned"); return MMASIM_ERR_ALIGN; }
    if ((st = check_device_ptr(A, "A")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(B, "B")) != MMASIM_OK) return st;
    if (C && (st = check_device_ptr(C, "C")) != MMASIM_OK) return st;
    const cudaStream_t s = static_cast<cudaStream_t>(stream);
    HostLane lane;
    cudaError_t err = take_lane(&lane);
    cudaMemPool_t pool = nullptr;
    if (err == cudaSuccess) err = scratch_pool(&pool);
    const size_t d_bytes = (size_t(M) * size_t(N) * model->info.acc_bytes + 255) / 256 * 256;
    unsigned char* base = nullptr;
    if (err == cudaSuccess) err = cudaMallocFromPoolAsync(reinterpret_cast<void**>(&base), d_bytes + deviation_scratch(M, N, K), pool, s);
    if (err == cudaSuccess) {
        *lane.gave_up = 0u;
        g.copy_timeouts = lane.gave_up_dev;
        st = launch_deviation_start(m.fmt_a, M, N, K, A, B, base + d_bytes, s);
        g.D = base;
        if (st == MMASIM_OK) st = run_gemm(model, g, 0, s);
        if (st == MMASIM_OK) st = launch_deviation_end(m.acc, M, N, K, C, g.D, base + d_bytes, reinterpret_cast<double*>(lane.gave_up_dev) + 8, s);
    }
    if (st == MMASIM_ERR_CUDA) cudaGetLastError();
    if (base) cudaFreeAsync(base, s);
    const cudaError_t e = cudaStreamSynchronize(s);
    if (err == cudaSuccess) err = e;
    const int device = lane.device;
    const unsigned int count = err == cudaSuccess ? *static_cast<volatile unsigned int*>(lane.gave_up) : 0u;
    if (err == cudaSuccess && st == MMASIM_OK && !count) std::memcpy(stats, lane.stats, 64);
    give_lane(lane, err == cudaSuccess);
    if (err != cudaSuccess) {
        cudaGetLastError();
        set_error("mmasim_deviation_stats: %s", cudaGetErrorString(err));
        return MMASIM_ERR_CUDA;
    }
    return given_up_waits(st, count, device, "mmasim_deviation_stats");
}

int mmasim_reference_fp64(const mmasim_model* model, int64_t M, int64_t N, int64_t K, const void* A, const void* B, const void* C,
                          double* ref, void* stream) {
    GemmArgs g;
    int st = build_args(model, M, N, K, A, B, C, ref, nullptr, &g);
    if (st != MMASIM_OK) return st;
    const DevModel& m = model->dev;
    if (!has_reference(m)) {
        set_error("mmasim_reference_fp64: unscaled models of FP32, TF32, BF16, FP16 and FP8 inputs of one type");
        return MMASIM_ERR_UNSUPPORTED;
    }
    if ((st = check_device_ptr(A, "A")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(B, "B")) != MMASIM_OK) return st;
    if ((st = check_device_ptr(ref, "ref")) != MMASIM_OK) return st;
    if (C && (st = check_device_ptr(C, "C")) != MMASIM_OK) return st;
    st = launch_reference_fp64(m.fmt_a, m.acc, M, N, K, A, B, C, ref, static_cast<cudaStream_t>(stream));
    if (st == MMASIM_ERR_CUDA) cudaGetLastError();
    return st;
}

int mmasim_host_release(void) {
    {
        std::lock_guard<std::mutex> lanes(g_lane_mutex);
        int current = 0;
        const bool known = cudaGetDevice(&current) == cudaSuccess;
        for (int d = 0; d < MAX_DEVICES; ++d) {
            if (g_lane_count[d]) cudaSetDevice(d);
            while (g_lane_count[d]) destroy_lane(g_lanes[d][--g_lane_count[d]]);
        }
        if (known) cudaSetDevice(current);
    }
    std::lock_guard<std::mutex> lock(g_pool_mutex);
    cudaError_t err = cudaSuccess;
    for (int d = 0; d < MAX_DEVICES; ++d)
        if (g_pools[d]) {
            const cudaError_t e = cudaMemPoolDestroy(g_pools[d]);
            if (err == cudaSuccess) err = e;
            g_pools[d] = nullptr;
        }
    if (err != cudaSuccess) {
        cudaGetLastError();
        set_error("mmasim_host_release: %s", cudaGetErrorString(err));
        return MMASIM_ERR_CUDA;
    }
    return MMASIM_OK;
}

const char* mmasim_last_kernel(void) { return g_kernel; }
const char* mmasim_last_variant(void) { return g_variant; }

int mmasim_copy_timeouts(uint64_t* count) {
    if (!count) { set_error("count is NULL"); return MMASIM_ERR_INVALID_ARG; }
    unsigned int* p = copy_timeout_counter();
    unsigned int v = 0u;
    int dev = 0;
    cudaError_t err = p ? cudaMemcpy(&v, p, sizeof(v), cudaMemcpyDeviceToHost) : cudaErrorUnknown;
    if (err == cudaSuccess) err = cudaGetDevice(&dev);
    if (err != cudaSuccess) { set_error("mmasim_copy_timeouts: %s", cudaGetErrorString(err)); return MMASIM_ERR_CUDA; }
    *count = v + (dev < MAX_DEVICES ? g_host_timeouts[dev].load() : 0u);
    return MMASIM_OK;
}
const char* mmasim_last_error(void) { return g_error; }

}  // extern "C"
