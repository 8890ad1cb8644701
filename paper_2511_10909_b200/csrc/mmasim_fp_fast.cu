// Tuned kernels for the models that run on the floating-point pipes:
//   Phi_FMA (Algorithm 4): d <- fma(a_k, b_k, d) in ascending k, FP32 or FP64, IEEE-754 round-to-nearest-even (FP64: on
//   the FP64 matrix instruction, see fma64_mma_kernel)
//   Phi_FTZ-AddMul (Algorithm 2): FTZ-Mul products, pairwise FTZ-Add over groups of P, FTZ-Add into d
// Register-tiled like a classic SGEMM (CTA tile in shared memory, k-major, one micro-tile of accumulators per
// thread), except that the order of operations inside one output is fixed by the model, so there is no split-K and
// no reassociation: every accumulator walks K sequentially.
//
// FTZ-Add / FTZ-Mul use the hardware flush-to-zero mode (`add.rn.ftz.f32`, `mul.rn.ftz.f32`), which flushes
// subnormal results to a zero of the same sign, exactly the last line of Algorithm 1.  "Round, then flush" and the
// hardware's flush coincide here: products of two BF16 / FP16 values have at most 22 significant bits, and sums of
// two normal-or-zero FP32 values below 2^-125 are multiples of 2^-149, so no result is rounded across the 2^-126
// boundary.  Inputs are never subnormal (Algorithm 2 flushes A, B and C to +0 first; every intermediate is flushed).
//
// Any K and any row stride: the last chunk is filled up with -0 in A and +0 in B, whose products are -0, which every accumulator
// (a -0 too) takes without a change.  Tiles in two sizes; see use_small.
#include <cuda_fp16.h>
#include <algorithm>
#include "mmasim_stats.cuh"

namespace mmasim {
namespace {

constexpr int NT = 256;

enum FpMode : int { FP_FMA32 = 0, FP_FTZ_F16 = 2, FP_FTZ_BF16 = 3 };

template <int MODE> struct ModeTraits;
template <> struct ModeTraits<FP_FMA32> { static constexpr int TM = 8, TN = 8, IN_BYTES = 4; };
template <> struct ModeTraits<FP_FTZ_F16> { static constexpr int TM = 8, TN = 4, IN_BYTES = 2; };
template <> struct ModeTraits<FP_FTZ_BF16> { static constexpr int TM = 8, TN = 4, IN_BYTES = 2; };

__device__ __forceinline__ float add_ftz(float x, float y) {
    float z;
    asm("add.rn.ftz.f32 %0, %1, %2;" : "=f"(z) : "f"(x), "f"(y));
    return z;
}
__device__ __forceinline__ float mul_ftz(float x, float y) {
    float z;
    asm("mul.rn.ftz.f32 %0, %1, %2;" : "=f"(z) : "f"(x), "f"(y));
    return z;
}

// FlushSubnormal of Algorithm 2 followed by the exact conversion to FP32.
__device__ __forceinline__ float load_flushed(uint32_t w, bool bf16) {
    if (bf16) return ((w & 0x7F80u) == 0u && (w & 0x007Fu)) ? 0.0f : __uint_as_float(w << 16);
    return ((w & 0x7C00u) == 0u && (w & 0x03FFu)) ? 0.0f : __half2float(__ushort_as_half((unsigned short)w));
}

// TM x TN: outputs per thread; KC: elements of K per chunk; rows at any address (ROWS_ANY), on 16 bytes (ROWS_16), or on 16 bytes with K a
// multiple of a chunk (ROWS_WHOLE: without the tests for the end of K, 2 - 5 % faster).
enum Rows : int { ROWS_ANY = 0, ROWS_16, ROWS_WHOLE };
template <int MODE, int P, int TM, int TN, int KC, int ROWS>
__global__ void __launch_bounds__(NT, TM >= 8 ? 2 : 3) fp_kernel(GemmArgs g) {
    after_previous();
    using T = ModeTraits<MODE>;
    using in_t = float;
    using acc_t = float;
    constexpr int BM = 16 * TM, BN = 16 * TN;
    constexpr bool FTZ = MODE == FP_FTZ_F16 || MODE == FP_FTZ_BF16;
    constexpr int EPT = 16 / T::IN_BYTES;                   // elements per 16-byte load
    constexpr int TPR = KC / EPT;                           // loads per row per chunk
    static_assert(KC % EPT == 0 && (!FTZ || KC % P == 0), "chunk layout");
    __shared__ __align__(16) in_t As[KC][BM];
    __shared__ __align__(16) in_t Bs[KC][BN];

    const int tid = threadIdx.x;
    const int tx = tid % 16, ty = tid / 16;
    const int64_t row0 = int64_t(blockIdx.y) * BM, col0 = int64_t(blockIdx.x) * BN;
    // Columns of a thread's micro-tile: groups of V (one 16-byte shared load), 16 * V columns apart, so that the sixteen
    // threads of a row of the thread grid read 256 contiguous bytes per load (no bank conflicts).
    constexpr int V = 16 / int(sizeof(in_t));
    auto col_of = [&](int c) { return (c / V) * (16 * V) + tx * V + (c % V); };

    acc_t d[TM][TN];
#pragma unroll
    for (int r = 0; r < TM; ++r)
#pragma unroll
        for (int c = 0; c < TN; ++c) {
            const int64_t i = row0 + ty * TM + r, j = col0 + col_of(c);
            acc_t v = acc_t(0);
            if (g.C && i < g.M && j < g.N) {
                if (FTZ) {
                    const uint32_t w = static_cast<const uint32_t*>(g.C)[i * g.ldc + j];
                    v = ((w & 0x7F800000u) == 0u && (w & 0x007FFFFFu)) ? 0.0f : __uint_as_float(w);   // FlushSubnormal(C)
                } else {
                    v = static_cast<const acc_t*>(g.C)[i * g.ldc + j];
                }
            }
            d[r][c] = v;
        }

    // The raw 16-byte words of the next chunk are fetched while the current one is computed.
    constexpr int TASKS = (BM + BN) * TPR, PER_THREAD = (TASKS + NT - 1) / NT;
    uint4 raw[PER_THREAD];
    auto fetch = [&](int64_t k0) {
#pragma unroll
        for (int it = 0; it < PER_THREAD; ++it) {
            const int task = it * NT + tid;
            const bool is_a = task < BM * TPR;
            const int u = is_a ? task : task - BM * TPR;
            const int rows = is_a ? BM : BN;
            const int r = u % rows, h = u / rows;
            const int64_t grow = (is_a ? row0 : col0) + r;
            const uint32_t pad = is_a ? (T::IN_BYTES == 4 ? 0x80000000u : 0x80008000u) : 0u;
            raw[it] = make_uint4(pad, pad, pad, pad);
            const int64_t k = k0 + h * EPT;
            if (task >= TASKS || grow >= (is_a ? g.M : g.N) || (ROWS != ROWS_WHOLE && k >= g.K)) continue;
            const unsigned char* p = static_cast<const unsigned char*>(is_a ? g.A : g.B) + (grow * (is_a ? g.lda : g.ldb) + k) * T::IN_BYTES;
            if (ROWS == ROWS_WHOLE || (ROWS == ROWS_16 && k + EPT <= g.K)) raw[it] = *reinterpret_cast<const uint4*>(p);
            else {
                uint32_t w[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    w[q] = pad;
                    if (T::IN_BYTES == 4) { if (k + q < g.K) w[q] = reinterpret_cast<const uint32_t*>(p)[q]; }
                    else {
                        if (k + 2 * q < g.K) w[q] = (w[q] & 0xFFFF0000u) | reinterpret_cast<const uint16_t*>(p)[2 * q];
                        if (k + 2 * q + 1 < g.K) w[q] = (w[q] & 0x0000FFFFu) | uint32_t(reinterpret_cast<const uint16_t*>(p)[2 * q + 1]) << 16;
                    }
                }
                raw[it] = make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
    };
    fetch(0);
    for (int64_t k0 = 0; k0 < g.K; k0 += KC) {
        __syncthreads();
        // ---- stage: decode the fetched words, stored k-major ----
#pragma unroll
        for (int it = 0; it < PER_THREAD; ++it) {
            const int task = it * NT + tid;
            if (task >= TASKS) break;
            const bool is_a = task < BM * TPR;
            const int u = is_a ? task : task - BM * TPR;
            const int rows = is_a ? BM : BN;
            const int r = u % rows, h = u / rows;
            const uint32_t wv[4] = {raw[it].x, raw[it].y, raw[it].z, raw[it].w};
#pragma unroll
            for (int q = 0; q < EPT; ++q) {
                in_t v;
                if (MODE == FP_FMA32) v = in_t(__uint_as_float(wv[q]));
                else v = in_t(load_flushed((wv[q / 2] >> (16 * (q % 2))) & 0xFFFFu, MODE == FP_FTZ_BF16));
                if (is_a) As[h * EPT + q][r] = v; else Bs[h * EPT + q][r] = v;
            }
        }
        __syncthreads();
        if (k0 + KC < g.K) fetch(k0 + KC);

        if (!FTZ) {
            // fully unrolled: with a partial unroll the compiler rotates the accumulators through register moves
#pragma unroll 16
            for (int kk = 0; kk < KC; ++kk) {
                in_t a[TM], b[TN];
#pragma unroll
                for (int r = 0; r < TM; ++r) a[r] = As[kk][ty * TM + r];
#pragma unroll
                for (int c = 0; c < TN; ++c) b[c] = Bs[kk][col_of(c)];
#pragma unroll
                for (int r = 0; r < TM; ++r)
#pragma unroll
                    for (int c = 0; c < TN; ++c) d[r][c] = fma(a[r], b[c], d[r][c]);   // one rounding (fmaf for float)
            }
        } else {
#pragma unroll 1
            for (int kg = 0; kg < KC; kg += P) {
                float s[TM][TN], u[P == 4 ? TM : 1][P == 4 ? TN : 1];
#pragma unroll
                for (int l = 0; l < P; ++l) {
                    float a[TM], b[TN];
#pragma unroll
                    for (int r = 0; r < TM; ++r) a[r] = float(As[kg + l][ty * TM + r]);
#pragma unroll
                    for (int c = 0; c < TN; ++c) b[c] = float(Bs[kg + l][col_of(c)]);
#pragma unroll
                    for (int r = 0; r < TM; ++r)
#pragma unroll
                        for (int c = 0; c < TN; ++c) {
                            const float p = mul_ftz(a[r], b[c]);
                            if (l == 0) s[r][c] = p;
                            else if (l == 1) s[r][c] = add_ftz(s[r][c], p);
                            else if (l == 2) u[P == 4 ? r : 0][P == 4 ? c : 0] = p;
                            else u[P == 4 ? r : 0][P == 4 ? c : 0] = add_ftz(u[P == 4 ? r : 0][P == 4 ? c : 0], p);
                        }
                }
#pragma unroll
                for (int r = 0; r < TM; ++r)
#pragma unroll
                    for (int c = 0; c < TN; ++c) {
                        float t = s[r][c];
                        if (P == 4) t = add_ftz(t, u[P == 4 ? r : 0][P == 4 ? c : 0]);
                        d[r][c] = acc_t(add_ftz(float(d[r][c]), t));
                    }
            }
        }
    }

#pragma unroll
    for (int r = 0; r < TM; ++r)
#pragma unroll
        for (int c = 0; c < TN; ++c) {
            const int64_t i = row0 + ty * TM + r, j = col0 + col_of(c);
            if (i >= g.M || j >= g.N) continue;
            const acc_t v = d[r][c];
            uint32_t w = __float_as_uint(v);
            if (v != v) w = 0x7FC00000u;
            static_cast<uint32_t*>(g.D)[i * g.ldd + j] = w;
        }
}

// ---- Phi_FMA in FP64 on the FP64 matrix instruction ----
// `mma.sync.m8n8k4.f64` is, per output, the chain d <- fma(a_k, b_k, d) over its four k in ascending order, each step
// rounded to nearest even: Phi_FMA itself (Algorithm 4; the B200's instruction agrees with the model bit for bit on every
// input class of Section 3.2).  A warp owns 32 x 32 outputs (sixteen accumulator tiles), eight warps a 128 x 64 tile; the
// raw doubles of A and B reach shared memory by 16-byte asynchronous copies, three chunks of 16 k in flight, rows with
// a pitch of 20 doubles so that the fragment loads (lane (g, t) reads element (row 8 i + g, k 4 s + t)) are conflict-free.
namespace dm {
constexpr int DKC = 16, KP = DKC + 4, STAGES = 3;
template <int BM, int BN>
struct Stage {
    double a[BM][KP];
    double b[BN][KP];
};
}  // namespace dm

// WR x WC warps of TI x TJ accumulator tiles; UNIT: bytes per asynchronous copy (16, or 8 where a row stride or K is odd); TAIL: K is no
// multiple of a chunk (the test for it in every chunk cost 2048 x 2048 x 2048 684 instead of 620 us).
// OUT_STATS_*: C and the outputs compared with are FP32 or FP16 words, and what leaves are the sums of the deviations (see launch_deviation_end).
enum Out : int { OUT_WORDS = 0, OUT_STATS_32, OUT_STATS_16 };
template <int WR, int WC, int TI, int TJ, int UNIT, bool TAIL, int OUT>
__global__ void __launch_bounds__(32 * WR * WC, 2) fma64_mma_kernel(GemmArgs g, DeviationArgs s_out) {
    after_previous();
    using namespace dm;
    constexpr int BM = 8 * WR * TI, BN = 8 * WC * TJ, DNT = 32 * WR * WC, SEGS = DKC * 8 / UNIT, PER = UNIT / 8;
    using ST = Stage<BM, BN>;
    extern __shared__ __align__(16) unsigned char dm_smem[];
    ST* stages = reinterpret_cast<ST*>(dm_smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int wr = warp / WC, wc = warp % WC, gq = lane >> 2, tq = lane & 3;
    const int64_t row0 = int64_t(blockIdx.y) * BM, col0 = int64_t(blockIdx.x) * BN;
    const int NCH = TAIL ? int((g.K + DKC - 1) / DKC) : int(g.K / DKC), tail = int(g.K % DKC);

    double acc[TI][TJ][2];
#pragma unroll
    for (int i = 0; i < TI; ++i)
#pragma unroll
        for (int j = 0; j < TJ; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int64_t r = row0 + 8 * (wr * TI + i) + gq, c = col0 + 8 * (wc * TJ + j) + 2 * tq + e;
                acc[i][j][e] = 0.0;
                if (g.C && r < g.M && c < g.N)
                    acc[i][j][e] = OUT == OUT_WORDS ? static_cast<const double*>(g.C)[r * g.ldc + c] : stats::output_value<OUT == OUT_STATS_16>(g.C, r * g.ldc + c);
            }

    // one chunk: consecutive threads on consecutive segments of a row; rows and K beyond the matrix are filled with zeros (a
    // shorter copy, or none)
    auto issue = [&](int n) {
        ST& s = stages[n % STAGES];
#pragma unroll
        for (int it = 0; it < (BM + BN) * SEGS / DNT; ++it) {
            const int task = it * DNT + tid;
            const bool is_a = task < BM * SEGS;
            const int u = is_a ? task : task - BM * SEGS;
            const int r = u / SEGS, seg = u % SEGS;
            const int64_t grow = (is_a ? row0 : col0) + r, k = int64_t(n) * DKC + PER * seg;
            const bool inside = grow < (is_a ? g.M : g.N) && (!TAIL || k < g.K);      // (all of a copy is inside, or nothing)
            const double* base = static_cast<const double*>(is_a ? g.A : g.B);
            const double* src = inside ? base + grow * (is_a ? g.lda : g.ldb) + k : base;
            const uint32_t dst = uint32_t(__cvta_generic_to_shared(is_a ? &s.a[r][PER * seg] : &s.b[r][PER * seg]));
            if (UNIT == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(inside ? 16 : 0) : "memory");
            else asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(inside ? 8 : 0) : "memory");
        }
    };
    issue(0);
    asm volatile("cp.async.commit_group;" ::: "memory");
    if (NCH > 1) issue(1);
    asm volatile("cp.async.commit_group;" ::: "memory");

    for (int n = 0; n < NCH; ++n) {
        asm volatile("cp.async.wait_group 1;" ::: "memory");    // chunk n has landed (n + 1 may still be in flight)
        __syncthreads();                                        // ... for every thread, and everybody has left chunk n - 1
        if (n + 2 < NCH) issue(n + 2);                          // into the buffer of chunk n - 1
        asm volatile("cp.async.commit_group;" ::: "memory");
        const ST& s = stages[n % STAGES];
        const bool last = TAIL && tail && n == NCH - 1;
#pragma unroll
        for (int ks = 0; ks < DKC / 4; ++ks) {
            double af[TI], bf[TJ];
#pragma unroll
            for (int i = 0; i < TI; ++i) {
                af[i] = s.a[8 * (wr * TI + i) + gq][4 * ks + tq];
                if (last && 4 * ks + tq >= tail) af[i] = -0.0;
            }
#pragma unroll
            for (int j = 0; j < TJ; ++j) bf[j] = s.b[8 * (wc * TJ + j) + gq][4 * ks + tq];
#pragma unroll
            for (int i = 0; i < TI; ++i)
#pragma unroll
                for (int j = 0; j < TJ; ++j)
                    asm volatile("mma.sync.aligned.m8n8k4.row.col.rn.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
                                 : "+d"(acc[i][j][0]), "+d"(acc[i][j][1]) : "d"(af[i]), "d"(bf[j]));
        }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");

    if constexpr (OUT != OUT_WORDS) {
        stats::Deviations s;
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
            for (int j = 0; j < TJ; ++j)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const int64_t r = row0 + 8 * (wr * TI + i) + gq, c = col0 + 8 * (wc * TJ + j) + 2 * tq + e;
                    if (r < g.M && c < g.N) s.add(stats::output_value<OUT == OUT_STATS_16>(s_out.D, r * g.ldd + c), acc[i][j][e]);
                }
        s.reduce_to<WR * WC>(s_out.sums);
        if (tid < 32) {                                 // the CTA that finishes last writes the sums out
            __threadfence();
            __syncwarp();
            unsigned int before = 0u;
            if (lane == 0) before = atomicAdd(s_out.finished, 1u);
            before = __shfl_sync(0xFFFFFFFFu, before, 0);
            if (before + 1u == gridDim.x * gridDim.y && lane < stats::NSTAT) {
                __threadfence();
                s_out.host[lane] = __ldcg(s_out.sums + lane);
            }
        }
        return;
    }
#pragma unroll
    for (int i = 0; i < TI; ++i)
#pragma unroll
        for (int j = 0; j < TJ; ++j)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const int64_t r = row0 + 8 * (wr * TI + i) + gq, c = col0 + 8 * (wc * TJ + j) + 2 * tq + e;
                if (r >= g.M || c >= g.N) continue;
                const double v = acc[i][j][e];
                unsigned long long w = (unsigned long long)__double_as_longlong(v);
                if (v != v) w = 0x7FF8000000000000ull;
                static_cast<unsigned long long*>(g.D)[r * g.ldd + c] = w;
            }
}

int64_t up_div(int64_t x, int64_t y) { return (x + y - 1) / y; }

// Small tiles where the large ones leave SMs idle: the work on the fullest SM, in large tiles; a small tile is its share of the outputs
// times `overhead` (more operand traffic per output), and a few of them take 0.35 of a large tile however small (latency).  Large / small
// in us: FP32 512^3 77 / 27, 1024^3 149 / 156; FP64 512^3 54 / 17, 1024 x 1024 x 256 34 / 31; CDNA2 FP16 560 x 192 x 128 20 / 11.
bool use_small(const GemmArgs& g, int bm, int bn, int sm, int sn, double overhead) {
    const double large = double(up_div(up_div(g.M, bm) * up_div(g.N, bn), 148));
    const double share = double(sm * sn) / double(bm * bn), n = double(up_div(up_div(g.M, sm) * up_div(g.N, sn), 148));
    return std::max(n * share * overhead, 0.35) < large;
}

template <int WR, int WC, int TI, int TJ, int OUT>
cudaError_t launch_fma64_tile(const GemmArgs& g, const DeviationArgs& s, cudaStream_t stream) {
    constexpr int BM = 8 * WR * TI, BN = 8 * WC * TJ;
    constexpr size_t sh = sizeof(dm::Stage<BM, BN>) * dm::STAGES;
    auto kernel = (g.lda | g.ldb | g.K) & 1 ? fma64_mma_kernel<WR, WC, TI, TJ, 8, true, OUT>
                                            : (g.K % dm::DKC ? fma64_mma_kernel<WR, WC, TI, TJ, 16, true, OUT> : fma64_mma_kernel<WR, WC, TI, TJ, 16, false, OUT>);
    const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sh));
    if (err != cudaSuccess) return err;
    return enqueue(kernel, dim3(unsigned(up_div(g.N, BN)), unsigned(up_div(g.M, BM))), 32 * WR * WC, sh, stream, g, s);
}
cudaError_t launch_fma64_mma(const GemmArgs& g, cudaStream_t stream) {
    const bool small = use_small(g, 128, 64, 32, 32, 1.15);
    set_kernel_name("fma_f64", small ? "small_tiles" : "large_tiles");
    return small ? launch_fma64_tile<2, 2, 2, 2, OUT_WORDS>(g, DeviationArgs{}, stream) : launch_fma64_tile<4, 2, 4, 4, OUT_WORDS>(g, DeviationArgs{}, stream);
}
template <int OUT>
cudaError_t launch_deviations(const GemmArgs& g, const DeviationArgs& s, cudaStream_t stream) {
    return use_small(g, 128, 64, 32, 32, 1.15) ? launch_fma64_tile<2, 2, 2, 2, OUT>(g, s, stream) : launch_fma64_tile<4, 2, 4, 4, OUT>(g, s, stream);
}

template <int MODE, int P, int TM, int TN, int KC>
cudaError_t launch_fp_tile(const GemmArgs& g, cudaStream_t stream) {
    constexpr int B = ModeTraits<MODE>::IN_BYTES;
    const dim3 grid(unsigned(up_div(g.N, 16 * TN)), unsigned(up_div(g.M, 16 * TM)), 1);
    if ((g.lda * B) % 16 || (g.ldb * B) % 16) return enqueue(fp_kernel<MODE, P, TM, TN, KC, ROWS_ANY>, grid, NT, 0, stream, g);
    if (g.K % KC) return enqueue(fp_kernel<MODE, P, TM, TN, KC, ROWS_16>, grid, NT, 0, stream, g);
    return enqueue(fp_kernel<MODE, P, TM, TN, KC, ROWS_WHOLE>, grid, NT, 0, stream, g);
}
template <int MODE, int P>
cudaError_t launch_fp(const GemmArgs& g, cudaStream_t stream) {
    using T = ModeTraits<MODE>;
    const bool small = use_small(g, 16 * T::TM, 16 * T::TN, 32, 64, MODE == FP_FMA32 ? 2.1 : 1.6);
    set_kernel_name(MODE == FP_FMA32 ? "fma_f32" : "ftz_addmul", small ? "small_tiles" : "large_tiles");
    if (small) return launch_fp_tile<MODE, P, 2, 4, 32>(g, stream);
    return launch_fp_tile<MODE, P, T::TM, T::TN, 16>(g, stream);
}

}  // namespace

bool fast_fp_supported(const DevModel& m, const GemmArgs& g) {
    if (g.dot_mode || g.k_chunk || g.row_scale) return false;
    if (m.family != FAM_FMA && m.family != FAM_FTZ) return false;
    if (g.K > 0x7FFF0000ll || g.M > 65535ll * 32) return false;
    // K off the chunks, or rows off 16 bytes, in FP32: while few CTAs (of 16 x 16 outputs) share an SM the generic kernels are the faster ones;
    // they have one output per thread and wait for less at a time.  Here / there in us, K = 1000, at 1.1 and 2.4 CTAs per SM and odd
    // strides: FP32 51 / 35 and 52 / 45, FP16 68 / 56 and 68 / 76, BF16 in pairs 70 / 64 and 70 / 89; on 16 bytes: FP32 43 / 35 and
    // 43 / 45, FP16 0.4 per SM 47 / 41 and 1.1 48 / 56, BF16 in pairs 47 / 54.  (FP64 is faster here at any size: 25 / 35.)
    const int bytes = fmt_desc(m.fmt_a).storage_bits / 8;
    const bool on16 = (g.lda * bytes) % 16 == 0 && (g.ldb * bytes) % 16 == 0;
    if (m.acc == ACC_F64 || (on16 && g.K % 16 == 0)) return true;
    const int64_t per_sm = up_div(up_div(g.M, 16) * up_div(g.N, 16), 148);
    const int generic_up_to = m.family == FAM_FMA ? (on16 ? 2 : 3) : (on16 ? (m.P == 4 ? 1 : 0) : 2);
    return per_sm > generic_up_to;
}

cudaError_t launch_fma64_deviations(int acc, const GemmArgs& g, const DeviationArgs& s, cudaStream_t stream) {
    return acc == ACC_F16 ? launch_deviations<OUT_STATS_16>(g, s, stream) : launch_deviations<OUT_STATS_32>(g, s, stream);
}

int launch_fast_fp(const DevModel& m, const GemmArgs& g, cudaStream_t stream) {
    cudaError_t err;
    if (m.family == FAM_FMA) {
        err = m.acc == ACC_F64 ? launch_fma64_mma(g, stream) : launch_fp<FP_FMA32, 2>(g, stream);
    } else {
        if (m.fmt_a == EF_F16) err = launch_fp<FP_FTZ_F16, 4>(g, stream);
        else if (m.P == 4) err = launch_fp<FP_FTZ_BF16, 4>(g, stream);
        else err = launch_fp<FP_FTZ_BF16, 2>(g, stream);
    }
    if (err != cudaSuccess) {
        set_error("floating-point kernel launch failed: %s", cudaGetErrorString(err));
        return MMASIM_ERR_CUDA;
    }
    return MMASIM_OK;
}

}  // namespace mmasim
