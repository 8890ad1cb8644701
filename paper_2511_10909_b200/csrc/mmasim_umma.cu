// Rows whose arithmetic is that of the B200's own fifth-generation matrix instruction, as a GEMM on that instruction.
//
// Which rows.  One tcgen05.mma per block of the model, chained through the accumulator in tensor memory, IS Algorithm 5 with the
// block function of Algorithms 7 (L = 16 / 8 / 32, F = 25), 8 and 9: the Hopper, Blackwell and RTX Blackwell FP16, BF16 and TF32
// rows and the Blackwell FP8 / FP6 / FP4, MX, MXFP4 and NVFP4 rows.  NaNs, infinities, signed zeros, subnormal results, overflow
// and NaN scale factors included they agree bit for bit (tests/test_gpu_matrix_instruction.py, mmasim_hw_umma);
// MMASIM_GEMM_LARGE_TILES and MMASIM_GEMM_FORCE_GENERIC keep the emulation reachable.  A shorter last (or only) block is filled up
// with zeros, which have no exponent and add nothing.
//
// Where they do not agree.  To the instruction a zero accumulator has the exponent -126, to the model it has none: a block that starts
// from zero and whose products all lie below 2^-126 is truncated on a finer grid by the model.  FP16 and unscaled 8-bit products
// do not get there (nor do NVFP4's scales); for BF16, TF32 and the E8M0 scales a tile whose smallest exponents of a row of A and a row
// of B add up to less is flagged, and the emulating kernel runs over the flagged tiles after the product.
//
// Work decomposition.  A tile is 128 lanes x BN columns of tensor memory: the lanes are rows of B (so that a warp's 32 lanes are 32
// neighbouring words of a row of C and D), the columns rows of A; few rows of A make narrow tiles, not idle ones.  CTAs are
// persistent, one per SM.  One warp brings in 128 bytes of K per row and stage (tiled bulk copies, 128-byte swizzle, rows and K
// beyond the matrix filled with zeros), one issues the instructions, eight put the next tile's C into tensor memory while the
// instructions run and take D out of it.  Four warps bring the scale factors, 16 bytes per row at a time, through a ring in shared
// memory into tensor memory: a 32-bit word holds four consecutive ones of a row, row r in lane r mod 32 of every quarter and
// column r / 32.  (tcgen05.cp does the storing too, but in the queue of the instructions, 32 ns per 512 bytes, and wants the words
// laid out by a pass beforehand, 4 us and a launch.)  FP6 and FP4 codes of the 8-bit containers are packed into the
// instruction's 16-element chunks first.
//
// Every wait is bounded: a role whose wait runs out raises a flag that ends the others' waits, the copies in flight are waited
// for, nothing more is stored, and the CTA counts itself in the library's counter of given-up waits.
#include <type_traits>
#include "mmasim_tma.cuh"

namespace mmasim {
namespace {

using namespace tma;
constexpr int LANES = 128;
constexpr int EPI_WARPS = 8;            // warps 0 - 7: C in, D out; 8: copies; 9: instructions; scaled kinds: 10 - 13: scale factors
constexpr int SMS = 148;

enum MmaKind : int { MK_F16 = 0, MK_TF32, MK_F8, MK_MX8, MK_MXF4, MK_NVF4 };
__host__ __device__ constexpr int sf_per_step(int kind) { return kind == MK_MX8 ? 1 : (kind == MK_MXF4 ? 2 : (kind == MK_NVF4 ? 4 : 0)); }

template <int MK, int BN>
struct Layout {
    static constexpr int SF = sf_per_step(MK);          // scale words per row and stage, too: four steps of SF bytes
    static constexpr int SPC = SF ? 4 / SF : 1;         // stages per 16 bytes of scale factors of a row
    static constexpr int NTHREADS = 32 * (EPI_WARPS + 2 + (SF ? 4 : 0));
    static constexpr int NRB = (BN + 127) / 128;        // blocks of (up to) 128 rows on the column side
    static constexpr int STAGES = BN >= 256 ? 4 : (BN >= 128 ? 6 : 8);
    static constexpr int L_BYTES = LANES * KBYTES, Q_BYTES = BN * KBYTES;
    static constexpr int STAGE = L_BYTES + Q_BYTES, SF_ROWS = SF ? LANES + BN : 0;
    static constexpr int SF_RING = SF == 4 ? 4 : 3;     // 16 bytes of scale factors of every row, that many in flight or in use
    static constexpr int SMEM = STAGES * STAGE + SF_RING * 16 * SF_ROWS + 1024;        // (the stages start on a multiple of 1024 bytes)
    // tensor memory: two accumulators of BN columns (one where there is no room for two), then per stage SF groups of 4 columns
    // (lane side) and of 4 NRB (column side)
    static constexpr int SF_COLS = SF * 4 * (1 + NRB), ACCS = 2 * BN + STAGES * SF_COLS <= 512 ? 2 : 1, USED = ACCS * BN + STAGES * SF_COLS;
    static constexpr int COLS = USED <= 32 ? 32 : (USED <= 64 ? 64 : (USED <= 128 ? 128 : (USED <= 256 ? 256 : 512)));
    static_assert(USED <= 512, "tensor memory");
};

struct UmmaArgs {
    const void* C;
    void* D;
    int64_t R, Q;                       // rows of the lane side (N), rows of the column side (M)
    int64_t ldc, ldd;
    const float* scale_l;               // col_scale
    const float* scale_q;               // row_scale
    const uint8_t* sf_l;                // scale factors, nsf per row
    const uint8_t* sf_q;
    int nsf, sf_wide;                   // (sf_wide: bytes that every row starts on: 16, 4 or 1)
    int64_t tiles;
    int tiles_q;                        // tiles along the columns
    unsigned char* redo;                // guarded kinds: per tile, whether the emulation has to do it
    const int* least_l;                 // BF16, TF32: the smallest exponent of every row
    const int* least_q;
    int least_sf;                       // E8M0: smallest exponents of the elements of a row of A and B together, less both biases
    const unsigned char* codes_l;       // E8M0: the elements themselves, rows `pitch` bytes apart, `row_bytes` of each; bits of a word that are
    const unsigned char* codes_q;       // magnitudes
    int64_t pitch_l, pitch_q;
    int row_bytes;
    uint32_t magnitude_l, magnitude_q;
    int steps;                          // instructions per output
    uint32_t idesc;
    unsigned int* timeouts;
};

// K-major operand in the 128-byte swizzle: groups of eight rows 1024 bytes apart.
__device__ __forceinline__ uint64_t operand_desc(uint32_t addr) {
    return uint64_t((addr & 0x3FFFFu) >> 4) | (uint64_t(1) << 16) | (uint64_t(1024 >> 4) << 32) | (uint64_t(1) << 46) | (uint64_t(2) << 61);
}
// One lane of the (converged) warp issues; `lead` is its predicate, the operands are the same in all lanes.  (Issued by a lane that had
// branched off on its own, an instruction took about 200 clocks instead of 80.)
#define MMASIM_UMMA(KINDSTR)                                                                                              \
    asm volatile("{\n\t.reg .pred p, l;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 l, %5, 0;\n\t@l tcgen05.mma.cta_group::1.kind::" KINDSTR " [%0], %1, %2, %3, p;\n\t}" \
                 :: "r"(d), "l"(ld), "l"(qd), "r"(idesc), "r"(uint32_t(add)), "r"(lead) : "memory")
#define MMASIM_UMMA_SCALED(KINDSTR)                                                                                       \
    asm volatile("{\n\t.reg .pred p, l;\n\tsetp.ne.b32 p, %6, 0;\n\tsetp.ne.b32 l, %7, 0;\n\t@l tcgen05.mma.cta_group::1.kind::" KINDSTR " [%0], %1, %2, %3, [%4], [%5], p;\n\t}" \
                 :: "r"(d), "l"(ld), "l"(qd), "r"(idesc), "r"(sfl), "r"(sfq), "r"(uint32_t(add)), "r"(lead) : "memory")
template <int MK>
__device__ __forceinline__ void issue(uint32_t lead, uint32_t d, uint64_t ld, uint64_t qd, uint32_t idesc, uint32_t sfl, uint32_t sfq, bool add) {
    if (MK == MK_F16) MMASIM_UMMA("f16");
    else if (MK == MK_TF32) MMASIM_UMMA("tf32");
    else if (MK == MK_F8) MMASIM_UMMA("f8f6f4");
    else if (MK == MK_MX8) MMASIM_UMMA_SCALED("mxf8f6f4.block_scale.scale_vec::1X");
    else if (MK == MK_MXF4) MMASIM_UMMA_SCALED("mxf4.block_scale.scale_vec::2X");
    else MMASIM_UMMA_SCALED("mxf4nvf4.block_scale.scale_vec::4X");
}
__device__ __forceinline__ void commit(uint32_t lead, uint32_t bar) {
    asm volatile("{\n\t.reg .pred l;\n\tsetp.ne.b32 l, %1, 0;\n\t@l tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" :: "r"(bar), "r"(lead) : "memory");
}
#define MMASIM_R16(x) "r"(x[0]), "r"(x[1]), "r"(x[2]), "r"(x[3]), "r"(x[4]), "r"(x[5]), "r"(x[6]), "r"(x[7]), "r"(x[8]), "r"(x[9]), "r"(x[10]), "r"(x[11]), "r"(x[12]), "r"(x[13]), "r"(x[14]), "r"(x[15])
#define MMASIM_W16(x) "=r"(x[0]), "=r"(x[1]), "=r"(x[2]), "=r"(x[3]), "=r"(x[4]), "=r"(x[5]), "=r"(x[6]), "=r"(x[7]), "=r"(x[8]), "=r"(x[9]), "=r"(x[10]), "=r"(x[11]), "=r"(x[12]), "=r"(x[13]), "=r"(x[14]), "=r"(x[15])
__device__ __forceinline__ void tmem_st16(uint32_t addr, const uint32_t* x) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" :: "r"(addr), MMASIM_R16(x) : "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t* x) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];" : MMASIM_W16(x) : "r"(addr) : "memory");
}

// The smallest of sixteen E8M0 scale factors (four words, from block `k0` of a row on) by byte position, without those of blocks of zeros:
// their products have no exponent, and quantisers give such a block the smallest factor there is.  Looked at are only the factors below
// `small`, which comes back as the smallest one that counts: of two that are not below the first `small` neither flags anything, and a row
// needs its smallest alone.  Eight blocks at a time, their loads in flight together.  (MXFP8 1024 x 4096 x 4096, one block in twenty zero
// under the smallest factor: 3531 us with every tile flagged, 2870 on the emulation alone.)
template <int MK>
__device__ __noinline__ uint2 without_zero_blocks(const unsigned char* p, int row_bytes, uint32_t magnitude, int k0, uint4 w, uint32_t small) {
    constexpr int BYTES = MK == MK_MXF4 ? 16 : 32;
    uint32_t least = 0xFFFFFFFFu;
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
        const uint32_t e[2] = {h ? w.z : w.x, h ? w.w : w.y};
        uint32_t any[8];
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const int at = (k0 + 8 * h + b) * BYTES;
            any[b] = magnitude;
            if ((e[b / 4] >> (8 * (b % 4)) & 0xFFu) >= small) continue;
            any[b] = 0u;
            if (at + BYTES <= row_bytes) {
#pragma unroll
                for (int v = 0; v < BYTES; v += 16) { const uint4 x = *reinterpret_cast<const uint4*>(p + at + v); any[b] |= x.x | x.y | x.z | x.w; }
            } else
                for (int v = at; v < row_bytes; ++v) any[b] |= p[v];
        }
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const uint32_t factor = any[b] & magnitude ? e[b / 4] >> (8 * (b % 4)) & 0xFFu : 255u;
            small = min(small, factor);
            least = __vminu4(least, factor | 0xFFFFFF00u);
        }
    }
    return make_uint2(least, small);
}

#define MMASIM_R4(x, i) "r"(x[i]), "r"(x[i + 1]), "r"(x[i + 2]), "r"(x[i + 3])
// N words of a lane into neighbouring columns.
template <int N>
__device__ __forceinline__ void tmem_st(uint32_t addr, const uint32_t (&x)[N]) {
    static_assert(N == 4 || N == 8 || N == 16 || N == 32, "shapes of the instruction");
    if constexpr (N == 4) asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" :: "r"(addr), MMASIM_R4(x, 0) : "memory");
    else if constexpr (N == 8) asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" :: "r"(addr), MMASIM_R4(x, 0), MMASIM_R4(x, 4) : "memory");
    else {
#pragma unroll
        for (int i = 0; i < N; i += 16) tmem_st16(addr + i, x + i);
    }
}
__device__ __forceinline__ uint4 lds16(uint32_t addr) {
    uint4 x;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w) : "r"(addr) : "memory");
    return x;
}

// Words of C or D at p, p + step, ...: all of them inside the matrix (FULL), or those below `valid`.
template <typename W, int CH, bool FULL>
__device__ __forceinline__ void load_words(const W* p, int64_t step, int valid, uint32_t (&x)[CH]) {
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        x[c] = 0u;
        if (FULL || c < valid) x[c] = *p;
        p += step;
    }
}
template <typename W, int CH, bool FULL>
__device__ __forceinline__ void store_words(W* p, int64_t step, int valid, const uint32_t (&x)[CH]) {
#pragma unroll
    for (int c = 0; c < CH; ++c) {
        if (FULL || c < valid) *p = W(x[c]);
        p += step;
    }
}

template <int MK, int BN, bool ACC16>
__global__ void __launch_bounds__(Layout<MK, BN>::NTHREADS, 1) umma_kernel(const __grid_constant__ CUtensorMap map_l, const __grid_constant__ CUtensorMap map_q, const UmmaArgs g) {
    using LY = Layout<MK, BN>;
    using W = typename std::conditional<ACC16, uint16_t, uint32_t>::type;
    constexpr int STAGES = LY::STAGES, SF = LY::SF;
    extern __shared__ unsigned char smem_raw[];
    __shared__ __align__(8) unsigned long long bars[3 * STAGES + 4];
    __shared__ uint32_t tmem_base_s;
    __shared__ volatile int gave_up;
    __shared__ int least_s[4][2];
    const int tid = threadIdx.x, warp = __shfl_sync(0xFFFFFFFFu, tid >> 5, 0), lane = tid & 31;
    const uint32_t stage0 = (smem_u32(smem_raw) + 1023u) & ~1023u;
    const uint32_t bar_full = smem_u32(bars), bar_empty = bar_full + 8 * STAGES, bar_c = bar_empty + 8 * STAGES, bar_d = bar_c + 16, bar_sf = bar_d + 16;
    const int nst = (g.steps + 3) / 4;

    if (tid == 0) {
#pragma unroll
        for (int s = 0; s < STAGES; ++s) { mbar_init(bar_full + 8 * s, 1); mbar_init(bar_empty + 8 * s, 1); mbar_init(bar_sf + 8 * s, 4); }
#pragma unroll
        for (int b = 0; b < 2; ++b) { mbar_init(bar_c + 8 * b, EPI_WARPS); mbar_init(bar_d + 8 * b, 1); }
        gave_up = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == EPI_WARPS + 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" :: "r"(smem_u32(&tmem_base_s)), "r"(LY::COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    after_previous();
    const uint32_t tmem = __shfl_sync(0xFFFFFFFFu, tmem_base_s, 0);
    // about a second, and longer for a K whose instructions alone take that long
    const long long budget = 2000000000ll + 4000ll * nst;
    const uint32_t lead = elect_one();

    if (warp == EPI_WARPS) {                            // ---- the copies ----
        constexpr uint32_t BYTES = LY::STAGE;
        int s = 0, issued = 0;
        uint32_t phase = 1u;                            // (the first round finds every stage empty)
        bool ok = true;
        for (int64_t t = blockIdx.x; t < g.tiles && ok; t += gridDim.x) {
            const int tq = int(t % g.tiles_q), tl = int(t / g.tiles_q);
            for (int n = 0; n < nst; ++n) {
                ok = warp_wait(bar_empty + 8 * s, phase, &gave_up, budget);
                if (!ok) break;
                const uint32_t bar = bar_full + 8 * s, base = stage0 + s * LY::STAGE;
                if (lead) {
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(BYTES) : "memory");
                    tma_load(base, &map_l, n * KBYTES, tl * LANES, bar);
                    tma_load(base + LY::L_BYTES, &map_q, n * KBYTES, tq * BN, bar);
                }
                __syncwarp();
                ++issued;
                if (++s == STAGES) { s = 0; phase ^= 1u; }
            }
        }
        if (!ok)                                        // the copies in flight land before the CTA leaves its shared memory
            for (int n = issued > STAGES ? issued - STAGES : 0; n < issued; ++n) {
                const long long t0 = clock64();
                while (!mbar_try(bar_full + 8 * (n % STAGES), (n / STAGES) & 1) && clock64() - t0 < 200000000ll) {}
            }
    } else if (warp == EPI_WARPS + 1) {                 // ---- the instructions ----
        int s = 0, local = 0;
        uint32_t phase = 0u;
        bool ok = true;
        for (int64_t t = blockIdx.x; t < g.tiles && ok; t += gridDim.x, ++local) {
            const int buf = local % LY::ACCS;
            ok = ok && warp_wait(bar_c + 8 * buf, (local / LY::ACCS) & 1, &gave_up, budget);    // C is in, and D of the tile before out
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t acc = tmem + buf * BN;
            for (int n = 0; n < nst && ok; ++n) {
                ok = warp_wait(bar_full + 8 * s, phase, &gave_up, budget) && (SF == 0 || warp_wait(bar_sf + 8 * s, phase, &gave_up, budget));
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t base = stage0 + s * LY::STAGE;
                const uint64_t ld = operand_desc(base), qd = operand_desc(base + LY::L_BYTES);
                const uint32_t sfl = tmem + LY::ACCS * BN + s * LY::SF_COLS, sfq = sfl + 4 * SF;
                const int left = g.steps - 4 * n;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    if (k >= left) break;
                    constexpr int B4 = SF == 1 ? 1 : (SF == 2 ? 2 : 0);                 // byte of this step's first scale factor in its word
                    const uint32_t byte = uint32_t(k * B4) & 3u;
                    const int word = (k * SF) >> 2;
                    issue<MK>(lead, acc, ld + 2 * k, qd + 2 * k, g.idesc | (byte << 4) | (byte << 29), sfl + 4 * word, sfq + 4 * LY::NRB * word, g.C || n + k > 0);
                }
                commit(lead, bar_empty + 8 * s);
                if (++s == STAGES) { s = 0; phase ^= 1u; }
            }
            commit(lead, bar_d + 8 * buf);
        }
    } else if (SF > 0 && warp > EPI_WARPS + 1) {        // ---- scale factors: every warp a copy for its quarter of the lanes ----
        constexpr int PER = SF ? (LY::SF_ROWS + 127) / 128 : 1, NR = SF ? (LY::SF_ROWS + 31) / 32 : 1;
        const int me = tid - 32 * (EPI_WARPS + 2), nchunk = (nst + LY::SPC - 1) / LY::SPC;
        const uint32_t ring = stage0 + STAGES * LY::STAGE, quarter = uint32_t(32 * (warp & 3)) << 16;
        int s = 0, slot = 0;
        uint32_t phase = 0u;
        bool ok = true;
        // a thread's rows, one of the lane side and the others of the column side: 16 bytes of each at a time, tile after tile
        // without a gap (16 bytes are a stage of NVFP4, 0.5 us; two of MXFP4, four of MX8)
        auto row_at = [&](int64_t t, int i) -> int64_t { return i == 0 ? t / g.tiles_q * LANES + me : t % g.tiles_q * BN + me + 128 * i - LANES; };
        auto row_of = [&](int64_t t, int i) -> const uint8_t* {
            const int64_t row = row_at(t, i);
            return me + 128 * i < LY::SF_ROWS && row < (i == 0 ? g.R : g.Q) ? (i == 0 ? g.sf_l : g.sf_q) + row * g.nsf : nullptr;
        };
        const uint8_t* src[PER];
        int64_t ft = blockIdx.x;
        int fc = 0;
        // (rows at odd addresses go byte by byte through registers, and into the ring with the next fetch)
        uint4 held[PER];
        int held_to = -1;
        auto fetch = [&](int to) {
            if (held_to >= 0) {
#pragma unroll
                for (int i = 0; i < PER; ++i)
                    if (me + 128 * i < LY::SF_ROWS)
                        asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" :: "r"(ring + 16 * (held_to * LY::SF_ROWS + me + 128 * i)), "r"(held[i].x), "r"(held[i].y), "r"(held[i].z), "r"(held[i].w) : "memory");
                held_to = -1;
            }
            if (ft < g.tiles) {
                if (fc == 0) {
#pragma unroll
                    for (int i = 0; i < PER; ++i) src[i] = row_of(ft, i);
                }
#pragma unroll
                for (int i = 0; i < PER; ++i) {
                    if (me + 128 * i >= LY::SF_ROWS) continue;
                    const uint32_t dst = ring + 16 * (to * LY::SF_ROWS + me + 128 * i);
                    const uint8_t* p = src[i] ? src[i] + 16 * fc : g.sf_l;
                    const int left = src[i] ? g.nsf - 16 * fc : 0;
                    if (g.sf_wide == 16)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" :: "r"(dst), "l"(p), "r"(left > 0 ? 16 : 0) : "memory");
                    else if (g.sf_wide == 4) {
#pragma unroll
                        for (int q = 0; q < 4; ++q)
                            asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" :: "r"(dst + 4 * q), "l"(left > 4 * q ? p + 4 * q : g.sf_l), "r"(left > 4 * q ? 4 : 0) : "memory");
                    } else {
                        uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
                        for (int b = 0; b < 16; ++b)
                            if (b < left) w[b / 4] |= uint32_t(p[b]) << (8 * (b % 4));
                        held[i] = make_uint4(w[0], w[1], w[2], w[3]);
                        held_to = to;
                    }
                }
                if (++fc == nchunk) { fc = 0; ft += gridDim.x; }
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
#pragma unroll
        for (int a = 0; a + 1 < LY::SF_RING; ++a) fetch(a);
        // (a wait that ran out ends the waits and the stores, not the loops: the four warps meet at barriers)
        for (int64_t t = blockIdx.x; t < g.tiles; t += gridDim.x) {
            uint32_t least[PER];
            uint32_t small[PER];                        // factors below this one are looked at
            bool inside[PER];
#pragma unroll
            for (int i = 0; i < PER; ++i) { least[i] = 0xFFFFFFFFu; small[i] = uint32_t(max(0, (-126 - g.least_sf + 1) / 2)); inside[i] = MK != MK_NVF4 && row_of(t, i); }
            for (int c = 0; c < nchunk; ++c) {
                const uint32_t buf = ring + 16 * slot * LY::SF_ROWS;
                asm volatile("cp.async.wait_group %0;" :: "n"(LY::SF_RING - 2) : "memory");
                asm volatile("bar.sync 1, 128;" ::: "memory");      // everybody's rows have landed, and everybody has left the slot before
                fetch(slot == 0 ? LY::SF_RING - 1 : slot - 1);
                slot = slot + 1 == LY::SF_RING ? 0 : slot + 1;
                uint4 x[NR];
#pragma unroll
                for (int j = 0; j < NR; ++j) x[j] = lds16(buf + 16 * (32 * j + lane < LY::SF_ROWS ? 32 * j + lane : 0));
                auto word = [&](int j, int w) -> uint32_t {         // word w of the rows 32 j ..., as far as the tile has them
                    if (j >= NR) return 0u;
                    const uint4 v = x[j < NR ? j : 0];
                    return w == 0 ? v.x : (w == 1 ? v.y : (w == 2 ? v.z : v.w));
                };
#pragma unroll
                for (int i = 0; i < LY::SPC; ++i) {
                    if (c * LY::SPC + i >= nst) break;
                    ok = ok && warp_wait(bar_full + 8 * s, phase, &gave_up, budget);       // (the stage's columns are free)
                    if (ok) {
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");    // behind the instructions that read them
                        const uint32_t sfl = tmem + quarter + LY::ACCS * BN + s * LY::SF_COLS, sfq = sfl + 4 * SF;
                        uint32_t wl[SF ? 4 * SF : 4], wq[SF ? 4 * SF * LY::NRB : 4];
#pragma unroll
                        for (int w = 0; w < SF; ++w)
#pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                wl[4 * w + j] = word(j, i * SF + w);
#pragma unroll
                                for (int b = 0; b < LY::NRB; ++b) wq[4 * LY::NRB * w + 4 * b + j] = word(4 + 4 * b + j, i * SF + w);
                            }
                        tmem_st(sfl, wl);
                        tmem_st(sfq, wq);
                        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                        __syncwarp();
                        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(bar_sf + 8 * s) : "memory");
                    }
                    if (++s == STAGES) { s = 0; phase ^= 1u; }
                }
                if (MK != MK_NVF4) {                    // (behind the stores, which the instructions wait for)
#pragma unroll
                    for (int i = 0; i < PER; ++i)
                        if (inside[i]) {
                            const uint4 v = lds16(buf + 16 * (me + 128 * i));
                            uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                            for (int q = 0; q < 4; ++q) {           // (bytes beyond the row's are not its exponents)
                                const int over = 16 * c + 4 * q + 4 - g.nsf;
                                w[q] |= over <= 0 ? 0u : (over >= 4 ? 0xFFFFFFFFu : ~(0xFFFFFFFFu >> (8 * over)));
                            }
                            uint32_t m4 = __vminu4(__vminu4(w[0], w[1]), __vminu4(w[2], w[3]));
                            if (__vcmpltu4(m4, small[i] * 0x01010101u)) {
                                const uint2 f = without_zero_blocks<MK>(i == 0 ? g.codes_l + row_at(t, i) * g.pitch_l : g.codes_q + row_at(t, i) * g.pitch_q, g.row_bytes,
                                                                        i == 0 ? g.magnitude_l : g.magnitude_q, 16 * c, make_uint4(w[0], w[1], w[2], w[3]), small[i]);
                                m4 = f.x;
                                small[i] = f.y;
                            }
                            least[i] = __vminu4(least[i], m4);
                        }
                }
            }
            if (MK != MK_NVF4) {                        // the tile's smallest scale factors of A and of B
                auto byte = [](uint32_t v) { const uint32_t h = __vminu4(v, v >> 16); return __vminu4(h, h >> 8) & 0xFFu; };
                uint32_t ll = byte(least[0]), lq = 255u;
#pragma unroll
                for (int i = 1; i < PER; ++i) lq = min(lq, byte(least[i]));
                ll = __reduce_min_sync(0xFFFFFFFFu, ll);
                lq = __reduce_min_sync(0xFFFFFFFFu, lq);
                if (lane == 0) { least_s[warp & 3][0] = int(ll); least_s[warp & 3][1] = int(lq); }
                asm volatile("bar.sync 1, 128;" ::: "memory");
                if (me == 0) {
                    const int a = min(min(least_s[0][0], least_s[1][0]), min(least_s[2][0], least_s[3][0]));
                    const int b = min(min(least_s[0][1], least_s[1][1]), min(least_s[2][1], least_s[3][1]));
                    g.redo[t] = a + b + g.least_sf < -126;
                }
                asm volatile("bar.sync 1, 128;" ::: "memory");
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
    } else {                                            // ---- C in, D out: thread = one lane of tensor memory, half of the columns ----
        constexpr int SHARE = BN >= 32 ? BN / 2 : BN, CH = SHARE < 64 ? SHARE : 64;      // columns per warp, and at a time
        const int quarter = warp & 3, half = warp >> 2;
        const bool idle = half * SHARE >= BN;           // (16 columns: the second four warps have nothing)
        const uint32_t taddr = tmem + (uint32_t(32 * quarter) << 16);
        auto load_c = [&](int64_t t, int buf) {
            const int64_t q0 = (t % g.tiles_q) * BN, l = (t / g.tiles_q) * LANES + 32 * quarter + lane;
            if (g.C && !idle) {
                const bool full = q0 + BN <= g.Q && (t / g.tiles_q + 1) * LANES <= g.R;
#pragma unroll 1
                for (int c0 = half * SHARE; c0 < half * SHARE + SHARE; c0 += CH) {
                    uint32_t x[CH];
                    const W* p = static_cast<const W*>(g.C) + (q0 + c0) * g.ldc + l;
                    if (full) load_words<W, CH, true>(p, g.ldc, CH, x);
                    else load_words<W, CH, false>(p, g.ldc, l < g.R ? int(min(int64_t(CH), g.Q - q0 - c0)) : 0, x);
#pragma unroll
                    for (int c = 0; c < CH; c += 16) tmem_st16(taddr + buf * BN + c0 + c, x + c);
                }
                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(bar_c + 8 * buf) : "memory");
        };
        int local = 0;
        if (int64_t(blockIdx.x) < g.tiles) load_c(blockIdx.x, 0);
        for (int64_t t = blockIdx.x; t < g.tiles; t += gridDim.x, ++local) {
            const int buf = local % LY::ACCS;
            const int64_t next = t + gridDim.x;
            if (SF == 0 && g.least_l && warp == 0) {
                const int64_t l0 = t / g.tiles_q * LANES, q0 = t % g.tiles_q * BN;
                int a = 1 << 20, b = 1 << 20;
                for (int r = lane; r < LANES; r += 32) if (l0 + r < g.R) a = min(a, g.least_l[l0 + r]);
                for (int r = lane; r < BN; r += 32) if (q0 + r < g.Q) b = min(b, g.least_q[q0 + r]);
                a = __reduce_min_sync(0xFFFFFFFFu, a);
                b = __reduce_min_sync(0xFFFFFFFFu, b);
                if (lane == 0) g.redo[t] = a + b < -126;
            }
            if (LY::ACCS == 2 && next < g.tiles) load_c(next, buf ^ 1);
            if (!warp_wait(bar_d + 8 * buf, (local / LY::ACCS) & 1, &gave_up, 2 * budget) || __any_sync(0xFFFFFFFFu, gave_up)) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int64_t q0 = (t % g.tiles_q) * BN, l = (t / g.tiles_q) * LANES + 32 * quarter + lane;
            const bool full = q0 + BN <= g.Q && (t / g.tiles_q + 1) * LANES <= g.R;
            if (!idle) {
#pragma unroll 1
                for (int c0 = half * SHARE; c0 < half * SHARE + SHARE; c0 += CH) {
                    uint32_t x[CH];
#pragma unroll
                    for (int c = 0; c < CH; c += 16) tmem_ld16(taddr + buf * BN + c0 + c, x + c);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                    const int valid = l < g.R ? int(min(int64_t(CH), g.Q - q0 - c0)) : 0;
                    if (g.scale_l && valid > 0) {
                        const float sl = g.scale_l[l];
#pragma unroll
                        for (int c = 0; c < CH; ++c) {
                            float sc = __fmul_rn(sl, c < valid ? g.scale_q[q0 + c0 + c] : 0.f);
                            if (sc != sc) sc = __uint_as_float(0x7FFFFFFFu);
                            float v = __fmul_rn(sc, __uint_as_float(x[c]));
                            if (v != v) v = __uint_as_float(0x7FFFFFFFu);
                            x[c] = __float_as_uint(v);
                        }
                    }
                    W* p = static_cast<W*>(g.D) + (q0 + c0) * g.ldd + l;
                    if (full) store_words<W, CH, true>(p, g.ldd, CH, x);
                    else store_words<W, CH, false>(p, g.ldd, valid, x);
                }
            }
            if (LY::ACCS == 1 && next < g.tiles) load_c(next, 0);
        }
    }
    __syncwarp();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == EPI_WARPS + 1) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"(LY::COLS) : "memory");
    if (tid == 0 && gave_up && g.timeouts) atomicAdd(g.timeouts, 1u);
}

// ---- operands in the instruction's layout, smallest exponents ----
struct Side {
    const unsigned char* src;
    unsigned char* dst;
    int64_t rows, ld;
    int bits;                           // width of a code (8: this side is not packed)
};
// One code per byte -> chunks of sixteen codes packed from bit 0 upwards, 16 bytes each; rows of ceil(K / 16) chunks.
__global__ void __launch_bounds__(256) pack_codes_kernel(Side a, Side b, int K) {
    after_previous();
    const Side s = blockIdx.y ? b : a;
    const int chunks = (K + 15) / 16;
    const int64_t q = int64_t(blockIdx.x) * 256 + threadIdx.x;
    if (!s.dst || q >= s.rows * chunks) return;
    const int64_t r = q / chunks;
    const int c = int(q % chunks), n = min(16, K - 16 * c);
    const unsigned char* p = s.src + r * s.ld + 16 * c;
    __align__(16) unsigned char code[16];
    if (n == 16) *reinterpret_cast<uint4*>(code) = *reinterpret_cast<const uint4*>(p);
    else
        for (int i = 0; i < 16; ++i) code[i] = i < n ? p[i] : 0;
    unsigned long long lo = 0ull, hi = 0ull;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const unsigned long long v = code[i] & ((1u << s.bits) - 1u);
        const int pos = s.bits * i;
        if (pos < 64) { lo |= v << pos; if (pos + s.bits > 64) hi |= v >> (64 - pos); }
        else hi |= v << (pos - 64);
    }
    *reinterpret_cast<uint4*>(s.dst + q * 16) = make_uint4(uint32_t(lo), uint32_t(lo >> 32), uint32_t(hi), uint32_t(hi >> 32));
}

struct LeastSide {
    const unsigned char* src;
    int* least;
    int64_t rows, pitch;
};
// The smallest exponent of the nonzero elements of a row (BF16, or TF32 as FP32 words), one warp per row; rows of `n` 32-bit words,
// 16-byte starts; `odd`: the last word holds one BF16 element only.
template <bool BF16>
__global__ void __launch_bounds__(256) least_exponent_kernel(LeastSide a, LeastSide b, int n, bool odd) {
    after_previous();
    const LeastSide s = blockIdx.y ? b : a;
    const int64_t r = int64_t(blockIdx.x) * 8 + threadIdx.x / 32;
    if (r >= s.rows) return;
    const uint32_t* p = reinterpret_cast<const uint32_t*>(s.src + r * s.pitch);
    uint32_t least = 0xFFFFFFFFu;                       // of magnitude - 1: zero wraps to the top
    auto word = [&](uint32_t w) {
        if (BF16) least = min(least, min(((w << 16) & 0x7FFF0000u) - 1u, (w & 0x7FFF0000u) - 1u));
        else least = min(least, (w & 0x7FFFE000u) - 1u);
    };
    const int whole = n - (odd ? 1 : 0);
#pragma unroll 4
    for (int i = threadIdx.x % 32 * 4; i < whole; i += 128) {
        if (i + 4 <= whole) {
            const uint4 v = *reinterpret_cast<const uint4*>(p + i);
            word(v.x); word(v.y); word(v.z); word(v.w);
        } else
            for (int k = i; k < whole; ++k) word(p[k]);
    }
    if (odd && threadIdx.x % 32 == 0) word(reinterpret_cast<const uint16_t*>(p)[2 * whole]);
    least = __reduce_min_sync(0xFFFFFFFFu, least);
    const uint32_t field = (least + 1u) >> 23;
    if (threadIdx.x % 32 == 0) s.least[r] = least == 0xFFFFFFFFu ? 1 << 20 : int(max(field, 1u)) - 127;
}

int code_bits(int fmt) { return fmt == EF_E2M1 ? 4 : (fmt == EF_E2M3 || fmt == EF_E3M2 ? 6 : 8); }
bool is8(int f) { return f == EF_E4M3 || f == EF_E5M2 || f == EF_E3M2 || f == EF_E2M3 || f == EF_E2M1; }

// The instruction that computes the model's block, or -1.
int kind_of(const DevModel& m) {
    if (m.literal_emax || m.inner_round) return -1;
    if (m.family == FAM_T && !m.packed4) {
        const bool f32 = m.rho == RHO_RZ_FP32 && m.acc == ACC_F32, f16 = m.rho == RHO_RNE_FP16 && m.acc == ACC_F16;
        if (m.F != 25 || !(f32 || f16)) return -1;
        if (is8(m.fmt_a) && is8(m.fmt_b)) return m.L == 32 ? MK_F8 : -1;
        if (m.fmt_a != m.fmt_b) return -1;
        if (m.fmt_a == EF_F16) return m.L == 16 ? MK_F16 : -1;
        if (m.fmt_a == EF_BF16) return m.L == 16 && f32 ? MK_F16 : -1;
        if (m.fmt_a == EF_TF32) return m.L == 8 && f32 ? MK_TF32 : -1;
        return -1;
    }
    if (m.rho != RHO_RZ_FP32 || m.acc != ACC_F32) return -1;
    if (m.family == FAM_ST) return is8(m.fmt_a) && is8(m.fmt_b) && m.F == 25 && m.L == 32 && m.k_block == 32 && m.scale_fmt == EF_E8M0 ? MK_MX8 : -1;
    if (m.family == FAM_GST && m.packed4 && m.L == 64 && m.G == 16 && m.F == 35) {
        if (m.scale_fmt == EF_E8M0 && m.k_block == 32) return MK_MXF4;
        if (m.scale_fmt == EF_UE4M3 && m.k_block == 16) return MK_NVF4;
    }
    return -1;
}
uint32_t format_code(int mk, int fmt) {
    if (mk == MK_F16) return fmt == EF_BF16 ? 1u : 0u;
    if (mk == MK_TF32) return 2u;
    if (mk >= MK_MXF4) return 1u;
    switch (fmt) { case EF_E4M3: return 0u; case EF_E5M2: return 1u; case EF_E2M3: return 3u; case EF_E3M2: return 4u; default: return 5u; }
}
constexpr int64_t up(int64_t x, int64_t to) { return (x + to - 1) / to * to; }
int64_t row_bytes(const DevModel& m, int64_t elems) { return m.packed4 ? elems / 2 : elems * (fmt_desc(m.fmt_a).storage_bits / 8); }

template <int MK, int BN, bool ACC16>
cudaError_t launch_tile(const CUtensorMap& l, const CUtensorMap& q, const UmmaArgs& a, cudaStream_t st) {
    auto kernel = umma_kernel<MK, BN, ACC16>;
    const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, Layout<MK, BN>::SMEM);
    if (err != cudaSuccess) return err;
    return enqueue(kernel, unsigned(a.tiles < SMS ? a.tiles : SMS), Layout<MK, BN>::NTHREADS, Layout<MK, BN>::SMEM, st, l, q, a);
}
template <int MK, bool ACC16>
cudaError_t launch_bn(int bn, const CUtensorMap& l, const CUtensorMap& q, const UmmaArgs& a, cudaStream_t st) {
    switch (bn) {
        case 16: return launch_tile<MK, 16, ACC16>(l, q, a, st);
        case 32: return launch_tile<MK, 32, ACC16>(l, q, a, st);
        case 64: return launch_tile<MK, 64, ACC16>(l, q, a, st);
        case 128: return launch_tile<MK, 128, ACC16>(l, q, a, st);
        default: return launch_tile<MK, 256, ACC16>(l, q, a, st);
    }
}

// Columns per tile.  Measured per instruction (32 bytes of K), in ns: the chain through the accumulator up to 64 columns, the
// operands' way from L2 (60 bytes per clock and SM) from 128 on; the warps that store scale words need 0.25 (MX8) to 0.35 us per stage.
// The rest is C and D, 40 bytes per ns and SM, beside the instructions of another tile where tensor memory holds two accumulators.
// 16 / 32 / 64 / 128 / 256 columns, us a call: FP16 4096^3 595 / 306 / 166 / 124 / 123, MXFP8 1024 x 4096 x 4096 120 / 64 / 43 / 30 / 25,
// NVFP4 1024^3 12 / 9 / 7 / 9 / 11.
int pick_columns(const GemmArgs& g, int mk, bool acc16, int steps) {
    const double plain[5] = {41, 41, 47, 70, 119}, mx8[5] = {62, 61, 66, 86, 122}, fp4[5] = {85, 87, 97, 125, 155};
    const double* step = sf_per_step(mk) == 0 ? plain : (sf_per_step(mk) == 1 ? mx8 : fp4);
    int best = 128;
    double least = 1e300;
    for (int i = 0; i < 5; ++i) {
        const int bn = 16 << i;
        const int64_t tiles = ((g.N + LANES - 1) / LANES) * ((g.M + bn - 1) / bn);
        const double per_sm = double((tiles + SMS - 1) / SMS), io = bn * LANES * (acc16 ? 2 : 4) * (g.C ? 2 : 1) / 40.0, run = steps * step[i];
        const bool overlap = bn < 256 || sf_per_step(mk) == 0;
        const double cost = overlap ? per_sm * (run > io ? run : io) + io : per_sm * (run + io);
        if (cost < least) { least = cost; best = bn; }
    }
    return best;
}

// Kinds with products below 2^-126 (see the top).
bool guarded(const DevModel& m, int mk) { return mk == MK_MX8 || mk == MK_MXF4 || mk == MK_TF32 || (mk == MK_F16 && m.fmt_a == EF_BF16); }
// Scratch of launch_umma: packed codes of A and B, the smallest exponents of their rows, flags of tiles.
struct UmmaScratch {
    int bits_a, bits_b;
    int64_t pk;                         // bytes of a row of packed codes
    size_t pa, pb, le, fl;
    UmmaScratch(const DevModel& m, const GemmArgs& g, int mk, int64_t tiles) {
        const bool narrow = mk == MK_F8 || mk == MK_MX8;
        bits_a = narrow ? code_bits(m.fmt_a) : 8;
        bits_b = narrow ? code_bits(m.fmt_b) : 8;
        pk = up(g.K, 16);
        pa = bits_a < 8 ? size_t(up(g.M * pk, 256)) : 0;
        pb = bits_b < 8 ? size_t(up(g.N * pk, 256)) : 0;
        le = guarded(m, mk) && sf_per_step(mk) == 0 ? size_t(4 * (g.M + g.N)) : 0;
        fl = guarded(m, mk) ? size_t(tiles) : 0;
    }
    size_t bytes() const { return pa + pb + le + fl; }
};
bool overlap(const GemmArgs& g) {
    const char *c = static_cast<const char*>(g.C), *d = static_cast<const char*>(g.D);
    return c && c < d + ((g.M - 1) * g.ldd + g.N) * 4 && d < c + ((g.M - 1) * g.ldc + g.N) * 4;
}

}  // namespace

bool umma_supported(const DevModel& m, const GemmArgs& g) {
    const int mk = kind_of(m);
    if (mk < 0 || g.dot_mode || g.k_chunk || !encode_fn()) return false;
    if (row_bytes(m, g.lda) % 16 || row_bytes(m, g.ldb) % 16) return false;            // 16-byte row starts for the tiled copies
    if (g.M >= 0x7FFF0000ll || g.N >= 0x7FFF0000ll || row_bytes(m, g.K) >= 0x7FFF0000ll) return false;      // 32-bit coordinates
    if (!guarded(m, mk)) return true;
    // The emulation goes last, so C has to be there still; and its launch and that of the exponents have to pay.
    if (overlap(g)) return false;
    if (mk == MK_MXF4) return fast_gst_supported(m, g);
    // Emulation / instruction in us, by launches around the instruction.  Two (BF16 and TF32: the exponents before, the flags after; packed MX
    // rows): BF16 512 x 512 x 64 9.4 / 14.6, 512 x 512 x 128 12.5 / 14.6, 384 x 384 x 256 14.7 / 14.6, 512 x 512 x 256 20.7 / 14.6, TF32
    // 512 x 512 x 128 14.6 / 14.6.  One (MXFP8: the flags): 256 x 256 x 128 8.4 / 11.2, 384 x 384 x 128 12.5 / 11.0, 64 x 64 x 512 15.5 / 10.1.
    double us = 0.0;
    direct_size(m, g, &us);
    return us > (mk == MK_MX8 && code_bits(m.fmt_a) == 8 && code_bits(m.fmt_b) == 8 ? 11.0 : 15.0);
}

size_t umma_scratch(const DevModel& m, const GemmArgs& g) {
    const int mk = kind_of(m), bn = pick_columns(g, mk, m.acc == ACC_F16, int((row_bytes(m, g.K) + 31) / 32));
    return UmmaScratch(m, g, mk, (g.N + LANES - 1) / LANES * ((g.M + bn - 1) / bn)).bytes();
}

int launch_umma(const DevModel& m, const GemmArgs& g, cudaStream_t stream) {
    const int mk = kind_of(m);
    if (warp_mma_supported(m, g)) {
        set_kernel_name("tfdpa_f16", "matrix_instruction");
        const cudaError_t err = launch_warp_mma(m, g, stream);
        if (err != cudaSuccess) {
            set_error("matrix-instruction kernel launch failed: %s", cudaGetErrorString(err));
            return MMASIM_ERR_CUDA;
        }
        return MMASIM_OK;
    }
    const int64_t kb = row_bytes(m, g.K);
    UmmaArgs a;
    a.steps = int((kb + 31) / 32);
    const int bn = pick_columns(g, mk, m.acc == ACC_F16, a.steps);
    a.C = g.C; a.D = g.D;
    a.R = g.N; a.Q = g.M;
    a.ldc = g.ldc; a.ldd = g.ldd;
    a.tiles_q = int((a.Q + bn - 1) / bn);
    a.tiles = (a.R + LANES - 1) / LANES * a.tiles_q;
    a.scale_l = g.col_scale;
    a.scale_q = g.row_scale;
    a.timeouts = g.copy_timeouts;
    // instruction descriptor (see mmasim_hw_umma.cu): result format, operand formats, N / 8, M / 16; scale type for the scaled kinds
    const bool scaled = sf_per_step(mk) > 0;
    a.idesc = (format_code(mk, m.fmt_b) << 7) | (format_code(mk, m.fmt_a) << 10) | (uint32_t(bn >> 3) << 17) | (uint32_t(LANES >> 4) << 24);
    if (scaled) a.idesc |= uint32_t(m.scale_fmt == EF_E8M0) << 23;
    else if (m.acc != ACC_F16) a.idesc |= 1u << 4;

    const bool guard = guarded(m, mk);
    const UmmaScratch sc(m, g, mk, a.tiles);
    const int bits_a = sc.bits_a, bits_b = sc.bits_b;
    const int64_t pk = sc.pk;
    const size_t pa = sc.pa, pb = sc.pb, le = sc.le, fl = sc.fl;
    cudaError_t err = cudaSuccess;
    unsigned char* scratch = nullptr;
    if (sc.bytes()) err = take_scratch(g, sc.bytes(), stream, reinterpret_cast<void**>(&scratch));
    if (err != cudaSuccess) scratch = nullptr;
    int* least = reinterpret_cast<int*>(scratch + pa + pb);
    a.least_l = le ? least + g.M : nullptr;
    a.least_q = le ? least : nullptr;
    a.redo = fl ? scratch + pa + pb + le : nullptr;
    a.sf_l = g.sfb;
    a.sf_q = g.sfa;
    a.nsf = scaled ? int((g.K + m.k_block - 1) / m.k_block) : 0;
    const uintptr_t starts = reinterpret_cast<uintptr_t>(g.sfa) | reinterpret_cast<uintptr_t>(g.sfb) | uintptr_t(a.nsf);
    a.sf_wide = starts % 16 == 0 ? 16 : (starts % 4 == 0 ? 4 : 1);
    // (an MXFP4 group's exponent is its scale factors'; sixteen binades are kept away from the edge)
    a.least_sf = (mk == MK_MXF4 ? -16 : 2 - fmt_desc(m.fmt_a).bias - fmt_desc(m.fmt_b).bias) - 254;
    const unsigned char* A = static_cast<const unsigned char*>(g.A);
    const unsigned char* B = static_cast<const unsigned char*>(g.B);
    int64_t pitch_a = row_bytes(m, g.lda), pitch_b = row_bytes(m, g.ldb), kb_a = kb, kb_b = kb;
    a.codes_l = B; a.pitch_l = pitch_b; a.magnitude_l = (mk == MK_MXF4 ? 0x77u : (1u << (bits_b - 1)) - 1u) * 0x01010101u;
    a.codes_q = A; a.pitch_q = pitch_a; a.magnitude_q = (mk == MK_MXF4 ? 0x77u : (1u << (bits_a - 1)) - 1u) * 0x01010101u;
    a.row_bytes = int(kb);
    const int64_t rows = g.M > g.N ? g.M : g.N;
    if (err == cudaSuccess && pa + pb) {
        const Side s[2] = {{A, pa ? scratch : nullptr, g.M, pitch_a, bits_a}, {B, pb ? scratch + pa : nullptr, g.N, pitch_b, bits_b}};
        err = enqueue(pack_codes_kernel, dim3(unsigned((rows * (pk / 16) + 255) / 256), 2), 256, 0, stream, s[0], s[1], int(g.K));
        if (pa) { A = s[0].dst; pitch_a = kb_a = pk; }
        if (pb) { B = s[1].dst; pitch_b = kb_b = pk; }
    }
    if (err == cudaSuccess && le) {
        const LeastSide sa{A, least, g.M, pitch_a}, sb{B, least + g.M, g.N, pitch_b};
        const dim3 grid(unsigned((rows + 7) / 8), 2);
        if (mk == MK_TF32) err = enqueue(least_exponent_kernel<false>, grid, 256, 0, stream, sa, sb, int(g.K), false);
        else err = enqueue(least_exponent_kernel<true>, grid, 256, 0, stream, sa, sb, int((g.K + 1) / 2), g.K % 2 != 0);
    }
    if (err == cudaSuccess) {
        CUtensorMap ml, mq;
        if (!encode(&ml, B, kb_b, a.R, pitch_b, LANES) || !encode(&mq, A, kb_a, a.Q, pitch_a, bn)) err = cudaErrorInvalidValue;
        else switch (mk) {
            case MK_F16: err = m.acc == ACC_F16 ? launch_bn<MK_F16, true>(bn, ml, mq, a, stream) : launch_bn<MK_F16, false>(bn, ml, mq, a, stream); break;
            case MK_TF32: err = launch_bn<MK_TF32, false>(bn, ml, mq, a, stream); break;
            case MK_F8: err = m.acc == ACC_F16 ? launch_bn<MK_F8, true>(bn, ml, mq, a, stream) : launch_bn<MK_F8, false>(bn, ml, mq, a, stream); break;
            case MK_MX8: err = launch_bn<MK_MX8, false>(bn, ml, mq, a, stream); break;
            case MK_MXF4: err = launch_bn<MK_MXF4, false>(bn, ml, mq, a, stream); break;
            default: err = launch_bn<MK_NVF4, false>(bn, ml, mq, a, stream); break;
        }
    }
    int st = MMASIM_OK;
    if (err == cudaSuccess && guard) {
        GemmArgs e = g;
        e.redo = a.redo;
        e.redo_rows = bn;
        e.redo_across = a.tiles_q;
        st = mk == MK_MXF4 ? launch_fast_gst(m, e, stream) : launch_direct(m, e, DIRECT_32x32, stream);
    }
    if (scratch) give_scratch(g, scratch, stream);
    set_kernel_name(mk >= MK_MXF4 ? "gstfdpa" : (mk == MK_TF32 ? "tfdpa_tf32" : (mk != MK_F16 ? "tfdpa_lut8" : (m.fmt_a == EF_F16 ? "tfdpa_f16" : "tfdpa_bf16"))), "matrix_instruction");
    if (err != cudaSuccess) {
        set_error("matrix-instruction kernel launch failed: %s", cudaGetErrorString(err));
        return MMASIM_ERR_CUDA;
    }
    return st;
}

}  // namespace mmasim
