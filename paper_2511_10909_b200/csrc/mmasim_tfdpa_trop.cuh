// T-FDPA for FP8 inputs with F = 13 (the Ada / Hopper FP8 rows, E4M3 and E5M2 in any combination; Algorithm 5 + 7 +
// Table 2): the sum of a block in an FP32 register, one fused multiply-add per term, and the block's exponent maximum
// taken by the tensor cores.
//
// The sum register.  Aligned terms are below 2^15 and block sums below 2^21, so the fixed-point sum S of Algorithm 7
// fits an FP32 register as (1.5 * 2^23 + S) * u with u = 2^(e_max - F): in [2^23 u, 2^24 u) one ulp is u, so
// fma.rm.f32(a, b, register) forms a * b + register exactly and rounds once, toward minus infinity, onto multiples of
// u - the shift by e_max - e_k, the truncation and the addition of Algorithm 7 in one instruction, the alignment
// distance carried by the register's exponent.  Operands are the element values (A) and the element values with an
// offset 2^-(pre + guard) below the last significand bit (B), so that a negative product is never on the grid and
// floors to the one's complement of its truncated magnitude; a population count over sign masks adds the number of
// negative terms back (a zero is staged as a tiny number of its sign, TINY: far below any unit, its negative products too
// fall one short, so that no mask of nonzero elements is needed).  The accumulator enters by one fused multiply-add rounded toward minus infinity (times
// 1 + 2^-23: with its last mantissa bit clear, a c off the grid moves by less than its distance to the next grid point and one on the
// grid leaves it, so that a negative c floors likewise; the +1 is added to the register's starting value),
// and the block's value S * u leaves by one exact subtraction of 1.5 * 2^23 * u; rho is a mask (RZ-E8M13) or a
// conversion (RNE-FP16).  The accumulator between blocks is the output word itself.
//
// e_max = max_k (Exp(a_k) + Exp(b_k)) is a (max, +) product.  Powers turn it into an ordinary one: with
// pe(x) = 2^(6 (Exp(x) - 1)) for a nonzero finite x and 0 otherwise (the B plane scaled by 2^5 more),
//     P = sum_k pe(a_k) * pe(b_k)  lies in  2^(6 (e_max + 20) - 127) * [1, 32]  (at most 32 terms, 32 < 2^6),
// so its FP32 exponent field is 6 (e_max + 20) + 0..5 and floor(field / 6) - 20 = e_max exactly, whatever the order,
// rounding or truncation of the summation (terms far below the largest may be dropped, they do not matter).  E4M3
// exponents span 15 values: 6 * (Exp - 1) stays within +-42 and P within the FP32 range; with E5M2 operands the base
// is 2^5 or 2^4 and P is taken over sub-blocks of 16 or 8 terms (see pe_shift below).  P for the 32 x 32 outputs
// of a warp and one block of 32 is sixteen mma.sync.m16n8k16 on BF16 planes of pe values (a power of two is exact in
// BF16), instead of sixteen fused add-max instructions per output; P = 0 (every product zero: no exponent) converts
// to an exponent below every real one.  The fragments come by ldmatrix.  The division by the base is one high multiply on the bits of P, which leaves
// the result as an FP32 exponent field in place, comparable with the bits of |c| and a mask away from the sum
// register's starting value.
//
// A warp owns 32 rows x 32 columns of the CTA tile (two by four accumulator fragments), and the micro-tile of a thread is
// its share of those fragments: rows g, g + 8, g + 16, g + 24 (g = lane / 4) and columns 8 j + 2 t, 8 j + 2 t + 1
// (t = lane % 4, j = 0..3), so that the maxima arrive in the registers of the thread that needs them.  The operand
// planes are stored with rows and columns permuted accordingly (the four rows of a thread adjacent, its eight
// columns contiguous): three 16-byte shared loads feed the 32 fused multiply-adds of one k, which are issued as
// sixteen packed ones (fma.rm.f32x2: two adjacent columns per instruction).
//
// What bounds it: the packed multiply-adds with their loads and moves (2.5 of the 3.97 ms at 4096^3 that the kernel took with every phase
// on; 1.9 at the nominal rate), then the integer work per output and block (0.95 ms) and the tensor-core pass (0.5 ms); the phases
// add up, integer and FP32 instructions of one SM partition do not run beside each other at full rate.  4096^3, Hopper E4M3 -> FP32:
// 4.21 ms -> 3.97 (zeros as tiny numbers, range test left out) -> 3.84 (accumulator by multiply-add, ldmatrix).
#pragma once
#include <type_traits>
#include "mmasim_tfdpa_fast.cuh"

namespace mmasim {
namespace trop {

using fast::BM;
using fast::KC;
using fast::NT;
using fast::CB;
using fast::Elem;
using fast::raw_elem;
using fast::mbar_init;
using fast::mbar_expect_tx;
using fast::bulk_load;
using fast::mbar_wait;
using fast::smem_addr;

constexpr int PE_STRIDE = KC + 8;       // BF16 elements per row of a pe plane: 80 bytes, fragment loads hit 32 different banks
constexpr int PE_CENTER = 1;            // pe(x) = 2^(6 (Exp(x) - PE_CENTER)); E4M3: Exp in [-6, 8]
// pe(x) = 2^(BASE (Exp(x) - PE_CENTER)), the B plane times 2^pe_shift so that 127 + pe_shift is a multiple of BASE and
// the exponent field of P is BASE * (e_max + constant) + 0..BASE-1.  A sum of at most 2^(BASE-1) terms stays within a
// factor 2^(BASE-1) of its largest term; the spread of the exponents decides which BASE fits the FP32 range:
//   BASE 8: blocks of up to 32 terms in one accumulation; E4M3 x E4M3 (product exponents -12..16: 8 * 28 = 224 binades,
//           plus the 5 binades a sum of 32 terms can grow; the division by 8 is a shift)
//   BASE 5: sub-blocks of 16 terms; E4M3 x E5M2 (-20..23: 5 * 43 = 215 binades)
//   BASE 4: sub-blocks of 8 terms;  E5M2 x E5M2 (-28..30: 4 * 58 = 232 binades)
// The block maximum is then the integer maximum of the sub-blocks' P words.
__host__ __device__ constexpr int pe_shift(int base) { return base == 8 ? 1 : (base == 5 ? 3 : 1); }
__host__ __device__ constexpr int pe_sub(int base) { return base == 8 ? 32 : (base == 5 ? 16 : 8); }
__host__ __device__ constexpr uint32_t pe_mul(int base) { return base == 5 ? 0x33333334u : 0u; }  // ceil(2^32 / BASE); powers of two shift
constexpr int TW = 8;                   // micro-tile: TH rows x 8 columns

// Geometry by the height TH of the micro-tile.  TH = 4: warps 4 x 2, warp tile 32 x 32, CTA tile 128 x 64.
// TH = 8: warps 2 x 4, warp tile 64 x 32, CTA tile 128 x 128 - sixteen operand words per 64 multiply-adds instead of
// twelve per 32, at the price of 64 accumulator registers (where nothing else has to live across the K loop, and the larger tiles
// fill the SMs as well; see tall_tile).
template <int TH>
struct Geo {
    static_assert(TH == 4 || TH == 8, "two or four accumulator fragments stacked");
    static constexpr int WROWS = 8 * TH;                // rows of a warp tile
    static constexpr int WARPS_R = BM / WROWS, WARPS_C = (NT / 32) / WARPS_R;
    static constexpr int BN = 32 * WARPS_C;
    static constexpr int NB = BN * KC / NT;             // elements of B staged per thread: 8 or 16
};

struct LutEntryT {      // 8 bytes: one shared load per staged element
    uint32_t op;        // staged FP32 operand
    uint32_t y;         // bits 0..14: BF16 word of pe(x); bit 15: infinity / NaN (a pe of -0: harmless in P);
                        // bit 16: sign; bit 24: zero
};

// One operand's share of a chunk of KC = 32 elements of K, decoded: R rows of A (or columns of B).  A decode kernel
// writes these blocks to scratch memory once per GEMM; the main kernel brings them in with one bulk copy each.
template <int R>
struct BlkT {
    uint32_t op[KC][R];                 // [k][permuted row]: FP32 operands
    uint16_t pe[R][PE_STRIDE];          // [row][k]: BF16 exponent powers for the tensor cores
    uint32_t sgn[R];                    // [permuted row]: bit k = sign of element k of the chunk
    uint32_t special;                   // nonzero: the block holds an infinity or a NaN
    uint32_t sparse;                    // nonzero: a row (of the matrix) has a block of L with half or more of its elements zero
    uint32_t pad[2];
};
static_assert(sizeof(BlkT<128>) == fast::blk_t_bytes(128) && sizeof(BlkT<64>) == fast::blk_t_bytes(64), "what fast_tfdpa_scratch counts with");
static_assert(sizeof(BlkT<128>) % 16 == 0 && sizeof(BlkT<64>) % 16 == 0, "bulk copies move multiples of 16 bytes");

template <int TH>
struct SmemT {
    BlkT<BM> a[2];
    BlkT<Geo<TH>::BN> b[2];
    unsigned long long full[2];         // mbarriers: the bulk copies of a buffer have landed
    unsigned long long flags[3][NT];    // per thread: outputs (bit h * TW + x) that have seen a NaN, +infinity, -infinity
    int error;                          // a bounded wait ran out
};

// Position of a row / column of the CTA tile inside the permuted planes: the TH rows of a thread (g, g + 8, ...)
// adjacent, its eight columns (8 j + 2 t, 8 j + 2 t + 1) contiguous.
template <int TH>
__device__ __forceinline__ int perm_row(int r) {
    return TH == 4 ? ((r & ~31) | ((r & 7) << 2) | ((r >> 3) & 3)) : ((r & ~63) | ((r & 7) << 3) | ((r >> 3) & 7));
}
__device__ __forceinline__ int perm_col(int c) { return (c & ~31) | (((c >> 1) & 3) << 3) | (((c >> 3) & 3) << 1) | (c & 1); }

// four 8 x 8 tiles of 16-bit elements, lane l gives row l % 8 of tile l / 8 (stride 80 bytes: eight rows in eight bank groups)
__device__ __forceinline__ void ldmatrix4(uint32_t* r, const void* row) {
    asm("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(smem_addr(row)) : "memory");
}

constexpr float TINY = 7.888609052210118e-31f;          // 2^-100: times an element below 2^-83, the smallest unit is 2^-43

template <int BASE>
__device__ __forceinline__ void init_lut_t(LutEntryT* lut_a, LutEntryT* lut_b, const FmtDesc& fa, const FmtDesc& fb, int pre, int guard, int tid) {
    const uint32_t da = decode_elem(fa, uint32_t(tid)), db = decode_elem(fb, uint32_t(tid));
    const bool fin_a = dec_cls(da) == CLS_FINITE, fin_b = dec_cls(db) == CLS_FINITE;
    const bool nz_a = fin_a && dec_sig(da) != 0u, nz_b = fin_b && dec_sig(db) != 0u;
    LutEntryT ea, eb;
    auto tiny = [](uint32_t d) { return __float_as_uint(dec_sign(d) ? -TINY : TINY); };
    ea.op = nz_a ? __float_as_uint(ldexpf(float(dec_ssig(da)), dec_exp(da))) : tiny(da);
    ea.y = (nz_a ? uint32_t((127 + BASE * (dec_exp(da) - PE_CENTER)) << 7) : 0u) | (fin_a ? 0u : 0x8000u) |
           (dec_sign(da) << 16) | (uint32_t(!nz_a) << 24);
    const int sb = fin_b ? dec_ssig(db) : 0;
    const int ub = dec_sign(db) ? -1 : 1;
    // a_op * b_op = a * b * (1 + 2^-(pre + guard) / |sig_b|): the true product with the offset that makes a negative one inexact
    eb.op = nz_b ? __float_as_uint(ldexpf(float(sb * (1 << (pre + guard)) + ub), dec_exp(db) - (fa.mbits + fb.mbits + pre + guard))) : tiny(db);
    eb.y = (nz_b ? uint32_t((127 + pe_shift(BASE) + BASE * (dec_exp(db) - PE_CENTER)) << 7) : 0u) | (fin_b ? 0u : 0x8000u) |
           (dec_sign(db) << 16) | (uint32_t(!nz_b) << 24);
    lut_a[tid] = ea;
    lut_b[tid] = eb;
}

// N = 16 or 8 elements of one row: operands k-major, pe words row-major, sign bits into the masks.  Returns the table's flags
// (bit 15: infinity / NaN) and in bits 16.. the number of zeros.
template <int N, int R>
__device__ __forceinline__ uint32_t stage_row(const LutEntryT* lut, BlkT<R>& s, const uint32_t (&w)[N / 4], int r, int pr, int part) {
    uint32_t* op = &s.op[part * N][pr];
    uint32_t acc = 0u, spec = 0u, zeros = 0u, pw[N / 2];
#pragma unroll
    for (int q = 0; q < N; q += 2) {
        const uint2 e0 = *reinterpret_cast<const uint2*>(&lut[(w[q / 4] >> (8 * (q % 4))) & 0xFFu]);
        const uint2 e1 = *reinterpret_cast<const uint2*>(&lut[(w[q / 4] >> (8 * (q % 4) + 8)) & 0xFFu]);
        op[q * R] = e0.x;
        op[(q + 1) * R] = e1.x;
        acc += ((e0.y >> 16 & 1u) << q) + ((e1.y >> 16 & 1u) << (q + 1));
        zeros += (e0.y >> 24) + (e1.y >> 24);
        spec |= e0.y | e1.y;
        pw[q / 2] = __byte_perm(e0.y, e1.y, 0x5410);
    }
    uint16_t* pe = &s.pe[r][part * N];
#pragma unroll
    for (int q = 0; q < N / 8; ++q)
        reinterpret_cast<uint4*>(pe)[q] = make_uint4(pw[4 * q], pw[4 * q + 1], pw[4 * q + 2], pw[4 * q + 3]);
    if (N == 16) {
        reinterpret_cast<uint16_t*>(&s.sgn[pr])[part] = uint16_t(acc);
    } else {
        reinterpret_cast<uint8_t*>(&s.sgn[pr])[part] = uint8_t(acc);
    }
    return (spec & 0x8000u) | zeros << 16;
}

// Decode pass: one CTA decodes one block (R rows of A or columns of B x 32 elements of K) through a 256-entry table of
// 8-byte entries into shared memory and copies it to its place in the scratch array dst[tile][chunk].  Every thread
// takes 16 (R = 128) or 8 (R = 64) consecutive elements of one row.  Rows beyond the matrix repeat the last one (their outputs are
// not stored, but as zeros they would take the rare paths); the elements in front that fill K up to whole chunks decode as zeros.
static_assert(BM == 128 && KC == 32 && NT == 256, "the task split of the decode pass");
template <int R>
struct SideT {
    const unsigned char* src;
    int64_t rows, ld;
    fast::Pad pad;
    BlkT<R>* dst;
};
template <int BASE, int R, bool IS_A, int TH>
__device__ __forceinline__ void decode_t(const DevModel& m, const SideT<R>& side, int F, LutEntryT* lut_a, LutEntryT* lut_b, BlkT<R>& blk, unsigned tile) {
    const int tid = threadIdx.x;
    const FmtDesc fa = fmt_desc(m.fmt_a), fb = fmt_desc(m.fmt_b);
    init_lut_t<BASE>(lut_a, lut_b, fa, fb, F - (fa.mbits + fb.mbits), fa.mbits + 1, tid);
    if (tid == 0) { blk.special = blk.sparse = 0u; blk.pad[0] = blk.pad[1] = 0u; }
    constexpr int N = R * KC / NT;                      // elements per thread: 16 or 8
    const int r = tid % R, part = tid / R;
    const int64_t i = min(int64_t(tile) * R + r, side.rows - 1), k0 = int64_t(blockIdx.x) * KC - side.pad.front;
    uint32_t w[N / 4];
    fast::load_task<fast::EK_LUT8>(w, side.src, i * side.ld, k0 + N * part, side.pad.wide);
    __syncthreads();
    const uint32_t spec = stage_row<N, R>(IS_A ? lut_a : lut_b, blk, w, r, IS_A ? perm_row<TH>(r) : perm_col(r), part);
    if (spec & 0x8000u) atomicOr(&blk.special, 1u);
    // (two rows with less than half of their elements zero meet in a nonzero product; a thread sees a part of a block of L, and
    // parts with less than half of theirs add up to one)
    if ((spec >> 16) * 2 >= uint32_t(N)) atomicOr(&blk.sparse, 1u);
    __syncthreads();
    uint4* out = reinterpret_cast<uint4*>(side.dst + (int64_t(tile) * gridDim.x + blockIdx.x));
    const uint4* in = reinterpret_cast<const uint4*>(&blk);
    for (int q = tid; q < int(sizeof(BlkT<R>) / 16); q += NT) out[q] = in[q];
}
// Both operands in one launch: the tile rows of A, then the tile columns of B (blockIdx.y).
template <int BASE, int TH>
__global__ void __launch_bounds__(NT) trop_decode_kernel(DevModel m, SideT<BM> a, SideT<Geo<TH>::BN> b, int F, unsigned tiles_a) {
    __shared__ __align__(16) LutEntryT lut_a[256];
    __shared__ __align__(16) LutEntryT lut_b[256];
    __shared__ __align__(16) unsigned char blk[sizeof(BlkT<BM>)];
    after_previous();
    if (blockIdx.y < tiles_a) decode_t<BASE, BM, true, TH>(m, a, F, lut_a, lut_b, *reinterpret_cast<BlkT<BM>*>(blk), blockIdx.y);
    else decode_t<BASE, Geo<TH>::BN, false, TH>(m, b, F, lut_a, lut_b, *reinterpret_cast<BlkT<Geo<TH>::BN>*>(blk), blockIdx.y - tiles_a);
}


template <int EK, int L, int F, int RHO, bool PROMOTE, int BASE, int TH>
__global__ void __launch_bounds__(NT, 2) tfdpa_trop_kernel(DevModel m, GemmArgs g, const BlkT<BM>* __restrict__ wa,
                                                           const BlkT<Geo<TH>::BN>* __restrict__ wb) {
    constexpr bool ACC16 = RHO == RHO_RNE_FP16;
    constexpr int NBLK = KC / L;
    static_assert(KC % L == 0 && L % 16 == 0, "a block is one or two k16 matrix instructions");
    static_assert(BASE == 4 || BASE == 5 || BASE == 8, "see pe_shift");
    constexpr int KSUB = pe_sub(BASE) < L ? pe_sub(BASE) : L, NSUB = L / KSUB;        // terms per accumulation of P
    static_assert(!Elem<EK>::SIGNMAG && F <= 13, "8-bit inputs with F <= 13");
    static_assert(RHO == RHO_RZ_E8M13 || RHO == RHO_RNE_FP16, "rho of the F = 13 rows of Table 4");
    using G = Geo<TH>;
    constexpr int BN = G::BN;
    using mask_t = std::conditional_t<(TH * TW > 32), unsigned long long, uint32_t>;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SmemT<TH>& sm = *reinterpret_cast<SmemT<TH>*>(smem_raw);

    const int tid = threadIdx.x;
    const int warp = tid >> 5, lane = tid & 31;
    const int gq = lane >> 2, tq = lane & 3;
    const int row0 = int(blockIdx.y) * BM, col0 = int(blockIdx.x) * BN;        // M, N < 2^31 (checked by the dispatcher)
    const int wr = warp / G::WARPS_C, wc = warp % G::WARPS_C;                  // the warp's part of the CTA tile
    auto row_of = [&](int h) { return wr * G::WROWS + 16 * (h >> 1) + 8 * (h & 1) + gq; };    // inside the CTA tile
    auto col_of = [&](int x) { return wc * 32 + 8 * (x >> 1) + 2 * tq + (x & 1); };
    const FmtDesc fa = fmt_desc(m.fmt_a), fb = fmt_desc(m.fmt_b);
    const int pre = F - (fa.mbits + fb.mbits);
    const int guard = fa.mbits + 1;
    // Exponents are handled as FP32 exponent fields in place (bits 23..30) with whatever lies below as a fraction:
    //   t1 = floor(bits(P) / BASE) + T1_ADD: field e_max + 127 for the largest product (P = 0: a field below that of
    //        the smallest nonzero product); the division is a high multiply, inexact by 2^-30 at most, and P is never
    //        closer than 1 / BASE to the next multiple;
    //   ca = |c|: field Exp(c) + 127.
    // Sum register: (1.5 * 2^23 + S) * 2^(e_max - F), exponent field e + (23 - F).
    constexpr uint32_t MUL = pe_mul(BASE), T1_ADD = uint32_t(127 - (127 + pe_shift(BASE)) / BASE + 2 * PE_CENTER) << 23;
    constexpr uint32_t FIELD = 0x7F800000u, HALF = 0x00400000u;
    constexpr uint32_t RHO_MASK = ACC16 ? 0xFFFFFFFFu : 0xFFFFFC00u;   // RZ-E8M13 of an FP32 word whose exponent stays
    constexpr uint32_t MAGIC_ADD = (uint32_t(23 - F) << 23) | HALF;
    // Below E_LOW no product is nonzero, above E_HIGH the register would overflow (and every product is far below one
    // unit of the accumulator): the result is rho of the accumulator alone.  Such an output rides through pass 2 as a
    // marker KEEP + payload whose unit exceeds every product, so that a term changes it by -1 or not at all, which the
    // sign correction undoes.  FP16 accumulators are never out of range.
    const uint32_t E_LOW = ACC16 ? 0u : uint32_t(127 + 2 - fa.bias - fb.bias) << 23;
    constexpr uint32_t E_HIGH = (241u << 23) - 1u;
    constexpr uint32_t E_KEEP = 243u << 23, KEEP = E_KEEP + MAGIC_ADD;
    static_assert(F == 13 || ACC16, "the kept word is carried as its upper 22 bits");
    // the decoded blocks of this tile row of A and tile column of B, chunk after chunk, land in two buffers by bulk copies
    const int NCH = int((g.K + KC - 1) / KC);
    const BlkT<BM>* src_a = wa + int64_t(blockIdx.y) * NCH;
    const BlkT<BN>* src_b = wb + int64_t(blockIdx.x) * NCH;
    after_previous();
    auto issue = [&](int n) {                              // one thread: both copies of chunk n into buffer n & 1
        unsigned long long* bar = &sm.full[n & 1];
        mbar_expect_tx(bar, uint32_t(sizeof(BlkT<BM>) + sizeof(BlkT<BN>)));
        bulk_load(&sm.a[n & 1], src_a + n, uint32_t(sizeof(BlkT<BM>)), bar);
        bulk_load(&sm.b[n & 1], src_b + n, uint32_t(sizeof(BlkT<BN>)), bar);
    };
    if (tid == 0) {
        sm.error = 0;
        mbar_init(&sm.full[0], 1u);
        mbar_init(&sm.full[1], 1u);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        issue(0);
        if (NCH > 1) issue(1);
    }

    uint32_t cw[TH][TW];
    // The sticky flags wait in shared memory: six registers that only rare events touch (90 bytes of spills with them, 48 without; 4096^3
    // 3828 -> 3746 us).
    volatile unsigned long long* const flags = &sm.flags[0][tid];
    enum { NAN_SEEN = 0, PINF = NT, NINF = 2 * NT };
    flags[NAN_SEEN] = flags[PINF] = flags[NINF] = 0ull;
    auto note = [&](int which, int h, int x) { flags[which] = flags[which] | 1ull << (h * TW + x); };
    float promoted[PROMOTE ? TH : 1][PROMOTE ? TW : 1];
    int big = 0;
#define MMASIM_SP_LOAD const mask_t sp_nan = mask_t(flags[NAN_SEEN]), sp_pinf = mask_t(flags[PINF]), sp_ninf = mask_t(flags[NINF])
#define MMASIM_SP_GET(h, x) (uint32_t((sp_nan >> ((h) * TW + (x))) & 1u) | (uint32_t((sp_pinf >> ((h) * TW + (x))) & 1u) << 1) | (uint32_t((sp_ninf >> ((h) * TW + (x))) & 1u) << 2))
#define MMASIM_SP_WORD(h, x, w) (MMASIM_SP_GET(h, x) ? special_word(((MMASIM_SP_GET(h, x) & 1u) || (MMASIM_SP_GET(h, x) & 6u) == 6u) ? 1 : ((MMASIM_SP_GET(h, x) & 2u) ? 2 : 3), ACC16, true) : (w))
#pragma unroll
    for (int h = 0; h < TH; ++h)
#pragma unroll
        for (int x = 0; x < TW; ++x) {
            const int64_t i = row0 + row_of(h), j = col0 + col_of(x);
            uint32_t w = 0u;
            if (g.C && i < g.M && j < g.N)
                w = ACC16 ? uint32_t(static_cast<const uint16_t*>(g.C)[i * g.ldc + j])
                          : static_cast<const uint32_t*>(g.C)[i * g.ldc + j];
            if (PROMOTE) { promoted[PROMOTE ? h : 0][PROMOTE ? x : 0] = __uint_as_float(w); w = 0u; }
            const AccDec d = decode_acc(w, ACC16);
            if (d.cls != CLS_FINITE) {
                note(d.cls == CLS_NAN ? NAN_SEEN : (d.sign ? NINF : PINF), h, x);
                w = 0u;
            }
            // an FP32 accumulator enters with the bits that its own exponent keeps (units of 2^(Exp(c) - F): the first block's are as
            // coarse or coarser), so that its last mantissa bit is clear; zeros are +0
            if (!ACC16) w = (w & 0x7FFFFFFFu & RHO_MASK) ? w & RHO_MASK : 0u;
            big = big || fabsf(__uint_as_float(w)) > 1.2676506e30f;         // 2^100
            cw[h][x] = w;
        }

    // (the barriers are initialised.)  An output can only leave the range of the sum register where it has no nonzero product, or
    // from a huge C: K products of at most 2^32 each move an accumulator by less than 2^64.
    big = __syncthreads_or(!ACC16 && !PROMOTE && big);
    for (int chunk = 0; chunk < NCH; ++chunk) {
        const int k0 = chunk * KC;                         // (g.K elements end with the last chunk; see fast::front_pad)
        // a wait that runs out is recorded and the chunk computed on whatever is there; every thread sees the flag after
        // the barrier at the end of the chunk, and the CTA leaves together without storing anything
        if (!mbar_wait(&sm.full[chunk & 1], uint32_t(chunk >> 1) & 1u)) *reinterpret_cast<volatile int*>(&sm.error) = 1;
        const BlkT<BM>& sa_blk = sm.a[chunk & 1];
        const BlkT<BN>& sb_blk = sm.b[chunk & 1];
        const bool chunk_special = (sa_blk.special | sb_blk.special) != 0u, chunk_range = big || (sa_blk.sparse | sb_blk.sparse) != 0u;

#pragma unroll 1
        for (int blk = 0; blk < NBLK; ++blk) {
            const int kb = blk * L;
            if (chunk_special) {                           // rare: special-value events of this block (Section 4.2)
                const int64_t first = k0 + kb - fast::front_pad(g.K);
#pragma unroll 1
                for (int h = 0; h < TH; ++h)
#pragma unroll 1
                    for (int x = 0; x < TW; ++x) {
                        const int64_t i = row0 + row_of(h), j = col0 + col_of(x);
                        if (i >= g.M || j >= g.N || first < 0) continue;
                        Special ev;
                        for (int kk = 0; kk < L; ++kk) {
                            const uint32_t xa = decode_elem(fa, raw_elem<EK>(g.A, i * g.lda + first + kk));
                            const uint32_t yb = decode_elem(fb, raw_elem<EK>(g.B, j * g.ldb + first + kk));
                            ev.product(xa, yb);
                        }
                        if (ev.nan) note(NAN_SEEN, h, x);
                        if (ev.pinf) note(PINF, h, x);
                        if (ev.ninf) note(NINF, h, x);
                    }
            }

            // ---- pass 1 on the tensor cores: P = sum_k pe(a_k) pe(b_k), one accumulation per sub-block of KSUB terms,
            // the block's P the integer maximum of their words; one accumulator fragment row (16 x 32 outputs of the
            // warp, two rows of the micro-tile) at a time, followed at once by its sum registers ----
            // (fragments by ldmatrix, the columns' kept for all rows: 12 instead of 96 loads per block of 32)
            constexpr int NK = KSUB >= 16 ? KSUB / 16 : 1, K8 = L / 8;     // matrix instructions per accumulation; tiles of 8 along K
            bool rare = false;
            uint32_t bf[4 * K8];                                           // [column tile j][k8]
#pragma unroll
            for (int q = 0; q < K8; ++q) {
                const int t = 4 * q + (lane >> 3);
                ldmatrix4(&bf[4 * q], &sb_blk.pe[wc * 32 + 8 * (t / K8) + (lane & 7)][kb + 8 * (t % K8)]);
            }
#pragma unroll
            for (int mt = 0; mt < TH / 2; ++mt) {
                uint32_t P[4][4], af[2 * K8];                              // af: [k8][upper / lower 8 rows]
#pragma unroll
                for (int q = 0; q < K8 / 2; ++q)
                    ldmatrix4(&af[4 * q], &sa_blk.pe[wr * G::WROWS + 16 * mt + (lane & 15)][kb + 8 * (2 * q + (lane >> 4))]);
#pragma unroll
                for (int sub = 0; sub < NSUB; ++sub) {
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        float d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
                        for (int ks = 0; ks < NK; ++ks) {
                            const int k8 = (sub * KSUB + 16 * ks) / 8;
                            if constexpr (KSUB >= 16)
                                asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                                             : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                                             : "r"(af[2 * k8]), "r"(af[2 * k8 + 1]), "r"(af[2 * k8 + 2]), "r"(af[2 * k8 + 3]),
                                               "r"(bf[j * K8 + k8]), "r"(bf[j * K8 + k8 + 1]));
                            else
                                asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
                                             : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                                             : "r"(af[2 * k8]), "r"(af[2 * k8 + 1]), "r"(bf[j * K8 + k8]));
                        }
#pragma unroll
                        for (int i = 0; i < 4; ++i)
                            P[j][i] = sub == 0 ? __float_as_uint(d[i]) : max(P[j][i], __float_as_uint(d[i]));
                    }
                }
                // e = max(exponent of the largest product, exponent of the accumulator), kept in the register of P
                uint32_t out_of_range = 0u;
#pragma unroll
                for (int hh = 0; hh < 2; ++hh)
#pragma unroll
                    for (int x = 0; x < TW; ++x) {
                        const int h = 2 * mt + hh;
                        uint32_t& p = P[x >> 1][2 * hh + (x & 1)];
                        const uint32_t t1 = (BASE == 5 ? __umulhi(p, MUL) : (p >> (BASE == 8 ? 3 : 2))) + T1_ADD;
                        uint32_t e;
                        if (ACC16) {
                            // a subnormal FP16 accumulator has the exponent -14, not that of its leading bit.  BASE 6: the
                            // floor also covers c = 0, harmlessly (every nonzero E4M3 product has an exponent of at least
                            // -12); with E5M2 operands products reach down to 2^-28 and a zero accumulator must not count
                            uint32_t ca = __float_as_uint(__half2float(__ushort_as_half((unsigned short)(cw[h][x] & 0x7FFFu))));
                            if (BASE == 8) e = uint32_t(__vimax3_s32(int(t1), int(ca), int(113u << 23)));
                            else { if (ca) ca = max(ca, 113u << 23); e = max(t1, ca); }
                        } else {
                            // |c| and t1 are positive FP32 patterns: their order as numbers is their order as words, and
                            // the absolute value rides on the instruction
                            e = __float_as_uint(fmaxf(__uint_as_float(t1), fabsf(__uint_as_float(cw[h][x]))));
                        }
                        p = e;
                    }
                if (!ACC16 && chunk_range) {
#pragma unroll
                    for (int j = 0; j < 4; ++j)
#pragma unroll
                        for (int i = 0; i < 4; ++i) out_of_range = __viaddmax_u32(P[j][i], 0u - E_LOW, out_of_range);
                }
                if (!ACC16 && chunk_range && out_of_range > E_HIGH - E_LOW) {     // rare: turn the outputs out of range into markers (see above)
                    rare = true;
#pragma unroll
                    for (int hh = 0; hh < 2; ++hh)
#pragma unroll
                        for (int x = 0; x < TW; ++x) {
                            const int h = 2 * mt + hh;
                            uint32_t& p = P[x >> 1][2 * hh + (x & 1)];
                            if (p - E_LOW > E_HIGH - E_LOW) {
                                const uint32_t c = cw[h][x];
                                const uint32_t kept = (c & 0x7FFFFFFFu) ? (c >> 10) : 0u;      // rho(c); an exactly zero sum is +0
                                p = E_KEEP;
                                cw[h][x] = __float_as_uint(__uint2float_rn(kept) * __uint_as_float(uint32_t(E_KEEP >> 23) + uint32_t(23 - F) - 23u << 23));
                            }
                        }
                }
                // the sum register with the accumulator term: floor((c + tiny) / unit); a negative c is one short
#pragma unroll
                for (int hh = 0; hh < 2; ++hh)
#pragma unroll
                    for (int xp = 0; xp < TW / 2; ++xp) {          // two adjacent columns per packed addition
                        const int h = 2 * mt + hh;
                        uint32_t magic[2], cb[2];
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            const uint32_t e = P[xp][2 * hh + q];
                            const uint32_t c = cw[h][2 * xp + q];
                            magic[q] = (e & FIELD) + MAGIC_ADD + (c >> (ACC16 ? 15 : 31));
                            const float cf = ACC16 ? __half2float(__ushort_as_half((unsigned short)c)) : __uint_as_float(c);
                            cb[q] = ACC16 ? __float_as_uint(cf) | 1u : c;
                        }
                        if (!ACC16)
                            asm("{\n\t.reg .b64 a, b, r;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tfma.rm.f32x2 r, a, %6, b;\n\tmov.b64 {%0, %1}, r;\n\t}"
                                : "=r"(cw[h][2 * xp]), "=r"(cw[h][2 * xp + 1]) : "r"(cb[0]), "r"(cb[1]), "r"(magic[0]), "r"(magic[1]), "l"(0x3F8000013F800001ull));
                        else
                        asm("{\n\t.reg .b64 a, b, r;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tadd.rm.f32x2 r, a, b;\n\tmov.b64 {%0, %1}, r;\n\t}"
                            : "=r"(cw[h][2 * xp]), "=r"(cw[h][2 * xp + 1]) : "r"(cb[0]), "r"(cb[1]), "r"(magic[0]), "r"(magic[1]));
                    }
            }
            // ---- pass 2: one fused multiply-add per term, rounding toward minus infinity onto the grid of S; two
            // columns of the micro-tile per instruction (fma.rm.f32x2: lanes (a_h, a_h) x (b_x, b_x+1) + (S_h,x, S_h,x+1)).
            // The columns are walked to and fro: every instruction shares its a or its b with the one before, which saves reads of
            // the register file, the packed instruction's bound beside its own pipe (five 32-bit reads in two cycles that have four):
            // 4096^3 3839 -> 3709 us; b kept for all rows instead of a 3735, to and fro that way 3790 ----
            {
                unsigned long long acc[TH][TW / 2];
#pragma unroll
                for (int h = 0; h < TH; ++h)
#pragma unroll
                    for (int xp = 0; xp < TW / 2; ++xp)
                        asm("mov.b64 %0, {%1, %2};" : "=l"(acc[h][xp]) : "r"(cw[h][2 * xp]), "r"(cw[h][2 * xp + 1]));
#pragma unroll
                for (int kk = kb; kk < kb + L; ++kk) {
                    float oas[TH];
#pragma unroll
                    for (int q = 0; q < TH / 4; ++q) {
                        const float4 oa = *reinterpret_cast<const float4*>(&sa_blk.op[kk][wr * G::WROWS + TH * gq + 4 * q]);
                        oas[4 * q] = oa.x; oas[4 * q + 1] = oa.y; oas[4 * q + 2] = oa.z; oas[4 * q + 3] = oa.w;
                    }
                    const ulonglong2 ob0 = *reinterpret_cast<const ulonglong2*>(&sb_blk.op[kk][wc * 32 + 8 * tq]);
                    const ulonglong2 ob1 = *reinterpret_cast<const ulonglong2*>(&sb_blk.op[kk][wc * 32 + 8 * tq + 4]);
                    const unsigned long long obv[TW / 2] = {ob0.x, ob0.y, ob1.x, ob1.y};
#pragma unroll
                    for (int h = 0; h < TH; ++h) {
                        unsigned long long oav;
                        asm("mov.b64 %0, {%1, %1};" : "=l"(oav) : "f"(oas[h]));
#pragma unroll
                        for (int xq = 0; xq < TW / 2; ++xq) {
                            const int xp = (h & 1) ? TW / 2 - 1 - xq : xq;
                            asm("fma.rm.f32x2 %0, %1, %2, %0;" : "+l"(acc[h][xp]) : "l"(oav), "l"(obv[xp]));
                        }
                    }
                }
#pragma unroll
                for (int h = 0; h < TH; ++h)
#pragma unroll
                    for (int xp = 0; xp < TW / 2; ++xp)
                        asm("mov.b64 {%0, %1}, %2;" : "=r"(cw[h][2 * xp]), "=r"(cw[h][2 * xp + 1]) : "l"(acc[h][xp]));
            }
            // ---- sign corrections and rho ----
            const uint32_t kmask = (L == 32) ? 0xFFFFFFFFu : (((1u << L) - 1u) << kb);
            uint32_t wmax = 0u;
            uint32_t sbv[TW];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint4 u = *reinterpret_cast<const uint4*>(&sb_blk.sgn[wc * 32 + 8 * tq + 4 * q]);
                sbv[4 * q] = u.x; sbv[4 * q + 1] = u.y; sbv[4 * q + 2] = u.z; sbv[4 * q + 3] = u.w;
            }
            auto finish = [&](auto with_markers) {
#pragma unroll
                for (int h = 0; h < TH; ++h) {
                    const uint32_t sa = sa_blk.sgn[wr * G::WROWS + TH * gq + h];
                    uint32_t bitsv[TW], vv[TW];
#pragma unroll
                    for (int x = 0; x < TW; ++x)                   // every negative term fell one unit short:
                        bitsv[x] = cw[h][x] + uint32_t(__popc((sa ^ sbv[x]) & kmask));   // (1.5 * 2^23 + S) * unit
#pragma unroll
                    for (int xp = 0; xp < TW / 2; ++xp)            // S * unit, exact; two columns per packed subtraction
                        asm("{\n\t.reg .b64 a, b, r;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tsub.rn.f32x2 r, a, b;\n\tmov.b64 {%0, %1}, r;\n\t}"
                            : "=r"(vv[2 * xp]), "=r"(vv[2 * xp + 1])
                            : "r"(bitsv[2 * xp]), "r"(bitsv[2 * xp + 1]), "r"((bitsv[2 * xp] & FIELD) | HALF), "r"((bitsv[2 * xp + 1] & FIELD) | HALF));
#pragma unroll
                    for (int x = 0; x < TW; ++x) {
                        const uint32_t bits = bitsv[x];
                        const float v = __uint_as_float(vv[x]);
                        uint32_t w;
                        if (ACC16) { w = uint32_t(__half_as_ushort(__float2half_rn(v))); wmax = max(wmax, w & 0x7FFFu); }
                        else w = __float_as_uint(v);     // RZ-E8M13 is applied where the word leaves the chain (below): the next
                                                         // block's alignment truncates on a grid at least as coarse
                        if (decltype(with_markers)::value && bits >= KEEP) w = (bits - KEEP) << 10;
                        cw[h][x] = w;
                    }
                }
            };
            if (rare) finish(std::true_type{}); else finish(std::false_type{});
            // RNE-FP16 overflowed: +-infinity from now on.  (Not rare: an output that has is likely to again, from zero.  With a load and a
            // store of the flags per output 185 us, flags in registers 171, this way 135: Hopper E4M3 -> FP16 512 x 1024 x 1024.)
            if (ACC16 && wmax >= 0x7C00u) {
                const mask_t seen = mask_t(flags[NAN_SEEN] | flags[PINF] | flags[NINF]);
                mask_t plus = 0, minus = 0;
#pragma unroll
                for (int h = 0; h < TH; ++h)
#pragma unroll
                    for (int x = 0; x < TW; ++x)
                        if ((cw[h][x] & 0x7FFFu) == 0x7C00u) {
                            const mask_t bit = mask_t(1) << (h * TW + x) & ~seen;
                            if (cw[h][x] >> 15) minus |= bit; else plus |= bit;
                            cw[h][x] = 0u;
                        }
                if (plus) flags[PINF] = flags[PINF] | plus;
                if (minus) flags[NINF] = flags[NINF] | minus;
            }
        }
        __syncthreads();                                   // everybody has finished with this buffer
        if (*reinterpret_cast<volatile int*>(&sm.error)) break;
        if (tid == 0 && chunk + 2 < NCH) issue(chunk + 2);
        if (PROMOTE && ((k0 + KC) % int(g.k_chunk)) == 0) {     // FP32 promotion of the partial sum every k_chunk elements
            MMASIM_SP_LOAD;
            if (sp_nan | sp_pinf | sp_ninf) {                  // (rare: the flags of 32 outputs one by one cost as much as a block of 32)
#pragma unroll
                for (int h = 0; h < TH; ++h)
#pragma unroll
                    for (int x = 0; x < TW; ++x) cw[h][x] = MMASIM_SP_WORD(h, x, cw[h][x]);
            }
#pragma unroll
            for (int h = 0; h < TH; ++h)
#pragma unroll
                for (int x = 0; x < TW; ++x) {
                    // (a NaN's word may lose low bits: every NaN becomes the same below)
                    const float part = __uint_as_float(positive_zero(cw[h][x] & RHO_MASK, 0x7FFFFFFFu));
                    float v = __fadd_rn(promoted[PROMOTE ? h : 0][PROMOTE ? x : 0], part);
                    if (v != v) v = __uint_as_float(0x7FFFFFFFu);
                    promoted[PROMOTE ? h : 0][PROMOTE ? x : 0] = v;
                    cw[h][x] = 0u;
                }
            flags[NAN_SEEN] = flags[PINF] = flags[NINF] = 0ull;
        }
    }

    if (*reinterpret_cast<volatile int*>(&sm.error)) {     // a copy never arrived: count it, give the copies in flight one more
        if (tid == 0) {                                    // bounded wait each, and store nothing
            if (g.copy_timeouts) atomicAdd(g.copy_timeouts, 1u);
            mbar_wait(&sm.full[0], 0u);
            mbar_wait(&sm.full[1], 0u);
        }
        return;
    }
    MMASIM_SP_LOAD;
#pragma unroll
    for (int h = 0; h < TH; ++h)
#pragma unroll
        for (int x = 0; x < TW; ++x) {
            const int64_t i = row0 + row_of(h), j = col0 + col_of(x);
            if (i >= g.M || j >= g.N) continue;
            // a chain's last word of magnitude zero is +0 (in between the sign of a zero does not matter: it has no exponent)
            uint32_t w = PROMOTE ? __float_as_uint(promoted[PROMOTE ? h : 0][PROMOTE ? x : 0])
                                 : MMASIM_SP_WORD(h, x, positive_zero(cw[h][x] & RHO_MASK, ACC16 ? 0x7FFFu : 0x7FFFFFFFu));
            if (g.row_scale) {
                float sc = __fmul_rn(g.row_scale[i], g.col_scale[j]);
                if (sc != sc) sc = __uint_as_float(0x7FFFFFFFu);
                float v = __fmul_rn(sc, __uint_as_float(w));
                if (v != v) v = __uint_as_float(0x7FFFFFFFu);
                w = __float_as_uint(v);
            }
            if (ACC16) static_cast<uint16_t*>(g.D)[i * g.ldd + j] = uint16_t(w);
            else static_cast<uint32_t*>(g.D)[i * g.ldd + j] = w;
        }
#undef MMASIM_SP_LOAD
#undef MMASIM_SP_GET
#undef MMASIM_SP_WORD
}

// Where the decoded blocks go: a fixed array (given != nullptr, capacity bytes) or, by default, the call's scratch.
struct Scratch {
    void* given = nullptr;
    size_t capacity = 0;
};

template <int TH>
size_t scratch_bytes_one(const GemmArgs& g) {
    constexpr int BN = Geo<TH>::BN;
    const int64_t tiles_m = (g.M + BM - 1) / BM, tiles_n = (g.N + BN - 1) / BN, nch = (g.K + KC - 1) / KC;
    return size_t(tiles_m * nch) * sizeof(BlkT<BM>) + size_t(tiles_n * nch) * sizeof(BlkT<BN>);
}

template <int EK, int L, int F, int RHO, bool PROMOTE, int BASE, int TH>
cudaError_t launch_one_t(const DevModel& m, const GemmArgs& g, cudaStream_t stream, const Scratch& sc) {
    constexpr int BN = Geo<TH>::BN;
    const size_t sh = sizeof(SmemT<TH>);
    cudaError_t err = cudaFuncSetAttribute(tfdpa_trop_kernel<EK, L, F, RHO, PROMOTE, BASE, TH>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sh));
    if (err != cudaSuccess) return err;
    const int64_t tiles_m = (g.M + BM - 1) / BM, tiles_n = (g.N + BN - 1) / BN, nch = (g.K + KC - 1) / KC;
    const size_t bytes_a = size_t(tiles_m * nch) * sizeof(BlkT<BM>), bytes_b = size_t(tiles_n * nch) * sizeof(BlkT<BN>);
    void* ws = sc.given;
    if (ws) {
        if (bytes_a + bytes_b > sc.capacity) return cudaErrorInvalidValue;      // the caller checked: never reached
    } else {
        if ((err = take_scratch(g, bytes_a + bytes_b, stream, &ws)) != cudaSuccess) return err;
    }
    BlkT<BM>* wa = static_cast<BlkT<BM>*>(ws);
    BlkT<BN>* wb = reinterpret_cast<BlkT<BN>*>(static_cast<unsigned char*>(ws) + bytes_a);
    const SideT<BM> a{static_cast<const unsigned char*>(g.A), g.M, g.lda, fast::pad_of<fast::EK_LUT8>(g.K, g.lda), wa};
    const SideT<BN> b{static_cast<const unsigned char*>(g.B), g.N, g.ldb, fast::pad_of<fast::EK_LUT8>(g.K, g.ldb), wb};
    // (blockIdx.y has 65535 values: what does not fit goes in two launches)
    auto decode = trop_decode_kernel<BASE, TH>;
    if (tiles_m + tiles_n <= 65535) err = enqueue(decode, dim3((unsigned)nch, (unsigned)(tiles_m + tiles_n)), NT, 0, stream, m, a, b, F, unsigned(tiles_m));
    else {
        err = enqueue(decode, dim3((unsigned)nch, (unsigned)tiles_m), NT, 0, stream, m, a, b, F, unsigned(tiles_m));
        if (err == cudaSuccess) err = enqueue(decode, dim3((unsigned)nch, (unsigned)tiles_n), NT, 0, stream, m, a, b, F, 0u);
    }
    if (err == cudaSuccess) err = enqueue(tfdpa_trop_kernel<EK, L, F, RHO, PROMOTE, BASE, TH>, dim3((unsigned)tiles_n, (unsigned)tiles_m, 1), NT, sh, stream, m, g, wa, wb);
    if (sc.given) return err;
    const cudaError_t err2 = give_scratch(g, ws, stream);
    return err != cudaSuccess ? err : err2;
}

// The tall micro-tile (128 x 128 outputs per CTA) or the short one (128 x 64)?  RNE-FP16 and promoted partial sums: the short one, they
// need the registers.  Otherwise what the fullest SM does decides; in given memory always the tall one, so that what fits there does
// not depend on the number of SMs.
inline bool tall_tile(const DevModel& m, const GemmArgs& g, bool given) {
    if (m.rho == RHO_RNE_FP16 || g.k_chunk) return false;
    return given || fast::f13_chunk_us(g, 128) < fast::f13_chunk_us(g, 64);
}
// (of a call in given memory)
inline size_t scratch_bytes(const DevModel& m, const GemmArgs& g) {
    return tall_tile(m, g, true) ? scratch_bytes_one<8>(g) : scratch_bytes_one<4>(g);
}

template <int EK, int L, int F, int RHO, int BASE>
cudaError_t launch_variant_t(const DevModel& m, const GemmArgs& g, cudaStream_t stream, const Scratch& sc) {
    if constexpr (RHO == RHO_RNE_FP16) {
        return launch_one_t<EK, L, F, RHO, false, BASE, 4>(m, g, stream, sc);
    } else {
        if (g.k_chunk) return launch_one_t<EK, L, F, RHO, true, BASE, 4>(m, g, stream, sc);
        if (tall_tile(m, g, sc.given != nullptr)) return launch_one_t<EK, L, F, RHO, false, BASE, 8>(m, g, stream, sc);
        return launch_one_t<EK, L, F, RHO, false, BASE, 4>(m, g, stream, sc);
    }
}

// BASE by the exponent spread of the two element types (see pe_shift): both E4M3, one E5M2, both E5M2.
template <int EK, int L, int F, int RHO>
cudaError_t launch_by_types_t(const DevModel& m, const GemmArgs& g, cudaStream_t stream, const Scratch& sc = Scratch()) {
    const int wide = (m.fmt_a == EF_E5M2) + (m.fmt_b == EF_E5M2);
    if ((m.fmt_a != EF_E4M3 && m.fmt_a != EF_E5M2) || (m.fmt_b != EF_E4M3 && m.fmt_b != EF_E5M2)) return cudaErrorInvalidValue;
    if (wide == 0) return launch_variant_t<EK, L, F, RHO, 8>(m, g, stream, sc);
    if (wide == 1) return launch_variant_t<EK, L, F, RHO, 5>(m, g, stream, sc);
    return launch_variant_t<EK, L, F, RHO, 4>(m, g, stream, sc);
}

}  // namespace trop
}  // namespace mmasim
