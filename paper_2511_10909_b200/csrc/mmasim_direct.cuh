// Small-tile FDPA kernels (T-, ST-, TR-, GTR- and E-FDPA; Algorithms 5-8, 10, 11) that read the raw operands themselves: one
// launch, no scratch memory, any K, any row stride.
//
// When they run.  The large kernels (mmasim_tfdpa_f64.cuh, mmasim_tfdpa_trop.cuh, mmasim_trfdpa_f64.cu, mmasim_efdpa_f64.cu)
// own 64 x 64 (F = 13: 128 x 64 or 128 x 128) outputs per CTA and read operands that a decode pass has laid out.  A matrix with few rows or few
// outputs gives them a handful of CTAs, each of which walks all of K at the full cost of its tile, most of it padding: every
// output is a serial chain over K (the accumulator is rounded after each block), so nothing but more and smaller tiles makes
// such a product faster.
//
// Work decomposition.  The first WR x WC warps of a CTA compute: a warp owns 8 TM x 8 CN outputs as accumulator tiles of the
// FP64 matrix instruction.  The other warps stage: every staging thread copies its share of the raw words of a chunk of 32
// elements of K into its own slots of a ring in shared memory (cp.async, three chunks ahead; the zero fill of a short copy is
// the padding of the last chunk) and decodes them, two chunks ahead of the multiply-adds, into operand planes (doubles), packed
// exponent pairs and sign / nonzero masks.  One barrier per chunk.  An element is decoded once per CTA, that is N / BN (or M / BM)
// times: about twenty instructions per element against the BN (BM) multiply-adds that it feeds.
//
// What bounds it: the chain of a block - exponent maximum, one FP64 addition, L / 4 dependent matrix instructions (26 cycles
// each), correction, rho - in one or two warps per scheduler, and the instructions around it.  So the next block's exponents and
// operand fragments are fetched between this block's matrix instructions, and a chunk runs through blocks without a branch: what
// needs one (subnormal or overflowing results, an inexact E-FDPA sum) is noted, and the chunk done again block by block;
// chunks with infinities or NaNs, of which the staging warps keep masks, go block by block at once.
// Against the large kernels (Hopper FP16): 16 x 4096 x 4096 1027 -> 112 us, 32 x 64 x 1536 353 -> 25, 128 x 2048 x 2048
// 337 -> 128, 656 x 256 x 2688 647 -> 165; against the generic kernel: 1000 x 1111 x 1000 (Ampere BF16) 3590 -> 330 us.  Versions
// on the way, 32 x 64 x 1536: staging by the computing warps 74 us, by warps of their own 45, branches out of the blocks 31;
// further helper warps for the exponent maxima: no gain alone and half the rate in a full grid, not kept.
//
// The arithmetic per block is that of the large kernels (see their headers): the sum register 1.5 * 2^52 * q + S * q, one
// multiply-add rounded toward minus infinity per term, the population count for the negative terms; F = 13 runs on the FP64
// pipe here as well (rho = RZ-E8M13 is a mask on the high word).
#pragma once
#include "mmasim_tfdpa_f64.cuh"

namespace mmasim {
namespace direct {

using fast::EB;
using fast::CB;
using fast::Elem;
using fast::raw_elem;
using fast64::imad;
using fast64::fmax3_abs;
using fast64::c_mul64;
using fast64::G_OFF;

constexpr int KC = 32;
constexpr int KP = KC + 4;              // doubles per row of an operand plane: fragment loads hit sixteen different bank pairs
constexpr int EP = KC / 2 + 4;          // exponent words per row: 80 bytes, 16-byte loads of eight rows hit different banks
constexpr int RING = 4;                 // raw chunks in flight or waiting to be decoded (eight: no gain)
constexpr int BUF = 3;                  // decoded chunks: one being computed, one whose exponents are looked ahead at, one being decoded

// TASK (4 or 8) raw elements as FP32 words of the same values (exact: every format here has at most 10 significand bits and, but for
// the subnormals of BF16 and TF32, a range inside that of the normal FP32 numbers; infinity and NaN stay what they are).
__device__ __forceinline__ uint32_t half_to_fp32(uint32_t h) { return __float_as_uint(__half2float(__ushort_as_half((unsigned short)h))); }
template <int EK, int TASK>
__device__ __forceinline__ void to_fp32(const uint32_t* w, int fmt, uint32_t (&x)[TASK]) {
    if (Elem<EK>::BYTES == 4) {
#pragma unroll
        for (int q = 0; q < TASK; ++q) x[q] = w[q] & ~((1u << Elem<EK>::LOW) - 1u);
    } else if (EK == fast::EK_BF16) {
#pragma unroll
        for (int q = 0; q < TASK; ++q) x[q] = (q & 1) ? w[q / 2] & 0xFFFF0000u : w[q / 2] << 16;
    } else if (EK == fast::EK_F16) {
#pragma unroll
        for (int q = 0; q < TASK; ++q) x[q] = half_to_fp32(w[q / 2] >> (16 * (q & 1)));
    } else {
        // Pairs of FP16 words.  One branch for all of them: a choice of the conversion inside the loop made the staging of eight elements
        // three times that of FP16 ones, and the small tiles of FP8 waited for it (with the blocks left out 20.2 of 21.2 us; Hopper E4M3
        // 64 x 256 x 1024 21.2 -> 15.3 us, Ada E5M2 32 x 384 x 2816 57.0 -> 42.0, CDNA3 E4M3 64 x 256 x 1024 23.7 -> 18.7).
        uint32_t h[TASK / 2];
        auto each = [&](auto convert) {
#pragma unroll
            for (int q = 0; q < TASK / 2; ++q) h[q] = convert((unsigned short)(w[q / 2] >> (16 * (q & 1))));
        };
        if (fmt == EF_E5M2) {                           // an FP16 word without its low byte
#pragma unroll
            for (int q = 0; q < TASK / 2; ++q) h[q] = __byte_perm(w[q / 2], 0u, q & 1 ? 0x3424 : 0x1404);
        } else if (fmt == EF_E4M3) {
            each([](unsigned short p) { uint32_t r; asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(r) : "h"(p)); return r; });
        } else if (fmt == EF_E3M2) {
            each([](unsigned short p) { uint32_t r; asm("cvt.rn.f16x2.e3m2x2 %0, %1;" : "=r"(r) : "h"((unsigned short)(p & 0x3F3Fu))); return r; });
        } else if (fmt == EF_E2M3) {
            each([](unsigned short p) { uint32_t r; asm("cvt.rn.f16x2.e2m3x2 %0, %1;" : "=r"(r) : "h"((unsigned short)(p & 0x3F3Fu))); return r; });
        } else {
            each([](unsigned short p) {                 // E2M1, one code per byte: both codes into one byte
                uint32_t r;
                const unsigned short b = (unsigned short)((p & 0xFu) | ((p >> 4) & 0xF0u));
                asm("{ .reg .b8 lo, hi; mov.b16 {lo, hi}, %1; cvt.rn.f16x2.e2m1x2 %0, lo; }" : "=r"(r) : "h"(b));
                return r;
            });
        }
#pragma unroll
        for (int q = 0; q < TASK; ++q) x[q] = half_to_fp32(h[q / 2] >> (16 * (q & 1)));
    }
}

// The offset bit of a staged B operand: far below the significand of a product, never zero (see mmasim_tfdpa_f64.cuh).
constexpr uint32_t OFFSET_BIT = 1u << 12;

// E-FDPA by the book (Algorithm 6): n elements of one row of A and one row of B, decoded from global memory.
template <int EK>
__device__ __noinline__ uint32_t by_the_book(DevModel m, const void* A, const void* B, int64_t ia, int64_t ib, int n, uint32_t c) {
    const FmtDesc fa = fmt_desc(m.fmt_a), fb = fmt_desc(m.fmt_b);
    uint32_t a[4], b[4];
    for (int k = 0; k < n; ++k) {
        a[k] = decode_elem(fa, raw_elem<EK>(A, ia + k));
        b[k] = decode_elem(fb, raw_elem<EK>(B, ib + k));
    }
    return efdpa_block(a, b, n, c, m);
}

// TASK: consecutive elements of one row per staging task.
template <int EK, int BM, int BN, int PT, int TASK>
struct Smem {
    static constexpr int TPR = KC / TASK;
    static constexpr int ROWS = BM + BN, TASKS = ROWS * TPR, SLOT = TASK * Elem<EK>::BYTES;
    static constexpr int PER = (TASKS + PT - 1) / PT;  // staging tasks per thread
    __align__(16) unsigned char raw[RING][PER * PT * SLOT];     // a thread's own slots: no barrier between its copy and its decode
    __align__(16) double d[BUF][ROWS][KP];              // rows of A, then rows of B
    __align__(16) uint32_t e[BUF][ROWS][EP];            // exponents of elements 2 p (low half) and 2 p + 1 (high half)
    uint32_t sgn[BUF][ROWS], nz[BUF][ROWS];             // bit k: sign / finite and nonzero
    uint32_t nan[BUF][ROWS], inf[BUF][ROWS];            // bit k: NaN (ST: all of them under a NaN scale factor) / infinity
    int special[BUF];                                   // n + 1: chunk n holds an infinity or a NaN (ST: or a NaN scale factor)
    int wild[BUF];                                      // n + 1: chunk n holds a nonzero element outside [2^-48, 2^40)
    uint32_t max_exp[BUF][2];                           // (n + 1) << 11 | largest Exp + EB of chunk n's A and B (TR-FDPA, wide formats)
};

template <int UNIT>
__device__ __forceinline__ void copy_async(void* dst, const void* src, int valid) {      // `valid` bytes and zeros up to UNIT
    const uint32_t d = uint32_t(__cvta_generic_to_shared(dst));
    if (UNIT == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" :: "r"(d), "l"(src), "r"(valid) : "memory");
    else asm volatile("cp.async.ca.shared.global [%0], [%1], %3, %2;" :: "r"(d), "l"(src), "r"(valid), "n"(UNIT) : "memory");
}

// Resident CTAs asked for: 80 registers per thread for warps of one or two tiles, 128 for larger ones and for the fragments of
// blocks of 32.
__host__ __device__ constexpr int min_ctas(int tiles, int L, int warps) {
    return (tiles <= 2 && L <= 16 ? 24 : 16) / warps > 0 ? (tiles <= 2 && L <= 16 ? 24 : 16) / warps : 1;
}

// unit_a / unit_b: bytes per asynchronous copy that the row starts allow (the natural 16, or 8 for 8-bit elements; 4), or 0:
// rows at odd addresses, read element by element in the decode step.
template <int FAM, int EK, int L, int RHO, bool PROMOTE, int TM, int CN, int WR, int WC, int PW, int TASK>
__device__ __forceinline__ void direct_tile(const DevModel& m, const GemmArgs& g, int unit_a, int unit_b, int64_t row0, int64_t col0) {
    static_assert(FAM == FAM_T || FAM == FAM_ST || FAM == FAM_TR || FAM == FAM_GTR || FAM == FAM_E, "FDPA families");
    constexpr bool T = FAM == FAM_T || FAM == FAM_ST, GTR = FAM == FAM_GTR, E = FAM == FAM_E;
    constexpr bool ACC16 = RHO == RHO_RNE_FP16, E8M13 = RHO == RHO_RZ_E8M13;
    constexpr int TN = 2 * CN, BM = 8 * TM * WR, BN = 8 * CN * WC, NTH = 32 * PW;     // NTH: the staging threads
    constexpr int BYTES = Elem<EK>::BYTES;
    constexpr bool TOP = FAM == FAM_TR && (EK == fast::EK_BF16 || EK == fast::EK_TF32);     // products that may reach 2^128
    // results are tested for the range of normal FP32 numbers only where they can leave it (see mmasim_tfdpa_f64.cuh); the small tiles
    // wait for the chain of a block, not for the integer pipe: a second body of code gained and lost 2 - 6 % from size to size
    constexpr bool TAMEABLE = FAM == FAM_T && !ACC16 && TM * CN >= 4;
    static_assert(TM * TN <= 16 && KC % L == 0 && TASK == 8, "sticky flags are 16-bit masks; blocks tile the chunk; a task fills a byte of the masks");
    constexpr int NC = WR * WC, NBLK = KC / L;
    using SM = Smem<EK, BM, BN, NTH, TASK>;
    constexpr int TPR = SM::TPR;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SM& sm = *reinterpret_cast<SM*>(smem_raw);

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool stager = warp >= NC;                     // the first WR * WC warps compute, the others decode
    const int tid = int(threadIdx.x) - 32 * NC;         // (of a staging thread)
    const int wr = warp / WC, wc = warp % WC, gq = lane >> 2, tq = lane & 3;
    auto row_at = [&](int r) { return wr * 8 * TM + 8 * r + gq; };                       // inside the CTA tile
    auto col_at = [&](int c) { return wc * 8 * CN + 8 * (c >> 1) + 2 * tq + (c & 1); };
    const FmtDesc fa = fmt_desc(m.fmt_a), fb = fmt_desc(m.fmt_b);
    constexpr bool WIDE = EK == fast::EK_BF16 || EK == fast::EK_TF32;       // subnormals below the normal FP32 range
    const uint32_t min_a = uint32_t(128 - fa.bias), min_b = uint32_t(128 - fb.bias);     // FP32 field of the smallest normal number
    const int K = int(g.K), NCH = (K + KC - 1) / KC;

    // ---- staging: task u = row * TPR + h takes elements 8 h .. 8 h + 7 of a row; consecutive threads, consecutive addresses ----
    const unsigned char* src[SM::PER];                  // the row's next eight elements
    int left[SM::PER];                                  // bytes from there to the end of the row (rows beyond the matrix: none)
    auto init_tasks = [&] {
#pragma unroll
        for (int it = 0; it < SM::PER; ++it) {
            const int task = it * NTH + tid, r = task / TPR, h = task % TPR;
            const bool is_a = r < BM;
            const int64_t grow = is_a ? row0 + r : col0 + (r - BM);
            const bool inside = task < SM::TASKS && grow < (is_a ? g.M : g.N);
            src[it] = static_cast<const unsigned char*>(is_a ? g.A : g.B) + (inside ? (grow * (is_a ? g.lda : g.ldb) + h * TASK) * BYTES : 0);
            left[it] = inside ? (K - h * TASK) * BYTES : 0;
        }
    };
    auto issue = [&](int n) {                           // every chunk in turn: the next raw words of the thread's tasks
#pragma unroll
        for (int it = 0; it < SM::PER; ++it) {
            const int task = it * NTH + tid;
            const int unit = task / TPR < BM ? unit_a : unit_b;
            constexpr int NATURAL = SM::SLOT < 16 ? SM::SLOT : 16;
            unsigned char* dst = &sm.raw[n % RING][task * SM::SLOT];
            if (SM::TASKS % NTH && task >= SM::TASKS) break;
            if (n < NCH) {
                if (unit == NATURAL) {
#pragma unroll
                    for (int b = 0; b < SM::SLOT; b += NATURAL) {
                        const int v = min(NATURAL, max(left[it] - b, 0));
                        copy_async<NATURAL>(dst + b, v ? src[it] + b : static_cast<const unsigned char*>(g.A), v);
                    }
                } else if (unit) {
#pragma unroll
                    for (int b = 0; b < SM::SLOT; b += 4) {
                        const int v = min(4, max(left[it] - b, 0));
                        copy_async<4>(dst + b, v ? src[it] + b : static_cast<const unsigned char*>(g.A), v);
                    }
                }
            }
            src[it] += KC * BYTES;
            left[it] -= KC * BYTES;
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    };
    auto stage = [&](int n) {                           // decode the thread's own raw words of chunk n into buffer n mod 3
        const int buf = n % BUF;
        const bool marked = sm.special[buf] != 0;
        uint32_t spec = 0u, wild = 0u, top_a = 0u, top_b = 0u;
#pragma unroll
        for (int it = 0; it < SM::PER; ++it) {
            const int task = it * NTH + tid;
            if (SM::TASKS % NTH && task >= SM::TASKS) break;
            const int r = task / TPR, h = task % TPR;
            const bool is_a = r < BM;
            const int64_t grow = is_a ? row0 + r : col0 + (r - BM);
            const bool inside = grow < (is_a ? g.M : g.N);
            constexpr int W = SM::SLOT / 4;                 // (8-bit elements: one word of four)
            uint32_t w[W];
            const uint32_t* slot = reinterpret_cast<const uint32_t*>(&sm.raw[n % RING][(it * NTH + tid) * SM::SLOT]);
#pragma unroll
            for (int q = 0; q < W; ++q) w[q] = slot[q];
            if ((is_a ? unit_a : unit_b) == 0) {
                const int k = n * KC + h * TASK;
                const int64_t at = grow * (is_a ? g.lda : g.ldb) + k;
#pragma unroll
                for (int q = 0; q < W; ++q) w[q] = 0u;
#pragma unroll
                for (int q = 0; q < TASK; ++q)
                    if (inside && k + q < K) w[q * BYTES / 4] |= raw_elem<EK>(is_a ? g.A : g.B, at + q) << (8 * ((q * BYTES) % 4));
            }
            uint32_t sc20 = 0u, sc_exp = uint32_t(EB - 127);
            bool sc_nan = false;
            if (FAM == FAM_ST && inside) {              // the row's E8M0 scale factor of this block of 32 multiplies its operands, exactly
                const uint32_t byte = is_a ? g.sfa[grow * g.ld_sfa + n] : g.sfb[grow * g.ld_sfb + n];
                sc20 = uint32_t(int(byte) - 127) << 20;
                sc_exp += byte - 127u;
                sc_nan = byte == 0xFFu;
            }
            uint32_t x[TASK], sbits = 0u, nbits = 0u, nans = 0u, infs = 0u, ep[TASK / 2], top = 0u, low = 0xFFFFFFFFu;
            to_fp32<EK, TASK>(w, is_a ? m.fmt_a : m.fmt_b, x);
            const uint32_t off = (E || is_a) ? 0u : OFFSET_BIT;
            const uint32_t min_field = is_a ? min_a : min_b;
            double v[TASK];
#pragma unroll
            for (int q = TASK - 1; q >= 0; --q) {
                const uint32_t mag = x[q] & 0x7FFFFFFFu;
                top = max(top, mag);
                if (WIDE) low = min(low, mag - 1u);
                const bool nonzero = mag != 0u;
                // an FP32 word as a double: the fields three bits down, the bias exchanged
                const uint32_t hi = nonzero ? ((mag >> 3) + (896u << 20) + sc20) | (x[q] & 0x80000000u) : 0u;
                v[q] = __hiloint2double(int(hi), int(nonzero ? off : 0u));
                // unnormalised exponents: a subnormal element counts with that of the smallest normal number
                const uint32_t expb = nonzero ? max(mag >> 23, min_field) + sc_exp : 0u;
                sbits = __funnelshift_l(x[q], sbits, 1);
                nbits = __funnelshift_l(mag + 0x7FFFFFFFu, nbits, 1);
                if (q & 1) ep[q / 2] = expb << 16; else ep[q / 2] |= expb;
            }
            if (WIDE && TAMEABLE) wild |= uint32_t(top >= uint32_t(127 + 40) << 23) | uint32_t(low < (uint32_t(127 - 48) << 23) - 1u);
            if (top >= 0x7F800000u || (WIDE && low < 0x007FFFFFu) || sc_nan) {
                // rare: infinities and NaNs are staged as zeros without exponent, like the rows of a NaN scale factor; an FP32
                // subnormal is a small integer times 2^-149
#pragma unroll
                for (int q = 0; q < TASK; ++q) {
                    const uint32_t mag = x[q] & 0x7FFFFFFFu;
                    const bool none = mag >= 0x7F800000u || sc_nan;
                    if (none) {
                        v[q] = 0.0;
                        nbits &= ~(1u << q);
                        ep[q / 2] &= (q & 1) ? 0x0000FFFFu : 0xFFFF0000u;
                        if (mag == 0x7F800000u && !sc_nan) infs |= 1u << q; else nans |= 1u << q;
                        spec = 1u;
                    } else if (WIDE && mag - 1u < 0x007FFFFFu) {
                        const double d = __dmul_rn(__uint2double_rn(mag), __hiloint2double((1023 - 149) << 20, 0));
                        v[q] = __hiloint2double(__double2hiint(d) | int(x[q] & 0x80000000u), int(off));
                    }
                }
            }
            if (TOP) {
                uint32_t t = 0u;
#pragma unroll
                for (int q = 0; q < TASK / 2; ++q) t = __vmaxu2(t, ep[q]);
                t = max(t & 0xFFFFu, t >> 16);
                if (is_a) top_a = max(top_a, t); else top_b = max(top_b, t);
            }
            double* dp = sm.d[buf][r];
            if (GTR) {                                  // even elements of a block of 16 first, then the odd ones
                double* eo = dp + (h * TASK / 16) * 16 + (h * TASK % 16) / 2;
#pragma unroll
                for (int q = 0; q < TASK; q += 4) {
                    *reinterpret_cast<double2*>(eo + q / 2) = make_double2(v[q], v[q + 2]);
                    *reinterpret_cast<double2*>(eo + 8 + q / 2) = make_double2(v[q + 1], v[q + 3]);
                }
            } else {
#pragma unroll
                for (int q = 0; q < TASK; q += 2) *reinterpret_cast<double2*>(dp + h * TASK + q) = make_double2(v[q], v[q + 1]);
            }
            if (!E) {
                *reinterpret_cast<uint4*>(&sm.e[buf][r][h * 4]) = make_uint4(ep[0], ep[1], ep[2], ep[3]);
                reinterpret_cast<uint8_t*>(&sm.sgn[buf][r])[h] = uint8_t(sbits);
                reinterpret_cast<uint8_t*>(&sm.nz[buf][r])[h] = uint8_t(nbits);
            }
            if (marked || (nans | infs)) {              // (zero until the buffer first holds a special value)
                reinterpret_cast<uint8_t*>(&sm.nan[buf][r])[h] = uint8_t(nans);
                reinterpret_cast<uint8_t*>(&sm.inf[buf][r])[h] = uint8_t(infs);
            }
        }
        if (spec) sm.special[buf] = n + 1;
        if (wild) sm.wild[buf] = n + 1;
        if (TOP) {
            if (top_a) atomicMax(&sm.max_exp[buf][0], uint32_t(n + 1) << 11 | top_a);
            if (top_b) atomicMax(&sm.max_exp[buf][1], uint32_t(n + 1) << 11 | top_b);
        }
    };

    // ---- the accumulators: doubles (T: bit 0 of the low word set, see the large kernel), or the plain word (E-FDPA) ----
    auto state_of = [](uint32_t w) {
        double d = 0.0;
        if (ACC16) { if (w & 0x7FFFu) d = double(__half2float(__ushort_as_half((unsigned short)w))); }
        else if (w & 0x7FFFFFFFu) d = double(__uint_as_float(w));
        return __hiloint2double(__double2hiint(d), __double2loint(d) | 1);
    };
    auto rz_word = [](double v) {                       // rho of a value below 2^128 (2^16) as a word
        if (ACC16) return uint32_t(__half_as_ushort(__double2half(v)));
        return __float_as_uint(__double2float_rz(v)) & (E8M13 ? 0xFFFFFC00u : 0xFFFFFFFFu);
    };
    auto clean = [](double st) { return __hiloint2double(__double2hiint(st), __double2loint(st) & ~1); };
    constexpr int EXP_LOW = ACC16 ? -14 : -126, EXP_TOP = ACC16 ? 16 : 128;
    double cs[E ? 1 : TM][E ? 1 : TN];
    uint32_t cw[E ? TM : 1][E ? TN : 1];
    float promoted[PROMOTE ? TM : 1][PROMOTE ? TN : 1];
    bool subnormal = false;                             // T: some accumulator is a nonzero subnormal: its Exp is EXP_LOW, not its field
    uint32_t sp_nan = 0u, sp_pinf = 0u, sp_ninf = 0u;   // per output (bit r * TN + c)
    auto set_state = [&](int r, int c, uint32_t w) {    // from a finite word
        if (E) { cw[E ? r : 0][E ? c : 0] = w; return; }
        double& st = cs[E ? 0 : r][E ? 0 : c];
        if (!T) { st = double(__uint_as_float(w)); return; }
        st = state_of(w);
        subnormal = subnormal || (ACC16 ? ((w & 0x7C00u) == 0u && (w & 0x03FFu) != 0u) : ((w & 0x7F800000u) == 0u && (w & 0x007FFFFFu) != 0u));
    };
    // (exponent sum + CB) << 20 becomes the exponent field e_max + 1023 (T), or that of the constant 1.5 * 2^52 * 2^(e_max - F) (TR)
    const int key_add = T ? -(1 << 20) : (1023 + 52 - m.F - CB) << 20;
    for (int i = threadIdx.x; i < BUF * (BM + BN); i += 32 * (NC + PW)) (&sm.nan[0][0])[i] = (&sm.inf[0][0])[i] = 0u;
    if (threadIdx.x < BUF) { sm.special[threadIdx.x] = sm.wild[threadIdx.x] = 0; sm.max_exp[threadIdx.x][0] = sm.max_exp[threadIdx.x][1] = 0u; }
    __syncthreads();
    if (stager) {
        // during chunk n, which looks ahead at the exponents of chunk n + 1, chunk n + 2 is decoded
        init_tasks();
        issue(0);
        issue(1);
        issue(2);
        for (int n = 0; n < NCH; ++n) {
            issue(n + 3);
            asm volatile("cp.async.wait_group 3;" ::: "memory");        // chunk n has landed (three more may be in flight)
            stage(n);
            if (n >= 1) __syncthreads();
        }
        __syncthreads();
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        return;
    }
#pragma unroll
    for (int r = 0; r < TM; ++r)
#pragma unroll
        for (int c = 0; c < TN; ++c) {
            const int64_t i = row0 + row_at(r), j = col0 + col_at(c);
            // outputs of the padding run at 1.0: like zero accumulators they meet zero products only, but stay out of the rare paths
            const bool inside = i < g.M && j < g.N;
            uint32_t w = inside ? 0u : (ACC16 ? 0x3C00u : 0x3F800000u);
            if (g.C && inside)
                w = ACC16 ? uint32_t(static_cast<const uint16_t*>(g.C)[i * g.ldc + j]) : static_cast<const uint32_t*>(g.C)[i * g.ldc + j];
            if (PROMOTE) { promoted[PROMOTE ? r : 0][PROMOTE ? c : 0] = __uint_as_float(w); w = 0u; }
            if (E) { cw[E ? r : 0][E ? c : 0] = w; continue; }
            const AccDec d = decode_acc(w, ACC16);
            if (d.cls != CLS_FINITE) {
                const uint32_t bit = 1u << (r * TN + c);
                if (d.cls == CLS_NAN) sp_nan |= bit; else if (d.sign) sp_ninf |= bit; else sp_pinf |= bit;
                w = 0u;
            }
            set_state(r, c, w);
        }
    auto output_word = [&](int r, int c) {              // the word that leaves a chain of blocks
        if (E) return cw[E ? r : 0][E ? c : 0];
        const uint32_t bit = r * TN + c;
        const uint32_t nan = (sp_nan >> bit) & 1u, pinf = (sp_pinf >> bit) & 1u, ninf = (sp_ninf >> bit) & 1u;
        if (nan | pinf | ninf) return special_word((nan || (pinf && ninf)) ? 1 : (pinf ? 2 : 3), ACC16, T);
        const double st = cs[E ? 0 : r][E ? 0 : c];
        if (!T) return __float_as_uint(__double2float_rn(st));
        return positive_zero(rz_word(clean(st)), ACC16 ? 0x7FFFu : 0x7FFFFFFFu);
    };

    __syncthreads();                                    // chunks 0 and 1 are decoded
    const int arow = wr * 8 * TM, brow = BM + wc * 8 * CN;
    // What a block needs from shared memory is in registers when the block begins: its product exponents and its operand
    // fragments (lane (g, t) of the matrix instruction holds element (row g, k t)) are fetched for the next block between the
    // matrix instructions of the one before, so that the chain from accumulator to accumulator is arithmetic alone.
    constexpr int NKS = (L + 3) / 4;
    double af[NKS][TM], bf[NKS][CN];
    uint32_t emp[E ? 1 : TM][E ? 1 : TN];               // largest Exp(a) + Exp(b): even elements in the low lane, odd ones in the high lane
    const bool used = L >= 4 || tq < 2;                 // blocks of two leave half of the matrix instruction empty
    auto fetch_fragments = [&](int b, int kb, int ks) {
#pragma unroll
        for (int r = 0; r < TM; ++r) af[ks][r] = L >= 4 ? sm.d[b][arow + 8 * r + gq][kb + 4 * ks + tq] : (used ? sm.d[b][arow + 8 * r + gq][kb + (tq & 1)] : 0.0);
#pragma unroll
        for (int j = 0; j < CN; ++j) bf[ks][j] = L >= 4 ? sm.d[b][brow + 8 * j + gq][kb + 4 * ks + tq] : (used ? sm.d[b][brow + 8 * j + gq][kb + (tq & 1)] : 0.0);
    };
    auto fetch_exponents = [&](int b, int kb, int ks) { // pairs 2 ks, 2 ks + 1 of the block
        if (E) return;
        uint2 ea[TM], eb[TN];
#pragma unroll
        for (int r = 0; r < TM; ++r) ea[r] = *reinterpret_cast<const uint2*>(&sm.e[b][row_at(r)][kb / 2 + 2 * ks]);
#pragma unroll
        for (int c = 0; c < TN; ++c) eb[c] = *reinterpret_cast<const uint2*>(&sm.e[b][BM + col_at(c)][kb / 2 + 2 * ks]);
#pragma unroll
        for (int r = 0; r < TM; ++r)
#pragma unroll
            for (int c = 0; c < TN; ++c) {
                uint32_t& m2 = emp[E ? 0 : r][E ? 0 : c];
                m2 = __viaddmax_s16x2(ea[r].y, eb[c].y, __viaddmax_s16x2(ea[r].x, eb[c].x, ks == 0 ? 0u : m2));
            }
    };
#pragma unroll
    for (int ks = 0; ks < NKS; ++ks) { fetch_fragments(0, 0, ks); fetch_exponents(0, 0, ks); }

    // One block, from accumulator to accumulator: elements kb .. kb + L - 1 of the decoded chunk `buf`; `nb`, `nkb`: where the
    // next block lives (behind the last one: anything decoded, the values are not used).  The plain form has no branch, keeps
    // no flags and only notes that some result needs more; the careful form does everything, block by block.
    constexpr int EXPF = 0x7FF00000, HALF = 0x00080000, LOW31 = int(0x80000000u);
    constexpr uint32_t LOWHI = uint32_t(1023 + EXP_LOW) << 20, TOPHI = uint32_t(1023 + EXP_TOP) << 20;
    uint32_t negm[E ? 1 : TM][E ? 1 : TN];              // bit k: product k of the chunk is negative and nonzero
    uint32_t seen_max = 0u, seen_min = 0xFFFFFFFFu;     // T: twice the high words of the results, and the same minus one
    float seen_top = 0.f;                               // TR, GTR: the largest magnitude
    bool rare = false;                                  // the chunk holds special values, or products that may reach 2^128
    uint32_t slow = 0u;                                 // E: outputs whose block sum needs the exact route
    auto mma = [&](double (&acc)[TM][TN], int ks, int nb, int nkb) {    // four terms per output, each rounded toward minus infinity
#pragma unroll
        for (int r = 0; r < TM; ++r)
#pragma unroll
            for (int j = 0; j < CN; ++j)
                asm volatile("mma.sync.aligned.m8n8k4.row.col.rm.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
                             : "+d"(acc[r][2 * j]), "+d"(acc[r][2 * j + 1]) : "d"(af[ks][r]), "d"(bf[ks][j]));
        fetch_fragments(nb, nkb, ks);
        fetch_exponents(nb, nkb, ks);
    };
    enum { PLAIN = 0, CAREFULLY, IN_RANGE };
    auto block = [&](int kb, int nb, int nkb, auto mode) {
        constexpr bool CAREFUL = decltype(mode)::value == CAREFULLY, TAME = decltype(mode)::value == IN_RANGE;
        const uint32_t kmask = (L == 32) ? 0xFFFFFFFFu : (((1u << (L % 32)) - 1u) << kb);
        if constexpr (T) {
            // blocks of at most 8 terms, and F = 13: the sum register's low word, started at 2^31, never carries
            constexpr bool NARROW = L <= 8 || E8M13;
            // blocks of 32 with few outputs per thread: the second half of the terms in a register of its own (the sums are
            // exact integers), half the chain of dependent matrix instructions
            constexpr bool SPLIT = L == 32 && TM * CN == 1;
            const int km = ((52 << 20) | HALF) - (m.F << 20);
            double acc[TM][TN], acc2[SPLIT ? TM : 1][SPLIT ? TN : 1];
            int mhi[TM][TN];
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int c = 0; c < TN; ++c) {
                    const double st = cs[r][c];
                    const int hi = __double2hiint(st);
                    const int klo = imad(int(emp[r][c]), c_mul64[0], key_add), khi = imad(int(emp[r][c]), c_mul64[1], key_add);
                    int keyc = hi;
                    if (CAREFUL) { const double x = fabs(clean(st)); if (x != 0.0 && x < (ACC16 ? 6.103515625e-05 : 1.1754943508222875e-38)) keyc = int(LOWHI); }
                    mhi[r][c] = (fmax3_abs(keyc, klo, khi) & EXPF) + km;
                    const int mlo = NARROW ? int(__funnelshift_l(uint32_t(hi), 0x40000000u, 1)) : int(uint32_t(hi) >> 31);
                    acc[r][c] = __dadd_rd(st, __hiloint2double(mhi[r][c], mlo));
                    if (SPLIT) acc2[SPLIT ? r : 0][SPLIT ? c : 0] = __hiloint2double(mhi[r][c], 0);
                }
            if constexpr (SPLIT) {
#pragma unroll
                for (int ks = 0; ks < NKS / 2; ++ks) { mma(acc, ks, nb, nkb); mma(acc2, ks + NKS / 2, nb, nkb); }
            } else {
#pragma unroll
                for (int ks = 0; ks < NKS; ++ks) mma(acc, ks, nb, nkb);
            }
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int c = 0; c < TN; ++c) {
                    const int nneg = __popc(negm[r][c] & kmask);
                    double v;
                    if (NARROW)
                        v = __dsub_rn(__hiloint2double(__double2hiint(acc[r][c]), __double2loint(acc[r][c]) + nneg), __hiloint2double(mhi[r][c], LOW31));
                    else
                        v = __dsub_rn(__longlong_as_double(__double_as_longlong(acc[r][c]) + (long long)nneg), __hiloint2double(mhi[r][c], 0));
                    if constexpr (SPLIT) v = __dadd_rn(v, __dsub_rn(acc2[r][c], __hiloint2double(mhi[r][c], 0)));
                    if (ACC16) asm("cvt.f64.f16 %0, %1;" : "=d"(v) : "h"(__half_as_ushort(__double2half(v))));
                    if (!TAME) {
                        const uint32_t twice = uint32_t(imad(__double2hiint(v), c_mul64[6], 0));      // (the sign leaves at the top)
                        seen_max = max(seen_max, twice);
                        seen_min = __viaddmin_u32(twice, 0xFFFFFFFFu, seen_min);                      // (zero wraps: it needs nothing)
                    }
                    if (ACC16) cs[r][c] = __hiloint2double(__double2hiint(v), __double2loint(v) | 1);
                    else if (E8M13) cs[r][c] = __hiloint2double(__double2hiint(v) & int(0xFFFFFF80u), 1);
                    else cs[r][c] = __hiloint2double(__double2hiint(v), (__double2loint(v) & int(0xE0000000u)) | 1);
                }
            if (CAREFUL) {                              // subnormal results and overflow
                subnormal = false;
#pragma unroll
                for (int r = 0; r < TM; ++r)
#pragma unroll
                    for (int c = 0; c < TN; ++c) {
                        const double v = clean(cs[r][c]);
                        const uint32_t bit = 1u << (r * TN + c);
                        if (fabs(v) >= (ACC16 ? 65536.0 : 3.402823669209385e38)) {
                            if (!((sp_nan | sp_pinf | sp_ninf) & bit)) { if (v < 0.0) sp_ninf |= bit; else sp_pinf |= bit; }
                            set_state(r, c, 0u);
                        } else if (fabs(v) < (ACC16 ? 6.103515625e-05 : 1.1754943508222875e-38)) {
                            set_state(r, c, rz_word(v));
                        }
                    }
            }
        } else if constexpr (!E) {
            // ---- TR- / GTR-FDPA: the sum registers start as bare constants; the accumulator joins in the merge ----
            double t0[TM][TN], t1[GTR ? TM : 1][GTR ? TN : 1];
            int m0[TM][TN], m1[GTR ? TM : 1][GTR ? TN : 1];
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int c = 0; c < TN; ++c) {
                    const int klo = imad(int(emp[r][c]), c_mul64[0], key_add), khi = imad(int(emp[r][c]), c_mul64[1], key_add);
                    m0[r][c] = ((GTR ? klo : max(klo, khi)) & EXPF) | HALF;
                    t0[r][c] = __hiloint2double(m0[r][c], LOW31);
                    if (GTR) {
                        m1[GTR ? r : 0][GTR ? c : 0] = (khi & EXPF) | HALF;
                        t1[GTR ? r : 0][GTR ? c : 0] = __hiloint2double(m1[GTR ? r : 0][GTR ? c : 0], LOW31);
                    }
                }
            if constexpr (GTR) {
#pragma unroll
                for (int ks = 0; ks < 2; ++ks) { mma(t0, ks, nb, nkb); mma(t1, ks + 2, nb, nkb); }     // (the plane holds the even elements first)
            } else {
#pragma unroll
                for (int ks = 0; ks < NKS; ++ks) mma(t0, ks, nb, nkb);
            }
            const uint32_t k_c = uint32_t(((52 - m.F2) << 20) | HALF) + 1u;
            constexpr uint32_t k_gtr = (53u << 20) + 1u;
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int c = 0; c < TN; ++c) {
                    const uint32_t neg = negm[r][c] & kmask;
                    auto value = [&](double u, int mh, int n) { return __dsub_rn(__hiloint2double(__double2hiint(u), __double2loint(u) + n), __hiloint2double(mh, LOW31)); };
                    double Y;
                    int m0hi = m0[r][c];
                    if constexpr (GTR) {
                        const double ye = value(t0[r][c], m0[r][c], __popc(neg & 0x55555555u)), yo = value(t1[r][c], m1[r][c], __popc(neg & 0xAAAAAAAAu));
                        m0hi = max(m0[r][c], m1[r][c]);
                        const double mm = __hiloint2double(m0hi, 0);
                        Y = __dsub_rn(__dadd_rd(yo, __dadd_rd(ye, mm)), mm);
                    } else Y = value(t0[r][c], m0[r][c], __popc(neg));
                    double st = cs[r][c];
                    const uint32_t ecm = __viaddmax_u32(uint32_t(__double2hiint(st) & EXPF), 0xFFFFFFFFu, LOWHI - 1u);
                    if (GTR && int(ecm + k_gtr) < m0hi - HALF) st = 0.0;                // special truncation (Algorithm 11 Step 4)
                    const double Mv = __hiloint2double(__viaddmax_s32(int(ecm), int(k_c), m0hi), 0);
                    const float w = __double2float_rn(__dsub_rn(__dadd_rd(Y, __dadd_rd(st, Mv)), Mv));
                    seen_top = fmaxf(fabsf(w), seen_top);
                    cs[r][c] = double(w);
                    if (CAREFUL && fabsf(w) > 3.4028234663852886e38f) {                 // RNE-FP32 overflowed
                        const uint32_t bit = 1u << (r * TN + c);
                        if (!((sp_nan | sp_pinf | sp_ninf) & bit)) { if (w < 0.f) sp_ninf |= bit; else sp_pinf |= bit; }
                        cs[r][c] = 0.0;
                    }
                }
        } else {
            // ---- E-FDPA: two chains, rounded toward minus and plus infinity: equal if and only if exact ----
            double lo[TM][TN], hi[TM][TN];
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int j = 0; j < CN; ++j) {
#pragma unroll
                    for (int q = 0; q < 2; ++q)         // adding +0 turns a -0 into +0
                        lo[r][2 * j + q] = hi[r][2 * j + q] = __dadd_rn(double(__uint_as_float(cw[r][2 * j + q])), 0.0);
                    asm volatile("mma.sync.aligned.m8n8k4.row.col.rm.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
                                 : "+d"(lo[r][2 * j]), "+d"(lo[r][2 * j + 1]) : "d"(af[0][r]), "d"(bf[0][j]));
                    asm volatile("mma.sync.aligned.m8n8k4.row.col.rp.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
                                 : "+d"(hi[r][2 * j]), "+d"(hi[r][2 * j + 1]) : "d"(af[0][r]), "d"(bf[0][j]));
                }
            fetch_fragments(nb, nkb, 0);
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int c = 0; c < TN; ++c) {
                    // the same double (bit for bit): the exact sum; block by block also bounds that round to one word, which leave no other for
                    // the sum between them (a zero only if both are zero, and no NaN)
                    bool fits = lo[r][c] == hi[r][c] && __double2hiint(lo[r][c]) == __double2hiint(hi[r][c]);
                    if (CAREFUL) {
                        const uint32_t w = __float_as_uint(__double2float_rn(lo[r][c]));
                        fits = fits || (w == __float_as_uint(__double2float_rn(hi[r][c])) && (w & 0x7FFFFFFFu) - 1u < 0x7F800000u);
                        if (lo[r][c] == 0.0 && hi[r][c] == 0.0) { lo[r][c] = 0.0; fits = true; }
                        fits = fits && !((slow >> (r * TN + c)) & 1u);
                    }
                    if (!fits) slow |= 1u << (r * TN + c);
                    if (!CAREFUL || fits) cw[r][c] = __float_as_uint(__double2float_rn(lo[r][c]));
                }
        }
    };

    int until = PROMOTE ? int(g.k_chunk) : 0;           // elements of K left before the next promotion
    auto promote = [&] {                                // FP32 promotion of the partial sum every k_chunk elements
        until = int(g.k_chunk);
#pragma unroll
        for (int r = 0; r < TM; ++r)
#pragma unroll
            for (int c = 0; c < TN; ++c) {
                float v = __fadd_rn(promoted[PROMOTE ? r : 0][PROMOTE ? c : 0], __uint_as_float(output_word(r, c)));
                if (v != v) v = __uint_as_float(0x7FFFFFFFu);
                promoted[PROMOTE ? r : 0][PROMOTE ? c : 0] = v;
                set_state(r, c, 0u);
            }
        sp_nan = sp_pinf = sp_ninf = 0u;
        subnormal = false;
    };
    bool c_tame = false;
    subnormal = __any_sync(0xFFFFFFFFu, subnormal);     // (matrix instructions need the whole warp: what they depend on is voted)
    for (int chunk = 0; chunk < NCH; ++chunk) {
        const int buf = chunk % BUF, next_buf = (chunk + 1) % BUF, k0 = chunk * KC, kc = min(KC, K - k0), nblk = (kc + L - 1) / L;
        const bool special = sm.special[buf] == chunk + 1;
        bool top_reached = false;                       // some product may reach 2^128
        if (TOP) {
            auto top = [&](int x) { const uint32_t v = sm.max_exp[buf][x]; return v >> 11 == uint32_t(chunk + 1) ? int(v & 0x7FFu) : 0; };
            top_reached = top(0) + top(1) - CB >= 126;
        }
        if (!E) {
            uint32_t sb[TN], nb[TN];
#pragma unroll
            for (int c = 0; c < TN; ++c) { sb[c] = sm.sgn[buf][BM + col_at(c)]; nb[c] = sm.nz[buf][BM + col_at(c)]; }
#pragma unroll
            for (int r = 0; r < TM; ++r) {
                const uint32_t sa = sm.sgn[buf][row_at(r)], na = sm.nz[buf][row_at(r)];
#pragma unroll
                for (int c = 0; c < TN; ++c) negm[E ? 0 : r][E ? 0 : c] = (sa ^ sb[c]) & na & nb[c];
            }
        }
        // Special-value events (Section 4.2) of the elements in `bits`, from the masks; the flags are sticky.  A loop, because they are rare
        // and registers are not: a second call behind the plain blocks made special values cheaper (0.38 ms) and everything else 1 %
        // dearer.  Read and decoded element by element for every output, raw bit patterns took 1000 x 1111 x 1000 7.8 ms (Ampere FP16;
        // the generic kernel 2.1, this way 0.78).
        auto note_specials = [&](uint32_t bits) {
#pragma unroll 1
            for (int o = 0; o < TM * TN; ++o) {
                const int a = row_at(o / TN), b = BM + col_at(o % TN);
                const uint32_t an = sm.nan[buf][a], ai = sm.inf[buf][a], bn = sm.nan[buf][b], bi = sm.inf[buf][b];
                const uint32_t az = ~(an | ai | sm.nz[buf][a]), bz = ~(bn | bi | sm.nz[buf][b]);
                const uint32_t bad = an | bn | (ai & bz) | (bi & az), infs = (ai | bi) & ~bad & bits, sign = sm.sgn[buf][a] ^ sm.sgn[buf][b];
                if (bad & bits) sp_nan |= 1u << o;
                if (infs & ~sign) sp_pinf |= 1u << o;
                if (infs & sign) sp_ninf |= 1u << o;
            }
        };
        auto note_overflows = [&](int kb) {             // products of 2^128 and more are infinities (the offset of a B operand does not get one there)
#pragma unroll 1
            for (int o = 0; o < TM * TN; ++o) {
                if (((sp_nan | (sp_pinf & sp_ninf)) >> o) & 1u) continue;       // a NaN already
#pragma unroll 1
                for (int k = kb; k < kb + L; ++k) {
                    const double p = __dmul_rn(sm.d[buf][row_at(o / TN)][k], sm.d[buf][BM + col_at(o % TN)][k]);
                    if (fabs(p) >= 3.402823669209385e38) { if (p < 0.0) sp_ninf |= 1u << o; else sp_pinf |= 1u << o; }
                }
            }
        };
        rare = special || top_reached;
        // ---- a whole chunk without special values, promotion or odd accumulators runs through plain blocks; if one of them
        // notes a result outside the normal range, the chunk is done again from the accumulators it began with ----
        bool again = true;
        const bool whole = !rare && !subnormal && nblk == NBLK && !(PROMOTE && until < KC);
        bool tame = TAMEABLE && whole && !(WIDE && sm.wild[buf] == chunk + 1);
        if (tame && !c_tame) {
            bool ok = true;
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int c = 0; c < TN; ++c) {
                    const uint32_t h = uint32_t(__double2hiint(cs[E ? 0 : r][E ? 0 : c])) & 0x7FFFFFFFu;
                    ok = ok && (h == 0u || h - (uint32_t(1023 - 100) << 20) < (200u << 20));
                }
            c_tame = __all_sync(0xFFFFFFFFu, ok);
        }
        tame = tame && c_tame;
        c_tame = tame;
        constexpr int UNROLL = NBLK * TM * TN <= 32 ? NBLK : (32 / (TM * TN) > 1 ? 32 / (TM * TN) : 1);
        if (TAMEABLE && tame) {
#pragma unroll UNROLL
            for (int blk = 0; blk < NBLK; ++blk)
                block(blk * L, blk + 1 < NBLK ? buf : next_buf, blk + 1 < NBLK ? blk * L + L : 0, std::integral_constant<int, TAMEABLE ? IN_RANGE : PLAIN>{});
            again = false;
            if (PROMOTE && (until -= KC) == 0) promote();
        } else if (whole) {
            double cs0[E ? 1 : TM][E ? 1 : TN];
            uint32_t cw0[E ? TM : 1][E ? TN : 1];
#pragma unroll
            for (int r = 0; r < TM; ++r)
#pragma unroll
                for (int c = 0; c < TN; ++c) { if (E) cw0[E ? r : 0][E ? c : 0] = cw[E ? r : 0][E ? c : 0]; else cs0[E ? 0 : r][E ? 0 : c] = cs[E ? 0 : r][E ? 0 : c]; }
            seen_max = 0u;
            seen_min = 0xFFFFFFFFu;
            seen_top = 0.f;
            slow = 0u;
#pragma unroll UNROLL
            for (int blk = 0; blk < NBLK; ++blk) block(blk * L, blk + 1 < NBLK ? buf : next_buf, blk + 1 < NBLK ? blk * L + L : 0, std::integral_constant<int, PLAIN>{});
            const bool done = T ? seen_max < 2u * TOPHI && seen_min >= 2u * LOWHI - 1u : (E ? slow == 0u : seen_top <= 3.4028234663852886e38f);
            again = __any_sync(0xFFFFFFFFu, !done);
            if (again) {
#pragma unroll
                for (int r = 0; r < TM; ++r)
#pragma unroll
                    for (int c = 0; c < TN; ++c) { if (E) cw[E ? r : 0][E ? c : 0] = cw0[E ? r : 0][E ? c : 0]; else cs[E ? 0 : r][E ? 0 : c] = cs0[E ? 0 : r][E ? 0 : c]; }
#pragma unroll
                for (int ks = 0; ks < NKS; ++ks) { fetch_fragments(buf, 0, ks); fetch_exponents(buf, 0, ks); }
            } else {
                if (PROMOTE && (until -= KC) == 0) promote();
            }
        }
        if (again) {
#pragma unroll 1
            for (int blk = 0; blk < nblk; ++blk) {
                const int kb = blk * L;
                // (before the block: a finite overflow counts if it comes first)
                if (special && !E) note_specials(L == 32 ? 0xFFFFFFFFu : ((1u << (L % 32)) - 1u) << kb);
                if (TOP && top_reached) note_overflows(kb);
                slow = 0u;
                if (E && special) {                     // outputs whose block holds a special value
#pragma unroll 1
                    for (int o = 0; o < TM * TN; ++o) {
                        const int a = row_at(o / TN), b = BM + col_at(o % TN);
                        const uint32_t any = sm.nan[buf][a] | sm.inf[buf][a] | sm.nan[buf][b] | sm.inf[buf][b];
                        if ((any >> kb) & ((1u << (L % 32)) - 1u)) slow |= 1u << o;
                    }
                }
                block(kb, blk + 1 < nblk ? buf : next_buf, blk + 1 < nblk ? kb + L : 0, std::integral_constant<int, CAREFULLY>{});
                if (E && slow) {                        // by the book on the raw words
#pragma unroll
                    for (int r = 0; r < TM; ++r)
#pragma unroll
                        for (int c = 0; c < TN; ++c)
                            if ((slow >> (r * TN + c)) & 1u) {
                                const int64_t i = row0 + row_at(r), j = col0 + col_at(c);
                                uint32_t& w = cw[E ? r : 0][E ? c : 0];
                                if ((w & 0x7FFFFFFFu) > 0x7F800000u) { w = special_word(1, false, false); continue; }      // a NaN stays one
                                w = (i < g.M && j < g.N) ? by_the_book<EK>(m, g.A, g.B, i * g.lda + k0 + kb, j * g.ldb + k0 + kb, min(L, kc - kb), w) : 0u;
                            }
                }
                if (PROMOTE && (until -= L) <= 0) promote();
            }
            subnormal = __any_sync(0xFFFFFFFFu, subnormal);
        }
        if (chunk + 1 < NCH) __syncthreads();
    }

#pragma unroll
    for (int r = 0; r < TM; ++r)
#pragma unroll
        for (int c = 0; c < TN; ++c) {
            const int64_t i = row0 + row_at(r), j = col0 + col_at(c);
            if (i >= g.M || j >= g.N) continue;
            uint32_t w = PROMOTE ? __float_as_uint(promoted[PROMOTE ? r : 0][PROMOTE ? c : 0]) : output_word(r, c);
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
}

template <int FAM, int EK, int L, int RHO, bool PROMOTE, int TM, int CN, int WR, int WC, int PW, int TASK>
__global__ void __launch_bounds__(32 * (WR * WC + PW), min_ctas(TM * CN, L, WR * WC + PW)) direct_kernel(DevModel m, GemmArgs g, int unit_a, int unit_b) {
    after_previous();
    direct_tile<FAM, EK, L, RHO, PROMOTE, TM, CN, WR, WC, PW, TASK>(m, g, unit_a, unit_b, int64_t(blockIdx.y) * (8 * TM * WR), int64_t(blockIdx.x) * (8 * CN * WC));
}

// The tiles that the matrix instruction has to leave to the emulation (GemmArgs::redo), on a fixed grid: almost always there are
// none, and every CTA reads the flags and leaves (1024 x 4096: a CTA per tile that looked for itself took 18 us).
template <int FAM, int EK, int L, int RHO, int TM, int CN, int WR, int WC, int PW, int TASK>
__global__ void __launch_bounds__(32 * (WR * WC + PW), min_ctas(TM * CN, L, WR * WC + PW)) direct_rest_kernel(DevModel m, GemmArgs g, int unit_a, int unit_b) {
    after_previous();
    constexpr int BM = 8 * TM * WR, BN = 8 * CN * WC;
    const int64_t flags = (g.N + 127) / 128 * g.redo_across;
    int any = 0;
    for (int64_t i = threadIdx.x; i < flags; i += blockDim.x) any |= g.redo[i];
    if (!__syncthreads_or(any)) return;
    const int64_t tn = (g.N + BN - 1) / BN, tiles = (g.M + BM - 1) / BM * tn;
    for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int64_t row0 = t / tn * BM, col0 = t % tn * BN;
        if (!tile_wanted(g, row0, BM, col0, BN)) continue;
        direct_tile<FAM, EK, L, RHO, false, TM, CN, WR, WC, PW, TASK>(m, g, unit_a, unit_b, row0, col0);
        __syncthreads();
    }
}

// Bytes per asynchronous copy that rows `ld` elements apart allow (bases are 16-byte aligned).
template <int EK, int TASK>
int copy_unit(int64_t ld) {
    constexpr int B = Elem<EK>::BYTES, SLOT = TASK * B;
    constexpr int NATURAL = SLOT < 16 ? SLOT : 16;
    return (ld * B) % NATURAL == 0 ? NATURAL : ((ld * B) % 4 == 0 ? 4 : 0);
}

template <int FAM, int EK, int L, int RHO, bool PROMOTE, int TM, int CN, int WR, int WC, int PW, int TASK>
cudaError_t launch_tile(const DevModel& m, const GemmArgs& g, cudaStream_t st) {
    constexpr int BM = 8 * TM * WR, BN = 8 * CN * WC, NTH = 32 * (WR * WC + PW);
    constexpr size_t sh = sizeof(Smem<EK, BM, BN, 32 * PW, TASK>);
    auto kernel = direct_kernel<FAM, EK, L, RHO, PROMOTE, TM, CN, WR, WC, PW, TASK>;
    if (sh > 48 * 1024) {
        const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sh));
        if (err != cudaSuccess) return err;
    }
    const dim3 grid((unsigned)((g.N + BN - 1) / BN), (unsigned)((g.M + BM - 1) / BM), 1);
    return enqueue(kernel, grid, NTH, sh, st, m, g, copy_unit<EK, TASK>(g.lda), copy_unit<EK, TASK>(g.ldb));
}

template <int FAM, int EK, int L, int RHO>
cudaError_t launch_rest(const DevModel& m, const GemmArgs& g, cudaStream_t st) {
    constexpr int PW = 4, TASK = 8, NTH = 32 * (4 + PW);
    constexpr size_t sh = sizeof(Smem<EK, 32, 32, 32 * PW, TASK>);
    auto kernel = direct_rest_kernel<FAM, EK, L, RHO, 2, 2, 2, 2, PW, TASK>;
    const cudaError_t err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, int(sh));
    if (err != cudaSuccess) return err;
    const int64_t tiles = (g.M + 31) / 32 * ((g.N + 31) / 32);
    return enqueue(kernel, unsigned(tiles < 296 ? tiles : 296), NTH, sh, st, m, g, copy_unit<EK, TASK>(g.lda), copy_unit<EK, TASK>(g.ldb));
}

// Accumulator tiles per warp, warps and staging warps per CTA for each size (chosen by direct_size in mmasim_tfdpa_fast.cu).
template <int FAM, int EK, int L, int RHO, bool PROMOTE>
cudaError_t launch_sizes(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t st) {
    switch (size) {
        case DIRECT_8x16: return launch_tile<FAM, EK, L, RHO, PROMOTE, 1, 1, 1, 2, 3, 8>(m, g, st);
        case DIRECT_16x16: return launch_tile<FAM, EK, L, RHO, PROMOTE, 1, 1, 2, 2, 4, 8>(m, g, st);
        default: return launch_tile<FAM, EK, L, RHO, PROMOTE, 2, 2, 2, 2, 4, 8>(m, g, st);
    }
}

template <int FAM, int EK, int L, int RHO>
cudaError_t launch(const DevModel& m, const GemmArgs& g, DirectSize size, cudaStream_t st) {
    if constexpr ((FAM == FAM_T || FAM == FAM_ST) && RHO != RHO_RNE_FP16) {
        if (g.k_chunk) return launch_sizes<FAM, EK, L, RHO, true>(m, g, size, st);
    }
    return launch_sizes<FAM, EK, L, RHO, false>(m, g, size, st);
}

}  // namespace direct
}  // namespace mmasim
