// matval.cuh -- the valuation as a matrix product on the 5th-generation tensor cores.
//
// With deterministic mortality the reserve of policy p under scenario s is
//   V(p, s) = amount_p [ sum_t D_s(t + 1) E_p(t) + D_s(S_p) B_p ],   D_s(t + 1) = v_0 ... v_t
// (Eq. basicReserveSummation; cashflow.cuh): a product of the policies' expected cash
// flows [policy][step] and the scenarios' discount products [step][scenario].  The
// recurrence kernels run it chain by chain on the FP32 pipe; here it runs as 16-bit
// matrix instructions with FP32 accumulation, on operands split into exact digits (the splitting
// of Ozaki, Ogita, Oishi & Rump, "Error-free transformations of matrix multiplication by using
// fast routines of matrix multiplication", Numer. Algorithms 59, 2012):
//
//   a = d1 + d2 + ...  with a in [0, 1]; d1: a to 7 bits.
//   Three digits: d2 and d3 the FP16 values (11 bits and sign) of the remainders, to 2^-32
//   of the row's largest entry; stored times 2^15.
//   Four and six: d2 and d3 the next 8 bits each (signed), the others BF16 values of the
//   remainders, to 2^-33 and 2^-48.
//   Eight (the FP64 form): seven more of 8 bits each (signed), to 2^-63.
//
// The products of digits i and j, i + j at most the last digit's number, are taken.  A digit is
// at most 2^7 units in size and a product 2^14, so that FP32 adds up 1,024 products of a level
// exactly whatever their signs.  Operands that hardly change (no interest and no mortality to
// speak of) have digits of one sign from step to step, so this is the bound that counts: one
// accumulator a level over 1,000 steps was off by 4e-9 on such operands.  With six and eight
// digits an accumulator takes one or two products of a level and sums at most 512 steps, a segment,
// which makes the levels 0 to 2 (eight digits: to 3) exact and leaves truncations below 2^-40
// (2^-46) of the sum at the very worst.  With three and four digits a segment is 1,024 steps, so
// that level 0 is exact; the truncations of the others, at most 2^-24 of a sum 2^-7 below for each
// block of 16 steps and pair of digits, stay within 2^-22.
// The epilogue adds the accumulators: the first ones with their rounding errors, the low ones as
// they are (to 2^-40, 2^-48 and 2^-56 with four, six and eight digits), and the segments as
// double-floats (eight digits: three floats).  A maturity payment is added there, from the
// discount products themselves, so that a row holds entries of one kind.
//
// Fixed point needs rows and columns of moderate range.  The discount products are
// tilted by a power of two per step, 2^tau(t) ~ 1 / (their geometric mean over the
// scenarios), and the cash flows by 2^-tau(t), so that what is left of a scenario is its
// deviation from the mean; a row is scaled by the power of two of its largest
// entry.  A scenario set whose tilted products vary by too much along a scenario (see
// mv_max_spread) keeps the recurrence kernels.
//
// Measured (one GB300, with the digits and the totals), before: the recurrence.
//   100,000 policies of every product, 1,000 scenarios: compensated 38.7 -> 1.67 ms
//   (annuities 1.5e-13 -> 6e-15 rms, assurances 2e-9 -> 1.2e-14), deflated 4.93 -> 0.88 ms
//   (rms 3e-8 -> 5e-9, with three digits 0.62 ms);
//   1,000,000 annuities, 600 steps, 1,000 scenarios, deflated: 30.6 -> 4.1 ms;
//   3,000 two-life policies, 333 scenarios, FP64: 5.17 -> 0.15 ms (1.4e-15 -> 1.3e-15).
// It is the faster path at every size measured: one policy and one scenario 53 -> 49 us
// compensated and 158 -> 37 us deflated (host call included), 1,000 policies under 157
// scenarios of the mix 276 -> 102 us and 282 -> 63 us.
#pragma once

#include <cuda.h>

#include "cashflow.cuh"

namespace rsv {

constexpr int kMvP = 128;          // policies per tile (MMA N)
constexpr int kMvM = 128;          // scenarios per tile (MMA M)
constexpr int kMvParts = 4;        // column groups of the epilogue
constexpr int kMvTilt = 60;        // largest |tau|
constexpr int kMvMaxSteps = 64 * 65535;   // of a scenario set: blocks of 64 along a grid's second dimension
constexpr size_t kMvPanelBytes = size_t(1) << 30;            // cash-flow digits held at a time
// A row's entries, survivor-column entry times cash-flow multiplier times tilt, are formed in FP32
// head and tail (in the FP64 form their heads, for the row's scale), and a row's scale times its
// amount is one too; beyond these an exponent would be clamped or a tail lost.
constexpr double kMvEntryMin = 0x1p-100, kMvEntryMax = 0x1p100;
constexpr double kMvScaleMin = 0x1p-90, kMvScaleMax = 0x1p110;
constexpr double kMvAmountMin = 0x1p-60, kMvAmountMax = 0x1p90;   // |amount|

// The spread of a scenario set: the largest difference of the binary exponents of a scenario's
// tilted discount products (Vasicek paths, sd of the rate 2.2%: 3 to 5 over 50 years, 5 to 7
// over 100).  The worst error is that of a single payment at the smallest, row entry
// >= 1/2 and column entry >= 2^-(spread + 1):
//   three digits (deflated, spread to 4): 2^-27 left out, 2^(spread - 25) of the payment,
//     within the form's bound of 15 x 2^-24; at larger spreads the truncations of the low
//     accumulator also grow past it (2e-6 measured at 7);
//   four (deflated, to 8): below 2^-30 left out, 2^(spread - 28);
//   six (compensated, to 10): about 2^-46 left out, 2^(spread - 44);
//   eight (FP64, to 8): about 2^-61, 2^(spread - 59).
inline int mv_max_spread(int form) { return form == F_COMP ? 10 : 8; }
inline int mv_digits_of(int form, int spread) {
    return form == F_F64 ? 8 : (form == F_COMP ? 6 : (spread <= 4 ? 3 : 4));
}
inline int mv_digit_set(int ns) { return ns == 8 ? 3 : (ns == 6 ? 2 : ns - 3); }   // index of a digit count
// rows of scenario sums that the product writes: one a tile, or one a half tile
inline int mv_part_rows(int ns, int n_tiles) { return ns < 6 ? n_tiles : 2 * n_tiles; }
inline int mv_pitch(int steps) { return steps < 1 ? 64 : (steps + 63) / 64 * 64; }

// Scenario side, from the FP64 plane [n_steps][s_pad]: the discount products, and
struct MvScen {
    int32_t* tau;       // [n_steps] tilt of each step
    float* tilt;        // [n_steps] 2^-tau and
    float* tilt_top;    // [n_steps] its running maximum
    int32_t* colexp;    // [s_pad] binary exponent of each column's largest tilted product
    int32_t* colmin;    // [s_pad] scratch
    int32_t* stat;      // largest spread of a column, largest |tau| (INT_MAX where a product is
                        // not a normal number)
    static size_t words(int n_steps, int s_pad) { return 3 * (size_t)n_steps + 2 * (size_t)s_pad + 2; }
    static MvScen at(void* p, int n_steps, int s_pad) {
        int32_t* w = static_cast<int32_t*>(p);
        float* t = reinterpret_cast<float*>(w + n_steps);
        int32_t* c = w + 3 * (size_t)n_steps;
        return MvScen{w, t, t + n_steps, c, c + s_pad, c + 2 * (size_t)s_pad};
    }
};
cudaError_t launch_mv_scenarios(const double* v64, int n_steps, int n_scen, int s_pad, float2* D, const MvScen& c,
                                cudaStream_t st);
// Its digits [slices][s_pad][pitch]; columns beyond n_scen and steps beyond n_steps are 0.
cudaError_t launch_mv_digits(int ns, const float2* D, const int32_t* tau, const int32_t* colexp, int n_steps, int n_scen,
                             int s_pad, int pitch, void* digits, cudaStream_t st);

// Policy side of one panel of tiles: digits [tile][slices][128][pitch] up to each tile's
// longest projection, and what the epilogue needs of each policy.
struct alignas(16) MvOut {   // 32 bytes
    float sc_h, sc_l;    // V = (sc_h + sc_l) 2^(colexp) U (three digits: 2^-30 of it) + (mat_h + mat_l) D(S)
    float mat_h, mat_l;  // the maturity payment times its probability
    int32_t pol, S, pad[2];
};
struct MvBuild {
    CfTables T;
    const SlotRec* slots;      // of the panel's first tile
    const int32_t* kinds;
    const double* amount;
    int32_t n_tiles, tab_pad, pitch;
    int32_t general_from;      // first tile of the panel whose policies have varying cash flows
    const double* cf;          // their multipliers [n_pol][cf_ld], or null
    int32_t cf_ld;
    int32_t n_steps;           // of the scenario set
    int32_t rows_per_warp;     // 1, or 4 once there are tiles enough to fill the chip
    const float* tilt;
    const float* tilt_top;
    void* digits;
    MvOut* out;
};
cudaError_t launch_mv_build(int ns, const MvBuild& b, cudaStream_t st);

// A contract on up to four lives (32 bytes; records of one tile in decreasing steps).
struct MvLives {
    int32_t idx[4];  // survivor-column index of each life at valuation, -1: no such life
    int32_t S;
    int32_t pol;     // -1: padding
    int32_t k;       // 1 .. 4
    int32_t flags;   // bit 0: assurance (on the k-th death), else annuity (k or more alive);
                     // bits 8..11: dead at valuation
};
static_assert(sizeof(MvLives) == sizeof(SlotRec), "record strides");
constexpr int kMvRecWords = sizeof(SlotRec) / 4;
cudaError_t launch_mv_build_lives(const CfTables& T, const MvLives* recs, const double* amount, int n_tiles, int pitch,
                                  int n_steps, const float* tilt, void* digits, MvOut* out, cudaStream_t st);

// The FP64 form's: FP64 discount products, their eight digits, and the rows of the records that
// launch_cf_records makes of the panel's slots.
cudaError_t launch_mv_products64(const double* v64, int n_steps, int s_pad, double* D, cudaStream_t st);
cudaError_t launch_mv_digits64(const double* D, const int32_t* tau, const int32_t* colexp, int n_steps, int n_scen, int s_pad,
                               int pitch, void* digits, cudaStream_t st);
cudaError_t launch_mv_build64(const MvBuild& b, const CfPol* pols, cudaStream_t st);

struct MvArgs {
    const int32_t* steps;      // the steps of the panel's first record; one record is kMvRecWords
    const int32_t* kinds;      // of the tiles, or null: no maturity payments
    const MvOut* out;
    const int32_t* colexp;     // of the first column
    const float2* D;           // the discount products [n_steps][s_pad], at the first column
    const double* D64;         // the same in FP64 (eight digits)
    const double* amount;
    int32_t n_tiles, n_chunks; // policy tiles of the panel, scenario tiles of the column block
    int32_t s_pad, n_scen, s0; // plane rows; valid columns of the block; the block's first column
    int32_t v0_ld, part_ld;
    float* V0f;                // at the block's first column
    double* V0d;
    double* partial;           // [mv_part_rows][part_ld], at the panel's first tile and the block's first column
    int32_t* status;
};
// digitsE: launch_mv_build's, digitsD: launch_mv_digits', both of ns digits.
cudaError_t launch_mv_product(int ns, const MvArgs& a, const void* digitsD, const void* digitsE, int pitchD, int pitchE,
                              int sm_count, cudaStream_t st);

// The matrix variant's index among a form's tunable variants is the last one.
const char* mv_variant_name(int form);

}  // namespace rsv
