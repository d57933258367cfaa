// Tile variants of the two-pass transforms and the rule that picks one by the
// size of a launch.  Host code without CUDA, so that it can be compiled and
// checked by itself.
#pragma once

// Columns or rows per CTA, resident CTAs per SM at 256-element passes, log2 of
// the elements per thread.  With sixteen elements 3/6/12 CTAs leave up to 80
// registers a thread and 16/8 up to 64; with eight, 8 CTAs of 128 threads leave
// 64.
constexpr int NVAR = 6;
constexpr int VAR_CT[NVAR] = {16, 8, 4, 4, 8, 4};
constexpr int VAR_MINB[NVAR] = {3, 6, 12, 16, 8, 8};
constexpr int VAR_LE[NVAR] = {4, 4, 4, 4, 4, 3};

enum PassKind { FWD_COLS = 0, FWD_ROWS = 1, INV_ROWS = 2, INV_COLS = 3 };

// Tile of variant v for a pass of S stages: at most 8 sub-transforms per CTA
// when they have 512 elements (static shared memory), and the resident-CTA
// target that keeps the threads per SM (hence the register budget) of the
// variant's 256-element form.
constexpr int ntt_tile_width(int v, int S) { return S >= 9 && VAR_CT[v] > 8 ? 8 : VAR_CT[v]; }
constexpr int ntt_tile_threads(int v, int S) { return (ntt_tile_width(v, S) << S) >> VAR_LE[v]; }
constexpr int ntt_tile_ctas(int v, int S)
{
    const int want = (((256 * VAR_CT[v]) >> VAR_LE[v]) * VAR_MINB[v]) / ntt_tile_threads(v, S);
    return want < 1 ? 1 : (want > 32 ? 32 : want);
}

// Resident-CTA target of the whole-limb pass of logN = 12 (512 threads).
constexpr int NTT_LIMB_CTAS = 2;

// Stages of the column and of the row pass.
constexpr int ntt_col_stages(int logN) { return logN <= 14 ? 7 : (logN <= 16 ? 8 : 9); }
constexpr int ntt_row_stages(int logN) { return logN - ntt_col_stages(logN); }

// The compiled tile that runs for variant v of a pass: with Shoup arithmetic the
// wide tile and, but for forward columns, the 64-register ones run as 1 and 2.
// (Forward transforms at 61-bit primes, columns within 80 against 64 registers,
// us: logN = 16, 30 limbs 25.9 26.3, 60: 43.8 42.8, 90: 65.3 63.8, 120: 86.2 84.8;
// logN = 17, 60: 98.2 95.9, 90: 144.6 140.5.)
constexpr int ntt_compiled(int v, bool fold, int kind)
{
    return fold || (v == 4 && kind == FWD_COLS) ? v : (v == 0 || v == 4 ? 1 : (v == 3 ? 2 : v));
}

// Variant of a pass over `total` limbs where no table was installed.  A small
// launch runs in one wave, whose length is one thread's instruction stream:
// eight elements per thread halve it and put twice the warps in flight.  Larger launches are bound by the
// multiply pipe and the twiddle reads, and sixteen elements exchange through
// shared memory once instead of twice.  The column pass crosses over at 22
// limbs of logN = 16 (1.4 M elements; the inverse one at 23: 180 limbs of
// logN = 13 17.1 against 16.9 us, 24 limbs of logN = 16 20.1 against 20.3), the
// forward row pass, whose twiddles
// come from L2, at 56, and the inverse row pass not within 120.  Chains of
// whole transforms, columns + rows with sixteen and sixteen elements per
// thread, eight and eight, sixteen and eight (folding arithmetic, us):
//   logN = 16 forward  1 limb 6.5 5.0 5.6, 10: 17.5 14.8 12.8, 20: 20.1 15.9
//     16.6, 24: 20.2 18.8 18.7, 30: 21.9 22.1 20.9, 60: 37.1 40.2 37.2,
//     90: 53.0 59.1 53.8
//   logN = 16 inverse  1: 7.3 5.0 6.2, 20: 22.5 17.6 17.6, 30: 25.8 23.7 23.4,
//     60: 44.4 43.1 41.1, 90: 63.0 62.3 59.2
//   logN = 17 forward  7: 15.6 15.4 17.7, 12: 21.3 21.1 20.1, 30: 43.6 44.7 43.7
//   logN = 14 forward  60: 18.7 14.6 15.4, 90: 19.1 17.1 17.0, 120: 20.5 21.4 19.3
// Large forward row passes take four rows a CTA, at logN = 13 eight: four rows
// of 64 elements are half a warp (480 limbs 43.4 us with four, 32.1 with eight,
// 32.5 with eight elements a thread; logN = 14 60.6 with four, 65.5).
// Forward columns of more than 64 limbs of logN = 17 run within 64 registers
// (90 limbs 125.8 -> 123.5 us; not at logN = 16: 180 limbs 106.3 -> 107.3).
//
// operands: a forward row pass whose epilogue reads operands (ModDown,
// Rescale: two or three words a coefficient against one) waits for HBM where
// the plain pass waits for the multiply pipe.  More warps are worth more than
// registers there, so the same tiles run within 64: a Rescale by its rows, 80
// against 64 registers (folding arithmetic, us), logN = 16, 58 limbs 54.6 53.3,
// 78: 69.6 68.8, 98: 88.3 84.5; logN = 17, 32: 66.1 63.4, 58: 115.9 109.9, 98:
// 177.7 170.1.  Plain passes lose: a transform
// of 60 limbs 35.5 36.1.
inline int ntt_default_variant(int kind, int logN, long total, bool operands = false)
{
    const long elements = total << logN;
    switch (kind) {
    case FWD_COLS: return elements <= (22L << 16) ? 5 : (logN == 17 && elements > (128L << 16) ? 4 : 1);
    case INV_COLS: return elements <= (23L << 16) ? 5 : 1;
    case FWD_ROWS:
        if (elements <= (56L << 16)) return 5;
        return logN == 13 ? (operands ? 4 : 1) : (operands ? 3 : 2);
    default: return 5;
    }
}

// Variant of a pass: what the tuned or installed table (n entries for the pass
// kind, limb counts from zero) says, whatever the epilogue, or the default.
// Launches past the table's end take its last entry.
inline int ntt_variant(const unsigned char *table, int n, bool tuned, int kind, int logN, int total, bool operands)
{
    if (!tuned) return ntt_default_variant(kind, logN, total, operands);
    return table[total < n ? total : n - 1];
}
