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
// eight elements per thread halve it and put twice the warps in flight.  Larger
// launches are bound by the multiply pipe and the twiddle reads, and sixteen
// elements exchange through shared memory once instead of twice.  The lines
// below, in limbs of logN = 16 (as many elements at other degrees), are where
// chains of whole transforms cross over, eight against sixteen elements in one
// of the passes (us):
//   forward columns, 22: folding, logN = 16, 22 limbs 17.6 18.5, 24: 19.1 18.7;
//     logN = 17, 11: 19.1 19.9, 12: 21.5 20.5; logN = 15, 40: 15.8 15.8, 60: 21.6
//     20.1.  Shoup, 20: 19.1 19.1, 24: 22.2 21.9
//   inverse columns, 23: folding, logN = 13, 180: 16.9 17.1; logN = 16, 24: 20.3
//     20.1; logN = 15, 60: 22.8 22.4.  Shoup, logN = 13, 180: 18.7 19.9; logN = 16,
//     24: 23.5 23.4
//   forward rows, 28 folding and 32 Shoup: folding, logN = 16, 24: 18.5 19.3, 30:
//     21.2 20.7, 36: 24.6 23.2, 60: 37.8 35.5; logN = 14, 90: 17.0 17.9, 120: 19.3
//     19.1, 240: 34.2 32.2; logN = 17, 12: 20.6 20.5, 20: 31.0 30.1.  Shoup, 30: 25.7
//     25.9, 36: 29.4 28.3
//   inverse rows, 32: folding, logN = 16, 24: 20.1 20.2, 30: 23.4 23.2, 36: 26.7
//     25.7, 60: 41.2 39.4, 120: 82.2 79.6; logN = 15, 60: 22.4 22.8, 90: 30.7 30.4;
//     logN = 17, 20: 32.9 32.2, 60: 94.4 90.4.  Shoup, 30: 27.5 27.7, 36: 31.4 30.8
// Large row passes take four rows a CTA, at logN = 13 eight: four rows of 64
// elements are half a warp (480 limbs forward 43.4 us with four, 32.1 with eight).
// Forward columns run within 64 registers past 64 limbs of logN = 17 with folding
// products (80 against 64: 90 limbs 125.8 123.5, 120: 165.0 162.0; logN = 16, 180
// limbs 106.3 107.3).  Plain transforms of 15 to 60 limbs of logN = 17 gain 1 % by
// it too, but the columns of a Rescale, which reduce their input, lose more (14
// limbs 31.9 35.7), and so with Shoup products.
//
// operands: a forward row pass whose epilogue reads operands (ModDown,
// Rescale: two or three words a coefficient against one) waits for HBM where
// the plain pass waits for the multiply pipe.  More warps are worth more than
// registers there.  With Shoup products the eight-element tile stays ahead at
// every size measured (a Rescale by its rows, eight and sixteen elements, logN =
// 16, 58: 62.0 64.6, 98: 98.3 102.4; logN = 17, 98: 196.6 205.9); folding ones
// cross over at 56 and then run sixteen elements within 64 registers (a Rescale,
// eight elements, sixteen within 80 and within 64: logN = 16, 46: 44.8 43.9 43.6,
// 58: 54.4 54.6 53.3, 98: 87.6 88.3 84.5; logN = 17, 32: 64.7 66.1 63.4, 98: 175.9
// 177.7 170.1; an HRotate, logN = 16, 48: 194.6 196.4 195.9, 56: 210.8 211.4 212.0,
// 72: 310.0 316.7 308.8).
inline int ntt_default_variant(int kind, int logN, bool fold, long total, bool operands = false)
{
    const long limbs = ((total << logN) + 65535) >> 16;   // of logN = 16, rounded up
    const int rows16 = logN == 13 ? 1 : 2;                // row passes with sixteen elements
    switch (kind) {
    case FWD_COLS: return limbs <= 22 ? 5 : (logN == 17 && fold && limbs > 128 ? 4 : 1);
    case INV_COLS: return limbs <= 23 ? 5 : 1;
    case FWD_ROWS:
        if (operands) return !fold || limbs <= 56 ? 5 : (logN == 13 ? 4 : 3);
        return limbs <= (fold ? 28 : 32) ? 5 : rows16;
    default: return limbs <= 32 ? 5 : rows16;
    }
}

// Variant of a pass: what the tuned or installed table says (n entries for the
// pass kind, limb counts from zero; launches past its end take the last), or
// the default.  An entry that is the default's leaves the default, also for the
// passes whose epilogue reads operands; any other is what runs in both.
inline int ntt_variant(const unsigned char *table, int n, bool tuned, int kind, int logN, bool fold, int total,
                       bool operands)
{
    const int at = total < n ? total : n - 1;
    if (!tuned || (operands && table[at] == ntt_default_variant(kind, logN, fold, at)))
        return ntt_default_variant(kind, logN, fold, total, operands);
    return table[at];
}
