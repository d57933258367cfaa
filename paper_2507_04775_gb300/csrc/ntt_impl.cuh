// NTT launchers for one ring degree, instantiated once per logN in its own
// translation unit (ntt_l12.cu .. ntt_l17.cu) so that the many kernel
// instances compile in parallel; ntt.cu dispatches on the context's logN.
//
// logN = 12: one tile per limb (KIND 2).  logN = 13..17: the paper's two-pass
// decomposition (Sec. III-F4) with a column pass of S_col stages on columns
// of stride 2^(logN - S_col) and a row pass of S_row stages on contiguous rows:
//   logN   13   14   15   16   17
//   S_col   7    7    8    8    9
//   S_row   6    7    7    8    8
// Each pass has up to six compiled tile variants (columns/rows per CTA, the
// resident-CTA target and the elements per thread, chosen per pass kind and
// size; see ntt_rules.h).
#pragma once

#include <algorithm>
#include <cstring>

#include "fides_internal.cuh"
#include "ntt.cuh"
#include "ntt_rules.h"
#include "rows_inner.cuh"

namespace {

// Variant of a pass of `total` limbs; operands: a forward row pass whose epilogue
// reads operands.
inline int variant_of(const fides_ctx *c, int kind, int total, bool operands = false)
{
    return ntt_variant(c->ntt_var[kind], FIDES_TUNE_MAX + 1, c->ntt_tuned, kind, c->logN, c->fold, total,
                       operands);
}

template <int LOGN>
struct Split {
    static constexpr int COL = ntt_col_stages(LOGN);
    static constexpr int ROW = ntt_row_stages(LOGN);
};

template <int LOGN, int V, int KIND, bool INV, bool NINV, bool FOLD, class Pro, class Epi>
void launch_pass(const fides_ctx *c, const LimbSet &set, const TwPair *tw, Pro pro, Epi epi, cudaStream_t st,
                 const char *name)
{
    constexpr int S = KIND == 0 ? Split<LOGN>::COL : Split<LOGN>::ROW;
    constexpr int CT = ntt_tile_width(V, S);
    auto k = k_ntt<LOGN, S, KIND, INV, NINV, CT, ntt_tile_ctas(V, S), VAR_LE[V], FOLD, Pro, Epi>;
    dim3 grid((1 << (LOGN - S)) / CT, set.total), block(ntt_tile_threads(V, S));
    FIDES_LAUNCH(name, st, k, grid, block, set, (const PrimeInfo *)c->d_prime, tw, pro, epi);
}

template <int LOGN, int KIND, bool INV, bool NINV, class Pro, class Epi>
void launch_pass_v(int v, const fides_ctx *c, const LimbSet &set, const TwPair *tw, Pro pro, Epi epi,
                   cudaStream_t st, const char *name)
{
    if (c->fold) {
        switch (v) {
        case 0: launch_pass<LOGN, 0, KIND, INV, NINV, true>(c, set, tw, pro, epi, st, name); break;
        case 1: launch_pass<LOGN, 1, KIND, INV, NINV, true>(c, set, tw, pro, epi, st, name); break;
        case 2: launch_pass<LOGN, 2, KIND, INV, NINV, true>(c, set, tw, pro, epi, st, name); break;
        case 3: launch_pass<LOGN, 3, KIND, INV, NINV, true>(c, set, tw, pro, epi, st, name); break;
        case 4: launch_pass<LOGN, 4, KIND, INV, NINV, true>(c, set, tw, pro, epi, st, name); break;
        default: launch_pass<LOGN, 5, KIND, INV, NINV, true>(c, set, tw, pro, epi, st, name); break;
        }
        return;
    }
    constexpr int kind = KIND == 0 ? (INV ? INV_COLS : FWD_COLS) : (INV ? INV_ROWS : FWD_ROWS);
    switch (ntt_compiled(v, false, kind)) {
    case 1: launch_pass<LOGN, 1, KIND, INV, NINV, false>(c, set, tw, pro, epi, st, name); break;
    case 2: launch_pass<LOGN, 2, KIND, INV, NINV, false>(c, set, tw, pro, epi, st, name); break;
    case 4:
        if constexpr (kind == FWD_COLS) launch_pass<LOGN, 4, KIND, INV, NINV, false>(c, set, tw, pro, epi, st, name);
        break;
    default: launch_pass<LOGN, 5, KIND, INV, NINV, false>(c, set, tw, pro, epi, st, name); break;
    }
}

template <int LOGN, class Pro, class Epi>
int forward(const fides_ctx *c, const LimbSet &set, Pro pro, Epi epi, cudaStream_t st)
{
    if (set.total == 0) return FIDES_OK;
    if constexpr (LOGN == 12) {
        auto k = c->fold ? k_ntt<12, 12, 2, false, false, 16, NTT_LIMB_CTAS, 3, true, Pro, Epi>
                         : k_ntt<12, 12, 2, false, false, 16, NTT_LIMB_CTAS, 3, false, Pro, Epi>;
        FIDES_LAUNCH("k_ntt_fwd_limb", st, k, dim3(1, set.total), dim3(512), set, (const PrimeInfo *)c->d_prime,
                     (const TwPair *)c->d_tw, pro, epi);
    } else {
        launch_pass_v<LOGN, 0, false, false>(variant_of(c, FWD_COLS, set.total), c, set, c->d_tw, pro, EpiLazy{},
                                             st, "k_ntt_fwd_cols");
        constexpr bool operands = !std::is_same_v<Epi, EpiCanon>;
        launch_pass_v<LOGN, 1, false, false>(variant_of(c, FWD_ROWS, set.total, operands), c, set, c->d_tw, ProDst{},
                                             epi, st, "k_ntt_fwd_rows");
    }
    return fides_check_cuda(cudaGetLastError(), "ntt forward launch");
}

template <int LOGN, class Pro, class Epi>
int inverse(const fides_ctx *c, const LimbSet &set, Pro pro, Epi epi, cudaStream_t st)
{
    if (set.total == 0) return FIDES_OK;
    if constexpr (LOGN == 12) {
        auto k = c->fold ? k_ntt<12, 12, 2, true, true, 16, NTT_LIMB_CTAS, 3, true, Pro, Epi>
                         : k_ntt<12, 12, 2, true, true, 16, NTT_LIMB_CTAS, 3, false, Pro, Epi>;
        FIDES_LAUNCH("k_ntt_inv_limb", st, k, dim3(1, set.total), dim3(512), set, (const PrimeInfo *)c->d_prime,
                     (const TwPair *)c->d_itw, pro, epi);
    } else {
        launch_pass_v<LOGN, 1, true, false>(variant_of(c, INV_ROWS, set.total), c, set, c->d_itw, pro, EpiLazy{}, st,
                                            "k_ntt_inv_rows");
        launch_pass_v<LOGN, 0, true, true>(variant_of(c, INV_COLS, set.total), c, set, c->d_itw, ProDst{}, epi, st,
                                           "k_ntt_inv_cols");
    }
    return fides_check_cuda(cudaGetLastError(), "ntt inverse launch");
}

// the column pass alone (see ntt.cuh)
template <int LOGN>
int forward_cols(const fides_ctx *c, const LimbSet &set, cudaStream_t st)
{
    if constexpr (LOGN != 12) {
        if (set.total == 0) return FIDES_OK;
        launch_pass_v<LOGN, 0, false, false>(variant_of(c, FWD_COLS, set.total), c, set, c->d_tw, ProSrc{}, EpiLazy{},
                                             st, "k_ntt_fwd_cols");
    }
    return fides_check_cuda(cudaGetLastError(), "ntt forward launch");
}

template <int LOGN>
int inverse_cols(const fides_ctx *c, const LimbSet &set, cudaStream_t st)
{
    if constexpr (LOGN != 12) {
        if (set.total == 0) return FIDES_OK;
        launch_pass_v<LOGN, 0, true, true>(variant_of(c, INV_COLS, set.total), c, set, c->d_itw, ProDst{}, EpiCanon{},
                                           st, "k_ntt_inv_cols");
    }
    return fides_check_cuda(cudaGetLastError(), "ntt inverse launch");
}

// the forward row pass of ModUp's limbs with the key inner product
// (rows_inner.cuh)
template <int LOGN, int MAXB>
int rows_inner_b(const fides_ctx *c, const IPArgs &A, int limbs, int max_beta, cudaStream_t st)
{
    constexpr int S = Split<LOGN>::ROW;
    constexpr int C = 1024 >> S;
    const dim3 grid((1 << (LOGN - S)) / C, limbs), block((C << S) >> RI_LE);
    FIDES_LAUNCH_SMEM("k_rows_inner", st, (k_rows_inner<LOGN, S, C, MAXB>), grid, block, rows_inner_smem(max_beta), A,
                      c->L, c->K, (const PrimeInfo *)c->d_prime, (const TwPair *)c->d_tw, (const TwPair *)c->d_itw);
    return fides_check_cuda(cudaGetLastError(), "rows + inner product launch");
}

template <int LOGN>
int rows_inner(const fides_ctx *c, const IPArgs &A, int limbs, int max_beta, cudaStream_t st)
{
    if constexpr (LOGN != 12) {
        switch (max_beta) {
        case 1:
        case 2: return rows_inner_b<LOGN, 2>(c, A, limbs, max_beta, st);
        case 3: return rows_inner_b<LOGN, 3>(c, A, limbs, max_beta, st);
        case 4: return rows_inner_b<LOGN, 4>(c, A, limbs, max_beta, st);
        default: return rows_inner_b<LOGN, 5>(c, A, limbs, max_beta, st);
        }
    }
    return fides_set_error(FIDES_ERR_UNSUPPORTED, "rows + inner product: logN = 12");   // rows_inner_ok is false
}

// What the autotuner times for variant v of pass kind `kind`: whole transforms,
// whose other pass runs the default tile.  Forward rows run twice, once with an
// epilogue that reads operands (the segments carry aux, out and constants): one
// choice serves both, the default with its own tile for the latter.
template <int LOGN>
void launch_one(const fides_ctx *c, int kind, int v, const LimbSet &set, cudaStream_t st)
{
    const char *name = "k_ntt_tune";
    auto tile = [&](int k) { return k == kind ? v : ntt_default_variant(k, LOGN, c->fold, set.total); };
    if (kind == FWD_COLS || kind == FWD_ROWS) {
        launch_pass_v<LOGN, 0, false, false>(tile(FWD_COLS), c, set, c->d_tw, ProSrc{}, EpiLazy{}, st, name);
        launch_pass_v<LOGN, 1, false, false>(tile(FWD_ROWS), c, set, c->d_tw, ProDst{}, EpiCanon{}, st, name);
        if (kind == FWD_COLS) return;
        launch_pass_v<LOGN, 0, false, false>(tile(FWD_COLS), c, set, c->d_tw, ProSrc{}, EpiLazy{}, st, name);
        const int def = ntt_default_variant(FWD_ROWS, LOGN, c->fold, set.total);
        launch_pass_v<LOGN, 1, false, false>(v == def ? ntt_default_variant(FWD_ROWS, LOGN, c->fold, set.total, true) : v,
                                             c, set, c->d_tw, ProDst{}, EpiSubMul{}, st, name);
    } else {
        launch_pass_v<LOGN, 1, true, false>(tile(INV_ROWS), c, set, c->d_itw, ProPlain{}, EpiLazy{}, st, name);
        launch_pass_v<LOGN, 0, true, true>(tile(INV_COLS), c, set, c->d_itw, ProDst{}, EpiCanon{}, st, name);
    }
}

}  // namespace

// The launchers of one ring degree (defined by FIDES_NTT_DEGREE in ntt_lNN.cu).
#define FIDES_NTT_DECLARE(L)                                                                      \
    int ntt_fwd_canon_##L(const fides_ctx *, const LimbSet &, cudaStream_t);                      \
    int ntt_fwd_submul_##L(const fides_ctx *, const LimbSet &, cudaStream_t);                     \
    int ntt_fwd_switch_submul_##L(const fides_ctx *, const LimbSet &, cudaStream_t);              \
    int ntt_fwd_submul_rot_##L(const fides_ctx *, const LimbSet &, cudaStream_t);                 \
    int ntt_fwd_raise_##L(const fides_ctx *, const LimbSet &, cudaStream_t);                      \
    int ntt_fwd_hmrs_##L(const fides_ctx *, const LimbSet &, cudaStream_t);                       \
    int ntt_inv_canon_##L(const fides_ctx *, const LimbSet &, cudaStream_t);                      \
    int ntt_fwd_cols_##L(const fides_ctx *, const LimbSet &, cudaStream_t);                       \
    int ntt_inv_cols_##L(const fides_ctx *, const LimbSet &, cudaStream_t);                       \
    int ntt_rows_inner_##L(const fides_ctx *, const IPArgs &, int, int, cudaStream_t);            \
    void ntt_tune_one_##L(const fides_ctx *, int, int, const LimbSet &, cudaStream_t);

#define FIDES_NTT_DEGREE(L)                                                                                       \
    int ntt_fwd_canon_##L(const fides_ctx *c, const LimbSet &s, cudaStream_t st)                                \
    {                                                                                                             \
        return forward<L>(c, s, ProSrc{}, EpiCanon{}, st);                                                        \
    }                                                                                                             \
    int ntt_fwd_submul_##L(const fides_ctx *c, const LimbSet &s, cudaStream_t st)                               \
    {                                                                                                             \
        return forward<L>(c, s, ProSrc{}, EpiSubMul{}, st);                                                       \
    }                                                                                                             \
    int ntt_fwd_switch_submul_##L(const fides_ctx *c, const LimbSet &s, cudaStream_t st)                        \
    {                                                                                                             \
        return forward<L>(c, s, ProSwitchMod{}, EpiSubMul{}, st);                                                 \
    }                                                                                                             \
    int ntt_fwd_submul_rot_##L(const fides_ctx *c, const LimbSet &s, cudaStream_t st)                           \
    {                                                                                                             \
        return forward<L>(c, s, ProSrc{}, EpiSubMulRot{c->logN}, st);                                             \
    }                                                                                                             \
    int ntt_fwd_raise_##L(const fides_ctx *c, const LimbSet &s, cudaStream_t st)                                \
    {                                                                                                             \
        return forward<L>(c, s, ProRaise{}, EpiCanon{}, st);                                                      \
    }                                                                                                             \
    int ntt_fwd_hmrs_##L(const fides_ctx *c, const LimbSet &s, cudaStream_t st)                                 \
    {                                                                                                             \
        return forward<L>(c, s, ProHmRs{}, EpiHmRs{}, st);                                                        \
    }                                                                                                             \
    int ntt_inv_canon_##L(const fides_ctx *c, const LimbSet &s, cudaStream_t st)                                \
    {                                                                                                             \
        if (s.modes == 0) return inverse<L>(c, s, ProPlain{}, EpiCanon{}, st);                                    \
        return inverse<L>(c, s, ProPrep{c->logN}, EpiCanon{}, st);                                                \
    }                                                                                                             \
    int ntt_fwd_cols_##L(const fides_ctx *c, const LimbSet &s, cudaStream_t st) { return forward_cols<L>(c, s, st); } \
    int ntt_inv_cols_##L(const fides_ctx *c, const LimbSet &s, cudaStream_t st) { return inverse_cols<L>(c, s, st); } \
    int ntt_rows_inner_##L(const fides_ctx *c, const IPArgs &A, int limbs, int max_beta, cudaStream_t st)       \
    {                                                                                                             \
        return rows_inner<L>(c, A, limbs, max_beta, st);                                                          \
    }                                                                                                             \
    void ntt_tune_one_##L(const fides_ctx *c, int kind, int v, const LimbSet &s, cudaStream_t st)               \
    {                                                                                                             \
        if constexpr (L != 12) launch_one<L>(c, kind, v, s, st);                                                  \
    }

FIDES_NTT_DECLARE(12)
FIDES_NTT_DECLARE(13)
FIDES_NTT_DECLARE(14)
FIDES_NTT_DECLARE(15)
FIDES_NTT_DECLARE(16)
FIDES_NTT_DECLARE(17)
