// NTT launchers and the tile-width autotuner.
//
// The paper trades launch overhead against locality with a "limb batch"
// context parameter (Sec. III-F1) whose best value depends on the GPU
// (Sec. IV).  Here one launch always covers every limb of a step; what is left
// to tune is the tile width of each pass, which decides how many CTAs a launch
// has and so how much of its last wave is empty, and the elements per thread.
// Six variants of each pass of a two-pass transform (logN 13..17) are compiled
// for folding products (three or four for Shoup products, ntt_compiled) -- at
// logN=16, sixteen elements per thread with 16, 8 or 4 columns/rows per
// CTA (256, 128 or 64 threads) and up to 80 registers (3, 6 or 12 resident
// CTAs per SM), or with 4 or 8 per CTA and up to 64 registers (16 or 8 per
// SM), and eight elements per thread with 4 per CTA (128 threads, 8 per SM, 64
// registers); other sizes scale the resident-CTA target to the same register
// budget (ntt_rules.h).  The variant of a launch is a default by its size, or
// after fides_ctx_autotune what a table of the context says per pass kind and
// limb count.  The launchers of each ring degree live in
// ntt_l12.cu .. ntt_l17.cu; this file dispatches on the context's logN.
#include <algorithm>
#include <cstring>
#include <vector>

#include "ntt_impl.cuh"

#define FIDES_NTT_DISPATCH(fn, ...)                                  \
    switch (c->logN) {                                               \
    case 12: return fn##_12(__VA_ARGS__);                            \
    case 13: return fn##_13(__VA_ARGS__);                            \
    case 14: return fn##_14(__VA_ARGS__);                            \
    case 15: return fn##_15(__VA_ARGS__);                            \
    case 16: return fn##_16(__VA_ARGS__);                            \
    default: return fn##_17(__VA_ARGS__);                            \
    }

int ntt_fwd_canon(const fides_ctx *c, const LimbSet &s, cudaStream_t st) { FIDES_NTT_DISPATCH(ntt_fwd_canon, c, s, st) }
int ntt_fwd_submul(const fides_ctx *c, const LimbSet &s, cudaStream_t st) { FIDES_NTT_DISPATCH(ntt_fwd_submul, c, s, st) }
int ntt_fwd_switch_submul(const fides_ctx *c, const LimbSet &s, cudaStream_t st)
{
    FIDES_NTT_DISPATCH(ntt_fwd_switch_submul, c, s, st)
}
int ntt_fwd_submul_rot(const fides_ctx *c, const LimbSet &s, cudaStream_t st)
{
    FIDES_NTT_DISPATCH(ntt_fwd_submul_rot, c, s, st)
}
int ntt_fwd_raise(const fides_ctx *c, const LimbSet &s, cudaStream_t st) { FIDES_NTT_DISPATCH(ntt_fwd_raise, c, s, st) }
int ntt_fwd_hmrs(const fides_ctx *c, const LimbSet &s, cudaStream_t st) { FIDES_NTT_DISPATCH(ntt_fwd_hmrs, c, s, st) }
int ntt_inv_canon(const fides_ctx *c, const LimbSet &s, cudaStream_t st) { FIDES_NTT_DISPATCH(ntt_inv_canon, c, s, st) }
int ntt_fwd_cols(const fides_ctx *c, const LimbSet &s, cudaStream_t st) { FIDES_NTT_DISPATCH(ntt_fwd_cols, c, s, st) }
int ntt_inv_cols(const fides_ctx *c, const LimbSet &s, cudaStream_t st) { FIDES_NTT_DISPATCH(ntt_inv_cols, c, s, st) }
int ntt_rows_inner(const fides_ctx *c, const IPArgs &A, int limbs, int max_beta, cudaStream_t st)
{
    FIDES_NTT_DISPATCH(ntt_rows_inner, c, A, limbs, max_beta, st)
}

namespace {
void tune_one(const fides_ctx *c, int kind, int v, const LimbSet &s, cudaStream_t st)
{
    FIDES_NTT_DISPATCH(ntt_tune_one, c, kind, v, s, st)
}

// The autotuner times whole transforms by themselves and in chains, as programs
// queue them.  By itself a transform is timed with its launch latency and an
// idle GPU around it; in a chain of one size, neighbours share the SMs as they
// do in no program.  Tables of single passes by themselves ran the calls of a
// context 5 % slower than the default on average, chains alone up to 29 %
// (Rescale of 4 limbs of logN = 17): a tile replaces the default where both say
// that it is faster, by more than such timings differ.
constexpr int TUNE_CHAIN = 4;
constexpr float TUNE_GAIN = 0.98f;

// Best of three runs of `chain` transforms after one to warm up.
int tune_time(const fides_ctx *c, int kind, int v, const LimbSet &s, int chain, cudaStream_t st, cudaEvent_t e0,
              cudaEvent_t e1, float *best)
{
    for (int r = 0; r < 4; ++r) {
        cudaEventRecord(e0, st);
        for (int k = 0; k < chain; ++k) tune_one(c, kind, v, s, st);
        cudaEventRecord(e1, st);
        if (int rc = fides_check_cuda(cudaEventSynchronize(e1), "fides_ctx_autotune")) return rc;
        float ms = 0.f;
        cudaEventElapsedTime(&ms, e0, e1);
        if (r == 1 || (r > 1 && ms < *best)) *best = ms;
    }
    return FIDES_OK;
}
}  // namespace

// The table that tells what runs before autotuning (ntt_rules.h; launches of
// more limbs than it holds go by their size, too).
void ntt_default_table(const fides_ctx *c, unsigned char (&table)[4][FIDES_TUNE_MAX + 1])
{
    for (int kind = 0; kind < 4; ++kind)
        for (int n = 0; n <= FIDES_TUNE_MAX; ++n)
            table[kind][n] = (unsigned char)ntt_default_variant(kind, c->logN, c->fold, n);
}

void ntt_default_variants(fides_ctx *c)
{
    ntt_default_table(c, c->ntt_var);
    c->ntt_tuned = 0;
}

extern "C" int fides_ctx_autotune(fides_ctx *c, int max_limbs, void *stream)
{
    if (!c) return fides_set_error(FIDES_ERR_ARG, "fides_ctx_autotune: ctx is NULL");
    if (c->logN == 12) return FIDES_OK;   // one variant only
    const size_t limbs_avail = c->scratch_words / c->N;
    int maxn = std::min(std::min(max_limbs, FIDES_TUNE_MAX), (int)limbs_avail);
    if (maxn < 1) return fides_set_error(FIDES_ERR_ARG, "fides_ctx_autotune: max_limbs < 1");
    cudaStream_t st = (cudaStream_t)stream;
    const int was = fides_trace_set(0);
    cudaEvent_t e0, e1;
    cudaEventCreate(&e0);
    cudaEventCreate(&e1);
    int rc = FIDES_OK;
    for (int n = 1; n <= maxn && !rc; ++n) {
        LimbSet S;
        memset(&S, 0, sizeof(S));
        // limbs under the q-primes, in place, with operands (the forward row pass
        // that reads them) from limbs of the pool that no other segment transforms,
        // where it has that many
        for (int z0 = 0; z0 < n && S.nseg < FIDES_MAX_SEG; z0 += c->L) {
            Seg &g = S.seg[S.nseg++];
            g.count = std::min(c->L, n - z0);
            u64 *p = c->scratch + (size_t)z0 * c->N;
            g.aux = c->scratch + std::min((size_t)(n + z0), limbs_avail - g.count) * c->N;
            g.src = p; g.dst = p; g.out = p; g.side = nullptr; g.cst = nullptr; g.g = 0;
            g.prime0 = 0; g.src_step = 1; g.mode = 0; g.pstride = 0;
            S.total += g.count;
        }
        for (int kind = 0; kind < 4 && !rc; ++kind) {
            // (an inverse pass would take the constants for its final scale)
            for (int i = 0; i < S.nseg; ++i) S.seg[i].cst = kind == FWD_ROWS ? c->d_md_pinv : nullptr;
            const int def = ntt_default_variant(kind, c->logN, c->fold, n);
            float alone[NVAR], chain[NVAR];
            for (int v = 0; v < NVAR && !rc; ++v) rc = tune_time(c, kind, v, S, 1, st, e0, e1, &alone[v]);
            if (!rc) rc = tune_time(c, kind, def, S, TUNE_CHAIN, st, e0, e1, &chain[def]);
            int best = def;
            for (int v = 0; v < NVAR && !rc; ++v) {
                if (alone[v] >= TUNE_GAIN * alone[def]) continue;
                rc = tune_time(c, kind, v, S, TUNE_CHAIN, st, e0, e1, &chain[v]);
                if (!rc && chain[v] < TUNE_GAIN * chain[def] && chain[v] < chain[best]) best = v;
            }
            if (rc) break;
            c->ntt_var[kind][n] = (unsigned char)best;
        }
    }
    // counts above the tuned range keep the widest tile when it won at the top
    for (int kind = 0; kind < 4; ++kind)
        for (int n = maxn + 1; n <= FIDES_TUNE_MAX; ++n) c->ntt_var[kind][n] = c->ntt_var[kind][maxn];
    c->ntt_tuned = 1;
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    fides_trace_set(was);
    return rc;
}

extern "C" int fides_ctx_ntt_tile(const fides_ctx *c, int pass, int n_limbs)
{
    if (!c || pass < 0 || pass > 3 || n_limbs < 0) return 0;
    if (c->logN == 12) return (1 << 8) | NTT_LIMB_CTAS;
    const int v = ntt_compiled(variant_of(c, pass, n_limbs), c->fold, pass);
    const int S = pass == FWD_COLS || pass == INV_COLS ? ntt_col_stages(c->logN) : ntt_row_stages(c->logN);
    return (ntt_tile_width(v, S) << 8) | ntt_tile_ctas(v, S);
}

extern "C" int fides_ctx_tune_table(fides_ctx *c, unsigned char *table, int set)
{
    if (!c || !table) return fides_set_error(FIDES_ERR_ARG, "fides_ctx_tune_table: NULL argument");
    const size_t n = sizeof(c->ntt_var);
    if (!set) {
        memcpy(table, c->ntt_var, n);
        return FIDES_OK;
    }
    for (size_t i = 0; i < n; ++i)
        if (table[i] >= NVAR) return fides_set_error(FIDES_ERR_ARG, "fides_ctx_tune_table: variant %d out of range", table[i]);
    memcpy(c->ntt_var, table, n);
    // (a default table that was read out and is put back means the defaults)
    unsigned char def[4][FIDES_TUNE_MAX + 1];
    ntt_default_table(c, def);
    c->ntt_tuned = memcmp(c->ntt_var, def, n) != 0;
    return FIDES_OK;
}
