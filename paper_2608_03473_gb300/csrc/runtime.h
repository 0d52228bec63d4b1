// runtime.h -- host-side runtime shared by the CUDA translation units: the
// context (scratch, pinned staging, graph cache, timing events) and the
// helpers that size its buffers and upload token-set tables.  Not part of the
// C ABI.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <utility>
#include <vector>

#include "internal.h"

// A launch configuration of the tile kernel for one token set and mode:
// the record column height and the CTAs per SM (capped by occupancy).
struct lx_tuned {
    const lx_tokenset *ts;
    int mode;
    uint32_t ks, ctas, cls;   // cls: class-indexed table
    float ms;   // measured by lx_autotune (0 when set by hand)
    // what lx_autotune found fastest: LX_KERNEL_TILE or _WARP; LX_KERNEL_AUTO
    // where the entry-row kernels were, or nothing was chosen
    int kernel = 0;
    uint32_t warps = 0;       // warps per CTA it chose for the warp-tile kernel (0: as many as fit)
};

// Bytes of the pinned buffer for a kernel's launch record (lx_ctx::h_res).
constexpr size_t LAUNCH_RECORD_BYTES = 64;

// Inputs of one kind that the entry-row kernels refuse one after the other
// (tokens that backtrack across slices) are not tried each time: a refused
// attempt costs up to a pass (64 MiB of C-like text with a line of them 1.55
// ms a call, 1.35 without).  After the second refusal in a row one call goes
// without, then 3, 7 and at most 15 between attempts; one that is taken ends
// it, so that inputs refused now and then are all tried.
struct Refusals {
    uint32_t streak = 0, skip = 0;
    bool skips()   // whether this call goes without an attempt
    {
        if (skip) {
            skip--;
            return true;
        }
        return false;
    }
    void note(bool refused)
    {
        streak = refused ? std::min(streak + 1, 5u) : 0u;
        skip = streak ? (1u << (streak - 1)) - 1 : 0u;
    }
};

struct lx_ctx {
    int device = 0;
    int num_sms = 0;
    void *scratch = nullptr;
    size_t scratch_bytes = 0;
    void *h_res = nullptr;   // pinned: the launch record read back by lx_lex (LAUNCH_RECORD_BYTES)
    uint64_t timeout_ns = 20ull * 1000 * 1000 * 1000;
    uint32_t withhold = 0xFFFFFFFFu;   // failure-detection tests (lx_ctx_debug_withhold)
    lx_debug_counts counts = {};       // route tests (lx_ctx_debug_counts)
    std::vector<std::pair<uint64_t, int>> occupancy;   // (form << 32 | shared bytes) -> CTAs per SM
    std::vector<lx_tuned> tuned;                       // per (token set, mode); default otherwise
    // lx_lex_batch: device scratch, pinned staging (descriptors up, records
    // down), the capture stream and the cached graph with its shape key
    void *b_dev = nullptr;
    size_t b_dev_bytes = 0;
    void *b_host = nullptr;
    size_t b_host_bytes = 0;
    cudaStream_t b_stream = nullptr;
    cudaGraphExec_t b_exec = nullptr;
    std::vector<uint64_t> b_key;
    // the same for batches from entry rows (rows.cu): a batch that they refuse
    // keeps both
    cudaGraphExec_t r_exec = nullptr;
    std::vector<uint64_t> r_key;
    // lx_lex_enumerative: device scratch
    void *e_dev = nullptr;
    size_t e_dev_bytes = 0;
    // device buffers of lx_lex_host, its copy streams, per-piece events and
    // pinned per-piece records
    void *d_in = nullptr;
    size_t d_in_bytes = 0;
    void *d_out = nullptr;
    size_t d_out_bytes = 0;
    void *h_scratch = nullptr;   // pinned
    size_t h_scratch_bytes = 0;
    cudaStream_t s_in = nullptr, s_out = nullptr;
    std::vector<cudaEvent_t> ev_in, ev_lex;
    // the failed-lookahead guard's prepass (liveness.cu): device scratch
    void *lv_dev = nullptr;
    size_t lv_dev_bytes = 0;
    // lx_lex kernel choice (lx_ctx_set_kernel): LX_KERNEL_AUTO, _TILE or _WARP
    int kernel = 0;
    // warps per CTA of the warp-tile kernel (0: as many as shared memory holds)
    uint32_t warps = 0;
    // lx_lex_batch on the warp-tile kernel: the combined table of the last
    // batch's token sets (key: mode and the sets' serial numbers)
    void *wb_dev = nullptr;
    size_t wb_dev_bytes = 0;
    std::vector<uint64_t> wb_key;
    uint32_t wb_blob_bytes = 0, wb_rows = 0, wb_acc_off = 0, wb_sets_off = 0;
    bool wb_sync = false;   // every set has a synchronizing byte; rows.cu's table lies behind the other
    // the warp-tile kernel's geometry (lx_ctx_set_warp_geometry) and, in
    // LX_WARP_GEOMETRY_AUTO, the choice per (token set serial * 8 + mode)
    int warp_geometry = 0;
    std::vector<std::pair<uint64_t, bool>> warp_dense;
    // the warp-tile kernel's per-warp spill slots (kept tokens of a tile beyond its shared stage)
    void *w_spill = nullptr;
    size_t w_spill_bytes = 0;
    // refusals per (token set serial * 8 + mode), and of the batches of wb_key
    std::vector<std::pair<uint64_t, Refusals>> refusals;
    Refusals wb_refusals;
    // rows.cu: the scratch of small launches (its first part is zero between
    // them while small_clean), and the last launch's sequence number
    void *small = nullptr;
    size_t small_bytes = 0;
    bool small_clean = false;
    uint32_t seq = 0;
    // optional kernel timing
    bool timing = false;
    cudaEvent_t ev[2] = {nullptr, nullptr};
};

namespace lx {

// Batches: a document's tiles are consecutive in the launch's tile sequence
// from first_tile; `set` indexes the WSet array staged with the tables.
struct WDoc {
    const uint8_t *in;
    uint64_t n;
    uint32_t first_tile;
    uint32_t set;
};

// One token set's rows and maps in a batch's combined table (offsets from
// the table's start; the rows of all sets lie in one 16-bit address window).
struct WSet {
    uint32_t p_start, p_pre, p_slow, kmap_off, cmap_off, cut_off, ctx_off;
    uint32_t n_pat, pat[4];   // synchronizing byte values where they are few (rows.cu)
};

struct WDocRes {
    unsigned long long total;          // kept tokens of the document's tiles (any after a failure included)
    unsigned long long inv_fail_pos;   // ~min failure offset within the document, 0 = none
    unsigned long long inv_fail_tok;   // ~output index at that failure
    unsigned long long out_off1;       // output index of its first token + 1 (0: not yet resolved)
};

// lx_lex_host on the warp-tile kernel (lexwarp.cu): the K pieces [b[i],
// b[i+1]) of the host input (cut at certified bytes) each copied to a
// 16-byte aligned place on the device, lexed by their own launch with their
// own output range, and their tokens copied out after the previous pieces'
// once their records are in (same contract as lx_lex_host).  Uses the
// context's s_in / s_out streams and K of its ev_in / ev_lex events.  With
// sparse_limit != 0, LX_SPARSE or LX_LOOKAHEAD as lex_warp_device (some
// piece stopped early; the host buffers then hold nothing defined).
int lex_warp_host(lx_ctx *c, const lx_tokenset *ts, const uint8_t *h_in, uint64_t n, int mode, uint16_t *h_kinds,
                  uint32_t *h_lens, uint64_t capacity, const uint64_t *b, uint32_t K, uint64_t *n_tokens,
                  uint64_t *consumed, cudaStream_t st, uint64_t sparse_limit);
// LX_OK, LX_E_NOMEM for an allocation failure, LX_E_CUDA otherwise.
int cuda_err(cudaError_t e);
// Grow a device (grow) or pinned host (grow_host) buffer to at least `need`
// bytes; contents are not kept.
int grow(void **p, size_t *have, size_t need);
int grow_host(void **p, size_t *have, size_t need);
// The token set's tables on `device` (uploaded on first use): the walk-table
// blobs of each mode (both forms where both exist) and the plain scan table
// (nullptr where a table does not exist for this token set).
int ensure_device_tables(const lx_tokenset *ts, int device, DeviceTables *out);
// The warp-tile kernel (lexwarp.cu): whether lx_lex can take it for this
// token set, mode and input pointer (an event-code walk table and a 16-byte
// aligned input), and the call itself (same contract as lx_lex).  With
// sparse_limit != 0 a chunk longer than that many bytes (certified bytes too
// far apart) makes the call stop early and return LX_SPARSE, and backtracking
// steps beyond a budget proportional to n (failed lookahead) make it return
// LX_LOOKAHEAD, leaving the input to the enumerative path (guarded).
constexpr int LX_SPARSE = -100;   // internal status, never returned by the C ABI
bool warp_path_ok(const lx_tokenset *ts, int mode, const uint8_t *d_in);
// Lexing from the entry rows of fixed slices (rows.cu; same contract as
// lx_lex, any input alignment), for token sets with a synchronizing byte.
// LX_ROWS: the entry rows were not found or do not fit together, or there is no
// memory for the scratch; the caller lexes the input another way.
// LX_FAR: only because synchronizing bytes (or, with rows given, the starts
// from which they were found) lie too far apart.
constexpr int LX_ROWS = -102;   // internal statuses, never returned by the C ABI
constexpr int LX_FAR = -103;
bool rows_path_ok(const lx_tokenset *ts, int mode);
// Rows already found, one every `step` bytes from the input's first 16-byte
// block on, and the error word of the kernels that find them.
struct RowsGiven {
    uint16_t *rows;
    uint32_t step;
    const unsigned int *error;
    bool open;   // whether a token may fail in a later slice than its own
};
int lex_rows_device(lx_ctx *c, const lx_tokenset *ts, const uint8_t *d_in, uint64_t n, int mode, uint16_t *d_kinds,
                    uint32_t *d_lens, uint64_t capacity, uint64_t *n_tokens, uint64_t *consumed, cudaStream_t st,
                    const RowsGiven *given = nullptr);
// lx_lex_host on the same kernels: the K pieces [b[i], b[i + 1]) of the host
// input (cut at certified bytes) each copied in, lexed by its own launch into
// its own output range, and copied out after the previous pieces' tokens.  Uses
// the context's s_in / s_out streams and K of its events where K > 1; LX_ROWS
// and LX_FAR as above (the host buffers then hold nothing defined).
int lex_rows_host(lx_ctx *c, const lx_tokenset *ts, const uint8_t *h_in, uint64_t n, int mode, uint16_t *h_kinds,
                  uint32_t *h_lens, uint64_t capacity, const uint64_t *b, uint32_t K, uint64_t *n_tokens,
                  uint64_t *consumed, cudaStream_t st);
// lx_lex_batch in one launch from entry rows (rows.cu), with the context's
// combined table (its key: part of the graph's); LX_ROWS, LX_FAR as above.
int lex_batch_rows(lx_ctx *c, const std::vector<uint64_t> &sets_key, const lx_doc *docs, uint32_t n_docs, int mode,
                   uint16_t *d_kinds, uint32_t *d_lens, uint64_t capacity, lx_doc_result *results, uint64_t *n_total,
                   cudaStream_t st);
// lex_rows_device with the entry rows found by enumerating contexts (ctxmap.cu): any
// token set with a walk and a scan table.  With `spec`, the speculative path's
// predictions and rounds as well (model: nullptr for BOUNDARY everywhere).
// LX_ROWS, LX_FAR as above.
bool contexts_path_ok(const lx_tokenset *ts, int mode);
int lex_contexts_device(lx_ctx *c, const lx_tokenset *ts, const uint8_t *d_in, uint64_t n, int mode, uint16_t *d_kinds,
                        uint32_t *d_lens, uint64_t capacity, uint64_t *n_tokens, uint64_t *consumed, cudaStream_t st,
                        lx_model *model, lx_spec_stats *spec);
// Warps per CTA of the warp-tile kernel (not of the entry-row kernels, whose
// shared memory differs: they take what fits) on (ts, mode): the context's
// setting, else lx_autotune's choice, else 0 (as many as fit).
uint32_t warps_setting(const lx_ctx *c, const lx_tokenset *ts, int mode);
// lx_lex_async (lexwarp.cu): the warp-tile kernel and a status kernel that
// writes the result record to device memory; no synchronization, no fallback.
int lex_warp_async(lx_ctx *c, const lx_tokenset *ts, const uint8_t *d_in, uint64_t n, int mode, uint16_t *d_kinds,
                   uint32_t *d_lens, uint64_t capacity, lx_async_result *d_result, cudaStream_t st);
// lx_lex_batch in one launch of the warp-tile kernel (lexwarp.cu): every
// document of every token set, the sets' class-form tables side by side in
// shared memory, the output in document order.  LX_SPARSE when not
// applicable (a table without a class form, rows beyond the 16-bit window,
// an unaligned document): the caller takes the per-set tile kernels.
int lex_batch_warp(lx_ctx *c, const lx_tokenset *const *sets, uint32_t n_sets, const lx_doc *docs, uint32_t n_docs,
                   int mode, uint16_t *d_kinds, uint32_t *d_lens, uint64_t capacity, lx_doc_result *results,
                   uint64_t *n_total, cudaStream_t st);
int lex_warp_device(lx_ctx *c, const lx_tokenset *ts, const uint8_t *d_in, uint64_t n, int mode, uint16_t *d_kinds,
                    uint32_t *d_lens, uint64_t capacity, uint64_t *n_tokens, uint64_t *consumed, cudaStream_t st,
                    uint64_t sparse_limit);
// Internal status: a scan ran past its step budget (failed lookahead, or a
// token spanning many chunks); the caller runs the input again with the
// failed-lookahead guard.  Never returned by the C ABI.
constexpr int LX_LOOKAHEAD = -101;
// lx_lex_enumerative (enumerate.cu) with the failed-lookahead guard from the
// start when `guard` (the caller saw a scan run past its budget already), on
// the chunks at once when `chunks` (the contexts of ctxmap.cu do not serve it).
int lex_enumerative_device(lx_ctx *c, const lx_tokenset *ts, const uint8_t *d_in, uint64_t n, int mode,
                           uint16_t *d_kinds, uint32_t *d_lens, uint64_t capacity, uint64_t *n_tokens,
                           uint64_t *consumed, cudaStream_t stream, bool guard, bool chunks);
// The guard's prepass (liveness.cu): the liveness automaton's state at every
// offset 0..n of the input into d_out[n + 1] (nullptr: the context's scratch);
// *live receives the array, *member the automaton's member bitsets on the
// device.  LX_E_TOOBIG when the token set has no liveness automaton.
int liveness_device(lx_ctx *c, const lx_tokenset *ts, const uint8_t *d_in, uint64_t n, uint8_t *d_out,
                    cudaStream_t s, const uint8_t **live, const uint32_t **member);
// The entry-context model (model.cu): number of contexts it scores, and the
// BF16 prediction of the entry context of every chunk start (0xFFFE =
// BOUNDARY) into guess[M], restricted to the candidates of the byte before.
uint32_t model_contexts(const lx_model *m);
int model_predict(lx_model *m, const uint8_t *in, uint64_t n, const uint64_t *start, const uint32_t *cinfo,
                  const uint8_t *scan_blob, uint32_t cbeg_off, uint32_t cand_off, uint32_t M, uint16_t *guess,
                  cudaStream_t s);

}  // namespace lx
