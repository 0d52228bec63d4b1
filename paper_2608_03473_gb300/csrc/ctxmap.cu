// ctxmap.cu -- entry contexts of every slice by enumeration, for token sets
// (or inputs) without synchronizing bytes: what lx_lex_enumerative and
// lx_lex_speculative take first, lex_rows (rows.cu) lexing from the rows
// found.  enumerate.cu keeps the forms these hand over to.
//
// enumerate.cu scans every 4096-byte chunk with one lane per candidate
// context, so a call costs a few thousand dependent byte steps however small
// the input is, and it scans all chunks once more to write their tokens.
// Here a lane has 128 bytes and all candidates at once:
//   cm_starts   per 4096-byte target the chunk start of enumerate.cu (within
//               256 bytes, after the byte with the fewest contexts), and per
//               128-byte slice a start of its own within its first 64 bytes by
//               the same rule (none: the slice joins the one before);
//   cm_maps     from each start to the next, the walk of lex_rows without its
//               events, from up to six candidates at a time (independent
//               chains, one class lookup for all): the context left in per
//               candidate, as eight 4-bit indexes, and the row at every
//               128-byte boundary passed.  A warp composes its tile's 32 maps;
//   cm_fold, cm_top   the tiles' maps composed: each tile's true entry;
//   cm_rows     the true row at every slice boundary, for lex_rows.
// Backtracking inside a slice is replayed (hard_run); a candidate that fails,
// or that would have to backtrack to before its slice, is dead (15).  Where
// the true chain dies without a lexing failure, lex_rows finds rows that do
// not fit and the caller takes the chunks of enumerate.cu.
// cm_guess, cm_round and cm_judge play the speculative path's rounds on the
// chunks' maps.
//
// 96 MiB of the refused C-like set, filtered: 7 143 -> 542 us a call (starts
// 32, maps 340, fold and top 7, rows 9, lex_rows 135); 160 MiB through the
// speculative call with a model 11.4 -> 1.20 ms (maps 480, the model 300,
// lex_rows 215).  cm_maps is bound by the shared-memory pipe: fifteen wavefronts
// a byte step (six rows and the class map, lanes in unrelated rows two to four
// apart; rows spread over the banks took it from 420 to 375).

#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "rows.cuh"
#include "runtime.h"

namespace lx {
namespace {

constexpr uint32_t CT = 4096;      // bytes per tile: one chunk target of enumerate.cu
constexpr uint32_t CL = 128;       // bytes per slice, one lane each
constexpr uint32_t CWIN = 256;     // a chunk start is searched in the target's first CWIN bytes
constexpr uint32_t SWIN = 64;      // a slice's own start in its first SWIN
constexpr uint32_t KMAX = 8;       // candidate contexts of a start (BOUNDARY included)
constexpr uint32_t DEAD = 15;      // context index: none
constexpr uint32_t IDENT = 0x76543210u;
constexpr uint32_t NO_START = 255;
constexpr int CM_NT = 512;
constexpr int MAP_NT = 640;        // two CTAs of 20 warps per SM
constexpr int TOP_NT = 1024;
// Tiles searched for the next start: one lane walks all bytes up to it, 70 ns
// each (64 MiB of C-like text with one line of 30 KiB, which has no start: 2.4
// ms; 14.1 through the chunks of enumerate.cu, where four tiles sent it).
constexpr uint32_t FAR_TILES = 16;
constexpr uint64_t HARD_MAX = 64 * 4 * CT + 4096;   // steps of a stretch replayed with backtracking, at most
constexpr uint64_t NOPOS64 = ~0ull;
constexpr int CLAIM = 12;          // P.counts: the tiles cm_maps has given out
constexpr int ROUNDS = 8;          // speculative fix-up rounds (enumerate.cu: SPEC_ROUNDS)

struct CParams {
    RParams R;                 // input, table, and the record whose error word the kernels flag
    const uint16_t *cbeg, *cand;   // scan table: candidate states after every byte
    uint8_t *starts;           // per slice: its start's offset, NO_START
    uint32_t *pmap;            // per slice: map of the slices before it in its tile
    uint32_t *tmap;            // per tile: its 32 slices' map
    uint32_t *bmap;            // per TOP_NT tiles: their map
    uint8_t *tent;             // per tile: context index at its first start
    uint16_t *rf;              // per slice boundary and candidate of the start before it: row there (0: dead)
    uint32_t n_tiles;
    // chunks (as enumerate.cu numbers them; positions relative to the input)
    uint64_t *cstart;          // [n_tiles] NOPOS64: none
    uint32_t *cinfo;           // byte before << 8 | candidates
    uint8_t *cur, *nxt;        // assumed context index of each chunk, before and after a round
    const uint16_t *guess;     // predicted contexts (nullptr: BOUNDARY)
    unsigned int *counts;      // [ROUNDS] chunks whose entry a round changed, then those the judge changed
};

__device__ __forceinline__ uint32_t map_at(uint32_t m, uint32_t k)   // context index k through m; DEAD stays
{
    return (uint32_t)(((0xFFFFFFFFull << 32) | m) >> (4 * k)) & 15u;
}
// `then` after `first`: its eight values as bytes, picked by PRMT with the
// nibbles of `first`; where one of those is DEAD (bit 3) the result is.
__device__ __forceinline__ uint32_t compose(uint32_t first, uint32_t then)
{
    const uint32_t x = then & 0x0F0F0F0Fu, y = (then >> 4) & 0x0F0F0F0Fu;
    const uint32_t lo = __byte_perm(x, y, 0x5140), hi = __byte_perm(x, y, 0x7362);
    uint32_t r0 = __byte_perm(lo, hi, first & 0x7777u), r1 = __byte_perm(lo, hi, (first >> 16) & 0x7777u);
    r0 = (r0 | (r0 >> 4)) & 0x00FF00FFu;
    r1 = (r1 | (r1 >> 4)) & 0x00FF00FFu;
    r0 = __byte_perm(r0, r1, 0x6420);
    return r0 | ((first & 0x88888888u) >> 3) * 15u;
}

__device__ __forceinline__ uint32_t n_cand(const CParams &P, uint32_t b)
{
    return 1u + __ldg(P.cbeg + b + 1) - __ldg(P.cbeg + b);
}

__global__ void __launch_bounds__(CM_NT) cm_starts(CParams P)
{
    __shared__ uint8_t cnt[256];
    for (uint32_t b = threadIdx.x; b < 256; b += blockDim.x) cnt[b] = (uint8_t)min(255u, n_cand(P, b));
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31, nw = gridDim.x * (blockDim.x / 32);
    const uint8_t *in = P.R.in;
    const uint64_t n = P.R.n;
    for (uint32_t t = (blockIdx.x * blockDim.x + threadIdx.x) / 32; t < P.n_tiles; t += nw) {
        const uint64_t T0 = (uint64_t)t * CT;
        // the chunk start: fewest candidates, then the first
        uint32_t key = NONE;
        if (t > 0) {
#pragma unroll
            for (uint32_t i = 0; i < CWIN / 32; i++) {
                const uint32_t o = (CWIN / 32) * lane + i;
                if (T0 + o < n) key = min(key, ((uint32_t)cnt[__ldg(in + T0 + o - 1)] << 16) | o);
            }
        }
        key = __reduce_min_sync(0xffffffffu, key);
        if (t == 0) key = (1u << 16) | P.R.lo;   // the input's start: BOUNDARY alone
        const uint32_t kc = key >> 16, co = key & 0xFFFFu;
        const bool chunk = kc <= KMAX;
        if (lane == 0) {
            P.cstart[t] = chunk ? T0 + co - P.R.lo : NOPOS64;
            P.cinfo[t] = chunk ? (t ? (uint32_t)__ldg(in + T0 + co - 1) << 8 : 0u) | kc : 0u;
        }
        // the slices' own starts, after the chunk's
        const uint32_t b0 = lane * CL;
        uint32_t s = NO_START;
        if (chunk && co / CL == lane) {
            s = co - b0;
        } else if (T0 + b0 < n && (!chunk || b0 > co)) {
            uint32_t best = KMAX + 1, prev = __ldg(in + T0 + b0 - 1);
            const uint64_t left = n - (T0 + b0);
            const uint32_t lim = left < SWIN ? (uint32_t)left : SWIN;
            for (uint32_t o = 0; o < lim; o += 16) {
                uint4 v = make_uint4(0, 0, 0, 0);
                if (o + 16 <= left) {
                    v = ldg16(in + T0 + b0 + o);
                } else {
                    uint32_t w[4] = {0, 0, 0, 0};
                    for (uint32_t k = 0; o + k < left; k++) w[k >> 2] |= (uint32_t)__ldg(in + T0 + b0 + o + k) << (8 * (k & 3));
                    v = make_uint4(w[0], w[1], w[2], w[3]);
                }
#pragma unroll
                for (uint32_t k = 0; k < 16; k++) {
                    const uint32_t c = cnt[prev];
                    if (c < best && o + k < lim) {
                        best = c;
                        s = o + k;
                    }
                    const uint32_t w = k < 4 ? v.x : k < 8 ? v.y : k < 12 ? v.z : v.w;
                    prev = (w >> (8 * (k & 3))) & 0xFFu;
                }
            }
        }
        const uint64_t sl = (uint64_t)t * 32 + lane;
        if (sl < P.R.n_slices) P.starts[sl] = (uint8_t)s;
    }
}

// Four byte steps over w from CH rows at once.  Six: the best start of nearly
// every slice has at most that many candidates (four after a newline of the
// refused C-like set, six after a space), and one lane with more makes its
// warp walk twice (four at a time: 27 % more instructions).
constexpr uint32_t CH = 6;
#define LXM_ROW(E) "lop3.b32 a, " E ", t, %7, 0xD8;\n\tld.shared.u16 " E ", [a];\n\t"
#define LXM_ROWS LXM_ROW("%0") LXM_ROW("%1") LXM_ROW("%2") LXM_ROW("%3") LXM_ROW("%4") LXM_ROW("%5")
#define LXM_SROW(E)                                                            \
    "shr.b32 a, " E ", 6;\n\tlop3.b32 a, a, 0x7C, t, 0x6A;\n\t"                \
    "lop3.b32 a, " E ", a, %7, 0xD8;\n\tld.shared.u16 " E ", [a];\n\t"
#define LXM_SROWS LXM_SROW("%0") LXM_SROW("%1") LXM_SROW("%2") LXM_SROW("%3") LXM_SROW("%4") LXM_SROW("%5")
#define LXM_C(SEL) "prmt.b32 t, %6, %8, " SEL ";\n\tld.shared.u8 t, [t];\n\t" LXM_SROWS
#define LXM_OPS(MASK)                                                          \
    : "+r"(e[0]), "+r"(e[1]), "+r"(e[2]), "+r"(e[3]), "+r"(e[4]), "+r"(e[5])   \
    : "r"(w), "r"(MASK), "r"(cm) : "memory"
template <int FORM>
__device__ __forceinline__ void wwords(uint32_t (&e)[CH], uint32_t w, uint32_t cm)
{
    if (FORM == FORM_BYTE)
        asm volatile("{\n\t.reg .b32 t, a;\n\tshl.b32 t, %6, 1;\n\t" LXM_ROWS "shr.b32 t, %6, 7;\n\t" LXM_ROWS
                     "shr.b32 t, %6, 15;\n\t" LXM_ROWS "shr.b32 t, %6, 23;\n\t" LXM_ROWS "}" LXM_OPS(0x1FEu));
    else
        asm volatile("{\n\t.reg .b32 t, a;\n\t" LXM_C("0x7650") LXM_C("0x7651") LXM_C("0x7652") LXM_C("0x7653") "}"
                     LXM_OPS(0xFFu));
}

// The row at boundary position p (a multiple of CL) entered with candidate k.
__device__ __forceinline__ void put_row(const CParams &P, const REnv &E, uint64_t p, uint32_t k, uint32_t e)
{
    if (p < P.R.n) P.rf[(p / CL) * KMAX + k] = (uint16_t)((e & ~0xFFu) - E.tb);
}

// [s, ne) from `row` token by token, with backtracking; returns the row at
// ne, or SLOW where the candidate fails or would backtrack to before s.
template <int FORM>
__device__ __noinline__ uint32_t hard_run(const CParams &P, const REnv &E, uint64_t s, uint64_t ne, uint32_t row,
                                          uint32_t k)
{
    uint32_t q = row;
    uint64_t r = acc_code(E, q) && q != E.start ? s : NOPOS64, p = s;
    for (uint64_t steps = min(64 * (ne - s) + 4096, HARD_MAX); p < ne; steps--) {
        if (steps == 0) {   // repeated failed lookahead: left to the guarded scans
            atomicOr(P.R.error(), ERR_ROWS);
            return E.slow;
        }
        const uint32_t v = wstep<FORM, true>(E, q, __ldg(P.R.in + p));
        if (v != E.slow && v != E.pre) {
            if (v & 0xFEu) r = NOPOS64;
            q = v;
            p++;
            if (p % CL == 0) put_row(P, E, p, k, q);   // (written again when the token backtracks)
            if (acc_code(E, q)) r = p;
        } else if (r == NOPOS64 || r == s) {
            // from s itself: the token ended there, which is another context's entry
            return E.slow;
        } else {
            p = r;
            q = E.start;
            r = NOPOS64;
        }
    }
    return q;
}

// SLOW of a row that neither accepts nor is free of accepting rows before it
// is a backtrack to be replayed: such rows' transitions to SLOW are sent to
// the PRE row (HARD here), which absorbs every byte like SLOW.  A chain that
// ends in SLOW is dead: its token ended at a byte that starts none, or has no
// accepting prefix.
__device__ void hard_rows(const CParams &P, uint8_t *smem, const REnv &E)
{
    const uint8_t *noacc = P.R.blob + P.R.noacc_off, *acc = P.R.blob + P.R.acc_off;
    uint32_t *tab = reinterpret_cast<uint32_t *>(smem + (E.tb - smem_u32(smem)));
    const uint32_t pre = P.R.p_pre >> E.shift, start = P.R.p_start >> E.shift, h = E.pre * 0x10001u, sl = E.slow * 0x10001u;
    for (uint32_t i = threadIdx.x; i < P.R.rows_bytes / 4; i += blockDim.x) {
        const uint32_t r = (4 * i) >> E.shift;
        if (r == pre) {
            tab[i] = h;
        } else if (r > 0 && r < start && !__ldg(acc + r) && !__ldg(noacc + r)) {
            const uint32_t d = __vcmpeq2(tab[i], sl);   // 0xFFFF where the entry is SLOW
            tab[i] = (tab[i] & ~d) | (h & d);
        }
    }
}

// A block of 16 bytes at p that a chain entered in `row` and left in HARD, byte
// by byte: its token's last accepting position mostly lies in the block (the
// wrong candidates read text as code and meet a "4en" at every turn).  HARD
// where it lies before.
template <int FORM>
__device__ uint32_t block_fix(const REnv &E, const uint8_t *in, uint64_t p, bool at_start, uint32_t row)
{
    uint32_t q = row, r = acc_code(E, row) ? 0u : NONE;
    for (uint32_t j = 0; j < 16;) {
        const uint32_t v = wstep<FORM, true>(E, q, __ldg(in + p + j));
        if (v == E.slow) return v;
        if (v == E.pre) {
            if (r == NONE) return v;
            if (r == 0 && at_start) return E.slow;   // as in hard_run
            j = r;
            q = E.start;
            r = NONE;
            continue;
        }
        if (v & 0xFEu) r = NONE;
        q = v;
        j++;
        if (acc_code(E, q)) r = j;
    }
    return q;
}

template <int FORM>
__global__ void __launch_bounds__(MAP_NT, 2) cm_maps(CParams P)
{
    extern __shared__ __align__(16) uint8_t smem[];
    REnv E;
    if (!stage_table<FORM, true>(P.R, smem, E)) return;
    __syncthreads();
    hard_rows(P, smem, E);
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31;
    const uint8_t *in = P.R.in;
    const uint64_t n = P.R.n;
    for (;;) {
        uint32_t t = 0;
        if (lane == 0) t = atomicAdd(P.counts + CLAIM, 1u);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= P.n_tiles) break;
        const uint64_t T0 = (uint64_t)t * CT, sl = (uint64_t)t * 32 + lane;
        const uint32_t so = sl < P.R.n_slices ? P.starts[sl] : NO_START;
        const bool has = so != NO_START;
        // the next start: in this tile, else in the next few
        const uint32_t hs = __ballot_sync(0xffffffffu, has);
        const uint32_t above = hs & ~((2u << lane) - 1u);
        uint64_t ne = 0;
        {
            const uint32_t src = above ? __ffs(above) - 1 : 0;
            const uint32_t o = __shfl_sync(0xffffffffu, so, src);
            uint64_t far = n;
            if (hs) {   // where the tile's last start leads
                bool found = false;
                for (uint32_t f = 1; f <= FAR_TILES && !found; f++) {
                    const uint64_t x = ((uint64_t)t + f) * 32 + lane;
                    if (((uint64_t)t + f) * 32 >= P.R.n_slices) {
                        found = true;
                        break;
                    }
                    const uint32_t fo = x < P.R.n_slices ? P.starts[x] : NO_START;
                    const uint32_t fs = __ballot_sync(0xffffffffu, fo != NO_START);
                    if (fs) {
                        const uint32_t fl = __ffs(fs) - 1;
                        far = ((uint64_t)t + f) * CT + fl * CL + __shfl_sync(0xffffffffu, fo, fl);
                        found = true;
                    }
                }
                if (!found && lane == 0) atomicOr(P.R.error(), ERR_FAR);   // starts too far apart
                if (!found) far = T0;   // walk nothing
            }
            ne = above ? T0 + src * CL + o : far;
        }
        const uint64_t s = T0 + lane * CL + so;
        const uint32_t pb = has && s > P.R.lo ? __ldg(in + s - 1) : 0u;    // the byte before
        const uint32_t c0 = has ? __ldg(P.cbeg + pb) : 0u;
        const uint32_t nc = !has ? 0u : s == P.R.lo ? 1u : 1u + __ldg(P.cbeg + pb + 1) - c0;
        const uint32_t b0 = has ? __ldg(in + s) : 0u;
        uint32_t map = has ? NONE : IDENT;   // every index DEAD, or the identity
#pragma unroll 1
        for (uint32_t g = 0; __any_sync(0xffffffffu, nc > g); g += CH) {
            if (nc <= g) continue;
            uint32_t e[CH];
            uint64_t p = s;
            // the candidates' rows; one whose token does not read the next
            // byte is not entered in, BOUNDARY stands for it
#pragma unroll
            for (uint32_t i = 0; i < CH; i++) {
                const uint32_t k = g + i;
                e[i] = E.slow;
                if (k == 0) {
                    e[i] = E.start;
                } else if (k < nc) {
                    const uint32_t row = E.tb + ((1u + __ldg(P.cand + c0 + k - 1)) << E.shift);
                    const uint32_t v = wstep<FORM, true>(E, row, b0);
                    if (v != E.slow && v != E.pre && !(v & 0xFEu)) e[i] = row;
                }
            }
            auto scalar = [&](uint64_t to) {
                for (; p < to; p++) {
                    const uint32_t b = __ldg(in + p);
                    const uint32_t x = FORM == FORM_BYTE ? b << 1 : lds_u8(E.cmap + b);
#pragma unroll
                    for (uint32_t i = 0; i < CH; i++)
                        e[i] = lds_u16(FORM == FORM_BYTE ? (e[i] & ~0x1FEu) | x
                                                         : (e[i] & ~0xFFu) | (x ^ ((e[i] >> 6) & 0x7Cu)));
                }
            };
            auto words = [&](uint64_t to) {   // p a multiple of 4
                for (; p + 4 <= to; p += 4) wwords<FORM>(e, __ldg(reinterpret_cast<const uint32_t *>(in + p)), E.cmap);
            };
            auto mark = [&]() {
                if (p % CL == 0 && p > s && p < n) {
                    uint32_t r[CH / 2];
#pragma unroll
                    for (uint32_t i = 0; i < CH / 2; i++)
                        r[i] = ((e[2 * i] & ~0xFFu) - E.tb) | (((e[2 * i + 1] & ~0xFFu) - E.tb) << 16);
                    uint16_t *q = P.rf + (p / CL) * KMAX;
                    if (g == 0) *reinterpret_cast<uint4 *>(q) = make_uint4(r[0], r[1], r[2], 0);
                    else *reinterpret_cast<uint32_t *>(q + CH) = r[0];   // candidates 6 and 7
                }
            };
            const uint64_t up = (s + 15) & ~(uint64_t)15, b16 = up < ne ? up : ne;
            scalar(min((s + 3) & ~(uint64_t)3, b16));
            words(b16);
            if (p < b16) scalar(b16);
            mark();
            uint4 A = p + 16 <= ne ? ldg16(in + p) : make_uint4(0, 0, 0, 0);
            while (p + 16 <= ne) {
                const uint4 c = A;
                if (p + 32 <= ne) A = ldg16(in + p + 16);
                const uint32_t w[CH] = {e[0], e[1], e[2], e[3], e[4], e[5]};
                wwords<FORM>(e, c.x, E.cmap);
                wwords<FORM>(e, c.y, E.cmap);
                wwords<FORM>(e, c.z, E.cmap);
                wwords<FORM>(e, c.w, E.cmap);
#pragma unroll
                for (uint32_t i = 0; i < CH; i++)
                    if (e[i] == E.pre && w[i] != E.pre) e[i] = block_fix<FORM>(E, in, p, p == s, w[i]);
                p += 16;
                mark();
            }
            if (p < ne) {
                words(ne);
                scalar(ne);
            }
#pragma unroll
            for (uint32_t i = 0; i < CH; i++)
                if (e[i] == E.pre)
                    e[i] = hard_run<FORM>(P, E, s, ne,
                                          g + i == 0 ? E.start : E.tb + ((1u + __ldg(P.cand + c0 + g + i - 1)) << E.shift), g + i);
            if (ne < n && ne > s) {   // the context at the next start
                const uint32_t nb = __ldg(in + ne), lb = __ldg(in + ne - 1);
                const uint32_t d0 = __ldg(P.cbeg + lb), dn = __ldg(P.cbeg + lb + 1) - d0;
#pragma unroll
                for (uint32_t i = 0; i < CH; i++) {
                    const uint32_t k = g + i;
                    if (k >= KMAX) break;
                    uint32_t x = DEAD;
                    if (e[i] != E.slow && e[i] < E.start) {
                        const uint32_t v = wstep<FORM, true>(E, e[i], nb);
                        if (v == E.slow ? acc_code(E, e[i]) != 0 : (v & 0xFEu) != 0) {
                            x = 0;   // the token ends there
                        } else if (v != E.slow && v != E.pre) {
                            const uint32_t st = ((e[i] - E.tb) >> E.shift) - 1u;
                            for (uint32_t j = 0; j < dn && j < KMAX - 1; j++)
                                if (__ldg(P.cand + d0 + j) == st) x = j + 1;
                        }
                    }
                    map = (map & ~(15u << (4 * k))) | (x << (4 * k));
                }
            }
        }
        // compose the tile's slices
        uint32_t incl = map;
        for (uint32_t o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl = compose(y, incl);
        }
        uint32_t excl = __shfl_up_sync(0xffffffffu, incl, 1);
        if (lane == 0) excl = IDENT;
        if (sl < P.R.n_slices) P.pmap[sl] = excl;
        if (lane == 31) P.tmap[t] = incl;
    }
}

// Inclusive compositions of the block's words, thread by thread.
__device__ __forceinline__ uint32_t block_compose(uint32_t x, uint32_t *sh)
{
    const uint32_t lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (uint32_t o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x = compose(y, x);
    }
    if (lane == 31) sh[w] = x;
    __syncthreads();
    if (w == 0) {
        uint32_t v = sh[lane];
        for (uint32_t o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
            if (lane >= o) v = compose(y, v);
        }
        sh[lane] = v;
    }
    __syncthreads();
    return w ? compose(sh[w - 1], x) : x;
}

// Every tile's true entry, in two launches: the maps of TOP_NT tiles composed
// by a block (cm_fold), then each block composes those of the blocks before it
// and follows its tiles from BOUNDARY at the input's start (cm_top).  (One
// block over all tiles took 21 us at 96 MiB and 40 at 160, on one SM.)
__global__ void __launch_bounds__(TOP_NT) cm_fold(CParams P)
{
    __shared__ uint32_t sh[32];
    const uint32_t t = blockIdx.x * TOP_NT + threadIdx.x;
    const uint32_t m = block_compose(t < P.n_tiles ? __ldg(P.tmap + t) : IDENT, sh);
    if (threadIdx.x == TOP_NT - 1) P.bmap[blockIdx.x] = m;
}

__global__ void __launch_bounds__(TOP_NT) cm_top(CParams P)
{
    __shared__ uint32_t sh[32], sh2[32], first;
    const uint32_t per = (blockIdx.x + TOP_NT - 1) / TOP_NT;   // blocks before this one, for each thread
    const uint32_t b0 = min(blockIdx.x, threadIdx.x * per), b1 = min(blockIdx.x, b0 + per);
    uint32_t m = IDENT;
    for (uint32_t i = b0; i < b1; i++) m = compose(m, __ldg(P.bmap + i));
    m = block_compose(m, sh);
    if (threadIdx.x == TOP_NT - 1) first = m;
    const uint32_t t = blockIdx.x * TOP_NT + threadIdx.x;
    const uint32_t incl = block_compose(t < P.n_tiles ? __ldg(P.tmap + t) : IDENT, sh2);   // (its barriers publish `first`)
    const uint32_t k = map_at(incl, map_at(first, 0));
    if (t == 0) P.tent[0] = 0;
    if (t + 1 < P.n_tiles) P.tent[t + 1] = (uint8_t)k;
}

// The true row at every slice boundary: each slice's start hands out those up
// to the next start.
__global__ void __launch_bounds__(CM_NT) cm_rows(CParams P)
{
    const uint64_t total = ((uint64_t)P.n_tiles * 32 + 31) & ~31ull;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (uint64_t)gridDim.x * blockDim.x) {
        if (i == 0) P.R.rows[0] = (uint16_t)P.R.p_start;
        if (i >= P.R.n_slices || P.starts[i] == NO_START) continue;
        const uint32_t k = map_at(P.pmap[i], P.tent[i / 32]);
        for (uint64_t m = i + 1; m < P.R.n_slices; m++) {
            const uint32_t r = k == DEAD ? 0u : P.rf[m * KMAX + k];
            P.R.rows[m] = (uint16_t)(r && r < P.R.p_start ? r : ROW_DEAD);
            const uint32_t so = P.starts[m];   // a start at offset 0 lies at the boundary itself
            if (so != NO_START) break;
        }
    }
}

// ---- the speculative path's rounds on the chunks' maps ----
// A chunk runs to the next chunk start; its map is its tile's, composed with
// those of tiles without one.
__device__ __forceinline__ uint32_t chunk_exit(const CParams &P, uint32_t j, uint32_t k)
{
    k = map_at(__ldg(P.tmap + j), k);
    for (uint32_t i = j + 1; i < P.n_tiles && P.cstart[i] == NOPOS64; i++) k = map_at(__ldg(P.tmap + i), k);
    return k;
}

__global__ void cm_guess(CParams P)
{
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < P.n_tiles; j += gridDim.x * blockDim.x) {
        uint32_t k = 0;
        const uint32_t g = j > 0 && P.guess && P.cstart[j] != NOPOS64 ? P.guess[j] : 0xFFFEu;
        if (g != 0xFFFEu) {
            const uint32_t b = P.cinfo[j] >> 8, c0 = P.cbeg[b], c1 = P.cbeg[b + 1];
            k = DEAD;
            for (uint32_t i = c0; i < c1 && i < c0 + KMAX - 1; i++)
                if (P.cand[i] == g) k = i - c0 + 1;
        }
        P.cur[j] = (uint8_t)k;
    }
}

// One round: every chunk's scan from its assumed entry, then every chunk
// takes its predecessor's exit; counts the chunks whose entry changed.
__global__ void cm_round(CParams P, uint32_t round)
{
    uint32_t changed = 0;
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < P.n_tiles; j += gridDim.x * blockDim.x) {
        uint32_t k = P.cur[j];
        if (j > 0 && P.cstart[j] != NOPOS64) {
            uint32_t q = j - 1;
            while (q > 0 && P.cstart[q] == NOPOS64) q--;
            const uint32_t x = chunk_exit(P, q, P.cur[q]);
            if (x != DEAD && x != k) {
                k = x;
                changed++;
            }
        }
        P.nxt[j] = (uint8_t)k;
    }
    changed = __reduce_add_sync(0xffffffffu, changed);
    if ((threadIdx.x & 31) == 0 && changed) atomicAdd(P.counts + round, changed);
}

// Chunks that the judge scans again: entries still changing (cur: before the
// last round, nxt: after it) or not the true ones.
__global__ void cm_judge(CParams P)
{
    uint32_t changed = 0;
    for (uint32_t j = blockIdx.x * blockDim.x + threadIdx.x; j < P.n_tiles; j += gridDim.x * blockDim.x) {
        if (P.cstart[j] == NOPOS64 || P.tent[j] == DEAD) continue;
        if (P.cur[j] != P.nxt[j] || P.nxt[j] != P.tent[j]) changed++;
    }
    changed = __reduce_add_sync(0xffffffffu, changed);
    if ((threadIdx.x & 31) == 0 && changed) atomicAdd(P.counts + ROUNDS, changed);
}

int allow_smem(lx_ctx *c)
{
    const uint64_t key = (2ull << 62) | (1ull << 40);
    for (auto &kv : c->occupancy)
        if (kv.first == key) return LX_OK;
    cudaError_t e = cudaFuncSetAttribute(cm_maps<FORM_BYTE>, cudaFuncAttributeMaxDynamicSharedMemorySize, 66 * 1024);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(cm_maps<FORM_CLASS>, cudaFuncAttributeMaxDynamicSharedMemorySize, 66 * 1024);
    if (e != cudaSuccess) return LX_E_CUDA;
    c->occupancy.emplace_back(key, 1);
    return LX_OK;
}

}  // namespace

bool contexts_path_ok(const lx_tokenset *ts, int mode)
{
    return ts->walk[mode].status == LX_OK && ts->scan.status == LX_OK;
}

int lex_contexts_device(lx_ctx *c, const lx_tokenset *ts, const uint8_t *d_in, uint64_t n, int mode, uint16_t *d_kinds,
                        uint32_t *d_lens, uint64_t capacity, uint64_t *n_tokens, uint64_t *consumed, cudaStream_t st,
                        lx_model *model, lx_spec_stats *spec)
{
    const WalkTable &w = ts->walk[mode];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != c->device) return LX_E_INVAL;
    DeviceTables dt;
    int rc = ensure_device_tables(ts, dev, &dt);
    if (rc == LX_OK) rc = allow_smem(c);
    if (rc != LX_OK) return rc;
    CParams P{};
    RParams &R = P.R;
    rows_table(ts, mode, dt, R);
    R.lo = (uint32_t)(reinterpret_cast<uintptr_t>(d_in) & 15u);
    R.in = d_in - R.lo;
    R.n = n + R.lo;
    R.slice = CL;
    R.n_slices = (R.n + CL - 1) / CL;
    const uint64_t tiles = (R.n + CT - 1) / CT;
    if (tiles > 0xFFFFFFF0ull) return LX_E_INVAL;
    P.n_tiles = (uint32_t)tiles;
    const uint8_t *scan = static_cast<const uint8_t *>(dt.d_scan);
    P.cbeg = reinterpret_cast<const uint16_t *>(scan + ts->scan.cbeg_off);
    P.cand = reinterpret_cast<const uint16_t *>(scan + ts->scan.cand_off);
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    const size_t S = R.n_slices, T = P.n_tiles;
    const size_t o_cnt = 64, o_rows = 256, o_starts = al(o_rows + 2 * S), o_pmap = al(o_starts + S);
    const size_t o_rf = al(o_pmap + 4 * S), o_tmap = al(o_rf + 2 * KMAX * S), o_tent = al(o_tmap + 4 * T);
    const size_t o_cs = al(o_tent + T), o_ci = al(o_cs + 8 * T), o_cur = al(o_ci + 4 * T), o_nxt = al(o_cur + T);
    const size_t o_guess = al(o_nxt + T), o_bmap = al(o_guess + 2 * T);
    const size_t total = al(o_bmap + 4 * ((T + TOP_NT - 1) / TOP_NT));
    rc = grow(&c->e_dev, &c->e_dev_bytes, total);
    if (rc == LX_E_NOMEM) return LX_ROWS;   // the chunks need a third of it
    if (rc != LX_OK) return rc;
    uint8_t *d = static_cast<uint8_t *>(c->e_dev);
    R.res = reinterpret_cast<RResult *>(d);
    P.counts = reinterpret_cast<unsigned int *>(d + o_cnt);
    R.rows = reinterpret_cast<uint16_t *>(d + o_rows);
    P.starts = d + o_starts;
    P.pmap = reinterpret_cast<uint32_t *>(d + o_pmap);
    P.rf = reinterpret_cast<uint16_t *>(d + o_rf);
    P.tmap = reinterpret_cast<uint32_t *>(d + o_tmap);
    P.tent = d + o_tent;
    P.bmap = reinterpret_cast<uint32_t *>(d + o_bmap);
    P.cstart = reinterpret_cast<uint64_t *>(d + o_cs);
    P.cinfo = reinterpret_cast<uint32_t *>(d + o_ci);
    P.cur = d + o_cur;
    P.nxt = d + o_nxt;
    rc = cuda_err(cudaMemsetAsync(d, 0, 256, st));
    if (rc != LX_OK) return rc;
    c->counts.contexts++;
    if (c->timing) cudaEventRecord(c->ev[0], st);
    const uint32_t wpb = CM_NT / 32, grid = (uint32_t)std::min<uint64_t>(4ull * c->num_sms, (tiles + wpb - 1) / wpb);
    const uint32_t smem = 512 + R.blob_bytes + 16;
    cm_starts<<<grid, CM_NT, 0, st>>>(P);
    // as many warps as make the last round of tiles a full one (a round's time is
    // its warps' share of the shared-memory pipe): 96 MiB are 4.04 rounds of 40
    // warps per SM, or 5 of 34, 597 -> 572 us a call.  The warps claim their tiles
    // (by turns they took 8 % longer: 542 us so).
    const uint32_t ctas = 2 * c->num_sms, rounds = (P.n_tiles + ctas * (MAP_NT / 32) - 1) / (ctas * (MAP_NT / 32));
    const uint32_t mwarps = (P.n_tiles + ctas * rounds - 1) / (ctas * rounds);
    const uint32_t mnt = 32 * std::max(mwarps, std::min(16u, (uint32_t)MAP_NT / 32));   // (sixteen stage the table)
    const uint32_t mgrid = std::min(ctas, (P.n_tiles + mnt / 32 - 1) / (mnt / 32));
    if (w.form == FORM_BYTE) cm_maps<FORM_BYTE><<<mgrid, mnt, smem, st>>>(P);
    else cm_maps<FORM_CLASS><<<mgrid, mnt, smem, st>>>(P);
    const uint32_t blocks = (P.n_tiles + TOP_NT - 1) / TOP_NT;
    cm_fold<<<blocks, TOP_NT, 0, st>>>(P);
    cm_top<<<blocks, TOP_NT, 0, st>>>(P);
    cm_rows<<<(uint32_t)std::min<uint64_t>(8ull * c->num_sms, (32 * tiles + CM_NT - 1) / CM_NT), CM_NT, 0, st>>>(P);
    unsigned int h[ROUNDS + 1] = {0};
    if (spec) {
        if (model) {
            uint16_t *guess = reinterpret_cast<uint16_t *>(d + o_guess);
            rc = model_predict(model, d_in, n, P.cstart, P.cinfo, scan, ts->scan.cbeg_off, ts->scan.cand_off, P.n_tiles,
                               guess, st);
            if (rc != LX_OK) return rc;
            P.guess = guess;
        }
        const uint32_t g2 = (uint32_t)std::min<uint64_t>(4ull * c->num_sms, (tiles + 255) / 256);
        cm_guess<<<g2, 256, 0, st>>>(P);
        for (uint32_t r = 0; r < (uint32_t)ROUNDS; r++) {
            cm_round<<<g2, 256, 0, st>>>(P, r);
            std::swap(P.cur, P.nxt);
        }
        std::swap(P.cur, P.nxt);
        cm_judge<<<g2, 256, 0, st>>>(P);
        rc = cuda_err(cudaMemcpyAsync(h, P.counts, sizeof h, cudaMemcpyDeviceToHost, st));
        if (rc != LX_OK) return rc;
    }
    rc = cuda_err(cudaGetLastError());
    if (rc != LX_OK) return rc;
    // (spec: a token that fails past its chunk ends the chunk's scan, which the maps do not show; the chunks count it)
    const RowsGiven given{R.rows, CL, &R.res->error, !spec};
    rc = lex_rows_device(c, ts, d_in, n, mode, d_kinds, d_lens, capacity, n_tokens, consumed, st, &given);
    if (spec && (rc == LX_OK || rc == LX_E_CAPACITY)) {
        // as the rounds of enumerate.cu count: a changed entry is scanned in
        // the next round, or after the judge
        uint32_t rescanned = 0, used = 0;
        for (int r = 0; r < ROUNDS; r++) {
            if (r + 1 < ROUNDS) rescanned += h[r];
            used += h[r] != 0;
        }
        spec->chunks = P.n_tiles;
        spec->rounds = 1 + used;
        spec->judged = h[ROUNDS - 1] != 0;
        spec->rescanned = rescanned + (spec->judged ? h[ROUNDS] : 0u);
    }
    return rc;
}

}  // namespace lx
