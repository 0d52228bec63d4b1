// rows.cu -- GB300 (sm_103a) lexing from known entry rows: the kernels that
// lx_lex takes first (lexwarp.cu and lex.cu hold the paths for what these
// refuse).
//
// The longest-match scanner of Section 3, as the event-code walk table of
// internal.h runs it, is in one row after every input byte.  If the row at
// the start of every slice of the input is known, all slices walk at once
// from there, each over its own bytes and no others.  Two kernels:
//
//   row_guess   the entry row of every slice.  After a synchronizing byte
//               every run over Q+ is in the same row (WalkTable::sync; the
//               certified bytes of the mode are among them), so a lane that
//               starts a few bytes before the slice in the PRE row, which
//               absorbs bytes up to the first synchronizing one, reaches the
//               slice in the scanner's row.  (Small inputs, and large ones
//               where 32 bytes nearly always suffice: lex_rows does it.)
//   lex_rows    every warp claims tiles of 32 slices; lane i walks slice i
//               from its entry row, stores the event codes in its part of
//               the warp's event buffer, counts them, and turns them into
//               (kind, length) pairs in a shared stage; the warp resolves
//               the tile's output offset (lookback.cuh) after its next
//               tile's walk and copies the stage out, coalesced.
//
// The entry rows need not be right: each lane checks that it leaves its slice
// in the next one's entry row (across tiles, when the offset is resolved).
// Where every slice agrees from START at offset 0 on, the rows are the serial
// scan's by induction.  A disagreement, an entry row that was not found or a
// backtrack to before a slice stops the call (ERR_ROWS) and the caller
// lexes the input another way; what was written is overwritten.  That costs up
// to a pass: C-like text with 40 lines of tokens that backtrack, alone among
// inputs that are taken, 2 MiB 80 us a call without the attempt, 140 with it, 64
// MiB 230 and 405 (250 when lexwarp.cu came first); one after the other
// (Refusals in runtime.h) they cost what they do without.
//
// Backtracking inside a slice (SLOW) is replayed by its lane (relex), and the
// first lexing failure ends the stream (Corollary 1); a token that fails in a
// later slice than its own, with no accepting prefix (WalkTable::noacc: an open
// string at the input's end), fails at the last event before.  Handing such
// inputs on took two passes: JSON cut inside a string 107 -> 32 us a call at
// 1.5 KB, 309 -> 135 at 64 MiB; what it adds to the others is a few bytes of
// spills: 512 MiB of JSON 519.3 -> 519.9 us, 512 documents 365.0 -> 367.0.
//
// Against the chunks of lexwarp.cu, which start at a certified byte and run
// on past their lane's bytes to the next one: no lane walks another's bytes
// (that tail was 16-26 % of the time), no halo, 16-byte event stores, and
// token-driven instead of byte-driven emission (instructions per input byte
// 1.02 -> 0.7).  A call: 512 MiB of JSON 1 003 -> 520 us, 192 MiB of C-like
// text 630 -> 334 us, 1 MiB of arith tokens 84 -> 30 us, 40 MiB not 16-byte
// aligned (formerly the tile kernel) 333 -> 79 us.  What bounds it: the
// load/store pipe, 66-80 % busy (1 460 wavefronts per 6 KiB tile of JSON: 614
// for the table lookups, 420 for the emission's code lookups and stage
// stores), with half the issue slots taken.

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cstdint>
#include <cstring>
#include <vector>

#include "rows.cuh"

namespace lx {
namespace {

// One input (of a batch: a document) as guess_row sees it.
struct GuessIn {
    const uint8_t *in;
    uint32_t lo, guess, n_pat, pat[4];
};

// Whether one of the few synchronizing byte values is among a block's bytes.
__device__ __forceinline__ bool has_sync(const GuessIn &P, const uint4 &c)
{
    uint32_t z = 0;
#pragma unroll
    for (uint32_t i = 0; i < 4; i++) {
        if (i >= P.n_pat) break;
        const uint32_t x = c.x ^ P.pat[i], y = c.y ^ P.pat[i], u = c.z ^ P.pat[i], v = c.w ^ P.pat[i];
        z |= ((x - 0x01010101u) & ~x) | ((y - 0x01010101u) & ~y) | ((u - 0x01010101u) & ~u) | ((v - 0x01010101u) & ~v);
    }
    return (z & 0x80808080u) != 0;
}

// The row at position p (a multiple of 16, 0 < p < n) by walking to it from
// the PRE row: from the block of the nearest synchronizing byte before it
// where few byte values synchronize (compared a word at a time, which takes
// no table lookups), else from `guess` bytes before, four times as many where
// none of them synchronizes; at most GUESS_MAX bytes back, and from START where
// the input begins there.  After SLOW (a token that backtracks) the next
// synchronizing byte is looked for; where none follows the row is lost, since
// a walk from farther back comes to the same place (looking there all the same
// took 1 ms of 64 MiB of C-like text with one line of them).  All lanes of a
// warp call it together.
template <int FORM>
__device__ uint32_t guess_row(const GuessIn &P, const REnv &E, uint64_t p, bool has)
{
    uint32_t e = E.pre, w = P.guess;
    bool hit = true;
    if (P.n_pat && has) {
        w = 0;
        hit = false;
        while (!hit && w < GUESS_MAX && w < p) {   // 64 bytes at a time
            uint4 c[4];
#pragma unroll
            for (uint32_t k = 0; k < 4; k++)
                c[k] = w + 16 * (k + 1) <= p ? ldg16(P.in + (p - w - 16 * (k + 1))) : make_uint4(0, 0, 0, 0);
            uint32_t back = 64;
#pragma unroll
            for (int k = 3; k >= 0; k--)
                if (w + 16 * (k + 1) <= p && has_sync(P, c[k])) {
                    back = 16 * (k + 1);
                    hit = true;
                }
            w += back;
        }
    }
    bool todo = has && (hit || w >= p), lost = false;   // (none in reach: nothing to walk from)
    while (__any_sync(0xffffffffu, todo)) {
        if (todo) {
            uint64_t a = p > w ? p - w : 0;
            e = E.pre;
            if (a == 0) {
                e = E.start;
                if (P.lo) {
                    for (uint32_t k = P.lo; k < 16; k++) e = wstep<FORM>(E, e, __ldg(P.in + k));
                    a = 16;
                }
            }
            for (; a < p; a += 16) {
                const uint4 c = ldg16(P.in + a);
                wword<FORM>(e, c.x, E.cmap);
                wword<FORM>(e, c.y, E.cmap);
                wword<FORM>(e, c.z, E.cmap);
                wword<FORM>(e, c.w, E.cmap);
                if (e == E.slow) e = E.pre, lost = true;
            }
            todo = e >= E.pre && w < GUESS_MAX && w < p && !lost;
        }
        w *= 4;
    }
    if (e >= E.pre || e == E.slow) return lost ? ROW_LOST : ROW_UNKNOWN;
    return (e & ~0xFFu) - E.tb;
}

__device__ __forceinline__ GuessIn guess_in(const RParams &P)
{
    return GuessIn{P.in, P.lo, P.guess, P.n_pat, {P.pat[0], P.pat[1], P.pat[2], P.pat[3]}};
}

// The tables of a batch's set, and its documents' synchronizing bytes.
__device__ __forceinline__ GuessIn use_set(const RParams &P, REnv &E, const WDoc &D)
{
    const uint32_t ws = E.tb + P.sets_off + D.set * (uint32_t)sizeof(WSet);
    E.start = E.tb + lds_u32(ws);
    E.pre = E.tb + lds_u32(ws + 4);
    E.slow = E.tb + lds_u32(ws + 8);
    E.kmap = E.tb + lds_u32(ws + 12);
    E.cmap = E.tb + lds_u32(ws + 16);
    return GuessIn{D.in, 0, P.guess, lds_u32(ws + 28), {lds_u32(ws + 32), lds_u32(ws + 36), lds_u32(ws + 40), lds_u32(ws + 44)}};
}

template <int FORM, bool BATCH>
__global__ void __launch_bounds__(GUESS_NT) row_guess(RParams P)
{
    extern __shared__ __align__(16) uint8_t smem[];
    // the scratch of lex_rows, which runs next on the stream
    uint4 *z = reinterpret_cast<uint4 *>(P.res);
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < P.zero_bytes / 16;
         i += (uint64_t)gridDim.x * blockDim.x)
        z[i] = make_uint4(0, 0, 0, 0);
    REnv E;
    if (!stage_table<FORM>(P, smem, E)) return;
    __syncthreads();
    GuessIn in = guess_in(P);
    for (uint64_t s0 = ((uint64_t)blockIdx.x * blockDim.x + threadIdx.x) & ~31ull; s0 < P.n_slices;
         s0 += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t s = s0 + (threadIdx.x & 31);
        uint64_t p = s * P.slice, n = P.n;   // the slice's position in its input
        if (BATCH) {   // a warp's 32 slices are one tile
            const uint32_t t = (uint32_t)(s0 / 32);
            const WDoc D = P.docs[__ldg(P.tile_doc + t)];
            in = use_set(P, E, D);
            p = (uint64_t)(t - D.first_tile) * 32 * P.slice + (uint64_t)(threadIdx.x & 31) * P.slice;
            n = D.n;
        }
        uint32_t r = guess_row<FORM>(in, E, p, p > 0 && p < n);
        if (p == 0) r = E.start - E.tb;
        if (p < n) P.rows[s] = (uint16_t)r;
    }
}

// The scratch of a lex_rows that finds its rows itself.
__global__ void rows_zero(RParams P)
{
    asm volatile("griddepcontrol.launch_dependents;");
    uint4 *z = reinterpret_cast<uint4 *>(P.res);
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < P.zero_bytes / 16;
         i += (uint64_t)gridDim.x * blockDim.x)
        z[i] = make_uint4(0, 0, 0, 0);
}

// The slice [ps, pe) of a lane token by token, from the last event that its
// walk stored (or from the entry row): the walk ran into SLOW, or the input
// ends at pe in a row that does not accept.  Codes go to ev + position - p0.
// Sets the exit row, the code that ends at pe == end of input (tail), a
// failure (twice its offset; twice ps + 1 where the token began before the
// slice and has no accepting prefix: an open string at the input's end, a
// control byte inside one), or `back` where the token in progress at ps does
// not accept in the slice but did before it (it has to be replayed from there).
template <int FORM>
__device__ __noinline__ void relex(const REnv &E, const uint8_t *noacc, const uint8_t *in, uint32_t ev, uint32_t p0,
                                   uint32_t ps, uint32_t pe, uint32_t e_in, bool at_end, uint32_t *exit, uint32_t *tail,
                                   uint32_t *fail, bool *back)
{
    uint32_t tok = ps, q = e_in, r = NONE, rc = 0, k;
    bool own = false;   // a token start lies in the slice
    for (uint32_t j = pe; j-- > ps;)
        if (lds_u8(ev + j - p0)) {
            tok = j;
            own = true;
            break;
        }
    if (own || q == E.start) {
        q = E.start;
        own = true;
    } else if ((rc = acc_code(E, q)) != 0) {
        r = ps;
    }
    k = tok;
    for (;;) {
        uint32_t v = E.slow;
        if (k < pe) {
            v = wstep<FORM>(E, q, __ldg(in + k));
        } else if (!at_end) {
            *exit = q & ~0xFFu;
            return;
        } else if (q != E.start) {
            const uint32_t ac = acc_code(E, q);
            if (ac) {
                *tail = ac;
                return;
            }
        } else {
            return;
        }
        if (v != E.slow) {
            const uint32_t code = v & 0xFEu;
            if (code) {   // the token ends before this byte
                sts_u8(ev + k - p0, code);
                tok = k;
                own = true;
                r = NONE;
            }
            q = v;
            k++;
            const uint32_t ac = acc_code(E, q);
            if (ac) {
                r = k;
                rc = ac;
            }
            continue;
        }
        if (r == NONE) {
            if (own) *fail = 2 * tok;
            else if (noacc && __ldg(noacc + ((e_in - E.tb) >> E.shift))) *fail = 2 * ps + 1;
            else *back = true;
            return;
        }
        sts_u8(ev + r - p0, rc);
        tok = k = r;
        own = true;
        q = E.start;
        r = NONE;
    }
}

// A failure of a token that began in an earlier tile (as a position in a tile).
constexpr uint32_t FAIL_BEFORE = NONE - 1;

// A tile whose tokens wait in the warp's stage for their output offset.
struct Pending {
    uint32_t tile;      // NONE: nothing pending
    uint32_t staged;    // kept tokens
    uint32_t split;     // of them in the shared stage (the rest: spill slot)
    uint32_t entry;     // entry row of its first lane
    uint32_t fail;      // failure position in the tile, or NONE, or FAIL_BEFORE
    uint32_t open;      // its first event ended a kept token that began in an earlier tile
    uint32_t lidx, llen;   // per lane: a token whose length the stage does not hold
    uint32_t doc, dtile, kmap;   // batches: its document, its index there, its set's kind map
};

// The staged tokens of a tile to the output from index G: each lane two
// consecutive tokens at a time from the first index where G + i is even, when
// the arrays are aligned for it and the capacity does not cut the tile.
__device__ __forceinline__ void copy_stage(const RParams &P, uint32_t kmap, uint32_t stage, const uint16_t *spill,
                                           uint32_t split, uint32_t staged, uint64_t G)
{
    const uint32_t lane = threadIdx.x & 31;
    auto val = [&](uint32_t i) { return i < split ? lds_u16(stage + 2 * i) : (uint32_t)spill[i - split]; };
    auto kind = [&](uint32_t v) { return lds_u16(kmap + ((v >> 8) & 0xFEu)); };
    auto one = [&](uint32_t i) {
        const uint64_t o = G + i;
        if (o < P.cap) {
            const uint32_t v = val(i);
            P.out_kinds[o] = (uint16_t)kind(v);
            P.out_lens[o] = v & 0x1FFu;
        }
    };
    const bool aligned = ((reinterpret_cast<uintptr_t>(P.out_kinds) & 3u) |
                          (reinterpret_cast<uintptr_t>(P.out_lens) & 7u)) == 0;
    if (!aligned || G + staged > P.cap) {
        for (uint32_t i = lane; i < staged; i += 32) one(i);
        return;
    }
    const uint32_t h = min((uint32_t)(G & 1u), staged);
    if (lane < h) one(lane);
    const uint32_t ng = (staged - h) / 2;
    uint16_t *const ok = P.out_kinds + G + h;
    uint32_t *const ol = P.out_lens + G + h;
    auto put = [&](uint32_t q, uint32_t v0, uint32_t v1, uint32_t k0, uint32_t k1) {
        *reinterpret_cast<uint32_t *>(ok + 2 * q) = k0 | (k1 << 16);
        *reinterpret_cast<uint2 *>(ol + 2 * q) = make_uint2(v0 & 0x1FFu, v1 & 0x1FFu);
    };
    uint32_t q = lane;
    if (split == staged)   // two pairs at a time: their stage and kind lookups overlap
        for (; q + 32 < ng; q += 64) {
            const uint32_t s0 = stage + 2 * h + 4 * q;
            const uint32_t v0 = lds_u16(s0), v1 = lds_u16(s0 + 2), v2 = lds_u16(s0 + 128), v3 = lds_u16(s0 + 130);
            const uint32_t k0 = kind(v0), k1 = kind(v1), k2 = kind(v2), k3 = kind(v3);
            put(q, v0, v1, k0, k1);
            put(q + 32, v2, v3, k2, k3);
        }
    for (; q < ng; q += 32) {
        const uint32_t i = h + 2 * q, v0 = val(i), v1 = val(i + 1);
        put(q, v0, v1, kind(v0), kind(v1));
    }
    const uint32_t t = h + 2 * ng;
    if (lane < staged - t) one(t + lane);
}

// Resolve the pending tile's output offset, check its entry row against the
// previous tile's exit row, and copy its tokens out.  False: stop (an error
// is flagged).
template <int NW, bool BATCH>
__device__ bool finish_tile(const RParams &P, const REnv &E, const Pending &D, uint32_t stage, const uint16_t *spill)
{
    const uint32_t lane = threadIdx.x & 31;
    constexpr uint32_t TILE = Geo<NW>::TILE;
    uint64_t G = 0, carry = 0;
    unsigned long long w;   // the previous tile's status word
    if (!resolve_tile(P, D.tile, G, w)) return false;
    const uint32_t dtile = BATCH ? D.dtile : D.tile;
    if (dtile) {
        const uint32_t x = (uint32_t)(w >> 32) & 0xFFFFu;
        if (x && x != D.entry) {
            if (lane == 0) atomicOr(P.error(), ERR_ROWS);
            return false;
        }
        if (D.open || D.fail == FAIL_BEFORE) {   // where that token began: the last event before the tile (every earlier tile has published)
            bool good = true;
            if (lane == 0) {
                Waiter W;
                uint32_t t = D.tile - 1;
                while (good && !((w >> 16) & 0xFFFFu) && t > D.tile - dtile) {
                    t--;
                    while ((w = ld_status(&P.status[t])) == 0 && (good = W.again(P))) {}
                }
                const uint32_t lp = (uint32_t)(w >> 16) & 0xFFFFu;
                carry = (uint64_t)(D.tile - t) * TILE - (lp ? lp - 1 : P.lo);
            }
            if (!__shfl_sync(0xffffffffu, good ? 1u : 0u, 0)) return false;
            carry = __shfl_sync(0xffffffffu, carry, 0);
        }
    }
    if (lane == 0) {
        unsigned long long *fp = BATCH ? &P.dres[D.doc].inv_fail_pos : &P.res->inv_fail_pos;
        unsigned long long *ft = BATCH ? &P.dres[D.doc].inv_fail_tok : &P.res->inv_fail_tok;
        if (D.fail != NONE) {
            const uint64_t f = (uint64_t)dtile * TILE;
            atomicMax(fp, ~(unsigned long long)(D.fail == FAIL_BEFORE ? f - carry : f + D.fail));
            atomicMax(ft, ~(unsigned long long)(G + D.staged));
        }
        if (BATCH) {
            if (dtile == 0) P.dres[D.doc].out_off1 = G + 1;
            if (D.staged) atomicAdd(&P.dres[D.doc].total, (unsigned long long)D.staged);
        }
        if (D.tile == P.n_tiles - 1) P.res->total = G + D.staged;
    }
    copy_stage(P, BATCH ? D.kmap : E.kmap, stage, spill, D.split, D.staged, G);
    __syncwarp();
    if (D.lidx != NONE && G + D.lidx < P.cap)
        P.out_lens[G + D.lidx] = (uint32_t)(D.llen + (D.open && D.lidx == 0 ? carry : 0));
    return true;
}

// The last CTA to finish hands the record over (a copy and a synchronization
// less per call than reading it back), and leaves a small launch's scratch
// zeroed (a memset less): 1 500 B of JSON 31.3 -> 24.7 us a call, 1 MiB of
// arith tokens 41 -> 36 us.
template <bool BATCH>
__device__ void finish_launch(const RParams &P)
{
    __threadfence();
    __syncthreads();   // (no static shared memory: the dynamic part takes all of it)
    if (!__syncthreads_or(threadIdx.x == 0 && atomicAdd(P.done, 1u) == gridDim.x - 1)) return;
    __threadfence();
    if (BATCH) {   // the record and, 64 bytes from it, the documents' records
        const uint32_t words = 8 + (uint32_t)(sizeof(WDocRes) / 8) * P.n_docs;
        const unsigned long long *src = reinterpret_cast<const unsigned long long *>(P.res);
        for (uint32_t i = threadIdx.x; i < words; i += blockDim.x)
            reinterpret_cast<volatile unsigned long long *>(P.down)[i] = __ldcg(src + i);
        __threadfence_system();
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence_system();
            reinterpret_cast<volatile unsigned long long *>(P.down)[words] = P.seq;
        }
        return;
    }
    if (threadIdx.x == 0) {
        RResult r;
        r.total = __ldcg(&P.res->total);
        r.inv_fail_pos = __ldcg(&P.res->inv_fail_pos);
        r.inv_fail_tok = __ldcg(&P.res->inv_fail_tok);
        r.error = __ldcg(&P.res->error);
        r.pad = 0;
        volatile unsigned long long *h = reinterpret_cast<volatile unsigned long long *>(&P.host->r);
        h[0] = r.total;
        h[1] = r.inv_fail_pos;
        h[2] = r.inv_fail_tok;
        h[3] = r.error;
    }
    __syncthreads();
    if (P.clean) {
        uint4 *z = reinterpret_cast<uint4 *>(P.res);
        for (uint32_t i = threadIdx.x; i < P.zero_bytes / 16; i += blockDim.x) z[i] = make_uint4(0, 0, 0, 0);
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        __threadfence_system();
        *reinterpret_cast<volatile uint32_t *>(&P.host->seq) = P.seq;
    }
}

template <int FORM, int NW, bool FIND, bool BATCH>
__global__ void __launch_bounds__(32 * MAX_WARPS, 1) lex_rows(RParams P)
{
    extern __shared__ __align__(16) uint8_t smem[];
    constexpr uint32_t SLICE = Geo<NW>::SLICE, TILE = Geo<NW>::TILE, STRIDE = Geo<NW>::STRIDE;
    const uint32_t STAGE = P.stage, WAREA = warp_area(NW, P.stage);
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    REnv E;
    bool go = stage_table<FORM>(P, smem, E);
    asm volatile("griddepcontrol.wait;" ::: "memory");   // the zeroed scratch and the rows of the kernel before
    if (!go && threadIdx.x == 0) atomicOr(P.error(), ERR_SMEM);   // (row_guess may have zeroed the first one)
    __syncthreads();
    const uint32_t area = ((E.tb + P.blob_bytes + 15u) & ~15u) + wid * WAREA;
    const uint32_t stage = area + 32 * STRIDE, evl = area + lane * STRIDE;
    uint16_t *const spill = P.spill + ((size_t)blockIdx.x * (blockDim.x >> 5) + wid) * (TILE + 1);
    const uint32_t ahead = gridDim.x * (blockDim.x / 32);
    const uint32_t lt = (1u << lane) - 1u;
    const uint32_t mbar = stage + 2 * STAGE;
    uint32_t phase = 0;
    if (lane == 0) mbar_init(mbar);
    fence_proxy_async();
    __syncwarp();
    if (P.before && *P.before != 0) {   // no rows to start from
        if (threadIdx.x == 0) atomicOr(P.error(), *P.before == ERR_FAR ? ERR_FAR : ERR_ROWS);
        go = false;
    }

    Pending pend;
    pend.tile = NONE;
    while (go) {
        uint32_t tile = 0;
        if (lane == 0) {
            tile = atomicAdd(P.tile_counter, 1u);
            if (*(volatile unsigned int *)P.error() != 0) tile = P.n_tiles;
        }
        tile = __shfl_sync(0xffffffffu, tile, 0);
        if (tile >= P.n_tiles) break;
        const uint8_t *in = P.in + (uint64_t)tile * TILE;
        uint64_t left = P.n - (uint64_t)tile * TILE;
        uint32_t doc = 0, dtile = tile;
        if (BATCH) {   // the tile's document and its set's tables
            doc = __ldg(P.tile_doc + tile);
            const WDoc D = P.docs[doc];
            dtile = tile - D.first_tile;
            in = D.in + (uint64_t)dtile * TILE;
            left = D.n - (uint64_t)dtile * TILE;
            use_set(P, E, D);
        }
        const uint32_t nrel = left < BIG ? (uint32_t)left : BIG;   // bytes from the tile's start on
        const uint32_t lo = BATCH || tile ? 0u : P.lo;
        if (!BATCH && lane == 0 && tile + ahead < P.n_tiles) {   // a tile some warp takes about one tile from now, into L2
            const uint64_t fb = (uint64_t)(tile + ahead) * TILE, fl = P.n - fb;
            const uint32_t bytes = (uint32_t)(fl < TILE ? fl : TILE) & ~15u;
            if (bytes)
                asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(P.in + fb), "r"(bytes) : "memory");
        }
        const uint32_t p0 = lane * SLICE;
        const bool has = p0 < nrel, whole = nrel >= TILE && lo == 0;
        if (whole) {   // every lane's slice into its place, while the entry row is read or found
            fence_proxy_async();   // (after the last tile's events were read there)
            if (lane == 0)
                asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(mbar), "r"(TILE) : "memory");
            __syncwarp();
            bulk_load(evl, in + p0, SLICE, mbar);
        }
        const uint64_t p = (uint64_t)tile * TILE + p0;
        const bool near = FIND && whole && !P.n_pat;   // rows from the slices' own bytes
        uint32_t er = 0, e;
        uint4 g0, g1;
        if (near) {
            if (lane == 0 && tile) {
                g0 = ldg16(in - 32);
                g1 = ldg16(in - 16);
            }
        } else if (FIND) {
            er = guess_row<FORM>(guess_in(P), E, p, has && p > 0);
            if (p == 0) er = P.p_start;
        } else if (has) {
            er = P.rows[((uint64_t)tile * 32 + lane) * P.row_step];
        }
        if (whole) {
            const bool there = mbar_wait(mbar, phase, P.timeout_ns);
            phase ^= 1u;
            if (!__all_sync(0xffffffffu, there)) {
                if (lane == 0) atomicOr(P.error(), ERR_TIMEOUT);
                mbar_wait(mbar, phase ^ 1u, P.timeout_ns);   // the copies must not land in a finished CTA
                break;
            }
        }
        if (near) {   // as guess_row, from the end of the lane before's slice
            if (lane) {
                g0 = lds16(evl - STRIDE + SLICE - 32);
                g1 = lds16(evl - STRIDE + SLICE - 16);
            }
            __syncwarp();   // (the walks below write over it)
            e = p > 32 ? E.pre : E.start;
            wword<FORM>(e, g0.x, E.cmap);
            wword<FORM>(e, g0.y, E.cmap);
            wword<FORM>(e, g0.z, E.cmap);
            wword<FORM>(e, g0.w, E.cmap);
            if (e == E.slow) e = E.pre;
            wword<FORM>(e, g1.x, E.cmap);
            wword<FORM>(e, g1.y, E.cmap);
            wword<FORM>(e, g1.z, E.cmap);
            wword<FORM>(e, g1.w, E.cmap);
            if (e == E.slow) e = E.pre;
            er = p ? (e & ~0xFFu) - E.tb : P.p_start;
            const bool open = p && e >= E.pre;
            if (__any_sync(0xffffffffu, open)) {   // no synchronizing byte there
                GuessIn I = guess_in(P);
                I.guess = 128;
                const uint32_t r = guess_row<FORM>(I, E, p, open);
                if (open) er = r;
            }
        }
        const bool act = has && er < ROW_DEAD;
        const uint32_t e_in = er + E.tb, ps = max(p0, lo), pe = min(p0 + SLICE, nrel);
        e = e_in;

        // walk the slice, its codes over its bytes.  (With 16-byte loads from
        // global memory instead, 32 lines a load, the input alone took a quarter
        // of the shared-memory and L1 pipe that bounds this kernel.)
        if (whole) {
            if (act) {
                uint4 A = lds16(evl);
#pragma unroll 2
                for (uint32_t b = 0; b < SLICE; b += 16) {
                    const uint4 c = A;
                    if (b + 16 < SLICE) A = lds16(evl + b + 16);
                    const uint32_t a0 = wword<FORM>(e, c.x, E.cmap), a1 = wword<FORM>(e, c.y, E.cmap);
                    const uint32_t a2 = wword<FORM>(e, c.z, E.cmap), a3 = wword<FORM>(e, c.w, E.cmap);
                    sts16(evl + b, a0, a1, a2, a3);
                }
            }
        } else if (act) {   // the input's first or last tile: partial blocks byte by byte
            for (uint32_t b = p0; b < pe; b += 16) {
                if (b >= lo && b + 16 <= nrel) {
                    const uint4 A = ldg16(in + b);
                    const uint32_t a0 = wword<FORM>(e, A.x, E.cmap), a1 = wword<FORM>(e, A.y, E.cmap);
                    const uint32_t a2 = wword<FORM>(e, A.z, E.cmap), a3 = wword<FORM>(e, A.w, E.cmap);
                    sts16(evl + b - p0, a0, a1, a2, a3);
                } else {
                    sts16(evl + b - p0, 0, 0, 0, 0);
                    for (uint32_t k = max(b, lo); k < min(b + 16, nrel); k++) {
                        e = wstep<FORM>(E, e, __ldg(in + k));
                        sts_u8(evl + k - p0, e & 0xFEu);
                    }
                }
            }
        }

        // the lane's end: backtracking, the end of the input, the exit row
        const bool at_end = act && pe == nrel;
        uint32_t tail = 0, fail = NONE, exit = e & ~0xFFu;   // without the event code
        bool back = has && er >= ROW_LOST;
        if (at_end && e != E.slow && e < E.pre) tail = acc_code(E, e);
        if (act && (e == E.slow || (at_end && !tail)))
            relex<FORM>(E, P.noacc_off ? P.blob + P.noacc_off : nullptr, in, evl, p0, ps, pe, e_in, at_end, &exit, &tail, &fail, &back);
        const uint32_t fmin2 = __reduce_min_sync(0xffffffffu, fail), fmin = fmin2 >> 1;   // (NONE: past every position)
        {
            const uint32_t ner = __shfl_down_sync(0xffffffffu, er, 1);
            bool bad = back;
            const bool far = has && er == ROW_UNKNOWN;
            if (lane < 31 && act && fail == NONE && !at_end && exit - E.tb != ner) bad = true;
            if (__any_sync(0xffffffffu, bad && p0 <= fmin)) {
                const unsigned err = __any_sync(0xffffffffu, far && p0 <= fmin) ? ERR_FAR : ERR_ROWS;
                if (lane == 0) atomicOr(P.error(), err);
                break;
            }
        }

        // (d) event masks (bit j: position 32 w + j of the slice) and the kept count
        uint32_t m[NW], cnt = 0;
        const uint32_t used = act && ps <= fmin ? pe - p0 : 0u;
#pragma unroll
        for (uint32_t w = 0; w < NW; w++) {
            m[w] = 0;
            if (32 * w < used) {
                const uint4 x = lds16(evl + 32 * w);
                uint4 y = make_uint4(0, 0, 0, 0);
                if (32 * w + 16 < used) y = lds16(evl + 32 * w + 16);
                const uint32_t s0 = __dp4a(event_mask(x.y), 0x80402010u, __dp4a(event_mask(x.x), 0x08040201u, 0u));
                const uint32_t s1 = __dp4a(event_mask(x.w), 0x80402010u, __dp4a(event_mask(x.z), 0x08040201u, 0u));
                const uint32_t s2 = __dp4a(event_mask(y.y), 0x80402010u, __dp4a(event_mask(y.x), 0x08040201u, 0u));
                const uint32_t s3 = __dp4a(event_mask(y.w), 0x80402010u, __dp4a(event_mask(y.z), 0x08040201u, 0u));
                m[w] = (s0 >> 7) | (s1 << 1) | (s2 << 9) | (s3 << 17);
                uint32_t c = __dp4a(kept_mask(x.x), 0x01010101u, __dp4a(kept_mask(x.y), 0x01010101u, 0u));
                c = __dp4a(kept_mask(x.z), 0x01010101u, __dp4a(kept_mask(x.w), 0x01010101u, c));
                c = __dp4a(kept_mask(y.x), 0x01010101u, __dp4a(kept_mask(y.y), 0x01010101u, c));
                c = __dp4a(kept_mask(y.z), 0x01010101u, __dp4a(kept_mask(y.w), 0x01010101u, c));
                cnt += c;
            }
        }
        cnt >>= 7;
        if (fmin2 != NONE) {   // nothing after the failure counts
            cnt = 0;
#pragma unroll
            for (uint32_t w = 0; w < NW; w++) {
                const uint32_t at = p0 + 32 * w;
                if (at > fmin) m[w] = 0;
                else if (fmin - at < 31) m[w] &= (2u << (fmin - at)) - 1u;
                for (uint32_t x = m[w]; x; x &= x - 1) cnt += lds_u8(evl + 32 * w + __ffs(x) - 1) >= 4 ? 1u : 0u;
            }
            if (pe > fmin) tail = 0;
        }
        cnt += tail >= 4 ? 1u : 0u;
        // the last event position of the lane (+ 1), and of the lanes before it
        uint32_t lp = 0;
#pragma unroll
        for (uint32_t w = 0; w < NW; w++)
            if (m[w]) lp = p0 + 32 * w + 32 - __clz(m[w]);
        if (tail) lp = pe + 1;
        const uint32_t evb = __ballot_sync(0xffffffffu, lp != 0);
        const uint32_t below = evb & lt;
        const uint32_t prev1 = __shfl_sync(0xffffffffu, lp, below ? 31 - __clz(below) : 0);
        const uint32_t last1 = __shfl_sync(0xffffffffu, lp, evb ? 31 - __clz(evb) : 0);
        uint32_t excl = cnt;
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, excl, o);
            if (lane >= (uint32_t)o) excl += y;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, excl, 31);
        excl -= cnt;
        const uint32_t xr = __shfl_sync(0xffffffffu, exit, 31);   // 0 where the input ended or failed
        const uint32_t x31 = __shfl_sync(0xffffffffu, (act && !at_end && fmin2 == NONE) ? 1u : 0u, 31) ? xr - E.tb : 0u;
        publish_word(P, tile, ((unsigned long long)x31 << 32) | ((unsigned long long)last1 << 16) | total);

        uint32_t pfail = fmin2 == NONE ? NONE : fmin;
        if (fmin2 != NONE && (fmin2 & 1u))   // a token that fails in a later slice than its own began at the last event before it
            pfail = last1 ? last1 - 1 : dtile == 0 ? lo : FAIL_BEFORE;

        // the previous tile's output: its predecessors have had a whole tile to publish
        if (pend.tile != NONE) {
            if (!finish_tile<NW, BATCH>(P, E, pend, stage, spill)) {
                pend.tile = NONE;
                break;
            }
            __syncwarp();
        }

        // (e) the kept events into the stage, in order
        pend.tile = tile;
        pend.staged = total;
        pend.fail = pfail;
        pend.entry = __shfl_sync(0xffffffffu, er, 0);
        pend.lidx = NONE;
        pend.llen = 0;
        if (BATCH) {
            pend.doc = doc;
            pend.dtile = dtile;
            pend.kmap = E.kmap;
        }
        bool open = false;
        uint32_t split = total;
        uint16_t *gp = nullptr;
        if (total > STAGE) {   // excl + cnt ascends with the lane: those that fit are a prefix
            const uint32_t fit = __popc(__ballot_sync(0xffffffffu, excl + cnt <= STAGE));
            split = fit == 32 ? total : __shfl_sync(0xffffffffu, excl, fit & 31u);
            if (lane >= fit) gp = spill + (excl - split);
        }
        pend.split = split;
        // the first event's token may begin in another lane or tile
        int prev = 0;   // the last event's position, relative to the slice
        if (lp) {
            uint32_t f = NONE;
#pragma unroll
            for (int w = NW - 1; w >= 0; w--)
                if (m[w]) f = 32 * w + __ffs(m[w]) - 1;
            const uint32_t fp = f == NONE ? pe - p0 : f;             // its position in the slice
            const uint32_t fc = f == NONE ? tail : lds_u8(evl + f);  // its code
            if (below) prev = (int)prev1 - 1 - (int)p0;
            else if (dtile == 0) prev = (int)lo - (int)p0;
            else prev = -(int)p0, open = true;
            const uint32_t d = (uint32_t)((int)fp - prev);
            if (open || d >= LEN_MAX) {
                if (fc >= 4) {
                    pend.lidx = excl;
                    pend.llen = d;
                } else {
                    open = false;
                }
                prev = (int)fp - (int)LEN_MAX;
            }
        }
        uint32_t sa = stage + 2 * excl;
        if (total <= STAGE) {
            // every lane its events in order, the warp as many steps per mask
            // word as its fullest lane has events, four at a time so that their
            // code lookups overlap
            uint32_t nmax[NW];
#pragma unroll
            for (uint32_t w = 0; w < NW; w++) nmax[w] = __reduce_max_sync(0xffffffffu, __popc(m[w]));
#pragma unroll
            for (uint32_t w = 0; w < NW; w++) {
                uint32_t x = m[w];
                for (int n = (int)nmax[w]; n > 0; n -= 4) {
                    uint32_t b[4], v[4], code[4];
#pragma unroll
                    for (int i = 0; i < 4; i++) {   // x's lowest one; 32 once the events have run out
                        v[i] = x;
                        b[i] = __popc((x - 1) & ~x);
                        x &= x - 1;
                    }
#pragma unroll
                    for (int i = 0; i < 4; i++) code[i] = event_code(evl + 32 * w + b[i], v[i]);
#pragma unroll
                    for (int i = 0; i < 4; i++) put_event(sa, prev, v[i], code[i], b[i] + 32 * w);
                }
            }
            if (tail >= 4) sts_u16(sa, (tail << 8) + (uint32_t)((int)(pe - p0) - prev));
        } else {
#pragma unroll
            for (uint32_t w = 0; w < NW; w++)
                for (uint32_t x = m[w]; x; x &= x - 1) {
                    const int pos = (int)(32 * w) + __ffs(x) - 1;
                    const uint32_t code = lds_u8(evl + pos), v = (code << 8) + (uint32_t)(pos - prev);
                    if (code >= 4) {
                        if (gp) *gp++ = (uint16_t)v;
                        else sts_u16(sa, v), sa += 2;
                    }
                    prev = pos;
                }
            if (tail >= 4) {
                const uint32_t v = (tail << 8) + (uint32_t)((int)(pe - p0) - prev);
                if (gp) *gp = (uint16_t)v;
                else sts_u16(sa, v);
            }
        }
        pend.open = __any_sync(0xffffffffu, open) ? 1u : 0u;
        __syncwarp();
    }
    if (pend.tile != NONE) finish_tile<NW, BATCH>(P, E, pend, stage, spill);
    finish_launch<BATCH>(P);
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
constexpr uint32_t SMEM_BUDGET = 227 * 1024;

struct RLaunch {
    RParams P;
    uint32_t grid = 0, nwarps = 0, smem = 0;
    uint32_t ggrid = 0, gsmem = 0;
    bool fused = false;   // its scratch is zero between launches
    bool find = false;    // lex_rows finds its entry rows itself
    int form = FORM_BYTE, nw = 1;
};

// Up to this many bytes lex_rows finds the entry rows itself: one launch less.
constexpr uint64_t FUSED_MAX = 4ull << 20;
// The part of a small launch's scratch that is zero between launches: status
// words for FUSED_MAX / 1 KiB + 1 tiles, group words, the record.
constexpr uint64_t SMALL_ZERO = 48 * 1024;
static_assert(64 + 8 * (FUSED_MAX / 1024 + 1) + 16 * (FUSED_MAX / 1024 / GS + 2) + 64 <= SMALL_ZERO, "small scratch");
// Where no word has to be searched for (n_pat = 0: the 32 bytes before a slice
// nearly always synchronize, and they are in shared memory as the end of the
// slice before), launches of three rounds of tiles and more find their rows
// themselves too, at slice lengths that such launches have.  512 MiB of JSON
// 546 -> 520 us, 256 MiB 306 -> 280, 64 MiB 109 -> 99; 256 MiB of arith tokens
// 641 -> 615: row_guess reads 128 bytes of memory for each 32 that it walks.
// In fewer rounds the rare lane that has to look 128 or 512 bytes back, one
// byte in 90 cycles beside 19 other warps, is a round's time by itself: 20 MiB
// of JSON 61 us with row_guess, 84 .. 93 without.
constexpr int FIND_NW_MIN = 5, FIND_NW_MAX = 7;
constexpr uint64_t FIND_ROUNDS = 3;
// A warp's time for a tile of 32 slices of 32 k bytes, in units of its fixed
// part, and the warps per SM past which more of them do not help (measured at
// 20 warps, 512 MiB of JSON: 669, 616, 581, 584 and 637 us for k = 4 to 8; 192
// MiB of C-like text: 380, 363, 342, 356, 360, and the same at 18); a launch
// takes its rounds of tiles and half a round more, the last one's share.
constexpr double TILE_FIXED = 1.0, TILE_STEP = 0.385;
constexpr uint32_t USEFUL_WARPS = 18;

using RowsKernel = void (*)(RParams);

// The kernel of a table form and geometry, and its per-warp shared bytes.
template <int FORM, bool BATCH>
RowsKernel rows_kernel(int nw, bool find)
{
    if constexpr (!BATCH)
        if (find) switch (nw) {
            case 1: return lex_rows<FORM, 1, true, false>;
            case 2: return lex_rows<FORM, 2, true, false>;
            case 5: return lex_rows<FORM, 5, true, false>;
            case 6: return lex_rows<FORM, 6, true, false>;
            default: return lex_rows<FORM, FIND_NW_MAX, true, false>;
            }
    switch (nw) {
    case 1: return lex_rows<FORM, 1, false, BATCH>;
    case 2: return lex_rows<FORM, 2, false, BATCH>;
    case 3: return lex_rows<FORM, 3, false, BATCH>;
    case 4: return lex_rows<FORM, 4, false, BATCH>;
    case 5: return lex_rows<FORM, 5, false, BATCH>;
    case 6: return lex_rows<FORM, 6, false, BATCH>;
    case 7: return lex_rows<FORM, 7, false, BATCH>;
    default: return lex_rows<FORM, 8, false, BATCH>;
    }
}
RowsKernel rows_kernel(int form, int nw, bool find, bool batch = false)
{
    if (batch) return rows_kernel<FORM_CLASS, true>(nw, false);
    return form == FORM_BYTE ? rows_kernel<FORM_BYTE, false>(nw, find) : rows_kernel<FORM_CLASS, false>(nw, find);
}

RowsKernel guess_kernel(int form, bool batch)
{
    if (batch) return row_guess<FORM_CLASS, true>;
    return form == FORM_BYTE ? row_guess<FORM_BYTE, false> : row_guess<FORM_CLASS, false>;
}

// Whether the kernels may use the shared memory they are launched with (once per context and kernel).
int allow_smem(lx_ctx *c, int form, int nw, bool find, bool batch = false)
{
    const uint64_t key = (2ull << 62) | ((uint64_t)batch << 9) | ((uint64_t)form << 8) | ((uint64_t)find << 7) | (uint64_t)nw;
    for (auto &kv : c->occupancy)
        if (kv.first == key) return LX_OK;
    cudaError_t e = cudaFuncSetAttribute(rows_kernel(form, nw, find, batch),
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BUDGET);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(guess_kernel(form, batch), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 batch ? SMEM_BUDGET : 66 * 1024);
    if (e != cudaSuccess) return LX_E_CUDA;
    c->occupancy.emplace_back(key, 1);
    return LX_OK;
}

// The slice length (32 nw bytes) for `tiles_of(nw)` tiles beside `fixed` bytes
// of tables, among 1 .. most and multiples of `step` bytes; 0: none fits.
template <class F>
int choose_nw(const lx_ctx *c, int mode, uint32_t fixed, int most, uint32_t step, F tiles_of)
{
    double best = 0;
    int nw = 0;
    for (int k = 1; k <= most; k++) {
        const uint32_t area = warp_area(k, stage_for(k, mode));
        if (fixed + area > SMEM_BUDGET) break;
        if (32 * k % step != 0) continue;
        const uint32_t warps = std::min<uint32_t>(USEFUL_WARPS, (SMEM_BUDGET - fixed) / area);
        const uint64_t all = (uint64_t)warps * c->num_sms;
        const double cost = ((double)tiles_of(k) / (double)all + 0.5) * (TILE_FIXED + TILE_STEP * k);
        if (!nw || cost < best) {
            best = cost;
            nw = k;
        }
    }
    return nw;
}

// Geometry of a launch over L.P.n bytes: the slice length, the warps per CTA
// and the grid (one CTA per SM).
int shape(lx_ctx *c, const lx_tokenset *ts, int mode, RLaunch &L, const RowsGiven *given)
{
    const WalkTable &w = ts->walk[mode];
    const uint32_t fixed = 512 + (uint32_t)w.blob.size() + 16;
    const uint64_t n = L.P.n;
    L.fused = !given && n <= FUSED_MAX;
    // a small launch takes one tile of 1 KiB per SM, or tiles of 2 KiB (1 MiB of
    // arith tokens 33 us in the former, 30 in the latter)
    const int nw = L.fused ? (n <= 1024ull * c->num_sms ? 1 : 2)
                           : choose_nw(c, mode, fixed, 8, given ? given->step : 1,
                                       [&](int k) { return (n + 1024 * k - 1) / (1024 * k); });
    if (L.fused && fixed + warp_area(nw, stage_for(nw, mode)) > SMEM_BUDGET) return LX_E_TOOBIG;
    if (!nw) return LX_E_TOOBIG;
    L.nw = nw;
    L.P.slice = 32 * nw;
    L.P.n_slices = (n + L.P.slice - 1) / L.P.slice;
    const uint64_t tiles = (n + 1024 * nw - 1) / (1024 * nw);
    if (tiles > 0xFFFFFFF0ull) return LX_E_INVAL;
    L.P.n_tiles = (uint32_t)tiles;
    L.P.stage = stage_for(nw, mode);
    const uint32_t area = warp_area(nw, L.P.stage);
    const uint32_t warps = std::min<uint32_t>(MAX_WARPS, (SMEM_BUDGET - fixed) / area);
    // few tiles: one CTA on every SM, no more warps than its share (sixteen stage the table)
    L.nwarps = (uint32_t)std::min<uint64_t>(warps, std::max<uint64_t>(16, (tiles + c->num_sms - 1) / c->num_sms));
    L.smem = fixed + L.nwarps * area;
    L.grid = (uint32_t)std::min<uint64_t>((uint64_t)c->num_sms, tiles);
    L.gsmem = fixed;
    L.find = L.fused || (!given && !L.P.n_pat && nw >= FIND_NW_MIN && nw <= FIND_NW_MAX &&
                         tiles >= FIND_ROUNDS * L.grid * L.nwarps);
    return allow_smem(c, w.form, nw, L.find);
}

void launch(const RLaunch &L, const RowsGiven *given, cudaStream_t st)
{
    if (!L.find && !given) guess_kernel(L.form, false)<<<L.ggrid, GUESS_NT, L.gsmem, st>>>(L.P);
    else if (L.find && !L.fused) rows_zero<<<32, 256, 0, st>>>(L.P);
    if (L.fused || given) {
        rows_kernel(L.form, L.nw, L.find)<<<L.grid, 32 * L.nwarps, L.smem, st>>>(L.P);
        return;
    }
    // lex_rows may start, and stage its table, while the last CTAs of row_guess
    // run (24 MiB of JSON 87 -> 79 us a call)
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(L.grid);
    cfg.blockDim = dim3(32 * L.nwarps);
    cfg.dynamicSmemBytes = L.smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1] = {};
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, rows_kernel(L.form, L.nw, L.find), L.P);
}

// The last CTA of a launch has written its record to pinned memory: a launch
// that takes long (or failed) is waited for by the runtime, at `ev` if given.
template <class F>
int wait_record(cudaStream_t st, cudaEvent_t ev, F there)
{
    const auto t0 = std::chrono::steady_clock::now();
    bool ok = there();
    for (uint32_t i = 1; !ok; i++, ok = there())
        if (i % 1024 == 0 && std::chrono::steady_clock::now() - t0 > std::chrono::milliseconds(2)) break;
    if (!ok) {
        const int rc = cuda_err(ev ? cudaEventSynchronize(ev) : cudaStreamSynchronize(st));
        if (rc != LX_OK) return rc;
        if (!there()) return LX_E_CUDA;
    }
    std::atomic_thread_fence(std::memory_order_acquire);
    return LX_OK;
}

}  // namespace

bool rows_path_ok(const lx_tokenset *ts, int mode)
{
    return ts->walk[mode].status == LX_OK && ts->walk[mode].n_sync > 0;
}

void rows_table(const lx_tokenset *ts, int mode, const DeviceTables &dt, RParams &P)
{
    const WalkTable &w = ts->walk[mode];
    P.blob = static_cast<const uint8_t *>(dt.d_walk[mode]);
    P.blob_bytes = (uint32_t)w.blob.size();
    P.rows_bytes = w.rows_bytes;
    P.row_shift = w.row_shift;
    P.sync_bytes = 2 * (uint32_t)w.sync.size();
    P.p_start = w.p_start;
    P.p_pre = w.p_pre;
    P.acc_off = w.acc_off;
    P.kmap_off = w.kmap_off;
    P.cmap_off = w.cmap_off;
    P.noacc_off = P.blob_bytes + P.sync_bytes;
}

namespace {

// One input's launch: its parameters and shape, with the scratch grown for it.
int rows_prepare(lx_ctx *c, const lx_tokenset *ts, const uint8_t *d_in, uint64_t n, int mode, uint16_t *d_kinds,
                 uint32_t *d_lens, uint64_t capacity, const RowsGiven *given, RLaunch &L)
{
    const WalkTable &w = ts->walk[mode];
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev != c->device) return LX_E_INVAL;
    DeviceTables dt;
    int rc = ensure_device_tables(ts, dev, &dt);
    if (rc != LX_OK) return rc;
    RParams &P = L.P;
    P = RParams{};
    P.lo = (uint32_t)(reinterpret_cast<uintptr_t>(d_in) & 15u);
    P.in = d_in - P.lo;
    P.n = n + P.lo;
    L.form = w.form;
    P.guess = 32;
    if (w.n_sync <= 4)   // few byte values synchronize: they are searched for
        for (uint32_t b = 0; b < 256; b++)
            if (w.sync[w.form == FORM_BYTE ? b : ts->byte_class[b]] != w.p_pre) P.pat[P.n_pat++] = b * 0x01010101u;
    rc = shape(c, ts, mode, L, given);
    if (rc == LX_E_TOOBIG) return LX_ROWS;
    if (rc != LX_OK) return rc;
    rows_table(ts, mode, dt, P);
    if (given && !given->open) P.noacc_off = 0;
    P.out_kinds = d_kinds;
    P.out_lens = d_lens;
    P.cap = capacity;
    P.timeout_ns = c->timeout_ns;
    P.withhold = c->withhold;
    // scratch: record and counters, status words, group words (zeroed), entry
    // rows, spill slots
    auto al = [](uint64_t x) { return (x + 255) & ~(uint64_t)255; };
    const uint64_t groups = (P.n_tiles + GS - 1) / GS;
    const uint64_t o_g = 64 + 8ull * P.n_tiles, o_i = o_g + 8 * groups, zero = (o_i + 8 * groups + 15) & ~15ull;
    const uint64_t o_rows = L.fused ? SMALL_ZERO : al(zero), o_spill = al(o_rows + (L.find || given ? 0 : 2 * P.n_slices));
    const uint64_t need = o_spill + 2ull * (32 * P.slice + 1) * L.grid * L.nwarps;
    void **buf = L.fused ? &c->small : &c->scratch;
    size_t *have = L.fused ? &c->small_bytes : &c->scratch_bytes;
    if (L.fused && *have < need) c->small_clean = false;
    rc = grow(buf, have, need);
    if (rc == LX_E_NOMEM) return LX_ROWS;   // (what comes next may need less)
    if (rc != LX_OK) return rc;
    uint8_t *scr = static_cast<uint8_t *>(*buf);
    P.res = reinterpret_cast<RResult *>(scr);
    P.tile_counter = reinterpret_cast<unsigned int *>(scr + sizeof(RResult));
    P.done = P.tile_counter + 1;
    P.status = reinterpret_cast<unsigned long long *>(scr + 64);
    P.gagg = reinterpret_cast<unsigned long long *>(scr + o_g);
    P.ginc = reinterpret_cast<unsigned long long *>(scr + o_i);
    P.zero_bytes = zero;
    P.rows = given ? given->rows : reinterpret_cast<uint16_t *>(scr + o_rows);
    P.row_step = given ? P.slice / given->step : 1;
    P.before = given ? given->error : nullptr;
    P.spill = reinterpret_cast<uint16_t *>(scr + o_spill);
    P.clean = L.fused;
    L.ggrid = (uint32_t)std::min<uint64_t>(4ull * c->num_sms, (P.n_slices + GUESS_NT - 1) / GUESS_NT);
    return LX_OK;
}

// Queue it on st; its record goes to `rec` (pinned).
int rows_queue(lx_ctx *c, RLaunch &L, const RowsGiven *given, HostRecord *rec, cudaStream_t st)
{
    RParams &P = L.P;
    P.host = rec;
    P.seq = ++c->seq ? c->seq : ++c->seq;
    // a small launch finds its scratch zeroed by the one before
    if (given || (L.fused && !c->small_clean)) {
        const int rc = cuda_err(cudaMemsetAsync(P.res, 0, L.fused ? SMALL_ZERO : P.zero_bytes, st));
        if (rc != LX_OK) return rc;
    }
    static_cast<volatile HostRecord *>(rec)->seq = 0;
    std::atomic_thread_fence(std::memory_order_seq_cst);
    if (L.fused) c->small_clean = false;   // until this launch has finished without an error
    launch(L, given, st);
    return cuda_err(cudaGetLastError());
}

// Wait for its record: the tokens, con(w) and whether it failed.  `ev`: an event
// behind it, where more work is queued on st.
int rows_collect(lx_ctx *c, const RLaunch &L, cudaStream_t st, cudaEvent_t ev, uint64_t *tokens, uint64_t *consumed,
                 bool *failed)
{
    const volatile HostRecord *hr = L.P.host;
    const int rc = wait_record(st, ev, [&] { return hr->seq == L.P.seq; });
    if (rc != LX_OK) return rc;
    const RResult r = L.P.host->r;
    if (L.fused && r.error == 0) c->small_clean = true;
    if (r.error == ERR_TIMEOUT) return LX_E_TIMEOUT;
    if ((r.error & ~ERR_TIMEOUT) == ERR_FAR) return LX_FAR;   // (waits end early once an error is flagged)
    if (r.error) return LX_ROWS;
    *failed = r.inv_fail_pos != 0;
    *tokens = *failed ? ~r.inv_fail_tok : r.total;
    *consumed = (*failed ? ~r.inv_fail_pos : L.P.n) - L.P.lo;
    return LX_OK;
}

}  // namespace

int lex_rows_device(lx_ctx *c, const lx_tokenset *ts, const uint8_t *d_in, uint64_t n, int mode, uint16_t *d_kinds,
                    uint32_t *d_lens, uint64_t capacity, uint64_t *n_tokens, uint64_t *consumed, cudaStream_t st,
                    const RowsGiven *given)
{
    static_assert(sizeof(RResult) == 32 && sizeof(HostRecord) <= LAUNCH_RECORD_BYTES, "record layout");
    if (n == 0) {
        *n_tokens = 0;
        *consumed = 0;
        return LX_OK;
    }
    RLaunch L;
    int rc = rows_prepare(c, ts, d_in, n, mode, d_kinds, d_lens, capacity, given, L);
    if (rc != LX_OK) return rc;
    if (!given) c->counts.rows++;
    if (c->timing && !given) cudaEventRecord(c->ev[0], st);
    rc = rows_queue(c, L, given, static_cast<HostRecord *>(c->h_res), st);
    if (c->timing) cudaEventRecord(c->ev[1], st);
    uint64_t tokens = 0, con = 0;
    bool failed = false;
    if (rc == LX_OK) rc = rows_collect(c, L, st, nullptr, &tokens, &con, &failed);
    if (rc != LX_OK) return rc;
    *n_tokens = tokens;
    *consumed = con;
    return tokens > capacity ? LX_E_CAPACITY : LX_OK;
}

// Bound by the two copies (84 MB in and 75 out for 80 MiB of JSON: 533 us when
// they overlap).  Pieces of 12 MiB, at most eight (lex.cu: ROWS_PIECE): the
// launches of a piece take a few microseconds of host time, the copy in of the
// first and the copy out of the last overlap nothing.  JSON, kinds 2, against
// the single-pass kernel in pieces of 32 MiB: 1.5 KB 60 -> 33 us, 1 MiB
// 83 -> 53, 24 MiB 361 -> 277, 48 MiB 632 -> 497, 80 MiB 832 -> 756..790 (with
// pieces of 8 MiB 814, of 16 MiB 783; tapered at both ends 790).
int lex_rows_host(lx_ctx *c, const lx_tokenset *ts, const uint8_t *h_in, uint64_t n, int mode, uint16_t *h_kinds,
                  uint32_t *h_lens, uint64_t capacity, const uint64_t *b, uint32_t K, uint64_t *n_tokens,
                  uint64_t *consumed, cudaStream_t st)
{
    auto al = [](uint64_t x, uint64_t a) { return (x + a - 1) / a * a; };
    // device layout: piece i's bytes at a 16-byte aligned offset; its tokens
    // (at most one per byte) in its own output range, 4-token aligned
    std::vector<uint64_t> in_off(K), out_off(K), cap(K);
    uint64_t in_total = 0, out_total = 0;
    for (uint32_t i = 0; i < K; i++) {
        const uint64_t len = b[i + 1] - b[i];
        in_off[i] = in_total;
        in_total = al(in_total + len, 16);
        cap[i] = al(len + 1, 4);
        out_off[i] = out_total;
        out_total += cap[i];
    }
    int rc = grow(&c->d_in, &c->d_in_bytes, in_total + 16);
    if (rc == LX_OK) rc = grow(&c->d_out, &c->d_out_bytes, 6 * out_total + 64);
    if (rc == LX_OK) rc = grow_host(&c->h_scratch, &c->h_scratch_bytes, sizeof(HostRecord) * (size_t)K);
    if (rc != LX_OK) return rc;
    uint8_t *d_in = static_cast<uint8_t *>(c->d_in);
    uint32_t *d_lens = static_cast<uint32_t *>(c->d_out);
    uint16_t *d_kinds = reinterpret_cast<uint16_t *>(d_lens + out_total);
    HostRecord *rec = static_cast<HostRecord *>(c->h_scratch);
    // every piece's parameters twice: the scratch has grown for all of them
    // before the first launch is queued
    std::vector<RLaunch> L(K);
    for (int pass = 0; pass < 2 && rc == LX_OK; pass++)
        for (uint32_t i = 0; i < K && rc == LX_OK; i++)
            rc = rows_prepare(c, ts, d_in + in_off[i], b[i + 1] - b[i], mode, d_kinds + out_off[i], d_lens + out_off[i],
                              cap[i], nullptr, L[i]);
    if (rc != LX_OK) return rc;
    // one piece: all on the caller's stream
    cudaStream_t si = K > 1 ? c->s_in : st, so = K > 1 ? c->s_out : st;
    for (uint32_t i = 0; i < K && rc == LX_OK; i++) {
        rc = cuda_err(cudaMemcpyAsync(d_in + in_off[i], h_in + b[i], b[i + 1] - b[i], cudaMemcpyHostToDevice, si));
        if (rc == LX_OK && K > 1) rc = cuda_err(cudaEventRecord(c->ev_in[i], si));
    }
    // the launches, in order on the caller's stream (one scratch, reused)
    c->counts.rows++;
    if (c->timing) cudaEventRecord(c->ev[0], st);
    for (uint32_t i = 0; i < K && rc == LX_OK; i++) {
        if (K > 1) rc = cuda_err(cudaStreamWaitEvent(st, c->ev_in[i], 0));
        if (rc == LX_OK) rc = rows_queue(c, L[i], nullptr, rec + i, st);
        if (rc == LX_OK && K > 1) rc = cuda_err(cudaEventRecord(c->ev_lex[i], st));
    }
    if (c->timing) cudaEventRecord(c->ev[1], st);
    // each piece's tokens out as soon as it is lexed, after the previous pieces'
    uint64_t out = 0, con = n;
    bool failed = false;
    for (uint32_t i = 0; i < K && !failed && rc == LX_OK; i++) {
        uint64_t m = 0, pc = 0;
        rc = rows_collect(c, L[i], st, K > 1 ? c->ev_lex[i] : nullptr, &m, &pc, &failed);
        if (rc != LX_OK) break;
        if (failed) con = b[i] + pc;   // Corollary 1: the first failing piece ends the stream
        const uint64_t lo = std::min(out, capacity), hi = std::min(out + m, capacity);
        if (hi > lo) {
            rc = cuda_err(cudaMemcpyAsync(h_lens + lo, d_lens + out_off[i], (hi - lo) * 4, cudaMemcpyDeviceToHost, so));
            if (rc == LX_OK)
                rc = cuda_err(cudaMemcpyAsync(h_kinds + lo, d_kinds + out_off[i], (hi - lo) * 2, cudaMemcpyDeviceToHost, so));
        }
        out += m;
    }
    int r2 = cuda_err(cudaStreamSynchronize(so));
    if (rc == LX_OK) rc = r2;
    if (K > 1) {
        r2 = cuda_err(cudaStreamSynchronize(st));
        if (rc == LX_OK) rc = r2;
        r2 = cuda_err(cudaStreamSynchronize(si));
        if (rc == LX_OK) rc = r2;
    }
    if (rc != LX_OK) return rc;
    *n_tokens = out;
    *consumed = con;
    return out > capacity ? LX_E_CAPACITY : LX_OK;
}

// ---------------------------------------------------------------------------
// batches: every document of every token set in one graph launch
// ---------------------------------------------------------------------------
namespace {

// One warp per document takes its descriptor from pinned memory and writes the
// document's index over its tiles.
__global__ void br_tile_docs(const WDoc *docs, uint32_t n_docs, uint32_t tile, WDoc *dev, uint32_t *tile_doc)
{
    const uint32_t lane = threadIdx.x & 31u, nw = gridDim.x * (blockDim.x / 32u);
    for (uint32_t d = (blockIdx.x * blockDim.x + threadIdx.x) / 32u; d < n_docs; d += nw) {
        const WDoc D = docs[d];
        if (lane == 0) dev[d] = D;
        const uint32_t nt = (uint32_t)((D.n + tile - 1) / tile);
        for (uint32_t k = lane; k < nt; k += 32) tile_doc[D.first_tile + k] = d;
    }
}

}  // namespace

int lex_batch_rows(lx_ctx *c, const std::vector<uint64_t> &sets_key, const lx_doc *docs, uint32_t n_docs, int mode,
                   uint16_t *d_kinds, uint32_t *d_lens, uint64_t capacity, lx_doc_result *results, uint64_t *n_total,
                   cudaStream_t st)
{
    const uint32_t fixed = 512 + c->wb_blob_bytes + 16;
    uint64_t bytes = 0;
    uint32_t D = 0;
    for (uint32_t i = 0; i < n_docs; i++)
        if (docs[i].n) {
            bytes += docs[i].n;
            D++;
        }
    if (!D) return LX_OK;
    // half a tile of every document is empty on average
    const int nw = choose_nw(c, mode, fixed, 8, 1, [&](int k) { return bytes / (1024 * k) + (D + 1) / 2; });
    if (!nw) return LX_ROWS;
    const uint32_t tile = 1024 * nw;
    std::vector<WDoc> hd;
    std::vector<uint32_t> idx;
    hd.reserve(D);
    idx.reserve(D);
    uint64_t TT = 0;
    for (uint32_t i = 0; i < n_docs; i++) {
        if (!docs[i].n) continue;
        hd.push_back(WDoc{docs[i].data, docs[i].n, (uint32_t)TT, docs[i].set});
        idx.push_back(i);
        TT += (docs[i].n + tile - 1) / tile;
        if (TT > 0xFFFFFFF0ull) return LX_E_INVAL;
    }
    const uint32_t area = warp_area(nw, stage_for(nw, mode));
    const uint32_t warps = std::min<uint32_t>(MAX_WARPS, (SMEM_BUDGET - fixed) / area);
    const uint32_t n_tiles = (uint32_t)TT;
    const uint32_t nwarps = (uint32_t)std::min<uint64_t>(warps, std::max<uint64_t>(16, (TT + c->num_sms - 1) / c->num_sms));
    const uint32_t smem = fixed + nwarps * area, grid = (uint32_t)std::min<uint64_t>((uint64_t)c->num_sms, TT);
    int rc = allow_smem(c, FORM_CLASS, nw, false, true);
    if (rc != LX_OK) return rc;

    // device scratch: [record, document records, statuses, group words: zeroed][documents][tile map][rows][spill]
    auto al = [](size_t x, size_t a) { return (x + a - 1) / a * a; };
    const size_t groups = (n_tiles + GS - 1) / GS;
    const size_t o_dres = 64, down = o_dres + sizeof(WDocRes) * D, o_status = al(down, 64);
    const size_t o_gagg = o_status + 8 * (size_t)n_tiles, o_ginc = o_gagg + 8 * groups, zero_end = al(o_ginc + 8 * groups, 16);
    const size_t o_docs = al(zero_end, 256), o_tdoc = al(o_docs + sizeof(WDoc) * D, 256);
    const size_t o_rows = al(o_tdoc + 4 * (size_t)n_tiles, 256), o_spill = al(o_rows + 64 * (size_t)n_tiles, 256);
    const size_t dev_total = o_spill + 2 * (size_t)(tile + 1) * grid * nwarps;
    const size_t h_down = al(sizeof(WDoc) * D, 64), host_total = h_down + down + 8;
    void *od = c->b_dev, *oh = c->b_host;
    rc = grow(&c->b_dev, &c->b_dev_bytes, dev_total);
    if (rc == LX_OK) rc = grow_host(&c->b_host, &c->b_host_bytes, host_total);
    if (rc == LX_E_NOMEM) return LX_ROWS;
    if (rc != LX_OK) return rc;
    const bool moved = od != c->b_dev || oh != c->b_host;
    uint8_t *dv = static_cast<uint8_t *>(c->b_dev), *hs = static_cast<uint8_t *>(c->b_host);
    std::memcpy(hs, hd.data(), sizeof(WDoc) * D);

    std::vector<uint64_t> gkey = {0xB47C6ull, D, TT, (uint64_t)mode, (uint64_t)(uintptr_t)d_kinds,
                                  (uint64_t)(uintptr_t)d_lens, capacity, (uint64_t)(uintptr_t)dv,
                                  (uint64_t)(uintptr_t)hs, c->timeout_ns, grid, nwarps, (uint64_t)nw,
                                  (uint64_t)(uintptr_t)c->wb_dev};
    gkey.insert(gkey.end(), sets_key.begin(), sets_key.end());
    if (moved || gkey != c->r_key || !c->r_exec) {
        if (c->r_exec) cudaGraphExecDestroy(c->r_exec);
        c->r_exec = nullptr;
        c->r_key.clear();
        if (!c->b_stream && cudaStreamCreateWithFlags(&c->b_stream, cudaStreamNonBlocking) != cudaSuccess)
            return LX_E_CUDA;
        cudaStream_t cs = c->b_stream;
        RParams P{};
        P.blob = static_cast<const uint8_t *>(c->wb_dev) + c->wb_blob_bytes;
        P.blob_bytes = c->wb_blob_bytes;
        P.rows_bytes = c->wb_rows;
        P.row_shift = 8;
        P.acc_off = c->wb_acc_off;
        P.noacc_off = c->wb_blob_bytes;
        P.sets_off = c->wb_sets_off;
        P.guess = 32;
        P.slice = 32 * nw;
        P.stage = stage_for(nw, mode);
        P.n_slices = 32ull * n_tiles;
        P.row_step = 1;
        P.out_kinds = d_kinds;
        P.out_lens = d_lens;
        P.cap = capacity;
        P.res = reinterpret_cast<RResult *>(dv);
        P.tile_counter = reinterpret_cast<unsigned int *>(dv + sizeof(RResult));
        P.done = P.tile_counter + 1;
        P.down = reinterpret_cast<unsigned long long *>(hs + h_down);
        P.n_docs = D;
        P.seq = 1;
        P.dres = reinterpret_cast<WDocRes *>(dv + o_dres);
        P.status = reinterpret_cast<unsigned long long *>(dv + o_status);
        P.gagg = reinterpret_cast<unsigned long long *>(dv + o_gagg);
        P.ginc = reinterpret_cast<unsigned long long *>(dv + o_ginc);
        P.zero_bytes = zero_end;
        P.docs = reinterpret_cast<const WDoc *>(dv + o_docs);
        P.tile_doc = reinterpret_cast<const uint32_t *>(dv + o_tdoc);
        P.rows = reinterpret_cast<uint16_t *>(dv + o_rows);
        P.spill = reinterpret_cast<uint16_t *>(dv + o_spill);
        P.n_tiles = n_tiles;
        P.timeout_ns = c->timeout_ns;
        P.withhold = NONE;
        const uint32_t gmax = SMEM_BUDGET / (fixed + 1024) * c->num_sms;   // guess CTAs resident at once, at most four per SM
        const uint32_t gg = std::min(std::min(gmax, 4u * (uint32_t)c->num_sms), (32u * n_tiles + GUESS_NT - 1) / GUESS_NT);
        if (cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return LX_E_CUDA;
        br_tile_docs<<<(D + 7) / 8, 256, 0, cs>>>(reinterpret_cast<const WDoc *>(hs), D, tile,
                                                 const_cast<WDoc *>(P.docs), const_cast<uint32_t *>(P.tile_doc));
        guess_kernel(FORM_CLASS, true)<<<std::max(1u, gg), GUESS_NT, fixed, cs>>>(P);
        rows_kernel(FORM_CLASS, nw, false, true)<<<grid, 32 * nwarps, smem, cs>>>(P);
        cudaGraph_t graph = nullptr;
        cudaError_t e = cudaStreamEndCapture(cs, &graph);
        if (e == cudaSuccess) e = cudaGraphInstantiate(&c->r_exec, graph, 0);
        if (graph) cudaGraphDestroy(graph);
        if (e != cudaSuccess) {
            c->r_exec = nullptr;
            cudaGetLastError();
            return LX_E_CUDA;
        }
        c->r_key = gkey;
        c->counts.graphs++;
    }
    c->counts.rows++;
    volatile unsigned long long *seq = reinterpret_cast<volatile unsigned long long *>(hs + h_down + down);
    *seq = 0;
    std::atomic_thread_fence(std::memory_order_seq_cst);
    if (c->timing) cudaEventRecord(c->ev[0], st);
    rc = cuda_err(cudaGraphLaunch(c->r_exec, st));
    if (c->timing) cudaEventRecord(c->ev[1], st);
    if (rc == LX_OK) rc = wait_record(st, nullptr, [&] { return *seq == 1; });
    if (rc != LX_OK) return rc;

    const RResult r = *reinterpret_cast<const RResult *>(hs + h_down);
    if (r.error == ERR_TIMEOUT) return LX_E_TIMEOUT;
    if (r.error) return LX_ROWS;
    const WDocRes *dres = reinterpret_cast<const WDocRes *>(hs + h_down + o_dres);
    for (uint32_t j = 0; j < D; j++) {
        const WDocRes &x = dres[j];
        lx_doc_result &o = results[idx[j]];
        if (x.out_off1 == 0) return LX_E_CUDA;   // every document's first tile reports its offset
        o.out_off = x.out_off1 - 1;
        if (x.inv_fail_pos) {
            o.consumed = ~x.inv_fail_pos;
            o.n_tokens = ~x.inv_fail_tok - o.out_off;
        } else {
            o.consumed = hd[j].n;
            o.n_tokens = x.total;
        }
    }
    *n_total = r.total;
    return r.total > capacity ? LX_E_CAPACITY : LX_OK;
}

}  // namespace lx
