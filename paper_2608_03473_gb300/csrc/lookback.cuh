// lookback.cuh -- the two-level decoupled look-back of the warp-owned tile
// kernels (lexwarp.cu, rows.cu).
// Tiles form groups of GS.  A tile publishes its kept count (ST_AGG) in its
// status word and adds it, with one in the top bits, to its group's word:
// a store and a reduction that nothing waits for (the earlier form, an
// acquire-release counter whose last arrival summed the group, held every
// warp about 3 900 cycles a tile).  A group whose word counts all its tiles
// holds its aggregate; a warp that has resolved a tile stores the inclusive
// prefix of the group before it.  A tile's output offset is the exclusive
// prefix of its group (a look-back over group words, a few dozen deep) plus
// the counts of the tiles before it in the group; all those words are read
// at once, in one L2 round trip.  A word carries all that is read from it,
// so relaxed accesses suffice.  Every wait is bounded by the time budget and
// ends early once another warp has given up.
// The parameter type P supplies status, gagg, ginc, n_tiles, timeout_ns,
// withhold, error() (the launch record's error word), COUNT (the bits of a
// tile's status word that hold its count) and SMALL (the counts of 32
// groups add up to less than 2^32).
#pragma once

#include "devutil.cuh"

namespace lx {

constexpr uint32_t GS = 256;                  // tiles per look-back group
constexpr unsigned ERR_TIMEOUT_BIT = 1u;      // the error word's "a wait ran out" bit
constexpr int GW_SHIFT = 54;                  // a group word: tiles that have published << 54 | their counts
constexpr int LB_IN = GS / 32;                // status words per lane of a tile's own group

// Polls back off exponentially (64 ns doubling to 4 us): while one slow tile
// (say, a chunk walked byte by byte) holds up its group, thousands of waiting
// warps must not flood L2 with status reads and starve that tile's own loads.
struct Waiter {
    uint64_t t0 = 0;
    uint32_t spins = 0;
    // false (and the error flag raised) once the budget is spent
    template <class PT>
    __device__ bool again(const PT &P)
    {
        if (spins == 0) t0 = globaltimer();
        if ((++spins & 3) == 0 &&
            (globaltimer() - t0 > P.timeout_ns || *(volatile const unsigned int *)P.error() != 0)) {
            if ((threadIdx.x & 31) == 0) atomicOr(P.error(), ERR_TIMEOUT_BIT);
            return false;
        }
        __nanosleep(64u << min(spins, 6u));
        return true;
    }
};

// `word`: the tile's count with whatever else its kernel keeps beside it.
template <class PT>
__device__ __forceinline__ void publish_word(const PT &P, uint32_t tile, unsigned long long word)
{
    if ((threadIdx.x & 31) == 0 && tile != P.withhold) {
        st_status(&P.status[tile], ST_AGG | word);
        asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(&P.gagg[tile / GS]),
                     "l"((1ull << GW_SHIFT) | (word & PT::COUNT)) : "memory");
    }
}

template <class PT>
__device__ __forceinline__ unsigned long long warp_sum(unsigned long long x)
{
    if (PT::SMALL) return __reduce_add_sync(0xffffffffu, (uint32_t)x);
    for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Lane 0 waits until done(); the warp learns whether the wait ended in time.
template <class PT, class F>
__device__ bool wait_for(const PT &P, Waiter &W, F done)
{
    uint32_t ok = 1;
    if ((threadIdx.x & 31) == 0)
        while (!done())
            if (!W.again(P)) {
                ok = 0;
                break;
            }
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

// The output offset of `tile` and the status word of the tile before it (0
// for tile 0); false when a wait ran out of time.  A wait polls one word, by
// lane 0, and then reads the round again.  (Groups of 256 tiles: with 64, the
// group words of a 4 KiB-tile launch are read so often that 512 MiB of JSON took
// 2.2 ms instead of 0.73.)
template <class PT>
__device__ __forceinline__ bool resolve_tile(const PT &P, uint32_t tile, uint64_t &G, unsigned long long &before)
{
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t g = tile / GS, f = g * GS, nt = tile - f;   // nt: tiles before it in its group
    Waiter W;
    int64_t base = (int64_t)g - 1;
    unsigned long long inc, agg, v[LB_IN];
    auto load_groups = [&]() {
        const int64_t k = base - (int64_t)lane;
        inc = k >= 0 ? ld_status(&P.ginc[k]) : ST_INCL;
        agg = k >= 0 ? ld_status(&P.gagg[k]) : 0ull;
    };
#pragma unroll
    for (int i = 0; i < LB_IN; i++) v[i] = lane + 32 * i < nt ? ld_status(&P.status[f + lane + 32 * i]) : ST_AGG;
    before = tile ? ld_status(&P.status[tile - 1]) : ST_AGG;
    load_groups();
    for (;;) {
        uint32_t miss = before == 0 ? tile - 1 : 0xFFFFFFFFu;
#pragma unroll
        for (int i = LB_IN - 1; i >= 0; i--) miss = v[i] == 0 ? f + lane + 32 * i : miss;
        const uint32_t m = __reduce_min_sync(0xffffffffu, miss);
        if (m == 0xFFFFFFFFu) break;
        if (!wait_for(P, W, [&] { return ld_status(&P.status[m]) != 0; })) return false;
#pragma unroll
        for (int i = 0; i < LB_IN; i++)
            if (v[i] == 0) v[i] = ld_status(&P.status[f + lane + 32 * i]);
        if (before == 0) before = ld_status(&P.status[tile - 1]);
    }
    unsigned long long own = 0;
#pragma unroll
    for (int i = 0; i < LB_IN; i++) own += v[i] & PT::COUNT;   // 0 past the tile
    const unsigned long long w = warp_sum<PT>(own);
    uint64_t GE = 0;
    bool found = base < 0, near = true;
    while (!found) {
        const unsigned vi = __ballot_sync(0xffffffffu, inc != 0);
        const unsigned va = __ballot_sync(0xffffffffu, (agg >> GW_SHIFT) == GS);
        const unsigned nearer = vi ? (vi & (0u - vi)) - 1u : 0xffffffffu;   // lanes before the nearest prefix
        if (nearer & ~va) {   // the farthest group before it that is not complete yet: wait, and sum again
            const int64_t k = base - (31 - __clz(nearer & ~va));
            if (!wait_for(P, W, [&] {
                    return (ld_status(&P.gagg[k]) >> GW_SHIFT) == GS || ld_status(&P.ginc[k]) != 0;
                }))
                return false;
            GE = 0;
            base = (int64_t)g - 1;
            load_groups();
            continue;
        }
        if (nearer) {
            GE += warp_sum<PT>((nearer >> lane) & 1u ? agg & ((1ull << GW_SHIFT) - 1) : 0ull);
            near = false;
        }
        if (vi) {
            GE += __shfl_sync(0xffffffffu, inc, __ffs(vi) - 1) & ST_VAL;
            found = true;
        } else {
            base -= 32;
            load_groups();
        }
    }
    // the inclusive prefix of the group before shortens later look-backs
    if (lane == 0 && g > 0 && !near) st_status(&P.ginc[g - 1], ST_INCL | GE);
    if (tile == 0) before = 0;
    G = GE + w;
    return true;
}

}  // namespace lx
