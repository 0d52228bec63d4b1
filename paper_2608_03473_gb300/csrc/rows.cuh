// rows.cuh -- device parts shared by the kernels that walk the event-code
// tables from known rows (rows.cu, ctxmap.cu): launch parameters, table
// staging, the byte and word steps.  Not part of the C ABI.
#pragma once

#include <cstdint>

#include "devutil.cuh"
#include "internal.h"
#include "lookback.cuh"
#include "runtime.h"

namespace lx {

struct RResult {
    unsigned long long total;          // kept tokens over all tiles
    unsigned long long inv_fail_pos;   // ~min failure position, 0 = none
    unsigned long long inv_fail_tok;   // ~output index at that failure
    unsigned int error;
    unsigned int pad;
};

struct HostRecord {
    RResult r;
    uint32_t seq;                      // of the last launch that has finished
};

struct RParams {
    const uint8_t *in;             // 16-byte aligned; the input is [lo, n) of it
    uint64_t n;
    uint32_t lo;                   // 0..15
    uint32_t slice;                // bytes per slice
    uint32_t stage;                // tokens a warp's stage holds
    const uint8_t *blob;           // walk table, then WalkTable::sync
    uint32_t blob_bytes, rows_bytes, row_shift, sync_bytes;   // multiples of 16 but the shift
    uint32_t p_start, p_pre, acc_off, kmap_off, cmap_off;
    uint32_t noacc_off;            // u8 per row (WalkTable::noacc), in global memory only; 0: failures in an earlier slice are not taken
    uint32_t guess;                // bytes walked before a slice at first
    uint16_t *rows;                // entry row of every slice (relative address)
    uint32_t row_step;             // rows per slice of lex_rows
    const unsigned int *before;    // an error word that the kernels before lex_rows may have set, or nullptr
    uint64_t n_slices;
    uint16_t *out_kinds;
    uint32_t *out_lens;
    uint64_t cap;
    uint16_t *spill;               // per warp of the grid: a tile's stage entries beyond the shared stage
    unsigned long long *status;    // per tile: ST_AGG | exit row << 32 | last event position + 1 << 16 | kept count
    unsigned long long *gagg, *ginc;   // per group of tiles (lookback.cuh)
    unsigned int *tile_counter;
    RResult *res;
    uint64_t zero_bytes;           // of the scratch from res on, zeroed by row_guess
    uint32_t n_tiles;
    uint64_t timeout_ns;
    uint32_t withhold;
    // the end of the launch: the last CTA writes the record and then `seq` to
    // pinned host memory, and with `clean` zeroes the scratch for the next call
    unsigned int *done;            // CTAs that have finished
    HostRecord *host;
    uint32_t seq, clean;
    uint32_t n_pat;                // synchronizing byte values where they are few (0: more than four)
    uint32_t pat[4];               // each four times
    // batches
    const WDoc *docs;
    const uint32_t *tile_doc;      // document of every tile
    WDocRes *dres;
    uint32_t sets_off;             // WSet array in the table
    unsigned long long *down;      // pinned: the record and the document records (D), then the sequence number
    uint32_t n_docs;
    static constexpr unsigned long long COUNT = 0xFFFFull;
    static constexpr bool SMALL = true;
    __device__ unsigned int *error() const { return &res->error; }
};

// The table parameters of a token set's walk table (rows.cu).
void rows_table(const lx_tokenset *ts, int mode, const DeviceTables &dt, RParams &P);

namespace {   // each translation unit its own copy

constexpr uint32_t NONE = 0xFFFFFFFFu;
constexpr uint32_t BIG = 0x7FFFFFFFu;
constexpr uint32_t ROW_UNKNOWN = 0xFFFFu;   // entry row: none found (rows are at even addresses)
constexpr uint32_t ROW_LOST = 0xFFFEu;      // entry row: a token before it backtracks
constexpr uint32_t ROW_DEAD = 0xFFFDu;      // entry row: after the first failure
constexpr int MAX_WARPS = 20;               // warps per CTA at most
constexpr uint32_t LEN_MAX = 511;           // a stage entry's length field; this value: kept aside
constexpr uint32_t GUESS_MAX = 8192;        // bytes before a slice searched for a synchronizing byte
constexpr int GUESS_NT = 512;
constexpr unsigned ERR_TIMEOUT = ERR_TIMEOUT_BIT;
constexpr unsigned ERR_SMEM = 2u;
constexpr unsigned ERR_ROWS = 4u;           // entry rows do not fit together: lex the input another way
constexpr unsigned ERR_FAR = 8u;            // no synchronizing byte near a slice

// A warp's shared memory: the slices' bytes and then, in their place, their
// event codes, SLICE + 16 bytes per lane (the 16-byte stores and loads of eight
// lanes then fall in different banks); the stage of P.stage tokens, 2 bytes each
// (event code << 8 | length); the mbarrier of the copies.
template <int NW>   // event mask words per lane
struct Geo {
    static constexpr uint32_t SLICE = 32 * NW;
    static constexpr uint32_t TILE = 32 * SLICE;
    static constexpr uint32_t STRIDE = SLICE + 16;
};
// Shared bytes of a warp with a stage of `stage` tokens (a multiple of 8).
__host__ __device__ constexpr uint32_t warp_area(uint32_t nw, uint32_t stage)
{
    return 32 * (32 * nw + 16) + 2 * stage + 16;
}
// Tokens of the stage: what a tile of 1024 nw bytes seldom exceeds, so that
// enough warps fit (a stage for every mode's tokens left 16 beside the C-like
// set's table at nw = 6, one for the filtered modes' tokens leaves 18).
constexpr uint32_t stage_for(int nw, int mode)
{
    return nw < 3 ? 1024 * nw : mode == LX_FULL_EXACT ? 352 * nw : 240 * nw;
}

// Shared addresses of the tables.
struct REnv {
    uint32_t tb, start, pre, slow, acc, kmap, cmap, shift;
};

__device__ __forceinline__ uint4 ldg16(const uint8_t *p)
{
    return __ldg(reinterpret_cast<const uint4 *>(p));
}
__device__ __forceinline__ void sts16(uint32_t a, uint32_t x, uint32_t y, uint32_t z, uint32_t w)
{
    asm volatile("st.shared.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(x), "r"(y), "r"(z), "r"(w) : "memory");
}
__device__ __forceinline__ uint4 lds16(uint32_t a)
{
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
    return v;
}
__device__ __forceinline__ void sts_u16(uint32_t a, uint32_t v)
{
    asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((unsigned short)v) : "memory");
}

__device__ __forceinline__ void mbar_init(uint32_t mbar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mbar) : "memory");
}
__device__ __forceinline__ void fence_proxy_async()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// `bytes` (a multiple of 16, both addresses 16-byte aligned) global -> shared.
__device__ __forceinline__ void bulk_load(uint32_t dst, const uint8_t *src, uint32_t bytes, uint32_t mbar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(src), "r"(bytes), "r"(mbar) : "memory");
}
// Bounded wait for a phase of the mbarrier; false when the time budget runs out.
__device__ __forceinline__ bool mbar_wait(uint32_t mbar, uint32_t parity, uint64_t timeout_ns)
{
    uint64_t t0 = 0;
    for (uint32_t it = 0;; it++) {
        uint32_t done;
        asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                     "selp.u32 %0, 1, 0, p;\n\t}" : "=r"(done) : "r"(mbar), "r"(parity) : "memory");
        if (done) return true;
        if (it % 16 == 0) {
            const uint64_t t = globaltimer();
            if (!t0) t0 = t;
            else if (t - t0 > timeout_ns) return false;
        }
    }
}

// SPREAD: the class form's rows as stage_table<FORM, true> lays them out.
template <int FORM, bool SPREAD = false>
__device__ __forceinline__ uint32_t wstep(const REnv &E, uint32_t e, uint32_t b)
{
    const uint32_t a = FORM == FORM_BYTE ? ((e & ~0x1FEu) | (b << 1))
                                         : ((e & ~0xFFu) | (lds_u8(E.cmap + b) ^ (SPREAD ? (e >> 6) & 0x7Cu : 0u)));
    return lds_u16(a);
}
__device__ __forceinline__ uint32_t acc_code(const REnv &E, uint32_t e)
{
    return lds_u8(E.acc + ((e - E.tb) >> E.shift));
}

// Four byte steps over the little-endian word w (per byte one LOP3 and the
// dependent table load; the class form adds a PRMT and the class map's load,
// which depend on the input alone); returns the four event codes.
#define LXR_B(XOP, VIN, VOUT)                                                  \
    XOP "lop3.b32 a, " VIN ", t, %4, 0xD8;\n\t"                                \
        "ld.shared.u16 " VOUT ", [a];\n\t"
#define LXR_C(SEL, VIN, VOUT)                                                  \
    "prmt.b32 t, %2, %3, " SEL ";\n\t"                                         \
    "ld.shared.u8 c, [t];\n\t"                                                 \
    "lop3.b32 a, " VIN ", c, %4, 0xD8;\n\t"                                    \
    "ld.shared.u16 " VOUT ", [a];\n\t"
#define LXR_HEAD "{\n\t.reg .b32 t, a, c, v0, v1, v2, t0, t1;\n\t"
#define LXR_PACK                                                               \
    "prmt.b32 t0, v0, v1, 0x0040;\n\t"                                         \
    "prmt.b32 t1, v2, %0, 0x0040;\n\t"                                         \
    "prmt.b32 %1, t0, t1, 0x5410;\n\t}"

template <int FORM>
__device__ __forceinline__ uint32_t wword(uint32_t &e, uint32_t w, uint32_t cm)
{
    uint32_t pk;
    if (FORM == FORM_BYTE)
        asm volatile(LXR_HEAD LXR_B("shl.b32 t, %2, 1;\n\t", "%0", "v0") LXR_B("shr.b32 t, %2, 7;\n\t", "v0", "v1")
                         LXR_B("shr.b32 t, %2, 15;\n\t", "v1", "v2") LXR_B("shr.b32 t, %2, 23;\n\t", "v2", "%0")
                             LXR_PACK
                     : "+r"(e), "=r"(pk) : "r"(w), "r"(cm), "r"(0x1FEu) : "memory");
    else
        asm volatile(LXR_HEAD LXR_C("0x7650", "%0", "v0") LXR_C("0x7651", "v0", "v1") LXR_C("0x7652", "v1", "v2")
                         LXR_C("0x7653", "v2", "%0") LXR_PACK
                     : "+r"(e), "=r"(pk) : "r"(w), "r"(cm), "r"(0xFFu) : "memory");
    return pk;
}

// The code at shared address a where v != 0 (else undefined): lanes without an
// event stay off the banks.
__device__ __forceinline__ uint32_t event_code(uint32_t a, uint32_t v)
{
    uint32_t c;
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p ld.shared.u8 %0, [%1];\n\t}"
                 : "=r"(c) : "r"(a), "r"(v));
    return c;
}

// An event at position pos: where there is one (v != 0), a kept token (code >=
// 4) from prev to pos goes into the stage at sa, which advances, and prev
// moves on.
__device__ __forceinline__ void put_event(uint32_t &sa, int &prev, uint32_t v, uint32_t code, uint32_t pos)
{
    asm volatile("{\n\t.reg .pred p, q;\n\t.reg .b32 d;\n\t"
                 "setp.ne.u32 p, %2, 0;\n\t"
                 "setp.gt.and.u32 q, %3, 3, p;\n\t"
                 "sub.u32 d, %4, %1;\n\t"
                 "mad.lo.u32 d, %3, 256, d;\n\t"
                 "@q st.shared.u16 [%0], d;\n\t"
                 "@q add.u32 %0, %0, 2;\n\t"
                 "@p mov.u32 %1, %4;\n\t}"
                 : "+r"(sa), "+r"(prev) : "r"(v), "r"(code), "r"(pos) : "memory");
}

__device__ __forceinline__ uint32_t kept_mask(uint32_t w)   // bit 7 of every byte >= 4 (a kept code)
{
    return (((w | 0x80808080u) - 0x04040404u) | w) & 0x80808080u;
}
__device__ __forceinline__ uint32_t event_mask(uint32_t w)  // bit 7 of every nonzero byte
{
    return (((w & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | w) & 0x80808080u;
}

// Stage the walk table (row offsets become shared addresses) with the PRE
// row replaced by the synchronizing one; false where the 16-bit row
// addresses would not reach every row.  Class-form rows start on 256-byte
// boundaries, so a class has the same bank in every row and lanes that read
// one class in different rows queue; SPREAD: the words of each row are XORed
// with its number.  That takes a sixth off the wavefronts of the C-like set's
// walk and two instructions more on each byte's chain: 6 % faster where six
// chains hide them (cm_maps), nothing on C-like text and 12 % slower on a
// batch in lex_rows, which therefore does without.
template <int FORM, bool SPREAD = false>
__device__ bool stage_table(const RParams &P, uint8_t *smem, REnv &E)
{
    const uint32_t sbase = smem_u32(smem), tb = (sbase + 511u) & ~511u;
    if (tb + P.rows_bytes > 65536u) {
        if (threadIdx.x == 0) atomicOr(P.error(), ERR_SMEM);
        return false;
    }
    uint4 *dst = reinterpret_cast<uint4 *>(smem + (tb - sbase));
    const uint4 *src = reinterpret_cast<const uint4 *>(P.blob);
    const uint32_t n = P.blob_bytes / 16, r = P.rows_bytes / 16, pre = P.p_pre / 16, tb2 = tb * 0x10001u;
    for (uint32_t i = threadIdx.x; i < n; i += blockDim.x) {
        uint4 v = __ldg(src + (i - pre < P.sync_bytes / 16 ? n + (i - pre) : i));
        if (i < r) v = make_uint4(__vadd2(v.x, tb2), __vadd2(v.y, tb2), __vadd2(v.z, tb2), __vadd2(v.w, tb2));
        if (SPREAD && FORM == FORM_CLASS && i < r) {   // word j of row q at j ^ (q mod 32), q as in the row's address
            const uint32_t at = tb + 16 * i, x = (at >> 6) & 0x7Cu;
            sts_u32(at ^ x, v.x);
            sts_u32((at + 4) ^ x, v.y);
            sts_u32((at + 8) ^ x, v.z);
            sts_u32((at + 12) ^ x, v.w);
        } else {
            dst[i] = v;
        }
    }
    E.tb = E.slow = tb;
    E.start = tb + P.p_start;
    E.pre = tb + P.p_pre;
    E.acc = tb + P.acc_off;
    E.kmap = tb + P.kmap_off;
    E.cmap = tb + P.cmap_off;
    E.shift = P.row_shift;
    return true;
}

}  // namespace
}  // namespace lx
