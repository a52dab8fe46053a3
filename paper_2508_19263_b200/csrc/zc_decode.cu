// Decoder kernel (table decode of the Huffman-coded streams fused with field merge) and zc_decompress.
//
// One warp per chunk, one lane per subchunk.  The chunk's compressed piece is staged in shared memory
// with a bulk asynchronous copy (TMA, non-multicast) completing on an mbarrier.  Work proceeds in
// rounds: every lane decodes R symbols of its own subchunk into a padded row of shared memory, then the
// whole warp merges 32 x R symbols with the other stream and writes 16-byte vectors, fully coalesced.
// The bytes of a raw stream come by bulk copies too in chunks of up to 4 KiB (run_small); in larger ones those of a round are
// prefetched into the L2 before it is decoded, as a delta's base tensor is, so that the DRAM latency hides behind the table lookups.
// Small chunks without a coded stream are only merged (run_plain).
#include "zc_device.cuh"

#include <atomic>
#include <chrono>

namespace zc {

struct DecParams {
    const uint8_t* comp;
    const uint8_t* base;     // XOR-delta form: the decoded tensor is XOR-ed with this one before it is written; or null
    uint8_t* out;
    Control* ctl;
    uint64_t comp_bytes, input_bytes, n_syms, n_elems;
    uint32_t n_chunks, cs, sub, chunk_bytes, format, group;
    uint32_t pool_bytes;     // per-warp shared memory: symbol rows first, the rest stages compressed pieces
    uint32_t c_begin, c_end; // chunks the launch decodes (zc_decompress: all of them)
    uint32_t spec;           // the container is long enough to read stream 0's tables before the header is checked
    uint32_t spin_limit;     // polls after which a wait for a staged piece gives up
    uint32_t skip_copy;      // test hook: the copies of the pieces are not started
    uint32_t sliced;         // large chunks: pieces are staged slice by slice and lane by lane (see run_chunks)
    uint32_t groups;         // decode_split_kernel: blocks a chunk's subchunks are dealt to (1, 2, 4 or 8)
    uint32_t active;         // warps of a block that decode chunks (they share the pools); the others only help to build the tables
    unsigned long long call_id;
};

// One tensor of a batch, and the parameters of a batched launch.  The tensors share format and chunk size;
// the chunks of all of them form one index space that is cut into contiguous slices (see kDecMaxPieces).
struct DecItem {
    const uint8_t* comp;
    const uint8_t* base;
    uint8_t* out;
    uint64_t comp_bytes, input_bytes, n_syms, n_elems;
    uint32_t n_chunks, first_chunk;          // first_chunk = chunks of all earlier tensors of the launch
};
// The chunk index space of a batched launch is cut into as many equal slices as there are blocks, and a slice into pieces that
// shrink.  A block takes the pieces of its own slice one after the other; when it is through, it takes pieces that the slices'
// owners have not come to yet, largest first, so that blocks end together although tensors, and SMs, differ in how fast they
// get through a piece.  Who takes a piece sets its bit in the control block (nobody else takes a slice's first piece).  The next
// piece of one's own slice is nearly always of the same tensor, whose tables are kept; another one costs about 12 us (waiting for
// the block's last warp, header, tables, first pieces).  (Dealt out in rounds over the whole index space by a ticket counter, every
// piece of a block was of another tensor; the step from that to slices, with the chunk loops as they were then: 1.74 GB of BF16 weights
// 621 -> 612 us, their delta of 872 MB 550 -> 524, 18 tensors of 66 MB in all 58 -> 53.  In one piece each, the delta took 659 us.)
constexpr uint32_t kDecMaxPieces = 5, kDecOneRound = 64;
constexpr uint32_t kDecMaxBlocks = 160, kDecClaimWords = kDecMaxBlocks / 32;
constexpr size_t kDecClaims = 128;           // where the bits are in the control block: [piece - 1][kDecClaimWords]
static_assert(sizeof(Control) <= kDecClaims && kDecClaims + 4 * (kDecMaxPieces - 1) * kDecClaimWords <= kControlBytes, "control block");
constexpr uint32_t kDecBatchMax = 448;       // tensors per launch: the parameter block stays below 32 KiB
struct DecBatchParams {
    Control* ctl;
    unsigned long long call_id;
    uint32_t cs, sub, chunk_bytes, format, group, pool_bytes;
    uint32_t n_tensors, n_empty, tensor_base, total;      // n_empty: tensors without chunks; total: chunks
    uint32_t n_pieces, piece_end[kDecMaxPieces];          // where a slice's pieces end, in 65536ths of it
    uint32_t spin_limit, skip_copy, sliced;
    DecItem item[kDecBatchMax];
};

constexpr uint32_t kLutBytes = kLutEntries * 4;       // one decode table: 4096 entries of 4 bytes
constexpr uint32_t kScratchBytes = 1280;           // code bookkeeping of build_lut (258 words)
constexpr uint32_t kDecMaxWarps = 28;              // 896 threads: 72 registers per thread fit the register file
// Launches that expect both streams to be coded (scale bytes, deltas) keep two bit readers per lane going and stage two
// pieces per warp: fewer warps fit the shared memory anyway, and the kernels built for them get more registers.
constexpr uint32_t kDecMaxWarpsBoth = 20;          // 640 threads: 96 registers per thread
template <int FMT, bool XOR>
constexpr uint32_t dec_block_warps() { return (XOR || FMT == ZC_FMT_SCALE_U8) ? kDecMaxWarpsBoth : kDecMaxWarps; }
// Launches of few chunks (at most kDecFewActive per SM) run kernels of their own: every SM takes a share of the chunks
// however few they are, all 16 warps of a block build the tables, and only as many warps as the block has chunks decode,
// each with room to stage whole pieces of both streams and with registers for two bit readers.  What such a launch takes
// is one lane's serial walk over its subchunk: 16 chunks of 64 KiB with both streams coded (FP8) took 230 us as 16 warps of
// one block that staged slices.
constexpr uint32_t kDecFewWarps = 16, kDecFewActive = 8;
constexpr int kDecMany = 0, kDecFew = 1, kDecSplit = 2;   // kernels of a single-tensor launch
constexpr uint32_t kDecStaticSmem = 2 * kLutBytes + 512;      // the decode tables (block_luts), and the kernels' variables
// The block's decode tables.  They are static shared memory: their addresses are constants and no register holds them.
__device__ __forceinline__ uint32_t* block_luts()
{
    __shared__ __align__(16) uint32_t s_lut[2 * kLutEntries];
    return s_lut;
}
constexpr uint32_t kSliceSyms = 128;               // symbols a lane decodes from one slice of its subchunk
constexpr uint32_t kSliceBytes = 256;              // copied per slice: 15 bytes of alignment + 128 * 12 bits + the window's look-ahead fit
constexpr uint32_t kSliceSlot = 272;               // a lane's slot

__device__ __forceinline__ void sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    ZC_DBG_SHARED(addr, 16, return);
    asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" :: "r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t addr)
{
    ZC_DBG_SHARED(addr, 16, return make_uint4(0, 0, 0, 0));
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}

__device__ __forceinline__ uint32_t lds16(uint32_t addr)
{
    ZC_DBG_SHARED(addr, 2, return 0);
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
    return v;
}

// ------------------------------------------------------------------------------------------------
// decode tables, built by every block from the container's code-length table
// ------------------------------------------------------------------------------------------------
// Canonical-code bookkeeping in shared memory, per code length l = 1..12:
//   count[l]  codes of that length            first[l]  value of the first one
//   offset[l] position of its symbols in the (length, symbol)-sorted list
//   limit[l]  windows below this value start with a code of length <= l
struct CodeBook {
    uint32_t* count;   // [16]
    uint32_t* first;   // [16]
    uint32_t* offset;  // [16]
    uint32_t* limit;   // [16]
    uint32_t* wcount;  // [8][16] per-warp counts, then exclusive prefix over warps
    uint8_t* sorted;   // [256]
    uint32_t* ok;      // [0] lengths usable, [1] symbols per lookup
};

__device__ __forceinline__ CodeBook codebook_views(uint32_t* scratch)
{
    CodeBook b;
    b.count = scratch; b.first = scratch + 16; b.offset = scratch + 32; b.limit = scratch + 48; b.wcount = scratch + 64;
    b.sorted = reinterpret_cast<uint8_t*>(scratch + 64 + 128);
    b.ok = scratch + 64 + 128 + 64;
    return b;
}

// Fills the table of one stream and decides how many symbols every lookup yields (returned in *per_lookup).
//   two-symbol mode   entry bits  7..0  bits the lookup consumes      15..8 first symbol     23..16 second symbol
//                                27..24 length of the first code       31   "only the first symbol is valid"
//   one-symbol mode   entry bits  7..0  length of the code              31..24 the symbol
// Two-symbol mode: a lookup normally yields the two symbols whose codes start the 12-bit window; when the two
// codes together are longer than 12 bits the entry carries the first one and bit 31, and the decoder fetches
// the second with one more lookup.  That mode is chosen when such pairs are rare (estimated from the code
// lengths with p(symbol) = 2^-length, an eighth of that for the two longest lengths); otherwise every lookup
// yields exactly one symbol.  A fixed number of
// symbols per lookup lets a lane assemble words of 4 symbols in registers without any bookkeeping.
// `single` is a 4096 x u16 scratch table (length << 8 | symbol of the first code of every window).
// Returns false to all threads if the lengths are not a complete prefix code (or the one-symbol code).
static __device__ bool build_lut(uint32_t my_len, uint32_t* lut, uint16_t* single, uint32_t* scratch, uint32_t* per_lookup)
{
    const CodeBook b = codebook_views(scratch);
    const uint32_t tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t my_rank = 0;                                        // my_len: length of symbol tid's code (threads < 256)
    if (tid < 64 + 128) scratch[tid] = 0;
    if (tid == 0) b.ok[0] = 1;
    __syncthreads();
    if (tid < 256) {
        if (my_len > kLmax) { b.ok[0] = 0; my_len = 0; }
        for (uint32_t l = 1; l <= kLmax; ++l) {
            const uint32_t m = __ballot_sync(0xFFFFFFFFu, my_len == l);
            if (my_len == l) my_rank = __popc(m & ((1u << lane) - 1));
            if (lane == 0) b.wcount[warp * 16 + l] = __popc(m);
        }
    }
    __syncthreads();
    if (warp == 0) {
        // Lane l looks after length l: adds up its codes over the 8 warps; the rest are prefix sums over the lengths.
        // weight = the share of the 2^12 windows that start with a code of length l (a code of length k < l takes 2^(l - k)
        // values of length l, so the first value of length l is the weight of all shorter ones >> (12 - l)).
        const uint32_t l = lane, use = l >= 1 && l <= kLmax;
        uint32_t cnt = 0;
        if (use)
            for (uint32_t w = 0; w < 8; ++w) { const uint32_t t = b.wcount[w * 16 + l]; b.wcount[w * 16 + l] = cnt; cnt += t; }
        const uint32_t weight = use ? cnt << (kLmax - l) : 0u;
        // weight of length l in units of 2^-12; codes at or next to the length limit belong to symbols that are rarer than
        // 2^-length says: the limit clipped them, or they are the never-seen symbols of a static dictionary
        const uint32_t p = l + 1 >= kLmax ? weight >> 3 : weight;
        uint32_t sum_w = weight, sum_c = cnt, sum_p = p;
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) {
            const uint32_t xw = __shfl_up_sync(0xFFFFFFFFu, sum_w, o), xc = __shfl_up_sync(0xFFFFFFFFu, sum_c, o), xp = __shfl_up_sync(0xFFFFFFFFu, sum_p, o);
            if (lane >= (uint32_t)o) { sum_w += xw; sum_c += xc; sum_p += xp; }
        }
        const uint32_t total = __shfl_sync(0xFFFFFFFFu, sum_w, kLmax), active = __shfl_sync(0xFFFFFFFFu, sum_c, kLmax);
        const uint32_t all_p = __shfl_sync(0xFFFFFFFFu, sum_p, kLmax), shorter_p = __shfl_sync(0xFFFFFFFFu, sum_p, use ? kLmax - l : 0u);
        const bool one = active == 1 && __shfl_sync(0xFFFFFFFFu, cnt, 1) == 1;
        // probability (units of 2^-24) that two consecutive codes need more than 12 bits: the first is of length l, the
        // second of length 13 - l or more
        unsigned long long pairs = use ? (unsigned long long)p * (all_p - shorter_p) : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) pairs += __shfl_xor_sync(0xFFFFFFFFu, pairs, o);
        if (use) {
            b.count[l] = cnt;
            b.first[l] = (sum_w - weight) >> (kLmax - l);
            b.offset[l] = sum_c - cnt;
            b.limit[l] = (l == 1 && one) ? kLutEntries : sum_w;   // the unused half of the windows reads as the one symbol
        }
        if (lane == 0) {
            if (!(total == kLutEntries || one || active == 0)) b.ok[0] = 0;      // Kraft sum is exactly one
            b.ok[1] = pairs <= (1ull << 24) / 32 ? 2u : 1u;
        }
    }
    __syncthreads();
    const uint32_t mode = b.ok[1];
    if (tid < 256 && my_len) b.sorted[b.offset[my_len] + b.wcount[warp * 16 + my_len] + my_rank] = (uint8_t)tid;
    uint32_t lim[kLmax + 1];
#pragma unroll
    for (uint32_t l = 1; l <= kLmax; ++l) lim[l] = b.limit[l];
    __syncthreads();
    // First code of every window: its length is the number of limits at or below the window value, plus one.  A thread takes
    // eight neighbouring windows at a time: they start with the same code when that is of 9 bits or less.
    const uint32_t single_s = smem_u32(single), lut_s = smem_u32(lut);
    auto first_code = [&](const uint32_t idx) -> uint32_t {
        uint32_t l = 1;
#pragma unroll
        for (uint32_t k = 1; k < kLmax; ++k) l += idx >= lim[k] ? 1u : 0u;
        uint32_t rel = (idx >> (kLmax - l)) - b.first[l];
        if (rel >= b.count[l]) rel = 0;                           // only reachable with damaged or one-symbol tables
        return (l << 8) | b.sorted[b.offset[l] + rel];
    };
    for (uint32_t idx = 8 * tid; idx < kLutEntries; idx += 8 * blockDim.x) {
        uint32_t e = first_code(idx) * 0x10001u, w[4] = {e, e, e, e};
        if ((e & 0xFF00u) > 0x900u) {
#pragma unroll
            for (uint32_t i = 0; i < 4; ++i) w[i] = first_code(idx + 2 * i) | first_code(idx + 2 * i + 1) << 16;
        }
        sts128(single_s + 2 * idx, w[0], w[1], w[2], w[3]);
    }
    __syncthreads();
    if (mode == 2) {
        // Neighbouring lanes look up the second codes of neighbouring windows.  (With eight windows to a lane those lookups
        // were up to 16-way bank conflicts: 16 BF16 chunks of 4 KiB 8.7 against 7.8 us, 300 BF16 tensors of 16 chunks in a
        // batch 55.6 against 51.3 us.)
        for (uint32_t idx = tid; idx < kLutEntries; idx += blockDim.x) {
            const uint32_t e1 = lds16(single_s + 2 * idx), l1 = e1 >> 8, s1 = e1 & 0xFF;
            const uint32_t e2 = lds16(single_s + 2 * ((idx << l1) & (kLutEntries - 1))), l2 = e2 >> 8, s2 = e2 & 0xFF;
            sts32(lut_s + 4 * idx, l1 + l2 <= kLmax ? (l1 + l2) | (s1 << 8) | (s2 << 16) | (l1 << 24) : l1 | (s1 << 8) | (l1 << 24) | 0x80000000u);
        }
    } else {
        for (uint32_t idx = 8 * tid; idx < kLutEntries; idx += 8 * blockDim.x) {
            const uint4 v = lds128(single_s + 2 * idx);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};          // two first codes each: length << 8 | symbol
            uint32_t e[8];
#pragma unroll
            for (uint32_t i = 0; i < 8; ++i) e[i] = __byte_perm(w[i / 2], 0, i & 1u ? 0x2443 : 0x0441);
            sts128(lut_s + 4 * idx, e[0], e[1], e[2], e[3]);
            sts128(lut_s + 4 * idx + 16, e[4], e[5], e[6], e[7]);
        }
    }
    __syncthreads();
    if (tid == 0) *per_lookup = mode;
    return b.ok[0] != 0;
}

// ------------------------------------------------------------------------------------------------
// per-lane decoding of one round
// ------------------------------------------------------------------------------------------------

__device__ __forceinline__ uint32_t load_sub_end(const uint8_t* tab, uint32_t width, uint32_t chunk, uint32_t lane)
{
    if (width == 2) return reinterpret_cast<const uint16_t*>(tab + 64ull * chunk)[lane];
    return reinterpret_cast<const uint32_t*>(tab + 128ull * chunk)[lane];
}

// A lane's place in its chunk's piece is the bit position `pos`.  Piece staged in shared memory: pos counts from shared
// address 0 (8 * byte address of the slot + bit in the piece), and the words around it are kept in registers (LaneBits), so a
// window is one funnel shift.  Piece read from global memory: pos counts from the start of the piece, a window loads its two
// words, and the word index is clamped to `lim`, the last place from which two words can be read.
// Bounds of the staged form: a lane starts inside its piece (checked against the tables before the chunk is
// decoded) and consumes at most 12 bits per symbol, so it reads less than 1.5 * sub + 16 bytes past the piece
// whatever the payload bits are; the block's shared memory ends with that much slack behind the last warp's
// slot.  With a valid container a lane reads at most 16 bytes past its piece (covered by the copy); with a
// damaged payload it decodes garbage in bounds and the consumed-bits check after the chunk reports the damage.

// A lane's bit reader.  w0, w1 = the aligned words that hold bits [32 i, 32 i + 64) of shared memory with i = pos / 32; with the
// look-ahead (see word_first) also w2 = the word behind them, addr = the address of the one after that.  A lane consumes at
// most 24 bits between two windows, so pos crosses at most one word boundary: then the words move up and one is loaded, in a
// predicated load in which only the lanes that crossed take part.
struct LaneBits { uint32_t pos, w0, w1, w2, addr; };

__device__ __forceinline__ void lane_start(LaneBits& L, const uint32_t at)
{
    const uint32_t a = (at >> 3) & ~3u;
    ZC_DBG_SHARED(a, 4, return); ZC_DBG_SHARED(a + 8, 4, return);
    L.pos = at;
    L.addr = a + 12;
    asm volatile("ld.shared.u32 %0, [%3];\n\tld.shared.u32 %1, [%3+4];\n\tld.shared.u32 %2, [%3+8];" : "=r"(L.w0), "=r"(L.w1), "=r"(L.w2) : "r"(a));
}
__device__ __forceinline__ uint32_t window_s(const LaneBits& L)
{
    return __funnelshift_l(L.w1, L.w0, L.pos);                  // the shift takes the low 5 bits of pos
}
// pos moves on to `to` (at most 32 bits further).  AHEAD: the word behind the window's is in a register already and the next one
// is requested; otherwise the window's second word is loaded when it is needed.
template <bool AHEAD>
__device__ __forceinline__ void lane_advance(LaneBits& L, const uint32_t to)
{
    const uint32_t cross = (L.pos ^ to) & 32u;
    L.pos = to;
    if (AHEAD) {
        if (cross) ZC_DBG_SHARED(L.addr, 4, return);
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t@p mov.u32 %0, %1;\n\t@p mov.u32 %1, %2;\n\t"
                     "@p ld.shared.u32 %2, [%3];\n\t@p add.u32 %3, %3, 4;\n\t}"
                     : "+r"(L.w0), "+r"(L.w1), "+r"(L.w2), "+r"(L.addr) : "r"(cross));
    } else {
        const uint32_t a = ((to >> 3) & ~3u) + 4;
        if (cross) ZC_DBG_SHARED(a, 4, return);
        L.w0 = cross ? L.w1 : L.w0;
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p ld.shared.u32 %0, [%1];\n\t}" : "+r"(L.w1) : "r"(a), "r"(cross));
    }
}
__device__ __forceinline__ uint32_t window_g(const uint32_t* __restrict__ pay, uint32_t pos, uint32_t lim)
{
    const uint32_t w = min(pos >> 5, lim);
    return __funnelshift_l(__ldg(pay + w + 1), __ldg(pay + w), pos);
}
// window = top 12 bits; the address by a multiply-add, off the integer ALU pipe
__device__ __forceinline__ uint32_t lut_peek(uint32_t win, uint32_t lut_s)
{
    uint32_t addr;
    asm("mad.lo.u32 %0, %1, 4, %2;" : "=r"(addr) : "r"(win >> (32 - kLmax)), "r"(lut_s));
    return lds32(addr);
}
// pos + low byte of x, in one multiply-add-like instruction off the integer ALU pipe
__device__ __forceinline__ uint32_t add_low_byte(uint32_t pos, uint32_t x) { return __dp4a(x, 1u, pos); }

// Decode one word of 4 symbols from a piece staged in shared memory.  K = symbols per lookup (1 or 2).
// A window of 32 bits serves two lookups of at most 12 bits each.
// Two-symbol mode: entry = bits | first symbol << 8 | second symbol << 16 | first length << 24 | flag << 31.  A
// lookup whose second code did not fit the window carries the flag (rare by construction of the mode) and
// consumes its first code only, so the two lookups still end on a code boundary, one symbol short (two if both
// carry the flag); the missing symbols come from a fresh window.
// One-symbol mode: entry = length | symbol << 24, so that `pos += entry` advances the position and leaves the
// symbol in bits the position does not use.
// word_first makes the window and the two lookups that every word needs; word_second finishes the word: two more lookups
// from a second window in one-symbol mode, the rare extra lookups of short pair entries in two-symbol mode.
// The one-symbol mode keeps a word in flight ahead of its windows, of which it has twice as many: without it 436 MB of FP8
// weights at 16 KiB take 200 instead of 193 us.  The two-symbol mode is bound by its instructions, and the look-ahead costs
// three registers to move at every window: 872 MB of BF16 weights 307 us with it, 301 us without.
template <int K>
__device__ __forceinline__ void word_first(LaneBits& L, const uint32_t lut_s, uint32_t& x, uint32_t& y)
{
    const uint32_t win = window_s(L);
    x = lut_peek(win, lut_s);
    y = lut_peek(__funnelshift_l(0, win, x), lut_s);            // consume: low 5 bits of the entry
    lane_advance<K == 1>(L, add_low_byte(add_low_byte(L.pos, x), y));
}
template <int K>
__device__ __forceinline__ uint32_t word_second(LaneBits& L, const uint32_t lut_s, const uint32_t e0, const uint32_t e1)
{
    if (K == 2) {
        if ((int)(e0 | e1) < 0) {
            const uint32_t win = window_s(L);
            const uint32_t f = lut_peek(win, lut_s), lf = (f >> 24) & 15;
            if ((int)(e0 & e1) < 0) {                            // both: first symbols of e0, e1, f and of one more lookup
                const uint32_t g = lut_peek(__funnelshift_l(0, win, lf), lut_s);
                lane_advance<false>(L, L.pos + lf + ((g >> 24) & 15));
                return __byte_perm(__byte_perm(e0, e1, 0x0051), __byte_perm(f, g, 0x0051), 0x5410);
            }
            lane_advance<false>(L, L.pos + lf);
            // e0 short: e0's first, e1's two; e1 short: e0's two, e1's first; then f's first
            return __byte_perm(__byte_perm(e0, e1, (int)e0 < 0 ? 0x0651 : 0x0521), f, 0x5210);
        }
        return __byte_perm(e0, e1, 0x6521);
    }
    uint32_t c, d;
    word_first<1>(L, lut_s, c, d);
    return __byte_perm(__byte_perm(e0, e1, 0x0073), __byte_perm(c, d, 0x0073), 0x5410);
}
template <int K>
__device__ __forceinline__ uint32_t decode_word(LaneBits& L, const uint32_t lut_s)
{
    uint32_t x, y;
    word_first<K>(L, lut_s, x, y);
    return word_second<K>(L, lut_s, x, y);
}

// Decoded symbols of a round, per coded stream and warp: lane L owns PPL quads (16 symbols = 16 bytes each);
// its quad q lives in 16-byte slot L * PPL + (q ^ f(L)), f(L) = (L >> (3 - log2 PPL)) & (PPL - 1).  With this
// placement both the writers (32 lanes, same q, one 16-byte store each) and the readers of the merge (lane l
// reads quad l % PPL of row l / PPL + i * 32 / PPL) touch eight different 16-byte bank groups per quarter warp:
// no bank conflicts on either side, one store per 16 symbols and one load per merged part.
template <int K, int PPL, bool FULL>
__device__ __forceinline__ void decode_round(LaneBits& L, const uint32_t lut_s, uint32_t wr_s, uint32_t fw, uint32_t n_quads)
{
#pragma unroll
    for (int q = 0; q < PPL; ++q) {
        if (!FULL && (uint32_t)q >= n_quads) break;
        const uint32_t s0 = decode_word<K>(L, lut_s);
        const uint32_t s1 = decode_word<K>(L, lut_s);
        const uint32_t s2 = decode_word<K>(L, lut_s);
        const uint32_t s3 = decode_word<K>(L, lut_s);
        sts128(wr_s + 16 * ((uint32_t)q ^ fw), s0, s1, s2, s3);
    }
}

// Two coded streams: the same words, decoded for both streams side by side.  A lane's two bit readers are independent
// chains of dependent operations (window -> lookup -> shift -> lookup); issued alternately, one chain's shared-memory
// latency is covered by the other's arithmetic.
template <int K0, int K1, int PPL, bool FULL>
__device__ __forceinline__ void decode_round2(LaneBits& A, const uint32_t luta_s, uint32_t wra_s, LaneBits& B, const uint32_t lutb_s, uint32_t wrb_s,
                                              uint32_t fw, uint32_t n_quads)
{
#pragma unroll
    for (int q = 0; q < PPL; ++q) {
        if (!FULL && (uint32_t)q >= n_quads) break;
        uint32_t a[4], b[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            uint32_t ax, ay, bx, by;
            word_first<K0>(A, luta_s, ax, ay);
            word_first<K1>(B, lutb_s, bx, by);
            a[j] = word_second<K0>(A, luta_s, ax, ay);
            b[j] = word_second<K1>(B, lutb_s, bx, by);
        }
        sts128(wra_s + 16 * ((uint32_t)q ^ fw), a[0], a[1], a[2], a[3]);
        sts128(wrb_s + 16 * ((uint32_t)q ^ fw), b[0], b[1], b[2], b[3]);
    }
}

// A chunk without payload bits holds nothing but the stream's fill symbol, the symbol with the all-zero code:
// the first symbol of the table entry for a window of zeros.
static __device__ __noinline__ void fill_quads(uint32_t lut_s, uint32_t pairs, uint32_t wr_s, uint32_t fw, uint32_t n_quads)
{
    const uint32_t e = lds32(lut_s);
    const uint32_t word = (pairs ? (e >> 8) & 0xFFu : e >> 24) * 0x01010101u;
    for (uint32_t q = 0; q < n_quads; ++q) sts128(wr_s + 16 * (q ^ fw), word, word, word, word);
}

// The same result as decode_round one symbol at a time, from the first code of every table entry (two-symbol
// tables: symbol in bits 15..8, length in bits 27..24; one-symbol tables: symbol in bits 31..24, length in bits
// 3..0), reading the piece from global memory.  Small and slow on purpose: it serves pieces that were too long
// to stage.  Returns the new position.
static __device__ __noinline__ uint32_t decode_quads_global(uint32_t pos, const uint32_t* __restrict__ pay, uint32_t lut_s, uint32_t pairs,
                                                     uint32_t wr_s, uint32_t fw, uint32_t n_quads, uint32_t lim)
{
    for (uint32_t i = 0; i < 4 * n_quads; ++i) {
        uint32_t word = 0, win = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            if ((k & 1) == 0) win = window_g(pay, pos, lim);
            const uint32_t e = lut_peek(win, lut_s);
            const uint32_t l = pairs ? (e >> 24) & 15 : e & 15, sy = pairs ? (e >> 8) & 0xFF : e >> 24;
            win = __funnelshift_l(0, win, l);
            pos += l;
            word |= sy << (8 * k);
        }
        sts32(wr_s + 16 * ((i >> 2) ^ fw) + 4 * (i & 3), word);
    }
    return pos;
}

// ------------------------------------------------------------------------------------------------
// chunk loop of one warp, specialised for which streams are Huffman-coded
// ------------------------------------------------------------------------------------------------

struct DecShared {                   // what the block's prologue leaves for the chunk loop
    uint32_t pairs0, pairs1;         // the stream's table yields two symbols per lookup
    unsigned long long sec0, sec1;   // byte offsets of the streams' sections
    unsigned long long payload_off, payload_bytes;
    uint32_t pool_bytes;             // bytes of this warp's pool
};

template <bool V> struct BoolTag { static constexpr bool value = V; };

// The warp waits for the copies on its two mbarriers (those it has on the way); false when a wait gave up.  The phases count only
// where every lane has seen the copies land: all lanes keep the same parity.
__device__ __forceinline__ bool pieces_here(const bool on0, const bool on1, uint64_t* const bar, uint32_t& parity0, uint32_t& parity1, const uint32_t spin_limit)
{
    bool late = false;
    if (on0) late = !mbar_wait(&bar[0], parity0, spin_limit);
    if (on1) late = !mbar_wait(&bar[1], parity1, spin_limit) || late;
    if (__any_sync(0xFFFFFFFFu, late)) return false;
    if (on0) parity0 ^= 1;
    if (on1) parity1 ^= 1;
    return true;
}

// Whether one of the block's copies did not land within the limit.  The block then takes no more parts: the copy may still write into
// the pools, and the phases of its mbarrier are not known any more.
__device__ __forceinline__ uint32_t& block_lost()
{
    __shared__ uint32_t s_lost;
    return s_lost;
}
// The wait of settle; out of line, since it is rare (in line it took registers of the chunk loops: 15 GB of BF16 weights 4.56 ms, so 4.51;
// of deltas 10.28 and 10.09).  False when the copy did not land.
static __device__ __noinline__ bool settle_wait(uint64_t* const bar, const uint32_t parity, const uint32_t spin_limit)
{
    const bool landed = mbar_wait(bar, parity, spin_limit);
    if (__all_sync(0xFFFFFFFFu, landed)) return true;
    if ((threadIdx.x & 31) == 0) block_lost() = 1;
    return false;
}
// A copy that was started and not waited for (the warp's loop ended early, on damage or on a wait that gave up) must land before the
// block goes on or leaves, and its phase counts: the warp's next wait on the mbarrier is for the next phase.
__device__ __forceinline__ bool settle(const bool flying, uint64_t* const bar, uint32_t& parity, const uint32_t spin_limit)
{
    if (!flying) return true;                                    // (the same in every lane)
    if (!settle_wait(bar, parity, spin_limit)) return false;
    parity ^= 1;
    return true;
}

// PPL = 16-symbol parts each lane merges per round = R / 16, R in {16, 32, 64}.
// SIDE: the streams of chunks with both streams coded are decoded side by side.
template <int FMT, int PPL, bool H0, bool H1, bool XOR, bool SIDE>
__device__ __forceinline__ uint32_t run_chunks(const DecParams& P, const DecShared& S, uint8_t* pool, uint64_t* bar,
                                               uint32_t first_end0, uint32_t first_off0,
                                               uint32_t c, const uint32_t c_end, const uint32_t step,
                                               uint32_t& parity0, uint32_t& parity1)
{
    constexpr uint32_t R = 16 * PPL;
    constexpr uint32_t kLog = PPL == 4 ? 2 : PPL == 2 ? 1 : 0;
    constexpr uint32_t kRowsBytes = 512 * PPL;                 // one stream's decoded symbols of a warp and round
    constexpr uint32_t kHuff = (H0 ? 1u : 0u) + (H1 ? 1u : 0u);
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t sub_w = P.chunk_bytes <= 8192 ? 2u : 4u;
    const uint64_t tab_chunk = 256, tab_sub = 256 + (((uint64_t)4 * P.n_chunks + 15) & ~15ull);
    const uint8_t* sec0 = P.comp + S.sec0;
    const uint8_t* sec1 = P.comp + S.sec1;
    const uint32_t lut0_s = smem_u32(block_luts()), lut1_s = lut0_s + kLutBytes;
    const uint8_t* payload = P.comp + S.payload_off;
    const uint64_t payload16 = S.payload_bytes >> 4;

    // pool: symbols of stream 0 (if coded), of stream 1 (if coded), then one staging slot per coded stream
    constexpr uint32_t rows1_off = H0 ? kRowsBytes : 0;
    constexpr uint32_t slots_off = rows1_off + (H1 ? kRowsBytes : 0);
    const uint32_t slot_room = S.pool_bytes > slots_off ? S.pool_bytes - slots_off : 0u;
    const uint32_t slot_bytes = kHuff ? (slot_room / (kHuff ? kHuff : 1)) & ~15u : 0u;
    const uint32_t rows0_s = smem_u32(pool), rows1_s = rows0_s + rows1_off;
    // A piece that does not fit its slot is staged in slices instead, lane by lane (where the geometry allows:
    // subchunks of a multiple of kSliceSyms symbols, slots of at least 32 lane slots): the stream's slot becomes 32
    // lane slots of kSliceSlot bytes, and every kSliceSyms symbols each lane copies the next kSliceBytes of its own
    // subchunk there.  The copy is waited for on the spot, so this is slower than staging the piece as a whole,
    // and much faster than decoding it from global memory.
    const bool can_slice = P.sliced && slot_bytes >= 32 * kSliceSlot;
    const uint32_t base0_s = rows0_s + slots_off, base1_s = base0_s + (H0 ? slot_bytes : 0u);
    uint32_t slot0_s = base0_s, slot1_s = base1_s;
    bool sliced0 = false, sliced1 = false;
    constexpr uint32_t kRoundsPerSlice = kSliceSyms / R;
    // where this lane writes its quads and reads the parts it merges (see decode_round)
    const uint32_t fw = (lane >> (3 - kLog)) & (PPL - 1);
    const uint32_t wr_off = 16 * PPL * lane;
    const uint32_t rl = lane / PPL, rq = lane % PPL;
    const uint32_t rd_off = 16 * (rl * PPL + (rq ^ ((rl >> (3 - kLog)) & (PPL - 1))));   // part i: + 512 * i
    uint32_t err = 0;
    const bool out32 = ((uintptr_t)P.out & 16) == 0;           // chunks start at multiples of 1024 bytes behind it

    // this lane's parts of a round: part i covers symbols k_lane + i * k_step (+ round offset) of the chunk
    const uint32_t k_lane = rl * P.sub + rq * 16, k_step = (32 / PPL) * P.sub;
    const uint32_t n_rounds = P.sub / R;
    // every chunk but possibly the last one is complete
    const uint32_t n_full = ((uint64_t)P.n_chunks * P.cs == P.n_syms && (uint64_t)P.n_chunks * P.chunk_bytes == P.input_bytes)
                                ? P.n_chunks : P.n_chunks - 1;

    uint32_t nx_end0 = first_end0, nx_off0 = first_off0, nx_end1 = 0, nx_off1 = 0;
    if (H1 && c < c_end) {
        nx_end1 = load_sub_end(sec1 + tab_sub, sub_w, c, lane);
        nx_off1 = reinterpret_cast<const uint32_t*>(sec1 + tab_chunk)[c];
    }

    // The pieces of one chunk at a time live in the warp's staging slots.  A chunk's pieces are requested as soon
    // as the chunk before it has been decoded (the slots are free then), so the copy runs while that chunk is
    // merged and written.  State of the chunk whose pieces are in the slots or on their way:
    uint32_t end0 = 0, end1 = 0, start0 = 0, start1 = 0, piece0 = 0, piece1 = 0;
    const uint32_t* pay0_g = nullptr;
    const uint32_t* pay1_g = nullptr;
    bool staged0 = false, staged1 = false, flying0 = false, flying1 = false;
    // Sliced pieces: bits of the piece before the current slice (rel), position at the slice's start (org), and the
    // slice that is on its way: its bytes per lane (by), where it starts in the piece (at), bytes of the whole warp (tot).
    uint32_t rel0 = 0, rel1 = 0, org0 = 0, org1 = 0;
    uint32_t by0 = 0, by1 = 0, at0 = 0, at1 = 0, tot0 = 0, tot1 = 0;
    // Every lane fetches the next slice of its own subchunk, from bit rel of the piece on: 16-byte aligned, long
    // enough for kSliceSyms symbols of 12 bits plus the window's look-ahead, not past the piece's guard (with a
    // damaged payload a lane may have run past its piece: the copy still stays inside piece + guard).  The copies
    // are waited for when the slice is needed; until then the warp merges and writes the symbols it has.
    auto issue_slices = [&](const bool more0, const bool more1) {
        by0 = by1 = 0;
        at0 = min(16 * (rel0 >> 7), piece0); at1 = min(16 * (rel1 >> 7), piece1);
        if (H0 && sliced0 && more0) by0 = min(kSliceBytes, piece0 + 16 - at0);
        if (H1 && sliced1 && more1) by1 = min(kSliceBytes, piece1 + 16 - at1);
        tot0 = H0 ? __reduce_add_sync(0xFFFFFFFFu, by0) : 0u;
        tot1 = H1 ? __reduce_add_sync(0xFFFFFFFFu, by1) : 0u;
        __syncwarp();                                            // every lane is done with the previous slices
        if (tot0) flying0 = true;
        if (tot1) flying1 = true;
        if (P.skip_copy) return;
        if (lane == 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            if (tot0) mbar_expect_tx(&bar[0], tot0);
            if (tot1) mbar_expect_tx(&bar[1], tot1);
        }
        __syncwarp();
        if (by0) bulk_g2s_addr(slot0_s, reinterpret_cast<const uint8_t*>(pay0_g) + at0, by0, &bar[0]);
        if (by1) bulk_g2s_addr(slot1_s, reinterpret_cast<const uint8_t*>(pay1_g) + at1, by1, &bar[1]);
    };
    // Takes the table entries in nx_* (of chunk `cc`), checks them, starts the copies, and requests the entries
    // of the chunk after it.
    auto prepare = [&](const uint32_t cc) {
        bool ok = true;
        if (H0) {
            const uint32_t off16 = nx_off0;
            end0 = nx_end0;
            start0 = __shfl_up_sync(0xFFFFFFFFu, end0, 1);
            if (lane == 0) start0 = 0;
            const uint32_t chunk_bits = __shfl_sync(0xFFFFFFFFu, end0, 31);
            piece0 = ((chunk_bits + 127) / 128) * 16;
            ok = ok && start0 <= end0 && end0 - start0 <= P.sub * kLmax && (uint64_t)off16 + piece0 / 16 <= payload16;
            pay0_g = reinterpret_cast<const uint32_t*>(payload + 16ull * off16);
        }
        if (H1) {
            const uint32_t off16 = nx_off1;
            end1 = nx_end1;
            start1 = __shfl_up_sync(0xFFFFFFFFu, end1, 1);
            if (lane == 0) start1 = 0;
            const uint32_t chunk_bits = __shfl_sync(0xFFFFFFFFu, end1, 31);
            piece1 = ((chunk_bits + 127) / 128) * 16;
            ok = ok && start1 <= end1 && end1 - start1 <= P.sub * kLmax && (uint64_t)off16 + piece1 / 16 <= payload16;
            pay1_g = reinterpret_cast<const uint32_t*>(payload + 16ull * off16);
        }
        staged0 = staged1 = false;
        if (kHuff && !__all_sync(0xFFFFFFFFu, ok)) { err = ZC_E_CORRUPT; return; }
        // the copy takes 16 bytes more than the piece (the next piece or the guard), so window peeks stay inside
        sliced0 = H0 && can_slice && piece0 + 16 > slot_bytes;
        sliced1 = H1 && can_slice && piece1 + 16 > slot_bytes;
        slot0_s = base0_s + (sliced0 ? lane * kSliceSlot : 0u);
        slot1_s = base1_s + (sliced1 ? lane * kSliceSlot : 0u);
        if (sliced0) staged0 = true;
        if (sliced1) staged1 = true;
        if (sliced0 || sliced1) {
            rel0 = start0; rel1 = start1;
            issue_slices(end0 > start0, end1 > start1);          // lanes that have bits at all
        }
        if (H0 && piece0 + 16 <= slot_bytes) {
            staged0 = flying0 = true;
            if (lane == 0 && !P.skip_copy) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_expect_tx(&bar[0], piece0 + 16);
                bulk_g2s(pool + slots_off, pay0_g, piece0 + 16, &bar[0]);
            }
        }
        if (H1 && piece1 + 16 <= slot_bytes) {
            staged1 = flying1 = true;
            if (lane == 0 && !P.skip_copy) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_expect_tx(&bar[1], piece1 + 16);
                bulk_g2s(pool + slots_off + (H0 ? slot_bytes : 0), pay1_g, piece1 + 16, &bar[1]);
            }
        }
        const uint32_t cn = cc + step;
        if (cn < c_end) {
            if (H0) { nx_end0 = load_sub_end(sec0 + tab_sub, sub_w, cn, lane);
                      nx_off0 = reinterpret_cast<const uint32_t*>(sec0 + tab_chunk)[cn]; }
            if (H1) { nx_end1 = load_sub_end(sec1 + tab_sub, sub_w, cn, lane);
                      nx_off1 = reinterpret_cast<const uint32_t*>(sec1 + tab_chunk)[cn]; }
        }
    };
    if (c < c_end) prepare(c);

    for (; c < c_end && !err; c += step) {
        // ---- the chunk; FULL: a complete chunk, every lane has P.sub symbols ----
        auto body = [&](auto full_tag) {
            constexpr bool FULL = decltype(full_tag)::value;
            const uint64_t c_lo = (uint64_t)c * P.cs;
            const uint32_t c_syms = FULL ? P.cs : (uint32_t)min((uint64_t)P.cs, P.n_syms - c_lo);
            const uint32_t out_bytes = FULL ? P.chunk_bytes : (uint32_t)min((uint64_t)P.chunk_bytes, P.input_bytes - 2 * c_lo);
            const uint32_t lo_sym = lane * P.sub;
            const uint32_t n_my = FULL ? P.sub : (lo_sym < c_syms ? min(P.sub, c_syms - lo_sym) : 0u);
            const uint32_t last_r = FULL ? n_rounds - 1 : (min(c_syms, P.sub) - 1) / R;   // lane 0 has the most symbols
            const uint8_t* raw0 = sec0 + c_lo + k_lane;             // my first part's bytes in a raw stream
            const uint8_t* raw1 = sec1 + c_lo + k_lane;
            uint8_t* dst_lane = P.out + 2 * c_lo + 2 * k_lane;      // two element bytes per symbol in every format
            LaneBits L0{}, L1{};                                 // (.pos also where the piece is read from global memory)
            uint32_t lim0 = 0, lim1 = 0;
            for (uint32_t r = 0; r <= last_r; ++r) {
                // ---- what this round is merged with (raw stream, base tensor) travels to the L2 while it is decoded ----
#pragma unroll
                for (int i = 0; i < PPL; ++i) {
                    if (!H1 && (FULL || k_lane + i * k_step + r * R < c_syms))
                        asm volatile("prefetch.global.L2 [%0];" :: "l"(raw1 + i * k_step + r * R));
                    if (XOR && P.base && (FULL || 2 * (k_lane + i * k_step + r * R) < out_bytes))
                        asm volatile("prefetch.global.L2 [%0];" :: "l"(P.base + (dst_lane - P.out) + 2 * (i * k_step + r * R)));
                }
                if (kHuff && (sliced0 || sliced1) && r % kRoundsPerSlice == 0) {
                    // the slice requested after the previous one was used up (or, for the chunk's first one, while
                    // the chunk before was merged) is needed now
                    if (!pieces_here(tot0 != 0, tot1 != 0, bar, parity0, parity1, P.spin_limit)) { err = ZC_E_DEVICE_TIMEOUT; return; }
                    if (tot0) flying0 = false;
                    if (tot1) flying1 = false;
                    if (by0) { org0 = 8 * slot0_s + min(rel0 - 8 * at0, 127u); lane_start(L0, org0); }
                    if (by1) { org1 = 8 * slot1_s + min(rel1 - 8 * at1, 127u); lane_start(L1, org1); }
                    tot0 = tot1 = 0;
                }
                if (kHuff && r == 0) {
                    if (!pieces_here(H0 && staged0 && !sliced0, H1 && staged1 && !sliced1, bar, parity0, parity1, P.spin_limit)) { err = ZC_E_DEVICE_TIMEOUT; return; }
                    if (!sliced0) flying0 = false;
                    if (!sliced1) flying1 = false;
                    // staged: positions count from shared address 0; from global memory: from the piece, and the last
                    // readable word pair ends with the guard (piece + 16 bytes)
                    if (H0 && !sliced0) { if (staged0) lane_start(L0, 8 * slot0_s + start0); else L0.pos = start0; lim0 = piece0 / 4 + 2; }
                    if (H1 && !sliced1) { if (staged1) lane_start(L1, 8 * slot1_s + start1); else L1.pos = start1; lim1 = piece1 / 4 + 2; }
                }
                // ---- every lane decodes R symbols of its subchunk ----
                if (kHuff) {
                    const uint32_t done = r * R;
                    // a ragged end decodes up to 15 symbols too many (from the bits that follow); they are not used
                    const uint32_t n_quads = FULL ? (uint32_t)PPL : (n_my > done ? (min(R, n_my - done) + 15) / 16 : 0u);
                    // (only in the kernels that have the registers for it)
                    constexpr bool kSideBySide = H0 && H1 && SIDE;
                    if (kSideBySide && n_quads && staged0 && staged1 && piece0 != 0 && piece1 != 0) {
                        // both streams come from staged pieces: their words are decoded side by side
                        const uint32_t wra_s = rows0_s + wr_off, wrb_s = rows1_s + wr_off;
                        if (S.pairs0) {
                            if (S.pairs1) decode_round2<2, 2, PPL, FULL>(L0, lut0_s, wra_s, L1, lut1_s, wrb_s, fw, n_quads);
                            else decode_round2<2, 1, PPL, FULL>(L0, lut0_s, wra_s, L1, lut1_s, wrb_s, fw, n_quads);
                        } else {
                            if (S.pairs1) decode_round2<1, 2, PPL, FULL>(L0, lut0_s, wra_s, L1, lut1_s, wrb_s, fw, n_quads);
                            else decode_round2<1, 1, PPL, FULL>(L0, lut0_s, wra_s, L1, lut1_s, wrb_s, fw, n_quads);
                        }
                    } else if (n_quads) {
                        if (H0) {
                            const uint32_t wr_s = rows0_s + wr_off;
                            if (piece0 == 0) fill_quads(lut0_s, S.pairs0, wr_s, fw, n_quads);   // a chunk without bits: nothing but the fill symbol
                            else if (!staged0) L0.pos = decode_quads_global(L0.pos, pay0_g, lut0_s, S.pairs0, wr_s, fw, n_quads, lim0);
                            else if (S.pairs0) decode_round<2, PPL, FULL>(L0, lut0_s, wr_s, fw, n_quads);
                            else decode_round<1, PPL, FULL>(L0, lut0_s, wr_s, fw, n_quads);
                        }
                        if (H1) {
                            const uint32_t wr_s = rows1_s + wr_off;
                            if (piece1 == 0) fill_quads(lut1_s, S.pairs1, wr_s, fw, n_quads);
                            else if (!staged1) L1.pos = decode_quads_global(L1.pos, pay1_g, lut1_s, S.pairs1, wr_s, fw, n_quads, lim1);
                            else if (S.pairs1) decode_round<2, PPL, FULL>(L1, lut1_s, wr_s, fw, n_quads);
                            else decode_round<1, PPL, FULL>(L1, lut1_s, wr_s, fw, n_quads);
                        }
                    }
                    __syncwarp();
                    if ((sliced0 || sliced1) && (r + 1) % kRoundsPerSlice == 0 && r < last_r) {
                        if (sliced0) { rel0 += L0.pos - org0; org0 = L0.pos; }
                        if (sliced1) { rel1 += L1.pos - org1; org1 = L1.pos; }
                        issue_slices(n_my > (r + 1) * R, n_my > (r + 1) * R);
                    }
                    if (r == last_r) {
                        // Every lane must have consumed exactly the bits of its subchunk (a ragged end decodes up to
                        // fifteen symbols too many, and a lane without symbols took no slice: nothing but its table entry can
                        // be wrong).  Anything else means the payload does not belong to the tables.  (Giving the lanes without
                        // symbols a slice origin of their own took a register of the chunk loop: 15 GB of BF16 5.05 -> 5.27 ms.)
                        bool good = true;
                        if (H0) {
                            const uint32_t used = sliced0 ? rel0 + L0.pos - org0 : L0.pos - (staged0 ? 8 * slot0_s : 0u);
                            good = good && (FULL ? used == end0 : n_my ? used - end0 <= 15 * kLmax : start0 == end0);
                        }
                        if (H1) {
                            const uint32_t used = sliced1 ? rel1 + L1.pos - org1 : L1.pos - (staged1 ? 8 * slot1_s : 0u);
                            good = good && (FULL ? used == end1 : n_my ? used - end1 <= 15 * kLmax : start1 == end1);
                        }
                        if (!__all_sync(0xFFFFFFFFu, good)) err = ZC_E_CORRUPT;
                        // the slots are free: the next chunk's pieces travel while this round is merged and written
                        if (!err && c + step < c_end) prepare(c + step);
                    }
                }
                // ---- cooperative merge: a part covers 16 symbols = 32 output bytes ----
#pragma unroll
                for (int i = 0; i < PPL; ++i) {
                    const uint32_t k = k_lane + i * k_step + r * R;
                    if ((!FULL && k >= c_syms)) continue;
                    uint32_t e[4], m[4];
                    if (H0) {
                        const uint4 v = lds128(rows0_s + rd_off + 512 * i);
                        e[0] = v.x; e[1] = v.y; e[2] = v.z; e[3] = v.w;
                    } else {
                        const uint4 v = ld_nc_v4(raw0 + i * k_step + r * R);
                        e[0] = v.x; e[1] = v.y; e[2] = v.z; e[3] = v.w;
                    }
                    if (H1) {
                        const uint4 v = lds128(rows1_s + rd_off + 512 * i);
                        m[0] = v.x; m[1] = v.y; m[2] = v.z; m[3] = v.w;
                    } else {
                        const uint4 v = ld_nc_v4(raw1 + i * k_step + r * R);
                        m[0] = v.x; m[1] = v.y; m[2] = v.z; m[3] = v.w;
                    }
                    uint32_t o[8];
                    merge16<FMT>(e, m, o);
                    merge16<FMT>(e + 2, m + 2, o + 4);
                    uint8_t* dst = dst_lane + 2 * (i * k_step + r * R);
                    if (XOR && P.base) {                              // delta form: XOR the base tensor back in
                        const uint64_t off = (uint64_t)(dst - P.out);
                        const uint4 b0 = FULL ? ld_nc_v4(P.base + off) : load16_guarded(P.base, off, P.input_bytes);
                        const uint4 b1 = FULL ? ld_nc_v4(P.base + off + 16) : load16_guarded(P.base, off + 16, P.input_bytes);
                        o[0] ^= b0.x; o[1] ^= b0.y; o[2] ^= b0.z; o[3] ^= b0.w;
                        o[4] ^= b1.x; o[5] ^= b1.y; o[6] ^= b1.z; o[7] ^= b1.w;
                    }
                    if (FULL || 2 * k + 32 <= out_bytes) {
                        if (out32) {
                            st_cs_v8(dst, o);
                        } else {                                 // an output that is aligned to 16 bytes only
                            st_cs_v4(dst, make_uint4(o[0], o[1], o[2], o[3]));
                            st_cs_v4(dst + 16, make_uint4(o[4], o[5], o[6], o[7]));
                        }
                    } else {
#pragma unroll
                        for (int t = 0; t < 32; ++t)
                            if (2 * k + t < out_bytes) dst[t] = (uint8_t)(o[t >> 2] >> (8 * (t & 3)));
                    }
                }
                if (kHuff) __syncwarp();
            }
        };
        if (c < n_full) body(BoolTag<true>{}); else body(BoolTag<false>{});
    }
    if (!P.skip_copy && !settle(flying0, &bar[0], parity0, P.spin_limit)) err = ZC_E_DEVICE_TIMEOUT;
    if (!P.skip_copy && !settle(flying1, &bar[1], parity1, P.spin_limit)) err = ZC_E_DEVICE_TIMEOUT;
    return err;
}

// ------------------------------------------------------------------------------------------------
// the same for chunks of up to 4 KiB
// ------------------------------------------------------------------------------------------------
constexpr uint32_t kSmallChunk = 4096;

// What the chunk loop has to know of the tensor, in shared memory: read where it is needed (a chunk needs each value once or
// twice), so that it takes no registers over the loop.
struct DecView {
    const uint8_t* sec[2];           // the streams' sections: tables of a coded one, bytes of a raw one
    const uint8_t* payload;
    const uint8_t* base;
    uint8_t* out;
    unsigned long long payload16;    // payload bytes / 16
    unsigned long long tab_sub;      // where a section's subchunk ends start
    unsigned long long n_syms, input_bytes;
    uint32_t n_full;                 // complete chunks (every lane has a whole subchunk)
};

// Merges 16 symbols of either stream (off: where their 32 element bytes are in the tensor, room: those the chunk has from there on).
template <int FMT, bool XOR, bool FULL>
__device__ __forceinline__ void merge_part(const volatile DecView& V, uint8_t* const dst, const uint4 ev, const uint4 mv, const uint64_t off,
                                           const uint32_t room, const bool out32)
{
    uint32_t e[4], m[4], o[8];
    e[0] = ev.x; e[1] = ev.y; e[2] = ev.z; e[3] = ev.w;
    m[0] = mv.x; m[1] = mv.y; m[2] = mv.z; m[3] = mv.w;
    merge16<FMT>(e, m, o);
    merge16<FMT>(e + 2, m + 2, o + 4);
    if (XOR && V.base) {                                         // delta form: XOR the base tensor back in
        const uint8_t* const base = V.base;
        const uint4 b0 = FULL ? ld_nc_v4(base + off) : load16_guarded(base, off, V.input_bytes);
        const uint4 b1 = FULL ? ld_nc_v4(base + off + 16) : load16_guarded(base, off + 16, V.input_bytes);
        o[0] ^= b0.x; o[1] ^= b0.y; o[2] ^= b0.z; o[3] ^= b0.w;
        o[4] ^= b1.x; o[5] ^= b1.y; o[6] ^= b1.z; o[7] ^= b1.w;
    }
    if (FULL || room >= 32) {
        if (out32) {
            st_cs_v8(dst, o);
        } else {                                                 // an output that is aligned to 16 bytes only
            st_cs_v4(dst, make_uint4(o[0], o[1], o[2], o[3]));
            st_cs_v4(dst + 16, make_uint4(o[4], o[5], o[6], o[7]));
        }
    } else {
#pragma unroll
        for (int t = 0; t < 32; ++t)
            if ((uint32_t)t < room) dst[t] = (uint8_t)(o[t >> 2] >> (8 * (t & 3)));
    }
}

// The bytes of chunk cc of the base tensor travel to the L2.  One lane calls it.
__device__ __forceinline__ void prefetch_base_chunk(const volatile DecView& V, const uint32_t cc, const uint32_t chunk_bytes)
{
    const uint8_t* const base = V.base;
    const uint32_t n = cc < V.n_full ? chunk_bytes : (uint32_t)min((unsigned long long)chunk_bytes, V.input_bytes - (uint64_t)cc * chunk_bytes) & ~15u;
    if (base && n) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(base + (uint64_t)cc * chunk_bytes), "r"(n) : "memory");
}

// Neither stream coded (chunks of up to 4 KiB): nothing is decoded, the symbols are merged in address order (a complete chunk
// is a multiple of the warp's 512 symbols) and the next chunk's bytes travel to the L2 a chunk ahead.  Bound by memory.  (Dealt to the
// lanes by subchunks and without the prefetch, these containers lived on the L1, of which the pools of this kernel leave 28 KB:
// at 1, 2, 3, 4 KiB 872 MB of BF16 took 330, 294, 417, 320 us, now 303, 290, 299, 318; as a delta 453, 411, 676, 559 us, now 417, 407,
// 418, 451; 3.75 GB of FP4 elements 1.53 ms, now 1.44.  By bulk copies into the pools BF16 takes 305 us at 4 KiB, but FP4 4 % more
// at 2 and 4 KiB.)
template <int FMT, bool XOR>
__device__ __forceinline__ uint32_t run_plain(const DecParams& P, const volatile DecView& V, uint32_t c, const uint32_t c_end, const uint32_t step)
{
    const uint32_t lane = threadIdx.x & 31, cs = P.cs, chunk_bytes = P.chunk_bytes;
    const uint8_t* const sec0 = V.sec[0];
    const uint8_t* const sec1 = V.sec[1];
    uint8_t* const out = V.out;
    const uint64_t n_syms = V.n_syms, input_bytes = V.input_bytes;
    const uint32_t n_full = V.n_full;
    const bool out32 = ((uintptr_t)out & 16) == 0;
    for (; c < c_end; c += step) {
        const uint32_t next = c + step;
        if (next < c_end) {
            const uint64_t lo = (uint64_t)next * cs;             // (a raw section is padded to 16 bytes)
            const uint32_t n = next < n_full ? cs : ((uint32_t)min((uint64_t)cs, n_syms - lo) + 15u) & ~15u;
            if (lane < 2) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"((lane ? sec1 : sec0) + lo), "r"(n) : "memory");
            if (XOR && lane == 2) prefetch_base_chunk(V, next, chunk_bytes);
        }
        auto body = [&](auto full_tag) {
            constexpr bool FULL = decltype(full_tag)::value;
            const uint64_t lo = (uint64_t)c * cs + 16 * lane;    // my first part's symbols
            const uint32_t syms = FULL ? cs : (uint32_t)min((uint64_t)cs, n_syms - (uint64_t)c * cs);
            const uint32_t bytes = FULL ? chunk_bytes : (uint32_t)min((uint64_t)chunk_bytes, input_bytes - (uint64_t)c * chunk_bytes);
            const uint8_t* const e_at = sec0 + lo;
            const uint8_t* const m_at = sec1 + lo;
            uint8_t* const dst = out + 2 * lo;                 // two element bytes per symbol in every format
#pragma unroll 1
            for (uint32_t at = FULL ? 0u : 16 * lane; at < syms; at += 1024) {   // two parts at a time, 512 symbols apart
                const bool two = at + 512 < syms;
                const uint32_t k = at - (FULL ? 0u : 16 * lane);
                uint4 e1{}, m1{};
                const uint4 e0 = ld_nc_v4(e_at + k), m0 = ld_nc_v4(m_at + k);
                if (two) { e1 = ld_nc_v4(e_at + k + 512); m1 = ld_nc_v4(m_at + k + 512); }
                merge_part<FMT, XOR, FULL>(V, dst + 2 * k, e0, m0, 2 * (lo + k), bytes - (32 * lane + 2 * k), out32);
                if (two) merge_part<FMT, XOR, FULL>(V, dst + 2 * k + 1024, e1, m1, 2 * (lo + k) + 1024, bytes - (32 * lane + 2 * k + 1024), out32);
            }
        };
        if (c < n_full) body(BoolTag<true>{}); else body(BoolTag<false>{});
    }
    return ZC_OK;
}

// Chunks of up to 4 KiB are decoded as run_chunks does it, but everything a chunk needs comes by bulk copies: its pieces,
// staged whole, and the bytes of a raw stream, so that the merge reads both streams from shared memory.  Both are requested as
// soon as the chunk before has been decoded; the raw bytes of 4 KiB chunks, for which the block's memory has one buffer per
// warp, when that has been written.  Subchunks of 32 and 64 symbols are one round, their addresses immediates.
__host__ __device__ constexpr uint32_t small_raw_buffers(uint32_t ppl) { return ppl == 4 ? 1u : 2u; }   // (ppl 4: 4 KiB)

template <int FMT, int PPL, bool H0, bool H1, bool XOR, bool SIDE>
__device__ __forceinline__ uint32_t run_small(const DecParams& P, const volatile DecView& V, const uint32_t pairs0, const uint32_t pairs1,
                                              uint8_t* const pool, const uint32_t pool_bytes, uint64_t* const bar,
                                              uint32_t nx_end0, uint32_t nx_off0,
                                              uint32_t c, const uint32_t c_end, const uint32_t step,
                                              uint32_t& parity0, uint32_t& parity1)
{
    constexpr uint32_t R = 16 * PPL;
    constexpr uint32_t kLog = PPL == 4 ? 2 : PPL == 2 ? 1 : 0;
    constexpr uint32_t kRowsBytes = 512 * PPL;
    constexpr uint32_t kHuff = (H0 ? 1u : 0u) + (H1 ? 1u : 0u);
    static_assert(kHuff != 0, "containers without a coded stream: run_plain");
    constexpr bool kCopyRaw = kHuff == 1;                        // one coded stream, one raw
    constexpr int kRaw = H0 ? 1 : 0;                             // the raw one, and its mbarrier
    constexpr uint32_t kRawBufs = small_raw_buffers(PPL);
    // 4 KiB chunks with one coded stream look ahead: the next chunk's table entries are taken and checked before a chunk is decoded,
    // and where both pieces fit half a slot they lie side by side and the next one's copy is requested then, too, not when the
    // slot is free.  (872 MB of BF16 weights 303 -> 283 us, of FP8 weights 372 -> 359 us.  With both streams coded the registers
    // for two more pieces spill: 436 MB of deltas 345 -> 356 us; chunks up to 3 KiB gain nothing.)
    constexpr bool kAhead = kHuff == 1 && PPL == 4;
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t sub = PPL > 1 ? R : P.sub, cs = 32 * sub, chunk_bytes = 2 * cs, n_rounds = PPL > 1 ? 1u : sub / R;
    const uint32_t lut0_s = smem_u32(block_luts()), lut1_s = lut0_s + kLutBytes;

    // pool: symbols of stream 0 (if coded), of stream 1 (if coded), raw bytes of a chunk, one staging slot per coded stream
    constexpr uint32_t rows1_off = H0 ? kRowsBytes : 0, raw_off = kHuff * kRowsBytes;
    const uint32_t slots_off = raw_off + (kCopyRaw ? kRawBufs * cs : 0u);
    const uint32_t slot_bytes = ((pool_bytes - slots_off) / kHuff) & ~15u;
    const uint32_t rows0_s = smem_u32(pool), rows1_s = rows0_s + rows1_off;
    uint32_t raw_s = rows0_s + raw_off;                          // of the chunk that is merged next
    const uint32_t slot0_s = rows0_s + slots_off, slot1_s = slot0_s + (H0 ? slot_bytes : 0u);
    // where this lane writes its quads and reads the parts it merges (see decode_round)
    const uint32_t fw = (lane >> (3 - kLog)) & (PPL - 1);
    const uint32_t wr_off = 16 * PPL * lane;
    const uint32_t rl = lane / PPL, rq = lane % PPL;
    const uint32_t rd_off = 16 * (rl * PPL + (rq ^ ((rl >> (3 - kLog)) & (PPL - 1))));   // part i: + 512 * i
    const uint32_t k_lane = rl * sub + rq * 16, k_step = (32 / PPL) * sub;
    const bool out32 = ((uintptr_t)V.out & 16) == 0;

    uint32_t err = 0, nx_end1 = 0, nx_off1 = 0;
    // the chunk whose pieces are in the slots or on their way
    uint32_t end0 = 0, end1 = 0, start0 = 0, start1 = 0, piece0 = 0, piece1 = 0, off0 = 0, off1 = 0;
    bool staged0 = false, staged1 = false, flying0 = false, flying1 = false;
    auto load_tables = [&](const int s, const uint32_t cc, uint32_t& end, uint32_t& off) {
        const uint8_t* const sec = V.sec[s];
        end = reinterpret_cast<const uint16_t*>(sec + V.tab_sub + 64ull * cc)[lane];
        off = reinterpret_cast<const uint32_t*>(sec + 256)[cc];
    };
    auto copy = [&](const uint32_t dst_s, const uint8_t* src, const uint32_t bytes, uint64_t* b) {   // one lane calls it
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_expect_tx(b, bytes);
        bulk_g2s_addr(dst_s, src, bytes, b);
    };
    // the raw bytes of a chunk (a raw section is padded to 16 bytes)
    auto copy_raw = [&](const uint32_t dst_s, const uint32_t cc) {
        const uint64_t lo = (uint64_t)cc * cs;
        const uint32_t n = cc < V.n_full ? cs : ((uint32_t)min((unsigned long long)cs, V.n_syms - lo) + 15u) & ~15u;
        if (kRaw == 1) flying1 = true; else flying0 = true;
        if (lane == 0 && !P.skip_copy) copy(dst_s, V.sec[kRaw] + lo, n, &bar[kRaw]);
    };
    auto check = [&](const uint32_t end, const uint32_t off, uint32_t& start, uint32_t& piece) -> bool {
        start = __shfl_up_sync(0xFFFFFFFFu, end, 1);
        if (lane == 0) start = 0;
        piece = (__shfl_sync(0xFFFFFFFFu, end, 31) + 127) / 128 * 16;
        return start <= end && end - start <= sub * kLmax && (uint64_t)off + piece / 16 <= V.payload16;
    };
    // Takes the table entries in nx_* (of chunk cc), checks them, starts the copies, and requests the entries of the chunk
    // after it.  A copy takes 16 bytes more than the piece (the next piece or the guard), for the windows' look-ahead.
    // (As prefetch_base_chunk has it; but with a call of that the compiler spills in the loop of two coded streams: 15 GB of deltas 10.1 ->
    // 10.7 ms.)
    auto prefetch_base = [&](const uint32_t cc) {                // the base tensor's bytes travel to the L2
        const uint8_t* const base = V.base;
        const uint32_t n = cc < V.n_full ? chunk_bytes : (uint32_t)min((unsigned long long)chunk_bytes, V.input_bytes - (uint64_t)cc * chunk_bytes) & ~15u;
        if (lane == 0 && base && n)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(base + (uint64_t)cc * chunk_bytes), "r"(n) : "memory");
    };
    auto prepare = [&](const uint32_t cc) {
        bool ok = true;
        if (H0) { end0 = nx_end0; off0 = nx_off0; ok = check(end0, off0, start0, piece0); }
        if (H1) { end1 = nx_end1; off1 = nx_off1; ok = check(end1, off1, start1, piece1) && ok; }
        staged0 = staged1 = false;
        if (!__all_sync(0xFFFFFFFFu, ok)) { err = ZC_E_CORRUPT; return; }
        if (H0 && piece0 + 16 <= slot_bytes) {
            staged0 = flying0 = true;
            if (lane == 0 && !P.skip_copy) copy(slot0_s, V.payload + 16ull * off0, piece0 + 16, &bar[0]);
        }
        if (H1 && piece1 + 16 <= slot_bytes) {
            staged1 = flying1 = true;
            if (lane == 0 && !P.skip_copy) copy(slot1_s, V.payload + 16ull * off1, piece1 + 16, &bar[1]);
        }
        if (XOR) prefetch_base(cc);
        if (cc + step < c_end) {
            if (H0) load_tables(0, cc + step, nx_end0, nx_off0);
            if (H1) load_tables(1, cc + step, nx_end1, nx_off1);
        }
    };
    // kAhead: the coded stream's next piece (see prepare for the present one), where it lies, and where the present one does
    uint32_t ne_start = 0, ne_end = 0, ne_bytes = 0, ne_off = 0, ne_at = 0, at_s = H0 ? slot0_s : slot1_s;
    auto ask_next = [&](const uint32_t dst_s) {
        ne_at = dst_s;
        if (H0) flying0 = true; else flying1 = true;
        if (lane == 0 && !P.skip_copy) copy(dst_s, V.payload + 16ull * ne_off, ne_bytes + 16, &bar[H0 ? 0 : 1]);
    };
    auto look_ahead = [&](const uint32_t cc) {
        ne_end = H0 ? nx_end0 : nx_end1; ne_off = H0 ? nx_off0 : nx_off1; ne_at = 0;
        const bool ok = check(ne_end, ne_off, ne_start, ne_bytes);
        if (!__all_sync(0xFFFFFFFFu, ok)) { err = ZC_E_CORRUPT; return; }
        const uint32_t half = slot_bytes / 2 & ~15u, first_s = H0 ? slot0_s : slot1_s;
        if (ne_bytes + 16 <= half && (H0 ? piece0 : piece1) + 16 <= half) ask_next(at_s == first_s ? first_s + half : first_s);
        if (XOR) prefetch_base(cc);
        if (cc + step < c_end) {
            if (H0) load_tables(0, cc + step, nx_end0, nx_off0);
            if (H1) load_tables(1, cc + step, nx_end1, nx_off1);
        }
    };
    // the next piece's copy, if it had to wait for the slot; and it becomes the present one (ne_at 0: it is not staged)
    auto ask_late = [&]() {
        if (!ne_at && ne_bytes + 16 <= slot_bytes) ask_next(H0 ? slot0_s : slot1_s);
    };
    auto adopt = [&]() {
        if (H0) { start0 = ne_start; end0 = ne_end; piece0 = ne_bytes; off0 = ne_off; staged0 = ne_at != 0; }
        if (H1) { start1 = ne_start; end1 = ne_end; piece1 = ne_bytes; off1 = ne_off; staged1 = ne_at != 0; }
        if (ne_at) at_s = ne_at;
    };
    // One-symbol tables: the next chunk's pieces travel to the L2 while a chunk is decoded (their table entries are in nx_*), so that
    // the copies are quicker than the merge they hide behind (436 MB of deltas 350 -> 345 us; with two-symbol tables it is more
    // instructions than it saves: BF16 weights 297 -> 302 us).
    auto prefetch_next = [&]() {
        if (lane != 31) return;                                  // its subchunk's end is the piece's
        const uint32_t n0 = (nx_end0 + 127) / 128, n1 = (nx_end1 + 127) / 128;
        if (H0 && n0 && (uint64_t)nx_off0 + n0 <= V.payload16)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(V.payload + 16ull * nx_off0), "r"(16 * n0) : "memory");
        if (H1 && n1 && (uint64_t)nx_off1 + n1 <= V.payload16)
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(V.payload + 16ull * nx_off1), "r"(16 * n1) : "memory");
    };
    auto other_raw = [&]() { return rows0_s + raw_off + (raw_s == rows0_s + raw_off ? cs : 0u); };
    auto wait_raw = [&]() -> bool {
        uint32_t& parity = kRaw == 1 ? parity1 : parity0;
        const bool here = mbar_wait(&bar[kRaw], parity, P.spin_limit);
        if (!__all_sync(0xFFFFFFFFu, here)) { err = ZC_E_DEVICE_TIMEOUT; return false; }
        parity ^= 1;
        if (kRaw == 1) flying1 = false; else flying0 = false;
        return true;
    };
    if (c < c_end) {
        if (H1) load_tables(1, c, nx_end1, nx_off1);
        prepare(c);
        if (kCopyRaw && !err) copy_raw(raw_s, c);
    }

    for (; c < c_end && !err; c += step) {
        // ---- the chunk; FULL: a complete chunk, every lane has `sub` symbols ----
        auto body = [&](auto full_tag) {
            constexpr bool FULL = decltype(full_tag)::value;
            const uint64_t c_lo = (uint64_t)c * cs;
            const uint32_t c_syms = FULL ? cs : (uint32_t)min((unsigned long long)cs, V.n_syms - c_lo);
            const uint32_t out_bytes = FULL ? chunk_bytes : (uint32_t)min((unsigned long long)chunk_bytes, V.input_bytes - 2 * c_lo);
            const uint32_t lo_sym = lane * sub;
            const uint32_t n_my = FULL ? sub : (lo_sym < c_syms ? min(sub, c_syms - lo_sym) : 0u);
            const uint32_t last_r = FULL ? n_rounds - 1 : (min(c_syms, sub) - 1) / R;         // lane 0 has the most symbols
            LaneBits L0{}, L1{};                                 // (.pos also where the piece is read from global memory)
            for (uint32_t r = 0; r <= last_r; ++r) {
                if (r == 0) {
                    if (!pieces_here(H0 && staged0, H1 && staged1, bar, parity0, parity1, P.spin_limit)) { err = ZC_E_DEVICE_TIMEOUT; return; }
                    if (H0) flying0 = false;
                    if (H1) flying1 = false;
                    if (H0) { if (staged0) lane_start(L0, 8 * (kAhead ? at_s : slot0_s) + start0); else L0.pos = start0; }
                    if (H1) { if (staged1) lane_start(L1, 8 * (kAhead ? at_s : slot1_s) + start1); else L1.pos = start1; }
                    if (kAhead && c + step < c_end) look_ahead(c + step);
                    if (!kAhead && ((H0 && !pairs0) || (H1 && !pairs1)) && c + step < c_end) prefetch_next();
                }
                // ---- every lane decodes R symbols of its subchunk ----
                if (kHuff) {
                    const uint32_t done = r * R;
                    // a ragged end decodes up to 15 symbols too many (from the bits that follow); they are not used
                    const uint32_t n_quads = FULL ? (uint32_t)PPL : (n_my > done ? (min(R, n_my - done) + 15) / 16 : 0u);
                    constexpr bool kSideBySide = H0 && H1 && SIDE;           // (only in the kernels that have the registers for it)
                    const uint32_t wr0_s = rows0_s + wr_off, wr1_s = rows1_s + wr_off;
                    if (kSideBySide && n_quads && staged0 && staged1 && piece0 != 0 && piece1 != 0) {
                        if (pairs0) {
                            if (pairs1) decode_round2<2, 2, PPL, FULL>(L0, lut0_s, wr0_s, L1, lut1_s, wr1_s, fw, n_quads);
                            else decode_round2<2, 1, PPL, FULL>(L0, lut0_s, wr0_s, L1, lut1_s, wr1_s, fw, n_quads);
                        } else {
                            if (pairs1) decode_round2<1, 2, PPL, FULL>(L0, lut0_s, wr0_s, L1, lut1_s, wr1_s, fw, n_quads);
                            else decode_round2<1, 1, PPL, FULL>(L0, lut0_s, wr0_s, L1, lut1_s, wr1_s, fw, n_quads);
                        }
                    } else if (n_quads) {
                        // (the last word pair that may be read from global memory ends with the guard, 16 bytes behind the piece)
                        if (H0) {
                            if (piece0 == 0) fill_quads(lut0_s, pairs0, wr0_s, fw, n_quads);   // a chunk without bits: nothing but the fill symbol
                            else if (!staged0) L0.pos = decode_quads_global(L0.pos, reinterpret_cast<const uint32_t*>(V.payload + 16ull * off0), lut0_s, pairs0, wr0_s, fw, n_quads, piece0 / 4 + 2);
                            else if (pairs0) decode_round<2, PPL, FULL>(L0, lut0_s, wr0_s, fw, n_quads);
                            else decode_round<1, PPL, FULL>(L0, lut0_s, wr0_s, fw, n_quads);
                        }
                        if (H1) {
                            if (piece1 == 0) fill_quads(lut1_s, pairs1, wr1_s, fw, n_quads);
                            else if (!staged1) L1.pos = decode_quads_global(L1.pos, reinterpret_cast<const uint32_t*>(V.payload + 16ull * off1), lut1_s, pairs1, wr1_s, fw, n_quads, piece1 / 4 + 2);
                            else if (pairs1) decode_round<2, PPL, FULL>(L1, lut1_s, wr1_s, fw, n_quads);
                            else decode_round<1, PPL, FULL>(L1, lut1_s, wr1_s, fw, n_quads);
                        }
                    }
                    __syncwarp();
                    if (kCopyRaw && kRawBufs == 2 && r == 0 && !wait_raw()) return;
                    if (r == last_r) {
                        // Every lane must have consumed exactly the bits of its subchunk (a ragged end decodes up to fifteen
                        // symbols too many).  Anything else means the payload does not belong to the tables.
                        bool good = true;
                        if (H0) {
                            const uint32_t used = L0.pos - (staged0 ? 8 * (kAhead ? at_s : slot0_s) : 0u);
                            good = good && (FULL ? used == end0 : n_my ? used - end0 <= 15 * kLmax : start0 == end0);
                        }
                        if (H1) {
                            const uint32_t used = L1.pos - (staged1 ? 8 * (kAhead ? at_s : slot1_s) : 0u);
                            good = good && (FULL ? used == end1 : n_my ? used - end1 <= 15 * kLmax : start1 == end1);
                        }
                        if (!__all_sync(0xFFFFFFFFu, good)) err = ZC_E_CORRUPT;
                        // the slots are free: the next chunk's pieces travel while this round is merged and written
                        if (!err && c + step < c_end) {
                            if (kAhead) ask_late(); else prepare(c + step);
                            if (kCopyRaw && kRawBufs == 2 && !err) copy_raw(other_raw(), c + step);
                        }
                    }
                }
                if (kCopyRaw && kRawBufs == 1 && r == 0 && !wait_raw()) return;
                // ---- cooperative merge: a part covers 16 symbols = 32 output bytes ----
                uint8_t* const dst0 = V.out + 2 * c_lo + 2 * (k_lane + r * R);   // two element bytes per symbol in every format
#pragma unroll
                for (int i = 0; i < PPL; ++i) {
                    const uint32_t k = k_lane + i * k_step + r * R;
                    if ((!FULL && k >= c_syms)) continue;
                    uint32_t e[4], m[4];
                    {
                        const uint4 v = H0 ? lds128(rows0_s + rd_off + 512 * i) : lds128(raw_s + k);
                        e[0] = v.x; e[1] = v.y; e[2] = v.z; e[3] = v.w;
                    }
                    {
                        const uint4 v = H1 ? lds128(rows1_s + rd_off + 512 * i) : lds128(raw_s + k);
                        m[0] = v.x; m[1] = v.y; m[2] = v.z; m[3] = v.w;
                    }
                    uint32_t o[8];
                    merge16<FMT>(e, m, o);
                    merge16<FMT>(e + 2, m + 2, o + 4);
                    uint8_t* const dst = dst0 + 2 * (i * k_step);
                    if (XOR && V.base) {                              // delta form: XOR the base tensor back in
                        const uint8_t* const base = V.base;
                        const uint64_t off = 2 * (c_lo + k);
                        const uint4 b0 = FULL ? ld_nc_v4(base + off) : load16_guarded(base, off, V.input_bytes);
                        const uint4 b1 = FULL ? ld_nc_v4(base + off + 16) : load16_guarded(base, off + 16, V.input_bytes);
                        o[0] ^= b0.x; o[1] ^= b0.y; o[2] ^= b0.z; o[3] ^= b0.w;
                        o[4] ^= b1.x; o[5] ^= b1.y; o[6] ^= b1.z; o[7] ^= b1.w;
                    }
                    if (FULL || 2 * k + 32 <= out_bytes) {
                        if (out32) {
                            st_cs_v8(dst, o);
                        } else {                                 // an output that is aligned to 16 bytes only
                            st_cs_v4(dst, make_uint4(o[0], o[1], o[2], o[3]));
                            st_cs_v4(dst + 16, make_uint4(o[4], o[5], o[6], o[7]));
                        }
                    } else {
#pragma unroll
                        for (int t = 0; t < 32; ++t)
                            if (2 * k + t < out_bytes) dst[t] = (uint8_t)(o[t >> 2] >> (8 * (t & 3)));
                    }
                }
                __syncwarp();
            }
            if (kCopyRaw && kRawBufs == 1 && !err && c + step < c_end) copy_raw(raw_s, c + step);   // everybody has read this chunk's
            if (kCopyRaw && kRawBufs == 2) raw_s = other_raw();
            if (kAhead && !err && c + step < c_end) adopt();
        };
        if (c < V.n_full) body(BoolTag<true>{}); else body(BoolTag<false>{});
    }
    if (!P.skip_copy && !settle(flying0, &bar[0], parity0, P.spin_limit)) err = ZC_E_DEVICE_TIMEOUT;
    if (!P.skip_copy && !settle(flying1, &bar[1], parity1, P.spin_limit)) err = ZC_E_DEVICE_TIMEOUT;
    return err;
}

// ------------------------------------------------------------------------------------------------
// the kernel
// ------------------------------------------------------------------------------------------------
// PPL = 16-symbol parts each lane merges per round = R / 16, R in {16, 32, 64}.

struct DecSmem {                     // the block's shared memory, carved up once per kernel
    uint32_t* lut0;                  // decode table of stream 0
    uint32_t* lut1;                  // decode table of stream 1
    uint32_t* scratch;
    uint8_t* pools;                  // all warps' pools
    uint8_t* pool;                   // this warp's pool
    uint64_t* bar;                   // this warp's two mbarriers
};

__device__ __forceinline__ DecSmem carve_smem(uint8_t* smem, uint32_t pool_bytes, uint32_t active)
{
    const uint32_t warp = threadIdx.x >> 5, n_warps = blockDim.x >> 5;
    DecSmem m;
    m.lut0 = block_luts();
    m.lut1 = m.lut0 + kLutEntries;
    m.scratch = reinterpret_cast<uint32_t*>(smem);
    uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kScratchBytes);
    m.pools = reinterpret_cast<uint8_t*>(bars + 2 * n_warps);
    m.pool = m.pools + (size_t)min(warp, active - 1) * pool_bytes;
    m.bar = bars + 2 * warp;
    if ((threadIdx.x & 31) == 0) { mbar_init(&m.bar[0], 1); mbar_init(&m.bar[1], 1); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    return m;
}

struct DecOpened {                   // what open_container leaves
    DecShared S;
    bool huff0, huff1;
};

struct DecHeader {                   // of the tensor whose tables the block has built, in shared memory
    uint32_t mode[2], per_lookup[2], ok;
    unsigned long long payload_off, payload_bytes, sec[2];
};
__device__ __forceinline__ DecHeader& block_header()
{
    __shared__ DecHeader s_header;
    return s_header;
}
__device__ __forceinline__ void opened_container(const DecParams& P, DecOpened& H)
{
    const DecHeader& T = block_header();
    H.huff0 = T.mode[0] == ZC_MODE_HUFF; H.huff1 = T.mode[1] == ZC_MODE_HUFF;
    H.S.pool_bytes = P.pool_bytes;
    H.S.pairs0 = H.huff0 && T.per_lookup[0] == 2;
    H.S.pairs1 = H.huff1 && T.per_lookup[1] == 2;
    H.S.sec0 = T.sec[0]; H.S.sec1 = T.sec[1];
    H.S.payload_off = T.payload_off; H.S.payload_bytes = T.payload_bytes;
}

// Checks the header against the plan and builds the decode tables of the coded streams; the whole block calls it.  Returns a
// zc_status, the same in every thread.
__device__ __forceinline__ uint32_t open_container(const DecParams& P, const DecSmem& M, DecOpened& H)
{
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t sub_w = P.chunk_bytes <= 8192 ? 2u : 4u;     // bytes per sub_end entry
    // Nearly every container has stream 0 coded, its table section right behind the header.  Its code lengths are requested
    // together with the header, and thrown away if the header says otherwise.
    uint32_t spec_len = 0;
    if (P.spec && threadIdx.x < 256) spec_len = P.comp[kHeaderBytes + threadIdx.x];
    // ---- header check against the plan ----
    __shared__ __align__(16) uint32_t s_hdr[32];
    DecHeader& T = block_header();
    if (warp == 0) {
        s_hdr[lane] = reinterpret_cast<const uint32_t*>(P.comp)[lane];      // the 128-byte header in one request
        __syncwarp();
    }
    if (threadIdx.x == 0) {
        const uint8_t* h = reinterpret_cast<const uint8_t*>(s_hdr);
        const uint32_t* h32 = s_hdr;
        const unsigned long long* h64 = reinterpret_cast<const unsigned long long*>(s_hdr);
        bool ok = h32[0] == kMagic && h[kHdrVersion] == 1 && h[kHdrVersion + 1] == 0 && h[kHdrFormat] == P.format &&
                  h[kHdrStreams] == 2 && h64[kHdrElems / 8] == P.n_elems && h32[kHdrChunkBytes / 4] == P.chunk_bytes &&
                  h32[kHdrChunks / 4] == P.n_chunks && h[kHdrLmax] == kLmax && h[kHdrGroup] == P.group && h[kHdrSubs] == kSubs &&
                  h[kHdrSubWidth] == sub_w;
        uint32_t mode[2] = {0, 0};
        for (int s = 0; s < 2 && ok; ++s) {
            const uint8_t* d = h + kHdrStream0 + kHdrStreamStride * s;
            mode[s] = d[kSdMode];
            ok = mode[s] <= 1 && reinterpret_cast<const unsigned long long*>(d)[1] == P.n_syms;
        }
        if (ok) {
            // recompute where everything must be and compare with what the header says
            uint64_t off = kHeaderBytes, sec[2] = {0, 0};
            const uint64_t tab = 256 + (((uint64_t)4 * P.n_chunks + 15) & ~15ull) + 32ull * sub_w * P.n_chunks;
            for (int s = 0; s < 2; ++s) if (mode[s] == ZC_MODE_HUFF) { sec[s] = off; off += tab; }
            for (int s = 0; s < 2; ++s) if (mode[s] == ZC_MODE_RAW) { sec[s] = off; off += (P.n_syms + 15) & ~15ull; }
            const bool any_huff = mode[0] == ZC_MODE_HUFF || mode[1] == ZC_MODE_HUFF;
            const uint64_t total = h64[kHdrTotal / 8], poff = h64[kHdrPayloadOff / 8], pbytes = h64[kHdrPayloadBytes / 8];
            ok = poff == off && (pbytes & 15) == 0 && payload_fits(P.comp_bytes, off, any_huff ? 16 : 0, pbytes, total);
            for (int s = 0; s < 2 && ok; ++s)
                ok = reinterpret_cast<const unsigned long long*>(h + kHdrStream0 + kHdrStreamStride * s)[3] == sec[s];
            T.mode[0] = mode[0]; T.mode[1] = mode[1];
            T.sec[0] = sec[0]; T.sec[1] = sec[1];
            T.payload_off = poff; T.payload_bytes = pbytes;
        }
        T.ok = ok ? 1u : 0u;
    }
    __syncthreads();
    if (!T.ok) return ZC_E_CORRUPT;

    const bool huff0 = T.mode[0] == ZC_MODE_HUFF, huff1 = T.mode[1] == ZC_MODE_HUFF;
    {
        // the warps' pools are free until the chunk loop: 8 KiB of them hold the one-symbol scratch table
        uint16_t* single = reinterpret_cast<uint16_t*>(M.pools);
        bool tables_ok = true;
        if (huff0) {
            uint32_t len = spec_len;                             // stream 0's section always starts behind the header
            if (!P.spec && threadIdx.x < 256) len = P.comp[T.sec[0] + threadIdx.x];
            tables_ok = build_lut(len, M.lut0, single, M.scratch, &T.per_lookup[0]) && tables_ok;
        }
        if (huff1) {
            uint32_t len = 0;
            if (threadIdx.x < 256) len = P.comp[T.sec[1] + threadIdx.x];
            tables_ok = build_lut(len, M.lut1, single, M.scratch, &T.per_lookup[1]) && tables_ok;
        }
        __syncthreads();
        if (!tables_ok) return ZC_E_CORRUPT;
    }
    opened_container(P, H);
    return ZC_OK;
}

// Decodes the chunks c0, c0 + step, ... (< c_end) of one tensor with this warp; the whole block calls it
// together (the header check and the table build are block-wide).  opened_before: the block has the tensor's tables already.
// Returns a zc_status, the same in every thread for the block-wide checks.
template <int FMT, int PPL, bool XOR, bool SIDE, bool SMALL>
__device__ __forceinline__ uint32_t decode_one(const DecParams& P, const DecSmem& M, const uint32_t chunk_base, const uint32_t c_end,
                                               const uint32_t block_index, const uint32_t n_blocks, const bool opened_before,
                                               uint32_t& parity0, uint32_t& parity1)
{
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    // chunk chunk_base + k goes to block k % n_blocks, warp (k / n_blocks) % P.active
    uint32_t c0 = warp < P.active ? chunk_base + block_index + warp * n_blocks : c_end, step = n_blocks * P.active;
    const uint32_t sub_w = P.chunk_bytes <= 8192 ? 2u : 4u;     // bytes per sub_end entry
    const uint64_t tab_chunk = 256, tab_sub = 256 + (((uint64_t)4 * P.n_chunks + 15) & ~15ull);
    // this warp's first table entries, on the guess that stream 0 is coded (see open_container)
    uint32_t spec_end = 0, spec_off = 0;
    if (P.spec && c0 < c_end) {
        spec_end = load_sub_end(P.comp + kHeaderBytes + tab_sub, sub_w, c0, lane);
        spec_off = reinterpret_cast<const uint32_t*>(P.comp + kHeaderBytes + tab_chunk)[c0];
    }
    DecOpened H;
    if (opened_before) {
        opened_container(P, H);
    } else {
        const uint32_t opened = open_container(P, M, H);
        if (opened != ZC_OK) return opened;
    }
    const bool huff0 = H.huff0, huff1 = H.huff1;
    DecShared& S = H.S;
    // Both streams coded where a warp's pool was sized for one of them (the plan does not say how many streams a container
    // codes): fewer warps then share the block's pools, each with room for both, and the chunks are dealt to those warps only.
    uint8_t* pool = M.pool;
    uint32_t pool_bytes = P.pool_bytes;
    if ((SMALL || P.sliced) && huff0 && huff1) {
        const uint32_t need = 2 * (512 * PPL + (SMALL ? P.cs + 32 : 32 * kSliceSlot));
        if (need > P.pool_bytes) {
            const uint32_t active = max(1u, P.active * P.pool_bytes / need);
            pool = M.pools + (size_t)min(warp, active - 1) * need;
            pool_bytes = need;
            c0 = warp < active ? chunk_base + block_index + warp * n_blocks : c_end;
            step = n_blocks * active;
            spec_end = spec_off = 0;
            if (c0 < c_end) {
                spec_end = load_sub_end(P.comp + kHeaderBytes + tab_sub, sub_w, c0, lane);
                spec_off = reinterpret_cast<const uint32_t*>(P.comp + kHeaderBytes + tab_chunk)[c0];
            }
        }
    }
    S.pool_bytes = pool_bytes;
    uint32_t first_end0 = spec_end, first_off0 = spec_off;
    if (huff0 && !P.spec && c0 < c_end) {
        first_end0 = load_sub_end(P.comp + S.sec0 + tab_sub, sub_w, c0, lane);
        first_off0 = reinterpret_cast<const uint32_t*>(P.comp + S.sec0 + tab_chunk)[c0];
    }
    if constexpr (SMALL) {
        __shared__ DecView s_view;
        if (threadIdx.x == 0) {
            s_view.sec[0] = P.comp + S.sec0;
            s_view.sec[1] = P.comp + S.sec1;
            s_view.payload = P.comp + S.payload_off;
            s_view.base = XOR ? P.base : nullptr;
            s_view.out = P.out;
            s_view.payload16 = S.payload_bytes >> 4;
            s_view.tab_sub = tab_sub;
            s_view.n_syms = P.n_syms;
            s_view.input_bytes = P.input_bytes;
            s_view.n_full = (uint64_t)P.n_chunks * P.cs == P.n_syms && (uint64_t)P.n_chunks * P.chunk_bytes == P.input_bytes ? P.n_chunks : P.n_chunks - 1;
        }
        __syncthreads();
        const volatile DecView& V = s_view;
        if (huff0 && !huff1) return run_small<FMT, PPL, true, false, XOR, SIDE>(P, V, S.pairs0, 0, pool, pool_bytes, M.bar, first_end0, first_off0, c0, c_end, step, parity0, parity1);
        if (!huff0 && !huff1) return run_plain<FMT, XOR>(P, V, c0, c_end, step);
        if (huff0) return run_small<FMT, PPL, true, true, XOR, SIDE>(P, V, S.pairs0, S.pairs1, pool, pool_bytes, M.bar, first_end0, first_off0, c0, c_end, step, parity0, parity1);
        return run_small<FMT, PPL, false, true, XOR, SIDE>(P, V, 0, S.pairs1, pool, pool_bytes, M.bar, 0, 0, c0, c_end, step, parity0, parity1);
    } else {
        if (huff0 && !huff1) return run_chunks<FMT, PPL, true, false, XOR, SIDE>(P, S, pool, M.bar, first_end0, first_off0, c0, c_end, step, parity0, parity1);
        if (!huff0 && !huff1) return run_chunks<FMT, PPL, false, false, XOR, SIDE>(P, S, pool, M.bar, 0, 0, c0, c_end, step, parity0, parity1);
        if (huff0) return run_chunks<FMT, PPL, true, true, XOR, SIDE>(P, S, pool, M.bar, first_end0, first_off0, c0, c_end, step, parity0, parity1);
        return run_chunks<FMT, PPL, false, true, XOR, SIDE>(P, S, pool, M.bar, 0, 0, c0, c_end, step, parity0, parity1);
    }
}

// One tensor per launch: the warps of all blocks take the chunks in turn.  FEW: see kDecFewWarps.
template <int FMT, int PPL, bool FEW, bool SMALL>
__global__ void __launch_bounds__((FEW ? kDecFewWarps : dec_block_warps<FMT, false>()) * 32, 1)
decode_kernel(const __grid_constant__ DecParams P)
{
    extern __shared__ __align__(16) uint8_t smem[];
    const DecSmem M = carve_smem(smem, P.pool_bytes, P.active);
    if (P.ctl && blockIdx.x == 0 && threadIdx.x == 0) P.ctl->call_id = P.call_id;
    uint32_t parity0 = 0, parity1 = 0;
    const uint32_t err = decode_one<FMT, PPL, false, FEW || FMT == ZC_FMT_SCALE_U8, SMALL>(P, M, P.c_begin, P.c_end, blockIdx.x, gridDim.x, false, parity0, parity1);
    if (err) raise_status(P.ctl, P.call_id, err);
}

// Launches of a few large chunks (see zc_decompress_chunks).  A lane's walk over its subchunk is serial, 1024 symbols at
// 64 KiB, and with a few chunks most of the GPU would watch.  Here a block takes a group of a chunk's subchunks, and every
// subchunk is cut into `parts` stretches of equal bits, a thread each: every thread decodes from its cut on, as if a code
// started there, up to the first code boundary at or behind the next cut, and counts.  Prefix codes find back into step within
// some codes, so where a thread ends is nearly always right even if it began inside a code; where its predecessor ended is
// where it must begin, and the threads whose beginning was wrong decode once more until nothing changes (the first is right
// from the start, so that ends after `parts` rounds whatever the payload is).  A code whose codes all have one length never
// finds back into step; its cuts are multiples of that length.  Then everybody's symbols have their place, and a last pass
// writes them.
// 1 MiB FP8 tensor, 64 KiB chunks, both streams coded: 63 us with a lane per subchunk (decode_kernel), 50 us here (its nearly
// uniform sign+mantissa code finds back into step late); one stream coded 57 against 25 us.
struct SplitBits {                   // 33 to 64 bits of the payload from the current position on, and the word behind them
    uint32_t hi, lo, n, next, addr;
};
__device__ __forceinline__ void split_start(SplitBits& B, uint32_t base_s, uint32_t at)
{
    B.addr = base_s + 4 * (at >> 5);
    const uint32_t w0 = lds32(B.addr), w1 = lds32(B.addr + 4);
    B.next = lds32(B.addr + 8);
    B.hi = __funnelshift_l(w1, w0, at);
    B.lo = w1 << (at & 31u);
    B.n = 64 - (at & 31u);
    B.addr += 12;
}
// back to 33 bits and more; two codes (of at most 12 bits, or whatever four bits of a damaged table say) fit between two calls
__device__ __forceinline__ void split_refill(SplitBits& B)
{
    if (B.n <= 32) {
        B.hi |= B.n == 32 ? 0u : B.next >> (B.n & 31u);
        B.lo = B.n == 32 ? B.next : B.next << (32 - B.n);
        B.n += 32;
        B.next = lds32(B.addr);
        B.addr += 4;
    }
}
// the table entry of the code at the current position; the position moves behind it
__device__ __forceinline__ uint32_t split_code(SplitBits& B, uint32_t lut_s, uint32_t len_shift, uint32_t& pos)
{
    const uint32_t e = lut_peek(B.hi, lut_s), l = (e >> len_shift) & 15u;
    B.hi = __funnelshift_l(B.lo, B.hi, l);
    B.lo <<= l;
    B.n -= l;
    pos += l;
    return e;
}

constexpr uint32_t kSplitThreads = 512;
// Shortest subchunk it is used for (chunks from 32 KiB on).  16 chunks of 16 KiB of BF16 weights, one stream coded, 24.6 us
// here, 18.4 us in decode_kernel; device times of longer ones, here / decode_kernel (few chunks) in us:
//                                  32 KiB, 16    32 KiB, 148   64 KiB, 16    64 KiB, 74    64 KiB, 148 chunks
//   BF16, one stream coded         20 / 24       22 / 25       21 / 43       23 / 44       26 / 43
//   scale bytes, both coded        25 / 33       28 / 36       25 / 59       28 / 61       45 / 62
//   FP8 weights, both coded        39 / 32       46 / 32       43 / 55       51 / 56       62 / 56
// The last kind's sign+mantissa code is nearly uniform and falls back into step late.  The host does not know the codes of
// the container, so the line is drawn for the others.
constexpr uint32_t kSplitMinSub = 512;

template <int FMT>
__global__ void __launch_bounds__(kSplitThreads, 1)
decode_split_kernel(const __grid_constant__ DecParams P)
{
    extern __shared__ __align__(16) uint8_t smem[];
    __shared__ uint32_t s_end[2][32], s_off[2], s_lens[2];
    const DecSmem M = carve_smem(smem, P.pool_bytes, 1);
    const uint32_t tid = threadIdx.x, lane = tid & 31;
    uint64_t* const bars = M.bar - 2 * (tid >> 5);               // the first warp's: one per stream
    if (tid < 2) s_lens[tid] = 0;
    if (P.ctl && blockIdx.x == 0 && tid == 0) P.ctl->call_id = P.call_id;
    DecOpened H;
    const uint32_t opened = open_container(P, M, H);
    if (opened != ZC_OK) { raise_status(P.ctl, P.call_id, opened); return; }
    const DecShared& S = H.S;
    const bool coded[2] = {H.huff0, H.huff1};
    const uint32_t sub_w = P.chunk_bytes <= 8192 ? 2u : 4u;
    const uint64_t tab_chunk = 256, tab_sub = 256 + (((uint64_t)4 * P.n_chunks + 15) & ~15ull);
    // my work: subchunks g_lo .. g_lo + g_subs - 1 of chunk c
    const uint32_t g_subs = 32 / P.groups, c = P.c_begin + blockIdx.x / P.groups, g_lo = (blockIdx.x % P.groups) * g_subs;
    const uint64_t c_lo = (uint64_t)c * P.cs;
    const uint32_t c_syms = c < P.c_end ? (uint32_t)min((uint64_t)P.cs, P.n_syms - c_lo) : 0u;
    const uint32_t out_bytes = c < P.c_end ? (uint32_t)min((uint64_t)P.chunk_bytes, P.input_bytes - 2 * c_lo) : 0u;
    if (c_syms <= g_lo * P.sub) return;                          // nothing of the (ragged) chunk is in my group; block-uniform
    // pool: the group's symbols of both streams, then its pieces (12 bits per symbol and 48 bytes each)
    const uint32_t g_syms = g_subs * P.sub, syms_s = smem_u32(M.pools), piece_room = ((g_syms + g_syms / 2 + 15) & ~15u) + 48;
    const uint32_t pieces_s = syms_s + 2 * g_syms;

    // ---- table entries (warp 0: stream 0, warp 1: stream 1), checked before anything is staged; code lengths in use ----
    bool bad = false;
    if (tid < 64 && coded[tid >> 5]) {
        const uint32_t s = tid >> 5;
        const uint8_t* sec = P.comp + (s == 0 ? S.sec0 : S.sec1);
        const uint32_t end = load_sub_end(sec + tab_sub, sub_w, c, lane), off16 = reinterpret_cast<const uint32_t*>(sec + tab_chunk)[c];
        uint32_t start = __shfl_up_sync(0xFFFFFFFFu, end, 1);
        if (lane == 0) start = 0;
        const uint32_t piece16 = (__shfl_sync(0xFFFFFFFFu, end, 31) + 127) / 128;
        bad = !(start <= end && end - start <= P.sub * kLmax && (uint64_t)off16 + piece16 <= (S.payload_bytes >> 4));
        s_end[s][lane] = end;
        if (lane == 0) s_off[s] = off16;
    }
    if (tid < 512 && coded[tid >> 8]) {
        const uint32_t m = __reduce_or_sync(0xFFFFFFFFu, 1u << (P.comp[(tid >> 8 ? S.sec1 : S.sec0) + (tid & 255)] & 31u));
        if (lane == 0) atomicOr(&s_lens[tid >> 8], m & ~1u);
    }
    if (__syncthreads_or(bad)) { if (tid == 0) raise_status(P.ctl, P.call_id, ZC_E_CORRUPT); return; }

    // ---- the group's part of the pieces ----
    const uint32_t bits[2] = {H.huff0 ? s_end[0][31] : 0u, H.huff1 ? s_end[1][31] : 0u};     // of the chunk
    uint32_t from_byte[2] = {0, 0};
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        if (!bits[s]) continue;
        const uint32_t lo = g_lo ? s_end[s][g_lo - 1] : 0u, hi = s_end[s][g_lo + g_subs - 1];
        from_byte[s] = (lo >> 7) * 16;
        if (tid == 0 && !P.skip_copy) {
            // 16 bytes more (bits of the next subchunk or piece, or the guard) for the window's look-ahead
            const uint32_t bytes = ((hi + 127) / 128) * 16 + 16 - from_byte[s];
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbar_expect_tx(&bars[s], bytes);
            bulk_g2s_addr(pieces_s + s * piece_room, P.comp + S.payload_off + 16ull * s_off[s] + from_byte[s], bytes, &bars[s]);
        }
    }
#pragma unroll
    for (int s = 0; s < 2; ++s)                                  // (a copy that was started must land before the block may leave: once more where the wait gave up)
        if (bits[s] && !mbar_wait(&bars[s], 0, P.spin_limit)) bad = P.skip_copy || !mbar_wait(&bars[s], 0, P.spin_limit) || bad;
    if (__syncthreads_or(bad)) { if (tid == 0) raise_status(P.ctl, P.call_id, ZC_E_DEVICE_TIMEOUT); return; }

    // ---- decode: my stream, subchunk and stretch ----
    const uint32_t per_stream = H.huff0 && H.huff1 ? kSplitThreads / 2 : kSplitThreads;
    uint32_t parts = per_stream / g_subs;                        // a power of two, at most 32 and of 64 symbols or more
    while (parts > 32 || (parts > 1 && parts * 64 > P.sub)) parts /= 2;
    const uint32_t st = H.huff0 ? tid / per_stream : 1u, q = tid % per_stream;
    if ((H.huff0 || H.huff1) && bits[st]) {
        const bool on = q < g_subs * parts;
        const uint32_t sub = g_lo + (on ? q / parts : 0u), part = q % parts;
        const uint32_t lut_s = smem_u32(st ? M.lut1 : M.lut0), pairs = st ? S.pairs1 : S.pairs0;
        const uint32_t len_shift = pairs ? 24u : 0u, sym_shift = pairs ? 8u : 24u;   // of an entry's first code
        const uint32_t piece_s = pieces_s + st * piece_room, base = 8 * from_byte[st];
        const uint32_t lo = (sub ? s_end[st][sub - 1] : 0u) - base, end_bit = s_end[st][sub] - base, len = end_bit - lo;
        const uint32_t lens = s_lens[st], unit = (lens & (lens - 1)) == 0 && lens ? (uint32_t)__ffs(lens) - 1 : 1u;
        auto cut_at = [&](const uint32_t k) { return k == parts ? end_bit : lo + len * k / parts / unit * unit; };
        const uint32_t cut = cut_at(part), stop = on ? cut_at(part + 1) : cut;
        // counts the codes from `at` to the first boundary at or behind `stop`
        uint32_t count = 0, end = cut, from = cut;
        auto walk = [&]() {
            count = 0;
            end = from;
            if (end < stop) {
                SplitBits B;
                split_start(B, piece_s, from);
                for (;;) {
                    split_code(B, lut_s, len_shift, end);
                    ++count;
                    if (end >= stop) break;
                    split_code(B, lut_s, len_shift, end);
                    ++count;
                    if (end >= stop) break;
                    split_refill(B);
                }
            }
        };
        walk();
        for (uint32_t round = 1; round < parts; ++round) {
            uint32_t should = __shfl_up_sync(0xFFFFFFFFu, end, 1);
            if (part == 0) should = lo;
            const bool wrong = on && should != from;
            if (!__any_sync(0xFFFFFFFFu, wrong)) break;
            if (wrong) { from = should; walk(); }
        }
        // symbols of the subchunk before mine
        uint32_t upto = count;
        for (uint32_t o = 1; o < parts; o <<= 1) {
            const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, upto, o);
            if (part >= o) upto += x;
        }
        // A subchunk must hold exactly its symbols and end with its last bit; anything else means that the payload does not
        // belong to the tables.
        const uint32_t first = sub * P.sub, want = c_syms > first ? min(P.sub, c_syms - first) : 0u;
        const uint32_t got = __shfl_sync(0xFFFFFFFFu, upto, lane | (parts - 1)), last = __shfl_sync(0xFFFFFFFFu, end, lane | (parts - 1));
        if (on && (got != want || last != end_bit)) {
            bad = true;
        } else if (count) {
            // the last pass: single symbols up to a word boundary, then whole words, then single symbols again
            SplitBits B;
            split_start(B, piece_s, from);
            uint32_t at = syms_s + st * g_syms + (sub - g_lo) * P.sub + upto - count, left = count, pos = 0;
            while (left) {
                if ((at & 3u) == 0 && left >= 4) {
                    uint32_t w = (split_code(B, lut_s, len_shift, pos) >> sym_shift) & 0xFFu;
                    w |= ((split_code(B, lut_s, len_shift, pos) >> sym_shift) & 0xFFu) << 8;
                    split_refill(B);
                    w |= ((split_code(B, lut_s, len_shift, pos) >> sym_shift) & 0xFFu) << 16;
                    w |= ((split_code(B, lut_s, len_shift, pos) >> sym_shift) & 0xFFu) << 24;
                    sts32(at, w);
                    at += 4;
                    left -= 4;
                } else {
                    sts8(at, (split_code(B, lut_s, len_shift, pos) >> sym_shift) & 0xFFu);
                    ++at;
                    --left;
                }
                split_refill(B);
            }
        }
    }
    if (__syncthreads_or(bad)) { if (tid == 0) raise_status(P.ctl, P.call_id, ZC_E_CORRUPT); return; }

    // ---- merge: 16 symbols of each stream, 32 output bytes per thread and step ----
    const uint8_t* raw[2] = {P.comp + S.sec0 + c_lo, P.comp + S.sec1 + c_lo};
    uint32_t fill4[2];                                           // a chunk without bits: nothing but the fill symbol
#pragma unroll
    for (int s = 0; s < 2; ++s) {
        const uint32_t e = lds32(smem_u32(s ? M.lut1 : M.lut0));
        fill4[s] = ((s ? S.pairs1 : S.pairs0) ? (e >> 8) & 0xFFu : e >> 24) * 0x01010101u;
    }
    const uint32_t k_lo = g_lo * P.sub, k_hi = min(c_syms, k_lo + g_syms);
    for (uint32_t k = k_lo + 16 * tid; k < k_hi; k += 16 * kSplitThreads) {
        uint32_t f[2][4];
#pragma unroll
        for (int s = 0; s < 2; ++s) {
            uint4 v;
            if (!coded[s]) v = ld_nc_v4(raw[s] + k);
            else if (bits[s]) v = lds128(syms_s + s * g_syms + k - k_lo);
            else v = make_uint4(fill4[s], fill4[s], fill4[s], fill4[s]);
            f[s][0] = v.x; f[s][1] = v.y; f[s][2] = v.z; f[s][3] = v.w;
        }
        uint32_t o[8];
        merge16<FMT>(f[0], f[1], o);
        merge16<FMT>(f[0] + 2, f[1] + 2, o + 4);
        uint8_t* dst = P.out + 2 * (c_lo + k);
        if (2 * k + 32 <= out_bytes) {
            st_cs_v4(dst, make_uint4(o[0], o[1], o[2], o[3]));
            st_cs_v4(dst + 16, make_uint4(o[4], o[5], o[6], o[7]));
        } else {
#pragma unroll
            for (int t = 0; t < 32; ++t)
                if (2 * k + t < out_bytes) dst[t] = (uint8_t)(o[t >> 2] >> (8 * (t & 3)));
        }
    }
}

// Many tensors per launch: the blocks take pieces of the concatenated chunk index space (see kDecMaxPieces) and go through a
// piece tensor by tensor, building a tensor's tables once for its part of it.
// XOR: the launch has base tensors (delta form); a kernel of its own so that the plain form pays nothing for it.
template <int FMT, int PPL, bool XOR, bool SMALL>
__global__ void __launch_bounds__(dec_block_warps<FMT, XOR>() * 32, 1)
decode_batch_kernel(const __grid_constant__ DecBatchParams B)
{
    extern __shared__ __align__(16) uint8_t smem[];
    const DecSmem M = carve_smem(smem, B.pool_bytes, blockDim.x >> 5);
    if (blockIdx.x == 0 && threadIdx.x == 0 && B.tensor_base == 0) B.ctl->call_id = B.call_id;
    uint32_t parity0 = 0, parity1 = 0;

    // Where the block is, in shared memory (the first warp's business; nobody keeps it in registers while decoding).
    constexpr uint32_t kNone = 0xFFFFFFFFu;
    __shared__ uint32_t s_t, s_lo, s_hi;                         // the part to decode next: chunks [s_lo, s_hi) of tensor s_t
    __shared__ uint32_t s_opened;                                // the tensor whose tables the block has
    __shared__ uint32_t s_empty, s_piece, s_g, s_g_hi, s_g_t;    // tensor to look at for an empty one; pieces taken of my slice; the rest of a piece
    if (threadIdx.x == 0) {
        s_opened = kNone;
        block_lost() = 0;
        // Block 0 first walks over the tensors, if there are any without chunks: their headers are still checked.  (The walk takes
        // 0.1 us a tensor, which the block is late for its slice: 64 BF16 pages of 129 chunks 37 us, without it 31 us.)
        s_empty = blockIdx.x == 0 && B.n_empty ? 0u : B.n_tensors;
        s_piece = s_g = s_g_hi = s_g_t = 0;
    }
    // The first warp: piece p of slice j is the block's now.
    auto enter = [&](const uint32_t p, const uint32_t j) {
        const uint32_t from = (uint32_t)((uint64_t)j * B.total / gridDim.x), len = (uint32_t)((uint64_t)(j + 1) * B.total / gridDim.x) - from;
        const uint32_t warps = blockDim.x >> 5;
        auto cut = [&](const uint32_t k) -> uint32_t {           // pieces are whole turns of the warps
            return k == B.n_pieces ? len : (uint32_t)((uint64_t)len * (k ? B.piece_end[k - 1] : 0u) >> 16) / warps * warps;
        };
        const uint32_t g = from + cut(p);
        // the last tensor that starts at or before g (tensors without chunks share their start with the next one)
        uint32_t lo = 0, hi = B.n_tensors;
        while (hi - lo > 1) {
            const uint32_t mid = (lo + hi) / 2;
            if (B.item[mid].first_chunk <= g) lo = mid; else hi = mid;
        }
        if (threadIdx.x == 0) { s_g = g; s_g_hi = from + cut(p + 1); s_g_t = lo; }
        __syncwarp();
    };
    uint32_t* const claims = reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(B.ctl) + kDecClaims);
    auto claim = [&](const uint32_t p, const uint32_t j) -> bool {
        const uint32_t bit = 1u << (j % 32);
        return (atomicOr(&claims[(p - 1) * kDecClaimWords + j / 32], bit) & bit) == 0;
    };
    // The first warp: looks for another piece; false when none is left.
    auto next_piece = [&]() -> bool {
        const uint32_t lane = threadIdx.x & 31, p = s_piece;
        if (p < B.n_pieces) {
            bool got = p == 0;
            if (p && lane == 0) got = claim(p, blockIdx.x);
            got = __shfl_sync(0xFFFFFFFFu, got, 0);
            __syncwarp();
            if (lane == 0) s_piece = got ? p + 1 : B.n_pieces;
            if (got) { enter(p, blockIdx.x); return true; }
        }
        // Lane l looks at word l of the bits, starting behind the block's own place, so that blocks do not all try the same one.
        const uint32_t q = lane / kDecClaimWords + 1, w = (lane + blockIdx.x / 32) % kDecClaimWords;
        const uint32_t in_word = gridDim.x > 32 * w ? min(32u, gridDim.x - 32 * w) : 0u;
        for (uint32_t tries = 0; tries < kDecMaxPieces * kDecMaxBlocks; ++tries) {
            uint32_t open = 0;
            if (q < B.n_pieces && lane < (kDecMaxPieces - 1) * kDecClaimWords && in_word)
                open = ~*reinterpret_cast<volatile uint32_t*>(&claims[(q - 1) * kDecClaimWords + w]) & (0xFFFFFFFFu >> (32 - in_word));
            const uint32_t have = __ballot_sync(0xFFFFFFFFu, open != 0);
            if (!have) return false;
            const uint32_t who = __ffs(have) - 1;
            const uint32_t behind = open & (0xFFFFFFFFu << (blockIdx.x % 32));
            const uint32_t j = 32 * w + __ffs(behind ? behind : open) - 1;
            bool got = false;
            if (lane == who) got = claim(q, j);
            if (__shfl_sync(0xFFFFFFFFu, got, who)) {
                enter(__shfl_sync(0xFFFFFFFFu, q, who), __shfl_sync(0xFFFFFFFFu, j, who));
                return true;
            }
        }
        return false;
    };
    // The first warp: the next part.
    auto next_part = [&]() {
        uint32_t t = kNone, lo = 0, hi = 0, e = s_empty;
        while (e < B.n_tensors && B.item[e].n_chunks != 0) ++e;
        const bool lost = block_lost() != 0;
        if (e < B.n_tensors && !lost) {
            t = e++;
        } else {
            bool more = !lost;
            while (s_g >= s_g_hi && more) more = next_piece();
            if (more) {
                const uint32_t g = s_g;
                t = s_g_t;
                while (g >= B.item[t].first_chunk + B.item[t].n_chunks) ++t;
                lo = g - B.item[t].first_chunk;
                hi = min(s_g_hi - B.item[t].first_chunk, B.item[t].n_chunks);
            }
        }
        __syncwarp();
        if (threadIdx.x == 0) {
            s_empty = e;
            s_t = t; s_lo = lo; s_hi = hi;
            if (hi > lo) { s_g += hi - lo; s_g_t = t; }
        }
    };
    for (;;) {
        __syncthreads();                                         // everybody is done with the previous part
        if (threadIdx.x < 32) next_part();
        __syncthreads();
        const uint32_t t = s_t;
        if (t == kNone) break;
        const bool opened_before = s_opened == t;
        DecParams P;
        P.comp = B.item[t].comp; P.base = XOR ? B.item[t].base : nullptr; P.out = B.item[t].out; P.ctl = B.ctl;
        P.comp_bytes = B.item[t].comp_bytes; P.input_bytes = B.item[t].input_bytes;
        P.n_syms = B.item[t].n_syms; P.n_elems = B.item[t].n_elems; P.n_chunks = B.item[t].n_chunks;
        P.cs = B.cs; P.sub = B.sub; P.chunk_bytes = B.chunk_bytes; P.format = B.format; P.group = B.group;
        P.pool_bytes = B.pool_bytes; P.call_id = B.call_id; P.c_begin = 0; P.c_end = P.n_chunks;
        P.spin_limit = B.spin_limit; P.skip_copy = B.skip_copy; P.sliced = B.sliced; P.active = blockDim.x >> 5;
        const uint64_t tables = 256 + (((uint64_t)4 * P.n_chunks + 15) & ~15ull) + 32ull * (P.chunk_bytes <= 8192 ? 2u : 4u) * P.n_chunks;
        P.spec = P.comp_bytes >= kHeaderBytes + tables ? 1u : 0u;
        const uint32_t err = decode_one<FMT, PPL, XOR, XOR || FMT == ZC_FMT_SCALE_U8, SMALL>(P, M, s_lo, s_hi, 0, 1, opened_before, parity0, parity1);
        if (err && raise_status(B.ctl, B.call_id, err)) B.ctl->failed = B.tensor_base + s_t + 1;
        // (a tensor that could not be opened is opened again, and refused again, in every part)
        if (!opened_before && threadIdx.x == 0) s_opened = err ? kNone : t;
    }
}


// ---- launchers, one set per element format -------------------------------------------------------------------
// The kernels of one format are instantiated where that format's launchers are defined.  This file can be compiled
// as a whole (ZC_DEC_PART undefined or 0) or in four parts (1: the C ABI and BF16, 2: FP8, 3: scale bytes, 4: FP4), one
// object each, so that a build compiles the formats side by side.
#ifndef ZC_DEC_PART
#define ZC_DEC_PART 0
#endif

// the buffers of a launch, for the development build's checks
struct DecRanges { const void* in; size_t in_bytes; const void* out; size_t out_bytes; const void* ws; size_t ws_bytes; };

template <int F>
cudaError_t dec_launch_single_t(uint32_t ppl, int kind, uint32_t grid, uint32_t threads, size_t smem, cudaStream_t st, const DecParams& P,
                                const DecRanges& R)
{
    cudaError_t e = cudaSuccess;
    auto launch = [&](auto kern) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return;
#if ZC_DEBUG_CHECKS
        dbg_set_ranges(st, R.in, R.in_bytes, R.out, R.out_bytes, R.ws, R.ws_bytes);
#else
        (void)R;
#endif
        kern<<<grid, threads, smem, st>>>(P);
        e = cudaGetLastError();
    };
    if (kind == kDecSplit) {
        launch(decode_split_kernel<F>);
    } else if (kind == kDecFew) {
        if (ppl == 4) launch(decode_kernel<F, 4, true, false>);
        else if (ppl == 2) launch(decode_kernel<F, 2, true, false>);
        else launch(decode_kernel<F, 1, true, false>);
    } else if (P.chunk_bytes <= kSmallChunk) {
        if (ppl == 4) launch(decode_kernel<F, 4, false, true>);
        else if (ppl == 2) launch(decode_kernel<F, 2, false, true>);
        else launch(decode_kernel<F, 1, false, true>);
    } else {
        if (ppl == 4) launch(decode_kernel<F, 4, false, false>);
        else if (ppl == 2) launch(decode_kernel<F, 2, false, false>);
        else launch(decode_kernel<F, 1, false, false>);
    }
    return e;
}

template <int F>
cudaError_t dec_launch_batch_t(uint32_t ppl, bool any_base, uint32_t grid, uint32_t threads, size_t smem, cudaStream_t st,
                               const DecBatchParams& B, const DecRanges& R)
{
    cudaError_t e = cudaSuccess;
    auto launch = [&](auto kern) {
        e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return;
#if ZC_DEBUG_CHECKS
        dbg_set_ranges(st, R.in, R.in_bytes, R.out, R.out_bytes, R.ws, R.ws_bytes);
#else
        (void)R;
#endif
        kern<<<grid, threads, smem, st>>>(B);
        e = cudaGetLastError();
    };
    auto pick = [&](auto xor_tag, auto small_tag) {
        constexpr bool XOR = decltype(xor_tag)::value, SMALL = decltype(small_tag)::value;
        if (ppl == 4) launch(decode_batch_kernel<F, 4, XOR, SMALL>);
        else if (ppl == 2) launch(decode_batch_kernel<F, 2, XOR, SMALL>);
        else launch(decode_batch_kernel<F, 1, XOR, SMALL>);
    };
    const bool small = B.chunk_bytes <= kSmallChunk;
    if (any_base) { if (small) pick(BoolTag<true>{}, BoolTag<true>{}); else pick(BoolTag<true>{}, BoolTag<false>{}); }
    else { if (small) pick(BoolTag<false>{}, BoolTag<true>{}); else pick(BoolTag<false>{}, BoolTag<false>{}); }
    return e;
}

#define ZC_DEC_DECLARE(NAME)                                                                                              \
    cudaError_t dec_launch_single_##NAME(uint32_t ppl, int kind, uint32_t grid, uint32_t threads, size_t smem, cudaStream_t st,     \
                                         const DecParams& P, const DecRanges& R);                                        \
    cudaError_t dec_launch_batch_##NAME(uint32_t ppl, bool any_base, uint32_t grid, uint32_t threads, size_t smem,        \
                                        cudaStream_t st, const DecBatchParams& B, const DecRanges& R);                   \
    void dec_debug_counts_##NAME(uint32_t out[2]);
ZC_DEC_DECLARE(bf16)
ZC_DEC_DECLARE(fp8)
ZC_DEC_DECLARE(scale)
ZC_DEC_DECLARE(fp4)
#undef ZC_DEC_DECLARE

#if ZC_DEBUG_CHECKS
#define ZC_DEC_COUNTS(out) dbg_read_counts(out)
#else
#define ZC_DEC_COUNTS(out) (void)(out)
#endif
#define ZC_DEC_DEFINE(NAME, F)                                                                                            \
    cudaError_t dec_launch_single_##NAME(uint32_t ppl, int kind, uint32_t grid, uint32_t threads, size_t smem, cudaStream_t st,     \
                                         const DecParams& P, const DecRanges& R)                                         \
    { return dec_launch_single_t<F>(ppl, kind, grid, threads, smem, st, P, R); }                                                \
    cudaError_t dec_launch_batch_##NAME(uint32_t ppl, bool any_base, uint32_t grid, uint32_t threads, size_t smem,        \
                                        cudaStream_t st, const DecBatchParams& B, const DecRanges& R)                    \
    { return dec_launch_batch_t<F>(ppl, any_base, grid, threads, smem, st, B, R); }                                       \
    void dec_debug_counts_##NAME(uint32_t out[2]) { ZC_DEC_COUNTS(out); }
#if ZC_DEC_PART == 0 || ZC_DEC_PART == 1
ZC_DEC_DEFINE(bf16, ZC_FMT_BF16)
#endif
#if ZC_DEC_PART == 0 || ZC_DEC_PART == 2
ZC_DEC_DEFINE(fp8, ZC_FMT_FP8_E4M3)
#endif
#if ZC_DEC_PART == 0 || ZC_DEC_PART == 3
ZC_DEC_DEFINE(scale, ZC_FMT_SCALE_U8)
#endif
#if ZC_DEC_PART == 0 || ZC_DEC_PART == 4
ZC_DEC_DEFINE(fp4, ZC_FMT_FP4_E2M1)
#endif
#undef ZC_DEC_DEFINE

}  // namespace zc

#if ZC_DEC_PART <= 1

using namespace zc;

extern "C" {

namespace {

// Launch shape for a plan: symbols per round and lane, per-warp pool, warps per block, shared memory.
struct DecShape { uint32_t ppl, pool_bytes, warps, sliced; size_t smem; };

// both_coded: expect both streams to be Huffman-coded (scale bytes, deltas) instead of one
zc_status dec_shape(const zc_plan_t* p, bool both_coded, DecShape* out)
{
    DecShape s{};
    // symbols per round and lane: the largest of 64 / 32 / 16 that divides the subchunk length
    s.ppl = (p->syms_per_sub % 64 == 0) ? 4 : (p->syms_per_sub % 32 == 0) ? 2 : 1;
    // scale bytes and deltas have both streams coded as a rule, plain tensors one (the other one is raw)
    const uint32_t coded = (both_coded || p->format == ZC_FMT_SCALE_U8) ? 2 : 1;
    const uint32_t rows_bytes = 512 * s.ppl;
    // per warp: the coded streams' rows plus room to stage, per coded stream, a piece as large as the raw chunk
    // stream; pieces that do not fit (or chunks above 16 KiB of symbols) are read from global memory instead
    s.sliced = p->syms_per_sub % kSliceSyms == 0 ? 1u : 0u;   // pieces beyond their slot can be staged slice by slice
    s.pool_bytes = std::max<uint32_t>(coded * (rows_bytes + std::min<uint32_t>(p->syms_per_chunk, 16384) + 32), 2 * rows_bytes);
    // up to 4 KiB: room for the bytes of a raw stream too (see run_small)
    if (p->chunk_bytes <= kSmallChunk) s.pool_bytes = std::max(s.pool_bytes, rows_bytes + p->syms_per_chunk + 32 + small_raw_buffers(s.ppl) * p->syms_per_chunk);
    // chunks above 16 KiB: whole pieces would leave room for a dozen warps at most; lane slots for sliced pieces
    // are enough, and more warps decode
    if (s.sliced && p->syms_per_chunk > 8192) s.pool_bytes = std::max<uint32_t>(coded * (rows_bytes + 32 * kSliceSlot), 2 * rows_bytes);
    // slack behind the last slot: what a lane can read past its piece when the payload is damaged (see window_s)
    const size_t slack = (size_t)round_up(p->syms_per_sub + p->syms_per_sub / 2 + 16, 16);
    const size_t fixed = kDecStaticSmem + kScratchBytes + slack;
    size_t per_warp = 16 + s.pool_bytes;
    const size_t max_warps = coded == 2 ? kDecMaxWarpsBoth : kDecMaxWarps;     // the kernels' launch bounds
    s.warps = (uint32_t)std::min<size_t>(max_warps, (kMaxSmem - fixed - 1024) / per_warp);
    if (s.warps < 8) {               // large chunks: stage less
        s.pool_bytes = std::max<uint32_t>(coded * (rows_bytes + 32 * kSliceSlot), 2 * rows_bytes);   // room for the lane slots of sliced pieces
        per_warp = 16 + s.pool_bytes;
        s.warps = (uint32_t)std::min<size_t>(max_warps, (kMaxSmem - fixed - 1024) / per_warp);
    }
    // the table build uses 8 KiB of the pools and 256 threads
    while (s.warps * (size_t)s.pool_bytes < 8192) ++s.warps;
    if (s.warps < 8 || s.warps > max_warps) return ZC_E_UNSUPPORTED;
    s.smem = kScratchBytes + s.warps * per_warp + slack;
    *out = s;
    return ZC_OK;
}

// Launch shape for n_chunks chunks of one tensor when they are few: `warps` build the tables, `active` of them decode.
DecShape few_shape(const zc_plan_t* p, uint32_t n_chunks, uint32_t* active)
{
    DecShape s{};
    s.ppl = (p->syms_per_sub % 64 == 0) ? 4 : (p->syms_per_sub % 32 == 0) ? 2 : 1;
    s.warps = kDecFewWarps;
    const size_t slack = (size_t)round_up(p->syms_per_sub + p->syms_per_sub / 2 + 16, 16);
    const size_t room = kMaxSmem - 1024 - kDecStaticSmem - kScratchBytes - 16 * s.warps - slack;
    *active = std::max<uint32_t>(1, (n_chunks + sm_count() - 1) / sm_count());
    // rows of both streams and room for whole pieces of 12-bit codes (less when the warps' shares are smaller: slices then)
    const uint32_t most = 2 * (512 * s.ppl + (uint32_t)round_up((uint64_t)p->syms_per_chunk * kLmax / 8, 16) + 32);
    const uint32_t share = (uint32_t)(room / *active) & ~15u;
    s.pool_bytes = std::max<uint32_t>(std::min(most, share), 8192);          // the table build uses 8 KiB of the pools
    // slices only where whole pieces might not fit (then the pools fill the block's memory, as decode_one's sharing of them
    // among fewer warps expects)
    s.sliced = share < most && p->syms_per_sub % kSliceSyms == 0 ? 1u : 0u;
    s.smem = kScratchBytes + 16 * s.warps + (size_t)*active * s.pool_bytes + slack;
    return s;
}

// Launch shape of decode_split_kernel: as many blocks per chunk as there are SMs for, up to 8 (4 subchunks each).
DecShape split_shape(const zc_plan_t* p, uint32_t n_chunks, uint32_t* groups)
{
    DecShape s{};
    s.ppl = 1;
    s.warps = kSplitThreads / 32;
    *groups = 1;
    while (*groups < 8 && 2ull * *groups * n_chunks <= (uint64_t)sm_count()) *groups *= 2;
    const uint32_t syms = p->syms_per_chunk / *groups;
    s.pool_bytes = std::max<uint32_t>(2 * syms + 2 * ((uint32_t)round_up((uint64_t)syms * kLmax / 8, 16) + 48), 8192);
    s.smem = kScratchBytes + 16 * s.warps + s.pool_bytes + 64;   // the bit readers look a few words past a piece's copy
    return s;
}

// Pieces of a slice of a batched launch (see kDecMaxPieces), as where they end in 65536ths of it; turn = one chunk for every warp.
// Seven eighths of what is left, until one is down to two chunks per warp; the last one is the rest.  Deltas: five eighths of the slice,
// then an eighth of it or half of what is left, whichever is less, since slices differ in speed (unchanged stretches take half of
// the time and less) and the piece that is taken last from a slow one is what the launch ends with.  (15 GB of deltas, most layers
// unchanged: 6.89 ms; 7.59 ms with a half, a quarter and so on, which left a quarter of a slow slice to the block that came first.  872
// MB with none, a quarter, half, three quarters unchanged: 657, 609, 523, 457 us against 658, 623, 520, 485.  Two more pieces: 6.75 ms,
// but 668, 611, 532, 457 us: another piece costs about 5 us.)  With fewer than kDecOneRound chunks per warp in all, another piece costs
// more than it evens out (FP8 at 16 KiB chunks, 9 chunks per warp: 219 us in one round, 270 us in three; BF16 at 1 KiB chunks, 44
// per warp: 119 us in one round, 140 in four).
uint32_t dec_pieces(uint64_t total, uint64_t turn, bool any_base, uint32_t* piece_end)
{
    uint32_t n = 0;
    for (uint64_t done = 0; done < 65536;) {
        const uint64_t left = 65536 - done;
        const uint64_t part = !any_base ? left - left / 8 : done ? std::min<uint64_t>(left / 2, 65536 / 8) : left / 8 * 5;
        const bool last = n + 1 == kDecMaxPieces || total < kDecOneRound * turn || (left - part) * total < 2 * turn * 65536;
        done = last ? 65536 : done + part;
        piece_end[n++] = (uint32_t)done;
    }
    return n;
}

// Blocks of a batched launch: one per SM, or fewer.  The chunk index space is cut into equal slices, and a slice that reaches
// over a tensor's end costs its block a second header, table and walk over a subchunk, one after the other.  A multiple of
// the number of tensors has no such ranges when the tensors are of one size.  Taken is what is shorter for the block with the
// longest way, in symbols of a lane's walk: a tensor's part costs kDecOpenSyms (9 us) and its chunks a walk for every round
// over the warps.  (64 BF16 tensors of 9 chunks of 64 KiB: 135 us in 148 ranges, 77 us in 128; 36 of 64 chunks of 32 KiB: 77
// and 52 us.)
constexpr uint32_t kDecOpenSyms = 160, kDecChunkSyms = 16;
uint32_t batch_grid(const DecItem* item, uint32_t n, uint32_t with_chunks, uint64_t total, uint32_t warps, uint32_t sub)
{
    const uint32_t most = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>({total, (uint64_t)sm_count(), kDecMaxBlocks}));
    const uint32_t even = with_chunks ? most / with_chunks * with_chunks : 0;
    if (with_chunks < 2 || even == 0 || even == most || total >= (uint64_t)kDecOneRound * most * warps) return most;
    auto longest = [&](const uint32_t ranges) {
        const uint32_t step = (uint32_t)(total / ranges), odd = (uint32_t)(total % ranges);
        uint32_t t = 0, g = 0, hi = 0, rest = 0, worst = 0;
        uint64_t end = item[0].n_chunks;                         // where tensor t ends
        for (uint32_t j = 0; j < ranges; ++j) {                  // range j ends at (j + 1) * total / ranges
            hi += step;
            rest += odd;
            if (rest >= ranges) { rest -= ranges; ++hi; }
            uint32_t way = 0;
            while (g < hi) {
                while (end <= g) end += item[++t].n_chunks;
                const uint32_t part = (uint32_t)std::min<uint64_t>(hi, end) - g;
                way += kDecOpenSyms + (part + warps - 1) / warps * (sub + kDecChunkSyms);
                g += part;
            }
            worst = std::max(worst, way);
        }
        return worst;
    };
    return longest(even) < longest(most) ? even : most;
}

// no clearing of the workspace: errors are tagged with the id of the call that raised them
unsigned long long new_call_id()
{
    static std::atomic<unsigned long long> next_call{(unsigned long long)std::chrono::steady_clock::now().time_since_epoch().count()};
    return (next_call.fetch_add(1) & ((1ull << 56) - 1)) | 1ull << 55;
}

}  // namespace

}  // extern "C"
namespace zc {
void debug_counts_decode(uint32_t out[2])
{
    dec_debug_counts_bf16(out);
    dec_debug_counts_fp8(out);
    dec_debug_counts_scale(out);
    dec_debug_counts_fp4(out);
}
}  // namespace zc
extern "C" {

uint32_t zc_test_decoder_warps(const zc_plan_t* p, uint32_t both_coded)
{
    DecShape sh;
    if (!p || dec_shape(p, both_coded != 0, &sh) != ZC_OK) return 0;
    return sh.warps;
}

uint32_t zc_test_decoder_pieces(const zc_plan_t* p, uint32_t any_base, uint64_t total_chunks, uint32_t* h_piece_end)
{
    DecShape sh;
    if (!p || !h_piece_end || !total_chunks || dec_shape(p, any_base != 0, &sh) != ZC_OK) return 0;
    return dec_pieces(total_chunks, std::min<uint64_t>({total_chunks, (uint64_t)sm_count(), kDecMaxBlocks}) * sh.warps, any_base != 0, h_piece_end);
}

zc_status zc_decompress(const zc_plan_t* p, const void* d_comp, size_t comp_bytes, void* d_out, void* d_workspace,
                        void* cuda_stream)
{
    return zc_decompress_xor(p, d_comp, comp_bytes, nullptr, d_out, d_workspace, cuda_stream);
}

zc_status zc_decompress_xor(const zc_plan_t* p, const void* d_comp, size_t comp_bytes, const void* d_base, void* d_out,
                            void* d_workspace, void* cuda_stream)
{
    if (d_base) {                                            // the delta form lives in the batched kernel
        if (!p) return ZC_E_INVALID_ARG;
        void* out1 = d_out;
        return zc_decompress_batch_xor(1, &p, &d_comp, &comp_bytes, &d_base, &out1, d_workspace, cuda_stream);
    }
    if (!p) return ZC_E_INVALID_ARG;
    return zc_decompress_chunks(p, d_comp, comp_bytes, 0, p->n_chunks, d_out, d_workspace, cuda_stream);
}

zc_status zc_decompress_chunks(const zc_plan_t* p, const void* d_comp, size_t comp_bytes, uint32_t first_chunk, uint32_t n_chunks,
                               void* d_out, void* d_workspace, void* cuda_stream)
{
    if (!p || !d_comp || !d_workspace || (!d_out && p->n_elems)) return ZC_E_INVALID_ARG;
    if ((uint64_t)first_chunk + n_chunks > p->n_chunks) return ZC_E_INVALID_ARG;
    if (!aligned16(d_comp) || !aligned16(d_out) || !aligned16(d_workspace)) return ZC_E_INVALID_ARG;
    if (comp_bytes < kHeaderBytes) return ZC_E_CORRUPT;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    DecShape shape;
    uint32_t active = 0;
    uint32_t groups = 1;
    // decode_split_kernel's rounds cost more than a lane's walk where subchunks are short (see kSplitMinSub), and more than
    // other warps' walks where a block would have several chunks.
    const int kind = p->syms_per_sub >= kSplitMinSub && n_chunks <= (uint32_t)sm_count() ? kDecSplit
                     : n_chunks <= kDecFewActive * (uint32_t)sm_count() ? kDecFew : kDecMany;
    if (kind == kDecSplit) {
        shape = split_shape(p, n_chunks, &groups);
        active = 1;
    } else if (kind == kDecFew) {
        shape = few_shape(p, n_chunks, &active);
    } else {
        const zc_status ss = dec_shape(p, false, &shape);
        if (ss != ZC_OK) return ss;
        active = shape.warps;
    }
    DecParams P{};
    P.comp = (const uint8_t*)d_comp;
    P.base = nullptr;
    // the kernel addresses the output by position in the tensor: d_out is where chunk first_chunk goes
    P.out = (uint8_t*)d_out - (size_t)first_chunk * p->chunk_bytes;
    P.c_begin = first_chunk; P.c_end = first_chunk + n_chunks;
    P.ctl = (Control*)d_workspace;
    P.comp_bytes = comp_bytes; P.input_bytes = p->input_bytes; P.n_syms = p->n_syms; P.n_elems = p->n_elems;
    P.n_chunks = p->n_chunks; P.cs = p->syms_per_chunk; P.sub = p->syms_per_sub; P.chunk_bytes = p->chunk_bytes;
    P.format = p->format; P.group = p->group;
    P.call_id = new_call_id();
    P.spec = comp_bytes >= kHeaderBytes + table_section_bytes(p->n_chunks, p->chunk_bytes) ? 1u : 0u;
    P.pool_bytes = shape.pool_bytes;
    P.spin_limit = test_knobs().spin_limit; P.skip_copy = test_knobs().skip_copy; P.sliced = shape.sliced; P.active = active; P.groups = groups;
    const uint32_t warps = shape.warps, ppl = shape.ppl;
    const size_t smem = shape.smem;
    // at least one block even for an empty range: the header is still checked
    const uint32_t want = std::max<uint32_t>(kind != kDecMany ? n_chunks : (n_chunks + warps - 1) / warps, 1);
    const uint32_t grid = kind == kDecSplit ? std::max<uint32_t>(n_chunks, 1) * groups : std::min<uint32_t>(want, (uint32_t)sm_count());
    const DecRanges R{d_comp, comp_bytes, d_out,
                      (size_t)std::min<uint64_t>((uint64_t)n_chunks * p->chunk_bytes, p->input_bytes - (uint64_t)first_chunk * p->chunk_bytes),
                      d_workspace, sizeof(Control)};
    cudaError_t e;
    switch (p->format) {
    case ZC_FMT_BF16: e = dec_launch_single_bf16(ppl, kind, grid, warps * 32, smem, st, P, R); break;
    case ZC_FMT_FP8_E4M3: case ZC_FMT_FP8_E5M2: e = dec_launch_single_fp8(ppl, kind, grid, warps * 32, smem, st, P, R); break;
    case ZC_FMT_SCALE_U8: e = dec_launch_single_scale(ppl, kind, grid, warps * 32, smem, st, P, R); break;
    default: e = dec_launch_single_fp4(ppl, kind, grid, warps * 32, smem, st, P, R); break;
    }
    return e == cudaSuccess ? ZC_OK : ZC_E_CUDA;
}

zc_status zc_decompress_batch(uint32_t n_tensors, const zc_plan_t* const* plans, const void* const* d_comp,
                              const size_t* comp_bytes, void* const* d_out, void* d_workspace, void* cuda_stream)
{
    return zc_decompress_batch_xor(n_tensors, plans, d_comp, comp_bytes, nullptr, d_out, d_workspace, cuda_stream);
}

zc_status zc_decompress_batch_xor(uint32_t n_tensors, const zc_plan_t* const* plans, const void* const* d_comp,
                                  const size_t* comp_bytes, const void* const* d_base, void* const* d_out,
                                  void* d_workspace, void* cuda_stream)
{
    if (!d_workspace || !aligned16(d_workspace)) return ZC_E_INVALID_ARG;
    if (n_tensors == 0) return ZC_OK;
    if (!plans || !d_comp || !comp_bytes || !d_out) return ZC_E_INVALID_ARG;
    for (uint32_t t = 0; t < n_tensors; ++t) {
        const zc_plan_t* p = plans[t];
        if (!p || !d_comp[t] || (!d_out[t] && p->n_elems)) return ZC_E_INVALID_ARG;
        if (!aligned16(d_comp[t]) || !aligned16(d_out[t]) || (d_base && !aligned16(d_base[t]))) return ZC_E_INVALID_ARG;
        if (p->format != plans[0]->format || p->chunk_bytes != plans[0]->chunk_bytes) return ZC_E_INVALID_ARG;
        if (comp_bytes[t] < kHeaderBytes) return ZC_E_CORRUPT;
    }
    cudaStream_t st = (cudaStream_t)cuda_stream;
    const zc_plan_t* p0 = plans[0];
    DecShape shape;
    bool delta = false;
    if (d_base) for (uint32_t t = 0; t < n_tensors; ++t) delta = delta || d_base[t] != nullptr;
    const zc_status ss = dec_shape(p0, delta, &shape);
    if (ss != ZC_OK) return ss;
    const unsigned long long call_id = new_call_id();
    static thread_local DecBatchParams B;                    // 28 KiB: kept off the stack
    for (uint32_t base = 0; base < n_tensors;) {
        B.ctl = (Control*)d_workspace;
        B.call_id = call_id;
        B.cs = p0->syms_per_chunk; B.sub = p0->syms_per_sub; B.chunk_bytes = p0->chunk_bytes;
        B.format = p0->format; B.group = p0->group; B.pool_bytes = shape.pool_bytes;
        B.tensor_base = base;
        B.spin_limit = test_knobs().spin_limit; B.skip_copy = test_knobs().skip_copy; B.sliced = shape.sliced;
        uint32_t n = 0;
        uint64_t total = 0;
        // as many tensors as fit one launch: at most kDecBatchMax, fewer than 2^32 chunks together
        while (base + n < n_tensors && n < kDecBatchMax && total + plans[base + n]->n_chunks < (1ull << 32)) {
            const zc_plan_t* p = plans[base + n];
            DecItem& it = B.item[n];
            it.comp = (const uint8_t*)d_comp[base + n];
            it.base = d_base ? (const uint8_t*)d_base[base + n] : nullptr;
            it.out = (uint8_t*)d_out[base + n];
            it.comp_bytes = comp_bytes[base + n]; it.input_bytes = p->input_bytes; it.n_syms = p->n_syms; it.n_elems = p->n_elems;
            it.n_chunks = p->n_chunks; it.first_chunk = (uint32_t)total;
            total += p->n_chunks;
            ++n;
        }
        B.n_tensors = n;
        bool any_base = false;
        B.n_empty = 0;
        for (uint32_t i = 0; i < n; ++i) {
            any_base = any_base || B.item[i].base != nullptr;
            B.n_empty += B.item[i].n_chunks == 0;
        }
        const uint32_t grid = batch_grid(B.item, n, n - B.n_empty, total, shape.warps, B.sub);
        B.total = (uint32_t)total;
        B.n_pieces = dec_pieces(total, (uint64_t)grid * shape.warps, any_base, B.piece_end);
        if (B.n_pieces > 1 && cudaMemsetAsync((uint8_t*)d_workspace + kDecClaims, 0, 4 * (kDecMaxPieces - 1) * kDecClaimWords, st) != cudaSuccess) return ZC_E_CUDA;
        DecRanges R{nullptr, 0, nullptr, 0, d_workspace, sizeof(Control)};
#if ZC_DEBUG_CHECKS
        DbgHull rd, wr;
        for (uint32_t i = 0; i < n; ++i) {
            rd.add(B.item[i].comp, B.item[i].comp_bytes);
            rd.add(B.item[i].base, B.item[i].input_bytes);
            wr.add(B.item[i].out, B.item[i].input_bytes);
        }
        R.in = rd.ptr(); R.in_bytes = rd.bytes(); R.out = wr.ptr(); R.out_bytes = wr.bytes();
#endif
        cudaError_t e;
        switch (p0->format) {
        case ZC_FMT_BF16: e = dec_launch_batch_bf16(shape.ppl, any_base, grid, shape.warps * 32, shape.smem, st, B, R); break;
        case ZC_FMT_FP8_E4M3: case ZC_FMT_FP8_E5M2: e = dec_launch_batch_fp8(shape.ppl, any_base, grid, shape.warps * 32, shape.smem, st, B, R); break;
        case ZC_FMT_SCALE_U8: e = dec_launch_batch_scale(shape.ppl, any_base, grid, shape.warps * 32, shape.smem, st, B, R); break;
        default: e = dec_launch_batch_fp4(shape.ppl, any_base, grid, shape.warps * 32, shape.smem, st, B, R); break;
        }
        if (e != cudaSuccess) return ZC_E_CUDA;
        base += n;
    }
    return ZC_OK;
}

zc_status zc_batch_status(const void* d_workspace, uint32_t* h_failed_tensor, void* cuda_stream)
{
    if (!d_workspace) return ZC_E_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    Control h;
    if (cudaMemcpyAsync(&h, d_workspace, sizeof(Control), cudaMemcpyDeviceToHost, st) != cudaSuccess) return ZC_E_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return ZC_E_CUDA;
    const bool mine = (h.status >> 8) == h.call_id && (h.status & 0xFF) != 0;
    if (h_failed_tensor) *h_failed_tensor = mine && h.failed ? h.failed - 1 : 0xFFFFFFFFu;
    return mine ? (zc_status)(h.status & 0xFF) : ZC_OK;
}

}  // extern "C"

#endif  // ZC_DEC_PART <= 1
