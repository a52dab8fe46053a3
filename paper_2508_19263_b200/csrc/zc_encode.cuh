// Encoder kernel: field split, code lookup, bit packing and placement of the chunks in one pass over the input.
//
// Work unit of a warp: a tile, 32 lanes x 64 (in one kernel shape 48) consecutive symbols, 4 KiB (3 KiB) of input.  Packing needs no serial walk over a
// subchunk: once every lane knows how many bits its symbols take, prefix sums give every lane its bit position, and a
// subchunk may end anywhere a lane has added up 16 symbols (subchunks are multiples of 16 symbols long).  A unit is one
// chunk, or as many whole chunks as fit a tile (chunks of 1 and 2 KiB); T warps, one per tile of a unit, form a team that
// codes one unit together (T = 1: nothing to agree on).  A block is several teams plus two service warps, and its batch is
// as many consecutive units of a tensor as it has teams.
//   A  the tile's input arrives in shared memory by a bulk asynchronous copy requested a tile ahead; it is split in
//      registers, the raw stream is stored as it is, the coded stream goes back into the same buffer as one row of 64
//      (48) bytes per lane (16-byte pieces of 64-byte rows swizzled so that neither side has bank conflicts)
//   B  every lane looks up its symbols and keeps the codes of two neighbouring symbols, joined, in one register each
//      (24 bits of code, 5 bits of length), adding up the bits; the warp scans the bit counts
//   C  the unit's size is posted, subchunk ends are written, and every lane ORs its codes into the chunk's piece in the
//      team's output ring in shared memory, at their final bit position
// Pieces lie in the ring exactly as they will lie in the payload area.  Once a batch's place is known a service warp
// sends each team's pieces there with one bulk copy (cp.async.bulk shared -> global).  The place is the sum of the sizes
// of all earlier batches of the tensor, found by a look-back over one word per batch; workers never wait for it, only
// for room in their ring (several chunks deep).
#pragma once
#include "zc_device.cuh"

namespace zc {

// The code tables of a codebook as they travel to the device: per symbol the code left-aligned in bits 15..4 and its
// length in bits 3..0, 0 for a symbol without a code.
struct EncTables {
    uint16_t enc[2][256];
    uint32_t fill[2];                            // fill symbol (the one with the all-zero code) | its code length << 8
    uint32_t pad[2];
};

// The entries of the tables in shared memory: the code left-aligned in bits 31..20, the length in bits 3..0.  A symbol
// without a code has a bit of its own; two of them add up to a bit that no sum of two lengths reaches.
constexpr uint32_t kNoCode = 0x40;
__device__ __forceinline__ uint32_t enc_entry(uint32_t v) { return v ? ((v & 0xFFF0u) << 16) | (v & 15u) : kNoCode; }

// One tensor of a launch.
struct EncItem {
    const uint8_t* in;
    const uint8_t* base;                         // XOR-delta form: what is coded is in XOR base; or null
    uint8_t* out;
    uint64_t input_bytes, n_syms, n_elems;
    Layout lay;
    uint32_t n_chunks, n_units;
    uint32_t first_batch;                        // batches of all earlier tensors of the launch
    uint32_t index;                              // position in the caller's arrays (counters, error reports)
    uint32_t table;                              // its code tables among the uploaded ones (tensors may share a codebook)
    uint32_t pad;
};
static_assert(sizeof(EncItem) % 8 == 0, "items are copied as 8-byte words");

struct EncParams {
    Control* ctl;
    TensorCounters* counters;                    // indexed by EncItem::index
    unsigned long long* flags;                   // one look-back word per batch of the launch
    const EncItem* items;                        // batched calls: the launch's tensors; null: `one`
    const uint32_t* first_batch;                 // batched calls: EncItem::first_batch of every tensor, densely
    const EncTables* tables;                     // batched calls: indexed by EncItem::table; null: `table`
    uint32_t cs, sub, chunk_bytes;               // symbols per chunk / per subchunk
    uint32_t format, group, sub_width;           // sub_width: bytes per sub_end entry (2 or 4)
    uint32_t mode[2];
    uint32_t sub_magic;                          // ceil(2^32 / sub): k / sub == umulhi(k, sub_magic) for k < 2^17
    uint32_t unit_syms, unit_chunks;             // symbols and chunks of a unit
    uint32_t tiles, teams;                       // T (tiles of a unit = warps of a team), units of a batch
    uint32_t ring16;                             // a team's output ring, in 16-byte units
    uint32_t n_tensors, total_batches;
    uint32_t ahead;                              // 1: a block holds one batch at a time, 2: the next one too, 3: and the ticket after it
    uint32_t spin_limit;                         // polls after which a bounded wait gives up
    uint32_t base_buf;                           // every worker has a second input buffer for the base tensor
    uint32_t buf_bytes;                          // a worker's input buffers
    EncItem one;
    EncTables table;
};

constexpr unsigned long long kFlagAggregate = 1ull << 62, kFlagPrefix = 2ull << 62, kFlagValue = (1ull << 62) - 1;

__device__ __forceinline__ unsigned long long ld_flag(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_flag(unsigned long long* p, unsigned long long v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" :: "l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ void sts64(uint32_t addr, uint32_t a, uint32_t b)
{
    ZC_DBG_SHARED(addr, 8, return);
    asm volatile("st.shared.v2.u32 [%0], {%1,%2};" :: "r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void sts128_zero(uint32_t addr)
{
    ZC_DBG_SHARED(addr, 16, return);
    asm volatile("st.shared.v4.u32 [%0], {%1,%1,%1,%1};" :: "r"(addr), "r"(0u) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t addr)
{
    ZC_DBG_SHARED(addr, 16, return make_uint4(0, 0, 0, 0));
    uint4 v;
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void red_or(uint32_t addr, uint32_t v)
{
    ZC_DBG_SHARED(addr, 4, return);
    asm volatile("red.shared.or.b32 [%0], %1;" :: "r"(addr), "r"(v) : "memory");
}

// Append the bits (at most 32, left-aligned in `code`, zero below them) at bit position t of a lane's bit string, of
// which w holds the bits of the word at `addr` so far; t_new is the position behind them.  A word that is full is ORed
// into shared memory (neighbouring lanes share their first and last words) and the bits that did not fit start the next
// one; the three operations are predicated, not branched around, since in every step some lanes fill a word and some don't.
__device__ __forceinline__ void put_bits(uint32_t code, uint32_t t_new, uint32_t& t, uint32_t& w, uint32_t& addr)
{
    w |= __funnelshift_r(code, 0, t);                           // code >> (t & 31)
    const uint32_t rest = __funnelshift_r(0, code, t);          // code << (32 - (t & 31)), 0 for t & 31 == 0
    const uint32_t cross = (t ^ t_new) & 32u;
    t = t_new;
    if (cross) ZC_DBG_SHARED(addr, 4, return);
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p red.shared.or.b32 [%1], %0;\n\t@p add.u32 %1, %1, 4;\n\t@p mov.u32 %0, %2;\n\t}"
                 : "+r"(w), "+r"(addr) : "r"(rest), "r"(cross) : "memory");
}

__device__ __forceinline__ unsigned long long ld_ctl(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Bulk asynchronous copy shared -> global, tracked by the issuing thread's bulk groups.
__device__ __forceinline__ void bulk_s2g(void* dst, uint32_t src_s, uint32_t bytes)
{
    ZC_DBG_GLOBAL(dst, bytes, 16, true, return); ZC_DBG_SHARED(src_s, 16, return); ZC_DBG_SHARED(src_s + bytes - 16, 16, return);
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" :: "l"(dst), "r"(src_s), "r"(bytes) : "memory");
}

// Writes the 128-byte header and the guard of one tensor; called by one thread once every chunk is accounted for.
static __device__ __noinline__ void write_header(const EncParams& P, const EncItem& I, TensorCounters* tc)
{
    const bool any_huff = P.mode[0] == ZC_MODE_HUFF || P.mode[1] == ZC_MODE_HUFF;
    const uint64_t payload_bytes = any_huff ? 16ull * ld_ctl(&tc->total16) : 0;
    uint8_t* h = I.out;
    uint32_t* h32 = reinterpret_cast<uint32_t*>(h);
    unsigned long long* h64 = reinterpret_cast<unsigned long long*>(h);
    for (int i = 0; i < 32; ++i) h32[i] = 0;
    h32[0] = kMagic;
    h[kHdrVersion] = 1; h[kHdrFormat] = (uint8_t)P.format; h[kHdrStreams] = 2;
    h64[kHdrElems / 8] = I.n_elems;
    h32[kHdrChunkBytes / 4] = P.chunk_bytes;
    h32[kHdrChunks / 4] = I.n_chunks;
    h[kHdrLmax] = kLmax; h[kHdrGroup] = (uint8_t)P.group; h[kHdrSubs] = kSubs; h[kHdrSubWidth] = (uint8_t)P.sub_width;
    const uint64_t total = I.lay.payload_off + payload_bytes + (any_huff ? 16 : 0);
    h64[kHdrTotal / 8] = total;
    h64[kHdrPayloadOff / 8] = I.lay.payload_off;
    h64[kHdrPayloadBytes / 8] = payload_bytes;
    for (int s = 0; s < 2; ++s) {
        uint8_t* d = h + kHdrStream0 + kHdrStreamStride * s;
        d[kSdMode] = (uint8_t)P.mode[s];
        reinterpret_cast<unsigned long long*>(d)[1] = I.n_syms;
        reinterpret_cast<unsigned long long*>(d)[2] = P.mode[s] == ZC_MODE_HUFF ? ld_ctl(&tc->payload_bits[s]) : 8 * I.n_syms;
        reinterpret_cast<unsigned long long*>(d)[3] = I.lay.section_off[s];
    }
    if (any_huff) {                              // 16 zero bytes behind the payload: decoders may peek past the last piece
        uint32_t* g = reinterpret_cast<uint32_t*>(I.out + I.lay.payload_off + payload_bytes);
        g[0] = g[1] = g[2] = g[3] = 0;
    }
    tc->total16 = total;                         // the host reads the container size from here
}

constexpr uint32_t kEncRing = 16;                // batches of a block whose bookkeeping is alive at the same time
constexpr uint32_t kTabSlots = 4;                // tensors (code tables and item) a block's live batches may belong to
constexpr uint32_t kNoSlot = 0xFFFFFFFFu;        // "no more batches"
constexpr uint32_t kConstTile = 0x80000000u;     // tile of nothing but the fill symbol
constexpr int kLookWide = 4;                     // look-back rounds cover 32 * kLookWide predecessors

// Kernel shapes:
//   kEncSolo    a chunk is one tile (4 KiB)
//   kEncTeam    a chunk is T whole tiles (8, 12, 16, .. KiB)
//   kEncUnit    a tile is several whole chunks (1 and 2 KiB); in one kernel with the odd sizes both streams' codes did not fit
//               the registers (96 MB at 2 KiB, both streams coded: FP8 152 -> 127 us, scale bytes 122 -> 96 us)
//   kEncAny     everything else, with lanes of 64 symbols (the last tile is not full)
//   kEncAny48   the same with lanes of 48 where that fills the tiles better (3, 6, 9 KiB; BF16 weights at 6 KiB: 95 against 119 us)
//   kEncBig     chunks that need more workers than the shape above has, or of which it fits twice the teams
//   kEncSolo80, kEncSolo96, kEncSolo112   a chunk of 5, 6 or 7 KiB with one coded stream is one tile of long lanes: two tiles
//               are a sixth to a quarter empty, and a team that meets twice per chunk is slower than a warp alone (128 MB of
//               BF16 weights in two tiles / one, and in the encoder with lane regions that packed subchunk by subchunk: 5 KiB
//               103 / 74 / 82 us, 6 KiB 86 / 69 / 82 us, 7 KiB 97 / 73 / 84 us)
constexpr int kEncSolo = 0, kEncTeam = 1, kEncAny = 2, kEncAny48 = 3, kEncBig = 4, kEncSolo80 = 5, kEncSolo96 = 6, kEncSolo112 = 7, kEncUnit = 8;
__host__ __device__ constexpr uint32_t enc_lane_syms(int shape) { return shape == kEncAny48 ? 48u : shape >= kEncSolo80 && shape <= kEncSolo112 ? 16u * shape : 64u; }   // (these are numbered by the KiB of their chunks)
constexpr uint32_t kMaxUnitChunks = 4;           // chunks of a unit (kEncUnit)
// Worker warps per block: the joined codes take half a register per symbol of a lane and coded stream; with the two service
// warps that makes 5 warps of 96 registers per scheduler for 32 or fewer of them, 4 of 128 for more.  kEncAny gets the 128
// with one coded stream too (with 18 workers it spills: BF16 weights at 1 KiB 83 -> 90 us, at 7 KiB 97 -> 106 us).
constexpr uint32_t kServiceWarps = 2;
__host__ __device__ constexpr uint32_t enc_max_workers(int shape, int n_huff) { return shape == kEncBig ? 16u : n_huff == 2 || shape == kEncAny || shape >= kEncSolo80 ? 14u : 18u; }

__device__ __forceinline__ uint32_t add_low_byte(uint32_t x, uint32_t acc) { return __dp4a(x, 1u, acc); }
// Joins the table entries of two neighbouring symbols: codes behind one another in bits 31..8, length in bits 7..0.
__device__ __forceinline__ uint32_t join_codes(uint32_t a, uint32_t b)
{
    return add_low_byte(b, a | (__funnelshift_r(b, 0, a) & 0xFFFFFF00u));   // the funnel shift takes the low five bits of a: its length
}

// Phase B for one coded stream: looks up the lane's symbols (its row of 2 N staged bytes at row_s, 16-byte pieces
// XORed with `swz`), leaves the joined codes in e[] and returns the lane's bit count.  longer: not 0 when some four
// neighbouring codes are longer than 32 bits together.  `ok` turns false when a symbol has no code: the caller then uses
// lookup_checked.  Tiles are multiples of 256 symbols, so only a lane of 48 can be filled in part, by 16 or 32 of them: what
// lies behind is left by another tile.
template <uint32_t N>
__device__ __forceinline__ uint32_t lookup_quick(uint32_t (&e)[N], const uint32_t row_s, const uint32_t swz,
                                                 const uint32_t tab_s, const uint32_t n_my, bool& ok, uint32_t& longer)
{
    uint32_t bits = 0, seen = 0, over = 0;
#pragma unroll
    for (uint32_t p = 0; p < N / 8; ++p) {
        if (N == 24 && 16 * p >= n_my) {
#pragma unroll
            for (uint32_t i = 0; i < 8; ++i) e[8 * p + i] = 0;
            bits += 4 * 95;
            continue;
        }
        const uint4 v = lds128(row_s + ((p ^ swz) << 4));
        const uint32_t q[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (uint32_t i = 0; i < 4; ++i) {
            // tab_s + 4 * byte k of the word, in one dot product
            const uint32_t a0 = lds32(__dp4a(q[i], 0x00000004u, tab_s)), a1 = lds32(__dp4a(q[i], 0x00000400u, tab_s));
            const uint32_t a2 = lds32(__dp4a(q[i], 0x00040000u, tab_s)), a3 = lds32(__dp4a(q[i], 0x04000000u, tab_s));
            const uint32_t e0 = join_codes(a0, a1), e1 = join_codes(a2, a3);
            seen |= e0 | e1;
            e[8 * p + 2 * i] = e0;
            e[8 * p + 2 * i + 1] = e1;
            const uint32_t len = e0 + e1 + 95;               // bit 7 of it: more than 32 bits
            over |= len;
            bits = add_low_byte(len, bits);
        }
    }
    ok = (seen & (3u * kNoCode)) == 0;                           // one or two of them in a pair
    longer = over & 0x80u;
    return bits - 95 * (N / 2);
}

// The same symbol by symbol for tiles that need care: a ragged end (only the first n_my symbols count) and symbols
// without a code (they take no bits; `bad` is set).
template <uint32_t N>
__device__ __forceinline__ uint32_t lookup_checked(uint32_t (&e)[N], const uint32_t row_s, const uint32_t swz,
                                                   const uint32_t tab_s, const uint32_t n_my, bool& bad)
{
    uint32_t bits = 0;
#pragma unroll
    for (uint32_t p = 0; p < N / 8; ++p) {
        const uint4 v = lds128(row_s + ((p ^ swz) << 4));
        const uint32_t q[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (uint32_t i = 0; i < 4; ++i) {
            uint32_t a[4];
#pragma unroll
            for (uint32_t k = 0; k < 4; ++k) {
                a[k] = 0;
                if (16 * p + 4 * i + k < n_my) a[k] = lds32(tab_s + 4u * __byte_perm(q[i], 0, 0x4440 + k));
                if (a[k] & kNoCode) { bad = true; a[k] = 0; }
            }
            e[8 * p + 2 * i] = join_codes(a[0], a[1]);
            e[8 * p + 2 * i + 1] = join_codes(a[2], a[3]);
            bits = add_low_byte(e[8 * p + 2 * i] + e[8 * p + 2 * i + 1], bits);
        }
    }
    return bits;
}

// Phase C for one coded stream: ORs the joined codes into shared memory from bit `at` of the piece at piece_s on.
// QUADS: four codes at a time (no four neighbouring ones in the warp are longer than 32 bits), else two at a time (choosing
// anew for every four costs more than it saves: FP8 505 against 474 us).
template <bool QUADS, uint32_t N>
__device__ __forceinline__ void emit_codes(const uint32_t (&e)[N], const uint32_t piece_s, const uint32_t at)
{
    uint32_t addr = piece_s + 4 * (at >> 5), t = at & 31u, w = 0;
#pragma unroll
    for (uint32_t i = 0; i < N / 2; ++i) {
        const uint32_t e0 = e[2 * i], e1 = e[2 * i + 1], c0 = e0 & 0xFFFFFF00u, c1 = e1 & 0xFFFFFF00u;
        if (QUADS) {
            put_bits(c0 | __funnelshift_r(c1, 0, e0), add_low_byte(e0 + e1, t), t, w, addr);
        } else {
            put_bits(c0, add_low_byte(e0, t), t, w, addr);
            put_bits(c1, add_low_byte(e1, t), t, w, addr);
        }
    }
    if (t & 31u) red_or(addr, w);
}

// The lanes whose n_my staged symbols all equal `symbol`; the whole warp calls it.  Rarely needed (tiles that might be
// constant), so it is kept out of line.
static __device__ __noinline__ uint32_t lanes_of_only(uint32_t row_s, uint32_t swz, uint32_t n_my, uint32_t symbol)
{
    bool same = true;
    for (uint32_t k = 0; k < n_my; k += 4) {
        const uint32_t left = min(n_my - k, 4u);
        const uint32_t x = lds32(row_s + (((k >> 4) ^ swz) << 4) + (k & 15u)) ^ (symbol * 0x01010101u);
        same = same && (x & (0xFFFFFFFFu >> (32 - 8 * left))) == 0;
    }
    return __ballot_sync(0xFFFFFFFFu, same);
}

__device__ __forceinline__ uint32_t warp_scan(uint32_t v, uint32_t lane)
{
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t x = __shfl_up_sync(0xFFFFFFFFu, v, o);
        if (lane >= (uint32_t)o) v += x;
    }
    return v;
}

template <int FMT, bool H0, bool H1, int SHAPE>
__global__ void __launch_bounds__((enc_max_workers(SHAPE, (H0 ? 1 : 0) + (H1 ? 1 : 0)) + kServiceWarps) * 32, 1)
encode_kernel(const __grid_constant__ EncParams P)
{
    constexpr int kHuff = (H0 ? 1 : 0) + (H1 ? 1 : 0);
    constexpr int kTabs = kHuff ? kHuff : 1;
    constexpr uint32_t kMaxW = enc_max_workers(SHAPE, kHuff);
    constexpr bool kUnit = SHAPE == kEncUnit, kSolo = SHAPE == kEncSolo || SHAPE >= kEncSolo80;   // kSolo: a unit is one full tile
    constexpr bool kAny = SHAPE >= kEncAny && SHAPE <= kEncBig;
    constexpr uint32_t kN = enc_lane_syms(SHAPE);               // symbols of a lane
    constexpr uint32_t kTileSyms = 32 * kN;
    extern __shared__ __align__(16) uint8_t smem[];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t n_workers = (blockDim.x >> 5) - kServiceWarps;
    const uint32_t T = kSolo ? 1u : P.tiles, teams = kSolo ? n_workers : P.teams;
    const uint32_t unit_syms = kSolo ? kTileSyms : P.unit_syms, unit_chunks = kUnit ? P.unit_chunks : 1u;

    // shared: rings[teams] | input buffers[workers] | tables[kTabSlots][kTabs][256]
    const uint32_t rings_s = smem_u32(smem);
    const uint32_t bufs_s = rings_s + teams * 16 * P.ring16;
    const uint32_t tabs_s = bufs_s + n_workers * P.buf_bytes;

    __shared__ EncItem s_item[kTabSlots];
    __shared__ uint32_t s_fill[kTabSlots][2];
    __shared__ uint32_t s_slot[kEncRing], s_c0[kEncRing], s_ticket[kEncRing], s_tensor[kEncRing], s_tot[kEncRing];
    __shared__ uint32_t s_bits[kEncRing][kTabs][kMaxW * (kUnit ? kMaxUnitChunks : 1)], s_src[kEncRing][kMaxW];
    __shared__ uint32_t s_tile[2][kTabs][kMaxW];
    __shared__ uint32_t s_freed_seq, s_end, s_fail;
    __shared__ uint64_t mb_in[kMaxW], mb_team[kMaxW], mb_info[kEncRing], mb_size[kEncRing], mb_posted[kEncRing], mb_done[kEncRing];

    if (threadIdx.x == 0) {
        s_freed_seq = s_fail = 0;
        s_end = 0xFFFFFFFFu;
        for (uint32_t i = 0; i < kEncRing; ++i) { mbar_init(&mb_info[i], 1); mbar_init(&mb_size[i], teams); mbar_init(&mb_posted[i], 1); mbar_init(&mb_done[i], n_workers); }
        for (uint32_t i = 0; i < n_workers; ++i) { mbar_init(&mb_in[i], 1); mbar_init(&mb_team[i], T); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();

    auto vol32 = [](const uint32_t* p) { return *reinterpret_cast<const volatile uint32_t*>(p); };
    auto counters = [&](const uint32_t index) -> TensorCounters* { return P.counters + index; };
    const EncItem* const items = P.items ? P.items : &P.one;

    if (warp == n_workers) {
        // =========================== the dealer warp ===========================
        // Takes tickets, turns them into batches and publishes those; posts the sizes of batches that have been packed.
        uint32_t published = 0, posted = 0;                      // batches of this block
        uint32_t ticket = 0;                                     // lane 0: ticket taken for the next batch
        bool have_ticket = false;
        uint32_t tcur = 0, next_first = 0;                       // tensor of the last ticket (tickets only grow), first batch of the next one
        uint32_t slot = 0, slot_tensor = kNoSlot;                // the newest table slot and whose it is
        uint32_t slot_last[kTabSlots] = {};                      // 1 + last batch that uses the slot
        bool ended = false;
        uint32_t idle = 0;
        for (;;) {
            bool did = false;
            // ---- sizes of batches that have been packed ----
            while (posted < published && __all_sync(0xFFFFFFFFu, mbar_test(&mb_size[posted % kEncRing], (posted / kEncRing) & 1u))) {
                const uint32_t r = posted % kEncRing;
                uint32_t p16 = 0;
#pragma unroll
                for (int h = 0; h < kHuff; ++h)
                    for (uint32_t k = 0; k < unit_chunks; ++k) p16 += lane < teams ? (s_bits[r][h][lane * unit_chunks + k] + 127) >> 7 : 0u;
                const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, p16);
                if (lane == 0) {
                    if (kHuff) st_flag(P.flags + s_ticket[r], (s_c0[r] == 0 ? kFlagPrefix : kFlagAggregate) | total);
                    s_tot[r] = total;
                    mbar_arrive(&mb_posted[r]);
                }
                __syncwarp();
                ++posted;
                did = true;
            }
            if (ended && posted == published) break;
            // ---- a new batch ----
            const uint32_t freed = __shfl_sync(0xFFFFFFFFu, vol32(&s_freed_seq), 0);
            if (!ended && published < posted + min(P.ahead, 2u) && published < freed + kEncRing) {
                if (!have_ticket && lane == 0) ticket = atomicAdd(&P.ctl->ticket, 1u);
                have_ticket = true;
                const uint32_t g = __shfl_sync(0xFFFFFFFFu, ticket, 0);
                const uint32_t r = published % kEncRing;
                if (g >= P.total_batches) {
                    ended = true;
                    if (lane == 0) {
                        s_slot[r] = kNoSlot;
                        *reinterpret_cast<volatile uint32_t*>(&s_end) = published;
                        mbar_arrive(&mb_info[r]);
                    }
                    __syncwarp();
                    continue;
                }
                // the last tensor that starts at or before the batch (tensors without chunks share their start with the next)
                if (P.items && g >= next_first) {
                    for (;;) {
                        const uint32_t cand = tcur + 1 + lane;
                        const uint32_t k = __popc(__ballot_sync(0xFFFFFFFFu, cand < P.n_tensors && P.first_batch[cand] <= g));
                        tcur += k;
                        if (k < 32) break;
                    }
                    next_first = tcur + 1 < P.n_tensors ? P.first_batch[tcur + 1] : 0xFFFFFFFFu;
                }
                bool publish = true;
                if (tcur != slot_tensor) {
                    // another tensor: it takes the next slot once every batch that uses it has left the block
                    const uint32_t ns = (slot + 1) % kTabSlots;
                    const uint32_t last = ns == 0 ? slot_last[0] : ns == 1 ? slot_last[1] : ns == 2 ? slot_last[2] : slot_last[3];
                    publish = freed >= last;
                    if (publish) {
                        slot = ns;
                        slot_tensor = tcur;
                        const unsigned long long* src = reinterpret_cast<const unsigned long long*>(items + tcur);
                        unsigned long long* dst = reinterpret_cast<unsigned long long*>(&s_item[ns]);
                        for (uint32_t i = lane; i < sizeof(EncItem) / 8; i += 32) dst[i] = src[i];
                        const EncTables& E = P.tables ? P.tables[items[tcur].table] : P.table;
                        uint32_t h = 0;
#pragma unroll
                        for (int s = 0; s < 2; ++s) {
                            if (!(s == 0 ? H0 : H1)) continue;
#pragma unroll
                            for (uint32_t i = 0; i < 4; ++i) {
                                const uint32_t two = reinterpret_cast<const uint32_t*>(E.enc[s])[lane + 32 * i];
                                sts64(tabs_s + 1024 * (kTabs * ns + h) + 8 * (lane + 32 * i), enc_entry(two & 0xFFFFu), enc_entry(two >> 16));
                            }
                            if (lane == 0) s_fill[ns][h] = E.fill[s];
                            ++h;
                        }
                        __syncwarp();
                    }
                }
                if (publish) {
                    const EncItem& I = s_item[slot];
                    const uint32_t c0 = (g - I.first_batch) * teams;
                    ++published;
                    have_ticket = false;
#pragma unroll
                    for (uint32_t k = 0; k < kTabSlots; ++k) if (k == slot) slot_last[k] = published;
                    if (lane == 0) {
                        s_slot[r] = slot; s_c0[r] = c0; s_ticket[r] = g; s_tensor[r] = tcur;
                        mbar_arrive(&mb_info[r]);
                    }
                    __syncwarp();
                    // With two coded streams to a tile, the batch's input travels to the L2: a worker requests its tile when it has
                    // staged the one before, and what is left of its turn is too short for DRAM's latency (two inputs of a delta;
                    // 872 MB 582 -> 553 us; FP8 with both streams coded 244 -> 234 us).  Elsewhere it gains nothing, and chunks of
                    // several tiles lose 3 %.
                    if (kHuff == 2 && T == 1 && lane < 2) {
                        const uint8_t* const src = lane ? I.base : I.in;
                        const unsigned long long lo = 2ull * unit_syms * c0, left = I.input_bytes > lo ? I.input_bytes - lo : 0ull;
                        const uint32_t n = (uint32_t)min(left, 2ull * unit_syms * teams) & ~15u;
                        if (src && n) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" :: "l"(src + lo), "r"(n) : "memory");
                    }
                    if (P.ahead > 2) {                           // the next one's ticket travels until it is looked at
                        if (lane == 0) ticket = atomicAdd(&P.ctl->ticket, 1u);
                        have_ticket = true;
                    }
                    if (c0 == 0) {
                        // the fixed parts of the tensor's container: code lengths, padding of the chunk offset table, tail
                        // padding of raw bodies
                        uint32_t h = 0;
#pragma unroll
                        for (int s = 0; s < 2; ++s) {
                            if (s == 0 ? H0 : H1) {
                                for (uint32_t v = lane; v < 256; v += 32)
                                    I.out[I.lay.section_off[s] + v] = (uint8_t)(lds32(tabs_s + 1024 * (kTabs * slot + h) + 4 * v) & 15u);
                                const uint32_t padded = (I.n_chunks + 3) & ~3u;
                                for (uint32_t i = I.n_chunks + lane; i < padded; i += 32)
                                    reinterpret_cast<uint32_t*>(I.out + I.lay.chunk_off_tab[s])[i] = 0;
                                ++h;
                            } else {
                                const uint64_t lo = (I.n_syms + 7) & ~7ull, hi = (I.n_syms + 15) & ~15ull;
                                for (uint64_t i = lo + lane; i < hi; i += 32) I.out[I.lay.section_off[s] + i] = 0;
                            }
                        }
                    }
                    did = true;
                }
            }
            if (__shfl_sync(0xFFFFFFFFu, vol32(&s_fail), 0)) break;
            if (did) { idle = 0; continue; }
            if (++idle > P.spin_limit) { s_fail = 1; break; }
            __nanosleep(200);                                    // nothing to do right now: leave the issue slots to the workers
        }
    } else if (warp == n_workers + 1) {
        // =========================== the placer warp ===========================
        // Finds the place of the block's oldest batch without one by a look-back over other blocks' words, sends its pieces
        // there, gives the ring space back, and keeps the tensors' counters.
        if (blockIdx.x == 0)                                     // tensors without chunks are all header
            for (uint32_t t = lane; t < P.n_tensors; t += 32)
                if (items[t].n_chunks == 0) write_header(P, items[t], counters(items[t].index));
        uint32_t placed = 0, freed = 0;                          // batches of this block
        bool lb_on = false, lb_done = false;
        uint32_t lb_sum = 0, lb_pos = 0;
        uint32_t idle = 0;
        // chunks this block has placed, per tensor; added to the tensor's counters when the tensor changes
        uint32_t acc_t = kNoSlot, acc_n = 0;
        unsigned long long acc_bits[2] = {0, 0};                 // per lane: payload bits of those chunks
        auto flush_acc = [&]() {
            if (acc_n == 0) return;
#pragma unroll
            for (int h = 0; h < kHuff; ++h)
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc_bits[h] += __shfl_xor_sync(0xFFFFFFFFu, acc_bits[h], o);
            if (lane == 0) {
                const EncItem& I = items[acc_t];
                TensorCounters* tc = counters(I.index);
                if (H0) atomicAdd(&tc->payload_bits[0], acc_bits[0]);
                if (H1) atomicAdd(&tc->payload_bits[1], acc_bits[H0 ? 1 : 0]);
                __threadfence();
                const uint32_t before = atomicAdd(&tc->done, acc_n);
                if (before + acc_n == I.n_chunks) {              // whoever completes a tensor writes its header
                    __threadfence();
                    write_header(P, I, tc);
                }
            }
            __syncwarp();
            acc_n = 0;
            acc_bits[0] = acc_bits[1] = 0;
        };
        for (;;) {
            bool did = false;
            const uint32_t r = placed % kEncRing;
            if (!lb_on && __all_sync(0xFFFFFFFFu, mbar_test(&mb_posted[r], (placed / kEncRing) & 1u))) {
                lb_sum = 0;                                      // sizes are 16-byte units: chunk_off16 has 32 bits
                lb_pos = 1;                                      // lane i looks lb_pos + i batches back
                lb_done = !kHuff || s_c0[r] == 0;
                lb_on = true;
                did = true;
            }
            if (lb_on) {
                const EncItem& I = s_item[s_slot[r]];
                const uint32_t c0 = s_c0[r], total = s_tot[r];
                if (!lb_done) {
                    // One round: 32 * kLookWide predecessors at a time, newest first, up to the first one that already knows
                    // its prefix.  All loads of a round are in flight together.  The look-back stays inside the tensor.
                    unsigned long long* const flags = P.flags + s_ticket[r];
                    const uint32_t b = s_ticket[r] - I.first_batch;
                    unsigned long long f[kLookWide];
#pragma unroll
                    for (int k = 0; k < kLookWide; ++k) {
                        const uint32_t back = lb_pos + 32 * k + lane;
                        f[k] = back <= b ? ld_flag(flags - back) : kFlagPrefix;      // before batch 0: prefix 0
                    }
#pragma unroll
                    for (int k = 0; k < kLookWide; ++k) {
                        const uint32_t ready = __ballot_sync(0xFFFFFFFFu, (f[k] >> 62) != 0);
                        const uint32_t prefix = __ballot_sync(0xFFFFFFFFu, (f[k] >> 62) == 2);
                        const uint32_t first = prefix ? (uint32_t)__ffs(prefix) - 1 : 32u;
                        const uint32_t need = first == 32 ? 0xFFFFFFFFu : (0xFFFFFFFFu >> (31 - first));
                        if ((ready & need) != need) break;       // somebody has not posted yet: again from here later
                        lb_sum += __reduce_add_sync(0xFFFFFFFFu, lane <= first ? (uint32_t)f[k] : 0u);
                        lb_pos += 32;
                        did = true;
                        if (first != 32) { lb_done = true; break; }
                    }
                    if (lb_done && lane == 0) st_flag(flags, kFlagPrefix | ((unsigned long long)lb_sum + total));
                }
                if (lb_done && __all_sync(0xFFFFFFFFu, mbar_test(&mb_done[r], (placed / kEncRing) & 1u))) {
                    const uint32_t n_mine = min(teams, I.n_units - c0);
                    if (s_tensor[r] != acc_t) { flush_acc(); acc_t = s_tensor[r]; }
                    acc_n += min(n_mine * unit_chunks, I.n_chunks - c0 * unit_chunks);
                    if (kHuff) {
                        uint32_t mine = 0;
                        for (uint32_t k = 0; k < unit_chunks; ++k)
#pragma unroll
                            for (int h = 0; h < kHuff; ++h)
                                if (lane < n_mine) {
                                    const uint32_t bits = s_bits[r][h][lane * unit_chunks + k];
                                    mine += (bits + 127) >> 7;
                                    acc_bits[h] += bits;
                                }
                        const uint32_t off = lb_sum + warp_scan(mine, lane) - mine;
                        if (lane < n_mine && mine)
                            bulk_s2g(I.out + I.lay.payload_off + 16ull * off, rings_s + 16 * (lane * P.ring16 + s_src[r][lane]), 16 * mine);
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                        if (lane < n_mine) {
                            uint32_t at = off;
                            for (uint32_t k = 0; k < unit_chunks; ++k) {
                                const uint32_t c = (c0 + lane) * unit_chunks + k;
#pragma unroll
                                for (int h = 0; h < kHuff; ++h) {
                                    if (c < I.n_chunks) reinterpret_cast<uint32_t*>(I.out + I.lay.chunk_off_tab[H0 ? h : 1])[c] = at;
                                    at += (s_bits[r][h][lane * unit_chunks + k] + 127) >> 7;
                                }
                            }
                        }
                        // the block that owns the last chunk knows the size of the whole payload area
                        if (lane == 0 && c0 + n_mine == I.n_units) counters(I.index)->total16 = lb_sum + total;
                    }
                    __syncwarp();
                    ++placed;
                    lb_on = false;
                    did = true;
                }
            }
            if (__shfl_sync(0xFFFFFFFFu, vol32(&s_fail), 0)) break;
            // ---- ring space of batches that have been sent: the newest one's copies are given time until nothing else is to do ----
            if (freed < placed) {
                if (did) asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
                else asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
                __syncwarp();
                const uint32_t now = placed - (did ? 1u : 0u);
                did = did || now != freed;
                freed = now;
                if (lane == 0) *reinterpret_cast<volatile uint32_t*>(&s_freed_seq) = freed;
            } else if (freed == __shfl_sync(0xFFFFFFFFu, vol32(&s_end), 0)) {
                break;
            }
            if (did) { idle = 0; continue; }
            if (++idle > P.spin_limit) { s_fail = 1; break; }
            __nanosleep(50);
        }
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
        flush_acc();
    } else {
        // =========================== a worker warp ===========================
        // Bounded wait of the whole warp for a phase of an mbarrier; false on the failure flag or when the wait gives up.
        // (A try_wait sleeps in hardware until the phase completes or a time limit is reached.  With a hint of 2 us for that limit 872
        // MB of BF16 weights at 16 KiB take 425 us, without 419.)
        auto wait_phase = [&](uint64_t* bar, const uint32_t parity) -> bool {
            bool ok = mbar_try_wait(bar, parity);
            for (uint32_t k = 0; !ok && k < P.spin_limit; ++k) {
                if (vol32(&s_fail)) break;
                ok = mbar_try_wait(bar, parity);
            }
            return __all_sync(0xFFFFFFFFu, ok);                  // decisions of the whole warp: no lane may leave alone
        };
        const uint32_t my_team = kSolo ? warp : warp / T, tw = kSolo ? 0u : warp - my_team * T;    // my team, my tile of its unit
        uint32_t ph_team = 0;
        auto team_sync = [&]() -> bool {
            __syncwarp();
            if (lane == 0) mbar_arrive(&mb_team[my_team]);
            const bool ok = wait_phase(&mb_team[my_team], ph_team & 1u);
            ++ph_team;
            return ok;
        };
        const uint32_t t_lo = tw * kTileSyms;                                          // my tile in the unit,
        const uint32_t t_full = kAny ? min(kTileSyms, unit_syms - t_lo) : kTileSyms;   // and its symbols (a multiple of 256)
        const uint32_t buf_s = bufs_s + warp * P.buf_bytes;
        const uint32_t ring_s = rings_s + my_team * 16 * P.ring16;
        // Staged symbols.  Rows of 64 bytes: 16-byte piece p of row r sits at p ^ (r >> 1 & 3); group g (8 symbols) is half of a
        // piece of row g / 8.  Lane l's groups l + 32 i go to row 4 i + l / 8: from one i to the next the swizzle flips bit 1
        // of the piece index.  Rows of 48 bytes have no bank conflicts as they are.
        const uint32_t swz = kN == 64 ? (lane >> 1) & 3u : 0u;
        const uint32_t at0 = kN == 64 ? (lane >> 3) * 64 + ((((lane & 7) >> 1) ^ (lane >> 4)) << 4) + 8 * (lane & 1u) : 8 * lane;
        auto stage_at = [&](const uint32_t i) { return (kN == 64 ? at0 ^ ((i & 1u) << 5) : at0) + 256 * i; };
        // several chunks in a unit: the lanes of my chunk
        const uint32_t chunk_lanes = kUnit ? P.cs / kN : 32u, my_k = kUnit ? lane / chunk_lanes : 0u;
        uint32_t k_lane = my_k * chunk_lanes;
        // (Knowing that it is 0, the compiler keeps more over the loop than the kernels of two coded streams have registers
        // for: 144 bytes of spills against 74.)
        if (kAny) asm("" : "+r"(k_lane));

        bool loaded = false;                                     // the next tile's input has been requested
        uint32_t ph_in = 0;
        auto whole_tile = [&](const EncItem& I, const uint64_t s_lo) { return s_lo + t_full <= I.n_syms && 2 * (s_lo + t_full) <= I.input_bytes; };
        // Requests my tile of unit u of tensor I, if it is a complete one (the buffer is free: every lane has passed a __syncwarp).
        auto request = [&](const EncItem& I, const uint32_t u) {
            const uint64_t s_lo = (uint64_t)u * unit_syms + t_lo;
            if (u >= I.n_units || !whole_tile(I, s_lo)) return;
            if (lane == 0) {
                const bool two = I.base && P.base_buf;
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_expect_tx(&mb_in[warp], two ? 4 * t_full : 2 * t_full);
                bulk_g2s_addr(buf_s, I.in + 2 * s_lo, 2 * t_full, &mb_in[warp]);
                if (two) bulk_g2s_addr(buf_s + 2 * kTileSyms, I.base + 2 * s_lo, 2 * t_full, &mb_in[warp]);
            }
            loaded = true;
        };

        uint32_t ring_pos = 0, virt = 0;                         // ring position and its running (virtual) form, 16-byte units
        uint32_t vend = 0;                                       // lane k: virtual end of the last batch it with it % 32 == k
        uint32_t bad = 0;
        bool failed = false;
        for (uint32_t it = 0;; ++it) {
            const uint32_t r = it % kEncRing;
            if (!wait_phase(&mb_info[r], (it / kEncRing) & 1u)) { failed = true; break; }
            const uint32_t use = vol32(&s_slot[r]);
            if (use == kNoSlot) break;
            const EncItem& I = s_item[use];
            const uint32_t u = vol32(&s_c0[r]) + my_team;
            const bool active = u < I.n_units;
            const uint32_t tab_s = tabs_s + 1024 * kTabs * use;

            uint32_t e[kTabs][kN / 2];                             // joined codes of my symbols
            uint32_t mine[kTabs] = {}, end[kTabs] = {};          // bits of my symbols, and where they end in their chunk
            uint32_t chunk_bits[kTabs] = {};                     // bits of my chunk (0: constant)
            uint32_t longer[kTabs] = {};                         // not 0: some four neighbouring codes of the tile are longer than 32 bits
            const uint64_t s_lo = (uint64_t)u * unit_syms + t_lo;       // first symbol of the tile in its stream
            auto request_next = [&]() {                          // my tile of the next batch, if that is known already
                const uint32_t r1 = (it + 1) % kEncRing;
                if (!__all_sync(0xFFFFFFFFu, mbar_test(&mb_info[r1], ((it + 1) / kEncRing) & 1u))) return;
                const uint32_t use1 = vol32(&s_slot[r1]);
                if (use1 != kNoSlot) request(s_item[use1], vol32(&s_c0[r1]) + my_team);
            };
            if (active) {
                // ---- phase A ----
                const uint32_t t_syms = s_lo < I.n_syms ? (uint32_t)min((uint64_t)t_full, I.n_syms - s_lo) : 0u;
                const bool whole = whole_tile(I, s_lo);
                uint8_t* const raw0 = I.out + I.lay.section_off[0] + s_lo;
                uint8_t* const raw1 = I.out + I.lay.section_off[1] + s_lo;
                // With both streams coded (delta checkpoints: stretches of unchanged weights are constant chunks in both
                // streams) every staged word is compared with the fill symbol on the way; with one coded stream constant
                // tiles are rare and are found by their bit count.
                constexpr bool kSpotConstant = kHuff == 2;
                uint32_t fill4[2] = {0, 0}, differs[2] = {0, 0};
                if (kSpotConstant) {
                    fill4[0] = (s_fill[use][0] & 0xFFu) * 0x01010101u;
                    fill4[1] = (s_fill[use][1] & 0xFFu) * 0x01010101u;
                }
                auto stage = [&](const uint4 x, const uint32_t g, const uint32_t at, const bool on) {
                    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
                    uint32_t sy[2][2];
                    split16<FMT>(w, sy[0], sy[1]);
                    if (H0) sts64(buf_s + at, sy[0][0], sy[0][1]);
                    else if (!kAny || on) st_cs_v2(raw0 + 8 * g, make_uint2(sy[0][0], sy[0][1]));
                    if (H1) sts64(buf_s + (H0 ? kTileSyms : 0u) + at, sy[1][0], sy[1][1]);
                    else if (!kAny || on) st_cs_v2(raw1 + 8 * g, make_uint2(sy[1][0], sy[1][1]));
                    if (kSpotConstant && (!kAny || on)) {
                        differs[0] |= (sy[0][0] ^ fill4[0]) | (sy[0][1] ^ fill4[0]);
                        differs[1] |= (sy[1][0] ^ fill4[1]) | (sy[1][1] ^ fill4[1]);
                    }
                };
                auto x4 = [](const uint4 a, const uint4 b) { return make_uint4(a.x ^ b.x, a.y ^ b.y, a.z ^ b.z, a.w ^ b.w); };
                if (whole) {
                    if (!loaded) request(I, u);
                    if (!wait_phase(&mb_in[warp], ph_in & 1u)) { failed = true; break; }
                    ++ph_in;
                    loaded = false;
                    // (a tile that is not full is read and staged to its end all the same: what lies behind is not looked at)
                    uint4 x[kN / 8];
#pragma unroll
                    for (uint32_t i = 0; i < kN / 8; ++i) x[i] = lds128(buf_s + 16 * (lane + 32 * i));
                    if (I.base) {
#pragma unroll
                        for (uint32_t i = 0; i < kN / 8; ++i) {
                            const uint32_t on = kAny ? min(i, t_full / 256 - 1) : i;
                            x[i] = x4(x[i], P.base_buf ? lds128(buf_s + 2 * kTileSyms + 16 * (lane + 32 * i)) : ld_nc_v4(I.base + 2 * s_lo + 16 * (lane + 32 * on)));
                        }
                    }
                    __syncwarp();                                // everybody has read: the buffer takes the staged symbols
#pragma unroll
                    for (uint32_t i = 0; i < kN / 8; ++i) stage(x[i], lane + 32 * i, stage_at(i), 256 * i < t_full);
                } else {
                    for (uint32_t i = 0; 256 * i + 8 * lane < t_syms; ++i) {
                        const uint32_t g = lane + 32 * i;
                        uint4 x = load16_guarded(I.in, 2 * (s_lo + 8ull * g), I.input_bytes);
                        if (I.base) x = x4(x, load16_guarded(I.base, 2 * (s_lo + 8ull * g), I.input_bytes));
                        stage(x, g, stage_at(i), true);
                    }
                }
                __syncwarp();

                // ---- phase B ----
                const uint32_t n_my = t_syms > kN * lane ? min(kN, t_syms - kN * lane) : 0u;
                const uint32_t k_syms = kUnit ? (t_syms > my_k * P.cs ? min(P.cs, t_syms - my_k * P.cs) : 0u) : t_syms;   // of my chunk in the tile
                uint32_t tile_bits[kTabs];
#pragma unroll
                for (int h = 0; h < kHuff; ++h) {
                    const uint32_t row = buf_s + h * kTileSyms + lane * kN;
                    const uint32_t fill = s_fill[use][h], fill_len = fill >> 8;
                    bool constant = false;
                    if (kSpotConstant && whole && fill_len <= kLmax && __all_sync(0xFFFFFFFFu, differs[h] == 0)) {
                        // nothing but the fill symbol (which has the all-zero code)
#pragma unroll
                        for (uint32_t i = 0; i < kN / 2; ++i) e[h][i] = kN != 48 || 16 * (i / 8) < n_my ? 2 * fill_len : 0u;
                        mine[h] = n_my * fill_len;
                        constant = true;
                        longer[h] = fill_len > 8;
                    } else {
                        bool ok = false;
                        uint32_t mine_longer = 0;
                        if (whole) {
                            if (!kAny || n_my) {
                                mine[h] = lookup_quick(e[h], row, swz, tab_s + 1024 * h, n_my, ok, mine_longer);
                            } else {
                                ok = true;
                            }
                        }
                        longer[h] = __reduce_or_sync(0xFFFFFFFFu, mine_longer);
                        if (!__all_sync(0xFFFFFFFFu, ok)) {
                            longer[h] = 1;
                            bool no_code = false;
                            mine[h] = lookup_checked(e[h], row, swz, tab_s + 1024 * h, n_my, no_code);
                            if (no_code) bad = I.index + 1;
                        }
                    }
                    const uint32_t inc = warp_scan(mine[h], lane);
                    uint32_t bits = __shfl_sync(0xFFFFFFFFu, inc, 31), lead = 0;         // of my chunk in the tile; of the chunks before it
                    if (kUnit) {
                        lead = __shfl_sync(0xFFFFFFFFu, inc, k_lane ? k_lane - 1 : 0);
                        if (k_lane == 0) lead = 0;
                        bits = __shfl_sync(0xFFFFFFFFu, inc, k_lane + chunk_lanes - 1) - lead;
                    }
                    const bool maybe = !constant && k_syms && bits == k_syms * fill_len;
                    if (__any_sync(0xFFFFFFFFu, maybe)) {
                        const uint32_t want = (0xFFFFFFFFu >> (32 - chunk_lanes)) << k_lane;
                        if ((lanes_of_only(row, swz, n_my, fill & 0xFFu) & want) == want) constant = constant || maybe;
                    }
                    end[h] = inc - lead;
                    // tiles without symbols (behind the end of a ragged chunk) do not keep a chunk from being constant
                    tile_bits[h] = bits | ((constant || k_syms == 0) ? kConstTile : 0u);
                }
                __syncwarp();                                    // the staged symbols are used up
                request_next();
                if (T == 1) {
#pragma unroll
                    for (int h = 0; h < kHuff; ++h) chunk_bits[h] = (tile_bits[h] & kConstTile) ? 0u : tile_bits[h];
                } else if (kHuff) {
                    // every warp of the team learns the bit counts of the chunk's tiles (the team meets once more before anybody
                    // can write the same buffer again)
                    if (lane == 0)
#pragma unroll
                        for (int h = 0; h < kHuff; ++h) s_tile[it & 1u][h][warp] = tile_bits[h];
                    if (!team_sync()) { failed = true; break; }
#pragma unroll
                    for (int h = 0; h < kHuff; ++h) {
                        const uint32_t v = lane < T ? s_tile[it & 1u][h][my_team * T + lane] : kConstTile;
                        const uint32_t a = warp_scan(v & ~kConstTile, lane);
                        const bool none = __all_sync(0xFFFFFFFFu, (v & kConstTile) != 0);
                        const uint32_t bits = __shfl_sync(0xFFFFFFFFu, a, 31);
                        chunk_bits[h] = none ? 0u : bits;
                        end[h] += __shfl_sync(0xFFFFFFFFu, a - (v & ~kConstTile), tw);
                    }
                }
            }

            // ---- the pieces: their sizes are posted, they get a stretch of the ring (every warp of the team follows the allocation) ----
            uint32_t p16[kTabs], total = 0, my_at = 0;           // my chunk's pieces; the unit's; where mine start among them
#pragma unroll
            for (int h = 0; h < kHuff; ++h) { p16[h] = (chunk_bits[h] + 127) >> 7; total += p16[h]; }
            if (kUnit) {
                const uint32_t own = total;
                total = 0;
                for (uint32_t k = 0; k < unit_chunks; ++k) {
                    const uint32_t x = __shfl_sync(0xFFFFFFFFu, own, k * chunk_lanes);
                    if ((int)k < (int)my_k) my_at += x;
                    total += x;
                }
            }
            if (ring_pos + total > P.ring16) { virt += P.ring16 - ring_pos; ring_pos = 0; }
            const uint32_t piece_at = ring_pos;
            ring_pos += total;
            virt += total;
            if (lane == (it & 31u)) vend = virt;
            if (tw == 0) {
                if (lane == k_lane) {
#pragma unroll
                    for (int h = 0; h < kHuff; ++h) s_bits[r][h][my_team * unit_chunks + my_k] = chunk_bits[h];
                }
                if (kUnit) __syncwarp();
                if (lane == 0) {
                    s_src[r][my_team] = piece_at;
                    mbar_arrive(&mb_size[r]);
                }
            }
            // ---- phase C ----
            if (kHuff && active) {
                if (total) {
                    bool room = false;
                    for (uint32_t k = 0; k < P.spin_limit && !room; ++k) {   // every value the same in all lanes
                        const uint32_t f = __shfl_sync(0xFFFFFFFFu, vol32(&s_freed_seq), 0);
                        const uint32_t freed_virt = __shfl_sync(0xFFFFFFFFu, vend, (f - 1) & 31u);
                        room = f == it || virt - (f ? freed_virt : 0u) <= P.ring16;
                        if (room || __shfl_sync(0xFFFFFFFFu, vol32(&s_fail), 0)) break;
                        __nanosleep(50);
                    }
                    if (!room) { failed = true; break; }
                    // my share of the pieces starts from zero
                    for (uint32_t q = tw * 32 + lane; q < total; q += 32 * T) sts128_zero(ring_s + 16 * (piece_at + q));
                }
                // The team meets for a constant chunk too, though nothing was zeroed: the next batch in which it has a chunk may
                // be two batches on (a tensor's last batch need not have one for every team), where the tiles' bit counts go
                // into the same buffer again, and nobody may still be reading them.
                if (T == 1) __syncwarp();
                else if (!team_sync()) { failed = true; break; }
                const uint32_t c = u * unit_chunks + my_k;
#pragma unroll
                for (int h = 0; h < kHuff; ++h) {
                    const int s = H0 ? h : 1;
                    uint8_t* const tab = I.out + I.lay.sub_end_tab[s] + (uint64_t)(32 * P.sub_width) * c;
                    auto put_end = [&](const uint32_t i, const uint32_t at) {
                        if (kSolo || P.sub_width == 2) reinterpret_cast<uint16_t*>(tab)[i] = (uint16_t)at;
                        else reinterpret_cast<uint32_t*>(tab)[i] = at;
                    };
                    if (kUnit) {
                        // subchunks are 16 or 32 symbols: a lane ends four, or two
                        uint32_t at = end[h] - mine[h];
                        const uint32_t two = P.sub >> 5;
#pragma unroll
                        for (uint32_t p = 0; p < kN / 16; ++p) {
#pragma unroll
                            for (uint32_t i = 0; i < 8; ++i) at = add_low_byte(e[h][8 * p + i], at);
                            if (c < I.n_chunks && !(two & ~p)) put_end(((4 * (lane - k_lane) + p + 1) >> two) - 1, chunk_bits[h] ? at : 0u);
                        }
                    } else if (kAny) {
                        // subchunks end where a lane has added up a multiple of 16 symbols
                        uint32_t at = end[h] - mine[h];
#pragma unroll
                        for (uint32_t p = 0; p < kN / 16; ++p) {
#pragma unroll
                            for (uint32_t i = 0; i < 8; ++i) at = add_low_byte(e[h][8 * p + i], at);
                            const uint32_t k = t_lo + kN * lane + 16 * (p + 1), i = __umulhi(k, P.sub_magic);
                            if (k <= P.cs && i * P.sub == k) put_end(i - 1, chunk_bits[h] ? at : 0u);
                        }
                    } else {
                        // T lanes are a subchunk: lane g of the chunk (counting through its tiles) ends subchunk (g + 1) / T - 1 if T divides g + 1
                        const uint32_t g1 = tw * 32 + lane + 1, i = kSolo ? g1 : g1 / T;
                        if (i * T == g1) put_end(i - 1, chunk_bits[h] ? end[h] : 0u);
                    }
                    if (chunk_bits[h] && (!(kAny || kUnit) || mine[h])) {
                        const uint32_t piece_s = ring_s + 16 * (piece_at + my_at + (h ? p16[0] : 0u));
                        if (longer[h] == 0) emit_codes<true>(e[h], piece_s, end[h] - mine[h]);
                        else emit_codes<false>(e[h], piece_s, end[h] - mine[h]);
                    }
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            __syncwarp();
            if (lane == 0) mbar_arrive(&mb_done[r]);
        }
        if (failed) s_fail = 1;
        if (loaded) mbar_wait(&mb_in[warp], ph_in & 1u, P.spin_limit);   // a copy that was requested must land before the block leaves
        if (bad && raise_status(P.ctl, 0, ZC_E_NO_CODE)) P.ctl->failed = bad;
    }
    __syncthreads();
    if (s_fail && threadIdx.x == 0) raise_status(P.ctl, 0, ZC_E_DEVICE_TIMEOUT);
}

// ---- launchers, one per element format (each in an object of its own, see zc_encode_fmt.cu) ----
struct EncRanges { const void* in; size_t in_bytes; const void* out; size_t out_bytes; const void* ws; size_t ws_bytes; };

#define ZC_ENC_DECLARE(NAME)                                                                                              \
    cudaError_t enc_launch_##NAME(int shape, uint32_t grid, uint32_t threads, size_t smem, cudaStream_t st,               \
                                  const EncParams& P, const EncRanges& R);                                                \
    void enc_debug_counts_##NAME(uint32_t out[2]);
ZC_ENC_DECLARE(bf16)
ZC_ENC_DECLARE(fp8)
ZC_ENC_DECLARE(scale)
ZC_ENC_DECLARE(fp4)
#undef ZC_ENC_DECLARE

}  // namespace zc
