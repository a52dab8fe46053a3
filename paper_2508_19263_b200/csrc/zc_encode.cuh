// Encoder kernel: field split, code lookup, bit packing and placement of the chunks in one pass over the input.
//
// Work unit of a warp: a tile, 32 lanes x n consecutive symbols of one chunk.  n is the largest of 64, 48, 32, 16 that
// divides the subchunk length, so a subchunk is T = sub / n lanes long and a chunk is T tiles (T = 1 up to 4 KiB chunks).
// Packing needs no serial walk over a subchunk: once every lane knows how many bits its symbols take, prefix sums give
// every lane its bit position.  T warps form a team that codes one chunk together (T = 1: nothing to agree on); a block
// is several teams plus one service warp, and its batch is as many consecutive chunks of a tensor as it has teams.
//   A  the tile's input arrives in shared memory by a bulk asynchronous copy requested a tile ahead; it is split in
//      registers, the raw stream is stored as it is, the coded stream goes back into the same buffer as one row of n bytes
//      per lane (16-byte pieces swizzled so that neither side has bank conflicts)
//   B  every lane looks up its symbols and keeps the codes of two neighbouring symbols, joined, in one register each
//      (24 bits of code, 5 bits of length), adding up the bits; the warp scans the bit counts
//   C  the chunk's size is posted, subchunk ends are written, and every lane ORs its codes into the chunk's piece in the
//      team's output ring in shared memory, at their final bit position
// Pieces lie in the ring exactly as they will lie in the payload area.  Once a batch's place is known the service warp
// sends each team's piece there with one bulk copy (cp.async.bulk shared -> global).  The place is the sum of the sizes
// of all earlier batches of the tensor, found by a look-back over one word per batch; workers never wait for it, only
// for room in their ring (several chunks deep).
#pragma once
#include "zc_device.cuh"

namespace zc {

// Per symbol: the code left-aligned in bits 31..20 and its length in bits 3..0; a symbol without a code is kNoCode.
struct EncTables {
    uint32_t enc[2][256];
    uint32_t fill[2];                            // fill symbol (the one with the all-zero code) | its code length << 8
    uint32_t pad[2];
};

// One tensor of a launch.
struct EncItem {
    const uint8_t* in;
    const uint8_t* base;                         // XOR-delta form: what is coded is in XOR base; or null
    uint8_t* out;
    uint64_t input_bytes, n_syms, n_elems;
    Layout lay;
    uint32_t n_chunks;
    uint32_t first_batch;                        // batches of all earlier tensors of the launch
    uint32_t index;                              // position in the caller's arrays (counters, error reports)
    uint32_t table;                              // its code tables among the uploaded ones (tensors may share a codebook)
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
    uint32_t lane_syms, tiles;                   // n, T
    uint32_t team, teams;                        // warps per chunk (T, or fewer: then each takes several tiles), chunks per batch
    uint32_t ring16;                             // a team's output ring, in 16-byte units
    uint32_t n_tensors, total_batches;
    uint32_t ahead;                              // batches a block may hold beyond those it has packed
    uint32_t spin_limit;                         // polls after which a bounded wait gives up
    uint32_t any_base;                           // some tensor has a base: every worker has a second input buffer
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

// Kernel shapes: lanes of 64 symbols and one warp per chunk (4 KiB chunks); lanes of 64 symbols and a warp per tile (chunks
// of 8, 12, 16, .. KiB); everything else.
constexpr int kEncSolo64 = 0, kEncTeam64 = 1, kEncAny = 2;
// Worker warps per block: the joined codes take 32 registers per lane and coded stream; with the service warp that makes
// 6 warps of 80 registers per scheduler with one coded stream, 4 of 128 with two.
__host__ __device__ constexpr uint32_t enc_max_workers(int n_huff) { return n_huff == 2 ? 15u : 23u; }
constexpr uint32_t kEncMaxTeam = 16;

__device__ __forceinline__ uint32_t add_low_byte(uint32_t x, uint32_t acc) { return __dp4a(x, 1u, acc); }
// Joins the table entries of two neighbouring symbols: codes behind one another in bits 31..8, length in bits 7..0.
__device__ __forceinline__ uint32_t join_codes(uint32_t a, uint32_t b)
{
    return add_low_byte(b, a | (__funnelshift_r(b, 0, a) & 0xFFFFFF00u));   // the funnel shift takes the low five bits of a: its length
}

// Phase B for one coded stream: looks up the lane's symbols (its row of 16 * parts staged bytes at row_s, 16-byte pieces
// XORed with `swz`), leaves the joined codes in e[] and returns the lane's bit count.  `ok` turns false when a symbol has
// no code: the caller then uses lookup_checked.
__device__ __forceinline__ uint32_t lookup_quick(uint32_t (&e)[32], const uint32_t row_s, const uint32_t swz, const uint32_t parts,
                                                 const uint32_t tab_s, bool& ok, bool& long_quad)
{
    uint32_t bits = 0, seen = 0, over = 0;
#pragma unroll
    for (uint32_t p = 0; p < 4; ++p) {
        if (p < parts) {
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
    }
    ok = (seen & (3u * kNoCode)) == 0;                           // one or two of them in a pair
    long_quad = (over & 0x80u) != 0;
    return bits - 4 * 95 * parts;
}

// The same symbol by symbol for tiles that need care: a ragged end (only the first n_my symbols count) and symbols
// without a code (they take no bits; `bad` is set).
__device__ __forceinline__ uint32_t lookup_checked(uint32_t (&e)[32], const uint32_t row_s, const uint32_t swz, const uint32_t parts,
                                                   const uint32_t tab_s, const uint32_t n_my, bool& bad)
{
    uint32_t bits = 0;
#pragma unroll
    for (uint32_t p = 0; p < 4; ++p) {
        if (p < parts) {
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
    }
    return bits;
}

// Phase C for one coded stream: ORs the joined codes into shared memory from bit `at` of the piece at piece_s on.
// QUADS: four codes at a time (no group of four in the warp is longer than 32 bits), else two at a time.
template <bool QUADS>
__device__ __forceinline__ void emit_codes(const uint32_t (&e)[32], const uint32_t parts, const uint32_t piece_s, const uint32_t at)
{
    uint32_t addr = piece_s + 4 * (at >> 5), t = at & 31u, w = 0;
#pragma unroll
    for (uint32_t p = 0; p < 4; ++p) {
        if (p < parts) {
#pragma unroll
            for (uint32_t i = 0; i < 4; ++i) {
                const uint32_t e0 = e[8 * p + 2 * i], e1 = e[8 * p + 2 * i + 1], c0 = e0 & 0xFFFFFF00u, c1 = e1 & 0xFFFFFF00u;
                if (QUADS) {
                    put_bits(c0 | __funnelshift_r(c1, 0, e0), add_low_byte(e0 + e1, t), t, w, addr);
                } else {
                    put_bits(c0, add_low_byte(e0, t), t, w, addr);
                    put_bits(c1, add_low_byte(e1, t), t, w, addr);
                }
            }
        }
    }
    if (t & 31u) red_or(addr, w);
}

// Whether the n_my staged symbols of every lane all equal `symbol`; the whole warp calls it.  Rarely needed (tiles that
// might be constant), so it is kept out of line.
static __device__ __noinline__ bool all_symbols_are(uint32_t row_s, uint32_t swz, uint32_t n_my, uint32_t symbol)
{
    bool same = true;
    for (uint32_t k = 0; k < n_my; k += 4) {
        const uint32_t left = min(n_my - k, 4u);
        const uint32_t x = lds32(row_s + (((k >> 4) ^ swz) << 4) + (k & 15u)) ^ (symbol * 0x01010101u);
        same = same && (x & (0xFFFFFFFFu >> (32 - 8 * left))) == 0;
    }
    return __all_sync(0xFFFFFFFFu, same);
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
__global__ void __launch_bounds__((enc_max_workers((H0 ? 1 : 0) + (H1 ? 1 : 0)) + 1) * 32, 1)
encode_kernel(const __grid_constant__ EncParams P)
{
    constexpr int kHuff = (H0 ? 1 : 0) + (H1 ? 1 : 0);
    constexpr int kTabs = kHuff ? kHuff : 1;
    constexpr uint32_t kMaxW = enc_max_workers(kHuff);
    constexpr uint32_t kMaxTiles = SHAPE == kEncAny ? 64 : kMaxW;        // tiles of a batch
    constexpr bool kSolo = SHAPE == kEncSolo64;
    extern __shared__ __align__(16) uint8_t smem[];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint32_t n_workers = (blockDim.x >> 5) - 1;
    const uint32_t T = kSolo ? 1u : P.tiles, team = kSolo ? 1u : P.team, teams = kSolo ? n_workers : P.teams;
    const uint32_t n = SHAPE != kEncAny ? 64u : P.lane_syms;            // symbols per lane

    // shared: rings[teams] | input buffers[workers][1 or 2][64 n] | tables[kTabSlots][kTabs][256]
    const uint32_t rings_s = smem_u32(smem);
    const uint32_t bufs_s = rings_s + teams * 16 * P.ring16;
    const uint32_t buf_bytes = P.any_base ? 128 * n : 64 * n;
    const uint32_t tabs_s = bufs_s + n_workers * buf_bytes;

    __shared__ EncItem s_item[kTabSlots];
    __shared__ uint32_t s_fill[kTabSlots][2];
    __shared__ uint32_t s_slot[kEncRing], s_c0[kEncRing], s_ticket[kEncRing], s_cnt[kEncRing], s_done[kEncRing], s_tot[kEncRing];
    __shared__ uint32_t s_bits[kEncRing][kTabs][kMaxW], s_src[kEncRing][kMaxW];
    __shared__ uint32_t s_tile[2][kTabs][kMaxTiles];
    __shared__ uint32_t s_freed_seq, s_fail;
    __shared__ uint64_t mb_in[kMaxW], mb_team[kMaxW], mb_info[kEncRing];

    if (threadIdx.x < kEncRing) s_cnt[threadIdx.x] = s_done[threadIdx.x] = 0;
    if (threadIdx.x == 0) {
        s_freed_seq = s_fail = 0;
        for (uint32_t i = 0; i < kEncRing; ++i) mbar_init(&mb_info[i], 1);
        for (uint32_t i = 0; i < n_workers; ++i) { mbar_init(&mb_in[i], 1); mbar_init(&mb_team[i], team); }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncthreads();

    auto vol32 = [](const uint32_t* p) { return *reinterpret_cast<const volatile uint32_t*>(p); };
    auto counters = [&](const uint32_t index) -> TensorCounters* { return P.counters + index; };

    if (warp == n_workers) {
        // =========================== the service warp ===========================
        // It never blocks on one thing: in a loop it publishes batches, posts the sizes of packed ones, advances the
        // look-back of the oldest batch without a place by one round, and sends out the batch whose place is known.
        const EncItem* const items = P.items ? P.items : &P.one;
        if (blockIdx.x == 0)                                     // tensors without chunks are all header
            for (uint32_t t = lane; t < P.n_tensors; t += 32)
                if (items[t].n_chunks == 0) write_header(P, items[t], counters(items[t].index));

        uint32_t published = 0, posted = 0, placed = 0, freed = 0;     // batches of this block
        uint32_t ticket = 0;                                     // lane 0: ticket taken for the next batch
        bool have_ticket = false;
        uint32_t tcur = 0, next_first = 0;                       // tensor of the last ticket (tickets only grow), first batch of the next one
        uint32_t slot = 0, slot_tensor = kNoSlot;                // the newest table slot and whose it is
        uint32_t slot_last[kTabSlots] = {};                      // 1 + last batch that uses the slot
        bool ended = false, lb_on = false, lb_done = false;
        unsigned long long lb_sum = 0;
        long long lb_pos = 0;
        uint32_t idle = 0;
        // chunks this block has placed, per tensor; added to the tensor's counters when the tensor changes
        uint32_t acc_slot = kNoSlot, acc_index = 0, acc_n = 0;
        unsigned long long acc_bits[2] = {0, 0};                 // per lane: payload bits of those chunks
        auto flush_acc = [&]() {                                 // before its slot is given to another tensor
            if (acc_n == 0) return;
#pragma unroll
            for (int h = 0; h < kHuff; ++h)
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) acc_bits[h] += __shfl_xor_sync(0xFFFFFFFFu, acc_bits[h], o);
            if (lane == 0) {
                const EncItem& I = s_item[acc_slot];
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
            // ---- post the sizes of batches that have been packed ----
            while (posted < published - (ended ? 1u : 0u) && __shfl_sync(0xFFFFFFFFu, vol32(&s_cnt[posted % kEncRing]), 0) == teams) {
                __threadfence_block();
                const uint32_t r = posted % kEncRing;
                uint32_t p16 = 0;
#pragma unroll
                for (int h = 0; h < kHuff; ++h) p16 += lane < teams ? (s_bits[r][h][lane] + 127) >> 7 : 0u;
                const uint32_t total = __reduce_add_sync(0xFFFFFFFFu, p16);
                if (lane == 0) {
                    s_cnt[r] = 0;
                    s_tot[r] = total;
                    if (kHuff) st_flag(P.flags + s_ticket[r], (s_c0[r] == 0 ? kFlagPrefix : kFlagAggregate) | total);
                }
                __syncwarp();
                ++posted;
                did = true;
            }
            // ---- a new batch ----
            if (!ended && published < posted + P.ahead && published < freed + kEncRing) {
                if (!have_ticket && lane == 0) ticket = atomicAdd(&P.ctl->ticket, 1u);
                have_ticket = true;
                const uint32_t next_g = __shfl_sync(0xFFFFFFFFu, ticket, 0);
                const uint32_t r = published % kEncRing;
                bool publish = true;
                uint32_t use = kNoSlot, c0 = 0;
                if (next_g < P.total_batches) {
                    // the last tensor that starts at or before the batch (tensors without chunks share their start with the next)
                    if (P.items && next_g >= next_first) {
                        for (;;) {
                            const uint32_t cand = tcur + 1 + lane;
                            const uint32_t k = __popc(__ballot_sync(0xFFFFFFFFu, cand < P.n_tensors && P.first_batch[cand] <= next_g));
                            tcur += k;
                            if (k < 32) break;
                        }
                        next_first = tcur + 1 < P.n_tensors ? P.first_batch[tcur + 1] : 0xFFFFFFFFu;
                    }
                    if (tcur != slot_tensor) {
                        // another tensor: it takes the next slot once every batch that uses it is placed
                        const uint32_t ns = (slot + 1) % kTabSlots;
                        const uint32_t last = ns == 0 ? slot_last[0] : ns == 1 ? slot_last[1] : ns == 2 ? slot_last[2] : slot_last[3];
                        if (placed < last) {
                            publish = false;
                        } else {
                            if (acc_slot == ns) flush_acc();
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
                                for (uint32_t i = 0; i < 8; ++i) sts32(tabs_s + 1024 * (kTabs * ns + h) + 4 * (lane + 32 * i), E.enc[s][lane + 32 * i]);
                                if (lane == 0) s_fill[ns][h] = E.fill[s];
                                ++h;
                            }
                            __syncwarp();
                        }
                    }
                    if (publish) {
                        use = slot;
                        const EncItem& I = s_item[slot];
                        c0 = (next_g - I.first_batch) * teams;
                        if (c0 == 0) {
                            // the fixed parts of the tensor's container: code lengths, padding of the chunk offset table,
                            // tail padding of raw bodies
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
                    }
                } else {
                    ended = true;
                }
                if (publish) {
                    ++published;
                    have_ticket = false;
                    if (use != kNoSlot) {
#pragma unroll
                        for (uint32_t k = 0; k < kTabSlots; ++k) if (k == use) slot_last[k] = published;
                    }
                    if (lane == 0) {
                        s_slot[r] = use; s_c0[r] = c0; s_ticket[r] = next_g;
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&mb_info[r]);
                    if (P.ahead > 1 && !ended) {                 // the next one's ticket travels until it is looked at
                        if (lane == 0) ticket = atomicAdd(&P.ctl->ticket, 1u);
                        have_ticket = true;
                    }
                    did = true;
                }
            }
            // ---- placement of the oldest batch without a place ----
            if (placed < posted) {
                const uint32_t r = placed % kEncRing;
                const uint32_t use = s_slot[r], c0 = s_c0[r];
                const EncItem& I = s_item[use];
                unsigned long long* const flags = P.flags + s_ticket[r];   // the batch's own word; the look-back stays inside the tensor
                const uint32_t total = s_tot[r];
                if (!lb_on) {
                    lb_sum = 0;
                    lb_pos = 1;                                  // lane i looks lb_pos + i batches back
                    lb_done = !kHuff || c0 == 0;
                    lb_on = true;
                }
                if (!lb_done) {
                    // One round: 32 * kLookWide predecessors at a time, newest first, up to the first one that already knows
                    // its prefix.  All loads of a round are in flight together.
                    const long long b = s_ticket[r] - I.first_batch;
                    unsigned long long f[kLookWide];
#pragma unroll
                    for (int k = 0; k < kLookWide; ++k) {
                        const long long back = lb_pos + 32 * k + lane;
                        f[k] = back <= b ? ld_flag(flags - back) : kFlagPrefix;      // before batch 0: prefix 0
                    }
#pragma unroll
                    for (int k = 0; k < kLookWide; ++k) {
                        if (lb_done) continue;
                        const uint32_t ready = __ballot_sync(0xFFFFFFFFu, (f[k] >> 62) != 0);
                        const uint32_t prefix = __ballot_sync(0xFFFFFFFFu, (f[k] >> 62) == 2);
                        const uint32_t first = prefix ? (uint32_t)__ffs(prefix) - 1 : 32u;
                        const uint32_t need = first == 32 ? 0xFFFFFFFFu : (0xFFFFFFFFu >> (31 - first));
                        if ((ready & need) != need) break;       // somebody has not posted yet: again from here later
                        unsigned long long x = lane <= first ? f[k] & kFlagValue : 0;
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
                        lb_sum += x;
                        lb_done = first != 32;
                        lb_pos += 32;
                        did = true;
                    }
                    if (lb_done && lane == 0) st_flag(flags, kFlagPrefix | (lb_sum + total));
                }
                if (lb_done && __shfl_sync(0xFFFFFFFFu, vol32(&s_done[r]), 0) == n_workers) {
                    __threadfence_block();
                    const uint32_t n_mine = min(teams, I.n_chunks - c0);
                    if (use != acc_slot || I.index != acc_index) { flush_acc(); acc_slot = use; acc_index = I.index; }
                    acc_n += n_mine;
                    if (kHuff) {
                        uint32_t bits[2] = {0, 0}, p16[2] = {0, 0};
#pragma unroll
                        for (int h = 0; h < kHuff; ++h) {
                            if (lane < n_mine) bits[h] = s_bits[r][h][lane];
                            p16[h] = (bits[h] + 127) >> 7;
                            acc_bits[h] += bits[h];
                        }
                        const uint32_t mine = p16[0] + p16[1];
                        const unsigned long long off = lb_sum + warp_scan(mine, lane) - mine;
                        if (lane < n_mine) {
                            reinterpret_cast<uint32_t*>(I.out + I.lay.chunk_off_tab[H0 ? 0 : 1])[c0 + lane] = (uint32_t)off;
                            if (kHuff == 2) reinterpret_cast<uint32_t*>(I.out + I.lay.chunk_off_tab[1])[c0 + lane] = (uint32_t)off + p16[0];
                            if (mine) bulk_s2g(I.out + I.lay.payload_off + 16 * off, rings_s + 16 * (lane * P.ring16 + s_src[r][lane]), 16 * mine);
                        }
                        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
                        // the block that owns the last chunk knows the size of the whole payload area
                        if (lane == 0 && c0 + n_mine == I.n_chunks) counters(I.index)->total16 = lb_sum + total;
                    }
                    __syncwarp();
                    if (lane == 0) s_done[r] = 0;
                    ++placed;
                    lb_on = false;
                    did = true;
                }
            }
            if (ended && freed == published - 1) break;
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
            }
            if (did) { idle = 0; continue; }
            if (++idle > P.spin_limit) { s_fail = 1; break; }
            __nanosleep(100);                                    // nothing to do right now: leave the issue slots to the workers
        }
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
        __syncwarp();
        flush_acc();
    } else {
        // =========================== a worker warp ===========================
        // Bounded wait of the whole warp for a phase of an mbarrier; false on the failure flag or when the wait gives up.
        // (A try_wait sleeps in hardware until the phase completes or a time limit is reached.)
        auto wait_phase = [&](uint64_t* bar, const uint32_t parity) -> bool {
            bool ok = mbar_try_wait(bar, parity);
            for (uint32_t k = 0; !ok && k < P.spin_limit; ++k) {
                if (vol32(&s_fail)) break;
                ok = mbar_try_wait(bar, parity);
            }
            return __all_sync(0xFFFFFFFFu, ok);                  // decisions of the whole warp: no lane may leave alone
        };
        const uint32_t my_team = kSolo ? warp : warp / team, tw = kSolo ? 0u : warp - my_team * team;    // my team, my place in it
        uint32_t ph_team = 0;
        auto team_sync = [&]() -> bool {
            __syncwarp();
            if (lane == 0) mbar_arrive(&mb_team[my_team]);
            const bool ok = wait_phase(&mb_team[my_team], ph_team & 1u);
            ++ph_team;
            return ok;
        };
        const uint32_t parts = n / 16;                           // 16-byte pieces of a lane's row
        const uint32_t tile_syms = 32 * n;
        const uint32_t buf_s = bufs_s + warp * buf_bytes;
        const uint32_t ring_s = rings_s + my_team * 16 * P.ring16;
        // rows of 64 bytes: 16-byte piece p of row r sits at p ^ (r >> 1 & 3); of 32 bytes: p ^ (r >> 2 & 1); the others as they are
        const uint32_t swz_shift = n == 64 ? 1u : 2u, swz_mask = n == 64 ? 3u : n == 32 ? 1u : 0u;
        const uint32_t swz = (lane >> swz_shift) & swz_mask;
        const uint32_t row_groups = n / 8, row_magic = (0xFFFFFFFFu / row_groups) + 1;   // g / row_groups == umulhi(g, magic), g < 2^16
        auto at_of = [&](const uint32_t g) {                     // where group g's 8 symbols are staged
            const uint32_t row = __umulhi(g, row_magic), k = g - row * row_groups;
            return row * n + (((k >> 1) ^ ((row >> swz_shift) & swz_mask)) << 4) + 8 * (k & 1u);
        };
        // lanes of 64 symbols: lane l's groups l + 32 i go to row 4 i + l / 8; from one i to the next the swizzle flips bit 1
        // of the piece index
        const uint32_t at0 = (lane >> 3) * 64 + ((((lane & 7) >> 1) ^ (lane >> 4)) << 4) + 8 * (lane & 1u);

        bool loaded = false;                                     // the next tile's input has been requested
        uint32_t ph_in = 0;
        auto whole_tile = [&](const EncItem& I, const uint64_t s_lo) { return s_lo + tile_syms <= I.n_syms && 2 * (s_lo + tile_syms) <= I.input_bytes; };
        // Requests tile j of chunk c of tensor I, if it is a complete one (the buffer is free: every lane has passed a __syncwarp).
        auto request = [&](const EncItem& I, const uint32_t c, const uint32_t j) {
            const uint64_t s_lo = (uint64_t)c * P.cs + j * tile_syms;
            if (c >= I.n_chunks || !whole_tile(I, s_lo)) return;
            if (lane == 0) {
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_expect_tx(&mb_in[warp], I.base ? 128 * n : 64 * n);
                bulk_g2s_addr(buf_s, I.in + 2 * s_lo, 64 * n, &mb_in[warp]);
                if (I.base) bulk_g2s_addr(buf_s + 64 * n, I.base + 2 * s_lo, 64 * n, &mb_in[warp]);
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
            const uint32_t c = vol32(&s_c0[r]) + my_team;
            const bool active = c < I.n_chunks;
            const uint64_t c_lo = (uint64_t)c * P.cs;
            const uint32_t c_syms = active ? (uint32_t)min((uint64_t)P.cs, I.n_syms - c_lo) : 0u;
            const uint32_t tab_s = tabs_s + 1024 * kTabs * use;

            uint32_t e[kTabs][32];                               // joined codes of my symbols
            uint32_t inc[kTabs], mine[kTabs];                    // my symbols' bits, and their inclusive scan over the tile
            uint32_t tile_bits[kTabs];
            bool quads[kTabs];                                   // no four neighbouring codes of the tile are longer than 32 bits
            // Phases A and B of tile j of my chunk; `raw`: store the raw stream too; next(): requests the tile after it.
            auto do_tile = [&](const uint32_t j, const bool raw, auto next) -> bool {
                const uint32_t t_lo = j * tile_syms;
                const uint32_t t_syms = c_syms > t_lo ? min(tile_syms, c_syms - t_lo) : 0u;
                const uint64_t s_lo = c_lo + t_lo;               // first symbol of the tile in its stream
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
                auto stage = [&](const uint4 x, const uint32_t g, const uint32_t at) {
                    const uint32_t w[4] = {x.x, x.y, x.z, x.w};
                    uint32_t sy[2][2];
                    split16<FMT>(w, sy[0], sy[1]);
                    if (H0) sts64(buf_s + at, sy[0][0], sy[0][1]);
                    else if (raw) st_cs_v2(raw0 + 8 * g, make_uint2(sy[0][0], sy[0][1]));
                    if (H1) sts64(buf_s + (H0 ? tile_syms : 0u) + at, sy[1][0], sy[1][1]);
                    else if (raw) st_cs_v2(raw1 + 8 * g, make_uint2(sy[1][0], sy[1][1]));
                    if (kSpotConstant) {
                        differs[0] |= (sy[0][0] ^ fill4[0]) | (sy[0][1] ^ fill4[0]);
                        differs[1] |= (sy[1][0] ^ fill4[1]) | (sy[1][1] ^ fill4[1]);
                    }
                };
                auto x4 = [](const uint4 a, const uint4 b) { return make_uint4(a.x ^ b.x, a.y ^ b.y, a.z ^ b.z, a.w ^ b.w); };
                const bool whole = t_syms == tile_syms;
                if (whole && whole_tile(I, s_lo)) {
                    if (!loaded) request(I, c, j);
                    if (!wait_phase(&mb_in[warp], ph_in & 1u)) return false;
                    ++ph_in;
                    loaded = false;
                    uint4 x[8];
#pragma unroll
                    for (uint32_t i = 0; i < 8; ++i)
                        if (SHAPE != kEncAny || i < row_groups) x[i] = lds128(buf_s + 16 * (lane + 32 * i));
                    if (I.base) {
#pragma unroll
                        for (uint32_t i = 0; i < 8; ++i)
                            if (SHAPE != kEncAny || i < row_groups) x[i] = x4(x[i], lds128(buf_s + 64 * n + 16 * (lane + 32 * i)));
                    }
                    __syncwarp();                                // everybody has read: the buffer takes the staged symbols
#pragma unroll
                    for (uint32_t i = 0; i < 8; ++i)
                        if (SHAPE != kEncAny || i < row_groups)
                            stage(x[i], lane + 32 * i, SHAPE != kEncAny ? (at0 ^ ((i & 1u) << 5)) + 256 * i : at_of(lane + 32 * i));
                } else {
                    for (uint32_t g = lane; g < (t_syms + 7) / 8; g += 32) {
                        uint4 x = load16_guarded(I.in, 2 * (s_lo + 8ull * g), I.input_bytes);
                        if (I.base) x = x4(x, load16_guarded(I.base, 2 * (s_lo + 8ull * g), I.input_bytes));
                        stage(x, g, at_of(g));
                    }
                }
                __syncwarp();

                const uint32_t n_my = t_syms > lane * n ? min(n, t_syms - lane * n) : 0u;
#pragma unroll
                for (int h = 0; h < kHuff; ++h) {
                    const uint32_t row = buf_s + h * tile_syms + lane * n;
                    const uint32_t fill = s_fill[use][h], fill_len = fill >> 8;
                    bool constant = false;
                    if (kSpotConstant && whole && fill_len <= kLmax && __all_sync(0xFFFFFFFFu, differs[h] == 0)) {
                        // nothing but the fill symbol (which has the all-zero code)
#pragma unroll
                        for (uint32_t i = 0; i < 32; ++i) e[h][i] = 2 * fill_len;
                        mine[h] = n * fill_len;
                        constant = true;
                        quads[h] = fill_len <= 8;
                    } else {
                        bool ok = false, long_quad = true;
                        if (whole) mine[h] = lookup_quick(e[h], row, swz, parts, tab_s + 1024 * h, ok, long_quad);
                        quads[h] = __all_sync(0xFFFFFFFFu, ok && !long_quad);
                        if (!quads[h] && !__all_sync(0xFFFFFFFFu, ok)) {
                            bool no_code = false;
                            mine[h] = lookup_checked(e[h], row, swz, parts, tab_s + 1024 * h, n_my, no_code);
                            if (no_code) bad = I.index + 1;
                        }
                    }
                    inc[h] = warp_scan(mine[h], lane);
                    uint32_t bits = __shfl_sync(0xFFFFFFFFu, inc[h], 31);
                    if (!constant && t_syms && bits == t_syms * fill_len) constant = all_symbols_are(row, swz, n_my, fill & 0xFFu);
                    // tiles without symbols (behind the end of a ragged chunk) do not keep a chunk from being constant
                    if (constant || t_syms == 0) bits |= kConstTile;
                    tile_bits[h] = bits;
                }
                __syncwarp();                                    // the buffer is free
                next();
                return true;
            };
            auto next_batch = [&]() {                            // the first tile of my next chunk, if that is known already
                const uint32_t r1 = (it + 1) % kEncRing;
                if (!__all_sync(0xFFFFFFFFu, mbar_test(&mb_info[r1], ((it + 1) / kEncRing) & 1u))) return;
                const uint32_t use1 = vol32(&s_slot[r1]);
                if (use1 != kNoSlot) request(s_item[use1], vol32(&s_c0[r1]) + my_team, tw);
            };

            // per coded stream: bits of the chunk, and of the tiles of it before mine (lane = tile when a warp has several)
            uint32_t chunk_bits[kTabs] = {}, before[kTabs] = {}, before2[kTabs] = {};
            const bool several = SHAPE == kEncAny && team < T;
            if (active) {
                if (several) {
                    for (uint32_t j = tw; j < T && !failed; j += team) {
                        failed = !do_tile(j, true, [&] { if (kHuff || j + team < T) request(I, c, j + team < T ? j + team : tw); else next_batch(); });
                        if (lane == 0)
                            for (int h = 0; h < kHuff; ++h) s_tile[it & 1u][h][j] = tile_bits[h];
                    }
                } else {
                    failed = !do_tile(tw, true, next_batch);
                    if (!kSolo && lane == 0)
                        for (int h = 0; h < kHuff; ++h) s_tile[it & 1u][h][warp] = tile_bits[h];
                }
                if (failed) break;
                if (kSolo) {
#pragma unroll
                    for (int h = 0; h < kHuff; ++h) chunk_bits[h] = (tile_bits[h] & kConstTile) ? 0u : tile_bits[h];
                } else if (kHuff) {
                    // every warp of the team learns the bit counts of the chunk's tiles
                    if (!team_sync()) { failed = true; break; }
#pragma unroll
                    for (int h = 0; h < kHuff; ++h) {
                        const uint32_t* tiles = &s_tile[it & 1u][h][several ? 0u : my_team * team];
                        const uint32_t v0 = lane < T ? tiles[lane] : kConstTile, v1 = lane + 32 < T ? tiles[lane + 32] : kConstTile;
                        const uint32_t a = warp_scan(v0 & ~kConstTile, lane), a31 = __shfl_sync(0xFFFFFFFFu, a, 31);
                        uint32_t b = 0;
                        if (SHAPE == kEncAny && T > 32) b = warp_scan(v1 & ~kConstTile, lane);
                        const bool none = __all_sync(0xFFFFFFFFu, (v0 & v1 & kConstTile) != 0);
                        chunk_bits[h] = none ? 0u : a31 + __shfl_sync(0xFFFFFFFFu, b, 31);
                        before[h] = a - (v0 & ~kConstTile);
                        before2[h] = a31 + b - (v1 & ~kConstTile);
                        if (!several) before[h] = __shfl_sync(0xFFFFFFFFu, before[h], tw);
                    }
                }
            }

            // ---- the piece: its size is posted, it gets a stretch of the ring (every warp of the team follows the allocation) ----
            uint32_t p16[kTabs], total = 0;
#pragma unroll
            for (int h = 0; h < kHuff; ++h) { p16[h] = (chunk_bits[h] + 127) >> 7; total += p16[h]; }
            if (ring_pos + total > P.ring16) { virt += P.ring16 - ring_pos; ring_pos = 0; }
            const uint32_t piece_at = ring_pos;
            ring_pos += total;
            virt += total;
            if (lane == (it & 31u)) vend = virt;
            if (tw == 0 && lane == 0) {
#pragma unroll
                for (int h = 0; h < kHuff; ++h) s_bits[r][h][my_team] = chunk_bits[h];
                s_src[r][my_team] = piece_at;
                __threadfence_block();
                atomicAdd(&s_cnt[r], 1u);
            }
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
                    // my share of the piece starts from zero
                    for (uint32_t u = tw * 32 + lane; u < total; u += 32 * team) sts128_zero(ring_s + 16 * (piece_at + u));
                    if (kSolo) __syncwarp();
                    else if (!team_sync()) { failed = true; break; }
                }
                auto finish_tile = [&](const uint32_t j, const uint32_t (&pre)[kTabs]) {
                    // subchunk ends: lane g of the chunk (counting through its tiles) ends subchunk (g + 1) / T - 1 if T divides g + 1
                    const uint32_t gl = j * 32 + lane + 1, sub_i = kSolo ? gl : gl / T;
#pragma unroll
                    for (int h = 0; h < kHuff; ++h) {
                        const int s = H0 ? h : 1;
                        const uint32_t end = chunk_bits[h] ? pre[h] + inc[h] : 0u;
                        if (sub_i * T == gl) {
                            if (SHAPE == kEncSolo64 || P.sub_width == 2) reinterpret_cast<uint16_t*>(I.out + I.lay.sub_end_tab[s] + 64ull * c)[sub_i - 1] = (uint16_t)end;
                            else reinterpret_cast<uint32_t*>(I.out + I.lay.sub_end_tab[s] + 128ull * c)[sub_i - 1] = end;
                        }
                        if (chunk_bits[h]) {
                            const uint32_t piece_s = ring_s + 16 * (piece_at + (h ? p16[0] : 0u));
                            if (quads[h]) emit_codes<true>(e[h], parts, piece_s, end - mine[h]);
                            else emit_codes<false>(e[h], parts, piece_s, end - mine[h]);
                        }
                    }
                };
                if (several) {
                    for (uint32_t j = tw; j < T && !failed; j += team) {
                        uint32_t pre[kTabs];
#pragma unroll
                        for (int h = 0; h < kHuff; ++h) pre[h] = __shfl_sync(0xFFFFFFFFu, j < 32 ? before[h] : before2[h], j & 31u);
                        // looked up again: the codes of one tile at a time are kept
                        failed = !do_tile(j, false, [&] { if (j + team < T) request(I, c, j + team); else next_batch(); });
                        if (!failed) finish_tile(j, pre);
                    }
                    if (failed) break;
                } else {
                    finish_tile(tw, before);
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            }
            __syncwarp();
            if (lane == 0) {
                __threadfence_block();
                atomicAdd(&s_done[r], 1u);
            }
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
