// Host side of the encoder: launch shapes and zc_compress, zc_compress_batch, zc_compress_noalloc, zc_device_status.
#include "zc_encode.cuh"

#include <atomic>
#include <cstdlib>
#include <cstring>
#include <unordered_map>
#include <vector>

using namespace zc;

namespace {

// Launch shape of the tensors of one launch (same format, chunk size and stream modes).
struct EncShape { int kind; uint32_t unit_chunks, tiles, teams, ring16, buf_bytes; bool base_buf; size_t smem; };

constexpr uint32_t kEncSmem = 216 * 1024;        // dynamic shared memory of a block; the rest is static

EncShape enc_shape(const zc_plan_t* p, uint32_t n_huff, bool any_base, uint64_t total_chunks)
{
    EncShape s{};
    const uint32_t cs = p->syms_per_chunk, full = 32 * enc_lane_syms(kEncAny), small = 32 * enc_lane_syms(kEncAny48);
    auto tiles = [&](uint32_t tile_syms) { return (cs + tile_syms - 1) / tile_syms; };
    // a unit is as many whole chunks as fit a tile (1 and 2 KiB), or one chunk of one tile or several
    s.unit_chunks = 2 * cs <= full && full % cs == 0 ? std::min(kMaxUnitChunks, full / cs) : 1;
    const int solo = (int)(cs / 512);                            // the shapes of long lanes are numbered by the chunk's KiB
    if (cs == full) s.kind = kEncSolo;
    else if (s.unit_chunks > 1) s.kind = kEncUnit;
    // (a launch of few chunks takes a warp's way through one, which is shorter in two tiles: 205 chunks of 5 KiB 16.2 against
    // 16.8 us; from about two chunks per SM on one tile is faster: 1184 chunks of 7 KiB 20.7 against 19.0 us)
    else if (n_huff == 1 && solo >= kEncSolo80 && solo <= kEncSolo112 && total_chunks > 2ull * sm_count()) s.kind = solo;
    else if (cs % full == 0) s.kind = kEncTeam;
    else if (tiles(small) * small < tiles(full) * full && tiles(small) <= enc_max_workers(kEncAny48, (int)n_huff)) s.kind = kEncAny48;
    else s.kind = kEncAny;
    s.tiles = tiles(32 * enc_lane_syms(s.kind));
    // kEncBig has the workers for 16 tiles, or with one coded stream for half as many teams again (29 to 31 KiB: two teams
    // instead of one, 128 MB of BF16 weights 124 -> 102 us; 19 KiB: three instead of two, 111 -> 102 us; not 13 and 14 KiB,
    // four instead of three: +2 %)
    const uint32_t workers = enc_max_workers(s.kind, (int)n_huff), big_teams = enc_max_workers(kEncBig, (int)n_huff) / tiles(full);
    if (s.tiles > workers || (n_huff == 1 && (s.kind == kEncAny || s.kind == kEncAny48) && 2 * big_teams >= 3 * (workers / s.tiles))) {
        s.kind = kEncBig;
        s.tiles = tiles(full);
    }
    const uint32_t tile_bytes = 64 * enc_lane_syms(s.kind);
    const uint32_t tables = 1024 * kTabSlots * std::max<uint32_t>(n_huff, 1);
    // a ring holds at least one unit of 12-bit codes; typical ones are a quarter to a half of that
    const uint32_t min_ring = n_huff * s.unit_chunks * (uint32_t)round_up((uint64_t)cs * kLmax / 8, 16);
    // The base tensor has an input buffer of its own, except for the largest chunks with both streams coded.  (The staged
    // symbols take the input's place: a buffer of their own would let the next tile be requested earlier, but what it takes
    // from the rings costs more: BF16 736 against 742 us, FP8 499 against 526 us.)
    const uint32_t max_teams = enc_max_workers(s.kind, (int)n_huff) / s.tiles;
    auto teams_with = [&](uint32_t worker_bytes) { return std::min<uint32_t>(max_teams, (kEncSmem - tables) / (s.tiles * worker_bytes + min_ring)); };
    s.base_buf = any_base && teams_with(2 * tile_bytes) > 0;
    s.buf_bytes = s.base_buf ? 2 * tile_bytes : tile_bytes;
    s.teams = teams_with(s.buf_bytes);
    const uint32_t buf = s.tiles * s.buf_bytes;
    // few chunks: rather more blocks than more teams in a block
    const uint64_t units = (total_chunks + s.unit_chunks - 1) / s.unit_chunks;
    s.teams = (uint32_t)std::max<uint64_t>(1, std::min<uint64_t>(s.teams, (units + sm_count() - 1) / sm_count()));
    s.ring16 = n_huff ? std::min<uint32_t>(((kEncSmem - tables) / s.teams - buf) / 16, std::max<uint32_t>(min_ring / 4, 1024)) : 0;
    s.smem = tables + (size_t)s.teams * (buf + 16 * s.ring16);
    return s;
}

void fill_common(EncParams& P, const zc_plan_t* p, const uint32_t mode[2], const EncShape& sh)
{
    P.cs = p->syms_per_chunk; P.sub = p->syms_per_sub; P.chunk_bytes = p->chunk_bytes;
    P.format = p->format; P.group = p->group;
    P.sub_width = sub_end_width(p->chunk_bytes);
    P.sub_magic = (uint32_t)(((1ull << 32) + p->syms_per_sub - 1) / p->syms_per_sub);
    P.mode[0] = mode[0]; P.mode[1] = mode[1];
    P.unit_syms = sh.unit_chunks * p->syms_per_chunk; P.unit_chunks = sh.unit_chunks;
    P.tiles = sh.tiles; P.teams = sh.teams; P.ring16 = sh.ring16;
    P.spin_limit = test_knobs().spin_limit;
    P.base_buf = sh.base_buf ? 1u : 0u;
    P.buf_bytes = sh.buf_bytes;
}

uint32_t units_of(const zc_plan_t* p, const EncShape& sh) { return (p->n_chunks + sh.unit_chunks - 1) / sh.unit_chunks; }
uint32_t batches_of(const zc_plan_t* p, const EncShape& sh) { return (uint32_t)((units_of(p, sh) + (uint64_t)sh.teams - 1) / sh.teams); }

void fill_item(EncItem& it, const zc_plan_t* p, const EncShape& sh, const uint32_t mode[2], const void* d_in, const void* d_base, void* d_out,
               uint32_t first_batch, uint32_t index, uint32_t table)
{
    it.in = (const uint8_t*)d_in;
    it.base = (const uint8_t*)d_base;
    it.out = (uint8_t*)d_out;
    it.input_bytes = p->input_bytes; it.n_syms = p->n_syms; it.n_elems = p->n_elems;
    it.n_chunks = p->n_chunks;
    it.n_units = units_of(p, sh);
    it.pad = 0;
    it.first_batch = first_batch;
    it.index = index;
    it.table = table;
    it.lay = make_layout(*p, mode);
}

void fill_tables(EncTables& T, const zc_codebook_t* cb)
{
    static_assert(sizeof(T.enc) == sizeof(cb->enc), "table layout");
    std::memcpy(T.enc, cb->enc, sizeof(T.enc));
    T.fill[0] = cb->fill[0]; T.fill[1] = cb->fill[1];
    T.pad[0] = T.pad[1] = 0;
}

cudaError_t launch_encode(EncParams& P, const EncShape& sh, const EncRanges& R, cudaStream_t st)
{
    const uint32_t grid = std::min<uint32_t>(std::max<uint32_t>(P.total_batches, 1), (uint32_t)sm_count());
    // Holding a second batch (and the ticket of a third) hides the way from a ticket to a batch and lets the workers request
    // its input while they code the first; with few batches per block it would only keep them from idle blocks.  (64 pages of
    // 527 KB, 3.5 batches per block: 70 us with one batch at a time, 54 us with two.)
    P.ahead = P.total_batches >= 4 * grid ? 3 : P.total_batches >= 2 * grid ? 2 : 1;
    const uint32_t threads = (sh.tiles * sh.teams + kServiceWarps) * 32;
    switch (P.format) {
    case ZC_FMT_BF16: return enc_launch_bf16(sh.kind, grid, threads, sh.smem, st, P, R);
    case ZC_FMT_FP8_E4M3: case ZC_FMT_FP8_E5M2: return enc_launch_fp8(sh.kind, grid, threads, sh.smem, st, P, R);
    case ZC_FMT_SCALE_U8: return enc_launch_scale(sh.kind, grid, threads, sh.smem, st, P, R);
    default: return enc_launch_fp4(sh.kind, grid, threads, sh.smem, st, P, R);
    }
}

#if ZC_DEBUG_CHECKS
// no container is larger than its tables plus 12 bits per symbol of either stream, padding and guard
size_t out_bound(const EncItem& it) { return it.lay.payload_off + 3 * it.n_syms + 32ull * it.n_chunks + 64; }
#endif

// Workspace of a batched call: control block | counters[n] | look-back words[batches] | items[n] | first batches[n] |
// tables[n].  Everything before the items starts from zero (one clear), the rest is uploaded in one copy.  A batch is
// one chunk or more, so the number of chunks bounds the number of batches.
struct BatchLayout { size_t counters, flags, items, first, tables, total; };

BatchLayout batch_layout(uint32_t n_tensors, uint64_t total_batches)
{
    BatchLayout L{};
    L.counters = kControlBytes;
    L.flags = (size_t)round_up(L.counters + sizeof(TensorCounters) * (uint64_t)n_tensors, 256);
    L.items = (size_t)round_up(L.flags + 8ull * total_batches, 256);
    L.first = L.items + sizeof(EncItem) * (size_t)n_tensors;
    L.tables = (size_t)round_up(L.first + 4ull * n_tensors, 16);
    L.total = (size_t)round_up(L.tables + sizeof(EncTables) * (uint64_t)n_tensors, 256);
    return L;
}

// Host-to-device copy of what a batched call needs on the device (tensor list, code tables).  A large copy from pageable memory holds the host
// until the stream has drained, which would make an asynchronous call wait for the previous call's kernel; so
// it goes through a pinned staging buffer, one per calling thread, that is reused once the previous copy
// out of it has been done (an event says so).  The buffer is never freed (a thread's last CUDA calls may come
// after the runtime has shut down).  Without pinned memory the copy falls back to the pageable one.
// A copy that is being captured into a graph is made anew by every replay, long after this call has returned and the
// buffers here hold another call's lists: its source is a block of its own that the graph, and what is instantiated from it,
// keeps.
struct TableStage { void* ptr = nullptr; size_t cap = 0; cudaEvent_t done = nullptr; int device = -1; };

cudaError_t upload_host(void* d_dst, const void* h_src, size_t bytes, cudaStream_t st)
{
    static thread_local TableStage stage;
    cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
    cudaGraph_t graph = nullptr;
    cudaError_t ec = cudaStreamGetCaptureInfo_v2(st, &capture, nullptr, &graph);
    if (ec != cudaSuccess) return ec;
    if (capture != cudaStreamCaptureStatusNone) {
        if (capture != cudaStreamCaptureStatusActive) return cudaErrorStreamCaptureInvalidated;
        void* const kept = std::malloc(bytes);
        if (!kept) return cudaErrorMemoryAllocation;
        std::memcpy(kept, h_src, bytes);
        cudaUserObject_t owner;
        ec = cudaUserObjectCreate(&owner, kept, std::free, 1, cudaUserObjectNoDestructorSync);
        if (ec != cudaSuccess) { std::free(kept); return ec; }
        ec = cudaGraphRetainUserObject(graph, owner, 1, cudaGraphUserObjectMove);
        if (ec != cudaSuccess) { cudaUserObjectRelease(owner, 1); return ec; }
        return cudaMemcpyAsync(d_dst, kept, bytes, cudaMemcpyHostToDevice, st);
    }
    if (bytes <= 48 * 1024)                      // small copies leave the caller's memory at once anyway
        return cudaMemcpyAsync(d_dst, h_src, bytes, cudaMemcpyHostToDevice, st);
    int device = -1;
    if (cudaGetDevice(&device) != cudaSuccess) return cudaErrorUnknown;
    if (stage.done) {
        if (cudaEventSynchronize(stage.done) != cudaSuccess) return cudaErrorUnknown;
        if (stage.device != device) { cudaEventDestroy(stage.done); stage.done = nullptr; }
    }
    if (stage.cap < bytes) {
        if (stage.ptr) cudaFreeHost(stage.ptr);
        stage.ptr = nullptr;
        stage.cap = 0;
        const size_t want = (size_t)round_up(bytes, 1u << 18);
        if (cudaHostAlloc(&stage.ptr, want, cudaHostAllocPortable) == cudaSuccess) stage.cap = want;
        else { stage.ptr = nullptr; (void)cudaGetLastError(); }
    }
    if (!stage.ptr) return cudaMemcpyAsync(d_dst, h_src, bytes, cudaMemcpyHostToDevice, st);
    if (!stage.done) {
        if (cudaEventCreateWithFlags(&stage.done, cudaEventDisableTiming) != cudaSuccess) {
            stage.done = nullptr;
            (void)cudaGetLastError();
            return cudaMemcpyAsync(d_dst, h_src, bytes, cudaMemcpyHostToDevice, st);
        }
        stage.device = device;
    }
    std::memcpy(stage.ptr, h_src, bytes);
    const cudaError_t e = cudaMemcpyAsync(d_dst, stage.ptr, bytes, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return e;
    return cudaEventRecord(stage.done, st);
}

}  // namespace

namespace zc {
void debug_counts_encode(uint32_t out[2])
{
    enc_debug_counts_bf16(out);
    enc_debug_counts_fp8(out);
    enc_debug_counts_scale(out);
    enc_debug_counts_fp4(out);
}
}  // namespace zc

extern "C" {

uint32_t zc_test_encoder_workers(const zc_plan_t* p, uint32_t n_coded, uint32_t any_base, uint64_t total_chunks)
{
    if (!p || n_coded > 2 || any_base > 1) return 0;
    const EncShape sh = enc_shape(p, n_coded, any_base != 0, total_chunks);
    const uint32_t workers = sh.tiles * sh.teams, unit = n_coded * sh.unit_chunks * (uint32_t)round_up((uint64_t)p->syms_per_chunk * kLmax / 8, 16);
    if (workers > enc_max_workers(sh.kind, (int)n_coded) || sh.smem > kEncSmem || 16 * sh.ring16 < unit) return 0;
    return sh.tiles * 32 * enc_lane_syms(sh.kind) >= sh.unit_chunks * p->syms_per_chunk ? workers : 0;
}

zc_status zc_compress(const zc_plan_t* p, const zc_codebook_t* cb, const void* d_in, void* d_out, size_t out_capacity,
                      void* d_workspace, uint64_t* h_out_bytes, void* cuda_stream)
{
    return zc_compress_xor(p, cb, d_in, nullptr, d_out, out_capacity, d_workspace, h_out_bytes, cuda_stream);
}

zc_status zc_compress_xor(const zc_plan_t* p, const zc_codebook_t* cb, const void* d_in, const void* d_base, void* d_out,
                          size_t out_capacity, void* d_workspace, uint64_t* h_out_bytes, void* cuda_stream)
{
    if (!p || !cb || !d_out || !d_workspace || (!d_in && p->n_elems)) return ZC_E_INVALID_ARG;
    if (!aligned16(d_in) || !aligned16(d_base) || !aligned16(d_out) || !aligned16(d_workspace)) return ZC_E_INVALID_ARG;
    if (out_capacity < zc_max_compressed_bytes(p)) return ZC_E_BUFFER_TOO_SMALL;
    cudaStream_t st = (cudaStream_t)cuda_stream;

    uint32_t mode[2], n_huff = 0;
    for (int s = 0; s < 2; ++s) {
        // an empty tensor has no symbols to code: both streams are stored raw
        mode[s] = p->n_syms ? cb->mode[s] : (uint32_t)ZC_MODE_RAW;
        n_huff += mode[s] == ZC_MODE_HUFF;
    }
    const EncShape sh = enc_shape(p, n_huff, d_base != nullptr, p->n_chunks);

    EncParams P{};
    fill_common(P, p, mode, sh);
    P.ctl = (Control*)d_workspace;
    P.counters = &P.ctl->tc;
    P.flags = (unsigned long long*)((uint8_t*)d_workspace + kControlBytes);
    P.n_tensors = 1;
    P.total_batches = batches_of(p, sh);
    fill_item(P.one, p, sh, mode, d_in, d_base, d_out, 0, 0, 0);
    fill_tables(P.table, cb);

    if (cudaMemsetAsync(d_workspace, 0, kControlBytes + 8ull * P.total_batches, st) != cudaSuccess) return ZC_E_CUDA;
    if (test_knobs().first_ticket) {             // test hook: the tickets start late, batch 0 is never packed
        static uint32_t first;
        first = test_knobs().first_ticket;
        if (cudaMemcpyAsync(&((Control*)d_workspace)->ticket, &first, sizeof(first), cudaMemcpyHostToDevice, st) != cudaSuccess) return ZC_E_CUDA;
    }
    EncRanges R{};
#if ZC_DEBUG_CHECKS
    DbgHull rd;
    rd.add(d_in, p->input_bytes);
    rd.add(d_base, p->input_bytes);
    R = EncRanges{rd.ptr(), rd.bytes(), d_out, out_bound(P.one), d_workspace, kControlBytes + 8ull * std::max<uint32_t>(P.total_batches, 1)};
#endif
    if (launch_encode(P, sh, R, st) != cudaSuccess) return ZC_E_CUDA;

    if (h_out_bytes) {
        Control h;
        if (cudaMemcpyAsync(&h, d_workspace, sizeof(Control), cudaMemcpyDeviceToHost, st) != cudaSuccess) return ZC_E_CUDA;
        if (cudaStreamSynchronize(st) != cudaSuccess) return ZC_E_CUDA;
        if (h.status & 0xFF) return (zc_status)(h.status & 0xFF);
        *h_out_bytes = h.tc.total16;
    }
    return ZC_OK;
}

size_t zc_compress_batch_workspace_bytes(uint32_t n_tensors, const zc_plan_t* const* plans)
{
    if (!plans) return 0;
    uint64_t chunks = 0;
    for (uint32_t t = 0; t < n_tensors; ++t) {
        if (!plans[t]) return 0;
        chunks += plans[t]->n_chunks;
    }
    return batch_layout(n_tensors, chunks).total;
}

zc_status zc_compress_batch(uint32_t n_tensors, const zc_plan_t* const* plans, const zc_codebook_t* const* codebooks,
                            const void* const* d_in, void* const* d_out, const size_t* out_capacity,
                            void* d_workspace, size_t workspace_bytes, uint64_t* h_out_bytes, void* cuda_stream)
{
    return zc_compress_batch_xor(n_tensors, plans, codebooks, d_in, nullptr, d_out, out_capacity, d_workspace, workspace_bytes,
                                 h_out_bytes, cuda_stream);
}

zc_status zc_compress_batch_xor(uint32_t n_tensors, const zc_plan_t* const* plans, const zc_codebook_t* const* codebooks,
                                const void* const* d_in, const void* const* d_base, void* const* d_out,
                                const size_t* out_capacity, void* d_workspace, size_t workspace_bytes,
                                uint64_t* h_out_bytes, void* cuda_stream)
{
    if (!d_workspace || !aligned16(d_workspace)) return ZC_E_INVALID_ARG;
    if (n_tensors == 0) return ZC_OK;
    if (!plans || !codebooks || !d_in || !d_out || !out_capacity) return ZC_E_INVALID_ARG;
    const zc_plan_t* p0 = plans[0];
    uint64_t all_chunks = 0;
    for (uint32_t t = 0; t < n_tensors; ++t) {
        const zc_plan_t* p = plans[t];
        if (!p || !codebooks[t] || !d_out[t] || (!d_in[t] && p->n_elems)) return ZC_E_INVALID_ARG;
        if (!aligned16(d_in[t]) || !aligned16(d_out[t]) || (d_base && !aligned16(d_base[t]))) return ZC_E_INVALID_ARG;
        if (p->format != p0->format || p->chunk_bytes != p0->chunk_bytes) return ZC_E_INVALID_ARG;
        if (out_capacity[t] < zc_max_compressed_bytes(p)) return ZC_E_BUFFER_TOO_SMALL;
        all_chunks += p->n_chunks;
    }
    if (workspace_bytes < batch_layout(n_tensors, all_chunks).total) return ZC_E_BUFFER_TOO_SMALL;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    uint8_t* ws = (uint8_t*)d_workspace;

    // One launch per combination of stream modes that occurs; the tensors of a combination lie next to each other in the
    // uploaded list.  Codebooks that several tensors share (the K/V pages of a step) are uploaded once.
    static thread_local std::vector<uint8_t> upload;
    static thread_local std::vector<uint8_t> combo_of;           // per tensor: mode0 | mode1 << 1
    static thread_local std::vector<const zc_codebook_t*> books; // the distinct codebooks
    static thread_local std::vector<uint32_t> table_of;          // per tensor: its tables among the uploaded ones
    static thread_local std::unordered_map<const zc_codebook_t*, uint32_t> seen;
    combo_of.resize(n_tensors); table_of.resize(n_tensors);
    books.clear(); seen.clear();
    uint32_t per_combo[4] = {};
    uint64_t chunks[4] = {};
    bool base[4] = {};
    for (uint32_t t = 0; t < n_tensors; ++t) {
        const auto found = seen.emplace(codebooks[t], (uint32_t)books.size());
        if (found.second) books.push_back(codebooks[t]);
        table_of[t] = found.first->second;
        // an empty tensor has no symbols to code: both streams are stored raw
        const uint32_t combo = plans[t]->n_syms ? codebooks[t]->mode[0] | (codebooks[t]->mode[1] << 1) : 0;
        combo_of[t] = (uint8_t)combo;
        ++per_combo[combo];
        chunks[combo] += plans[t]->n_chunks;
        base[combo] = base[combo] || (d_base && d_base[t]);
    }
    EncShape shapes[4];
    for (uint32_t combo = 0; combo < 4; ++combo) shapes[combo] = enc_shape(p0, (combo & 1u) + (combo >> 1), base[combo], chunks[combo]);
    uint32_t begin[5] = {};
    uint64_t batches[4] = {}, all_batches = 0;
    for (uint32_t t = 0; t < n_tensors; ++t) batches[combo_of[t]] += batches_of(plans[t], shapes[combo_of[t]]);
    for (uint32_t combo = 0; combo < 4; ++combo) {
        begin[combo + 1] = begin[combo] + per_combo[combo];
        all_batches += batches[combo];
        if (batches[combo] >= (1ull << 32)) return ZC_E_UNSUPPORTED;
    }
    const BatchLayout L = batch_layout(n_tensors, all_batches);
    const size_t upload_bytes = L.tables - L.items + sizeof(EncTables) * books.size();
    upload.resize(upload_bytes);
    EncItem* items = reinterpret_cast<EncItem*>(upload.data());
    uint32_t* first = reinterpret_cast<uint32_t*>(upload.data() + (L.first - L.items));
    EncTables* tables = reinterpret_cast<EncTables*>(upload.data() + (L.tables - L.items));
    for (size_t k = 0; k < books.size(); ++k) fill_tables(tables[k], books[k]);
    uint32_t at[4] = {begin[0], begin[1], begin[2], begin[3]}, next[4] = {};
    for (uint32_t t = 0; t < n_tensors; ++t) {
        const uint32_t combo = combo_of[t], i = at[combo]++;
        const uint32_t mode[2] = {combo & 1u, combo >> 1};
        fill_item(items[i], plans[t], shapes[combo], mode, d_in[t], d_base ? d_base[t] : nullptr, d_out[t], next[combo], t, table_of[t]);
        first[i] = next[combo];
        next[combo] += batches_of(plans[t], shapes[combo]);
    }
    // control block, counters and look-back words start from zero
    if (cudaMemsetAsync(ws, 0, L.items, st) != cudaSuccess) return ZC_E_CUDA;
    if (upload_host(ws + L.items, upload.data(), upload_bytes, st) != cudaSuccess) return ZC_E_CUDA;

    uint64_t flag_base = 0;
    bool first_launch = true;
    for (uint32_t combo = 0; combo < 4; ++combo) {
        if (!per_combo[combo]) continue;
        const uint32_t mode[2] = {combo & 1u, combo >> 1};
        EncParams P{};
        fill_common(P, p0, mode, shapes[combo]);
        P.ctl = (Control*)ws;
        P.counters = (TensorCounters*)(ws + L.counters);
        P.flags = (unsigned long long*)(ws + L.flags) + flag_base;
        P.items = (const EncItem*)(ws + L.items) + begin[combo];
        P.first_batch = (const uint32_t*)(ws + L.first) + begin[combo];
        P.tables = (const EncTables*)(ws + L.tables);
        P.n_tensors = per_combo[combo];
        P.total_batches = (uint32_t)batches[combo];
        flag_base += batches[combo];
        // the ticket counter restarts for every launch (the first one finds it cleared)
        if (!first_launch && cudaMemsetAsync(&((Control*)ws)->ticket, 0, sizeof(uint32_t), st) != cudaSuccess) return ZC_E_CUDA;
        first_launch = false;
        EncRanges R{};
#if ZC_DEBUG_CHECKS
        DbgHull rd, wr;
        for (uint32_t i = begin[combo]; i < begin[combo + 1]; ++i) {
            rd.add(items[i].in, items[i].input_bytes);
            rd.add(items[i].base, items[i].input_bytes);
            wr.add(items[i].out, out_bound(items[i]));
        }
        R = EncRanges{rd.ptr(), rd.bytes(), wr.ptr(), wr.bytes(), ws, L.total};
#endif
        if (launch_encode(P, shapes[combo], R, st) != cudaSuccess) return ZC_E_CUDA;
    }

    if (h_out_bytes) {
        // control block and counters lie next to each other: one copy
        static thread_local std::vector<uint8_t> h_state;
        const size_t bytes = L.counters + sizeof(TensorCounters) * (size_t)n_tensors;
        h_state.resize(bytes);
        if (cudaMemcpyAsync(h_state.data(), ws, bytes, cudaMemcpyDeviceToHost, st) != cudaSuccess) return ZC_E_CUDA;
        if (cudaStreamSynchronize(st) != cudaSuccess) return ZC_E_CUDA;
        Control h;
        std::memcpy(&h, h_state.data(), sizeof(Control));
        if (h.status & 0xFF) return (zc_status)(h.status & 0xFF);
        for (uint32_t t = 0; t < n_tensors; ++t) {
            TensorCounters tc;
            std::memcpy(&tc, h_state.data() + L.counters + sizeof(TensorCounters) * (size_t)t, sizeof(tc));
            h_out_bytes[t] = tc.total16;
        }
    }
    return ZC_OK;
}

// ---- compression without a caller-supplied workspace ---------------------------------------------
// The scratch zc_compress needs (control block + one look-back word per chunk) for up to
// ZC_NOALLOC_MAX_CHUNKS chunks, resident in every GPU that loads the library.  Host code must not pass
// this symbol to a kernel: on the host its name is only a stand-in, the device address comes from
// cudaGetSymbolAddress and differs per device.
static __device__ __align__(256) unsigned char g_noalloc_scratch[ZC_NOALLOC_SCRATCH_BYTES];

namespace {
constexpr int kMaxDevices = 64;
std::atomic<void*> g_noalloc_ptr[kMaxDevices];

// Device address of the scratch array on the current device; looked up once per device (two host threads that
// make the first call together both look it up and store the same address).
zc_status noalloc_scratch(void** out)
{
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return ZC_E_CUDA;
    void* ptr = g_noalloc_ptr[dev].load(std::memory_order_acquire);
    if (!ptr) {
        if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) return ZC_E_CUDA;
        g_noalloc_ptr[dev].store(ptr, std::memory_order_release);
    }
    *out = ptr;
    return ZC_OK;
}
}  // namespace

zc_status zc_compress_noalloc(const zc_plan_t* p, const zc_codebook_t* cb, const void* d_in, void* d_out,
                              size_t out_capacity, uint64_t* h_out_bytes, void* cuda_stream)
{
    if (!p) return ZC_E_INVALID_ARG;
    if (p->n_chunks > ZC_NOALLOC_MAX_CHUNKS || zc_workspace_bytes(p) > ZC_NOALLOC_SCRATCH_BYTES) return ZC_E_TOO_LARGE;
    void* scratch = nullptr;
    const zc_status st = noalloc_scratch(&scratch);
    if (st != ZC_OK) return st;
    // zc_compress clears the control block and the look-back words it uses before launching
    return zc_compress(p, cb, d_in, d_out, out_capacity, scratch, h_out_bytes, cuda_stream);
}

zc_status zc_noalloc_status(void* cuda_stream)
{
    void* scratch = nullptr;
    const zc_status st = noalloc_scratch(&scratch);
    if (st != ZC_OK) return st;
    cudaStream_t stream = (cudaStream_t)cuda_stream;
    unsigned long long word[2] = {0, 0};            // status, call id
    if (cudaMemcpyAsync(word, scratch, sizeof(word), cudaMemcpyDeviceToHost, stream) != cudaSuccess) return ZC_E_CUDA;
    if (cudaStreamSynchronize(stream) != cudaSuccess) return ZC_E_CUDA;
    return (word[0] >> 8) == word[1] ? (zc_status)(word[0] & 0xFF) : ZC_OK;
}

zc_status zc_device_status(const zc_plan_t* p, const void* d_workspace, void* cuda_stream)
{
    if (!p || !d_workspace) return ZC_E_INVALID_ARG;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    unsigned long long word[2] = {0, 0};            // status, call id
    if (cudaMemcpyAsync(word, d_workspace, sizeof(word), cudaMemcpyDeviceToHost, st) != cudaSuccess) return ZC_E_CUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return ZC_E_CUDA;
    // an error word left by an earlier call carries that call's id and does not count
    return (word[0] >> 8) == word[1] ? (zc_status)(word[0] & 0xFF) : ZC_OK;
}

}  // extern "C"
