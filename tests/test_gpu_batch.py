"""The batched entry points against the CPU oracle: many tensors per call, bit-exact.

Containers given to the batched decoder are made by the oracle; containers made by the batched encoder are
compared with the oracle's byte for byte.  Everything goes through the C ABI (via the ctypes binding).
"""
import numpy as np
import pytest
import torch

import oracle as zo
from paper_2508_19263_b200 import binding as zc
from test_gpu_parity import _weights

pytestmark = pytest.mark.gpu
FORMATS = [zc.FMT_BF16, zc.FMT_FP8_E4M3, zc.FMT_FP4_E2M1, zc.FMT_SCALE_U8, zc.FMT_FP8_E5M2]
DEV = "cuda"


def _sizes(fmt, chunk_bytes):
    """Element counts from nothing to dozens of chunks, ragged ends included."""
    G = zo.group(fmt)
    cs = chunk_bytes // 2
    sizes = [0, 2 * G, cs * G, cs * G + 2 * G, 3 * cs * G - 2 * G, 40 * cs * G + 6 * G, 0, 7 * cs * G, 29 * cs * G + cs * G // 2,
             64 * cs * G, 2 * G, 11 * cs * G + 10 * G]
    return [n - (n % 2) if fmt == zc.FMT_FP4_E2M1 else n for n in sizes]


def _oracle_containers(fmt, sizes, chunk_bytes, seed):
    policies = [zc.POLICY_AUTO, zc.POLICY_HUFF_ALL, zc.POLICY_RAW_ALL]
    datas, conts = [], []
    for i, n in enumerate(sizes):
        data = _weights(fmt, n, seed + i)
        cb = zo.build_codebook(zo.histogram(fmt, data, n), policies[i % 3])
        datas.append(data)
        conts.append(zo.compress(fmt, data, n, chunk_bytes, cb))
    return datas, conts


def _to_dev(a, pad=0):
    t = torch.full((max(a.size, 16) + pad,), 0xEE, dtype=torch.uint8, device=DEV)
    t[: a.size] = torch.from_numpy(a.copy()).to(DEV)
    return t


@pytest.mark.parametrize("fmt", FORMATS)
@pytest.mark.parametrize("chunk_bytes", [1024, 4096, 16384])
def test_batched_decoder_restores_every_tensor(fmt, chunk_bytes):
    sizes = _sizes(fmt, chunk_bytes)
    datas, conts = _oracle_containers(fmt, sizes, chunk_bytes, 1000 * fmt + chunk_bytes)
    plans = [zc.plan(fmt, n, chunk_bytes) for n in sizes]
    d_comps = [_to_dev(c) for c in conts]
    d_outs = [torch.full((p.input_bytes + 64,), 0xEE, dtype=torch.uint8, device=DEV) for p in plans]
    ws = torch.full((256,), 0x5A, dtype=torch.uint8, device=DEV)
    batch = zc.DecompressBatch(plans, d_comps, [c.size for c in conts], d_outs)
    for _ in range(2):                                               # the second call reuses the workspace as it is
        zc.decompress_batch(batch, ws)
        assert zc.batch_status(ws) == (zc.OK, None)
        for p, data, out in zip(plans, datas, d_outs):
            back = out.cpu().numpy()
            assert np.array_equal(back[: p.input_bytes], data[: p.input_bytes])
            assert (back[p.input_bytes:] == 0xEE).all()


def test_batched_decoder_many_small_tensors_span_several_launches():
    fmt, chunk_bytes = zc.FMT_BF16, 1024
    rng = np.random.default_rng(7)
    sizes = [int(v) for v in rng.integers(0, 3000, 1100)]
    datas, conts = _oracle_containers(fmt, sizes, chunk_bytes, 5)
    plans = [zc.plan(fmt, n, chunk_bytes) for n in sizes]
    d_comps = [_to_dev(c) for c in conts]
    d_outs = [torch.full((p.input_bytes + 16,), 0xEE, dtype=torch.uint8, device=DEV) for p in plans]
    ws = torch.zeros(256, dtype=torch.uint8, device=DEV)
    zc.decompress_batch(zc.DecompressBatch(plans, d_comps, [c.size for c in conts], d_outs), ws)
    assert zc.batch_status(ws) == (zc.OK, None)
    for p, data, out in zip(plans, datas, d_outs):
        back = out.cpu().numpy()
        assert np.array_equal(back[: p.input_bytes], data[: p.input_bytes])
        assert (back[p.input_bytes:] == 0xEE).all()


@pytest.mark.parametrize("victim", [0, 5, 11])
def test_batched_decoder_names_the_damaged_tensor_and_decodes_the_rest(victim):
    fmt, chunk_bytes = zc.FMT_FP8_E4M3, 4096
    sizes = _sizes(fmt, chunk_bytes)
    datas, conts = _oracle_containers(fmt, sizes, chunk_bytes, 77)
    bad = conts[victim].copy()
    bad[17] ^= 0x40                                                  # chunk_bytes field of the header
    conts[victim] = bad
    plans = [zc.plan(fmt, n, chunk_bytes) for n in sizes]
    d_comps = [_to_dev(c) for c in conts]
    d_outs = [torch.full((p.input_bytes + 16,), 0xEE, dtype=torch.uint8, device=DEV) for p in plans]
    ws = torch.zeros(256, dtype=torch.uint8, device=DEV)
    zc.decompress_batch(zc.DecompressBatch(plans, d_comps, [c.size for c in conts], d_outs), ws)
    assert zc.batch_status(ws) == (zc.E_CORRUPT, victim)
    for t, (p, data, out) in enumerate(zip(plans, datas, d_outs)):
        back = out.cpu().numpy()
        if t == victim:
            assert (back == 0xEE).all()                              # nothing of it was written
        else:
            assert np.array_equal(back[: p.input_bytes], data[: p.input_bytes])


def test_batch_argument_checks():
    pa, pb = zc.plan(zc.FMT_BF16, 5000, 4096), zc.plan(zc.FMT_BF16, 5000, 8192)
    pc = zc.plan(zc.FMT_FP8_E4M3, 5000, 4096)
    d = [torch.zeros(1 << 15, dtype=torch.uint8, device=DEV) for _ in range(2)]
    o = [torch.zeros(1 << 15, dtype=torch.uint8, device=DEV) for _ in range(2)]
    ws = torch.zeros(256, dtype=torch.uint8, device=DEV)
    for plans in ([pa, pb], [pa, pc]):
        with pytest.raises(zc.ZcError) as e:
            zc.decompress_batch(zc.DecompressBatch(plans, d, [1 << 15] * 2, o), ws)
        assert e.value.status == zc.E_INVALID_ARG
    with pytest.raises(zc.ZcError) as e:
        zc.decompress_batch(zc.DecompressBatch([pa, pa], d, [1 << 15, 64], o), ws)
    assert e.value.status == zc.E_CORRUPT
    zc.decompress_batch(zc.DecompressBatch([], [], [], []), ws)      # nothing to do


# ---- the batched encoder ----

def _batch_compress(fmt, sizes, chunk_bytes, seed, policies):
    datas = [_weights(fmt, n, seed + i) for i, n in enumerate(sizes)]
    plans = [zc.plan(fmt, n, chunk_bytes) for n in sizes]
    hists = [zo.histogram(fmt, d, n) for d, n in zip(datas, sizes)]
    cbs = [zc.build_codebook(p, h, policies[i % len(policies)]) for i, (p, h) in enumerate(zip(plans, hists))]
    ocbs = [zo.build_codebook(h, policies[i % len(policies)]) for i, h in enumerate(hists)]
    d_ins = [_to_dev(d) for d in datas]
    d_outs = [torch.full((p.max_compressed_bytes + 64,), 0xA5, dtype=torch.uint8, device=DEV) for p in plans]
    batch = zc.CompressBatch(plans, d_ins, [o[: p.max_compressed_bytes] for o, p in zip(d_outs, plans)])
    batch.set_codebooks(cbs)
    ws = torch.full((batch.workspace_bytes,), 0x5A, dtype=torch.uint8, device=DEV)
    return datas, plans, ocbs, d_outs, batch, ws


@pytest.mark.parametrize("fmt", FORMATS)
@pytest.mark.parametrize("chunk_bytes", [1024, 4096, 16384])
def test_batched_encoder_writes_the_oracle_s_containers(fmt, chunk_bytes):
    sizes = _sizes(fmt, chunk_bytes)
    policies = [zc.POLICY_AUTO, zc.POLICY_HUFF_ALL, zc.POLICY_RAW_ALL]
    datas, plans, ocbs, d_outs, batch, ws = _batch_compress(fmt, sizes, chunk_bytes, 3000 * fmt + chunk_bytes, policies)
    for _ in range(2):                                               # twice in a row on the same workspace
        got_sizes = zc.compress_batch(batch, ws)
        assert zc.batch_status(ws) == (zc.OK, None)
        for n, data, p, ocb, out, nbytes in zip(sizes, datas, plans, ocbs, d_outs, got_sizes):
            want = zo.compress(fmt, data, n, chunk_bytes, ocb)
            cont = out.cpu().numpy()
            assert nbytes == want.size
            assert np.array_equal(cont[:nbytes], want)
            assert (cont[p.max_compressed_bytes:] == 0xA5).all()     # canary after the buffer


def test_batched_encoder_many_small_tensors_and_the_batched_decoder_after_it():
    fmt, chunk_bytes = zc.FMT_BF16, 1024
    rng = np.random.default_rng(11)
    sizes = [int(v) for v in rng.integers(0, 6000, 700)]
    datas, plans, ocbs, d_outs, batch, ws = _batch_compress(fmt, sizes, chunk_bytes, 9, [zc.POLICY_AUTO, zc.POLICY_HUFF_ALL])
    got_sizes = zc.compress_batch(batch, ws)
    for n, data, ocb, out, nbytes in zip(sizes, datas, ocbs, d_outs, got_sizes):
        want = zo.compress(fmt, data, n, chunk_bytes, ocb)
        assert nbytes == want.size and np.array_equal(out[:nbytes].cpu().numpy(), want)
    backs = [torch.full((p.input_bytes + 16,), 0xEE, dtype=torch.uint8, device=DEV) for p in plans]
    zc.decompress_batch(zc.DecompressBatch(plans, d_outs, got_sizes, backs), ws)
    assert zc.batch_status(ws) == (zc.OK, None)
    for p, data, back in zip(plans, datas, backs):
        assert np.array_equal(back[: p.input_bytes].cpu().numpy(), data[: p.input_bytes])


@pytest.mark.parametrize("fmt", [zc.FMT_BF16, zc.FMT_FP8_E4M3])
def test_batched_encoder_with_codebooks_shared_between_tensors(fmt):
    """Pages of a K/V cache share their dictionaries (Sec. 3.3): three static codebooks serve 40 tensors, a few
    tensors bring their own; every container equals the oracle's with the same code."""
    chunk_bytes = 4096
    rng = np.random.default_rng(3)
    G = zo.group(fmt)
    sizes = [int(v) * 2 * G for v in rng.integers(1, 12000, 40)] + [0, 2 * G]
    datas = [_weights(fmt, n, 500 + i) for i, n in enumerate(sizes)]
    plans = [zc.plan(fmt, n, chunk_bytes) for n in sizes]
    hists = [zo.histogram(fmt, d, n) for d, n in zip(datas, sizes)]
    shared = [zc.build_codebook(plans[k], hists[k], zc.POLICY_STATIC) for k in range(3)]
    oshared = [zo.build_codebook(hists[k], zo.POLICY_STATIC) for k in range(3)]
    cbs, ocbs = [], []
    for i in range(len(sizes)):
        if i % 7 == 6:                                               # its own codebook
            cbs.append(zc.build_codebook(plans[i], hists[i], zc.POLICY_AUTO))
            ocbs.append(zo.build_codebook(hists[i], zo.POLICY_AUTO))
        else:
            cbs.append(shared[i % 3])
            ocbs.append(oshared[i % 3])
    d_ins = [_to_dev(d) for d in datas]
    d_outs = [torch.full((p.max_compressed_bytes,), 0xA5, dtype=torch.uint8, device=DEV) for p in plans]
    batch = zc.CompressBatch(plans, d_ins, d_outs)
    batch.set_codebooks(cbs)
    ws = torch.full((batch.workspace_bytes,), 0x5A, dtype=torch.uint8, device=DEV)
    for _ in range(2):
        got = zc.compress_batch(batch, ws)
        for n, data, ocb, out, nbytes in zip(sizes, datas, ocbs, d_outs, got):
            want = zo.compress(fmt, data, n, chunk_bytes, ocb)
            assert nbytes == want.size and np.array_equal(out[:nbytes].cpu().numpy(), want)
    backs = [torch.full((p.input_bytes + 16,), 0xEE, dtype=torch.uint8, device=DEV) for p in plans]
    dws = torch.zeros(256, dtype=torch.uint8, device=DEV)
    zc.decompress_batch(zc.DecompressBatch(plans, d_outs, got, backs), dws)
    assert zc.batch_status(dws) == (zc.OK, None)
    for p, data, back in zip(plans, datas, backs):
        assert np.array_equal(back[: p.input_bytes].cpu().numpy(), data[: p.input_bytes])


@pytest.mark.parametrize("count", [5, 90])
def test_a_captured_batched_encode_keeps_its_arguments(count):
    """A serving step with static dictionaries in a CUDA graph: replayed after other calls of the same thread, on the pages'
    new contents, it still codes its own tensors with its own tables (few and many: small and large uploads)."""
    fmt, chunk_bytes, n = zc.FMT_BF16, 4096, 9000
    sizes = [n + 16 * i for i in range(count)]
    plans = [zc.plan(fmt, m, chunk_bytes) for m in sizes]
    hists = [zo.histogram(fmt, _weights(fmt, m, 60 + i), m) for i, m in enumerate(sizes)]
    cbs = [zc.build_codebook(p, h, zc.POLICY_STATIC) for p, h in zip(plans, hists)]
    ocbs = [zo.build_codebook(h, zc.POLICY_STATIC) for h in hists]
    d_ins = [_to_dev(_weights(fmt, m, 60 + i)) for i, m in enumerate(sizes)]
    d_outs = [torch.zeros(p.max_compressed_bytes, dtype=torch.uint8, device=DEV) for p in plans]
    batch = zc.CompressBatch(plans, d_ins, d_outs)
    batch.set_codebooks(cbs)
    ws = torch.empty(batch.workspace_bytes, dtype=torch.uint8, device=DEV)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        zc.compress_batch(batch, ws, sync=False)
    for seed in (200, 500):
        _, _, _, _, other, other_ws = _batch_compress(fmt, [7000 + 100 * i for i in range(2 * count)], chunk_bytes, seed, [zc.POLICY_HUFF_ALL])
        zc.compress_batch(other, other_ws)
        datas = [_weights(fmt, m, seed + 7 * i) for i, m in enumerate(sizes)]
        for t, d, o in zip(d_ins, datas, d_outs):
            t[: d.size] = torch.from_numpy(d).to(DEV)
            o.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert zc.batch_status(ws) == (zc.OK, None)
        for m, d, ocb, o in zip(sizes, datas, ocbs, d_outs):
            want = zo.compress(fmt, d, m, chunk_bytes, ocb)
            assert np.array_equal(o[: want.size].cpu().numpy(), want)


def test_batched_encoder_reports_a_symbol_without_code_and_its_tensor():
    fmt, chunk_bytes = zc.FMT_BF16, 4096
    sizes = [30000, 50000, 20000]
    datas = [_weights(fmt, n, 40 + i) for i, n in enumerate(sizes)]
    plans = [zc.plan(fmt, n, chunk_bytes) for n in sizes]
    hists = [zo.histogram(fmt, d, n) for d, n in zip(datas, sizes)]
    missing = int(np.flatnonzero(hists[1][0] == 0)[0])
    bad = datas[1].copy().view(np.uint16); bad[777] = missing << 7
    datas[1] = bad.view(np.uint8)
    cbs = [zc.build_codebook(p, h, zc.POLICY_HUFF_ALL) for p, h in zip(plans, hists)]
    d_ins = [_to_dev(d) for d in datas]
    d_outs = [torch.zeros(p.max_compressed_bytes, dtype=torch.uint8, device=DEV) for p in plans]
    batch = zc.CompressBatch(plans, d_ins, d_outs)
    batch.set_codebooks(cbs)
    ws = torch.zeros(batch.workspace_bytes, dtype=torch.uint8, device=DEV)
    with pytest.raises(zc.ZcError) as e:
        zc.compress_batch(batch, ws)
    assert e.value.status == zc.E_NO_CODE
    assert zc.batch_status(ws) == (zc.E_NO_CODE, 1)


def test_compress_batch_argument_checks():
    pa, pb = zc.plan(zc.FMT_BF16, 5000, 4096), zc.plan(zc.FMT_BF16, 5000, 8192)
    d = [torch.zeros(1 << 15, dtype=torch.uint8, device=DEV) for _ in range(2)]
    o = [torch.zeros(1 << 15, dtype=torch.uint8, device=DEV) for _ in range(2)]
    cb = zc.build_codebook(pa, np.ones((2, 256)), zc.POLICY_AUTO)
    batch = zc.CompressBatch([pa, pb], d, o)
    batch.set_codebooks([cb, cb])
    ws = torch.zeros(1 << 16, dtype=torch.uint8, device=DEV)
    with pytest.raises(zc.ZcError) as e:
        zc.compress_batch(batch, ws)
    assert e.value.status == zc.E_INVALID_ARG
    batch = zc.CompressBatch([pa, pa], d, [o[0], o[1][:100]])
    batch.set_codebooks([cb, cb])
    with pytest.raises(zc.ZcError) as e:
        zc.compress_batch(batch, ws)
    assert e.value.status == zc.E_BUFFER_TOO_SMALL
    batch = zc.CompressBatch([pa, pa], d, o)
    batch.set_codebooks([cb, cb])
    with pytest.raises(zc.ZcError) as e:
        zc.compress_batch(batch, ws[:256])
    assert e.value.status == zc.E_BUFFER_TOO_SMALL


# ---- the batched histogram ----

@pytest.mark.parametrize("fmt", FORMATS)
def test_batched_histogram_counts_every_tensor(fmt):
    G = zo.group(fmt)
    rng = np.random.default_rng(fmt)
    sizes = [0, 2 * G, 8 * G - 2 * G, 8 * G, 8 * G + 2 * G, 100000 * G + 6 * G, 0, 16 * G, 3 * G * 2, 1 << 21, 12345 * 2 * G] + \
            [int(v) * 2 * G for v in rng.integers(0, 5000, 40)]
    datas = [_weights(fmt, n, 500 + i) for i, n in enumerate(sizes)]
    plans = [zc.plan(fmt, n, 4096) for n in sizes]
    d_ins = [_to_dev(d) for d in datas]
    d_hists = torch.full((len(sizes), 2, 256), -1, dtype=torch.int64, device=DEV)
    zc.histogram_batch(zc.HistogramBatch(plans, d_ins), d_hists)
    got = d_hists.cpu().numpy().astype(np.uint64)
    for i, (n, data) in enumerate(zip(sizes, datas)):
        assert np.array_equal(got[i], zo.histogram(fmt, data, n)), f"tensor {i} ({n} elements)"


# ---- XOR-delta forms (delta checkpoints, Sec. 3.1 / 4.1) ----

def _checkpoint_pair(fmt, n, seed):
    """Two tensors that differ little: the second one is the first with a few low mantissa bits flipped here and
    there and a sprinkling of completely different elements."""
    rng = np.random.default_rng(seed)
    a = _weights(fmt, n, seed)
    b = a.copy()
    if b.size:
        flip = rng.random(b.size) < 0.3
        b[flip] ^= rng.integers(0, 4, int(flip.sum()), dtype=np.uint8)
        wild = rng.random(b.size) < 0.002
        b[wild] = rng.integers(0, 256, int(wild.sum()), dtype=np.uint8)
    return a, b


@pytest.mark.parametrize("fmt", [zc.FMT_BF16, zc.FMT_FP8_E4M3])
@pytest.mark.parametrize("chunk_bytes", [1024, 4096, 16384])
def test_xor_delta_single_calls_match_the_oracle_on_the_xor(fmt, chunk_bytes):
    G = zo.group(fmt)
    cs = chunk_bytes // 2
    for n in [0, 2 * G, 5 * cs * G + cs * G // 3 + 2 * G, 23 * cs * G + 6 * G]:
        base, cur = _checkpoint_pair(fmt, n, chunk_bytes + n)
        delta = base ^ cur                                            # the plain definition of what is coded
        p = zc.plan(fmt, n, chunk_bytes)
        d_cur, d_base = _to_dev(cur), _to_dev(base)
        hist = zc.histogram(p, d_cur, d_base=d_base).cpu().numpy().astype(np.uint64)
        assert np.array_equal(hist, zo.histogram(fmt, delta, n))
        cb, ocb = zc.build_codebook(p, hist, zc.POLICY_AUTO), zo.build_codebook(hist, zc.POLICY_AUTO)
        d_out = torch.full((p.max_compressed_bytes,), 0xA5, dtype=torch.uint8, device=DEV)
        ws = torch.empty(p.workspace_bytes, dtype=torch.uint8, device=DEV)
        nbytes = zc.compress(p, cb, d_cur, d_out, ws, d_base=d_base)
        want = zo.compress(fmt, delta, n, chunk_bytes, ocb)
        assert nbytes == want.size and np.array_equal(d_out[:nbytes].cpu().numpy(), want)
        d_back = torch.full((p.input_bytes + 32,), 0xEE, dtype=torch.uint8, device=DEV)
        zc.decompress(p, d_out, nbytes, d_back, ws, d_base=d_base)
        assert zc.device_status(p, ws) == zc.OK
        back = d_back.cpu().numpy()
        assert np.array_equal(back[: p.input_bytes], cur[: p.input_bytes]) and (back[p.input_bytes:] == 0xEE).all()


def _mixed_delta(fmt, chunk_bytes):
    """base, current, their XOR and the element count: chunks 0, 3, 5, 8, 10 and the ragged end unchanged; 1-2 mantissa
    bits only; 4 lowest exponent bit only; 6-7 everything; 9 mantissa bits in its first half."""
    G = zo.group(fmt)
    cs = chunk_bytes // 2
    n_syms = 11 * cs + cs // 3 + 5
    n = n_syms * G
    rng = np.random.default_rng(chunk_bytes + fmt)
    base = _weights(fmt, n, 5 + chunk_bytes)[: 2 * n_syms].copy()
    delta = np.zeros_like(base)
    if fmt == zc.FMT_BF16:
        view, mant, expo, full = delta.view(np.uint16), 0x0003, 0x0080, 0x10000     # sign 15, exponent 14..7, mantissa 6..0
    else:
        view, mant, expo, full = delta, 0x03, 0x08, 0x100                             # sign 7, exponent 6..3, mantissa 2..0
    per_chunk = 2 * cs // view.itemsize
    def span(c0, c1): return view[c0 * per_chunk: c1 * per_chunk]
    d = span(1, 3); d[:] = rng.integers(0, mant + 1, d.size) * (rng.random(d.size) < 0.4)
    d = span(4, 5); d[:] = (rng.random(d.size) < 0.05) * expo
    d = span(6, 8); d[:] = rng.integers(0, full, d.size) * (rng.random(d.size) < 0.2)
    d = span(9, 10); d[: d.size // 2] = rng.integers(0, mant + 1, d.size // 2)
    return base, base ^ delta, delta, n


@pytest.mark.parametrize("fmt", [zc.FMT_BF16, zc.FMT_FP8_E4M3])
@pytest.mark.parametrize("chunk_bytes", [2048, 4096, 16384, 65536])
def test_xor_delta_with_unchanged_stretches(fmt, chunk_bytes):
    """A later checkpoint in which whole stretches did not move, stretches where only the low mantissa bits moved (the
    exponent stream of those chunks is constant, the other stream is not), stretches where only exponent bits
    moved, ordinary stretches, and an unchanged ragged end: every mix of constant and coded chunks in the two
    streams, with both streams Huffman-coded."""
    cs = chunk_bytes // 2
    base, cur, delta, n = _mixed_delta(fmt, chunk_bytes)
    p = zc.plan(fmt, n, chunk_bytes)
    d_cur, d_base = _to_dev(cur), _to_dev(base)
    hist = zc.histogram(p, d_cur, d_base=d_base).cpu().numpy().astype(np.uint64)
    assert np.array_equal(hist, zo.histogram(fmt, delta, n))
    for policy in (zc.POLICY_HUFF_ALL, zc.POLICY_AUTO):
        cb, ocb = zc.build_codebook(p, hist, policy), zo.build_codebook(hist, policy)
        d_out = torch.full((p.max_compressed_bytes,), 0xA5, dtype=torch.uint8, device=DEV)
        ws = torch.empty(p.workspace_bytes, dtype=torch.uint8, device=DEV)
        nbytes = zc.compress(p, cb, d_cur, d_out, ws, d_base=d_base)
        want = zo.compress(fmt, delta, n, chunk_bytes, ocb)
        assert nbytes == want.size and np.array_equal(d_out[:nbytes].cpu().numpy(), want)
        if policy == zc.POLICY_HUFF_ALL:
            hd = zo.parse_header(want)
            assert all(st["payload_bits"] < 8 * 4 * cs for st in hd["streams"])      # most chunks of either stream cost nothing
        d_back = torch.full((p.input_bytes + 32,), 0xEE, dtype=torch.uint8, device=DEV)
        zc.decompress(p, d_out, nbytes, d_back, ws, d_base=d_base)
        assert zc.device_status(p, ws) == zc.OK
        back = d_back.cpu().numpy()
        assert np.array_equal(back[: p.input_bytes], cur[: p.input_bytes]) and (back[p.input_bytes:] == 0xEE).all()


def test_xor_delta_batched_calls():
    fmt, chunk_bytes = zc.FMT_BF16, 4096
    sizes = _sizes(fmt, chunk_bytes)
    pairs = [_checkpoint_pair(fmt, n, 900 + i) for i, n in enumerate(sizes)]
    plans = [zc.plan(fmt, n, chunk_bytes) for n in sizes]
    d_bases = [_to_dev(a) for a, _ in pairs]
    d_curs = [_to_dev(b) for _, b in pairs]
    d_bases[3] = None                                                 # one tensor of the batch without a base
    deltas = [(b if i == 3 else a ^ b) for i, (a, b) in enumerate(pairs)]
    d_hists = torch.zeros((len(sizes), 2, 256), dtype=torch.int64, device=DEV)
    zc.histogram_batch(zc.HistogramBatch(plans, d_curs, d_bases), d_hists)
    hists = d_hists.cpu().numpy().astype(np.uint64)
    for i, (n, d) in enumerate(zip(sizes, deltas)):
        assert np.array_equal(hists[i], zo.histogram(fmt, d, n))
    cbs = zc.build_codebooks(plans, hists, zc.POLICY_AUTO)
    d_outs = [torch.zeros(p.max_compressed_bytes, dtype=torch.uint8, device=DEV) for p in plans]
    batch = zc.CompressBatch(plans, d_curs, d_outs, d_bases)
    batch.set_codebooks(cbs)
    ws = torch.empty(batch.workspace_bytes, dtype=torch.uint8, device=DEV)
    got = zc.compress_batch(batch, ws)
    for i, (n, d) in enumerate(zip(sizes, deltas)):
        want = zo.compress(fmt, d, n, chunk_bytes, zo.build_codebook(hists[i], zc.POLICY_AUTO))
        assert got[i] == want.size and np.array_equal(d_outs[i][: got[i]].cpu().numpy(), want)
    backs = [torch.full((p.input_bytes + 16,), 0xEE, dtype=torch.uint8, device=DEV) for p in plans]
    zc.decompress_batch(zc.DecompressBatch(plans, d_outs, got, backs, d_bases), ws)
    assert zc.batch_status(ws) == (zc.OK, None)
    for p, (a, b), back in zip(plans, pairs, backs):
        out = back.cpu().numpy()
        assert np.array_equal(out[: p.input_bytes], b[: p.input_bytes]) and (out[p.input_bytes:] == 0xEE).all()


@pytest.mark.parametrize("fmt,chunk_bytes", [(zc.FMT_BF16, 8192), (zc.FMT_BF16, 13312), (zc.FMT_BF16, 24576), (zc.FMT_FP8_E4M3, 16384)])
def test_batched_delta_of_tensors_that_end_in_constant_chunks_and_a_partial_batch(fmt, chunk_bytes):
    """Chunks of several warps' tiles, both streams coded.  A constant chunk is coded without the team of warps meeting a
    second time, and in a tensor's last batch some teams have no chunk at all: tensors of every length on both sides of a
    batch whose chunks are constant up to the end, so that teams go from a constant chunk over a batch without one to the
    next tensor's first chunk."""
    G = zo.group(fmt)
    cs = chunk_bytes // 2
    rng = np.random.default_rng(chunk_bytes)
    sizes, bases, curs, deltas = [], [], [], []
    for i in range(360):
        chunks = 1 + i % 17
        n = (chunks * cs - (int(rng.integers(1, cs)) if i % 5 == 4 else 0)) * G
        base = _weights(fmt, n, 3000 + i)
        delta = np.zeros_like(base)
        head = min(base.size, chunk_bytes * (1 + i % 3))                 # what is not constant
        delta[:head] = rng.integers(0, 4, head, dtype=np.uint8) * (rng.random(head) < 0.3)
        sizes.append(n); bases.append(base); curs.append(base ^ delta); deltas.append(delta)
    plans = [zc.plan(fmt, n, chunk_bytes) for n in sizes]
    hists = [zo.histogram(fmt, d, n) for d, n in zip(deltas, sizes)]
    ocbs = [zo.build_codebook(h, zc.POLICY_HUFF_ALL) for h in hists]
    d_bases, d_curs = [_to_dev(b) for b in bases], [_to_dev(c) for c in curs]
    d_outs = [torch.empty(p.max_compressed_bytes, dtype=torch.uint8, device=DEV) for p in plans]
    batch = zc.CompressBatch(plans, d_curs, d_outs, d_bases)
    batch.set_codebooks([zc.build_codebook(p, h, zc.POLICY_HUFF_ALL) for p, h in zip(plans, hists)])
    ws = torch.empty(batch.workspace_bytes, dtype=torch.uint8, device=DEV)
    wants = [zo.compress(fmt, d, n, chunk_bytes, ocb) for d, n, ocb in zip(deltas, sizes, ocbs)]
    for _ in range(5):
        for o in d_outs:
            o.fill_(0xA5)
        got = zc.compress_batch(batch, ws)
        for t, (want, out, nbytes) in enumerate(zip(wants, d_outs, got)):
            assert nbytes == want.size and np.array_equal(out[:nbytes].cpu().numpy(), want), t
    backs = [torch.full((max(p.input_bytes, 16),), 0xEE, dtype=torch.uint8, device=DEV) for p in plans]
    zc.decompress_batch(zc.DecompressBatch(plans, d_outs, got, backs, d_bases), ws)
    assert zc.batch_status(ws) == (zc.OK, None)
    for p, cur, back in zip(plans, curs, backs):
        assert np.array_equal(back[: p.input_bytes].cpu().numpy(), cur[: p.input_bytes])


def test_batched_calls_at_bench_size_on_sampled_chunks():
    """Tensors of the size class the benchmark times (a 14336 x 4096 and a 4096 x 4096 BF16 matrix and a 1024 x 4096
    one, 4 KiB chunks, the batched calls): the oracle decodes sampled chunks one by one, properties that hold at
    any size cover the rest."""
    fmt, chunk_bytes = zc.FMT_BF16, 4096
    shapes = [(14336, 4096), (4096, 4096), (1024, 4096)]
    g = torch.Generator(device=DEV); g.manual_seed(99)
    d_ins, plans = [], []
    for r, c in shapes:
        x = (torch.randn(r * c, generator=g, device=DEV) * 0.02).to(torch.bfloat16)
        d_ins.append(x.view(torch.uint8))
        plans.append(zc.plan(fmt, r * c, chunk_bytes))
    n_t = len(plans)
    d_hists = torch.zeros((n_t, 2, 256), dtype=torch.int64, device=DEV)
    zc.histogram_batch(zc.HistogramBatch(plans, d_ins), d_hists)
    hists = d_hists.cpu().numpy().astype(np.uint64)
    for t in range(n_t):
        assert int(hists[t, 0].sum()) == plans[t].n_syms and int(hists[t, 1].sum()) == plans[t].n_syms
    cbs = zc.build_codebooks(plans, hists, zc.POLICY_AUTO)
    d_outs = [torch.empty(p.max_compressed_bytes, dtype=torch.uint8, device=DEV) for p in plans]
    enc = zc.CompressBatch(plans, d_ins, d_outs)
    enc.set_codebooks(cbs)
    ws = torch.empty(enc.workspace_bytes, dtype=torch.uint8, device=DEV)
    sizes = zc.compress_batch(enc, ws)
    rng = np.random.default_rng(0)
    for t in range(n_t):
        p = plans[t]
        cont = d_outs[t][: sizes[t]].cpu().numpy()
        assert zc.validate_container(p, cont) == zc.OK
        hd = zo.parse_header(cont)
        assert hd["total_bytes"] == sizes[t] and hd["n_chunks"] == p.n_chunks
        for s in range(2):
            mode, lens, _ = cbs[t].get(s)
            want_bits = int((hists[t, s].astype(np.int64) * lens).sum()) if mode == zc.MODE_HUFF else 8 * p.n_syms
            assert hd["streams"][s]["payload_bits"] == want_bits
        data = d_ins[t].cpu().numpy()
        for c in [0, 1, p.n_chunks - 1] + [int(v) for v in rng.integers(0, p.n_chunks, 10)]:
            got = zo.decompress_chunk(cont, c, chunk_bytes)
            assert np.array_equal(got, data[c * chunk_bytes: c * chunk_bytes + got.size]), (t, c)
    d_backs = [torch.empty(p.input_bytes, dtype=torch.uint8, device=DEV) for p in plans]
    zc.decompress_batch(zc.DecompressBatch(plans, d_outs, sizes, d_backs), ws)
    assert zc.batch_status(ws) == (zc.OK, None)
    for b, x in zip(d_backs, d_ins):
        assert torch.equal(b, x)


@pytest.mark.parametrize("fmt", [zc.FMT_BF16, zc.FMT_FP8_E4M3])
@pytest.mark.parametrize("chunk_bytes", [2048, 4096, 65536])
def test_whole_containers_at_bench_size_equal_the_oracle_s(fmt, chunk_bytes):
    """Tensors of the size class the benchmark times, in one batched call that crosses tensor boundaries: every byte
    of every container against the oracle (not a sample).  The large tensor has thousands of batches, far more
    than blocks run at a time, so its chunks are placed through many rounds of the look-back; the ragged one ends
    in the middle of a chunk."""
    G = zo.group(fmt)
    sizes = [(24 << 20) * G, (3 << 20) * G + 1234 * G + 2 * G, 0, (7 << 20) * G]     # 48 MiB, 6 MiB + a bit, nothing, 14 MiB of BF16
    g = torch.Generator(device=DEV); g.manual_seed(7 + chunk_bytes)
    d_ins, plans, datas = [], [], []
    for i, n in enumerate(sizes):
        x = torch.randn(max(n, 16), generator=g, device=DEV) * (0.02 / (1 + i))
        if fmt == zc.FMT_BF16:
            b = x.to(torch.bfloat16).view(torch.uint8)[: 2 * n]
        else:
            b = (x / (x.abs().max() / 448)).clamp(-448, 448).to(torch.float8_e4m3fn).view(torch.uint8)[:n]
        d_ins.append(b.contiguous() if n else torch.zeros(16, dtype=torch.uint8, device=DEV))
        datas.append(b.cpu().numpy().copy() if n else np.zeros(0, np.uint8))
        plans.append(zc.plan(fmt, n, chunk_bytes))
    n_t = len(plans)
    d_hists = torch.zeros((n_t, 2, 256), dtype=torch.int64, device=DEV)
    zc.histogram_batch(zc.HistogramBatch(plans, d_ins), d_hists)
    hists = d_hists.cpu().numpy().astype(np.uint64)
    cbs = zc.build_codebooks(plans, hists, zc.POLICY_AUTO)
    d_outs = [torch.empty(p.max_compressed_bytes, dtype=torch.uint8, device=DEV) for p in plans]
    enc = zc.CompressBatch(plans, d_ins, d_outs)
    enc.set_codebooks(cbs)
    ws = torch.empty(enc.workspace_bytes, dtype=torch.uint8, device=DEV)
    got_sizes = zc.compress_batch(enc, ws)
    for t in range(n_t):
        assert np.array_equal(hists[t], zo.histogram(fmt, datas[t], sizes[t]))
        want = zo.compress(fmt, datas[t], sizes[t], chunk_bytes, zo.build_codebook(hists[t], zo.POLICY_AUTO))
        assert got_sizes[t] == want.size
        assert np.array_equal(d_outs[t][: got_sizes[t]].cpu().numpy(), want), f"container of tensor {t} differs"
    d_backs = [torch.empty(max(p.input_bytes, 16), dtype=torch.uint8, device=DEV) for p in plans]
    zc.decompress_batch(zc.DecompressBatch(plans, d_outs, got_sizes, d_backs), ws)
    assert zc.batch_status(ws) == (zc.OK, None)
    for p, b, x in zip(plans, d_backs, d_ins):
        assert torch.equal(b[: p.input_bytes], x[: p.input_bytes])


@pytest.mark.parametrize("fmt,chunk_bytes,chunks", [(zc.FMT_BF16, 4096, k) for k in (1, 31, 149, 2500, 5500)] +
                         [(zc.FMT_FP8_E4M3, 16384, k) for k in (1, 149, 700)] + [(zc.FMT_BF16, 1024, k) for k in (60000, 150000)])
def test_batches_from_one_chunk_to_several_rounds(fmt, chunk_bytes, chunks):
    """The batched encoder holds one to three batches of a block, by the number of chunks, and the batched decoder's blocks go
    from less than a chunk to dozens per warp: totals on both sides of those lines, in a large, a ragged and an empty tensor."""
    cs = chunk_bytes // 2 * zo.group(fmt)
    a = chunks * 2 // 3
    sizes = [a * cs, 0, max((chunks - a) * cs - 3, 1)]
    datas, plans, ocbs, d_outs, batch, ws = _batch_compress(fmt, sizes, chunk_bytes, 40 + chunks, [zc.POLICY_AUTO, zc.POLICY_HUFF_ALL])
    got_sizes = zc.compress_batch(batch, ws)
    assert zc.batch_status(ws) == (zc.OK, None)
    for n, data, ocb, out, nbytes in zip(sizes, datas, ocbs, d_outs, got_sizes):
        assert np.array_equal(out[:nbytes].cpu().numpy(), zo.compress(fmt, data, n, chunk_bytes, ocb))
    backs = [torch.full((p.input_bytes + 16,), 0xEE, dtype=torch.uint8, device=DEV) for p in plans]
    zc.decompress_batch(zc.DecompressBatch(plans, d_outs, got_sizes, backs), ws)
    assert zc.batch_status(ws) == (zc.OK, None)
    for p, data, back in zip(plans, datas, backs):
        back = back.cpu().numpy()
        assert np.array_equal(back[: p.input_bytes], data[: p.input_bytes]) and (back[p.input_bytes:] == 0xEE).all()


def _encoded_batch(fmt, chunk_bytes, d_ins, sizes, d_bases=None, policy=None):
    """Containers of tensors on the device, by the library's own encoder (compared with the oracle's elsewhere)."""
    plans = [zc.plan(fmt, n, chunk_bytes) for n in sizes]
    d_hists = torch.zeros((len(plans), 2, 256), dtype=torch.int64, device=DEV)
    zc.histogram_batch(zc.HistogramBatch(plans, d_ins, d_bases), d_hists)
    d_outs = [torch.empty(p.max_compressed_bytes, dtype=torch.uint8, device=DEV) for p in plans]
    enc = zc.CompressBatch(plans, d_ins, d_outs, d_bases)
    enc.set_codebooks(zc.build_codebooks(plans, d_hists.cpu().numpy(), policy or (zc.POLICY_HUFF_ALL if d_bases else zc.POLICY_AUTO)))
    return plans, d_outs, zc.compress_batch(enc, torch.empty(enc.workspace_bytes, dtype=torch.uint8, device=DEV))


@pytest.mark.parametrize("kind,chunks", [("plain", 300_000), ("plain", 750_000), ("scale", 200_000), ("delta", 200_000)])
def test_batched_decoder_deals_chunks_out_in_several_rounds(kind, chunks):
    """Launches of 64 chunks per warp and more, a block's slice in two to five pieces: a large tensor, an empty one, a ragged one, one
    without a base."""
    fmt = zc.FMT_SCALE_U8 if kind == "scale" else zc.FMT_BF16
    cs = 512 * zo.group(fmt)
    sizes = [(chunks * 5 // 8) * cs, 0, (chunks // 4) * cs - 77, (chunks // 8) * cs + 1]
    tile = torch.from_numpy(_weights(fmt, 8 << 20, chunks)).to(DEV)
    nbytes = [zo.input_bytes(fmt, n) for n in sizes]
    d_ins = [tile.repeat(-(-max(b, 16) // tile.numel()))[: max(b, 16)].clone() for b in nbytes]
    d_bases = None
    if kind == "delta":
        g = torch.Generator(device=DEV); g.manual_seed(1)
        d_bases = [x ^ (torch.rand(x.numel(), generator=g, device=DEV) < 0.1).to(torch.uint8) for x in d_ins]
        d_bases[3] = None
    plans, d_outs, got = _encoded_batch(fmt, 1024, d_ins, sizes, d_bases)
    backs = [torch.zeros_like(x) for x in d_ins]
    ws = torch.zeros(256, dtype=torch.uint8, device=DEV)
    zc.decompress_batch(zc.DecompressBatch(plans, d_outs, got, backs, d_bases), ws)
    assert zc.batch_status(ws) == (zc.OK, None)
    for b, x, n in zip(backs, d_ins, nbytes):
        assert torch.equal(b[:n], x[:n])


@pytest.mark.parametrize("kind,chunks,pieces", [("plain", 300_000, 2), ("plain", 750_000, 3), ("plain", 4_400_000, 4), ("scale", 200_000, 2),
                                                ("delta", 200_000, 5)])
def test_launches_in_several_rounds_have_two_to_five_pieces(kind, chunks, pieces):
    """The launches of the test above, and one of four pieces (plain launches have a fifth from 34 million chunks on)."""
    p = zc.plan(zc.FMT_SCALE_U8 if kind == "scale" else zc.FMT_BF16, 1 << 20, 1024)
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the numbers are those of 148 SMs")
    assert len(zc.test_decoder_pieces(p, kind == "delta", chunks)) == pieces
    if pieces == 4:
        test_batched_decoder_deals_chunks_out_in_several_rounds(kind, chunks)


@pytest.mark.parametrize("unchanged", ["first_half", "every_other", "last_quarter"])
def test_batched_decoder_with_slices_of_unlike_speed(unchanged):
    """Deltas whose unchanged stretches are as long as many blocks' slices: blocks that are through take the other slices' pieces,
    of which there are five."""
    chunks, cs = 400_000, 512
    assert len(zc.test_decoder_pieces(zc.plan(zc.FMT_BF16, cs, 1024), True, chunks)) == 5
    parts = {"first_half": [(300_000, True), (100_000 - 3, False)], "every_other": [(50_000, k % 2 == 0) for k in range(8)],
             "last_quarter": [(299_999, False), (100_001, True)]}[unchanged]
    sizes = [n * cs - 7 * k for k, (n, _) in enumerate(parts)]
    tile = torch.from_numpy(_weights(zc.FMT_BF16, 8 << 20, 5)).to(DEV)
    d_ins = [tile.repeat(-(-2 * n // tile.numel()))[: 2 * n].clone() for n in sizes]
    g = torch.Generator(device=DEV); g.manual_seed(2)
    d_bases = []
    for k, (x, (_, same)) in enumerate(zip(d_ins, parts)):
        step = (torch.rand(x.numel(), generator=g, device=DEV) < 0.3).to(torch.uint8) * 3
        if same:
            step[: x.numel() * 2 // 3 if unchanged == "first_half" else x.numel()] = 0
        d_bases.append(x ^ step)
    plans, d_outs, got = _encoded_batch(zc.FMT_BF16, 1024, d_ins, sizes, d_bases)
    ws = torch.zeros(256, dtype=torch.uint8, device=DEV)
    backs = [torch.zeros_like(x) for x in d_ins]
    for _ in range(3):
        zc.decompress_batch(zc.DecompressBatch(plans, d_outs, got, backs, d_bases), ws)
        assert zc.batch_status(ws) == (zc.OK, None)
        for b, x in zip(backs, d_ins):
            assert torch.equal(b, x)
            b.zero_()


@pytest.mark.parametrize("chunk_bytes", [4096, 32768])
@pytest.mark.parametrize("count", [2, 20, 64, 147, 149])
def test_batched_decoder_with_tensors_of_one_size_and_of_several(count, chunk_bytes):
    """As many ranges as a multiple of the number of tensors, or as there are SMs, whichever is shorter for the longest
    block: tensors of 1, 9 and 20 chunks, the last chunk ragged or not, alone and with empty and unlike tensors among them."""
    fmt, cs = zc.FMT_FP8_E4M3, chunk_bytes
    for chunks in (1, 9, 20):
        n = chunks * cs - (chunks == 9) * 1000
        for mixed in (False, True):
            sizes = [n] * count
            if mixed:
                sizes[0], sizes[count // 2] = 0, 3 * n + 16
            x = torch.from_numpy(_weights(fmt, 4 * n + 16 * count + 16, chunks)).to(DEV)
            d_ins = [x[16 * i: 16 * i + max(m, 16)] for i, m in enumerate(sizes)]
            plans, d_outs, got = _encoded_batch(fmt, chunk_bytes, d_ins, sizes)
            backs = [torch.full((m + 16,), 0xEE, dtype=torch.uint8, device=DEV) for m in sizes]
            ws = torch.zeros(256, dtype=torch.uint8, device=DEV)
            zc.decompress_batch(zc.DecompressBatch(plans, d_outs, got, backs), ws)
            assert zc.batch_status(ws) == (zc.OK, None)
            for b, d, m in zip(backs, d_ins, sizes):
                assert torch.equal(b[:m], d[:m]) and bool((b[m:] == 0xEE).all())


@pytest.mark.parametrize("fmt", FORMATS)
@pytest.mark.parametrize("chunk_bytes", [1024, 2048, 3072, 4096, 5120])
def test_decoder_of_small_chunks_with_one_and_two_coded_streams(fmt, chunk_bytes):
    """Chunks up to 4 KiB have a loop of their own (one or two buffers for raw bytes), in which a container with both streams
    coded goes to fewer warps: tensors of either kind in turn, from one symbol to more chunks than the kernel for few chunks
    takes, ragged and complete, in one batched call and each on its own."""
    cs = chunk_bytes // 2 * zo.group(fmt)
    sizes = [1300 * cs, 2, 0, 1300 * cs - 2, 40 * cs + 8 * zo.group(fmt), cs, cs - 4 * zo.group(fmt), 29 * cs + 2]
    datas, plans, ocbs, d_outs, batch, ws = _batch_compress(fmt, sizes, chunk_bytes, 70, [zc.POLICY_AUTO, zc.POLICY_HUFF_ALL])
    got_sizes = zc.compress_batch(batch, ws)
    backs = [torch.full((p.input_bytes + 16,), 0xEE, dtype=torch.uint8, device=DEV) for p in plans]

    def check():
        for p, data, back in zip(plans, datas, backs):
            back = back.cpu().numpy()
            assert np.array_equal(back[: p.input_bytes], data[: p.input_bytes]) and (back[p.input_bytes:] == 0xEE).all()

    zc.decompress_batch(zc.DecompressBatch(plans, d_outs, got_sizes, backs), ws)
    assert zc.batch_status(ws) == (zc.OK, None)
    check()
    for p, out, nbytes, back in zip(plans, d_outs, got_sizes, backs):
        back.fill_(0xEE)
        zc.decompress(p, out, nbytes, back, ws)
        assert zc.device_status(p, ws) == zc.OK
    check()


@pytest.mark.parametrize("fmt", FORMATS)
@pytest.mark.parametrize("chunk_bytes", [1024, 2048, 3072, 4096, 5120])
def test_decoder_of_small_chunks_without_coded_streams(fmt, chunk_bytes):
    """Containers with both streams raw have a loop of their own up to 4 KiB: several chunks per warp, the last one ragged at every kind of
    place, outputs aligned to 32 and to 16 bytes, batched and alone, plain and (BF16) as a delta."""
    G = zo.group(fmt)
    cs = chunk_bytes // 2 * G
    sizes = [13000 * cs, 9000 * cs - 2, 5000 * cs + 16 * G, 300 * cs + cs // 2 + 8 * G, cs - 2, 2 * cs + 2, 2, 0]
    nbytes = [zo.input_bytes(fmt, n) for n in sizes]
    g = torch.Generator(device=DEV); g.manual_seed(chunk_bytes + fmt)
    d_ins = [torch.randint(0, 256, (max(b, 16),), dtype=torch.uint8, device=DEV, generator=g) for b in nbytes]
    for delta in (False, True)[: 2 if fmt == zc.FMT_BF16 else 1]:
        d_bases = [torch.randint(0, 256, (x.numel(),), dtype=torch.uint8, device=DEV, generator=g) for x in d_ins] if delta else None
        plans, d_outs, got = _encoded_batch(fmt, chunk_bytes, d_ins, sizes, d_bases, zc.POLICY_RAW_ALL)
        for shift in (0, 16):
            bufs = [torch.full((b + 64,), 0xEE, dtype=torch.uint8, device=DEV) for b in nbytes]
            assert all(b.data_ptr() % 32 == 0 for b in bufs)
            backs = [b[shift:] for b in bufs]
            ws = torch.zeros(256, dtype=torch.uint8, device=DEV)

            def check():
                for n, x, b in zip(nbytes, d_ins, bufs):
                    assert torch.equal(b[shift: shift + n], x[:n]) and bool((b[:shift] == 0xEE).all()) and bool((b[shift + n:] == 0xEE).all())
                    b.fill_(0xEE)

            zc.decompress_batch(zc.DecompressBatch(plans, d_outs, got, backs, d_bases), ws)
            assert zc.batch_status(ws) == (zc.OK, None)
            check()
            if not delta:
                for p, out, n, back in zip(plans, d_outs, got, backs):
                    zc.decompress(p, out, n, back, ws)
                    assert zc.device_status(p, ws) == zc.OK
                check()
