"""Parity of the CUDA path with the CPU oracle: bit-exact histograms, containers and round trips.

Everything goes through the C ABI (via the ctypes binding).  Integer work: no tolerance.
"""
import numpy as np
import pytest
import torch

import oracle as zo
from paper_2508_19263_b200 import binding as zc
from paper_2508_19263_b200 import workloads as wl

pytestmark = pytest.mark.gpu
FORMATS = [zc.FMT_BF16, zc.FMT_FP8_E4M3, zc.FMT_FP4_E2M1, zc.FMT_SCALE_U8, zc.FMT_FP8_E5M2]
DEV = "cuda"


def _gpu_round_trip(fmt, data_np, n, chunk_bytes, policy, oracle_codebook_hist=None, check_container=True):
    """Run histogram -> codebook -> compress -> decompress on the GPU and compare every stage with the oracle."""
    p = zc.plan(fmt, n, chunk_bytes)
    d_in = torch.from_numpy(data_np.copy()).to(DEV) if data_np.size else torch.zeros(16, dtype=torch.uint8, device=DEV)
    # histogram
    d_hist = zc.histogram(p, d_in)
    hist = d_hist.cpu().numpy().astype(np.uint64)
    want_hist = zo.histogram(fmt, data_np, n)
    assert np.array_equal(hist, want_hist)
    # codebook (possibly from another histogram: static dictionary)
    hsrc = hist if oracle_codebook_hist is None else oracle_codebook_hist
    cb = zc.build_codebook(p, hsrc, policy)
    ocb = zo.build_codebook(hsrc, policy)
    # compress
    d_out = torch.full((p.max_compressed_bytes + 64,), 0xA5, dtype=torch.uint8, device=DEV)
    d_ws = torch.full((p.workspace_bytes,), 0x5A, dtype=torch.uint8, device=DEV)
    nbytes = zc.compress(p, cb, d_in, d_out[: p.max_compressed_bytes], d_ws)
    cont = d_out[:nbytes].cpu().numpy()
    assert (d_out[p.max_compressed_bytes:].cpu().numpy() == 0xA5).all()        # canary after the buffer
    if check_container:
        want = zo.compress(fmt, data_np, n, chunk_bytes, ocb)
        assert nbytes == want.size
        if not np.array_equal(cont, want):
            bad = np.flatnonzero(cont != want)
            raise AssertionError(f"container differs at {bad[:8]} of {want.size} (first: got {cont[bad[0]]:#x} want {want[bad[0]]:#x})")
        assert zc.validate_container(p, cont) == zc.OK
    # decompress the GPU container on the GPU
    d_back = torch.full((p.input_bytes + 64,), 0xEE, dtype=torch.uint8, device=DEV)
    zc.decompress(p, d_out, nbytes, d_back, d_ws)
    assert zc.device_status(p, d_ws) == zc.OK
    back = d_back.cpu().numpy()
    assert np.array_equal(back[: p.input_bytes], data_np[: p.input_bytes])
    assert (back[p.input_bytes:] == 0xEE).all()
    # and the oracle decodes it too
    assert np.array_equal(zo.decompress(cont, p.input_bytes), data_np[: p.input_bytes])
    return p, cb, hist, cont


def _compress_with_modes(fmt, data_np, n, chunk_bytes, hist, modes):
    """Compress with a HUFF_ALL codebook whose stream modes are overridden (one stream raw), against the oracle."""
    ocb = zo.build_codebook(hist, zo.POLICY_HUFF_ALL)
    ocb.modes = list(modes)
    want = zo.compress(fmt, data_np, n, chunk_bytes, ocb)
    # the library has no call that overrides modes; the policies give the same two combinations on suitable counts
    p = zc.plan(fmt, n, chunk_bytes)
    d_back = torch.full((p.input_bytes + 64,), 0xEE, dtype=torch.uint8, device=DEV)
    d_ws = torch.empty(p.workspace_bytes, dtype=torch.uint8, device=DEV)
    d_comp = torch.from_numpy(want.copy()).to(DEV)
    zc.decompress(p, d_comp, want.size, d_back, d_ws)
    assert zc.device_status(p, d_ws) == zc.OK
    assert np.array_equal(d_back.cpu().numpy()[: p.input_bytes], data_np[: p.input_bytes])


def _weights(fmt, n, seed):
    rng = np.random.default_rng(seed)
    if n == 0:
        return np.zeros(0, np.uint8)
    if fmt == zc.FMT_SCALE_U8:                                       # E8M0-like scale bytes: a narrow bell around 120
        return np.clip(np.round(rng.normal(120, 1.5, n)), 0, 255).astype(np.uint8)
    if fmt == zc.FMT_BF16:
        x = torch.from_numpy((rng.standard_normal(n) * 0.02).astype(np.float32))
        return x.to(torch.bfloat16).view(torch.uint8).numpy().reshape(-1).copy()
    if fmt == zc.FMT_FP8_E4M3:
        x = rng.standard_normal(n).astype(np.float32)
        x = x / (np.abs(x).max() / 448.0)
        return torch.from_numpy(x).to(torch.float8_e4m3fn).view(torch.uint8).numpy().reshape(-1).copy()
    if fmt == zc.FMT_FP8_E5M2:
        x = torch.from_numpy((rng.standard_normal(n) * 0.02).astype(np.float32))
        return x.to(torch.float8_e5m2).view(torch.uint8).numpy().reshape(-1).copy()
    v = rng.choice(16, size=n, p=np.array([6, 5, 4, 3, 2, 1, 1, 1, 6, 5, 4, 3, 2, 1, 1, 1]) / 46.0).astype(np.uint8)
    return (v[0::2] | (v[1::2] << 4)).astype(np.uint8)


@pytest.mark.parametrize("fmt", FORMATS)
@pytest.mark.parametrize("policy", [zc.POLICY_AUTO, zc.POLICY_HUFF_ALL, zc.POLICY_RAW_ALL])
@pytest.mark.parametrize("chunk_bytes", [1024, 2048, 3072, 8192, 16384, 65536])
def test_round_trip_several_chunks_and_ragged_tail(fmt, policy, chunk_bytes):
    G = zo.group(fmt)
    cs = chunk_bytes // 2
    n = (5 * cs + cs // 3 + 11) * G
    if fmt == zc.FMT_FP4_E2M1:
        n -= n % 2
    _gpu_round_trip(fmt, _weights(fmt, n, chunk_bytes + fmt), n, chunk_bytes, policy)


@pytest.mark.parametrize("fmt", FORMATS)
def test_edge_sizes(fmt):
    G = zo.group(fmt)
    chunk_bytes = 1024
    cs = chunk_bytes // 2
    sizes = {0, 1, G - 1, G, G + 1, 2 * G, 7 * G, 8 * G, 9 * G, cs * G - 1, cs * G, cs * G + 1, cs * G + G,
             2 * cs * G, 33 * cs * G + 5 * G, 16 * G - 1, 16 * G + 1}
    for n in sorted(sizes):
        if n < 0 or (fmt == zc.FMT_FP4_E2M1 and n % 2):
            continue
        for policy in (zc.POLICY_AUTO, zc.POLICY_HUFF_ALL):
            _gpu_round_trip(fmt, _weights(fmt, n, 100 + n), n, chunk_bytes, policy)


def test_special_bit_patterns():
    z = np.zeros(20000, np.uint16).view(np.uint8)                     # one active symbol per stream
    _gpu_round_trip(zc.FMT_BF16, z, 20000, 4096, zc.POLICY_HUFF_ALL)
    pats = np.array([0x7FC0, 0xFFC1, 0x7F80, 0xFF80, 0x8000, 0x0001, 0x807F, 0x7FFF] * 3000, np.uint16).view(np.uint8)
    _gpu_round_trip(zc.FMT_BF16, pats, 24000, 4096, zc.POLICY_HUFF_ALL)
    allb = np.tile(np.arange(256, dtype=np.uint8), 100)
    _gpu_round_trip(zc.FMT_FP8_E4M3, allb, allb.size, 2048, zc.POLICY_HUFF_ALL)
    _gpu_round_trip(zc.FMT_FP4_E2M1, allb, 2 * allb.size, 2048, zc.POLICY_HUFF_ALL)
    rng = np.random.default_rng(9)                                    # one exponent value, noise below it: [HUFF, RAW], and
    noisy = (np.uint16(0x3F80) | rng.integers(0, 128, 30000).astype(np.uint16) | (rng.integers(0, 2, 30000).astype(np.uint16) << 15))
    p, cb, _, cont = _gpu_round_trip(zc.FMT_BF16, noisy.view(np.uint8), 30000, 4096, zc.POLICY_AUTO)
    assert cb.modes == [zc.MODE_HUFF, zc.MODE_RAW]                    # the constant exponent chunks cost nothing
    assert zo.parse_header(cont)["streams"][0]["payload_bits"] == 0
    rng = np.random.default_rng(1)
    uni = rng.integers(0, 256, 1 << 18, dtype=np.uint8)               # incompressible: every code length near 8
    _gpu_round_trip(zc.FMT_BF16, uni, 1 << 17, 8192, zc.POLICY_HUFF_ALL)


@pytest.mark.parametrize("fmt", FORMATS)
@pytest.mark.parametrize("chunk_bytes", [1024, 4096, 16384])
def test_chunks_of_nothing_but_the_fill_symbol_take_no_bits(fmt, chunk_bytes):
    """Unchanged stretches of a delta checkpoint or the unused part of a cache page: chunks whose symbols are all the
    symbol with the all-zero code have empty pieces; chunks next to them are coded as usual."""
    G = zo.group(fmt)
    cs = chunk_bytes // 2
    per_sym = 2                                                      # element bytes per symbol in every format
    body = _weights(fmt, 2 * cs * G + 6 * G, 77 + fmt)               # two chunks and a bit of ordinary data
    zeros = lambda n_syms: np.zeros(n_syms * per_sym, np.uint8)
    data = np.concatenate([zeros(3 * cs), body[: (2 * cs + 6) * per_sym], zeros(cs - 6), zeros(4 * cs + cs // 3)])
    n = data.size // per_sym * G
    for policy in (zc.POLICY_HUFF_ALL, zc.POLICY_AUTO):
        _gpu_round_trip(fmt, data, n, chunk_bytes, policy)
    cb = zo.build_codebook(zo.histogram(fmt, data, n), zo.POLICY_HUFF_ALL)
    hd = zo.parse_header(zo.compress(fmt, data, n, chunk_bytes, cb))
    assert hd["streams"][0]["payload_bits"] < 8 * 3 * cs           # far below one bit per symbol of the whole tensor
    # a tensor that is constant altogether: header and tables only
    flat = zeros(5 * cs + 9)
    _gpu_round_trip(fmt, flat, flat.size // per_sym * G, chunk_bytes, zc.POLICY_HUFF_ALL)
    # one stream raw: the coded stream's constant chunks cost nothing all the same
    h = zo.histogram(fmt, data, n)
    p = zc.plan(fmt, n, chunk_bytes)
    for modes in ((zc.MODE_HUFF, zc.MODE_RAW), (zc.MODE_RAW, zc.MODE_HUFF)):
        _compress_with_modes(fmt, data, n, chunk_bytes, h, modes)


def test_long_codes_and_skew():
    """Exponentially skewed exponents: the 12-bit limit binds and codes of every length occur."""
    rng = np.random.default_rng(5)
    n = 300000
    e = np.minimum(rng.geometric(0.45, n) + 100, 254).astype(np.uint16)
    m = rng.integers(0, 128, n).astype(np.uint16)
    s = rng.integers(0, 2, n).astype(np.uint16)
    data = ((s << 15) | (e << 7) | m).astype(np.uint16).view(np.uint8)
    p, cb, hist, cont = _gpu_round_trip(zc.FMT_BF16, data, n, 16384, zc.POLICY_AUTO)
    assert cb.get(0)[1].max() == 12


@pytest.mark.parametrize("policy", [zc.POLICY_AUTO, zc.POLICY_HUFF_ALL])
@pytest.mark.parametrize("chunk_bytes", [1024, 4096, 6144, 8192, 32768])
def test_subchunks_above_eight_bits_per_symbol(chunk_bytes, policy):
    """A static dictionary meets runs of its rarest symbols: some subchunks need 12 bits per symbol, more than
    the staging slot of the encoder holds, in the first, the last, neighbouring and isolated chunks (the chunk
    sizes and the number of coded streams cover every staging layout of the encoder)."""
    rng = np.random.default_rng(chunk_bytes)
    cs = chunk_bytes // 2
    n = 41 * cs + cs // 2 + 3
    common = rng.choice([120, 121, 122, 123], size=n, p=[0.5, 0.25, 0.15, 0.1]).astype(np.uint16)
    e = common.copy()
    rare = np.arange(10, 74, dtype=np.uint16)                      # 64 exponents the dictionary barely knows
    for c in (0, 1, 2, 7, 9, 10, 11, 12, 20, 33, 40, 41):
        lo = c * cs + int(rng.integers(0, cs // 2))
        hi = min(n, lo + int(rng.integers(cs // 16, cs)))
        e[lo:hi] = rare[rng.integers(0, rare.size, hi - lo)]
    m = rng.integers(0, 128, n).astype(np.uint16)
    sgn = rng.integers(0, 2, n).astype(np.uint16)
    data = ((sgn << 15) | (e << 7) | m).astype(np.uint16).view(np.uint8)
    dict_hist = np.zeros((2, 256), np.uint64)
    dict_hist[0, 120:124] = [500000, 250000, 150000, 100000]
    dict_hist[0, rare] = 1
    dict_hist[1] = zo.histogram(zo.BF16, data, n)[1]
    p, cb, hist, cont = _gpu_round_trip(zc.FMT_BF16, data, n, chunk_bytes, policy, oracle_codebook_hist=dict_hist)
    assert cb.get(0)[1][rare].min() > 8
    off16, sub_end, _ = zo.read_tables(cont, 0)
    sub_bits = np.diff(np.concatenate([np.zeros((sub_end.shape[0], 1), np.int64), sub_end.astype(np.int64)], axis=1), axis=1)
    assert (sub_bits > 8 * (cs // 32)).any()                       # the case this test is about did occur


def test_static_dictionary_and_missing_code():
    a = _weights(zc.FMT_BF16, 50000, 1)
    b = _weights(zc.FMT_BF16, 50000, 2)
    ha = zo.histogram(zo.BF16, a, 50000)
    _gpu_round_trip(zc.FMT_BF16, b, 50000, 8192, zc.POLICY_HUFF_ALL, oracle_codebook_hist=ha + 1)
    # a symbol without a code: the device reports it
    p = zc.plan(zc.FMT_BF16, 50000, 8192)
    cb = zc.build_codebook(p, ha, zc.POLICY_HUFF_ALL)
    missing = int(np.flatnonzero(ha[0] == 0)[0])
    bad = b.copy().view(np.uint16); bad[777] = missing << 7
    d_in = torch.from_numpy(bad.view(np.uint8)).to(DEV)
    d_out = torch.empty(p.max_compressed_bytes, dtype=torch.uint8, device=DEV)
    d_ws = torch.empty(p.workspace_bytes, dtype=torch.uint8, device=DEV)
    with pytest.raises(zc.ZcError) as e:
        zc.compress(p, cb, d_in, d_out, d_ws)
    assert e.value.status == zc.E_NO_CODE


def test_decoder_accepts_oracle_containers_and_flags_damage():
    n = 70000
    data = _weights(zc.FMT_BF16, n, 3)
    hist = zo.histogram(zo.BF16, data, n)
    for policy in (zo.POLICY_AUTO, zo.POLICY_HUFF_ALL):
        cont = zo.compress(zo.BF16, data, n, 8192, zo.build_codebook(hist, policy))
        p = zc.plan(zc.FMT_BF16, n, 8192)
        d_ws = torch.empty(p.workspace_bytes, dtype=torch.uint8, device=DEV)
        d_back = torch.zeros(p.input_bytes, dtype=torch.uint8, device=DEV)
        d_c = torch.from_numpy(cont).to(DEV)
        zc.decompress(p, d_c, cont.size, d_back, d_ws)
        assert zc.device_status(p, d_ws) == zc.OK
        assert np.array_equal(d_back.cpu().numpy(), data)
        # header damage and table damage are reported, never trapped on
        hd = zo.parse_header(cont)
        sec = hd["streams"][0]["section_off"]
        used = int(np.flatnonzero(cont[sec:sec + 256])[0])
        _, _, tab = zo.read_tables(cont, 0)
        w = hd["sub_end_bytes"]
        for off, val in ((0, 0x58), (6, 2), (8, 1), (17, 0x40), (27, 3), (64, 7), (sec + used, 13), (tab + w * 31 + w - 1, 0xFF)):
            bad = cont.copy(); bad[off] = val
            zc.decompress(p, torch.from_numpy(bad).to(DEV), bad.size, d_back, d_ws)
            assert zc.device_status(p, d_ws) == zc.E_CORRUPT, off
        # a plan that does not match
        p2 = zc.plan(zc.FMT_BF16, n + 1, 8192)
        d_ws2 = torch.empty(p2.workspace_bytes, dtype=torch.uint8, device=DEV)
        d_back2 = torch.zeros(p2.input_bytes, dtype=torch.uint8, device=DEV)
        zc.decompress(p2, d_c, cont.size, d_back2, d_ws2)
        assert zc.device_status(p2, d_ws2) == zc.E_CORRUPT


@pytest.mark.parametrize("fmt", FORMATS)
def test_random_access_decodes_chunk_ranges_like_the_oracle(fmt):
    """Sec. 3.1: chunks decode independently.  Ranges of chunks (first, last, single, all, empty) against the
    oracle's chunk-by-chunk decoder; bytes outside the range stay untouched."""
    chunk_bytes = 2048
    G = zo.group(fmt)
    cs = chunk_bytes // 2
    n = (37 * cs + cs // 2 + 5) * G
    if fmt == zc.FMT_FP4_E2M1:
        n -= n % 2
    data = _weights(fmt, n, 321 + fmt)
    for policy in (zc.POLICY_AUTO, zc.POLICY_HUFF_ALL):
        p, cb, hist, cont = _gpu_round_trip(fmt, data, n, chunk_bytes, policy)
        d_c = torch.from_numpy(cont).to(DEV)
        ws = torch.empty(p.workspace_bytes, dtype=torch.uint8, device=DEV)
        for first, count in [(0, 1), (0, p.n_chunks), (p.n_chunks - 1, 1), (5, 1), (7, 13), (30, p.n_chunks - 30), (9, 0)]:
            want = np.concatenate([zo.decompress_chunk(cont, c, chunk_bytes) for c in range(first, first + count)] + [np.zeros(0, np.uint8)])
            d_out = torch.full((want.size + 64,), 0xEE, dtype=torch.uint8, device=DEV)
            zc.decompress_chunks(p, d_c, cont.size, first, count, d_out[32:], ws)
            assert zc.device_status(p, ws) == zc.OK
            got = d_out.cpu().numpy()
            assert np.array_equal(got[32: 32 + want.size], want), (first, count)
            assert (got[:32] == 0xEE).all() and (got[32 + want.size:] == 0xEE).all()
        with pytest.raises(zc.ZcError) as e:
            zc.decompress_chunks(p, d_c, cont.size, p.n_chunks - 1, 2, d_out, ws)
        assert e.value.status == zc.E_INVALID_ARG


def test_argument_checks():
    p = zc.plan(zc.FMT_BF16, 1000, 1024)
    d = torch.zeros(4096, dtype=torch.uint8, device=DEV)
    ws = torch.zeros(p.workspace_bytes, dtype=torch.uint8, device=DEV)
    cb = zc.build_codebook(p, np.ones((2, 256)), zc.POLICY_AUTO)
    with pytest.raises(zc.ZcError) as e:
        zc.compress(p, cb, d, d[:100], ws)
    assert e.value.status == zc.E_BUFFER_TOO_SMALL
    big = torch.zeros(p.max_compressed_bytes + 16, dtype=torch.uint8, device=DEV)
    with pytest.raises(zc.ZcError) as e:
        zc.compress(p, cb, d[1:], big, ws)                            # misaligned input
    assert e.value.status == zc.E_INVALID_ARG


def test_small_versions_of_the_five_configurations():
    for name, fmt, t, n in wl.small_cases(DEV):
        data = t.cpu().numpy()
        for chunk_bytes in (8192, 65536):
            for policy in (zc.POLICY_AUTO, zc.POLICY_HUFF_ALL):
                _gpu_round_trip(fmt, data, n, chunk_bytes, policy)


def test_config1_exact():
    """Config 1 in full: 1024x1024 FP8 E4M3, N(0, 0.02), per-tensor scale, seed 0, 64 KiB chunks."""
    t, n = wl.config1_tensor(DEV)
    data = t.cpu().numpy()
    p, cb, hist, cont = _gpu_round_trip(zc.FMT_FP8_E4M3, data, n, 65536, zc.POLICY_AUTO)
    assert p.n_chunks == 16
    assert cb.modes == [zc.MODE_HUFF, zc.MODE_RAW]
    st = zc.stats(p, cb, hist, cont[:128])
    assert 0.78 < st.ratio_container < 0.86                       # the paper's abstract quotes "up to 83%" for FP8


def test_large_tensor_sampled_chunks():
    """A tensor of bench size class (64 Mi BF16 elements, 16 KiB chunks): the oracle checks sampled chunks
    one by one, properties cover the rest."""
    n = 1 << 26
    g = torch.Generator(device=DEV); g.manual_seed(123)
    x = (torch.randn(n, generator=g, device=DEV) * 0.02).to(torch.bfloat16)
    d_in = x.view(torch.uint8)
    chunk_bytes = 16384
    p = zc.plan(zc.FMT_BF16, n, chunk_bytes)
    hist = zc.histogram(p, d_in).cpu().numpy().astype(np.uint64)
    assert int(hist[0].sum()) == n and int(hist[1].sum()) == n
    cb = zc.build_codebook(p, hist, zc.POLICY_AUTO)
    d_out = torch.empty(p.max_compressed_bytes, dtype=torch.uint8, device=DEV)
    d_ws = torch.empty(p.workspace_bytes, dtype=torch.uint8, device=DEV)
    nbytes = zc.compress(p, cb, d_in, d_out, d_ws)
    cont = d_out[:nbytes].cpu().numpy()
    assert zc.validate_container(p, cont) == zc.OK
    hd = zo.parse_header(cont)
    mode0, lens0, _ = cb.get(0)
    assert hd["streams"][0]["payload_bits"] == int((hist[0].astype(np.int64) * lens0).sum())
    data = d_in.cpu().numpy()
    rng = np.random.default_rng(0)
    for c in [0, 1, p.n_chunks - 1] + [int(v) for v in rng.integers(0, p.n_chunks, 12)]:
        got = zo.decompress_chunk(cont, c, chunk_bytes)
        assert np.array_equal(got, data[c * chunk_bytes:(c + 1) * chunk_bytes])
    d_back = torch.empty(p.input_bytes, dtype=torch.uint8, device=DEV)
    zc.decompress(p, d_out, nbytes, d_back, d_ws)
    assert zc.device_status(p, d_ws) == zc.OK
    assert torch.equal(d_back, d_in)


@pytest.mark.parametrize("fmt", [zc.FMT_BF16, zc.FMT_FP8_E4M3])
@pytest.mark.parametrize("policy", [zc.POLICY_AUTO, zc.POLICY_HUFF_ALL])
@pytest.mark.parametrize("chunk_kib,extra", [(1, 0), (2, 1), (4, 0), (5, -1), (6, 17), (7, 1), (9, 0), (12, -16), (13, 1), (28, -1), (32, 16),
                                             (33, 0), (61, 1), (64, 0)])
def test_encoder_at_every_kind_of_chunk_size(fmt, policy, chunk_kib, extra):
    """Chunks that fill a worker's lanes exactly, several workers, part of one, and more symbols than the workers of a block
    hold at once; 11 chunks and a tail that ends just before or behind a chunk's, a subchunk's or a word's edge."""
    n = (11 * 512 * chunk_kib + extra) * zo.group(fmt)
    _gpu_round_trip(fmt, _weights(fmt, n, chunk_kib + fmt), n, 1024 * chunk_kib, policy)


@pytest.mark.parametrize("fmt,policy", [(zc.FMT_BF16, zc.POLICY_AUTO), (zc.FMT_BF16, zc.POLICY_HUFF_ALL), (zc.FMT_FP8_E4M3, zc.POLICY_AUTO)])
@pytest.mark.parametrize("chunk_kib", [4, 31, 32, 64])
def test_decoder_at_the_chunk_counts_where_its_kernel_changes(fmt, policy, chunk_kib):
    """Ranges of one chunk up to a few per SM and beyond, below and from the subchunk length on that is cut into stretches."""
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    counts = sorted({1, 2, 18, 19, 37, 74, 75, sm, sm + 1, 8 * sm, 8 * sm + 1} if chunk_kib == 4 else {1, 2, 18, 19, 37, 74, 75, sm, sm + 1})
    cs = 512 * chunk_kib
    n = ((counts[-1] + 1) * cs - cs // 3 - 5) * zo.group(fmt)        # a ragged chunk follows the longest range
    data = _weights(fmt, n, chunk_kib)
    cont = zo.compress(fmt, data, n, 1024 * chunk_kib, zo.build_codebook(zo.histogram(fmt, data, n), policy))
    p = zc.plan(fmt, n, 1024 * chunk_kib)
    d_comp, d_ws = torch.from_numpy(cont).to(DEV), torch.zeros(p.workspace_bytes, dtype=torch.uint8, device=DEV)
    want = torch.from_numpy(data).to(DEV)
    for count in counts:
        for first in (0, p.n_chunks - count):
            lo, hi = first * p.chunk_bytes, min((first + count) * p.chunk_bytes, p.input_bytes)
            back = torch.full((hi - lo + 64,), 0xEE, dtype=torch.uint8, device=DEV)
            zc.decompress_chunks(p, d_comp, cont.size, first, count, back, d_ws)
            assert zc.device_status(p, d_ws) == zc.OK
            assert torch.equal(back[: hi - lo], want[lo:hi]) and bool((back[hi - lo:] == 0xEE).all())


@pytest.mark.parametrize("counts", [[255 - k for k in range(256)], [2 ** max(0, 40 - k) for k in range(256)], [1] * 256,
                                    [2 ** max(0, 11 - k) for k in range(256)], [10 ** 6] + [1] * 255, [7] + [0] * 255, [7, 7] + [0] * 254])
def test_decode_tables_of_every_shape_of_code(counts):
    """Codes of all lengths from 1 to 12, of one length only, and of one or two symbols: windows that start with a code of up
    to 9 bits, of 10 to 12 bits, and of no symbol."""
    rng = np.random.default_rng(5)
    c = np.array(counts, dtype=np.float64)
    n = 40 * 2048
    lo = rng.choice(256, n, p=c / c.sum()).astype(np.uint32)         # the exponent byte of BF16 carries the counts
    rest = rng.integers(0, 256, n, dtype=np.uint32)
    v = ((rest & 0x80) << 8) | (lo << 7) | (rest & 0x7F)
    data = v.astype(np.uint16).view(np.uint8)
    for chunk_bytes in (4096, 65536):
        _gpu_round_trip(zc.FMT_BF16, data, n, chunk_bytes, zc.POLICY_HUFF_ALL)


@pytest.mark.parametrize("fmt", [zc.FMT_BF16, zc.FMT_FP8_E4M3])
@pytest.mark.parametrize("chunk_kib", [40, 48, 56, 64])
def test_ragged_large_chunk_behind_complete_ones_of_the_same_warp(fmt, chunk_kib):
    """Both streams coded, pieces staged slice by slice, more chunks than warps: the last chunk, long enough for slices and
    with lanes that have no symbols, is decoded by a warp that has decoded a complete one before, in the single and in the
    batched form."""
    cs = chunk_kib * 512
    n = (1500 * cs + cs * 3 // 4 + 5) * zo.group(fmt)
    g = torch.Generator(device=DEV); g.manual_seed(chunk_kib)
    x = torch.randn(n, generator=g, device=DEV)
    d_in = ((x * 0.02).to(torch.bfloat16) if fmt == zc.FMT_BF16 else (x * 80).clamp(-448, 448).to(torch.float8_e4m3fn)).view(torch.uint8)
    p = zc.plan(fmt, n, chunk_kib * 1024)
    cb = zc.build_codebook(p, zc.histogram(p, d_in).cpu().numpy(), zc.POLICY_HUFF_ALL)
    d_out = torch.empty(p.max_compressed_bytes, dtype=torch.uint8, device=DEV)
    ws = torch.empty(p.workspace_bytes, dtype=torch.uint8, device=DEV)
    nbytes = zc.compress(p, cb, d_in, d_out, ws)
    assert zc.validate_container(p, d_out[:nbytes].cpu().numpy()) == zc.OK
    back = torch.zeros(p.input_bytes, dtype=torch.uint8, device=DEV)
    zc.decompress(p, d_out, nbytes, back, ws)
    assert zc.device_status(p, ws) == zc.OK and torch.equal(back, d_in)
    back.zero_()
    zc.decompress_batch(zc.DecompressBatch([p], [d_out], [nbytes], [back]), ws)
    assert zc.batch_status(ws) == (zc.OK, None) and torch.equal(back, d_in)


@pytest.mark.parametrize("fmt", FORMATS)
@pytest.mark.parametrize("chunk_kib,chunks", [(5, 296), (5, 297), (6, 300), (7, 620), (13, 30), (19, 40), (29, 25), (30, 300), (31, 20)])
@pytest.mark.parametrize("coded", [0, 1])
def test_one_coded_stream_at_chunk_sizes_with_kernels_of_their_own(fmt, chunk_kib, chunks, coded):
    """Chunks of 5 to 7 KiB that one warp codes (launches of more than two chunks per SM) and chunks of odd sizes whose teams
    need the larger block, either stream coded and the other one raw, with and without a base tensor, a ragged end."""
    cs = chunk_kib * 512
    n = (chunks * cs - cs // 3 - 5) * zo.group(fmt)
    data, base = _weights(fmt, n, chunk_kib), _weights(fmt, n, 100 + chunk_kib)
    skewed, even = np.full((2, 256), 0, np.uint64), np.full(256, 1000, np.uint64)
    skewed[0] = skewed[1] = (1 << 20) // (1 + np.arange(256)) ** 2 + 1
    hist = np.stack([skewed[0], even] if coded == 0 else [even, skewed[1]])  # the AUTO rule: one stream coded, one raw
    p = zc.plan(fmt, n, chunk_kib * 1024)
    cb, ocb = zc.build_codebook(p, hist, zc.POLICY_STATIC), zo.build_codebook(hist, zo.POLICY_STATIC)
    assert cb.modes == [1 - coded, coded]
    d_base = torch.from_numpy(base).to(DEV)
    for d_in, d_b in ((data, None), (data ^ base, d_base)):
        d_out = torch.full((p.max_compressed_bytes + 64,), 0xA5, dtype=torch.uint8, device=DEV)
        ws = torch.empty(p.workspace_bytes, dtype=torch.uint8, device=DEV)
        nbytes = zc.compress(p, cb, torch.from_numpy(d_in).to(DEV), d_out[: p.max_compressed_bytes], ws, d_base=d_b)
        want = zo.compress(fmt, data, n, chunk_kib * 1024, ocb)
        got = d_out.cpu().numpy()
        assert nbytes == want.size and np.array_equal(got[:nbytes], want) and (got[p.max_compressed_bytes:] == 0xA5).all()
        back = torch.full((p.input_bytes + 32,), 0xEE, dtype=torch.uint8, device=DEV)
        zc.decompress(p, d_out, nbytes, back, ws)
        assert zc.device_status(p, ws) == zc.OK
        back = back.cpu().numpy()
        assert np.array_equal(back[: p.input_bytes], data[: p.input_bytes]) and (back[p.input_bytes:] == 0xEE).all()
