"""rANS decoder on hand-made chunks, as the oracle's coder writes them from
explicit coding operations or as bare states and words: escape prefixes up to
the limit give their values and longer ones are reported; lanes without a
symbol read no words; states below 2^16 decode as the format defines; a
corrupt chunk stops early."""
import numpy as np
import pytest

import synthetic as S
from oracle import codec as K
from oracle import entropy as E
from oracle import rans as R
from tests._lib import ensure_built
from tests.test_zz_no_alloc import _noalloc

pytestmark = pytest.mark.gpu
ensure_built()

KMAX = 30                                   # longest escape prefix of the format


@pytest.fixture(scope="module")
def pw():
    import paper_2405_12631_gb300 as m
    return m


@pytest.fixture(scope="module")
def codec(pw):
    c = pw.Codec(0, "fp32")
    yield c
    c.close()


@pytest.fixture(scope="module")
def bank():
    return E.cdf_bank().astype(np.int64)


def _esc_ops(cdf, right, k, low):
    """An escape of k ones, a zero and the k bits of low; and its residual."""
    s = R.ESC_R if right else R.ESC_L
    bits = [1] * k + [0] + [(low >> (k - 1 - i)) & 1 for i in range(k)]
    ops = [(int(cdf[s]), int(cdf[s + 1]) - int(cdf[s]))] + [(b * R.HALF, R.HALF) for b in bits]
    e = (1 << k) + low - 1
    return ops, (e if right else -e) + (R.T + 1 if right else -R.T - 1)


def _chunk(rng, bank, n, nl, escapes):
    """n symbols on nl lanes, `escapes` {symbol: prefix length} among small
    residuals: (payload, packed indices, values)."""
    tid = rng.integers(0, 2048, n)
    tid = (tid & ~127) | np.clip(tid & 127, 0, 80)
    ctr = rng.integers(-30, 30, n)
    ops, vals = [], []
    for p in range(n):
        if p in escapes:
            k = escapes[p]
            low = int(rng.integers(0, 1 << k)) if k < KMAX else int(rng.integers(0, (1 << k) - 4096))
            o, r = _esc_ops(bank[tid[p]], bool(rng.integers(2)), k, low)
        else:
            r = int(rng.integers(-3, 4))
            o = R.symbol_ops(r, bank[tid[p]])
        ops.append(o)
        vals.append(int(ctr[p]) + r)
    st, words = R.encode_chunk(ops, nl)
    t = 16 * ctr + (tid // 128 - 8)
    idx = (((t + (1 << 23)) << 7) | (tid % 128)).astype(np.uint32)
    return R.pack_chunk(st, words), idx, vals


def _both(pw, codec, buf, n, nl, idx):
    """(status, values) of the regular and the allocation-free decoder."""
    u32 = lambda v: np.asarray([v], dtype=np.uint32)
    a = (buf, u32(0), u32(len(buf)), u32(n), u32(nl), idx)
    try:
        reg = pw.PW_OK, codec.rans_decode(*a)
    except pw.PwError as e:
        reg = e.code, None
    rc, got = _noalloc(pw, *a)
    assert rc == reg[0], (rc, reg[0])
    return rc, got if reg[1] is None else reg[1]


@pytest.mark.parametrize("nl", [1, 5, 32])
@pytest.mark.parametrize("k", [30, 31, 32, 35, 45])
def test_escape_prefix_limit(pw, codec, bank, nl, k):
    """The state's fill when the escape starts decides where its passes of up
    to 16 bits end: 48 chunks with other symbols before it."""
    rng = np.random.default_rng(100 * nl + k)
    for _ in range(48):
        n = int(rng.integers(1, 3 * nl + 2))
        buf, idx, vals = _chunk(rng, bank, n, nl, {int(rng.integers(0, n)): k})
        rc, got = _both(pw, codec, buf, n, nl, idx)
        if k <= KMAX:
            assert rc == pw.PW_OK and got.tolist() == vals
        else:
            assert rc == pw.PW_ECORRUPT, "an over-long prefix was accepted"


@pytest.mark.parametrize("nl", [1, 3, 32])
def test_every_prefix_length(pw, codec, bank, nl):
    """Prefixes of 0 to 30 at every state, on neighbouring lanes and alone."""
    rng = np.random.default_rng(nl)
    n = 40 * 31
    esc = {p: int(k) for p, k in zip(rng.permutation(n)[:31 * 16], np.tile(np.arange(31), 16))}
    buf, idx, vals = _chunk(rng, bank, n, nl, esc)
    rc, got = _both(pw, codec, buf, n, nl, idx)
    assert rc == pw.PW_OK and got.tolist() == vals


@pytest.mark.parametrize("k", [30, 31, 33, 40])
def test_escape_prefix_limit_ragged(pw, k, monkeypatch):
    """The last chunk of a stream, on which no other depends, in a ragged
    batch and alone."""
    cfg = S.ModelConfig(levels=4, C=32, ll_mode=0)
    blob = S.pack_blob(cfg, S.random_model(cfg, 1))
    rng = np.random.default_rng(k)
    img = S.gray_sinusoids(16, 32, seed=1)
    encode, tables_of = R.encode_chunk, K.coding_tables
    tables, seen, last = [None], [0], [0]

    def keep_tables(*args):
        ctr, tables[0] = tables_of(*args)
        return ctr, tables[0]

    def escape_in_last(ops, nl):
        seen[0] += 1
        if seen[0] == last[0]:
            p = int(rng.integers(0, len(ops)))
            ops = list(ops)
            ops[p], _ = _esc_ops(tables[0][p], True, k, 5)
        return encode(ops, nl)

    monkeypatch.setattr(K, "coding_tables", keep_tables)
    monkeypatch.setattr(R, "encode_chunk", escape_in_last)
    streams = []
    for _ in range(13):   # the first one as it is
        seen[0] = 0
        streams.append(K.encode_image(blob, img, q=8.0, integer=True))
        last[0] = seen[0]
    codec = pw.Codec(0, "int8")
    model = codec.load_model(blob)
    other = codec.encode_image(model, S.gray_sinusoids(33, 20, seed=2), q=8.0)
    codec.decode_ragged(model, [other, streams[0]])
    for bs in streams[1:]:
        for call in (lambda: codec.decode_ragged(model, [other, bs]),
                     lambda: codec.decode_symbols(model, bs)):
            if k <= KMAX:
                call()
            else:
                with pytest.raises(pw.PwError) as e:
                    call()
                assert e.value.code == pw.PW_ECORRUPT
    model.close()
    codec.close()


def _row(bank, tid):
    """Table tid's packed index with centre 0 and its entries."""
    t = tid // 128 - 8
    return np.uint32(((t + (1 << 23)) << 7) | (tid % 128)), bank[tid]


def test_lane_without_symbols_keeps_its_state(pw, codec, bank):
    """One symbol on two lanes: the second lane's state has to be 2^16 as it
    stands. A state of 1 that a spare zero word would lift to 2^16 is corrupt."""
    pk, cdf = _row(bank, 8 * 128 + 20)
    for r in (0, 1, -2, 7):
        st, words = R.encode_chunk([R.symbol_ops(r, cdf)], 2)
        idx = np.asarray([pk])
        rc, got = _both(pw, codec, R.pack_chunk(st, words), 1, 2, idx)
        assert rc == pw.PW_OK and got.tolist() == [r]
        rc, _ = _both(pw, codec, R.pack_chunk([st[0], 1], words + [0]), 1, 2, idx)
        assert rc == pw.PW_ECORRUPT


@pytest.mark.parametrize("n", [1, 3, 8, 9, 30])
def test_padded_rounds_read_no_words(pw, codec, bank, n):
    """One lane whose state is 1 after its last symbol, and a spare zero word
    (the rounds that fill up the last group of eight must not take it)."""
    pk, cdf = _row(bank, 8 * 128 + 20)
    s = R.T + 1                              # residual 0
    c = int(cdf[s])
    idx = np.full(n, pk)
    # state c -> 0 -> the next word: c again (a symbol a word) or, last, 1
    words = [c] * (n - 1)
    rc, _ = _both(pw, codec, R.pack_chunk([c], words + [1, 0]), n, 1, idx)
    assert rc == pw.PW_ECORRUPT
    rc, _ = _both(pw, codec, R.pack_chunk([c], words + [1]), n, 1, idx)
    assert rc == pw.PW_ECORRUPT
    # the same symbols from a state that ends at 2^16 (c + 1 -> 1 -> 1 0000h):
    # low states of lanes with symbols are the coder's business, and accepted
    words = [c] * (n - 2) + [c + 1] if n > 1 else []
    st = [c] if n > 1 else [c + 1]
    out, used, xf = R.decode_chunk(st, words + [0], n, 1, lambda p: cdf)
    assert out == [0] * n and used == n and xf == [R.L]
    rc, got = _both(pw, codec, R.pack_chunk(st, words + [0]), n, 1, idx)
    assert rc == pw.PW_OK and got.tolist() == [0] * n


def test_low_states_between_escapes(pw, codec, bank):
    """An escape read from states below 2^16, a word for every bit: the words
    4000h give ones until a zero word ends the prefix."""
    pk, cdf = _row(bank, 8 * 128 + 20)
    c = int(cdf[R.ESC_R])
    idx = np.asarray([pk])
    for k in (1, 5, 6, 17, 30):
        # c -> 0 -> 4000h (k times a one) -> 0 -> zero bit, then k bits of 0; the
        # last word is 2^16's low half after 1 has been lifted: 4001h -> 1 on a one
        words = [0x4000] * k + [0] + [0] * k
        out, used, xf = R.decode_chunk([c], words + [0], 1, 1, lambda p: cdf)
        e = (1 << k) - 1
        assert out == [e + R.T + 1] and used == len(words) + 1
        rc, got = _both(pw, codec, R.pack_chunk([c], words + [0]), 1, 1, idx)
        # the end state is 0, not 2^16
        assert xf == [0] and rc == pw.PW_ECORRUPT
        words[-1] = 1
        words.append(0)
        out, used, xf = R.decode_chunk([c], words, 1, 1, lambda p: cdf)
        assert out == [e + R.T + 1] and used == len(words) and xf == [R.L]
        rc, got = _both(pw, codec, R.pack_chunk([c], words), 1, 1, idx)
        assert rc == pw.PW_OK and got.tolist() == [e + R.T + 1]


@pytest.mark.parametrize("nl", [1, 8, 32])
def test_corrupt_chunk_stops_early(pw, codec, bank, nl):
    """Words that run out, or an escape that cannot be, end the chunk: what
    lies far behind is not decoded (the output keeps its fill value)."""
    rng = np.random.default_rng(nl)
    n = 160 * nl
    buf, idx, vals = _chunk(rng, bank, n, nl, {n // 2: 3})
    rc, got = _both(pw, codec, buf, n, nl, idx)
    assert rc == pw.PW_OK and got.tolist() == vals
    cut = 4 * nl + 2 * ((len(buf) - 4 * nl) // 8)
    rc, got = _both(pw, codec, buf[:cut], n, nl, idx)
    assert rc == pw.PW_ECORRUPT and np.all(got[n * 3 // 4:] == -7)
    buf, idx, vals = _chunk(rng, bank, n, nl, {n // 4: 40})
    rc, got = _both(pw, codec, buf, n, nl, idx)
    assert rc == pw.PW_ECORRUPT and np.all(got[n * 3 // 4:] == -7)
    assert got[:n // 4 - 32 * nl].tolist() == vals[:n // 4 - 32 * nl]
