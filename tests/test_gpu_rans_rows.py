"""rANS decoder: table rows in shared memory, their overflow to global memory,
several chunks per block and the batch edges of the helper warps. The encoder
(checked against the oracle elsewhere) writes the payload; the decoder must
return the values, on chunk lengths around the eight-round batches and on
index sets with more distinct tables than fit in shared memory."""
import numpy as np
import pytest

from tests._lib import ensure_built

pytestmark = pytest.mark.gpu
ensure_built()


@pytest.fixture(scope="module")
def codec():
    import paper_2405_12631_gb300 as pw
    c = pw.Codec(0, "fp32")
    yield c
    c.close()


def _round_trip(codec, counts, lanes, tables, seed):
    """tables: number of distinct scale bins (of 128) the indices spread over;
    every one of the 16 phases is used."""
    rng = np.random.default_rng(seed)
    n = int(np.sum(counts))
    j = rng.integers(64 - tables // 2, 64 - tables // 2 + tables, n)
    t = rng.integers(-400, 400, n)
    idx = (((t + 2**23) << 7) | j).astype(np.uint32)
    ctr = (t + 8) >> 4
    scale = 0.125 * 2.0 ** (j / 8.0)
    r = np.rint(rng.laplace(0.0, np.minimum(scale, 200.0)))
    vals = (ctr + r).astype(np.int32)
    if n:
        vals[rng.integers(0, n, max(1, n // 500))] += rng.choice([-70000, 63, -63, 2**30])
    pay, off, nb = codec.rans_encode(counts, lanes, idx, vals)
    assert np.array_equal(codec.rans_decode(pay, off, nb, counts, lanes, idx), vals)
    return pay, off, nb, idx


@pytest.mark.parametrize("lanes", [1, 2, 31, 32])
def test_batch_edges(codec, lanes):
    rounds = [1, 2, 7, 8, 9, 15, 16, 17, 24, 25]
    counts = [lanes * r for r in rounds] + [lanes * r - lanes // 2 for r in rounds]
    counts = [c for c in counts if c > 0]
    _round_trip(codec, counts, [lanes] * len(counts), 24, lanes)


@pytest.mark.parametrize("tables", [1, 40, 60, 128])
def test_row_capacity(codec, tables):
    """1 .. 2048 distinct tables in one chunk (about 770 rows fit)."""
    _round_trip(codec, [16384], [32], tables, tables)


@pytest.mark.parametrize("nchunks", [152, 153, 305, 700, 1300])
def test_chunks_per_block(codec, nchunks):
    rng = np.random.default_rng(nchunks)
    counts = rng.integers(0, 300, nchunks)
    lanes = rng.integers(1, 33, nchunks)
    _round_trip(codec, counts, lanes, 100, nchunks)


def test_corrupt_words(codec):
    """A missing last word is reported, as before."""
    import paper_2405_12631_gb300 as pw
    pay, off, nb, idx = _round_trip(codec, [5000], [32], 16, 9)
    with pytest.raises(pw.PwError) as e:
        codec.rans_decode(pay[:-2], off, nb - 2, [5000], [32], idx)
    assert e.value.code == pw.PW_ECORRUPT
