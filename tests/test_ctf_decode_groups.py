"""The host decoder around the ends of chunks and of groups of four chunks, where it changes
between its two loops, against the oracle's decoder; damaged blobs rejected by both."""
import numpy as np
import pytest

import oracle
from helpers import float_tf
from paper_2106_03636_gb300 import o2tpc


def _blob(n):
    rng = np.random.default_rng(n)
    tf = float_tf(rng.integers(0, 36, n), rng.integers(0, 152, n), rng.uniform(-10, 10, n), rng.uniform(5, 240, n))
    tf.z = np.where(tf.sector < 18, tf.z, -tf.z).astype(np.float32)
    return oracle.run(tf, compress=True)["ctf"]


@pytest.mark.parametrize("n", [1, 4095, 4096, 4097, 16383, 16384, 16385, 20480, 150000])
def test_equals_the_oracle_around_chunk_ends(n):
    blob = _blob(n)
    got, want = o2tpc.ctf_decode(blob), oracle.ctf_decode(blob)
    assert len(got["sector"]) == n
    for k, kw in (("sector", "sector"), ("row", "row"), ("y", "y"), ("zeta", "z")):
        assert np.array_equal(got[k], want[kw]), k


@pytest.mark.parametrize("n", [16384, 40000])
def test_damage_anywhere_is_rejected(n):
    """One bit of a chunk state or payload byte: the coder no longer ends in its initial state
    with its bytes used up (a changed symbol run could by chance; not with these seeds)."""
    blob = _blob(n)
    head = 24 + sum(8 + 512 + 4 * (((n if s < 8 else 0) + 4095) // 4096) for s in range(10))
    rng = np.random.default_rng(n + 1)
    for at in rng.integers(head, len(blob), 24):
        bad = blob.copy()
        bad[at] ^= 1 << int(rng.integers(0, 8))
        with pytest.raises(o2tpc.O2TPCError):
            o2tpc.ctf_decode(bad)
    with pytest.raises(o2tpc.O2TPCError):
        o2tpc.ctf_decode(blob[:-1])
