"""Cell sort at the ends of its range of shared counters: rows that ask for the largest
shared memory (from 107 M clusters) and rows of a few hits, against other launch shapes."""
import numpy as np
import pytest

from paper_2106_03636_gb300 import o2tpc, synth

pytestmark = pytest.mark.gpu


def _run(tf, threads):
    with o2tpc.Tracker(sort_threads_per_row=threads) as t:
        return t.poll(t.submit(tf))


@pytest.mark.parametrize("orbits", [0, 64])
def test_cell_sort_shapes(orbits):
    tf = synth.full_tf(seed=5, orbits=orbits) if orbits else synth.single_sector(seed=5, ntracks=6)
    ref = _run(tf, 512)
    assert ref["status"] == 0 and ref["n_tracks"] > 0
    for threads in (0, 128):
        res = _run(tf, threads)
        assert res["status"] == 0
        for k, v in ref.items():
            if isinstance(v, np.ndarray):
                assert np.array_equal(v, res[k], equal_nan=v.dtype.kind == "f"), k
