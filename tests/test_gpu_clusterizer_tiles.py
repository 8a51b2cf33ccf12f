"""Clusterizer at the edges of its tiles and halos: full (row, bin)s of 256 pads, so that a
neighbour lies as far away as it can, and sizes around a tile, on aligned and odd addresses."""
import numpy as np
import pytest

import oracle
from paper_2106_03636_gb300 import o2tpc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 3071, 3072, 3073, 3344, 8192])
def test_full_bins_across_tiles(n, shift):
    rng = np.random.default_rng(n)
    i = np.arange(n)

    class D:
        pass

    d = D()
    cut = 2 * n // 3  # the rest on another row
    d.sector = np.full(n, 35, np.uint8)
    d.row = np.where(i < cut, 4, 5).astype(np.uint8)
    d.time = (np.where(i < cut, i, i - cut) // 256 + 2).astype(np.uint32)
    d.pad = (np.where(i < cut, i, i - cut) % 256).astype(np.uint8)
    d.adc = rng.integers(2, 7, n).astype(np.uint16)
    dev = {}
    for k in ("sector", "row", "pad", "time", "adc"):
        whole = np.concatenate([np.zeros(shift, getattr(d, k).dtype), getattr(d, k)])
        dev[k] = torch.from_numpy(whole).cuda()[shift:]
    rc, rec, m = o2tpc.clusterize(dev)
    assert rc == o2tpc.O2TPC_OK
    want = oracle.clusterize(d)
    assert m == len(want) and np.array_equal(rec.cpu().numpy(), want)
