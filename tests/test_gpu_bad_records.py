"""Bytes that are no cluster records: refused after the batch has run to its end over them, on
the regular and the captured path and by the static sort, and good input is served afterwards."""
import numpy as np
import pytest

from paper_2106_03636_gb300 import o2tpc, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _noise(n):
    """Records of uniform words: nine in ten go to row 0, their times all over 32 bits."""
    tf = synth.single_sector(fmt=synth.FMT_FIXED)
    rec = np.random.default_rng(n).integers(0, 256, (n, 12), dtype=np.uint8)
    tf.n, tf.packed, tf.coll_time = n, rec, None
    tf.sector = tf.row = None
    return tf


@pytest.mark.parametrize("captured", [False, True])
def test_noise_is_refused(captured):
    n = 200000
    bad, good = _noise(n), synth.single_sector(fmt=synth.FMT_FIXED)
    with o2tpc.Tracker(graph_max_clusters=n if captured else 0, graph_max_tfs=1) as t:
        assert t.track(bad)["status"] == o2tpc.O2TPC_EINVAL
        r = t.track(good)
        assert r["status"] == 0 and r["n_tracks"] > 10


def test_static_sort_refuses_noise():
    n = 200000
    dev = torch.device("cuda", 0)
    rec = torch.from_numpy(_noise(n).packed).to(dev)
    t = o2tpc.o2tpc_tf()
    t.n, t.format, t.location, t.packed = n, o2tpc.O2TPC_FMT_FIXED, o2tpc.O2TPC_LOC_DEVICE, rec.data_ptr()
    rows = 36 * 152
    cap = n // 4 + 46 * rows + 2
    grid = torch.empty((rows, 8), dtype=torch.int32, device=dev)
    cs, yz = torch.empty(cap, dtype=torch.int32, device=dev), torch.empty((n, 2), dtype=torch.int32, device=dev)
    orig = torch.empty(n, dtype=torch.int32, device=dev)
    rc = o2tpc.o2tpc_sort_tf_static(t, 2.58, orig.data_ptr(), yz.data_ptr(), grid.data_ptr(), cs.data_ptr(), cap,
                                    torch.cuda.current_stream().cuda_stream)
    assert rc == o2tpc.O2TPC_EINVAL
