"""The FP64 refit of a track gives the same bits by a warp (few queued tracks) and by a thread
(many), so that a Time Frame's result is the same alone and in a batch."""
import numpy as np
import pytest

from paper_2106_03636_gb300 import o2tpc, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, o2tpc.O2TPC_FLAG_ANGULAR_ERRORS])
@pytest.mark.parametrize("seed", [21, 22, 23])
def test_same_bits_alone_and_in_a_batch(seed, flags):
    tf = synth.full_tpc_1ms(seed=seed, n_coll=1, ntracks=1200, fmt=synth.FMT_FIXED)
    with o2tpc.Tracker(flags=o2tpc.O2TPC_FLAG_FORCE_FP64 | flags, max_batch=8) as t:
        few = t.track(tf)  # below 2048 queued tracks
        many = [t.poll(k) for k in t.submit_many([tf, tf, tf])]  # above
    assert 1024 < few["n_tracks"] <= 2048 and few["stats"]["n_fp64_fallback"] == few["n_tracks"]
    assert np.count_nonzero(few["flags"] & 2) > 100  # over several sectors: with rotations
    for m in many:
        assert m["stats"]["batch_size"] == 3
        for k, v in few.items():
            if isinstance(v, np.ndarray):
                assert np.array_equal(v, m[k], equal_nan=v.dtype.kind == "f"), k


def test_few_tracks_use_the_whole_gpu():
    """A warp per track spreads over all SMs: one frame's tracks take no longer than three frames'
    by a thread each (0.9 against 1.7 ms; 11.5 ms with a sixteenth of the GPU)."""
    tf = synth.full_tpc_1ms(seed=21, n_coll=1, ntracks=1200, fmt=synth.FMT_FIXED, with_truth=False)
    with o2tpc.Tracker(flags=o2tpc.O2TPC_FLAG_FORCE_FP64, max_batch=8) as t:
        refit = lambda tfs: min(t.poll(k)["stats"]["ms_stage"][8] for k in t.submit_many(tfs))
        few, many = (min(refit(tfs) for _ in range(6)) for tfs in ([tf], [tf, tf, tf]))
    assert few <= many, (few, many)
