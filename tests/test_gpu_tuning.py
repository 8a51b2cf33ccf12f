"""o2tpc_get_tuning names the cell sort's shape that the last batch ran with."""
import pytest

from paper_2106_03636_gb300 import o2tpc, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("captured", [False, True])
def test_sort_shape_of_the_last_batch(captured):
    small, large = synth.single_sector(seed=5, ntracks=6), synth.full_tpc_1ms(seed=5, n_coll=20, with_truth=False)
    assert small.n // 5472 < 1000 <= large.n // 5472 < 8000
    room = dict(graph_max_clusters=large.n, graph_max_tfs=1) if captured else {}
    with o2tpc.Tracker(**room) as t:
        assert t.tuning()["sort_threads_per_row"] == 256
        t.track(small)
        assert t.tuning()["sort_threads_per_row"] == (256 if captured else 128)  # captured: by the room
        t.track(large)
        assert t.tuning()["sort_threads_per_row"] == 256
    with o2tpc.Tracker(sort_threads_per_row=512, **room) as t:
        t.track(small)
        assert t.tuning()["sort_threads_per_row"] == 512
