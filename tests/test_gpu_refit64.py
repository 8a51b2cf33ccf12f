"""The FP64 refit by a warp per track (few tracks) and by a thread per track (many): the same
forced-FP64 results to FP64 rounding, on merged tracks with rotations too."""
import numpy as np
import pytest

from paper_2106_03636_gb300 import o2tpc, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("angular", [0, o2tpc.O2TPC_FLAG_ANGULAR_ERRORS])
def test_warp_and_thread_forms_agree(angular):
    tf = synth.full_tpc_1ms(seed=21, n_coll=1, ntracks=1200, fmt=synth.FMT_FIXED)
    flags = o2tpc.O2TPC_FLAG_FORCE_FP64 | angular
    with o2tpc.Tracker(flags=flags, max_batch=8) as t:
        few = t.track(tf)  # below 2048 queued tracks: a warp each
        many = [t.poll(k) for k in t.submit_many([tf, tf, tf])]  # above: a thread each
    assert 0 < few["n_tracks"] <= 2048 < 3 * few["n_tracks"]
    assert all(m["stats"]["batch_size"] == 3 for m in many)
    assert few["stats"]["n_fp64_fallback"] == few["n_tracks"]
    for m in many:
        assert np.array_equal(few["cluster_idx"], m["cluster_idx"]) and np.array_equal(few["ndf"], m["ndf"])
        assert np.array_equal(few["flags"], m["flags"])
        for k in ("par", "cov", "chi2"):
            # single-precision outputs of double-precision sums: equal but for the last place, where the
            # order of a double sum decides a rounding (ulp 6e-8); cancellation in the covariance's
            # y-zeta terms is relative to the diagonal, so the scale is the column's
            a, b = few[k].astype(np.float64), m[k].astype(np.float64)
            scale = np.abs(a).reshape(len(a), -1) + 1e-3
            d = np.abs(a - b).reshape(len(a), -1) / scale
            assert np.quantile(d, 0.999) <= 2.0 ** -23, k
