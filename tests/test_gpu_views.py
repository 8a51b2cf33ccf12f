"""Searches in the drift-ordered views at the edges of their rule: rows so dense that the
cells are searched, sparse rows with few wide bins, rows in one bin, single hits."""
import numpy as np
import pytest

import oracle
from parity import compare_stages
from paper_2106_03636_gb300 import o2tpc, synth

pytestmark = pytest.mark.gpu


def _frame(kind):
    if kind == "dense":  # inner rows past both density limits, outer rows below them
        return synth.single_sector(seed=3, ntracks=5000)
    if kind == "lumps":  # two collisions 20 ms apart: bins tens of cm wide
        return synth.generate(seed=4, t0=[0.0, 20000.0], ntracks=[900, 900], zvtx_sigma=5.0)
    if kind == "sparse":  # a few hits a row
        return synth.single_sector(seed=5, ntracks=6)
    tf = synth.single_sector(seed=6, ntracks=300)  # every hit at one drift time: one bin, equal metrics
    tf.z[:] = 100.0
    return tf


@pytest.mark.parametrize("kind", ["dense", "lumps", "sparse", "one_time"])
def test_views_against_the_oracle(kind):
    tf = _frame(kind)
    with o2tpc.Tracker(flags=o2tpc.O2TPC_FLAG_KEEP_STAGES) as t:
        ticket = t.submit(tf)
        res = t.poll(ticket, keep=True)
        assert res["status"] == 0
        o = oracle.run(tf)
        compare_stages(t, ticket, o)  # links and start hits bit for bit
        nh = t.stage(ticket, "tl_nhits")
        assert len(nh) == len(o["tl_nhits"])
        if kind != "one_time":  # degenerate fits amplify FP32 rounding into the hit choice
            assert np.mean(nh == o["tl_nhits"]) >= 0.999
        t.release(ticket, res)


@pytest.mark.parametrize("kind", ["dense", "lumps", "sparse", "one_time"])
def test_row_step2_views_against_the_oracle(kind):
    """Links across a missing row, bit for bit, with a seventh of the rows' hits gone."""
    tf = _frame(kind)
    keep = np.random.default_rng(1).random(tf.n) > 1.0 / 7.0
    tf.sector, tf.row, tf.y, tf.z = (np.ascontiguousarray(a[keep]) for a in (tf.sector, tf.row, tf.y, tf.z))
    tf.n = int(keep.sum())
    with o2tpc.Tracker(flags=o2tpc.O2TPC_FLAG_KEEP_STAGES | o2tpc.O2TPC_FLAG_ROW_STEP2) as t:
        ticket = t.submit(tf)
        res = t.poll(ticket, keep=True)
        assert res["status"] == 0
        compare_stages(t, ticket, oracle.run(tf, row_step2=True))
        t.release(ticket, res)


@pytest.mark.parametrize("kind", ["dense", "lumps", "sparse", "one_time"])
def test_cooperative_search_in_the_cells_agrees(kind):
    """The warp-cooperative search looks through the cells: the same tracks."""
    tf = _frame(kind)
    with o2tpc.Tracker() as a, o2tpc.Tracker(flags=o2tpc.O2TPC_FLAG_COOP_SEARCH) as b:
        x, y = a.track(tf), b.track(tf)
    for k in ("offsets", "cluster_idx", "par", "cov", "chi2"):
        assert np.array_equal(x[k], y[k]), k
