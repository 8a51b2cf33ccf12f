"""Rows whose sorted and drift orders lie further apart than a view's 16-bit index distances
reach, and rows on both sides of 65 535 hits, where the bin starts become 32-bit: the links
against the oracle bit for bit, with and without links across a missing row."""
import numpy as np
import pytest

import oracle
from helpers import float_tf
from parity import compare_stages
from paper_2106_03636_gb300 import o2tpc

pytestmark = pytest.mark.gpu

ZUNIT = 0.003125 * 2.58  # cm per drift unit
ROW = 20


def _frame(kind, n):
    """Straight tracks over the rows ROW - 6 to ROW + 6 of the first sector; row ROW is filled up
    to n hits, spread in drift (a late one among them, so that one cell row holds the others), all
    at one drift time, or spread so far that the views are searched."""
    rng = np.random.default_rng(n)
    span = {"late": 320000, "one_time": 0, "long": 3000000}[kind]
    ntrk = 300 if kind == "one_time" else 3000
    zu = lambda k: 1000 + np.round(rng.random(k) * span)
    row, y, z = [], [], []
    ty, tz = rng.uniform(-10, 10, ntrk), zu(ntrk)
    for r in range(ROW - 6, ROW + 7):
        k = ntrk
        row.append(np.full(k, r)), y.append(ty + rng.normal(0, 0.05, k)), z.append(tz + np.round(rng.normal(0, 8, k)))
    k = n - ntrk - (kind == "late")
    row.append(np.full(k, ROW)), y.append(rng.uniform(-10, 10, k)), z.append(zu(k))
    if kind == "late":
        row.append([ROW]), y.append([0.0]), z.append([1.0e9])
    row, y, z = np.concatenate(row), np.concatenate(y), np.concatenate(z)
    p = rng.permutation(len(row))
    tf = float_tf(np.zeros(len(p)), row[p], y[p], 250.0 - z[p] * ZUNIT)
    return tf


def _least_distance(o):
    """Largest over the hits of row ROW of the least distance between a hit's sorted index and a
    place of its drift bin (bins of at least 62 units, at most one per hit)."""
    a, n = int(o["row_start"][ROW]), int(o["row_count"][ROW])
    z = o["sorted_z"][a:a + n].astype(np.int64)
    rng = np.float32(z.max() - z.min()) + np.float32(1)
    nzb = int(max(1, min(int(rng / np.float32(62)), n)))
    b = np.minimum(((z - z.min()).astype(np.float32) * (np.float32(nzb) / rng)).astype(np.int64), nzb - 1)
    first = np.concatenate([[0], np.cumsum(np.bincount(b, minlength=nzb))])
    h = np.arange(n)
    return int(np.maximum(first[b] - h, h - (first[b + 1] - 1)).max())


@pytest.mark.parametrize("row_step2", [False, True])
@pytest.mark.parametrize("kind,n", [("late", 40000), ("late", 70000), ("one_time", 40000), ("long", 65535),
                                    ("long", 65536)])
def test_links_of_rows_with_many_hits(kind, n, row_step2):
    tf = _frame(kind, n)
    o = oracle.run(tf, row_step2=row_step2)
    assert o["row_count"][ROW] == n
    assert (_least_distance(o) > 32768) == (kind == "late")
    assert np.count_nonzero(o["up_raw"] >= 0) > (200 if kind == "one_time" else 10000)
    flags = o2tpc.O2TPC_FLAG_KEEP_STAGES | (o2tpc.O2TPC_FLAG_ROW_STEP2 if row_step2 else 0)
    with o2tpc.Tracker(flags=flags) as t:
        ticket = t.submit(tf)
        res = t.poll(ticket, keep=True)
        assert res["status"] == 0
        compare_stages(t, ticket, o)
        t.release(ticket, res)
