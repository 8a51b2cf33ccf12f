"""Cell sort of frames with few filled rows, which a launch of its own takes: rows on both sides of
its least size, of its shared counters' (11 520 cells) and of one sector filled, against the oracle."""
import numpy as np
import pytest

import oracle
from helpers import float_tf, npads
from parity import compare_stages
from paper_2106_03636_gb300 import o2tpc

pytestmark = pytest.mark.gpu


def test_few_filled_rows_against_the_oracle():
    rng = np.random.default_rng(5)
    rows = np.arange(0, 152, 4)  # none adjacent: no links
    counts = np.full(len(rows), 30000)
    ny = -(-64 * npads(int(rows[1])) // 320)
    counts[:6] = 90000, 4 * 2048, 4 * 2048 + 4 * ny, 100, 4 * 11520, 4 * 11520 + 4 * ny
    counts[-1] = 200000
    row = np.repeat(rows, counts)
    n = len(row)
    assert n // (152 * 4) > 4 * 512  # or no row is taken apart
    p = rng.permutation(n)
    z = 250.0 - 0.003125 * 2.58 * np.round(rng.random(n) * 3000000)
    tf = float_tf(np.full(n, 7), row[p], rng.uniform(-9, 9, n), z)
    o = oracle.run(tf)
    cells = (o["row_ny"] * o["row_nz"])[7 * 152 + rows]
    assert cells.max() > 11520 and np.any((cells > 2048) & (cells <= 11520)) and np.any(cells <= 2048)
    with o2tpc.Tracker(flags=o2tpc.O2TPC_FLAG_KEEP_STAGES) as t:
        ticket = t.submit(tf)
        res = t.poll(ticket, keep=True)
        assert res["status"] == 0
        compare_stages(t, ticket, o)
        t.release(ticket, res)
