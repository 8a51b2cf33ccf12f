"""Clusterizer with the records written over one of the digit arrays."""
import numpy as np
import pytest

import oracle
from paper_2106_03636_gb300 import o2tpc, synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("over", ["time", "adc", "pad"])
def test_records_over_a_digit_array(over):
    d = synth.digits_from(synth.full_tpc_1ms(seed=6, n_coll=1, ntracks=400, fmt=synth.FMT_FIXED), seed=3)
    want = oracle.clusterize(d)
    dev = {}
    for k in ("sector", "row", "pad", "time", "adc"):
        a = np.ascontiguousarray(getattr(d, k))
        room = np.zeros(max(a.nbytes, want.nbytes) + 16, np.uint8)
        room[:a.nbytes] = a.view(np.uint8)
        dev[k] = torch.from_numpy(room).cuda()
    dig = o2tpc.o2tpc_digits(n=len(d.adc), **{k: v.data_ptr() for k, v in dev.items()})
    rc, n = o2tpc.o2tpc_clusterize(dig, dev[over].data_ptr(), len(want), torch.cuda.current_stream().cuda_stream)
    assert rc == o2tpc.O2TPC_OK and n == len(want)
    assert np.array_equal(dev[over].cpu().numpy()[:want.nbytes].reshape(-1, 12), want)
