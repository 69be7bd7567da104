"""How a layer's rows are dealt out to the CTAs, and which rows are gathered: sizes at the edges of each rule."""
import numpy as np
import pytest

from paper_2509_24899_b200 import workloads as W
from _util import oracle_mask, to_cuda_bf16

pytestmark = pytest.mark.gpu


def _inputs(B, H, N, d, rate, seed, F=None, hidden=0):
    import torch
    wl = W.Workload("split", B=B, H=H, d=d, F=F or d, grid=(1, 1, N), block=(1, 1, N), rate=rate, seed=seed,
                    layers=2 if hidden else 1, hidden=hidden)
    dev = {k: to_cuda_bf16(v) for k, v in W.generate(wl, wq_gain=2e-3 if rate else 1.0).items()}
    return wl, dev


@pytest.mark.parametrize("d,F,hidden", [(64, 64, 64), (128, 128, 128), (128, 256, 256)])
@pytest.mark.parametrize("N,rate", [(5, 2), (128, 1000), (128, 2), (131, 3), (400, 7)])
def test_softmax_rows_of_a_two_layer_map_are_gathered_bit_for_bit(N, rate, d, F, hidden):
    """One row of a tile, every second one, the last rows of a ragged tile."""
    import torch
    from paper_2509_24899_b200 import HybridAttention
    wl, dev = _inputs(2, 3, N, d, rate, 72, F, hidden)
    op = HybridAttention.from_workload(wl)
    ks, vs, _, _ = op.key_pass(dev["k"], dev["v"], dev["wq"], dev["wk"], wq2=dev["wq2"], wk2=dev["wk2"])
    at = torch.from_numpy(np.flatnonzero(oracle_mask(wl))).cuda()
    assert op.last_status() == 0
    for got, x in ((ks, dev["k"]), (vs, dev["v"])):
        assert torch.equal(got.view(torch.int16), x[:, :, at].reshape(6, len(at), d).view(torch.int16))
