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


# 128-row tiles per head: one; two; three; five - with as many heads as make (on 148 SMs) no full round or one or several, a
# last round of whole units, of units cut in two, of single tiles, of both
@pytest.mark.parametrize("rate", [0, 5])
@pytest.mark.parametrize("B,H,N", [(1, 3, 100), (1, 5, 129), (2, 35, 300), (1, 100, 300), (2, 40, 620), (1, 74, 620), (2, 45, 620), (1, 148, 256),
                                   (1, 160, 257)])
def test_every_tile_of_every_head_is_worked_on(B, H, N, rate):
    """The tensor path next to the fp32 check path: 2.5e-3 and 1.7e-3 off the exact result (bf16 operands; bf16 output), so 5e-3 apart."""
    import torch
    from paper_2509_24899_b200 import HybridAttention, binding
    wl, dev = _inputs(B, H, N, 64, rate, 71)
    args = [dev[n] for n in ("q", "k", "v", "wq", "wk")]
    out = []
    for path in (binding.AS_PATH_TENSOR, binding.AS_PATH_SIMT):
        op = HybridAttention.from_workload(wl, kernel_path=path)
        out.append(op.forward(*args, out=torch.full_like(args[0], float("nan"))).double())
        assert op.last_status() == 0
    err = (out[0] - out[1]).norm(dim=-1) / out[1].norm(dim=-1)
    assert bool(torch.isfinite(out[0]).all())
    assert float((out[0] - out[1]).norm() / out[1].norm()) <= 5e-3
    assert float(err.max()) <= 5e-2                          # no row left out or taken twice


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
