"""Kernels that set up while the kernel before them in the stream drains: nothing of theirs may be read or written before that one has
ended, whatever it is - one of the library's or the caller's - and a captured sequence has to keep that."""
import numpy as np
import pytest

from paper_2509_24899_b200 import workloads as W
from _util import to_cuda_bf16

pytestmark = pytest.mark.gpu

LAYERS = {
    "softmax_d128": dict(d=128, rate=1), "softmax_d64": dict(d=64, rate=1), "hybrid_d128": dict(d=128, rate=4), "hybrid_d64": dict(d=64, rate=4),
    "linear_d128": dict(d=128, rate=0), "linear_d64": dict(d=64, rate=0), "two_layers": dict(d=128, rate=4, F=256, hidden=256),
}


def _layer(d, rate, F=None, hidden=0):
    from paper_2509_24899_b200 import HybridAttention
    wl = W.Workload("order", B=1, H=4, d=d, F=F or d, grid=(1, 20, 26), block=(1, 4, 4), rate=rate, seed=81, layers=2 if hidden else 1,
                    hidden=hidden)
    dev = {k: to_cuda_bf16(v) for k, v in W.generate(wl, wq_gain=2e-3 if rate else 1.0).items()}
    return wl, dev, HybridAttention.from_workload(wl), {n: dev[n] for n in ("wq2", "wk2") if n in dev}


def _late(dst, src):
    """Writes src into dst by a kernel on the current stream, a millisecond from now."""
    import torch
    torch.cuda._sleep(2_000_000)
    torch.mul(src, 1.0, out=dst)


@pytest.mark.parametrize("name", sorted(LAYERS))
def test_a_forward_right_behind_the_kernel_that_writes_its_input(name):
    import torch
    wl, dev, op, second = _layer(**LAYERS[name])
    want = op.forward(dev["q"], dev["k"], dev["v"], dev["wq"], dev["wk"], **second).clone()
    for n in ("q", "k", "v"):
        x = dict(dev, **{n: torch.full_like(dev[n], 3.0)})
        torch.cuda.synchronize()
        _late(x[n], dev[n])
        got = op.forward(x["q"], x["k"], x["v"], x["wq"], x["wk"], **second)
        assert op.last_status() == 0
        assert torch.equal(got, want), n


@pytest.mark.parametrize("name", ["hybrid_d128", "hybrid_d64", "linear_d128", "linear_d64", "two_layers"])
def test_a_forward_right_behind_the_kernel_that_writes_its_weights(name):
    """Weights and biases written by an ordinary kernel, and by one of the library's, which lets dependents in long before it writes: a query stage of a
    few CTAs beside which the whole call finds room to set up."""
    import torch
    from paper_2509_24899_b200 import HybridAttention
    wl, dev, op, second = _layer(**LAYERS[name])
    g = torch.Generator(device="cuda").manual_seed(7)
    before = HybridAttention(1, 1, 4096, 64, (1, 1, 4096), (1, 1, 4096), 1)
    x = [torch.randn((1, 1, 4096, 64), device="cuda", generator=g).bfloat16() for _ in range(2)] + \
        [torch.randn((1, 1, 4096, 64), device="cuda", generator=g).bfloat16() * 8]
    written = before.forward(*x).clone()
    H, hid, F = wl.H, wl.hidden or op.F, op.F
    sizes = {"wq": (H, hid, wl.d), "wk": (H, hid, wl.d), "bq1": (H, hid), "bk1": (H, hid)}
    if second:
        sizes.update(wq2=(H, F, hid), wk2=(H, F, hid), bq2=(H, F), bk2=(H, F))

    def run(w):
        bias = {n: w[n] for n in sizes if n[0] == "b"}
        out = op.forward(dev["q"], dev["k"], dev["v"], w["wq"], w["wk"], biases=bias, **{n: w[n] for n in second})
        return out.view(torch.int16)                             # (bits: a row without a feature above 0 is no number)

    w = {n: dev[n] if n in dev else torch.randn(size, device="cuda", generator=g).bfloat16() for n, size in sizes.items()}
    for n, size in sizes.items():
        late = dict(w, **{n: torch.full_like(w[n], 3.0)})
        want = run(w).clone()
        torch.cuda.synchronize()
        _late(late[n], w[n])
        got = run(late)
        assert op.last_status() == 0
        assert torch.equal(got, want), n
        count = late[n].numel()
        want = run(dict(w, **{n: written.flatten()[-count:].view(size)})).clone()
        out = torch.full_like(written, 3.0)
        torch.cuda.synchronize()
        before.forward(*x, out=out)
        got = run(dict(w, **{n: out.flatten()[-count:].view(size)}))
        assert op.last_status() == 0
        assert torch.equal(got, want), n


@pytest.mark.parametrize("with_state", [False, True])
@pytest.mark.parametrize("d", [64, 128])
def test_a_query_pass_right_behind_the_kernel_that_writes_its_input(d, with_state):
    import torch
    wl, dev, op, _ = _layer(d, 4)
    ks, vs, S, z = (x.clone() for x in op.key_pass(dev["k"], dev["v"], dev["wq"], dev["wk"]))
    state = (S, z) if with_state else (None, None)
    want = op.query_pass(dev["q"], dev["wq"], dev["wk"], ks, vs, *state).clone()
    inputs = {"q": dev["q"], "ks": ks, "S": S} if with_state else {"q": dev["q"], "ks": ks}
    for n, src in inputs.items():
        x = dict(q=dev["q"], ks=ks, S=state[0])
        x[n] = torch.full_like(src, 3.0)
        torch.cuda.synchronize()
        _late(x[n], src)
        got = op.query_pass(x["q"], dev["wq"], dev["wk"], x["ks"], vs, x["S"], state[1])
        assert op.last_status() == 0
        assert torch.equal(got, want), n


@pytest.mark.parametrize("name", ["hybrid_d128", "hybrid_d64"])
def test_a_gradient_right_behind_the_kernel_that_writes_the_teacher(name):
    import torch
    wl, dev, op, _ = _layer(**LAYERS[name])
    args = [dev[n] for n in ("q", "k", "v", "wq", "wk")]
    y = to_cuda_bf16(W.teacher_output(wl))
    aux = torch.empty((wl.B, wl.H, wl.N, 3), dtype=torch.float32, device="cuda")
    y_hat = op.forward(*args, aux=aux)
    want = op.backward_phi(*args, y, y_hat, aux)
    late = torch.full_like(y, 3.0)
    torch.cuda.synchronize()
    _late(late, y)
    got = op.backward_phi(*args, late, y_hat, aux)
    assert op.last_status() == 0
    for a, b in zip(got, want):
        assert torch.equal(a, b)


@pytest.mark.parametrize("name", sorted(LAYERS))
def test_a_captured_step_gives_the_results_of_the_calls(name):
    """Forward (and gradient, where the layer has one) captured into a graph and replayed on other inputs in the same buffers."""
    import torch
    wl, dev, op, second = _layer(**LAYERS[name])
    args = [dev[n] for n in ("q", "k", "v", "wq", "wk")]
    gradient = wl.rate != 1 and not second
    y = to_cuda_bf16(W.teacher_output(wl))
    aux = torch.empty((wl.B, wl.H, wl.N, 3), dtype=torch.float32, device="cuda")
    out = torch.empty_like(dev["q"])

    def step():
        op.forward(*args, out=out, aux=aux, **second)
        return op.backward_phi(*args, y, out, aux) if gradient else ()

    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(side):
        step()                                           # workspaces are there before the capture
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            captured = step()
    torch.cuda.synchronize()
    dev["q"].copy_(dev["q"].flip(2))
    dev["v"].copy_(dev["v"].flip(1))
    want = [x.clone() for x in step()] + [out.clone(), aux.clone()]
    out.zero_()
    for _ in range(2):
        graph.replay()
    torch.cuda.synchronize()
    assert op.last_status() == 0
    got = list(captured) + [out, aux]
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    del graph


@pytest.mark.parametrize("name", sorted(LAYERS) + ["two_layers_128", "two_layers_d64", "biased_linear"])
def test_nothing_is_written_behind_a_time_out_of_the_kernel_before(name):
    """The kernel whose wait runs out lets dependents in first: they have looked at the status word when it is raised.  Neither outputs nor the workspace change, and
    the handle works again once the status has been read."""
    import torch
    from paper_2509_24899_b200 import binding
    layers = dict(LAYERS, two_layers_128=dict(d=128, rate=4, F=128, hidden=128), two_layers_d64=dict(d=64, rate=4, F=64, hidden=64),
                  biased_linear=dict(d=128, rate=0))
    wl, dev, op, second = _layer(**layers[name])
    bias = {n: torch.ones((wl.H, op.F), dtype=torch.bfloat16, device="cuda") for n in ("bq1", "bk1")} if name == "biased_linear" else None
    args = [dev[n] for n in ("q", "k", "v", "wq", "wk")]
    aux = torch.empty((wl.B, wl.H, wl.N, 3), dtype=torch.float32, device="cuda")

    def run(out=None, k=args[1]):
        return op.forward(args[0], k, *args[2:], out=out, aux=aux, biases=bias, **second)

    good, stats = run().clone(), aux.clone()
    assert op.last_status() == 0
    out, other = torch.full_like(good, 7.0), torch.randn_like(args[1])
    aux.fill_(7.0)
    before = op.workspace().clone()
    torch.cuda.synchronize()
    binding.as_hybrid_attn_debug_expire_wait(op.handle, 2_000_000, torch.cuda.current_stream().cuda_stream)
    for _ in range(2):
        run(out, other)
    torch.cuda.synchronize()
    assert torch.equal(out, torch.full_like(good, 7.0)) and torch.equal(aux, torch.full_like(aux, 7.0))
    assert torch.equal(op.workspace(), before)
    assert op.last_status() == binding.AS_ERR_DEVICE_TIMEOUT and op.last_status() == 0
    assert torch.equal(run(out), good) and torch.equal(aux, stats)
    assert op.last_status() == 0


@pytest.mark.parametrize("d", [64, 128])
def test_no_partial_gradient_is_written_behind_a_time_out(d):
    import torch
    from paper_2509_24899_b200 import binding
    wl, dev, op, _ = _layer(d, 4)
    args = [dev[n] for n in ("q", "k", "v", "wq", "wk")]
    y = to_cuda_bf16(W.teacher_output(wl))
    aux = torch.empty((wl.B, wl.H, wl.N, 3), dtype=torch.float32, device="cuda")
    y_hat = op.forward(*args, aux=aux)
    want = [x.clone() for x in op.backward_phi(*args, y, y_hat, aux)]
    assert op.last_status() == 0
    other, before = args[0].flip(2).contiguous(), op._bws.clone()
    torch.cuda.synchronize()
    binding.as_hybrid_attn_debug_expire_wait(op.handle, 2_000_000, torch.cuda.current_stream().cuda_stream)
    op.backward_phi(other, *args[1:], y, y_hat, aux)             # (sums over the chunks of dS and dz, formed again from the same partials, are the same)
    torch.cuda.synchronize()
    assert torch.equal(op._bws, before)
    assert op.last_status() == binding.AS_ERR_DEVICE_TIMEOUT and op.last_status() == 0
    assert all(torch.equal(a, b) for a, b in zip(op.backward_phi(*args, y, y_hat, aux), want))


@pytest.mark.parametrize("H,N,rate,d", [(2, 10000, 1, 128), (1, 8000, 1, 64), (5, 9467, 2, 64)])
def test_key_loops_in_parts_write_nothing_behind_a_time_out(H, N, rate, d):
    import torch
    from paper_2509_24899_b200 import HybridAttention, binding
    from _query_plan import plan
    assert plan(N, H, rate, d, d)["parts"]
    g = torch.Generator(device="cuda").manual_seed(N)
    q, k, v = (torch.randn((1, H, N, d), device="cuda", generator=g).bfloat16() for _ in range(3))
    w = {} if rate == 1 else {n: (torch.randn((H, d, d), device="cuda", generator=g) * 0.05).bfloat16() for n in ("wq", "wk")}
    op = HybridAttention(1, H, N, d, (1, 1, N), (1, 1, N), rate)
    good = op.forward(q, k, v, **w).clone()
    assert op.last_status() == 0
    out, before = torch.full_like(good, 7.0), op.workspace().clone()
    other = q.flip(2).contiguous()
    torch.cuda.synchronize()
    binding.as_hybrid_attn_debug_expire_wait(op.handle, 2_000_000, torch.cuda.current_stream().cuda_stream)
    for _ in range(2):
        op.forward(other, k, v, out=out, **w)
    torch.cuda.synchronize()
    assert torch.equal(out, torch.full_like(good, 7.0)) and torch.equal(op.workspace(), before)
    assert op.last_status() == binding.AS_ERR_DEVICE_TIMEOUT
    for _ in range(2):
        assert torch.equal(op.forward(q, k, v, out=out, **w), good)
    assert op.last_status() == 0
