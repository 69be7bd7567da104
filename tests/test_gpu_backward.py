"""Gradient of the value-distillation loss w.r.t. the feature-map weights: CUDA library against the float64 oracle.

The library differentiates at ITS forward output (bf16) while the oracle differentiates at the exact one.  The L1
loss has a kink where the student's output equals the teacher's: an element on which the two outputs fall on
different sides of the teacher's value flips sign(y_hat - y), and a fraction p of flipped terms moves a sum of
randomly signed terms by about 2 sqrt(p) of its size, whatever the arithmetic.  So there are two kinds of case:
  * teacher outputs kept at least 0.05 away from the oracle's student output (built from the oracle's forward pass):
    no flips, the comparison sees the arithmetic alone - fp32 sums and the bf16 roundings of the forward pass (y_hat,
    S, z, aux).  Bound: relative L2 <= 5e-3 on dW_q and dW_k.
  * free-standing random teacher outputs (`workloads.teacher_output`, what the benchmark uses): flips happen on about
    one element in several thousand.  Bound: relative L2 <= 3e-2.
The loss itself is compared to 2e-3 relative in both.
"""
import numpy as np
import pytest

from oracle import hybrid_attention as O
from oracle import hybrid_backward as G
from paper_2509_24899_b200 import workloads as W
from _util import balanced_gain, errors, from_cuda_bf16, oracle_inputs, oracle_mask, to_cuda_bf16, _record

pytestmark = pytest.mark.gpu

CASES = {
    "ragged_d128": W.Workload("bw_ragged_d128", B=1, H=2, d=128, F=128, grid=(3, 10, 13), block=(1, 6, 8), rate=4, seed=61),
    "batch_d64": W.Workload("bw_batch_d64", B=2, H=3, d=64, F=64, grid=(2, 9, 31), block=(1, 4, 4), rate=2, seed=62,
                            rms_norm_qk=False),
    "rate0": W.Workload("bw_rate0", B=1, H=2, d=128, F=128, grid=(2, 10, 13), block=(1, 6, 8), rate=0, seed=63),
    "degree1": W.Workload("bw_degree1", B=1, H=2, d=128, F=128, grid=(3, 10, 13), block=(1, 6, 8), rate=3, seed=64, degree=1),
    "degree4_chunks": W.Workload("bw_degree4", B=1, H=1, d=128, F=128, grid=(6, 30, 52), block=(1, 6, 8), rate=8, seed=65, degree=4),
    # several 128-token tiles per chunk (accumulation across tiles, tiles loaded ahead) and a batch to sum over
    "tiles_per_chunk_batch": W.Workload("bw_tiles", B=2, H=20, d=128, F=128, grid=(1, 30, 52), block=(1, 6, 8), rate=4, seed=66),
}


def _teacher_with_margin(wl, d64, mode, margin=0.05):
    """Teacher outputs at least `margin` away from the oracle's student output, either side at random."""
    y_hat, _ = O.hybrid_attention(d64["q"], d64["k"], d64["v"], d64["wq"], d64["wk"], oracle_mask(wl), None, mode, wl.degree)
    rng = np.random.default_rng(wl.seed + 78)
    off = (margin + np.abs(0.5 * rng.standard_normal(y_hat.shape))) * rng.choice([-1.0, 1.0], size=y_hat.shape)
    return W.f32_to_bf16_bits(np.nan_to_num(y_hat + off).astype(np.float32))


def _run(wl, mode, gain, margin, simt=False):
    import torch
    from paper_2509_24899_b200 import HybridAttention, binding
    data = W.generate(wl, wq_gain=gain)
    y_bits = _teacher_with_margin(wl, oracle_inputs(data), mode) if margin else W.teacher_output(wl)
    dev = {k: to_cuda_bf16(v) for k, v in data.items()}
    y_dev = to_cuda_bf16(y_bits)
    # (the default path runs the products on the tensor cores; the fp32 CUDA-core kernels are the check path)
    kw = {"kernel_path": binding.AS_PATH_SIMT} if simt else {}
    op = HybridAttention.from_workload(wl, stab_mode=mode, **kw)
    aux = torch.empty((wl.B, wl.H, wl.N, 3), dtype=torch.float32, device="cuda")
    y_hat = op.forward(dev["q"], dev["k"], dev["v"], dev["wq"], dev["wk"], aux=aux)
    dwq, dwk, loss = op.backward_phi(dev["q"], dev["k"], dev["v"], dev["wq"], dev["wk"], y_dev, y_hat, aux)
    again = op.backward_phi(dev["q"], dev["k"], dev["v"], dev["wq"], dev["wk"], y_dev, y_hat, aux)
    torch.cuda.synchronize()
    assert op.last_status() == 0
    assert torch.equal(dwq, again[0]) and torch.equal(dwk, again[1]) and torch.equal(loss, again[2])   # fixed-order sums
    d64 = oracle_inputs(data)
    ref_loss, ref_q, ref_k = G.phi_weight_gradients(d64["q"], d64["k"], d64["v"], d64["wq"], d64["wk"], oracle_mask(wl),
                                                    W.bf16_bits_to_f64(y_bits), None, mode, wl.degree)
    return (dwq.cpu().numpy().astype(np.float64), dwk.cpu().numpy().astype(np.float64), float(loss.item()),
            ref_q, ref_k, ref_loss)


@pytest.mark.parametrize("margin", [True, False])
@pytest.mark.parametrize("mode", [O.STAB_PAPER, O.STAB_EXACT])
@pytest.mark.parametrize("name", sorted(CASES))
def test_phi_weight_gradients_match_the_oracle(mode, name, margin):
    wl = CASES[name]
    gain = balanced_gain(wl, mode)
    dwq, dwk, loss, ref_q, ref_k, ref_loss = _run(wl, mode, gain, margin)
    eq, ek = errors(dwq, ref_q)[0], errors(dwk, ref_k)[0]
    _record({"case": "backward/%s/%s/%s" % (name, "exact" if mode == O.STAB_EXACT else "paper",
                                            "teacher-with-margin" if margin else "free-teacher"),
             "rel_l2_dWq": eq, "rel_l2_dWk": ek, "loss_rel_err": abs(loss - ref_loss) / ref_loss})
    assert np.abs(ref_q).max() > 0 and np.abs(ref_k).max() > 0
    tol = 5e-3 if margin else 3e-2
    assert eq <= tol and ek <= tol, (eq, ek)
    assert abs(loss - ref_loss) <= 2e-3 * ref_loss


@pytest.mark.parametrize("name", ["ragged_d128", "rate0", "degree1"])
def test_phi_weight_gradients_on_the_cuda_core_path(name):
    """d = F = 128 on the fp32 check path (the default path takes these shapes to the tensor cores)."""
    wl = CASES[name]
    dwq, dwk, loss, ref_q, ref_k, ref_loss = _run(wl, O.STAB_PAPER, balanced_gain(wl, O.STAB_PAPER), True, simt=True)
    eq, ek = errors(dwq, ref_q)[0], errors(dwk, ref_k)[0]
    _record({"case": "backward/%s/paper/teacher-with-margin/cuda-cores" % name, "rel_l2_dWq": eq, "rel_l2_dWk": ek,
             "loss_rel_err": abs(loss - ref_loss) / ref_loss})
    assert eq <= 5e-3 and ek <= 5e-3, (eq, ek)
    assert abs(loss - ref_loss) <= 2e-3 * ref_loss


# B, H, grid, block, rate, degree, stab_mode: less than a tile, one row past a tile, whole tiles, several tiles a chunk (odd
# and even counts), more (batch, head) pairs than SMs, no softmax tokens
D64_SHAPES = [(1, 1, (1, 7, 9), (1, 4, 4), 2, 2, O.STAB_PAPER), (1, 2, (1, 3, 43), (1, 4, 4), 0, 1, O.STAB_PAPER),
              (1, 1, (1, 16, 16), (1, 4, 4), 4, 2, O.STAB_EXACT), (2, 40, (2, 20, 21), (1, 4, 4), 8, 2, O.STAB_EXACT),
              (3, 60, (1, 29, 31), (1, 4, 4), 32, 1, O.STAB_PAPER), (1, 30, (2, 30, 52), (1, 6, 8), 0, 2, O.STAB_PAPER)]


@pytest.mark.parametrize("offset", [0, 1])
@pytest.mark.parametrize("shape", D64_SHAPES, ids=str)
def test_narrow_head_gradient_has_the_precision_of_the_cuda_core_kernels(shape, offset):
    """d = 64: the tensor-core kernels (three bf16 pieces) next to the fp32 kernels of the check path, on the same y_hat, row
    statistics and state, and against the chain rule in 64 bits on those.  Sums over up to 3120 tokens in fp32, in blocks of 128:
    a few times 2^-24 sqrt(log2(3120)) each, so 1e-6 (the fp32 kernels: up to 6e-7 here).  `offset`: a teacher tensor that starts
    2 bytes off, which TMA cannot address."""
    import torch
    from paper_2509_24899_b200 import HybridAttention, binding
    B, H, grid, block, rate, degree, mode = shape
    N, d = int(np.prod(grid)), 64
    wl = W.Workload("bw_d64", B=B, H=H, d=d, F=d, grid=grid, block=block, rate=rate, seed=67, degree=degree)
    dev = {k: to_cuda_bf16(v) for k, v in W.generate(wl, wq_gain=2e-3 if rate else 1.0).items()}
    flat = torch.empty(B * H * N * d + 8, dtype=torch.bfloat16, device="cuda")
    y = flat[offset:offset + B * H * N * d].view(B, H, N, d)
    y.copy_(to_cuda_bf16(W.teacher_output(wl)))
    ops = [HybridAttention.from_workload(wl, stab_mode=mode, kernel_path=k) for k in (binding.AS_PATH_TENSOR, binding.AS_PATH_SIMT)]
    aux = torch.empty((B, H, N, 3), dtype=torch.float32, device="cuda")
    args = [dev[n] for n in ("q", "k", "v", "wq", "wk")]
    y_hat = ops[0].forward(*args, aux=aux)
    ops[1]._ws = ops[0].workspace()                     # S and z of the tensor path's forward
    got = [op.backward_phi(*args, y, y_hat, aux) for op in ops]
    S, z = (x.double() for x in ops[0].linear_state())
    assert ops[0].last_status() == 0

    def phi(x, w):
        a = x.double() @ w.double().transpose(-1, -2)
        power = torch.arange(d, device="cuda") // (d // degree)
        return a.relu() ** (power + 1), (a > 0) * (power + 1) * a.relu() ** power

    q, k, v, wq, wk = args
    lam = torch.exp(-aux[..., 0].double()) if mode == O.STAB_EXACT and rate else torch.ones_like(aux[..., 0], dtype=torch.float64)
    w = (lam / (aux[..., 1].double() + lam * aux[..., 2].double()))[..., None]
    diff = y_hat.double() - y.double()
    G = diff.sign()
    t = -(G * y_hat.double()).sum(-1, keepdim=True)
    phi_q, slope_q = phi(q, wq)
    dwq = ((w * (G @ S.transpose(-1, -2) + z[:, :, None] * t) * slope_q).transpose(-1, -2) @ q.double()).sum(0)
    dS, dz = (w * phi_q).transpose(-1, -2) @ G, (w * phi_q * t).sum(2)
    linear = torch.from_numpy(~oracle_mask(wl)).cuda()[:, None]
    dwk = (((v.double() @ dS.transpose(-1, -2) + dz[:, :, None]) * phi(k, wk)[1] * linear).transpose(-1, -2) @ k.double()).sum(0)
    for dq, dk, loss in got:
        # a pre-activation whose rounding changes its sign flips a slope of one: one row of one token, so the median over the features
        for a, r in ((dq, dwq), (dk, dwk)):
            err = (a.double() - r).norm(dim=-1) / r.norm(dim=-1)
            assert err.median() <= 1e-6 and (err > 1e-5).sum() <= 2, err.max()
        assert abs(loss.item() - diff.abs().sum().item()) <= 1e-5 * diff.abs().sum().item()


def test_narrow_head_gradient_takes_a_copy_of_the_state_at_any_float_boundary():
    """d = 64, the forward workspace copied to an address 4 bytes past a 16-byte boundary: the CUDA-core kernels' results, bit for bit."""
    import torch
    from paper_2509_24899_b200 import HybridAttention, binding
    wl = W.Workload("bw_d64_copy", B=1, H=2, d=64, F=64, grid=(1, 9, 31), block=(1, 4, 4), rate=4, seed=69)
    dev = {k: to_cuda_bf16(v) for k, v in W.generate(wl, wq_gain=2e-3).items()}
    y = to_cuda_bf16(W.teacher_output(wl))
    ops = [HybridAttention.from_workload(wl, kernel_path=k) for k in (binding.AS_PATH_TENSOR, binding.AS_PATH_SIMT)]
    aux = torch.empty((wl.B, wl.H, wl.N, 3), dtype=torch.float32, device="cuda")
    args = [dev[n] for n in ("q", "k", "v", "wq", "wk")]
    y_hat = ops[0].forward(*args, aux=aux)
    ws = ops[0].workspace()
    copy = torch.empty(ws.numel() + 16, dtype=torch.uint8, device="cuda")[4:4 + ws.numel()]
    assert copy.data_ptr() % 16 == 4
    copy.copy_(ws)
    ops[0]._ws, ops[1]._ws = copy, ws
    got = [op.backward_phi(*args, y, y_hat, aux) for op in ops]
    assert ops[0].last_status() == 0
    for a, b in zip(*got):
        assert torch.equal(a, b) and bool(torch.isfinite(a).all())


# less than a tile of 64, whole tiles, one row more, an odd number of tiles, more tiles a chunk than the ring has slots; every power
@pytest.mark.parametrize("B,H,N,rate,degree,mode", [(1, 1, 40, 2, 2, O.STAB_PAPER), (1, 2, 64, 0, 1, O.STAB_PAPER), (1, 2, 65, 4, 4, O.STAB_EXACT),
                                                    (1, 3, 192, 3, 2, O.STAB_EXACT), (2, 75, 700, 4, 4, O.STAB_PAPER), (1, 150, 321, 0, 2, O.STAB_PAPER)])
def test_gradient_at_the_edges_of_tiles(B, H, N, rate, degree, mode):
    """d = 128: the tensor-core kernels and (up to degree 2, which they take) the fp32 ones against the chain rule in 64 bits on the same
    y_hat, row statistics and state.  The operands g, lambda phi_q, dL/da, S, dS of the first are rounded to bf16 (2^-9 each, at random):
    2e-3 to 4e-3 in relative L2; 6e-3 asserted.  The fp32 kernels as at d = 64: 1e-6 for the median feature."""
    import torch
    from paper_2509_24899_b200 import HybridAttention, binding
    wl = W.Workload("bw_edges", B=B, H=H, d=128, F=128, grid=(1, 1, N), block=(1, 1, N), rate=rate, seed=68, degree=degree)
    dev = {k: to_cuda_bf16(v) for k, v in W.generate(wl, wq_gain=2e-3 if rate else 1.0).items()}
    y = to_cuda_bf16(W.teacher_output(wl))
    paths = [binding.AS_PATH_TENSOR] + ([binding.AS_PATH_SIMT] if degree <= 2 else [])
    ops = [HybridAttention.from_workload(wl, stab_mode=mode, kernel_path=k) for k in paths]
    aux = torch.empty((B, H, N, 3), dtype=torch.float32, device="cuda")
    args = [dev[n] for n in ("q", "k", "v", "wq", "wk")]
    y_hat = ops[0].forward(*args, aux=aux)
    for op in ops[1:]:
        op._ws = ops[0].workspace()                     # S and z of the tensor path's forward
    got, *got_fp32 = [op.backward_phi(*args, y, y_hat, aux) for op in ops]
    S, z = (x.double() for x in ops[0].linear_state())
    assert ops[0].last_status() == 0
    q, k, v, wq, wk = (x.double() for x in args)
    power = torch.arange(128, device="cuda") // (128 // degree)

    def phi(x, w):
        a = x @ w.transpose(-1, -2)
        return a.relu() ** (power + 1), (a > 0) * (power + 1) * a.relu() ** power

    lam = torch.exp(-aux[..., 0].double()) if mode == O.STAB_EXACT and rate else torch.ones_like(aux[..., 0], dtype=torch.float64)
    w = (lam / (aux[..., 1].double() + lam * aux[..., 2].double()))[..., None]
    diff = y_hat.double() - y.double()
    G = diff.sign()
    t = -(G * y_hat.double()).sum(-1, keepdim=True)
    phi_q, slope_q = phi(q, wq)
    dwq = ((w * (G @ S.transpose(-1, -2) + z[:, :, None] * t) * slope_q).transpose(-1, -2) @ q).sum(0)
    dS, dz = (w * phi_q).transpose(-1, -2) @ G, (w * phi_q * t).sum(2)
    linear = torch.from_numpy(~oracle_mask(wl)).cuda()[:, None]
    dwk = (((v @ dS.transpose(-1, -2) + dz[:, :, None]) * phi(k, wk)[1] * linear).transpose(-1, -2) @ k).sum(0)
    for a, r in ((got[0], dwq), (got[1], dwk)):
        assert float((a.double() - r).norm() / r.norm()) <= 6e-3
    assert abs(got[2].item() - diff.abs().sum().item()) <= 1e-5 * diff.abs().sum().item()
    for dq, dk, loss in got_fp32:
        for a, r in ((dq, dwq), (dk, dwk)):
            err = (a.double() - r).norm(dim=-1) / r.norm(dim=-1)
            assert err.median() <= 1e-6 and (err > 1e-5).sum() <= 2, err.max()
        assert abs(loss.item() - diff.abs().sum().item()) <= 1e-5 * diff.abs().sum().item()


def _small_step(d, degree=2, seed=74):
    """A layer of 200 tokens after its forward: (handle, arguments of the gradient, y_hat, aux)."""
    import torch
    from paper_2509_24899_b200 import HybridAttention
    wl = W.Workload("bw_small", B=1, H=2, d=d, F=d, grid=(1, 1, 200), block=(1, 1, 200), rate=4, seed=seed, degree=degree)
    dev = {k: to_cuda_bf16(v) for k, v in W.generate(wl, wq_gain=2e-3).items()}
    op = HybridAttention.from_workload(wl)
    aux = torch.empty((wl.B, wl.H, wl.N, 3), dtype=torch.float32, device="cuda")
    args = [dev[n] for n in ("q", "k", "v", "wq", "wk")]
    return op, args, op.forward(*args, aux=aux), aux


@pytest.mark.parametrize("d", [64, 128])
def test_signs_at_the_edges_of_bf16(d):
    """sign(y_hat - y) where the difference is the smallest bf16 number, and where it is infinity less infinity: that is no number, and
    neither is the loss, nor the gradient (which y_hat enters)."""
    import torch
    op, args, y_hat, aux = _small_step(d)
    g = torch.Generator(device="cuda").manual_seed(75)
    negative = torch.rand(y_hat.shape, device="cuda", generator=g) < 0.5
    least = (negative.to(torch.int16) * -32768 + 1).to(torch.int16).view(torch.bfloat16)
    zero, far = torch.zeros_like(y_hat), torch.where(negative, 1.0, -1.0).bfloat16()
    got = [op.backward_phi(*args, y, least, aux)[:2] for y in (zero, far)]
    for a, b in zip(*got):
        assert torch.equal(a, b) and bool(a.any())
    y = zero.clone()
    y[0, 1, 77, 5] = y_hat[0, 1, 77, 5] = float("inf")
    dwq, dwk, loss = op.backward_phi(*args, y, y_hat, aux)
    assert op.last_status() == 0
    assert bool(loss.isnan().all()) and not bool(dwq[1].isfinite().all()) and not bool(dwk[1].isfinite().all())
    assert bool(dwq[0].isfinite().all()) and bool(dwk[0].isfinite().all())


@pytest.mark.parametrize("d,degree", [(64, 1), (64, 2), (128, 1), (128, 2), (128, 4)])
def test_a_student_output_that_is_no_number_reaches_every_feature(d, degree):
    """One NaN in y_hat: dL/dphi of that token is NaN, and its product with a slope of zero as well, whatever the feature's power."""
    op, args, y_hat, aux = _small_step(d, degree)
    y = y_hat.clone()
    y_hat[0, 1, 77, 5] = float("nan")
    dwq, dwk, loss = op.backward_phi(*args, y, y_hat, aux)
    assert op.last_status() == 0
    assert bool(loss.isnan().all()) and bool(dwq[1].isnan().all()) and bool(dwk[1].isnan().all())
    assert not bool(dwq[0].any()) and not bool(dwk[0].any())


@pytest.mark.parametrize("d", [64, 128])
def test_loss_keeps_its_precision_near_the_teacher(d):
    """y_hat one bf16 unit from y on half of the elements and equal on the rest, values spread over several decades.  The loss is a sum
    of positive fp32 terms, each exact; a term goes through some 16 + 3 + 5 + 8 + 12 + 5 additions of 2^-24 each at most: 1e-6 with their
    roundings at random (square root of 49 times 2^-24: 4e-7), 3e-6 at worst."""
    import torch
    from paper_2509_24899_b200 import HybridAttention
    wl = W.Workload("bw_near", B=1, H=2, d=d, F=d, grid=(1, 1, 500), block=(1, 1, 500), rate=4, seed=70)
    dev = {k: to_cuda_bf16(v) for k, v in W.generate(wl, wq_gain=2e-3).items()}
    op = HybridAttention.from_workload(wl)
    aux = torch.empty((wl.B, wl.H, wl.N, 3), dtype=torch.float32, device="cuda")
    args = [dev[n] for n in ("q", "k", "v", "wq", "wk")]
    op.forward(*args, aux=aux)
    g = torch.Generator(device="cuda").manual_seed(70)
    r = [torch.randn(aux.shape[:3] + (d,), device="cuda", generator=g) for _ in range(3)]
    y = ((4.0 * r[0]).exp() * r[1].sign()).bfloat16()
    bits = y.view(torch.int16)
    y_hat = torch.where(r[2] > 0.5, bits + 1, torch.where(r[2] < -0.8, bits - 1, bits)).view(torch.bfloat16)
    _, _, loss = op.backward_phi(*args, y, y_hat, aux)
    assert op.last_status() == 0
    want = (y_hat.double() - y.double()).abs().sum().item()
    assert abs(loss.item() - want) <= 1e-6 * want


def test_backward_argument_errors_and_zero_gradient_without_linear_tokens():
    import torch
    from paper_2509_24899_b200 import HybridAttention, binding, AsError
    wl = CASES["ragged_d128"].with_rate(1)
    dev = {k: to_cuda_bf16(v) for k, v in W.generate(wl).items()}
    y = to_cuda_bf16(W.teacher_output(wl))
    op = HybridAttention.from_workload(wl)
    aux = torch.empty((wl.B, wl.H, wl.N, 3), dtype=torch.float32, device="cuda")
    y_hat = op.forward(dev["q"], dev["k"], dev["v"], aux=aux)
    dwq, dwk, _ = op.backward_phi(dev["q"], dev["k"], dev["v"], dev["wq"], dev["wk"], y, y_hat, aux, want_loss=False)
    torch.cuda.synchronize()
    assert not dwq.any() and not dwk.any()                      # rate 1: the output does not depend on phi
    two = W.Workload("bw_two", B=1, H=1, d=128, F=128, grid=(1, 4, 8), block=(1, 4, 8), rate=2, seed=1, layers=2)
    op2 = HybridAttention.from_workload(two)
    with pytest.raises(AsError) as e:
        binding.as_hybrid_attn_backward_workspace_bytes(op2.handle)
    assert e.value.status == binding.AS_ERR_UNSUPPORTED
