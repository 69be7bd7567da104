"""Key loops in parts behind full rounds of whole units, whose ring items and phases the parts go on from, and with few of them; every feature map, biases, a state and keys
from outside; outputs and row statistics compared with the layer in 64 bits."""
import pytest

from _query_plan import plan

pytestmark = pytest.mark.gpu

# (heads, N, one softmax token in, d, F, hidden, biases, powers, exact)
LAYERS = [(5, 8513, 2, 128, 128, 0, False, 2, False), (5, 8650, 2, 128, 256, 0, False, 2, True), (5, 8513, 2, 128, 384, 0, False, 2, False),
          (8, 7143, 2, 128, 256, 256, False, 2, False), (7, 8102, 3, 128, 128, 128, False, 2, True), (8, 7143, 3, 64, 64, 0, False, 2, False),
          (7, 8102, 3, 64, 64, 64, False, 2, True), (8, 7143, 3, 64, 64, 0, True, 2, False), (8, 7143, 2, 128, 128, 0, True, 2, True),
          (7, 8102, 3, 64, 64, 64, True, 2, False), (2, 10726, 2, 128, 256, 256, True, 2, False), (2, 11976, 2, 128, 256, 0, True, 4, True)]


def _phi(x, w, b, side, P, hidden):
    import torch
    a = torch.relu(x @ w["w" + side].transpose(-1, -2) + b.get("b%s1" % side, 0))
    if hidden:                                                # rounded as the kernels keep it
        a = torch.relu(a.bfloat16().double() @ w["w%s2" % side].transpose(-1, -2) + b.get("b%s2" % side, 0))
    part = a.shape[-1] // P
    return torch.cat([a[..., i * part:(i + 1) * part] ** (i + 1) for i in range(P)], -1)


def _check(out, aux, q, k, v, w, b, at, P, hidden, exact, rows):
    """One head at a time: out [rows, d] and aux [rows, 3] of q's rows against all keys."""
    import torch
    d = q.shape[-1]
    soft = torch.zeros(k.shape[1], dtype=torch.bool, device=q.device)
    soft[at] = True
    for h in range(q.shape[0]):
        qq, kk, vv = q[h].double(), k[h].double(), v[h].double()
        wh = {n: x[h].double() for n, x in w.items()}
        bh = {n: x[h].double() for n, x in b.items()}
        s = qq @ kk[soft].T / d ** 0.5
        c = s.amax(-1, keepdim=True)
        e = torch.exp(s - c)
        pk, pq = _phi(kk[~soft], wh, bh, "k", P, hidden), _phi(qq, wh, bh, "q", P, hidden)
        lam = torch.exp(-c) if exact else 1.0
        den_s, den_l = e.sum(-1, keepdim=True), pq @ pk.sum(0)[:, None]
        ref = (e @ vv[soft] + lam * (pq @ (pk.T @ vv[~soft]))) / (den_s + lam * den_l)
        assert float((out[h].double() - ref).norm() / ref.norm()) <= 5e-3, h       # the tolerances of every forward pass and its statistics here
        assert float((aux[h, :, 0].double() - c[:, 0]).abs().max()) <= 2e-3, h
        assert float((aux[h, :, 1].double() - den_s[:, 0]).norm() / den_s.norm()) <= 5e-3, h
        assert float((aux[h, :, 2].double() - den_l[:, 0]).norm() / den_l.norm()) <= 5e-3, h


def _layer(H, N, rate, d, F, hidden, biases, P, exact):
    import torch
    from paper_2509_24899_b200 import AS_STAB_EXACT, AS_STAB_PAPER, HybridAttention
    g = torch.Generator(device="cuda").manual_seed(N + d + F)

    def draw(*shape, gain=1.0):
        return (torch.randn(shape, device="cuda", generator=g) * gain).bfloat16()

    q, k, v = draw(1, H, N, d), draw(1, H, N, d), draw(1, H, N, d)
    k[:, :, N // 2] *= 3.0                                    # a key that some rows' maximum jumps at, in the middle of their loop
    wide = hidden or F
    w = {"wq": draw(H, wide, d, gain=0.02 if not hidden else 0.1), "wk": draw(H, wide, d, gain=0.1)}
    if hidden:
        w.update(wq2=draw(H, F, hidden, gain=0.01), wk2=draw(H, F, hidden, gain=0.1))
    b = {} if not biases else {"bq1": draw(H, wide, gain=0.02), "bk1": draw(H, wide, gain=0.2)}
    if biases and hidden:
        b.update(bq2=draw(H, F, gain=0.02), bk2=draw(H, F, gain=0.2))

    def make(n, **tokens):
        return HybridAttention(1, H, n, d, (1, 1, n), (1, 1, n), rate, phi_dim=F, poly_degree=P, stab_mode=AS_STAB_EXACT if exact else AS_STAB_PAPER,
                               phi_layers=2 if hidden else 1, phi_hidden=hidden or None, **tokens)
    return q, k, v, w, b, make


@pytest.mark.parametrize("layer", LAYERS)
def test_outputs_and_statistics(layer):
    import torch
    H, N, rate, d, F, hidden, biases, P, exact = layer
    planned = plan(N, H, rate, d, F, hidden, biases or P > 2)
    assert planned["parts"] and (planned["rounds"] > 0) == (H > 2)
    q, k, v, w, b, make = _layer(*layer)
    op = make(N)
    aux = torch.empty((1, H, N, 3), dtype=torch.float32, device="cuda")
    out = op.forward(q, k, v, aux=aux, biases=b or None, **w)
    first, stats = out.clone(), aux.clone()
    assert torch.equal(op.forward(q, k, v, aux=aux, biases=b or None, **w), first) and torch.equal(aux, stats)
    assert op.last_status() == 0
    _check(first[0], stats[0], q[0], k[0], v[0], w, b, torch.tensor(op.softmax_indices(), device="cuda"), P, hidden, exact, N)


# what a rank of several has: its own queries against keys from all ranges and the sum of their states
RANGES = [(12, 12, 8190, 8, 128, 128, 0, False, 2, False), (5, 3, 8513, 3, 128, 256, 256, True, 2, True), (8, 2, 7143, 3, 64, 64, 0, False, 2, True), (3, 2, 7000, 4, 64, 64, 64, True, 2, False)]


@pytest.mark.parametrize("ranges", RANGES)
def test_keys_and_state_from_outside(ranges):
    import torch
    H, parts, n, rate, d, F, hidden, biases, P, exact = ranges
    world = parts if parts < 4 else 4
    N = n * world
    q, k, v, w, b, make = _layer(H, N, rate, d, F, hidden, biases, P, exact)
    local = list(range(0, n, rate))
    n_keys = len(local) * world
    assert plan(n, H, rate, d, F, hidden, biases or P > 2, n_keys=n_keys)["parts"]
    op = make(n, softmax_idx=local)
    keys = []
    for r in range(world):
        kk, vv = (x[:, :, r * n:(r + 1) * n].contiguous() for x in (k, v))
        keys.append([x.clone() for x in op.key_pass(kk, vv, w["wq"], w["wk"], biases=b or None, **{m: w[m] for m in w if m[-1] == "2"})])
    ks, vs = (torch.cat([x[i] for x in keys], 1).contiguous() for i in (0, 1))
    S, z = (sum(x[i] for x in keys) for i in (2, 3))
    at = torch.tensor([r * n + i for r in range(world) for i in local], device="cuda")
    r = world - 1
    qq = q[:, :, r * n:(r + 1) * n].contiguous()
    aux = torch.empty((1, H, n, 3), dtype=torch.float32, device="cuda")
    out = op.query_pass(qq, w["wq"], w["wk"], ks, vs, S, z, aux=aux, biases=b or None, **{m: w[m] for m in w if m[-1] == "2"})
    assert op.last_status() == 0
    _check(out[0], aux[0], qq[0], k[0], v[0], w, b, at, P, hidden, exact, n)
