"""Query stages whose last round of units has its key loops cut across CTAs: shares that begin and end inside, at the border of and across units, with and
without a linear branch, in both head dims and all feature maps, and calls in a row on the flags that the one before has left."""
import pytest

pytestmark = pytest.mark.gpu


def _reference(q, k, v, w, idx, P, exact, two):
    """The layer in 64 bits, plain torch; the hidden units rounded to bf16 as the kernels keep them."""
    import torch
    q, k, v = (x.double() for x in (q, k, v))
    w = {n: x.double() for n, x in w.items()}
    N, d = q.shape[2], q.shape[3]
    soft = torch.zeros(N, dtype=torch.bool, device=q.device)
    soft[idx] = True
    s = q @ k[:, :, soft].transpose(-1, -2) / d ** 0.5
    c = s.amax(-1, keepdim=True)
    e = torch.exp(s - c)
    num, den = e @ v[:, :, soft], e.sum(-1, keepdim=True)
    if not bool(soft.all()):
        def phi(x, side):
            a = torch.relu(x @ w["w" + side].transpose(-1, -2))
            if two:
                a = torch.relu(a.bfloat16().double() @ w["w%s2" % side].transpose(-1, -2))
            part = a.shape[-1] // P
            return torch.cat([a[..., i * part:(i + 1) * part] ** (i + 1) for i in range(P)], -1)
        pk, pq = phi(k[:, :, ~soft], "k"), phi(q, "q")
        lam = torch.exp(-c) if exact else 1.0
        num = num + lam * (pq @ (pk.transpose(-1, -2) @ v[:, :, ~soft]))
        den = den + lam * (pq @ pk.sum(2)[..., None])
    return num / den


# (B, H, N, one softmax token in, d, F, hidden, powers, exact), on 148 SMs: two CTAs to a unit and five to three, five and eight CTAs to a unit, 88 units behind two
# full rounds; odd numbers of tiles (half of a unit empty), the last key tile ragged; no linear branch, every feature map
CASES = [(1, 2, 12288, 2, 128, 128, 0, 2, False), (1, 2, 12301, 2, 128, 128, 0, 4, True), (2, 1, 9999, 1, 128, 128, 0, 2, False), (1, 1, 8000, 1, 128, 128, 0, 2, False),
         (1, 1, 7900, 1, 64, 64, 0, 2, False), (1, 3, 8200, 2, 64, 64, 0, 2, True), (1, 12, 8190, 2, 128, 128, 0, 2, False), (1, 2, 12288, 2, 128, 256, 0, 2, False),
         (1, 2, 12200, 2, 128, 256, 256, 2, False), (1, 2, 12288, 2, 128, 128, 128, 4, True), (1, 3, 7000, 3, 64, 64, 64, 2, False), (1, 7, 3999, 1, 128, 128, 0, 2, False),
         (1, 1, 4000, 1, 64, 64, 0, 2, False), (1, 1, 20000, 4, 128, 128, 0, 2, False)]


@pytest.mark.parametrize("B,H,N,rate,d,F,hidden,P,exact", CASES)
def test_key_loops_cut_across_ctas(B, H, N, rate, d, F, hidden, P, exact):
    import torch
    from paper_2509_24899_b200 import AS_STAB_EXACT, AS_STAB_PAPER, HybridAttention
    g = torch.Generator(device="cuda").manual_seed(N)

    def draw(*shape, gain=1.0):
        return (torch.randn(shape, device="cuda", generator=g) * gain).bfloat16()

    q, k, v = draw(B, H, N, d), draw(B, H, N, d), draw(B, H, N, d)
    k[:, :, N // 2] *= 3.0                                    # a key that some rows' maximum jumps at, in the middle of their loop
    wide = hidden or F
    w = {"wq": draw(H, wide, d, gain=0.02 if not hidden else 0.1), "wk": draw(H, wide, d, gain=0.1)}
    if hidden:
        w.update(wq2=draw(H, F, hidden, gain=0.01), wk2=draw(H, F, hidden, gain=0.1))
    op = HybridAttention(B, H, N, d, (1, 1, N), (1, 1, N), rate, phi_dim=F, poly_degree=P, stab_mode=AS_STAB_EXACT if exact else AS_STAB_PAPER,
                         phi_layers=2 if hidden else 1, phi_hidden=hidden or None)
    aux = torch.empty((B, H, N, 3), dtype=torch.float32, device="cuda")
    out = op.forward(q, k, v, aux=aux, **w)
    first, stats = out.clone(), aux.clone()
    assert torch.equal(op.forward(q, k, v, aux=aux, **w), first) and torch.equal(aux, stats)
    assert op.last_status() == 0
    at = torch.tensor(op.softmax_indices(), device="cuda")
    for b in range(B):                                        # the tolerance of every forward pass here: relative 2-norm 5e-3
        for h0 in range(0, H, 2):
            sl = (slice(b, b + 1), slice(h0, h0 + 2))
            ref = _reference(q[sl], k[sl], v[sl], {n: x[h0:h0 + 2] for n, x in w.items()}, at, P, exact, hidden > 0)
            err = float((first[sl].double() - ref).norm() / ref.norm())
            assert err <= 5e-3, (b, h0, err)
