"""The key stage by itself: the softmax tokens' rows, bit by bit, and the linear state, at the edges of its tiles and for sets of softmax tokens
from one to all but one."""
import pytest

pytestmark = pytest.mark.gpu

# softmax tokens of N: one in R; a run; all but one, in the last tile; one alone
SETS = {
    "one_in_2": lambda n: range(0, n, 2), "one_in_3": lambda n: range(1, n, 3), "one_in_4": lambda n: range(0, n, 4), "one_in_32": lambda n: range(31, n, 32),
    "run": lambda n: range(n // 3, n // 3 + 70), "all_but_one": lambda n: [i for i in range(n) if i != n - 2], "one": lambda n: [n - 1],
}
# (B, H, N, d, F, layers): one tile, a tile and a row, chunks of several tiles (the ring goes round), more features than lanes
SHAPES = [(1, 2, 128, 64, 64, 1), (1, 3, 129, 128, 128, 1), (2, 1, 255, 64, 64, 2), (1, 40, 1537, 64, 64, 1), (2, 20, 1409, 128, 128, 1), (1, 70, 901, 128, 256, 1),
          (1, 40, 1283, 128, 256, 2)]


@pytest.mark.parametrize("tokens", sorted(SETS))
@pytest.mark.parametrize("B,H,N,d,F,layers", SHAPES)
def test_rows_and_state(B, H, N, d, F, layers, tokens):
    import torch
    from paper_2509_24899_b200 import HybridAttention
    idx = list(SETS[tokens](N))
    g = torch.Generator(device="cuda").manual_seed(N + d)

    def draw(*shape):
        return torch.randn(shape, device="cuda", generator=g).bfloat16()

    k, v, wk = draw(B, H, N, d), draw(B, H, N, d), draw(H, F, d) * 0.1
    second = {"wk2": draw(H, F, F) * 0.1, "wq2": draw(H, F, F)} if layers == 2 else {}
    op = HybridAttention(B, H, N, d, (1, 1, N), (1, 1, N), 2, softmax_idx=idx, phi_dim=F, phi_layers=layers, phi_hidden=F)
    for _ in range(2):                                        # the second call on counters that the first one left
        ks, vs, S, z = op.key_pass(k, v, wk, wk, **second)
    assert op.last_status() == 0
    at = torch.tensor(idx, device="cuda")
    assert torch.equal(ks, k[:, :, at].reshape(B * H, len(idx), d)) and torch.equal(vs, v[:, :, at].reshape(B * H, len(idx), d))
    linear = torch.ones(N, device="cuda", dtype=torch.float64)
    linear[at] = 0
    a = k.double() @ wk.double().transpose(-1, -2)
    if layers == 2:
        a = torch.relu(a).bfloat16().double() @ second["wk2"].double().transpose(-1, -2)
    phi = torch.relu(a) * linear[:, None]
    phi[..., F // 2:] **= 2
    # A feature is rounded to bf16, by at most 2^-8 of itself (half of a spacing of 2^-7); S adds up phi v and z phi, 1e-5 for sums in 32 bits.  Two
    # layers: a hidden unit's sum in 32 bits may fall on the other side of a rounding, so features differ by more, but few of them: the norms are held.
    for got, ref, size in ((S, phi.transpose(-1, -2) @ v.double(), phi.transpose(-1, -2) @ v.double().abs()), (z, phi.sum(2), phi.sum(2))):
        diff = (got.double().reshape(ref.shape) - ref).abs()
        if layers == 1:
            assert bool((diff <= 2.0 ** -8 * size + 1e-5 * size.max()).all()), float((diff / (size + 1e-9)).max())
        else:
            assert float(diff.norm()) <= 2.0 ** -8 * float(size.norm())


# (B, H, N, d, width): one tile; fewer tiles than SMs; two tiles a head, so that a run of tiles goes through several heads (of one batch row and the next);
# runs of a few tiles and of ten, which end inside heads
@pytest.mark.parametrize("B,H,N,d,width", [(1, 1, 128, 64, 64), (2, 3, 300, 128, 128), (3, 50, 130, 128, 128), (2, 97, 200, 64, 64), (2, 40, 701, 64, 64),
                                           (1, 60, 1031, 128, 256), (2, 1, 20001, 128, 256), (1, 12, 15600, 128, 256)])
@pytest.mark.parametrize("bias", [False, True])
def test_first_layer_over_runs_of_tiles(B, H, N, d, width, bias):
    import torch
    from paper_2509_24899_b200 import HybridAttention
    g = torch.Generator(device="cuda").manual_seed(N + d)

    def draw(*shape):
        return torch.randn(shape, device="cuda", generator=g).bfloat16()

    k, v, w1, w2 = draw(B, H, N, d), draw(B, H, N, d), draw(H, width, d) * 0.1, draw(H, width, width) * 0.1
    b1 = draw(H, width)
    biases = {n: b1 if n == "bk1" else torch.zeros_like(b1) for n in ("bq1", "bk1", "bq2", "bk2")} if bias else None
    idx = list(range(0, N, 3))
    op = HybridAttention(B, H, N, d, (1, 1, N), (1, 1, N), 3, softmax_idx=idx, phi_dim=width, phi_layers=2, phi_hidden=width)
    for _ in range(2):
        ks, vs, S, z = op.key_pass(k, v, w1, w1, wk2=w2, wq2=w2, biases=biases)
    assert op.last_status() == 0
    at = torch.tensor(idx, device="cuda")
    assert torch.equal(ks, k[:, :, at].reshape(B * H, len(idx), d)) and torch.equal(vs, v[:, :, at].reshape(B * H, len(idx), d))
    linear = torch.ones(N, device="cuda", dtype=torch.float64)
    linear[at] = 0
    h1 = torch.relu(k.double() @ w1.double().transpose(-1, -2) + (b1.double()[:, None] if bias else 0)).bfloat16().double()
    phi = torch.relu(h1 @ w2.double().transpose(-1, -2)) * linear[:, None]
    phi[..., width // 2:] **= 2
    # features rounded to bf16, 2^-8 of themselves at most; head by head, so that one head with another's weights cannot hide among the others
    for got, ref, size in ((S, phi.transpose(-1, -2) @ v.double(), phi.transpose(-1, -2) @ v.double().abs()), (z, phi.sum(2), phi.sum(2))):
        diff = (got.double().reshape(ref.shape) - ref).flatten(2).norm(dim=2)
        assert bool((diff <= 2.0 ** -8 * size.flatten(2).norm(dim=2)).all())
