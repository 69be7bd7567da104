"""Key loops in parts on values at and past the end of the range: what a part has to leave out and what it must not, compared with the layer in 64 bits."""
import pytest

from _query_plan import plan

pytestmark = pytest.mark.gpu

# (heads, N, one softmax token in, d, F, hidden): one and two threads a row; parts only, and behind full rounds
LAYERS = [(2, 10000, 1, 128, 128, 0), (1, 8000, 1, 64, 64, 0), (2, 12288, 2, 128, 128, 0), (5, 9467, 1, 64, 64, 0), (8, 7121, 2, 64, 64, 64), (5, 9467, 1, 128, 128, 0)]


def _run(layer, change):
    """(output, reference) after `change(k, v, keys)`, whose scores are all of one sign per key: q is positive."""
    import torch
    from paper_2509_24899_b200 import HybridAttention
    H, N, rate, d, F, hidden = layer
    assert plan(N, H, rate, d, F, hidden)["parts"]
    g = torch.Generator(device="cuda").manual_seed(N)

    def draw(*shape):
        return torch.randn(shape, device="cuda", generator=g).bfloat16()

    q, k, v = draw(1, H, N, d).abs(), draw(1, H, N, d), draw(1, H, N, d)
    op = HybridAttention(1, H, N, d, (1, 1, N), (1, 1, N), rate, phi_layers=2 if hidden else 1, phi_hidden=hidden or None)
    keys = torch.tensor(op.softmax_indices(), device="cuda")
    change(k, v, keys)
    w = {} if rate == 1 else {"wq": draw(H, hidden or d, d) * 0.02, "wk": torch.zeros((H, hidden or d, d), device="cuda").bfloat16()}   # no linear branch to speak of
    if hidden:
        w.update(wq2=draw(H, F, hidden), wk2=torch.zeros((H, F, hidden), device="cuda").bfloat16())
    out = op.forward(q, k, v, **w)
    assert op.last_status() == 0
    scores = q[0].double() @ k[0, :, keys].double().transpose(-1, -2) / d ** 0.5
    return out[0].double(), scores, v[0, :, keys].double()


def _close(out, ref):
    assert bool(out.isfinite().all())
    err = float((out - ref).norm() / ref.norm())
    assert err <= 5e-3, err                                   # the tolerance of every forward pass here


@pytest.mark.parametrize("layer", LAYERS)
@pytest.mark.parametrize("begin,end", [(0.2, 0.7), (0.45, 1.0)])
def test_keys_with_scores_of_minus_infinity(layer, begin, end):
    """In 32 bits; a run of them long enough that parts begin with some."""
    import torch

    def change(k, v, keys):
        k[:, :, keys[int(begin * len(keys)):int(end * len(keys))]] = -3e38
    out, scores, v = _run(layer, change)
    _close(out, torch.softmax(scores, -1) @ v)


@pytest.mark.parametrize("layer", LAYERS)
def test_values_at_the_end_of_the_range_under_keys_that_weigh_nothing(layer):
    """The lowest number of the type in every such value: their sum alone is past the end."""
    import torch

    def change(k, v, keys):
        run = keys[int(0.4 * len(keys)):]
        k[:, :, run] = -1e4
        v[:, :, run] = torch.finfo(torch.bfloat16).min
    out, scores, v = _run(layer, change)
    _close(out, torch.softmax(scores, -1) @ v)


@pytest.mark.parametrize("layer", LAYERS)
@pytest.mark.parametrize("value", ["inf", "nan"])
@pytest.mark.parametrize("at", [0.1, 0.9])
def test_a_value_that_is_no_number_shows_in_its_column(layer, value, at):
    """Under a key that weighs nothing: 0 times it, wherever in the loop it comes.  The other columns are right, and finite."""
    import torch
    col = 5

    def change(k, v, keys):
        # all keys but the last tenth - or, for a value there, but the first tenth - weigh nothing
        n = len(keys)
        k[:, :, keys[:int(0.85 * n)] if at < 0.5 else keys[int(0.15 * n):]] = -1e4
        v[:, :, keys[int(at * n)], col] = float(value)
    out, scores, v = _run(layer, change)
    assert not bool(out[..., col].isfinite().any())
    rest = [c for c in range(out.shape[-1]) if c != col]
    _close(out[..., rest], torch.softmax(scores, -1) @ v[..., rest])
