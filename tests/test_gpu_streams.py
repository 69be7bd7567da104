"""Several layers at once, each with a handle and a stream of its own: CTAs of one launch that wait for one another (the sum over the key stage's chunks, key
loops in parts) while those of other launches take the SMs that some of them would need."""
import pytest

pytestmark = pytest.mark.gpu

# (H, N, one softmax token in, d, hidden): key stages that fill the GPU, few long key loops in parts, two layers, no softmax tokens
LAYERS = [(12, 3120, 8, 128, 0), (2, 12288, 2, 128, 0), (1, 7900, 1, 64, 0), (20, 1170, 4, 64, 0), (3, 4000, 4, 128, 128), (7, 6001, 0, 128, 0)]


def test_layers_on_streams_of_their_own_give_what_they_give_alone():
    import torch
    from paper_2509_24899_b200 import HybridAttention
    g = torch.Generator(device="cuda").manual_seed(5)

    def draw(*shape, gain=1.0):
        return (torch.randn(shape, device="cuda", generator=g) * gain).bfloat16()

    work = []
    for H, N, rate, d, hidden in LAYERS:
        op = HybridAttention(1, H, N, d, (1, 1, N), (1, 1, N), rate, phi_layers=2 if hidden else 1, phi_hidden=hidden or None)
        q, k, v = draw(1, H, N, d), draw(1, H, N, d), draw(1, H, N, d)
        w = {"wq": draw(H, hidden or d, d, gain=0.05), "wk": draw(H, hidden or d, d, gain=0.1)}
        if hidden:
            w.update(wq2=draw(H, d, hidden, gain=0.05), wk2=draw(H, d, hidden, gain=0.1))
        want = op.forward(q, k, v, **w).clone()
        work.append((op, (q, k, v), w, want, torch.cuda.Stream(), []))
    torch.cuda.synchronize()
    for _ in range(25):
        for op, qkv, w, _, stream, outs in work:
            with torch.cuda.stream(stream):
                outs.append(op.forward(*qkv, **w))
    torch.cuda.synchronize()
    for op, _, _, want, _, outs in work:
        assert op.last_status() == 0
        assert all(torch.equal(out, want) for out in outs)
