"""What the speed of this library is measured on: the calls a user's program makes, over the range of layers it makes them for.

A case names one layer and one use of it:

  forward   `HybridAttention.forward` on device tensors, as a DiT's sampling loop calls it once per layer and step
  step      one step of the value distillation: a forward that keeps its row statistics, then the gradient of the loss
            w.r.t. the feature-map weights (`backward_phi`)
  shard     one rank's share of a layer whose tokens are spread over several GPUs (`SeqShardedAttention.forward`), the
            other ranks' contributions being there already (the exchange itself needs the other GPUs)
  host      `forward_host`: q, k, v and the output in pinned host memory, as an offloading pipeline holds them

`listed` are the library's own benchmark layers and the ragged, biased and narrow-head relatives of them that its tests run;
`draw` gives more layers of the same ranges.
"""
import math

import torch

from paper_2509_24899_b200 import AS_STAB_EXACT, AS_STAB_PAPER, HybridAttention
from paper_2509_24899_b200.seq_shard import SeqShardedAttention

# 480x832 video: 30 x 52 tokens per latent frame, spatial block 6 x 8
WAN = {"gh": 30, "gw": 52, "bt": 1, "bh": 6, "bw": 8}


def _case(use, B, H, d, gt, gh, gw, bt, bh, bw, rate, F=None, hidden=0, degree=2, bias=False, exact=False, ranks=1, **name):
    return dict(name, use=use, B=B, H=H, d=d, gt=gt, gh=gh, gw=gw, bt=bt, bh=bh, bw=bw, rate=rate, F=d if F is None else F,
                hidden=hidden, degree=degree, bias=bias, exact=exact, ranks=ranks)


def listed():
    return [
        # a toy model's layer, N = 1024: a call whose time is launches and latency
        _case("forward", 1, 2, 64, 4, 16, 16, 2, 4, 4, 32, name="forward tiny d64"),
        # 17 frames of 480p, N = 7800: short clips and the coarse stage of a cascade
        _case("forward", 1, 12, 128, 5, rate=8, **WAN, name="forward 17 frames"),
        # 81 frames of 480p, N = 32760, one softmax token in eight: the layer most of the surgery's layers become
        _case("forward", 1, 12, 128, 21, rate=8, **WAN, name="forward 81 frames"),
        # the same layer left as full softmax attention: about a quarter of the layers of a cost-aware stack
        _case("forward", 1, 12, 128, 21, rate=1, **WAN, name="forward 81 frames softmax"),
        # and with no softmax tokens at all: a fifth of them
        _case("forward", 1, 12, 128, 21, rate=0, **WAN, name="forward 81 frames linear"),
        # 161 frames with both branches of classifier-free guidance in the batch, N = 63960: the longest clip
        _case("forward", 2, 12, 128, 41, rate=16, **WAN, name="forward 161 frames cfg"),
        # 81 frames with the paper's default feature map, two layers d -> 2d -> 2d
        _case("forward", 1, 12, 128, 21, rate=8, F=256, hidden=256, **WAN, name="forward 81 frames two-layer map"),
        # narrow heads, a ragged grid whose blocks are clipped, biases, weights exp(s) beside phi phi: the other options in one layer
        _case("forward", 2, 16, 64, 7, 27, 45, 2, 4, 4, 4, bias=True, exact=True, name="forward ragged d64 bias exact"),
        # distilling the 81-frame layer
        _case("step", 1, 12, 128, 21, rate=8, **WAN, name="step 81 frames"),
        # distilling a narrow-head layer on a ragged grid, a batch of two
        _case("step", 2, 12, 64, 2, 27, 45, 1, 4, 4, 4, name="step ragged d64"),
        # a quarter of the 81-frame layer: one rank of four
        _case("shard", 1, 12, 128, 21, rate=8, ranks=4, **WAN, name="shard 81 frames of 4"),
        # 17 frames whose activations live in host memory
        _case("host", 1, 12, 128, 5, rate=8, **WAN, name="host 17 frames"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# the most that a drawn case may cost, below the largest listed one (81 frames of full softmax)
MOST_FLOPS = 6.0e12
MOST_TOKENS = 2 * 12 * 63960             # rows of q over all heads: bounds memory and the linear layers
MOST_STEP_TOKENS_D64 = 250_000           # the narrow-head gradient runs in fp32


def draw(rng):
    """One more case: any use, any grid from a few hundred to some tens of thousands of tokens (odd sides among them), every rate, both
    head dims, the feature maps the library has."""
    while True:
        use = rng.choices(["forward", "step", "shard", "host"], [12, 4, 3, 1])[0]
        d = rng.choices([128, 64], [3, 1])[0]
        B, H = rng.choice([1, 1, 2]), _log_int(rng, 1, 24)
        n = _log_int(rng, 500, 64000)
        gh, gw = (30, 52) if n > 1560 and rng.random() < 0.4 else (rng.randint(9, 34), rng.randint(9, 56))
        gt = max(1, n // (gh * gw))
        bt, bh, bw = rng.choice([(1, 6, 8), (1, 6, 8), (2, 4, 4), (1, 4, 4), (gt, gh, gw)])
        rate = rng.choice([0, 1, 2, 4, 8, 8, 16, 32])
        F, hidden, degree, bias, ranks = d, 0, 2, False, 1
        if use == "step":
            degree = rng.choice([1, 2, 2, 2] if d == 64 else [1, 2, 2, 4])
            rate = rate if rate != 1 else 2                  # full softmax has nothing to distil
        else:
            kind = rng.random()
            if kind < 0.25:
                F, hidden = (64, 64) if d == 64 else rng.choice([(128, 128), (256, 256), (256, 256)])
            elif kind < 0.40 and d == 128:
                F = 256
            degree = rng.choice([1, 2, 2, 2] if F == 64 else [1, 2, 2, 2, 4])
            bias = rng.random() < 0.2
        if use == "shard":
            ranks = rng.choice([2, 4, 8])
        c = _case(use, B, H, d, gt, gh, gw, bt, bh, bw, rate, F, hidden, degree, bias, rng.random() < 0.3, ranks)
        tokens = B * H * gt * gh * gw
        if tokens > MOST_TOKENS or work(c)["flops"] > MOST_FLOPS:
            continue
        if use == "step" and d == 64 and tokens > MOST_STEP_TOKENS_D64:
            continue
        if use == "host" and tokens * d > 12 * 16384 * 128:  # pinned buffers take long to make
            continue
        if use == "shard" and gt * gh * gw < 256 * ranks:
            continue
        return c


def _n_tokens(c):
    return c["gt"] * c["gh"] * c["gw"]


def _n_softmax(c):
    """Softmax tokens of the layer: one in `rate` of every block, the blocks clipped at the grid's border."""
    if c["rate"] <= 1:
        return _n_tokens(c) * c["rate"]
    sides = [[min(b, g - o) for o in range(0, g, b)] for g, b in ((c["gt"], c["bt"]), (c["gh"], c["bh"]), (c["gw"], c["bw"]))]
    return sum(-(-(t * h * w) // c["rate"]) for t in sides[0] for h in sides[1] for w in sides[2])


class _State:
    pass


class _OtherRanks:
    """What the exchanges of a sharded layer bring in: the other ranks' keys and values and their share of the state have arrived.
    Keeps what this rank sends, which is part of its result."""

    def __init__(self, totals, gathered):
        self.totals, self.gathered, self.sent = totals, gathered, []

    def all_reduce_sum(self, t):
        self.sent.append(t)
        return self.totals[t.dim()]

    def all_gather_rows(self, t, rows_per_rank):
        self.sent.append(t)
        return self.gathered[len([x for x in self.sent if x.dtype == torch.bfloat16]) - 1]


def _phi(c, x, w, side, dtype=torch.float32, slope=False):
    """The feature map of rows x [B, H, n, d], of the queries ("q") or the keys ("k"); with `slope` its derivative w.r.t. the last
    layer's sums beside it."""
    a = x.to(dtype) @ w["w" + side].to(dtype).transpose(-1, -2) + (w["biases"]["b%s1" % side].to(dtype)[:, None] if c["bias"] else 0.0)
    if c["hidden"]:
        a = torch.relu(a) @ w["w%s2" % side].to(dtype).transpose(-1, -2)
        a = a + (w["biases"]["b%s2" % side].to(dtype)[:, None] if c["bias"] else 0.0)
    r, part = torch.relu(a), c["F"] // c["degree"]
    cols = [slice(p * part, (p + 1) * part) for p in range(c["degree"])]
    phi = torch.cat([r[..., x] ** (p + 1) for p, x in enumerate(cols)], dim=-1)
    if not slope:
        return phi
    return phi, torch.cat([(a[..., x] > 0) * (p + 1) * r[..., x] ** p for p, x in enumerate(cols)], dim=-1)


def _inputs(c, seed):
    """(q, k, v, weights, teacher's output or None) of a case: whole layers, on the GPU."""
    B, H, N, d, F = c["B"], c["H"], _n_tokens(c), c["d"], c["F"]
    g = torch.Generator(device="cuda").manual_seed(seed)

    def rows(unit_rms):
        x = torch.randn((B, H, N, d), device="cuda", generator=g)
        if unit_rms:                                         # the DiT's QK-norm
            x /= x.square().mean(dim=-1, keepdim=True).sqrt()
        return x.bfloat16()

    def uniform(shape, a):
        return ((2 * torch.rand(shape, device="cuda", generator=g) - 1) * a).bfloat16()

    q, k, v = rows(True), rows(True), rows(False)
    wide = c["hidden"] or F
    a1 = math.sqrt(6.0 / (d + wide))
    w = {"wq": uniform((H, wide, d), a1), "wk": uniform((H, wide, d), a1)}
    if c["hidden"]:
        a2 = math.sqrt(6.0 / (wide + F))
        w["wq2"], w["wk2"] = uniform((H, F, wide), a2), uniform((H, F, wide), a2)
    # a trained map gives the two branches comparable weight; with a map as drawn the linear one holds nearly all of it
    if c["rate"] > 0:
        last = "wq2" if c["hidden"] else "wq"
        w[last] = (w[last].float() * 2e-3).bfloat16()
    if c["bias"]:
        w["biases"] = {n: uniform((H, wide), 0.1) for n in ("bq1", "bk1")}
        if c["hidden"]:
            w["biases"].update({n: uniform((H, F), 0.1) for n in ("bq2", "bk2")})
        if c["rate"] > 0:
            last = "bq2" if c["hidden"] else "bq1"
            w["biases"][last] = (w["biases"][last].float() * 2e-3).bfloat16()
    teacher = (0.5 * torch.randn((B, H, N, d), device="cuda", generator=g)).bfloat16() if c["use"] == "step" else None
    return q, k, v, w, teacher


def prepare(case, seed):
    c, s = case, _State()
    B, H, N, d, F = c["B"], c["H"], _n_tokens(c), c["d"], c["F"]
    q, k, v, w, s.teacher = _inputs(c, seed)
    s.use, s.w = c["use"], w
    kw = {"phi_dim": F, "poly_degree": c["degree"], "stab_mode": AS_STAB_EXACT if c["exact"] else AS_STAB_PAPER,
          "phi_layers": 2 if c["hidden"] else 1, "phi_hidden": c["hidden"] or None}
    grid, block = (c["gt"], c["gh"], c["gw"]), (c["bt"], c["bh"], c["bw"])
    s.op = HybridAttention(B, H, N, d, grid, block, c["rate"], **kw)
    if c["use"] == "shard":
        idx = s.op.softmax_indices()
        at = torch.tensor(idx, dtype=torch.long, device="cuda")
        gathered = [x[:, :, at].reshape(B * H, len(idx), d) for x in (k, v)]
        totals = {}
        if len(idx) < N:
            linear = torch.ones(N, device="cuda")
            linear[at] = 0
            phi = _phi(c, k, w, "k") * linear[:, None]
            totals = {3: (phi.transpose(-1, -2) @ v.float()).reshape(B * H, F, d), 2: phi.sum(dim=2).reshape(B * H, F)}
        s.comm = _OtherRanks(totals, gathered)
        s.op = SeqShardedAttention(B, H, N, d, idx, c["ranks"] // 2, c["ranks"], comm=s.comm, **kw)
        q, k, v = (x[:, :, s.op.n0:s.op.n1].contiguous() for x in (q, k, v))
    if c["use"] == "host":
        q, k, v = (x.cpu().pin_memory() for x in (q, k, v))
        s.out = torch.empty_like(q).pin_memory()
    if c["use"] == "step":
        s.aux = torch.empty((B, H, N, 3), dtype=torch.float32, device="cuda")
    s.q, s.k, s.v = q, k, v
    return s


def run(s):
    if s.use == "forward":
        return s.op.forward(s.q, s.k, s.v, **s.w)
    if s.use == "step":
        out = s.op.forward(s.q, s.k, s.v, aux=s.aux, **s.w)
        dwq, dwk, loss = s.op.backward_phi(s.q, s.k, s.v, s.w["wq"], s.w["wk"], s.teacher, out, s.aux)
        return {"out": out, "aux": s.aux, "dwq": dwq, "dwk": dwk, "loss": loss}
    if s.use == "shard":
        s.comm.sent.clear()
        out = s.op.forward(s.q, s.k, s.v, **s.w)
        return [out] + s.comm.sent
    return s.op.forward_host(s.q, s.k, s.v, out_host=s.out, **s.w)


def work(case):
    """Operations of the method (multiply and add counted as two) and the bytes of its inputs and outputs."""
    c = case
    N, n_s, pairs, d, F, hid = _n_tokens(c), _n_softmax(c), c["B"] * c["H"], c["d"], c["F"], c["hidden"]
    n_l = N - n_s
    share = 1.0 / c["ranks"]
    phi = 2 * d * hid + 2 * hid * F if hid else 2 * d * F
    apply = 2 * F * (d + 1)
    flops = pairs * share * (n_l * (phi + apply) + N * (4 * n_s * d + (phi + apply if n_l else 0)))
    rows = pairs * N * d * 2 * share                         # q, k, v in, the output out
    weights = c["H"] * (2 * d * hid + 2 * hid * F if hid else 2 * d * F) * 2 if n_l else 0
    total = 4 * rows + weights
    if c["use"] == "shard":                                  # the other ranks' keys in, this rank's keys and state out, the summed state in
        total += pairs * n_s * d * 2 * 2 * (1 + (share if n_l else 0)) + (2 * pairs * F * (d + 1) * 4 if n_l else 0)
    if c["use"] == "step":                                   # the teacher's output in, the row statistics and the gradients out
        flops += pairs * (N * 6 * d * F + n_l * 4 * d * F)   # dphi_q, dS, dW_q per query; dphi_k, dW_k per linear key
        total += rows + pairs * N * 3 * 4 + 2 * c["H"] * F * d * 4
    return {"bytes": total, "flops": flops}


def tolerance(case):
    """Outputs are bf16 with bf16 operands inside: the listed layers are 2.1e-3 to 2.5e-3 away from the same layers with fp32 operands
    (`AS_PATH_SIMT`)."""
    if case["use"] == "step":
        # 3e-3 to 4.8e-3 on the gradients of the listed layers in the same comparison, up to 2.1e-2 on layers of a few hundred tokens: the
        # loss |y - y_hat| has a kink, and where another rounding of y_hat falls on the other side of y a whole unit changes sign
        return {"rel": 0.03}
    return {"rel": 0.01}


def _softmax_mask(c):
    """True for the softmax tokens: the raster index inside the token's block, clipped at the grid's border, is a multiple of the rate."""
    sides = [torch.arange(n, device="cuda") for n in (c["gt"], c["gh"], c["gw"])]
    blocks, grid = (c["bt"], c["bh"], c["bw"]), (c["gt"], c["gh"], c["gw"])
    inner = [x % b for x, b in zip(sides, blocks)]
    extent = [torch.clamp(n - x // b * b, max=b) for x, b, n in zip(sides, blocks, grid)]
    at = (inner[0][:, None, None] * extent[1][None, :, None] + inner[1][None, :, None]) * extent[2][None, None, :] + inner[2][None, None, :]
    return (at.reshape(-1) % c["rate"] == 0) if c["rate"] else torch.zeros(_n_tokens(c), dtype=torch.bool, device="cuda")


def exact(case, seed):
    """What `run` returns, in 64 bits from the method's equations."""
    c, f64 = case, torch.float64
    B, H, N, d, F = c["B"], c["H"], _n_tokens(c), c["d"], c["F"]
    q, k, v, w, teacher = _inputs(c, seed)
    soft = _softmax_mask(c)
    lin = ~soft
    n_s = int(soft.sum())
    n0, n1 = 0, N
    if c["ranks"] > 1:                                       # contiguous near-equal ranges, the first ones a token longer
        rank, (base, extra) = c["ranks"] // 2, divmod(N, c["ranks"])
        n0 = rank * base + min(rank, extra)
        n1 = n0 + base + (rank < extra)
    mine = torch.zeros_like(soft)
    mine[n0:n1] = True
    out = torch.empty((B, H, n1 - n0, d), dtype=f64, device="cuda")
    aux = torch.zeros((B, H, N, 3), dtype=f64, device="cuda") if c["use"] == "step" else None
    part = []
    dw = [torch.zeros((H, F, d), dtype=f64, device="cuda") for _ in range(2)]
    loss = torch.zeros(1, dtype=f64, device="cuda")
    step = max(1, (1 << 26) // max(n_s, 4 * F))
    for b in range(B):
        for h in range(H):
            wh = {n: ({m: y[h:h + 1] for m, y in x.items()} if n == "biases" else x[h:h + 1]) for n, x in w.items()}
            phi_of = lambda x, side, **kw: _phi(c, x[None, None], wh, side, f64, **kw)
            ks, vs = k[b, h][soft].to(f64), v[b, h][soft].to(f64)
            S, z, pS, pz = (torch.zeros(x, dtype=f64, device="cuda") for x in ((F, d), (F,), (F, d), (F,)))
            for i in range(0, N, step):
                rows = lin[i:i + step, None].to(f64)
                phi, val = phi_of(k[b, h, i:i + step], "k")[0, 0] * rows, v[b, h, i:i + step].to(f64)
                S += phi.T @ val
                z += phi.sum(dim=0)
                if c["use"] == "shard":
                    phi = phi * mine[i:i + step, None].to(f64)
                    pS += phi.T @ val
                    pz += phi.sum(dim=0)
            part.append((pS, pz))
            dS, dz = torch.zeros_like(S), torch.zeros_like(z)
            for i in range(n0, n1, step):
                j = min(n1, i + step)
                x = q[b, h, i:j]
                num, den, top = torch.zeros((j - i, d), dtype=f64, device="cuda"), torch.zeros(j - i, dtype=f64, device="cuda"), None
                if n_s:
                    e = (x.to(f64) @ ks.T) / math.sqrt(d)
                    top = e.max(dim=1).values
                    e = torch.exp_(e.sub_(top[:, None]))
                    num, den = e @ vs, e.sum(dim=1)
                    del e
                lam = torch.exp(-top) if n_s and c["exact"] else torch.ones_like(den)
                if aux is not None:
                    aux[b, h, i:j, 1] = den
                    if n_s:
                        aux[b, h, i:j, 0] = top
                if n_s < N:
                    phi, slope = (y[0, 0] for y in phi_of(x, "q", slope=True))
                    num = num + lam[:, None] * (phi @ S)
                    den = den + lam * (phi @ z)
                    if aux is not None:
                        aux[b, h, i:j, 2] = phi @ z
                y = num / den[:, None]
                out[b, h, i - n0:j - n0] = y
                if c["use"] == "step":
                    diff = y - teacher[b, h, i:j].to(f64)
                    loss += diff.abs().sum()
                    gy = diff.sign()
                    if n_s < N:
                        g, sden = gy / den[:, None], -(gy * y).sum(dim=1) / den
                        dphi = lam[:, None] * (g @ S.T + sden[:, None] * z)
                        dw[0][h] += (dphi * slope).T @ x.to(f64)
                        phi = lam[:, None] * phi
                        dS += phi.T @ g
                        dz += phi.T @ sden
            if c["use"] == "step" and n_s < N:
                for i in range(0, N, step):
                    x = k[b, h, i:i + step]
                    slope = phi_of(x, "k", slope=True)[1][0, 0] * lin[i:i + step, None]
                    dw[1][h] += ((v[b, h, i:i + step].to(f64) @ dS.T + dz) * slope).T @ x.to(f64)
    if c["use"] == "step":
        return {"out": out, "aux": aux, "dwq": dw[0], "dwk": dw[1], "loss": loss}
    if c["use"] == "shard":
        sent = [torch.stack([x[n] for x in part]) for n in (0, 1)] if n_s < N else []
        own = [x[:, :, soft & mine].reshape(B * H, -1, d).to(f64) for x in (k, v)]
        return [out] + sent + own
    return out.cpu() if c["use"] == "host" else out
