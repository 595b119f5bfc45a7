"""Performance cases of the blockBP decoder: what its users have it do, through its public entry points.

Five kinds of work, each over the range it is used in:

* ``decode``: a batch of syndromes of one distance (``decode``), from one
  syndrome (a real-time loop) to the 10^4 of a Monte-Carlo step; fused form
  (Remark 9) in FP32 or FP64 with 4 x 4 blocks, 6 x 6 blocks for large
  distances, and the boundary-MPS form (Sec. III.D);
* ``mixed``: syndromes of several distances in one persistent launch
  (``decode_mixed``);
* ``learned``: the decoder started from the network's proposals
  (``decode_warm``);
* ``train``: one optimiser step of that network (``WarmStart.train_step``).

Inputs are the paper's synthetic workload (Sec. IV): i.i.d. depolarizing
errors, drawn from the seed, and their syndromes.
"""

from __future__ import annotations

import math

import torch

import paper_2402_04834_gb300 as bbp
from paper_2402_04834_gb300 import warmstart
from paper_2402_04834_gb300.decoder import decode_mixed

OUTPUTS = ("logp", "delta", "iters", "flags", "decision")
DELTA0, DELTA1, ETA = 1e-4, 1e-2, 0.1        # Sec. IV
F, H, O = 256, 256, 16                       # the warm-start network


def _decode(name, d, B, p=0.10, k=4, D=8, precision="fp32", algorithm="fused", max_iter=20):
    return {"name": name, "kind": "decode", "d": d, "B": B, "p": p, "k": k, "D": D, "precision": precision,
            "algorithm": algorithm, "max_iter": max_iter}


def listed():
    return [
        # A real-time loop hands over one syndrome at a time: latency.
        _decode("single_d11", 11, 1),
        # A short queue of a smaller code at a lower noise level.
        _decode("queue_d9", 9, 64, p=0.08),
        # The benchmark's step: 10^4 syndromes at d = 11, p = 0.10.
        _decode("batch_d11", 11, 10000),
        # The largest distance of the 4 x 4-block studies.
        _decode("batch_d21", 21, 2000),
        # Even distances leave blocks three nodes wide at the far edges.
        _decode("batch_d12", 12, 2000),
        # d = 31 with 6 x 6 blocks.
        _decode("batch_d31_k6", 31, 152, p=0.12, k=6),
        # The FP64 decoder that the FP32 one is checked and compared with.
        _decode("fp64_d11", 11, 1000, precision="fp64"),
        # Plain FP64 blockBP with MPS messages: the smallest studied code, and the benchmark's distance.
        _decode("mps_d5", 5, 200, k=3, D=4, precision="fp64", algorithm="mps", max_iter=10),
        _decode("mps_d11", 11, 24, precision="fp64", algorithm="mps"),
        # Uneven distances in one launch, every distance odd.
        {"name": "mixed", "kind": "mixed", "d_list": "7,9,13,17,21", "B": 4096, "p": 0.10, "odd_kernels": True},
        # The benchmark's headline decoder: 10^4 syndromes started from the network's proposals.
        {"name": "learned_d11", "kind": "learned", "d": 11, "B": 10000, "p": 0.10},
        # One minibatch of the network's training.
        {"name": "train", "kind": "train", "N": 8192},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fused", "fused", "fused", "fp64", "k6", "small_k", "mps64", "mps32", "mixed", "learned",
                       "train"])
    p = round(rng.uniform(0.05, 0.15), 3)
    if kind == "fused":
        d = rng.randint(5, 21)
        case = _decode("", d, _log(rng, 1, min(10000, 600000 // (d * d))), p=p)
    elif kind == "fp64":
        d = rng.randint(5, 15)
        case = _decode("", d, _log(rng, 1, min(1500, 120000 // (d * d))), p=p, precision="fp64")
    elif kind == "k6":
        d = rng.randint(9, 31)
        case = _decode("", d, _log(rng, 1, 140000 // (d * d)), p=p, k=6)
    elif kind == "small_k":
        d, k = rng.randint(5, 13), rng.choice([2, 3])
        case = _decode("", d, _log(rng, 1, 200000 // (d * d)), p=p, k=k)
    elif kind == "mps64":
        d = rng.randint(4, 9)
        case = _decode("", d, _log(rng, 1, 4000 // (d * d)), p=p, k=3, D=4, precision="fp64", algorithm="mps",
                       max_iter=10)
    elif kind == "mps32":
        d = rng.randint(5, 11)
        case = _decode("", d, _log(rng, 1, 2900 // (d * d)), p=p, precision="fp32", algorithm="mps")
    elif kind == "mixed":
        odd = rng.random() < 0.5
        ds = sorted(rng.sample(range(5, 22, 2) if odd else range(5, 20), rng.randint(2, 5)))
        case = {"kind": "mixed", "d_list": ",".join(map(str, ds)), "B": _log(rng, 16, 3000), "p": p,
                "odd_kernels": odd}
    elif kind == "learned":
        d = rng.randint(7, 15)
        case = {"kind": "learned", "d": d, "B": _log(rng, 1, min(8000, 500000 // (d * d))), "p": p}
    else:
        case = {"kind": "train", "N": rng.randint(700, 8000)}
    return {k: v for k, v in case.items() if k != "name"}


# --- inputs -----------------------------------------------------------------

def _syndromes(d, p, B, seed):
    """Syndromes [B, 2 d (d - 1)] of i.i.d. depolarizing errors on the planar code.

    Grid of side 2 d - 1: qubits where i + j is even; checks A (even, odd) see
    the x bits of their neighbours, checks B (odd, even) the z bits."""
    W = 2 * d - 1
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for b0 in range(0, B, 4096):
        n = min(4096, B - b0)
        r = torch.rand(n, W, W, device="cuda", generator=gen)
        i = torch.arange(W, device="cuda")
        qubit = ((i[:, None] + i[None, :]) % 2 == 0)
        x = ((r < 2 * p / 3) & qubit).to(torch.uint8)                       # X or Y
        z = ((r >= p / 3) & (r < p) & qubit).to(torch.uint8)                # Y or Z

        def around(g):
            q = torch.nn.functional.pad(g, (1, 1, 1, 1))
            return q[:, :-2, 1:-1] ^ q[:, 2:, 1:-1] ^ q[:, 1:-1, :-2] ^ q[:, 1:-1, 2:]
        a = around(x)[:, 0::2, 1::2].reshape(n, -1)
        b = around(z)[:, 1::2, 0::2].reshape(n, -1)
        out.append(torch.cat((a, b), 1))
    return torch.cat(out).contiguous()


def _training_rows(N, seed):
    """A minibatch: 0/1 window features, one-hot direction and length, 10 p and 1; unit targets; a network
    and its Adam moments in the middle of a run."""
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def rand(*shape):
        return torch.rand(*shape, device="cuda", generator=gen)

    def randn(*shape):
        return torch.randn(*shape, device="cuda", generator=gen)
    rows = torch.arange(N, device="cuda")
    feats = torch.zeros(N, F, device="cuda")
    feats[:, :245] = (rand(N, 245) < 0.35).float()
    feats[rows, 245 + (rand(N) * 4).long()] = 1.0
    width = torch.where(rand(N) < 0.85, 4, 1)
    feats[rows, 248 + width] = 1.0
    feats[:, 253] = 0.5 + rand(N)
    feats[:, 254] = 1.0
    lens = (2 ** width).to(torch.int32)
    t = torch.exp(1.5 * randn(N, O)) * (torch.arange(O, device="cuda")[None, :] < lens[:, None])
    targets = (t / t.norm(dim=1, keepdim=True)).contiguous()
    theta = torch.cat([q.reshape(-1) for a, b in ((F, H), (H, H), (H, O))
                       for q in (randn(a, b) * math.sqrt(2.0 / (a + b)), 0.02 * randn(b))])
    m = 1e-4 * randn(theta.numel())
    v = 1e-7 * (0.1 + rand(theta.numel()))
    return feats, targets, lens, theta, m, v


def _params(case):
    return bbp.DecoderParams(d=case["d"], k=case.get("k", 4), D=case.get("D", 8), p=case["p"],
                             max_iter=case.get("max_iter", 20), eta=ETA, delta0=DELTA0, delta1=DELTA1,
                             precision=case.get("precision", "fp32"), algorithm=case.get("algorithm", "fused"))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "decode":
        return {"kind": kind, "prm": _params(case), "s": _syndromes(case["d"], case["p"], case["B"], seed),
                "ws": bbp.Workspace()}
    if kind == "learned":
        # The benchmark's network architecture; random parameters stand for trained ones.
        return {"kind": kind, "prm": _params(case), "s": _syndromes(case["d"], case["p"], case["B"], seed),
                "net": warmstart.WarmStart(seed=seed)}
    if kind == "mixed":
        ds = [int(t) for t in case["d_list"].split(",")]
        B = case["B"]
        gen = torch.Generator().manual_seed(seed)
        d_of = torch.tensor(ds)[torch.randint(len(ds), (B,), generator=gen)]
        d_of[0] = ds[-1]
        m_of = 2 * d_of * (d_of - 1)
        offsets = (torch.cumsum(m_of, 0) - m_of).cuda()
        packed = torch.empty(int(m_of.sum()), dtype=torch.uint8, device="cuda")
        for j, d in enumerate(ds):
            mine = (d_of == d).nonzero()[:, 0].cuda()
            if mine.numel():
                s = _syndromes(d, case["p"], mine.numel(), seed + 1000 * (j + 1))
                at = offsets[mine][:, None] + torch.arange(s.shape[1], device="cuda")[None, :]
                packed[at.reshape(-1)] = s.reshape(-1)
        d_dev = d_of.to(torch.int32).cuda()
        prm = bbp.DecoderParams(d=ds[-1], k=4, p=case["p"], max_iter=20, eta=ETA, delta0=DELTA0, delta1=DELTA1,
                                precision="fp32", algorithm="fused", messages=3 if case["odd_kernels"] else 0)
        order = torch.argsort(d_dev, descending=True, stable=True).to(torch.int32)
        counter = torch.empty(256 + bbp.workspace_bytes(prm, B), dtype=torch.uint8, device="cuda")
        return {"kind": kind, "prm": prm, "packed": packed, "offsets": offsets, "d_of": d_dev, "order": order,
                "d_max": ds[-1], "counter": counter}
    feats, targets, lens, theta, m, v = _training_rows(case["N"], seed)
    net = warmstart.WarmStart(seed=seed)
    net.theta.copy_(theta)
    net.m.copy_(m)
    net.v.copy_(v)
    net.step = 100
    return {"kind": kind, "net": net, "feats": feats, "targets": targets, "lens": lens}


def run(state):
    kind = state["kind"]
    if kind == "decode":
        out = bbp.decode(state["s"], state["prm"], workspace=state["ws"])
    elif kind == "learned":
        out = warmstart.decode_warm(state["s"], state["prm"], state["net"])
    elif kind == "mixed":
        out = decode_mixed(state["packed"], state["offsets"], state["d_of"], state["prm"], order=state["order"],
                           d_max=state["d_max"], counter=state["counter"])
    else:
        net = state["net"]
        loss = net.train_step(state["feats"], state["targets"], state["lens"], lr=1e-3)
        return {"loss": loss, "grad": net.grad, "theta": net.theta}
    return {q: out[q] for q in OUTPUTS}


# --- work -------------------------------------------------------------------

def _update_flops(h, c, algorithm, D):
    """One block update: per column t a butterfly per row bit over the 2^h rows and the open legs of the two
    side messages (fused form); the QR and SVD sweeps of c columns and the damping (MPS form)."""
    if algorithm == "mps":
        return 7 * D ** 3 * max(h - 1, 1) * (c + 1)
    return 2 * 2 ** h * h * sum(4 ** min(t, c - 1 - t) for t in range(c))


def _decode_flops(d, k, max_iter, algorithm="fused", D=8):
    W = 2 * d - 1
    sizes = [min(k, W - a) for a in range(0, W, k)]
    n, total = len(sizes), 0
    for I, h in enumerate(sizes):
        for J, c in enumerate(sizes):
            total += ((J + 1 < n) + (J > 0)) * _update_flops(h, c, algorithm, D)
            total += ((I + 1 < n) + (I > 0)) * _update_flops(c, h, algorithm, D)
    return 4 * 0.7 * max_iter * total          # four cosets; they converge after 0.7 max_iter on average


def work(case):
    kind = case["kind"]
    if kind == "train":
        params = F * H + H + H * H + H + H * O + O
        return {"bytes": 4 * (case["N"] * (F + O + 1) + 7 * params), "flops": 6 * case["N"] * (F * H + H * H + H * O)}
    per_out = 4 * (8 + 8 + 4 + 4) + 1
    if kind == "mixed":
        ds = [int(t) for t in case["d_list"].split(",")]
        share = case["B"] / len(ds)
        return {"bytes": sum(share * (2 * d * (d - 1) + 12 + per_out) for d in ds),
                "flops": sum(share * _decode_flops(d, 4, 20) for d in ds)}
    d, B, k = case["d"], case["B"], case.get("k", 4)
    flops = B * _decode_flops(d, k, case.get("max_iter", 20), case.get("algorithm", "fused"), case.get("D", 8))
    return {"bytes": B * (2 * d * (d - 1) + per_out), "flops": flops}


# --- 64-bit results ---------------------------------------------------------

def _exact_decode(s, d, k, p, max_iter):
    """log P and Delta [B, 4] of dense block belief propagation in FP64: every k x k block contracted into one
    tensor of the messages' legs, Remarks 2-8 and Lemma 1 as written."""
    dev, W = s.device, 2 * d - 1
    B = s.shape[0]
    a = s[:, :d * (d - 1)].reshape(B, d, d - 1).to(torch.int64)
    b = s[:, d * (d - 1):].reshape(B, d - 1, d).to(torch.int64)
    fx = torch.zeros(B, 4, W, W, dtype=torch.int64, device=dev)
    fz = torch.zeros_like(fx)
    fx[:, :, 0::2, 2::2] = (torch.cumsum(a, 2) % 2)[:, None]
    fz[:, :, 2::2, 0::2] = (torch.cumsum(b, 1) % 2)[:, None]
    fx[:, 1:3, 0, 0::2] ^= 1
    fz[:, 2:4, 0::2, 0] ^= 1
    N = 4 * B
    fx, fz = fx.reshape(N, W, W), fz.reshape(N, W, W)
    bits = [torch.arange(2, device=dev)]

    def node(i, j):
        """[N or 1, left, right, up, down]; legs that leave the grid have one value."""
        n = (1 if j == 0 else 2, 1 if j == W - 1 else 2, 1 if i == 0 else 2, 1 if i == W - 1 else 2)
        l, r, u, dn = (bits[0][:m].reshape([1] + [m if q == e else 1 for e in range(4)]) for q, m in enumerate(n))
        if (i + j) % 2:
            legs = [g for g, m in zip((l, r, u, dn), n) if m == 2]
            t = torch.ones((1,) + n, dtype=torch.float64, device=dev)
            for g in legs[1:]:
                t = t * (g == legs[0])
            return t
        x, z = (u ^ dn, l ^ r) if i % 2 == 0 else (l ^ r, u ^ dn)
        same = (fx[:, i, j].reshape(N, 1, 1, 1, 1) == x) & (fz[:, i, j].reshape(N, 1, 1, 1, 1) == z)
        return torch.full_like(same, p / 3, dtype=torch.float64).masked_fill_(same, 1 - p)

    nb = (W + k - 1) // k
    span = [(q * k, min(q * k + k, W)) for q in range(nb)]
    blocks = {}
    for I in range(nb):
        for J in range(nb):
            (r0, r1), (c0, c1) = span[I], span[J]
            T = None                                   # [N, left legs, right legs, up legs, down legs]
            for i in range(r0, r1):
                row = None                             # one row of nodes: [N, left, right, up, down]
                for j in range(c0, c1):
                    t = node(i, j).expand(N, -1, -1, -1, -1)
                    if row is None:
                        row = t
                    else:
                        q = torch.einsum("nlaud,narvw->nlruvdw", row, t)
                        row = q.reshape(N, q.shape[1], q.shape[2], q.shape[3] * q.shape[4], q.shape[5] * q.shape[6])
                if T is None:
                    T = row
                else:
                    q = torch.einsum("nlrua,nLRad->nlLrRud", T, row)
                    T = q.reshape(N, q.shape[1] * q.shape[2], q.shape[3] * q.shape[4], q.shape[5], q.shape[6])
            blocks[I, J] = T
    step = {"R": (0, 1), "L": (0, -1), "D": (1, 0), "U": (-1, 0)}
    back = {"R": "L", "L": "R", "D": "U", "U": "D"}
    axis = {"L": "l", "R": "r", "U": "u", "D": "d"}

    def near(I, J, q):
        i, j = I + step[q][0], J + step[q][1]
        return (i, j) if 0 <= i < nb and 0 <= j < nb else None

    edges = [(I, J, q) for I in range(nb) for J in range(nb) for q in "RLDU" if near(I, J, q)]
    size = {(I, J, q): 2 ** (span[I][1] - span[I][0] if q in "RL" else span[J][1] - span[J][0]) for I, J, q in edges}
    msg = {e: torch.full((N, size[e]), size[e] ** -0.5, dtype=torch.float64, device=dev) for e in edges}
    one = torch.ones(N, 1, dtype=torch.float64, device=dev)

    def close(I, J, out):
        """The block with every incoming message but the one from ``out`` (None: all of them)."""
        ins = {}
        for q in "LRUD":
            if q != out:
                at = near(I, J, q)
                ins[q] = msg[at[0], at[1], back[q]] if at else one
        T, legs = blocks[I, J], "lrud"
        for q in sorted(ins, key="UDLR".index):
            rest = legs.replace(axis[q], "")
            T = torch.einsum("n%s,n%s->n%s" % (legs, axis[q], rest), T, ins[q])
            legs = rest
        return T

    act = torch.ones(N, dtype=torch.bool, device=dev)
    delta = torch.zeros(N, dtype=torch.float64, device=dev)
    for _ in range(max_iter if edges else 0):
        total = torch.zeros(N, dtype=torch.float64, device=dev)
        for colour in (0, 1):
            for e in (e for e in edges if (e[0] + e[1]) % 2 == colour):
                new, old = close(*e), msg[e]
                new = (1 - ETA) * new / new.norm(dim=1, keepdim=True) + ETA * old
                new = new / new.norm(dim=1, keepdim=True)
                total += 2 - 2 * (new * old).sum(1) ** 2
                msg[e] = torch.where(act[:, None], new, old)
        now = total.clamp_min(0).sqrt() / len(edges)
        delta = torch.where(act, now, delta)
        act = act & ~(now < DELTA0)
        if not bool(act.any()):
            break
    logp = torch.zeros(N, dtype=torch.float64, device=dev)
    for I in range(nb):
        for J in range(nb):
            logp += close(I, J, None).abs().log()
    for I, J, q in edges:
        if q in "RD":
            at = near(I, J, q)
            logp -= (msg[I, J, q] * msg[at[0], at[1], back[q]]).sum(1).abs().log()
    return logp.reshape(B, 4), delta.reshape(B, 4)


def _exact_train(N, seed):
    feats, targets, lens, theta, m, v = _training_rows(N, seed)
    th = theta.double().requires_grad_(True)
    parts, at = [], 0
    for a, b in ((F, H), (H, H), (H, O)):
        parts += [th[at:at + a * b].reshape(a, b), th[at + a * b:at + a * b + b]]
        at += a * b + b
    x = feats.double()
    x = torch.nn.functional.gelu(x @ parts[0] + parts[1])
    x = torch.nn.functional.gelu(x @ parts[2] + parts[3])
    o = (x @ parts[4] + parts[5]).masked_fill(torch.arange(O, device="cuda")[None, :] >= lens[:, None], -math.inf)
    u = torch.exp(o - o.max(1, keepdim=True).values)
    u = u / u.norm(dim=1, keepdim=True)
    loss = (1 - (u * targets.double()).sum(1) ** 2).mean()
    loss.backward()
    g = th.grad
    m1, v1 = 0.9 * m.double() + 0.1 * g, 0.999 * v.double() + 0.001 * g * g
    new = theta.double() - 1e-3 * (m1 / (1 - 0.9 ** 101)) / ((v1 / (1 - 0.999 ** 101)).sqrt() + 1e-8)
    return {"loss": loss.detach(), "grad": g, "theta": new}


def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case["N"], seed)
    if case["kind"] != "decode":
        return None                                    # thousands of syndromes in FP64: minutes
    d, k, B = case["d"], case["k"], case["B"]
    blocks = B * 4 * ((2 * d - 1 + k - 1) // k) ** 2
    if blocks * 2 ** (4 * k) > 1e10 or k > 4:          # the dense block tensors
        return None
    s = _syndromes(d, case["p"], B, seed)
    logp, delta = _exact_decode(s, d, k, case["p"], case["max_iter"])
    return {"logp": logp, "delta": delta, "iters": None, "flags": None, "decision": None}
