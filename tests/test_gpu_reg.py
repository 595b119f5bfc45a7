"""The register-form block updates at the edges of their passes: eight jobs
(message, coset) of one shape per warp pass, so small codes leave passes
partly empty (d = 3: one 4 x 4 block and the three one-node-wide ones), and
cosets that stop at different iterations leave one, two or three jobs per
message; even distances have blocks three nodes wide.  Against the dense oracle, with the repository's bars: |delta log P|
<= 1e-9 in FP64 and 1e-3 in FP32."""

import numpy as np
import pytest

import paper_2402_04834_gb300 as pkg
import synth
from oracle.lattice import Lattice
from oracle.naive import run_naive
from oracle.tn import coset_network

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-9), ("fp32", 1e-3)])
@pytest.mark.parametrize("d,B,delta0", [(3, 3, 0.0), (3, 3, 1e-3), (4, 3, 0.0), (5, 3, 1e-3),
                                        (6, 2, 1e-3), (7, 2, 1e-4), (8, 1, 1e-4)])
def test_partly_filled_passes(precision, tol, d, B, delta0):
    p, iters = 0.1, 12
    _, _, S = synth.sample_syndromes(8800 + d, 0, B, d, p)
    want = np.empty((B, 4))
    its = np.empty((B, 4), dtype=np.int64)
    for b in range(B):
        for c in range(4):
            want[b, c], _, its[b, c], _ = run_naive(coset_network(Lattice(d), S[b], c, p), 4, iters, 0.1, delta0)
    first = None
    for warps, cosets, messages in ((0, 0, 0), (8, 1, 1), (8, 2, 3), (4, 2, 1), (4, 4, 1)):
        if messages == 3 and d % 2 == 0:
            continue                                      # odd distances only
        if messages == 3 and precision == "fp64":
            warps, cosets = 4, 2
        prm = pkg.DecoderParams(d=d, k=4, p=p, max_iter=iters, delta0=delta0, precision=precision, algorithm="fused",
                                warps=warps, cosets=cosets, messages=messages)
        out = pkg.decode(torch.from_numpy(S).cuda(), prm)
        got = out["logp"].cpu().numpy()
        same = out["iters"].cpu().numpy() == its          # FP32 may stop an iteration apart at the threshold
        assert same.mean() >= (1.0 if precision == "fp64" else 0.75)
        assert np.max(np.abs(got - want)[same]) <= tol, (warps, cosets, messages)
        if first is None:
            first = out
        for key in ("logp", "delta", "iters", "flags", "decision"):
            assert torch.equal(out[key], first[key]), (warps, cosets, messages, key)


@pytest.mark.gpu
@pytest.mark.parametrize("d,B", [(3, 700), (5, 1), (5, 80), (7, 200), (9, 400), (11, 39), (11, 77), (11, 153), (11, 305),
                                 (11, 2500), (13, 400), (17, 320), (21, 160), (27, 160), (29, 3), (29, 160), (41, 2),
                                 (53, 2), (2, 700), (4, 1), (6, 80), (8, 160), (12, 320), (12, 1000), (20, 400), (26, 3),
                                 (30, 160), (40, 2), (52, 2)])
def test_default_kernel_of_every_size_gives_the_same_bits(d, B):
    # The default launch takes a kernel by geometry and batch; each gives the
    # bits of a kernel asked for by shape (messages in shared memory, or in
    # workspace slots where they do not fit).
    _, _, S = synth.sample_syndromes(9900 + d, 0, B, d, 0.11)
    s = torch.from_numpy(S).cuda()
    base = dict(d=d, k=4, p=0.11, max_iter=6, delta0=2e-3, precision="fp32", algorithm="fused")
    a = pkg.decode(s, pkg.DecoderParams(**base))
    b = pkg.decode(s, pkg.DecoderParams(**base, messages=1 if d <= 46 else 2))
    for key in ("logp", "delta", "iters", "flags", "decision"):
        assert torch.equal(a[key], b[key]), key


@pytest.mark.gpu
@pytest.mark.parametrize("d,k,B", [(4, 6, 5), (7, 6, 60), (8, 6, 3), (9, 6, 60), (13, 6, 3), (13, 5, 60), (16, 6, 45)])
def test_default_kernel_of_large_blocks_gives_the_same_bits(d, k, B):
    # Side remainders 1, 3 and 5 (partial blocks of every width share the
    # launch with full 6 x 6 blocks), one CTA of 16 warps and two of 8 per SM.
    _, _, S = synth.sample_syndromes(9700 + d, 0, B, d, 0.11)
    s = torch.from_numpy(S).cuda()
    base = dict(d=d, k=k, p=0.11, max_iter=5, delta0=2e-3, precision="fp32", algorithm="fused")
    a = pkg.decode(s, pkg.DecoderParams(**base))
    b = pkg.decode(s, pkg.DecoderParams(**base, warps=4, cosets=1, messages=2))
    for key in ("logp", "delta", "iters", "flags", "decision"):
        assert torch.equal(a[key], b[key]), key
