"""Block sides 5 and 6 by the call without a launch shape, against the dense
oracle with the repository's bars: every remainder of the grid's side (last
blocks one to five nodes wide), a batch of one and, in FP32, one that takes the
kernel with two CTAs per SM.  d = 6 and 9 at k = 6 have 6 x 5 blocks, whose
states do not fit the small buffers, and run the full-size ones."""

import numpy as np
import pytest

import paper_2402_04834_gb300 as pkg
import synth
from oracle.lattice import Lattice
from oracle.naive import run_naive
from oracle.tn import coset_network

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("k,d", [(6, 4), (6, 5), (6, 6), (6, 7), (6, 8), (6, 9), (5, 4), (5, 5), (5, 6), (5, 7)])
def test_default_call_matches_the_dense_oracle(k, d):
    p, iters = 0.1, 5
    _, _, S = synth.sample_syndromes(9300 + d, 0, 60, d, p)
    want = [run_naive(coset_network(Lattice(d), S[0], c, p), k, iters, 0.1, 0.0)[0] for c in range(4)]
    s = torch.from_numpy(S).cuda()
    for precision, tol in (("fp64", 1e-9), ("fp32", 1e-3)):
        prm = pkg.DecoderParams(d=d, k=k, p=p, max_iter=iters, delta0=0.0, precision=precision, algorithm="fused")
        one, many = pkg.decode(s[:1].contiguous(), prm), pkg.decode(s, prm)
        assert np.max(np.abs(one["logp"][0].cpu().numpy() - np.array(want))) <= tol
        for key in ("logp", "delta", "iters", "flags", "decision"):
            assert torch.equal(one[key], many[key][:1]), (precision, key)
