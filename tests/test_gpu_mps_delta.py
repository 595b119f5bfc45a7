"""Delta (Remark 4) of a network that a cluster of thread blocks shares.  Every
block of the cluster sums its own copy of the overlaps and stops by its own
Delta, so the sum has to be ordered before the stores of the next half-round:
otherwise blocks of one cluster may leave the iteration at different times.
The window is widest at k = 1, where an update is shortest and M, the length of
the sum, largest."""

import pytest

import paper_2402_04834_gb300 as pkg
import synth

torch = pytest.importorskip("torch")

KEYS = ("logp", "delta", "iters", "flags", "decision")


@pytest.mark.gpu
@pytest.mark.parametrize("d,sizes", [(9, (1, 4, 13, 24, 60, 200)), (13, (1, 5, 13, 24, 100)), (15, (2, 9, 40))])
def test_early_exit_of_single_node_blocks(d, sizes):
    # M = 1088, 2400 and 3248 messages; with a rule of (warps, blocks per
    # network) by the batch these sizes run, on 152 SMs in FP64, as 8 x 8, 4 x 8,
    # 4 x 5, 4 x 3 and 8 x 2, in FP32 as 8 x 8 down to 8 x 2 and without a cluster.
    p, n = 0.06, max(sizes)
    _, _, S = synth.sample_syndromes(8100 + d, 0, n, d, p)
    S = torch.from_numpy(S).cuda()
    base = dict(d=d, k=1, p=p, max_iter=30, delta0=2e-4, delta1=1e-2)
    fused = pkg.decode(S, pkg.DecoderParams(precision="fp64", algorithm="fused", **base))
    assert len(torch.unique(fused["iters"])) > 3                # networks stop at different iterations
    for precision in ("fp64", "fp32"):
        prm = pkg.DecoderParams(D=2, precision=precision, algorithm="mps", **base)
        whole = pkg.decode(S, prm)
        for b in sizes:
            for _ in range(3):
                out = pkg.decode(S[:b].contiguous(), prm)
                for key in KEYS:
                    assert torch.equal(out[key], whole[key][:b]), (precision, b, key)
        if precision == "fp64":                                 # nothing is truncated at k = 1
            assert torch.equal(whole["iters"], fused["iters"])
            assert float((whole["logp"] - fused["logp"]).abs().max()) <= 1e-9


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("d,k,D,sizes", [(11, 4, 8, (1, 5, 13, 17, 24, 48)), (9, 3, 4, (1, 7, 13, 24, 50, 100)),
                                         (8, 4, 3, (1, 24, 50))])
def test_early_exit_does_not_depend_on_the_cluster_size(precision, d, k, D, sizes):
    # Each batch size here runs another shape than its neighbours in at least
    # one precision, pairs of eight-warp blocks at D > 4 among them.
    _, _, S = synth.sample_syndromes(8200 + d, 0, max(sizes), d, 0.08)
    S = torch.from_numpy(S).cuda()
    prm = pkg.DecoderParams(d=d, k=k, D=D, p=0.08, max_iter=8, delta0=2e-3, precision=precision, algorithm="mps")
    whole = pkg.decode(S, prm)
    assert len(torch.unique(whole["iters"])) > 1
    for b in sizes:
        out = pkg.decode(S[:b].contiguous(), prm)
        for key in KEYS:
            assert torch.equal(out[key], whole[key][:b]), (b, key)
