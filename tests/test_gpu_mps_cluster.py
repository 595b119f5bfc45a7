"""MPS decode with a network shared by a cluster of thread blocks: the cluster
size goes by the batch, each update is the same arithmetic in whichever block
it runs, so a syndrome's outputs do not depend on the batch it comes in.  Batch
sizes reach every cluster size from eight to one of both precisions, networks
without messages, half-rounds smaller than one block's warps, and bond caps
that truncate."""

import pytest

import paper_2402_04834_gb300 as pkg
import synth

torch = pytest.importorskip("torch")


@pytest.mark.gpu
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("d,k,D,sizes", [(3, 4, 8, (1, 9)), (2, 4, 8, (1, 40)), (4, 2, 4, (1, 6, 90)),
                                         (5, 3, 4, (1, 13, 39, 200)), (6, 1, 2, (1, 2, 20)), (8, 4, 3, (1, 3, 7, 20)),
                                         (11, 4, 8, (1, 3, 9, 13)), (21, 4, 4, (1, 2))])
def test_outputs_do_not_depend_on_the_cluster_size(precision, d, k, D, sizes):
    _, _, S = synth.sample_syndromes(7700 + d, 0, max(sizes), d, 0.1)
    S = torch.from_numpy(S).cuda()
    prm = pkg.DecoderParams(d=d, k=k, D=D, p=0.1, max_iter=4, delta0=1e-4, precision=precision, algorithm="mps")
    outs = [pkg.decode(S[:n].contiguous(), prm) for n in sizes]
    for n, out in zip(sizes, outs):
        again = pkg.decode(S[:n].contiguous(), prm)
        for key in ("logp", "delta", "iters", "flags", "decision"):
            assert torch.equal(out[key], outs[-1][key][:n]), (n, key)
            assert torch.equal(out[key], again[key]), (n, key)


@pytest.mark.gpu
@pytest.mark.parametrize("k,d,B", [(1, 3, 5), (1, 4, 40), (2, 2, 3), (2, 3, 300), (2, 4, 1), (2, 5, 30), (2, 7, 9)])
def test_small_bond_instance_equals_the_fused_form(k, d, B):
    # k <= 2 and D = 4 truncate nothing, so the instance for D <= 4 gives the
    # fused form's log P (FP64 bar 1e-9) and, iteration by iteration, its stops.
    _, _, S = synth.sample_syndromes(7900 + d, 0, B, d, 0.1)
    S = torch.from_numpy(S).cuda()
    prm = dict(d=d, k=k, D=4, p=0.1, max_iter=6, delta0=0.0, precision="fp64")
    a = pkg.decode(S, pkg.DecoderParams(algorithm="mps", **prm))
    b = pkg.decode(S, pkg.DecoderParams(algorithm="fused", **prm))
    assert torch.equal(a["iters"], b["iters"])
    assert float((a["logp"] - b["logp"]).abs().max()) <= 1e-9
