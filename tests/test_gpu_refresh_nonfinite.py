"""A refresh on a gradient that is not finite, or whose products overflow, keeps
the projector, and the next refresh of the same context is as if it had not
been.  With and without orthogonal iterations, with a sketch of full width (no
column of the Ritz vectors is left out), on both kinds of products."""

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("what", ["nan", "inf", "overflow"])
@pytest.mark.parametrize("ritz_iters", [0, 3])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_projector_kept(dtype, ritz_iters, what):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15037_gb300 as M
    m, n, r = 72, 136, 72                       # l = r = 72: more than one block, every column gathered
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    good = torch.tensor(synth.lowrank_grad(m, n, 8, 10.0, 0.5, 1, seed=3, noise_rel=True), dtype=torch.float32).to(tdt).cuda()
    bad = good.clone()
    if what == "overflow":
        bad.mul_(1e25)
    else:
        bad[5, 7] = float(what)
    outs = []
    for seq in ([bad, good], [good, good]):
        g = M.MoaraGroup(block_size=64, decompose=0, ritz_iters=ritz_iters)
        mid = g.add(m, n, r, dtype)
        P0 = torch.eye(m, r, device="cuda")
        g.load_projector(mid, P0)
        g.refresh(seq[:1])
        torch.cuda.synchronize()
        assert g.status() == 0
        if seq[0] is bad:
            assert torch.equal(g.modules[0].P, P0)
        g.refresh(seq[1:])
        torch.cuda.synchronize()
        assert g.status() == 0
        outs.append(g.modules[0].P.clone())
        g.close()
    assert torch.equal(*outs) and not torch.equal(outs[0], P0)
    P = outs[0].double().cpu().numpy()
    assert np.abs(P.T @ P - np.eye(r)).max() <= 1e-5
