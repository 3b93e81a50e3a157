"""Bounded waits that run out in the products on CTA pairs (refreshes and
alignments of few weights, and the alignment's second product), left and right
projectors, at limits from far below a copy's latency (every wait gives up) to
above a whole product's: the pair gives up anywhere in between, in one CTA or
both.  Each time the host reads the status, no copy is left in flight, and the
context goes on: with the default bound the next refresh and alignment are
those of a context that was never interrupted."""

import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("side", ["left", "smaller"])
@pytest.mark.parametrize("shapes", [
    [(264, 2048, 40)],                                 # a pair tile each, K of 32 and of 1 stages
    [(2312, 1304, 96), (130, 1304, 24), (3000, 2056, 264)],    # persistent pairs with several tiles
])
def test_pairs_give_up_and_recover(shapes, side):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15037_gb300 as M
    gs = [torch.tensor(synth.lowrank_grad(m, n, 16, 10.0, 0.05, 1, seed=2, module=i, noise_rel=True),
                       dtype=torch.float32).to(torch.bfloat16).cuda() for i, (m, n, _) in enumerate(shapes)]
    limits = [100, 100, 500, 1000, 2000, 4000, 8000, 16000, 100000]
    outs = []
    for interrupt in (False, True):
        g = M.MoaraGroup(block_size=64, proj_rule=M.MOARA_PROJ_SMALLER if side == "smaller" else M.MOARA_PROJ_LEFT)
        for m, n, r in shapes:
            g.add(m, n, r, "bf16")
        seen = []
        for limit in limits:
            g.refresh(gs)
            torch.cuda.synchronize()
            assert g.status() == 0
            if interrupt:
                M.moara_set_wait_limit(g.ctx, limit)
            g.alignment(gs)
            torch.cuda.synchronize()
            seen.append(g.status())
            g.refresh(gs)
            torch.cuda.synchronize()
            seen.append(g.status())
            M.moara_set_wait_limit(g.ctx, 0)
        if interrupt:
            assert set(seen) <= {0, M.MOARA_ERR_DEVICE_TIMEOUT} and seen[:4] == [M.MOARA_ERR_DEVICE_TIMEOUT] * 4
        else:
            assert not any(seen)
        g.refresh(gs)
        S = g.alignment(gs)
        torch.cuda.synchronize()
        assert g.status() == 0
        outs.append((S.clone(), [b.P.clone() for b in g.modules]))
        g.close()
    assert (outs[0][0] - outs[1][0]).abs().max() <= 1e-6      # atomic additions of the sums, any order
    for a, b in zip(outs[0][1], outs[1][1]):
        assert torch.equal(a, b)
