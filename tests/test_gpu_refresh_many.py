"""A refresh of more modules than have a cluster of their own for the
factorisation's chain (39 and more in one launch: a CTA each) gives what
refreshes of fewer give.  Sketch widths of one block and less, of several, with
and without 16-byte rows and whole blocks, on both kinds of products.  Bit for
bit: the chain adds the same terms in the same order on one CTA as on four, and
the products' sums follow from each problem alone."""

import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("count", [38, 39, 60])
def test_many_modules_as_few(dtype, count):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15037_gb300 as M
    step = 8 if dtype == "bf16" else 1                   # l = r + 32 from 33 (40) to about 230
    shapes = [(232 + 3 * k, 240 + 8 * (k % 11), step * (1 + (37 * k) % (200 // step))) for k in range(count)]
    gs = [torch.tensor(synth.lowrank_grad(m, n, 16, 10.0, 0.3, 1, seed=4, module=i, noise_rel=True),
                       dtype=torch.float32).to(torch.bfloat16 if dtype == "bf16" else torch.float32).cuda()
          for i, (m, n, _) in enumerate(shapes)]
    outs = []
    for per_call in (count, 20):
        g = M.MoaraGroup(block_size=64, refresh_workspace_bytes=1 << 30)
        for m, n, r in shapes:
            g.add(m, n, r, dtype)
        assert sum(M.moara_refresh_workspace_bytes(g.ctx, *s) for s in shapes) <= 1 << 30     # one launch group
        for a in range(0, count, per_call):
            g.refresh(gs[a:a + per_call], ids=g.ids[a:a + per_call])
        torch.cuda.synchronize()
        assert g.status() == 0
        outs.append([b.P.clone() for b in g.modules])
        g.close()
    for (m, n, r), a, b in zip(shapes, *outs):
        assert torch.equal(a, b), (m, n, r)
        assert (a.T @ a - torch.eye(r, device="cuda")).abs().max() <= 1e-4      # a refreshed projector (fp32 check)
