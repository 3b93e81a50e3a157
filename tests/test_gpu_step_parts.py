"""A group step whose gradients fill several parts (0.8 GB each: one, two and
three here, small weights at both ends) gives what a step of each weight by
itself gives.  Bit-exact."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("big", [5, 6, 9])
def test_parts(big):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15037_gb300 as M
    shapes = [(264, 136, 8)] + [(16384, 8192, 64)] * big + [(130, 520, 40)]
    gen = torch.Generator(device="cuda")

    def setup(idx):
        g = M.MoaraGroup(block_size=128)
        for k, i in enumerate(idx):
            m, n, r = shapes[i]
            gen.manual_seed(i)
            mid = g.add(m, n, r, "bf16")
            g.modules[k].W.normal_(0.0, 0.02, generator=gen)
            g.load_projector(mid, torch.randn(m, r, device="cuda", generator=gen) / m ** 0.5)
        return g

    def grad(i, t):
        m, n, _ = shapes[i]
        gen.manual_seed(100 * t + i)
        return torch.randn(m, n, device="cuda", generator=gen, dtype=torch.bfloat16)

    group = setup(range(len(shapes)))
    for t in (1, 2):
        group.step([grad(i, t) for i in range(len(shapes))], t, 1e-3)
    torch.cuda.synchronize()
    assert group.status() == 0
    for i in range(len(shapes)):
        one = setup([i])
        for t in (1, 2):
            one.step([grad(i, t)], t, 1e-3)
        torch.cuda.synchronize()
        a, b = one.modules[0], group.modules[i]
        assert torch.equal(a.W, b.W) and torch.equal(a.exp_avg, b.exp_avg) and torch.equal(a.mag_avg, b.mag_avg)
        one.close()
    group.close()
