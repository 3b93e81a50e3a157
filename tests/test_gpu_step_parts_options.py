"""Steps of several parts (0.8 GB of gradients each) with what the plain step
does not have: clipping, whose Optimizer_M and K2 run once after all parts,
2-byte states, right projectors, and blocks below 32 columns, whose Optimizer_M
is a pass of its own beside the other part's products.  Against steps of each
weight by itself: bit for bit, and with clipping (the other weights' share of
the norm goes in as one fp32 number, so the coefficients differ by an ulp or
two) to 1e-6 of each result's norm, 1e-3 where the results are rounded to
2 bytes: an ulp's difference crosses a rounding boundary in about one entry of
10^4, by 2^-8 of it."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("states,clip,side,B", [
    ("f32", 1.0, "left", 128), ("bf16", 0.0, "left", 64), ("bf16", 1.0, "smaller", 128), ("f32", 0.0, "smaller", 32),
    ("f32", 0.0, "left", 16), ("f32", 1.0, "smaller", 16), ("f32", 0.0, "left", 8)])
def test_parts_with_options(states, clip, side, B):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15037_gb300 as M
    shapes = [(264, 136, 8)] + [(16384, 8192, 64)] * 6 + [(130, 520, 40)]      # 1.6 GB: two parts
    gen = torch.Generator(device="cuda")

    def setup(idx):
        g = M.MoaraGroup(block_size=B, clip_norm=clip,
                         state_dtype=M.MOARA_DTYPE_BF16 if states == "bf16" else M.MOARA_DTYPE_F32,
                         proj_rule=M.MOARA_PROJ_SMALLER if side == "smaller" else M.MOARA_PROJ_LEFT)
        for k, i in enumerate(idx):
            m, n, r = shapes[i]
            gen.manual_seed(i)
            mid = g.add(m, n, r, "bf16")
            g.modules[k].W.normal_(0.0, 0.02, generator=gen)
            rows = n if side == "smaller" and m > n else m
            g.load_projector(mid, torch.randn(rows, r, device="cuda", generator=gen) / rows ** 0.5)
        return g

    def grad(i, t):
        m, n, _ = shapes[i]
        gen.manual_seed(100 * t + i)
        return torch.randn(m, n, device="cuda", generator=gen, dtype=torch.bfloat16)

    def sq(i, t):
        return float(grad(i, t).float().square().sum(dtype=torch.float64))

    group = setup(range(len(shapes)))
    coef = {}
    for t in (1, 2):
        group.step([grad(i, t) for i in range(len(shapes))], t, 1e-3)
        torch.cuda.synchronize()
        if clip:
            total = sum(sq(i, t) for i in range(len(shapes)))
            coef[t] = [float(x) for x in group.clip_state()]
            assert coef[t][0] == pytest.approx(total ** 0.5, rel=1e-6) and coef[t][1] < 1e-3
    assert group.status() == 0
    for i in range(len(shapes)):
        one = setup([i])
        for t in (1, 2):
            if clip:
                one.set_clip_extra(torch.tensor([coef[t][0] ** 2 - sq(i, t)], dtype=torch.float32, device="cuda"))
            one.step([grad(i, t)], t, 1e-3)
        torch.cuda.synchronize()
        a, b = one.modules[0], group.modules[i]
        for name in ("W", "exp_avg", "exp_avg_sq", "mag_avg", "mag_avg_sq"):
            x, y = getattr(a, name), getattr(b, name)
            if not clip:
                assert torch.equal(x, y), (i, name)
            else:
                bar = 1e-3 if x.dtype == torch.bfloat16 else 1e-6
                assert float((x.double() - y.double()).norm()) <= bar * float(x.double().norm()), (i, name)
        one.close()
    group.close()
