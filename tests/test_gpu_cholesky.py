"""The refresh's blocked Cholesky and superblock inverse at sketch widths l
around its tiles: below, at and past one 64-column block, several blocks, the
2304-column superblock and the levels of the inverse past it.  The projector's
columns come through up to sixteen such factorisations, so orthonormality to
1e-5 and the leading singular vectors of a spectrum with clear gaps pin them.
The noise floor (per-direction, of the largest singular value) is that of the
arithmetic: 1e-3 with fp32 products, 1e-1 with bf16 operands, whose Gram
matrices carry 16 bits before the last pass."""

import numpy as np
import pytest

import synth

from gpu_helpers import top_subspace
from oracle import rsi_ref as R

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("bf16,l", [(False, 1), (False, 2), (False, 63), (False, 64), (False, 65), (False, 130),
                                    (False, 511), (False, 512), (False, 513), (False, 579), (False, 640),
                                    (True, 72), (True, 512), (True, 520), (True, 1032),
                                    (False, 2318), (True, 2320)])
def test_refresh_sketch_widths(bf16, l):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15037_gb300 as M
    m, n = (2400, 4800) if l > 1096 else (1152, 1096) if l > 640 else (704, 656)
    r = 1 if l < 8 else 8
    u, v = synth.lowrank_factors(m, n, 8, seed=l)
    G = (u * (10.0 * 0.8 ** np.arange(8))) @ v.T
    G += (0.5 if bf16 else 0.01) / np.sqrt(n) * np.random.default_rng(l).standard_normal((m, n))
    G = synth.to_bf16_exact(G) if bf16 else G.astype(np.float32).astype(np.float64)
    g = M.MoaraGroup(block_size=64, decompose=0, oversample=l - r)
    g.add(m, n, r, "bf16" if bf16 else "f32")
    t = torch.tensor(G, dtype=torch.float32).cuda()
    g.refresh([t.to(torch.bfloat16) if bf16 else t])
    torch.cuda.synchronize()
    assert g.status() == 0
    P = g.modules[0].P.double().cpu().numpy()
    g.close()
    assert np.abs(P.T @ P - np.eye(r)).max() <= 1e-5
    U = top_subspace(G, r)[0]
    if l >= 8:
        assert np.min(np.abs(np.sum(P * U, axis=0))) >= 0.9999
    else:           # a one- or two-column sketch holds a mixture of close directions: the same sketch in 64 bits
        ref = R.randomized_projector(G, r, l - r, 4, R.sketch_key(0, 0, 0))
        assert np.abs(P - ref).max() <= 1e-4 * np.abs(ref).max()      # ten products with V in fp32, about 1e-6 each


@pytest.mark.parametrize("shapes,noise", [
    ([(264, 2048, 40)], 0.05),                       # two row tiles, the second of 8 rows; one column tile of 72
    ([(130, 1304, 24), (2312, 1160, 96)], 0.01),     # mixed K, column tiles of 56 and of 128
    ([(1304, 1032, 232), (1032, 1304, 264)], 0.01),  # l = 264 and 296: a second column tile of 8 and 40
])
def test_refresh_product_tiles(shapes, noise):
    """Refreshes whose products have few tiles and a long K (2-CTA pairs), at
    row and column tiles with remainders, V and G read both ways; the usual
    energy bar."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15037_gb300 as M
    from gpu_helpers import check_refresh
    from oracle import moara_ref as o
    B = 64
    for rule in (M.MOARA_PROJ_LEFT, M.MOARA_PROJ_SMALLER):
        g = M.MoaraGroup(block_size=B, proj_rule=rule)
        gs, Xs = [], []
        for i, (m, n, r) in enumerate(shapes):
            G = synth.to_bf16_exact(synth.lowrank_grad(m, n, 16, 10.0, noise, 1, seed=2, module=i, noise_rel=True))
            g.add(m, n, r, "bf16")
            gs.append(torch.tensor(G, dtype=torch.float32).to(torch.bfloat16).cuda())
            Xs.append(o.decompose(G, B)[1])
        g.refresh(gs)
        torch.cuda.synchronize()
        assert g.status() == 0
        for mid, (m, n, r), X in zip(g.ids, shapes, Xs):
            right = rule == M.MOARA_PROJ_SMALLER and m > n
            P = g.modules[mid].P.double().cpu().numpy()
            check_refresh(P, X.T if right else X, r, g.hp.oversample, g.hp.power_iters, R.sketch_key(g.hp.seed, mid, 0))
        g.close()
