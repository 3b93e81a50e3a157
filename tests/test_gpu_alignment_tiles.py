"""The alignment diagnostic at the edges of its tiles: one 8 x 8 block, one
row or column tile plus a remainder, ranks of one 64-deep stage and past
several, every block size (two norms per 16 entries at B = 8), more column
tiles than one, and both projection sides.  Bar 1e-4 as for the other
alignment tests (R in two bf16 planes, fp32 sums)."""

import numpy as np
import pytest

from oracle import moara_ref as o
import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("B", [8, 16, 32, 64, 128])
@pytest.mark.parametrize("side", ["left", "smaller"])
def test_alignment_tile_edges(B, side):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15037_gb300 as M
    shapes = [(8, 8, 8), (9, 264, 8), (257, 248, 72), (128, 256, 64), (1300, 136, 136), (300, 1032, 264)]
    g = M.MoaraGroup(block_size=B, precision=M.MOARA_PREC_BF16_TC,
                     proj_rule=M.MOARA_PROJ_SMALLER if side == "smaller" else M.MOARA_PROJ_LEFT)
    grads, refs = [], []
    for i, (m, n, r) in enumerate(shapes):
        right = side == "smaller" and m > n
        G = synth.to_bf16_exact(synth.lowrank_grad(m, n, min(16, m, n), 10.0, 0.01, 0, seed=B, module=i, noise_rel=True))
        P = synth.to_bf16_exact(synth.random_orthonormal(n if right else m, r, seed=B, module=i))
        g.load_projector(g.add(m, n, r, "bf16"), P)
        grads.append(torch.tensor(G, dtype=torch.float32).to(torch.bfloat16).cuda())
        refs.append(o.alignment(G, P, B, right=right))
    S = g.alignment(grads).cpu().numpy()
    assert g.status() == 0
    g.close()
    assert np.max(np.abs(S - np.array(refs))) <= 1e-4, (S, refs)
