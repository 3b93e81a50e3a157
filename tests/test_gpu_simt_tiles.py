"""The fp32 products at the edges of their two tilings: 64 x 64 tiles with the
K range split over a cluster (one to eight CTAs, ranks with an empty range),
and 128 x 128 tiles from 304 tiles on.  fp32 arithmetic, so both R (through
exp_avg) and W agree with the float64 oracle to 1e-5 of their largest entry
(a dot product of K <= 2500 terms rounds by about sqrt(K) 2^-24 = 3e-6; the
large Adam eps keeps the sign-like first step from amplifying it)."""

import numpy as np
import pytest

from oracle import moara_ref as o
import synth

from gpu_helpers import rel_err, make_inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = [
    # (m, n, r, B, bf16)
    [(1, 1, 1, 1, False)],
    [(31, 33, 7, 8, False)],               # K below one slice
    [(64, 64, 64, 64, False)],
    [(65, 63, 40, 16, True)],
    [(97, 130, 65, 48, False)],            # three slices over two CTAs
    [(2049, 71, 64, 64, True)],            # K = 2049: eight CTAs
    [(500, 1003, 91, 64, True), (33, 65, 20, 64, True), (1367, 40, 7, 64, True)],   # mixed K in one launch
    [(70, 66, 9, 32, False)] * 9,          # more problems than the small parameter block holds
    [(2300, 2201, 20, 64, False)],         # update: 18 x 18 = 324 wide tiles
]


@pytest.mark.parametrize("mods", SHAPES)
@pytest.mark.parametrize("decompose", [1, 0])
def test_fp32_products(mods, decompose):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15037_gb300 as M
    B, bf16 = mods[0][3], mods[0][4]
    shapes = [w[:3] for w in mods]
    grads, W0 = make_inputs(shapes, B, 2, bf16, seed=7)
    hp = o.Hparams(block_size=B, adam_eps=1e-2, decompose=bool(decompose))
    g = M.MoaraGroup(block_size=B, adam_eps=1e-2, decompose=decompose, precision=M.MOARA_PREC_FP32)
    refs = []
    for i, (m, n, r) in enumerate(shapes):
        P = synth.random_orthonormal(m, r, seed=7, module=i).astype(np.float32).astype(np.float64)
        refs.append(o.run(o.init_state(W0[i], r, B, P=P), grads[i], 1e-3, hp, auto_refresh=False))
        g.load_projector(g.add(m, n, r, "bf16" if bf16 else "f32", W0=W0[i]), P)
    for t in (1, 2):
        g.step([torch.tensor(x[t - 1], dtype=torch.float32).to(torch.bfloat16 if bf16 else torch.float32).cuda()
                for x in grads], t, 1e-3)
    torch.cuda.synchronize()
    for b, ref in zip(g.modules, refs):
        assert rel_err(b.exp_avg.double().cpu().numpy(), ref.exp_avg) <= 1e-5
        assert rel_err(b.W.double().cpu().numpy(), ref.W) <= 1e-5
    g.close()
