"""A step, a refresh and the alignment diagnostic recorded in a CUDA graph and
replayed give what the same calls give when they are enqueued: the kernels'
early launches (programmatic dependent launch) become edges of the graph.
Bit-exact."""

import pytest

import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_captured_calls(dtype):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15037_gb300 as M
    shapes = [(320, 264, 40), (130, 520, 64), (64, 72, 8)]
    tdt = torch.bfloat16 if dtype == "bf16" else torch.float32
    gs = [torch.tensor(synth.lowrank_grad(m, n, 8, 10.0, 0.05, 1, seed=3, module=i, noise_rel=True),
                       dtype=torch.float32).to(tdt).cuda() for i, (m, n, r) in enumerate(shapes)]
    outs = []
    for captured in (False, True):
        g = M.MoaraGroup(block_size=64)
        for i, (m, n, r) in enumerate(shapes):
            g.add(m, n, r, dtype, W0=synth.init_weight(m, n, seed=i))

        S = torch.zeros(len(shapes), dtype=torch.float32, device="cuda")

        def calls(t, stream):
            g.refresh(gs, stream=stream)
            g.step(gs, t, 1e-3, stream=stream)
            if dtype == "bf16":
                M.moara_alignment(g.ctx, g.ids, [x.data_ptr() for x in gs], S.data_ptr(), stream)

        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        calls(1, s.cuda_stream)                   # work lists and module tables are made here
        s.synchronize()
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=s):
                calls(2, s.cuda_stream)
            graph.replay()
        else:
            calls(2, s.cuda_stream)
        torch.cuda.synchronize()
        assert g.status() == 0
        outs.append([S.clone()] + [x.clone() for b in g.modules for x in (b.W, b.P, b.exp_avg)])
        g.close()
    for a, b in zip(*outs):
        assert torch.equal(a, b)
