"""The alignment diagnostic on subsets of a context's modules: recorded in a graph
without a call on the same subset before, with and without a work list (more
subsets than the context keeps lists of), in any order of the modules, and with
more modules than one launch carries.  The scores of a subset are those of the
calls on one module each; 1e-6 apart for the order of the atomic additions (each
sum is of fp32 partial sums added in fp64)."""

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _group(M, shapes):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    g = M.MoaraGroup(block_size=64, precision=M.MOARA_PREC_BF16_TC)
    Gs = []
    for m, n, r in shapes:
        g.load_projector(g.add(m, n, r, "bf16"), torch.randn(m, r, device="cuda", generator=gen) / m ** 0.5)
        Gs.append(torch.randn(m, n, device="cuda", generator=gen).to(torch.bfloat16))
    return g, Gs


def _one_by_one(g, Gs):
    return torch.stack([g.alignment([G], ids=[mid])[0] for mid, G in zip(g.ids, Gs)])


def _cuda():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2609_15037_gb300 as M
    return M


def test_first_call_on_a_subset_is_capturable():
    M = _cuda()
    g, Gs = _group(M, [(320, 264, 40), (130, 520, 64), (64, 72, 8)])
    s = torch.cuda.Stream()
    S = torch.zeros(3, device="cuda")
    torch.cuda.synchronize()
    M.moara_alignment(g.ctx, g.ids, [G.data_ptr() for G in Gs], S.data_ptr(), s.cuda_stream)
    torch.cuda.synchronize()
    ref = S.clone()
    for pick in ([2, 0], [1], [1, 2]):
        S.zero_()
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            M.moara_alignment(g.ctx, [g.ids[i] for i in pick], [Gs[i].data_ptr() for i in pick], S.data_ptr(),
                              s.cuda_stream)
        graph.replay()
        torch.cuda.synchronize()
        assert g.status() == 0
        assert (S[:len(pick)] - ref[pick]).abs().max() <= 1e-6
    g.close()


@pytest.mark.parametrize("shapes", [
    [(512, 512, 8), (1030, 776, 264), (257, 264, 72), (2304, 1288, 8), (8, 8, 8), (300, 2056, 136)],   # ranks out of order
    [(40 + i % 90, 8 * (1 + i % 40), 8 * (1 + i % 3) if i % 40 > 2 else 8) for i in range(230)],       # two launches
    [(2600, 9000, 8), (264, 520, 72)],                # several rounds of tiles per cluster, the last one partial
])
def test_modules_of_one_call(shapes):
    M = _cuda()
    g, Gs = _group(M, shapes)
    S = g.alignment(Gs)                               # a list is made
    ref = _one_by_one(g, Gs)
    assert (S - ref).abs().max() <= 1e-6
    few = g.ids[:2]
    for k in range(70):                               # as many lists as a context keeps, and more
        m = g.add(8 + k, 16, 8, "bf16")
        g.load_projector(m, torch.eye(8 + k, 8, device="cuda"))
        g.alignment([Gs[0], Gs[1], torch.ones(8 + k, 16, device="cuda", dtype=torch.bfloat16)], ids=few + [m])
    ids = g.ids[:len(shapes)][::-1]                   # a new list of modules: dealt out in turn
    S = g.alignment(Gs[::-1], ids=ids).flip(0)
    torch.cuda.synchronize()
    assert g.status() == 0
    assert (S - ref).abs().max() <= 1e-6
    g.close()
