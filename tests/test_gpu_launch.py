"""A stage's kernels are launched so that each launch overlaps the end of the kernel before: several
steps in one call, the same steps one by one with a synchronisation after each, and a captured graph of
them replayed twice on new states give the same bits (no markers: nothing is summed in random order).
"""
import pytest

from paper_1905_00182_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("charwise", [False, True])
@pytest.mark.parametrize("re", [0.0, 200.0])
@pytest.mark.parametrize("form", ["strict", "fast", "fp32"])
@pytest.mark.parametrize("n", [(48, 37), (130, 96), (24, 19, 13)])
def test_order_of_kernels(n, form, re, charwise):
    from paper_1905_00182_gb300 import ibfsa as ib
    dim = len(n)
    vel = (0.1, 0.05, -0.05)
    spec = W.GridSpec(dim=dim, n=tuple(n) + (1,) * (3 - dim), lo=(-1.0,) * 3, hi=(1.0,) * 3,
                      gamma=1.4, Re=re, qinf=W.freestream(dim, 1.4, vel=vel), scheme=W.TENO5,
                      precision=W.FP32_PERTURB if form == "fp32" else W.FP64, charwise=charwise,
                      sponge_cells=3, sponge_sigma=2.0)
    states = [W.random_smooth_state(spec, seed=s, amp=2e-3, vel0=vel) for s in (51, 52)]
    dt, steps = 0.1 * min(spec.h), 4
    stream = torch.cuda.Stream()
    g = ib.Grid(spec, strict=form == "strict", stream=stream)

    def run(Q, how):
        torch.cuda.synchronize()
        g.set_state(Q)
        torch.cuda.synchronize()
        how()
        torch.cuda.synchronize()
        assert g.status() == 0
        return g.get_state().clone()

    def one_by_one():
        for _ in range(steps):
            g.rk3_step(dt, 1)
            torch.cuda.synchronize()

    want = [run(Q, one_by_one) for Q in states]
    g.set_state(states[0])  # the FP32 form's first stage on a new state rounds it once more
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        g.rk3_step(dt, steps)
    for Q, w in zip(states, want):
        assert torch.equal(run(Q, lambda: g.rk3_step(dt, steps)), w)
        assert torch.equal(run(Q, graph.replay), w)
    g.close()
