"""The plate's step of a coupled step runs beside the fluid's last stage, and in line while kernel timing
is on.  In the strict form, whose sums have one order, both schedules, the same steps one call and one
synchronisation at a time, and a captured graph of them replayed twice give the same bits of fluid, penalty
integral and plate.
"""
import pytest

from oracle import oracle as O
from paper_1905_00182_gb300 import workloads as W
from tests.test_gpu_plate import _coupled_case

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,scheme", [((96, 64), W.TENO5), ((61, 47), W.WENO5JS)])
def test_schedules_give_the_same_bits(n, scheme):
    from paper_1905_00182_gb300 import ibfsa as ib
    spec, ps, Q, e, v, dt = _coupled_case(n=n, scheme=scheme)
    steps = 4
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):  # the copies that set the state are the stream's own
        g, p = ib.Grid(spec, strict=True, stream=stream), ib.Plate(ps, stream=stream)
        X, U, dS = O.plate_markers(ps, e, v)

        def start():
            g.set_state(Q)
            g.set_markers(X, U, dS)
            g.set_time(0.0)
            p.set_state(e, v, 0.0)
            torch.cuda.synchronize()

        def run(how):
            start()
            how()
            torch.cuda.synchronize()
            assert g.status() == 0 and p.status()[0] == 0
            return [t.clone() for t in (g.get_state(), g.penalty_integral(), *p.get_state()[:2])]

        def one_by_one():
            for _ in range(steps):
                ib.fsi_step(g, p, dt, 1)
                torch.cuda.synchronize()

        def in_line():
            ib.ibfsa_profile_enable(g.h, 1)
            ib.fsi_step(g, p, dt, steps)
            ib.ibfsa_profile_enable(g.h, 0)

        want = run(one_by_one)
        assert (want[2].cpu().numpy() != e).any()  # the plate moved
        start()
        graph = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        ib.fsi_step(g, p, dt, steps)
    with torch.cuda.stream(stream):
        for how in (in_line, lambda: ib.fsi_step(g, p, dt, steps), graph.replay, graph.replay):
            for a, b in zip(run(how), want):
                assert torch.equal(a, b)
        g.close()
        p.close()
