"""More than 2^28 markers in 3D: 16 lanes each are more threads than 32 bits count.  All markers lie at one of
a few positions, so that every marker's penalty force (arXiv:1905.00182, Eq. 7-8) is, to the bit, the one of
the same position among the first markers, which a grid of these alone gives as well.
"""
import pytest

from paper_1905_00182_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

FEW = 1 << 12


@pytest.mark.parametrize("precision", [W.FP64, W.FP32_PERTURB])
def test_more_markers_than_threads_in_32_bits(precision):
    from paper_1905_00182_gb300 import ibfsa as ib
    nm = (1 << 28) + 37
    if torch.cuda.mem_get_info()[0] < 300 * nm:  # 152 bytes a marker in the workspace
        pytest.skip("not enough device memory")
    spec = W.GridSpec(dim=3, n=(64, 60, 56), lo=(-1.0,) * 3, hi=(1.0,) * 3, gamma=1.4, Re=0.0,
                      qinf=W.freestream(3, 1.4), scheme=W.TENO5, precision=precision)
    spec.alpha_pen, spec.beta_pen = -3.0, -2.0
    Q = W.random_smooth_state(spec, seed=31, amp=2e-3)
    pos = torch.from_numpy(1.5 * W.splitmix64(41, 3 * FEW).reshape(3, FEW) - 0.75).cuda()
    few = torch.zeros(3, FEW, dtype=torch.float64, device="cuda")

    def forces(n):
        spec.max_markers = n
        at = torch.arange(n, device="cuda") % FEW
        g = ib.Grid(spec)
        g.set_state(Q)
        g.set_markers(pos[:, at], few[:, at], torch.zeros(n, dtype=torch.float64, device="cuda"))
        g.rhs()
        F = g.marker_forces()
        assert g.status() == 0
        g.close()
        return F

    want = forces(FEW)
    assert (want != 0.0).all()
    F = forces(nm)
    for a in range(3):
        full = F[a, : nm // FEW * FEW].view(-1, FEW)
        assert (full == want[a]).all()
        assert torch.equal(F[a, nm // FEW * FEW:], want[a, : nm % FEW])
    del F
    torch.cuda.empty_cache()
