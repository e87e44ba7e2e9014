"""Mixed solves to a relative residual of 1e-12 on meshes of 256^2 with scattering up to 1e4, where the fluxes are thousands of
times the source: the certifying FP64 residual has to round well below that.  Draws in which one instance of 16 stalled at
2e-12 to 4e-12 while the partial fluxes of an apply were added up in one chain."""
import numpy as np
import pytest

from gpu_common import lib, spec2d, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("seed", [41, 42, 57])
def test_every_instance_reaches_1e12(seed):
    torch = torch_cuda()
    B = lib()
    n, R = 16, 64
    rs = np.random.RandomState(seed)
    ss, sa = np.exp(rs.uniform(0.0, np.log(1e4), (n, R))), rs.uniform(0.0, 1.0, (n, R))
    spec = spec2d([256] * n, [256] * n, n_polar=8, n_azim=24, rx=8, ry=8, src_q=1.0, src_box=(0.4, 0.6, 0.4, 0.6), inflow_g=0.0)
    gp = B.Problem(spec, ss, sa)
    phi = torch.zeros(gp.n_dof, dtype=torch.float64, device="cuda")
    st = B.fgmres_solve(gp, None, phi, restart=40, rtol=1e-12, max_iter=400, post_mode=B.RTE_POST_DSA, mode=B.RTE_MODE_MIXED,
                        inner_rtol=1e-3, max_outer=30, raise_on_fail=False)
    assert [s["status"] for s in st] == [0] * n
