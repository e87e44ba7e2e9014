"""A pinned sweep kernel on a mesh too wide for the traces of the pinned number of directions in FP64: the wider arithmetics
take fewer directions a task.  Against the oracle; tolerances as for the other sweep tests, relative l2."""
import numpy as np
import pytest

from gpu_common import lib, oracle_problems, rel, spec2d, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("variant", [0, 1])
def test_four_directions_on_4096_columns(variant):
    torch = torch_cuda()
    B = lib()
    from oracle import transport as OT
    spec = spec2d([4096], [40], n_polar=4, n_azim=8, rx=2, ry=2)
    rs = np.random.RandomState(variant)
    ss, sa = np.exp(rs.uniform(0.0, 3.0, (1, 4))), rs.uniform(0.0, 0.5, (1, 4))
    gp = B.Problem(spec, ss, sa)
    gp.set_sweep_variant(variant, 4)
    op = oracle_problems(spec, ss, sa)[0]
    z = rs.standard_normal(gp.n_dof)
    w64, wdf = (torch.empty(gp.n_dof, dtype=torch.float64, device="cuda") for _ in range(2))
    w32 = torch.empty(gp.n_dof, device="cuda")
    gp.apply_op(to_dev(z), w64)
    gp.apply_op(to_dev(z), wdf, double_float=True)
    gp.apply_op(to_dev(z, torch.float32), w32)
    ref = OT.Atilde_apply(op, z)
    assert rel(w64.cpu().numpy(), ref) < 1e-13
    assert rel(wdf.cpu().numpy(), ref) < 1e-12
    assert rel(w32.cpu().numpy(), OT.Atilde_apply(op, z.astype(np.float32).astype(np.float64))) < 2e-5
