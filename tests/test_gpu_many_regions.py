"""Operator applies of problems with more regions than the FP64 or double-float tables of a task have room for in shared
memory (they are read from global memory then), against the oracle.  Tolerances as for the other sweep tests: 1e-13 (FP64),
1e-12 (double-float), relative l2."""
import dataclasses

import numpy as np
import pytest

from gpu_common import lib, oracle_problems, rel, spec2d, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def _problem(B, n, regions, n_polar, n_azim):
    spec = dataclasses.replace(spec2d([n], [n], n_polar=n_polar, n_azim=n_azim, rx=regions, ry=regions), inflow_g=0.4,
                               inflow_faces=("x-", "y+"))
    rs = np.random.RandomState(n + n_polar)
    ss, sa = np.exp(rs.uniform(0.0, np.log(300.0), (1, regions**2))), rs.uniform(0.0, 0.5, (1, regions**2))
    return B.Problem(spec, ss, sa), oracle_problems(spec, ss, sa)[0], rs.standard_normal(4 * n * n)


@pytest.mark.parametrize("n,D", [(44, 1), (32, 2), (24, 4), (56, 1)])
def test_pinned(n, D):
    torch = torch_cuda()
    B = lib()
    from oracle import transport as OT
    gp, op, z = _problem(B, n, n, 2, 4 * D)
    gp.set_sweep_variant(0, D)
    w64, wdf, t64, b64 = (torch.empty(gp.n_dof, dtype=torch.float64, device="cuda") for _ in range(4))
    gp.apply_op(to_dev(z), w64)
    gp.apply_op(to_dev(z), wdf, double_float=True)
    gp.apply_T(to_dev(z), t64)
    gp.rhs(b64)
    ref = OT.Atilde_apply(op, z)
    assert rel(w64.cpu().numpy(), ref) < 1e-13
    assert rel(wdf.cpu().numpy(), ref) < 1e-12
    assert rel(t64.cpu().numpy(), OT.T_apply(op, z)) < 1e-13
    assert rel(b64.cpu().numpy(), OT.rhs_btilde(op)) < 1e-13


@pytest.mark.parametrize("n,regions,n_polar,n_azim", [(44, 44, 2, 4), (80, 40, 4, 48), (80, 40, 8, 48)])
def test_without_allocation(n, regions, n_polar, n_azim):
    """The fixed scratch asks for one, two and four directions a task."""
    torch = torch_cuda()
    B = lib()
    from oracle import transport as OT
    gp, op, z = _problem(B, n, regions, n_polar, n_azim)
    w = torch.empty(gp.n_dof, dtype=torch.float64, device="cuda")
    gp.apply_op_noalloc(to_dev(z), w)
    assert rel(w.cpu().numpy(), OT.Atilde_apply(op, z)) < 1e-13
