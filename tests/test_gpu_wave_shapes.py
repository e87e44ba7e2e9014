"""Every launch shape of the operator sweeps that is built, pinned one by one, against the oracle: meshes with more bands than
warps, fewer, and a last band of one row, quadrants of 15 directions (which no task of 2, 4, 8, 12 or 16 divides), inflow.
Tolerances as for the other sweep tests: 1e-13 (FP64), 1e-12 (double-float), 2e-5 (FP32), relative l2."""
import dataclasses
import functools

import numpy as np
import pytest

from gpu_common import lib, oracle_problems, rel, spec2d, split, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

NX = [33, 96, 12, 39]
NY = {1: [65, 97, 7, 300], 2: [66, 130, 8, 322]}   # rows a lane: two need an even number of rows in every region


@functools.lru_cache(maxsize=None)
def _case(rows):
    from oracle import transport as OT
    spec = dataclasses.replace(spec2d(NX, NY[rows], n_polar=6, n_azim=20, rx=3, ry=1), inflow_g=0.7, inflow_faces=("x-", "y+"))
    rs = np.random.RandomState(rows)
    ss, sa = np.exp(rs.uniform(0.0, np.log(300.0), (4, 3))), rs.uniform(0.0, 0.5, (4, 3))
    gp = lib().Problem(spec, ss, sa)
    z = rs.standard_normal(gp.n_dof)
    zr = z.astype(np.float32).astype(np.float64)
    ops = oracle_problems(spec, ss, sa)
    ref = [OT.Atilde_apply(op, v) for op, v in zip(ops, split(z, gp.offsets))]
    ref32 = [OT.Atilde_apply(op, v) for op, v in zip(ops, split(zr, gp.offsets))]
    return gp, z, ref, ref32, [OT.rhs_btilde(op) for op in ops]


@pytest.mark.parametrize("warps", [1, 2, 4, 8])
@pytest.mark.parametrize("arith,D,rows", [("f32", D, 1) for D in (1, 2, 4, 8, 12, 16)] + [("f32", 8, 2)] +
                         [("f64", D, 1) for D in (1, 2, 3, 4)] + [("df", D, 1) for D in (1, 2, 4)])
def test_shape_matches_oracle(arith, D, rows, warps):
    torch = torch_cuda()
    B = lib()
    gp, z, ref, ref32, rhs = _case(rows)
    code = {"f32": B.RTE_F32, "f64": B.RTE_F64, "df": B.RTE_F64_DF}[arith]
    gp.set_sweep_shape(code, D, warps, rows)
    try:
        v = to_dev(z, torch.float32 if arith == "f32" else torch.float64)
        w, b = torch.full_like(v, float("nan")), torch.full_like(v, float("nan"))
        gp.apply_op(v, w, double_float=arith == "df")
        if arith != "df":
            gp.rhs(b)
    finally:
        gp.set_sweep_shape(code, 0)
    tol = {"f32": 2e-5, "f64": 1e-13, "df": 1e-12}[arith]
    hw, hb = (split(x.cpu().numpy().astype(np.float64), gp.offsets) for x in (w, b))
    for k in range(4):
        assert rel(hw[k], (ref32 if arith == "f32" else ref)[k]) < tol, k
        if arith != "df":
            assert rel(hb[k], rhs[k]) < tol, k


def test_shapes_that_are_not_built_are_refused():
    B = lib()
    torch_cuda()
    gp = _case(1)[0]
    for code, D, warps, rows in ((B.RTE_F32, 3, 1, 1), (B.RTE_F64, 8, 1, 1), (B.RTE_F64_DF, 3, 1, 1), (B.RTE_F64, 1, 1, 2),
                                 (B.RTE_F32, 8, 1, 2), (B.RTE_F32, 1, 9, 1), (B.RTE_F32, 1, 1, 11)):
        with pytest.raises(B.RteError):
            gp.set_sweep_shape(code, D, warps, rows)   # (two rows a lane: the case has odd row counts)
