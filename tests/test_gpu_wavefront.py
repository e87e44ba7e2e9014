"""Operator sweeps (csrc/wavefront.cu) against the oracle where tiles, bands and direction chunks end: ragged meshes, one
cell, more bands than warps, a region per cell, direction counts that the chunk does not divide, inflow on the faces.
Tolerances as for the other sweep tests: 1e-13 (FP64), 1e-12 (double-float), 2e-5 (FP32), relative l2."""
import dataclasses

import numpy as np
import pytest

from gpu_common import lib, oracle_problems, rel, spec2d, split, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

CASES = {
    "one_cell_and_slivers": dict(nx=[1, 33, 7, 64], ny=[1, 65, 40, 1], n_polar=2, n_azim=4, rx=1, ry=1),
    "rows_past_two_bands": dict(nx=[31, 32, 34], ny=[97, 33, 32], n_polar=3, n_azim=6, rx=1, ry=1),
    "nine_bands": dict(nx=[40, 24], ny=[260, 300], n_polar=4, n_azim=8, rx=4, ry=2),
    "region_per_cell": dict(nx=[30], ny=[42], n_polar=2, n_azim=8, rx=30, ry=42),
    "odd_regions": dict(nx=[36, 60], ny=[33, 99], n_polar=4, n_azim=8, rx=12, ry=11),
    "twenty_four_per_quadrant": dict(nx=[48] * 24, ny=[64] * 24, n_polar=8, n_azim=24, rx=2, ry=2),
    "unequal_quadrants": dict(nx=[40] * 10, ny=[40] * 10, n_polar=6, n_azim=30, rx=4, ry=4),
    "two_rows_a_lane": dict(nx=[64] * 90, ny=[128] * 90, n_polar=4, n_azim=16, rx=2, ry=2),
}


@pytest.mark.parametrize("name", list(CASES))
def test_operator_sweeps_match_oracle(name):
    torch = torch_cuda()
    B = lib()
    from oracle import transport as OT
    spec = dataclasses.replace(spec2d(**CASES[name]), inflow_g=0.7, inflow_faces=("x-", "y+"))
    n, R = spec.n_instances, spec.n_regions
    rs = np.random.RandomState(len(name))
    ss, sa = np.exp(rs.uniform(0.0, np.log(300.0), (n, R))), rs.uniform(0.0, 0.5, (n, R))
    ss[0], sa[0, : max(1, R // 2)] = 0.0, 0.0          # a void and a pure absorber
    gp = B.Problem(spec, ss, sa)
    z = rs.standard_normal(gp.n_dof)
    w64, wdf, t64 = (torch.empty(gp.n_dof, dtype=torch.float64, device="cuda") for _ in range(3))
    b64, w32, b32 = torch.empty_like(w64), torch.empty_like(w64, dtype=torch.float32), torch.empty_like(w64, dtype=torch.float32)
    gp.apply_op(to_dev(z), w64)
    gp.apply_op(to_dev(z), wdf, double_float=True)
    gp.apply_op(to_dev(z, torch.float32), w32)
    gp.apply_T(to_dev(z), t64)
    gp.rhs(b64)
    gp.rhs(b32)
    host = {k: split(v.cpu().numpy().astype(np.float64), gp.offsets)
            for k, v in dict(w64=w64, wdf=wdf, w32=w32, t64=t64, b64=b64, b32=b32).items()}
    zr = z.astype(np.float32).astype(np.float64)
    for b in sorted({0, 1 % n, n // 2, n - 1}):        # a void first instance and some of the others
        op = oracle_problems(dataclasses.replace(spec, nx=[spec.nx[b]], ny=[spec.ny[b]]), ss[b:b + 1], sa[b:b + 1])[0]
        zb, zrb = split(z, gp.offsets)[b], split(zr, gp.offsets)[b]
        ref, rhs = OT.Atilde_apply(op, zb), OT.rhs_btilde(op)
        assert rel(host["w64"][b], ref) < 1e-13, b
        assert rel(host["wdf"][b], ref) < 1e-12, b
        assert rel(host["w32"][b], OT.Atilde_apply(op, zrb)) < 2e-5, b
        assert rel(host["t64"][b], OT.T_apply(op, zb)) < 1e-13, b
        assert rel(host["b64"][b], rhs) < 1e-13, b
        assert rel(host["b32"][b], rhs) < 2e-5, b


@pytest.mark.parametrize("D", [1, 2])
def test_columns_that_share_a_trace_slot_across_bands(D):
    """Two warps per task and rows a little longer than a multiple of 32: the next band's first columns take the slots
    of the last ones, which the other warp still has to read."""
    torch = torch_cuda()
    B = lib()
    from oracle import transport as OT
    spec = spec2d([97, 73, 100, 129, 96], [130, 160, 100, 97, 128], n_polar=2, n_azim=8, rx=1, ry=1)
    rs = np.random.RandomState(D)
    ss, sa = np.exp(rs.uniform(0.0, np.log(3.0), (5, 1))), rs.uniform(0.0, 0.1, (5, 1))
    gp = B.Problem(spec, ss, sa)
    gp.set_sweep_variant(2, D)
    ops = oracle_problems(spec, ss, sa)
    z = rs.standard_normal(gp.n_dof)
    w64, w32 = torch.empty(gp.n_dof, dtype=torch.float64, device="cuda"), torch.empty(gp.n_dof, device="cuda")
    wdf = torch.empty_like(w64)
    gp.apply_op(to_dev(z), w64)
    gp.apply_op(to_dev(z), wdf, double_float=True)
    gp.apply_op(to_dev(z, torch.float32), w32)
    for b, op in enumerate(ops):
        zb = split(z, gp.offsets)[b]
        ref, ref32 = OT.Atilde_apply(op, zb), OT.Atilde_apply(op, zb.astype(np.float32).astype(np.float64))
        assert rel(split(w64.cpu().numpy(), gp.offsets)[b], ref) < 1e-13, b
        assert rel(split(wdf.cpu().numpy(), gp.offsets)[b], ref) < 1e-12, b
        assert rel(split(w32.cpu().numpy().astype(np.float64), gp.offsets)[b], ref32) < 2e-5, b


@pytest.mark.parametrize("n,D", [(40, 1), (28, 2)])
def test_regions_beyond_the_legendre_tables(n, D):
    """A region per cell, more than the sixteen-entry tables of D directions hold in shared memory: FP64 applies with a
    task of D directions, chosen and without allocations."""
    torch = torch_cuda()
    B = lib()
    from oracle import transport as OT
    spec = spec2d([n], [n], n_polar=2, n_azim=4 * D, rx=n, ry=n)
    rs = np.random.RandomState(n)
    ss, sa = np.exp(rs.uniform(0.0, np.log(300.0), (1, n * n))), rs.uniform(0.0, 0.5, (1, n * n))
    op = oracle_problems(spec, ss, sa)[0]
    z = rs.standard_normal(4 * n * n)
    ref = OT.Atilde_apply(op, z)
    for how in ("pinned", "noalloc", "chosen"):
        gp = B.Problem(spec, ss, sa)
        w = torch.empty(gp.n_dof, dtype=torch.float64, device="cuda")
        if how == "pinned":
            gp.set_sweep_variant(0, D)
        (gp.apply_op_noalloc if how == "noalloc" else gp.apply_op)(to_dev(z), w)
        assert rel(w.cpu().numpy(), ref) < 1e-13, how
