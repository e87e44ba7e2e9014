"""DSA V-cycle (csrc/dsa.cu) where its 32 x 16 tiles and its classes of cells end: meshes of one row, of part of a tile and
of a tile and a bit, blocks of one, two and many cells, one set of coefficients per cell, and vectors off the 16-byte
boundary.  The tolerance is that of the other V-cycle comparisons (5e-5 relative, FP32 set-up and cycle)."""
import numpy as np
import pytest

from gpu_common import lib, oracle_problems, rel, spec2d, split, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

CASES = {
    "slivers": ([9, 40, 1, 8], [9, 1, 24, 48], 1, 1),
    "tile_and_a_bit": ([36, 64, 72, 40], [20, 16, 40, 24], 1, 1),
    "one_cell_blocks": ([16], [16], 16, 16),
    "one_by_many_blocks": ([48], [32], 48, 2),
    "two_cell_blocks": ([64], [48], 32, 3),
    "few_regions": ([64, 32], [32, 64], 4, 2),
}


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("name", list(CASES))
def test_vcycle_matches_oracle_at_tile_and_class_edges(name, dtype):
    torch = torch_cuda()
    B = lib()
    from oracle import dsa as ODSA
    nx, ny, rx, ry = CASES[name]
    spec = spec2d(nx, ny, n_polar=2, n_azim=8, rx=rx, ry=ry)
    rs = np.random.RandomState(len(name))
    ss, sa = np.exp(rs.uniform(np.log(5.0), np.log(50.0), (len(nx), rx * ry))), rs.uniform(0.05, 0.5, (len(nx), rx * ry))
    gp = B.Problem(spec, ss, sa)
    tdt = torch.float64 if dtype == "f64" else torch.float32
    v = to_dev(rs.standard_normal(gp.n_dof), tdt)
    z = torch.empty_like(v)
    gp.dsa_apply(v, z)
    off = torch.empty(gp.n_dof + 1, dtype=tdt, device="cuda")
    off[1:] = v
    z1 = torch.empty_like(off)
    gp.dsa_apply(off[1:], z1[1:])
    assert rel(z1[1:].cpu().numpy(), z.cpu().numpy()) < 1e-6
    zg, vv = z.double().cpu().numpy(), v.double().cpu().numpy()
    for b, op in enumerate(oracle_problems(spec, ss, sa)):
        vb = split(vv, gp.offsets)[b]
        assert rel(split(zg, gp.offsets)[b] - vb, ODSA.MultigridDsa(op, "partial").apply(vb) - vb) < 5e-5, b
