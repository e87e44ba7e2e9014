"""Slabs in batches large and small: a thread marches each chain of cells where there are many, a warp scans it where there
are few.  Applies, right-hand sides and angular sweeps of both against the oracle, on lengths that the lanes of a warp do and
do not divide.  Tolerances as for the other sweep tests: 1e-13 (FP64), 1e-12 (double-float), 2e-5 (FP32), relative l2."""
import dataclasses

import numpy as np
import pytest

from gpu_common import lib, oracle_problems, rel, spec1d, split, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,copies", [([4, 36, 128, 520], 1), ([4, 36, 128], 900), ([520], 2100)])
def test_slabs_match_oracle(nx, copies):
    torch = torch_cuda()
    B = lib()
    from oracle import transport as OT
    spec = dataclasses.replace(spec1d(nx * copies, n_polar=8), inflow_g=0.6)
    n = spec.n_instances
    rs = np.random.RandomState(n)
    ss, sa = np.exp(rs.uniform(0.0, np.log(100.0), (n, 4))), rs.uniform(0.0, 0.5, (n, 4))
    ss[0], sa[0] = 0.0, 0.0    # a void
    gp = B.Problem(spec, ss, sa)
    z = rs.standard_normal(gp.n_dof)
    z64, z32 = to_dev(z), to_dev(z, torch.float32)
    w64, wdf, b64, p64 = (torch.empty_like(z64) for _ in range(4))
    w32, p32 = torch.empty_like(z32), torch.empty_like(z32)
    gp.apply_op(z64, w64)
    gp.apply_op(z64, wdf, double_float=True)
    gp.apply_op(z32, w32)
    gp.rhs(b64)
    for v, p in ((z64, p64), (z32, p32)):
        psi = torch.empty(int(gp.info.n_angular_total), dtype=v.dtype, device="cuda")
        gp.sweep(v, psi)
        gp.scalar_flux(psi, p)
    host = {k: split(v.cpu().numpy().astype(np.float64), gp.offsets)
            for k, v in dict(w64=w64, wdf=wdf, w32=w32, b64=b64, p64=p64, p32=p32).items()}
    zr = z.astype(np.float32).astype(np.float64)
    for b in sorted({0, 1 % n, 2 % n, 3 % n, n // 2, n - 1}):
        op = oracle_problems(dataclasses.replace(spec, nx=[spec.nx[b]], ny=[1]), ss[b:b + 1], sa[b:b + 1])[0]
        zb, zrb = split(z, gp.offsets)[b], split(zr, gp.offsets)[b]
        ref = OT.Atilde_apply(op, zb)
        assert rel(host["w64"][b], ref) < 1e-13, b
        assert rel(host["wdf"][b], ref) < 1e-12, b
        assert rel(host["w32"][b], OT.Atilde_apply(op, zrb)) < 2e-5, b
        assert rel(host["b64"][b], OT.rhs_btilde(op)) < 1e-13, b
        assert rel(host["p64"][b], OT.T_apply(op, zb)) < 1e-13, b
        assert rel(host["p32"][b], OT.T_apply(op, zrb)) < 2e-5, b
