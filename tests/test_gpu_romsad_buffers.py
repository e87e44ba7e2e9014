"""romsad_apply keeps its work buffers from one call to the next: no allocation per call, and calls on several threads and
streams of one ROM have buffers of their own."""
import threading

import numpy as np
import pytest

from gpu_common import lib, rel, spec2d, to_dev, torch_cuda

pytestmark = pytest.mark.gpu


def _setup(n, rank=6, seed=1):
    B = lib()
    spec = spec2d([16] * n, [16] * n, n_polar=2, n_azim=8)
    rs = np.random.RandomState(seed)
    gp = B.Problem(spec, np.exp(rs.uniform(0.0, 3.0, (n, 4))), rs.uniform(0.1, 0.5, (n, 4)))
    ndir, ndof = 16, 16 * 16 * 4
    Q, _ = np.linalg.qr(rs.standard_normal((ndir * ndof, rank)))
    return B, gp, B.Rom.from_basis(gp, Q.T.reshape(rank, ndir, ndof).copy(), instance=0)


@pytest.mark.parametrize("dtype_name", ["float32", "float64"])
def test_second_call_allocates_nothing(dtype_name):
    torch = torch_cuda()
    from torch.profiler import ProfilerActivity, profile
    B, gp, rom = _setup(5)
    v = to_dev(np.random.RandomState(2).standard_normal(gp.n_dof), getattr(torch, dtype_name))
    z = torch.empty_like(v)
    rom.apply(gp, v, z)
    torch.cuda.synchronize()
    for _ in range(2):   # the first recording of a process may miss its calls
        with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as p:
            rom.apply(gp, v, z)
            torch.cuda.synchronize()
    names = [e.name for e in p.events()]
    if not any("LaunchKernel" in k for k in names):
        pytest.skip("the runtime's calls are not recorded here")
    assert not [k for k in names if "Malloc" in k or "cudaFree" in k]


def test_calls_on_two_threads_and_sizes():
    """One ROM, two problems of different batch sizes, each on a thread and stream of its own, against the same calls one
    after the other: the same kernels on the same inputs, so the same bits."""
    torch = torch_cuda()
    B, g1, rom = _setup(3)
    spec = spec2d([16] * 9, [16] * 9, n_polar=2, n_azim=8)
    rs = np.random.RandomState(3)
    g2 = B.Problem(spec, np.exp(rs.uniform(0.0, 3.0, (9, 4))), rs.uniform(0.1, 0.5, (9, 4)))
    work = []
    for gp in (g1, g2):
        v = to_dev(rs.standard_normal(gp.n_dof), torch.float32)
        want, got = torch.empty_like(v), torch.empty_like(v)
        rom.apply(gp, v, want)
        work.append((gp, v, want, got, torch.cuda.Stream()))
    torch.cuda.synchronize()
    bad = []

    def run(gp, v, want, got, st):
        for _ in range(20):
            got.fill_(0.0)
            torch.cuda.synchronize()
            rom.apply(gp, v, got, stream=st)
            if not torch.equal(got, want):
                bad.append(gp.n_dof)

    threads = [threading.Thread(target=run, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
