"""Batches whose chunks of iterations run as two halves on two streams: every
system against its solve alone (never split), bit for bit.

The batches are just above and below the work from which chunks split (2^21
complex numbers in a vector of the running systems, FP64 mode 2^14), with odd numbers of systems
and masses far apart, so that the halves empty at different times and the chunk
falls back to a whole one on the way.
"""
import pytest

import lattice_synth as ls

pytestmark = pytest.mark.gpu

OPS = {"sw": 0, "wilson": 1, "wilson_eo": 2}


@pytest.fixture(scope="module")
def sw():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1312_3265_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("op,prec,dims,nsys", [
    ("wilson", 1, (12, 12, 12, 24), 4), ("wilson", 1, (12, 12, 12, 24), 5), ("wilson", 2, (12, 12, 12, 24), 7),
    ("wilson_eo", 1, (14, 14, 14, 26), 5), ("sw", 1, (16, 16, 16, 16), 11), ("sw", 2, (14, 16, 16, 18), 13),
    ("wilson", 0, (4, 4, 6, 8), 2), ("wilson", 0, (6, 6, 6, 6), 2), ("wilson", 0, (48, 48, 10, 6), 3),
    ("wilson_eo", 0, (6, 6, 6, 6), 5), ("sw", 0, (4, 6, 8, 10), 3), ("sw", 0, (6, 6, 10, 10), 7)])
def test_halves_equal_single_solves(sw, op, prec, dims, nsys):
    import torch
    g = torch.Generator("cuda").manual_seed(11)
    V = ls.volume(dims)
    # SU(3): unitary factor of a Gaussian near 1, its determinant's phase divided out
    z = torch.eye(3, dtype=torch.complex128, device="cuda") + 0.2 * torch.randn(
        (V * 4, 3, 3), dtype=torch.complex128, device="cuda", generator=g)
    Q, R = torch.linalg.qr(z)
    d = torch.diagonal(R, dim1=-2, dim2=-1)
    Q = Q * (d / d.abs())[:, None, :]
    U = (Q / torch.linalg.det(Q)[:, None, None] ** (1.0 / 3.0)).reshape(V, 4, 3, 3).contiguous()
    W = None
    if op == "sw":
        W = torch.empty((V, 8, 3, 3), dtype=torch.complex128, device="cuda")
        sw.sw_hypercube_build(dims, U, W, False)
    chi = torch.randn((nsys, V) + ((3,) if op == "sw" else (4, 3)), dtype=torch.complex128, device="cuda", generator=g)
    masses = [0.1 * 1.6 ** (k if k % 2 else -0.2 * k) for k in range(nsys)]
    x = torch.zeros_like(chi)
    rc, infos = sw.cgne_solve_batch(dims, OPS[op], U, W, chi, x, masses, 1.0, 1e-9, 5000, prec, False)
    assert rc == sw.SW_OK
    for k, m in enumerate(masses):
        one = torch.zeros_like(chi[k])
        info = sw.cgne_solve(dims, OPS[op], U, W, chi[k].contiguous(), one, m, 1.0, 1e-9, 5000, prec, False)
        assert info.iters == infos[k].iters and info.reliable_updates == infos[k].reliable_updates
        assert torch.equal(one, x[k])
