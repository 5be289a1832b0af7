"""Solves on lattices small enough for the one-launch iteration (small.cuh), in
every operator and storage: the FP64 residual of the returned solution, taken
by the library's own FP64 operators (pinned to the oracle elsewhere), and a
batch against each of its systems alone, bit for bit.

The lattices are those where the blocks can go wrong: fewer sites than a warp
holds, half lattices that end in a partial group of 16 (every extent 2 mod 4), a
partial last block, one block, and the largest volumes that take this path
(Wilson 29184 sites, staggered Wilson 14592 with 152 SMs).
"""
import pytest

import lattice_synth as ls

pytestmark = pytest.mark.gpu

TOL = 1e-9
OPS = {"sw": 0, "wilson": 1, "wilson_eo": 2}


@pytest.fixture(scope="module")
def sw():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1312_3265_gb300 as m
    m.lib()
    return m


def residual(sw, op, dims, U, W, chi, x, m, r, apbc):
    import torch

    def D(v, dag):
        o = torch.empty_like(v)
        if op == "sw":
            sw.sw_dslash_apply(dims, U, W, v, o, m, r, dag, apbc)
        else:
            sw.wilson_dslash_apply(dims, U, v, o, m, r, dag, apbc)
        return o

    b = D(chi, True)
    return ((b - D(D(x, False), True)).norm() / b.norm()).item()


@pytest.mark.parametrize("op,prec", [("sw", 1), ("sw", 2), ("wilson", 1), ("wilson", 2), ("wilson_eo", 1)])
@pytest.mark.parametrize("dims,r,nsys", [((2, 2, 2, 2), 1.0, 3), ((2, 6, 2, 6), 0.75, 1), ((6, 6, 6, 6), 1.0, 5),
                                         ((4, 6, 10, 2), 0.75, 4), ((8, 8, 8, 28), 1.0, 2),
                                         ((12, 12, 12, 16), 1.0, 3)])
def test_small_lattice_solves(sw, op, prec, dims, r, nsys):
    import torch
    g = torch.Generator("cuda").manual_seed(7)
    V = ls.volume(dims)
    apbc = dims[3] % 4 == 2
    if V <= 4096:
        U = torch.from_numpy(ls.su3_links(dims, 5, ls.PLAQ_EPS)).cuda()
    else:  # SU(3): unitary factor of a Gaussian near 1, its determinant's phase divided out
        z = torch.eye(3, dtype=torch.complex128, device="cuda") + 0.3 * torch.randn(
            (V * 4, 3, 3), dtype=torch.complex128, device="cuda", generator=g)
        Q, R = torch.linalg.qr(z)
        d = torch.diagonal(R, dim1=-2, dim2=-1)
        Q = Q * (d / d.abs())[:, None, :]
        U = (Q / torch.linalg.det(Q)[:, None, None] ** (1.0 / 3.0)).reshape(V, 4, 3, 3).contiguous()
    W = None
    inner = (3,) if op == "sw" else (4, 3)
    if op == "sw":
        W = torch.empty((V, 8, 3, 3), dtype=torch.complex128, device="cuda")
        sw.sw_hypercube_build(dims, U, W, apbc)
    chi = torch.randn((nsys, V) + inner, dtype=torch.complex128, device="cuda", generator=g)
    masses = [0.1 + 0.15 * k for k in range(nsys)]  # they stop at different iterations
    x = torch.zeros_like(chi)
    rc, infos = sw.cgne_solve_batch(dims, OPS[op], U, W, chi, x, masses, r, TOL, 5000, prec, apbc)
    assert rc == sw.SW_OK
    for k, m in enumerate(masses):
        assert residual(sw, op, dims, U, W, chi[k], x[k], m, r, apbc) <= 1.01 * TOL
        if k in (0, nsys - 1):
            one = torch.zeros_like(chi[k])
            info = sw.cgne_solve(dims, OPS[op], U, W, chi[k].contiguous(), one, m, r, TOL, 5000, prec, apbc)
            assert info.iters == infos[k].iters and torch.equal(one, x[k])
