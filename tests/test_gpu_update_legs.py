"""How often a mixed-precision solve recomputes its residual in FP64: the legs
between the updates are equal and end at the tolerance, so a solve takes at
most one update more than the legs of the trigger's size that its tolerance
needs, in every operator and storage, from a zero guess and from a rough one;
and it stops at a true residual within the tolerance.
"""
import math

import pytest

import lattice_synth as ls

pytestmark = pytest.mark.gpu

OPS = {"sw": 0, "wilson": 1, "wilson_eo": 2}
DELTA = {1: 3e-5, 2: 1e-3}


@pytest.fixture(scope="module")
def sw():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1312_3265_gb300 as m
    m.lib()
    return m


@pytest.mark.parametrize("op,prec", [("sw", 1), ("sw", 2), ("wilson", 1), ("wilson", 2), ("wilson_eo", 1)])
@pytest.mark.parametrize("tol", [1e-3, 1e-6, 1e-8, 1e-10, 1e-12])
def test_update_counts(sw, op, prec, tol):
    import torch
    dims = (8, 6, 8, 8)
    V = ls.volume(dims)
    U = torch.from_numpy(ls.su3_links(dims, 5, ls.PLAQ_EPS)).cuda()
    W = None
    if op == "sw":
        W = torch.empty((V, 8, 3, 3), dtype=torch.complex128, device="cuda")
        sw.sw_hypercube_build(dims, U, W, False)
    g = torch.Generator("cuda").manual_seed(3)
    chi = torch.randn((3, V) + ((3,) if op == "sw" else (4, 3)), dtype=torch.complex128, device="cuda", generator=g)
    legs = math.ceil(math.log(tol) / math.log(DELTA[prec]))
    for guess in (0.0, 0.01):  # (a solve from a guess starts with an FP64 residual of its own)
        x = guess * chi
        rc, infos = sw.cgne_solve_batch(dims, OPS[op], U, W, chi, x, [0.1, 0.3, 0.6], 1.0, tol, 5000, prec, False)
        assert rc == sw.SW_OK
        for info in infos:
            assert info.true_rel_resid <= tol
            assert info.reliable_updates <= legs + 1 + (guess != 0.0)
