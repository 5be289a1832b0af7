"""The inner operator of the one-launch iterations is as exact as the one of the
kernels of larger lattices: three CG iterations from zero in a mixed mode, on a
lattice just below and one just above the limit of the one-launch path, against
the same iterations in FP64.

Bound: both errors are averages over more than 80000 numbers (0.3%) of the same
distribution, and rounding each gauge matrix entry once more, or adding up
unscaled, shows as 8% (Wilson, r != 1) and 70% (staggered Wilson) of the
operator's own error; 2% over the other path's error lies between.
"""
import pytest

import lattice_synth as ls

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sw():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1312_3265_gb300 as m
    m.lib()
    return m


def cg_error(sw, op, dims, r, k=3, mass=0.3):
    import torch
    g = torch.Generator("cuda").manual_seed(13)
    V = ls.volume(dims)
    # random SU(3): two rows by Gram-Schmidt, the third the conjugate of their cross product
    z = torch.randn((V, 4, 2, 3), dtype=torch.complex128, device="cuda", generator=g)
    u = z[..., 0, :] / z[..., 0, :].norm(dim=-1, keepdim=True)
    v = z[..., 1, :] - (z[..., 1, :] * u.conj()).sum(-1, keepdim=True) * u
    v = v / v.norm(dim=-1, keepdim=True)
    U = torch.stack([u, v, torch.linalg.cross(u, v).conj()], dim=-2).contiguous()
    W = None
    if op == 0:
        W = torch.empty((V, 8, 3, 3), dtype=torch.complex128, device="cuda")
        sw.sw_hypercube_build(dims, U, W)
    chi = torch.randn((V, 3) if op == 0 else (V, 4, 3), dtype=torch.complex128, device="cuda", generator=g)

    def D(v, dag):
        o = torch.empty_like(v)
        if op == 0:
            sw.sw_dslash_apply(dims, U, W, v, o, mass, r, dag)
        else:
            sw.wilson_dslash_apply(dims, U, v, o, mass, r, dag)
        return o

    dot = lambda a: (a.real ** 2 + a.imag ** 2).sum()
    res = D(chi, True)
    p, ref, rr = res.clone(), torch.zeros_like(chi), dot(res)
    for _ in range(k):
        t = D(p, False)
        alpha = rr / dot(t)
        ref = ref + alpha * p
        res = res - alpha * D(t, True)
        new = dot(res)
        p, rr = res + (new / rr) * p, new
    x = torch.zeros_like(chi)
    info = sw.cgne_solve(dims, op, U, W, chi, x, mass, r, 1e-12, k, sw.SW_PREC_F32_RELIABLE)
    assert info.iters == k
    return ((x - ref).norm() / ref.norm()).item()


@pytest.mark.parametrize("op,below,above", [(0, (8, 8, 8, 28), (8, 8, 8, 30)), (1, (12, 12, 12, 16), (12, 12, 12, 18))])
@pytest.mark.parametrize("r", [1.0, 0.75, 1.3])
def test_operator_error_below_and_above_the_limit(sw, op, below, above, r):
    assert cg_error(sw, op, below, r) <= 1.02 * cg_error(sw, op, above, r)
