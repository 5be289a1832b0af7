"""The solves' general path -- a launch per kernel, chunks of iterations, CUDA
graphs, reliable updates on a side stream -- on lattices just above those that
take the one-launch iterations (with 152 SMs: Wilson 29184 sites, staggered
Wilson 14592), and the autotuners, which time that path on any lattice.  The
number of launches shows that it ran.
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


class Batch:
    """A gauge field and nsys Gaussian sources, all from the seed."""

    def __init__(self, sw, op, dims, nsys, seed, apbc=False):
        import torch
        g = torch.Generator("cuda").manual_seed(seed)
        V = ls.volume(dims)
        # SU(3): unitary factor of a Gaussian near 1, its determinant's phase divided out
        z = torch.eye(3, dtype=torch.complex128, device="cuda") + 0.3 * torch.randn(
            (V * 4, 3, 3), dtype=torch.complex128, device="cuda", generator=g)
        Q, R = torch.linalg.qr(z)
        d = torch.diagonal(R, dim1=-2, dim2=-1)
        Q = Q * (d / d.abs())[:, None, :]
        self.sw, self.op, self.dims, self.apbc = sw, op, dims, apbc
        self.U = (Q / torch.linalg.det(Q)[:, None, None] ** (1.0 / 3.0)).reshape(V, 4, 3, 3).contiguous()
        self.W = None
        if op == "sw":
            self.W = torch.empty((V, 8, 3, 3), dtype=torch.complex128, device="cuda")
            sw.sw_hypercube_build(dims, self.U, self.W, apbc)
        self.chi = torch.randn((nsys, V) + ((3,) if op == "sw" else (4, 3)), dtype=torch.complex128, device="cuda",
                               generator=g)

    def solve(self, masses, prec, r=1.0, tol=1e-9, max_iter=5000):
        """(solutions, infos, launches) of the batch."""
        import torch
        x = torch.zeros_like(self.chi)
        before = self.sw.sw_kernel_launches()
        rc, infos = self.sw.cgne_solve_batch(self.dims, OPS[self.op], self.U, self.W, self.chi, x, masses, r, tol,
                                             max_iter, prec, self.apbc)
        assert rc == self.sw.SW_OK
        return x, infos, self.sw.sw_kernel_launches() - before

    def residual(self, x, k, m, r=1.0):
        """The FP64 residual of system k, by the library's FP64 operators (pinned to the oracle elsewhere)."""
        import torch

        def D(v, dag):
            o = torch.empty_like(v)
            if self.op == "sw":
                self.sw.sw_dslash_apply(self.dims, self.U, self.W, v, o, m, r, dag, self.apbc)
            else:
                self.sw.wilson_dslash_apply(self.dims, self.U, v, o, m, r, dag, self.apbc)
            return o

        b = D(self.chi[k], True)
        return ((b - D(D(x[k], False), True)).norm() / b.norm()).item()


class param:
    """Process-wide tunables set for a block."""

    def __init__(self, sw, **kv):
        self.sw, self.kv = sw, {getattr(sw, "SW_PARAM_" + k): v for k, v in kv.items()}

    def __enter__(self):
        self.old = {k: self.sw.sw_get_param(k) for k in self.kv}
        for k, v in self.kv.items():
            self.sw.sw_set_param(k, v)

    def __exit__(self, *_):
        for k, v in self.old.items():
            self.sw.sw_set_param(k, v)


@pytest.mark.parametrize("op", ["sw", "wilson"])
@pytest.mark.parametrize("prec", [1, 2])
def test_autotuners_time_the_kernels_they_tune(sw, op, prec):
    b = Batch(sw, op, (4, 4, 4, 8), 1, 2)
    iters = 24
    with param(sw, NS_SW=2, NS_WILSON=1, SITE_BLOCKING=0):
        before = sw.sw_kernel_launches()
        sw.sw_autotune(b.dims, OPS[op], b.U, b.W, 5, prec, iters=iters)
        one = sw.sw_kernel_launches() - before
        sw.sw_autotune_layout(b.dims, OPS[op], b.U, b.W, 5, prec, iters=iters)
        layout = sw.sw_kernel_launches() - before - one
    # three launches an iteration, two solves a candidate
    assert one >= 3 * 2 * 3 * iters and layout >= 3 * sw.SW_SITE_SHAPES * 2 * 3 * iters
