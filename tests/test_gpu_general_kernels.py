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
        # SU(3) near 1: two rows by Gram-Schmidt, the third the conjugate of their cross product
        z = torch.eye(3, dtype=torch.complex128, device="cuda") + 0.3 * torch.randn(
            (V, 4, 3, 3), dtype=torch.complex128, device="cuda", generator=g)
        u = z[..., 0, :] / z[..., 0, :].norm(dim=-1, keepdim=True)
        v = z[..., 1, :] - (z[..., 1, :] * u.conj()).sum(-1, keepdim=True) * u
        v = v / v.norm(dim=-1, keepdim=True)
        self.sw, self.op, self.dims, self.apbc = sw, op, dims, apbc
        self.U = torch.stack([u, v, torch.linalg.cross(u, v).conj()], dim=-2).contiguous()
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


WILSON, SW, EO = (18, 14, 12, 10), (10, 12, 14, 10), (18, 16, 16, 14)  # 30240, 16800, 32256 sites (of a half)
MASSES = [0.05, 0.1, 0.2, 0.07, 0.3, 0.02, 0.15]


@pytest.mark.parametrize("op,dims", [("sw", SW), ("wilson", WILSON), ("wilson_eo", EO)])
def test_widths_and_orders(sw, op, dims):
    """Widths 1, 2 and 4 (7 systems: ragged groups) in two site orders and both
    grid orders solve the same systems; the grid order does not change a bit."""
    import torch
    b = Batch(sw, op, dims, 7, 3, apbc=True)
    for prec in ((1,) if op == "wilson_eo" else (1, 2)):
        for width in (1, 2, 4):
            for blocking in ((0,) if op == "wilson_eo" else (0, 1 + width)):
                out = []
                for gfast in (0, 1):
                    with param(sw, NS_SW=width, NS_WILSON=width, SITE_BLOCKING=blocking, GROUP_FAST=gfast):
                        x, infos, launches = b.solve(MASSES, prec)
                    assert launches > 3 * max(i.iters for i in infos)
                    out.append(x)
                    for k in (0, 3, 6):
                        assert b.residual(x, k, MASSES[k]) <= 1.01e-9
                assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("op,dims,prec", [("sw", SW, 1), ("sw", SW, 2), ("wilson", WILSON, 1), ("wilson", WILSON, 2),
                                          ("wilson_eo", EO, 1), ("sw", SW, 0), ("wilson", WILSON, 0)])
def test_graphs_and_device_driven_rounds_are_bitwise_launches(sw, op, dims, prec):
    """Chunks as graphs, updates on the side stream, and the whole solve as one
    graph, on a stream that can be captured, against launches one by one."""
    import torch
    b = Batch(sw, op, dims, 3, 4, apbc=True)
    masses = [0.05, 0.1, 0.2]
    torch.cuda.synchronize()
    ref = None
    with torch.cuda.stream(torch.cuda.Stream()):
        for graphs, persistent in ((0, 0), (1, 0), (1, 1)):
            with param(sw, GRAPHS=graphs, PERSISTENT=persistent):
                x, infos, launches = b.solve(masses, prec)
            torch.cuda.synchronize()
            assert launches > 3 * max(i.iters for i in infos) > 3 * 16
            got = [(i.iters, i.reliable_updates) for i in infos]
            ref = (x, got) if ref is None else ref
            assert got == ref[1] and torch.equal(x, ref[0])


def test_wilson_lean_and_default_forms(sw):
    import torch
    b = Batch(sw, "wilson", WILSON, 5, 5, apbc=True)
    out = []
    for form in (0, 1):
        with param(sw, WILSON_LEAN=form):
            out.append(b.solve(MASSES[:5], 1))
    assert [i.iters for i in out[0][1]] == [i.iters for i in out[1][1]]
    assert torch.equal(out[0][0], out[1][0])


@pytest.mark.parametrize("op,dims,prec", [("sw", SW, 1), ("sw", SW, 2), ("wilson", WILSON, 1), ("wilson", WILSON, 2),
                                          ("wilson_eo", EO, 1)])
def test_other_wilson_parameters(sw, op, dims, prec):
    b = Batch(sw, op, dims, 3, 6)
    for r in (0.75, 1.3):
        x, infos, launches = b.solve(MASSES[:3], prec, r=r)
        assert launches > 3 * max(i.iters for i in infos)
        for k in range(3):
            assert b.residual(x, k, MASSES[k], r) <= 1.01e-9


@pytest.mark.parametrize("op,dims,nsys,prec,r,kw", [
    ("wilson", WILSON, 9, 1, 1.0, dict(NS_WILSON=4)), ("wilson", WILSON, 7, 1, 0.75, dict(NS_WILSON=2, GROUP_FAST=1)),
    ("wilson", WILSON, 8, 2, 0.75, dict(SITE_BLOCKING=4)), ("wilson", WILSON, 9, 1, 1.0, dict(SITE_BLOCKING=2)),
    ("sw", (18, 14, 16, 16), 13, 1, 1.0, dict(NS_SW=4)), ("sw", (18, 14, 16, 16), 13, 2, 1.3, dict(GROUP_FAST=1)),
    ("sw", (18, 14, 16, 16), 12, 1, 0.75, dict(SITE_BLOCKING=5, NS_SW=1)), ("wilson_eo", EO, 7, 1, 0.75, {}),
    ("wilson", WILSON, 3, 0, 0.75, {}), ("wilson_eo", EO, 3, 0, 1.0, {}), ("sw", SW, 5, 0, 1.3, {})])
def test_halves_in_every_layout(sw, op, dims, nsys, prec, r, kw):
    """Chunks as two halves: twice the launches, the same bits as every system alone."""
    import torch
    b = Batch(sw, op, dims, nsys, 8, apbc=True)
    masses = [0.1 + 0.01 * (k % 5) for k in range(nsys)]
    with param(sw, **kw), torch.cuda.stream(torch.cuda.Stream()):
        torch.cuda.synchronize()
        x, infos, launches = b.solve(masses, prec, r=r)
        assert launches > 5 * max(i.iters for i in infos)
        for k, m in enumerate(masses):
            one = torch.zeros_like(b.chi[k])
            info = sw.cgne_solve(dims, OPS[op], b.U, b.W, b.chi[k].contiguous(), one, m, r, 1e-9, 5000, prec, True)
            assert info.iters == infos[k].iters and torch.equal(one, x[k])
        torch.cuda.synchronize()


@pytest.mark.parametrize("op,dims,prec", [("sw", SW, 1), ("wilson", WILSON, 1), ("wilson", WILSON, 2),
                                          ("sw", SW, 0)])
def test_server_engines(sw, op, dims, prec):
    """Requests that join while others run, more of them than slots, against single solves."""
    import torch
    n = 9
    b = Batch(sw, op, dims, n, 9, apbc=True)
    torch.cuda.synchronize()  # the engine copies U on a stream of its own
    srv = sw.Server(8 << 30)
    try:
        e = srv.add_engine(dims, OPS[op], b.U, precision=prec, slots=5, t_antiperiodic=True)
        chi = b.chi.cpu().pin_memory()
        x = torch.zeros_like(chi).pin_memory()
        masses = [0.05 + 0.03 * ((5 * k) % n) for k in range(n)]
        ids = {srv.submit(e, chi[k], x[k], m, 1e-9): k for k, m in enumerate(masses)}
        srv.drain(120)
        done = srv.poll()
        assert len(done) == n
        for rid, info in done:
            k = ids[rid]
            one = torch.zeros_like(b.chi[k])
            ref = sw.cgne_solve(dims, OPS[op], b.U, b.W, b.chi[k].contiguous(), one, masses[k], 1.0, 1e-9, 100000,
                                prec, True)
            assert info.iters == ref.iters and torch.equal(one.cpu(), x[k])
    finally:
        srv.close()


@pytest.mark.parametrize("persistent", [0, 1])
def test_a_system_resumes_within_a_long_chunk(sw, persistent):
    """Two systems, chunks of 64 iterations: the heavy one's update runs beside the
    second chunk, in which it goes on to its end, while the light one runs to its
    iteration limit of 128.  Two chunks, then, and on the device a third round for
    the last updates; a system that resumed only with the next chunk takes one more."""
    import torch
    b = Batch(sw, "wilson", WILSON, 2, 3)
    V = ls.volume(WILSON)
    b.U = torch.eye(3, dtype=torch.complex128, device="cuda").expand(V, 4, 3, 3).contiguous()  # free: slow at mass 0.01
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()), param(sw, CHUNK=64, PERSISTENT=persistent):
        x = torch.zeros_like(b.chi)
        before = sw.sw_kernel_launches()
        rc, infos = sw.cgne_solve_batch(b.dims, 1, b.U, None, b.chi, x, [6.0, 0.01], 1.0, 1e-10, 128, 1)
        launches = sw.sw_kernel_launches() - before
        torch.cuda.synchronize()
    assert infos[0].status == sw.SW_OK and infos[0].iters < 40
    assert infos[1].status == sw.SW_NOT_CONVERGED and infos[1].iters == 128
    assert launches < 3.9 * 64 * 3
