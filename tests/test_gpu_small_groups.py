"""The one-launch iterations of small lattices (small.cuh) with many systems in a
group of blocks: more than two a warp of a block, those that stop first (heavy
masses) at the front of the batch, so that every warp's first systems have
stopped while most of the group runs on; and more systems than the groups
resident at once hold, so that a round takes several launches.  Every system is
compared bit for bit with its solve alone, and the batch with itself.
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


def su3_field(V, g):
    """SU(3): unitary factor of a Gaussian near 1, its determinant's phase divided out."""
    import torch
    z = torch.eye(3, dtype=torch.complex128, device="cuda") + 0.3 * torch.randn(
        (V * 4, 3, 3), dtype=torch.complex128, device="cuda", generator=g)
    Q, R = torch.linalg.qr(z)
    d = torch.diagonal(R, dim1=-2, dim2=-1)
    Q = Q * (d / d.abs())[:, None, :]
    return (Q / torch.linalg.det(Q)[:, None, None] ** (1.0 / 3.0)).reshape(V, 4, 3, 3).contiguous()


# with 152 SMs: 6 warps a block and 2 groups; 12 warps, one group, two launches
# (70 systems); 9 warps, one group; staggered Wilson 6 warps, 3 groups; 12 warps,
# one group, two launches
@pytest.mark.parametrize("op,prec,dims,nsys", [
    ("wilson", 1, (6, 10, 12, 14), 48), ("wilson", 2, (6, 10, 12, 14), 48), ("wilson", 1, (12, 12, 12, 16), 70),
    ("wilson_eo", 1, (12, 12, 12, 24), 40), ("sw", 1, (8, 8, 8, 8), 61), ("sw", 2, (8, 8, 8, 8), 61),
    ("sw", 1, (8, 8, 8, 28), 75)])
def test_many_systems_a_group(sw, op, prec, dims, nsys):
    import torch
    g = torch.Generator("cuda").manual_seed(17)
    V = ls.volume(dims)
    U = su3_field(V, g)
    W = None
    if op == "sw":
        W = torch.empty((V, 8, 3, 3), dtype=torch.complex128, device="cuda")
        sw.sw_hypercube_build(dims, U, W, False)
    chi = torch.randn((nsys, V) + ((3,) if op == "sw" else (4, 3)), dtype=torch.complex128, device="cuda", generator=g)
    heavy = (nsys + 2) // 3
    masses = [4.0] * heavy + [0.1 + 0.2 * k / nsys for k in range(nsys - heavy)]
    ref = None
    for _ in range(3):
        x = torch.zeros_like(chi)
        rc, infos = sw.cgne_solve_batch(dims, OPS[op], U, W, chi, x, masses, 1.0, 1e-9, 5000, prec, False)
        assert rc == sw.SW_OK and all(i.true_rel_resid <= 1e-9 for i in infos)
        ref = x if ref is None else ref
        assert torch.equal(x, ref)
    assert max(i.iters for i in infos[:heavy]) < min(i.iters for i in infos[heavy:])
    for k, m in enumerate(masses):
        one = torch.zeros_like(chi[k])
        info = sw.cgne_solve(dims, OPS[op], U, W, chi[k].contiguous(), one, m, 1.0, 1e-9, 5000, prec, False)
        assert info.iters == infos[k].iters and info.reliable_updates == infos[k].reliable_updates
        assert torch.equal(one, x[k])


def test_long_lived_engine(sw):
    """A server engine that has run more launches of the small-lattice kernel
    than its inboxes keep epochs for (1024), with one group of blocks, then
    takes a burst of many groups: every result equals the solve's, bit for bit."""
    import torch
    dims, slots = (4, 4, 4, 4), 96
    V = ls.volume(dims)
    g = torch.Generator("cuda").manual_seed(5)
    U = su3_field(V, g)
    chi = torch.randn((slots, V, 4, 3), dtype=torch.complex128, device="cuda", generator=g).cpu().pin_memory()
    x = torch.zeros_like(chi).pin_memory()
    srv = sw.Server(4 << 30)
    try:
        e = srv.add_engine(dims, sw.SW_OP_WILSON, U, slots=slots)
        for i in range(1100):  # each takes a launch at least
            srv.submit(e, chi[0], x[0], 4.0, 1e-2)
            srv.drain()
            (_, info), = srv.poll()
            assert info.status == sw.SW_OK
        masses = [0.1 + 0.01 * k for k in range(slots)]
        ids = {srv.submit(e, chi[k], x[k], m, 1e-9): k for k, m in enumerate(masses)}
        srv.drain()
        for rid, info in srv.poll():
            k = ids[rid]
            one = torch.zeros((V, 4, 3), dtype=torch.complex128, device="cuda")
            ref = sw.cgne_solve(dims, sw.SW_OP_WILSON, U, None, chi[k].cuda(), one, masses[k], 1.0, 1e-9, 100000,
                                sw.SW_PREC_F32_RELIABLE)
            assert info.iters == ref.iters and torch.equal(one.cpu(), x[k])
    finally:
        srv.close()


@pytest.mark.parametrize("op,prec", [("sw", 1), ("sw", 2), ("wilson", 1), ("wilson_eo", 1)])
def test_a_wait_that_gives_up_is_a_timeout(sw, op, prec):
    """With one poll allowed, a wait for 100 other blocks runs out: the call
    returns SW_ERR_TIMEOUT at once, for every system of the batch and to a
    request of a server, and the next calls, with the default limit, solve."""
    import torch
    dims, nsys = (8, 8, 8, 16) if op != "wilson_eo" else (8, 8, 16, 16), 3
    V = ls.volume(dims)
    g = torch.Generator("cuda").manual_seed(3)
    U = su3_field(V, g)
    W = None
    if op == "sw":
        W = torch.empty((V, 8, 3, 3), dtype=torch.complex128, device="cuda")
        sw.sw_hypercube_build(dims, U, W, False)
    chi = torch.randn((nsys, V) + ((3,) if op == "sw" else (4, 3)), dtype=torch.complex128, device="cuda", generator=g)
    solve = lambda x: sw.cgne_solve_batch(dims, OPS[op], U, W, chi, x, [0.2, 0.3, 0.4], 1.0, 1e-9, 5000, prec, False)
    old = sw.sw_get_param(sw.SW_PARAM_WAIT_POLLS)
    srv = sw.Server(4 << 30)
    try:
        sw.sw_set_param(sw.SW_PARAM_WAIT_POLLS, 1)
        x = torch.zeros_like(chi)
        before = sw.sw_kernel_launches()
        with pytest.raises(sw.SWError) as e:
            solve(x)
        assert e.value.code == -7
        assert sw.sw_kernel_launches() - before < 40  # admission and one round
        if op != "wilson_eo":
            eng = srv.add_engine(dims, OPS[op], U, precision=prec, slots=2)
            ch, xh = chi[0].cpu().pin_memory(), torch.zeros_like(chi[0]).cpu().pin_memory()
            srv.submit(eng, ch, xh, 0.2, 1e-9)
            srv.drain(60)
            (_, info), = srv.poll()
            assert info.status == -7
    finally:
        sw.sw_set_param(sw.SW_PARAM_WAIT_POLLS, old)
        srv.close()
    x = torch.zeros_like(chi)
    rc, infos = solve(x)
    assert rc == sw.SW_OK and all(i.true_rel_resid <= 1e-9 for i in infos)


@pytest.mark.parametrize("op,dims,nsys,base", [("sw", (8, 8, 8, 8), 600, 3 * 64), ("wilson", (12, 12, 12, 16), 90, 12 * 64)])
def test_scratch_of_a_large_batch_stays_small(sw, op, dims, nsys, base):
    """The workspace of a batch on a small lattice is that of larger lattices (two
    FP64 vectors, p, t, r and x: `base` bytes a site and system, and the packed
    gauge field) and at most a fifth of it."""
    import torch
    g = torch.Generator("cuda").manual_seed(1)
    V = ls.volume(dims)
    U = su3_field(V, g)
    W = None
    if op == "sw":
        W = torch.empty((V, 8, 3, 3), dtype=torch.complex128, device="cuda")
        sw.sw_hypercube_build(dims, U, W, False)
    chi = torch.randn((nsys, V) + ((3,) if op == "sw" else (4, 3)), dtype=torch.complex128, device="cuda", generator=g)
    x = torch.zeros_like(chi)
    torch.cuda.synchronize()
    sw.sw_trim_workspace()
    held = sw.sw_workspace_reserved()
    rc, infos = sw.cgne_solve_batch(dims, OPS[op], U, W, chi, x, [0.5] * nsys, 1.0, 1e-6, 5000, 1, False)
    assert rc == sw.SW_OK and all(i.true_rel_resid <= 1e-6 for i in infos)
    used = sw.sw_workspace_reserved() - held
    assert used <= 1.2 * (base * V * nsys + 864 * V) + (32 << 20)  # (and the pool's granularity)
