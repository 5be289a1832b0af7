"""A request that reaches a busy server engine on a small lattice does not wait
for the running systems' legs to end: its launches are short where a group of
blocks holds many systems."""
import time

import pytest

import lattice_synth as ls

pytestmark = pytest.mark.gpu


def test_request_beside_long_solves():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1312_3265_gb300 as sw
    dims, slots = (12, 12, 12, 12), 41
    V = ls.volume(dims)
    U = torch.eye(3, dtype=torch.complex128, device="cuda").expand(V, 4, 3, 3).contiguous()
    g = torch.Generator("cuda").manual_seed(2)
    chi = torch.randn((V, 4, 3), dtype=torch.complex128, device="cuda", generator=g).cpu().pin_memory()
    x = torch.zeros((slots, V, 4, 3), dtype=torch.complex128).pin_memory()
    torch.cuda.synchronize()
    srv = sw.Server(16 << 30)
    try:
        e = srv.add_engine(dims, sw.SW_OP_WILSON, U, slots=slots)
        srv.submit(e, chi, x[0], 2.0, 1e-6)  # the engine's first launches
        srv.drain(60)
        srv.poll()
        # free links and a small mass: hundreds of iterations in two legs
        slow = {srv.submit(e, chi, x[k], 0.02, 1e-8) for k in range(slots - 1)}
        time.sleep(0.02)  # they run
        quick = srv.submit(e, chi, x[slots - 1], 2.0, 1e-6)
        srv.drain(120)
        done = dict(srv.poll())
    finally:
        srv.close()
    assert all(done[k].status == sw.SW_OK for k in slow | {quick})
    assert min(done[k].iters for k in slow) > 150
    # a launch of their iterations up to the leg's end would take half of their time
    assert done[quick].seconds < 0.25 * min(done[k].seconds for k in slow)
