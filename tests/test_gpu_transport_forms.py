"""The two builds of the hypercube transports against each other.

sw_hypercube_build works through two-link sums held in a workspace (the whole
lattice, or slabs of time slices on lattices whose sums exceed it); a stream
that is being captured takes the kernel without a workspace.  Both compute W(x,s)
in FP64: an entry is 1/24 of the sum of 24 products of four unitary matrices,
each product a chain of at most 3 x 3 rounded complex multiply-adds on numbers
of magnitude at most 1, so each build is within 24/24 * 4 * 9 * u of the exact
value and the two are within 72 u (u = 2^-53) of each other.
"""
import pytest

import lattice_synth as ls

pytestmark = pytest.mark.gpu

BOUND = 72 * 2.0 ** -53


# extents of 2 (hops alias), ragged ones, one time slice pair, and a lattice
# built in slabs that do not divide its extent
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 2, 6, 2), (2, 6, 4, 10), (8, 8, 8, 8), (16, 18, 20, 30)])
def test_builds_agree(dims):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1312_3265_gb300 as sw
    V = ls.volume(dims)
    th = torch.randn((V * 4, 3, 3), dtype=torch.complex128, device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    U = torch.linalg.qr(th)[0].reshape(V, 4, 3, 3).contiguous()
    W = torch.full((V, 8, 3, 3), float("nan"), dtype=torch.complex128, device="cuda")
    C = torch.full_like(W, float("nan"))
    sw.sw_hypercube_build(dims, U, W)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        sw.sw_hypercube_build(dims, U, C)
    g.replay()
    torch.cuda.synchronize()
    assert (W - C).abs().max().item() <= BOUND
