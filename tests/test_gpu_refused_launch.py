"""Small lattices where the runtime refuses the cooperative launch (a fake of
the failing call, linked into a copy of the library): the solve goes on with the
kernels of larger lattices, from its start or from the middle, and meets its
tolerance.  The copy is loaded by a child process.
"""
import glob
import json
import os
import shutil
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

pytestmark = pytest.mark.gpu

CHILD = r"""
import ctypes, json, sys
sys.path.insert(0, sys.argv[2])
import torch
import lattice_synth as ls
import paper_1312_3265_gb300 as sw
from paper_1312_3265_gb300 import _binding
_binding._lib_path = lambda: sys.argv[1]
L = sw.lib()
allowed, refused = ctypes.c_int.in_dll(L, "refused_allowed"), ctypes.c_int.in_dll(L, "refused_calls")
dims, V = (6, 4, 6, 8), 1152
U = torch.from_numpy(ls.su3_links(dims, 5, ls.PLAQ_EPS)).cuda()
W = torch.empty((V, 8, 3, 3), dtype=torch.complex128, device="cuda")
sw.sw_hypercube_build(dims, U, W)
out = []
for op, prec, nsys, n in [(0, 1, 5, 0), (0, 2, 5, 1), (1, 1, 5, 0), (1, 1, 1, 1), (1, 2, 3, 1), (2, 1, 4, 0), (2, 1, 4, 1)]:
    g = torch.Generator("cuda").manual_seed(op)
    chi = torch.randn((nsys, V) + ((3,) if op == 0 else (4, 3)), dtype=torch.complex128, device="cuda", generator=g)
    x = torch.zeros_like(chi)
    allowed.value, refused.value = n, 0
    before = sw.sw_kernel_launches()
    rc, infos = sw.cgne_solve_batch(dims, op, U, W if op == 0 else None, chi, x, [0.1 + 0.1 * k for k in range(nsys)],
                                    1.0, 1e-9, 5000, prec)
    def D(v, m, dag):
        o = torch.empty_like(v)
        if op == 0: sw.sw_dslash_apply(dims, U, W, v, o, m, 1.0, dag)
        else: sw.wilson_dslash_apply(dims, U, v, o, m, 1.0, dag)
        return o
    res = []
    for k in range(nsys):
        m = 0.1 + 0.1 * k
        b = D(chi[k], m, True)
        res.append(((b - D(D(x[k], m, False), m, True)).norm() / b.norm()).item())
    out.append(dict(rc=rc, res=max(res), iters=max(i.iters for i in infos), refused=refused.value,
                    launches=sw.sw_kernel_launches() - before))
print(json.dumps(out))
"""


def test_refused_cooperative_launch_takes_the_other_kernels(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1312_3265_gb300 import build as b
    objs = sorted(glob.glob(os.path.join(b.BUILD, "*.o")))
    cxx = shutil.which("g++")
    if not objs or not cxx:
        pytest.skip("no objects of the library, or no host compiler")
    cc = b.nvcc()
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(cc))), "include")
    shim, lib = str(tmp_path / "shim.o"), str(tmp_path / "librefused.so")
    subprocess.run([cxx, "-std=c++17", "-fPIC", "-I", inc, "-I", "/usr/local/cuda/include", "-c",
                    os.path.join(HERE, "host", "refused_launch.cc"), "-o", shim], check=True)
    subprocess.run([cc, *b.ARCH, "-shared", "-o", lib, *objs, shim, "-Xlinker",
                    "--wrap=cudaLaunchCooperativeKernel"], check=True)
    run = subprocess.run([sys.executable, "-c", CHILD, lib, ROOT], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stderr[-2000:]
    for r in json.loads(run.stdout.splitlines()[-1]):
        assert r["rc"] == 0 and r["res"] <= 1.01e-9
        assert r["refused"] == 1  # asked once, then the kernels of larger lattices
        assert r["launches"] > r["iters"]  # three an iteration
