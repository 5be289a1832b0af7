"""The work this library is used for, as cases to measure: operator applications,
transport builds and CGNE solves through the package's public entry points.

listed() names the cases, draw() gives more of the same ranges, prepare() makes
what a user's program holds before the call, run() is one pass, work() counts
what a pass cannot do without, exact() gives its result from plain torch in
64 bits (no code of this library).

Gauge fields follow the library's synthetic recipe: U = reunitarise(exp(i eps H)),
H = sum_a theta_a lambda_a, theta_a ~ N(0, 1), eps = 0.219 (mean plaquette 0.59).
Solves start from x = 0 and run to a relative residual of the case's `tol`.
"""
import math

import torch

import paper_1312_3265_gb300 as sw

EPS = 0.219
OPS = {"sw": sw.SW_OP_STAGGERED_WILSON, "wilson": sw.SW_OP_WILSON, "wilson_eo": sw.SW_OP_WILSON_EVEN_ODD}
PREC = {"f64": sw.SW_PREC_F64, "f32": sw.SW_PREC_F32_RELIABLE, "f16": sw.SW_PREC_F16_RELIABLE}
MASSES = (0.02, 0.05, 0.1, 0.2)
MAX_ITER = 20000


def _dims(case):
    return (case["l0"], case["l1"], case["l2"], case["l3"])


def _lattice(l0, l1, l2, l3, **more):
    return dict(l0=l0, l1=l1, l2=l2, l3=l3, **more)


def _apply(name, op, dims, mass=0.1, r=1.0, dagger=False, apbc=False):
    return dict(_lattice(*dims), name=name, kind="apply", op=op, mass=mass, r=r, dagger=dagger, apbc=apbc)


def _solve(name, op, prec, dims, source, nsrc, nmass, r=1.0, apbc=False, tol=1e-10):
    return dict(_lattice(*dims), name=name, kind="solve", op=op, prec=prec, source=source, nsrc=nsrc, nmass=nmass,
                r=r, apbc=apbc, tol=tol)


def listed():
    return [
        # one matrix application inside a user's own solver or measurement, small lattice: launch and latency
        _apply("apply_sw_8x8x8x8", "sw", (8, 8, 8, 8)),
        # the same on the paper's lattice, the usual Wilson operator
        _apply("apply_wilson_16x16x16x32", "wilson", (16, 16, 16, 32)),
        # the adjoint with the antiperiodic time boundary on the batched runs' lattice
        _apply("apply_sw_dag_24x24x24x48", "sw", (24, 24, 24, 48), dagger=True, apbc=True),
        # hypercube transports, once per gauge configuration of the paper's lattice
        dict(_lattice(16, 16, 16, 32), name="transports_16x16x16x32", kind="transports", apbc=False),
        # one interactive or test solve: a single point source on a small lattice
        _solve("solve_sw_f32_8x8x8x8", "sw", "f32", (8, 8, 8, 8), "point", 1, 1),
        # one noise source on a ragged lattice with antiperiodic time and r != 1
        _solve("solve_wilson_f32_6x10x12x14", "wilson", "f32", (6, 10, 12, 14), "gaussian", 1, 1, r=0.75, apbc=True),
        # plain FP64 CG of one quark's twelve spin-colour sources, the option without mixed precision
        _solve("batch_wilson_f64_8x8x8x16", "wilson", "f64", (8, 8, 8, 16), "point", 12, 1),
        # the paper's staggered Wilson batch: three colour sources x four masses
        _solve("batch_sw_f32_16x16x16x32", "sw", "f32", (16, 16, 16, 32), "point", 3, 4),
        # the paper's Wilson batch: twelve spin-colour sources x four masses
        _solve("batch_wilson_f32_16x16x16x32", "wilson", "f32", (16, 16, 16, 32), "point", 12, 4),
        # one propagator by the even-odd preconditioned solver
        _solve("batch_wilson_eo_f32_16x16x16x32", "wilson_eo", "f32", (16, 16, 16, 32), "point", 12, 1),
        # half-precision storage, a propagator on a lattice between the small and the paper's, to a tight residual
        # (where this storage needs most residual replacements)
        _solve("batch_wilson_f16_12x12x12x24", "wilson", "f16", (12, 12, 12, 24), "point", 12, 1, tol=1e-11),
        # noise sources x masses on the larger lattice of the batched runs
        _solve("batch_sw_f32_24x24x24x48", "sw", "f32", (24, 24, 24, 48), "z2", 6, 4, apbc=True),
    ]


def _volume(case):
    return case["l0"] * case["l1"] * case["l2"] * case["l3"]


def _iters(case):
    """CG iterations of a solve, from the condition numbers these gauge fields show."""
    root_kappa = {"sw": 4.7, "wilson": 15.0, "wilson_eo": 6.0}[case["op"]]
    return 0.42 * root_kappa * math.log(2.0 / case["tol"])


def _cost(case):
    """Rough arithmetic of a case, FP64 work weighted by what it costs beside FP32's."""
    w = work(case)["flops"]
    return w * (16 if case["kind"] != "solve" or case["prec"] == "f64" else 1)


def draw(rng):
    biggest = max(_cost(c) for c in listed())
    while True:
        volume = math.exp(rng.uniform(math.log(256), math.log(24 ** 3 * 48)))
        base = (volume / 2) ** 0.25
        sp = [max(2, 2 * round(base * rng.uniform(0.75, 1.3) / 2)) for _ in range(3)]
        lt = min(64, max(2, 2 * round(volume / (sp[0] * sp[1] * sp[2]) / 2)))
        case = _lattice(sp[0], sp[1], sp[2], lt, apbc=rng.random() < 0.5)
        kind = rng.choice(["apply", "apply", "transports", "solve", "solve", "solve", "solve", "solve"])
        case["kind"] = kind
        if kind == "apply":
            case.update(op=rng.choice(["sw", "wilson"]), mass=rng.choice(MASSES), r=rng.choice([1.0, 1.0, 1.0, 0.75]),
                        dagger=rng.random() < 0.5)
        elif kind == "solve":
            op = rng.choice(["sw", "sw", "wilson", "wilson", "wilson_eo"])
            prec = rng.choice(["f32", "f32", "f32", "f32", "f16", "f64"])
            if op == "wilson_eo" and prec == "f16":
                prec = "f32"
            source = rng.choice(["point", "z2", "gaussian"])
            nsrc = rng.choice([1, 2, 3, 5, 12])
            if source == "point":
                nsrc = min(nsrc, 3 if op == "sw" else 12)
            case.update(op=op, prec=prec, source=source, nsrc=nsrc, nmass=rng.choice([1, 1, 2, 4]),
                        r=rng.choice([1.0, 1.0, 1.0, 0.75]), tol=1e-11 if prec == "f16" else 1e-10)
        if _volume(case) <= 24 ** 3 * 48 and _cost(case) <= biggest:
            return case


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _links(dims, gen):
    """SU(3) links [V][4][3][3], complex128."""
    V = dims[0] * dims[1] * dims[2] * dims[3]
    th = torch.randn((V * 4, 8), dtype=torch.float64, device="cuda", generator=gen)
    H = torch.zeros((V * 4, 3, 3), dtype=torch.complex128, device="cuda")
    for k, (i, j) in ((0, (0, 1)), (3, (0, 2)), (5, (1, 2))):
        H[:, i, j] = torch.complex(th[:, k], -th[:, k + 1])
        H[:, j, i] = torch.complex(th[:, k], th[:, k + 1])
    d8 = th[:, 7] / math.sqrt(3.0)
    H[:, 0, 0], H[:, 1, 1], H[:, 2, 2] = th[:, 2] + d8, d8 - th[:, 2], -2 * d8
    A = 1j * EPS * H
    M = torch.eye(3, dtype=torch.complex128, device="cuda").expand_as(A)
    for k in range(12, 0, -1):  # exp(A) by Horner; the projection below makes it SU(3) to rounding
        M = torch.eye(3, dtype=torch.complex128, device="cuda") + (A @ M) / k
    r0 = M[:, 0] / torch.linalg.vector_norm(M[:, 0], dim=1, keepdim=True)
    r1 = M[:, 1] - (r0.conj() * M[:, 1]).sum(1, keepdim=True) * r0
    r1 = r1 / torch.linalg.vector_norm(r1, dim=1, keepdim=True)
    r2 = torch.linalg.cross(r0, r1, dim=1).conj()
    return torch.stack([r0, r1, r2], dim=1).reshape(V, 4, 3, 3).contiguous()


def _noise(shape, gen, z2=False):
    if z2:
        s = torch.randint(0, 2, shape, device="cuda", generator=gen)
        return (2 * s - 1).to(torch.complex128)
    return torch.complex(torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen),
                         torch.randn(shape, dtype=torch.float64, device="cuda", generator=gen))


def _internal(op):
    return (3,) if op == "sw" else (4, 3)


def _inputs(case, seed):
    """Links, source vectors and masses: what both prepare() and exact() start from."""
    gen = _generator(seed)
    dims, V = _dims(case), _volume(case)
    U = _links(dims, gen)
    if case["kind"] == "transports":
        return U, None, None
    if case["kind"] == "apply":
        return U, _noise((V,) + _internal(case["op"]), gen), None
    n, inner = case["nsrc"], _internal(case["op"])
    if case["source"] == "point":
        site = int(torch.randint(0, V, (1,), device="cuda", generator=gen))
        src = torch.zeros((n, V, 3 if len(inner) == 1 else 12), dtype=torch.complex128, device="cuda")
        src[torch.arange(n, device="cuda"), site, torch.arange(n, device="cuda")] = 1.0
        src = src.reshape((n, V) + inner)
    else:
        src = _noise((n, V) + inner, gen, case["source"] == "z2")
    masses = [m for m in (MASSES if case["nmass"] > 1 else MASSES[1:2])[: case["nmass"]] for _ in range(n)]
    return U, src.repeat((case["nmass"],) + (1,) * (src.dim() - 1)).contiguous(), masses


def prepare(case, seed):
    U, v, masses = _inputs(case, seed)
    dims, V = _dims(case), _volume(case)
    s = dict(case=case, dims=dims, U=U, v=v, masses=masses, W=None)
    if case["kind"] == "transports" or case["op"] == "sw":
        s["W"] = torch.empty((V, 8, 3, 3), dtype=torch.complex128, device="cuda")
    if case["kind"] != "transports":
        s["out"] = torch.zeros_like(v)
        if case["op"] == "sw":
            sw.sw_hypercube_build(dims, U, s["W"], case["apbc"])
    return s


def run(state):
    c, dims = state["case"], state["dims"]
    if c["kind"] == "transports":
        sw.sw_hypercube_build(dims, state["U"], state["W"], c["apbc"])
        return state["W"]
    if c["kind"] == "apply":
        if c["op"] == "sw":
            sw.sw_dslash_apply(dims, state["U"], state["W"], state["v"], state["out"], c["mass"], c["r"], c["dagger"],
                               c["apbc"])
        else:
            sw.wilson_dslash_apply(dims, state["U"], state["v"], state["out"], c["mass"], c["r"], c["dagger"],
                                   c["apbc"])
        return state["out"]
    x = state["out"].zero_()  # the initial guess
    if len(state["masses"]) == 1:
        sw.cgne_solve(dims, OPS[c["op"]], state["U"], state["W"], state["v"], x, state["masses"][0], c["r"], c["tol"],
                      MAX_ITER, PREC[c["prec"]], c["apbc"])
    else:
        sw.cgne_solve_batch(dims, OPS[c["op"]], state["U"], state["W"], state["v"], x, state["masses"], c["r"],
                            c["tol"], MAX_ITER, PREC[c["prec"]], c["apbc"])
    return x


def work(case):
    V = _volume(case)
    links, transports = 4 * 9 * 16, 8 * 9 * 16
    if case["kind"] == "transports":
        # per stored transport: six products of two two-link sums, each sum two products of two links,
        # shared over the lattice (12 sums per site); a complex 3x3 product: 198 flops
        return {"bytes": V * (links + transports), "flops": V * (8 * 6 + 12 * 2) * 198}
    nc, flops = (3, 1743) if case["op"] == "sw" else (12, 1392)
    gauge = links + (transports if case["op"] == "sw" else 0)
    if case["kind"] == "apply":
        return {"bytes": V * (gauge + 2 * 16 * nc), "flops": V * flops}
    n = case["nsrc"] * case["nmass"]
    # sources in, solutions out; two applications an iteration and two for the residual that decides
    return {"bytes": V * (gauge + 2 * 16 * nc * n), "flops": V * n * flops * 2 * (_iters(case) + 1)}


# ------------------------------------------------------------------ 64-bit results from plain torch


def _shifted(dims):
    """idx(s): for every site x the index of x + s (periodic)."""
    grid = torch.arange(dims[0] * dims[1] * dims[2] * dims[3], device="cuda").reshape(dims[3], dims[2], dims[1], dims[0])

    def idx(s):
        return torch.roll(grid, shifts=[-s[3], -s[2], -s[1], -s[0]], dims=[0, 1, 2, 3]).reshape(-1)

    return idx


def _coords(dims):
    n = torch.arange(dims[0] * dims[1] * dims[2] * dims[3], device="cuda")
    x = []
    for L in dims:
        x.append(n % L)
        n = n // L
    return x


def _unit(mu, s):
    e = [0, 0, 0, 0]
    e[mu] = s
    return e


def _transports(dims, U, signs):
    """Average over the 24 orderings of the four-link path x -> x + signs."""
    idx = _shifted(dims)

    def link(mu):  # the link walked from x in direction signs[mu]
        if signs[mu] > 0:
            return U[:, mu]
        return U[idx(_unit(mu, -1)), mu].conj().transpose(-1, -2)

    L = [link(mu) for mu in range(4)]

    def two(a, b):
        return L[a] @ L[b][idx(_unit(a, signs[a]))] + L[b] @ L[a][idx(_unit(b, signs[b]))]

    W = 0
    for a in range(4):
        for b in range(a + 1, 4):
            c, d = [m for m in range(4) if m not in (a, b)]
            s = [signs[m] if m in (a, b) else 0 for m in range(4)]
            W = W + two(a, b) @ two(c, d)[idx(s)]
    return W / 24.0


def _k_signs(k):
    return [-1 if k & 1 else 1, -1 if k & 2 else 1, -1 if k & 4 else 1, 1]


class _Operator:
    """D + m and its adjoint on [V][3][columns] (staggered) or [V][3][4 x columns] (Wilson, spin slowest)."""

    def __init__(self, case, U):
        self.dims, self.op, self.r = _dims(case), "sw" if case["op"] == "sw" else "wilson", case["r"]
        x, idx = _coords(self.dims), _shifted(self.dims)
        V = U.shape[0]
        one = torch.ones(V, dtype=torch.float64, device="cuda")
        fw, bw = one.clone(), one.clone()
        if case["apbc"]:
            fw[x[3] == self.dims[3] - 1] = -1
            bw[x[3] == 0] = -1
        self.hops = []  # (matrix [V][3][3] with the boundary sign, neighbour index, direction, sign)
        for mu in range(4):
            for s in (1, -1):
                i = idx(_unit(mu, s))
                M = U[:, mu] if s > 0 else U[i, mu].conj().transpose(-1, -2)
                sign = (fw if s > 0 else bw) if mu == 3 else one
                self.hops.append((sign[:, None, None] * M, i, mu, s))
        if self.op == "sw":
            par = 0
            for mu in range(4):
                eta = (1 - 2 * (par % 2)).to(torch.float64) if mu else one
                for h in (2 * mu, 2 * mu + 1):
                    M, i, m, s = self.hops[h]
                    self.hops[h] = (0.5 * s * eta[:, None, None] * M, i, m, s)
                par = par + x[mu]
            g5 = (1 - 2 * ((x[1] + x[3]) % 2)).to(torch.float64)
            self.corners = []
            for k in range(8):
                W = _transports(self.dims, U, _k_signs(k))
                i, j = idx(_k_signs(k)), idx([-s for s in _k_signs(k)])
                c = (-self.r / 16) * g5
                self.corners.append(((c * fw)[:, None, None] * W, i))
                self.corners.append(((c * bw)[:, None, None] * W[j].conj().transpose(-1, -2), j))
        else:
            s1 = torch.tensor([[0, 1], [1, 0]], dtype=torch.complex128)
            s2 = torch.tensor([[0, -1j], [1j, 0]], dtype=torch.complex128)
            s3 = torch.tensor([[1, 0], [0, -1]], dtype=torch.complex128)
            eye = torch.eye(2, dtype=torch.complex128)
            self.gamma = []
            for A in (1j * s1, -1j * s2, 1j * s3, eye):
                g = torch.zeros((4, 4), dtype=torch.complex128)
                g[:2, 2:], g[2:, :2] = A, A.conj().T
                self.gamma.append(g.cuda())

    def __call__(self, v, mass, dagger=False):
        """v: [V][3][S][n] (S = 1 or 4), mass: [n]."""
        V, _, S, n = v.shape
        if self.op == "sw":
            flat = v.reshape(V, 3, n)
            sg = -1.0 if dagger else 1.0
            out = 0
            for M, i, _, _ in self.hops:
                out = out + sg * (M @ flat[i])
            for M, i in self.corners:
                out = out + M @ flat[i]
            return out.reshape(v.shape) + (self.r + mass) * v
        out = (4 * self.r + mass) * v
        eye = torch.eye(4, dtype=torch.complex128, device="cuda")
        for M, i, mu, s in self.hops:
            P = -0.5 * (self.r * eye - (-s if dagger else s) * self.gamma[mu])
            h = (M @ v[i].reshape(V, 3, S * n)).reshape(V, 3, S, n)
            for a in range(4):
                for b in P[a].nonzero().reshape(-1).tolist():
                    out[:, :, a] += P[a, b] * h[:, :, b]
        return out


def _to_columns(v, op):
    """[n][V][(4)][3] -> [V][3][S][n]"""
    if op == "sw":
        return v.permute(1, 2, 0).unsqueeze(2).contiguous()
    return v.permute(1, 3, 2, 0).contiguous()


def _from_columns(v, op):
    return (v.squeeze(2).permute(2, 0, 1) if op == "sw" else v.permute(3, 0, 2, 1)).contiguous()


def exact(case, seed):
    U, v, masses = _inputs(case, seed)
    dims = _dims(case)
    if case["kind"] == "transports":
        return torch.stack([_transports(dims, U, _k_signs(k)) for k in range(8)], dim=1)
    D = _Operator(case, U)
    if case["kind"] == "apply":
        m = torch.tensor([case["mass"]], dtype=torch.float64, device="cuda")
        return _from_columns(D(_to_columns(v[None], case["op"]), m, case["dagger"]), case["op"])[0]
    m = torch.tensor(masses, dtype=torch.float64, device="cuda")
    # textbook CG on the normal equations, each column by itself, down to rounding
    r = D(_to_columns(v, case["op"]), m, True)
    x, p = torch.zeros_like(r), r.clone()

    def norm2(a):
        return torch.view_as_real(a).square().sum(dim=(0, 1, 2, 4))

    rr = norm2(r)
    stop = rr * 1e-26
    for _ in range(2000):
        t = D(p, m)
        alpha = torch.where(rr > stop, rr / norm2(t), 0.0)
        x += alpha * p
        r -= alpha * D(t, m, True)
        new = norm2(r)
        beta = torch.where(rr > stop, new / rr, 0.0)
        p = r + beta * p
        rr = new
        if bool((rr <= stop).all()):
            break
    return _from_columns(x, case["op"])
