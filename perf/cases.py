"""The workloads whose speed is measured, as a user's program runs them.

Each case is one pass through the library's public calls (dw_apply,
sap_precondition, fgmresdr_solve, the solve server) on a lattice, storage
precision and right-hand-side count that its users run: the operator alone,
the Schwarz preconditioner alone, whole solves, and a served burst of solves.
``prepare`` makes what such a program has in hand (seeded fields on the GPU, a
context with its gauge field, a server with its requests), ``run`` is the pass,
``work`` the bytes and operations that the method cannot do without, ``exact``
the same results in 64 bits from plain torch.

Gauge links are exp(i eps H) with H Gaussian, the recipe of ``fieldgen`` drawn
on the GPU; eps and the distance of the bare mass from the left edge of the
spectrum are those of the repository's workloads. Solves run to 1e-12, so that
the solution itself, and not only its residual, is determined to the accuracy
that its FP64 type promises.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_1204_5463_gb300 as dw

# left edge of the spectrum of D at m0 = 0 by link disorder eps (fieldgen/spectral_edges.json)
EDGE = {0.3: 0.2285, 0.5: 0.6135, 0.6: 0.8645}
PREC = {"f64": dw.DW_F64, "f32": dw.DW_F32, "f16": dw.DW_F16, "bf16": dw.DW_BF16, "df64": dw.DW_DF64}
LINK_BYTES = {"f64": 576, "f32": 288, "f16": 144, "bf16": 144}
# sap_precondition widens its result to FP64 at the boundary; a program keeps
# the vectors in the type that holds what the storage precision gave
KEPT = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
SOLVE_STEPS = 40  # Arnoldi steps that these masses take to 1e-12, about


def _dims(c):
    return tuple(int(x) for x in c["dims"].split("x"))


def _block(c):
    return tuple(int(x) for x in c["block"].split("x"))


def _volume(c):
    return math.prod(_dims(c))


def _apply(name, dims, block, prec, nrhs, eps=0.5, csw=0.0):
    return dict(name=name, kind="apply", dims=dims, block=block, prec=prec, nrhs=nrhs, eps=eps, delta=0.01, csw=csw)


def _sap(name, dims, block, prec, nrhs, cycles, mr, eps=0.5, csw=0.0):
    return dict(name=name, kind="sap", dims=dims, block=block, prec=prec, nrhs=nrhs, eps=eps, delta=0.01, csw=csw,
                cycles=cycles, mr=mr)


def _solve(name, dims, block, prec, nrhs, outer="df64", m=30, k=10, cycles=5, mr=4, eps=0.5, delta=0.05):
    return dict(name=name, kind="solve", dims=dims, block=block, prec=prec, nrhs=nrhs, eps=eps, delta=delta, csw=0.0,
                outer=outer, m=m, k=k, cycles=cycles, mr=mr)


def listed():
    return [
        # the smallest call: one operator application on the tiny lattice, all latency
        _apply("apply_f32_4x4x4x4", "4x4x4x4", "2x2x2x2", "f32", 1, eps=0.3),
        # the operator alone on the lattice whose bandwidth the benchmark reports
        _apply("apply_f32_24x24x24x48", "24x24x24x48", "4x4x4x4", "f32", 1),
        # twelve spin-colour sources sharing one gauge field, 16-bit storage
        _apply("apply_f16_12rhs_24x24x24x48", "24x24x24x48", "4x4x4x4", "f16", 12),
        # an FP64 residual check of a solution
        _apply("apply_f64_16x16x16x32", "16x16x16x32", "4x4x4x4", "f64", 1),
        # an irregular lattice and batch with the improved operator
        _apply("apply_bf16_5rhs_clover_12x10x14x18", "12x10x14x18", "3x5x7x3", "bf16", 5, csw=1.91),
        # the preconditioner of the benchmark solve
        _sap("sap_f32_16x16x16x32", "16x16x16x32", "4x4x4x4", "f32", 1, 5, 4),
        # the preconditioner of the batched solve: twelve sources, 16-bit storage
        _sap("sap_f16_12rhs_24x24x24x48", "24x24x24x48", "4x4x4x4", "f16", 12, 5, 4),
        # domains of odd extent (81 sites), a small batch, another 16-bit format
        _sap("sap_bf16_3rhs_12x12x12x18", "12x12x12x18", "3x3x3x3", "bf16", 3, 4, 5, eps=0.3),
        # the improved operator with the paper's five MR steps and eight cycles
        _sap("sap_f32_clover_16x16x16x32", "16x16x16x32", "4x4x4x4", "f32", 1, 8, 5, csw=1.91),
        # one whole solve with the default parameters
        _solve("solve_f32_16x16x16x32", "16x16x16x32", "4x4x4x4", "f32", 1),
        # twelve right-hand sides solved together, 16-bit preconditioner
        _solve("solve_f16_12rhs_16x16x16x32", "16x16x16x32", "4x4x4x4", "f16", 12),
        # a burst of small requests at the solve server (host buffers, overlapping streams)
        dict(name="serve_6req_8x8x8x16", kind="serve", dims="8x8x8x16", block="4x4x4x4", prec="f32", nrhs=2, eps=0.6,
             delta=0.05, csw=0.0, requests=6, slots=4, m=30, k=10, cycles=5, mr=4),
    ]


BLOCKS = [(2, 2, 2, 2), (4, 4, 4, 4), (4, 4, 4, 4), (4, 4, 2, 4), (3, 3, 3, 3), (2, 4, 4, 6), (4, 2, 6, 2),
          (6, 3, 4, 3), (8, 4, 4, 2), (3, 5, 7, 2)]


def _lattice(rng, vmax):
    """Extents around a volume drawn over its logarithm, in even numbers of one of BLOCKS per direction."""
    block = rng.choice([b for b in BLOCKS if 16 * math.prod(b) <= vmax])
    n = [2, 2, 2, 2]
    target = math.exp(rng.uniform(math.log(16 * math.prod(block)), math.log(vmax)))
    while True:
        j = rng.randrange(4)
        grown = [x + 2 if i == j else x for i, x in enumerate(n)]
        if math.prod(grown) * math.prod(block) > target:
            break
        n = grown
    return "x".join(str(b * k) for b, k in zip(block, n)), "x".join(map(str, block))


def draw(rng):
    kind = rng.choice(["apply", "apply", "sap", "sap", "solve", "serve"])
    eps = rng.choice(sorted(EDGE))
    if kind == "serve":
        dims, block = _lattice(rng, 8192)
        return dict(kind=kind, dims=dims, block=block, prec=rng.choice(["f32", "f16", "bf16"]), nrhs=rng.randint(1, 3),
                    eps=eps, delta=0.05, csw=0.0, requests=rng.randint(2, 6), slots=rng.randint(2, 4), m=30, k=10,
                    cycles=5, mr=4)
    nrhs = rng.choice([1, 1, 1, 2, 3, 5, 12])
    dims, block = _lattice(rng, 663552 if kind != "solve" else 131072)
    if kind == "apply":
        c = _apply("", dims, block, rng.choice(["f64", "f32", "f32", "f16", "bf16"]), nrhs, eps, rng.choice([0.0, 0.0, 1.91]))
    elif kind == "sap":
        c = _sap("", dims, block, rng.choice(["f64", "f32", "f32", "f16", "bf16"]), nrhs, rng.randint(2, 5),
                 rng.randint(3, 6), eps, rng.choice([0.0, 0.0, 1.91]))
        if c["prec"] == "f64":  # FP64 preconditioning is a check, on small lattices
            c["dims"], c["block"] = _lattice(rng, 32768)
            c["nrhs"] = 1
    else:
        c = _solve("", dims, block, rng.choice(["f32", "f16", "bf16"]), min(nrhs, 5), rng.choice(["df64", "df64", "f32", "f64"]),
                   rng.choice([24, 30, 40]), rng.choice([0, 8, 10, 16]), rng.randint(3, 5), rng.randint(3, 6), eps,
                   rng.choice([0.05, 0.1]))
    del c["name"]
    return c


# ---- inputs ------------------------------------------------------------------


def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed(1000003 * int(seed) + stream)


def _gell_mann():
    lam = np.zeros((8, 3, 3), dtype=np.complex128)
    lam[0][0, 1] = lam[0][1, 0] = lam[3][0, 2] = lam[3][2, 0] = lam[5][1, 2] = lam[5][2, 1] = 1
    for i, (a, b) in ((1, (0, 1)), (4, (0, 2)), (6, (1, 2))):
        lam[i][a, b], lam[i][b, a] = -1j, 1j
    lam[2][0, 0], lam[2][1, 1] = 1, -1
    lam[7] = np.diag([1, 1, -2]) / math.sqrt(3)
    return torch.from_numpy(lam).cuda()


def _mul3(a, b):
    return (a.unsqueeze(-1) * b.unsqueeze(-3)).sum(-2)


def _links(V, eps, seed, stream=0):
    """SU(3) links (V, 4, 3, 3), complex128: exp(i eps H) by scaling, Taylor series and squaring."""
    omega = torch.randn(V * 4, 8, dtype=torch.float64, device="cuda", generator=_gen(seed, stream))
    X = (omega.to(torch.complex128) @ _gell_mann().reshape(8, 9)).reshape(-1, 3, 3) * (0.5j * eps / 32)
    eye = torch.eye(3, dtype=torch.complex128, device="cuda").expand_as(X)
    U = eye
    for n in range(9, 0, -1):
        U = eye + _mul3(X, U) / n
    for _ in range(5):
        U = _mul3(U, U)
    return U.reshape(V, 4, 3, 3).contiguous()


def _sources(nrhs, V, seed, stream=1):
    """Complex Gaussian spinor fields (nrhs, V, 4, 3), complex128."""
    return torch.view_as_complex(torch.randn(nrhs, V, 4, 3, 2, dtype=torch.float64, device="cuda", generator=_gen(seed, stream)))


def _m0(c):
    return c["delta"] - EDGE[c["eps"]]


def _params(c, **kw):
    return dw.dw_default_params(m=c["m"], k=c["k"], tol=1e-12, sap_cycles=c["cycles"], mr_steps=c["mr"],
                                sap_prec=PREC[c["prec"]], nrhs=c["nrhs"], **kw)


class _Lattice:
    """A context with its gauge field, the input fields and the output buffer."""

    def __init__(self, c, seed):
        self.case, V = c, _volume(c)
        self.ctx = dw.dw_create(_dims(c), _block(c), _m0(c), torch.cuda.current_stream().cuda_stream)
        dw.dw_set_gauge(self.ctx, _links(V, c["eps"], seed), True)
        if c["csw"]:
            dw.dw_set_clover(self.ctx, c["csw"])
        self.b = _sources(c["nrhs"], V, seed)
        self.x = torch.empty_like(self.b)
        self.params = _params(c, outer_prec=PREC[c["outer"]]) if c["kind"] == "solve" else None

    def __del__(self):
        if getattr(self, "ctx", None):
            dw.dw_destroy(self.ctx)


class _Served:
    """A server and the requests of a burst: each its own gauge field, all in host memory."""

    def __init__(self, c, seed):
        self.case, V = c, _volume(c)
        self.U = [_links(V, c["eps"], seed, 2 * i).cpu().numpy() for i in range(c["requests"])]
        self.b = [_sources(c["nrhs"], V, seed, 2 * i + 1).cpu().numpy() for i in range(c["requests"])]
        self.x = [np.zeros_like(b) for b in self.b]
        self.reqs = [dw.make_request(_dims(c), _block(c), _m0(c), U, b, x, _params(c)) for U, b, x in
                     zip(self.U, self.b, self.x)]
        self.server = dw.dw_server_create(32 << 30, c["slots"])

    def __del__(self):
        if getattr(self, "server", None):
            dw.dw_server_destroy(self.server)


def prepare(case, seed):
    return _Served(case, seed) if case["kind"] == "serve" else _Lattice(case, seed)


def run(state):
    c = state.case
    if c["kind"] == "apply":
        dw.dw_apply(state.ctx, state.b, state.x, PREC[c["prec"]], c["nrhs"])
        return state.x
    if c["kind"] == "sap":
        dw.sap_precondition(state.ctx, state.b, state.x, c["cycles"], c["mr"], PREC[c["prec"]], c["nrhs"])
        return list(torch.view_as_real(state.x).to(KEPT[c["prec"]]))
    if c["kind"] == "solve":
        dw.fgmresdr_solve(state.ctx, state.b, state.x, state.params)
        return list(state.x)
    ids = [dw.dw_server_submit(state.server, r) for r in state.reqs]
    for i in ids:
        status, _, _ = dw.dw_server_wait(state.server, i)
        if status != dw.DW_OK:
            raise RuntimeError(f"request {i} ended with status {status}")
    return state.x


# ---- what a pass cannot do without ---------------------------------------------


def _sap_flops(c):
    """FP32 operations per site of one application: every site's residual once per cycle and its MR steps."""
    hops = sum(2.0 * (b - 1) / b for b in _block(c))
    clover = 576.0 if c["csw"] else 0.0
    return c["cycles"] * (1392.0 + clover + c["mr"] * (165.0 * hops + 48.0 + 336.0 + clover))


def work(case):
    c, V = case, _volume(case)
    links = V * (LINK_BYTES[c["prec"]] + ((576 if c["prec"] == "f64" else 288) if c["csw"] else 0))
    fields = 2.0 * 192 * V * c["nrhs"]
    if c["kind"] == "apply":
        return {"bytes": fields + links, "flops": c["nrhs"] * V * (1392.0 + (576.0 if c["csw"] else 0.0))}
    if c["kind"] == "sap":
        return {"bytes": fields + links, "flops": c["nrhs"] * V * _sap_flops(c)}
    # a solve: per Arnoldi step the preconditioner, one product and the two
    # sweeps of Gram-Schmidt over a basis of half its full length on average
    vec = V * (96 if c.get("outer") == "f32" else 192)
    step = {"bytes": 2.0 * (c["m"] / 2 + 1) * vec + V * 480.0, "flops": V * (_sap_flops(c) + 1392.0 + 8 * 12 * 2 * c["m"] / 2)}
    n = SOLVE_STEPS * c["nrhs"] * c.get("requests", 1)
    return {"bytes": fields + links + n * step["bytes"], "flops": n * step["flops"]}


# ---- the same in 64 bits ---------------------------------------------------------


class _Operator:
    """D, its clover term and its restriction to the domains, in complex128 on a
    grid (d4, d3, d2, d1): plain rolls and 3x3 products."""

    def __init__(self, c, U):
        self.d, self.b, self.diag = _dims(c), _block(c), 4.0 + _m0(c)
        self.grid = self.d[::-1]
        self.U = U.reshape(*self.grid, 4, 3, 3)
        z, o = torch.zeros(2, 2, dtype=torch.complex128), torch.eye(2, dtype=torch.complex128)
        s = [torch.tensor(p, dtype=torch.complex128) for p in ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]])]
        up = [-1j * p for p in s] + [o]
        self.gamma = [torch.cat([torch.cat([z, a], 1), torch.cat([a.conj().T, z], 1)]).cuda() for a in up]
        self.eye = torch.eye(4, dtype=torch.complex128, device="cuda")
        self.coord = []
        for mu in range(4):
            shape = [1] * 4
            shape[3 - mu] = self.d[mu]
            self.coord.append(torch.arange(self.d[mu], device="cuda").reshape(shape))
        self.A = None
        if c["csw"]:
            self.A = self._clover(c["csw"])

    def field(self, v):
        return v.reshape(*self.grid, 4, 3)

    def _shift(self, f, mu, n):  # value at site + n mu
        return torch.roll(f, -n, 3 - mu)

    def _clover(self, csw):
        A = torch.zeros(*self.grid, 4, 3, 4, 3, dtype=torch.complex128, device="cuda")
        mm = lambda *m: _mul3(m[0], m[1]) if len(m) == 2 else _mul3(mm(*m[:-1]), m[-1])  # noqa: E731
        H = lambda m: m.conj().transpose(-1, -2)  # noqa: E731
        for mu in range(4):
            for nu in range(mu + 1, 4):
                a, b = self.U[..., mu, :, :], self.U[..., nu, :, :]
                at = self._shift
                Q = mm(a, at(b, mu, 1), H(at(a, nu, 1)), H(b))
                Q = Q + mm(b, H(at(at(a, mu, -1), nu, 1)), H(at(b, mu, -1)), at(a, mu, -1))
                Q = Q + mm(H(at(a, mu, -1)), H(at(at(b, mu, -1), nu, -1)), at(at(a, mu, -1), nu, -1), at(b, nu, -1))
                Q = Q + mm(H(at(b, nu, -1)), at(a, nu, -1), at(at(b, mu, 1), nu, -1), H(a))
                F = (Q - H(Q)) / 8
                F = F - torch.einsum("...aa->...", F)[..., None, None] / 3 * torch.eye(3, device="cuda")
                s = 0.5j * (self.gamma[mu] @ self.gamma[nu] - self.gamma[nu] @ self.gamma[mu])
                A = A + 0.5j * csw * torch.einsum("st,...ab->...satb", s, F)
        return A.reshape(*self.grid, 12, 12)

    def hops(self, psi, local):
        acc = torch.zeros_like(psi)
        for mu in range(4):
            U = self.U[..., mu, :, :]
            for sign in (1, -1):
                P = self.eye + sign * self.gamma[mu]
                if sign > 0:
                    h = torch.einsum("st,...tb->...sb", P, self._shift(psi, mu, 1))
                    t = torch.matmul(h, U.transpose(-1, -2))
                else:
                    h = torch.einsum("st,...tb->...sb", P, psi)
                    t = self._shift(torch.matmul(h, U.conj()), mu, -1)
                if local:
                    edge = self.b[mu] - 1 if sign > 0 else 0
                    t = t * (self.coord[mu] % self.b[mu] != edge)[..., None, None]
                acc = acc + t
        return acc

    def __call__(self, psi, local=False):
        out = self.diag * psi - 0.5 * self.hops(psi, local)
        if self.A is not None:
            out = out + torch.matmul(self.A, psi.reshape(*self.grid, 12, 1)).reshape(psi.shape)
        return out

    def domain_sum(self, f):
        """Sum of a grid of numbers over each domain, given back on every site of it."""
        n, b = [d // k for d, k in zip(self.d, self.b)][::-1], self.b[::-1]
        shape = [x for p in zip(n, b) for x in p]
        s = f.reshape(shape).sum(dim=(1, 3, 5, 7), keepdim=True)
        return s.expand(shape).reshape(f.shape)

    def sap(self, v, cycles, mr):
        parity = sum(self.coord[mu] // self.b[mu] for mu in range(4)) % 2
        x = torch.zeros_like(v)
        for _ in range(cycles):
            for colour in (0, 1):
                on = (parity == colour)[..., None, None]
                r = (v - self(x)) * on
                for _ in range(mr):
                    p = self(r, local=True) * on
                    pp = self.domain_sum((p.real**2 + p.imag**2).sum((-1, -2)))
                    pr = self.domain_sum((p.conj() * r).sum((-1, -2)))
                    alpha = torch.where(pp > 0, pr / torch.where(pp > 0, pp, 1.0), 0.0)[..., None, None]
                    x, r = x + alpha * r, r - alpha * p
        return x

    def solve(self, b):
        """D^-1 b by BiCGStab to 1e-14, restarted from the true residual."""
        x, norm = torch.zeros_like(b), b.norm()
        dot = lambda a, c: torch.vdot(a.reshape(-1), c.reshape(-1))  # noqa: E731
        for _ in range(20):
            r = b - self(x)
            if r.norm() <= 1e-14 * norm:
                break
            r0, p, rho, goal = r, r, dot(r, r), max(1e-15 * norm, 1e-6 * r.norm())
            for _ in range(2000):
                q = self(p)
                alpha = rho / dot(r0, q)
                s = r - alpha * q
                t = self(s)
                w = dot(t, s) / dot(t, t)
                x, r = x + alpha * p + w * s, s - w * t
                if r.norm() <= goal:
                    break
                new = dot(r0, r)
                p = r + (new / rho) * (alpha / w) * (p - w * q)
                rho = new
        return x


def exact(case, seed):
    c, V = case, _volume(case)
    if c["kind"] == "serve":
        got = []
        for i in range(c["requests"]):
            D = _Operator(c, _links(V, c["eps"], seed, 2 * i))
            got.append(torch.stack([D.solve(D.field(f)).reshape(V, 4, 3) for f in _sources(c["nrhs"], V, seed, 2 * i + 1)]))
        return got
    D = _Operator(c, _links(V, c["eps"], seed))
    b = [D.field(f) for f in _sources(c["nrhs"], V, seed)]
    if c["kind"] == "apply":
        return torch.stack([D(f).reshape(V, 4, 3) for f in b])
    # each right-hand side is an output of its own: as many as the time allows
    few = max(1, 700000 // V) if c["kind"] == "sap" else max(1, 131072 // V)
    if c["kind"] == "sap":
        got = [torch.view_as_real(D.sap(f, c["cycles"], c["mr"]).reshape(V, 4, 3)) for f in b[:few]]
    else:
        got = [D.solve(f).reshape(V, 4, 3) for f in b[:few]]
    return got + [None] * (c["nrhs"] - len(got))
