"""Performance cases of the library: what a user's program has it do, as calls of the public entry points.

A case names its kind of call, the decomposition and the options:

    kind    stencil | solve | action | w | force | md | net
    cells   per direction (time first, "/" between) the cells the lattice is cut into, e.g. "8,10/8,10/9,9/18*": a cell
            is one core and its frame, and a "*" leaves the direction undecomposed (one periodic extent)
    frame   thickness of the frame in sites
    nrhs    right-hand sides per block, or multi-boson fields, or network pairs per block
    kappa, eps (roughness of the links exp(i eps H)), csw (clover coefficient, 0 for none)
    prec    storage of the stencil, or the inner precision of the solves
    and, where they apply, tune and graph (solver options) and steps (leapfrog steps)

prepare() holds what such a program keeps: the context with its links and decomposition, the network, the right-hand
sides on the GPU and the output buffers.  exact() repeats the mathematics in 64 bits with plain torch.
"""

import math

import numpy as np
import torch

from paper_2211_06902_gb300 import dd4d

TOL = 1e-10            # the tolerance every solve of the repository's benchmark and tests runs to
CHANNELS = (4, 16, 16, 16, 4)
APPLICATIONS = 40      # applications of D that a Krylov solve to TOL needs at these kappas, at the least


def _case(kind, cells, frame, nrhs, kappa=0.135, eps=0.5, csw=0.0, prec="f32", tune=False, graph=False, steps=0):
    return {"kind": kind, "cells": cells, "frame": frame, "nrhs": nrhs, "kappa": kappa, "eps": eps, "csw": csw,
            "prec": prec, "tune": tune, "graph": graph, "steps": steps}


def _uniform(n, cell):
    return "/".join([",".join([str(cell)] * n)] * 4)


def listed():
    return [
        # one application of the FP64 stencil to the 16 framed 5^4 blocks of an 8^4 lattice: the smallest call, where
        # launches count (the residual check and the pseudofermion heat-bath of a program on a small lattice)
        dict(_case("stencil", _uniform(2, 4), 1, 1, 0.13, 0.3, prec="f64"), name="stencil f64 8x4"),
        # the FP32 stencil on framed 9^4 blocks with 12 right-hand sides, the library's central kernel on its own
        dict(_case("stencil", _uniform(3, 8), 1, 12, prec="f32"), name="stencil f32 24x4"),
        # mixed-precision block solves on the 8^4 lattice (5^4 blocks): a solve bound by its launches
        dict(_case("solve", _uniform(2, 4), 1, 4, 0.13, 0.3), name="solve 8x4"),
        # uneven blocks of odd sides, a thick frame in one direction's cells, an odd count of right-hand sides, and a
        # direction that is not decomposed
        dict(_case("solve", "8,10/7,9/10,8/6*", 2, 5, 0.136, 0.6), name="solve uneven"),
        # the benchmark's batch: 32^4, 256 framed 9^4 blocks, 12 right-hand sides, launch form tuned
        dict(_case("solve", _uniform(4, 8), 1, 12, tune=True), name="solve 32x4"),
        # the same blocks with the clover term on a smaller lattice
        dict(_case("solve", _uniform(2, 8), 1, 12, csw=1.0), name="solve clover 16x4"),
        # plain FP64 solves: the training targets of the network and the dense check use them
        dict(_case("solve", _uniform(2, 8), 1, 3, prec="f64"), name="solve f64 16x4"),
        # one evaluation of the multi-boson action on 8^4 (frame pieces, frame, blocks, reductions)
        dict(_case("action", _uniform(2, 4), 1, 2, 0.13, 0.3), name="action 8x4"),
        # the operator w for 12 fields on uneven blocks: what the action, the heat-bath of the fields and the
        # reweighting samples apply again and again
        dict(_case("w", "7,9,7,9/7,9/7,9/7,9", 1, 12, 0.136, 0.6, tune=True, graph=True), name="w 32x16x3"),
        # the force on the active links for 12 fields (two block solves and the link contraction)
        dict(_case("force", _uniform(3, 8), 1, 12), name="force 24x4"),
        # a leapfrog trajectory of the active links: every step has new links
        dict(_case("md", _uniform(2, 8), 1, 4, steps=2), name="md 16x4"),
        # loss and weight gradients of the network preconditioner: its forward and backward layers, one training step
        dict(_case("net", _uniform(2, 8), 1, 4), name="net gradient 16x4"),
    ]


def draw(rng):
    kind = rng.choice(("stencil", "solve", "solve", "solve", "action", "w", "force", "md", "net"))
    small = rng.random() < 0.4
    extents = (4, 5, 6) if small else (6, 7, 8, 9, 10)
    frame = rng.choice((1, 1, 1, 2))
    dirs = []
    for m in range(4):
        n = 2 if small or m else rng.choice((2, 2, 3, 4))
        while True:
            cells = [rng.choice([e for e in extents if e >= frame + 2]) for _ in range(n)]
            if sum(cells) % 2 == 0:
                break
        dirs.append(",".join(map(str, cells)))
    if rng.random() < 0.15:
        dirs[3] = "%d*" % rng.choice((4, 6, 8))
    most = {"net": 6, "md": 4, "force": 12}.get(kind, 16)
    nrhs = max(1, min(most, round(math.exp(rng.uniform(0.0, math.log(most + 0.5))))))
    case = _case(kind, "/".join(dirs), frame, nrhs, round(rng.uniform(0.120, 0.136), 4), round(rng.uniform(0.3, 0.6), 2),
                 steps=rng.choice((1, 2)) if kind == "md" else 0)
    if kind == "stencil":
        case["prec"] = rng.choice(("f64", "f32", "bf16"))
    elif kind == "solve":
        case["prec"] = rng.choice(("f32", "f32", "f32", "bf16", "f64"))
        case["csw"] = rng.choice((0.0, 0.0, 0.0, 1.0))
    if kind in ("solve", "action", "w"):
        case["tune"], case["graph"] = rng.random() < 0.3, rng.random() < 0.3
    return case


# ---- the decomposition ------------------------------------------------------------------------

def _geometry(case):
    """Extents, cores per direction (the call's argument) and per block (origin, side, core) of its box."""
    L, cores = [], []
    for d in case["cells"].split("/"):
        if d.endswith("*"):
            L.append(int(d[:-1]))
            cores.append([])
            continue
        at, c = 0, []
        for n in map(int, d.split(",")):
            c.append((at, at + n - case["frame"] - 1))
            at += n
        L.append(at)
        cores.append(c)
    per = []
    for m in range(4):
        c, k = cores[m], len(cores[m])
        if not c:
            per.append([(0, L[m], 0, L[m])])
            continue
        row = []
        for i in range(k):
            o = (c[i - 1][1] + 1) % L[m]
            side = (c[(i + 1) % k][0] - o) % L[m]
            lo = (c[i][0] - o) % L[m]
            row.append((o, side, lo, lo + c[i][1] - c[i][0] + 1))
        per.append(row)
    boxes = [tuple(zip(a, b, c, d)) for a in per[0] for b in per[1] for c in per[2] for d in per[3]]
    return tuple(L), cores, boxes


def _sites(box):
    return math.prod(box[1])


def work(case):
    L, _, boxes = _geometry(case)
    V, R, k = math.prod(L), case["nrhs"], case["kind"]
    omega = sum(_sites(b) for b in boxes)
    links = 144.0 * 4 * V
    apply_flops = 1368.0 * omega * R
    field = 192.0 * omega * R
    if k == "stencil":
        return {"bytes": 2 * field + links, "flops": apply_flops}
    if k == "solve":
        return {"bytes": 2 * field + links, "flops": APPLICATIONS * apply_flops}
    planes = 1.0
    for m in range(4):
        n = len(case["cells"].split("/")[m].split(",")) if not case["cells"].split("/")[m].endswith("*") else 0
        planes *= 1.0 - min(1.0, 2.0 * n / L[m])
    chi = 192.0 * V * (1.0 - planes) * R
    if k in ("action", "w"):
        return {"bytes": (2 if k == "w" else 1) * chi + links, "flops": 2 * APPLICATIONS * apply_flops}
    force = 256.0 * V
    if k == "force":
        return {"bytes": chi + links + force, "flops": 3 * APPLICATIONS * apply_flops}
    if k == "md":
        return {"bytes": chi + 2 * links + 2 * force, "flops": (case["steps"] + 1) * 3 * APPLICATIONS * apply_flops}
    taps = sum(9 * a * b for a, b in zip(CHANNELS, CHANNELS[1:]))
    return {"bytes": 2 * field + links, "flops": 3 * 24.0 * taps * omega * R}


# ---- inputs -----------------------------------------------------------------------------------

def _generator(seed, tag):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 64 + tag)


def _gauss(gen, *shape):
    """Complex Gaussians with Re, Im ~ N(0, 1/2)."""
    return torch.view_as_complex(torch.randn(*shape, 2, generator=gen, device="cuda", dtype=torch.float64) * math.sqrt(0.5))


def _gell_mann():
    m = torch.zeros(8, 3, 3, dtype=torch.complex128)
    m[0, 0, 1] = m[0, 1, 0] = m[3, 0, 2] = m[3, 2, 0] = m[5, 1, 2] = m[5, 2, 1] = 1
    m[1, 0, 1] = m[4, 0, 2] = m[6, 1, 2] = -1j
    m[1, 1, 0] = m[4, 2, 0] = m[6, 2, 1] = 1j
    m[2, 0, 0], m[2, 1, 1] = 1, -1
    m[7] = torch.diag(torch.tensor([1, 1, -2], dtype=torch.complex128)) / math.sqrt(3.0)
    return m.cuda()


def _links(case, seed):
    """SU(3) links exp(i eps H), H = sum_a h_a lambda_a / 2, h_a ~ N(0, 1): [V, 4, 3, 3]."""
    V = math.prod(_geometry(case)[0])
    gen, lam, out = _generator(seed, 1), _gell_mann().reshape(8, 9), torch.empty(V * 4, 9, dtype=torch.complex128, device="cuda")
    for part in out.split(1 << 20):
        h = torch.randn(part.shape[0], 8, generator=gen, device="cuda", dtype=torch.float64)
        part.copy_(torch.linalg.matrix_exp(((0.5j * case["eps"] * h.to(torch.complex128)) @ lam).reshape(-1, 3, 3)).reshape(-1, 9))
    return out.reshape(V, 4, 3, 3)


def _context(case, seed):
    L, cores, _ = _geometry(case)
    ctx = dd4d.Context(L, case["kappa"])
    ctx.gauge_upload(_links(case, seed).reshape(*L, 4, 3, 3).cpu().numpy())
    ctx.set_geometry(cores)
    if case["csw"]:
        ctx.set_clover(case["csw"])
    return ctx


def _rhs(case, seed, tag=2):
    """Right-hand sides on every block, the layout of solve_blocks: [block][rhs][site][12]."""
    return _gauss(_generator(seed, tag), sum(_sites(b) for b in _geometry(case)[2]) * case["nrhs"] * 12)


def _n_dpi(case):
    L, cores, _ = _geometry(case)
    inside = 1
    for m in range(4):
        planes = {x for lo, hi in cores[m] for x in (lo, hi)}
        inside *= L[m] - len(planes)
    return math.prod(L) - inside


def _fields(case, seed):
    return _gauss(_generator(seed, 3), case["nrhs"], _n_dpi(case), 12)


def _roots(case):
    """u_k, k = 1..N/2 of the N = 2 nrhs roots at c = 0.5."""
    n = 2 * case["nrhs"]
    t = 2 * math.pi * np.arange(1, case["nrhs"] + 1) / (n + 1)
    return np.cos(t) + 1j * math.sqrt(0.75) * np.sin(t)


def _momenta(case, seed):
    V = math.prod(_geometry(case)[0])
    return torch.randn(V * 32, generator=_generator(seed, 4), device="cuda", dtype=torch.float64)


def _weights(seed):
    """Near-identity network weights of few significant bits, one [9, c_out, c_in] array per layer."""
    rng = np.random.default_rng(seed)
    out = []
    for a, b in zip(CHANNELS, CHANNELS[1:]):
        w = 0.08 / math.sqrt(a) * (rng.standard_normal((9, b, a)) + 1j * rng.standard_normal((9, b, a)))
        for c in range(min(a, b)):
            w[0, c, c] += 1.0
        out.append(np.round(w * 128) / 128)
    return out


def _real(t):
    return torch.view_as_real(t).reshape(-1).contiguous()


def prepare(case, seed):
    k = case["kind"]
    s = {"kind": k, "case": dict(case), "ctx": _context(case, seed)}
    s["ids"] = list(range(len(_geometry(case)[2])))
    inner = {"bf16": 1e-3}.get(case["prec"], 3e-6)
    s["prm"] = dd4d.params(TOL, inner_prec=case["prec"], inner_tol=inner, autotune=case["tune"], graph=case["graph"])
    if k in ("stencil", "solve"):
        s["b"] = _real(_rhs(case, seed))
        s["x"] = torch.zeros_like(s["b"])
    elif k == "net":
        s["b"] = _real(_rhs(case, seed))
        s["x"] = _real(_rhs(case, seed) + 0.3 * _rhs(case, seed, 5))
        s["net"] = dd4d.Net(s["ctx"], _weights(seed), CHANNELS)
    else:
        s["u"] = _roots(case)
        s["chi"] = _real(_fields(case, seed))
        if k == "w":
            s["w"] = torch.zeros_like(s["chi"])
        elif k == "force":
            s["F"] = torch.zeros(math.prod(_geometry(case)[0]) * 32, dtype=torch.float64, device="cuda")
        elif k == "md":
            eta = _real(_rhs(dict(case, nrhs=1), seed))
            s["phi"] = torch.zeros_like(eta)
            s["ctx"].pf_heatbath(eta, s["phi"])
            s["P0"] = _momenta(case, seed)
            s["P"] = torch.zeros_like(s["P0"])
            s["sign"] = 1.0
    return s


def run(s):
    k, case, ctx = s["kind"], s["case"], s["ctx"]
    if k == "stencil":
        ctx.apply_D_block("omega", s["ids"], case["nrhs"], s["b"], s["x"], case["prec"])
        return {"Db": s["x"]}
    if k == "solve":
        st = ctx.solve_blocks("omega", s["ids"], case["nrhs"], s["b"], s["x"], s["prm"])
        return {"x": s["x"], "status": st["status"]}
    if k == "action":
        S, S_block, S_r, status = ctx.multiboson_action(s["u"], s["chi"], s["prm"])
        return {"S": S, "S_block": S_block, "S_r": S_r, "status": status}
    if k == "w":
        status = ctx.apply_w(case["nrhs"], s["chi"], s["w"], s["prm"])
        return {"w": s["w"], "status": status}
    if k == "force":
        F, status = ctx.mb_force(s["u"], s["chi"], s["F"], s["prm"])
        return {"F": F, "status": status}
    if k == "md":
        # a short trajectory there, the next one back: the links stay near where they began
        torch.mul(s["P0"], s["sign"], out=s["P"])
        s["sign"] = -s["sign"]
        st = ctx.md_trajectory(s["u"], s["chi"], s["phi"], s["P"], 0.02 * case["steps"], case["steps"], s["prm"])
        return {"P": s["P"], "H0": st["H0"], "H1": st["H1"], "S_mb": st["s_mb1"], "S_pf": st["s_pf1"], "status": st["status"]}
    loss, grads = s["net"].loss_grad(s["ids"], case["nrhs"], s["b"], s["x"])
    return {"loss": loss, "grads": grads}


# ---- the same in 64 bits, in plain torch --------------------------------------------------------

def _gammas():
    s = torch.zeros(3, 2, 2, dtype=torch.complex128)
    s[0, 0, 1] = s[0, 1, 0] = 1
    s[1, 0, 1], s[1, 1, 0] = -1j, 1j
    s[2, 0, 0], s[2, 1, 1] = 1, -1
    g = torch.zeros(4, 4, 4, dtype=torch.complex128)
    g[0, :2, 2:] = g[0, 2:, :2] = -torch.eye(2)
    for k in range(3):
        g[k + 1, :2, 2:], g[k + 1, 2:, :2] = -1j * s[k], 1j * s[k]
    return g.cuda()


class _Lattice:
    """Links of the lattice and D restricted to boxes of it (periodic in space, antiperiodic in time)."""

    def __init__(self, case, seed):
        self.L, self.cores, self.boxes = _geometry(case)
        self.kappa, self.gamma = case["kappa"], _gammas()
        self.one = torch.eye(4, dtype=torch.complex128, device="cuda")
        U = _links(case, seed).reshape(*self.L, 4, 3, 3)
        self.A = self._clover(U, case["csw"]) if case["csw"] else None
        self.U = U.clone()
        self.U[-1, :, :, :, 0] *= -1
        self.U = self.U.reshape(-1, 4, 3, 3)

    def _clover(self, U, csw):
        A = torch.eye(12, dtype=torch.complex128, device="cuda").expand(*self.L, 12, 12).clone()
        at = lambda f, mu, n: torch.roll(f, -n, mu)  # noqa: E731
        for mu in range(4):
            for nu in range(mu + 1, 4):
                m, n = U[..., mu, :, :], U[..., nu, :, :]
                mm, nn = at(m, mu, -1), at(n, nu, -1)
                q = m @ at(n, mu, 1) @ at(m, nu, 1).mH @ n.mH
                q = q + n @ at(mm, nu, 1).mH @ at(n, mu, -1).mH @ mm
                q = q + mm.mH @ at(nn, mu, -1).mH @ at(mm, nu, -1) @ nn
                q = q + nn.mH @ at(m, nu, -1) @ at(nn, mu, 1) @ m.mH
                g = self.gamma
                sigma = 0.5j * (g[mu] @ g[nu] - g[nu] @ g[mu])
                A += 1j * self.kappa * csw * torch.einsum("st,...ab->...satb", sigma, (q - q.mH) / 8).reshape(*self.L, 12, 12)
        return A.reshape(-1, 12, 12)

    def index(self, origin, side):
        """Global site of every site of a box, in its own order."""
        x = torch.zeros(*side, dtype=torch.long, device="cuda")
        for m in range(4):
            c = (torch.arange(side[m], device="cuda") + origin[m]) % self.L[m]
            x = x * self.L[m] + c.reshape([-1 if k == m else 1 for k in range(4)])
        return x.reshape(-1)

    def wraps(self, whole=False):
        return [whole or not self.cores[m] for m in range(4)]

    def D(self, psi, side, idx, wrap):
        """D on a box: psi [R, n, 12] -> the same; hops out of it are dropped unless the direction wraps."""
        R = psi.shape[0]
        p = psi.reshape(R, *side, 4, 3)
        U = self.U[idx].reshape(*side, 4, 3, 3)
        out = p.clone() if self.A is None else (self.A[idx] @ psi.unsqueeze(-1)).reshape(p.shape)
        for mu in range(4):
            Um = U[..., mu, :, :]
            f, last, first = torch.roll(p, -1, mu + 1), self._face(mu, side[mu] - 1), self._face(mu, 0)
            if not wrap[mu]:
                f[last] = 0
            out -= self.kappa * ((self.one - self.gamma[mu]) @ (f @ Um.transpose(-1, -2)))
            b = torch.roll(p @ Um.conj(), 1, mu + 1)
            if not wrap[mu]:
                b[first] = 0
            out -= self.kappa * ((self.one + self.gamma[mu]) @ b)
        return out.reshape(R, -1, 12)

    @staticmethod
    def _face(mu, at):
        return (slice(None),) * (mu + 1) + (at,)

    def solve(self, b, side, idx, wrap, mask=None):
        """BiCGstab for D_X x = b to rounding, X the box or the sites of it that `mask` [n] keeps."""
        m = 1.0 if mask is None else mask.to(torch.float64)[None, :, None]
        op = lambda v: m * self.D(m * v, side, idx, wrap)  # noqa: E731
        dot = lambda u, v: (u.conj() * v).sum((1, 2), keepdim=True)  # noqa: E731
        div = lambda u, v: torch.where(v == 0, torch.zeros_like(u), u / torch.where(v == 0, torch.ones_like(v), v))  # noqa: E731
        x, r = torch.zeros_like(b), m * b
        h, p, rho, b2 = r.clone(), r.clone(), dot(r, r), dot(r, r).real
        for _ in range(400):
            v = op(p)
            alpha = div(rho, dot(h, v))
            s = r - alpha * v
            t = op(s)
            omega = div(dot(t, s), dot(t, t))
            x = x + alpha * p + omega * s
            r = s - omega * t
            if bool((dot(r, r).real <= 1e-28 * b2).all()):
                break
            new = dot(h, r)
            p = r + div(new, rho) * div(alpha, omega) * (p - omega * v)
            rho = new
        return x

    def ext(self, origin, side):
        """A box with one more layer of sites around it where it does not wrap, and where it lies in that one."""
        w = self.wraps()
        o = [origin[m] if w[m] else (origin[m] - 1) % self.L[m] for m in range(4)]
        d = [side[m] if w[m] else side[m] + 2 for m in range(4)]
        inner = torch.zeros(*d, dtype=torch.bool, device="cuda")
        inner[tuple(slice(None) if w[m] else slice(1, -1) for m in range(4))] = True
        return o, d, inner.reshape(-1)

    def core_mask(self, box):
        m = torch.zeros(*box[1], dtype=torch.bool, device="cuda")
        m[tuple(slice(a, b) for a, b in zip(box[2], box[3]))] = True
        return m.reshape(-1)

    def sets(self):
        """Sites of dPi (increasing), and for every site whether it lies on dPi and in a core."""
        core = torch.zeros(math.prod(self.L), dtype=torch.bool, device="cuda")
        for b in self.boxes:
            core[self.index(b[0], b[1])[self.core_mask(b)]] = True
        plane = torch.zeros(*self.L, dtype=torch.bool, device="cuda")
        for m in range(4):
            for lo, hi in self.cores[m]:
                plane[self._face(m - 1, lo)] = True
                plane[self._face(m - 1, hi)] = True
        plane = plane.reshape(-1)
        return torch.nonzero(plane).reshape(-1), plane, core

    def blocks_of(self, chi, frame=True):
        """(w chi as a lattice field, y_a = D_Omega^-1 D_{Omega,ext} chi' per block) for fields chi [f, V, 12] on dPi."""
        _, plane, core = self.sets()
        w, q = torch.zeros_like(chi), torch.zeros_like(chi)
        c = (plane & ~core)[None, :, None]
        wrap = self.wraps()
        if bool(c.any()):
            for b in self.boxes:
                idx, own = self.index(b[0], b[1]), self.core_mask(b)
                s = self.D(chi[:, idx] * own[None, :, None], b[1], idx, wrap) * ~own[None, :, None]
                q[:, idx] += self.solve(s, b[1], idx, wrap, ~own) * ~own[None, :, None]
            q = q * c
            if frame:
                every = torch.arange(math.prod(self.L), device="cuda")
                s = self.D(chi * core[None, :, None], self.L, every, self.wraps(True)) * ~core[None, :, None]
                w = c * (q - self.solve(s, self.L, every, self.wraps(True), ~core))
        ys, chi = [], chi - q
        for b in self.boxes:
            idx = self.index(b[0], b[1])
            o, d, inner = self.ext(b[0], b[1])
            big = self.index(o, d)
            s = self.D(chi[:, big] * ~inner[None, :, None], d, big, wrap)[:, inner]
            y = self.solve(s, b[1], idx, wrap)
            own = (self.core_mask(b) & plane[idx])[None, :, None]
            w[:, idx] -= y * own
            ys.append(y)
        return w, ys


def _on_lattice(lat, chi):
    at, _, _ = lat.sets()
    full = torch.zeros(chi.shape[0], math.prod(lat.L), 12, dtype=torch.complex128, device="cuda")
    full[:, at] = chi
    return full, at


def _exact_force(lat, chi, u):
    full, _ = _on_lattice(lat, chi)
    _, plane, _ = lat.sets()
    _, ys = lat.blocks_of(full, frame=False)
    V = math.prod(lat.L)
    F, T = torch.zeros(V, 4, 8, dtype=torch.float64, device="cuda"), _gell_mann() / 2
    g5 = torch.tensor([1.0] * 6 + [-1.0] * 6, dtype=torch.float64, device="cuda")
    wrap = lat.wraps()
    for b, y in zip(lat.boxes, ys):
        idx, own = lat.index(b[0], b[1]), lat.core_mask(b)
        r = (u[:, None, None] * full[:, idx] + y) * (own & plane[idx])[None, :, None]
        z = g5 * lat.solve(g5 * r, b[1], idx, wrap)
        shape = (-1, *b[1], 4, 3)
        yb, zb, U = y.reshape(shape), z.reshape(shape), lat.U[idx].reshape(*b[1], 4, 3, 3)
        box = own.reshape(b[1])
        for mu in range(4):
            Um = U[..., mu, :, :].transpose(-1, -2)
            up, uz = torch.roll(yb, -1, mu + 1) @ Um, torch.roll(zb, -1, mu + 1) @ Um
            M = torch.einsum("r...sa,st,r...tb->...ab", zb.conj(), lat.one - lat.gamma[mu], up)
            M = M - torch.einsum("r...sa,st,r...tb->...ab", uz.conj(), lat.one + lat.gamma[mu], yb)
            both = box & torch.roll(box, -1, mu)
            if not wrap[mu]:
                both[lat._face(mu - 1, b[1][mu] - 1)] = False
            f = -2 * lat.kappa * torch.einsum("tab,...ab->...t", T, M).imag * both[..., None]
            F[idx, mu] += f.reshape(-1, 8)
    return F.reshape(-1)


def _exact_net(lat, case, seed):
    W = [torch.from_numpy(w).cuda().requires_grad_() for w in _weights(seed)]
    R, wrap, total, at = case["nrhs"], lat.wraps(), 0.0, 0
    b = _rhs(case, seed)
    x = b + 0.3 * _rhs(case, seed, 5)
    systems = R * len(lat.boxes)
    for box in lat.boxes:
        n, side = _sites(box), box[1]
        U = lat.U[lat.index(box[0], side)].reshape(*side, 4, 3, 3)
        phi = b[at:at + 12 * n * R].reshape(R, *side, 4, 3)
        want = x[at:at + 12 * n * R].reshape(R, *side, 4, 3)
        at += 12 * n * R
        for w in W:
            taps = [phi]
            for mu in range(4):
                f = torch.roll(phi, -1, mu + 1).clone()
                if not wrap[mu]:
                    f[lat._face(mu, side[mu] - 1)] = 0
                taps.append(f @ U[..., mu, :, :].transpose(-1, -2))
            for mu in range(4):
                g = torch.roll(phi @ U[..., mu, :, :].conj(), 1, mu + 1).clone()
                if not wrap[mu]:
                    g[lat._face(mu, 0)] = 0
                taps.append(g)
            phi = sum(w[d] @ taps[d] for d in range(9))
        off = (phi - want).abs().square().flatten(1).sum(1)
        loss = (off / want.abs().square().flatten(1).sum(1)).sum() / systems
        loss.backward()
        total += float(loss.detach())
    return {"loss": total, "grads": [w.grad.cpu().numpy() for w in W]}


def exact(case, seed):
    L, _, boxes = _geometry(case)
    k, R = case["kind"], case["nrhs"]
    omega = sum(_sites(b) for b in boxes) * R
    if k == "md" or omega > {"stencil": 8e6, "net": 5e5}.get(k, 1.5e6) or len(boxes) > (100 if k == "stencil" else 40):
        return None          # a trajectory, or more solves than 20 seconds hold
    lat = _Lattice(case, seed)
    if k in ("stencil", "solve"):
        b, out, at = _rhs(case, seed), [], 0
        for box in boxes:
            n, idx = _sites(box), lat.index(box[0], box[1])
            v = b[at:at + 12 * n * R].reshape(R, n, 12)
            at += 12 * n * R
            out.append((lat.D(v, box[1], idx, lat.wraps()) if k == "stencil" else lat.solve(v, box[1], idx, lat.wraps())).reshape(-1))
        return {"Db" if k == "stencil" else "x": _real(torch.cat(out))}
    if k == "net":
        return _exact_net(lat, case, seed)
    chi, u = _fields(case, seed), torch.from_numpy(_roots(case)).cuda()
    if k == "force":
        return {"F": _exact_force(lat, chi, u)}
    full, at = _on_lattice(lat, chi)
    w, _ = lat.blocks_of(full)
    if k == "w":
        return {"w": _real(w[:, at])}
    s = (u[:, None, None] * full - w).abs().square().sum((0, 2))
    _, plane, core = lat.sets()
    per = [float(s[lat.index(b[0], b[1])[lat.core_mask(b)]][plane[lat.index(b[0], b[1])[lat.core_mask(b)]]].sum()) for b in boxes]
    rest = float(s[plane & ~core].sum())
    return {"S": sum(per) + rest, "S_block": np.array(per), "S_r": rest}
