"""The work that programs have this package do, as timed cases.

A program builds a `Plan` for its mesh once, keeps it, and then evaluates magnetisations on it: one
state at a time in a relaxation, many states at once in a service, several meshes in one submission,
inside the LLG stepper, from host or device memory.  Each case names one such use:

  entry   the public entry point: "eval" (Plan.eval), "energy" (Plan.eval then Plan.energy), "multi"
          (eval_multi_into), "host" (Plan.eval_host on pinned host buffers), "llg" (Plan.llg_rk4)
  mesh    "cube" (Kuhn cube, n cells an edge), "ball" (Delaunay ball, spacing h), "film" (Kuhn film,
          n x n/2 x 2 cells), "batch" (n meshes of uneven size, cubes, balls and ellipsoids)
  p, leaf, precision, near, batch
          the plan's options: expansion order, tets per leaf, arithmetic, stored (1) or integrated
          (0) near field, states in one call

`exact` is the defining integral itself, in FP64 on the faces of the mesh: with a continuous,
piecewise affine M the face charges of two tets sharing a face cancel, so
    4 pi u(r) = sum over boundary faces int (M.n) / R dS  -  sum over tets div M int 1 / R dV,
both in closed form (Wilton et al. 1984).  It holds no truncation, so the difference of a case from
it is the FMM's truncation error together with rounding.
"""
import functools
import math

import numpy as np
import torch

from paper_1606_00247_gb300 import inputs
from paper_1606_00247_gb300.api import Plan, eval_multi_into

THETA = 0.5
DEVICE = "cuda"
FILM_SIZE = (2000.0, 1000.0, 10.0)


# ---------------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------------
def _case(name, entry, mesh, size, p, leaf, precision, near, batch):
    c = dict(entry=entry, mesh=mesh, size=size, p=p, leaf=leaf, precision=precision, near=near, batch=batch)
    return dict(name=name, **c) if name else c


def listed():
    return [
        # a first script: a small cube with the library's default options, one state (FP64, near field
        # integrated in every call); latency
        _case("cube_default_b1", "eval", "cube", 8, 4, 32, "fp64", 0, 1),
        # FP64 on a plan too short-lived to store near-field coefficients: three states of a ball
        _case("ball_integrated_b3", "eval", "ball", 0.12, 8, 128, "fp64", 0, 3),
        # the FP64 reference evaluation of a production mesh that mixed results are checked against
        _case("ball_fp64_b1", "eval", "ball", 0.0505, 8, 128, "fp64", 1, 1),
        # a batched FP64 study on a small mesh (hysteresis samples)
        _case("ball_fp64_b16", "eval", "ball", 0.1, 8, 128, "fp64", 1, 16),
        # FP32 arithmetic at a lower order, an odd number of states
        _case("ball_fp32_b37", "eval", "ball", 0.1, 6, 64, "fp32", 1, 37),
        # one state of a production mesh with its energy: the inner call of a minimiser
        _case("ball_bf16x3_energy_b1", "energy", "ball", 0.0505, 8, 128, "bf16x3", 1, 1),
        # a service's ordinary batch, ragged against the 128-state tiles
        _case("ball_bf16x3_b83", "eval", "ball", 0.075, 8, 128, "bf16x3", 1, 83),
        # a service's largest batch
        _case("ball_bf16x3_b256", "eval", "ball", 0.0505, 8, 128, "bf16x3", 1, 256),
        # a thin film with flux-closure domains, two states (a step and its trial step)
        _case("film_bf16x3_b2", "eval", "film", 288, 8, 128, "bf16x3", 1, 2),
        # several meshes of uneven size, one state each, in one submission
        _case("meshes_bf16x3_b1", "multi", "batch", 6, 8, 128, "bf16x3", 1, 1),
        # host arrays in and out through pinned memory
        _case("ball_host_b24", "host", "ball", 0.1, 8, 128, "bf16x3", 1, 24),
        # dynamics: one Runge-Kutta step of sixteen states (four evaluations)
        _case("ball_llg_b16", "llg", "ball", 0.1, 8, 128, "bf16x3", 1, 16),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    entry = rng.choice(["integrated", "fp64", "fp64", "mixed", "mixed", "mixed", "mixed", "film", "multi", "host", "llg"])
    h = round(_log_uniform(rng, 0.0505, 0.14), 4)
    if entry == "integrated":
        if rng.random() < 0.4:
            return _case(None, "eval", "cube", rng.randint(3, 11), rng.choice([4, 6]), rng.choice([16, 32, 64]), "fp64",
                         0, rng.randint(1, 3))
        return _case(None, "eval", "ball", round(rng.uniform(0.12, 0.2), 4), rng.choice([4, 6, 8]),
                     rng.choice([32, 64, 128]), "fp64", 0, rng.randint(1, 3))
    if entry == "fp64":
        h = max(h, 0.07) if rng.random() < 0.7 else h
        top = 16 if h > 0.09 else (4 if h > 0.065 else 1)
        return _case(None, "eval", "ball", h, rng.choice([4, 5, 6, 8]), 128, "fp64", 1, round(_log_uniform(rng, 1, top)))
    if entry == "film":
        return _case(None, "eval", "film", rng.choice([96, 130, 192, 250, 288]), rng.choice([6, 8]), 128, "bf16x3", 1,
                     rng.randint(1, 12))
    if entry == "multi":
        return _case(None, "multi", "batch", rng.randint(2, 6), rng.choice([6, 8]), 128, "bf16x3", 1, rng.randint(1, 3))
    if entry == "host":
        return _case(None, "host", "ball", max(h, 0.075), 8, 128, "bf16x3", 1, round(_log_uniform(rng, 1, 48)))
    if entry == "llg":
        return _case(None, "llg", "ball", max(h, 0.075), rng.choice([6, 8]), 128, "bf16x3", 1,
                     round(_log_uniform(rng, 1, 48)))
    precision = rng.choice(["fp32", "tf32", "bf16x3", "bf16x3", "bf16x3", "bf16x6"])
    p = rng.choice([4, 6, 8, 8]) if precision != "fp32" else rng.choice([4, 5, 6])
    leaf = 128 if p == 8 or h < 0.08 else rng.choice([64, 128])
    top = 256 if precision == "bf16x3" else (128 if h > 0.07 else 24)
    return _case(None, rng.choice(["eval", "eval", "energy"]), "ball", h, p, leaf, precision, 1,
                 round(_log_uniform(rng, 1, top)))


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=32)
def _meshes(kind, size):
    if kind == "cube":
        return (inputs.unit_cube(size),)
    if kind == "ball":
        return (inputs.sphere(h=size),)
    if kind == "film":
        return (inputs.thin_film(size, size // 2, 2, size=FILM_SIZE),)
    return tuple(inputs.batch_meshes(n=size, min_tets=3e3, max_tets=6e4))


def _textures(nodes, batch, seed):
    """Unit vectors (batch, N, 3): a few long waves of random direction and phase, and a tilt of
    every node, normalised (smooth magnetisation with thermal noise)."""
    g = torch.Generator(DEVICE).manual_seed(int(seed))
    x = torch.as_tensor(nodes, device=DEVICE)
    x = (x - x.mean(0)) / (x.max(0).values - x.min(0).values).max()
    m = 0.1 * torch.randn((batch, x.shape[0], 3), dtype=torch.float64, device=DEVICE, generator=g)
    for _ in range(4):
        q = 6.0 * torch.randn((batch, 1, 3), dtype=torch.float64, device=DEVICE, generator=g)
        a = torch.randn((batch, 1, 3), dtype=torch.float64, device=DEVICE, generator=g)
        ph = 6.3 * torch.rand((batch, 1), dtype=torch.float64, device=DEVICE, generator=g)
        m += a * torch.cos((x[None] * q).sum(-1) + ph)[..., None]
    return m / m.norm(dim=-1, keepdim=True)


def _states(case, seed):
    """One (batch, N, 3) magnetisation per mesh of the case."""
    out = []
    for k, (nodes, _) in enumerate(_meshes(case["mesh"], case["size"])):
        if case["mesh"] == "film":
            m = np.stack([inputs.landau_m(nodes, size=FILM_SIZE[:2], seed=1000 * seed + b) for b in range(case["batch"])])
            out.append(torch.as_tensor(m, device=DEVICE))
        else:
            out.append(_textures(nodes, case["batch"], 1000 * seed + k))
    return out


LLG = dict(Ms=1.0, alpha=0.1, h_ext=(0.0, 0.02, 0.1), dt=0.05, steps=1)


def prepare(case, seed):
    s = {"case": case, "M": _states(case, seed)}
    s["plans"] = [Plan(nodes, tets, p=case["p"], leaf_size=case["leaf"], theta=THETA, precision=case["precision"],
                       near_mode=case["near"], max_batch=case["batch"], device=DEVICE)
                  for nodes, tets in _meshes(case["mesh"], case["size"])]
    if case["entry"] == "multi":  # the outputs of a submission are kept, as its captured work is
        s["u"] = [torch.empty(m.shape[:2], dtype=torch.float64, device=DEVICE) for m in s["M"]]
        s["H"] = [torch.empty_like(m) for m in s["M"]]
    if case["entry"] == "host":
        m = s["M"][0]
        s["M"] = [m.cpu().pin_memory().numpy()]
        s["u"] = torch.empty(m.shape[:2], dtype=torch.float64, pin_memory=True).numpy()
        s["H"] = torch.empty(m.shape, dtype=torch.float64, pin_memory=True).numpy()
    return s


def run(state):
    entry, plan, m = state["case"]["entry"], state["plans"][0], state["M"][0]
    if entry == "multi":
        u, h = eval_multi_into(state["plans"], state["M"], state["u"], state["H"])
        return {"u": u, "H": h}
    if entry == "host":
        u, h = plan.eval_host(m, u=state["u"], H=state["H"])
        return {"u": u, "H": h}
    if entry == "llg":  # from the same start each time: the stepper advances its argument
        return {"m": plan.llg_rk4(m.clone(), **LLG)}
    u, h = plan.eval(m)
    if entry == "energy":
        return {"u": u, "H": h, "e": plan.energy(m, h)}
    return {"u": u, "H": h}


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
def work(case):
    """M read, u and H written, the stored coefficients read (12 B a coefficient vector in 32 bits,
    24 B in FP64), and the operations of the method: 2 C(p+6, 6) per M2L pair and state, C(p+3, 3)
    multiply-adds per node for P2M (3 components) and L2P, 6 per stored coefficient vector and state,
    250 per integrated (node, tet) pair.  Near and far pairs by the volume rule of theta = 0.5: a node's
    near region holds the nodes of ~310 boxes (a ball of 4.2 box sides; 55 in a film), a cell takes
    ~290 far cells (60 in a film)."""
    p, leaf, b = case["p"], case["leaf"], case["batch"]
    reps = 4 * LLG["steps"] if case["entry"] == "llg" else 1
    nbytes = flops = 0.0
    film = case["mesh"] == "film"
    for nodes, tets in _meshes(case["mesh"], case["size"]):
        n, t = nodes.shape[0], tets.shape[0]
        near = min(n, (55 if film else 310) * leaf / 3.0 * n / t)
        cells = 1.7 * t / leaf
        nbytes += b * n * 56
        flops += b * (cells * min(cells, 60 if film else 290) * 2 * math.comb(p + 6, 6) + 8 * n * math.comb(p + 3, 3))
        if case["near"]:
            nbytes += n * near * (24 if case["precision"] == "fp64" else 12)
            flops += 6.0 * n * near * b
        else:
            flops += 250.0 * n * near * t / n
    return {"bytes": int(reps * nbytes), "flops": int(reps * flops)}


def tolerance(case):
    """Four times the largest difference seen, over the listed and drawn cases, between a result and
    another evaluation with the same tree and order: FP64 against a plain C FMM on the CPU, which takes
    the near field from the face charges instead (up to 2.1e-14), the other precisions against FP64.
    A film's flux-closure domains cancel more than the balls' textures, and the stepper's state moves
    by dt times the field only."""
    if case["entry"] == "llg":
        return {"rel": 2e-7}
    if case["mesh"] == "film":
        return {"rel": 1.2e-4}
    return {"rel": {"fp64": 1e-13, "fp32": 6e-6, "tf32": 1.6e-3, "bf16x3": 3e-5, "bf16x6": 6e-6}[case["precision"]]}


# ---------------------------------------------------------------------------------------------
# the definition in FP64
# ---------------------------------------------------------------------------------------------
EXACT_PAIRS = 2e10  # (node, face) pairs times evaluations, up to which the definition is summed


class _Direct:
    """u = W M by the boundary-face and volume charges of one mesh."""

    def __init__(self, nodes, tets):
        self.x = torch.as_tensor(nodes, dtype=torch.float64, device=DEVICE)
        t = torch.as_tensor(tets, dtype=torch.int64, device=DEVICE)
        x = self.x
        e1, e2, e3 = (x[t[:, k]] - x[t[:, 0]] for k in (1, 2, 3))
        det = (e1 * torch.linalg.cross(e2, e3)).sum(-1)
        t = torch.where((det < 0)[:, None], t[:, [0, 1, 3, 2]], t)
        e1, e2, e3 = (x[t[:, k]] - x[t[:, 0]] for k in (1, 2, 3))
        det = det.abs()[:, None]
        g = torch.stack([torch.linalg.cross(e2, e3), torch.linalg.cross(e3, e1), torch.linalg.cross(e1, e2)], 1) / det[:, None]
        self.grad = torch.cat([-g.sum(1, keepdim=True), g], 1)  # (T, 4, 3) gradients of the hat functions
        self.vol, self.tets = det[:, 0] / 6.0, t
        faces = torch.cat([t[:, f] for f in ([1, 2, 3], [0, 3, 2], [0, 1, 3], [0, 2, 1])])  # outward
        owner = torch.arange(t.shape[0], device=DEVICE).repeat(4)
        key, inv = torch.unique(faces.sort(1).values, dim=0, return_inverse=True)
        order = torch.argsort(inv, stable=True)
        first = torch.searchsorted(inv[order], torch.arange(key.shape[0], device=DEVICE))
        self.face, self.own = faces[order[first]], owner[order[first]]
        nxt = (first + 1).clamp(max=inv.shape[0] - 1)
        two = (inv[order[nxt]] == torch.arange(key.shape[0], device=DEVICE)) & (first + 1 < inv.shape[0])
        self.other = torch.where(two, owner[order[nxt]], torch.full_like(self.own, -1))
        self.bnd = torch.nonzero(~two)[:, 0]
        v = x[self.face]  # (F, 3, 3)
        n = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
        self.area2 = n.norm(dim=-1)
        self.n = n / self.area2[:, None]
        ev = self.face[:, [[0, 1], [1, 2], [2, 0]]]  # (F, 3 edges, 2)
        self.edge, self.fe = torch.unique(ev.sort(-1).values.reshape(-1, 2), dim=0, return_inverse=True)
        self.fe = self.fe.reshape(-1, 3)
        self.len = (x[self.edge[:, 1]] - x[self.edge[:, 0]]).norm(dim=-1)
        d = x[ev[..., 1]] - x[ev[..., 0]]
        self.t = d / d.norm(dim=-1, keepdim=True)
        self.m = torch.linalg.cross(self.t, self.n[:, None].expand(-1, 3, -1))  # outward in the face's plane
        self.p = x[ev[..., 0]]
        self.elen = d.norm(dim=-1)

    def charges(self, M):
        """Jump of div M over every face (F, B), M (B, N, 3)."""
        div = torch.zeros((M.shape[0], self.tets.shape[0]), dtype=torch.float64, device=DEVICE)
        for k in range(4):
            div += (M[:, self.tets[:, k]] * self.grad[None, :, k]).sum(-1)
        jump = div[:, self.own] - torch.where(self.other >= 0, div[:, self.other.clamp(min=0)], 0.0)
        return jump.T.contiguous()

    def parts(self, r):
        """For targets r (C, 3): a I_F over all faces (C, F), and int lambda_k / R over the boundary
        faces (C, 3, boundary)."""
        R = torch.cdist(r, self.x, compute_mode="donot_use_mm_for_euclid_dist")
        s = R[:, self.edge[:, 0]] + R[:, self.edge[:, 1]]
        gap = s - self.len
        # ln((R+ + R- + l) / (R+ + R- - l)); its factor vanishes on the edge itself
        L = torch.where(gap > 1e-13 * self.len, torch.log1p(2.0 * self.len / gap.clamp(min=1e-300)), 0.0)
        a = (self.n * self.p[:, 0]).sum(-1) - r @ self.n.T
        I = torch.zeros_like(a)
        for e in range(3):
            I += ((self.m[:, e] * self.p[:, e]).sum(-1) - r @ self.m[:, e].T) * L[:, self.fe[:, e]]
        R1, R2, R3 = (R[:, self.face[:, k]] for k in range(3))
        l = self.len[self.fe]
        den = R1 * R2 * R3 + 0.5 * ((R1 * R1 + R2 * R2 - l[:, 0] ** 2) * R3 + (R2 * R2 + R3 * R3 - l[:, 1] ** 2) * R1
                                    + (R3 * R3 + R1 * R1 - l[:, 2] ** 2) * R2)
        I -= 2.0 * a.abs() * torch.atan2(a.abs() * self.area2, den)
        b = self.bnd
        lin = torch.zeros((r.shape[0], b.shape[0], 3), dtype=torch.float64, device=DEVICE)  # int (r' - r_proj) / R
        h = a[:, b]
        for e in range(3):
            rel = self.p[b, e][None] - r[:, None]
            d = (rel * self.m[b, e]).sum(-1)
            sm = (rel * self.t[b, e]).sum(-1)
            i0, i1 = self.face[b, e], self.face[b, (e + 1) % 3]
            v = (d * d + h * h) * L[:, self.fe[b, e]] + (sm + self.elen[b, e]) * R[:, i1] - sm * R[:, i0]
            lin += 0.5 * v[..., None] * self.m[b, e]
        lam = []
        for k in range(3):
            opp = (k + 1) % 3  # the edge opposite vertex k runs from vertex k + 1 to vertex k + 2
            grad = -self.m[b, opp] * (self.elen[b, opp] / self.area2[b])[:, None]
            at = ((r[:, None] - self.p[b, opp][None]) * grad).sum(-1)  # lambda_k at the projection of r
            lam.append(at * I[:, b] + (lin * grad).sum(-1))
        return a * I, torch.stack(lam, 1)

    def potential(self, M):
        jump = self.charges(M)
        sig = torch.stack([(M[:, self.face[self.bnd, k]] * self.n[self.bnd]).sum(-1) for k in range(3)], 1)  # (B, 3, b)
        sig = sig.reshape(M.shape[0], -1).T.contiguous()
        u = torch.empty(M.shape[:2], dtype=torch.float64, device=DEVICE)
        step = max(1, int(6e7 // self.face.shape[0]))
        for i in range(0, self.x.shape[0], step):
            vol, lam = self.parts(self.x[i:i + step])
            u[:, i:i + step] = ((lam.reshape(lam.shape[0], -1) @ sig - 0.5 * (vol @ jump)) / (4.0 * math.pi)).T
        return u

    def field(self, u):
        """The mass-lumped -grad u at the nodes."""
        g = torch.zeros((u.shape[0], self.tets.shape[0], 3), dtype=torch.float64, device=DEVICE)
        for k in range(4):
            g += u[:, self.tets[:, k], None] * self.grad[None, :, k]
        g *= self.vol[:, None]
        H = torch.zeros(u.shape + (3,), dtype=torch.float64, device=DEVICE)
        V = torch.zeros(self.x.shape[0], dtype=torch.float64, device=DEVICE)
        for k in range(4):
            H.index_add_(1, self.tets[:, k], g)
            V.index_add_(0, self.tets[:, k], self.vol)
        return -H / V[None, :, None], V


def _llg_exact(D, m):
    hx = torch.tensor(LLG["h_ext"], dtype=torch.float64, device=DEVICE)

    def rhs(y):
        h = D.field(D.potential(LLG["Ms"] * y))[0] / LLG["Ms"] + hx
        c = torch.linalg.cross(y, h)
        return -(c + LLG["alpha"] * torch.linalg.cross(y, c)) / (1.0 + LLG["alpha"] ** 2)

    dt = LLG["dt"]
    for _ in range(LLG["steps"]):
        k1 = rhs(m)
        k2 = rhs(m + 0.5 * dt * k1)
        k3 = rhs(m + 0.5 * dt * k2)
        k4 = rhs(m + dt * k3)
        m = m + dt / 6.0 * (k1 + 2.0 * k2 + 2.0 * k3 + k4)
        m = m / m.norm(dim=-1, keepdim=True)
    return m


def exact(case, seed):
    meshes = _meshes(case["mesh"], case["size"])
    pairs = sum(2.0 * nodes.shape[0] * tets.shape[0] for nodes, tets in meshes)
    if pairs * (4 if case["entry"] == "llg" else 1) * (1.0 + case["batch"] / 256.0) > EXACT_PAIRS:
        return None
    us, hs = [], []
    for (nodes, tets), M in zip(meshes, _states(case, seed)):
        D = _Direct(nodes, tets)
        if case["entry"] == "llg":
            return {"m": _llg_exact(D, M)}
        u = D.potential(M)
        H, V = D.field(u)
        us.append(u)
        hs.append(H)
    if case["entry"] == "multi":
        return {"u": us, "H": hs}
    out = {"u": us[0], "H": hs[0]}
    if case["entry"] == "energy":  # the lumped volume of a node is a quarter of the tets around it
        out["e"] = -0.5 * 0.25 * (V[None, :, None] * M * H).sum((1, 2))
    return out
