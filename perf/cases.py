"""Measured workloads of the solver, through its public entry points (paper_2209_01877_gb300.dg and
.adjoint), with a plain 64-bit torch evaluation of what each of them returns.

A case is one call sequence of a user's program on one mesh:

  step      set the state, take n SSP-RK3 steps, read the state back
  march     one step of a monitored run: set the state, the stable time step, one SSP-RK3 step, the
            conserved totals and kinetic energy, the boundary flux, the status check, the state
  ns_step   set the state, take n SSP-RK3 steps of the Navier-Stokes equations, read the state back
  residual  the semi-discrete right-hand side of a caller's state
  vjp       the vector-Jacobian product of the residual
  adjoint   the checkpointed gradient of the final kinetic energy with respect to the initial state

Meshes are the seeded Kuhn-split boxes of paper_2209_01877_gb300.inputs: a periodic unit cube, or a
channel with slip walls and far-field ends.  The state is an isentropic vortex (cube) or a density
pulse in a Mach 0.3 stream (channel), projected onto the basis, with a 1% perturbation per element;
position and perturbation come from the seed.  The time step is CFL 0.1.

Values that the library holds in 32 bits (states of FP32 meshes, residuals of FP32 and mixed meshes)
are returned in 32 bits; states of the mixed forms (float-float) and of FP64 meshes in 64.
"""
import functools
import itertools
import math

import numpy as np
import torch

from paper_2209_01877_gb300 import adjoint, dg
from paper_2209_01877_gb300 import inputs as I

PREC = {"fp64": dg.DG_FP64, "fp32": dg.DG_FP32, "f16": dg.DG_MIXED_FP16, "bf16": dg.DG_MIXED_BF16}
FLUX = {"rusanov": dg.DG_RUSANOV, "roe": dg.DG_ROE}
ORDER = {"rcm": dg.DG_ORDER_RCM, "morton": dg.DG_ORDER_MORTON, "hilbert": dg.DG_ORDER_HILBERT}
NB, NQ, NQF = {1: 4, 2: 10, 3: 20}, {1: 4, 2: 14, 3: 24}, {1: 3, 2: 6, 3: 12}
GAMMA, CFL, MU, PRANDTL = 1.4, 0.1, 1e-3, 0.72


def _case(name, kind, p, prec, flux, dims, order, box=False, n=1, conservative=False):
    c = dict(kind=kind, p=p, prec=prec, flux=flux, nx=dims[0], ny=dims[1], nz=dims[2], order=order, box=box, n=n,
             conservative=conservative)
    return dict(c, name=name) if name else c


def listed():
    return [
        # a small first-order mesh in double precision: the launch-bound time loop
        _case("step_p1_fp64_small", "step", 1, "fp64", "rusanov", (6, 6, 6), "rcm", n=10),
        # a mid-sized first-order run in mixed precision (still replayed as a graph)
        _case("step_p1_f16", "step", 1, "f16", "rusanov", (20, 20, 20), "morton", n=16),
        # single precision, second order, renumbered by RCM: the FP32 throughput workload
        _case("step_p2_fp32", "step", 2, "fp32", "rusanov", (48, 48, 48), "rcm", n=2),
        # double precision, third order, Roe: the FP64 reference run
        _case("step_p3_fp64", "step", 3, "fp64", "roe", (32, 32, 32), "morton"),
        # mixed precision, third order, Roe, the largest mesh: the production run
        _case("step_p3_f16", "step", 3, "f16", "roe", (64, 64, 64), "morton", n=2),
        # one monitored step of a channel with walls and far field, cell averages kept conservative
        _case("march_p3_f16_box", "march", 3, "f16", "roe", (48, 24, 24), "morton", box=True, conservative=True),
        # the same loop in double precision on a small channel: latency of the diagnostics
        _case("march_p2_fp64_box", "march", 2, "fp64", "roe", (24, 12, 12), "rcm", box=True),
        # viscous time stepping in double precision
        _case("ns_p2_fp64", "ns_step", 2, "fp64", "rusanov", (32, 32, 32), "morton"),
        # viscous time stepping in single precision with no-slip walls
        _case("ns_p3_fp32_box", "ns_step", 3, "fp32", "roe", (40, 20, 20), "morton", box=True, n=2),
        # the right-hand side alone in bf16 pairs on a mesh of odd extents (a ragged last tile)
        _case("residual_p3_bf16", "residual", 3, "bf16", "roe", (31, 29, 23), "hilbert"),
        # one adjoint application in single precision on a small ragged mesh
        _case("vjp_p3_fp32", "vjp", 3, "fp32", "roe", (17, 13, 11), "rcm"),
        # the checkpointed gradient over four steps: forward steps and their reverse
        _case("adjoint_p2_fp64", "adjoint", 2, "fp64", "rusanov", (32, 32, 32), "morton", n=4),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "march", "ns_step", "residual", "vjp", "adjoint"])
    prec = rng.choice(["fp64", "fp32"] if kind in ("vjp", "adjoint") else ["fp64", "fp32", "f16", "bf16"])
    p, box = rng.choice([1, 2, 3]), rng.random() < 0.4
    top = {"adjoint": 40_000, "ns_step": 120_000}.get(kind, 200_000)   # elements
    cells = math.exp(rng.uniform(math.log(60), math.log(top / 6)))
    a, b = math.exp(rng.uniform(-0.4, 0.4)), math.exp(rng.uniform(-0.4, 0.4))
    s = (cells / (a * b)) ** (1 / 3)
    dims = [min(64, max(3, int(round(x)))) for x in (a * s, b * s, s)]
    n = {"step": rng.choice([1, 2, 9]) if cells < 2000 else 1, "ns_step": 1, "adjoint": 3}.get(kind, 1)
    return _case(None, kind, p, prec, rng.choice(["rusanov", "roe"]), dims, rng.choice(["rcm", "morton", "hilbert"]), box, n,
                 kind == "march" and prec in ("f16", "bf16") and rng.random() < 0.5)


# ---- inputs ---------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=2)
def _host_mesh(nx, ny, nz, box):
    if box:
        return I.make_box_channel(nx, ny, nz, jitter=0.15)
    return I.make_box_mesh((nx, ny, nz), jitter=0.12)


def _mesh_arrays(case):
    return _host_mesh(case["nx"], case["ny"], case["nz"], case["box"])


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _cons(rho, u, v, w, p):
    return torch.stack([rho, rho * u, rho * v, rho * w, p / (GAMMA - 1) + 0.5 * rho * (u * u + v * v + w * w)], -1)


def _field(case, x, g):
    """Pointwise conserved state at x [..., 3]; its position from the generator."""
    r = torch.rand(3, generator=g, dtype=torch.float64).tolist()
    one = torch.ones_like(x[..., 0])
    if case["box"]:
        c = (0.6 + 0.8 * r[0], 0.35 + 0.3 * r[1], 0.35 + 0.3 * r[2])
        r2 = sum((x[..., d] - c[d]) ** 2 for d in range(3))
        rho = 1 + 0.1 * torch.exp(-r2 / 0.05 ** 2)
        v, w = (0.05 * (t - 0.5) * one for t in torch.rand(2, generator=g, dtype=torch.float64).tolist())   # a slight cross-flow
        return _cons(rho, 0.3 * math.sqrt(GAMMA) * one, v, w, one)
    rad = min(0.2, max(1 / 16, 1.5 / min(case["nx"], case["ny"])))
    d = [x[..., k] - (0.3 + 0.4 * r[k]) for k in (0, 1)]
    dx, dy = (t - torch.round(t) for t in d)
    e = torch.exp(0.5 * (1 - (dx * dx + dy * dy) / rad ** 2))
    beta = 5.0
    T = 1 - (GAMMA - 1) * beta ** 2 / (8 * GAMMA * math.pi ** 2) * e * e
    rho = T ** (1 / (GAMMA - 1))
    return _cons(rho, 0.5 * math.sqrt(GAMMA) - beta / (2 * math.pi) * dy / rad * e, beta / (2 * math.pi) * dx / rad * e, 0 * one,
                 rho ** GAMMA)


def _inputs(case, seed):
    """The state U [ne, 5, nb], the direction lam (vjp) and the time step, from the seed alone."""
    m, p, dev = _mesh_arrays(case), case["p"], _device()
    g = torch.Generator().manual_seed(int(seed) % (1 << 62))
    X, w, phi, _ = _volume(p)
    xyz = torch.from_numpy(m.tet_xyz).to(dev)
    J = (xyz[:, 1:] - xyz[:, :1]).transpose(1, 2)                     # columns: edges from vertex 0
    X, w, phi = (torch.from_numpy(t).to(dev) for t in (X, w, phi))
    U = torch.empty(m.ne, 5, NB[p], dtype=torch.float64, device=dev)
    state = g.get_state()
    for s in range(0, m.ne, 1 << 18):
        x = xyz[s:s + (1 << 18), None, 0] + torch.einsum("edk,qk->eqd", J[s:s + (1 << 18)], X)
        g.set_state(state)
        U[s:s + (1 << 18)] = torch.einsum("q,eqv,qj->evj", w, _field(case, x, g), phi)
    xi = (2 * torch.rand(2, m.ne, generator=g, dtype=torch.float64) - 1).to(dev)
    a, b = 1 + 0.01 * xi[0], 1 + 0.01 * xi[1]
    U[:, 0] *= a[:, None]
    U[:, 1:4] *= (a * b)[:, None, None]
    lam = None
    if case["kind"] == "vjp":
        lam = torch.randn(U.shape, generator=g, dtype=torch.float64).to(dev)
    return U, lam, _stable_dt(p, U, xyz)


def _stable_dt(p, U, xyz):
    """CFL min_e h_e / ((2p+1)(|u|+c)), h_e = 3 vol / max face area, from the element means."""
    ub = math.sqrt(6.0) * U[..., 0]
    u = torch.linalg.norm(ub[:, 1:4], dim=1) / ub[:, 0]
    c = torch.sqrt(GAMMA * (GAMMA - 1) * (ub[:, 4] - 0.5 * ub[:, 0] * u * u) / ub[:, 0])
    a, b, d = (xyz[:, 1:] - xyz[:, :1]).unbind(1)
    vol = (torch.linalg.cross(a, b) * d).sum(1).abs() / 6
    area = torch.stack([torch.linalg.norm(torch.linalg.cross(xyz[:, v[1]] - xyz[:, v[0]], xyz[:, v[2]] - xyz[:, v[0]]), dim=1) / 2
                        for v in FV]).amax(0)
    return CFL * float((3 * vol / area / ((2 * p + 1) * (u + c))).min())


def _freestream():
    return tuple(float(t) for t in I.freestream_state(0.3))


def prepare(case, seed):
    m = _mesh_arrays(case)
    U, lam, dt = _inputs(case, seed)
    M = dg.Mesh(m.tet_vid, m.tet_xyz, m.bc_tag if case["box"] else None, order=case["p"], precision=PREC[case["prec"]],
                flux=FLUX[case["flux"]], renumber=ORDER[case["order"]], freestream=_freestream() if case["box"] else (0,) * 5)
    if case["conservative"]:
        dg.dg_set_conservative(M.handle, True)
    return dict(case=case, M=M, U=U, lam=lam, dt=dt, out=torch.empty_like(U))


def run(state):
    c, M, U, out, dt = state["case"], state["M"], state["U"], state["out"], state["dt"]
    h, kind = M.handle, c["kind"]
    if kind == "adjoint":
        J, g, _ = adjoint.rk3_adjoint(M, U, dt, c["n"], ckpt_every=2)
        return {"J": J, "grad": g if c["prec"] == "fp64" else g.float()}
    if kind == "vjp":
        dg.dg_residual_vjp(h, U, state["lam"], out)
        return out if c["prec"] == "fp64" else out.float()
    if kind == "residual":
        dg.dg_residual(h, U, out)
        return out if c["prec"] == "fp64" else out.float()
    dg.dg_set_state(h, U)
    more = {}
    if kind == "march":
        dt = dg.dg_stable_dt(h, CFL)
        dg.dg_rk3_step(h, dt, 1)
        more["dt"] = dt
        more["totals"], more["ke"] = dg.dg_integrals(h)
        if c["box"]:
            more["bflux"] = dg.dg_boundary_flux(h)
        dg.dg_sync_status(h)
    elif kind == "ns_step":
        dg.dg_ns_rk3_step(h, dt, c["n"], MU, PRANDTL)
    else:
        dg.dg_rk3_step(h, dt, c["n"])
    dg.dg_get_state(h, out)
    more["state"] = out.float() if c["prec"] == "fp32" else out
    return more


def work(case):
    """Bytes: a caller's FP64 arrays in and out once each, and per residual the stored state in and out
    (4 bytes a value in FP32, else 8) with 32 bytes of connectivity and geometry.  Flops of a residual:
    each face's traces and flux once, the volume and lift contractions; a viscous residual adds the
    gradient's and the viscous flux's; a reverse residual counts twice a forward one."""
    p = case["p"]
    nb, nq, nqf, ne = NB[p], NQ[p], NQF[p], 6 * case["nx"] * case["ny"] * case["nz"]
    nv, s = 5 * nb, 4 if case["prec"] == "fp32" else 8
    f = 2 * 2 * nqf * nv * 2 + 2 * nqf * (160 if case["flux"] == "roe" else 70) + nq * nv * 2 + nq * 115 + nv * 3 * nq * 2 \
        + nv * 4 * nqf * 2 + 4 * nv
    if case["kind"] == "ns_step":
        f += nv * 3 * nq * 2 + 3 * nv * 4 * nqf * 2 + (nq + 4 * nqf) * (3 * nv * 2 + 120) + 4 * nb * (3 * nq + 4 * nqf) * 2
    io, b = 2 * nv * 8, 2 * nv * s + 32
    fwd, rev = {"step": (3 * case["n"], 0), "march": (3, 0), "ns_step": (3 * case["n"], 0), "residual": (1, 0), "vjp": (0, 1),
                "adjoint": (3 * case["n"], 3 * case["n"])}[case["kind"]]
    return {"bytes": ne * (io + fwd * b + rev * (b + nv * s)), "flops": ne * (fwd + 2 * rev) * f}


# ---- the method in plain 64-bit torch -------------------------------------------------------------
FV = ((1, 2, 3), (0, 2, 3), (0, 1, 3), (0, 1, 2))          # local face f is opposite local vertex f
REF = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]], dtype=np.float64)
# orbits (barycentric values, pattern, weight) of the symmetric Gauss rules exact to degree 2p
TET = {
    1: [((0.1381966011250105, 0.5854101966249685), (0, 0, 0, 1), 1 / 24)],
    2: [((0.09273525031089122, 0.7217942490673264), (0, 0, 0, 1), 0.012248840519393659),
        ((0.3108859192633006, 0.06734224221009821), (0, 0, 0, 1), 0.018781320953002643),
        ((0.04550370412564965, 0.45449629587435036), (0, 0, 1, 1), 0.007091003462846911)],
    3: [((0.214602871259152, 0.356191386222544), (0, 0, 0, 1), 0.006653791709694585),
        ((0.04067395853461136, 0.877978124396166), (0, 0, 0, 1), 0.0016795351758867741),
        ((0.32233789014227554, 0.03298632957317338), (0, 0, 0, 1), 0.009226196923942453),
        ((0.06366100187501753, 0.2696723314583158, 0.6030056647916491), (0, 0, 1, 2), 0.008035714285714285)],
}
TRI = {
    1: [((1 / 6, 2 / 3), (0, 0, 1), 1 / 6)],
    2: [((0.4459484909159649, 0.10810301816807022), (0, 0, 1), 0.11169079483900574),
        ((0.09157621350977074, 0.8168475729804585), (0, 0, 1), 0.054975871827660935)],
    3: [((0.2492867451709104, 0.5014265096581791), (0, 0, 1), 0.0583931378631897),
        ((0.06308901449150223, 0.8738219710169955), (0, 0, 1), 0.02542245318510341),
        ((0.05314504984481694, 0.3103524510337844, 0.6365024991213987), (0, 1, 2), 0.04142553780918678)],
}


def _rule(orbits):
    pts, w = [], []
    for vals, pat, wt in orbits:
        for q in sorted(set(itertools.permutations(pat))):
            pts.append([vals[i] for i in q])
            w.append(wt)
    return np.array(pts), np.array(w)


def _jacobi(n, a, x):
    """Jacobi P_n^(a,0) of unit norm under (1-x)^a on [-1, 1], and its derivative (n <= 3)."""
    P, D = [np.ones_like(x), ((a + 2) * x + a) / 2], [np.zeros_like(x), np.full_like(x, (a + 2) / 2)]
    for k in range(2, n + 1):
        s = 2 * k + a
        c1, c2, c3, c4 = 2 * k * (k + a) * (s - 2), (s - 1) * a * a, (s - 2) * (s - 1) * s, 2 * (k + a - 1) * (k - 1) * s
        P.append(((c2 + c3 * x) * P[-1] - c4 * P[-2]) / c1)
        D.append(((c2 + c3 * x) * D[-1] + c3 * P[-2] - c4 * D[-2]) / c1)
    f = math.sqrt((2 * n + a + 1) / 2 ** (a + 1))
    return f * P[n], f * D[n]


def _basis(p, X):
    """Orthonormal Proriol-Koornwinder-Dubiner basis phi [n, nb] and gradient [n, nb, 3] at X [n, 3]."""
    x, y, z = X.T
    A, B = 1 - y - z, 1 - z
    a, b, c = 2 * x / A - 1, 2 * y / B - 1, 2 * z - 1
    phi, grad = [], []
    for d in range(p + 1):
        for i in range(d + 1):
            for j in range(d - i + 1):
                (P, dP), (Q, dQ), (R, dR) = _jacobi(i, 0, a), _jacobi(j, 2 * i + 1, b), _jacobi(d - i - j, 2 * i + 2 * j + 2, c)
                f, h = P * A ** i, Q * B ** j
                fx = 2 * dP * A ** (i - 1) if i else 0 * A
                fy = (dP * (1 + a) - i * P) * A ** (i - 1) if i else 0 * A     # d f / d y = d f / d z
                hy = 2 * dQ * B ** (j - 1) if j else 0 * B
                hz = (dQ * (1 + b) - j * Q) * B ** (j - 1) if j else 0 * B
                s = 8 * 2 ** (2 * i + j)
                phi.append(s * f * h * R)
                grad.append(np.stack([s * fx * h * R, s * (fy * h + f * hy) * R, s * (fy * h * R + f * hz * R + 2 * f * h * dR)], -1))
    return np.stack(phi, 1), np.stack(grad, 1)


def _volume(p):
    lam, w = _rule(TET[p])
    X = np.ascontiguousarray(lam[:, 1:])
    phi, grad = _basis(p, X)
    return X, w, phi, grad


def _abs(x):
    """|x| with the derivative +1 at 0: the rule of the adjoint at a kink."""
    return torch.where(x < 0, -x, x)


class _Plain:
    """Residual, its transpose, and the Navier-Stokes residual of a case, element by element in chunks."""
    CHUNK = 1 << 16

    def __init__(self, case):
        m, p, dev = _mesh_arrays(case), case["p"], _device()
        self.p, self.roe, self.ne = p, case["flux"] == "roe", m.ne
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a)).to(dev)   # noqa: E731
        _, w, phi, grad = _volume(p)
        bary, wf = _rule(TRI[p])
        self.w, self.phi, self.grad, self.wf = t(w), t(phi), t(grad), t(wf)
        self.phif = [t(_basis(p, bary @ REF[list(v)])[0]) for v in FV]
        self.xyz = t(m.tet_xyz)
        J = (self.xyz[:, 1:] - self.xyz[:, :1]).transpose(1, 2)
        self.det, self.Jinv = torch.linalg.det(J), torch.linalg.inv(J)
        glam = torch.cat([-self.Jinv.sum(1, keepdim=True), self.Jinv], 1)   # gradients of the barycentrics
        size = torch.linalg.norm(glam, dim=2)
        self.normal, self.sf = -glam / size[..., None], size                # outward; 2 |S_f| / |det J|
        self.tag = t(m.bc_tag.astype(np.int64))
        self.finf = t(np.array(_freestream()))
        # neighbours by sorted vertex triples, then the point permutation by vertex ids
        vid = t(m.tet_vid.astype(np.int64))
        tri = torch.stack([vid[:, list(v)] for v in FV], 1).reshape(-1, 3)
        k = tri.sort(1).values
        key = (k[:, 0] << 42) | (k[:, 1] << 21) | k[:, 2]
        srt, idx = key.sort()
        same = srt[1:] == srt[:-1]
        a, b = idx[:-1][same], idx[1:][same]
        part = torch.full_like(key, -1)
        part[a], part[b] = b, a
        self.inner = (part >= 0).reshape(-1, 4)
        other = part.clamp(min=0)
        where = (tri[other][:, :, None] == tri[:, None, :]).double().argmax(2)   # own position of the other's vertex
        perms = list(itertools.permutations(range(3)))
        pt = np.zeros((27, len(wf)), dtype=np.int64)
        for q3 in perms:
            for q in range(len(wf)):
                pt[q3[0] * 9 + q3[1] * 3 + q3[2], q] = int(np.argmin(np.abs(bary - bary[q][list(q3)]).sum(1)))
        row = t(pt)[where[:, 0] * 9 + where[:, 1] * 3 + where[:, 2]]
        self.point = (other[:, None] * len(wf) + row).reshape(m.ne, 4, len(wf))   # into the trace table

    def chunks(self):
        for s in range(0, self.ne, self.CHUNK):
            yield slice(s, min(self.ne, s + self.CHUNK))

    def traces(self, U):
        T = torch.stack([torch.einsum("qj,e...j->eq...", ph, U) for ph in self.phif], 1)
        return T

    @staticmethod
    def pressure(U):
        return (GAMMA - 1) * (U[..., 4] - 0.5 * (U[..., 1:4] ** 2).sum(-1) / U[..., 0])

    def flux(self, U):
        u, p = U[..., 1:4] / U[..., :1], self.pressure(U)
        F = u[..., :, None] * U[..., None, :]                      # [.., d, v]
        eye = torch.eye(3, dtype=U.dtype, device=U.device)
        return torch.cat([F[..., :1], F[..., 1:4] + p[..., None, None] * eye, F[..., 4:] + (p[..., None] * u)[..., None]], -1)

    def riemann(self, L, R, n):
        rl, rr, pl, pr = L[..., 0], R[..., 0], self.pressure(L), self.pressure(R)
        ul, ur = L[..., 1:4] / rl[..., None], R[..., 1:4] / rr[..., None]
        nl, nr = (ul * n).sum(-1), (ur * n).sum(-1)
        z = torch.zeros_like(rl)[..., None]
        Fl = L * nl[..., None] + torch.cat([z, pl[..., None] * n, (pl * nl)[..., None]], -1)
        Fr = R * nr[..., None] + torch.cat([z, pr[..., None] * n, (pr * nr)[..., None]], -1)
        if not self.roe:
            sl, sr = _abs(nl) + torch.sqrt(GAMMA * pl / rl), _abs(nr) + torch.sqrt(GAMMA * pr / rr)
            return 0.5 * (Fl + Fr) - 0.5 * torch.where(sl >= sr, sl, sr)[..., None] * (R - L)
        ql, qr = torch.sqrt(rl), torch.sqrt(rr)
        av = lambda a, b, x, y: (x * a + y * b) / (x + y)   # noqa: E731
        u = av(ul, ur, ql[..., None], qr[..., None])
        H = av((L[..., 4] + pl) / rl, (R[..., 4] + pr) / rr, ql, qr)
        k = 0.5 * (u * u).sum(-1)
        c2 = (GAMMA - 1) * (H - k)
        c, rho, un = torch.sqrt(c2), ql * qr, (u * n).sum(-1)
        du, dp = ur - ul, pr - pl
        dn = nr - nl
        a1, a5 = 0.5 * (dp - rho * c * dn) / c2, 0.5 * (dp + rho * c * dn) / c2
        a2 = rr - rl - dp / c2
        l2 = _abs(un)
        w1, w2, w5 = _abs(un - c) * a1, l2 * a2, _abs(un + c) * a5
        sh = (l2 * rho)[..., None] * (du - dn[..., None] * n)
        D = torch.cat([(w1 + w2 + w5)[..., None],
                       (w1 + w2 + w5)[..., None] * u + ((w5 - w1) * c)[..., None] * n + sh,
                       (w1 * (H - c * un) + w2 * k + (u * sh).sum(-1) + w5 * (H + c * un))[..., None]], -1)
        return 0.5 * (Fl + Fr) - 0.5 * D

    def ghost(self, U, n, wall):
        """Boundary state: mirrored momentum on walls, Riemann invariants on far-field faces."""
        m = U[..., 1:4]
        W = torch.cat([U[..., :1], m - 2 * (m * n).sum(-1, keepdim=True) * n, U[..., 4:]], -1)
        O = self.finf.expand_as(U)
        g1 = GAMMA - 1
        vi, vo, pi, po = m / U[..., :1], O[..., 1:4] / O[..., :1], self.pressure(U), self.pressure(O)
        ci, co = torch.sqrt(GAMMA * pi / U[..., 0]), torch.sqrt(GAMMA * po / O[..., 0])
        ni, no = (vi * n).sum(-1), (vo * n).sum(-1)
        Rp, Rm = ni + 2 * ci / g1, no - 2 * co / g1
        vn, cb = 0.5 * (Rp + Rm), 0.25 * g1 * (Rp - Rm)
        out = vn > 0
        s = torch.where(out, pi / U[..., 0] ** GAMMA, po / O[..., 0] ** GAMMA)
        v = torch.where(out[..., None], vi - ni[..., None] * n, vo - no[..., None] * n) + vn[..., None] * n
        rb = (cb * cb / (GAMMA * s)) ** (1 / g1)
        F = _cons(rb, v[..., 0], v[..., 1], v[..., 2], rb * cb * cb / GAMMA)
        F = torch.where((ni.abs() >= ci)[..., None], torch.where((ni < 0)[..., None], O, U), F)
        return torch.where(wall[..., None], W, F)

    def others(self, T, c):
        """The neighbour's traces at the own face points of the chunk c."""
        return T.reshape((-1,) + T.shape[3:])[self.point[c]]

    def face_flux(self, T, c):
        Um, Up, n = T[c], self.others(T, c), self.normal[c][:, :, None].expand(-1, -1, T.shape[2], -1)
        if not bool(self.inner.all()):
            G = self.ghost(Um, n, (self.tag[c] == 1)[:, :, None].expand(-1, -1, T.shape[2]))
            Up = torch.where(self.inner[c][:, :, None, None], Up, G)
        return self.riemann(Um, Up, n)

    def residual(self, U):
        T, out = self.traces(U), []
        for c in self.chunks():
            F = self.flux(torch.einsum("qj,evj->eqv", self.phi, U[c]))
            G = torch.einsum("ekd,eqdv->ekqv", self.Jinv[c], F)
            R = torch.einsum("q,ekqv,qjk->evj", self.w, G, self.grad)
            H = self.face_flux(T, c) * self.sf[c][:, :, None, None]
            for f in range(4):
                R = R - torch.einsum("q,eqv,qj->evj", self.wf, H[:, f], self.phif[f])
            out.append(R)
        return torch.cat(out)

    def vjp(self, U, lam):
        with torch.enable_grad():
            V = U.detach().requires_grad_(True)
            return torch.autograd.grad(self.residual(V), V, lam)[0]

    def viscous_flux(self, U, Z):
        """F_v [.., d, (momentum, energy)] from U and its gradient Z [.., d, v]; constant viscosity."""
        r, u = U[..., 0], U[..., 1:4] / U[..., :1]
        du = (Z[..., 1:4] - u[..., None, :] * Z[..., :1]) / r[..., None, None]      # [.., d, i]
        T = self.pressure(U) / r
        dp = (GAMMA - 1) * (Z[..., 4] - (u[..., None, :] * Z[..., 1:4]).sum(-1) + 0.5 * (u * u).sum(-1)[..., None] * Z[..., 0])
        dT = (dp - T[..., None] * Z[..., 0]) / r[..., None]
        div = du.diagonal(dim1=-2, dim2=-1).sum(-1)
        eye = torch.eye(3, dtype=U.dtype, device=U.device)
        tau = MU * (du + du.transpose(-1, -2) - 2 / 3 * div[..., None, None] * eye)
        kappa = MU * GAMMA / ((GAMMA - 1) * PRANDTL)
        return torch.cat([tau, ((tau * u[..., None, :]).sum(-1) + kappa * dT)[..., None]], -1)

    @staticmethod
    def wall_state(U):
        Q = torch.zeros_like(U)
        Q[..., 0] = U[..., 0]
        Q[..., 4] = U[..., 4] - 0.5 * (U[..., 1:4] ** 2).sum(-1) / U[..., 0]
        return Q

    def ns_residual(self, U):
        R, T, Z = self.residual(U), self.traces(U), []
        inner = self.inner[:, :, None, None]
        wall = ((self.tag == 1) & ~self.inner)[:, :, None, None]
        for c in self.chunks():
            Q = torch.where(inner[c], 0.5 * (T[c] + self.others(T, c)), torch.where(wall[c], self.wall_state(T[c]), T[c]))
            Uq = torch.einsum("qj,evj->eqv", self.phi, U[c])
            z = -torch.einsum("ekd,q,eqv,qjk->edvj", self.Jinv[c], self.w, Uq, self.grad)
            for f in range(4):
                z = z + torch.einsum("ed,q,eqv,qj->edvj", self.normal[c, f] * self.sf[c, f, None], self.wf, Q[:, f], self.phif[f])
            Z.append(z)
        Z = torch.cat(Z)
        TZ = self.traces(Z)
        Q = torch.where(wall, self.wall_state(T), T)
        Fn = torch.empty(T.shape[:3] + (4,), dtype=T.dtype, device=T.device)
        for c in self.chunks():
            Fn[c] = (self.viscous_flux(Q[c], TZ[c]) * self.normal[c][:, :, None, :, None]).sum(-2)
        for c in self.chunks():
            own = Fn[c].clone()
            own[..., 3] = torch.where(wall[c][..., 0], torch.zeros_like(own[..., 3]), own[..., 3])
            H = torch.where(inner[c], 0.5 * (Fn[c] - self.others(Fn, c)), own) * self.sf[c][:, :, None, None]
            Fq = self.viscous_flux(torch.einsum("qj,evj->eqv", self.phi, U[c]), torch.einsum("qj,edvj->eqdv", self.phi, Z[c]))
            R[c, 1:] -= torch.einsum("q,ekd,eqdv,qjk->evj", self.w, self.Jinv[c], Fq, self.grad)
            for f in range(4):
                R[c, 1:] += torch.einsum("q,eqv,qj->evj", self.wf, H[:, f], self.phif[f])
        return R

    def step(self, U, dt, rhs=None):
        rhs = rhs or self.residual
        U1 = U + dt * rhs(U)
        U2 = 0.75 * U + 0.25 * (U1 + dt * rhs(U1))
        return U / 3 + 2 / 3 * (U2 + dt * rhs(U2))

    def step_vjp(self, U, dt, lam):
        U1 = U + dt * self.residual(U)
        U2 = 0.75 * U + 0.25 * (U1 + dt * self.residual(U1))
        m2 = 2 / 3 * (lam + dt * self.vjp(U2, lam))
        m1 = 0.25 * (m2 + dt * self.vjp(U1, m2))
        return lam / 3 + 0.75 * m2 + m1 + dt * self.vjp(U, m1)

    def kinetic_energy(self, U):
        e = torch.zeros((), dtype=U.dtype, device=U.device)
        for c in self.chunks():
            q = torch.einsum("qj,evj->eqv", self.phi, U[c])
            e = e + torch.einsum("q,e,eq->", self.w, self.det[c], 0.5 * (q[..., 1:4] ** 2).sum(-1) / q[..., 0])
        return e

    def boundary_flux(self, U):
        T, B = self.traces(U), torch.zeros(5, dtype=U.dtype, device=U.device)
        for c in self.chunks():
            H = self.face_flux(T, c) * (self.sf[c] * self.det[c, None] * ~self.inner[c])[:, :, None, None]
            B += torch.einsum("q,efqv->v", self.wf, H)
        return B


@torch.no_grad()
def exact(case, seed):
    P, (U, lam, dt), kind = _Plain(case), _inputs(case, seed), case["kind"]
    if kind == "residual":
        return P.residual(U)
    if kind == "vjp":
        return P.vjp(U, lam)
    if kind == "adjoint":
        states = [U]
        for _ in range(case["n"]):
            states.append(P.step(states[-1], dt))
        with torch.enable_grad():
            V = states[-1].clone().requires_grad_(True)
            J = P.kinetic_energy(V)
            g = torch.autograd.grad(J, V)[0]
        for S in reversed(states[:-1]):
            g = P.step_vjp(S, dt, g)
        return {"J": float(J.detach()), "grad": g}
    out = {}
    for _ in range(case["n"]):
        U = P.step(U, dt, P.ns_residual if kind == "ns_step" else None)
    if kind == "march":
        out = {"dt": dt, "totals": (P.det[:, None] * U[..., 0]).sum(0) / math.sqrt(6.0), "ke": float(P.kinetic_energy(U))}
        if case["box"]:
            out["bflux"] = P.boundary_flux(U)
    out["state"] = U
    return out
