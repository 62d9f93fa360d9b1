"""Performance cases of the framework's public entry points: what a program that tunes loop
arrays has the library do, from one loop with one configuration up to 1024 ports.

A case is a plain dict. `kind` says which entry points it goes through:

  train   Simulator(C) -> (B, loss), then loss.sum().backward()            (autograd)
  field   the same call, differentiated through a cotangent on the whole field B
          (and on the loss too where cot is "both")
  fit     AdamFit: a fit of the capacitances from its start, `epochs` epochs
  ragged  one call over many structures of uneven port counts, then loss.sum().backward()
  sroute  rc_reflection -> SRoute -> (Bcomb, loss), then loss.sum().backward()
  basis   mts_build_basis for a new geometry, and the export of H and M

Programs that use the FP32-class precisions ("mixed", "bf16") keep their parameters, losses
and gradients in float32, as torch programs do; those that use "fp64" keep float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2503_18479_gb300 import native as nv
from paper_2503_18479_gb300 import workloads as W
from paper_2503_18479_gb300.optimize import AdamFit
from paper_2503_18479_gb300.simulator import Simulator
from paper_2503_18479_gb300.sroute import SRoute, rc_reflection

MU0 = 4e-7 * math.pi
WIRE = 0.001
SIDE, PITCH = 0.050, 0.055
LR = 1e-13


def listed():
    return [
        # the single tuned loop of a bench set-up: one capacitance, a frequency sweep, FP64
        dict(name="loop_1x101_fp64", kind="train", shape="loop", nx=1, ny=1, seg=64, n_cfg=1,
             n_freq=101, grid=32, planes=1, precision="fp64", loss="abs"),
        # a line of 8 loops over a band: many small systems, a large field
        dict(name="line8_1024x201", kind="train", shape="square", nx=8, ny=1, seg=16, n_cfg=1024,
             n_freq=201, grid=64, planes=1, precision="mixed", loss="abs"),
        # the 8x8 metasurface, the batch that the benchmark reports: field, objective, gradient
        dict(name="array64_4096", kind="train", shape="square", nx=8, ny=8, seg=16, n_cfg=4096,
             n_freq=1, grid=128, planes=4, precision="mixed", loss="abs"),
        # fitting that metasurface: 4096 fits of 64 capacitances, a first stretch of 20 epochs
        dict(name="array64_fit", kind="fit", shape="square", nx=8, ny=8, seg=16, n_cfg=4096,
             n_freq=1, grid=16, planes=1, precision="mixed", loss="abs", epochs=20),
        # the same array inside a larger model: a gradient comes back for the whole field
        dict(name="array64_field", kind="field", shape="square", nx=8, ny=8, seg=16, n_cfg=3000,
             n_freq=1, grid=128, planes=4, precision="mixed", loss="abs", cot="field"),
        # an odd array and odd grid over three frequencies in the fast, coarse precision
        dict(name="array63_bf16", kind="train", shape="square", nx=9, ny=7, seg=16, n_cfg=1000,
             n_freq=3, grid=101, planes=1, precision="bf16", loss="abs"),
        # the metasurface in full double precision (reference runs, ill-conditioned tunings)
        dict(name="array64_fp64", kind="train", shape="square", nx=8, ny=8, seg=16, n_cfg=1024,
             n_freq=1, grid=64, planes=4, precision="fp64", loss="abs"),
        # a catalogue of different arrays in one call: 1 to 128 ports, 1 to 16 frequencies each
        dict(name="ragged_300", kind="ragged", mix=0, n_struct=300, grid=64, max_freq=16,
             max_ports=128, precision="mixed"),
        # an array past the register kernels, complex targets, gradients through field and loss
        dict(name="array80_both", kind="field", shape="square", nx=10, ny=8, seg=16, n_cfg=500,
             n_freq=2, grid=75, planes=1, precision="mixed", loss="complex", cot="both"),
        # the largest array: 1024 ports
        dict(name="array1024_256", kind="train", shape="square", nx=32, ny=32, seg=16, n_cfg=256,
             n_freq=1, grid=256, planes=2, precision="mixed", loss="abs"),
        # the scattering-parameter route on exported fields: 65 structure ports, RC loads
        dict(name="sroute65_4096", kind="sroute", nx=8, ny=8, n_cfg=4096, n_freq=1, grid=128,
             planes=4, precision="mixed"),
        # a new geometry: field basis and inductances of the 8x8 array
        dict(name="basis64", kind="basis", shape="square", nx=8, ny=8, seg=16, grid=128, planes=4,
             precision="mixed"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["train", "train", "train", "field", "fit", "ragged", "sroute", "basis", "large"])
    if kind == "ragged":
        return dict(kind=kind, mix=rng.randint(1, 999), n_struct=_log(rng, 20, 300), grid=rng.randint(9, 64),
                    max_freq=rng.randint(1, 16), max_ports=rng.choice([16, 64, 128]),
                    precision=rng.choice(["mixed", "mixed", "bf16"]))
    if kind == "sroute":
        nx, ny = rng.randint(1, 10), rng.randint(1, 9)
        c = dict(kind=kind, nx=nx, ny=ny, n_cfg=_log(rng, 16, 4096), n_freq=rng.randint(1, 3),
                 grid=_log(rng, 8, 90), planes=rng.randint(1, 2), precision="mixed")
        return _fit_in(c, 2.7e8)
    if kind == "basis":
        shape = rng.choice(["square", "square", "circle"])
        nx, ny = (rng.randint(1, 5), rng.randint(1, 5)) if shape == "circle" else (rng.randint(1, 12), rng.randint(1, 12))
        return dict(kind=kind, shape=shape, nx=nx, ny=ny,
                    seg=rng.randint(24, 64) if shape == "circle" else rng.randint(1, 16),
                    grid=_log(rng, 10, 128), planes=rng.randint(1, 4),
                    precision=rng.choice(["mixed", "mixed", "bf16"]))
    if kind == "large":
        nx, ny = rng.choice([(10, 8), (11, 11), (16, 8), (13, 11), (16, 12), (19, 17), (24, 20)])
        c = dict(kind="train", shape="square", nx=nx, ny=ny, seg=rng.choice([1, 2, 4, 8]),
                 n_cfg=_log(rng, 16, 256 if nx * ny > 150 else 2000), n_freq=1,
                 grid=_log(rng, 16, 128), planes=rng.randint(1, 2),
                 precision=rng.choice(["mixed", "mixed", "bf16"]), loss=rng.choice(["abs", "complex"]))
        return _fit_in(c, 1.3e8)
    nx, ny = rng.randint(1, 8), rng.randint(1, 8)
    c = dict(kind=kind, shape="square", nx=nx, ny=ny, seg=rng.choice([1, 4, 16]),
             n_cfg=_log(rng, 1, 4096), n_freq=_log(rng, 1, 64), grid=_log(rng, 8, 128),
             planes=rng.randint(1, 4), precision="mixed", loss=rng.choice(["abs", "complex"]))
    if kind == "fit":
        c.update(n_freq=rng.randint(1, 3), grid=16, planes=1, epochs=rng.randint(3, 20), loss="abs")
        return c
    if kind == "field":
        c.update(cot=rng.choice(["field", "both"]))
        return _fit_in(c, 2.7e8)
    c.update(precision=rng.choice(["mixed", "mixed", "mixed", "bf16", "fp64"]))
    return _fit_in(c, 1.7e7 if c["precision"] == "fp64" else 4e8)


def _fit_in(c, most):
    """The case with fewer configurations where its field would hold over `most` values, or its
    solves would cost more than those of the largest listed case."""
    P = c["planes"] * c["grid"] ** 2 + c["nx"] * c["ny"]
    most = min(most / P, 2e10 / (c["nx"] * c["ny"]) ** 3)
    c["n_cfg"] = max(1, min(c["n_cfg"], int(most / c["n_freq"])))
    return c


# ---------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------
def _geometry(case, rng):
    """(loops, corner loops, L_self, omega, points) of an array; the corner loops are the same
    polygons without the vertices that lie inside a straight side."""
    nx, ny, seg = case["nx"], case["ny"], case["seg"]
    side, pitch = SIDE, PITCH
    if case["kind"] == "basis":  # another seed is another geometry
        side, pitch = rng.uniform(0.046, 0.052), rng.uniform(0.054, 0.060)
    ctr = [((i - (nx - 1) / 2.0) * pitch, (j - (ny - 1) / 2.0) * pitch) for j in range(ny) for i in range(nx)]
    L_self = None
    if case["shape"] == "square":
        loops = W.square_array(nx, ny, side, pitch, seg)
        corners = [tuple(v[::seg] for v in l) for l in loops]
    else:
        a = 0.050 if case["shape"] == "loop" else side / 2
        loops = corners = [W.circular_loop(a, seg, x, y) for x, y in ctr]
        L_self = np.full(nx * ny, MU0 * a * (math.log(8 * a / WIRE) - 2))
    hx, hy = (nx + 1) * pitch / 2, (ny + 1) * pitch / 2
    z0 = 0.020 if case["planes"] == 1 else 0.010
    pts = [W.grid_plane(case["grid"], hx, z0 + 0.010 * k, half_span_y=hy) for k in range(case["planes"])]
    pts.append((np.array([x for x, _ in ctr]), np.array([y for _, y in ctr]), np.full(nx * ny, 0.040)))
    pts = tuple(np.concatenate([p[i] for p in pts]) for i in range(3))
    F = case.get("n_freq", 1)
    omega = 2 * math.pi * (np.array([63.6e6]) if F == 1 else np.linspace(60e6, 68e6, F))
    return loops, corners, L_self, omega, pts


def _workload(case, seed):
    """(Workload, corner loops of each structure); capacitances are uniform in 20..200 pF."""
    rng = np.random.default_rng(seed)
    if case["kind"] == "ragged":
        ports = [n for n in W.RAGGED_SHAPES if n <= case["max_ports"]]
        wl = W.ragged(seed=case["mix"], n_struct=case["n_struct"], grid=case["grid"],
                      max_freq=case["max_freq"], port_choices=ports)  # the catalogue
        corners = []
        for st in wl.structures:
            off = st.loop_vtx_off
            corners.append([tuple(v[off[k]:off[k + 1]][::16] for v in (st.vx, st.vy, st.vz))
                            for k in range(st.n_ports)])
        wl.C = rng.uniform(20e-12, 200e-12, size=wl.C.shape).astype(np.float32).astype(np.float64)
        wl.target = rng.standard_normal(wl.target.shape) * 1e-6
        return wl, corners
    loops, corners, L_self, omega, pts = _geometry(case, rng)
    off, vx, vy, vz = W.loops_to_arrays(loops)
    N, F, P = len(loops), len(omega), len(pts[0])
    st = W.Structure(loop_vtx_off=off, vx=vx, vy=vy, vz=vz, px=pts[0], py=pts[1], pz=pts[2],
                     R=np.full(N, 0.1), omega=omega, V=W.drive_uniform_field(loops, omega),
                     loss_idx=np.arange(P - N, P, dtype=np.int64), L_self=L_self)
    cplx = case.get("loss") == "complex"
    C = rng.uniform(20e-12, 200e-12, size=(case.get("n_cfg", 1), N))
    if case["precision"] != "fp64":
        C = C.astype(np.float32).astype(np.float64)
    target = rng.standard_normal(F * N * (2 if cplx else 1)) * 1e-6
    return W.Workload("case", [st], C, WIRE, loss_mode=int(cplx), target=target), [corners]


def _cotangents(case, seed, n_cfg, n_field):
    g = torch.Generator(device="cuda").manual_seed(seed)
    gB = torch.randn((n_cfg, n_field, 2), dtype=torch.float32, device="cuda", generator=g)
    gl = torch.rand((n_cfg, 1), dtype=torch.float32, device="cuda", generator=g) * 1e13
    return torch.view_as_complex(gB), gl


def prepare(case, seed):
    if case["kind"] == "sroute":
        sw = _sroute_inputs(case, seed)
        dev = {k: torch.from_numpy(getattr(sw, k)).cuda() for k in ("R", "omega")}
        sr = SRoute(sw.S0, sw.field, sw.rows, sw.cols, sw.n1, sc_const=sw.sc_const,
                    loss_idx=sw.loss_idx, target=sw.target, precision=case["precision"])
        C = torch.from_numpy(sw.C.astype(np.float32)).cuda().requires_grad_(True)
        return dict(case=case, sr=sr, C=C, Z0=sw.Z0, **dev)
    wl, _ = _workload(case, seed)
    if case["kind"] == "basis":
        pb = nv.Problem(wl.flat(), wl.wire_radius)
        st = wl.structures[0]
        return dict(case=case, pb=pb, basis=nv.alloc_bytes(nv.mts_basis_bytes(pb, case["precision"])),
                    H=torch.empty((st.n_points, st.n_ports), dtype=torch.float64, device="cuda"),
                    M=torch.empty((st.n_ports, st.n_ports), dtype=torch.float64, device="cuda"))
    sim = Simulator(wl, case["precision"])
    C = torch.from_numpy(wl.C).cuda()
    if case["precision"] != "fp64":
        C = C.float()
    s = dict(case=case, sim=sim, C=C)
    if case["kind"] != "fit":
        C.requires_grad_(True)
    if case["kind"] == "field":
        s["gB"], s["gl"] = _cotangents(case, seed, wl.n_cfg, sim.sumFP)
    return s


def run(s):
    kind = s["case"]["kind"]
    if kind == "basis":
        prec = s["case"]["precision"]
        nv.mts_build_basis(s["pb"], prec, s["basis"])
        nv.mts_basis_export(s["pb"], prec, s["basis"], s["H"], s["M"])
        return {"H": s["H"].float(), "M": s["M"]}
    if kind == "fit":
        epochs = s["case"]["epochs"]
        C, history = AdamFit(s["sim"], s["C"], lr=LR, max_epochs=epochs).run(epochs)
        return {"C": C.float(), "history": history.float()}
    C = s["C"]
    C.grad = None
    if kind == "sroute":
        B, loss = s["sr"](rc_reflection(s["R"], C, s["omega"], s["Z0"]))
    else:
        B, loss = s["sim"](C)
    loss = loss.to(C.dtype)
    if kind != "field":
        loss.sum().backward()
    elif s["case"]["cot"] == "both":
        torch.autograd.backward([B, loss], [s["gB"], s["gl"]])
    else:
        B.backward(s["gB"])
    return {"B": B.detach(), "loss": loss.detach(), "grad_C": C.grad}


# ---------------------------------------------------------------------------------------
# the least work of a pass
# ---------------------------------------------------------------------------------------
def _solve_flops(N, systems):
    """LU, a forward and an adjoint triangular pair, and one residual of each."""
    return systems * (8 / 3 * N ** 3 + 4 * 8 * N ** 2)


def work(case):
    kind = case["kind"]
    elem = 16 if case["precision"] == "fp64" else 8
    if kind == "ragged":
        ports = [n for n in W.RAGGED_SHAPES if n <= case["max_ports"]]
        each = case["n_struct"] / len(ports)
        F, g2 = (case["max_freq"] + 1) / 2, case["grid"] ** 2
        by = sum(each * (g2 + n) * (F * elem + 4 * n) for n in ports)
        fl = sum(each * F * (_solve_flops(n, 1) + 4 * n * (g2 + n)) for n in ports)
        return {"bytes": by, "flops": fl}
    N = case["nx"] * case["ny"]
    P = case["planes"] * case["grid"] ** 2 + N
    if kind == "basis":
        segs = N * (case["seg"] if case["shape"] == "circle" else 4)  # straight sides
        return {"bytes": P * (24 + 4 * N) + 8 * N * N, "flops": 30 * P * segs + 60 * segs ** 2}
    S = case["n_cfg"] * case["n_freq"]
    if kind == "fit":
        e = case["epochs"]
        return {"bytes": e * case["n_cfg"] * (16 * N + 8), "flops": e * (_solve_flops(N, S) + 8 * S * N * N)}
    if kind == "sroute":
        n0 = N + 1
        return {"bytes": elem * P * (S + case["n_freq"] * n0), "flops": _solve_flops(n0, S) + 8 * S * P * n0}
    by = elem * P * S + elem // 2 * P * N + 16 * case["n_cfg"] * N
    fl = _solve_flops(N, S) + 4 * S * P * N
    if kind == "field":
        by, fl = by + elem * P * S, fl + 4 * S * P * N + 16 * S * N * N
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------------------
# the same results in plain 64-bit torch
# ---------------------------------------------------------------------------------------
def _dev(a):
    return torch.as_tensor(np.asarray(a), device="cuda")


def _sides(loops):
    """Start and end of every straight side, and the loop that it belongs to: [S, 3], [S, 3], [S]."""
    a = np.concatenate([np.stack(l, 1) for l in loops])
    b = np.concatenate([np.roll(np.stack(l, 1), -1, axis=0) for l in loops])
    return _dev(a), _dev(b), _dev(np.repeat(np.arange(len(loops)), [len(l[0]) for l in loops]))


def _field_basis(loops, pts):
    """H [P, N]: Bz of the Biot-Savart integral over straight sides carrying 1 A."""
    a, b, own = _sides(loops)
    H = torch.zeros((len(pts[0]), len(loops)), dtype=torch.float64, device="cuda")
    step = max(1, int(6e7) // len(a))
    for p0 in range(0, len(pts[0]), step):
        p = torch.stack([_dev(x[p0:p0 + step]) for x in pts], 1)
        u, v = p[:, None] - a[None], p[:, None] - b[None]
        cz = u[..., 0] * v[..., 1] - u[..., 1] * v[..., 0]
        ru, rv = u.norm(dim=-1), v.norm(dim=-1)
        dot = (u * v).sum(-1)
        cross2 = torch.linalg.cross(u, v).square().sum(-1)
        den = torch.where(dot > 0, ru * rv + dot, cross2 / (ru * rv - dot))
        H[p0:p0 + step].index_add_(1, own, MU0 / (4 * math.pi) * cz * (ru + rv) / (ru * rv * den))
    return H


def _inductance(loops, L_self):
    """M [N, N]: Neumann's double integral; parallel sides in closed form, others by Gauss
    quadrature (loops that do not touch), the self terms from L_self where it is given."""
    N = len(loops)
    a, b, own = _sides(loops)
    d = b - a
    l = d.norm(dim=-1)
    M = torch.zeros((N, N), dtype=torch.float64, device="cuda")
    if L_self is not None:
        x, w = np.polynomial.legendre.leggauss(16)
        x = _dev(np.concatenate([(k + (1 + x) / 2) / 4 for k in range(4)]))  # four panels a side
        w = _dev(np.tile(w, 4) / 8)
        q = (a[:, None] + x[None, :, None] * d[:, None]).reshape(N, -1, 3)
        dl = (w[None, :, None] * d[:, None]).reshape(N, -1, 3)
        for i in range(N):
            for j in range(i + 1, N):
                dist = (q[i][:, None] - q[j][None]).norm(dim=-1)
                M[i, j] = M[j, i] = MU0 / (4 * math.pi) * ((dl[i] @ dl[j].T) / dist).sum()
        return M + torch.diag(_dev(L_self))
    t = d / l[:, None]
    step = max(1, int(3e7) // len(a))
    for s0 in range(0, len(a), step):
        s = slice(s0, s0 + step)
        cos = t[s] @ t.T
        along = (t[s][:, None] * (a[None] - a[s][:, None])).sum(-1)  # start of the other side
        far = along + cos * l[None]
        off = (a[None] - a[s][:, None]) - along[..., None] * t[s][:, None]
        dist = off.norm(dim=-1)
        line = dist < 1e-9  # on one line

        def G(u):
            y = torch.where(line, torch.ones_like(dist), dist)
            return torch.where(line, torch.xlogy(u.abs(), u.abs()) - u.abs(),
                               u * torch.asinh(u / y) - torch.sqrt(u * u + y * y))

        ls = l[s][:, None]
        pair = MU0 / (4 * math.pi) * (G(ls - along) - G(-along) - G(ls - far) + G(-far))
        pair = torch.where(cos.abs() > 0.5, pair, torch.zeros_like(pair))
        k = torch.arange(s0, s0 + cos.shape[0], device="cuda")
        pair[k - s0, k] = MU0 / (2 * math.pi) * l[s] * (torch.log(2 * l[s] / WIRE) - 1)
        rows = torch.zeros((cos.shape[0], N), dtype=torch.float64, device="cuda").index_add_(1, own, pair)
        M.index_add_(0, own[s], rows)
    return M


def _assemble(M, R, C, omega):
    A = 1j * omega[:, None, None] * M[None] + torch.diag(R)[None]
    A = A[None].expand(C.shape[0], -1, -1, -1).clone()
    z = 1 / (1j * omega[None, :, None] * C[:, None])
    A.diagonal(dim1=-2, dim2=-1).add_(z)
    return A


def _fields(H, I):
    """H I for real H [P, N] and complex I [..., N]."""
    return torch.complex(I.real @ H.T, I.imag @ H.T)


def _objective(B, target, cplx):
    """Per configuration: the mean objective and its cotangent dL/dRe + j dL/dIm."""
    n = B.shape[1] * B.shape[2]
    if cplx:
        e = B - target
        return e.abs().square().mean(dim=(1, 2)), 2 * e / n
    r = B.abs()
    return (r - target).square().mean(dim=(1, 2)), 2 * (r - target) * torch.where(r > 0, B / r, B) / n


def _structure(st, corners, C, target, cplx, cot=None, gB=None, gl=None, want_B=True):
    """(B [b, F P], loss [b], grad_C [b, N]) of one structure in 64 bits."""
    pts = (st.px, st.py, st.pz)
    M = _inductance(corners, st.L_self)
    R, omega, V = _dev(st.R), _dev(st.omega), _dev(st.V)
    F = len(st.omega)
    target = _dev(target)
    target = torch.view_as_complex(target.reshape(F, -1, 2).contiguous()) if cplx else target.reshape(F, -1)
    H = _field_basis(corners, pts) if want_B else None
    Hl = _field_basis(corners, tuple(x[st.loss_idx] for x in pts))
    Bs, losses, grads = [], [], []
    step = max(1, int(2e8) // (F * M.shape[0] ** 2))
    for c0 in range(0, C.shape[0], step):
        c = slice(c0, c0 + step)
        A = _assemble(M, R, C[c], omega)
        LU, piv = torch.linalg.lu_factor(A)
        I = torch.linalg.lu_solve(LU, piv, V[None, :, :, None].expand(A.shape[0], -1, -1, -1).contiguous())[..., 0]
        loss, G = _objective(_fields(Hl, I), target, cplx)
        u = torch.zeros_like(I)
        if cot != "field":
            scale = 1.0 if gl is None else gl[c].double()[:, None, None]
            u = u + _fields(Hl.T, G.conj()) * scale
        if gB is not None:
            g = gB[c].reshape(A.shape[0], F, -1)
            u = u + torch.complex(g.real.double() @ H, -(g.imag.double() @ H))
        mu = torch.linalg.lu_solve(LU, piv, u[..., None])[..., 0]
        grads.append(((mu * I).imag / omega[None, :, None]).sum(1) / C[c].square())
        losses.append(loss)
        if want_B:
            Bs.append(_fields(H, I).reshape(A.shape[0], -1))
    return torch.cat(Bs) if want_B else None, torch.cat(losses), torch.cat(grads)


def _sroute_inputs(case, seed):
    freqs = (63.6e6,) if case["n_freq"] == 1 else tuple(np.linspace(60e6, 68e6, case["n_freq"]))
    sw = W.sroute_array(case["nx"], case["ny"], seed=seed, n_cfg=case["n_cfg"], grid=case["grid"],
                        planes=tuple(0.010 * (k + 1) for k in range(case["planes"])), freqs_hz=freqs)
    sw.C = sw.C.astype(np.float32).astype(np.float64)
    return sw


def _exact_sroute(case, seed):
    sw = _sroute_inputs(case, seed)
    n0 = sw.S0.shape[1]
    S0, field, omega, R = _dev(sw.S0), _dev(sw.field), _dev(sw.omega), _dev(sw.R)
    S12 = _dev(sw.sc_const)[:, :n0, n0:]
    C = _dev(sw.C).requires_grad_(True)
    Z = R[:, None] - 1j / (omega[None, :, None] * C[:, None])
    gamma = (Z - sw.Z0) / (Z + sw.Z0)
    gamma = torch.cat([gamma, torch.zeros_like(gamma[..., :1])], -1)  # the drive port is matched
    A = torch.eye(n0, device="cuda") - gamma[..., None] * S0[None]
    V = torch.linalg.solve(A, S12[None].expand(A.shape[0], -1, -1, -1))  # [b, F, n0, n1]
    Bl = torch.einsum("flk,bfkc->bcfl", field[:, _dev(sw.loss_idx)], V)
    loss = (Bl.abs() - _dev(sw.target).transpose(0, 1)[None]).square().mean(dim=(1, 2, 3))
    loss.sum().backward()
    B = torch.stack([field[f] @ V.detach()[:, f, :, 0].T for f in range(len(omega))])  # [F, P, b]
    return {"B": B.permute(2, 0, 1)[:, None], "loss": loss.detach(), "grad_C": C.grad}


def _exact_fit(case, wl, corners):
    """Adam (Kingma and Ba) on the exact objective and gradient."""
    st, C = wl.structures[0], _dev(wl.C).clone()
    m, v = torch.zeros_like(C), torch.zeros_like(C)
    history = []
    for t in range(1, case["epochs"] + 1):
        _, loss, g = _structure(st, corners[0], C, wl.target, False, want_B=False)
        history.append(loss[:, None])
        m = 0.9 * m + 0.1 * g
        v = 0.999 * v + 0.001 * g * g
        C = C - LR / (1 - 0.9 ** t) * m / (v.sqrt() / math.sqrt(1 - 0.999 ** t) + 1e-8)
    return {"C": C, "history": torch.stack(history)}


def exact(case, seed):
    kind = case["kind"]
    if kind == "sroute":
        return _exact_sroute(case, seed)
    wl, corners = _workload(case, seed)
    if kind == "basis":
        st = wl.structures[0]
        return {"H": _field_basis(corners[0], (st.px, st.py, st.pz)), "M": _inductance(corners[0], st.L_self)}
    if kind == "fit":
        return _exact_fit(case, wl, corners)
    gB = gl = None
    cot = case.get("cot")
    if kind == "field":
        st = wl.structures[0]
        gB, gl = _cotangents(case, seed, wl.n_cfg, st.n_freq * st.n_points)
        gl = gl[:, 0]
    parts, target_off, cplx = [], wl.target_off() * (1 + wl.loss_mode), wl.loss_mode == 1
    for s, st in enumerate(wl.structures):
        t = wl.target[target_off[s]:target_off[s + 1]]
        parts.append(_structure(st, corners[s], _dev(wl.structure_C(s)), t, cplx, cot, gB, gl))
    return {"B": torch.cat([p[0] for p in parts], 1), "loss": torch.stack([p[1] for p in parts], 1),
            "grad_C": torch.cat([p[2] for p in parts], 1)}
