"""Performance cases: the calls a program that uses this library makes, over the sizes it makes them at.

A case is a dict of plain values.  ``op`` says which entry points one pass goes through:

* ``solve``: whole load steps of Algorithm 1 from a fresh state (fftm_reset_state, fftm_set_load,
  fftm_solve_step, then the stress field and, where the stencil leaves no free hourglass mode in it,
  the displacement), the main use;
* ``serve``: a batch of independent requests through the serving runtime (fftm_server_submit,
  fftm_server_poll), results on the host;
* ``residual``: fftm_residual_noalloc on a caller's displacement field (equilibrium checks, outer
  solvers that own their fields);
* ``green``: fftm_apply of the Green update on a caller's polarisation field (the operator alone, as
  a preconditioner of an outer solver).

Grid sizes are the library's own, 2^a 3^b voxels per axis.  ``iters`` is the typical number of
fixed-point iterations (for ``work`` only).  ``exact`` is plain FP64 torch: dense transform
matrices, stencils as shifted sums, the fixed point run far below the case's tolerance.
"""

import math

import numpy as np
import torch

from paper_2607_05929_gb300 import fftm as F

DEV = torch.device("cuda" if torch.cuda.is_available() else "cpu")
SIZES = (16, 18, 24, 27, 32, 36, 48, 54, 64, 72, 81, 96, 108, 128, 144, 162, 192, 216, 243, 256)
CUBIC = (168.0, 121.0, 75.0)  # C11, C12, C44 (GPa)
CP = CUBIC + (1e-3, 20.0, 0.03, 0.09, 0.3, 1.0)  # gdot0, n, tau0, tau_inf, h0, dt
VOIGT = ((0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1))


def lame(E, nu):
    return E * nu / ((1 + nu) * (1 - 2 * nu)), E / (2 * (1 + nu))


def case(name, op, n, precision, scheme, bc, law, load="tension", tol=1e-6, steps=1, iters=1, out="stress", grains=0):
    return {"name": name, "op": op, "n1": n[0], "n2": n[1], "n3": n[2], "precision": precision, "scheme": scheme,
            "bc": bc, "law": law, "load": load, "tol": tol, "steps": steps, "iters": iters, "out": out,
            "grains": grains}


def listed():
    return [
        # the smallest problem of a parameter study: a stiff inclusion, double precision to 1e-8
        case("inclusion_32_fp64", "solve", (32, 32, 32), "fp64", "HEX1", "D N P", "iso10", tol=1e-8, iters=120,
             out="u,stress"),
        # the headline workload: a 500-grain cubic polycrystal, TF32 tensor-core transforms
        case("polycrystal_256_tf32", "solve", (256, 256, 256), "fp32_tf32", "TETRA2", "D N P", "cubic", iters=21,
             out="u", grains=500),
        # a flat specimen on a ragged grid, FP32 FFT transforms, stresses read out
        case("specimen_162x96x243_fp32", "solve", (162, 96, 243), "fp32", "TETRA2", "D N P", "cubic", iters=21,
             out="u,stress", grains=120),
        # the double-precision run that a single-precision one is checked against
        case("polycrystal_128_fp64", "solve", (128, 128, 128), "fp64", "TETRA2", "D N P", "cubic", iters=21,
             out="u,stress", grains=200),
        # elasto-plastic composite under bending, two load steps (the second from a committed state)
        case("composite_j2_128_tf32", "solve", (128, 128, 128), "fp32_tf32", "HEX1", "D N N", "j2bend", "bending",
             steps=2, iters=90),
        # finite-strain crystal plasticity, one torsion-bending increment
        case("crystal_32_fp32", "solve", (32, 32, 32), "fp32", "TETRA2", "D N N", "cp", "torsion", tol=1e-5,
             iters=27, out="u,stress", grains=24),
        # finite-strain porous medium (logarithmic J2), stretched past yield
        case("porous_48_fp64", "solve", (48, 48, 48), "fp64", "TETRA2", "D N P", "logj2", "stretch", iters=60),
        # a uniaxial test: one strain component imposed, the others free (normal-mixed loading)
        case("uniaxial_64_fp64", "solve", (64, 64, 64), "fp64", "HEX1", "dnn ndn nnd", "iso2", "mixed", iters=27),
        # eight mixed requests at once through the server
        case("serve_8_tf32", "serve", (64, 64, 64), "fp32_tf32", "mixed", "mixed", "request", "tension", iters=40),
        # an equilibrium check of a caller's field on a mid-size polycrystal
        case("residual_192_fp32", "residual", (192, 192, 192), "fp32", "TETRA2", "D N P", "cubic", grains=300),
        # the Green operator alone: double precision on an odd grid with quarter-wave axes, and FP32
        # at full size
        case("green_108x81x72_fp64", "green", (108, 81, 72), "fp64", "HEX1", "dnn:nnn P dnd:nnn", "iso2"),
        case("green_256_fp32", "green", (256, 256, 256), "fp32", "TETRA2", "D N P", "iso2"),
    ]


def draw(rng):
    def side(lo, hi):
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        return min(SIZES, key=lambda s: abs(math.log(s / v)))

    def grid(lo, hi):
        b = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        return tuple(side(max(lo, 0.6 * b), min(hi, 1.4 * b)) for _ in range(3))

    scheme = rng.choice(["HEX1", "TETRA2"])
    kind = rng.choices(["cubic", "iso2", "j2", "porous", "cp", "mixed", "serve", "residual", "green"],
                       [5, 2, 2, 1, 1, 1, 1, 3, 3])[0]
    low = rng.choice(["fp32", "fp32_tf32"])
    if kind in ("cubic", "iso2"):
        prec = rng.choice(["fp64", "fp32", "fp32_tf32"])
        c = case("", "solve", grid(24, 128 if prec == "fp64" else 243), prec, scheme,
                 rng.choice(["D N P", "D N N", "D P N", "D P P"] + (["N D P", "D D P"] if prec == "fp64" else [])),
                 kind, iters=21,
                 grains=rng.randint(20, 300))
    elif kind == "j2":
        c = case("", "solve", grid(24, 108), rng.choice(["fp64", low]), scheme, "D N N", "j2bend", "bending", steps=2,
                 iters=40)
    elif kind == "porous":
        c = case("", "solve", grid(16, 54), "fp64", "TETRA2", "D N P", "logj2", "stretch", iters=60)
    elif kind == "cp":
        c = case("", "solve", grid(16, 36), "fp32", "TETRA2", "D N N", "cp", "torsion", tol=1e-5, iters=60,
                 grains=rng.randint(8, 30))
    elif kind == "mixed":
        c = case("", "solve", grid(24, 96), "fp64", scheme, "dnn ndn nnd", "iso2", "mixed",
                 iters=60)
    elif kind == "serve":
        s = side(36, 81)
        c = case("", "serve", (s, s, s), low, "mixed", "mixed", "request", "tension", iters=40)
    elif kind == "residual":
        c = case("", "residual", grid(24, 243), rng.choice(["fp64", "fp32"]), scheme,
                 rng.choice(["D N P", "D N N", "P P P", "dnn ndn nnd"]), rng.choice(["cubic", "iso2"]),
                 grains=rng.randint(20, 300))
    else:
        c = case("", "green", grid(24, 243), rng.choice(["fp64", "fp32"]), scheme,
                 rng.choice(["D N P", "D N N", "P P P", "dnn:nnn P dnd:nnn", "dnn ndn nnd"]), "iso2")
    del c["name"]
    return c


# ---- inputs ----------------------------------------------------------------------------------
def bc_table(text):
    """bc[axis][face][component] of "x y z": one letter an axis, three letters (components), or
    three:three (the two faces)."""
    out = []
    for t in text.split():
        t = t.upper()
        f = t.split(":") if ":" in t else [t, t]
        out.append([list(v * 3 if len(v) == 1 else v) for v in f])
    return out


def voronoi(n, grains, gen):
    """Grain index of the nearest of `grains` random points (ties to the lowest index), [x, y, z]."""
    box = torch.tensor([16 * v for v in n])
    pts = (torch.rand((grains, 3), generator=gen, dtype=torch.float64) * box).long().to(DEV)
    ax = [16 * torch.arange(n[a], device=DEV) + 8 for a in range(3)]
    best = torch.full(n, 1 << 60, dtype=torch.int64, device=DEV)
    for g in range(grains):
        d = [(ax[a] - pts[g, a]) ** 2 for a in range(3)]
        xy = ((d[0][:, None] + d[1][None, :]) << 16) + g
        torch.minimum(best, xy[:, :, None] + (d[2] << 16), out=best)
    return (best & 0xFFFF).to(torch.int32)


def spheres(n, fraction, gen):
    """Overlapping random spheres of about this volume fraction, radii in [n/32, n/12.8] (1 inside)."""
    lo, hi = min(n) / 32.0, min(n) / 12.8
    vol = 4.0 / 3.0 * math.pi * (hi ** 4 - lo ** 4) / (4.0 * (hi - lo))
    count = max(1, round(-math.log(1.0 - fraction) * n[0] * n[1] * n[2] / vol))
    u = torch.rand((count, 4), generator=gen, dtype=torch.float64).tolist()
    mask = torch.zeros(n, dtype=torch.bool, device=DEV)
    for c in u:
        r = lo + (hi - lo) * c[3]
        at = [c[a] * n[a] for a in range(3)]
        s = [slice(max(0, math.floor(at[a] - r - 1)), min(n[a], math.ceil(at[a] + r + 1))) for a in range(3)]
        d = [(torch.arange(s[a].start, s[a].stop, device=DEV) + 0.5 - at[a]) ** 2 for a in range(3)]
        mask[s[0], s[1], s[2]] |= d[0][:, None, None] + d[1][None, :, None] + d[2] <= r * r
    return mask.to(torch.int32)


def problem_data(case, gen):
    """Phase map [x, y, z], materials (law, params, quat), reference medium and loads of a case."""
    n = (case["n1"], case["n2"], case["n3"])
    law, one = case["law"], (1.0, 0.0, 0.0, 0.0)
    bc = bc_table(case["bc"])
    if law in ("cubic", "cp"):
        g = case["grains"]
        phase = voronoi(n, g, gen)
        q = torch.randn((g, 4), generator=gen, dtype=torch.float64)
        q = (q / q.norm(dim=1, keepdim=True)).tolist()
        mats = [(F.FFTM_LAW_CUBIC_ELASTIC, CUBIC, v) if law == "cubic" else (F.FFTM_LAW_CP_FCC, CP, v) for v in q]
        ref = (CUBIC[1], 0.5 * (CUBIC[2] + 0.5 * (CUBIC[0] - CUBIC[1])))
    elif law == "iso10":  # one sphere, ten times stiffer, its centre within a few voxels of the middle
        r = n[0] / 4.0
        c = [0.5 * v + 4.0 * (float(torch.rand((), generator=gen)) - 0.5) for v in n]
        d = [(torch.arange(n[a], device=DEV) + 0.5 - c[a]) ** 2 for a in range(3)]
        phase = (d[0][:, None, None] + d[1][None, :, None] + d[2] <= r * r).to(torch.int32)
        a, b = lame(1.0, 0.3), lame(10.0, 0.3)
        mats = [(F.FFTM_LAW_ISO_ELASTIC, a, one), (F.FFTM_LAW_ISO_ELASTIC, b, one)]
        ref = (0.5 * (a[0] + b[0]), 0.5 * (a[1] + b[1]))
    elif law == "logj2":  # soft Neo-Hookean pores in a perfectly plastic matrix
        phase = spheres(n, 0.12, gen)
        a = lame(200.0, 0.3)
        mats = [(F.FFTM_LAW_LOG_J2, a + (0.3,), one), (F.FFTM_LAW_NEO_HOOKE, (20.0, 40.0), one)]
        ref = a
    else:
        phase = spheres(n, 0.30, gen)
        a, b = lame(200.0, 0.3), lame(200.0 if law == "j2bend" else 400.0, 0.3)
        matrix = (F.FFTM_LAW_J2_LINHARD, a + (0.3, 2.0), one) if law.startswith("j2") else (F.FFTM_LAW_ISO_ELASTIC, a, one)
        mats = [matrix, (F.FFTM_LAW_ISO_ELASTIC, b, one)]
        ref = (0.5 * (a[0] + b[0]), 0.5 * (a[1] + b[1]))
    loads = []
    for k in range(1, case["steps"] + 1):
        A, Q, mixed = np.zeros((3, 3)), np.zeros((3, 6)), 0
        if case["load"] == "bending":  # rotation of the x = L face about its mid-line, past yield
            th = 0.0016 * k * n[0] / n[1]
            A[0, 0], Q[0, 5] = -th * n[1] / (2.0 * n[0]), th / n[0]
        elif case["load"] == "torsion":  # rigid turn of the x = L face, linear in x
            s = 0.05 / 30
            Q[1, 4], Q[2, 5] = -s / n[0], s / n[0]
            A[1, 0], A[2, 0] = s * n[2] / (2.0 * n[0]), -s * n[1] / (2.0 * n[0])
        elif case["load"] == "stretch":
            A[0, 0] = 0.002
        else:
            a = next((a for a in range(3) if bc[a][0][a] == "D"), 0)
            A[a, a] = 1e-3 * k
            mixed = 0b111110 if case["load"] == "mixed" else 0
        for a in range(3):  # u* may not depend on a periodic coordinate
            if bc[a][0][0] == "P":
                A[:, a] = 0.0
        loads.append((A, Q, mixed))
    return n, phase, mats, bc, ref, loads


def nodes(n, bc):
    return tuple(n[a] if bc[a][0][0] == "P" else n[a] + 1 for a in range(3))


def field_of(case, gen):
    """A caller's node field (3, N1, N2, N3) in FP64: smooth displacements for ``residual``, the
    rough polarisation of a random medium for ``green``, zero where a component is not transformed."""
    n, bc = (case["n1"], case["n2"], case["n3"]), bc_table(case["bc"])
    N = nodes(n, bc)
    if case["op"] == "residual":
        c = torch.randn((1, 3, 7, 7, 7), generator=gen, dtype=torch.float64).to(DEV)
        f = torch.nn.functional.interpolate(c, size=N, mode="trilinear", align_corners=True)[0] * (1e-4 * min(n))
    else:
        small = torch.Generator(device=DEV)
        small.manual_seed(int(torch.randint(1 << 40, (), generator=gen)))
        f = torch.randn((3,) + N, generator=small, dtype=torch.float64, device=DEV)
    f = f.to(torch.float32).double() if case["precision"] != "fp64" else f
    return f * Reference.masks(n, bc)


class Handle:
    """A library problem on the current stream, freed with the state that holds it."""

    def __init__(self, case, n, phase, mats, bc, ref):
        self.ctx = F.fftm_ctx_create(0, torch.cuda.current_stream())
        desc, keep = F.make_desc(n, phase.cpu().numpy(), mats, bc, scheme=case["scheme"], lambda0=ref[0], mu0=ref[1],
                                 precision=case["precision"], tol=case["tol"], max_iter=2000)
        self.p = F.fftm_problem_create(self.ctx, desc)

    def __del__(self):
        if getattr(self, "p", None):
            F.fftm_problem_destroy(self.p)
            F.fftm_ctx_destroy(self.ctx)


def requests(case, seed):
    """The requests of a ``serve`` case: grids around the case's size, every family of the stream."""
    top = case["n1"]
    sides = [s for s in SIZES if top / 2 <= s <= top]
    bcs = ("D N P", "D N N", "D P P", "D D N", "N D P", "D P N", "D N P", "D N N")
    out = []
    for k in range(8):
        gen = torch.Generator().manual_seed(1000 * seed + k)
        s = sides[(3 * k) % len(sides)]
        c = dict(case, op="solve", n1=s, n2=s, n3=s, scheme="TETRA2" if k % 2 else "HEX1", bc=bcs[k],
                 law="cubic" if k % 3 == 0 else "iso2" if k % 3 == 1 else "j2", steps=2 if k % 3 == 2 else 1,
                 grains=s // 2)
        out.append((c, problem_data(c, gen)))
    return out


class Server:
    def __init__(self):
        self.s = F.fftm_server_create(0, 16 << 30, 4)

    def __del__(self):
        if getattr(self, "s", None):
            F.fftm_server_destroy(self.s)


def dtype_of(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def prepare(case, seed):
    torch.cuda.set_device(0)
    dt = dtype_of(case)
    if case["op"] == "serve":
        jobs = []
        for c, (n, phase, mats, bc, ref, loads) in requests(case, seed):
            desc = F.make_desc(n, phase.cpu().numpy(), mats, bc, scheme=c["scheme"], lambda0=ref[0], mu0=ref[1],
                               precision=c["precision"], tol=c["tol"], max_iter=2000)
            N = nodes(n, bc)
            u = np.zeros((3, N[2], N[1], N[0]), dtype=np.float64 if dt == torch.float64 else np.float32)
            jobs.append((desc, [(A, (0.0, 0.0, 0.0), Q) for A, Q, _ in loads], u))
        return {"op": "serve", "server": Server(), "jobs": jobs}
    gen = torch.Generator().manual_seed(seed)
    n, phase, mats, bc, ref, loads = problem_data(case, gen)
    h = Handle(case, n, phase, mats, bc, ref)
    N = nodes(n, bc)
    st = {"op": case["op"], "h": h, "loads": loads, "u": torch.empty((3, N[2], N[1], N[0]), dtype=dt, device=DEV)}
    st["u_out"] = "u" in case["out"].split(",")
    if case["op"] == "solve" and "stress" in case["out"]:
        size = F.fftm_field_bytes(h.p, F.FFTM_FIELD_STRESS) // dt.itemsize
        st["stress"] = torch.empty(size, dtype=dt, device=DEV)
    if case["op"] in ("residual", "green"):
        st["f"] = field_of(case, gen).permute(0, 3, 2, 1).to(dt).contiguous()
        st["norms"] = torch.empty(3, dtype=torch.float64, device=DEV)
        if case["op"] == "residual":
            F.fftm_set_load(h.p, loads[0][0])
    return st


def run(state):
    if state["op"] == "serve":
        s = state["server"].s
        ids = {}
        for k, (desc, loads, u) in enumerate(state["jobs"]):
            ids[F.fftm_server_submit(s, desc[0], loads, u_out=u)] = k
        left = len(ids)
        while left:
            for r in F.fftm_server_poll(s):
                if r["status"] != F.FFTM_OK:
                    raise RuntimeError("request %d: status %d %s" % (ids[r["id"]], r["status"], r["message"]))
                left -= 1
        return [u for _, _, u in state["jobs"]]
    p, u = state["h"].p, state["u"]
    if state["op"] == "residual":
        F.fftm_residual_noalloc(p, state["f"], u, state["norms"])
        return {"D": u, "norms": state["norms"].to(u.dtype)}
    if state["op"] == "green":
        F.fftm_set_field(p, F.FFTM_FIELD_WORK, state["f"])
        F.fftm_apply(p, F.FFTM_OP_GREEN_UPDATE)
        F.fftm_get_field(p, F.FFTM_FIELD_U, u)
        return {"u": u}
    F.fftm_reset_state(p)
    for A, Q, mixed in state["loads"]:
        F.fftm_set_load(p, A, Q=Q, mixed=mixed)
        st, rep, _, _ = F.fftm_solve_step(p)
        if st != F.FFTM_OK:
            raise RuntimeError("load step not converged: err %g after %d iterations" % (rep["err"], rep["iterations"]))
    out = {"mean_P": torch.tensor(rep["mean_P"], dtype=u.dtype)}
    if state["u_out"]:
        F.fftm_get_field(p, F.FFTM_FIELD_U, u)
        out["u"] = u
    if "stress" in state:
        F.fftm_get_field(p, F.FFTM_FIELD_STRESS, state["stress"])
        out["stress"] = state["stress"]
    return out


def work(case):
    """Per iteration: u and D of every node read or written once each in the residual (with the
    phase of every voxel) and once in the Green update, the four stored couples in every third
    iteration; the stencils, the law and five radix-2 transform passes for the arithmetic."""
    e = 8 if case["precision"] == "fp64" else 4
    if case["op"] == "serve":
        total = {"bytes": 0.0, "flops": 0.0}
        for k in range(8):
            sides = [s for s in SIZES if case["n1"] / 2 <= s <= case["n1"]]
            s = sides[(3 * k) % len(sides)]
            w = work(dict(case, op="solve", n1=s, n2=s, n3=s, scheme="TETRA2" if k % 2 else "HEX1", bc="D N N",
                          law="iso2", steps=2 if k % 3 == 2 else 1))
            total = {m: total[m] + w[m] for m in total}
        return total
    n = (case["n1"], case["n2"], case["n3"])
    vox, npp = n[0] * n[1] * n[2], 2 if case["scheme"] == "TETRA2" else 1
    N = nodes(n, bc_table(case["bc"]))
    nod = N[0] * N[1] * N[2]
    res_b, res_f = 6 * e * nod + 2 * vox, vox * (npp * (60 + (4000 if case["law"] == "cp" else 70)) + 60)
    lg = sum(math.log2(v) for v in n)
    green_b, green_f = 6 * e * nod, 3 * nod * (2 * 2.5 * lg + 20)
    if case["op"] == "residual":
        return {"bytes": res_b, "flops": res_f}
    if case["op"] == "green":
        return {"bytes": green_b, "flops": green_f}
    it = case["iters"] * case["steps"]
    out = (3 * e * nod if "u" in case["out"].split(",") else 0) + (6 * npp * e * vox if "stress" in case["out"] else 0)
    return {"bytes": it * (res_b + green_b + 27 * e * nod / 3) + out, "flops": it * (res_f + green_f + 66 * nod / 3)}


# ---- the same in 64 bits ---------------------------------------------------------------------
class Reference:
    """The discrete problem in plain FP64 torch, fields indexed [q, x, y, z]."""

    KIND = {("P", "P"): "DFT", ("N", "N"): "DCT1", ("N", "D"): "DCT3", ("D", "D"): "DST1", ("D", "N"): "DST3"}

    def __init__(self, case, data):
        self.n, self.phase, self.mats, self.bc, (self.lam0, self.mu0), _ = data
        self.tetra = case["scheme"] == "TETRA2"
        self.per = [self.bc[a][0][0] == "P" for a in range(3)]
        self.N = nodes(self.n, self.bc)
        self.kind = [[self.KIND[(self.bc[a][0][q], self.bc[a][1][q])] for a in range(3)] for q in range(3)]
        self.mask = self.masks(self.n, self.bc)
        self.phase = self.phase.long()
        self.C = torch.stack([self.stiffness(m) for m in self.mats]).to(DEV)
        j2 = [m[0] == F.FFTM_LAW_J2_LINHARD for m in self.mats]
        self.j2 = torch.tensor(j2, device=DEV)[self.phase] if any(j2) else None
        if self.j2 is not None:
            self.par = next(m[1] for m in self.mats if m[0] == F.FFTM_LAW_J2_LINHARD)
            pts = 2 if self.tetra else 1
            self.ep = torch.zeros((pts, 6) + self.n, dtype=torch.float64, device=DEV)
            self.pl = torch.zeros((pts,) + self.n, dtype=torch.float64, device=DEV)
        self.mat = {}
        for q in range(3):
            for a in range(3):
                k = (self.kind[q][a], self.n[a])
                if k not in self.mat:
                    fwd = self.matrix(*k)
                    self.mat[k] = (fwd.to(DEV), torch.linalg.inv(fwd).to(DEV))

    @staticmethod
    def span(kind, n):
        return {"DFT": (0, n), "DCT1": (0, n + 1), "DCT3": (0, n), "DST1": (1, n), "DST3": (1, n + 1)}[kind]

    @classmethod
    def masks(cls, n, bc):
        N = nodes(n, bc)
        m = torch.zeros((3,) + N, dtype=torch.float64, device=DEV)
        for q in range(3):
            s = [slice(*cls.span(cls.KIND[(bc[a][0][q], bc[a][1][q])], n[a])) for a in range(3)]
            m[q][s[0], s[1], s[2]] = 1.0
        return m

    @staticmethod
    def xi(kind, n):
        lo, hi = Reference.span(kind, n)
        k = torch.arange(hi - lo, dtype=torch.float64)
        return {"DFT": 2 * math.pi * k / n, "DCT1": math.pi * k / n, "DCT3": math.pi * (k + 0.5) / n,
                "DST1": math.pi * (k + 1) / n, "DST3": math.pi * (k + 0.5) / n}[kind]

    @staticmethod
    def matrix(kind, n):
        """Rows: outputs; columns: the node range (the DFT as real cosine and sine rows)."""
        lo, hi = Reference.span(kind, n)
        j = torch.arange(lo, hi, dtype=torch.float64)
        if kind == "DFT":
            k = torch.arange(n)
            arg = 2 * math.pi * ((torch.minimum(k, n - k)[:, None] * k) % n).double() / n
            return torch.where((2 * k <= n)[:, None], torch.cos(arg), -torch.sin(arg))
        arg = torch.outer(Reference.xi(kind, n), j)
        w = torch.full((hi - lo,), 2.0, dtype=torch.float64)
        if kind in ("DCT1", "DCT3"):
            w[0] = 1.0
        if kind in ("DCT1", "DST3"):
            w[-1] = 1.0
        return w * (torch.cos(arg) if kind in ("DCT1", "DCT3") else torch.sin(arg))

    @staticmethod
    def stiffness(m):
        """6 x 6 stiffness on (11, 22, 33, 23, 13, 12) strains, shears counted once (tensor values)."""
        law, c, quat = m
        C = torch.zeros((3, 3, 3, 3), dtype=torch.float64)
        I = torch.eye(3, dtype=torch.float64)
        if law == F.FFTM_LAW_CUBIC_ELASTIC:
            w, x, y, z = quat
            R = torch.tensor([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                              [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                              [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]], dtype=torch.float64)
            lam, mu, extra = c[1], c[2], c[0] - c[1] - 2 * c[2]
            C += extra * torch.einsum("ia,ja,ka,la->ijkl", R, R, R, R)
        else:
            lam, mu = c[0], c[1]
        C += lam * torch.einsum("ij,kl->ijkl", I, I)
        C += mu * (torch.einsum("ik,jl->ijkl", I, I) + torch.einsum("il,jk->ijkl", I, I))
        return torch.stack([torch.stack([C[i, j, k, l] * (1.0 if k == l else 2.0) for k, l in VOIGT]) for i, j in VOIGT])

    def corners(self, r, i):
        """(offset, sign) of the difference along axis i at point r; the scale goes with it."""
        for o in range(8):
            b = ((o >> 0) & 1, (o >> 1) & 1, (o >> 2) & 1)
            if not self.tetra:
                yield b, (1.0 if b[i] else -1.0) * 0.25
            elif (sum(b) & 1) == r:
                yield b, (1.0 if b[i] else -1.0) * 0.5

    def full(self, u):
        for a in range(3):
            if self.per[a]:
                u = torch.cat([u, u.narrow(1 + a, 0, 1)], dim=1 + a)
        return u

    def strain(self, uf, r):
        """sym grad (11, 22, 33, 23, 13, 12) at point r of a field on all n + 1 nodes."""
        n = self.n
        G = [[None] * 3 for _ in range(3)]
        for i in range(3):
            acc = 0.0
            for b, s in self.corners(r, i):
                acc = acc + s * uf[:, b[0]:b[0] + n[0], b[1]:b[1] + n[1], b[2]:b[2] + n[2]]
            for q in range(3):
                G[i][q] = acc[q]
        return torch.stack([0.5 * (G[i][j] + G[j][i]) for i, j in VOIGT])

    def ustar(self, A, Q):
        x = torch.meshgrid(*[torch.arange(v + 1, dtype=torch.float64, device=DEV) for v in self.n], indexing="ij")
        mono = (x[0] * x[0], x[1] * x[1], x[2] * x[2], x[1] * x[2], x[0] * x[2], x[0] * x[1])
        return torch.stack([sum(float(A[q][a]) * x[a] for a in range(3)) + sum(
            float(Q[q][k]) * mono[k] for k in range(6) if Q[q][k]) for q in range(3)])

    def stress(self, e, r):
        """(6, ...) stress at point r and the committed state that goes with it."""
        if self.mats[0][0] == F.FFTM_LAW_CUBIC_ELASTIC:
            s = torch.zeros_like(e)
            for i in range(6):
                for j in range(6):
                    s[i] += self.C[:, i, j][self.phase] * e[j]
            return s, None
        lam = torch.tensor([m[1][0] for m in self.mats], dtype=torch.float64, device=DEV)
        mu = torch.tensor([m[1][1] for m in self.mats], dtype=torch.float64, device=DEV)
        lam, mu = lam[self.phase], mu[self.phase]
        ee = e if self.j2 is None else e - self.ep[r]
        s = 2 * mu * ee
        s[:3] += lam * (ee[0] + ee[1] + ee[2])
        if self.j2 is None:
            return s, None
        d = s.clone()
        d[:3] -= (s[0] + s[1] + s[2]) / 3
        seq = torch.sqrt(1.5 * ((d[:3] ** 2).sum(0) + 2 * (d[3:] ** 2).sum(0)))
        _, m, sy, H = self.par
        dp = torch.where(self.j2, torch.clamp(seq - sy - H * self.pl[r], min=0.0), 0.0) / (3 * m + H)
        de = 1.5 * dp / seq.clamp(min=1e-300) * d
        return s - 2 * m * de, (self.ep[r] + de, self.pl[r] + dp)

    def divergence(self, S):
        """Node divergence of the point stresses S (points, 6, n): mirrored one layer outside, each
        component with the sign of its displacement's symmetry (minus across its own axis), the two
        tetrahedra exchanged; periodic axes wrap."""
        pts = S.shape[0]
        D = torch.zeros((3,) + self.N, dtype=torch.float64, device=DEV)
        for q in range(3):
            for i in range(3):
                c = i if i == q else 6 - i - q
                E = S[:, c]
                for a in range(3):
                    lo, hi = E.narrow(1 + a, 0, 1), E.narrow(1 + a, self.n[a] - 1, 1)
                    if self.per[a]:
                        lo, hi = hi, lo
                    else:
                        sg = [(1.0 if self.bc[a][f][q] == "N" else -1.0) * (-1.0 if i == a else 1.0) for f in (0, 1)]
                        lo, hi = sg[0] * lo.flip(0), sg[1] * hi.flip(0)
                    E = torch.cat([lo, E, hi], dim=1 + a)
                for r in range(pts):
                    for b, s in self.corners(1 - r if self.tetra else 0, i):
                        D[q] += (0.5 if self.tetra else 1.0) * s * E[r][
                            b[0]:b[0] + self.N[0], b[1]:b[1] + self.N[1], b[2]:b[2] + self.N[2]]
        return D * self.mask

    def evaluate(self, u, us):
        """D, stresses (points, 6, n) and states of u^f = u under the prescribed field us."""
        uf = self.full(u) + us
        S, states = [], []
        for r in range(2 if self.tetra else 1):
            s, z = self.stress(self.strain(uf, r), r)
            S.append(s)
            states.append(z)
        S = torch.stack(S)
        return self.divergence(S), S, states

    def green(self, f):
        out = torch.zeros_like(f)
        for q in range(3):
            k, n = self.kind[q], self.n
            s = tuple(slice(*self.span(k[a], n[a])) for a in range(3))
            x = f[q][s]
            sq = []
            for a in range(3):
                xi = self.xi(k[a], n[a])
                if k[a] == "DFT":
                    xi = torch.minimum(xi, 2 * math.pi - xi)
                sn, cs = torch.sin(xi / 2), torch.cos(xi / 2)
                cs[cs.abs() < 1e-14] = 0.0
                shape = [1, 1, 1]
                shape[a] = -1
                sq.append(((sn * sn).reshape(shape).to(DEV), (cs * cs).reshape(shape).to(DEV)))
            t = []
            for a in range(3):
                b, c = [v for v in range(3) if v != a]
                v = 4 * sq[a][0] * sq[b][1] * sq[c][1]
                t.append(v + 4 * sq[a][1] * sq[b][0] * sq[c][0] if self.tetra else v)
            den = 2 * self.mu0 * (t[0] + t[1] + t[2]) + self.lam0 * t[q]
            for a in range(3):
                x = torch.movedim(torch.movedim(x, a, -1) @ self.mat[(k[a], n[a])][0].T, -1, a)
            x = torch.where(den > 0, -x / den, 0.0)
            for a in range(3):
                x = torch.movedim(torch.movedim(x, a, -1) @ self.mat[(k[a], n[a])][1].T, -1, a)
            out[q][s] = x
        return out

    def solve(self, u, A, Q, mixed, tol, limit):
        """The fixed point u - Gamma(D), mixed by least squares over the last four iterates."""
        A, U, R = np.array(A), [], []
        for m in range(limit):
            D, S, states = self.evaluate(u, self.ustar(A, Q))
            err = math.sqrt(float((D * D).sum()) / (float((S[:, :3] ** 2).sum() + 2 * (S[:, 3:] ** 2).sum()) / S.shape[0]))
            mean = S.mean(dim=(0, 2, 3, 4)).tolist()
            free = [k for k in range(6) if (mixed >> k) & 1]
            norm = math.sqrt(sum(v * v for v in mean))
            if err < tol and all(abs(mean[k]) < tol * norm for k in free):
                break
            U, R = (U + [u])[-4:], (R + [D])[-4:]
            v, d = u, D
            if m % 3 == 2 and len(R) == 4:
                X = torch.stack([(x - D).reshape(-1) for x in R[:-1]])
                g = torch.linalg.lstsq((X @ X.T).cpu(), -(X @ D.reshape(-1)).cpu()).solution.tolist()
                v = u + sum(c * (x - u) for c, x in zip(g, U[:-1]))
                d = D + sum(c * (x - D) for c, x in zip(g, R[:-1]))
            u = v - self.green(d)
            nf = [k for k in free if k < 3]
            if nf:
                M = np.full((len(nf), len(nf)), self.lam0) + 2 * self.mu0 * np.eye(len(nf))
                for k, dv in zip(nf, np.linalg.solve(M, [-mean[k] for k in nf])):
                    A[k, k] += dv
            for k in free:
                if k >= 3:
                    i, j = VOIGT[k]
                    A[i, j] -= mean[k] / (2 * self.mu0)
                    A[j, i] -= mean[k] / (2 * self.mu0)
        if self.j2 is not None:
            for r, (ep, pl) in enumerate(states):
                self.ep[r], self.pl[r] = ep, pl
        return u, S


def exact(case, seed):
    if case["law"] in ("cp", "logj2"):
        return None
    if case["op"] == "serve":
        return [exact_solve(dict(c, out="u"), d, 1e-9)["u"] for c, d in requests(case, seed)]
    gen = torch.Generator().manual_seed(seed)
    data = problem_data(case, gen)
    if case["op"] == "solve":
        return exact_solve(case, data, 1e-3 * case["tol"])
    ref = Reference(case, data)
    f = field_of(case, gen)
    if case["op"] == "green":
        return {"u": ref.green(f).permute(0, 3, 2, 1)}
    D, S, _ = ref.evaluate(f, ref.ustar(data[5][0][0], np.zeros((3, 6))))
    sd = float((D * D).sum())
    sp = float((S[:, :3] ** 2).sum() + 2 * (S[:, 3:] ** 2).sum()) / S.shape[0]
    return {"D": D.permute(0, 3, 2, 1), "norms": torch.tensor([sd, sp, math.sqrt(sd / sp)], dtype=torch.float64)}


def exact_solve(case, data, tol):
    ref = Reference(case, data)
    u = torch.zeros((3,) + ref.N, dtype=torch.float64, device=DEV)
    for A, Q, mixed in data[5]:
        u, S = ref.solve(u, A, Q, mixed, tol, 500)
    out = {"mean_P": S.mean(dim=(0, 2, 3, 4))}
    if case["op"] != "solve" or "u" in case["out"].split(","):
        out["u"] = u.permute(0, 3, 2, 1)
    if "stress" in case["out"]:
        out["stress"] = S.permute(0, 1, 4, 3, 2).reshape(-1)
    return out
