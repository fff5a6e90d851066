"""Timed workloads of the GB300 strain-gradient crystal-plasticity increment.

Each case is work that a user of the library has it do through its public
entry points, from the blocks of an increment (the Galerkin projection with
and without a handle, the GND hardening, the local update with its tangent)
to whole increments: small and latency-bound, the 64^3 polycrystal, mixed
precision, a batch of different RVEs, and an increment that carries the
parameter sensitivities.  Inputs are made from a seed: periodic Voronoi
polycrystals, uniformly random orientations, and states as a tension test
passes through them.  ``exact`` evaluates the same equations with torch in 64
bits, with no code of the library.
"""
import math

import numpy as np
import torch

import paper_1910_01946_gb300 as pkg

# Slip rate, exponent and interaction coefficients as in rvegen, four FCC metals
FLOW = dict(alpha=0.3, q=(0.122, 0.122, 0.657, 0.084, 0.137, 0.118), q_normalise=True, gdot0=1e-3, n=20.0,
            rho0_total=1e12, mu=0.0, gnd_enabled=True)
METALS = {
    "Cu": dict(C11=168.4e3, C12=121.4e3, C44=75.4e3, b=0.256e-9, tau0=10.0, K=6.0, yc=15e-9, **FLOW),
    "Al": dict(C11=108.2e3, C12=61.3e3, C44=28.5e3, b=0.286e-9, tau0=5.0, K=9.0, yc=56e-9, **FLOW),
    "Ag": dict(C11=124.0e3, C12=93.4e3, C44=46.1e3, b=0.289e-9, tau0=10.0, K=5.0, yc=12.5e-9, **FLOW),
    "Ni": dict(C11=246.5e3, C12=147.3e3, C44=124.7e3, b=0.249e-9, tau0=10.0, K=11.0, yc=14e-9, **FLOW),
}
RATE = 1e-3                                   # strain rate [1/s]
# strain of the increments that lead a specimen through its plastic onset
# before the increment that is timed
ONSET = (2e-4, 2e-4, 3e-4, 3e-4)
STEP = 1e-3
# strain-controlled components: uniaxial tension along x, or full strain control
MASKS = {"uniaxial": (1, 0, 0, 1, 0, 0, 1, 1, 0), "strain": (1,) * 9}


# ------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest projection: a few launches, all latency
        dict(name="project-16", kind="project", n0=16, n1=16, n2=16, control="uniaxial"),
        # ragged box with an odd edge: mixed-radix transforms, no row-strip stencils
        dict(name="project-36x54x27", kind="project", n0=36, n1=54, n2=27, control="strain"),
        # the projection of the largest workload (128^3 voxels)
        dict(name="project-128", kind="project", n0=128, n1=128, n2=128, control="uniaxial"),
        # the projection for callers that cannot allocate: nine fields in Fourier space
        dict(name="noalloc-64", kind="noalloc", n0=64, n1=64, n2=64, control="uniaxial"),
        # Nye tensor, GND densities and critical stresses at the start of an increment
        dict(name="hardening-64", kind="hardening", n0=64, n1=64, n2=64, grains=100, metal="Cu"),
        # material-point evaluations with the consistent tangent, as a caller with a solver of its own uses them
        dict(name="constitutive-32", kind="constitutive", n0=32, n1=32, n2=32, grains=40, metal="Cu", precision=0),
        dict(name="constitutive-64-mixed", kind="constitutive", n0=64, n1=64, n2=64, grains=100, metal="Al",
             precision=1),
        # one increment of a small RVE (parameter studies, tests): latency-bound
        dict(name="step-16", kind="step", n0=16, n1=16, n2=16, grains=8, metal="Cu", precision=0),
        # one increment of the benchmark polycrystal in both precisions
        dict(name="step-64", kind="step", n0=64, n1=64, n2=64, grains=100, metal="Cu", precision=0),
        dict(name="step-64-mixed", kind="step", n0=64, n1=64, n2=64, grains=100, metal="Cu", precision=1),
        # several RVEs of a grain-size study advanced together
        dict(name="batch-32-48-64", kind="batch", edges="32,48,64", grains=30, metals="Cu,Al,Ni", precision=1),
        # calibration: an increment that also carries d<P>/d(tau0, K, alpha, b)
        dict(name="sensitivity-32", kind="sensitivity", n0=32, n1=32, n2=32, grains=16, metal="Cu", precision=0),
    ]


def draw(rng):
    def edge(lo, hi, even=True):
        sizes = [2 ** a * 3 ** b for a in range(10) for b in range(6)]
        sizes = [s for s in sizes if lo <= s <= hi and (s % 2 == 0 or not even)]
        want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        return min(sizes, key=lambda s: abs(math.log(s / want)))

    def box(lo, hi):
        return dict(n0=edge(lo, hi), n1=edge(lo, hi), n2=edge(lo, hi, even=False))

    kind = rng.choice(("project", "noalloc", "hardening", "constitutive", "step", "step", "batch", "sensitivity"))
    metal = rng.choice(sorted(METALS))
    if kind == "project":
        return dict(kind=kind, **box(8, 128), control=rng.choice(sorted(MASKS)))
    if kind == "noalloc":
        return dict(kind=kind, **box(8, 64), control=rng.choice(sorted(MASKS)))
    if kind == "hardening":
        return dict(kind=kind, **box(16, 96), grains=rng.randint(4, 200), metal=metal)
    if kind == "constitutive":
        return dict(kind=kind, **box(8, 64), grains=rng.randint(4, 100), metal=metal, precision=rng.randint(0, 1))
    if kind == "step":
        return dict(kind=kind, **box(12, 54), grains=rng.randint(4, 40), metal=metal, precision=rng.randint(0, 1))
    if kind == "sensitivity":
        return dict(kind=kind, **box(8, 24), grains=rng.randint(4, 12), metal=metal, precision=0)
    return dict(kind=kind, edges=",".join(str(edge(16, 48)) for _ in range(rng.randint(2, 4))),
                grains=rng.randint(4, 30), metals="%s,%s" % (metal, rng.choice(sorted(METALS))), precision=1)


def parts(case):
    """The RVEs of a case, each as a case of its own."""
    if case["kind"] != "batch":
        return [case]
    metals = case["metals"].split(",")
    return [dict(kind="step", n0=int(e), n1=int(e), n2=int(e), grains=case["grains"], metal=metals[i % len(metals)],
                 precision=case["precision"]) for i, e in enumerate(case["edges"].split(","))]


# ------------------------------------------------------------------ inputs
def microstructure(case, seed):
    """Grain map (n2, n1, n0), quaternions (w, x, y, z) and edge length [m]."""
    rng = np.random.default_rng((seed, 1))
    g = case.get("grains", 1)
    pts, quat = rng.random((g, 3)), rng.standard_normal((g, 4))
    axes = [(torch.arange(case[k], dtype=torch.float64, device="cuda") + 0.5) / case[k] for k in ("n2", "n1", "n0")]
    best = torch.full([len(a) for a in axes], 9.0, dtype=torch.float64, device="cuda")
    gid = torch.zeros_like(best, dtype=torch.int32)
    for i in range(g):
        d = [(a - float(pts[i, k])).abs() for a, k in zip(axes, (2, 1, 0))]
        z, y, x = (torch.minimum(t, 1 - t) ** 2 for t in d)
        dist = z[:, None, None] + y[None, :, None] + x[None, None, :]
        gid = torch.where(dist < best, i, gid)
        best = torch.minimum(best, dist)
    edge = 20e-6 * (math.pi * g / 6) ** (1 / 3)
    return gid.cpu().numpy(), quat / np.linalg.norm(quat, axis=1, keepdims=True), edge


def noise(case, seed, ncomp):
    """Standard normal values (ncomp, nvox) on the GPU."""
    gen = torch.Generator("cuda").manual_seed(seed)
    nvox = case["n0"] * case["n1"] * case["n2"]
    return torch.randn(ncomp, nvox, generator=gen, device="cuda", dtype=torch.float64)


def eye9():
    return torch.eye(3, dtype=torch.float64, device="cuda").reshape(9, 1)


def stress_field(case, seed):
    """A stress-like field: a macroscopic tension and its fluctuations [MPa]."""
    X = 15.0 * noise(case, seed, 9)
    X[0] += 60.0
    return X


def plastic_state(case, seed):
    """F, Fp and rho_SSD (component, voxel) of a specimen some increments into a tension test."""
    z = noise(case, seed, 9 + 9 + 12)
    stretch = torch.diag(torch.tensor([2e-3, -8e-4, -8e-4], dtype=torch.float64, device="cuda")).reshape(9, 1)
    slip = 5e-4 * z[9:18]
    slip[0::4] -= slip[0::4].mean(dim=0)                    # isochoric to first order
    return eye9() + stretch + 5e-4 * z[:9], eye9() + 0.8 * stretch + slip, (1e12 / 12) * torch.exp(0.5 * z[18:])


def increment(strain):
    """Macroscopic step and its duration."""
    return np.array([strain] + [0.0] * 8), strain / RATE


# ------------------------------------------------------------------ the library's side
def put(rve, name, field):
    """Sets a committed field from device memory."""
    torch.cuda.current_stream().synchronize()
    which, _ = pkg.FIELDS[name]
    status = pkg.rve_set_fields(rve.h, which, field.data_ptr(), field.numel() * 8, 1)
    if status != pkg.RVE_OK:
        raise RuntimeError("rve_set_fields: %d" % status)


def specimen(case, seed):
    """An RVE with the plastic onset behind it, and its checkpoint in pinned host memory."""
    gid, quat, edge = microstructure(case, seed)
    rve = pkg.RVE(gid, quat, METALS[case["metal"]], edge, own_stream=True, precision=case["precision"])
    for strain in ONSET:
        dF, dt = increment(strain)
        rve.step(dF, MASKS["uniaxial"], np.zeros(9), dt)
    held = torch.empty(pkg.rve_checkpoint_bytes(rve.h), dtype=torch.uint8, pin_memory=True)
    if pkg.rve_checkpoint(rve.h, held.numpy()) != pkg.RVE_OK:
        raise RuntimeError("rve_checkpoint")
    return rve, held


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("project", "noalloc"):
        X = stress_field(case, seed)
        s = dict(X=X, Y=torch.empty_like(X), mask=np.array(MASKS[case["control"]], dtype=np.uint8))
        if kind == "project":
            gid = np.zeros((case["n2"], case["n1"], case["n0"]), dtype=np.int32)
            s["rve"] = pkg.RVE(gid, [[1.0, 0, 0, 0]], METALS["Cu"], 1e-5)
    elif kind in ("hardening", "constitutive"):
        gid, quat, edge = microstructure(case, seed)
        rve = pkg.RVE(gid, quat, METALS[case["metal"]], edge, precision=case.get("precision", 0))
        for name, field in zip(("F", "FP", "RHO_SSD"), plastic_state(case, seed)):
            put(rve, name, field)
        s = dict(rve=rve)
    else:
        s = dict(rves=[specimen(c, seed + 1000 * i) for i, c in enumerate(parts(case))])
        if kind == "sensitivity":
            s["rves"][0][0].enable_sensitivity()
    return dict(s, case=case)


def fields(rve, *names):
    return {name: rve.field(name, device=True) for name in names}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "project":
        return state["rve"].project(state["mask"], state["X"], state["Y"])
    if kind == "noalloc":
        status = pkg.rve_project_noalloc(case["n0"], case["n1"], case["n2"], 1e-5, state["mask"],
                                         state["X"].data_ptr(), state["Y"].data_ptr(),
                                         torch.cuda.current_stream().cuda_stream)
        if status != pkg.RVE_OK:
            raise RuntimeError("rve_project_noalloc: %d" % status)
        return state["Y"]
    if kind == "hardening":
        state["rve"].eval_hardening()
        return fields(state["rve"], "NYE", "RHO_GND18", "RHO_GND", "TAUC")
    if kind == "constitutive":
        _, failed = state["rve"].eval_constitutive(STEP / RATE)
        return dict(fields(state["rve"], "P_EVAL", "S_EVAL", "DGAM", "TANGENT"), failed=failed)
    rves = [r for r, _ in state["rves"]]
    for rve, held in state["rves"]:
        rve.restore(held.numpy())
    dF, dt = increment(STEP)
    if kind == "batch":
        pkg.step_batch(rves, dF, MASKS["uniaxial"], np.zeros(9), dt)
    else:
        rves[0].step(dF, MASKS["uniaxial"], np.zeros(9), dt)
    out = [dict(fields(r, "F", "FP", "P", "S", "RHO_SSD", "RHO_GND"), macro=np.stack(r.macro_stress())) for r in rves]
    if kind == "sensitivity":
        out[0]["dP"] = rves[0].stress_sensitivity()
    return out


# ------------------------------------------------------------------ work
def work(case):
    """Bytes and operations of one pass.  An increment reads and writes its
    state once; its operations assume four local evaluations, three tangents
    and 60 conjugate-gradient iterations per tangent."""
    if case["kind"] == "batch":
        each = [work(c) for c in parts(case)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    n = case["n0"] * case["n1"] * case["n2"]
    fft = 5.0 * math.log2(n)                        # per field, forward and inverse, real data
    if case["kind"] == "project":
        return {"bytes": 144.0 * n, "flops": (54 + 3 * fft) * n}
    if case["kind"] == "noalloc":
        return {"bytes": 144.0 * n, "flops": (25 + 9 * fft) * n}
    if case["kind"] == "hardening":
        return {"bytes": 8.0 * (9 + 12 + 51) * n, "flops": (700 + 9 * fft) * n}
    if case["kind"] == "constitutive":
        return {"bytes": 8.0 * (9 + 9 + 12 + 9 + 6 + 12 + 81) * n, "flops": (450 + 4 * 500 + 3 * 1442 + 7744) * n}
    solves = 3 + (4 if case["kind"] == "sensitivity" else 0)
    return {"bytes": 8.0 * 2 * 54 * n,
            "flops": (4 * (450 + 3 * 500 + 2 * 1442) + 3 * 7744 + 60 * solves * (198 + 118 + 3 * fft)) * n}


# ------------------------------------------------------------------ the same in 64 bits with torch
def outer(a, b):
    return torch.einsum("...i,...j->...ij", a, b)


def inv3(A):
    """Inverse of 3 x 3 matrices by cross products (torch's batched inverse is slow on so many small ones)."""
    a, b, c = A.unbind(dim=-1)
    rows3 = torch.stack([torch.linalg.cross(b, c), torch.linalg.cross(c, a), torch.linalg.cross(a, b)], dim=-2)
    return rows3 / (a * rows3[..., 0, :]).sum(dim=-1)[..., None, None]


def solve6(A, b):
    """x of A x = b for many 6 x 6 matrices close to a positive definite one, by Gauss-Jordan elimination."""
    M = torch.cat([A, b.unsqueeze(-1)], dim=-1)
    for k in range(6):
        row = M[:, k:k + 1] / M[:, k:k + 1, k:k + 1]
        M = M - M[:, :, k:k + 1] * row
        M[:, k:k + 1] = row
    return M[:, :, 6]


def crystal():
    """Unit slip directions and normals of the 12 systems, unit screw directions."""
    s = [(0, 1, -1), (-1, 0, 1), (1, -1, 0), (0, 1, -1), (1, 0, 1), (1, 1, 0),
         (0, 1, 1), (1, 0, -1), (1, 1, 0), (0, 1, 1), (1, 0, 1), (1, -1, 0)]
    m = [(1, 1, 1)] * 3 + [(-1, 1, 1)] * 3 + [(1, -1, 1)] * 3 + [(1, 1, -1)] * 3
    w = [(0, 1, -1), (1, 0, -1), (1, -1, 0), (0, 1, 1), (1, 0, 1), (1, 1, 0)]
    return [torch.tensor(v, dtype=torch.float64, device="cuda") / math.sqrt(sum(x * x for x in v[0])) for v in (s, m, w)]


def interaction(metal):
    """12 x 12 interaction matrix from the geometry of each pair."""
    s, m, _ = (v.cpu().numpy() for v in crystal())
    q = np.zeros((12, 12))
    for a in range(12):
        for b in range(12):
            ss, mm = s[a] @ s[b], m[a] @ m[b]
            j = s[a] - np.sign(ss) * s[b]
            k = (0 if a == b else 1 if abs(mm) > 0.99 else 2 if abs(ss) > 0.99 else 3 if abs(ss) < 0.01
                 else 4 if min(abs(j @ m[a]), abs(j @ m[b])) < 1e-9 else 5)
            q[a, b] = metal["q"][k] / metal["q"][0]
    return torch.tensor(q, device="cuda")


class Material64:
    """The constitutive law on all voxels at once, in the crystal frame."""

    def __init__(self, case, seed):
        gid, quat, self.edge = microstructure(case, seed)
        self.m = m = METALS[case["metal"]]
        self.h = self.edge / case["n0"]
        w, x, y, z = quat.T
        R = np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y)],
                      [2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x)],
                      [2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)]])
        self.R = torch.tensor(R, device="cuda").permute(2, 0, 1)[torch.from_numpy(gid.reshape(-1).astype(np.int64)).cuda()]
        self.mu = 3 * m["C44"] * (m["C11"] - m["C12"]) / (4 * m["C44"] + m["C11"] - m["C12"])
        s, n, w = crystal()
        self.schmid = outer(s, n)                                       # (12, 3, 3)
        A = torch.cat([outer(s, torch.linalg.cross(n, s)), outer(w, w)]).reshape(18, 9).T
        self.Ainv = A.T @ torch.linalg.inv(A @ A.T) / m["b"]
        self.screw = (s @ w.T).abs().argmax(dim=1)
        self.q = interaction(m)
        self.I = torch.eye(3, dtype=torch.float64, device="cuda")
        E = torch.zeros(6, 3, 3, dtype=torch.float64, device="cuda")    # symmetric basis, Voigt order
        self.voigt = [(0, 0), (1, 1), (2, 2), (1, 2), (0, 2), (0, 1)]
        for k, (i, j) in enumerate(self.voigt):
            E[k, i, j] = E[k, j, i] = 1.0
        self.basis = E
        self.tau_of = torch.einsum("kij,aij->ak", E, self.schmid)       # tau^a = tau_of[a] . S

    def to_crystal(self, X):
        return self.R.mT @ X @ self.R

    def to_sample(self, X):
        return self.R @ X @ self.R.mT

    def pick(self, X):
        return torch.stack([X[..., i, j] for i, j in self.voigt], dim=-1)

    def stiff(self, E):
        """Cubic stiffness on tensor components in Voigt order."""
        m = self.m
        tr = E[..., :1] + E[..., 1:2] + E[..., 2:3]
        return torch.cat([(m["C11"] - m["C12"]) * E[..., :3] + m["C12"] * tr, 2 * m["C44"] * E[..., 3:]], dim=-1)

    def hardening(self, nye, rho_ssd):
        m = self.m
        rho18 = self.to_crystal(nye).reshape(-1, 9) @ self.Ainv.T
        gnd = rho18[:, :12].abs() + 0.5 * rho18[:, 12:].abs()[:, self.screw]
        rho = rho_ssd + gnd
        tauc = m["tau0"] + m["alpha"] * self.mu * m["b"] * torch.sqrt(rho @ self.q.T)
        return rho18, gnd, tauc, m["K"] / torch.sqrt(rho.sum(dim=1, keepdim=True) - rho)

    def residual(self, S, Fe0, tauc, dt):
        m = self.m
        x = (S @ self.tau_of.T) / tauc
        dg = dt * m["gdot0"] * x.abs() ** m["n"] * x.sign()
        far = ~(dg.abs() <= 0.1).all(dim=1, keepdim=True)              # beyond the slips a step may take
        dg = torch.where(far, 0.0, dg)
        slope = dt * m["gdot0"] * m["n"] * x.abs() ** (m["n"] - 1) / tauc
        Minv = inv3(self.I + torch.einsum("va,aij->vij", dg, self.schmid))
        Fe = Fe0 @ Minv
        r = S - self.stiff(self.pick(0.5 * (Fe.mT @ Fe - self.I)))
        return torch.where(far, torch.inf, r), dg, slope, Minv, Fe

    def dM(self, slope):
        """dM/dS: (v, 6, 3, 3)."""
        return torch.einsum("va,ak,aij->vkij", slope, self.tau_of, self.schmid)

    def jacobian(self, slope, Minv, Fe):
        X = (Fe.mT @ Fe)[:, None] @ self.dM(slope) @ Minv[:, None]
        return torch.eye(6, dtype=torch.float64, device="cuda") + self.stiff(self.pick(0.5 * (X + X.mT))).mT

    def update(self, F, Fp0, tauc, S, dt):
        """S (crystal, Voigt), slips, P (sample) and what the tangent needs."""
        Ft, Fi = self.to_crystal(F), self.to_crystal(inv3(Fp0))
        Fe0 = Ft @ Fi
        S = S.clone()
        r = self.residual(S, Fe0, tauc, dt)[0]
        reset = ~torch.isfinite(r).all(dim=1)
        S[reset] = 0.0
        norm = self.residual(S, Fe0, tauc, dt)[0].abs().amax(dim=1)
        live = torch.arange(len(S), device="cuda")
        for _ in range(60):
            live = live[norm[live] > 2e-16 * self.mu]
            if not len(live):
                break
            r, _, slope, Minv, Fe = self.residual(S[live], Fe0[live], tauc[live], dt)
            step = solve6(self.jacobian(slope, Minv, Fe), -r)
            lam = torch.ones(len(live), 1, dtype=torch.float64, device="cuda")
            better = torch.zeros(len(live), dtype=torch.bool, device="cuda")
            for _ in range(30):
                trial = S[live] + lam * step
                tn = self.residual(trial, Fe0[live], tauc[live], dt)[0].abs().amax(dim=1)
                better = tn < norm[live]
                if bool((better | (norm[live] < 1e-13 * self.mu)).all()):
                    break
                lam = torch.where(better[:, None], lam, 0.5 * lam)
            S[live[better]] = trial[better]
            norm[live[better]] = tn[better]
            live = live[better]
        _, dg, slope, Minv, Fe = self.residual(S, Fe0, tauc, dt)
        Sf = torch.einsum("vk,kij->vij", S, self.basis)
        Fpi = Fi @ Minv
        P = self.to_sample(Ft @ Fpi @ Sf @ Fpi.mT)
        return S, dg, P, (Ft, Fpi, Sf, slope, Minv, Fe)

    def tangent(self, kept):
        """dP_ij / dF_kl as (v, 9, 9), sample frame."""
        Ft, Fpi, Sf, slope, Minv, Fe = kept
        J, dM = self.jacobian(slope, Minv, Fe), self.dM(slope)
        Q, W = Fpi @ Sf @ Fpi.mT, Sf @ Fpi.mT
        K = torch.empty(len(Ft), 9, 9, dtype=torch.float64, device="cuda")
        for k in range(3):
            for l in range(3):
                dF = outer(self.R[:, k], self.R[:, l])                  # R^T e_k e_l^T R
                X = Fe.mT @ dF @ Fpi
                dS = solve6(J, self.stiff(self.pick(0.5 * (X + X.mT))))
                A = -Fpi @ torch.einsum("vk,vkij->vij", dS, dM) @ Minv @ W
                dQ = A + A.mT + Fpi @ torch.einsum("vk,kij->vij", dS, self.basis) @ Fpi.mT
                K[:, :, 3 * k + l] = self.to_sample(dF @ Q + Ft @ dQ).reshape(-1, 9)
        return K


class Spectral64:
    """The rotated-scheme derivative and what is built from it."""

    def __init__(self, case):
        self.shape = (case["n2"], case["n1"], case["n0"])
        shift, wave = [], []
        for n in (case["n0"], case["n1"], case["n2"]):
            k = torch.fft.fftfreq(n, dtype=torch.float64, device="cuda")
            e = torch.exp(2j * math.pi * k)
            wave.append(torch.where(k == -0.5, -1.0 + 0j, e))
        ex, ey, ez = wave[0][None, None, :], wave[1][None, :, None], wave[2][:, None, None]
        self.D = torch.stack([(ex - 1) * (ey + 1) * (ez + 1), (ex + 1) * (ey - 1) * (ez + 1),
                              (ex + 1) * (ey + 1) * (ez - 1)])
        # symbols that vanish at a Nyquist frequency do so exactly
        norm = (self.D.abs() ** 2).sum(dim=0)
        self.unit = torch.where(norm > 0, self.D / torch.sqrt(torch.where(norm > 0, norm, 1.0)), 0)

    def spectrum(self, X):                                              # (9, nvox) -> (3, 3, grid)
        return torch.fft.fftn(X.reshape((3, 3) + self.shape), dim=(2, 3, 4))

    def project(self, X, mask):
        """G* of a field (9, nvox): compatible part, and the mean of the stress-controlled components."""
        Y = torch.einsum("jzyx,izyx->ijzyx", self.unit,
                         torch.einsum("lzyx,ilzyx->izyx", self.unit.conj(), self.spectrum(X)))
        Y = torch.fft.ifftn(Y, dim=(2, 3, 4)).real.reshape(9, -1)
        keep = torch.tensor([0.0 if c else 1.0 for c in mask], dtype=torch.float64, device="cuda").reshape(9, 1)
        return Y + keep * X.mean(dim=1, keepdim=True)

    def nye(self, Fp, h):
        """G_ij = -eps_jkl d_k Fp_il, (9, nvox) -> (nvox, 3, 3)."""
        f, D = self.spectrum(Fp), self.D / (4 * h)
        G = torch.stack([D[2] * f[:, 1] - D[1] * f[:, 2], D[0] * f[:, 2] - D[2] * f[:, 0],
                         D[1] * f[:, 0] - D[0] * f[:, 1]], dim=1)
        return torch.fft.ifftn(G, dim=(2, 3, 4)).real.reshape(9, -1).T.reshape(-1, 3, 3)


def rows(X):
    """(9, nvox) -> (nvox, 3, 3)"""
    return X.T.reshape(-1, 3, 3)


def columns(X):
    """(nvox, ...) -> (components, nvox)"""
    return X.reshape(len(X), -1).T.contiguous()


def tension64(case, seed):
    """The tension test of a step case from the pristine state, its last increment's fields."""
    mat, spec = Material64(case, seed), Spectral64(case)
    m, mask = mat.m, MASKS["uniaxial"]
    nv = len(mat.R)
    F = eye9().repeat(1, nv)
    Fp, S = rows(F), torch.zeros(nv, 6, dtype=torch.float64, device="cuda")
    rho = torch.full((nv, 12), m["rho0_total"] / 12, dtype=torch.float64, device="cuda")
    for strain in ONSET + (STEP,):
        dF, dt = increment(strain)
        _, gnd, tauc, ell = mat.hardening(spec.nye(columns(Fp), mat.h), rho)
        F = F + torch.tensor(dF, device="cuda").reshape(9, 1)

        def evaluate(F, S):
            S, dg, P, kept = mat.update(rows(F), Fp, tauc, S, dt)
            P = columns(P)
            R = spec.project(P, mask)
            return S, dg, P, kept, R, float(R.norm()) / float(P.mean(dim=1).norm()) / math.sqrt(nv)

        S, dg, P, kept, R, res = evaluate(F, S)
        polished = False
        for _ in range(60):
            if polished:
                break
            polished = res <= 1e-11                         # one iteration beyond the usual tolerance
            K = mat.tangent(kept)
            x, r = torch.zeros_like(R), -R
            p, rr = r, r.square().sum()
            stop = rr * max(1e-12, min(1e-2, res)) ** 2
            for it in range(2000):
                q = spec.project(columns(K @ p.T.unsqueeze(-1)), mask)
                a = rr / (p * q).sum()
                x, r = x + a * p, r - a * q
                rr, old = r.square().sum(), rr
                if it % 8 == 7 and bool(rr <= stop):
                    break
                p = r + (rr / old) * p
            lam = 1.0
            while lam > 1e-3:
                new = evaluate(F + lam * x, S)
                if new[5] < res:
                    break
                lam *= 0.5
            if not new[5] < res:
                break
            F = F + lam * x
            S, dg, P, kept, R, res = new
        M = mat.I + torch.einsum("va,aij->vij", dg, mat.schmid)
        Fp = mat.to_sample(M) @ Fp
        rho = (rho + dg.abs() / (m["b"] * ell)) / (1 + 2 * m["yc"] * dg.abs() / m["b"])
    f, p = rows(F), rows(P)
    cauchy = p @ f.mT / torch.linalg.det(f)[:, None, None]
    sample = mat.pick(mat.to_sample(torch.einsum("vk,kij->vij", S, mat.basis)))
    return dict(F=F, FP=columns(Fp), P=P, S=columns(sample), RHO_SSD=columns(rho), RHO_GND=columns(gnd),
                macro=torch.stack([P.mean(dim=1).reshape(3, 3), cauchy.mean(dim=0)]).cpu().numpy())


def exact(case, seed):
    kind = case["kind"]
    if kind in ("project", "noalloc"):
        return Spectral64(case).project(stress_field(case, seed), MASKS[case["control"]])
    if kind in ("hardening", "constitutive"):
        mat, spec = Material64(case, seed), Spectral64(case)
        F, Fp, rho = plastic_state(case, seed)
        nye = spec.nye(Fp, mat.h)
        rho18, gnd, tauc, _ = mat.hardening(nye, rho.T)
        if kind == "hardening":
            return dict(NYE=columns(nye), RHO_GND18=columns(rho18), RHO_GND=columns(gnd), TAUC=columns(tauc))
        S, dg, P, kept = mat.update(rows(F), rows(Fp), tauc, torch.zeros(len(rho.T), 6, dtype=torch.float64, device="cuda"),
                                    STEP / RATE)
        sample = mat.pick(mat.to_sample(torch.einsum("vk,kij->vij", S, mat.basis)))
        return dict(P_EVAL=columns(P), S_EVAL=columns(sample), DGAM=columns(dg), TANGENT=columns(mat.tangent(kept)),
                    failed=None)
    # whole tension tests take torch too long beyond some thousand voxels, and
    # the sensitivities would need many of them
    if kind == "sensitivity" or sum(c["n0"] * c["n1"] * c["n2"] for c in parts(case)) > 5000:
        return None
    return [tension64(c, seed + 1000 * i) for i, c in enumerate(parts(case))]
