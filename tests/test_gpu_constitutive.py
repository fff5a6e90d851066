"""The local update (FP32 directions, FP64 residual) and the consistent tangent
in the sample frame against the oracle, at the edges of their dispatch: voxel
counts that fill no warp, one and two voxels past a block, flow-rule exponents
with and without the integer fast path, a stiffness without a positive definite
compliance; and the mixed-precision entry point (FP64 directions, FP32 tangent)
against the FP64 one."""
import numpy as np
import pytest

import rvegen
from oracle import solver

pytestmark = pytest.mark.gpu

CASES = {
    "one block": (dict(), (4, 4, 4)),
    "two voxels": (dict(), (1, 2, 2)),
    "past a block": (dict(), (9, 6, 12)),
    "integer exponent": (dict(n=7.0), (3, 4, 6)),
    "real exponent": (dict(n=12.5), (3, 4, 6)),
    "linear flow": (dict(n=1.0), (2, 4, 4)),
    "soft bulk": (dict(C11=100e3, C12=-55e3, C44=60e3, mu=45e3), (2, 4, 6)),
}


@pytest.fixture(scope="module")
def pkg():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1910_01946_gb300 import _build
    _build.build()
    import paper_1910_01946_gb300 as p
    p.load_library()
    return p


def relerr(a, b):
    return float(np.abs(a - b).max() / max(np.abs(b).max(), 1e-300))


def state(case, seed=23):
    over, shape = CASES[case]
    n2, n1, n0 = shape
    gid, _ = rvegen.voronoi_grain_map(0, 3, seed, shape=(n0, n1, n2))
    mat = rvegen.material("Cu", **over)
    rng = np.random.default_rng(seed)
    F = np.eye(3) + np.diag([2e-3, -6e-4, -6e-4]) + 5e-4 * rng.standard_normal(shape + (3, 3))
    Fp = np.eye(3) + 5e-4 * rng.standard_normal(shape + (3, 3))
    return gid, rvegen.random_quaternions(3, seed + 1), mat, F, Fp


def evaluate(pkg, args, **options):
    gid, quat, mat, F, Fp = args
    g = pkg.RVE(gid, quat, mat, 2e-5, **options)
    g.set_field("F", F.reshape(gid.shape + (9,)))
    g.set_field("FP", Fp.reshape(gid.shape + (9,)))
    _, failed = g.eval_constitutive(1.0)
    assert failed == 0
    out = {k: g.field(k).reshape(gid.size, -1) for k in ("P_EVAL", "S_EVAL", "DGAM", "TANGENT")}
    g.close()
    return out


@pytest.mark.parametrize("case", sorted(CASES))
def test_local_update_and_tangent_match_oracle(pkg, case):
    args = state(case)
    gid, quat, mat, F, Fp = args
    out = evaluate(pkg, args)
    o = solver.RVE(gid, quat, mat, 2e-5)
    o.Fp = Fp.reshape(-1, 3, 3).copy()
    tauc, _ = o.hardening()
    P, K, S, M, dg, iters, failed = o.constitutive(F.reshape(-1, 3, 3), tauc, np.zeros_like(o.S), 1.0)
    assert failed == 0
    assert relerr(out["P_EVAL"], P.reshape(-1, 9)) < 1e-11
    assert relerr(out["DGAM"], dg.reshape(-1, 12)) < 1e-9
    assert relerr(out["TANGENT"], K.reshape(-1, 81)) < 1e-10


@pytest.mark.parametrize("case", ["one block", "past a block", "linear flow", "soft bulk"])
def test_tangent_entries_resolve_the_largest_one_to_58_bits(pkg, case):
    """K is kept as integers on one scale per voxel, the largest entry at 2^58
    or more: half of the small entries (below 2^53 of those units, so exact as
    doubles) have their lowest set bit in the last of them or the one above, 2^-58
    or less of the power of two above the largest entry."""
    K = evaluate(pkg, state(case))["TANGENT"]
    top = np.frexp(np.abs(K).max(axis=1))[1][:, None]
    m, e = np.frexp(K)
    i = np.abs(m * 2.0 ** 53).astype(np.int64)
    small = (i > 0) & (np.abs(K) <= np.ldexp(1.0, top - 8))
    low = (e - 53 + np.log2(np.where(i > 0, i & -i, 1)) - top)[small]
    assert low.size > 50
    assert np.median(low) <= -58


@pytest.mark.parametrize("case", ["one block", "past a block", "real exponent"])
def test_mixed_evaluation_is_the_fp64_one_with_a_rounded_tangent(pkg, case):
    """FP32 rounding of the tangent: half a unit of the last place, 2^-24."""
    args = state(case)
    a, b = evaluate(pkg, args), evaluate(pkg, args, precision=1)
    for k in ("P_EVAL", "S_EVAL"):
        assert relerr(b[k], a[k]) < 1e-11
    assert relerr(b["DGAM"], a["DGAM"]) < 1e-9
    K = b["TANGENT"]
    assert np.array_equal(K, K.astype(np.float32).astype(np.float64))
    assert np.all(np.abs(K - a["TANGENT"]) <= 2.0 ** -24 * np.abs(a["TANGENT"]) + 1e-10 * np.abs(a["TANGENT"]).max())


@pytest.mark.parametrize("shape", [(1, 2, 2), (27, 36, 36), (27, 36, 48)])
def test_tangent_apply_forms_reach_one_increment(pkg, shape):
    """K in tiles of 256 voxels, the last one part full, on both sides of the
    line between the two FP64 forms of the apply (38912 voxels): conjugate
    gradients in FP64 and in mixed precision (staged and plain loads) reach the increment
    that BiCGStab reaches with its own product K : p, to the 1e-9 of the other
    comparisons of two converged increments."""
    n2, n1, n0 = shape
    wl = rvegen.WORKLOADS["cu16"]
    gid, _ = rvegen.voronoi_grain_map(0, 4, 3, shape=(n0, n1, n2))
    quat, mat = rvegen.random_quaternions(4, 5), rvegen.material("Cu")
    out = []
    for options in (dict(krylov=1), dict(), dict(precision=1), dict(precision=1, tma=0)):
        g = pkg.RVE(gid, quat, mat, wl.edge, **options)
        assert g.step(wl.dFbar(), rvegen.UNIAXIAL_X_MASK, np.zeros(9), wl.dt)["converged"]
        out.append([g.field(k).reshape(gid.size, -1) for k in ("P", "F", "RHO_GND")])
        g.close()
    for other in out[1:]:
        for a, b in zip(other, out[0]):
            assert np.abs(a - b).max() <= 1e-9 * np.abs(b).max()


@pytest.mark.parametrize("precision", [0, 1])
def test_tangent_of_a_step_is_the_oracles(pkg, precision):
    """TANGENT after rve_step: the kernel the conjugate gradients of either precision read
    from, at the increment's own state.  FP32 storage: half a unit of the last
    place, 2^-24; the rest as in the other comparisons with the oracle (1e-10 of the largest)."""
    wl = rvegen.Workload("cu8", 8, 5, "Cu", 0.004, 4, seed=31)
    gid, quat, mat = wl.inputs()
    g = pkg.RVE(gid, quat, mat, wl.edge, precision=precision)
    o = solver.RVE(gid, quat, mat, wl.edge)
    for _ in range(3):
        o.Fp, o.rho_ssd = g.field("FP").reshape(-1, 3, 3).copy(), g.field("RHO_SSD").reshape(-1, 12).copy()
        assert g.step(wl.dFbar(), rvegen.UNIAXIAL_X_MASK, np.zeros(9), wl.dt)["converged"]
    tauc, _ = o.hardening()
    K = o.constitutive(g.field("F").reshape(-1, 3, 3), tauc, np.zeros_like(o.S), wl.dt)[1].reshape(-1, 81)
    out = g.field("TANGENT").reshape(-1, 81)
    if precision:
        assert np.array_equal(out, out.astype(np.float32).astype(np.float64))
    assert np.all(np.abs(out - K) <= (2.0 ** -24 if precision else 0.0) * np.abs(K) + 1e-10 * np.abs(K).max())
    g.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shear", [1e-7, 1e-5, 1e-3])
def test_increments_of_a_lattice_soft_in_one_shear(pkg, precision, shear):
    """Increments of lattices with C11 - C12 = 1e-7, 1e-5 (FP64 Newton matrices) and
    1e-3 C11 (FP32 ones) converge to the Newton tolerance, in both precisions to the
    same mean stress (1e-9, as the other comparisons of two converged increments)."""
    wl = rvegen.Workload("cu8", 8, 5, "Cu", 0.002, 4, seed=31)
    gid, quat, _ = wl.inputs()
    mat = rvegen.material("Cu", C11=120e3 * (1 + shear), C12=120e3, C44=75e3, mu=45e3)
    P = []
    for p in {precision, 0}:
        g = pkg.RVE(gid, quat, mat, wl.edge, precision=p)
        for _ in range(2):
            info = g.step(wl.dFbar(), rvegen.UNIAXIAL_X_MASK, np.zeros(9), wl.dt)
            assert info["converged"] and info["newton_iters"] <= 12
        P.append(g.macro_stress()[0])
        g.close()
    assert relerr(P[0], P[-1]) < 1e-9


@pytest.mark.parametrize("shear", [1e-7, 1e-9])
def test_voxels_whose_fp32_direction_breaks_down_are_solved_in_fp64(pkg, shear):
    """A lattice with almost no stiffness in one shear (C11 - C12 = 1e-7 and 1e-9
    C11): the FP32 factorisation of the compliance plus the slip terms is no
    descent direction, the FP64 one with pivoting solves every voxel.  Both
    handles end at residuals of 10 local_tol mu = 4.5e-9 MPa or less, and an
    error of S is no larger than its residual, within a factor 3 in P:
    2.7e-8 MPa of 667."""
    gid, quat, _, F, Fp = state("past a block")
    args = gid, quat, rvegen.material("Cu", C11=120e3 * (1 + shear), C12=120e3, C44=75e3, mu=45e3), F, Fp
    a, b = evaluate(pkg, args), evaluate(pkg, args, precision=1)
    assert relerr(a["P_EVAL"], b["P_EVAL"]) < 5e-11
    assert relerr(a["S_EVAL"], b["S_EVAL"]) < 5e-11


def test_voxels_that_fail_are_tried_again_in_fp64(pkg):
    """C44 = 1e4 C11: strains of 5e-4 ask for trial shears of 1e6 MPa, and a few
    voxels fail from either Newton iteration (4 and 10 of 648 by themselves); those
    that the FP32 directions leave are solved by the FP64 ones, the others keep
    their result."""
    gid, quat, _, F, Fp = state("past a block")
    out = evaluate(pkg, (gid, quat, rvegen.material("Cu", C44=75e7, mu=45e3), F, Fp))
    assert all(np.isfinite(v).all() for v in out.values())


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("field", ["TANGENT", "P_EVAL", "DGAM"])
def test_fields_go_to_device_memory_of_any_alignment(pkg, precision, field):
    """Device destinations that start 8, 4 and 1 bytes past a 16-byte boundary get
    the bytes that a host destination gets."""
    import torch
    gid, quat, mat, F, Fp = state("past a block")
    g = pkg.RVE(gid, quat, mat, 2e-5, precision=precision)
    g.set_field("F", F.reshape(gid.shape + (9,)))
    g.set_field("FP", Fp.reshape(gid.shape + (9,)))
    assert g.eval_constitutive(1.0)[1] == 0
    which, nc = pkg.FIELDS[field]
    n = nc * gid.size * 8
    host = np.empty(n, dtype=np.uint8)
    assert pkg.rve_get_fields(g.h, which, host.ctypes.data, n, 0) == pkg.RVE_OK
    for shift in (0, 8, 4, 1):
        dst = torch.zeros(n + 16, dtype=torch.uint8, device="cuda")
        assert pkg.rve_get_fields(g.h, which, dst.data_ptr() + shift, n, 1) == pkg.RVE_OK
        assert np.array_equal(dst[shift:shift + n].cpu().numpy(), host)
        assert not dst[shift + n:].any() and not dst[:shift].any()
    g.close()
