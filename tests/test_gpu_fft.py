"""The hand-written transforms behind the two projections, at axis lengths that
exercise every radix (8, 6, 4, 3, 2), plans of one to five passes and
transforms wider than a warp, against numpy's FP64 FFT; and the edges of the
fixed-point arithmetic inside the FP64 transforms (scales, zeros, NaN)."""
import numpy as np
import pytest

import rvegen
from oracle import spectral as sp

pytestmark = pytest.mark.gpu

MASK = rvegen.UNIAXIAL_X_MASK
LENGTHS = (2, 4, 6, 12, 16, 18, 24, 32, 36, 54, 64, 96, 108, 128, 162, 192, 256, 324, 432, 486, 512)


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


def device_field(X):
    import torch
    return torch.from_numpy(np.ascontiguousarray(np.moveaxis(X.reshape(X.shape[:3] + (9,)), -1, 0).reshape(9, -1))).cuda()


def handle(pkg, shape):
    n2, n1, n0 = shape
    return pkg.RVE(np.zeros(shape, dtype=np.int32), np.array([[1.0, 0, 0, 0]]), rvegen.material("Cu"), 1e-5)


def noalloc(pkg, shape, Xd):
    import torch
    n2, n1, n0 = shape
    Y = torch.empty_like(Xd)
    assert pkg.rve_project_noalloc(n0, n1, n2, 1e-5, MASK, Xd.data_ptr(), Y.data_ptr(), 0) == pkg.RVE_OK
    torch.cuda.synchronize()
    return Y


@pytest.mark.parametrize("axis", [0, 1, 2])
def test_every_axis_length_matches_numpy(pkg, axis):
    """Tolerances: a transform's rounding errors stay within a few 2^-53 of its
    largest value, and the Fourier-space projection (noalloc) has norm one:
    1e-14.  The stencil-factored projection divides by the symbol of the
    derivative, as small as about pi / n near the Nyquist frequencies, so
    errors of 2^-52 grow by up to n: 4e-15 n."""
    lengths = LENGTHS + ((1, 3, 9, 27, 81, 243) if axis == 2 else ())
    for n in lengths:
        size = [4, 6, 3]
        size[axis] = n
        shape = (size[2], size[1], size[0])
        X = np.random.default_rng(100 * axis + n).standard_normal(shape + (3, 3))
        ref = device_field(sp.project(X, MASK, 1e-5 / size[0])).cpu()
        scale = float(ref.abs().max())
        Xd = device_field(X)
        r = handle(pkg, shape)
        Y = r.project(MASK, Xd).cpu()
        r.close()
        assert float((Y - ref).abs().max()) < 4e-15 * max(size) * scale, (axis, n, "handle")
        assert float((noalloc(pkg, shape, Xd).cpu() - ref).abs().max()) < 1e-14 * scale, (axis, n, "noalloc")


@pytest.mark.parametrize("shape", [(6, 12, 16), (9, 18, 64)])
def test_fixed_point_scales(pkg, shape):
    """Powers of two pass through the projection exactly; near the ends of the
    FP64 range (where the conversion takes its checked path) the result is the
    scaled one to round-off; a zero field gives zero."""
    import torch
    Xd = device_field(np.random.default_rng(7).standard_normal(shape + (3, 3)))
    r = handle(pkg, shape)
    for run in (lambda x: r.project(MASK, x).clone(), lambda x: noalloc(pkg, shape, x)):
        Y = run(Xd)
        for k in (-600, -40, 300, 900):
            assert torch.equal(run(Xd * 2.0 ** k), Y * 2.0 ** k), k
        big = run(Xd * 2.0 ** 1000) * 2.0 ** -1000
        assert float((big - Y).abs().max()) < 1e-13 * float(Y.abs().max())
        assert float(run(torch.zeros_like(Xd)).abs().max()) == 0.0
    r.close()


@pytest.mark.parametrize("n0", [4, 24, 48, 54, 64, 72, 108, 128])
def test_projection_of_fields_on_an_odd_eight_byte_boundary(pkg, n0):
    """The row strips load 16 bytes at a time where the caller's field allows
    it; one that starts 8 bytes off gives the same bits, and so does a run of
    many rows per warp (sums of the means are taken down in between)."""
    import torch
    shape = (36, 54, n0) if n0 < 8 else (3, 4, n0)
    Xd = device_field(np.random.default_rng(n0).standard_normal(shape + (3, 3)) + 5.0)
    shifted = torch.empty(Xd.numel() + 1, dtype=Xd.dtype, device=Xd.device)[1:].view_as(Xd)
    shifted.copy_(Xd)
    assert shifted.data_ptr() % 16 == 8
    r = handle(pkg, shape)
    out = torch.empty(Xd.numel() + 1, dtype=Xd.dtype, device=Xd.device)[1:].view_as(Xd)
    Y = r.project(MASK, Xd)
    assert torch.equal(r.project(MASK, shifted, out), Y)
    assert float((Y[8].mean() - Xd[8].mean()).abs()) < 1e-14 * float(Xd.abs().max())
    r.close()


def test_columns_of_very_different_size_keep_their_digits(pkg):
    """A field whose rows differ by 2^-30 along y and z: the small tensor row's
    projection is as accurate as when it stands alone (each transform has its
    own scale)."""
    import torch
    shape = (8, 12, 32)
    X = np.random.default_rng(11).standard_normal(shape + (3, 3))
    X[..., 1, :] *= 2.0 ** -30
    X[..., 2, :] *= 2.0 ** 30
    ref = device_field(sp.project(X, MASK, 1e-5 / 32)).cpu()
    Xd = device_field(X)
    r = handle(pkg, shape)
    for Y in (r.project(MASK, Xd).cpu(), noalloc(pkg, shape, Xd).cpu()):
        for i in range(3):
            rows = slice(3 * i, 3 * i + 3)
            assert float((Y[rows] - ref[rows]).abs().max()) < 2e-13 * float(ref[rows].abs().max())
    r.close()


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
def test_non_finite_values_reach_every_value_of_their_rows(pkg, bad):
    import torch
    shape = (6, 12, 16)
    Xd = device_field(np.random.default_rng(13).standard_normal(shape + (3, 3)))
    Xd[4, 77] = bad                                     # component 11: tensor row 1
    r = handle(pkg, shape)
    for Y in (r.project(MASK, Xd), noalloc(pkg, shape, Xd)):
        # (the mean and the constant modes of the other rows do not see it)
        assert not torch.isfinite(Y[3:6]).any()
        assert torch.isfinite(Y[:3]).all() and torch.isfinite(Y[6:]).all()
    r.close()


@pytest.mark.parametrize("shape", [(3, 54, 48), (1, 8, 512), (3, 12, 486)])
def test_rows_that_share_a_block_with_another_tensor_row(pkg, shape):
    """Transforms along x whose threads are no power of two up to 32 (6, 64 and
    81 of them): the last rows of one tensor row lie in a block with the first of the
    next, 2^60 as large or with a NaN in it, and keep their digits (4e-15 n, as
    above) all the same."""
    import torch
    X = np.random.default_rng(17).standard_normal(shape + (3, 3))
    X[..., 1, :] *= 2.0 ** -30
    X[..., 2, :] *= 2.0 ** 30
    ref = device_field(sp.project(X, MASK, 1e-5 / shape[2])).cpu()
    Xd = device_field(X)
    Xn = Xd.clone()
    Xn[4, 5] = float("nan")
    r = handle(pkg, shape)
    for run in (lambda x: r.project(MASK, x).clone(), lambda x: noalloc(pkg, shape, x)):
        Y = run(Xd)
        for i in range(3):
            rows = slice(3 * i, 3 * i + 3)
            assert float((Y.cpu()[rows] - ref[rows]).abs().max()) < 4e-15 * max(shape) * float(ref[rows].abs().max()), i
        Z = run(Xn)
        assert not torch.isfinite(Z[3:6]).any()
        assert torch.equal(Z[:3], Y[:3]) and torch.equal(Z[6:], Y[6:])
    r.close()


@pytest.mark.parametrize("shape", [(1, 16, 16), (3, 2, 432), (2, 512, 2), (6, 128, 8), (3, 32, 64), (4, 48, 48), (3, 54, 36),
                                   (3, 54, 48), (2, 64, 64)])
def test_planes_in_one_block_and_above_the_line(pkg, shape):
    """The X and Y passes fused per plane, up to the largest planes that take
    them, and the separate passes just above: as accurate as the axis-length
    test asks (4e-15 n), powers of two exact, zeros stay zero, a NaN stays
    in its tensor row."""
    import torch
    X = np.random.default_rng(sum(shape)).standard_normal(shape + (3, 3))
    ref = device_field(sp.project(X, MASK, 1e-5 / shape[2])).cpu()
    Xd = device_field(X)
    r = handle(pkg, shape)
    Y = r.project(MASK, Xd).clone()
    assert float((Y.cpu() - ref).abs().max()) < 4e-15 * max(shape) * float(ref.abs().max())
    assert torch.equal(r.project(MASK, Xd * 2.0 ** -40), Y * 2.0 ** -40)
    assert float(r.project(MASK, torch.zeros_like(Xd)).abs().max()) == 0.0
    Xd[4, 5] = float("nan")
    Z = r.project(MASK, Xd)
    assert not torch.isfinite(Z[3:6]).any()
    assert torch.equal(Z[:3], Y[:3]) and torch.equal(Z[6:], Y[6:])
    r.close()


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("shape", [(6, 12, 16), (27, 8, 64), (1, 6, 12)])
def test_curl_components_see_only_the_fields_they_depend_on(pkg, scheme, shape):
    """G_ij = -eps_jkl D_k Fp_il: component i0 does not depend on Fp_i0, which
    may be 2^60 as large as the others or hold a NaN without a bit of G_i0
    changing (each field's inverse transform has its own scale)."""
    rng = np.random.default_rng(sum(shape))
    Fp = np.eye(3) + 1e-3 * rng.standard_normal(shape + (3, 3))
    r = handle(pkg, shape)

    def nye(F):
        r.set_field("FP", F.reshape(shape + (9,)))
        assert pkg.load_library().rve_eval_nye(r.h, scheme) == pkg.RVE_OK
        return r.field("NYE").reshape(-1, 3, 3)

    G = nye(Fp)
    for bad in (2.0 ** 60, np.nan):
        for l in range(3):
            F = Fp.copy()
            F[..., 1, l] *= bad if bad == bad else 1.0
            if bad != bad:
                F[0, 1, 2, 1, l] = bad
            H = nye(F)
            assert np.array_equal(H[:, 1, l], G[:, 1, l]), (bad, l)
            assert np.array_equal(H[:, [0, 2]], G[:, [0, 2]])
            for j in (j for j in range(3) if j != l and shape != (1, 6, 12)):
                assert not np.array_equal(H[:, 1, j], G[:, 1, j])
    r.close()


@pytest.mark.parametrize("options", [dict(), dict(stencils=1)])
@pytest.mark.parametrize("shape", [(6, 12, 16), (9, 18, 64), (3, 8, 144)])
def test_small_fields_keep_their_digits(pkg, shape, options):
    """The projections and the curl are linear down to the bottom of the FP64
    range: fields of 2^-800 and 2^-920 give the scaled result (1e-13, the
    tolerance at the top of the range)."""
    import torch
    X = np.random.default_rng(7).standard_normal(shape + (3, 3))
    Xd = device_field(X)
    r = pkg.RVE(np.zeros(shape, dtype=np.int32), np.array([[1.0, 0, 0, 0]]), rvegen.material("Cu"), 1e-5, **options)

    def nye(x):
        r.set_field("FP", x.reshape(9, -1).T.reshape(shape + (9,)).cpu().numpy())
        r.eval_nye()
        return torch.from_numpy(np.ascontiguousarray(r.field("NYE"))).cuda()

    for run in (lambda x: r.project(MASK, x).clone(), lambda x: noalloc(pkg, shape, x), nye):
        Y = run(Xd)
        for k in (-800, -920):
            Z = run(Xd * 2.0 ** k) * 2.0 ** -k
            assert float((Z - Y).abs().max()) < 1e-13 * float(Y.abs().max()), k
    r.close()
