"""The float64 sums of CP-ALS (the tensor's norm, the update's column norms, the
fit's inner products) over the whole range of float32 inputs, infinities among
them. Reference: the same sums in float64 on the host, whose terms are exact
(products of 24-bit numbers) or off by one rounding.

Bounds: n nonnegative terms added in any order in float64 are off by at most
n 2^-53 of their sum; a norm's square root halves that and adds a rounding."""

import math

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

blco = pytest.importorskip("paper_2201_12523_gb300.blco")

SCALES = [1e-25, 1e-22, 1e-20, 1e-18, 1e-9, 1.0, 1e9, 1e18, 1e30]
EPS = 2.0 ** -53


def _squares(x):
    return math.fsum((x.astype(np.float64) ** 2).tolist())


def _store(vals, dims=(40, 30, 20)):
    rng = np.random.default_rng(len(vals))
    c = np.stack([rng.integers(0, d, len(vals)) for d in dims], 1).astype(np.uint32).view(np.int32)
    return blco.Tensor.build(torch.from_numpy(np.ascontiguousarray(c)).cuda(), torch.from_numpy(vals).cuda(), dims)


def _norm2(vals):
    t = _store(vals)  # the handle lives as long as its Tensor
    out = torch.empty(1, dtype=torch.float64, device="cuda")
    blco.blco_norm2(t.handle, out)
    norm2 = float(out.item())
    t.destroy()
    return norm2


@pytest.mark.parametrize("scale", SCALES)
@pytest.mark.parametrize("n", [1, 777, 30_001])
def test_norm2(scale, n):
    v = (np.random.default_rng(n).standard_normal(n) * scale).astype(np.float32)
    ref = _squares(v)
    assert abs(_norm2(v) - ref) <= n * EPS * ref


def test_norm2_of_mixed_scales_zeros_and_infinities():
    v = np.zeros(5000, np.float32)
    assert _norm2(v) == 0.0
    v[::3], v[1::7], v[4999] = 1e-25, 3e-21, 1e-19
    ref = _squares(v)
    assert abs(_norm2(v) - ref) <= v.size * EPS * ref
    v[17] = 1e25
    ref = _squares(v)
    assert abs(_norm2(v) - ref) <= v.size * EPS * ref
    v[99] = -np.inf
    assert _norm2(v) == np.inf
    v[100] = np.nan
    assert math.isnan(_norm2(v))


def _update(Mh, fn):
    """The update with V the identity: M's columns and their norms."""
    I, R = Mh.shape
    eye = torch.eye(R, dtype=torch.float64, device="cuda")
    M = torch.from_numpy(Mh).cuda()
    A = torch.empty_like(M)
    lam = torch.empty(R, dtype=torch.float64, device="cuda")
    info = torch.empty(1, dtype=torch.int32, device="cuda")
    fn([eye, eye, eye], 3, 1, R, M, I, A, lam, None, info)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    return A.cpu().numpy(), lam.cpu().numpy()


def _check_columns(Mh, fn):
    A, lam = _update(Mh, fn)
    ref = np.sqrt([_squares(Mh[:, r]) for r in range(Mh.shape[1])])
    assert np.all(np.abs(lam - ref) <= (Mh.shape[0] + 2) * EPS * ref)
    unit = Mh / np.where(ref > 0, ref, 1.0)
    assert np.all(np.abs(A - unit) <= 2.0 ** -22 * np.abs(unit) + 2.0 ** -149)


@pytest.mark.parametrize("fn", [blco.blco_cpals_update, blco.blco_cpals_update_noalloc])
@pytest.mark.parametrize("scale", SCALES)
@pytest.mark.parametrize("I,R", [(1, 1), (500, 5), (4099, 64)])
def test_column_norms(I, R, scale, fn):
    _check_columns((np.random.default_rng(I + R).standard_normal((I, R)) * scale).astype(np.float32), fn)


@pytest.mark.parametrize("R", [7, 16])
def test_column_norms_of_columns_of_different_scales(R):
    rng = np.random.default_rng(R)
    Mh = rng.standard_normal((3001, R))
    Mh[:, 0] = 0.0
    for r, s in enumerate((1e-25, 1e-20, 1e18, 1e30)):
        Mh[:, r + 1] *= s
    Mh[5::9, 5] *= 1e-23  # tiny entries beside ordinary ones
    _check_columns(Mh.astype(np.float32), blco.blco_cpals_update)


def test_column_norm_with_an_infinity():
    Mh = np.ones((900, 1), np.float32)
    Mh[400] = np.inf
    A, lam = _update(Mh, blco.blco_cpals_update)
    assert lam[0] == np.inf and np.isnan(A[400, 0]) and np.all(A[:400] == 0)


@pytest.mark.parametrize("scale", SCALES)
@pytest.mark.parametrize("I,R", [(1, 3), (2039, 32), (70_001, 10)])
def test_fit(I, R, scale):
    """M and A both scaled, so that their products leave float32's range; model
    norm and ||X|| scaled alike, so that the fit does not depend on the scale."""
    rng = np.random.default_rng(I)
    M, A = [(rng.random((I, R)) * scale).astype(np.float32) for _ in range(2)]
    inner = math.fsum((M.astype(np.float64) * A.astype(np.float64)).ravel().tolist())
    lam = np.full(R, 0.5)
    G = [np.eye(R) * (2.0 * inner / R), np.eye(R), np.eye(R)]
    xh2, normX2 = 0.25 * R * (2.0 * inner / R), 3.0 * inner
    ref = 1.0 - math.sqrt(normX2 + xh2 - inner) / math.sqrt(normX2)
    fit = torch.empty(1, dtype=torch.float64, device="cuda")
    blco.blco_cpals_fit(normX2, [torch.from_numpy(g).cuda() for g in G], 3, R, torch.from_numpy(lam).cuda(),
                        torch.from_numpy(M).cuda(), torch.from_numpy(A).cuda(), I, fit)
    # the inner product is a third of what is under the root
    assert abs(float(fit.item()) - ref) <= (I * R + 16) * EPS


@pytest.mark.parametrize("exponent", [-80, 64])
def test_cp_als_does_not_depend_on_the_units_of_the_values(exponent):
    """Values times a power of two: the same factors and fits, lambda times it.
    The two runs differ by the order of float32 sums only; 100 times the
    rounding of a sum over the longest slice covers the update's condition."""
    rng = np.random.default_rng(3)
    dims, R, nnz = (60, 50, 40), 8, 20_000
    c = np.stack([rng.integers(0, d, nnz) for d in dims], 1).astype(np.uint32).view(np.int32)
    coords = torch.from_numpy(np.ascontiguousarray(c)).cuda()
    v = rng.random(nnz).astype(np.float32) + 0.5
    A0 = [torch.from_numpy(rng.random((d, R)).astype(np.float32)).cuda() for d in dims]
    got = []
    for s in (0, exponent):
        t = blco.Tensor.build(coords, torch.from_numpy(np.ldexp(v, s).astype(np.float32)).cuda(), dims)
        A, lam, fits = blco.cp_als(t, [a.clone() for a in A0], 2)
        got.append(([a.cpu().numpy() for a in A], np.ldexp(lam.cpu().numpy(), -s), fits))
    tol = 100 * 600 * 2.0 ** -24
    np.testing.assert_allclose(got[1][2], got[0][2], atol=tol)
    np.testing.assert_allclose(got[1][1], got[0][1], rtol=tol)
    for a, b in zip(got[0][0], got[1][0]):
        assert np.linalg.norm(a - b) <= tol * np.linalg.norm(a)


@pytest.mark.parametrize("scale", [1e-25, 1e-22, 1.0, 1e30])
def test_sums_over_mostly_empty_rows(scale):
    """Threads that see nothing but zeros (of either sign) beside threads that do not."""
    rng = np.random.default_rng(8)
    Mh = np.zeros((200_003, 10))
    rows = rng.choice(200_003, 900, replace=False)
    Mh[rows] = rng.standard_normal((900, 10)) * scale
    Mh[:, 3] = 0.0
    Mh[::5] *= -1.0
    _check_columns(Mh.astype(np.float32), blco.blco_cpals_update)
    v = Mh[:, 0].astype(np.float32)
    ref = _squares(v)
    assert abs(_norm2(v) - ref) <= v.size * EPS * ref
