"""The CP-ALS update's kernels (inverse, apply, scaling with the Gram) at the
edges of their tiles: ranks that are no multiple of 4, row counts around a tile
of rows and a stage of 32, A in place of M, pointers off a 16-byte boundary, no
Gram asked for, no rows. Reference: float64 numpy on the same float32 inputs.

Bounds, with u = 2^-24: a float32 sum of R products with a rounded inverse is
off by at most (R + 2) u sum_k |M_ik| |W_kr|; a column's norm by the norm of its
entries' bounds; the scaling adds two roundings. The Gram's reference is that
of the returned A, which its pairs of floats give to 1e-12 of sum |a b|."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

blco = pytest.importorskip("paper_2201_12523_gb300.blco")
U = 2.0 ** -24


def _run(I, R, mode, in_place, offset, gram, fn):
    rng = np.random.default_rng(I * 131 + R)
    dims = [I if k == mode else 200 + 3 * R for k in range(3)]
    facs = [rng.standard_normal((max(d, 1), R)) for d in dims]
    Gs = [torch.from_numpy(f.T @ f).cuda() for f in facs]
    buf = torch.zeros(2 * (I * R + 8), dtype=torch.float32, device="cuda")
    M = buf[offset:offset + I * R].view(I, R)
    M.copy_(torch.from_numpy(rng.standard_normal((I, R)).astype(np.float32)))
    Mh = M.cpu().numpy().astype(np.float64)
    A = M if in_place else buf[I * R + 8 + offset:2 * I * R + 8 + offset].view(I, R)
    lam = torch.full((R,), -1.0, dtype=torch.float64, device="cuda")
    G = torch.full((R, R), 7.0, dtype=torch.float64, device="cuda") if gram else None
    info = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    # (an empty view has no address: the buffer stands in for it)
    fn(Gs, 3, mode, R, M if I else buf, I, A if I else buf, lam, G, info)
    torch.cuda.synchronize()
    V = np.ones((R, R))
    for k in range(3):
        if k != mode:
            V *= Gs[k].cpu().numpy()
    W = np.linalg.inv(V)
    raw = Mh @ W
    off = (R + 2) * U * (np.abs(Mh) @ np.abs(W)) + 1e-11 * np.abs(raw).max(initial=0.0)
    norm = np.linalg.norm(raw, axis=0)
    return A.cpu().numpy().astype(np.float64), lam.cpu().numpy(), G, int(info.item()), raw, off, norm


@pytest.mark.parametrize("R", [1, 3, 4, 5, 10, 16, 31, 33, 50, 63, 64])
@pytest.mark.parametrize("I,in_place,offset,gram", [
    (1, False, 0, True), (31, True, 0, True), (65, False, 1, True), (1025, True, 3, True), (4099, False, 0, False),
    (70_001, False, 0, True)])
@pytest.mark.parametrize("fn", [blco.blco_cpals_update, blco.blco_cpals_update_noalloc])
def test_update_at_the_edges(R, I, in_place, offset, gram, fn):
    A, lam, G, info, raw, off, norm = _run(I, R, 1, in_place, offset, gram, fn)
    assert info == 0
    dl = np.linalg.norm(off, axis=0)
    assert np.all(np.abs(lam - norm) <= dl + 1e-12 * norm)
    safe = norm > 100 * dl  # a column of rounding errors only has no direction
    assert np.all((np.abs(A - raw / norm) <= (off + np.abs(raw) * dl / norm) / (norm - dl) + 4 * U * np.abs(A))[:, safe])
    if gram:
        err = np.abs(G.cpu().numpy() - A.T @ A)
        assert np.all(err <= 1e-12 * (np.abs(A).T @ np.abs(A)))


def test_update_without_rows():
    A, lam, G, info, *_ = _run(0, 8, 1, False, 0, True, blco.blco_cpals_update)
    assert info == 0 and np.all(lam == 0) and torch.all(G == 0)
