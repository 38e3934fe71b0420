"""The MTTKRP of stores that keep the order inside tiles of 1024 positions
(2^16 nonzeros and more), at the edges of its tiles, its rank and gather counts
and its row widths, against the FP64 oracle and against the kernel that orders
32 nonzeros at a time (which computes blco_mttkrp_range)."""

import numpy as np
import pytest
import torch

import oracle
from tests._util import FP32_TOL

pytestmark = pytest.mark.gpu

blco = pytest.importorskip("paper_2201_12523_gb300.blco")


def _coo(dims, nnz, seed, power=3):
    rng = np.random.default_rng(seed)
    c = np.stack([np.minimum((d * rng.random(nnz) ** power).astype(np.int64), d - 1) for d in dims], 1)
    c[0] = [d - 1 for d in dims]
    return rng, c


def _i32(c):
    return torch.from_numpy(np.ascontiguousarray(c.astype(np.uint32).view(np.int32))).cuda()


@pytest.mark.parametrize("dims,nnz,line,R,dtype", [
    ((300, 200, 100), 65_536, 64, 32, torch.float32),             # whole tiles, smallest size
    ((5000, 4000, 70), 65_537, 64, 16, torch.float32),            # one nonzero in the last tile
    ((5000, 4000, 7), 66_559, 64, 64, torch.float32),             # last tile one short; a mode of 7 rows
    ((40_000, 3), 70_001, 64, 32, torch.float32),                 # 2 modes: no row but the partner's
    ((900, 800, 70, 60), 70_003, 64, 32, torch.bfloat16),
    ((900, 800, 70, 60, 5), 70_004, 20, 16, torch.float16),       # blocks
    ((90, 80, 70, 6, 5, 4), 70_005, 64, 8, torch.float32),        # generic gather count
    ((90, 80, 70, 6, 5, 4, 3, 2), 70_006, 64, 128, torch.float32),
    (((1 << 23) + 5, 1 << 14, 900), 70_007, 40, 32, torch.float32),  # a row does not fit 22 bits; blocks
    ((1000, 1, 900), 70_008, 64, 32, torch.float32),              # a mode of one row
])
def test_tiled_mttkrp(dims, nnz, line, R, dtype):
    rng, c = _coo(dims, nnz, nnz + R)
    vals = rng.standard_normal(nnz).astype(np.float32)
    t = blco.Tensor.build(_i32(c), torch.from_numpy(vals).cuda(), dims, line_bits=line)
    A = [torch.from_numpy(rng.standard_normal((d, R)).astype(np.float32)).cuda().to(dtype) for d in dims]
    Af = [a.double().cpu().numpy() for a in A]
    for n in range(len(dims)):
        got = t.mttkrp(n, A)
        M, S = oracle.mttkrp(c, vals.astype(np.float64), dims, Af, n)
        assert oracle.max_rel_err(got.cpu().numpy(), M, S) <= FP32_TOL
        part = torch.empty_like(got)
        blco.blco_mttkrp_range(t.handle, n, 0, nnz, A, blco._DTYPE_CODE[dtype], R, part)
        assert oracle.max_rel_err(part.cpu().numpy(), M, S) <= FP32_TOL


def test_tiled_adjoint_takes_an_unaligned_gradient():
    dims, nnz, R = (700, 600, 50), 66_001, 32
    rng, c = _coo(dims, nnz, 5)
    t = blco.Tensor.build(_i32(c), torch.ones(nnz, device="cuda"), dims)
    A = [torch.from_numpy(rng.standard_normal((d, R)).astype(np.float32)).cuda() for d in dims]
    buf = torch.from_numpy(rng.standard_normal(nnz + 1).astype(np.float32)).cuda()
    g = buf[1:]  # starts 4 bytes past a 16-byte boundary
    assert g.data_ptr() % 16 == 4
    perm = t.perm()
    for n in range(3):
        M, S = oracle.mttkrp(c[perm], g.double().cpu().numpy(), dims, [a.double().cpu().numpy() for a in A], n)
        assert oracle.max_rel_err(t.cp_bwd(n, g, A).cpu().numpy(), M, S) <= FP32_TOL


@pytest.mark.parametrize("R", [8, 16, 32, 64])
@pytest.mark.parametrize("dims", [(500, 400, 30), (200, 90, 30, 7), (300, 4), (60, 50, 9, 8, 7)])
def test_tiled_mttkrp_f64(dims, R):
    nnz = 65_700
    rng, c = _coo(dims, nnz, R)
    vals = rng.standard_normal(nnz)
    t = blco.Tensor.build(_i32(c), torch.from_numpy(vals).cuda(), dims)
    A = [torch.from_numpy(rng.standard_normal((d, R))).cuda() for d in dims]
    Af = [a.cpu().numpy() for a in A]
    for n in range(len(dims)):
        M, S = oracle.mttkrp(c, vals, dims, Af, n)
        assert oracle.max_rel_err(t.mttkrp_f64(n, A).cpu().numpy(), M, S) <= 1e-12


def test_tiled_f64_nonfinite_rows_are_summed_term_by_term():
    """An infinite partner row times a fiber whose terms are zero, cancel or
    differ in sign gives what the sum of the terms gives (NaN or infinity), not
    what the product with the fiber's sum would give."""
    dims, nnz, R = (40, 500, 30), 65_600, 16
    rng, c = _coo(dims, nnz, 11, power=1)
    vals = rng.standard_normal(nnz)
    vals[:: 97] = 0.0
    A = [rng.standard_normal((d, R)) for d in dims]
    A[1][7] = np.inf
    A[1][8, ::2] = -np.inf
    A[1][9, 3] = np.nan
    A[2][4] = 0.0
    t = blco.Tensor.build(_i32(c), torch.from_numpy(vals).cuda(), dims)
    for n in (0, 2):
        got = t.mttkrp_f64(n, [torch.from_numpy(a).cuda() for a in A]).cpu().numpy()
        with np.errstate(invalid="ignore"):
            terms = vals[:, None].copy() * np.ones((1, R))
            for k in (2, 0):
                if k != n:
                    terms = terms * A[k][c[:, k]]
            terms = terms * A[1][c[:, 1]]
            ref = np.zeros((dims[n], R))
            np.add.at(ref, c[:, n], terms)
        assert np.array_equal(np.isnan(got), np.isnan(ref))
        assert np.array_equal(np.isposinf(got), np.isposinf(ref))
        assert np.array_equal(np.isneginf(got), np.isneginf(ref))


@pytest.mark.parametrize("dims,nnz,line,R,dtype,skip", [
    ((900, 800, 70, 60, 5), 65_536, 64, 16, torch.float32, None),
    ((900, 800, 70, 60, 5), 65_537, 20, 32, torch.float32, None),    # blocks; one nonzero in the last tile
    ((60, 70, 5000, 8, 9), 66_559, 64, 64, torch.float32, 2),       # the longest mode in the middle, not asked for
    ((90, 80, 70, 60, 1), 70_001, 64, 16, torch.bfloat16, None),    # a mode of one row
    ((1 << 24, 300, 20, 12, 10), 70_003, 40, 32, torch.float16, 1),  # the longest mode the kernel takes
])
def test_tiled_all_modes_in_one_pass(dims, nnz, line, R, dtype, skip):
    rng, c = _coo(dims, nnz, nnz + R)
    vals = rng.standard_normal(nnz).astype(np.float32)
    t = blco.Tensor.build(_i32(c), torch.from_numpy(vals).cuda(), dims, line_bits=line)
    A = [torch.from_numpy(rng.standard_normal((d, R)).astype(np.float32)).cuda().to(dtype) for d in dims]
    outs = [None if n == skip else torch.full((d, R), 3.0, device="cuda") for n, d in enumerate(dims)]
    blco.blco_mttkrp_all(t.handle, A, blco._DTYPE_CODE[dtype], R, outs)
    Af = [a.double().cpu().numpy() for a in A]
    for n in range(5):
        if n == skip:
            continue
        M, S = oracle.mttkrp(c, vals.astype(np.float64), dims, Af, n)
        assert oracle.max_rel_err(outs[n].cpu().numpy(), M, S) <= FP32_TOL
