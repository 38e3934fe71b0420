"""The kernels over the order inside tiles of 1024 positions at the edges of their
tiles, ranks, gather counts and row widths, on stores large enough to use them
(2^20 nonzeros; 2^19 at R = 8 and 128 and in float64), against the FP64 oracle and
against the kernel that orders 32 nonzeros at a time (blco_mttkrp_range).
Tolerances: float32 sums as everywhere else, float64 sums 1e-12."""

import numpy as np
import pytest
import torch

import oracle
from tests import test_gpu_tiled as tiled
from tests._util import FP32_TOL

pytestmark = pytest.mark.gpu

blco = pytest.importorskip("paper_2201_12523_gb300.blco")

M, H = 1 << 20, 1 << 19


@pytest.mark.parametrize("dims,nnz,line,R,dtype", [
    ((300, 200, 100), M, 64, 32, torch.float32),                       # whole tiles, smallest size
    ((5000, 4000, 70), M + 1, 64, 16, torch.float32),                  # one nonzero in the last tile
    ((5000, 4000, 7), M + 1023, 64, 64, torch.float32),                # last tile one short; a mode of 7 rows
    ((40_000, 3), M + 4465, 64, 32, torch.float32),                    # 2 modes: no row but the partner's
    ((900, 800, 70, 60), M + 4467, 64, 32, torch.bfloat16),
    ((900, 800, 70, 60, 5), M + 4468, 20, 16, torch.float16),          # blocks
    ((90, 80, 70, 6, 5, 4), M + 4469, 64, 8, torch.float32),           # generic gather count
    ((90, 80, 70, 6, 5, 4, 3, 2), H + 4470, 64, 128, torch.float32),
    ((500, 400, 30), H + 1, 64, 128, torch.bfloat16),
    ((500, 400, 30), H + 5, 64, 8, torch.float32),
    (((1 << 23) + 5, 1 << 14, 900), M + 4471, 40, 32, torch.float32),  # a row does not fit 22 bits; blocks
    ((1000, 1, 900), M + 4472, 64, 32, torch.float32),                 # a mode of one row
])
def test_mttkrp(dims, nnz, line, R, dtype):
    tiled.test_tiled_mttkrp(dims, nnz, line, R, dtype)


@pytest.mark.parametrize("R", [8, 16, 32, 64])
@pytest.mark.parametrize("dims,nnz", [((500, 400, 30), H), ((200, 90, 30, 7), H + 1), ((4000, 1, 3000), H + 1023),
                                      ((40_000, 30_000, 2000), M + 7)])  # modes with 0.85 run ends per nonzero and more
def test_mttkrp_f64(dims, nnz, R):
    rng, c = tiled._coo(dims, nnz, R)
    vals = rng.standard_normal(nnz)
    t = blco.Tensor.build(tiled._i32(c), torch.from_numpy(vals).cuda(), dims)
    A = [rng.standard_normal((d, R)) for d in dims]
    for n in range(len(dims)):
        M, S = oracle.mttkrp(c, vals, dims, A, n)
        got = t.mttkrp_f64(n, [torch.from_numpy(a).cuda() for a in A]).cpu().numpy()
        assert oracle.max_rel_err(got, M, S) <= 1e-12


def test_f64_nonfinite_rows_are_summed_term_by_term():
    dims, nnz, R = (40, 500, 30), H + 77, 16
    rng, c = tiled._coo(dims, nnz, 11, power=1)
    vals = rng.standard_normal(nnz)
    vals[:: 97] = 0.0
    A = [rng.standard_normal((d, R)) for d in dims]
    A[1][7] = np.inf
    A[1][8, ::2] = -np.inf
    A[1][9, 3] = np.nan
    A[2][4] = 0.0
    t = blco.Tensor.build(tiled._i32(c), torch.from_numpy(vals).cuda(), dims)
    for n in (0, 2):
        got = t.mttkrp_f64(n, [torch.from_numpy(a).cuda() for a in A]).cpu().numpy()
        with np.errstate(invalid="ignore"):
            terms = vals[:, None] * A[2 - n][c[:, 2 - n]] * A[1][c[:, 1]]
            ref = np.zeros((dims[n], R))
            np.add.at(ref, c[:, n], terms)
        assert np.array_equal(np.isnan(got), np.isnan(ref))
        assert np.array_equal(np.isposinf(got), np.isposinf(ref))
        assert np.array_equal(np.isneginf(got), np.isneginf(ref))


def test_adjoint_takes_an_unaligned_gradient():
    dims, nnz, R = (700, 600, 50), M + 465, 32
    rng, c = tiled._coo(dims, nnz, 5)
    t = blco.Tensor.build(tiled._i32(c), torch.ones(nnz, device="cuda"), dims)
    A = [torch.from_numpy(rng.standard_normal((d, R)).astype(np.float32)).cuda() for d in dims]
    g = torch.from_numpy(rng.standard_normal(nnz + 1).astype(np.float32)).cuda()[1:]
    assert g.data_ptr() % 16 == 4
    perm = t.perm()
    for n in range(3):
        ref, S = oracle.mttkrp(c[perm], g.double().cpu().numpy(), dims, [a.double().cpu().numpy() for a in A], n)
        assert oracle.max_rel_err(t.cp_bwd(n, g, A).cpu().numpy(), ref, S) <= FP32_TOL


@pytest.mark.parametrize("dims,nnz,line,R,dtype,skip", [
    ((900, 800, 70, 60, 5), M, 64, 16, torch.float32, None),
    ((900, 800, 70, 60, 5), M + 1, 20, 32, torch.float32, None),         # blocks; one nonzero in the last tile
    ((60, 70, 5000, 8, 9), M + 1023, 64, 64, torch.float32, 2),          # the longest mode in the middle, not asked for
    ((90, 80, 70, 60, 1), M + 4465, 64, 16, torch.bfloat16, None),       # a mode of one row
    ((1 << 24, 300, 20, 12, 10), M + 4467, 40, 32, torch.float16, 1),    # the longest mode the kernel takes
])
def test_all_modes_in_one_pass(dims, nnz, line, R, dtype, skip):
    tiled.test_tiled_all_modes_in_one_pass(dims, nnz, line, R, dtype, skip)
