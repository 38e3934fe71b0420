"""Which stores keep the order inside tiles of 1024 positions: those whose calls
are faster with it. A store built with a device budget never keeps it, so the
difference of the two stores' device memory is the order's."""

import numpy as np
import pytest
import torch

import oracle
from tests._util import FP32_TOL
from tests.test_gpu_tiled import _coo, _i32

pytestmark = pytest.mark.gpu

blco = pytest.importorskip("paper_2201_12523_gb300.blco")


def _order_bytes(dims, nnz, dtype):
    rng = np.random.default_rng(nnz)
    c = np.stack([rng.integers(0, d, nnz) for d in dims], 1).astype(np.uint32).view(np.int32)
    coords, vals = torch.from_numpy(np.ascontiguousarray(c)).cuda(), torch.ones(nnz, dtype=dtype, device="cuda")
    plain = blco.Tensor.build(coords, vals, dims)
    bare = blco.Tensor.build(coords, vals, dims, device_budget_bytes=1 << 33)
    n = blco.blco_info(plain.handle).device_bytes - blco.blco_info(bare.handle).device_bytes
    plain.destroy()
    bare.destroy()
    return n


# per mode and tile: a 2-byte word per position, a bit per position, and in
# float64 stores a second one
def _expected(order, nnz, f64):
    return order * -(-nnz // 1024) * (2048 + 128 * (2 if f64 else 1))


@pytest.mark.parametrize("order,kept", [(1, False), (2, False), (3, True), (4, True), (5, False), (6, False), (8, False)])
def test_float64_stores_keep_the_order_for_3_and_4_modes(order, kept):
    nnz = 600_001
    got = _order_bytes((3000, 700, 300, 90, 40, 9, 5, 3)[:order], nnz, torch.float64)
    assert got == (_expected(order, nnz, True) if kept else 0)


@pytest.mark.parametrize("dtype,dims,least", [
    (torch.float32, (700, 90), 1 << 19), (torch.float32, (700, 300, 90, 40, 9), 1 << 19),
    (torch.float64, (700, 300, 90), 3 << 16)])
def test_small_stores_keep_no_order(dtype, dims, least):
    for nnz in (66_000, least - 1):
        assert _order_bytes(dims, nnz, dtype) == 0
    for nnz in (least, least + 1):
        assert _order_bytes(dims, nnz, dtype) == _expected(len(dims), nnz, dtype == torch.float64)


def test_small_float64_stores_need_longer_runs():
    """1024 neighbours fall on about 3100 rows of 300k nonzeros (0.85 run ends per
    nonzero) and 2048 rows of 2^20 (0.79): more than 0.7, less than 0.98."""
    dims = (20_000, 15_000, 10_000)
    assert _order_bytes(dims, 300_000, torch.float64) == 0
    assert _order_bytes(dims, 1 << 20, torch.float64) == _expected(3, 1 << 20, True)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_modes_whose_rows_hardly_repeat_keep_no_order(dtype):
    """Of 2^20 uniform nonzeros, 1024 neighbours in the store have about 2^16 rows
    of the long modes to fall on (0.99 of them end a run), and 300 of the short."""
    nnz = 1 << 20
    assert _order_bytes((1 << 22, 1 << 21, 300), nnz, dtype) == _expected(1, nnz, dtype == torch.float64)
    assert _order_bytes((1 << 22, 1 << 21, 1 << 20), nnz, dtype) == 0


def test_a_store_with_the_order_of_one_mode_serves_all():
    dims, nnz, R = (1 << 22, 1 << 21, 300), (1 << 20) + 5, 16
    rng, c = _coo(dims, nnz, 9, power=1)
    vals = rng.standard_normal(nnz).astype(np.float32)
    t = blco.Tensor.build(_i32(c), torch.from_numpy(vals).cuda(), dims)
    A = [rng.standard_normal((d, R)).astype(np.float32) for d in dims]
    dA = [torch.from_numpy(a).cuda() for a in A]
    every = t.mttkrp_all(dA)
    for n in range(3):
        M, S = oracle.mttkrp(c, vals.astype(np.float64), dims, [a.astype(np.float64) for a in A], n)
        assert oracle.max_rel_err(t.mttkrp(n, dA).cpu().numpy(), M, S) <= FP32_TOL
        assert oracle.max_rel_err(every[n].cpu().numpy(), M, S) <= FP32_TOL


def test_one_pass_over_5_modes_without_every_modes_order():
    dims, nnz, R = (1 << 22, 1 << 20, 40, 30, 20), (1 << 20) + 5, 16
    rng, c = _coo(dims, nnz, 10, power=1)
    vals = rng.standard_normal(nnz).astype(np.float32)
    t = blco.Tensor.build(_i32(c), torch.from_numpy(vals).cuda(), dims)
    A = [rng.standard_normal((d, R)).astype(np.float32) for d in dims]
    every = t.mttkrp_all([torch.from_numpy(a).cuda() for a in A])
    for n in range(5):
        M, S = oracle.mttkrp(c, vals.astype(np.float64), dims, [a.astype(np.float64) for a in A], n)
        assert oracle.max_rel_err(every[n].cpu().numpy(), M, S) <= FP32_TOL
