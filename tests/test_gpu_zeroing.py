"""blco_mttkrp_all overwrites whatever its outputs held: zeroed by one launch where
they are small, by one each where they are not, through private copies in short
modes at large ranks."""

import numpy as np
import pytest
import torch

import oracle
from tests._util import FP32_TOL

pytestmark = pytest.mark.gpu

blco = pytest.importorskip("paper_2201_12523_gb300.blco")


def _tensor(dims, nnz):
    rng = np.random.default_rng(nnz + len(dims))
    c = np.stack([rng.integers(0, d, nnz) for d in dims], 1)
    vals = rng.standard_normal(nnz).astype(np.float32)
    t = blco.Tensor.build(torch.from_numpy(np.ascontiguousarray(c.astype(np.uint32).view(np.int32))).cuda(),
                          torch.from_numpy(vals).cuda(), dims)
    return t, c, vals, rng


@pytest.mark.parametrize("dims,R,skip", [
    ((300, 200, 100), 8, None), ((1, 5000, 7), 16, None), ((5000, 1, 1, 300), 32, 1), ((300, 5000, 40), 64, None),
    ((90, 80, 70, 6, 5, 4), 128, 0), ((90, 80, 70, 6, 5, 4, 3, 1), 16, 7), ((700, 900), 32, None)])
def test_outputs_are_overwritten(dims, R, skip):
    t, c, vals, rng = _tensor(dims, 4001)
    A = [rng.standard_normal((d, R)).astype(np.float32) for d in dims]
    outs = [None if n == skip else torch.full((d, R), float("nan"), device="cuda") for n, d in enumerate(dims)]
    blco.blco_mttkrp_all(t.handle, [torch.from_numpy(a).cuda() for a in A], blco.BLCO_F32, R, outs)
    for n in range(len(dims)):
        if n != skip:
            M, S = oracle.mttkrp(c, vals.astype(np.float64), dims, [a.astype(np.float64) for a in A], n)
            assert oracle.max_rel_err(outs[n].cpu().numpy(), M, S) <= FP32_TOL


@pytest.mark.parametrize("dims,R,launches", [
    ((5000, 4000, 900), 32, 1),              # 1.2 MB: one launch
    ((400_000, 200_000, 1000), 32, 3),       # 77 MB: one each
    ((300, 5000, 4000), 64, 3),              # short modes (16 copies in 48 MB: up to 12288 rows): their copies only
])
def test_zeroing_launches(dims, R, launches):
    t, *_ = _tensor(dims, 3000)
    A = [torch.rand(d, R, device="cuda") for d in dims]
    blco.blco_profile_enable(t.handle, True)
    t.mttkrp_all(A)
    blco.blco_profile_enable(t.handle, False)
    assert blco.blco_profile_read(t.handle)["zero"][0] == launches
