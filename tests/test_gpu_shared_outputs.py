"""blco_mttkrp_all with requested outputs in the same memory: the modes run one
after another, each overwriting its output, so the later mode's result stands
where two share memory."""

import numpy as np
import pytest
import torch

import oracle
from tests._util import FP32_TOL

pytestmark = pytest.mark.gpu

blco = pytest.importorskip("paper_2201_12523_gb300.blco")


@pytest.mark.parametrize("dims", [(300, 300, 50), (300, 200, 50), (200, 300, 50), (90, 300, 120, 300)])
@pytest.mark.parametrize("R", [16, 64])
def test_the_later_mode_stands_where_outputs_share_memory(dims, R):
    rng = np.random.default_rng(R)
    nnz = 20_003
    c = np.stack([rng.integers(0, d, nnz) for d in dims], 1)
    vals = rng.standard_normal(nnz).astype(np.float32)
    coords = torch.from_numpy(np.ascontiguousarray(c.astype(np.uint32).view(np.int32))).cuda()
    t = blco.Tensor.build(coords, torch.from_numpy(vals).cuda(), dims)
    A = [rng.standard_normal((d, R)).astype(np.float32) for d in dims]
    scratch = torch.full((max(dims), R), 7.0, device="cuda")
    own = torch.empty((dims[2], R), device="cuda")
    outs = [scratch[:dims[0]], scratch[:dims[1]], own] + [scratch[:d] for d in dims[3:]]
    blco.blco_mttkrp_all(t.handle, [torch.from_numpy(a).cuda() for a in A], blco.BLCO_F32, R, outs)
    got = scratch.cpu().numpy()
    ref = [oracle.mttkrp(c, vals.astype(np.float64), dims, [a.astype(np.float64) for a in A], n)
           for n in range(len(dims))]
    want, scale = np.full(got.shape, 7.0), np.ones(got.shape)
    for n in [0, 1] + list(range(3, len(dims))):
        want[:dims[n]], scale[:dims[n]] = ref[n]
    assert oracle.max_rel_err(got, want, scale) <= FP32_TOL
    assert oracle.max_rel_err(own.cpu().numpy(), *ref[2]) <= FP32_TOL
