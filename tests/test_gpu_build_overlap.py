"""A build waits for its own stream only: the scratch of a construction is given
back without a device-wide synchronization, so another stream's kernel may still
be running when blco_build returns."""

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

blco = pytest.importorskip("paper_2201_12523_gb300.blco")

CYCLES = 1_500_000_000  # of a kernel that only counts cycles: 0.7 s at 2.07 GHz


@pytest.mark.parametrize("dims,nnz,line", [
    ((5000, 4000, 300), 300_000, 64),
    ((5000, 4000, 300), 5_000_000, 64),                # scratch of more than 32 MB
    ((5000, 4000, 300), 300_000, 20),                  # blocks: their keys are scratch
    ((5000, 4000, 300), 5_000_000, 20),
    ((1 << 30, 1 << 22, 1 << 21), 300_000, 64),        # 73 bits: two more key buffers, and blocks
])
def test_build_returns_while_another_stream_works(dims, nnz, line):
    rng = np.random.default_rng(nnz)
    c = np.stack([rng.integers(0, d, nnz) for d in dims], 1).astype(np.uint32).view(np.int32)
    coords, vals = torch.from_numpy(np.ascontiguousarray(c)).cuda(), torch.ones(nnz, device="cuda")
    blco.Tensor.build(coords, vals, dims, line_bits=line).destroy()  # kernels loaded
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(1000)
    torch.cuda.synchronize()
    done = torch.cuda.Event()
    with torch.cuda.stream(side):
        torch.cuda._sleep(CYCLES)
        done.record()
    t = blco.Tensor.build(coords, vals, dims, line_bits=line)
    running = not done.query()
    side.synchronize()
    keys = torch.empty(nnz, dtype=torch.int64, device="cuda")
    blco.blco_keys(t.handle, keys)
    t.destroy()
    assert running
