"""Construction at the sizes where its sort, byte tables and re-encoding change
path: odd and even numbers of 8-bit passes over the low and the high word,
index bits that fill a byte or run one over, edges of the 4096-item sort tile.
The store is an exact object: every array equals the oracle's."""

import numpy as np
import pytest
import torch

import oracle
from tests.test_gpu_parity import _store_equal

pytestmark = pytest.mark.gpu

blco = pytest.importorskip("paper_2201_12523_gb300.blco")


@pytest.mark.parametrize("dims,line", [
    ((2, 1, 3), 64),                          # 3 bits: one pass; a mode without bits
    ((1 << 8, 1 << 8), 64),                   # 16 bits: two passes, whole bytes
    ((257, 129, 5), 64),                      # 9 + 8 + 3 bits: three passes, a byte and one bit
    ((1 << 22, 1 << 21, 1 << 21), 64),        # 64 bits: the widest single word
    ((1 << 22, 1 << 21, 1 << 22), 64),        # 65 bits: one pass over the high word
    ((1 << 30, 1 << 22, 1 << 21), 64),        # 73 bits: two passes over the high word
    ((1 << 31, 1 << 30, 1 << 20), 64),        # 81 bits: three
    ((1 << 14, 1 << 9, 1 << 9), 20),          # 32 bits over a 20-bit line: block keys of a single word
])
@pytest.mark.parametrize("nnz", [1, 4095, 4096, 4097, 12_345])
def test_store_bit_exact_at_the_sorts_edges(dims, line, nnz):
    rng = np.random.default_rng(nnz + sum(dims) % 1000)
    # skewed towards low indices, so that keys repeat, with both ends present
    c = np.stack([np.minimum((d * rng.random(nnz) ** 4).astype(np.int64), d - 1) for d in dims], 1)
    c[0] = [d - 1 for d in dims]
    coords = torch.from_numpy(np.ascontiguousarray(c.astype(np.uint32).view(np.int32)))
    vals = torch.from_numpy(rng.random(nnz).astype(np.float32))
    t = blco.Tensor.build(coords.cuda(), vals.cuda(), dims, line_bits=line)
    _store_equal(t, coords, vals, dims, line, 1 << 27)
