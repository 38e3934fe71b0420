"""Host threads with handles and streams of their own call the library at once:
no call may fail because of the shared memory that another thread's call of the
same kernel asks for."""

import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

blco = pytest.importorskip("paper_2201_12523_gb300.blco")


def _run_together(jobs, calls):
    errors, start = [], threading.Barrier(len(jobs))

    def work(job):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                call = job()
                start.wait()
                for _ in range(calls):
                    call()
            stream.synchronize()
        except Exception as e:  # noqa: BLE001 - told to the main thread
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors[:2]


def _update(R):
    def job():
        G = [torch.eye(R, dtype=torch.float64, device="cuda") for _ in range(3)]
        M = torch.rand(300, R, device="cuda")
        A, lam = torch.empty_like(M), torch.empty(R, dtype=torch.float64, device="cuda")
        info = torch.empty(1, dtype=torch.int32, device="cuda")
        return lambda: blco.blco_cpals_update(G, 3, 0, R, M, 300, A, lam, None, info)
    return job


def test_updates_of_different_ranks():
    _run_together([_update(64), _update(8), _update(64), _update(16)], 1500)


def _wide_build(dims):
    rng = np.random.default_rng(len(dims))
    c = np.stack([rng.integers(0, d, 1000) for d in dims], 1).astype(np.uint32).view(np.int32)

    def job():
        coords, vals = torch.from_numpy(np.ascontiguousarray(c)).cuda(), torch.ones(1000, device="cuda")
        return lambda: blco.Tensor.build(coords, vals, dims).destroy()
    return job


def test_builds_of_different_index_widths():
    # 69 bits in 3 modes and 128 in 8: 72 and 128 KB of byte tables
    _run_together([_wide_build((1 << 23,) * 3), _wide_build((1 << 16,) * 8)], 50)
