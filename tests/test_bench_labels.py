"""What bench.py's line says ran and what bound it (CPU only)."""

import bench


def _info(nnz, order, streamed=0, ordered=True):
    held = 16 * nnz + (order * (-(-nnz // 1024)) * 2176 if ordered else 0)
    return {"nnz": nnz, "order": order, "streamed": streamed, "device_bytes": held}


def test_the_kernel_named_is_the_one_that_the_store_runs():
    big, small = 500_000_000, 600_000
    assert bench.mttkrp_kernel(_info(big, 4), 32, False) == "k_mttkrp_tiled<float,32,3>"
    assert bench.mttkrp_kernel(_info(big, 4, ordered=False), 32, False) == "k_mttkrp<float,32,3>"
    assert bench.mttkrp_kernel(_info(big, 5), 16, True) == "k_mttkrp_fused_tiled<float,16,5>"
    assert bench.mttkrp_kernel(_info(big, 5, streamed=1), 16, True) == "k_mttkrp_fused<float,16,5>"
    assert bench.mttkrp_kernel(_info(small, 3), 64, False) == "k_mttkrp<float,64,2>"
    assert bench.mttkrp_kernel(_info(small, 3), 128, False) == "k_mttkrp_tiled<float,128,2>"


def test_a_streamed_step_is_bound_by_its_uploads_where_they_fill_it():
    assert bench.streamed_bound(125.2, 125.2, 70.2, 56.7).startswith("uploads: under way for 125 of the step's 125 ms")
    assert bench.streamed_bound(86.0, 60.0, 85.8, 56.7).startswith("kernels")
