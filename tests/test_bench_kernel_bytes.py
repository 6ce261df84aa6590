"""bench.py's bytes per launch against the arrays that the step's kernels read and write."""
import pytest

import bench


@pytest.mark.parametrize("nq,ng", [(512, 1536), (256, 768), (200, 400)])
def test_kernel_bytes_count_the_arrays_in_use(nq, ng):
    Np, Mc = float(nq**3), ng * ng * (ng // 2 + 1) * 8.0
    pos, key, rank, record, slots, offset = 12, 4, 4, 16, 48, 4
    # count: positions read, key and rank written; scatter: positions, key, rank and the
    # bin's offset read, record and sorted position written; the counts cleared,
    # added to, scanned and read
    assert bench.kernel_bytes("bins", nq, ng) == (
        (pos + key + rank + pos + key + rank + offset + record + rank) * Np + 4 * 4 * ng**2)
    assert bench.kernel_bytes("dep_r2c", nq, ng) == record * Np + Mc
    assert bench.kernel_bytes("c2r_gather", nq, ng) == 3 * Mc + (record + slots) * Np
    for same in ("deposit", "fft_z_r2c_fix", "fft_y_fwd", "fft_x_green", "fft_y_inv", "fft_z_c2r",
                 "gather_kick_drift", "kick_drift", "not_a_kernel"):
        assert bench.kernel_bytes(same, nq, ng) == bench.algorithmic_bytes(same, nq, ng)
