"""bench.py's names and traffic model of the A kernels (CPU)."""
import bench


def test_the_kernel_that_runs_is_the_one_named():
    assert bench.fwd_kernel_name(3, 2) == bench.fwd_kernel_name(3, 8) == "k_line_fwd"
    assert bench.fwd_kernel_name(3, 16) == bench.fwd_kernel_name(2, 64) == "k_fwd<w8,r2>"
    assert bench.fwd_kernel_name(1, 64) == "k_fwd<w8,r4>"
    assert bench.fwd_kernel_name(1, 8) == bench.fwd_kernel_name(0, 64) == bench.fwd_kernel_name(-1, 64) == "k_fwd"


def test_bytes_gathered_follow_the_table():
    n, M, nnz, nb = 512, 60 * 736, 28793597, 2
    N = n * n
    # the library's algorithmic bytes of a launch on either table (adm.cu, add_profile_bytes)
    csr = 8.0 * nnz + 8.0 * (M + 1) + 4.0 * nb * (N + M)
    lines = 4.0 * M * n + 4.0 * nb * (N + M)
    assert bench.gathered_by_a("k_fwd", csr, n, N, M, nnz) == (nb, 4.0 * nb * nnz)
    assert bench.gathered_by_a("k_line_fwd", lines, n, N, M, nnz) == (nb, 4.0 * nb * 2 * M * n)
