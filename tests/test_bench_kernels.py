"""bench.py's names and traffic model of the A kernels (CPU)."""
import bench


def test_the_kernel_that_runs_is_the_one_named():
    assert bench.fwd_kernel_name(3, 2) == bench.fwd_kernel_name(3, 8) == "k_line_fwd"
    assert bench.fwd_kernel_name(3, 16) == bench.fwd_kernel_name(2, 64) == "k_fwd<w8,r2>"
    assert bench.fwd_kernel_name(1, 64) == "k_fwd<w8,r4>"
    assert bench.fwd_kernel_name(1, 8) == bench.fwd_kernel_name(0, 64) == bench.fwd_kernel_name(-1, 64) == "k_fwd"


def test_bytes_gathered_follow_the_width():
    n, M, nnz = 512, 60 * 736, 28793597
    N = n * n

    def bwd(nb):  # the library's algorithmic bytes of A^T (adm.cu, add_profile_bytes)
        return 8.0 * nnz + 8.0 * (N + 1) + 4.0 * nb * (M + 3 * N)

    assert bench.gathered_by_a("k_fwd<w8,r2>", bwd(64), n, N, M, nnz) == (64, 4.0 * 64 * nnz)
    assert bench.gathered_by_a("k_line_fwd", bwd(2), n, N, M, nnz) == (2, 4.0 * 2 * 2 * M * n)
    # half of the launches narrowed to 2 channels, where A has another table: 33 on average
    assert bench.gathered_by_a("k_fwd<w8,r2>", (bwd(64) + bwd(2)) / 2, n, N, M, nnz)[0] == 33
