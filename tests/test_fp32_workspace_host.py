"""What an fp32 product asks of its workspace (no GPU needed: the queries look at sizes and strides only)."""
from paper_2608_13426_b200 import binding

PARTIALS = 2 * 148 * 65536      # room for the sums of cut tiles


def mat(rows, cols, batch=1):
    return binding.rmm_mat_t(256, binding.RMM_F32, batch, rows, cols, rows * cols if batch > 1 else 0, cols, 1)


def gemm(M, K, N, k, batch=1):
    return binding.lib().rmm_reduced_gemm_workspace_bytes(mat(M, K, batch), mat(K, N, batch), k, mat(M, N, batch))


def product(M, K, N):
    return binding.lib().rmm_product_workspace_bytes(mat(M, K), mat(K, N), mat(M, N))


def test_the_parts_are_bounded():
    most = 4096 + (512 << 20) + PARTIALS + (8 << 20)
    for M, K, N in [(32768, 28672, 8192), (8192, 28672, 32768), (100000, 4096, 300), (300, 200000, 300)]:
        for k in (K, K // 2, K // 16):
            assert 4096 <= gemm(M, K, N, k) <= most, (M, K, N, k)
        assert product(M, K, N) <= most
    assert gemm(2048, 4096, 2048, 2048, batch=64) <= most


def test_the_parts_follow_the_kept_count():
    M, K, N = 4096, 8192, 4096
    sizes = [gemm(M, K, N, k) for k in (512, 1024, 2048, 4096, 8192)]
    assert sizes == sorted(sizes)
    for k, size in zip((512, 1024, 2048, 4096, 8192), sizes):
        assert size <= 4096 + 6 * (M + N) * k + PARTIALS + (4 << 20)
    assert product(M, K, N) == sizes[-1]


def test_products_of_the_fma_kernel_do_not_ask_for_parts():
    # few rows: estimates prefer the FMA kernel, whose slices fit in far less than the parts of B
    assert gemm(64, 4096, 4096, 2048) < 6 * 4096 * 2048
    assert gemm(64, 28672, 8192, 14336) < 6 * 8192 * 14336


def test_a_kept_count_that_the_call_refuses_asks_for_no_parts():
    assert gemm(777, 3000, 1500, 10 ** 7) < 64 << 20
