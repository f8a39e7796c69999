"""rgf_zgemm_tc with leading dimensions whose product with an inner index passes
2^31: every entry is addressed in 64 bits (128 rows of B that lie 17 million
elements apart, about 35 GB of which only the rows are touched).  Against
torch's complex128 product; tolerance as documented, 2^-50 k max|A| max|B| per
real part."""
import pytest

pytestmark = pytest.mark.gpu


def product_error(rgflib, m, n, k, lda, ldb, ldc):
    import torch
    if torch.cuda.mem_get_info()[0] < 2 * 16 * max(m * lda, k * ldb, m * ldc):
        pytest.skip("not enough device memory")
    g = torch.Generator("cuda").manual_seed(m + n + k)

    def matrix(rows, cols, ld):
        flat = torch.empty((rows - 1) * ld + cols, dtype=torch.complex128, device="cuda")
        v = flat.as_strided((rows, cols), (ld, 1))
        v.copy_(torch.randn(rows, cols, dtype=torch.complex128, device="cuda", generator=g))
        return v

    A, B, C = matrix(m, k, lda), matrix(k, n, ldb), matrix(m, n, ldc)
    torch.cuda.synchronize()
    st = rgflib.lib.rgf_zgemm_tc(m, n, k, A.data_ptr(), lda, B.data_ptr(), ldb, C.data_ptr(), ldc, None)
    assert st == 0
    bound = 2.0 ** -50 * k * A.abs().max() * B.abs().max()
    d = torch.view_as_real(C - A.contiguous() @ B.contiguous()).abs().max()
    del A, B, C
    torch.cuda.empty_cache()
    return float(d / bound)


@pytest.mark.parametrize("m,n,k,lda,ldb,ldc", [(16, 8, 128, 128, 17_000_000, 8),
                                              (130, 5, 40, 17_000_000, 5, 9)])
def test_wide_leading_dimensions(rgflib, m, n, k, lda, ldb, ldc):
    assert product_error(rgflib, m, n, k, lda, ldb, ldc) < 1.0
