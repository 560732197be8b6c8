"""The FP64-class product (csrc/crt_gemm.cu) in blocks of fewer rows than columns, at its most K splits
and in blocks of K."""
import pytest

from test_gpu_crt import _check, _normal, product  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def up256(x):
    return (x + 255) // 256 * 256


# rows are halved first, to 384 of 520 and 256 of 330, below a number of columns that is no multiple of 16: the
# scratch lies between 384 x 520 (256 x 330) bytes per modulus, which do not hold the block, and its padded columns'
@pytest.mark.parametrize("m,n,mb,K", [(520, 520, 384, 64), (330, 330, 256, 72)])
def test_crt_blocks_of_fewer_rows_than_columns(product, m, n, mb, K):  # noqa: F811
    A, B = _normal(m, K), _normal(n, K, seed=2)
    need = sum(up256(16 * r * K * 2) + up256(4 * r) for r in (mb, n)) + up256(16 * n * mb)
    C = torch.empty(m, n, dtype=torch.float64, device="cuda")
    _check(product(A, B, C, 1, 1, scratch=need), A, B)


# operands of one sign just below a power of two: residues' sums over 19 splits of K near their largest
def test_crt_splits_of_one_sign(product):  # noqa: F811
    A, B = 1.0 - _normal(3, 20000).abs() * 2.0 ** -40, 1.0 - _normal(9, 20000, seed=2).abs() * 2.0 ** -45
    C = torch.empty(3, 9, dtype=torch.float64, device="cuda")
    _check(product(A, B, C, 1, 1), A, B)


# more than 2^17 terms: the operands' last bit, 2^-53 below the power of two above their row, decides the result
@pytest.mark.parametrize("K", [1 << 17, (1 << 17) + 2, 500000])
def test_crt_long_contractions_keep_53_bits(product, K):  # noqa: F811
    sign = torch.ones(K, dtype=torch.float64, device="cuda")
    sign[1::2] = -1.0
    A = (0.75 + 2.0 ** -53 * (sign > 0).double())[None].repeat(2, 1)
    assert A.dtype == torch.float64
    B = (0.75 * sign)[None].repeat(3, 1)
    C = product(A, B, torch.empty(2, 3, dtype=torch.float64, device="cuda"), 1, 1)
    assert bool((C == K // 2 * 0.75 * 2.0 ** -53).all())
