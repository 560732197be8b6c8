"""The FP64-class product (csrc/crt_gemm.cu) in blocks of fewer rows than columns, at its most K splits,
in blocks of K, and with rows down to the least numbers."""
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


def test_crt_rows_near_the_least_numbers(product):  # noqa: F811
    """Rows near 2^-1022 keep their relative accuracy, and rows of subnormal numbers are exact."""
    A, B = _normal(20, 100), _normal(30, 100, seed=2)
    C = product(A, B, torch.empty(20, 30, dtype=torch.float64, device="cuda"), 1, 1)
    for e in (-920, -1000):
        tiny = A * 2.0 ** -500 * 2.0 ** (e + 500)
        S = product(tiny, B * 2.0 ** 950, torch.empty_like(C), 1, 1)
        assert torch.equal(S, C * 2.0 ** (e + 950))
    whole = torch.round(A * 2.0 ** 45)
    C = product(whole, B, torch.empty_like(C), 1, 1)
    S = product(whole * 2.0 ** -600 * 2.0 ** -474, B * 2.0 ** 950, torch.empty_like(C), 1, 1)
    assert torch.equal(S, C * 2.0 ** -124)
