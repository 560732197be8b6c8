"""The t1-dressed ladder of an FP64 plan under a change of scale of the virtual
orbitals: B_ac -> s_a s_c B_ac, Bov_kc -> s_c Bov_kc, t_k^a -> s_a t_k^a, tau^cd ->
tau^cd / (s_c s_d) gives s_a s_b R^ab, bit for bit where s are powers of two."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("o,v,n", [(1, 5, 3), (3, 29, 37), (6, 50, 20)])
def test_orbital_scales_are_exact(o, v, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_08142_gb300 as lad
    rng = np.random.default_rng(v)
    B, Bov = rng.standard_normal((n, v, v)), rng.standard_normal((n, o, v))
    t1, tau = 0.1 * rng.standard_normal((o, v)), rng.standard_normal((o, o, v, v))
    tau = 0.5 * (tau + tau.transpose(1, 0, 3, 2))
    s = 2.0 ** rng.integers(-40, 41, v)
    L = lad.Ladder(o, v, n, mode="fp64", dressed=True)

    def apply(*x):
        return L.apply_dressed(*[torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in x]).cpu().numpy()
    R0 = apply(B, Bov, t1, tau)
    R1 = apply(B * s[:, None] * s, Bov * s, t1 * s, tau / (s[:, None] * s))
    L.close()
    assert np.array_equal(R1, R0 * s[:, None] * s)
    # zero amplitudes at some (c, d), and all zero
    tau[:, :, ::2, 1] = tau[:, :, 1, ::2] = 0.0
    L = lad.Ladder(o, v, n, mode="fp64", dressed=True)
    R0 = apply(B, Bov, t1, tau)
    Bd = B - np.einsum("kb,Pkd->Pbd", t1, Bov)
    ref = np.einsum("Pac,Pbd,ijcd->ijab", Bd, Bd, tau, optimize=True)
    X = np.einsum("Pkc,Pld,ijcd->ijkl", Bov, Bov, tau, optimize=True)
    ref -= np.einsum("ka,lb,ijkl->ijab", t1, t1, X, optimize=True)
    assert np.abs(R0 - ref).max() <= 1e-12 * np.abs(ref).max()
    assert not apply(B, Bov, t1, np.zeros_like(tau)).any()
    L.close()
