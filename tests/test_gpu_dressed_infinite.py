"""The t1-dressed ladder of an FP64 plan keeps the infinities of FP64 arithmetic:
with an infinite amplitude, positive integrals and one occupied orbital, R^ab is
+inf - t^a t^b inf, +inf where t^a t^b < 0 and NaN where it is positive."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("v,n", [(3, 2), (41, 70)])
def test_infinite_amplitude(v, n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_08142_gb300 as lad
    rng = np.random.default_rng(v)
    B, Bov = rng.uniform(0.5, 1.0, (n, v, v)), rng.uniform(0.5, 1.0, (n, 1, v))
    t1 = rng.uniform(0.05, 0.1, (1, v)) * rng.choice([-1.0, 1.0], (1, v))
    t1[0, 0], t1[0, 1] = -0.1, 0.1
    tau = rng.uniform(0.5, 1.0, (1, 1, v, v))
    tau = 0.5 * (tau + tau.transpose(0, 1, 3, 2))
    tau[0, 0, 1, 1] = np.inf
    L = lad.Ladder(1, v, n, mode="fp64", dressed=True)
    R = L.apply_dressed(*[torch.from_numpy(x).cuda() for x in (B, Bov, t1, tau)])[0, 0].cpu().numpy()
    L.close()
    negative = np.outer(t1[0], t1[0]) < 0.0
    assert (R[negative] == np.inf).all() and np.isnan(R[~negative]).all()
