"""The sixth slice of V+- in the error-free mode (csrc/ladder_oz.cu) is cut to
the nearest multiple of its last place.

One auxiliary function, one occupied orbital and one amplitude, tau^00 = 1, make
R^ab = B_a0 B_b0, an integer of 48 bits, and everything but the slices of V+-
exact: 2 R^ab is one slot of a row whose largest, 2 B_a1 B_b1 = 2^53, puts the
last place of slice 6 at 2^(54 - 8 - 40) = 64.  So R^ab may be off by half of
that, halved: 16."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("sym", [0, 1])
def test_last_slice_is_rounded_to_nearest(sym):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_08142_gb300 as lad
    v = 64
    L = lad.Ladder(1, v, 1, mode="ozaki", tuning={"oz_slices": 6, "sym_b": sym})
    tau = torch.zeros(1, 1, v, v, dtype=torch.float64, device="cuda")
    tau[0, 0, 0, 0] = 1.0
    for seed in range(4):
        b = (np.random.default_rng(seed).integers(1 << 23, 1 << 24, v) | 1).astype(np.float64)
        B = np.zeros((1, v, v))
        B[0, :, 0], B[0, :, 1] = b, 2.0 ** 26
        if sym:
            B[0, 0, :], B[0, 1, :] = B[0, :, 0], B[0, :, 1]
        R = L.apply(torch.from_numpy(B).cuda(), tau)
        L.check_device()
        off = np.abs(R[0, 0].cpu().numpy() - np.outer(b, b))[2:, 2:]
        assert off.max() <= 16.0
    L.close()
