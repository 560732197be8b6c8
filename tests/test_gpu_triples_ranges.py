"""FP64 E(T) keeps its relative accuracy where orbitals differ by powers of ten.

The factors and amplitudes carry a scale per orbital.  With one dominant occupied
orbital its own triple vanishes (W and V are symmetric then), so E(T) comes from
terms that lie the scale of the next orbital below those of that triple, which
have to cancel, and the residues of W have to keep the bits of small operands.  The
reference evaluates E(T) in numpy's extended type (64 bits of
mantissa or more).

Tolerance: W rounded once, about 20 FP64 operations per term and sums of terms of
one sign: 1e-13 leaves room for the terms' own cancellations."""
import itertools

import numpy as np
import pytest

from gpu_util import to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
LD = np.longdouble
PERMS = list(itertools.permutations(range(3)))


def reference(B, Bov, Boo, t1, t2, e_occ, e_vir):
    b, bo, boo, s, t = (x.astype(LD) for x in (B, Bov, Boo, t1, t2))
    f = np.einsum("Pbd,Pia->ibda", b, bo)
    f = np.einsum("ibda,kjcd->ijkabc", f, t) - np.einsum("klcj,ilab->ijkabc", np.einsum("Pkc,Pjl->klcj", bo, boo), t)
    W = sum(np.transpose(f, np.argsort(p + tuple(3 + x for x in p))) for p in PERMS)
    I = np.einsum("Pjb,Pkc->jkbc", bo, bo)
    V = W + np.einsum("jkbc,ia->ijkabc", I, s) + np.einsum("ikac,jb->ijkabc", I, s) + np.einsum("ijab,kc->ijkabc", I, s)
    e, v = e_occ.astype(LD), e_vir.astype(LD)
    D = (e[:, None, None] + e[:, None] + e)[..., None, None, None] - (v[:, None, None] + v[:, None] + v)
    Z = 4 * W + np.transpose(W, (0, 1, 2, 5, 3, 4)) + np.transpose(W, (0, 1, 2, 4, 5, 3))
    return float((Z * (V - np.transpose(V, (0, 1, 2, 5, 4, 3))) / (3 * D)).sum())


@pytest.mark.parametrize("bits", [0, 3, 5, 10, 20, 30])
@pytest.mark.parametrize("flat_t2", [False, True])
@pytest.mark.parametrize("singles", [0.0, 0.01])
def test_wide_orbital_ranges(bits, flat_t2, singles):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_08142_gb300 as lad
    o, v, n = 3, 9, 20
    for seed in range(3):
        rng = np.random.default_rng(seed)
        so, sv = 2.0 ** -np.array([0, bits, bits + 1]), 2.0 ** -rng.integers(0, bits + 1, v)

        def sym(x):
            return 0.5 * (x + x.transpose(0, 2, 1))
        B = sym(rng.standard_normal((n, v, v))) * sv[:, None] * sv
        Bov = rng.standard_normal((n, o, v)) * so[:, None] * sv
        Boo = sym(rng.standard_normal((n, o, o))) * so[:, None] * so
        t2 = rng.standard_normal((o, o, v, v))
        t2 = 0.5 * (t2 + t2.transpose(1, 0, 3, 2)) * so[:, None, None, None] * so[:, None, None]
        if not flat_t2:
            t2 = t2 * sv[:, None] * sv
        t1 = singles * rng.standard_normal((o, v)) * so[:, None] * (1.0 if flat_t2 else sv)
        e_occ, e_vir = rng.uniform(-1.5, -0.3, o), rng.uniform(0.1, 3.0, v)
        E = lad.triples(*[to_dev(x) for x in (B, Bov, Boo, t1, t2, e_occ, e_vir)]).item()
        E_ref = reference(B, Bov, Boo, t1, t2, e_occ, e_vir)
        assert abs(E - E_ref) <= 1e-13 * abs(E_ref), (seed, E, E_ref)

def test_orbitals_without_integrals_or_amplitudes():
    """Rows of zeros: an occupied and a virtual orbital without coupling leave E(T) of the others (to the order of its sum)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_08142_gb300 as lad
    import synthetic
    x = synthetic.make_inputs(3, 9, 12, 5)
    E = lad.triples(*[to_dev(a) for a in (x.B, x.B_ov, x.B_oo, x.t1, x.t2, x.e_occ, x.e_vir)]).item()
    z = synthetic.make_inputs(4, 10, 12, 5)
    for name in ("B", "B_ov", "B_oo", "t1", "t2"):
        a, b = getattr(z, name), getattr(x, name)
        a[...] = 0.0
        a[tuple(slice(0, k) for k in b.shape)] = b
    z.e_occ[:3], z.e_vir[:9] = x.e_occ, x.e_vir
    E2 = lad.triples(*[to_dev(a) for a in (z.B, z.B_ov, z.B_oo, z.t1, z.t2, z.e_occ, z.e_vir)]).item()
    assert abs(E2 - E) <= 1e-14 * abs(E)
    zero = [np.zeros_like(a) for a in (z.B, z.B_ov, z.B_oo, z.t1, z.t2)] + [z.e_occ, z.e_vir]
    assert lad.triples(*[to_dev(a) for a in zero]).item() == 0.0
