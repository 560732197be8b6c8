"""Plans and triples with the least workspace: the FP64 ladder on the FP64 units,
FP64 triples on the CUDA cores, and the dressing's products in their smallest
blocks, against the CPU oracle with the bars of the usual forms (FP64 1e-12,
error-free 1e-10).  Sizes between the two choose the least form, and smaller
ones are refused."""
import numpy as np
import pytest

import oracle
import synthetic
from gpu_util import rel_err, run_dressed, run_forward, to_dev

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# one occupied orbital; ragged tiles; two chunks of occupied pairs of each sign (o = 17)
SHAPES = [(1, 5, 3, 11), (5, 17, 33, 12), (17, 24, 20, 15), (7, 41, 70, 14)]


@pytest.fixture(scope="module")
def lad():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1810_08142_gb300 as lad
    return lad


def shrink(lad, L, spare=0):
    """L with its least workspace (and `spare` bytes more)."""
    least, size = lad.ladder_workspace_least(L.plan), lad.ladder_workspace_size(L.plan)
    assert least + spare < size == L.workspace.numel()
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    with pytest.raises(lad.LadderError) as e:
        lad.ladder_set_workspace(L.plan, ws[:least - 1])
    assert lad.STATUS[e.value.status] == "LADDER_EWORKSPACE"
    L.workspace = torch.empty(least + spare, dtype=torch.uint8, device="cuda")
    lad.ladder_set_workspace(L.plan, L.workspace)
    assert lad.ladder_workspace_size(L.plan) == size and lad.ladder_workspace_least(L.plan) == least
    return L


@pytest.mark.parametrize("o,v,n,seed", SHAPES)
def test_fp64_ladder_and_gradient(lad, o, v, n, seed):
    x = synthetic.make_inputs(o, v, n, seed)
    L = shrink(lad, lad.Ladder(o, v, n, mode="fp64", backward=True), spare=256)
    tau, R, E = run_forward(L, x)
    assert rel_err(R, oracle.ladder(x.B, tau)) < 1e-12
    W = oracle.energy_weights(x.t2)
    dtau, dB = L.backward(to_dev(x.B), to_dev(tau), to_dev(W))
    assert rel_err(dtau.cpu().numpy(), oracle.grad_tau(x.B, W)) < 1e-12
    assert rel_err(dB.cpu().numpy(), oracle.grad_B(x.B, tau, W)) < 1e-12
    # and back to the full one
    L.workspace = torch.empty(lad.ladder_workspace_size(L.plan), dtype=torch.uint8, device="cuda")
    lad.ladder_set_workspace(L.plan, L.workspace)
    full = L.apply(to_dev(x.B), to_dev(tau)).cpu().numpy()
    fresh = lad.Ladder(o, v, n, mode="fp64").apply(to_dev(x.B), to_dev(tau)).cpu().numpy()
    assert np.array_equal(full, fresh)


@pytest.mark.parametrize("mode,tol", [("fp64", 1e-12), ("ozaki", 1e-10)])
@pytest.mark.parametrize("o,v,n,seed", [(5, 17, 33, 12), (12, 140, 150, 21)])
def test_dressed(lad, mode, tol, o, v, n, seed):
    x = synthetic.make_inputs(o, v, n, seed)
    tau, R, _ = run_dressed(shrink(lad, lad.Ladder(o, v, n, mode=mode, dressed=True)), x)
    assert rel_err(R, oracle.ladder_dressed(x.B, x.B_ov, x.t1, tau)) < tol


@pytest.mark.parametrize("o,v,n,seed", [(3, 5, 4, 7), (5, 17, 33, 12), (3, 140, 60, 23), (17, 33, 40, 24)])
def test_triples(lad, o, v, n, seed):
    x = synthetic.make_inputs(o, v, n, seed)
    args = [to_dev(a) for a in (x.B, x.B_ov, x.B_oo, x.t1, x.t2, x.e_occ, x.e_vir)]
    least = lad.ladder_triples_workspace_least(o, v, n, 0)
    assert least < lad.ladder_triples_workspace_size(o, v, n, 0)
    ws = torch.empty(least, dtype=torch.uint8, device="cuda")
    E = lad.triples(*args, workspace=ws).item()
    E_o = oracle.triples(x.B, x.B_ov, x.B_oo, x.t1, x.t2, x.e_occ, x.e_vir)
    assert abs(E - E_o) < 1e-12 * abs(E_o)
    with pytest.raises(lad.LadderError):
        lad.triples(*args, workspace=ws[:least - 1])


def test_other_forms_have_one_size(lad):
    for mode in ("bf16x3", "bf16x6", "ozaki"):
        L = lad.Ladder(4, 24, 96, mode=mode)
        size = lad.ladder_workspace_size(L.plan)
        assert lad.ladder_workspace_least(L.plan) == size
        with pytest.raises(lad.LadderError):
            lad.ladder_set_workspace(L.plan, L.workspace[:size - 1])
    for prec in (1, 2):
        assert lad.ladder_triples_workspace_least(4, 24, 96, prec) == lad.ladder_triples_workspace_size(4, 24, 96, prec)


def test_binding_takes_the_least_where_memory_is_short(lad, monkeypatch):
    o, v, n, seed = 5, 17, 33, 12
    x = synthetic.make_inputs(o, v, n, seed)
    args = [to_dev(a) for a in (x.B, x.B_ov, x.B_oo, x.t1, x.t2, x.e_occ, x.e_vir)]
    sizes = {lad.ladder_triples_workspace_size(o, v, n, 0)}
    L = lad.Ladder(o, v, n, mode="fp64")
    sizes.add(lad.ladder_workspace_size(L.plan))
    empty = torch.empty

    def short(*shape, **kw):
        if kw.get("dtype") is torch.uint8 and shape[0] in sizes:
            raise torch.cuda.OutOfMemoryError("no room")
        return empty(*shape, **kw)
    monkeypatch.setattr(torch, "empty", short)
    L = lad.Ladder(o, v, n, mode="fp64")
    assert L.workspace.numel() == lad.ladder_workspace_least(L.plan)
    tau, R, _ = run_forward(L, x)
    assert rel_err(R, oracle.ladder(x.B, tau)) < 1e-12
    E_o = oracle.triples(x.B, x.B_ov, x.B_oo, x.t1, x.t2, x.e_occ, x.e_vir)
    assert abs(lad.triples(*args).item() - E_o) < 1e-12 * abs(E_o)
