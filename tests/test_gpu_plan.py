"""GPU: the work items of a build (jk_plan_kernel) cover every candidate once,
whatever the chunk, the partition and the grouping of class pairs into
launches, at the edges of their ranges."""
import numpy as np
import pytest

import oracle
from paper_2507_09772_gb300 import jk, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    mol = synth.batched_molecule(5, natm=11)
    J, K, nq = oracle.jk(mol, cutoff=1e-13)
    return mol, J, K, nq


def build(mol, options, parts=1, **kw):
    eng = jk.JK(mol)
    try:
        for k, v in options.items():
            eng.set_option(k, v)
        D = torch.tensor(mol.D, dtype=torch.float64, device="cuda")
        J = K = nq = 0
        for p in range(parts):
            if parts > 1:
                eng.set_option("part_count", parts)
                eng.set_option("part_index", p)
            j, k, st = eng.build(D, cutoff=1e-13, stats=True, **kw)
            J, K = J + j, K + k
            nq += st["quartets_fp64"] + st["quartets_fp32"]
        return J.cpu().numpy(), K.cpu().numpy(), nq
    finally:
        eng.close()


@pytest.mark.parametrize("options,parts", [
    ({}, 1), ({"chunk": 32}, 1), ({"chunk": 65536}, 1), ({"chunk": 33}, 7), ({}, 300),
    ({"profile": 1}, 1), ({"profile": 1, "branches": 8}, 2), ({"branches": 1}, 1),
    ({"use_graph": 1, "chunk": 41}, 3)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_every_candidate_once(case, options, parts, precision):
    mol, Jr, Kr, nq = case
    if precision == "mixed" and parts == 300:
        parts = 2
    J, K, n = build(mol, options, parts, precision=precision)
    assert n == nq
    tol = 1e-10 if precision == "fp64" else 1e-8
    assert np.abs(J - Jr).max() <= tol and np.abs(K - Kr).max() <= tol


@pytest.mark.parametrize("scale", [1.0, 1e-9, 30.0])
@pytest.mark.parametrize("use_dmax", [0, 1])
def test_item_bound_follows_the_density(case, scale, use_dmax):
    """The items are listed from this build's largest density element: a small
    change of the density and one far above 1 keep the oracle's quartets."""
    mol = case[0]
    D = mol.D * scale
    Jr, Kr, nq = oracle.jk(mol, D=D, cutoff=1e-13, use_dmax=bool(use_dmax))
    eng = jk.JK(mol)
    try:
        eng.set_option("use_dmax", use_dmax)
        J, K, st = eng.build(torch.tensor(D, dtype=torch.float64, device="cuda"), cutoff=1e-13, stats=True)
    finally:
        eng.close()
    assert st["quartets_fp64"] == nq
    assert np.abs(J.cpu().numpy() - Jr).max() <= 1e-10 * max(scale, 1e-3)
    assert np.abs(K.cpu().numpy() - Kr).max() <= 1e-10 * max(scale, 1e-3)
