"""GPU: the work items of a build (jk_plan_kernel) cover every candidate once,
whatever the chunk, the partition and the grouping of class pairs into
launches, at the edges of their ranges."""
import itertools

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


def build(mol, options, parts=1, full=False, **kw):
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
        return (J.cpu().numpy(), K.cpu().numpy(), nq) + ((st,) if full else ())
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


def tuning_table(path, only=None):
    """Other shapes for the s and p classes than the built-in rule's, as another rank's autotuner might have stored."""
    p = torch.cuda.get_device_properties(0)
    name = "".join(c if c.isalnum() and c.isascii() else "_" for c in p.name)
    shape = {"1010": "3 1 1 1", "1011": "1 1 3 1", "1110": "3 1 1 1", "1100": "3 1 1 1", "1000": "3 1 1 1"}
    with open(path / f"tune_{name}_sm{p.major}{p.minor}_{p.multi_processor_count}.txt", "w") as f:
        for k, v in shape.items():
            for n in [only] if only else itertools.product([1, 3, 6], repeat=4):
                for t in (0, 1, 2):
                    f.write("%s/%d_%d_%d_%d/%d %s\n" % (k, *n, t, v))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_parts_of_differently_tuned_handles_sum_to_the_build(case, precision, tmp_path, monkeypatch):
    """Ranks tune, chunk and profile by themselves: the parts still hold every quartet once."""
    mol, Jr, Kr, nq = case
    J = K = n = 0
    shapes = []
    for part in range(3):
        where = tmp_path / str(part)
        where.mkdir()
        if part == 1:
            tuning_table(where)
        monkeypatch.setenv("JK_TUNING_DIR", str(where))
        eng = jk.JK(mol)
        for k, v in {"part_count": 3, "part_index": part, "profile": int(part == 2), "chunk": 41 if part == 2 else 64}.items():
            eng.set_option(k, v)
        j, k, st = eng.build(torch.tensor(mol.D, dtype=torch.float64, device="cuda"), cutoff=1e-13, precision=precision,
                             stats=True)
        J, K, n = J + j.cpu().numpy(), K + k.cpu().numpy(), n + st["quartets_fp64"] + st["quartets_fp32"]
        eng.set_option("profile", 1)
        eng.build(torch.tensor(mol.D, dtype=torch.float64, device="cuda"), precision=precision, stats=True)
        shapes.append({(p["la"], p["lb"], p["lc"], p["ld"], p["tier"]): p["threads_per_quartet"] for p in jk.jk_profile(eng.h)})
        eng.close()
    assert shapes[1] != shapes[0]     # the table took effect
    assert n == nq
    tol = 1e-10 if precision == "fp64" else 1e-8
    assert np.abs(J - Jr).max() <= tol and np.abs(K - Kr).max() <= tol


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("use_graph", [0, 1])
def test_branches_1_keeps_the_build_on_the_callers_stream(case, precision, use_graph):
    mol, Jr, Kr, _ = case
    eng = jk.JK(mol)
    eng.set_option("use_graph", use_graph)
    assert eng.get_option("branches") == 1
    D = torch.tensor(mol.D, dtype=torch.float64, device="cuda")
    tol = 1e-10 if precision == "fp64" else 1e-8
    for branches, streams in ((None, 24), (1, 1), (4, 24), (1, 1)):
        if branches:
            eng.set_option("branches", branches)
        J, K, st = eng.build(D, precision=precision, stats=True)
        assert eng.get_option("streams") == min(streams, st["kernel_launches"])
        assert np.abs(J.cpu().numpy() - Jr).max() <= tol and np.abs(K.cpu().numpy() - Kr).max() <= tol
    assert eng.get_option("graphs") == 2 * use_graph
    eng.close()


def test_an_eager_build_keeps_the_priority_of_the_callers_stream(case):
    mol, Jr, Kr, _ = case
    eng = jk.JK(mol)
    D = torch.tensor(mol.D, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for priority in (0, -1, 0):
        s = torch.cuda.Stream(priority=priority)
        with torch.cuda.stream(s):
            J, K, _ = eng.build(D)
        s.synchronize()
        assert eng.get_option("stream_priority") == priority
        assert np.abs(J.cpu().numpy() - Jr).max() <= 1e-10 and np.abs(K.cpu().numpy() - Kr).max() <= 1e-10
    eng.close()


@pytest.mark.parametrize("prims", [(3, 3, 3, 3), (1, 3, 1, 3), None])
def test_tuned_class_pairs_still_share_a_launch(case, prims, tmp_path, monkeypatch):
    """Shapes stored for some class pairs of an angular momentum do not split its launch."""
    mol, Jr, Kr, nq = case
    launches = []
    for tuned in (False, True):
        where = tmp_path / str(tuned)
        where.mkdir()
        if tuned:
            tuning_table(where, prims)
        monkeypatch.setenv("JK_TUNING_DIR", str(where))
        J, K, n, st = build(mol, {}, full=True)
        launches.append(st["kernel_launches"])
        assert n == nq and np.abs(J - Jr).max() <= 1e-10 and np.abs(K - Kr).max() <= 1e-10
    assert launches[0] == launches[1]


@pytest.mark.parametrize("shells", [
    [(1, [0.3])], [(2, [0.4])], [(0, [2.0, 0.3]), (1, [0.4])], [(2, [0.6]), (2, [0.25])], [(0, [0.4]), (3, [0.7])]])
@pytest.mark.parametrize("precision", ["fp64", "mixed", "fp32"])
def test_uncontracted_and_mixed_launches_of_many_quartets(shells, precision):
    """Launches whose items keep many kets, with the primitive loops and (all
    class pairs uncontracted) without them, against the oracle."""
    rng = np.random.default_rng(3)
    natm = 10 if shells[-1][0] == 3 else 22
    xyz = synth._rejection_box(rng, natm, (natm / 0.08) ** (1.0 / 3.0), 0.9)
    mol = synth.custom_basis_molecule(xyz, [shells] * natm, rng)
    Jr, Kr, nq = oracle.jk(mol, cutoff=1e-13)
    J, K, n = build(mol, {}, precision=precision)
    assert n == nq
    tol = {"fp64": 1e-10, "mixed": 1e-8, "fp32": 1e-3}[precision]
    assert np.abs(J - Jr).max() <= tol and np.abs(K - Kr).max() <= tol
