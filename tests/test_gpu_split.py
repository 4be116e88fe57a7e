"""GPU: the split tier (FP64-tier quartets below the split threshold evaluated
in pairs of floats).

Two floats carry 48 bits; an integral takes some hundred operations, each
within 2^-46 of its result, a relative error of at most 2e-12 (J and K so built
were 1e-14 off for s, p, d shells, 4e-13 with f shells), so with every quartet
in two floats (split = 1) and |J|, |K| below 50 the result stays within 1e-10;
at the default threshold, 1/128 of the largest bound, within 1e-12 of the
all-FP64 build.
"""
import numpy as np
import pytest

import oracle
from paper_2507_09772_gb300 import jk, synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")


def build(mol, split, options=(), **kw):
    eng = jk.JK(mol)
    try:
        eng.set_option("split", split)
        for k, v in dict(options).items():
            eng.set_option(k, v)
        D = torch.tensor(mol.D, dtype=torch.float64, device="cuda")
        J, K, st = eng.build(D, cutoff=1e-13, stats=True, **kw)
        return [None if x is None else x.cpu().numpy() for x in (J, K)], st["quartets_fp64"]
    finally:
        eng.close()


def one_l(l, seed):
    """Two atoms with one shell type of angular momentum l and an s shell."""
    rng = np.random.default_rng(seed)
    xyz = np.array([[0.0, 0.1, -0.2], [1.1, -0.4, 0.7]])
    return synth.custom_basis_molecule(xyz, [[(l, [2.3, 0.4][: 2 if l < 3 else 1]), (0, [30.0, 0.5])]] * 2, rng)


CASES = {
    "tiny": lambda: (synth.tiny_631gs(), {}, {}),
    "two densities": lambda: (synth.random_small_molecule(5, natm=3, lmax=2, n_dm=2), {}, {}),
    "j only": lambda: (synth.batched_molecule(4, natm=10), {}, {"with_k": False}),
    "k only": lambda: (synth.batched_molecule(4, natm=10), {}, {"with_j": False}),
    "erf": lambda: (synth.random_small_molecule(6, natm=3, lmax=2), {"omega": 0.4}, {}),
    "erfc": lambda: (synth.random_small_molecule(6, natm=3, lmax=2), {"omega": -0.4}, {}),
    "no dmax": lambda: (synth.random_small_molecule(8, natm=3, lmax=2), {"use_dmax": 0}, {}),
    "spherical": lambda: (synth.random_small_molecule(9, natm=2, lmax=3, spherical=True), {}, {}),
    "p": lambda: (one_l(1, 1), {}, {}), "d": lambda: (one_l(2, 2), {}, {}), "f": lambda: (one_l(3, 3), {}, {}),
    "g": lambda: (one_l(4, 4), {}, {}),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_two_float_quartets(name):
    mol, options, kw = CASES[name]()
    ref, n0 = build(mol, 0.0, options, **kw)
    for split, tol in ((1.0, 1e-10), (1.0 / 128, 1e-12)):
        got, n = build(mol, split, options, **kw)
        assert n == n0            # every quartet in exactly one of the tiers
        for a, b in zip(got, ref):
            if b is not None:
                assert np.abs(a - b).max() <= tol * max(1.0, np.abs(b).max() / 50)


def test_every_quartet_in_two_floats_against_the_oracle():
    mol = synth.batched_molecule(2, natm=12)
    (J, K), n = build(mol, 1.0)
    Jr, Kr, nq = oracle.jk(mol, cutoff=1e-13)
    assert n == nq
    assert np.abs(J - Jr).max() <= 1e-10 and np.abs(K - Kr).max() <= 1e-10


def test_scaled_density_keeps_the_relative_error():
    """The threshold follows the density: a small change of it is built as
    exactly, relative to its own size, as a whole density."""
    mol = synth.tiny_631gs()
    mol.D = mol.D * 2.0 ** -12
    (J0, K0), _ = build(mol, 0.0)
    (J1, K1), _ = build(mol, 1.0 / 128)
    assert np.abs(J1 - J0).max() <= 1e-12 * 2.0 ** -12 and np.abs(K1 - K0).max() <= 1e-12 * 2.0 ** -12


def test_a_basis_outside_the_fp32_range_stays_in_fp64():
    rng = np.random.default_rng(3)
    mol = synth.custom_basis_molecule(np.array([[0.0, 0, 0], [1.2, 0, 0.3]]), [[(0, [3e8]), (0, [0.7]), (1, [1.1])]] * 2, rng)
    (J0, K0), n0 = build(mol, 0.0)
    (J1, K1), n1 = build(mol, 1.0)
    assert n0 == n1
    assert np.abs(J1 - J0).max() <= 1e-13 * np.abs(J0).max() and np.abs(K1 - K0).max() <= 1e-13 * np.abs(K0).max()


@pytest.mark.parametrize("split", [1.0, 1.0 / 128])
def test_a_nan_in_the_density_stays_one(split):
    """A queued build of a density with a NaN leaves NaN wherever the all-FP64
    build does, nothing finite in its place, and the error word is raised."""
    mol = synth.batched_molecule(4, natm=10)
    mol.D = mol.D.copy()
    mol.D[0, 5, 11] = mol.D[0, 11, 5] = np.nan
    got = []
    for s in (0.0, split):
        eng = jk.JK(mol)
        eng.set_option("split", s)
        J, K, _ = eng.build(torch.tensor(mol.D, dtype=torch.float64, device="cuda"), cutoff=1e-13, check=False)
        with pytest.raises(jk.JKError):
            jk.jk_check(eng.h)
        got.append((J.cpu().numpy(), K.cpu().numpy()))
        eng.close()
    for a, b in zip(*got):
        assert not np.isfinite(a).all()
        assert (np.isfinite(a) == np.isfinite(b)).all()
        m = np.isfinite(a)
        assert np.abs(a - b)[m].max(initial=0.0) <= 1e-10


@pytest.mark.parametrize("scale", [1e-34, 1e-22, 1e18, 1e37])
@pytest.mark.parametrize("use_dmax", [0, 1])
def test_densities_near_the_ends_of_the_fp32_range(scale, use_dmax):
    """Whatever the screening takes for the density's size, a density outside
    1e-15 .. 1e15 is built in FP64 instructions: the same result but for the
    order of the sums (1e-13 of the largest element)."""
    mol = synth.tiny_631gs()
    mol.D = mol.D * scale
    eng = jk.JK(mol)
    D = torch.tensor(mol.D, dtype=torch.float64, device="cuda")
    eng.set_option("use_dmax", use_dmax)
    got = []
    for split in (0.0, 1.0):
        eng.set_option("split", split)
        J, K, st = eng.build(D, cutoff=1e-13 if scale > 1 or not use_dmax else 1e-28, stats=True)
        got.append((J.cpu().numpy() / scale, K.cpu().numpy() / scale, st["quartets_fp64"]))
    eng.close()
    assert got[0][2] == got[1][2]
    for a, b in zip(got[0][:2], got[1][:2]):
        assert np.isfinite(b).all() and np.abs(a - b).max() <= 1e-13 * max(1.0, np.abs(a).max())


@pytest.mark.parametrize("omega", [1e-40, 1e-9, 1e-6, 1e6, -1e6, 1e16, 1e17, 2e19, -2e19, 1e100])
def test_range_separation_at_the_ends_of_the_fp32_range(omega):
    """omega^2 enters the roots of erf(omega r)/r: where FP32 cannot hold it to
    48 bits the build takes FP64 instructions."""
    mol = synth.tiny_631gs()
    (J0, K0), n0 = build(mol, 0.0, {"omega": omega})
    (J1, K1), n1 = build(mol, 1.0, {"omega": omega})
    assert n0 == n1
    for a, b in ((J0, J1), (K0, K1)):
        # erfc is the difference of 1/r (|J| and |K| up to 50) and erf
        top = 50.0 if omega < 0 else np.abs(a).max()
        # in range: two floats (1e-10 of |J| up to 50); outside: the order of the sums
        assert np.isfinite(b).all() and np.abs(a - b).max() <= (2e-12 if 1e-6 <= abs(omega) <= 1e6 else 1e-13) * top


def two_float_quartets(mol):
    eng = jk.JK(mol)
    try:
        eng.set_option("profile", 1)
        eng.build(torch.tensor(mol.D, dtype=torch.float64, device="cuda"), cutoff=1e-13, stats=True)
        return sum(p["quartets"] for p in jk.jk_profile(eng.h) if p["tier"] == 2)
    finally:
        eng.close()


@pytest.mark.parametrize("alpha,coef", [(1.1e-5, 2e-8), (1.1e-5, 1e-7), (3e-6, 9e7)])
def test_intermediates_beyond_the_fp32_range_stay_in_fp64(alpha, coef):
    """A diffuse g shell passes (1 / 2p)^8 in one table entry, 3e41 here, although
    its integrals and the products with the density are in range."""
    rng = np.random.default_rng(8)
    mol = synth.custom_basis_molecule(np.array([[0.0, 0, 0], [40.0, 5.0, -9.0]]), [[(4, [alpha]), (0, [0.4])]] * 2, rng)
    mol.coeffs = np.where(mol.exps < 1e-3, coef, mol.coeffs)
    (J0, K0), n0 = build(mol, 0.0)
    (J1, K1), n1 = build(mol, 1.0)
    assert n0 == n1 and two_float_quartets(mol) == 0
    for a, b in ((J0, J1), (K0, K1)):
        assert np.isfinite(b).all() and np.abs(a - b).max() <= 1e-13 * np.abs(a).max()


@pytest.mark.parametrize("name", ["tiny", "spherical", "g", "batch"])
def test_ordinary_bases_take_two_floats(name):
    mol = synth.batched_molecule(3, natm=12) if name == "batch" else CASES[name]()[0]
    assert two_float_quartets(mol) > 0


def test_the_range_is_judged_molecule_by_molecule():
    rng = np.random.default_rng(8)
    wide = synth.custom_basis_molecule(np.array([[0.0, 0, 0], [1.2, 0, 0.3]]), [[(0, [3e8]), (0, [0.7]), (1, [1.1])]] * 2, rng)
    eng = jk.JK([wide, synth.batched_molecule(3, natm=6)])
    eng.set_option("profile", 1)
    eng.build([torch.tensor(m.D, dtype=torch.float64, device="cuda") for m in (wide, synth.batched_molecule(3, natm=6))], stats=True)
    assert sum(p["quartets"] for p in jk.jk_profile(eng.h) if p["tier"] == 2) > 0
    eng.close()


@pytest.mark.parametrize("cutoff,precision,tau32,set_split,taken", [
    (1e-13, "fp64", 1e-4, False, True), (9.9e-14, "fp64", 1e-4, False, False), (1e-15, "fp64", 1e-4, False, False),
    (1e-15, "fp64", 1e-4, True, True), (1e-15, "mixed", 1e-4, False, True), (1e-15, "mixed", 9e-9, False, False),
    (1e-13, "mixed", 1e-12, False, True), (1e-12, "fp64", 1e-4, False, True)])
def test_two_floats_only_where_the_cutoff_covers_their_error(cutoff, precision, tau32, set_split, taken):
    mol = synth.tiny_631gs()
    eng = jk.JK(mol)
    eng.set_option("tau32", tau32)
    D = torch.tensor(mol.D, dtype=torch.float64, device="cuda")
    if set_split:
        eng.set_option("split", eng.get_option("split"))
    eng.set_option("profile", 1)
    eng.build(D, cutoff=cutoff, precision=precision, stats=True)
    assert (sum(p["quartets"] for p in jk.jk_profile(eng.h) if p["tier"] == 2) > 0) == taken
    eng.close()
