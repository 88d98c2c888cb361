"""S, T, V where the warp-per-pair kernel's split changes: one atom, fewer and more (primitive pair,
nucleus) items than lanes, more nuclei than lanes, more than 32 primitive pairs, every class up to
(d|d); Schwarz factors of contracted shells for every lane count.  FP64 against the oracle: 1e-12 of
the largest element (a few hundred rounded terms)."""
import numpy as np
import pytest

import mess_inputs as mi

pytestmark = pytest.mark.gpu

MOLECULES = {"o": lambda: mi.Molecule("o", np.array([8], dtype=np.int32), np.array([[0.3, -0.2, 0.1]])),
             "h2": lambda: mi.h2(1.4), "water1": mi.h2o, "water11": lambda: mi.water_cluster(11, 13.3, 5),
             "c4h10": lambda: mi.alkane(4, np.random.default_rng(2))}


@pytest.mark.parametrize("mol,basis", [("o", "6-31gs"), ("h2", "sto-3g"), ("water1", "6-31gs"), ("water11", "6-31gs"),
                                       ("c4h10", "6-31g"), ("c4h10", "sto-3g")])
def test_one_electron_matrices(mess, oracle_mod, mol, basis):
    m = MOLECULES[mol]()
    path = mi.basis_path(basis)
    g, o = mess.Basis.from_molecule(m, path), oracle_mod.basis_for(m, path)
    for got, ref in zip((g.overlap(), g.kinetic(), g.nuclear()), oracle_mod.one_e(o)):
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
        assert np.array_equal(got, got.T)


# pair counts per class either side of the Schwarz kernels' lane rule (1, 8 or 32 lanes per pair), and
# contracted d pairs, one block each
@pytest.mark.parametrize("mol,basis", [("h2", "sto-3g"), ("water1", "6-31gs"), ("water11", "6-31gs")])
def test_schwarz_factors(mess, oracle_mod, mol, basis):
    m = MOLECULES[mol]()
    path = mi.basis_path(basis)
    g, o = mess.Basis.from_molecule(m, path), oracle_mod.basis_for(m, path)
    Q, Qr = g.schwarz(), oracle_mod.schwarz(o)
    assert np.abs(Q - Qr).max() <= 1e-11 * Qr.max()
