"""E_xc and V_xc at the sizes where the grid kernels change shape: one function, fewer functions than
the V_xc groups, a part tile, two function tiles (more than 64 functions), and a batch of unequal
molecules; against the oracle on the same grid.  V is a sum of at most 4e5 signed FP64 terms: 1e-9
absolute on elements of order one leaves four digits over their accumulated rounding."""
import numpy as np
import pytest

import mess_inputs as mi
from oracle import dft

pytestmark = pytest.mark.gpu

MOLECULES = {"h": lambda: mi.Molecule("h", np.array([1], dtype=np.int32), np.zeros((1, 3))),
             "h2": lambda: mi.h2(1.4), "h2o": mi.h2o, "water4": lambda: mi.water_cluster(4, 9.5, 3)}


@pytest.mark.parametrize("mol,basis,kind", [("h", "sto-3g", "lda"), ("h2", "sto-3g", "pbe"), ("h2", "6-31g", "lda"),
                                            ("h2o", "6-31g", "pbe"), ("water4", "6-31gs", "lda"),
                                            ("water4", "6-31gs", "pbe")])
def test_xc_shapes(mess, oracle_mod, mol, basis, kind):
    m = MOLECULES[mol]()
    path = mi.basis_path(basis)
    g, o = mess.Basis.from_molecule(m, path), oracle_mod.basis_for(m, path)
    D = mi.random_symmetric_density(g.nbf, 11, nocc=max(1, m.nelectron // 2))
    E, V, npts = g.xc(D, kind)
    pts, w = dft.molecular_grid(o.Z, o.xyz)
    assert npts == len(w)
    Er, Vr = dft.xc(o, D, pts, w, kind)
    assert abs(E - Er) <= 1e-10 * max(1.0, abs(Er)), (E, Er)
    assert np.abs(V - Vr).max() <= 1e-9


def test_batch_of_unequal_molecules(mess):
    """Each molecule of a Kohn-Sham batch ends at the energy of its own single SCF."""
    mols = [mi.h2(1.4), mi.h2o(), mi.h2(2.0)]
    bases = [mess.Basis.from_molecule(m, mi.basis_path("6-31g")) for m in mols]
    res, _ = mess.scf_batch(bases, xc="pbe")
    for b, r in zip(bases, res):
        assert abs(b.scf(xc="pbe")["E_total"] - r["E_total"]) <= 1e-9
