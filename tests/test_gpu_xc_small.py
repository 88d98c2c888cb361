"""E_xc and V_xc of molecules with one to four functions, whose V_xc the functional kernel sums itself, against the
oracle on the same grid, and a batch in which the molecules differ in size.  The bounds are those of the
larger molecules: V is a sum of FP64 terms of order one or less."""
import numpy as np
import pytest

import mess_inputs as mi
from oracle import dft

pytestmark = pytest.mark.gpu


def _chain(n):
    return mi.Molecule(f"h{n}", np.ones(n, dtype=np.int32), np.array([[0.1 * k, 0.3 * (k % 2), 1.5 * k] for k in range(n)]))


@pytest.mark.parametrize("n,basis", [(1, "sto-3g"), (2, "sto-3g"), (3, "sto-3g"), (4, "sto-3g"), (2, "6-31g"), (5, "sto-3g")])
@pytest.mark.parametrize("kind", ["lda", "pbe"])
def test_small_molecules(mess, oracle_mod, n, basis, kind):
    m, path = _chain(n), mi.basis_path(basis)
    g, o = mess.Basis.from_molecule(m, path), oracle_mod.basis_for(m, path)
    D = mi.random_symmetric_density(g.nbf, 7, nocc=max(1, n // 2))
    E, V, npts = g.xc(D, kind)
    pts, w = dft.molecular_grid(o.Z, o.xyz)
    assert npts == len(w)
    Er, Vr = dft.xc(o, D, pts, w, kind)
    assert abs(E - Er) <= 1e-10 * max(1.0, abs(Er)), (E, Er)
    assert np.abs(V - Vr).max() <= 1e-9


@pytest.mark.parametrize("kind", ["lda", "pbe"])
def test_batch_of_unequal_small_molecules(mess, kind):
    bases = [mess.Basis.from_molecule(_chain(n), mi.basis_path("sto-3g")) for n in (2, 4, 2)]
    res, _ = mess.scf_batch(bases, xc=kind)
    for b, r in zip(bases, res):
        assert abs(b.scf(xc=kind)["E_total"] - r["E_total"]) <= 1e-9
