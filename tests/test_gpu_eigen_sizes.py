"""The eigensolver at the sizes where it changes shape: two functions, odd and even matrices, every block
size, and a matrix too large for shared memory; in FP64 and double-float.  The density of a converged
closed-shell SCF is idempotent in the overlap metric, D S D = 2 D, exactly as far as the eigenvectors
and X = S^-1/2 are orthonormal: 1e-11 of the largest element in FP64, 1e-10 in double-float (48 bits through
a few hundred rotations)."""
import numpy as np
import pytest

import mess_inputs as mi

pytestmark = pytest.mark.gpu

MOLECULES = {"h2": lambda: mi.h2(1.4), "h2o": mi.h2o, "c2h6": lambda: mi.alkane(2, np.random.default_rng(1)),
             "c5h12": lambda: mi.alkane(5, np.random.default_rng(1)), "water9": lambda: mi.water_cluster(9, 12.5, 4)}


@pytest.mark.parametrize("mol,basis,n", [("h2", "sto-3g", 2), ("h2o", "sto-3g", 7), ("c2h6", "sto-3g", 16),
                                         ("h2o", "6-31gs", 19), ("c2h6", "6-31gs", 42), ("c5h12", "6-31g", 69),
                                         ("water9", "6-31gs", 171)])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-11), ("mixed", 1e-10)])
def test_density_is_idempotent(mess, mol, basis, n, prec, tol):
    g = mess.Basis.from_molecule(MOLECULES[mol](), mi.basis_path(basis))
    assert g.nbf == n
    r = g.scf(prec=prec, split_df32=prec == "mixed", schwarz_tau=1e-10, guess=mess.MESS_GUESS_SAD)
    assert r["converged"] == 1
    D, S = r["D"], g.overlap()
    assert np.abs(D @ S @ D - 2.0 * D).max() <= tol * max(1.0, np.abs(D).max())
    assert abs(float((D * S).sum()) - g.nelectron) <= 1e-9 * g.nelectron
