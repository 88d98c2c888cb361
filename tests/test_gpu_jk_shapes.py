"""The kernel shape that the cost estimate picks for every part exists for its class and computes the
same J/K as one thread (or warp) per quartet, from one quartet per part to parts that fill the GPU.
FP64 against FP64: 1e-11 of the largest element (another summation order); double-float on every quartet:
1e-9 (48-bit arithmetic, a few thousand terms per element)."""
import numpy as np
import pytest

import mess_inputs as mi

pytestmark = pytest.mark.gpu

MOLECULES = {"h2": lambda: mi.h2(1.4), "water1": mi.h2o, "water6": lambda: mi.water_cluster(6, 10.9, 2),
             "c3h8": lambda: mi.alkane(3, np.random.default_rng(1))}


@pytest.mark.parametrize("mol,basis", [("h2", "sto-3g"), ("water1", "sto-3g"), ("water1", "6-31gs"), ("c3h8", "6-31g"),
                                       ("water6", "6-31gs")])
@pytest.mark.parametrize("kw,tol", [(dict(prec="fp64", schwarz_tau=1e-10), 1e-11),
                                    (dict(prec="mixed", split_df32=True, fp64_tau=1e-300, schwarz_tau=1e-10), 1e-9)])
def test_estimated_shapes(mess, mol, basis, kw, tol):
    m = MOLECULES[mol]()
    g = mess.Basis.from_molecule(m, mi.basis_path(basis))
    D = mi.random_symmetric_density(g.nbf, 7)
    J, K, _ = g.jk(D, **kw)
    table = g.jk_tuning(**kw)
    g.jk_set_tuning(table, **kw)                     # rejects a shape that its class does not have
    assert g.jk_tuning(**kw) == table
    g.jk_set_variant(G=1, team=0, **kw)
    J1, K1, _ = g.jk(D, **kw)
    assert np.abs(J - J1).max() <= tol * np.abs(J1).max()
    assert np.abs(K - K1).max() <= tol * np.abs(K1).max()
