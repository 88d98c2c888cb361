"""Parts of few quartets with many primitive quartets, split over blocks (a warp or a block per quartet), against one
thread per quartet: FP64 and double-float sums of the same integrals in another order, 1e-12 and 1e-9 of elements
of order ten.  One molecule has fewer primitive quartets than lanes, one a single (pp|pp) quartet, one parts of more
quartets than are split."""
import numpy as np
import pytest

import mess_inputs as mi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mol,basis", [("h2", "sto-3g"), ("h2o", "sto-3g"), ("h2o", "6-31gs"), ("c2h6", "6-31gs")])
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("shape", [dict(G=32, team=0), dict(G=1, team=3)])
def test_split_matches_one_thread(mess, mol, basis, prec, shape):
    m = {"h2": lambda: mi.h2(1.4), "h2o": mi.h2o, "c2h6": lambda: mi.alkane(2, np.random.default_rng(2))}[mol]()
    g = mess.Basis.from_molecule(m, mi.basis_path(basis))
    D = mi.random_symmetric_density(g.nbf, 5, nocc=max(1, m.nelectron // 2))
    # (mixed: every quartet in double-float)
    kw = dict(prec=prec) if prec == "fp64" else dict(prec=prec, split_df32=True, fp64_tau=1e-300)
    g.jk(D, **kw)
    g.jk_set_variant(G=1, team=0, **kw)
    J1, K1, _ = g.jk(D, **kw)
    g.jk_set_variant(**shape, **kw)
    J, K, _ = g.jk(D, **kw)
    tol = 1e-12 if prec == "fp64" else 1e-9
    scale = max(1.0, np.abs(J1).max())
    assert np.abs(J - J1).max() <= tol * scale and np.abs(K - K1).max() <= tol * scale
