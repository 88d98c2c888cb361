"""FP32 parts laid out in bra runs (from 2^19 quartets with few primitives on) against the same basis in FP64: the classes of s, p
and d shells, and a threshold low enough that kets and bras differ in
their ranges.  The reduced-precision matrices carry the FP32 integrals' relative error (1e-7 of the split
threshold per quartet): 2e-5 per element, the bound of the other reduced-precision tests; the energy of
the same density 1e-6 hartree."""
import numpy as np
import pytest

import mess_inputs as mi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,basis", [(28, "6-31gs"), (20, "6-31g")])
@pytest.mark.parametrize("tau", [1e-10, 1e-8])
def test_bra_runs_match_fp64(mess, n, basis, tau):
    m = mi.water_cluster(n, 19.0 * (n / 32.0) ** (1.0 / 3.0), 9)
    g = mess.Basis.from_molecule(m, mi.basis_path(basis))
    D = np.eye(g.nbf) + 0.1 * mi.random_symmetric_density(g.nbf, 3) * np.exp(-np.abs(np.subtract.outer(
        np.arange(g.nbf), np.arange(g.nbf))) / 20.0)
    kw = dict(prec="mixed", split_df32=True, schwarz_tau=tau)
    J64, K64, i64 = g.jk(D, prec="fp64", schwarz_tau=tau)
    J, K, i32 = g.jk(D, **kw)
    assert i64["function_quartets"] == i32["function_quartets"]
    assert np.abs(J - J64).max() <= 2e-5 and np.abs(K - K64).max() <= 2e-5
    g.jk_set_variant(G=4, team=0, **kw)              # by quartets: the same FP32 integrals in another order
    J4, K4, _ = g.jk(D, **kw)
    assert np.abs(J - J4).max() <= 2e-5 and np.abs(K - K4).max() <= 2e-5
    e = lambda A, B: 0.5 * float(np.sum(D * (A - 0.5 * B)))  # noqa: E731
    assert abs(e(J, K) - e(J64, K64)) <= 1e-6 * max(1.0, n / 8.0)
