"""FP32 quartets whose primitive quartets are split over 4, 8 or 32 lanes: K is no further from FP64 than with one thread
per quartet.  A lane's chain of additions is shorter than the thread's, and the lanes' sums are rounded once; so the
error is smaller, and 1.05 leaves room for the scatter of a mean over eight molecules and densities."""
import numpy as np
import pytest

import mess_inputs as mi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def errors(mess):
    """Relative error of K per lane count, one row per molecule."""
    out = []
    for seed in range(40, 48):
        m = mi.alkane(7, np.random.default_rng(seed))
        g = mess.Basis.from_molecule(m, mi.basis_path("6-31g"))
        near = np.exp(-np.abs(np.subtract.outer(np.arange(g.nbf), np.arange(g.nbf))) / 20.0)
        D = mi.random_symmetric_density(g.nbf, seed, nocc=m.nelectron // 2) * near
        kw = dict(prec="mixed", schwarz_tau=1e-10, fp64_tau=1e-3, split_df32=True)
        _, ref, _ = g.jk(D, prec="fp64", schwarz_tau=1e-10)
        row = []
        for G in (1, 4, 8, 32):
            g.jk(D, **kw)
            g.jk_set_variant(G=G, team=0, **kw)
            row.append(np.linalg.norm(g.jk(D, **kw)[1] - ref) / np.linalg.norm(ref))
        out.append(row)
    return np.array(out)


@pytest.mark.parametrize("k,G", [(1, 4), (2, 8), (3, 32)])
def test_lanes_round_no_more_than_one_thread(errors, k, G):
    assert (errors[:, k] / errors[:, 0]).mean() <= 1.05, errors
