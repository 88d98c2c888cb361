"""Bra runs in a batch: several molecules share a part, molecules leave as they converge, and late incremental builds screen
single quartets of a run by their density.  256 stretched or squeezed water trimers / 6-31G in reduced precision
against the same batch in FP64 (held to the oracle by the batch tests): 1e-6 hartree after the final energy, the bound
of those tests, and 1e-5 per water for the iterations' own energies."""
import numpy as np
import pytest

import mess_inputs as mi

pytestmark = pytest.mark.gpu

RUN_MIN, RUN_PRIM = 1 << 19, 16      # quartets of a part, and primitive quartets of each, from which it is laid out in runs
RUN_CLASSES = {(0, 0, 0, 0), (1, 0, 0, 0), (1, 0, 1, 0), (1, 1, 0, 0), (1, 1, 1, 0)}   # those of s and p shells


def test_batch_in_runs_matches_fp64(mess):
    torch = pytest.importorskip("torch")
    path = mi.basis_path("6-31g")
    m0 = mi.water_cluster(3, 8.0, 6)
    mols = [mi.Molecule("w3", m0.Z, m0.xyz * f) for f in np.linspace(0.92, 1.15, 256)]
    bases = [mess.Basis.from_molecule(m, path) for m in mols]
    kw = dict(prec="mixed", split_df32=True, schwarz_tau=1e-10)
    # the parts of a batch are those of its molecules put together
    g = bases[128]
    D = torch.eye(g.nbf, dtype=torch.float64, device="cuda")
    parts = g.jk_profile(D, torch.empty_like(D), torch.empty_like(D), **kw)
    taken = {tuple(p[k] for k in ("la", "lb", "lc", "ld")) for p in parts
             if not p["fp64"] and 256 * 0.9 * p["shell_quartets"] >= RUN_MIN
             and p["primitive_quartets"] <= RUN_PRIM * p["shell_quartets"]}
    assert len(taken & RUN_CLASSES) >= 2, taken
    ref, st = mess.scf_batch(bases, prec="fp64", schwarz_tau=1e-12)
    assert st == mess.MESS_OK
    res, st = mess.scf_batch(bases, **kw)
    assert st == mess.MESS_OK
    E, Ei, E64 = (np.array([r[k] for r in rs]) for rs, k in ((res, "E_total"), (res, "E_iter"), (ref, "E_total")))
    assert np.abs(E - E64).max() <= 1e-6, np.abs(E - E64).max()
    assert np.abs(Ei - E64).max() <= 3e-5, np.abs(Ei - E64).max()
    assert len({r["iterations"] for r in res}) > 1   # molecules left at different iterations
