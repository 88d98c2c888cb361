"""S and T of a contracted d shell with itself are symmetric to the last bit: the elements (m, n) and (n, m) of such a
block are sums of the same terms in different orders, and one of the two has to stand for both."""
import numpy as np
import pytest

import mess_inputs as mi

pytestmark = pytest.mark.gpu


# primitives per shell: their pairs fill part of a warp, or take a second pass of it
@pytest.mark.parametrize("prims", [3, 4, 6])
def test_contracted_d_shells(mess, oracle_mod, tmp_path, prims):
    rng = np.random.default_rng(prims)
    path = str(tmp_path / "d.basis")
    with open(path, "w") as fh:
        fh.write("element O\n")
        for _ in range(16):
            fh.write(f"D {prims}\n")
            for k in range(prims):
                fh.write(f"  {rng.uniform(0.1, 0.3) * 3.0 ** k:.12f} {rng.uniform(0.2, 1.0):.12f}\n")
    m = mi.Molecule("o", np.array([8], dtype=np.int32), np.array([[0.3, -0.2, 0.1]]))
    g, o = mess.Basis.from_molecule(m, path), oracle_mod.basis_for(m, path)
    for got, ref in zip((g.overlap(), g.kinetic(), g.nuclear()), oracle_mod.one_e(o)):
        assert np.abs(got - ref).max() <= 1e-12 * np.abs(ref).max()
        assert np.array_equal(got, got.T)
