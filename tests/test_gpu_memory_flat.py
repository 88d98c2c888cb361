"""Calls that allocate their own workspaces give them back: the free memory of the device after many
repetitions is what it was after the first ones.  Each of these calls takes at least 0.4 MB, which 24
repetitions would show beside the allocator's 2 MB granularity."""
import numpy as np
import pytest

import mess_inputs as mi

pytestmark = pytest.mark.gpu

STO = mi.basis_path("sto-3g")


def _gradient(mess, tmp_path):
    g = mess.Basis.from_molecule(mi.alkane(2, np.random.default_rng(1)), mi.basis_path("6-31g"))
    return lambda: g.gradient()


def _network(mess, tmp_path):
    X, T, M = (np.zeros((64, k), dtype=np.float32) for k in (112, 25, 25))
    M[:, 0] = 1.0

    def call():
        net = mess.MLP(seed=1)
        net.loss_grad(X, T, M)
        net.close()
    return call


def _features(mess, tmp_path):
    g = mess.Basis.from_molecule(mi.alkane(12, np.random.default_rng(2)), STO)
    D = mi.random_symmetric_density(g.nbf, 3)
    return lambda: mess.mlp_features(g, D)


def _predict(mess, tmp_path):
    g = mess.Basis.from_molecule(mi.alkane(12, np.random.default_rng(2)), STO)
    net = mess.MLP(seed=1)
    return lambda: net.predict(g)


def _guess(mess, tmp_path):
    bases = [mess.Basis.from_molecule(m, STO) for m in mi.alkane_batch(8, 6, 8, 4)]
    w = str(tmp_path / "w.bin")
    mess.MLP(seed=1).save(w)
    return lambda: mess.scf_batch(bases, prec="mixed", split_df32=True, guess=mess.MESS_GUESS_MLP, mlp_weights=w, max_iter=2)


def _train(mess, tmp_path):
    bases = [mess.Basis.from_molecule(m, STO) for m in mi.alkane_batch(8, 3, 5, 5)]
    net = mess.MLP(seed=1)
    return lambda: net.train(bases, epochs=1, batch_rows=256)


@pytest.mark.parametrize("make", [_gradient, _network, _features, _predict, _guess, _train], ids=lambda f: f.__name__[1:])
def test_free_memory_stays(mess, tmp_path, make):
    torch = pytest.importorskip("torch")
    call = make(mess, tmp_path)
    for _ in range(3):
        call()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for _ in range(24):
        call()
    torch.cuda.synchronize()
    assert before - torch.cuda.mem_get_info()[0] <= 4 << 20
