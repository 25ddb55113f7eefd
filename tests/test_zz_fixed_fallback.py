"""gd_neighbors_fixed where its walks cannot settle a query and the exact search does, at sizes of
several leaves: coincident particles beyond every buffer, shells of equal distances, a crowd whose sort
keys are all equal (a walk reaches more leaves than its table holds), and coordinates that are not
finite (a row of -1, no one's neighbour).  Lists and distances bit-exact against brute force."""
import numpy as np
import pytest

from paper_2609_35967_gb300 import workloads as W
from test_zz_no_alloc import _fixed

pytestmark = pytest.mark.gpu


def _shape(shape):
    rng = np.random.default_rng(5)
    if shape == "point":
        x, y, z = (np.full(900, 1.5) for _ in range(3))
        x[:70] = np.arange(70.0)
    elif shape == "lattice":
        x, y, z = (a.ravel() for a in np.meshgrid(*(np.arange(10.0),) * 3))
    elif shape == "crowd":
        x, y, z = (rng.normal(size=12000) for _ in range(3))
        x[7], y[11] = 1e9, -1e9
    else:
        x, y, z = (rng.normal(size=3000) for _ in range(3))
    p = rng.permutation(len(x))
    return [np.ascontiguousarray(a[p]) for a in (x, y, z)]


@pytest.mark.parametrize("K", [16, 48, 64])
@pytest.mark.parametrize("shape", ["point", "lattice", "crowd"])
def test_fixed_exact_search(gd, oracle, shape, K):
    x, y, z = _shape(shape)
    ins = dict(W.disk_instance(64, seed=3, K=K), x=x, y=y, z=z)
    idx = np.unique(np.linspace(0, len(x) - 1, 300).astype(np.int64))
    ref, rd = oracle.knn(oracle.params(dict(ins["params"], K=K)), x, y, z, idx)
    for nbr, d in _fixed(gd, ins, K):
        assert np.array_equal(nbr[idx], ref)
        assert np.array_equal(d[idx], rd)


def test_fixed_non_finite(gd, oracle):
    x, y, z = _shape("cloud")
    K, bad = 32, [5, 700, 2999]
    x[5], y[700], z[2999] = np.nan, np.inf, -np.inf
    ins = dict(W.disk_instance(64, seed=3, K=K), x=x, y=y, z=z)
    keep = np.delete(np.arange(len(x)), bad)
    ref, rd = oracle.knn(oracle.params(dict(ins["params"], K=K)), x[keep], y[keep], z[keep], np.arange(len(keep)))
    for nbr, d in _fixed(gd, ins, K):
        assert np.array_equal(nbr[keep], keep[ref])
        assert np.array_equal(d[keep], rd)
        assert np.all(nbr[bad] == -1) and np.all(d[bad] == -1.0)
