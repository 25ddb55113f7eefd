"""Elongated instances: a narrow column and a long box (one axis far longer), a thin ring (one far
shorter), at the most particles that 24-bit keys order.  Lists and distances exact on a sample, and the
order good enough that the warp's search settles nearly all queries: at most one in twenty reaches the
exact search (a leaf whose particles share a key and little else overruns the walk's tables)."""
import numpy as np
import pytest

from paper_2609_35967_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _instance(shape, n, K):
    rng = np.random.default_rng(11)
    if shape == "ring":
        ins = W.disk_instance(n, seed=3, K=K)
        R, phi = 50 * W.AU * (1.0 + 1e-3 * rng.uniform(-1, 1, n)), rng.uniform(0, 2 * np.pi, n)
        ins["x"], ins["y"], ins["z"] = R * np.cos(phi), R * np.sin(phi), 2e-5 * R * rng.normal(size=n)
        return ins
    ins = W.patch_instance(n, seed=4, K=K)
    L = ins["params"]["box_x"]
    if shape == "column":
        ins["z"] = 30.0 * L * rng.normal(size=n)
    else:
        ins["params"] = dict(ins["params"], box_x=100.0 * L)
        ins["x"] = 100.0 * ins["x"]
    return ins


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("shape", ["column", "long", "ring"])
def test_elongated_instances(gd, oracle, shape, precision):
    n, K = 1 << 18, 32
    ins = _instance(shape, n, K)
    sess = gd.Session([ins], K=K, precision=precision)
    P = oracle.params(ins["params"])
    idx = np.random.default_rng(1).choice(n, 64, replace=False)
    ref, rd = oracle.knn(P, ins["x"], ins["y"], ins["z"], idx)
    for _ in range(2):
        nbr, d = sess.build_neighbors(want=True)
        assert np.array_equal(nbr.cpu().numpy()[idx], ref)
        assert np.array_equal(d.cpu().numpy()[idx], rd)
    if precision == 1:
        assert sess.stats()["knn_redo"] <= 2 * n // 20
    sess.close()
