"""The tree search at its branches, against brute force (bit-exact lists and distances): first
builds, static builds (the radius of the build before), positions changed by the caller without a
push (every stale radius fails), every kernel size, partial leaves and blocks, periodic images
near half a box, exact ties, particles on one point or line, and coordinates that are not finite."""
import numpy as np
import pytest
import torch

from paper_2609_35967_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _same(oracle, sess, ins, xyz, K):
    P = oracle.params(dict(ins["params"], K=K))
    n = len(xyz[0])
    nbr, d = sess.build_neighbors(want=True)
    onbr, od = oracle.knn(P, *xyz, np.arange(n))
    assert np.array_equal(nbr.cpu().numpy(), onbr)
    assert np.array_equal(d.cpu().numpy(), od)


def _move(sess, xyz):
    for k, v in zip(("x", "y", "z"), xyz):
        sess.t[k].copy_(torch.as_tensor(v))
    torch.cuda.synchronize()


@pytest.mark.parametrize("n,K", [(33, 32), (1025, 32), (700, 33), (2049, 48), (1500, 49), (1111, 64), (901, 65),
                                 (777, 128), (1300, 129), (640, 256)])
@pytest.mark.parametrize("disk", [False, True])
def test_first_static_and_changed_positions(gd, oracle, n, K, disk):
    make = (lambda s: W.disk_instance(n, seed=s, K=K)) if disk else (lambda s: W.patch_instance(n, seed=s, K=K))
    ins, other = make(n), make(n + 1)
    sess = gd.Session([ins], K=K, precision=n % 2)
    for data in (ins, ins, other, other, ins):
        xyz = [data[k] for k in ("x", "y", "z")]
        _move(sess, xyz)
        _same(oracle, sess, ins, xyz, K)
    assert sess.stats()["status"] == 0
    sess.close()


@pytest.mark.parametrize("shape", ["lattice", "line", "plane", "point", "clusters"])
def test_ties_and_degenerate_shapes(gd, oracle, shape):
    """Shells of equal distances, coincident particles beyond every buffer, points on a line or
    plane, and two clusters a million times their size apart."""
    n, K = 512, 20
    ins = W.disk_instance(n, seed=3, K=K)
    rng = np.random.default_rng(5)
    g = np.arange(8.0)
    x, y, z = (a.ravel() for a in np.meshgrid(g, g, g))
    if shape == "line":
        x, y, z = np.arange(float(n)), np.zeros(n), np.zeros(n)
    elif shape == "plane":
        x, y, z = rng.normal(size=n), rng.normal(size=n), np.full(n, 0.25)
    elif shape == "point":
        x, y, z = (np.full(n, 1.5) for _ in range(3))
        x[:40] = np.arange(40.0)
    elif shape == "clusters":
        x, y, z = (rng.normal(size=n) + (1e6 * (np.arange(n) % 2)) for _ in range(3))
    p = rng.permutation(n)
    xyz = [np.ascontiguousarray(a[p]) for a in (x, y, z)]
    sess = gd.Session([ins], K=K, precision=1)
    _move(sess, xyz)
    for _ in range(3):
        _same(oracle, sess, ins, xyz, K)
    sess.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_non_finite_coordinate_touches_one_particle(gd, oracle, precision):
    n, K = 600, 16
    ins = W.patch_instance(n, K=K, seed=6)
    sess = gd.Session([ins], precision=precision)
    sess.t["y"][77] = float("nan")
    torch.cuda.synchronize()
    keep = np.delete(np.arange(n), 77)
    P = oracle.params(ins["params"])
    onbr, od = oracle.knn(P, *[ins[k][keep] for k in ("x", "y", "z")], np.arange(n - 1))
    for _ in range(2):
        nbr, d = sess.build_neighbors(want=True)
        assert np.array_equal(nbr.cpu().numpy()[keep], keep[onbr])
        assert np.array_equal(d.cpu().numpy()[keep], od)
        assert np.all(nbr.cpu().numpy()[77] == 77)
    assert sess.stats(check=False)["status"] & gd.ST_KNN
    sess.close()
