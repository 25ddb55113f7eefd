"""The per-particle passes at the edges of their tiles: instances one below, at and one above the
smallest tile, equal grains (a warp's lanes in one bin) and a broad distribution (many bins), and
the same instance in small and in large tiles.  The bars are those of the interval parity tests:
FP64 moments 1e-12 relative, mixed 2e-4."""
import numpy as np
import pytest

from paper_2609_35967_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {0: 1e-12, 1: 2e-4}


def _broad(ins, seed):
    ins["s"] = ins["s"] * 10.0 ** np.random.default_rng(seed).uniform(-2.0, 2.0, len(ins["s"]))
    return ins


def _bins(sess, b):
    return [np.array(a) for a in sess.controller_bins(b)]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("broad", [False, True])
def test_tile_edges_match_oracle(gd, oracle, precision, broad):
    insts = [W.patch_instance(n, K=32, seed=n) for n in (255, 256, 257, 513, 33, 4097)]
    if broad:
        insts = [_broad(ins, 9) for ins in insts]
    sess = gd.Session(insts, precision=precision)
    sess.build_neighbors()
    sess.collision_rates()
    got = [_bins(sess, b) for b in range(len(insts))]
    sess.sample_collisions()
    stats = sess.stats(check=False)
    for b, ins in enumerate(insts):
        P = oracle.params(ins["params"])
        st = oracle.new_state(P)
        ref = oracle.interval_step(P, st, ins["x"], ins["y"], ins["z"], ins["s"].copy(), ins["M"],
                                   want=("A_b", "B_b"))
        n = st.n_groups
        for k, g in zip(("A_b", "B_b"), got[b]):
            assert len(g) == n
            r = ref[k][:n]
            assert np.array_equal(r == 0.0, g == 0.0)
            assert np.all(np.abs(g - r) <= TOL[precision] * r), (b, k)
        inst = stats["instances"][b]
        near = inst["near_dt"] + inst["near_audit"] + st.near_dt + st.near_audit
        assert near > 0 or abs(inst["dt_exe"] / st.dt_exe - 1.0) <= TOL[precision]
        assert near > 0 or inst["C"] == st.C
    sess.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_small_and_large_tiles_agree(gd, precision):
    """700,000 particles beside it take the tile of 1,500 particles from 256 to 1,024."""
    small = _broad(W.patch_instance(1500, K=32, seed=2), 4)
    big = W.patch_instance(700000, K=32, seed=3)
    out = []
    for insts in ([small], [small, big]):
        sess = gd.Session(insts, precision=precision)
        sess.build_neighbors()
        sess.collision_rates()
        out.append(_bins(sess, 0))
        sess.close()
    for a, b in zip(*out):
        assert len(a) == len(b)
        assert np.all(np.abs(a - b) <= TOL[precision] * np.abs(a))
