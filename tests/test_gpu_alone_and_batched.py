"""An instance's results do not depend on what else is in the context: alone and in a batch with larger
ones, every sum is formed in the same order, so moments, intervals, diameters and statistics are the
same bit for bit (in both forms; with a larger instance before and behind it)."""
import numpy as np
import pytest

from paper_2609_35967_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(gd, insts, at, precision, groups):
    sess = gd.Session(insts, K=32, precision=precision)
    lo, hi = sess.offsets[at], sess.offsets[at + 1]
    out = []
    for _ in range(3):
        sess.build_neighbors()
        lam, _ = sess.collision_rates(want=groups == 1)    # (a round of groups leaves idle ones' rates)
        A, B = sess.controller_bins(at)
        sess.sample_collisions()
        i = sess.stats(check=False)["instances"][at]
        keys = ("dt_exe", "C", "sum_M", "sum_Mm", "sum_Ms", "events_total")
        out.append([np.array(A), np.array(B), sess.t["s"].cpu().numpy()[lo:hi], np.array([i[k] for k in keys]),
                    np.array(i["spectrum"])])
        if lam is not None:
            out[-1].append(lam.cpu().numpy()[lo:hi])
    sess.close()
    return out


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,groups", [(1500, 1), (20011, 1), (9000, 3)])
def test_alone_equals_batched(gd, precision, n, groups):
    extra = dict(spatial_groups=groups) if groups > 1 else {}
    one = (W.disk_instance(n, seed=6, K=32, sizes=("lognormal", 10.0, 1.0), **extra) if groups > 1
           else W.patch_instance(n, K=32, seed=2))
    if groups == 1:
        one["s"] = one["s"] * 10.0 ** np.random.default_rng(4).uniform(-2.0, 2.0, n)
    big = W.patch_instance(700000, K=32, seed=3)
    alone = _run(gd, [one], 0, precision, groups)
    for insts, at in (([one, big], 0), ([big, one], 1)):
        for a, b in zip(alone, _run(gd, insts, at, precision, groups)):
            for u, v in zip(a, b):
                assert np.array_equal(u, v)
