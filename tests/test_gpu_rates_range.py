"""FP64 pair rates over the regimes of the turbulent relative speed and past them: a gas without
turbulence (Re^-1/2 infinite), grains of every regime in one patch, and grains so far above or
below the gas disk's that products of their Stokes numbers leave the range of the shared quotient.
Every channel rate within 1e-12 relative of the oracle's, the bar of the interval parity tests.
Past the disk a rate can hang on one difference of two stopping-time terms (no turbulence, no
thermal motion): each side's terms are within 4 roundings, so 16 2^-53 over the relative gap of
the two sizes comes on top."""
import numpy as np
import pytest

from paper_2609_35967_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("alpha", [0.0, 1e-8, 1e-3, 1e-1])
@pytest.mark.parametrize("lo,hi", [(-1.0, 1.0), (-2.0, 6.0), (-12.0, 30.0), (-31.0, -25.0), (28.0, 33.0)])
def test_channel_rates(gd, oracle, alpha, lo, hi):
    n, K = 777, 32
    ins = W.patch_instance(n, K=K, seed=8, alpha=alpha)
    rng = np.random.default_rng(17)
    ins["s"] = ins["s"] * 10.0 ** rng.uniform(lo, hi, n)
    sess = gd.Session([ins], K=K, precision=0)
    nbr, d = sess.build_neighbors(want=True)
    lam, chan = sess.collision_rates(want=True, chan=True)
    sess.close()
    P = oracle.params(ins["params"])
    ref = oracle.rates_subset(P, *[ins[k] for k in ("x", "y", "z", "s", "M")], np.arange(n),
                              nbr.cpu().numpy(), d.cpu().numpy(), chan=True)
    got, r = chan.cpu().numpy(), ref["chan"]
    assert np.isfinite(r).all()
    assert np.array_equal(r == 0.0, got == 0.0)
    si, sj = ins["s"][:, None], ins["s"][nbr.cpu().numpy()]
    gap = np.abs(si - sj) / np.maximum(si, sj)
    tol = 1e-12 + 16 * 2.0**-53 / np.where(gap > 0.0, gap, 1.0)
    assert np.all(np.abs(got - r) <= tol[:, :, None] * r)
    assert np.all(np.abs(lam.cpu().numpy() - ref["lam"]) <= tol.max(axis=1) * ref["lam"])
