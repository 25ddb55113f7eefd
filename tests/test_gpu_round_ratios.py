"""Grains of round mass ratios: diameters 100:1 and 1000:1 (the grouping threshold psi = 1e-6 and whole
counts 1e-4/psi) and masses 10:1 (the erosion threshold psi = 0.1), as equal grains grow into.  The
decisions hang on the last bit of psi = m_j/m_i there, so the FP64 form takes the rounded quotient, as
the oracle does: rates within 1e-12, events and counts identical although every such pair is a flagged
near tie.  The mixed form settles such pairs in FP64, so its events are the same."""
import numpy as np
import pytest

from paper_2609_35967_gb300 import workloads as W
from test_gpu_parity import _check_channels, _step_both

pytestmark = pytest.mark.gpu


def round_patch(v_frag):
    n = 777
    ins = W.patch_instance(n, K=32, seed=31, v_frag=v_frag)
    rng = np.random.default_rng(8)
    base = 2e-4 * rng.uniform(0.5, 2.0, 12)
    tenth = base * 10.0 ** (1.0 / 3.0)
    # the diameters around the cube root whose mass ratio comes nearest to 1/10
    for k in range(12):
        near = tenth[k] * (1.0 + np.arange(-4, 5) * 2.0**-53)
        tenth[k] = near[np.argmin(np.abs(base[k] ** 3 / near**3 - 0.1))]
    pool = np.concatenate([base, base, 100.0 * base, 1000.0 * base, tenth])
    ins["s"] = rng.choice(pool, n)
    return ins


@pytest.mark.parametrize("v_frag", [1e9, 1e-3])
@pytest.mark.parametrize("precision", [0, 1])
def test_round_ratios_match_oracle(gd, oracle, precision, v_frag):
    ins = round_patch(v_frag)
    sess = gd.Session([ins], K=32, precision=precision)
    P = oracle.params(ins["params"])
    st = oracle.new_state(P)
    ref, got = _step_both(gd, oracle, sess, P, st, ins, ins["s"].copy())
    inst = sess.stats(check=False)["instances"][0]
    sess.close()
    if precision == 0:
        _check_channels(ref, got, 1e-12)
        assert np.abs(got["lam"] / ref["lam"] - 1.0).max() < 1e-12
    assert inst["dt_exe"] == st.dt_exe or precision == 1
    if inst["dt_exe"] == st.dt_exe:
        assert np.array_equal(got["ev_count"], ref["ev_count"])
        assert np.array_equal(got["ev_hash"], ref["ev_hash"])
