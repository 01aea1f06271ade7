"""The lane-group walkers (several lanes and several SMs per run) against the
other shapes of the same run: a run alone takes up to eight lanes per walker on
a cluster of blocks, the same run in a batch that fills the GPU one thread per
walker, and one in between something in between.  Every shape takes the same
FP32 operations in the same order, so all of a run's buffers are equal bit
for bit: the tolerance is zero."""
import numpy as np
import pytest

from paper_2608_28514_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nat():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2608_28514_gb300 import _native
    _native.lib()
    return _native


BUFFERS = ("live_x", "live_l", "live_cid", "new_x", "new_l", "hist_len", "walker_evals", "walker_flags", "chol")


def _state(nat, h, r):
    out = {k: nat.ns_copy_run_buffer(h, r, k) for k in BUFFERS}
    n = out["hist_len"]
    hl = nat.ns_copy_run_buffer(h, r, "hist_l").reshape(len(n), -1)
    hx = nat.ns_copy_run_buffer(h, r, "hist_x").reshape(len(n), hl.shape[1], -1)
    out["hist_l"] = np.concatenate([hl[i, :n[i]] for i in range(len(n))])  # the entries in use
    out["hist_x"] = np.concatenate([hx[i, :n[i]].ravel() for i in range(len(n))])
    s = nat.ns_summary(h, r)
    out["scalars"] = np.array([s[k] for k in ("log_z", "info", "n_dead", "n_evals", "n_relaxed", "n_capped")])
    return out


# family and dimension (both sides of the register classes' edges), N, m (one
# walker, a warp's edge, the most lanes, the largest batch), the caps
CASES = [
    (W.gauss_iso(2, 0.5, -5, 5), 100, 1, {}),
    (W.gauss_corr(1, 3), 64, 31, {}),
    (W.gauss_corr(10, 4), 400, 100, {}),
    (W.gauss_corr(12, 5), 300, 33, dict(e_max=1, s_max=4, t_max=1)),
    (W.gauss_corr(13, 6), 300, 129, dict(s_max=2, t_max=3)),
    (W.rosenbrock(7), 520, 256, dict(e_max=2, s_max=5, t_max=4)),
    (W.mixture(5, 2), 300, 17, dict(depth=2)),
    (W.mixture(17, 2), 200, 70, dict(depth=1, s_max=1)),
    (W.gauss_iso(32, 1.0, -7, 7), 520, 256, {}),
    (W.bimodal(9), 200, 40, dict(bracket=1)),
    (W.shell2d(), 200, 64, dict(correction=3)),
]


@pytest.mark.parametrize("case", range(len(CASES)), ids=lambda i: CASES[i][0].name + f"_m{CASES[i][2]}")
@pytest.mark.parametrize("mapping", [0, 1])
def test_every_shape_of_a_run_is_the_same_run(nat, case, mapping):
    p, N, m, kw = CASES[case]
    if mapping and kw.get("correction"):
        pytest.skip("one mapping is enough here")
    opt = nat.ns_default_options(walker_mapping=mapping, dead_cap=N + 8 * m, **kw)
    got = []
    for copies in (1, 24, 700):
        runs = [(p, N, m, min(5 * p.d, 40), 1e-3, 77 + r) for r in range(copies)]
        h = nat.ns_create_batch(runs, opt)
        nat.ns_step(h, 2)
        nat.ns_step(h, 3)
        got.append((_state(nat, h, 0), _state(nat, h, copies - 1)))
        nat.ns_destroy(h)
    for other in got[1:]:
        for k, v in got[0][0].items():
            np.testing.assert_array_equal(v, other[0][k], err_msg=k)
    if kw.get("s_max") or kw.get("e_max"):
        assert got[0][0]["walker_flags"].any()  # the caps were met
