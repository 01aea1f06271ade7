"""Evaluation counts beyond 32 bits: on a plateau (a Gaussian so wide that every
log L is the same FP32 value) no shrink candidate is ever accepted, so each of
the 256 walkers of the iteration takes s_max of them, 2.2e9 per block of the
run's cluster."""
import numpy as np
import pytest

from paper_2608_28514_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def test_an_iterations_count_is_the_sum_of_its_walkers():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2608_28514_gb300 import _native as nat
    p, N, m, s_max = W.gauss_iso(2, 1e30, -5.0, 5.0), 512, 256, 68_000_000
    h = nat.ns_create_batch([(p, N, m, 1, 1e-3, 5)], nat.ns_default_options(s_max=s_max))
    nat.ns_step(h, 1)
    per = nat.ns_copy_run_buffer(h, 0, "walker_evals").astype(np.int64)
    s = nat.ns_summary(h, 0)
    nat.ns_destroy(h)
    assert per.sum() > 8 * 2**31  # (the first candidates may lie outside the cube, which costs no evaluation)
    assert s["n_evals"] == N + per.sum()
    assert s["n_capped"] == m
