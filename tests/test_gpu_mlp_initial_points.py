"""The initial live points of an MLP run, shared out over the CTAs of its
cluster: the same points and the same FP32 log L, bit for bit, as one CTA
computes, and a first iteration of tensor-core passes on top of them."""
import numpy as np
import pytest

from paper_2608_28514_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


# N below, at and across the batches (min(32, 2 m + 8) points) of four CTAs
@pytest.mark.parametrize("precision", [1, 2])
@pytest.mark.parametrize("N,m", [(7, 1), (104, 9), (131, 9), (300, 16)])
def test_initial_points_do_not_depend_on_the_cluster(N, m, precision):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2608_28514_gb300 import _native as nat
    p = W.mlp_emulator(1)
    got = []
    for cluster in (1, 2, 4):
        opt = nat.ns_default_options(precision=precision, mlp_cluster=cluster)
        h = nat.ns_create_batch([(p, N, m, 2, 1e-3, 5)], opt)
        nat.ns_step(h, 1)
        s = nat.ns_summary(h, 0)
        assert s["status"] == 0 and s["n_iter"] == 1
        got.append((nat.ns_copy_run_buffer(h, 0, "live_x").reshape(p.d, -1)[:, :N], nat.ns_copy_run_buffer(h, 0, "live_l")[:N]))
        nat.ns_destroy(h)
    x1, l1 = got[0]
    assert np.isfinite(l1).all()
    for x, l in got[1:]:
        # the m replaced points may differ where a comparison was borderline
        same = np.all(x == x1, axis=0)
        assert same.sum() >= N - m
        assert (l[same] == l1[same]).sum() >= N - m
