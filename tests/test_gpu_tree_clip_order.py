"""Trees with more singular nodes than eigen-clip slots: the factors, leaves and
volumes are the same bits from call to call and in every shape of a run (the
clips share warps differently and the list of nodes is filled in any order)."""
import numpy as np
import pytest

from paper_2608_28514_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def nat():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2608_28514_gb300 import _native
    _native.lib()
    return _native


# d, N, depth: 41 to 113 singular nodes, 2 to 32 lanes each
@pytest.mark.parametrize("d,N,depth", [(14, 127, 6), (14, 185, 5), (25, 274, 4), (32, 100, 2), (3, 90, 6)])
def test_tree_is_the_same_from_call_to_call(nat, d, N, depth):
    rng = np.random.default_rng([2, d, N])
    x = 0.5 + np.where((np.arange(N) % 2)[:, None] == 0, -0.2, 0.2) + 0.03 * rng.standard_normal((N, d))
    n_pad, nn = (N + 31) // 32 * 32, (1 << (depth + 1)) - 1
    live = np.zeros((d, n_pad), np.float32)
    live[:, :N] = x.T
    live = torch.from_numpy(live).cuda()
    i32 = dict(dtype=torch.int32, device="cuda")
    first = None
    for _ in range(8):
        o = dict(centres=torch.zeros(nn, d, device="cuda"), chol=torch.zeros(nn, d, d, device="cuda"),
                 chol64=torch.zeros(nn, d, d, dtype=torch.float64, device="cuda"), logvol=torch.zeros(nn, device="cuda"),
                 count=torch.zeros(nn, **i32), split=torch.zeros(nn, **i32), mask=torch.zeros(nn, **i32),
                 cid=torch.full((N,), -1, **i32))
        nat.ns_cluster(N, n_pad, d, live, nat.ns_default_options(depth=depth), 3, 0, **o)
        first = first or o
        for k, v in o.items():
            assert torch.equal(v.view(torch.uint8), first[k].view(torch.uint8)), k


@pytest.mark.parametrize("d,N,m,depth", [(10, 150, 15, 5), (14, 185, 12, 5), (24, 120, 20, 3)])
def test_every_shape_of_a_run_has_the_same_tree(nat, d, N, m, depth):
    """A run alone (points staged in shared memory), among 24 and among 700 (one
    walker per thread, points in global memory)."""
    p = W.gauss_corr(d, 4)
    opt = nat.ns_default_options(depth=depth, dead_cap=N + 8 * m)
    got = []
    for copies in (1, 24, 700):
        h = nat.ns_create_batch([(p, N, m, 10, 1e-3, 77 + r) for r in range(copies)], opt)
        nat.ns_step(h, 3)
        got.append({k: nat.ns_copy_run_buffer(h, 0, k) for k in ("chol", "live_x", "live_l", "live_cid")})
        nat.ns_destroy(h)
    for other in got[1:]:
        for k, v in got[0].items():
            np.testing.assert_array_equal(v.view(np.int32), other[k].view(np.int32), err_msg=k)
