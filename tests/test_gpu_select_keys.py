"""Selection over live sets whose keys leave nothing to choose by: equal values,
infinities and NaN (which ranks by its bits, above +infinity).  The oracle
selects over the keys' ranks, which order the same; all outputs are equal."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _keys(l):
    b = l.view(np.uint32)
    return np.where(b & 0x80000000, ~b, b | np.uint32(0x80000000)).astype(np.uint32)


def _live(what, N):
    nan = np.array([0x7FFFFFFF], np.uint32).view(np.float32)[0]  # what the device's arithmetic returns
    if what == "numbers_and_nan":
        l = np.random.default_rng(N).normal(size=N).astype(np.float32)
        l[N // 2] = nan
        return l
    return np.full(N, {"equal": -1.5, "zero": 0.0, "-inf": -np.inf, "inf": np.inf, "nan": nan}[what], np.float32)


@pytest.mark.parametrize("what", ["equal", "zero", "-inf", "inf", "nan", "numbers_and_nan"])
@pytest.mark.parametrize("N,m", [(2, 1), (33, 1), (100, 1), (1537, 1), (5000, 1), (65536, 1), (33, 16), (1537, 77)])
def test_select_without_distinct_keys(oracle, what, N, m):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2608_28514_gb300 import _native as nat
    l = _live(what, N)
    worst = torch.full((1, m), -1, dtype=torch.int32, device="cuda")
    Wv = torch.zeros(1, m, device="cuda")
    seed_slot = torch.full((1, m), -1, dtype=torch.int32, device="cuda")
    nat.ns_select_worst(torch.from_numpy(l.view(np.int32)[None]).cuda().view(torch.float32), m, [17], 3, worst, Wv,
                        seed_slot)
    torch.cuda.synchronize()
    rank = np.unique(_keys(l), return_inverse=True)[1].astype(np.float64)
    w, s = oracle.select(rank, m, 17, 3)
    np.testing.assert_array_equal(worst[0].cpu().numpy(), w)
    np.testing.assert_array_equal(seed_slot[0].cpu().numpy(), s)
    np.testing.assert_array_equal(Wv[0].view(torch.int32).cpu().numpy(), l[w].view(np.int32))
