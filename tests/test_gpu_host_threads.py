"""Host threads that launch the same kernel with different amounts of shared
memory, each on a stream of its own: every call succeeds and returns what it
returns alone."""
import threading

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


def _together(jobs):
    """Runs the jobs in a thread each; the first exception is raised."""
    errors, go = [], threading.Barrier(len(jobs))

    def body(job):
        try:
            go.wait()
            job()
        except Exception as e:  # noqa: BLE001 (raised below)
            errors.append(e)

    ts = [threading.Thread(target=body, args=(j,)) for j in jobs]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    if errors:
        raise errors[0]


def test_select_of_different_sizes(nat):
    def job(N):
        l = np.random.default_rng(N).normal(size=(1, N)).astype(np.float32)
        want = np.argsort(l[0], kind="stable")[:8]

        def run():
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                ll = torch.from_numpy(l).cuda()
                worst = torch.zeros(1, 8, dtype=torch.int32, device="cuda")
                Wv, seed = torch.zeros(1, 8, device="cuda"), torch.zeros(1, 8, dtype=torch.int32, device="cuda")
                for _ in range(1500):
                    nat.ns_select_worst(ll, 8, [1], 2, worst, Wv, seed, stream=s)
                s.synchronize()
                np.testing.assert_array_equal(worst[0].cpu().numpy(), want)

        return run

    _together([job(N) for N in (13000, 56000, 20000, 40000)])


def test_runs_of_different_sizes(nat):
    def state(N, m, depth, steps, stream=None):
        h = nat.ns_create_batch([(W.gauss_corr(10, 4), N, m, 5, 1e-3, 7)], nat.ns_default_options(depth=depth))
        for _ in range(steps):
            nat.ns_step(h, 1, stream=stream)
        out = nat.ns_copy_run_buffer(h, 0, "live_x")
        nat.ns_destroy(h)
        return out

    sizes = [(100, 10, 0), (900, 90, 3), (300, 30, 1)]
    alone = [state(*s, 40) for s in sizes]

    def job(k):
        def run():
            s = torch.cuda.Stream()
            np.testing.assert_array_equal(state(*sizes[k], 40, s), alone[k])

        return run

    _together([job(k) for k in range(len(sizes))])
