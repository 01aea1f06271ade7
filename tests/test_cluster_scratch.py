"""The cluster tree's shared-memory layout (make_carve) and trees whose
eigen-clips fill their work space."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_28514_gb300", "csrc")

# Host code over make_carve.  clip_overrun: the bytes by which the eigen-clips'
# work slots reach past the staged points (into the child bits behind them),
# the largest over N, or past an unstaged run's shared memory; every block's
# warps.  blocks: those that an SM holds of a thread-walker run that does not
# spill (-1: it does).
HOST = r"""
#include "ns_run.cuh"
using namespace nsd;
extern "C" long long clip_overrun(int d, int depth, int n_hi, long long room, int* n_worst, int* n_staged) {
  const int n_nodes = (1 << (depth + 1)) - 1;
  const bool spill = make_carve(d, 1, n_nodes, kMaxDim).base > kRunSmemBudget;
  const size_t per = sizeof(double) * (2 * d * d + d);
  long long worst = -(1LL << 40);
  *n_staged = 0;
  for (int w = 4; w <= 8; ++w) {
    for (int N = 2; N <= n_hi; ++N) {
      const Carve c = make_carve(d, 1, n_nodes, kMaxDim, false, spill, 0, N, (size_t)room, true, w);
      if (!c.staged) continue;
      ++*n_staged;
      const size_t slots = c.work_bytes / per;
      const long long over = (long long)(c.pbuf + slots * per) - (long long)(c.stage + sizeof(float) * (size_t)d * N);
      if (slots < 1 || c.total > (size_t)room) return 1LL << 40;
      if (over > worst) {
        worst = over;
        *n_worst = N;
      }
    }
    const Carve c = make_carve(d, 1, n_nodes, kMaxDim, false, spill, 0, 100, (size_t)room, false, w);
    if (c.work_bytes < per || c.pbuf + c.work_bytes > c.total ||
        c.pbuf + sizeof(float) * w * c.rows * 33 > c.total || c.total > kRunSmemBudget) return 1LL << 41;
  }
  return worst;
}
extern "C" int blocks(int d, int m, int depth, int dmax, int block, int k) {
  const int n_nodes = (1 << (depth + 1)) - 1;
  if (make_carve(d, m, n_nodes, dmax).base > kRunSmemBudget) return -1;
  const size_t t = make_carve(d, m, n_nodes, dmax, false, false, 0, 0, block_room(k), false, block / 32).total;
  const int fit = smem_blocks(t);
  return fit < k ? fit : k;
}
extern "C" long long point_at(int i, int n_pad, int j) {
  const PointIndex<false> ld = n_pad;
  return (long long)(i * ld + j);
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    nvcc = os.environ.get("NVCC", "nvcc")
    if shutil.which(nvcc) is None:
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("carve")
    (d / "carve.cu").write_text(HOST)
    so = str(d / "carve.so")
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "--expt-relaxed-constexpr", "-shared",
                        "-Xcompiler", "-fPIC", "-I", CSRC, str(d / "carve.cu"), "-o", so], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(so)
    lib.clip_overrun.restype = lib.point_at.restype = ctypes.c_longlong
    return lib


@pytest.mark.parametrize("depth", range(1, 7))
def test_clip_slots_end_before_the_child_bits(host, depth):
    n, k = ctypes.c_int(), ctypes.c_int()
    staged = 0
    for d in range(1, 33):
        for room in (227 * 1024 - 3072, 114688, 56320):
            over = host.clip_overrun(d, depth, 2000, ctypes.c_longlong(room), ctypes.byref(n), ctypes.byref(k))
            staged += k.value
            assert over <= 0, (d, depth, room, n.value, over)
    assert staged > 1000


@pytest.mark.parametrize("n_pad", [2**26, 2**26 + 32, 2**30])
def test_points_in_global_memory_are_indexed_in_64_bits(host, n_pad):
    assert host.point_at(31, n_pad, n_pad - 1) == 32 * n_pad - 1


def test_full_batches_of_trees_keep_their_blocks(host):
    """What an SM holds of a batch of thread-walker runs, 128-thread blocks (4 by
    their registers, 2 above 12 dimensions): as many as with the tables that
    the tree of a run needs and the factorisation's work space of 48 KB, by
    which a run's tables are laid out in its arena."""
    for d, m, depth, want in [(2, 100, 1, 4), (5, 100, 1, 4), (5, 100, 3, 4), (5, 100, 4, 4), (10, 100, 1, 3),
                              (10, 100, 2, 3), (10, 100, 3, 2), (8, 64, 3, 3), (12, 128, 2, 2), (16, 100, 1, 2),
                              (20, 128, 1, 2), (3, 30, 6, 4)]:
        dmax = next(c for c in (2, 4, 6, 8, 10, 12, 16, 20) if c >= d)
        assert host.blocks(d, m, depth, dmax, 128, 4 if dmax <= 12 else 2) >= want, (d, m, depth)


def two_modes(d, N):
    """Two Gaussian modes far apart, shuffled."""
    rng = np.random.default_rng([1, d, N])
    x = 0.5 + np.where((np.arange(N) % 2)[:, None] == 0, -0.2, 0.2) + 0.03 * rng.standard_normal((N, d))
    return rng.permutation(x.astype(np.float32))


# d, N, depth with d N not a multiple of 4 and more nodes of at most d members
# (singular covariances, which take the eigen-clip) than work slots.  The
# oracle's partitions and leaves are the same for points moved by 2e-7.
@pytest.mark.gpu
@pytest.mark.parametrize("d,N,depth", [(14, 185, 5), (14, 127, 6), (17, 126, 5), (25, 274, 4), (26, 205, 4)])
def test_tree_with_full_clip_slots_matches_oracle(oracle, d, N, depth):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2608_28514_gb300 import _native as nat
    x = two_modes(d, N)
    n_pad, nn = (N + 31) // 32 * 32, (1 << (depth + 1)) - 1
    live = np.zeros((d, n_pad), np.float32)
    live[:, :N] = x.T
    i32 = dict(dtype=torch.int32, device="cuda")
    o = dict(centres=torch.zeros(nn, d, device="cuda"), chol=torch.zeros(nn, d, d, device="cuda"),
             chol64=torch.zeros(nn, d, d, dtype=torch.float64, device="cuda"), logvol=torch.zeros(nn, device="cuda"),
             count=torch.zeros(nn, **i32), split=torch.zeros(nn, **i32), mask=torch.zeros(nn, **i32),
             cid=torch.full((N,), -1, **i32))
    nat.ns_cluster(N, n_pad, d, torch.from_numpy(live).cuda(), nat.ns_default_options(depth=depth), 3, 0, **o)
    torch.cuda.synchronize()
    g = {k: v.cpu().numpy() for k, v in o.items()}
    want = oracle.cluster(x.astype(np.float64), oracle.opts(d, 1, depth=depth), 3, 0)
    np.testing.assert_array_equal(g["cid"][:12], want["assign"][:12])
    for k, w in (("split", "split"), ("mask", "mask"), ("count", "count"), ("cid", "assign")):
        np.testing.assert_array_equal(g[k], want[w])
    # volumes: as in the parity tests of the tree (nodes with enough members)
    used = (want["count"] > 4 * (d + 1)) & np.isfinite(want["logvol"])
    np.testing.assert_allclose(g["logvol"][used], want["logvol"][used], rtol=1e-4, atol=1e-3)
