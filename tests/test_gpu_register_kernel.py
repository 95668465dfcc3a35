"""GPU parity of the one-warp-per-instance kernels (matrices in registers, blocks of eight) at the sizes where their block
structure can go wrong: one short of a block, exactly a block, one past it, the smallest sizes and m > n."""
import numpy as np
import pytest
import torch

from paper_2603_09221_b200 import lqr
from tests import parity_util as pu
from tests.test_gpu_affine import affine_workload, check, run_both
from tests.test_gpu_parity import small_workload

pytestmark = pytest.mark.gpu
SIZES = [(1, 1), (2, 7), (7, 8), (8, 7), (8, 9), (9, 8), (15, 1), (16, 8), (15, 16), (16, 15), (17, 5), (24, 24), (25, 8),
         (31, 32), (32, 16), (20, 30), (33, 7), (40, 16), (39, 24), (33, 40), (41, 9), (48, 32), (47, 48), (49, 3), (57, 24), (64, 16), (55, 64), (64, 63),
         (17, 9), (24, 16), (25, 17), (32, 24), (33, 25), (40, 32), (49, 33), (64, 48)]


@pytest.mark.parametrize("n,m", SIZES)
def test_block_edges_time_invariant(n, m):
    w = small_workload(n, m, 6, (2, 3, 3), seed=40 + 17 * n + m)
    idx = np.arange(18)
    g = pu.run_gpu(w)
    pu.compare(g, pu.run_oracle(w), idx, 1e-4)
    for k in ("K", "P", "x", "u"):
        assert not torch.any(g[k] == 123456.0), "canary left in %s" % k
    f = pu.run_gpu(w, want=("P", "u", "info"), first_only=True)
    pu.compare(f, pu.run_oracle(w, first_only=True), idx, 1e-4, names=("P", "u"))


@pytest.mark.parametrize("n,m", [(1, 2), (8, 9), (9, 8), (15, 16), (17, 31), (32, 24)])
def test_block_edges_time_varying_with_linear_term(n, m):
    w = affine_workload(n, m, 5, (1, 2, 4), seed=90 + 17 * n + m)
    check(*run_both(w), False)
    check(*run_both(w, first_only=True, want=("P", "pvec", "u", "info")), True)


@pytest.mark.parametrize("n,m", [(5, 4), (8, 8), (12, 5), (16, 16), (21, 20), (32, 32), (40, 12)])
def test_odd_strides_and_failed_instances(n, m):
    """Operands whose matrices start at odd element offsets, and an instance whose R is not positive definite at the last
    pivot: reported with that pivot, filled with NaN, its neighbours untouched."""
    w = small_workload(n, m, 4, (1, 1, 6), seed=7 + n)
    for k, shp in (("A", (n, n)), ("B", (n, m)), ("Q", (n, n)), ("R", (m, m))):
        size = shp[0] * shp[1]
        buf = torch.zeros((6, size + 1), device=w[k].device)
        buf[:, :size] = w[k].expand((1, 1, 6) + shp).reshape(6, size)
        w[k] = buf.as_strided((1, 1, 6) + shp, (0, 0, size + 1, shp[1], 1))
    w["R"][0, 0, 4, m - 1, m - 1] = -1e6
    g = pu.run_gpu(w)
    good = np.array([0, 1, 2, 3, 5])
    for k in ("K", "P", "x", "u"):
        assert torch.isnan(g[k][4]).all(), k
    ref = pu.run_oracle(w, idx=good)
    sub = {k: g[k][torch.as_tensor(good, device=g[k].device)] for k in ("K", "P", "x", "u", "info")}
    pu.compare(sub, ref, np.arange(5), 1e-4)
    assert int(g["info"][4]) == 3 * m + m
