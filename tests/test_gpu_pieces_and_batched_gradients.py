"""Edges of the scan over the horizon (number, length and remainder of its pieces) and of the gradient kernels that batches
of more than four instances per SM take (one launch; a last CTA that is not full, more instances than are resident)."""
import numpy as np
import pytest
import torch

from oracle import ttc_layer_grad as olg
from paper_2603_09221_b200 import lqr, workloads
from tests import parity_util as pu
from tests import test_gpu_grad as tg
from tests.test_gpu_parity import small_workload
from tests.test_gpu_time_varying import tv_workload

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


# one piece, exactly two, a last piece of one step, of one step less than the others, the next number of squarings
@pytest.mark.parametrize("n", [16, 32])
@pytest.mark.parametrize("H", [7, 8, 9, 11, 31, 32, 33, 128, 131])
def test_pieces_of_the_horizon(n, H):
    w = small_workload(n, n, H, (1, 2, 3), seed=500 + n + H)
    idx = np.arange(6)
    full = pu.run_gpu(w, method=lqr.TTC_SCAN)
    pu.compare(full, pu.run_oracle(w), idx, 1e-4)
    for k in ("K", "P", "x", "u"):
        assert not torch.any(full[k] == 123456.0), "canary left in %s" % k
    first = pu.run_gpu(w, method=lqr.TTC_SCAN, want=("P", "u", "info"), first_only=True)
    pu.compare(first, pu.run_oracle(w, first_only=True), idx, 1e-4, names=("P", "u"))


# one instance more than the threshold (a last CTA that is not full), and more instances than are resident at once
@pytest.mark.parametrize("n,extra", [(16, 1), (16, 2600), (32, 1), (32, 1203)])
def test_gradients_of_batches_that_fill_the_machine(n, extra):
    N = 4 * torch.cuda.get_device_properties(0).multi_processor_count + extra
    w = tv_workload(n, n, 5, (1, 1, N), seed=60 + n + extra)
    g = tg.draw_g(N, n, 3)
    out = tg.run_gpu(w, g)
    assert out["launches"] == 1 and int(out["info"].abs().max()) == 0
    idx = sorted({0, 1, N // 3, N // 2, N - 4, N - 2, N - 1})
    errs = tg.errors(out, tg.run_oracle(w, g, idx=idx), idx=idx)
    assert all(v <= 1e-4 for v in errs.values()), errs
    for k in tg.NAMES:
        assert torch.isfinite(out[k]).all() and not torch.any(out[k] == 123456.0), k


@pytest.mark.parametrize("key,extra,r", [("layer16", 3, 1), ("layer16", 1900, 15), ("layer32", 1, 17), ("layer32", 900, 5)])
def test_layer_gradients_of_batches_that_fill_the_machine(key, extra, r):
    """Numbers of basis matrices that are no multiple of the sixteen a reduction block takes; twice, for the second call
    finds the workspace as the first one left it."""
    N, T = 4 * torch.cuda.get_device_properties(0).multi_processor_count + extra, 4
    w = workloads.make_layer_workload(key, device=DEV, batch=(1, 1, N), seed=70 + extra)
    full = w["r"]
    take = torch.arange(r, device=DEV) % full
    for k in ("s_b", "s_q", "s_qf"):
        w[k] = (w[k][:, take] * (full / r) ** 0.5).contiguous()
    for k in ("B_basis", "Q_basis"):
        w[k] = w[k][take].contiguous()
    n = w["n"]
    gen = torch.Generator(device=DEV)
    gen.manual_seed(5)
    g = torch.randn((N, n), generator=gen, device=DEV)
    s = lqr.LqrSolver(n, n, T, (1, 1, N))
    for _ in range(2):
        grads = {k: torch.full_like(w[k], 777.0) for k in lqr.LAYER_GRAD_KEYS}
        info = torch.full((N,), -5, dtype=torch.int32, device=DEV)
        s.layer_grad(*(w[k] for k in workloads.LAYER_KEYS), T, g, grads, info=info)
    torch.cuda.synchronize()
    s.close()
    assert int(info.abs().max()) == 0
    f64 = lambda t: t.to(torch.float64).cpu().numpy()
    host = {k: f64(w[k]) for k in workloads.LAYER_KEYS}
    total = {"B_basis": 0.0, "Q_basis": 0.0}
    sampled = set(range(0, N, 211)) | {N - 1}
    for i in range(N):
        ref = olg.grad(*(host[k][i] for k in workloads.LAYER_KEYS[:9]), host["B_basis"], host["Q_basis"], T, f64(g[i]))
        for k in total:
            total[k] = total[k] + ref[k]
        if i in sampled:
            for k in lqr.LAYER_GRAD_KEYS[:9]:
                got = f64(grads[k][i])
                assert np.abs(got - ref[k]).max() <= 1e-4 * max(np.abs(ref[k]).max(), 1e-7), (k, i)
    for k in total:
        assert np.abs(f64(grads[k]) - total[k]).max() <= 1e-4 * np.abs(total[k]).max(), k
