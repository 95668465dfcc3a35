"""Costs, units and couplings at which the matrix products of the one-warp kernel could lose digits or leave their range.
Everything is compared with the float64 oracles."""
import numpy as np
import pytest
import torch

from paper_2603_09221_b200 import lqr
from tests import parity_util as pu
from tests import test_gpu_affine as aff
from tests import test_gpu_grad as grad
from tests.test_gpu_parity import small_workload
from tests.test_gpu_time_varying import run_both, tv_workload

pytestmark = pytest.mark.gpu


def scale_costs(w, e):
    for k in ("Q", "Qf", "R"):
        if k in w:
            w[k] = w[k] * 2.0 ** e
    return w


@pytest.mark.parametrize("e", [-24, -27, -30, -50])
@pytest.mark.parametrize("n,m", [(5, 5), (16, 16), (20, 12), (32, 32)])
def test_small_costs_without_terminal_weight(n, m, e):
    """The value matrix is zero at the end of the horizon and small, not zero, from then on."""
    w = scale_costs(tv_workload(n, m, 6, (1, 2, 4), seed=50 + n), e)
    w["Qf"].zero_()
    out, ref = run_both(w)
    pu.compare(out, ref, np.arange(8), 1e-4)


@pytest.mark.parametrize("n", [16, 32])
def test_small_costs_affine_and_gradients(n):
    w = scale_costs(aff.affine_workload(n, n, 6, (1, 2, 4), seed=70 + n), -30)
    w["r"] = w["r"] * 2.0 ** -30
    w["Qf"].zero_()
    out, ref = aff.run_both(w)
    aff.check(out, ref, False)
    w = scale_costs(tv_workload(n, n, 6, (1, 2, 4), seed=90 + n), -30)
    w["Qf"].zero_()
    g = grad.draw_g(8, n, 3)
    out = grad.run_gpu(w, g)
    errs = grad.errors(out, grad.run_oracle(w, g))
    assert int(out["info"].abs().max()) == 0 and all(v <= 1e-4 for v in errs.values()), errs


@pytest.mark.parametrize("e", [-63, -70, 63])
@pytest.mark.parametrize("n,m", [(9, 9), (16, 16), (32, 32), (40, 12)])
def test_costs_far_from_one_time_invariant(n, m, e):
    w = scale_costs(small_workload(n, m, 6, (1, 2, 4), seed=110 + n), e)
    pu.compare(pu.run_gpu(w), pu.run_oracle(w), np.arange(8), 1e-4)


def test_sixty_four_equal_contributions():
    """Every contraction index contributes 8 * 128 to a row of A'P: 64 * 8 * 128 is above the largest float16.  P_1 =
    1 + 8^2 64^2 R / (R + 64^2) passes through 128 over the heads.  It is what is left of 262144 after a cancellation by 2^11,
    so float32 products (2^-20 each) give it to 2^-9, K (no cancellation) to the usual bound; P_0 cancels once more by the
    same and is only finite."""
    heads = 24
    w = small_workload(64, 1, 2, (1, heads, 1), seed=1)
    w["A"].fill_(8.0)
    w["B"].fill_(1.0)
    w["Q"].fill_(1.0)
    w["R"].copy_(torch.linspace(1.983, 1.987, heads).reshape(w["R"].shape))
    gpu, ref = pu.run_gpu(w, want=("K", "P", "info")), pu.run_oracle(w)
    assert 127.8 < ref["P"][0, 1].max() and ref["P"][-1, 1].max() < 128.2
    assert int(gpu["info"].abs().max()) == 0 and bool(torch.isfinite(gpu["P"]).all())
    assert pu.block_rel_err(gpu["K"][:, 1:].cpu(), ref["K"][:, 1:], 2) <= 1e-4
    assert pu.block_rel_err(gpu["P"][:, 1:].cpu(), ref["P"][:, 1:], 2) <= 2.0 ** -9


@pytest.mark.parametrize("n,m", [(16, 16), (32, 32)])
def test_weights_far_from_the_terminal_weight(n, m):
    w = tv_workload(n, m, 6, (1, 2, 4), seed=130 + n)
    w["Qf"] *= 2.0 ** -58
    w["Q"] *= 2.0 ** 73
    w["R"] *= 2.0 ** 73
    out, ref = run_both(w)
    pu.compare(out, ref, np.arange(8), 1e-4)


@pytest.mark.parametrize("n,m", [(16, 5), (32, 12), (40, 12)])
def test_small_control_weight_of_a_control_without_effect(n, m):
    """R_22 = 2^-70 beside P = 2^60, and column 2 of B is zero: S_22 = R_22, row 2 of K is zero."""
    w = small_workload(n, m, 6, (1, 2, 4), seed=150 + n)
    w["Q"] *= 2.0 ** 59
    w["R"] = torch.diag_embed(torch.full((1, 2, 1, m), 2.0 ** -70, device=w["R"].device)).contiguous()
    w["R"][..., torch.arange(m) != 2, torch.arange(m) != 2] = 2.0 ** 55
    w["B"][..., 2] = 0.0
    pu.compare(pu.run_gpu(w), pu.run_oracle(w), np.arange(8), 1e-4)
