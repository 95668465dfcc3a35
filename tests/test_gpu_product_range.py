"""Costs, units and couplings at which the matrix products of the one-warp kernel could lose digits or leave their range.
Everything is compared with the float64 oracles."""
import numpy as np
import pytest
import torch

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


def entrywise(got, ref, floor=1e-7):
    """Largest relative error of the single entries above `floor` of the largest of their block."""
    got, ref = got.double().cpu().numpy(), np.asarray(ref)
    big = np.abs(ref) > floor * np.abs(ref).max(axis=(-2, -1), keepdims=True)
    return float((np.abs(got - ref)[big] / np.abs(ref)[big]).max())


def systems(n, m, seed, eps):
    """Weakly coupled: A = 0.9 I + eps G, B = [I + eps G], Q = I + eps (G + G'), R = I."""
    w = small_workload(n, m, 8, (1, 2, 4), seed=seed)
    g = torch.Generator(device="cuda:0")
    g.manual_seed(seed)
    rn = lambda *shape: torch.randn(shape, generator=g, device="cuda:0")
    eye = torch.eye(n, device="cuda:0")
    q = rn(1, 2, 4, n, n)
    w["A"] = (0.9 * eye + eps * rn(1, 2, 1, n, n)).contiguous()
    w["B"] = (eye[:, :m] + eps * rn(1, 2, 1, n, m)).contiguous()
    w["Q"] = (eye + eps * (q + q.transpose(-1, -2))).contiguous()
    w["R"] = torch.eye(m, device="cuda:0").expand(1, 2, 1, m, m).contiguous()
    return w


def coupling_error(got, ref):
    """Largest error of the off-diagonal entries, relative to the largest of them in their block."""
    got, ref = got.double().cpu().numpy(), np.asarray(ref)
    off = ~np.eye(ref.shape[-2], ref.shape[-1], dtype=bool)
    return float((np.abs(got - ref)[..., off].max(axis=-1) / np.abs(ref)[..., off].max(axis=-1)).max())


# An operand is represented to 2^-21 of each element, an off-diagonal entry is the sum of a few products of one coupling and
# one number of order one, over eight steps: some ten roundings of 2^-21, 5e-6.
@pytest.mark.parametrize("eps", [1e-2, 1e-3, 1e-4, 1e-5, 1e-6])
@pytest.mark.parametrize("n,m", [(16, 16), (24, 24), (32, 20), (40, 12)])
def test_weak_couplings_keep_their_digits(n, m, eps):
    w = systems(n, m, 7 * n, eps)
    gpu, ref = pu.run_gpu(w, want=("K", "P", "info")), pu.run_oracle(w)
    errs = coupling_error(gpu["K"], ref["K"]), coupling_error(gpu["P"], ref["P"])
    assert max(errs) <= 1e-5, errs


@pytest.mark.parametrize("n", [16, 32])
def test_neighbours_of_a_chain_keep_their_digits(n):
    w = systems(n, n, 3, 0.0)
    w["A"] += 0.02 * (torch.diag(torch.ones(n - 1), 1) + torch.diag(torch.ones(n - 1), -1)).to(w["A"].device)
    gpu, ref = pu.run_gpu(w, want=("K", "P", "info")), pu.run_oracle(w)
    errs = entrywise(gpu["K"], ref["K"]), entrywise(gpu["P"], ref["P"])
    assert max(errs) <= 1e-5, errs


@pytest.mark.parametrize("n", [16, 24, 32])
def test_small_products_of_operands_of_ordinary_size(n):
    """B'P is 2^-8 of the largest elements throughout and R small: an error of B'P reaches the gains undiminished.  Single
    float32 roundings of B'P give 4e-7 in K."""
    w = small_workload(n, n, 12, (1, 2, 4), seed=n)
    g = torch.Generator(device="cuda:0")
    g.manual_seed(n)
    u = lambda *shape: torch.rand(shape, generator=g, device="cuda:0")
    d = 0.063 + 0.004 * u(1, 2, 4, n)
    d[..., 0] = 1.0
    w["Q"] = torch.diag_embed(d).contiguous()
    w["A"] = (w["A"] * 0.01 + 0.05 * torch.eye(n, device="cuda:0")).contiguous()
    w["B"] = torch.diag_embed(0.063 + 0.012 * u(1, 2, 1, n)).contiguous()
    w["R"] = (1e-6 * torch.eye(n, device="cuda:0")).expand(1, 2, 1, n, n).contiguous()
    gpu, ref = pu.run_gpu(w, want=("K", "P", "info")), pu.run_oracle(w)
    pu.compare(gpu, ref, np.arange(8), 5e-6, names=("K", "P"))


def scaled(x, top):
    """x times the power of two that brings `top` into [2^14, 2^15)."""
    return np.ldexp(x, 15 - np.frexp(top)[1])


def operand_fits(M):
    """Conditions of the one-warp kernel for A and B on pairs of halves (riccati_frag.cuh), restated: M is one matrix."""
    a = scaled(np.abs(M.T), np.abs(M).max())
    rows = a.sum(axis=1)
    return a.min() >= 2.0 ** -15 and rows.min() >= 2.0 ** -5 * 2.0 ** np.frexp(rows.max())[1]


def small_elements(P):
    """Elements of a value matrix below the limit, after scaling."""
    return int((scaled(np.abs(P), np.diagonal(P).max()) < 2.0 ** -9).sum())


# Ten roundings of 2^-21 in a step, over five steps (which damp them) and amplified by a few in S: 2e-5 of the largest entry of a
# block, a fifth of the bound of the other parity tests.
EDGE_TOL = 2e-5


def edge_workload(n, m, H=5):
    w = small_workload(n, m, H, (1, 6, 3), seed=200 + n + m)
    for k in ("A", "B"):                                   # no element that is small by accident
        w[k] = (w[k] + 0.02 * torch.where(w[k] < 0, -1.0, 1.0)).contiguous()
    return w


@pytest.mark.parametrize("n,m", [(17, 17), (24, 20), (32, 32), (33, 12), (40, 40), (56, 9)])
def test_operands_at_their_limits(n, m):
    """Elements and rows of A' and B' just inside the range of the halves and just outside, one head each."""
    w = edge_workload(n, m)
    A, B = w["A"][0, :, 0], w["B"][0, :, 0]
    two = lambda e: 2.0 ** e
    A[1, 1, 2] = two(np.frexp(float(A[1].abs().max()))[1] - 1 - 28)            # 2^-14 after scaling
    A[2, 1, 2] = two(np.frexp(float(A[2].abs().max()))[1] - 1 - 30)            # 2^-16
    B[3, :, 0] *= two(-3)
    B[4, :, 0] *= two(-9)
    B[5, 3, m - 1] = 0.0
    fits = [operand_fits(A[h].double().cpu().numpy()) and operand_fits(B[h].double().cpu().numpy()) for h in range(6)]
    assert fits == [True, True, False, True, False, False]
    gpu, ref = pu.run_gpu(w, want=("K", "P", "info")), pu.run_oracle(w)
    pu.compare(gpu, ref, np.arange(18), EDGE_TOL, names=("K", "P"))
    rows = lambda a: np.moveaxis(np.asarray(a), -2, 0)     # every control by itself: row j of K is as large as 1 / |B_j|
    assert max(pu.block_rel_err(g[..., None, :], r[..., None, :], 2) for g, r in zip(rows(gpu["K"].cpu()), rows(ref["K"]))) <= 1e-4


@pytest.mark.parametrize("n", [17, 24, 32, 40])
def test_value_matrices_at_their_limits(n):
    """Q (and so P at the end of the horizon) with no, one, two pairs of small elements, diagonal, with a state of other
    units, and with a factor of 2^40: what the last steps run in changes, the results do not."""
    w = edge_workload(n, n)
    Q = w["Q"][0]
    for h, pairs in ((1, 1), (2, 2)):
        for i in range(pairs):
            Q[h, :, i, i + 3] = Q[h, :, i + 3, i] = 2.0 ** -26
    Q[3] = torch.diag_embed(torch.diagonal(Q[3], dim1=-2, dim2=-1))
    Q[4, :, 5, :] *= 2.0 ** -14
    Q[4, :, :, 5] *= 2.0 ** -14
    Q[5] *= 2.0 ** 40
    w["R"][0, 5] *= 2.0 ** 40
    small = [small_elements(Q[h, 0].double().cpu().numpy()) for h in range(6)]
    assert small[1:4] == [2, 4, n * (n - 1)] and small[4] >= 1 and small[5] == small[0] == 0
    gpu, ref = pu.run_gpu(w, want=("K", "P", "info")), pu.run_oracle(w)
    pu.compare(gpu, ref, np.arange(18), EDGE_TOL, names=("K", "P"))


@pytest.mark.parametrize("n,m", [(17, 17), (32, 32), (20, 31)])
@pytest.mark.parametrize("tv", [("A", "B", "Q", "R"), ("A",), ("B",), ("Q",)])
def test_time_varying_operands_enter_and_leave_the_range(n, m, tv):
    """Steps whose A_t or B_t is out of range between steps inside, with operands that change and operands that stay."""
    w = tv_workload(n, m, 9, (1, 3, 4), seed=300 + n, tv=tv)
    if "A" in tv:
        w["A"][:, 1, :, 2, 0, 1] = w["A"][:, 1, :, 6, 3, 3] = 0.0
    if "B" in tv:
        w["B"][:, 2, :, 4, :, 1] *= 2.0 ** -10
        w["B"][:, 1, :, 7] = 0.0
    if "Q" in tv:
        w["Q"][:, 0, :, 5] = torch.diag_embed(torch.diagonal(w["Q"][:, 0, :, 5], dim1=-2, dim2=-1))
    out, ref = run_both(w, want=("K", "P", "info"))
    pu.compare(out, ref, np.arange(12), EDGE_TOL, names=("K", "P"))
