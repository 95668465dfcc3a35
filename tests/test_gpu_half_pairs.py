"""Range of the pairs of halves in the one-warp kernel: inside it, outside it, and across it in the middle of a horizon.
Every case is compared with the float64 oracle within the float32 bound of the other parity tests."""
import numpy as np
import pytest
import torch

from paper_2603_09221_b200 import lqr
from tests import parity_util as pu
from tests.test_gpu_parity import small_workload
from tests.test_gpu_time_varying import run_both, tv_workload

pytestmark = pytest.mark.gpu
HEADS = 6


def units(n, m):
    """Per head: units of the states (x -> T x), of the controls (u -> D u) and of the cost, all powers of two, so that the
    problem in these units has the same solution in units of its own to the last bit of the inputs."""
    T, D, c = np.ones((HEADS, n)), np.ones((HEADS, m)), np.ones(HEADS)
    c[1], c[2] = 2.0 ** 21, 2.0 ** -17
    D[3, 0] = 2.0 ** 12                                    # column 0 of B and R_00 become small
    T[4, 0], T[4, -1] = 2.0 ** 10, 2.0 ** -6
    T[5, n // 2], D[5, -1], c[5] = 2.0 ** -3, 2.0 ** -5, 2.0 ** 9
    return T, D, c


def in_units(w, T, D, c):
    dev = w["Q"].device
    shape = lambda a, tail: torch.as_tensor(a, dtype=torch.float32, device=dev).reshape((1, HEADS, 1) + tail)
    extra = lambda k: (1,) if k in w.get("tv", ()) else ()  # room for the time axis
    row = lambda a, k: shape(a, extra(k) + (a.shape[1], 1))
    col = lambda a, k: shape(a, extra(k) + (1, a.shape[1]))
    cost = lambda k: shape(c, extra(k) + (1, 1))
    v = dict(w)
    v["A"] = w["A"] * row(T, "A") / col(T, "A")
    v["B"] = w["B"] * row(T, "B") / col(D, "B")
    v["R"] = w["R"] * cost("R") / row(D, "R") / col(D, "R")
    for k in ("Q", "Qf"):
        if k in w:
            v[k] = w[k] * cost(k) / row(T, k) / col(T, k)
    v["x0"] = w["x0"] * shape(T, (T.shape[1],))
    return {k: a.contiguous() if isinstance(a, torch.Tensor) else a for k, a in v.items()}


def back(out, T, D, c, tokens):
    per = lambda a: np.repeat(a, tokens, axis=0)
    T, D, c = per(T), per(D), per(c)
    g = {k: out[k].double().cpu().numpy() for k in ("K", "P", "x", "u")}
    g["K"] = g["K"] * T[:, None, None, :] / D[:, None, :, None]
    g["P"] = g["P"] * T[:, None, None, :] * T[:, None, :, None] / c[:, None, None, None]
    g["x"] = g["x"] / T[:, None]
    g["u"] = g["u"] / D[:, None]
    return dict({k: torch.from_numpy(v) for k, v in g.items()}, info=out["info"])


@pytest.mark.parametrize("n,m", [(9, 9), (16, 16), (16, 5), (17, 20), (24, 24), (32, 32), (33, 7), (40, 40), (58, 41)])
def test_units_time_invariant(n, m):
    w = small_workload(n, m, 7, (1, HEADS, 3), seed=900 + 17 * n + m)
    u = units(n, m)
    pu.compare(back(pu.run_gpu(in_units(w, *u)), *u, 3), pu.run_oracle(w), np.arange(3 * HEADS), 1e-4)


@pytest.mark.parametrize("n,m", [(9, 9), (16, 16), (16, 11), (31, 20), (32, 32)])
@pytest.mark.parametrize("tv", [("A", "B", "Q", "R"), ("B", "R")])
def test_units_time_varying(n, m, tv):
    w = tv_workload(n, m, 6, (1, HEADS, 3), seed=300 + 17 * n + m, tv=tv)
    u = units(n, m)
    out, _ = run_both(in_units(w, *u))
    _, ref = run_both(w)
    pu.compare(back(out, *u, 3), ref, np.arange(3 * HEADS), 1e-4)


@pytest.mark.parametrize("n,m", [(12, 12), (16, 16), (24, 9), (32, 32), (40, 12)])
def test_value_matrix_leaves_the_range(n, m):
    """Open-loop unstable dynamics and expensive controls: P_t grows by a factor of about two a step, past 128 times its
    start within the horizon; every second head stays inside."""
    w = small_workload(n, m, 14, (1, 4, 5), seed=70 + n)
    w["A"][:, ::2] *= 1.6
    w["R"][:, ::2] *= 1e5
    g, ref = pu.run_gpu(w), pu.run_oracle(w)
    top = np.abs(ref["P"]).max(axis=(2, 3))
    assert (top[:5, 0] > 512 * top[:5, -1]).all() and (top[5:10, 0] < 64 * top[5:10, -1]).all()
    pu.compare(g, ref, np.arange(20), 1e-4)


@pytest.mark.parametrize("n", [16, 32])
def test_no_terminal_weight_and_zero_columns(n):
    """P_H = 0, a control without effect, and a step whose A_t is above the range in one head."""
    w = tv_workload(n, n, 8, (1, 3, 4), seed=11 + n)
    w["Qf"].zero_()
    w["B"][:, 1, :, :, :, 2] = 0.0
    w["A"][:, 2, :, 4] *= 14.0
    out, ref = run_both(w)
    pu.compare(out, ref, np.arange(12), 1e-4)
