"""GPU parity of the several-rows-a-step dense kernels (n <= 2048, native arithmetic) at the
edges of their column slots (32 W k), team widths (256, 512, 1024) and row groups (4, 8)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_2507_13204_gb300 import workloads as W
from tests.helpers import TOL, f32_round, rel_l2, rel_scalar

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api(cuda_ok):
    from paper_2507_13204_gb300 import build
    build.build()
    from paper_2507_13204_gb300 import api as A
    return A


# one CTA, the last CTA's sum, a second launch; full and ragged row groups; every team width
SHAPES = [(1, 1), (7, 31), (8, 33), (9, 64), (65, 97), (300, 128), (1000, 129), (40000, 100), (8, 256),
          (513, 257), (20001, 255), (70, 512), (3001, 513), (5, 1024), (2049, 1025), (4, 2048), (1999, 2047)]


@pytest.mark.parametrize("m,n", SHAPES)
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_value_and_both_gradients(api, m, n, dtype):
    dt = torch.float64 if dtype == "f64" else torch.float32
    A, x = W.quadform_inputs(n, m=m, seed=m + 3 * n)
    if dtype == "f32":
        A, x = f32_round(A), f32_round(x)
    f_ref, g_ref, gA_ref = O.quadform_grad(A, x, fbar=-0.75, want_gA=True)
    # team: FP32 rows of n >= 1024, n % 4 == 0 otherwise run the TMA-streamed kernel
    p = api.QuadForm(torch.tensor(A, dtype=dt, device="cuda"), arith="native", team=0 if n < 1024 else 256)
    xt = torch.tensor(x, dtype=dt, device="cuda")
    gA = torch.full((m, n), 0.25, dtype=dt, device="cuda")
    gx = torch.full((n,), 0.5, dtype=dt, device="cuda")
    seed = torch.tensor(-0.75, dtype=dt, device="cuda")
    f, _ = p.grad(xt, gx=gx, gdata=gA, seed=seed, accumulate=True)
    f1, g1 = p.grad(xt, seed=seed)
    f2, g2 = p.grad(xt, seed=seed)
    fe = p.eval(xt)
    p.sync()
    tol = TOL[dtype]
    for v in (f, f1, fe):
        assert rel_scalar(v.item(), f_ref if v is not fe else O.quadform_value(A, x)) <= tol
    assert rel_l2(g1.cpu().numpy(), g_ref) <= tol
    assert torch.equal(f1, f2) and torch.equal(g1, g2)  # fixed summation order
    # onto the prefill: one more rounding of the sum
    assert rel_l2(gx.cpu().numpy(), 0.5 + g_ref) <= tol
    assert rel_l2(gA.cpu().numpy(), 0.25 + gA_ref) <= tol
    p.close()


@pytest.mark.parametrize("team,n", [(32, 50), (128, 50), (128, 1000), (256, 50), (256, 1300)])
@pytest.mark.parametrize("strategy", ["fused", "transpose", "atomic"])
def test_team_widths_and_strategies(api, team, n, strategy):
    A, x = W.quadform_inputs(n, m=203, seed=team + n)
    f_ref, g_ref = O.quadform_grad(A, x)
    p = api.QuadForm(torch.tensor(A, device="cuda"), arith="native", team=team, strategy=strategy)
    f, g = p.grad(torch.tensor(x, device="cuda"))
    p.sync()
    assert rel_scalar(f.item(), f_ref) <= TOL["f64"]
    assert rel_l2(g.cpu().numpy(), g_ref) <= TOL["f64"]
    p.close()


@pytest.mark.parametrize("m,n", [(9, 40), (3, 300), (1, 2000)])
def test_infinite_x_and_ragged_row_group(api, m, n):
    # the empty rows of the last group must not turn an infinite x into NaN
    A = np.ones((m, n))
    x = np.ones(n)
    x[n - 1] = np.inf
    p = api.QuadForm(torch.tensor(A, device="cuda"), arith="native", team=0 if n < 1024 else 256)
    f, g = p.grad(torch.tensor(x, device="cuda"))
    p.sync()
    assert f.item() == np.inf and bool((g == np.inf).all())
    p.close()
