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
          (513, 257), (20001, 255), (70, 512), (3001, 513), (5, 1024), (2049, 1025), (4, 2048), (1999, 2047),
          (333, 1024), (700, 2048), (1300, 2049), (610, 3000), (5, 3585), (400, 4096), (399, 4097), (301, 5121),
          (77, 6200), (200, 7169), (310, 8191), (153, 8193), (31, 9300), (305, 10241), (160, 11300), (3, 12288)]


@pytest.mark.parametrize("m,n", SHAPES)
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_value_and_both_gradients(api, m, n, dtype):
    dt = torch.float64 if dtype == "f64" else torch.float32
    A, x = W.quadform_inputs(n, m=m, seed=m + 3 * n)
    if dtype == "f32":
        A, x = f32_round(A), f32_round(x)
    f_ref, g_ref, gA_ref = O.quadform_grad(A, x, fbar=-0.75, want_gA=True)
    # team: FP32 problems of n >= 1024, n % 4 == 0 otherwise offer no gradient w.r.t. A
    team = 0 if n < 1024 or n % 4 else 256 if n <= 2048 else 512
    p = api.QuadForm(torch.tensor(A, dtype=dt, device="cuda"), arith="native", team=team)
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


@pytest.mark.parametrize("team,n", [(32, 50), (128, 50), (128, 1000), (256, 50), (256, 1300), (512, 50),
                                   (512, 2000), (512, 4500)])
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


@pytest.mark.parametrize("m,n", [(1, 1024), (3, 1026), (4, 1536), (5, 1538), (1217, 2046), (1300, 2048), (9001, 1500),
                                 (611, 2050), (700, 2562), (1001, 3074), (613, 3586), (1216, 4096), (609, 4098),
                                 (615, 5122), (700, 6146), (801, 7170), (608, 8192)])
def test_float_pair_rows_paths_agree_bitwise(api, m, n, monkeypatch):
    # float pairs, several rows a step: every width of a thread, ragged steps of four or two
    # rows, one and many CTAs; prepared and per-load split, one launch and two (also taken by
    # grids of up to 64 CTAs), give the same bits
    from paper_2507_13204_gb300 import _lib as L
    A, x = W.quadform_inputs(n, m=m, seed=2 * m + n)
    f_ref, g_ref = O.quadform_grad(A, x, fbar=0.5)
    At, xt = torch.tensor(A, device="cuda"), torch.tensor(x, device="cuda")
    seed = torch.tensor(0.5, dtype=torch.float64, device="cuda")
    out = []
    for coop, budget in ((1, 0), (0, 0), (1, 8)):  # a budget of 8 bytes: no prepared copy
        if coop:
            monkeypatch.delenv("KG_TEST_NO_COOP", raising=False)
        else:
            monkeypatch.setenv("KG_TEST_NO_COOP", "1")
        p = api.QuadForm(At, tape_budget_bytes=budget)
        assert p.config == ("fused", "recompute", "pair")
        f, g = p.grad(xt, seed=seed)
        assert L.kg_last_launch_count() == (1 if coop and m > 256 else 2) or budget and n > 4096
        g2 = torch.full_like(g, 0.25)
        p.grad(xt, gx=g2, seed=seed, accumulate=True)
        fe = p.eval(xt)
        p.sync()
        out.append((f.item(), g.cpu().numpy(), g2.cpu().numpy(), fe.item()))
        p.close()
    f, g, g2, fe = out[0]
    assert rel_scalar(f, f_ref) <= TOL["f64"] and rel_scalar(fe, f_ref) <= TOL["f64"]
    assert rel_l2(g, g_ref) <= TOL["f64"] and np.array_equal(g2, 0.25 + g)
    for o in out[1:]:
        assert o[3] == fe
        if n <= 4096 or o is out[1]:  # (longer rows: the per-load split's gradient is another kernel)
            assert o[0] == f and np.array_equal(o[1], g) and np.array_equal(o[2], g2)


@pytest.mark.parametrize("m,n", [(304, 1024), (1001, 1500), (9001, 2048)])
def test_f32_short_rows_run_several_a_step(api, m, n):
    # FP32, n % 4 == 0, 1024 <= n <= 2048: the streamed kernel's shapes by the several-rows
    # kernel; what the streamed kernel refuses stays refused (misaligned x, a gradient w.r.t. A)
    from paper_2507_13204_gb300 import _lib as L
    A, x = W.quadform_inputs(n, m=m, seed=m + n)
    A, x = f32_round(A), f32_round(x)
    f_ref, g_ref = O.quadform_grad(A, x, fbar=0.5)
    p = api.QuadForm(torch.tensor(A, dtype=torch.float32, device="cuda"))
    xt = torch.tensor(x, dtype=torch.float32, device="cuda")
    seed = torch.tensor(0.5, dtype=torch.float32, device="cuda")
    f, g = p.grad(xt, seed=seed)
    fe = p.eval(xt)
    g2 = p.grad(xt, seed=seed)[1]
    p.sync()
    assert rel_scalar(f.item(), f_ref) <= TOL["f32"] and rel_scalar(fe.item(), f_ref) <= TOL["f32"]
    assert rel_l2(g.cpu().numpy(), g_ref) <= TOL["f32"] and torch.equal(g, g2)
    off = torch.empty(n + 1, dtype=torch.float32, device="cuda")[1:].copy_(xt)
    for call in (lambda: p.grad(off), lambda: p.grad(xt, gx=off), lambda: p.eval(off),
                 lambda: p.grad(xt, gdata=torch.empty(m, n, dtype=torch.float32, device="cuda"))):
        with pytest.raises(L.KGError):
            call()
    p.close()


@pytest.mark.parametrize("fbar", [np.inf, -np.inf])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("m,n", [(9, 40), (611, 100), (3, 300), (611, 300), (613, 1001), (305, 2001), (611, 3001),
                                 (613, 5501), (613, 6501), (305, 8197), (611, 9001)])
def test_infinite_seed_and_ragged_row_group(api, m, n, dtype, fbar):
    # positive A and x: 2 fbar y_i A_ij and 2 fbar y_i x_j are infinities of fbar's sign, and so
    # are their sums.  The rows missing from the last group (of 8, 4 or 2) and the teams past
    # the end must not add infinity times zero
    dt = torch.float64 if dtype == "f64" else torch.float32
    rng = np.random.default_rng(m + n)
    A, x = f32_round(rng.uniform(0.5, 1, (m, n))), f32_round(rng.uniform(0.5, 1, n))
    ybar = 2 * fbar * (A @ x)
    assert (ybar @ A == fbar).all() and (np.outer(ybar, x) == fbar).all()
    p = api.QuadForm(torch.tensor(A, dtype=dt, device="cuda"), arith="native")
    gA = torch.zeros((m, n), dtype=dt, device="cuda")
    f, g = p.grad(torch.tensor(x, dtype=dt, device="cuda"), gdata=gA,
                  seed=torch.tensor(fbar, dtype=dt, device="cuda"))
    p.sync()
    assert rel_scalar(f.item(), O.quadform_value(A, x)) <= TOL[dtype]
    assert bool((g == fbar).all()) and bool((gA == fbar).all())
    p.close()


@pytest.mark.parametrize("m,n", [(401280, 1024), (50160, 6000), (50160, 10242)])
def test_pair_value_of_a_tall_matrix_of_equal_rows(api, m, n):
    # y_i^2 the same for every row: a thread that adds 330 of them (two CTAs an SM and four rows a
    # step, or a CTA an SM and a row a step) keeps their bits only with its accumulator renormalised; in float arithmetic, 1.0e-11
    # without and 2.7e-13 with it
    a = 1.972628813822955
    A = torch.zeros((m, n), dtype=torch.float64, device="cuda")
    A[:, 0] = a
    x = torch.zeros(n, dtype=torch.float64, device="cuda")
    x[0] = 1.0
    p = api.QuadForm(A, tape_budget_bytes=8 << 30)
    assert p.config[2] == "pair"
    f, g = p.grad(x)
    fe = p.eval(x)
    p.sync()
    assert rel_scalar(fe.item(), m * a * a) <= TOL["f64"]
    assert rel_scalar(f.item(), m * a * a) <= TOL["f64"]
    assert rel_scalar(g[0].item(), 2 * m * a * a) <= TOL["f64"]
    p.close()


# more rows than two an SM (the FP64 one-row kernels take fewer), not a whole number of groups,
# in the widths whose other shapes above are short: 13 to 14 and 21 to 28 columns a lane
@pytest.mark.parametrize("m,n", [(611, 3073), (613, 3584), (611, 5500), (613, 6500), (609, 7167)])
def test_wide_rows_in_ragged_groups(api, m, n):
    for dtype in ("f64", "f32"):
        dt = torch.float64 if dtype == "f64" else torch.float32
        rnd = f32_round if dtype == "f32" else (lambda a: a)
        A, x = (rnd(a) for a in W.quadform_inputs(n, m=m, seed=m + n))
        f_ref, g_ref, gA_ref = O.quadform_grad(A, x, fbar=-0.75, want_gA=True)
        # FP32 problems of n % 4 == 0 otherwise offer no gradient w.r.t. A
        p = api.QuadForm(torch.tensor(A, dtype=dt, device="cuda"), arith="native", team=512)
        xt = torch.tensor(x, dtype=dt, device="cuda")
        gA = torch.empty((m, n), dtype=dt, device="cuda")
        f, g = p.grad(xt, gdata=gA, seed=torch.tensor(-0.75, dtype=dt, device="cuda"))
        fe = p.eval(xt)
        p.sync()
        assert rel_scalar(f.item(), f_ref) <= TOL[dtype]
        assert rel_scalar(fe.item(), O.quadform_value(A, x)) <= TOL[dtype]
        assert rel_l2(g.cpu().numpy(), g_ref) <= TOL[dtype]
        assert rel_l2(gA.cpu().numpy(), gA_ref) <= TOL[dtype]
        p.close()


@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("m,n", [(611, 300), (613, 1001), (613, 2001), (611, 3001), (613, 5501)])
def test_infinite_x_and_ragged_row_group_of_several_warps(api, m, n, dtype):
    dt = torch.float64 if dtype == "f64" else torch.float32
    x = torch.ones(n, dtype=dt, device="cuda")
    x[n - 1] = np.inf
    p = api.QuadForm(torch.ones((m, n), dtype=dt, device="cuda"), arith="native")
    f, g = p.grad(x)
    fe = p.eval(x)
    p.sync()
    assert bool((g == np.inf).all())
    if dtype == "f64":  # (FP32: the compensated sum of squares has no infinity)
        assert f.item() == np.inf and fe.item() == np.inf
    p.close()


# few columns: one CTA's rounds end at 128 rows (FP64) and 320 (FP32) of up to 4096 entries in
# all; the forward has a grid of its own
@pytest.mark.parametrize("m,n", [(64, 1), (128, 8), (129, 8), (320, 8), (321, 12), (1000, 3), (4096, 1), (4097, 1),
                                 (150, 16), (8, 512), (4, 700)])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
def test_few_columns(api, m, n, dtype):
    dt = torch.float64 if dtype == "f64" else torch.float32
    A, x = W.quadform_inputs(n, m=m, seed=7 * m + n)
    if dtype == "f32":
        A, x = f32_round(A), f32_round(x)
    f_ref, g_ref = O.quadform_grad(A, x)
    p = api.QuadForm(torch.tensor(A, dtype=dt, device="cuda"), arith="native")
    xt = torch.tensor(x, dtype=dt, device="cuda")
    f, g = p.grad(xt)
    fe = p.eval(xt)
    f2, g2 = p.grad(xt)
    p.sync()
    assert rel_scalar(f.item(), f_ref) <= TOL[dtype] and rel_scalar(fe.item(), f_ref) <= TOL[dtype]
    assert rel_l2(g.cpu().numpy(), g_ref) <= TOL[dtype]
    assert torch.equal(f, f2) and torch.equal(g, g2)
    p.close()


@pytest.mark.parametrize("m,n", [(1, 129), (16, 129), (16, 256), (17, 240), (64, 250), (150, 193), (304, 256),
                                 (305, 255)])
def test_few_rows_of_one_and_two_warps(api, m, n):
    # FP64 rows of 129 to 256 entries, up to two an SM: a team of two warps, one row a step
    A, x = W.quadform_inputs(n, m=m, seed=5 * m + n)
    f_ref, g_ref, gA_ref = O.quadform_grad(A, x, fbar=0.5, want_gA=True)
    p = api.QuadForm(torch.tensor(A, device="cuda"), arith="native")
    xt = torch.tensor(x, device="cuda")
    gA = torch.empty((m, n), dtype=torch.float64, device="cuda")
    f, g = p.grad(xt, gdata=gA, seed=torch.tensor(0.5, dtype=torch.float64, device="cuda"))
    fe = p.eval(xt)
    p.sync()
    assert rel_scalar(f.item(), f_ref) <= TOL["f64"] and rel_scalar(fe.item(), f_ref) <= TOL["f64"]
    assert rel_l2(g.cpu().numpy(), g_ref) <= TOL["f64"]
    assert rel_l2(gA.cpu().numpy(), gA_ref) <= TOL["f64"]
    p.close()
