"""GPU parity: sparse (CSR) ||A x||^2 value and gradients (w.r.t. x and the stored
values), atomic scatter and the atomic-free transpose gather, through the C ABI
vs the CPU oracle."""
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


def _problem(api, A, dtype=torch.float64, **kw):
    dev = "cuda"
    return api.SpQuadForm(torch.tensor(A.rowptr, device=dev), torch.tensor(A.col, device=dev),
                          torch.tensor(A.val, dtype=dtype, device=dev), A.n, **kw)


# (m, n, degree range): ragged rows, empty rows, repeated columns, wide and tall shapes
SHAPES = [(1, 1, (1, 1)), (7, 5, (0, 4)), (300, 200, (0, 9)), (5000, 3000, (8, 24)),
          (1000, 70000, (20, 60)), (40000, 100, (1, 3))]


@pytest.mark.parametrize("m,n,deg", SHAPES)
@pytest.mark.parametrize("strategy", ["atomic", "transpose"])
@pytest.mark.parametrize("arith", ["pair", "native"])
def test_f64_matches_oracle(api, m, n, deg, strategy, arith):
    A, x = W.spquadform_inputs(m, n, d_lo=deg[0], d_hi=deg[1], seed=m + n)
    f_ref, g_ref, gv_ref = O.spquadform_grad(A.rowptr, A.col, A.val, x, fbar=0.5, want_gval=True)
    p = _problem(api, A, strategy=strategy, arith=arith)
    assert p.config[0] == strategy and p.config[2] == arith
    xt = torch.tensor(x, device="cuda")
    gval = torch.empty(A.nnz, dtype=torch.float64, device="cuda")
    f, g = p.grad(xt, gdata=gval, seed=torch.tensor(0.5, dtype=torch.float64, device="cuda"))
    fe = p.eval(xt)
    p.sync()
    assert rel_scalar(f.item(), f_ref) <= TOL["f64"]
    assert rel_scalar(fe.item(), O.spquadform_value(A.rowptr, A.col, A.val, x)) <= TOL["f64"]
    assert rel_l2(g.cpu().numpy(), g_ref) <= TOL["f64"]
    assert rel_l2(gval.cpu().numpy(), gv_ref) <= TOL["f64"]


@pytest.mark.parametrize("strategy", ["atomic", "transpose"])
def test_f32_matches_oracle_on_rounded_inputs(api, strategy):
    A, x = W.spquadform_inputs(20000, 15000, seed=3)
    A.val = f32_round(A.val)
    x = f32_round(x)
    f_ref, g_ref = O.spquadform_grad(A.rowptr, A.col, A.val, x)
    p = _problem(api, A, torch.float32, strategy=strategy)
    f, g = p.grad(torch.tensor(x, dtype=torch.float32, device="cuda"))
    p.sync()
    assert rel_scalar(f.item(), f_ref) <= TOL["f32"]
    assert rel_l2(g.cpu().numpy(), g_ref) <= TOL["f32"]


@pytest.mark.parametrize("strategy", ["atomic", "transpose"])
def test_accumulate_adds_to_both_gradients(api, strategy):
    A, x = W.spquadform_inputs(900, 700, seed=8)
    _, g_ref, gv_ref = O.spquadform_grad(A.rowptr, A.col, A.val, x, want_gval=True)
    p = _problem(api, A, strategy=strategy)
    g = torch.full((A.n,), 1.5, dtype=torch.float64, device="cuda")
    gv = torch.full((A.nnz,), -2.0, dtype=torch.float64, device="cuda")
    p.grad(torch.tensor(x, device="cuda"), gx=g, gdata=gv, accumulate=True)
    p.sync()
    assert rel_l2(g.cpu().numpy() - 1.5, g_ref) <= TOL["f64"]
    assert rel_l2(gv.cpu().numpy() + 2.0, gv_ref) <= TOL["f64"]


def test_transpose_is_bitwise_reproducible_and_close_to_atomic(api):
    A, x = W.spquadform_inputs(30000, 30000, seed=9)
    xt = torch.tensor(x, device="cuda")
    pt = _problem(api, A, strategy="transpose")
    pa = _problem(api, A, strategy="atomic")
    g1 = pt.grad(xt)[1].clone()
    g2 = pt.grad(xt)[1].clone()
    ga = pa.grad(xt)[1]
    torch.cuda.synchronize()
    assert torch.equal(g1, g2)
    assert rel_l2(ga.cpu().numpy(), g1.cpu().numpy()) <= TOL["f64"]


def test_edge_cases(api):
    from paper_2507_13204_gb300 import _lib as L
    dev = "cuda"
    # no stored entries: f = 0, gradient 0
    for strategy in ("atomic", "transpose"):
        p = api.SpQuadForm(torch.zeros(6, dtype=torch.int32, device=dev),
                           torch.zeros(0, dtype=torch.int32, device=dev),
                           torch.zeros(0, dtype=torch.float64, device=dev), 4, strategy=strategy)
        f, g = p.grad(torch.ones(4, dtype=torch.float64, device=dev))
        p.sync()
        assert f.item() == 0.0 and torch.equal(g, torch.zeros(4, dtype=torch.float64, device=dev))
    # one dense row much longer than a team, and one column shared by every row
    rowptr = np.array([0, 3000], np.int32)
    col = np.arange(3000, dtype=np.int32)
    val = np.random.default_rng(1).standard_normal(3000)
    x = np.random.default_rng(2).uniform(-1, 1, 3000)
    A1 = W.CsrMatrix(rowptr, col, val, 1, 3000)
    rowptr2 = np.arange(0, 5001, dtype=np.int32)
    A2 = W.CsrMatrix(rowptr2, np.zeros(5000, np.int32), np.random.default_rng(3).standard_normal(5000),
                     5000, 1)
    for A, xv in ((A1, x), (A2, np.array([0.7]))):
        f_ref, g_ref = O.spquadform_grad(A.rowptr, A.col, A.val, xv)
        for strategy in ("atomic", "transpose"):
            p = _problem(api, A, strategy=strategy)
            f, g = p.grad(torch.tensor(xv, device=dev))
            p.sync()
            assert rel_scalar(f.item(), f_ref) <= TOL["f64"]
            assert rel_l2(g.cpu().numpy(), g_ref) <= TOL["f64"]
    # invalid structures are rejected at create
    bad = [(np.array([0, 2, 1, 3], np.int32), np.array([0, 1, 2], np.int32)),  # decreasing rowptr
           (np.array([0, 1, 3], np.int32), np.array([0, 1, 9], np.int32)),     # column >= n
           (np.array([1, 2, 3], np.int32), np.array([0, 1, 2], np.int32))]     # rowptr[0] != 0
    for rp, cl in bad:
        for strategy in ("atomic", "transpose"):
            with pytest.raises(L.KGError) as ei:
                api.SpQuadForm(torch.tensor(rp, device=dev), torch.tensor(cl, device=dev),
                               torch.ones(cl.shape[0], dtype=torch.float64, device=dev), 4,
                               strategy=strategy)
            assert ei.value.status == L.KG_ERR_BOUNDS
    q = api.SpQuadForm(torch.tensor([0, 1], dtype=torch.int32, device=dev),
                       torch.tensor([0], dtype=torch.int32, device=dev),
                       torch.ones(1, dtype=torch.float64, device=dev), 2)
    assert q.config == ("atomic", "recompute", "pair")
    with pytest.raises(L.KGError) as ei:
        api.SpQuadForm(torch.tensor([0, 1], dtype=torch.int32, device=dev),
                       torch.tensor([0], dtype=torch.int32, device=dev),
                       torch.ones(1, dtype=torch.float64, device=dev), 2, strategy="csr")
    assert ei.value.status == L.KG_ERR_UNSUPPORTED


def test_pair_range_rules(api):
    from paper_2507_13204_gb300 import _lib as L
    A, x = W.spquadform_inputs(2000, 1500, seed=21)
    A.val[17] = 1e-70  # below the pair range: AUTO falls back to native FP64
    p = _problem(api, A)
    assert p.config[2] == "native"
    f, g = p.grad(torch.tensor(x, device="cuda"))
    p.sync()
    assert rel_l2(g.cpu().numpy(), O.spquadform_grad(A.rowptr, A.col, A.val, x)[1]) <= TOL["f64"]
    with pytest.raises(L.KGError) as ei:
        _problem(api, A, arith="pair")
    assert ei.value.status == L.KG_ERR_UNSUPPORTED
    # an x out of range is reported through kg_sync; the next good call is clean
    A.val[17] = 0.5
    q = _problem(api, A, arith="pair")
    xb = x.copy()
    xb[A.col[5]] = 1e300
    q.grad(torch.tensor(xb, device="cuda"))
    with pytest.raises(L.KGError) as ei:
        q.sync()
    assert ei.value.status == L.KG_ERR_RANGE
    q.grad(torch.tensor(x, device="cuda"))
    q.sync()
    # the prepared copy is 8 bytes per stored value; with a smaller budget AUTO stays native
    small = _problem(api, A, tape_budget_bytes=8 * A.nnz - 8)
    assert small.config[2] == "native"


@pytest.mark.parametrize("team", [2, 4, 16, 32])
def test_team_widths(api, team):
    A, x = W.spquadform_inputs(3000, 2500, d_lo=0, d_hi=70, seed=team)
    f_ref, g_ref = O.spquadform_grad(A.rowptr, A.col, A.val, x)
    for strategy in ("atomic", "transpose"):
        p = _problem(api, A, strategy=strategy, team=team)
        f, g = p.grad(torch.tensor(x, device="cuda"))
        p.sync()
        assert rel_scalar(f.item(), f_ref) <= TOL["f64"]
        assert rel_l2(g.cpu().numpy(), g_ref) <= TOL["f64"]


def test_full_size_workload_f64(api):
    A, x = W.spquadform_inputs()  # 2^20 x 2^20, 8..24 entries per row (16.8e6 stored)
    f_ref, g_ref = O.spquadform_grad(A.rowptr, A.col, A.val, x)
    xt = torch.tensor(x, device="cuda")
    for strategy in ("atomic", "transpose"):
        p = _problem(api, A, strategy=strategy)
        f, g = p.grad(xt)
        p.sync()
        assert rel_scalar(f.item(), f_ref) <= TOL["f64"], strategy
        assert rel_l2(g.cpu().numpy(), g_ref) <= TOL["f64"], strategy
        p.close()


def _csr_of_degrees(deg, n, seed):
    rng = np.random.default_rng(seed)
    rowptr = np.concatenate([[0], np.cumsum(deg)]).astype(np.int32)
    nnz = int(rowptr[-1])
    return W.CsrMatrix(rowptr, rng.integers(0, n, nnz).astype(np.int32), rng.standard_normal(nnz), len(deg), n)


# Row blocks: 256 / TW rows, TW the power of two with 2.4 to 4.8 entries a lane; at most 1536
# entries in a block, longer ones by a warp per row
BLOCKS = {
    "capacity": [48] * 32 + [48] * 31 + [49] + [0] * 30 + [3, 97] + [1] * 5,  # 1536, 1537, ragged last block
    "tw1": [3] * 300 + [0] * 7, "tw2": [9] * 200, "tw4": [17] * 131, "tw16": [70] * 33 + [0, 1, 140],
    "tw32": [150] * 19 + [192] * 8 + [1, 0], "row teams": [300, 1, 170],
    "one long row": [2] * 500 + [4000] + [2] * 500,
}


@pytest.mark.parametrize("name", sorted(BLOCKS))
@pytest.mark.parametrize("kind", ["pair", "native", "f32"])
@pytest.mark.parametrize("strategy", ["atomic", "transpose"])
def test_row_blocks(api, name, kind, strategy):
    A = _csr_of_degrees(BLOCKS[name], 211, seed=len(name))
    x = np.random.default_rng(5).uniform(-1, 1, A.n)
    dt = torch.float32 if kind == "f32" else torch.float64
    tol = TOL["f32" if kind == "f32" else "f64"]
    if kind == "f32":
        A.val, x = f32_round(A.val), f32_round(x)
    f_ref, g_ref, gv_ref = O.spquadform_grad(A.rowptr, A.col, A.val, x, fbar=0.5, want_gval=True)
    p = _problem(api, A, dt, strategy=strategy, arith="auto" if kind == "f32" else kind)
    xt = torch.tensor(x, dtype=dt, device="cuda")
    seed = torch.tensor(0.5, dtype=dt, device="cuda")
    gv = torch.full((A.nnz,), 0.25, dtype=dt, device="cuda")
    f, g = p.grad(xt, gdata=gv, seed=seed, accumulate=False)
    f2, g2 = p.grad(xt, gdata=gv, gx=g.clone(), seed=seed, accumulate=True)
    fe = p.eval(xt)
    p.sync()
    for v in (f, f2, fe):
        assert rel_scalar(v.item(), f_ref) <= tol
    assert rel_l2(g.cpu().numpy(), g_ref) <= tol
    assert rel_l2(g2.cpu().numpy(), 2 * g_ref) <= tol
    assert rel_l2(gv.cpu().numpy(), 2 * gv_ref) <= tol
    if strategy == "transpose":
        g3 = p.grad(xt, gdata=gv, seed=seed)[1].clone()
        assert torch.equal(f, f2) and torch.equal(g3, g)
        g4, g5 = p.grad(xt, seed=seed)[1].clone(), p.grad(xt, seed=seed)[1]
        assert torch.equal(g4, g5) and rel_l2(g4.cpu().numpy(), g_ref) <= tol
    p.close()


@pytest.mark.parametrize("strategy", ["atomic", "transpose"])
@pytest.mark.parametrize("name", ["no entries", "tw1", "tw4", "tw16"])
def test_an_x_that_no_entry_reads_has_no_range(api, name, strategy):
    from paper_2507_13204_gb300 import _lib as L
    # column 0 has no entries; the blocks' lanes without an entry must not look at x[0] either
    A = _csr_of_degrees([0] * 40 if name == "no entries" else BLOCKS[name], 211, seed=len(name))
    A.col[A.col == 0] = 1
    x = np.random.default_rng(6).uniform(0.5, 1, A.n)
    f_ref, g_ref, gv_ref = O.spquadform_grad(A.rowptr, A.col, A.val, x, want_gval=True)
    p = _problem(api, A, strategy=strategy, arith="pair")
    for x0 in (1e-30, np.inf):
        x[0] = x0
        gv = torch.zeros(A.nnz, dtype=torch.float64, device="cuda")
        f, g = p.grad(torch.tensor(x, device="cuda"), gdata=gv if A.nnz else None)
        fe = p.eval(torch.tensor(x, device="cuda"))
        p.sync()
        assert rel_scalar(f.item(), f_ref) <= TOL["f64"] and rel_scalar(fe.item(), f_ref) <= TOL["f64"]
        assert rel_l2(g.cpu().numpy(), g_ref) <= TOL["f64"] and rel_l2(gv.cpu().numpy(), gv_ref) <= TOL["f64"]
    if name != "no entries":  # one that an entry reads is refused
        x[0], x[1] = 1.0, 1e-30
        p.grad(torch.tensor(x, device="cuda"))
        with pytest.raises(L.KGError):
            p.sync()
    p.close()


@pytest.mark.parametrize("strategy", ["atomic", "transpose"])
@pytest.mark.parametrize("team", [0, 8])
@pytest.mark.parametrize("dtype", ["f64", "f32"])
@pytest.mark.parametrize("name", ["tw2", "tw4", "tw16", "row teams"])
def test_an_infinite_x_stays_in_its_rows(api, name, dtype, team, strategy):
    # column 0 is in row 0 only, and x[0] is infinite: y_0 is, and the gradient of row 0's
    # columns; lanes without an entry, which load x[0] or y_0, must not spread it
    A = _csr_of_degrees(BLOCKS[name], 3000, seed=3)
    rng = np.random.default_rng(9)
    A.val, x = f32_round(rng.uniform(0.5, 1, A.nnz)), f32_round(rng.uniform(0.5, 1, A.n))
    A.col[A.col == 0] = 1
    A.col[0] = 0
    x[0] = np.inf
    dt = torch.float32 if dtype == "f32" else torch.float64
    rows = np.repeat(np.arange(A.m), np.diff(A.rowptr))
    y = np.zeros(A.m)
    np.add.at(y, rows, A.val * x[A.col])
    ref = np.zeros(A.n)
    np.add.at(ref, A.col, 2 * A.val * y[rows])
    hit = np.isinf(ref)
    assert hit[0] and hit.sum() < A.n // 2 and not np.isnan(ref).any()
    p = _problem(api, A, dt, strategy=strategy, arith="native", team=team)
    g = p.grad(torch.tensor(x, dtype=dt, device="cuda"))[1].cpu().numpy()
    p.sync()
    assert np.array_equal(np.isinf(g), hit)
    assert rel_l2(g[~hit], ref[~hit]) <= TOL[dtype]
    p.close()


@pytest.mark.parametrize("deg", [6, 10, 21, 39, 60, 100])
@pytest.mark.parametrize("kind", ["pair", "native"])
def test_many_blocks_of_fp64_rows(api, deg, kind):
    # more than 20 row blocks an SM: some passes of these row lengths go to the row teams
    A = _csr_of_degrees([deg] * 200000, 5000, seed=deg)
    x = np.random.default_rng(8).uniform(-1, 1, A.n)
    f_ref, g_ref, gv_ref = O.spquadform_grad(A.rowptr, A.col, A.val, x, want_gval=True)
    xt = torch.tensor(x, device="cuda")
    for strategy in ("atomic", "transpose"):
        p = _problem(api, A, strategy=strategy, arith=kind)
        gv = torch.empty(A.nnz, dtype=torch.float64, device="cuda")
        f, g = p.grad(xt, gdata=gv)
        f2, g2 = p.grad(xt)
        fe = p.eval(xt)
        p.sync()
        for v in (f, f2, fe):
            assert rel_scalar(v.item(), f_ref) <= TOL["f64"]
        for v in (g, g2):
            assert rel_l2(v.cpu().numpy(), g_ref) <= TOL["f64"]
        assert rel_l2(gv.cpu().numpy(), gv_ref) <= TOL["f64"]
        p.close()
