"""GPU parity for the meta-game solvers (Sec. 4.2 meta-solver, App. C.2
aggregation) against the oracle:

* fictitious play is bit-exact: identical play counts (so identical mixtures)
  and identical fp64 bounds, including tie-heavy integer tables, ragged and
  1 x n shapes, tables held off chip, batches, and the stride-4 read of an
  evaluation output;
* the LP's value is within 1e-9 of the oracle's (scaled by the payoff range)
  and its mixtures form an equilibrium (NashConv <= 1e-8); equilibria need not
  be unique, so the mixtures are checked by that property, not element-wise;
* aggregation is within 1e-12 (relative) of the oracle's matrix products.
"""
import numpy as np
import pytest

from gpu_util import context, need_gpu
from oracle import meta_solver as ms

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = context()
    yield c
    c.close()


def run_fp(ctx, tables, iters, stride=1, raw=None):
    torch = need_gpu()
    G, m, n = tables.shape
    src = raw if raw is not None else tables
    P = torch.from_numpy(np.ascontiguousarray(src)).cuda()
    x = torch.empty((G, m), dtype=torch.float64, device="cuda")
    y = torch.empty((G, n), dtype=torch.float64, device="cuda")
    b = torch.empty((G, 2), dtype=torch.float64, device="cuda")
    ctx.meta_fictitious_play(P, iters, x, y, b, stride=stride)
    ctx.sync()
    return x.cpu().numpy(), y.cpu().numpy(), b.cpu().numpy()


def check_fp_exact(tables, iters, gx, gy, gb):
    for g in range(tables.shape[0]):
        x, y, lo, hi, _, _ = ms.fictitious_play(tables[g], iters)
        assert np.array_equal(gx[g], x), g
        assert np.array_equal(gy[g], y), g
        assert gb[g, 0] == lo and gb[g, 1] == hi, (g, gb[g], lo, hi)


@pytest.mark.parametrize("m,n", [(1, 1), (1, 7), (6, 1), (2, 2), (37, 53), (64, 64), (100, 100)])
@pytest.mark.parametrize("iters", [1, 2, 500])
def test_fp_bit_exact_normal(ctx, m, n, iters):
    rng = np.random.default_rng(1000 * m + n)
    tables = rng.normal(size=(3, m, n))
    check_fp_exact(tables, iters, *run_fp(ctx, tables, iters))


def test_fp_bit_exact_ties(ctx):
    rng = np.random.default_rng(9)
    tables = rng.integers(-2, 3, size=(8, 20, 30)).astype(np.float64)
    tables[0] = 0.0                                  # every play ties
    check_fp_exact(tables, 777, *run_fp(ctx, tables, 777))


def test_fp_bit_exact_off_chip_and_max(ctx):
    rng = np.random.default_rng(4)
    t1 = rng.normal(size=(2, 300, 257))             # 300 x 257 fp64 > 200 KB: read from L2
    check_fp_exact(t1, 300, *run_fp(ctx, t1, 300))
    t2 = rng.normal(size=(1, 1024, 1024))           # the largest supported table
    check_fp_exact(t2, 50, *run_fp(ctx, t2, 50))
    t3 = rng.normal(size=(3, 256, 200))             # 256 rows, one per thread, read from L2
    check_fp_exact(t3, 120, *run_fp(ctx, t3, 120))
    t4 = rng.normal(size=(2, 257, 100))             # 257 rows: two per thread for some
    check_fp_exact(t4, 120, *run_fp(ctx, t4, 120))
    for m, n in ((512, 40), (40, 512), (513, 40)):  # two and three rows per thread
        t5 = rng.normal(size=(1, m, n))
        check_fp_exact(t5, 120, *run_fp(ctx, t5, 120))


def test_fp_many_games(ctx):
    rng = np.random.default_rng(21)
    tables = rng.normal(size=(700, 8, 8))           # more games than CTAs in the grid
    gx, gy, gb = run_fp(ctx, tables, 200)
    for g in range(0, 700, 37):
        x, y, lo, hi, _, _ = ms.fictitious_play(tables[g], 200)
        assert np.array_equal(gx[g], x) and np.array_equal(gy[g], y)
        assert gb[g, 0] == lo and gb[g, 1] == hi


def test_fp_reads_mean_column_of_eval_output(ctx):
    rng = np.random.default_rng(8)
    m, n = 5, 6
    raw = rng.normal(size=(1, m, n, 4))            # [pairs][mean, SE, sum, sumsq] layout
    tables = np.ascontiguousarray(raw[..., 0])
    check_fp_exact(tables, 321, *run_fp(ctx, tables, 321, stride=4, raw=raw))


def run_lp(ctx, tables):
    torch = need_gpu()
    G, m, n = tables.shape
    P = torch.from_numpy(np.ascontiguousarray(tables)).cuda()
    x = torch.empty((G, m), dtype=torch.float64, device="cuda")
    y = torch.empty((G, n), dtype=torch.float64, device="cuda")
    v = torch.empty((G,), dtype=torch.float64, device="cuda")
    ctx.meta_lp_nash(P, x, y, v)
    ctx.sync()
    return x.cpu().numpy(), y.cpu().numpy(), v.cpu().numpy()


def check_lp(tables, gx, gy, gv):
    for g in range(tables.shape[0]):
        A = tables[g]
        scale = max(1.0, float(A.max() - A.min()))
        _, _, v = ms.lp_nash(A)
        assert abs(gv[g] - v) <= 1e-9 * scale, (g, gv[g], v)
        assert gx[g].min() >= -1e-12 and gy[g].min() >= -1e-12
        assert abs(gx[g].sum() - 1) < 1e-9 and abs(gy[g].sum() - 1) < 1e-9
        assert ms.nash_conv(A, gx[g], gy[g]) <= 1e-8 * scale


@pytest.mark.parametrize("m,n", [(1, 1), (1, 5), (4, 1), (2, 2), (5, 5), (16, 20), (64, 64),
                                 (100, 100)])
def test_lp_value_and_equilibrium(ctx, m, n):
    rng = np.random.default_rng(50 + m * n)
    tables = rng.normal(size=(3, m, n))
    check_lp(tables, *run_lp(ctx, tables))


@pytest.mark.parametrize("G,m,n,whole", [(1, 40, 40, 0), (1, 40, 40, 1), (1, 39, 41, 0), (1, 39, 41, 1), (4, 100, 17, 1),
                                         (20, 45, 83, 1), (50, 64, 33, 1), (3, 33, 130, 1), (2, 512, 9, 1),
                                         (1, 300, 290, 0), (1, 300, 290, 1), (40, 300, 200, 1), (70, 200, 150, 1)])
def test_lp_games_over_clusters(ctx, G, m, n, whole):
    """Columns dealt over 8, 4, 2 and 1 CTAs, CTAs with fewer columns or none,
    tableaus on and off chip; the last `whole` tables hold small integers, which tie
    often, the others normal deviates."""
    rng = np.random.default_rng(m * n + G)
    tables = rng.normal(size=(G, m, n))
    if whole:
        tables[-1] = rng.integers(-2, 3, size=(m, n))
    gx, gy, gv = run_lp(ctx, tables)
    some = sorted({0, G // 2, G - 1})
    check_lp(tables[some], gx[some], gy[some], gv[some])


def test_lp_clusters_back_to_back(ctx):
    """One game on a cluster of eight CTAs, launched 40 times in a row: every launch
    starts its clusters anew and gives the same bits."""
    torch = need_gpu()
    rng = np.random.default_rng(5)
    tables = rng.normal(size=(1, 64, 64))
    P = torch.from_numpy(tables).cuda()
    x, y = (torch.zeros((40, 1, 64), dtype=torch.float64, device="cuda") for _ in range(2))
    v = torch.zeros((40, 1), dtype=torch.float64, device="cuda")
    for i in range(40):
        ctx.meta_lp_nash(P, x[i], y[i], v[i])
    ctx.sync()
    check_lp(tables, x[0].cpu().numpy(), y[0].cpu().numpy(), v[0].cpu().numpy())
    assert torch.equal(x, x[:1].expand_as(x)) and torch.equal(y, y[:1].expand_as(y)) and torch.equal(v, v[:1].expand_as(v))


def test_lp_closed_forms_and_degenerate(ctx):
    rps = np.array([[0, -1, 1], [1, 0, -1], [-1, 1, 0]], float)
    two = np.array([[3.0, -1.0], [-2.0, 1.0]])
    tables = np.zeros((4, 3, 3))
    tables[0] = rps
    tables[1, :2, :2] = two
    tables[1, 2, :] = -10.0                          # dominated row
    tables[1, :, 2] = 10.0                           # dominated column
    tables[2] = 0.25                                 # constant game
    tables[3] = np.array([[1, 1, 2], [1, 1, 2], [0, 0, 3]], float)   # ties everywhere
    gx, gy, gv = run_lp(ctx, tables)
    check_lp(tables, gx, gy, gv)
    assert abs(gv[0]) < 1e-12 and np.abs(gx[0] - 1 / 3).max() < 1e-9
    assert abs(gv[1] - (3 * 1 - (-1) * (-2)) / (3 + 1 + 1 + 2)) < 1e-12
    assert abs(gv[2] - 0.25) < 1e-15


@pytest.mark.parametrize("table,x,y", [
    ([[-3, -1, 2], [3, -1, 2], [3, 1, -2]], [0, 1 / 2, 1 / 2], [0, 2 / 3, 1 / 3]),
    ([[3, 1, 2, -3], [3, -3, -1, 1], [-2, 0, 2, -2], [-3, -3, -1, 1]], [1 / 2, 1 / 2, 0, 0], [0, 1 / 2, 0, 1 / 2]),
    ([[2, 3, 0], [2, -2, -3], [-1, -3, 1], [-3, -2, -2], [-2, 3, 0]], [4 / 7, 0, 3 / 7, 0, 0], [0, 1 / 7, 6 / 7]),
    ([[3, 3, 3, 3, 1, -3], [-2, 3, -3, 3, -3, -3], [0, -1, 2, -2, 2, 2], [2, 0, 1, 0, -3, -2], [-2, 0, 2, -1, -2, 0]],
     [2 / 5, 0, 3 / 5, 0, 0], [0, 0, 0, 1 / 2, 0, 1 / 2])])
def test_lp_equal_ratios_tie(ctx, table, x, y):
    """Rows whose ratios are equal rationals tie, and the lowest basic variable leaves:
    the equilibrium is the one that the same rules reach in exact rational arithmetic
    (these games have others)."""
    gx, gy, _ = run_lp(ctx, np.array([table], float))
    assert np.abs(gx[0] - x).max() < 1e-12 and np.abs(gy[0] - y).max() < 1e-12, (gx, gy)


def test_lp_off_chip(ctx):
    rng = np.random.default_rng(77)
    tables = rng.normal(size=(2, 300, 200))          # tableau 301 x 501 fp64 > 200 KB
    check_lp(tables, *run_lp(ctx, tables))


def test_lp_pivot_limit_reports_not_converged(ctx):
    """A game that needs more simplex pivots than the caller's limit raises
    ENOTCONVERGED at the next sync; the flag is cleared once read and the
    context stays usable. Rock-paper-scissors needs at least 3 pivots (its
    optimal basis holds all 3 columns, one enters per pivot); a 1 x 1 game
    needs exactly 1, so a limit of 1 still converges."""
    torch = need_gpu()
    from paper_2106_07551_gb300 import MALIB_ENOTCONVERGED, MalibError
    rps = np.array([[[0, -1, 1], [1, 0, -1], [-1, 1, 0]]], float)
    P = torch.from_numpy(rps).cuda()
    x = torch.empty((1, 3), dtype=torch.float64, device="cuda")
    y = torch.empty((1, 3), dtype=torch.float64, device="cuda")
    v = torch.empty((1,), dtype=torch.float64, device="cuda")
    ctx.meta_lp_nash(P, x, y, v, max_pivots=2)
    with pytest.raises(MalibError) as e:
        ctx.sync()
    assert e.value.code == MALIB_ENOTCONVERGED and "ENOTCONVERGED" in str(e.value)
    ctx.sync()                                       # cleared once reported
    ctx.meta_lp_nash(P, x, y, v, max_pivots=3 * 6)
    ctx.sync()
    check_lp(rps, x.cpu().numpy(), y.cpu().numpy(), v.cpu().numpy())
    one = torch.full((1, 1, 1), 0.5, dtype=torch.float64, device="cuda")
    x1 = torch.empty((1, 1), dtype=torch.float64, device="cuda")
    ctx.meta_lp_nash(one, x1, x1.clone(), v, max_pivots=1)
    ctx.sync()
    assert abs(float(v[0]) - 0.5) < 1e-15
    with pytest.raises(MalibError):
        ctx.meta_lp_nash(P, x, y, v, max_pivots=-1)


def test_aggregate(ctx):
    torch = need_gpu()
    rng = np.random.default_rng(13)
    G, m, n = 4, 33, 65
    tables = rng.normal(size=(G, m, n))
    x = rng.dirichlet(np.ones(m), size=G)
    y = rng.dirichlet(np.ones(n), size=G)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    ay = torch.empty((G, m), dtype=torch.float64, device="cuda")
    xa = torch.empty((G, n), dtype=torch.float64, device="cuda")
    val = torch.empty((G,), dtype=torch.float64, device="cuda")
    ctx.meta_aggregate(d(tables), d(x), d(y), ay, xa, val)
    ctx.sync()
    for g in range(G):
        r_ay, r_xa, r_v = ms.aggregate(tables[g], x[g], y[g])
        s = np.abs(tables[g]).max()
        assert np.abs(ay[g].cpu().numpy() - r_ay).max() <= 1e-12 * s * n
        assert np.abs(xa[g].cpu().numpy() - r_xa).max() <= 1e-12 * s * m
        assert abs(float(val[g]) - r_v) <= 1e-12 * s * (m + n)


@pytest.mark.parametrize("G,m,n", [(3, 1, 1), (5000, 2, 2), (2, 7, 16), (2, 15, 17), (2, 16, 16), (2, 17, 16), (2, 60, 10),
                                   (2, 100, 13), (2, 300, 16), (2, 3, 65), (2, 32, 32), (2, 33, 33), (700, 45, 70),
                                   (2, 64, 64), (2, 70, 70), (2, 20, 256), (2, 5, 257), (1, 3, 1000), (1, 2000, 1)])
def test_aggregate_shapes(ctx, G, m, n):
    """Both sides of the dispatch: tables of up to 256, 1,024, 4,096 and more entries, up to
    16, 256 and more columns, more games than resident blocks; entry 0 of 4. The bound is
    that of fp64 sums of m, n or m n terms in any order."""
    torch = need_gpu()
    rng = np.random.default_rng(m * n)
    raw = rng.normal(size=(G, m, n, 4))
    x, y = rng.dirichlet(np.ones(m), size=G), rng.dirichlet(np.ones(n), size=G)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    ay, xa, val = (torch.full(s, np.nan, dtype=torch.float64, device="cuda") for s in ((G, m), (G, n), (G,)))
    ctx.meta_aggregate(d(raw), d(x), d(y), ay, xa, val, stride=4)
    ctx.sync()
    A, u = raw[..., 0], 2.0 ** -53
    size = [np.einsum(e, *o) for e, o in (("gij,gj->gi", (abs(A), y)), ("gi,gij->gj", (x, abs(A))),
                                          ("gi,gij,gj->g", (x, abs(A), y)))]
    for got, want, s, terms in ((ay, np.einsum("gij,gj->gi", A, y), size[0], n), (xa, np.einsum("gi,gij->gj", x, A), size[1], m),
                                (val, np.einsum("gi,gij,gj->g", x, A, y), size[2], m + n)):
        assert np.all(np.abs(got.cpu().numpy() - want) <= 2 * (terms + 2) * u * s)


def test_errors(ctx):
    torch = need_gpu()
    from paper_2106_07551_gb300 import MalibError
    P = torch.zeros((1, 4, 4), dtype=torch.float64, device="cuda")
    x = torch.empty((1, 4), dtype=torch.float64, device="cuda")
    b = torch.empty((1, 2), dtype=torch.float64, device="cuda")
    with pytest.raises(MalibError):
        ctx.meta_fictitious_play(P, 0, x, x, b)                     # iters < 1
    with pytest.raises(MalibError):
        ctx.meta_fictitious_play(P.cpu(), 5, x, x, b)               # host table
    big = torch.zeros((1, 1025, 2), dtype=torch.float64, device="cuda")
    with pytest.raises(MalibError):
        ctx.meta_fictitious_play(big, 5, torch.empty((1, 1025), dtype=torch.float64, device="cuda"),
                                 torch.empty((1, 2), dtype=torch.float64, device="cuda"), b)
