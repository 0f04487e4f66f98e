"""The pruned FP32 search (rows in locality order, from 16,384 rows on)
against the full scan and the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2603_02402_gb300 import synth
from test_knn_gpu import rsc, run_knn  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _both(rsc, X, k, metric="euclidean"):
    p = run_knn(rsc, X, k, metric=metric, precision="fp32")
    f = run_knn(rsc, X, k, metric=metric, precision="fp32", prune="off")
    return p, f


@pytest.mark.parametrize("n,d,k,comp,metric", [
    (16_384, 50, 15, 30, "euclidean"), (16_385, 50, 15, 30, "cosine"), (16_447, 3, 16, 5, "euclidean"),
    (20_001, 8, 1, 12, "euclidean"), (33_333, 50, 17, 60, "euclidean"), (20_000, 64, 32, 20, "euclidean"),
    (18_000, 63, 30, 20, "cosine"), (40_011, 17, 5, 9, "euclidean"), (30_000, 1, 15, 4, "euclidean"),
    (70_000, 50, 15, 40, "euclidean"),
])
def test_pruned_equals_full_scan(rsc, n, d, k, comp, metric):  # noqa: F811
    # tiles of 64 and 128 rows with ragged ends, both list lengths (k <= 16,
    # k <= 32), component counts around the four-component step; more than one
    # chunk of 512 tiles at 40,011 and 70,000 rows
    X = synth.mixture(n, d, n_comp=comp, seed=n + k)
    (pi, pd), (fi, fd) = _both(rsc, X, k, metric)
    np.testing.assert_array_equal(pd, fd)
    np.testing.assert_array_equal(pi, fi)


def test_unclustered_and_far_from_the_origin(rsc):  # noqa: F811
    # rows that no sphere separates, then a cluster pair with a large offset
    rng = np.random.Generator(np.random.PCG64(5))
    U = rng.uniform(-1, 1, (20_000, 12)).astype(np.float32)
    M = synth.mixture(20_000, 50, n_comp=2, seed=6) + np.float32(1e3)
    for X in (U, M):
        (pi, pd), (fi, fd) = _both(rsc, X, 15)
        np.testing.assert_array_equal(pi, fi)
        np.testing.assert_array_equal(pd, fd)


@pytest.mark.parametrize("case", ["grid", "duplicates", "one point"])
def test_more_ties_than_a_list_holds(rsc, case):  # noqa: F811
    # equal distances beyond the list's length: the lowest ids win, as in the
    # oracle.  Integer coordinates: the squared distances are exact in FP32
    # and in FP64, so ids must agree exactly.
    rng = np.random.Generator(np.random.PCG64(7))
    if case == "grid":      # 24 and 32 neighbours at equal distance
        X = np.stack(np.meshgrid(*[np.arange(12)] * 4), -1).reshape(-1, 4).astype(np.float32)
    elif case == "duplicates":
        X = np.repeat(rng.integers(0, 9, (410, 6)), 50, axis=0).astype(np.float32)
    else:
        X = np.full((17_000, 5), 3, dtype=np.float32)
    X = X[rng.permutation(len(X))]
    gi, gd = run_knn(rsc, X, 15, precision="fp32")
    q = synth.query_sample(len(X), 300, seed=3)
    oi, od, _ = oracle.knn(X, 15, queries=q)
    np.testing.assert_array_equal(gi[q], oi)
    np.testing.assert_allclose(gd[q], od, rtol=1e-6)


def test_cosine_rows_that_are_zero_or_not_numbers(rsc):  # noqa: F811
    X = synth.mixture(18_000, 20, n_comp=10, seed=8)
    X[[5, 9_000, 17_999]] = 0.0
    X[100, 3] = np.nan
    X[200, 4] = np.inf
    (pi, pd), (fi, fd) = _both(rsc, X, 15, "cosine")
    np.testing.assert_array_equal(pi, fi)
    np.testing.assert_array_equal(pd, fd)
    assert pi[5].tolist()[:3] == [5, 9_000, 17_999]


def test_scan_stats_of_the_pruned_search(rsc):  # noqa: F811
    n = 30_000
    X = torch.from_numpy(synth.mixture(n, 50, n_comp=40, seed=1)).cuda()
    for prune in ("auto", "off"):
        ws = torch.empty(rsc.rsc_knn_workspace_size(n, 50, 15, prune=prune), dtype=torch.uint8, device="cuda")
        rsc.rsc_knn(X, 15, workspace=ws, prune=prune)
        scanned, total = rsc.rsc_knn_scan_stats(n, 50, 15, ws, precision="fp32", prune=prune)
        tiles = -(-n // 128)
        assert total == tiles * tiles
        assert scanned == total if prune == "off" else 0 < scanned < 0.3 * total


@pytest.mark.parametrize("n,d,k,metric", [
    (1, 50, 1, "euclidean"), (20, 3, 20, "euclidean"), (64, 50, 15, "euclidean"), (65, 8, 16, "cosine"),
    (129, 64, 17, "euclidean"), (2_700, 50, 15, "euclidean"), (2_701, 50, 32, "cosine"), (5_000, 7, 32, "euclidean"),
    (10_001, 33, 5, "euclidean"), (16_383, 50, 16, "euclidean"),
])
def test_parts_of_small_inputs_equal_one_scan(rsc, n, d, k, metric):  # noqa: F811
    # fewer rows than the ordering pays for: the database in parts, the lists
    # merged within reach of the k-th; explicit splits keep the plain scan
    X = synth.mixture(n, d, n_comp=7, seed=n)
    pi, pd = run_knn(rsc, X, k, metric=metric, precision="fp32")
    fi, fd = run_knn(rsc, X, k, metric=metric, precision="fp32", db_splits=1)
    np.testing.assert_array_equal(pd, fd)
    np.testing.assert_array_equal(pi, fi)


@pytest.mark.parametrize("case", ["grid", "duplicates", "one point"])
def test_ties_of_small_inputs(rsc, case):  # noqa: F811
    rng = np.random.Generator(np.random.PCG64(17))
    if case == "grid":      # 24 and 32 neighbours at equal distance
        X = np.stack(np.meshgrid(*[np.arange(8)] * 4), -1).reshape(-1, 4).astype(np.float32)
    elif case == "duplicates":   # 80 rows at distance zero: more than are scored at once
        X = np.repeat(rng.integers(0, 9, (40, 6)), 80, axis=0).astype(np.float32)
    else:
        X = np.full((3_000, 5), 3, dtype=np.float32)
    X = X[rng.permutation(len(X))]
    for k in (15, 32):
        gi, gd = run_knn(rsc, X, k, precision="fp32")
        oi, od, _ = oracle.knn(X, k)
        np.testing.assert_array_equal(gi, oi)
        np.testing.assert_allclose(gd, od, rtol=1e-6)


@pytest.mark.parametrize("n", [100, 5_000, 20_000])
def test_search_that_gave_up_leaves_no_id_outside_the_rows(rsc, n):  # noqa: F811
    # A wait budget of a few hundred SM clocks makes the search's first wait
    # give up, so its lists keep what the workspace held: here every other
    # entry is an id far past the rows (1.26e9, the bits of 8388608.0f) and
    # the rest, the lists' last ones among them, are empty (-1).  The status
    # word tells, no such id is followed or returned (what else that call
    # returns is unspecified), and the next call is correct.
    X = synth.mixture(n, 50, n_comp=7, seed=n)
    fi, fd = run_knn(rsc, X, 15, precision="fp32", prune="off")
    Xd = torch.from_numpy(X).cuda()
    ws = torch.empty(rsc.rsc_knn_workspace_size(n, 50, 15, precision="fp32") // 4 * 4, dtype=torch.uint8, device="cuda")
    ws.view(torch.int32).fill_(-1)
    ws.view(torch.int32)[::2] = 0x4B000000
    rsc.rsc_set_wait_budget(300)
    try:
        gi, _ = rsc.rsc_knn(Xd, 15, precision="fp32", workspace=ws)
        assert rsc.rsc_workspace_status(ws) == rsc.RSC_ERR_TIMEOUT
    finally:
        rsc.rsc_set_wait_budget(0)
    gi = gi.cpu().numpy()
    assert ((gi >= -1) & (gi < n)).all()
    gi, gd = rsc.rsc_knn(Xd, 15, precision="fp32", workspace=ws)
    assert rsc.rsc_workspace_status(ws) == rsc.RSC_OK
    np.testing.assert_array_equal(gi.cpu().numpy(), fi)
    np.testing.assert_array_equal(gd.cpu().numpy(), fd)


@pytest.mark.parametrize("case,n,k", [
    ("binary", 17_000, 15), ("binary", 20_011, 32), ("binary", 9_001, 16), ("binary", 129, 32),
    ("copies", 30_000, 15), ("copies", 20_000, 32), ("copies", 12_000, 17),
    ("few", 20_000, 15), ("few", 16_400, 32), ("few", 5_000, 15),
    ("line", 40_000, 15), ("line", 20_000, 32), ("line", 9_000, 15),
])
def test_ties_pass_finds_the_k_nearest(rsc, case, n, k):  # noqa: F811
    # rows for the ties pass in most items or in few (their database in parts),
    # with hits that one row has alone or all rows share, both list lengths,
    # with and without the ordering.  Integer coordinates and copies have equal
    # distances in FP32 and FP64 alike, so the ids must agree; the line's
    # distances are those of FP64 to the rounding of two subtractions.
    rng = np.random.Generator(np.random.PCG64(n + k))
    if case == "binary":      # nothing separates these: all tiles are kept
        X = rng.integers(0, 2, (n, 20)).astype(np.float32)
    elif case == "copies":    # 100 groups of 60 copies among clusters
        X = synth.mixture(n, 30, n_comp=20, seed=n)
        X[:6000] = np.repeat(X[:100], 60, axis=0)
        X = X[rng.permutation(n)]
    elif case == "few":       # ten rows as far from all the others, which are one row
        X = rng.standard_normal((n, 50)).astype(np.float32)
        X[: n - 10] = X[0]
        X = X[rng.permutation(n)]
    else:                     # s of rows on a line loses what separates neighbours
        X = rng.uniform(0, 1, (n, 1)).astype(np.float32)
    gi, gd = run_knn(rsc, X, k, precision="fp32")
    q = np.arange(n) if n < 500 else synth.query_sample(n, 300, seed=3)
    if case in ("copies", "few"):   # some of the rows in question
        q = np.unique(np.r_[q, np.argsort(gd.max(1), kind="stable")[[0, -1, -2, -3]]])
    oi, od, _ = oracle.knn(X, k, queries=q)
    np.testing.assert_allclose(gd[q], od, rtol=1e-5, atol=1e-7)
    if case != "line":
        same = gi[q] == oi
        if case == "copies":   # neighbours of a mixture closer than FP32 tells may change places
            same |= np.isclose(od, np.roll(od, 1, 1), rtol=1e-6) | np.isclose(od, np.roll(od, -1, 1), rtol=1e-6)
            zero = od == 0
            assert (gi[q] == oi)[zero].all()
        assert same.all()


@pytest.mark.parametrize("n", [17_000, 4_000])
def test_ties_pass_of_cosine_rows(rsc, n):  # noqa: F811
    # small whole numbers in three components: many rows along one direction
    # and rows of zeros; distances to the rounding of normalised rows
    rng = np.random.Generator(np.random.PCG64(n))
    X = rng.integers(0, 4, (n, 3)).astype(np.float32)
    gi, gd = run_knn(rsc, X, 15, metric="cosine", precision="fp32")
    q = synth.query_sample(n, 300, seed=3)
    _, od, _ = oracle.knn(X, 15, metric=oracle.COSINE, queries=q)
    np.testing.assert_allclose(gd[q], od, rtol=0, atol=1e-6)
    zeros = np.flatnonzero((X == 0).all(1))
    assert (gi[zeros] == zeros[:15]).all()


@pytest.mark.parametrize("n,k,clustered", [
    (20_000, 15, 0), (40_000, 15, 0), (40_000, 32, 0), (150_000, 15, 0), (180_000, 15, 90_000),
])
def test_rows_that_no_sphere_separates(rsc, n, k, clustered):  # noqa: F811
    # every item keeps most tiles: fewer items than a wave of CTAs (all are
    # split), a wave and a few more (these are), several waves, parts longer
    # than a chunk of tiles; and beside as many clustered rows, where more
    # items are put off than the list holds (640)
    rng = np.random.Generator(np.random.PCG64(n + k))
    X = rng.uniform(-1, 1, (n, 12)).astype(np.float32)
    if clustered:
        X[:clustered] = synth.mixture(clustered, 12, n_comp=60, seed=1)
        X = X[rng.permutation(n)]
    (pi, pd), (fi, fd) = _both(rsc, X, k)
    np.testing.assert_array_equal(pi, fi)
    np.testing.assert_array_equal(pd, fd)


@pytest.mark.parametrize("n,strays", [(30_000, 60), (30_000, 900), (100_003, 2_500)])
def test_rows_far_from_every_cluster(rsc, n, strays):  # noqa: F811
    # strays get small leaves of their own: tiles of few rows where these are
    # few, small leaves in common tiles where they would be many
    X = synth.mixture(n, 50, n_comp=30, seed=n)
    rng = np.random.Generator(np.random.PCG64(strays))
    X[rng.permutation(n)[:strays]] = 20 * rng.standard_normal((strays, 50)).astype(np.float32)
    (pi, pd), (fi, fd) = _both(rsc, X, 15)
    np.testing.assert_array_equal(pi, fi)
    np.testing.assert_array_equal(pd, fd)
