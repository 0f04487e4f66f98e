"""GPU tests of the learned partitioner: training-kernel gradients against the
FP64 oracle, recall of the partitioned search against the exact oracle, and
the gain of the network over nearest-centroid routing with the same parts and
probe budget."""
import numpy as np
import pytest

import oracle
from paper_2603_02402_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rsc():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2603_02402_gb300 import rsc as mod
    mod.lib()
    return mod


def _batch(seed, B, d, P):
    rng = np.random.Generator(np.random.PCG64(seed))
    X = rng.standard_normal((B, d)).astype(np.float32)
    T = rng.uniform(size=(B, P)).astype(np.float32)
    T /= T.sum(axis=1, keepdims=True)
    return X, T


@pytest.mark.parametrize("bf16,rtol", [(False, 2e-4), (True, 1e-2)])
def test_loss_and_gradient_match_oracle(rsc, bf16, rtol):
    d, P, H, B = 12, 16, 24, 37
    part = rsc.Partitioner(d, P, H, bf16_weights=bf16, seed=3)
    params = (np.random.Generator(np.random.PCG64(4)).standard_normal(part.param_count) * 0.3).astype(np.float32)
    part.set_params(params)
    X, T = _batch(5, B, d, P)
    loss, grad = part.loss_grad(torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda())
    grad = grad.cpu().numpy().astype(np.float64)
    ref_loss, ref_grad = oracle.mlp_loss_grad(X, T, params, (d, H, H, P), bf16=bf16)
    assert abs(loss - ref_loss) <= rtol * abs(ref_loss)
    scale = np.abs(ref_grad).max()
    # per-element agreement relative to the gradient's scale
    np.testing.assert_allclose(grad, ref_grad, rtol=0, atol=rtol * scale)
    assert np.dot(grad, ref_grad) / (np.linalg.norm(grad) * np.linalg.norm(ref_grad)) > 1 - rtol


def _recall(gi, oi, gd, od):
    ok = gd <= od[:, -1:] * (1 + 1e-6)
    return float(ok.mean())


def test_partitioned_search_recall_and_gain(rsc):
    # 60,000 anisotropic cells, 64 parts: recall@15 of the partitioned search
    # against the exact oracle for 1, 2 and 4 probed parts, with the network's
    # routing and with the nearest-centroid routing over the same parts (the
    # method without the network, same candidate budget).  The network must
    # beat the centroids at one probe by a clear margin (measured on this
    # workload: 0.850 against 0.818) and never fall behind.
    n, d, k = 60_000, 50, 15
    X = synth.anisotropic(n, d, n_comp=40, seed=7)
    Xd = torch.from_numpy(X).cuda()
    rng = np.random.Generator(np.random.PCG64(8))
    perm = rng.permutation(n)
    train = torch.from_numpy(np.sort(perm[:8000]).astype(np.int32)).cuda()
    queries = np.sort(perm[8000:9000]).astype(np.int32)
    part = rsc.Partitioner(d, n_parts=64, hidden=64, bf16_weights=True, seed=9)
    loss = part.train(Xd, train, k=k, kmeans_iters=8, epochs=8, batch=512, lr=2e-3)
    assert np.isfinite(loss) and loss > 0
    q = torch.from_numpy(queries).cuda()
    oi, od, _ = oracle.knn(X, k, queries=queries)
    res = {}
    for probes in (1, 2, 4):
        for routing in ("network", "centroids"):
            gi, gd = part.knn(Xd, k=k, n_probe=probes, routing=routing, query_rows=q)
            gi, gd = gi.cpu().numpy(), gd.cpu().numpy()
            assert (np.diff(gd, axis=1) >= 0).all()
            # every returned distance is exact for its id
            ex = np.sqrt(((X[queries][:, None, :].astype(np.float64) - X[gi].astype(np.float64)) ** 2).sum(-1))
            np.testing.assert_allclose(gd, ex, rtol=1e-5, atol=1e-6)
            res[(routing, probes)] = _recall(gi, oi, gd, od)
    print("recall@15 by (routing, probes)", res)
    assert res[("network", 1)] >= res[("centroids", 1)] + 0.015
    for probes in (2, 4):
        assert res[("network", probes)] >= res[("centroids", probes)]
    assert res[("network", 4)] >= 0.99
    # more probes never lose a neighbour
    assert res[("network", 1)] <= res[("network", 2)] <= res[("network", 4)]


def test_save_load_roundtrip(rsc, tmp_path):
    part = rsc.Partitioner(10, 16, 16, seed=11)
    p0 = part.get_params()
    path = str(tmp_path / "part.bin")
    part.save(path)
    other = rsc.Partitioner.load(path)
    np.testing.assert_array_equal(other.get_params(), p0)


@pytest.mark.parametrize("n,d,k,probes", [(20_000, 50, 15, 8), (5_003, 33, 16, 8), (9_001, 48, 1, 4), (300, 7, 10, 8),
                                          (40, 50, 16, 8)])
def test_probes_bounded_by_the_first_part_lose_nothing(rsc, n, d, k, probes):
    # with as many probes as parts the search is exact: the bound taken from
    # the first probed part (which may hold fewer than k rows, or none) must
    # not drop a neighbour that lies in another part.  Row starts on 4-, 8-
    # and 16-byte boundaries (d = 33 and 7, 50, 48).  Distances as in the
    # exact search: 1e-5 relative of FP64.
    parts = 8
    X = synth.mixture(n, d, n_comp=12, seed=n)
    Xd = torch.from_numpy(X).cuda()
    part = rsc.Partitioner(d, parts, 32, bf16_weights=True, seed=d)
    part.build_index(Xd)
    rng = np.random.Generator(np.random.PCG64(n + 1))
    queries = rng.integers(0, n, size=min(n, 1500)).astype(np.int32)
    q = torch.from_numpy(queries).cuda()
    oi, od, _ = oracle.knn(X, k, queries=queries.astype(np.int64))
    full_i, full_d = (t.cpu().numpy() for t in part.knn(Xd, k=k, n_probe=8, query_rows=q))
    np.testing.assert_allclose(full_d, od, rtol=1e-5, atol=1e-6)
    # fewer probes: every query's list is a subset of the exact order, never closer
    gi, gd = (t.cpu().numpy() for t in part.knn(Xd, k=k, n_probe=probes, query_rows=q))
    finite = np.isfinite(gd)
    assert (gd[finite] >= od[finite] * (1 - 1e-5) - 1e-6).all()
    assert ((gi >= 0) == finite).all()
    # all rows as queries: the same lists as the sampled rows got
    ai, ad = (t.cpu().numpy() for t in part.knn(Xd, k=k, n_probe=8))
    np.testing.assert_array_equal(ai[queries], full_i)
    np.testing.assert_array_equal(ad[queries], full_d)


def _bf16(a):
    u = np.ascontiguousarray(a, dtype=np.float32).view(np.uint32).astype(np.uint64)
    u = (u + 0x7FFF + ((u >> 16) & 1)) & 0xFFFF0000
    return u.astype(np.uint32).view(np.float32).astype(np.float64)


def _logits(part, X, d, P, H):
    """The network on BF16-rounded operands, sums in FP64."""
    w = part.get_params()
    sizes = [H * d, H, H * H, H, P * H, P]
    W1, b1, W2, b2, W3, b3 = np.split(w, np.cumsum(sizes)[:-1])
    h = np.maximum(_bf16(X) @ _bf16(W1).reshape(H, d).T + b1, 0)
    h = np.maximum(_bf16(h) @ _bf16(W2).reshape(H, H).T + b2, 0)
    return _bf16(h) @ _bf16(W3).reshape(P, H).T + b3


@pytest.mark.parametrize("n,d,P,H", [(20_001, 50, 600, 256), (5_000, 33, 9, 130), (3_000, 61, 256, 8),
                                     (4_000, 20, 1024, 64), (3_000, 50, 257, 300)])
def test_routing_follows_the_network(rsc, n, d, P, H):
    # part counts around the 256-wide accumulators, hidden sizes around the K
    # blocks, H = 300 through the GEMMs.  Each query's list comes from the part
    # its largest logit names (rows whose two largest logits are closer than
    # the network's rounding, 2^-7 of their size, may go either way).
    X = synth.mixture(n, d, n_comp=30, seed=P)
    Xd = torch.from_numpy(X).cuda()
    part = rsc.Partitioner(d, P, H, bf16_weights=True, seed=H)
    part.build_index(Xd)
    z = _logits(part, X, d, P, H)
    order = np.sort(z, axis=1)
    clear = order[:, -1] - order[:, -2] > 2.0 ** -7 * np.abs(z).max(axis=1)
    label = z.argmax(axis=1)
    k = 10
    gi = part.knn(Xd, k=k, n_probe=1)[0].cpu().numpy()
    found = gi >= 0
    near = np.where(found, gi, 0)
    same = (label[near] == label[:, None]) | ~clear[near] | ~clear[:, None] | ~found
    assert clear.mean() > 0.5
    assert same.all()
    size = np.bincount(label[clear], minlength=P)
    assert (found.sum(axis=1)[clear] >= np.minimum(size[label[clear]], k)).all()


@pytest.mark.parametrize("n,P,H", [(100, 9, 8), (20_001, 600, 256)])
def test_routing_that_gave_up_is_recorded_and_the_next_call_recovers(rsc, n, P, H):
    # a wait budget of a few hundred SM clocks makes the routing kernel's first
    # waits give up (three weight blocks in all and one tile of rows, then many
    # of both): the status word tells, and the next calls are those of a
    # partitioner that never saw it
    X = torch.from_numpy(synth.mixture(n, 50, n_comp=7, seed=n)).cuda()
    part, other = (rsc.Partitioner(50, P, H, bf16_weights=True, seed=H) for _ in range(2))
    ws = torch.zeros(part.workspace_size(n, 0, 10, n, 8), dtype=torch.uint8, device="cuda")
    rsc.rsc_set_wait_budget(300)
    try:
        part.build_index(X, workspace=ws)
        assert rsc.rsc_workspace_status(ws) == rsc.RSC_ERR_TIMEOUT
    finally:
        rsc.rsc_set_wait_budget(0)
    for p in (part, other):
        p.build_index(X, workspace=ws)
        assert rsc.rsc_workspace_status(ws) == rsc.RSC_OK
    got, want = (p.knn(X, k=10, n_probe=8, workspace=ws) for p in (part, other))
    assert rsc.rsc_workspace_status(ws) == rsc.RSC_OK
    for a, b in zip(got, want):
        np.testing.assert_array_equal(a.cpu().numpy(), b.cpu().numpy())


@pytest.mark.parametrize("H", [32, 300])
def test_probes_without_a_part_are_left_out(rsc, H):
    # eight parts, some of whose logits are made NaN, -inf or very small by
    # their bias, through the fused routing kernel and (H = 300) the GEMMs.
    # A part with a NaN logit is not probed and nothing is probed twice; one at
    # -inf is probed last.
    n, d, P, k = 5_000, 20, 8, 10
    X = torch.from_numpy(synth.mixture(n, d, n_comp=12, seed=4)).cuda()
    part = rsc.Partitioner(d, P, H, bf16_weights=True, seed=1)
    part.build_index(X)
    params = part.get_params()

    def knn(bias, n_probe):
        w = params.copy()
        w[-P:] += np.asarray(bias, dtype=np.float32)
        part.set_params(w)
        return [t.cpu().numpy() for t in part.knn(X, k=k, n_probe=n_probe)]

    def same(a, b):
        np.testing.assert_array_equal(a[0], b[0])
        np.testing.assert_array_equal(a[1], b[1])

    zero, low = np.zeros(P), -1e6
    last = lambda v: np.r_[np.zeros(P - 4), np.full(4, v)]   # noqa: E731
    four = knn(last(low), 4)
    same(knn(last(np.nan), 8), four)
    for row in four[0]:
        found = row[row >= 0]
        assert len(set(found.tolist())) == len(found)
    same(knn(last(-np.inf), 8), knn(zero, 8))
    same(knn(np.r_[0, np.full(P - 1, -np.inf)], 2), knn(np.r_[0, -1e5, np.full(P - 2, -1e6)], 2))
    same(knn(np.full(P, np.nan), 8), knn(np.r_[0, np.full(P - 1, low)], 1))


def test_training_with_a_row_that_is_no_number(rsc):
    # the row has no nearest centroid: it joins no cluster and is nobody's
    # target, and the centroids of the others stay numbers (with a NaN centroid,
    # or none, eight probes would not reach every part)
    n, d, k = 2_000, 20, 10
    X = synth.mixture(n, d, n_comp=12, seed=9)
    bad = X.copy()
    bad[100, 3] = np.nan
    part = rsc.Partitioner(d, 8, 32, bf16_weights=True, seed=2)
    train = torch.arange(n, dtype=torch.int32, device="cuda")
    part.train(torch.from_numpy(bad).cuda(), train, k=k, kmeans_iters=4, epochs=1, batch=256)
    part.set_params(rsc.Partitioner(d, 8, 32, bf16_weights=True, seed=2).get_params())
    Xd = torch.from_numpy(X).cuda()
    part.build_index(Xd)
    gi, gd = part.knn(Xd, k=k, n_probe=8, routing="centroids")
    oi, od, _ = oracle.knn(X, k)
    np.testing.assert_allclose(gd.cpu().numpy(), od, rtol=1e-5, atol=1e-6)
    assert (gi.cpu().numpy() >= 0).all()


def test_build_index_starts_with_a_clear_status_word(rsc):
    # whatever the workspace held before: a word left there would read as a
    # failure, and a failure would not be recorded over it
    X = torch.from_numpy(synth.mixture(2_000, 20, n_comp=5, seed=1)).cuda()
    part = rsc.Partitioner(20, 16, 32, bf16_weights=True, seed=1)
    ws = torch.full((part.workspace_size(2_000, 0, 10, 2_000, 8),), 7, dtype=torch.uint8, device="cuda")
    part.build_index(X, workspace=ws)
    assert rsc.rsc_workspace_status(ws) == rsc.RSC_OK
    ws.fill_(7)
    rsc.rsc_set_wait_budget(300)
    try:
        part.build_index(X, workspace=ws)
        assert rsc.rsc_workspace_status(ws) == rsc.RSC_ERR_TIMEOUT
    finally:
        rsc.rsc_set_wait_budget(0)
