"""Batched persistent path: every matrix against the FP64 oracle (FP32 tolerance 5e-6 N)."""
import numpy as np
import pytest

import oracle
from paper_2608_21227_gb300 import inputs
from _util import err_rel, to_device_colmajor

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nla():
    from paper_2608_21227_gb300 import nla as _nla

    _nla.lib()
    return _nla


def make_batch(nla, mats):
    return nla.Batch([to_device_colmajor(A, torch.float32) for A in mats])


def check(batch_S, info, mats, tol_scale=5e-6):
    torch.cuda.synchronize()
    assert np.all(info.cpu().numpy()[: len(mats)] == 0)
    for A, S in zip(mats, batch_S):
        ref = oracle.svdvals(A.astype(np.float64))
        assert err_rel(S.cpu().numpy(), ref) <= tol_scale * max(A.shape), A.shape


def test_uneven_shapes_vs_oracle(nla):
    ms, ns = inputs.batch_shapes(300, seed=33)
    mats = [inputs.gaussian(int(m), int(n), [33, i], dtype=np.float32) for i, (m, n) in enumerate(zip(ms, ns))]
    # every fifth matrix is handed over wide (m < n)
    mats = [A.T.copy() if i % 5 == 0 else A for i, A in enumerate(mats)]
    b = make_batch(nla, mats)
    S, info = nla.gesvd_vals_batched(b)
    check(S, info, mats)


def test_tiny_and_degenerate(nla):
    g = np.random.default_rng(5)
    mats = [g.standard_normal((1, 1)), g.standard_normal((1, 6)), g.standard_normal((6, 1)), np.zeros((8, 8)),
            np.outer(np.arange(1.0, 11.0), np.ones(5)), g.standard_normal((17, 16)), g.standard_normal((256, 256)),
            g.standard_normal((1024, 256))]
    mats = [A.astype(np.float32) for A in mats]
    b = make_batch(nla, mats)
    S, info = nla.gesvd_vals_batched(b)
    torch.cuda.synchronize()
    assert np.all(info.cpu().numpy() == 0)
    for A, s in zip(mats, S):
        ref = oracle.svdvals(A.astype(np.float64))
        assert np.max(np.abs(s.cpu().numpy() - ref)) <= 5e-6 * max(A.shape) * max(ref[0], 1e-30) + 1e-30


def test_ten_thousand_matrices_sampled(nla):
    # the batched workload: 10,000 FP32 matrices, n ~ U{8..256}, m/n ~ U[1, 4], N(0, 1)
    ms, ns = inputs.batch_shapes(10000, seed=3)
    mats = [inputs.gaussian(int(m), int(n), [3, i], dtype=np.float32) for i, (m, n) in enumerate(zip(ms, ns))]
    b = make_batch(nla, mats)
    S, info = nla.gesvd_vals_batched(b)
    torch.cuda.synchronize()
    assert np.all(info.cpu().numpy() == 0)
    sample = np.random.default_rng(0).choice(10000, size=60, replace=False)
    for i in sample:
        ref = oracle.svdvals(mats[i].astype(np.float64))
        assert err_rel(S[i].cpu().numpy(), ref) <= 5e-6 * max(mats[i].shape)


def test_graph_capture_replay(nla):
    # the whole batched call (prep + persistent kernel) is captured once and replayed;
    # work is handed out dynamically, so replays agree with the direct call to rounding
    ms, ns = inputs.batch_shapes(200, seed=7)
    mats = [inputs.gaussian(int(m), int(n), [7, i], dtype=np.float32) for i, (m, n) in enumerate(zip(ms, ns))]
    b = make_batch(nla, mats)
    S0, _ = nla.gesvd_vals_batched(b)
    torch.cuda.synchronize()
    first = [s.clone() for s in S0]
    for s in b.S:
        s.fill_(float("nan"))
    st = torch.cuda.Stream()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        with torch.cuda.graph(g, stream=st):
            nla.gesvd_vals_batched(b, stream=st)
    for _ in range(2):
        g.replay()
        torch.cuda.synchronize()
        assert np.all(b.info.cpu().numpy() == 0)
        for A, a, s in zip(mats, first, b.S):
            sv = s.cpu().numpy().astype(np.float64)
            assert np.all(np.isfinite(sv))
            assert err_rel(sv, a.cpu().numpy().astype(np.float64)) <= 5e-6 * max(A.shape)
    check(b.S, b.info, mats[:40])


def test_unsorted_batch_over_the_sort_limit(nla):
    # above 16,384 matrices the batch is not sorted: the persistent kernel then also takes
    # the matrices too large for shared memory (global scratch); every 1000th is one
    g = np.random.default_rng(11)
    count = 16400
    mats = []
    for i in range(count):
        if i % 1000 == 500:
            mats.append(g.standard_normal((300, 200)).astype(np.float32))  # 60,000 elements
        else:
            n = int(g.integers(2, 9))
            mats.append(g.standard_normal((n + int(g.integers(0, 5)), n)).astype(np.float32))
    b = make_batch(nla, mats)
    S, info = nla.gesvd_vals_batched(b)
    torch.cuda.synchronize()
    assert np.all(info.cpu().numpy() == 0)
    check_ids = [i for i in range(count) if i % 1000 == 500] + list(range(0, count, 997))
    for i in check_ids:
        ref = oracle.svdvals(mats[i].astype(np.float64))
        assert err_rel(S[i].cpu().numpy(), ref) <= 5e-6 * max(mats[i].shape), (i, mats[i].shape)


@pytest.mark.parametrize("groups", [None, 32, 128, 256])
def test_class_and_chunk_edges(nla, groups, tmp_path):
    # column counts around the five classes, rows around the register tiles and the chunks of the QR
    # reduction, wide matrices, leading dimensions beyond the rows; the table's least threads per matrix
    from paper_2608_21227_gb300 import kt

    if groups is None:
        kt.load_config(None)
    else:
        path = tmp_path / "t.kt"
        for b in range(5):
            kt.write_table(path, 2, b, 0, nla.F32, 0, (groups, 0, 0, 0, 0), 1.0)
        kt.load_config(path)
    try:
        g = np.random.default_rng(77)
        shapes = [(n, n) for n in (1, 2, 3, 31, 32, 33, 63, 64, 65, 127, 128, 129, 191, 192, 193, 255, 256)]
        shapes += [(65, 32), (129, 32), (64, 33), (65, 64), (129, 64), (257, 60), (129, 100), (257, 128), (513, 77),
                   (193, 150), (385, 192), (577, 130), (257, 200), (385, 256), (1024, 256), (3000, 17), (2000, 1)]
        mats, dev = [], []
        for k, (m, n) in enumerate(shapes):
            A = g.standard_normal((m, n)).astype(np.float32)
            if k % 4 == 1:
                A = (A * 1e-12).astype(np.float32)
            if k % 3 == 2:
                A = np.ascontiguousarray(A.T)  # wide
            pad = 3 if k % 2 else 0
            t = torch.zeros(A.shape[1], A.shape[0] + pad, device="cuda")
            t[:, : A.shape[0]] = torch.from_numpy(np.ascontiguousarray(A.T)).cuda()
            mats.append(A)
            dev.append(t[:, : A.shape[0]])  # column-major m x n, lda = m + pad
        b = nla.Batch(dev)
        S, info = nla.gesvd_vals_batched(b)
        torch.cuda.synchronize()
        assert np.all(info.cpu().numpy() == 0)
        for A, s in zip(mats, S):
            ref = np.linalg.svd(A.astype(np.float64), compute_uv=False)
            assert err_rel(s.cpu().numpy(), ref) <= 5e-6 * max(A.shape), A.shape
    finally:
        kt.load_config(None)


@pytest.mark.parametrize("m,n", [(1, 1), (3, 1), (1, 9), (32, 32), (33, 33), (96, 64), (64, 96), (128, 129), (192, 192),
                                 (250, 200), (256, 256), (257, 256), (300, 40), (40, 700), (2000, 30), (3000, 250)])
def test_single_small_matrix(nla, m, n):
    # nla_gesvd_vals on both sides of the small-matrix rule, padded leading dimension, A left as it was
    # when asked; the configuration given explicitly takes the two-stage path
    A = np.random.default_rng(5 * m + n).standard_normal((m, n)).astype(np.float32)
    t = torch.zeros(n, m + 2, device="cuda")
    t[:, :m] = torch.from_numpy(np.ascontiguousarray(A.T)).cuda()
    keep = t.clone()
    ref = np.linalg.svd(A.astype(np.float64), compute_uv=False)
    for kw in ({}, {"cfg": nla.Cfg.make(band=16)}):
        S, info = nla.gesvd_vals(t[:, :m], preserve_a=True, **kw)
        torch.cuda.synchronize()
        assert int(info.item()) == 0 and torch.equal(t, keep)
        assert err_rel(S.cpu().numpy(), ref) <= 5e-6 * max(m, n)


@pytest.mark.parametrize("shapes,max_m,max_n", [([(200, 250), (200, 246), (3, 250)], 200, 250),
                                                ([(100, 1000), (7, 999)], 100, 1000), ([(1000, 100)], 1000, 100),
                                                ([(255, 3001), (256, 256)], 256, 3001)])
def test_bounds_of_rows_and_columns(nla, shapes, max_m, max_n):
    # bounds given for m_i and n_i (the binding gives the larger and the smaller dimension): wide matrices at them
    mats = [np.random.default_rng(m + n).standard_normal((m, n)).astype(np.float32) for m, n in shapes]
    b = make_batch(nla, mats)
    b.max_m, b.max_n = max_m, max_n
    S, info = nla.gesvd_vals_batched(b)
    check(S, info, mats)


def test_matrices_beyond_the_bounds_are_refused(nla):
    mats = [np.random.default_rng(i).standard_normal(s).astype(np.float32) for i, s in enumerate([(300, 260), (400, 200), (20, 10)])]
    b = make_batch(nla, mats)
    b.max_m, b.max_n = 200, 200
    for s in b.S:
        s.fill_(-1.0)
    _, info = nla.gesvd_vals_batched(b)
    torch.cuda.synchronize()
    assert info.tolist() == [-7, -7, 0] and float(b.S[0].max()) == -1.0 and float(b.S[1].max()) == -1.0
    b.max_m, b.max_n = 300, 257
    with pytest.raises(nla.NLAError):
        nla.gesvd_vals_batched(b)
