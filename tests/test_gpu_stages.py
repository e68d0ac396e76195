"""Stage-level GPU parity: each stage's output checked by the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2608_21227_gb300 import inputs
from _util import band_dense, err_rel, from_device_colmajor, to_device_colmajor, tol_for

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def nla():
    from paper_2608_21227_gb300 import nla as _nla

    _nla.lib()
    return _nla


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("m,n,b", [(300, 200, 16), (256, 256, 32), (150, 150, 64), (90, 45, 8),
                                   # FP32: several 128-row strips, column splits and ragged tails of the
                                   # TMA / tensor-core projections on both sides
                                   (1100, 900, 16), (1032, 1000, 32), (1064, 1064, 64)])
def test_stage1_band(nla, dt, m, n, b):
    A = inputs.gaussian(m, n, 500 + m + b)
    tdt = torch.float64 if dt == 0 else torch.float32
    if dt == 1:
        A = A.astype(np.float32).astype(np.float64)
    t = to_device_colmajor(A, tdt)
    tauq, taup, info = nla.gebrd_band(t, b)
    ABt = nla.band_extract(t, b)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    D = band_dense(ABt, b)
    # structure: nothing outside the upper band 0 <= j - i <= b
    i, j = np.indices(D.shape)
    assert np.all(D[(j - i < 0) | (j - i > b)] == 0)
    # Frobenius norm and singular values preserved (Section 5.1.1: orthogonal reduction)
    fro = np.linalg.norm(A)
    tolf = (1e-13 if dt == 0 else 1e-6) * m
    assert abs(np.linalg.norm(D) - fro) <= tolf * fro
    assert err_rel(oracle.svdvals(D), oracle.svdvals(A)) <= tol_for(dt, m)
    # the lower part of the panel holds reflectors, the band the reduced matrix
    full = from_device_colmajor(t)
    assert np.allclose(np.triu(full[:n, :n]) * ((j - i) <= b), D, atol=0, rtol=0)


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("n,b", [(200, 16), (256, 32), (130, 64), (50, 2), (64, 3), (3, 2)])
def test_stage2_bulge_chase(nla, dt, n, b):
    g = np.random.default_rng(600 + n + b)
    D = np.triu(g.standard_normal((n, n))) * (np.subtract.outer(np.arange(n), np.arange(n)) >= -b)
    if dt == 1:
        D = D.astype(np.float32).astype(np.float64)
    tdt = torch.float64 if dt == 0 else torch.float32
    t = to_device_colmajor(D, tdt)
    ABt = nla.band_extract(t, b)
    d, e, info = nla.band2bd(ABt, b)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    dn, en = d.cpu().numpy(), e.cpu().numpy()
    fro2 = float(np.sum(D * D))
    tolf = (1e-13 if dt == 0 else 1e-6) * n
    assert abs(np.sum(dn * dn) + np.sum(en * en) - fro2) <= tolf * fro2
    assert err_rel(oracle.bdsvd(dn, en), oracle.svdvals(D)) <= tol_for(dt, n)


@pytest.mark.parametrize("n", [1, 2, 3, 50, 333, 1024])
def test_stage3_bisection_vs_oracle(nla, n):
    g = np.random.default_rng(700 + n)
    d = g.standard_normal(n)
    e = g.standard_normal(max(n - 1, 0))
    S, info = nla.bdsvd_vals(torch.from_numpy(d).cuda(), torch.from_numpy(e).cuda())
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    assert err_rel(S.cpu().numpy(), oracle.bdsvd(d, e)) <= 1e-12 * max(n, 1)


def test_stage3_closed_forms(nla):
    n = 400
    S, _ = nla.bdsvd_vals(torch.ones(n, dtype=torch.float64).cuda(), torch.ones(n - 1, dtype=torch.float64).cuda())
    k = np.arange(1, n + 1)
    assert err_rel(S.cpu().numpy(), 2 * np.cos(k * np.pi / (2 * n + 1))) <= 1e-13 * n
    d = np.array([3.0, 0.0, -2.0, 0.0, 1.0, 5.0])
    S, _ = nla.bdsvd_vals(torch.from_numpy(d).cuda(), torch.zeros(5, dtype=torch.float64).cuda())
    assert err_rel(S.cpu().numpy(), np.sort(np.abs(d))[::-1]) <= 1e-15
    e = np.array([1.0, 2.0, 0.5, 1.5, 0.25])
    S, _ = nla.bdsvd_vals(torch.from_numpy(d).cuda(), torch.from_numpy(e).cuda())
    assert err_rel(S.cpu().numpy(), oracle.bdsvd(d, e)) <= 1e-13


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("n", [8, 9, 17, 40, 609, 1217])
@pytest.mark.parametrize("kind", ["graded", "decoupled", "identity", "no_diagonal"])
def test_stage3_minors_keep_their_signs(nla, dt, n, kind):
    # graded and decoupled bidiagonals make the minors of a Sturm count shrink or vanish; the sizes
    # straddle its blocks of 16 terms and the lanes-per-value limits.  Bound: the search stops at
    # 2^-51 (FP64) / 2^-23 (FP32) of the Gershgorin bound <= 2 sigma_1, plus a few roundings.
    d, e = np.ones(n), np.zeros(n - 1)
    if kind == "graded":
        d = 10.0 ** -np.linspace(0, 16, n)
        e = 0.5 * d[:-1]
    elif kind == "decoupled":
        g = np.random.default_rng(40 + n)
        d, e = g.standard_normal(n), g.standard_normal(n - 1)
        e[::3] = 0.0
        d[::5] = 0.0
    elif kind == "no_diagonal":
        d, e = np.zeros(n), np.ones(n - 1)
    tdt = torch.float64 if dt == 0 else torch.float32
    S, info = nla.bdsvd_vals(torch.from_numpy(d).cuda(), torch.from_numpy(e).cuda(), dtype=tdt)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    B = np.diag(d) + np.diag(e, 1)
    assert err_rel(S.double().cpu().numpy(), np.linalg.svd(B, compute_uv=False)) <= (n * 2.0 ** -51 if dt == 0 else 2.0 ** -20)


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("b", [7, 8, 16, 32, 64])
@pytest.mark.parametrize("n", ["3", "b", "b+1", "2*b", "2*b+2", "5*b+3"])
@pytest.mark.parametrize("store", ["packed", "plain", "wide", "counters_only"])
def test_stage2_widths_edges_and_storage(nla, dt, b, n, store):
    # sizes around one and two block steps; the band in the chase's own leading dimension, in the
    # compact one, in a wider one, and with a workspace that holds the counters only
    import ctypes

    n = max(3, eval(n, {"b": b}))
    per = 2 if dt == 0 else 4
    ldab = {"packed": (3 * b + per) // per * per, "plain": 3 * b + 1, "wide": 3 * b + 6,
            "counters_only": 3 * b + 1}[store]
    g = np.random.default_rng(50 * b + n)
    i, j = np.indices((n, n))
    D = np.where((j - i >= 0) & (j - i <= b), g.standard_normal((n, n)), 0.0)
    tdt = torch.float64 if dt == 0 else torch.float32
    if dt == 1:
        D = D.astype(np.float32).astype(np.float64)
    AB = np.zeros((n, ldab))
    for c in range(n):
        for r in range(max(0, c - b), c + 1):
            AB[c, 2 * b + r - c] = D[r, c]
    t = torch.from_numpy(AB).to("cuda", tdt)
    L = nla.lib()
    need = ctypes.c_size_t(0)
    assert L.nla_band2bd_workspace(n, b, dt, ctypes.byref(need)) == 0
    bytes_ = 4 * n if store == "counters_only" else need.value
    work = torch.empty(max(bytes_, 256), dtype=torch.uint8, device="cuda")
    d = torch.empty(n, dtype=torch.float64, device="cuda")
    e = torch.empty(n, dtype=torch.float64, device="cuda")
    info = torch.zeros(1, dtype=torch.int32, device="cuda")
    st = L.nla_band2bd(n, b, dt, t.data_ptr(), ldab, d.data_ptr(), e.data_ptr(), work.data_ptr(), bytes_,
                       info.data_ptr(), None, torch.cuda.current_stream().cuda_stream)
    assert st == 0
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    dn, en = d.cpu().numpy(), e.cpu().numpy()[: n - 1]
    assert err_rel(oracle.bdsvd(dn, en), oracle.svdvals(D)) <= tol_for(dt, n)
    # the band storage holds the bidiagonal
    got = t.double().cpu().numpy()
    assert np.array_equal(got[:, 2 * b], dn)
    assert np.array_equal(got[1:, 2 * b - 1], en)


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("m,n,b", [(5, 5, 16), (16, 16, 16), (17, 16, 16), (31, 20, 8), (33, 33, 32), (129, 40, 4), (192, 64, 32),
                                   (1025, 40, 16), (2049, 37, 32), (4097, 33, 16), (7681, 33, 16), (8193, 33, 32),
                                   (15361, 20, 16), (16385, 40, 32)])
def test_stage1_panel_row_limits(nla, dt, m, n, b):
    # panels around the rows a warp, a block and a cluster hold (odd leading dimensions: no vector
    # loads), widths below and at the compiled ones, and rows beyond every register variant
    A = np.random.default_rng(m + n + b).standard_normal((m, n))
    if dt == 1:
        A = A.astype(np.float32).astype(np.float64)
    t = to_device_colmajor(A, torch.float64 if dt == 0 else torch.float32)
    tq, tp, info = nla.gebrd_band(t, b)
    ABt = nla.band_extract(t, min(b, n))
    d, e, info2 = nla.band2bd(ABt, min(b, n))
    torch.cuda.synchronize()
    assert int(info.item()) == 0 and int(info2.item()) == 0
    assert err_rel(oracle.bdsvd(d.cpu().numpy(), e.cpu().numpy()), np.linalg.svd(A, compute_uv=False)) <= tol_for(dt, m)


@pytest.mark.parametrize("m,n,b,pad", [(17, 17, 16, 0), (40, 37, 16, 1), (513, 513, 16, 0), (515, 130, 16, 1),
                                       (1030, 600, 16, 2), (2500, 60, 16, 0), (700, 650, 32, 0), (1537, 200, 32, 3),
                                       (2433, 300, 16, 3)])
def test_stage1_one_launch_update(nla, m, n, b, pad):
    # the FP32 update that keeps a strip of lines in a block: ragged strips, long dimensions around its
    # chunks (512 and 256), every lines-per-strip choice, with and without 16-byte alignment; against
    # the two-kernel path (which explicit update parameters select) and the values themselves
    A = np.random.default_rng(3 * m + n).standard_normal((m, n)).astype(np.float32)
    buf = torch.zeros(n, m + pad, device="cuda")
    buf[:, :m] = torch.from_numpy(np.ascontiguousarray(A.T)).cuda()
    ref = np.linalg.svd(A.astype(np.float64), compute_uv=False)
    cfg = nla.Cfg.make(band=b, tile=32, threads=128, cols_per_block=2, unroll=1)
    for c in (nla.Cfg.make(band=b), cfg):
        S, info = nla.gesvd_vals(buf[:, :m].clone() if pad == 0 else buf.clone()[:, :m], cfg=c)
        torch.cuda.synchronize()
        assert int(info.item()) == 0
        assert err_rel(S.double().cpu().numpy(), ref) <= tol_for(1, m)


@pytest.mark.parametrize("cfg", [(16, 64, 256, 2, 4), (32, 64, 128, 2, 1), (64, 64, 256, 4, 2), (16, 128, 512, 4, 1),
                                 (8, 32, 64, 1, 2), (32, 32, 32, 1, 4)])
@pytest.mark.parametrize("m,n", [(70, 40), (300, 257), (1100, 90), (257, 300)])
def test_fp64_update_shapes(nla, cfg, m, n):
    # the FP64 update halves its blocks and splits its sums by the trailing size: 1, 2, 4 and 8
    # reflectors a thread, tiles of 4, 2 and 1 lines, strips and splits that end raggedly
    A = np.random.default_rng(m * n + cfg[0]).standard_normal((m, n))
    if cfg[0] > min(m, n):  # the band is cut to 40, five reflectors a thread: refused
        with pytest.raises(nla.NLAError):
            nla.gesvd_vals(to_device_colmajor(A, torch.float64), cfg=nla.Cfg.make(*cfg))
        return
    S, info = nla.gesvd_vals(to_device_colmajor(A, torch.float64), cfg=nla.Cfg.make(*cfg))
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    assert err_rel(S.cpu().numpy(), np.linalg.svd(A, compute_uv=False)) <= tol_for(0, max(m, n))


@pytest.mark.parametrize("b", [16, 32])
def test_fp64_panel_reflectors_are_orthogonal(nla, b):
    # tau (1 + |v|^2) / 2 = 1 for the stored reflectors.  In units u = 2^-53, rounding independently to
    # nearest: v's entries and their scale, the norm, its root, the sum in tau and tau itself leave
    # about 0.8 u (rms) for 9 to 24 entries, whatever the method; a scalar that loses a bit shows as
    # 1.9 u.  1.2 u lies between.
    m, bad = b + 8, []
    for seed in range(40):
        t = to_device_colmajor(np.random.default_rng(seed).standard_normal((m, b)), torch.float64)
        tauq, _, info = nla.gebrd_band(t, b)
        A, tau = from_device_colmajor(t), tauq.cpu().numpy()
        for j in range(b):
            if m - j - 1 < 24:
                v = A[j + 1:, j].astype(np.longdouble)
                bad.append(float(tau[j] * (1 + v @ v) / 2 - 1) * 2.0 ** 53)
    assert int(info.item()) == 0
    assert np.sqrt(np.mean(np.square(bad))) <= 1.2


# The tensor core rounds its accumulator toward zero: -2.7e-8 of sigma_1 per MMA that a projection
# sums one after another, on each side.  2,100 x 2,000 in 8 splits of 264: 33 K steps on 8 / 4 / 2
# accumulators (band 16 / 32 / 64) on the QR side; on the LQ side blocks of 16 steps, of 48 MMAs at
# band 32 and 99 of one split at band 64.  With 3e-7 for the unbiased rounding: 1.0e-6, 1.9e-6,
# 3.5e-6.  (One accumulator a side at band 16 is 66 MMAs: 2.1e-6.)
@pytest.mark.parametrize("b,tol", [(16, 1.0e-6), (32, 1.9e-6), (64, 3.5e-6)])
def test_fp32_two_kernel_update_accuracy(nla, b, tol):
    A = np.random.default_rng(b).uniform(-1.0, 1.0, (2100, 2000)).astype(np.float32)
    cfg = nla.Cfg.make(*nla.plan_cfg(2100, 2000, nla.F32, cfg=nla.Cfg.make(band=b)))  # named: no one-launch update
    t = to_device_colmajor(A, torch.float32)
    S, info = nla.gesvd_vals(t, cfg=cfg, preserve_a=True)
    again, _ = nla.gesvd_vals(t, cfg=cfg, preserve_a=True)
    torch.cuda.synchronize()
    assert int(info.item()) == 0
    assert torch.equal(S, again)
    assert err_rel(S.double().cpu().numpy(), np.linalg.svd(A.astype(np.float64), compute_uv=False)) <= tol


@pytest.mark.parametrize("m,n,b,pad", [(1100, 900, 16, 0), (1101, 901, 16, 1), (1700, 1500, 16, 0), (1701, 1503, 16, 2),
                                       (900, 800, 32, 0), (640, 30, 16, 0)])
def test_one_launch_update_is_taken(nla, m, n, b, pad):
    # more trailing columns than SMs hold at 4 and at 8 a block (4 x 152, 8 x 152), so that the QR side
    # takes 8 and 16 lines a strip; the same configuration by name turns the one-launch update off, and
    # sums in another order
    A = np.random.default_rng(m + n).standard_normal((m, n)).astype(np.float32)
    buf = torch.zeros(n, m + pad, device="cuda")
    buf[:, :m] = torch.from_numpy(np.ascontiguousarray(A.T)).cuda()
    ref = np.linalg.svd(A.astype(np.float64), compute_uv=False)
    out = []
    for c in (nla.Cfg.make(band=b), nla.Cfg.make(*nla.plan_cfg(m, n, nla.F32, cfg=nla.Cfg.make(band=b)))):
        S, info = nla.gesvd_vals(buf.clone()[:, :m], cfg=c)  # (in place: the leading dimension is the caller's)
        torch.cuda.synchronize()
        assert int(info.item()) == 0
        assert err_rel(S.double().cpu().numpy(), ref) <= tol_for(1, m)
        out.append(S)
    assert not torch.equal(out[0], out[1])


@pytest.mark.parametrize("dt", [0, 1])
@pytest.mark.parametrize("n,b", [(700, 8), (1500, 16), (900, 32), (600, 64), (900, 24), (400, 5)])
def test_chase_storage_forms_agree(nla, dt, n, b):
    # the same chase whether columns move as bulk copies (packed), element by element (a workspace of
    # counters only, no workspace at all, other leading dimensions), and every time: d and e bit for bit
    import ctypes

    i, j = np.indices((n, n))
    D = np.where((j - i >= 0) & (j - i <= b), np.random.default_rng(n + b).standard_normal((n, n)), 0.0)
    tdt = torch.float64 if dt == 0 else torch.float32
    L, st = nla.lib(), torch.cuda.current_stream().cuda_stream
    vp = ctypes.c_void_p
    L.nla_band2bd_noalloc.argtypes = [ctypes.c_int] * 3 + [vp, ctypes.c_int, vp, vp, vp, vp]
    need = ctypes.c_size_t(0)
    assert L.nla_band2bd_workspace(n, b, dt, ctypes.byref(need)) == 0
    AB0 = nla.band_extract(to_device_colmajor(D, tdt), b)
    results = []
    for ldab, work_bytes in [(3 * b + 1, need.value), (3 * b + 1, 4 * n), (3 * b + 7, 4 * n), (3 * b + 1, None)] * 2:
        AB = torch.zeros(n, ldab, dtype=tdt, device="cuda")
        AB[:, :3 * b + 1] = AB0[:, :3 * b + 1]
        d = torch.zeros(n, dtype=torch.float64, device="cuda")
        e = torch.zeros(n, dtype=torch.float64, device="cuda")
        info = torch.zeros(1, dtype=torch.int32, device="cuda")
        args = (n, b, dt, AB.data_ptr(), ldab, d.data_ptr(), e.data_ptr())
        if work_bytes is None:
            assert L.nla_band2bd_noalloc(*args, info.data_ptr(), st) == 0
        else:
            work = torch.empty(max(work_bytes, 256), dtype=torch.uint8, device="cuda")
            assert L.nla_band2bd(*args, work.data_ptr(), work_bytes, info.data_ptr(), None, st) == 0
        torch.cuda.synchronize()
        assert int(info.item()) == 0
        results.append((d, e[:n - 1]))
    for d, e in results[1:]:
        assert torch.equal(d, results[0][0]) and torch.equal(e, results[0][1])
    assert err_rel(oracle.bdsvd(d.cpu().numpy(), e.cpu().numpy()), np.linalg.svd(D, compute_uv=False)) <= tol_for(dt, n)
