"""Alternative execution paths that environment switches select (read once per
process, so each runs in a subprocess): the SIMT projections instead of the
tensor-core ones (both sides, or the LQ side alone), the one-sweep-per-block bulge chase, the grid-wide panel, the
shared-memory cluster panel, programmatic dependent launch and other sweep-group sizes.  Each must give the same
singular values as the FP64 oracle within the parity tolerance."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, sys
import numpy as np, torch
sys.path.insert(0, sys.argv[1]); sys.path.insert(0, sys.argv[1] + "/tests")
from paper_2608_21227_gb300 import nla, inputs
import oracle
from _util import err_rel, tol_for
out = []
for (m, n, b, dt) in [(300, 260, 16, 1), (512, 512, 32, 1), (257, 200, 16, 0), (640, 640, 64, 1)]:
    A = inputs.gaussian(m, n, 900 + m + b)
    if dt == 1:
        A = A.astype(np.float32).astype(np.float64)
    t = torch.from_numpy(np.ascontiguousarray(A.T)).cuda().to(torch.float32 if dt == 1 else torch.float64)
    S, info = nla.gesvd_vals(t, cfg=nla.Cfg.make(band=b))
    torch.cuda.synchronize()
    e = err_rel(S.double().cpu().numpy(), oracle.svdvals(A))
    out.append({"m": m, "n": n, "b": b, "dt": dt, "info": int(info.item()), "err": e, "tol": tol_for(dt, max(m, n))})
print(json.dumps(out))
"""

VARIANTS = {
    "simt_projections": {"NLA_PROJ_TC": "0"},
    "simt_lq_projection": {"NLA_PROJ_TC": "1"},
    "chase_one_sweep_per_block": {"NLA_CHASE_GROUP": "0"},
    "chase_group_4": {"NLA_CHASE_GROUP": "4"},
    "grid_panel": {"NLA_PANEL_CLUSTER": "0"},
    "shared_memory_cluster_panel": {"NLA_PANEL_REG": "0"},
    "programmatic_dependent_launch": {"NLA_PDL": "1"},
}


@pytest.mark.parametrize("name", sorted(VARIANTS))
def test_variant_matches_oracle(name):
    env = dict(os.environ, **VARIANTS[name])
    r = subprocess.run([sys.executable, "-c", CHILD, ROOT], env=env, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    for rec in json.loads(r.stdout.strip().splitlines()[-1]):
        assert rec["info"] == 0, rec
        assert rec["err"] <= rec["tol"], rec


@pytest.mark.parametrize("env", [{}, {"NLA_PDL": "0"}])
def test_whole_svd_captured_and_replayed(env):
    # programmatic dependent launch is on by default: plain, captured in a graph and replayed on new
    # data, and with it off, the values agree with the reference
    child = r"""
import sys
import numpy as np, torch
sys.path.insert(0, sys.argv[1]); sys.path.insert(0, sys.argv[1] + "/tests")
from paper_2608_21227_gb300 import nla
from _util import err_rel, tol_for
for (m, n, dt) in [(700, 500, torch.float32), (2500, 300, torch.float32), (260, 200, torch.float64)]:
    code = 1 if dt == torch.float32 else 0
    g = torch.Generator(device="cuda"); g.manual_seed(m)
    A = torch.randn(n, m, generator=g, device="cuda", dtype=dt)
    work = nla.workspace(nla.gesvd_vals_workspace(m, n, code, preserve_a=True))
    S = torch.empty(n, dtype=dt, device="cuda"); info = torch.zeros(1, dtype=torch.int32, device="cuda")
    run = lambda: nla.gesvd_vals(A, preserve_a=True, work=work, S=S, info=info)
    run(); torch.cuda.synchronize()
    st = torch.cuda.Stream(); gr = torch.cuda.CUDAGraph()
    with torch.cuda.stream(st):
        with torch.cuda.graph(gr, stream=st):
            run()
    for _ in range(2):
        A.copy_(torch.randn(n, m, generator=g, device="cuda", dtype=dt))
        S.fill_(float("nan"))
        gr.replay(); torch.cuda.synchronize()
        ref = np.linalg.svd(A.double().cpu().numpy(), compute_uv=False)
        assert int(info.item()) == 0 and err_rel(S.double().cpu().numpy(), ref) <= tol_for(code, m)
print("ok")
"""
    r = subprocess.run([sys.executable, "-c", child, ROOT], env=dict(os.environ, **env), capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stderr[-2000:]


# The switches on shapes and configurations that do reach what they switch: with the update's parameters named, the
# two-kernel FP32 update runs (leading dimensions of whole 16 bytes) at bands 16, 32 and 64, over enough columns to
# go round its accumulators.
TWO_KERNEL_CHILD = r"""
import json, sys
import numpy as np, torch
sys.path.insert(0, sys.argv[1]); sys.path.insert(0, sys.argv[1] + "/tests")
from paper_2608_21227_gb300 import nla
from _util import err_rel, tol_for
out = []
for (m, n, b) in [(1100, 900, 16), (1032, 1000, 32), (1064, 1064, 64), (2100, 300, 16), (700, 650, 32)]:
    A = np.random.default_rng(m + n + b).standard_normal((m, n)).astype(np.float32)
    t = torch.from_numpy(np.ascontiguousarray(A.T)).cuda()
    S, info = nla.gesvd_vals(t, cfg=nla.Cfg.make(*nla.plan_cfg(m, n, nla.F32, cfg=nla.Cfg.make(band=b))))
    torch.cuda.synchronize()
    e = err_rel(S.double().cpu().numpy(), np.linalg.svd(A.astype(np.float64), compute_uv=False))
    out.append({"m": m, "n": n, "b": b, "info": int(info.item()), "err": e, "tol": tol_for(1, max(m, n)),
                "values": S.cpu().numpy().tolist()})
print(json.dumps(out))
"""


def _two_kernel(env):
    r = subprocess.run([sys.executable, "-c", TWO_KERNEL_CHILD, ROOT], env=dict(os.environ, **env), capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    out = json.loads(r.stdout.strip().splitlines()[-1])
    for rec in out:
        assert rec["info"] == 0 and rec["err"] <= rec["tol"], {k: v for k, v in rec.items() if k != "values"}
    return [rec["values"] for rec in out]


@pytest.fixture(scope="module")
def two_kernel_default():
    return _two_kernel({})


@pytest.mark.parametrize("mask", ["0", "1", "2"])
def test_two_kernel_update_projections(two_kernel_default, mask):
    # other sums, so other last digits: the switch has an effect on every shape
    for a, b in zip(_two_kernel({"NLA_PROJ_TC": mask}), two_kernel_default):
        assert a != b


def test_two_kernel_update_in_plain_stream_order(two_kernel_default):
    assert _two_kernel({"NLA_PDL": "0"}) == two_kernel_default
