"""The bounds-checked build (libfrpcpf_checked.so: every partner index read
from the connectivity is checked on the device before use, and an index out
of range ends the run with FR_EBOUNDS instead of an access outside the
arrays) runs the GPU parity suites with no check firing: the residual, RK4,
preconditioning, tile-variant, batch, partitioned-march and adjoint parity
tests pass on it, and every field they create is destroyed with a status
free of FR_EBOUNDS (the package reads it at destruction under
FRP_BOUNDS_CHECK=1; the tests' conftest fails the test otherwise)."""
import os
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.gpu
@pytest.mark.parametrize("suite,select", [
    ("tests/test_gpu_parity.py", "rhs_parity or march or pseudo or tile_variants or noflux"),
    ("tests/test_gpu_adjoint.py", ""),
    ("tests/test_gpu_batch.py", ""),
    ("tests/test_gpu_partition.py", ""),
])
def test_parity_suites_pass_on_the_bounds_checked_build(suite, select):
    from paper_2006_10967_gb300 import build
    build.build(checked=True)
    env = dict(os.environ, FRP_BOUNDS_CHECK="1")
    probe = subprocess.run([sys.executable, "-c", "import paper_2006_10967_gb300._capi as c; c.lib(); print(c.LIB_PATH)"],
                           cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert probe.stdout.strip().endswith("libfrpcpf_checked.so"), probe.stdout + probe.stderr
    cmd = [sys.executable, "-m", "pytest", suite, "-m", "gpu", "-q", "-x", "-p", "no:cacheprovider"]
    if select:
        cmd += ["-k", select]
    r = subprocess.run(cmd, cwd=ROOT, env=env, capture_output=True, text=True, timeout=1500)
    tail = "\n".join(r.stdout.splitlines()[-15:])
    assert r.returncode == 0, tail
    assert " passed" in tail and "failed" not in tail, tail


_BAD_EDGE = """
import numpy as np
import synthetic as S
import paper_2006_10967_gb300 as G
from paper_2006_10967_gb300 import _capi
N = {order} + 1
w = S.workload("c2t")
w.order, w.n_precond, w.pseudo_kmax = {order}, 1, 2
M = G.Mesh.from_synthetic(S.tri_split(1, 1, periodic=(False, False)), w.order)
n = 2 * 3 * N
for case in ("before the array", "unread word", "wall off its L side"):
    F = G.Field(M, G.make_params(w, "mixed", pseudo_fixed=True), ic=w.circle)
    assert F.sync() == 0
    words = F._ws[F._base - F._ws.data_ptr():][:F.workspace_bytes // 4 * 4].view(F.torch.int32)
    v = words.cpu().numpy()
    at = [i for i in range(0, len(v) - n, 64) if (v[i:i + n] >= 0).all() and (v[i:i + n] < 2 * n).all()
          and (np.sort(v[i:i + n] >> 1) == np.arange(n)).all()]
    assert len(at) == 1, at
    c = v[at[0]:at[0] + n]
    shared = int(np.flatnonzero(c & 1 == 0)[0])     # first point of the shared edge on its R side
    where, word = {{"before the array": (shared, 0 << 1), "unread word": (shared + 1, (1 << 30) - 2),
                   "wall off its L side": (0 if c[0] == 1 else N, None)}}[case]
    words[at[0] + where] = int(c[where]) - 1 if word is None else word
    F.step(1)
    F.precondition()
    assert F.sync() == _capi.FR_EBOUNDS, case
print("checked")
"""


@pytest.mark.gpu
@pytest.mark.parametrize("order", [1, 4])
def test_checked_build_reports_a_broken_triangle_edge(order):
    """A triangle edge whose words do not lead to one whole partner edge ends
    the run of the thread-per-element kernels with FR_EBOUNDS: a partner at the
    array's start, a word beyond the edge's first, a wall marked as an R side."""
    from paper_2006_10967_gb300 import build
    build.build(checked=True)
    r = subprocess.run([sys.executable, "-c", _BAD_EDGE.format(order=order)], cwd=ROOT, capture_output=True, text=True,
                       env=dict(os.environ, FRP_BOUNDS_CHECK="1"), timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "checked", r.stdout + r.stderr
