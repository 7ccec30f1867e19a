"""Host threads that call the library at the same time, each on its own stream
and workspace, with scenes of different sizes: the kernels' shared-memory
limits are per kernel and not per call, so one call's must not undo another's.
"""
import threading

import pytest
import torch

import paper_2608_13226_gb300 as cp
from gpu_util import scene, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2608_13226_gb300 import build
    build.build()
    cp.load()


@pytest.mark.parametrize("call,sizes,kw", [
    ("select", (700, 2600, 1100, 1900), dict()),  # 2600: few picks
    ("select", (2100, 2600, 3300, 4500), dict()),
    ("select", (900, 3100, 1300), dict(g=20)),
    ("select", (6500, 7900), dict(sgs_mode=1)),
    ("lite", (5200, 9000, 6100), dict(norm_mode=1)),
    ("select", (13000, 15000), dict(sgs_mode=2))])
def test_threads_with_different_sizes(call, sizes, kw):
    fn = cp.coverprune_select if call == "select" else cp.coverprune_lite_select
    op = cp.CP_OP_SELECT if call == "select" else cp.CP_OP_LITE
    K = 3 if kw.get("sgs_mode") else 12
    prm = cp.Params(**kw)
    jobs = []
    for N in sizes:
        f, pos, fr = to_dev(scene("long_video", N, N=N, D=64))
        ws = cp.workspace(op, 1, N, 64, K, cp.CP_BF16, prm)
        ref = fn(f, pos, fr, K, prm, ws=ws)
        jobs.append((f, pos, fr, ws, ref["kept"].clone()))
    torch.cuda.synchronize()
    errors = []

    def run(f, pos, fr, ws, kept):
        s = torch.cuda.Stream()
        out = torch.empty_like(kept)[None]
        with torch.cuda.stream(s):
            for _ in range(100 if K == 12 else 20):
                try:
                    fn(f, pos, fr, K, prm, ws=ws, out={"kept": out})
                except cp.CoverPruneError as e:
                    errors.append((f.shape[0], str(e)))
            if cp.coverprune_check(ws) != cp.CP_OK or not torch.equal(out[0], kept):
                errors.append((f.shape[0], "result"))

    threads = [threading.Thread(target=run, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, (len(errors), errors[:3])
