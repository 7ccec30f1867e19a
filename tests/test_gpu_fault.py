"""Failure detection without a GPU fault: every device-side wait of the
library is bounded.  The self-test launches co-resident blocks on a grid
barrier that expects more arrivals than there are blocks -- a flag nobody
sets -- and the kernel must give up after the time limit, record
CP_ETIMEOUT in the workspace status word and return, leaving the context
usable."""
import time

import pytest
import torch

import paper_2608_13226_gb300 as cp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2608_13226_gb300 import build
    build.build()
    cp.load()


def test_barrier_times_out_and_context_survives():
    ws = torch.empty(256, dtype=torch.uint8, device="cuda")
    t0 = time.time()
    st = cp.coverprune_barrier_selftest(4, 5, 50.0, ws)  # 4 blocks, 5 expected
    dt = time.time() - t0
    assert st == cp.CP_ETIMEOUT
    assert dt < 5.0
    # the context still works: a passing barrier and a real call
    assert cp.coverprune_barrier_selftest(4, 4, 50.0, ws) == cp.CP_OK
    f = torch.randn(64, 16, device="cuda").to(torch.bfloat16)
    pos = torch.rand(64, 3, device="cuda")
    fr = torch.zeros(64, dtype=torch.int32, device="cuda")
    r = cp.coverprune_select(f, pos, fr, 8)
    assert cp.coverprune_check(r["ws"]) == cp.CP_OK
    assert r["kept"].shape == (8,)


def test_select_reports_ok_status():
    f = torch.randn(300, 64, device="cuda").to(torch.bfloat16)
    pos = torch.rand(300, 3, device="cuda")
    fr = torch.arange(300, dtype=torch.int32, device="cuda") // 30
    for g in (0, 12):
        r = cp.coverprune_select(f, pos, fr, 30, cp.Params(g=g))
        assert cp.coverprune_check(r["ws"]) == cp.CP_OK
    lt = cp.coverprune_lite_select(f, pos, fr, 30)
    assert cp.coverprune_check(lt["ws"]) == cp.CP_OK


@pytest.mark.parametrize("eps", [0.05, 1e-3])  # the factors alone; both forms of the iterations
def test_literal_rule_gives_up_as_a_cluster(eps):
    """Waits of the transport rule's iterations limited to a nanosecond: a
    block may give up where its peers did not have to wait, and then none of
    the cluster may go on to the second form.  The call returns, its status is
    one of the two, and the context and the workspace work afterwards."""
    gen = torch.Generator(device="cuda").manual_seed(3)
    f = torch.randn(5, 1024, 64, generator=gen, device="cuda")
    pos = torch.rand(5, 1024, 3, generator=gen, device="cuda") * 6
    fr = (torch.arange(1024, device="cuda") // 128).to(torch.int32).expand(5, 1024).contiguous()
    ref = cp.coverprune_select(f, pos, fr, 12, cp.Params(sgs_mode=2, sot_eps=eps))
    assert cp.coverprune_check(ref["ws"]) == cp.CP_OK
    t0 = time.time()
    for _ in range(3):
        r = cp.coverprune_select(f, pos, fr, 12, cp.Params(sgs_mode=2, sot_eps=eps, timeout_ms=1e-6),
                                 ws=ref["ws"])
        assert cp.coverprune_check(r["ws"]) in (cp.CP_OK, cp.CP_ETIMEOUT)
    assert time.time() - t0 < 5.0
    r = cp.coverprune_select(f, pos, fr, 12, cp.Params(sgs_mode=2, sot_eps=eps), ws=ref["ws"])
    assert cp.coverprune_check(r["ws"]) == cp.CP_OK
    for k in ("kept", "order", "gains", "objective"):
        assert torch.equal(r[k], ref[k]), k
