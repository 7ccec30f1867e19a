"""The default selection (gains kept up to date over lists of live
candidates) against the full sweep, which sums every gain afresh every step:
both add the same fixed-point terms, so picks, gains and objectives are equal
bit for bit.  Sizes sit at the edges of the kernels' tiles (32 rows, 128
columns, 8 to 32 lanes a list, clusters of 1 to 16 blocks), at the smallest and
the largest selections, and at coverage costs that move the fixed-point scale.
"""
import numpy as np
import pytest
import torch

import paper_2608_13226_gb300 as cp
from gpu_util import batch_to_dev, check_sgs_teacher_forced, scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    from paper_2608_13226_gb300 import build
    build.build()
    cp.load()


def host(t):
    return t.cpu().numpy()


def _same(f, pos, fr, K, **kw):
    a = cp.coverprune_select(f, pos, fr, K, cp.Params(sgs_mode=0, **kw))
    b = cp.coverprune_select(f, pos, fr, K, cp.Params(sgs_mode=1, **kw))
    assert cp.coverprune_check(a["ws"]) == cp.CP_OK
    assert cp.coverprune_check(b["ws"]) == cp.CP_OK
    for k in ("kept", "order", "gains", "objective"):
        assert torch.equal(a[k], b[k]), k
    return a


@pytest.mark.parametrize("N,K,g,B", [(1, 1, 0, 1), (2, 2, 0, 3), (31, 31, 0, 1), (33, 33, 0, 2),
                                     (127, 127, 0, 1), (129, 60, 0, 3), (511, 200, 0, 1),
                                     (513, 513, 0, 2), (1025, 300, 0, 5), (2051, 500, 0, 1),
                                     (4099, 400, 0, 9), (8191, 300, 0, 1), (12289, 90, 0, 1),
                                     (33, 20, 2, 2), (100, 100, 99, 1), (257, 120, 33, 3),
                                     (1500, 700, 65, 2), (3001, 500, 100, 1), (12289, 200, 7, 1),
                                     (16384, 300, 64, 1)])
def test_push_equals_full_sweep(N, K, g, B):
    scs = [scene("long_video", sd, N=N, D=64) for sd in range(min(B, 3))]
    f, pos, fr = batch_to_dev((scs * B)[:B])
    _same(f, pos, fr, K, g=g, n_cap=min(8, max(1, N - 1)))


@pytest.mark.parametrize("g", [0, 24])
@pytest.mark.parametrize("m0", [1e-12, 0.05, 0.7, 40.0, 1e12])
def test_push_scale_of_the_coverage_cost(m0, g):
    """m0 sets the first fixed-point scale (and, below the costs, what is live).
    Both modes share the rule of the scales; the gains themselves are compared
    with the oracle's below."""
    s = scene("short_clip", 3, N=700, D=64)
    f, pos, fr = batch_to_dev([s])
    r = _same(f, pos, fr, 150, g=g, m0=m0)
    gains = host(r["gains"])[0].astype(np.float64)
    assert np.all(np.diff(gains) <= 0) and np.all(gains >= 0)
    # F = sum v_j m_j starts at m0 (sum v = 1 up to fp32 rounding) and each
    # step lowers it by its gain: fp32 terms and a gain cut to 24 bits, so
    # relative 2^-23 a step of the sum, and N 2^-24 for the sum of v
    F = float(host(r["objective"])[0])
    assert abs((m0 - gains.sum()) - F) <= m0 * (700 * 2.0 ** -24 + 2.0 ** -20)


@pytest.mark.parametrize("N,B", [(1, 1), (2, 2), (300, 3), (2047, 1), (2048, 2), (4099, 5),
                                 (9000, 1)])
@pytest.mark.parametrize("kw", [dict(), dict(m0=1e12), dict(capacity_mode=1, lambda_x=0.0)])
def test_few_picks_equal_full_sweep(N, B, kw):
    """Few picks sweep their candidates behind bounds; the lists take over
    beyond 8 (16 from 2048 tokens on)."""
    for name in ("long_video", "tiny"):  # bf16: bounds from the cost pass; fp32: none at first
        scs = [scene(name, sd, N=N, D=64) for sd in range(min(B, 2))]
        f, pos, fr = batch_to_dev((scs * B)[:B])
        for K in (1, 2, 8, 9, 16, 17):
            if K <= N:
                _same(f, pos, fr, K, n_cap=min(8, max(1, N - 1)), **kw)


@pytest.mark.parametrize("N,K,g", [(1500, 200, 0), (1500, 400, 24), (300, 300, 0)])
@pytest.mark.parametrize("m0", [1e-3, 1e3, 1e6, 1e9, 1e12, 1e30])
def test_push_coverage_cost_against_the_oracle(orc, m0, N, K, g):
    """Whatever an uncovered token costs, the gains are those of the oracle's
    greedy forced to the same picks, and each pick is its best one, within
    the bars of the default m0; K = N runs the gains down to nothing."""
    s = scene("long_video", 9, N=N, D=64)
    f, pos, fr = batch_to_dev([s])
    r = _same(f, pos, fr, K, g=g, m0=m0)
    c = cp.coverprune_cost(f, pos, fr, cp.Params(g=g))
    nbr = orc.knn_others(s["pos"], g - 1) if g else None
    check_sgs_teacher_forced(orc, host(c["cost"])[0].astype(np.float64),
                             host(c["capacity"])[0].astype(np.float64), host(r["order"])[0],
                             host(r["gains"])[0], float(host(r["objective"])[0]),
                             float(np.float32(m0)), g, nbr)


@pytest.mark.parametrize("K", [6, 40])
@pytest.mark.parametrize("m0", [5.0, 1e3, 1e12])
def test_push_uncovered_after_the_first_pick(m0, K):
    """A token at infinity has no cost to any other: the first pick leaves it
    uncovered, and it is the second for its own m0 v (C(j, j) = 0)."""
    s = scene("long_video", 2, N=400, D=64)
    s["pos"][13, 1] = np.inf
    f, pos, fr = batch_to_dev([s, scene("long_video", 4, N=400, D=64)])
    r = _same(f, pos, fr, K, m0=m0)
    v = host(cp.coverprune_cost(f, pos, fr, cost=False)["capacity"])[0, 13]
    if m0 * v > 1.0:
        assert host(r["order"])[0, 1] == 13
        assert host(r["gains"])[0, 1] == np.float32(v) * np.float32(m0)


@pytest.mark.parametrize("weights", [dict(lambda_f=0.0, lambda_x=0.0, lambda_tau=0.0),
                                     dict(lambda_x=0.0, lambda_tau=0.0), dict(lambda_f=0.0)])
def test_push_ties(weights):
    """Duplicate tokens and vanishing weights: gains tie exactly and the
    lowest index wins (with every weight zero all gains are zero)."""
    s = scene("tiny", 1, N=300, D=64)
    s = {**s, "feats": np.repeat(s["feats"][:100], 3, axis=0),
         "pos": np.repeat(s["pos"][:100], 3, axis=0)}
    f, pos, fr = batch_to_dev([s])
    for g in (0, 17):
        r = _same(f, pos, fr, 250, g=g, **weights)
    if not any(weights.get(k, 1.0) for k in ("lambda_f", "lambda_x", "lambda_tau")):
        assert host(r["order"])[0].tolist() == list(range(250))


@pytest.mark.parametrize("g", [0, 20])
def test_push_in_the_least_workspace(g):
    """Any workspace from the least size on gives the same results; one byte
    less is refused."""
    B, N, D, K = 7, 1025, 64, 120
    scs = [scene("long_video", sd, N=N, D=D) for sd in range(B)]
    f, pos, fr = batch_to_dev(scs)
    prm = cp.Params(g=g)
    ref = cp.coverprune_select(f, pos, fr, K, prm)
    size = cp.coverprune_workspace_size(cp.CP_OP_SELECT, B, N, D, K, cp.CP_BF16, prm)
    least = cp.coverprune_workspace_least(cp.CP_OP_SELECT, B, N, D, K, cp.CP_BF16, prm)
    assert least < size
    for n in (least, (least + size) // 2, size - 1):
        ws = torch.empty(n, dtype=torch.uint8, device="cuda")
        a = cp.coverprune_select(f, pos, fr, K, prm, ws=ws)
        assert cp.coverprune_check(ws) == cp.CP_OK
        for k in ("kept", "order", "gains", "objective"):
            assert torch.equal(a[k], ref[k]), (n, k)
    with pytest.raises(cp.CoverPruneError) as e:
        cp.coverprune_select(f, pos, fr, K, prm, ws=ws[:least - 1])
    assert e.value.status == cp.CP_EWORKSPACE


def test_push_batch_in_waves():
    """A batch whose lists exceed the bound on them runs in waves of scenes:
    every scene equals the same scene alone."""
    N, K, B = 8192, 40, 50
    scs = [scene("long_video", sd, N=N, D=64) for sd in range(2)]
    f, pos, fr = batch_to_dev((scs * B)[:B])
    a = cp.coverprune_select(f, pos, fr, K)
    assert cp.coverprune_check(a["ws"]) == cp.CP_OK
    for i in range(2):
        one = cp.coverprune_select(f[i], pos[i], fr[i], K)
        for b in range(i, B, 2):
            for k in ("kept", "order", "gains", "objective"):
                assert torch.equal(a[k][b], one[k]), (b, k)
