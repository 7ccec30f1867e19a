"""The calls a program that prunes 3D scene tokens makes, with their sizes, inputs and expected accuracy.

A case names one public entry point ("op"), the sizes of its input and the options that program would set.  Inputs are
synthetic scenes of the shape the method is used on: a camera walking through a room, one token per image patch with a
back-projected position, features that repeat where the same surface is seen again (noise around a heavy-tailed set of
modes) and a few outliers.  The workspace is kept between calls, as a serving program keeps it; outputs are allocated by
each call.
"""
import math

import torch

import paper_2608_13226_gb300 as cp

ROOM = (8.0, 8.0, 3.0)
SELECT, LITE, COST, KNN, GATHER = "select", "lite", "cost", "knn", "gather"


def _case(op, N, D, B=1, K=0, dtype="bf16", tpf=256, modes=64, **options):
    c = {"op": op, "B": B, "N": N, "D": D, "K": K, "dtype": dtype, "tpf": tpf, "modes": modes,
         "g": 0, "norm_mode": 0, "sgs_mode": 0, "n_cap": 8, "k": 0}
    c.update(options)
    return c


def listed():
    return [
        # the smallest scene of the workloads, fp32 features: one interactive call, latency
        dict(_case(SELECT, 1024, 256, K=102, dtype="f32", tpf=128, modes=16), name="select tiny f32"),
        # a short clip, one scene alone: the latency a user waits for before decoding starts
        dict(_case(SELECT, 4096, 1280, K=410, modes=32), name="select short clip"),
        # a long video, one scene alone, 15% kept
        dict(_case(SELECT, 8192, 3584, K=1229), name="select long video"),
        # the throughput batch: 32 long videos a call
        dict(_case(SELECT, 8192, 3584, B=32, K=1229), name="select batch of 32"),
        # local neighbourhoods (64 tokens), throughput batch
        dict(_case(SELECT, 8192, 3584, B=32, K=1229, g=64), name="select local batch of 32"),
        # local neighbourhoods without the all-pairs pass, 32 frames of 14 x 14 patches, 10% kept
        dict(_case(SELECT, 6272, 1280, B=4, K=628, tpf=196, g=64, norm_mode=1), name="select local bounded"),
        # the light selection over the throughput batch, exact feature normaliser
        dict(_case(LITE, 8192, 3584, B=32, K=1229), name="lite batch of 32"),
        # the light selection of the longest scene alone, without the all-pairs pass
        dict(_case(LITE, 16384, 3584, K=1638, norm_mode=1), name="lite long bounded"),
        # cost and capacity for a program with its own selection; odd sizes, rows not 16-byte aligned
        dict(_case(COST, 3001, 1160, B=2, tpf=196, modes=32), name="cost ragged"),
        # the selection rule that solves a transport problem per step, small scene (an ablation)
        dict(_case(SELECT, 1024, 256, K=102, dtype="f32", tpf=128, modes=16, sgs_mode=2), name="select transport rule"),
        # neighbour lists alone, for a program that builds its own graph
        dict(_case(KNN, 7000, 8, B=8, tpf=196, k=63), name="neighbours 63"),
        # the kept rows of the throughput batch, compacted for the language model
        dict(_case(GATHER, 8192, 3584, B=32, K=1229), name="gather batch of 32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice([SELECT, SELECT, SELECT, SELECT, LITE, LITE, COST, KNN, GATHER])
    f32 = op in (SELECT, LITE, COST) and rng.random() < 0.2
    N = _log(rng, 300, 3000 if f32 else 16384)
    D = 4 * _log(rng, 16, 128) if f32 else 8 * _log(rng, 8, 448)
    # within the work of the largest listed case, and three states on the card
    most = 32 * 8192 * 8192 // 2
    B = _log(rng, 1, max(1, min(32, most // (N * N))))
    K = math.ceil(rng.choice([0.05, 0.1, 0.15, 0.25]) * N)
    c = _case(op, N, D, B, K, "f32" if f32 else "bf16", rng.choice([100, 128, 196, 256]), rng.choice([16, 32, 64]))
    if op == SELECT:
        kind = rng.random()
        if kind < 0.35:
            c["g"] = rng.choice([16, 24, 33, 64, 100])
            c["norm_mode"] = rng.choice([0, 1])
        elif kind < 0.42:
            c.update(sgs_mode=2, N=min(N, 1500), K=min(K, 100), B=1)
        c["n_cap"] = rng.choice([8, 8, 8, 4, 12])
    elif op == LITE:
        c["norm_mode"] = rng.choice([0, 1])
        c["n_cap"] = rng.choice([8, 8, 8, 4, 12])
    elif op == COST:
        c.update(N=min(N, 6000), K=0)
    elif op == KNN:
        c.update(D=8, K=0, k=rng.choice([4, 8, 16, 40, 63, 100]))
    return c


# ------------------------------------------------------------------ inputs
def _positions(c, gen):
    """[B, N, 3] fp32: frames of a walking pinhole camera, one point per patch of a square grid."""
    B, N, tpf = c["B"], c["N"], c["tpf"]
    side = max(1, math.isqrt(tpf))
    frames = -(-N // tpf)
    step = torch.randn(B, frames, 2, generator=gen, device="cuda") * 0.25
    turn = torch.randn(B, frames, generator=gen, device="cuda") * math.radians(20)
    yaw = turn.cumsum(1) + 2 * math.pi * torch.rand(B, 1, generator=gen, device="cuda")
    eye = torch.cat([(step.cumsum(1) + 4.0).clamp(1.0, 7.0), torch.full((B, frames, 1), 1.5, device="cuda")], 2)
    i = torch.arange(tpf, device="cuda")
    u = ((i % side) + 0.5) / side * 2 - 1
    w = ((i // side) + 0.5) / -(-tpf // side) * 2 - 1
    co, si = yaw.cos()[..., None], yaw.sin()[..., None]
    d = torch.stack([co + u * si, si - u * co, (-w).expand(B, frames, tpf)], -1)
    d = d / d.norm(dim=-1, keepdim=True)
    p = eye[:, :, None, :]
    room = torch.tensor(ROOM, device="cuda")
    t = torch.where(d > 0, (room - p) / d, torch.where(d < 0, -p / d, torch.full_like(d, 1e9))).amin(-1)
    depth = t.clamp(1.0, 6.0) * (1 + 0.02 * torch.randn(t.shape, generator=gen, device="cuda"))
    return (p + depth[..., None] * d).reshape(B, frames * tpf, 3)[:, :N].contiguous()


def _inputs(case, seed):
    c = case
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    B, N, D, M = c["B"], c["N"], c["D"], c["modes"]
    pos = _positions(c, gen)
    frame = (torch.arange(N, device="cuda") // c["tpf"]).to(torch.int32).expand(B, N).contiguous()
    if c["op"] == KNN:
        return None, pos, frame
    # contiguous runs of surface (height band, azimuth about the room's centre) share a feature mode, sizes heavy-tailed
    key = pos[..., 2].floor().clamp(0, 2) * 10 + torch.atan2(pos[..., 1] - 4.0, pos[..., 0] - 4.0)
    share = torch.arange(1, M + 1, device="cuda", dtype=torch.float64) ** -1.2
    edge = (share / share.sum()).cumsum(0)
    run = torch.searchsorted(edge, (torch.arange(N, device="cuda", dtype=torch.float64) + 0.5) / N).clamp(max=M - 1)
    dt = torch.bfloat16 if c["dtype"] == "bf16" else torch.float32
    feats = torch.empty(B, N, D, dtype=dt, device="cuda")
    for b in range(B):
        name = torch.randperm(M, generator=gen, device="cuda")
        centre = torch.randn(M, D, generator=gen, device="cuda")
        centre = centre / centre.norm(dim=1, keepdim=True)
        label = torch.empty(N, dtype=torch.int64, device="cuda")
        label[key[b].argsort(stable=True)] = name[run]
        f = torch.randn(N, D, generator=gen, device="cuda") * (0.3 / math.sqrt(D)) + centre[label]
        odd = torch.rand(N, generator=gen, device="cuda") < 0.05
        other = (torch.rand(N, D, generator=gen, device="cuda") * 2 - 1) * math.sqrt(3.0 / D)
        feats[b] = torch.where(odd[:, None], other, f).to(dt)
    return feats, pos, frame


def _params(c):
    return cp.Params(g=c["g"], norm_mode=c["norm_mode"], sgs_mode=c["sgs_mode"], n_cap=c["n_cap"])


def prepare(case, seed):
    c = case
    feats, pos, frame = _inputs(c, seed)
    s = {"op": c["op"], "feats": feats, "pos": pos, "frame": frame, "K": c["K"], "k": c["k"], "prm": _params(c)}
    dt = cp.CP_BF16 if c["dtype"] == "bf16" else cp.CP_F32
    kind = {SELECT: cp.CP_OP_SELECT, LITE: cp.CP_OP_LITE, COST: cp.CP_OP_COST, KNN: cp.CP_OP_KNN}.get(c["op"])
    if kind is not None:
        s["ws"] = cp.workspace(kind, c["B"], c["N"], c["D"], c["K"], dt, s["prm"])
    if c["op"] == GATHER:
        gen = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
        order = torch.rand(c["B"], c["N"], generator=gen, device="cuda").argsort(1)
        s["kept"] = order[:, :c["K"]].sort(1).values.contiguous()
    return s


def run(s):
    if s["op"] == SELECT:
        r = cp.coverprune_select(s["feats"], s["pos"], s["frame"], s["K"], s["prm"], ws=s["ws"])
        return {k: r[k] for k in ("kept", "order", "gains", "objective")}
    if s["op"] == LITE:
        r = cp.coverprune_lite_select(s["feats"], s["pos"], s["frame"], s["K"], s["prm"], ws=s["ws"])
        return {k: r[k] for k in ("kept", "group_start", "objective")}
    if s["op"] == COST:
        r = cp.coverprune_cost(s["feats"], s["pos"], s["frame"], s["prm"], ws=s["ws"])
        return {k: r[k] for k in ("cost", "capacity", "norms")}
    if s["op"] == KNN:
        nbr, diameter = cp.coverprune_knn(s["pos"], s["k"], ws=s["ws"])
        return {"nbr": nbr, "diameter": diameter}
    f, p, t = cp.coverprune_gather(s["feats"], s["pos"], s["frame"], s["kept"])
    return {"feats": f, "pos": p, "frame": t}


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    c = case
    B, N, D, K = c["B"], c["N"], c["D"], c["K"]
    e = 2 if c["dtype"] == "bf16" else 4
    inputs = B * N * (D * e + 12 + 4)
    pairs = B * N * (N + 1) / 2       # unordered pairs, one dot product of 2 D flops each
    near = B * N * c["n_cap"]         # the pairs of the capacity score
    if c["op"] == SELECT:
        out = B * K * (8 + 8 + 4) + 8 * B
        g = c["g"]
        if g and c["norm_mode"]:      # only neighbourhood pairs are ever needed, each once
            return {"bytes": inputs + out, "flops": B * N * g / 2 * 2 * D}
        return {"bytes": inputs + out, "flops": pairs * 2 * D}
    if c["op"] == LITE:
        out = B * K * (8 + 4) + 8 * B
        if c["norm_mode"]:            # the capacity's pairs, and the pairs within groups of N / K tokens
            return {"bytes": inputs + out, "flops": (near + B * N * (N / max(1, K)) / 2) * 2 * D}
        return {"bytes": inputs + out, "flops": pairs * 2 * D}
    if c["op"] == COST:
        return {"bytes": inputs + B * N * N * 4 + B * N * 4 + B * 24, "flops": pairs * 2 * D}
    if c["op"] == KNN:                # its compulsory traffic; the search's own arithmetic depends on the scene
        return {"bytes": B * N * (12 + 4 * c["k"]) + 4 * B, "flops": B * N * c["k"] * 8}
    return {"bytes": B * K * (2 * (D * e + 12 + 4) + 8), "flops": 0}


def tolerance(case):
    op = case["op"]
    if op in (KNN, GATHER):
        return "exact"                # integers decided in pinned fp32, a correctly rounded root, copied bytes
    # About four times what the calls show against 64 bits (see exact), seen over these ranges: fp32 features 1e-7 to 2e-7
    # (single values 1e-6); bf16 features, whose dot products the tensor cores sum, cost 5e-7, capacity 4e-6, gains 1e-6, and
    # an objective whose costs are all small 9e-6 up to D = 2048 and 5e-5 at D = 3584.
    # Order and kept: two candidates whose gains agree to fp32 rounding may swap places in the order.
    f32 = case["dtype"] == "f32"
    if op == COST:
        return {"rel": 1e-6, "max": 5e-6} if f32 else {"rel": 1.5e-5, "max": 2e-5}
    if op == LITE:
        return {"rel": 1e-6, "max": 5e-6, "differ": 0.01} if f32 else {"rel": 5e-6, "max": 2e-5, "differ": 0.01}
    if f32:
        return {"rel": 1e-6, "max": 5e-6, "differ": 0.01}
    rel = 4e-5 if case["D"] <= 2048 else 2e-4
    return {"rel": rel, "max": rel, "differ": 0.01}


# ------------------------------------------------------------------ the same values in 64 bits
def _neighbours(pos, n):
    """[N, n] nearest other tokens by the squared distance in fp32, one rounding per operation, ties by index."""
    N = pos.shape[0]
    x, y, z = pos[:, 0], pos[:, 1], pos[:, 2]
    rows = []
    for a in range(0, N, 1024):
        dx, dy, dz = x[a:a + 1024, None] - x, y[a:a + 1024, None] - y, z[a:a + 1024, None] - z
        d2 = (dx * dx + dy * dy) + dz * dz
        key = (d2.view(torch.int32).to(torch.int64) << 32) | torch.arange(N, device="cuda")
        i = torch.arange(a, min(a + 1024, N), device="cuda")
        key[i - a, i] = 2 ** 63 - 1
        rows.append(key.topk(n, largest=False, sorted=True).values & 0xFFFFFFFF)
    return torch.cat(rows)


class _Scene:
    """One scene in 64 bits: normalisers, neighbours, capacity, and the cost of any rows."""

    def __init__(self, c, feats, pos, frame, nn):
        f = feats.double()
        self.f = f / f.norm(dim=1, keepdim=True).clamp(min=1e-300)
        self.x, self.t = pos.double(), frame.double()
        N = f.shape[0]
        lo, hi, far = 2.0, 0.0, 0.0
        for a in range(0, N, 2048):
            far = max(far, float(torch.cdist(self.x[a:a + 2048], self.x).max()))
            if c["norm_mode"] == 0:
                d = self._df(torch.arange(a, min(a + 2048, N), device="cuda"))
                lo, hi = min(lo, float(d.min())), max(hi, float(d.max()))
        self.norms = (lo, hi, 0.0, far, 0.0, float(self.t.max() - self.t.min()))
        if c["norm_mode"]:
            self.norms = (0.0, 2.0) + self.norms[2:]
        self.inv = [1.0 / r if r > 1e-6 else 0.0 for r in (self.norms[1] - self.norms[0], far, self.norms[5])]
        self.nbr = _neighbours(pos, min(nn, N - 1))
        k = self.nbr[:, :c["n_cap"]]
        terms = 0.0
        for q in range(k.shape[1]):
            o = k[:, q]
            terms = terms + ((1 - (self.f * self.f[o]).sum(1).clamp(-1, 1)) - self.norms[0]) * self.inv[0]
            terms = terms + (self.x - self.x[o]).norm(dim=1) * self.inv[1]
            terms = terms + (self.t - self.t[o]).clamp(min=0) * self.inv[2]
        r = terms / max(1, k.shape[1])
        self.v = r / r.sum()

    def _df(self, i):
        g = (self.f[i] @ self.f.T).clamp(-1, 1)
        g[torch.arange(i.numel(), device="cuda"), i] = 1.0
        return 1 - g

    def fst(self, df, dist, dt):
        return (df - self.norms[0]) * self.inv[0] + torch.log1p(10.0 * dist * self.inv[1]) / math.log(11.0) \
            + dt.clamp(min=0) * self.inv[2]

    def rows(self, i):
        diff = self.x[i][:, None, :] - self.x[None]
        return self.fst(self._df(i), diff.norm(dim=2), self.t[i][:, None] - self.t[None])

    def cost(self):
        N = self.f.shape[0]
        return torch.cat([self.rows(torch.arange(a, min(a + 1024, N), device="cuda")) for a in range(0, N, 1024)])


def _greedy(s, K, g):
    C = s.cost()
    N = C.shape[0]
    if 0 < g < N:                     # targets outside M_g(t) are out of t's reach
        near = torch.zeros(N, N, dtype=torch.bool, device="cuda")
        near.scatter_(1, s.nbr[:, :g - 1], True)
        near.fill_diagonal_(True)
        C = torch.where(near, C, torch.full_like(C, math.inf))
    CT = C.T.contiguous()
    m = torch.full((N,), 3.0, dtype=torch.float64, device="cuda")
    gain = torch.zeros(N, dtype=torch.float64, device="cuda")
    for a in range(0, N, 1024):
        gain += s.v[a:a + 1024] @ (m[a:a + 1024, None] - CT[a:a + 1024]).clamp(min=0)
    gains, free = [], torch.zeros(N, dtype=torch.float64, device="cuda")
    for _ in range(K):
        best, w = (gain + free).max(0)
        gains.append(best)
        free[w] = -math.inf
        row = C[w]
        low = (row < m).nonzero()[:, 0]
        for a in range(0, low.numel(), 1024):
            j = low[a:a + 1024]
            c = CT[j]
            gain -= s.v[j] @ ((m[j, None] - c).clamp(min=0) - (row[j, None] - c).clamp(min=0))
        m = torch.minimum(m, row)
    return torch.stack(gains), (s.v * m).sum()


def _transport(s, K, g):
    C = s.cost()
    N = C.shape[0]
    eps, lv = 0.05, s.v.log()
    pot = torch.zeros(N, dtype=torch.float64, device="cuda")
    rest, picked, scores, free = s.v, [], [], torch.zeros(N, dtype=torch.float64, device="cuda")
    for step in range(K):
        if step:
            S = C[picked]
            for _ in range(20):
                f = eps * (-math.log(K) - ((pot - S) / eps).logsumexp(1))
                pot = (eps * (lv - ((f[:, None] - S) / eps).logsumexp(0))).clamp(max=0)
            rest = (s.v - ((f[:, None] + pot - S) / eps).exp().sum(0)).clamp(min=0)
        score = C @ rest
        best, w = (score + free).min(0)
        scores.append(best)
        free[w] = math.inf
        picked.append(int(w))
    m = C[picked].amin(0).clamp(max=3.0)
    return torch.stack(scores), (s.v * m).sum()


def _spread(q):
    r = torch.zeros_like(q)
    for i in range(10):
        r |= ((q >> i) & 1) << (3 * i)
    return r


def _groups(s, pos, K):
    """Objective of the light selection: Morton order, groups of capacity 1 / K, the cheapest member of each."""
    N = pos.shape[0]
    cell = ((pos - pos.amin(0)) / torch.tensor(0.2, device="cuda")).floor().clamp(0, 1023).to(torch.int64)
    code = _spread(cell[:, 0]) | _spread(cell[:, 1]) << 1 | _spread(cell[:, 2]) << 2
    perm = (code * N + torch.arange(N, device="cuda")).argsort()
    mass = (s.v[perm].float().double() * 2.0 ** 40).round().cumsum(0)
    q = torch.arange(1, K, device="cuda", dtype=torch.float64)
    ideal = torch.searchsorted(mass, q / K * mass[-1]) + 1
    at = torch.arange(1, K, device="cuda")
    start = at + (ideal - at).cummax(0).values.clamp(max=N - K) if K > 1 else at
    start = [0] + start.tolist() + [N]
    total = 0.0
    a = 0
    while a < K:                      # runs of groups, at most about 256 tokens a product
        e = a + 1
        while e < K and start[e + 1] - start[a] <= 256:
            e += 1
        i = perm[start[a]:start[e]]
        df = 1 - (s.f[i] @ s.f[i].T).clamp(-1, 1).fill_diagonal_(1.0)
        C = s.fst(df, (s.x[i][:, None] - s.x[i][None]).norm(dim=2), s.t[i][:, None] - s.t[i][None])
        of = torch.repeat_interleave(torch.arange(a, e, device="cuda"),
                                     torch.tensor([start[b + 1] - start[b] for b in range(a, e)], device="cuda"))
        score = torch.where(of[:, None] == of[None], C, torch.zeros_like(C)) @ s.v[i]
        total = total + torch.full((e - a,), math.inf, dtype=torch.float64, device="cuda").scatter_reduce(
            0, of - a, score, "amin").sum()
        a = e
    return total


def exact(case, seed):
    c = case
    B, N, D, K = c["B"], c["N"], c["D"], c["K"]
    # 64-bit products run at about 1 TFLOP/s here; a greedy step costs a few launches a scene
    all_pairs = c["op"] in (SELECT, COST) or (c["op"] == LITE and c["norm_mode"] == 0)
    seconds = B * (4 * N * N * D / 1e12 * all_pairs + N * N * 4e-9 + 4e-4 * K)
    if c["sgs_mode"] == 2:
        seconds += B * K * 20 * (4e-4 + K * N * 4e-11)
    if c["op"] not in (KNN, GATHER) and seconds > 12:
        return None
    feats, pos, frame = _inputs(c, seed)
    if c["op"] == GATHER:
        return None                   # a copy: the comparison is on its bytes
    if c["op"] == KNN:
        far = [max(float(torch.cdist(p[a:a + 2048], p).max()) for a in range(0, N, 2048)) for p in pos.double()]
        return {"nbr": None, "diameter": torch.tensor(far, dtype=torch.float64)}
    scenes = (_Scene(c, feats[b], pos[b], frame[b], max(c["n_cap"], c["g"] - 1)) for b in range(B))
    if c["op"] == COST:
        got = [(s.cost(), s.v, torch.tensor(s.norms, dtype=torch.float64)) for s in scenes]
        return {"cost": torch.stack([x[0] for x in got]), "capacity": torch.stack([x[1] for x in got]),
                "norms": torch.stack([x[2] for x in got])}
    if c["op"] == LITE:
        return {"kept": None, "group_start": None,
                "objective": torch.stack([_groups(s, pos[b], K) for b, s in enumerate(scenes)])}
    pick = _transport if c["sgs_mode"] == 2 else _greedy
    got = [pick(s, K, c["g"]) for s in scenes]
    return {"kept": None, "order": None, "gains": torch.stack([x[0] for x in got]),
            "objective": torch.stack([x[1] for x in got])}
