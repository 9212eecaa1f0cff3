"""GPU order of calls that depend on one another only through a buffer set to a value: every pass finds other valid contents in the
buffers it overwrites, so a kernel that reads ahead of its producer, or is overtaken by its successor, is seen."""
import numpy as np
import pytest
import torch

from oracle import c2r_oracle as O
from paper_2504_01337_b200 import inputs as G
from tests.util import dev, host, mask_of, random_sets

pytestmark = pytest.mark.gpu

N, E, K, T, P, D = 16384, 60, 4, 16, 4, 64


def _volume(idx, part, P):
    """O.dispatch_volume by numpy counting (naive, dedup, both send matrices), pinned to it on a sample."""
    n, k = idx.shape
    home, q = np.arange(n) * P // n, part[idx]
    first = np.array([[True] * k] * n)
    for j in range(1, k):
        first[:, j] = (q[:, :j] != q[:, j:j + 1]).all(1)
    naive, dedup = (np.bincount((home[:, None] * P + q)[m], minlength=P * P).reshape(P, P) for m in (np.ones((n, k), bool), first))
    return naive, dedup, first


def test_the_numpy_volume_is_the_oracles():
    rng = np.random.default_rng(0)
    idx = rng.permuted(np.tile(np.arange(E), (300, 1)), axis=1)[:, :K]
    part = rng.integers(0, P, E)
    ref = O.dispatch_volume(idx, part, P)
    naive, dedup, _ = _volume(idx, part, P)
    assert np.array_equal(naive, ref["send_naive"]) and np.array_equal(dedup, ref["send_dedup"])


def _count(idx):
    """Eq. 2 as a product of indicator matrices."""
    m = np.zeros((idx.shape[0], E), np.float64)
    np.put_along_axis(m, idx, 1.0, axis=1)
    return (m.T @ m).astype(np.int64)


class _Calls:
    """Buffers of a calibration and of a dispatch batch, two sets of logits, and what every pass over them has to give."""

    def __init__(self, B, n=N, seed=0):
        self.B = B
        rng = np.random.default_rng(seed)
        self.logits = [rng.standard_normal((n, E)).astype(np.float32) for _ in range(2)]
        self.part = (np.arange(E) % P).astype(np.int32)
        self.idx_ref = [O.topk_route(L, K)[0] for L in self.logits]
        self.C_ref = [_count(i) for i in self.idx_ref]
        self.sets_ref = [O.collab_sets(c, T) for c in self.C_ref]
        self.vol_ref = [_volume(i, self.part, P) for i in self.idx_ref]
        i32, i64 = dict(dtype=torch.int32, device="cuda"), dict(dtype=torch.int64, device="cuda")
        self.src = [dev(L) for L in self.logits]
        self.other = (dev(np.tile(np.arange(K, dtype=np.int32), (n, 1))), dev(np.tile(np.arange(E - K, E, dtype=np.int32), (n, 1))))
        self.cfg = B.make_config(n, D, E, 16, K, T, P, 0, B.F32, 1)
        self.L = torch.empty((n, E), device="cuda")
        self.idx, self.w = torch.zeros((n, K), **i32), torch.empty((n, K), device="cuda")
        self.C, self.I_T, self.mask = torch.zeros((E, E), **i32), torch.zeros((E, T), **i32), torch.zeros(E, **i64)
        self.vol = [torch.zeros(s, **i64) for s in ((4,), (P, P), (P, P))]
        self.part_d = dev(self.part)

    def preset(self, i):
        """Other, valid contents: the other logits' place is taken, idx names experts that routing would rarely pick."""
        self.idx.copy_(self.other[i % 2])
        self.L.copy_(self.src[i % 2])

    def calibrate(self):
        self.B.route(self.cfg, self.L, None, self.idx, self.w)
        self.B.collab_count(self.cfg, self.idx, self.cfg.N, self.C)
        self.B.collab_sets(self.cfg, self.C, self.I_T, self.mask)

    def check_calibrated(self, i, C, I_T, mask):
        assert np.array_equal(host(C), self.C_ref[i % 2])
        assert np.array_equal(host(I_T), self.sets_ref[i % 2])
        assert np.array_equal(host(mask).view(np.uint64), mask_of(self.sets_ref[i % 2], E))

    def volume(self):
        self.B.route(self.cfg, self.L, None, self.idx, self.w)
        self.B.dispatch_volume(self.cfg, self.idx, self.part_d, *self.vol)

    def check_volume(self, i, totals, naive, dedup):
        rn, rd, _ = self.vol_ref[i % 2]
        assert np.array_equal(host(naive), rn) and np.array_equal(host(dedup), rd)
        assert host(totals).tolist() == [rn.sum(), rd.sum(), rn.sum() - np.trace(rn), rd.sum() - np.trace(rd)]


@pytest.fixture(scope="module")
def calls():
    from paper_2504_01337_b200 import binding as B
    return _Calls(B)


@pytest.mark.parametrize("what", ["calibrate", "volume"])
@pytest.mark.parametrize("captured", [False, True])
def test_passes_in_a_row_with_changing_inputs(calls, what, captured):
    """Twelve passes without a synchronisation between them, eagerly and from a graph, results copied aside on the stream."""
    c = calls
    step = getattr(c, what)
    out = (c.C, c.I_T, c.mask) if what == "calibrate" else tuple(c.vol)
    c.preset(0)
    step()  # per-device set-up outside a capture
    torch.cuda.synchronize()
    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            step()
        step = graph.replay
    got = []
    for i in range(12):
        c.preset(i)
        step()
        got.append([t.clone() for t in out])
    torch.cuda.synchronize()
    for i, g in enumerate(got):
        (c.check_calibrated if what == "calibrate" else c.check_volume)(i, *g)


def test_a_fresh_count_does_not_overtake_readers_of_the_old_one(calls):
    """Routing of a large batch keeps the stream busy while sets and degree of the old counts, a fresh count and a second one
    that adds to it are queued behind it."""
    B, c = calls.B, calls
    big = 16 * N
    cfg = B.make_config(big, D, E, 16, K, T, P, 0, B.F32, 1)
    L = c.src[0].repeat(16, 1)
    idx, w = torch.zeros((big, K), dtype=torch.int32, device="cuda"), torch.empty((big, K), device="cuda")
    idx0, idx1 = (dev(i.astype(np.int32)) for i in c.idx_ref)
    deg = torch.zeros(E, device="cuda")
    for _ in range(4):
        B.collab_count(c.cfg, idx1, N, c.C)
        torch.cuda.synchronize()
        B.route(cfg, L, None, idx, w)
        B.collab_sets(c.cfg, c.C, c.I_T, c.mask)
        B.collab_degree(c.cfg, c.C, deg)
        B.collab_count(c.cfg, idx0, N, c.C)
        B.collab_count(c.cfg, idx0, N, c.C, accumulate=True)
        torch.cuda.synchronize()
        assert np.array_equal(host(c.I_T), c.sets_ref[1])
        assert np.abs(host(deg) - O.collab_degree(c.C_ref[1])[0]).max() < 1e-4
        assert np.array_equal(host(c.C), 2 * c.C_ref[0])


@pytest.mark.parametrize("n,k", [(9000, 4), (263000, 2)])
def test_dispatches_in_a_row_with_changing_inputs(n, k):
    """Routing result -> two-stage dispatch -> volume, below and beyond 1024 blocks of the counting sort, alternating between two
    batches in the same buffers and workspace: rows, receive counts and volumes of every pass."""
    from paper_2504_01337_b200 import binding as B
    e, p, d = 9, 2, 8
    rng = np.random.default_rng(n)
    part = (np.arange(e) % p).astype(np.int32)
    batches = [rng.permuted(np.tile(np.arange(e, dtype=np.int32), (n, 1)), axis=1)[:, :k].copy() for _ in range(2)]
    cfg = B.make_config(n, d, e, 16, k, 0, p, 0, B.F32, 1)
    R, cap = B.permuted_rows(cfg), n * min(k, p)
    i32, i64 = dict(dtype=torch.int32, device="cuda"), dict(dtype=torch.int64, device="cuda")
    out = {x: torch.full((m,), -7, **i32) for x, m in (("counts", e), ("offsets", e + 1), ("row_of_slot", n * k), ("slot_of_row", R),
                                                       ("recv_counts", p), ("recv_offsets", p + 1), ("recv_row_of_slot", n * k),
                                                       ("token_of_recv_row", cap))}
    vol = [torch.zeros(s, **i64) for s in ((4,), (p, p), (p, p))]
    X = dev(rng.standard_normal((n, d)).astype(np.float32))
    Xr, Xp = torch.zeros((cap, d), device="cuda"), torch.zeros((R, d), device="cuda")
    ws = torch.empty(B.workspace_bytes(cfg, B.WS_DISPATCH_DEDUP), dtype=torch.uint8, device="cuda")
    status = torch.zeros(1, **i32)
    src, idx, part_d = [dev(b) for b in batches], torch.zeros((n, k), **i32), dev(part)
    got = []
    for i in range(6):
        idx.copy_(src[i % 2])
        B.dispatch_dedup(cfg, idx, part_d, None, X, *out.values(), Xr, Xp, status, ws)
        B.dispatch_volume(cfg, idx, part_d, *vol)
        got.append([t.clone() for t in (out["recv_counts"], out["token_of_recv_row"], out["row_of_slot"], *vol)])
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    for i, (recv_counts, tokens, rows, totals, naive, dedup) in enumerate(got):
        b = batches[i % 2]
        rn, rd, first = _volume(b, part, p)
        q = part[b]
        recv = [np.nonzero((first & (q == x)).any(1))[0] for x in range(p)]
        assert host(recv_counts).tolist() == [r.size for r in recv] == rd.sum(0).tolist()
        flat = np.concatenate(recv)
        assert np.array_equal(host(tokens), np.concatenate([flat, np.full(cap - flat.size, -1)]))
        order = np.argsort(b.reshape(-1), kind="stable")
        assert np.array_equal(host(rows)[order], np.arange(n * k))
        assert np.array_equal(host(naive), rn) and np.array_equal(host(dedup), rd) and int(totals[0]) == n * k


@pytest.mark.parametrize("captured", [False, True])
def test_small_layer_with_volume(captured):
    """A layer so small that all its kernels fit the chip at once: routing and volume of every pass while the input alternates."""
    from paper_2504_01337_b200.layer import C2RLayer
    wl = G.Workload("chain", N=512, d=256, E=8, I=128, K=2, T=4, P=2, I_s=0, bf16=False, seed=5)
    Wg, _ = G.gate_weights(wl)
    sets = random_sets(wl.E, wl.T, seed=1)
    part = (np.arange(wl.E) % wl.P).astype(np.int32)
    lay = C2RLayer(wl.N, wl.d, wl.E, wl.I, wl.K, wl.T, wl.P, 0, False, backward=False)
    lay.set_params(Wg, *G.expert_weights(wl))
    lay.set_routing(mask=mask_of(sets, wl.E), part=part)
    xs = [dev(G.hidden(wl)), dev(G.hidden(wl)[::-1].copy())]
    x = torch.empty_like(xs[0])
    lay.set_input(x)
    x.copy_(xs[0])
    lay.forward()
    torch.cuda.synchronize()
    step = lay.forward
    if captured:
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            lay.forward()
        step = graph.replay
    got = []
    for i in range(8):
        x.copy_(xs[i % 2])
        lay.t["idx"].fill_(i % wl.E)
        step()
        got.append([lay.t[n].clone() for n in ("L", "idx", "volume")])
    torch.cuda.synchronize()
    for L, idx, vol in got:
        ridx, _ = O.c2r_route(host(L), sets, wl.K)
        assert np.array_equal(host(idx), ridx)
        ref = O.dispatch_volume(ridx, part, wl.P)
        v = host(vol)
        assert v[:4].tolist() == [ref["naive"], ref["dedup"], ref["naive_x"], ref["dedup_x"]]
        assert np.array_equal(v[4:8].reshape(2, 2), ref["send_naive"]) and np.array_equal(v[8:].reshape(2, 2), ref["send_dedup"])
