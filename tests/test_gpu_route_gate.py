"""GPU parity of the routing kernel and of the gate's token tiles at the edges of their blocks."""
import numpy as np
import pytest
import torch

from oracle import c2r_oracle as O
from paper_2504_01337_b200 import inputs as G
from tests.util import assert_close_abs, dev, host, mask_of, random_sets

pytestmark = pytest.mark.gpu


# every K (its own blocking of the tokens), expert counts on both staging paths, token counts around a block; logits on a
# coarse grid so that most arg-max rounds are decided by the lower-index rule
@pytest.mark.parametrize("K,E,N", [(1, 5, 513), (2, 8, 256), (3, 33, 161), (4, 60, 129), (5, 64, 97), (6, 12, 79), (7, 60, 65), (8, 63, 64)])
@pytest.mark.parametrize("masked", [False, True])
def test_routing_with_ties(K, E, N, masked):
    from paper_2504_01337_b200 import binding as B
    rng = np.random.default_rng(K * 100 + E)
    L = (np.round(4 * rng.standard_normal((N, E))) / 4).astype(np.float32)
    L[rng.random((N, E)) < 0.1] = -np.inf
    L[rng.random((N, E)) < 0.1] = -0.0
    L[:, 0] = np.maximum(L[:, 0], -8.0)  # a finite logit in every row
    T = max(K - 1, 1)
    sets = random_sets(E, T, seed=K)
    cfg = B.make_config(N, 8, E, 16, K, T, 1, 0, B.F32, 1)
    idx = torch.zeros((N, K), dtype=torch.int32, device="cuda")
    w, p = torch.zeros((N, K), device="cuda"), torch.zeros((N, E), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.route(cfg, dev(L), dev(mask_of(sets, E).view(np.int64)) if masked else None, idx, w, p, status)
    ridx, rw = O.c2r_route(L, sets, K) if masked else O.topk_route(L, K)
    assert np.array_equal(host(idx), ridx)
    assert_close_abs(host(w), rw, 1e-6, "w")
    e = np.exp(L.astype(np.float64) - L.max(1, keepdims=True))
    assert_close_abs(host(p), e / e.sum(1, keepdims=True), 1e-6, "p")
    assert int(status.item()) == 0


@pytest.mark.parametrize("N,d,E,shared", [(1, 2048, 60, True), (33, 1088, 33, False), (4737, 272, 64, False), (4736, 240, 12, True),
                                          (9473, 336, 63, True), (18945, 64, 7, False)])
def test_gate_logits_do_not_depend_on_the_token_tile(N, d, E, shared):
    """Tiles of 32, 64 and 128 tokens: against the oracle (1e-4, as for whole tiles), and bit for bit against another batch size."""
    from paper_2504_01337_b200 import binding as B
    X, Wg, wsg = (G.round_bf16(G.normal(1, s, shp, sd)) for s, shp, sd in
                  ((G.S_X, (N, d), 1.0), (G.S_WG, (E, d), 0.02), (G.S_WSG, (d,), 0.02)))
    bf = torch.bfloat16

    def gate(x):
        n = x.shape[0]
        cfg = B.make_config(n, d, E, 16, 2, 3, 1, 16 if shared else 0, B.BF16, 1)
        L, z = torch.full((n, E), 7.0, device="cuda"), torch.full((n,), 7.0, device="cuda")
        B.gate_logits(cfg, x, dev(Wg, bf), dev(wsg, bf) if shared else None, L, z if shared else None)
        return L, z

    x = dev(X, bf)
    L, z = gate(x)
    assert_close_abs(host(L), O.gate_logits(X, Wg), 1e-4, "L")
    if shared:
        assert_close_abs(host(z), X.astype(np.float64) @ wsg.astype(np.float64), 1e-4, "z")
    big, zb = gate(x.repeat(20000 // N + 1, 1))
    assert torch.equal(big[:N], L) and torch.equal(zb[:N], z)


# experts in tiles of 16 and of 32, a last one that is not full, whole, or alone; contractions shorter and longer than the ring
@pytest.mark.parametrize("N,d,E,shared", [(64, 4096, 63, True), (1184, 328, 64, False), (1600, 1040, 50, True), (1600, 64, 33, False), (2300, 528, 17, True)])
def test_gate_logits_do_not_depend_on_the_expert_tile(N, d, E, shared):
    test_gate_logits_do_not_depend_on_the_token_tile(N, d, E, shared)


# expert counts at both ends of what a token's threads hold together (8, 16, 24, 32, 48, 64), a thread with fewer selections than
# rounds and with more; enough tokens for every number of threads per block, and for two threads per token of 25 to 32 experts
@pytest.mark.parametrize("E,K,N", [(2, 1, 37), (8, 8, 700), (9, 5, 700), (16, 3, 700), (17, 8, 700), (24, 2, 700), (25, 3, 700), (32, 8, 700), (33, 5, 700),
                                   (48, 8, 700), (49, 3, 700), (64, 2, 700), (17, 4, 19000), (24, 8, 9500), (33, 8, 9500), (48, 4, 19000), (49, 4, 19000), (25, 8, 76000), (32, 4, 76000), (31, 5, 76000), (60, 4, 76000), (64, 8, 38000)])
def test_route_at_the_edges_of_a_thread(E, K, N):
    from paper_2504_01337_b200 import binding as B
    rng = np.random.default_rng(E + K)
    L = (rng.integers(-6, 7, (N, E)) / 4).astype(np.float32)  # many ties
    L[rng.random((N, E)) < 0.02] = -np.inf
    nan = rng.random(N) < 0.1
    L[nan, rng.integers(0, E, N)[nan]] = np.nan
    T = max(K - 1, 1)
    sets = random_sets(E, T, seed=E) if T <= E - 1 else None
    ref = np.where(np.isnan(L), -np.inf, L)
    ref[np.isinf(ref).all(1), 0] = 0.0  # (a row of -inf alone has no weights)
    Lin = np.where(np.isinf(np.where(np.isnan(L), -np.inf, L)).all(1)[:, None], ref, L)
    i32 = dict(dtype=torch.int32, device="cuda")
    for masked in ((False, True) if sets is not None else (False,)):
        for want_p in (False, True):
            cfg = B.make_config(N, 64, E, 16, K, T, 1, 0, B.F32, 1)
            idx, w, status = torch.zeros((N, K), **i32), torch.zeros((N, K), device="cuda"), torch.zeros(1, **i32)
            p = torch.zeros((N, E), device="cuda") if want_p else None
            ws = torch.zeros(B.workspace_bytes(cfg, B.WS_PERMUTE), dtype=torch.uint8, device="cuda")
            B.route(cfg, dev(Lin), dev(mask_of(sets, E).view(np.int64)) if masked else None, idx, w, p, status, ws)
            ridx, rw = O.c2r_route(ref, sets, K) if masked else O.topk_route(ref, K)
            assert np.array_equal(host(idx), ridx)
            assert_close_abs(host(w), rw, 1e-6, "w")
            if want_p:
                e = np.exp(ref.astype(np.float64) - ref.max(1, keepdims=True))
                assert_close_abs(host(p), e / e.sum(1, keepdims=True), 1e-6, "p")
            assert int(status.item()) == 1  # NaN logits, and nothing else
            counts = host(ws.view(torch.int32))[:ws.numel() // 4 // E * E].reshape(-1, E).sum(0)
            assert np.array_equal(counts, np.bincount(ridx.ravel(), minlength=E))


# whole tiles of 16, 32, 48 and 64 experts, with and without the shared gate, against the general form (a batch below 64 tokens per
# SM): contractions of one k-block, with a partial last one and longer than the ring; the first E of each tile's range and the last
@pytest.mark.parametrize("N,d,E,shared", [(77, 64, 2, True), (77, 1096, 16, False), (300, 72, 17, False), (300, 712, 32, True), (1000, 136, 33, True),
                                          (1000, 704, 48, True), (9472, 200, 49, False), (9472, 72, 63, True)])
def test_gate_logits_of_whole_tiles(N, d, E, shared):
    test_gate_logits_do_not_depend_on_the_token_tile(N, d, E, shared)


@pytest.mark.parametrize("N,K,P", [(1, 3, 4), (150, 7, 2), (1700, 6, 5), (40000, 4, 3), (525000, 1, 3), (263000, 2, 1),
                                   (176000, 3, 2)])
def test_two_stage_dispatch_against_numpy(N, K, P):
    """Both index paths (up to and beyond 1024 blocks of the counting sort), tokens that meet a partition several times; the
    receive side is a stable sort of the first slots by partition, so numpy gives it directly."""
    from paper_2504_01337_b200 import binding as B
    E, d, align = 9, 8, 4
    rng = np.random.default_rng(N + K)
    idx = rng.permuted(np.tile(np.arange(E, dtype=np.int32), (N, 1)), axis=1)[:, :K].copy()
    part = (np.arange(E) % P).astype(np.int32)
    X = rng.standard_normal((N, d)).astype(np.float32)
    cfg = B.make_config(N, d, E, 16, K, 0, P, 0, B.F32, align)
    R, cap = B.permuted_rows(cfg), N * min(K, P)
    i32 = dict(dtype=torch.int32, device="cuda")
    out = {k: torch.full((n,), -7, **i32) for k, n in (("counts", E), ("offsets", E + 1), ("row_of_slot", N * K), ("slot_of_row", R),
                                                       ("recv_counts", P), ("recv_offsets", P + 1), ("recv_row_of_slot", N * K),
                                                       ("token_of_recv_row", cap))}
    Xr, Xp = torch.full((cap, d), 7.0, device="cuda"), torch.full((R, d), 7.0, device="cuda")
    status = torch.zeros(1, **i32)
    ws = torch.empty(B.workspace_bytes(cfg, B.WS_DISPATCH_DEDUP), dtype=torch.uint8, device="cuda")
    B.dispatch_dedup(cfg, dev(idx), dev(part), None, dev(X), *out.values(), Xr, Xp, status, ws)
    got = {k: host(v) for k, v in out.items()}
    assert int(status.item()) == 0
    # per-expert layout: a stable sort of the slots by expert, segments aligned
    flat = idx.reshape(-1)
    counts = np.bincount(flat, minlength=E)
    offsets = np.concatenate([[0], np.cumsum((counts + align - 1) // align * align)])
    order = np.argsort(flat, kind="stable")
    rank = np.arange(N * K) - np.repeat(np.cumsum(counts) - counts, counts)
    row_of_slot = np.empty(N * K, np.int64)
    row_of_slot[order] = offsets[flat[order]] + rank
    assert np.array_equal(got["counts"], counts) and np.array_equal(got["offsets"], offsets)
    assert np.array_equal(got["row_of_slot"], row_of_slot)
    # receive side
    q = part[idx]
    first = np.stack([(q[:, :k] != q[:, k:k + 1]).all(1) for k in range(K)], axis=1)
    slots = np.nonzero(first.reshape(-1))[0]
    qs = q.reshape(-1)[slots]
    recv = slots[np.argsort(qs, kind="stable")]
    assert np.array_equal(got["recv_counts"], np.bincount(qs, minlength=P))
    assert np.array_equal(got["recv_offsets"], np.concatenate([[0], np.cumsum(np.bincount(qs, minlength=P))]))
    assert np.array_equal(got["token_of_recv_row"], np.concatenate([recv // K, np.full(cap - recv.size, -1)]))
    Xph = np.zeros((R, d), np.float32)
    Xph[row_of_slot] = np.repeat(X, K, axis=0)
    assert np.array_equal(host(Xp), Xph) and np.array_equal(host(Xr)[:recv.size], X[recv // K])
    rrs = got["recv_row_of_slot"]
    assert np.array_equal(got["token_of_recv_row"][rrs], np.repeat(np.arange(N), K))
    assert ((rrs[:, None] >= got["recv_offsets"][None, :-1]) & (rrs[:, None] < got["recv_offsets"][None, 1:])).argmax(1).tolist() == q.reshape(-1).tolist()


# full softmax by warps: every K at its block size, one token, a batch of one block, two warps' worth of experts; N on both
# sides of the line on blocks (592 blocks of 64 tokens) and of a small batch (128 tokens)
@pytest.mark.parametrize("K,E,N", [(1, 33, 128), (1, 33, 129), (2, 64, 1), (3, 60, 127), (4, 33, 130), (5, 60, 97), (6, 64, 161), (7, 33, 65),
                                   (8, 60, 1), (8, 34, 592 * 64), (8, 34, 592 * 64 + 1)])
@pytest.mark.parametrize("renorm", [0, 1])
def test_full_softmax_of_small_batches(K, E, N, renorm):
    from paper_2504_01337_b200 import binding as B
    rng = np.random.default_rng(K * 100 + E + N)
    L = (2 * rng.standard_normal((N, E))).astype(np.float32)
    L[rng.random((N, E)) < 0.05] = -np.inf
    L[:, E - 1] = np.maximum(L[:, E - 1], -8.0)  # a finite logit in every row
    cfg = B.make_config(N, 8, E, 16, K, K, 1, 0, B.F32, 1, renorm)
    idx, w, p = torch.zeros((N, K), dtype=torch.int32, device="cuda"), torch.zeros((N, K), device="cuda"), torch.zeros((N, E), device="cuda")
    B.route(cfg, dev(L), None, idx, w, p)
    ridx, rw = O.topk_route(L, K, bool(renorm))
    assert np.array_equal(host(idx), ridx)
    # expf and a division: a few units in the last place of values up to 1
    assert_close_abs(host(w), rw, 1e-6, "w")
    assert_close_abs(host(p), O.softmax_rows(L), 1e-6, "p")


# blocks of the ranking at two, three, four, eight and nine per SM, where its share of an SM's shared memory changes
@pytest.mark.parametrize("N,K,P", [(9600, 4, 3), (19100, 4, 9), (28600, 4, 1), (66300, 4, 3), (75900, 4, 4)])
def test_two_stage_dispatch_at_the_edges_of_a_share(N, K, P):
    test_two_stage_dispatch_against_numpy(N, K, P)
