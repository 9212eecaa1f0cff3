"""GPU parity of the row passes (gather, weighted sum, un-permute) at the edges of their rules on batch and row length."""
import numpy as np
import pytest
import torch

from paper_2504_01337_b200 import inputs as G
from tests.util import dev, host

pytestmark = pytest.mark.gpu


def _index(B, cfg, idx):
    E, NK, R = cfg.E, cfg.N * cfg.K, B.permuted_rows(cfg)
    t = [torch.full((n,), -7, dtype=torch.int32, device="cuda") for n in (E, E + 1, NK, R)]
    ws = torch.empty(B.workspace_bytes(cfg, B.WS_PERMUTE), dtype=torch.uint8, device="cuda")
    B.permute(cfg, idx, None, None, *t, None, torch.zeros(1, dtype=torch.int32, device="cuda"), ws)
    return t, R


# several warps per token (1, 2368 tokens) against one; the split form in one wave (4736), between (4737, 7104), in two
# (7105, 9472) and past them; rows shorter than, equal to and longer than what a warp holds at once, with remainders
@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("N,d,K", [(1, 1032, 4), (2368, 264, 3), (2369, 64, 8), (4736, 8, 1), (4737, 1032, 2), (7104, 256, 4),
                                   (7105, 1024, 2), (9472, 72, 2), (9473, 264, 1), (20001, 40, 7)])
def test_combine_and_unpermute(N, d, K, bf16):
    """Against fp64 sums: fp32 accumulation of at most 10 terms of size ~1 stays below 4e-6; a bf16 result carries half an ulp more."""
    from paper_2504_01337_b200 import binding as B
    E = 9
    dt = torch.bfloat16 if bf16 else torch.float32
    rng = np.random.default_rng(N + d)
    idx = dev(rng.permuted(np.tile(np.arange(E, dtype=np.int32), (N, 1)), axis=1)[:, :K].copy())
    cfg = B.make_config(N, d, E, 16, K, 0, 1, 0, B.BF16 if bf16 else B.F32, 16)
    (counts, offsets, rows, _), R = _index(B, cfg, idx)
    Yp, Ys = (rng.standard_normal((n, d)).astype(np.float32) for n in (R, N))
    w, z, dz = (rng.standard_normal(s).astype(np.float32) for s in ((N, K), (N,), (N,)))
    Wg, wsg = (G.round_bf16(rng.standard_normal(s).astype(np.float32)) for s in ((E, d), (d,)))
    out = torch.full((N, d), 7.0, dtype=dt, device="cuda")
    r = host(rows).reshape(N, K)
    terms = sum(w[:, k:k + 1].astype(np.float64) * Yp[r[:, k]] for k in range(K))

    def check(ref):
        err = np.abs(host(out) - ref)
        assert (err <= 4e-6 * (1 + np.abs(ref)) + (2.0 ** -8 * np.abs(ref) if bf16 else 0)).all()

    B.combine(cfg, dev(Yp), dev(w), rows, dev(Ys), dev(z), out)
    check(terms + Ys / (1 + np.exp(-z.astype(np.float64)))[:, None])
    B.unpermute_grad(cfg, dev(Yp), rows, dev(Ys), idx, dev(w), dev(Wg, dt), dev(dz), dev(wsg, dt), out)
    e = host(idx)
    check(sum(Yp[r[:, k]].astype(np.float64) for k in range(K)) + Ys + dz[:, None].astype(np.float64) * wsg
          + sum(w[:, k:k + 1].astype(np.float64) * Wg[e[:, k]] for k in range(K)))


@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("N,K,d,align,used", [(2, 2, 16, 128, 2), (1, 1, 8, 128, 9), (300, 2, 264, 128, 3), (700, 8, 1032, 5, 9), (9000, 3, 64, 96, 4)])
def test_rows_without_a_slot_of_the_two_stage_dispatch_are_zero(N, K, d, align, used, bf16):
    """The rows that close each segment and the rows past the last one, with experts nobody chose: bit for bit the plain
    gather's rows, and zeros everywhere else."""
    from paper_2504_01337_b200 import binding as B
    E, P = 9, 4
    dt = torch.bfloat16 if bf16 else torch.float32
    rng = np.random.default_rng(N + K)
    pool = np.arange(max(used, K), dtype=np.int32)
    idx = dev(rng.permuted(np.tile(pool, (N, 1)), axis=1)[:, :K].copy().reshape(N, K))
    cfg = B.make_config(N, d, E, 16, K, 0, P, 0, B.BF16 if bf16 else B.F32, align)
    R, cap = B.permuted_rows(cfg), N * min(K, P)
    t = [torch.full((n,), -7, dtype=torch.int32, device="cuda") for n in (E, E + 1, N * K, R, P, P + 1, N * K, cap)]
    X = dev(rng.standard_normal((N, d)).astype(np.float32).reshape(N, d), dt)
    Xr, Xp = torch.full((cap, d), 7.0, dtype=dt, device="cuda"), torch.full((R, d), 7.0, dtype=dt, device="cuda")
    ws = torch.empty(B.workspace_bytes(cfg, B.WS_DISPATCH_DEDUP), dtype=torch.uint8, device="cuda")
    rank = dev(rng.permutation(E).astype(np.int32))
    B.dispatch_dedup(cfg, idx, dev((np.arange(E) % P).astype(np.int32)), rank, X, *t, Xr, Xp, torch.zeros(1, dtype=torch.int32, device="cuda"), ws)
    slot = host(t[3])
    ref = torch.zeros((R, d), dtype=dt, device="cuda")
    live = np.nonzero(slot >= 0)[0]
    assert live.size == N * K
    ref[dev(live)] = X[dev(slot[live] // K)]
    assert torch.equal(Xp, ref)


# a row within one group of 32 16-byte chunks per lane, exactly one, one more, and several per warp; several warps per token
@pytest.mark.parametrize("bf16", [True, False])
@pytest.mark.parametrize("N,K,d", [(1, 8, 2056), (40, 3, 264), (3000, 2, 128), (3000, 1, 256), (3000, 5, 264), (5000, 8, 1032), (5001, 4, 24)])
def test_row_gather(N, K, d, bf16):
    from paper_2504_01337_b200 import binding as B
    E = 9
    dt = torch.bfloat16 if bf16 else torch.float32
    rng = np.random.default_rng(N + d)
    idx = dev(rng.permuted(np.tile(np.arange(E, dtype=np.int32), (N, 1)), axis=1)[:, :K].copy())
    cfg = B.make_config(N, d, E, 16, K, 0, 1, 0, B.BF16 if bf16 else B.F32, 32)
    (counts, offsets, rows, slot), R = _index(B, cfg, idx)
    X = dev(rng.standard_normal((N, d)).astype(np.float32), dt)
    Xp = torch.full((R, d), 7.0, dtype=dt, device="cuda")
    B.permute_rows(cfg, X, rows, counts, offsets, Xp)
    end, s = int(offsets[E]), slot.long()
    ref = torch.full((R, d), 7.0, dtype=dt, device="cuda")  # rows past the layout are left alone
    ref[:end] = 0
    ref[s >= 0] = X[s[s >= 0] // K]
    assert torch.equal(Xp, ref)
