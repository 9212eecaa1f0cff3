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
