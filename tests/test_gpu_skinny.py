"""GPU parity of the weight-streaming expert kernels (a handful of rows per expert) against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import c2r_oracle as O
from paper_2504_01337_b200 import inputs as G
from tests.util import assert_close_elem, assert_close_rms, dev, host, live_rows, mask_of, random_sets, row_weights

pytestmark = pytest.mark.gpu


# token counts at the edges of the 16-column MMA tile and of the 48-row rule; widths below one k-block, with a partial last
# k-block and with a partial last 128-channel block of the packed layout; with and without the shared expert in the launch
@pytest.mark.parametrize("N,d,E,I,K,T,I_s", [(1, 16, 4, 16, 2, 3, 0), (1, 2048, 8, 272, 4, 6, 1024), (16, 64, 3, 48, 1, 2, 16),
                                             (17, 80, 33, 112, 4, 9, 112), (33, 336, 5, 688, 2, 3, 144), (65, 256, 8, 400, 4, 5, 528),
                                             (128, 128, 12, 160, 3, 4, 208), (192, 1024, 16, 128, 4, 8, 0)])
def test_forward_with_few_rows_per_expert(N, d, E, I, K, T, I_s):
    from paper_2504_01337_b200.layer import C2RLayer
    wl = G.Workload("skinny", N=N, d=d, E=E, I=I, K=K, T=T, P=2, I_s=I_s, bf16=True, seed=3)
    X = G.hidden(wl)
    Wg, wsg = G.gate_weights(wl)
    W1, W3, W2 = G.expert_weights(wl)
    sh = G.shared_weights(wl) if I_s else None
    sets = random_sets(E, T, seed=7)
    rank = np.random.default_rng(9).permutation(E)
    lay = C2RLayer(N, d, E, I, K, T, 2, I_s, True, backward=False)
    lay.set_params(Wg, W1, W3, W2, wsg, sh)
    lay.set_routing(mask=mask_of(sets, E), expert_rank=rank)
    lay.set_input(X)
    lay.forward()
    torch.cuda.synchronize()
    assert int(lay.t["status"].item()) == 0
    f = O.layer_fwd(X, Wg, W1, W3, W2, sets, K, expert_rank=rank, row_align=lay.cfg.row_align, shared=sh, wsg=wsg,
                    logits=lay.host("L"))
    assert np.array_equal(lay.host("idx"), f["idx"])
    rows, wr = live_rows(f["counts"], f["offsets"]), row_weights(f)[:, None]
    n = f["slot_of_row"].size
    assert_close_elem(lay.host("H")[:n][rows], (wr * f["H"])[rows], what="H")
    # an element of Yp is a sum over I products with one bf16-rounded factor (standard deviation 2^-9 / sqrt(3) of it):
    # 3e-2 of the RMS is over 20 standard deviations for Gaussian sums, and leaves room for the few-term sums of I = 16
    assert_close_rms(lay.host("Yp")[:n][rows], (wr * f["Yp"])[rows], 3e-2, "Yp", out_bf16=False)
    assert_close_rms(lay.host("Y"), f["Y"], 3e-2, "Y")


@pytest.mark.parametrize("counts", [[0, 37, 1, 16, 0, 140], [300, 0, 0, 0, 0, 0], [0, 0, 0, 0, 0, 0]])
def test_uneven_counts_take_the_same_kernel(counts):
    """Counts the host cannot foresee: empty experts, several token chunks per expert, one expert with everything."""
    from paper_2504_01337_b200 import binding as B
    E, d, I, align = len(counts), 192, 176, 128
    cfg = B.make_config(100, d, E, I, 2, 3, 1, 0, B.BF16, align)
    offsets = np.concatenate([[0], np.cumsum([(c + align - 1) // align * align for c in counts])]).astype(np.int32)
    R = int(offsets[-1]) + 7
    rng = np.random.default_rng(4)
    Xp = G.round_bf16(rng.standard_normal((R, d)).astype(np.float32))
    W1, W3, W2 = (G.round_bf16((0.05 * rng.standard_normal(s)).astype(np.float32)) for s in ((E, I, d), (E, I, d), (E, d, I)))
    bf = torch.bfloat16
    W13p = torch.empty((E, 2 * I, d), dtype=bf, device="cuda")
    B.pack_weights(cfg, E, I, dev(W1, bf), dev(W3, bf), W13p)
    H = torch.full((R, I), 7.0, dtype=bf, device="cuda")
    Yp = torch.full((R, d), 7.0, device="cuda")
    scale = rng.random(R).astype(np.float32)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    B.grouped_swiglu_fwd(cfg, E, I, R, dev(Xp, bf), dev(np.asarray(counts, np.int32)), dev(offsets), W13p, dev(W2, bf), None, H, Yp,
                         status, B.expert_opts(dev(scale), B.SCALE_ROW))
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    _, _, Href, Yref = O.swiglu_fwd(Xp, np.asarray(counts), offsets, W1, W3, W2)
    rows = live_rows(np.asarray(counts), offsets)
    s = scale[:, None].astype(np.float64)
    if rows.size:
        assert_close_elem(host(H)[rows], (s * Href)[rows], what="H")
        assert_close_rms(host(Yp)[rows], (s * Yref)[rows], 3e-2, "Yp", out_bf16=False)
    other = np.setdiff1d(np.arange(R), rows)  # rows that belong to no expert are left alone
    assert (host(Yp)[other] == 7.0).all() and (host(H)[other] == 7.0).all()


@pytest.mark.parametrize("n", [1, 17, 100, 129])
def test_a_token_gets_the_same_bits_from_either_kernel(n):
    """Batches on both sides of the rule, alone and with the shared expert in the launch, against a large batch's first tokens."""
    from paper_2504_01337_b200.layer import C2RLayer
    wl = G.Workload("either", N=1500, d=336, E=8, I=400, K=3, T=4, P=2, I_s=528, bf16=True, seed=11)
    X = G.hidden(wl)
    Wg, wsg = G.gate_weights(wl)
    W, sh, sets = G.expert_weights(wl), G.shared_weights(wl), random_sets(wl.E, wl.T, seed=5)
    got = []
    for m in (n, wl.N):
        lay = C2RLayer(m, wl.d, wl.E, wl.I, wl.K, wl.T, wl.P, wl.I_s, True, backward=False)
        lay.set_params(Wg, *W, wsg, sh)
        lay.set_routing(mask=mask_of(sets, wl.E))
        lay.set_input(X[:m])
        lay.forward()
        rows = lay.t["row_of_slot"].long()[:n * wl.K]
        got.append([lay.t[x][:n] for x in ("L", "idx", "Ys", "Hs", "Y")] + [lay.t[x][rows] for x in ("H", "Yp")])
    assert all(torch.equal(a, b) for a, b in zip(*got))


@pytest.mark.parametrize("n", [1, 100, 200])
def test_a_forward_pass_has_the_same_bits_when_a_backward_pass_follows(n):
    """The kernels that keep nothing (streaming, alone and with the shared expert in the launch, and pair tiles) against the one that
    keeps the local derivatives."""
    from paper_2504_01337_b200.layer import C2RLayer
    wl = G.Workload("kept", N=n, d=336, E=8, I=400, K=3, T=4, P=2, I_s=528, bf16=True, seed=11)
    X = G.hidden(wl)
    Wg, wsg = G.gate_weights(wl)
    W, sh, sets = G.expert_weights(wl), G.shared_weights(wl), random_sets(wl.E, wl.T, seed=5)
    got = []
    for backward in (False, True):
        lay = C2RLayer(n, wl.d, wl.E, wl.I, wl.K, wl.T, wl.P, wl.I_s, True, backward=backward)
        lay.set_params(Wg, *W, wsg, sh)
        lay.set_routing(mask=mask_of(sets, wl.E))
        lay.set_input(X)
        lay.forward()
        rows = lay.t["row_of_slot"].long()
        got.append([lay.t[x] for x in ("L", "idx", "Ys", "Hs", "Y")] + [lay.t[x][rows] for x in ("H", "Yp")])
    assert all(torch.equal(a, b) for a, b in zip(*got))
