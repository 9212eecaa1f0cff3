"""GPU parity of the CUDA-core expert GEMMs over both tile sizes and every edge of a tile, against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import c2r_oracle as O
from paper_2504_01337_b200 import inputs as G
from tests.util import assert_close_abs, dev, host, mask_of, random_sets

pytestmark = pytest.mark.gpu


# 32-wide tiles with remainders in every direction; 64 x 64 tiles (enough rows and columns to fill the chip twice); an expert
# that gets nothing (T = K - 1 fixes every set); contractions shorter than one k-tile and no multiple of one
@pytest.mark.parametrize("N,d,E,I,K,T,I_s", [(1, 8, 4, 16, 2, 3, 0), (33, 40, 7, 48, 3, 2, 16), (500, 72, 33, 80, 2, 1, 144),
                                             (2600, 200, 5, 336, 2, 3, 208), (4000, 264, 9, 144, 4, 5, 0)])
def test_fp32_layer_over_tile_sizes(N, d, E, I, K, T, I_s):
    from paper_2504_01337_b200.layer import C2RLayer
    wl = G.Workload("simt", N=N, d=d, E=E, I=I, K=K, T=T, P=2, I_s=I_s, bf16=False, seed=6)
    X, dY = G.hidden(wl), G.grad_out(wl)
    Wg, wsg = G.gate_weights(wl)
    W1, W3, W2 = G.expert_weights(wl)
    sh = G.shared_weights(wl) if I_s else None
    sets = random_sets(E, T, seed=2)
    rank = np.random.default_rng(1).permutation(E)
    lay = C2RLayer(N, d, E, I, K, T, 2, I_s, False, backward=True)
    lay.set_params(Wg, W1, W3, W2, wsg, sh)
    lay.set_routing(mask=mask_of(sets, E), expert_rank=rank)
    lay.set_input(X, dY)
    lay.forward()
    lay.backward()
    torch.cuda.synchronize()
    assert_close_abs(lay.host("L"), O.gate_logits(X, Wg), 1e-4, "L")
    f = O.layer_fwd(X, Wg, W1, W3, W2, sets, K, expert_rank=rank, row_align=1, shared=sh, wsg=wsg, logits=lay.host("L"))
    assert np.array_equal(lay.host("idx"), f["idx"])
    assert_close_abs(lay.host("Y"), f["Y"], 1e-4, "Y")
    g = O.layer_bwd(X, Wg, W1, W3, W2, f, dY, shared=sh, wsg=wsg)
    dW1, dW3 = lay.unpacked_grads()[:2]
    # gradients sum over the expert's rows: fp32 rounding of n terms of size ~1 stays below 1e-6 sqrt(n), here under 1e-4
    for name, got, ref in (("dX", lay.host("dX"), g["dX"]), ("dW1", host(dW1), g["dW1"]), ("dW3", host(dW3), g["dW3"]),
                           ("dW2", lay.host("dW2"), g["dW2"]), ("dWg", lay.host("dWg"), g["dWg"])):
        assert_close_abs(got, ref, 1e-4 * max(1.0, float(np.abs(ref).max())), name)


@pytest.mark.parametrize("offset", [1, 2, 4])
def test_gate_logits_of_unaligned_arrays(offset):
    """Arrays that start off a 16-byte boundary take element-wise loads."""
    from paper_2504_01337_b200 import binding as B
    N, d, E = 45, 72, 9
    for bf16 in (False, True):
        dt = torch.bfloat16 if bf16 else torch.float32
        X, Wg = G.normal(1, G.S_X, (N, d)), G.normal(1, G.S_WG, (E, d), 0.02)
        if bf16:
            X, Wg = G.round_bf16(X), G.round_bf16(Wg)
        flat = torch.zeros(N * d + 16, dtype=dt, device="cuda")
        flat[offset:offset + N * d] = dev(X, dt).reshape(-1)
        L = torch.full((N, E), 7.0, device="cuda")
        cfg = B.make_config(N, d, E, 16, 2, 3, 1, 0, B.BF16 if bf16 else B.F32, 1)
        B.gate_logits(cfg, flat[offset:offset + N * d].view(N, d), dev(Wg, dt), None, L, None)
        assert_close_abs(host(L), O.gate_logits(X, Wg), 1e-4, "L")


# a batch that takes 32-wide tiles inside one that takes the large tiles in every product; contractions that end inside a part
@pytest.mark.parametrize("n,N,d,E,I,K,I_s,bf16", [(37, 4096, 200, 5, 336, 2, 0, False), (300, 4100, 264, 4, 528, 3, 400, False),
                                                  (37, 6000, 200, 5, 336, 2, 272, True)])
def test_results_of_a_token_do_not_depend_on_the_batch(n, N, d, E, I, K, I_s, bf16):
    """The CUDA-core kernels (fp32, and bf16 with d no multiple of 16), forward and backward, bit for bit."""
    from paper_2504_01337_b200.layer import C2RLayer
    wl = G.Workload("batch", N=N, d=d, E=E, I=I, K=K, T=E - 1, P=2, I_s=I_s, bf16=bf16, seed=8)
    X, dY = G.hidden(wl), G.grad_out(wl)
    Wg, wsg = G.gate_weights(wl)
    W1, W3, W2 = G.expert_weights(wl)
    sh = G.shared_weights(wl) if I_s else None
    got = []
    for m in (n, N):
        lay = C2RLayer(m, d, E, I, K, E - 1, 2, I_s, bf16, row_align=1, backward=True)
        lay.set_params(Wg, W1, W3, W2, wsg, sh)
        lay.set_routing()
        lay.set_input(X[:m], dY[:m])
        lay.forward()
        lay.backward()
        rows = lay.t["row_of_slot"].long()[:n * K]
        t = {x: lay.t[x][:n] for x in ("L", "idx", "w", "Y", "dl", "dX") + (("Ys", "dXs", "dz") if I_s else ())}
        t.update({x: lay.t[x][rows] for x in ("H", "AB", "Yp", "dAB", "dXp")})
        got.append(t)
    for x in got[0]:
        assert torch.equal(got[0][x], got[1][x]), x
