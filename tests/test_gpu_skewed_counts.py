"""Expert call that keeps nothing for a backward pass, with routing skewed so far that the mean says nothing, against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import c2r_oracle as O
from paper_2504_01337_b200 import inputs as G
from tests.util import assert_close_elem, assert_close_rms, dev, host, live_rows

pytestmark = pytest.mark.gpu


# The counts that 11500 tokens of the skewed-logits recipe give 60 experts (mean 767), and a tenth of them (mean 77): four experts
# with nearly every token, a falling tail, most experts empty.
@pytest.mark.parametrize("tenth", [False, True])
def test_most_rows_in_four_experts(tenth):
    from paper_2504_01337_b200 import binding as B
    E, K, d, I, align = 60, 4, 128, 144, 128
    counts = np.zeros(E, np.int64)
    counts[:18] = [11488, 11435, 11085, 10296, 813, 428, 200, 114, 55, 32, 23, 13, 13, 0, 2, 0, 1, 2]
    if tenth:
        counts = (counts + 9) // 10
    cfg = B.make_config(int(counts.sum()) // K, d, E, I, K, 3, 1, 0, B.BF16, align)
    offsets = np.concatenate([[0], np.cumsum((counts + align - 1) // align * align)]).astype(np.int32)
    R = int(offsets[-1]) + 128
    rng = np.random.default_rng(8)
    Xp = G.round_bf16(rng.standard_normal((R, d)).astype(np.float32))
    W1, W3, W2 = (G.round_bf16((0.05 * rng.standard_normal(s)).astype(np.float32)) for s in ((E, I, d), (E, I, d), (E, d, I)))
    bf = torch.bfloat16
    W13p = torch.empty((E, 2 * I, d), dtype=bf, device="cuda")
    B.pack_weights(cfg, E, I, dev(W1, bf), dev(W3, bf), W13p)
    rows = live_rows(counts, offsets)
    got = []
    for AB in (None, torch.empty((R, 2 * I), dtype=bf, device="cuda")):
        H, Yp = torch.empty((R, I), dtype=bf, device="cuda"), torch.empty((R, d), device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        for _ in range(3):
            B.grouped_swiglu_fwd(cfg, E, I, R, dev(Xp, bf), dev(counts.astype(np.int32)), dev(offsets), W13p, dev(W2, bf), AB, H, Yp, status)
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        got.append((host(H)[rows], host(Yp)[rows]))
    assert all(np.array_equal(a, b) for a, b in zip(*got))  # the same bits whether or not a backward pass follows
    _, _, Href, Yref = O.swiglu_fwd(Xp, counts, offsets, W1, W3, W2)
    assert_close_elem(got[0][0], Href[rows], what="H")
    # bound of tests/test_gpu_skinny.py: sums over I products with one bf16-rounded factor
    assert_close_rms(got[0][1], Yref[rows], 3e-2, "Yp", out_bf16=False)
