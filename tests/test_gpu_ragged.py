"""GPU parity of the forward kernel with tokens as the N operand of pair MMAs against the fp64 oracle."""
import numpy as np
import pytest
import torch

from oracle import c2r_oracle as O
from paper_2504_01337_b200 import inputs as G
from tests.util import assert_close_elem, assert_close_rms, dev, host, live_rows

pytestmark = pytest.mark.gpu


# Counts at the steps of the MMA's N (32), at the largest single MMA (256) and at the largest chunk (384), empty experts among
# them; widths below a 128-channel block, with a partial last block (rest 16 .. 112) and with a partial last k-block; enough
# units per CTA pair that neighbours share tensor memory (first and last case) and fewer units than pairs.
@pytest.mark.parametrize("counts,d,I", [([384, 1, 383, 257, 300, 0, 288, 256, 31, 352, 770, 385], 128, 1424),
                                        ([33, 64, 0, 1], 48, 16), ([890], 272, 112), ([0, 130, 0, 511, 97], 336, 128),
                                        ([320, 160, 384, 384, 290, 384, 410, 65, 384], 2320, 176)])
def test_uneven_counts(counts, d, I):
    from paper_2504_01337_b200 import binding as B
    E, align = len(counts), 128
    cfg = B.make_config(200 * E, d, E, I, 1, 0, 1, 0, B.BF16, align)  # 200 rows per expert are expected: the rule for this kernel
    offsets = np.concatenate([[0], np.cumsum([(c + align - 1) // align * align for c in counts])]).astype(np.int32)
    R = int(offsets[-1]) + 7
    rng = np.random.default_rng(4)
    Xp = G.round_bf16(rng.standard_normal((R, d)).astype(np.float32))
    W1, W3, W2 = (G.round_bf16((0.05 * rng.standard_normal(s)).astype(np.float32)) for s in ((E, I, d), (E, I, d), (E, d, I)))
    bf = torch.bfloat16
    W13p = torch.empty((E, 2 * I, d), dtype=bf, device="cuda")
    B.pack_weights(cfg, E, I, dev(W1, bf), dev(W3, bf), W13p)
    # factors below 1: a row's error grows with its factor, and at 3.5 (Gaussian factors) the largest of some 1e6 errors of
    # 1.6e-3 of the row's RMS each, 5 to 6 standard deviations out, would pass 3e-2 of the tensor's RMS
    scale = rng.random(R).astype(np.float32)
    _, _, Href, Yref = O.swiglu_fwd(Xp, np.asarray(counts), offsets, W1, W3, W2)
    rows = live_rows(np.asarray(counts), offsets)
    other = np.setdiff1d(np.arange(R), rows)
    for kind in (B.SCALE_NONE, B.SCALE_ROW, B.SCALE_SIGMOID):
        H = torch.full((R, I), 7.0, dtype=bf, device="cuda")
        Yp = torch.full((R, d), 7.0, device="cuda")
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        B.grouped_swiglu_fwd(cfg, E, I, R, dev(Xp, bf), dev(np.asarray(counts, np.int32)), dev(offsets), W13p, dev(W2, bf), None, H, Yp,
                             status, None if kind == B.SCALE_NONE else B.expert_opts(dev(scale), kind))
        torch.cuda.synchronize()
        assert int(status.item()) == 0
        s = {B.SCALE_NONE: np.ones(R), B.SCALE_ROW: scale, B.SCALE_SIGMOID: O.sigmoid(scale.astype(np.float64))}[kind][:, None]
        assert_close_elem(host(H)[rows], (s * Href)[rows], what="H")
        # bounds of tests/test_gpu_skinny.py: sums over I products with one bf16-rounded factor
        assert_close_rms(host(Yp)[rows], (s * Yref)[rows], 3e-2, "Yp", out_bf16=False)
        assert (host(Yp)[other] == 7.0).all() and (host(H)[other] == 7.0).all()  # rows of no expert are left alone
