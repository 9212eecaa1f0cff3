"""fp32 gate logits: each one chain of products in k order, whatever the batch, the tile and the alignment."""
import numpy as np
import pytest
import torch

from tests.util import dev, host

pytestmark = pytest.mark.gpu


# batches below, at and above one block per SM; tiles of one and of eight outputs per thread; contractions that fit one buffer and
# that take several with a remainder; a gate of one row and of 64
@pytest.mark.parametrize("N,d,E,shared", [(1, 8, 1, False), (149, 264, 8, True), (512, 256, 7, False), (1300, 512, 63, True), (1500, 3400, 33, True),
                                          (4736, 72, 64, False), (4737, 520, 60, True), (9000, 64, 12, False)])
def test_gate_logits_fp32(N, d, E, shared):
    from paper_2504_01337_b200 import binding as B
    rng = np.random.default_rng(3)
    X, Wg, wsg = (rng.standard_normal(s).astype(np.float32) for s in ((N, d), (E, d), (d,)))

    def gate(x, w, v):
        n = x.shape[0]
        L, z = torch.full((n, E), 9.0, device="cuda"), torch.full((n,), 9.0, device="cuda")
        B.gate_logits(B.make_config(n, d, E, 16, 1, 0, 1, 16 if shared else 0, B.F32, 1), x, w, v if shared else None, L, z if shared else None)
        return L, z

    dX, dW, dv = dev(X), dev(Wg), dev(wsg)
    L, z = gate(dX, dW, dv)
    W = np.concatenate([Wg, wsg[None]]) if shared else Wg
    got = np.concatenate([host(L), host(z)[:, None]], 1) if shared else host(L)
    # a chain of d products in fp32: each rounding is at most 2^-24 of a partial sum, and those are below the sum of magnitudes
    bound = d * 2.0 ** -24 * (np.abs(X).astype(np.float64) @ np.abs(W).astype(np.float64).T)
    assert (np.abs(got - X.astype(np.float64) @ W.astype(np.float64).T) <= bound).all()
    # the same bits from other batches and from rows that lie on no 16-byte boundary
    n = min(N, 37)
    assert all(torch.equal(a[:n], b) for a, b in zip((L, z), gate(dX[:n].contiguous(), dW, dv)))
    shifted = torch.empty(N * d + 1, device="cuda")[1:].view(N, d)
    shifted.copy_(dX)
    assert all(torch.equal(a, b) for a, b in zip((L, z), gate(shifted, dW, dv)))
