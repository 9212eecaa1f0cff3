"""CUDA-core expert GEMMs on arrays that start off a 16-byte boundary (element-wise loads): the same bits as on aligned ones."""
import pytest
import torch

pytestmark = pytest.mark.gpu


# contractions with a remainder beyond a 32-wide tile and shorter than one; tiles of 32 and (last case) of 64; an empty expert
@pytest.mark.parametrize("bf16,offset", [(False, 1), (False, 2), (True, 1), (True, 4)])
@pytest.mark.parametrize("counts,d,I", [([37, 0, 5, 64], 40, 48), ([1, 2], 8, 16), ([700, 650, 800], 520, 144)])
def test_unaligned_arrays(counts, d, I, bf16, offset):
    from paper_2504_01337_b200 import binding as B
    E, R = len(counts), sum(counts)
    dt = torch.bfloat16 if bf16 else torch.float32
    cfg = B.make_config(R, d, E, I, 1, 0, 1, 0, B.BF16 if bf16 else B.F32, 1)  # several experts, rows not aligned to 128: off the tensor cores
    g = torch.Generator(device="cuda").manual_seed(d)
    cnt = torch.tensor(counts, dtype=torch.int32, device="cuda")
    off = torch.tensor([sum(counts[:i]) for i in range(E + 1)], dtype=torch.int32, device="cuda")
    shapes = dict(X=(R, d), W13=(E, 2 * I, d), W2=(E, d, I), dY=(R, d))
    flat = {k: torch.empty(torch.Size(s).numel(), dtype=dt, device="cuda").normal_(0, 0.3, generator=g) for k, s in shapes.items()}

    def run(shift):
        t = {}
        for k, s in shapes.items():
            a = torch.zeros(flat[k].numel() + 16, dtype=dt, device="cuda")
            a[shift:shift + flat[k].numel()] = flat[k]
            t[k] = a[shift:shift + flat[k].numel()].view(s)
        AB, H, Yp = torch.empty((R, 2 * I), dtype=dt, device="cuda"), torch.empty((R, I), dtype=dt, device="cuda"), torch.empty((R, d), device="cuda")
        dAB, dXp, dW13, dW2 = torch.empty_like(AB), torch.empty_like(Yp), torch.empty_like(t["W13"]), torch.empty_like(t["W2"])
        B.grouped_swiglu_fwd(cfg, E, I, R, t["X"], cnt, off, t["W13"], t["W2"], AB, H, Yp)
        B.grouped_swiglu_bwd(cfg, E, I, R, t["X"], cnt, off, t["W13"], t["W2"], AB, H, t["dY"], dAB, dXp, dW13, dW2)
        torch.cuda.synchronize()
        return AB, H, Yp, dAB, dXp, dW13, dW2

    assert all(torch.isfinite(a).all() and torch.equal(a, b) for a, b in zip(run(0), run(offset)))


# bf16 arrays on a 4-byte boundary and no better one
@pytest.mark.parametrize("counts,d,I", [([37, 0, 5, 64], 40, 48), ([700, 650, 800], 520, 144)])
def test_arrays_on_a_four_byte_boundary(counts, d, I):
    test_unaligned_arrays(counts, d, I, True, 2)


# launches small enough for a ring of two stages and larger ones; contractions of one tile, of a few and with a remainder
@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("d,I", [(256, 128), (24, 16), (520, 48)])
def test_two_stages_and_four_give_the_same_bits(d, I, bf16):
    from paper_2504_01337_b200 import binding as B
    E, few, many = 8, 40, 1200
    dt = torch.bfloat16 if bf16 else torch.float32
    g = torch.Generator(device="cuda").manual_seed(d)
    X, dY = (torch.empty((E, many, d), device="cuda").normal_(0, 0.5, generator=g).to(dt) for _ in range(2))
    W13, W2 = (torch.empty(s, device="cuda").normal_(0, 0.1, generator=g).to(dt) for s in ((E, 2 * I, d), (E, d, I)))
    got = []
    for n in (few, many):
        R = E * n
        cfg = B.make_config(R, d, E, I, 1, 0, 1, 0, B.BF16 if bf16 else B.F32, 1)
        cnt = torch.full((E,), n, dtype=torch.int32, device="cuda")
        off = torch.arange(E + 1, dtype=torch.int32, device="cuda") * n
        x, dy = X[:, :n].reshape(R, d).contiguous(), dY[:, :n].reshape(R, d).contiguous()
        AB, H, Yp = torch.empty((R, 2 * I), dtype=dt, device="cuda"), torch.empty((R, I), dtype=dt, device="cuda"), torch.empty((R, d), device="cuda")
        dAB, dXp, dW13, dW2 = torch.empty_like(AB), torch.empty_like(Yp), torch.empty_like(W13), torch.empty_like(W2)
        B.grouped_swiglu_fwd(cfg, E, I, R, x, cnt, off, W13, W2, AB, H, Yp)
        B.grouped_swiglu_bwd(cfg, E, I, R, x, cnt, off, W13, W2, AB, H, dy, dAB, dXp, dW13, dW2)
        got.append([t.view(E, n, -1)[:, :few] for t in (AB, H, Yp, dAB, dXp)])
        # the weight gradients from the stored dY, H, dAB and X: sums of n products, each rounding at most 2^-24 of the sum of
        # magnitudes, and for bf16 the rounding of the result
        for dW, a, b in ((dW2, dy, H), (dW13, dAB, x)):
            a, b = a.view(E, n, -1).double(), b.view(E, n, -1).double()
            ref, mag = a.transpose(1, 2) @ b, a.abs().transpose(1, 2) @ b.abs()
            assert ((dW.double() - ref).abs() <= n * 2.0 ** -24 * mag + (2.0 ** -8 * ref.abs() if bf16 else 0)).all()
    assert all(torch.equal(a, b) for a, b in zip(*got))
