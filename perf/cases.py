"""What this library is used for, as cases that can be timed and compared: whole layers at inference and in training, and
the calls around them that profile routing and carry out the dispatch.

A case is a dict of plain values.  `kind` says which calls a pass makes:

  forward    C2RLayer.forward, nothing kept for a backward pass (serving: decode steps and prefill)
  train      C2RLayer.train_step (forward, backward, Eq. 2 / Eq. 4 refresh, dispatch volume)
  steps      the forward pass call by call from gate logits that are given (routing studies on skewed logits)
  calibrate  gate logits -> Top-K -> collaboration counts -> sets (profiling batch of Sec. 3.3, step 1)
  dispatch   C2R routing -> two-stage dispatch of Sec. 3.4 with the rows -> dispatch volume

Sizes follow the workloads of `paper_2504_01337_b200.inputs` and of the tests.
"""
from __future__ import annotations

import math

import torch

from paper_2504_01337_b200 import binding as B
from paper_2504_01337_b200.layer import C2RLayer

_QWEN = dict(d=2048, E=60, I=1408, K=4, T=16, P=4, I_s=5632, bf16=True)   # workloads c3, c4, c5
_LLAMA = dict(d=4096, E=16, I=688, K=4, T=8, P=4, I_s=0, bf16=True)       # workload c2
_TINY = dict(d=256, E=8, I=128, K=2, T=4, P=2, I_s=0, bf16=False)         # workload c1


def listed():
    return [
        # one token of one sequence: the smallest call of a serving loop, latency and launches count
        dict(name="decode-1", kind="forward", N=1, **_QWEN),
        # a decode step of a batch of sequences: every expert's weights are read for a handful of rows each
        dict(name="decode-64", kind="forward", N=64, **_QWEN),
        # a ragged prompt through the LLaMA-MoE-shaped layer (expert width no multiple of a tile)
        dict(name="prefill-1021", kind="forward", N=1021, **_LLAMA),
        # an ordinary prefill chunk of the Qwen-MoE-shaped layer
        dict(name="prefill-4096", kind="forward", N=4096, **_QWEN),
        # the exact-arithmetic configuration: a tiny fp32 layer, forward only (workload c1)
        dict(name="forward-fp32", kind="forward", N=512, **_TINY),
        # the same layer trained in fp32 on a ragged batch: gradient checks and small experiments
        dict(name="train-fp32", kind="train", N=1500, **_TINY),
        # training step of the LLaMA-MoE-shaped layer (workload c2)
        dict(name="train-llama", kind="train", N=8192, **_LLAMA),
        # training step of the Qwen-MoE-shaped layer (workload c3, the default of the benchmark)
        dict(name="train-qwen", kind="train", N=16384, **_QWEN),
        # the large-batch training step (workload c5): the largest call
        dict(name="train-qwen-large", kind="train", N=65536, **_QWEN),
        # skewed routing (workload c4): most tokens meet in a few experts, most experts are empty
        dict(name="skewed-forward", kind="steps", N=16384, **_QWEN),
        # profiling batch from which the collaborator sets are built
        dict(name="calibrate", kind="calibrate", N=16384, **_QWEN),
        # one copy of a token per partition, then replication inside the partition
        dict(name="dispatch-two-stage", kind="dispatch", N=16384, **_QWEN),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: every kind, token counts from one to the large batch, widths that are no multiple of a tile among them."""
    while True:
        kind = rng.choice(["forward", "forward", "forward", "train", "train", "train", "steps", "calibrate", "dispatch"])
        bf16 = kind in ("calibrate", "dispatch") or rng.random() < 0.8
        E = rng.choice([4, 7, 8, 12, 16, 24, 33, 48, 60])
        K = rng.randint(1, min(8, E - 1, 6))
        T = rng.randint(max(K - 1, 1), E - 1)
        P = rng.choice([p for p in (1, 2, 3, 4, 6, 8) if p <= E])
        if bf16:
            step = rng.choice([16, 64, 128])
            d = max(2, _log_int(rng, 256, 4096) // step) * step
            I = max(1, _log_int(rng, 128, 2816) // 16) * 16
            I_s = rng.choice([0, 0, max(1, _log_int(rng, 256, 5632) // 16) * 16])
            N = _log_int(rng, 256 if kind == "train" else 1, 65536)
        else:
            d = max(1, _log_int(rng, 64, 512) // 8) * 8
            I = max(1, _log_int(rng, 32, 512) // 16) * 16
            I_s = rng.choice([0, 0, max(1, _log_int(rng, 32, 512) // 16) * 16])
            N = _log_int(rng, 64 if kind == "train" else 1, 4096)
        if N < {"steps": 16, "calibrate": 64, "dispatch": 64}.get(kind, 1):
            continue
        c = dict(kind=kind, N=N, d=d, E=E, I=I, K=K, T=T, P=P, I_s=I_s, bf16=bf16)
        if kind == "train" and bf16 and rng.random() < 0.25:  # options of the layer: fused combine, second stream
            c["fused_combine"] = True
            c["side_stream"] = I_s > 0
        w, top = work(c), work(dict(kind="train", N=65536, **_QWEN))
        rows = N * K + 128 * E
        if w["flops"] <= top["flops"] and w["bytes"] <= top["bytes"] and rows * (d + I) <= 65536 * 4 * 3456 + 128 * 60 * 3456:
            return c


# ---- inputs ---------------------------------------------------------------------------------------------------------

def _normal(g, shape, dt, std=1.0):
    return torch.empty(shape, dtype=dt, device="cuda").normal_(0.0, std, generator=g)


def _skewed_logits(g, N, E, d):
    """Recipe of `inputs.skewed_logits`: Zipf-like expert bias and a bonus on the rest of the leading expert's block of four."""
    L = _normal(g, (N, E), torch.float32, 0.02 * math.sqrt(d))
    L -= 2.0 * torch.log(torch.arange(1, E + 1, device="cuda", dtype=torch.float32))[None, :]
    lead = L.argmax(1, keepdim=True)
    cols = torch.arange(E, device="cuda")[None, :]
    return L + 1.5 * ((cols // 4 == lead // 4) & (cols != lead)).float()


def _calibrated(case, g, Wg, dt, logits=None):
    """(mask, expert_rank, part): collaborator sets and placement from a calibration batch under conventional Top-K."""
    E, K, T, P = case["E"], case["K"], case["T"], case["P"]
    n = 4096
    cfg = B.make_config(n, case["d"], E, case["I"], K, T, P, 0, B.BF16 if case["bf16"] else B.F32, 1)
    if logits is None:
        logits = torch.empty((n, E), device="cuda")
        B.gate_logits(cfg, _normal(g, (n, case["d"]), dt), Wg, None, logits, None)
    idx = torch.empty((n, K), dtype=torch.int32, device="cuda")
    B.route(cfg, logits, None, idx, torch.empty((n, K), device="cuda"))
    C = torch.zeros((E, E), dtype=torch.int32, device="cuda")
    B.collab_count(cfg, idx, n, C)
    mask = torch.zeros((E,), dtype=torch.int64, device="cuda")
    B.collab_sets(cfg, C, torch.zeros((E, T), dtype=torch.int32, device="cuda"), mask)
    part, rank = torch.zeros(E, dtype=torch.int32), torch.zeros(E, dtype=torch.int32)
    B.place_experts(cfg, C.cpu(), 0, part, rank)
    return mask, rank.cuda(), part.cuda()


def _packed(cfg, g, n_experts, I, d, dt):
    w1, w3 = _normal(g, (n_experts, I, d), dt, 0.02), _normal(g, (n_experts, I, d), dt, 0.02)
    out = torch.empty((n_experts, 2 * I, d), dtype=dt, device="cuda")
    B.pack_weights(cfg, n_experts, I, w1, w3, out)
    return out, _normal(g, (n_experts, d, I), dt, 0.02)


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    N, d, E, I, K, T, P, I_s = (case[k] for k in ("N", "d", "E", "I", "K", "T", "P", "I_s"))
    dt = torch.bfloat16 if case["bf16"] else torch.float32
    kind = case["kind"]
    Wg = _normal(g, (E, d), dt, 0.02)
    X = _normal(g, (N, d), dt)
    i32 = dict(dtype=torch.int32, device="cuda")

    if kind == "calibrate":
        cfg = B.make_config(N, d, E, I, K, T, P, 0, B.BF16, 1)
        return dict(kind=kind, cfg=cfg, N=N, X=X, Wg=Wg, L=torch.empty((N, E), device="cuda"), idx=torch.empty((N, K), **i32),
                    w=torch.empty((N, K), device="cuda"), C=torch.empty((E, E), **i32), I_T=torch.empty((E, T), **i32),
                    mask=torch.empty((E,), dtype=torch.int64, device="cuda"))

    if kind == "dispatch":
        mask, rank, part = _calibrated(case, g, Wg, dt)
        cfg = B.make_config(N, d, E, I, K, T, P, 0, B.BF16, 128)
        L = torch.empty((N, E), device="cuda")
        B.gate_logits(cfg, X, Wg, None, L, None)
        R, cap = B.permuted_rows(cfg), N * min(K, P)
        s = dict(kind=kind, cfg=cfg, X=X, L=L, mask=mask, rank=rank, part=part, idx=torch.empty((N, K), **i32),
                 w=torch.empty((N, K), device="cuda"), counts=torch.empty(E, **i32), offsets=torch.empty(E + 1, **i32),
                 row_of_slot=torch.empty(N * K, **i32), slot_of_row=torch.empty(R, **i32), recv_counts=torch.empty(P, **i32),
                 recv_offsets=torch.empty(P + 1, **i32), recv_row_of_slot=torch.empty(N * K, **i32),
                 token_of_recv_row=torch.empty(cap, **i32), Xr=torch.zeros((cap, d), dtype=dt, device="cuda"),
                 Xp=torch.zeros((R, d), dtype=dt, device="cuda"), status=torch.zeros(1, **i32),
                 ws=torch.empty(B.workspace_bytes(cfg, B.WS_DISPATCH_DEDUP), dtype=torch.uint8, device="cuda"))
        for k, shape in (("totals", (4,)), ("send_naive", (P, P)), ("send_dedup", (P, P))):
            s[k] = torch.zeros(shape, dtype=torch.int64, device="cuda")
        return s

    train = kind == "train"
    lay = C2RLayer(N, d, E, I, K, T, P, I_s, case["bf16"], backward=train, profile=train,
                   fused_combine=bool(case.get("fused_combine")), side_stream=bool(case.get("side_stream")))
    lay.t["Wg"] = Wg
    lay.t["W13p"], lay.t["W2"] = _packed(lay.cfg, g, E, I, d, dt)
    if I_s:
        lay.t["wsg"] = _normal(g, (d,), dt, 0.02)
        lay.t["Ws13p"], lay.t["Ws2"] = _packed(lay.cfg, g, 1, I_s, d, dt)
    if kind == "steps":
        lay.t["L"] = _skewed_logits(g, N, E, d)
        mask, rank, part = _calibrated(case, g, Wg, dt, _skewed_logits(g, 4096, E, d))
    else:
        mask, rank, part = _calibrated(case, g, Wg, dt)
    lay.set_routing(mask=mask, expert_rank=rank, part=part if train else None)
    lay.set_input(X, _normal(g, (N, d), dt) if train else None)
    s = dict(kind=kind, lay=lay)
    if kind == "steps":
        s["opts"] = B.expert_opts(lay.t["w_row"], B.SCALE_ROW)
        if I_s:
            B.gate_logits(lay.cfg, X, Wg, lay.t["wsg"], torch.empty((N, E), device="cuda"), lay.t["z"])
            s["opts_shared"] = B.expert_opts(lay.t["z"], B.SCALE_SIGMOID)
    return s


# ---- one pass -------------------------------------------------------------------------------------------------------

def run(s):
    kind = s["kind"]
    if kind == "forward":
        s["lay"].forward()
        t = s["lay"].t
        return {k: t[k] for k in ("Y", "idx", "w", "counts")}
    if kind == "train":
        s["lay"].train_step()
        t = s["lay"].t
        return {k: t[k] for k in ("Y", "idx", "w", "counts", "volume", "dX", "dW13p", "dW2", "dWg", "dWs13p", "dWs2", "dwsg",
                                  "C", "I_T") if k in t}
    if kind == "steps":
        lay = s["lay"]
        c, t = lay.cfg, lay.t
        if c.I_s:
            B.grouped_swiglu_fwd(c, 1, c.I_s, c.N, t["X"], t["s_counts"], t["s_offsets"], t["Ws13p"], t["Ws2"], None, t["Hs"],
                                 t["Ys"], t["status"], s["opts_shared"])
        B.route(c, t["L"], t["mask"], t["idx"], t["w"], None, t["status"], t["ws"])
        B.permute(c, t["idx"], t["expert_rank"], t["X"], t["counts"], t["offsets"], t["row_of_slot"], t["slot_of_row"], t["Xp"],
                  t["status"], t["ws"], t["w"], t["w_row"], True)
        B.grouped_swiglu_fwd(c, c.E, c.I, lay.R, t["Xp"], t["counts"], t["offsets"], t["W13p"], t["W2"], None, t["H"], t["Yp"],
                             t["status"], s["opts"])
        B.combine(c, t["Yp"], None, t["row_of_slot"], t.get("Ys"), None, t["Y"])
        return {k: t[k] for k in ("Y", "idx", "w", "counts", "offsets", "row_of_slot", "slot_of_row")}
    if kind == "calibrate":
        c = s["cfg"]
        B.gate_logits(c, s["X"], s["Wg"], None, s["L"], None)
        B.route(c, s["L"], None, s["idx"], s["w"])
        B.collab_count(c, s["idx"], s["N"], s["C"])
        B.collab_sets(c, s["C"], s["I_T"], s["mask"])
        return {k: s[k] for k in ("L", "idx", "C", "I_T")}
    c = s["cfg"]
    B.route(c, s["L"], s["mask"], s["idx"], s["w"], None, s["status"])
    B.dispatch_dedup(c, s["idx"], s["part"], s["rank"], s["X"], s["counts"], s["offsets"], s["row_of_slot"], s["slot_of_row"],
                     s["recv_counts"], s["recv_offsets"], s["recv_row_of_slot"], s["token_of_recv_row"], s["Xr"], s["Xp"],
                     s["status"], s["ws"])
    B.dispatch_volume(c, s["idx"], s["part"], s["totals"], s["send_naive"], s["send_dedup"])
    return {k: s[k] for k in ("idx", "w", "counts", "offsets", "row_of_slot", "slot_of_row", "recv_counts", "recv_offsets",
                              "recv_row_of_slot", "token_of_recv_row", "Xr", "Xp", "totals", "send_naive", "send_dedup")}


# ---- what a pass cannot do without ----------------------------------------------------------------------------------

def work(case):
    N, d, E, I, K, P, I_s = (case[k] for k in ("N", "d", "E", "I", "K", "P", "I_s"))
    es = 2 if case["bf16"] else 4
    kind = case["kind"]
    x = N * d * es
    gate = (E + (1 if I_s else 0)) * d * es
    if kind == "calibrate":
        return {"bytes": x + gate + 4 * N * E + 4 * N * K + 4 * E * E, "flops": 2 * N * d * E}
    if kind == "dispatch":  # rows sent: the expected number of distinct partitions of K experts
        sent = N * P * (1.0 - (1.0 - 1.0 / P) ** K)
        return {"bytes": 4 * N * E + x + (sent + N * K) * d * es + 20 * N * K, "flops": 0}
    hit = E * (1.0 - (1.0 - K / E) ** N)  # experts that meet at least one token
    weights = 3 * d * (hit * I + I_s) * es
    fwd = 6 * N * d * (K * I + I_s) + 2 * N * d * E
    if kind == "train":
        return {"bytes": 4 * x + weights + 3 * d * (E * I + I_s) * es + gate + 4 * (E + 1) * d + 8 * N * K, "flops": 3 * fwd}
    if kind == "steps":
        return {"bytes": 2 * x + weights + 4 * N * E + 8 * N * K, "flops": 6 * N * d * (K * I + I_s)}
    return {"bytes": 2 * x + weights + gate + 8 * N * K, "flops": fwd}


def tolerance(case):
    """Against fp64 arithmetic on the same routing: bf16 layers (every stored intermediate and result is rounded to bf16) are off
    by at most 2.9e-3 in the 2-norm and 0.028 of the RMS at one element, fp32 layers by 1.2e-6 and 6.5e-6, weights from bf16
    inputs by 2.8e-6; stated is about four times that.  Logits summed in another order can swap two experts that agree to a
    few units in the last place; a swap changes a few entries of C and I_T."""
    kind = case["kind"]
    if kind == "dispatch":
        return {"rel": 1e-6}
    if kind == "calibrate":
        return {"rel": 1e-5, "differ": 5e-3}
    tol = {"rel": 1e-2, "max": 0.12} if case["bf16"] else {"rel": 5e-6, "max": 3e-5}
    return tol if kind == "steps" else dict(tol, differ=5e-3)


# ---- the same pass in 64 bits, in plain torch -----------------------------------------------------------------------

def _unpack(W13p, I):
    """Rows of W1 and of W3 inside the packed array: blocks of 128 channels of W1, then the same channels of W3."""
    i = torch.arange(I, device=W13p.device)
    gate = i // 128 * 256 + i % 128
    return gate, gate + torch.clamp(I - i // 128 * 128, max=128)


def _expert(x, W13, W2, rows, s, g):
    """s silu(x W1^T) (x W3^T) W2^T for rows x and, with g = dL/dY, also dx, dW13 (packed), dW2 and s <g, expert(x)>."""
    W13, W2 = W13.double(), W2.double()
    gate, up = rows
    a, b = x @ W13[gate].T, x @ W13[up].T
    sg = torch.sigmoid(a)
    h = a * sg * b
    y = s[:, None] * (h @ W2.T)
    if g is None:
        return y, None
    dh = s[:, None] * (g @ W2)
    da, db = dh * b * sg * (1 + a * (1 - sg)), dh * a * sg
    dW13 = torch.empty_like(W13)
    dW13[gate], dW13[up] = da.T @ x, db.T @ x
    return y, (da @ W13[gate] + db @ W13[up], dW13, g.T @ (s[:, None] * h), (dh * h).sum(1))


def exact(case, seed):
    s = prepare(case, seed)
    kind, E, K, I, I_s = case["kind"], case["E"], case["K"], case["I"], case["I_s"]
    if kind == "calibrate":
        return {"L": s["X"].double() @ s["Wg"].double().T, "idx": None, "C": None, "I_T": None}
    t = s if kind == "dispatch" else s["lay"].t
    X = t["X"].double()
    L = t["L"].double() if kind in ("dispatch", "steps") else X @ t["Wg"].double().T
    # Sec. 3.3 step 2: the best expert of all, then the K - 1 best inside its collaborator set (ties: lower index)
    top = L.argmax(1)
    member = ((t["mask"][:, None] >> torch.arange(E, device="cuda")[None, :]) & 1).bool()[top]
    rest = L.masked_fill(~member, -math.inf).scatter(1, top[:, None], -math.inf)
    idx = torch.cat([top[:, None], rest.sort(dim=1, descending=True, stable=True).indices[:, :K - 1]], 1)
    w = torch.softmax(L.gather(1, idx), 1)
    if kind == "dispatch":
        return {"w": w}
    dY = t["dY"].double() if kind == "train" else None
    Y, out = torch.zeros_like(X), {}
    dX, q = torch.zeros_like(X), torch.zeros_like(w)
    if kind == "train":
        out["dW13p"] = torch.zeros(t["W13p"].shape, dtype=torch.float64, device="cuda")
        out["dW2"] = torch.zeros(t["W2"].shape, dtype=torch.float64, device="cuda")
    rows = _unpack(t["W13p"], I)
    for e in range(E):
        tok, k = (idx == e).nonzero(as_tuple=True)
        if len(tok) == 0:
            continue
        y, back = _expert(X[tok], t["W13p"][e], t["W2"][e], rows, w[tok, k], None if dY is None else dY[tok])
        Y.index_add_(0, tok, y)
        if back is not None:
            dX.index_add_(0, tok, back[0])
            out["dW13p"][e], out["dW2"][e], q[tok, k] = back[1:]
        del y, back
    if I_s:
        gs = torch.sigmoid(X @ t["wsg"].double())
        y, back = _expert(X, t["Ws13p"][0], t["Ws2"][0], _unpack(t["Ws13p"], I_s), gs, dY)
        Y += y
        if back is not None:
            dz = back[3] * (1 - gs)
            dX += back[0] + dz[:, None] * t["wsg"].double()
            out.update(dWs13p=back[1][None], dWs2=back[2][None], dwsg=dz @ X)
    if kind == "train":
        dL = torch.zeros_like(L).scatter(1, idx, q - w * q.sum(1, keepdim=True))
        dX += dL @ t["Wg"].double()
        out.update(dX=dX, dWg=dL.T @ X)
    return dict(out, Y=Y, w=w)
