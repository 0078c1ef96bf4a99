"""The work that is measured: Step 2 of Gradient Cache (loss and representation-gradient cache) over
the sizes its users have, the calls around it, and Step 3 on a linear encoder.

A case is a dict of plain values.  `op` names what a training program does:

  build   gc_build_cache: loss, row_lse, positive logits, dQ, dP of one batch
  split   gc_loss_fwd, then gc_loss_bwd with the row_lse it gave (a program that wants the loss first)
  cosine  cosine similarity with a learnable temperature, both directions: gc_row_normalize of both
          sides, gc_build_cache_two_direction on the unit rows, gc_cosine_bwd of both, gc_dtau
  rank    one rank's share of a batch that is spread over `world` GPUs: gc_shard_fwd_dq for its
          queries, gc_shard_dp for its passages (the gathered matrices are in hand)
  apply   gc_cache_apply over a batch in `parts` sub-batches: dW = sum of U^T X

All buffers (outputs, workspace) are made once in prepare(), as a training loop keeps them.
"""
from __future__ import annotations

import math

import torch

from paper_2101_06983_b200 import binding as gc
from paper_2101_06983_b200.sharded import row_ranges

EXTREME = 65536 * 131072 * 768          # the largest batch, in multiply-adds of one product


def listed():
    return [
        # the smallest batches a retriever is trained with: one launch, latency only
        dict(name="batch64_f32", op="build", dtype="f32", B=64, N=128, d=768, tau=1.0, views=0),
        dict(name="batch128_bf16", op="build", dtype="bf16", B=128, N=256, d=768, tau=1.0, views=0),
        # ordinary retriever batches (one positive and one hard negative per query); the second is
        # the ragged last batch of an epoch
        dict(name="batch512_bf16", op="build", dtype="bf16", B=512, N=1024, d=768, tau=1.0, views=0),
        dict(name="batch1531_bf16", op="build", dtype="bf16", B=1531, N=3062, d=768, tau=1.0, views=0),
        # pre-training scale, and the batch that forbids storing the logits
        dict(name="batch4096_bf16", op="build", dtype="bf16", B=4096, N=8192, d=768, tau=1.0, views=0),
        dict(name="batch65536_bf16", op="build", dtype="bf16", B=65536, N=131072, d=768, tau=1.0,
             views=0),
        # full-precision training at an ordinary large batch
        dict(name="batch2048_f32", op="build", dtype="f32", B=2048, N=4096, d=768, tau=1.0, views=0),
        # two views of each item, shared rows, the diagonal masked, short rows
        dict(name="views8192_d128", op="build", dtype="bf16", B=8192, N=8192, d=128, tau=0.1, views=1),
        # wide rows, loss first, gradients in a second call
        dict(name="split4096_d1024", op="split", dtype="bf16", B=4096, N=8192, d=1024, tau=1.0,
             views=0),
        # image-text style batch: cosine similarity, both directions, learnable temperature
        dict(name="cosine4096_d512", op="cosine", dtype="bf16", B=4096, N=4096, d=512, tau=0.07,
             views=0),
        # one of eight ranks of the pre-training batch
        dict(name="rank4096_of8", op="rank", dtype="bf16", B=4096, N=8192, d=768, tau=1.0, views=0,
             world=8),
        # Step 3: the cache of a batch taken to the encoder matrix in two sub-batches
        dict(name="apply8192_d768", op="apply", dtype="bf16", B=8192, N=768, d=768, tau=1.0, views=0,
             parts=2),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["build", "build", "build", "build32", "views", "split", "cosine", "rank", "apply"])
    wide = [256, 384, 512, 640, 768, 1024]
    if op == "apply":
        d = rng.choice([128, 384, 512, 768, 1024])
        return dict(op="apply", dtype="bf16", B=_log_int(rng, 128, 32768), N=rng.choice([384, 768, 1024]),
                    d=d, tau=1.0, views=0, parts=rng.choice([1, 2, 4]))
    if op == "views":
        B = 2 * _log_int(rng, 96, 8192)
        return dict(op="build", dtype="bf16", B=B, N=B, d=rng.choice([64, 128, 256]),
                    tau=rng.choice([0.1, 0.2, 0.5]), views=1)
    if op == "build32":
        B = _log_int(rng, 32, 4096)
        return dict(op="build", dtype="f32", B=B, N=B * rng.choice([1, 2]),
                    d=rng.choice([64, 128, 256, 384, 512, 768]), tau=1.0, views=0)
    d = rng.choice(wide)
    hard = rng.choice([1, 2, 2, 3])
    if op == "cosine":
        B = _log_int(rng, 128, 16384)
        return dict(op="cosine", dtype="bf16", B=B, N=B, d=d, tau=rng.choice([0.05, 0.07, 0.2]), views=0)
    if op == "rank":
        B = _log_int(rng, 1024, 16384)
        return dict(op="rank", dtype="bf16", B=B, N=hard * B, d=d, tau=1.0, views=0,
                    world=rng.choice([2, 4, 8]))
    B = _log_int(rng, 96, 40000)
    while B * hard * B * d > EXTREME:
        B //= 2
    return dict(op=op, dtype="bf16", B=B, N=hard * B, d=d, tau=1.0, views=0)


def _normal(gen, rows, d, sigma):
    return torch.randn(rows, d, generator=gen, device="cuda") * sigma


def _rows(case, gen):
    """Representations: queries near the unit sphere; per query a positive close to it, a hard negative
    less close, the rest of the passages unrelated.  Two views: noisy copies, L2-normalised."""
    B, N, d = case["B"], case["N"], case["d"]
    if case["views"]:
        M = B // 2
        x = _normal(gen, M, d, 1.0)
        X = torch.cat([x + 0.3 * _normal(gen, M, d, 1.0), x + 0.3 * _normal(gen, M, d, 1.0)])
        X /= X.norm(dim=1, keepdim=True)
        pos = (torch.arange(B, device="cuda") + M) % B
        return X, X, pos.to(torch.int32)
    s = d ** -0.5
    Q = _normal(gen, B, d, s)
    per = N // B
    P = _normal(gen, N, d, s)
    P[0::per] = 0.8 * Q + 0.6 * P[0::per]
    if per > 1:
        P[1::per] = 0.5 * Q + 0.866 * P[1::per]
    pos = torch.arange(B, device="cuda") * per
    return Q, P, pos.to(torch.int32)


def prepare(case, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    B, N, d, op = case["B"], case["N"], case["d"], case["op"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    f32 = dict(dtype=torch.float32, device="cuda")
    s = dict(case)
    if op == "apply":                       # d x N is the encoder matrix, B the rows of the cache
        scale = torch.exp2(8.0 * torch.rand(B, 1, generator=gen, device="cuda") - 4.0) / B
        s["U"] = _normal(gen, B, d, 1.0) * scale
        s["X"] = _normal(gen, B, N, 1.0).to(dt)
        s["ranges"] = [(a, n) for a, n in row_ranges(B, case["parts"]) if n > 0]
        s["dW"] = torch.empty(d, N, **f32)
        most = max(n for _, n in s["ranges"])
        s["ws"] = torch.empty(max(gc.gc_cache_apply_workspace_bytes(most, d, N), 256),
                              dtype=torch.uint8, device="cuda")
        return s
    Q, P, s["pos"] = _rows(case, gen)
    shared = P is Q
    s["Q"] = Q.to(dt)
    s["P"] = s["Q"] if shared else P.to(dt)
    del Q, P
    code = gc.GC_BF16 if dt == torch.bfloat16 else gc.GC_F32
    if op in ("build", "split"):
        s["out"] = gc.Outputs(B, N, d, code)
        return s
    s["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    s["loss"] = torch.zeros(1, **f32)
    if op == "cosine":
        # encoder outputs of any length: the loss normalises them
        s["Q"] = (s["Q"].float() * (0.5 + 4.0 * torch.rand(B, 1, generator=gen, device="cuda"))).to(dt)
        s["P"] = (s["P"].float() * (0.5 + 4.0 * torch.rand(N, 1, generator=gen, device="cuda"))).to(dt)
        s["Qn"], s["Pn"] = torch.empty_like(s["Q"]), torch.empty_like(s["P"])
        s["iq"], s["ip"] = torch.empty(B, **f32), torch.empty(N, **f32)
        s["row_lse"] = torch.empty(B, **f32)
        s["dQ"], s["dP"] = torch.empty(B, d, **f32), torch.empty(N, d, **f32)
        s["dtau"] = torch.empty(1, **f32)
        need = max(int(gc._lib.gc_two_direction_workspace_bytes(B, N, d, code)),
                   int(gc._lib.gc_dtau_workspace_bytes(B)), 256)
        s["ws"] = torch.empty(need, dtype=torch.uint8, device="cuda")
        return s
    # rank: a rank in the middle of the batch
    r = case["world"] // 2
    s["q0"], s["qn"] = row_ranges(B, case["world"])[r]
    s["p0"], s["pn"] = row_ranges(N, case["world"])[r]
    s["row_lse"] = torch.empty(B, **f32)
    # the logsumexp of the other ranks' queries arrives through the exchange
    for a in range(0, B, 4096):
        s["row_lse"][a:a + 4096] = torch.logsumexp(
            (s["Q"][a:a + 4096].float() @ s["P"].float().T) / case["tau"], dim=1)
    s["dQ"], s["dP"] = torch.empty(s["qn"], d, **f32), torch.empty(s["pn"], d, **f32)
    need = max(gc.gc_shard_workspace_bytes(B, N, d, code, s["qn"], N),
               gc.gc_shard_workspace_bytes(B, N, d, code, B, s["pn"]), 256)
    s["ws"] = torch.empty(need, dtype=torch.uint8, device="cuda")
    return s


def run(s):
    op, tau = s["op"], s["tau"]
    mask = gc.GC_MASK_SELF if s["views"] else gc.GC_MASK_NONE
    if op == "build":
        o = s["out"]
        gc.gc_build_cache(s["Q"], s["P"], s["pos"], tau, mask, o.loss, o.row_lse, o.dQ, o.dP,
                          o.pos_logit, o.ws, o.dev_status)
        return o.loss, o.row_lse, o.pos_logit, o.dQ, o.dP, o.dev_status
    if op == "split":
        o = s["out"]
        gc.gc_loss_fwd(s["Q"], s["P"], s["pos"], tau, mask, o.loss, o.row_lse, o.pos_logit, o.ws,
                       o.dev_status)
        gc.gc_loss_bwd(s["Q"], s["P"], s["pos"], tau, mask, o.row_lse, o.dQ, o.dP, o.ws, o.dev_status)
        return o.loss, o.row_lse, o.pos_logit, o.dQ, o.dP, o.dev_status
    if op == "cosine":
        gc.gc_row_normalize(s["Q"], s["Qn"], s["iq"])
        gc.gc_row_normalize(s["P"], s["Pn"], s["ip"])
        gc.gc_build_cache_two_direction(s["Qn"], s["Pn"], s["pos"], tau, s["loss"], s["row_lse"],
                                        s["dQ"], s["dP"], s["ws"], s["status"])
        gc.gc_dtau(s["Qn"], s["dQ"], tau, s["dtau"], s["ws"])
        gc.gc_cosine_bwd(s["Q"], s["iq"], s["dQ"], s["dQ"])
        gc.gc_cosine_bwd(s["P"], s["ip"], s["dP"], s["dP"])
        return s["loss"], s["row_lse"], s["dQ"], s["dP"], s["dtau"], s["status"]
    if op == "rank":
        gc.gc_shard_fwd_dq(s["Q"], s["P"], s["pos"], tau, s["q0"], s["qn"], s["loss"], s["row_lse"],
                           s["dQ"], ws=s["ws"], dev_status=s["status"], mask_mode=mask)
        gc.gc_shard_dp(s["Q"], s["P"], s["pos"], tau, s["row_lse"], s["p0"], s["pn"], s["dP"],
                       ws=s["ws"], dev_status=s["status"], mask_mode=mask)
        return s["loss"], s["row_lse"], s["dQ"], s["dP"], s["status"]
    for k, (a, n) in enumerate(s["ranges"]):
        gc.gc_cache_apply(s["U"][a:a + n], s["X"][a:a + n], s["dW"], k > 0, s["ws"])
    return s["dW"]


def work(case):
    B, N, d, op = case["B"], case["N"], case["d"], case["op"]
    es = 2 if case["dtype"] == "bf16" else 4
    if op == "apply":
        return {"bytes": 4 * B * d + es * B * N + 4 * d * N, "flops": 2 * B * d * N}
    rows_in = es * d * (B if case["views"] else B + N) + 4 * B
    out = 4 * d * (B + N) + 8 * B + 4
    three = 6 * B * N * d                    # S, dQ and dP: one product of B x N x d each
    if op == "rank":
        qn, pn = row_ranges(B, case["world"])[0][1], row_ranges(N, case["world"])[0][1]
        return {"bytes": rows_in + 4 * d * (qn + pn) + 8 * B,
                "flops": 4 * qn * N * d + 4 * B * pn * d}     # S and dQ; S and dP of other pairs
    if op == "cosine":                       # both directions share the logits of the B positive pairs
        return {"bytes": rows_in + out, "flops": three}
    return {"bytes": rows_in + out, "flops": three}


def tolerance(case):
    """fp32 rows: 32-bit products and sums (measured against 64 bits: up to 3e-6).  bf16 rows: the
    softmax weights are bf16 operands of the gradient products (up to 2e-3; 4.5e-3 with unit rows
    rounded to bf16 in between)."""
    if case["op"] == "apply" or case["dtype"] == "f32":
        return {"rel": 2e-5}
    return {"rel": 1e-2}
