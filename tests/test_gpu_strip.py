"""GPU parity of the strip plan (three products over strips of query rows) against the CPU oracle, at
the sizes where it can go wrong: single columns and rows, ragged last tiles and groups of 64 columns,
column tiles of every width, whole-tile and cut-tile dealing of the gradients, several strips with the
masked diagonal running through them, one gradient without the other, rows whose logits span hundreds
of powers of two.  Tolerances are those of the other parity tests."""
import numpy as np
import pytest
import torch

from paper_2101_06983_b200 import inputs

from gpu_util import TOL, check_against_oracle, grad_err, run_build, to_device
from test_gpu_parity import _check_properties, _check_sampled, _oracle_full

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2101_06983_b200 import binding as b
    return b


SHAPES = [
    # B, N, d, dtype, mask, tau
    (129, 1, 64, "bf16", 0, 1.0), (1, 257, 8, "bf16", 0, 1.0), (1, 129, 8, "f32", 0, 1.0),
    (255, 321, 72, "bf16", 1, 0.3), (257, 511, 136, "f32", 1, 0.3), (400, 1601, 448, "bf16", 0, 0.5),
    (1100, 63, 1088, "bf16", 0, 0.5), (2305, 2561, 192, "bf16", 1, 0.2), (3000, 5000, 576, "bf16", 0, 0.5),
    (5200, 700, 768, "bf16", 0, 0.5), (1900, 2100, 384, "f32", 0, 0.5), (600, 9001, 512, "f32", 0, 0.5),
    # logits spanning hundreds of powers of two.  fp32: a weight is 2^(s - lse) of two fp32 numbers, so its
    # relative error is at least ln 2 times half an ulp of lse log2(e): at tau = 0.01 lse reaches 2800
    # (4000 in log2 units, 1.7e-4, beyond the 1e-4 of these tests), at 0.1 it stays below 300 (1.1e-5).
    (300, 520, 768, "bf16", 0, 0.004), (300, 520, 64, "f32", 0, 0.1),
]


@pytest.mark.parametrize("B,N,d,dtype,mask,tau", SHAPES)
def test_build_and_split_calls(binding, oracle, B, N, d, dtype, mask, tau):
    prob = inputs.random_problem(B, N, d, dtype, seed=B + N + d, tau=tau, mask_mode=mask,
                                 scale=1.0 if tau <= 0.1 else d ** -0.5)
    out = run_build(prob)
    ref = _oracle_full(oracle, prob)
    check_against_oracle(prob, out, ref)
    Q, P, pos = to_device(prob)
    b = binding.Outputs(B, N, d, binding._dtype_code(Q))
    args = (Q, P, pos, prob.tau, prob.mask_mode)
    binding.gc_loss_fwd(*args, b.loss, b.row_lse, b.pos_logit, b.ws, b.dev_status)
    binding.gc_loss_bwd(*args, b.row_lse, b.dQ, None, b.ws, b.dev_status)
    binding.gc_loss_bwd(*args, b.row_lse, None, b.dP, b.ws, b.dev_status)
    torch.cuda.synchronize()
    check_against_oracle(prob, b, ref)


@pytest.mark.parametrize("B,N", [(333, 4100), (66, 33000), (650, 17000), (1300, 16500), (3, 270000)])
def test_long_rows_of_the_row_pass(binding, oracle, B, N):
    """Four warps to a row with the last one idle; segments of one, two and three rounds; a grid beyond
    six blocks per SM; more slots than a lane holds at once."""
    prob = inputs.random_problem(B, N, 64, "bf16", seed=B + N, tau=0.2, scale=0.125)
    check_against_oracle(prob, run_build(prob), _oracle_full(oracle, prob))


def test_logits_formed_twice(binding, oracle):
    """Rows of at most 384 values and many pairs: no row pass, one launch more per strip."""
    n, d = 16700, 320
    prob = inputs.random_problem(n, n, d, "bf16", seed=7, tau=0.5, mask_mode=inputs.MASK_SELF,
                                 scale=d ** -0.5)
    assert binding.gc_kernel_launches(binding.GC_OP_BUILD, n, n, d, binding.GC_BF16) == 4
    out = run_build(prob)
    assert int(out.dev_status.item()) == 0
    _check_sampled(oracle, prob, out, 48, 24, full_lse=out.row_lse.cpu().numpy().astype(np.float64))
    Q, P, _ = to_device(prob)
    _check_properties(prob, out, Q, P)


def test_several_strips_f32_self_mask(binding, oracle):
    """8200 x 8200 pairs are two strips; the diagonal runs through both."""
    prob = inputs.random_problem(8200, 8200, 16, "f32", seed=5, tau=0.5, mask_mode=inputs.MASK_SELF,
                                 scale=0.25)
    assert binding.gc_kernel_launches(binding.GC_OP_BUILD, 8200, 8200, 16, binding.GC_F32) == 1 + 2 * 3
    out = run_build(prob)
    check_against_oracle(prob, out, _oracle_full(oracle, prob))


def test_several_strips_bf16_self_mask(binding, oracle):
    """33 000 x 33 000 pairs are two strips: sampled rows of both, and the identities."""
    n, d = 33000, 448
    prob = inputs.random_problem(n, n, d, "bf16", seed=6, tau=0.5, mask_mode=inputs.MASK_SELF,
                                 scale=d ** -0.5)
    assert binding.gc_kernel_launches(binding.GC_OP_BUILD, n, n, d, binding.GC_BF16) == 2 * 3
    out = run_build(prob)
    assert int(out.dev_status.item()) == 0
    _check_sampled(oracle, prob, out, 48, 24, full_lse=out.row_lse.cpu().numpy().astype(np.float64))
    Q, P, _ = to_device(prob)
    _check_properties(prob, out, Q, P)


@pytest.mark.parametrize("B,N,d,tau", [(300, 310, 136, 0.3), (500, 320, 64, 0.2), (1030, 1200, 448, 0.5)])
def test_two_directions_with_few_spare_passages(binding, oracle, B, N, d, tau):
    """Up to 1.25 B passages the column direction runs over all passages: passages that are nobody's
    positive, and passages that are the positive of several queries."""
    prob = inputs.random_problem(B, N, d, "bf16", seed=B + N, tau=tau, scale=d ** -0.5)
    ref = oracle.build_variant(prob.Q, prob.P, prob.pos_idx, prob.tau, 0, two_direction=True)
    assert np.unique(prob.pos_idx).size < min(B, N)
    Q, P, pos = to_device(prob)
    f = dict(dtype=torch.float32, device="cuda")
    loss, lse = torch.zeros(1, **f), torch.empty(B, **f)
    dQ, dP = torch.full((B, d), float("nan"), **f), torch.full((N, d), float("nan"), **f)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    binding.gc_build_cache_two_direction(Q, P, pos, prob.tau, loss, lse, dQ, dP, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    tol = TOL["bf16"]
    assert abs(loss.item() - ref["loss"]) <= tol["loss"] * abs(ref["loss"])
    assert grad_err(dQ.cpu().numpy(), ref["dQ"]) <= tol["grad"]
    assert grad_err(dP.cpu().numpy(), ref["dP"]) <= tol["grad"]
    bad = pos.clone()
    bad[3] = N
    binding.gc_build_cache_two_direction(Q, P, bad, prob.tau, loss, lse, dQ, dP, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == binding.GC_DEV_POS_RANGE and bool(torch.isfinite(dP).all())


@pytest.mark.parametrize("B,N,d,mask", [(128, 128, 8, 0), (33, 127, 72, 0), (97, 97, 136, 1),
                                        (128, 1, 192, 0), (1, 128, 264, 0), (65, 66, 1000, 1)])
def test_one_tile_f32_clusters(binding, oracle, B, N, d, mask):
    """One, two and four CTAs per cluster, slices that do not fill the last cluster; both gradients from
    the build and each alone from the backward call."""
    prob = inputs.random_problem(B, N, d, "f32", seed=B + N + d, tau=0.5, mask_mode=mask, scale=d ** -0.5)
    ref = _oracle_full(oracle, prob)
    check_against_oracle(prob, run_build(prob), ref)
    Q, P, pos = to_device(prob)
    b = binding.Outputs(B, N, d, binding.GC_F32)
    args = (Q, P, pos, prob.tau, prob.mask_mode)
    binding.gc_loss_fwd(*args, b.loss, b.row_lse, b.pos_logit, b.ws, b.dev_status)
    binding.gc_loss_bwd(*args, b.row_lse, b.dQ, None, b.ws, b.dev_status)
    binding.gc_loss_bwd(*args, b.row_lse, None, b.dP, b.ws, b.dev_status)
    torch.cuda.synchronize()
    check_against_oracle(prob, b, ref)


@pytest.mark.parametrize("B,N,d", [(768, 64, 3072), (705, 1, 3008), (768, 65, 3072)])
def test_few_logit_tiles_clear_every_counter(binding, oracle, B, N, d):
    """Three logit tiles (six CTAs), gradient tiles cut between CTA pairs: the counters of every cut tile
    start at zero whatever the workspace held, in a first call and in a second one on other inputs."""
    out = binding.Outputs(B, N, d, binding.GC_F32)
    out.ws.fill_(0xA5)
    for seed in (1, 2):
        prob = inputs.random_problem(B, N, d, "f32", seed=seed, tau=0.5, scale=d ** -0.5)
        Q, P, pos = to_device(prob)
        out.dQ.fill_(float("nan"))
        out.dP.fill_(float("nan"))
        binding.build_cache(Q, P, pos, prob.tau, prob.mask_mode, out)
        torch.cuda.synchronize()
        check_against_oracle(prob, out, _oracle_full(oracle, prob))


def _hard_negatives(B, N, d, seed):
    """Unit rows; passage i is the positive of query i (cosine 0.8), passage B + i its hard negative (0.95)."""
    rng = np.random.default_rng(seed)
    unit = lambda x: x / np.linalg.norm(x, axis=1, keepdims=True)
    Q, P = unit(rng.standard_normal((B, d))), unit(rng.standard_normal((N, d)))
    for first, cos in ((0, 0.8), (B, 0.95)):
        side = P[first:first + B] - (P[first:first + B] * Q).sum(1, keepdims=True) * Q
        P[first:first + B] = cos * Q + (1 - cos * cos) ** 0.5 * unit(side)
    return Q.astype(np.float32), P.astype(np.float32)


@pytest.mark.parametrize("B,N,d,tau", [(512, 2048, 512, 0.05), (512, 2048, 512, 0.02), (300, 1000, 448, 0.012),
                                       (300, 1111, 512, 0.2), (130, 900, 64, 0.03), (200, 5000, 64, 0.03),
                                       (150, 17001, 512, 0.05)])
def test_rows_of_small_weights_keep_their_precision(binding, B, N, d, tau):
    """dP row by row, for passages whose every weight lies up to a hundred powers of two below their row's
    largest.  A weight is rounded at most twice, to 8 bits of mantissa (2^-9 of it) in between and to bf16
    (2^-8) in the end, and 2^(s - lse) of two fp32 numbers below 2^8 in magnitude is off by 2^-15 at most; a
    row of dP therefore by at most that share of the sum of its terms' norms."""
    Qn, Pn = _hard_negatives(B, N, d, seed=B + N)
    Q, P = (torch.from_numpy(x).to(torch.bfloat16).cuda() for x in (Qn, Pn))
    pos = torch.arange(B, dtype=torch.int32, device="cuda")
    o = binding.Outputs(B, N, d, binding.GC_BF16)
    binding.gc_build_cache(Q, P, pos, tau, 0, o.loss, o.row_lse, o.dQ, o.dP, o.pos_logit, o.ws, o.dev_status)
    both = torch.empty_like(o.dP)
    binding.gc_loss_bwd(Q, P, pos, tau, 0, o.row_lse, o.dQ, both, o.ws, o.dev_status)
    torch.cuda.synchronize()
    assert int(o.dev_status.item()) == 0
    Q64, P64 = Q.double().cpu(), P.double().cpu()
    S = Q64 @ P64.T / tau
    W = torch.exp(S - torch.logsumexp(S, 1, keepdim=True))
    W[torch.arange(B), torch.arange(B)] -= 1.0
    dP = W.T @ Q64 / (B * tau)
    terms = W.abs().T @ Q64.norm(dim=1) / (B * tau)
    bound = (2.0 ** -8 + 2.0 ** -9 + 2.0 ** -13) * terms + B * 2.0 ** -118
    for got in (o.dP, both):
        err = (got.double().cpu() - dP).norm(dim=1)
        assert bool((err <= bound).all()), float((err / bound).max())


@pytest.mark.parametrize("B,N,d,dtype", [
    (256, 256, 64, "bf16"), (2048, 2304, 64, "bf16"), (3328, 4096, 64, "bf16"), (4100, 5700, 64, "bf16"),
    (512, 300, 40, "f32"), (1800, 1900, 72, "f32"), (2600, 2700, 64, "f32"),
])
def test_chained_calls_of_pairs_with_one_to_four_tiles(binding, oracle, B, N, d, dtype):
    """The CTAs of a pair leave together after one, two, three and four uses of their accumulators, and the
    next kernel takes their place at once: forty calls in a row, no wait that runs out, the same bits."""
    prob = inputs.random_problem(B, N, d, dtype, seed=B + N, tau=0.5, scale=d ** -0.5)
    Q, P, pos = to_device(prob)
    a = binding.Outputs(B, N, d, binding._dtype_code(Q))
    b = binding.Outputs(B, N, d, binding._dtype_code(Q))
    args = (Q, P, pos, prob.tau, prob.mask_mode)
    for o in [a] + [b] * 20:
        binding.gc_build_cache(*args, o.loss, o.row_lse, o.dQ, o.dP, o.pos_logit, o.ws, o.dev_status)
        binding.gc_loss_bwd(*args, o.row_lse, o.dQ, None, o.ws, o.dev_status)
    torch.cuda.synchronize()
    check_against_oracle(prob, a, _oracle_full(oracle, prob))
    assert int(b.dev_status.item()) == 0
    for name in ("loss", "row_lse", "pos_logit", "dQ", "dP"):
        assert torch.equal(getattr(a, name), getattr(b, name)), name


@pytest.mark.parametrize("B,N,d,dtype", [
    (8191, 200, 64, "bf16"), (8192, 1, 64, "bf16"), (9001, 512, 128, "bf16"), (8500, 1024, 64, "bf16"),
    (8500, 1025, 64, "bf16"), (1, 512, 24, "f32"), (1300, 511, 24, "f32"), (9600, 5, 16, "f32"),
    (700, 513, 24, "f32"),
])
def test_short_rows_of_the_row_pass(binding, oracle, B, N, d, dtype):
    """A thread per row of the loss (at most eight slots, many rows), a warp per row of fp32 logits: both
    sides of each limit, last blocks and warps that are not full, unusable positives."""
    prob = inputs.random_problem(B, N, d, dtype, seed=B + N, tau=0.5, scale=d ** -0.5)
    Q, P, pos = to_device(prob)
    b = binding.Outputs(B, N, d, binding._dtype_code(Q))
    args = (Q, P, pos, prob.tau, prob.mask_mode)
    binding.gc_loss_fwd(*args, b.loss, b.row_lse, b.pos_logit, b.ws, b.dev_status)
    binding.gc_loss_bwd(*args, b.row_lse, b.dQ, b.dP, b.ws, b.dev_status)
    torch.cuda.synchronize()
    ref = _oracle_full(oracle, prob)
    check_against_oracle(prob, b, ref)
    check_against_oracle(prob, run_build(prob), ref)
    bad = pos.clone()
    bad[0], bad[B // 2] = N, -1
    binding.gc_loss_fwd(Q, P, bad, *args[3:], b.loss, b.row_lse, b.pos_logit, b.ws, b.dev_status)
    torch.cuda.synchronize()
    assert int(b.dev_status.item()) == binding.GC_DEV_POS_RANGE
    assert b.pos_logit[0].item() == 0 and b.pos_logit[B // 2].item() == 0


@pytest.mark.parametrize("B,N,d", [(4671, 30, 128), (4000, 64, 512), (7, 9470, 128), (2000, 100, 2048)])
def test_one_side_far_longer_than_the_other(binding, oracle, B, N, d):
    """Gradient tiles of one or two contraction blocks beside tiles of very many."""
    prob = inputs.random_problem(B, N, d, "bf16", seed=B + N, tau=0.5, scale=d ** -0.5)
    check_against_oracle(prob, run_build(prob), _oracle_full(oracle, prob))


def test_several_strips_given_row_lse(binding, oracle):
    """gc_loss_fwd, then gc_loss_bwd over two strips with the self mask: row_lse, the masked diagonal, the
    counters and the sums into dP of the second strip."""
    n, d = 33000, 448
    prob = inputs.random_problem(n, n, d, "bf16", seed=16, tau=0.5, mask_mode=inputs.MASK_SELF, scale=d ** -0.5)
    assert binding.gc_kernel_launches(binding.GC_OP_BWD, n, n, d, binding.GC_BF16) == 2 * 2
    Q, P, pos = to_device(prob)
    o = binding.Outputs(n, n, d, binding.GC_BF16)
    args = (Q, P, pos, prob.tau, prob.mask_mode)
    binding.gc_loss_fwd(*args, o.loss, o.row_lse, o.pos_logit, o.ws, o.dev_status)
    binding.gc_loss_bwd(*args, o.row_lse, o.dQ, o.dP, o.ws, o.dev_status)
    torch.cuda.synchronize()
    assert int(o.dev_status.item()) == 0
    _check_sampled(oracle, prob, o, 48, 24, full_lse=o.row_lse.cpu().numpy().astype(np.float64))
    _check_properties(prob, o, Q, P)


def test_logits_formed_twice_over_several_strips(binding, oracle):
    n, d = 28800, 320
    prob = inputs.random_problem(n, n, d, "bf16", seed=17, tau=0.5, scale=d ** -0.5)
    assert binding.gc_kernel_launches(binding.GC_OP_BUILD, n, n, d, binding.GC_BF16) == 2 * 4
    out = run_build(prob)
    assert int(out.dev_status.item()) == 0
    _check_sampled(oracle, prob, out, 48, 24, full_lse=out.row_lse.cpu().numpy().astype(np.float64))
    Q, P, _ = to_device(prob)
    _check_properties(prob, out, Q, P)


def test_two_directions_over_several_strips(binding):
    """Both directions in one set of weights over two strips, against 64-bit sums in blocks of rows."""
    n, d, tau = 28800, 192, 0.5
    g = torch.Generator(device="cuda").manual_seed(18)
    Q = (torch.randn(n, d, generator=g, device="cuda") * d ** -0.5).bfloat16()
    P = (torch.randn(n, d, generator=g, device="cuda") * d ** -0.5).bfloat16()
    pos = torch.randint(0, n, (n,), generator=g, device="cuda")
    f = dict(dtype=torch.float32, device="cuda")
    loss, lse, dQ, dP = torch.zeros(1, **f), torch.empty(n, **f), torch.empty(n, d, **f), torch.empty(n, d, **f)
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    binding.gc_build_cache_two_direction(Q, P, pos.int(), tau, loss, lse, dQ, dP, dev_status=st)
    torch.cuda.synchronize()
    assert int(st.item()) == 0
    q, p = Q.double(), P.double()
    rows = [slice(a, min(a + 3200, n)) for a in range(0, n, 3200)]
    row_lse = torch.cat([torch.logsumexp(q[r] @ p.T / tau, 1) for r in rows])
    col_lse = torch.cat([torch.logsumexp(p[r] @ q.T / tau, 1) for r in rows])
    mult = torch.bincount(pos, minlength=n).double()
    pl = (q * p[pos]).sum(1) / tau
    want = 0.5 * ((row_lse - pl) + (col_lse[pos] - pl)).mean().item()
    rQ, rP = torch.empty_like(q), torch.zeros_like(p)
    for r in rows:
        S = q[r] @ p.T / tau
        W = torch.exp(S - row_lse[r, None]) + mult * torch.exp(S - col_lse)
        W[torch.arange(W.shape[0], device="cuda"), pos[r]] -= 2.0
        rQ[r] = W @ p / (2 * n * tau)
        rP += W.T @ q[r] / (2 * n * tau)
    tol = TOL["bf16"]
    assert abs(loss.item() - want) <= tol["loss"] * abs(want)
    assert grad_err(dQ.cpu().numpy(), rQ.cpu().numpy()) <= tol["grad"]
    assert grad_err(dP.cpu().numpy(), rP.cpu().numpy()) <= tol["grad"]


@pytest.mark.parametrize("B,N,d,dtype", [
    (512, 8192, 768, "bf16"),                           # dQ in up to 12 shares a tile
    (300, 4000, 200, "bf16"), (4001, 300, 200, "bf16"), # 200: the last column tile holds 72 of 128; ragged rows
    (777, 3130, 320, "bf16"), (9001, 700, 640, "bf16"), # tiles of 128, the last of 320 half filled; dQ, dP
    (1300, 16500, 640, "bf16"),                         # both: tiles of 256 columns, the last one at half width
    (40, 16500, 72, "f32"), (2100, 260, 136, "f32"), (260, 2100, 136, "f32"),
])
def test_sums_of_cut_gradient_tiles(binding, oracle, B, N, d, dtype):
    """Each gradient alone and both, over long contractions: tiles in up to dozens of shares, summed in pieces by
    whoever is there.  Ragged last rows and columns; outputs inside wider and longer buffers, of which nothing else
    is written; the same bits in every run."""
    prob = inputs.random_problem(B, N, d, dtype, seed=B + N + d, tau=0.5, scale=d ** -0.5)
    Q, P, pos = to_device(prob)
    code = binding._dtype_code(Q)
    assert binding.gc_kernel_launches(binding.GC_OP_BWD, B, N, d, code) == (2 if dtype == "bf16" else 4)   # one strip
    b = binding.Outputs(B, N, d, code)
    args = (Q, P, pos, prob.tau, prob.mask_mode)
    binding.gc_loss_fwd(*args, b.loss, b.row_lse, b.pos_logit, b.ws, b.dev_status)
    wide = {k: torch.full((n + 3, d + 8), float("nan"), device="cuda") for k, n in (("dQ", B), ("dP", N))}
    b.dQ, b.dP = wide["dQ"][:B, :d], wide["dP"][:N, :d]

    def grads(*which):
        for w in wide.values():
            w.fill_(float("nan"))
        binding.gc_loss_bwd(*args, b.row_lse, *(getattr(b, k) if k in which else None for k in ("dQ", "dP")), b.ws,
                            b.dev_status)
        for k, w in wide.items():
            g = getattr(b, k)
            assert bool(torch.isfinite(g).all() if k in which else torch.isnan(g).all())
            assert bool(torch.isnan(w[:, d:]).all()) and bool(torch.isnan(w[g.shape[0]:]).all())
        return [getattr(b, k).clone() for k in which]

    large = B * N * d > 1 << 33
    ref = None if large else _oracle_full(oracle, prob)
    alone = grads("dQ") + grads("dP")
    both = grads("dQ", "dP")
    for b.dQ, b.dP in (alone, both):
        torch.cuda.synchronize()
        if large:
            _check_sampled(oracle, prob, b, 48, 24, full_lse=b.row_lse.cpu().numpy().astype(np.float64))
        else:
            check_against_oracle(prob, b, ref)
    b.dQ, b.dP = wide["dQ"][:B, :d], wide["dP"][:N, :d]
    for _ in range(20):
        again = grads("dQ") + grads("dP"), grads("dQ", "dP")
        assert all(torch.equal(x, y) for got, want in zip(again, (alone, both)) for x, y in zip(got, want))
    assert int(b.dev_status.item()) == 0


@pytest.mark.parametrize("B,N,d,dtype,lse2,tau2", [(32768, 25000, 448, "bf16", 15, 112), (32768, 25000, 1024, "bf16", 15, 112),
                                                   (8192, 8250, 136, "f32", 13, 114)])
def test_subnormal_gradients_of_a_second_strip(binding, B, N, d, dtype, lse2, tau2):
    """Weights of 2^-lse2 (2^-lse2 - 1 at the positives, in bf16 rounded to -1), rows of +-2^-6 and a temperature of
    2^tau2: every entry of dP is a sum of subnormal numbers, exact but for that rounding.  The second strip adds to
    the first through a bulk reduction or, where a cut tile is summed in pieces, in registers: the same sums."""
    g = torch.Generator(device="cuda").manual_seed(B + d)
    dt = torch.bfloat16 if dtype == "bf16" else torch.float32
    Q, P = ((torch.randint(0, 2, (n, d), generator=g, device="cuda") * 2.0 ** -5 - 2.0 ** -6).to(dt) for n in (B, N))
    pos = torch.randint(0, N, (B,), generator=g, device="cuda").int()
    code = binding._dtype_code(Q)
    assert binding.gc_kernel_launches(binding.GC_OP_BWD, B, N, d, code) == (4 if dtype == "bf16" else 1 + 2 * 3)
    o = binding.Outputs(B, N, d, code)
    o.row_lse.fill_(lse2 * float(np.log(2.0)))
    want = Q.double().sum(0).mul(2.0 ** -lse2).repeat(N, 1).index_add_(0, pos.long(), Q.double(), alpha=-1.0)
    want = want * 2.0 ** -tau2 / B
    assert float(want.abs().max()) < 2.0 ** -127
    for dQ in (o.dQ, None):
        for _ in range(5):
            o.dP.fill_(float("nan"))
            binding.gc_loss_bwd(Q, P, pos, 2.0 ** tau2, 0, o.row_lse, dQ, o.dP, o.ws, o.dev_status)
            err = (o.dP.double() - want).abs().max()      # up to 15 positives to a passage, 2^-149 per strip's sum
            assert float(err) <= 2.0 ** -lse2 * float(want.abs().max()) + 2 * 2.0 ** -149
    assert int(o.dev_status.item()) == 0


@pytest.mark.parametrize("B,N,d,side", [(256, 16384, 768, "dQ"), (16384, 256, 768, "dP"), (512, 8192, 448, "dQ")])
def test_cut_tiles_on_a_busy_device(binding, B, N, d, side):
    """Two streams with an output and a workspace each: pairs of one launch start when pairs of the other have left.
    The same bits as alone, and no share that waits for a pair which cannot start."""
    prob = inputs.random_problem(B, N, d, "bf16", seed=B + N, tau=0.5, scale=d ** -0.5)
    Q, P, pos = to_device(prob)
    args = (Q, P, pos, prob.tau, prob.mask_mode)
    outs = [binding.Outputs(B, N, d, binding.GC_BF16) for _ in range(2)]
    want = run_build(prob)

    def grad(o):
        grads = (o.dQ, None) if side == "dQ" else (None, o.dP)
        binding.gc_loss_bwd(*args, want.row_lse, *grads, o.ws, o.dev_status)

    grad(outs[0])
    alone = getattr(outs[0], side).clone()
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in outs]
    for _ in range(5):
        for o in outs:
            getattr(o, side).fill_(float("nan"))
        torch.cuda.synchronize()
        for _ in range(10):
            for o, st in zip(outs, streams):
                with torch.cuda.stream(st):
                    grad(o)
        torch.cuda.synchronize()
        for o in outs:
            assert torch.equal(getattr(o, side), alone) and int(o.dev_status.item()) == 0
