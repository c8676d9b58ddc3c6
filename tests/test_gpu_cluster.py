"""GPU parity of the cluster row kernel, the emitted sequences, the paired tensor-core contraction and the affinity builds
at the sizes where their tiles and segments end, against the CPU checker (or a float64 product of the same operands)."""
import numpy as np
import pytest
import torch

import parity_util as PU
import workloads as W
from oracle import rdk_oracle as O
from test_gpu_linear import KIND, _run_linear

pytestmark = pytest.mark.gpu


def _rdk():
    import paper_2506_03206_b200 as rdk
    return rdk


def _reference(inp, kept_ids=None, prior=None):
    cfg, kappa = inp["cfg"], (inp["kept_ids"] if kept_ids is None else kept_ids).numpy()
    return {r: O.rdk_row(W.to_f64(inp["target"][r]), W.to_f64(inp["drafter"][r]), kappa, np.zeros((1, 4)), "linear",
                         drafter_kind=cfg.drafter_kind, prior=None if prior is None else W.to_f64(prior)) for r in range(cfg.rows)}


# N around the change of variant (4096), segments of one and several 256-token chunks, odd sizes (every row at another
# alignment), one to sixteen CTAs a row, more than one round of trials (16), more kept tokens than fit a warp's registers
@pytest.mark.parametrize("N,n,rows,trials,dtype,kind", [
    (4095, 1000, 3, 17, "f32", "logits"), (4096, 1024, 3, 1, "bf16", "logits"), (4097, 4000, 3, 2, "bf16", "probs"),
    (8193, 8193, 2, 33, "f32", "logits"), (20001, 2500, 40, 1, "bf16", "logits"), (50257, 25000, 2, 8, "bf16", "logits"),
    (65537, 300, 2, 3, "f32", "probs"), (131075, 40000, 1, 16, "bf16", "logits")])
def test_cluster_kernel_shapes(N, n, rows, trials, dtype, kind):
    cfg = W.tiny_config(N=N, n=n, rows=rows, dtype=dtype, trials=trials, rho=0.6, seed=N, drafter_kind=kind, zipf_bias=True)
    _run_linear(cfg, W.make_inputs(cfg), check_qtilde=N < 60000).assert_ok()


def test_cluster_kernel_unsorted_ids_and_sequences_longer_than_the_accept_bits():
    cfg = W.tiny_config(N=5003, n=700, rows=60, dtype="bf16", trials=3, rho=0.9, seed=5)
    cfg = cfg.with_rows(2, 30)                       # 30 positions: arrivals are counted, the flags read again
    inp = W.make_inputs(cfg)
    ids = inp["kept_ids"][torch.randperm(cfg.n, generator=torch.Generator().manual_seed(2))].clone()
    ids[3], ids[cfg.n - 1] = -1, cfg.N + 4           # two drafter tokens outside the vocabulary
    _run_linear(cfg, inp, kept_override=ids).assert_ok()


def test_cluster_kernel_scale_that_does_not_fit_the_segment():
    """The first tokens of a segment give the scale of its exponentials; here they are far below the others or -inf, so that
    the sums overflow the limit and the visit is repeated with the maximum."""
    cfg = W.tiny_config(N=16411, n=3000, rows=4, dtype="f32", trials=4, rho=0.5, seed=12)
    inp = W.make_inputs(cfg)
    inp["target"][0, 256:] += 150.0
    inp["target"][1, :4000] = -float("inf")
    inp["target"][2, 700:9000] -= 400.0
    inp["drafter"][3, 2000:] += 120.0
    _run_linear(cfg, inp).assert_ok()


@pytest.mark.parametrize("shift", [0.0, 30.0, -30.0])
def test_cluster_kernel_prior_above_and_below_the_target(shift):
    """theta pi / N is the smaller of the two nearly everywhere, or for half of the tokens, or hardly anywhere: the second visit
    decides it from the difference of the logits."""
    rdk = _rdk()
    cfg = W.tiny_config(N=9001, n=1500, rows=3, dtype="bf16", trials=5, rho=0.7, seed=31)
    inp = W.make_inputs(cfg)
    g = torch.Generator().manual_seed(3)
    prior = torch.randn(cfg.N, generator=g)
    prior[: cfg.N // 2] += shift
    prior[11] = -float("inf")
    inp["target"][:, 13] = -float("inf")
    prior = prior.to(torch.bfloat16)
    idx = rdk.rdk_prepare_ids(inp["kept_ids"].cuda(), cfg.N)
    out = rdk.rdk_sample_and_verify_prior(idx, inp["target"].cuda(), prior.cuda(), inp["drafter"].cuda(), inp["uniforms"].cuda(),
                                          cfg.batch, cfg.positions)
    qt, _, _ = rdk.rdk_redistribute_linear_prior(idx, inp["target"].cuda(), prior.cuda(), inp["drafter"].cuda(), cfg.batch, cfg.positions)
    torch.cuda.synchronize()
    PU.compare_sampling(inp, out, range(cfg.rows), "linear", prior=prior).assert_ok()
    PU.compare_accepted_len(out, cfg.batch, cfg.positions, cfg.trials)
    PU.compare_qtilde(qt, _reference(inp, prior=prior), True)


@pytest.mark.parametrize("N,batch,positions,trials,counters", [(4096, 3, 2, 20, True), (33000, 2, 3, 1, False), (70001, 1, 1, 4, True)])
def test_cluster_kernel_given_weights(N, batch, positions, trials, counters):
    rdk = _rdk()
    B = rdk.binding
    cfg = W.tiny_config(N=N, n=50, rows=batch * positions, dtype="bf16", trials=trials, seed=N).with_rows(batch, positions)
    inp = W.make_inputs(cfg)
    # a total of about 1, as the exact redistribution gives: S is an fp32 number, so its bound of 1e-5 holds for such totals
    # (a rounding error is 2^-24 of the total, 2e-4 for one of several thousand)
    w = torch.rand(cfg.rows, N, generator=torch.Generator().manual_seed(N)) ** 8
    w = w / w.sum(1, keepdim=True)
    idx = rdk.rdk_prepare_ids(inp["kept_ids"].cuda(), N)
    # with room for the counters accepted_len is counted in the same launch, without it in one more
    ws = torch.full((8 * batch * trials if counters else 4,), 0xA5, dtype=torch.uint8, device="cuda")
    for _ in range(2):
        out = rdk.rdk_sample_and_verify(idx, B.RDK_MODE_PRECOMPUTED_W, inp["target"].cuda(), None, w.cuda(), inp["uniforms"].cuda(),
                                        batch, positions, ws=ws)
        torch.cuda.synchronize()
        PU.compare_sampling(inp, out, range(cfg.rows), "given", w_given=w.double().numpy()).assert_ok()
        PU.compare_accepted_len(out, batch, positions, trials)


@pytest.mark.parametrize("N,batch,positions,trials", [(300, 700, 3, 2), (40001, 90, 40, 1), (140000, 3, 1, 1), (1001, 20, 2, 2), (4001, 400, 2, 1),
                                                      (65537, 400, 1, 1), (70001, 70, 2, 1)])
def test_emitted_sequences_of_many_pairs(N, batch, positions, trials):
    """More pairs than clusters, more positions than a warp's lanes, one to eight CTAs a row; the accept patterns mix all
    accepted, none and everything between."""
    rdk = _rdk()
    g = torch.Generator().manual_seed(N)
    bonus = (torch.randn(batch, N, generator=g) * 2).to(torch.bfloat16)
    u = torch.from_numpy(W.uniforms(N, batch * positions, trials))
    cut = torch.randint(0, positions + 2, (batch, trials), generator=g)           # leading accepts; beyond it at random
    acc = torch.rand(batch, positions, trials, generator=g) < 0.5
    k = torch.arange(positions).view(1, positions, 1)
    acc = (k < cut.unsqueeze(1)) | (acc & (k > cut.unsqueeze(1)))
    draft = torch.randint(0, N, (batch, positions, trials), generator=g, dtype=torch.int32)
    resid = torch.randint(0, N, (batch, positions, trials), generator=g, dtype=torch.int32)
    seq, ln = rdk.rdk_emit_sequences(N, batch, positions, bonus.cuda(), u.cuda(), draft.cuda(), acc.to(torch.uint8).cuda(), resid.cuda())
    torch.cuda.synchronize()
    seq, ln, un, near = seq.cpu().numpy(), ln.cpu().numpy(), u.numpy().reshape(batch, positions, trials, 4), 0
    for b in range(batch):
        cdf = None
        for t in range(trials):
            a = acc[b, :, t].numpy()
            j = positions if a.all() else int(np.argmin(a))
            assert ln[b, t] == j + 1 and np.array_equal(seq[b, t, :j], draft[b, :j, t].numpy()) and np.all(seq[b, t, j + 1:] == -1)
            if j < positions:
                assert seq[b, t, j] == resid[b, j, t]
            else:
                cdf = np.cumsum(O.softmax(W.to_f64(bonus[b]))) if cdf is None else cdf
                thr, tok = float(un[b, positions - 1, t, 3]) * cdf[-1], int(seq[b, t, j])
                near += tok != int(np.searchsorted(cdf, thr, side="right"))
                assert PU.interval_distance(cdf, tok, thr) <= PU.BOUNDARY_TOL
    assert near <= max(1, 0.01 * batch * trials)


# rows: one instruction of the smallest width, the steps of 16, both instructions, several row tiles, halves of the last
# round; tokens: less than, exactly and just over a CTA's 128 and a pair's 256; contraction: around one block of 64
@pytest.mark.parametrize("N,n,rows", [(127, 63, 1), (128, 64, 16), (129, 65, 33), (255, 8, 256), (257, 129, 257), (5000, 200, 300),
                                      (300, 1000, 513), (19200, 72, 1024), (38000, 640, 320), (4096, 192, 1100),
                                      # two instructions of R rows each, 74 pairs: R = 144, in one round and with halved items; 176,
                                      # 208 and 240; two and three row tiles; a last row tile of one instruction
                                      (18944, 300, 257), (19100, 300, 288), (25000, 200, 340), (25000, 200, 410), (30000, 136, 470),
                                      (20000, 100, 700), (33000, 70, 1030), (2000, 70, 8200)])
def test_paired_contraction_at_tile_edges(N, n, rows):
    rdk = _rdk()
    B = rdk.binding
    g = torch.Generator(device="cuda").manual_seed(N + rows)
    ids = torch.sort(torch.randperm(N, generator=g, device="cuda")[: min(n, N)]).values.to(torch.int32)
    ids = torch.cat([ids, torch.full((n - ids.numel(),), -1, dtype=torch.int32, device="cuda")])        # n > N: tokens outside the vocabulary
    idx = rdk.rdk_prepare_ids(ids, N)
    # probabilities that are multiples of 2^-12 and add up to 1: exact in bf16, so that q' is too
    q = torch.zeros(rows, n, device="cuda")
    live = min(n, N, 16)                             # columns of its own for every row: a row in another's place shows
    q.scatter_(1, torch.rand(rows, min(n, N), generator=g, device="cuda").argsort(1)[:, :live], 1.0 / (1 << (live.bit_length() - 1)))
    q = q / q.sum(1, keepdim=True) if live & (live - 1) else q
    M = {"data": torch.rand(N, (n + 7) // 8 * 8, generator=g, device="cuda").to(torch.bfloat16), "layout": B.RDK_AFF_BF16_COLS, "ld": (n + 7) // 8 * 8}
    w = torch.full((rows, N), float("nan"), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    _, S, _ = rdk.rdk_redistribute_exact(idx, q, M, rows, 1, B.RDK_PROBS, w_out=w, status_word=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    ref = q.to(torch.bfloat16).double() @ M["data"][:, :n].double().T
    # fp32 accumulation of n products: n rounding errors of 2^-24 of the result at most
    assert ((w.double() - ref).abs() <= (n + 2) * 2.0 ** -24 * ref.abs() + 1e-12).all()
    assert ((S.double() - ref.sum(1)).abs() <= (N + n) * 2.0 ** -24 * ref.sum(1) + 1e-12).all()


@pytest.mark.parametrize("N,n,rows", [(31, 5, 1), (33, 257, 9), (1024, 300, 80), (4736, 1000, 70)])
def test_fp32_contraction_at_tile_edges(N, n, rows):
    """One and four columns a thread (the last shape), ragged rows, columns and contraction."""
    rdk = _rdk()
    B = rdk.binding
    g = torch.Generator(device="cuda").manual_seed(N)
    ids = torch.sort(torch.randperm(N, generator=g, device="cuda")[: min(n, N)]).values.to(torch.int32)
    ids = torch.cat([ids, torch.full((n - ids.numel(),), -1, dtype=torch.int32, device="cuda")])
    idx = rdk.rdk_prepare_ids(ids, N)
    y = torch.randn(rows, n, generator=g, device="cuda")
    M = {"data": torch.rand(n, N, generator=g, device="cuda"), "layout": B.RDK_AFF_F32_ROWS, "ld": N}
    w, S, _ = rdk.rdk_redistribute_exact(idx, y, M, rows, 1)
    torch.cuda.synchronize()
    q = torch.softmax(torch.where(ids >= 0, y.double(), torch.tensor(-float("inf"), device="cuda", dtype=torch.float64)), -1)
    ref = q @ M["data"].double()
    # q' carries a few rounding errors of its own (exponential, sum, quotient): 1e-6; the products add n of 2^-24
    assert ((w.double() - ref).abs() <= (1e-6 + n * 2.0 ** -24) * ref).all()
    assert ((S.double() - ref.sum(1)).abs() <= (1e-6 + (N + n) * 2.0 ** -24) * ref.sum(1)).all()


@pytest.mark.parametrize("N,n,d,dtype,tau", [(257, 129, 20, "bf16", 0.1), (1030, 260, 100, "bf16", 0.05), (515, 64, 65, "bf16", 0.1),
                                             (9000, 2400, 64, "f32", 0.1), (1001, 17, 33, "f32", 0.02)])
def test_affinity_builds_at_tile_edges(N, n, d, dtype, tau):
    """Ragged tiles on both routes, embedding dimensions whose rows are not whole 16-byte units, a zero embedding (equally near to
    every token), ids outside the vocabulary, four columns and one a thread."""
    rdk = _rdk()
    B = rdk.binding
    g = torch.Generator(device="cuda").manual_seed(N)
    E = torch.randn(N, d, generator=g, device="cuda").to(torch.bfloat16 if dtype == "bf16" else torch.float32)
    ids = torch.sort(torch.randperm(N, generator=g, device="cuda")[:n]).values.to(torch.int32)
    E[ids[1].long()] = 0
    ids[2], ids[n - 1] = -1, N
    M = rdk.rdk_build_affinity(E, ids, tau, B.RDK_AFF_BF16_COLS if dtype == "bf16" else B.RDK_AFF_F32_ROWS)
    torch.cuda.synchronize()
    ok = (ids >= 0) & (ids < N)
    En = torch.nn.functional.normalize(E.double(), dim=1, eps=1e-12)
    ref = torch.softmax(En[ids.clamp(0, N - 1).long()] @ En.T / tau, -1) * ok.unsqueeze(1)
    got = M["data"][:, :n].T.double() if dtype == "bf16" else M["data"].double()
    # the exponent (cos - 1) / tau log2 e carries rounding errors of 2^-24 of its size, d of them in the dot product, in units of
    # 1 / tau; storing in bf16 adds half a unit in the last place, 2^-9
    tol = 4 * (d ** 0.5 + 8) * 2.0 ** -24 / tau + (2.0 ** -8 if dtype == "bf16" else 0.0)
    assert ((got - ref).abs() <= tol * ref).all()
    assert torch.all(got[~ok] == 0)
    if dtype == "bf16":
        assert torch.all(M["data"][:, n:] == 0)


@pytest.mark.parametrize("N,n,d", [(3000, 700, 64), (1111, 300, 200)])
def test_affinity_of_a_small_temperature_is_the_identity(N, n, d):
    """At tau = 1e-5 every other token is thousands of units of the exponent away, so a kept id's own entry is its whole sum and
    has to be 1 to the last bit, whatever rounding errors the cosine carries (units of 1e-2 of the exponent here): entry and sum
    are the same number.  Some 1e-2 off shows as another bf16 number, of which there is one every 2^-8 below 1.  A zero embedding
    is equally near to every token."""
    rdk = _rdk()
    B = rdk.binding
    g = torch.Generator(device="cuda").manual_seed(d)
    E = torch.randn(N, d, generator=g, device="cuda").to(torch.bfloat16)
    ids = torch.randperm(N, generator=g, device="cuda")[:n].to(torch.int32)
    E[ids[7].long()] = 0
    M = rdk.rdk_build_affinity(E, ids, 1e-5, B.RDK_AFF_BF16_COLS)["data"][:, :n].double()
    ref = torch.zeros_like(M)
    ref[ids.long(), torch.arange(n, device="cuda")] = 1.0
    ref[:, 7] = torch.tensor(1.0 / N).to(torch.bfloat16).double()
    assert torch.equal(M, ref)


@pytest.mark.parametrize("N,n,dtype,order", [(50257, 12565, "bf16", "ascending"), (32000, 8000, "f32", "ranked"), (9001, 3000, "f32", "ascending")])
def test_cluster_kernel_errors_against_64_bits(N, n, dtype, order):
    """alpha and the residual's mass of 320 long-tailed rows, relative error in the 2-norm: an exponential is off by 2^-24 of itself
    in the mean; its sum, the reciprocal, the product and the sum of the products by a rounding each (2^-24 / sqrt 3): sqrt(7 / 3) in
    units of 2^-24 in all where one token has the weight, and less where several share it.  Scales that are rounded for each segment apart, and exponents far
    above zero, show here."""
    rdk = _rdk()
    B = rdk.binding
    rows, dt, g = 32, {"bf16": torch.bfloat16, "f32": torch.float32}[dtype], torch.Generator(device="cuda").manual_seed(N)
    square = {"alpha": 0.0, "residual_mass": 0.0}
    for _ in range(10):
        ranking = torch.randperm(N, generator=g, device="cuda")
        ids = ranking[:n] if order == "ranked" else torch.sort(ranking[:n]).values
        bias = torch.empty(N, device="cuda")
        bias[ranking] = -1.1 * torch.log(torch.arange(1, N + 1, device="cuda", dtype=torch.float32))
        z0 = torch.randn(rows, N, generator=g, device="cuda")
        z = (3 * z0 + bias).to(dt)
        y = (bias[ids] + 3 * (0.8 * z0[:, ids] + 0.6 * torch.randn(rows, n, generator=g, device="cuda"))).to(dt)
        out = rdk.rdk_sample_and_verify(rdk.rdk_prepare_ids(ids.to(torch.int32), N), B.RDK_MODE_LINEAR, z, y, None,
                                        torch.rand(rows, 4, 4, generator=g, device="cuda"), rows, 1)
        B.check_status_word(out)
        p, q = torch.softmax(z.double(), 1), torch.zeros(rows, N, dtype=torch.float64, device="cuda")
        q[:, ids] = torch.softmax(y.double(), 1)
        theta = (p * q).sum(1, keepdim=True)
        w = (N * q + theta * p) / (N + p)
        m = torch.minimum(p, w / w.sum(1, keepdim=True))
        for k, ref in (("alpha", m.sum(1)), ("residual_mass", (p - m).sum(1))):
            square[k] += float(((out[k].double() - ref) ** 2).sum() / (ref ** 2).sum()) / 10
    assert max(square.values()) ** 0.5 <= (7 / 3) ** 0.5 * 2.0 ** -24, {k: v ** 0.5 * 2 ** 24 for k, v in square.items()}


@pytest.mark.parametrize("N,n", [(128256, 12826), (262143, 90000)])
def test_written_out_q_errors_against_64_bits(N, n):
    """q~ of 64 long-tailed rows, relative error in the 2-norm: the exponential's 2^-24 and a rounding (2^-24 / sqrt 3) each for the
    reciprocal of the sum, the product and the redistribution; the sum's own, which all of a row would share, are not among them."""
    rdk = _rdk()
    rows, g, square = 8, torch.Generator(device="cuda").manual_seed(N), 0.0
    for _ in range(8):
        ranking = torch.randperm(N, generator=g, device="cuda")
        ids = torch.sort(ranking[:n]).values
        bias = torch.empty(N, device="cuda")
        bias[ranking] = -1.1 * torch.log(torch.arange(1, N + 1, device="cuda", dtype=torch.float32))
        z = (3 * torch.randn(rows, N, generator=g, device="cuda") + bias).to(torch.bfloat16)
        y = (bias[ids] + 3 * torch.randn(rows, n, generator=g, device="cuda")).to(torch.bfloat16)
        got, _, _ = rdk.rdk_redistribute_linear(rdk.rdk_prepare_ids(ids.to(torch.int32), N), z, y, rows, 1)
        p, q = torch.softmax(z.double(), 1), torch.zeros(rows, N, dtype=torch.float64, device="cuda")
        q[:, ids] = torch.softmax(y.double(), 1)
        w = (N * q + (p * q).sum(1, keepdim=True) * p) / (N + p)
        w = w / w.sum(1, keepdim=True)
        square += float(((got.double() - w) ** 2).sum() / (w ** 2).sum()) / 8
    assert square ** 0.5 <= 2.0 ** 0.5 * 2.0 ** -24, square ** 0.5 * 2 ** 24


@pytest.mark.parametrize("mode,N,rows,trials", [("given", 4096, 100, 16), ("given", 33001, 20, 256), ("given", 262144, 40, 64), ("given", 70001, 2, 256), ("linear", 5000, 160, 64),
                                                ("linear", 70001, 5, 2048), ("prior", 9000, 150, 64)])
def test_many_draws_take_the_row_kernel(mode, N, rows, trials):
    """Where draws outweigh the sweep the one-CTA-per-row kernel serves, so every output has that kernel's bits."""
    rdk = _rdk()
    B = rdk.binding
    g = torch.Generator(device="cuda").manual_seed(N)
    ids = torch.randperm(N, generator=g, device="cuda")[: N // 4].to(torch.int32)      # (not ascending: the streaming kernels cannot serve)
    idx = rdk.rdk_prepare_ids(ids, N)
    z = torch.randn(rows, N, generator=g, device="cuda").to(torch.bfloat16)
    y = torch.randn(rows, N // 4, generator=g, device="cuda").to(torch.bfloat16) if mode != "given" else None
    w = torch.softmax(torch.randn(rows, N, generator=g, device="cuda"), -1) if mode == "given" else None
    u = torch.rand(rows, trials, 4, generator=g, device="cuda")
    m = B.RDK_MODE_LINEAR if mode != "given" else B.RDK_MODE_PRECOMPUTED_W
    if mode == "prior":      # (the call with a prior has no flags: the row kernel's numbers are those of a prior that is the target)
        a = rdk.rdk_sample_and_verify_prior(idx, z, z, y, u, rows, 1)
        b = rdk.rdk_sample_and_verify(idx, m, z, y, None, u, rows, 1, flags=B.RDK_FLAG_ROW_KERNEL)
    else:
        a, b = (rdk.rdk_sample_and_verify(idx, m, z, y, w, u, rows, 1, flags=f) for f in (0, B.RDK_FLAG_ROW_KERNEL))
    for k in ("draft_token", "out_token", "accepted", "accept_prob", "alpha", "S", "residual_mass", "accepted_len"):
        assert torch.equal(a[k], b[k]), k


def test_index_written_by_the_kernel_queued_just_before_the_call():
    """An index is an input like any other: a copy of one, made on the stream just before the call into a buffer that held another
    list's, is the one that the call uses.  The strided copy is a kernel that a long one holds up."""
    rdk = _rdk()
    B = rdk.binding
    N, n, rows = 20011, 3001, 4
    g = torch.Generator(device="cuda").manual_seed(4)
    lists = [torch.randperm(N, generator=g, device="cuda")[:n].to(torch.int32) for _ in range(2)]
    idx = [rdk.rdk_prepare_ids(x, N) for x in lists]
    z = torch.randn(rows, N, generator=g, device="cuda").to(torch.bfloat16)
    y, u = torch.randn(rows, n, generator=g, device="cuda").to(torch.bfloat16), torch.rand(rows, 1, 4, generator=g, device="cuda")
    want = [rdk.rdk_sample_and_verify(i, B.RDK_MODE_LINEAR, z, y, None, u, rows, 1) for i in idx]
    wide = [torch.stack([i.buffer, i.buffer], 1) for i in idx]
    moved, big = B.KeptIndex(torch.empty_like(idx[0].buffer), N, n, n), torch.zeros(1 << 27, device="cuda")
    moved.buffer.copy_(idx[0].buffer)
    for k in range(1, 9):
        big.add_(1.0)
        moved.buffer.copy_(wide[k & 1][:, 0])
        out = rdk.rdk_sample_and_verify(moved, B.RDK_MODE_LINEAR, z, y, None, u, rows, 1)
        for name in ("draft_token", "alpha", "theta", "S"):
            assert torch.equal(out[name], want[k & 1][name]), (k, name)


# Shapes on clusters of other sizes than powers of two, of eight and of sixteen warps, with many and with few registers; more
# than one wave of them; more kept tokens than fit a warp's registers
@pytest.mark.parametrize("N,n,rows,trials,dtype", [
    (5001, 500, 40, 1, "bf16"), (20011, 2000, 20, 1, "f32"), (33333, 8333, 40, 1, "bf16"), (33333, 8333, 45, 4, "f32"),
    (50257, 12565, 80, 1, "bf16"), (50257, 12565, 330, 2, "bf16"), (90001, 30000, 20, 1, "f32"), (128257, 3000, 24, 5, "bf16"),
    (262143, 100000, 5, 1, "bf16"), (16001, 4000, 16, 4, "f32"), (32001, 8000, 33, 4, "f32"), (32001, 8000, 34, 4, "bf16")])
def test_cluster_kernel_cluster_sizes(N, n, rows, trials, dtype):
    cfg = W.tiny_config(N=N, n=n, rows=rows, dtype=dtype, trials=trials, rho=0.8, seed=rows, zipf_bias=True)
    inp = W.make_inputs(cfg)
    rdk = _rdk()
    B = rdk.binding
    idx = rdk.rdk_prepare_ids(inp["kept_ids"].cuda(), N)
    z, y, u = inp["target"].cuda(), inp["drafter"].cuda(), inp["uniforms"].cuda()
    out = rdk.rdk_sample_and_verify(idx, B.RDK_MODE_LINEAR, z, y, None, u, cfg.batch, cfg.positions)
    ref = rdk.rdk_sample_and_verify(idx, B.RDK_MODE_LINEAR, z, y, None, u, cfg.batch, cfg.positions, flags=B.RDK_FLAG_ROW_KERNEL)
    torch.cuda.synchronize()
    B.check_status_word(out)
    PU.compare_sampling(inp, out, sorted({0, rows // 2, rows - 1}), "linear").assert_ok()
    for k in ("alpha", "theta", "S", "residual_mass"):
        assert float((out[k] - ref[k]).abs().max()) < 1e-5, k
    # a draw on the other side of a boundary: prefix sums 1e-7 apart, some 2 n interval ends (as in assert_ok_at_scale)
    assert int((out["draft_token"] != ref["draft_token"]).sum()) <= 2 + 6e-7 * n * rows * trials
    if trials == 1:
        w = torch.softmax(z.float(), -1)
        given = rdk.rdk_sample_and_verify(idx, B.RDK_MODE_PRECOMPUTED_W, z, None, w, u, cfg.batch, cfg.positions)
        torch.cuda.synchronize()
        assert float(given["accepted"].float().mean()) > 0.99 and float((given["alpha"] - 1).abs().max()) < 1e-5
        if N < 100000:
            qt, _, _ = rdk.rdk_redistribute_linear(idx, z, y, cfg.batch, cfg.positions)
            torch.cuda.synchronize()
            PU.compare_qtilde(qt, {0: O.rdk_row(W.to_f64(inp["target"][0]), W.to_f64(inp["drafter"][0]), inp["kept_ids"].numpy(), np.zeros((1, 4)), "linear")}, dtype == "bf16")


# One prior row for all rows through the streaming kernels, and the same shapes without it: groups of unequal length and of one
# row; kept tokens per segment from none to all of them (segments that outgrow the cached slots), one to six steps of 64 slots;
# sequences of one position, of several and of more than the accept bits; draw kernels of 256 and of 128 threads (beyond 1184 draws)
@pytest.mark.parametrize("N,n,batch,positions,kept", [
    (16384, 900, 90, 5, "random"), (65536, 8000, 38, 5, "random"), (65536, 11000, 149, 1, "highest"), (65536, 13000, 131, 1, "random"),
    (65536, 20000, 20, 8, "lowest"), (131072, 7000, 3, 30, "highest"), (131064, 34000, 83, 1, "random"), (262144, 4000, 14, 5, "random")])
@pytest.mark.parametrize("shared_prior", [False, True])
def test_stream_kernel_shared_prior(N, n, batch, positions, kept, shared_prior):
    rows, trials = batch * positions, 3
    cfg = W.tiny_config(N=N, n=n, rows=rows, dtype="bf16", trials=trials, rho=0.7, seed=n, zipf_bias=True).with_rows(batch, positions)
    g = torch.Generator().manual_seed(n)
    ids = {"random": torch.sort(torch.randperm(N, generator=g)[:n]).values, "lowest": torch.arange(n), "highest": torch.arange(N - n, N)}[kept]
    inp = W.make_inputs(cfg)
    inp["kept_ids"] = ids.to(inp["kept_ids"].dtype)
    rdk = _rdk()
    idx = rdk.rdk_prepare_ids(inp["kept_ids"].to(torch.int32).cuda(), N)
    z, y, u = inp["target"].cuda(), inp["drafter"].cuda(), inp["uniforms"].cuda()
    z[rows // 2, : N // 3] = -float("inf")               # whole segments without weight
    y[rows - 1, n // 2:] += 60.0                         # the first kept value is a poor scale
    inp["target"], inp["drafter"] = z, y
    B = rdk.binding
    prior = None
    if shared_prior:
        prior = (torch.randn(N, generator=g) * 2).to(torch.bfloat16)
        prior[5] = -float("inf")
        pb = B.make_problem(idx, z, y, cfg.batch, cfg.positions)
        wanted = B.lib().rdk_sample_prior_workspace_bytes(B.C.byref(pb), z.data_ptr(), prior.cuda().data_ptr(), 0, y.data_ptr(), trials)
        assert wanted > 0                                # the streaming kernels serve
        out = rdk.rdk_sample_and_verify_prior(idx, z, prior.cuda(), y, u, cfg.batch, cfg.positions)
    else:
        out = rdk.rdk_sample_and_verify(idx, B.RDK_MODE_LINEAR, z, y, None, u, cfg.batch, cfg.positions)
        route, why = rdk.rdk_sample_route(idx, B.RDK_MODE_LINEAR, z, y, batch, positions, trials, out["_ws"])
        assert route == B.RDK_ROUTE_STREAM_KERNEL, why
    torch.cuda.synchronize()
    B.check_status_word(out)
    some = sorted({0, 1, rows // 2, rows - 2, rows - 1})
    PU.compare_sampling(inp, out, some, "linear", prior=prior).assert_ok()
    PU.compare_accepted_len(out, batch, positions, trials)
    # every row against the one-CTA-per-row or the cluster kernel
    if shared_prior:
        ref = rdk.rdk_sample_and_verify_prior(idx, z, prior.cuda().expand(rows, N).contiguous(), y, u, cfg.batch, cfg.positions)
    else:
        ref = rdk.rdk_sample_and_verify(idx, B.RDK_MODE_LINEAR, z, y, None, u, cfg.batch, cfg.positions, flags=B.RDK_FLAG_ROW_KERNEL)
    torch.cuda.synchronize()
    for k in ("alpha", "theta", "S", "residual_mass"):
        assert float((out[k] - ref[k]).abs().max()) < 1e-5, k
    # a draw on the other side of a boundary: prefix sums 1e-7 apart, some 2 n interval ends (as in assert_ok_at_scale)
    assert int((out["draft_token"] != ref["draft_token"]).sum()) <= 2 + 6e-7 * n * rows * trials
