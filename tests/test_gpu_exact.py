"""GPU parity of the affinity construction (Eq. symbolic-m), the exact redistribution w = M^T q'
(Algorithm 1 step 2) and the sampler fed with a precomputed w, against the CPU checker."""
import numpy as np
import pytest
import torch

import parity_util as PU
import workloads as W
from oracle import rdk_oracle as O

pytestmark = pytest.mark.gpu

KIND = {"logits": 0, "probs": 1}


def _rdk():
    import paper_2506_03206_b200 as rdk
    return rdk


def _oracle_M(cfg, inp):
    return O.build_affinity(W.to_f64(inp["embeddings"]), inp["kept_ids"].numpy(), cfg.tau)


def _upload_affinity(M64, layout, B):
    """Put the checker's matrix into one of the library's two layouts on the GPU."""
    n, N = M64.shape
    A = B.affinity_alloc(N, n, layout, "cuda")
    if layout == B.RDK_AFF_F32_ROWS:
        A["data"].copy_(torch.from_numpy(M64).to(torch.float32))
    else:
        A["data"][:, :n].copy_(torch.from_numpy(O.round_to_bf16(M64).T.copy()).to(torch.bfloat16))
    return A


@pytest.mark.parametrize("which", ["C1", "tiny16", "odd"])
def test_build_affinity_fp32_rows(which):
    rdk = _rdk()
    B = rdk.binding
    cfg = {"C1": W.CONFIGS["C1"], "tiny16": W.tiny_config(N=16, n=4, emb_dim=8),
           "odd": W.tiny_config(N=777, n=45, emb_dim=33, dtype="bf16")}[which]
    inp = W.make_inputs(cfg, with_embeddings=True)
    M_ref = _oracle_M(cfg, inp)
    M = rdk.rdk_build_affinity(inp["embeddings"].cuda(), inp["kept_ids"].cuda(), cfg.tau, B.RDK_AFF_F32_ROWS)
    torch.cuda.synchronize()
    got = M["data"].cpu().double().numpy()
    assert np.abs(got - M_ref).max() <= PU.ABS_TOL
    sel = M_ref > 1e-30
    assert (np.abs(got - M_ref)[sel] / M_ref[sel]).max() <= 1e-4
    assert np.abs(got.sum(axis=1) - 1.0).max() < 1e-5                 # Assumption 4.1


def test_build_affinity_bf16_cols_and_dropped_rows():
    rdk = _rdk()
    B = rdk.binding
    cfg = W.tiny_config(N=1500, n=200, emb_dim=32, dtype="bf16")
    inp = W.make_inputs(cfg, with_embeddings=True)
    ids = inp["kept_ids"].clone()
    ids[3] = -1
    ids[17] = cfg.N + 1
    M_ref = O.build_affinity(W.to_f64(inp["embeddings"]), ids.numpy(), cfg.tau)
    M = rdk.rdk_build_affinity(inp["embeddings"].cuda(), ids.cuda(), cfg.tau, B.RDK_AFF_BF16_COLS)
    torch.cuda.synchronize()
    got = M["data"][:, : cfg.n].cpu().double().numpy().T               # back to [n, N]
    # bf16 storage (8 significant bits): the stored value is the checker's value rounded to
    # nearest-even, except where the fp32 arithmetic lands on the other side of a rounding
    # boundary -- then it is the neighbouring bf16 number (one unit in the last place, 2^-7).
    M_rnd = O.round_to_bf16(M_ref)
    assert np.mean(got == M_rnd) >= 0.99
    assert np.all(np.abs(got - M_rnd) <= 2.0 ** -7 * M_rnd + 1e-38)
    assert np.all(np.abs(got - M_ref) <= (2.0 ** -8 + 1e-4) * M_ref + 1e-38)
    assert np.all(got[3] == 0) and np.all(got[17] == 0)


@pytest.mark.parametrize("N,n,d", [(3000, 300, 72), (4100, 2300, 128), (700, 64, 64)])
def test_build_affinity_on_the_tensor_cores(N, n, d):
    """bf16 embeddings of dimension >= 64 into the bf16 layout: the dot products run on the tensor cores (ragged
    embedding dimension, ragged tiles, more kept rows than one chunk, ids outside the vocabulary), compared with the
    checker's matrix rounded to bf16: equal except where fp32 arithmetic lands on the other side of a rounding
    boundary (then the neighbouring bf16 number)."""
    rdk = _rdk()
    B = rdk.binding
    cfg = W.tiny_config(N=N, n=n, emb_dim=d, dtype="bf16", seed=N + d)
    inp = W.make_inputs(cfg, with_embeddings=True)
    assert inp["embeddings"].dtype == torch.bfloat16
    ids = inp["kept_ids"].clone()
    ids[5] = -3
    ids[n - 2] = N
    M_ref = O.build_affinity(W.to_f64(inp["embeddings"]), ids.numpy(), cfg.tau)
    emb = inp["embeddings"].cuda()
    if d == 72:      # rows inside a wider buffer: a row stride of 80 elements (16-byte aligned rows)
        wide = torch.zeros(N, 80, dtype=torch.bfloat16, device="cuda")
        wide[:, :d] = emb
        emb = wide[:, :d]
        assert emb.stride(0) == 80
    M = rdk.rdk_build_affinity(emb, ids.cuda(), cfg.tau, B.RDK_AFF_BF16_COLS)
    torch.cuda.synchronize()
    got = M["data"][:, :n].cpu().double().numpy().T
    assert not np.isnan(got).any()
    M_rnd = O.round_to_bf16(M_ref)
    assert np.mean(got == M_rnd) >= 0.99
    assert np.all(np.abs(got - M_rnd) <= 2.0 ** -7 * M_rnd + 1e-38)
    assert np.all(np.abs(got - M_ref) <= (2.0 ** -8 + 1e-4) * M_ref + 1e-38)
    assert np.all(got[5] == 0) and np.all(got[n - 2] == 0)
    assert np.all(np.abs(got.sum(axis=1)[[0, 1, n - 1]] - 1.0) < 5e-3)


def _flip_allowance(qp, Mcols):
    """The left operand q' is rounded to bf16 on the GPU from an fp32 value and in the checker from a
    float64 value.  An element whose exact value lies within fp32 rounding error (2e-6 relative) of a
    bf16 rounding boundary may legitimately land on either neighbour; this returns, for each output
    column, the largest change of w such flips can cause (zero when no element is that close).
    qp: [..., n] float64 q' at the kept ids; Mcols: [n, cols]."""
    _, e = np.frexp(qp)
    ulp = np.ldexp(1.0, e - 8)
    dist_to_boundary = 0.5 * ulp - np.abs(qp - O.round_to_bf16(qp))
    near = dist_to_boundary <= 2e-6 * np.abs(qp)
    return (np.where(near, ulp, 0.0)) @ Mcols


def _exact_case(cfg, layout_name, identity=False):
    rdk = _rdk()
    B = rdk.binding
    layout = {"f32": B.RDK_AFF_F32_ROWS, "bf16": B.RDK_AFF_BF16_COLS}[layout_name]
    inp = W.make_inputs(cfg, with_embeddings=True)
    kappa = inp["kept_ids"].numpy()
    if identity:
        M64 = np.zeros((cfg.n, cfg.N))
        M64[np.arange(cfg.n), kappa] = 1.0
    else:
        M64 = _oracle_M(cfg, inp)
    if layout == B.RDK_AFF_BF16_COLS:
        M64 = O.round_to_bf16(M64)           # both sides contract the stored (rounded) matrix
    A = _upload_affinity(M64, layout, B)
    idx = rdk.rdk_prepare_ids(inp["kept_ids"].cuda(), cfg.N)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    w, S, _ = rdk.rdk_redistribute_exact(idx, inp["drafter"].cuda(), A, cfg.batch, cfg.positions,
                                         KIND[cfg.drafter_kind], status_word=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    bf = layout == B.RDK_AFF_BF16_COLS
    w_ref = np.zeros((cfg.rows, cfg.N))
    for r in range(cfg.rows):
        ref = O.rdk_row(W.to_f64(inp["target"][r]), W.to_f64(inp["drafter"][r]), kappa, np.zeros((1, 4)), "exact",
                        M=M64, drafter_kind=cfg.drafter_kind, operand_bf16=bf)
        w_ref[r] = ref["w"]
        g = w[r].cpu().double().numpy()
        assert np.abs(g - ref["w"]).max() <= PU.ABS_TOL
        if bf:
            valid = (kappa >= 0) & (kappa < cfg.N)
            allow = _flip_allowance(np.where(valid, ref["qprime"][np.where(valid, kappa, 0)], 0.0), M64)
            assert np.all(np.abs(g - ref["w"]) <= PU.REL_TOL_BF16 * ref["w"] + allow + 1e-12)
            assert abs(float(S[r]) - ref["S"]) <= PU.ABS_TOL + allow.sum()
        else:
            if cfg.dtype == "bf16":
                assert np.all(np.abs(g - ref["w"]) <= PU.REL_TOL_BF16 * ref["w"] + 1e-12)
            assert PU.close(float(S[r]), ref["S"], False)
        if identity and not bf:
            assert np.allclose(g / g.sum(), ref["qprime"], atol=1e-6)   # M = I: RDK reduces to TLI
    # the sampler takes w as an input: both sides get the checker's w, stored as float32
    w_in = torch.from_numpy(w_ref).to(torch.float32)
    out = rdk.rdk_sample_and_verify(idx, B.RDK_MODE_PRECOMPUTED_W, inp["target"].cuda(), None, w_in.cuda(),
                                    inp["uniforms"].cuda(), cfg.batch, cfg.positions)
    torch.cuda.synchronize()
    t = PU.compare_sampling(inp, out, range(cfg.rows), "given", w_given=w_in.double().numpy())
    PU.compare_accepted_len(out, cfg.batch, cfg.positions, cfg.trials)
    print(cfg.name, layout_name, t.summary())
    t.assert_ok(max_ambiguous_frac=0.1)
    return w_ref


def test_config1_tiny_rdk_exact():
    _exact_case(W.CONFIGS["C1"], "f32")


@pytest.mark.parametrize("N,n,rows", [(2, 1, 3), (16, 4, 5), (16, 16, 2), (300, 33, 9), (2050, 130, 17)])
def test_exact_small_shapes_fp32(N, n, rows):
    _exact_case(W.tiny_config(N=N, n=n, rows=rows, trials=8, emb_dim=8, seed=N + n), "f32")


def test_exact_identity_affinity_is_tli():
    _exact_case(W.tiny_config(N=64, n=10, rows=4, trials=8), "f32", identity=True)


def test_exact_probability_drafter_fp32():
    _exact_case(W.tiny_config(N=512, n=64, rows=4, trials=4, drafter_kind="probs", dtype="bf16", rho=0.8), "f32")


# ---------------------------------------------------------------- tensor-core layout (bf16, transposed)
@pytest.mark.parametrize("N,n,rows", [(300, 33, 9), (2050, 130, 17), (1000, 520, 300), (4096, 1024, 384),
                                      (777, 64, 129), (256, 8, 1)])
def test_exact_tensor_core_shapes(N, n, rows):
    # several tiles of 256 tokens, ragged edges in all three dimensions, up to five row tiles of one instruction each
    _exact_case(W.tiny_config(N=N, n=n, rows=rows, trials=2, emb_dim=8, seed=N + n + rows, dtype="bf16"), "bf16")


def test_exact_tensor_core_identity_affinity_is_tli():
    # M = I in bf16 is exact, so w must equal the bf16-rounded q' at the kept ids and 0 elsewhere
    rdk = _rdk()
    B = rdk.binding
    cfg = W.tiny_config(N=600, n=72, rows=5, trials=1, dtype="bf16", seed=8)
    inp = W.make_inputs(cfg)
    kappa = inp["kept_ids"].numpy()
    M64 = np.zeros((cfg.n, cfg.N))
    M64[np.arange(cfg.n), kappa] = 1.0
    A = _upload_affinity(M64, B.RDK_AFF_BF16_COLS, B)
    idx = rdk.rdk_prepare_ids(inp["kept_ids"].cuda(), cfg.N)
    w, S, _ = rdk.rdk_redistribute_exact(idx, inp["drafter"].cuda(), A, cfg.batch, cfg.positions)
    torch.cuda.synchronize()
    for r in range(cfg.rows):
        qp = O.drafter_qprime(W.to_f64(inp["drafter"][r]), kappa, cfg.N, "logits")
        g = w[r].cpu().double().numpy()
        assert np.all(g[np.setdiff1d(np.arange(cfg.N), kappa)] == 0)
        # the operand is the fp32 q' rounded to bf16; against the float64 q' that is one rounding step
        assert np.all(np.abs(g[kappa] - qp[kappa]) <= 2.0 ** -8 * qp[kappa] + 1e-12)


def test_exact_tensor_core_probability_drafter():
    _exact_case(W.tiny_config(N=1024, n=256, rows=40, trials=2, drafter_kind="probs", dtype="bf16", rho=0.8, emb_dim=16),
                "bf16")


def test_config5_full_size_sampled_outputs():
    """N = 32768, n = 8192, 1024 rows: the checker builds the whole affinity matrix (float64, rounded to
    bf16 for storage), the library contracts it on the tensor cores, and a seeded sample of output
    columns is recomputed by the checker for every row; the sampler then runs on the library's w."""
    rdk = _rdk()
    B = rdk.binding
    cfg = W.CONFIGS["C5"]
    inp = W.make_inputs(cfg, with_embeddings=True)
    kappa = inp["kept_ids"].numpy()
    E64 = W.to_f64(inp["embeddings"])
    Mt = torch.zeros(cfg.N, cfg.n, dtype=torch.bfloat16)
    rng = np.random.default_rng(5)
    cols = np.sort(rng.choice(cfg.N, 48, replace=False))
    Mcols = np.zeros((cfg.n, cols.size))
    for i0 in range(0, cfg.n, 1024):                      # the matrix in blocks of kept rows
        blk = O.round_to_bf16(O.build_affinity(E64, kappa[i0:i0 + 1024], cfg.tau))
        Mt[:, i0:i0 + 1024] = torch.from_numpy(blk.T.copy()).to(torch.bfloat16)
        Mcols[i0:i0 + 1024] = blk[:, cols]
    A = {"data": Mt.cuda(), "layout": B.RDK_AFF_BF16_COLS, "ld": cfg.n}
    idx = rdk.rdk_prepare_ids(inp["kept_ids"].cuda(), cfg.N)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    drafter = inp["drafter"].cuda()
    w, S, _ = rdk.rdk_redistribute_exact(idx, drafter, A, cfg.batch, cfg.positions, KIND[cfg.drafter_kind],
                                         status_word=status)
    torch.cuda.synchronize()
    assert int(status.item()) == 0
    # sampled columns of every row against the checker (operand rounded to bf16 as in the library)
    q = W.to_f64(inp["drafter"])
    qp64 = q / q.sum(axis=1, keepdims=True)
    ref = O.round_to_bf16(qp64) @ Mcols
    got = w[:, torch.from_numpy(cols).cuda()].cpu().double().numpy()
    assert np.all(np.abs(got - ref) <= PU.REL_TOL_BF16 * ref + _flip_allowance(qp64, Mcols) + 1e-12)
    assert np.abs(got - ref).max() <= PU.ABS_TOL
    assert torch.all((S - 1).abs() < 5e-3)                # bf16 rows of M sum to 1 only approximately
    # the library's own affinity construction at this size, on the same sampled columns
    Mg = rdk.rdk_build_affinity(inp["embeddings"].cuda(), inp["kept_ids"].cuda(), cfg.tau, B.RDK_AFF_BF16_COLS)
    torch.cuda.synchronize()
    got_cols = Mg["data"][torch.from_numpy(cols).cuda(), : cfg.n].cpu().double().numpy().T
    assert np.mean(got_cols == Mcols) >= 0.99
    assert np.all(np.abs(got_cols - Mcols) <= 2.0 ** -7 * Mcols + 1e-38)
    # sampler (precomputed-w mode) at full size: its w input is the checker's product for a sample of
    # rows (float32), placed in the rows the checker recomputes; the other rows keep the library's w
    rows = sorted(set([0, cfg.rows - 1] + rng.choice(cfg.rows, 10, replace=False).tolist()))
    w_rows = torch.from_numpy(O.round_to_bf16(qp64[rows]) @ np.vstack([O.round_to_bf16(O.build_affinity(E64, kappa[i0:i0 + 1024], cfg.tau))
                                                                      for i0 in range(0, cfg.n, 1024)])).to(torch.float32)
    w[torch.tensor(rows).cuda()] = w_rows.cuda()
    out = rdk.rdk_sample_and_verify(idx, B.RDK_MODE_PRECOMPUTED_W, inp["target"].cuda(), None, w, inp["uniforms"].cuda(),
                                    cfg.batch, cfg.positions)
    torch.cuda.synchronize()
    t = PU.compare_sampling(inp, out, rows, "given", w_given=w_rows.double().numpy())
    print("C5", t.summary())
    t.assert_ok(max_ambiguous_frac=0.2)


@pytest.mark.parametrize("n,dropped", [(1, False), (255, False), (257, True), (2048, False), (2049, True), (5000, False), (8197, True)])
def test_drafter_sum_has_a_fixed_order(n, dropped):
    """q' of a probability drafter is a quotient of two fp32 numbers, so it can be had to the last bit: the row's sum is taken over
    256 interleaved runs, the runs of 32 neighbours are added in pairs and these eight one after the other.  With the identity as
    affinity the contraction returns it unchanged."""
    rdk = _rdk()
    B = rdk.binding
    N, rows = n + 3, 3
    g = torch.Generator().manual_seed(n)
    q = torch.rand(rows, n, generator=g) ** 4
    ids = torch.arange(n, dtype=torch.int32)
    if dropped:
        ids[5], ids[n - 2] = -1, N
    valid = ((ids >= 0) & (ids < N)).numpy()
    M = torch.zeros(n, N)
    M[torch.arange(n)[valid], ids[valid].long()] = 1.0
    idx = rdk.rdk_prepare_ids(ids.cuda(), N)
    w, _, _ = rdk.rdk_redistribute_exact(idx, q.cuda(), {"data": M.cuda(), "layout": B.RDK_AFF_F32_ROWS, "ld": N}, rows, 1, B.RDK_PROBS)
    v = np.zeros((rows, (n + 255) // 256 * 256), dtype=np.float32)
    v[:, :n] = np.where(valid, q.numpy(), np.float32(0))
    run = np.zeros((rows, 256), dtype=np.float32)
    for part in v.reshape(rows, -1, 256).transpose(1, 0, 2):
        run = run + part
    run = run.reshape(rows, 8, 32)
    for o in (16, 8, 4, 2, 1):
        run = run + run[:, :, np.arange(32) ^ o]
    total = np.zeros(rows, dtype=np.float32)
    for k in range(8):
        total = total + run[:, k, 0]
    want = np.zeros((rows, N), dtype=np.float32)
    want[:, ids.numpy()[valid]] = (q.numpy() * (np.float32(1) / total)[:, None])[:, valid]
    assert np.array_equal(w.cpu().numpy(), want)


@pytest.mark.parametrize("N,rows", [(31, 1), (1024, 4), (4096, 21), (4097, 9), (20000, 5)])
def test_fp32_row_sums_are_repeatable(N, rows):
    """S of the fp32 layout: runs of 16 fp32 additions carried in fp64, in a fixed order, so the same bits every time, and within 15
    roundings of 2^-24 of the terms (16 with the result's own) of the sum of w."""
    rdk = _rdk()
    B = rdk.binding
    n = 64
    g = torch.Generator(device="cuda").manual_seed(N)
    ids = torch.cat([torch.arange(min(n, N)), torch.full((max(0, n - N),), -1)]).to(torch.int32).cuda()
    idx = rdk.rdk_prepare_ids(ids, N)
    M = {"data": torch.rand(n, N, generator=g, device="cuda") ** 6, "layout": B.RDK_AFF_F32_ROWS, "ld": N}
    y = torch.randn(rows, n, generator=g, device="cuda")
    first = None
    for _ in range(20):
        w, S, _ = rdk.rdk_redistribute_exact(idx, y, M, rows, 1)
        first = S.clone() if first is None else first
        assert torch.equal(S, first)
    ref = w.double().sum(1)
    assert ((S.double() - ref).abs() <= 16 * 2.0 ** -24 * ref).all()


@pytest.mark.parametrize("N,rows", [(128000, 320), (100003, 40), (70000, 700), (8192, 300), (33000, 1500)])
def test_bf16_row_sums_take_one_addition_per_cta(N, rows):
    """S of the bf16 layout: a CTA keeps the sums of its rows and adds them to S once, in whatever order.  k fp32 additions of equal
    terms, each off by up to 2^-24 of a running sum that grows to the total, leave a root mean square error of 2^-24 sqrt(k / 3)
    at most; k is one for each SM, and 16 for what a CTA adds up by itself."""
    rdk = _rdk()
    B = rdk.binding
    n = 64
    g = torch.Generator(device="cuda").manual_seed(N)
    idx = rdk.rdk_prepare_ids(torch.arange(n, dtype=torch.int32, device="cuda"), N)
    M = {"data": torch.rand(N, n, generator=g, device="cuda").to(torch.bfloat16), "layout": B.RDK_AFF_BF16_COLS, "ld": n}
    w, S, _ = rdk.rdk_redistribute_exact(idx, torch.randn(rows, n, generator=g, device="cuda"), M, rows, 1)
    ref = torch.cat([x.double().sum(1) for x in w.split(64)])
    k = torch.cuda.get_device_properties(0).multi_processor_count + 16
    assert float(((S.double() / ref - 1) ** 2).mean().sqrt()) <= 2.0 ** -24 * (k / 3) ** 0.5


@pytest.mark.parametrize("N,n,rows", [(18945, 300, 5), (56833, 200, 17), (19000, 130, 33), (20011, 1001, 20), (32768, 520, 250), (40001, 64, 1)])
def test_panels_lower_than_the_instruction(N, n, rows):
    """Up to 256 rows a CTA takes fewer tokens than the instruction has rows where the panels of two CTAs do not fit one round, so that
    every round is full (72 to 112 tokens here, the last panel ragged): every entry of w against a float64 product of the same
    bf16 operands, and its row sums."""
    rdk = _rdk()
    B = rdk.binding
    ctas = torch.cuda.get_device_properties(0).multi_processor_count // 2 * 2
    rounds = -(-(-(-N // 256)) // (ctas // 2))
    assert rounds > 1 and -(-(-(-N // (rounds * ctas))) // 8) * 8 < 128 and N % (-(-(-(-N // (rounds * ctas))) // 8) * 8)
    g = torch.Generator(device="cuda").manual_seed(N)
    idx = rdk.rdk_prepare_ids(torch.arange(n, dtype=torch.int32).cuda(), N)
    ld = (n + 7) // 8 * 8
    Mt = torch.rand(N, ld, generator=g, device="cuda").to(torch.bfloat16)
    q = torch.rand(rows, n, generator=g, device="cuda")
    w, S, _ = rdk.rdk_redistribute_exact(idx, q, {"data": Mt, "layout": B.RDK_AFF_BF16_COLS, "ld": ld}, rows, 1, B.RDK_PROBS)
    torch.cuda.synchronize()
    # the operand as the library rounds it: q / sum in fp32, to bf16; a quotient next to a boundary may be its neighbour (2^-8)
    a = (q.double() / q.double().sum(1, keepdim=True)).to(torch.bfloat16).double()
    ref = a @ Mt[:, :n].double().t()
    # products exact, n fp32 additions of terms of one sign, rounded or cut off; and a neighbour or two moves w by 2^-8 of a term,
    # of which the largest is some four times the mean
    assert float(((w.double() - ref).abs() / ref).max()) <= n * 2.0 ** -23 + 2.0 ** -8 * (2 + n / 4096) * 4 / n
    assert float((S.double() - w.double().sum(1)).abs().max()) <= 3e-6 * float(S.max())
