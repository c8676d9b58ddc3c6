"""The calls with one prior row for all rows that the streaming kernels serve: workspace, capture, several draws and positions, odd
sizes, a wait that gives up, precision."""
import numpy as np
import pytest
import torch

import parity_util as PU
import workloads as W
from oracle import rdk_oracle as O

pytestmark = pytest.mark.gpu

OUTPUTS = ("draft_token", "out_token", "accepted", "accept_prob", "alpha", "theta", "S", "residual_mass", "accepted_len")


def _rdk():
    import paper_2506_03206_b200 as rdk
    return rdk


def _device_inputs(N, n, batch, positions, trials, seed):
    """Random inputs made on the device, where no row is compared with the oracle."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    rows = batch * positions
    z = (torch.randn(rows, N, generator=g, device="cuda") * 2).to(torch.bfloat16)
    y = (torch.randn(rows, n, generator=g, device="cuda") * 2).to(torch.bfloat16)
    prior = (torch.randn(N, generator=g, device="cuda") * 2).to(torch.bfloat16)
    u = torch.randint(0, 1 << 24, (rows, trials, 4), generator=g, device="cuda").float() / (1 << 24)
    ids = torch.sort(torch.randperm(N, generator=g, device="cuda")[:n]).values.to(torch.int32)
    return z, prior, y, u, ids


def _wanted(rdk, idx, z, prior, y, batch, positions, trials):
    """Bytes of workspace with which the streaming kernels serve (0: they do not)."""
    B = rdk.binding
    pb = B.make_problem(idx, z, y, batch, positions)
    return B.lib().rdk_sample_prior_workspace_bytes(B.C.byref(pb), z.data_ptr(), prior.data_ptr(), 0, y.data_ptr(), trials)


def test_no_memory_for_a_workspace_is_no_error():
    """The call needs no workspace; where the allocator has none to give, the cluster kernel serves."""
    rdk = _rdk()
    N, n, rows = 16384, 2000, 5000
    z, prior, y, u, ids = _device_inputs(N, n, rows, 1, 1, 3)
    idx = rdk.rdk_prepare_ids(ids, N)
    assert _wanted(rdk, idx, z, prior, y, rows, 1, 1) > 24 << 20
    want = rdk.rdk_sample_and_verify_prior(idx, z, prior, y, u, rows, 1)
    out = rdk.binding.alloc_outputs(rows, rows, 1, "cuda")
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    total = torch.cuda.get_device_properties(0).total_memory
    try:
        torch.cuda.set_per_process_memory_fraction((torch.cuda.memory_reserved() + (4 << 20)) / total)
        held, size = [], 1 << 28                         # what is left over in the allocator's blocks
        while size > 1 << 21:
            try:
                held.append(torch.empty(size, dtype=torch.uint8, device="cuda"))
            except torch.cuda.OutOfMemoryError:
                size >>= 1
        rdk.rdk_sample_and_verify_prior(idx, z, prior, y, u, rows, 1, out=out)
    finally:
        held = None
        torch.cuda.set_per_process_memory_fraction(1.0)
    torch.cuda.synchronize()
    rdk.binding.check_status_word(out)
    for k in ("alpha", "theta", "S", "residual_mass"):
        assert float((out[k] - want[k]).abs().max()) < 1e-5, k
    # a draw on the other side of a boundary: prefix sums 1e-7 apart, some 2 n interval ends (as in assert_ok_at_scale)
    assert int((out["draft_token"] != want["draft_token"]).sum()) <= 2 + 6e-7 * n * rows


def test_a_workspace_of_the_callers_also_under_capture():
    """With `ws` the call is the same in a graph as outside of one, bit for bit and with new inputs in the same buffers; without, a captured
    call takes the cluster kernel, as does one with a workspace that is too small.  The streaming kernels leave a record of each
    row at the start of the workspace."""
    rdk = _rdk()
    B = rdk.binding
    N, n, batch, positions, trials = 50264, 9000, 40, 5, 2
    sets = [_device_inputs(N, n, batch, positions, trials, 70 + k) for k in range(3)]
    ids = sets[0][4]
    idx = rdk.rdk_prepare_ids(ids, N)
    buf = [t.clone() for t in sets[0][:4]]
    z, prior, y, u = buf
    need = _wanted(rdk, idx, z, prior, y, batch, positions, trials)
    assert need > 0
    ws = B.sample_workspace(B.make_problem(idx, z, y, batch, positions), B.RDK_MODE_LINEAR, trials, "cuda")
    assert ws.numel() >= need
    head = 4160 * batch * positions

    def call(out, ws):
        return rdk.rdk_sample_and_verify_prior(idx, z, prior, y, u, batch, positions, out=out, ws=ws)

    def outs():
        return B.alloc_outputs(batch * positions, batch, trials, "cuda")

    for given, streams in ((ws, True), (ws[: need // 2], False), (ws[:0], False)):
        ws.fill_(0xA5)
        call(outs(), given)
        torch.cuda.synchronize()
        assert bool((ws[:head] != 0xA5).any()) == streams, given.numel()
    captured, plain = outs(), outs()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        call(captured, ws)
    for inputs in sets + sets[:1]:
        for b, t in zip(buf, inputs):
            b.copy_(t)
        ws.fill_(0xA5)
        graph.replay()
        torch.cuda.synchronize()
        assert bool((ws[:head] != 0xA5).any())
        call(plain, ws)
        torch.cuda.synchronize()
        B.check_status_word(captured)
        for k in OUTPUTS:
            assert torch.equal(captured[k], plain[k]), k
    without, graph = outs(), torch.cuda.CUDAGraph()
    call(without, ws[:0])
    with torch.cuda.graph(graph):
        call(captured, None)
    graph.replay()
    torch.cuda.synchronize()
    for k in OUTPUTS:
        assert torch.equal(captured[k], without[k]), k


@pytest.mark.parametrize("shared_prior", [False, True])
def test_alpha_is_the_records_sum_rounded_once(shared_prior):
    """The draw kernel adds the segments' shares of alpha up in fp64, as it does those of the weights: the result is the sum of the
    row's records (16 scalars, then four sums a segment, the second of min(p, q~)) rounded to fp32 once."""
    rdk = _rdk()
    B = rdk.binding
    N, n, rows = 131072, 600, 300
    z, prior, y, u, ids = _device_inputs(N, n, rows, 1, 1, 11)
    idx = rdk.rdk_prepare_ids(ids, N)
    ws = B.sample_workspace(B.make_problem(idx, z, y, rows, 1), B.RDK_MODE_LINEAR, 1, "cuda")
    if shared_prior:
        assert _wanted(rdk, idx, z, prior, y, rows, 1, 1) > 0
        out = rdk.rdk_sample_and_verify_prior(idx, z, prior, y, u, rows, 1, ws=ws)
    else:
        assert rdk.rdk_sample_route(idx, B.RDK_MODE_LINEAR, z, y, rows, 1, 1, ws)[0] == B.RDK_ROUTE_STREAM_KERNEL
        out = rdk.rdk_sample_and_verify(idx, B.RDK_MODE_LINEAR, z, y, None, u, rows, 1, ws=ws)
    torch.cuda.synchronize()
    B.check_status_word(out)
    geo = rdk.rdk_stream_geometry(N, n)
    record = ws[: 4160 * rows].view(rows, 4160)[:, 64:].contiguous().view(torch.float32).view(rows, 256, 4)
    sums = record[:, : geo["ctas_per_row"] * geo["warps_per_cta"], 1].double().sum(1)
    assert torch.equal(out["alpha"], sums.float())


# Beside each: what the streaming kernels / the cluster kernel take, in us
@pytest.mark.parametrize("N,n,rows,trials,streams", [
    (200000, 8000, 1, 1, False), (262144, 65536, 6, 1, False), (100032, 25008, 8, 2, False), (16384, 4096, 96, 1, False),       # 16.8 / 10.1, 19.4 / 12.3, 17.3 / 10.7, 17.5 / 11.0
    (128256, 32064, 4, 1, False), (128256, 32064, 64, 1, True), (200000, 50000, 48, 1, True), (128256, 32064, 8, 16, True),    # 16.9 / 10.3, 25.0 / 33.0, 25.8 / 36.9, 18.3 / 26.1
    (32000, 4000, 160, 64, True), (16384, 2048, 640, 16, True)])                                                            # beside one CTA per row: 85 / 105, 89 / 125
def test_route_of_few_rows_with_a_prior(N, n, rows, trials, streams):
    rdk = _rdk()
    z, prior, y, u, ids = _device_inputs(N, n, rows, 1, trials, N)
    idx = rdk.rdk_prepare_ids(ids, N)
    assert (_wanted(rdk, idx, z, prior, y, rows, 1, trials) > 0) == streams


@pytest.mark.parametrize("N,n,rows,trials", [(50264, 9000, 200, 2), (128256, 32064, 8, 16), (16384, 4000, 700, 1)])
def test_a_wait_that_runs_out_with_a_prior(N, n, rows, trials):
    """With the limit of the device-side waits at one failed try, the waits for the exchange (and now and then for the copies, those of the
    prior's slice among them) run out; every warp still reaches the end of the kernel, which takes up its copies, and the status word says
    so.  With the default limit restored the same call on the same workspace is right again.  Groups of several rows and of one."""
    rdk = _rdk()
    B = rdk.binding
    z, prior, y, u, ids = _device_inputs(N, n, rows, 1, trials, 5)
    idx = rdk.rdk_prepare_ids(ids, N)
    assert _wanted(rdk, idx, z, prior, y, rows, 1, trials) > 0
    ws = B.sample_workspace(B.make_problem(idx, z, y, rows, 1), B.RDK_MODE_LINEAR, trials, "cuda")
    want = rdk.rdk_sample_and_verify_prior(idx, z, prior, y, u, rows, 1, ws=ws)
    torch.cuda.synchronize()
    B.check_status_word(want)
    try:
        rdk.rdk_test_set_spin_limit(1)
        for _ in range(5):
            out = rdk.rdk_sample_and_verify_prior(idx, z, prior, y, u, rows, 1, ws=ws)
            torch.cuda.synchronize()
            assert int(out["status_word"].item()) == B.RDK_ERR_TIMEOUT
    finally:
        rdk.rdk_test_set_spin_limit(0)
    out = rdk.rdk_sample_and_verify_prior(idx, z, prior, y, u, rows, 1, ws=ws)
    torch.cuda.synchronize()
    B.check_status_word(out)
    for k in OUTPUTS:
        assert torch.equal(out[k], want[k]), k


# Rows padded to 64 elements, so that any N has them on 16-byte boundaries: the prior's slice and the target's end inside a vector
@pytest.mark.parametrize("N,n,batch,positions,trials", [(50257, 12566, 30, 5, 3), (24583, 2000, 120, 4, 1), (65543, 9000, 3, 40, 4), (131071, 20002, 12, 7, 16)])
def test_shared_prior_of_any_size(N, n, batch, positions, trials):
    rdk = _rdk()
    B = rdk.binding
    rows = batch * positions
    cfg = W.tiny_config(N=N, n=n, rows=rows, dtype="bf16", trials=trials, rho=0.8, seed=N, zipf_bias=True).with_rows(batch, positions)
    inp = W.make_inputs(cfg)
    idx = rdk.rdk_prepare_ids(inp["kept_ids"].cuda(), N)
    wide = torch.full((rows, -(-N // 64) * 64), 50.0, dtype=torch.bfloat16, device="cuda")       # (what lies beyond N must not count)
    wide[:, :N] = inp["target"].cuda()
    z, y, u = wide[:, :N], inp["drafter"].cuda(), inp["uniforms"].cuda()
    g = torch.Generator().manual_seed(N)
    prior = (inp["target"][0].float() * 0.8 + torch.randn(N, generator=g)).to(torch.bfloat16)
    prior_dev = torch.full((N + 8,), 50.0, dtype=torch.bfloat16, device="cuda")[:N].copy_(prior)
    assert _wanted(rdk, idx, z, prior_dev, y, batch, positions, trials) > 0
    out = rdk.rdk_sample_and_verify_prior(idx, z, prior_dev, y, u, batch, positions)
    ref = rdk.rdk_sample_and_verify_prior(idx, z, prior_dev.expand(rows, N).contiguous(), y, u, batch, positions)
    torch.cuda.synchronize()
    for o in (out, ref):
        B.check_status_word(o)
        PU.compare_accepted_len(o, batch, positions, trials)
    PU.compare_sampling(inp, out, sorted({0, 1, rows // 2, rows - 2, rows - 1}), "linear", prior=prior).assert_ok()
    for k in ("alpha", "theta", "S", "residual_mass"):
        assert float((out[k] - ref[k]).abs().max()) < 1e-5, k
    assert int((out["draft_token"] != ref["draft_token"]).sum()) <= 2 + 6e-7 * n * rows * trials


@pytest.mark.parametrize("shift", [0.0, 12.0, 30.0, -30.0])
def test_shared_prior_above_and_below_the_target(shift):
    """theta pi / N is the smaller of the two nearly everywhere, or for half of the tokens, or hardly anywhere: the second visit takes
    away what it is above p, where the smallest difference of a lane's logits says that there is any."""
    rdk = _rdk()
    B = rdk.binding
    N, n, rows, trials = 37003, 5000, 160, 2
    cfg = W.tiny_config(N=N, n=n, rows=rows, dtype="bf16", trials=trials, rho=0.7, seed=31)
    inp = W.make_inputs(cfg)
    g = torch.Generator().manual_seed(3)
    prior = torch.randn(N, generator=g)
    prior[: N // 2] += shift
    prior[11] = -float("inf")
    inp["target"][:, 13] = -float("inf")
    inp["target"][7, N // 2:] = -float("inf")            # every token of a segment where there is none of the target
    prior = prior.to(torch.bfloat16)
    idx = rdk.rdk_prepare_ids(inp["kept_ids"].cuda(), N)
    wide = torch.zeros(rows, -(-N // 64) * 64, dtype=torch.bfloat16, device="cuda")
    wide[:, :N] = inp["target"].cuda()
    z, y, u = wide[:, :N], inp["drafter"].cuda(), inp["uniforms"].cuda()
    assert _wanted(rdk, idx, z, prior.cuda(), y, rows, 1, trials) > 0
    out = rdk.rdk_sample_and_verify_prior(idx, z, prior.cuda(), y, u, rows, 1)
    torch.cuda.synchronize()
    B.check_status_word(out)
    PU.compare_sampling(inp, out, sorted({0, 1, 7, *range(8, rows, 13)}), "linear", prior=prior).assert_ok()
    # tokens that are not kept and lie below theta pi / N, all rows: the share of alpha that the test is about
    p, pi = torch.softmax(z.double(), 1), torch.softmax(prior.cuda().double(), 0)
    q = torch.zeros_like(p)
    q[:, inp["kept_ids"].cuda().long()] = torch.softmax(y.double(), 1)
    theta = (pi * q).sum(1, keepdim=True)
    w = (N * q + theta * pi) / (N + pi)
    w = w / w.sum(1, keepdim=True)
    assert bool(((theta * pi / N > p) & (q == 0)).any())
    assert float((out["alpha"].double() - torch.minimum(p, w).sum(1)).abs().max()) < 1e-5
