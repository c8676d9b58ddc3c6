"""The work a user has this library do, as measurable cases.

A case is one pass of one of five jobs, each through the entry points of `paper_2506_03206_b200`:

  step      one verification step of speculative decoding: first-order redistribution, draft draw, rejection test,
            residual draw, then the tokens every sequence emits (rdk_sample_and_verify + rdk_emit_sequences)
  prior     the same with a static prior in place of the target inside the first-order formula, which is what can be
            evaluated before the target model has run (rdk_sample_and_verify_prior)
  exact     exact redistribution through the token-affinity matrix, then the draws from it (rdk_redistribute_exact +
            rdk_sample_and_verify on the weights)
  qtilde    the redistributed drafter written out for all target tokens (rdk_redistribute_linear)
  affinity  the token-affinity matrix itself (rdk_build_affinity)

Sizes are those of `workloads/configs.py` and of the tests, and generic ones between and around them.
"""
import math

import torch

import paper_2506_03206_b200 as rdk

B = rdk.binding
DTYPE = {"bf16": torch.bfloat16, "f32": torch.float32}


def _case(job, N, n, batch=1, positions=1, dtype="bf16", kind="logits", order="ascending", trials=1, pad=1, shared=True,
          layout="bf16", d=0, **more):
    """pad: rows are slices of a buffer whose width is N rounded up to that; order: of the kept ids; layout, d: of the
    affinity matrix and the embeddings that it is built from; shared: one prior row for all rows."""
    c = dict(job=job, N=N, n=n, batch=batch, positions=positions, dtype=dtype, kind=kind, order=order, trials=trials, pad=pad)
    if job == "prior":
        c["shared"] = shared
    if job in ("exact", "affinity"):
        c.update(layout=layout, d=d)
    return dict(more, **c)


def listed():
    return [
        # one user, five drafts, a 128k vocabulary pruned to a quarter: latency of an interactive session
        _case("step", 128256, 32064, 1, 5, name="step_1x5_v128k"),
        # a serving batch on the same model sizes: the benchmark's workload
        _case("step", 128256, 32064, 64, 5, name="step_64x5_v128k"),
        # the largest serving batch, with the largest vocabulary in use
        _case("step", 262144, 32768, 512, 4, name="step_512x4_v262k"),
        # fp32 logits of a small-vocabulary model, kept ids in the order of a frequency ranking, four draws a position
        _case("step", 32000, 8000, 8, 4, dtype="f32", order="ranked", trials=4, name="step_8x4_v32k_f32_ranked"),
        # a vocabulary of odd size: no two rows start at the same alignment
        _case("step", 50257, 12565, 32, 5, name="step_32x5_v50257"),
        # drafting against a static prior, one row for all
        _case("prior", 128256, 32064, 64, 5, name="prior_64x5_v128k"),
        # exact redistribution of the smallest configuration: launches and latency
        _case("exact", 1024, 256, 1, 4, dtype="f32", trials=16, layout="f32", d=64, name="exact_1x4_v1k_f32"),
        # exact redistribution for a few sequences: the affinity matrix is read for twenty rows
        _case("exact", 32768, 8192, 4, 5, kind="probs", d=128, name="exact_4x5_v32k"),
        # exact redistribution for a large batch: a dense contraction
        _case("exact", 32768, 8192, 1024, 1, kind="probs", d=128, name="exact_1024_v32k"),
        # the same at a 128k vocabulary, rows that do not fill whole tiles
        _case("exact", 128256, 32064, 64, 5, d=256, name="exact_64x5_v128k"),
        # the redistributed distribution itself, for analysis and for samplers of one's own
        _case("qtilde", 128256, 12826, 16, 5, name="qtilde_16x5_v128k"),
        # once for each model and kept-id list, before serving
        _case("affinity", 32768, 8192, d=128, name="affinity_v32k"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _vocabulary(rng, lo, hi):
    """Half of the sizes are multiples of 64, as padded heads have; the others are whatever comes."""
    N = _log(rng, lo, hi)
    return max(lo, N // 64 * 64) if rng.random() < 0.5 else N


def _rows(rng, most):
    """(batch, positions) with at most `most` rows."""
    positions = rng.randint(1, max(1, min(8, most)))
    return _log(rng, 1, max(1, min(512, most // positions))), positions


def draw(rng):
    job = rng.choices(("step", "prior", "exact", "qtilde", "affinity"), (55, 10, 15, 10, 10))[0]
    if job == "affinity":
        f32 = rng.random() < 0.25
        N = _vocabulary(rng, 1000, 8000 if f32 else 65536)
        d = rng.choice((64, 72, 100, 128, 256, 384, 512))
        n = max(16, min(int(N * rng.uniform(0.05, 0.3)), int((2e9 / d if f32 else 268e6) / N)))
        return _case(job, N, n, dtype="f32" if f32 else "bf16", layout="f32" if f32 else "bf16", d=d)
    if job == "exact":
        f32 = rng.random() < 0.25
        N = _vocabulary(rng, 1000, 2048 if f32 else 65536)
        n = int(N * rng.uniform(0.05, 0.3))
        batch, positions = _rows(rng, 16 if f32 else min(1024, int(2.7e11 / N / n)))
        return _case(job, N, n, batch, positions, dtype="f32" if f32 else "bf16", kind=rng.choice(("logits", "probs")),
                     trials=rng.choice((1, 1, 4)), layout="f32" if f32 else "bf16", d=rng.choice((64, 128, 256)))
    N = _vocabulary(rng, 1000, 262144)
    n = max(4, int(N * math.exp(rng.uniform(math.log(0.0025), math.log(0.5)))))
    batch, positions = _rows(rng, int({"step": 134e6, "prior": 41e6, "qtilde": 20e6}[job] / N))
    return _case(job, N, n, batch, positions, dtype="f32" if rng.random() < 0.25 else "bf16",
                 kind="probs" if rng.random() < 0.2 else "logits", order="ranked" if rng.random() < 0.2 else "ascending",
                 trials=1 if job == "qtilde" or rng.random() < 0.75 else rng.randint(2, 8),
                 pad=64 if rng.random() < 0.5 else 1, shared=rng.random() < 0.7)


def _wide(rows, N, pad, dtype):
    return torch.empty(rows, -(-N // pad) * pad, dtype=dtype, device="cuda")[:, :N]


def prepare(case, seed):
    c, dev = case, "cuda"
    N, n, batch, positions, job = c["N"], c["n"], c["batch"], c["positions"], c["job"]
    rows, dtype = batch * positions, DTYPE[c["dtype"]]
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    # a frequency ranking of the vocabulary; the drafter keeps the most frequent n tokens
    ranking = torch.randperm(N, generator=g, device=dev)
    ids = (ranking[:n] if c["order"] == "ranked" else torch.sort(ranking[:n]).values).to(torch.int32)
    s = {"case": dict(c), "ids": ids}
    if job in ("exact", "affinity"):
        s["embeddings"] = torch.randn(N, c["d"], generator=g, device=dev).to(dtype)
        s["layout"] = B.RDK_AFF_F32_ROWS if c["layout"] == "f32" else B.RDK_AFF_BF16_COLS
    if job == "affinity":
        return s
    # logits as language models give them: long-tailed over the frequency ranks, a per-row spread of 2 to 4, the
    # drafter correlated with the target
    sigma, rho = 3.0, 0.8
    bias = torch.empty(N, device=dev)
    bias[ranking] = -1.1 * torch.log(torch.arange(1, N + 1, device=dev, dtype=torch.float32))
    target, drafter = _wide(rows, N, c["pad"], dtype), torch.empty(rows, n, dtype=dtype, device=dev)
    at = ids.long()
    for r in range(0, rows, 128):
        e = min(rows, r + 128)
        z = torch.randn(e - r, N, generator=g, device=dev)
        y = bias[at] + sigma * (rho * z[:, at] + math.sqrt(1 - rho * rho) * torch.randn(e - r, n, generator=g, device=dev))
        target[r:e] = (z * sigma + bias).to(dtype)
        drafter[r:e] = (torch.softmax(y, -1) if c["kind"] == "probs" else y).to(dtype)
    s.update(index=rdk.rdk_prepare_ids(ids, N), target=target, drafter=drafter,
             kind=B.RDK_PROBS if c["kind"] == "probs" else B.RDK_LOGITS)
    # uniforms are 24-bit numbers in [0, 1)
    s["uniforms"] = torch.randint(0, 1 << 24, (rows, c["trials"], 4), generator=g, device=dev).float() / (1 << 24)
    if job == "qtilde":
        return s
    if job == "prior":
        prior = torch.randn(1 if c["shared"] else rows, N, generator=g, device=dev) * 0.5 + bias
        s["prior"] = prior[0].to(dtype) if c["shared"] else prior.to(dtype)
    if job == "exact":
        s["M"] = rdk.rdk_build_affinity(s.pop("embeddings"), ids, 0.1, s["layout"])
        torch.cuda.synchronize()
        s["M"].pop("_ws", None)
        s["w"] = torch.empty(rows, N, device=dev)
        problem = B.make_problem(s["index"], None, drafter, batch, positions, s["kind"])
        s["exact_ws"] = torch.empty(max(256, B.lib().rdk_exact_workspace_bytes(B.C.byref(problem), s["layout"])),
                                    dtype=torch.uint8, device=dev)
    if job == "step":
        s["bonus"] = _wide(batch, N, c["pad"], dtype)
        s["bonus"].copy_((torch.randn(batch, N, generator=g, device=dev) * sigma + bias).to(dtype))
    # a decoding loop keeps its output buffers and workspace; it does not ask for the acceptance probability of each
    # draw, only for the draws, whether they were accepted, and the row statistics
    out = B.alloc_outputs(rows, batch, c["trials"], dev)
    del out["accept_prob"]
    s["out"] = out
    problem = B.make_problem(s["index"], target, drafter, batch, positions, s["kind"])
    s["mode"] = B.RDK_MODE_PRECOMPUTED_W if job == "exact" else B.RDK_MODE_LINEAR
    s["ws"] = B.sample_workspace(problem, s["mode"], c["trials"], dev)
    return s


def run(s):
    c = s["case"]
    batch, positions, job = c["batch"], c["positions"], c["job"]
    if job == "affinity":
        return rdk.rdk_build_affinity(s["embeddings"], s["ids"], 0.1, s["layout"])["data"]
    if job == "qtilde":
        return rdk.rdk_redistribute_linear(s["index"], s["target"], s["drafter"], batch, positions, s["kind"])
    more = {}
    if job == "prior":
        out = rdk.rdk_sample_and_verify_prior(s["index"], s["target"], s["prior"], s["drafter"], s["uniforms"], batch,
                                              positions, s["kind"], out=s["out"])
    elif job == "exact":
        more["w"], more["w_sum"], _ = rdk.rdk_redistribute_exact(s["index"], s["drafter"], s["M"], batch, positions, s["kind"],
                                                                 w_out=s["w"], ws=s["exact_ws"],
                                                                 status_word=s["out"]["status_word"])
        out = rdk.rdk_sample_and_verify(s["index"], s["mode"], s["target"], None, s["w"], s["uniforms"], batch, positions,
                                        out=s["out"], ws=s["ws"])
    else:
        out = rdk.rdk_sample_and_verify(s["index"], s["mode"], s["target"], s["drafter"], None, s["uniforms"], batch,
                                        positions, s["kind"], out=s["out"], ws=s["ws"])
        more["seq_tokens"], more["seq_len"] = rdk.rdk_emit_sequences(c["N"], batch, positions, s["bonus"], s["uniforms"],
                                                                     out["draft_token"], out["accepted"], out["out_token"])
    return dict({k: v for k, v in out.items() if k != "_ws"}, **more)


def work(case):
    """Each input read once, each output written once. The bonus rows of a step are not counted: only a sequence whose
    drafts were all accepted needs one."""
    c = case
    N, n, rows, job = c["N"], c["n"], c["batch"] * c["positions"], c["job"]
    size = 2 if c["dtype"] == "bf16" else 4
    if job == "affinity":
        m = 2 if c["layout"] == "bf16" else 4
        return {"bytes": N * c["d"] * size + 4 * n + m * n * N, "flops": 2 * n * N * c["d"]}
    target, drafter = rows * N * size, rows * n * size
    draws = rows * c["trials"] * (16 + 9) + rows * 16
    if job == "qtilde":
        return {"bytes": target + drafter + 4 * rows * N, "flops": rows * (6 * N + 6 * n)}
    if job == "exact":
        m = 2 if c["layout"] == "bf16" else 4
        return {"bytes": drafter + m * n * N + 4 * rows * N + target + draws, "flops": 2 * rows * n * N}
    prior = 0 if job == "step" else (1 if c["shared"] else rows) * N * size
    return {"bytes": target + drafter + prior + draws, "flops": rows * (6 * N + 10 * n)}


def tolerance(case):
    """Sums are taken in fp32, over values that are exact in their own type. The drafter operand and the affinity matrix
    of the bf16 layout are rounded to bf16, where two correct fp32 values may land on either side of a boundary. A draw
    whose threshold lies within rounding of a boundary of the distribution may give the neighbouring token."""
    bf16_matrix = case["job"] in ("exact", "affinity") and case["layout"] == "bf16"
    t = {"rel": 2e-3, "max": 1e-2} if bf16_matrix else {"rel": 2e-5}
    if case["job"] in ("step", "prior", "exact"):
        t["differ"] = 0.01
    return t
