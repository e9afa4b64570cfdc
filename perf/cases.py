"""Performance cases of the solve + verify path: the calls a serving stack or an acceptance study makes, over the range
of vocabularies, batches, draft counts, supports and element types that the library takes.

A case is a dict of plain values:
  call      "two"    gr_solve followed by gr_verify (binding: solve, verify)
            "fused"  gr_solve_verify, one call
            "alpha"  gr_alpha_star for every draft count in `n_list`
            "host"   solve_verify_host: pinned host logits in, host tokens out
  config    which of the seeded input families of `workloads` the logits come from (1..5)
  V, n, topk (0 = the whole vocabulary), batch, dtype; sigma (config 4: distance between draft and target logits);
  tau       error threshold of Algorithm 1 (0 = the exact rule)

`prepare` makes what a caller has in hand (logits, drafted tokens, uniforms on the device; pinned host buffers for
"host") and the result objects it keeps from call to call.
"""
from __future__ import annotations

import math

import torch

import paper_2511_15898_b200 as G
from paper_2511_15898_b200 import workloads as W


def _case(name, call, config, V, n, topk, batch, dtype="f32", sigma=0.0, tau=0.0, n_list=""):
    return {"name": name, "call": call, "config": config, "V": V, "n": n, "topk": topk, "batch": batch, "dtype": dtype,
            "sigma": sigma, "tau": tau, "n_list": n_list}


def listed():
    return [
        # one sequence being decoded: latency of a single position at the headline shape
        _case("decode-one", "two", 3, 128256, 8, 50, 1),
        # tiny vocabulary, untruncated draft, acceptance close to one (heavy weights, many iterations)
        _case("tiny-full", "two", 1, 16, 2, 0, 64),
        # a 32k-vocabulary model with short drafts and a narrow sampler
        _case("v32k-n4-k8", "two", 2, 32000, 4, 8, 256),
        # the headline: a full decode batch of a 128k-vocabulary model
        _case("headline", "two", 3, 128256, 8, 50, 1024),
        # the same model served with bf16 logits at an ordinary batch, drafts known beforehand: one fused call
        _case("bf16-fused-128", "fused", 3, 128256, 8, 50, 128, dtype="bf16"),
        # long drafts on an odd vocabulary (rows are not 16-byte aligned)
        _case("v50k-n16-k20", "fused", 4, 50257, 16, 20, 512, sigma=2.0),
        # more than 16 drafts: the general solver, with dominant draft tokens
        _case("v50k-n32-k20", "two", 4, 50257, 32, 20, 512, sigma=1.0),
        # untruncated draft on a large vocabulary: optimal acceptance, then a sample of the target
        _case("v50k-whole", "two", 4, 50257, 8, 0, 512, sigma=1.0),
        # acceptance against the number of drafts from one pass over the logits
        _case("alpha-sweep-k20", "alpha", 4, 50257, 32, 20, 512, sigma=1.0, n_list="2,4,8,16,32"),
        # the error-threshold variant of Algorithm 1 at the paper's threshold
        _case("tau-1e-3", "two", 3, 128256, 8, 50, 512, tau=1e-3),
        # large serving batch: 152k vocabulary, 16 drafts of a top-100 sampler, bf16 logits
        _case("serving-4096", "two", 5, 152064, 16, 100, 4096, dtype="bf16"),
        # logits that live in host memory (an engine whose models run elsewhere)
        _case("host-32", "host", 3, 128256, 8, 50, 32),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(["two", "two", "two", "fused", "fused", "alpha", "tau", "long", "whole", "tiny", "host"])
    dtype = rng.choice(["f32", "f32", "bf16"])
    sigma = rng.choice([0.25, 0.5, 1.0, 2.0])
    if kind == "tiny":
        return _strip(_case("", rng.choice(["two", "fused"]), 1, 16, 2, 0, _log_int(rng, 1, 256)))
    V = _log_int(rng, 300, 152064)
    most = 150_000_000 // V                       # logits of one model per call
    if kind == "whole":
        V = min(V, 60000)
        call, n = rng.choice([("two", rng.randint(2, 32)), ("alpha", 32)])
        return _strip(_case("", call, 4, V, n, 0, _log_int(rng, 1, 512), dtype=dtype, sigma=sigma,
                            n_list="2,8,32" if call == "alpha" else ""))
    if kind == "alpha":
        return _strip(_case("", "alpha", rng.choice([3, 4]), V, 32, _log_int(rng, 4, 128),
                            min(most, _log_int(rng, 1, 1024)), dtype=dtype, sigma=sigma,
                            n_list=rng.choice(["2,4,8,16,32", "1,2,3,4,5,6,7,8", "8"])))
    if kind == "long":
        return _strip(_case("", rng.choice(["two", "fused"]), 4, V, rng.randint(17, 32), _log_int(rng, 4, 32),
                            min(most, _log_int(rng, 1, 512)), dtype=dtype, sigma=sigma))
    if kind == "host":
        return _strip(_case("", "host", 3, V, rng.randint(2, 8), _log_int(rng, 4, 64),
                            min(most, 6_000_000 // V + 1, _log_int(rng, 1, 64)), dtype=dtype))
    config = rng.choice([3, 3, 4])
    n, topk = rng.randint(2, 16), _log_int(rng, 4, 128)
    batch = min(most, _log_int(rng, 1, 2048))
    tau = 1e-3 if kind == "tau" else 0.0
    return _strip(_case("", "two" if kind == "tau" else kind, config, V, n, topk, batch, dtype=dtype,
                        sigma=sigma, tau=tau))


def _strip(case):
    return {k: v for k, v in case.items() if k != "name"}


def _workload(case, seed, device):
    config, B, V, n, topk = case["config"], case["batch"], case["V"], case["n"], case["topk"]
    if config == 1:
        return W.config1(batch=B, device=device, seed=seed)
    if config == 2:
        return W.config2(batch=B, device=device, seed=seed, V=V)
    if config == 3:
        return W.config3(batch=B, device=device, seed=seed, V=V, n=n, topk=topk)
    if config == 4:
        return W.config4(n, topk, case["sigma"], batch=B, device=device, seed=seed, V=V)
    return W.config5(batch=B, device=device, seed=seed, V=V, n=n, topk=topk)


def prepare(case, seed):
    dev = torch.device("cuda")
    wl = _workload(case, seed, dev)
    q, p, toks, uni = wl.q_logits, wl.p_logits, wl.draft_tokens, wl.uniforms
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    if q.dtype != dtype:
        q, p = q.to(dtype), p.to(dtype)
        # (rounding the logits can change the support: the draft model samples from the rounded ones)
        g = torch.Generator(device=dev)
        g.manual_seed(seed)
        toks = W.sample_draft_tokens(p, case["topk"], wl.temp_draft, case["n"], g)
    state = {"case": case, "n": case["n"], "topk": case["topk"], "tt": wl.temp_target, "td": wl.temp_draft,
             "opt": G.Options(tau=case["tau"]) if case["tau"] > 0 else None}
    if case["call"] == "host":
        state.update(q=q.cpu().pin_memory(), p=p.cpu().pin_memory(), toks=toks.cpu().pin_memory(),
                     uni=uni.cpu().pin_memory(), buffers={})
    else:
        state.update(q=q, p=p, toks=toks, uni=uni, solved=None, verified=None)
    if case["call"] == "alpha":
        state["n_list"] = [int(x) for x in case["n_list"].split(",")]
    return state


def run(state):
    s, call = state, state["case"]["call"]
    if call == "alpha":
        alpha, status = G.alpha_star(s["q"], s["p"], s["n_list"], s["topk"], s["tt"], s["td"])
        return {"alpha_star": alpha, "status": status}
    if call == "host":
        token, accepted, alpha, status = G.solve_verify_host(s["q"], s["p"], s["toks"], s["uni"], s["n"], s["topk"],
                                                             s["tt"], s["td"], s["opt"], "cuda:0", s["buffers"])
        return {"token": token, "accepted": accepted, "alpha_star": alpha, "status": status}
    if call == "fused":
        pair = (s["solved"], s["verified"]) if s["solved"] is not None else None
        s["solved"], s["verified"] = G.solve_verify(s["q"], s["p"], s["toks"], s["uni"], s["topk"], s["tt"], s["td"],
                                                    s["opt"], pair)
    else:
        s["solved"] = G.solve(s["q"], s["p"], s["n"], s["topk"], s["tt"], s["td"], s["opt"], s["solved"])
        s["verified"] = G.verify(s["solved"], s["toks"], s["uni"], s["verified"])
    v = s["verified"]
    return {"token": v.token, "accepted": v.accepted, "alpha_star": s["solved"].alpha_star,
            "solve_status": s["solved"].status, "status": v.status}


def work(case):
    """Both logit rows read once, drafted tokens and uniforms read, results written.  Operations: two per logit for
    the target's (and an untruncated draft's) exponential sum, and one evaluation of the gradient of the convex
    programs at the solution (series of n terms per token at 26 quadrature nodes)."""
    B, V, n, topk = case["batch"], case["V"], case["n"], case["topk"]
    esize = 2 if case["dtype"] == "bf16" else 4
    k = V if (topk <= 0 or topk >= V) else topk
    counts = len(case["n_list"].split(",")) if case["call"] == "alpha" else 0
    nbytes = B * (2 * V * esize + (4 * counts + 4 if counts else 4 * n + 8 + 13))
    flops = 2.0 * B * V * (2 if k > G.binding.GR_MAX_SUPPORT else 1)
    if not counts and k <= G.binding.GR_MAX_SUPPORT:
        flops += 2.0 * B * 26 * (k * (n * (n - 1) / 2 + 2 * n) + n * (n + 1) / 2)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Optimal acceptance: an fp32 sum over the row (a few 1e-7 absolute).  Tokens: a draw within about 1e-6 of a
    boundary of its cumulative distribution may fall on either side; under an error threshold tau any rule within
    15 tau of the target in L1 is a correct one."""
    return {"rel": 1e-5, "max": 4e-4, "differ": min(0.01, 7.5 * case["tau"]) if case["tau"] > 0 else 1e-3}
